"""GPU: the protein search kernel (ga_prot.cuh) at the edges of its tiles, stages and
row batches, for alphabets and gap costs at the ends of their ranges."""
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402

NTHREADS = os.cpu_count() or 8
WIDTHS = [128, 192, 256, 320, 384, 448, 512, 640, 768, 896, 1024]


@pytest.mark.parametrize("A,alpha,beta,lo,hi", [(20, 11, 1, -4, 11), (5, 1, 1, -1, 1), (31, 4096, 4096, -127, 127),
                                                (24, 1, 1, -2, 9)])
def test_tile_stage_and_batch_edges(A, alpha, beta, lo, hi):
    rng = np.random.default_rng(A)
    mat = rng.integers(lo, 1, size=(A, A)).astype(np.int8)
    np.fill_diagonal(mat, hi)
    qlens = [0, 1, 2] + [w + d for w in WIDTHS for d in (-1, 0, 1)]
    qs = [rng.integers(0, A, size=n).astype(np.uint8) for n in qlens]
    ts = [rng.integers(0, A, size=n).astype(np.uint8) for n in
          [0, 1, 2, 14, 15, 16, 17, 18, 30, 31, 32, 33, 47, 48, 49, 63, 64, 65, 130]]
    # related targets: alignments that cross stage edges and end in the last rows and columns
    for k in range(8, len(qs), 3):
        t = np.delete(qs[k], rng.integers(0, len(qs[k]), size=len(qs[k]) // 30))
        ts += [t, t[-int(rng.integers(20, 60)):]]
    qc, qo = synth.pack_csr(qs)
    tc, to = synth.pack_csr(ts)
    dev = [torch.from_numpy(a).cuda() for a in (qc, qo, tc, to)]
    got, st = ga.align_cross(*dev, mat, alpha, beta, "local", stats=True)
    want, _ = oracle.cross(qc, qo, tc, to, mat, alpha, beta, "local", nthreads=NTHREADS)
    assert np.array_equal(got.cpu().numpy().ravel(), want.ravel()) and st["status"] == 0
    # one query, so that its bin is the only launch; the same scores
    for k in (1, 12, len(qs) - 1):
        one = ga.align_cross(dev[0], dev[1][k:k + 2].contiguous(), *dev[2:], mat, alpha, beta, "local")
        assert torch.equal(one.ravel(), got[k])


@pytest.mark.parametrize("nq,long_targets", [(1, 3), (8, 40), (30, 5)])
def test_long_targets_beside_many_short_ones(nq, long_targets):
    # the longest targets run as strips beside the search kernel: every pair once,
    # invalid and empty targets as before
    rng = np.random.default_rng(nq)
    mat = synth.blosum62()
    qs = [rng.integers(0, 20, size=int(n)).astype(np.uint8) for n in rng.integers(1, 700, size=nq)]
    lens = np.concatenate([rng.integers(0, 150, size=900), rng.integers(1000, 2600, size=long_targets)])
    ts = [rng.integers(0, 20, size=int(n)).astype(np.uint8) for n in rng.permutation(lens)]
    longest = int(np.argmax([len(t) for t in ts]))
    ts[longest][200:200 + len(qs[0])] = qs[0]
    qc, qo = synth.pack_csr(qs)
    tc, to = synth.pack_csr(ts)
    want, _ = oracle.cross(qc, qo, tc, to, mat, 11, 1, "local", nthreads=NTHREADS)
    want = np.asarray(want).reshape(nq, len(ts)).copy()
    for bad in (False, True):
        if bad:
            tc[to[longest] + 5] = 40
            want[:, longest] = np.iinfo(np.int32).min
        dev = [torch.from_numpy(a).cuda() for a in (qc, qo, tc, to)]
        got, st = ga.align_cross(*dev, mat, 11, 1, "local", stats=True)
        assert np.array_equal(got.cpu().numpy(), want)
        assert st["pairs_int16"] == nq * (len(ts) - bad) and (st["status"] != 0) == bad


@pytest.mark.parametrize("mode", ["global", "semiglobal"])
def test_more_pairs_than_one_plan_holds(mode):
    # protein searches in the whole-sequence modes are planned 2^20 pairs at a time
    rng = np.random.default_rng(6)
    mat = synth.blosum62()
    qs = [rng.integers(0, 20, size=int(n)).astype(np.uint8) for n in rng.integers(0, 8, size=1100)]
    ts = [rng.integers(0, 20, size=int(n)).astype(np.uint8) for n in rng.integers(0, 8, size=1000)]
    qc, qo = synth.pack_csr(qs)
    tc, to = synth.pack_csr(ts)
    dev = [torch.from_numpy(a).cuda() for a in (qc, qo, tc, to)]
    want, _ = oracle.cross(qc, qo, tc, to, mat, 11, 1, mode, nthreads=NTHREADS)
    got = ga.align_cross(*dev, mat, 11, 1, mode)
    assert np.array_equal(got.cpu().numpy().ravel(), np.asarray(want).ravel())
