"""GPU: band doubling decided by the exact score (ga_bandfull.cuh) gives the scores,
the accepted widths and the counts of the attempts that the doubling itself gives."""
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


def _dev(b):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.q_codes, b.q_off, b.t_codes, b.t_off)]


@pytest.mark.parametrize("matrix,alpha,beta", [(synth.dna_matrix(2, -3), 5, 2), (synth.dna_matrix(1, -1), 1, 1),
                                               (synth.dna_matrix(2, -1), 2, 2)])
@pytest.mark.parametrize("w0", [0, 1, 3])
def test_small_pairs_and_ties(matrix, alpha, beta, w0):
    # short related and unrelated pairs under small scores: the exact score often
    # equals the bound of some attempt, which is then run
    rng = np.random.default_rng(5 + w0)
    qs, ts = [], []
    for k in range(1500):
        a = rng.integers(0, 4, int(rng.integers(1, 90))).astype(np.uint8)
        b = np.delete(a, rng.integers(0, len(a), size=int(rng.integers(0, 6))))
        if k % 3 == 0:
            b = rng.integers(0, 4, int(rng.integers(1, 90))).astype(np.uint8)
        if len(b) == 0:
            b = a[:1]
        qs.append(a)
        ts.append(b)
    qc, qo = synth.pack_csr(qs)
    tc, to = synth.pack_csr(ts)
    b = synth.Batch(qc, qo, tc, to, matrix, alpha, beta, "ties")
    sc, wu, st = ga.align_banded(*_dev(b), matrix, alpha, beta, default_w0=w0, stats=True)
    sc, wu = sc.cpu().numpy(), wu.cpu().numpy()
    ties = 0
    for p in range(b.npairs):
        ref = oracle.banded_doubling_blocks(qs[p], ts[p], matrix, alpha, beta, w0, 16)
        assert (int(sc[p]), int(wu[p])) == (ref[0], ref[1]), (p, len(qs[p]), len(ts[p]), sc[p], wu[p], ref)
        m, n = len(qs[p]), len(ts[p])
        w = w0
        while w <= wu[p]:
            lo, hi = min(0, n - m) - w, max(0, n - m) + w
            ub = max([oracle.band_ub(m, n, int(matrix.max()), alpha, beta, d)
                      for d, inside in ((lo - 1, lo - 1 >= -m), (hi + 1, hi + 1 <= n)) if inside], default=None)
            ties += ub == sc[p]
            w = 2 * w if w else 1
    assert ties > 0 and st["status"] == 0


@pytest.mark.parametrize("w0", [64, 700])
def test_one_call_equals_calls_of_a_few_pairs(w0):
    # a few pairs take their full matrices, many the band kernel and, where they
    # fail, the strips: the same scores, widths and counts
    b = synth.long_dna_pairs(npairs=1300, lmin=900, lmax=9000, seed=61)
    d = _dev(b)
    sc, wu, st = ga.align_banded(*d, b.matrix, b.alpha, b.beta, default_w0=w0, stats=True)
    full = ga.align_batch(*d, b.matrix, b.alpha, b.beta, "global")
    assert torch.equal(sc, full) and st["status"] == 0
    cells = retries = 0
    for k in range(0, b.npairs, 20):
        sub = b.subset(range(k, min(k + 20, b.npairs)))
        s2, w2, t2 = ga.align_banded(*_dev(sub), b.matrix, b.alpha, b.beta, default_w0=w0, stats=True)
        assert torch.equal(s2, sc[k:k + 20]) and torch.equal(w2, wu[k:k + 20])
        cells += t2["banded_cells"]
        retries += t2["band_retries"]
    assert (cells, retries) == (st["banded_cells"], st["band_retries"])
    assert retries > 0


def test_widths_per_pair_and_unscored_pairs():
    b = synth.long_dna_pairs(npairs=40, lmin=300, lmax=5000, seed=62)
    rng = np.random.default_rng(4)
    w0 = rng.integers(-2, 900, size=b.npairs).astype(np.int32)
    codes = b.q_codes.copy()
    codes[b.q_off[7]] = 9  # an invalid residue
    d = _dev(b)
    d[0] = torch.from_numpy(codes).cuda()
    sc, wu = ga.align_banded(*d, b.matrix, b.alpha, b.beta, w0=torch.from_numpy(w0).cuda())
    sc, wu = sc.cpu().numpy(), wu.cpu().numpy()
    for p in range(b.npairs):
        if p == 7:
            assert sc[p] == -2 ** 31 and wu[p] == -1
            continue
        q, t = b.q_codes[b.q_off[p]:b.q_off[p + 1]], b.t_codes[b.t_off[p]:b.t_off[p + 1]]
        ref = oracle.banded_doubling_blocks(q, t, b.matrix, b.alpha, b.beta, max(0, int(w0[p])), 16)
        assert (int(sc[p]), int(wu[p])) == (ref[0], ref[1]), p
