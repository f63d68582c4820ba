"""GPU parity of the one-launch kernel of small batches (alphabets of <= 4
symbols) against the CPU oracle: the edges of its strips (256, 512, 768 columns),
batches that mix it with pairs too long for it, empty and invalid sequences, as
one call, several modes and a plan."""
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

MODES = ["local", "global", "semiglobal"]
NTHREADS = max(1, min(32, os.cpu_count() or 1))
INT32_MIN = -2 ** 31


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def _lengths(longest):
    edges = [0, 1, 2, 4, 31, 32, 33, 63, 64, 65, 128, 255, 256, 257, 300, 511, 512, 513, 767, 768, 769, 900, 1500]
    edges = [e for e in edges if e <= longest]
    return [(a, b) for a in edges for b in edges]


def _batch(longest, seed=1):
    rng = np.random.default_rng(seed)
    qs, ts = [], []
    for a, b in _lengths(longest):
        x = rng.integers(0, 4, max(a, b)).astype(np.uint8)
        y = np.where(rng.random(len(x)) < 0.1, rng.integers(0, 4, len(x)), x).astype(np.uint8)
        qs.append(x[:a])
        ts.append(y[len(y) - b:] if len(qs) % 3 == 0 else y[:b])
    return (*synth.pack_csr(qs), *synth.pack_csr(ts))


@pytest.mark.parametrize("scoring", [(synth.dna_matrix(2, -3), 5, 2), (synth.dna_matrix(100, -90), 28, 28),
                                     (np.full((1, 1), 3, np.int8), 2, 1)])
@pytest.mark.parametrize("longest", [768, 1500])
def test_edges(longest, scoring):
    qc, qo, tc, to = _batch(longest)
    if scoring[0].shape[0] == 1:
        qc, tc = qc * 0, tc * 0
    d = _dev(qc, qo, tc, to)
    want = [oracle.batch(qc, qo, tc, to, *scoring, md, nthreads=NTHREADS)[0] for md in MODES]
    cells = int(np.sum(np.diff(qo) * np.diff(to)))
    for md, w in zip(MODES, want):
        got, st = ga.align_batch(*d, *scoring, md, stats=True)
        np.testing.assert_array_equal(got.cpu().numpy(), w)
        assert st["status"] == 0 and st["cells"] == cells
        if longest <= 768:
            with ga.Plan(*scoring, md, len(qo) - 1, max(len(qc), len(tc)), longest) as plan:
                np.testing.assert_array_equal(plan.run(*d).cpu().numpy(), w)
                assert plan.stats()["cells"] == cells
    got = ga.align_batch_modes(*d, *scoring, MODES).cpu().numpy()
    np.testing.assert_array_equal(got, np.stack(want))


@pytest.mark.parametrize("longest", [768, 1500])
def test_invalid_sequences(longest):
    qc, qo, tc, to = _batch(longest, seed=2)
    lens = np.stack([np.diff(qo), np.diff(to)])
    scoring = (synth.dna_matrix(2, -3), 5, 2)
    want, _ = oracle.batch(qc, qo, tc, to, *scoring, "semiglobal", nthreads=NTHREADS)
    # a bad code in some queries (the last residue) and targets (the first), among
    # them pairs whose other sequence is empty
    bad_q = [p for p in range(5, lens.shape[1], 29) if lens[0, p]] + [int(np.nonzero((lens[1] == 0) & (lens[0] > 0))[0][2])]
    bad_t = [p for p in range(11, lens.shape[1], 31) if lens[1, p]] + [int(np.nonzero((lens[0] == 0) & (lens[1] > 0))[0][3])]
    qc, tc = qc.copy(), tc.copy()
    qc[qo[np.array(bad_q) + 1] - 1] = 4
    tc[to[np.array(bad_t)]] = 255
    d = _dev(qc, qo, tc, to)
    want = want.copy()
    want[bad_q + bad_t] = INT32_MIN
    got, st = ga.align_batch(*d, *scoring, "semiglobal", stats=True)
    np.testing.assert_array_equal(got.cpu().numpy(), want)
    assert st["status"] == 5
    if longest <= 768:
        with ga.Plan(*scoring, "semiglobal", len(qo) - 1, max(len(qc), len(tc)), longest) as plan:
            np.testing.assert_array_equal(plan.run(*d).cpu().numpy(), want)
            assert plan.stats()["status"] == 5


def test_decreasing_offsets_and_chunks_of_a_larger_buffer():
    qc, qo, tc, to = _batch(300, seed=3)
    scoring = (synth.dna_matrix(2, -3), 5, 2)
    n = len(qo) - 1
    want, _ = oracle.batch(qc, qo, tc, to, *scoring, "global", nthreads=NTHREADS)
    a = 40  # pairs a .. n - 1 of the buffers: the first offset is not 0
    got = ga.align_batch(*_dev(qc, qo[a:], tc, to[a:]), *scoring, "global").cpu().numpy()
    np.testing.assert_array_equal(got, want[a:])
    broken = qo.copy()
    k = int(np.nonzero(np.diff(qo) > 100)[0][3])
    broken[k + 1] = broken[k] - 1  # pair k ends before it starts
    got, st = ga.align_batch(*_dev(qc, broken, tc, to), *scoring, "global", stats=True)
    got = got.cpu().numpy()
    assert got[k] == INT32_MIN and st["status"] == 1
    keep = [p for p in range(n) if p not in (k, k + 1)]
    np.testing.assert_array_equal(got[keep], want[keep])
