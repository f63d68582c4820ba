"""GPU parity of semi-global scores where the last column's free end parts it from
the column beside it by more than int16: H(., C) keeps the largest value of its
column while the cells to its left fall by the gap extension a row.  Every kernel of
relative cells, the last column at every place of a lane (first, inner and last of
its K columns, either half, lane 0), and rows past several renormalisations."""
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

NTHREADS = max(1, min(32, os.cpu_count() or 1))
STEEP = (synth.dna_matrix(8, -127), 120, 100)


def _free_end_pair(rows, cols, hit):
    """The query's residue `hit` matches the target's last one and nothing else
    matches: 8 at (hit + 1, cols), falling columns everywhere else."""
    q = np.zeros(rows, np.uint8)
    q[hit] = 2
    t = np.ones(cols, np.uint8)
    t[-1] = 2
    return q, t


def _both_ways(pairs):
    return [p for q, t in pairs for p in ((q, t), (t, q))]


def _batch(pairs):
    qc, qo = synth.pack_csr([p[0] for p in pairs])
    tc, to = synth.pack_csr([p[1] for p in pairs])
    return qc, qo, tc, to


def _dev(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def _check(got, want, pairs, what):
    got = np.asarray(got, dtype=np.int64)
    bad = np.nonzero(got != want)[0]
    assert len(bad) == 0, (what, len(bad), [(len(pairs[b][0]), len(pairs[b][1]), int(got[b]), int(want[b])) for b in bad[:5]])


def _oracle(batch, sc):
    return oracle.batch(*batch, *sc, "semiglobal", nthreads=NTHREADS)[0]


def test_one_launch_batches():
    pairs = [_free_end_pair(400, 421, 0)]
    rng = np.random.default_rng(21)
    for cols in (*range(129, 137), 160, 256, *range(257, 274), 384, 385, 420, 511, 512, 513, 524, 525, 640, 641, 767, 768):
        for rows in (cols, cols - 1, max(1, cols - 40)):
            pairs.append(_free_end_pair(rows, cols, int(rng.integers(0, min(rows, 60)))))
    pairs = _both_ways(pairs)
    b = _batch(pairs)
    want, d = _oracle(b, STEEP), _dev(*b)
    assert want[0] == 8
    _check(ga.align_batch(*d, *STEEP, "semiglobal").cpu().numpy(), want, pairs, "batch")
    _check(ga.align_batch_modes(*d, *STEEP, ["local", "semiglobal"]).cpu().numpy()[1], want, pairs, "modes")
    with ga.Plan(*STEEP, "semiglobal", len(pairs), max(len(b[0]), len(b[2])), 768) as plan:
        _check(plan.run(*d).cpu().numpy(), want, pairs, "plan")


# (scoring, longest): the columns part by beta x rows
@pytest.mark.parametrize("sc,rows", [(STEEP, 1500), ((synth.dna_matrix(2, -3), 12, 10), 4200),
                                     ((synth.dna_matrix(2, -9), 5, 4), 9000)])
def test_long_pairs(sc, rows):
    rng = np.random.default_rng(22)
    pairs = []
    for cols in (rows, rows + 1, rows + 7, rows + 40, rows + 255, rows + 256, rows + 257, rows + 513):
        pairs.append(_free_end_pair(rows, cols, int(rng.integers(0, 200))))
    # related sequences that end in the last column early, then unrelated rows
    for n in (500, 700):
        t = rng.integers(0, 4, rows + n).astype(np.uint8)
        pairs.append((np.concatenate([t[-n:], rng.integers(0, 4, rows - n).astype(np.uint8)]), t))
    pairs = _both_ways(pairs)
    b = _batch(pairs)
    want, d = _oracle(b, sc), _dev(*b)
    _check(ga.align_batch(*d, *sc, "semiglobal").cpu().numpy(), want, pairs, "strips")
    with ga.Plan(*sc, "semiglobal", len(pairs), max(len(b[0]), len(b[2])), rows + 700) as plan:
        _check(plan.run(*d).cpu().numpy(), want, pairs, "one warp a pair")
    one = [int(ga.align_long(*_dev(q, t), *sc, "semiglobal").item()) for q, t in pairs[:6]]
    _check(one, want[:6], pairs[:6], "single pairs")
    with ga.Server(arena_bytes=1 << 28, idle_us=200) as srv:
        sid = srv.add_scoring(*sc)
        srv.submit(*b, 2, sid)
        srv.drain(30_000)
        got = np.sort(srv.poll(), order="id")
    assert (got["status"] == 0).all()
    _check(got["score"], want, pairs, "server")


def test_profile_strips():
    rng = np.random.default_rng(23)
    mat = np.full((5, 5), -9, np.int8)
    np.fill_diagonal(mat, 8)
    sc = (mat, 12, 10)
    pairs = []
    for rows, cols in ((3400, 3401), (3400, 3585), (3500, 3841), (4000, 4100), (5000, 5121)):
        pairs.append(_free_end_pair(rows, cols, int(rng.integers(0, 90))))
    pairs = _both_ways(pairs)
    b = _batch(pairs)
    want, d = _oracle(b, sc), _dev(*b)
    _check(ga.align_batch(*d, *sc, "semiglobal").cpu().numpy(), want, pairs, "batch")
    k = len(pairs)
    cross = ga.align_cross(*d, *sc, "semiglobal").cpu().numpy().reshape(k, k)
    _check(np.diagonal(cross), want, pairs, "cross")
