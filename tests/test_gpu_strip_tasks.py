"""GPU parity of the strip tasks (long pairs and alphabets of more than 4
symbols) against the CPU oracle, bit for bit, at the edges of a strip: widths
around multiples of 256 columns (64 K for K = 4 .. 20), rows around the batches
of 32, the 63 rows of a strip's drain and the renormalisation every 128, both
orientations, and batches of the sizes at which each strip width is chosen."""
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
DNA = (synth.dna_matrix(2, -3), 5, 2)
PROTEIN = (synth.blosum62(), 11, 1)


def _related(rng, n, m, A):
    """Two sequences of n and m residues that share most of the shorter one."""
    a = rng.integers(0, A, size=n).astype(np.uint8)
    b = np.concatenate([a, rng.integers(0, A, size=max(0, m - n)).astype(np.uint8)])[:m].copy()
    hit = rng.random(m) < 0.1
    b[hit] = rng.integers(0, A, size=int(hit.sum()))
    if m > 40:
        b = np.concatenate([b[:m // 3], b[m // 3 + 5:], b[:5]])
    return a, b


def _check(pairs, scoring, mode):
    qc, qo = synth.pack_csr([p[0] for p in pairs])
    tc, to = synth.pack_csr([p[1] for p in pairs])
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]
    got, st = ga.align_batch(*d, *scoring, mode, stats=True)
    want, errs = oracle.batch(qc, qo, tc, to, *scoring, mode, nthreads=NTHREADS)
    assert not errs.any() and st["status"] == 0
    got = got.cpu().numpy().astype(np.int64)
    bad = np.nonzero(got != want)[0]
    assert len(bad) == 0, (mode, len(bad), [(len(pairs[b][0]), len(pairs[b][1]), int(got[b]), int(want[b])) for b in bad[:5]])


@pytest.mark.parametrize("mode", MODES)
def test_protein_edges(mode):
    rng = np.random.default_rng(7)
    lens = [1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 128, 129, 160, 255, 256, 257, 511, 512, 513, 769, 1025]
    pairs = [_related(rng, a, b, 24) for a in lens for b in lens]
    _check(pairs, PROTEIN, mode)


@pytest.mark.parametrize("mode", MODES)
def test_dna_long_edges(mode):
    rng = np.random.default_rng(8)
    lens = [513, 640, 767, 768, 769, 1023, 1024, 1025, 1280, 1281, 1536, 2049]
    pairs = [_related(rng, a, b, 4) for a in lens for b in lens]
    _check(pairs, DNA, mode)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("npairs,length", [(2, 6000), (30, 6000), (60, 6000), (90, 6000), (110, 6000), (700, 1400)])
def test_dna_batches_of_every_width(mode, npairs, length):
    rng = np.random.default_rng(npairs)
    pairs = [_related(rng, int(rng.integers(length // 2, length)), int(rng.integers(length - 300, length)), 4)
             for _ in range(npairs)]
    _check(pairs, DNA, mode)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("npairs,length", [(3, 3000), (200, 1600), (2600, 260)])
def test_protein_batches_of_every_width(mode, npairs, length):
    rng = np.random.default_rng(npairs)
    pairs = [_related(rng, int(rng.integers(length // 2, length)), int(rng.integers(length // 2, length)), 20)
             for _ in range(npairs)]
    _check(pairs, PROTEIN, mode)


@pytest.mark.parametrize("mode", MODES)
def test_single_pairs_and_scorings(mode):
    rng = np.random.default_rng(9)
    asym = rng.integers(-6, 7, size=(4, 4)).astype(np.int8)
    five = rng.integers(-9, 10, size=(5, 5)).astype(np.int8)
    # linear gaps, the largest packed step (sigma_max + alpha = 128), small and odd alphabets
    scorings = [DNA, PROTEIN, (asym, 4, 4), (synth.dna_matrix(3, -127), 125, 1), (synth.dna_matrix(1, -1), 127, 127),
                (five, 10, 3), (np.full((1, 1), 2, np.int8), 3, 1)]
    for k, sc in enumerate(scorings):
        for m, n in ((700, 5000), (5000, 701), (1, 3000), (3000, 1), (4097, 4097)):
            a, b = _related(rng, m, n, sc[0].shape[0])
            got = ga.align_long(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), *sc, mode)
            assert int(got.item()) == oracle.score(a, b, *sc, mode), (k, m, n)


@pytest.mark.parametrize("mode", MODES)
def test_bases_that_move_far_at_the_last_rows(mode):
    """Steep scorings (sigma_max + alpha = 128) on identical sequences: a base
    moves by thousands per 128 rows, also while lane 0 is past the last row (its
    left input is -inf there).  Batches and the server run strip tasks, plans the
    one-warp kernel."""
    rng = np.random.default_rng(11)
    mat, alpha, beta = synth.dna_matrix(100, -100), 28, 1
    seqs = [rng.integers(0, 4, n).astype(np.uint8) for n in range(960, 1100, 5)]
    # a row sequence that ends where its alignment has just entered a strip
    longer = [np.concatenate([s, rng.integers(0, 4, 150).astype(np.uint8)]) for s in seqs]
    _check([(s, s.copy()) for s in seqs] + list(zip(seqs, longer)), (mat, alpha, beta), mode)
    qc, qo = synth.pack_csr(seqs)
    tc, to = synth.pack_csr(longer)
    want, _ = oracle.batch(qc, qo, tc, to, mat, alpha, beta, mode, nthreads=NTHREADS)
    with ga.Server(arena_bytes=1 << 26, idle_us=200) as srv:
        sid = srv.add_scoring(mat, alpha, beta)
        srv.submit(qc, qo, tc, to, MODES.index(mode), sid)
        srv.drain(30_000)
        got = np.sort(srv.poll(), order="id")
    assert (got["score"] == want).all() and (got["status"] == 0).all()
    qc, qo = synth.pack_csr(seqs)
    d = [torch.from_numpy(a).cuda() for a in (qc, qo, qc.copy(), qo.copy())]
    with ga.Plan(mat, alpha, beta, mode, len(seqs), len(qc), 1100) as plan:
        got = plan.run(*d).cpu().numpy()
    assert (got == [100 * len(s) for s in seqs]).all()
