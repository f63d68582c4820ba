"""GPU: batches around the limits of the one-launch kernel (by pairs, and by residues
beyond them) give the scores of the same pairs in small calls."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402


@pytest.mark.parametrize("npairs,lmin,lmax", [(8192, 60, 120), (8193, 60, 120), (8193, 280, 320), (16_384, 100, 180),
                                              (16_385, 20, 60)])
def test_around_the_limits(npairs, lmin, lmax):
    rng = np.random.default_rng(npairs)
    mat, alpha, beta = synth.dna_matrix(2, -3), 5, 2
    qs = [rng.integers(0, 4, int(n)).astype(np.uint8) for n in rng.integers(lmin, lmax + 1, size=npairs)]
    ts = [np.delete(q, rng.integers(0, len(q), size=len(q) // 20)) for q in qs]
    # an empty sequence, a pair beyond the kernel's 768 residues, an invalid code
    qs[17] = qs[17][:0]
    ts[npairs - 2] = rng.integers(0, 4, 900).astype(np.uint8)
    qc, qo = synth.pack_csr(qs)
    tc, to = synth.pack_csr(ts)
    qc[qo[40]] = 7
    d = [torch.from_numpy(a).cuda() for a in (qc, qo, tc, to)]
    for mode in ("local", "global", "semiglobal"):
        parts = [ga.align_batch(d[0], d[1][k:min(k + 4000, npairs) + 1].contiguous(), d[2],
                                d[3][k:min(k + 4000, npairs) + 1].contiguous(), mat, alpha, beta, mode)
                 for k in range(0, npairs, 4000)]
        got, st = ga.align_batch(*d, mat, alpha, beta, mode, stats=True)
        assert torch.equal(got, torch.cat(parts)) and int(got[40]) == -2 ** 31 and st["status"] != 0
    both = ga.align_batch_modes(*d, mat, alpha, beta, ["global", "semiglobal"])
    assert torch.equal(both[1], got)
