"""GPU: the counts of a small batch in one launch are those of the planned path: cells
and pairs without a sequence that has an invalid code."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402


@pytest.mark.parametrize("mode", ["local", "global", "semiglobal"])
def test_invalid_pairs_are_not_counted(mode):
    rng = np.random.default_rng(71)
    n = 60
    qc, qo = synth.random_sequences(rng, rng.integers(1, 300, n), 4)
    tc, to = synth.random_sequences(rng, rng.integers(1, 300, n), 4)
    bad = [3, 17, 58]
    qc[qo[3]] = 4
    tc[to[18] - 1] = 9
    qc[qo[59] - 1] = 200
    good = np.array([k not in bad for k in range(n)])
    cells = int((np.diff(qo) * np.diff(to))[good].sum())
    sc = (synth.dna_matrix(2, -3), 5, 2)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]
    scores, one = ga.align_batch(*d, *sc, mode, stats=True)
    assert (scores.cpu().numpy()[bad] == -2 ** 31).all() and one["status"] == 5
    assert (one["cells"], one["pairs_int16"], one["pairs_int32"]) == (cells, n - len(bad), 0)
    with ga.Plan(*sc, mode, n, max(len(qc), len(tc)), 300) as plan:
        for tuning in (None, ga.Tuning((1 << 17) - 1, (1 << 17) - 1, 1, 0)):
            if tuning is not None:
                plan.tuning = tuning
            plan.run(*d)
            st = plan.stats()
            assert (st["cells"], st["pairs_int16"], st["pairs_int32"]) == (cells, n - len(bad), 0), tuning
