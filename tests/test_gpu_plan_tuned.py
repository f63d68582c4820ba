"""GPU: tunings of plans of small capacity, which run one launch without bins as long
as they have none.  A tuning that is set is run as it stands, and the autotuner drops
the tiles that hold no pair of the sample."""
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
ALL = (1 << len(ga.TILE_K)) - 1


def _reads(n, length, seed):
    rng = np.random.default_rng(seed)
    qc, qo = synth.random_sequences(rng, np.full(n, length), 4)
    tc, to = synth.random_sequences(rng, np.full(n, length), 4)
    return (qc, qo, tc, to), [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]


@pytest.mark.parametrize("conc", [0, 1])
def test_a_tuning_that_is_set_is_run(conc):
    # bounds beyond int16: the bins take these pairs in int32, the one-launch kernel in
    # relative int16 cells
    sc = (synth.dna_matrix(8, -127), 120, 100)
    host, d = _reads(50, 400, 61)
    want, _ = oracle.batch(*host, *sc, "global", nthreads=NTHREADS)
    with ga.Plan(*sc, "global", 50, len(host[0]), 400) as plan:
        np.testing.assert_array_equal(plan.run(*d).cpu().numpy(), want)
        st = plan.stats()
        assert (st["pairs_int16"], st["pairs_int32"]) == (50, 0)
        plan.tuning = ga.Tuning(ALL, ALL, conc, 0)
        np.testing.assert_array_equal(plan.run(*d).cpu().numpy(), want)
        st = plan.stats()
        assert (st["pairs_int16"], st["pairs_int32"]) == (0, 50)


@pytest.mark.parametrize("given", [True, False])
@pytest.mark.parametrize("mode", ["global", "local"])
def test_autotuner_drops_unused_tiles(mode, given):
    sc = (synth.dna_matrix(2, -3), 5, 2)
    host, d = _reads(4000, 150, 62)
    want, _ = oracle.batch(*host, *sc, mode, nthreads=NTHREADS)
    with ga.Plan(*sc, mode, 4000, len(host[0]), 200) as plan:
        if given:
            plan.tuning = ga.Tuning(ALL, ALL, 0, 0)
        tuning, ms = plan.autotune(*d, reps=5)
        # 150 columns: tile 10 (160 columns); the widest one stays
        assert tuning["tiles16"] == [10, 32] and tuning["tiles32"] == []
        assert plan.tuning.as_dict() == tuning and ms > 0
        np.testing.assert_array_equal(plan.run(*d).cpu().numpy(), want)
        plan.tuning = plan.tuning
        np.testing.assert_array_equal(plan.run(*d).cpu().numpy(), want)
