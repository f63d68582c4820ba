"""GPU parity of long pairs in plans (one warp a pair, relative int16 cells) whose
alignment enters a super-stage (1,536 columns in local and global mode, 1,280 in
semi-global) within the last rows: the base of the first columns moves by tens of
thousands while their left input is already -inf."""
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


@pytest.mark.parametrize("mode", ["local", "global", "semiglobal"])
@pytest.mark.parametrize("sc", [(synth.dna_matrix(24, -24), 1, 1), (synth.dna_matrix(100, -100), 28, 1)])
def test_alignments_that_end_behind_a_stage_edge(sc, mode):
    rng = np.random.default_rng(91)
    width = 1280 if mode == "semiglobal" else 1536
    pairs = []
    for k in range(1, 150, 3):
        s = rng.integers(0, 4, width + 150).astype(np.uint8)
        rows = np.concatenate([rng.integers(0, 4, 200 + k).astype(np.uint8), s[:width + k]])
        pairs += [(rows, s), (s, rows)]
    qc, qo = synth.pack_csr([p[0] for p in pairs])
    tc, to = synth.pack_csr([p[1] for p in pairs])
    want, _ = oracle.batch(qc, qo, tc, to, *sc, mode, nthreads=NTHREADS)
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]
    with ga.Plan(*sc, mode, len(pairs), max(len(qc), len(tc)), width + 500) as plan:
        got = plan.run(*d).cpu().numpy()
    np.testing.assert_array_equal(got, want)
