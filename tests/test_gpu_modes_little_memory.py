"""GPU: a call in several modes whose strip workspace fits for one mode only runs its
long pairs on the kernels that need less.  In a process of its own, because the
library's pool keeps what it once mapped."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import numpy as np, torch, oracle, synth
import paper_2205_07610_gb300 as ga
MODES = ["local", "global", "semiglobal"]
rng = np.random.default_rng(81)
n, length = 13_000, 10_000
codes = rng.integers(0, 4, (n, length)).astype(np.uint8)
other = codes.copy()
other[:, 1::9] = rng.integers(0, 4, other[:, 1::9].shape)
off = np.arange(n + 1, dtype=np.int64) * length
mat = synth.dna_matrix(2, -3)
dev = [torch.from_numpy(a).cuda() for a in (codes.reshape(-1), off, other.reshape(-1), off.copy())]
scores = torch.empty((3, n), dtype=torch.int32, device="cuda")
small = [d[:2] if k % 2 else d[:length] for k, d in enumerate(dev)]
ga.align_batch_modes(*small, mat, 5, 2, MODES)
torch.cuda.synchronize()
# a mode's strip edges take 1,040 MB, its edges at one warp a pair 200
free = torch.cuda.mem_get_info()[0]
full = torch.empty(free - (1170 << 20), dtype=torch.uint8, device="cuda")
got = ga.align_batch_modes(*dev, mat, 5, 2, MODES, scores=scores).cpu().numpy()
for k in (0, 1, 4999, n - 1):
    for m, mode in enumerate(MODES):
        assert int(got[m, k]) == oracle.score(codes[k], other[k], mat, 5, 2, mode), (k, mode)
"""


def test_modes_fall_back_together():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
