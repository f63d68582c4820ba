"""GPU: a banded call that runs every pair on the band kernel takes no workspace for
exact scores.  In a process of its own, because the library's pool keeps what it once
mapped."""
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
n, length = 20_000, 3000
rng = np.random.default_rng(41)
base = rng.integers(0, 4, (n, length)).astype(np.uint8)
other = base.copy()
hit = rng.random(other.shape) < 0.02
other[hit] = rng.integers(0, 4, int(hit.sum()))
off = np.arange(n + 1, dtype=np.int64) * length
dev = [torch.from_numpy(a).cuda() for a in (base.reshape(-1), off, other.reshape(-1), off.copy())]
scores = torch.empty(n, dtype=torch.int32, device="cuda")
mat = synth.dna_matrix(2, -3)
ga.align_batch(*[d[:2] if k % 2 else d[:length] for k, d in enumerate(dev)], mat, 5, 2, "global")
torch.cuda.synchronize()
used = torch.empty_like(scores)
before = torch.cuda.mem_get_info()[0]
got = ga.align_banded(*dev, mat, 5, 2, default_w0=64, scores=scores, w_used=used)[0]
torch.cuda.synchronize()
took = before - torch.cuda.mem_get_info()[0]
got = got.cpu().numpy()
pick = rng.choice(n, 40, replace=False)
for k in pick:
    assert int(got[k]) == oracle.score(base[k], other[k], mat, 5, 2, "global"), k
# packed sequences 30 MB, edges of the resident warps 90 MB, lists; the edges of 20,000
# full matrices are 480 MB
print("took", took >> 20)
assert took < 320 << 20, took >> 20
"""


def test_no_workspace_for_exact_scores():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
