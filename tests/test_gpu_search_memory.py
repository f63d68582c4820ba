"""GPU: a search that runs in chunks of pairs holds the workspace of one chunk.  In a
process of its own, because the library's pool keeps what it once mapped."""
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
mode = "{mode}"
rng = np.random.default_rng(31)
# 2^20 pairs a chunk: 4 queries of two strips each (850 MB of edges), then 24
nt = 1 << 18
tc, to = synth.random_sequences(rng, np.full(nt, 100), 20)
qc, qo = synth.random_sequences(rng, np.full(24, 700), 20)
mat = synth.blosum62()
dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]
scores = torch.empty((24, nt), dtype=torch.int32, device="cuda")
def search(k):
    ga.align_cross(dev[0], dev[1][:k + 1].contiguous(), dev[2], dev[3], mat, 11, 1, mode, scores=scores[:k])
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
before = torch.cuda.mem_get_info()[0]
one, six = search(4), search(24)
print("chunks", before - one, one - six)
assert before - one > 700 << 20, "the edges of a chunk are what this test is about"
# six chunks plan with buffers of the same size; 256 MB of allowance for the pool's rounding
assert one - six < 256 << 20, (one - six) >> 20
cols = rng.choice(nt, 5, replace=False)
for k in (0, 3, 4, 11, 23):
    for c in cols:
        want = oracle.score(qc[qo[k]:qo[k + 1]], tc[to[c]:to[c + 1]], mat, 11, 1, mode)
        assert int(scores[k, c].item()) == want, (k, c)
"""


@pytest.mark.parametrize("mode", ["global", "semiglobal"])
def test_workspace_does_not_grow_with_the_chunks(mode):
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(mode=mode)], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
