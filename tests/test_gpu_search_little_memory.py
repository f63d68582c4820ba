"""GPU: a search whose launches keep their stage edges side by side where they fit
runs them one after another over one buffer where only that fits.  In a process of its
own, because the library's pool keeps what it once mapped."""
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
rng = np.random.default_rng(51)
mat = synth.blosum62()
# queries of two stages in four tile widths; one target of 26,000 residues makes a
# launch's edges about 1 GB, all four 3.5 GB
qc, qo = synth.random_sequences(rng, np.repeat([640, 768, 896, 1024], 8), 20)
tc, to = synth.random_sequences(rng, np.concatenate([[26000], rng.integers(30, 90, 1300)]), 20)
dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]
scores = torch.empty((32, 1301), dtype=torch.int32, device="cuda")
ga.align_cross(dev[0], dev[1][:2].contiguous(), dev[2], (dev[3][:3] - 0).contiguous(), mat, 11, 1, "local")
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
full = torch.empty(free - (2300 << 20), dtype=torch.uint8, device="cuda")
got = ga.align_cross(*dev, mat, 11, 1, "local", scores=scores).cpu().numpy()
want, _ = oracle.cross(qc, qo, tc, to, mat, 11, 1, "local", nthreads=16)
assert (got == want).all(), int((got != want).sum())
"""


def test_search_falls_back_to_one_edge_buffer():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
