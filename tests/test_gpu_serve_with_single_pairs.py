"""GPU: a server keeps working when other calls of the process use its kernel."""
import time

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402


def test_server_after_a_single_pair_of_a_smaller_alphabet():
    """A single pair on int32 strips (sigma_max + alpha > 128) launches the
    server's kernel with a 4-symbol profile; the server's next launch still gets
    the shared memory of its 24-symbol one."""
    rng = np.random.default_rng(3)
    q = rng.integers(0, 20, 1500).astype(np.uint8)
    t = rng.integers(0, 20, 1400).astype(np.uint8)
    prot = (synth.blosum62(), 11, 1)
    want = oracle.score(q, t, *prot, "local")
    a = rng.integers(0, 4, 900).astype(np.uint8)
    dna = (synth.dna_matrix(2, -3), 140, 2)
    with ga.Server(arena_bytes=1 << 26, idle_us=200) as srv:
        sid = srv.add_scoring(*prot)
        for _ in range(2):
            srv.submit(q, [0, len(q)], t, [0, len(t)], 0, sid)
            srv.drain(30_000)
            assert int(srv.poll()["score"][0]) == want
            time.sleep(0.05)  # past idle_us: the next request launches the kernel again
            x = torch.from_numpy(a).cuda()
            got = ga.align_long(x, x, *dna, "global")
            assert int(got.item()) == oracle.score(a, a, *dna, "global")
