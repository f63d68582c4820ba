"""GPU: a burst whose long requests come last, which are queued before the others."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402


def test_long_requests_submitted_last():
    rng = np.random.default_rng(8)
    scoring = (synth.dna_matrix(2, -3), 5, 2)
    lens = np.concatenate([rng.integers(1, 900, size=400), [32767, 32768, 33001]])
    qs = [rng.integers(0, 4, int(n)).astype(np.uint8) for n in lens]
    ts = [np.delete(q, rng.integers(0, len(q), size=len(q) // 50)) if len(q) > 50 else q for q in qs]
    ts[-2] = ts[-2][:100]
    qc, qo = synth.pack_csr(qs)
    tc, to = synth.pack_csr(ts)
    dev = [torch.from_numpy(a).cuda() for a in (qc, qo, tc, to)]
    modes = (np.arange(len(qs)) % 2).astype(np.int32)  # local, global
    want = np.stack([ga.align_batch(*dev, *scoring, m).cpu().numpy() for m in ("local", "global")])
    with ga.Server(arena_bytes=1 << 28) as srv:
        sid = srv.add_scoring(*scoring)
        first = srv.submit(qc, qo, tc, to, modes, sid)
        srv.drain(60_000)
        got = srv.poll()
    assert len(got) == len(qs) and not got["status"].any()
    scores = np.empty(len(qs), np.int32)
    scores[got["id"] - first] = got["score"]
    assert np.array_equal(scores, want[modes, np.arange(len(qs))])
