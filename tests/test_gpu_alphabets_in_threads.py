"""GPU: calls from several host threads with alphabets of different size.  The kernels
with a scoring profile need shared memory by the alphabet; the limit set for one
thread's call must not fail the launch of another's."""
import threading

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402


def _run(kind, A, reps, errors, start):
    try:
        rng = np.random.default_rng(A)
        mat = rng.integers(-4, 8, (A, A)).astype(np.int8)
        n = 2600 if kind == "batch" else 8  # (a batch that fills the chip runs 512-column strips)
        qc, qo = synth.random_sequences(rng, np.full(n, 450 if kind == "search" else 300), A)
        tc, to = synth.random_sequences(rng, np.full(n, 280), A)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (qc, qo, tc, to)]
            s.synchronize()
            plan = ga.Plan(mat, 11, 1, "global", 8, 4000, 512) if kind == "plan" else None
            mode = "local" if kind == "search" else "global"
            fn = {"batch": lambda: ga.align_batch(*d, mat, 11, 1, mode, stream=s),
                  "search": lambda: ga.align_cross(*d, mat, 11, 1, mode, stream=s),
                  "plan": lambda: plan.run(*d, stream=s)}[kind]
            start.wait(60)
            for _ in range(reps):
                got = fn()
            s.synchronize()
            got = got.cpu().numpy()
        if kind == "search":
            want, _ = oracle.cross(qc, qo, tc, to, mat, 11, 1, mode, nthreads=4)
        else:
            want, _ = oracle.batch(qc, qo, tc, to, mat, 11, 1, mode, nthreads=4)
        np.testing.assert_array_equal(got.ravel(), np.asarray(want).ravel())
        if plan:
            plan.close()
    except BaseException as e:  # noqa: BLE001 - reported by the test
        errors.append((A, repr(e)[:300]))


@pytest.mark.parametrize("kind", ["batch", "search", "plan"])
def test_two_alphabets_at_once(kind):
    errors, start = [], threading.Barrier(4)
    # 24..31 symbols: every profile beyond the default limit of 48 KB
    threads = [threading.Thread(target=_run, args=(kind, A, 400 if kind == "batch" else 1500, errors, start)) for A in (24, 31, 27, 30)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
