"""GPU: an untuned plan beyond the one-launch capacity runs its bins as parallel
branches: the scores of ga_align_batch on any stream, replayed, and under capture."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2205_07610_gb300 as ga  # noqa: E402


@pytest.mark.parametrize("mode", ["local", "global", "semiglobal"])
@pytest.mark.parametrize("npairs,lmin,lmax", [(20_000, 20, 200), (3000, 100, 900)])
def test_untuned_plan_beyond_one_launch(mode, npairs, lmin, lmax):
    b = synth.mutated_dna_pairs(npairs=npairs, lmin=lmin, lmax=lmax, seed=9)
    d = [torch.from_numpy(a).cuda() for a in (b.q_codes, b.q_off, b.t_codes, b.t_off)]
    want = ga.align_batch(*d, b.matrix, b.alpha, b.beta, mode)
    cap = max(len(b.q_codes), len(b.t_codes))
    scores = torch.zeros(npairs, dtype=torch.int32, device="cuda")
    with ga.Plan(b.matrix, b.alpha, b.beta, mode, max(npairs, 17_000), cap, 2 * lmax) as plan:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        for _ in range(2):
            scores.zero_()
            side.wait_stream(torch.cuda.current_stream())
            plan.run(*d, scores, stream=side)
            # work enqueued behind the run on its stream sees every branch's scores
            with torch.cuda.stream(side):
                copy = scores.clone()
            side.synchronize()
            assert torch.equal(copy, want) and plan.stats()["status"] == 0
        scores.zero_()
        torch.cuda.synchronize()
        plan.capture(*d, scores)
        for _ in range(2):
            plan.launch()
            torch.cuda.synchronize()
            assert torch.equal(scores, want)
            scores.zero_()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            plan.run(*d, scores)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(scores, want)
