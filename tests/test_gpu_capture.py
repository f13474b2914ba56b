"""Plan calls recorded in a CUDA graph and replayed: the same bits as direct calls.  On meshes up to
256 the launches are programmatic dependents, also behind nodes that are no kernels (copies, memsets);
at 384 passes are persistent and park in tensor memory."""
import pytest
import torch

from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_p,ng", [(32, 64), (48, 96), (64, 256), (64, 384)])
def test_captured_calls_replay_the_same_bits(n_p, ng):
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as cola
    box = 0.5 * ng
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    noise = plan.noise(7)
    s0, v0, s1, s2 = plan.ic_2lpt(noise)
    s_in, v_in, x_in = torch.empty_like(s0), torch.empty_like(v0), torch.empty_like(noise)
    s, v, x = torch.empty_like(s0), torch.empty_like(v0), torch.empty_like(noise)

    def calls():
        x.copy_(x_in)
        out = list(plan.ic_2lpt(x))
        s.copy_(s_in)
        v.zero_()
        v.add_(v_in)
        plan.step(3, s, v, s1, s2)
        rho, delta = plan.density(s)
        out += [s, v, rho, delta, *plan.power(delta, ng // 2), *plan.density_power(s, ng // 2), plan.force(s)]
        return out

    def inputs_of(seed):
        x_in.copy_(plan.noise(seed))
        s_in.copy_(torch.from_numpy(inputs.gaussian_displacements(n_p, 1.0, seed)))
        v_in.copy_(torch.from_numpy(inputs.gaussian_displacements(n_p, 0.5, seed + 1)))

    inputs_of(1)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        calls()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        recorded = calls()
    for seed in (1, 11):
        inputs_of(seed)
        graph.replay()
        got = [t.clone() for t in recorded]
        want = [t.clone() for t in calls()]
        plan.status()
        for i, (a, b) in enumerate(zip(got, want)):
            assert torch.equal(a, b), i
