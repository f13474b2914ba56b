"""Plans on two streams at a time: the column passes of both park in the tensor memory of the same
SMs (from 256 up), where a block waits until another's columns are free; the results are those of one
stream after the other."""
import pytest
import torch

from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("meshes", [(384, 384), (256, 512), (512, 768)])
def test_two_plans_on_two_streams(meshes):
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as cola
    n_p, evaluations = 64, 8
    plans = [cola.Plan(np_side=n_p, ng=ng, box=0.4 * ng) for ng in meshes]
    pos = [torch.from_numpy(inputs.gaussian_displacements(n_p, 1.0, 3 + i)).cuda() for i in range(2)]
    want = [p.force(s) for p, s in zip(plans, pos)]
    streams = [torch.cuda.Stream() for _ in plans]
    out = [[], []]
    for st in streams:
        st.wait_stream(torch.cuda.current_stream())
    for _ in range(evaluations):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                out[i].append(plans[i].force(pos[i]))
    torch.cuda.synchronize()
    for i in range(2):
        plans[i].status()
        for g in out[i]:
            assert torch.equal(g, want[i])
