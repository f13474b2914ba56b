"""cola_density writes buffers that the caller owns, at any alignment of their elements: slices of
larger tensors receive what aligned ones do, and nothing around them changes."""
import pytest
import torch

from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_p,ng", [(32, 32), (48, 64), (64, 192)])
@pytest.mark.parametrize("rho_at,delta_at", [(1, None), (None, 1), (1, 1), (1, 0), (0, 1), (1, 2), (2, 3), (0, 2)])
def test_density_into_slices(n_p, ng, rho_at, delta_at):
    # (offsets in elements of a 256-byte aligned buffer; None: the output is not asked for)
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as cola
    from paper_1301_0322_gb300 import cola as binding
    box = 0.5 * ng
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    s = torch.from_numpy(inputs.clustered_displacements(n_p, box, 3)).cuda()
    want = [x.reshape(-1) for x in plan.density(s)]
    bufs, outs = [], []
    for at, dtype, guard in ((rho_at, torch.int64, -7), (delta_at, torch.float32, -7.0)):
        if at is None:
            bufs.append(None)
            outs.append(None)
            continue
        buf = torch.full((ng**3 + 8,), guard, dtype=dtype, device="cuda")
        assert buf.data_ptr() % 256 == 0
        bufs.append(buf)
        outs.append(buf[at:at + ng**3])
    binding.cola_density(plan.handle, s, *outs)
    plan.status()
    for at, buf, out, ref in zip((rho_at, delta_at), bufs, outs, want):
        if out is not None:
            assert torch.equal(out, ref)
            assert bool((buf[:at] == -7).all()) and bool((buf[at + ng**3:] == -7).all())
