"""The fused deposit's tiles on meshes small enough that its blocks deposit with more threads than
they transform with: P(k) through it equals P(k) of the integer deposit bit for bit (the same
correctly rounded overdensities and transforms), for spread and for clumped particles (tiles of
a few and of thousands of particles, cell sums beyond 32 bits)."""
import pytest
import torch

from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_p,ng", [(32, 32), (48, 48), (32, 64), (32, 96), (64, 128), (96, 192), (64, 256), (96, 384)])
@pytest.mark.parametrize("clumps", [False, True])
def test_fused_deposit_equals_the_integer_deposit(n_p, ng, clumps):
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as cola
    box = 0.5 * ng
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    s32 = inputs.clustered_displacements(n_p, box, 3) if clumps else inputs.gaussian_displacements(n_p, 3.0, 4)
    s = torch.from_numpy(s32).cuda()
    rho, delta = plan.density(s)
    assert int(rho.sum()) % 2**64 == (n_p**3 << 48) % 2**64  # (the sum of the cells wraps at 2^63)
    want, got = plan.power(delta, ng // 2), plan.density_power(s, ng // 2)
    plan.status()
    for a, b in zip(want, got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n_p,ng,bits", [(48, 64, 16), (48, 128, 12), (64, 96, 16), (96, 256, 16), (96, 256, 20), (48, 64, 8)])
def test_positions_on_a_mesh_that_is_no_multiple_of_the_lattice(n_p, ng, bits):
    # the 32-bit lattice offset floor(i ng 2^F / np) against the oracle's, small and box-crossing
    # displacements (96 on 256: the last size whose bins one block scans)
    import numpy as np

    import paper_1301_0322_gb300 as cola
    from oracle import mesh as omesh
    box = 0.5 * ng
    plan = cola.Plan(np_side=n_p, ng=ng, box=box, fixed_bits=bits)
    for sigma in (0.3, 40.0):
        s = inputs.gaussian_displacements(n_p, sigma, 5)
        rho, _ = plan.density(torch.from_numpy(s).cuda(), delta=False)
        got = rho.cpu().numpy().reshape(ng, ng, ng)
        assert np.array_equal(got, omesh.cic_deposit_fixed(s, n_p, ng, box, bits))
