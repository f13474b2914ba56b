"""The binning on meshes where the scatter takes its places from running cursors (finer than the
lattice, 512 and up): the integer density equals the oracle's cell by cell, for spread and for
clumped particles, and again in later calls on the same workspace (counts and cursors are left as
the next call needs them)."""
import numpy as np
import pytest
import torch

from oracle import mesh as omesh
from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_p", [32, 48])
def test_bins_with_cursors(n_p):
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as cola
    ng = 512
    box = 0.5 * ng
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    for s32 in (inputs.clustered_displacements(n_p, box, 3), inputs.gaussian_displacements(n_p, 40.0, 5),
                inputs.gaussian_displacements(n_p, 0.1, 6)):
        rho, _ = plan.density(torch.from_numpy(s32).cuda(), delta=False)
        plan.status()
        want = omesh.cic_deposit_fixed(s32, n_p, ng, box, 16).reshape(-1)
        assert torch.equal(rho, torch.from_numpy(np.ascontiguousarray(want)).cuda())


def test_both_forms_of_the_binning_bin_the_same_particles():
    # the same positions on a mesh on either side of the rule: particles per bin add up to the lattice,
    # and the density of the finer mesh summed over its cells is that of the lattice
    import paper_1301_0322_gb300 as cola
    n_p = 64
    for ng, bits in ((384, 16), (512, 16), (768, 12)):
        plan = cola.Plan(np_side=n_p, ng=ng, box=100.0, fixed_bits=bits)
        s = torch.from_numpy(inputs.clustered_displacements(n_p, 100.0, 4)).cuda()
        for _ in range(2):
            rho, _ = plan.density(s, delta=False)
            assert int(rho.sum()) % 2**64 == (n_p**3 << (3 * bits)) % 2**64
            k, pk, nm = plan.density_power(s, 32)
            assert bool(torch.isfinite(pk).all())
        plan.status()
        del plan, rho
        torch.cuda.empty_cache()


@pytest.mark.parametrize("bits", [8, 16, 19, 20])
@pytest.mark.parametrize("n_p,ng", [(32, 32), (32, 96), (48, 32), (48, 64), (96, 128), (192, 256), (384, 256), (192, 512),
                                    (384, 512)])
def test_lattice_offsets(n_p, ng, bits):
    # undisplaced particles: the density is the product of the axes' lines, which follow from
    # floor(i ng 2^F / np) alone
    import paper_1301_0322_gb300 as cola
    one = 1 << bits
    f = torch.tensor([i * ng * one // n_p for i in range(n_p)], device="cuda")
    cell, up = f // one, f % one
    line = torch.zeros(ng, dtype=torch.int64, device="cuda")
    line.index_add_(0, cell, one - up)
    line.index_add_(0, (cell + 1) % ng, up)
    plan = cola.Plan(np_side=n_p, ng=ng, box=100.0, fixed_bits=bits)
    rho, _ = plan.density(torch.zeros(3, n_p**3, device="cuda"), delta=False)
    want = line.view(ng, 1, 1) * line.view(1, ng, 1) * line.view(1, 1, ng)
    assert torch.equal(rho.view(ng, ng, ng), want)
