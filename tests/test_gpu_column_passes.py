"""The column passes at the mesh sizes whose strips, groups and blocks differ from those of the
small parity meshes (one or two columns per thread, strips of 8 or 16 columns, one wave of
persistent blocks): the force of a plane wave along each axis against the oracle's exact
one-dimensional reduction (the tolerance of the full-size checks, 3e-4 of max |g|), and the
forward transform against float64 (float32 rounding of three passes of log2 N stages,
6e-8 sqrt(3 log2 N) < 1e-6 of the norm).
"""
import numpy as np
import pytest
import torch

from oracle import mesh as omesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cola():
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as c
    c.load_library()
    return c


@pytest.mark.parametrize("n_p,ng", [(96, 192), (128, 384), (128, 512), (256, 1024), (384, 1536)])
def test_plane_wave_force(cola, n_p, ng):
    free, _ = torch.cuda.mem_get_info()
    if free < 8 * 4 * ng**3:
        pytest.skip("not enough free device memory")
    box = 0.4 * ng
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    for axis, m in ((0, 1), (1, 3), (2, 5)):
        k = 2 * np.pi * m / box
        line = (0.4 / k * np.sin(k * np.arange(n_p) * box / n_p)).astype(np.float32)
        shape = [1, 1, 1]
        shape[2 - axis] = n_p  # [iz][iy][ix]
        s = torch.zeros((3, n_p, n_p, n_p), dtype=torch.float32, device="cuda")
        s[axis].copy_(torch.from_numpy(line).cuda().view(shape).expand(n_p, n_p, n_p))
        g = plan.force(s.view(3, -1)).view(3, n_p, n_p, n_p).double()
        plan.status()
        ref = omesh.unit_force_axis_wave(line.astype(np.float64), axis, n_p, ng, box, deconv=1)
        scale = np.abs(ref).max()
        want = torch.zeros_like(g)
        want[axis] += torch.from_numpy(ref).cuda().view(shape)
        assert float((g - want).abs().max()) <= 3e-4 * scale, (axis, float((g - want).abs().max()) / scale)
    del plan
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [384, 512, 768])
def test_forward_transform(cola, n):
    plan = cola.Plan(np_side=32, ng=n, box=100.0)
    x = torch.randn(n**3, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    got = plan.fft_r2c(x)
    want = torch.fft.rfftn(x.double().view(n, n, n))
    err = torch.linalg.vector_norm(torch.view_as_real(got.to(torch.complex128) - want))
    assert float(err) <= 1e-6 * float(torch.linalg.vector_norm(torch.view_as_real(want)))
    del plan, got, want
    torch.cuda.empty_cache()
