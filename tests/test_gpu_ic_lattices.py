"""2LPT displacements at the lattices whose inverse passes transform two columns per thread (256 up;
persistent from 384), element by element against a float64 evaluation on the GPU of the same filter,
gradients and second-order source.  Tolerances: those of the check against the oracle on small lattices
(2e-5 of max |s1|, 2e-4 of max |s2|)."""
import numpy as np
import pytest
import torch

from oracle.cosmology import Cosmology
from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu


def lpt64(noise, n, box):
    """s1 and s2 at a = 1, [3][n^3] float64 (first derivatives zero on their Nyquist plane)."""
    cosmo = Cosmology(**inputs.COSMOLOGY)
    kf = 2 * np.pi / box
    full = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    half = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    m2 = full[:, None, None] ** 2 + full[None, :, None] ** 2 + half[None, None, :] ** 2
    # P(k) depends on the whole number |n|^2 alone: one host evaluation per value
    values, where = torch.unique(m2.to(torch.int64), return_inverse=True)
    k = kf * np.sqrt(values.cpu().numpy().astype(np.float64))
    k[0] = 1.0
    amp = np.sqrt(cosmo.pk_linear(k) * n**3 / box**3)
    amp[0] = 0.0
    inv_k2 = 1.0 / (kf * kf * m2.clamp_min(1.0))
    d = torch.fft.rfftn(noise.double().view(n, n, n)) * torch.from_numpy(amp).cuda()[where] * inv_k2
    del where, m2
    gfull, ghalf = kf * full, kf * half
    gfull[n // 2] = 0.0
    ghalf[n // 2] = 0.0
    grad = [ghalf[None, None, :], gfull[None, :, None], gfull[:, None, None]]

    def back(f):
        return torch.fft.irfftn(f, s=(n, n, n)).reshape(-1)

    s1 = torch.stack([back(1j * g * d) for g in grad])
    xx, yy, zz = (back(-g * g * d) for g in grad)
    mu = xx * yy + xx * zz + yy * zz
    del xx, yy, zz
    for i, j in ((0, 1), (0, 2), (1, 2)):
        mu -= back(-grad[i] * grad[j] * d) ** 2
    m = torch.fft.rfftn(mu.view(n, n, n)) * inv_k2
    m[0, 0, 0] = 0.0
    return s1, cosmo.growth([1.0])["d2u1"] * torch.stack([back(-1j * g * m) for g in grad])


@pytest.mark.parametrize("n", [128, 256, 384, 512])
def test_ic_2lpt_of_large_lattices(n):
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as cola
    box = 0.4 * n
    plan = cola.Plan(np_side=n, ng=n, box=box)
    noise = plan.noise(n)
    s, v, s1, s2 = plan.ic_2lpt(noise)
    plan.status()
    del plan
    r1, r2 = lpt64(noise, n, box)
    assert float((s1.double() - r1).abs().max()) <= 2e-5 * float(r1.abs().max())
    assert float((s2.double() - r2).abs().max()) <= 2e-4 * float(r2.abs().max())
    assert bool((v == 0).all())
    del r1, r2, s, v, s1, s2
    torch.cuda.empty_cache()
