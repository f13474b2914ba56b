"""GPU friends-of-friends (Sec. 3.2) against the oracle's brute-force groups.

Both sides use the same fixed-point positions and the exact integer linking rule, so the
groups, their labels (smallest member index), sizes and the mass function must agree exactly.
"""
import numpy as np
import pytest
import torch

from oracle import fof as ofof
from oracle import mesh as omesh
from paper_1301_0322_gb300 import inputs

pytestmark = pytest.mark.gpu

THRESHOLDS = [25, 50, 100, 200, 400, 800, 1600]


@pytest.fixture(scope="module")
def cola():
    from paper_1301_0322_gb300 import build
    build.build(verbose=False)
    import paper_1301_0322_gb300 as c
    c.load_library()
    return c


def check(cola, plan, s32, n_p, ng, box, b=(1, 5), nmin=25):
    group, size, n_ge = plan.fof(torch.from_numpy(s32).cuda(), nmin=nmin, b=b, thresholds=THRESHOLDS)
    plan.status()
    g, sz, ng_ = (t.cpu().numpy() for t in (group, size, n_ge))
    f = omesh.fixed_point_coords(s32, n_p, ng, box, 16)
    rg, rs = ofof.fof_groups(f, ng << 16, (ng // n_p) << 16, nmin, *b)
    assert np.array_equal(g, rg)
    assert np.array_equal(sz, rs)
    assert np.array_equal(ng_, ofof.mass_function(rg, rs, THRESHOLDS))
    return int(np.unique(rg[rg >= 0]).size)


@pytest.mark.parametrize("n_p,ng,box,seed", [(32, 64, 50.0, 3), (32, 96, 40.0, 4)])
def test_fof_of_clustered_particles(cola, n_p, ng, box, seed):
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    s32 = inputs.clustered_displacements(n_p, box, seed)
    nhalo = check(cola, plan, s32, n_p, ng, box)
    assert nhalo >= 4


def test_fof_of_an_evolved_cola_box_and_other_linking_length(cola):
    n_p, ng, box = 32, 64, 25.0
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    s, v, s1, s2 = plan.run(plan.noise(5))
    s32 = s.cpu().numpy()
    nhalo = check(cola, plan, s32, n_p, ng, box)
    print("halos at z = 0 (32^3 particles, L = 25 Mpc/h):", nhalo)
    check(cola, plan, s32, n_p, ng, box, b=(1, 4), nmin=10)


def test_union_retry_limit_reports_timeout_and_recovers(cola):
    # The union-find is a bounded loop: when its retries run out, cola_fof latches COLA_ETIMEOUT
    # (read by cola_status) instead of spinning.  With 0 tries every union gives up at once; with
    # 1 try on a dense clump the run either reports the timeout or has exact groups; afterwards
    # the default limit gives exact groups on the same plan (the context stays usable).
    n_p, ng, box = 32, 64, 50.0
    plan = cola.Plan(np_side=n_p, ng=ng, box=box)
    s32 = inputs.clustered_displacements(n_p, box, 3, nclump=2, frac=0.8, radius=0.3)
    s_dev = torch.from_numpy(s32).cuda()
    cola.cola_set_fof_union_tries(plan.handle, 0)
    plan.fof(s_dev, nmin=25, b=(1, 5), thresholds=THRESHOLDS)
    with pytest.raises(cola.ColaError) as e:
        plan.status()
    assert e.value.code == 6 and "union-find" in str(e.value)
    cola.cola_set_fof_union_tries(plan.handle, 1)
    group, size, n_ge = plan.fof(s_dev, nmin=25, b=(1, 5), thresholds=THRESHOLDS)
    try:
        plan.status()
        exact = True
    except cola.ColaError as err:
        assert err.code == 6
        exact = False
    if exact:
        f = omesh.fixed_point_coords(s32, n_p, ng, box, 16)
        rg, _ = ofof.fof_groups(f, ng << 16, (ng // n_p) << 16, 25, 1, 5)
        assert np.array_equal(group.cpu().numpy(), rg)
    with pytest.raises(cola.ColaError):
        cola.cola_set_fof_union_tries(plan.handle, -1)
    cola.cola_set_fof_union_tries(plan.handle, 1 << 20)
    assert check(cola, plan, s32, n_p, ng, box) >= 1


@pytest.mark.parametrize("n_p,ng", [(32, 64), (32, 96), (32, 32)])
def test_fof_stays_inside_its_workspace(cola, n_p, ng):
    # linking cells of one mesh cell need the most scratch: nothing behind the workspace may change
    from paper_1301_0322_gb300 import cola as binding
    cfg = binding._make_config(n_p, ng, 50.0)
    h = binding.cola_plan_create(cfg)
    nbytes = binding.cola_workspace_bytes(h)
    buf = torch.full((nbytes + (1 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
    assert buf.data_ptr() % 256 == 0
    binding.cola_set_workspace(h, buf[:nbytes])
    s = torch.from_numpy(inputs.clustered_displacements(n_p, 50.0, 3)).cuda()
    group = torch.empty(n_p**3, dtype=torch.int32, device="cuda")
    size = torch.empty_like(group)
    binding.cola_fof(h, s, 1, 5, 25, group, size, None, None)
    binding.cola_status(h)
    assert bool((buf[nbytes:] == 0x5A).all())
    binding.cola_plan_destroy(h)


@pytest.mark.parametrize("n_p,ng,b,kind", [(32, 32, (1, 5), "clumps"), (32, 64, (1, 1), "random"), (32, 192, (1, 5), "clumps"),
                                           (48, 96, (1, 6), "clumps"), (32, 96, (3, 5), "random"), (32, 64, (1, 5), "one cell")])
def test_fof_linking_cells(cola, n_p, ng, b, kind):
    # cells of one and of several mesh cells, groups across the faces of the box, and every particle
    # in a few cells (more candidates than a particle has lanes)
    box = 40.0
    if kind == "clumps":
        s32 = inputs.clustered_displacements(n_p, box, 7)
    elif kind == "random":
        s32 = inputs.gaussian_displacements(n_p, box, 8)
    else:
        p = np.arange(n_p**3)
        q = np.stack([p % n_p, (p // n_p) % n_p, p // (n_p * n_p)]) * (box / n_p)
        away = np.random.default_rng(9).normal(0, 0.15 * box / n_p, size=q.shape)
        pull = p % 29 == 0  # a clump around the corner of the box, the others stay near the lattice
        s32 = np.where(pull, np.where(q > box / 2, box - q, -q) + away, 0.1 * away).astype(np.float32)
    check(cola, cola.Plan(np_side=n_p, ng=ng, box=box), s32, n_p, ng, box, b=b, nmin=5)
