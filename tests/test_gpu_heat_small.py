"""heat7's choices of kernel: small windows without a march, pairs of steps on
128-column tiles (level s of the two columns beside a tile point by point),
and overlapped launches, also under stream capture.  All give the same bits."""
import numpy as np
import pytest

from synth import smooth_random_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ooc():
    import paper_2109_05410_gb300 as m
    m.build()
    m.lib()
    return m


def steps(ooc, u, n):
    v = u.clone()
    ooc.ooc_heat7_steps(v, torch.empty_like(v), n)
    return v


@pytest.mark.parametrize("ny,nx", [(512, 512), (484, 516)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_large_grid_equals_its_parts(ooc, ny, nx, n):
    # 48 planes: marched steps and pairs; parts of 24 planes: steps without a
    # march.  A part's planes further than n from its cut do not see it.
    u = torch.from_numpy(np.random.default_rng(3).standard_normal((48, ny, nx)).astype(np.float32)).cuda()
    whole = steps(ooc, u, n)
    for z0, z1, keep in ((0, 24, slice(0, 24 - n)), (24, 48, slice(24 + n, 48))):
        part = steps(ooc, u[z0:z1].contiguous(), n)
        assert torch.equal(whole[keep].view(torch.int32), part[keep.start - z0:keep.stop - z0].view(torch.int32))


@pytest.mark.parametrize("nx", [4, 124, 128, 132, 248, 256])
@pytest.mark.parametrize("T,k", [(8, 2), (12, 5), (64, 4)])
def test_pairs_in_plans_equal_single_steps(ooc, nx, T, k):
    # 128 and 256 columns take 128-column tiles; slabs pass level-s bands
    u0 = smooth_random_field((40, 20, nx), 5.0, seed=4)
    got = []
    for spl in (1, 2):
        plan = ooc.Plan(nx=nx, ny=20, nz=40, stencil="heat7", k=k, slab_planes=T, heat_steps_per_launch=spl)
        try:
            plan.set_field(0, u0)
            plan.step(2 * k + 1)
            got.append(plan.get_field(0))
        finally:
            plan.close()
    ref = steps(ooc, torch.from_numpy(u0).cuda(), 2 * k + 1).cpu().numpy()
    for g in got:
        assert np.array_equal(g.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("shape", [(4, 4, 4), (8, 12, 36), (64, 64, 64), (13 * 4, 40, 260)])
def test_overlapped_steps_between_other_work(ooc, shape):
    # the field changes right before and right after the steps, in the same
    # stream: nothing is read early, nothing late
    u = torch.from_numpy(smooth_random_field(shape, 3.0, seed=5)).cuda()
    a, tmp = u.clone(), torch.empty_like(u)
    for _ in range(20):
        a.mul_(1.5)
        ooc.ooc_heat7_steps(a, tmp, 7)
        a.add_(u)
    b = u.clone()
    for _ in range(20):
        b.mul_(1.5)
        for _ in range(7):
            torch.cuda.synchronize()
            ooc.ooc_heat7_steps(b, tmp, 1)
        torch.cuda.synchronize()
        b.add_(u)
    assert torch.equal(a.view(torch.int32), b.view(torch.int32))


def test_overlapped_steps_under_capture(ooc):
    u = torch.from_numpy(smooth_random_field((32, 40, 64), 4.0, seed=6)).cuda()
    ref = steps(ooc, steps(ooc, u, 6), 6)
    p, pm = u.clone(), 0.9 * u
    kap = torch.full_like(u, 0.05)
    rp, rpm = p.clone(), pm.clone()
    for _ in range(2):
        ooc.ooc_wave25_steps(rp, rpm, kap, 4)
    a, tmp = u.clone(), torch.empty_like(u)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        ooc.ooc_heat7_steps(a, tmp, 6, stream=s)
        ooc.ooc_wave25_steps(p, pm, kap, 4, stream=s)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(a.view(torch.int32), ref.view(torch.int32))
    assert torch.equal(p.view(torch.int32), rp.view(torch.int32))
    assert torch.equal(pm.view(torch.int32), rpm.view(torch.int32))
