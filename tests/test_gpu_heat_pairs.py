"""The fused heat7 pairs (two steps per launch, packed FP32) against single
steps, bit for bit.

The single steps are calls with nsteps = 1, which never pair; the pairs are
in-core calls above the size up to which the step loops run single steps only
(11 Mi points) with at least three steps, and plans with two steps per launch.
ooc_heat7_steps and ooc_heat7_steps_fused choose alike, so neither is the
other's reference."""
import numpy as np
import pytest

import oracle
from synth import sine_modes_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL = 11 << 20  # points of the largest grid that steps singly


@pytest.fixture(scope="module")
def ooc():
    import paper_2109_05410_gb300 as m
    m.build()
    m.lib()
    return m


def values(kind, shape):
    g = np.random.default_rng({"normal": 0, "subnormal": 1, "mixed": 2, "large": 3}[kind])
    u = g.standard_normal(shape, dtype=np.float32)
    if kind == "subnormal":  # with zeros of both signs
        u = (u * np.float32(1e-40)).astype(np.float32)
        u[g.random(shape) < 0.1] = 0.0
        u[g.random(shape) < 0.05] = -0.0
    elif kind == "mixed":  # over the whole exponent range
        u = np.ldexp(u, g.integers(-146, 124, size=shape, dtype=np.int32)).astype(np.float32)
    elif kind == "large":  # sums of six stay finite
        u = (g.uniform(-1.0, 1.0, shape) * 5e37).astype(np.float32)
    assert np.all(np.isfinite(u))
    return u


def singly(ooc, u, n):
    v, tmp = u.clone(), torch.empty_like(u)
    for _ in range(n):
        ooc.ooc_heat7_steps(v, tmp, 1)
    return v


def same(a, b):
    return torch.equal(a.view(torch.int32), b.view(torch.int32))


# Whole waves of whole tiles and z-chunks of the rest (1024 x 1024, 1000 x
# 1016), 128-column tiles (512 wide), ragged tiles (516, 1016 wide).
@pytest.mark.parametrize("shape", [(24, 1024, 1024), (20, 1000, 1016), (48, 512, 512), (12, 2048, 516)])
@pytest.mark.parametrize("kind", ["normal", "subnormal", "mixed", "large"])
def test_incore_pairs(ooc, shape, kind):
    assert np.prod(shape) > SMALL
    u = torch.from_numpy(values(kind, shape)).cuda()
    for n in (3, 4, 6):
        ref = singly(ooc, u, n)
        if kind == "subnormal":
            assert bool(((ref != 0) & (ref.abs() < torch.finfo(torch.float32).tiny)).any())  # they survive
        for call in (ooc.ooc_heat7_steps, ooc.ooc_heat7_steps_fused):
            v = u.clone()
            call(v, torch.empty_like(v), n)
            assert same(v, ref)


@pytest.mark.parametrize("shape", [(20, 36, 260), (24, 20, 128), (40, 68, 244)])
@pytest.mark.parametrize("kind", ["normal", "subnormal", "mixed", "large"])
def test_plan_pairs(ooc, shape, kind):
    nz, ny, nx = shape
    u = values(kind, shape)
    plan = ooc.Plan(nx=nx, ny=ny, nz=nz, stencil="heat7", k=4, slab_planes=8, heat_steps_per_launch=2)
    try:
        plan.set_field(0, u)
        plan.step(6)
        got = plan.get_field(0)
    finally:
        plan.close()
    ref = singly(ooc, torch.from_numpy(u).cuda(), 6).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("shape", [(2048, 4, 2048), (2048, 8, 1024), (4096, 1024, 4), (8192, 60, 32), (8192, 64, 32),
                                   (640, 512, 36)])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 6])
def test_few_rows_or_columns(ooc, shape, n):
    # 4 rows run single steps; many rows of at most 32 points an odd number
    # of launches and a copy
    assert np.prod(shape) > SMALL
    u = torch.from_numpy(values("normal", shape)).cuda()
    v = u.clone()
    ooc.ooc_heat7_steps(v, torch.empty_like(v), n)
    assert same(v, singly(ooc, u, n))


def test_incore_pairs_match_fp64(ooc):
    shape = (16, 768, 1024)
    assert np.prod(shape) > SMALL
    u0, _ = sine_modes_field(shape, seed=2)
    d = torch.from_numpy(u0).cuda()
    ooc.ooc_heat7_steps(d, torch.empty_like(d), 8)
    # the tolerance of the single steps' test: FP32 rounding of eight steps
    assert oracle.error_metrics(d.cpu().numpy(), oracle.heat7_run(u0.astype(np.float64), 8))["rel_l2"] < 1e-6


def test_incore_pairs_past_2_32(ooc):
    # a field of more than 2^32 points: pairs on chip-wide 64-bit offsets
    if torch.cuda.mem_get_info()[0] < 80e9:
        pytest.skip("needs 80 GB of free device memory")
    shape = (4104, 1024, 1024)
    u = torch.empty(shape, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(5)
    for z in range(0, shape[0], 513):
        u[z:z + 513].normal_(generator=g)
    ref = singly(ooc, u, 3)
    ooc.ooc_heat7_steps(u, torch.empty_like(u), 3)
    assert same(u, ref)
    del u, ref
    torch.cuda.empty_cache()
