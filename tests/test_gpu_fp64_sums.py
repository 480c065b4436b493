"""The FP64 kernels' integer neighbour sums (stencil64.cu) at the sizes and
values where they can go wrong: edges of the 64-wide row tiles and of the row
blocks, exponents far apart, zeros, the ends of the range (which take the
FP64 instructions), infinities and NaN.  Reference: the operators evaluated
in numpy's extended precision.

Bounds.  A heat7 step in FP64 rounds at most eight times and the integer form
less often, each time by at most eps = 2^-53 of a partial sum; a partial sum
is at most A = |c| + |r| (sum |neighbours| + 6 |c|).  A wave25 step rounds at
most 26 times, of partial sums below B = kappa sum |c_m| |p_m| + 2|p| +
|p_prev|; the double coefficients differ from the rationals by at most eps
each.  So 8 eps A and 27 eps B bound the errors, plus the smallest subnormal
for results at the bottom of the range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
C = [-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0]
SHAPES = [(4, 4, 4), (12, 12, 64), (8, 20, 68), (20, 8, 132), (36, 4, 60)]
KINDS = ["normal", "wide", "steep", "steps", "sparse", "tiny", "huge"]


@pytest.fixture(scope="module")
def ooc():
    import paper_2109_05410_gb300 as m
    m.build()
    m.lib()
    return m


def field(kind, shape, seed):
    g = np.random.default_rng(seed)
    v = g.standard_normal(shape)
    if kind == "wide":  # neighbours up to 2^120 apart
        v = np.ldexp(v, g.integers(-60, 60, size=shape))
    elif kind == "steep":  # a factor of 8 to 64 per cell, along a diagonal
        z, y, x = np.indices(shape)
        v = np.ldexp(v, 3 * z + 6 * y - 4 * x)
    elif kind == "steps":  # exact powers of two and equal values: sums that cancel
        v = np.ldexp(g.choice([-1.0, 1.0], size=shape), g.integers(0, 3, size=shape))
    elif kind == "sparse":  # zeros of both signs around isolated values
        v = np.where(g.random(shape) < 0.01, v, g.choice([0.0, -0.0], size=shape))
    elif kind == "tiny":  # across the exponent below which FP64 instructions take over, and subnormals
        v = np.ldexp(v, g.integers(-1074, -860, size=shape))
    elif kind == "huge":
        v = np.ldexp(v, g.integers(860, 1010, size=shape))
    return v


def neighbours(u, m):
    """The six arrays of values m cells away (zero outside), u's dtype."""
    out = []
    for ax in range(3):
        for s in (m, -m):
            w = np.zeros_like(u)
            n = u.shape[ax]
            if m < n:
                d, f = [slice(None)] * 3, [slice(None)] * 3
                d[ax], f[ax] = (slice(m, n), slice(0, n - m)) if s > 0 else (slice(0, n - m), slice(m, n))
                w[tuple(d)] = u[tuple(f)]
            out.append(w)
    return out


def heat_ref(u, r):
    q = u.astype(np.longdouble)
    nb = neighbours(q, 1)
    ref = q + np.longdouble(r) * (sum(nb) - 6 * q)
    mag = np.abs(q) + abs(r) * (sum(np.abs(v) for v in nb) + 6 * np.abs(q))
    return ref, mag


def wave_ref(p, pm, kap):
    q = p.astype(np.longdouble)
    lap, mag = 3 * np.longdouble(C[0]) * q, abs(3 * C[0]) * np.abs(q)
    for m in range(1, 5):
        nb = neighbours(q, m)
        lap = lap + np.longdouble(C[m]) * sum(nb)
        mag = mag + abs(C[m]) * sum(np.abs(v) for v in nb)
    kq = kap.astype(np.longdouble)
    return kq * lap + 2 * q - pm, kq * mag + 2 * np.abs(q) + np.abs(pm).astype(np.longdouble)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", KINDS)
def test_heat7_f64_step_within_rounding(ooc, shape, kind):
    u = field(kind, shape, 3)
    for r in (1.0 / 6.0, -0.05):
        d = torch.from_numpy(u.copy()).cuda()
        ooc.ooc_heat7_steps_f64(d, torch.empty_like(d), 1, r=r)
        got = d.cpu().numpy()
        ref, mag = heat_ref(u, r)
        assert np.all(np.abs(got - ref) <= 8 * EPS * mag + 2.0 ** -1074)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", KINDS)
def test_wave25_f64_step_within_rounding(ooc, shape, kind):
    p, pm = field(kind, shape, 4), 0.9 * field(kind, shape, 4)
    kap = np.random.default_rng(5).uniform(0.01, 0.15, size=shape)
    dp, dpm = torch.from_numpy(p.copy()).cuda(), torch.from_numpy(pm.copy()).cuda()
    ooc.ooc_wave25_steps_f64(dp, dpm, torch.from_numpy(kap).cuda(), 1)
    ref, mag = wave_ref(p, pm, kap)
    assert np.all(np.abs(dp.cpu().numpy() - ref) <= 27 * EPS * mag + 2.0 ** -1074)
    assert np.array_equal(dpm.cpu().numpy(), p)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinities_and_nan_spread_as_in_fp64(ooc, bad):
    shape = (12, 12, 68)
    u = field("normal", shape, 6)
    u[5, 6, 31] = bad
    u[2, 3, 64] = bad
    d = torch.from_numpy(u.copy()).cuda()
    ooc.ooc_heat7_steps_f64(d, torch.empty_like(d), 1)
    got = d.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref, mag = heat_ref(u, 1.0 / 6.0)
        same = np.isfinite(ref)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(got[np.isinf(got)], ref[np.isinf(ref)])
        assert np.all(np.abs(got - ref)[same] <= 8 * EPS * mag[same])
    kap = np.full(shape, 0.1)
    dp, dpm = torch.from_numpy(u.copy()).cuda(), torch.zeros(shape, dtype=torch.float64, device="cuda")
    ooc.ooc_wave25_steps_f64(dp, dpm, torch.from_numpy(kap).cuda(), 1)
    got = dp.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref, mag = wave_ref(u, np.zeros(shape), kap)
        same = np.isfinite(ref)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(got[np.isinf(got)], ref[np.isinf(ref)])
        assert np.all(np.abs(got - ref)[same] <= 27 * EPS * mag[same])


@pytest.mark.parametrize("kind", ["normal", "smooth", "wide", "steep"])
def test_error_no_larger_than_the_fp64_sequence(ooc, kind):
    # the same step as a sequence of FP64 operations (fused multiply-adds
    # formed in extended precision), both against extended precision
    shape = (32, 40, 128)
    if kind == "smooth":
        from synth import smooth_random_field
        p = smooth_random_field(shape, 8.0, seed=8, dtype=np.float64)
    else:
        p = field(kind, shape, 7)
    pm, kap = 0.95 * p, np.random.default_rng(9).uniform(0.01, 0.15, size=shape)

    def fma(a, b, c):
        return (np.longdouble(a) * b + c).astype(np.float64)

    d = torch.from_numpy(p.copy()).cuda()
    ooc.ooc_heat7_steps_f64(d, torch.empty_like(d), 1)
    ref, mag = heat_ref(p, 1.0 / 6.0)
    n = neighbours(p, 1)
    seq = fma(1.0 / 6.0, fma(-6.0, p, ((n[4] + n[5]) + (n[2] + n[3])) + (n[0] + n[1])), p)
    err = [float(np.sqrt(np.mean(((v - ref) / mag) ** 2))) for v in (d.cpu().numpy(), seq)]
    assert err[0] <= err[1], err

    dp = torch.from_numpy(p.copy()).cuda()
    ooc.ooc_wave25_steps_f64(dp, torch.from_numpy(pm.copy()).cuda(), torch.from_numpy(kap).cuda(), 1)
    ref, mag = wave_ref(p, pm, kap)
    lap = (3.0 * C[0]) * p
    for m in range(1, 5):
        n = neighbours(p, m)
        lap = fma(C[m], ((n[4] + n[5]) + (n[2] + n[3])) + (n[0] + n[1]), lap)
    seq = fma(kap, lap, fma(2.0, p, -pm))
    err = [float(np.sqrt(np.mean(((v - ref) / mag) ** 2))) for v in (dp.cpu().numpy(), seq)]
    assert err[0] <= err[1], err
