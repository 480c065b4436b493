"""The FP64 stencils over many steps: errors that would add up from step to
step, and the sign symmetry of FP64 arithmetic, f(-u) = -f(u).

Reference: the steps in numpy's extended precision (113 bits on this
platform) and the same steps as a sequence of FP64 operations, with the fused
multiply-adds formed in extended precision.

Bounds.  A CPU emulation of the kernels' integers over 12 random fields each
(12 x 16 x 72) gives, as the ratio of the rms error to the FP64 sequence's:
heat7 at r = 1/6, point release and half-empty checkerboard, 200 steps, 1.00
(2.04 and 1.85 with shifts that cut off towards minus infinity); smooth, 32
steps, 0.81, at most 0.87 (about 3 if 6 c comes off before the sum is
rounded); wave25, 100 steps, rough 0.76, smooth 0.66, point release 0.76, at
most 0.93 (2.09, 0.87 and 2.00 with rational weights).  The bounds lie
between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (12, 16, 72)
C = [-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0]
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
    z, y, x = np.indices(shape)
    if kind == "wide":
        v = np.ldexp(v, g.integers(-60, 60, size=shape))
    elif kind == "steep":
        v = np.ldexp(v, 3 * z + 6 * y - 4 * x)
    elif kind == "steps":
        v = np.ldexp(g.choice([-1.0, 1.0], size=shape), g.integers(0, 3, size=shape))
    elif kind == "sparse":
        v = np.where(g.random(shape) < 0.01, v, g.choice([0.0, -0.0], size=shape))
    elif kind == "tiny":
        v = np.ldexp(v, g.integers(-1074, -860, size=shape))
    elif kind == "huge":
        v = np.ldexp(v, g.integers(860, 1010, size=shape))
    elif kind == "point":
        v = np.zeros(shape)
        v[tuple(g.integers(0, n) for n in shape)] = g.uniform(1.0, 2.0)
    elif kind == "checker":
        v = np.where((x + y + z) % 2 == 0, g.uniform(1.0, 1.3, size=shape), 0.0)
    elif kind == "smooth":
        from synth import smooth_random_field
        v = smooth_random_field(shape, 8.0, seed=seed, dtype=np.float64)
    return v


def shifted(u, ax, s):
    w = np.zeros_like(u)
    n = u.shape[ax]
    d, f = [slice(None)] * 3, [slice(None)] * 3
    d[ax], f[ax] = (slice(s, n), slice(0, n - s)) if s > 0 else (slice(0, n + s), slice(-s, n))
    if abs(s) < n:
        w[tuple(d)] = u[tuple(f)]
    return w


def six(u, m):
    """((x- + x+) + (y- + y+)) + (z- + z+), zero outside, in u's type."""
    x, y, z = (shifted(u, ax, m) + shifted(u, ax, -m) for ax in (2, 1, 0))
    return (x + y) + z


def fma(a, b, c):
    return (np.longdouble(a) * b + c).astype(np.float64)


def heat_gpu(ooc, u, n, r=1.0 / 6.0):
    d = torch.from_numpy(u.copy()).cuda()
    ooc.ooc_heat7_steps_f64(d, torch.empty_like(d), n, r=r)
    return d.cpu().numpy()


@pytest.mark.parametrize("kind,steps,bound", [("point", 200, 1.25), ("checker", 200, 1.25), ("smooth", 32, 1.0)])
def test_heat7_error_does_not_add_up(ooc, kind, steps, bound):
    r, err = 1.0 / 6.0, np.zeros(2)
    for seed in range(4):
        u = field(kind, SHAPE, 20 + seed)
        got = heat_gpu(ooc, u, steps)
        q, s = u.astype(np.longdouble), u.copy()
        for _ in range(steps):
            q = q + np.longdouble(r) * (six(q, 1) - 6 * q)
            s = fma(r, fma(-6.0, s, six(s, 1)), s)
        norm = np.sqrt(np.mean(q * q))
        err += [float(np.mean(((v - q) / norm) ** 2)) for v in (got, s)]
    assert np.sqrt(err[0]) <= bound * np.sqrt(err[1]), np.sqrt(err / 4)


@pytest.mark.parametrize("kind", KINDS + ["point", "checker", "smooth"])
def test_heat7_is_odd(ooc, kind):
    u = field(kind, SHAPE, 30)
    for r in (1.0 / 6.0, 0.11):
        assert np.array_equal(heat_gpu(ooc, -u, 5, r), -heat_gpu(ooc, u, 5, r))


@pytest.mark.parametrize("kind", ["normal", "steps", "wide", "sparse"])
def test_heat7_keeps_a_node_plane(ooc, kind):
    # odd about plane 5 and zero far from it: the grid's ends are too far
    # away to be felt there
    u = np.zeros(SHAPE)
    u[6:8] = field(kind, SHAPE, 31)[6:8]
    u[3:5] = -u[7:5:-1]
    got = heat_gpu(ooc, u, 6)
    assert not np.any(got[5])
    assert np.array_equal(got[4], -got[6]) and np.any(got[4])


def wave_gpu(ooc, p, pm, kap, n):
    dp, dpm = torch.from_numpy(p.copy()).cuda(), torch.from_numpy(pm.copy()).cuda()
    ooc.ooc_wave25_steps_f64(dp, dpm, torch.from_numpy(kap).cuda(), n)
    return dp.cpu().numpy()


def layers(shape):
    z = np.indices(shape)[0]
    return 0.07 * (1.0 + 0.02 * z / shape[0])


@pytest.mark.parametrize("kind", ["normal", "smooth", "point"])
def test_wave25_error_does_not_add_up(ooc, kind):
    steps, err, kap = 100, np.zeros(2), layers(SHAPE)
    for seed in range(2):
        p = field(kind, SHAPE, 40 + seed)
        got = wave_gpu(ooc, p, 0.95 * p, kap, steps)
        q, qm, s, sm = p.astype(np.longdouble), (0.95 * p).astype(np.longdouble), p, 0.95 * p
        for _ in range(steps):
            lap = np.longdouble(3.0 * C[0]) * q
            seq = (3.0 * C[0]) * s
            for m in range(1, 5):
                lap = lap + np.longdouble(C[m]) * six(q, m)
                seq = fma(C[m], six(s, m), seq)
            q, qm = kap * lap + 2 * q - qm, q
            s, sm = fma(kap, seq, fma(2.0, s, -sm)), s
        norm = np.sqrt(np.mean(q * q))
        err += [float(np.mean(((v - q) / norm) ** 2)) for v in (got, s)]
    assert err[0] <= err[1], np.sqrt(err / 2)


@pytest.mark.parametrize("kind", KINDS + ["point", "checker", "smooth"])
def test_wave25_is_odd(ooc, kind):
    p, pm, kap = field(kind, SHAPE, 50), 0.9 * field(kind, SHAPE, 50), layers(SHAPE)
    assert np.array_equal(wave_gpu(ooc, -p, -pm, kap, 4), -wave_gpu(ooc, p, pm, kap, 4))


@pytest.mark.parametrize("kind", ["normal", "steps", "wide", "sparse"])
def test_wave25_keeps_a_node_plane(ooc, kind):
    shape = (36, 16, 72)
    u = np.zeros(shape)
    u[18:20] = field(kind, shape, 51)[18:20]
    u[15:17] = -u[19:17:-1]
    got = wave_gpu(ooc, u, 0.9 * u, np.full(shape, 0.1), 6)
    assert not np.any(got[17])
    assert np.array_equal(got[16], -got[18]) and np.any(got[16])
