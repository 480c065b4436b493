"""The encoders code whole warps of blocks together: warps in which some lanes
have no block, a block of zeros, no plane above the mode's lowest, or planes
that start and end elsewhere than the others'.  Bit for bit against the
oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ooc():
    import paper_2109_05410_gb300 as m
    m.build()
    m.lib()
    return m


def blocks(n, seed, zeros, dtype=np.float32, spread=40):
    """[4, 4, 4n]: rough and smooth blocks of differing size, a share of zeros."""
    g = np.random.default_rng(seed)
    scale = np.repeat(2.0 ** -g.integers(0, spread, n).astype(np.float64), 4)
    f = np.linspace(0.5, 1.5, 4 * n) * scale * np.where(np.repeat(g.random(n) < 0.5, 4), 1.0,
                                                        g.standard_normal((4, 4, 4 * n)))
    return (f * np.repeat(g.random(n) >= zeros, 4)).astype(dtype)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 131])
@pytest.mark.parametrize("zeros", [0.0, 0.5, 0.97, 1.0])
@pytest.mark.parametrize("rate", [1, 8, 16, 64])
def test_fixed_rate(ooc, n, zeros, rate):
    f = blocks(n, 3 * n, zeros)
    got = ooc.ooc_compress(torch.from_numpy(f).cuda(), rate)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), oracle.fr4_encode(f, rate))
    d = blocks(n, 3 * n + 1, zeros, np.float64)
    got = ooc.ooc_compress64(torch.from_numpy(d).cuda(), rate)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), oracle.fr4d_encode(d, rate))


@pytest.mark.parametrize("n", [1, 33, 131])
@pytest.mark.parametrize("zeros", [0.0, 0.5, 1.0])
@pytest.mark.parametrize("mode,param", [(1, 1), (1, 17), (1, 32), (2, 1e-9), (2, 1e-3), (2, 64.0)])
def test_variable(ooc, n, zeros, mode, param):
    f = blocks(n, 5 * n, zeros)
    words, index = oracle.fr4_encode_var(f, mode, param)
    got, got_index = ooc.ooc_compress_var(torch.from_numpy(f).cuda(), mode, param)
    assert np.array_equal(got_index.cpu().numpy().astype(np.uint64), index)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), words)
