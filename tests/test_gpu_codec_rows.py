"""The any-shape codec kernels' two kinds of row access (16-byte rows when nx
is a multiple of 4 and the field 16-byte aligned, single values otherwise) and
the variable-size decoder's rounds (blocks that do not fit its staging buffer
together), bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from synth import random_blocks, smooth_random_field

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(4, 5, 8), (5, 4, 4), (7, 9, 132), (33, 6, 20)]


@pytest.fixture(scope="module")
def ooc():
    import paper_2109_05410_gb300 as m
    m.build()
    m.lib()
    return m


def on_gpu(a, shift):
    """The array on the GPU, `shift` values past a 16-byte boundary."""
    flat = torch.zeros(a.size + 4, dtype=torch.float32, device="cuda")
    v = flat[shift:shift + a.size].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return v


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("rate", [1, 13, 16, 64])
def test_fixed_rate_rows(ooc, shape, shift, rate):
    f = smooth_random_field(shape, 3.0, seed=5) * 2.0
    ref = oracle.fr4_encode(f, rate)
    assert np.array_equal(ooc.ooc_compress(on_gpu(f, shift), rate).cpu().numpy().view(np.uint32), ref)
    out = on_gpu(np.zeros_like(f), shift)
    ooc.ooc_decompress(torch.from_numpy(ref.view(np.uint8)).cuda(), shape, rate, d_out=out)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.fr4_decode(ref, shape, rate).view(np.uint32))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("mode,param", [(1, 1), (1, 20), (1, 32), (2, 1e-5)])
def test_variable_rows(ooc, shape, shift, mode, param):
    f = smooth_random_field(shape, 3.0, seed=6) * 2.0
    words, index = oracle.fr4_encode_var(f, mode, param)
    got, got_index = ooc.ooc_compress_var(on_gpu(f, shift), mode, param)
    assert np.array_equal(got_index.cpu().numpy().astype(np.uint64), index)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), words)
    out = on_gpu(np.zeros_like(f), shift)
    ooc.ooc_decompress_var(got, got_index, shape, mode, param, d_out=out)
    ref = oracle.fr4_decode_var(words, index, shape, mode, param)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("kind", ["normal", "bits", "sparse"])
def test_variable_decoder_rounds(ooc, kind):
    # 32 blocks of up to 68 words against a staging buffer of 38 words per
    # block: one to two rounds per warp, three partly filled warps
    f = random_blocks(kind, 70, seed=12)
    words, index = oracle.fr4_encode_var(f, 1, 32)
    got, got_index = ooc.ooc_compress_var(torch.from_numpy(f).cuda(), 1, 32)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), words)
    out = ooc.ooc_decompress_var(got, got_index, f.shape, 1, 32)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.fr4_decode_var(words, index, f.shape, 1, 32).view(np.uint32))
    # any offsets decode: blocks of 0 and of the clamped 130 words among others
    index2 = np.asarray(index).copy()
    index2[5:40:3] = index2[-1]
    index2[6:41:7] = 0
    out = ooc.ooc_decompress_var(got, torch.from_numpy(index2.astype(np.int64)).cuda(), f.shape, 1, 32)
    torch.cuda.synchronize()
    assert out.shape == f.shape


def test_block_exponents_of_special_values(ooc):
    # a block's header holds the exponent of its largest bit pattern without
    # the sign: zeros, subnormals, the largest values, infinities and NaN of
    # any payload
    specials = np.array([0x00000000, 0x80000000, 0x00000001, 0x80000001, 0x007fffff, 0x00800000, 0x3f800000,
                         0xff7fffff, 0x7f800000, 0xff800000, 0x7fc00000, 0xffc00001, 0x7f800001], dtype=np.uint32)
    rng = np.random.default_rng(8)
    blocks = np.zeros((2 * specials.size, 64), dtype=np.uint32)
    for i, v in enumerate(specials):  # alone, and among smaller ones
        blocks[2 * i, rng.integers(64)] = v
        m = (int(v) & 0x7fffffff) >> 23
        blocks[2 * i + 1] = rng.integers(0, max(m, 1) << 23, 64).astype(np.uint32) if m else 0
        blocks[2 * i + 1, rng.integers(64)] = v
    mx = (blocks & 0x7fffffff).max(axis=1)
    want = np.where(mx == 0, 0, 1 | (((mx >> 23) + 1 & 0xff) << 1))
    f = blocks.reshape(-1, 4, 4, 4).transpose(1, 2, 0, 3).reshape(4, 4, -1).view(np.float32)
    words = ooc.ooc_compress(torch.from_numpy(np.ascontiguousarray(f)).cuda(), 16).cpu().numpy().view(np.uint32)
    assert np.array_equal(words.reshape(-1, 32)[:, 0] & 0x1ff, want)


@pytest.mark.parametrize("rate", [1, 3, 9, 16, 40, 64])
def test_first_planes_of_mixed_warps(ooc, rate):
    # neighbouring blocks from constant to rough, so that the lanes of a warp
    # leave the encoder's one-field planes at different ones, or never do
    rng = np.random.default_rng(rate)
    f = np.broadcast_to(np.linspace(-1, 1.5, 4 * 67, dtype=np.float32), (8, 4, 4 * 67)).copy()
    rough = rng.standard_normal(f.shape).astype(np.float32) * np.repeat(np.float32(2.0) ** -rng.integers(0, 40, 67), 4)
    f += rough.astype(np.float32)
    f[:, :, 40:44] = 0.25
    f[4:, :, 96:100] = 0.0
    ref = oracle.fr4_encode(f, rate)
    assert np.array_equal(ooc.ooc_compress(on_gpu(f, 0), rate).cpu().numpy().view(np.uint32), ref)
