"""The checkpointed gradient over segments of every small length (odd and
even, one step, a shorter last one): the pairs of terms added inside the
adjoint steps and the one or two added at a segment's end."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ooc():
    import paper_2109_05410_gb300 as ooc
    return ooc


@pytest.mark.parametrize("every", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("shape", [(12, 16, 20), (36, 8, 132)])
def test_gradient_over_short_segments(ooc, shape, every):
    # FP32 steps, uncompressed checkpoints: two fields of 11 steps with some 12
    # roundings of 6e-8 each give 1.6e-5 if none cancel
    N = 11
    nz, ny, nx = shape
    rng = np.random.default_rng(17 + every)
    kap = rng.uniform(0.02, 0.12, shape).astype(np.float32)
    kap64 = kap.astype(np.float64)
    src = (nx // 2, ny // 2, nz // 2)
    src_flat = (src[2] * ny + src[1]) * nx + src[0]
    w = rng.standard_normal(N).astype(np.float32)
    rec = np.arange(0, ny * nx, 3, dtype=np.int64) + (nz // 2) * ny * nx
    res = rng.standard_normal((N, rec.size)).astype(np.float32)
    want = oracle.wave25_adjoint_grad(kap64, src_flat, w.astype(np.float64), N, rec, res.astype(np.float64))

    d_kap, d_rec = torch.from_numpy(kap).cuda(), torch.from_numpy(rec).cuda()
    traces = torch.empty((N, rec.size), device="cuda")
    h_ckpt = torch.empty(ooc.ooc_wave25_ckpt_bytes(shape, N, every, 0), dtype=torch.uint8, pin_memory=True)
    # what the work buffer held before has no effect (all ones: NaN)
    work = torch.full((ooc.ooc_wave25_adjoint_work_bytes(shape, every, 0),), 255, dtype=torch.uint8, device="cuda")
    streams = [torch.cuda.current_stream(), torch.cuda.Stream()]
    ooc.ooc_wave25_forward_ckpt(d_kap, N, d_rec, traces, every, 0, h_ckpt, work, streams, src=src, w=w)
    work.fill_(255)
    g = torch.empty(shape, dtype=torch.float64, device="cuda")
    ooc.ooc_wave25_backward_ckpt(d_kap, N, d_rec, torch.from_numpy(res).cuda(), every, 0, h_ckpt, g, work, streams,
                                 src=src, w=w)
    err = np.linalg.norm(g.cpu().numpy() - want) / np.linalg.norm(want)
    assert err < 2e-5, err
