"""The image is the same bit for bit with and without the per-pixel intermediates
(kernels of their own) for every draw and grid, integer and real counts; and a
frame in host memory equals glint_shade's bit for bit with the surrogate and real
counts where the whole frame and its bands take different fused kernels."""
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("draw,grid", [(0, 0), (0, 1), (1, 0), (2, 0), (3, 0)])
@pytest.mark.parametrize("real", [False, True])
def test_intermediates_do_not_change_a_bit(gl, K, draw, grid, real):  # noqa: F811
    glint, render, ctx, torch = gl
    n = 20037
    fr = render.Frame(ctx, synth.env_hdr(seed=6, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=64)))
    fr.update_env()
    planes = render.gbuffer_tensors(synth.gbuffer_random(n, seed=K, width=n))
    kw = dict(seed=5, count_mode=glint.COUNT_REAL if real else glint.COUNT_INTEGER, draw=draw, grid=grid,
              gamma=0.01 if draw == 3 else 0.0)
    want = fr.shade(planes, n, 1, debug=glint.debug_buffers(n, K, samples=12 if grid else 6), **kw)
    got = fr.shade(planes, n, 1, **kw)
    torch.cuda.synchronize()
    assert torch.equal(got, want)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("staged", [False, True])
def test_bands_of_a_large_surrogate_frame(gl, real, staged):  # noqa: F811
    glint, render, ctx, torch = gl
    K, w, h = 8, 733, 701  # above four rounds of 768 pixels an SM; the bands of 50 rows are below
    n = w * h
    fr = render.Frame(ctx, synth.env_hdr(seed=6, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=128)))
    fr.update_env()
    gb = synth.gbuffer_random(n, seed=5, width=w)
    host = render.gbuffer_tensors(gb, device="cpu", pinned=True)
    tan = torch.from_numpy(gb.tangents()).pin_memory()
    net = glint.Mlp(ctx, K, 256)
    net.set_params(synth.mlp_params(seed=10, K=K))
    kw = dict(seed=4, count_mode=glint.COUNT_REAL if real else glint.COUNT_INTEGER, evaluator=glint.EVAL_MLP, mlp=net)
    ref = fr.shade([p.cuda() for p in host], w, h, tangent=tan.cuda(), **kw)
    out = torch.zeros(n, 4).pin_memory()
    pipe = glint.HostPipe(ctx, band_pixels=w * 50, slots=2)
    pipe.shade(fr.env, host, w, h, out, tangent=tan, p_scratch=torch.empty(n, K, device="cuda"), rows_per_band=50,
               staged=staged, **kw)
    torch.cuda.synchronize()
    assert torch.equal(out, ref.cpu())
    pipe.close()
