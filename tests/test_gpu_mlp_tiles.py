"""The network's warp tiles and the fused kernel's two sizes: ragged row counts,
outputs at odd addresses, and frames large enough for the halves of a block to
take turns."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 4, 8])
def test_rows_do_not_depend_on_their_number_or_address(gl, K):  # noqa: F811
    glint, render, ctx, torch = gl
    n = 100003
    gen = torch.Generator(device="cuda").manual_seed(K)
    x = torch.zeros(n, 64, device="cuda")
    x[:, :6 * K + 3] = torch.rand(n, 6 * K + 3, device="cuda", generator=gen)
    x = x.to(torch.bfloat16).view(torch.int16)
    lp = torch.log_softmax(torch.randn(n, K, device="cuda", generator=gen) * 2, -1)
    net = glint.Mlp(ctx, K, 256)
    net.set_params(synth.mlp_params(seed=3, K=K))
    ref = net.forward(x, lp)
    assert torch.allclose(ref.sum(1), torch.ones(n, device="cuda"), atol=1e-5)
    for m in (1, 15, 16, 31, 32, 33, 127, 129, 4097):
        guard = torch.full((m * K + 9,), -7.0, device="cuda")
        moved = torch.empty(m * K + 1, device="cuda")
        moved[1:] = lp[:m].reshape(-1)
        out = guard[1:1 + m * K].view(m, K)  # 4-byte aligned only
        net.forward(x[:m].contiguous(), moved[1:].view(m, K), out=out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref[:m]), m
        assert guard[0] == -7.0 and torch.all(guard[1 + m * K:] == -7.0)


@pytest.mark.parametrize("K,width,height", [(8, 733, 701), (8, 1283, 717), (8, 997, 3), (4, 733, 701), (2, 311, 97)])
def test_fused_frames_equal_shading_with_the_network_p(gl, K, width, height):  # noqa: F811
    """Integer counts bit for bit; with real counts, whose products the kernels
    may contract differently, to FP32 rounding."""
    glint, render, ctx, torch = gl
    n = width * height
    gb = synth.gbuffer_random(n, seed=5, width=width)
    planes, tan = render.gbuffer_tensors(gb), render.tangent_tensor(gb)
    planes[0][::11, 3] = 0.0  # background
    fr = render.Frame(ctx, synth.env_hdr(seed=6, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=128)))
    fr.update_env()
    net = glint.Mlp(ctx, K, 256)
    net.set_params(synth.mlp_params(seed=10, K=K))
    p = net.infer(fr.env, planes, width, height, tan, torch.empty(n, K, device="cuda"))
    for mode in (glint.COUNT_INTEGER, glint.COUNT_REAL):
        got = fr.shade(planes, width, height, seed=4, count_mode=mode, tangent=tan, evaluator=glint.EVAL_MLP, mlp=net)
        want = fr.shade(planes, width, height, seed=4, count_mode=mode, evaluator=glint.EVAL_GIVEN, p_scratch=p)
        torch.cuda.synchronize()
        if mode == glint.COUNT_INTEGER:
            assert torch.equal(got, want)
        else:
            same = torch.isclose(got, want, rtol=1e-5, atol=1e-6 * float(want.max())).all(1).float().mean()
            assert same > 0.9999, float(same)
