"""A launch that the runtime refuses is reported by the call that made it and by no
later one.  The refusal is a stream whose capture was invalidated (by an
allocation during it): nothing reaches the GPU."""
import ctypes

import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["shade", "shade_grid", "shade_mlp", "probs", "probs_e2", "update"])
def test_refused_launch_is_reported_once(gl, call):  # noqa: F811
    glint, render, ctx, torch = gl
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])  # the one the library and torch use
    K, n = 4, 300
    fr = render.Frame(ctx, synth.env_hdr(seed=3, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=64)))
    fr.update_env()
    gb = synth.gbuffer_random(n, seed=5, width=n)
    planes, tan = render.gbuffer_tensors(gb), render.tangent_tensor(gb)
    net = glint.Mlp(ctx, K, 256)
    net.set_params(synth.mlp_params(seed=3, K=K))
    out, p = torch.empty(n, 4, device="cuda"), torch.empty(n, K, device="cuda")
    x, lp = torch.zeros(n, 64, device="cuda", dtype=torch.int16), torch.zeros(n, K, device="cuda")
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    handle, graph, ptr = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 0) == 0  # global: an allocation invalidates it
    try:
        assert rt.cudaMalloc(ctypes.byref(ptr), 256) != 0
        rt.cudaGetLastError()
        with pytest.raises(glint.GlintError):
            if call == "update":
                fr.update_env(stream=s)
            elif call == "probs":
                fr.probs(planes, n, 1, out=p, stream=s)
            elif call == "probs_e2":
                fr.probs(planes, n, 1, evaluator=glint.EVAL_E2, tangent=tan, out=p, stream=s)
            elif call == "shade_mlp":
                fr.shade(planes, n, 1, out=out, evaluator=glint.EVAL_MLP, mlp=net, tangent=tan, stream=s)
            else:
                fr.shade(planes, n, 1, out=out, grid=int(call == "shade_grid"), stream=s)
        assert rt.cudaGetLastError() == 0
    finally:
        rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
        rt.cudaGetLastError()
    net.forward(x, lp, out=p)  # ends in cudaGetLastError(): reports only its own launch
    torch.cuda.synchronize()
    assert torch.allclose(p.sum(1), torch.ones(n, device="cuda"), atol=1e-5)
