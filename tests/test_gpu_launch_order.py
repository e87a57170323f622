"""Kernels launched before their predecessor in the stream has ended read what it
wrote and overwrite what it has read: calls in a row without a host wait, each
reading the last one's output, with frames of less and more than a block an SM
(both ways of letting the next kernel start), against the same calls with a wait
after each."""
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix", [1, 152 * 128, 152 * 128 + 1, 80003, 200003])
def test_calls_in_a_row(gl, npix):  # noqa: F811
    glint, render, ctx, torch = gl
    K = 4
    fr = [render.Frame(ctx, synth.env_hdr(seed=s, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=64))) for s in (3, 4)]
    gb = synth.gbuffer_random(npix, seed=5, width=npix)
    planes, tan = render.gbuffer_tensors(gb), render.tangent_tensor(gb)
    p = torch.empty(npix, K, device="cuda")

    def frames(wait):
        out = []
        for i in range(8):
            f = fr[i % 2]
            f.update_env()
            wait()
            ev = (glint.EVAL_E1, glint.EVAL_E2, glint.EVAL_E1_ANISO)[i % 3]
            f.probs(planes, npix, 1, evaluator=ev, e2_samples=(3, 16)[i % 2], tangent=tan, out=p)  # overwrites p
            wait()
            out.append(f.shade(planes, npix, 1, seed=i, evaluator=glint.EVAL_GIVEN, p_scratch=p))
            wait()
            out.append(f.shade(planes, npix, 1, seed=i, grid=i % 2))
            wait()
        torch.cuda.synchronize()
        return out

    ref = frames(torch.cuda.synchronize)
    for _ in range(3):
        for a, b in zip(frames(lambda: None), ref):
            assert torch.equal(a, b)
