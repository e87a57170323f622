"""The comparison draws and the anisotropic grid give the same image with and
without the per-pixel intermediates (two kernels each), ragged tail included."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("draw,grid", [(0, 1), (1, 0), (2, 0), (3, 0)])
def test_intermediates_leave_the_image_alone(gl, K, draw, grid):  # noqa: F811
    glint, render, ctx, torch = gl
    env = synth.env_hdr(seed=6, W=256, H=128)
    gb = synth.gbuffer_random(2000 + 37, seed=K, width=2037)
    fr = render.Frame(ctx, env, _cfg(glint, MethodParams(K=K, Wo=64)))
    fr.update_env()
    planes = render.gbuffer_tensors(gb)
    for mode in (glint.COUNT_INTEGER, glint.COUNT_REAL):
        kw = dict(seed=5, count_mode=mode, draw=draw, grid=grid, gamma=0.01 if draw == 3 else 0.0)
        dbg = glint.debug_buffers(2037, K, samples=12 if grid else 6)
        want = fr.shade(planes, gb.width, gb.height, debug=dbg, **kw).clone()
        got = fr.shade(planes, gb.width, gb.height, **kw)
        torch.cuda.synchronize()
        np.testing.assert_allclose(got.cpu().numpy(), want.cpu().numpy(), rtol=1e-4, atol=1e-9)
