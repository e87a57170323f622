"""Real counts of pixels with at most one microfacet, whose warps draw them by
their gates alone: the same image as beside dense pixels, which take the whole
draw's path."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu

ONE = np.float32(1)
COUNTS = [1e-6, 0.03, 0.5, float(np.nextafter(ONE, ONE * 0)), 1.0]


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("grid", [0, 1])
def test_sparse_warps_draw_as_mixed_ones(gl, K, grid):  # noqa: F811
    glint, render, ctx, torch = gl
    n = 4099
    fr = render.Frame(ctx, synth.env_hdr(seed=6, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=64)))
    fr.update_env()
    gb = synth.gbuffer_random(n, seed=33 + K, width=n)
    planes = [t.clone() for t in render.gbuffer_tensors(gb)]
    planes[0][:, 3] = torch.tensor(COUNTS, device="cuda").repeat(n // len(COUNTS) + 1)[:n] * 2.0 ** 10
    planes[0][::29, 3] = 0.0  # background
    planes[3][:] = torch.tensor([2.0 ** -5, 0.0, 0.0, 2.0 ** -5], device="cuda")  # footprint 2^-10: N_P is the count
    kw = dict(seed=4, count_mode=glint.COUNT_REAL, grid=grid)
    sparse = fr.shade(planes, n, 1, **kw)
    mixed = [t.repeat_interleave(2, 0) for t in planes]
    mixed[0][1::2, 3] = 2.0 ** 17  # a dense pixel beside each
    both = fr.shade(mixed, 2 * n, 1, **kw)
    torch.cuda.synchronize()
    assert (sparse[:, :3] > 0).any()
    assert torch.equal(both[::2], sparse)
