"""The map update's two filter kernels, its 8- and 16-byte texel loads and its
smallest pyramids."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


def _filtered(gl, mp, env, texels=None):  # noqa: F811
    glint, render, ctx, torch = gl
    fr = render.Frame(ctx, env, _cfg(glint, mp))
    if texels is not None:
        fr.texels = texels
    fr.update_env()
    torch.cuda.synchronize()
    widths, flat = fr.env.export(glint.ENV_FILTERED)
    at = np.concatenate([[0], np.cumsum(widths.astype(int) * (widths.astype(int) // 2))])
    return fr, [flat[a:b] for a, b in zip(at, at[1:])]


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("S,wfmt,H", [(1, 0, 64), (2, 1, 256), (63, 0, 256), (64, 2, 32), (65, 0, 256), (200, 3, 128)])
def test_both_filter_kernels_give_the_same_texels(gl, K, S, wfmt, H):  # noqa: F811
    """Levels of the same width filtered among 7456 texels (a thread a sample) and
    among 43552 (a thread a texel and sample parity) are equal bit for bit."""
    env = synth.env_hdr(seed=4, W=2 * H, H=H)
    _, small = _filtered(gl, MethodParams(K=K, S=S, Wo=64, wfmt=wfmt), env)
    _, large = _filtered(gl, MethodParams(K=K, S=S, Wo=256, wfmt=wfmt), env)
    same = [r for r in range(len(small)) if small[r].shape == large[r].shape]
    assert len(same) >= 6
    for r in same:
        assert np.array_equal(small[r].view(np.uint32), large[r].view(np.uint32)), r


def test_texels_aligned_to_8_bytes(gl):  # noqa: F811
    glint, render, ctx, torch = gl
    env = synth.env_hdr(seed=5, W=128, H=64)
    mp = MethodParams(K=8, Wo=64)
    ref, a = _filtered(gl, mp, env)
    buf = torch.empty(ref.texels.numel() + 4, dtype=torch.float16, device="cuda")
    odd = buf[4:].view(ref.texels.shape)
    odd.copy_(ref.texels)
    assert odd.data_ptr() % 16 == 8
    got, b = _filtered(gl, mp, env, odd)
    assert np.array_equal(ref.env.levels(), got.env.levels())
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("H", [2, 4, 8, 16, 64])
@pytest.mark.parametrize("K", [2, 8, 16])
def test_small_pyramids_match_oracle(gl, orc, H, K):  # noqa: F811
    """Maps of a single tile or less, and one whose upper levels the last block
    builds; tolerances as the pyramid's parity test has them."""
    env = synth.env_hdr(seed=6, W=2 * H, H=H)
    mp = MethodParams(K=K, Wo=16)
    fr, _ = _filtered(gl, mp, env)
    e = orc.env_full(env.rgba32(), env.scale, mp.K, mp.ell)
    assert np.allclose(fr.env.levels().astype(np.float64), e.levels, rtol=3e-6, atol=0)
    for m in range(fr.env.M):
        g, o = fr.env.export(gl[0].ENV_PYRAMID, m).astype(np.float64), e.mips[m]
        assert g.shape == o.shape
        assert np.max(np.abs(g[..., 3:] - o[..., 3:])) < 4e-6, m
        assert np.max(np.abs(g[..., :3] - o[..., :3]) / np.abs(o[..., :3])) < 2e-6, m
