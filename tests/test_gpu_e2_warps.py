"""E2's p_k by a warp a pixel (glint_reflect_probs): every K, point counts that
do and do not fill whole steps of a warp, maps down to a few texels, background
and single-pixel frames, several pixels a warp, against the oracle's quadrature
under its E2 tie model."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams, oracle_shade
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("S,H", [(4, 8), (5, 128), (8, 32), (13, 128), (16, 128), (32, 256), (33, 64)])
def test_warp_quadrature_matches_oracle(gl, orc, K, S, H):  # noqa: F811
    glint, render, ctx, torch = gl
    mp = MethodParams(K=K, Wo=32)
    env = synth.env_hdr(seed=9, W=2 * H, H=H)
    gb = synth.gbuffer_random(203, seed=61 + K + S, width=203, a_lo=0.02, a_hi=1.0)
    rows = gb.rows16()
    rows[::17, 3] = 0.0  # background
    gb.planes = [rows[:, 4 * i:4 * i + 4].reshape(gb.height, gb.width, 4).copy() for i in range(4)]
    fr = render.Frame(ctx, env, _cfg(glint, mp))
    fr.update_env()
    planes, tan = render.gbuffer_tensors(gb), render.tangent_tensor(gb)
    p = fr.probs(planes, gb.width, 1, evaluator=glint.EVAL_E2, e2_samples=S, tangent=tan).cpu().numpy()
    one = fr.probs([t[1:2].contiguous() for t in planes], 1, 1, evaluator=glint.EVAL_E2, e2_samples=S,
                   tangent=tan[1:2].contiguous()).cpu().numpy()
    assert np.array_equal(one[0], p[1])
    bg = rows[:, 3] == 0
    assert np.all(p[bg] == 0)
    o = oracle_shade(orc, gb.rows16(), env, mp, evaluator=1, tangents=gb.tangents(), e2_S=S)
    sure = ~bg & (o.e2_flags == 0)
    assert sure.sum() > 0.9 * (~bg).sum()
    rtol, atol = orc.TIE_E2[0], orc.TIE_E2[4]
    err = np.abs(p[sure].astype(np.float64) - o.pk[sure])
    assert np.all(err <= rtol * o.pk[sure] + atol), (err / (rtol * o.pk[sure] + atol)).max()


def test_pixels_do_not_depend_on_the_frame(gl):  # noqa: F811
    """Frames large enough for 2, 4 and 8 pixels a warp give each pixel the p_k
    it has in a frame of its own size class."""
    glint, render, ctx, torch = gl
    K, S = 8, 16
    fr = render.Frame(ctx, synth.env_hdr(seed=9, W=256, H=128), _cfg(glint, MethodParams(K=K, Wo=32)))
    fr.update_env()
    gb = synth.gbuffer_random(130003, seed=3, width=130003)
    planes, tan = render.gbuffer_tensors(gb), render.tangent_tensor(gb)

    def probs(n):
        return fr.probs([t[:n].contiguous() for t in planes], n, 1, evaluator=glint.EVAL_E2, e2_samples=S,
                        tangent=tan[:n].contiguous())

    ref = probs(2001)
    for n in (30001, 60007, 130003):
        assert torch.equal(probs(n)[:2001], ref), n
