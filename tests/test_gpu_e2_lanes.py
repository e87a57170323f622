"""E2's p_k by 1, 8 and 32 lanes a pixel (glint_reflect_probs): both sides of every
line of the rule that chooses them, several rings a lane, several pixels a group
of lanes, and frames of different size, against the oracle's quadrature under
its E2 tie model and against one another."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams, oracle_shade
from tests.test_gpu_parity import _cfg, gl  # noqa: F401

pytestmark = pytest.mark.gpu


def _frame(gl, n, K, H=128):  # noqa: F811
    glint, render, ctx, torch = gl
    mp = MethodParams(K=K, Wo=32)
    env = synth.env_hdr(seed=9, W=2 * H, H=H)
    gb = synth.gbuffer_random(n, seed=61 + K, width=n, a_lo=0.02, a_hi=1.0)
    rows = gb.rows16()
    rows[::17, 3] = 0.0  # background
    gb.planes = [rows[:, 4 * i:4 * i + 4].reshape(gb.height, gb.width, 4).copy() for i in range(4)]
    fr = render.Frame(ctx, env, _cfg(glint, mp))
    fr.update_env()
    planes, tan = render.gbuffer_tensors(gb), render.tangent_tensor(gb)

    def probs(S, m=n):
        return fr.probs([t[:m].contiguous() for t in planes], m, 1, evaluator=glint.EVAL_E2, e2_samples=S,
                        tangent=tan[:m].contiguous()).cpu().numpy()

    def shaded(S):
        dbg = glint.debug_buffers(n, K)
        fr.shade(planes, n, 1, evaluator=glint.EVAL_E2, e2_samples=S, tangent=tan, debug=dbg)
        return dbg["p"].cpu().numpy()

    return env, mp, gb, rows, probs, shaded


def _near_oracle(orc, p, env, mp, rows, tangents, S):
    o = oracle_shade(orc, rows, env, mp, evaluator=1, tangents=tangents, e2_S=S)
    bg = rows[:, 3] == 0
    assert np.all(p[bg] == 0)
    sure = ~bg & (o.e2_flags == 0)
    assert 2 * sure.sum() > (~bg).sum()  # (the oracle leaves out more pixels the more points there are)
    err = np.abs(p[sure].astype(np.float64) - o.pk[sure])
    bound = orc.TIE_E2[0] * o.pk[sure] + orc.TIE_E2[4]
    assert np.all(err <= bound), (err / bound).max()


@pytest.mark.parametrize("K,S", [(2, 8), (2, 16), (2, 23), (2, 24), (4, 15), (4, 16), (4, 17), (8, 11), (8, 12),
                                 (8, 16), (8, 20), (8, 21), (16, 7), (16, 8), (16, 16), (16, 19), (16, 20), (16, 21)])
def test_lanes_match_oracle(gl, orc, K, S):  # noqa: F811
    env, mp, gb, rows, probs, _ = _frame(gl, 205, K)
    _near_oracle(orc, probs(S), env, mp, rows, gb.tangents(), S)


@pytest.mark.parametrize("K", [4, 8, 16])
@pytest.mark.parametrize("S", [64, 256])
def test_many_rings_match_oracle(gl, orc, K, S):  # noqa: F811
    env, mp, gb, rows, probs, _ = _frame(gl, 37, K)
    _near_oracle(orc, probs(S), env, mp, rows, gb.tangents(), S)


@pytest.mark.parametrize("K,S", [(4, 13), (4, 16), (8, 7), (8, 13), (8, 16), (8, 24), (16, 7), (16, 16), (16, 33)])
def test_large_frames_match_oracle(gl, orc, K, S):  # noqa: F811
    """A frame large enough for several pixels a group, a few hundred of its pixels."""
    n = 130003
    env, mp, gb, rows, probs, _ = _frame(gl, n, K)
    pick = np.unique(np.concatenate([np.random.default_rng(S).integers(0, n, 300), [0, 1, n - 2, n - 1]]))
    _near_oracle(orc, probs(S)[pick], env, mp, rows[pick], gb.tangents()[pick], S)


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("S", [4, 5, 7, 8, 11, 12, 13, 16, 20, 23, 24, 32])
def test_frames_of_different_size(gl, orc, K, S):  # noqa: F811
    """A crop's p_k equals the whole frame's, bit for bit unless glint.h names K and S;
    there, and from glint_shade's own, it differs by less than the tie model allows
    two evaluations (twice its bound)."""
    n, m = 60007, 2003
    _, _, _, rows, probs, shaded = _frame(gl, n, K)
    whole, crop = probs(S), probs(S, m)
    by_size = 5 <= S < {2: 24, 4: 24, 8: 12, 16: 8}[K] and not (K <= 4 and S == 16)
    if not by_size:
        assert np.array_equal(whole[:m], crop)

    def near(a, b):
        return np.all(np.abs(a.astype(np.float64) - b) <= 2 * (orc.TIE_E2[0] * b + orc.TIE_E2[4]))

    assert near(whole[:m], crop)
    assert near(whole, shaded(S))
