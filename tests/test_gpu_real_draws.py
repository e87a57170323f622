"""Real-valued draws at the ends of their range, and the stored codes of every
compressed weight format, for every number of bins."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams, oracle_shade
from tests.test_gpu_draw_edges import COUNTS
from tests.test_gpu_parity import _cfg, _check, _run, gl  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 4, 8, 16])
def test_real_draws_at_the_ends_of_their_range(gl, orc, K):  # noqa: F811
    glint, render, ctx, torch = gl
    mp = MethodParams(K=K, Wo=64, seed=29, integer_mode=False)
    env = synth.env_tiny(2)
    counts = [0.0] + COUNTS
    half = np.zeros((2, K), np.float32)
    half[0, :K // 2] = half[1, K // 2:] = 2.0 / K
    pk = np.concatenate([np.eye(K, dtype=np.float32), half, np.full((1, K), 1.0 / K, np.float32),
                         synth.distributions(4, K, seed=6)])
    pk = np.repeat(pk, len(counts), axis=0)
    n = len(pk)
    gb = synth.gbuffer_random(n, seed=33, width=n)
    rows = gb.rows16()
    rows[:, 3] = np.maximum(np.tile(np.array(counts, np.float32), n // len(counts)) * 2.0 ** 10, 2.0 ** -100)
    rows[:, 12:16] = [2.0 ** -5, 0.0, 0.0, 2.0 ** -5]  # footprint 2^-10: N_P is the count
    gb.planes = [rows[:, 4 * i:4 * i + 4].reshape(gb.height, gb.width, 4).copy() for i in range(4)]
    fr = render.Frame(ctx, env, _cfg(glint, mp))
    fr.update_env()
    planes = render.gbuffer_tensors(gb)
    dbg = glint.debug_buffers(n, K)
    out = fr.shade(planes, gb.width, gb.height, seed=mp.seed, count_mode=glint.COUNT_REAL, debug=dbg,
                   evaluator=glint.EVAL_GIVEN, p_scratch=torch.from_numpy(pk).cuda())
    torch.cuda.synchronize()
    res = {k: v.cpu().numpy() for k, v in dbg.items()}
    res["rgb"] = out[:, :3].cpu().numpy().astype(np.float64)
    o = oracle_shade(orc, gb.rows16(), env, mp, evaluator=2, pk_in=pk.astype(np.float64))
    _check(orc, o, res, integer_mode=False)


@pytest.mark.parametrize("K", [2, 4, 8, 16])
@pytest.mark.parametrize("wfmt", [1, 2, 3])
def test_probabilities_from_stored_codes(gl, K, wfmt):  # noqa: F811
    """p_k = V W_k (+ U for k = 0) with V <= 1 and W_k a convex sum of stored
    weights in [0, 1]: storing them moves p_k by half a code at most (float16
    2^-12, unorm16 2^-17, unorm8 2^-9), plus FP32 rounding."""
    env = synth.env_hdr(seed=6, W=256, H=128)
    gb = synth.gbuffer_random(1500 + 13, seed=K, width=1513)
    exact = _run(gl, env, gb, MethodParams(K=K, Wo=128, seed=3))["p"].astype(np.float64)
    stored = _run(gl, env, gb, MethodParams(K=K, Wo=128, seed=3, wfmt=wfmt))["p"].astype(np.float64)
    assert np.abs(stored - exact).max() <= {1: 2.0 ** -12, 2: 2.0 ** -17, 3: 2.0 ** -9}[wfmt] + 2.0 ** -19
