"""The packed sibling draws at the ends of their range: trial counts from none
to the uint32 saturation, certain and impossible outcomes, empty subtrees,
probabilities below the small-p bias, for every number of bins."""
import numpy as np
import pytest

from paper_2507_02674_gb300 import synth
from tests._pipeline import MethodParams, oracle_shade
from tests.test_gpu_parity import _cfg, _check, gl  # noqa: F401

pytestmark = pytest.mark.gpu

COUNTS = [0.25, 1.0, 1.5, 2.0, 3.0, 17.25, 1000.0, 2.0 ** 23 + 1.0, 2.0 ** 25 + 4.0, 4.0e9, 1.0e12]


@pytest.mark.parametrize("K", [2, 4, 8, 16])
def test_draws_at_the_ends_of_their_range(gl, orc, K):  # noqa: F811
    glint, render, ctx, torch = gl
    mp = MethodParams(K=K, Wo=64, seed=23)
    env = synth.env_tiny(2)
    eye = np.eye(K, dtype=np.float32)
    half = np.zeros((2, K), np.float32)
    half[0, :K // 2] = half[1, K // 2:] = 2.0 / K
    tiny = np.full((1, K), 1e-5, np.float32)
    tiny[0, 0] = 1.0 - 1e-5 * (K - 1)
    pk = np.concatenate([eye, half, tiny, np.full((1, K), 1.0 / K, np.float32), synth.distributions(3, K, seed=5)])
    pk = np.repeat(pk, len(COUNTS), axis=0)
    n = len(pk)
    gb = synth.gbuffer_random(n, seed=31, width=n)
    rows = gb.rows16()
    rows[:, 3] = np.tile(np.array(COUNTS, np.float32), n // len(COUNTS)) * 2.0 ** 10
    rows[:, 12:16] = [2.0 ** -5, 0.0, 0.0, 2.0 ** -5]  # footprint 2^-10: N_P is the count
    gb.planes = [rows[:, 4 * i:4 * i + 4].reshape(gb.height, gb.width, 4).copy() for i in range(4)]
    fr = render.Frame(ctx, env, _cfg(glint, mp))
    fr.update_env()
    planes = render.gbuffer_tensors(gb)
    dbg = glint.debug_buffers(n, K)
    out = fr.shade(planes, gb.width, gb.height, seed=mp.seed, debug=dbg, evaluator=glint.EVAL_GIVEN,
                   p_scratch=torch.from_numpy(pk).cuda())
    torch.cuda.synchronize()
    res = {k: v.cpu().numpy() for k, v in dbg.items()}
    res["rgb"] = out[:, :3].cpu().numpy().astype(np.float64)
    # every trial ends in a bin, exactly
    assert np.array_equal(res["counts"].astype(np.float64).sum(-1)[rows[:, 3] < 2.0 ** 34],
                          res["nroot"].astype(np.float64)[rows[:, 3] < 2.0 ** 34])
    o = oracle_shade(orc, gb.rows16(), env, mp, evaluator=2, pk_in=pk.astype(np.float64))
    _check(orc, o, res)
