"""glint_normal_quantile beyond the uniforms that the kernels draw: any p in
(0, 1), where 2p - 1 is rounded and, below 2^-25, is -1."""
import numpy as np
import pytest

from tests.test_gpu_parity import gl  # noqa: F401

pytestmark = pytest.mark.gpu


def _quantile(gl, p):  # noqa: F811
    glint, render, ctx, torch = gl
    return glint.normal_quantile(torch.from_numpy(p).cuda()).cpu().numpy().astype(np.float64)


def test_any_p(gl):  # noqa: F811
    """2^-20 relative, 2^-22 absolute near the median: the polynomials' fit (6e-8),
    lg2.approx (2^-22) and a dozen roundings of 2^-24 stay below half of it."""
    from scipy import special
    rng = np.random.default_rng(7)
    p = np.concatenate([rng.random(1 << 20), 2.0 ** rng.uniform(-25, 0, 1 << 20),
                        1 - 2.0 ** rng.uniform(-24, 0, 1 << 18), 0.5 + rng.uniform(-1e-3, 1e-3, 4096),
                        [2.0 ** -25, 1e-7, 3e-7, 1 - 2.0 ** -24]]).astype(np.float32)
    p = p[(p >= 2.0 ** -25) & (p < 1)]
    z, ref = _quantile(gl, p), special.ndtri(p.astype(np.float64))
    big = np.abs(ref) > 0.25
    assert (np.abs(z - ref)[big] / np.abs(ref[big])).max() < 2.0 ** -20
    assert np.abs(z - ref)[~big].max() < 2.0 ** -22


def test_extrapolated_tail(gl):  # noqa: F811
    """Below 2^-25 the fit is extrapolated; in exact arithmetic it is 1.1e-6 off
    at 1e-8, 2.7e-4 at 1e-10."""
    from scipy import special
    for lo, bound in ((1e-8, 1.1e-6 + 2.0 ** -20), (1e-10, 2.7e-4)):
        p = np.geomspace(lo, 2.0 ** -25, 1001).astype(np.float32)[1:]
        z, ref = _quantile(gl, p), special.ndtri(p.astype(np.float64))
        assert (np.abs(z - ref) / np.abs(ref)).max() < bound
