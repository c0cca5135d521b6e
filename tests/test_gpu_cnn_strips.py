"""Strip heights of the CNN's work lists: what the autotuner times, and strips of one row."""
import numpy as np
import pytest

import synth
from oracle import cnn as ocnn

from gpu_common import pnp, rel_l2, require_gpu, to_dev_f32, to_host

pytestmark = pytest.mark.gpu

BF16_U = 2.0 ** -8


def _params(seed):
    return synth.cnn_init(np.random.default_rng(seed), 64, 8, 1.0)


def test_autotuner_times_the_default():
    """2048^2 in one piece is 216 rows an SM, more than twice the tallest of the low heights: all seven heights have lists of
    their own, and the tuner times each, the default among them (it once timed six and installed the best of those)."""
    require_gpu()
    n, reps = 2048, 2
    den = pnp.CnnDenoiser(_params(3), n, halo=0)
    z = to_dev_f32(np.random.default_rng(4).random((n, n)))
    k0 = pnp.kernel_launches()
    base = to_host(den.denoise(z))
    per = pnp.kernel_launches() - k0
    tune = den.autotune(z, reps=reps)
    assert pnp.kernel_launches() - k0 - per == 7 * (reps + 1) * per
    assert tune["strip_rows"] in (16, 24, 32, 48, 64, 96, 1024) and tune["denoise_ms"] > 0
    den.set_strip_rows(300)    # the default's lists
    k0 = pnp.kernel_launches()
    den.autotune(z, reps=reps)
    assert pnp.kernel_launches() - k0 == 7 * (reps + 1) * per
    den.set_strip_rows(7)      # a list of its own
    k0 = pnp.kernel_launches()
    den.autotune(z, reps=reps)
    assert pnp.kernel_launches() - k0 == 8 * (reps + 1) * per
    assert np.array_equal(to_host(den.denoise(z)), base)


def test_facets_of_one_row():
    """306 facets of one row: the SMs' shares are 6 or 7 strips of one row, and the shorter lists are filled up with
    empty strips."""
    require_gpu()
    n = 306
    params = _params(5)
    z = np.random.default_rng(6).random((n, n))
    den = pnp.CnnDenoiser(params, n, facet_rows=[1] * n, halo=0)
    zd = to_dev_f32(z)
    base = to_host(den.denoise(zd))
    for rows in (4, 1024):
        den.set_strip_rows(rows)
        assert np.array_equal(to_host(den.denoise(zd)), base)
    assert den.device_status() == 0
    zf = z.astype(np.float32).astype(np.float64)
    assert rel_l2(base, ocnn.denoise_faceted(params, zf, [1] * n, [n], 0, bf16=True)) <= BF16_U
