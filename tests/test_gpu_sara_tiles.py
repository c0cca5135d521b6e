"""The SARA dictionary's tiled transforms at sides where a tile, a run or a filter does not fit: blocks shorter than a
filter at the coarsest level, one coefficient left, tiles with a ragged edge.  Bounds: those of the dictionary test,
relative L2 <= 1e-6 against the oracle, for the analysis and the synthesis of the oracle's coefficients."""
import numpy as np
import pytest

from oracle import sara as osara

from gpu_common import pnp, rel_l2, require_gpu, to_dev_f32, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels", [(2, 1), (16, 4), (34, 1), (68, 2), (130, 1), (144, 4), (256, 8)])
def test_dictionary_at_ragged_sides(n, levels):
    require_gpu()
    rng = np.random.default_rng(n + levels)
    x = rng.standard_normal((n, n))
    psi = osara.Sara(levels=levels)
    den = pnp.SaraDenoiser(n, 0.1, 0.1, 1, levels=levels)
    c = psi.analysis(x.astype(np.float32).astype(np.float64))
    assert rel_l2(to_host(den.analysis(to_dev_f32(x))), c) <= 1e-6
    assert rel_l2(to_host(den.synthesis(to_dev_f32(c))), psi.synthesis(c.astype(np.float32).astype(np.float64))) <= 1e-6
