"""Units dealt to the warps of the gridding kernels: one per warp without a counter, and batches from the counter, at
the sizes where one gives way to the other; plain and compensated flushes.

Tolerance: relative L2 <= 1e-5, the operator bound for FP32 weights."""
import numpy as np
import pytest

import synth
from oracle import nufft as onu

from gpu_common import pnp, rel_l2, require_gpu, to_dev_c64, to_dev_f32, to_host

pytestmark = pytest.mark.gpu

TOL = 1e-5


# units of one row each: 4 warps a CTA, up to 6 CTAs on each of 152 SMs, batches of 2 from 32 units a warp on
@pytest.mark.parametrize("M", [1, 3, 607, 609, 3039, 3041, 3647, 3648, 3649, 2 * 3648 + 1, 33 * 3648])
def test_units_around_the_warp_count(M):
    require_gpu()
    n, K = 64, 128
    rng = np.random.default_rng(M)
    omega = rng.uniform(-np.pi, np.pi, (M, 2))
    plan, ora = pnp.Plan(n, K, omega), onu.Operator(n, K, omega)
    plan.set_unit_nnz(49)
    assert plan.info["n_units"] == M
    x, r = rng.random((n, n)) + 0.1, synth.complex_normal(M, rng)
    xd, rd = to_dev_f32(x), to_dev_c64(r)
    adj = ora.adjoint(r)
    for comp in (False, True, False):   # a counter left behind by one call would show in the next
        plan.set_compensated(comp)
        assert rel_l2(to_host(plan.phi_forward(xd)), ora.forward(x)) <= TOL
        assert rel_l2(to_host(plan.phi_adjoint(rd)), adj) <= TOL
        assert rel_l2(x - to_host(plan.grad_step(xd, rd, 1.0)), ora.adjoint(ora.forward(x) - r)) <= TOL
    assert plan.device_status() == 0
