"""Gridding of sparse uv coverage: a grid that does not stay in L2, and few rows per grid tile.

Tolerances: relative L2 <= 1e-5, the operator bound for FP32 weights."""
import numpy as np
import pytest

import synth
from oracle import nufft as onu

from gpu_common import pnp, rel_l2, require_gpu, to_dev_c64, to_dev_f32, to_host

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _gridding_ms(plan, call, reps=5):
    call()
    plan.set_timing(True)
    for _ in range(reps):
        call()
    ms = plan.read_timing()["gridding"][0] / reps
    plan.set_timing(False)
    return ms


def test_gridding_beyond_l2():
    """Rows spread over a 4096^2 grid (134 MB), taps across both grid edges: parity, and the gridding pass takes at
    most twice the de-gridding pass, which reads the same rows and touches the same cells (atomics on lines that
    were not in L2 made it three times)."""
    n, K, M = 2048, 4096, 300_000
    rng = np.random.default_rng(21)
    omega = rng.uniform(-np.pi, np.pi, (M, 2))
    omega[0] = (np.pi * (1 - 1e-6), -np.pi)
    plan, ora = pnp.Plan(n, K, omega), onu.Operator(n, K, omega)
    x, r = rng.random((n, n)), synth.complex_normal(M, rng)
    xd, rd = to_dev_f32(x), to_dev_c64(r)
    assert rel_l2(to_host(plan.phi_adjoint(rd)), ora.adjoint(r)) <= TOL
    g = to_host(plan.grad_step(xd, rd, 1.0))
    assert rel_l2(x - g, ora.adjoint(ora.forward(x) - r)) <= TOL
    assert plan.device_status() == 0
    assert _gridding_ms(plan, lambda: plan.phi_adjoint(rd)) <= 2.0 * _gridding_ms(plan, lambda: plan.phi_forward(xd))
