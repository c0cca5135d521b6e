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


@pytest.mark.parametrize("wd", ["c64", "bf16"])
@pytest.mark.parametrize("supports", [(7, 9, 12, 16), (7, 8, 9), (2, 3, 5, 8, 9, 13)])
def test_thin_units_share_their_tile_regions(supports, wd):
    """About one row of a support in an 8 x 8 tile over a 2048^2 grid: the plan takes 16 x 16 tiles whose regions all
    supports share.  Forward, adjoint, the fused gradient and compensated gridding against the oracle (BF16 plans: the
    oracle's rows replaced by the plan's rounded ones), with rows across both grid edges and tiles of many rows."""
    n, K, M = 64, 2048, 130_000
    rng = np.random.default_rng(31)
    omega = rng.uniform(-np.pi, np.pi, (M, 2))
    omega[:900] = (rng.integers(-9, 9, (900, 2)) + rng.random((900, 2))) * (2 * np.pi / K) - np.pi
    omega[:900] = (omega[:900] + np.pi) % (2 * np.pi) - np.pi
    w, dl = rng.uniform(-1, 1, M), np.sqrt(2.0 / (n * K))
    Jr = np.asarray(supports, np.int8)[rng.integers(0, len(supports), M)]
    plan = pnp.Plan(n, K, omega, w, dl, Jr, J=min(supports), weight_dtype=wd)
    ora = onu.Operator(n, K, omega, w, dl, Jr, J=min(supports))
    assert plan.info["tile"] == 16
    if wd == "bf16":
        off, wts, cols = plan.export_rows(np.arange(M))
        ora.G = type(ora.G)((wts.astype(np.complex128), cols, off), shape=ora.G.shape)
        ora.GH = ora.G.conj().T.tocsr()
    x, r = rng.random((n, n)), synth.complex_normal(M, rng)
    xd, rd = to_dev_f32(x), to_dev_c64(r)
    adj = ora.adjoint(r)
    for _ in range(2):   # a stale accumulator or counter of the first call would show in the second
        assert rel_l2(to_host(plan.phi_forward(xd)), ora.forward(x)) <= TOL
        assert rel_l2(to_host(plan.phi_adjoint(rd)), adj) <= TOL
        assert rel_l2(x - to_host(plan.grad_step(xd, rd, 1.0)), ora.adjoint(ora.forward(x) - r)) <= TOL
        plan.set_unit_nnz(3000)
    plan.set_compensated(True)
    assert rel_l2(to_host(plan.phi_adjoint(rd)), adj) <= TOL
    assert plan.device_status() == 0
