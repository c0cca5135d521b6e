"""GPU parity of the BF16 gridding kernels' classes of supports: forward, adjoint and the fused gradient against FP64
sums over the plan's own rounded rows, so that a misplaced or dropped small tap shows; one row, lane groups without a
row, windows across the grid's edges; and a visibility that is not finite.

Tolerance: relative L2 <= 1e-5, the operator bound for FP32 sums (the rows' rounding is on both sides)."""
import numpy as np
import pytest

import synth
from oracle import nufft as onu

from gpu_common import pnp, rel_l2, require_gpu, to_dev_c64, to_dev_f32, to_host

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _problem(J, M, n, K, rng):
    omega = rng.uniform(-np.pi, np.pi, (M, 2))
    dense = M // 3
    omega[:dense] = (rng.integers(-2, 2, (dense, 2)) + rng.uniform(0, 1, (dense, 2))) * (2 * np.pi / K) - np.pi
    omega[:dense] = (omega[:dense] + np.pi) % (2 * np.pi) - np.pi
    args = (omega, None, 0.0, None) if J <= 14 else (omega, rng.uniform(-1, 1, M), np.sqrt(4.0 / (n * K)),
                                                     np.full(M, J, np.int8))
    plan = pnp.Plan(n, K, *args, J=min(J, 7 if J > 14 else J), weight_dtype="bf16")
    ora = onu.Operator(n, K, *args, J=min(J, 7 if J > 14 else J))
    off, wts, cols = plan.export_rows(np.arange(M))
    ora.G = type(ora.G)((wts.astype(np.complex128), cols, off), shape=ora.G.shape)
    ora.GH = ora.G.conj().T.tocsr()
    return plan, ora


@pytest.mark.parametrize("J", [2, 4, 6, 7, 8, 9, 10, 12, 14, 15, 16])
@pytest.mark.parametrize("M", [1, 5, 4001])
def test_bf16_supports(J, M):
    require_gpu()
    n, K = 64, 128
    rng = np.random.default_rng(3000 * J + M)
    plan, ora = _problem(J, M, n, K, rng)
    x, r = np.maximum(rng.standard_normal((n, n)), 0) + 0.1, synth.complex_normal(M, rng)
    x = x.astype(np.float32).astype(np.float64)
    r = r.astype(np.complex64).astype(np.complex128)
    xd, rd = to_dev_f32(x), to_dev_c64(r)
    assert rel_l2(to_host(plan.phi_forward(xd)), ora.forward(x)) <= TOL
    adj = ora.adjoint(r)
    assert rel_l2(to_host(plan.phi_adjoint(rd)), adj) <= TOL
    g = to_host(plan.grad_step(xd, rd, 1.0))
    assert rel_l2(x - g, ora.adjoint(ora.forward(x) - r)) <= TOL
    bad = r.copy()
    bad[M // 2] = np.nan
    assert not np.isfinite(to_host(plan.phi_adjoint(to_dev_c64(bad)))).any()
    assert rel_l2(to_host(plan.phi_adjoint(rd)), adj) <= TOL
    assert plan.device_status() == 0
