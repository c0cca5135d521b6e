"""GPU parity of the gridding kernels' classes of supports against the FP64 oracle: one row, a few rows (lane
groups without one), many rows per window, windows that wrap around both grid edges; and a visibility that is
not finite stays within the call that brought it (the padding taps of its window must not reach grid cells
outside the uv support, which nothing zeroes again).

Tolerance: relative L2 <= 1e-5, the operator bound for FP32 weights."""
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


def _rows(J, M, K, rng):
    omega = rng.uniform(-np.pi, np.pi, (M, 2))
    dense = M // 3                                      # a third of the rows in a few cells at the grid's corner
    omega[:dense] = (rng.integers(-2, 2, (dense, 2)) + rng.uniform(0, 1, (dense, 2))) * (2 * np.pi / K) - np.pi
    omega[:dense] = (omega[:dense] + np.pi) % (2 * np.pi) - np.pi
    if J <= 14:
        return omega, None, 0.0, None, J                # KB rows of support J
    return omega, rng.uniform(-1, 1, M), np.sqrt(4.0 / (64 * K)), np.full(M, J, np.int8), 7


@pytest.mark.parametrize("J", [2, 5, 7, 8, 9, 10, 12, 13, 14, 15, 16])
@pytest.mark.parametrize("M", [1, 5, 4001])
def test_supports_against_oracle(J, M):
    n, K = 64, 128
    rng = np.random.default_rng(1000 * J + M)
    omega, w, dl, Jr, J0 = _rows(J, M, K, rng)
    gpu = pnp.Plan(n, K, omega, w, dl, Jr, J=J0)
    ora = onu.Operator(n, K, omega, w, dl, Jr, J=J0)
    x = np.maximum(rng.standard_normal((n, n)), 0) + 0.1
    r = synth.complex_normal(M, rng)
    assert rel_l2(to_host(gpu.phi_forward(to_dev_f32(x))), ora.forward(x)) <= TOL
    assert rel_l2(to_host(gpu.phi_adjoint(to_dev_c64(r))), ora.adjoint(r)) <= TOL
    g = to_host(gpu.grad_step(to_dev_f32(x), to_dev_c64(r), 1.0))
    assert gpu.device_status() == 0
    assert rel_l2(x - g, ora.adjoint(ora.forward(x) - r)) <= TOL


@pytest.mark.parametrize("supports", [(7,), (9, 12, 16)])
def test_non_finite_visibility_does_not_outlive_its_call(supports):
    n, K, M = 64, 128, 900
    rng = np.random.default_rng(5)
    omega = rng.uniform(-0.3 * np.pi, 0.3 * np.pi, (M, 2))   # a support well inside the grid
    w, dl, Jr = None, 0.0, None
    if len(supports) > 1:
        w, dl = rng.uniform(-1, 1, M), np.sqrt(4.0 / (n * K))
        Jr = np.asarray(supports, np.int8)[rng.integers(0, len(supports), M)]
    gpu = pnp.Plan(n, K, omega, w, dl, Jr)
    r = synth.complex_normal(M, rng)
    clean = to_host(gpu.phi_adjoint(to_dev_c64(r)))
    for bad in (np.nan, np.inf):
        q = r.copy()
        q[M // 2] = bad
        assert not np.isfinite(to_host(gpu.phi_adjoint(to_dev_c64(q)))).any()
        assert rel_l2(to_host(gpu.phi_adjoint(to_dev_c64(r))), clean) <= TOL
