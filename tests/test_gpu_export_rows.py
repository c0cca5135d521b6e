"""Exported rows of G are the definition's weights rounded once to complex64, whatever the plan keeps (2^-24 relative per
component), and in BF16 plans those rounded to BF16, bit for bit: data weights, w-kernels, rows across both grid edges.

The definition is evaluated in FP64 on both sides by different routes; 1e-11 of the row's largest weight allows for that."""
import numpy as np
import pytest

from oracle import nufft as onu

from gpu_common import pnp, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("supports", [(2,), (7,), (7, 9, 12, 16)])
def test_exported_rows_are_rounded_once(supports):
    require_gpu()
    n, K, M = 64, 128, 3000
    rng = np.random.default_rng(17)
    omega, w, dl, Jr = rng.uniform(-np.pi, np.pi, (M, 2)), None, 0.0, None
    if len(supports) > 1:
        w, dl = rng.uniform(-1, 1, M), np.sqrt(4.0 / (n * K))
        Jr = np.asarray(supports, np.int8)[rng.integers(0, len(supports), M)]
    d = rng.uniform(0.1, 2.0, M)
    plan = pnp.Plan(n, K, omega, w, dl, Jr, J=supports[0], row_scale=d)
    G = onu.Operator(n, K, omega, w, dl, Jr, J=supports[0], row_scale=d).G
    rows = rng.permutation(M)[:1000]
    u = 2.0 ** -24
    off, wts, cols = plan.export_rows(rows)
    for i, m in enumerate(rows):
        sl = slice(off[i], off[i + 1])
        got, ref = np.zeros(K * K, np.complex128), np.zeros(K * K, np.complex128)
        got[cols[sl]] = wts[sl]
        ref[G[m].indices] = G[m].data
        tol = 1e-11 * np.abs(ref).max()
        assert np.all(np.abs(got.real - ref.real) <= u * np.abs(ref.real) + tol), m
        assert np.all(np.abs(got.imag - ref.imag) <= u * np.abs(ref.imag) + tol), m
    bf = pnp.Plan(n, K, omega, w, dl, Jr, J=supports[0], weight_dtype="bf16", row_scale=d)
    off_b, wts_b, cols_b = bf.export_rows(rows)
    assert np.array_equal(off_b, off) and np.array_equal(cols_b, cols)
    rounded = torch.view_as_real(torch.from_numpy(wts)).to(torch.bfloat16).to(torch.float32)
    assert np.array_equal(torch.view_as_real(torch.from_numpy(wts_b)).numpy(), rounded.numpy())
