"""Settings without an effect on the kernels cost nothing."""
import time

import numpy as np

import pytest

from gpu_common import pnp, require_gpu, to_dev_c64, torch
import synth

pytestmark = pytest.mark.gpu


def test_row_batch_does_not_drop_the_captured_loop():
    """The row batch is kept and reported only: alternating it must not make each run capture its loop again (a capture
    of this loop takes several times as long as the two iterations run)."""
    require_gpu()
    n, K, M = 64, 128, 2000
    rng = np.random.default_rng(8)
    plan = pnp.Plan(n, K, rng.uniform(-np.pi, np.pi, (M, 2)))
    den, y = pnp.HaarDenoiser(0.01), to_dev_c64(synth.complex_normal(M, rng))

    def ms(batches, reps=40):
        out = []
        for i in range(reps):
            plan.set_row_batch(batches[i % len(batches)])
            torch.cuda.synchronize()
            t = time.perf_counter()
            plan.fb_run(den, y, gamma=1e-6, L=1.0, max_iter=2)
            torch.cuda.synchronize()
            out.append((time.perf_counter() - t) * 1e3)
        return float(np.median(out))

    ms([2])
    kept, changed = ms([2]), ms([1, 4])
    print(f"two iterations: {kept:.3f} ms, with the row batch changed before each run {changed:.3f} ms")
    assert plan.info["row_batch"] == 4
    assert changed <= 1.5 * kept
