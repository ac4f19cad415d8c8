"""Failure detection of the resident iteration without a fault: a block waits
for a barrier and for a sum that never come, gives up after a short limit, and
the call returns LQCD_ETIMEOUT although the job's first block ended well and
wrote "converged".  The same context then solves correctly, through the
resident iteration."""
import time

import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_bounded_resident_wait_times_out_and_context_survives(gpu):
    dims = (4, 6, 8, 10)
    b = inputs.gaussian_field(dims, k=121)
    with gpu.Context(dims) as c:
        c.links_upload(inputs.random_links(dims, seed=121))
        x0, i0 = c.mscg_solve(0.05, [1e-3, 0.1], 1e-10, b)
        for limit in (0.02, 0.1):
            t0 = time.perf_counter()
            with pytest.raises(gpu.LqcdError) as e:
                c.selftest_resident_wait(limit)
            dt = time.perf_counter() - t0
            assert e.value.status == gpu.LQCD_ETIMEOUT
            assert 2 * limit <= dt < 2 * limit + 5.0
        with pytest.raises(gpu.LqcdError) as e:
            c.selftest_resident_wait(0.0)
        assert e.value.status == gpu.LQCD_EINVAL
        x1, i1 = c.mscg_solve(0.05, [1e-3, 0.1], 1e-10, b)
        assert i1["kernel_launches"] < i1["iters"]
        assert np.array_equal(x0, x1) and max(i1["true_resid"]) <= 1e-10
