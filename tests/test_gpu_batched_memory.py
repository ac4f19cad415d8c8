"""The batched CG where there is no room for all fields' FP64 residuals at once:
it forms them one at a time, with the same bits.  The k-th device allocation of
the call is refused for every k in turn; the one refusal that the call can do
without leaves (n - 1) fields less on the device, every other one is LQCD_ENOMEM
and leaves a context that solves."""
import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n", [((4, 6, 10, 2), 3), ((8, 8, 8, 8), 16)])
def test_refused_allocations(gpu, orc, dims, n):
    U = inputs.random_links(dims, seed=160)
    b = np.stack([inputs.gaussian_field(dims, k=j) for j in range(n)])
    field = 3 * int(np.prod(dims)) // 2 * 16

    def run(k):
        with gpu.Context(dims, prec=gpu.PREC_FP32, recon=12) as c:
            c.links_upload(U)
            gpu.inject_alloc_failure(k)
            try:
                x, infos = c.cg_solve_mrhs(0.05, 0.0, 1e-11, b)
                return x, [(i["iters"], i["reliable_updates"], i["true_resid"]) for i in infos], c.device_bytes()
            except gpu.LqcdError as e:
                assert e.status == gpu.LQCD_ENOMEM
            finally:
                gpu.inject_alloc_failure(0)
            return None, c.cg_solve_mrhs(0.05, 0.0, 1e-11, b)[0], 0

    x0, i0, held = run(0)
    assert max(orc.true_residual(dims, U, 0.05, 0.0, b[j], x0[j]) for j in range(n)) <= 1e-11
    assert max(i[1] for i in i0) > 0, "no restart was tested"
    without = 0
    for k in range(1, 12):
        x, i, bytes_held = run(k)
        if x is None:
            assert np.array_equal(i, x0)
            continue
        assert np.array_equal(x, x0) and i == i0
        without += bytes_held == held - (n - 1) * field
    assert without == 1
