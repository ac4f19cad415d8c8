"""The batched CG's reductions and kept workspace at the edges of their ranges:
batches that are and are not a multiple of the fields of a 16-byte access, and
lattices whose last block is ragged or smaller than one block.

The FP64 true residual of every field is recomputed by the oracle: bar tol, as
the solver tests its own.  A repeated call takes the kept workspace and graph:
the same bits, and no device memory beyond that of the first call."""
import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 5, 16])
@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (4, 6, 10, 2), (6, 8, 4, 14)])
def test_batched_cg_ragged_and_repeated(gpu, orc, n, dims):
    U = inputs.random_links(dims, seed=140)
    b = np.stack([inputs.gaussian_field(dims, k=j) for j in range(n)])
    other = np.stack([inputs.gaussian_field(dims, k=j + 20) for j in range(max(1, n - 1))])
    with gpu.Context(dims, prec=gpu.PREC_FP32, recon=12) as c:
        c.links_upload(U)
        x, infos = c.cg_solve_mrhs(0.1, 0.0, 1e-10, b)
        held = c.device_bytes()
        c.cg_solve_mrhs(0.2, 0.0, 1e-8, other)     # another batch through the same workspace
        x2, infos2 = c.cg_solve_mrhs(0.1, 0.0, 1e-10, b)
        assert c.device_bytes() == held
    assert np.array_equal(x, x2) and [i["iters"] for i in infos] == [i["iters"] for i in infos2]
    for j in range(n):
        assert orc.true_residual(dims, U, 0.1, 0.0, b[j], x[j]) <= 1e-10
