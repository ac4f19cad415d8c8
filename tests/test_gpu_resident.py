"""The resident iteration of small lattices (many iterations in one cooperative
launch) against the four-kernel iteration, which a context with pdl = 1 runs.

Both do the same arithmetic in the same order, so the bar is bitwise equality
of the solutions, the iteration counts and the true residuals.  Lattices: one
partial sub-tile (2^4: 8 sites), partial last sub-tiles, one block, several
sub-tiles per block, more than 32 tiles (totals formed by several warps), the
largest lattices of each precision's range and ones just beyond it; 1, 3 and
32 shifts; packed solves of uneven lattices."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FORMATS = {"fp64": {}, "mixed_12r": dict(prec=1, recon=12, fp64_until=1e-2),
           "fp32_18r": dict(prec=1, recon=18, fp64_until=0.0), "fp16": dict(prec=2, recon=12)}


def solve(lqcd, inputs, dims, opts, pdl, n_shift, U, b):
    with lqcd.Context(dims, pdl=pdl, **opts) as c:
        c.links_upload(U)
        x, info = c.mscg_solve(0.1, inputs.log_shifts(n_shift), 1e-9, b)
        launches = info["kernel_launches"]
        return x, [info["iters"], info["refine_iters"], info["reliable_updates"], info["shift_iters"]], \
            info["true_resid"], launches


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("dims,n_shift", [((2, 2, 2, 2), 1), ((4, 4, 4, 4), 3), ((4, 6, 8, 10), 32), ((6, 6, 10, 8), 1),
                                          ((8, 8, 8, 8), 3), ((12, 10, 14, 12), 3), ((16, 16, 16, 16), 3),
                                          ((16, 16, 16, 20), 1), ((18, 16, 18, 20), 3), ((18, 18, 18, 20), 1)])
def test_resident_bitwise_equal_to_four_kernels(gpu, fmt, dims, n_shift):
    from paper_1701_00426_gb300 import inputs
    U = inputs.random_links(dims, seed=31)
    b = inputs.gaussian_field(dims, k=5)
    a = solve(gpu, inputs, dims, FORMATS[fmt], 0, n_shift, U, b)
    r = solve(gpu, inputs, dims, FORMATS[fmt], 1, n_shift, U, b)
    assert np.array_equal(a[0], r[0])
    assert a[1] == r[1] and a[2] == r[2]
    assert max(a[2]) <= 1e-9
    if fmt == "fp64" and int(np.prod(dims)) // 2 <= 40960:
        assert a[3] < r[3], "the resident iteration did not run"


def test_resident_packed_equals_solo(gpu):
    from paper_1701_00426_gb300 import inputs
    sizes = [(2, 2, 2, 2), (8, 8, 8, 8), (4, 6, 8, 10), (12, 12, 12, 12)]
    ctxs, bs, solo = [], [], []
    for k, d in enumerate(sizes):
        c = gpu.Context(d)
        c.links_upload(inputs.random_links(d, seed=90 + k))
        ctxs.append(c)
        bs.append(inputs.gaussian_field(d, k=k))
        solo.append(c.mscg_solve(0.1, inputs.log_shifts(k + 1), 1e-9, bs[k]))
    xs, infos = gpu.mscg_solve_packed(ctxs, [0.1] * 4, [inputs.log_shifts(k + 1) for k in range(4)], [1e-9] * 4, bs)
    for k in range(4):
        assert np.array_equal(xs[k], solo[k][0])
        assert infos[k]["iters"] == solo[k][1]["iters"]
    for c in ctxs:
        c.close()
