"""The exponential of the link update and of stout smearing (a Taylor series
reduced by Cayley-Hamilton) and its derivative in the force chain, over the
branches of their argument's size: the three degrees and one or more
halvings, zero and degenerate eigenvalues.

Against the FP64 oracle (a matrix Taylor series).  Bars: 1e-13 relative, times
the growth of a rounding error under k squarings, 2^k <= 2 r, where r ~ 3 eps
is the largest eigenvalue of eps H (r <= 6 rho for a stout level); 1e-12 for the
force chain, which is linear in the derivative and in 1 + 12 rho staples."""
import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("eps", [0.0, 1e-4, 0.02, 0.07, 0.3, 1.5, 6.0])
def test_link_update_over_sizes_of_the_argument(gpu, orc, prec, eps):
    dims = (4, 2, 4, 6)
    U = inputs.random_links(dims, seed=130)
    H = inputs.random_momenta(dims, seed=131)
    H[0, :8] = 0.0                                        # the identity
    H[1, :8] = np.diag([1.0, 1.0, -2.0])                  # two equal eigenvalues
    H[2, :8] = np.diag([1.0, 1.0 + 1e-9, -2.0 - 1e-9])    # nearly equal
    ref = orc.link_update(dims, U, H, eps)
    with gpu.Context(dims) as c:
        c.links_upload(U)
        c.mom_upload(H)
        c.gauge_link_update(eps, prec)
        got = c.links_download()
    assert rel(got, ref) <= 1e-13 * max(1.0, 6.0 * eps)
    assert np.array_equal(got[0, :8], U[0, :8]) or rel(got[0, :8], U[0, :8]) <= 1e-14


@pytest.mark.parametrize("rho,levels", [(0.0, 1), (0.003, 1), (0.05, 1), (0.5, 1), (1.5, 1), (0.15, 4)])
def test_stout_over_sizes_of_rho(gpu, orc, rho, levels):
    dims = (4, 2, 4, 6)
    U = inputs.random_links(dims, seed=132)
    F = inputs.random_momenta(dims, seed=133)
    with gpu.Context(dims) as c:
        c.links_upload(U)
        c.stout_smear(rho, levels)
        got = c.links_download()
        force = c.stout_force(F)
    grow = max(1.0, 12.0 * rho)
    assert rel(got, orc.stout_smear(dims, U, rho, levels)) <= 1e-13 * grow * levels
    assert rel(force, orc.stout_force(dims, U, rho, F, levels)) <= 1e-12 * (1.0 + 12.0 * rho) ** levels


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 4, 4), (4, 4, 6, 10)])
@pytest.mark.parametrize("fail", [0, 1])
def test_momentum_update_from_stored_staples(gpu, orc, prec, dims, fail):
    """The force from stored plaquette staples against the oracle's paths: wrapping
    sides of 2, a ragged last block, all six planes at once and (first scratch
    allocation refused) three at a time.  Bars as for the momentum update:
    1e-12 double-float, 1e-13 native."""
    U = inputs.random_links(dims, seed=134)
    H = inputs.random_momenta(dims, seed=135)
    eps, beta = 0.03, 5.52
    ref = orc.mom_update(dims, U, H, beta, eps)
    with gpu.Context(dims) as c:
        c.links_upload(U)
        c.mom_upload(H)
        gpu.inject_alloc_failure(fail)
        try:
            c.gauge_mom_update(beta, eps, prec)
        finally:
            gpu.inject_alloc_failure(0)
        got = c.mom_download()
    assert rel(got - H, ref - H) <= (1e-12 if prec == 0 else 1e-13)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 4, 4), (4, 4, 6, 10), (8, 2, 6, 12)])
def test_fp32_momentum_update(gpu, orc, dims):
    """The FP32 force, its links through the per-thread ring, against the FP64
    oracle: wrapping sides of 2 (a double step returns to the site) and ragged last
    blocks.  Bar: five products in a row, each 6 roundings of 2^-24 = 6e-8 per
    entry, 2e-6 at worst; H itself, rounded to FP32 before and after, adds 2 x
    6e-8 of |H| against |eps F| >= 0.1 |H|, 1.2e-6."""
    U = inputs.random_links(dims, seed=136)
    H = inputs.random_momenta(dims, seed=137)
    eps, beta = 0.5, 5.52
    ref = orc.mom_update(dims, U, H, beta, eps)
    assert np.linalg.norm(ref - H) >= 0.1 * np.linalg.norm(H)
    with gpu.Context(dims) as c:
        c.links_upload(U)
        c.mom_upload(H)
        c.gauge_mom_update(beta, eps, 1)
        got = c.mom_download()
    assert rel(got - H, ref - H) <= 3.5e-6
