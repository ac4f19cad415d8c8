"""The FP64 momentum update does not depend on how much device memory is free:
with the scratch for the stored plaquette staples refused, every thread forms
the staples itself, with the same bits.  And its passes over the planes, as
many as the lattice's size asks for (6, 3, 2 or 1 planes each), give the force.

Passes: a small lattice's links and momenta repeated periodically over a large
one have the small lattice's force, which the oracle computes; bars as for the
momentum update, 1e-12 double-float, 1e-13 native."""
import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 4, 4), (4, 4, 6, 10), (8, 8, 8, 8)])
def test_bits_do_not_depend_on_the_scratch(gpu, prec, dims):
    U = inputs.random_links(dims, seed=150)
    H = inputs.random_momenta(dims, seed=151)

    def run(fail, calls):
        with gpu.Context(dims) as c:
            c.links_upload(U)
            c.mom_upload(H)
            before = c.device_bytes()
            for f in calls:
                gpu.inject_alloc_failure(fail)
                try:
                    f(c)
                finally:
                    gpu.inject_alloc_failure(0)
            return c.mom_download(), c.links_download(), c.device_bytes() - before

    for calls in ([lambda c: c.gauge_mom_update(5.52, 0.03, prec)], [lambda c: c.gauge_md_steps(5.52, 0.02, 3, prec)],
                  [lambda c: c.gauge_mom_update(5.52, 0.03, prec)] * 2):
        stored, refused = run(0, calls), run(1, calls)
        assert np.array_equal(stored[0], refused[0]) and np.array_equal(stored[1], refused[1])
        assert stored[2] > 0 and refused[2] == 0


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("dims,planes", [((8, 8, 8, 8), 6), ((32, 32, 32, 32), 3), ((32, 32, 32, 40), 2), ((32, 32, 40, 48), 1)])
def test_passes_over_the_planes(gpu, orc, prec, dims, planes):
    tile = (4, 4, 4, 4)
    u, h = inputs.random_links(tile, seed=152), inputs.random_momenta(tile, seed=153)
    eps, beta = 0.03, 5.52
    want = orc.mom_update(tile, u, h, beta, eps) - h
    rep = [dims[3 - k] // tile[3 - k] for k in range(4)]   # the first coordinate is the fastest

    def spread(f):
        return np.tile(f.reshape((4,) + tile[::-1] + (3, 3)), [1] + rep + [1, 1]).reshape(4, -1, 3, 3)

    V = int(np.prod(dims))
    with gpu.Context(dims) as c:
        c.links_upload(spread(u))
        c.mom_upload(spread(h))
        before = c.device_bytes()
        c.gauge_mom_update(beta, eps, prec)
        assert c.device_bytes() - before == planes * 1152 * (V // 2)
        got = c.mom_download() - spread(h)
    assert rel(got, spread(want)) <= (1e-12 if prec == 0 else 1e-13)


def test_scratch_is_given_back_to_calls_that_need_memory(gpu):
    """An allocation that fails while the context holds the scratch is tried again
    without it; the momentum update then takes it anew, with the same bits."""
    dims = (8, 8, 8, 8)
    H = inputs.random_momenta(dims, seed=154)
    b = inputs.gaussian_field(dims, k=9)
    scratch = 6 * 1152 * 8 ** 4 // 2
    with gpu.Context(dims) as c:
        c.links_upload(inputs.random_links(dims, seed=154))
        c.mom_upload(H)
        c.gauge_mom_update(5.52, 0.03)
        first = c.mom_download()
        held = c.device_bytes()
        gpu.inject_alloc_failure(1)
        try:
            x, info = c.mscg_solve(0.1, [1e-3], 1e-10, b)
            assert c.device_bytes() < held                  # given back
            gpu.inject_alloc_failure(1)
            with pytest.raises(gpu.LqcdError) as e:         # nothing left to give
                c.mscg_solve(0.1, inputs.log_shifts(8), 1e-10, b)
            assert e.value.status == gpu.LQCD_ENOMEM
        finally:
            gpu.inject_alloc_failure(0)
        assert max(info["true_resid"]) <= 1e-10
        before = c.device_bytes()
        c.mom_upload(H)
        c.gauge_mom_update(5.52, 0.03)
        assert c.device_bytes() == before + scratch
        assert np.array_equal(c.mom_download(), first)
