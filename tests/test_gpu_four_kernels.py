"""The four kernels of a solver iteration on small lattices, which by default run
many iterations per launch instead: contexts with pdl = 1 take the four kernels
at every size.

* Staged against per-thread stencils, packed against solo, up to the 64 jobs
  whose mask the persistent finalisers keep in 64 bits (one K3 block per job
  forms its shifted coefficients): bitwise.
* Persistent reductions against one block per tile (read once per process, so in
  child processes), FP64, hybrid, FP16 and packed: bitwise.
* The bounds-checked library: no index out of range, and the bits of the
  default library's resident iteration.
* The resident iteration itself, every storage format and packed batches,
  against the four kernels, with the launches counted: it did run."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1701_00426_gb300 import inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FORMATS = {"fp64": {}, "mixed_12r": dict(prec=1, recon=12, fp64_until=1e-2),
           "fp32_18r": dict(prec=1, recon=18, fp64_until=0.0), "fp16": dict(prec=2, recon=12, fp64_until=0.0)}


def solve(gpu, dims, n_shift, **opts):
    with gpu.Context(dims, **opts) as c:
        c.links_upload(inputs.random_links(dims, seed=170))
        return c.mscg_solve(0.05, inputs.log_shifts(n_shift), 1e-10, inputs.gaussian_field(dims, k=17))


def packed(gpu, sizes, n_shift, **opts):
    ctxs = []
    for k, d in enumerate(sizes):
        ctxs.append(gpu.Context(d, **opts))
        ctxs[-1].links_upload(inputs.random_links(d, seed=171 + k % 5))
    n = len(sizes)
    r = gpu.mscg_solve_packed(ctxs, [0.05] * n, [inputs.log_shifts(n_shift)] * n, [1e-10] * n,
                              [inputs.gaussian_field(d, k=k % 7) for k, d in enumerate(sizes)])
    for c in ctxs:
        c.close()
    return r


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 6, 8, 10), (12, 12, 12, 12)])
@pytest.mark.parametrize("opts", [{}, dict(prec=1, recon=12, fp64_until=1e-3)], ids=["fp64", "hybrid"])
def test_staged_equals_per_thread(gpu, dims, opts):
    (x1, i1), (x0, i0) = (solve(gpu, dims, 8, staged=s, pdl=1, **opts) for s in (1, 0))
    assert i1["kernel_launches"] >= 4 * i1["iters"]
    assert np.array_equal(x1, x0) and i1["iters"] == i0["iters"] and i1["true_resid"] == i0["true_resid"]


@pytest.mark.parametrize("n", [4, 64])
def test_packed_equals_solo(gpu, n):
    sizes = ([(4, 4, 4, 4), (8, 8, 8, 8), (12, 12, 12, 12), (4, 6, 8, 10)] if n == 4 else
             [(6, 6, 6, 6) if k % 4 == 0 else (4, 4, 4, 4) for k in range(n)])   # 3 tiles or 1, ragged
    xs, infos = packed(gpu, sizes, 3, pdl=1)
    for k, d in enumerate(sizes):
        with gpu.Context(d, staged=0, pdl=1) as c:
            c.links_upload(inputs.random_links(d, seed=171 + k % 5))
            x, info = c.mscg_solve(0.05, inputs.log_shifts(3), 1e-10, inputs.gaussian_field(d, k=k % 7))
        assert np.array_equal(xs[k], x), k
        assert infos[k]["iters"] == info["iters"] and max(infos[k]["true_resid"]) <= 1e-10


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("dims", [(4, 6, 8, 10), (16, 16, 16, 16), (16, 18, 18, 20)])
def test_resident_ran_and_equals_four_kernels(gpu, fmt, dims):
    if fmt == "fp64" and int(np.prod(dims)) // 2 > 40960:
        dims = (16, 16, 16, 20)   # the largest of the double-float range
    (a, ia), (b, ib) = (solve(gpu, dims, 3, pdl=p, **FORMATS[fmt]) for p in (0, 1))
    assert np.array_equal(a, b) and ia["iters"] == ib["iters"] and ia["true_resid"] == ib["true_resid"]
    # four launches per multi-shift iteration against one per 256 of them; the
    # refinement's are the same
    assert ib["kernel_launches"] - ia["kernel_launches"] >= 3 * ia["iters"], "the resident iteration did not run"


@pytest.mark.parametrize("fmt", list(FORMATS))
def test_resident_packed_equals_four_kernels(gpu, fmt):
    sizes = [(2, 2, 2, 2), (8, 8, 8, 8), (4, 6, 8, 10), (12, 12, 12, 12), (6, 6, 6, 6)]
    (a, ia), (b, ib) = (packed(gpu, sizes, 4, pdl=p, **FORMATS[fmt]) for p in (0, 1))
    for k in range(len(sizes)):
        assert np.array_equal(a[k], b[k]), k
        assert ia[k]["iters"] == ib[k]["iters"] and ia[k]["true_resid"] == ib[k]["true_resid"]


CHILD = r'''
import sys, numpy as np
sys.path.insert(0, sys.argv[1])
from paper_1701_00426_gb300 import build, inputs, lqcd
checked, pdl = sys.argv[3] == "1", int(sys.argv[4])
lqcd.load(build.build(checked=checked))
out = {}
formats = {"fp64": {}, "per_thread": dict(staged=0), "hybrid": dict(prec=1, recon=12, fp64_until=1e-3),
           "fp32_18r": dict(prec=1, recon=18, fp64_until=1e-3), "fp16": dict(prec=2, recon=12, fp64_until=0.0)}
for dims in ((2, 2, 2, 2), (4, 6, 8, 10), (12, 12, 12, 12)):
    for name, opts in formats.items():
        with lqcd.Context(dims, pdl=pdl, **opts) as c:
            c.links_upload(inputs.random_links(dims, seed=172))
            x, info = c.mscg_solve(0.05, inputs.log_shifts(6), 1e-10, inputs.gaussian_field(dims, k=18))
        out[f"{name} {dims}"] = x
        out[f"{name} {dims} info"] = np.array([info["iters"], info["refine_iters"], info["reliable_updates"]])
sizes = [(4, 4, 4, 4), (8, 8, 8, 8), (6, 6, 6, 6)]
for name, opts in formats.items():
    ctxs = []
    for k, d in enumerate(sizes):
        ctxs.append(lqcd.Context(d, pdl=pdl, **opts))
        ctxs[-1].links_upload(inputs.random_links(d, seed=173 + k))
    xs, _ = lqcd.mscg_solve_packed(ctxs, [0.05] * 3, [inputs.log_shifts(6)] * 3, [1e-10] * 3,
                                   [inputs.gaussian_field(d, k=k) for k, d in enumerate(sizes)])
    for k, x in enumerate(xs):
        out[f"{name} packed {k}"] = x
    for c in ctxs:
        c.close()
np.savez(sys.argv[2], **out)
print("bounds", lqcd.bounds_errors() if checked else 0)
'''


def child(tmp_path, tag, checked=0, pdl=1, persist="1"):
    script, npz = tmp_path / "child.py", tmp_path / f"{tag}.npz"
    script.write_text(CHILD)
    r = subprocess.run([sys.executable, str(script), ROOT, str(npz), str(checked), str(pdl)],
                       env=dict(os.environ, LQCD_PERSIST_REDUCTIONS=persist), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    assert r.stdout.strip().splitlines()[-1] == "bounds 0"
    return np.load(npz)


def test_reductions_and_bounds_checked_build(gpu, tmp_path):
    ref = child(tmp_path, "resident", pdl=0)
    for tag, kw in [("four kernels", {}), ("one block per tile", dict(persist="0")), ("checked", dict(checked=1)),
                    ("checked, one block per tile", dict(checked=1, persist="0"))]:
        got = child(tmp_path, tag, **kw)
        assert sorted(got.files) == sorted(ref.files)
        for k in ref.files:
            assert np.array_equal(got[k], ref[k]), (tag, k)
