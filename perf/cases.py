"""Performance cases: what a lattice-QCD program has this library do.

Each case is one call, or the short run of calls, that such a program makes
through the public binding (``paper_1701_00426_gb300.lqcd``), on the seeded
synthetic inputs the repository uses elsewhere (hot random SU(3) links,
Gaussian sources, Gaussian momenta), drawn here on the GPU.

Kinds (``case["kind"]``) and what they stand for:

deo        D_oe, then D_eo of its result: one hop to the odd sites and back,
           the operator every measurement and solver applies.  Options:
           the arithmetic (FP64 with 18- or 12-real links, native FP64, FP32
           with 18- or 12-real links, FP16 links).
mrhs       the same pair on 1..16 fields that share the links (FP32).
solve      a multi-shift solve on device spinors: the pseudofermion heatbath,
           action and force of the RHMC; 1..16 shifts, FP64 or mixed precision.
cg_mrhs    a batched CG on several sources (propagators), through the host call.
packed     independent multi-shift solves on lattices of different sizes in one
           call (host buffers), as a parameter scan or a solve service has them.
gauge_md   a trajectory's gauge updates: n steps of the tree-level Symanzik
           force and the link update, then the moved links and momenta on the
           host.
stout      smearing of the fermion links, the smeared links on the host, and
           the chain of a force on them back to the thin links.
"""
import math

import numpy as np
import torch

from paper_1701_00426_gb300 import lqcd

FP64, FP32, FP16, NATIVE = lqcd.PREC_FP64, lqcd.PREC_FP32, lqcd.PREC_FP16, lqcd.PREC_FP64_NATIVE
BETA = 5.52          # gauge coupling of the workloads
RHO = 0.15           # stout weight
C0, C1 = 5.0 / 3.0, -1.0 / 12.0
LAMBDA_MAX = 7.4     # effective largest eigenvalue of -D_eo D_oe on hot links, for iteration counts


def _case(kind, dims, name=None, **kw):
    c = {"kind": kind, "n0": dims[0], "n1": dims[1], "n2": dims[2], "n3": dims[3], **kw}
    if name:
        c["name"] = name
    return c


def listed():
    c8, c16, c24, c32 = ((n,) * 4 for n in (8, 16, 24, 32))
    return [
        # the smallest operator call: a test lattice, where latency counts
        _case("deo", c8, "deo_fp64_8", prec=FP64, recon=18),
        # the operator at a production size
        _case("deo", c32, "deo_fp64_32", prec=FP64, recon=18),
        # 16 sources of a propagator calculation sharing one configuration
        _case("mrhs", c24, "mrhs16_fp32_24", n=16, recon=12, layout=1),
        # single-shift FP64 CG on a test lattice
        _case("solve", c8, "cg_fp64_8", prec=FP64, recon=18, n_shift=1, mass=0.1, tol=1e-10),
        # the RHMC's 15-pole solve on a small, an ordinary and a large lattice
        _case("solve", c16, "mscg_fp64_16", prec=FP64, recon=18, n_shift=15, mass=0.01, tol=1e-10),
        _case("solve", c24, "mscg_mixed_24", prec=FP32, recon=12, n_shift=15, mass=0.01, tol=1e-10),
        _case("solve", c32, "mscg_fp64_32", prec=FP64, recon=18, n_shift=15, mass=0.01, tol=1e-10),
        # propagators of 16 sources
        _case("cg_mrhs", c24, "cg_mrhs16_24", n=16, recon=12, mass=0.1, tol=1e-10),
        # four lattices of uneven size in one call
        _case("packed", c8, "packed_8_12_16_20", count=4, step=4, prec=FP64, n_shift=4, mass=0.05, tol=1e-10),
        # gauge updates of a trajectory in FP64 and, on a larger lattice, in FP32
        _case("gauge_md", c16, "gauge_md_fp64_16", prec=FP64, steps=20, eps=0.01),
        _case("gauge_md", c24, "gauge_md_fp32_24", prec=FP32, steps=40, eps=0.01),
        # two stout levels and their force chain
        _case("stout", c16, "stout2_16", levels=2),
    ]


# ------------------------------------------------------------------ drawn cases
def _dims(rng, lo, hi):
    """Even sides with a volume between lo^4 and hi^4 (log-uniform), rarely equal."""
    while True:
        side = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        d = [max(4, 2 * round(0.5 * side * math.exp(rng.uniform(-0.4, 0.4)))) for _ in range(4)]
        v = math.prod(d)
        if lo ** 4 <= v <= hi ** 4 and max(d) <= 48:
            return d


def draw(rng):
    kind = rng.choice(["deo", "mrhs", "solve", "solve", "cg_mrhs", "packed", "gauge_md", "stout"])
    if kind == "deo":
        prec, recon = rng.choice([(FP64, 18), (FP64, 18), (FP64, 12), (NATIVE, 18), (FP32, 18), (FP32, 12), (FP16, 12)])
        return _case(kind, _dims(rng, 6, 32), prec=prec, recon=recon)
    if kind == "mrhs":
        return _case(kind, _dims(rng, 8, 24), n=rng.randint(1, 16), recon=rng.choice([12, 18]), layout=rng.choice([0, 1]))
    if kind == "solve":
        prec, recon = rng.choice([(FP64, 18), (FP64, 18), (FP32, 12), (FP32, 18)])
        return _case(kind, _dims(rng, 6, 24), prec=prec, recon=recon, n_shift=rng.randint(1, 16),
                     mass=rng.choice([0.01, 0.02, 0.05, 0.1]), tol=rng.choice([1e-8, 1e-10]))
    if kind == "cg_mrhs":
        return _case(kind, _dims(rng, 8, 24), n=rng.randint(2, 16), recon=rng.choice([12, 18]),
                     mass=rng.choice([0.05, 0.1, 0.2]), tol=rng.choice([1e-8, 1e-10]))
    if kind == "packed":
        d = _dims(rng, 6, 10)
        return _case(kind, d, count=rng.randint(2, 4), step=rng.choice([2, 4]), prec=FP64,
                     n_shift=rng.randint(1, 8), mass=rng.choice([0.05, 0.1]), tol=rng.choice([1e-8, 1e-10]))
    if kind == "gauge_md":
        prec = rng.choice([FP64, FP64, FP32, NATIVE])
        steps = rng.randint(4, 10) if prec == NATIVE else rng.randint(10, 40)
        return _case(kind, _dims(rng, 8, 20), prec=prec, steps=steps, eps=rng.choice([0.005, 0.01, 0.02]))
    return _case(kind, _dims(rng, 6, 18), levels=rng.randint(1, 3))


# ------------------------------------------------------------------ inputs
def _sides(case):
    return tuple(int(case[k]) for k in ("n0", "n1", "n2", "n3"))


def _packed_dims(case):
    """Lattice k of a packed call is k * step longer in every direction."""
    return [tuple(n + k * case["step"] for n in _sides(case)) for k in range(case["count"])]


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + 7919 * stream + 1701) % (1 << 62))


def _normal(shape, gen):
    """Complex N(0,1) real and imaginary parts."""
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=gen))


def _links(dims, seed, stream=0):
    """Hot SU(3) links [4, V, 3, 3] complex128 on the GPU: rows of Gaussian
    matrices orthonormalised (two passes), third row conj(r0 x r1)."""
    a = _normal((4, math.prod(dims), 2, 3), _gen(seed, stream))
    r0, r1 = a[..., 0, :], a[..., 1, :]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    for _ in range(2):
        r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], dim=-2)


def _hermitian(dims, seed, stream):
    """Traceless Hermitian Gaussian matrices [4, V, 3, 3], density exp(-Tr H^2 / 2)."""
    a = _normal((4, math.prod(dims), 3, 3), _gen(seed, stream)) / math.sqrt(2.0)
    h = 0.5 * (a + a.mH)
    tr = torch.diagonal(h, dim1=-2, dim2=-1).real.sum(-1) / 3.0
    return h - tr[..., None, None] * torch.eye(3, dtype=h.dtype, device=h.device)


def _shifts(case):
    return np.logspace(-5.0, 2.0, case["n_shift"]) if case["n_shift"] > 1 else np.array([0.0])


def _host(t):
    return np.ascontiguousarray(t.cpu().numpy())


def _spinor_dtype(prec):
    return torch.complex128 if prec in (FP64, NATIVE) else torch.complex64


def _source(case, seed):
    """The case's input field(s) on the GPU, complex128, [..., Vh, 3] or the device layout."""
    kind, dims = case["kind"], _sides(case)
    vh = math.prod(dims) // 2
    if kind in ("deo", "solve"):
        return _normal((3, vh), _gen(seed, 1))
    if kind == "mrhs":
        shape = (3, vh, case["n"]) if case["layout"] == 0 else (3, case["n"], vh)
        return _normal(shape, _gen(seed, 1))
    if kind == "cg_mrhs":
        return _normal((case["n"], vh, 3), _gen(seed, 1))
    if kind == "packed":
        return [_normal((math.prod(d) // 2, 3), _gen(seed, 10 + k)) for k, d in enumerate(_packed_dims(case))]
    return _hermitian(dims, seed, 1)


def prepare(case, seed):
    kind, dims = case["kind"], _sides(case)
    src = _source(case, seed)
    if kind == "packed":
        ctxs = []
        for k, d in enumerate(_packed_dims(case)):
            c = lqcd.Context(d, prec=case["prec"])
            c.links_upload(_host(_links(d, seed, 20 + k)))
            ctxs.append(c)
        return {"case": case, "ctxs": ctxs, "b": [_host(b) for b in src], "shifts": _shifts(case)}
    opts = {"prec": case["prec"], "recon": case["recon"]} if kind == "solve" else {}
    if kind == "cg_mrhs":
        opts = {"prec": FP32, "recon": case["recon"]}
    ctx = lqcd.Context(dims, **opts)
    ctx.links_upload(_host(_links(dims, seed)))
    s = {"case": case, "ctx": ctx}
    if kind in ("deo", "mrhs"):
        t = torch.complex64 if kind == "mrhs" else _spinor_dtype(case["prec"])
        s["in"] = src.to(t).contiguous()
        s["odd"], s["even"] = torch.empty_like(s["in"]), torch.empty_like(s["in"])
    elif kind == "solve":
        s["shifts"], s["b"] = _shifts(case), src
        s["x"] = torch.empty((case["n_shift"], *src.shape), dtype=src.dtype, device="cuda")
    elif kind == "cg_mrhs":
        s["b"] = _host(src)
    elif kind == "gauge_md":
        ctx.mom_upload(_host(src))
    else:
        s["F"] = _host(src)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "packed":
        n = case["count"]
        x, _ = lqcd.mscg_solve_packed(s["ctxs"], [case["mass"]] * n, [s["shifts"]] * n, [case["tol"]] * n, s["b"])
        return x
    ctx = s["ctx"]
    if kind == "deo":
        ctx.deo_apply_ex(1, case["prec"], case["recon"], s["in"], s["odd"])
        ctx.deo_apply_ex(0, case["prec"], case["recon"], s["odd"], s["even"])
        return s["odd"], s["even"]
    if kind == "mrhs":
        ctx.deo_apply_mrhs(1, case["n"], case["recon"], s["in"], s["odd"], layout=case["layout"])
        ctx.deo_apply_mrhs(0, case["n"], case["recon"], s["odd"], s["even"], layout=case["layout"])
        return s["odd"], s["even"]
    if kind == "solve":
        ctx.mscg_solve_dev(case["mass"], s["shifts"], case["tol"], s["b"], s["x"])
        return s["x"]
    if kind == "cg_mrhs":
        return ctx.cg_solve_mrhs(case["mass"], 0.0, case["tol"], s["b"])[0]
    if kind == "gauge_md":
        ctx.gauge_md_steps(BETA, case["eps"], case["steps"], prec=case["prec"])
        return ctx.links_download(), ctx.mom_download()
    ctx.stout_smear(RHO, case["levels"])
    smeared = ctx.links_download()
    thin = ctx.stout_force(s["F"])
    ctx.stout_restore()
    return smeared, thin


# ------------------------------------------------------------------ work
def _iterations(case, shift=0.0):
    """CG iterations to tol at mass^2 + shift, from the condition number."""
    kappa = LAMBDA_MAX / (case["mass"] ** 2 + shift)
    return max(4.0, 0.5 * math.sqrt(1.0 + kappa) * math.log(2.0 / case["tol"]))


def work(case):
    """Bytes and floating-point operations of one pass.  A hop term is 8
    link-vector products per site: 570 operations; a 3x3 product 198."""
    kind = case["kind"]
    v = math.prod(_sides(case))
    vh = v // 2
    if kind == "deo":
        spin = 48 if case["prec"] in (FP64, NATIVE) else 24
        real = {FP64: 8, NATIVE: 8, FP32: 4, FP16: 2}[case["prec"]]
        return {"bytes": 2 * vh * (8 * case["recon"] * real + 2 * spin), "flops": 2 * vh * 570}
    if kind == "mrhs":
        return {"bytes": 2 * vh * (8 * case["recon"] * 4 + 48 * case["n"]), "flops": 2 * vh * 570 * case["n"]}
    if kind in ("solve", "packed"):
        vhs = [math.prod(d) // 2 for d in _packed_dims(case)] if kind == "packed" else [vh]
        sh = _shifts(case)
        its = [_iterations(case, s) for s in sh]
        if case["prec"] == FP64:
            link, spin = 144, 48
        else:  # the bulk of a mixed solve runs on FP32 links and vectors
            link, spin = 4 * case["recon"], 24
        per_iter = 16 * link + 9 * spin          # two hop terms; r, q, t, p
        per_shift = 4 * spin                     # x_i and p_i read and written
        total = its[0] * per_iter + sum(its) * per_shift
        return {"bytes": sum(vhs) * total, "flops": sum(vhs) * (its[0] * 1200 + sum(its) * 36)}
    if kind == "cg_mrhs":
        it = _iterations(case)
        return {"bytes": vh * it * (16 * 4 * case["recon"] + case["n"] * 11 * 24), "flops": vh * it * case["n"] * 1260}
    if kind == "gauge_md":
        real = 4 if case["prec"] == FP32 else 8
        # force: per link 24 staple products with shared sides and U A; update: the exponential and E U
        return {"bytes": case["steps"] * v * 4 * real * (18 + 8 + 8 + 8 + 18 + 18) + v * 4 * 288,
                "flops": case["steps"] * v * 4 * 198 * 38}
    # smearing: 12 staple products, Q, the exponential, E U; chain: the same, the
    # derivative and 18 staple terms, per link and level
    return {"bytes": case["levels"] * v * 4 * (2 * 144 + 144 + 2 * 64) + v * 4 * 3 * 144,
            "flops": case["levels"] * v * 4 * 198 * (16 + 60)}


# ------------------------------------------------------------------ 64-bit reference
class _Hop:
    """D_oe / D_eo in complex128 torch: gathered neighbours times signed links."""

    def __init__(self, links, dims):
        n0, n1, n2, n3 = dims
        dev = links.device
        V = math.prod(dims)
        lex = torch.arange(V, device=dev)
        x = [lex % n0, lex // n0 % n1, lex // (n0 * n1) % n2, lex // (n0 * n1 * n2)]
        par = (x[0] + x[1] + x[2] + x[3]) & 1
        stride = [1, n0, n0 * n1, n0 * n1 * n2]
        self.W, self.idx = [], []
        for P in (0, 1):
            site = lex[par == P]                     # in the order of the half index lex // 2
            site = site[torch.argsort(site // 2)]
            W, idx = [], []
            for mu in range(4):
                eta = sum(x[:mu], torch.zeros_like(lex)) & 1
                s = 1.0 - 2.0 * eta.double()
                if mu == 3:
                    s = torch.where(x[3] == n3 - 1, -s, s)
                n = dims[mu]
                fwd = lex + torch.where(x[mu] == n - 1, -(n - 1), 1) * stride[mu]
                bwd = lex + torch.where(x[mu] == 0, n - 1, -1) * stride[mu]
                f, b = fwd[site], bwd[site]
                W += [0.5 * s[site, None, None] * links[mu, site], -0.5 * s[b, None, None] * links[mu, b].mH]
                idx += [f // 2, b // 2]
            self.W.append(torch.stack(W))            # [8, Vh, 3, 3]
            self.idx.append(torch.stack(idx))        # [8, Vh]

    def __call__(self, P, v):
        """v [n, Vh, 3] -> [n, Vh, 3] on the sites of parity P."""
        out = torch.zeros_like(v)
        for h in range(8):
            g = v[:, self.idx[P][h]]
            for b in range(3):
                out += self.W[P][h][None, :, :, b] * g[:, :, b, None]
        return out


def _exact_shifted(hop, mass, shifts, b):
    """(m^2 - D_eo D_oe + shift)^-1 b for every shift (n systems at once), b [n, Vh, 3]
    of one source repeated or of several; CG in complex128 to 1e-14 with restarts."""
    n = b.shape[0]
    a = torch.as_tensor(np.asarray(shifts) + mass * mass, device=b.device).reshape(n, 1, 1)
    A = lambda v: a * v - hop(0, hop(1, v))  # noqa: E731
    dot = lambda u, v: (torch.view_as_real(u) * torch.view_as_real(v)).sum((1, 2, 3)).reshape(n, 1, 1)  # noqa: E731
    x, bb = torch.zeros_like(b), dot(b, b)
    for _ in range(3):
        r = b - A(x)
        p, rr = r.clone(), dot(r, r)
        for k in range(20000):
            q = A(p)
            alpha = rr / dot(p, q).clamp_min(1e-300)
            x += alpha * p
            r -= alpha * q
            new = dot(r, r)
            p = r + (new / rr.clamp_min(1e-300)) * p
            rr = new
            if k % 50 == 49 and bool((rr <= 1e-28 * bb).all()):
                break
    return x


def _staple(U, mu, nu, sh):
    """Upper and lower staple of U_mu in the plane nu: x -> x+nu -> x+nu+mu -> x+mu, and mirrored."""
    up = U[nu] @ sh(U[mu], nu, 1) @ sh(U[nu], mu, 1).mH
    low = sh(U[nu].mH @ U[mu] @ sh(U[nu], mu, 1), nu, -1)
    return up, low


def _shifter(dims):
    n0, n1, n2, n3 = dims

    def sh(f, mu, d):
        """f(x + d mu) for f [V, ...]."""
        g = f.reshape(n3, n2, n1, n0, *f.shape[1:])
        return torch.roll(g, -d, 3 - mu).reshape(f.shape)
    return sh


def _exact_md(U, H, dims, eps, steps):
    """n steps of H -= eps F, U <- exp(i eps H) U in complex128."""
    sh = _shifter(dims)
    for _ in range(steps):
        F = []
        for mu in range(4):
            A = torch.zeros_like(U[mu])
            for nu in range(4):
                if nu == mu:
                    continue
                for s in (1, -1):
                    def step(d, sg, mu=mu, nu=nu):
                        """link of a step of sign sg in direction d as a field of its starting site"""
                        return U[d] if sg > 0 else sh(U[d], d, -1).mH

                    def path(moves, mu=mu, nu=nu):
                        """ordered product of steps starting at x + mu, as a field of x"""
                        M, pos = None, [(mu, 1)]
                        for d, sg in moves:
                            L = step(d, sg)
                            for dd, k in pos:
                                L = sh(L, dd, k)
                            M = L if M is None else M @ L
                            pos.append((d, sg))
                        return M
                    A += C0 * path([(nu, s), (mu, -1), (nu, -s)])
                    A += C1 * path([(mu, 1), (nu, s), (mu, -1), (mu, -1), (nu, -s)])
                    A += C1 * path([(nu, s), (mu, -1), (mu, -1), (nu, -s), (mu, 1)])
                    A += C1 * path([(nu, s), (nu, s), (mu, -1), (nu, -s), (nu, -s)])
            M = U[mu] @ A
            f = -1j * (BETA / 6.0) * (M - M.mH)
            tr = torch.diagonal(f, dim1=-2, dim2=-1).sum(-1) / 3.0
            F.append(f - tr[..., None, None] * torch.eye(3, dtype=f.dtype, device=f.device))
        H = H - eps * torch.stack(F)
        U = torch.linalg.matrix_exp(1j * eps * H) @ U
    return U, H


def _smear(U, dims):
    sh = _shifter(dims)
    out = []
    for mu in range(4):
        C = sum(sum(_staple(U, mu, nu, sh)) for nu in range(4) if nu != mu) * RHO
        om = C @ U[mu].mH
        q = 0.5j * (om.mH - om)
        tr = torch.diagonal(q, dim1=-2, dim2=-1).sum(-1) / 3.0
        q = q - tr[..., None, None] * torch.eye(3, dtype=q.dtype, device=q.device)
        out.append(torch.linalg.matrix_exp(1j * q) @ U[mu])
    return torch.stack(out)


def _exact_stout(U, F, dims, levels):
    """Smeared links, and the thin links' force from the gradient of the linear
    functional whose differential at the smeared links is Tr(X' F)."""
    U = U.clone().requires_grad_(True)
    W = U
    for _ in range(levels):
        W = _smear(W, dims)
    S = (-1j * W.detach().mH @ F @ W).diagonal(dim1=-2, dim2=-1).sum().real
    (g,) = torch.autograd.grad(S, U)
    m = 1j * U.detach() @ g.mH
    f = 0.5 * (m + m.mH)
    tr = torch.diagonal(f, dim1=-2, dim2=-1).sum(-1) / 3.0
    return W.detach(), f - tr[..., None, None] * torch.eye(3, dtype=f.dtype, device=f.device)


def exact(case, seed):
    kind, dims = case["kind"], _sides(case)
    src = _source(case, seed)
    if kind == "deo":
        hop = _Hop(_links(dims, seed), dims)
        v = src.to(_spinor_dtype(case["prec"])).to(torch.complex128).T[None]
        odd = hop(1, v)
        return odd[0].T.contiguous(), hop(0, odd)[0].T.contiguous()
    if kind == "mrhs":
        hop = _Hop(_links(dims, seed), dims)
        order = (2, 1, 0) if case["layout"] == 0 else (1, 2, 0)
        back = (2, 1, 0) if case["layout"] == 0 else (2, 0, 1)
        v = src.to(torch.complex64).to(torch.complex128).permute(*order).contiguous()
        odd = hop(1, v)
        return odd.permute(*back).contiguous(), hop(0, odd).permute(*back).contiguous()
    # solves: on the lattices where complex128 CG takes seconds
    if kind == "solve":
        n = case["n_shift"]
        if math.prod(dims) * n * _iterations(case) > 3e9:
            return None
        b = src.T[None].expand(n, -1, -1).contiguous()
        x = _exact_shifted(_Hop(_links(dims, seed), dims), case["mass"], _shifts(case), b)
        return x.permute(0, 2, 1).contiguous()
    if kind == "cg_mrhs":
        if math.prod(dims) * case["n"] * _iterations(case) > 3e9:
            return None
        x = _exact_shifted(_Hop(_links(dims, seed), dims), case["mass"], [0.0] * case["n"], src)
        return x.cpu().numpy()
    if kind == "packed":
        out = []
        for k, d in enumerate(_packed_dims(case)):
            n = case["n_shift"]
            if math.prod(d) * n * _iterations(case) > 1e9:
                out.append(None)
                continue
            hop = _Hop(_links(d, seed, 20 + k), d)
            out.append(_exact_shifted(hop, case["mass"], _shifts(case), src[k][None].expand(n, -1, -1).contiguous()).cpu().numpy())
        return out
    U = _links(dims, seed)
    if kind == "gauge_md":
        if math.prod(dims) * case["steps"] > 1.5e7:
            return None
        U, H = _exact_md(U, src, dims, case["eps"], case["steps"])
        return U.cpu().numpy(), H.cpu().numpy()
    W, F = _exact_stout(U, src, dims, case["levels"])
    return W.cpu().numpy(), F.cpu().numpy()
