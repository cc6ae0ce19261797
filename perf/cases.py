"""Performance cases of the gschur library: what its users run, through the public binding.

A case is a dict of plain values.  "kind" names the entry point, "dims" the lattice extents
(x0 fastest), "m0" the bare mass and "eps" the roughness of the gauge field U = exp(i eps H),
H a Gaussian traceless Hermitian matrix per link: the recipe of this repository's synthetic
fields (eps = 0.38 has the plaquette of the benchmark's beta = 5.4 field).  Sources are complex
Gaussian.  Solver tolerances lie below the 1e-10 of the benchmark, so that two correct solvers
agree in nine digits.
"""
import math

import numpy as np
import torch

import paper_0704_2341_gb300 as gs
from paper_0704_2341_gb300 import learned

PERMS = ((1, 0, 0), (2, 0, 0), (1, 0, 1), (2, 0, 1))    # P_I, P_II, P_I^T, P_II^T
TOL, INNER_TOL = 2e-12, 1e-13
C64, C128 = torch.complex64, torch.complex128


def listed():
    return [
        # One D x on the 8^4 lattice of the benchmark: the smallest call, as a user's own Krylov loop makes it.
        {"name": "wilson_8x4", "kind": "wilson", "dims": "8x8x8x8", "m0": -0.4, "eps": 0.38},
        # The same on the lattice of the batched workload: the largest FP64 vector work (0.64 GB a pass).
        {"name": "wilson_24x48", "kind": "wilson", "dims": "24x24x24x48", "m0": -0.35, "eps": 0.2},
        # The low-precision stencil at the largest lattice in use: the dslash bandwidth the benchmark reports.
        {"name": "stencil_f32_32x64", "kind": "stencil", "dims": "32x32x32x64", "m0": -0.38, "eps": 0.2,
         "type": 0, "dir": 0, "inverse": 0, "prec": "f32"},
        # D_rr in BF16 storage on the rest set of the batched workload, through its neighbour table.
        {"name": "stencil_bf16_rest_24x48", "kind": "stencil", "dims": "24x24x24x48", "m0": -0.35, "eps": 0.2,
         "type": 1, "dir": 0, "inverse": 0, "prec": "bf16"},
        # One application of S_bb with FP64 inner solve on 8^4: the operator itself, latency bound.
        {"name": "schur_apply_8x4", "kind": "schur_apply", "dims": "8x8x8x8", "m0": -0.4, "eps": 0.38,
         "type": 1, "dir": 0, "inverse": 0, "prec": "f64"},
        # S_bb of the mixed-precision workload: 16^3 x 32, Type II, FP32 inner solve.
        {"name": "schur_apply_f32_16x32", "kind": "schur_apply", "dims": "16x16x16x32", "m0": -0.3, "eps": 0.25,
         "type": 2, "dir": 0, "inverse": 0, "prec": "f32"},
        # The benchmark's step: the complete solves of the four permutations of one 8^4 field at once, FP64.
        {"name": "solve_batched_8x4", "kind": "batched", "dims": "8x8x8x8", "m0": -0.4, "eps": 0.38, "prec": "f64"},
        # Four sources on one 8^4 lattice sharing every launch, FP32 inner solves (the small lattices of the
        # batched workload).
        {"name": "solve_multi_8x4", "kind": "multi", "dims": "8x8x8x8", "m0": -0.35, "eps": 0.2,
         "type": 1, "dir": 0, "inverse": 0, "prec": "f32", "nrhs": 4},
        # Section 3's approximation of S_bb on a lattice of uneven extents and an inverse permutation.
        {"name": "reusken_ragged", "kind": "reusken", "dims": "18x14x10x22", "m0": -0.4, "eps": 0.38,
         "type": 2, "dir": 1, "inverse": 1},
        # The inner solve with the 24-channel network inside flexible GMRES.
        {"name": "learned_rr_16x32", "kind": "learned_rr", "dims": "16x16x16x32", "m0": -0.2, "eps": 0.2,
         "type": 1, "dir": 0, "inverse": 0},
        # One Adam step of that network on 8^4 with the batch its training uses: forward, backward, update.
        {"name": "train_8x4", "kind": "train", "dims": "8x8x8x8", "m0": -0.38, "eps": 0.2,
         "type": 1, "dir": 0, "inverse": 0, "batch": 4},
        # Section 4: BiCGStab on D preconditioned by the 3-level V-cycle (Type I inverse at both steps), 8^4.
        {"name": "vcycle_8x4", "kind": "vcycle", "dims": "8x8x8x8", "m0": -0.4, "eps": 0.38},
    ]


def _extents(rng, lo, hi, even):
    """Four extents with the volume spread over its logarithm in [lo, hi]."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        w = [math.exp(rng.uniform(-0.5, 0.5)) for _ in range(4)]
        s = (v / (w[0] * w[1] * w[2] * w[3])) ** 0.25
        L = [max(4, round(s * x)) for x in w]
        if even:
            L = [max(4, 2 * round(x / 2)) for x in L]
        n = L[0] * L[1] * L[2] * L[3]
        if lo <= n <= hi:
            return "x".join(str(x) for x in L)


def draw(rng):
    kind = rng.choice(("wilson", "wilson", "stencil", "stencil", "schur_apply", "schur_apply", "batched", "multi",
                       "reusken", "learned_rr", "train", "vcycle"))
    eps = round(rng.uniform(0.2, 0.38), 3)
    m0 = round(-rng.uniform(0.2, 0.35 + 0.8 * (eps - 0.2)), 3)        # rougher fields take a lighter bare mass
    ptype, mu, inv = rng.choice((1, 2)), 0, rng.choice((0, 0, 1))
    if ptype == 2:
        mu = rng.randrange(4)
    case = {"kind": kind, "m0": m0, "eps": eps}
    if kind == "wilson":
        return dict(case, dims=_extents(rng, 256, 663552, False))
    if kind == "stencil":
        whole = rng.random() < 0.4
        case["prec"] = rng.choice(("f32", "bf16"))
        if whole:
            return dict(case, dims=_extents(rng, 256, 2097152, False), type=0, dir=0, inverse=0)
        return dict(case, dims=_extents(rng, 256, 1048576, True), type=ptype, dir=mu, inverse=inv)
    case.update(type=ptype, dir=mu, inverse=inv)
    if kind == "schur_apply":
        prec = rng.choice(("f64", "f32", "bf16"))
        return dict(case, dims=_extents(rng, 256, 32768 if prec == "f64" else 262144, True), prec=prec)
    if kind == "reusken":
        return dict(case, dims=_extents(rng, 256, 262144, True))
    if kind == "multi":
        return dict(case, dims=_extents(rng, 256, 8192, True), prec=rng.choice(("f32", "bf16")),
                    nrhs=rng.choice((2, 3, 4, 6, 12)))
    if kind == "learned_rr":
        return dict(case, m0=-0.2, dims=_extents(rng, 1024, 131072, True))
    if kind == "train":
        return dict(case, dims=_extents(rng, 256, 4096, True), batch=rng.choice((1, 2, 3, 4)))
    for k in ("type", "dir", "inverse"):
        del case[k]
    if kind == "batched":
        return dict(case, dims=_extents(rng, 256, 8192, True), prec=rng.choice(("f64", "f32")))
    return dict(case, dims=rng.choice(("4x4x4x4", "8x4x4x8", "8x8x4x8", "8x8x8x4", "8x8x8x8", "8x8x8x12")))


# ---- inputs ---------------------------------------------------------------------------------------------

def _dims(case):
    return tuple(int(x) for x in case["dims"].split("x"))


def _volume(case):
    return math.prod(_dims(case))


def _generator(seed):
    return torch.Generator("cuda").manual_seed(1000003 * int(seed) + 17)


def _gaussian(gen, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=gen))


def _mm(a, b):
    return a[:, 0, None] * b[None, 0] + a[:, 1, None] * b[None, 1] + a[:, 2, None] * b[None, 2]


def _gauge(case, gen):
    """exp(i eps H) for every link, complex128 [V][4][3][3]; entry (i, j) of all links is one vector meanwhile."""
    n = 4 * _volume(case)
    a = _gaussian(gen, 3, 3, n)
    x = 0.5 * (a + a.transpose(0, 1).conj())
    trace = (x[0, 0] + x[1, 1] + x[2, 2]) / 3.0
    for i in range(3):
        x[i, i] -= trace
    x = x * (1j * case["eps"] / 16)
    del a
    u = torch.zeros_like(x)
    for i in range(3):
        u[i, i] = 1.0
    term = u.clone()
    for k in range(1, 15):
        term = _mm(term, x) / k
        u += term
    for _ in range(4):
        u = _mm(u, u)
    return u.permute(2, 0, 1).reshape(n // 4, 4, 3, 3).contiguous()


def _rest_and_coarse(case, ptype=None, mu=None, inv=None):
    """Sites of the coarse set and of the rest set, each in label order."""
    ptype = case["type"] if ptype is None else ptype
    mu = case["dir"] if mu is None else mu
    inv = case["inverse"] if inv is None else inv
    dims, V = _dims(case), _volume(case)
    if ptype == 0:
        return None, torch.arange(V, device="cuda")
    s, even = torch.arange(V, device="cuda"), []
    for L in dims:
        even.append(s % L % 2 == 0)
        s = s // L
    b = even[0] & even[1] & even[2] & even[3] if ptype == 1 else even[mu]
    p = torch.cat([b.nonzero().reshape(-1), (~b).nonzero().reshape(-1)])
    if inv:
        q = torch.empty_like(p)
        q[p] = torch.arange(V, device="cuda")
        p = q
    nb = int(b.sum())
    return p[:nb], p[nb:]


def _opts(case):
    prec = {"f64": gs.GS_F64, "f32": gs.GS_F32, "bf16": gs.GS_BF16}[case["prec"]]
    return gs.gs_default_opts(tol=TOL, inner_tol=INNER_TOL, inner_prec=prec)


def _context(case, U, stream=None):
    s = torch.cuda.current_stream() if stream is None else stream
    ctx = gs.Context(_dims(case), case["m0"], s.cuda_stream)
    ctx.set_gauge(U)
    return ctx


def _lowp_layout(x, prec):
    """The library's component-major layout of [n][24] reals: FP32 [6][n][4], BF16 [3][n][8]."""
    g = 8 if prec == "bf16" else 4
    return x.reshape(x.shape[0], 24 // g, g).transpose(0, 1).contiguous()


def _inputs(case, seed):
    """Gauge field and vectors of a case, in plain torch; the same for prepare() and exact()."""
    gen, kind, V = _generator(seed), case["kind"], _volume(case)
    U = _gauge(case, gen)
    if kind in ("wilson", "vcycle", "batched"):
        return U, _gaussian(gen, V, 12)
    if kind == "multi":
        return U, _gaussian(gen, case["nrhs"], V, 12)
    b, r = _rest_and_coarse(case)
    if kind == "stencil":
        x = torch.view_as_real(_gaussian(gen, r.numel(), 12)).reshape(-1, 24)
        return U, x.to(torch.bfloat16 if case["prec"] == "bf16" else torch.float32)
    if kind in ("schur_apply", "reusken"):
        return U, _gaussian(gen, b.numel(), 12)
    if kind == "learned_rr":
        return U, _gaussian(gen, r.numel(), 12)
    D = _Wilson(case, U)                                   # train: pairs (t = D_rr z, z)
    z = _gaussian(gen, case["batch"], r.numel(), 12)
    t = torch.stack([D.block(r, r, v) for v in z])
    return U, (t.to(C64).contiguous(), z.to(C64).contiguous())


def prepare(case, seed):
    kind = case["kind"]
    U, x = _inputs(case, seed)
    st = {"case": case, "x": x}
    if kind == "batched":
        st["streams"] = [torch.cuda.Stream() for _ in PERMS]
        torch.cuda.current_stream().synchronize()
        st["ctxs"] = [_context(case, U, s) for s in st["streams"]]
        st["out"] = [torch.empty_like(x) for _ in PERMS]
        st["problems"] = [{"ctx": c.handle, "type": t, "dir": m, "inverse": i, "nrhs": 1, "f": x, "x": y}
                          for c, (t, m, i), y in zip(st["ctxs"], PERMS, st["out"])]
        for s in st["streams"]:
            s.synchronize()
        st["opts"] = _opts(case)
        return st
    ctx = st["ctx"] = _context(case, U)
    if kind == "stencil":
        st["x"] = _lowp_layout(x, case["prec"])
        st["prec"] = gs.GS_BF16 if case["prec"] == "bf16" else gs.GS_F32
    if kind in ("learned_rr", "train"):
        net = st["net"] = gs.Net(24)
        for layer, w in enumerate(learned.identity_like_weights(24, case["m0"], 4)):
            net.set_weights(layer, w)
        if kind == "learned_rr":
            ctx.set_net(net)
            st["opts"] = learned.fgmres_net_opts(inner_tol=INNER_TOL, inner_restart=64, lowp_tol=1e-2)
    if kind == "vcycle":
        st["vc"] = gs.VCycle(ctx, [(1, 0, 1), (1, 0, 1)])
    if kind in ("schur_apply", "multi"):
        st["opts"] = _opts(case)
    if kind != "train":
        st["y"] = torch.empty_like(st["x"])
    return st


def run(st):
    case = st["case"]
    kind, x, ctx = case["kind"], st["x"], st.get("ctx")
    if kind == "batched":
        status, _ = gs.schur_solve_batched(st["problems"], st["opts"])
        if status != gs.GS_OK:
            raise RuntimeError("schur_solve_batched: status %d" % status)
        return st["out"]
    if kind == "wilson":
        ctx.wilson_apply(x, st["y"])
        return st["y"]
    if kind == "vcycle":
        ctx.solve_bicgstab(st["vc"], x, st["y"], tol=TOL)
        return st["y"]
    where = (case["type"], case["dir"], case["inverse"])
    if kind == "train":
        loss = st["net"].train_step(ctx.handle, *where, case["batch"], x[0], x[1], 1e-3)
        return [loss] + [st["net"].get(1, layer) for layer in range(3)]
    if kind == "stencil":
        ctx.wilson_apply_lowp(*where, st["prec"], x, st["y"])
    elif kind == "schur_apply":
        ctx.schur_apply(*where, x, st["y"], st["opts"])
    elif kind == "reusken":
        ctx.schur_apply_reusken(*where, x, st["y"])
    elif kind == "multi":
        ctx.schur_solve_multi(*where, case["nrhs"], x, st["y"], st["opts"])
    else:
        ctx.solve_rr(*where, x, st["y"], st["opts"])
    return st["y"]


# ---- what a pass cannot do without ----------------------------------------------------------------------

def work(case):
    """Bytes: links once, inputs once, outputs once.  Flops: 1368 a site of D (168 a hop, 48 on the diagonal);
    iterative solves count the operator applications that Gaussian sources on these fields need in FP64."""
    V, kind = _volume(case), case["kind"]
    D = 1368.0
    if kind == "wilson":
        return {"bytes": V * (192 + 192 + 576), "flops": V * D}
    if kind in ("batched", "multi", "vcycle"):
        n = {"batched": 4, "multi": case.get("nrhs", 1), "vcycle": 1}[kind]
        # outer steps x inner iterations x two D_rr each; the V-cycle counts its level-0 solves
        applies = {"batched": 4 * 25 * 12 * 2, "multi": n * 25 * 12 * 2, "vcycle": 6 * 2 * 2 * 8}[kind]
        return {"bytes": V * (576 + 192 + 192 * n), "flops": applies * V * D}
    nb = V // 16 if case["type"] == 1 else V // 2 if case["type"] == 2 else 0
    nr = V - nb
    if kind == "stencil":
        s = 0.5 if case["prec"] == "bf16" else 1.0
        return {"bytes": nr * 384 * s, "flops": nr * D}
    if kind == "reusken":
        return {"bytes": V * 576 + nb * 384 + nr * 2304, "flops": V * 3 * D + nr * 1152.0}
    if kind == "schur_apply":
        return {"bytes": V * 576 + nb * 384, "flops": 2 * 30 * nr * D}
    if kind == "learned_rr":
        return {"bytes": V * 576 + nr * 384, "flops": 60 * V * (1.99e6 + 2 * 8.3e4)}
    # forward 1 x, backward 2 x the contractions of the network
    return {"bytes": case["batch"] * nr * 192 + V * 288, "flops": 3 * case["batch"] * V * (1.99e6 + 2 * 8.3e4)}


# ---- the same results in 64 bits, from plain torch ------------------------------------------------------

_i = 1j
_GAMMA = np.array([[[0, 0, 0, _i], [0, 0, _i, 0], [0, -_i, 0, 0], [-_i, 0, 0, 0]],
                   [[0, 0, 0, -1], [0, 0, 1, 0], [0, 1, 0, 0], [-1, 0, 0, 0]],
                   [[0, 0, _i, 0], [0, 0, 0, -_i], [-_i, 0, 0, 0], [0, _i, 0, 0]],
                   [[0, 0, 1, 0], [0, 0, 0, 1], [1, 0, 0, 0], [0, 1, 0, 0]]], dtype=np.complex128)


def _neighbours(dims):
    """(forward, backward) site indices per direction."""
    grid = torch.arange(math.prod(dims), device="cuda").reshape(*reversed(dims))
    return [(torch.roll(grid, -1, 3 - mu).reshape(-1), torch.roll(grid, 1, 3 - mu).reshape(-1)) for mu in range(4)]


def _move(T, v):
    """T[x] on the colour index of v [V][k][3]."""
    return T[:, None, :, 0] * v[..., 0:1] + T[:, None, :, 1] * v[..., 1:2] + T[:, None, :, 2] * v[..., 2:3]


class _Wilson:
    """D of a field in site order, on [V][12] vectors."""

    def __init__(self, case, U):
        self.V, self.diag = _volume(case), case["m0"] + 4.0
        self.hops = []
        for mu, (f, b) in enumerate(_neighbours(_dims(case))):
            g = torch.from_numpy(_GAMMA[mu]).to("cuda")
            one = torch.eye(4, dtype=C128, device="cuda")
            self.hops.append((U[:, mu], f, -0.5 * (one - g)))
            self.hops.append((U[b, mu].conj().transpose(1, 2), b, -0.5 * (one + g)))

    def __call__(self, x):
        v = x.reshape(self.V, 4, 3)
        out = self.diag * v
        for T, n, P in self.hops:
            m = _move(T, v[n])
            for s in range(4):
                for k in range(4):
                    if P[s, k] != 0:
                        out[:, s] += P[s, k] * m[:, k]
        return out.reshape(self.V, 12)

    def block(self, rows, cols, x):
        v = torch.zeros(self.V, 12, dtype=C128, device="cuda")
        v[cols] = x.reshape(-1, 12)
        return self(v)[rows]


def _solve(A, b):
    """x with ||b - A x|| / ||b|| near the rounding limit: BiCGStab, restarted from the true residual."""
    x, norm = torch.zeros_like(b), torch.linalg.vector_norm(b)
    for _ in range(6):
        r = b - A(x)
        start = torch.linalg.vector_norm(r)
        if start <= 3e-15 * norm:
            break
        h, p, rho = r.clone(), r.clone(), torch.vdot(r.reshape(-1), r.reshape(-1))
        y = torch.zeros_like(b)
        for it in range(600):
            v = A(p)
            alpha = rho / torch.vdot(h.reshape(-1), v.reshape(-1))
            s = r - alpha * v
            t = A(s)
            omega = torch.vdot(t.reshape(-1), s.reshape(-1)) / torch.vdot(t.reshape(-1), t.reshape(-1))
            y = y + alpha * p + omega * s
            r = s - omega * t
            if it % 5 == 4 and torch.linalg.vector_norm(r) <= max(1e-12 * start, 1e-15 * norm):
                break
            new = torch.vdot(h.reshape(-1), r.reshape(-1))
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
        x = x + y
    return x


def _site_inverse_of_row_sums(D, r):
    """Inverse 12 x 12 blocks of d~_x = sum_y (D_rr)_xy."""
    cols = []
    for k in range(12):
        e = torch.zeros(r.numel(), 12, dtype=C128, device="cuda")
        e[:, k] = 1.0
        cols.append(D.block(r, r, e))
    return torch.linalg.inv(torch.stack(cols, 2))


def exact(case, seed):
    kind = case["kind"]
    U, x = _inputs(case, seed)
    if kind == "train":
        return _exact_train(case, U, *x)
    D = _Wilson(case, U)
    if kind == "wilson":
        return D(x)
    if kind == "vcycle":
        return _solve(D, x)
    if kind == "batched":
        y = _solve(D, x)
        return [y for _ in PERMS]
    if kind == "multi":
        return torch.stack([_solve(D, f) for f in x])
    b, r = _rest_and_coarse(case)
    if kind == "stencil":
        y = D.block(r, r, torch.view_as_complex(x.double().reshape(-1, 12, 2)))
        return _lowp_layout(torch.view_as_real(y).reshape(-1, 24), case["prec"])
    if kind == "learned_rr":
        return _solve(lambda v: D.block(r, r, v), x)
    t = D.block(r, b, x)
    if kind == "schur_apply":
        z = _solve(lambda v: D.block(r, r, v), t)
    else:
        w = (_site_inverse_of_row_sums(D, r) @ t[..., None])[..., 0]
        z = t / D.diag + w - D.block(r, r, w) / D.diag
    return D.block(b, b, x) - D.block(b, r, z)


def _exact_train(case, U, t, z):
    V, batch = _volume(case), case["batch"]
    _, r = _rest_and_coarse(case)
    near = _neighbours(_dims(case))
    trans = [(None, None)] + [(U[:, mu], near[mu][0]) for mu in range(4)]
    trans += [(U[near[mu][1], mu].conj().transpose(1, 2), near[mu][1]) for mu in range(4)]
    W = [torch.from_numpy(w).to("cuda", C128).requires_grad_() for w in learned.identity_like_weights(24, case["m0"], 4)]
    total = 0.0
    for k in range(batch):                 # one pair at a time: the activations of 24 channels are large
        act = torch.zeros(V, 12, dtype=C128, device="cuda")
        act[r] = t[k].to(C128)
        act = act.reshape(V, 4, 3)
        for w in W:
            out = 0.0
            for d, (T, n) in enumerate(trans):
                out = out + torch.einsum("ok,vka->voa", w[d], act if T is None else _move(T, act[n]))
            act = out
        target = z[k].to(C128).reshape(-1)
        diff = act.reshape(V, 12)[r].reshape(-1) - target
        loss = torch.vdot(diff, diff).real / torch.vdot(target, target).real / batch
        loss.backward()
        total += float(loss.detach())
    return [total] + [w.grad for w in W]
