"""The work that users of this library have it do, as cases that can be timed.

Each case is one call, or the few calls of one step, through the public entry
points of ``paper_1310_1194_gb300.api`` on seeded synthetic meshes: forward
integration at the smallest and the largest batches and in the precisions a
caller chooses, a mixed-degree plan, training steps (forward and adjoint),
fused assembly, and a batch in host memory.  ``exact`` evaluates the same
definitions (Gauss-Legendre, collapsed prism rule, Dubiner x Legendre basis,
the weak form) densely in FP64 with numpy and torch.

Kinds of case:
  forward  api.fei_integrate                         -> A, b, status
  plan     api.Plan.execute on a degree array        -> A, b, status
  step     api.integrate and its backward            -> A, b, status, 5 gradients
  quad     api.fei_integrate and the quadratic-loss
           adjoint                                   -> A, b, status, 5 gradients
  assemble api.Assembly.integrate_assemble           -> values, rhs, status
  host     api.Pipeline.integrate_host               -> A, b, status
"""
import math

import numpy as np
import torch

from paper_1310_1194_gb300 import api

# share of each degree 1..7 in a mixed batch
MIXED = (0.25, 0.2, 0.15, 0.15, 0.1, 0.1, 0.05)


def listed():
    return [
        # one small mesh at the lowest degree: launch and latency
        dict(name="p1_small", kind="forward", p=1, n=4096, precision="auto"),
        # a large mesh at the lowest degree
        dict(name="p1_million", kind="forward", p=1, n=1000000, precision="auto"),
        # the ordinary large batch of middle degree, fastest path
        dict(name="p4_batch", kind="forward", p=4, n=100000, precision="auto"),
        # the call's default precision, a ragged count
        dict(name="p5_fp32", kind="forward", p=5, n=10007, precision="fp32"),
        # symmetric form in the upper-triangle layout on the tensor-core precision
        dict(name="p4_upper", kind="forward", p=4, n=30001, precision="tc_f16x3", upper=True),
        # the highest degree on a strongly distorted mesh; the largest outputs
        dict(name="p7_batch", kind="forward", p=7, n=16384, precision="auto", jitter=0.25),
        # every degree in one batch, through a plan kept by the caller
        dict(name="mixed_plan", kind="plan", n=50000, precision="auto"),
        # training step: coefficients per quadrature point, general cotangents
        dict(name="p5_step", kind="step", p=5, n=20000, precision="auto", per_qp=True),
        # energy minimisation step: the adjoint of the quadratic loss
        dict(name="p5_quadratic", kind="quad", p=5, n=20000, precision="auto", per_qp=True),
        # reference-accuracy step, all in FP64
        dict(name="p4_fp64_step", kind="step", p=4, n=4096, precision="fp64"),
        # integration and assembly into CSR on one mesh
        dict(name="p4_assemble", kind="assemble", p=4, nx=30, ny=30, nz=20, precision="tc_f16x3"),
        # a batch that lives in (pinned) host memory
        dict(name="p4_host", kind="host", p=4, n=12000, precision="tc_f16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "plan", "step", "step", "quad", "assemble", "host"])
    p = rng.randint(1, 7)
    precision = rng.choice(["auto", "auto", "fp32", "fp64", "tc_f16x3", "sf_fp32"])
    if kind == "plan":
        return dict(kind=kind, n=_log(rng, 300, 2000 if precision == "fp64" else 30000), precision=precision)
    if kind == "assemble":
        cap = _cap(p, precision, False)
        k = max(2, min(rng.randint(4, 24), int(round((cap / 2) ** (1 / 3)))))
        return dict(kind=kind, p=p, nx=k, ny=max(2, k - rng.randint(0, 2)), nz=rng.randint(2, k), precision=precision)
    per_qp = kind in ("step", "quad") and rng.random() < 0.5
    # an element costs two to three times the forward's in a training step
    n = _log(rng, 50, max(100, _cap(p, precision, kind in ("step", "quad"))))
    case = dict(kind=kind, p=p, n=n, precision=precision)
    if per_qp:
        case["per_qp"] = True
    if kind == "forward" and rng.random() < 0.2:
        case["upper"] = True
    if kind == "forward" and rng.random() < 0.3:
        case["jitter"] = 0.25
    return case


def _cap(p, precision, adjoint):
    """Most elements of a drawn case: bounded by its outputs and by the flops
    of the dense contraction, below the largest listed cases."""
    s, q = api.nsh(p), api.nq(p)
    dense = 8.0 * s * s * q * (3 if adjoint else 1)
    by_flops = (4.0e10 if precision == "fp64" else 2.5e11) / dense
    by_bytes = 1.5e9 / (4.0 * s * s * (2 if adjoint else 1))
    return int(max(60, min(by_flops, by_bytes, 300000)))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _mesh_size(n):
    k = max(1, int(round((n / 2) ** (1 / 3))))
    return k, k, -(-n // (2 * k * k))


def _vertex_ids(nx, ny, nz, dev):
    """Vertex ids [2 nx ny nz, 6]: each cell split into two prisms."""
    r = torch.arange
    k, j, i = (t.reshape(-1) for t in torch.meshgrid(r(nz, device=dev), r(ny, device=dev), r(nx, device=dev),
                                                     indexing="ij"))
    at = lambda di, dj: (k * (ny + 1) + j + dj) * (nx + 1) + i + di  # noqa: E731
    tri = torch.stack([torch.stack([at(0, 0), at(1, 0), at(1, 1)], 1),
                       torch.stack([at(0, 0), at(1, 1), at(0, 1)], 1)], 1).reshape(-1, 3)
    return torch.cat([tri, tri + (nx + 1) * (ny + 1)], 1)


def _mesh(nx, ny, nz, n, jitter, gen):
    """Jittered prisms of the unit cube, FP64 [n, 6, 3]; an element that the
    jitter folds keeps its regular vertices."""
    dev = gen.device
    lin = lambda m: torch.linspace(0, 1, m + 1, dtype=torch.float64, device=dev)  # noqa: E731
    z, y, x = torch.meshgrid(lin(nz), lin(ny), lin(nx), indexing="ij")
    base = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)
    h = torch.tensor([1 / nx, 1 / ny, 1 / nz], dtype=torch.float64, device=dev)
    move = (torch.rand(base.shape, generator=gen, dtype=torch.float64, device=dev) * 2 - 1) * jitter * h
    ids = _vertex_ids(nx, ny, nz, dev)[:n]
    geom, flat = (base + move)[ids], base[ids]
    P, Q = geom[:, :3], geom[:, 3:]
    ok = torch.ones(len(geom), dtype=torch.bool, device=dev)
    for t in torch.linspace(0, 1, 9).tolist():
        s = (1 - t) * P + t * Q
        normal = torch.linalg.cross(s[:, 1] - s[:, 0], s[:, 2] - s[:, 0])
        for a in range(3):
            ok &= (normal * (Q[:, a] - P[:, a])).sum(1) > 0.05 * h.prod()
    return torch.where(ok[:, None, None], geom, flat).contiguous()


def _rotations(m, gen):
    q = torch.randn(m, 4, generator=gen, dtype=torch.float64, device=gen.device)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(m, 3, 3)


def _coefficients(n, gen, symmetric):
    """Per element: diffusion K = Q diag(0.5..2) Q^T, velocity b, reaction c, source f."""
    dev = gen.device
    u = lambda *s: torch.rand(*s, generator=gen, dtype=torch.float64, device=dev)  # noqa: E731
    R = _rotations(n, gen)
    K = (R * (0.5 + 1.5 * u(n, 1, 3))) @ R.transpose(1, 2)
    K = (0.5 * (K + K.transpose(1, 2))).contiguous()
    b = torch.zeros(n, 3, dtype=torch.float64, device=dev) if symmetric else u(n, 3) * 2 - 1
    return K, b, u(n), u(n) * 2 - 1


def _fields(geom, p, gen):
    """Per quadrature point: smooth fields of position, [n (p+1)^3, ...]."""
    n, dev = geom.shape[0], geom.device
    pts = torch.from_numpy(_points(p)).to(dev)
    lam = torch.stack([1 - pts[:, 0] - pts[:, 1], pts[:, 0], pts[:, 1]], 1)
    N = torch.cat([lam * (0.5 * (1 - pts[:, 2:3])), lam * (0.5 * (1 + pts[:, 2:3]))], 1)
    x = torch.einsum("qv,nvk->nqk", N, geom).reshape(-1, 3)
    u = lambda *s: torch.rand(*s, generator=gen, dtype=torch.float64, device=dev)  # noqa: E731
    R = _rotations(1, gen)[0]
    K0 = (R * (0.75 + u(1, 3))) @ R.T
    K0 = 0.5 * (K0 + K0.T)
    wave = lambda: torch.sin(x @ (1 + 3 * u(3)) + 6.28 * u(1))  # noqa: E731
    K = K0 + (0.25 * wave())[:, None, None] * torch.eye(3, dtype=torch.float64, device=dev)
    b = torch.stack([wave() for _ in range(3)], 1)
    return K.contiguous(), b.contiguous(), 0.5 * (1 + wave()), wave()


def _degrees(n, gen):
    """The shares of MIXED, shuffled."""
    counts = [int(n * w) for w in MIXED]
    counts[0] += n - sum(counts)
    degree = torch.repeat_interleave(torch.arange(1, 8), torch.tensor(counts)).to(gen.device, torch.int32)
    return degree[torch.randperm(n, generator=gen, device=gen.device)].contiguous()


def _inputs(case, seed):
    """geom, K, b, c, f (FP64), degree (plan) and the generator, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    if case["kind"] == "assemble":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        n = 2 * nx * ny * nz
    else:
        n = case["n"]
        nx, ny, nz = _mesh_size(n)
    geom = _mesh(nx, ny, nz, n, case.get("jitter", 0.1), gen)
    degree = _degrees(n, gen) if case["kind"] == "plan" else None
    if case.get("per_qp"):
        coef = _fields(geom, case["p"], gen)
    else:
        coef = _coefficients(n, gen, case.get("upper", False))
    return geom, coef, degree, gen


def _fp32(case):
    return case["precision"] != "fp64"


def _parameters(case, seed):
    """A training step's parameters: the mesh, a displacement of its element
    vertices and the coefficients, in the precision the optimiser keeps (FP32
    unless the step is FP64), and the cotangents of A and b."""
    geom, coef, _, gen = _inputs(case, seed)
    dt = torch.float32 if _fp32(case) else torch.float64
    n, s = case["n"], api.nsh(case["p"])
    move = (1e-3 * (n / 2) ** (-1 / 3)
            * torch.randn(geom.shape, generator=gen, dtype=torch.float64, device=gen.device)).to(dt)
    gA = torch.randn(n * s * s, generator=gen, dtype=dt, device=gen.device)
    gb = torch.randn(n * s, generator=gen, dtype=dt, device=gen.device)
    return geom, [move] + [t.to(dt) for t in coef], gA, gb


def _l2g(case, dev):
    """Global numbers [n, N_sh]: the first six functions of an element carry
    its mesh vertices, the others are its own; and their count."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    v = _vertex_ids(nx, ny, nz, dev)
    nv, n, own = (nx + 1) * (ny + 1) * (nz + 1), v.shape[0], api.nsh(case["p"]) - 6
    private = nv + torch.arange(n * own, device=dev).reshape(n, own)
    return torch.cat([v, private], 1), nv + n * own


def prepare(case, seed):
    st = dict(case=case)
    kind = case["kind"]
    if kind == "step":
        geom, params, gA, gb = _parameters(case, seed)
        st.update(geom=geom, params=[t.requires_grad_(True) for t in params], gA=gA, gb=gb)
        return st
    geom, coef, degree, gen = _inputs(case, seed)
    if kind == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        n, s = case["n"], api.nsh(case["p"])
        dt = torch.float32 if _fp32(case) else torch.float64
        st["args"] = [pin(t) for t in (geom, *coef)]
        st["out"] = (torch.empty(n * s * s, dtype=dt, pin_memory=True), torch.empty(n * s, dtype=dt, pin_memory=True),
                     torch.empty(n, dtype=torch.int32, pin_memory=True))
        st["pipe"] = api.Pipeline(degrees=[case["p"]], precision=case["precision"])
        return st
    st["args"] = (geom, *coef)
    if kind == "plan":
        st["degree"] = degree
        st["layout"] = api.fei_plan_offsets(degree)
        st["plan"] = api.Plan(max_elem=case["n"], precision=case["precision"])
        dt = torch.float32 if _fp32(case) else torch.float64
        st["out"] = (torch.empty(st["layout"].A_total, dtype=dt, device="cuda"),
                     torch.empty(st["layout"].b_total, dtype=dt, device="cuda"),
                     torch.empty(case["n"], dtype=torch.int32, device="cuda"))
    elif kind == "quad":
        st["u"] = torch.randn(case["n"] * api.nsh(case["p"]), generator=gen, dtype=torch.float64, device="cuda")
    elif kind == "assemble":
        l2g, n_dof = _l2g(case, "cpu")
        st["asm"] = api.Assembly(l2g.reshape(-1).numpy(), n_dof, p=case["p"])
    return st


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    precision = case["precision"]
    if kind == "forward":
        A, b, status, _ = api.fei_integrate(*state["args"], p=case["p"], precision=precision,
                                            upper=case.get("upper", False))
        return A, b, status
    if kind == "plan":
        A, b, status, _ = state["plan"].execute(*state["args"], degree=state["degree"], layout=state["layout"],
                                                out=state["out"])
        return A, b, status
    if kind == "step":
        # parameters in the optimiser's precision, the library's inputs in FP64
        move, K, bc, c, f = state["params"]
        A, b, status = api.integrate(state["geom"] + move, K.double(), bc.double(), c.double(), f.double(),
                                     p=case["p"], per_qp=case.get("per_qp", False), precision=precision)
        return A, b, status, torch.autograd.grad((A, b), state["params"], (state["gA"], state["gb"]))
    if kind == "quad":
        per_qp = case.get("per_qp", False)
        A, b, status, layout = api.fei_integrate(*state["args"], p=case["p"], per_qp=per_qp, precision=precision)
        grads = api.fei_integrate_backward_quadratic(*state["args"], state["u"], p=case["p"], per_qp=per_qp,
                                                     precision=precision, layout=layout)
        # handed on to an optimiser that keeps FP32 unless the step is FP64
        return A, b, status, [g.float() for g in grads] if _fp32(case) else list(grads)
    if kind == "assemble":
        return state["asm"].integrate_assemble(*state["args"], precision=precision)
    return state["pipe"].integrate_host(*state["args"], p=case["p"], out=state["out"])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    """bytes: inputs read once, outputs written once.  flops: the three
    one-dimensional sums of the collapsed tensor-product rule (13 pairs of
    separable gradient factors over u and v, then 4 pairs of zeta factors),
    once per direction."""
    out = 4 if _fp32(case) else 8

    def per_degree(p, n):
        m, t, s, q = p + 1, (p + 1) * (p + 2) // 2, api.nsh(p), api.nq(p)
        flops = 2.0 * (13 * (m ** 5 + t * t * m * m) + 4 * t * t * m * m * m) + 220.0 * q
        rec = q if case.get("per_qp") else 1
        read, write = 144.0 + 112 * rec, float(out * (s * s + s) + 4)
        if case.get("upper"):
            write = out * (s * (s + 1) / 2 + s) + 4.0
        if case["kind"] == "step":
            # the cotangents read and the gradients written as well
            read, write, flops = read + out * (s * s + s), write + out * (18 + 14 * rec), 2 * flops
        if case["kind"] == "quad":
            read, write, flops = read + 8 * s, write + out * (18 + 14 * rec), flops + 8.0 * s * m * 3 + 400.0 * q
        return n * (read + write), n * flops

    if case["kind"] == "plan":
        parts = [per_degree(p, case["n"] * w) for p, w in zip(range(1, 8), MIXED)]
        return dict(bytes=sum(x for x, _ in parts), flops=sum(y for _, y in parts))
    n = 2 * case["nx"] * case["ny"] * case["nz"] if case["kind"] == "assemble" else case["n"]
    byts, flops = per_degree(case["p"], n)
    return dict(bytes=byts, flops=flops)


# --------------------------------------------------------------------------
# the definitions in FP64
# --------------------------------------------------------------------------
def _points(p):
    """[N_q, 4]: xi1, xi2, zeta, weight; zeta slowest, then v, then u."""
    x, w = np.polynomial.legendre.leggauss(p + 1)
    z, v, u = (t.reshape(-1) for t in np.meshgrid(x, x, x, indexing="ij"))
    wz, wv, wu = (t.reshape(-1) for t in np.meshgrid(w, w, w, indexing="ij"))
    return np.stack([(1 + u) * (1 - v) / 4, (1 + v) / 2, z, wu * wv * wz * (1 - v) / 8], 1)


def _jacobi(n, a, b, x):
    """P_n^(a,b)(x) by the three-term recurrence."""
    prev, cur = np.zeros_like(x), np.ones_like(x)
    for k in range(n):
        if k == 0:
            prev, cur = cur, 0.5 * (a - b + (a + b + 2) * x)
            continue
        s = 2 * k + a + b
        lead = 2 * (k + 1) * (k + a + b + 1) * s
        nxt = ((s + 1) * (a * a - b * b + s * (s + 2) * x) * cur - 2 * (k + a) * (k + b) * (s + 2) * prev) / lead
        prev, cur = cur, nxt
    return cur


def _djacobi(n, a, b, x):
    return np.zeros_like(x) if n == 0 else 0.5 * (n + a + b + 1) * _jacobi(n - 1, a + 1, b + 1, x)


def _basis(p):
    """[N_q, 4, N_sh]: value and reference gradient of every function."""
    pts = _points(p)
    xi1, xi2, z = pts[:, 0], pts[:, 1], pts[:, 2]
    v = 2 * xi2 - 1
    u = 4 * xi1 / (1 - v) - 1
    out = np.empty((len(pts), 4, api.nsh(p)))
    i = 0
    for k in range(p + 1):
        L, dL = (math.sqrt(k + 0.5) * fn(k, 0, 0, z) for fn in (_jacobi, _djacobi))
        for d in range(p + 1):
            for n in range(d + 1):
                m = d - n
                c = math.sqrt(2.0 * (2 * m + 1) * (m + n + 1))
                h = (1 - v) / 2
                A, dA = _jacobi(m, 0, 0, u), _djacobi(m, 0, 0, u)
                J, dJ = _jacobi(n, 2 * m + 1, 0, v), _djacobi(n, 2 * m + 1, 0, v)
                B = c * h ** m * J
                dB = c * (h ** m * dJ - (0.5 * m * h ** (m - 1) * J if m else 0.0))
                # du/dxi1 = 4/(1-v), du/dxi2 = 2(1+u)/(1-v), dv/dxi2 = 2
                out[:, 0, i] = A * B * L
                out[:, 1, i] = dA * 4 / (1 - v) * B * L
                out[:, 2, i] = (dA * 2 * (1 + u) / (1 - v) * B + 2 * A * dB) * L
                out[:, 3, i] = A * B * dL
                i += 1
    return out


def _operators(geom, K, b, c, f, p):
    """The 4 x 4 point operators [n, N_q, 4, 4] and the load weights [n, N_q];
    K, b, c, f with a point axis of length 1 or N_q."""
    pts = torch.from_numpy(_points(p)).to(geom.device)
    x1, x2, z, w = pts.unbind(1)
    one, nil = torch.ones_like(z), torch.zeros_like(z)
    lam = torch.stack([1 - x1 - x2, x1, x2], 1)
    lo, hi = (0.5 * (1 - z))[:, None], (0.5 * (1 + z))[:, None]
    e1, e2 = torch.stack([-one, one, nil], 1), torch.stack([-one, nil, one], 1)
    dN = torch.stack([torch.cat([e1 * lo, e1 * hi], 1), torch.cat([e2 * lo, e2 * hi], 1),
                      torch.cat([-0.5 * lam, 0.5 * lam], 1)], 1)
    c1, c2, c3 = torch.einsum("qlv,nvk->lnqk", dN, geom)
    adj = torch.stack([torch.linalg.cross(c2, c3), torch.linalg.cross(c3, c1), torch.linalg.cross(c1, c2)], 2)
    det = (adj[:, :, 2] * c3).sum(2)
    top = torch.cat([(w * det * c)[..., None], w[:, None] * (adj @ b[..., None])[..., 0]], 2)
    low = (w / det)[..., None, None] * (adj @ (K @ adj.transpose(2, 3)))
    D = torch.cat([top[:, :, None, :], torch.cat([torch.zeros_like(low[..., :1]), low], 3)], 2)
    return D, w * det * f


def _split(t, n):
    """A coefficient array with its element and point axes."""
    return t.reshape(n, t.shape[0] // n, *t.shape[1:])


def _chunks(n, p):
    step = max(1, int(3e8 / (4 * api.nq(p) * api.nsh(p))))
    return [slice(i, min(n, i + step)) for i in range(0, n, step)]


def _dense(geom, coef, p):
    """A [n, N_sh, N_sh], b [n, N_sh] of the elements given."""
    n, s = geom.shape[0], api.nsh(p)
    G = torch.from_numpy(_basis(p)).to(geom.device)
    A = torch.empty(n, s, s, dtype=torch.float64, device=geom.device)
    b = torch.empty(n, s, dtype=torch.float64, device=geom.device)
    coef = [_split(t, n) for t in coef]
    for k in _chunks(n, p):
        D, F = _operators(geom[k], *(t[k] for t in coef), p)
        H = torch.einsum("nqab,qai->niqb", D, G).reshape(-1, 4 * G.shape[0])
        A[k] = (H @ G.reshape(-1, s)).reshape(-1, s, s)
        b[k] = F @ G[:, 0]
    return A, b


def _dense_grads(geom, params, p, loss):
    """d loss / d (geometry, K, b, c, f), chunk by chunk; loss(D, F, G, chunk)."""
    n = geom.shape[0]
    G = torch.from_numpy(_basis(p)).to(geom.device)
    got = []
    split = [_split(t, n) for t in params]
    for k in _chunks(n, p):
        x = [t[k].clone().requires_grad_(True) for t in (geom, *split)]
        D, F = _operators(*x, p)
        got.append(torch.autograd.grad(loss(D, F, G, k), x))
    whole = [torch.cat(t) for t in zip(*got)]
    return [whole[0]] + [t.reshape(q.shape) for t, q in zip(whole[1:], params)]


def exact(case, seed):
    kind, p = case["kind"], case.get("p")
    if kind == "step":
        geom, (move, *coef), gA, gb = _parameters(case, seed)
        geom, coef = geom + move, [t.double() for t in coef]
        n, s = case["n"], api.nsh(p)
        A, b = _dense(geom, coef, p)

        def loss(D, F, G, k):
            # <gA, A> = sum D[a][b] (G_a gA G_b^T)
            X = gA.reshape(n, s, s)[k].double()
            W = (X.reshape(-1, s) @ G.reshape(-1, s).T).reshape(X.shape[0], s, -1, 4)
            gD = torch.einsum("qai,niqb->nqab", G, W)
            return (D * gD).sum() + ((F @ G[:, 0]) * gb.reshape(n, s)[k].double()).sum()

        return A.reshape(-1), b.reshape(-1), None, _dense_grads(geom, coef, p, loss)
    geom, coef, degree, gen = _inputs(case, seed)
    n = geom.shape[0]
    if kind == "plan":
        s = (degree.long() + 1) ** 2 * (degree.long() + 2) // 2
        sq = s * s
        at, bt = sq.cumsum(0) - sq, s.cumsum(0) - s
        A = torch.empty(int(sq.sum()), dtype=torch.float64, device="cuda")
        b = torch.empty(int(s.sum()), dtype=torch.float64, device="cuda")
        for q in range(1, 8):
            for ids in torch.nonzero(degree == q)[:, 0].split(4096):
                if len(ids):
                    Ae, be = _dense(geom[ids], [t[ids] for t in coef], q)
                    m = api.nsh(q)
                    A[at[ids, None] + torch.arange(m * m, device="cuda")] = Ae.reshape(-1, m * m)
                    b[bt[ids, None] + torch.arange(m, device="cuda")] = be
        return A, b, None
    A, b = _dense(geom, coef, p)
    s = api.nsh(p)
    if kind == "assemble":
        l2g, n_dof = _l2g(case, "cuda")
        key = (l2g[:, :, None] * n_dof + l2g[:, None, :]).reshape(-1)
        places, where = torch.unique(key, return_inverse=True)
        values = torch.zeros(len(places), dtype=torch.float64, device="cuda").index_add_(0, where, A.reshape(-1))
        rhs = torch.zeros(n_dof, dtype=torch.float64, device="cuda").index_add_(0, l2g.reshape(-1), b.reshape(-1))
        return values, rhs, None
    if kind == "quad":
        u = torch.randn(n * s, generator=gen, dtype=torch.float64, device="cuda").reshape(n, s)

        def loss(D, F, G, k):
            v = (u[k] @ G.reshape(-1, s).T).reshape(-1, G.shape[0], 4)
            return ((D @ v[..., None])[..., 0] * v).sum() - ((F @ G[:, 0]) * u[k]).sum()

        return A.reshape(-1), b.reshape(-1), None, _dense_grads(geom, coef, p, loss)
    if case.get("upper"):
        i, j = torch.triu_indices(s, s, device="cuda")
        A = A[:, i, j]
    A, b = A.reshape(-1), b.reshape(-1)
    return (A.cpu(), b.cpu(), None) if kind == "host" else (A, b, None)
