"""The sum-factorised forward at the sizes where it can go wrong: counts
around a block's batch of elements (1 to 4), more batches than resident
blocks (the persistent loop and its record prefetch), a bucketed list, flat
and tiny elements (w det J formed again in FP64), against the FP64 oracle.
Tolerances are the paths' own bars."""
import numpy as np
import pytest

import oracle
from paper_1310_1194_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-12, "fp32": 1e-5, "sf_fp32": 1e-5}


def run(w, precision, p=None, degree=None, **kw):
    from paper_1310_1194_gb300 import api
    g = [torch.from_numpy(np.ascontiguousarray(w[k])).cuda() for k in ("geom", "K", "b", "c", "f")]
    d = None if degree is None else torch.from_numpy(np.ascontiguousarray(degree)).to(torch.int32).cuda()
    A, b, st, _ = api.fei_integrate(*g, p=p, degree=d, precision=precision, **kw)
    torch.cuda.synchronize()
    return A.double().cpu().numpy(), b.double().cpu().numpy(), st.cpu().numpy()


def per_elem_err(got, want, offsets, sizes):
    return np.array([np.linalg.norm(got[o:o + k] - want[o:o + k]) / max(np.linalg.norm(want[o:o + k]), 1e-300)
                     for o, k in zip(offsets, sizes)])


def take(w, idx):
    return {k: np.ascontiguousarray(w[k][idx]) for k in ("geom", "K", "b", "c", "f")}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("p", range(2, 8))
def test_counts_around_a_batch(p, precision):
    """1..5, 7 elements and, on sampled elements, a batch several times the
    resident blocks: the same element must not depend on its place."""
    big = {2: 9001, 3: 7001, 4: 5003, 5: 3001, 6: 1201, 7: 701}[p]
    w = inputs.workload("p4", n_max=big)
    s = (p + 1) ** 2 * (p + 2) // 2
    Ab, bb, stb = run(w, precision, p=p)
    assert not stb.any()
    idx = np.r_[0:7, big // 2, big - 4:big]
    ref = oracle.integrate(*(take(w, idx)[k] for k in ("geom", "K", "b", "c", "f")), p=p)
    off = np.arange(len(idx) + 1)
    ea = per_elem_err(Ab.reshape(big, -1)[idx].reshape(-1), ref[0], off * s * s, np.full(len(idx), s * s))
    eb = per_elem_err(bb.reshape(big, -1)[idx].reshape(-1), ref[1], off * s, np.full(len(idx), s))
    assert ea.max() < TOL[precision] and eb.max() < TOL[precision]
    for n in (1, 2, 3, 4, 5, 7):
        A, b, st = run(take(w, np.arange(n)), precision, p=p)
        assert not st.any()
        assert np.array_equal(A, Ab[:n * s * s]) and np.array_equal(b, bb[:n * s])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_bucketed_equals_uniform(precision):
    """Elements of a list (a degree array) give the uniform call's bits."""
    w = inputs.workload("pr1", n_max=60)
    degree = np.tile(np.arange(2, 8, dtype=np.int32), 10)
    A, b, st = run(w, precision, degree=degree)
    assert not st.any()
    s = (degree + 1) ** 2 * (degree + 2) // 2
    Ao, bo = np.r_[0, np.cumsum(s * s)], np.r_[0, np.cumsum(s)]
    for e in range(0, 60, 7):
        Au, bu, _ = run(take(w, [e]), precision, p=int(degree[e]))
        assert np.array_equal(Au, A[Ao[e]:Ao[e + 1]]) and np.array_equal(bu, b[bo[e]:bo[e + 1]])


@pytest.mark.parametrize("p", [2, 3, 4, 6, 7])
def test_status_of_flat_and_scaled_elements(p):
    """Mirrored, exactly flat and almost flat elements and meshes scaled to
    1e-6 and 1e6: the FP32 path's statuses equal the FP64 path's and the
    oracle's, and unflagged results hold the bar."""
    w = inputs.workload("pr1", n_max=12)
    w = {k: w[k].copy() for k in ("geom", "K", "b", "c", "f")}
    g = w["geom"]
    g[1] = g[1][[0, 2, 1, 3, 5, 4]]
    g[3, 3:] = g[3, :3]
    g[5, 3:] = g[5, :3] + 1e-5 * (g[5, 3:] - g[5, :3])
    g[7] *= 1e-6
    g[8] *= 1e6
    g[10, 2, 1] = np.inf
    A64, b64, s64 = run(w, "fp64", p=p)
    A32, b32, s32 = run(w, "fp32", p=p)
    Ao, bo, so, (Aoff, _, _) = oracle.integrate(w["geom"], w["K"], w["b"], w["c"], w["f"], p=p)
    assert np.array_equal(s64, so) and np.array_equal(s32, so)
    assert set(np.flatnonzero(so)) == {1, 3, 10}
    s = (p + 1) ** 2 * (p + 2) // 2
    sizes = np.full(12, s * s)
    keep = so == 0
    assert per_elem_err(A64, Ao, Aoff, sizes)[keep].max() < 1e-12
    assert per_elem_err(A32, Ao, Aoff, sizes)[keep].max() < 1e-5
    assert not A32.reshape(12, -1)[~keep].any() and not b32.reshape(12, -1)[~keep].any()


@pytest.mark.parametrize("p", [3, 4])
def test_auto_follows_the_whole_batch(p):
    """FEI_AUTO at p = 3, 4 picks its kernel by the size of the caller's batch:
    at most 512 elements give FEI_TC_F16X3's bits and more FEI_SF_FP32's, in
    chunks through host memory as well."""
    from paper_1310_1194_gb300 import api
    for n, same in ((512, "tc_f16x3"), (513, "sf_fp32")):
        w = inputs.workload("pr1", n_max=n)
        w = take(w, np.arange(n))
        A, b, st = run(w, "auto", p=p)
        As, bs, _ = run(w, same, p=p)
        assert not st.any() and np.array_equal(A, As) and np.array_equal(b, bs)
        pipe = api.Pipeline(degrees=[p], precision="auto", slot_bytes=1 << 20)
        Ah, bh, _ = pipe.integrate_host(*(torch.from_numpy(w[k]).pin_memory() for k in ("geom", "K", "b", "c", "f")), p=p)
        torch.cuda.synchronize()
        assert pipe.n_chunks > 1
        assert np.array_equal(Ah.double().numpy(), A) and np.array_equal(bh.double().numpy(), b)


@pytest.mark.parametrize("precision,tol_elem,tol_rec", [("fp64", 1e-10, 1e-10), ("fp32", 1e-6, 1e-5)])
@pytest.mark.parametrize("p", range(1, 8))
def test_adjoint_counts_and_lists(p, precision, tol_elem, tol_rec):
    """The general and the quadratic-loss adjoint on more elements than
    resident blocks (the persistent loop reuses every buffer): sampled
    elements against the oracle; single elements, and elements of a list
    among other degrees, give the same bits."""
    from paper_1310_1194_gb300 import api
    from parity_util import assert_grads_close
    n = {1: 8001, 2: 8001, 3: 5001, 4: 2501, 5: 1601, 6: 901, 7: 701}[p]
    w = inputs.workload("p4", n_max=n)
    s = (p + 1) ** 2 * (p + 2) // 2
    dt = torch.float64 if precision == "fp64" else torch.float32
    rng = np.random.default_rng(p)
    gA, gb, u = (torch.from_numpy(rng.standard_normal(m)).cuda() for m in (n * s * s, n * s, n * s))
    gA, gb = gA.to(dt), gb.to(dt)
    dev = lambda ww: [torch.from_numpy(np.ascontiguousarray(ww[k])).cuda() for k in ("geom", "K", "b", "c", "f")]  # noqa: E731
    g = dev(w)
    full = api.fei_integrate_backward(*g, gA, gb, p=p, precision=precision)
    quad = api.fei_integrate_backward_quadratic(*g, u, p=p, precision=precision)
    idx = np.r_[0, 1, n // 2, n - 2, n - 1]
    sub = take(w, idx)
    Ai, bi = gA.view(n, -1)[idx].contiguous(), gb.view(n, -1)[idx].contiguous()
    ui = u.view(n, -1)[idx].cpu().numpy()
    args = [sub[k] for k in ("geom", "K", "b", "c", "f")]
    ref = oracle.integrate_backward(*args, Ai.double().cpu().numpy().reshape(-1), bi.double().cpu().numpy().reshape(-1), p=p)
    nq = np.full(len(idx), (p + 1) ** 3)
    assert_grads_close([t[idx].cpu().numpy() for t in full], ref, len(idx), False, nq, tol_elem, tol_rec, where=f"general p={p}")
    uu = np.einsum("ni,nj->nij", ui, ui)
    ref = oracle.integrate_backward(*args, uu.reshape(-1), -ui.reshape(-1), p=p)
    assert_grads_close([t[idx].cpu().numpy() for t in quad], ref, len(idx), False, nq, tol_elem, tol_rec, where=f"quad p={p}")
    # a list of the same elements between elements of another degree
    other = 1 + p % 7
    so = (other + 1) ** 2 * (other + 2) // 2
    degree = torch.tensor([p, other] * len(idx), dtype=torch.int32, device="cuda")
    mixed = dev({k: np.repeat(sub[k], 2, axis=0) for k in sub})
    pad = lambda t, m: torch.cat([t, torch.zeros(len(idx), m, dtype=t.dtype, device="cuda")], 1).reshape(-1).contiguous()  # noqa: E731
    got = api.fei_integrate_backward(*mixed, pad(Ai, so * so), pad(bi, so), degree=degree, precision=precision)
    for x, y in zip(got, full):
        assert torch.equal(x[::2], y[idx])
    one = api.fei_integrate_backward(*(t[2:3].contiguous() for t in dev(sub)), Ai[2].contiguous(), bi[2].contiguous(), p=p,
                                     precision=precision)
    for x, y in zip(one, full):
        assert torch.equal(x[0], y[idx[2]])


def test_p1_kernels_agree_in_and_out_of_the_pair_range():
    """p = 1: the one-thread kernel (above 16384 elements) and the eight-lane
    kernel give the same bits, tiles with a ragged end, elements of a list,
    and elements whose vertex differences are outside the FP32 pairs' range
    (an axis scaled to 1e-19) included; sampled elements against the oracle."""
    n = 16384 + 77
    w = inputs.workload("p1m", n_max=n)
    w = take(w, np.arange(n))
    odd = np.arange(5, n, 1000)
    w["geom"][odd] *= np.array([1e-19, 1e9, 1e9])
    A, b, st = run(w, "fp32", p=1)
    assert not st.any()
    idx = np.r_[0, 5, 127, 128, 1005, 16389, n - 1]
    As, bs, _ = run(take(w, idx), "fp32", p=1)
    assert np.array_equal(A.reshape(n, 36)[idx], As.reshape(-1, 36))
    assert np.array_equal(b.reshape(n, 6)[idx], bs.reshape(-1, 6))
    sub = take(w, idx)
    Ao, bo, so, _ = oracle.integrate(*(sub[k] for k in ("geom", "K", "b", "c", "f")), p=1)
    off, sizes = np.arange(len(idx)) * 36, np.full(len(idx), 36)
    assert not so.any() and per_elem_err(As, Ao, off, sizes).max() < 1e-5
    assert per_elem_err(bs, bo, off // 6, sizes // 6).max() < 1e-5
    # as every second element of a list of 2 n elements of degrees 1 and 2
    m = 200
    both = {k: np.repeat(w[k][:m], 2, axis=0) for k in w}
    degree = np.tile(np.array([2, 1], dtype=np.int32), m)
    Al, bl, sl = run(both, "fp32", degree=degree)
    at = np.r_[0, np.cumsum(np.where(degree == 1, 36, 324))]
    got = np.stack([Al[at[2 * i + 1]:at[2 * i + 2]] for i in range(m)])
    assert np.array_equal(got, A.reshape(n, 36)[:m])


@pytest.mark.parametrize("p,per_qp", [(3, False), (4, False), (5, True)])
def test_adjoint_wide_cotangents_past_the_resident_blocks(p, per_qp):
    """Cotangents whose rows differ by six orders of magnitude, on about twice
    as many elements as there are resident blocks: the loop reuses Y, X and D
    and takes the next element's rows; sampled elements against the oracle
    (the FP32 adjoint's bars)."""
    from paper_1310_1194_gb300 import api
    from parity_util import assert_grads_close
    n, s, q = {3: 4001, 4: 2003, 5: 1601}[p], api.nsh(p), api.nq(p)
    w = inputs.workload("diff" if per_qp else "p4", n_max=n)
    n = len(w["geom"])
    rng = np.random.default_rng(40 + p)
    gA = (rng.standard_normal((n, s, s)) * 10.0 ** rng.integers(-3, 4, size=(n, s, 1))).astype(np.float32)
    gb = rng.standard_normal((n, s)).astype(np.float32)
    dev = [torch.from_numpy(np.ascontiguousarray(w[k])).cuda() for k in ("geom", "K", "b", "c", "f")]
    got = api.fei_integrate_backward(*dev, torch.from_numpy(gA).cuda(), torch.from_numpy(gb).cuda(), p=p, per_qp=per_qp,
                                     precision="fp32")
    idx = np.r_[0, 1, n // 2, n - 903, n - 2, n - 1]
    rec = (idx[:, None] * q + np.arange(q)).reshape(-1) if per_qp else idx
    sub = [w["geom"][idx]] + [w[k][rec] for k in ("K", "b", "c", "f")]
    ref = oracle.integrate_backward(*(np.ascontiguousarray(x) for x in sub), gA[idx].astype(np.float64).reshape(-1),
                                    gb[idx].astype(np.float64).reshape(-1), p=p, per_qp=per_qp)
    out = [got[0].cpu().numpy()[idx]] + [t.cpu().numpy()[rec] for t in got[1:]]
    assert_grads_close(out, ref, len(idx), per_qp, np.full(len(idx), q), 1e-6, 1e-5, where=f"p={p}")
