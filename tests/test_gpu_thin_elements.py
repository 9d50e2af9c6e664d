"""Thin, collapsed and mirrored triangles: n3 = c1 x c2 cancels, so the FP32
paths must not flag or scale these elements by an FP32 pair's last bits.

The elements: a mesh element moved to the origin (the vertices' rounding
scales with the element), its third vertices drawn to the line through the
other two: P2 = P0 + 0.4 (P1 - P0) + eps (P2 - P0), the top alike.  Then c1 x
c2 is eps times the element's own at every zeta, so det J has the sign of eps
at every point.  FP64 arithmetic forms w det J to about 10 2^-53 / eps
(relative), FP32 pairs to at worst 10 2^-44 / eps."""
import numpy as np
import pytest

import oracle
from paper_1310_1194_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KEYS = ("geom", "K", "b", "c", "f")
NEGATIVE = 3


def thin(n, eps, at=0.4):
    w = inputs.workload("pr1", n_max=max(n, 1))
    w = {k: np.ascontiguousarray(np.resize(w[k], (n,) + w[k].shape[1:])) for k in KEYS}
    g = w["geom"] - w["geom"][:, :1]
    for o in (0, 3):
        g[:, o + 2] = g[:, o] + at * (g[:, o + 1] - g[:, o]) + eps * (g[:, o + 2] - g[:, o])
    w["geom"] = np.ascontiguousarray(g)
    return w


def device(w):
    return [torch.from_numpy(w[k]).cuda() for k in KEYS]


def forward(w, precision, p):
    from paper_1310_1194_gb300 import api
    A, b, st, _ = api.fei_integrate(*device(w), p=p, precision=precision)
    torch.cuda.synchronize()
    n = len(w["geom"])
    return A.view(n, -1).double().cpu().numpy(), b.view(n, -1).double().cpu().numpy(), st.cpu().numpy()


def rel(x, y):
    return (np.linalg.norm(x - y, axis=1) / np.linalg.norm(y, axis=1)).max()


def check_accuracy(p, precision, n):
    # FP64 and oracle together: 2 x 10 x 2^-53 / 1e-9 = 2.2e-6, the FP32 path's
    # own error below 1e-6; its bar is 1e-5
    w = thin(n, 1e-9)
    A, b, st = forward(w, precision, p)
    Ao, bo, so, _ = oracle.integrate(*(w[k] for k in KEYS), p=p)
    assert not st.any() and not so.any()
    assert rel(A, Ao.reshape(n, -1)) < 1e-5 and rel(b, bo.reshape(n, -1)) < 1e-5


def check_mirrored(p, precision, n):
    for eps in (-1e-9, -1e-12, -1e-14):
        A, b, st = forward(thin(n, eps), precision, p)
        assert (st == NEGATIVE).all(), (eps, int((st != NEGATIVE).sum()))
        assert not A.any() and not b.any()


@pytest.mark.parametrize("n", [3000, 20000])
def test_p1_thin_and_mirrored(n):
    """Both p = 1 kernels (one thread per element above 16384)."""
    check_accuracy(1, "fp32", n)
    check_mirrored(1, "fp32", n)


@pytest.mark.parametrize("n", [3000, 20000])
def test_p1_collapsed_triangles_are_flagged(n):
    """P1 == P2 and Q1 == Q2: c1 == c2 at every node, so n3 is 0 exactly."""
    w = inputs.workload("p1m", n_max=n)
    w = {k: np.ascontiguousarray(w[k][:n]) for k in KEYS}
    w["geom"][:, 2] = w["geom"][:, 1]
    w["geom"][:, 5] = w["geom"][:, 4]
    A, b, st = forward(w, "fp32", 1)
    assert (st == NEGATIVE).all(), int((st != NEGATIVE).sum())
    assert not A.any() and not b.any()


def test_p1_kernels_agree_on_thin_elements():
    """Elements of every kind give the same bits in both kernels."""
    n, m = 16384 + 300, 300
    parts = [thin(m, e) for e in (1e-3, 1e-4, 1e-5, 1e-9, 1e-13, -1e-4, -1e-13)]
    w = inputs.workload("p1m", n_max=n)
    w = {k: np.ascontiguousarray(w[k][:n]) for k in KEYS}
    for i, q in enumerate(parts):
        for k in KEYS:
            w[k][i::50][:m] = q[k]
    A, b, st = forward(w, "fp32", 1)
    As, bs, ss = forward({k: np.ascontiguousarray(w[k][:16000]) for k in KEYS}, "fp32", 1)
    assert np.array_equal(A[:16000], As) and np.array_equal(b[:16000], bs) and np.array_equal(st[:16000], ss)
    assert 0 < np.count_nonzero(st) < n


SAMPLE = {2: 2000, 3: 600, 4: 300, 5: 100, 6: 60, 7: 40}  # the oracle's share: seconds


def fractions(n):
    return np.random.default_rng(7).uniform(0.1, 0.9, (n, 1))


@pytest.mark.parametrize("precision", ["fp32", "sf_fp32"])
@pytest.mark.parametrize("p", range(2, 8))
def test_thin_accuracy(p, precision):
    """eps = 1e-10, the foot of the height anywhere on the edge.  An FP64 n3
    has at most 3 roundings of two products of size al |c1|^2 where n3 is
    eps |c1| |v| sin: 6 x 2^-53 / eps = 0.7e-5, say 1e-5 at 1e-10, in the path and
    in the oracle; doubled.  FP32 pairs: 2^-44 in the place of 2^-53."""
    n = SAMPLE[p]
    w = thin(n, 1e-10, fractions(n))
    A, b, st = forward(w, precision, p)
    Ao, bo, so, _ = oracle.integrate(*(w[k] for k in KEYS), p=p)
    assert not st.any() and not so.any()
    assert rel(A, Ao.reshape(n, -1)) < 4e-5 and rel(b, bo.reshape(n, -1)) < 4e-5


@pytest.mark.parametrize("p,n", [(2, 60000), (3, 20000)])
def test_thin_mirrored_at_the_end_of_the_pairs(p, n):
    """-5e-15: above FP64's rounding (1e-15 by the bound above), below a pair's."""
    A, b, st = forward(thin(n, -5e-15, fractions(n)), "fp32", p)
    assert (st == NEGATIVE).all(), int((st != NEGATIVE).sum())
    assert not A.any() and not b.any()


@pytest.mark.parametrize("p", range(2, 8))
def test_thin_mirrored(p):
    check_mirrored(p, "fp32", {2: 6000, 3: 5000, 4: 4000, 5: 2000, 6: 1000, 7: 500}[p])


@pytest.mark.parametrize("p", [2, 5])
def test_thin_elements_do_not_depend_on_their_neighbours(p):
    """Elements that take the FP64 setup between elements that do not."""
    n = 700
    w = inputs.workload("p4", n_max=n)
    w = {k: np.ascontiguousarray(w[k][:n]) for k in KEYS}
    alone, _, _ = forward(w, "fp32", p)
    parts = thin(n, 1e-9)
    both = {k: np.ascontiguousarray(np.stack([w[k], parts[k]], 1).reshape((2 * n,) + w[k].shape[1:])) for k in KEYS}
    A, _, st = forward(both, "fp32", p)
    assert not st.any() and np.array_equal(A[::2], alone)
    At, _, _ = forward(parts, "fp32", p)
    assert np.array_equal(A[1::2], At)


def adjoints(w, p, precision):
    """Both adjoints on a load of the constant function: dL/df is +- its value
    times the sum of w det J, in which nothing cancels."""
    from paper_1310_1194_gb300 import api
    g, n, s = device(w), len(w["geom"]), api.nsh(p)
    dt = torch.float64 if precision == "fp64" else torch.float32
    gA, gb = torch.zeros(n * s * s, dtype=dt, device="cuda"), torch.zeros(n, s, dtype=dt, device="cuda")
    gb[:, 0] = 1.0
    general = api.fei_integrate_backward(*g, gA, gb.reshape(-1), p=p, precision=precision)
    u = torch.zeros(n, s, dtype=torch.float64, device="cuda")
    u[:, 0] = 1.0
    return general, api.fei_integrate_backward_quadratic(*g, u.reshape(-1), p=p, precision=precision)


def flat(n, eps):
    """Oblique flat elements: regular triangles, the vertical edge in their plane
    up to eps of its normal part, so that n3 . c3 cancels and n3 does not."""
    w = thin(n, 1.0)
    g = w["geom"]
    at = np.random.default_rng(8).uniform(0.2, 0.8, (2, n, 1))
    edge = at[0] * (g[:, 1] - g[:, 0]) + at[1] * (g[:, 2] - g[:, 0]) + eps * (g[:, 3] - g[:, 0])
    g[:, 3:] = g[:, :3] + edge[:, None]
    return w


MANY = {1: 60000, 2: 60000, 3: 20000, 4: 5000, 5: 500, 6: 500, 7: 500}


@pytest.mark.parametrize("kind", ["thin", "flat"])
@pytest.mark.parametrize("p", range(1, 8))
def test_adjoint_of_thin_and_flat_elements(p, kind):
    """The FP32 adjoints against the FP64 ones (the bound of test_thin_accuracy:
    the three products of n3 . c3 round as the two of n3 do), and zero gradients
    where the forward flags an element."""
    def make(n, eps):
        return thin(n, eps, fractions(n)) if kind == "thin" else flat(n, eps)
    w = make({1: 2000, **SAMPLE}[p], 1e-10)
    for got, want in zip(adjoints(w, p, "fp32"), adjoints(w, p, "fp64")):
        assert float(((got[4] - want[4]).abs() / want[4].abs()).max()) < 4e-5
    n = MANY[p]
    w = make(n, -5e-15)
    assert (forward(w, "fp32", p)[2] == NEGATIVE).all()
    for grads in adjoints(w, p, "fp32"):
        for t in grads:
            assert not t.any(), int(t.reshape(n, -1).any(1).sum())
