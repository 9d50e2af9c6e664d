"""The FP32 quadratic-loss adjoint against the FP64 one: v_q = G_q u by three
one-dimensional sums is no further off than one dense FP32 sum with a rounded
table, whose errors average out over the points of an element."""
import numpy as np
import pytest

from paper_1310_1194_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("p,dense", [(3, 6.6e-8), (4, 5.0e-8)])
def test_factor_roundings_do_not_add_up(p, dense):
    """rms over elements of the relative error of dL/dK; dense: the dense sum's
    (GB300, 2000 and 1500 of these elements), and a tenth for the sample."""
    from paper_1310_1194_gb300 import api
    n, s = 2000, api.nsh(p)
    w = inputs.workload("p4", n_max=n)
    a = [torch.from_numpy(np.ascontiguousarray(w[k][:n])).cuda() for k in ("geom", "K", "b", "c", "f")]
    u = torch.from_numpy(np.random.default_rng(p).standard_normal(n * s)).cuda()
    got, want = (api.fei_integrate_backward_quadratic(*a, u, p=p, precision=q)[1].reshape(n, -1) for q in ("fp32", "fp64"))
    err = (got - want).norm(dim=1) / want.norm(dim=1)
    assert float(err.pow(2).mean().sqrt()) < 1.1 * dense
