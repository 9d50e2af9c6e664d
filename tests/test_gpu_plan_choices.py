"""Stored and default choices of plans (include/fei.h)."""
import json

import numpy as np
import pytest

from paper_1310_1194_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_choices_of_other_kernels_are_not_applied(tmp_path):
    """A tuning cache written for an earlier revision of the kernels (its key
    held the GPU model and precision only) changes nothing, and stays in the
    file beside new choices."""
    from paper_1310_1194_gb300 import api
    plan = api.Plan(max_elem=8, precision="auto")
    before = [plan.choice(p) for p in range(1, 8)]
    old = {f"{torch.cuda.get_device_name()}|auto": {str(p): {"variant": 0, "grid_cap": 304, "tuned_ms": 1.0}
                                                    for p in range(1, 8)}}
    path = str(tmp_path / "tune.json")
    with open(path, "w") as fh:
        json.dump(old, fh)
    assert not plan.load_choices(path)
    assert [plan.choice(p) for p in range(1, 8)] == before and plan.kernel(4) == "sum_factorised"
    plan.set_choice(4, 0, 0)
    plan.save_choices(path)
    other = api.Plan(max_elem=8, precision="auto")
    assert other.load_choices(path) and other.kernel(4) == "tensor_core"
    with open(path) as fh:
        data = json.load(fh)
    assert len(data) == 2 and all(data[k] == v for k, v in old.items())


@pytest.mark.parametrize("n", [1, 300, 512, 513])
def test_untuned_plan_equals_the_direct_call(n):
    """Every precision and degree, on both sides of FEI_AUTO's 512 elements, and
    a mixed batch."""
    from paper_1310_1194_gb300 import api
    w = inputs.workload("mixed", n_max=n)
    a = [torch.from_numpy(np.ascontiguousarray(w[k][:n])).cuda() for k in ("geom", "K", "b", "c", "f")]
    degree = torch.from_numpy(np.ascontiguousarray(w["degree"][:n])).cuda()
    stream = torch.cuda.Stream()
    for precision in ("auto", "fp32", "fp64", "tc_f16x3", "sf_fp32"):
        plan = api.Plan(max_elem=n, precision=precision)
        for kw in [dict(p=p) for p in range(1, 6)] + [dict(degree=degree)]:
            with torch.cuda.stream(stream):
                got = plan.execute(*a, **kw)
                want = api.fei_integrate(*a, precision=precision, **kw)
            stream.synchronize()
            for x, y in zip(got[:3], want[:3]):
                assert torch.equal(x, y), (precision, kw.get("p"))
