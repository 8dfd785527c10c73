"""The bytes and operations mgr_profile gives for the time passes of a 4D plan: what
such a pass cannot do without (every coarse slice read once), from level sizes alone."""
import numpy as np
import pytest

import paper_2105_12764_gb300 as mgr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("steps", [9, 10])
@pytest.mark.parametrize("dtype,prec,item,work_item", [(mgr.MGR_F64, mgr.MGR_PREC_NATIVE, 8, 8),
                                                       (mgr.MGR_F32, mgr.MGR_PREC_MIXED, 4, 8)])
def test_time_pass_work(steps, dtype, prec, item, work_item):
    shape = (steps, 17, 18, 19)
    ctx = mgr.Context(0)
    plan = mgr.Plan(ctx, shape, None, -1, dtype, prec)
    td = torch.float64 if dtype == mgr.MGR_F64 else torch.float32
    x, y = torch.randn(shape, dtype=td, device="cuda"), torch.empty(shape, dtype=td, device="cuda")
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    want, n = {}, list(shape)
    for l in range(plan.levels, 0, -1):
        m = [k // 2 + 1 for k in n]
        space, coarse = int(np.prod(n[1:])), int(np.prod(m[1:]))
        fine = n[0] - m[0]
        value = item if l == plan.levels else work_item
        if fine:
            want[l] = ((fine + 1) * (space * value + (space - coarse) * item) + fine * space * (value + item),
                       (fine + 1) * space + 4 * fine * space)
        n = m
    try:
        for op, name, src, dst in ((0, "time_coef", x, y), (1, "time_interp", y, x)):
            got = {r["level"]: (r["bytes"], r["flops"]) for r in plan.profile(op, src, dst, ws) if r["name"] == name}
            assert {l: got[l] for l in want} == want
    finally:
        plan.close()
        ctx.close()
