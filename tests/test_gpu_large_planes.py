"""Planes near the largest the library takes (2^31 elements), whose coarse levels
have rows so far apart that row index times pitch needs the clamp to the last row
before it fits in 32 bits (tests/test_row_offsets.py has the expression itself).

The oracle cannot run at this scale, but the method is a tensor product: with
u = a x b, the level values are a_l x b_l (both factors projected axis by axis) and
the coefficients a_l x b_l - (P a_l) x (P b_l), P the interpolant of the coarse
nodes, so 1D projections of the factors (`project`, compared with the oracle on
short ones) give whole rows of the result."""
import numpy as np
import pytest

import oracle
import paper_2105_12764_gb300 as mgr

pytestmark = pytest.mark.gpu

solve_banded = pytest.importorskip("scipy.linalg").solve_banded
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


def project(x, v):
    """Coarse nodes of the level with nodes x, and its values v there after the correction:
    v + M_c^-1 P^T M (v - P v), M and M_c the P1 mass matrices of the two levels."""
    n = len(x)
    coarse = np.array(sorted({*range(0, n, 2), n - 1}))
    c = v - np.interp(x, x[coarse], v[coarse])
    h = np.diff(x)
    g = np.zeros(n)
    g[:-1] += h * (2 * c[:-1] + c[1:]) / 6
    g[1:] += h * (c[:-1] + 2 * c[1:]) / 6
    fine = np.arange(1, n - 1, 2)
    left = (x[fine + 1] - x[fine]) / (x[fine + 1] - x[fine - 1])
    f = g[coarse]
    f[fine // 2] += left * g[fine]
    f[fine // 2 + 1] += (1 - left) * g[fine]
    hc = np.diff(x[coarse])
    band = np.zeros((3, len(coarse)))
    band[0, 1:] = band[2, :-1] = hc / 6
    band[1, :-1] += hc / 3
    band[1, 1:] += hc / 3
    return coarse, v[coarse] + solve_banded((1, 1), band, f)


class Factor:
    """One axis of a separable field: its values, projections and interpolants by level."""

    def __init__(self, v, L):
        self.N, self.L = len(v), L
        self.nodes, self.values, self.interp = [], [], []  # by level 0 .. L, on the full grid's nodes
        self.node_level = np.zeros(self.N, dtype=int)      # the level in which a node is fine (0: none)
        nodes, vals = np.arange(self.N), v
        for l in range(L, -1, -1):
            full, it = np.full(self.N, np.nan), np.full(self.N, np.nan)
            full[nodes] = vals
            if l:
                coarse, vals_c = project(nodes.astype(float), vals)
                it[nodes] = np.interp(nodes, nodes[coarse], vals[coarse])
                self.node_level[np.delete(nodes, coarse)] = l
            self.nodes.insert(0, nodes)
            self.values.insert(0, full)
            self.interp.insert(0, it)
            if l:
                nodes, vals = nodes[coarse], vals_c


def expected_row(fa, fb, r):
    """Row r of the decomposition of a x b."""
    out = np.empty(fb.N)
    level = np.maximum(fa.node_level[r], fb.node_level)
    for l in range(fa.L + 1):
        at = np.nonzero(level == l)[0]
        out[at] = fa.values[l][r] * fb.values[l][at]
        if l:
            out[at] -= fa.interp[l][r] * fb.interp[l][at]
    return out


def factors(shape, L):
    rng = np.random.default_rng(5)
    return [Factor(rng.standard_normal(n).astype(np.float32).astype(np.float64), L) for n in shape]


@pytest.mark.parametrize("shape", [(20, 36), (17, 50), (23, 41)])
def test_expected_rows_small(shape):
    fa, fb = factors(shape, oracle.default_levels(shape))
    ref = oracle.decompose(np.outer(fa.values[-1], fb.values[-1]))
    for r in range(shape[0]):
        np.testing.assert_allclose(expected_row(fa, fb, r), ref[r], rtol=0, atol=1e-12)


# 514 x 2097152: the level of 4 rows, 256 apart.  40000 x 53000: the level of 80
# rows, 512 apart.
@pytest.mark.parametrize("shape", [(514, 2_097_152), (40_000, 53_000)], ids=lambda s: "x".join(map(str, s)))
def test_large_planes(shape):
    ctx = mgr.Context(0)
    plan = mgr.Plan(ctx, shape, None, -1, mgr.MGR_F32)
    L = plan.levels
    fa, fb = factors(shape, L)
    a, b = (torch.from_numpy(f.values[L]).float().cuda() for f in (fa, fb))
    u = torch.outer(a, b)
    y, z = torch.empty_like(u), torch.empty_like(u)
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    scale = float(u.abs().max())
    # every coarsest row, and the nearest fine row of each level to the end of the axis
    rows = list(fa.nodes[0]) + [int(np.nonzero(fa.node_level == l)[0][-1]) for l in range(1, L + 1)]

    def check_rows(t):
        for r in rows:
            err = np.abs(t[r].cpu().numpy().astype(np.float64) - expected_row(fa, fb, r)).max() / scale
            assert err <= 1e-5, (r, err)

    def check_field():
        assert float((z - u).abs().max()) / scale <= 1e-5

    try:
        plan.decompose(u, y, ws)
        check_rows(y)
        plan.recompose(y, z, ws)
        check_field()
        # class-packed: the finest level reads its coefficients through 32-bit row offsets too
        plan.decompose_packed(u, y, ws)
        z.zero_()
        plan.recompose_packed(y, L + 1, z, ws)
        check_field()
        if shape[0] < 1000:
            return
        # batched (its autotuner times several shapes: not with the longest lines)
        y.zero_()
        z.zero_()
        torch.cuda.synchronize()
        assert ctx.batch_poll(ctx.batch_submit([(mgr.MGR_OP_DECOMPOSE, plan, u, y)]))[0] == mgr.MGR_OK
        check_rows(y)
        assert ctx.batch_poll(ctx.batch_submit([(mgr.MGR_OP_RECOMPOSE, plan, y, z)]))[0] == mgr.MGR_OK
        check_field()
    finally:
        plan.close()
        ctx.close()
