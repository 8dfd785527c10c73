"""The level passes where their warps and strips end: coarse rows of one lane
group and one more or less (groups of 32 lanes share two with their
neighbours), several short rows per group, strips that start on the last node
of an axis, axes of even length, few planes.  Decomposition, recomposition
and the class-packed forms against the oracle at the library's tolerances
(1e-12 FP64, 1e-5 FP32 and mixed)."""
import zlib

import numpy as np
import pytest

import oracle
import paper_2105_12764_gb300 as mgr
from gpu_util import Runner, rel_linf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def ctx():
    return mgr.Context(0)


def stretched(n):
    return np.concatenate([[0.0], np.cumsum(1.01 ** np.arange(n - 1))])


# coarse widths 31, 32, 33, 61, 62 and 63 from odd and even lengths; 2 to 16 for
# rows shorter than a group; heights around 7, 10, 13 and 16 coarse rows
SHAPES = [(5, 19, 61), (4, 20, 62), (6, 26, 63), (3, 27, 64), (9, 13, 121), (8, 14, 122), (7, 33, 123), (5, 34, 124),
          (33, 25, 3), (34, 41, 4), (12, 70, 5), (40, 38, 6), (21, 24, 17), (26, 60, 31), (3, 3, 200), (61, 3), (62, 28),
          (15, 1001)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype,prec,tol", [(mgr.MGR_F64, 0, 1e-12), (mgr.MGR_F32, 0, 1e-5), (mgr.MGR_F32, 1, 1e-5)])
def test_strip_edges(ctx, shape, dtype, prec, tol):
    rng = np.random.default_rng(sum(shape))
    coords = [stretched(n) for n in shape]
    u = rng.standard_normal(shape)
    if dtype == mgr.MGR_F32:
        u = u.astype(np.float32)
    for levels in sorted({1, oracle.max_levels(shape)}):
        r = Runner(ctx, shape, coords, levels, dtype, prec)
        ref = oracle.decompose(u.astype(np.float64), coords, levels)
        assert rel_linf(r.decompose(u), ref) <= tol, (shape, levels)
        assert rel_linf(r.recompose(ref.astype(u.dtype)), u) <= tol, (shape, levels)
        packed = torch.empty(u.size, dtype=r.a.dtype, device="cuda")
        r.a.copy_(torch.from_numpy(u))
        r.plan.decompose_packed(r.a, packed, r.ws)
        r.plan.recompose_packed(packed, levels + 1, r.b, r.ws)
        torch.cuda.synchronize()
        assert rel_linf(packed.cpu().numpy(), oracle.pack_classes(ref, levels)) <= tol, (shape, levels)
        assert rel_linf(r.b.cpu().numpy(), u) <= tol, (shape, levels)
        r.plan.close()


# FP32 codes show the last bit of a coefficient when the tolerance is far below
# the field's precision; their checksums are those of the earlier level pass,
# whose codes the current one reproduces.
CODES = [
    ((45, 66, 71), mgr.MGR_PREC_NATIVE, 3505642234),
    ((45, 66, 71), mgr.MGR_PREC_MIXED, 3647058172),
    ((31, 34, 130), mgr.MGR_PREC_NATIVE, 2561608840),
    ((31, 34, 130), mgr.MGR_PREC_MIXED, 1467654686),
    ((64, 50, 93), mgr.MGR_PREC_NATIVE, 4191757017),
    ((64, 50, 93), mgr.MGR_PREC_MIXED, 626166548),
    ((131, 200), mgr.MGR_PREC_NATIVE, 3216810082),
    ((131, 200), mgr.MGR_PREC_MIXED, 2252108792),
]


@pytest.mark.parametrize("shape,prec,crc", CODES)
def test_fp32_codes_keep_their_values(ctx, shape, prec, crc):
    u = np.random.default_rng(sum(shape)).standard_normal(shape).astype(np.float32)
    plan = mgr.Plan(ctx, shape, [stretched(n) for n in shape], -1, mgr.MGR_F32, prec)
    x = torch.from_numpy(u).cuda()
    codes = torch.empty(u.size, dtype=torch.int32, device="cuda")
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    plan.decompose_quantized(x, codes, 1e-7, ws)
    torch.cuda.synchronize()
    got = zlib.crc32(codes.cpu().numpy().tobytes())
    plan.close()
    assert got == crc, (shape, prec)


@pytest.mark.parametrize("shape", [(33, 33, 33), (40, 37, 66), (34, 36, 130), (150, 171), (9, 33, 17, 18)])
@pytest.mark.parametrize("dtype", [mgr.MGR_F64, mgr.MGR_F32])
def test_infinite_coarse_value_stays_in_its_support(ctx, shape, dtype):
    """An infinite value on a coarse node reaches the nodes that are interpolated from it and no
    others: it is no coefficient, and the load vector of its level does not see it, at the ends of
    the axes either."""
    for at in (0, -1):
        r = Runner(ctx, shape, None, 1, dtype)
        c = np.random.default_rng(3).standard_normal(shape)
        c[(at,) * len(shape)] = np.inf
        v = r.recompose(c)
        near = np.zeros(shape, bool)
        near[tuple(slice(0, 2) if at == 0 else slice(-2 if n % 2 else -1, None) for n in shape)] = True
        assert np.array_equal(~np.isfinite(v), near), at
        r.close()
