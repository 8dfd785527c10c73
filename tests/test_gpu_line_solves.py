"""Line solves at the edges of their layouts: lines staged 32, 16 and 8 at a time
and ones too long to be staged, one line more or less than a group, contiguous
lines shorter and longer than a CTA's rows; and the spatiotemporal fine slices,
odd and even counts of them.  Against the oracle at the library's tolerances (1e-12 FP64,
1e-5 FP32 and mixed)."""
import numpy as np
import pytest

import oracle
import paper_2105_12764_gb300 as mgr
from gpu_util import Runner, rel_linf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

FORMS = [(mgr.MGR_F64, 0, 1e-12), (mgr.MGR_F32, 0, 1e-5), (mgr.MGR_F32, 1, 1e-5)]


@pytest.fixture(scope="module")
def ctx():
    return mgr.Context(0)


def stretched(n):
    return np.concatenate([[0.0], np.cumsum(1.01 ** (np.arange(n - 1) % 200))])


def check(ctx, shape, dtype, prec, tol, levels):
    rng = np.random.default_rng(sum(shape))
    coords = [stretched(n) for n in shape]
    u = rng.standard_normal(shape)
    if dtype == mgr.MGR_F32:
        u = u.astype(np.float32)
    r = Runner(ctx, shape, coords, levels, dtype, prec)
    ref = oracle.decompose(u.astype(np.float64), coords, levels)
    assert rel_linf(r.decompose(u), ref) <= tol
    assert rel_linf(r.recompose(ref.astype(u.dtype)), u) <= tol
    r.close()


# (coarse lines 31 to 33, 15 to 17, 7 to 9 by 64 to 9000 long along y; many lines; z lines)
LINES = [(127, 300), (1300, 61), (1300, 63), (1300, 65), (2500, 33), (4000, 30), (6500, 17), (6500, 15), (12000, 40),
         (18000, 18), (9, 900, 37), (700, 5, 41), (3, 3, 3000), (400, 23, 25), (260, 370, 360)]


@pytest.mark.parametrize("shape", LINES)
@pytest.mark.parametrize("dtype,prec,tol", FORMS)
def test_lines(ctx, shape, dtype, prec, tol):
    check(ctx, shape, dtype, prec, tol, 1)


@pytest.mark.parametrize("shape", [(3, 6, 7, 8), (4, 9, 5, 6), (5, 5, 6, 7), (8, 7, 7, 5), (9, 12, 13, 14), (34, 5, 6, 5),
                                   (66, 4, 5, 3), (17, 20, 33, 41)])
@pytest.mark.parametrize("dtype,prec,tol", FORMS)
def test_fine_slices(ctx, shape, dtype, prec, tol):
    for levels in sorted({1, oracle.max_levels(shape)}):
        check(ctx, shape, dtype, prec, tol, levels)
