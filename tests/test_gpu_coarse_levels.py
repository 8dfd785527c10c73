"""The coarse levels of one cluster: fewer planes than CTAs and one plane more or
less than they share evenly, levels on either side of the size that every CTA
does by itself, grids of one plane or one row (their slabs lie along another
axis), axes of even length, grids that are coarse as a whole
(in place, too) and ones with a finer level above.  Against the oracle at the
library's tolerances (1e-12 FP64, 1e-5 FP32 and mixed)."""
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
    return np.concatenate([[0.0], np.cumsum(1.01 ** (np.arange(n - 1) % 200))])


SHAPES = [(17, 17, 17), (15, 18, 20), (16, 16, 16), (19, 19, 19), (3, 40, 60), (4, 44, 41), (6, 30, 31),
          (65, 11, 10), (129, 7, 9), (700, 3, 3), (9, 9, 9), (10, 10, 10), (11, 10, 10), (13, 9, 9), (5, 5, 5),
          (90, 91), (31, 33), (3, 2000), (2000, 4), (9,), (100,), (1030,), (1500,), (5000,),
          (33, 34, 35), (40, 3, 300), (130, 131), (16400,)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype,prec,tol", [(mgr.MGR_F64, 0, 1e-12), (mgr.MGR_F32, 0, 1e-5), (mgr.MGR_F32, 1, 1e-5)])
def test_coarse_levels(ctx, shape, dtype, prec, tol):
    rng = np.random.default_rng(sum(shape))
    coords = [stretched(n) for n in shape]
    u = rng.standard_normal(shape)
    if dtype == mgr.MGR_F32:
        u = u.astype(np.float32)
    for levels in sorted({1, oracle.max_levels(shape)}):
        r = Runner(ctx, shape, coords, levels, dtype, prec)
        ref = oracle.decompose(u.astype(np.float64), coords, levels)
        for inplace in (False, True):
            assert rel_linf(r.decompose(u, inplace), ref) <= tol, (levels, inplace)
            assert rel_linf(r.recompose(ref.astype(u.dtype), inplace), u) <= tol, (levels, inplace)
        r.close()
