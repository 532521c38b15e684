"""How the FP32 operations round: an FP32 result against the FP64 one over many problems, and sums that have to
be formed in one order everywhere."""
import numpy as np
import pytest

from gpu_helpers import context, dev, host, rel, sinker, torch

from paper_2107_00820_gb300 import alstokes as A

pytestmark = pytest.mark.gpu

F32, F64 = A.ALS_PREC_FP32, A.ALS_PREC_FP64


def _free(n, seed):
    """A random vector, zero at the boundary nodes, exact in FP32."""
    v = np.random.default_rng(seed).standard_normal((len(n),) + tuple(2 * m + 1 for m in reversed(n)))
    for a in range(1, v.ndim):
        np.moveaxis(v, a, 0)[0] = 0.0
        np.moveaxis(v, a, 0)[-1] = 0.0
    return v.astype(np.float32).astype(np.float64).ravel()


def test_2d_cycle_error_over_many_problems():
    """One FP32 cycle at contrast 1e6 has a few times the unit roundoff as its error, but a single problem's error
    varies by a factor of ten with the order of any sum, so the distribution is what is bounded.  Over 240 problems
    of this kind the median and the 90th percentile are 2.2e-7 and 3.1e-7 with the smoother's small numbers and its
    combinations of columns in double-float, 3.1e-7 and 5.8e-7 with these in plain FP32, 2.9e-7 and 5.4e-7 with one
    launch per operation and divisions in place of reciprocals.  The bounds are the geometric means of the first two."""
    n, levels, errs = (96, 96), 5, []
    for seed in range(80):
        ctx = context(sinker(2, n, levels, 100.0, 1e6, 1000 + seed), schur=A.ALS_SCHUR_P2, mode=A.ALS_MODE_MIXED)
        b = _free(n, 2000 + seed)
        x32 = torch.zeros(b.size, dtype=torch.float32, device="cuda")
        x64 = torch.zeros(b.size, dtype=torch.float64, device="cuda")
        ctx.vcycle(dev(b, torch.float32), x32, F32)
        ctx.vcycle(dev(b), x64)
        errs.append(rel(host(x32), host(x64)))
        ctx.close()
    assert np.median(errs) <= 2.6e-7
    assert np.quantile(errs, 0.9) <= 4.2e-7


# ragged tiles; sizes of one tile and less
@pytest.mark.parametrize("n", [(4, 4), (20, 12), (16, 34)])
def test_robust_prolongation_interpolates_as_the_standard_one(n):
    """With the stars' inverses set to 0 the robust prolongation is the interpolation alone, and that has the
    standard prolongation's bits: the robust correction amplifies a change of its rounding by gamma / mu."""
    pb = sinker(2, n, 2, 100.0, 1e4, 7)
    robust, standard = context(pb), context(pb, transfer=A.ALS_TRANSFER_STANDARD)
    stride = (18 * 19 // 2 + 3) // 4 * 4
    robust.load_patch_inverses(1, np.zeros((n[0] + 1) * (n[1] + 1) * stride))
    xc = dev(_free((n[0] // 2, n[1] // 2), 8), torch.float32)
    out = [torch.zeros(robust.nu(), dtype=torch.float32, device="cuda") for _ in range(2)]
    robust.prolong(1, xc, out[0], F32)
    standard.prolong(1, xc, out[1], F32)
    assert torch.equal(out[0], out[1])
