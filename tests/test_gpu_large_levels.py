"""Levels whose reductions have more blocks than every consumer adds up for itself (a kernel folds the partials in
between): the finest of 512^2, 48^3 and, at order 3, 288^2 cells."""
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_helpers import context, dev, host, rel, sinker, torch
from synthetic import problems as P

from paper_2107_00820_gb300 import Batch, alstokes as A

pytestmark = pytest.mark.gpu

F32, F64 = A.ALS_PREC_FP32, A.ALS_PREC_FP64
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _composed_cycle(ctx, b, sweeps):
    """The V-cycle from the context's own single steps, with GMRES(s) and its sums formed by torch in 64 bits."""
    def zeros(l):
        return torch.zeros(ctx.nu(l), dtype=torch.float64, device="cuda")

    def apply(l, x):
        y = zeros(l)
        ctx.apply_agamma(x, y, l)
        return y

    def smooth(l, x, b):
        V, Z, H = [b - apply(l, x)], [], torch.zeros(sweeps + 1, sweeps, dtype=torch.float64)
        beta = V[0].norm()
        V[0] = V[0] / beta
        for j in range(sweeps):
            Z.append(zeros(l))
            ctx.star_smooth(l, V[j], Z[j])
            w = apply(l, Z[j])
            h = torch.stack(V) @ w
            w = w - h @ torch.stack(V)
            H[:j + 1, j], H[j + 1, j] = h.cpu(), float(w.norm())
            V.append(w / w.norm())
        e = torch.zeros(sweeps + 1, 1, dtype=torch.float64)
        e[0] = float(beta)
        y = torch.linalg.lstsq(H, e).solution[:, 0]
        return x + y.cuda() @ torch.stack(Z)

    def cycle(l, b):
        x = zeros(l)
        if l == 0:
            ctx.coarse_solve(b, x)
            return x
        x = smooth(l, x, b)
        rc, xf = zeros(l - 1), zeros(l)
        ctx.restrict(l, b - apply(l, x), rc)
        ctx.prolong(l, cycle(l - 1, rc), xf)
        return smooth(l, x + xf, b)

    return cycle(ctx.levels - 1, b)


# tolerances of the parity tests for cycles at mild contrast
@pytest.mark.parametrize("d,n,levels,order", [(2, 512, 7, 2), (3, 48, 5, 2), (2, 288, 6, 3)])
def test_cycle_on_a_folding_level(d, n, levels, order):
    if order == 2:
        pb = sinker(d, n, levels, 1.0, 1e2, 21)
    else:
        pb = P.sinker_problem_k((n,) * d, levels, order, 8, 0.1, 200.0, 1e2, 10.0, 1.0, 21, d=d)
    ctx = context(pb, sweeps=3, order=order)
    b = torch.randn(ctx.nu(), dtype=torch.float32, device="cuda", generator=torch.Generator("cuda").manual_seed(22))
    x32, x64 = torch.zeros_like(b), torch.zeros_like(b, dtype=torch.float64)
    ctx.vcycle(b, x32, F32)
    ctx.vcycle(b.double(), x64)
    ref = host(_composed_cycle(ctx, b.double(), 3))
    assert rel(host(x64), ref) <= 1e-12
    assert rel(host(x32), ref) <= 1e-4


def test_merged_cycle_with_a_folding_level():
    """A large instance beside small ones: the merged launches give the single cycles' bits."""
    pbs = [sinker(2, 512, 7, 1.0, 1e2, 23), sinker(2, 16, 2, 1.0, 1e2, 24), sinker(3, 8, 2, 1.0, 1e2, 25)]
    opts = {"mode": A.ALS_MODE_MIXED, "schur": A.ALS_SCHUR_P2, "sweeps": 3}
    batch = Batch([{"dim": p.d, "n": p.n, "levels": p.levels, "coeffs": p.mu, "gamma": p.gamma, "options": opts}
                   for p in pbs])
    rng = np.random.default_rng(26)
    bs = [dev(rng.standard_normal(s[0]), torch.float32) for s in batch.shapes]
    xs = [torch.zeros_like(b) for b in bs]
    batch.vcycle(bs, xs, F32)
    for pb, b, xm in zip(pbs, bs, xs):
        ctx = context(pb, **opts)
        x = torch.zeros_like(b)
        ctx.vcycle(b, x, F32)
        assert torch.equal(x, xm)
        ctx.close()
    batch.close()


def test_large_levels_in_one_piece_take_separate_kernels():
    """A 2D level of 32,768 vertices and more whose stars are stored whole (a switch) takes its smoother steps as
    separate kernels like one with split stars: the operator's cell kernel is timed there, and is not where a step is
    one launch."""
    code = """if True:
        import sys
        import numpy as np
        import torch
        sys.path.insert(0, "tests")
        from gpu_helpers import context, sinker
        from paper_2107_00820_gb300 import alstokes as A
        for n, separate in ((128, False), (192, True)):
            ctx = context(sinker(2, n, 6, 1.0, 1e2, 27), mode=A.ALS_MODE_MIXED, sweeps=2)
            ctx.profile(True)
            b = torch.randn(ctx.nu(), dtype=torch.float32, device="cuda")
            x = torch.zeros_like(b)
            ctx.vcycle(b, x, A.ALS_PREC_FP32)
            assert (ctx.profile_read_kernel(1)[1] > 0) == separate, n
            ctx.close()
    """
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, ALS_SPLIT_STARS="0"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
