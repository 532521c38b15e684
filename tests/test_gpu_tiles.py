"""Kernels that split a level into tiles, lanes or register blocks, at the sizes where the split can go
wrong: levels smaller than a tile, ragged last tiles, remainders of a warp's or block's share, both sides
of the size rules, the fewest and the most basis columns.

Tolerances (relative l2), those of the parity tests for the same quantities: FP64 applies 1e-12, FP64
transfers and smoothers 1e-11 (inverses by another factorisation than the oracle's), FP64 cycles at mild
contrast 1e-12; FP32 applies 2e-5, FP32 smoothers, transfers and cycles at mild contrast 1e-4 (inverses
stored in single precision)."""
import numpy as np
import pytest

from gpu_helpers import context, dev, host, oracle, random_free, rel, sinker, torch
from oracle.fem import Level
from oracle.qk import HierarchyK, LevelK, robust_prolongation_k, star_patches_k
from synthetic import problems as P

from paper_2107_00820_gb300 import Batch, Context, alstokes as A

pytestmark = pytest.mark.gpu

F32, F64 = A.ALS_PREC_FP32, A.ALS_PREC_FP64


def _zeros(n, prec):
    return torch.zeros(n, dtype=torch.float32 if prec == F32 else torch.float64, device="cuda")


def _dt(prec):
    return torch.float32 if prec == F32 else torch.float64


# 2D, FP32: tiles of 8 x 8 cells.  4: less than one; 20 x 12, 36 x 20, 18 x 34: ragged last tiles on every
# level, in both axes; sweeps 1 and 8: no earlier column, and no room for the norm beside eight dots
@pytest.mark.parametrize("n,levels,sweeps", [((4, 4), 2, 5), ((20, 12), 3, 1), ((36, 20), 3, 3), ((18, 34), 2, 8),
                                             ((16, 8), 2, 2)])
@pytest.mark.parametrize("cycle", [A.ALS_CYCLE_V, A.ALS_CYCLE_F])
def test_tiled_2d_cycle(n, levels, sweeps, cycle):
    pb = sinker(2, n, levels, 10.0, dr=1e2, seed=71)
    ctx = context(pb, sweeps=sweeps, cycle=cycle)
    H = oracle(pb, steps=sweeps, cycle="F" if cycle == A.ALS_CYCLE_F else "V")
    b = random_free(H.levels[-1], 72)
    x = _zeros(b.shape[0], F32)
    ctx.vcycle(dev(b, torch.float32), x, F32)
    assert rel(host(x), H.cycle(b)) <= 1e-4


def test_tiled_2d_cycle_merged_equals_single():
    """Ragged 2D levels beside a 3D instance: the merged launches give the single cycles' bits, boundary
    values in the right-hand sides included."""
    pbs = [sinker(2, (20, 12), 2, 10.0, 1e2, 73), sinker(2, (36, 20), 3, 10.0, 1e2, 74), sinker(3, 4, 2, 10.0, 1e2, 75)]
    opts = {"mode": A.ALS_MODE_MIXED, "schur": A.ALS_SCHUR_P2, "sweeps": 3}
    batch = Batch([{"dim": p.d, "n": p.n, "levels": p.levels, "coeffs": p.mu, "gamma": p.gamma, "options": opts}
                   for p in pbs])
    rng = np.random.default_rng(76)
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


def test_tiled_2d_cycle_wait_timeout_is_reported_and_recoverable():
    """With the poll limit of the waits for the stars' inverses at 0 every tile gives up at once, waits for the
    copies in flight and returns; the call reports the timeout, and the next one is as before."""
    pb = sinker(2, (20, 12), 2, 10.0, dr=1e2, seed=77)
    ctx = context(pb)
    b = dev(np.random.default_rng(78).standard_normal(ctx.nu()), torch.float32)
    x0, x1 = torch.zeros_like(b), torch.zeros_like(b)
    ctx.vcycle(b, x0, F32)
    ctx.set_wait_limit(0)
    with pytest.raises(A.ALSError) as e:
        ctx.vcycle(b, torch.zeros_like(b), F32)
    assert e.value.status == A.ALS_ETIMEOUT
    ctx.set_wait_limit(-1)
    ctx.vcycle(b, x1, F32)
    assert torch.equal(x0, x1)


# transfers: 2D tiles of 4 x 4 coarse cells (FP32) and of 8 x 16 coarse nodes; 3D of 8 x 4 x 4 coarse nodes, four
# fine nodes a thread
@pytest.mark.parametrize("d,n", [(2, (4, 4)), (2, (20, 12)), (2, (16, 34)), (3, (6, 10, 4)), (3, (16, 6, 8)), (3, (4, 4, 6))])
@pytest.mark.parametrize("transfer", [A.ALS_TRANSFER_ROBUST, A.ALS_TRANSFER_STANDARD])
@pytest.mark.parametrize("prec", [F64, F32])
def test_transfer_tiles(d, n, transfer, prec):
    pb = sinker(d, n, 2, 10.0, dr=1e2, seed=79)
    ctx = context(pb, transfer=transfer)
    H = oracle(pb, smoother="richardson", steps=1, transfer="robust" if transfer == A.ALS_TRANSFER_ROBUST else "standard")
    c, f = H.levels[0], H.levels[1]
    tol = 1e-11 if prec == F64 else 1e-4
    xc, xf = random_free(c, 80), _zeros(f.mesh.nu, prec)
    ctx.prolong(1, dev(xc, _dt(prec)), xf, prec)
    assert rel(host(xf), H.P[1] @ xc) <= tol
    rf, rc = random_free(f, 81), _zeros(c.mesh.nu, prec)
    ctx.restrict(1, dev(rf, _dt(prec)), rc, prec)
    assert rel(host(rc), H.P[1].T @ rf) <= tol


# stars: FP64 rows 256 a block over star boundaries (3 x 3, 7 x 3, 9 x 5, 3^3, 3 x 7 x 3 and 5 x 3 x 3 interior stars),
# every kind of boundary star; FP32 2D groups of 32 lanes
@pytest.mark.parametrize("d,n", [(2, (4, 4)), (2, (8, 4)), (2, (10, 6)), (3, (4, 4, 4)), (3, (4, 8, 4)), (3, (6, 4, 4))])
@pytest.mark.parametrize("prec", [F64, F32])
def test_star_products_at_remainders(d, n, prec):
    pb = sinker(d, n, 2, 10.0, dr=1e2, seed=82)
    ctx = context(pb)
    H = oracle(pb, smoother="richardson", steps=1)
    r = random_free(H.levels[1], 83)
    z = _zeros(r.shape[0], prec)
    ctx.star_smooth(1, dev(r, _dt(prec)), z, prec)
    assert rel(host(z), H.patches[1].apply(r)) <= (1e-11 if prec == F64 else 1e-4)


# 3D cell applies: FP64 line form below 2500 cells, register form (10 cells a warp) from there on
@pytest.mark.parametrize("n", [(14, 12, 14), (14, 14, 14)])
def test_cell_applies_about_the_fp64_rule(n):
    pb = sinker(3, n, 2, 1e2, dr=1e4, seed=84)
    ctx = context(pb)
    lv = Level(3, pb.n, pb.mu[1], pb.gamma)
    x = np.random.default_rng(85).standard_normal(lv.mesh.nu)
    y = _zeros(lv.mesh.nu, F64)
    ctx.apply_agamma(dev(x), y, 1)
    assert rel(host(y), lv.A @ x) <= 1e-12


# FP32 line form below 5000 cells, register form (32 cells a block) from there on, against FP64
@pytest.mark.parametrize("n", [(20, 12, 20), (20, 16, 16)])
@pytest.mark.parametrize("schur", [A.ALS_SCHUR_P1, A.ALS_SCHUR_P2])
def test_cell_applies_about_the_fp32_rule(n, schur):
    pb = sinker(3, n, 3, 1e2, dr=1e4, seed=86)
    ctx = context(pb, schur=schur)
    x = np.random.default_rng(87).standard_normal(ctx.nu()).astype(np.float32).astype(np.float64)
    y32, y64 = _zeros(x.shape[0], F32), _zeros(x.shape[0], F64)
    ctx.apply_agamma(dev(x, torch.float32), y32, 2, F32)
    ctx.apply_agamma(dev(x), y64, 2)
    assert rel(host(y32), host(y64)) <= 2e-5


# the smoother's reductions with 1 .. 8 columns, 3D, both precisions
@pytest.mark.parametrize("sweeps", [1, 2, 6, 7, 8])
def test_gmres_columns(sweeps):
    pb = sinker(3, (6, 4, 4), 2, 1.0, dr=1e2, seed=88)
    ctx = context(pb, sweeps=sweeps)
    H = oracle(pb, steps=sweeps)
    b = random_free(H.levels[-1], 89)
    ref = H.vcycle(b)
    x, x32 = _zeros(b.shape[0], F64), _zeros(b.shape[0], F32)
    ctx.vcycle(dev(b), x)
    assert rel(host(x), ref) <= 1e-12
    ctx.vcycle(dev(b, torch.float32), x32, F32)
    assert rel(host(x32), ref) <= 1e-4


# order 3, 2D: FP32 cells 16 a warp, two lanes each (4; 32 + 3; 64 less 4), FP64 a warp a cell
@pytest.mark.parametrize("n", [(2, 2), (5, 7), (10, 6)])
@pytest.mark.parametrize("prec", [F64, F32])
def test_q3_cells_2d(n, prec):
    pb = P.sinker_problem_k(n, 1, 3, 4, 0.1, 200.0, 1e3, 10.0, 1e2, 90)
    ctx = Context(2, pb.n, 1, pb.mu, pb.gamma, order=3)
    lv = LevelK(2, pb.n, 3, pb.mu[0], pb.gamma)
    x = np.random.default_rng(91).standard_normal(lv.mesh.nu)
    y = _zeros(lv.mesh.nu, prec)
    ctx.apply_agamma(dev(x, _dt(prec)), y, 0, prec)
    assert rel(host(y), lv.A @ x) <= (1e-12 if prec == F64 else 2e-5)


# order 3: FP32 cycles on ragged levels (the cells form the nodal sums of the stars), 2D and 3D
@pytest.mark.parametrize("d,n", [(2, (6, 10)), (2, (4, 4)), (3, (4, 4, 8))])
def test_q3_cycle_fp32(d, n):
    pb = P.sinker_problem_k(n, 2, 3, 4, 0.1, 200.0, 1e2, 10.0, 1.0, 92, d=d)
    ctx = Context(d, pb.n, 2, pb.mu, pb.gamma, order=3, sweeps=3)
    H = HierarchyK(d, pb.n, 3, pb.mu, pb.gamma, steps=3)
    lv = H.levels[-1]
    b = np.random.default_rng(93).standard_normal(lv.mesh.nu)
    b[lv.bdof] = 0.0
    x = _zeros(b.shape[0], F32)
    ctx.vcycle(dev(b, torch.float32), x, F32)
    assert rel(host(x), H.vcycle(b)) <= 1e-4


# order 3, 2D transfers on a ragged level
def test_q3_transfers_ragged():
    pb = P.sinker_problem_k((6, 10), 2, 3, 4, 0.1, 200.0, 1e2, 10.0, 1.0, 94)
    ctx = Context(2, pb.n, 2, pb.mu, pb.gamma, order=3)
    c = LevelK(2, pb.level_n[0], 3, pb.mu[0], pb.gamma)
    f = LevelK(2, pb.n, 3, pb.mu[1], pb.gamma)
    P_ = robust_prolongation_k(c.mesh, f)[0]
    xc = np.random.default_rng(95).standard_normal(c.mesh.nu)
    xc[c.bdof] = 0.0
    rf = np.random.default_rng(96).standard_normal(f.mesh.nu)
    rf[f.bdof] = 0.0
    xf, rc = _zeros(f.mesh.nu, F64), _zeros(c.mesh.nu, F64)
    ctx.prolong(1, dev(xc), xf)
    assert rel(host(xf), P_ @ xc) <= 1e-11
    ctx.restrict(1, dev(rf), rc)
    assert rel(host(rc), P_.T @ rf) <= 1e-11


# order 3, 3D FP32 stars: fewer and more interior stars (27, 175 = 7 x 5 x 5) than the ring kernel has blocks, and
# the boundary stars of a face, an edge and a corner
@pytest.mark.parametrize("n", [(4, 4, 4), (8, 6, 6)])
def test_q3_3d_star_ring(n):
    pb = P.sinker_problem_k(n, 2, 3, 4, 0.1, 200.0, 1e2, 10.0, 1.0, 97, d=3)
    ctx = Context(3, pb.n, 2, pb.mu, pb.gamma, order=3)
    r = np.random.default_rng(98).standard_normal(ctx.nu()).astype(np.float32).astype(np.float64)
    z32, z64 = _zeros(r.shape[0], F32), _zeros(r.shape[0], F64)
    ctx.star_smooth(1, dev(r, torch.float32), z32, F32)
    ctx.star_smooth(1, dev(r), z64)
    if n == (4, 4, 4):
        lv = LevelK(3, pb.n, 3, pb.mu[1], pb.gamma)
        free = r.copy()
        free[lv.bdof] = 0.0
        assert rel(host(z64), star_patches_k(lv).apply(free)) <= 1e-11
    assert rel(host(z32), host(z64)) <= 1e-4
    ctx.set_wait_limit(0)
    with pytest.raises(A.ALSError) as e:
        ctx.star_smooth(1, dev(r, torch.float32), torch.zeros_like(z32), F32)
    assert e.value.status == A.ALS_ETIMEOUT
    ctx.set_wait_limit(-1)
    z1 = torch.zeros_like(z32)
    ctx.star_smooth(1, dev(r, torch.float32), z1, F32)
    assert torch.equal(z32, z1)


# the tiled 2D cycle with tensor coefficients (C = M M^T + I / 2 at every point), and with the P2 pairing's per-cell
# W^-1, against the FP64 cycle
@pytest.mark.parametrize("tensor,schur", [(True, A.ALS_SCHUR_P1), (True, A.ALS_SCHUR_P2), (False, A.ALS_SCHUR_P2)])
def test_tiled_2d_cycle_coefficients(tensor, schur):
    n, levels = (20, 12), 3
    if tensor:
        rng, iu = np.random.default_rng(99), np.triu_indices(3)
        Cs = []
        for l in range(levels):
            m = rng.standard_normal((n[0] * n[1] // 4 ** (levels - 1 - l), 9, 3, 3))
            Cs.append(np.einsum("cqij,cqkj->cqik", m, m) + 0.5 * np.eye(3))
        ctx = Context(2, n, levels, [np.ascontiguousarray(C[:, :, iu[0], iu[1]]) for C in Cs], 1.0,
                      mu_eff=[np.ascontiguousarray(C[:, :, 0, 0] / 2) for C in Cs], schur=schur, sweeps=3)
    else:
        ctx = context(sinker(2, n, levels, 1.0, dr=1e2, seed=99), schur=schur, sweeps=3)
    b = np.random.default_rng(100).standard_normal(ctx.nu()).astype(np.float32).astype(np.float64)
    x32, x64 = _zeros(b.shape[0], F32), _zeros(b.shape[0], F64)
    ctx.vcycle(dev(b, torch.float32), x32, F32)
    ctx.vcycle(dev(b), x64)
    assert rel(host(x32), host(x64)) <= 1e-4
