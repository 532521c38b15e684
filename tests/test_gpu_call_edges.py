"""Calls about the edges of the binding: what the autotuners time, how a call is ordered after the caller's stream,
which buffers it takes."""
import ctypes

import numpy as np
import pytest

from gpu_helpers import dev, sinker, torch

from paper_2107_00820_gb300 import Batch, Context, alstokes as A

pytestmark = pytest.mark.gpu

F32, F64 = A.ALS_PREC_FP32, A.ALS_PREC_FP64


def _batch(pbs, **opts):
    opts = {"mode": A.ALS_MODE_MIXED, "schur": A.ALS_SCHUR_P2, "sweeps": 3, **opts}
    return Batch([{"dim": p.d, "n": p.n, "levels": p.levels, "coeffs": p.mu, "gamma": p.gamma, "options": opts}
                  for p in pbs])


def test_merged_tuner_times_the_launches_that_run():
    """Tiled 2D levels launch neither star products nor interior solves of their own: beside a 3D instance the tuner
    leaves them out, and a level that has only those is not timed."""
    batch = _batch([sinker(2, (20, 12), 3, 10.0, 1e2, 31), sinker(2, (16, 16), 2, 10.0, 1e2, 32), sinker(3, 4, 2, 10.0, 1e2, 33)])
    batch.set_grouping(0)
    bs = [dev(np.random.default_rng(34).standard_normal(s[0]), torch.float32) for s in batch.shapes]
    batch.vcycle(bs, [torch.zeros_like(b) for b in bs], F32)
    assert min(batch.merged_tune(0, 1)[2]) > 0          # the 3D instance's
    assert batch.merged_tune(0, 2)[:3] == (0, 0, [0.0] * 6)
    batch.close()


@pytest.mark.parametrize("batch", [False, True])
def test_create_waits_for_the_default_stream(batch):
    """Coefficients that are still being written on the caller's stream, the default one included, are waited for."""
    pb = sinker(2, (16, 16), 2, 10.0, 1e2, 35)
    made = [dev(m) for m in pb.mu]
    late = [torch.zeros_like(m) for m in made]
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)          # about a tenth of a second
    for m, v in zip(late, made):
        m.copy_(v)
    if batch:
        ctx = Batch([{"dim": 2, "n": pb.n, "levels": 2, "coeffs": late, "gamma": pb.gamma, "options": {}}])
    else:
        ctx = Context(2, pb.n, 2, late, pb.gamma)
    ctx.close()


def test_merged_cycle_takes_vectors_of_any_alignment():
    """Vectors that do not start on a float's boundary are copied in and out like others."""
    batch = _batch([sinker(2, (20, 12), 2, 10.0, 1e2, 36), sinker(3, 4, 2, 10.0, 1e2, 37)])
    bs = [dev(np.random.default_rng(38).standard_normal(s[0]), torch.float32) for s in batch.shapes]
    xs = [torch.zeros_like(b) for b in bs]
    batch.vcycle(bs, xs, F32)

    def odd(t):
        raw = torch.zeros(4 * t.numel() + 1, dtype=torch.uint8, device="cuda")
        raw[1:] = t.view(torch.uint8)
        return raw

    b1, x1 = [odd(b) for b in bs], [odd(torch.zeros_like(b)) for b in bs]
    torch.cuda.synchronize()
    arrays = [(ctypes.c_void_p * 2)(*[t.data_ptr() + 1 for t in ts]) for ts in (b1, x1)]
    assert A.load().als_batch_vcycle(batch._b, F32, *arrays) == A.ALS_OK
    for x, raw in zip(xs, x1):
        assert torch.equal(x.view(torch.uint8), raw[1:])
    batch.close()
