"""ALS_FUSE_GATHER=0 (separate kernels for the node sums of the star outputs, and for every operation of the 2D FP32
order-2 cycle) against the default: the same bits where the sums run in the same order, the same results to FP32
rounding where they do not (tolerance of the FP32 cycles at mild contrast)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCRIPT = """if True:
    import sys
    import numpy as np
    import torch
    sys.path.insert(0, "tests")
    from gpu_helpers import context, dev, sinker
    from synthetic import problems as P
    from paper_2107_00820_gb300 import Context, alstokes as A
    out = {}
    cases = {"2d": (context(sinker(2, (20, 12), 3, 10.0, 1e2, 41), schur=A.ALS_SCHUR_P2)),
             "3d": (context(sinker(3, (8, 12, 8), 3, 10.0, 1e2, 42)))}
    for d, n in ((2, (10, 6)), (3, (4, 4, 6))):
        pb = P.sinker_problem_k(n, 2, 3, 4, 0.1, 200.0, 1e2, 10.0, 1.0, 43, d=d)
        cases["q3_%dd" % d] = Context(d, pb.n, 2, pb.mu, pb.gamma, order=3, sweeps=3)
    for name, ctx in cases.items():
        b = np.random.default_rng(44).standard_normal(ctx.nu())
        for dt, prec in ((torch.float32, A.ALS_PREC_FP32), (torch.float64, A.ALS_PREC_FP64)):
            x = torch.zeros(ctx.nu(), dtype=dt, device="cuda")
            ctx.vcycle(dev(b, dt), x, prec)
            out[name + "_" + str(dt)[-2:]] = x.cpu().numpy()
    np.savez(sys.argv[1], **out)
"""


@pytest.fixture(scope="module")
def both(tmp_path_factory):
    got = []
    for flag in ("1", "0"):
        path = str(tmp_path_factory.mktemp("fuse") / ("x%s.npz" % flag))
        r = subprocess.run([sys.executable, "-c", SCRIPT, path], cwd=ROOT, env=dict(os.environ, ALS_FUSE_GATHER=flag),
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
        got.append(dict(np.load(path)))
    return got


@pytest.mark.parametrize("case", ["2d_64", "3d_32", "3d_64", "q3_2d_32", "q3_2d_64", "q3_3d_32", "q3_3d_64"])
def test_same_bits(both, case):
    assert np.isfinite(both[0][case]).all()
    assert np.array_equal(both[0][case], both[1][case])


def test_2d_fp32_to_rounding(both):
    a, b = (g["2d_32"].astype(np.float64) for g in both)
    assert not np.array_equal(a, b)          # two forms
    assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
