"""Scans of every size class of the plain path against the CPU oracle, bit for bit: one point, the edges of
a warp and of the tiles of the one-kernel path, the sizes around the change to the ray list, and marches
long enough that several CTAs share a tile's steps."""
import numpy as np
import pytest

from paper_2310_05766_gb300 import synth
from helpers import assert_same, run_gpu, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _points(n, seed, lo, hi):
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    pts = np.zeros((n, 4), np.float32)
    pts[:, :3] = d * rng.uniform(lo, hi, (n, 1))
    pts[rng.random(n) < 0.2, 0] = np.nan          # beams without a return
    return pts


@pytest.mark.parametrize("reduce,flags", [(0, 0), (1, 1)])
@pytest.mark.parametrize("n", [1, 31, 33, 64, 255, 257, 2049, 29184, 29185, 32767, 32768, 32769, 58369])
def test_scan_sizes_exact(n, reduce, flags):
    p = synth.params_dict((64, 64, 64), 0.1, 0.25, 64, 0.05, 0.3, 6.0, reduce, (-32, -32, -32), flags)
    pose = synth.pose12(synth.rot_zyx(0.4, 0.1, -0.2), np.array([0.05, -0.1, 0.02]))
    steps = [("scan", _points(n, n, 0.5, 5.0), pose), ("scan", _points(n, n + 1, 0.5, 3.0), pose)]
    assert_same(run_gpu(p, steps, torch), run_oracle(p, steps), f"n={n}")


@pytest.mark.parametrize("reduce", [0, 1])
@pytest.mark.parametrize("n,tau", [(1, 6.0), (40, 3.0), (700, 1.5)])
def test_long_marches_exact(n, tau, reduce):
    """Few points, many steps: the steps of a tile are shared by several CTAs."""
    p = synth.params_dict((128, 64, 64), 0.05, tau, 64, 0.1, 0.3, 6.0, reduce, (-64, -32, -32))
    pose = synth.pose12(synth.rot_zyx(-0.3, 0.05, 0.1), np.array([0.02, 0.1, -0.05]))
    steps = [("scan", _points(n, 5 * n, 0.5, 2.5), pose)] * 2
    assert_same(run_gpu(p, steps, torch), run_oracle(p, steps), f"n={n} tau={tau}")


@pytest.mark.parametrize("reduce,flags", [(0, 0), (0, 2), (1, 0)])
@pytest.mark.parametrize("w_max", [1, 64, 32767])
def test_weighted_mean_extremes_exact(w_max, reduce, flags):
    """Eq. 1 / Eq. 2 on voxels of every weight up to the cap, values at both ends of the code range and at the
    roundings' ties, and on scans that put thousands of contributions into one voxel."""
    p = synth.params_dict((32, 32, 32), 0.1, 0.3, w_max, 0.2, 0.1, 6.0, reduce, (-16, -16, -16), flags)
    rng = np.random.default_rng(w_max + reduce)
    value = rng.choice(np.array([-32767, -32766, -1, 0, 1, 2, 16383, 32766, 32767], np.int16), (32, 32, 32))
    weight = rng.integers(0, w_max + 1, (32, 32, 32)).astype(np.int16)
    weight[::2] = w_max
    pose = synth.pose12(np.eye(3), np.zeros(3))
    pts = _points(3000, 3, 0.3, 1.5)
    pts[::3] = np.array([0.9, 0.4, 0.1, 0.0], np.float32)
    steps = [("scan", pts, pose)] * 2
    assert_same(run_gpu(p, steps, torch, prefill=(value, weight)), run_oracle(p, steps, prefill=(value, weight)), "mean")
