"""The launch-graph option on a map whose scans change between the one-kernel path and the ray list, and scans
captured into the caller's own graph mixed with direct calls."""
import time

import numpy as np
import pytest

from paper_2310_05766_gb300 import synth
from helpers import assert_same, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PARAMS = dict(dims=(128, 128, 64), voxel_size=0.1, tau=0.3, w_max=64, delta_z=0.05, r_min=0.3, r_max=6.0)


def _case(sizes, reduce=0):
    p = synth.params_dict(PARAMS["dims"], 0.1, 0.3, 64, 0.05, 0.3, 6.0, reduce, (-64, -64, -32))
    rng = np.random.default_rng(sum(sizes))
    scans, poses = [], []
    for i, n in enumerate(sizes):
        d = rng.normal(size=(n, 3))
        pts = np.zeros((n, 4), np.float32)
        pts[:, :3] = d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(0.5, 5.0, (n, 1))
        scans.append(pts)
        poses.append(synth.pose12(synth.rot_zyx(0.3 + 0.1 * i, 0.1, -0.1), np.array([0.05 * i, 0.1, -0.02])))
    return p, scans, poses


@pytest.mark.parametrize("reduce", [0, 1])
def test_launch_graph_alternating_sizes(reduce):
    """Sizes on both sides of the change of path: exact, and at about the host time of scans of one size."""
    from paper_2310_05766_gb300 import binding as b
    sizes = [32768, 32769, 5, 60000, 32000, 40000]
    p, scans, poses = _case(sizes, reduce)
    m = b.TsdfMap(p)
    try:
        b.tsdf_set_option(m.handle, b.TSDF_OPT_LAUNCH_GRAPH, 1)
        dev = [torch.from_numpy(s).cuda() for s in scans]
        stats = []
        for d, q in zip(dev, poses):
            m.integrate(d, q)
            stats.append(m.stats())
        v, w = m.read()
        assert_same((v, w, stats, m.origin), run_oracle(p, [("scan", s, q) for s, q in zip(scans, poses)]))

        def host_us(ids):
            best = None
            for _ in range(5):
                torch.cuda.synchronize()
                t = time.perf_counter()
                for i in ids:
                    m.integrate(dev[i], poses[i])
                t = (time.perf_counter() - t) * 1e6 / len(ids)
                best = t if best is None else min(best, t)
            torch.cuda.synchronize()
            return best

        same = host_us([3] * 20)
        assert host_us([3, 4] * 10) < 3 * same
    finally:
        m.close()


@pytest.mark.parametrize("sizes", [[40000, 60000, 50000], [2000, 60000, 40000], [60000, 3000, 32769]])
def test_captured_scans_mixed_with_direct_calls(sizes):
    """Scans captured into the caller's graphs, one and three at a time, replayed in any order among direct calls:
    the same map as the scans in that order."""
    from paper_2310_05766_gb300 import binding as b
    p, scans, poses = _case(sizes)
    m = b.TsdfMap(p)
    try:
        dev = [torch.from_numpy(s).cuda() for s in scans]
        order = []

        def direct(i):
            m.integrate(dev[i], poses[i])
            order.append(i)

        for i in range(3):
            direct(i)
        m.stats()
        graphs = []
        for ids in ([0], [1], [0, 1, 2]):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                for i in ids:
                    m.integrate(dev[i], poses[i])
            graphs.append((g, ids))
        rng = np.random.default_rng(sum(sizes))
        for k in rng.integers(0, 6, 24):
            if k < 3:
                graphs[k][0].replay()
                order.extend(graphs[k][1])
            else:
                direct(int(k) - 3)
        stats = m.stats()
        v, w = m.read()
        ref = run_oracle(p, [("scan", scans[i], poses[i]) for i in order])
        assert_same((v, w, [stats], m.origin), (ref[0], ref[1], ref[2][-1:], ref[3]))
    finally:
        m.close()
