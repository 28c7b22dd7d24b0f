"""Scans that find the pool full, on the one-kernel path and on the ray list: dropped whole and reported, the map
and its later scans unharmed, and at no more than the cost of a scan that fits."""
import numpy as np
import pytest

from paper_2310_05766_gb300 import synth
from helpers import assert_same, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _time_us(m, dev, pose, passes=20):
    best = None
    for _ in range(5):
        a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(passes):
            m.integrate(dev, pose)
        e.record()
        torch.cuda.synchronize()
        t = a.elapsed_time(e) * 1e3 / passes
        best = t if best is None else min(best, t)
    return best


@pytest.mark.parametrize("reduce", [0, 1])
@pytest.mark.parametrize("beams,azimuths", [(16, 1024), (64, 1024)])
def test_full_pool_drops_the_scan_and_nothing_else(beams, azimuths, reduce):
    from paper_2310_05766_gb300 import binding as b
    w = synth.workload_outdoor(n_scans=1, beams=beams, azimuths=azimuths, reduce=reduce)
    pts, pose = w.scans[0], w.poses[0]
    m = b.TsdfMap(w.params)
    try:
        dev = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
        b.tsdf_set_option(m.handle, b.TSDF_OPT_REDUCTION, b.TSDF_REDUCTION_POOL)
        stats = []
        for slots in (0, 64, 1000, 0):
            b.tsdf_set_option(m.handle, b.TSDF_OPT_POOL_BRICKS, slots)
            for _ in range(2):
                m.integrate(dev, pose)
                if slots:
                    with pytest.raises(b.TsdfError):
                        m.stats()
                else:
                    stats.append(m.stats())
        v, wt = m.read()
        assert_same((v, wt, stats, m.origin), run_oracle(w.params, [("scan", pts, pose)] * 4))
        fits = _time_us(m, dev, pose)
        b.tsdf_set_option(m.handle, b.TSDF_OPT_POOL_BRICKS, 64)
        m.integrate(dev, pose)
        assert _time_us(m, dev, pose) < 3 * fits
    finally:
        m.close()
