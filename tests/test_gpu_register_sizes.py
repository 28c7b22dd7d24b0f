"""Normal equations of scan-to-map registration against the oracle at the sizes where the kernel's partition of
the points changes (one point, a warp, a CTA, one point per thread of the device and beyond), on windows whose
codes are mostly truncated: a point between eight truncated voxels is used or not as the interpolation in
binary64 rounds. The tolerance is that of a sum of the same binary64 terms in another order."""
import numpy as np
import pytest

import oracle
from paper_2310_05766_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [0.2, 0.3, 0.6])
@pytest.mark.parametrize("n", [0, 1, 31, 33, 192, 193, 29184, 29185, 60001])
def test_register_system_sizes(n, tau):
    from paper_2310_05766_gb300 import binding as b
    p = synth.params_dict((32, 16, 64), 0.1, tau, 64, 0.0, 0.1, 10.0, 0, (-16, 8, -32))
    rng = np.random.default_rng(n + int(tau * 10))
    shape = (64, 16, 32)
    z = np.arange(64)[:, None, None] + rng.uniform(-0.4, 0.4, shape)
    value = np.rint(np.clip((z - 20) * 6000, -32767, 32767)).astype(np.int16)
    weight = rng.integers(0, 40, shape).clip(0, 5).astype(np.int16)
    pts = np.zeros((n, 4), np.float32)
    pts[:, :3] = rng.uniform((-1.9, 0.5, -3.6), (1.9, 2.7, 3.6), (n, 3))
    pts[::17, 1] = np.nan
    pose = synth.pose12(synth.rot_zyx(0.05, -0.02, 0.03), np.array([0.01, 0.02, -0.03]))
    m, om = b.TsdfMap(p), oracle.OracleMap(p)
    try:
        m.write(value, weight)
        om.load_window(value, weight)
        dev = torch.from_numpy(pts).cuda() if n else torch.zeros((0, 4), device="cuda")
        got, ref = b.tsdf_register_system(m.handle, dev, pose), om.register_system(pts, pose)
        assert got[28] == ref[28]
        assert np.allclose(got, ref, rtol=1e-9, atol=1e-12 * np.abs(ref).max())
    finally:
        m.close()
