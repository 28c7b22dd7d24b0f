"""First use of a map on a side stream while the default stream is busy: the buffers that a call allocates
then are filled before its kernels run, whatever the default stream still has to do."""
import numpy as np
import pytest

import oracle
from paper_2310_05766_gb300 import synth
from helpers import assert_same, run_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _busy_default_stream():
    """Copies that keep the default stream busy for tens of milliseconds."""
    a = torch.ones(1 << 28, device="cuda")
    c = torch.empty_like(a)
    torch.cuda.synchronize()
    for _ in range(60):
        c.copy_(a)
    return a, c


def _dirty_free_memory():
    """Memory that the next allocations may get back is not zero."""
    x = torch.full((1 << 26,), 7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("reduction", ["ATOMIC", "SORT", "POOL"])
@pytest.mark.parametrize("n", [2000, 40000])
def test_first_scan_on_side_stream(n, reduction):
    from paper_2310_05766_gb300 import binding as b
    p = synth.params_dict((128, 128, 64), 0.1, 0.3, 64, 0.05, 0.3, 6.0, 0, (-64, -64, -32))
    rng = np.random.default_rng(n)
    d = rng.normal(size=(n, 3))
    pts = np.zeros((n, 4), np.float32)
    pts[:, :3] = d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(0.5, 5.0, (n, 1))
    pose = synth.pose12(synth.rot_zyx(0.3, 0.1, -0.1), np.array([0.05, 0.1, -0.02]))
    _dirty_free_memory()
    m = b.TsdfMap(p)
    try:
        b.tsdf_set_option(m.handle, b.TSDF_OPT_REDUCTION, getattr(b, "TSDF_REDUCTION_" + reduction))
        dev = torch.from_numpy(pts).cuda()
        side = torch.cuda.Stream()
        busy = _busy_default_stream()
        with torch.cuda.stream(side):
            m.integrate(dev, pose)
            m.integrate(dev, pose)
            stats = m.stats()
        torch.cuda.synchronize()
        del busy
        v, w = m.read()
        got = (v, w, [stats], m.origin)
    finally:
        m.close()
    ref = run_oracle(p, [("scan", pts, pose)] * 2)
    assert_same(got, (ref[0], ref[1], ref[2][-1:], ref[3]), reduction)


@pytest.mark.parametrize("n", [100, 60001])
def test_first_registration_on_side_stream(n):
    from paper_2310_05766_gb300 import binding as b
    p = synth.params_dict((32, 16, 64), 0.1, 0.3, 64, 0.0, 0.1, 10.0, 0, (-16, 8, -32))
    rng = np.random.default_rng(n)
    shape = (64, 16, 32)
    value = np.rint(np.clip((np.arange(64)[:, None, None] + rng.uniform(-0.4, 0.4, shape) - 20) * 6000, -32767, 32767))
    value, weight = value.astype(np.int16), rng.integers(1, 5, shape).astype(np.int16)
    pts = np.zeros((n, 4), np.float32)
    pts[:, :3] = rng.uniform((-1.5, 0.9, -1.5), (1.5, 2.3, -0.9), (n, 3))
    pose = synth.pose12(synth.rot_zyx(0.05, -0.02, 0.03), np.array([0.01, 0.02, -0.03]))
    om = oracle.OracleMap(p)
    om.load_window(value, weight)
    ref = om.register_system(pts, pose)
    _dirty_free_memory()
    m = b.TsdfMap(p)
    try:
        m.write(value, weight)
        dev = torch.from_numpy(pts).cuda()
        side = torch.cuda.Stream()
        busy = _busy_default_stream()
        with torch.cuda.stream(side):
            got = [b.tsdf_register_system(m.handle, dev, pose) for _ in range(3)]
        torch.cuda.synchronize()
        del busy
        for g in got:
            assert g[28] == ref[28] > 0
            assert np.allclose(g, ref, rtol=1e-9, atol=1e-12 * np.abs(ref).max())
    finally:
        m.close()


def test_registration_leaves_its_stream_idle():
    """A registration synchronises its stream: whatever it returns, the stream has nothing left to do, and the
    next evaluation may use another one."""
    from paper_2310_05766_gb300 import binding as b
    p = synth.params_dict((64, 64, 64), 0.1, 0.3, 64, 0.0, 0.1, 10.0, 0, (-32, -32, -32))
    g = np.stack(np.meshgrid(*[np.arange(-32, 32) + 0.5] * 3, indexing="ij"), -1)[..., ::-1] * 0.1
    value = np.rint(np.clip(2.0 - np.linalg.norm(g, axis=-1), -0.3, 0.3) * 32767 / 0.3).astype(np.int16)
    rng = np.random.default_rng(3)
    d = rng.normal(size=(20000, 3))
    pts = np.zeros((20000, 4), np.float32)
    pts[:, :3] = d / np.linalg.norm(d, axis=1, keepdims=True) * 2.0
    pose = synth.pose12(synth.rot_zyx(0.01, -0.02, 0.01), np.array([0.02, -0.03, 0.01]))
    m = b.TsdfMap(p)
    try:
        m.write(value, np.ones_like(value))
        dev = torch.from_numpy(pts).cuda()
        far = dev + 1000.0
        streams = [torch.cuda.Stream() for _ in range(2)]
        ref = b.tsdf_register_system(m.handle, dev, pose)
        assert ref[28] > 10000
        for k in range(200):
            s = streams[k & 1]
            with torch.cuda.stream(s):
                got = b.tsdf_register_system(m.handle, dev, pose)
                assert s.query() and np.array_equal(got, ref)
                if k % 10 == 0:
                    with pytest.raises(b.TsdfError):
                        b.tsdf_register(m.handle, far, pose, iterations=3)
                    assert s.query()
                    b.tsdf_register(m.handle, dev, pose, iterations=2)
                    assert s.query()
    finally:
        m.close()


def test_device_bytes_count_registration():
    """What a map's first registration allocates on the device is in tsdf_map_device_bytes."""
    from paper_2310_05766_gb300 import binding as b
    p = synth.params_dict((64, 64, 64), 0.1, 0.3, 64, 0.0, 0.1, 10.0, 0, (-32, -32, -32))
    m = b.TsdfMap(p)
    try:
        before = b.tsdf_map_device_bytes(m.handle)
        pts = torch.zeros((100, 4), device="cuda")
        pose = synth.pose12(np.eye(3), np.zeros(3))
        b.tsdf_register_system(m.handle, pts, pose)
        after = b.tsdf_map_device_bytes(m.handle)
        assert after >= before + 512 * 32 * 8
        b.tsdf_register_system(m.handle, pts, pose)
        assert b.tsdf_map_device_bytes(m.handle) == after
    finally:
        m.close()
