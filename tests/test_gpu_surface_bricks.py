"""Surface points and triangles of windows as small as one brick, of uneven shapes and at every ring offset,
on random voxels (values at both ends of the code range and around zero, so that vertices come within a
rounding of their corners and triangles degenerate), against the oracle as exact sets."""
import numpy as np
import pytest

import oracle
from paper_2310_05766_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(a):
    a = np.asarray(a, np.float32)
    if not len(a):
        return np.zeros((0, 0), np.float32)
    a = np.ascontiguousarray(a.reshape(len(a), -1))
    return a[np.lexsort(a.T[::-1])]


def _cyclic(tri):
    """Each triangle rotated so that its smallest vertex comes first (its orientation kept)."""
    t = np.asarray(tri, np.float32).reshape(-1, 3, 3)
    keys = [tuple(map(tuple, x)) for x in t.tolist()]
    return _rows(np.array([x[k:] + x[:k] for x in keys for k in [min(range(3), key=lambda i: x[i:] + x[:i])]],
                          np.float32).reshape(len(t), 9))


@pytest.mark.parametrize("dims", [(8, 8, 8), (8, 16, 32), (32, 8, 16)])
@pytest.mark.parametrize("origin", [(0, 0, 0), (-24, 8, 40), (1 << 20, -(1 << 20), 16)])
@pytest.mark.parametrize("kind", ["noise", "extremes", "sparse"])
def test_random_windows_exact(dims, origin, kind):
    from paper_2310_05766_gb300 import binding as b
    p = synth.params_dict(dims, 0.05, 0.2, 64, 0.05, 0.3, 5.0, 0, origin)
    rng = np.random.default_rng(dims[0] * 100 + abs(origin[0]) % 97)
    shape = dims[::-1]
    if kind == "extremes":
        value = rng.choice(np.array([-32767, -1, 0, 1, 32767], np.int16), shape)
    else:
        value = rng.integers(-200, 200, shape).astype(np.int16)
    weight = rng.integers(0, 4, shape).astype(np.int16)
    if kind == "sparse":
        weight[rng.random(shape) < 0.6] = 0
    m, om = b.TsdfMap(p), oracle.OracleMap(p)
    try:
        m.write(value, weight)
        om.load_window(value, weight)
        for mw in (1, 2):
            assert np.array_equal(_rows(m.surface(mw).cpu().numpy()), _rows(om.surface(mw)))
            got, ref = m.mesh(mw).cpu().numpy(), om.mesh(mw)
            assert len(got) == len(ref) and np.array_equal(_cyclic(got), _cyclic(ref))
    finally:
        m.close()
