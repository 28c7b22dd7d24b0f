"""Batches with many contribution items per warp: the march claims chunks of
them from a counter instead of striding over them. A small grid (1 % of the
device) brings small maps there; the smallest grid of the test has more items
than a whole device's, so both sides of the rule and a last chunk that is not
full are run. Every result equals the per-map call's, bit for bit."""
import pytest

from test_gpu_batch import _run_batch, _run_single, _same, _small_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fraction", [1, 3, 100])
@pytest.mark.parametrize("config,cta_cache", [(0, 1), (2, 0), (4, 1), (6, 1), (8, 1), (9, 0), (12, 1)])
def test_claimed_chunks_match_single_maps(fraction, config, cta_cache):
    from paper_2310_05766_gb300 import binding as b
    ws = _small_batch(7, seed=41)
    mb = _run_batch(b, ws, prefill_steps=1,
                    options={b.TSDF_BATCH_OPT_CONFIG: config, b.TSDF_BATCH_OPT_GRID_FRACTION: fraction,
                             b.TSDF_BATCH_OPT_CTA_BRICK_CACHE: cta_cache})
    ms = _run_single(b, ws, repeats=2)
    _same(b, mb, ms)
    for m in mb + ms:
        m.close()
