"""Batched calls of one, two and five pairs of one, two and five assets (every pruning variant, with and without texel
windows, a CTA's shared memory handed from asset to asset, dense tiles), against the oracle asset by asset
(tests/test_gpu_batch.py's comparison)."""
import pytest

import oracle
import synth
from tests.test_gpu_batch import _check_against_oracle, _run_batch, _small_assets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    scs = _small_assets()
    return scs, [oracle.render_targets(sc, synth.target_scene(sc)) for sc in scs]


@pytest.mark.parametrize("n", [1, 2, 5])
@pytest.mark.parametrize("pairs", [1, 2, 5])
def test_short_batches_match_oracle(small, pairs, n):
    scs, targets = small[0][-n:], small[1][-n:]
    gs, bufs, sts, _ = _run_batch(scs, targets, pairs)
    assert sum(g.bin_stats()[0] for g in gs) > 0
    _check_against_oracle(scs, targets, bufs, sts, pairs)
