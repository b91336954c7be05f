"""Unlit calls of one or two pairs on both sides of the line above which tiles keep a texel window (six items and
pairs per CTA of the estimator's grid), against the oracle (tolerances: tests/parity.py)."""
import numpy as np
import pytest

import oracle
from tests.parity import assert_parity, run_both
from tests.test_gpu_fast_groups import _quads, _sphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nearest", [False, True], ids=["bilinear", "nearest"])
@pytest.mark.parametrize("make,pairs,many", [
    (lambda: _quads(700, 600), 1, False),
    (lambda: _quads(700, 600), 2, True),
    (lambda: _sphere(24, 40, 30, 288, 272, views=8), 2, True),
    (lambda: _sphere(24, 2, 2, 288, 272, views=8), 2, True),
], ids=["quads_1", "quads_2", "sphere_2", "sphere_2_texture_2x2"])
def test_windows_of_short_calls_match_oracle(make, pairs, many, nearest):
    import torch
    from paper_2404_09758_gb300 import FOOT_NEAREST
    sc = make()
    tg = np.random.default_rng(2).uniform(size=(sc.n_views, sc.height, sc.width, 3)).astype(np.float32)
    r = run_both(sc, tg, seed=13, it=2, views=list(range(sc.n_views)), pairs=pairs,
                 footprint=oracle.FOOT_NEAREST if nearest else 0,
                 gpu_kwargs={"footprint": FOOT_NEAREST} if nearest else {})
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert (r["bins"][0] * pairs > 6 * ctas) == many
    assert_parity(sc, r)
