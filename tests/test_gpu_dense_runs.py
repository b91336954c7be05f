"""Dense tiles with explicit runs of pairs (pairs_per_item): fewer than the kernel runs at a time, ones that do not
divide the call's pairs, the longest; against the oracle (tolerances: tests/parity.py)."""
import numpy as np
import pytest

from tests.parity import assert_parity, run_both
from tests.test_gpu_fast_groups import _sphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [1, 5])
@pytest.mark.parametrize("ppi", [1, 2, 3, 7, 8, 13, 64])
def test_explicit_runs_of_dense_tiles_match_oracle(ppi, pairs):
    sc = _sphere(96, 40, 30, 32, 30)
    tg = np.random.default_rng(2).uniform(size=(1, sc.height, sc.width, 3)).astype(np.float32)
    r = run_both(sc, tg, seed=13, it=2, views=[0], pairs=pairs, gpu_kwargs={"pairs_per_item": ppi})
    assert r["bins"][1] > 0
    assert_parity(sc, r)


@pytest.mark.parametrize("pairs", [1, 2, 5])
@pytest.mark.parametrize("ppi", [1, 2, 3, 7])
def test_short_explicit_runs_of_light_tiles_match_oracle(ppi, pairs):
    sc = _sphere(40, 40, 30, 61, 45)  # tiles on both sides of the line between small and large light ones
    tg = np.random.default_rng(2).uniform(size=(1, sc.height, sc.width, 3)).astype(np.float32)
    r = run_both(sc, tg, seed=13, it=2, views=[0], pairs=pairs, gpu_kwargs={"pairs_per_item": ppi})
    assert r["bins"][0] > 0
    assert_parity(sc, r)
