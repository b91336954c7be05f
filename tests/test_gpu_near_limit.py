"""Light tiles with a triangle that may cross the near limit: the limit runs through the box a vertex is perturbed in,
so the triangle is drawn on some sides and not on others, and where it is drawn its depth begins at that vertex.  Over
a farther triangle whose depth lies between its vertices' depths, against the oracle (tolerances: tests/parity.py)."""
import numpy as np
import pytest

import synth
from tests.parity import assert_parity, run_both

pytestmark = pytest.mark.gpu

NEAR, EPS = 0.1, 1e-3


def _scene(front, n_middle):
    """Camera: w = z, depth 1 - near / z.  front: z of the three vertices of the triangle in front, given at its
    screen places; behind it n_middle quads over the whole image at depths 0.5, 0.55, ..."""
    M = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -NEAR], [0, 0, 1, 0]], np.float32)
    ndc = [(0.05, -0.8), (-0.8, 0.7), (0.75, 0.8)]
    pos = [(x * z, y * z, z) for (x, y), z in zip(ndc, front)]
    tri = [(0, 1, 2)]
    for k in range(n_middle):
        z = NEAR / (0.5 - 0.05 * k)
        b = len(pos)
        pos += [(x * z, y * z, z) for x, y in ((-1.2, -1.2), (1.2, -1.2), (1.2, 1.2), (-1.2, 1.2))]
        tri += [(b, b + 1, b + 2), (b, b + 2, b + 3)]
    pos, tri = np.array(pos, np.float32), np.array(tri, np.int32)
    uv = np.random.default_rng(3).uniform(0.1, 0.9, size=(len(pos), 2)).astype(np.float32)
    tex = [synth.Texture(synth.sinusoid_texture(40, 30, 3, seed=5), 1.0 / 255.0, synth.ROLE_ALBEDO)]
    return synth.Scene("near", pos, tri, uv, tri.copy(), tex, EPS, M[None], np.zeros((1, 3), np.float32), 61, 50,
                       near=NEAR)


@pytest.mark.parametrize("n_middle", [1, 4])
@pytest.mark.parametrize("front", [
    (NEAR + 0.4 * EPS, 1.0, 1.2),        # one vertex whose box the limit runs through: above it,
    (NEAR - 0.4 * EPS, 1.0, 1.2),        # below it
    (NEAR + 0.4 * EPS, NEAR - 0.3 * EPS, 1.0),
    (NEAR + 0.5 * EPS, NEAR + 0.2 * EPS, NEAR + 0.4 * EPS),  # all three
], ids=["one_above", "one_below", "two", "three"])
def test_triangle_across_the_near_limit_matches_oracle(front, n_middle):
    sc = _scene(front, n_middle)
    tg = np.random.default_rng(2).uniform(size=(1, sc.height, sc.width, 3)).astype(np.float32)
    r = run_both(sc, tg, seed=13, it=2, views=[0], pairs=16)
    assert r["bins"][1] == 0  # every tile is a light one
    assert r["C"][:9].sum() > 0  # the triangle is drawn on some side
    assert_parity(sc, r)
