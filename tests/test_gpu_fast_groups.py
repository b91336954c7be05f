"""The fast estimator's groups of pairs, texel windows and hashed footprints at the sizes where they
can go wrong, against the oracle: group remainders (1..17 pairs, runs of 1..32), triangles too large
for the 32-bit edge functions, windows that hold a tile's footprints, are cut, or do not exist
(textures one texel wide or high, 2 x 2, minified until the hash table is full), candidate lists of
17..32 and of more, every shading model and both footprints.  Tolerances: tests/parity.py."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests.parity import assert_parity, run_both
from tests.tiny import flat_scene

pytestmark = pytest.mark.gpu


def _sphere(n, tex_w, tex_h, w, h, channels=3, views=1, seed=5):
    sc = synth.sphere_scene("t", n, n, 8, w, synth.random_eyes(views, seed))
    mvp = np.stack([synth.mvp_matrix(e, w, h) for e in synth.random_eyes(views, seed)]).astype(np.float32)
    t = synth.Texture(synth.sinusoid_texture(tex_w, tex_h, channels, seed=4), 1.0 / 255.0, synth.ROLE_ALBEDO)
    return dataclasses.replace(sc, width=w, height=h, mvp=mvp, textures=[t],
                               target_textures=[synth.sinusoid_texture(tex_w, tex_h, channels, seed=9)])


def _quads(w, h):
    """Two screen-filling triangles behind a few small ones: edges of hundreds of pixels."""
    tris = [[(-40, -30, 0.7), (2 * w + 60, -30, 0.8), (-40, 2 * h + 60, 0.6)],
            [(-900, h + 20, 0.5), (w + 500, -700, 0.9), (w + 90, h + 80, 0.6)],
            [(w / 2, h / 2, 0.2), (w / 2 + 9, h / 2 + 1, 0.2), (w / 2 + 2, h / 2 + 8, 0.3)]]
    tex = synth.Texture(synth.sinusoid_texture(50, 40, 3, seed=4), 1.0 / 255.0, synth.ROLE_ALBEDO)
    sc = flat_scene(tris, 512, 512, textures=[tex], eps_pos=2e-3)
    sc.width, sc.height = w, h
    sc.mvp = np.array([[[512 / w, 0, 0, 512 / w - 1], [0, 512 / h, 0, 1 - 512 / h], [0, 0, 1, 0], [0, 0, 0, 1]]], np.float32)
    return sc


def _lit(make, sizes, **kw):
    sc = make(n_views=1, pairs=1, render=72, tex=16, **kw)
    out, goal = [], []
    for (tw, th), t in zip(sizes, sc.textures):
        normal = t.role == synth.ROLE_NORMAL
        f = (lambda s: synth.normal_map_texture(tw, th, seed=s)) if normal else \
            (lambda s: 0.2 + 0.6 * synth.sinusoid_texture(tw, th, t.data.shape[2], seed=s))
        out.append(synth.Texture(f(3).astype(np.float32), t.eps, t.role))
        goal.append(f(7).astype(np.float32))
    return dataclasses.replace(sc, textures=out, target_textures=goal)


CASES = {
    "pairs_1": (lambda: _sphere(24, 40, 30, 61, 45), 1, {}),
    "pairs_9": (lambda: _sphere(24, 40, 30, 61, 45), 9, {}),
    "pairs_17_run_32": (lambda: _sphere(24, 40, 30, 61, 45), 17, {"pairs_per_item": 32}),
    "run_5": (lambda: _sphere(40, 40, 30, 61, 45), 11, {"pairs_per_item": 5}),
    "big_triangles": (lambda: _quads(331, 273), 3, {}),
    "texture_1x64": (lambda: _sphere(24, 1, 64, 48, 48), 3, {}),
    "texture_64x1": (lambda: _sphere(24, 64, 1, 48, 48), 3, {}),
    "texture_2x2": (lambda: _sphere(24, 2, 2, 48, 48), 3, {}),
    "texture_1x1_1ch": (lambda: _sphere(24, 1, 1, 48, 48, 1), 3, {}),
    "texture_3x2_4ch": (lambda: _sphere(24, 3, 2, 48, 48, 4), 3, {}),
    "window_cut": (lambda: _sphere(24, 160, 120, 64, 48, views=2), 3, {}),
    "hash_full": (lambda: _sphere(16, 1500, 1400, 48, 40), 3, {}),
    "many_candidates": (lambda: _sphere(72, 64, 64, 64, 64, views=2), 3, {}),
    "lambert_group_cut": (lambda: _lit(synth.config_autograd, [(150, 130)] * 2), 3, {}),
    "lambert_two_sizes": (lambda: _lit(synth.config_autograd, [(37, 29), (90, 3)]), 3, {}),
    "ggx_group": (lambda: _lit(synth.config_scale, [(40, 40)] * 4, n_lon=48, n_lat=24), 5, {}),
    "ggx_four_sizes": (lambda: _lit(synth.config_scale, [(40, 30), (1, 9), (300, 200), (16, 2)], n_lon=48, n_lat=24), 3, {}),
}


@pytest.mark.parametrize("nearest", [False, True], ids=["bilinear", "nearest"])
@pytest.mark.parametrize("case", list(CASES))
def test_fast_groups_match_oracle(case, nearest):
    from paper_2404_09758_gb300 import FOOT_NEAREST
    make, pairs, kw = CASES[case]
    sc = make()
    tg = oracle.render_targets(sc, synth.target_scene(sc)) if sc.target_positions is not None else \
        np.random.default_rng(2).uniform(size=(sc.n_views, sc.height, sc.width, 3)).astype(np.float32)
    r = run_both(sc, tg, seed=21, it=4, views=list(range(sc.n_views)), pairs=pairs,
                 footprint=oracle.FOOT_NEAREST if nearest else 0,
                 gpu_kwargs=dict(kw, footprint=FOOT_NEAREST) if nearest else kw)
    assert r["C"].sum() > 0
    assert_parity(sc, r)
