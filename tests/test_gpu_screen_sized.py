"""Triangles far larger than a tile, whose edge functions need 64 bits, of both windings: renders of tiles with few and
with hundreds of them, the plain path, light and dense tiles of the estimator and transparent tiles, against the oracle
(tolerances: tests/parity.py).  On the pixel grid the vertices, perturbed or not, are pixel centres, so that edges run
through the centres of pixels and the top/left rule decides."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests.parity import BG, U32, assert_parity, color_k, gpu_scene, run_both, torch_keys_to_u64

pytestmark = pytest.mark.gpu

R = 64  # a power of two: pixel centres and the perturbation of one pixel are exact


def _scene(n, reach, grid, seed=7, flat=False):
    """n triangles, every other one turned, that reach `reach` pixels beyond the image, each with an edge through it; half
    of them are slivers.  flat: at one of two neighbouring depths."""
    rng = np.random.default_rng(seed)
    c = rng.integers(0, R, size=(n, 2)) + (0.5 if grid else rng.uniform(size=(n, 2)))
    d = rng.integers(-3, 4, size=(n, 2))
    d[(d == 0).all(axis=1)] = (1, 1)
    if not grid:
        d = d + rng.uniform(-0.4, 0.4, size=(n, 2))
    far = rng.integers(reach // 4, reach // 3, size=(2, n, 1))
    p0, p1 = c + far[0] * d, c - far[1] * d
    p2 = np.where(np.arange(n)[:, None] % 4 < 2, p1 + rng.integers(-6, 7, size=(n, 2)),
                  c + np.stack([-d[:, 1], d[:, 0]], axis=1) * far[0])
    px = np.stack([p0, p1, p2], axis=1)
    z = rng.uniform(0.2, 0.8, size=(n, 3, 1))
    if flat:
        z = np.repeat(rng.choice([np.float32(0.7), np.nextafter(np.float32(0.7), np.float32(1))], size=(n, 1, 1)), 3, axis=1)
    pos = np.concatenate([2 * px[..., :1] / R - 1, 1 - 2 * px[..., 1:] / R, z], axis=2)
    pos[::2] = pos[::2, ::-1]
    sc, tg = synth.triangle_soup(n, render=R, seed=seed)
    uvs = rng.uniform(0.05, 0.95, size=sc.uvs.shape).astype(np.float32)
    tex = [synth.Texture(synth.sinusoid_texture(37, 29, 3, seed=5), 1.0 / 255.0, synth.ROLE_ALBEDO)]
    return dataclasses.replace(sc, positions=pos.reshape(-1, 3).astype(np.float32), uvs=uvs, textures=tex), tg


GRID = pytest.mark.parametrize("grid", [False, True], ids=["float", "grid"])
SHAPES = pytest.mark.parametrize("n,reach", [(12, 8000), (100, 100), (100, 2000), (400, 600), (600, 30000), (600, 90)])


@pytest.mark.parametrize("flat", [False, True], ids=["depths", "flat"])
@GRID
@SHAPES
def test_renders_match_oracle(n, reach, grid, flat):
    import torch
    sc, tg = _scene(n, reach, grid, flat=flat)
    g, osc = gpu_scene(sc, tg, bin_capacity=n * 16 + 64), oracle.OracleScene(sc, tg)
    for pair, side in ((0, 0), (2, 1), (2, -1)):
        keys, uv, rgb = g.render_idb(0, seed=5, it=3, pair=pair, side=side)
        torch.cuda.synchronize()
        ok, ouv, orgb = oracle.render(osc, 0, 5, 3, pair, side)
        assert np.array_equal(torch_keys_to_u64(keys), ok)
        cov = ok != BG
        assert np.array_equal(uv.cpu().numpy()[cov].view(np.uint32), ouv[cov].view(np.uint32))
        assert (np.abs(rgb.cpu().numpy().astype(np.float64) - orgb) <= color_k(sc) * U32 * (1.0 + np.abs(orgb))).all()
    assert g.status() == 0


@pytest.mark.parametrize("plain", [False, True], ids=["fused", "plain"])
@GRID
@SHAPES
def test_estimates_match_oracle(n, reach, grid, plain):
    sc, tg = _scene(n, reach, grid)
    r = run_both(sc, tg, seed=13, it=2, views=[0], pairs=3, plain=plain, gpu_kwargs={"bin_capacity": n * 16 + 64})
    assert r["C"][: sc.n_pos_params].sum() > 0
    assert_parity(sc, r)


@GRID
@pytest.mark.parametrize("n,reach", [(6, 8000), (40, 400), (300, 90)])
def test_transparent_estimates_match_oracle(n, reach, grid):
    sc, tg = _scene(n, reach, grid)
    sc = dataclasses.replace(sc, shading=synth.SHADE_TRANSPARENT, background=(0.3, 0.3, 0.3),
                             textures=[synth.Texture(synth.rgba_texture(37, 29, seed=0), 1.0 / 255.0, synth.ROLE_ALBEDO)])
    r = run_both(sc, tg, seed=3, it=1, views=[0], pairs=2, gpu_kwargs={"bin_capacity": n * 16 + 64})
    assert r["C"][: sc.n_pos_params].sum() > 0
    assert_parity(sc, r)


@pytest.mark.parametrize("n,pairs", [(6, 1), (40, 9), (400, 3)])
def test_flat_colours_match_oracle(n, pairs):
    """A triangle's colour is one texel of a one-row texture, whose footprints at the texel's centre differ by rounding
    between the sides: the texels left over on side - go through the hash."""
    sc, tg = _scene(n, 200, False)
    soup = synth.triangle_soup(n, render=R, seed=3)[0]
    sc = dataclasses.replace(sc, uvs=soup.uvs, textures=soup.textures)
    r = run_both(sc, tg, seed=13, it=2, views=[0], pairs=pairs, gpu_kwargs={"bin_capacity": n * 16 + 64})
    assert r["C"][sc.n_pos_params:].sum() > 0
    assert_parity(sc, r)
