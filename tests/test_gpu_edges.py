"""The pruning, the dense tiles, the renders, the binning, the transparent estimator and the step at the sizes where
their branches change, against the oracle: bins of one and of several chunks, grids of each pruning variant, dense
tiles of few and of many pairs (every model, grouped or not, both footprints), more than 1,024 tiles, textures one
texel wide or high, groups and buffers off the 16-byte grid.  Tolerances of estimates and renders: tests/parity.py."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests.parity import BG, U32, assert_parity, color_k, gpu_scene, run_both, torch_keys_to_u64
from tests.test_gpu_fast_groups import _lit, _quads, _sphere

pytestmark = pytest.mark.gpu


def _targets(sc):
    return np.random.default_rng(2).uniform(size=(sc.n_views, sc.height, sc.width, 3)).astype(np.float32)


def _lambert_dense(sizes, n):
    sc = _lit(synth.config_scale, [sizes[0]] * 4, n_lon=n, n_lat=n)
    keep = [k for k, t in enumerate(sc.textures) if t.role in (synth.ROLE_ALBEDO, synth.ROLE_NORMAL)]
    tex = [synth.Texture(np.ascontiguousarray(np.resize(sc.textures[k].data, (s[1], s[0], sc.textures[k].data.shape[2]))),
                         sc.textures[k].eps, sc.textures[k].role) for k, s in zip(keep, sizes)]
    return dataclasses.replace(sc, shading=synth.SHADE_LAMBERT, textures=tex, target_textures=None, target_positions=None,
                               width=40, height=36)


def _grown_soup(n, scale, render):
    """Triangles of all sizes up to several tiles, hundreds in every tile."""
    sc, _ = synth.triangle_soup(n, render=render)
    p = sc.positions.reshape(-1, 3, 3).astype(np.float64)
    c = p.mean(1, keepdims=True)
    p[..., :2] = c[..., :2] + np.linspace(0.2, scale, n)[:, None, None] * (p - c)[..., :2]
    return dataclasses.replace(sc, positions=p.reshape(-1, 3).astype(np.float32))


ESTIMATES = {
    # bins of more than 256 triangles of which a light tile's worth stays: marked, then listed
    "prune_chunks": (lambda: _sphere(52, 40, 30, 64, 64), 3),
    # 306 and 4 x 306 tiles: the one-wave and the throughput variants of the pruning
    "prune_grid_306": (lambda: _sphere(24, 40, 30, 288, 272), 2),
    "prune_grid_1224": (lambda: _sphere(24, 40, 30, 288, 272, views=4), 1),
    "prune_big": (lambda: _quads(700, 600), 1),
    # dense tiles: more live triangles than are kept in shared memory, one to nine pairs
    "dense_pairs_1": (lambda: _sphere(96, 40, 30, 32, 30), 1),
    "dense_pairs_9": (lambda: _sphere(96, 40, 30, 32, 30), 9),
    "dense_grown_soup": (lambda: _grown_soup(6000, 3.0, 72), 2),
    "dense_texture_1x1": (lambda: _sphere(72, 1, 1, 32, 30, 1), 3),
    "dense_hash": (lambda: _sphere(72, 900, 700, 32, 30), 3),
    "dense_lambert_group": (lambda: _lambert_dense([(40, 40)] * 2, 72), 3),
    "dense_lambert_two_sizes": (lambda: _lambert_dense([(37, 29), (90, 3)], 72), 3),
    "dense_ggx": (lambda: dataclasses.replace(_lit(synth.config_scale, [(40, 40)] * 4, n_lon=96, n_lat=72), width=40,
                                              height=36, target_positions=None), 3),
}


@pytest.mark.parametrize("nearest", [False, True], ids=["bilinear", "nearest"])
@pytest.mark.parametrize("case", list(ESTIMATES))
def test_estimate_branches_match_oracle(case, nearest):
    from paper_2404_09758_gb300 import FOOT_NEAREST
    make, pairs = ESTIMATES[case]
    sc = make()
    r = run_both(sc, _targets(sc), seed=13, it=2, views=list(range(sc.n_views)), pairs=pairs,
                 footprint=oracle.FOOT_NEAREST if nearest else 0,
                 gpu_kwargs={"footprint": FOOT_NEAREST} if nearest else {})
    assert r["C"].sum() > 0
    if case.startswith("dense"):
        assert r["bins"][1] > 0
    assert_parity(sc, r)


RENDERS = {
    "bins_of_thousands": lambda: _sphere(72, 40, 30, 32, 30),
    "bins_of_thousands_lambert": lambda: _lambert_dense([(37, 29), (90, 3)], 72),
    "bins_of_thousands_ggx": lambda: dataclasses.replace(_lit(synth.config_scale, [(40, 30)] * 4, n_lon=96, n_lat=72),
                                                         width=40, height=36),
    "big_triangles_1672_tiles": lambda: _quads(700, 600),
    # bins of several chunks with boxes on both sides of a lane's limit
    "grown_soup": lambda: _grown_soup(3000, 6.0, 72),
}


@pytest.mark.parametrize("case", list(RENDERS))
def test_renders_and_loss_match_oracle(case):
    import torch
    sc = RENDERS[case]()
    tg = _targets(sc)
    g, osc = gpu_scene(sc, tg), oracle.OracleScene(sc, tg)
    for pair, side in ((0, 0), (2, 1), (2, -1)):
        keys, uv, rgb = g.render_idb(0, seed=5, it=3, pair=pair, side=side)
        torch.cuda.synchronize()
        ok, ouv, orgb = oracle.render(osc, 0, 5, 3, pair, side)
        assert np.array_equal(torch_keys_to_u64(keys), ok)
        cov = ok != BG
        assert np.array_equal(uv.cpu().numpy()[cov].view(np.uint32), ouv[cov].view(np.uint32))
        assert (np.abs(rgb.cpu().numpy().astype(np.float64) - orgb) <= color_k(sc) * U32 * (1.0 + np.abs(orgb))).all()
    # a colour's error d = k u (1 + |I|) moves (I - T)^2 by at most 2 |I - T| d + d^2; the sum adds 256 terms by
    # tree and one float atomic per tile
    d = color_k(sc) * U32 * (1.0 + np.abs(ok_rgb := oracle.render(osc, 0)[2]))
    want = oracle.loss(osc, 0)
    tiles = ((sc.width + 15) // 16) * ((sc.height + 15) // 16)
    tol = (2 * np.abs(ok_rgb - tg[0]) * d + d * d).sum() + (tiles + 16) * U32 * want
    assert abs(float(g.loss([0])[0]) - want) <= tol
    assert g.status() == 0


@pytest.mark.parametrize("nearest", [False, True], ids=["bilinear", "nearest"])
@pytest.mark.parametrize("tw,th", [(1, 64), (64, 1), (2, 2), (3, 2), (200, 150)])
def test_transparent_textures_match_oracle(tw, th, nearest):
    from paper_2404_09758_gb300 import FOOT_NEAREST
    sc = synth.config_transparent(n_views=1, pairs=2, render=56, tex=16, n_lon=16, n_lat=16)
    sc = dataclasses.replace(sc, textures=[synth.Texture(synth.rgba_texture(tw, th, seed=0), 1.0 / 255.0, synth.ROLE_ALBEDO)],
                             target_textures=[synth.rgba_texture(tw, th, seed=1)], width=61, height=53)
    r = run_both(sc, _targets(sc), seed=3, it=1, views=[0], pairs=2, footprint=oracle.FOOT_NEAREST if nearest else 0,
                 gpu_kwargs={"footprint": FOOT_NEAREST} if nearest else {})
    assert r["C"][sc.n_pos_params:].sum() > 0
    assert_parity(sc, r)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_step_off_the_16_byte_grid_matches_oracle(kind, off):
    """Group starts that are no multiples of four, a last quad cut short, buffers `off` floats from a
    16-byte boundary; and parameters nothing touches: sums of 0 and moments down to denormals, whose
    step is below theta's rounding.  Tolerance: theta as in the step's other test; the gradient is two
    products and a quotient, 4 u relative."""
    import torch
    sc = _lambert_dense([(37, 29), (5, 3)], 12)
    g = gpu_scene(sc, _targets(sc))
    rng = np.random.default_rng(kind)
    d = g.n_params
    sizes = [sc.n_pos_params] + [t.data.size for t in sc.textures]
    assert sum(sizes) == d and sizes[0] % 4 and (d % 4)
    S = rng.normal(size=d).astype(np.float32)
    Cn = rng.integers(0, 20, size=d).astype(np.int32)
    idle = rng.uniform(size=d) < 0.5
    S[idle] = 0.0
    m0 = np.where(idle, 10.0 ** rng.uniform(-44, -6, size=d), 0.01 * rng.normal(size=d)).astype(np.float32)
    v0 = np.where(idle, 10.0 ** rng.uniform(-44, -6, size=d), 0.001 * rng.uniform(size=d)).astype(np.float32)
    theta0 = np.concatenate([p.detach().cpu().numpy().ravel() for p in g.param_groups()])
    per = lambda xs: np.concatenate([np.full(n, x, np.float32) for n, x in zip(sizes, xs)])
    eps, lr = per([sc.eps_pos] + [t.eps for t in sc.textures]), per([1e-3, 2e-3, 3e-3])

    def put(x):
        t = torch.zeros(d + 4, dtype=torch.int32 if x.dtype == np.int32 else torch.float32, device=g.device)[off:off + d]
        t.copy_(torch.tensor(x))
        return t

    grad, counts, m, v = put(S), put(Cn), put(m0), put(v0)
    out = g.gradient(grad, 8, out=put(S))
    g.step(kind, grad, counts, 8, 1e-3, [2e-3, 3e-3], m=m, v=v, t=3)
    torch.cuda.synchronize()
    want = S.astype(np.float64) / (2 * eps.astype(np.float64) * 8)
    assert (np.abs(out.cpu().numpy() - want) <= 4 * U32 * np.abs(want)).all()
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    th, mo, vo = oracle.step(kind, theta0, S.astype(np.float64), Cn.astype(np.uint64), eps, lr, 8, t=3, m=m0, v=v0, b1=b1, b2=b2)
    got = np.concatenate([p.detach().cpu().numpy().ravel() for p in g.param_groups()]).astype(np.float64)
    assert np.abs(got - th).max() <= 1e-6 * (1 + np.abs(th).max())
    if kind == 1:
        tiny = np.float64(2.0 ** -148)  # denormal moments round by up to two units
        gr = want
        assert (np.abs(m.cpu().numpy() - mo) <= 8 * U32 * (np.abs(b1 * m0) + np.abs((1 - b1) * gr)) + tiny).all()
        assert (np.abs(v.cpu().numpy() - vo) <= 16 * U32 * (np.abs(b2 * v0) + np.abs((1 - b2) * gr * gr)) + tiny).all()
    assert grad.abs().sum().item() == 0 and counts.abs().sum().item() == 0
