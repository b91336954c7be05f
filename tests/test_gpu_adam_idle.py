"""Adam's step on parameters whose step lies around theta's rounding and far below it (the bound under which the
divisions are left out), and for an adam_eps that is negative or zero, element by element against the oracle's
float64 step.

Tolerance: theta' = theta - step is rounded once (u |theta'|); the step is formed from four float32 products and
sums, two quotients by the bias corrections (formed by expm1f and logf, 2 ulp each) and a root: 32 u relative at
most where adam_eps is positive, and by cond = (|sqrt(v hat)| + |adam_eps|) / |sqrt(v hat) + adam_eps| more where
its sign lets the denominator cancel.  Every moment and product is a normal number."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests.parity import U32, gpu_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("adam_eps", [1e-8, 1e-3, 1e30, 0.0, -1e-8, -1e-3])
def test_small_steps_match_oracle(adam_eps, off):
    import torch
    sc = dataclasses.replace(synth.sphere_scene("s", 24, 20, 33, 32, synth.random_eyes(1, seed=2)))
    g = gpu_scene(sc, None)
    d = g.n_params
    rng = np.random.default_rng(5)
    sizes = [sc.n_pos_params] + [t.data.size for t in sc.textures]
    lrs = [1e-3, 2e-3]
    per = lambda xs: np.concatenate([np.full(n, x, np.float32) for n, x in zip(sizes, xs)])
    eps, lr = per([sc.eps_pos] + [t.eps for t in sc.textures]), per(lrs)
    t, b1, b2 = 7, float(np.float32(0.9)), float(np.float32(0.999))
    theta0 = (rng.choice([-1.0, 1.0], size=d) * 10.0 ** rng.uniform(-12, 3, size=d)).astype(np.float32)
    # sqrt(v hat) is far below adam_eps for most, so a step is about lr m hat / adam_eps: from 2^-44 to 2 of theta
    scale = max(abs(adam_eps), 1e-10)
    m0 = theta0.astype(np.float64) * 2.0 ** rng.uniform(-44, 1, size=d) * scale / lr.astype(np.float64) * (1 - b1 ** t)
    m0 = np.clip(m0 * rng.choice([-1.0, 1.0], size=d), -1e30, 1e30).astype(np.float32)
    v0 = np.clip((scale * 10.0 ** rng.uniform(-6, -1, size=d)) ** 2, 0, 1e30).astype(np.float32)
    o = 0
    for p, n in zip(g.param_groups(), sizes):
        p.copy_(torch.tensor(theta0[o:o + n]).view(p.shape))
        o += n

    def put(x):
        a = torch.zeros(d + 4, dtype=torch.float32, device=g.device)[off:off + d]
        a.copy_(torch.tensor(x))
        return a

    grad, m, v = put(np.zeros(d, np.float32)), put(m0), put(v0)
    counts = torch.zeros(d, dtype=torch.int32, device=g.device)
    g.step(1, grad, counts, 8, lrs[0], lrs[1:], m=m, v=v, t=t, adam_eps=adam_eps)
    torch.cuda.synchronize()
    eps32 = float(np.float32(adam_eps))
    th, mo, vo = oracle.step(1, theta0, np.zeros(d), np.zeros(d, np.uint64), eps, lr, 8, t=t, m=m0, v=v0, b1=b1, b2=b2,
                             adam_eps=eps32)
    got = np.concatenate([p.detach().cpu().numpy().ravel() for p in g.param_groups()]).astype(np.float64)
    step = np.abs(theta0.astype(np.float64) - th)
    root = np.sqrt(vo / (1 - b2 ** t))
    den = np.abs(root + eps32)
    cond = (root + abs(eps32)) / np.maximum(den, 1e-300)
    ok = (den > 0) & (cond < 1e3) & np.isfinite(th) & (np.abs(th) < 1e38)
    assert ok.mean() > 0.9
    assert (lr * np.abs(mo))[m0 != 0].min() > 2.0 ** -126 and vo.min() > 2.0 ** -126
    tol = U32 * np.abs(th) + 32 * U32 * cond * step
    bad = ok & (np.abs(got - th) > tol)
    assert not bad.any(), (int(bad.sum()), theta0[bad][:4], th[bad][:4], got[bad][:4])
    # the states on both sides of the bound were there
    rel = step[ok] / np.abs(theta0[ok])
    assert (rel > 2.0 ** -24).any() and (rel < 2.0 ** -34).any()
