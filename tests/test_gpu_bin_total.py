"""A call whose bin entries pass 2^32 while their low 32 bits would fit the capacity: reported, nothing rendered or
credited from bins that were not stored, and the next call on the scene is sound."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_entries_past_32_bits_are_an_overflow():
    import torch
    from paper_2404_09758_gb300 import ERR_BIN_OVERFLOW, OK, Scene
    free, _ = torch.cuda.mem_get_info()
    if free < 16 << 30:
        pytest.skip("needs 16 GB")
    # every triangle may cross the near limit, so it is binned into all 16,384 tiles of each of 16 views
    n, views, near, eps = 16_400, 16, 0.1, 1e-3
    tiles = (2048 // 16) ** 2
    total = n * tiles * views
    capacity = 6_000_000
    assert total >= 2 ** 32 and total % 2 ** 32 <= capacity
    rng = np.random.default_rng(0)
    pos = np.concatenate([rng.uniform(-0.1, 0.1, size=(3 * n, 2)), np.full((3 * n, 1), near)], axis=1).astype(np.float32)
    idx = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    M = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -near], [0, 0, 1, 0]], np.float32)
    tex = [(np.full((4, 4, 3), 0.5, np.float32), 1.0 / 255.0, synth.ROLE_ALBEDO)]
    g = Scene(pos, idx, np.full((3 * n, 2), 0.5, np.float32), idx, tex, eps, np.repeat(M[None], views, 0),
              np.zeros((views, 3), np.float32), 2048, 2048, near=near, bin_capacity=capacity, max_pairs_per_call=1)
    grad, counts = g.new_grad_buffers()
    g.estimate_grad(1, 0, list(range(views)), 1, grad, counts)
    light, heavy, entries = g.bin_stats()
    assert g.status() == ERR_BIN_OVERFLOW
    assert entries == total and light == 0 and heavy == 0
    assert not counts.any() and not grad.any()
    # moved away from the limit, every triangle within 22 pixels of the image's centre (16 tiles), it fits again
    g.positions[:, 2] = 5.0
    g.estimate_grad(1, 0, [0], 1, grad, counts)
    light, heavy, entries = g.bin_stats()
    assert g.status() == OK and light + heavy > 0 and 0 < entries <= capacity
    assert int(counts.sum()) > 0
