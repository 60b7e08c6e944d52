"""Sizes at which the kernels' work splits change: edges of tiles, remainders, the ends of a dispatch range."""
import math
import random

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2402_01798_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 64, 4096])
def test_params_device_record_counts(tq, mode, n):
    """Four records share a block: counts around a block's edge up to the largest, some records outside the domain.
    Device and host use their own log / exp: fp32 rounding of alpha and the levels (a few ulp, 6e-8 each)."""
    r = random.Random(n * 3 + mode)
    stats = []
    for i in range(n):
        s = tq.Stats()
        s.d, s.g_min = 10 ** r.randint(4, 9), math.exp(r.uniform(-12, -2))
        s.n_tail = 0 if i % 7 == 5 else max(1, int(2 * s.d * r.uniform(0.01, 0.2)))
        s.sum_log_tail, s.max_abs = s.n_tail / r.uniform(1.5, 3.0), s.g_min * math.exp(r.uniform(3, 8))
        stats.append(s)
    raw = torch.from_numpy(np.frombuffer(b"".join(bytes(s) for s in stats), dtype=np.uint8).copy()).cuda()
    got = tq.params_to_host(tq.tq_params_device(raw, n, 16, mode))
    for i in random.Random(1).sample(range(n), min(n, 200)):
        try:
            want = tq.tq_params(stats[i], 16, mode)
        except tq.TqError as e:
            assert got[i].flags == tq.FLAG_INVALID and got[i].iterations == e.status and got[i].alpha == 0.0
            continue
        assert (got[i].flags, got[i].bits, got[i].mode) == (want.flags, want.bits, want.mode)
        assert math.isclose(got[i].alpha, want.alpha, rel_tol=3e-7)
        assert np.allclose(list(got[i].levels), list(want.levels), rtol=5e-7, atol=0)
