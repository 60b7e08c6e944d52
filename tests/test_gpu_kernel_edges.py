"""Sizes at which the kernels' work splits change: edges of tiles, remainders, the ends of a dispatch range."""
import math
import random
import threading

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


def _two_step_levels(g_min, rho, gamma, alpha, L):
    """The two-step quantizer's upper levels below alpha, one row per record, with 64-bit significands: k* is where Q_B turns on either side of
    the best of 2048 grid points, closed in on by halving.  Second result: records whose k* is beyond doubt (one best turn,
    not beside the jump of the density)."""
    def masses(k, a, rho, gamma):
        inside = lambda t: np.where(t <= 1, (1 - 2 * rho) * t, 1 - 2 * rho * np.maximum(t, 1) ** (1 - gamma))
        u = inside(k * a)
        return u, np.maximum(inside(a) - u, 0)

    a, rho, gamma = (alpha / g_min)[:, None], rho[:, None], gamma[:, None]
    k = np.arange(1, 2048)[None, :] / 2048
    u, w = masses(k, a, rho, gamma)
    q = np.cbrt(w * (1 - k) ** 2) + np.cbrt(u * k * k)
    best = q.argmin(1)
    low = np.zeros(q.shape, bool)
    low[:, 1:-1] = (q[:, 1:-1] <= q[:, :-2]) & (q[:, 1:-1] <= q[:, 2:])
    other = np.where(low & (np.abs(np.arange(2047)[None, :] - best[:, None]) > 2), q, np.inf).min(1)
    sure = (a[:, 0] > 1.1) & (best > 1) & (best < 2045) & (other > q.min(1) * (1 + 1e-9))

    a, rho, gamma, g_min = (v.astype(np.longdouble) for v in (a, rho, gamma, g_min[:, None]))

    def rises(k):
        u, w = masses(k, a, rho, gamma)
        du = np.where(k * a <= 1, (1 - 2 * rho) * a, 2 * rho * (gamma - 1) * a ** (1 - gamma) * k ** -gamma)
        return w * w * (1 - k) * (du * k + 2 * u) ** 3 >= u * u * k * (du * (1 - k) + 2 * w) ** 3

    lo, hi = np.maximum(best, 1)[:, None].astype(np.longdouble) / 2048, (best[:, None] + 2).astype(np.longdouble) / 2048
    sure &= (~rises(lo) & rises(hi))[:, 0]
    for _ in range(64):
        mid = (lo + hi) / 2
        up = rises(mid)
        lo, hi = np.where(up, lo, mid), np.where(up, mid, hi)
    k, s = (lo + hi) / 2, L - 1
    u, w = masses(k, a, rho, gamma)
    beta = k * a
    c_in, c_out = np.cbrt(u / beta), np.cbrt(w / (a - beta))
    denom = 2 * a * (c_out * (1 - k) + c_in * k)
    c, lam_in, lam_out = np.arange(L // 2, s)[None, :] - np.longdouble(s) / 2, s * c_in / denom, s * c_out / denom
    return g_min * np.where(c <= lam_in * beta, c / lam_in, beta + (c - lam_in * beta) / lam_out), sure


@pytest.mark.parametrize("alpha", [None, 2.5e-3, 2e-2])
@pytest.mark.parametrize("L", [4, 8, 16])
def test_two_step_levels_are_rounded_once(tq, alpha, L):
    """Only the warp's form cuts the split's bracket 33-fold at a time.  Its levels are those of the exact split, rounded once to fp32, for
    exponents up to 10 and splits close to either end, alpha solved for or given.  In double precision the slope's own rounding moves a level by
    up to 2^-33 of itself, so those that stand closer than 2^-32 to the middle between two fp32 numbers may go either way."""
    n, d, r = 4096, 1_000_003, np.random.default_rng(L)
    tail, g_min, gamma = (d * 2 * r.uniform(0.005, 0.24, n)).astype(np.int64), np.exp(r.uniform(-9, -6.5, n)).astype(np.float32), r.uniform(2.05, 10, n)
    stats = [tq.Stats(d=d, n_tail=int(t), g_min=float(m), sum_log_tail=float(t / (g - 1)), max_abs=float(m) * 1e4) for t, m, g in zip(tail, g_min, gamma)]
    gamma = 1 + tail / np.array([s.sum_log_tail for s in stats])          # as the library reads it back from the record
    raw = torch.from_numpy(np.frombuffer(b"".join(bytes(s) for s in stats), dtype=np.uint8).copy()).cuda()
    rule = {} if alpha is None else dict(alpha_rule=tq.ALPHA_USER, alpha_user=alpha)
    got = tq.params_to_host(tq.tq_params_device(raw, n, L, tq.BISCALED, **rule))
    ok = np.array([p.flags & tq.FLAG_INVALID == 0 and p.alpha > 0 for p in got])
    top = np.array([p.alpha if v else 1.0 for p, v in zip(got, ok)], np.float32)
    want, sure = _two_step_levels(g_min.astype(np.float64), tail / (2.0 * d), gamma, top.astype(np.float64), L)
    sure &= ok
    assert sure.sum() > n // 8
    levels = np.array([list(p.levels)[L // 2:L - 1] for p in got], np.float32)
    lo, hi = (want * (1 - np.longdouble(2) ** -32)).astype(np.float32), (want * (1 + np.longdouble(2) ** -32)).astype(np.float32)
    wrong = sure[:, None] & (levels != lo) & (levels != hi)
    assert not wrong.any(), (int(wrong.sum()), int(sure.sum()), [(gamma[i], float(top[i])) for i in np.flatnonzero(wrong.any(1))[:4]])


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.lib()
    return oracle


def _oracle_params(orc, p):
    q = orc.Params()
    for f in ("bits", "num_levels", "mode", "flags", "alpha", "inv_step", "gamma", "g_min", "rho", "iterations"):
        setattr(q, f, getattr(p, f))
    for k in range(16):
        q.levels[k], q.inv_width[k] = p.levels[k], p.inv_width[k]
    return q


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("L,mode", [(2, 0), (8, 0), (4, 1), (8, 1), (16, 1)])
@pytest.mark.parametrize("lengths", [(8192, 8191, 1, 8193, 31, 32, 33), (1, 2, 3), (500_000, 17, 1_300_000, 4097)])
def test_ranges_that_cross_jobs(tq, orc, dtype, L, mode, lengths):
    """A block's range of tiles may end anywhere in a job and hold many short ones: every job's statistics (exact counts and
    maxima; sums of 16-element fp32 partials, 2e-6), packed words and updates (bit-exact) against the oracle."""
    n, bits, table, at = 3, {2: 1, 4: 2, 8: 3, 16: 4}[L], [], 0
    for ln in lengths:
        table.append((at, ln))
        at += (ln + 15) // 16 * 16
    gen = torch.Generator(device="cuda").manual_seed(at)
    g = (torch.randn((n, at), device="cuda", generator=gen) * torch.rand((n, at), device="cuda", generator=gen).pow(-0.4)).to(dtype)
    S = len(table)
    stats_dev = tq.tq_stats_segments(g, table)
    host = g.float().cpu().numpy()
    for i, r in enumerate(tq.stats_to_host(stats_dev)):
        off, ln = table[i % S]
        o = orc.stats(host[i // S, off:off + ln], g_min=r.g_min) if r.g_min > 0 else None
        assert r.d == ln and (o is None or (r.n_tail, r.max_abs) == (o.n_tail, o.max_abs))
        assert o is None or math.isclose(r.sum_abs, o.sum_abs, rel_tol=2e-6)
    params_dev = tq.tq_params_device(stats_dev, n * S, L, mode, 3.0)
    ps = tq.params_to_host(params_dev)
    packed = tq.tq_compress_segments(g, table, params_dev, L, mode, seed=99)
    out = torch.zeros(at, device="cuda")
    tq.tq_decompress_aggregate_segments(packed, table, params_dev, L, out=out)
    got, res, w = packed.cpu().numpy().view(np.uint32), out.cpu().numpy(), 0
    for s, (off, ln) in enumerate(table):
        words = tq.tq_packed_words(ln, bits)
        rows = np.ascontiguousarray(got[:, w:w + words])
        for i in range(n):
            p = ps[i * S + s]
            want = np.zeros(words, np.uint32) if p.flags & tq.FLAG_INVALID else orc.compress(host[i, off:off + ln], _oracle_params(orc, p), 99, i)
            assert np.array_equal(rows[i], want), (s, i)
        assert np.array_equal(res[off:off + ln], orc.decompress_aggregate(rows, ln, [_oracle_params(orc, ps[i * S + s]) for i in range(n)]))
        w += words


@pytest.mark.parametrize("bits,n", [(1, 3), (2, 17), (3, 64), (4, 5)])
@pytest.mark.parametrize("d", [1, 1023, 1025, 4097, 295 * 4096 - 5, 295 * 4096 + 5, 300 * 4096 + 1])
def test_aggregation_forms(tq, orc, bits, n, d):
    """One unit per thread up to 295 tiles of 4096 outputs, bulk copies beyond; rows one by one, weights, and the fused update
    (its own split up to 4096 tiles).  Sums are taken in worker order with one rounding per operation: equal to the oracle."""
    L = 1 << bits
    r = random.Random(d)
    ps = [tq.tq_params_from_levels(sorted([-1.0 - i] + [r.uniform(-0.9, 0.9) for _ in range(L - 2)] + [1.0 + i])) for i in range(n)]
    ops = [_oracle_params(orc, p) for p in ps]
    words = tq.tq_packed_words(d, bits)
    gen = torch.Generator(device="cuda").manual_seed(d)
    packed = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, words), dtype=torch.int32, device="cuda", generator=gen)
    host = packed.cpu().numpy().view(np.uint32)
    want = orc.decompress_aggregate(host, d, ops)
    assert np.array_equal(tq.tq_decompress_aggregate(packed, d, ps).cpu().numpy(), want)
    weights = [0.01 * (i + 1) for i in range(n)]
    rows = [packed[i].clone() for i in range(n)]
    got = tq.tq_decompress_aggregate_rows(rows, d, ps, weights=weights)
    assert np.array_equal(got.cpu().numpy(), orc.decompress_aggregate(host, d, ops, np.array(weights, np.float32)))
    theta, mom = torch.randn(d, device="cuda", generator=gen), torch.randn(d, device="cuda", generator=gen)
    t0, m0, f = theta.cpu().numpy(), mom.cpu().numpy(), np.float32
    tq.tq_decompress_aggregate_apply(packed, d, ps, theta, mom, lr=0.1, momentum=0.9, weight_decay=1e-3)
    g = want + f(1e-3) * t0
    m1 = f(0.9) * m0 + g
    assert np.array_equal(mom.cpu().numpy(), m1) and np.array_equal(theta.cpu().numpy(), t0 - f(0.1) * m1)
    assert tq.tq_wait_expired_count() == 0


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("weighted", [False, True])
def test_first_two_workers_of_two_bit_rows(tq, orc, n, weighted):
    """The bulk kernel looks up the sum of the first two workers' values at once: one worker, exactly two, short and full steps of four.  The
    additions are those of the oracle, so the results are equal; host and device parameters."""
    d, r = 300 * 4096 + 21, random.Random(n)
    ps = [tq.tq_params_from_levels(sorted([-1.0 - i, r.uniform(-0.9, -0.1), r.uniform(0.0, 0.9), 1.0 + i])) for i in range(n)]
    w = [r.uniform(0.1, 0.9) for _ in range(n)] if weighted else None
    packed = torch.randint(-2 ** 31, 2 ** 31, (n, tq.tq_packed_words(d, 2)), dtype=torch.int64, generator=torch.Generator().manual_seed(n)).to(torch.int32).cuda()
    want = orc.decompress_aggregate(packed.cpu().numpy().view(np.uint32), d, [_oracle_params(orc, p) for p in ps], w)
    assert np.array_equal(tq.tq_decompress_aggregate(packed, d, ps, weights=w).cpu().numpy(), want)
    raw = torch.frombuffer(bytearray(b"".join(bytes(p) for p in ps)), dtype=torch.uint8).cuda()
    assert np.array_equal(tq.tq_decompress_aggregate_device_params(packed, d, raw, 4, weights=w).cpu().numpy(), want)


@pytest.mark.parametrize("bits,n,momentum", [(3, 2, 0.9), (4, 1, 0.0), (4, 33, 0.9)])
@pytest.mark.parametrize("d", [4095 * 4096, 4096 * 4096 - 2047, 4096 * 4096 + 2049])
def test_fused_update_of_long_rows(tq, bits, n, momentum, d):
    """From 4096 tiles on two units per thread (one below; four beyond 32 workers).  The aggregate comes from the plain
    kernel and the update is one rounding per operation: equal."""
    s = (1 << bits) - 1
    ps = [tq.tq_params_from_levels([(2 * k - s) * (1.0 + i) / s for k in range(s + 1)]) for i in range(n)]
    gen = torch.Generator(device="cuda").manual_seed(d)
    packed = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, tq.tq_packed_words(d, bits)), dtype=torch.int32, device="cuda", generator=gen)
    g = tq.tq_decompress_aggregate(packed, d, ps)
    theta = torch.randn(d, device="cuda", generator=gen)
    mom = torch.randn(d, device="cuda", generator=gen) if momentum else None
    m1 = momentum * mom + g if momentum else g
    t1 = theta - 0.1 * m1
    tq.tq_decompress_aggregate_apply(packed, d, ps, theta, mom, lr=0.1, momentum=momentum)
    assert torch.equal(theta, t1) and (mom is None or torch.equal(mom, m1))
    assert tq.tq_wait_expired_count() == 0


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("chunks", [0, 1, 4096, 4097, 8192, 8193, 16384, 16385])
@pytest.mark.parametrize("n", [1, 8, 9])
def test_statistics_of_short_rows(tq, orc, dtype, chunks, n):
    """Up to 16384 chunks of 64 bytes and 8 rows one cluster per row does everything; beyond, two launches.  Counts and maxima
    exact, sums of fp32 partials of at most 16 terms (2e-6), logarithms by the hardware (5e-6), with a few odd values in the row."""
    d = chunks * (16 if dtype == torch.float32 else 32) + (5 if chunks % 2 else 0)
    gen = torch.Generator(device="cuda").manual_seed(chunks + n)
    g = torch.zeros((n, (d + 15) // 16 * 16 + 16), dtype=dtype, device="cuda")
    g[:, :d] = (torch.randn((n, d), device="cuda", generator=gen) * torch.rand((n, d), device="cuda", generator=gen).add(1e-3).pow(-0.5)).to(dtype)
    if d > 100:
        g[0, 17], g[n - 1, d - 1] = float("nan"), float("-inf")
    host = g.float().cpu().numpy()
    hint = tq.new_gmin_hint(n)
    records = {"given": tq.tq_stats(g, d, g_min=0.7), "mean": tq.tq_stats(g, d, kappa=1.5), "pow2": tq.tq_stats_hinted(g, hint, d),
               "again": tq.tq_stats_hinted(g, hint, d)}
    assert torch.equal(records["pow2"], records["again"])
    for name, rec in records.items():
        for i, r in enumerate(tq.stats_to_host(rec)):
            x = host[i, :d]
            o = orc.stats_pow2(x) if name in ("pow2", "again") else orc.stats(x, g_min=0.7 if name == "given" else 0.0, kappa=1.5)
            assert (r.d, r.n_nonfinite, r.max_abs) == (d, o.n_nonfinite, o.max_abs)
            assert math.isclose(r.sum_abs, o.sum_abs, rel_tol=2e-6) and math.isclose(r.sum_sq, o.sum_sq, rel_tol=2e-6)
            assert math.isclose(r.g_min, o.g_min, rel_tol=2e-6)
            ref = orc.stats(x, g_min=r.g_min) if r.g_min > 0 else o
            assert r.n_tail == ref.n_tail and math.isclose(r.sum_log_tail, ref.sum_log_tail, rel_tol=5e-6, abs_tol=1e-9)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("L,alpha,inner", [(16, 1.0, 2.0 ** -20), (16, 3e-3, 3e-3 * 2.0 ** -63), (8, 5e30, 1e25), (8, 1e-30, 1e-37), (16, 0.37, 0.37 * 1.07 ** -6)])
def test_codebooks_of_the_logarithmic_grid(tq, orc, dtype, L, alpha, inner):
    """Levels in geometric steps from `inner` to alpha, of both signs and on one side only: too close together for 2048 equal cells
    (but for the last, whose neighbours are 1.07 apart), up to 64 binades deep, large and small.  Values at every level and one
    ulp beside it, at the edges of cells, NaN, infinities, zeros.  Codes equal the oracle's, parameters on the host and on the device."""
    f = np.float32
    mags = np.geomspace(inner, alpha, L // 2).astype(f)
    books = [np.concatenate([-mags[::-1], mags]), np.concatenate([[-f(alpha)], np.geomspace(inner, alpha, L - 1).astype(f)])]
    d = 20_003
    for lv in books:
        lv[-1] = -lv[0]
        p = tq.tq_params_from_levels([float(x) for x in lv])
        r = np.random.default_rng(L)
        at = np.concatenate([lv, np.nextafter(lv, f(np.inf)), np.nextafter(lv, f(-np.inf)), mags.view(np.uint32).__and__(0xFFF80000).view(f),
                             np.array([0.0, -0.0, np.nan, -np.nan, np.inf, -np.inf, 1e-45, -1e-45, 3e38, -3e38], f)]).astype(f)
        x = (np.exp2(r.uniform(np.log2(float(inner)) - 3, np.log2(alpha) + 2, d)) * r.choice([-1.0, 1.0], d)).astype(f)
        x[: 8 * at.size] = np.tile(at, 8)
        g = torch.zeros(2, (d + 31) // 32 * 32, dtype=dtype, device="cuda")
        g[:, :d] = torch.from_numpy(x).to(dtype).cuda()
        host = g[:, :d].float().cpu().numpy()
        got = tq.tq_compress(g, [p, p], seed=11, first_worker=3, d=d).cpu().numpy().view(np.uint32)
        raw = torch.frombuffer(bytearray(bytes(p) * 2), dtype=torch.uint8).cuda()
        dev = tq.tq_compress_device_params(g, raw, L, tq.NONUNIFORM, seed=11, first_worker=3, d=d).cpu().numpy().view(np.uint32)
        for i in range(2):
            want = orc.compress(host[i], _oracle_params(orc, p), 11, 3 + i)
            assert np.array_equal(got[i], want) and np.array_equal(dev[i], want)


@pytest.mark.parametrize("bits,d,n", [(4, 8_200_003, 1), (4, 9_500_001, 1), (3, 2_000_003, 8), (2, 300_001, 40), (4, 200_000, 64), (1, 17_000_033, 1), (4, 20_000_016, 2)])
def test_decision_table_dispatch(tq, orc, bits, d, n):
    """bf16 rows on both sides of the line from which the decision table serves a call (earlier with host parameters than with
    device ones), few and many rows per SM, ragged ends.  The same codes whichever kernel ran: the oracle's on the last row."""
    L = 1 << bits
    mags = np.geomspace(1e-5, 3e-3, L // 2).astype(np.float32) if L > 2 else np.array([3e-3], np.float32)
    p = tq.tq_params_from_levels([float(x) for x in np.concatenate([-mags[::-1], mags])])
    gen = torch.Generator(device="cuda").manual_seed(d)
    g = torch.zeros(n, (d + 31) // 32 * 32, dtype=torch.bfloat16, device="cuda")
    for i in range(n):
        g[i, :d] = (torch.randn(d, device="cuda", generator=gen) * torch.exp(torch.randn(d, device="cuda", generator=gen)) * 2e-4).to(torch.bfloat16)
    g[:, 5], g[:, d - 1] = float("nan"), float("-inf")
    got = tq.tq_compress(g, [p] * n, seed=3, d=d)
    raw = torch.frombuffer(bytearray(bytes(p) * n), dtype=torch.uint8).cuda()
    assert torch.equal(got, tq.tq_compress_device_params(g, raw, L, tq.NONUNIFORM, seed=3, d=d))
    assert np.array_equal(got[n - 1].cpu().numpy().view(np.uint32), orc.compress(g[n - 1, :d].float().cpu().numpy(), _oracle_params(orc, p), 3, n - 1))


@pytest.mark.parametrize("bits", [1, 2, 3, 4])
@pytest.mark.parametrize("top", [0x0200, 0x3A80, 0x3A81, 0x3A82, 0x3A83, 0x61FF, 0x6200, 0x6203, 0x7EFF])
def test_decision_table_of_every_pattern(tq, orc, bits, top):
    """The table is indexed by the bf16 pattern up to the smallest one >= alpha and filled in four entries at a time below the
    evaluated ones: alpha at each place of a group of four, at the smallest normal numbers, at the largest pattern that has an entry, at the
    next, from which on values enter with a factor, and near the largest of all.  Rows hold every pattern there is but signalling NaN (which C's fmaxf, unlike the GPU's, does not drop)."""
    d, n, L = 1_100_003, 16, 1 << bits
    alpha = float(np.array([top << 16], np.uint32).view(np.float32)[0])
    p = tq.tq_params_from_levels([float(np.float32(alpha) * np.float32((2 * k - (L - 1)) / (L - 1))) for k in range(L)])
    every = torch.arange(65536, dtype=torch.int32)
    every = torch.where((every & 0x7FFF) > 0x7F80, every | 0x40, every).to(torch.int16)
    near = torch.randint(max(top - 1500, 0), top + 40, (d,), generator=torch.Generator().manual_seed(top), dtype=torch.int32)
    row = torch.cat([every, (near + (torch.arange(d) % 2).int() * 0x8000).to(torch.int16)])[:d].cuda()
    g = torch.zeros(n, (d + 15) // 16 * 16, dtype=torch.int16, device="cuda")
    for i in range(n):
        g[i, :d] = torch.roll(row, 1237 * i)
    g = g.view(torch.bfloat16)
    got = tq.tq_compress(g, [p] * n, seed=8, d=d)
    raw = torch.frombuffer(bytearray(bytes(p) * n), dtype=torch.uint8).cuda()
    assert torch.equal(got, tq.tq_compress_device_params(g, raw, L, tq.NONUNIFORM, seed=8, d=d))
    for i in (0, n - 1):
        assert np.array_equal(got[i].cpu().numpy().view(np.uint32), orc.compress(g[i, :d].float().cpu().numpy(), _oracle_params(orc, p), 8, i))


def _kernels(call, path):
    """The kernels that a call launches: the nodes of a graph captured from it, as text."""
    call()                                                       # the first launch of some kernels sets a function attribute
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph):
        call()
    graph.debug_dump(str(path))
    return path.read_text()


def _one_book(tq, L, alpha):
    mags = np.geomspace(alpha * 1e-3, alpha, L // 2).astype(np.float32) if L > 2 else np.array([alpha], np.float32)
    return tq.tq_params_from_levels([float(x) for x in np.concatenate([-mags[::-1], mags])])


@pytest.mark.parametrize("L,d,n,table", [(8, 8_200_000, 1, True), (8, 9_000_000, 1, False), (2, 562_500, 16, False), (8, 10_500_000, 1, True), (8, 656_250, 16, True), (16, 9_000_000, 1, True), (4, 562_500, 16, True)])
def test_decision_table_from_where_it_pays_on_an_idle_gpu(tq, tmp_path, L, d, n, table):
    """With host parameters nothing may be running that hides the table: codes of 1 and 3 bits, whose threads then take a third long piece, use it
    from a little later on."""
    g = torch.zeros(n, (d + 31) // 32 * 32, dtype=torch.bfloat16, device="cuda")
    ps, out = [_one_book(tq, L, 3e-3)] * n, torch.empty(n, tq.tq_packed_words(d, {2: 1, 4: 2, 8: 3, 16: 4}[L]), dtype=torch.int32, device="cuda")
    names = _kernels(lambda: tq.tq_compress(g, ps, seed=5, d=d, packed=out), tmp_path / "graph.dot")
    assert ("compress_lut_kernel" in names) == table and ("compress_kernel" in names) == (not table), names


@pytest.mark.parametrize("alphas", [(3e-3, 3e-3), (3e-3, 1e20), (3e-3, 1e25), (1e25, 1e37)])
def test_decision_table_serves_every_alpha(tq, tmp_path, alphas):
    """Rows with an alpha beyond the table's patterns (2^69) neither leave the table themselves nor take the call's other rows with them."""
    d = 6_000_001
    g = torch.zeros(2, (d + 31) // 32 * 32, dtype=torch.bfloat16, device="cuda")
    ps, out = [_one_book(tq, 16, a) for a in alphas], torch.empty(2, tq.tq_packed_words(d, 4), dtype=torch.int32, device="cuda")
    names = _kernels(lambda: tq.tq_compress(g, ps, seed=5, d=d, packed=out), tmp_path / "graph.dot")
    assert "compress_lut_kernel" in names and "compress_kernel" not in names, names


@pytest.mark.parametrize("bits", [1, 2, 3, 4])
@pytest.mark.parametrize("alpha", [3e-3, 1e30])
def test_decision_table_and_signalling_nan(tq, bits, alpha):
    """The oracle treats signalling NaN otherwise (see above): the table's codes for every pattern are those of the element-wise kernel, which
    serves a call of the first 65536 elements alone."""
    d, n = 17_000_016, 1
    p = _one_book(tq, 1 << bits, alpha)
    g = torch.arange(d, device="cuda").to(torch.int16).view(torch.bfloat16).view(1, d)
    few = tq.tq_compress(g[:, :65536], [p], seed=8, d=65536)
    words = few.shape[1] // 4 * 4
    assert torch.equal(tq.tq_compress(g, [p], seed=8, d=d)[:, :words], few[:, :words])
    raw = torch.frombuffer(bytearray(bytes(p)), dtype=torch.uint8).cuda()
    assert torch.equal(tq.tq_compress_device_params(g, raw, 1 << bits, tq.NONUNIFORM, seed=8, d=d)[:, :words], few[:, :words])


@pytest.mark.parametrize("bits,bad", [(4, False), (3, True), (1, False)])
def test_decision_table_of_layer_groups(tq, orc, bits, bad):
    """bf16 layer groups large enough for a table per piece: lengths from one element up, ranges that cross several jobs, one job whose
    codebook the table does not serve and one that is invalid (zeros).  Equal to the element-wise kernels, which serve the
    groups one call each would be too short for, and to the oracle on a few jobs."""
    L, n = 1 << bits, 3
    lens = [16_000_000, 1, 5_000_001, 33, 9_000_016, 12_289, 3_000_007]
    segs, off = [], 0
    for ln in lens:
        segs.append((off, ln))
        off += (ln + 15) // 16 * 16
    gen = torch.Generator(device="cuda").manual_seed(bits)
    g = (torch.randn(n, off, device="cuda", generator=gen) * torch.exp(torch.randn(n, off, device="cuda", generator=gen)) * 2e-4).to(torch.bfloat16)
    g[:, 7], g[:, off - 17] = float("nan"), float("inf")
    ps = []
    for j in range(n * len(lens)):
        mags = np.geomspace((1e-5 if not (bad and j == 2) else 1e-30) * (1 + j), 3e-3 * (1 + 0.1 * j), L // 2).astype(np.float32) if L > 2 else np.array([3e-3], np.float32)
        ps.append(tq.tq_params_from_levels([float(x) for x in np.concatenate([-mags[::-1], mags])]))
    recs = [bytes(p) for p in ps]
    if bad:
        recs[len(lens) + 4] = bytes(len(recs[0]))                # alpha = 0: never served, all codes 0
    raw = torch.frombuffer(bytearray(b"".join(recs)), dtype=torch.uint8).cuda()
    got = tq.tq_compress_segments(g, segs, raw, L, tq.NONUNIFORM, seed=21).cpu().numpy().view(np.uint32)
    w = 0
    for s, (o, ln) in enumerate(segs):
        words = tq.tq_packed_words(ln, bits)
        for i in range(n):
            j = i * len(lens) + s
            part = got[i, w:w + words]
            if bad and j == len(lens) + 4:
                assert not part.any()
            elif s != 0 or i == 2:
                assert np.array_equal(part, orc.compress(g[i, o:o + ln].float().cpu().numpy(), _oracle_params(orc, ps[j]), 21, i)), (s, i)
        w += words


def test_two_pass_threshold_is_one_number(tq):
    """The tail pass derives g_min = mean|g| in every block from the 512 block sums of the row.  Here the mean lies on the tie between
    two fp32 numbers, and the order in which the warps' sums are added decides to which side it falls; 1 + 2^-23 stands in every
    block, above the one threshold and not above the other.  Each block's sum is exact in fp64, so the sum over the blocks is the
    tree's, bit for bit, and the tail holds all of those elements or none."""
    T, P = 512, 1.0 + 2.0 ** -23

    def fold(rec, tree):                                       # as one block of 256 threads adds the records
        v = (rec[:256] + rec[256:]).reshape(8, 32)
        for o in (16, 8, 4, 2, 1):
            v = v[:, :o] + v[:, o:2 * o]
        w = v[:, 0]
        if tree:
            for o in (4, 2, 1):
                w = w[:o] + w[o:2 * o]
            return float(w[0])
        s = 0.0
        for x in w:
            s += float(x)
        return s

    r = np.random.default_rng(1)
    large = np.full(T, 47.0 + 2.0 ** -12)
    large[:16] -= 2.0 ** -18                                   # the blocks' sums without `small` add up to the tie, T * 4096 * (1 + 2^-24)
    while True:
        small = np.where(r.random(T) < 0.03, r.integers(1, 17, T), 0) * 2.0 ** -38
        rec = 253 * 16 + P + large + small
        tree, turn = fold(rec, True), fold(rec, False)
        if np.float32(tree / (T * 4096)) != np.float32(turn / (T * 4096)):
            break
    x = np.ones((T, 256, 16), np.float32)                      # a block's tile: 256 chunks of 16
    x[:, :3] = 0.0
    x[:, 0, 0], x[:, 1, 0], x[:, 2, 0] = P, small, large
    g = torch.from_numpy(x.reshape(-1)).cuda()
    for st in (tq.stats_to_host(tq.tq_stats(g))[0], tq.stats_to_host(tq.tq_stats_segments(g, [(0, g.numel())]))[0]):
        assert st.sum_abs == tree and st.g_min == float(np.float32(tree / (T * 4096)))
        assert st.n_tail == T + (T if st.g_min == 1.0 else 0)


def test_decision_tables_of_two_threads(tq):
    """Two threads compress bf16 rows whose quantizers need tables of different sizes (they reach up to alpha's pattern: 1e-30 and 1e20), each
    on its own stream: every call is accepted and gives what it gives alone."""
    d = 17_000_000
    x = torch.randn(1, d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    rows, books = [(x * a / 3).to(torch.bfloat16) for a in (1e-30, 1e20)], [[_one_book(tq, 16, a)] for a in (1e-30, 1e20)]
    want = [tq.tq_compress(g, p, seed=5, d=d) for g, p in zip(rows, books)]
    torch.cuda.synchronize()
    failed = []

    def work(k):
        try:
            stream, out = torch.cuda.Stream(), torch.empty_like(want[k])
            with torch.cuda.stream(stream):
                for _ in range(2000):
                    tq.tq_compress(rows[k], books[k], seed=5, d=d, packed=out)
                stream.synchronize()
                assert torch.equal(out, want[k])
        except BaseException as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not failed, failed
