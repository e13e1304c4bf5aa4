"""Sketch pass whose lanes keep their cells (states without a projection of vectors of many tiles): every
number of walker warps and of items to a warp, sketch rows in one part and in two, partial worker groups and
tiles, rows that are not aligned; hashes whose lists are too uneven for it; and the calls of such a
context that the other list kernels serve.  Tolerance: the usual one of a state (the sums of a tile's list in
fp32, added to the cell's in fp32 once per tile, as in the other kernels)."""
import numpy as np
import pytest

from fda_testlib import check_states

pytestmark = pytest.mark.gpu

P = (1 << 61) - 1


def schedule_bytes(F, l, m, coeffs, d, K):
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        return ctx.fda_context_info()["schedule_bytes"]


def check(l, m, K, d, coeffs, aligned, seed, even=True):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pitch = (d + 3) // 4 * 4 + (0 if aligned else 1)
    w0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = torch.full((K, pitch), 1e6, device="cuda")[:, :d]
    w.copy_(w0 + torch.randn((K, d), device="cuda", generator=gen) * 1e-3)
    xi = torch.randn(d, device="cuda", generator=gen)
    xi /= xi.norm()
    ks = [0, K // 2, K - 1]
    ora = oracle.local_state(w[ks].cpu().numpy(), w0.cpu().numpy(), xi.cpu().numpy(), coeffs, l, m, threads=8)
    without = ora.copy()
    without[:, 1] = 0.0
    # a second schedule is there exactly when the hash is even (the same vector with few workers has none)
    few = schedule_bytes(F, l, m, coeffs, d, 4)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        assert (ctx.fda_context_info()["schedule_bytes"] > 3 * few // 2) == even
        for flags, want in ((5, without), (7, ora)):
            st = [torch.full((K, ctx.state_len), float("nan"), device="cuda") for _ in range(2)]
            for s in st:
                ctx.fda_local_state(w, w0, xi, flags, s)
            assert ctx.fda_debug_last_kernel() == "k_local_state_gather"
            assert ctx.fda_debug_last_schedule() == (2 if flags == 5 and even else 1)
            assert bool(torch.isfinite(st[0]).all())
            check_states(st[0][ks].cpu().numpy(), want, l, m, d)
            if flags == 5 and even:            # no sum's order is left to chance
                assert torch.equal(st[0], st[1])
        part = torch.full((K, ctx.state_len), float("nan"), device="cuda")      # fewer workers, a shorter vector
        ctx.fda_local_state(w[:7, :70_001], w0[:70_001], None, 5, part)
        assert ctx.fda_debug_last_schedule() == 1
        ora = oracle.local_state(w[:7, :70_001].cpu().numpy(), w0[:70_001].cpu().numpy(), None, coeffs, l, m, threads=8)
        check_states(part[:7].cpu().numpy(), ora, l, m, 70_001)


@pytest.mark.parametrize("l,m", [(1, 250), (3, 250), (4, 250), (5, 250), (6, 250), (7, 250), (9, 250), (7, 500), (4, 1000),
                                 (4, 1200), (8, 1000), (2, 129)])
@pytest.mark.parametrize("K,d,aligned", [(57, 800_001, False), (60, 800_000, True)])
def test_sketches(l, m, K, d, aligned):
    import fda_synth as S
    check(l, m, K, d, S.hash_coefficients(3, l), aligned, l * m + d)


# the split of the warps: 12, 16, 20, 23 or 24 walkers with one item each and more (the first hash that is even)
@pytest.mark.parametrize("l,m", [(4, 64), (4, 96), (4, 128), (5, 128), (3, 200), (7, 96), (5, 160), (4, 288), (6, 200), (6, 250), (3, 500),
                                 (5, 384), (4, 500), (6, 384), (2, 1000), (3, 800), (5, 500), (6, 500), (8, 480), (4, 1000), (8, 560)])
@pytest.mark.parametrize("K,d,aligned", [(57, 900_001, False)])
def test_every_split_of_the_warps(l, m, K, d, aligned):
    import fda_synth as S
    import paper_2405_20988_b200 as F
    few = [schedule_bytes(F, l, m, S.hash_coefficients(s, l), d, k) for s in range(20) for k in (4, K)]
    seed = next(s for s in range(20) if few[2 * s + 1] > 3 * few[2 * s] // 2)
    check(l, m, K, d, S.hash_coefficients(seed, l), aligned, l * m + d)


# both sides of the line for narrow sketches: lanes without a cell, tiles of two batches, and rows
@pytest.mark.parametrize("l,m,lanes", [(8, 71, False), (8, 72, True), (5, 54, False), (5, 55, True), (12, 65, False), (13, 65, True), (8, 100, True)])
def test_narrow_sketches(l, m, lanes):
    import fda_synth as S
    import paper_2405_20988_b200 as F
    K, d = 60, 700_001
    both = [schedule_bytes(F, l, m, S.hash_coefficients(s, l), d, k) for s in range(20) for k in (4, K)]
    even = [s for s in range(20) if both[2 * s + 1] > 3 * both[2 * s] // 2]
    assert (len(even) > 0) == lanes
    seed = even[0] if lanes else 3
    check(l, m, K, d, S.hash_coefficients(seed, l), True, l * m, lanes)


@pytest.mark.parametrize("kind,even", [("one bucket", False), ("short period", False), ("index mod m", True)])
def test_uneven_hashes(kind, even):
    import fda_synth as S
    l, m = 5, 250
    c = S.hash_coefficients(3, l).copy()
    if kind == "one bucket":
        c[6], c[7] = m, 11                     # every index in bucket 11
    elif kind == "short period":
        c[12] = m * pow(7, -1, P) % P           # buckets repeat every seven indices
    else:
        c[18], c[19] = 1, 0                    # neighbours in neighbouring buckets
    check(l, m, 60, 700_003, c, True, 5, even)


# a context that is larger than the call: fewer workers (other groups, so other blocks walk the records), the last tile cut
# in the middle of its record; with K = 60 the first call goes through three launches, the last two at shifted programs
@pytest.mark.parametrize("l,m,d", [(5, 250, 3_000_017), (7, 500, 3_100_002), (8, 1000, 1_000_003), (3, 250, 2_900_001)])
@pytest.mark.parametrize("aligned", [True, False])
def test_calls_below_the_limits_of_the_context(l, m, d, aligned):
    import torch
    import oracle
    import fda_synth as S
    import paper_2405_20988_b200 as F
    K, coeffs = 60, S.hash_coefficients(3, l)
    gen = torch.Generator(device="cuda").manual_seed(d)
    w0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = torch.empty((K, (d + 3) // 4 * 4 + (0 if aligned else 1)), device="cuda")[:, :d]
    w.copy_(w0 + torch.randn((K, d), device="cuda", generator=gen) * 1e-3)
    with F.FdaContext(l, m, coeffs, d_max=d + 50_000, K_max=K + 3) as ctx:
        for k, n, launches in ((K, d, 4 if m < 1000 else 2), (K - 15, d - 130_001, 2), (K, d // 2 // 4 * 4, 2)):
            st = torch.full((k, ctx.state_len), float("nan"), device="cuda")
            ctx.fda_local_state(w[:k, :n], w0[:n], None, 5, st)
            assert (ctx.fda_debug_last_schedule(), ctx.fda_debug_last_launches()) == (2, launches)
            again = torch.empty_like(st)
            ctx.fda_local_state(w[:k, :n], w0[:n], None, 5, again)
            assert torch.equal(st, again)
            rows = [r for r in (0, 3, 44, 51, 52, 55, 59) if r < k]       # of every launch
            ora = oracle.local_state(w[rows, :n].cpu().numpy(), w0[:n].cpu().numpy(), None, coeffs, l, m, threads=8)
            check_states(st[rows].cpu().numpy(), ora, l, m, n)


# tiles to a block below the line from which the idle SMs get the last tiles, and behind it
@pytest.mark.parametrize("tiles,launches", [(35, 2), (40, 4), (41, 4)])
def test_line_of_the_tail_launches(tiles, launches):
    import torch
    import oracle
    import fda_synth as S
    import paper_2405_20988_b200 as F
    l, m, K, coeffs = 5, 250, 60, S.hash_coefficients(3, 5)
    d = tiles * 9 * 6144 - 3
    gen = torch.Generator(device="cuda").manual_seed(d)
    w0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = torch.empty((K, d + 3), device="cuda")[:, :d]
    w.copy_(w0 + torch.randn((K, d), device="cuda", generator=gen) * 1e-3)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        st = torch.full((K, ctx.state_len), float("nan"), device="cuda")
        ctx.fda_local_state(w, w0, None, 5, st)
        assert (ctx.fda_debug_last_schedule(), ctx.fda_debug_last_launches()) == (2, launches)
        rows = [0, 51, 52, 59]
        ora = oracle.local_state(w[rows].cpu().numpy(), w0.cpu().numpy(), None, coeffs, l, m, threads=8)
        check_states(st[rows].cpu().numpy(), ora, l, m, d)


# NaN and infinity of one worker show in its norm and in one cell of every row, and nowhere else
@pytest.mark.parametrize("l,m,K,d", [(5, 250, 60, 900_001), (8, 1000, 57, 600_000)])
@pytest.mark.parametrize("lanes", [True, False])
def test_values_that_are_not_finite(l, m, K, d, lanes):
    import torch
    import oracle
    import fda_synth as S
    import paper_2405_20988_b200 as F
    coeffs = S.hash_coefficients(3, l)
    gen = torch.Generator(device="cuda").manual_seed(9)
    w0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = w0 + torch.randn((K, d), device="cuda", generator=gen) * 1e-3
    xi = None if lanes else torch.full((d,), 1e-3, device="cuda")
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        clean, got = (torch.empty((K, ctx.state_len), device="cuda") for _ in range(2))
        ctx.fda_local_state(w, w0, xi, 7, clean)
        bad = {(1, d - 1): float("nan"), (2, 6143): float("inf"), (K - 1, 0): float("-inf")}
        for (k, j), v in bad.items():
            w[k, j] = v
        ctx.fda_local_state(w, w0, xi, 7, got)
        assert ctx.fda_debug_last_schedule() == (2 if lanes else 1)
    want, got = clean.cpu().numpy(), got.cpu().numpy()
    for (k, j), v in bad.items():
        bucket, sign = oracle.hash_dump(coeffs, l, m, j, 1)
        want[k, 0] = v * v
        if not lanes:
            want[k, 1] = v
        for i in range(l):
            want[k, 2 + i * m + int(bucket[i, 0])] = v * float(sign[i, 0])
    assert np.array_equal(want, got, equal_nan=True)


# the records that the lanes walk: as test_schedule_gpu.py has them, at most 1.6 steps to an entry
@pytest.mark.parametrize("l,m,d", [(5, 250, 800_001), (7, 500, 800_000), (8, 1000, 700_001), (3, 250, 800_000), (2, 129, 800_000)])
def test_records(l, m, d):
    import torch
    import fda_synth as S
    import paper_2405_20988_b200 as F
    from test_schedule_gpu import check_record
    with F.FdaContext(l, m, S.hash_coefficients(3, l), d_max=d, K_max=60) as ctx:
        _, info = ctx.fda_debug_lane_schedule(0)
        T = info["tile_indices"]
        tiles = -(-d // T)
        parts = info["tiles"] // tiles
        assert info["tiles"] == parts * tiles and l % parts == 0
        rows, steps, entries, cells = l // parts, 0, 0, {}
        for record in (0, 1, tiles - 1, info["tiles"] - 1):
            part, tile = divmod(record, tiles)
            b, s = torch.empty((l, T), dtype=torch.int16, device="cuda"), torch.empty((l, T), dtype=torch.int8, device="cuda")
            ctx.fda_debug_hash(tile * T, T, b, s)
            rec, info = ctx.fda_debug_lane_schedule(record)
            own = slice(part * rows, (part + 1) * rows)
            n, e = check_record(rec, info, rows, m, b.cpu().numpy().view(np.uint16).astype(np.int64)[own], s.cpu().numpy()[own])
            steps, entries = steps + n, entries + e
            # a lane's cell is the same in every tile (l*m where the tile has no index of it)
            items = int(rec[:4].view(np.uint32)[0])
            at = (16 + 8 * items + 63) // 64 * 64
            of = rec[at:at + 64 * items].view(np.uint16).astype(np.int64)
            known = cells.setdefault(part, of.copy())
            assert ((of == known) | (of == rows * m) | (known == rows * m)).all()
            assert not (of & 0x8000).any()
        assert steps <= 1.6 * entries
        with pytest.raises(F.FdaError):
            ctx.fda_debug_lane_schedule(info["tiles"])
    with F.FdaContext(l, m, S.hash_coefficients(3, l), d_max=50_000, K_max=60) as ctx:
        with pytest.raises(F.FdaError):
            ctx.fda_debug_lane_schedule(0)


def test_a_second_schedule_that_does_not_fit_is_reported():
    import torch
    import fda_synth as S
    import paper_2405_20988_b200 as F
    l, m, d, K = 5, 250, 800_000, 60
    coeffs = S.hash_coefficients(3, l)
    first = schedule_bytes(F, l, m, coeffs, d, 4)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K, schedule_limit_bytes=first + 1000) as ctx:
        info = ctx.fda_context_info()
        assert info["schedule_bytes"] == first and first // 2 < info["schedule_dropped_bytes"] < 2 * first
        st = torch.empty((K, ctx.state_len), device="cuda")
        ctx.fda_local_state(torch.ones((K, d), device="cuda"), torch.zeros(d, device="cuda"), None, 5, st)
        assert ctx.fda_debug_last_schedule() == 1


def test_the_second_schedule_can_be_left_out():
    import torch
    import fda_synth as S
    import paper_2405_20988_b200 as F
    l, m, d, K = 5, 250, 800_000, 60
    coeffs = S.hash_coefficients(3, l)
    gen = torch.Generator(device="cuda").manual_seed(1)
    w0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = w0 + torch.randn((K, d), device="cuda", generator=gen) * 1e-3
    xi = torch.randn(d, device="cuda", generator=gen)
    got = []
    for one in (True, False):
        with F.FdaContext(l, m, coeffs, d_max=d, K_max=K, one_schedule=one) as ctx:
            info = ctx.fda_context_info()
            assert info["list_kernel"] == 1 and info["schedule_dropped_bytes"] == 0
            st, xi_st = (torch.empty((K, ctx.state_len), device="cuda") for _ in range(2))
            mean = torch.empty(ctx.state_len, device="cuda")
            ctx.fda_local_state(w, w0, None, 5, st)
            assert ctx.fda_debug_last_schedule() == (1 if one else 2)
            ctx.fda_local_state(w, w0, xi, 7, xi_st)
            ctx.fda_mean_state(w, w0, xi, 7, mean)
            got.append((info["schedule_bytes"], st.cpu().numpy(), xi_st, mean))
    assert got[0][0] == schedule_bytes(F, l, m, coeffs, d, 4) < got[1][0]
    check_states(got[0][1], got[1][1].astype(np.float64), l, m, d)
    assert torch.equal(got[0][2], got[1][2]) and torch.equal(got[0][3], got[1][3])
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K, one_schedule=True, schedule_limit_bytes=-1) as ctx:
        assert ctx.fda_context_info()["list_kernel"] == 0
