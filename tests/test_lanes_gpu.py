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
            assert bool(torch.isfinite(st[0]).all())
            check_states(st[0][ks].cpu().numpy(), want, l, m, d)
            if flags == 5 and even:            # no sum's order is left to chance
                assert torch.equal(st[0], st[1])
        part = torch.full((K, ctx.state_len), float("nan"), device="cuda")      # fewer workers, a shorter vector
        ctx.fda_local_state(w[:7, :70_001], w0[:70_001], None, 5, part)
        ora = oracle.local_state(w[:7, :70_001].cpu().numpy(), w0[:70_001].cpu().numpy(), None, coeffs, l, m, threads=8)
        check_states(part[:7].cpu().numpy(), ora, l, m, 70_001)


@pytest.mark.parametrize("l,m", [(1, 250), (3, 250), (4, 250), (5, 250), (6, 250), (7, 250), (9, 250), (7, 500), (4, 1000),
                                 (4, 1200), (8, 1000), (2, 129)])
@pytest.mark.parametrize("K,d,aligned", [(57, 800_001, False), (60, 800_000, True)])
def test_sketches(l, m, K, d, aligned):
    import fda_synth as S
    check(l, m, K, d, S.hash_coefficients(3, l), aligned, l * m + d)


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
