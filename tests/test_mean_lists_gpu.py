"""The averaged state from the lists, over the vector of averaged drifts (k_mean_sketch_short)."""
import numpy as np
import pytest

from fda_testlib import check_mean_state

pytestmark = pytest.mark.gpu
SMS = 148
ROUTE = "k_mean_model + k_mean_state_gather"


# 5 x 250 and 1 x 250 (tiles of 6144): three, two and one block to a tile, ends of a tile, the last d before a block has two tiles;
# 7 x 500 (5120): one tile a block, two blocks to an SM, several tiles a block; 8 x 1000: rows in parts, a tile of which has one,
# two and more blocks; 16 x 120: cells with several lists; 6 x 200 and 12 x 300: items of more than the chunks asked for at once
@pytest.mark.parametrize("l,m,K,d", [
    (5, 250, 11, 1), (5, 250, 11, 6143), (5, 250, 20, 6145), (5, 250, 12, 49 * 6144), (5, 250, 12, 49 * 6144 + 1),
    (1, 250, 11, 74 * 6144 + 3), (5, 250, 11, SMS * 6144 - 1), (6, 200, 13, 40_001),
    (7, 500, 15, 5121), (7, 500, 15, SMS * 5120 + 1), (7, 500, 16, 2 * SMS * 5120 + 5), (7, 500, 15, 900 * 5120 + 7),
    (8, 1000, 4, 4_099), (8, 1000, 17, 24 * 5120 + 2), (8, 1000, 17, 37 * 5120 + 1), (8, 1000, 3, SMS * 5120 + 9),
    (16, 120, 11, 30_001), (12, 300, 25, 50_003)])
def test_lists_over_the_averaged_drifts(l, m, K, d):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(l * 1000 + K + d)
    coeffs = rng.integers(1, (1 << 61) - 1, size=6 * l, dtype=np.uint64)
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    wbuf = np.zeros((K, d + 1), dtype=np.float32)              # (an odd pitch or an odd start: the rows are not 16-byte aligned)
    wbuf[:, :d] = w_t0 + rng.normal(2e-4, 1e-3, size=(K, d)).astype(np.float32)
    u = wbuf[:, :d].astype(np.float64) - w_t0
    ubar = u.mean(axis=0)
    # linear: the state of the averaged drift has the averaged cells
    ora = oracle.local_state(ubar.astype(np.float32)[None], np.zeros(d, np.float32), None, coeffs, l, m, threads=8)
    ora = np.repeat(ora, K, axis=0)
    ora[:, 0] = (u * u).sum(axis=1)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        assert ctx.fda_context_info()["list_kernel"] == 1
        buf = torch.zeros(K * (d + 1) + 1, device="cuda")
        w = buf[1:].view(K, d + 1)
        w.copy_(torch.from_numpy(wbuf))
        w0 = torch.from_numpy(w_t0).cuda()
        first, again = (torch.full((ctx.state_len,), float("nan"), device="cuda") for _ in range(2))
        for out in (first, again):
            ctx.fda_mean_state(w[:, :d], w0, None, 5, out)
        assert ctx.fda_debug_last_kernel() == ROUTE and ctx.fda_debug_last_schedule() == 1
        assert ctx.fda_context_info()["table_bytes"] == 0
        if (l, m) != (16, 120):                                 # (lists of one cell are added atomically there)
            assert torch.equal(first, again)
        check_mean_state(first.cpu().numpy(), ora, float(ubar @ ubar), l, m, d, K)
        # a shorter vector on the same context
        if d > 12_000:
            n = d // 2 | 1
            part = oracle.local_state(ubar[:n].astype(np.float32)[None], np.zeros(n, np.float32), None, coeffs, l, m, threads=8)
            part = np.repeat(part, K, axis=0)
            part[:, 0] = (u[:, :n] ** 2).sum(axis=1)
            ctx.fda_mean_state(w[:, :n], w0[:n], None, 5, first)
            check_mean_state(first.cpu().numpy(), part, float(ubar[:n] @ ubar[:n]), l, m, n, K)
