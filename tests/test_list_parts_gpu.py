"""Branches of the list kernel's dispatch: sketches whose rows are in several parts with records of
their own (lists of five entries fit a part where the whole sketch leaves no room for them), and
vectors of so few tiles that several blocks share the items of one.  States and averaged states
against the oracle at the edges of tiles, worker groups and parts."""
import numpy as np
import pytest

from fda_testlib import check_mean_state, check_states

pytestmark = pytest.mark.gpu

P = (1 << 61) - 1


@pytest.mark.parametrize("l,m,K,d,aligned", [
    (8, 1000, 5, 1, True), (8, 1000, 20, 5 * 5120 - 1, True), (8, 1000, 21, 150_001, False),       # two parts
    (16, 600, 9, 40_961, True), (4, 1200, 3, 30_720, False),
    (5, 250, 5, 6144, True), (5, 250, 4, 6145, False), (5, 250, 37, 12_289, True),                 # shared tiles
    (7, 500, 10, 10_241, True), (3, 100, 6, 61_706, False),
    (7, 500, 21, 150_001, True), (8, 1000, 9, 120_003, False), (16, 600, 8, 200_002, True)])       # finalize, four workers to a lane
def test_parts_and_shared_tiles(l, m, K, d, aligned):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(l * m + d)
    coeffs = rng.integers(0, P, size=6 * l, dtype=np.uint64)
    coeffs[0::6] |= np.uint64(1)
    coeffs[2::6] |= np.uint64(1)
    pitch = (d + 3) // 4 * 4 + (0 if aligned else 3)
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    wbuf = np.full((K, pitch), 1e6, dtype=np.float32)
    wbuf[:, :d] = w_t0 + rng.normal(2e-4, 1e-3, size=(K, d)).astype(np.float32)
    xi = rng.normal(size=d)
    xi = (xi / np.linalg.norm(xi)).astype(np.float32)
    ora = oracle.local_state(wbuf[:, :d], w_t0, xi, coeffs, l, m, threads=4)
    ubar_sq = float(np.sum((wbuf[:, :d].astype(np.float64) - w_t0).mean(axis=0) ** 2))
    w, w0, xg = (torch.from_numpy(a).cuda() for a in (wbuf, w_t0, xi))
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        assert ctx.fda_context_info()["list_kernel"] == 1
        for _ in range(2):
            st = torch.full((K, ctx.state_len), float("nan"), device="cuda")
            ctx.fda_local_state(w[:, :d], w0, xg, 7, st)
            assert ctx.fda_debug_last_kernel() == "k_local_state_gather" and ctx.fda_debug_last_launches() == 2
            check_states(st.cpu().numpy(), ora, l, m, d)
        mean = torch.full((ctx.state_len,), float("nan"), device="cuda")
        ctx.fda_mean_state(w[:, :d], w0, xg, 7, mean)
        check_mean_state(mean.cpu().numpy(), ora, ubar_sq, l, m, d, K)
