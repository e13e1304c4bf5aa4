"""Passes that combine the rows of w index by index at any alignment (fda_quads.cuh), at the sizes
where quads, windows and warps' runs end: the model average with and without broadcast and direction,
exactly in the order of its sums, and the averaged norm of fda_mean_state; and the averaged state in
one pass when a quad's rows arrive in several slots."""
import numpy as np
import pytest

from fda_testlib import check_mean_state

pytestmark = pytest.mark.gpu

P = (1 << 61) - 1


def at(torch, a, misalign):
    buf = torch.zeros(a.size + 8, dtype=torch.float32, device="cuda")
    view = buf[misalign:misalign + a.size].view(a.shape)
    view.copy_(torch.from_numpy(a))
    return view


@pytest.mark.parametrize("d", [1, 11, 12, 17, 139, 140, 1029, 75_776, 75_777, 75_916, 76_803])   # (both sides of the lines: test_rules_gpu.py)
@pytest.mark.parametrize("K,extra,mis", [(1, 0, (1, 0, 0)), (3, 1, (0, 0, 0)), (4, 2, (0, 3, 0)), (5, 3, (2, 2, 2)), (9, 1, (3, 1, 2)),
                                         (33, 3, (0, 0, 0)), (4, 0, (0, 0, 0))])
def test_average_at_any_alignment(d, K, extra, mis):
    import torch
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(100 * d + K)
    pitch = (d + 3) // 4 * 4 + extra
    wbuf = rng.normal(0, 0.05, size=(K, pitch)).astype(np.float32)
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    acc = np.zeros(d, dtype=np.float32)
    for k in range(K):
        acc = acc + wbuf[k, :d]
    mean = acc * (np.float32(1.0) / np.float32(K))
    delta = (mean - w_t0).astype(np.float64)
    xi_ref = delta / np.linalg.norm(delta)
    norms = ((wbuf[:, :d].astype(np.float64) - w_t0) ** 2).sum(axis=1)
    with F.FdaContext(0, 0, None, d_max=d, K_max=K) as ctx:
        w, w0 = at(torch, wbuf, mis[0]), at(torch, w_t0, mis[1])
        st = torch.empty(2, device="cuda")
        ctx.fda_mean_state(w[:, :d], w0, None, 1, st)
        assert abs(float(st[0]) - norms.mean()) <= 1e-5 * norms.mean()
        for bc in (0, F.FDA_AVG_BROADCAST):
            w, w0 = at(torch, wbuf, mis[0]), at(torch, w_t0, mis[1])
            ctx.fda_average_models(w[:, :d], w0, None, bc)
            got = w.cpu().numpy()
            assert np.array_equal(w0.cpu().numpy(), mean)
            assert np.array_equal(got[:, d:], wbuf[:, d:])                      # nothing between the rows is written
            assert np.array_equal(got[:, :d], np.tile(mean, (K, 1)) if bc else wbuf[:, :d])
        w, w0, xi = at(torch, wbuf, mis[0]), at(torch, w_t0, mis[1]), at(torch, np.zeros(d, np.float32), mis[2])
        ctx.fda_average_models_xi(w[:, :d], w0, xi, None, F.FDA_AVG_BROADCAST)
        assert np.array_equal(w0.cpu().numpy(), mean) and np.array_equal(w.cpu().numpy()[:, :d], np.tile(mean, (K, 1)))
        assert np.max(np.abs(xi.cpu().numpy() - xi_ref)) <= 1e-5


@pytest.mark.parametrize("rounds,extra,pitch_extra", [(4, 0, 0), (4, 1, 0), (5, 1023, 0), (8, 3, 1), (8, 12, 1), (9, 501, 2)])
def test_average_of_long_vectors(rounds, extra, pitch_extra):
    # around the size from which blocks take chunks by ticket (4 rounds of the grid, 8 when rows are not aligned), called again and again
    import torch
    import paper_2405_20988_b200 as F
    K, d = 3, rounds * torch.cuda.get_device_properties(0).multi_processor_count * 8 * 1024 + extra
    pitch = (d + 3) // 4 * 4 + pitch_extra
    gen = torch.Generator(device="cuda").manual_seed(d)
    with F.FdaContext(0, 0, None, d_max=d, K_max=K) as ctx:
        for bc in (0, F.FDA_AVG_BROADCAST, 0):
            wbuf = torch.randn((K, pitch), device="cuda", generator=gen)
            before, w0 = wbuf.clone(), torch.zeros(d, device="cuda")
            rows = before.cpu().numpy()[:, :d]
            mean = (rows[0] + rows[1] + rows[2]) * (np.float32(1.0) / np.float32(K))
            ctx.fda_average_models(wbuf[:, :d], w0, None, bc)
            assert np.array_equal(w0.cpu().numpy(), mean)
            assert torch.equal(wbuf[:, d:], before[:, d:])
            assert torch.equal(wbuf[:, :d], w0.expand(K, d) if bc else before[:, :d])


@pytest.mark.parametrize("K,tiles,extra,pitch_extra", [(11, 2, 13, 0), (21, 2, 0, 0), (3, 8, 2, 1)])
def test_averaged_state_in_one_pass(K, tiles, extra, pitch_extra):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    l, m = 3, 100
    d = tiles * torch.cuda.get_device_properties(0).multi_processor_count * 6144 + extra
    rng = np.random.default_rng(K)
    coeffs = rng.integers(1, P, size=6 * l, dtype=np.uint64)
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    pitch = (d + 3) // 4 * 4 + pitch_extra
    wbuf = np.zeros((K, pitch), dtype=np.float32)
    for k in range(K):
        wbuf[k, :d] = w_t0 + rng.standard_normal(d, dtype=np.float32) * np.float32(1e-3) + np.float32(2e-4)
    xi = rng.standard_normal(d, dtype=np.float32) / np.float32(np.sqrt(d))
    ora = oracle.local_state(wbuf[:, :d], w_t0, xi, coeffs, l, m, threads=8)
    _, _, ubar_sq = oracle.variance(wbuf[:, :d], w_t0)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        mean = torch.full((ctx.state_len,), float("nan"), device="cuda")
        ctx.fda_mean_state(torch.from_numpy(wbuf).cuda()[:, :d], torch.from_numpy(w_t0).cuda(), torch.from_numpy(xi).cuda(),
                           7, mean)
        assert ctx.fda_debug_last_kernel() == "k_mean_state_gather"
        check_mean_state(mean.cpu().numpy(), ora, ubar_sq, l, m, d, K)
