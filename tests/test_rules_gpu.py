"""Both sides of the lines at which a call goes to another kernel, against the oracle."""
import numpy as np
import pytest

import fda_synth as S
from fda_testlib import REL, check_estimate, check_states

pytestmark = pytest.mark.gpu

SMS = 148


def _inputs(l, K, d, pitch_extra, seed):
    rng = np.random.default_rng(seed)
    pitch = (d + 3) // 4 * 4 + pitch_extra
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    wbuf = np.full((K, pitch), 1e6, dtype=np.float32)
    wbuf[:, :d] = w_t0 + rng.normal(2e-4, 1e-3, size=(K, d)).astype(np.float32)
    xi = rng.normal(size=d)
    return wbuf, w_t0, (xi / np.linalg.norm(xi)).astype(np.float32), S.hash_coefficients(seed, l)


# blocks of one tile: the most that still share tiles (74), one more, one for every SM, and the first vector with
# two tiles to a block; sketches of up to six rows and of more go to different kernels in between
@pytest.mark.parametrize("pitch_extra", [0, 1])
@pytest.mark.parametrize("l,m,K,tiles,more", [(5, 250, 10, 24, 0), (5, 250, 10, 24, 1), (5, 250, 9, 49, 0), (5, 250, 10, 49, 1),
                                              (6, 400, 5, 74, 0), (6, 400, 20, 14, 5), (7, 500, 10, 25, -3), (7, 500, 3, 75, 0),
                                              (1, 250, 3, 148, -1)])
def test_vectors_of_one_tile_per_block(l, m, K, tiles, more, pitch_extra):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    T = 6144 if m == 250 else 5120
    d = tiles * T + more
    wbuf, w_t0, xi, coeffs = _inputs(l, K, d, pitch_extra, l * m + tiles)
    ora = oracle.local_state(wbuf[:, :d], w_t0, xi, coeffs, l, m, threads=8)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        assert ctx.fda_context_info()["tile_indices"] == T
        st = torch.full((K, ctx.state_len), float("nan"), device="cuda")
        ctx.fda_local_state(torch.from_numpy(wbuf).cuda()[:, :d], torch.from_numpy(w_t0).cuda(), torch.from_numpy(xi).cuda(), 7, st)
        assert ctx.fda_debug_last_kernel() == "k_local_state_gather"
    check_states(st.cpu().numpy(), ora, l, m, d)


# round trips of a warp: 3 | 4 of one batch of columns, 2 | 4 of two, 4 of four, 3 | 4 of batches of columns
@pytest.mark.parametrize("l,m,K", [(3, 100, 24), (3, 100, 25), (5, 250, 8), (5, 250, 9), (7, 500, 1), (16, 96, 8), (16, 97, 8), (1, 960, 24), (1, 960, 25)])
def test_combine_by_one_block_and_by_several(l, m, K):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(l * m + K)
    st = rng.normal(0, 0.1, size=(K, 2 + l * m)).astype(np.float32)
    st[:, 0] = np.abs(st[:, 0]) + 1.0
    with F.FdaContext(l, m, S.hash_coefficients(2, l), d_max=1000, K_max=K) as ctx:
        g, buf = torch.from_numpy(st).cuda(), ctx.new_estimate_buffer()
        for variant in (0, 1, 1):
            est = ctx.fda_combine_estimate(g, K, variant, float(np.float32(0.06)), 0.5, buf)
            check_estimate(est.as_dict(), oracle.combine(st, l, m, variant, 0.06, 0.5), l)
            assert bytes(buf.cpu().numpy()) == bytes(est)


def _at(torch, a, misalign):
    buf = torch.zeros(a.size + 8, dtype=torch.float32, device="cuda")
    view = buf[misalign:misalign + a.size].view(a.shape)
    view.copy_(torch.from_numpy(a))
    return view


# indices per SM up to which an index has a thread of its own; behind that line the quads, whose edges the offsets meet
@pytest.mark.parametrize("over", [0, 1, 2, 140, 1027])
@pytest.mark.parametrize("K,per_sm,extra,mis", [(4, 768, 0, (0, 0, 0)), (7, 768, 1, (1, 3, 2)), (8, 1536, 0, (0, 1, 0)), (11, 1536, 3, (3, 0, 1)),
                                                (32, 768, 0, (0, 0, 0)), (33, 1536, 0, (0, 0, 0)), (33, 4096, 2, (0, 0, 3))])
def test_average_by_index_and_by_quads(K, per_sm, extra, mis, over):
    import torch
    import paper_2405_20988_b200 as F
    d = SMS * per_sm + over
    rng = np.random.default_rng(d + K)
    wbuf = rng.normal(0, 0.05, size=(K, (d + 3) // 4 * 4 + extra)).astype(np.float32)
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    acc = np.zeros(d, dtype=np.float32)
    for k in range(K):
        acc = acc + wbuf[k, :d]
    mean = acc * (np.float32(1.0) / np.float32(K))
    delta = (mean - w_t0).astype(np.float64)
    delta /= np.linalg.norm(delta)
    with F.FdaContext(0, 0, None, d_max=d, K_max=K) as ctx:
        for bc in (0, F.FDA_AVG_BROADCAST):
            w, w0 = _at(torch, wbuf, mis[0]), _at(torch, w_t0, mis[1])
            ctx.fda_average_models(w[:, :d], w0, None, bc)
            got = w.cpu().numpy()
            assert np.array_equal(w0.cpu().numpy(), mean)
            assert np.array_equal(got[:, d:], wbuf[:, d:])
            assert np.array_equal(got[:, :d], np.broadcast_to(mean, (K, d)) if bc else wbuf[:, :d])
        w, w0, xi = _at(torch, wbuf, mis[0]), _at(torch, w_t0, mis[1]), _at(torch, np.zeros(d, np.float32), mis[2])
        ctx.fda_average_models_xi(w[:, :d], w0, xi, None, F.FDA_AVG_BROADCAST)
        assert np.array_equal(w0.cpu().numpy(), mean) and np.array_equal(w.cpu().numpy()[:, :d], np.broadcast_to(mean, (K, d)))
        # single precision on both sides of a difference of numbers around mean |w|, unit length
        assert np.max(np.abs(xi.cpu().numpy() - delta)) <= 1e-5


# the split of the warps: l * (1 + 10 * m / T) below ten and from ten on, seven rows on either side of it, eight and more
@pytest.mark.parametrize("l,m", [(5, 500), (5, 600), (6, 250), (6, 400), (7, 250), (7, 300), (8, 100)])
@pytest.mark.parametrize("K,d,pitch_extra", [(9, 200_003, 0), (4, 2_500_001, 2)])
def test_both_splits_of_the_warps(l, m, K, d, pitch_extra):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    wbuf, w_t0, xi, coeffs = _inputs(l, K, d, pitch_extra, l * m)
    ora = oracle.local_state(wbuf[:, :d], w_t0, xi, coeffs, l, m, threads=8)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        st = torch.full((K, ctx.state_len), float("nan"), device="cuda")
        ctx.fda_local_state(torch.from_numpy(wbuf).cuda()[:, :d], torch.from_numpy(w_t0).cuda(), torch.from_numpy(xi).cuda(), 7, st)
        assert ctx.fda_debug_last_kernel() == "k_local_state_gather"
    check_states(st.cpu().numpy(), ora, l, m, d)


# rows that are not 16-byte aligned: one pass up to ten workers or twice the sketch rows, from eight tiles per SM where
# the second kernel of the other route has lane-private bins, from two where it walks the lists too
@pytest.mark.parametrize("l,m,K,tiles,one_pass", [(3, 100, 10, 8, True), (3, 100, 11, 8, False), (3, 100, 3, 7, False), (5, 250, 10, 8, True),
                                                  (7, 500, 14, 2, True), (7, 500, 15, 2, False), (7, 500, 3, 1, False)])
def test_averaged_state_of_unaligned_rows(l, m, K, tiles, one_pass):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    T = 5120 if m == 500 else 6144
    d = tiles * SMS * T - 7
    wbuf, w_t0, xi, coeffs = _inputs(l, K, d, 2, l * m + K)
    # the sketch is linear: the oracle's state of the averaged drift, and the averages of the scalars
    u = wbuf[:, :d].astype(np.float64) - w_t0
    ubar = u.mean(axis=0)
    ora = oracle.local_state(ubar.astype(np.float32)[None], np.zeros(d, np.float32), xi, coeffs, l, m, threads=8)[0]
    norm, proj = float((u * u).sum(axis=1).mean()), float((u @ xi.astype(np.float64)).mean())
    ubar_sq = float(ubar @ ubar)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        assert ctx.fda_context_info()["tile_indices"] == T
        mean = torch.full((ctx.state_len,), float("nan"), device="cuda")
        ctx.fda_mean_state(torch.from_numpy(wbuf).cuda()[:, :d], torch.from_numpy(w_t0).cuda(), torch.from_numpy(xi).cuda(), 7, mean)
        assert (ctx.fda_debug_last_kernel() == "k_mean_state_gather") == one_pass
        assert (ctx.fda_context_info()["other_lazy_bytes"] == 0) == one_pass
    got = mean.cpu().numpy().astype(np.float64)
    assert abs(got[0] - norm) <= REL * norm
    assert abs(got[1] - proj) <= REL * max(abs(proj), np.sqrt(ubar_sq / d))
    # u-bar reaches the oracle in single precision (2^-24), a cell is held to REL of its scale
    assert np.max(np.abs(got[2:] - ora[2:]) / np.maximum(np.abs(ora[2:]), np.sqrt(ubar_sq / m))) <= REL


# more worker groups than SMs: the plain-load kernels, also on a context with a schedule
@pytest.mark.parametrize("l,m,K", [(2, 16, 4 * SMS), (2, 16, 4 * SMS + 1), (8, 1000, 2 * SMS), (8, 1000, 2 * SMS + 1)])
def test_more_worker_groups_than_sms(l, m, K):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    d = 1027
    wbuf, w_t0, xi, coeffs = _inputs(l, K, d, 0, K)
    ora = oracle.local_state(wbuf[:, :d], w_t0, xi, coeffs, l, m, threads=8)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        assert ctx.fda_context_info()["list_kernel"] == 1
        st = torch.full((K, ctx.state_len), float("nan"), device="cuda")
        ctx.fda_local_state(torch.from_numpy(wbuf).cuda()[:, :d], torch.from_numpy(w_t0).cuda(), torch.from_numpy(xi).cuda(), 7, st)
        assert (ctx.fda_debug_last_kernel() == "k_local_state_gather") == (K % SMS == 0)
    check_states(st.cpu().numpy(), ora, l, m, d)
