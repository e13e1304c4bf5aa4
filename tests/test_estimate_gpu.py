"""The estimate of fda_combine_estimate as its host caller gets it: what is promised when the call
returns, and contexts beyond those that the library keeps mapped host memory for."""
import ctypes

import numpy as np
import pytest

import fda_synth as S

pytestmark = pytest.mark.gpu


def _fields(raw):
    import paper_2405_20988_b200 as F
    e = F.Estimate.from_buffer_copy(bytes(raw))
    return (e.mean_sq_norm, e.est_sq_norm_of_mean, e.H, e.theta, e.trigger, e.l, tuple(e.row_sq_norm))


# states of 24 x (2 + 5 x 250) floats are taken by several blocks, of 3 x (2 + 16 x 64) and of a context without sketch by one
@pytest.mark.parametrize("l,m,K", [(5, 250, 24), (16, 64, 3), (0, 1, 5)])
def test_device_estimate_is_complete_when_the_call_returns(l, m, K):
    """est_dev is read on another stream, with nothing but the call's return in front of it."""
    import torch
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(l + K)
    size, calls = ctypes.sizeof(F.Estimate), 300
    with F.FdaContext(l, m, S.hash_coefficients(3, l), d_max=64, K_max=K) as ctx:
        variant = F.FDA_VARIANT_SKETCH if l else F.FDA_VARIANT_LINEAR
        states = torch.from_numpy(rng.normal(0, 1, size=(calls, K, ctx.state_len)).astype(np.float32)).cuda()
        states[:, :, 0].abs_()
        est = ctx.new_estimate_buffer()
        read = torch.zeros((calls, size), dtype=torch.uint8, device="cuda")
        writer, reader = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        host = []
        for t in range(calls):
            host.append(_fields(ctx.fda_combine_estimate(states[t], K, variant, 0.06, 0.5, est, stream=writer)))
            with torch.cuda.stream(reader):
                read[t].copy_(est)
            reader.synchronize()                 # (the next call writes est again)
        got = read.cpu().numpy()
    assert len(set(host)) == calls               # every call's estimate is another one
    for t in range(calls):
        assert _fields(got[t]) == host[t]


@pytest.mark.parametrize("m", [4, 5000])              # one block, several blocks
@pytest.mark.parametrize("cells", [[1, np.nan, np.nan, np.nan, 2], [3, np.nan, 1, 2, 5], [np.nan] * 5, [np.inf, 1, np.inf, np.inf, 2],
                                   [1, np.nan, 2, 3], [np.nan, 1, np.nan, 2], [2, np.inf, np.nan, 1], [4, 4, 1, 4, np.nan, 1]])
def test_median_of_rows_that_are_not_all_numbers(cells, m):
    """NaN counts as the largest: the median is a number while fewer than half of the rows are NaN."""
    import torch
    import paper_2405_20988_b200 as F
    l = len(cells)
    state = np.zeros((1, 2 + l * m), dtype=np.float32)
    state[0, 0] = 7.0
    state[0, 3::m] = cells
    rows = np.sort(np.square(np.array(cells, dtype=np.float64)))
    want = rows[l // 2] if l % 2 else 0.5 * (rows[l // 2 - 1] + rows[l // 2])
    with F.FdaContext(l, m, S.hash_coefficients(3, l), d_max=64, K_max=1) as ctx:
        est = ctx.fda_combine_estimate(torch.from_numpy(state).cuda(), 1, F.FDA_VARIANT_SKETCH, 0.0, 1.0, ctx.new_estimate_buffer())
    assert np.array_equal(np.float32(est.est_sq_norm_of_mean), np.float32(want), equal_nan=True)
    assert np.array_equal(np.float32(est.H), np.float32(7.0 - want), equal_nan=True)
    assert est.trigger == int(7.0 - want > 1.0)


def test_contexts_beyond_the_mapped_page():
    """The page of mapped host memory has 32 slots: the contexts beyond them copy the estimate, and
    a slot that a context has given back serves another one, whose first estimate is not the old one."""
    import torch
    import paper_2405_20988_b200 as F
    K, l, m = 3, 2, 16
    rng = np.random.default_rng(1)

    def estimate(ctx):
        states = torch.from_numpy(np.abs(rng.normal(0, 1, size=(K, ctx.state_len))).astype(np.float32)).cuda()
        est = ctx.new_estimate_buffer()
        host = ctx.fda_combine_estimate(states, K, F.FDA_VARIANT_SKETCH, 0.06, 0.5, est)
        mean = states.double().mean(dim=0).cpu().numpy()
        rows = np.square(mean[2:].reshape(l, m)).sum(axis=1)
        assert host.mean_sq_norm == pytest.approx(mean[0], rel=1e-6)
        assert host.est_sq_norm_of_mean == pytest.approx(rows.mean() / 1.06, rel=1e-6)
        assert list(host.row_sq_norm[:l]) == pytest.approx(rows, rel=1e-6)
        assert _fields(est.cpu().numpy()) == _fields(bytes(host))

    held = [F.FdaContext(l, m, S.hash_coefficients(k, l), d_max=64, K_max=K) for k in range(36)]
    try:
        for _ in range(2):
            for ctx in held:
                estimate(ctx)
            for k in range(0, 36, 5):            # slots go round, to contexts that had none among others
                held[k].close()
                held[k] = F.FdaContext(l, m, S.hash_coefficients(k, l), d_max=64, K_max=K)
    finally:
        for ctx in held:
            ctx.close()
