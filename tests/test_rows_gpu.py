"""The streaming pass of fda_rows.cuh behind both entry points that use it, at the sizes where its
quads, windows and row groups have edges, with rows, w_t0 and xi each at an alignment of their own;
and the two shapes of the combine kernel on either side of the size where the choice changes."""
import numpy as np
import pytest

from fda_testlib import check_estimate, check_states

pytestmark = pytest.mark.gpu


def at(torch, a, misalign):
    """The array on the device, starting `misalign` elements behind a 16-byte boundary."""
    buf = torch.zeros(a.size + 8, dtype=torch.float32, device="cuda")
    view = buf[misalign:misalign + a.size].view(a.shape)
    view.copy_(torch.from_numpy(a))
    return view


@pytest.mark.parametrize("d", [1, 7, 8, 11, 12, 1023, 1031, 5003])
@pytest.mark.parametrize("K,pitch_extra,mis", [(1, 0, (0, 0, 0)), (5, 1, (0, 0, 0)), (6, 2, (1, 0, 0)), (11, 3, (2, 3, 3)),
                                               (4, 4, (3, 1, 2)), (10, 0, (0, 2, 1))])
def test_rows_at_any_alignment(d, K, pitch_extra, mis):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(1000 * d + K)
    pitch = (d + 3) // 4 * 4 + pitch_extra
    w_t0 = rng.normal(0, 0.05, size=d).astype(np.float32)
    wbuf = np.full((K, pitch), 1e6, dtype=np.float32)            # what lies between the rows must not be read into the sums
    wbuf[:, :d] = w_t0 + rng.normal(0, 1e-3, size=(K, d)).astype(np.float32)
    xi = rng.normal(size=d)
    xi = (xi / np.linalg.norm(xi)).astype(np.float32)
    w, w0, xg = at(torch, wbuf, mis[0])[:, :d], at(torch, w_t0, mis[1]), at(torch, xi, mis[2])
    ora = oracle.local_state(wbuf[:, :d], w_t0, xi, None, 0, 0)
    with F.FdaContext(0, 0, None, d_max=d, K_max=K) as ctx:
        for flags, x in ((3, xg), (1, None)):
            ref = ora.copy()
            if not flags & 2:
                ref[:, 1] = 0.0
            for _ in range(2):                                   # the group tickets are back at zero
                st = torch.full((K, 2), float("nan"), device="cuda")
                ctx.fda_local_state(w, w0, x, flags, st)
                hook = torch.full((K, 2), float("nan"), device="cuda")
                F.fda_local_state_linear_noalloc(w, w0, x, flags, hook)
                check_states(st.cpu().numpy(), ref, 0, 0, d)
                check_states(hook.cpu().numpy(), ref, 0, 0, d)


@pytest.mark.parametrize("l,m,K", [(1, 1, 1), (5, 250, 9), (5, 250, 10), (6, 65, 31), (6, 65, 32), (16, 64, 12), (2, 600, 70)])
def test_combine_on_both_sides_of_its_rule(l, m, K):
    import torch
    import oracle
    import paper_2405_20988_b200 as F
    rng = np.random.default_rng(l * m + K)
    st = rng.normal(0, 0.1, size=(K, 2 + l * m)).astype(np.float32)
    st[:, 0] = np.abs(st[:, 0]) + 1.0
    coeffs = rng.integers(1, 1 << 60, size=6 * l, dtype=np.uint64)
    with F.FdaContext(l, m, coeffs, d_max=1000, K_max=K) as ctx:
        g, buf = torch.from_numpy(st).cuda(), ctx.new_estimate_buffer()
        for variant in (0, 1, 1):
            ref = oracle.combine(st, l, m, variant, 0.06, 0.5)
            est = ctx.fda_combine_estimate(g, K, variant, float(np.float32(0.06)), 0.5, buf)
            check_estimate(est.as_dict(), ref, l)
            assert bytes(buf.cpu().numpy()) == bytes(est)
