"""The line from which cells stay with their lanes on vectors of a few tiles to a block: four tiles (the list kernel,
also with the sketch rows in parts, whose warps form the first tile together) and more (lanes), with a last tile that
ends inside a batch.  Tolerance: the usual one of a state."""
import pytest

from fda_testlib import check_states

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l,m,K", [(5, 250, 14), (3, 100, 41), (7, 500, 44), (7, 250, 30), (4, 1000, 20), (8, 1000, 26)])
@pytest.mark.parametrize("full,more", [(0, 1), (1, 0), (3, 1), (4, 0), (4, 1), (5, 0), (12, 1)])
@pytest.mark.parametrize("aligned", [True, False])
def test_few_tiles_to_a_block(l, m, K, full, more, aligned):
    import torch
    import oracle
    import fda_synth as S
    import paper_2405_20988_b200 as F
    groups = (K + 3) // 4 * (2 if l * m == 8000 else 1)
    cpg = torch.cuda.get_device_properties(0).multi_processor_count // groups
    for seed in range(20):                             # the first hash whose lists are even
        coeffs = S.hash_coefficients(seed, l)
        with F.FdaContext(l, m, coeffs, d_max=5 * cpg * 7168, K_max=K) as ctx:
            try:
                T = ctx.fda_debug_lane_schedule(0)[1]["tile_indices"]
                break
            except F.FdaError:
                continue
    d = (full * cpg + more) * T - 1029
    gen = torch.Generator(device="cuda").manual_seed(d)
    w0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = torch.full((K, (d + 3) // 4 * 4 + (0 if aligned else 1)), 1e6, device="cuda")[:, :d]
    w.copy_(w0 + torch.randn((K, d), device="cuda", generator=gen) * 1e-3)
    rows = [0, K // 2, K - 1]
    ora = oracle.local_state(w[rows].cpu().numpy(), w0.cpu().numpy(), None, coeffs, l, m, threads=8)
    with F.FdaContext(l, m, coeffs, d_max=d, K_max=K) as ctx:
        st = torch.full((K, ctx.state_len), float("nan"), device="cuda")
        ctx.fda_local_state(w, w0, None, 5, st)
        assert ctx.fda_debug_last_kernel() == "k_local_state_gather"
        assert ctx.fda_debug_last_schedule() == (2 if full * cpg + more > 4 * cpg else 1)
        assert bool(torch.isfinite(st).all())
        check_states(st[rows].cpu().numpy(), ora, l, m, d)
