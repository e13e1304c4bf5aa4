"""Kernels that start while the one before them is ending (programmatic dependent launches) see what
that one has written: after a broadcast average every drift is zero, so a state formed directly behind
it is zero to the last bit, whichever kernel forms it; one value of the models from before the average would show."""
import numpy as np
import pytest

import fda_synth as S

pytestmark = pytest.mark.gpu


# one tile per block, two tiles, long vectors, sketch rows in parts, no schedule (limit -1); aligned and packed rows
@pytest.mark.parametrize("l,m,K,d,limit", [(5, 250, 5, 61_706, None), (5, 250, 20, 300_000, None), (5, 250, 4, 12_000_003, None),
                                           (7, 500, 13, 2_000_001, None), (8, 1000, 6, 200_001, None), (5, 250, 6, 150_003, -1),
                                           (0, 1, 7, 150_003, None)])
@pytest.mark.parametrize("packed", [False, True])
def test_states_behind_an_average_are_zero(l, m, K, d, limit, packed):
    import torch
    import paper_2405_20988_b200 as F
    gen = torch.Generator(device="cuda").manual_seed(d)
    pitch = d if packed else (d + 31) // 32 * 32
    w_t0 = torch.randn(d, device="cuda", generator=gen) * 0.05
    w = torch.empty((K, pitch), device="cuda")[:, :d]
    xi = torch.randn(d, device="cuda", generator=gen)
    flags = 7 if l else 3
    with F.FdaContext(l, m, S.hash_coefficients(9, l), d_max=d, K_max=K, schedule_limit_bytes=limit) as ctx:
        states = torch.empty((6, K, ctx.state_len), device="cuda")
        means = torch.empty((6, ctx.state_len), device="cuda")
        for t in range(6):
            w.normal_(0.0, 1e-3, generator=gen)
            w += w_t0
            ctx.fda_local_state(w, w_t0, xi, flags, states[t])
            assert float(states[t, :, 0].min()) > 0.0
            ctx.fda_average_models(w, w_t0, None, F.FDA_AVG_BROADCAST)
            ctx.fda_local_state(w, w_t0, xi, flags, states[t])
            w.normal_(0.0, 1e-3, generator=gen)
            w += w_t0
            ctx.fda_average_models_xi(w, w_t0, xi, None, F.FDA_AVG_BROADCAST)
            ctx.fda_mean_state(w, w_t0, xi, flags, means[t])
        assert not states.any() and not means.any()


# lane-private bins (5 x 250) and compare-and-swap bins (7 x 500, 9 x 700); the first call builds the hash table
@pytest.mark.parametrize("l,m", [(5, 250), (7, 500), (9, 700)])
def test_first_averaged_state_of_a_context_equals_the_second(l, m):
    import torch
    import paper_2405_20988_b200 as F
    K, d = 4, 40_003
    gen = torch.Generator(device="cuda").manual_seed(l)
    w_t0 = torch.zeros(d, device="cuda")
    # quarters of whole numbers: every sum is exact, so the order of the additions does not show
    w = torch.randint(-8, 9, (K, d), device="cuda", generator=gen).float()
    for seed in range(8):
        with F.FdaContext(l, m, S.hash_coefficients(seed, l), d_max=d, K_max=K, schedule_limit_bytes=-1) as ctx:
            first, second = (torch.full((ctx.state_len,), float("nan"), device="cuda") for _ in range(2))
            ctx.fda_mean_state(w, w_t0, None, 5, first)
            assert ctx.fda_debug_last_kernel() == "k_mean_model + k_sketch_vector"
            ctx.fda_mean_state(w, w_t0, None, 5, second)
            assert torch.equal(first, second)
