"""The model average on both sides of every line between one index per thread and quads: rows at any alignment and
aligned ones, with and without broadcast.  The sum of an index is one of fp32 additions in the order of the workers on either
side, so the result is the same bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [4, 6, 7, 8, 9, 10, 18, 33])
@pytest.mark.parametrize("per_sm", [768, 1300, 1536, 1800, 2200, 2600, 3400, 4096, 4800, 6400])
@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("offset", [None, 0, 1])
def test_both_sides_of_the_lines(K, per_sm, more, offset):
    import torch
    import fda_synth as S
    import paper_2405_20988_b200 as F
    d = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + more
    pitch = (d + 3) // 4 * 4 + (0 if offset is None else 1 + d % 2)
    gen = torch.Generator(device="cuda").manual_seed(K + d)
    base = torch.randn(K * pitch + 4, device="cuda", generator=gen)
    first = offset or 0
    w = base[first:first + K * pitch].view(K, pitch)[:, :d]
    want = w[0].clone()
    for k in range(1, K):
        want += w[k]
    want *= torch.tensor(1.0, device="cuda") / torch.tensor(float(K), device="cuda")
    before = base.clone()
    with F.FdaContext(1, 8, S.hash_coefficients(1, 1), d_max=d, K_max=K) as ctx:
        for flags in (0, F.FDA_AVG_BROADCAST):
            guard = torch.full((d + 8,), 7.0, device="cuda")
            w0 = guard[4:4 + d]
            ctx.fda_average_models(w, w0, None, F.FDA_AVG_UNCONDITIONAL | flags)
            assert torch.equal(w0, want) and bool((guard[:4] == 7).all()) and bool((guard[4 + d:] == 7).all())
            if flags == 0:
                assert torch.equal(base, before)
        assert torch.equal(w, want.expand(K, d))
        w.copy_(before[first:first + K * pitch].view(K, pitch)[:, :d])
        assert torch.equal(base, before)          # nothing between the rows was touched
