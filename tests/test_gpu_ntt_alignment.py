"""fg_ntt on a buffer that starts 8 but not 16 bytes into an allocation, at
every ring degree, with one limb and with enough limbs for either pass form:
the words of the aligned call, and nothing written beside the buffer."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", range(10, 17))
@pytest.mark.parametrize("rows", [1, 60])
def test_odd_word_offset_gives_the_aligned_words(log_n, rows):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    ctx = fg.Context(log_n=log_n, q_bits=[60, 45], p_bits=[60], alpha=1, log_scale=40)
    g = torch.Generator(device="cuda")
    g.manual_seed(log_n)
    x = torch.stack([torch.randint(0, q, (rows, ctx.n), generator=g, device="cuda") for q in ctx.q], 1)
    x = x.reshape(-1, ctx.n).contiguous()
    room = torch.full((x.numel() + 2,), -7, dtype=torch.int64, device="cuda")
    odd = room[1:-1].view(x.shape)
    assert odd.data_ptr() % 16 == 8
    for inverse in (False, True):
        odd.copy_(x)
        want = fg.ntt(ctx, x.clone(), [0, 1], inverse=inverse)
        fg.ntt(ctx, odd, [0, 1], inverse=inverse)
        assert torch.equal(odd, want)
        assert room[0] == -7 and room[-1] == -7
    ctx.close()
