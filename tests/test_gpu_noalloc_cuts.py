"""GPU: key ranges of the allocation-free call that are cut and merged - equal pieces of few query-tile pairs (up to more parts
than the short merge takes at a time), equal shares of a line of many - at the edges of the cuts."""
import pytest

from test_gpu_attention_edges import MAX_ABS, MEAN_ABS, check, reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("heads,n_q,tiles", [
    (1, 1, 9), (3, 129, 11),               # one pair, or one per head; a lone query tile, one row of a second one
    (1, 256, 17), (1, 130, 60), (2, 5, 148),  # more than sixteen pieces of a pair
    (9, 2048, 3), (37, 512, 5),            # 72 and 74 pairs: two pieces each
    (15, 1280, 19), (10, 2560, 27),        # 75 and 100 pairs: shares of a line, a pair in two or three of them
    (25, 1500, 35),                        # 150 pairs: two whole waves but for a few
])
@pytest.mark.parametrize("ragged", [0, 1])
def test_cut_key_ranges(head_dim, heads, n_q, tiles, ragged):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(heads * 1000 + tiles)
    n_k = 128 * tiles - 127 * ragged
    check(*(torch.randn(n, heads, head_dim, device="cuda", generator=gen).bfloat16() for n in (n_q, n_k, n_k)))


def test_calls_of_every_route_back_to_back():
    """Each call overwrites the list, the partial results and the merge entries that the one before still works on."""
    import torch
    from paper_2607_20125_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(5)
    cases = []
    for heads, n_q, n_k in ((10, 2560, 3456), (2, 5, 2560), (4, 129, 64), (1, 256, 1100), (25, 1500, 4400), (64, 300, 200)) * 2:
        q, k, v = (torch.randn(n, heads, 64, device="cuda", generator=gen).bfloat16() for n in (n_q, n_k, n_k))
        cases.append((q, k, v, torch.empty_like(q), torch.empty_like(q)))
    for again in (3, 4):
        torch.cuda.synchronize()
        for c in cases:
            binding.dense_attend_noalloc(*c[:3], c[again])
        binding.noalloc_status()
    for q, k, v, out, out2 in cases:
        err = (out.float() - reference(q, k, v)).abs()
        assert err.max().item() <= MAX_ABS and err.mean().item() <= MEAN_ABS
        assert torch.equal(out, out2)
