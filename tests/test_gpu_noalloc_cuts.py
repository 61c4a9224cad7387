"""GPU: key ranges of the allocation-free call that are cut and merged - equal pieces of few query-tile pairs (up to more parts
than the short merge takes at a time), equal shares of a line of many - at the edges of the cuts."""
import pytest

from test_gpu_attention_edges import MAX_ABS, MEAN_ABS, reference

pytestmark = pytest.mark.gpu

# heads, queries, key tiles, pieces of every pair (-1: shares of a line); test_noalloc_plan.py holds the last to the rule
CASES = [
    (1, 1, 9, 9), (3, 129, 11, 11),        # one pair, or one per head; a lone query tile, one row of a second one
    (1, 256, 17, 17), (1, 130, 60, 20), (2, 5, 148, 37),  # more than sixteen pieces of a pair
    (9, 2048, 10, 2), (37, 512, 12, 2),    # 72 and 74 pairs: two pieces each, 148 CTAs in use
    (12, 1024, 12, 3), (9, 1024, 16, 4), (9, 512, 24, 8),
    (15, 1280, 19, -1), (10, 2560, 36, -1),  # 75 and 100 pairs: a pair in two or three shares
    (25, 1500, 35, -1),                    # 150 pairs: two whole waves but for a few
]
# Largest relative error (2-norm) of one row of one head: bf16 rounds outputs and probabilities by 2^-9 at most, which is 0.4 %
# together; a lost piece changes some row of its pair by 17 % or more (computed without the piece, all cases).
ROW_ERROR = 1e-2


def planted(heads, n_q, n_k, head_dim, device, gen):
    """q, k, v in which, for every head, query-tile pair and key tile, one key of the tile draws one row of the pair 16 nats above
    the average: every piece of every pair decides a row, also where it is the single key of the last tile."""
    import torch
    q, k, v = (torch.randn(n, heads, head_dim, device=device, generator=gen).bfloat16().float() for n in (n_q, n_k, n_k))
    drawn = torch.zeros_like(k)
    for pair in range(-(-n_q // 256)):
        rows = min(256, n_q - 256 * pair)
        for tile in range(-(-n_k // 128)):
            row = q[256 * pair + tile % rows]
            drawn[128 * tile + pair % min(128, n_k - 128 * tile)] += 16.0 * head_dim ** 0.5 * row / row.square().sum(-1, keepdim=True)
    k = torch.where(drawn.abs().sum(-1, keepdim=True) > 0, drawn, k)
    return q.bfloat16(), k.bfloat16(), v.bfloat16()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("heads,n_q,tiles,pieces", CASES)
@pytest.mark.parametrize("ragged", [0, 1])
def test_cut_key_ranges(head_dim, heads, n_q, tiles, pieces, ragged):
    import torch
    from paper_2607_20125_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(heads * 1000 + tiles)
    q, k, v = planted(heads, n_q, 128 * tiles - 127 * ragged, head_dim, "cuda", gen)
    out = torch.full_like(q, float("nan"))
    binding.dense_attend_noalloc(q, k, v, out)
    binding.noalloc_status()
    want = reference(q, k, v)
    assert ((out.float() - want).norm(dim=-1) <= ROW_ERROR * want.norm(dim=-1)).all()


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
