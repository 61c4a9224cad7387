"""GPU: the attention kernel at the edges of its tiles - 128-row query tiles in pairs, 128-key tiles in four chunks of 32,
P handed over in two parts, O rescaled when a row's maximum grows - against float32 attention of the same bf16 values."""
import pytest

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3  # the repository's bars: bf16 probabilities and outputs of order one


def reference(q, k, v):
    import torch
    s = torch.einsum("qhd,khd->hqk", q.float(), k.float()) / q.shape[-1] ** 0.5
    return torch.einsum("hqk,khd->qhd", torch.softmax(s, -1), v.float())


def check(q, k, v):
    import torch
    from paper_2607_20125_b200 import binding
    out = torch.full_like(q, float("nan"))
    binding.dense_attend_noalloc(q, k, v, out)
    binding.noalloc_status()
    err = (out.float() - reference(q, k, v)).abs()
    assert err.max().item() <= MAX_ABS and err.mean().item() <= MEAN_ABS, (q.shape, k.shape, err.max().item(), err.mean().item())


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("n_keys", [1, 31, 32, 33, 64, 65, 96, 97, 127, 128, 129, 255, 257, 640])
def test_ragged_queries_and_keys(head_dim, n_keys):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(n_keys * 1000 + head_dim)
    for n_q in (1, 32, 33, 127, 128, 129, 255, 256, 257, 385):
        q, k, v = (torch.randn(n, 3, head_dim, device="cuda", generator=gen).bfloat16() for n in (n_q, n_keys, n_keys))
        check(q, k, v)


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("n_q", [100, 256])
def test_row_maximum_grows_and_falls_from_tile_to_tile(head_dim, n_q):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(7)
    u = torch.nn.functional.normalize(torch.randn(1, 2, head_dim, device="cuda", generator=gen), dim=-1)
    q, k, v = (torch.randn(n, 2, head_dim, device="cuda", generator=gen) for n in (n_q, 128 * 6 + 5, 128 * 6 + 5))
    tile = torch.arange(k.shape[0], device="cuda") // 128
    steps = torch.tensor([0.0, 1.0, 0.3, 2.0, 2.9, 2.9, 2.5], device="cuda")[tile]
    # a third of the rows climbs by about 13 nats a step, a third falls behind, the rest sees noise
    sign = torch.tensor([1.0, -1.0, 0.0], device="cuda")[torch.arange(n_q, device="cuda") % 3]
    q = q + 12.0 * head_dim ** 0.25 * sign[:, None, None] * u
    k = k + 1.1 * head_dim ** 0.25 * steps[:, None, None] * u
    check(q.bfloat16(), k.bfloat16(), v.bfloat16())


@pytest.mark.parametrize("heads,n_q", [(1, 1), (3, 256 * 49), (4, 256 * 37), (4, 256 * 37 + 1), (5, 256 * 59 + 130), (64, 256 * 32)])
def test_work_list_of_the_allocation_free_call(heads, n_q):
    """1, 147, 148, 152, 300 and 2048 (the limit) work items: fewer than, as many as and more than one per SM."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(heads)
    q, k, v = (torch.randn(n, heads, 64, device="cuda", generator=gen).bfloat16() for n in (n_q, 70, 70))
    check(q, k, v)


def test_allocation_free_calls_of_different_sizes_back_to_back():
    """Every call rewrites the list that the call before it still works on: nothing waits in between on the host."""
    import torch
    from paper_2607_20125_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(3)
    cases = []
    for heads, n_q, n_k in ((16, 1373, 5492), (1, 5, 3), (12, 3000, 900), (2, 129, 64)) * 3:
        q, k, v = (torch.randn(n, heads, 64, device="cuda", generator=gen).bfloat16() for n in (n_q, n_k, n_k))
        cases.append((q, k, v, torch.empty_like(q)))
    torch.cuda.synchronize()
    for q, k, v, out in cases:
        binding.dense_attend_noalloc(q, k, v, out)
    binding.noalloc_status()
    for q, k, v, out in cases:
        err = (out.float() - reference(q, k, v)).abs()
        assert err.max().item() <= MAX_ABS and err.mean().item() <= MEAN_ABS
