"""GPU: NaN queries and keys reach the output as NaN and touch no other row or head, whether a key range is one work item or is
cut into pieces that are merged."""
import pytest

pytestmark = pytest.mark.gpu


def check(attend, q, k, v, heads_of_nan_keys=()):
    """`attend(q, k, v, out)` with two NaN query rows and, per head listed, 600 NaN keys in a row."""
    import torch
    rows, heads = q.shape[:2]
    want = torch.zeros(rows, heads, dtype=torch.bool, device="cuda")
    for row, head in ((0, 0), (rows - 1, heads - 1)):
        q[row, head] = float("nan")
        want[row, head] = True
    for head in heads_of_nan_keys:
        k[:600, head] = float("nan")
        want[:, head] = True
    out = torch.zeros_like(q)
    attend(q, k, v, out)
    got = out.isnan()
    assert torch.equal(got, want[:, :, None].expand_as(got))


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("heads,n_q,n_k", [(5, 300, 700), (8, 687, 2748), (2, 40, 5000), (15, 1280, 2432)])  # whole, pieces, > 16 pieces, a line
def test_allocation_free_call(head_dim, heads, n_q, n_k):
    import torch
    from paper_2607_20125_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(n_k)
    q, k, v = (torch.randn(n, heads, head_dim, device="cuda", generator=gen).bfloat16() for n in (n_q, n_k, n_k))
    check(binding.dense_attend_noalloc, q, k, v, heads_of_nan_keys=[1])


@pytest.mark.parametrize("grid_h,grid_w,heads,head_dim", [(8, 8, 4, 64), (13, 22, 6, 128), (30, 52, 8, 128)])
def test_context(grid_h, grid_w, heads, head_dim):
    import torch
    from paper_2607_20125_b200.binding import HeadCast
    gen = torch.Generator(device="cuda").manual_seed(grid_h)
    draw = lambda: torch.randn(3 * grid_h * grid_w, heads, head_dim, device="cuda", generator=gen).bfloat16()  # noqa: E731
    hc = HeadCast(heads, head_dim, grid_h, grid_w, 3, keep_monolithic=True)
    for _ in range(3):
        hc.append(draw(), draw())
    hc.set_labels([(3 + i) % 4 for i in range(heads)])
    hc.split_cache()
    check(lambda q, k, v, out: hc.full_attend(q, out), draw(), draw(), None)
    check(lambda q, k, v, out: hc.attend(q, out), draw(), draw(), None)
    hc.check()
    hc.destroy()
