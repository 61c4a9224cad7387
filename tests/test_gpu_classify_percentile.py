"""GPU: the last kernel of a classification (sums, 5th percentile) at the sizes where its layout changes - fewer rows than its
1024 threads, a few more, more than the 24 values per thread that it keeps in registers - against the same in 64 bits."""
import math

import pytest

pytestmark = pytest.mark.gpu

RADIUS = 2


def reference(grid_h, grid_w, blocks, q):
    """(mean, 5th percentile, mean squared error) of the Spatial proxy of one head in 64 bits."""
    import torch
    k, v = (torch.cat([b[i][:, 0] for b in blocks]).double() for i in (0, 1))
    tf, scale = grid_h * grid_w, 1.0 / math.sqrt(q.shape[-1])
    at = torch.arange(k.shape[0], device="cuda") % tf
    ky, kx = at // grid_w, at % grid_w
    cos, sq = [], 0.0
    for rows in torch.arange(q.shape[0], device="cuda").split(1024):
        s = scale * (q[rows, 0].double() @ k.T)
        py, px = (rows % tf) // grid_w, (rows % tf) % grid_w
        near = ((ky - py[:, None]).abs() <= RADIUS) & ((kx - px[:, None]).abs() <= RADIUS)
        ref, proxy = torch.softmax(s, -1) @ v, torch.softmax(s.masked_fill(~near, -math.inf), -1) @ v
        cos.append((ref * proxy).sum(1) / (ref.norm(dim=1) * proxy.norm(dim=1)))
        sq += (ref - proxy).square().sum().item()
    cos = torch.cat(cos).sort().values
    rank = 0.05 * (len(cos) - 1)
    lo, hi = cos[int(rank)].item(), cos[min(int(rank) + 1, len(cos) - 1)].item()
    return cos.mean().item(), lo + (rank - int(rank)) * (hi - lo), sq / q.numel()


@pytest.mark.parametrize("grid_h,grid_w", [(1, 1), (11, 31), (19, 18), (91, 91)])  # 3, 1023, 1026 and 24843 rows
def test_percentile_and_sums(grid_h, grid_w):
    import torch
    from paper_2607_20125_b200.binding import HeadCast
    gen = torch.Generator(device="cuda").manual_seed(grid_h)
    rows = 3 * grid_h * grid_w
    draw = lambda: torch.randn(rows, 1, 64, device="cuda", generator=gen).bfloat16()  # noqa: E731
    blocks, q = [(draw(), draw()) for _ in range(2)], draw()
    hc = HeadCast(1, 64, grid_h, grid_w, 2, proxy_radius=RADIUS)
    for k, v in blocks:
        hc.append(k, v)
    scores = hc.classify(q)[1].flatten().tolist()
    again = hc.classify(q)[1].flatten().tolist()
    hc.destroy()
    mean, p5, mse = reference(grid_h, grid_w, blocks, q)
    assert scores == again
    assert abs(scores[2] - mean) <= 5e-3 and abs(scores[3] - p5) <= 1e-2 and abs(scores[4] - mse) <= 2e-3
