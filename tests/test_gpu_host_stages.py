"""GPU: headcast_attend_host on both sides of the size up to which a block is copied and attended as one."""
import pytest

pytestmark = pytest.mark.gpu

LABELS = [0, 1, 2, 3, 2, 3, 1, 0, 2, 3, 3, 2]


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("grid_h,grid_w,one", [(13, 35, True), (19, 24, False)])  # 1365 and 1368 rows of 3072 bytes; 4 MiB are 1365.3
def test_host_buffers_on_both_sides_of_the_one_stage_limit(grid_h, grid_w, one, pinned):
    import torch
    from paper_2607_20125_b200.binding import HeadCast
    gen = torch.Generator(device="cuda").manual_seed(grid_w)
    hc = HeadCast(12, 128, grid_h, grid_w, 3)
    draw = lambda: torch.randn(3 * grid_h * grid_w, 12, 128, device="cuda", generator=gen).bfloat16()  # noqa: E731
    host = lambda t: t.cpu().pin_memory() if pinned else t.cpu()  # noqa: E731
    for _ in range(2):
        hc.append(draw(), draw())
    hc.set_labels(LABELS)
    hc.split_cache()
    hc.append_host(host(draw()), host(draw()))
    queries = [draw() for _ in range(3)]
    want = [torch.empty_like(q) for q in queries]
    for q, out in zip(queries, want):
        hc.attend(q, out)
    torch.cuda.synchronize()
    inputs, outs = [host(q) for q in queries], [host(torch.full_like(q, float("nan"))) for q in queries]
    launches = hc.launch_count()
    for q, out in zip(inputs, outs):
        hc.attend_host(q, out)
    torch.cuda.current_stream().synchronize()
    assert (hc.launch_count() - launches <= 3 * 2) == one  # an attention and a merge launch per call
    for out, ref in zip(outs, want):
        if one:
            assert torch.equal(out, ref.cpu())
        err = (out.float() - ref.cpu().float()).abs()  # cut elsewhere: the sums differ in order, the outputs by a bf16 step
        assert err.max().item() <= 2e-2 and err.mean().item() <= 2e-3
    hc.check()
    hc.destroy()
