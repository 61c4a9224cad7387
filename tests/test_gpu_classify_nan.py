"""GPU: a NaN among the values of a head makes every score of that head that looks at outputs NaN, and touches no other head."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid_h,grid_w", [(4, 5), (11, 31), (20, 26)])
def test_nan_values_reach_the_percentile(grid_h, grid_w):
    import torch
    from paper_2607_20125_b200.binding import HeadCast
    gen = torch.Generator(device="cuda").manual_seed(grid_w)
    draw = lambda: torch.randn(3 * grid_h * grid_w, 3, 64, device="cuda", generator=gen).bfloat16()  # noqa: E731
    keys, values, q = [draw(), draw()], [draw(), draw()], draw()

    def scores():
        hc = HeadCast(3, 64, grid_h, grid_w, 2)
        for k, v in zip(keys, values):
            hc.append(k, v)
        labels, result = hc.classify(q)
        hc.destroy()
        return labels, torch.from_numpy(result)

    labels, before = scores()
    values[0][7, 1] = float("nan")
    labels_nan, after = scores()
    assert before.isfinite().all() and after[[0, 2]].equal(before[[0, 2]])
    assert after[1, [0, 2, 3, 4, 5]].isnan().all() and after[1, 6:].equal(before[1, 6:])  # cosines, percentile, error, score; the masses
    assert labels_nan[1] == 3 and (labels_nan == labels)[[0, 2]].all()
