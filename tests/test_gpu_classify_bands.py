"""GPU: the classification on grids where the Spatial proxy's query pairs are dealt per frame (more than 256 tokens a
frame: a last pair of few rows, bands clipped at the frame's ends, radii from nothing to the whole frame) and on the
largest grid where they are not, against the float64 oracle."""
import numpy as np
import pytest

from oracle import headcast_oracle as orc
from paper_2607_20125_b200 import synth
from test_gpu_parity import Pair, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gh,gw,radius", [(16, 16, 2), (17, 16, 2), (19, 27, 1), (19, 27, 0), (27, 19, 7), (1, 300, 2), (300, 1, 3), (16, 17, 400)])
def test_classification_of_frames_dealt_into_pairs(gh, gw, radius):
    w = synth.Workload("bands", 4, 64, gh, gw, 3, labels=(0, 1, 2, 3))
    p = Pair(w, keep_monolithic=True, proxy_radius=radius)
    p.append(2)
    q = synth.make_q(w, 1, 0)
    labels, scores = p.hc.classify(to_dev(q))
    want_labels, want = orc.classify(q, p.cache, p.geom, r=radius)
    for i, name in enumerate(orc.SCORE_NAMES):
        # fp32 statistics of bf16 probabilities against float64: cosines and masses 5e-3, mse 2e-3, and the score, which
        # takes gamma = 5 times the mse, 1e-2 + 5 * 2e-3
        tol = {"mse_spatial": 2e-3, "p5_spatial": 1e-2, "score": 2e-2}.get(name, 5e-3)
        assert np.abs(scores[:, i] - want[:, i]).max() <= tol, (name, scores[:, i], want[:, i])
    assert list(labels) == list(want_labels)


@pytest.mark.parametrize("gh,gw", [(16, 17), (8, 9)])
def test_any_radius_beyond_the_frame_means_the_whole_frame(gh, gw):
    w = synth.Workload("whole", 4, 64, gh, gw, 3, labels=(0, 1, 2, 3))
    results = []
    for radius in (max(gh, gw), 10**6, 2**31 - 1):
        p = Pair(w, keep_monolithic=True, proxy_radius=radius)
        p.append(2)
        results.append(p.hc.classify(to_dev(synth.make_q(w, 1, 0))))
    for labels, scores in results[1:]:
        assert np.array_equal(labels, results[0][0]) and np.array_equal(scores, results[0][1])
