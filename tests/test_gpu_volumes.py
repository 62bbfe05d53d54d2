"""The FP32 volumes in device memory (stereo_cost_volume / _aggregate_volume / _wta_volume) at
the edges of their tiling: columns off 32, rows off 16, disparities off 4, 16 and 32, every
window radius, volumes that start off a 16-byte boundary; and the scan's treatment of ties,
infinities and NaNs.  Costs and aggregated costs are held to the parity tests' 1e-4 (floor 1e-2);
the WTA of a given volume is exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_1904_06017_gb300 as sg
import synth
from gpu_helpers import check_rel, dev_f32, dev_img, pitch_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1904_06017_gb300 import build
    build.build()
    oracle.build()


def _empty(shape, offset):
    """A float32 CUDA tensor that starts `offset` floats past a 16-byte boundary."""
    n = int(np.prod(shape))
    return torch.empty(n + 4, dtype=torch.float32, device="cuda")[offset:offset + n].view(shape)


@pytest.mark.parametrize("W,H,D,win,bil,offset", [(1, 1, 1, 3, 1, 0), (33, 17, 5, 3, 3, 0), (31, 15, 32, 5, 5, 0),
                                                  (65, 33, 36, 7, 7, 1), (40, 48, 34, 9, 11, 0), (64, 16, 64, 11, 13, 0),
                                                  (50, 30, 40, 11, 15, 3), (97, 20, 31, 9, 9, 2)])
def test_volumes_at_tile_edges(W, H, D, win, bil, offset):
    rng = np.random.default_rng(W * 1000 + H * 10 + D)
    ref, tgt = synth.texture(rng, H, W), synth.texture(rng, H, W)
    c_o = oracle.cost_volume(ref, tgt, D, win)
    e_o = oracle.aggregate(ref, c_o, bil, 3.0, 10.0)
    cost, agg = _empty((H, W, D), offset), _empty((H, W, D), offset)
    r = dev_img(ref, pitch_of(W))
    with sg.Stereo(W, H, D, win=win, bil=bil, sigma0=3.0, sigma1=10.0, pitch=pitch_of(W)) as st:
        st.cost_volume(r, dev_img(tgt, pitch_of(W)), cost)
        st.aggregate_volume(r, cost, agg)
    check_rel(cost.cpu().numpy(), c_o)
    check_rel(agg.cpu().numpy(), e_o)


@pytest.mark.parametrize("D", [1, 2, 7, 8, 9, 33])
def test_wta_volume_scan(D):
    H, W = 5, 37
    rng = np.random.default_rng(D)
    e = rng.integers(0, 4, (H, W, D)).astype(np.float32)          # many ties
    e[rng.random((H, W, D)) < 0.2] = np.inf
    e[rng.random((H, W, D)) < 0.1] = np.nan
    e[0, :4] = np.inf
    e[0, 4:8] = np.nan
    e[1, :3, 0] = np.nan
    e[1, 3:6] = -np.inf
    best, second = np.zeros((H, W), np.int64), np.full((H, W), np.inf, np.float32)
    for v in range(H):
        for u in range(W):
            x, b = e[v, u], 0
            for d in range(1, D):
                if x[d] < x[b]:
                    b = d
            best[v, u] = b
            for d in range(D):
                if d != b and x[d] < second[v, u]:
                    second[v, u] = x[d]
    shift = rng.uniform(-6, 6, H).astype(np.float32)
    disp = torch.empty((H, W), device="cuda")
    wta = torch.empty((H, W), dtype=torch.int32, device="cuda")
    best2 = torch.empty((H, W, 2), device="cuda")
    with sg.Stereo(W, H, D, win=3, bil=3, pitch=pitch_of(W)) as st:
        st.wta_volume(dev_f32(e), dev_f32(shift), disp, wta, best2)
    assert np.array_equal(wta.cpu().numpy(), best)
    b2 = best2.cpu().numpy()
    assert np.array_equal(b2[..., 0], np.take_along_axis(e, best[..., None], 2)[..., 0], equal_nan=True)
    assert np.array_equal(b2[..., 1], second)


@pytest.mark.parametrize("sigma1", [1e16, 1e17, 1e18, 1e19, 1e25, 3e38])
def test_aggregation_without_a_range_term(sigma1):
    """A sigma1 so large that intensities don't matter: at the borders too, only the neighbours inside
    the image count."""
    W, H, D, bil = 37, 21, 9, 11
    rng = np.random.default_rng(5)
    ref = synth.texture(rng, H, W)
    cost = rng.uniform(0, 2, (H, W, D)).astype(np.float32)
    agg = torch.empty((H, W, D), device="cuda")
    with sg.Stereo(W, H, D, win=3, bil=bil, sigma0=3.0, sigma1=sigma1, pitch=pitch_of(W)) as st:
        st.aggregate_volume(dev_img(ref, pitch_of(W)), dev_f32(cost), agg)
    check_rel(agg.cpu().numpy(), oracle.aggregate(ref, cost, bil, 3.0, sigma1))
