"""The tensor-core pass down strips (k_march) at the edges of its split: strips of 32 columns, bands
of 4 rows, search ranges at and around the chunk sizes 32, 64, 96 and 128 and over several chunks,
every block and window radius, and both sides of the size limit between its refinement and the
tiles'.  FP32 storage equals the SIMT form bit for bit; 16-bit storage is held to the oracle by the
tensor-form tests' derived gap (2e-2 FP16, 1e-1 BF16), and its validity mask is exact."""
import numpy as np
import pytest
import torch

import oracle
import paper_1904_06017_gb300 as sg
from gpu_helpers import dev_f32, dev_img, pitch_of
from test_gpu_screened import assert_same, pair, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1904_06017_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("W,H,D,win,bil", [
    (1, 1, 1, 3, 1), (33, 5, 33, 3, 1), (31, 3, 34, 5, 3), (64, 8, 64, 7, 5), (65, 9, 65, 9, 7), (96, 12, 96, 11, 9),
    (40, 70, 97, 9, 11), (34, 37, 128, 11, 11), (50, 20, 129, 5, 13), (64, 33, 192, 9, 13), (45, 21, 193, 7, 11),
    (70, 18, 256, 11, 13), (60, 40, 170, 3, 9), (32, 4, 31, 9, 13), (95, 23, 32, 11, 13), (63, 90, 16, 9, 11),
    (303, 270, 32, 9, 11), (304, 270, 32, 9, 11)])
def test_fp32_equals_simt_at_the_edges(W, H, D, win, bil):
    if W == 1:
        ref, tgt = np.full((1, 1), 7, np.uint8), np.full((1, 1), 9, np.uint8)
    else:
        ref, tgt, _ = pair(W, H, min(5, W - 1), W * 131 + H + D)
    shift = (np.arange(H) % 5 - 2).astype(np.float32)
    assert_same(run(ref, tgt, shift, D, win, bil, 3.0, 10.0, sg.STEREO_FUSED_SIMT),
                run(ref, tgt, shift, D, win, bil, 3.0, 10.0, sg.STEREO_FUSED_TENSOR))


@pytest.mark.parametrize("sigma1", [2.0, 10.0])
@pytest.mark.parametrize("W,H,D,bil", [(140, 60, 30, 9), (150, 50, 32, 13), (90, 44, 60, 11)])
def test_fp32_equals_simt_where_candidates_tie(W, H, D, bil, sigma1):
    """Low contrast, repeated texture and flat rows: pixels with two candidates far apart, with many,
    and ranges clipped at the flat run, in one image."""
    rng = np.random.default_rng(W + D)
    tile = rng.integers(100, 104, (H, 12), dtype=np.uint8)
    ref = np.tile(tile, (1, W // 12 + 1))[:, :W].copy()
    tgt = np.roll(ref, -4, axis=1)
    ref[: H // 3, W // 2:] = rng.integers(0, 256, (H // 3, W - W // 2), dtype=np.uint8)
    tgt[: H // 3, : W - 4] = ref[: H // 3, 4:]
    for v in range(H):
        tgt[v, : (v * 7) % (W - 8)] = tgt[v, 0]
    shift = np.zeros(H, np.float32)
    assert_same(run(ref, tgt, shift, D, 7, bil, 3.0, sigma1, sg.STEREO_FUSED_SIMT),
                run(ref, tgt, shift, D, 7, bil, 3.0, sigma1, sg.STEREO_FUSED_TENSOR))


@pytest.mark.parametrize("dtype,gap", [(sg.STEREO_F16, 2e-2), (sg.STEREO_BF16, 1e-1)])
@pytest.mark.parametrize("W,H,D,win,bil", [(33, 9, 20, 3, 5), (70, 30, 33, 9, 11), (64, 21, 96, 5, 7), (90, 22, 129, 9, 11),
                                           (80, 25, 200, 7, 13), (97, 17, 256, 11, 9)])
def test_16_bit_forms_over_chunks(dtype, gap, W, H, D, win, bil):
    ref, tgt, shift = pair(W, H, 5, W * 17 + D)
    p = pitch_of(W)
    disp, b2 = torch.empty((H, W), device="cuda"), torch.empty((H, W, 2), device="cuda")
    wta, wta2 = (torch.empty((H, W), dtype=torch.int32, device="cuda") for _ in range(2))
    valid = torch.empty((H, W), dtype=torch.uint8, device="cuda")
    disp2 = torch.empty_like(disp)
    with sg.Stereo(W, H, D, win=win, bil=bil, sigma0=3.0, sigma1=10.0, pitch=p, cost_dtype=dtype) as st:
        a = (dev_img(ref, p), dev_img(tgt, p), dev_f32(shift))
        st.cost_aggregate_wta(*a, disp, wta, valid)
        st.cost_aggregate_wta(*a, disp2, wta2, valid, best2=b2)
    assert torch.equal(disp, disp2) and torch.equal(wta, wta2)
    d_o, ds_o, eb, es = oracle.stereo(ref, tgt, shift, D, win, bil, 3.0, 10.0)
    sure = es - eb > gap
    assert sure.mean() > 0.3
    assert np.array_equal(wta.cpu().numpy()[sure], ds_o[sure])
    b = b2.cpu().numpy()
    assert np.abs(b[..., 0] - eb).max() <= gap / 2 and np.abs(b[..., 1] - es)[sure].max() <= gap / 2
    assert np.array_equal(valid.cpu().numpy(), oracle.valid_mask(W, H, D, win, bil, shift))


@pytest.mark.parametrize("W,H,D,bil", [(70, 21, 160, 11), (70, 21, 161, 11), (40, 30, 224, 7), (65, 17, 225, 9),
                                       (50, 26, 160, 13), (50, 26, 161, 13), (97, 13, 224, 13), (97, 13, 225, 13)])
def test_fp32_range_in_two_passes_equals_simt(W, H, D, bil):
    """On both sides of the ranges whose last chunk is a pass of its own."""
    ref, tgt, _ = pair(W, H, 5, W * 7 + H + D)
    shift = (np.arange(H) % 5 - 2).astype(np.float32)
    assert_same(run(ref, tgt, shift, D, 7, bil, 3.0, 10.0, sg.STEREO_FUSED_SIMT),
                run(ref, tgt, shift, D, 7, bil, 3.0, 10.0, sg.STEREO_FUSED_TENSOR))


@pytest.mark.parametrize("W,H,D,win,bil", [(40, 11, 40, 9, 11), (33, 12, 40, 9, 11), (64, 13, 64, 5, 9), (70, 24, 36, 11, 7),
                                           (33, 25, 50, 9, 13), (96, 37, 40, 3, 5), (300, 120, 140, 9, 11),
                                           (960, 540, 40, 9, 11), (960, 541, 40, 9, 11)])
def test_refinement_tile_heights_equal_simt(W, H, D, win, bil):
    """Frames around the low refinement tiles' 12 rows, and on both sides of the size where the tiles
    have 36 rows (960 x 541 has 480 of them)."""
    ref, tgt, _ = pair(W, H, 5, W * 3 + H + D)
    shift = (np.arange(H) % 5 - 2).astype(np.float32)
    assert_same(run(ref, tgt, shift, D, win, bil, 3.0, 10.0, sg.STEREO_FUSED_SIMT),
                run(ref, tgt, shift, D, win, bil, 3.0, 10.0, sg.STEREO_FUSED_TENSOR))


@pytest.mark.parametrize("form", ["f32", "simt", "f16", "tiles", "small", "batch"])
def test_context_runs_after_others_of_smaller_windows_and_ranges(form):
    """A context whose kernels need much shared memory, then contexts that need less of the same kernels
    (other windows and ranges, a warp estimator, a batch): the first one runs as before."""
    W, H, D = (400, 300, 30) if form == "tiles" else (200, 80, 30) if form == "small" else (200, 80, 128)
    ref, tgt, shift = pair(W, H, 5, 3)
    pitch = pitch_of(W)
    args = dict(ref=dev_img(ref, pitch), tgt=dev_img(tgt, pitch), shift=dev_f32(shift))
    disp, wta = torch.empty((H, W), device="cuda"), torch.empty((H, W), dtype=torch.int32, device="cuda")
    valid = torch.empty((H, W), dtype=torch.uint8, device="cuda")

    def batch(D, win):
        q = dict(args, max_disp=D, disp=torch.empty((H, W), device="cuda"), disp_out=disp, valid=valid,
                 tgt_warped=torch.zeros((H, pitch), dtype=torch.uint8, device="cuda"),
                 res=torch.zeros(64, dtype=torch.uint8, device="cuda"))
        return sg.StereoBatch([q], win=win, bil=11, sigma0=3.0, sigma1=10.0, tile_wc=32, tile_dc=32), q

    def frame(win, D, **kw):
        return sg.Stereo(W, H, D, win=win, bil=11, sigma0=3.0, sigma1=10.0, pitch=pitch, **kw)

    kw = dict(simt=dict(fused_form=sg.STEREO_FUSED_SIMT), f16=dict(cost_dtype=sg.STEREO_F16)).get(form, {})
    if form == "batch":
        b, q = batch(D, 11)

        def run_it():
            q["disp"].fill_(-1)
            b.run()
            torch.cuda.synchronize()
            return q["disp"].clone()
    else:
        st = frame(11, D, **kw)

        def run_it():
            disp.fill_(-1)
            st.cost_aggregate_wta(args["ref"], args["tgt"], args["shift"], disp, wta, valid)
            torch.cuda.synchronize()
            return disp.clone()
    before = run_it()
    others = [frame(3, d, **k) for d in (100, 40, 5) for k in (kw, {})]
    others += [sg.WarpEstimator(W, H, 64, factor=2, win=3, bil=11, pitch=pitch), batch(100, 3)[0], batch(5, 3)[0]]
    assert torch.equal(run_it(), before)
    del others
