"""Order 0 with one window scale (lpa_mean): every pixel against the oracle, and the same bits from
every entry point.

Covered where its tiles and windows can go wrong: outputs around the 64-pixel tile width and the 8
P rows of a tile, axis-parallel and rotated rigs, 1x, enlarged, reduced and mirrored outputs, both
candidate-cell sizes and the windows between them, odd sensors with calibration frames, outputs past the
sensors, one and eight sensors, and the larger tiles of big frames on sampled pixels. Tolerance: the parity
rule of tests/parity.py, unchanged.
"""
import dataclasses
import math

import numpy as np
import pytest

import oracle
from paper_1308_4908_gb300 import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1308_4908_gb300 import hdr
    c = hdr.Context(0)
    yield c
    c.close()


def _frame(w, h, rot, n=2, sigma=0.7, seed=1500, calibrated=False, **over):
    p = synth.Params(order=0, sigmas=(sigma,), out_w=w, out_h=h)
    fr = synth._build_frame(seed + n, n, w, h, [2.0 ** (-2 * k) for k in range(n)], 1.3, rot, 0.0, p, "mean")
    if calibrated:
        r = np.random.default_rng(seed)
        s = fr.sensors[0]
        s.bias_frame = (s.black + r.uniform(-2, 2, (h, w))).astype(np.float32)
        s.prnu_frame = r.uniform(0.95, 1.05, (h, w)).astype(np.float32)
        s.read_var_frame = r.uniform(6, 12, (h, w)).astype(np.float32)
        s.sat_frame = r.integers(200, 4096, (h, w)).astype(np.uint16)
    return dataclasses.replace(fr, params=dataclasses.replace(p, **over))


def _run(ctx, fr, rig=0):
    p = fr.params
    ctx.set_rig(rig, fr.sensors)
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]
    ch = torch.full((3, p.out_h, p.out_w), 77, dtype=torch.uint8, device="cuda")
    dt = torch.float16 if p.out_dtype else torch.float32
    out = torch.full((3, p.out_h, p.out_w), -7.0, dtype=dt, device="cuda")
    ctx.reconstruct(rig, p, raws, out=out, choice=ch)
    ctx.check()
    return out.float().cpu().numpy(), ch.cpu().numpy(), raws


def _against_oracle(fr, out, ch, pix, extra=0.0):
    p = fr.params
    o = oracle.reconstruct(fr.sensors, p, pix, levels=True)
    parity.compare(out[:, pix[:, 1], pix[:, 0]], ch[:, pix[:, 1], pix[:, 0]], o, pix, 1, 0, p.ici_gamma, p.min_pivot,
                   extra_rel=extra)


def _every_pixel(p):
    vv, uu = np.mgrid[0:p.out_h, 0:p.out_w]
    return np.stack([uu.ravel(), vv.ravel()], axis=1)


@pytest.mark.parametrize("rot", [0.0, 0.3, 7.0])
@pytest.mark.parametrize("w,h", [(1, 1), (63, 7), (64, 8), (65, 9), (131, 34)])
def test_tile_edges(ctx, w, h, rot):
    fr = _frame(w, h, rot)
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


@pytest.mark.parametrize("rot", [0.0, 0.4])
@pytest.mark.parametrize("sigma,green", [(0.3, 1.0), (0.66, 0.5), (0.7, 0.70710678), (0.99, 0.7), (1.2, 0.8), (1.3, 0.6)])
def test_window_sizes(ctx, sigma, green, rot):
    """Windows of 1 to 4 cells a side, green as large as the others, and one just too large for the
    kernel (1.34 x 3 px reaches five cells), with calibration frames and saturated pixels."""
    fr = _frame(71, 45, rot, sigma=sigma, green_ratio=green, calibrated=True)
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))
    fr = dataclasses.replace(fr, params=dataclasses.replace(fr.params, sigmas=(1.34,)))
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


@pytest.mark.parametrize("rot", [0.0, 0.3])
@pytest.mark.parametrize("ow,oh", [(142, 90), (107, 68), (50, 31), (18, 12), (9, 6)])
def test_resampled_outputs(ctx, ow, oh, rot):
    """Enlarged and reduced outputs; the eightfold reduction outgrows every kernel's staging and stays
    refused."""
    from paper_1308_4908_gb300 import hdr
    fr = _frame(71, 45, rot, out_w=ow, out_h=oh, out_affine=synth.output_affine(71, 45, ow, oh))
    if ow == 9:
        with pytest.raises(hdr.HdrError) as e:
            _run(ctx, fr)
        assert e.value.status == hdr.HDR_E_UNSUPPORTED
        return
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


@pytest.mark.parametrize("affine", [[[-1.0, 0, 70.0], [0, 1.0, 0]], [[0, 1.0, 0.2], [1.0, 0, -0.3]],
                                    [[1.0, 0, -20.0], [0, -1.0, 60.0]]])
def test_mirrored_transposed_and_outside(ctx, affine):
    """Output mappings that mirror, transpose, and reach past the sensors (NaN, level 255 there)."""
    fr = _frame(71, 45, 0.0, out_affine=np.array(affine))
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))
    assert np.array_equal(np.isnan(out), ch == 255)


@pytest.mark.parametrize("w,h,scale", [(131, 34, 1.0), (97, 66, 1.4)])
def test_sheared_sensors(ctx, w, h, scale):
    """Sensors whose axes are neither orthogonal nor evenly scaled: the windows are ellipses in the
    sensor and the Gaussian does not factor."""
    fr = _frame(w, h, 1.0, n=3, out_affine=np.array([[1 / scale, 0.01, 0.3], [-0.02, 1 / scale, 0.6]]))
    for k, s in enumerate(fr.sensors):
        s.affine = s.affine @ np.array([[1.0, 0.03 * (k + 1), 0.0], [0.0, 1.0 + 0.04 * k, 0.0], [0.0, 0.0, 1.0]])
        s.raw = synth.simulate_raw(fr.scene, s, 1500, k)
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


@pytest.mark.parametrize("n", [1, 8])
@pytest.mark.parametrize("rot", [0.0, 2.0])
def test_sensor_counts_and_half(ctx, n, rot):
    fr = _frame(80, 33, rot, n=n, out_dtype=1)
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params), extra=parity.HALF_TOL)


@pytest.mark.parametrize("w,h,rot", [(832, 760, 0.0), (832, 760, 0.2), (1250, 1010, 0.0), (1250, 1010, 0.2)])
def test_larger_tiles_and_every_entry_point(ctx, w, h, rot):
    """Two and four rows per thread (the frame sizes that choose them): sampled pixels and the border
    against the oracle; batches of every launch configuration, the host-buffer bands and a server that
    takes the frame in steps of odd tile counts return the same bits."""
    from paper_1308_4908_gb300 import hdr
    fr = _frame(w, h, rot)
    out, ch, raws = _run(ctx, fr)
    p = fr.params
    r = np.random.default_rng(w)
    pix = np.concatenate([np.stack([r.integers(0, w, 1500), r.integers(0, h, 1500)], 1),
                          [[0, 0], [w - 1, 0], [0, h - 1], [w - 1, h - 1]]])
    _against_oracle(fr, out, ch, pix)
    for cfg in (hdr.hdr_batch_config(16, 0, 1, 0), hdr.hdr_batch_config(8, 0, 1, 0),
                hdr.hdr_batch_config(16, 0, 1, 0, 2, 1), hdr.hdr_batch_config(16, 0, 1, 0, 1, 2)):
        o = torch.full((3, h, w), -7.0, device="cuda")
        c = torch.full((3, h, w), 77, dtype=torch.uint8, device="cuda")
        keep = [raws]
        ctx.reconstruct_batch([ctx.frame(0, p, raws, o, c, keep)], cfg)
        ctx.check()
        np.testing.assert_array_equal(o.cpu().numpy(), out)
        np.testing.assert_array_equal(c.cpu().numpy(), ch)
    host = [np.ascontiguousarray(s.raw) for s in fr.sensors]
    o, c = np.full((3, h, w), -7.0, np.float32), np.full((3, h, w), 77, np.uint8)
    ctx.reconstruct_host(0, p, host, o, c)
    np.testing.assert_array_equal(o, out)
    np.testing.assert_array_equal(c, ch)
    own = hdr.Context(0)
    try:
        own.set_rig(0, fr.sensors)
        srv = hdr.Server(own, max_frames=2, pool_bytes=256 << 20, step_tiles=777)
        o[:], c[:] = -7.0, 77
        assert srv.poll(srv.submit(0, p, host, o, c)).status == hdr.HDR_OK
        srv.close()
    finally:
        own.close()
    np.testing.assert_array_equal(o, out)
    np.testing.assert_array_equal(c, ch)


@pytest.mark.parametrize("rot", [0.0, 0.3])
@pytest.mark.parametrize("scale,shear", [(1.0, 0.0), (1.5, 0.0), (1.5, 0.05)])
@pytest.mark.parametrize("sigma", [0.7, 1.2])
def test_compensated_sums(ctx, sigma, scale, shear, rot):
    """accum 1 in every form and window size, around the 64 x 16 tiles of its two rows per thread."""
    w, h = round(90 * scale) + 1, round(33 * scale)
    fr = _frame(90, 33, rot, n=3, sigma=sigma, accum=1, out_w=w, out_h=h,
                out_affine=np.array([[1 / scale, 0.0, 0.2], [0.0, 1 / scale, -0.1]]))
    if shear:
        for k, s in enumerate(fr.sensors):
            s.affine = s.affine @ np.array([[1.0, shear, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
            s.raw = synth.simulate_raw(fr.scene, s, 1500, k)
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


@pytest.mark.parametrize("shift,w", [(-9.0e6, 9_000_064), (-5.0e5, 500_064)])
def test_far_coordinates(ctx, shift, w):
    """Sensors that only the last pixels of a very wide output reach: the terms of a position are
    large there and cancel, on both sides of the line up to which FP32 box origins serve."""
    fr = _frame(64, 8, 0.3)
    fr = dataclasses.replace(fr, params=dataclasses.replace(fr.params, out_w=w, out_h=2, out_affine=(0.9999, 0, 0.9999 * shift, 0, 0.9999, 0)))
    out, ch, _ = _run(ctx, fr)
    pix = _every_pixel(dataclasses.replace(fr.params, out_w=96)) + [w - 96, 0]
    assert np.isfinite(out[:, pix[:, 1], pix[:, 0]]).mean() > 0.5
    _against_oracle(fr, out, ch, pix)


@pytest.mark.parametrize("n,reduce,rot", [(8, 1.0, 0.3), (8, 2.0, 0.3), (8, 2.6, 0.0), (8, 3.2, 0.3), (4, 4.0, 0.3), (2, 6.0, 0.3), (1, 7.0, 0.0)])
def test_refused_as_by_the_general_kernel(ctx, n, reduce, rot):
    """Outputs that outgrow the general kernel's staging (order 1 has the same) are refused at order 0
    too, although its own kernel could stage the sensors in turn."""
    from paper_1308_4908_gb300 import hdr
    fr = _frame(96, 64, rot, n=n, out_w=40, out_h=30, out_affine=np.array([[reduce, 0, 1.0], [0, reduce, 0.5]]))
    refused = []
    for order in (0, 1):
        try:
            _run(ctx, dataclasses.replace(fr, params=dataclasses.replace(fr.params, order=order)))
            refused.append(0)
        except hdr.HdrError as e:
            refused.append(e.status)
    assert refused[0] == refused[1] and refused[0] in (0, hdr.HDR_E_UNSUPPORTED)
    if (n, reduce) in ((8, 1.0), (8, 3.2)):
        assert (refused[0] == 0) == (reduce == 1.0)


@pytest.mark.parametrize("nudge", [-1e-6, 0.0, 1e-6])
@pytest.mark.parametrize("scale,rot", [(1.0, 0.0), (1.5, 0.0), (1.0, 0.2), (1.3, 0.0)])
def test_boxes_on_an_alignment_boundary(ctx, scale, rot, nudge):
    """Sensors displaced by the reach of the staging box, so that its corner falls on a multiple of 8 px, or a
    rounding to either side, in every tile of an unrotated frame: the fetched samples and the position tables must
    agree on it."""
    w, h = round(131 * scale), round(34 * scale)
    fr = _frame(131, 34, rot, out_w=w, out_h=h, out_affine=np.array([[1 / scale, 0.0, 0.0], [0.0, 1 / scale, 0.0]]))
    for k, s in enumerate(fr.sensors):
        s.affine = np.array(s.affine, dtype=np.float64)
        s.affine[:, 2] = -(3 * 0.7 + 2e-3 + 1.0 + nudge) + 8.0 * k
        s.raw = synth.simulate_raw(fr.scene, s, 1500, k)
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


def _edge_frame(**over):
    """Three exactly translated sensors whose red samples lie within 1e-5 px of the edge of every even pixel's
    window, so that their window values are a few 1e-7 of the centre's."""
    fr = _frame(70, 41, 0.0, n=3, sigma=1.3 / 3, **over)
    for k, s in enumerate(fr.sensors):
        s.affine = np.array([[1.0, 0.0, 1.0], [0.0, 1.0, math.sqrt((1.3 - 1e-5 * (k + 1)) ** 2 - 1.0)]])
        s.raw = synth.simulate_raw(fr.scene, s, 1500, k)
    return fr


def _without_window_rounding(fr, out):
    """Every pixel within the parity rule's terms for conversion and FP32 sums alone: window values that are exact
    to one rounding need nothing of the term for their evaluation (ew)."""
    p = fr.params
    pix = _every_pixel(p)
    o = oracle.reconstruct(fr.sensors, p, pix, levels=True)
    g = out[:, pix[:, 1], pix[:, 0]].T
    tol = parity.level_tol(o["out"], o["efit"][:, :, 0], 0.0)
    assert np.array_equal(np.isnan(g), np.isnan(o["out"]))
    m = ~np.isnan(g)
    assert (np.abs(g - o["out"])[m] <= tol[m]).all(), float((np.abs(g - o["out"])[m] / tol[m]).max())


def test_tabulated_weights_at_the_window_edge(ctx):
    """tab_weights 1: window values formed in FP64. In FP32 they are off by parts in a thousand at the edge of
    a window, and so are the estimates there."""
    fr = _edge_frame()
    _without_window_rounding(fr, _run(ctx, fr)[0])


@pytest.mark.parametrize("scale,shear", [(5e-13, 0.0), (0.0, 5e-13), (-4e-13, -3e-13)])
def test_nearly_exact_translations(ctx, scale, shear):
    """Sensors whose linear part is the identity to the tolerance of the tabulated weights, but not exactly."""
    fr = _frame(131, 34, 0.0)
    for s in fr.sensors:
        s.affine = np.array(s.affine) + np.array([[scale, shear, 0.0], [-shear, scale, 0.0]])
    out, ch, _ = _run(ctx, fr)
    _against_oracle(fr, out, ch, _every_pixel(fr.params))


@pytest.mark.parametrize("w,h", [(832, 380), (832, 760), (1250, 1010)])  # one, two and eight rows per thread
@pytest.mark.parametrize("sigma,accum", [(0.7, 0), (1.2, 0), (1.2, 1)])
def test_tabulated_weights_in_every_entry_point(ctx, w, h, sigma, accum):
    """Sampled pixels against the oracle, and the same bits from a batch, the host-buffer bands and a first call
    under stream capture, whose table is not there yet."""
    from paper_1308_4908_gb300 import hdr
    fr = _frame(w, h, 0.0, n=3, sigma=sigma, accum=accum)
    out, ch, raws = _run(ctx, fr)
    p = fr.params
    r = np.random.default_rng(w)
    pix = np.concatenate([np.stack([r.integers(0, w, 1500), r.integers(0, h, 1500)], 1),
                          [[0, 0], [w - 1, 0], [0, h - 1], [w - 1, h - 1]]])
    _against_oracle(fr, out, ch, pix)
    o = torch.full((3, h, w), -7.0, device="cuda")
    keep = [raws]
    ctx.reconstruct_batch([ctx.frame(0, p, raws, o, None, keep)])
    ctx.check()
    np.testing.assert_array_equal(o.cpu().numpy(), out)
    host = np.full((3, h, w), -7.0, np.float32)
    ctx.reconstruct_host(0, p, [np.ascontiguousarray(s.raw) for s in fr.sensors], host)
    np.testing.assert_array_equal(host, out)
    own = hdr.Context(0)
    try:
        own.set_rig(0, fr.sensors)
        o.fill_(-7.0)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            own.reconstruct(0, p, raws, out=o)
        g.replay()
        torch.cuda.synchronize()
        own.check()
    finally:
        own.close()
    np.testing.assert_array_equal(o.cpu().numpy(), out)


@pytest.mark.parametrize("trunc_k", [0.05, 0.3, 0.99])
def test_windows_cut_close_in(ctx, trunc_k):
    """Windows cut below one sigma, where the window value is the difference of nearly equal exponentials: left to
    the tabulated windows' general kernel."""
    fr = _frame(71, 45, 0.0, n=3, sigma=2.0 / trunc_k, trunc_k=trunc_k)
    _without_window_rounding(fr, _run(ctx, fr)[0])


@pytest.mark.parametrize("sigma,rot,n", [(1.2, 0.0, 2), (1.2, 0.2, 2), (0.7, 0.0, 4), (1.2, 0.0, 4)])
def test_largest_tiles_enlarged(ctx, sigma, rot, n):
    """Twofold output of at least four tiles of 64 x 32 per SM and CTA: the largest tiles of each form and window size,
    sampled pixels and the border."""
    fr = _frame(625, 505, rot, n=n, sigma=sigma, out_w=1250, out_h=1010, out_affine=synth.output_affine(625, 505, 1250, 1010))
    out, ch, _ = _run(ctx, fr)
    r = np.random.default_rng(n)
    pix = np.concatenate([np.stack([r.integers(0, 1250, 2000), r.integers(0, 1010, 2000)], 1),
                          np.stack([np.arange(1250), np.full(1250, 1009)], 1), np.stack([np.full(1010, 1249), np.arange(1010)], 1)])
    _against_oracle(fr, out, ch, pix)
