"""Frames with one window scale, whose kernels leave the variance sums out.

The interval rule has nothing to compare with one scale, so Var C_0 is not formed; the values must
stay the same bits. Two pixels per thread and two staging buffers run the kernels that keep the
variance sums, so batches with these settings are the reference of the single-frame call.
"""
import dataclasses

import numpy as np
import pytest

from paper_1308_4908_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1308_4908_gb300 import hdr
    c = hdr.Context(0)
    yield c
    c.close()


def _frame(translational, order):
    fr = synth.paper_scale(size=61, seed=1400 + order)
    if translational:
        for k, s in enumerate(fr.sensors):
            s.affine = np.asarray(synth.affine_about_center(61, 61, 0.3 * k - 0.4, 0.7 - 0.9 * k))
            s.raw = synth.simulate_raw(fr.scene, s, 1400, k)
    return fr


@pytest.mark.parametrize("cond_fallback", [1e6, 1.0])  # FP32 only; the FP64 re-solve compiled in
@pytest.mark.parametrize("accum", [0, 1])
@pytest.mark.parametrize("translational", [False, True])
@pytest.mark.parametrize("order", [1, 2])
def test_values_do_not_depend_on_the_variance_sums(ctx, order, translational, accum, cond_fallback):
    from paper_1308_4908_gb300 import hdr
    fr = _frame(translational, order)
    p = dataclasses.replace(fr.params, order=order, sigmas=(1.1,), out_w=59, out_h=35, accum=accum,
                            cond_fallback=cond_fallback)
    ctx.set_rig(0, fr.sensors)
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]

    def buffers():
        return (torch.full((3, p.out_h, p.out_w), -7.0, device="cuda"),
                torch.empty((3, p.out_h, p.out_w), dtype=torch.uint8, device="cuda"))

    out, ch = buffers()
    ctx.reconstruct(0, p, raws, out=out, choice=ch)
    for cfg in (hdr.hdr_batch_config(16, 0, 1, 0, 2, 1), hdr.hdr_batch_config(16, 0, 1, 0, 1, 2),
                hdr.hdr_batch_config(8, 0, 1, 0, 1, 1)):
        o, c = buffers()
        keep = [raws]
        ctx.reconstruct_batch([ctx.frame(0, p, raws, o, c, keep)], cfg)
        ctx.check()
        np.testing.assert_array_equal(c.cpu().numpy(), ch.cpu().numpy())
        np.testing.assert_array_equal(o.cpu().numpy(), out.cpu().numpy())


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("sigma,green,zoom", [(0.34, 1.0, 1.0), (0.67, 0.5, 1.0), (0.99, 0.7, 1.0), (1.0, 1.0, 1.0),
                                              (1.33, 0.5, 1.0), (1.34, 0.76, 1.0), (0.7, 0.9, 0.55)])
def test_window_sizes_of_the_fixed_walk(ctx, order, sigma, green, zoom):
    """Windows on both sides of the reaches (1, 2, 3 and 4 px, also unequal on a stretched sensor) between which
    single-scale kernels take a fixed block of cells: the same bits as the kernels that search every
    window (two pixels per thread)."""
    from paper_1308_4908_gb300 import hdr
    fr = _frame(False, order)
    if zoom != 1.0:
        for s in fr.sensors:
            s.affine = s.affine @ np.array([[zoom, 0.0, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    p = dataclasses.replace(fr.params, order=order, sigmas=(sigma,), green_ratio=green, out_w=50, out_h=47)
    ctx.set_rig(0, fr.sensors)
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]
    got = []
    for batch in (False, True):
        out = torch.full((3, 47, 50), -7.0, device="cuda")
        ch = torch.empty((3, 47, 50), dtype=torch.uint8, device="cuda")
        if batch:
            keep = [raws]
            ctx.reconstruct_batch([ctx.frame(0, p, raws, out, ch, keep)], hdr.hdr_batch_config(16, 0, 1, 0, 2, 1))
        else:
            ctx.reconstruct(0, p, raws, out=out, choice=ch)
        ctx.check()
        got.append((out.cpu().numpy(), ch.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("sigma,green", [(0.79, 1.0), (0.81, 0.9), (0.99, 0.7), (1.0, 0.8), (1.12, 1.0), (1.14, 0.7), (1.33, 0.6), (1.34, 0.6)])
def test_fixed_walk_at_order_0(ctx, sigma, green):
    """Order 0 outside its own kernel (a pivot threshold next to 1), on both sides of the reaches from which its
    windows take a fixed block of cells (2.4 to 3 and 3.4 to 4 px): the same bits as the kernels that search."""
    from paper_1308_4908_gb300 import hdr
    fr = _frame(False, 1)
    p = dataclasses.replace(fr.params, order=0, sigmas=(sigma,), green_ratio=green, min_pivot=0.995, out_w=50, out_h=47)
    ctx.set_rig(0, fr.sensors)
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]
    got = []
    for batch in (False, True):
        out = torch.full((3, 47, 50), -7.0, device="cuda")
        ch = torch.empty((3, 47, 50), dtype=torch.uint8, device="cuda")
        if batch:
            keep = [raws]
            ctx.reconstruct_batch([ctx.frame(0, p, raws, out, ch, keep)], hdr.hdr_batch_config(16, 0, 1, 0, 2, 1))
        else:
            ctx.reconstruct(0, p, raws, out=out, choice=ch)
        ctx.check()
        got.append((out.cpu().numpy(), ch.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
    assert np.isfinite(got[0][0]).mean() > 0.5
