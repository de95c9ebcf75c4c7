"""Assignment of a tile's pixels to threads by phase class (PixelMap).

Each axis takes every 1st to 4th pixel in turn by the output's scale; the value of a pixel must not
depend on the thread that computes it. Every pixel is compared with the oracle (the parity rule of
tests/parity.py) at scales that select every stride, unequal on the two axes, on ragged outputs;
tiles of 8 rows and of two pixels per thread, whose maps differ, return the same bits.
"""
import dataclasses

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


@pytest.mark.parametrize("order", [0, 2])
@pytest.mark.parametrize("sx,sy", [(0.5, 1.0), (1.0, 1.5), (1.5, 1.5), (2.0, 0.6), (1.875, 1.0547), (3.0, 2.0)])
def test_every_stride(ctx, order, sx, sy):
    from paper_1308_4908_gb300 import hdr
    fr = synth.paper_scale(size=40, seed=1600)
    w, h = round(40 * sx) - 1, round(40 * sy) - 1
    p = dataclasses.replace(fr.params, order=order, sigmas=(0.6, 1.1), out_w=w, out_h=h,
                            out_affine=synth.output_affine(40, 40, w, h))
    ctx.set_rig(0, fr.sensors)
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]

    def buffers():
        return (torch.full((3, h, w), -7.0, device="cuda"), torch.full((3, h, w), 77, dtype=torch.uint8, device="cuda"))

    out, ch = buffers()
    ctx.reconstruct(0, p, raws, out=out, choice=ch)
    ctx.check()
    g, gc = out.cpu().numpy(), ch.cpu().numpy()
    vv, uu = np.mgrid[0:h, 0:w]
    pix = np.stack([uu.ravel(), vv.ravel()], axis=1)
    o = oracle.reconstruct(fr.sensors, p, pix, levels=True, kappa=True)
    parity.compare(g[:, pix[:, 1], pix[:, 0]], gc[:, pix[:, 1], pix[:, 0]], o, pix, 2, order, p.ici_gamma, p.min_pivot)
    for cfg in (hdr.hdr_batch_config(8, 0, 1, 0), hdr.hdr_batch_config(16, 0, 1, 0, 2, 1)):
        o2, c2 = buffers()
        keep = [raws]
        ctx.reconstruct_batch([ctx.frame(0, p, raws, o2, c2, keep)], cfg)
        ctx.check()
        np.testing.assert_array_equal(o2.cpu().numpy(), g)
        np.testing.assert_array_equal(c2.cpu().numpy(), gc)


@pytest.mark.parametrize("order", [0, 2])
@pytest.mark.parametrize("step", [1.5, 2.5, 3.0, 3.5])
def test_strides_of_reduced_outputs(ctx, order, step):
    """Reduced outputs whose 2nd or 4th pixels repeat the samples' fractions, ragged and half tiles."""
    fr = synth.paper_scale(size=120, seed=1601)
    w, h = round(120 / step) + 1, round(100 / step) - 3
    p = dataclasses.replace(fr.params, order=order, sigmas=(0.6, 1.1), out_w=w, out_h=h,
                            out_affine=np.array([[step, 0.0, 0.3], [0.0, step, 0.6]]))
    ctx.set_rig(0, fr.sensors)
    ch = torch.full((3, h, w), 77, dtype=torch.uint8, device="cuda")
    out = ctx.reconstruct(0, p, [torch.from_numpy(s.raw).cuda() for s in fr.sensors], choice=ch)
    ctx.check()
    g, gc = out.cpu().numpy(), ch.cpu().numpy()
    vv, uu = np.mgrid[0:h, 0:w]
    pix = np.stack([uu.ravel(), vv.ravel()], axis=1)
    o = oracle.reconstruct(fr.sensors, p, pix, levels=True, kappa=True)
    parity.compare(g[:, pix[:, 1], pix[:, 0]], gc[:, pix[:, 1], pix[:, 0]], o, pix, 2, order, p.ici_gamma, p.min_pivot)
