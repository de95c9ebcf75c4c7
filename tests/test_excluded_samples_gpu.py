"""Samples that FP32 cannot hold are left out as saturated ones are.

A per-pixel sensitivity near the smallest float makes the weight 0 and the value infinite, a bias that is no
number makes the value none, a read variance near the smallest float makes the weight infinite. A frame with
such pixels must return the bits of the frame whose same pixels are marked saturated: every pixel, in
every kernel (windows searched, tabulated, small and fixed; frames converted ahead or in the kernel).
"""
import dataclasses

import numpy as np
import pytest

from paper_1308_4908_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MARKS = [("prnu_frame", 1e-38), ("prnu_frame", 1e-41), ("bias_frame", np.nan), ("bias_frame", np.inf),
         ("bias_frame", -np.inf), ("read_var_frame", 1e-45)]


@pytest.fixture(scope="module")
def ctx():
    from paper_1308_4908_gb300 import hdr
    c = hdr.Context(0)
    yield c
    c.close()


def _frames(w, h, rot, params):
    """(frame with unusable pixels, the same with these saturated)."""
    fr = synth._build_frame(1900 + w, 2, w, h, (1.0, 1 / 8), 1.2, rot, 0.0, params, "excluded")
    pair = []
    for marked in (True, False):
        r = np.random.default_rng(w)
        sensors = []
        for s in fr.sensors:
            s = dataclasses.replace(s)
            s.raw = s.raw.copy()
            s.bias_frame = (s.black + r.uniform(-2, 2, (h, w))).astype(np.float32)
            s.prnu_frame = r.uniform(0.95, 1.05, (h, w)).astype(np.float32)
            s.read_var_frame = r.uniform(6, 12, (h, w)).astype(np.float32)
            s.sat_frame = np.full((h, w), 4000, np.uint16)
            for k, at in enumerate(r.choice(w * h, 4 * len(MARKS), replace=False)):
                y, x = divmod(int(at), w)
                s.raw[y, x] = 0 if MARKS[k % len(MARKS)][0] == "read_var_frame" else 900
                if marked:
                    name, value = MARKS[k % len(MARKS)]
                    getattr(s, name)[y, x] = value
                else:
                    s.sat_frame[y, x] = 0
            sensors.append(s)
        pair.append(sensors)
    return pair


@pytest.mark.parametrize("weight_mode", [0, 1])
@pytest.mark.parametrize("w,h", [(61, 45), (260, 170)])  # converted in the kernel; ahead of it
@pytest.mark.parametrize("rot", [0.0, 0.3])
@pytest.mark.parametrize("order,sigmas", [(0, (0.7,)), (0, (1.2,)), (0, (1.6,)), (0, synth.PAPER_SCALES), (1, (1.2,)),
                                          (1, synth.PAPER_SCALES), (2, (1.2,)), (2, synth.PAPER_SCALES)])
def test_as_saturated(ctx, order, sigmas, rot, w, h, weight_mode):
    p = synth.Params(order=order, sigmas=sigmas, out_w=w, out_h=h, weight_mode=weight_mode)
    got = []
    for sensors in _frames(w, h, rot, p):
        ctx.set_rig(0, sensors)
        raws = [torch.from_numpy(s.raw).cuda() for s in sensors]
        ch = torch.empty((3, h, w), dtype=torch.uint8, device="cuda")
        out = ctx.reconstruct(0, p, raws, choice=ch)
        ctx.check()
        got.append((out.cpu().numpy(), ch.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
    assert np.isfinite(got[0][0]).mean() > 0.9


@pytest.mark.parametrize("grad_sigma", [1.2, 2.4])  # the gradient pass's own kernel; the general one
def test_gradients_as_saturated(ctx, grad_sigma):
    from paper_1308_4908_gb300 import hdr
    p = synth.Params(order=2, out_w=61, out_h=45)
    got = []
    for sensors in _frames(61, 45, 0.3, p):
        ctx.set_rig(0, sensors)
        raws = [torch.from_numpy(s.raw).cuda() for s in sensors]
        got.append(ctx.calpa_gradients(0, p, hdr.hdr_calpa_params_default(grad_sigma=grad_sigma), raws).cpu().numpy())
        ctx.check()
    np.testing.assert_array_equal(got[0], got[1])
    assert np.isfinite(got[0]).all()
