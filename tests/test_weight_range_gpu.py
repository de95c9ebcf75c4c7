"""Rigs whose units take the weights to the ends of FP32's range.

Scaling every exposure by 2^m scales radiances by 2^-m and inverse variances by 2^2m, and changes no rounding: the
estimates must be those of the ordinary rig times 2^-m, bit for bit, with the same choices, and the level maps'
variances times 2^-2m. Unscaled, sums of such weights are denormal (their reciprocals infinite) or overflow.
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


def _sensors(fr, m, calibrated):
    out = []
    for k, s in enumerate(fr.sensors):
        s = dataclasses.replace(s, exposure=s.exposure * 2.0 ** m)
        if calibrated:
            r = np.random.default_rng(k)
            s.prnu_frame = r.uniform(0.95, 1.05, (s.height, s.width)).astype(np.float32)
            s.read_var_frame = r.uniform(6, 12, (s.height, s.width)).astype(np.float32)
        out.append(s)
    return out


@pytest.mark.parametrize("m", [-60, -52, 50])
@pytest.mark.parametrize("rot,calibrated", [(0.0, False), (0.3, True)])
@pytest.mark.parametrize("order,sigmas,over", [
    (0, (0.7,), {}), (0, (0.7,), {"accum": 1}), (0, (1.6,), {}), (0, synth.PAPER_SCALES, {}), (1, (1.2,), {}),
    (1, synth.PAPER_SCALES, {}), (2, (1.2,), {"accum": 1}), (2, synth.PAPER_SCALES, {}),
    (2, synth.PAPER_SCALES, {"cond_fallback": 10.0}), (2, synth.PAPER_SCALES, {"weight_mode": 1})])
def test_scaled_exposures(ctx, order, sigmas, over, rot, calibrated, m):
    p = synth.Params(order=order, sigmas=sigmas, out_w=70, out_h=41, **over)
    fr = synth._build_frame(1950, 2, 70, 41, (1.0, 1 / 8), 1.2, rot, 0.0, p, "range")
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]
    levels = over.get("weight_mode", 0) == 0
    got = []
    for e in (0, m):
        ctx.set_rig(0, _sensors(fr, e, calibrated))
        ch = torch.empty((3, 41, 70), dtype=torch.uint8, device="cuda")
        out = ctx.reconstruct(0, p, raws, choice=ch)
        ctx.check()
        lv = torch.zeros((3, len(sigmas) + order, 41, 70, 2), device="cuda")
        if levels:
            ctx.reconstruct(0, p, raws, choice=ch, levels=lv)
            ctx.check()
        got.append((out.cpu().numpy(), ch.cpu().numpy(), lv.cpu().numpy()))
    np.testing.assert_array_equal(np.ldexp(got[1][0], m), got[0][0])
    np.testing.assert_array_equal(got[1][1], got[0][1])
    with np.errstate(over="ignore"):  # variances beyond FP32 are infinite
        np.testing.assert_array_equal(got[1][2], np.ldexp(got[0][2], np.array([-m, -2 * m])))
    assert np.isfinite(got[0][0]).mean() > 0.9


def test_scaled_gradients(ctx):
    from paper_1308_4908_gb300 import hdr
    p = synth.Params(order=2, out_w=70, out_h=41)
    fr = synth._build_frame(1951, 3, 70, 41, (1.0, 1 / 8, 1 / 64), 1.2, 0.3, 0.0, p, "range")
    raws = [torch.from_numpy(s.raw).cuda() for s in fr.sensors]
    got = []
    for e in (0, -52):
        ctx.set_rig(0, _sensors(fr, e, False))
        got.append(ctx.calpa_gradients(0, p, hdr.hdr_calpa_params_default(), raws).cpu().numpy())
        ctx.check()
    np.testing.assert_array_equal(np.ldexp(got[1], -52), got[0])
