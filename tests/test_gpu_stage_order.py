"""The staged pipelines of the tensor-core S4 kernels over many groups per CTA.

One channel: with more stages per group than the ring holds (TF32x3 from m = 11,
FP16x3 from m = 16), and with one stage per group over thousands of short groups,
a product must wait for its own load and not for the ring's previous use.
Several channels: a staged coefficient must not be overwritten before every lane
has used it, so passes over one record agree to the rounding of the float64 sums.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def P():
    import paper_2505_01231_gb300 as mod
    return mod


@pytest.mark.parametrize("precision,m,G", [("tf32x3", 11, 900), ("tf32x3", 16, 700),
                                           ("fp16x3", 16, 700), ("fp16x3", 32, 500),
                                           ("tf32x3", 32, 500)])
def test_more_stages_per_group_than_the_ring_holds(precision, m, G):
    T = 64
    z = synth.ar1_quadratic(T * m * G + 7, seed=m)
    ref = oracle.polyspectra(z, T, 0.5, m, orders=(4,), group_chunk=64)
    plan = P().Plan(T=T, dt=0.5, m=m, orders=(4,), precision=precision)
    for _ in range(3):
        plan.reset()
        plan.accumulate(torch.from_numpy(z).cuda())
        got = plan.finalize()
        # the bar of every FP32-level precision: 1e-5 of the peak
        assert np.max(np.abs(got["S4"][0] - ref["S4"])) <= 1e-5 * np.max(np.abs(ref["S4"]))
    plan.close()


@pytest.mark.parametrize("precision", ["tf32x3", "fp16x3"])
def test_one_stage_per_group_over_many_short_groups(precision):
    T, m, n = 64, 10, 1 << 24
    z = torch.from_numpy(synth.ar1_quadratic(n, seed=3)).cuda()
    outs = []
    for prec in ("fp32", precision):
        plan = P().Plan(T=T, dt=0.5, m=m, orders=(4,), precision=prec)
        for _ in range(1 if prec == "fp32" else 4):
            plan.reset()
            plan.accumulate(z)
            outs.append(plan.finalize()["S4"][0])
        plan.close()
    peak = np.max(np.abs(outs[0]))
    for o in outs[1:]:  # both within 1e-5 of the definition
        assert np.max(np.abs(o - outs[0])) <= 2e-5 * peak


@pytest.mark.parametrize("precision", ["fp16x3", "tf32x3"])
def test_cross_channel_passes_agree(precision):
    T, m, G = 512, 20, 1200
    z = torch.from_numpy(synth.multichannel_shared(2, T * m * G, seed=4)).cuda()
    plan = P().Plan(channels=2, T=T, dt=0.5, m=m, orders=(4,), precision=precision)
    outs = []
    for _ in range(4):
        plan.reset()
        plan.accumulate(z)
        outs.append(plan.finalize())
    plan.close()
    for key in ("S4", "S4_err"):
        peak = np.max(np.abs(outs[0][key]))
        for o in outs[1:]:
            # the order of the float64 additions is all that differs between passes
            # (the variance behind an error bar cancels: 1e-9 of the peak)
            assert np.max(np.abs(o[key] - outs[0][key])) <= 1e-9 * peak, key
