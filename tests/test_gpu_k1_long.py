"""K1 for long frames against the oracle: the power spectrum alone from registers (T =
1024, 2048, 4096; odd numbers of frames in the last batch of a group, chunks that start
anywhere, so that samples come from the carry-over and from unaligned addresses, int16,
several channels, S1) and transform and centring in two kernels (groups that do not fit
in shared memory, with every consumer of the spectra).
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL, TOL_ERR = 1e-5, 1e-4


def check(got, ref, keys):
    for key in keys:
        a, e = got[key][0], got[key + "_err"][0]
        r, re = ref[key], ref[key + "_err"].reshape(e.shape)
        assert np.max(np.abs(a - r.reshape(a.shape))) <= TOL * np.max(np.abs(r)), key
        assert np.max(np.abs(e - re)) <= TOL_ERR * np.max(re), key


@pytest.mark.parametrize("T,m,G", [(1024, 2, 3), (1024, 5, 40), (2048, 3, 7), (2048, 16, 5),
                                   (4096, 2, 2), (4096, 7, 4), (1024, 90, 3)])
@pytest.mark.parametrize("cuts", [(), (1, 4097, 9001)])
def test_power_spectrum_alone(T, m, G, cuts):
    import paper_2505_01231_gb300 as mod
    n = T * m * G + T + 5
    z = synth.ar1_quadratic(n, seed=T + m) + np.float32(3.0)   # an offset: S1 is not zero
    ref = oracle.polyspectra(z, T, 0.5, m, orders=(1, 2), group_chunk=8)
    plan = mod.Plan(T=T, dt=0.5, m=m, orders=(1, 2))
    zd = torch.from_numpy(z).cuda()
    cuts = [0] + [c for c in cuts if c < n] + [n]
    for a, b in zip(cuts, cuts[1:]):
        plan.accumulate(zd[a:b])
    out = plan.finalize()
    plan.close()
    assert out["G"] == ref["G"]
    check(out, ref, ("S2",))
    assert abs(out["S1"][0] - ref["S1"]) <= TOL * abs(ref["S1"])


def test_power_spectrum_alone_int16_and_channels():
    import paper_2505_01231_gb300 as mod
    T, m, G, C = 2048, 5, 9, 3
    n = T * m * G + 33
    z = np.rint(500 * synth.multichannel_shared(C, n, seed=6)).astype(np.int16)
    recs = [(2, c, c, -1, -1) for c in range(C)]
    plan = mod.Plan(channels=C, T=T, dt=0.5, m=m, orders=(2,), dtype="i16", combos=recs)
    plan.accumulate(torch.from_numpy(z).cuda())
    out = plan.finalize()
    plan.close()
    for c in range(C):
        ref = oracle.polyspectra(z[c].astype(np.float64), T, 0.5, m, orders=(2,), group_chunk=8)
        assert np.max(np.abs(out["S2"][c] - ref["S2"])) <= TOL * np.max(np.abs(ref["S2"]))


@pytest.mark.parametrize("T,m,G,precision,k1", [(2048, 16, 3, "fp32", "auto"),
                                                (4096, 6, 3, "fp16x3", "auto"),
                                                (4096, 5, 3, "tf32x3", "auto"),
                                                (1024, 5, 70, "bf16x3", "frames"),
                                                (2048, 40, 3, "fp32", "auto")])
def test_transform_and_centring_in_two_kernels(T, m, G, precision, k1):
    import paper_2505_01231_gb300 as mod
    z = synth.ar1_quadratic(T * m * G + 9, seed=T + m)
    ref = oracle.polyspectra(z, T, 0.5, m, orders=(2, 4), group_chunk=4)
    plan = mod.Plan(T=T, dt=0.5, m=m, orders=(1, 2, 4), precision=precision)
    mod.ss_set_tuning(plan.handle, f"k1={k1}")
    plan.accumulate(torch.from_numpy(z).cuda())
    out = plan.finalize()
    plan.close()
    check(out, ref, ("S2",))
    tol = 5e-5 if precision == "bf16x3" else TOL
    assert np.max(np.abs(out["S4"][0] - ref["S4"])) <= tol * np.max(np.abs(ref["S4"]))
