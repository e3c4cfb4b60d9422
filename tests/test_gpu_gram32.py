"""The FP32 S4 as one contraction of the frame Gram (m <= 16) against the oracle, and
against the five-sum form on both sides of the limit: ragged tiles (T = 8 .. 64), the
column l = M - 1 of its own (T >= 128), entry counts around multiples of 8 (m = 5: 16,
m = 10: 56, m = 12: 79), both estimators.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,m,G", [(8, 4, 50), (16, 5, 40), (64, 12, 30), (128, 10, 24),
                                   (256, 16, 9), (256, 17, 9), (512, 7, 6), (4096, 4, 3),
                                   (32, 9, 4000)])
@pytest.mark.parametrize("natural", [False, True])
def test_gram_form_matches_the_oracle(T, m, G, natural):
    import paper_2505_01231_gb300 as mod
    z = synth.ar1_quadratic(T * m * G + 2 * T + 3, seed=T + m)
    est = "natural" if natural else "unbiased"
    ref = oracle.polyspectra(z, T, 0.5, m, orders=(4,), group_chunk=64, estimator=est)
    plan = mod.Plan(T=T, dt=0.5, m=m, orders=(4,), estimator=est)
    plan.accumulate(torch.from_numpy(z).cuda())
    out = plan.finalize()
    plan.close()
    a, e = out["S4"][0], out["S4_err"][0]
    # 1e-5 of the peak as for every FP32 path; T = 8: the terms of Eq. 85 cancel strongly
    tol = 2e-5 if T == 8 else 1e-5
    assert np.max(np.abs(a - ref["S4"])) <= tol * np.max(np.abs(ref["S4"]))
    er = ref["S4_err"].reshape(e.shape)
    assert np.max(np.abs(e - er)) <= 1e-4 * np.max(er)
    assert np.array_equal(a, a.T)
