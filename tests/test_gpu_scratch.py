"""A device batch so large that the float32 operand image beside the spectra exceeds the
GPU's memory, of which the spectra alone take 0.42: the plan takes fewer groups a batch.
One group a batch or nine, a small record's float32 sums over groups differ by rounding
alone, some 9 x 2^-24 of the spectrum's peak (1e-5 asked, as elsewhere).
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_batch_beyond_memory():
    import paper_2505_01231_gb300 as mod
    T, m = 1024, 10
    x = torch.from_numpy(synth.ar1_quadratic(T * m * 9, seed=5).astype(np.float32)).cuda()
    spectra = m * 528 * 8                    # bytes a group
    groups = int(0.42 * torch.cuda.mem_get_info()[0] / spectra)
    got = []
    for batch in (0, groups):
        plan = mod.Plan(channels=1, T=T, m=m, orders=(3, 4), precision="fp32")
        if batch:
            mod.ss_set_batch(plan.handle, batch)
        plan.accumulate(x)
        got.append(plan.finalize())
        plan.close()
    for key in got[0]:
        a, b = np.asarray(got[0][key]), np.asarray(got[1][key])
        assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(a)), key
