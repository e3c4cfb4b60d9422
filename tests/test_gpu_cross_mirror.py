"""S4 of several channels where the rows k < 0 are mirrored (first pair or second pair of
equal channels) beside combinations that are not, FP32 and on the tensor cores, below and
from the frame length on where the tensor-core tiles split (T = 256, the row k = M - 1 of
its own), two device batches, against the oracle on the whole grid.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COMBOS = [(0, 0, 1, 1), (0, 0, 0, 1), (0, 1, 1, 1), (1, 0, 2, 2), (0, 1, 0, 2), (2, 2, 2, 2)]


@pytest.mark.parametrize("precision", ["fp32", "fp16x3", "tf32x3"])
@pytest.mark.parametrize("T,m,G", [(16, 5, 7), (128, 9, 5), (256, 5, 6), (512, 4, 3)])
def test_mirrored_combinations_match_the_oracle(T, m, G, precision):
    import paper_2505_01231_gb300 as mod
    C = 3
    z = synth.multichannel_shared(C, T * m * G + 7, seed=T + m)
    ref = oracle.cross_polyspectra(z, T, 0.5, m, s4_combos=COMBOS, group_chunk=8)
    plan = mod.Plan(channels=C, T=T, dt=0.5, m=m, orders=(4,), precision=precision,
                    combos=[(4,) + c for c in COMBOS])
    mod.ss_set_batch(plan.handle, 4)
    plan.accumulate(torch.from_numpy(z).cuda())
    out = plan.finalize()
    plan.close()
    for i, c in enumerate(COMBOS):
        v, e = ref[("S4", c)]
        assert np.max(np.abs(out["S4"][i].reshape(v.shape) - v)) <= 1e-5 * np.max(np.abs(v)), c
        e = e.reshape(out["S4_err"][i].shape)
        assert np.max(np.abs(out["S4_err"][i] - e)) <= 1e-4 * np.max(e), c
