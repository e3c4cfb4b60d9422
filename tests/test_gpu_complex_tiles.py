"""Complex-signal spectra where the tiles and chunks of the kernels can go wrong: planes
of several 32 x 64 tiles and less than one, a segment longer than a chunk of 8 frames and
not a multiple of it, runs of more groups than one float32 sum takes, and the first row
and column of the T x T plane, each stored twice.  Against the oracle; float32 sums of at
most 64 groups of m frames leave a rounding of some sqrt(64 m) 2^-24 of a point's terms,
below 1e-5 of the peak for m <= 17, and ten times that for a standard error.
"""
import numpy as np
import pytest

import oracle
from test_gpu_complex import P, check, gpu_records, signals

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,m,G,shift", [(8, 4, 3000, 1), (64, 17, 24, -70), (128, 9, 40, 0),
                                         (256, 5, 14, 95)])
def test_tiles_and_chunks(T, m, G, shift):
    real, z = signals(T, m, G, seed=3 * T + m)
    s2 = [((0, False), (1, True))]
    s3 = [((0, False), (1, False), (0, True)), ((1, True), (1, False), (0, False))]
    s4 = [((0, False), (1, True), (1, False), (0, True))]
    ref = oracle.complex_polyspectra(z, T, 0.5, m, s2_combos=s2, s3_combos=s3, s4_combos=s4,
                                     s4_shift=shift)
    mod = P()
    plan = mod.Plan(channels=4, T=T, dt=0.5, m=m, orders=(2,), combos=[(2, 0, 0, -1, -1)])
    recs = gpu_records(s2 + s3 + s4)
    mod.ss_set_complex(plan.handle, recs, shift)
    plan.accumulate(torch.from_numpy(real).cuda())
    got = plan.complex_spectra(recs)
    plan.close()
    keys = [("S2", c) for c in s2] + [("S3", c) for c in s3] + [("S4", c) for c in s4]
    for key, g in zip(keys, got):
        check(g, ref[key], str(key[0]))
    s4got = np.asarray(got[-1][0])
    assert np.array_equal(s4got[0], s4got[-1]) and np.array_equal(s4got[:, 0], s4got[:, -1])
