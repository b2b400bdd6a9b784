"""Mixed prediction at the edges of its tiles, against the FP64 oracle.

The contraction takes 64x64 station tiles, sources in steps of eight (scalar)
or sixteen (full Stokes; 32x32 tiles) through two buffers, and ranges of
(timeslot, channel) pairs; the station phasors take 128 stations, ranges of
timeslots and 32 channels at a time.  Sizes lie on, one below and one above
those edges.  Tolerance: 1e-5 of the cluster's flux scale sum_s S_s(f), the
bound of the mixed path (float32 phasors, float32 sums of at most 33 terms).
"""
import numpy as np
import pytest

import oracle as O
from paper_1910_13908_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402


def tdev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("N,T,F,counts", [(63, 2, 1, [1, 8, 16]), (64, 1, 2, [7, 15, 0]), (65, 3, 2, [9, 17]),
                                          (129, 2, 1, [33, 1]), (3, 1, 33, [8, 2]), (2, 1300, 1, [3])])
def test_mixed_prediction_at_tile_edges(full, N, T, F, counts):
    spec = synth.JobSpec(N=N, T=T, F=F, K=len(counts), S=max(counts), f_lo=140e6, f_hi=160e6, seed=N + F,
                         alpha=-0.7)
    uvw, f = synth.station_uvw(spec), synth.freqs(spec)
    if full:
        sky = synth.sky_pol(spec, sources_per_cluster=counts, frac_extended=0.5, max_circ_pol=0.1)
        amp, ref = np.abs(sky.I) + np.abs(sky.Q) + np.abs(sky.U) + np.abs(sky.V), O.predict_sky_full(uvw, f, sky)
    else:
        sky = synth.sky(spec, counts)
        amp, ref = sky.flux, O.predict_sky(uvw, f, sky)
    shp = sc.Shape(N, T, F, len(counts), max(counts))
    ws = sc.workspace(shp, sc.SC_MIXED)
    predict = sc.predict_coherencies_full if full else sc.predict_coherencies
    dev = (sc.DeviceSkyFull if full else sc.DeviceSky).from_synth(sky)
    got = predict(shp, tdev(uvw), tdev(f), dev, sc.SC_MIXED, ws).cpu().numpy()
    for k in range(len(counts)):
        a, b = int(sky.offsets[k]), int(sky.offsets[k + 1])
        scale = (amp[a:b, None] * (f[None, :] / sky.f0) ** sky.alpha[a:b, None]).sum(0)  # [F]
        err = np.abs(got[k] - ref[k]).reshape(T, -1, F, 4 if full else 1)
        assert np.all(err <= 1e-5 * scale[None, None, :, None]), (k, err.max())
    assert sc.device_status(ws) == 0
