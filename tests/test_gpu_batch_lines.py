"""A lock-step batch large enough that its launches take other kernels than a
job alone does, against the jobs alone, bit for bit.

A launch of few tile pairs evaluates the LM step in the short form and solves
on one cluster per job; a batch goes over to the general forms.  Jobs of 70
stations have 15 tile pairs: 24 of them make 360, above the short form's line
of two blocks per SM, and 24 clusters of 16 CTAs more than the GPU holds.  Of
20 stations (3 pairs, 3 tile rows) 30 jobs stay below the first line and cross
the second (30 clusters of 8 CTAs), and 110 cross both.  In float64 200 jobs have
more blocks of the factorisation than the GPU holds."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402
from paper_1910_13908_gb300 import synth  # noqa: E402


def _job(N, T, F, K, seed, prec):
    spec = synth.JobSpec(N=N, T=T, F=F, K=K, S=4, f_lo=140e6, f_hi=160e6, seed=seed)
    shp = sc.Shape(N, T, F, K, spec.S)
    uvw, freqs = torch.as_tensor(synth.station_uvw(spec)).cuda(), torch.as_tensor(synth.freqs(spec)).cuda()
    sky, ws = sc.DeviceSky.from_synth(synth.sky(spec)), sc.workspace(shp, prec)
    C = sc.predict_coherencies(shp, uvw, freqs, sky, prec, ws)
    J = torch.as_tensor(synth.jones_true(spec)).to("cuda", C.dtype)
    p, q = torch.triu_indices(N, N, 1, device="cuda")
    V = sum(C[k][..., None, None] * (J[k][p] @ J[k][q].mH)[None, :, None] for k in range(K))
    noise = torch.Generator(device="cuda").manual_seed(seed)
    V = V + 0.01 * torch.randn(V.shape, generator=noise, dtype=V.dtype, device="cuda")
    return sc.Job(shape=shp, uvw=uvw, freqs=freqs, sky=sky, V=V.contiguous(),
                  jones=torch.as_tensor(synth.identity_jones(K, N)).cuda(),
                  costs=torch.zeros(K, dtype=torch.float64, device="cuda"), ws=ws, stream=torch.cuda.current_stream())


@pytest.mark.parametrize("n_jobs,N,prec", [(24, 70, "mixed"), (30, 20, "mixed"), (110, 20, "mixed"), (24, 70, "fp64"),
                                            (200, 20, "fp64")])
def test_large_lockstep_batch_equals_jobs_alone(n_jobs, N, prec):
    prec = sc.SC_MIXED if prec == "mixed" else sc.SC_FP64
    shapes = [(N, 1 + i % 7, 1 + i % 3, 2, 100 + i) for i in range(n_jobs)]
    batch, alone = [_job(*s, prec) for s in shapes], [_job(*s, prec) for s in shapes]
    sc.calibrate_batched(batch, prec, sc.batched_workspace(batch, prec), n_em=1, n_lm=5)
    for j in alone:
        sc.calibrate_sage(j.shape, j.uvw, j.freqs, j.sky, j.V, j.jones, prec, j.ws, n_em=1, n_lm=5, costs=j.costs)
    torch.cuda.synchronize()
    for i, (a, b) in enumerate(zip(batch, alone)):
        assert torch.equal(a.jones, b.jones), i
        assert torch.equal(a.costs, b.costs), i
        assert sc.device_status(a.ws) == 0
