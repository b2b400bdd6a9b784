"""Which kernel solves for a job that shares the device.

A thread-block cluster waits long for its multiprocessors while other streams'
factorisations hold them, so a job whose factorisation is capped (the caller's
max_ctas, a batch on streams) solves without one; the bands of a consensus keep
it.  The kernels that ran are read from the profiler's trace; the results are the
same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1910_13908_gb300 import sagecal as sc  # noqa: E402
from paper_1910_13908_gb300 import synth  # noqa: E402


def _job(seed):
    spec = synth.JobSpec(N=40, T=2, F=1, K=1, S=4, f_lo=150e6, f_hi=150e6, seed=seed)
    shp = sc.Shape(spec.N, spec.T, spec.F, spec.K, spec.S)
    uvw, freqs = torch.as_tensor(synth.station_uvw(spec)).cuda(), torch.as_tensor(synth.freqs(spec)).cuda()
    sky, ws = sc.DeviceSky.from_synth(synth.sky(spec)), sc.workspace(shp, sc.SC_MIXED)
    C = sc.predict_coherencies(shp, uvw, freqs, sky, sc.SC_MIXED, ws)[0]
    J = torch.as_tensor(synth.jones_true(spec)[0]).to("cuda", C.dtype)
    p, q = torch.triu_indices(spec.N, spec.N, 1, device="cuda")
    V = (C[..., None, None] * (J[p] @ J[q].mH)[None, :, None]).contiguous()
    return sc.Job(shp, uvw, freqs, sky, V, torch.as_tensor(synth.identity_jones(1, spec.N)).cuda(),
                  torch.zeros(1, dtype=torch.float64, device="cuda"), ws, torch.cuda.Stream())


def _solvers(call):
    """Names of the solve kernels that ran in call()."""
    for _ in range(3):  # a process's first trace can come back empty
        torch.cuda.synchronize()
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        names = {e.key for e in prof.key_averages()}
        if any("k_chol" in n for n in names):
            return {"cluster" if "k_chol_solve_cluster" in n else "general" for n in names if "k_chol_solve" in n}
    pytest.skip("no kernel names from the profiler here")


def _sage(j, cap):
    j.jones = torch.as_tensor(synth.identity_jones(1, 40)).cuda()
    sc.calibrate_sage(j.shape, j.uvw, j.freqs, j.sky, j.V, j.jones, sc.SC_MIXED, j.ws, n_em=1, n_lm=4, costs=j.costs,
                      max_ctas=cap)


def test_a_capped_job_solves_without_a_cluster():
    j = _job(1)
    assert _solvers(lambda: _sage(j, 0)) == {"cluster"}
    alone = j.jones.clone(), j.costs.clone()
    assert _solvers(lambda: _sage(j, 38)) == {"general"}
    assert torch.equal(j.jones, alone[0]) and torch.equal(j.costs, alone[1])


@pytest.mark.parametrize("n_jobs,solver", [(1, "cluster"), (3, "general")])
def test_jobs_on_streams(n_jobs, solver):
    jobs = [_job(10 + i) for i in range(n_jobs)]

    def batch():
        for j in jobs:
            j.jones = torch.as_tensor(synth.identity_jones(1, 40)).cuda()
        sc.calibrate_batch(jobs, sc.SC_MIXED, n_em=1, n_lm=4)

    assert _solvers(batch) == {solver}
    for j in jobs:
        jones, costs = j.jones.clone(), j.costs.clone()
        _sage(j, 0)
        torch.cuda.synchronize()
        assert torch.equal(j.jones, jones) and torch.equal(j.costs, costs)


def test_concurrent_bands_keep_the_cluster():
    j, n_bands = _job(20), 3
    freqs = (j.freqs + 1e6 * torch.arange(n_bands, device="cuda", dtype=torch.float64)[:, None]).contiguous()
    V = j.V[None].repeat(n_bands, 1, 1, 1, 1, 1).contiguous()
    basis = torch.ones((n_bands, 1), dtype=torch.float64, device="cuda")
    out = {}

    def consensus(concurrent):
        jones = j.jones[None].repeat(n_bands, 1, 1, 1, 1).contiguous()
        ws = sc.consensus_workspace(j.shape, sc.SC_MIXED, concurrent)
        out[concurrent] = sc.calibrate_consensus(j.shape, j.uvw, freqs, j.sky, V, basis, jones, sc.SC_MIXED, ws, 1.0,
                                                 n_admm=2, n_em=1, n_lm=3)

    assert _solvers(lambda: consensus(n_bands)) == {"cluster"}
    assert _solvers(lambda: consensus(1)) == {"cluster"}
    assert all(torch.equal(a, b) for a, b in zip(out[n_bands], out[1]))
