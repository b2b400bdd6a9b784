"""The work a user of this framework has it do, as cases that can be timed.

Every case goes through the Python binding of the C ABI
(paper_1910_13908_gb300.sagecal), with the inputs a calibration program has in
hand on the GPU: station coordinates, a sky model, visibilities, Jones
matrices and the caller-owned workspace.  Inputs are drawn from the seed with
the distributions of paper_1910_13908_gb300.synth (stations in a 3 km disc,
fluxes log-uniform in 0.1..10 Jy, Jones I + CN(0, 0.1), noise 0.01 Jy); the
visibilities are simulated here with torch, not with the library.

Kinds of work:
  residual      sc.residual: one cluster's residual and cost
  solve         sc.solve_cluster: Levenberg-Marquardt on one cluster
  sage          sc.calibrate_sage: a whole calibration
  batched       sc.calibrate_batched: many jobs of uneven length in lock step
  cholesky      sc.cholesky_solve: the dense solve on its own
  predict       sc.predict_coherencies: point sources
  predict_full  sc.predict_coherencies_full: polarised, Gaussian sources
  residual_all  sc.residual_all: the output after calibration
"""
import math

import numpy as np
import torch

from paper_1910_13908_gb300 import sagecal as sc
from paper_1910_13908_gb300 import synth

DEV = "cuda"


# ---- the cases -----------------------------------------------------------------


def listed():
    return [
        # the smallest call: the residual of one direction of a 64-station sub-band, as a monitor asks for it
        dict(name="residual_64", kind="residual", prec="mixed", N=64, T=10, F=1, S=20),
        # one direction of a LOFAR-like array solved from scratch: latency and launches
        dict(name="solve_64", kind="solve", prec="mixed", N=64, T=10, F=1, S=20, n_lm=10),
        # the plain float64 calibration of the same array (the first workload of the study)
        dict(name="sage_64_fp64", kind="sage", prec="fp64", N=64, T=10, F=1, K=1, S=20, n_em=1, n_lm=10),
        # a whole mixed-precision calibration: 128 stations, 10 directions, 8 channels, 3 sweeps
        dict(name="sage_128", kind="sage", prec="mixed", N=128, T=20, F=8, K=10, S=25, n_em=3, n_lm=10),
        # float64 on a mid-size array whose matrix is no multiple of the tile
        dict(name="solve_150_fp64", kind="solve", prec="fp64", N=150, T=10, F=2, S=25, n_lm=5),
        # a ragged station and channel count (order 2408)
        dict(name="solve_301", kind="solve", prec="mixed", N=301, T=7, F=3, S=50, n_lm=10),
        # one direction at SKA1-LOW scale (order 4096): the step the 512-station calibration repeats
        dict(name="solve_512", kind="solve", prec="mixed", N=512, T=10, F=4, S=100, n_lm=10),
        # sub-bands of 256 stations and uneven length calibrated side by side
        dict(name="batched_256", kind="batched", prec="mixed", jobs=16, N=256, F=1, K=2, S=50, n_em=1, n_lm=5),
        # the dense solve alone at an order above the solver's, with a ragged last tile
        dict(name="cholesky_6000", kind="cholesky", prec="mixed", n=6000),
        # model coherencies at SKA1-LOW scale
        dict(name="predict_512", kind="predict", prec="mixed", N=512, T=10, F=4, K=8, S=100),
        # polarised, partly extended sky
        dict(name="predict_full_256", kind="predict_full", prec="mixed", N=256, T=10, F=4, K=5, S=50),
        # every direction removed from the data, corrected towards one: what imaging receives
        dict(name="residual_all_512", kind="residual_all", prec="mixed", N=512, T=10, F=4, K=40, S=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "solve", "solve", "solve", "sage", "sage", "batched", "cholesky", "predict",
                       "predict_full", "residual_all"])
    T, F, S = rng.randint(1, 20), rng.randint(1, 8), _log(rng, 5, 100)
    if kind == "residual":
        return dict(kind=kind, prec=rng.choice(["mixed", "mixed", "fp64"]), N=_log(rng, 16, 256), T=T, F=F, S=S)
    if kind == "solve":
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        return dict(kind=kind, prec=prec, N=_log(rng, 16, 512 if prec == "mixed" else 150), T=rng.randint(1, 10),
                    F=rng.randint(1, 4), S=S, n_lm=rng.randint(2, 10))
    if kind == "sage":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        N = _log(rng, 16, 128 if prec == "mixed" else 64)
        return dict(kind=kind, prec=prec, N=N, T=T, F=F, K=rng.randint(1, 6), S=min(S, 40), n_em=rng.randint(1, 2),
                    n_lm=rng.randint(3, 10))
    if kind == "batched":
        return dict(kind=kind, prec="mixed", jobs=_log(rng, 2, 16), N=_log(rng, 32, 256), F=rng.randint(1, 2),
                    K=rng.randint(1, 2), S=min(S, 50), n_em=1, n_lm=rng.randint(2, 5))
    if kind == "cholesky":
        return dict(kind=kind, prec="mixed", n=_log(rng, 64, 6000))
    if kind == "predict":
        return dict(kind=kind, prec="mixed", N=_log(rng, 32, 512), T=rng.randint(1, 10), F=rng.randint(1, 4),
                    K=rng.randint(1, 8), S=S)
    if kind == "predict_full":
        return dict(kind=kind, prec="mixed", N=_log(rng, 32, 256), T=rng.randint(1, 10), F=rng.randint(1, 4),
                    K=rng.randint(1, 5), S=min(S, 50))
    return dict(kind=kind, prec="mixed", N=_log(rng, 32, 512), T=rng.randint(1, 10), F=rng.randint(1, 4),
                K=rng.randint(1, 40), S=min(S, 20))


# ---- inputs ----------------------------------------------------------------------


def _prec(case):
    return sc.SC_MIXED if case["prec"] == "mixed" else sc.SC_FP64


def _cdt(case):
    return torch.complex64 if case["prec"] == "mixed" else torch.complex128


def _spec(case, seed, T=None):
    F = case["F"]
    return synth.JobSpec(N=case["N"], T=case["T"] if T is None else T, F=F, K=case.get("K", 1), S=case["S"],
                         f_lo=140e6 if F > 1 else 150e6, f_hi=160e6 if F > 1 else 150e6,
                         alpha=-0.7 if F > 1 else 0.0, seed=int(seed) & 0x7FFFFFFF)


def _dev(a):
    return torch.as_tensor(a, device=DEV)


def _pairs(N):
    i = torch.triu_indices(N, N, 1, device=DEV)
    return i[0], i[1]


def _phasors(uvw, freqs, l, m):
    """exp(-2 pi i f/c (u l + v m + w (n - 1))) of every station, [T][F][S][N] complex128."""
    r2 = l * l + m * m
    nm1 = -r2 / (1.0 + torch.sqrt(1.0 - r2))
    path = torch.einsum("tnx,xs->tsn", uvw, torch.stack([l, m, nm1]))
    turns = path[:, None] * (freqs / synth.C_LIGHT)[None, :, None, None]
    turns = turns - torch.round(turns)
    return torch.polar(torch.ones_like(turns), -2.0 * math.pi * turns)


def _coherencies(uvw, freqs, sky, k, cdt):
    """[T][B][F] of cluster k, summed in cdt."""
    a, b = int(sky.offsets[k]), int(sky.offsets[k + 1])
    l, m, flux, al = (_dev(x[a:b]) for x in (sky.l, sky.m, sky.flux, sky.alpha))
    E = _phasors(uvw, freqs, l, m)
    Sf = flux[None] * (freqs[:, None] / sky.f0) ** al[None]  # [F][S]
    p, q = _pairs(uvw.shape[1])
    out = torch.empty((uvw.shape[0], p.numel(), freqs.numel()), dtype=cdt, device=DEV)
    for t in range(uvw.shape[0]):
        full = torch.einsum("fsp,fsq->fpq", (E[t] * Sf[:, :, None]).to(cdt), E[t].conj().to(cdt))
        out[t] = full[:, p, q].T
    return out


def _gains(J, cdt):
    """J_p J_q^H of every baseline, [B][2][2]."""
    p, q = _pairs(J.shape[0])
    Jc = J.to(cdt)
    return Jc[p] @ Jc[q].mH


def _observed(spec, uvw, freqs, sky, cdt, seed, C=None):
    """sum_k C_k J_p J_q^H + noise."""
    Jt = _dev(synth.jones_true(spec))
    V = None
    for k in range(spec.K):
        Ck = _coherencies(uvw, freqs, sky, k, cdt) if C is None else C[k]
        M = Ck[..., None, None] * _gains(Jt[k], cdt)[None, :, None]
        V = M if V is None else V + M
    rdt = torch.float32 if cdt == torch.complex64 else torch.float64
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return V + spec.sigma * torch.view_as_complex(torch.randn(V.shape + (2,), generator=g, dtype=rdt, device=DEV))


def _near_truth(spec, off=0.02):
    """Jones as a calibration hands them on: near the true ones."""
    z = synth.normal(spec.seed + 1, synth.TAG_JONES, 8 * spec.K * spec.N)
    d = (z[0::2] + 1j * z[1::2]).reshape(spec.K, spec.N, 2, 2) * off
    return _dev(synth.jones_true(spec) + d)


def _job(case, seed, T=None):
    spec = _spec(case, seed, T)
    uvw, freqs, sky = _dev(synth.station_uvw(spec)), _dev(synth.freqs(spec)), synth.sky(spec)
    return spec, uvw, freqs, sky


def _batch_slots(case, seed):
    """Timeslots of the jobs of a batch: 5..40, uneven."""
    return [int(t) for t in synth.uneven_time_chunks(case["jobs"], seed=int(seed) & 0x7FFFFFFF)]


def _spd(n, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    M = torch.randn((n, n), generator=g, device=DEV)
    A = M @ M.T / n
    A = 0.5 * (A + A.T)
    A.diagonal().add_(0.05)
    return A.contiguous(), torch.randn((n,), generator=g, dtype=torch.float64, device=DEV)


def prepare(case, seed):
    kind, prec, cdt = case["kind"], _prec(case), _cdt(case)
    if kind == "cholesky":
        A, b = _spd(case["n"], seed)
        return dict(kind=kind, prec=prec, A=A, b=b, ws=sc.cholesky_workspace(case["n"], prec))
    if kind == "batched":
        jobs, starts = [], []
        for i, T in enumerate(_batch_slots(case, seed)):
            spec, uvw, freqs, sky = _job(case, seed + 1000 * i, T)
            shape = sc.Shape(spec.N, spec.T, spec.F, spec.K, spec.S)
            J0 = _dev(synth.identity_jones(spec.K, spec.N))
            starts.append(J0)
            jobs.append(sc.Job(shape, uvw, freqs, sc.DeviceSky.from_synth(sky),
                               _observed(spec, uvw, freqs, sky, cdt, seed + i), J0.clone(),
                               torch.zeros(spec.K, dtype=torch.float64, device=DEV), sc.workspace(shape, prec),
                               torch.cuda.current_stream()))
        return dict(kind=kind, prec=prec, jobs=jobs, J0=starts, ws=sc.batched_workspace(jobs, prec),
                    opts=dict(n_em=case["n_em"], n_lm=case["n_lm"]))
    spec, uvw, freqs, sky = _job(case, seed)
    shape = sc.Shape(spec.N, spec.T, spec.F, spec.K, spec.S)
    state = dict(kind=kind, prec=prec, shape=shape, uvw=uvw, freqs=freqs)
    if kind == "predict":
        state["sky"] = sc.DeviceSky.from_synth(sky)
    elif kind == "predict_full":
        state["sky"] = sc.DeviceSkyFull.from_synth(synth.sky_pol(spec))
    elif kind == "sage":
        state.update(sky=sc.DeviceSky.from_synth(sky), V=_observed(spec, uvw, freqs, sky, cdt, seed),
                     J0=_dev(synth.identity_jones(spec.K, spec.N)),
                     opts=dict(n_em=case["n_em"], n_lm=case["n_lm"]))
    elif kind == "residual_all":
        C = torch.stack([_coherencies(uvw, freqs, sky, k, cdt) for k in range(spec.K)])
        state.update(C=C, V=_observed(spec, uvw, freqs, sky, cdt, seed, C), J=_near_truth(spec))
    else:  # residual, solve: one cluster
        C = _coherencies(uvw, freqs, sky, 0, cdt)
        state.update(C=C, V=_observed(spec, uvw, freqs, sky, cdt, seed, C[None]))
        if kind == "residual":
            state["J"] = _near_truth(spec)[0].contiguous()
        else:
            state.update(J0=_dev(synth.identity_jones(1, spec.N))[0].contiguous(), n_lm=case["n_lm"])
    state["ws"] = sc.workspace(shape, prec)
    return state


def run(state):
    kind, prec, ws = state["kind"], state["prec"], state["ws"]
    if kind == "cholesky":
        L, x = sc.cholesky_solve(state["A"].clone(), state["b"], prec, ws)
        return L.tril_(), x
    if kind == "batched":
        for job, J0 in zip(state["jobs"], state["J0"]):
            job.jones = J0.clone()
        sc.calibrate_batched(state["jobs"], prec, ws, **state["opts"])
        return [(job.jones, job.costs) for job in state["jobs"]]
    shape = state["shape"]
    if kind == "residual":
        return sc.residual(shape, state["V"], state["C"], state["J"], prec, ws)
    if kind == "solve":
        return sc.solve_cluster(shape, state["V"], state["C"], state["J0"].clone(), prec, ws, n_lm=state["n_lm"])
    if kind == "sage":
        return sc.calibrate_sage(shape, state["uvw"], state["freqs"], state["sky"], state["V"], state["J0"].clone(),
                                 prec, ws, **state["opts"])
    if kind == "predict":
        return sc.predict_coherencies(shape, state["uvw"], state["freqs"], state["sky"], prec, ws)
    if kind == "predict_full":
        return sc.predict_coherencies_full(shape, state["uvw"], state["freqs"], state["sky"], prec, ws)
    return sc.residual_all(shape, state["V"], state["C"], state["J"], prec, ws, corr=0)


def work(case):
    rs = 4 if case["prec"] == "mixed" else 8
    if case["kind"] == "cholesky":
        n = case["n"]  # the lower triangle read and written, the right-hand side and the solution
        return dict(bytes=rs * n * (n + 1) + 16 * n, flops=n ** 3 / 3 + 2 * n * n)
    N, F, K = case["N"], case["F"], case.get("K", 1)
    # a batch has 22.5 timeslots a job on average
    T, jobs = (22.5, case["jobs"]) if case["kind"] == "batched" else (case["T"], 1)
    B, P = N * (N - 1) // 2, 8 * N
    vis, c = T * B * F, 2 * rs  # visibilities of a job, bytes of one complex number
    lm = P ** 3 / 3 + 4 * P * P  # one LM step: factorisation and two substitutions
    pred = 8 * case["S"] * vis  # one cluster's coherencies
    jones = 128 * K * N
    if case["kind"] == "residual":
        return dict(bytes=vis * 9 * c + jones, flops=40 * vis)
    if case["kind"] == "solve":
        return dict(bytes=vis * 5 * c + 2 * jones, flops=60 * vis + case["n_lm"] * lm)
    if case["kind"] in ("sage", "batched"):
        steps = K * case["n_em"]
        return dict(bytes=jobs * (vis * 4 * c + 2 * jones),
                    flops=jobs * (K * pred + steps * (140 * vis + case["n_lm"] * lm)))
    if case["kind"] == "predict":
        return dict(bytes=K * vis * c, flops=K * pred)
    if case["kind"] == "predict_full":
        return dict(bytes=K * vis * 4 * c, flops=K * case["S"] * vis * 25)
    return dict(bytes=vis * (8 + K) * c + jones, flops=vis * (32 * K + 130))


# ---- the same in 64 bits, in plain torch -------------------------------------------------


class _Cluster:
    """One cluster's least-squares problem: data X [T][B][F][2][2], coherencies c [T][B][F]."""

    def __init__(self, X, c):
        self.S = X.abs().square().sum(dim=(0, 2, 3, 4))
        self.rho = (c.conj()[..., None, None] * X).sum(dim=(0, 2))
        self.W = c.abs().square().sum(dim=(0, 2))
        self.N = (1 + math.isqrt(1 + 8 * self.W.numel())) // 2
        self.p, self.q = _pairs(self.N)
        full = torch.zeros((self.N, self.N), dtype=torch.float64, device=DEV)
        full[self.p, self.q] = self.W
        self.full = full + full.T

    def evaluate(self, J):
        """cost, J^T r as [N][2][2] complex, H [N][2][2]"""
        G = J[self.p] @ J[self.q].mH
        cost = (self.S - 2.0 * (G.conj() * self.rho).sum(dim=(1, 2)).real
                + self.W * G.abs().square().sum(dim=(1, 2))).sum()
        r = self.rho - self.W[:, None, None] * G
        g = torch.zeros_like(J)
        g.index_add_(0, self.p, r @ J[self.q])
        g.index_add_(0, self.q, r.mH @ J[self.p])
        H = torch.einsum("so,oab->sab", self.full.to(J.dtype), J.mH @ J)
        return cost, g, H

    def matrix(self, J, H, mu):
        """J^T J + mu I, [8N][8N]: row (s, i, j, x), column (o, b, a, y)"""
        N = self.N
        Z = torch.einsum("so,sia,obj->sijoba", self.full.to(J.dtype), J, J)
        A = torch.stack([torch.stack([Z.real, Z.imag], -1), torch.stack([Z.imag, -Z.real], -1)], 3)
        # A: s i j x o b a y
        Hd = H.mT  # [s][j][a] = H[a][j]
        D = torch.stack([torch.stack([Hd.real, -Hd.imag], -1), torch.stack([Hd.imag, Hd.real], -1)], 2)
        s = torch.arange(N, device=DEV)
        for i in range(2):  # D: s j x a y
            A[s, i, :, :, s, i] += D
        A = A.reshape(8 * N, 8 * N)
        A.diagonal().add_(mu)
        return A


def _solve(X, c, J, n_lm, tau=1e-3, eps=1e-12):
    """Levenberg-Marquardt (Madsen, Nielsen & Tingleff 2004, Alg. 3.16) in float64."""
    P = _Cluster(X, c)
    cost, g, H = P.evaluate(J)
    vec = lambda z: torch.view_as_real(z.contiguous()).reshape(-1)  # noqa: E731
    top = lambda z: float(vec(z).abs().max())  # noqa: E731
    mu, nu, it = tau * float(torch.diagonal(H, dim1=1, dim2=2).real.abs().max()), 2.0, 0
    while it < n_lm and not top(g) <= eps * (1.0 + float(cost)):
        it += 1
        L, bad = torch.linalg.cholesky_ex(P.matrix(J, H, mu))
        rho = -1.0
        if int(bad) == 0:
            gv = vec(g)
            d = torch.cholesky_solve(gv[:, None], L)[:, 0]
            Jt = J + torch.view_as_complex(d.reshape(P.N, 2, 2, 2))
            pred = float((d * (mu * d + gv)).sum())
            ct, gt, Ht = P.evaluate(Jt)
            if pred > 0:
                rho = float(cost - ct) / pred
        if rho > 0:
            J, cost, g, H = Jt, ct, gt, Ht
            mu, nu = mu * max(1.0 / 3.0, 1.0 - (2.0 * rho - 1.0) ** 3), 2.0
        else:
            mu, nu = mu * nu, 2.0 * nu
    return J, cost


def _sage(V, C, J, n_em, n_lm):
    J, K = list(J), len(C)
    model = lambda k: C[k][..., None, None] * _gains(J[k], torch.complex128)[None, :, None]  # noqa: E731
    R = V - sum(model(k) for k in range(K))
    costs = [None] * K
    for _ in range(n_em):
        for k in range(K):
            X = R + model(k)
            J[k], costs[k] = _solve(X, C[k], J[k], n_lm)
            R = X - model(k)
    return torch.stack(J), torch.stack(costs)


def _full_coherencies(uvw, freqs, sky, k):
    """[T][B][F][2][2] of cluster k of a polarised sky, in complex128."""
    a, b = int(sky.offsets[k]), int(sky.offsets[k + 1])
    l, m, I, Q, U, Vs, al, maj, mnr, pa = (_dev(np.ascontiguousarray(getattr(sky, n)[a:b])) for n in sc.FULL_FIELDS)
    E = _phasors(uvw, freqs, l, m)
    Bm = torch.stack([torch.stack([I + Q + 0j, U + 1j * Vs], -1), torch.stack([U - 1j * Vs, I - Q + 0j], -1)], -2)
    Sf = (freqs[:, None] / sky.f0) ** al[None]
    p, q = _pairs(uvw.shape[1])
    sig = 1.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    out = torch.empty((uvw.shape[0], p.numel(), freqs.numel(), 2, 2), dtype=torch.complex128, device=DEV)
    for t in range(uvw.shape[0]):
        uv = uvw[t, p] - uvw[t, q]
        for f in range(freqs.numel()):
            u, v = uv[:, :1] * (freqs[f] / synth.C_LIGHT), uv[:, 1:2] * (freqs[f] / synth.C_LIGHT)
            ua = u * torch.sin(pa) + v * torch.cos(pa)
            ub = u * torch.cos(pa) - v * torch.sin(pa)
            G = torch.exp(-2.0 * math.pi ** 2 * ((sig * maj * ua) ** 2 + (sig * mnr * ub) ** 2))
            e = (E[t, f][:, p] * E[t, f][:, q].conj()).T * G * Sf[f]  # [B][S]
            out[t, :, f] = (e @ Bm.reshape(-1, 4)).reshape(-1, 2, 2)
    return out


def exact(case, seed):
    kind, c128 = case["kind"], torch.complex128
    if kind == "cholesky":
        A, b = _spd(case["n"], seed)
        L = torch.linalg.cholesky(A.double())
        return L, torch.cholesky_solve(b[:, None], L)[:, 0]
    if kind == "batched":
        out = []
        for i, T in enumerate(_batch_slots(case, seed)):
            spec, uvw, freqs, sky = _job(case, seed + 1000 * i, T)
            V = _observed(spec, uvw, freqs, sky, _cdt(case), seed + i).to(c128)
            C = [_coherencies(uvw, freqs, sky, k, c128) for k in range(spec.K)]
            out.append(_sage(V, C, _dev(synth.identity_jones(spec.K, spec.N)), case["n_em"], case["n_lm"]))
        return out
    spec, uvw, freqs, sky = _job(case, seed)
    if kind == "predict":
        return torch.stack([_coherencies(uvw, freqs, sky, k, c128) for k in range(spec.K)])
    if kind == "predict_full":
        pol = synth.sky_pol(spec)
        return torch.stack([_full_coherencies(uvw, freqs, pol, k) for k in range(spec.K)])
    if kind == "sage":
        V = _observed(spec, uvw, freqs, sky, _cdt(case), seed).to(c128)
        C = [_coherencies(uvw, freqs, sky, k, c128) for k in range(spec.K)]
        return _sage(V, C, _dev(synth.identity_jones(spec.K, spec.N)), case["n_em"], case["n_lm"])
    if kind == "residual_all":
        C = torch.stack([_coherencies(uvw, freqs, sky, k, _cdt(case)) for k in range(spec.K)])
        R, J = _observed(spec, uvw, freqs, sky, _cdt(case), seed, C).to(c128), _near_truth(spec)
        for k in range(spec.K):
            R = R - C[k].to(c128)[..., None, None] * _gains(J[k], c128)[None, :, None]
        cost = R.abs().square().sum()
        inv = torch.linalg.inv(J[0])
        p, q = _pairs(spec.N)
        return inv[p][None, :, None] @ R @ inv[q].mH[None, :, None], cost
    C = _coherencies(uvw, freqs, sky, 0, _cdt(case))
    V = _observed(spec, uvw, freqs, sky, _cdt(case), seed, C[None]).to(c128)
    if kind == "residual":
        R = V - C.to(c128)[..., None, None] * _gains(_near_truth(spec)[0], c128)[None, :, None]
        return R, R.abs().square().sum()
    J, cost = _solve(V, C.to(c128), _dev(synth.identity_jones(1, spec.N))[0], case["n_lm"])
    return J, cost, None
