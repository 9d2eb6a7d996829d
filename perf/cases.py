"""What the imager is timed on: the calls its users make, over the sizes they make them at.

Four kinds of work, each through the package's public entry points:

* ``bounds``  a new sample covariance, its dirty image and its MVDR bound
              (the quick-look images of an observation, and the first step
              of every solve);
* ``ops``     one forward product Psi x and one adjoint Psi^H u on device
              tensors, queued without a host wait: what an iterative method
              written by the user (its own LSQR, CLEAN, ...) calls per step;
* ``image``   a new covariance and its bounded least-squares image, alone or
              (``jobs`` > 1) as a batch of frequency channels;
* ``ls``      the unconstrained WLS image, every pixel free.

Data follow the model of the paper's Sec. II: point sources on the grid
(lognormal powers), an array in a disk, N time samples, a signal-to-noise
ratio near 0 dB per antenna.  A state holds what a program keeps between
images (the context: geometry, steering tables, buffers) and the inputs of
the next pass; the covariance is handed over anew in every pass.
"""
from __future__ import annotations

import math

import torch

import paper_1505_01348_gb300 as G

PRECISION = {"fp32": G.PREC_FP32, "f16x3": G.PREC_F16X3, "bf16x3": G.PREC_BF16X3}
COST = {"pwls": G.COST_PWLS, "ls": G.COST_LS}
KAPPA = 6.0


def listed():
    return [
        # the smallest image: a 16-antenna station, host arrays in and out
        {"name": "image_p16_32x32", "kind": "image", "p": 16, "n_l": 32, "n_m": 32, "sources": 5, "N": 1000,
         "precision": "f16x3", "cost": "pwls", "max_outer": 0, "jobs": 1, "host": True},
        # one frequency channel of a 48-antenna array, the grid not square
        {"name": "image_p48_96x80", "kind": "image", "p": 48, "n_l": 96, "n_m": 80, "sources": 10, "N": 10000,
         "precision": "f16x3", "cost": "pwls", "max_outer": 0, "jobs": 1, "host": False},
        # a 100-antenna station (the size of the paper's simulations)
        {"name": "image_p100_64x64", "kind": "image", "p": 100, "n_l": 64, "n_m": 64, "sources": 8, "N": 1000,
         "precision": "f16x3", "cost": "pwls", "max_outer": 0, "jobs": 1, "host": False},
        # the first passes of the largest workload (six clusters of 48 antennas)
        {"name": "image_p288_256x256", "kind": "image", "p": 288, "n_l": 256, "n_m": 256, "sources": 50, "N": 10000,
         "precision": "f16x3", "cost": "pwls", "max_outer": 200, "jobs": 1, "host": False},
        # channels of one observation in one call, arrays of three sizes,
        # with a cap on the passes as a real-time program sets it
        {"name": "batch_16_channels", "kind": "image", "p": 48, "n_l": 64, "n_m": 64, "sources": 10, "N": 10000,
         "precision": "f16x3", "cost": "pwls", "max_outer": 300, "jobs": 16, "host": False},
        # quick-look images: a 64-antenna array, the largest array, and the
        # default arithmetic (FP32 on CUDA cores)
        {"name": "bounds_p64_128x128", "kind": "bounds", "p": 64, "n_l": 128, "n_m": 128, "sources": 20, "N": 10000,
         "precision": "f16x3", "host": False},
        {"name": "bounds_p288_256x256", "kind": "bounds", "p": 288, "n_l": 256, "n_m": 256, "sources": 50, "N": 10000,
         "precision": "f16x3", "host": False},
        {"name": "bounds_p128_100x90_fp32", "kind": "bounds", "p": 128, "n_l": 100, "n_m": 90, "sources": 10,
         "N": 2000, "precision": "fp32", "host": True},
        # the operator pair: small and odd, the widest streamed operand on a
        # large grid, and beyond it
        {"name": "ops_p45_61x47", "kind": "ops", "p": 45, "n_l": 61, "n_m": 47, "sources": 5, "precision": "f16x3"},
        {"name": "ops_p256_512x512", "kind": "ops", "p": 256, "n_l": 512, "n_m": 512, "sources": 50,
         "precision": "f16x3"},
        {"name": "ops_p330_256x256", "kind": "ops", "p": 330, "n_l": 256, "n_m": 256, "sources": 50,
         "precision": "f16x3"},
        # the WLS image of a 128-antenna array, run to convergence
        {"name": "ls_p128_72x64", "kind": "ls", "p": 128, "n_l": 72, "n_m": 64, "sources": 20, "N": 10000,
         "precision": "f16x3", "cost": "pwls", "maxit": 100},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["bounds", "ops", "ops", "image", "ls"])
    p = _log_int(rng, 10, 384)
    precision = rng.choice(["f16x3", "f16x3", "f16x3", "bf16x3", "fp32"])
    if kind == "bounds":
        # CUDA cores (and the FP32 default) on the sizes where they are usable
        p = min(p, 288) if precision == "fp32" else p
        top = 128 if precision == "fp32" else 300
        return {"kind": kind, "p": p, "n_l": _log_int(rng, 20, top), "n_m": _log_int(rng, 20, top),
                "sources": rng.randint(1, 40), "N": 10 * p + rng.randint(1, 9000), "precision": precision,
                "host": rng.random() < 0.5}
    if kind == "ops":
        p, top = (min(p, 128), 128) if precision == "fp32" else (p, 400)
        return {"kind": kind, "p": p, "n_l": _log_int(rng, 20, top), "n_m": _log_int(rng, 20, top),
                "sources": rng.randint(1, 40), "precision": precision}
    if kind == "ls":
        p = max(64, min(p, 256))
        return {"kind": kind, "p": p, "n_l": _log_int(rng, 16, p * 3 // 5), "n_m": _log_int(rng, 16, p * 3 // 5),
                "sources": rng.randint(2, 30), "N": 10 * p + rng.randint(1, 9000),
                "precision": "bf16x3" if precision == "bf16x3" else "f16x3", "cost": rng.choice(["pwls", "ls"]),
                "maxit": 10 * rng.randint(6, 12)}
    wide = p > 64
    top = 128 if wide else 80
    return {"kind": "image", "p": p, "n_l": _log_int(rng, 20, top), "n_m": _log_int(rng, 20, top),
            "sources": rng.randint(2, 12), "N": 10 * p + rng.randint(1, 9000),
            "precision": "f16x3" if wide else precision,
            "cost": rng.choice(["pwls", "pwls", "ls"]), "max_outer": 100, "jobs": rng.choice([1, 1, 3]),
            "host": rng.random() < 0.3}


# ---------------------------------------------------------------- inputs
def _geometry(p, n_l, n_m, gen):
    """Antennas in a disk (radius grown with their number), pixel grid on [-0.5, 0.5]^2."""
    radius = 10.0 if p <= 32 else 50.0 if p <= 128 else 200.0
    r = radius * torch.sqrt(torch.rand(p, generator=gen, dtype=torch.float64))
    th = 2.0 * math.pi * torch.rand(p, generator=gen, dtype=torch.float64)
    ant = torch.stack([r * torch.cos(th), r * torch.sin(th), torch.zeros(p, dtype=torch.float64)], dim=1)
    return ant, torch.linspace(-0.5, 0.5, n_l, dtype=torch.float64), torch.linspace(-0.5, 0.5, n_m, dtype=torch.float64)


def _steering(ant, l, m, lam, idx):
    """Columns a_i (p x len(idx)) of the steering matrix, complex128 on the GPU."""
    n_l = l.shape[0]
    u = l.cuda()[idx % n_l]
    v = m.cuda()[torch.div(idx, n_l, rounding_mode="floor")]
    a = ant.cuda()
    ph = (a[:, 0:1] * u[None, :] + a[:, 1:2] * v[None, :]) / lam
    ph = -2.0 * math.pi * (ph - torch.round(ph))
    return torch.polar(torch.full_like(ph, a.shape[0] ** -0.5), ph)


def _sky(case, gen):
    Q = case["n_l"] * case["n_m"]
    idx = torch.randperm(Q, generator=gen)[: case["sources"]].cuda()
    power = torch.exp(torch.randn(case["sources"], generator=gen, dtype=torch.float64)).cuda()
    return idx, power


def _covariance(ant, l, m, lam, idx, power, N, gen):
    """Sample covariance of N snapshots of the sources in white noise (0 dB per antenna)."""
    p = ant.shape[0]
    A = _steering(ant, l, m, lam, idx)
    noise = float(power.sum()) / p

    def normal(rows):
        z = torch.randn(rows, N, 2, generator=gen, dtype=torch.float64, device="cuda") * math.sqrt(0.5)
        return torch.view_as_complex(z)

    Y = (A * torch.sqrt(power)) @ normal(idx.shape[0]) + math.sqrt(noise) * normal(p)
    R = Y @ Y.conj().T / N
    return 0.5 * (R + R.conj().T)


def _jobs(case, seed):
    """(ant, l, m, lam, R, N) of every job of a case; R in column-major order on the GPU."""
    gen = torch.Generator().manual_seed(int(seed))
    dgen = torch.Generator(device="cuda").manual_seed(int(seed))
    jobs = case.get("jobs", 1)
    sizes = [case["p"], case["p"] * 4 // 3, case["p"] * 2]
    out = []
    for c in range(jobs):
        p = min(sizes[c % 3], 384) if jobs > 1 else case["p"]
        ant, l, m = _geometry(p, case["n_l"], case["n_m"], gen)
        lam = 1.0 + 0.5 * c / max(jobs - 1, 1)
        idx, power = _sky(case, gen)
        N = max(case["N"], 5 * p)
        R = _covariance(ant, l, m, lam, idx, power, N, dgen)
        out.append((ant, l, m, lam, R, N))
    return out


def _imager(case, ant, l, m, lam):
    kw = {"precision": PRECISION[case["precision"]], "kappa": KAPPA}
    if "cost" in case:
        kw["cost"] = COST[case["cost"]]
    if case.get("max_outer"):
        kw["max_outer"] = case["max_outer"]
    return G.Imager(ant.numpy(), l.numpy(), m.numpy(), lam, **kw)


def _matrix(R, host):
    """A p x p matrix as the package takes it: a column-major host array or device tensor."""
    return R.cpu().numpy().T.copy().T if host else R.T.contiguous().T


def _out(Q, host):
    return None if host else torch.empty(Q, dtype=torch.float64, device="cuda")


def _ops_inputs(case, seed):
    """x (pixel powers) and a Hermitian U (the residual of that sky against another)."""
    gen = torch.Generator().manual_seed(int(seed))
    ant, l, m = _geometry(case["p"], case["n_l"], case["n_m"], gen)
    Q = case["n_l"] * case["n_m"]
    x = 0.01 * torch.rand(Q, generator=gen, dtype=torch.float64).cuda()
    idx, power = _sky(case, gen)
    x[idx] += power
    other, weight = _sky(case, gen)
    A, B = _steering(ant, l, m, 1.0, idx), _steering(ant, l, m, 1.0, other)
    U = (A * power) @ A.conj().T - (B * weight) @ B.conj().T
    U = 0.5 * (U + U.conj().T) + 0.01 * torch.eye(case["p"], dtype=torch.complex128, device="cuda")
    return ant, l, m, x, U


def prepare(case, seed):
    Q = case["n_l"] * case["n_m"]
    if case["kind"] == "ops":
        ant, l, m, x, U = _ops_inputs(case, seed)
        p = case["p"]
        state = {"case": case, "im": _imager(case, ant, l, m, 1.0), "x": x, "U": _matrix(U, False),
                 "K": torch.empty(p, p, dtype=torch.complex128, device="cuda"), "y": _out(Q, False)}
        torch.cuda.synchronize()
        return state
    host = bool(case.get("host"))
    jobs = _jobs(case, seed)
    state = {"case": case, "ims": [_imager(case, *j[:4]) for j in jobs], "R": [_matrix(j[4], host) for j in jobs],
             "N": [j[5] for j in jobs]}
    for name in ("dirty", "bound", "sigma"):
        state[name] = [_out(Q, host) for _ in jobs]
    # the inputs were made on another stream than the contexts'
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "ops":
        im = state["im"]
        return {"K": im.psi(state["x"], state["K"], wait=False), "y": im.psi_adj(state["U"], state["y"], wait=False)}
    ims = state["ims"]
    for im, R, N in zip(ims, state["R"], state["N"]):
        im.set_covariance(R, N)
    if case["kind"] == "bounds":
        return {"dirty": ims[0].dirty(state["dirty"][0]), "bound": ims[0].mvdr_bound(state["bound"][0])}
    if case["kind"] == "ls":
        sigma, info = ims[0].ls_image(maxit=case["maxit"], out=state["sigma"][0])
        return {"sigma": sigma, "iterations": info.lsqr_iters}
    if len(ims) > 1:
        sigma, infos = G.solve_batch(ims, None if case["host"] else state["sigma"])
        return {"sigma": sigma, "passes": [i.outer for i in infos]}
    dirty = ims[0].dirty(state["dirty"][0])
    bound = ims[0].mvdr_bound(state["bound"][0])
    sigma, info = ims[0].solve(state["sigma"][0])
    return {"dirty": dirty, "bound": bound, "sigma": sigma, "passes": info.outer, "free": info.n_free}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes of the inputs and outputs, and flops of the definitions: 4 p^2 per pixel for Psi, 8 p^2 for
    Psi^H, 16/3 p^3 for the Cholesky factor and its inverse.  A solve cannot do with fewer gradients than
    sources: each is found by one."""
    if case["kind"] == "ops":
        p, Q = case["p"], case["n_l"] * case["n_m"]
        return {"bytes": 2 * 16 * p * p + 2 * 8 * Q, "flops": 12.0 * p * p * Q}
    jobs = case.get("jobs", 1)
    sizes = [case["p"], case["p"] * 4 // 3, case["p"] * 2]
    bytes_, flops = 0, 0.0
    for c in range(jobs):
        p = min(sizes[c % 3], 384) if jobs > 1 else case["p"]
        Q = case["n_l"] * case["n_m"]
        images = {"bounds": 2, "ls": 1}.get(case["kind"], 3 if jobs == 1 else 1)
        bytes_ += 16 * p * p + 8 * Q * images
        flops += 16.0 * p * p * Q + 16.0 / 3.0 * p ** 3
        if case["kind"] == "ls":
            flops += 12.0 * p * p * Q * case["maxit"]
        elif case["kind"] == "image":
            flops += 8.0 * p * p * Q * min(case["sources"], case["max_outer"] or case["sources"])
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64-bit values
def _adjoint64(A, U):
    return (A.conj() * (U @ A)).real.sum(dim=0)


def _lsqr64(A, R, pwls, maxit, tol):
    """Paige-Saunders LSQR in 64 bits on M = W Psi D^-1 (PWLS) or Psi, stopping tests every 10 iterations."""
    p = A.shape[0]
    if pwls:
        Li = torch.linalg.inv(torch.linalg.cholesky(R))
        C = Li @ A
        scale = (C.abs() ** 2).sum(dim=0) ** -2
        u = torch.eye(p, dtype=A.dtype, device=A.device)
    else:
        C, u = A, R.clone()
        scale = torch.ones(A.shape[1], dtype=torch.float64, device=A.device)
    beta = u.norm()
    u = u / beta
    v = scale * _adjoint64(C, u)
    alpha = v.norm()
    v = v / alpha
    w, x = v.clone(), torch.zeros_like(v)
    bnorm, phibar, rhobar, anorm2 = beta, beta, alpha, 0.0
    for it in range(1, maxit + 1):
        u = (C * (scale * v)) @ C.conj().T - alpha * u
        beta = u.norm()
        u = u / beta
        anorm2 = anorm2 + alpha ** 2 + beta ** 2
        v = scale * _adjoint64(C, u) - beta * v
        alpha = v.norm()
        v = v / alpha
        rho = torch.sqrt(rhobar ** 2 + beta ** 2)
        c, s = rhobar / rho, beta / rho
        phi, phibar = c * phibar, s * phibar
        x = x + (phi / rho) * w
        w = v - (s * alpha / rho) * w
        rhobar = -c * alpha
        if it % 10 == 0:
            anorm = anorm2 ** 0.5
            if phibar <= tol * bnorm + tol * anorm * x.norm() or alpha * c.abs() <= tol * anorm:
                break
    return scale * x


def exact(case, seed):
    Q = case["n_l"] * case["n_m"]
    idx = torch.arange(Q, device="cuda")
    if case["kind"] == "ops":
        ant, l, m, x, U = _ops_inputs(case, seed)
        A = _steering(ant, l, m, 1.0, idx)
        # K is column-major in the tensor's memory: its rows are K's columns
        return {"K": ((A * x) @ A.conj().T).T.contiguous(), "y": _adjoint64(A, U)}
    jobs = _jobs(case, seed)
    if len(jobs) > 1:
        return None
    ant, l, m, lam, R, N = jobs[0]
    A = _steering(ant, l, m, lam, idx)
    if case["kind"] == "ls":
        # Before convergence the iterates of a 32-bit and a 64-bit Lanczos process part by percents, whatever
        # the products' accuracy: only a determined problem run to its end has a value to compare with.
        if Q > 0.3 * case["p"] ** 2 or case["maxit"] < 60:
            return None
        # a different count of iterations would be another image of the same tolerance
        return {"sigma": _lsqr64(A, R, case["cost"] == "pwls", case["maxit"], 1e-6), "iterations": None}
    out = {"dirty": _adjoint64(A, R), "bound": 1.0 / _adjoint64(A, torch.linalg.inv(R))}
    if case["kind"] == "image":
        # the active set is a sequence of strict comparisons: where two candidates are within rounding of
        # each other either is a correct step, so the image has no value apart from the decisions taken
        out.update(sigma=None, passes=None, free=None)
    return out
