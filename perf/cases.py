"""What a user of this library has it do, as timed cases.

Data of mixed-precision plans are complex64 (the scanner's type), of FP64 plans complex128 or complex64.

A case names an encoding (grid, trajectory, coils, off-resonance), how the plan is set up
(precision, Recon kept or implicit, residual, refinement steps) and one call pattern:

  oneshot   host arrays in, images out: Plan -> build -> apply -> close, all in one pass
  step      an existing plan is built again and applied to its frames (a new trajectory
            calibration per series; the benchmark's step)
  apply     a built plan reconstructs frames (one frame: the real-time loop; many: a series)
  batch     several uneven plans built and applied together, replayed from CUDA graphs
  serve     a burst of requests on a server whose plans are resident
  spectrum  eigenvalue decomposition of the Gram and a truncated reconstruction

prepare() makes the inputs from the seed alone (trajectory rotation, coil phases, off-resonance,
phantom, noise) with the synthetic generators of the package: k-space data are the continuous
Fourier transform of an ellipse phantom plus 1 % noise, never the discrete model.
"""
import math
import random

import numpy as np
import torch

from paper_2410_06129_gb300 import _lib as L
from paper_2410_06129_gb300 import synth
from paper_2410_06129_gb300.batch import Batch
from paper_2410_06129_gb300.plan import Plan
from paper_2410_06129_gb300.serve import Server

PREC = {"fp64": L.FP64, "bf16x6": L.MIXED_BF16X6, "bf16x3": L.MIXED_BF16X3}
RECON = {"store": L.RECON_STORE, "none": L.RECON_NONE}
DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
ELLIPSES = 10


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------
def _case(kind, nx, ny=0, nz=1, coils=1, traj="spiral", samples=0, b0=False, keep=1.0, prec="bf16x6",
          recon="none", frames=1, dtype="c64", iters=3, lam=1e-3):
    """nx x ny x nz grid (ny = 0: square); samples per coil and slice encoding; keep < 1: only that
    share of the voxels (an elliptical mask) is reconstructed."""
    ny = ny or nx
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, coils=coils, traj=traj, samples=samples or 2 * nx * ny, b0=b0,
                keep=keep, prec=prec, recon=recon, frames=frames, dtype=dtype, iters=iters, lam=lam)


def listed():
    return [
        # the plain FP64 workload, as a user's first script runs it: 32x32, one coil, one spiral of
        # 2048 samples, one complex128 frame, library defaults, host arrays to image
        dict(_case("oneshot", 32, samples=2048, prec="fp64", recon="store", dtype="c128", iters=1),
             name="oneshot fp64 32x32"),
        # FP64 multi-coil reconstruction with the explicit Recon of the library's defaults, built and
        # applied to a short series; an odd grid and a sample count that is no multiple of anything
        dict(_case("step", 37, coils=4, traj="radial", samples=2701, prec="fp64", recon="store", frames=13,
                   dtype="c128", iters=1), name="step fp64 37x37 4 coils"),
        # the real-time loop: one frame at a time through a plan built once (64x64, 8 coils)
        dict(_case("apply", 64, coils=8, frames=1, lam=1e-4), name="apply 64x64 8 coils 1 frame"),
        # a 64-frame series through the same encoding with the explicit Recon (the default of a mixed plan)
        dict(_case("apply", 64, coils=8, recon="store", frames=64, lam=1e-4), name="apply 64x64 8 coils Recon"),
        # the benchmark's step: factor-only build and 64 frames
        dict(_case("step", 64, coils=8, frames=64, lam=1e-4), name="step 64x64 8 coils"),
        # explicit Recon built and applied (workload sizes of the batched series), ragged everywhere
        dict(_case("step", 45, 51, coils=5, traj="radial", samples=5003, recon="store", frames=33),
             name="step 45x51 5 coils Recon"),
        # off-resonance: the reduced high-resolution radial workload (B0, no Toeplitz structure)
        dict(_case("step", 56, coils=8, traj="radial", samples=5600, b0=True, frames=16, lam=1e-4),
             name="step 56x56 8 coils B0"),
        # a masked 3D stack of spirals (in-vivo masks; the paper's 3D dataset class)
        dict(_case("step", 26, 22, 7, coils=3, samples=601, keep=0.7, frames=6),
             name="step 3D masked"),
        # the largest side of the serving workload: 128x128, 8 coils
        dict(_case("step", 128, coils=8, frames=16), name="step 128x128 8 coils"),
        # the batched dynamic series: uneven plans (side 24-64, 1-8 coils, spiral and radial, 1-4x N samples)
        dict(kind="batch", plans=6, lo=24, hi=64, mix=3000, prec="bf16x6", recon="store", frames=48, iters=3,
             lam=1e-3, name="batch of 6 plans"),
        # the serving loop: a burst of requests (1-64 frames) over resident plans of mixed sizes
        dict(kind="serve", plans=8, lo=16, hi=64, mix=4000, requests=40, slots=4, prec="bf16x6", recon="store",
             iters=3, lam=1e-3, name="serve burst of 40"),
        # the conditioning diagnostic and a truncated reconstruction of 64 frames
        dict(_case("spectrum", 20, samples=800, prec="fp64", frames=64, iters=1), name="spectrum 20x20"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case; no FP64 case does more work than the listed FP64 step, no other more than the
    largest listed one."""
    top = {fp64: max(work(c)["flops"] for c in listed() if (c["prec"] == "fp64") == fp64) for fp64 in (True, False)}
    while True:
        c = _drawn(rng)
        if work(c)["flops"] <= top[c["prec"] == "fp64"]:
            return c


def _drawn(rng):
    kind = rng.choice(["oneshot", "step", "step", "step", "apply", "apply", "batch", "serve", "spectrum"])
    if kind == "spectrum":
        side = rng.randint(8, 20)
        return _case(kind, side, samples=_log(rng, side * side, 4 * side * side), prec="fp64",
                     frames=_log(rng, 1, 64), iters=1, dtype=rng.choice(["c64", "c128"]))
    if kind == "batch":
        return dict(kind=kind, plans=rng.randint(2, 8), lo=rng.randint(16, 24), hi=rng.randint(32, 64),
                    mix=rng.randint(1, 10 ** 6), prec="bf16x6", recon=rng.choice(["none", "store"]),
                    frames=_log(rng, 8, 128), iters=3, lam=1e-3)
    if kind == "serve":
        return dict(kind=kind, plans=rng.randint(2, 10), lo=rng.randint(16, 24), hi=rng.randint(32, 64),
                    mix=rng.randint(1, 10 ** 6), requests=rng.randint(8, 60), slots=rng.randint(1, 6),
                    prec="bf16x6", recon=rng.choice(["none", "store"]), iters=3, lam=1e-3)
    coils = rng.choice([1, 2, 3, 4, 5, 8])
    traj = rng.choice(["spiral", "radial"])
    frames = _log(rng, 1, 64)
    form = rng.choice(["fp64", "x6", "x6", "x6", "x6 b0", "x6 3d", "x3"])
    if form == "fp64":
        side = _log(rng, 12, 36)
        return _case(kind, side, coils=coils, traj=traj, samples=_log(rng, side * side, 3 * side * side), prec="fp64",
                     recon=rng.choice(["none", "store"]), frames=min(frames, 24), dtype=rng.choice(["c64", "c128"]),
                     iters=1)
    if form == "x6 3d":
        nx, ny, nz = rng.randint(12, 28), rng.randint(12, 28), rng.randint(3, 9)
        return _case(kind, nx, ny, nz, coils=coils, samples=_log(rng, nx * ny, 2 * nx * ny),
                     keep=rng.choice([1.0, rng.uniform(0.4, 0.8)]), recon="none", frames=frames)
    if form == "x6 b0":
        side = _log(rng, 16, 60)
        return _case(kind, side, coils=coils, traj=traj, samples=_log(rng, side * side, 2 * side * side), b0=True,
                     recon="none", frames=min(frames, 32))
    if form == "x3":
        side = _log(rng, 12, 32)
        return _case(kind, side, coils=coils, traj=traj, samples=_log(rng, side * side, 2 * side * side),
                     prec="bf16x3", recon="none", frames=frames, iters=4)
    nx = _log(rng, 16, 100)
    ny = min(100, max(12, round(nx * rng.uniform(0.8, 1.25))))
    store = nx * ny <= 64 * 64 and rng.random() < 0.5
    return _case(kind, nx, ny, coils=coils, traj=traj, samples=_log(rng, nx * ny, 3 * nx * ny),
                 recon="store" if store else "none", frames=frames)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _members(case):
    """The encodings of a batch or server: sizes from the case's own `mix`, not from the seed."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["plans"]):
        side = rng.randint(case["lo"], case["hi"])
        out.append(_case(case["kind"], side, coils=rng.randint(1, 8), traj=rng.choice(["spiral", "radial"]),
                         samples=int(side * side * rng.uniform(1, 4 if case["kind"] == "batch" else 2)),
                         prec=case["prec"], recon=case["recon"], frames=case.get("frames", 64),
                         iters=case["iters"], lam=case["lam"]))
    return out


def _requests(case):
    """(plan, frames) of each request of a burst."""
    rng = random.Random(case["mix"] + 1)
    return [(rng.randrange(case["plans"]), rng.randint(1, 64)) for _ in range(case["requests"])]


def _mask(case):
    """Flat indices of the voxels reconstructed, or None for the whole grid."""
    if case["keep"] >= 1.0:
        return None
    r = synth.voxel_positions((case["nx"], case["ny"], case["nz"]))
    rad = np.sqrt((2 * r[:, 0]) ** 2 + (1.9 * r[:, 1]) ** 2 + (0.3 * r[:, 2]) ** 2)
    return np.sort(np.argsort(rad, kind="stable")[: max(1, int(case["keep"] * r.shape[0]))])


def _geometry(case, seed):
    """Plan inputs on the host: dims, traj, coil_maps, b0_hz, times, voxel_index."""
    rng = np.random.default_rng([int(seed), 7])
    nx, ny, nz, M2 = case["nx"], case["ny"], case["nz"], case["samples"]
    side = max(nx, ny)
    if case["traj"] == "spiral":
        J = max(1, side // 16)
        S = -(-M2 // J)
        k, idx = synth.spiral(side, J, S)
    else:
        S = max(2, min(2 * side, M2))
        k, idx = synth.radial(side, -(-M2 // S), S)
    k, idx = k[:M2], idx[:M2]
    th = rng.uniform(0, 2 * math.pi)
    k = k @ np.array([[math.cos(th), math.sin(th)], [-math.sin(th), math.cos(th)]])
    k = k * np.array([nx / side, ny / side])
    dims = (nx, ny)
    if nz > 1:  # a stack: the in-plane trajectory at every slice encoding
        kz = np.arange(nz) - nz // 2
        k = np.concatenate([np.concatenate([k, np.full((M2, 1), float(z))], axis=1) for z in kz])
        idx = np.tile(idx, nz)
        dims = (nx, ny, nz)
    vi = _mask(case)
    maps = synth.coil_maps(dims, case["coils"], rng) if case["coils"] > 1 else None
    b0 = synth.b0_map(dims, rng) if case["b0"] else None
    if vi is not None:
        maps = None if maps is None else np.ascontiguousarray(maps[:, vi])
        b0 = None if b0 is None else b0[vi]
    return dict(dims=dims, traj=k, coil_maps=maps, b0_hz=b0,
                times=(idx * synth.DWELL_S).astype(np.float64) if case["b0"] else None, voxel_index=vi)


def _data(case, geo, seed):
    """[F][C][M_k] k-space frames on the GPU: analytic ellipse spectra (one basis signal per
    ellipse), modulated by decaying time courses, plus 1 % noise."""
    C, F, k = case["coils"], case["frames"], geo["traj"]
    e = synth.ellipses(np.random.default_rng([int(seed), 8]), ELLIPSES)
    n_vox = case["nx"] * case["ny"] * case["nz"]
    basis = []
    for i in range(ELLIPSES):
        one = synth.Ellipses(e.centre[i:i + 1], e.axes[i:i + 1], e.angle[i:i + 1], np.ones(1, complex), e.tau[i:i + 1])
        rng = np.random.default_rng([int(seed), 9])  # the same coil offsets for every ellipse
        basis.append(synth.kspace_data(one, k[:, :2], n_vox, C, 1, rng, noise_frac=0.0)[0])
    basis = torch.from_numpy(np.stack(basis)).cuda()
    if k.shape[1] == 3:  # a Gaussian slab profile along the slice direction
        basis = basis * torch.exp(-(0.35 * torch.from_numpy(k[:, 2].copy()).cuda()) ** 2)
    f = np.arange(F)
    amps = torch.from_numpy(e.amp[None, :] * np.exp(-f[:, None] / e.tau[None, :])).cuda()
    data = (amps @ basis.reshape(ELLIPSES, -1)).reshape(F, C, k.shape[0])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 31 + 5)
    sigma = 0.01 * torch.sqrt(data.abs().square().mean())
    data += sigma * torch.randn(data.shape, generator=gen, device="cuda", dtype=torch.complex128)
    return data.to(DTYPE[case["dtype"]]).contiguous()


def _plan_args(case, geo):
    return dict(geo, lam=case["lam"], precision=PREC[case["prec"]], recon_mode=RECON[case["recon"]],
                refine_max_iters=case["iters"])


def _parts(case, seed):
    """(case, geometry, data) of every encoding of the case."""
    if case["kind"] not in ("batch", "serve"):
        g = _geometry(case, seed)
        return [(case, g, _data(case, g, seed))]
    out = []
    for i, c in enumerate(_members(case)):
        g = _geometry(c, seed * 100 + i)
        out.append((c, g, _data(c, g, seed * 100 + i)))
    return out


def prepare(case, seed):
    parts = _parts(case, seed)
    kind = case["kind"]
    if kind == "oneshot":
        return dict(kind=kind, args=_plan_args(*parts[0][:2]), data=parts[0][2])
    if kind == "serve":
        server = Server(budget_bytes=120 << 30, max_slots=case["slots"])
        ids = []
        for c, g, _ in parts:
            a = _plan_args(c, g)
            ids.append(server.register(**a))
        reqs = [(ids[i], parts[i][2][:f].contiguous()) for i, f in _requests(case)]
        outs = [torch.empty((f, _sizes(parts[i][0])[0]), dtype=torch.complex64, device="cuda")
                for i, f in _requests(case)]
        for pid, d in dict(reqs).items():  # plans resident, as in a running server
            assert server.wait(server.enqueue(pid, d[:1])[0]) == L.OK
        return dict(kind=kind, server=server, reqs=reqs, outs=outs)
    if kind == "batch":
        plans = [Plan(**_plan_args(c, g)) for c, g, _ in parts]
        stream = torch.cuda.Stream()  # graph capture needs a created stream
        datas = [d for _, _, d in parts]
        outs = [torch.empty((d.shape[0], p.n_vox), dtype=d.dtype, device="cuda") for d, p in zip(datas, plans)]
        return dict(kind=kind, batch=Batch(plans, graph=True), datas=datas, outs=outs, stream=stream)
    c, g, data = parts[0]
    plan = Plan(**_plan_args(c, g), keep_gram=kind == "spectrum")
    if kind in ("apply", "spectrum"):
        plan.build()
    return dict(kind=kind, plan=plan, data=data)


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["plan"].apply(state["data"])
    if kind == "step":
        return state["plan"].build().apply(state["data"])
    if kind == "oneshot":
        with Plan(**state["args"]) as plan:
            return plan.build().apply(state["data"])
    if kind == "batch":
        state["stream"].wait_stream(torch.cuda.current_stream())
        state["batch"].build(stream=state["stream"])
        outs = state["batch"].apply(state["datas"], state["outs"], stream=state["stream"])
        torch.cuda.current_stream().wait_stream(state["stream"])
        return outs
    if kind == "serve":
        sv = state["server"]
        tickets = [sv.enqueue(pid, d, out)[0] for (pid, d), out in zip(state["reqs"], state["outs"])]
        status = [sv.wait(t) for t in tickets]
        return {"status": np.array(status), "images": state["outs"]}
    plan, data = state["plan"], state["data"]
    mu, P, _ = plan.eig()
    images, rank, _ = plan.tsvd_apply(mu, P, data, energy=0.95, lam=0.0)
    return {"mu": mu, "images": images, "rank": rank}


# --------------------------------------------------------------------------
# the work a pass cannot do without
# --------------------------------------------------------------------------
def _sizes(c):
    N = c["nx"] * c["ny"] * c["nz"]
    if c["keep"] < 1.0:
        N = max(1, int(c["keep"] * N))
    return N, c["samples"] * c["nz"]


def _build_work(c):
    """Complex multiply-adds: without B0 the Gram follows from its table of grid offsets, with B0
    from all samples; Cholesky and inverse N^3 / 6 each; an explicit Recon N^2 per row of Encode."""
    N, Mk = _sizes(c)
    table = 4.0 * c["nx"] * c["ny"] * c["nz"] * Mk
    gram = 0.5 * N * N * Mk if c["b0"] else min(table, 0.5 * N * N * Mk)
    gram += 0.5 * N * N * c["coils"]
    recon = 1.0 * N * N * Mk * c["coils"] if c["recon"] == "store" else 0.0
    e = 16 if c["prec"] == "fp64" else 8
    return gram + N ** 3 / 3.0 + recon, 8.0 * N * N + (e * N * Mk * c["coils"] if c["recon"] == "store" else 0)


def _apply_work(c, frames):
    """E^H d once per frame, then per correction two triangular products and a residual (the exact
    Gram without B0, E and E^H with it). A FP64 plan with Recon multiplies by it instead."""
    N, Mk = _sizes(c)
    M = Mk * c["coils"]
    resid = 2.0 * N * M if c["b0"] or c["prec"] == "fp64" else 1.0 * N * N
    per_frame = N * M + N * N + c["iters"] * (resid + N * N)
    item = 8 if c["dtype"] == "c64" else 16
    factor = 16.0 * N * M if c["prec"] == "fp64" and c["recon"] == "store" else 8.0 * N * N
    return per_frame * frames, item * frames * (M + N) + factor


def work(case):
    kind = case["kind"]
    cmac, nbytes = 0.0, 0.0
    if kind == "spectrum":
        N, Mk = _sizes(case)
        cmac = 4.0 * N ** 3 + case["frames"] * (N * Mk + 2.0 * N * N)
        nbytes = 32.0 * N * N + 16.0 * case["frames"] * (N + Mk)
    elif kind == "batch":
        for c in _members(case):
            for w in (_build_work(c), _apply_work(c, case["frames"])):
                cmac, nbytes = cmac + w[0], nbytes + w[1]
    elif kind == "serve":
        members = _members(case)
        for i, f in _requests(case):
            w = _apply_work(members[i], f)
            cmac, nbytes = cmac + w[0], nbytes + w[1]
    else:
        parts = [_apply_work(case, case["frames"])]
        if kind != "apply":
            parts.append(_build_work(case))
        cmac, nbytes = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": nbytes, "flops": 8.0 * cmac}


# --------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# --------------------------------------------------------------------------
def _encode(c, g, rows):
    """[len(rows)][N] exp(-i 2 pi (k . r + df t)) of the samples `rows`."""
    r = synth.voxel_positions(g["dims"])
    if g["voxel_index"] is not None:
        r = r[g["voxel_index"]]
    k = torch.from_numpy(np.ascontiguousarray(g["traj"][rows])).cuda()
    ph = k @ torch.from_numpy(np.ascontiguousarray(r.T)).cuda()
    if g["b0_hz"] is not None:
        ph += torch.outer(torch.from_numpy(g["times"][rows]).cuda(), torch.from_numpy(g["b0_hz"]).cuda())
    return torch.polar(torch.ones_like(ph), -2 * math.pi * ph)


def _gram_and_rhs(c, g, data):
    """E^H E (without lambda) [N][N] and E^H d [N][F] in complex128. Without B0, A^H A depends only
    on the difference of two voxels' grid indices, so it is gathered from the table of differences."""
    Mk, F, C = g["traj"].shape[0], data.shape[0], c["coils"]
    S = torch.from_numpy(g["coil_maps"]).cuda() if g["coil_maps"] is not None else None
    N = S.shape[1] if S is not None else (len(g["voxel_index"]) if g["voxel_index"] is not None else
                                          int(np.prod(g["dims"])))
    d = data.to(torch.complex128)
    b = torch.zeros((C, N, F), dtype=torch.complex128, device="cuda")
    G = torch.zeros((N, N), dtype=torch.complex128, device="cuda") if c["b0"] else None
    dims = tuple(g["dims"]) + (1,) * (3 - len(g["dims"]))
    diff = [torch.arange(-(n - 1), n, device="cuda", dtype=torch.float64) / n for n in dims]
    T = torch.zeros([len(x) for x in diff], dtype=torch.complex128, device="cuda")
    for s in range(0, Mk, 4096):
        rows = slice(s, min(s + 4096, Mk))
        A = _encode(c, g, rows)
        for q in range(C):
            b[q] += A.conj().T @ d[:, q, rows].T
        if c["b0"]:
            G += A.conj().T @ A
        else:  # T[d] = sum_m exp(+i 2 pi k_m . d), d = difference (row voxel - column voxel)
            k = torch.from_numpy(np.ascontiguousarray(g["traj"][rows])).cuda()
            e = [torch.polar(torch.ones(k.shape[0], len(x), dtype=torch.float64, device="cuda"),
                             2 * math.pi * torch.outer(k[:, a], x)) if a < k.shape[1]
                 else torch.ones((k.shape[0], 1), dtype=torch.complex128, device="cuda") for a, x in enumerate(diff)]
            for z in range(e[2].shape[1]):
                T[:, :, z] += (e[0] * e[2][:, z:z + 1]).T @ e[1]
    if not c["b0"]:
        flat = torch.arange(int(np.prod(dims))) if g["voxel_index"] is None else torch.from_numpy(g["voxel_index"])
        flat = flat.cuda()
        ix = [flat % dims[0], (flat // dims[0]) % dims[1], flat // (dims[0] * dims[1])]
        G = torch.empty((N, N), dtype=torch.complex128, device="cuda")
        for s in range(0, N, 2048):
            at = [i[s:s + 2048, None] - i[None, :] + (n - 1) for i, n in zip(ix, dims)]
            G[s:s + 2048] = T[at[0], at[1], at[2]]
    if S is not None:
        for s in range(0, N, 2048):
            G[s:s + 2048] *= S[:, s:s + 2048].conj().T @ S
        b = (b * S.conj()[:, :, None]).sum(0)
    else:
        b = b[0]
    return G, b


def _solve(c, g, data):
    """Images [F][N] of (E^H E + lambda I) x = E^H d."""
    G, b = _gram_and_rhs(c, g, data)
    lam = c["lam"] * G.diagonal().real.mean()
    G.diagonal().add_(lam)
    Lf = torch.linalg.cholesky(G)
    del G
    y = torch.linalg.solve_triangular(Lf, b, upper=False)
    return torch.linalg.solve_triangular(Lf.mH, y, upper=True).T.contiguous()


def exact(case, seed):
    parts = _parts(case, seed)
    if case["kind"] == "batch":
        return [_solve(c, g, d) for c, g, d in parts]
    if case["kind"] == "serve":
        every = [_solve(c, g, d) for c, g, d in parts]
        return {"status": np.zeros(case["requests"], dtype=np.int64), "images": [every[i][:f] for i, f in _requests(case)]}
    c, g, data = parts[0]
    if case["kind"] != "spectrum":
        return _solve(c, g, data)
    G, b = _gram_and_rhs(c, g, data)
    mu, P = torch.linalg.eigh(G)
    mu, P = mu.flip(0).clamp_min(0), P.flip(1)
    rank = int((torch.cumsum(mu, 0) / mu.sum() < 0.95).sum()) + 1
    images = (P[:, :rank] @ ((P[:, :rank].mH @ b) / mu[:rank, None])).T.contiguous()
    return {"mu": mu, "images": images, "rank": rank}
