"""The calls by which the library's speed is judged: what a transport calculation asks of it.

A calculation on one transition region is: solve the unperturbed Green's function for a block of
boundary columns and a set of energies (shifted COCG), get the lead self-energies (closed form or
decimation), take the Dyson step to the perturbed boundary Green's function, read the transmission.
The cases below are those calls, each through the package's public functions, over the sizes of the
repository's workloads and tests: the 8 x 8 x 12 wire (launches and latency count), slab and sampled
columns of middle-sized regions, the 64 x 64 x 128 and 72 x 72 x 256 grids, and boundary solves from
128 to 2048 rows.

A production solve takes thousands of seed iterations of equal cost; the cases on larger grids stop
after a fixed number of them (the iteration cap, as the repository's full-size tests do), so that the
iterates are a well-defined result at every precision.  Only the Green's functions, self-energies and
transmissions are returned: residual norms and iteration counts are stopping diagnostics.
"""

import math

import numpy as np
import torch

import paper_1502_00081_gb300 as rs

DEV = "cuda" if torch.cuda.is_available() else "cpu"
PREC = {"fp64": rs.RSFD_FP64, "df64": rs.RSFD_DF64, "c64": rs.RSFD_MIXED}
TOL_OFF = 1e-30   # no energy converges: the iteration cap ends the solve
H_WIRE = 0.5      # grid spacing of the wires with closed-form boundary Green's functions
C2 = (-2.0, 1.0)
C4 = (-2.5, 4.0 / 3.0, -1.0 / 12.0)


def listed():
    return [
        # the whole chain on the smallest wire, every plane column, to convergence: G0 -> Sigma -> G -> T
        dict(name="wire_chain_fp64", kind="chain", nx=8, ny=8, nz=12, order=2, K=8, eta=1e-3, tol=1e-12),
        # every slab column of a short wire, untuned options: many columns of a small grid
        dict(name="slab_columns_df64", kind="cocg", prec="df64", nx=16, ny=16, nz=48, order=4, n_face=2, cols=1024,
             K=16, eta=1e-2, iters=63, tuned=False, atoms=0),
        # complex128 vectors on a small ragged grid, the accurate mode used to check the others
        dict(name="ragged_fp64", kind="cocg", prec="fp64", nx=37, ny=26, nz=19, order=4, n_face=2, cols=24, K=8,
             eta=5e-2, iters=63, tuned=False, atoms=0),
        # three regions of uneven size in one call, one stream each
        dict(name="uneven_regions_df64", kind="regions", prec="df64", sizes="32x32x64,40x40x96,48x48x128",
             energies="48,100,64", cols=32, order=4, n_face=1, eta=1e-3, iters=63),
        # complex64 vectors (broad levels), untuned options
        dict(name="region_c64", kind="cocg", prec="c64", nx=56, ny=56, nz=80, order=4, n_face=1, cols=64, K=64,
             eta=1e-1, iters=63, tuned=False, atoms=0),
        # a block of sampled columns of the 64 x 64 x 128 region, tuned as the benchmark does
        dict(name="sampled_columns_df64", kind="cocg", prec="df64", nx=64, ny=64, nz=128, order=4, n_face=1, cols=38,
             K=128, eta=1e-3, iters=127, tuned=True, atoms=0),
        # the peapod-shaped region with a nonlocal projector on each of 460 atoms, tuned
        dict(name="peapod_projectors_df64", kind="cocg", prec="df64", nx=72, ny=72, nz=256, order=4, n_face=2, cols=16,
             K=100, eta=1e-3, iters=95, tuned=True, atoms=460),
        # the boundary step in complex128 throughout (the accurate mode)
        dict(name="dyson_fp64", kind="dyson", prec="fp64", nx=16, ny=16, nz=24, K=8, eta=2e-2, left=False, T=False),
        # all columns of G_bb for a batch of energies, reduced-precision handle
        dict(name="dyson_df64", kind="dyson", prec="df64", nx=32, ny=16, nz=24, K=16, eta=2e-2, left=False, T=False),
        # a large boundary, only what the transmission needs, and the transmission
        dict(name="dyson_transmission_df64", kind="dyson", prec="df64", nx=32, ny=32, nz=24, K=4, eta=2e-2, left=True,
             T=True),
        # the boundary step with two interior planes for the density of states
        dict(name="interior_planes_df64", kind="tracked", prec="df64", nx=12, ny=10, nz=24, planes=2, K=8, eta=2e-2),
        # self-energies of leads with their own layer potential
        dict(name="lead_decimation", kind="leads", nx=10, ny=10, order=4, K=8, eta=2e-2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "cocg", "cocg", "cocg", "cocg", "projectors", "regions", "dyson", "dyson", "dyson",
                       "tracked", "leads"])
    if kind == "chain":
        return dict(kind="chain", nx=rng.randint(4, 10), ny=rng.randint(4, 10), nz=rng.randint(6, 16), order=2,
                    K=rng.randint(2, 12), eta=rng.choice([1e-3, 3e-3, 1e-2, 3e-2]), tol=1e-12)
    if kind == "regions":
        sizes = ",".join("%dx%dx%d" % (rng.randint(20, 56), rng.randint(20, 56), rng.randint(32, 128)) for _ in range(3))
        return dict(kind="regions", prec=rng.choice(["df64", "df64", "fp64", "c64"]), sizes=sizes,
                    energies=",".join(str(rng.randint(16, 100)) for _ in range(3)), cols=rng.randint(4, 24),
                    order=rng.choice([2, 4]), n_face=1, eta=rng.choice([5e-2, 1e-1]), iters=rng.choice([31, 63]))
    if kind == "dyson":
        prec = rng.choice(["fp64", "df64", "df64", "c64"])
        area = _log_int(rng, 16, 300 if prec == "fp64" else 900)
        nx = rng.randint(max(2, int(area ** 0.5 / 2)), int(area ** 0.5 * 2))
        ny = max(1, round(area / nx))
        K = max(1, min(32, int((1 if prec == "fp64" else 8) * (512 / (nx * ny)) ** 3)))
        return dict(kind="dyson", prec=prec, nx=nx, ny=ny, nz=rng.randint(4, 40), K=rng.randint(1, K),
                    eta=rng.choice([2e-2, 5e-2]), left=rng.random() < 0.5, T=rng.random() < 0.5)
    if kind == "tracked":
        return dict(kind="tracked", prec=rng.choice(["fp64", "df64"]), nx=rng.randint(3, 14), ny=rng.randint(3, 12),
                    nz=rng.randint(8, 32), planes=rng.randint(1, 3), K=rng.randint(1, 8),
                    eta=rng.choice([2e-2, 5e-2]))
    if kind == "leads":
        return dict(kind="leads", nx=rng.randint(2, 11), ny=rng.randint(2, 11), order=rng.choice([2, 4]),
                    K=rng.randint(1, 10), eta=rng.choice([1e-2, 2e-2, 5e-2]))
    prec = "df64" if kind == "projectors" else rng.choice(["df64", "df64", "df64", "fp64", "c64"])
    order = rng.choice([2, 4, 4])
    n_face = rng.choice([1, order // 2])
    # complex128 arithmetic is about ten times as slow, so its grids stop earlier
    N = _log_int(rng, 2000, 60000 if prec == "fp64" else (300000 if kind == "projectors" else 500000))
    nz = _log_int(rng, max(8, N // 4096), max(9, min(256, N // 64)))
    nx = _log_int(rng, max(5, int((N / nz) ** 0.5 / 1.6)), max(6, min(80, int((N / nz) ** 0.5 * 1.6))))
    ny = max(4, min(80, N // (nz * nx)))
    pool = 2 * n_face * nx * ny
    cols = max(1, min(pool, _log_int(rng, 4, 1024), int(2e7 / (nx * ny * nz)) if prec != "fp64" else int(2e6 / (nx * ny * nz)) + 2))
    return dict(kind="cocg", prec=prec, nx=nx, ny=ny, nz=nz, order=order, n_face=n_face, cols=cols,
                K=_log_int(rng, 4, 160), eta=rng.choice([5e-2, 1e-1, 1e-1] if prec == "c64" else [1e-3, 1e-2, 5e-2]),
                iters=rng.choice([31, 63]), tuned=False, atoms=_log_int(rng, 3, 60) if kind == "projectors" else 0)


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _axes(nx, ny, nz, h):
    return ((np.arange(nx) + 1.0) * h, (np.arange(ny) + 1.0) * h, np.arange(nz) * h)


def _wells(rng, nx, ny, nz, h, centres, depths, width):
    """Sum of Gaussian wells on the grid, [nz, ny, nx]."""
    ax = _axes(nx, ny, nz, h)
    g = [torch.from_numpy(np.exp(-(a[None, :] - centres[:, k:k + 1]) ** 2 / (2.0 * width * width))).to(DEV)
         for k, a in enumerate(ax)]
    gz = g[2] * torch.from_numpy(-depths).to(DEV)[:, None]
    xy = (g[1][:, :, None] * g[0][:, None, :]).reshape(len(depths), -1)
    return (gz.T @ xy).reshape(nz, ny, nx).cpu().numpy()


class _Proj:
    """Kleinman-Bylander projectors in the binding's CSR form."""


def _projectors(centres, nx, ny, nz, h, sigma=1.2, r_cut=3.0, energy=0.5):
    ax = _axes(nx, ny, nz, h)
    ptr, idx, val = [0], [], []
    for c in centres:
        w = [np.nonzero(np.abs(a - c[k]) <= r_cut)[0] for k, a in enumerate(ax)]
        d2 = ((ax[2][w[2]] - c[2]) ** 2)[:, None, None] + ((ax[1][w[1]] - c[1]) ** 2)[None, :, None] + \
             ((ax[0][w[0]] - c[0]) ** 2)[None, None, :]
        lin = (w[2][:, None, None] * ny + w[1][None, :, None]) * nx + w[0][None, None, :]
        inside = d2 <= r_cut * r_cut
        p = np.exp(-d2[inside] / (2.0 * sigma * sigma))
        idx.append(lin[inside].astype(np.int64))
        val.append(p / math.sqrt(max(float(np.sum(p * p)) * h ** 3, 1e-300)))
        ptr.append(ptr[-1] + idx[-1].size)
    q = _Proj()
    q.n_atoms, q.ptr, q.idx, q.val = len(centres), np.asarray(ptr, np.int64), np.concatenate(idx), np.concatenate(val)
    q.E = np.full(len(centres), energy)
    return q


def _peapod_sites(rng, nx, ny, nz, h, n):
    """A tube of rings around a sphere at mid-length (400 + 60 sites at full size), n sites in all."""
    box = np.array([(nx + 1) * h, (ny + 1) * h, (nz - 1) * h])
    n_s = max(1, n * 60 // 460)
    rings = max(1, (n - n_s) // 20)
    radius, rad_s = min(12.8, 0.43 * min(box[0], box[1])), min(6.7, 0.23 * min(box[0], box[1]))
    spacing = min(2.3, 0.9 * box[2] / max(rings, 1))
    k = np.arange(n_s) + 0.5
    polar, azim = np.arccos(1.0 - 2.0 * k / n_s), np.pi * (1.0 + 5 ** 0.5) * k
    pts = np.stack([np.sin(polar) * np.cos(azim), np.sin(polar) * np.sin(azim), np.cos(polar)], 1)
    q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    sites = [box / 2 + p for p in pts @ q.T * rad_s]
    for i in range(n - n_s):
        r, s = divmod(i, 20)
        a = 2.0 * np.pi * s / 20 + (np.deg2rad(9.0) if r % 2 else 0.0)
        sites.append(np.array([box[0] / 2 + radius * np.cos(a), box[1] / 2 + radius * np.sin(a),
                               box[2] / 2 + (r - (rings - 1) / 2.0) * spacing]))
    return np.asarray(sites)


def _region(seed, nx, ny, nz, order, n_face, K, cols, atoms=0, erange=(-0.5, 0.5), h=0.4, wells=None):
    """Potential, projectors, energies and boundary columns of one region."""
    rng = np.random.Generator(np.random.PCG64(seed))
    box = np.array([(nx + 1) * h, (ny + 1) * h, (nz - 1) * h])
    r = dict(grid=(nx, ny, nz), h=h, order=order, n_face=n_face, proj=None)
    if atoms:
        c = _peapod_sites(rng, nx, ny, nz, h, atoms)
        r["V"] = _wells(rng, nx, ny, nz, h, c, np.ones(atoms), 0.8)
        r["proj"] = _projectors(c, nx, ny, nz, h)
        erange = (-0.3, 0.3)
    else:
        n = wells or max(2, int(round(200 * nx * ny * nz / (64 * 64 * 128))))
        r["V"] = _wells(rng, nx, ny, nz, h, rng.uniform(size=(n, 3)) * box, rng.uniform(0.5, 1.5, size=n), 1.0)
    nxy = nx * ny
    planes = list(range(n_face)) + list(range(nz - n_face, nz))
    pool = np.concatenate([np.arange(nxy, dtype=np.int64) + z * nxy for z in planes])
    r["rows"] = pool
    r["cols"] = pool if cols >= pool.size else np.sort(rng.choice(pool, size=cols, replace=False))
    r["E"] = np.linspace(erange[0], erange[1], K)
    return r


def _regions_of(case, seed):
    out = []
    for i, (s, k) in enumerate(zip(case["sizes"].split(","), case["energies"].split(","))):
        nx, ny, nz = (int(v) for v in s.split("x"))
        out.append(_region(seed * 16 + i, nx, ny, nz, case["order"], case["n_face"], int(k), case["cols"]))
    return out


def _chain_region(case, seed):
    return _region(seed, case["nx"], case["ny"], case["nz"], case["order"], case["order"] // 2, case["K"], 10 ** 9,
                   erange=(0.1, 0.8), h=H_WIRE, wells=3)


def _modes(nx, h, v=None):
    """Eigenpairs of the 1-D operator -1/2 d^2/dx^2 + v (2nd order, walls)."""
    A = np.diag(np.full(nx, 1.0 / h ** 2) + (0.0 if v is None else v)) + \
        np.diag(np.full(nx - 1, -0.5 / h ** 2), 1) + np.diag(np.full(nx - 1, -0.5 / h ** 2), -1)
    return np.linalg.eigh(A)


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _wire_blocks(case, seed, interior=0):
    """Boundary Green's function of a wire with a separable potential and the self-energies of its
    uniform leads, in closed form: G0 [K, n, n] on the first and last plane (then `interior` planes),
    Sigma_L, Sigma_R [K, ns, ns], complex128; all are complex symmetric."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny, nz, K = case["nx"], case["ny"], case["nz"], case["K"]
    h, ns = H_WIRE, nx * ny
    vx, vy, vz = (rng.uniform(-0.4, 0.0, size=n) for n in (nx, ny, nz))
    E = np.linspace(0.4, 2.4, K) + rng.uniform(0.0, 0.1)
    Z = _t(E + 1j * case["eta"])

    def transverse(ax, ay):
        (ex, ux), (ey, uy) = ax, ay
        e = (ey[:, None] + ex[None, :]).reshape(-1)
        U = np.einsum("ya,xb->yxab", uy, ux).reshape(ns, ns)
        return _t(e), _t(U)

    e, U = transverse(_modes(nx, h, vx), _modes(ny, h, vy))
    ez, uz = (_t(a) for a in _modes(nz, h, vz))
    zs = [0, nz - 1] + sorted(int(z) for z in rng.permutation(np.arange(1, nz - 1))[:interior])
    w = 1.0 / (Z[:, None, None] - e[None, :, None] - ez[None, None, :])           # [K, mode, n]

    def dense(g, U):                                                             # U diag(g) U^T per energy
        return torch.complex((U[None] * g.real[:, None, :]) @ U.T, (U[None] * g.imag[:, None, :]) @ U.T)

    G0 = torch.empty((K, len(zs) * ns, len(zs) * ns), dtype=torch.complex128, device=DEV)
    for a, za in enumerate(zs):
        for b, zb in enumerate(zs[:a + 1]):
            blk = dense((w * (uz[za] * uz[zb])).sum(2), U)
            G0[:, a * ns:(a + 1) * ns, b * ns:(b + 1) * ns] = blk
            G0[:, b * ns:(b + 1) * ns, a * ns:(a + 1) * ns] = blk
    # leads without a potential: Sigma = t lam per mode, t lam^2 - (Z - e - d) lam + t = 0, |lam| < 1
    e0, U0 = transverse(_modes(nx, h), _modes(ny, h))
    t, q = -0.5 / h ** 2, Z[:, None] - e0[None, :] - 1.0 / h ** 2
    s = torch.sqrt(q * q - 4 * t * t)
    lam = torch.where(((q + s) / (2 * t)).abs() < 1, (q + s) / (2 * t), (q - s) / (2 * t))
    S = dense(t * lam, U0)
    return G0, S, S.clone(), zs


def _layers(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    R = case["order"] // 2
    V = [rng.uniform(-0.5, 0.0, size=(R, case["ny"], case["nx"])) for _ in range(2)]
    return V[0], V[1], np.linspace(0.3, 2.0, case["K"]) + rng.uniform(0.0, 0.1)


# ------------------------------------------------------------------------------------------------
# what a program keeps, and one pass
# ------------------------------------------------------------------------------------------------
def _handle(r, prec):
    return rs.Handle(r["grid"], r["h"], r["order"], r["V"], n_face=r["n_face"], proj=r["proj"], precision=PREC[prec])


def _empty(h, K, ncols, n):
    return torch.empty((K, ncols, n), dtype=h.complex_dtype, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        r = _chain_region(case, seed)
        h = _handle(r, "fp64")
        G0 = _empty(h, case["K"], h.nb, h.nb)
        return dict(case=case, r=r, h=h, G0=G0, G=torch.empty_like(G0))
    if kind == "cocg":
        r = _region(seed, case["nx"], case["ny"], case["nz"], case["order"], case["n_face"], case["K"], case["cols"],
                    case["atoms"])
        h = _handle(r, case["prec"])
        if case["tuned"]:
            rs.rsfd_autotune(h.ptr, r["E"], case["eta"], slots=int(r["cols"].size), iters=64)
        return dict(case=case, r=r, h=h, G0=_empty(h, case["K"], r["cols"].size, h.nb))
    if kind == "regions":
        regions = _regions_of(case, seed)
        handles = [_handle(r, case["prec"]) for r in regions]
        outs = [_empty(h, r["E"].size, r["cols"].size, h.nb) for r, h in zip(regions, handles)]
        jobs = [dict(h=h.ptr, cols=r["cols"], energies=r["E"], eta=case["eta"], tol=TOL_OFF, maxit=case["iters"], G0_bb=o)
                for r, h, o in zip(regions, handles, outs)]
        return dict(case=case, handles=handles, outs=outs, jobs=jobs)
    if kind in ("dyson", "tracked"):
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        G0, SL, SR, zs = _wire_blocks(case, seed, case.get("planes", 0))
        h = rs.Handle((nx, ny, nz), H_WIRE, 2, np.zeros(nx * ny * nz), n_face=1, precision=PREC[case["prec"]])
        if kind == "tracked":
            rs.rsfd_set_tracked_planes(h.ptr, zs[2:])
        elif case["left"]:
            rs.rsfd_set_solve_options(h.ptr, dyson_cols=1)
        G0 = G0.to(h.complex_dtype).contiguous()
        return dict(case=case, h=h, G0=G0, SL=SL, SR=SR, G=torch.empty_like(G0))
    nx, ny, R = case["nx"], case["ny"], case["order"] // 2
    VL, VR, E = _layers(case, seed)
    h = rs.Handle((nx, ny, 2 * R + 2), H_WIRE, case["order"], np.zeros(nx * ny * (2 * R + 2)), precision=rs.RSFD_FP64)
    return dict(case=case, h=h, VL=VL, VR=VR, E=E)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "cocg":
        r = state["r"]
        rs.rsfd_shifted_cocg(state["h"].ptr, r["cols"], r["E"], case["eta"], TOL_OFF, case["iters"], state["G0"])
        return state["G0"]
    if kind == "regions":
        rs.rsfd_shifted_cocg_regions(state["jobs"])
        return state["outs"]
    if kind == "chain":
        r, h = state["r"], state["h"]
        rs.rsfd_shifted_cocg(h.ptr, h.rows, r["E"], case["eta"], case["tol"], 20000, state["G0"])
        SL, SR = rs.rsfd_lead_sigma_uniform(case["nx"], case["ny"], r["h"], r["order"], r["E"], case["eta"])
        SL, SR = torch.from_numpy(SL).to(DEV), torch.from_numpy(SR).to(DEV)
        rs.rsfd_dyson_boundary(h.ptr, state["G0"], SL, SR, state["G"])
        return dict(G0=state["G0"], G=state["G"], T=rs.rsfd_transmission(h.ptr, state["G"], SL, SR))
    if kind == "dyson":
        rs.rsfd_dyson_boundary(state["h"].ptr, state["G0"], state["SL"], state["SR"], state["G"])
        if not case["T"]:
            return dict(G=state["G"])
        return dict(G=state["G"], T=rs.rsfd_transmission(state["h"].ptr, state["G"], state["SL"], state["SR"]))
    if kind == "tracked":
        rs.rsfd_dyson_tracked(state["h"].ptr, state["G0"], state["SL"], state["SR"], state["G"])
        return state["G"]
    SL, SR, steps = rs.rsfd_lead_sigma_decimation(state["h"].ptr, state["E"], case["eta"], state["VL"], state["VR"],
                                                  ns=(case["order"] // 2) * case["nx"] * case["ny"])
    return dict(SL=SL, SR=SR, steps=steps)


# ------------------------------------------------------------------------------------------------
# what one pass cannot do without
# ------------------------------------------------------------------------------------------------
def _cocg_work(N, nb, ncols, K, iters, order, prec, nnz=0):
    """One seed iteration of one column reads r_{n-1}, r_{n-2} and writes r_n; the vectors of a call that
    fit in the chip's caches need not move.  About 55 + 12 R real operations a point (stencil, three-term
    update, dots), 16 per boundary row and energy (p and x of the shifted systems), 8 per projector entry."""
    v = 8 if prec == "c64" else 16
    krylov = 3 * v * N * ncols
    out = K * nb * ncols * v
    move = krylov * iters if krylov > 120e6 else 0
    flops = iters * ncols * (N * (55 + 6 * order) + 16 * K * nb + 8 * nnz)
    return dict(bytes=float(move + out + 8 * N), flops=float(flops))


def work(case):
    kind, K = case["kind"], case.get("K", 0)
    if kind == "cocg":
        N, nb = case["nx"] * case["ny"] * case["nz"], 2 * case["n_face"] * case["nx"] * case["ny"]
        return _cocg_work(N, nb, min(case["cols"], nb), K, case["iters"] + 1, case["order"], case["prec"],
                          1700 * case["atoms"])
    if kind == "regions":
        b = f = 0.0
        for s, k in zip(case["sizes"].split(","), case["energies"].split(",")):
            nx, ny, nz = (int(v) for v in s.split("x"))
            w = _cocg_work(nx * ny * nz, 2 * nx * ny, min(case["cols"], 2 * nx * ny), int(k), case["iters"] + 1,
                           case["order"], case["prec"])
            b, f = b + w["bytes"], f + w["flops"]
        return dict(bytes=b, flops=f)
    if kind == "chain":
        N, nb = case["nx"] * case["ny"] * case["nz"], case["order"] * case["nx"] * case["ny"]
        # a column of so small a grid takes about as many iterations as the grid has points
        w = _cocg_work(N, nb, nb, K, min(N, 800), case["order"], "fp64")
        w["flops"] += K * (8 / 3 + 8 + 4) * 8 / 8 * nb ** 3
        return w
    v = 8 if case.get("prec") == "c64" else 16
    if kind in ("dyson", "tracked"):
        ns = case["nx"] * case["ny"]
        nb = 2 * ns
        nr = nb + case.get("planes", 0) * ns
        nc = ns if case.get("left") else nr
        # M = I - G0 Sigma, an LU, nc right-hand sides
        f = 8.0 * nb * nb * ns + 8 / 3 * nb ** 3 + 8.0 * nb * nb * nc
        if kind == "tracked":
            f += 8.0 * ns * nb * nr + 8.0 * nr * nr * nb
        if case.get("T"):
            f += 16.0 * ns ** 3
        return dict(bytes=float(K * (2 * nr * nr * v + 2 * ns * ns * 16)), flops=float(K * f))
    n = (case["order"] // 2) * case["nx"] * case["ny"]
    # about a dozen doublings to the decay length: an LU, 2 n right-hand sides, four products; two leads
    return dict(bytes=float(2 * K * n * n * 16), flops=float(2 * K * 12 * (8 / 3 + 16 + 32) * n ** 3))


# ------------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------------
def _cocg64(r, eta, iters):
    """x_b [K, ncols, nb] of the shifted COCG after iters + 1 residuals (r_0 ... r_iters, the last one
    without its update), seed at the middle energy; no energy converges in so few iterations."""
    nx, ny, nz = r["grid"]
    N, h, R = nx * ny * nz, r["h"], r["order"] // 2
    c = C2 if R == 1 else C4
    cols, rows = _t(r["cols"]), _t(r["rows"])
    W = cols.numel()
    V = _t(r["V"].reshape(nz, ny, nx)) + 3.0 * (-0.5 * c[0] / h ** 2)
    Z = _t(r["E"] + 1j * eta)
    K, s = Z.numel(), Z.numel() // 2
    if r["proj"] is not None:
        p = r["proj"]
        atom = _t(np.repeat(np.arange(p.n_atoms), np.diff(p.ptr)))
        pidx, pval, pE = _t(p.idx), _t(p.val), _t(p.E)

    def apply(v):                                                   # (Z_s - H) v, v [W, N]
        g = v.view(W, nz, ny, nx)
        Hv = V * g
        for k in range(1, R + 1):
            a = -0.5 * c[k] / h ** 2
            for d in (1, 2, 3):
                n = g.shape[d]
                if n > k:
                    Hv.narrow(d, 0, n - k).add_(g.narrow(d, k, n - k), alpha=a)
                    Hv.narrow(d, k, n - k).add_(g.narrow(d, 0, n - k), alpha=a)
        Hv = Hv.view(W, N)
        if r["proj"] is not None:
            q = torch.zeros((W, p.n_atoms), dtype=v.dtype, device=DEV).index_add_(1, atom, v[:, pidx] * pval)
            Hv.index_add_(1, pidx, (q * (pE * h ** 3))[:, atom] * pval)
        return Z[s] * v - Hv

    one = torch.ones((W, 1), dtype=torch.complex128, device=DEV)
    r0 = torch.zeros((W, N), dtype=torch.complex128, device=DEV)     # r_n
    r0[torch.arange(W, device=DEV), cols] = 1.0
    rm = torch.zeros_like(r0)                                        # r_{n-1}
    x = torch.zeros((W, K, rows.numel()), dtype=torch.complex128, device=DEV)
    pb = torch.zeros_like(x)
    pi, pim = one.expand(W, K).clone(), one.expand(W, K).clone()
    am, rrm = one.clone(), one.clone()
    for n in range(iters):
        q = apply(r0)
        rr = (r0 * r0).sum(1, keepdim=True)
        beta = rr / rrm if n else torch.zeros_like(one)
        al = rr / ((r0 * q).sum(1, keepdim=True) - beta / am * rr)
        cc = beta * al / am
        bi = (pim / pi) ** 2 * beta
        pn = (1.0 + cc + al * (Z[None, :] - Z[s])) * pi - cc * pim
        pb.mul_(bi[:, :, None]).add_(r0[:, None, rows] / pi[:, :, None])
        x.add_(pb * (pi / pn * al)[:, :, None])
        pim, pi = pi, pn
        rm = (1.0 + cc) * r0 - cc * rm - al * q
        r0, rm, am, rrm = rm, r0, al, rr
    return x.transpose(0, 1).contiguous()


def _dyson64(G0, SL, SR, ns):
    """G_bb of matrices [K, nb, nb] in the row-column sense (all inputs symmetric)."""
    G0S = torch.cat([G0[:, :, :ns] @ SL, G0[:, :, ns:2 * ns] @ SR], 2)
    return torch.linalg.solve(torch.eye(2 * ns, dtype=G0.dtype, device=DEV) - G0S, G0)


def _T64(G, SL, SR, ns):
    gL, gR = (1j * (S - S.transpose(1, 2).conj()) for S in (SL, SR))
    A = G[:, ns:2 * ns, :ns]
    return torch.einsum("kab,kba->k", gL @ A.transpose(1, 2).conj(), gR @ A).real.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "cocg":
        r = _region(seed, case["nx"], case["ny"], case["nz"], case["order"], case["n_face"], case["K"], case["cols"],
                    case["atoms"])
        return _cocg64(r, case["eta"], case["iters"])
    if kind == "regions":
        return [_cocg64(r, case["eta"], case["iters"]) for r in _regions_of(case, seed)]
    if kind == "chain":
        r = _chain_region(case, seed)
        nx, ny, nz = r["grid"]
        ns, h = nx * ny, r["h"]
        D = [_t(_modes(n, h)[1] * _modes(n, h)[0]) @ _t(_modes(n, h)[1]).T for n in (nx, ny, nz)]
        I = [torch.eye(n, dtype=torch.float64, device=DEV) for n in (nx, ny, nz)]
        H = torch.kron(D[2], torch.kron(I[1], I[0])) + torch.kron(I[2], torch.kron(D[1], I[0])) + \
            torch.kron(I[2], torch.kron(I[1], D[0])) + torch.diag(_t(r["V"].reshape(-1)))
        rows = _t(r["rows"])
        ez, Uz = torch.linalg.eigh(H)
        Ub = Uz[rows].to(torch.complex128)
        Z = _t(r["E"] + 1j * case["eta"])
        G0 = torch.stack([(Ub / (z - ez)) @ Ub.T for z in Z])
        (ex, ux), (ey, uy) = _modes(nx, h), _modes(ny, h)
        e0, U0 = _t((ey[:, None] + ex[None, :]).reshape(-1)), _t(np.einsum("ya,xb->yxab", uy, ux).reshape(ns, ns))
        t, q = -0.5 / h ** 2, Z[:, None] - e0[None, :] - 1.0 / h ** 2
        s = torch.sqrt(q * q - 4 * t * t)
        lam = torch.where(((q + s) / (2 * t)).abs() < 1, (q + s) / (2 * t), (q - s) / (2 * t))
        U0 = U0.to(torch.complex128)
        S = (U0[None] * (t * lam)[:, None, :]) @ U0.T
        G = _dyson64(G0, S, S, ns)
        return dict(G0=G0.transpose(1, 2).contiguous(), G=G.transpose(1, 2).contiguous(), T=_T64(G, S, S, ns))
    if kind in ("dyson", "tracked"):
        ns = case["nx"] * case["ny"]
        G0, SL, SR, _ = _wire_blocks(case, seed, case.get("planes", 0))
        if case["prec"] == "c64":
            G0 = G0.to(torch.complex64).to(torch.complex128)
        if kind == "tracked":
            nb = 2 * ns
            Y = torch.linalg.solve(torch.eye(nb, dtype=G0.dtype, device=DEV) -
                                   torch.cat([G0[:, :nb, :ns] @ SL, G0[:, :nb, ns:nb] @ SR], 2), G0[:, :nb, :])
            G = G0 + G0[:, :, :ns] @ (SL @ Y[:, :ns]) + G0[:, :, ns:nb] @ (SR @ Y[:, ns:])
            return G.transpose(1, 2).contiguous()
        G = _dyson64(G0, SL, SR, ns)
        T = _T64(G, SL, SR, ns)
        if case["left"]:
            G[:, :, ns:] = 0
        out = dict(G=G.transpose(1, 2).contiguous())
        return {**out, "T": T} if case["T"] else out
    VL, VR, E = _layers(case, seed)
    nx, ny, R, h = case["nx"], case["ny"], case["order"] // 2, H_WIRE
    c = C2 if R == 1 else C4
    nxy, n = nx * ny, R * nx * ny

    def kin(m):
        A = np.zeros((m, m))
        for k in range(R + 1):
            A += -0.5 * c[k] / h ** 2 * (np.eye(m, k=k) + (np.eye(m, k=-k) if k else 0.0))
        return A

    plane = np.kron(kin(ny), np.eye(nx)) + np.kron(np.eye(ny), kin(nx))
    two = kin(2 * R)                                  # z couplings inside a layer and to the next one
    h01 = _t(np.kron(two[:R, R:], np.eye(nxy)) + 0j)
    out = []
    for V, a0, b0 in ((VL, h01.T, h01), (VR, h01, h01.T)):
        h00 = _t(np.kron(np.eye(R), plane) + np.kron(two[:R, :R], np.eye(nxy)) + np.diag(V.reshape(-1)) + 0j)
        Zs = _t(E + 1j * case["eta"])[:, None, None] * torch.eye(n, dtype=torch.complex128, device=DEV)
        es, ee = h00.expand_as(Zs).clone(), h00.expand_as(Zs).clone()
        al, be = a0.expand_as(Zs).contiguous(), b0.expand_as(Zs).contiguous()
        for _ in range(60):
            if max(al.abs().max().item(), be.abs().max().item()) < 1e-16:
                break
            g = torch.linalg.solve(Zs - ee, torch.cat([al, be], 2))
            ga, gb = g[:, :, :n], g[:, :, n:]
            ab = al @ gb
            es, ee = es + ab, ee + ab + be @ ga
            al, be = al @ ga, be @ gb
        out.append((a0 @ torch.linalg.solve(Zs - es, b0.expand_as(Zs).contiguous())).transpose(1, 2).contiguous())
    return dict(SL=out[0], SR=out[1], steps=None)
