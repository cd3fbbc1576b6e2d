"""Performance cases of the Galerkin-FFT solver, through the calls that user
programs make (paper_1806_10599_gb300.gff).

Every case is a dict of plain values; `kind` selects the call:

  apply       gff_apply_operator on device vectors, the hot operation of the
              conjugate gradients, on elastic (St.Venant-Kirchhoff) polycrystals
  project     gff_project, the bare projection of a stress field (residuals)
  small       gff_apply_operator of the small-strain variant (symmetric projection)
  host        gff_apply_operator_host, for callers with host buffers only
  linearise   gff_constitutive of a crystal-plasticity RVE in FP64 (return maps and
              consistent tangents), the stress read back, and one operator apply
              with the new tangent
  history     a new crystal-plasticity RVE in a handle, a few load increments of a
              cyclic history in mixed precision, the deformation gradient and the
              fatigue indicators read back
  batch       the same for several RVEs of different sizes through gff_batch_run
  unet        the warm-start network: output, loss and all parameter gradients

Inputs come from the seed alone.  Grids are periodic Voronoi polycrystals.
"""

import math

import numpy as np
import torch

from paper_1806_10599_gb300 import gff as g

# axis lengths the solver takes: even, 4 ... 128, factors 2, 3 and 5
AXES = [n for n in range(4, 129, 2) if not [m for m in (7, 11, 13, 17, 19, 23, 29, 31, 37, 41, 43, 47, 53, 59, 61)
                                            if n % m == 0]]
C11, C12, C44 = 168.4e9, 121.4e9, 75.4e9
CP = dict(gdot0=1e-3, p_exp=20.0, tau0=50e6, c_af=20e9, d_af=200.0)
MIXED_CONTROL = [0, 1, 1, 1, 1, 1, 1, 0, 1]  # uniaxial stress: F11 and F32 prescribed


def listed():
    return [
        # the smallest RVE of the examples, a mixed-control residual's projection: latency and launches
        {"name": "project_f64_16", "kind": "project", "nx": 16, "ny": 16, "nz": 16, "f64": True, "discrete": False,
         "mask": True, "grains": 8},
        # one CG operator of the 64^3 polycrystal, FP64
        {"name": "apply_f64_64", "kind": "apply", "nx": 64, "ny": 64, "nz": 64, "f64": True, "discrete": False,
         "mask": False, "grains": 200},
        # the apply benchmark: 128^3, 500 grains, FP64 and FP32
        {"name": "apply_f64_128", "kind": "apply", "nx": 128, "ny": 128, "nz": 128, "f64": True, "discrete": False,
         "mask": False, "grains": 500},
        {"name": "apply_f32_128", "kind": "apply", "nx": 128, "ny": 128, "nz": 128, "f64": False, "discrete": False,
         "mask": False, "grains": 500},
        # non-cubic RVEs: the discrete projection under mixed control, sizes off the powers of two
        {"name": "apply_f32_80x96x48", "kind": "apply", "nx": 80, "ny": 96, "nz": 48, "f64": False, "discrete": True,
         "mask": True, "grains": 60},
        {"name": "apply_f64_90x100x60", "kind": "apply", "nx": 90, "ny": 100, "nz": 60, "f64": True, "discrete": True,
         "mask": True, "grains": 120},
        # linear elastic small-strain homogenisation
        {"name": "small_f64_64", "kind": "small", "nx": 64, "ny": 64, "nz": 64, "f64": True, "discrete": True,
         "mask": False, "grains": 150},
        # the operator as a service to a program that holds its vectors on the host (pinned)
        {"name": "host_f64_128", "kind": "host", "nx": 128, "ny": 128, "nz": 128, "f64": True, "discrete": False,
         "mask": False, "grains": 500},
        # FP64 linearisation of a plastic state: what each FP64 Newton correction starts with
        {"name": "linearise_f64_48", "kind": "linearise", "nx": 48, "ny": 48, "nz": 48, "f64": True, "discrete": False,
         "mask": False, "grains": 100},
        # the 64^3, 200-grain cyclic simulation from its start, mixed precision, extrapolated starts
        {"name": "history_mixed_64", "kind": "history", "n": 64, "grains": 200, "steps": 4, "discrete": False},
        # a statistical volume element: RVEs of several sizes through one history
        {"name": "batch_mixed_5", "kind": "batch", "rves": 5, "n0": 32, "n1": 48, "n2": 64, "grains": 50, "steps": 2},
        # one training gradient of the warm-start network on a 64^3 sample
        {"name": "unet_grad_64", "kind": "unet", "n": 64},
    ]


def _axis(rng, lo, hi):
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(AXES, key=lambda n: abs(n - target))


def draw(rng):
    kind = rng.choices(["apply", "project", "small", "host", "linearise", "history", "batch", "unet"],
                       weights=[8, 3, 2, 2, 2, 1, 1, 1])[0]
    if kind == "history":
        return {"kind": kind, "n": rng.choice([16, 20, 24, 30, 32, 36, 40, 48, 50, 54, 60, 64]),
                "grains": rng.randint(8, 200), "steps": rng.randint(2, 4), "discrete": rng.random() < 0.5}
    if kind == "batch":
        n = [rng.choice([16, 20, 24, 32, 40, 48, 60, 64]) for _ in range(3)]
        return {"kind": kind, "rves": rng.randint(2, 5), "n0": n[0], "n1": n[1], "n2": n[2],
                "grains": rng.randint(8, 60), "steps": rng.randint(1, 2)}
    if kind == "unet":
        return {"kind": kind, "n": rng.choice([8, 16, 24, 32, 40, 48, 56, 64])}
    hi = 48 if kind == "linearise" else 128
    nx, ny, nz = _axis(rng, 8, hi), _axis(rng, 8, hi), _axis(rng, 8, hi)
    if rng.random() < 0.4:
        ny = nz = nx
    f64 = True if kind == "linearise" else rng.random() < 0.5
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "f64": f64, "discrete": rng.random() < 0.5,
            "mask": rng.random() < 0.5, "grains": rng.randint(4, 500 if kind != "linearise" else 100)}


# ---------------------------------------------------------------------------- inputs
def _gen(seed):
    r = torch.Generator(device="cuda")
    r.manual_seed(1000003 * seed + 17)
    return r


def _voronoi(nx, ny, nz, grains, r):
    """Periodic Voronoi grain ids [nz][ny][nx] (int32, device) and unit quaternions (host)."""
    seeds = torch.rand(grains, 3, generator=r, device="cuda")
    q = torch.randn(grains, 4, generator=r, device="cuda", dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True)
    q = torch.where(q[:, :1] < 0, -q, q)
    ax = [(torch.arange(n, device="cuda") + 0.5) / n for n in (nx, ny, nz)]

    def part(a, s):  # squared minimum-image distance along one axis [n][grains]
        d = (a[:, None] - s[None, :]).abs()
        return torch.minimum(d, 1 - d) ** 2

    dx, dy, dz = (part(a, seeds[:, k]) for k, a in enumerate(ax))
    gid = torch.empty(nz, ny, nx, dtype=torch.int32, device="cuda")
    for z in range(nz):
        gid[z] = (dz[z][None, None, :] + dy[:, None, :] + dx[None, :, :]).argmin(dim=2).int()
    return gid, q


def _noise(r, n, scale):
    return torch.randn(n, generator=r, device="cuda", dtype=torch.float64) * scale


def _field_inputs(case, seed):
    """Everything of an apply-like case that comes from the seed."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    r = _gen(seed)
    gid, quat = _voronoi(nx, ny, nz, case["grains"], r)
    eye = torch.eye(3, device="cuda", dtype=torch.float64).reshape(9, 1)
    inp = {"gid": gid, "quat": quat}
    if case["kind"] == "linearise":
        # a strain beyond yield with grain-scale scatter, small plastic distortions and backstresses
        a = 0.0009 + 0.0004 * torch.rand(1, generator=r, device="cuda", dtype=torch.float64)
        mac = torch.diag(torch.stack([a[0], -0.45 * a[0], -0.45 * a[0]])).reshape(9, 1)
        inp["F"] = eye + mac + _noise(r, (9, N), 1e-4)
        inp["Fpi"] = eye + _noise(r, (9, N), 1e-4)
        inp["chi"] = _noise(r, (12, N), 2e6)
    else:
        inp["F"] = (0 if case["kind"] == "small" else eye) + _noise(r, (9, N), 0.004)
    x = _noise(r, (9, N), 1.0)
    if case["kind"] == "project":  # a stress field: mean stresses with fluctuations
        x = 1e8 * (x + 2 * torch.randn(9, 1, generator=r, device="cuda", dtype=torch.float64))
    inp["x"] = x if case["f64"] else x.float()
    return inp


class _Handles:
    """Handles (and a network) that live as long as the state."""

    def __init__(self):
        self.hs, self.u = [], None

    def __del__(self):
        for h in self.hs:
            g.gff_destroy(h)
        if self.u is not None:
            g.gff_unet_destroy(self.u)


def _mask(case):
    return np.array(MIXED_CONTROL, dtype=np.uint8) if case["mask"] else None


def _strain_path(steps):
    """The first increments of a +-1 % cycle at 20 increments per quarter and 4 s per cycle."""
    F = np.zeros((steps, 9))
    for k in range(steps):
        f11 = 1 + 0.0005 * (k + 1)
        F[k, 0], F[k, 4], F[k, 8] = f11, f11 ** -0.5, f11 ** -0.5
    return np.full(steps, 0.05), F, np.zeros((steps, 9), np.uint8), np.zeros((steps, 9)), np.arange(steps) == 0


def _cp_options(discrete=False):
    return g.make_options(precision=g.GFF_PREC_MIXED, projection=int(discrete), newton_tol=1e-10, cg_tol=1e-6,
                          warm_start=g.GFF_WARM_EXTRAPOLATE)


def _rves(case, seed):
    """(n, gid [n^3], quaternions) of a history or batch case, on the host."""
    r = _gen(seed)
    sizes = [case["n"]] if case["kind"] == "history" else [case["n%d" % (i % 3)] for i in range(case["rves"])]
    out = []
    for n in sizes:
        gid, quat = _voronoi(n, n, n, case["grains"], r)
        out.append((n, gid.cpu().numpy().reshape(-1), quat.cpu().numpy()))
    return out


def prepare(case, seed):
    kind = case["kind"]
    own = _Handles()
    s = {"case": case, "own": own}
    if kind == "unet":
        n = case["n"]
        r = np.random.default_rng(seed)
        own.u = g.gff_unet_create(seed)
        w = g.gff_unet_get_params(own.u)
        w[-9 * 16 - 9:] = (0.2 * r.standard_normal(9 * 16 + 9)).astype(np.float32)  # the head starts at zero
        g.gff_unet_set_params(own.u, w)
        s["n"], s["w"] = n, w
        s["x"] = r.standard_normal((n ** 3, g.UNET_IN), dtype=np.float32)
        s["target"] = 0.3 * r.standard_normal((n ** 3, 9), dtype=np.float32)
        return s
    if kind in ("history", "batch"):
        s["rves"] = _rves(case, seed)
        s["path"] = _strain_path(case["steps"])
        for n, gid, quat in s["rves"]:
            h = g.gff_create(g.make_grid(n, n, n), _cp_options(case.get("discrete", False)))
            own.hs.append(h)
            g.gff_set_material(h, 0, g.make_material(g.GFF_MAT_CP_FCC, C11=C11, C12=C12, C44=C44, **CP))
            g.gff_set_microstructure(h, gid, len(quat), quat, np.zeros(len(quat), np.int32))
            g.gff_autotune(h)
        return s
    inp = _field_inputs(case, seed)
    h = g.gff_create(g.make_grid(case["nx"], case["ny"], case["nz"]), g.make_options(projection=int(case["discrete"])))
    own.hs.append(h)
    if kind == "small":
        g.gff_set_strain_measure(h, g.GFF_STRAIN_SMALL)
    mat = g.GFF_MAT_CP_FCC if kind == "linearise" else g.GFF_MAT_SVK_CUBIC
    g.gff_set_material(h, 0, g.make_material(mat, C11=C11, C12=C12, C44=C44, **CP))
    ng = case["grains"]
    g.gff_set_microstructure(h, inp["gid"].cpu().numpy().reshape(-1), ng, inp["quat"].cpu().numpy(),
                             np.zeros(ng, np.int32))
    g.gff_autotune(h)
    g.gff_set_field(h, g.GFF_FIELD_F, inp["F"].cpu().numpy())
    if kind == "linearise":
        g.gff_set_field(h, g.GFF_FIELD_FP_INV, inp["Fpi"].cpu().numpy())
        g.gff_set_field(h, g.GFF_FIELD_CHI, inp["chi"].cpu().numpy())
    elif kind != "project":
        g.gff_constitutive(h, 1.0)
    s["h"], s["mask"] = h, _mask(case)
    s["prec"] = g.GFF_PREC_FP64 if case["f64"] else g.GFF_PREC_MIXED
    s["x"], s["y"] = inp["x"], torch.empty_like(inp["x"])
    if kind == "host":
        s["x"], s["y"] = inp["x"].cpu().pin_memory(), torch.empty_like(inp["x"], device="cpu").pin_memory()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "unet":
        y, loss, grads = g.gff_unet_eval_host(s["own"].u, s["n"], s["x"], s["target"])
        return {"y": y, "loss": loss, "grads": grads}
    if kind == "history":
        h, (n, gid, quat) = s["own"].hs[0], s["rves"][0]
        g.gff_set_microstructure(h, gid, len(quat), quat, np.zeros(len(quat), np.int32))
        P, _ = g.gff_run_history(h, *s["path"])
        pc, w, fs = g.gff_get_fips(h, len(quat))
        return {"P": P, "F": g.gff_get_field(h, g.GFF_FIELD_F, n ** 3), "pcyc": pc, "wcyc": w, "fs": fs}
    if kind == "batch":
        for h, (n, gid, quat) in zip(s["own"].hs, s["rves"]):
            g.gff_set_microstructure(h, gid, len(quat), quat, np.zeros(len(quat), np.int32))
        P, _, _ = g.gff_batch_run(s["own"].hs, *s["path"])
        return {"P": P, "F": [g.gff_get_field(h, g.GFF_FIELD_F, n ** 3) for h, (n, _, _) in zip(s["own"].hs, s["rves"])],
                "fips": [g.gff_get_fips(h, len(q)) for h, (_, _, q) in zip(s["own"].hs, s["rves"])]}
    h, prec, mask, x, y = s["h"], s["prec"], s["mask"], s["x"], s["y"]
    if kind == "project":
        g.gff_project(h, prec, mask, x, y)
        return y
    if kind == "host":
        g.gff_apply_operator_host(h, prec, mask, x, y)
        return y
    if kind == "linearise":
        g.gff_constitutive(h, 0.05)
        P = g.gff_get_field(h, g.GFF_FIELD_P, case["nx"] * case["ny"] * case["nz"])
        g.gff_apply_operator(h, prec, mask, x, y)
        return {"P": P, "y": y}
    g.gff_apply_operator(h, prec, mask, x, y)
    return y


# ---------------------------------------------------------------------------- work
_UNET = [(32, 16, 0), (16, 16, 0), (16, 32, 1), (32, 32, 1), (32, 64, 2), (64, 64, 2), (64, 64, 3), (64, 64, 3),
         (128, 64, 2), (64, 64, 2), (96, 32, 1), (32, 32, 1), (48, 16, 0), (16, 16, 0)]


def _fft_flops(N):
    return 2 * 9 * 2.5 * N * math.log2(N)  # nine real fields, there and back


def work(case):
    kind = case["kind"]
    if kind == "unet":
        V = case["n"] ** 3
        mac = sum(27 * ci * co * V / 8 ** lev for ci, co, lev in _UNET)
        return {"bytes": 4.0 * V * (32 + 9 + 9) + 2 * 4 * sum(27 * ci * co for ci, co, _ in _UNET), "flops": 6.0 * mac}
    if kind in ("history", "batch"):
        sizes = [case["n"]] if kind == "history" else [case["n%d" % (i % 3)] for i in range(case["rves"])]
        N = sum(n ** 3 for n in sizes)
        # per increment: state in and out (F, Fp^-1, chi, slips, FIPs) and, at the least, one return map of one
        # local iteration, one tangent and three operator applies
        state = 8.0 * N * 2 * (9 + 9 + 12 + 12 + 61)
        per = N * (900 + 4000 + 3 * 162) + 3 * _fft_flops(N)
        return {"bytes": case["steps"] * (state + 3 * 4.0 * N * 99), "flops": case["steps"] * per}
    N = case["nx"] * case["ny"] * case["nz"]
    e = 8 if case["f64"] else 4
    if kind == "project":
        return {"bytes": e * 18.0 * N, "flops": _fft_flops(N) + 45.0 * N}
    w = {"bytes": e * 99.0 * N, "flops": 162.0 * N + _fft_flops(N) + 45.0 * N}
    if kind == "linearise":  # state in, P and K out (K used by the apply), return map and exact tangent
        w["bytes"] += 8.0 * N * (9 + 9 + 12 + 9 + 81)
        w["flops"] += 2 * 6000.0 * N
    return w


# ---------------------------------------------------------------------------- 64-bit values
def _rot(q):
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _stiff(E, R):
    """C : E of rotated cubic crystals, E symmetric [V][3][3], R [V][3][3] (crystal axes in columns)."""
    tr = E.diagonal(dim1=1, dim2=2).sum(1)
    ee = torch.einsum("via,vij,vja->va", R, E, R)
    eye = torch.eye(3, device=E.device, dtype=E.dtype)
    return C12 * tr[:, None, None] * eye + 2 * C44 * E + (C11 - C12 - 2 * C44) * torch.einsum("via,va,vja->vij", R, ee, R)


def _vox(a):  # [9][V] -> [V][3][3]
    return a.t().reshape(-1, 3, 3)


def _project(case, x):
    """G_M of x [9][N] (float64)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    X = torch.fft.fftn(x.reshape(3, 3, nz, ny, nx), dim=(2, 3, 4))
    q, nyq = [], []
    for n in (nx, ny, nz):
        k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64).round()
        nyq.append(k.abs() * 2 == n)
        q.append(torch.tan(math.pi * torch.where(nyq[-1], 0 * k, k) / n) * n if case["discrete"] else 2 * math.pi * k)
    Q = [q[0].reshape(1, 1, nx), q[1].reshape(1, ny, 1), q[2].reshape(nz, 1, 1)]
    zero = nyq[0].reshape(1, 1, nx) | nyq[1].reshape(1, ny, 1) | nyq[2].reshape(nz, 1, 1)
    q2 = Q[0] ** 2 + Q[1] ** 2 + Q[2] ** 2
    q2 = torch.where(q2 == 0, torch.ones_like(q2), q2)
    M = torch.tensor(MIXED_CONTROL if case["mask"] else [0] * 9, device="cuda", dtype=torch.float64).reshape(3, 3)
    dc = X[:, :, 0, 0, 0] * M
    if case["kind"] == "small":
        X = 0.5 * (X + X.transpose(0, 1))
        inv = 1 / q2.sqrt()
        nn = [c * inv for c in Q]
        a = [sum(X[i, j] * nn[j] for j in range(3)) for i in range(3)]
        na = sum(nn[i] * a[i] for i in range(3))
        Y = torch.stack([torch.stack([nn[i] * a[j] + a[i] * nn[j] - na * nn[i] * nn[j] for j in range(3)])
                         for i in range(3)])
    else:
        Y = torch.empty_like(X)
        for i in range(3):
            t = sum(X[i, j] * Q[j] for j in range(3)) / q2
            for j in range(3):
                Y[i, j] = t * Q[j]
    Y = torch.where(zero, torch.zeros_like(Y), Y)
    Y[:, :, 0, 0, 0] = dc
    return torch.fft.ifftn(Y, dim=(2, 3, 4)).real.reshape(9, -1)


def _slip_systems():
    nrm = [(1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)]
    dirs = [(0, 1, -1), (0, 1, 1), (1, -1, 0), (1, 0, -1), (1, 0, 1), (1, 1, 0)]
    S = [np.outer(d, m) / math.sqrt(6.0) for m in nrm for d in dirs if np.dot(m, d) == 0]
    return torch.tensor(np.array(S), device="cuda", dtype=torch.float64)


def _plasticity(F, A, chin, R, x, dt):
    """P and K : x of the crystal-plasticity law, by damped Newton on the slips of every voxel and the derivative of
    the converged return map."""
    S0 = torch.einsum("vij,ajk,vlk->vail", R, _slip_systems(), R)
    eye = torch.eye(3, device="cuda", dtype=torch.float64)
    coef, p, tau0, c, d = dt * CP["gdot0"], CP["p_exp"], CP["tau0"], CP["c_af"], CP["d_af"]

    def stress(F, dg):
        Fpi = A @ (eye - torch.einsum("va,vaij->vij", dg, S0))
        Fe = F @ Fpi
        S = _stiff(0.5 * (Fe.mT @ Fe - eye), R)
        return Fpi, Fe, S

    def resid(F, dg):
        Fpi, Fe, S = stress(F, dg)
        tau = torch.einsum("vij,vaij->va", Fe.mT @ Fe @ S, S0)
        y = (tau - (chin + c * dg) / (1 + d * dg.abs())) / tau0
        return dg - coef * y.abs() ** p * y.sign()

    def P_of(F, dg):
        Fpi, Fe, S = stress(F, dg)
        return Fe @ S @ Fpi.mT

    def jac(dg):
        cols = []
        for b in range(12):
            e = torch.zeros_like(dg)
            e[:, b] = 1
            cols.append(torch.func.jvp(lambda z: resid(F, z), (dg,), (e,))[1])
        return torch.stack(cols, 2)

    dg = torch.zeros_like(chin)
    r = resid(F, dg)
    best = r.norm(dim=1)
    for it in range(200):
        step = torch.linalg.solve(jac(dg), r.unsqueeze(2)).squeeze(2)
        t = torch.ones_like(best)
        for _ in range(12):
            rn = resid(F, dg - t[:, None] * step)
            bad = ~(rn.norm(dim=1) < best)
            if not bad.any():
                break
            t = torch.where(bad, 0.5 * t, t)
        nn = rn.norm(dim=1)
        ok = nn < best
        dg = torch.where(ok[:, None], dg - t[:, None] * step, dg)
        r = torch.where(ok[:, None], rn, r)
        done = bool((~ok).all()) or float(step.abs().max()) < 1e-17
        best = torch.where(ok, nn, best)
        if done or float(best.max()) < 1e-17:
            break
    P, dP = torch.func.jvp(lambda z: P_of(z, dg), (F,), (x,))
    dr = torch.func.jvp(lambda z: resid(z, dg), (F,), (x,))[1]
    ddg = -torch.linalg.solve(jac(dg), dr.unsqueeze(2)).squeeze(2)
    dP = dP + torch.func.jvp(lambda z: P_of(F, z), (dg,), (ddg,))[1]
    return P, dP


def _unet_reference(case, s):
    """Output, loss and parameter gradients of the network in 64 bits (no bfloat16 rounding)."""
    n = case["n"]
    w = torch.tensor(s["w"], device="cuda", dtype=torch.float64, requires_grad=True)
    off = 0
    layers = []
    for ci, co, _ in _UNET:
        layers.append((w[off:off + 27 * co * ci].reshape(27, co, ci), w[off + 27 * co * ci:off + 27 * co * ci + co]))
        off += 27 * co * ci + co
    head, hb = w[off:off + 144].reshape(9, 16), w[off + 144:]

    def conv(l, a):  # a [m][m][m][C], periodic
        W, b = layers[l]
        z = b
        for t in range(27):
            o = (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)
            z = z + torch.roll(a, (-o[0], -o[1], -o[2]), (0, 1, 2)) @ W[t].t()
        return torch.where(z > 0, z, 0.125 * z)

    def pool(a):
        m = a.shape[0] // 2
        return a.reshape(m, 2, m, 2, m, 2, -1).mean((1, 3, 5))

    def up(a):
        return a.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)

    a = torch.tensor(s["x"], device="cuda", dtype=torch.float64).reshape(n, n, n, -1)
    e1 = conv(1, conv(0, a))
    e2 = conv(3, conv(2, pool(e1)))
    e3 = conv(5, conv(4, pool(e2)))
    e4 = conv(7, conv(6, pool(e3)))
    d3 = conv(9, conv(8, torch.cat([up(e4), e3], 3)))
    d2 = conv(11, conv(10, torch.cat([up(d3), e2], 3)))
    d1 = conv(13, conv(12, torch.cat([up(d2), e1], 3)))
    y = (d1 @ head.t() + hb).reshape(-1, 9)
    loss = ((y - torch.tensor(s["target"], device="cuda", dtype=torch.float64)) ** 2).mean()
    loss.backward()
    return {"y": y.detach(), "loss": float(loss), "grads": w.grad}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("history", "batch"):
        return None  # a whole nonlinear solve: minutes in plain numpy
    if kind == "unet":
        s = prepare(case, seed)
        return _unet_reference(case, s)
    inp = _field_inputs(case, seed)
    x = inp["x"].double()
    if kind == "project":
        return _project(case, x)
    R = _rot(inp["quat"])[inp["gid"].reshape(-1).long()]
    F, X = _vox(inp["F"]), _vox(x)
    if kind == "small":
        Kx = _stiff(0.5 * (X + X.mT), R)
    elif kind == "linearise":
        P, Kx = _plasticity(F, _vox(inp["Fpi"]), inp["chi"].t().contiguous(), R, X, 0.05)
    else:
        eye = torch.eye(3, device="cuda", dtype=torch.float64)
        FX = F.mT @ X
        Kx = X @ _stiff(0.5 * (F.mT @ F - eye), R) + F @ _stiff(0.5 * (FX + FX.mT), R)
    y = _project(case, Kx.reshape(-1, 9).t().contiguous())
    if kind == "host":
        return y.cpu()
    return {"P": P.reshape(-1, 9).t().reshape(-1), "y": y} if kind == "linearise" else y
