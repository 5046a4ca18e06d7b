"""Workloads of the homogenization library whose run time matters to its users.

A case is one call sequence a program makes on a handle it keeps: a cell problem solved to its
tolerance and its corrector fields read back (``solve``), one Lippmann-Schwinger step on the caller's
device fields (``ls``), or a group of requests sent through the request server (``serve``).

Sizes and materials are those of the package's own configurations, tests and benchmark: random
spheres (128^3, contrast 100), three-phase spheres (64^3, orders 0 and 1), the 256-grain Voronoi
tessellation (up to 512^3), the centred sphere (32^3, FP64 Basic Scheme), Hashin's two-dimensional
structure, and the serving stream's grids.  Geometry, moduli and fields are drawn from the seed.

Results of the FP32 mode (FP32 fields and transforms, certified at a residual of 1e-6) are good to
about six digits; a program keeps them in single precision, as the passes here return them.  The FP64
mode's results stay double.

``exact`` solves the same problems with torch's FFTs in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1712_05145_gb300 import hom, synthetic

UNIT = np.eye(6)
SCHEMES = {"basic": hom.HOM_BASIC, "cg": hom.HOM_CG, "bicgstab": hom.HOM_BICGSTAB}


def listed():
    return [
        # the serving stream's smallest grid: launch latency and host reads count
        {"name": "spheres_32", "kind": "solve", "geometry": "spheres", "n1": 32, "n2": 32, "n3": 32, "contrast": 30.0,
         "precision": "fp32", "scheme": "cg", "loads": 6, "order": 0, "tol": 1e-6},
        # the serving stream's non-power-of-two grid
        {"name": "spheres_96", "kind": "solve", "geometry": "spheres", "n1": 96, "n2": 96, "n3": 96, "contrast": 10.0,
         "precision": "fp32", "scheme": "cg", "loads": 6, "order": 0, "tol": 1e-6},
        # the ordinary job: a random-sphere composite, all six unit strains, C_eff and the strain fields
        {"name": "spheres_128", "kind": "solve", "geometry": "spheres", "n1": 128, "n2": 128, "n3": 128,
         "contrast": 100.0, "precision": "fp32", "scheme": "cg", "loads": 6, "order": 0, "tol": 1e-6},
        # the serving stream's anisotropic grid with the Krylov solver the paper ran
        {"name": "bicgstab_32x64x128", "kind": "solve", "geometry": "spheres", "n1": 32, "n2": 64, "n3": 128,
         "contrast": 10.0, "precision": "fp32", "scheme": "bicgstab", "loads": 6, "order": 0, "tol": 1e-6},
        # a polycrystal whose planes no longer fit one thread block, the three axial strains (the grains'
        # spread of moduli amplifies the residual into the strain: five digits of it ask for 2e-7)
        {"name": "voronoi_256", "kind": "solve", "geometry": "voronoi", "n1": 256, "n2": 256, "n3": 256,
         "contrast": 0.0, "precision": "fp32", "scheme": "cg", "loads": 3, "order": 0, "tol": 2e-7},
        # half of the benchmark's grid, one load case (the whole grid's six take several seconds)
        {"name": "voronoi_512_one_load", "kind": "solve", "geometry": "voronoi", "n1": 512, "n2": 256, "n3": 512,
         "contrast": 0.0, "precision": "fp32", "scheme": "cg", "loads": 1, "order": 0, "tol": 2e-7},
        # the paper's higher-order problem: order 0, then the 18 loads of order 1
        {"name": "three_phase_64_order1", "kind": "solve", "geometry": "three_phase", "n1": 64, "n2": 64, "n3": 64,
         "contrast": 100.0, "precision": "fp32", "scheme": "cg", "loads": 6, "order": 1, "tol": 1e-6},
        # the paper's Basic Scheme in double precision on its smallest three-dimensional example
        {"name": "basic_32_fp64", "kind": "solve", "geometry": "centred", "n1": 32, "n2": 32, "n3": 32, "contrast": 10.0,
         "precision": "fp64", "scheme": "basic", "loads": 1, "order": 0, "tol": 1e-8},
        # the paper's two-dimensional example (plane stress) on a fine grid, double precision
        {"name": "hashin_2d_512_fp64", "kind": "solve", "geometry": "hashin", "n1": 512, "n2": 512, "n3": 1,
         "contrast": 10.0, "precision": "fp64", "scheme": "cg", "loads": 2, "order": 0, "tol": 1e-8},
        # a program with its own solver: one FP64 step for the six loads, and one large FP32 step
        {"name": "ls_step_64_fp64", "kind": "ls", "n1": 64, "n2": 64, "n3": 64, "precision": "fp64", "loads": 6},
        {"name": "ls_step_256x192x128_fp32", "kind": "ls", "n1": 256, "n2": 192, "n3": 128, "precision": "fp32",
         "loads": 2},
        # requests of several grids and both orders that arrive together
        {"name": "serve_8", "kind": "serve", "requests": 8, "max_contrast": 100.0},
    ]


_AXES = [16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512]


def draw(rng):
    def log_uniform(lo, hi):
        return float("%.4g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(["cg", "cg", "cg", "bicgstab", "order1", "fp64", "hashin", "ls", "ls", "serve"])
    if kind in ("cg", "bicgstab"):
        most = 1 << rng.randrange(13, 24 if kind == "cg" else 21)   # voxels: the grids' logarithms are spread
        while True:
            n1, n2, n3 = (rng.choice(_AXES) for _ in range(3))
            if most // 3 < n1 * n2 * n3 <= most:
                break
        shape = max(n1, n2, n3) / min(n1, n2, n3)
        # spheres need room along the shortest axis and are placed one by one on the host
        geometry = rng.choice(["spheres", "three_phase", "voronoi"]) if shape <= 4 and n1 * n2 * n3 <= 1 << 21 else "voronoi"
        contrast = {"spheres": log_uniform(2.0, 100.0 if kind == "cg" else 30.0), "three_phase": log_uniform(4.0, 100.0),
                    "voronoi": 0.0}[geometry]
        return {"kind": "solve", "geometry": geometry, "n1": n1, "n2": n2, "n3": n3, "contrast": contrast,
                "precision": "fp32", "scheme": kind, "loads": rng.choice([1, 3, 6, 6]), "order": 0,
                "tol": 2e-7 if geometry == "voronoi" else 1e-6}
    if kind == "order1":
        n = rng.choice([32, 48, 64, 96])
        return {"kind": "solve", "geometry": "three_phase", "n1": n, "n2": n, "n3": rng.choice([32, 48, n]),
                "contrast": log_uniform(4.0, 100.0), "precision": "fp32", "scheme": "cg", "loads": 6, "order": 1,
                "tol": 1e-6}
    if kind == "fp64":
        n = rng.choice([16, 24, 32, 48, 64])
        scheme = rng.choice(["basic", "cg"])
        return {"kind": "solve", "geometry": "centred", "n1": n, "n2": n, "n3": n, "contrast": log_uniform(2.0, 30.0),
                "precision": "fp64", "scheme": scheme, "loads": rng.choice([1, 6]), "order": 0, "tol": 1e-8}
    if kind == "hashin":
        n = rng.choice([64, 96, 128, 192, 256, 384, 512])
        return {"kind": "solve", "geometry": "hashin", "n1": n, "n2": n, "n3": 1, "contrast": log_uniform(0.1, 100.0),
                "precision": "fp64", "scheme": "cg", "loads": rng.choice([1, 2]), "order": 0, "tol": 1e-8}
    if kind == "ls":
        fp64 = rng.random() < 0.5
        most = 1 << rng.randrange(14, 22 if fp64 else 24)
        while True:
            n1, n2, n3 = (rng.choice([8, 12] + _AXES) for _ in range(3))
            loads = rng.choice([1, 2, 3, 6])
            if most // 3 < n1 * n2 * n3 * loads <= most:
                break
        return {"kind": "ls", "n1": n1, "n2": n2, "n3": n3, "precision": "fp64" if fp64 else "fp32", "loads": loads}
    return {"kind": "serve", "requests": rng.randrange(3, 11), "max_contrast": log_uniform(5.0, 100.0)}


# ---- inputs ------------------------------------------------------------------------------------------
_SERVE_GRIDS = [(32, 32, 32), (48, 48, 48), (64, 64, 64), (96, 96, 96), (32, 64, 128)]


def _microstructure(case, seed):
    grid = (case["n1"], case["n2"], case["n3"])
    rng = np.random.default_rng(seed)
    geometry, contrast = case["geometry"], case["contrast"]
    if geometry == "spheres":
        return synthetic.random_spheres(grid, seed=seed, inclusion_e=contrast)
    if geometry == "three_phase":
        return synthetic.three_phase_spheres(grid, seed=seed, youngs=(1.0, math.sqrt(contrast), contrast))
    if geometry == "voronoi":
        return synthetic.voronoi_torch(grid, seed=seed, n_grains=256)
    stiff = contrast * rng.uniform(0.8, 1.0)   # fixed geometries: the seed draws the moduli
    if geometry == "centred":
        return synthetic.centred_sphere(grid[0], inclusion=(stiff, stiff))
    return synthetic.hashin_2d(grid[0], e_core=100.0 * rng.uniform(0.8, 1.2), e_coat=100.0 * stiff)


def _requests(case, seed):
    """(microstructure, order) of each request of the serving stream."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case["requests"]):
        grid = _SERVE_GRIDS[(k + case["requests"]) % len(_SERVE_GRIDS)]
        contrast = math.exp(rng.uniform(math.log(2.0), math.log(case["max_contrast"])))
        ms = synthetic.random_spheres(grid, seed=seed + 97 * k, inclusion_e=contrast)
        out.append((ms, k % 2))
    return out


def _step_material(case, seed):
    """Three random phases, as in the parity tests of the step."""
    rng = np.random.default_rng(seed)
    lame = np.array([[1.0, 1.0], [8.0, 5.0], [0.4, 0.3]]) * rng.uniform(0.8, 1.2, size=(3, 1))
    phase = rng.choice(3, size=(case["n3"], case["n2"], case["n1"]), p=[0.5, 0.3, 0.2]).astype(np.uint8)
    return synthetic.Microstructure(phase, lame, 4.0, 2.5)


def _step_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["loads"], 6, case["n3"], case["n2"], case["n1"])
    eps = torch.empty(shape, dtype=torch.float64, device="cuda").uniform_(-1.0, 1.0, generator=g)
    return eps, UNIT[: case["loads"]]


class _Server:
    def __init__(self):
        self.s = hom.hom_server_create(24 << 30, 4, 8)

    def __del__(self):
        hom.hom_server_destroy(self.s)


def prepare(case, seed):
    if case["kind"] == "serve":
        return {"kind": "serve", "server": _Server(), "requests": _requests(case, seed)}
    single = case["precision"] == "fp32"
    precision = hom.HOM_FP32_REFINE if single else hom.HOM_FP64
    stream = torch.cuda.Stream()   # the library and the caller's own operations share one stream
    if case["kind"] == "ls":
        H = hom.Homogenization(_step_material(case, seed), precision=precision, stream=stream.cuda_stream)
        eps, E = _step_inputs(case, seed)
        return {"kind": "ls", "handle": H, "stream": stream, "eps": eps, "E": E, "out": torch.empty_like(eps),
                "loads": case["loads"], "single": single}
    H = hom.Homogenization(_microstructure(case, seed), precision=precision, scheme=SCHEMES[case["scheme"]],
                           max_iter=5000, stream=stream.cuda_stream)
    return {"kind": "solve", "handle": H, "stream": stream, "loads": UNIT[: case["loads"]], "order": case["order"],
            "tol": case["tol"], "single": single}


# ---- one pass ----------------------------------------------------------------------------------------
def run(state):
    if state["kind"] == "serve":
        s = state["server"].s
        ids = [hom.hom_server_submit(s, ms, order, 1e-6) for ms, order in state["requests"]]
        res = [hom.hom_server_wait(s, i) for i in ids]
        if any(r["status"] for r in res):
            raise RuntimeError("a request failed: %s" % [r["message"] for r in res if r["status"]])
        out = {"c_eff": np.stack([r["c_eff"] for r in res]).astype(np.float32)}
        d1 = [r["d1"] for r in res if r["d1"] is not None]
        if d1:
            out["d1"] = np.stack(d1).astype(np.float32)
        return out
    H = state["handle"]
    with torch.cuda.stream(state["stream"]):
        if state["kind"] == "ls":
            hom.hom_ls_apply(H.h, state["loads"], state["eps"], state["E"], state["out"])
            return state["out"].float() if state["single"] else state["out"]
        info = H.solve(0, state["tol"], loads=state["loads"])
        out = {"c_eff": H.effective(0)}
        if state["order"] >= 1:
            info += H.solve(1, state["tol"])
            out["d1"] = H.effective(1)
        if any(i["status"] for i in info):
            raise RuntimeError("not converged: %s" % info)
        # the strain fields of the highest order solved (of the first six loads)
        fields = [H.field(state["order"], k, device=True) for k in range(len(state["loads"]))]
        if state["single"]:
            out = {k: v.astype(np.float32) for k, v in out.items()}
            fields = [f.float() for f in fields]
        out["strain"] = fields
        return out


# ---- what one pass cannot do without -----------------------------------------------------------------
def _iterations(case):
    """Krylov (or fixed-point) steps a load of this contrast takes to the tolerance, to the usual bounds."""
    kappa = case["contrast"] if case["contrast"] > 1.0 else 1.0 / case["contrast"] if case["contrast"] > 0 else 220.0
    digits = math.log(2.0 / case["tol"])
    if case["scheme"] == "basic":
        return max(4.0, 0.5 * kappa * digits)
    return max(4.0, 0.5 * math.sqrt(kappa) * digits)


def _step_work(voxels, elem):
    """One Lippmann-Schwinger step of one load: the strain read and the result written once; twelve real
    transforms, the polarization and the contraction."""
    return {"bytes": 12.0 * voxels * elem, "flops": 12 * 2.5 * voxels * math.log2(max(2, voxels)) + 100.0 * voxels}


def work(case):
    if case["kind"] == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for k in range(case["requests"]):
            n1, n2, n3 = _SERVE_GRIDS[(k + case["requests"]) % len(_SERVE_GRIDS)]
            w = work({"kind": "solve", "geometry": "spheres", "n1": n1, "n2": n2, "n3": n3, "precision": "fp32",
                      "contrast": math.sqrt(2.0 * case["max_contrast"]), "scheme": "cg", "loads": 6, "order": k % 2,
                      "tol": 1e-6})
            total = {q: total[q] + w[q] for q in total}
        return total
    voxels = case["n1"] * case["n2"] * case["n3"]
    if case["kind"] == "ls":
        w = _step_work(voxels * case["loads"], 8)
        return {"bytes": w["bytes"] + voxels, "flops": w["flops"]}
    elem = 4 if case["precision"] == "fp32" else 8
    solved = case["loads"] + (18 if case["order"] else 0)
    w = _step_work(voxels, elem)
    steps = _iterations(case) * solved * (2 if case["scheme"] == "bicgstab" else 1)
    fields = 6.0 * voxels * elem * case["loads"]
    return {"bytes": steps * w["bytes"] + voxels + fields, "flops": steps * w["flops"]}


# ---- the same results in 64 bits ---------------------------------------------------------------------
# Symmetric tensors are (11, 22, 33, 23, 13, 12) components here, fields [..., 6, N3, N2, N1].
_PAIRS = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
_IDX = [[0, 5, 4], [5, 1, 3], [4, 3, 2]]
_W = [1.0, 1.0, 1.0, 2.0, 2.0, 2.0]


class _Exact:
    def __init__(self, ms, tol=1e-10):
        self.tol = tol   # relative residual: far below what the compared solves ask for
        phase = ms.phase if isinstance(ms.phase, torch.Tensor) else torch.from_numpy(ms.phase).cuda()
        lame = torch.tensor(np.asarray(ms.lame), dtype=torch.float64, device="cuda")
        phase = phase.long()
        self.lam, self.mu = lame[:, 0][phase], lame[:, 1][phase]
        self.lam0, self.mu0 = ms.lam0, ms.mu0
        n3, n2, n1 = phase.shape
        self.shape = (n3, n2, n1)

        def wave(n, half):
            k = np.arange(n // 2 + 1) if half else np.fft.fftfreq(n, 1.0 / n)
            k = np.where(2 * np.abs(k) == n, 0, k) if n % 2 == 0 else k
            return torch.tensor(2.0 * math.pi * max(n1, n2, n3) / n * k, dtype=torch.float64, device="cuda")

        self.xi = [wave(n1, True)[None, None, :], wave(n2, False)[None, :, None], wave(n3, False)[:, None, None]]
        q = self.xi[0] ** 2 + self.xi[1] ** 2 + self.xi[2] ** 2
        self.iq = torch.where(q > 0, 1.0 / torch.where(q > 0, q, torch.ones_like(q)), torch.zeros_like(q))

    def stress(self, e):
        tr = self.lam * (e[..., 0, :, :, :] + e[..., 1, :, :, :] + e[..., 2, :, :, :])
        s = 2.0 * self.mu * e
        for i in range(3):
            s[..., i, :, :, :] += tr
        return s

    def c0_dot(self, a, b):
        """Voxel mean of a : C0 : b per load."""
        tr = (a[..., 0, :, :, :] + a[..., 1, :, :, :] + a[..., 2, :, :, :]) * \
             (b[..., 0, :, :, :] + b[..., 1, :, :, :] + b[..., 2, :, :, :])
        return self.lam0 * tr.mean(dim=(-3, -2, -1)) + 2.0 * self.mu0 * self.dot(a, b)

    def dot(self, a, b):
        return sum(w * (a[..., i, :, :, :] * b[..., i, :, :, :]).mean(dim=(-3, -2, -1)) for i, w in enumerate(_W))

    def times_xi(self, t):
        return [sum(t[..., _IDX[i][j], :, :, :] * self.xi[j] for j in range(3)) for i in range(3)]

    def gamma(self, t, g=None):
        """Gamma0 * (t + theta), i theta_hat xi = g_hat; t and g are real fields."""
        dims = (-3, -2, -1)
        w = self.times_xi(torch.fft.rfftn(t, dim=dims))
        if g is not None:
            gh = torch.fft.rfftn(g, dim=dims)
            w = [w[i] - 1j * gh[..., i, :, :, :] for i in range(3)]
        s = (w[0] * self.xi[0] + w[1] * self.xi[1] + w[2] * self.xi[2]) * self.iq
        c = (self.lam0 + self.mu0) / (self.lam0 + 2.0 * self.mu0)
        v = [(w[i] - c * s * self.xi[i]) * self.iq / (2.0 * self.mu0) for i in range(3)]
        e = torch.stack([v[i] * self.xi[j] + v[j] * self.xi[i] for i, j in _PAIRS], dim=-4)
        return torch.fft.irfftn(e, s=self.shape, dim=dims)

    def solve(self, b, most=3000):
        """CG on Gamma0 * (C : x) = b in the C0 product, all loads at once."""
        x, r = torch.zeros_like(b), b.clone()
        p = r.clone()
        rho = self.c0_dot(r, r)
        b2 = self.dot(b, b)
        for _ in range(most):
            q = self.gamma(self.stress(p))
            den = self.c0_dot(p, q)
            alpha = torch.where(den > 0, rho / torch.where(den > 0, den, torch.ones_like(den)), torch.zeros_like(den))
            x += alpha[..., None, None, None, None] * p
            r -= alpha[..., None, None, None, None] * q
            new = self.c0_dot(r, r)
            if bool((self.dot(r, r) <= self.tol * self.tol * b2).all()):
                break
            beta = torch.where(rho > 0, new / torch.where(rho > 0, rho, torch.ones_like(rho)), torch.zeros_like(rho))
            p = r + beta[..., None, None, None, None] * p
            rho = new
        return x

    def order0(self, loads):
        """(strain fluctuations, stresses) of Mandel loads."""
        e = torch.tensor(np.asarray(loads), dtype=torch.float64, device="cuda") / _mandel()
        e = e[:, :, None, None, None].expand(-1, -1, *self.shape)
        x = self.solve(-self.gamma(self.stress(e)))
        return x, self.stress(x + e)

    def order1(self, x0, s0):
        """(strain fluctuations, stresses) of the 18 loads of order 1, load 3 A + k."""
        eh = torch.fft.rfftn(x0, dim=(-3, -2, -1))
        w = self.times_xi(eh)
        s = (w[0] * self.xi[0] + w[1] * self.xi[1] + w[2] * self.xi[2]) * self.iq
        u = torch.stack([-1j * (2.0 * w[i] - s * self.xi[i]) * self.iq for i in range(3)], dim=-4)
        u = torch.fft.irfftn(u, s=self.shape, dim=(-3, -2, -1))
        t = torch.zeros((18, 6) + self.shape, dtype=torch.float64, device="cuda")
        g = torch.zeros((18, 3) + self.shape, dtype=torch.float64, device="cuda")
        for a in range(6):
            for k in range(3):
                for i in range(3):
                    t[3 * a + k, _IDX[i][k]] += u[a, i] * (1.0 if i == k else 0.5)
                    g[3 * a + k, i] = s0[a, _IDX[i][k]]
        p = self.stress(t)
        x = self.solve(-self.gamma(p, g))
        return x, self.stress(x) + p


def _mandel():
    """Factors from tensor components to Mandel components."""
    return torch.tensor(_W, dtype=torch.float64, device="cuda").sqrt()


def _mandel_field(x):
    return x * _mandel()[:, None, None, None]


def _mean_mandel(s):
    return (s.mean(dim=(-3, -2, -1)) * _mandel()).T.contiguous()


def exact(case, seed):
    if case["kind"] == "serve":
        c_eff, d1 = [], []
        for ms, order in _requests(case, seed):
            pb = _Exact(ms)
            x0, s0 = pb.order0(UNIT)
            c_eff.append(_mean_mandel(s0))
            if order:
                d1.append(_mean_mandel(pb.order1(x0, s0)[1]))
        out = {"c_eff": torch.stack(c_eff)}
        if d1:
            out["d1"] = torch.stack(d1)
        return out
    if case["kind"] == "ls":
        ms = _step_material(case, seed)
        pb = _Exact(ms)
        eps, E = _step_inputs(case, seed)
        out = torch.empty_like(eps)
        for k in range(case["loads"]):
            e = eps[k] / _mandel()[:, None, None, None]
            e = e + (torch.tensor(E[k], dtype=torch.float64, device="cuda") / _mandel())[:, None, None, None]
            tau = pb.stress(e)
            tr = ms.lam0 * (e[0] + e[1] + e[2])
            tau -= 2.0 * ms.mu0 * e
            tau[:3] -= tr
            out[k] = _mandel_field(-pb.gamma(tau))
        return out
    voxels = case["n1"] * case["n2"] * case["n3"]
    if voxels * (case["loads"] + 3 * case["order"] * 6) > 24 << 20:
        return None   # minutes in 64 bits
    pb = _Exact(_microstructure(case, seed), 1e-10 if case["precision"] == "fp32" else 1e-13)
    if voxels > 1 << 21:   # load by load, for the memory
        parts = [pb.order0(UNIT[k:k + 1]) for k in range(case["loads"])]
        return {"c_eff": torch.cat([_mean_mandel(s) for _, s in parts], dim=1),
                "strain": [_mandel_field(x[0]) for x, _ in parts]}
    x, s = pb.order0(UNIT[: case["loads"]])
    out = {"c_eff": _mean_mandel(s)}
    if case["order"]:
        x, s = pb.order1(x, s)
        out["d1"] = _mean_mandel(s)
    out["strain"] = [_mandel_field(x[k]) for k in range(case["loads"])]
    return out
