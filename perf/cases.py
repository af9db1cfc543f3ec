"""Workloads of the single-layer BEM library as its users run them, with plain 64-bit references.

A case is one of five kinds:

* ``apply``: one application of the compressed Galerkin operator to ``nrhs`` vectors
  (``ibem_matvec``), the step that every Krylov iteration repeats;
* ``batch``: one application of many uneven instances together (``ibem_batch_matvec``);
* ``potential``: the field of ``nrhs`` densities at points off the surface, by the
  direct sum (``ibem_potential``) or with the interpolated far field
  (``ibem_potential_fmm``);
* ``network``: the learned preconditioner's network, inference or one
  forward and backward pass of its training, in BF16;
* ``scatter``: a whole sound-soft scattering computation, from the surface to the
  scattered field (create, assemble, right-hand side, solve, potential).

All surfaces are spheres of six cube-sphere patches.  The outputs of the FP32
operator are handed on as float32, those of the BF16 network as bfloat16: the
accuracy that these paths compute with.
"""
import math

import numpy as np
import torch

from paper_1708_09162_gb300 import ibem

ETA = 1.6
GAUSS = 8
POINT_RADIUS = 3.0


def listed():
    return [
        # The smallest operator that the tests and a first trial use: launches and latency.
        dict(name="laplace_p2_m2", kind="apply", kernel="laplace", kappa=0.0, p=2, m=2, q=6, nrhs=1,
             precision="fp64", coupling="df", store=False),
        # A converged electrostatics mesh inside conjugate gradients: stored double-float coupling.
        dict(name="laplace_p3_m5", kind="apply", kernel="laplace", kappa=0.0, p=3, m=5, q=6, nrhs=1,
             precision="fp64", coupling="df", store=False),
        # One incident wave inside GMRES on an ordinary mesh: stored complex coupling.
        dict(name="helmholtz_p2_m4", kind="apply", kernel="helmholtz", kappa=4.0, p=2, m=4, q=6, nrhs=1,
             precision="fp64", coupling="df", store=False),
        # The benchmark's scattering operator a level down, FP64-accurate, 64 incident waves: the largest step.
        dict(name="helmholtz_p2_m5_r64", kind="apply", kernel="helmholtz", kappa=4.0, p=2, m=5, q=8, nrhs=64,
             precision="fp64", coupling="sliced", store=False),
        # The inner operator of a mixed-precision solve with 16 waves, coupling generated per application.
        dict(name="helmholtz_fp32_m5_r16", kind="apply", kernel="helmholtz", kappa=4.0, p=2, m=5, q=8, nrhs=16,
             precision="fp32", coupling="sliced", store=False),
        # The same with 64 waves and the coupling stored once, as long solves keep it.
        dict(name="helmholtz_fp32_stored_m5_r64", kind="apply", kernel="helmholtz", kappa=4.0, p=2, m=5, q=8,
             nrhs=64, precision="fp32", coupling="sliced", store=True),
        # Many small uneven problems in one application.
        dict(name="batch_8", kind="batch", count=8, m_max=4, plan=5),
        # The scattered field of 64 solved densities at 200 points, direct sum over all Gauss points.
        dict(name="potential_m5_r64", kind="potential", kernel="helmholtz", kappa=4.0, p=2, m=5, q=8, nrhs=64,
             points=200, far=False),
        # A field map: many points, few densities, interpolated far field.
        dict(name="potential_far_m6_r4", kind="potential", kernel="helmholtz", kappa=4.0, p=2, m=6, q=8, nrhs=4,
             points=5000, far=True),
        # Preconditioner inference for 16 right-hand sides at level 7 (6 patches of 130 x 130 pixels each).
        dict(name="network_forward_130", kind="network", images=96, height=130, width=130, gradients=False),
        # A training minibatch of 16 vectors at level 5.
        dict(name="network_gradients_34", kind="network", images=96, height=34, width=34, gradients=True),
        # From the surface to the scattered field of 8 waves on a small mesh.
        dict(name="scatter_p2_m3_r8", kind="scatter", kappa=4.0, p=2, m=3, q=6, nrhs=8, points=100),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["apply", "apply", "apply", "apply", "batch", "potential", "potential", "network", "network",
                       "scatter"])
    kappa = round(rng.uniform(1.0, 8.0), 3)
    if kind == "apply":
        kernel = rng.choice(["laplace", "helmholtz"])
        precision = rng.choice(["fp64", "fp32"])
        nrhs = log_int(1, 64)
        wide = kernel == "helmholtz" and nrhs >= 4
        m = rng.randint(1, 5 if kernel == "laplace" else 4 if nrhs < 16 else 5)
        p = rng.randint(1, 3) if m > 2 else rng.randint(0, 4)
        store = kernel == "helmholtz" and precision == "fp32" and nrhs >= 16 and rng.random() < 0.5
        return dict(kind="apply", kernel=kernel, kappa=kappa if kernel == "helmholtz" else 0.0, p=p, m=m,
                    q=8 if wide else rng.randint(4, 7), nrhs=nrhs, precision=precision,
                    coupling="sliced" if wide else "df", store=store)
    if kind == "batch":
        return dict(kind="batch", count=log_int(2, 10), m_max=rng.randint(3, 4), plan=rng.randint(0, 10 ** 6))
    if kind == "potential":
        far = rng.random() < 0.5
        return dict(kind="potential", kernel=rng.choice(["laplace", "helmholtz"]), kappa=kappa, p=rng.randint(1, 3),
                    m=rng.randint(2, 6 if far else 5), q=rng.randint(4, 8), nrhs=log_int(1, 64),
                    points=log_int(10, 5000 if far else 400), far=far)
    if kind == "network":
        gradients = rng.random() < 0.5
        n = log_int(8, 66 if gradients else 130)
        return dict(kind="network", images=log_int(1, 96), height=n, width=n if rng.random() < 0.7 else log_int(8, n),
                    gradients=gradients)
    return dict(kind="scatter", kappa=kappa, p=rng.randint(1, 2), m=rng.randint(1, 3), q=rng.randint(4, 7),
                nrhs=log_int(1, 12), points=log_int(10, 200))


# ---- what a program holds before the call -------------------------------------------
class Held:
    """Library objects of one program, released with it."""

    def __init__(self):
        self.handles, self.batch, self.network = [], None, None

    def __del__(self):
        if self.batch is not None:
            ibem.ibem_batch_destroy(self.batch)
        if self.network is not None:
            ibem.ibem_cnn_destroy(self.network)
        for h in self.handles:
            ibem.ibem_destroy(h)


COUPLING = {"df": ibem.IBEM_COUPLING_DF, "sliced": ibem.IBEM_COUPLING_SLICED, "none": ibem.IBEM_COUPLING_NONE}


def _params(case, coupling="df", store=False):
    helm = case["kernel"] == "helmholtz"
    return ibem.make_params(case["p"], case["m"], q_cheb=case["q"], eta=ETA,
                            kernel=ibem.IBEM_HELMHOLTZ if helm else ibem.IBEM_LAPLACE,
                            kappa=case["kappa"] if helm else 0.0, gauss_regular=GAUSS, gauss_singular=8,
                            fp64_coupling=COUPLING[coupling],
                            fp32_coupling=ibem.IBEM_FP32_COUPLING_STORE if store else
                            ibem.IBEM_FP32_COUPLING_GENERATE)


def _ndof(case):
    return 6 * (2 ** case["m"] + case["p"]) ** 2


def _vectors(rng, case):
    """Seeded normal coefficient vectors [nrhs][ndof] (complex: [..][2])."""
    shape = (case["nrhs"], _ndof(case)) + ((2,) if case["kernel"] == "helmholtz" else ())
    return rng.normal(size=shape)


def _directions(rng, n):
    d = rng.normal(size=(n, 3))
    return d / np.linalg.norm(d, axis=1)[:, None]


def _batch_plan(case):
    """The instances of a batch: levels 2 to m_max, degrees 1 to 3, both kernels, 1 to 16
    right-hand sides, radii from 0.5 to 2."""
    rng = np.random.default_rng(case["plan"])
    out = []
    for _ in range(case["count"]):
        helm = int(rng.integers(0, 2))
        out.append(dict(kernel="helmholtz" if helm else "laplace", kappa=float(rng.uniform(2.0, 8.0)) if helm else 0.0,
                        p=int(rng.integers(1, 4)), m=int(rng.integers(2, case["m_max"] + 1)),
                        q=int(rng.choice([6, 8])), nrhs=int(rng.integers(1, 17)),
                        radius=float(rng.uniform(0.5, 2.0))))
    return out


def _network_parameters(rng, channels=32):
    """He-initialised parameters, W[cout][cin][3][3] then bias, the last layer scaled by 1/4."""
    out = []
    layers = [(2, channels), (channels, channels), (channels, channels), (channels, 2)]
    for i, (cin, cout) in enumerate(layers):
        w = rng.normal(size=cout * cin * 9) * math.sqrt(2.0 / (9 * cin)) * (0.25 if i == 3 else 1.0)
        out += [w, 0.05 * rng.normal(size=cout)]
    return np.concatenate(out).astype(np.float32)


def _inputs(case, seed):
    """The seeded inputs of a case, as host arrays: what both the library and the reference start from."""
    rng = np.random.default_rng([17, seed])
    if case["kind"] == "apply":
        return {"x": _vectors(rng, case)}
    if case["kind"] == "batch":
        return {"x": [_vectors(rng, inst) for inst in _batch_plan(case)]}
    if case["kind"] == "potential":
        w = _vectors(rng, case)
        return {"w": w, "points": POINT_RADIUS * _directions(rng, case["points"]) * rng.uniform(0.5, 1.0, size=(case["points"], 1))}
    if case["kind"] == "network":
        theta = _network_parameters(rng)
        shape = (case["images"], 2, case["height"], case["width"])
        return {"theta": theta, "image": rng.standard_normal(shape, dtype=np.float32),
                "target": rng.standard_normal(shape, dtype=np.float32)}
    return {"waves": _directions(rng, case["nrhs"]), "points": POINT_RADIUS * _directions(rng, case["points"])}


def prepare(case, seed):
    held, inp = Held(), _inputs(case, seed)
    s = {"case": case, "held": held}
    gpu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    if case["kind"] == "apply":
        h = ibem.ibem_create(ibem.sphere_patches(), _params(case, case["coupling"], case["store"]))
        held.handles.append(h)
        ibem.ibem_assemble(h)
        s["x"] = gpu(inp["x"])
        s["y"] = torch.empty_like(s["x"])
        s["precision"] = ibem.IBEM_FP64 if case["precision"] == "fp64" else ibem.IBEM_FP32
    elif case["kind"] == "batch":
        plan = _batch_plan(case)
        s["stream"] = torch.cuda.Stream()
        for inst in plan:
            h = ibem.ibem_create(ibem.sphere_patches(inst["radius"]), _params(inst, "none"))
            held.handles.append(h)
            ibem.ibem_assemble(h)
        held.batch = ibem.ibem_batch_create(held.handles, [inst["nrhs"] for inst in plan], s["stream"])
        s["x"] = gpu(np.concatenate([x.reshape(-1) for x in inp["x"]]))
        s["y"] = torch.empty_like(s["x"])
    elif case["kind"] == "potential":
        held.handles.append(ibem.ibem_create(ibem.sphere_patches(), _params(case)))
        s["w"], s["points"] = gpu(inp["w"]), gpu(inp["points"])
        s["u"] = torch.empty((case["nrhs"], case["points"]) + inp["w"].shape[2:], dtype=torch.float64, device="cuda")
    elif case["kind"] == "network":
        held.network = ibem.ibem_cnn_create(32, seed=1)
        ibem.ibem_cnn_params(held.network, inp["theta"])
        s["image"], s["target"] = gpu(inp["image"]), gpu(inp["target"])
        s["out"] = torch.empty_like(s["image"])
    else:
        s["waves"], s["points"] = gpu(inp["waves"]), gpu(inp["points"])
    return s


# ---- one pass ---------------------------------------------------------------------------
def run(state):
    case, held = state["case"], state["held"]
    if case["kind"] == "apply":
        ibem.ibem_matvec(held.handles[0], state["x"], state["y"], case["nrhs"], state["precision"])
        return state["y"] if case["precision"] == "fp64" else state["y"].float()
    if case["kind"] == "batch":
        here = torch.cuda.current_stream()
        state["stream"].wait_stream(here)
        ibem.ibem_batch_matvec(held.batch, state["x"], state["y"])
        here.wait_stream(state["stream"])
        return state["y"].float()
    if case["kind"] == "potential":
        call = ibem.ibem_potential_fmm if case["far"] else ibem.ibem_potential
        call(held.handles[0], state["w"], case["nrhs"], state["points"], state["u"])
        return state["u"]
    if case["kind"] == "network":
        if case["gradients"]:
            loss, grad = ibem.ibem_cnn_gradients(held.network, state["image"], state["target"], ibem.IBEM_BF16)
            return {"loss": torch.tensor(loss).bfloat16(), "grad": torch.from_numpy(grad).bfloat16()}
        ibem.ibem_cnn_forward(held.network, state["image"], state["out"], ibem.IBEM_BF16)
        return state["out"].bfloat16()
    return _scatter(case, state["waves"], state["points"])


def _scatter(case, waves, points):
    """Sound-soft scattering of plane waves: g = -e^{i kappa d.x} on the surface, solve, evaluate."""
    n = case["nrhs"]
    h = ibem.ibem_create(ibem.sphere_patches(), _params(dict(case, kernel="helmholtz")))
    try:
        ibem.ibem_assemble(h)
        info = ibem.ibem_get_info(h)
        xyz = torch.empty((info.n_quad_points, 3), dtype=torch.float64, device="cuda")
        ibem.ibem_quad_points(h, xyz)
        phase = case["kappa"] * (waves @ xyz.T)
        g = -torch.stack((torch.cos(phase), torch.sin(phase)), dim=-1).contiguous()
        b = torch.empty((n, info.ndof, 2), dtype=torch.float64, device="cuda")
        ibem.ibem_rhs(h, g, n, b)
        w = torch.empty_like(b)
        ibem.ibem_solve(h, b, w, n, rtol=1e-11, maxit=2000, precond=ibem.IBEM_PRECOND_BLOCK_JACOBI)
        u = torch.empty((n, points.shape[0], 2), dtype=torch.float64, device="cuda")
        ibem.ibem_potential(h, w, n, points, u)
    finally:
        ibem.ibem_destroy(h)
    return {"density": w, "field": u}


# ---- what a pass cannot do without -----------------------------------------------------
def _operator_work(case, kept):
    """Bytes and operations of one application.  The near blocks are read; of the coupling, what the
    handle keeps (``kept`` bytes per far block) is read and the rest is evaluated."""
    helm = case["kernel"] == "helmholtz"
    near, far = ibem.ibem_block_tree(ibem.sphere_patches(), _params(case))
    n_near, n_far, nb, q2 = len(near), len(far), (case["p"] + 1) ** 2, case["q"] ** 2
    word = (8 if case.get("precision") == "fp64" else 4) * (2 if helm else 1)
    macs = case["nrhs"] * (n_near * nb * nb + n_far * q2 * q2)
    evaluate = 0 if kept else n_far * q2 * q2 * (20 if helm else 10)
    return {"bytes": n_near * nb * nb * word + n_far * kept + 16 * (2 if helm else 1) * case["nrhs"] * _ndof(case),
            "flops": macs * (8 if helm else 2) + evaluate}


def work(case):
    if case["kind"] == "apply":
        q4, kept = case["q"] ** 4, 0
        if case["precision"] == "fp64" and case["coupling"] == "df":
            kept = q4 * 16 if case["kernel"] == "helmholtz" else q4 * 4  # double-float; Laplace: one of two mirrored blocks
        elif case["store"]:
            kept = q4 * 4
        return _operator_work(case, kept)
    if case["kind"] == "batch":
        parts = [_operator_work(dict(inst, precision="fp32"), 0) for inst in _batch_plan(case)]
        return {k: sum(part[k] for part in parts) for k in ("bytes", "flops")}
    if case["kind"] == "potential":
        helm = case["kernel"] == "helmholtz"
        word, nq = 16 if helm else 8, 6 * 4 ** case["m"] * GAUSS ** 2
        bytes_ = word * case["nrhs"] * (_ndof(case) + case["points"]) + 24 * case["points"]
        if case["far"]:  # about 40 clusters of q^2 points for each point
            pairs = case["points"] * 40 * case["q"] ** 2
        else:
            pairs, bytes_ = case["points"] * nq, bytes_ + 32 * nq
        return {"bytes": bytes_, "flops": pairs * ((20 if helm else 10) + case["nrhs"] * (8 if helm else 2))}
    if case["kind"] == "network":
        pixels = case["images"] * case["height"] * case["width"]
        macs = 9 * (2 * 32 + 32 * 32 + 32 * 32 + 32 * 2)
        return {"bytes": pixels * 16, "flops": pixels * 2 * macs * (3 if case["gradients"] else 1)}
    # scatter: the assembly's kernel evaluations (regular pairs alone) and some 30 applications
    op = _operator_work(dict(case, kernel="helmholtz", precision="fp64"), case["q"] ** 4 * 16)
    near, _ = ibem.ibem_block_tree(ibem.sphere_patches(), _params(dict(case, kernel="helmholtz")))
    return {"bytes": 30 * op["bytes"], "flops": 30 * op["flops"] + len(near) * GAUSS ** 4 * 20.0}


# ---- plain 64-bit references --------------------------------------------------------------
FACES = np.array([  # n, t1, t2 of the cube-sphere faces +x, -x, +y, -y, +z, -z
    [[1, 0, 0], [0, 1, 0], [0, 0, 1]], [[-1, 0, 0], [0, 0, 1], [0, 1, 0]], [[0, 1, 0], [0, 0, 1], [1, 0, 0]],
    [[0, -1, 0], [1, 0, 0], [0, 0, 1]], [[0, 0, 1], [1, 0, 0], [0, 1, 0]], [[0, 0, -1], [0, 1, 0], [1, 0, 0]]],
    dtype=np.float64)
# The symmetries of the square: (s, t) -> (a0 + a1 s + a2 t, b0 + b1 s + b2 t).
SYMMETRIES = [(0, 1, 0, 0, 0, 1), (1, 0, -1, 0, 1, 0), (1, -1, 0, 1, 0, -1), (0, 0, 1, 1, -1, 0),
              (0, 0, 1, 0, 1, 0), (1, -1, 0, 0, 0, 1), (1, 0, -1, 1, -1, 0), (0, 1, 0, 1, 0, -1)]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _gauss(n):
    t, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (t + 1.0), 0.5 * w


def _tensor(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(_device())


def _sphere(radius, patch, u, v):
    """Points and surface measure; u, v: tensors, patch: integer tensor that broadcasts against them."""
    frames = _tensor(FACES)[patch]
    n, t1, t2 = frames[..., 0, :], frames[..., 1, :], frames[..., 2, :]
    c = n + (2.0 * u - 1.0)[..., None] * t1 + (2.0 * v - 1.0)[..., None] * t2
    r2 = (c * c).sum(-1)
    # F = R c / |c|; the measure of the central projection of the plane at distance 1, twice the parameter each way
    return radius * c / r2.sqrt()[..., None], 4.0 * radius ** 2 / (r2 * r2.sqrt())


class Surface:
    """B-splines, trees and rules of one discretised sphere, from the definitions (no nested bases)."""

    def __init__(self, case, radius=1.0):
        self.p, self.m, self.q, self.radius = case["p"], case["m"], case["q"], radius
        self.kappa = case["kappa"] if case["kernel"] == "helmholtz" else None
        self.ne, self.n1 = 2 ** self.m, 2 ** self.m + self.p
        self.knots = np.array([0.0] * (self.p + 1) + [i / self.ne for i in range(1, self.ne)] + [1.0] * (self.p + 1))
        a = np.arange(self.q)
        self.nodes = 0.5 * (1.0 - np.cos((2 * a + 1) * np.pi / (2 * self.q)))
        self.balls = [self._balls(level) for level in range(self.m + 1)]
        self.dtype = torch.float64 if self.kappa is None else torch.complex128

    def cells(self, level):
        """(patch, ix, iy) of the clusters of a level; index patch 4^l + iy 2^l + ix."""
        n = 2 ** level
        c = np.arange(6 * n * n)
        return c // (n * n), c % n, (c // n) % n

    def _balls(self, level):
        patch, ix, iy = self.cells(level)
        g = np.linspace(0.0, 1.0, 5)
        su, sv = np.meshgrid(g, g, indexing="xy")
        h = 1.0 / 2 ** level

        def points(s, t):
            f = FACES[patch][:, None]
            u, v = (ix[:, None] + s) * h, (iy[:, None] + t) * h
            c = f[:, :, 0] + (2 * u - 1)[..., None] * f[:, :, 1] + (2 * v - 1)[..., None] * f[:, :, 2]
            return self.radius * c / np.sqrt(np.sum(c * c, axis=-1))[..., None]

        mid = points(np.array([0.5]), np.array([0.5]))
        r = np.sqrt(np.max(np.sum((points(su.ravel(), sv.ravel()) - mid) ** 2, axis=-1), axis=1))
        if level == self.m:
            self.corners = points(np.array([0.0, 1.0, 1.0, 0.0]), np.array([0.0, 0.0, 1.0, 1.0]))
        return mid[:, 0], r

    def _children(self, level, c):
        n = 2 ** level
        patch, ix, iy = c // (n * n), c % n, (c // n) % n
        return np.stack([patch * 4 * n * n + (2 * iy + dy) * 2 * n + 2 * ix + dx for dy in (0, 1) for dx in (0, 1)], -1)

    def block_tree(self):
        """Near element pairs and, by level, the far cluster pairs; with the near pairs' distances and diameters."""
        far = []
        s, t = (a.ravel() for a in np.meshgrid(np.arange(6), np.arange(6), indexing="ij"))
        for level in range(self.m + 1):
            c, r = self.balls[level]
            d = np.sqrt(np.sum((c[s] - c[t]) ** 2, axis=-1)) - r[s] - r[t]
            dist, diam = np.maximum(d, 0.0), 2.0 * np.maximum(r[s], r[t])
            ok = ETA * diam < dist
            far.append((s[ok], t[ok]))
            s, t = s[~ok], t[~ok]
            if level < self.m:
                sc, tc = self._children(level, s), self._children(level, t)
                s, t = np.repeat(sc, 4, axis=1).ravel(), np.tile(tc, (1, 4)).ravel()
        return s, t, dist[~ok], diam[~ok], far

    def basis(self, i, x):
        """The p + 1 B-splines of the 1D element i at local coordinates x: (..., p + 1)."""
        u = (i + x) / self.ne
        knots = _tensor(self.knots)
        at = lambda k: knots[i + k] + torch.zeros_like(u)  # noqa: E731
        b = [torch.ones_like(u)]
        for d in range(1, self.p + 1):
            new, carry = [], torch.zeros_like(u)
            for r in range(d):
                right, left = at(self.p + 1 + r), at(self.p + 1 - d + r)
                f = b[r] / (right - left)
                new.append(carry + (right - u) * f)
                carry = (u - left) * f
            b = new + [carry]
        return torch.stack(b, -1)

    def element(self, e, s, t):
        """Points, measures and the (p + 1)^2 basis values of the elements e at local (s, t)."""
        patch, ix, iy = e // self.ne ** 2, e % self.ne, (e // self.ne) % self.ne
        F, k = _sphere(self.radius, patch, (ix + s) / self.ne, (iy + t) / self.ne)
        bu, bv = self.basis(ix, s), self.basis(iy, t)
        return F, k, (bv[..., :, None] * bu[..., None, :]).flatten(-2)

    def dofs(self, e):
        ix, iy, patch = e % self.ne, (e // self.ne) % self.ne, e // self.ne ** 2
        a = torch.arange(self.p + 1, device=e.device)
        j = (iy[:, None] + a)[:, :, None] * self.n1 + (ix[:, None] + a)[:, None, :]
        return (patch[:, None, None] * self.n1 ** 2 + j).flatten(1)

    def green(self, X, Y):
        d = X - Y
        r = (d * d).sum(-1).sqrt()
        if self.kappa is None:
            return 1.0 / (4.0 * math.pi * r)
        return torch.polar(1.0 / (4.0 * math.pi * r), self.kappa * r)

    def moments(self, level):
        """mu[i, a, j] = int over the level's 1D cluster i of L_a b_j."""
        ng, per = math.ceil((self.q + self.p) / 2) + 1, 2 ** (self.m - level)
        g, w = _gauss(ng)
        i = torch.arange(self.ne, device=_device())
        b = self.basis(i[:, None], _tensor(g)[None].expand(self.ne, ng)) * _tensor(w)[:, None] / self.ne
        local = ((np.arange(self.ne) % per)[:, None] + g) / per
        L = np.ones((self.ne, ng, self.q))
        for a in range(self.q):
            for c in range(self.q):
                if c != a:
                    L[..., a] *= (local - self.nodes[c]) / (self.nodes[a] - self.nodes[c])
        part = torch.einsum("ega,egt->eat", _tensor(L), b)
        mu = torch.zeros((2 ** level, self.q, self.n1), dtype=torch.float64, device=_device())
        for k in range(self.p + 1):
            mu.index_put_((i[:, None] // per, torch.arange(self.q, device=_device())[None], (i + k)[:, None]),
                          part[..., k], accumulate=True)
        return mu.to(self.dtype)

    def node_points(self, level):
        zu, zv = np.meshgrid(self.nodes, self.nodes, indexing="xy")
        patch, ix, iy = (_tensor(a)[:, None] for a in self.cells(level))
        h = 1.0 / 2 ** level
        return _sphere(self.radius, patch, (ix + _tensor(zu.ravel())) * h, (iy + _tensor(zv.ravel())) * h)

    def forward(self, level, x):
        """Moments of every cluster of a level: x (N, R) -> (clusters, q^2, R)."""
        mu = self.moments(level).flatten(0, 1)
        X = x.reshape(6, self.n1, self.n1, -1)
        Z = torch.einsum("cu,pvur->pvcr", mu, X)
        Z = torch.einsum("dv,pvcr->pdcr", mu, Z).reshape(6, 2 ** level, self.q, 2 ** level, self.q, -1)
        return Z.permute(0, 1, 3, 2, 4, 5).reshape(6 * 4 ** level, self.q ** 2, -1)

    def backward(self, level, y):
        mu = self.moments(level).flatten(0, 1)
        n = 2 ** level
        Z = y.reshape(6, n, n, self.q, self.q, -1).permute(0, 1, 3, 2, 4, 5).reshape(6, n * self.q, n * self.q, -1)
        Z = torch.einsum("cu,pdcr->pdur", mu, Z)
        return torch.einsum("dv,pdur->pvur", mu, Z).reshape(6 * self.n1 ** 2, -1)

    # -- near field -----------------------------------------------------------------------
    def _rules(self):
        """Touching pairs: (x1, x2, y1, y2, weight) of the identical, common-edge and common-vertex rules."""
        g, w = _gauss(8)
        a, b, c, d = (v.ravel() for v in np.meshgrid(g, g, g, g, indexing="ij"))
        W = np.multiply.outer(np.multiply.outer(w, w), np.multiply.outer(w, w)).ravel()

        def ordered(z, s, swap):
            lo = (1.0 - z) * s
            return (lo + z, lo) if swap else (lo, lo + z)

        same, edge, vertex = [], [], []
        for z1, z2 in ((a, a * b), (a * b, a)):
            for o1 in (0, 1):
                for o2 in (0, 1):
                    x1, y1 = ordered(z1, c, o1)
                    x2, y2 = ordered(z2, d, o2)
                    same.append((x1, x2, y1, y2, W * a * (1 - z1) * (1 - z2)))
        for x1, y1, z in ((a, a * b, a * c), (a * b, a, a * c), (a * b, a * c, a)):
            for o in (0, 1):
                x2, y2 = ordered(z, d, o)
                edge.append((x1, x2, y1, y2, W * a * a * (1 - z)))
        for k in range(4):
            co = [a * b, a * c, a * d]
            co.insert(k, a)
            vertex.append((*co, W * a ** 3))
        return [tuple(np.concatenate(col) for col in zip(*rule)) for rule in (same, edge, vertex)]

    def _touching(self, s, t, diam):
        """Class 0 (edge 1, vertex 2) and orientation of touching pairs, -1 for pairs that do not touch."""
        P, Q = self.corners[s], self.corners[t]
        meet = np.sqrt(np.sum((P[:, :, None] - Q[:, None]) ** 2, axis=-1)) <= (1e-10 * diam)[:, None, None]
        count = meet.sum((1, 2))
        cls = np.where(s == t, 0, np.where(count >= 2, 1, np.where(count == 1, 2, -1)))
        ids = {(0, 0): 0, (1, 0): 1, (1, 1): 2, (0, 1): 3}
        corner = [[ids[(a0 + a1 * u + a2 * v, b0 + b1 * u + b2 * v)] for u, v in ((0, 0), (0, 1))]
                  for a0, a1, a2, b0, b1, b2 in SYMMETRIES]
        ka, kb = np.full(len(s), -1), np.full(len(s), -1)
        for i in range(8):
            for j in range(8):
                ok = meet[:, corner[i][0], corner[j][0]] & ((cls != 1) | meet[:, corner[i][1], corner[j][1]])
                new = ok & (ka < 0) & (cls > 0)
                ka[new], kb[new] = i, j
        ka[cls == 0], kb[cls == 0] = 0, 0
        return cls, ka, kb

    def _pair_blocks(self, s, t, rule):
        """Blocks of pairs with a joint rule over both elements."""
        x1, x2, y1, y2, w = (_tensor(v)[None] for v in rule)
        F, k, b = self.element(s[:, None], x1.expand(len(s), -1), x2.expand(len(s), -1))
        G, l, c = self.element(t[:, None], y1.expand(len(s), -1), y2.expand(len(s), -1))
        wk = self.green(F, G) * (k * l * w / self.ne ** 4)
        return b.to(self.dtype).transpose(1, 2) @ (wk[..., None] * c)

    def _product_blocks(self, s, t, tables):
        """Blocks of pairs with one rule on each element (points, weighted measures and basis values by element)."""
        F, k, b = tables
        wk = self.green(F[s][:, :, None], F[t][:, None]) * (k[s][:, :, None] * k[t][:, None])
        return b[s].to(self.dtype).transpose(1, 2) @ (wk @ b[t].to(self.dtype))

    def _gauss_tables(self, split):
        g, w = _gauss(GAUSS)
        u, v = np.meshgrid(g, g, indexing="xy")
        wt = np.outer(w, w).ravel()
        cells = [(0.0, 0.0), (0.5, 0.0), (0.0, 0.5), (0.5, 0.5)]
        if split:
            u, v = (np.concatenate([o[k] + 0.5 * z.ravel() for o in cells]) for k, z in ((0, u), (1, v)))
            wt = np.tile(wt / 4.0, 4)
        e = torch.arange(6 * self.ne ** 2, device=_device())[:, None]
        shape = (len(e), wt.size)
        F, k, b = self.element(e, _tensor(u.ravel())[None].expand(shape), _tensor(v.ravel())[None].expand(shape))
        return F, k * _tensor(wt) / self.ne ** 2, b

    def near_blocks(self, s, t, dist, diam):
        """(targets, sources, blocks) in chunks, over all near pairs."""
        touch = np.full(len(s), -1)
        ka, kb = touch.copy(), touch.copy()
        at = np.nonzero(dist <= 1e-9 * diam)[0]
        touch[at], ka[at], kb[at] = self._touching(s[at], t[at], diam[at])
        rules = self._rules()
        for cls in range(3):
            for i in range(8):
                for j in range(8):
                    pick = np.nonzero((touch == cls) & (ka == i) & (kb == j))[0]
                    if not len(pick):
                        continue
                    x1, x2, y1, y2, w = rules[cls]
                    a, b = SYMMETRIES[i], SYMMETRIES[j]
                    rule = (a[0] + a[1] * x1 + a[2] * x2, a[3] + a[4] * x1 + a[5] * x2,
                            b[0] + b[1] * y1 + b[2] * y2, b[3] + b[4] * y1 + b[5] * y2, w)
                    for part in np.array_split(pick, -(-len(pick) * w.size // 2_000_000)):
                        ss, tt = _tensor(s[part]), _tensor(t[part])
                        yield ss, tt, self._pair_blocks(ss, tt, rule)
        for split in (True, False):
            pick = np.nonzero((touch < 0) & ((dist < 0.5 * diam) == split))[0]
            if len(pick):
                tables = self._gauss_tables(split)
                for part in np.array_split(pick, -(-len(pick) // (256 if split else 4096))):
                    ss, tt = _tensor(s[part]), _tensor(t[part])
                    yield ss, tt, self._product_blocks(ss, tt, tables)

    # -- operator and potential -------------------------------------------------------------
    def apply(self, x):
        """The compressed Galerkin matrix times x (N, R)."""
        s, t, dist, diam, far = self.block_tree()
        E = 6 * self.ne ** 2
        y = torch.zeros_like(x)
        dofs = self.dofs(torch.arange(E, device=_device()))
        near = torch.zeros((E, dofs.shape[1], x.shape[1]), dtype=x.dtype, device=x.device)
        for ss, tt, blocks in self.near_blocks(s, t, dist, diam):
            near.index_add_(0, ss, blocks @ x[dofs[tt]])
        y.index_add_(0, dofs.flatten(), near.flatten(0, 1))
        del near
        for level, (s, t) in enumerate(far):
            if not len(s):
                continue
            xh = self.forward(level, x)
            yh = torch.zeros_like(xh)
            F, k = self.node_points(level)
            for part in np.array_split(np.arange(len(s)), -(-len(s) // 4096)):
                ss, tt = _tensor(s[part]), _tensor(t[part])
                K = self.green(F[ss][:, :, None], F[tt][:, None]) * (k[ss][:, :, None] * k[tt][:, None])
                yh.index_add_(0, ss, K @ xh[tt])
            y += self.backward(level, yh)
        return y

    def density(self, w):
        """Weighted density values at the Gauss points: points (E Q^2, 3) and values (E Q^2, R)."""
        F, k, b = self._gauss_tables(False)
        dofs = self.dofs(torch.arange(6 * self.ne ** 2, device=_device()))
        return F, k[..., None] * (b.to(self.dtype) @ w[dofs])

    def potential(self, w, points):
        F, d = self.density(w)
        F, d = F.flatten(0, 1), d.flatten(0, 1)
        u = torch.zeros((len(points), w.shape[1]), dtype=self.dtype, device=w.device)
        for a, b in zip(F.split(8192), d.split(8192)):
            u += self.green(points[:, None], a[None]) @ b
        return u

    def potential_far(self, w, points):
        """The walk of the cluster tree by point: an admissible cluster by its moments, an element that never
        is by its Gauss sum."""
        X = points.cpu().numpy()
        u = torch.zeros((len(X), w.shape[1]), dtype=self.dtype, device=w.device)
        pt, cl = (a.ravel() for a in np.meshgrid(np.arange(len(X)), np.arange(6), indexing="ij"))

        def add(pt, cl, F, values):
            for part in np.array_split(np.arange(len(pt)), -(-len(pt) * values[0].numel() // 20_000_000) or 1):
                i, c = _tensor(pt[part]), _tensor(cl[part])
                g = self.green(points[i][:, None], F[c])
                u.index_add_(0, i, (g[:, None] @ values[c])[:, 0])

        for level in range(self.m + 1):
            c, r = self.balls[level]
            ok = ETA * 2.0 * r[cl] < np.maximum(np.sqrt(np.sum((X[pt] - c[cl]) ** 2, axis=-1)) - r[cl], 0.0)
            if ok.any():
                F, k = self.node_points(level)
                add(pt[ok], cl[ok], F, k[..., None] * self.forward(level, w))
            pt, cl = pt[~ok], cl[~ok]
            if level < self.m:
                pt, cl = np.repeat(pt, 4), self._children(level, cl).ravel()
        if len(pt):
            add(pt, cl, *self.density(w))
        return u


def _columns(x):
    """[R][N] or [R][N][2] host values -> (N, R) on the device, real or complex."""
    x = _tensor(x)
    return (torch.view_as_complex(x) if x.dim() == 3 else x).T.contiguous()


def _rows(y):
    y = y.T.contiguous()
    return torch.view_as_real(y).contiguous() if y.is_complex() else y


def _network(theta, x):
    c, off = [(2, 32), (32, 32), (32, 32), (32, 2)], 0
    for i, (cin, cout) in enumerate(c):
        W = theta[off:off + cout * cin * 9].reshape(cout, cin, 3, 3)
        b = theta[off + cout * cin * 9:off + cout * cin * 9 + cout]
        off += cout * cin * 9 + cout
        x = torch.nn.functional.conv2d(x, W, b, padding=1)
        x = torch.relu(x) if i < 3 else x
    return x


def exact(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "apply":
        return _rows(Surface(case).apply(_columns(inp["x"])))
    if case["kind"] == "batch":
        return torch.cat([_rows(Surface(inst, inst["radius"]).apply(_columns(x))).flatten()
                          for inst, x in zip(_batch_plan(case), inp["x"])])
    if case["kind"] == "potential":
        s = Surface(case)
        return _rows((s.potential_far if case["far"] else s.potential)(_columns(inp["w"]), _tensor(inp["points"])))
    if case["kind"] == "network":
        theta = _tensor(inp["theta"]).double().requires_grad_(case["gradients"])
        if not case["gradients"]:
            return torch.cat([_network(theta, x.double()) for x in _tensor(inp["image"]).split(8)])
        loss = 0.0
        for x, y in zip(_tensor(inp["image"]).split(8), _tensor(inp["target"]).split(8)):
            part = ((_network(theta, x.double()) - y.double()) ** 2).sum() / (2 * case["images"])
            part.backward()
            loss += float(part)
        return {"loss": torch.tensor(loss, dtype=torch.float64), "grad": theta.grad}
    s = Surface(dict(case, kernel="helmholtz"))
    F, k, b = s._gauss_tables(False)
    g = -torch.polar(torch.ones((), dtype=torch.float64, device=F.device), case["kappa"] * (F @ _tensor(inp["waves"]).T))
    N = 6 * s.n1 ** 2
    rhs = torch.zeros((N, case["nrhs"]), dtype=s.dtype, device=F.device)
    rhs.index_add_(0, s.dofs(torch.arange(len(F), device=F.device)).flatten(),
                   (b.to(s.dtype).transpose(1, 2) @ (k[..., None] * g)).flatten(0, 1))
    A = s.apply(torch.eye(N, dtype=s.dtype, device=F.device))
    w = torch.linalg.solve(A, rhs)
    return {"density": _rows(w), "field": _rows(s.potential(w, _tensor(inp["points"])))}
