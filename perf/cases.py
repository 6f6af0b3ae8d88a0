"""The work that a user of this framework has it do, as cases that can be timed and compared.

Three ways in, as in the README and the benchmark:
  * `predict`: one space-time predictor per element of an isolated population, device buffers in and out
    (`poro_predict_dev`), for Biot's equations in the three precision forms and for the other systems in binary64;
  * `host`: the same end to end from pinned host memory (`poro_predict_host`);
  * `advance`: time stepping of a mesh (`poro_advance`: predictor, corrector, source, receivers), with one step
    for all elements or with clustered local time stepping, and the wavefield read back at the end.

`exact` states the same mathematics in plain 64-bit torch: basis and matrices by quadrature, the degree-block
solve with dense matrices, Riemann solver by eigenvectors.
"""
import math
from functools import lru_cache

import numpy as np
import torch

from paper_2108_10565_gb300 import _lib as L
from paper_2108_10565_gb300 import inputs

PRECISION = {"fp64": L.PORO_FP64, "tf32": L.PORO_FP32_REFINE, "bf16": L.PORO_BF16X3_REFINE}
SYSTEM = {"biot": L.PORO_SYSTEM_BIOT, "maxwell": L.PORO_SYSTEM_MAXWELL, "visco": L.PORO_SYSTEM_VISCOELASTIC,
          "subcell": L.PORO_SYSTEM_BIOT}
QUANTITIES = {"biot": 13, "maxwell": 6, "visco": 27, "subcell": 13}


def modes(N):
    return (N + 1) * (N + 2) * (N + 3) // 6


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smoke test's population: a handful of elements, launch and call overhead
        dict(name="predict fp64 N3 tiny", kind="predict", system="biot", precision="fp64", degree=3, elements=7, sweeps=1),
        # the benchmark's binary64 arm at the size of its profiles
        dict(name="predict fp64 N6", kind="predict", system="biot", precision="fp64", degree=6, elements=20000, sweeps=1),
        # the benchmark's headline form, the largest population here; not a multiple of anything
        dict(name="predict bf16 N6 large", kind="predict", system="biot", precision="bf16", degree=6, elements=40009, sweeps=1),
        # the tf32 form at a middle degree
        dict(name="predict tf32 N4", kind="predict", system="biot", precision="tf32", degree=4, elements=20011, sweeps=1),
        # the end-to-end leg of the benchmark: pinned host memory in and out, chunked pipeline
        dict(name="host bf16 N5", kind="host", system="biot", precision="bf16", degree=5, elements=16384, sweeps=1),
        # the small periodic point-source run (384 tetrahedra, degree 2): launches and latency
        dict(name="advance fp64 N2 small", kind="advance", mesh="periodic", boxes=4, precision="fp64", degree=2, clusters=1, cycles=10),
        # global time stepping in binary64 on a periodic cube, the corrector's profile workload scaled down
        dict(name="advance fp64 N5", kind="advance", mesh="periodic", boxes=10, precision="fp64", degree=5, clusters=1, cycles=2),
        # the layer over a half-space on a graded mesh, six rate-2 clusters, one step of the largest cluster
        dict(name="advance bf16 N3 LTS", kind="advance", mesh="layered", boxes=8, precision="bf16", degree=3, clusters=6, cycles=1),
        # one served run: box mesh with free surface, degree 6, two clusters
        dict(name="advance bf16 N6 served", kind="advance", mesh="box", boxes=6, precision="bf16", degree=6, clusters=2, cycles=2),
        # the other systems of the paper, binary64
        dict(name="predict maxwell N4", kind="predict", system="maxwell", precision="fp64", degree=4, elements=20000, sweeps=1),
        dict(name="predict visco N5", kind="predict", system="visco", precision="fp64", degree=5, elements=4001, sweeps=1),
        dict(name="predict subcell N4", kind="predict", system="subcell", precision="fp64", degree=4, elements=500, sweeps=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: populations of 1 to 40,000 elements (fewer for the costlier systems), meshes of
    162 to 13,824 tetrahedra, all degrees and precision forms."""
    kind = rng.choice(["predict"] * 5 + ["host"] + ["advance"] * 4)
    if kind == "advance":
        mesh = rng.choice(["periodic", "layered", "box"])
        precision = rng.choice(["fp64", "tf32", "bf16"])
        N = rng.randint(1, 6)
        top = {"periodic": 13 - N, "layered": 9 - N // 2, "box": 9 - N // 2}[mesh]
        boxes = rng.randint(3, top)
        clusters = 1 if mesh == "periodic" else rng.randint(1, 5)
        return dict(kind=kind, mesh=mesh, boxes=boxes, precision=precision, degree=N, clusters=clusters,
                    cycles=rng.randint(1, 4 if clusters < 3 else 1))
    system = "biot" if kind == "host" or rng.random() < 0.7 else rng.choice(["maxwell", "visco", "subcell"])
    precision = rng.choice(["fp64", "tf32", "bf16"]) if system == "biot" else "fp64"
    N = rng.randint(2, 6)
    top = {"biot": 40000, "maxwell": 30000, "visco": 4000, "subcell": 500}[system]
    if precision == "fp64" and N == 6:
        top = min(top, 16000)
    if system == "subcell" and N >= 5:
        top = 200
    sweeps = 2 if precision != "fp64" and rng.random() < 0.2 else 1
    return dict(kind=kind, system=system, precision=precision, degree=N, elements=_log_int(rng, 1, top), sweeps=sweeps)


# ------------------------------------------------------------------ inputs
def _population(case, seed):
    """Geometry, material rows, time steps (host) and the random initial modes (device)."""
    n, N, system = case["elements"], case["degree"], case["system"]
    rng = np.random.Generator(np.random.PCG64([seed, 1]))
    vert = inputs.random_tetrahedra(rng, n)
    if system == "biot":
        mat = inputs.perturbed_materials(rng, n)
        dt = L.poro_cfl_dt(N, vert, mat)
    elif system == "maxwell":
        mat = np.stack([rng.uniform(1.0, 4.0, n), rng.uniform(1.0, 2.0, n), rng.uniform(0.5, 1.5, n)], axis=1)
        dt = L.poro_cfl_dt_system(L.PORO_SYSTEM_MAXWELL, N, vert, mat)
    elif system == "visco":
        rho, cs = rng.uniform(2000.0, 3000.0, n), rng.uniform(1500.0, 3500.0, n)
        mu = rho * cs ** 2
        lam = rho * (cs * rng.uniform(1.7, 2.0, n)) ** 2 - 2 * mu
        om = np.tile(2 * np.pi * np.array([0.1, 1.0, 10.0]), (n, 1))
        mat = np.concatenate([rho[:, None], lam[:, None], mu[:, None], om, lam[:, None] * rng.uniform(0.005, 0.03, (n, 3)),
                              mu[:, None] * rng.uniform(0.005, 0.03, (n, 3))], axis=1)
        dt = L.poro_cfl_dt_system(L.PORO_SYSTEM_VISCOELASTIC, N, vert, mat)
    else:
        centre = inputs.perturbed_materials(rng, n, tie_skeleton=True)
        f = rng.uniform(0.9, 1.1, (n, 4, 10))
        f[:, :, 2] = f[:, :, 0]
        f[:, :, 3] = f[:, :, 0]
        mat = np.ascontiguousarray(centre[:, None, :] * f)
        dt = np.minimum.reduce([L.poro_cfl_dt(N, vert, np.ascontiguousarray(mat[:, v, :])) for v in range(4)])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    q0 = torch.randn((n, QUANTITIES[system], modes(N)), dtype=torch.float64, device="cuda", generator=gen)
    return vert, mat, dt, q0


def _mesh(case):
    """(mesh, materials, source, receivers) of a time-stepping case."""
    k = case["boxes"]
    w = np.zeros(13)
    if case["mesh"] == "periodic":
        mesh = inputs.kuhn_box_mesh(k)
        mats = np.tile(inputs.REFERENCE_MATERIAL, (mesh["tets"].shape[0], 1))
        w[9] = 1.0
        source = dict(x=np.array([0.5, 0.5, 0.5]), w=w, f0=1e4, t0=1e-4, amplitude=1.0)
        rec = np.random.Generator(np.random.PCG64(7)).uniform(0.1, 0.9, (4, 3))
    elif case["mesh"] == "layered":
        mesh, mats = inputs.layered_graded_mesh(k)
        source = dict(x=np.array([0.0, 0.0, -1010.0]), w=inputs.EXPLOSIVE_WEIGHTS, f0=5.0, t0=0.25, amplitude=1e9)
        rec = inputs.LOH_RECEIVERS
    else:
        mesh = inputs.uniform_box_mesh_for(24 * k ** 3)
        depth = -mesh["vertices"][mesh["tets"]].mean(axis=1)[:, 2]
        mats = np.where((depth < 2500.0)[:, None], inputs.LAYER_MATERIAL[None, :], inputs.HALFSPACE_MATERIAL[None, :])
        source = dict(x=np.array([9000.0, 9500.0, -4100.0]), w=inputs.EXPLOSIVE_WEIGHTS, f0=1.0, t0=1.2, amplitude=1e9)
        rec = np.array([[4000.0, 5000.0, -1.0], [12000.0, 9000.0, -1.0], [9100.0, 9600.0, -6000.0]])
    return mesh, np.ascontiguousarray(mats), source, rec


def _mesh_q0(case, seed, ne):
    return np.random.Generator(np.random.PCG64([seed, 2])).standard_normal((ne, 13, modes(case["degree"])))


class State:
    """A context and the buffers that a program keeps beside it."""

    def __init__(self, case):
        self.kind = case["kind"]
        self.ctx = L.poro_create(0, case["degree"], PRECISION[case["precision"]], system=SYSTEM[case.get("system", "biot")])

    def __del__(self):
        if getattr(self, "ctx", None):
            torch.cuda.synchronize()
            L.poro_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    s = State(case)
    N, B, T = case["degree"], modes(case["degree"]), case["degree"] + 1
    if case["kind"] == "advance":
        mesh, mats, src, rec = _mesh(case)
        L.poro_set_mesh(s.ctx, mesh["vertices"], mesh["tets"], mesh["neighbors"], mesh["face_tag"])
        L.poro_set_materials(s.ctx, mats)
        s.dt, _ = L.poro_set_clusters(s.ctx, 0.5, case["clusters"])
        L.poro_add_point_source(s.ctx, src["x"], src["w"], src["f0"], src["t0"], src["amplitude"])
        for x in rec:
            L.poro_add_receiver(s.ctx, x)
        ne = mesh["tets"].shape[0]
        L.poro_set_dofs(s.ctx, _mesh_q0(case, seed, ne))
        s.step = case["cycles"] * 2 ** (case["clusters"] - 1) * s.dt
        s.time = 0.0
        s.out = torch.empty((ne, 13, B), dtype=torch.float64, pin_memory=True).numpy()
        return s
    vert, mat, dt, q0 = _population(case, seed)
    if case["precision"] != "fp64":
        L.poro_set_refinement(s.ctx, case["sweeps"])
    {"biot": L.poro_set_isolated, "maxwell": L.poro_set_isolated_maxwell, "visco": L.poro_set_isolated_viscoelastic,
     "subcell": L.poro_set_isolated_subcell}[case["system"]](s.ctx, vert, mat, dt)
    s.n = case["elements"]
    if case["kind"] == "host":
        s.q0 = q0.cpu().pin_memory().numpy()
        s.out = torch.empty(q0.shape, dtype=torch.float64, pin_memory=True).numpy()
        return s
    s.q0 = q0
    s.qt = torch.empty(tuple(q0.shape) + (T,), dtype=torch.float64, device="cuda")
    s.i = torch.empty_like(q0)
    s.ptr = (s.q0.data_ptr(), s.qt.data_ptr(), s.i.data_ptr())
    return s


def run(s):
    if s.kind == "predict":
        L.poro_predict_dev(s.ctx, 0, s.n, *s.ptr, stream=torch.cuda.current_stream().cuda_stream)
        return {"predictor": s.qt, "integrated": s.i}
    if s.kind == "host":
        return {"integrated": L.poro_predict_host(s.ctx, s.q0, out=s.out)}
    s.time += s.step
    L.poro_advance(s.ctx, s.time)
    return {"dofs": L.poro_get_dofs(s.ctx, out=s.out)}


# ------------------------------------------------------------------ floors and tolerances
STAR = {"biot": 54, "maxwell": 12, "visco": 51, "subcell": 54}
#: structural non-zeros of the three matrices M^{-1} K by degree
KHAT_NNZ = {1: 6, 2: 46, 3: 202, 4: 647, 5: 1708, 6: 3920}


def _predict_flops(system, N):
    """Multiply-adds that the structural non-zeros ask for, as 2 flops: time solves, star products, block products."""
    nq, B, T = QUANTITIES[system], modes(N), N + 1
    return 2.0 * (nq * B * T * T + 3 * STAR[system] * (B - 1) * T + KHAT_NNZ[N] * nq * T)


def work(case):
    N, B, T = case["degree"], modes(case["degree"]), case["degree"] + 1
    if case["kind"] == "advance":
        ne = {"periodic": 6 * case["boxes"] ** 3, "layered": 24 * case["boxes"] ** 3, "box": 24 * case["boxes"] ** 3}[case["mesh"]]
        df = (N + 1) * (N + 2) // 2
        corrector = 2.0 * (3 * 54 * B + KHAT_NNZ[N] * 13 + 3 * 4 * 13 * df * B + 4 * 2 * 169 * df)
        # per cycle every element steps at least once (a uniform mesh with C clusters: all in the smallest)
        steps = case["cycles"] * (2 ** (case["clusters"] - 1) if case["mesh"] == "box" else 1)
        # modes in and out, the flux solvers of four faces, and the wavefield's copy to the host
        per_step = 8.0 * (2 * 13 * B + 4 * 2 * 169)
        return {"bytes": ne * (steps * per_step + 8.0 * 13 * B), "flops": ne * steps * (_predict_flops("biot", N) + corrector)}
    n, system = case["elements"], case["system"]
    nq = QUANTITIES[system]
    out = nq * B * (1 if case["kind"] == "host" else T + 1)
    flops = _predict_flops(system, N) * (10 if system == "subcell" else 1)
    return {"bytes": 8.0 * n * (nq * B + out + 3 * STAR[system] + T * T), "flops": n * flops}


def tolerance(case):
    """Relative errors of another correct implementation: about four times what each path shows against `exact`."""
    if case["precision"] == "fp64":
        return {"rel": 3e-14, "max": 3e-12}
    # the mixed forms promise 1e-10; one correction sweep leaves 1.4e-12 at degree 6, up to 3e-12 in an element
    return {"rel": 6e-12, "max": 6e-10}


# ------------------------------------------------------------------ the same in plain 64 bits
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _jacobi(n, a, x, y):
    """y^n P_n^(a,0)(x / y), n = 0 .. n, polynomials in (x, y)."""
    p = [torch.ones_like(x), 0.5 * ((a + 2) * x + a * y)]
    for m in range(1, n):
        c = 2 * (m + 1) * (m + a + 1) * (2 * m + a)
        p.append(((2 * m + a + 1) * ((2 * m + a + 2) * (2 * m + a) * x + a * a * y) * p[m]
                  - 2 * (m + a) * m * (2 * m + a + 2) * y * y * p[m - 1]) / c)
    return p[: n + 1]


def _basis(N, pts):
    """phi_l at reference points [n][3] -> [n][B]: ordered by degree, then k, then j."""
    x, y, z = pts[:, 0], pts[:, 1], pts[:, 2]
    one = torch.ones_like(x)
    P = _jacobi(N, 0, 2 * x - (1 - y - z), 1 - y - z)
    Q = [_jacobi(N, 2 * i + 1, 2 * y - (1 - z), 1 - z) for i in range(N + 1)]
    R = [_jacobi(N, 2 * s + 2, 2 * z - one, one) for s in range(N + 1)]
    return torch.stack([P[g - j - k] * Q[g - j - k][j] * R[g - k][k] for g in range(N + 1) for k in range(g + 1)
                        for j in range(g - k + 1)], dim=1)


@lru_cache(maxsize=None)
def _reference(N):
    """M (diagonal), K^j_kl = int phi_k d_j phi_l, Khat^j = M^{-1} K^j, and the time matrices; on the CPU."""
    x, w = np.polynomial.legendre.leggauss(N + 3)
    a, wa = (1 + x) / 2, w / 2
    zz, yy, xx = np.meshgrid(a, a, a, indexing="ij")
    wz, wy, wx = np.meshgrid(wa, wa, wa, indexing="ij")
    pts = np.stack([xx * (1 - yy) * (1 - zz), yy * (1 - zz), zz], -1).reshape(-1, 3)
    wt = torch.from_numpy((wx * wy * wz * (1 - yy) * (1 - zz) ** 2).reshape(-1))
    pts = torch.from_numpy(pts)
    phi = _basis(N, pts)
    K = []
    for j in range(3):
        e = torch.zeros_like(pts)
        e[:, j] = 1.0
        d = torch.func.jvp(lambda p: _basis(N, p), (pts,), (e,))[1]
        K.append((phi * wt[:, None]).T @ d)
    M = ((phi * phi) * wt[:, None]).sum(0)
    K = torch.stack(K)
    Kh = K / M[None, :, None]
    deg = torch.tensor([g for g in range(N + 1) for _ in range((g + 1) * (g + 2) // 2)])
    Kh = torch.where((deg[:, None] < deg[None, :])[None], Kh, torch.zeros_like(Kh))  # zero by degree
    T = N + 1
    Z = torch.tensor([[(2 * u + 1.0) * (-1.0 if u > s and (u - s) % 2 else 1.0) for s in range(T)] for u in range(T)],
                     dtype=torch.float64)
    sw = torch.tensor([(2 * u + 1.0) * (-1) ** u for u in range(T)], dtype=torch.float64)
    mass3 = torch.stack([(phi * (wt * phi[:, r])[:, None]).T @ phi for r in range(4)]) / M[None, :, None]
    return dict(M=M, K=K, Kh=Kh, Z=Z, sw=sw, mass3=mass3)


def _biot(mat):
    """A_d [n][3][13][13] and E [n][13][13] of material rows [n][10] (torch)."""
    KS, rS, lam, mu, kap, phi, tor, KF, rF, nu = mat.T
    rho, KM = phi * rF + (1 - phi) * rS, lam + 2.0 / 3.0 * mu
    al = 1 - KM / KS
    M = KS / ((1 - KM / KS) - phi * (1 - KS / KF))
    lc, m = lam + M * al * al, rF * tor / phi
    D = rho * m - rF * rF
    b = nu / kap
    n = mat.shape[0]
    A = torch.zeros((n, 3, 13, 13), dtype=torch.float64, device=mat.device)
    E = torch.zeros((n, 13, 13), dtype=torch.float64, device=mat.device)
    sig = [[0, 3, 5], [3, 1, 4], [5, 4, 2]]
    for d in range(3):
        for k in range(3):
            A[:, d, k, 6 + d] = -(lc + 2 * mu) if k == d else -lc
            A[:, d, k, 10 + d] = -M * al
            if k != d:
                A[:, d, sig[k][d], 6 + k] = -mu
            A[:, d, 6 + k, sig[k][d]] = -m / D
            A[:, d, 10 + k, sig[k][d]] = rF / D
        A[:, d, 9, 6 + d] = M * al
        A[:, d, 9, 10 + d] = M
        A[:, d, 6 + d, 9] = -rF / D
        A[:, d, 10 + d, 9] = rho / D
        E[:, 6 + d, 10 + d] = rF * b / D
        E[:, 10 + d, 10 + d] = -rho * b / D
    return A, E


def _maxwell(mat):
    n = mat.shape[0]
    A = torch.zeros((n, 3, 6, 6), dtype=torch.float64, device=mat.device)
    E = torch.zeros((n, 6, 6), dtype=torch.float64, device=mat.device)
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3  # (curl F)_a = d_b F_c - d_c F_b
        A[:, b, a, 3 + c], A[:, c, a, 3 + b] = -1 / mat[:, 0], 1 / mat[:, 0]
        A[:, b, 3 + a, c], A[:, c, 3 + a, b] = 1 / mat[:, 1], -1 / mat[:, 1]
        E[:, a, a] = -mat[:, 2] / mat[:, 0]
    return A, E


def _visco(mat):
    n = mat.shape[0]
    A = torch.zeros((n, 3, 27, 27), dtype=torch.float64, device=mat.device)
    E = torch.zeros((n, 27, 27), dtype=torch.float64, device=mat.device)
    rho, lam, mu = mat[:, 0], mat[:, 1], mat[:, 2]
    sig = [[0, 3, 5], [3, 1, 4], [5, 4, 2]]
    for d in range(3):
        for k in range(3):
            A[:, d, k, 6 + d] = -(lam + 2 * mu) if k == d else -lam
            if k != d:
                A[:, d, sig[k][d], 6 + k] = -mu
            A[:, d, 6 + k, sig[k][d]] = -1 / rho
            for l in range(3):
                A[:, d, 9 + 6 * l + sig[k][d], 6 + k] = -mat[:, 3 + l] * (1.0 if k == d else 0.5)
    for l in range(3):
        om, yl, ym = mat[:, 3 + l], mat[:, 6 + l], mat[:, 9 + l]
        for k in range(6):
            E[:, 9 + 6 * l + k, 9 + 6 * l + k] = -om
            E[:, k, 9 + 6 * l + k] = -2 * ym
        for i in range(3):
            for k in range(3):
                E[:, i, 9 + 6 * l + k] = -(yl + 2 * ym) if i == k else -yl
    return A, E


def _geometry(vert):
    J = (vert[:, 1:] - vert[:, :1]).transpose(1, 2)  # columns x_v - x_0
    return J, torch.linalg.inv(J)


def _solve(N, As, Es, rhs):
    """Q of (Z (x) I - E* + sum_j A^{j*} (x) Khat^j) Q = rhs, by degree blocks; rhs [n][q][B][T]."""
    R = {k: v.to(rhs.device) for k, v in _reference(N).items()}
    nq, T = Es.shape[1], N + 1
    b, Q = rhs.clone(), torch.zeros_like(rhs)
    eye = torch.eye(T, dtype=torch.float64, device=rhs.device)
    Zi = torch.linalg.inv(R["Z"] - torch.diagonal(Es, dim1=1, dim2=2)[:, :, None, None] * eye)
    off = 0
    blocks = []
    for g in range(N + 1):
        d = (g + 1) * (g + 2) // 2
        blocks.append((off, off + d))
        off += d
    coupled = [[bool((Es[:, o, p] != 0).any()) for p in range(nq)] for o in range(nq)]
    for g in range(N, -1, -1):
        lo, hi = blocks[g]
        for p in range(nq - 1, -1, -1):
            Q[:, p, lo:hi] = b[:, p, lo:hi] @ Zi[:, p].transpose(1, 2)
            for o in range(p):
                if coupled[o][p]:
                    b[:, o, lo:hi] += Es[:, o, p, None, None] * Q[:, p, lo:hi]
        if lo == 0:
            break
        for j in range(3):
            X = torch.einsum("npq,nqmu->npmu", As[:, j], Q[:, :, lo:hi])
            b[:, :, :lo] -= torch.einsum("lm,npmu->nplu", R["Kh"][j, :lo, lo:hi], X)
    return Q


def _operators(system, vert, mat, dt):
    A, E = {"biot": _biot, "maxwell": _maxwell, "visco": _visco}[system](mat)
    _, Ji = _geometry(vert)
    return dt[:, None, None, None] * torch.einsum("njd,ndpq->njpq", Ji, A), dt[:, None, None] * E


def _exact_predict(case, seed):
    vert, mat, dt, q0 = _population(case, seed)
    dev, N, system = q0.device, case["degree"], case["system"]
    vert, mat, dt = (torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (vert, mat, dt))
    sw = _reference(N)["sw"].to(dev)
    out = []
    for lo in range(0, q0.shape[0], 4096):
        s = slice(lo, lo + 4096)
        rhs = q0[s, :, :, None] * sw
        if system != "subcell":
            out.append(_solve(N, *_operators(system, vert[s], mat[s], dt[s]), rhs))
            continue
        # linear variation inside the element: f_r = sum_v P_rv f_v, fixed-point iteration on the mean operator
        V = _basis(1, torch.tensor([[0.0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=torch.float64))
        P = torch.linalg.inv(V).to(dev)
        ops = [_operators("biot", vert[s], mat[s, v], dt[s]) for v in range(4)]
        Ar = [sum(P[r, v] * ops[v][0] for v in range(4)) for r in range(4)]
        Er = [sum(P[r, v] * ops[v][1] for v in range(4)) for r in range(4)]
        Kh, m3 = _reference(N)["Kh"].to(dev), _reference(N)["mass3"].to(dev)
        Q = _solve(N, Ar[0], Er[0], rhs)
        for _ in range(60):
            b = rhs.clone()
            for r in range(1, 4):
                W = -torch.einsum("npq,nqlu->nplu", Er[r], Q)
                for j in range(3):
                    W += torch.einsum("lm,npmu->nplu", Kh[j], torch.einsum("npq,nqmu->npmu", Ar[r][:, j], Q))
                b -= torch.einsum("kl,nplu->npku", m3[r], W)
            new = _solve(N, Ar[0], Er[0], b)
            done = float((new - Q).abs().max()) <= 1e-16 * float(new.abs().max())
            Q = new
            if done:
                break
        out.append(Q)
    Q = torch.cat(out)
    i = dt[:, None, None] * Q[..., 0]
    return {"integrated": i.cpu().numpy()} if case["kind"] == "host" else {"predictor": Q, "integrated": i}


# Riemann solvers: waves of the x-direction Jacobian in impedance units, rotated into each face's frame
def _waves(A, z):
    """(R^-, R^+, A^+) of one Jacobian: real bases of the waves with negative and positive speed, and the positive part."""
    s = np.ones(13)
    s[[0, 1, 2, 3, 4, 5, 9]] = z
    lam, V = np.linalg.eig(A * s[None, :] / s[:, None])
    Vi, lam = np.linalg.inv(V), lam.real
    tol = 1e-6 * np.abs(lam).max()

    def part(mask, w):
        return ((V * np.where(mask, w, 0.0)[None, :]) @ Vi).real

    span = [np.linalg.svd(part(m, np.ones(13)))[0][:, :4] * s[:, None] for m in (lam < -tol, lam > tol)]
    return span[0], span[1], part(lam > tol, lam) * s[:, None] / s[None, :]


def _flux_x(matL, matR, kind):
    """F^-, F^+ for a face whose normal is x."""
    def side(m):
        A = _biot(torch.from_numpy(m[None]))[0][0, 0].numpy()
        rho = m[5] * m[8] + (1 - m[5]) * m[1]
        z = rho * np.abs(np.linalg.eigvals(A).real).max()
        return A, z

    A, z = side(matL)
    Rm, _, Ap = _waves(A, z)
    if kind == 2:
        return Ap, np.zeros((13, 13))
    C = np.zeros((8, 13))
    for r, q in enumerate((0, 3, 5, 9, 6, 7, 8, 10)):  # traction, pressure, solid velocity, normal fluid velocity
        C[r, q] = 1.0 / (z if r < 4 else 1.0)
    if kind == 1:
        return A @ (np.eye(13) - Rm @ np.linalg.solve(C[:4] @ Rm, C[:4])), np.zeros((13, 13))
    Rp = _waves(*side(matR))[1]
    K = Rm @ np.linalg.solve(np.hstack([C @ Rm, -C @ Rp]), C)[:4]
    return A @ (np.eye(13) - K), A @ K


def _rotations(nr):
    """[n][13][13] from the frame whose x axis is the normal to the global frame, and back."""
    ref = torch.where((nr[:, :1].abs() < 0.7), torch.tensor([1.0, 0, 0], dtype=nr.dtype, device=nr.device),
                      torch.tensor([0, 1.0, 0], dtype=nr.dtype, device=nr.device))
    s = torch.linalg.cross(nr, ref.expand_as(nr))
    s = s / torch.linalg.vector_norm(s, dim=1, keepdim=True)
    G = torch.stack([nr, s, torch.linalg.cross(nr, s)], dim=2)
    pair = [(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)]
    out = []
    for r in (G, G.transpose(1, 2)):
        T = torch.zeros((nr.shape[0], 13, 13), dtype=nr.dtype, device=nr.device)
        for a, (i, j) in enumerate(pair):
            for b, (k, l) in enumerate(pair):
                T[:, a, b] = r[:, i, k] * r[:, j, l] + (r[:, i, l] * r[:, j, k] if k != l else 0.0)
        T[:, 6:9, 6:9] = r
        T[:, 9, 9] = 1.0
        T[:, 10:, 10:] = r
        out.append(T)
    return out


def _exact_advance(case, seed):
    N, C, T = case["degree"], case["clusters"], case["degree"] + 1
    mesh, mats, src, _ = _mesh(case)
    dev = _dev()
    ne = mesh["tets"].shape[0]
    Q = torch.from_numpy(_mesh_q0(case, seed, ne)).to(dev)
    hv = mesh["vertices"][mesh["tets"]]
    dte = L.poro_cfl_dt(N, hv, mats)
    dt = dte.min()
    cl = np.minimum(C - 1, np.floor(np.log2(dte / dt) + 1e-12)).astype(int).clip(0)
    R = {k: v.to(dev) for k, v in _reference(N).items()}
    vert, mat = torch.from_numpy(hv).to(dev), torch.from_numpy(mats).to(dev)
    A, E = _biot(mat)
    J, Ji = _geometry(vert)
    Aj = torch.einsum("njd,ndpq->njpq", Ji, A)
    detJ = torch.linalg.det(J).abs()
    # faces: quadrature points in both elements' coordinates, by tables over (face, neighbour's face, permutation)
    x, w = np.polynomial.legendre.leggauss(N + 2)
    a, wa = (1 + x) / 2, w / 2
    pb, pa = np.meshgrid(a, a, indexing="ij")
    wq = torch.from_numpy((wa[:, None] * wa[None, :] * (1 - pb)).reshape(-1)).to(dev)
    pa, pb = torch.from_numpy((pa * (1 - pb)).reshape(-1)), torch.from_numpy(pb.reshape(-1))
    ref = torch.tensor([[0.0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=torch.float64)
    fv = [[v for v in range(4) if v != f] for f in range(4)]
    perms = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]

    def trace(c):  # basis at the quadrature points of the triangle with corners c[0], c[1], c[2]
        return _basis(N, c[0] + pa[:, None] * (c[1] - c[0]) + pb[:, None] * (c[2] - c[0]))

    own = torch.stack([trace(ref[fv[f]]) for f in range(4)]).to(dev)
    other = torch.stack([trace(ref[[fv[h][p[i]] for i in range(3)]]) for h in range(4) for p in perms]).to(dev)
    nb = mesh["neighbors"]
    flux = {}
    area2, tab, Fm, Fp = [], [], [], []
    key = np.unique(mats, axis=0, return_inverse=True)[1].reshape(-1)
    for f in range(4):
        c = hv[:, fv[f]]
        nr = np.cross(c[:, 1] - c[:, 0], c[:, 2] - c[:, 0])
        ln = np.linalg.norm(nr, axis=1)
        nr /= ln[:, None]
        nr *= np.where(np.einsum("nd,nd->n", nr, hv[:, f] - c[:, 0]) > 0, -1.0, 1.0)[:, None]
        area2.append(torch.from_numpy(ln).to(dev))
        t = np.full(ne, -1)
        r = np.maximum(nb[:, f], 0)
        for h in range(4):
            o = hv[r][:, fv[h]]
            shift = o.mean(axis=1) - c.mean(axis=1)
            for k, p in enumerate(perms):
                same = np.abs(o[:, p] - c - shift[:, None]).max(axis=(1, 2)) < 1e-9 * (1 + np.abs(c).max())
                t = np.where(same & (nb[:, f] >= 0) & (t < 0), h * 6 + k, t)
        tab.append(torch.from_numpy(t).to(dev))
        kind = np.where(nb[:, f] >= 0, 0, mesh["face_tag"][:, f])
        code = np.stack([key, np.where(nb[:, f] >= 0, key[r], -1), kind], 1)
        uniq, inv = np.unique(code, axis=0, return_inverse=True)
        fx = []
        for u in uniq:
            if tuple(u) not in flux:
                i = int(np.nonzero((code == u).all(axis=1))[0][0])
                flux[tuple(u)] = _flux_x(mats[i], mats[r[i]], int(u[2]))
            fx.append(flux[tuple(u)])
        to, back = _rotations(torch.from_numpy(nr).to(dev))
        inv = torch.from_numpy(inv.reshape(-1)).to(dev)
        for k, dst in ((0, Fm), (1, Fp)):
            F = torch.from_numpy(np.stack([v[k] for v in fx])).to(dev)[inv]
            dst.append(to @ F @ back)
    # the source's element and modes
    xi = np.einsum("njd,nd->nj", np.linalg.inv((hv[:, 1:] - hv[:, :1]).transpose(0, 2, 1)), src["x"] - hv[:, 0])
    se = int(np.nonzero((xi >= -1e-12).all(axis=1) & (1 - xi.sum(axis=1) >= -1e-12))[0][0])
    phi_s = _basis(N, torch.from_numpy(xi[se:se + 1]))[0].to(dev)
    coef = src["amplitude"] * torch.from_numpy(np.asarray(src["w"], float)).to(dev)[:, None] * phi_s / (detJ[se] * R["M"])

    def ricker(t):
        return (t - src["t0"]) * math.exp(-(math.pi * src["f0"] * (t - src["t0"])) ** 2)

    def legendre_integrals(lo, hi):  # int_lo^hi P_s(2 tau - 1) dtau
        return [0.5 * float(np.polynomial.Legendre.basis(s).integ()(2 * hi - 1)
                            - np.polynomial.Legendre.basis(s).integ()(2 * lo - 1)) for s in range(T)]

    tcl, tnb = torch.from_numpy(cl).to(dev), torch.from_numpy(np.ascontiguousarray(nb)).to(dev)
    Qt = torch.zeros((ne, 13, modes(N), T), dtype=torch.float64, device=dev)
    I = torch.zeros_like(Q)
    sums = [torch.zeros_like(Q) for _ in range(C)]
    dtc = dt * 2.0 ** tcl.double()
    els = [torch.nonzero(tcl == c).reshape(-1) for c in range(C)]
    for k in range(case["cycles"] * 2 ** (C - 1)):
        for c in range(C):
            if k % 2 ** c == 0 and len(els[c]):
                for e in els[c].split(4096):
                    h = dtc[e]
                    Qt[e] = _solve(N, h[:, None, None, None] * Aj[e], h[:, None, None] * E[e], Q[e][..., None] * R["sw"])
                    I[e] = h[:, None, None] * Qt[e][..., 0]
                    for big in range(c + 1, C):
                        sums[big][e] = I[e] if k % 2 ** big == 0 else sums[big][e] + I[e]
        for c in range(C):
            if (k + 1) % 2 ** c or not len(els[c]):
                continue
            ks = k + 1 - 2 ** c
            for e in els[c].split(4096):
                d = sum(torch.einsum("npl,lk->npk", Aj[e][:, j] @ I[e], R["K"][j]) for j in range(3)) / R["M"] + E[e] @ I[e]
                for f in range(4):
                    u = Fm[f][e] @ (I[e] @ own[f].T)
                    r = tnb[e, f].clamp(min=0)
                    Ir = torch.where((tcl[r] < c)[:, None, None], sums[c][r], I[r])
                    for big in range(c + 1, C):
                        m = (ks >> big) << big
                        wts = torch.tensor(legendre_integrals((ks - m) / 2 ** big, (k + 1 - m) / 2 ** big),
                                           dtype=torch.float64, device=dev)
                        at = torch.nonzero(tcl[r] == big).reshape(-1)
                        Ir[at] = dt * 2.0 ** big * (Qt[r[at]] @ wts)
                    P = other[tab[f][e].clamp(min=0)]
                    u = u + torch.where((tnb[e, f] >= 0)[:, None, None], Fp[f][e] @ (Ir @ P.transpose(1, 2)), 0.0)
                    d = d - (area2[f][e] / detJ[e])[:, None, None] * ((u * wq) @ own[f]) / R["M"]
                Q[e] += d
            if cl[se] == c:
                Q[se] += coef * (ricker((k + 1) * dt) - ricker(ks * dt))
    return {"dofs": Q.cpu().numpy()}


def exact(case, seed):
    return _exact_advance(case, seed) if case["kind"] == "advance" else _exact_predict(case, seed)
