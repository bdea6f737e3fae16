"""The work that users of this package have it do, as timed cases.

A case names one call of the package's public entry points (the forward solve, J s, J^T t, both at once, the
prior solve, a batch of forward solves on uneven meshes, a short reconstruction, the U-Net's prediction and its
gradient) with its mesh, its number of illuminations and its solver options.  Meshes are Kuhn cubes of n nodes
a side and cylinders mapped from such grids; the fields are smooth random optical coefficients of tissue.
"""
import itertools
import math
from collections import OrderedDict

import numpy as np
import torch

import paper_1512_02796_gb300 as Q

DEV = "cuda"
F64 = torch.float64
CONVS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (192, 64), (64, 64),
         (96, 32), (32, 32), (48, 16), (16, 16), (16, 16)]  # (c_in, c_out) of the U-Net's convolutions


def listed():
    return [
        # the smallest call: one illumination of a coarse first reconstruction mesh, all launches and latency
        {"name": "forward_cube11_k1", "kind": "forward", "mesh": "cube", "n": 11, "K": 1},
        # a J s on the curved body of the phantom experiments: general tet shapes, an odd number of illuminations
        {"name": "jvp_cyl21x27_k3", "kind": "jvp", "mesh": "cyl", "n": 21, "nz": 27, "K": 3},
        # a whole call: a few priorconditioned LSQR rounds of Algorithm 1 from host arrays
        {"name": "reconstruct_cube24_k2", "kind": "reconstruct", "mesh": "cube", "n": 24, "K": 2, "lin": 2, "rounds": 4},
        # many small bodies at once (meshes of 16 to 48 nodes a side) in one replayed launch
        {"name": "batch12_16to48", "kind": "batch", "meshes": 12, "lo": 16, "hi": 48, "pick": 3},
        # one LSQR round's K solves on the ordinary mesh, with the default solver
        {"name": "pair_cube64_k4", "kind": "pair", "mesh": "cube", "n": 64, "K": 4},
        # the same with the FP32 solver inside FP64 refinement
        {"name": "pair_cube64_k4_mixed", "kind": "pair", "mesh": "cube", "n": 64, "K": 4, "precision": 1},
        # the other half of that round: M_delta^-1 with the default solver
        {"name": "prior_cube64", "kind": "prior", "mesh": "cube", "n": 64},
        # a fine mesh with 8 illuminations, FP32 multigrid cycles inside FP64 conjugate gradients
        {"name": "pair_cube96_k8_mg32", "kind": "pair", "mesh": "cube", "n": 96, "K": 8, "multigrid": 2},
        # the largest mesh, FP64 throughout: the operator work of one LSQR round
        {"name": "pair_cube128_k8_mg", "kind": "pair", "mesh": "cube", "n": 128, "K": 8, "multigrid": 1},
        {"name": "prior_cube128_mg", "kind": "prior", "mesh": "cube", "n": 128, "multigrid": 1},
        # learned initial guesses of all illuminations on the largest grid
        {"name": "unet_predict_128_b8", "kind": "unet_predict", "n": 128, "B": 8},
        # one training step's loss and gradient on the smallest grid
        {"name": "unet_grad_32_b4", "kind": "unet_grad", "n": 32, "B": 4},
    ]


def draw(rng):
    """Sizes are log-uniform over the listed range; the solver follows what one takes at that size."""
    kind = rng.choice(["forward", "jvp", "vjp", "pair", "pair", "prior", "prior", "reconstruct", "batch",
                       "unet_predict", "unet_grad"])
    size = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    if kind == "unet_predict":
        return {"kind": kind, "n": 16 * rng.randint(2, 8), "B": rng.randint(1, 8)}
    if kind == "unet_grad":
        return {"kind": kind, "n": 16 * rng.randint(2, 5), "B": rng.randint(1, 4)}
    if kind == "batch":
        lo = rng.randint(8, 20)
        return {"kind": kind, "meshes": rng.randint(2, 14), "lo": lo, "hi": lo + rng.randint(4, 28), "pick": rng.randint(0, 99)}
    if kind == "reconstruct":
        return {"kind": kind, "mesh": "cube", "n": size(9, 30), "K": rng.randint(1, 4), "lin": rng.randint(1, 2), "rounds": rng.randint(2, 4)}
    n = size(9, 120)
    case = {"kind": kind, "mesh": "cube", "n": n}
    if n < 60 and rng.random() < 0.3:
        case.update(mesh="cyl", n=max(9, n), nz=max(8, int(n * rng.uniform(0.5, 1.5))))
    if kind != "prior":
        case["K"] = rng.randint(1, 8)
    if n >= 32:
        case["multigrid"] = rng.choice([0, 1, 2]) if n < 90 else rng.choice([1, 2])
    if kind != "prior" and not case.get("multigrid"):
        case["precision"] = rng.choice([0, 0, 1])
    return case


# ---------------------------------------------------------------- meshes

def grid(case):
    """(nx, ny, nz, x, y, z) of the structured grid under the mesh; x runs fastest."""
    n, nz = case["n"], case.get("nz", case["n"])
    if case["mesh"] == "cube":
        side = 40.0 if n >= 32 else 20.0
        g = np.arange(n) * (side / (n - 1))
        z, y, x = np.meshgrid(g, g, g, indexing="ij")
        return n, nz, np.stack([x.ravel(), y.ravel(), z.ravel()], 1), side
    g = np.linspace(-1.0, 1.0, n)
    z, y, x = np.meshgrid(np.linspace(0.0, 25.0, nz), g, g, indexing="ij")
    x, y = x.ravel(), y.ravel()
    rho = np.hypot(x, y)
    f = 12.5 * np.maximum(np.abs(x), np.abs(y)) / np.where(rho > 0, rho, 1.0)
    return n, nz, np.stack([x * f, y * f, z.ravel()], 1), 25.0


def geometry(case):
    """Nodes, tets and the boundary faces in canonical order (node triples ascending, sorted)."""
    n, nz, xyz, side = grid(case)
    k, j, i = np.meshgrid(np.arange(nz - 1), np.arange(n - 1), np.arange(n - 1), indexing="ij")
    base = (i + n * (j + n * k)).ravel()
    step = (1, n, n * n)
    tets = np.stack([np.stack([base, base + step[a], base + step[a] + step[b], base + sum(step)], 1)
                     for a, b, _ in itertools.permutations(range(3))], 1).reshape(-1, 4)
    # a tet's face lies on the boundary when its three nodes lie in one boundary plane of the grid
    tri = np.sort(tets, 1)[:, [[0, 1, 2], [0, 1, 3], [0, 2, 3], [1, 2, 3]]]
    keep = []
    for s, m in ((1, n), (n, n), (n * n, nz)):
        c = tri // s % m if s < n * n else tri // s
        for v in (0, m - 1):
            keep.append(tri[(c == v).all(2)])
    faces = np.concatenate(keep)
    faces = faces[np.lexsort((faces[:, 2], faces[:, 1], faces[:, 0]))]
    return xyz, tets.astype(np.int32), faces, side


_MESHES = OrderedDict()


def mesh_of(case, patch_nodes=None):
    """A program prepares its mesh once and solves on it many times, so the handle is kept for the next inputs."""
    key = (case["mesh"], case["n"], case.get("nz"), patch_nodes)
    if key not in _MESHES:
        while len(_MESHES) >= 24:
            _MESHES.popitem(last=False)
        xyz, tets, faces, side = geometry(case)
        _MESHES[key] = (Q.qpat_mesh(xyz, tets, patch_nodes), xyz, faces, side)
    _MESHES.move_to_end(key)
    return _MESHES[key]


# ---------------------------------------------------------------- inputs

def generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def smooth(x, side, g, lo, hi, blobs=20):
    """A field of random blobs, mapped onto [lo, hi] in its logarithm."""
    c = torch.rand((blobs, 3), generator=g, device=DEV, dtype=F64) * side
    s = (0.05 + 0.1 * torch.rand(blobs, generator=g, device=DEV, dtype=F64)) * side
    a = torch.randn(blobs, generator=g, device=DEV, dtype=F64)
    f = torch.zeros(x.shape[0], device=DEV, dtype=F64)
    for b in range(blobs):
        f += a[b] * torch.exp(-((x - c[b]) ** 2).sum(1) / (2 * s[b] ** 2))
    t = (f - f.min()) / (f.max() - f.min())
    return torch.exp(math.log(lo) + t * math.log(hi / lo))


def optics(x, side, g):
    mua = smooth(x, side, g, 0.005, 0.05)
    mus = smooth(x, side, g, 0.5, 2.0)
    return 1.0 / (3.0 * (mua + mus)), mua


def fluxes(case, xyz, faces, side, K, g):
    """Patches on the six faces of a cube, or cosine profiles on the side of a cylinder: K x F."""
    mid = torch.from_numpy(xyz[faces].mean(1)).to(DEV)
    corner = torch.from_numpy(xyz[faces]).to(DEV)
    move = torch.rand((K, 3), generator=g, device=DEV, dtype=F64)
    out = torch.zeros((K, len(faces)), device=DEV, dtype=F64)
    for k in range(K):
        if case["mesh"] == "cube":
            axis, end = ((2, 1), (2, 0), (0, 1), (0, 0), (1, 1), (1, 0))[k % 6]
            on = ((corner[:, :, axis] - end * side).abs() < 1e-9 * side).all(1)
            centre = side * (0.4 + 0.2 * move[k])
            for b in range(3):
                if b != axis:
                    on &= (mid[:, b] - centre[b]).abs() <= side / 4
            out[k] = on.double()
        else:
            on = ((torch.hypot(corner[:, :, 0], corner[:, :, 1]) - 12.5).abs() < 1e-9 * side).all(1)
            d = torch.atan2(mid[:, 1], mid[:, 0]) - (k * math.pi / 2 + 0.2 * move[k, 0])
            d = torch.remainder(d + math.pi, 2 * math.pi) - math.pi
            out[k] = torch.where(on & (d.abs() <= math.pi / 8), torch.cos(4 * d), torch.zeros_like(d))
    return out


def fluences(x, side, K, g):
    """What forward solutions look like: light that decays from each source."""
    c = torch.rand((K, 3), generator=g, device=DEV, dtype=F64) * side
    d = torch.stack([((x - c[k]) ** 2).sum(1).sqrt() for k in range(K)])
    return torch.exp(-0.3 * d) / (1.0 + d)


def fields(case, seed, xyz, faces, side):
    """The inputs of one call, on the GPU."""
    g = generator(seed)
    x = torch.from_numpy(xyz).to(DEV)
    N, K = x.shape[0], case.get("K", 1)
    kappa, mu = optics(x, side, g)
    v = {"kappa": kappa, "mu": mu}
    if case["kind"] in ("forward", "reconstruct"):
        v["flux"] = fluxes(case, xyz, faces, side, K, g)
    if case["kind"] in ("jvp", "vjp", "pair"):
        v["phi"] = fluences(x, side, K, g)
        h = mu * v["phi"]
        v["w"] = 1.0 / (0.01 * h + 1e-3 * h.max())
        v["s"] = 0.1 * torch.randn(2 * N, generator=g, device=DEV, dtype=F64)
        v["t"] = torch.randn((K, N), generator=g, device=DEV, dtype=F64)
    if case["kind"] == "prior":
        v["kt"], v["mt"] = (kappa / kappa.median()).log(), (mu / mu.median()).log()
        v["rhs"] = torch.randn(2 * N, generator=g, device=DEV, dtype=F64)
    if case["kind"] == "reconstruct":
        v["noise"] = torch.randn((K, N), generator=g, device=DEV, dtype=F64)
    return v


def params(case):
    return Q.qpat_default_params(precision=case.get("precision", 0), fp32_operator=case.get("precision", 0),
                                 multigrid=case.get("multigrid", 0))


def bodies(case):
    """The meshes of a batch, as cases of their own."""
    r = np.random.RandomState(case["pick"])
    return [{"kind": "forward", "mesh": "cube", "n": int(r.randint(case["lo"], case["hi"] + 1)), "K": int(r.randint(1, 5))}
            for _ in range(case["meshes"])]


def network(case, seed):
    """Weights (He-normal, biases small), features and targets of the U-Net."""
    r = np.random.RandomState(int(seed) % (1 << 32))
    w = []
    for i, (cin, cout) in enumerate(CONVS):
        fan = 27 * (3 if i == 0 else cin)
        w.append((r.standard_normal(27 * cin * cout) * math.sqrt((2.0 if i < 14 else 0.5) / fan)).astype(np.float32))
        w.append((0.01 * r.standard_normal(cout)).astype(np.float32))
    g, n, B = generator(seed), case["n"], case["B"]
    at = torch.arange(n, device=DEV, dtype=F64) * (40.0 / (n - 1))
    z, y, x = torch.meshgrid(at, at, at, indexing="ij")
    x = torch.stack([x.ravel(), y.ravel(), z.ravel()], 1)
    feats, targets = [], []
    for b in range(B):
        kappa, mu = optics(x, 40.0, g)
        phi = fluences(x, 40.0, 1, g)[0]
        lit = torch.where(x[:, b % 3] < 1e-9, (phi > phi.median()).double(), torch.zeros_like(phi))
        feats.append(torch.stack([(mu / 0.01).log(), (kappa / 0.33).log(), lit], 1).float())
        targets.append(phi.float())
    return np.concatenate(w), torch.stack(feats).contiguous(), torch.stack(targets).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("unet_predict", "unet_grad"):
        w, x, t = network(case, seed)
        net = Q.UNet(case["n"], seed=1)
        net.set_params(w)
        return {"kind": kind, "net": net, "x": x, "t": t, "y": torch.empty(x.shape[:2], device=DEV)}
    if kind == "batch":
        bs = bodies(case)
        got = [mesh_of(b, 256) for b in bs]
        batch = Q.qpat_batch_create([m for m, *_ in got], [b["K"] for b in bs], Q.qpat_default_params(poly_degree=0))
        for j, (b, (_, xyz, faces, side)) in enumerate(zip(bs, got)):
            v = fields(b, int(seed) * 64 + j, xyz, faces, side)
            for to, name in zip(batch.inputs(j), ("kappa", "mu", "flux")):
                to.copy_(v[name])
        return {"kind": kind, "batch": batch, "phi": [torch.empty_like(batch.phi(j)) for j in range(len(bs))]}
    mesh, xyz, faces, side = mesh_of(case)
    v = fields(case, seed, xyz, faces, side)
    state = {"kind": kind, "mesh": mesh, "params": params(case), **v}
    N, K = mesh.N, case.get("K", 1)
    for name, shape in {"forward": {"phi": (K, N), "h": (K, N)}, "jvp": {"jv": (K, N)}, "vjp": {"jt": (2 * N,)},
                        "pair": {"jv": (K, N), "jt": (2 * N,)}, "prior": {"out": (2 * N,)}}.get(kind, {}).items():
        state[name] = torch.empty(shape, device=DEV, dtype=F64)
    if kind == "reconstruct":
        state["params"] = Q.qpat_default_params(T=2e-2, max_lin=case["lin"], max_lsqr=case["rounds"], fixed_counts=1)
        phi, h = Q.qpat_forward(mesh, v["kappa"].cpu().numpy(), v["mu"].cpu().numpy(), v["flux"].cpu().numpy())
        noise = v["noise"].cpu().numpy()
        state["chi"] = h + 0.01 * np.abs(h) * noise
        state["sigma"] = 0.01 * np.abs(h) + 1e-3 * np.abs(h).max()
        state["flux"] = v["flux"].cpu().numpy()
        state["background"] = np.array([float(v["kappa"].median()), float(v["mu"].median())])
    return state


def run(state):
    kind, s = state["kind"], state
    if kind == "forward":
        return Q.qpat_forward_dev(s["mesh"], s["kappa"], s["mu"], s["flux"], s["phi"], s["h"], s["params"])
    if kind == "jvp":
        return Q.qpat_jvp_dev(s["mesh"], s["kappa"], s["mu"], s["phi"], s["w"], s["s"], s["jv"], s["params"])
    if kind == "vjp":
        return Q.qpat_vjp_dev(s["mesh"], s["kappa"], s["mu"], s["phi"], s["w"], s["t"], s["jt"], s["params"])
    if kind == "pair":
        return Q.qpat_jvp_vjp_pair_dev(s["mesh"], s["kappa"], s["mu"], s["phi"], s["w"], s["s"], s["t"], s["jv"], s["jt"], s["params"])
    if kind == "prior":
        return Q.qpat_prior_solve_dev(s["mesh"], s["kt"], s["mt"], s["rhs"], s["out"], s["params"])
    if kind == "reconstruct":
        kappa, mu, _ = Q.qpat_reconstruct(s["mesh"], s["flux"], s["chi"], s["sigma"], s["params"], s["background"])
        return kappa, mu
    if kind == "batch":
        s["batch"].forward()
        # the batch's own buffers live and change with it: a program that goes on with the solutions takes them out
        return [to.copy_(s["batch"].phi(j)) for j, to in enumerate(s["phi"])]
    if kind == "unet_predict":
        return s["net"].predict(s["x"], s["y"])
    loss, grad = s["net"].grad(s["x"], s["t"])
    return np.float32(loss), grad


# ---------------------------------------------------------------- work

def sizes(case):
    n, nz = case["n"], case.get("nz", case["n"])
    return n * n * nz, 6 * (n - 1) ** 2 * (nz - 1), 4 * (n - 1) ** 2 + 8 * (n - 1) * (nz - 1)


def work(case):
    """Inputs and outputs once, and the operations of one application of the operator to every right-hand side (15
    entries a row for K, 7 for each block of M_delta): what no solver can do without."""
    kind = case["kind"]
    if kind.startswith("unet"):
        n, B = case["n"], case["B"]
        level = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
        macs = sum(27 * cin * cout * (n >> lv) ** 3 for (cin, cout), lv in zip(CONVS, level))
        weights = sum(27 * a * b + b for a, b in CONVS)
        if kind == "unet_predict":
            return {"bytes": B * n ** 3 * 16 + 4 * weights, "flops": 2 * macs * B}
        return {"bytes": B * n ** 3 * 16 + 8 * weights, "flops": 6 * macs * B}
    if kind == "batch":
        parts = [work(b) for b in bodies(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    (N, E, F), K = sizes(case), case.get("K", 1)
    mesh = 24 * N + 16 * E
    if kind == "prior":
        return {"bytes": mesh + 8 * 6 * N, "flops": 2 * 7 * 2 * N}
    values = {"forward": 2 * N + K * F + 2 * K * N, "jvp": 2 * N + 2 * K * N + 2 * N + K * N, "vjp": 2 * N + 3 * K * N + 2 * N,
              "pair": 2 * N + 3 * K * N + 2 * N + K * N + 2 * N, "reconstruct": K * F + 2 * K * N + 2 * N}[kind]
    times = {"pair": 2, "reconstruct": 2 * case.get("lin", 1) * case.get("rounds", 1)}.get(kind, 1)
    return {"bytes": mesh + 8 * values, "flops": 2 * 15 * N * K * times}


# ---------------------------------------------------------------- the same in plain torch, 64 bits

class Plain:
    """P1 elements of a mesh: gradients of the hat functions, volumes, and sparse matrices from element matrices."""

    def __init__(self, case):
        xyz, tets, self.faces, self.side = geometry(case)
        self.xyz = xyz
        x, self.t = torch.from_numpy(xyz).to(DEV), torch.from_numpy(tets).to(DEV).long()
        self.N = len(xyz)
        p = x[self.t]
        d = torch.stack([p[:, 1] - p[:, 0], p[:, 2] - p[:, 0], p[:, 3] - p[:, 0]], 1)
        c = torch.stack([torch.linalg.cross(d[:, 1], d[:, 2]), torch.linalg.cross(d[:, 2], d[:, 0]), torch.linalg.cross(d[:, 0], d[:, 1])], 1)
        det = (d[:, 0] * c[:, 0]).sum(1)
        g = c / det[:, None, None]
        self.g = torch.cat([-g.sum(1, keepdim=True), g], 1)
        self.vol = det.abs() / 6
        self.f = torch.from_numpy(self.faces).to(DEV)
        q = x[self.f]
        self.area = torch.linalg.cross(q[:, 1] - q[:, 0], q[:, 2] - q[:, 0]).norm(dim=1) / 2
        m = torch.full((4, 4, 4), 1.0 / 120, device=DEV, dtype=F64)  # int l_i l_j l_k = |T| / 20, / 60, / 120
        for i, j, k in itertools.product(range(4), repeat=3):
            m[i, j, k] *= {1: 6, 2: 2, 3: 1}[len({i, j, k})]
        self.m = m

    def sparse(self, ids, values):
        k = ids.shape[1]
        i = torch.stack([ids[:, :, None].expand(-1, k, k).reshape(-1), ids[:, None, :].expand(-1, k, k).reshape(-1)])
        return torch.sparse_coo_tensor(i, values.reshape(-1), (self.N, self.N)).coalesce()

    def stiffness(self, c):
        return torch.einsum("tid,tjd->tij", self.g, self.g) * (c * self.vol)[:, None, None]

    def K(self, kappa, mu, robin=True):
        e = self.stiffness(kappa[self.t].mean(1)) + torch.einsum("ijk,tk->tij", self.m, mu[self.t]) * self.vol[:, None, None]
        a = self.sparse(self.t, e)
        if robin:
            b = (torch.ones(3, 3, device=DEV, dtype=F64) + torch.eye(3, device=DEV, dtype=F64)) / 24
            a = (a + self.sparse(self.f, self.area[:, None, None] * b)).coalesce()
        return a.to_sparse_csr()

    def prior(self, u, T):
        grad = torch.einsum("tid,ti->td", self.g, u[self.t])
        g2 = (grad ** 2).sum(1)
        c = 1 / (1 + g2 / (T * T))
        eye = torch.arange(self.N, device=DEV)
        d = torch.sparse_coo_tensor(torch.stack([eye, eye]), torch.full((self.N,), 1e-6, device=DEV, dtype=F64), (self.N, self.N))
        return (self.sparse(self.t, self.stiffness(c)) + d).coalesce().to_sparse_csr()

    def load(self, flux):
        f = torch.zeros((flux.shape[0], self.N), device=DEV, dtype=F64)
        for v in range(3):
            f.index_add_(1, self.f[:, v], 2.0 / 3.0 * flux * self.area)
        return f


def diagonal(A):
    rows = torch.repeat_interleave(torch.arange(A.shape[0], device=DEV), A.crow_indices().diff())
    return A.values()[rows == A.col_indices()]


def solve(A, B, limit=6000):
    """A X = B (right-hand sides as rows) by conjugate gradients, refined with the true residual."""
    inv, X = 1.0 / diagonal(A)[:, None], torch.zeros_like(B).T.contiguous()
    B = B.T.contiguous()
    for _ in range(3):
        R = B - A @ X
        target = 1e-11 * R.norm(dim=0)
        D, Z = torch.zeros_like(X), inv * R
        P, rz = Z.clone(), (R * Z).sum(0)
        for i in range(limit):
            W = A @ P
            a = rz / (P * W).sum(0).clamp_min(1e-300)
            D += a * P
            R -= a * W
            if i % 20 == 19 and bool((R.norm(dim=0) <= target).all()):
                break
            Z = inv * R
            new = (R * Z).sum(0)
            P, rz = Z + new / rz.clamp_min(1e-300) * P, new
        X += D
    return X.T.contiguous()


def plain_unet(w, x, n):
    """The network on float64 weights: x (B, n^3, 3) -> channel 0 of its output, (B, n^3)."""
    at, parts = 0, []
    for cin, cout in CONVS:
        parts.append((w[at:at + 27 * cin * cout].view(27, cout, cin), w[at + 27 * cin * cout:at + 27 * cin * cout + cout]))
        at += 27 * cin * cout + cout

    def conv(i, a, relu=True):
        k, b = parts[i]
        m = a.shape[1]
        p = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        y = b.expand(*a.shape[:4], -1)
        for t in range(27):
            z, yy, xx = t // 9, t // 3 % 3, t % 3
            y = y + p[:, z:z + m, yy:yy + m, xx:xx + m] @ k[t].T
        return y.clamp_min(0) if relu else y

    pool = lambda a: a.view(a.shape[0], a.shape[1] // 2, 2, a.shape[2] // 2, 2, a.shape[3] // 2, 2, -1).mean((2, 4, 6))  # noqa: E731
    up = lambda a: a.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    a = torch.nn.functional.pad(x.view(x.shape[0], n, n, n, 3), (0, 13))
    s0 = conv(1, conv(0, a))
    s1 = conv(3, conv(2, pool(s0)))
    s2 = conv(5, conv(4, pool(s1)))
    bt = conv(7, conv(6, pool(s2)))
    d2 = conv(9, conv(8, torch.cat([up(bt), s2], -1)))
    d1 = conv(11, conv(10, torch.cat([up(d2), s1], -1)))
    d0 = conv(13, conv(12, torch.cat([up(d1), s0], -1)))
    return conv(14, d0, relu=False)[..., 0].reshape(x.shape[0], -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "reconstruct":  # Algorithm 1 as a whole has no short form in plain torch
        return None
    if kind.startswith("unet"):
        w, x, t = network(case, seed)
        w = torch.from_numpy(w).to(DEV).double()
        if kind == "unet_predict":
            with torch.no_grad():
                return torch.cat([plain_unet(w, x[b:b + 1].double(), case["n"]) for b in range(case["B"])])
        w.requires_grad_(True)
        loss = ((plain_unet(w, x.double(), case["n"]) - t.double()) ** 2).mean()
        loss.backward()
        return loss.detach(), w.grad
    if kind == "batch":
        out = []
        for j, b in enumerate(bodies(case)):
            P = Plain(b)
            v = fields(b, int(seed) * 64 + j, P.xyz, P.faces, P.side)
            out.append(solve(P.K(v["kappa"], v["mu"]), P.load(v["flux"])))
        return out
    P = Plain(case)
    v = fields(case, seed, P.xyz, P.faces, P.side)
    N = P.N
    if kind == "prior":
        T = Q.qpat_default_params().T
        return torch.cat([solve(P.prior(u, T), r[None])[0] for u, r in ((v["kt"], v["rhs"][:N]), (v["mt"], v["rhs"][N:]))])
    kappa, mu = v["kappa"], v["mu"]
    A = P.K(kappa, mu)
    if kind == "forward":
        phi = solve(A, P.load(v["flux"]))
        return phi, mu * phi
    phi, w, s, t = v["phi"], v["w"], v["s"], v["t"]
    rhs = []
    if kind in ("jvp", "pair"):
        rhs.append(-(P.K(kappa * s[:N], mu * s[N:], robin=False) @ phi.T).T)
    if kind in ("vjp", "pair"):
        rhs.append(mu * w * t)
    X = solve(A, torch.cat(rhs))
    K = phi.shape[0]
    jv = jt = None
    if kind in ("jvp", "pair"):
        jv = w * (mu * X[:K] + phi * (mu * s[N:]))
    if kind in ("vjp", "pair"):
        z = X[-K:]
        o1, o2 = torch.zeros(N, device=DEV, dtype=F64), torch.zeros(N, device=DEV, dtype=F64)
        for k in range(K):
            a, b = phi[k][P.t], z[k][P.t]
            e = (torch.einsum("tid,ti->td", P.g, a) * torch.einsum("tid,ti->td", P.g, b)).sum(1) * P.vol / 4
            o1.index_add_(0, P.t.reshape(-1), -e[:, None].expand(-1, 4).reshape(-1))
            q = torch.einsum("ijk,tj,tk->ti", P.m, a, b) * P.vol[:, None]
            o2.index_add_(0, P.t.reshape(-1), -q.reshape(-1))
        jt = torch.cat([kappa * o1, mu * (o2 + (phi * w * t).sum(0))])
    return {"jvp": jv, "vjp": jt}[kind] if kind != "pair" else (jv, jt)
