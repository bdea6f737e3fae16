"""The persistent solvers by name (pcg_variant = 1), at sizes where a call that
names no solver takes the multigrid CG: the patch-local polynomial and Jacobi for
M_delta, the FP32 solver inside FP64 refinement with both operators and both forms of
restart, batches with many illuminations; and the multigrid CG against them, on
meshes without a grid behind them and on two streams at once.

Bars as in the tests of the same calls at small sizes: 1e-10 for K solves against
the oracle (residual 1e-13, cond(K) < 1e3), residuals below 1e-12 and backward errors
below 1e-13 where the oracle cannot factorise, 1e-8 between two M_delta solutions (cond(M_delta) < 1e5 on this
body, residual 1e-13)."""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S
from tests.gpu_common import Case, rel
from tests.test_gpu_fullsize import smooth_phi

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def big():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Case(S.config("c1_cube64"), solve=False)
    c.lib = Q.qpat_mesh(c.xyz, c.tets)
    c.kt, c.mt = np.log(c.kappa / np.median(c.kappa)), np.log(c.mu / np.median(c.mu))
    c.rhs = np.random.default_rng(123).standard_normal(2 * c.N)
    yield c
    c.lib.close()


def prior(c, **prm):
    c.lib.reset_stats()
    x = Q.qpat_prior_solve(c.lib, c.kt, c.mt, c.rhs, Q.qpat_default_params(**prm))
    return x, c.lib.stats()["pcg_iters"]


def test_prior_polynomial_and_jacobi(big):
    p = Q.qpat_default_params()
    Md = O.prior_matrix(big.om, big.kt, big.mt, p.T, p.b_over_a, p.delta)
    norm = abs(Md).sum(axis=0).max()
    (x0, it0), (x2, it2), (xm, itm) = prior(big, pcg_variant=1, prior_poly_degree=0), prior(big, pcg_variant=1), prior(big, multigrid=1)
    for x in (x0, x2, xm):
        assert np.linalg.norm(Md @ x - big.rhs, 1) / (norm * np.linalg.norm(x, 1) + np.linalg.norm(big.rhs, 1)) < 1e-13
    assert rel(x2, x0) < 1e-8 and rel(xm, x0) < 1e-8
    assert it2 < 0.7 * it0  # the polynomial roughly halves the count
    assert itm < 0.2 * it2


@pytest.mark.parametrize("op", [0, 1])
def test_refinement(big, op):
    p = Q.qpat_default_params(precision=1, fp32_operator=op, pcg_variant=1)
    big.lib.reset_stats()
    phi, h = Q.qpat_forward(big.lib, big.kappa, big.mu, big.flux, p)
    assert big.lib.stats()["refinements"] >= 2 and big.lib.stats()["fp64_fallbacks"] == 0
    for k in range(big.K):
        f = O.load_vector(big.om, big.flux[k])
        assert np.linalg.norm(big.Kmat @ phi[k] - f) / np.linalg.norm(f) < 1e-12
    rng = np.random.default_rng(3)
    s, t, lin = rng.standard_normal(2 * big.N), rng.standard_normal((big.K, big.N)), smooth_phi(big.xyz, big.K, big.cfg.L, 5)
    jv, jt = Q.qpat_jvp_vjp_pair(big.lib, big.kappa, big.mu, lin, s, t, None, p)
    assert abs(np.sum(jv * t) - s @ jt) <= 1e-10 * abs(np.sum(jv * t))


@pytest.fixture(scope="module")
def middle():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Case(S.small_config(13, 12.0, 5, 3))
    c.lib = Q.qpat_mesh(c.xyz, c.tets, patch_nodes=128)
    yield c
    c.lib.close()


@pytest.mark.parametrize("restart", [0, 1])
@pytest.mark.parametrize("op", [0, 1])
def test_reliable_updates_and_restarts(middle, restart, op):
    c = middle
    p = Q.qpat_default_params(precision=1, fp32_operator=op, mixed_restart=restart, pcg_variant=1)
    c.lib.reset_stats()
    assert rel(Q.qpat_forward(c.lib, c.kappa, c.mu, c.flux, p)[0], c.phi) < 1e-10
    assert c.lib.stats()["refinements"] >= 2
    s = np.random.default_rng(12).standard_normal(2 * c.N)
    assert rel(Q.qpat_jvp(c.lib, c.kappa, c.mu, c.phi, s, c.w, p), O.jvp(c.om, c.kappa, c.mu, c.phi, s, c.w, c.fac)) < 1e-10


@pytest.mark.parametrize("deg", [1, 2, 4, 8])
def test_prior_degrees(middle, deg):
    c = middle
    rng = np.random.default_rng(13)
    kt, mt, rhs = 0.3 * rng.standard_normal(c.N), np.log(c.mu / c.mu.mean()), rng.standard_normal(2 * c.N)
    Md = O.prior_matrix(c.om, kt, mt, 1e-2, 0.7, 1e-6)
    iters = []
    for d in (0, deg):
        c.lib.reset_stats()
        x = Q.qpat_prior_solve(c.lib, kt, mt, rhs, Q.qpat_default_params(T=1e-2, b_over_a=0.7, prior_poly_degree=d, pcg_variant=1))
        iters.append(c.lib.stats()["pcg_iters"])
        norm = abs(Md).sum(axis=0).max()
        assert np.linalg.norm(Md @ x - rhs, 1) / (norm * np.linalg.norm(x, 1) + np.linalg.norm(rhs, 1)) < 1e-13
    assert iters[1] <= iters[0]


def test_coarsest_level(middle, big):
    for c in (middle, big):
        Q.qpat_forward(c.lib, c.kappa, c.mu, c.flux, Q.qpat_default_params(multigrid=1))
        assert c.lib.multigrid_levels()[-1] <= 64


@pytest.mark.parametrize("deg", [0, 2])
def test_batch_of_many_illuminations(deg):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bodies = [Case(S.small_config(n, 12.0, K, 3)) for n, K in ((13, 8), (12, 6), (15, 5), (11, 1))]
    meshes = [Q.qpat_mesh(c.xyz, c.tets, patch_nodes=256) for c in bodies]
    batch = Q.qpat_batch_create(meshes, [c.K for c in bodies], Q.qpat_default_params(poly_degree=deg))
    for j, c in enumerate(bodies):
        for to, a in zip(batch.inputs(j), (c.kappa, c.mu, c.flux)):
            to.copy_(torch.tensor(a))
    batch.forward()
    torch.cuda.synchronize()
    for j, c in enumerate(bodies):
        assert rel(batch.phi(j).cpu().numpy(), c.phi) < 1e-10
    batch.close()
    for m in meshes:
        m.close()


class FreeBody:
    """A cube whose inner nodes are displaced at random and whose nodes and tets are renumbered and turned over."""

    def __init__(self, n, seed):
        xyz, tets = S.kuhn_cube(n, 20.0)
        rng = np.random.default_rng(seed)
        inner = (xyz > 1e-9) & (xyz < 20.0 - 1e-9)
        xyz = xyz + np.where(inner, rng.uniform(-0.25, 0.25, xyz.shape) * 20.0 / (n - 1), 0.0)
        to = rng.permutation(len(xyz))
        xyz, tets = xyz[np.argsort(to)], to[tets][rng.permutation(len(tets))]
        turned = rng.random(len(tets)) < 0.5
        tets[turned] = tets[turned][:, [1, 0, 2, 3]]
        self.xyz, self.tets = xyz, tets.astype(np.int32)
        self.kappa, self.mu = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0]), 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
        self.mesh = Q.qpat_mesh(self.xyz, self.tets)
        self.flux = rng.uniform(0.0, 1.0, (16, self.mesh.F))
        self.rhs = rng.standard_normal(2 * len(xyz))


@pytest.mark.parametrize("n", [9, 14, 29])
def test_free_mesh_defaults(n):
    """29^3 nodes x 16 right-hand sides lie above the line of such meshes, the others below."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = FreeBody(n, n)
    om = O.Mesh(b.xyz, b.tets)
    Kmat = O.system_matrix(om, b.kappa, b.mu)
    for prm in (dict(), dict(precision=1), dict(multigrid=1), dict(multigrid=2)):
        phi, _ = Q.qpat_forward(b.mesh, b.kappa, b.mu, b.flux, Q.qpat_default_params(**prm))
        for k in (0, 15):
            f = O.load_vector(om, b.flux[k])
            assert np.linalg.norm(Kmat @ phi[k] - f) / np.linalg.norm(f) < 1e-12
    kt, mt = np.log(b.kappa / 0.3), np.log(b.mu / 0.02)
    p = Q.qpat_default_params(T=2e-2)
    Md = O.prior_matrix(om, kt, mt, p.T, p.b_over_a, p.delta)
    x = Q.qpat_prior_solve(b.mesh, kt, mt, b.rhs, p)
    norm = abs(Md).sum(axis=0).max()
    assert np.linalg.norm(Md @ x - b.rhs, 1) / (norm * np.linalg.norm(x, 1) + np.linalg.norm(b.rhs, 1)) < 1e-13
    b.mesh.close()


def test_two_handles_on_two_streams():
    """Solves of two meshes whose calls alternate between two streams give the bits of the meshes one after the other."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bodies = [FreeBody(14, 1), FreeBody(16, 2)]
    streams = [torch.cuda.Stream() for _ in bodies]
    data = [[torch.tensor(a, device="cuda") for a in (np.log(b.kappa / 0.3), np.log(b.mu / 0.02), b.rhs)] for b in bodies]
    p = Q.qpat_default_params(T=2e-2)
    torch.cuda.synchronize()
    want = [Q.qpat_prior_solve_dev(b.mesh, *d, torch.empty_like(d[2]), p).clone() for b, d in zip(bodies, data)]
    torch.cuda.synchronize()
    for _ in range(3):
        out = []
        for b, d, s in zip(bodies, data, streams):
            with torch.cuda.stream(s):
                out.append(Q.qpat_prior_solve_dev(b.mesh, *d, torch.empty_like(d[2]), p))
        torch.cuda.synchronize()
        for a, c in zip(out, want):
            assert torch.equal(a, c)
    for b in bodies:
        b.mesh.close()
