"""Element sums taken as gathers over the mesh's element plan (assembly of K
and of M_delta, the right-hand side of J s, the accumulation of J^T t) against
the oracle, at the sizes where the plan's lists are short or ragged: the
smallest cube, odd cubes, a cylinder, and a cube whose nodes and tets are
numbered at random and turned over; 1 to 16 illuminations (padded widths 1,
2, 4, 8, 16).

Tolerances: the assembled product differs from the oracle's by summation
order only (about 30 terms a row, a few eps each: 1e-13 of the result's
norm); J s and J^T t by the solves' relative residual 1e-13 times cond(K) < 1e3
(1e-10); the M_delta solve has a normwise backward error below 1e-13.
"""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


def mesh_arrays(name):
    if name == "cyl":
        return S.cylinder_mesh(7, 5, 10.0, 8.0)
    n = {"n2": 2, "n3": 3, "n10": 10, "n10mixed": 10}[name]
    xyz, tets = S.kuhn_cube(n, 10.0)
    if name == "n10mixed":
        rng = np.random.default_rng(4)
        to = rng.permutation(len(xyz))
        tets = to[tets][rng.permutation(len(tets))]
        turned = rng.random(len(tets)) < 0.5
        tets[turned] = tets[turned][:, [1, 0, 2, 3]]
        xyz = xyz[np.argsort(to)]
    return xyz, tets.astype(np.int32)


@pytest.fixture(scope="module", params=["n2", "n3", "n10", "n10mixed", "cyl"])
def body(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = mesh_arrays(request.param)
    om = O.Mesh(xyz, tets)
    rng = np.random.default_rng(11)
    kappa, mu = rng.uniform(0.2, 0.5, om.N), rng.uniform(0.005, 0.05, om.N)
    mesh = Q.qpat_mesh(xyz, tets, patch_nodes=32)
    yield om, kappa, mu, mesh
    mesh.close()


def test_assembled_K(body):
    om, kappa, mu, mesh = body
    x = np.random.default_rng(1).standard_normal((om.N, 4))
    t = [torch.tensor(a, device="cuda") for a in (kappa, mu, x)]
    y = Q.qpat_apply_K_dev(mesh, *t, torch.empty_like(t[2]), 2).cpu().numpy()
    assert rel(y, O.system_matrix(om, kappa, mu) @ x) < 1e-13


@pytest.mark.parametrize("K", [1, 2, 3, 7, 16])
def test_jacobian_products(body, K):
    om, kappa, mu, mesh = body
    rng = np.random.default_rng(K)
    phi, w, t = rng.uniform(0.1, 1.0, (K, om.N)), rng.uniform(0.5, 2.0, (K, om.N)), rng.standard_normal((K, om.N))
    s = rng.standard_normal(2 * om.N)
    fac = O.Factor(O.system_matrix(om, kappa, mu))
    assert rel(Q.qpat_jvp(mesh, kappa, mu, phi, s, w), O.jvp(om, kappa, mu, phi, s, w, fac)) < 1e-10
    out, ref = Q.qpat_vjp(mesh, kappa, mu, phi, t, w), O.vjp(om, kappa, mu, phi, t, w, fac)
    assert rel(out[:om.N], ref[:om.N]) < 1e-10
    assert rel(out[om.N:], ref[om.N:]) < 1e-10


@pytest.mark.parametrize("prior", [0, 1])
def test_prior_blocks(body, prior):
    om, kappa, mu, mesh = body
    rng = np.random.default_rng(prior)
    kt, mt, rhs = 0.3 * rng.standard_normal(om.N), 0.3 * rng.standard_normal(om.N), rng.standard_normal(2 * om.N)
    prm = Q.qpat_default_params(prior=prior, prior_q=0.7, T=2e-2)
    x = Q.qpat_prior_solve(mesh, kt, mt, rhs, prm)
    M = O.prior_matrix(om, kt, mt, prm.T, prm.b_over_a, prm.delta, prior=prior, q=0.7)
    eta = np.linalg.norm(M @ x - rhs, 1) / (abs(M).sum(axis=0).max() * np.linalg.norm(x, 1) + np.linalg.norm(rhs, 1))
    assert eta < 1e-13
