"""The lagged weights of M_delta for fields and scales far from the ordinary:
gradients whose square overflows, T at the ends of its range, on a grid and on
tets of many shapes (whose stiffness factors have both signs).

Tolerances: weights of 0 leave delta I, which the solve inverts to a residual of 1e-13; elsewhere the
normwise backward error of a solve of that residual, 1e-12."""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


def backward_error(M, x, b):
    return np.linalg.norm(M @ x - b, 1) / (abs(M).sum(axis=0).max() * np.linalg.norm(x, 1) + np.linalg.norm(b, 1))


def body(kind):
    return S.kuhn_cube(7, 10.0) if kind == "cube" else S.cylinder_mesh(7, 5, 10.0, 8.0)


@pytest.mark.parametrize("prior,q", [(0, 1.0), (1, 1.0), (1, 0.5)])
@pytest.mark.parametrize("kind", ["cube", "cyl"])
def test_gradients_beyond_the_range_of_their_square(kind, prior, q):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = body(kind)
    om, mesh = O.Mesh(xyz, tets), Q.qpat_mesh(xyz, tets)
    rng = np.random.default_rng(0)
    rhs = rng.standard_normal(2 * om.N)
    flat, steep = np.zeros(om.N), 1e160 * rng.standard_normal(om.N)
    prm = Q.qpat_default_params(prior=prior, prior_q=q)
    half = O.prior_matrix(om, flat, flat, prm.T, prm.b_over_a, prm.delta, prior=prior, q=q)
    for kt, mt, order in ((steep, flat, (0, 1)), (flat, steep, (1, 0))):
        out = Q.qpat_prior_solve(mesh, kt, mt, rhs, prm).reshape(2, -1)
        loose, plain = order
        assert rel(out[loose], rhs.reshape(2, -1)[loose] / prm.delta) < 1e-12
        full = np.zeros((2, om.N))
        full[plain], b = out[plain], np.zeros((2, om.N))
        b[plain] = rhs.reshape(2, -1)[plain]
        assert backward_error(half, full.ravel(), b.ravel()) < 1e-12
    mesh.close()


@pytest.mark.parametrize("kind", ["cube", "cyl"])
@pytest.mark.parametrize("T", [1e-150, 1e-80, 1e-3, 1e3, 1e150])
def test_edge_scales(kind, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = body(kind)
    om, mesh = O.Mesh(xyz, tets), Q.qpat_mesh(xyz, tets)
    rng = np.random.default_rng(0)
    kt, mt, rhs = rng.standard_normal(om.N), rng.standard_normal(om.N), rng.standard_normal(2 * om.N)
    prm = Q.qpat_default_params(T=T)
    out = Q.qpat_prior_solve(mesh, kt, mt, rhs, prm)
    M = O.prior_matrix(om, kt, mt, T, prm.b_over_a, prm.delta)
    assert backward_error(M, out, rhs) < 1e-12
    mesh.close()
