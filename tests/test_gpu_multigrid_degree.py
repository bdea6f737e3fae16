"""mg_degree: the smoothing polynomial on the fine level.  Every degree gives the
same solution, a higher one takes no more iterations, and it adds two kernels an
iteration for each degree and five for the second, however many levels there are
(the coarser levels take one step each).

Tolerances: 1e-10 between K solves of residual 1e-13 (cond(K) < 1e3), a normwise backward error of 1e-13 for M_delta."""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["cube13", "cube21", "cyl11x14", "cube3"])
def body(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = {"cube13": lambda: S.kuhn_cube(13, 20.0), "cube21": lambda: S.kuhn_cube(21, 20.0),
                 "cyl11x14": lambda: S.cylinder_mesh(11, 14, 10.0, 12.0), "cube3": lambda: S.kuhn_cube(3, 20.0)}[request.param]()
    mesh = Q.qpat_mesh(xyz, tets)
    kappa, mu = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0]), 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
    yield mesh, O.Mesh(xyz, tets), kappa, mu, np.random.default_rng(5).uniform(0.0, 1.0, (16, mesh.F))
    mesh.close()


def counted(mesh, call):
    mesh.reset_stats()
    before = Q.qpat_launch_count()
    out = call()
    return out, mesh.stats()["pcg_iters"], Q.qpat_launch_count() - before


@pytest.mark.parametrize("cycle", [1, 2])
@pytest.mark.parametrize("K", [1, 2, 4, 7, 16])
def test_forward(body, cycle, K):
    mesh, om, kappa, mu, flux = body
    want = O.forward(om, kappa, mu, flux[:K], O.Factor(O.system_matrix(om, kappa, mu)))[0]
    kernels, iters = {}, {}
    for d in (1, 2, 3, 5, 8):
        run = lambda rtol: counted(mesh, lambda: Q.qpat_forward(  # noqa: E731
            mesh, kappa, mu, flux[:K], Q.qpat_default_params(multigrid=cycle, mg_degree=d, pcg_rtol=rtol))[0])
        out, iters[d], n = run(1e-13)
        assert rel(out, want) < 1e-10
        _, few, m = run(1e-3)
        if iters[d] > few:
            assert (n - m) % (iters[d] - few) == 0
            kernels[d] = (n - m) // (iters[d] - few)
    if len(mesh.multigrid_levels()) > 1:
        assert iters[8] <= iters[5] <= iters[3] <= iters[1]
        for d in kernels:
            assert kernels[d] == kernels[1] + (0 if d == 1 else 5 + 2 * (d - 2) + (cycle == 2))


def test_prior(body):
    mesh, om, kappa, mu, _ = body
    kt, mt = np.log(kappa / 0.3), np.log(mu / 0.02)
    rhs = np.random.default_rng(1).standard_normal(2 * om.N)
    iters = {}
    for d in (1, 2, 3, 8):
        prm = Q.qpat_default_params(multigrid=1, mg_degree=d, T=2e-2)
        x, iters[d], _ = counted(mesh, lambda: Q.qpat_prior_solve(mesh, kt, mt, rhs, prm))
        M = O.prior_matrix(om, kt, mt, prm.T, prm.b_over_a, prm.delta)
        eta = np.linalg.norm(M @ x - rhs, 1) / (abs(M).sum(axis=0).max() * np.linalg.norm(x, 1) + np.linalg.norm(rhs, 1))
        assert eta < 1e-13
    assert iters[8] <= iters[3] <= iters[1]
