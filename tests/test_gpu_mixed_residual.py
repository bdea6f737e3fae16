"""precision 1 stops on the FP64 residual f - K phi, whichever solver the library
takes for it, and goes as far beyond the target as its last sweep takes it.

Tolerance: with the defaults the sweeps end at a residual of 1e-16 |f| or, where
rounding does not allow that, near the residual of the rounded solution; the
last sweep's dozen or so additions to phi, the final sum and the rounding of K
itself each add about as much again, so 20 times that residual bounds it.  The
residuals are formed in extended precision (on the oracle's K)."""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


class Exact:
    """K, the solution and residual norms in extended precision."""

    def __init__(self, xyz, tets, kappa, mu, flux):
        om = O.Mesh(xyz, tets)
        A = O.system_matrix(om, kappa, mu)
        fac, c = O.Factor(A), A.tocoo()
        self.row, self.col, self.val = c.row, c.col, c.data.astype(np.longdouble)
        self.b = np.stack([O.load_vector(om, f) for f in flux]).astype(np.longdouble)
        x = O.forward(om, kappa, mu, flux, fac)[0].astype(np.longdouble)
        for _ in range(3):
            x = x + np.stack([fac.solve(np.asarray(r, dtype=float)) for r in self.residual(x)])
        self.floor = self.norm(x.astype(float))

    def residual(self, x):
        out = self.b.copy()
        for k, v in enumerate(np.asarray(x, dtype=np.longdouble)):
            np.subtract.at(out[k], self.row, self.val * v[self.col])
        return out

    def norm(self, x):
        return np.sqrt((self.residual(x) ** 2).sum(1) / (self.b ** 2).sum(1)).astype(float)


@pytest.mark.parametrize("n", [9, 13, 21])
@pytest.mark.parametrize("prm", [{}, dict(fp32_operator=1), dict(pcg_variant=1), dict(fp32_operator=1, pcg_variant=1)], ids=str)
@pytest.mark.parametrize("guess", [False, True])
def test_residual(n, prm, guess):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = S.kuhn_cube(n, 20.0)
    kappa = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0])
    mu = 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
    mesh = Q.qpat_mesh(xyz, tets)
    flux = np.random.default_rng(n).uniform(0.0, 1.0, (3, mesh.F))
    exact = Exact(xyz, tets, kappa, mu, flux)
    d = [torch.tensor(a, device="cuda") for a in (kappa, mu, flux, np.ones((3, mesh.N)))]
    phi, h = torch.empty_like(d[3]), torch.empty_like(d[3])
    p = Q.qpat_default_params(precision=1, **prm)
    mesh.reset_stats()
    Q.qpat_forward_guess_dev(mesh, *d, phi, h, p) if guess else Q.qpat_forward_dev(mesh, *d[:3], phi, h, p)
    assert mesh.stats()["refinements"] >= 2
    assert (exact.norm(phi.cpu().numpy()) < 20 * exact.floor).all()
    mesh.close()


@pytest.mark.parametrize("prm", [{}, dict(fp32_operator=1)], ids=str)
def test_target_below_rounding(prm):
    """Coefficients over ten decades, so that no FP64 vector has a residual of 1e-13 |f|: the call still ends, and its
    residual is of the size of the FP64 solver's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = S.kuhn_cube(13, 20.0)
    rng = np.random.default_rng(0)
    kappa, mu = 10.0 ** rng.uniform(-5, 5, len(xyz)), 10.0 ** rng.uniform(-5, 0, len(xyz))
    mesh = Q.qpat_mesh(xyz, tets)
    flux = rng.uniform(0.0, 1.0, (3, mesh.F))
    exact = Exact(xyz, tets, kappa, mu, flux)
    assert exact.floor.min() > 2e-13
    fp64 = exact.norm(Q.qpat_forward(mesh, kappa, mu, flux, Q.qpat_default_params(pcg_variant=1))[0])
    got = exact.norm(Q.qpat_forward(mesh, kappa, mu, flux, Q.qpat_default_params(precision=1, **prm))[0])
    assert (got < 20 * np.maximum(exact.floor, fp64)).all()
    assert mesh.stats()["fp64_fallbacks"] == 1
    mesh.close()
