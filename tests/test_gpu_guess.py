"""Initial guesses of the forward solve (qpat_forward_guess_dev) change the
work, not the answer, for every solver: an unlit illumination has the
solution 0 whatever its guess, and a guess that already meets the target is
returned.

Tolerances: a solve of residual 1e-13 lies within 1e-10 of the oracle
(cond(K) < 1e3); an unlit column is compared with the lit ones' scale, of
which the guess is of order 1, so it lies within 1e-10 of that scale."""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu

# the persistent solvers, the library's choice (multigrid at this size) and the multigrid CG by name
SOLVERS = [dict(), dict(multigrid=1), dict(multigrid=2), dict(multigrid=1, mg_degree=2), dict(pcg_variant=1),
           dict(precision=1), dict(precision=1, fp32_operator=1), dict(precision=1, fp32_operator=1, pcg_variant=1)]


@pytest.fixture(scope="module")
def body():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = S.kuhn_cube(21, 20.0)
    om = O.Mesh(xyz, tets)
    kappa = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0])
    mu = 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
    flux = np.random.default_rng(5).uniform(0.0, 1.0, (16, om.F))
    phi, _ = O.forward(om, kappa, mu, flux, O.Factor(O.system_matrix(om, kappa, mu)))
    mesh = Q.qpat_mesh(xyz, tets)
    yield mesh, kappa, mu, flux, phi
    mesh.close()


def forward(mesh, kappa, mu, flux, guess, prm):
    d = [torch.tensor(a, device="cuda") for a in (kappa, mu, flux, guess)]
    phi, h = torch.empty_like(d[3]), torch.empty_like(d[3])
    Q.qpat_forward_guess_dev(mesh, *d, phi, h, Q.qpat_default_params(**prm))
    return phi.cpu().numpy(), h.cpu().numpy()


@pytest.mark.parametrize("K", [2, 3, 8, 16])
@pytest.mark.parametrize("prm", SOLVERS, ids=str)
def test_unlit_illumination(body, prm, K):
    mesh, kappa, mu, flux, ref = body
    dark = np.zeros(K, bool)
    dark[1::2] = True
    f, want = flux[:K] * ~dark[:, None], ref[:K] * ~dark[:, None]
    guess = ref[:K] * (1.0 + 1e-2 * np.cos(np.arange(mesh.N)))
    phi, h = forward(mesh, kappa, mu, f, guess, prm)
    assert rel(phi, want) < 1e-10
    assert rel(h, mu * want) < 1e-10


@pytest.mark.parametrize("prm", SOLVERS, ids=str)
def test_all_unlit(body, prm):
    mesh, kappa, mu, flux, ref = body
    phi, h = forward(mesh, kappa, mu, 0.0 * flux[:3], ref[:3], prm)
    assert np.linalg.norm(phi) < 1e-10 * np.linalg.norm(ref[:3])
    assert np.linalg.norm(h) < 1e-10 * np.linalg.norm(mu * ref[:3])


@pytest.mark.parametrize("prm", SOLVERS, ids=str)
def test_guess_that_is_the_solution(body, prm):
    """Solved to 1e-13 and handed in against a target of 1e-9: nothing is left to do; mixed with a poor guess."""
    mesh, kappa, mu, flux, ref = body
    phi, _ = forward(mesh, kappa, mu, flux[:4], 0.0 * ref[:4], prm)
    loose = dict(prm, pcg_rtol=1e-9)
    again, _ = forward(mesh, kappa, mu, flux[:4], phi, loose)
    assert rel(again, phi) < 1e-10
    half = phi.copy()
    half[2:] = 0.0
    mixed, _ = forward(mesh, kappa, mu, flux[:4], half, loose)
    assert rel(mixed[:2], phi[:2]) < 1e-10
    assert rel(mixed[2:], phi[2:]) < 1e-6  # residual 1e-9 times cond(K) < 1e3
