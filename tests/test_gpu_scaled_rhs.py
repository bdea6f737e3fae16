"""Small and large right-hand sides: K phi = f is linear and every number of a
solve is scaled by a power of two without rounding, so phi / 2^e for the fluxes
times 2^e has the same bits for every e, also where 2^e is far outside FP32's
range and the multigrid cycle runs in FP32."""
import numpy as np
import pytest

import qpat_synth as S

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def body():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = S.kuhn_cube(13, 20.0)
    mesh = Q.qpat_mesh(xyz, tets)
    kappa = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0])
    mu = 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
    yield mesh, kappa, mu, np.random.default_rng(5).uniform(0.0, 1.0, (8, mesh.F))
    mesh.close()


@pytest.mark.parametrize("K", [1, 3, 8])
@pytest.mark.parametrize("prm", [dict(multigrid=1), dict(multigrid=2), dict(multigrid=2, mg_degree=2), dict(precision=1)], ids=str)
def test_power_of_two(body, prm, K):
    mesh, kappa, mu, flux = body
    p = Q.qpat_default_params(**prm)
    # one column stays as it is: every right-hand side has a scale of its own
    keep = np.arange(K) == 1
    want = Q.qpat_forward(mesh, kappa, mu, flux[:K], p)[0]
    for e in (-400, -100, -40, 40, 100, 400):
        s = np.where(keep, 1.0, 2.0 ** e)[:, None]
        got = Q.qpat_forward(mesh, kappa, mu, s * flux[:K], p)[0]
        np.testing.assert_array_equal(got / s, want)
