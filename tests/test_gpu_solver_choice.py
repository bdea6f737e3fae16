"""Solves that name no solver (the defaults) take the persistent PCG or the
multigrid CG by size; both reach the same residual, so over every form of
call, on grids and cylinders around the sizes where the choice changes, the
default's result is the persistent PCG's (pcg_variant = 1) within the bars of
either: 1e-10 for the K solves (two solutions of residual 1e-13, cond(K) < 1e3),
and for M_delta 10 cond(M_delta) 1e-13, twice."""
import numpy as np
import pytest

import oracle as O
import qpat_synth as S
from tests.gpu_common import rel
from tests.test_gpu_parity import cond_mdelta

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu

# nodes below, around and above the lines of the choice (512, 1,500 and 8,000 nodes; 180,000 nodes x right-hand sides)
MESHES = {"cube7": (7, None), "cube9": (9, None), "cube17": (17, None), "cube13": (13, None), "cube21": (21, None), "cube25": (25, None), "cyl9x7": (9, 7),
          "cyl25x27": (25, 27)}


@pytest.fixture(scope="module", params=list(MESHES))
def body(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, nz = MESHES[request.param]
    xyz, tets = S.kuhn_cube(n, 20.0) if nz is None else S.cylinder_mesh(n, nz, 10.0, 12.0)
    mesh = Q.qpat_mesh(xyz, tets)
    rng = np.random.default_rng(2)
    x = xyz / 20.0
    kappa = 0.3 + 0.2 * np.sin(3 * x[:, 0] + x[:, 1])
    mu = 0.02 + 0.01 * np.cos(2 * x[:, 1] - 3 * x[:, 2])
    yield mesh, O.Mesh(xyz, tets), kappa, mu, rng
    mesh.close()


@pytest.mark.parametrize("K", [1, 3, 8, 16])
@pytest.mark.parametrize("precision,fp32_operator", [(0, 0), (1, 0), (1, 1)])
def test_default_equals_persistent(body, K, precision, fp32_operator):
    mesh, om, kappa, mu, rng = body
    N = mesh.N
    phi, t, s = rng.uniform(0.1, 1.0, (K, N)), rng.standard_normal((K, N)), rng.standard_normal(2 * N)
    flux = rng.uniform(0.0, 1.0, (K, mesh.F))
    out = []
    for variant in (0, 1):
        p = Q.qpat_default_params(precision=precision, fp32_operator=fp32_operator, pcg_variant=variant)
        o = list(Q.qpat_forward(mesh, kappa, mu, flux, p))
        o += [Q.qpat_jvp(mesh, kappa, mu, phi, s, None, p), Q.qpat_vjp(mesh, kappa, mu, phi, t, None, p)]
        if K <= 8:
            o += list(Q.qpat_jvp_vjp_pair(mesh, kappa, mu, phi, s, t, None, p))
        guess = torch.tensor(o[0] * (1 + 1e-3 * np.cos(np.arange(N))), device="cuda")
        d = [torch.tensor(a, device="cuda") for a in (kappa, mu, flux)]
        g, h = torch.empty_like(guess), torch.empty_like(guess)
        Q.qpat_forward_guess_dev(mesh, *d, guess, g, h, p)
        out.append(o + [g.cpu().numpy(), h.cpu().numpy()])
    for a, b in zip(*out):
        assert rel(a, b) < 1e-10


@pytest.mark.parametrize("prior", [0, 1])
def test_default_prior_equals_persistent(body, prior):
    mesh, om, kappa, mu, rng = body
    kt, mt, rhs = np.log(kappa / 0.3), np.log(mu / 0.02), rng.standard_normal(2 * mesh.N)
    a, b = (Q.qpat_prior_solve(mesh, kt, mt, rhs, Q.qpat_default_params(T=1e-2, prior=prior, pcg_variant=v)) for v in (0, 1))
    cond = cond_mdelta(O.prior_matrix(om, kt, mt, 1e-2, 1.0, 1e-6, prior=prior), 1e-6)
    assert rel(a, b) < 20 * cond * 1e-13
