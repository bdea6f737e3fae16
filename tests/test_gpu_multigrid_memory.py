"""The multigrid solver with too little device memory (a limit on what it may
hold, so that each of its allocations is the one that fails for some limit): a
solve that names it fails with an error and leaves nothing half-built, however
often it is called; one that leaves the choice to the library gets the
persistent solver's result; and once the memory is there the next solve runs.

Tolerances: two K solves of residual 1e-13 differ by less than 1e-10 (cond(K) < 1e3);
the same solver on the same inputs gives the same bits, but for the matrix-free
FP32 operator, whose shared-memory sums run in no fixed order."""
import numpy as np
import pytest

import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu

N_SIDE = 21  # above every line of the library's choice for K


@pytest.fixture(scope="module")
def inputs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = S.kuhn_cube(N_SIDE, 20.0)
    rng = np.random.default_rng(1)
    kappa = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0])
    mu = 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
    return xyz, tets, kappa, mu, rng.uniform(0.0, 1.0, (4, 12 * (N_SIDE - 1) ** 2)), rng.standard_normal(2 * len(xyz))


def solve(mesh, kind, inputs, **prm):
    _, _, kappa, mu, flux, rhs = inputs
    p = Q.qpat_default_params(**prm)
    if kind == "prior":
        return Q.qpat_prior_solve(mesh, np.log(kappa / 0.3), np.log(mu / 0.02), rhs, p)
    return Q.qpat_forward(mesh, kappa, mu, flux, p)[0]


FORMS = [("K", dict(multigrid=1)), ("K", dict(multigrid=2)), ("K", dict(multigrid=1, mg_degree=2)), ("prior", dict(multigrid=1))]


@pytest.mark.parametrize("kind,named", FORMS, ids=str)
def test_every_allocation_can_fail(inputs, kind, named):
    mesh = Q.qpat_mesh(*inputs[:2])
    want = solve(mesh, kind, inputs, **named)
    full = mesh.multigrid_bytes()
    assert full > 0
    mesh.close()
    for part in np.linspace(0.0, 1.0, 41)[:-1]:
        mesh = Q.qpat_mesh(*inputs[:2])
        mesh.set_multigrid_limit(max(1, int(part * full)))
        for _ in range(2):
            with pytest.raises(Q.QpatError, match="multigrid"):
                solve(mesh, kind, inputs, **named)
            assert mesh.multigrid_bytes() <= max(1, int(part * full))
        mesh.set_multigrid_limit(0)
        np.testing.assert_array_equal(solve(mesh, kind, inputs, **named), want)
        assert mesh.multigrid_bytes() == full
        mesh.close()


@pytest.mark.parametrize("kind,prm,bits", [("K", {}, True), ("K", dict(precision=1), False), ("prior", {}, True)], ids=str)
def test_default_solves_go_on(inputs, kind, prm, bits):
    mesh = Q.qpat_mesh(*inputs[:2])
    chosen = solve(mesh, kind, inputs, **prm)
    full = mesh.multigrid_bytes()
    assert full > 0  # the library's choice at this size is multigrid
    persistent = solve(mesh, kind, inputs, pcg_variant=1, **prm)
    if kind == "K":
        assert rel(chosen, persistent) < 1e-10
    mesh.close()
    for part in (0.0, 0.1, 0.3, 0.5, 0.7, 0.8, 0.9, 0.95, 0.99):
        mesh = Q.qpat_mesh(*inputs[:2])
        mesh.set_multigrid_limit(max(1, int(part * full)))
        for _ in range(3):
            again = solve(mesh, kind, inputs, **prm)
            assert np.array_equal(again, persistent) if bits else rel(again, persistent) < 1e-10
        mesh.close()


def test_failed_form_leaves_the_others(inputs):
    """The FP32 cycle's values do not fit beside the FP64 cycle's: those are rebuilt and still give the same bits."""
    mesh = Q.qpat_mesh(*inputs[:2])
    a = solve(mesh, "K", inputs, multigrid=1)
    mesh.set_multigrid_limit(mesh.multigrid_bytes())
    with pytest.raises(Q.QpatError, match="multigrid"):
        solve(mesh, "K", inputs, multigrid=2)
    np.testing.assert_array_equal(solve(mesh, "K", inputs, multigrid=1), a)
    mesh.close()


@pytest.mark.parametrize("K", [8, 16])
def test_vectors_of_the_default_cycle(inputs, K):
    """Per unknown: CG's five vectors, the fine residual, and three vectors on levels that together have a sixth of the fine
    level's rows."""
    xyz, tets, kappa, mu, flux, _ = inputs
    mesh = Q.qpat_mesh(xyz, tets)
    p = Q.qpat_default_params(multigrid=1)
    Q.qpat_forward(mesh, kappa, mu, flux[:1], p)
    before = mesh.multigrid_bytes()
    Q.qpat_forward(mesh, kappa, mu, np.tile(flux, (4, 1))[:K], p)
    assert mesh.multigrid_bytes() - before < 8 * 6.6 * K * mesh.N + (1 << 20)
    mesh.close()
