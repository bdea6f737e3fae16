"""Which solver a call that names none takes, seen by whether the multigrid
solver holds memory afterwards: only one that was measured faster on meshes of
its kind.  The persistent solver on meshes that are no grids of right-angled tets
for K with one right-hand side, whatever their size, and with several below
350,000 unknowns; its FP32 form with the operator that fp32_operator names but
on large grids; the multigrid CG on grids and for M_delta."""
import numpy as np
import pytest

import qpat_synth as S

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


def body(kind, n):
    """A cube's grid, or one whose inner nodes are displaced at random and whose nodes are renumbered."""
    xyz, tets = S.kuhn_cube(n, 20.0)
    if kind == "grid":
        return xyz, tets
    rng = np.random.default_rng(n)
    inner = (xyz > 1e-9) & (xyz < 20.0 - 1e-9)
    xyz = xyz + np.where(inner, rng.uniform(-0.2, 0.2, xyz.shape) * 20.0 / (n - 1), 0.0)
    to = rng.permutation(len(xyz))
    return xyz[np.argsort(to)], to[tets].astype(np.int32)


# (mesh, nodes a side, K right-hand sides or "prior", parameters, multigrid)
CALLS = [("grid", 9, 1, {}, False), ("grid", 21, 2, {}, True), ("grid", 37, 1, {}, True), ("grid", 25, 1, {}, False),
         ("free", 21, 8, {}, False), ("free", 37, 1, {}, False), ("free", 37, 2, {}, False), ("free", 37, 8, {}, True),
         ("free", 29, 16, {}, True), ("grid", 9, "prior", {}, False), ("free", 13, "prior", {}, True),
         ("grid", 9, 1, dict(precision=1), False), ("grid", 13, 1, dict(precision=1), True), ("free", 13, 1, dict(precision=1), False),
         ("free", 13, 4, dict(precision=1), True), ("grid", 37, 8, dict(precision=1, fp32_operator=1), False),
         ("free", 37, 16, dict(precision=1, fp32_operator=1), False), ("grid", 59, 1, dict(precision=1, fp32_operator=1), True),
         ("grid", 37, 8, dict(pcg_variant=1), False), ("grid", 37, 8, dict(poly_degree=1), False), ("grid", 13, "prior", dict(prior_poly_degree=0), False)]


@pytest.mark.parametrize("kind,n,what,prm,multigrid", CALLS, ids=lambda v: str(v))
def test_choice(kind, n, what, prm, multigrid):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets = body(kind, n)
    mesh = Q.qpat_mesh(xyz, tets)
    kappa = 0.3 + 0.1 * np.sin(0.3 * xyz[:, 0])
    mu = 0.02 + 0.01 * np.cos(0.2 * xyz[:, 1])
    rng = np.random.default_rng(0)
    p = Q.qpat_default_params(**prm)
    if what == "prior":
        Q.qpat_prior_solve(mesh, np.log(kappa / 0.3), np.log(mu / 0.02), rng.standard_normal(2 * mesh.N), p)
    else:
        Q.qpat_forward(mesh, kappa, mu, rng.uniform(0.0, 1.0, (what, mesh.F)), p)
    assert (mesh.multigrid_bytes() > 0) == multigrid
    mesh.close()
