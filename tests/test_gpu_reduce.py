"""Grid reductions of the persistent solvers at launches of few CTAs, at the
edges of the CTA groups and of many CTAs."""
import numpy as np
import pytest

import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


def solve(mesh, patches, kap, mu, **prm):
    flux = np.stack([Q.qpat_flux_patch(mesh, p.center, p.normal, p.half_w, p.amp) for p in patches])
    phi, _ = Q.qpat_forward(mesh, kap, mu, flux, params=Q.qpat_default_params(**prm))
    return phi


@pytest.mark.parametrize("variant", [1, 2, 3])
@pytest.mark.parametrize("n,K", [
    (3, 1),      # one CTA
    (12, 1),     # 54: every CTA reads all the others
    (13, 4),     # 69: five groups, the last of five CTAs
    (13, 8),
    (24, 1),     # 432: 27 groups, or two patches a CTA where fewer are resident
    (16, 16),    # 48 totals in the first reduction
])
def test_reductions_by_number_of_ctas(n, K, variant):
    """One system cut into different numbers of CTAs: both solves stop at a
    relative residual of 1e-13, so that their solutions agree to 1e-10."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfg = S.small_config(n, 2.0 * n, K, 700 + n)
    xyz, tets = cfg.mesh()
    kap, mu = cfg.coefficients(xyz)
    few = Q.qpat_mesh(xyz, tets, patch_nodes=256)
    many = Q.qpat_mesh(xyz, tets, patch_nodes=32)
    try:
        ref = solve(few, cfg.patches, kap, mu, pcg_variant=1)
        for rep in range(2):  # the second starts from the first's slots
            assert rel(solve(many, cfg.patches, kap, mu, pcg_variant=variant), ref) < 1e-10
    finally:
        few.close()
        many.close()
