"""Problems of one batch with different numbers of illuminations: each is
solved with its own number of right-hand sides (1, 2, 4 or 8), whatever the
largest of the batch, and with its share of the launch's CTAs."""
import numpy as np
import pytest

import qpat_synth as S
from tests.gpu_common import rel

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg", [0, 2])
@pytest.mark.parametrize("sizes", [
    [(4, 8), (11, 1), (6, 2), (9, 3)],   # every kernel width in one launch
    [(3, 1), (14, 1)],                   # width 1 alone, a mesh of one patch beside one of many
    [(8, 2), (5, 1), (12, 2)],
    [(10, 5)],                           # one problem has the launch for itself
])
def test_each_problem_at_its_own_width(sizes, deg):
    """Both solvers stop at a residual of 1e-13; the single solve of the same
    mesh and flux is the reference (1e-10, as for batches of any kind)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfgs = [S.small_config(n, 2.0 * n, K, 300 + i) for i, (n, K) in enumerate(sizes)]
    meshes, data = [], []
    for cfg in cfgs:
        xyz, tets = cfg.mesh()
        kap, mu = cfg.coefficients(xyz)
        m = Q.qpat_mesh(xyz, tets, patch_nodes=32)
        flux = np.stack([Q.qpat_flux_patch(m, p.center, p.normal, p.half_w, p.amp) for p in cfg.patches])
        meshes.append(m)
        data.append((kap, mu, flux))
    batch = Q.qpat_batch_create(meshes, [c.K for c in cfgs], Q.qpat_default_params(poly_degree=deg))
    try:
        for j, (kap, mu, flux) in enumerate(data):
            for to, v in zip(batch.inputs(j), (kap, mu, flux)):
                to.copy_(torch.tensor(v))
        batch.forward()
        torch.cuda.synchronize()
        st, it, ct = batch.status()
        assert all(s == 0 for s in st), st
        assert all(c >= 1 for c in ct)
        for j, (kap, mu, flux) in enumerate(data):
            ref, _ = Q.qpat_forward(meshes[j], kap, mu, flux)
            assert rel(batch.phi(j).cpu().numpy(), ref) < 1e-10
    finally:
        batch.close()
        for m in meshes:
            m.close()
