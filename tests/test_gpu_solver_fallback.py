"""Where the library's own attempt at multigrid cannot solve a system, the call
is the persistent solver's call: the same bits, the same counts, the message of
the last error left alone, and no attempt that is repeated for parts of the
system or, on a mesh without memory for it, by later calls."""
import numpy as np
import pytest

import qpat_synth as S

torch = pytest.importorskip("torch")
Q = pytest.importorskip("paper_1512_02796_gb300")

pytestmark = pytest.mark.gpu


class Body:
    def __init__(self, n, scale=1.0):
        xyz, tets = S.kuhn_cube(n, 20.0)
        self.mesh = Q.qpat_mesh(xyz, tets)
        rng = np.random.default_rng(3)
        self.kappa = scale * (0.3 + 0.1 * np.sin(0.3 * xyz[:, 0]))
        self.mu = scale * (0.02 + 0.01 * np.cos(0.2 * xyz[:, 1]))
        self.flux = rng.uniform(0.0, 1.0, (16, self.mesh.F))
        self.guess = rng.uniform(0.5, 1.0, (16, self.mesh.N)) / scale
        self.rhs = rng.standard_normal(2 * self.mesh.N)

    def forward(self, K, guess, **prm):
        d = [torch.tensor(a, device="cuda") for a in (self.kappa, self.mu, self.flux[:K], self.guess[:K])]
        phi, h = torch.empty_like(d[3]), torch.empty_like(d[3])
        p = Q.qpat_default_params(**prm)
        if guess:
            Q.qpat_forward_guess_dev(self.mesh, *d, phi, h, p)
        else:
            Q.qpat_forward_dev(self.mesh, *d[:3], phi, h, p)
        return phi.cpu().numpy()

    def prior(self, **prm):
        return Q.qpat_prior_solve(self.mesh, np.log(self.kappa / 0.3), np.log(self.mu / 0.02), self.rhs, Q.qpat_default_params(**prm))


def counted(mesh, call):
    mesh.reset_stats()
    before = Q.qpat_launch_count()
    out = call()
    return out, mesh.stats(), Q.qpat_launch_count() - before


def message():
    return Q.load().qpat_last_error().decode()


@pytest.fixture(scope="module")
def device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("what", ["prior", "K4", "K16", "K4 guess", "K16 guess", "K4 mixed", "K16 mixed guess"])
def test_no_memory(device, what):
    b = Body(59 if "mixed" in what else 21)  # sizes at which the library's choice is multigrid
    K = 4 if "K4" in what else 16
    prm = dict(precision=1, fp32_operator=1) if "mixed" in what else {}
    call = (lambda **p: b.prior(**p)) if what == "prior" else (lambda **p: b.forward(K, "guess" in what, **prm, **p))
    call(pcg_variant=1)
    want, counts, launches = counted(b.mesh, lambda: call(pcg_variant=1))
    b.mesh.set_multigrid_limit(1)
    with pytest.raises(Q.QpatError):
        Q.qpat_prior_solve(b.mesh, b.kappa, b.mu, b.rhs, Q.qpat_default_params(T=-1.0))
    text = message()
    for again in range(2):
        out, c, l = counted(b.mesh, lambda: call())
        np.testing.assert_array_equal(out, want)
        assert c == counts
        assert l == launches
        assert message() == text
        assert b.mesh.multigrid_bytes() == 0
    b.mesh.close()


@pytest.mark.parametrize("guess", [False, True])
@pytest.mark.parametrize("n,K", [(13, 1), (13, 8), (21, 16)])
def test_coefficients_beyond_fp32(device, n, K, guess):
    """K's entries overflow FP32: the FP32 cycle and the FP32 solver both break down, the FP64 solver answers."""
    b = Body(n, 1e39)
    prm = dict(precision=1)
    want, counts, launches = counted(b.mesh, lambda: b.forward(K, guess, pcg_variant=1, **prm))
    assert counts["fp64_fallbacks"] >= 1
    text = message()  # the FP32 solver's own

    def named():
        with pytest.raises(Q.QpatError):
            b.forward(K, guess, multigrid=2)

    attempt = counted(b.mesh, named)[2]
    out, c, l = counted(b.mesh, lambda: b.forward(K, guess, **prm))
    np.testing.assert_array_equal(out, want)
    assert c == counts
    assert message() == text
    assert l <= launches + attempt  # one attempt, not one for every part
    b.mesh.close()
