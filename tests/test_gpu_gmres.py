"""GMRES's vector kernels at their edges: numbers of basis vectors around the
blocks of eight they are compiled for, vectors shorter than a CTA, and vectors
long enough for the larger grid."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import close

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1007_4591_gb300 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("s", [0, 2])  # 20 and 320 panels
@pytest.mark.parametrize("restart", [1, 2, 3, 4, 5, 6, 7, 8, 9, 16, 17, 26, 40])
def test_restart_lengths(pkg, s, restart):
    """40 iterations to the rounding of FP64, whatever the basis's length: one
    leaf holds every panel, so the product is the dense one (error 1e-15) and
    sigma's error the residual's times the condition number, below 100."""
    m = synth.small_molecule(s, n_charges=12)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    ref, _ = P.solve(tol=1e-14)
    most = 40 if restart > 3 else 400
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=pkg.BEM_FP64, depth=-1, gmres_restart=restart,
                  max_iter=most, tol=1e-13) as g:
        sig, st = g.solve(allow_noconv=True)
        assert st["true_resid"] < 1e-12
        close(sig.cpu().numpy(), ref, 1e-10, what="sigma")


def test_long_basis(pkg):
    """A basis as long as the system allows (it breaks down when the residual
    reaches rounding, past two blocks of vectors): the solution stays."""
    m = synth.small_molecule(2, n_charges=12)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    ref, _ = P.solve(tol=1e-14)
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=pkg.BEM_FP64, depth=-1, gmres_restart=40,
                  max_iter=40, tol=1e-40) as g:
        sig, st = g.solve(allow_noconv=True)
        assert st["iterations"] > 16 and st["true_resid"] < 1e-12
        close(sig.cpu().numpy(), ref, 1e-10, what="sigma")


def test_large_system(pkg):
    """2.2 million rows (the larger grid, a last stride that is not whole): the
    residual that the rotations carry is that of the solution, to the rounding
    of FP64 products and sums (1e-15 of the right-hand side a step)."""
    m = synth.lattice(n_side=3)
    with pkg.Mesh(m.panels, np.zeros((0, 4)), m.eps_in, m.eps_out, precision=pkg.BEM_FP64, p=4) as g:
        g.set_charges(m.charges[::400])
        _, st = g.solve()
        assert st["converged"] and st["iterations"] > 6
        assert abs(st["true_resid"] - st["resid"]) < 1e-12
