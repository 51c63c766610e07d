"""All-pairs sums between charges and surface at the edges of their tiles:
B q at the collocation points, C s at the charges, and (C s, its gradient,
B^T lam) through the adjoint, against the dense FP64 oracle.

Tolerance: FP32 pair terms with split coordinates carry about 4e-7 each
(rsqrt cubed, three products) and tile sums of 256 terms in FP32 add a few
2^-24 of the partial sums, so 2e-6 of the vector's norm bounds every sum here.
"""
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


def _mol(s, n_c):
    return synth.small_molecule(s, n_charges=n_c) if s < 6 else synth.globular(s, n_charges=n_c)


# around one tile and one block of targets (256), two splits, five tiles
@pytest.mark.parametrize("n_c", [1, 2, 255, 256, 257, 513, 1025])
@pytest.mark.parametrize("fp64", [False, True])
def test_direct_sums_match_oracle(pkg, n_c, fp64):
    m = _mol(2, n_c)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    tol = 1e-12 if fp64 else 2e-6
    sig = np.random.default_rng(n_c).standard_normal(m.n_p)
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=int(fp64), depth=-1,
                  charge_mode=pkg.BEM_CHARGE_DIRECT) as g:
        close(g.rhs().cpu().numpy(), -P.ehat * P.bq(), tol, what="B q")
        dg, phi = g.energy(torch.from_numpy(sig).cuda(), want_phi=True)
        ref = P.c(sig)
        close(phi.cpu().numpy(), ref / m.eps_in, tol, what="C s")
        # C^T q . s, built from the potential at the quadrature points
        e = 4 * np.pi * 332.0637 / (2 * m.eps_in) * float(m.charges[:, 3] @ ref)
        scale = 4 * np.pi * 332.0637 / (2 * m.eps_in) * float(np.abs(m.charges[:, 3]) @ np.abs(ref))
        assert abs(g.energy(torch.from_numpy(sig).cuda()) - e) < 4 * tol * scale
        dq, dx = g.energy_backward()
    _, rq, rx = P.gradients()[:3]
    gtol = 1e-7 if fp64 else 1e-5  # the solves in between run to 1e-8
    close(dq.cpu().numpy(), rq, gtol, what="dq")
    if n_c > 2:
        close(dx.cpu().numpy(), rx, gtol, what="dx")


def test_sources_in_several_segments(pkg):
    """2,293,760 points (three segments of source records) at 600 charges: the
    splits do not end where the segments do."""
    m = _mol(7, 600)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    sig = P.bq()
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out) as g:
        _, phi = g.energy(torch.from_numpy(sig).cuda(), want_phi=True)
        close(phi.cpu().numpy(), P.c(sig) / m.eps_in, 2e-6, what="C s")


@pytest.mark.parametrize("fp64", [False, True])
def test_charge_sets_replaced_without_a_charge_tree(pkg, fp64):
    """Direct charge sums keep no charge tree: sets of other sizes (none, more,
    fewer) give what a mesh made with them gives."""
    m = _mol(2, 40)
    tol = 1e-12 if fp64 else 2e-6
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=int(fp64), depth=2) as g:
        sig = torch.from_numpy(np.random.default_rng(3).standard_normal(m.n_p)).cuda()
        g.set_charges(np.zeros((0, 4)))
        assert float(g.rhs().abs().max()) == 0.0 and g.energy(sig) == 0.0
        for n_c in (600, 3):
            w = _mol(2, n_c)
            P = oracle.Problem(w.panels, w.charges, w.eps_in, w.eps_out)
            g.set_charges(w.charges)
            close(g.rhs().cpu().numpy(), -P.ehat * P.bq(), tol, what="B q")
            close(g.energy(sig, want_phi=True)[1].cpu().numpy(), P.c(sig.cpu().numpy()) / w.eps_in, tol, what="C s")
            dq, dx = g.energy_backward()
            _, rq, rx = P.gradients()[:3]
            close(dq.cpu().numpy(), rq, 1e-5, what="dq")  # p = 10 products
            close(dx.cpu().numpy(), rx, 1e-5, what="dx")
