"""Translation tables built on the device, over the range of orders and both
separations: the dense real operators (m2l_mode 1) against the complex sums
over the tabulated solid harmonics (m2l_mode 2), and the highest order against
the dense FP64 oracle."""
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


@pytest.mark.parametrize("p", [1, 2, 9, 11, 16])
def test_dense_operators_match_harmonic_tables(pkg, p):
    # the same FP64 sums in another order: at most 289 terms, 1e-16 each
    m = synth.small_molecule(3)
    x = torch.from_numpy(np.random.default_rng(p).standard_normal(m.n_p)).cuda()
    y, b = [], []
    for mode in (pkg.BEM_M2L_DENSE, pkg.BEM_M2L_DIRECT):
        with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=pkg.BEM_FP64, p=p, depth=3, m2l_mode=mode,
                      charge_mode=pkg.BEM_CHARGE_FMM) as g:
            y.append(g.matvec(x).cpu().numpy())
            b.append(g.rhs().cpu().numpy())
    close(y[0], y[1], 1e-12, what="product")
    close(b[0], b[1], 1e-12, what="right-hand side")


def test_highest_order_against_oracle(pkg):
    # truncation falls by about 2 an order from 3.7e-6 at p = 10
    m = synth.small_molecule(4)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    x = P.bq()
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=pkg.BEM_FP64, p=16, depth=3) as g:
        close(g.matvec(torch.from_numpy(x).cuda()).cpu().numpy(), P.A(x), 1e-6, what="p = 16")


@pytest.mark.parametrize("p", [1, 4, 5, 6, 7, 8, 9, 10])
def test_tensor_core_m2l_orders(pkg, p):
    """Every number of K-blocks of the tensor-core M2L (32 coefficients each,
    the last one ragged) against the dense FP32 form: products kept to 2^-21
    by the split on one side and FP32 sums of up to 121 terms on both."""
    m = synth.small_molecule(4)
    x = torch.from_numpy(np.random.default_rng(p).standard_normal(m.n_p)).cuda()
    y = []
    for mode in (pkg.BEM_M2L_TC, pkg.BEM_M2L_DENSE):
        with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, p=p, depth=3, m2l_mode=mode,
                      flags=pkg.BEM_FLAG_NO_NEAR) as g:
            y.append((g.matvec(x) - x).cpu().numpy())
    close(y[0], y[1], 4e-6, what="far field")


def test_tensor_core_m2l_keeps_nan_and_infinity(pkg):
    m = synth.small_molecule(4)
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, depth=3) as g:
        for bad in (float("nan"), float("inf")):
            x = torch.ones(m.n_p, dtype=torch.float64, device="cuda")
            x[7] = bad
            # every panel lies in the near or the far field of panel 7
            assert not torch.isfinite(g.matvec(x)).any()
        assert torch.isfinite(g.matvec(torch.ones_like(x))).all()


@pytest.mark.parametrize("p", [2, 4, 6, 10])
def test_tensor_core_m2l_many_items(pkg, p):
    """Hundreds of offset classes and thousands of tiles, where the kernel's
    producers run ahead of its MMAs (by tiles and items at low orders)."""
    m = synth.globular(6)
    x = torch.from_numpy(np.random.default_rng(p).uniform(0.5, 1.5, m.n_p)).cuda()
    y = []
    for mode in (pkg.BEM_M2L_TC, pkg.BEM_M2L_DENSE):
        with pkg.Mesh(m.panels, np.zeros((0, 4)), m.eps_in, m.eps_out, p=p, leaf_size=32, m2l_mode=mode,
                      flags=pkg.BEM_FLAG_NO_NEAR) as g:
            y.append((g.matvec(x) - x).cpu().numpy())
    close(y[0], y[1], 4e-6, what="far field")


@pytest.mark.parametrize("p", [1, 2, 3, 8, 12, 16])
@pytest.mark.parametrize("galerkin", [0, 1])
def test_dipole_multipoles_at_every_order(pkg, p, galerkin):
    """<u, A x> = <A^T u, x> holds for the far fields of the product and its
    transpose only as far as both are converged, so the order is tested by the
    difference from the dense oracle falling with p: below 2^-p of the
    product's norm (measured 4e-6 at p = 10), and FP64 rounding at the top."""
    m = synth.small_molecule(3)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    x = np.random.default_rng(p).uniform(0.5, 1.5, m.n_p)
    ref = x + P.ehat * (P.kprime_t_galerkin(x) if galerkin else P.kprime_t(x))
    for prec in (pkg.BEM_FP64, pkg.BEM_MIXED):
        with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=prec, p=p, depth=2, galerkin=galerkin) as g:
            y = g.matvec_t(torch.from_numpy(x).cuda()).cpu().numpy()
        close(y, ref, max(2.0 ** -p, 3e-6) if p < 16 else 3e-6, inf=1.0 if p < 3 else None, what="K'^T")
