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
