"""Every M2L form in both directions against the default one: the same
translations in another order of operations (FP64 1e-16 a term, mixed 2^-21)."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("galerkin", [0, 1])
@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("p", [3, 10, 12, 15, 16])
def test_m2l_forms(pkg, p, fp64, galerkin):
    m = synth.small_molecule(4)
    x = torch.from_numpy(np.random.default_rng(p).uniform(0.5, 1.5, m.n_p)).cuda()
    r = []
    for mode, graph in ((pkg.BEM_M2L_AUTO, 0), (pkg.BEM_M2L_DENSE, 0), (pkg.BEM_M2L_DIRECT, 0), (pkg.BEM_M2L_AUTO, 1)):
        with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=fp64, p=p, depth=3, m2l_mode=mode, graph=graph,
                      galerkin=galerkin) as g:
            r.append([f(x).cpu().numpy() for f in (g.matvec, g.matvec, g.matvec_t)])
    tol = 1e-12 if fp64 else 4e-6
    for y in r:
        for a, b in zip(y, r[0]):
            close(a, b, tol)
