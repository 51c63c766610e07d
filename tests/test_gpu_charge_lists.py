"""A charge tree's M2L pairs per direction: built in one sort for small trees,
one list after the other for large ones; nothing of a tree that no pass reads."""
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


# a few pairs, charges in every cell of the volume, tens of millions of pairs
@pytest.mark.parametrize("mol", [lambda: synth.small_molecule(3, n_charges=2), lambda: synth.small_molecule(4, n_charges=4000),
                                 lambda: synth.lattice(n_side=3)])
def test_multipole_passes_match_direct_sums(pkg, mol):
    """Truncation at p = 10 with two cells' separation: 1e-5 of the vector, as for
    the products."""
    m = mol()
    sig = torch.from_numpy(np.random.default_rng(1).uniform(0.5, 1.5, m.n_p)).cuda()
    r = []
    for mode in (pkg.BEM_CHARGE_FMM, pkg.BEM_CHARGE_DIRECT):
        with pkg.Mesh(m.panels, m.charges[: max(1, len(m.charges) // 2)], m.eps_in, m.eps_out, charge_mode=mode) as g:
            g.set_charges(m.charges)
            r.append((g.rhs().cpu().numpy(), g.energy(sig, want_phi=True)[1].cpu().numpy()))
    close(r[0][0], r[1][0], 1e-5, inf=1e-3, what="B q")
    close(r[0][1], r[1][1], 1e-5, inf=1e-3, what="C s")


def test_direct_mesh_keeps_no_translation_lists(pkg):
    """With exact charge-panel pairs the direct form has a charge tree, for its
    neighbour lists alone: the mesh is smaller than one whose passes read it."""
    m = synth.globular(5)
    held = {}
    for mode in (pkg.BEM_CHARGE_FMM, pkg.BEM_CHARGE_DIRECT):
        with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, charge_mode=mode,
                      flags=pkg.BEM_FLAG_CHARGE_NEAR_EXACT) as g:
            pairs = g.info()["m2l_pairs"]
            g.rhs()
            held[mode] = g.info()["device_bytes"]
    # at least the pair of cells of every translation of the panel tree's size, beside the wider tables
    assert held[pkg.BEM_CHARGE_FMM] - held[pkg.BEM_CHARGE_DIRECT] > 8 * pairs
