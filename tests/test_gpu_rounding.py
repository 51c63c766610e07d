"""The far field's rounding, and how far an energy moves from call to call.

Expansions of cells with several children or M2L partners are sums in order of
arrival, so a product in mixed precision repeats itself only to a few 1e-8 and
an energy to a few 1e-9.  Where every expansion is a single translation the
product is the same bits in every run: those are held to values recorded with
multipoles and operators split by cvt.rna.tf32.f32 ahead of the M2L kernel."""
import json
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "mixed_rounding.json")
DIAGONALS = [(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
ORDERS = [4, 10]
MOLECULES = {"small-s4": lambda: synth.small_molecule(4), "globular-s5": lambda: synth.globular(5, n_charges=500)}


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1007_4591_gb300 as pkg
    pkg.load_library()
    return pkg


@pytest.fixture(scope="module")
def golden():
    with open(GOLDEN) as f:
        return json.load(f)


def two_clusters(diagonal, n=24):
    """Small triangles in two opposite corner cells of a tree of depth 3: every
    cell has one child and one M2L partner."""
    rng = np.random.default_rng([7, *(d + 1 for d in diagonal)])
    pan = []
    for side in (-20.0, 20.0):
        c = side * np.asarray(diagonal, dtype=np.float64) + rng.uniform(-1.0, 1.0, (n, 3))
        e = 0.4 * rng.standard_normal((n, 2, 3))
        pan.append(np.stack([c, c + e[:, 0], c + e[:, 1]], 1))
    return np.concatenate(pan), rng.uniform(0.5, 1.5, 2 * n)


def far_field(pkg, p, diagonal):
    pan, x = two_clusters(diagonal)
    with pkg.Mesh(pan, np.zeros((0, 4)), 4.0, 80.0, p=p, depth=3, near_table=0, flags=pkg.BEM_FLAG_NO_NEAR) as g:
        assert g.info()["m2l_pairs"] == 2
        return g.matvec(torch.from_numpy(x).cuda()).cpu().numpy() - x


@pytest.mark.parametrize("diagonal", DIAGONALS)
@pytest.mark.parametrize("p", ORDERS)
def test_single_translations_keep_their_bits(pkg, golden, p, diagonal):
    ref = [float.fromhex(v) for v in golden["far field"]["%d %s" % (p, list(diagonal))]]
    assert far_field(pkg, p, diagonal).tolist() == ref


POTENTIALS = {"small-s4, 60 charges": lambda: synth.small_molecule(4, n_charges=60),
              "globular-s6, 700 charges": lambda: synth.globular(6, n_charges=700)}


def potential(pkg, name):
    """C s at the charges for a fixed density: the right-hand side's, which no
    multipole pass has touched."""
    m = POTENTIALS[name]()
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, charge_mode=pkg.BEM_CHARGE_DIRECT) as g:
        return g.energy(g.rhs(), want_phi=True)[1].cpu().numpy()[::20]


@pytest.mark.parametrize("name", sorted(POTENTIALS))
def test_direct_sums_keep_their_bits(pkg, golden, name):
    """All-pairs sums have no order of arrival: normal field and potential, tile
    by tile in splits of the same length.  The last FP64 sum over the splits may
    be shared out differently (2^-52 a term, at most some thousands)."""
    ref = np.array([float.fromhex(v) for v in golden["potential"][name]])
    assert np.abs(potential(pkg, name) / ref - 1).max() < 1e-12


@pytest.mark.parametrize("name", sorted(MOLECULES))
def test_energy_from_call_to_call(pkg, golden, name):
    """200 calls before the multipoles were split inside the M2L kernel: mean as
    recorded, standard deviation 2.0-2.6e-9 of it.  Other timings change the
    order of arrival and with it the mean by about one deviation; a deviation of
    20 calls is itself known to a sixth.  So 3 deviations for the mean (with
    2.5e-9 / sqrt(20) of its own) and 2 for the spread."""
    m = MOLECULES[name]()
    ch = torch.from_numpy(m.charges).cuda().requires_grad_(True)
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out) as g:
        v = np.array([float(pkg.solvation_energy(g, ch).detach()) for _ in range(20)])
    mean = golden["energy"][name]
    assert abs(v.mean() / mean - 1) < 7.5e-9
    assert v.std() / abs(mean) < 5e-9
