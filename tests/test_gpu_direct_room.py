"""All-pairs sums over sources packed in several segments: the records live in
whatever memory the mesh has at hand, the sums do not depend on how much."""
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


# 140 and 2,240 points (a tile, several tiles), 143,360 (many)
@pytest.mark.parametrize("s, n_c", [(0, 3), (0, 700), (2, 40), (2, 3000), (5, 500)])
def test_potential_before_and_after_a_solve(pkg, s, n_c):
    """Before a solve half the points' records fit at once, with its basis all of
    them: the same tiles, so the same bits."""
    m = synth.small_molecule(s, n_charges=n_c)
    sig = torch.from_numpy(np.random.default_rng(s).standard_normal(m.n_p)).cuda()
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, charge_mode=pkg.BEM_CHARGE_DIRECT) as g:
        rhs, (dg, phi) = g.rhs(), g.energy(sig, want_phi=True)
        g.solve()
        assert torch.equal(g.rhs(), rhs)
        dg2, phi2 = g.energy(sig, want_phi=True)
        assert torch.equal(phi2, phi) and dg2 == dg
        g.set_charges(m.charges)
        assert torch.equal(g.energy(sig, want_phi=True)[1], phi) and g.energy(sig) == pytest.approx(dg, rel=1e-5)


@pytest.mark.parametrize("galerkin", [0, 1])
def test_gradients_in_segments(pkg, galerkin):
    """A short basis leaves room for half of the points at a time (the sums of
    potential and gradient, and of dipoles in the Galerkin form): the gradients
    of a long one up to the solves' tolerance of 1e-8 times their condition."""
    m = synth.globular(5, n_charges=300)
    r = []
    for restart in (4, 30):
        with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, gmres_restart=restart, galerkin=galerkin) as g:
            r.append([v.cpu().numpy() for v in g.energy_backward()])
    close(r[0][0], r[1][0], 1e-6, what="dq")
    close(r[0][1], r[1][1], 1e-6, what="dx")


@pytest.mark.parametrize("n_c", [1, 2])
@pytest.mark.parametrize("fp64", [False, True])
def test_gradient_of_one_and_two_charges(pkg, n_c, fp64):
    """Targets that leave lanes of the packed kernel idle.  A gradient is the
    difference of two fields of the size of energy over distance to the surface,
    and can be small against them: the bound is relative to that size."""
    m = synth.small_molecule(2, n_charges=n_c)
    P = oracle.Problem(m.panels, m.charges, m.eps_in, m.eps_out)
    _, rq, rx = P.gradients()[:3]
    with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out, precision=int(fp64), depth=-1) as g:
        dq, dx = g.energy_backward()
    depth = m.radius - np.linalg.norm(m.charges[:, :3], axis=1)
    size = np.abs(rq * m.charges[:, 3]).max() / depth.min()
    assert np.abs(dx.cpu().numpy() - rx).max() < (1e-7 if fp64 else 1e-5) * size


def test_sums_without_room_for_their_parts(pkg):
    """Under a memory cap just above what the mesh holds, sums take fewer parts:
    potentials of the same bits, gradients from longer FP32 sums (2e-6 as for every
    direct sum, over products that repeat to 1e-7)."""
    m = synth.globular(6, n_charges=3000)
    r = []
    try:
        for capped in (False, True):
            with pkg.Mesh(m.panels, m.charges, m.eps_in, m.eps_out) as g:
                sig, _ = g.solve()
                if capped:
                    g.matvec_t(sig)  # the transposed product's own tables
                    pkg.bem_set_device_memory_cap(g.info()["device_bytes"] + (8 << 20))
                r.append([g.energy(g.rhs(), want_phi=True)[1], *g.energy_backward()])
                held = g.info()["device_bytes"]
            pkg.bem_set_device_memory_cap(0)
            r[-1].append(held)
    finally:
        pkg.bem_set_device_memory_cap(0)
    assert r[1][3] < r[0][3]
    assert np.abs((r[1][0] / r[0][0] - 1).cpu().numpy()).max() < 1e-12
    for a, b, what in zip(r[1][1:3], r[0][1:3], ("dq", "dx")):
        close(a.cpu().numpy(), b.cpu().numpy(), 2e-6, what=what)
