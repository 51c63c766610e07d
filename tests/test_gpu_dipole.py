"""Dipole multipoles against truncated series of the kernel itself.

On a tree of depth 2 every pair of leaves that do not touch interacts by one
M2L, so the far field of the transposed product (one-point rule) is, for a
dipole at a from its leaf's centre and a point at b from its own, the part of
n . grad_a 1 / |D + b - a| of degree at most p in b and (before the gradient) in
a.  That part comes from the Taylor series of (|D + t b - s a|^2)^(-3/2) in s and
t, without any harmonics.  Every degree counts: the leaves are full and some two
cells apart, where the series falls by a factor of two a degree.
"""
import numpy as np
import pytest

from gpu_util import close

LEAVES = {(0, 0, 0): 131, (2, 0, 1): 33, (0, 2, 2): 32, (3, 3, 3): 5, (3, 1, 0): 1}


def scene():
    """Tiny triangles in a few leaves of a cube of four cells a side."""
    rng = np.random.default_rng(9)
    c = np.concatenate([np.asarray(k) + rng.uniform(0.04, 0.96, (n, 3)) for k, n in LEAVES.items()])
    c[0], c[-2] = 0.0, 4.0  # the corners of the root cube
    e = 0.01 * rng.standard_normal((len(c), 2, 3))
    pan = np.stack([c, c + e[:, 0], c + e[:, 1]], 1)
    return pan, rng.uniform(0.5, 1.5, len(c))


def far_field(pan, lam, p, eps_in=4.0, eps_out=80.0):
    cen, n = pan.mean(1), np.cross(pan[:, 1] - pan[:, 0], pan[:, 2] - pan[:, 0])
    two = np.linalg.norm(n, axis=1)
    n, area = n / two[:, None], 0.5 * two
    lo, hi = pan.reshape(-1, 3).min(0), pan.reshape(-1, 3).max(0)
    side = (hi - lo).max() * (1 + 1e-6) + 1e-12
    root, h = 0.5 * (lo + hi) - 0.5 * side, side / 4
    cell = np.floor((cen - root) / h).astype(int)
    mid = root + (cell + 0.5) * h
    j, i = np.nonzero(np.abs(cell[:, None] - cell[None]).max(2) >= 2)  # target, source
    dot = lambda u, v: (u * v).sum(1)  # noqa: E731
    d, a, b, ni = mid[j] - mid[i], cen[i] - mid[i], cen[j] - mid[j], n[i]
    zero = np.zeros((p + 1, len(i)))

    def mul(u, v):  # polynomials in t of degree <= p
        w = zero.copy()
        for k in range(p + 1):
            w[k:] += u[k] * v[: p + 1 - k]
        return w

    def poly(*coef):
        w = zero.copy()
        for k, x in enumerate(coef[: p + 1]):
            w[k] = x
        return w

    q = [poly(dot(d, d), 2 * dot(d, b), dot(b, b)), poly(-2 * dot(d, a), -2 * dot(a, b)), poly(dot(a, a))]
    power = -1.5
    f0, inv = zero.copy(), zero.copy()  # q0^power and 1 / q0
    f0[0], inv[0] = q[0][0] ** power, 1 / q[0][0]
    for m in range(1, p + 1):
        for k in range(1, min(m, 2) + 1):
            f0[m] += (k * (power + 1) - m) * q[0][k] * f0[m - k] / (m * q[0][0])
            inv[m] -= q[0][k] * inv[m - k] / q[0][0]
    f = [f0]
    for m in range(1, p + 1):
        s = sum((k * (power + 1) - m) * mul(q[k], f[m - k]) for k in range(1, min(m, 2) + 1))
        f.append(mul(s, inv) / m)
    dq = [None, poly(-2 * dot(d, ni), -2 * dot(ni, b)), poly(2 * dot(a, ni))]  # d q / d a along n
    g = sum(-0.5 * mul(dq[k], f[m - k]) for m in range(1, p + 1) for k in range(1, min(m, 2) + 1)).sum(0)
    out = np.zeros(len(cen))
    np.add.at(out, j, lam[i] * g)
    return 2 * (eps_in - eps_out) / (eps_in + eps_out) / (4 * np.pi) * area * out


def test_series_converges_to_the_kernel():
    pan, lam = scene()
    exact = None
    err = []
    for p in (6, 12, 24):
        y = far_field(pan, lam, p)
        if exact is None:
            cen, n = pan.mean(1), np.cross(pan[:, 1] - pan[:, 0], pan[:, 2] - pan[:, 0])
            two = np.linalg.norm(n, axis=1)
            lo, hi = pan.reshape(-1, 3).min(0), pan.reshape(-1, 3).max(0)
            side = (hi - lo).max() * (1 + 1e-6) + 1e-12
            cell = np.floor((cen - 0.5 * (lo + hi) + 0.5 * side) / (side / 4)).astype(int)
            r = cen[:, None] - cen[None]
            k = ((r * (n / two[:, None])[None]).sum(2)) / np.maximum(np.linalg.norm(r, axis=2), 1e-9) ** 3
            k[np.abs(cell[:, None] - cell[None]).max(2) < 2] = 0
            exact = 2 * (4.0 - 80.0) / 84.0 / (4 * np.pi) * 0.5 * two * (k @ lam)
        err.append(np.linalg.norm(y - exact) / np.linalg.norm(exact))
    assert err[0] < 3e-2 and err[1] < err[0] / 10 and err[2] < err[1] / 50


@pytest.mark.gpu
@pytest.mark.parametrize("p", range(1, 17))
def test_dipole_multipoles(p):
    """FP64 sums of some 200 terms of 289 products; mixed precision 2^-21 of the
    harmonics' products, as for the M2L forms.  (Without degree p the far field is
    off by 2e-6 at p = 16, 1e-4 at p = 10.)"""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1007_4591_gb300 as pkg
    pkg.load_library()
    pan, lam = scene()
    ref = far_field(pan, lam, p)
    for prec, tol in ((pkg.BEM_FP64, 1e-11), (pkg.BEM_MIXED, 4e-6)):
        with pkg.Mesh(pan, np.zeros((0, 4)), 4.0, 80.0, precision=prec, p=p, depth=2, near_table=0, quad_points=1,
                      flags=pkg.BEM_FLAG_NO_NEAR) as g:
            y = g.matvec_t(torch.from_numpy(lam).cuda()).cpu().numpy() - lam
        close(y, ref, tol, what="far field")
