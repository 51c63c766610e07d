"""The work that users of the solver have it do, as timed cases.

A case is one call (or one short sequence of calls) of the Python package on
a seeded synthetic molecule: a star-shaped closed surface (a geodesic sphere
of 20 f^2 triangles with smooth bumps and a random orientation) around point
charges, eps_in = 4, eps_out = 80.  The sizes are those of the repository's
benchmark and tests (Born ion 1,280 panels, globular molecule 81,920 panels
with 2,000 charges, uneven batches, rotated copies on a lattice) and odd ones
between them: the frequency f need not be a power of two.

kind      one pass
--------  ------------------------------------------------------------------
matvec    y = (I + Ehat K') x: the product inside GMRES
matvec_t  y = (I + Ehat K')^T x: the product inside the adjoint's GMRES
solve     right-hand side, GMRES to 1e-8, energy and reaction potential
bibee     the two BIBEE bounds (charge-to-surface sums, no solve)
gradient  new charges on a kept surface: energy and its gradient (autograd)
batch     many uneven molecules solved at once with their BIBEE bounds
molecule  panels and charges to energy: mesh, solve, energy, release
"""
import math

import numpy as np
import torch

import paper_1007_4591_gb300 as bem

EPS_IN, EPS_OUT = 4.0, 80.0
KCAL = 332.0637
EHAT = 2.0 * (EPS_IN - EPS_OUT) / (EPS_IN + EPS_OUT)
DIRECT_PAIRS = 4e10  # n_c n_p 7 up to which the charge sums run over all pairs
BATCH_SPREAD = (0.5, 0.6, 0.65, 0.75, 0.8, 0.9, 0.95, 1.0)  # frequencies in a batch, over the largest


def _case(name, kind, f, n_c=0, copies=1, p=10, leaf=64, fp64=False, galerkin=False, exact_near=False):
    c = {"kind": kind, "f": f, "n_c": n_c, "copies": copies, "p": p, "leaf": leaf, "fp64": fp64,
         "galerkin": galerkin, "exact_near": exact_near}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the Born ion: the smallest system anyone solves, bound by latency
        _case("born_solve", "solve", 8, n_c=1),
        # a small solute's operator product, ragged sizes, the screening order
        _case("small_matvec", "matvec", 15, p=6, leaf=32),
        # the benchmark's product: a globular protein, default options
        _case("globular_matvec", "matvec", 64),
        # the benchmark's solve with the reaction potential at every charge
        _case("globular_solve", "solve", 64, n_c=2000),
        # bounds of the solvation energy for ranking many charge sets, a finer mesh
        _case("globular_bibee", "bibee", 91, n_c=3000),
        # one step of a design or titration loop: new charges, energy, gradient
        _case("charge_gradient", "gradient", 45, n_c=1200),
        # the double-precision form, used to check the mixed one
        _case("fp64_matvec", "matvec", 40, fp64=True),
        # the Galerkin form of the product
        _case("galerkin_matvec", "matvec", 40, galerkin=True),
        # crowded solution: the product over many rotated copies
        _case("lattice_matvec", "matvec", 64, copies=27),
        # crowded solution, solved; the charge sums are multipole passes
        _case("crowded_solve", "solve", 64, n_c=2000, copies=8),
        # a screening batch of uneven molecules
        _case("batch_solve", "batch", 56, n_c=2000, copies=8),
        # a new geometry: the whole way from panels to an energy
        _case("new_molecule", "molecule", 53, n_c=1500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec"] * 4 + ["matvec_t"] * 2 + ["solve"] * 3 + ["bibee", "gradient", "batch", "molecule"])
    p, leaf = rng.choice([6, 8, 10, 10, 10, 12]), rng.choice([32, 64, 64, 64, 128])
    if kind in ("matvec", "matvec_t"):
        form = rng.choice(["mixed"] * 6 + ["fp64", "galerkin", "exact_near", "copies"])
        if form == "copies":
            return _case("", kind, _log(rng, 24, 64), copies=rng.randint(2, 20), p=p, leaf=leaf)
        return _case("", kind, _log(rng, 8, 44 if form in ("fp64", "galerkin") else 128), p=p, leaf=leaf,
                     fp64=form == "fp64", galerkin=form == "galerkin", exact_near=form == "exact_near")
    if kind == "solve" and rng.random() < 0.3:
        return _case("", kind, _log(rng, 24, 64), n_c=rng.randint(500, 2000), copies=rng.randint(2, 8), p=p, leaf=leaf)
    if kind == "batch":
        return _case("", kind, _log(rng, 32, 64), n_c=rng.randint(500, 2500), copies=rng.randint(4, 10), p=p, leaf=leaf)
    f = _log(rng, *{"solve": (8, 90), "bibee": (32, 128), "gradient": (16, 64), "molecule": (12, 64)}[kind])
    return _case("", kind, f, n_c=_log(rng, 1 if kind == "solve" else 50, 4000), p=p, leaf=leaf)


# ---------------------------------------------------------------- geometry
def _geodesic(f):
    """Unit-sphere triangles [20 f^2, 3, 3]: each face of the icosahedron cut
    into f^2 triangles, projected on the sphere, counter-clockwise outside."""
    t = (1.0 + 5.0 ** 0.5) / 2.0
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    face = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                     [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5],
                     [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]])
    i, j = np.meshgrid(np.arange(f), np.arange(f), indexing="ij")
    up = np.stack([i, j], -1)[i + j < f]      # triangles (i, j), (i+1, j), (i, j+1)
    dn = np.stack([i, j], -1)[i + j < f - 1]  # and (i+1, j), (i+1, j+1), (i, j+1)
    tri = np.concatenate([np.stack([up, up + [1, 0], up + [0, 1]], 1), np.stack([dn + [1, 0], dn + [1, 1], dn + [0, 1]], 1)])
    w = np.stack([f - tri.sum(-1), tri[..., 0], tri[..., 1]], -1) / float(f)  # barycentric
    p = np.einsum("tck,fkx->ftcx", w, v[face]).reshape(-1, 3, 3)
    return p / np.linalg.norm(p, axis=-1, keepdims=True)


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q *= np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _molecule(f, n_c, copies, rng):
    """Panels [copies 20 f^2, 3, 3] and charges [copies n_c, 4] on the GPU."""
    radius = 20.0 * (f / 64.0) ** 0.5 if f > 8 else 2.0
    u = torch.from_numpy(_geodesic(f) @ _rotation(rng)).cuda()
    if f > 8:  # bumps of at most 4 % of the radius, some panels wide
        k = torch.from_numpy(rng.standard_normal((6, 3)) * 2.5).cuda()
        ph = torch.from_numpy(rng.uniform(0, 2 * math.pi, 6)).cuda()
        u = u * (1.0 + (0.04 / 6) * torch.cos(u @ k.T + ph).sum(-1, keepdim=True))
    pan = radius * u
    if n_c == 1:
        ch = np.concatenate([0.1 * radius * rng.uniform(-1, 1, (1, 3)), [[1.0]]], 1)
    else:  # uniform in a ball 15 % inside the surface, values shifted to a net charge
        d = rng.standard_normal((max(n_c, 1), 3))
        d *= 0.85 * radius * rng.random((len(d), 1)) ** (1 / 3) / np.linalg.norm(d, axis=1, keepdims=True)
        q = rng.uniform(-0.8, 0.8, len(d))
        ch = np.concatenate([d, (q + (8.0 - q.sum()) / len(d))[:, None]], 1)[:n_c]
    ch = torch.from_numpy(ch).cuda()
    if copies == 1:
        return pan.contiguous(), ch.contiguous()
    side = math.ceil(copies ** (1 / 3))
    pans, chs = [], []
    for c in range(copies):
        rot = torch.from_numpy(_rotation(rng)).cuda()
        off = 2.5 * radius * torch.tensor([c // side ** 2, c // side % side, c % side], dtype=torch.float64, device="cuda")
        pans.append(pan @ rot + off)
        chs.append(torch.cat([ch[:, :3] @ rot + off, ch[:, 3:]], 1))
    return torch.cat(pans).contiguous(), torch.cat(chs).contiguous()


def _density(panels, rng, copies):
    """A panel vector like those GMRES meets: the normal-field-like trace of
    interior charges, one set per copy, with a little unresolved noise."""
    c = panels.mean(1)
    n = c.shape[0] // copies
    x = torch.empty(c.shape[0], dtype=torch.float64, device="cuda")
    for k in range(copies):
        ck = c[k * n:(k + 1) * n]
        mid = ck.mean(0)
        rad = (ck - mid).norm(dim=1).mean()
        d = torch.from_numpy(rng.standard_normal((32, 3))).cuda()
        at = mid + 0.8 * rad * d / d.norm(dim=1, keepdim=True)
        q = torch.from_numpy(rng.uniform(-1, 1, 32)).cuda()
        x[k * n:(k + 1) * n] = _square_distance(ck, at).reciprocal_() @ q
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    return x / x.std() + 0.05 * torch.randn(x.shape, generator=g, dtype=torch.float64, device="cuda")


def _options(case):
    o = {"p": case["p"], "leaf_size": case["leaf"]}
    if case["fp64"]:
        o["precision"] = bem.BEM_FP64
    if case["galerkin"]:
        o["galerkin"] = 1
    if case["exact_near"]:
        o["near_table"] = bem.BEM_NEAR_EXACT
    return o


def _inputs(case, seed):
    """The case's molecules and, for products, the panel vector."""
    rng = np.random.default_rng([seed, 20 * case["f"] ** 2, case["copies"]])
    if case["kind"] == "batch":
        mols = []
        for k in range(case["copies"]):
            s = BATCH_SPREAD[k % len(BATCH_SPREAD)]
            mols.append(_molecule(max(9, int(case["f"] * s)), max(50, int(case["n_c"] * s)), 1, rng))
        return mols, None
    pan, ch = _molecule(case["f"], case["n_c"], case["copies"], rng)
    x = _density(pan, rng, case["copies"]) if case["kind"].startswith("matvec") else None
    return [(pan, ch)], x


# ------------------------------------------------------------ prepare, run
def prepare(case, seed):
    mols, x = _inputs(case, seed)
    s = {"kind": case["kind"], "opt": _options(case)}
    if case["kind"] == "molecule":
        s["panels"], s["charges"] = mols[0]
        return s
    s["mesh"] = [bem.Mesh(p, c, EPS_IN, EPS_OUT, **s["opt"]) for p, c in mols]
    if case["kind"] == "gradient":
        s["charges"] = mols[0][1].requires_grad_(True)
    elif case["kind"] == "batch":
        s["sigma"] = [torch.empty(m.n_p, dtype=torch.float64, device="cuda") for m in s["mesh"]]
    s["x"] = x
    return s


def run(s):
    kind = s["kind"]
    if kind == "molecule":
        with bem.Mesh(s["panels"], s["charges"], EPS_IN, EPS_OUT, **s["opt"]) as m:
            sigma, _ = m.solve()
            dg, phi = m.energy(sigma, want_phi=True)
        return {"sigma": sigma, "dG": dg, "phi": phi}
    m = s["mesh"][0]
    if kind == "matvec":
        return m.matvec(s["x"])
    if kind == "matvec_t":
        return m.matvec_t(s["x"])
    if kind == "solve":
        sigma, _ = m.solve()
        dg, phi = m.energy(sigma, want_phi=True)
        return {"sigma": sigma, "dG": dg, "phi": phi}
    if kind == "bibee":
        cfa, sigma = m.bibee(bem.BEM_BIBEE_CFA, want_sigma=True)
        return {"sigma_cfa": sigma, "dG_cfa": cfa, "dG_p": m.bibee(bem.BEM_BIBEE_P)}
    if kind == "gradient":
        dg = bem.solvation_energy(m, s["charges"])
        return {"dG": dg.detach(), "grad": torch.autograd.grad(dg, s["charges"])[0]}
    dg, cfa, p, _ = bem.bem_batch_solve(s["mesh"], sigmas=s["sigma"])
    return {"sigma": s["sigma"], "dG": dg, "dG_cfa": cfa, "dG_p": p}


# -------------------------------------------------------------------- work
def _product_flops(n, case):
    """One product: the method's near pairs (20 flop each, 1,869 per panel at
    64 panels a leaf), translations (8,866 flop at p = 10 by rotation, 3.53
    per panel) and leaf expansions, each as on the 81,920-panel molecule."""
    outer = 7 if case["galerkin"] else 1
    pairs = outer * min(7.0 * n, 1869.0 * case["leaf"] / 64)
    trans = 3.53 * 64 / case["leaf"] * 8866 * (case["p"] / 10) ** 3
    return n * (20 * pairs + trans + (8 * 7 + 12 * outer) * (case["p"] + 1) ** 2)


def work(case):
    """Credited work of one pass.  Bytes: the surface's records (7 points, a
    centroid and a normal per panel in the working precision), the charges,
    and each vector of the call once."""
    spread = [BATCH_SPREAD[k % len(BATCH_SPREAD)] for k in range(case["copies"])] if case["kind"] == "batch" else [1.0]
    flops = nbytes = 0.0
    for s in spread:
        copies = 1 if case["kind"] == "batch" else case["copies"]
        n = 20.0 * int(case["f"] * s) ** 2 * copies
        nc = float(int(case["n_c"] * s) * copies)
        # a charge meets every quadrature point, or by multipoles about 4,000 of them
        qp = nc * min(7.0 * n, 4000.0 if nc * 7 * n > DIRECT_PAIRS else 7.0 * n)
        rec = 32 if case["fp64"] else 16
        nbytes += n * (9 * rec + 16) + nc * 40
        prod = _product_flops(n, case)
        kind = case["kind"]
        if kind.startswith("matvec"):
            flops += prod
        elif kind == "bibee":
            flops += 20 * qp / 7 + 4 * n
        elif kind == "gradient":  # two solves of 7 products, B q, C^T q, (phi, grad) of both layers
            flops += 16 * prod + 20 * qp / 7 + 10 * qp + 24 * qp + 30 * qp / 7
        else:  # 7 iterations and the final residual; B q, C sigma
            flops += 8 * prod + 20 * qp / 7 + 10 * qp
            if kind == "molecule":
                nbytes += n * 72
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- exact
def _surface(pan):
    e1, e2 = pan[:, 1] - pan[:, 0], pan[:, 2] - pan[:, 0]
    nrm = torch.linalg.cross(e1, e2)
    two = nrm.norm(dim=1, keepdim=True)
    r = 15.0 ** 0.5
    a, b = (6 - r) / 21, (6 + r) / 21  # Radon's seven-point rule of degree 5
    bary = [[1 / 3] * 3] + [[1 - 2 * t if k == j else t for k in range(3)] for t in (a, b) for j in range(3)]
    w = [9 / 40] + [(155 - r) / 1200] * 3 + [(155 + r) / 1200] * 3
    bary, w = (torch.tensor(v, dtype=torch.float64, device=pan.device) for v in (bary, w))
    area = 0.5 * two[:, 0]
    return {"pan": pan, "cen": pan.mean(1), "nrm": nrm / two, "area": area, "w": w,
            "qp": torch.einsum("qk,nkx->nqx", bary, pan), "qw": area[:, None] * w}


def _square_distance(t, y):
    r2 = (t[:, 0:1] - y[:, 0]).square_()
    for c in (1, 2):
        d = t[:, c:c + 1] - y[:, c]
        r2.addcmul_(d, d)
    return r2


def _normal_field(t, nt, y):
    """-(t - y).n / |t - y|^3 for all pairs [t, y]; coincident points give 0."""
    r = _square_distance(t, y).rsqrt_()
    r.masked_fill_(torch.isinf(r), 0.0)
    k = torch.addmm((nt * t).sum(1, keepdim=True), nt, y.T, beta=-1.0)
    return k.mul_(r.pow_(3))


def _triangle_field(t, n, v):
    """-n . int_T (t - y) / |t - y|^3 dA over the flat triangles v [m, 3, 3]:
    the solid angle along the triangle's normal, a logarithm per edge in its plane."""
    a = v - t[:, None]
    nu = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    nu = nu / nu.norm(dim=1, keepdim=True)
    ln = a.norm(dim=2)
    dot = lambda p, q: (p * q).sum(-1)  # noqa: E731
    den = ln.prod(1) + dot(a[:, 0], a[:, 1]) * ln[:, 2] + dot(a[:, 0], a[:, 2]) * ln[:, 1] + dot(a[:, 1], a[:, 2]) * ln[:, 0]
    f = nu * (-2.0 * torch.atan2(dot(a[:, 0], torch.linalg.cross(a[:, 1], a[:, 2])), den))[:, None]
    for e in range(3):
        b = (e + 1) % 3
        te = a[:, b] - a[:, e]
        te = te / te.norm(dim=1, keepdim=True)
        sa, sb = dot(a[:, e], te), dot(a[:, b], te)
        lg = torch.where(sa + sb >= 0, torch.log((ln[:, b] + sb) / (ln[:, e] + sa)), torch.log((ln[:, e] - sa) / (ln[:, b] - sb)))
        f = f + torch.linalg.cross(te, nu) * lg[:, None]
    return -dot(n, f)


def _near_pairs(g):
    """(i, j), j != i, with centroids within 2.5 sqrt(A_i)."""
    out, n = [], g["cen"].shape[0]
    for i0 in range(0, n, 4096):
        d2 = _square_distance(g["cen"][i0:i0 + 4096], g["cen"])
        ij = (d2 <= 6.25 * g["area"][i0:i0 + 4096, None]).nonzero()
        ij[:, 0] += i0
        out.append(ij[ij[:, 0] != ij[:, 1]])
    return torch.cat(out).T


def _rows(g, case):
    """4 pi K' row block by row block: yields (first row, block [rows, n])."""
    n = g["cen"].shape[0]
    outer = g["qp"] if case["galerkin"] else g["cen"][:, None]
    wo = g["w"] if case["galerkin"] else torch.ones(1, dtype=torch.float64, device="cuda")
    corr = None
    if case["galerkin"] or case["exact_near"]:  # near pairs take the exact inner integral
        i, j = _near_pairs(g)
        val = torch.zeros(len(i), dtype=torch.float64, device="cuda")
        for q in range(outer.shape[1]):
            t, nt = outer[i, q], g["nrm"][i]
            d = t[:, None] - g["qp"][j]
            rule = (-(d * nt[:, None]).sum(-1) / d.norm(dim=2).pow(3) * g["qw"][j]).sum(1)
            val += wo[q] * (_triangle_field(t, nt, g["pan"][j]) - rule)
        corr = (i, j, val)
    step = max(1, int(8e6 / n))  # blocks that stay in L2
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        own = torch.arange(i0, i1, device="cuda")
        blk = torch.zeros(i1 - i0, n, dtype=torch.float64, device="cuda")
        for q in range(outer.shape[1]):
            for e in range(7):
                blk.addcmul_(_normal_field(outer[i0:i1, q], g["nrm"][i0:i1], g["qp"][:, e]), wo[q] * g["qw"][:, e])
        blk[own - i0, own] = 0.0  # a flat panel on itself
        if corr is not None:
            sel = (corr[0] >= i0) & (corr[0] < i1)
            blk.index_put_((corr[0][sel] - i0, corr[1][sel]), corr[2][sel], accumulate=True)
        yield i0, blk


def _apply(g, case, x, transpose):
    y = x.clone()
    for i0, blk in _rows(g, case):
        c = EHAT / (4 * math.pi)
        if transpose:
            y += c * (blk.T @ x[i0:i0 + blk.shape[0]])
        else:
            y[i0:i0 + blk.shape[0]] += c * (blk @ x)
    return y


def _matrix(g, case):
    n = g["cen"].shape[0]
    a = torch.empty(n, n, dtype=torch.float64, device="cuda")
    for i0, blk in _rows(g, case):
        a[i0:i0 + blk.shape[0]] = blk.mul_(EHAT / (4 * math.pi))
    a.diagonal().add_(1.0)
    return a


def _gmres(mul, b, tol=1e-13, most=80):
    beta = b.norm()
    v, h = [b / beta], np.zeros((most + 1, most))
    for j in range(most):
        w = mul(v[j])
        for i, vi in enumerate(v):
            h[i, j] = float(vi @ w)
            w = w - h[i, j] * vi
        h[j + 1, j] = float(w.norm())
        e = np.zeros(j + 2)
        e[0] = float(beta)
        z, *_ = np.linalg.lstsq(h[:j + 2, :j + 1], e, rcond=None)
        if np.linalg.norm(h[:j + 2, :j + 1] @ z - e) <= tol * e[0]:
            break
        v.append(w / h[j + 1, j])
    return sum(float(zk) * vk for zk, vk in zip(z, v))


def _charge_blocks(x, y):
    for k0 in range(0, x.shape[0], max(1, int(2e7 / y.shape[0]))):
        yield slice(k0, k0 + max(1, int(2e7 / y.shape[0])))


def _bq(g, ch):
    out = torch.empty_like(g["area"])
    for s in _charge_blocks(g["cen"], ch):
        out[s] = _normal_field(g["cen"][s], g["nrm"][s], ch[:, :3]) @ ch[:, 3]
    return out / (4 * math.pi)


def _c_sigma(g, ch, sigma, grad=False):
    """C sigma at the charges, and its gradient."""
    y, s = g["qp"].reshape(-1, 3), (g["qw"] * sigma[:, None]).reshape(-1)
    phi, gr = torch.empty_like(ch[:, 0]), torch.empty_like(ch[:, :3])
    for b in _charge_blocks(ch, y):
        x = ch[b, :3]
        r = _square_distance(x, y).rsqrt_()
        phi[b] = r @ s
        if grad:
            r = r * r * r
            gr[b] = r @ (s[:, None] * y) - x * (r @ s)[:, None]
    return phi / (4 * math.pi), gr / (4 * math.pi)


def _dipole(g, ch, lam):
    """B^T lam at the charges (dipoles lam_i n_i at the centroids), and its gradient."""
    c, p = g["cen"], lam[:, None] * g["nrm"]
    phi, gr = torch.empty_like(ch[:, 0]), torch.empty_like(ch[:, :3])
    for b in _charge_blocks(ch, c):
        x = ch[b, :3]
        r = _square_distance(x, c).rsqrt_()
        pd = (x @ p.T - (p * c).sum(1)) * r ** 3
        phi[b] = pd.sum(1)
        t = 3 * pd * r * r
        gr[b] = r ** 3 @ p - (x * t.sum(1, keepdim=True) - t @ c)
    return phi / (4 * math.pi), gr / (4 * math.pi)


def _energy(ch, phi):
    return 4 * math.pi * KCAL / (2 * EPS_IN) * float(ch[:, 3] @ phi)


def exact(case, seed):
    mols, x = _inputs(case, seed)
    kind, n = case["kind"], max(p.shape[0] for p, _ in mols)
    pairs = sum(7.0 * p.shape[0] ** 2 for p, _ in mols) * (7 if case["galerkin"] else 1)
    if kind != "bibee" and (pairs > 1.2e11 or (not kind.startswith("matvec") and n > 90000)):
        return None  # over about 20 seconds, or a matrix larger than the card
    gs = [_surface(p) for p, _ in mols]
    if kind.startswith("matvec"):
        return _apply(gs[0], case, x, kind == "matvec_t")
    out = []
    for g, (_, ch) in zip(gs, mols):
        bq = _bq(g, ch)
        dg = [_energy(ch, _c_sigma(g, ch, -EHAT / (1 + EHAT * lam) * bq)[0]) for lam in (-0.5, 0.0)]
        if kind == "bibee":
            return {"sigma_cfa": -EHAT / (1 - 0.5 * EHAT) * bq, "dG_cfa": dg[0], "dG_p": dg[1]}
        a = _matrix(g, case)
        sigma = _gmres(lambda v: a @ v, -EHAT * bq)
        phi, dphi = _c_sigma(g, ch, sigma, grad=kind == "gradient")
        if kind == "gradient":
            ctq = torch.empty_like(g["qw"]).reshape(-1)
            y = g["qp"].reshape(-1, 3)
            for s in _charge_blocks(y, ch):
                ctq[s] = _square_distance(y[s], ch[:, :3]).rsqrt_() @ ch[:, 3]
            ctq = (ctq.view(-1, 7) * g["qw"]).sum(1) / (4 * math.pi)
            lam = _gmres(lambda v: a.T @ v, ctq)
            bl, dbl = _dipole(g, ch, lam)
            f = 4 * math.pi * KCAL / (2 * EPS_IN)
            dx = f * ch[:, 3:] * (dphi - EHAT * dbl)
            return {"dG": torch.tensor(_energy(ch, phi), dtype=torch.float64),
                    "grad": torch.cat([dx, f * (phi - EHAT * bl)[:, None]], 1)}
        out.append((sigma, _energy(ch, phi), phi / EPS_IN, *dg))
        del a
    if kind == "batch":
        return {"sigma": [o[0] for o in out], "dG": np.array([o[1] for o in out]), "dG_cfa": np.array([o[3] for o in out]),
                "dG_p": np.array([o[4] for o in out])}
    return {"sigma": out[0][0], "dG": out[0][1], "phi": out[0][2]}
