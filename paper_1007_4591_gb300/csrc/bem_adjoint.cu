// Transposed operator and adjoint gradients of the solvation energy.
//
// dG(q, x) = kappa/(2 eps_in) q^T C(x) sigma,  (I + Ehat K') sigma = -Ehat B(x) q,
// kappa = 4 pi 332.0637 (the matrix form of Sec. 2.1; the mesh, hence K', does
// not depend on the charges).  With lam solving A^T lam = C^T q:
//   d dG / d q_k = kappa/(2 eps_in) [ (C sigma)_k - Ehat (B^T lam)_k ]
//   d dG / d x_k = kappa/(2 eps_in) q_k [ grad_x (C sigma)_k - Ehat sum_i lam_i grad_{x_k} B_ik ].
// B^T lam at x is the potential of dipoles lam_i n_i placed at the collocation
// points, and sum_i lam_i grad_{x_k} B_ik its gradient; C^T q is the
// potential of the charges at the quadrature points summed over each panel.
// The products between charges and surface are direct sums here; K'^T is a
// fast multipole pass (fmm_pass_t) plus the transposed near-singular table.
// In the Galerkin form K' and B are K'_G and B_G (every row averaged over its
// panel by the rule): their transposes place the dipoles lam_i w_q n_i at the
// quadrature points of panel i instead of lam_i n_i at its centroid.
#include <algorithm>

#include "bem_internal.cuh"

namespace bem {

int gmres_solve(Mesh &m, const double *b, double *x, bool transpose, bool x_zero, bem_solve_stats *st);

enum AdjSrc { AS_QUAD = 0, AS_CHARGE = 1, AS_DIPOLE = 2 };
enum AdjTgt { AT_CHG_GRAD = 0, AT_QUAD_PHI = 1 };
constexpr int ADJ_THREADS = 256;

// FP64 direct sums of G = 1/(4 pi r) and its gradient (the 1/(4 pi) is applied
// in the reduction; the FP32 form is direct_partials).  Monopole s at y:
// phi = s/r, grad = -s d/r^3 (d = x - y).  Dipole p at c: phi = p.d/r^3,
// grad = p/r^3 - 3 (p.d) d/r^5.
template <int SK, int TK>
__global__ void __launch_bounds__(ADJ_THREADS)
k_direct_adj(int64_t ntgt, int64_t nsrc, int64_t chunk, const double *tpos, const double *spos,
             const double *sw, const double *snrm, const int *qpanel, const double *dens, double ox,
             double oy, double oz, double *part) {
    __shared__ double4 sa[ADJ_THREADS], sb[ADJ_THREADS];
    const int64_t i = blockIdx.x * (int64_t)ADJ_THREADS + threadIdx.x;
    const int64_t s0 = (int64_t)blockIdx.y * chunk, s1 = min(nsrc, s0 + chunk);
    double x = 0, y = 0, z = 0;
    if (i < ntgt) {
        x = tpos[3 * i] - ox;
        y = tpos[3 * i + 1] - oy;
        z = tpos[3 * i + 2] - oz;
    }
    double o0 = 0, o1 = 0, o2 = 0, o3 = 0;
    for (int64_t b = s0; b < s1; b += ADJ_THREADS) {
        __syncthreads();
        const int64_t k = b + threadIdx.x;
        double4 a, c;
        a.x = a.y = a.z = a.w = 0;
        c.x = c.y = c.z = c.w = 0;
        if (k < s1) {
            a.x = spos[3 * k] - ox;
            a.y = spos[3 * k + 1] - oy;
            a.z = spos[3 * k + 2] - oz;
            if (SK == AS_QUAD) a.w = sw[k] * dens[qpanel[k]];
            else if (SK == AS_CHARGE) a.w = sw[k];
            else {
                const double l = dens[k];
                c.x = l * snrm[3 * k];
                c.y = l * snrm[3 * k + 1];
                c.z = l * snrm[3 * k + 2];
            }
        }
        sa[threadIdx.x] = a;
        sb[threadIdx.x] = c;
        __syncthreads();
        const int cnt = (int)min((int64_t)ADJ_THREADS, s1 - b);
        double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
        for (int j = 0; j < cnt; ++j) {
            const double4 sp = sa[j];
            const double dx = x - sp.x, dy = y - sp.y, dz = z - sp.z;
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            if (r2 == 0.0) continue;  // a dummy slot or a coincident point
            const double ri = rsqrt(r2), ri3 = ri * ri * ri;
            if (SK != AS_DIPOLE) {
                a0 = fma(sp.w, ri, a0);
                if (TK == AT_CHG_GRAD) {
                    const double f = -sp.w * ri3;
                    a1 = fma(f, dx, a1);
                    a2 = fma(f, dy, a2);
                    a3 = fma(f, dz, a3);
                }
            } else {
                const double4 pm = sb[j];
                const double pd = fma(pm.x, dx, fma(pm.y, dy, pm.z * dz));
                a0 = fma(pd, ri3, a0);
                if (TK == AT_CHG_GRAD) {
                    const double f = 3.0 * pd * ri3 * ri * ri;
                    a1 += pm.x * ri3 - f * dx;
                    a2 += pm.y * ri3 - f * dy;
                    a3 += pm.z * ri3 - f * dz;
                }
            }
        }
        o0 += a0;
        o1 += a1;
        o2 += a2;
        o3 += a3;
    }
    if (i < ntgt) {
        double *pp = part + ((size_t)blockIdx.y * ntgt + i) * (TK == AT_CHG_GRAD ? 4 : 1);
        pp[0] = o0;
        if (TK == AT_CHG_GRAD) {
            pp[1] = o1;
            pp[2] = o2;
            pp[3] = o3;
        }
    }
}

// out = (phi, grad phi) / (4 pi) [ntgt][4], or phi / (4 pi) [ntgt] for AT_QUAD_PHI
static void direct_adjoint(Mesh &m, AdjSrc sk, AdjTgt tk, const double *dens, double *out) {
    cudaStream_t s = m.stream;
    const int64_t ntgt = (tk == AT_CHG_GRAD) ? m.nc : m.nqp;
    // Galerkin: the dipoles of B_G^T sit at every quadrature point, their
    // moments lam_j w_q in m.lamq (galerkin_moments)
    const bool gq = sk == AS_DIPOLE && m.opt.galerkin;
    const int64_t nsrc = (sk == AS_QUAD) ? m.nqp : (sk == AS_CHARGE ? m.nc : (gq ? m.nqp : m.np));
    if (ntgt == 0) return;
    const int no = tk == AT_CHG_GRAD ? 4 : 1;
    if (nsrc == 0) {
        BEM_CUDA(cudaMemsetAsync(out, 0, ntgt * no * sizeof(double), s));
        return;
    }
    const bool f32 = m.opt.precision == BEM_MIXED;
    const int tblocks = cdiv(ntgt, ADJ_THREADS);
    // splits of at least 4,096 sources (FP64) or 512 (FP32: a CTA is four warps,
    // and a thousand charges give few blocks of targets)
    const int few = std::max(1, std::min(cdiv(nsrc, 4096), 1216 / tblocks));
    int nsplit = few;
    if (f32) nsplit = std::max(few, std::min({cdiv(nsrc, 512), 4 * 8 * 152 / tblocks, splits_limit(m, ntgt * no)}));
    int64_t chunk = 0;
    auto cut = [&](int n) {
        n = std::min(n, 65535);
        chunk = (nsrc + n - 1) / n;
        chunk = ((chunk + ADJ_THREADS - 1) / ADJ_THREADS) * ADJ_THREADS;
        nsplit = (int)((nsrc + chunk - 1) / chunk);
    };
    cut(nsplit);
    if (f32 && m.dpart_f.n < (size_t)nsplit * ntgt * no) {
        try {
            m.dpart_f.alloc((size_t)nsplit * ntgt * no);
        } catch (const Error &e) {  // no room for so many splits
            if (e.code != BEM_ENOMEM) throw;
            cut(few);
            m.dpart_f.alloc((size_t)nsplit * ntgt * no);
        }
    }
    DirectSum d;
    d.dipole = sk == AS_DIPOLE;
    d.skip_coincident = true;
    d.kind = tk == AT_CHG_GRAD ? DO_PHI_GRAD : DO_PHI;
    d.nsrc = nsrc;
    d.ntgt = ntgt;
    d.spos = sk == AS_CHARGE ? m.chgg64.p : (sk == AS_QUAD || gq ? m.qpg64.p : m.cen64.p);
    d.sw = sk == AS_QUAD ? m.qw64.p : (sk == AS_CHARGE ? m.q64.p : nullptr);
    d.snrm = sk == AS_DIPOLE ? (gq ? m.nrmq64.p : m.nrm64.p) : nullptr;
    d.qpanel = sk == AS_QUAD ? m.qp_panel.p : nullptr;
    d.dens = gq ? m.lamq.p : (sk == AS_CHARGE ? nullptr : dens);
    d.tpos = (tk == AT_CHG_GRAD) ? m.chgg64.p : m.qpg64.p;
    d.to_quad_values = out == quad_values(m);
    const size_t need = (size_t)nsplit * ntgt * no;
    if (f32) {
        direct_partials(m, d, chunk, nsplit, m.dpart_f.p);
        direct_reduce(m.dpart_f.p, nsplit, 1, ntgt, no, out, s);
        return;
    }
    if (m.dpart_d.n < need) m.dpart_d.alloc(need);
    const double ox = m.root_min[0] + 0.5 * m.side, oy = m.root_min[1] + 0.5 * m.side,
                 oz = m.root_min[2] + 0.5 * m.side;
    auto go = [&](auto kern) {
        kern<<<dim3(tblocks, nsplit), ADJ_THREADS, 0, s>>>(ntgt, nsrc, chunk, d.tpos, d.spos, d.sw, d.snrm, d.qpanel,
                                                           d.dens, ox, oy, oz, m.dpart_d.p);
        BEM_CHECK_LAUNCH();
    };
    if (sk == AS_QUAD && tk == AT_CHG_GRAD) go(k_direct_adj<AS_QUAD, AT_CHG_GRAD>);
    else if (sk == AS_DIPOLE && tk == AT_CHG_GRAD) go(k_direct_adj<AS_DIPOLE, AT_CHG_GRAD>);
    else if (sk == AS_CHARGE && tk == AT_QUAD_PHI) go(k_direct_adj<AS_CHARGE, AT_QUAD_PHI>);
    else throw Error(BEM_EUNSUPPORTED, "direct adjoint combination not built");
    direct_reduce(m.dpart_d.p, nsplit, 1, ntgt, no, out, s);
}

// y = A^T x = x + Ehat (K'^T x)
// four lanes per row, as k_apply_A
__global__ void k_apply_At(const double *x, const double *ktx, const int *off, const int *col,
                           const double *val, double ehat, int64_t n, double *y) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 2;
    const int sub = threadIdx.x & 3;
    double k = 0.0;
    if (i < n && off)
        for (int e = off[i] + sub; e < off[i + 1]; e += 4) k += val[e] * x[col[e]];
    k += __shfl_xor_sync(0xffffffffu, k, 1);
    k += __shfl_xor_sync(0xffffffffu, k, 2);
    if (i < n && sub == 0) y[i] = x[i] + ehat * (ktx[i] + k);
}

void matvec_t_sorted(Mesh &m, const double *xs, double *ys) {
    const bool nt = m.nt_nnz > 0 && !(m.opt.flags & (BEM_FLAG_NO_NEARTAB | BEM_FLAG_NO_NEAR));
    if (nt) transpose_near_table(m);
    fmm_pass_t(m, xs, m.zs.p);
    k_apply_At<<<cdiv(4 * m.np, 256), 256, 0, m.stream>>>(xs, m.zs.p, nt ? m.ntT_off.p : nullptr,
                                                       m.ntT_col.p, m.ntT_val.p, m.ehat, m.np, ys);
    BEM_CHECK_LAUNCH();
}

__global__ void k_gradients(const double *cs4, const double *bl4, const double *q, double ehat,
                            double pref, int64_t nc, double *dq, double *dx) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= nc) return;
    dq[k] = pref * (cs4[4 * k] - ehat * bl4[4 * k]);
    for (int c = 0; c < 3; ++c) dx[3 * k + c] = pref * q[k] * (cs4[4 * k + 1 + c] - ehat * bl4[4 * k + 1 + c]);
}

void build_qp_of_panel(Mesh &m);

AdjointVectors adjoint_vectors(Mesh &m) {
    const size_t nc = (size_t)m.nc, np = (size_t)m.np, need = 12 * nc + np;
    if (m.adj.n < need) m.adj.alloc(need);
    double *p = m.adj.p;
    return AdjointVectors{p, p + 4 * nc, p + 8 * nc, p + 9 * nc, p + 12 * nc};
}

void adjoint_gradients(Mesh &m, double grad_out, double *dq_s, double *dx_s) {
    cudaStream_t s = m.stream;
    build_qp_of_panel(m);
    const int64_t np = m.np, nc = m.nc;
    const AdjointVectors v = adjoint_vectors(m);
    double *cs4 = v.cs4, *bl4 = v.bl4, *lam = v.lam, *rhs = rhs_vector(m), *psi = quad_values(m);
    // C sigma and its gradient at the charges
    direct_adjoint(m, AS_QUAD, AT_CHG_GRAD, m.sigma_s.p, cs4);
    charge_near_phi(m, m.sigma_s.p, cs4, 4, 4);
    // C^T q: potential of the charges at the quadrature points, summed per panel
    direct_adjoint(m, AS_CHARGE, AT_QUAD_PHI, nullptr, psi);
    panel_wsum(m, psi, rhs);
    charge_near_ct(m, m.q64.p, rhs);
    // A^T lam = C^T q
    BEM_CUDA(cudaMemsetAsync(lam, 0, np * sizeof(double), s));
    bem_solve_stats st{};
    gmres_solve(m, rhs, lam, true, true, &st);
    // B^T lam and its gradient: dipoles lam_i n_i at the collocation points
    // (Galerkin: lam_i w_q n_i at the quadrature points)
    if (m.opt.galerkin) galerkin_moments(m, lam);
    direct_adjoint(m, AS_DIPOLE, AT_CHG_GRAD, lam, bl4);
    const double pref = grad_out * FOUR_PI * KCAL / (2.0 * m.eps_in);
    k_gradients<<<cdiv(nc, 256), 256, 0, s>>>(cs4, bl4, m.q64.p, m.ehat, pref, nc, dq_s, dx_s);
    BEM_CHECK_LAUNCH();
    BEM_CUDA(cudaStreamSynchronize(s));
}

}  // namespace bem
