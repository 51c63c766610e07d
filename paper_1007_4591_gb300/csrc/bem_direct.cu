// Direct (all-pairs) products between the point charges and the surface:
// (B q)_i at the collocation points and (C s)_k at the charges.
//
// For the sizes where n_c * n_p * quad_points is modest (every molecule in
// the single-molecule and batched workloads) the direct sum is both cheaper
// and exact to rounding, while the fast multipole pass over a
// one-cell-separated octree has a worst case (a charge at a cell corner)
// whose truncation error converges only like (sqrt(3)/2)^p.  Large systems
// (many molecules) use the fast multipole pass; opt.charge_mode selects.
//
// Coordinates are taken relative to the root-cube centre; in FP32 each one is
// carried as a pair hi + lo (hi = the FP32 rounding, lo = the FP32 rounding of
// the rest) and a difference is formed as (hi_t - hi_s) + (lo_t - lo_s): the
// first term is exact for nearby points, so a pair's difference keeps about
// 2^-24 of its own length instead of 2^-24 of the distance from the centre
// (charges a few hundredths of an A from a quadrature or collocation point).
// Each thread sums one tile in a short accumulator and adds the tile total
// to a second one, and the partial sums of the source splits are reduced in
// FP64.  FP32 sums (two targets to a packed operand) and FP64 sums are separate
// kernels.
#include <type_traits>

#include "bem_device.cuh"

namespace bem {

void axpby(Mesh &m, double a, const double *x, double b, const double *y, double *out, int64_t n);

constexpr int DIRECT_THREADS = 256;  // FP64 kernel
constexpr int DIRECT_TILE = 256;     // sources per tile of either kernel

template <int SRC, int TGT>
__global__ void __launch_bounds__(DIRECT_THREADS)
k_direct(int64_t ntgt, int64_t nsrc, int64_t chunk, const double *tpos, const double *tnrm,
         const double *spos, const double *sw, const int *qpanel, const double *dens, double ox,
         double oy, double oz, double *part) {
    __shared__ double4 sh[DIRECT_TILE];
    const int64_t i = blockIdx.x * (int64_t)DIRECT_THREADS + threadIdx.x;
    const int64_t sb = (int64_t)blockIdx.y * chunk;
    const int64_t se = min(nsrc, sb + chunk);
    constexpr bool DN = TGT == TGT_CEN_DN || TGT == TGT_QUAD_DN;  // normal field, else potential
    double cx = 0, cy = 0, cz = 0, nx = 0, ny = 0, nz = 0;
    if (i < ntgt) {
        cx = tpos[3 * i] - ox;
        cy = tpos[3 * i + 1] - oy;
        cz = tpos[3 * i + 2] - oz;
        if (DN) {
            nx = tnrm[3 * i];
            ny = tnrm[3 * i + 1];
            nz = tnrm[3 * i + 2];
        }
    }
    double outer = 0;
    for (int64_t b = sb; b < se; b += DIRECT_TILE) {
        __syncthreads();
        const int64_t k = b + threadIdx.x;
        double4 r;
        r.x = r.y = r.z = r.w = 0;
        if (k < se) {
            r.x = spos[3 * k] - ox;
            r.y = spos[3 * k + 1] - oy;
            r.z = spos[3 * k + 2] - oz;
            if (SRC == SRC_QUAD) r.w = sw[k] * dens[qpanel[k]];
            else r.w = dens ? dens[k] : sw[k];
        }
        sh[threadIdx.x] = r;
        __syncthreads();
        const int cnt = (int)min((int64_t)DIRECT_TILE, se - b);
        double acc = 0;
#pragma unroll 4
        for (int j = 0; j < cnt; ++j) {
            const double4 y = sh[j];
            const double dx = cx - y.x, dy = cy - y.y, dz = cz - y.z;
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            const double ri = rsqrt(r2);
            if (DN) {
                const double nd = fma(nx, dx, fma(ny, dy, nz * dz));
                acc = fma(y.w * nd, ri * ri * ri, acc);
            } else {
                acc = fma(y.w, ri, acc);
            }
        }
        outer += acc;
    }
    if (i < ntgt) part[(size_t)blockIdx.y * ntgt + i] = DN ? -outer : outer;
}

// Source records of the FP32 kernel: (-x, -y, -z, w), (-lx, -ly, -lz, px) and,
// for dipoles, (py, pz, 0, 0), with hi + lo = the position about the root
// cube's centre, w the strength, p a dipole moment.
constexpr int DREC_MONO = 2, DREC_DIPOLE = 3;

template <bool DIPOLE>
__global__ void k_direct_pack(int64_t n, const double *spos, const double *sw, const double *snrm, const int *qpanel,
                              const double *dens, double ox, double oy, double oz, float4 *rec) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double p[3] = {spos[3 * k] - ox, spos[3 * k + 1] - oy, spos[3 * k + 2] - oz};
    float h[3], l[3], v[4] = {0.f, 0.f, 0.f, 0.f};  // v: w, px, py, pz
    for (int c = 0; c < 3; ++c) {
        h[c] = (float)p[c];
        l[c] = (float)(p[c] - (double)h[c]);
    }
    if (DIPOLE) {
        const double d = dens[k];
        for (int c = 0; c < 3; ++c) v[1 + c] = (float)(d * snrm[3 * k + c]);
    } else {
        v[0] = (float)(qpanel ? sw[k] * dens[qpanel[k]] : (dens ? dens[k] : sw[k]));
    }
    float4 *r = rec + (DIPOLE ? DREC_DIPOLE : DREC_MONO) * k;
    r[0] = make_float4(-h[0], -h[1], -h[2], v[0]);
    r[1] = make_float4(-l[0], -l[1], -l[2], v[1]);
    if (DIPOLE) r[2] = make_float4(v[2], v[3], 0.f, 0.f);
}

// FP32 pairs, bound by the FMA pipe (19 operations a pair for the normal
// field, 13 for the potential, 9 of them the split difference): a thread holds
// two targets in packed operands, so an FP32x2 instruction does two pairs
// while every target's sum keeps the order of a scalar loop; the records come
// ready from k_direct_pack, two tiles in flight by cp.async.  Measured in
// pairs/clk/SM over 4 waves of CTAs: 7.5 for the potential (bound 9.8; four
// targets a thread 7.5, records with every value twice in shared memory 6.0:
// an LDS.128 takes four cycles even as a broadcast) and 5.2 for the normal
// field (bound 6.7; four targets 4.7: 98 registers).  One target a thread with
// the records formed from FP64 in every CTA ran at 5.0 and 4.4.
constexpr int DPK_THREADS = 128;
constexpr int DPK_NPK = 1;                               // packed operands (target pairs) per thread
constexpr int DPK_TARGETS = 2 * DPK_NPK * DPK_THREADS;   // targets per CTA
__device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }

template <bool DIPOLE, int KIND, bool SKIP0>
__global__ void __launch_bounds__(DPK_THREADS)
k_direct_pk(int64_t ntgt, int64_t nsrc, int64_t chunk, int64_t seg0, int64_t seg1, int split0, const double *tpos,
            const double *tnrm, const float4 *__restrict__ rec, double ox, double oy, double oz, float *part) {
    constexpr int RS = DIPOLE ? DREC_DIPOLE : DREC_MONO, NPK = DPK_NPK;
    constexpr int NO = KIND == DO_PHI_GRAD ? 4 : 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    float4 *sh = reinterpret_cast<float4 *>(smraw);  // [2][DIRECT_TILE][RS]
    const int split = split0 + blockIdx.y;
    const int64_t c0 = (int64_t)split * chunk;
    const int64_t sb = max(seg0, c0), se = min(min(nsrc, seg1), c0 + chunk);
    const float4 *src = rec + RS * (sb - seg0);
    auto tgt = [&](int u, int e) { return ((int64_t)blockIdx.x * NPK + u) * (2 * DPK_THREADS) + 2 * threadIdx.x + e; };
    auto copy = [&](int64_t t, int bf) {  // tile t of [sb, se)
        const int64_t b = t * DIRECT_TILE;
        const int n = (int)min((int64_t)DIRECT_TILE, se - sb - b) * RS;
        for (int e = threadIdx.x; e < n; e += DPK_THREADS)
            cp_async_16(sh + bf * DIRECT_TILE * RS + e, src + b * RS + e, true);
        cp_async_commit();
    };
    copy(0, 0);
    float2 cx[NPK], cy[NPK], cz[NPK], lx[NPK], ly[NPK], lz[NPK], nx[NPK], ny[NPK], nz[NPK], outer[NPK][NO];
    float *const pp = part + (size_t)split * ntgt * NO;
#pragma unroll
    for (int u = 0; u < NPK; ++u) {
        float h[2][3], l[2][3], n[2][3], o[2][NO];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int64_t i = tgt(u, e);
#pragma unroll
            for (int c = 0; c < 3; ++c) h[e][c] = l[e][c] = n[e][c] = 0.f;
#pragma unroll
            for (int c = 0; c < NO; ++c) o[e][c] = 0.f;
            if (i < ntgt) {
                const double p[3] = {tpos[3 * i] - ox, tpos[3 * i + 1] - oy, tpos[3 * i + 2] - oz};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    h[e][c] = (float)p[c];
                    l[e][c] = (float)(p[c] - (double)h[e][c]);
                    if (KIND == DO_DN) n[e][c] = (float)tnrm[3 * i + c];
                }
                if (sb > c0)  // the chunk began in an earlier segment
#pragma unroll
                    for (int c = 0; c < NO; ++c) o[e][c] = KIND == DO_DN ? -pp[i * NO + c] : pp[i * NO + c];
            }
        }
        cx[u] = make_float2(h[0][0], h[1][0]);
        cy[u] = make_float2(h[0][1], h[1][1]);
        cz[u] = make_float2(h[0][2], h[1][2]);
        lx[u] = make_float2(l[0][0], l[1][0]);
        ly[u] = make_float2(l[0][1], l[1][1]);
        lz[u] = make_float2(l[0][2], l[1][2]);
        nx[u] = make_float2(n[0][0], n[1][0]);
        ny[u] = make_float2(n[0][1], n[1][1]);
        nz[u] = make_float2(n[0][2], n[1][2]);
#pragma unroll
        for (int c = 0; c < NO; ++c) outer[u][c] = make_float2(o[0][c], o[1][c]);
    }
    const int64_t ntile = (se - sb + DIRECT_TILE - 1) / DIRECT_TILE;
    for (int64_t t = 0; t < ntile; ++t) {
        const int bf = (int)(t & 1);
        cp_async_wait<0>();
        __syncthreads();  // tile t is in place; the other buffer's readers are done
        if (t + 1 < ntile) copy(t + 1, bf ^ 1);
        const int cnt = (int)min((int64_t)DIRECT_TILE, se - sb - t * DIRECT_TILE);
        const float4 *r = sh + bf * DIRECT_TILE * RS;
        float2 acc[NPK][NO];
#pragma unroll
        for (int u = 0; u < NPK; ++u)
#pragma unroll
            for (int c = 0; c < NO; ++c) acc[u][c] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int j = 0; j < cnt; ++j, r += RS) {
            const float4 a = r[0], b = r[1];
            const float2 yx = two(a.x), yy = two(a.y), yz = two(a.z), w = two(a.w);
            const float2 ylx = two(b.x), yly = two(b.y), ylz = two(b.z), px = two(b.w);
            float2 py, pz;
            if (DIPOLE) {
                const float2 f = *reinterpret_cast<const float2 *>(r + 2);
                py = two(f.x);
                pz = two(f.y);
            }
#pragma unroll
            for (int u = 0; u < NPK; ++u) {
                const float2 dx = __fadd2_rn(__fadd2_rn(cx[u], yx), __fadd2_rn(lx[u], ylx));
                const float2 dy = __fadd2_rn(__fadd2_rn(cy[u], yy), __fadd2_rn(ly[u], yly));
                const float2 dz = __fadd2_rn(__fadd2_rn(cz[u], yz), __fadd2_rn(lz[u], ylz));
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                float2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
                if (SKIP0) {
                    if (r2.x == 0.f) ri.x = 0.f;
                    if (r2.y == 0.f) ri.y = 0.f;
                }
                if (KIND == DO_PHI && !DIPOLE) {
                    acc[u][0] = __ffma2_rn(w, ri, acc[u][0]);
                    continue;
                }
                const float2 ri2 = __fmul2_rn(ri, ri), ri3 = __fmul2_rn(ri2, ri);
                if (KIND == DO_DN) {
                    const float2 nd = __ffma2_rn(nx[u], dx, __ffma2_rn(ny[u], dy, __fmul2_rn(nz[u], dz)));
                    acc[u][0] = __ffma2_rn(__fmul2_rn(w, nd), ri3, acc[u][0]);
                } else if (!DIPOLE) {  // potential and -gradient
                    acc[u][0] = __ffma2_rn(w, ri, acc[u][0]);
                    const float2 f = __fmul2_rn(w, ri3);
                    acc[u][1] = __ffma2_rn(f, dx, acc[u][1]);
                    acc[u][2] = __ffma2_rn(f, dy, acc[u][2]);
                    acc[u][3] = __ffma2_rn(f, dz, acc[u][3]);
                } else {  // potential p.d / r^3 and gradient p / r^3 - 3 (p.d) d / r^5
                    const float2 pd = __ffma2_rn(px, dx, __ffma2_rn(py, dy, __fmul2_rn(pz, dz)));
                    acc[u][0] = __ffma2_rn(pd, ri3, acc[u][0]);
                    const float2 f = __fmul2_rn(__fmul2_rn(__fmul2_rn(pd, make_float2(-3.f, -3.f)), ri3), ri2);
                    acc[u][1] = __fadd2_rn(acc[u][1], __ffma2_rn(f, dx, __fmul2_rn(px, ri3)));
                    acc[u][2] = __fadd2_rn(acc[u][2], __ffma2_rn(f, dy, __fmul2_rn(py, ri3)));
                    acc[u][3] = __fadd2_rn(acc[u][3], __ffma2_rn(f, dz, __fmul2_rn(pz, ri3)));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < NPK; ++u)
#pragma unroll
            for (int c = 0; c < NO; ++c) {
                const float2 v = acc[u][c];
                const bool neg = KIND == DO_PHI_GRAD && !DIPOLE && c > 0;
                outer[u][c] = __fadd2_rn(outer[u][c], neg ? make_float2(-v.x, -v.y) : v);
            }
    }
#pragma unroll
    for (int u = 0; u < NPK; ++u)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int64_t i = tgt(u, e);
            if (i >= ntgt) continue;
#pragma unroll
            for (int c = 0; c < NO; ++c) {
                const float v = e ? outer[u][c].y : outer[u][c].x;
                pp[i * NO + c] = KIND == DO_DN ? -v : v;
            }
        }
}

double *quad_values(Mesh &m) {
    return reinterpret_cast<double *>(m.opt.precision == BEM_MIXED ? (void *)m.str32.p : (void *)m.str64.p);
}

size_t direct_space(const Mesh &m) { return (size_t)(m.nqp + 1) / 2 + DREC_DIPOLE * DIRECT_TILE; }

// The records of a call live in memory that only products and GMRES use
// otherwise: the near field's strength records (16 bytes a quadrature point,
// less the values at the points when the call writes those) or, once a solve
// has run, its basis (31 vectors: room for every point's two records).
static void record_space(Mesh &m, bool values, float4 *&rec, size_t &n) {
    const size_t keep = values ? (size_t)(m.nqp + 1) / 2 : 0;
    rec = m.str32.p + keep;
    n = m.str32.n - keep;
    if (m.V.n / 2 > n) {
        rec = reinterpret_cast<float4 *>(m.V.p);
        n = m.V.n / 2;
    }
}

// Sources are packed and summed a segment at a time: as many whole tiles as
// there is room for (the tiles' sums do not depend on it).
void direct_partials(Mesh &m, const DirectSum &d, int64_t chunk, int nsplit, float *part) {
    cudaStream_t s = m.stream;
    const int rs = d.dipole ? DREC_DIPOLE : DREC_MONO;
    float4 *rec;
    size_t room;
    record_space(m, d.to_quad_values, rec, room);
    // (at most 32,768 splits a launch)
    const int64_t seg = std::min((int64_t)(room / rs / DIRECT_TILE), (int64_t)1 << 15) * DIRECT_TILE;
    if (seg == 0) throw Error(BEM_ECUDA, "direct sums: no room for a tile of records");
    const double ox = m.root_min[0] + 0.5 * m.side, oy = m.root_min[1] + 0.5 * m.side,
                 oz = m.root_min[2] + 0.5 * m.side;
    const size_t sm = (size_t)2 * DIRECT_TILE * rs * sizeof(float4);
    for (int64_t s0 = 0; s0 < d.nsrc; s0 += seg) {
        const int64_t s1 = std::min(d.nsrc, s0 + seg), n = s1 - s0;
        const double *sw = d.sw ? d.sw + s0 : nullptr, *dens = d.dens && !d.qpanel ? d.dens + s0 : d.dens;
        auto pack = d.dipole ? k_direct_pack<true> : k_direct_pack<false>;
        pack<<<cdiv(n, 256), 256, 0, s>>>(n, d.spos + 3 * s0, sw, d.snrm ? d.snrm + 3 * s0 : nullptr,
                                          d.qpanel ? d.qpanel + s0 : nullptr, dens, ox, oy, oz, rec);
        BEM_CHECK_LAUNCH();
        const int y0 = (int)(s0 / chunk), y1 = std::min(nsplit, (int)((s1 - 1) / chunk) + 1);
        auto go = [&](auto kern) {
            kern<<<dim3(cdiv(d.ntgt, DPK_TARGETS), y1 - y0), DPK_THREADS, sm, s>>>(
                d.ntgt, d.nsrc, chunk, s0, s1, y0, d.tpos, d.tnrm, rec, ox, oy, oz, part);
            BEM_CHECK_LAUNCH();
        };
        if (d.dipole && d.kind == DO_PHI_GRAD) go(k_direct_pk<true, DO_PHI_GRAD, true>);
        else if (d.dipole) throw Error(BEM_EUNSUPPORTED, "direct dipole sums: potential and gradient only");
        else if (d.kind == DO_DN) go(k_direct_pk<false, DO_DN, false>);
        else if (d.kind == DO_PHI_GRAD) go(k_direct_pk<false, DO_PHI_GRAD, true>);
        else if (d.skip_coincident) go(k_direct_pk<false, DO_PHI, true>);
        else go(k_direct_pk<false, DO_PHI, false>);
    }
}

// out[i] = mul x scale x the sum of the splits' parts: `group` consecutive splits in
// T (as if one CTA had summed their sources), then FP64 over the groups, shared
// by `lanes` threads (one thread loading 280 splits in turn took 20 us); n
// values, one to four of them a target.
template <class T>
__global__ void k_direct_reduce(const T *part, int nsplit, int group, int64_t n, double scale, double mul, int lanes,
                                double *out) {
    __shared__ double sh[256];
    const int per = blockDim.x / lanes, t = threadIdx.x % per, lane = threadIdx.x / per;
    const int64_t i = blockIdx.x * (int64_t)per + t;
    double s = 0.0;
    if (i < n)
        for (int k = lane * group; k < nsplit; k += lanes * group) {
            T g = part[(size_t)k * n + i];
            for (int e = k + 1; e < min(nsplit, k + group); ++e) g += part[(size_t)e * n + i];
            s += (double)g;
        }
    sh[threadIdx.x] = s;
    __syncthreads();
    if (lane == 0 && i < n) {
        for (int l = 1; l < lanes; ++l) s += sh[l * per + t];
        const double v = scale * s;
        out[i] = mul == 1.0 ? v : mul * v + 0.0 * v;  // as axpby does (a value that is not finite gives NaN)
    }
}

template <class T>
void direct_reduce(const T *part, int nsplit, int group, int64_t n, int no, double *out, cudaStream_t s, double mul) {
    const int ng = (nsplit + group - 1) / group, lanes = ng > 1024 ? 256 : (ng > 128 ? 32 : (ng > 16 ? 8 : 1));
    k_direct_reduce<T><<<cdiv(n * no, 256 / lanes), 256, 0, s>>>(part, nsplit, group, n * no, 1.0 / FOUR_PI, mul, lanes, out);
    BEM_CHECK_LAUNCH();
}
template void direct_reduce<float>(const float *, int, int, int64_t, int, double *, cudaStream_t, double);
template void direct_reduce<double>(const double *, int, int, int64_t, int, double *, cudaStream_t, double);

// out_j = mul sum_q (qw_jq / A_j) v_jq: the rule's average over panel j
__global__ void k_panel_avg(const double *v, const int *qp_of_panel, const double *qw, const double *area,
                            int nq, int64_t np, double mul, double *out) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= np) return;
    double a = 0.0;
    for (int q = 0; q < nq; ++q) {
        const int k = qp_of_panel[j * nq + q];
        a += qw[k] * v[k];
    }
    const double r = a / area[j];
    out[j] = mul == 1.0 ? r : mul * r + 0.0 * r;
}

// How a sum is cut: splits of `chunk` sources, `group` of them added in T before
// FP64.  With tiles = false a CTA sums a whole split: the same sums from fewer
// parts, for a device that has no room for more.
struct DirectCut {
    int64_t chunk;
    int nsplit, group;
};
static DirectCut direct_cut(const Mesh &m, bool tiles, SrcKind sk, int64_t nsrc, int64_t ntgt) {
    const int tblocks = cdiv(ntgt, DIRECT_THREADS);
    // enough CTAs to fill the GPU about twice (16 per SM), splits of at least 512 sources
    int nsplit = std::max(1, (int)std::min<int64_t>(cdiv(nsrc, 512), std::max(1, 2432 / tblocks)));
    nsplit = std::min(nsplit, 65535);
    int64_t chunk = (nsrc + nsplit - 1) / nsplit;
    chunk = ((chunk + DIRECT_THREADS - 1) / DIRECT_THREADS) * DIRECT_THREADS;
    // FP32: a CTA per tile of a split, the split's tiles added in order by the
    // reduction: bit for bit the sums that a CTA per split gives, in shorter CTAs
    // (81,920 targets, 2,000 charges are 1.2 waves of splits; 100 targets, 28.7M
    // points 1.6: 4.30 ms, 5.08 with a CTA per split)
    int group = 1;
    if (tiles && chunk <= 64 * DIRECT_TILE &&
        (double)cdiv(nsrc, DIRECT_TILE) * ntgt <= (sk == SRC_QUAD ? 1.5 : 1.0) * parts_limit(m)) {
        group = (int)(chunk / DIRECT_TILE);
        chunk = DIRECT_TILE;
    }
    return DirectCut{chunk, (int)((nsrc + chunk - 1) / chunk), group};
}

template <class T>
static void direct_impl(Mesh &m, SrcKind sk, TgtKind tk, const double *dens, double *out, DArray<T> &part, double mul) {
    cudaStream_t s = m.stream;
    const int64_t ntgt = (tk == TGT_CEN_DN) ? m.np : ((tk == TGT_QUAD_DN || tk == TGT_QUAD_PHI) ? m.nqp : m.nc);
    // Galerkin rows: the values at the quadrature points, then the rule's
    // average over each panel
    double *const final_out = out;
    if (tk == TGT_QUAD_DN) {
        if (!m.nrmq64.p || m.gq_tmp.n < (size_t)m.nqp) throw Error(BEM_EUNSUPPORTED, "Galerkin geometry not built");
        out = m.gq_tmp.p;
    }
    const int64_t nsrc = (sk == SRC_QUAD) ? m.nqp : m.nc;
    if (ntgt == 0) return;
    if (nsrc == 0) {
        BEM_CUDA(cudaMemsetAsync(final_out, 0, (tk == TGT_QUAD_DN ? m.np : ntgt) * sizeof(double), s));
        return;
    }
    DirectCut cut = direct_cut(m, std::is_same<T, float>::value, sk, nsrc, ntgt);
    if (part.n < (size_t)cut.nsplit * ntgt) {
        try {
            part.alloc((size_t)cut.nsplit * ntgt);
        } catch (const Error &e) {
            if (e.code != BEM_ENOMEM || cut.group == 1) throw;
            cut = direct_cut(m, false, sk, nsrc, ntgt);
            part.alloc((size_t)cut.nsplit * ntgt);
        }
    }
    const int64_t chunk = cut.chunk;
    const int nsplit = cut.nsplit, group = cut.group;
    [[maybe_unused]] const int tblocks = cdiv(ntgt, DIRECT_THREADS);
    [[maybe_unused]] const double ox = m.root_min[0] + 0.5 * m.side, oy = m.root_min[1] + 0.5 * m.side,
                                  oz = m.root_min[2] + 0.5 * m.side;
    const double *tpos = (tk == TGT_CEN_DN) ? m.cen64.p : ((tk == TGT_QUAD_DN || tk == TGT_QUAD_PHI) ? m.qpg64.p : m.chgg64.p);
    const double *spos = (sk == SRC_QUAD) ? m.qpg64.p : m.chgg64.p;
    const double *sw = (sk == SRC_QUAD) ? m.qw64.p : m.q64.p;
    const double *tnrm = tk == TGT_CEN_DN ? m.nrm64.p : (tk == TGT_QUAD_DN ? m.nrmq64.p : nullptr);
    const int *qpanel = sk == SRC_QUAD ? m.qp_panel.p : nullptr;
    if (sk == SRC_QUAD && (tk == TGT_QUAD_DN || tk == TGT_QUAD_PHI))
        throw Error(BEM_EUNSUPPORTED, "direct quadrature-to-quadrature sums not built");
    if constexpr (std::is_same<T, float>::value) {
        DirectSum d;
        d.kind = tnrm ? DO_DN : DO_PHI;
        d.nsrc = nsrc;
        d.ntgt = ntgt;
        d.spos = spos;
        d.sw = sw;
        d.dens = dens;
        d.qpanel = qpanel;
        d.tpos = tpos;
        d.tnrm = tnrm;
        d.to_quad_values = out == quad_values(m);
        direct_partials(m, d, chunk, nsplit, part.p);
    } else {
        dim3 grid(tblocks, nsplit);
        auto go = [&](auto kern) {
            kern<<<grid, DIRECT_THREADS, 0, s>>>(ntgt, nsrc, chunk, tpos, tnrm, spos, sw, qpanel, dens, ox, oy, oz,
                                                 part.p);
            BEM_CHECK_LAUNCH();
        };
        if (sk == SRC_QUAD && tk == TGT_CHG_PHI) go(k_direct<SRC_QUAD, TGT_CHG_PHI>);
        else if (sk == SRC_QUAD && tk == TGT_CEN_DN) go(k_direct<SRC_QUAD, TGT_CEN_DN>);
        else if (tnrm) go(k_direct<SRC_CHARGE, TGT_CEN_DN>);
        else go(k_direct<SRC_CHARGE, TGT_CHG_PHI>);
    }
    direct_reduce<T>(part.p, nsplit, group, ntgt, 1, out, s, tk == TGT_QUAD_DN ? 1.0 : mul);
    if (tk == TGT_QUAD_DN) {
        k_panel_avg<<<cdiv(m.np, 256), 256, 0, s>>>(out, m.qp_of_panel.p, m.qw64.p, m.area64.p, (int)m.nq,
                                                    m.np, mul, final_out);
        BEM_CHECK_LAUNCH();
    }
}

// out_j = sum_q qw_jq v_jq (the rule's weights include the panel area)
__global__ void k_panel_wsum(const double *v, const int *qp_of_panel, const double *qw, int nq, int64_t np,
                             double *out) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= np) return;
    double a = 0.0;
    for (int q = 0; q < nq; ++q) {
        const int k = qp_of_panel[j * nq + q];
        a += qw[k] * v[k];
    }
    out[j] = a;
}

void panel_wsum(Mesh &m, const double *v, double *out) {
    k_panel_wsum<<<cdiv(m.np, 256), 256, 0, m.stream>>>(v, m.qp_of_panel.p, m.qw64.p, (int)m.nq, m.np, out);
    BEM_CHECK_LAUNCH();
}

// C^T q in the sorted panel order: (C^T q)_j = sum_q A_j w_q psi(y_jq) with
// psi(y) = sum_k q_k G(x_k, y), so that q . (C sigma) = (C^T q) . sigma and
// the solvation energy of any sigma is one dot product (Eq. energy).  Built
// in the product's precision for meshes whose charge sums are direct.
void build_ctq(Mesh &m) {
    m.ctq_ok = false;
    if (m.nc == 0 || !charge_direct(m)) return;
    if (m.ctq.n < (size_t)m.np) m.ctq.alloc(m.np);
    if (m.opt.precision == BEM_MIXED) {  // room for both sums over the charges, not left to the first right-hand side
        const int64_t nt = m.opt.galerkin ? m.nqp : m.np;
        const size_t need = std::max((size_t)direct_cut(m, true, SRC_CHARGE, m.nc, nt).nsplit * nt,
                                     (size_t)direct_cut(m, true, SRC_CHARGE, m.nc, m.nqp).nsplit * m.nqp);
        if (m.dpart_f.n < need) {
            try {
                m.dpart_f.alloc(need);
            } catch (const Error &e) {  // no room: each sum takes what it needs
                if (e.code != BEM_ENOMEM) throw;
            }
        }
    }
    double *psi = quad_values(m);
    direct_pass(m, SRC_CHARGE, TGT_QUAD_PHI, nullptr, psi);
    panel_wsum(m, psi, m.ctq.p);
    charge_near_ct(m, m.q64.p, m.ctq.p);
    BEM_CUDA(cudaStreamSynchronize(m.stream));
    m.ctq_ok = true;
}

void direct_pass(Mesh &m, SrcKind sk, TgtKind tk, const double *dens, double *out, double mul) {
    if (m.opt.precision == BEM_MIXED) direct_impl<float>(m, sk, tk, dens, out, m.dpart_f, mul);
    else direct_impl<double>(m, sk, tk, dens, out, m.dpart_d, mul);
}

bool charge_direct(const Mesh &m) {
    if (m.opt.charge_mode == BEM_CHARGE_DIRECT) return true;
    if (m.opt.charge_mode == BEM_CHARGE_FMM) return false;
    return (double)m.nc * (double)m.nqp <= 4e10;
}

void charge_pass(Mesh &m, SrcKind sk, TgtKind tk, const double *dens, double *out, double mul) {
    if (charge_direct(m)) {
        direct_pass(m, sk, tk, dens, out, mul);
        return;
    }
    fmm_pass(m, m.tc, sk, tk, dens, out, false);
    if (mul != 1.0) axpby(m, mul, out, 0.0, out, out, tk == TGT_CHG_PHI ? m.nc : m.np);
}

}  // namespace bem
