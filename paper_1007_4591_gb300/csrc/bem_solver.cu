// BEM operator, restarted GMRES and energy reductions (Sec. 2.1, Sec. 2.2).
//
// All vectors here are FP64 and in the sorted panel order; the public entry
// points gather/scatter at the boundary.  GMRES (Saad & Schultz) runs on the
// device: classical Gram-Schmidt applied twice (CGS2) for the Arnoldi step,
// Givens rotations for the least-squares update, one 8-byte residual written to
// pinned host memory per iteration to decide convergence.
#include <cmath>
#include <type_traits>
#include <vector>

#include "bem_internal.cuh"

namespace bem {

constexpr int RED_THREADS = 256;

// ------------------------------------------------------------ permutations
__global__ void k_gather(const double *src, const int *perm, double *dst, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) dst[i] = src[perm[i]];
}
__global__ void k_scatter(const double *src, const int *perm, double *dst, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) dst[perm[i]] = src[i];
}
__global__ void k_scatter_scaled(double a, const double *src, const int *perm, double *dst, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) dst[perm[i]] = a * src[i] + 0.0 * src[i];  // as axpby does (a value that is not finite gives NaN)
}
__global__ void k_scatter3(const double *src, const int *perm, double *dst, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t j = perm[i];
    dst[3 * j] = src[3 * i];
    dst[3 * j + 1] = src[3 * i + 1];
    dst[3 * j + 2] = src[3 * i + 2];
}

void gather_f64(const double *src, const int *perm, double *dst, int64_t n, cudaStream_t s) {
    k_gather<<<cdiv(n, 256), 256, 0, s>>>(src, perm, dst, n);
    BEM_CHECK_LAUNCH();
}
void scatter_f64(const double *src, const int *perm, double *dst, int64_t n, cudaStream_t s) {
    k_scatter<<<cdiv(n, 256), 256, 0, s>>>(src, perm, dst, n);
    BEM_CHECK_LAUNCH();
}
void scatter_scaled(double a, const double *src, const int *perm, double *dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    k_scatter_scaled<<<cdiv(n, 256), 256, 0, s>>>(a, src, perm, dst, n);
    BEM_CHECK_LAUNCH();
}
void scatter_rows3(const double *src, const int *perm, double *dst, int64_t n, cudaStream_t s) {
    k_scatter3<<<cdiv(n, 256), 256, 0, s>>>(src, perm, dst, n);
    BEM_CHECK_LAUNCH();
}

// --------------------------------------------------------------- operator
// y = x + Ehat (K'x): kx holds the fast multipole K' x (sorted order); the
// FP64 near-singular table replaces the FP32 near-field values of the pairs
// it lists.
// y = x + Ehat (K'x + table x): four lanes per row share the row's table
// entries (a dozen or so gathers each row), then add up by shuffles.
__global__ void k_apply_A(const double *x, const double *kx, const int *nt_off, const int *nt_col,
                          const double *nt_val, double ehat, int64_t n, double *y) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 2;
    const int sub = threadIdx.x & 3;
    double k = 0.0;
    if (i < n && nt_off)
        for (int e = nt_off[i] + sub; e < nt_off[i + 1]; e += 4) k += nt_val[e] * x[nt_col[e]];
    k += __shfl_xor_sync(0xffffffffu, k, 1);
    k += __shfl_xor_sync(0xffffffffu, k, 2);
    if (i < n && sub == 0) y[i] = x[i] + ehat * (kx[i] + k);
}

static void matvec_launch(Mesh &m, const double *xs, double *ys) {
    if (!m.opt.galerkin) {
        kprime_apply(m, xs, ys);  // the pass ends in the epilogue itself
    } else {
        const bool nt = m.nt_nnz > 0 && !(m.opt.flags & (BEM_FLAG_NO_NEARTAB | BEM_FLAG_NO_NEAR));
        fmm_pass(m, m.tp, SRC_QUAD, TGT_QUAD_DN, xs, m.zs.p, true);
        k_apply_A<<<cdiv(4 * m.np, 256), 256, 0, m.stream>>>(xs, m.zs.p, nt ? m.nt_off.p : nullptr,
                                                          m.nt_col.p, m.nt_val.p, m.ehat, m.np, ys);
        BEM_CHECK_LAUNCH();
    }
    if (m.tm.on) BEM_CUDA(cudaEventRecord(m.tm.ev[7], m.stream));
}

// The K' product is a fixed sequence of ~20 kernels and memsets; with
// opt.graph it is captured once (on the buffers gx -> gy, after one ordinary
// run has set every kernel attribute) and replayed as a single graph launch.
static cudaError_t set_node_priorities(cudaGraph_t g) {
    int prio_lo = 0, prio_hi = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi);
    size_t n = 0;
    if (e == cudaSuccess) e = cudaGraphGetNodes(g, nullptr, &n);
    std::vector<cudaGraphNode_t> nodes(n);
    if (e == cudaSuccess && n > 0) e = cudaGraphGetNodes(g, nodes.data(), &n);
    for (size_t i = 0; e == cudaSuccess && i < n; ++i) {
        cudaGraphNodeType ty;
        e = cudaGraphNodeGetType(nodes[i], &ty);
        if (e != cudaSuccess || ty != cudaGraphNodeTypeKernel) continue;
        cudaKernelNodeParams kp{};
        e = cudaGraphKernelNodeGetParams(nodes[i], &kp);
        if (e != cudaSuccess) break;
        cudaLaunchAttributeValue v{};
        v.priority = is_near_field_kernel(kp.func) ? prio_lo : prio_hi;
        e = cudaGraphKernelNodeSetAttribute(nodes[i], cudaLaunchAttributePriority, &v);
    }
    return e;
}

void matvec_sorted(Mesh &m, const double *xs, double *ys) {
    if (!m.opt.graph || m.tm.on) {
        matvec_launch(m, xs, ys);
        return;
    }
    if (!m.g_mv) {
        if (m.gx.n < (size_t)m.np) {
            m.gx.alloc(m.np);
            m.gy.alloc(m.np);
        }
        matvec_launch(m, xs, ys);  // warm-up outside the capture
        cudaGraph_t g = nullptr;
        BEM_CUDA(cudaStreamBeginCapture(m.stream, cudaStreamCaptureModeThreadLocal));
        m.capturing = true;
        try {
            matvec_launch(m, m.gx.p, m.gy.p);
        } catch (...) {
            m.capturing = false;
            cudaStreamEndCapture(m.stream, &g);
            if (g) cudaGraphDestroy(g);
            throw;
        }
        m.capturing = false;
        BEM_CUDA(cudaStreamEndCapture(m.stream, &g));
        // Kernel nodes do not keep their capturing stream's priority: give the
        // near-field kernels the lowest and every other kernel the highest, so
        // that the graph runs the two branches as the streams would.
        cudaError_t e = set_node_priorities(g);
        if (e == cudaSuccess) e = cudaGraphInstantiateWithFlags(&m.g_mv, g, cudaGraphInstantiateFlagUseNodePriority);
        cudaGraphDestroy(g);
        BEM_CUDA(e);
        return;
    }
    if (xs != m.gx.p)
        BEM_CUDA(cudaMemcpyAsync(m.gx.p, xs, m.np * sizeof(double), cudaMemcpyDeviceToDevice, m.stream));
    BEM_CUDA(cudaGraphLaunch(m.g_mv, m.stream));
    if (ys != m.gy.p)
        BEM_CUDA(cudaMemcpyAsync(ys, m.gy.p, m.np * sizeof(double), cudaMemcpyDeviceToDevice, m.stream));
}

// --------------------------------------------------------------- BLAS-1
// Reductions end in the kernel that starts them: the last CTA to arrive
// (a ticket that wraps to zero) adds the CTAs' parts in a fixed order.  Up to
// some 100,000 panels these kernels are launches and latency, not bandwidth
// (8 n bytes a vector, 0.1 us at 81,920 panels): an Arnoldi step was 11 launches
// and a copy, is four launches, and the host reads the residual from pinned
// memory the device writes.  Above, FP64 issue and the passes over the basis
// count: the second pass of Gram-Schmidt subtracts and forms its products in
// one.  Kernels of a step, averages of 7 to 10 steps, against the eleven:
// 81,920 panels 38 us (60), 655,360 74 us (92), 2.6M 0.170 ms (0.208), 12.3M
// 0.640 ms (0.778).

// CTAs of a reduction over n rows, each a stride of the grid apart so that the
// CTAs sweep a vector together: 152 while the vectors lie in L2 and the end of
// the reduction costs more than a sparse sweep (655,360 rows: 74 us with 152,
// 77 with 304), from 24 rows a thread on twice as many (1.3M rows 115 and 104
// us, 12.3M 0.942 and 0.640 ms; 608: 119 us and 0.652 ms).
static int ctas_for(int64_t n) {
    const int64_t most = n < (int64_t)152 * RED_THREADS * 24 ? 152 : 304;
    return (int)std::min<int64_t>(cdiv(n, RED_THREADS), most);
}

__device__ __forceinline__ bool last_cta(unsigned *ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// nvec vectors are `full` blocks of VEC_BLOCK and a last one of NV (1 to
// VEC_BLOCK), a compile-time parameter (MORE: full > 0): FP64 issue bounds these kernels once
// they fill the chip, and a lane that a predicate turns off takes its slot all
// the same.  A thread has the loads of a whole block in flight.
constexpr int VEC_BLOCK = 8;

// part[i][CTA] = the CTA's sum of s[i]
template <int NV>
__device__ __forceinline__ void cta_parts(double (&s)[NV], double *part) {
    __shared__ double sh[NV][RED_THREADS / 32];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        for (int o = 16; o > 0; o >>= 1) s[i] += __shfl_down_sync(0xffffffffu, s[i], o);
        if (lane == 0) sh[i][wp] = s[i];
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int k = 0; k < RED_THREADS / 32; ++k) t += sh[threadIdx.x][k];
        part[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = t;
    }
}

// sum_i h[i] V_i[r] over `full` blocks and the last one, whose values are v
template <int NV, bool MORE>
__device__ __forceinline__ double row_sum(const double *__restrict__ V, size_t ld, int full, const double *h, int64_t r,
                                          const double (&v)[NV]) {
    double a = 0.0;
    for (int i0 = 0; MORE && i0 < VEC_BLOCK * full; i0 += VEC_BLOCK) {
        double u[VEC_BLOCK];
#pragma unroll
        for (int i = 0; i < VEC_BLOCK; ++i) u[i] = V[(size_t)(i0 + i) * ld + r];
#pragma unroll
        for (int i = 0; i < VEC_BLOCK; ++i) a += h[i0 + i] * u[i];
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) a += h[(MORE ? VEC_BLOCK * full : 0) + i] * v[i];
    return a;
}

// part[i][CTA] = the CTA's rows' share of (last block)_i . w; with SUB,
// w -= sum_i h[i] V_i over all blocks first, in the same pass
template <int NV, bool SUB, bool MORE>
__device__ __forceinline__ void dot_block(const double *__restrict__ V, size_t ld, int full, const double *h,
                                          double *__restrict__ w, int64_t n, double *part) {
    constexpr int U = NV >= 5 ? 1 : (NV >= 3 ? 2 : 4);  // rows of a thread in flight
    const double *__restrict__ Vl = V + (size_t)VEC_BLOCK * full * ld;
    double s[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] = 0.0;
#pragma unroll U
    for (int64_t r = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; r < n; r += (int64_t)gridDim.x * RED_THREADS) {
        double v[NV], x = w[r];
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = Vl[(size_t)i * ld + r];
        if (SUB) {
            x -= row_sum<NV, MORE>(V, ld, full, h, r, v);
            w[r] = x;
        }
#pragma unroll
        for (int i = 0; i < NV; ++i) s[i] += v[i] * x;
    }
    cta_parts<NV>(s, part + (size_t)VEC_BLOCK * full * gridDim.x);
}

// out[i] = the sum of vector i's parts (a warp per vector)
__device__ __forceinline__ void sum_parts(const double *part, int nvec, double *out) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < nvec; i += RED_THREADS / 32) {
        double t = 0.0;
        for (int k = lane; k < (int)gridDim.x; k += 32) t += __ldcg(part + (size_t)i * gridDim.x + k);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) out[i] = t;
    }
}

// out[0] = V . w (mode 0) or its square root (mode 1), also written to `host`
__global__ void __launch_bounds__(RED_THREADS)
k_dot(const double *V, const double *w, int64_t n, double *part, unsigned *ticket, int mode, double *out,
      volatile double *host) {
    dot_block<1, false, false>(V, 0, 0, nullptr, const_cast<double *>(w), n, part);  // reads w only
    if (!last_cta(ticket)) return;
    __shared__ double t;
    sum_parts(part, 1, &t);
    if (threadIdx.x == 0) {
        const double v = mode ? sqrt(t) : t;
        out[0] = v;
        *host = v;
        __threadfence_system();
    }
}

// First pass of classical Gram-Schmidt, h = V^T w, or (SUB) the second:
// w -= V hsub, then h = V^T w.
template <int NV, bool SUB, bool MORE>
__global__ void __launch_bounds__(RED_THREADS, MORE ? 3 : 4)
k_cgs(const double *V, size_t ld, int full, const double *hsub, double *w, int64_t n, double *part,
      unsigned *ticket, double *h) {
    // every thread reads back the rows it writes
    dot_block<NV, SUB, MORE>(V, ld, full, hsub, w, n, part);
    for (int f = 0; MORE && f < full; ++f) dot_block<VEC_BLOCK, false, false>(V, ld, f, nullptr, w, n, part);  // block f
    if (last_cta(ticket)) sum_parts(part, VEC_BLOCK * full + NV, h);
}

// Givens update of Hessenberg column j (column-major, leading dimension m1).
__device__ void givens(double *H, int m1, const double *hcol, int j, double *cs, double *sn, double *g, double inv_bnorm,
                       double *out /* [0]=resid, [1]=1/norm */) {
    double *h = H + (size_t)j * m1;
    for (int i = 0; i <= j + 1; ++i) h[i] = hcol[i];
    const double wn = h[j + 1];
    for (int i = 0; i < j; ++i) {
        const double t = cs[i] * h[i] + sn[i] * h[i + 1];
        h[i + 1] = -sn[i] * h[i] + cs[i] * h[i + 1];
        h[i] = t;
    }
    const double den = hypot(h[j], h[j + 1]);
    if (den > 0.0) {
        cs[j] = h[j] / den;
        sn[j] = h[j + 1] / den;
    } else {
        cs[j] = 1.0;
        sn[j] = 0.0;
    }
    h[j] = den;
    h[j + 1] = 0.0;
    g[j + 1] = -sn[j] * g[j];
    g[j] = cs[j] * g[j];
    out[0] = fabs(g[j + 1]) * inv_bnorm;
    out[1] = (wn > 0.0) ? 1.0 / wn : 0.0;
}

// The Arnoldi step's end: w -= V h2, |w|, the Hessenberg column h + h2 | |w|
// through the Givens rotations, the residual to the host.
template <int NV, bool MORE>
__global__ void __launch_bounds__(RED_THREADS, MORE ? 3 : 4)
k_cgs_end(const double *V, size_t ld, int full, double *h, const double *h2, double *w, int64_t n, double *part,
          unsigned *ticket, double *H, int m1, double *cs, double *sn, double *g, double inv_bnorm, double *out,
          volatile double *host) {
    constexpr int U = NV >= 5 ? 1 : (NV >= 3 ? 2 : 4);
    const int j = VEC_BLOCK * full + NV - 1;
    const double *__restrict__ Vl = V + (size_t)VEC_BLOCK * full * ld;
    double *__restrict__ wr = w;
    double s[1] = {0.0};
#pragma unroll U
    for (int64_t r = blockIdx.x * (int64_t)RED_THREADS + threadIdx.x; r < n; r += (int64_t)gridDim.x * RED_THREADS) {
        double v[NV], x = wr[r];
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = Vl[(size_t)i * ld + r];
        x -= row_sum<NV, MORE>(V, ld, full, h2, r, v);
        wr[r] = x;
        s[0] += x * x;
    }
    cta_parts<1>(s, part);
    if (!last_cta(ticket)) return;
    __shared__ double t;
    sum_parts(part, 1, &t);
    for (int i = threadIdx.x; i <= j; i += RED_THREADS) h[i] += h2[i];
    __syncthreads();
    if (threadIdx.x == 0) {
        h[j + 1] = sqrt(t);
        givens(H, m1, h, j, cs, sn, g, inv_bnorm, out);
        *host = out[0];
        __threadfence_system();
    }
}

// x += sum_i h[i] V_i
__global__ void k_multi_axpy(const double *V, size_t ld, int nvec, const double *h, double *x, int64_t n) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    double a = 0.0;
    for (int i = 0; i < nvec; ++i) a += h[i] * V[(size_t)i * ld + r];
    x[r] += a;
}

__global__ void k_scale_by(double *w, const double *sc, int64_t n) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n) w[r] *= sc[0];
}

// v = u / d[0] (u may be v), and g = (d[0], 0, ..., 0) with m1 entries
__global__ void k_start_basis(const double *u, const double *d, double *v, int64_t n, double *g, int m1) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n) v[r] = u[r] / d[0];
    if (r < m1) g[r] = r == 0 ? d[0] : 0.0;
}

__global__ void k_axpby(double a, const double *x, double b, const double *y, double *out,
                        int64_t n) {
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n) out[r] = a * x[r] + b * y[r];
}

// Back substitution H[:k,:k] y = g[:k], column by column: a thread per row
// (one thread alone waits for every entry in turn).
__global__ void k_backsolve(const double *H, int m1, const double *g, int k, double *y) {
    __shared__ double yi;
    const int l = threadIdx.x;
    double s = l < k ? g[l] : 0.0;
    for (int i = k - 1; i >= 0; --i) {
        const double v = l <= i ? H[(size_t)i * m1 + l] : 0.0;
        if (l == i) {
            yi = v != 0.0 ? s / v : 0.0;
            y[i] = yi;
        }
        __syncthreads();
        if (l < i) s -= v * yi;
        __syncthreads();
    }
}

// V . w (mode 0) or its square root (mode 1), left in *out and read by the host
static double dot_read(Mesh &m, const double *V, const double *w, int64_t n, int mode, double *out) {
    k_dot<<<ctas_for(n), RED_THREADS, 0, m.stream>>>(V, w, n, m.part.p, m.ticket.p, mode, out, m.h_pinned);
    BEM_CHECK_LAUNCH();
    BEM_CUDA(cudaStreamSynchronize(m.stream));
    return *const_cast<volatile double *>(m.h_pinned);
}

double norm2(Mesh &m, const double *w) { return dot_read(m, w, w, m.np, 1, m.red.p); }

// the right-hand side of the system at hand
double *rhs_vector(Mesh &m) {
    if (m.bvec.n < (size_t)m.np) m.bvec.alloc(m.np);
    return m.bvec.p;
}

// f(NV, MORE) of nvec vectors
template <int NV = 1, class F>
static void with_blocks(int nvec, F &&f) {
    if ((nvec - 1) % VEC_BLOCK + 1 == NV) {
        if (nvec > VEC_BLOCK) f(std::integral_constant<int, NV>(), std::true_type());
        else f(std::integral_constant<int, NV>(), std::false_type());
    } else if constexpr (NV < VEC_BLOCK) {
        with_blocks<NV + 1>(nvec, f);
    }
}

// Solve A x = b (sorted order).  x holds the initial guess on entry; with
// x_zero the caller knows it to be zero.
int gmres_solve(Mesh &m, const double *b, double *x, bool transpose, bool x_zero, bem_solve_stats *st) {
    const int64_t n = m.np;
    const int mr = std::max(1, m.opt.gmres_restart);
    const int m1 = mr + 1;
    const size_t ld = (size_t)n;
    cudaStream_t s = m.stream;
    if (m.V.n < (size_t)m1 * ld) m.V.alloc((size_t)m1 * ld);
    if (m.H.n < (size_t)m1 * mr) m.H.alloc((size_t)m1 * mr);
    if (m.gv.n < (size_t)m1) m.gv.alloc(m1);
    if (m.cs.n < (size_t)mr) { m.cs.alloc(mr); m.sn.alloc(mr); }
    if (m.yv.n < (size_t)mr) m.yv.alloc(mr);
    if (m.hv.n < (size_t)m1 + 2) m.hv.alloc(m1 + 2);
    const int nb = cdiv(n, 256);
    auto apply = [&](const double *in, double *out) {
        if (!transpose) matvec_sorted(m, in, out);
        else {
            matvec_t_sorted(m, in, out);
        }
    };
    const double bnorm = norm2(m, b);
    int it = 0, restarts = 0;
    double rec = 1.0;
    bool conv = false, stagnated = false;
    std::vector<double> hist;
    if (bnorm == 0.0) {
        BEM_CUDA(cudaMemsetAsync(x, 0, n * sizeof(double), s));
        rec = 0.0;
        conv = true;
    }
    // an all-zero initial guess skips one product: the residual is b
    const bool told = x_zero;  // red[0] still holds |b|
    if (!x_zero && !conv) x_zero = norm2(m, x) == 0.0;
    const int ncta = ctas_for(n);
    while (!conv && it < m.opt.max_iter && !stagnated) {
        double *V0 = m.V.p;
        const double *r0 = b;
        if (!x_zero) {
            apply(x, V0);
            k_axpby<<<nb, 256, 0, s>>>(1.0, b, -1.0, V0, V0, n);
            BEM_CHECK_LAUNCH();
            r0 = V0;
        }
        const double beta = told && it == 0 ? bnorm : norm2(m, r0);
        rec = beta / bnorm;
        if (rec <= m.opt.tol) {
            conv = true;
            break;
        }
        // V0 = r0 / beta, with beta read on the device (left in red[0] by norm2)
        k_start_basis<<<std::max(nb, cdiv(m1, 256)), 256, 0, s>>>(r0, m.red.p, V0, n, m.gv.p, m1);
        BEM_CHECK_LAUNCH();
        int k = 0;
        for (int j = 0; j < mr; ++j) {
            double *w = m.V.p + (size_t)(j + 1) * ld;
            apply(m.V.p + (size_t)j * ld, w);
            ++it;
            // CGS2: two passes of classical Gram-Schmidt
            with_blocks(j + 1, [&](auto nv, auto more) {
                constexpr int NV = decltype(nv)::value;
                constexpr bool MORE = decltype(more)::value;
                const int full = j / VEC_BLOCK;
                k_cgs<NV, false, MORE><<<ncta, RED_THREADS, 0, s>>>(m.V.p, ld, full, nullptr, w, n, m.part.p, m.ticket.p,
                                                                    m.hv.p);
                BEM_CHECK_LAUNCH();
                k_cgs<NV, true, MORE><<<ncta, RED_THREADS, 0, s>>>(m.V.p, ld, full, m.hv.p, w, n, m.part.p, m.ticket.p,
                                                                   m.yv.p);
                BEM_CHECK_LAUNCH();
                k_cgs_end<NV, MORE><<<ncta, RED_THREADS, 0, s>>>(m.V.p, ld, full, m.hv.p, m.yv.p, w, n, m.part.p,
                                                                 m.ticket.p, m.H.p, m1, m.cs.p, m.sn.p, m.gv.p,
                                                                 1.0 / bnorm, m.red.p, m.h_pinned);
                BEM_CHECK_LAUNCH();
            });
            k_scale_by<<<nb, 256, 0, s>>>(w, m.red.p + 1, n);
            BEM_CHECK_LAUNCH();
            BEM_CUDA(cudaStreamSynchronize(s));
            rec = *const_cast<volatile double *>(m.h_pinned);
            hist.push_back(rec);
            k = j + 1;
            if (!(rec == rec)) {  // NaN
                stagnated = true;
                break;
            }
            if (rec <= m.opt.tol || it >= m.opt.max_iter) break;
            const size_t hs = hist.size();
            if (hs > 60 && rec > 0.5 * hist[hs - 51]) {
                stagnated = true;
                break;
            }
        }
        k_backsolve<<<1, RED_THREADS, 0, s>>>(m.H.p, m1, m.gv.p, k, m.yv.p);
        BEM_CHECK_LAUNCH();
        k_multi_axpy<<<nb, 256, 0, s>>>(m.V.p, ld, k, m.yv.p, x, n);
        BEM_CHECK_LAUNCH();
        x_zero = false;
        if (rec <= m.opt.tol) conv = true;
        else ++restarts;
    }
    double true_res = rec;
    if (st) {
        // true residual from one more product
        apply(x, m.ys.p);
        k_axpby<<<nb, 256, 0, s>>>(1.0, b, -1.0, m.ys.p, m.ys.p, n);
        BEM_CHECK_LAUNCH();
        true_res = (bnorm > 0) ? norm2(m, m.ys.p) / bnorm : 0.0;
        st->iterations = it;
        st->restarts = restarts;
        st->converged = conv ? 1 : 0;
        st->resid = rec;
        st->true_resid = true_res;
    }
    BEM_CUDA(cudaStreamSynchronize(s));
    return conv ? BEM_OK : BEM_ENOCONV;
}

// dG = 4 pi 332.0637 / (2 eps_in) * (C^T q) . sigma
double energy_from_ctq(Mesh &m, const double *sig_s) {
    return FOUR_PI * KCAL / (2.0 * m.eps_in) * dot_read(m, m.ctq.p, sig_s, m.np, 0, m.red.p + 2);
}

// dG = 4 pi 332.0637 / (2 eps_in) * q . phi   (phi = C sigma, G = 1/(4 pi r))
double energy_from_phi(Mesh &m, const double *phi_s) {
    return FOUR_PI * KCAL / (2.0 * m.eps_in) * dot_read(m, m.q64.p, phi_s, m.nc, 0, m.red.p + 2);
}

void axpby(Mesh &m, double a, const double *x, double b, const double *y, double *out, int64_t n) {
    k_axpby<<<cdiv(n, 256), 256, 0, m.stream>>>(a, x, b, y, out, n);
    BEM_CHECK_LAUNCH();
}

}  // namespace bem
