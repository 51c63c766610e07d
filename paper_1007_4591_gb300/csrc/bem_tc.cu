// M2L translations on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// The M2L step of the downward sweep (Sec. 2.3) is, for every offset class
// o of the interaction list, the dense product L_t += T_o M_s over all pairs
// (t, s) with that offset: with the pairs of one class gathered as columns
// this is a GEMM  D[128 x 128] = T_o[128 x 128] . B[128 x 128 pairs]
// ((p+1)^2 = 121 coefficients padded to 128; p <= 10).  It runs as
// tcgen05.mma kind::tf32 with the 3xTF32 split a b ~ a_hi b_hi + a_hi b_lo +
// a_lo b_hi (tf32 keeps 11 significant bits; the split recovers FP32-level
// products).  The operator (A) and the accumulators live in tensor memory;
// the multipoles (B) are staged in shared memory one K-block (32
// coefficients, 128 bytes of a row) at a time in the K-major layout with the
// 128-byte swizzle: a warp's load reads four 128-byte pieces of rows from
// global memory in FP32 and the producers split them as they store.  A persistent, warp-specialised kernel
// runs the pairs of one class as a stream of 128-pair tiles (producers, one
// MMA thread, epilogue; see k_m2l_tc).  The epilogue adds each pair's
// local-expansion row into its target cell with a bulk reduction
// (cp.reduce.async.bulk, add.f32): the targets' local expansions (a few MB)
// stay in L2, which absorbs the reductions, and no per-pair
// buffer is written or read back.  Every wait is bounded: the pipeline waits by
// the mesh's wait budget (bem_set_wait_budget), after which the kernel
// raises an error flag; the last wait for its own MMAs (always about a
// second) comes before it frees its tensor memory and returns.
#include <algorithm>
#include <cstring>
#include <vector>

#include "bem_internal.cuh"

namespace bem {

constexpr int TC_BN = 128;           // pairs per MMA tile (N)
constexpr int TC_K = TC_TABLE_DIM;   // padded coefficients (K and M)
constexpr int TC_KB = 32;            // K-block: one 128-byte swizzled row of TF32 values
constexpr int TC_NKB = TC_K / TC_KB; // K-blocks per tile
constexpr int TC_TMEM_COLS = 512;    // A hi [0,128), A lo [128,256), 2 accumulators of 128
constexpr int TC_A_HI = 0, TC_A_LO = 128, TC_D0 = 256;
constexpr int TC_CHUNKS_PER_ITEM = 16;  // 64-pair chunks per work item (8 tiles)
constexpr long long TC_WAIT_CYCLES = 2000000000ll;  // about one second of SM clock

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor of a K-major operand with the 128-byte
// swizzle: start address, 8-row groups 1024 B apart (stride byte offset),
// descriptor version 1, swizzle mode 2 (128 B).  The leading byte offset is
// not used: one MMA reads 8 TF32 values (32 B) of a row, inside one swizzle
// row; the K-steps inside a K-block advance the start address by 32 B.
__device__ __forceinline__ uint64_t tc_desc_sw128(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor: D f32, A and B tf32, both K-major, N = 128, M = 128.
constexpr uint32_t TC_IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(TC_BN >> 3) << 17) |
                              ((uint32_t)(128 >> 4) << 24);

// x as the sum of two TF32 values (11 significant bits each), both the nearest
// with ties away from zero, bit for bit what cvt.rna.tf32.f32 gives for x and
// for x - h.  The tie rule is not free: the rest has at most 13 significant
// bits, so a quarter of all values tie, and rounding those to even moved the
// mean of a product by 1.7e-8 and of an energy by up to 8e-9 (four times what
// it moves from call to call).  Integer arithmetic runs on pipes that this
// kernel leaves idle (with cvt.rna k_m2l_tc took 106 us, against 70, on 81,920
// panels).  The last step keeps NaN and infinity, whose rest is NaN and could
// wrap to zero in the integer rounding.
__device__ __forceinline__ void split_tf32(float x, uint32_t &h, uint32_t &l) {
    h = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
    const float r = x - __uint_as_float(h);
    const float t = __uint_as_float((__float_as_uint(r) + 0x1000u) & 0xffffe000u);
    l = __float_as_uint(__fmaf_rn(r, 0.f, t));
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(phase)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t phase,
                                                  long long budget = TC_WAIT_CYCLES) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, phase))
        if (clock64() - t0 > budget) return false;
    return true;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

// D += A (tensor memory) . B (shared-memory descriptor)
__device__ __forceinline__ void tc_mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
        "r"(a), "l"(b), "r"(TC_IDESC), "r"(acc));
}

// Warp roles of the pipelined kernel.
constexpr int TC_NS = 5;                       // B stages: one K-block of a tile, hi | lo (32 KB)
constexpr int TC_STAGE_BYTES = 2 * TC_BN * TC_KB * 4;
constexpr int TC_ND = 2;                       // TMEM accumulators of TC_BN columns
constexpr int TC_RING = 16;                    // work items in flight between the roles
constexpr int TC_WARP_MMA = 0;                 // lane 0 issues the MMAs
constexpr int TC_WARP_EPI0 = 1;                // warps 1..4: epilogue (TMEM lane quadrant = warp % 4)
constexpr int TC_WARP_PROD0 = 5;               // warps 5..12: staging of B, operator into TMEM
constexpr int TC_NPROD = 8 * 32, TC_NEPI = 4 * 32;
constexpr int TC_THREADS = 13 * 32;
constexpr int TC_ROWS_PER_PROD = TC_BN * 8 / TC_NPROD;  // rows of a stage per producer thread (8 granules each)

__device__ __forceinline__ void bulk_prefetch_l2(const void *g, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(g), "r"(bytes) : "memory");
}

// The persistent kernel: one CTA per SM takes work items (offset class,
// first pair, number of pairs: up to 8 tiles of 128 pairs) from a global
// counter, largest first.  Tiles are numbered continuously across a CTA's
// items and each tile passes through nkb stages (one per K-block of 32
// coefficients: 4 at p = 10, 2 at p = 6), so the pipeline never drains between
// items:
//  * producers (warps 5-12): the leader fetches the next item, publishes it
//    in a shared ring (mbarrier itemFull) and prefetches its operator into
//    L2; all 256 hold a whole tile of multipoles in registers (FP32, 4 rows x
//    16 bytes per K-block and thread): each K-block is split into its TF32 hi
//    and lo parts and stored to stage g % TC_NS in the 128-byte swizzle
//    (mbarrier fullB), and its registers are loaded with the next tile's
//    K-block at once, a tile of time ahead.  After the first tile of an item
//    they wait for the last MMA of the previous item (aFree) and write the
//    item's operator into tensor memory (aReady), split the same way.  (A
//    barrier of its own: a parity wait must not run two phases ahead, and with
//    one K-block a tile the producers are several tiles ahead of fullD.)
//  * MMA (warp 0, lane 0): per item waits aReady; per tile waits a free
//    accumulator (emptyD), per K-block its stage (fullB), issues its K-steps x
//    3 products with A from tensor memory and commits to emptyB; after the
//    last K-block it commits to fullD, after an item's last tile to aFree.
//  * epilogue (warps 1-4): reads its TMEM lane quadrant, frees the
//    accumulator, transposes the tile into shared memory rows (one local
//    expansion row of cs floats per pair), then adds every row into its target
//    cell of `out` by one bulk reduction.
// What bounds it, on 2.7M pairs (81,920-panel molecules, 27 of them; 461 us, 6.7k
// cycles a tile): nothing alone.  Without the reductions 424, operator writes
// 428, two of the three MMAs 395, stores to the stages 371, with nothing but
// the MMAs 348 us: the MMAs issue at 106 cycles each (5.1k a tile).  Multipoles
// split beforehand (1 KB a pair, copied) took 514 us and a split kernel;
// reductions by vector instructions 512.  An FP16 split in three products with
// scaled operands, half the MMAs, took 479: the tiles then wait for copies and
// reductions, 128 KB of L2 traffic each.
__global__ void __launch_bounds__(TC_THREADS, 1)
k_m2l_tc(const float *__restrict__ A_all,
         const int4 *__restrict__ items, int nitems, int *__restrict__ next_item,
         const int *__restrict__ p_out, const int *__restrict__ p_in, int nc, int cs,
         const float *__restrict__ M, float *__restrict__ out, int *__restrict__ err,
         long long budget) {
    const int nkb = (nc + TC_KB - 1) / TC_KB;  // K-blocks that hold coefficients
    extern __shared__ __align__(1024) unsigned char smraw[];
    // 1024-byte aligned base (the 128-byte swizzle repeats every 1024 B)
    unsigned char *sm = smraw + ((1024u - (smem_u32(smraw) & 1023u)) & 1023u);
    const uint32_t sbase = smem_u32(sm);
    float *Ct = reinterpret_cast<float *>(sm + (size_t)TC_NS * TC_STAGE_BYTES);  // [TC_BN][cs]
    __shared__ __align__(8) uint64_t fullB[TC_NS], emptyB[TC_NS], fullD[TC_ND], emptyD[TC_ND];
    __shared__ __align__(8) uint64_t aReady, aFree, itemFull[TC_RING];
    __shared__ int4 s_item[TC_RING];
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < TC_NS; ++i) {
            mbar_init(smem_u32(&fullB[i]), TC_NPROD);
            mbar_init(smem_u32(&emptyB[i]), 1);
        }
        for (int i = 0; i < TC_ND; ++i) {
            mbar_init(smem_u32(&fullD[i]), 1);
            mbar_init(smem_u32(&emptyD[i]), TC_NEPI);
        }
        mbar_init(smem_u32(&aReady), TC_NPROD);
        mbar_init(smem_u32(&aFree), 1);
        for (int i = 0; i < TC_RING; ++i) mbar_init(smem_u32(&itemFull[i]), 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tm = s_tmem;
    // (An ordinary launch: as a programmatic dependent of the last M2M level its
    // CTAs would hold their SMs, idle, until that level ends: 8 uneven
    // molecules at once 10.17 against 10.57 ms.)
    int ntile_done = 0;  // tiles whose MMAs were all issued (MMA thread)
    int nitem_done = 0;  // items whose MMAs were all issued (MMA thread)
    int nstage_done = 0; // K-block stages whose MMAs were issued and committed (MMA thread)

    if (warp >= TC_WARP_PROD0) {
        // ---------------- producers
        const int ptid = tid - TC_WARP_PROD0 * 32;
        const int pw = ptid >> 5;                            // producer warp 0..7
        const int quad = warp & 3, row = 32 * quad + lane;  // TMEM lane of this thread
        const int gq = lane & 7, r4 = lane >> 3;            // 16-byte granule, row within a group of 4
        // every wait is made warp-uniform (__all_sync) and every item starts with
        // a vote of all producers, so that on a timeout they leave together
        bool fail = false;
        int t = 0;
        for (int i = 0;; ++i) {
            const int slot = i % TC_RING;
            uint32_t all_ok;
            asm volatile(
                "{\n .reg .pred p, q;\n setp.eq.u32 p, %1, 0;\n bar.red.and.pred q, 2, %2, p;\n"
                " selp.u32 %0, 1, 0, q;\n}\n"
                : "=r"(all_ok)
                : "r"((uint32_t)fail), "n"(TC_NPROD));
            if (!all_ok) break;
            if (ptid == 0) {
                const int idx = atomicAdd(next_item, 1);
                const int4 it = idx < nitems ? items[idx] : make_int4(-1, 0, 0, 0);
                if (it.x >= 0) {
                    bulk_prefetch_l2(A_all + (size_t)it.x * TC_K * TC_K, TC_K * TC_K * 4);
                }
                s_item[slot] = it;
                mbar_arrive(smem_u32(&itemFull[slot]));
            }
            asm volatile("bar.sync 2, %0;" ::"n"(TC_NPROD) : "memory");
            const int4 sc = s_item[slot];
            if (sc.x < 0) break;
            const int ntl = (sc.z + TC_BN - 1) / TC_BN;
            // source cells of the tile rows this thread stages
            auto load_srcs = [&](int c, int *dst) {
                const int y = sc.y + TC_BN * c, z = min(TC_BN, sc.z - TC_BN * c);  // z <= 0 past the item
#pragma unroll
                for (int i = 0; i < TC_ROWS_PER_PROD; ++i) {
                    const int n = 4 * TC_ROWS_PER_PROD * pw + 4 * i + r4;
                    dst[i] = (n < z) ? p_in[y + n] : -1;
                }
            };
            // K-block kb of the tile whose source cells are src, FP32; zero beyond
            // the coefficients (a row's padding is not initialised)
            float4 v[TC_NKB][TC_ROWS_PER_PROD];
            auto load_kb = [&](int kb, const int *src) {
                const int k0 = TC_KB * kb + 4 * gq;
#pragma unroll
                for (int i = 0; i < TC_ROWS_PER_PROD; ++i) {
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (src[i] >= 0 && k0 < nc) x = __ldcg(reinterpret_cast<const float4 *>(M + (size_t)src[i] * cs + k0));
                    v[kb][i] = x;
                }
            };
            int nxt[TC_ROWS_PER_PROD];
            load_srcs(0, nxt);
#pragma unroll
            for (int kb = 0; kb < TC_NKB; ++kb) load_kb(kb, nxt);
            load_srcs(1, nxt);
            for (int c = 0; c < ntl; ++c, ++t) {
#pragma unroll
                for (int kb = 0; kb < TC_NKB; ++kb) {
                    if (kb >= nkb || fail) continue;
                    const int g = nkb * t + kb;
                    const int st = g % TC_NS, k = g / TC_NS;
                    const bool okB = __all_sync(0xffffffffu, k < 1 || mbar_wait_bounded(smem_u32(&emptyB[st]),
                                                                                       (uint32_t)((k - 1) & 1), budget));
                    if (!okB) {
                        atomicExch(err, 1);
                        fail = true;
                        continue;
                    }
                    unsigned char *bh = sm + (size_t)st * TC_STAGE_BYTES, *bl = bh + TC_BN * TC_KB * 4;
                    const int left = nc - (TC_KB * kb + 4 * gq);  // coefficients from this granule on
#pragma unroll
                    for (int i = 0; i < TC_ROWS_PER_PROD; ++i) {
                        const int n = 4 * TC_ROWS_PER_PROD * pw + 4 * i + r4;
                        const float x[4] = {v[kb][i].x, left > 1 ? v[kb][i].y : 0.f, left > 2 ? v[kb][i].z : 0.f,
                                            left > 3 ? v[kb][i].w : 0.f};
                        uint4 h, l;
                        split_tf32(x[0], h.x, l.x);
                        split_tf32(x[1], h.y, l.y);
                        split_tf32(x[2], h.z, l.z);
                        split_tf32(x[3], h.w, l.w);
                        const uint32_t off = (uint32_t)(n * 128 + ((gq ^ (n & 7)) << 4));
                        *reinterpret_cast<uint4 *>(bh + off) = h;
                        *reinterpret_cast<uint4 *>(bl + off) = l;
                    }
                    // the stage was written through the generic proxy: order it before
                    // the tensor core's (async proxy) reads
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    mbar_arrive(smem_u32(&fullB[st]));
                    if (c > 0 && c + 1 < ntl) load_kb(kb, nxt);
                }
                if (fail) break;
                if (c == 0) {
                    // the item's operator into tensor memory, once the previous
                    // item's MMAs (which read the old one) have completed
                    const bool okA = __all_sync(0xffffffffu, i < 1 || mbar_wait_bounded(smem_u32(&aFree),
                                                                                       (uint32_t)((i - 1) & 1), budget));
                    if (!okA) {
                        atomicExch(err, 1);
                        fail = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    // operator layout [k / 4][row][k % 4]: the warp's rows read 512
                    // contiguous bytes per load; 16 coefficients at a time, each
                    // split into its TF32 hi part and the TF32 rest (the 3xTF32
                    // operands) and stored to both halves of the operator's columns
                    const float4 *ga = reinterpret_cast<const float4 *>(A_all + (size_t)sc.x * TC_K * TC_K) + row;
#pragma unroll 2
                    for (int part = pw >> 2; part < 2 * nkb; part += 2) {  // two warps per lane quadrant
                        const float4 *gp = ga + part * 4 * TC_K;
                        uint32_t vh[16], vl[16];
#pragma unroll
                        for (int q = 0; q < 16; q += 4) {
                            const float4 f = __ldg(gp + (q >> 2) * TC_K);
                            const float x[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) split_tf32(x[e], vh[q + e], vl[q + e]);
                        }
#pragma unroll
                        for (int hl = 0; hl < 2; ++hl) {
                            const uint32_t *w = hl ? vl : vh;
                            asm volatile(
                                "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
                                "%15,%16};" ::"r"(tm + ((uint32_t)(32 * quad) << 16) +
                                                  (uint32_t)(hl ? TC_A_LO : TC_A_HI) + (uint32_t)(16 * part)),
                                "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]),
                                "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]),
                                "r"(w[15]));
                        }
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    mbar_arrive(smem_u32(&aReady));
                    // the second tile: its latency passes under the first tile's MMAs
                    if (ntl > 1) {
#pragma unroll
                        for (int kb = 0; kb < TC_NKB; ++kb) load_kb(kb, nxt);
                    }
                }
                load_srcs(c + 2, nxt);  // needed after the next tile's first stage
            }
        }
    } else if (warp == TC_WARP_MMA) {
        // ---------------- MMA issue (one thread)
        if (lane == 0) {
            bool fail = false;
            int t = 0;
            for (int i = 0; !fail; ++i) {
                const int slot = i % TC_RING;
                if (!mbar_wait_bounded(smem_u32(&itemFull[slot]), (uint32_t)((i / TC_RING) & 1), budget)) {
                    atomicExch(err, 1);
                    break;
                }
                const int4 sc = s_item[slot];
                if (sc.x < 0) break;
                if (!mbar_wait_bounded(smem_u32(&aReady), (uint32_t)(i & 1), budget)) {
                    atomicExch(err, 1);
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const int ntl = (sc.z + TC_BN - 1) / TC_BN;
                for (int c = 0; c < ntl && !fail; ++c, ++t) {
                    const int d = t % TC_ND, jd = t / TC_ND;
                    if (jd >= 1 && !mbar_wait_bounded(smem_u32(&emptyD[d]), (uint32_t)((jd - 1) & 1), budget)) {
                        atomicExch(err, 1);
                        fail = true;
                        break;
                    }
                    const uint32_t dt = tm + (uint32_t)(TC_D0 + d * TC_BN);
                    for (int kb = 0; kb < nkb; ++kb) {
                        const int g = nkb * t + kb;
                        const int st = g % TC_NS, k = g / TC_NS;
                        if (!mbar_wait_bounded(smem_u32(&fullB[st]), (uint32_t)(k & 1), budget)) {
                            atomicExch(err, 1);
                            fail = true;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;");
                        const uint32_t bh = sbase + (uint32_t)(st * TC_STAGE_BYTES);
                        const uint32_t bl = bh + TC_BN * TC_KB * 4;
#pragma unroll
                        for (int ks = 0; ks < TC_KB / 8; ++ks) {
                            const uint64_t dbh = tc_desc_sw128(bh + 32u * ks), dbl = tc_desc_sw128(bl + 32u * ks);
                            const uint32_t kc = (uint32_t)(TC_KB * kb + 8 * ks);
                            tc_mma_ts(dt, tm + TC_A_HI + kc, dbh, (kb | ks) ? 1u : 0u);
                            tc_mma_ts(dt, tm + TC_A_HI + kc, dbl, 1u);
                            tc_mma_ts(dt, tm + TC_A_LO + kc, dbh, 1u);
                        }
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                         smem_u32(&emptyB[st]))
                                     : "memory");
                        nstage_done = g + 1;
                    }
                    if (fail) break;
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     smem_u32(&fullD[d]))
                                 : "memory");
                    if (c == ntl - 1)  // the item's MMAs all issued: its operator is free when they end
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                         smem_u32(&aFree))
                                     : "memory");
                }
                if (!fail) nitem_done = i + 1;
            }
            ntile_done = t;
        }
    } else {
        // ---------------- epilogue: TMEM lane quadrant (warp % 4), 128 pairs per tile
        const int quad = warp & 3;
        const int row = 32 * quad + lane;
        const int etid = tid - TC_WARP_EPI0 * 32;  // 0 .. TC_NEPI - 1
        bool fail = false;
        int t = 0;
        for (int i = 0; !fail; ++i) {
            const int slot = i % TC_RING;
            const bool okI = mbar_wait_bounded(smem_u32(&itemFull[slot]), (uint32_t)((i / TC_RING) & 1), budget);
            uint32_t all_ok;
            asm volatile(
                "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n"
                " selp.u32 %0, 1, 0, q;\n}\n"
                : "=r"(all_ok)
                : "r"((uint32_t)okI), "n"(TC_NEPI));
            if (!all_ok) {
                atomicExch(err, 1);
                break;
            }
            const int4 sc = s_item[slot];
            if (sc.x < 0) break;
            const int ntl = (sc.z + TC_BN - 1) / TC_BN;
            for (int c = 0; c < ntl; ++c, ++t) {
                const int d = t % TC_ND, jd = t / TC_ND;
                const bool ok = mbar_wait_bounded(smem_u32(&fullD[d]), (uint32_t)(jd & 1), budget);
                // the four epilogue warps leave together (they meet at named barriers below)
                asm volatile(
                    "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n"
                    " selp.u32 %0, 1, 0, q;\n}\n"
                    : "=r"(all_ok)
                    : "r"((uint32_t)ok), "n"(TC_NEPI));
                if (!all_ok) {
                    atomicExch(err, 1);
                    fail = true;
                    break;
                }
                // the previous tile's reductions have read Ct
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                asm volatile("bar.sync 1, %0;" ::"n"(TC_NEPI) : "memory");
                asm volatile("tcgen05.fence::after_thread_sync;");
                const int y = sc.y + TC_BN * c, z = min(TC_BN, sc.z - TC_BN * c);
                const int tgt = etid < z ? p_out[y + etid] : -1;
#pragma unroll 1
                for (int cg = 0; cg < TC_BN; cg += 32) {
                    uint32_t r[32];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
                          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
                          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                        : "r"(tm + ((uint32_t)(32 * quad) << 16) + (uint32_t)(TC_D0 + d * TC_BN + cg)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (row < cs) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) Ct[(cg + j) * cs + row] = __uint_as_float(r[j]);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                mbar_arrive(smem_u32(&emptyD[d]));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("bar.sync 1, %0;" ::"n"(TC_NEPI) : "memory");
                // every pair's row added into its target cell by one bulk reduction
                if (tgt >= 0)
                    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(
                                     out + (size_t)tgt * cs),
                                 "r"(smem_u32(Ct + etid * cs)), "r"((nc + 3) / 4 * 16)
                                 : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    // before the CTA's shared memory and tensor memory go away, every commit
    // arrival must have landed: the MMA thread waits (bounded) for the last
    // completion of each B stage (which follows all MMAs issued before it,
    // also those of a tile left unfinished by a failed wait) and of the last
    // accumulator and operator release
    if (warp == TC_WARP_MMA && lane == 0 && nstage_done > 0) {
        const int ng = nstage_done;
        for (int st = 0; st < TC_NS && st < ng; ++st) {
            const int g = st + ((ng - 1 - st) / TC_NS) * TC_NS;  // last stage use on st
            mbar_wait_bounded(smem_u32(&emptyB[st]), (uint32_t)((g / TC_NS) & 1));
        }
        if (ntile_done > 0) {
            const int t = ntile_done - 1;
            mbar_wait_bounded(smem_u32(&fullD[t % TC_ND]), (uint32_t)((t / TC_ND) & 1));
        }
        if (nitem_done > 0) mbar_wait_bounded(smem_u32(&aFree), (uint32_t)((nitem_done - 1) & 1));
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(TC_TMEM_COLS));
}

// ---------------------------------------------------------------- host side
bool tc_m2l_available(const Mesh &m) {
    return m.opt.precision == BEM_MIXED && (m.opt.p + 1) * (m.opt.p + 1) <= TC_K;
}

// dynamic shared memory: alignment slack, the B stages, the transposed tile
size_t tc_smem_bytes() { return 1024 + (size_t)TC_NS * TC_STAGE_BYTES + (size_t)TC_BN * TC_K * sizeof(float); }

// Work items of the persistent kernel: (offset class, first pair, number of
// pairs), up to TC_CHUNKS_PER_ITEM consecutive 64-pair chunks of one class
// (tiles of 128 pairs), largest first.
std::vector<int4> tc_items(const std::vector<int4> &chunks_m2l) {
    std::vector<int4> sup;
    int i = 0;
    const int n = (int)chunks_m2l.size();
    while (i < n) {  // chunks of one class cover consecutive pairs
        int j = i + 1, np = chunks_m2l[i].z;
        while (j < n && j - i < TC_CHUNKS_PER_ITEM && chunks_m2l[j].x == chunks_m2l[i].x) np += chunks_m2l[j++].z;
        sup.push_back(make_int4(chunks_m2l[i].x, chunks_m2l[i].y, np, 0));
        i = j;
    }
    std::stable_sort(sup.begin(), sup.end(), [](const int4 &a, const int4 &b) { return a.z > b.z; });
    return sup;
}

// L (levels >= 2, cleared by the pass) += sum over the M2L pairs of T_o M_s.
void m2l_tc(Mesh &m, const Tree &t, const Tree::M2LPairs &g, const float *M, float *L, bool timed) {
    const Tables &tb = tables_for(m, t);
    const int nc = (m.opt.p + 1) * (m.opt.p + 1);
    const int cs = cell_stride(m);
    if (g.nsuper == 0) return;
    const bool tk = timed && m.tm.on && m.tm.kev[0];
    auto kev = [&](int k) {
        if (tk) BEM_CUDA(cudaEventRecord(m.tm.kev[k], m.stream));
    };
    kev(0);
    if (cs % 4 != 0) throw Error(BEM_ECUDA, "tensor-core staging: cell stride not a multiple of 4");
    const size_t sm = tc_smem_bytes();
    int dev = 0, nsm = 0;
    BEM_CUDA(cudaGetDevice(&dev));
    BEM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int grid = std::max(1, std::min(g.nsuper, nsm));
    kev(1);
    ensure_smem_attr(reinterpret_cast<const void *>(k_m2l_tc), sm);
    k_m2l_tc<<<grid, TC_THREADS, sm, m.stream>>>(tb.Tc_f.p, g.super.p, g.nsuper, m.dev_err.p + 1, g.out.p,
                                                 g.in.p, nc, cs, M, L, m.dev_err.p, m.wait_budget);
    BEM_CHECK_LAUNCH();
    kev(2);
    kev(3);
}

}  // namespace bem
