// Multi-right-hand-side HMVM on the fifth-generation tensor cores: Y = H X for k slip-rate
// vectors at once (Eq. 20 applied to k inputs).
//
// With one right-hand side the product performs one FMA per stored entry and is bound by
// HBM; with k of them every stored entry feeds k FMAs, so from k of about 16 up the product
// needs more arithmetic than the CUDA cores give at full bandwidth, and it becomes a dense
// contraction that belongs on the tensor cores.  Both phases of Eq. 20 are batched GEMMs:
//   V^T phase: for each column group (low-rank blocks sharing a column cluster), the stacked
//              V^T rows (ranks x group columns) times the group's slice of X;
//   UY phase:  for each leaf row unit, its row panel [dense near-field | U of the low-rank
//              blocks] times the gathered [X | T] rows.
// A = the stored panel (FP16, per-column power-of-two scales as in the 2-byte storage; the
// FP32 near field of HBI_MIXED as an FP16 pair hi + 2^-11 lo), packed at build time in the
// canonical no-swizzle K-major tcgen05 layout (8 x 8 core matrices of 128 contiguous bytes),
// in chunks of MR_CW columns, so that one cp.async.bulk lands a chunk in shared memory ready
// for the MMA.  B = the input rows, scaled per right-hand side to FP16 range and split into
// hi + 2^-11 lo FP16 parts (22 significant bits) once per row (mr_split_kernel), [hi | lo] of one
// row side by side; a chunk's rows are fetched by index with 16-byte asynchronous copies straight
// into the swizzled MN-major layout the MMA reads.  The MMA (kind::f16, M = 128 panel rows,
// K = 16) accumulates in FP32 in tensor memory: D1 = A_hi B_hi and D2 = A_hi B_lo + A_lo B_hi;
// y = (D1 + 2^-11 D2) / s.
//
// Persistent CTAs, warp-specialised: one thread streams the A pieces into a ring of
// shared-memory stages (bulk copies on mbarriers), four warps gather the B chunks into a second
// ring, one warp allocates tensor memory and issues the MMAs, releasing each stage with
// tcgen05.commit, and four warps run the epilogue (tcgen05.ld, one TMEM lane per panel row)
// from one of two accumulators while the next task's MMAs fill the other.
// Every wait is bounded; a CTA that gives up raises the error flag, lets its copies and MMAs
// in flight finish and frees its tensor memory.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <type_traits>
#include <vector>

#include "hbi_internal.h"

namespace hbi {

constexpr int MR_CW = 64;                          // K columns per chunk
// Ring stages of A (a panel piece of 16 KB each) and of B (MR_CW rows of 4 kp bytes): what lets two
// CTAs share an SM, so that one's epilogue and waits run beside the other's MMAs (64 right-hand
// sides at 40,000 elements, both phases: 316 us; one CTA with seven and six stages 420 us, two
// with three and three 346 us; 32 right-hand sides 260 us, three CTAs 294 us, one 363 us).
__host__ __device__ constexpr int mr_stages_a(int kp) { return kp == 64 ? 4 : 5; }
__host__ __device__ constexpr int mr_stages_b(int kp) { return kp == 16 ? 6 : 3; }
constexpr int MR_GW = 4;                           // epilogue warps (TMEM lanes 0..127)
constexpr int MR_BW = 4;                           // B producer warps
static_assert(mr_stages_a(16) >= 2 && mr_stages_a(32) >= 2 && mr_stages_a(64) >= 2,
              "a dense chunk with a lo part holds two A stages");
constexpr int MR_THREADS = 32 * (MR_GW + 2 + MR_BW);   // epilogue, A producer, MMA and B producer warps
constexpr int MR_ROWS = 128;                       // MMA M: panel rows of a task
constexpr int MR_A_STAGE = MR_ROWS * MR_CW * 2;    // bytes: one part (hi or lo) of a 128-row chunk
constexpr int MR_KP_MAX = 64;                      // right-hand sides per call (padded to 16, 32 or 64)
constexpr int MR_ZERO = 2 * MR_KP_MAX;             // halves before row 0 of x16: row -1 is zeros, whatever the row length
constexpr int MR_KSLICE = 2048;                    // V^T: widest K of one task (wider groups are cut)
constexpr unsigned long long MR_WAIT_NS = 1000000000ull;   // 1 s

// One task: rows [0, rows) of one panel (a 128-row slice of a column group's V^T rows or of
// a leaf row unit).  Its K columns are kd dense columns (hi and, if lo, lo parts) followed by
// kl factor columns (U or V^T), each segment a multiple of 16 and cut into chunks of MR_CW.
struct MrTask {
    int64_t a_off;     // byte offset of the first chunk in the panel stream
    int64_t g_off;     // offset of the task's B row indices (MR_CW per chunk)
    int64_t out_off;   // first output row (V^T: row of T inside xt; UY: row of yp)
    int64_t s_off;     // V^T: rowscale index of row 0; UY: -1
    int rows;          // 1..128
    int kd, kl;        // dense and factor columns (multiples of 16)
    int kreal;         // V^T: the group's columns (the padding gathers zeros)
    int lo;            // the dense chunks carry a lo part
    int partial;       // V^T: a K slice of a wide column group; its rows are partial sums
};

// A V^T row tile of a wide column group, cut into nsl K slices: slice q wrote its partial rows
// (already scaled) at xt rows p_row + q MR_ROWS; their sum in slice order is t.
struct MrSplit {
    int64_t t_row, p_row;
    int rows, nsl;
};

}  // namespace hbi

// Everything the handle keeps for the multi-RHS product.
struct hbi::MultiRhs {
    unsigned char *d_panels = nullptr;
    int64_t panel_bytes = 0;
    MrTask *d_vt = nullptr, *d_uy = nullptr;
    int n_vt = 0, n_uy = 0;
    MrSplit *d_split = nullptr;   // V^T row tiles cut along K (reduced after the V^T phase)
    int n_split = 0;
    int64_t n_prow = 0;           // partial rows after T in xt
    int *d_bidx = nullptr;        // B row indices of every task's chunks (rows of x16; padding: -1, its row of zeros)
    float *d_cscale = nullptr;    // per X row: the scale of its dense columns (largest over the blocks)
    int *d_iperm = nullptr;       // original element -> permuted position
    float *d_rowscale = nullptr;  // V^T output row scales (sv su)
    int64_t n_t = 0;              // rows of T
    int64_t nx = 0;               // rows of X (n_in N)
    int lo = 0;
    int grid = 0;
    // per-call buffers, sized for kp_cap right-hand sides
    int kp_cap = 0;
    float *d_xt = nullptr, *d_yp = nullptr;
    __half *d_x16 = nullptr;      // MR_ZERO zeros, then rows of X, of X with the dense column scales and of T, each [hi | lo]
    int row_kp = 0;               // the row length the grid is for
    unsigned *d_vmax = nullptr;   // per right-hand side: [0, 64) max |x|, [64, 128) max |t|,
                                  // [128, 192) max |x| x its row's dense column scale
    int *h_err = nullptr;         // error flag of bounded device waits (pinned; the kernels write it)
    int64_t bytes_panels_alg = 0;     // stored entries (hi + lo for the FP32 near field) + scales
    int64_t vec_bytes_per_rhs = 0;    // x read, t written and read, y written (FP32)
    double flops_per_rhs = 0;         // 2 x (dense + U + V entries)
    double mma_flops_per_rhs = 0;     // as issued (padding, hi / lo passes)
};

namespace hbi {
namespace {

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ unsigned mr_smem(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long mr_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mr_bar_init(uint64_t *b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mr_smem(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mr_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mr_smem(b)) : "memory");
}
__device__ __forceinline__ void mr_expect_tx(uint64_t *b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mr_smem(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mr_try(uint64_t *b, unsigned parity) {
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(mr_smem(b)), "r"(parity)
                 : "memory");
    return ok != 0;
}
// One thread waits for the phase of the given parity; false once *fail is set or after MR_WAIT_NS.
__device__ __forceinline__ bool mr_wait(uint64_t *b, unsigned parity, volatile int *fail) {
    if (mr_try(b, parity)) return true;   // already complete: no timer read
    const unsigned long long t0 = mr_ns();
    for (unsigned it = 0;; ++it) {
        if (mr_try(b, parity)) return true;
        if ((it & 63u) == 63u && (*fail || mr_ns() - t0 > MR_WAIT_NS)) {
            *fail = 1;
            return false;
        }
    }
}
// The same for a whole warp, with a warp-uniform outcome.
__device__ __forceinline__ bool mr_warp_wait(uint64_t *b, unsigned parity, volatile int *fail) {
    if (__all_sync(0xffffffffu, mr_try(b, parity))) return true;   // already complete: no timer read
    const unsigned long long t0 = mr_ns();
    for (unsigned it = 0;; ++it) {
        if (__all_sync(0xffffffffu, mr_try(b, parity))) return true;
        if ((it & 63u) == 63u && __any_sync(0xffffffffu, *fail != 0 || mr_ns() - t0 > MR_WAIT_NS)) {
            *fail = 1;
            return false;
        }
    }
}
__device__ __forceinline__ void mr_bulk(void *dst, const void *src, unsigned bytes, uint64_t *b) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     mr_smem(dst)),
                 "l"(src), "r"(bytes), "r"(mr_smem(b))
                 : "memory");
}
__device__ __forceinline__ void mr_copy16(unsigned dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// arrives on the barrier once the thread's copies so far have landed
__device__ __forceinline__ void mr_copy_arrive(uint64_t *b) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(mr_smem(b)) : "memory");
}
// Shared-memory matrix descriptor: start address, LBO and SBO byte strides, version 1 (bits
// 46-47), swizzle mode (bits 61-63: 0 none, 2 128-byte, 4 64-byte).  No swizzle, K-major: LBO
// between core matrices along K, SBO between 8-row groups.  Swizzled, MN-major: LBO between
// atoms along N (one swizzle row of N elements each), SBO between groups of 8 K rows.
__device__ __forceinline__ uint64_t mr_desc(unsigned saddr, unsigned lbo, unsigned sbo, unsigned swizzle) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46) | ((uint64_t)swizzle << 61);
}
__device__ __forceinline__ void mr_mma(unsigned d_tmem, uint64_t a, uint64_t b, unsigned idesc, unsigned acc) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
                 "l"(a), "l"(b), "r"(idesc), "r"(acc)
                 : "memory");
}
__device__ __forceinline__ void mr_commit(uint64_t *b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mr_smem(b))
                 : "memory");
}
__device__ __forceinline__ void mr_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void mr_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void mr_ld16(unsigned taddr, float *v) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}
__device__ __forceinline__ void mr_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Chunk c of a task: dense or factor, its first column in the task's K, width, bytes of one
// part, parts (a dense chunk with a lo part holds its hi part, then its lo part) and offset.
struct MrChunk {
    int dense, col0, w, parts;
    unsigned bytes;   // of one part
    int64_t off;
};
__device__ __forceinline__ int mr_nchunks(const MrTask &t) { return (t.kd + MR_CW - 1) / MR_CW + (t.kl + MR_CW - 1) / MR_CW; }
__device__ __forceinline__ MrChunk mr_chunk(const MrTask &t, int c) {
    const int rg = (t.rows + 7) / 8, parts = 1 + t.lo;
    const int nchd = (t.kd + MR_CW - 1) / MR_CW;
    MrChunk k;
    if (c < nchd) {
        k.dense = 1;
        k.col0 = c * MR_CW;
        k.w = min(MR_CW, t.kd - k.col0);
        k.off = t.a_off + (int64_t)c * rg * MR_CW * 16 * parts;
        k.parts = parts;
    } else {
        const int cu = c - nchd;
        k.dense = 0;
        k.col0 = t.kd + cu * MR_CW;
        k.w = min(MR_CW, t.kl - cu * MR_CW);
        k.off = t.a_off + (int64_t)rg * t.kd * 16 * parts + (int64_t)cu * rg * MR_CW * 16;
        k.parts = 1;
    }
    k.bytes = (unsigned)(rg * k.w * 16);
    return k;
}

// Power of two s with max |v| s in (2^13, 2^14] (1 for 0): keeps the scaled B operand, whose
// largest entry is m s, inside FP16 range with the most significant bits.
__device__ __forceinline__ float mr_scale_for(float m) {
    if (!(m > 0.0f) || !isfinite(m)) return 1.0f;
    int e;
    const float f = frexpf(m, &e);   // m = f 2^e, f in [0.5, 1)
    const int c = f == 0.5f ? e - 1 : e;   // ceil(log2 m)
    return ldexpf(1.0f, 14 - c);
}

// The scale of right-hand side r: of the V^T phase from max |x|, of the UY phase from the larger of
// max |x| with the dense column scales and max |t|.
__device__ __forceinline__ float mr_phase_scale(const unsigned *vmax, int vt, int r) {
    const float m = vt ? __uint_as_float(vmax[r]) : fmaxf(__uint_as_float(vmax[128 + r]), __uint_as_float(vmax[64 + r]));
    return mr_scale_for(m);
}

// Rows [row0, row0 + nrows) of xt (KP FP32 words) times the phase's scales into x16 rows [hi | lo]:
// hi = fp16(b), lo = fp16((b - hi) 2^11), b = x s.  Eight right-hand sides a thread.  One pass over
// the inputs of a phase (bound by its traffic: 8 KP bytes a row) in place of a conversion of every
// gathered row in the product kernel, where each row serves several chunks.
template <int KP>
__global__ void mr_split_kernel(const float *xt, const unsigned *vmax, int vt, int64_t row0, int64_t nrows,
                                __half *x16) {
    constexpr int PER = KP / 8;   // threads a row
    pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int r0 = 8 * (int)(t0 % PER);   // stride is a multiple of PER
    float sc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) sc[q] = mr_phase_scale(vmax, vt, r0 + q);
    for (int64_t e = t0; e < nrows * PER; e += stride) {
        const int64_t row = row0 + e / PER;
        const float4 u = *reinterpret_cast<const float4 *>(xt + row * KP + r0);
        const float4 v = *reinterpret_cast<const float4 *>(xt + row * KP + r0 + 4);
        const float xs[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        __align__(16) __half hi[8], lo[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float b = xs[q] * sc[q];
            hi[q] = __float2half_rn(b);
            lo[q] = __float2half_rn((b - __half2float(hi[q])) * 2048.0f);
        }
        *reinterpret_cast<uint4 *>(x16 + row * 2 * KP + r0) = *reinterpret_cast<const uint4 *>(hi);
        *reinterpret_cast<uint4 *>(x16 + row * 2 * KP + KP + r0) = *reinterpret_cast<const uint4 *>(lo);
    }
}

// ------------------------------------------------------------------ the product kernel
// vt = 1: V^T phase (outputs T rows scaled by rowscale, max |t| per right-hand side into
// vmax[64 + r]); vt = 0: UY phase (outputs yp).  Warps 0-3 run the epilogue from one of two
// tensor-memory accumulators while the MMAs of the next task fill the other; warp 4 streams the A
// pieces (which depend on the operator alone, so it does not wait for the kernels before); warp
// 5 allocates tensor memory and issues the MMAs; warps 6-9 gather each chunk's B rows by index.
template <int KP>
__global__ void __launch_bounds__(MR_THREADS, 1)
    mr_kernel(const MrTask *__restrict__ tasks, int ntasks, int vt, const unsigned char *__restrict__ panels,
              const __half *x16, const int *__restrict__ bidx, const float *__restrict__ rowscale,
              float *out, unsigned *vmax, int *err) {
    constexpr int MR_SA = mr_stages_a(KP), MR_SB = mr_stages_b(KP);   // ring stages
    constexpr int ROWB = 4 * KP < 128 ? 4 * KP : 128;   // bytes of a K row in one swizzle atom
    constexpr int NATOM = 4 * KP / ROWB;                // atoms along N: one, or hi and lo for KP = 64
    constexpr int BATOM = MR_CW * ROWB;                 // bytes of an atom column of a chunk
    constexpr int BSTAGE = NATOM * BATOM;
    constexpr unsigned SWZ = ROWB == 128 ? 2u : 4u;
    constexpr unsigned TCOLS = 4 * KP <= 64 ? 64 : (4 * KP <= 128 ? 128 : 256);   // 2 accumulators x (D1 | D2)
    extern __shared__ __align__(1024) unsigned char mr_sm[];
    unsigned char *sA = mr_sm;                                        // MR_SA x MR_A_STAGE
    unsigned char *sB = sA + MR_SA * MR_A_STAGE;                      // MR_SB x BSTAGE
    __shared__ uint64_t a_full[MR_SA], a_empty[MR_SA], b_full[MR_SB], b_empty[MR_SB];
    __shared__ uint64_t acc_full[2], acc_empty[2], fin;
    __shared__ unsigned s_taddr;
    __shared__ float s_inv[KP];
    __shared__ unsigned s_tmax[KP];
    __shared__ volatile int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int W_PROD = MR_GW, W_MMA = MR_GW + 1, W_BPROD = MR_GW + 2;
    if (mr_smem(mr_sm) % 1024u != 0) {   // the swizzle goes by the address
        if (threadIdx.x == 0) *(volatile int *)err = 1;
        return;
    }

    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < MR_SA; ++s) { mr_bar_init(&a_full[s], 1); mr_bar_init(&a_empty[s], 1); }
        for (int s = 0; s < MR_SB; ++s) { mr_bar_init(&b_full[s], 32 * MR_BW); mr_bar_init(&b_empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mr_bar_init(&acc_full[s], 1); mr_bar_init(&acc_empty[s], 32 * MR_GW); }
        mr_bar_init(&fin, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < KP) s_tmax[threadIdx.x] = 0u;
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(mr_smem(&s_taddr)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    mr_fence_before();
    __syncthreads();
    mr_fence_after();
    const unsigned taddr = s_taddr;
    volatile int *fail = &s_fail;

    if (warp == W_PROD) {
        // ---------------------------------------------------------------- A producer (one lane)
        if (lane == 0) {
            unsigned g = 0;
            bool ok = true;
            MrTask tn;
            if (blockIdx.x < ntasks) tn = tasks[blockIdx.x];
            for (int ti = blockIdx.x; ti < ntasks && ok && !*fail; ti += gridDim.x) {
                const MrTask t = tn;
                if (ti + (int)gridDim.x < ntasks) tn = tasks[ti + gridDim.x];   // the next task, in flight
                const int nch = mr_nchunks(t);
                for (int c = 0; c < nch && ok; ++c) {
                    const MrChunk k = mr_chunk(t, c);
                    for (int p = 0; p < k.parts; ++p) {
                        const int s = g % MR_SA;
                        if (g >= (unsigned)MR_SA && !mr_wait(&a_empty[s], ((g / MR_SA) - 1) & 1, fail)) { ok = false; break; }
                        mr_expect_tx(&a_full[s], k.bytes);
                        mr_bulk(sA + (size_t)s * MR_A_STAGE, panels + k.off + (int64_t)p * k.bytes, k.bytes, &a_full[s]);
                        ++g;
                    }
                }
            }
            if (*fail) {   // let the copies in flight land before the CTA exits
                for (int s = 0; s < MR_SA; ++s) {
                    const unsigned uses = g / MR_SA + (s < (int)(g % MR_SA) ? 1u : 0u);
                    if (uses == 0) continue;
                    const unsigned long long t0 = mr_ns();
                    while (!mr_try(&a_full[s], (uses - 1) & 1) && mr_ns() - t0 < MR_WAIT_NS) {
                    }
                }
            }
        }
        pdl_wait();
    } else if (warp >= W_BPROD) {
        // ---------------------------------------------------------------- B producers
        // VPR threads copy a row (16 bytes each), so the 128 threads take RPS rows a step; a
        // thread's row indices of the next chunk are loaded ahead.  16-byte vector j of K row kc
        // goes to vector j ^ (kc mod 8) of its 128-byte swizzle row (64-byte rows: j ^ (kc / 2 mod
        // 4)).  Row-gathering bulk tensor copies (tile::gather4) in their place took 395 against
        // 193 us for the UY phase of 64 right-hand sides at 40,000 elements: about 90 cycles
        // per four 128-byte rows.
        constexpr int VPR = 4 * KP / 16, RPS = 32 * MR_BW / VPR, NST = MR_CW / RPS;
        const int bt = threadIdx.x - 32 * W_BPROD, brow = bt / VPR, v = bt % VPR;
        unsigned g = 0;
        bool ok = true;
        MrTask tn;
        if (blockIdx.x < ntasks) tn = tasks[blockIdx.x];
        int nxt[NST];
        auto load = [&](const MrTask &t, int c) {
#pragma unroll
            for (int u = 0; u < NST; ++u) nxt[u] = bidx[t.g_off + (int64_t)c * MR_CW + u * RPS + brow];
        };
        if (blockIdx.x < ntasks) load(tn, 0);
        pdl_wait();
        for (int ti = blockIdx.x; ti < ntasks && ok; ti += gridDim.x) {
            const MrTask t = tn;
            const bool more = ti + (int)gridDim.x < ntasks;
            if (more) tn = tasks[ti + gridDim.x];
            const int nch = mr_nchunks(t);
            for (int c = 0; c < nch; ++c, ++g) {
                int r[NST];
#pragma unroll
                for (int u = 0; u < NST; ++u) r[u] = nxt[u];
                if (c + 1 < nch) load(t, c + 1);
                else if (more) load(tn, 0);
                const int w = mr_chunk(t, c).w;
                const int s = g % MR_SB;
                if (g >= (unsigned)MR_SB && !mr_warp_wait(&b_empty[s], ((g / MR_SB) - 1) & 1, fail)) { ok = false; break; }
                const unsigned stage = mr_smem(sB + (size_t)s * BSTAGE);
#pragma unroll
                for (int u = 0; u < NST; ++u) {
                    const int kc = u * RPS + brow;
                    if (kc < w) {
                        const int at = v / (ROWB / 16), j = v % (ROWB / 16);
                        const int sj = ROWB == 128 ? j ^ (kc & 7) : j ^ ((kc >> 1) & 3);
                        mr_copy16(stage + (unsigned)(at * BATOM + kc * ROWB + sj * 16), x16 + (int64_t)r[u] * 2 * KP + v * 8);
                    }
                }
                mr_copy_arrive(&b_full[s]);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");   // the copies in flight land before the CTA exits
    } else if (warp == W_MMA) {
        // ---------------------------------------------------------------- MMA issuer
        pdl_wait();
        if (lane == 0) {
            // D F32 (bits 4-5 = 1), A and B F16, A K-major, B MN-major (bit 16), M = 128; N = 2 KP
            // for A_hi [B_hi | B_lo] into the adjacent accumulators D1 | D2, N = KP for A_lo B_hi
            const unsigned idesc2 = (1u << 4) | (1u << 16) | ((unsigned)((2 * KP) >> 3) << 17) |
                                    ((unsigned)(MR_ROWS >> 4) << 24);
            const unsigned idesc1 = (1u << 4) | (1u << 16) | ((unsigned)(KP >> 3) << 17) | ((unsigned)(MR_ROWS >> 4) << 24);
            unsigned ga = 0, gb = 0, nt = 0;
            bool ok = true;
            MrTask tn;
            if (blockIdx.x < ntasks) tn = tasks[blockIdx.x];
            for (int ti = blockIdx.x; ti < ntasks && ok && !*fail; ti += gridDim.x) {
                const MrTask t = tn;
                if (ti + (int)gridDim.x < ntasks) tn = tasks[ti + gridDim.x];
                const unsigned ab = nt & 1;
                if (nt >= 2 && !mr_wait(&acc_empty[ab], ((nt >> 1) - 1) & 1, fail)) break;
                mr_fence_after();
                const unsigned d1 = taddr + ab * 2 * KP, d2 = d1 + KP;
                const int nch = mr_nchunks(t);
                unsigned acc1 = 0;
                for (int c = 0; c < nch; ++c) {
                    const MrChunk k = mr_chunk(t, c);
                    const int sa = ga % MR_SA, sa2 = (ga + 1) % MR_SA, sb = gb % MR_SB;
                    if (!mr_wait(&a_full[sa], (ga / MR_SA) & 1, fail) ||
                        (k.parts == 2 && !mr_wait(&a_full[sa2], ((ga + 1) / MR_SA) & 1, fail)) ||
                        !mr_wait(&b_full[sb], (gb / MR_SB) & 1, fail)) {
                        ok = false;
                        break;
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the copied B rows, for the MMA
                    mr_fence_after();
                    const unsigned a0 = mr_smem(sA + (size_t)sa * MR_A_STAGE);
                    const unsigned a1 = mr_smem(sA + (size_t)sa2 * MR_A_STAGE);
                    const unsigned bst = mr_smem(sB + (size_t)sb * BSTAGE);
                    const unsigned sbo_a = (unsigned)k.w * 16u;
                    // descriptors of the chunk's first K step; a K step of 16 columns moves A by
                    // two core matrices (256 bytes) and B by 16 K rows (16 ROWB bytes), i.e. the
                    // start-address field (address / 16, low bits) by 16 and ROWB.  The N = KP MMA
                    // reads the hi half of the same operand.
                    uint64_t ah = mr_desc(a0, 128u, sbo_a, 0u), al = mr_desc(a1, 128u, sbo_a, 0u);
                    uint64_t bd = mr_desc(bst, (unsigned)BATOM, 8u * ROWB, SWZ);
                    const int nk = k.w / 16;
                    for (int kk = 0; kk < nk; ++kk) {
                        mr_mma(d1, ah, bd, idesc2, acc1);
                        acc1 = 1;
                        if (k.parts == 2) mr_mma(d2, al, bd, idesc1, 1u);
                        ah += 16u;
                        al += 16u;
                        bd += (unsigned)ROWB;
                    }
                    mr_commit(&a_empty[sa]);
                    if (k.parts == 2) mr_commit(&a_empty[sa2]);
                    mr_commit(&b_empty[sb]);
                    ga += k.parts;
                    ++gb;
                }
                if (!ok) break;
                mr_commit(&acc_full[ab]);
                ++nt;
            }
            // every MMA issued so far has completed once this phase does
            mr_commit(&fin);
            const unsigned long long t0 = mr_ns();
            while (!mr_try(&fin, 0) && mr_ns() - t0 < MR_WAIT_NS) {
            }
        }
    } else {
        // ---------------------------------------------------------------- epilogue (warps 0-3)
        pdl_wait();
        if (threadIdx.x < KP) s_inv[threadIdx.x] = 1.0f / mr_phase_scale(vmax, vt, threadIdx.x);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * MR_GW) : "memory");
        const int row = threadIdx.x;                       // 0..127 = TMEM lane = panel row
        const unsigned lane_base = (unsigned)(32 * warp) << 16;
        unsigned nt = 0;
        MrTask tn;
        if (blockIdx.x < ntasks) tn = tasks[blockIdx.x];
        for (int ti = blockIdx.x; ti < ntasks; ti += gridDim.x, ++nt) {
            const MrTask t = tn;
            if (ti + (int)gridDim.x < ntasks) tn = tasks[ti + gridDim.x];
            const unsigned ab = nt & 1;
            const float rs0 = (vt && row < t.rows && rowscale) ? rowscale[t.s_off + row] : 1.0f;
            if (!mr_warp_wait(&acc_full[ab], (nt >> 1) & 1, fail)) break;
            mr_fence_after();
            const bool live = row < t.rows;
            const float rs = rs0;
            float *orow = out + (t.out_off + row) * KP;
            const unsigned base = taddr + lane_base + ab * 2 * KP;
#pragma unroll 1
            for (int c0 = 0; c0 < KP; c0 += 16) {
                float a[16], b[16];
                mr_ld16(base + c0, a);
                mr_ld16(base + KP + c0, b);
                mr_ld_wait();
                float y[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) y[q] = (a[q] + b[q] * (1.0f / 2048.0f)) * s_inv[c0 + q] * rs;
                if (live) {
#pragma unroll
                    for (int q = 0; q < 16; q += 4)
                        *reinterpret_cast<float4 *>(orow + c0 + q) = make_float4(y[q], y[q + 1], y[q + 2], y[q + 3]);
                }
                if (vt && !t.partial) {
                    // max |t| per right-hand side over the warp's rows: non-negative floats order
                    // as their bit patterns, so one integer warp reduction per column
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        float m = live ? fabsf(y[q]) : 0.0f;
                        if (!(m == m)) m = 0.0f;
                        const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
                        if (lane == 0 && mb) atomicMax(&s_tmax[c0 + q], mb);
                    }
                }
            }
            mr_fence_before();
            mr_arrive(&acc_empty[ab]);
        }
    }
    mr_fence_before();
    __syncthreads();
    mr_fence_after();
    if (threadIdx.x == 0 && s_fail) {   // err is host memory
        *(volatile int *)err = 1;
        __threadfence_system();
    }
    if (vt && threadIdx.x < KP && s_tmax[threadIdx.x]) atomicMax(vmax + 64 + threadIdx.x, s_tmax[threadIdx.x]);
    if (warp == W_MMA)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TCOLS) : "memory");
}

constexpr int MR_TILE = 32;   // rows of the shared-memory transpose tiles of the input and output kernels

// The k inputs (caller's order, component-major, FP64) into [X | X with the dense column
// scales] in the permuted row order, KP FP32 words per row (right-hand sides k .. KP - 1 zero),
// and the largest magnitudes per right-hand side into vmax[r] (X) and vmax[128 + r] (scaled X).
// A tile of 32 consecutive elements of the caller's order, one component, goes through shared
// memory: read with consecutive threads on consecutive elements of one right-hand side
// (coalesced, a thread's KP / 8 reads in flight together), written as whole rows of KP words at the
// elements' permuted positions (iperm).  A thread writes one right-hand side throughout and keeps
// its maxima in registers (one shared and one global atomic per right-hand side and block).  Every
// call writes the row of zeros (`zeros`, MR_ZERO halves) itself: nothing remembers that one has, so a call
// that fails (refused under stream capture) leaves nothing wrong behind.
template <int KP>
__global__ void __launch_bounds__(256) mr_in_kernel(const double *X, const int *__restrict__ iperm, int n, int nin, int k,
                                                    const float *__restrict__ cscale, float *xt, unsigned *vmax,
                                                    uint4 *zeros) {
    __shared__ float tile[MR_TILE][KP + 1];
    __shared__ unsigned s_m[2][KP];
    constexpr int NL = KP * MR_TILE / 256;   // values of a tile per thread
    const int tid = threadIdx.x;
    const int64_t nx = (int64_t)nin * n;
    const int64_t ntile = ((int64_t)n + MR_TILE - 1) / MR_TILE * nin;
    for (int q = tid; q < 2 * KP; q += 256) s_m[q / KP][q % KP] = 0u;
    pdl_wait();
    if (blockIdx.x == 0 && tid < MR_ZERO / 8) zeros[tid] = make_uint4(0u, 0u, 0u, 0u);
    float m = 0.0f, mc = 0.0f;
    const int jl = tid % MR_TILE, rr = tid / MR_TILE;   // reading: element, first right-hand side
    const int wr = tid % KP, wj = tid / KP;             // writing: right-hand side, first element
    for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x) {
        const int c = (int)(t % nin);
        const int64_t j0 = t / nin * MR_TILE, j = j0 + jl;
        double v[NL];
#pragma unroll
        for (int u = 0; u < NL; ++u) {
            const int r = rr + u * (256 / MR_TILE);
            v[u] = r < k && j < n ? X[(int64_t)r * nx + (int64_t)c * n + j] : 0.0;
        }
        __syncthreads();   // the previous tile is written out
#pragma unroll
        for (int u = 0; u < NL; ++u) tile[jl][rr + u * (256 / MR_TILE)] = (float)v[u];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NL; ++u) {
            const int e = wj + u * (256 / KP);
            if (j0 + e >= n) break;
            const int64_t row = (int64_t)iperm[j0 + e] * nin + c;
            const float x = tile[e][wr], xc = x * cscale[row];
            xt[row * KP + wr] = x;              // X, the V^T phase's input
            xt[(nx + row) * KP + wr] = xc;      // X with the row's dense column scale, the near field's input
            const float a = fabsf(x), ac = fabsf(xc);
            if (isfinite(a)) m = fmaxf(m, a);
            if (isfinite(ac)) mc = fmaxf(mc, ac);
        }
    }
    if (m > 0.0f) atomicMax(&s_m[0][wr], __float_as_uint(m));
    if (mc > 0.0f) atomicMax(&s_m[1][wr], __float_as_uint(mc));
    __syncthreads();
    if (tid < KP) {
        if (s_m[0][tid]) atomicMax(vmax + tid, s_m[0][tid]);
        if (s_m[1][tid]) atomicMax(vmax + 128 + tid, s_m[1][tid]);
    }
}

// t of the V^T row tiles cut along K: the sum of their slices' partial rows, in slice order
// (deterministic), and its largest magnitude per right-hand side into vmax[64 + r].  MR_RED_ROWS rows
// of a tile per block, so that the few tiles of the wide groups spread over the chip.
constexpr int MR_RED_ROWS = 16;
template <int KP>
__global__ void __launch_bounds__(256) mr_reduce_kernel(const MrSplit *__restrict__ sp, float *xt, unsigned *vmax) {
    __shared__ unsigned s_m[KP];
    const MrSplit S = sp[blockIdx.x];
    if (threadIdx.x < KP) s_m[threadIdx.x] = 0u;
    __syncthreads();
    pdl_wait();
    const int r1 = min(S.rows, ((int)blockIdx.y + 1) * MR_RED_ROWS);
    for (int e = (int)blockIdx.y * MR_RED_ROWS * KP + (int)threadIdx.x; e < r1 * KP; e += 256) {
        const int r = e / KP, j = e - r * KP;
        float v = 0.0f;
        for (int q = 0; q < S.nsl; ++q) v += xt[(S.p_row + (int64_t)q * MR_ROWS + r) * KP + j];
        xt[(S.t_row + r) * KP + j] = v;
        const float a = fabsf(v);
        if (a > 0.0f && isfinite(a)) atomicMax(&s_m[j], __float_as_uint(a));
    }
    __syncthreads();
    if (threadIdx.x < KP && s_m[threadIdx.x]) atomicMax(vmax + 64 + threadIdx.x, s_m[threadIdx.x]);
}

// The permuted outputs (KP FP32 words per row) into the caller's order, component-major, FP64:
// a tile of 32 consecutive elements of the caller's order, one component, read as whole rows at
// the elements' permuted positions (a thread's reads in flight together) and written with
// consecutive threads on consecutive elements of one right-hand side (coalesced).
template <int KP>
__global__ void __launch_bounds__(256) mr_out_kernel(const float *yp, const int *__restrict__ iperm, int n, int nout, int k,
                                                     double *Y) {
    __shared__ float tile[MR_TILE][KP + 1];
    constexpr int NL = KP * MR_TILE / 256;
    const int tid = threadIdx.x;
    const int64_t ny = (int64_t)nout * n;
    const int64_t ntile = ((int64_t)n + MR_TILE - 1) / MR_TILE * nout;
    const int jl = tid % MR_TILE, rr = tid / MR_TILE;   // writing
    const int wr = tid % KP, wj = tid / KP;             // reading
    pdl_wait();
    for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x) {
        const int c = (int)(t % nout);
        const int64_t j0 = t / nout * MR_TILE, j = j0 + jl;
        float v[NL];
#pragma unroll
        for (int u = 0; u < NL; ++u) {
            const int e = wj + u * (256 / KP);
            v[u] = j0 + e < n ? yp[((int64_t)iperm[j0 + e] * nout + c) * KP + wr] : 0.0f;
        }
        __syncthreads();   // the previous tile is written out
#pragma unroll
        for (int u = 0; u < NL; ++u) tile[wj + u * (256 / KP)][wr] = v[u];
        __syncthreads();
        if (j < n)
#pragma unroll
            for (int u = 0; u < NL; ++u) {
                const int r = rr + u * (256 / MR_TILE);
                if (r < k) Y[(int64_t)r * ny + (int64_t)c * n + j] = (double)tile[jl][r];
            }
    }
}

// ------------------------------------------------------------------ packing
// Panel sources.  V^T task row: V(:, k) of one low-rank block (contiguous over the group's
// columns) times inv_scale.  UY term: like the main path's UyTerm.
struct MrRowSrc {
    const double *v;
    float inv_scale;
};
struct MrTerm {
    const double *src;   // U (column-major, ld = m) or dense (row-major, ld = nc)
    int64_t ld, roff;    // leading dimension, block row of the task's row 0
    int width, coloff;   // columns, first column inside its segment
    int dense;
    const float *inv_scales; // per-column 1 / scale (device), or null
};
struct MrPackTask {
    MrTask t;
    int src0, nsrc;      // V^T: rows [src0, src0 + rows); UY: terms [src0, src0 + nsrc)
};

__device__ __forceinline__ int64_t mr_elem_off(const MrTask &t, int i, int kc, int part) {
    // byte offset of panel entry (row i, task column kc) of part 0 (hi / factor) or 1 (lo)
    const int rg = (t.rows + 7) / 8, parts = 1 + t.lo;
    int64_t base;
    int w, k;
    if (kc < t.kd) {
        const int c = kc / MR_CW;
        k = kc - c * MR_CW;
        w = min(MR_CW, t.kd - c * MR_CW);
        base = t.a_off + (int64_t)c * rg * MR_CW * 16 * parts + (int64_t)part * rg * w * 16;
    } else {
        const int cu = (kc - t.kd) / MR_CW;
        k = kc - t.kd - cu * MR_CW;
        w = min(MR_CW, t.kl - cu * MR_CW);
        base = t.a_off + (int64_t)rg * t.kd * 16 * parts + (int64_t)cu * rg * MR_CW * 16;
    }
    return base + ((int64_t)(i >> 3) * (w >> 3) + (k >> 3)) * 128 + (i & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ void mr_put(unsigned char *panels, const MrTask &t, int i, int kc, double v, bool split) {
    const __half hi = __double2half(v);
    *reinterpret_cast<__half *>(panels + mr_elem_off(t, i, kc, 0)) = hi;
    if (split) {
        const __half lo = __double2half((v - (double)__half2float(hi)) * 2048.0);
        *reinterpret_cast<__half *>(panels + mr_elem_off(t, i, kc, 1)) = lo;
    }
}

// one CTA per task; the panel bytes were zeroed (row and column padding stays zero)
__global__ void mr_pack_kernel(const MrPackTask *__restrict__ pt, int vt, const MrRowSrc *__restrict__ rows,
                               const MrTerm *__restrict__ terms, unsigned char *__restrict__ panels) {
    const MrPackTask P = pt[blockIdx.x];
    const MrTask &t = P.t;
    if (vt) {
        const int64_t tot = (int64_t)t.rows * t.kreal;
        for (int64_t e = threadIdx.x; e < tot; e += blockDim.x) {
            const int i = (int)(e / t.kreal), kc = (int)(e % t.kreal);
            const MrRowSrc R = rows[P.src0 + i];
            mr_put(panels, t, i, t.kd + kc, R.v[kc] * (double)R.inv_scale, false);
        }
    } else {
        for (int q = P.src0; q < P.src0 + P.nsrc; ++q) {
            const MrTerm T = terms[q];
            const int64_t tot = (int64_t)t.rows * T.width;
            for (int64_t e = threadIdx.x; e < tot; e += blockDim.x) {
                const int i = (int)(e / T.width), c = (int)(e % T.width);
                double v = T.dense ? T.src[(T.roff + i) * T.ld + c] : T.src[(int64_t)c * T.ld + T.roff + i];
                if (T.inv_scales) v *= (double)T.inv_scales[c];
                mr_put(panels, t, i, (T.dense ? 0 : t.kd) + T.coloff + c, v, T.dense && t.lo);
            }
        }
    }
}

int64_t mr_round(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

template <typename X>
hbi_status mr_upload(X **dst, const std::vector<X> &v) {
    HBI_ALLOC_TRY((void **)dst, std::max<size_t>(1, v.size()) * sizeof(X));
    if (!v.empty()) HBI_CUDA_TRY(cudaMemcpy(*dst, v.data(), v.size() * sizeof(X), cudaMemcpyHostToDevice));
    return HBI_OK;
}

int64_t mr_task_bytes(const MrTask &t) {
    const int64_t rg = (t.rows + 7) / 8;
    return rg * 16 * ((int64_t)t.kd * (1 + t.lo) + t.kl);
}

template <int KP> const void *mr_fn() { return (const void *)mr_kernel<KP>; }
const void *mr_fn_for(int kp) { return kp == 16 ? mr_fn<16>() : (kp == 32 ? mr_fn<32>() : mr_fn<64>()); }
int mr_smem_bytes(int kp) { return mr_stages_a(kp) * MR_A_STAGE + mr_stages_b(kp) * MR_CW * kp * 4; }

}  // namespace

void multi_free(hbi_handle *h) {
    MultiRhs *m = h->mr;
    if (!m) return;
    void *ptrs[] = {m->d_panels, m->d_vt, m->d_uy, m->d_split, m->d_bidx, m->d_cscale, m->d_iperm, m->d_rowscale,
                    m->d_xt, m->d_yp, m->d_x16, m->d_vmax};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (m->h_err) cudaFreeHost(m->h_err);
    delete m;
    h->mr = nullptr;
}

// Pack the tensor-core panels of H from the FP64 blocks (build time).
hbi_status pack_multi(hbi_handle *h, std::vector<Block> &blocks, const std::vector<int> &leaf_starts) {
    if (h->storage != HBI_FP16 && h->storage != HBI_MIXED) {
        set_error("the multi-RHS product needs HBI_FP16 or HBI_MIXED storage");
        return HBI_ERR_INVALID_ARG;
    }
    const int n = h->n, nin = h->nin, nout = h->nout;
    const int lo = h->storage == HBI_MIXED ? 1 : 0;
    MultiRhs *M = new MultiRhs();
    h->mr = M;
    M->lo = lo;
    M->nx = (int64_t)nin * n;

    // ---- per-column scales: U, V columns of low-rank blocks and dense columns
    std::vector<ColRef> cols;
    std::vector<int64_t> soffU(blocks.size(), -1), soffV(blocks.size(), -1), soffD(blocks.size(), -1);
    for (size_t b = 0; b < blocks.size(); ++b) {
        const Block &B = blocks[b];
        if (B.lowrank) {
            if (B.rank == 0) continue;
            soffU[b] = (int64_t)cols.size();
            for (int k = 0; k < B.rank; ++k) cols.push_back(ColRef{B.d_src + (size_t)k * B.m, B.m, 1});
            soffV[b] = (int64_t)cols.size();
            for (int k = 0; k < B.rank; ++k) cols.push_back(ColRef{B.d_src2 + (size_t)k * B.nc, B.nc, 1});
        } else {
            soffD[b] = (int64_t)cols.size();
            for (int64_t j = 0; j < B.nc; ++j) cols.push_back(ColRef{B.d_src + j, B.m, B.nc});
        }
    }
    std::vector<float> cs;
    hbi_status st = column_scales(cols, cs);
    if (st) return st;
    std::vector<float> inv_cs(cs.size());
    for (size_t i = 0; i < cs.size(); ++i) inv_cs[i] = 1.0f / cs[i];
    float *d_inv_cs = nullptr;
    DevScratch tmp;   // build tables, freed on every return path
    if ((st = tmp.upload(&d_inv_cs, inv_cs))) return st;
    // The dense columns of one X row (one slip component of one element) get one scale, the
    // largest over the near-field blocks that hold the column: the input gather then needs no
    // per-column scale (mr_in_kernel writes the scaled X beside X), and the near-field entries
    // of a column, within a few decades of their maximum, stay far from FP16's subnormal range.
    std::vector<float> cglob(M->nx, 0.0f);
    for (size_t b = 0; b < blocks.size(); ++b)
        if (!blocks[b].lowrank)
            for (int64_t j = 0; j < blocks[b].nc; ++j)
                cglob[blocks[b].col0 + j] = std::max(cglob[blocks[b].col0 + j], cs[soffD[b] + j]);
    std::vector<float> inv_cglob(M->nx);
    for (int64_t j = 0; j < M->nx; ++j) {
        if (!(cglob[j] > 0.0f)) cglob[j] = 1.0f;
        inv_cglob[j] = 1.0f / cglob[j];
    }
    float *d_inv_cglob = nullptr;
    if ((st = tmp.upload(&d_inv_cglob, inv_cglob)) || (st = mr_upload(&M->d_cscale, cglob))) return st;
    {
        std::vector<int> iperm(n);
        for (int p = 0; p < n; ++p) iperm[h->perm[p]] = p;
        if ((st = mr_upload(&M->d_iperm, iperm))) return st;
    }

    // ---- V^T phase: column groups, 128-row tasks
    std::map<std::pair<int64_t, int64_t>, std::vector<int>> groups;
    for (size_t b = 0; b < blocks.size(); ++b)
        if (blocks[b].lowrank && blocks[b].rank > 0) groups[{blocks[b].col0, blocks[b].nc}].push_back((int)b);
    std::vector<int64_t> toff(blocks.size(), -1);
    std::vector<MrPackTask> pvt, puy;
    std::vector<MrRowSrc> vrows;
    std::vector<MrSplit> splits;
    int64_t prow = 0;
    std::vector<float> rowscale;
    int64_t aoff = 0, tcount = 0;
    int64_t alg = 0;
    double flops = 0, mma = 0;
    for (auto &kv : groups) {
        const int64_t col0 = kv.first.first, nc = kv.first.second;
        const int64_t tbase = tcount;
        std::vector<MrRowSrc> rs;
        for (int b : kv.second) {
            const Block &B = blocks[b];
            toff[b] = tbase + (int64_t)rs.size();
            for (int k = 0; k < B.rank; ++k) {
                const float sv = cs[soffV[b] + k], su = cs[soffU[b] + k];
                rs.push_back(MrRowSrc{B.d_src2 + (size_t)k * B.nc, 1.0f / sv});
                rowscale.push_back(sv * su);
            }
            alg += 2 * B.nc * B.rank + 4 * B.rank;
            flops += 2.0 * (double)B.nc * B.rank;
        }
        const int64_t R = (int64_t)rs.size();
        const int nsl = (int)((nc + MR_KSLICE - 1) / MR_KSLICE);
        for (int64_t q = 0; q < R; q += MR_ROWS) {
            const int rows = (int)std::min<int64_t>(MR_ROWS, R - q);
            if (nsl > 1) splits.push_back(MrSplit{2 * M->nx + tbase + q, prow, rows, nsl});
            for (int sl = 0; sl < nsl; ++sl) {
                const int64_t c0 = (int64_t)sl * MR_KSLICE, w = std::min<int64_t>(MR_KSLICE, nc - c0);
                MrPackTask P{};
                P.t.a_off = aoff;
                P.t.g_off = col0 + c0;
                P.t.out_off = nsl > 1 ? prow + (int64_t)sl * MR_ROWS : 2 * M->nx + tbase + q;   // partial rows: fixed below
                P.t.s_off = tbase + q;
                P.t.rows = rows;
                P.t.kd = 0;
                P.t.kl = (int)mr_round(w, 16);
                P.t.kreal = (int)w;
                P.t.lo = 0;
                P.t.partial = nsl > 1;
                P.src0 = (int)vrows.size();
                P.nsrc = rows;
                for (int i = 0; i < rows; ++i) vrows.push_back(MrRowSrc{rs[q + i].v + c0, rs[q + i].inv_scale});
                aoff += mr_round(mr_task_bytes(P.t), 256);
                mma += 2.0 * 2.0 * MR_ROWS * P.t.kl;
                pvt.push_back(P);
            }
            if (nsl > 1) prow += (int64_t)nsl * MR_ROWS;
        }
        tcount += R;
    }
    M->n_t = tcount;
    M->n_prow = prow;
    // partial rows live after T in xt
    for (auto &P : pvt)
        if (P.t.partial) P.t.out_off += 2 * M->nx + tcount;
    for (auto &S : splits) S.p_row += 2 * M->nx + tcount;

    // ---- UY phase: leaf row units, 128-row tasks, [dense | U] columns
    const int nleaves = (int)leaf_starts.size() - 1;
    std::vector<std::vector<int>> unit_terms(nleaves);
    {
        std::vector<int> leaf_of(n);
        for (int u = 0; u < nleaves; ++u)
            for (int e = leaf_starts[u]; e < leaf_starts[u + 1]; ++e) leaf_of[e] = u;
        for (size_t b = 0; b < blocks.size(); ++b) {
            const Block &B = blocks[b];
            if (B.lowrank && B.rank == 0) continue;
            const int e0 = (int)(B.row0 / nout), e1 = (int)((B.row0 + B.m) / nout);
            for (int u = leaf_of[e0]; u < nleaves && leaf_starts[u] < e1; ++u) unit_terms[u].push_back((int)b);
        }
    }
    std::vector<MrTerm> terms;
    std::vector<int> gidx;
    for (int u = 0; u < nleaves; ++u) {
        const int64_t r0 = (int64_t)nout * leaf_starts[u], R = (int64_t)nout * (leaf_starts[u + 1] - leaf_starts[u]);
        const int64_t goff = (int64_t)gidx.size();
        std::vector<MrTerm> ut;
        int64_t Cd = 0, Cl = 0;
        for (int pass = 0; pass < 2; ++pass) {
            for (int b : unit_terms[u]) {
                const Block &B = blocks[b];
                if ((pass == 0) == (bool)B.lowrank) continue;
                MrTerm T{};
                T.roff = r0 - B.row0;
                if (!B.lowrank) {
                    T.src = B.d_src; T.ld = B.nc; T.width = (int)B.nc; T.dense = 1; T.coloff = (int)Cd;
                    T.inv_scales = d_inv_cglob + B.col0;
                    for (int64_t j = 0; j < B.nc; ++j) gidx.push_back((int)(M->nx + B.col0 + j));   // scaled X
                    Cd += B.nc;
                    alg += R * B.nc * (lo ? 4 : 2) + 4 * B.nc;
                    flops += 2.0 * (double)R * B.nc;
                } else {
                    T.src = B.d_src; T.ld = B.m; T.width = B.rank; T.dense = 0; T.coloff = (int)Cl;
                    T.inv_scales = d_inv_cs + soffU[b];
                    for (int k = 0; k < B.rank; ++k) gidx.push_back((int)(2 * M->nx + toff[b] + k));   // T
                    Cl += B.rank;
                    alg += 2 * R * B.rank;
                    flops += 2.0 * (double)R * B.rank;
                }
                ut.push_back(T);
            }
            if (pass == 0)
                for (int64_t c = Cd; c < mr_round(Cd, 16); ++c) gidx.push_back(-1);
        }
        for (int64_t c = Cl; c < mr_round(Cl, 16); ++c) gidx.push_back(-1);
        const int64_t kd = mr_round(Cd, 16), kl = mr_round(Cl, 16);
        for (int64_t q = 0; q < R; q += MR_ROWS) {
            MrPackTask P{};
            P.t.a_off = aoff;
            P.t.g_off = goff;
            P.t.out_off = r0 + q;
            P.t.s_off = -1;
            P.t.rows = (int)std::min<int64_t>(MR_ROWS, R - q);
            P.t.kd = (int)kd;
            P.t.kl = (int)kl;
            P.t.kreal = (int)(kd + kl);
            P.t.lo = lo;
            P.src0 = (int)terms.size();
            P.nsrc = (int)ut.size();
            for (const MrTerm &T0 : ut) {
                MrTerm T = T0;
                T.roff += q;
                terms.push_back(T);
            }
            aoff += mr_round(mr_task_bytes(P.t), 256);
            mma += 2.0 * MR_ROWS * (double)(3 * kd * lo + 2 * kd * (1 - lo) + 2 * kl);
            puy.push_back(P);
        }
    }
    if ((int64_t)gidx.size() > (int64_t)INT32_MAX || 2 * M->nx + tcount > (int64_t)INT32_MAX) {
        set_error("operator too large for the multi-RHS gather indices");
        return HBI_ERR_INVALID_ARG;
    }
    // every task's chunks lie inside the panel stream and fit one A stage; its rows fit the MMA
    for (const auto *L : {&pvt, &puy})
        for (const MrPackTask &P : *L) {
            const MrTask &t = P.t;
            const bool ok = t.rows >= 1 && t.rows <= MR_ROWS && t.kd % 16 == 0 && t.kl % 16 == 0 && t.kd + t.kl > 0 &&
                            t.a_off % 256 == 0 && t.a_off + mr_task_bytes(t) <= aoff &&
                            (int64_t)((t.rows + 7) / 8) * MR_CW * 16 <= MR_A_STAGE;
            if (!ok) {
                set_error("internal error: a multi-RHS task exceeds its buffers");
                return HBI_ERR_INVALID_ARG;
            }
        }

    // ---- device data and packing
    M->panel_bytes = aoff;
    HBI_ALLOC_TRY(&M->d_panels, std::max<int64_t>(256, aoff));
    HBI_CUDA_TRY(cudaMemset(M->d_panels, 0, std::max<int64_t>(256, aoff)));
    MrPackTask *d_pvt = nullptr, *d_puy = nullptr;
    MrRowSrc *d_rows = nullptr;
    MrTerm *d_terms = nullptr;
    if ((st = tmp.upload(&d_pvt, pvt)) || (st = tmp.upload(&d_puy, puy)) || (st = tmp.upload(&d_rows, vrows)) ||
        (st = tmp.upload(&d_terms, terms)))
        return st;
    if (!pvt.empty()) mr_pack_kernel<<<(unsigned)pvt.size(), 256>>>(d_pvt, 1, d_rows, d_terms, M->d_panels);
    HBI_CUDA_TRY(cudaGetLastError());
    if (!puy.empty()) mr_pack_kernel<<<(unsigned)puy.size(), 256>>>(d_puy, 0, d_rows, d_terms, M->d_panels);
    HBI_CUDA_TRY(cudaGetLastError());
    HBI_CUDA_TRY(cudaDeviceSynchronize());

    // B row indices: MR_CW per chunk of every task, padding columns at the row of zeros before X
    // (the row tiles of one leaf row unit share theirs)
    std::vector<int> bidx;
    int64_t last_gather = -1, last_off = 0;
    auto add_rows = [&](MrTask &t, int phase) {
        const int64_t gather = t.g_off;   // V^T: first X row of the slice; UY: the unit's gather list
        if (phase == 1 && gather == last_gather) {
            t.g_off = last_off;
            return;
        }
        t.g_off = (int64_t)bidx.size();
        if (phase == 1) { last_gather = gather; last_off = t.g_off; }
        const int nchd = (t.kd + MR_CW - 1) / MR_CW, nch = nchd + (t.kl + MR_CW - 1) / MR_CW;
        for (int c = 0; c < nch; ++c) {
            const int col0 = c < nchd ? c * MR_CW : t.kd + (c - nchd) * MR_CW;
            const int end = c < nchd ? t.kd : t.kd + t.kl;
            for (int kc = 0; kc < MR_CW; ++kc) {
                const int col = col0 + kc;
                int64_t j = -1;
                if (phase == 0) j = col < t.kreal ? gather + col : -1;
                else if (col < end) j = gidx[gather + col];
                bidx.push_back(j >= 0 ? (int)j : -1);
            }
        }
    };
    std::vector<MrTask> tv, tu;
    for (auto &P : pvt) tv.push_back(P.t);
    for (auto &P : puy) tu.push_back(P.t);
    // V^T tasks largest first (they are independent); UY tasks in tree order, so that the
    // units running at the same time share far-field t entries in L2
    std::stable_sort(tv.begin(), tv.end(), [](const MrTask &a, const MrTask &b) { return mr_task_bytes(a) > mr_task_bytes(b); });
    for (MrTask &t : tv) add_rows(t, 0);
    for (MrTask &t : tu) add_rows(t, 1);
    M->n_vt = (int)tv.size();
    M->n_uy = (int)tu.size();
    M->n_split = (int)splits.size();
    if ((st = mr_upload(&M->d_vt, tv)) || (st = mr_upload(&M->d_uy, tu)) || (st = mr_upload(&M->d_split, splits)) ||
        (st = mr_upload(&M->d_rowscale, rowscale)) || (st = mr_upload(&M->d_bidx, bidx)))
        return st;
    HBI_CUDA_TRY(cudaMallocHost((void **)&M->h_err, sizeof(int)));
    *M->h_err = 0;
    M->bytes_panels_alg = alg;
    M->vec_bytes_per_rhs = 4 * (M->nx + 2 * tcount + (int64_t)nout * n);
    M->flops_per_rhs = flops;
    M->mma_flops_per_rhs = mma;
    return HBI_OK;
}

namespace {
hbi_status mr_prepare(hbi_handle *h, int kp) {
    MultiRhs *M = h->mr;
    const int64_t rows16 = 2 * M->nx + M->n_t;
    if (M->kp_cap < kp) {
        if (M->d_xt) cudaFree(M->d_xt);
        if (M->d_yp) cudaFree(M->d_yp);
        if (M->d_x16) cudaFree(M->d_x16);
        M->d_xt = M->d_yp = nullptr;
        M->d_x16 = nullptr;
        M->kp_cap = M->row_kp = 0;
        // xt rows: X, X scaled per row for the near field, T, partial rows of cut V^T tiles; x16
        // rows: the first three, split, behind the row of zeros
        HBI_ALLOC_TRY(&M->d_xt, (size_t)(2 * M->nx + M->n_t + M->n_prow) * kp * sizeof(float));
        HBI_ALLOC_TRY(&M->d_yp, (size_t)h->nout * h->n * kp * sizeof(float));
        HBI_ALLOC_TRY(&M->d_x16, (MR_ZERO + (size_t)rows16 * 2 * kp) * sizeof(__half));
        M->kp_cap = kp;
    }
    if (!M->d_vmax) HBI_ALLOC_TRY(&M->d_vmax, 192 * sizeof(unsigned));
    if (M->row_kp != kp) {
        const void *fn = mr_fn_for(kp);
        const int smem = mr_smem_bytes(kp);
        HBI_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        HBI_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        // CTAs per SM from shared memory, registers and tensor memory (each CTA holds 4 kp columns,
        // two accumulators, of the SM's 512)
        int dev = 0, sms = 0, smem_sm = 0, resv = 0, regs_sm = 0;
        HBI_CUDA_TRY(cudaGetDevice(&dev));
        HBI_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        HBI_CUDA_TRY(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
        HBI_CUDA_TRY(cudaDeviceGetAttribute(&resv, cudaDevAttrReservedSharedMemoryPerBlock, dev));
        HBI_CUDA_TRY(cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev));
        cudaFuncAttributes fa;
        HBI_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
        const int by_smem = smem_sm / (smem + (int)fa.sharedSizeBytes + resv);
        const int regs_warp = (fa.numRegs * 32 + 255) / 256 * 256;
        const int by_regs = regs_sm / (regs_warp * (MR_THREADS / 32));
        const int per_sm = std::max(1, std::min(std::min(by_smem, by_regs), 512 / (4 * kp)));
        M->grid = sms * per_sm;
        M->row_kp = kp;
    }
    return HBI_OK;
}

// Calls f with kp (16, 32 or 64) as a constant.
template <typename F> hbi_status mr_dispatch(int kp, F &&f) {
    if (kp == 16) return f(std::integral_constant<int, 16>());
    if (kp == 32) return f(std::integral_constant<int, 32>());
    return f(std::integral_constant<int, 64>());
}

// phase 0: V^T (split of X, the V^T product, sums of its cut tiles); 1: UY (split of scaled X and T,
// the row product)
template <int KP>
hbi_status mr_launch_phase(hbi_handle *h, int phase, cudaStream_t s) {
    MultiRhs *M = h->mr;
    const int smem = mr_smem_bytes(KP), sms = std::max(1, h->num_sms);
    auto split = [&](int vt, int64_t row0, int64_t nrows) {
        const int64_t blocks = (nrows * (KP / 8) + 255) / 256;
        return launch_dependent(mr_split_kernel<KP>, (int)std::max<int64_t>(1, std::min<int64_t>(blocks, 8 * sms)), 256, 0,
                                s, M->d_xt, M->d_vmax, vt, row0, nrows, M->d_x16 + MR_ZERO);
    };
    if (phase == 0 && M->n_vt) {
        HBI_CUDA_TRY(split(1, 0, M->nx));
        HBI_CUDA_TRY(launch_dependent(mr_kernel<KP>, std::min(M->grid, M->n_vt), MR_THREADS, smem, s, M->d_vt, M->n_vt, 1,
                                      M->d_panels, M->d_x16 + MR_ZERO, M->d_bidx, M->d_rowscale, M->d_xt, M->d_vmax, M->h_err));
        if (M->n_split) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)M->n_split, MR_ROWS / MR_RED_ROWS);
            cfg.blockDim = dim3(256);
            cfg.stream = s;
            HBI_CUDA_TRY(cudaLaunchKernelEx(&cfg, mr_reduce_kernel<KP>, (const MrSplit *)M->d_split, M->d_xt, M->d_vmax));
        }
    }
    if (phase == 1 && M->n_uy) {
        HBI_CUDA_TRY(split(0, M->nx, M->nx + M->n_t));
        HBI_CUDA_TRY(launch_dependent(mr_kernel<KP>, std::min(M->grid, M->n_uy), MR_THREADS, smem, s, M->d_uy, M->n_uy, 0,
                                      M->d_panels, M->d_x16 + MR_ZERO, M->d_bidx, M->d_rowscale, M->d_yp, M->d_vmax, M->h_err));
    }
    return HBI_OK;
}
hbi_status mr_phase(hbi_handle *h, int kp, int phase, cudaStream_t s) {
    return mr_dispatch(kp, [&](auto kc) { return mr_launch_phase<decltype(kc)::value>(h, phase, s); });
}

// the whole product on `s`, no synchronisation
hbi_status mr_enqueue(hbi_handle *h, int k, int kp, const double *d_X, double *d_Y, cudaStream_t s) {
    MultiRhs *M = h->mr;
    HBI_CUDA_TRY(cudaMemsetAsync(M->d_vmax, 0, 192 * sizeof(unsigned), s));
    const int64_t ntile = ((int64_t)h->n + MR_TILE - 1) / MR_TILE, most = 8 * std::max(1, h->num_sms);
    const int gin = (int)std::min<int64_t>(ntile * h->nin, most), gout = (int)std::min<int64_t>(ntile * h->nout, most);
    hbi_status st = mr_dispatch(kp, [&](auto kc) -> hbi_status {
        HBI_CUDA_TRY(launch_dependent(mr_in_kernel<decltype(kc)::value>, gin, 256, 0, s, d_X, M->d_iperm, h->n, h->nin, k,
                                      M->d_cscale, M->d_xt, M->d_vmax, reinterpret_cast<uint4 *>(M->d_x16)));
        return HBI_OK;
    });
    if (st || (st = mr_phase(h, kp, 0, s)) || (st = mr_phase(h, kp, 1, s))) return st;
    return mr_dispatch(kp, [&](auto kc) -> hbi_status {
        HBI_CUDA_TRY(launch_dependent(mr_out_kernel<decltype(kc)::value>, gout, 256, 0, s, M->d_yp, M->d_iperm, h->n,
                                      h->nout, k, d_Y));
        return HBI_OK;
    });
}

hbi_status mr_check(hbi_handle *h) {
    if (*(volatile int *)h->mr->h_err) {
        *h->mr->h_err = 0;
        set_error("a multi-RHS product wait timed out");
        return HBI_ERR_TIMEOUT;
    }
    return HBI_OK;
}

hbi_status mr_args(hbi_handle *h, int k, int &kp) {
    if (!h) { set_error("handle is required"); return HBI_ERR_INVALID_ARG; }
    if (!h->mr) {
        set_error("the handle was built without the multi-RHS panels (hbi_build_params.multi_rhs = 0)");
        return HBI_ERR_INVALID_ARG;
    }
    if (k < 1 || k > MR_KP_MAX) { set_error("need 1 <= k <= 64 right-hand sides"); return HBI_ERR_INVALID_ARG; }
    // 33 to 48 as 64: a third more row bytes and buffers than rows of 48 would take, which do not fill a
    // swizzle row (k = 40 at 40,000 elements 362 us a call, 64 right-hand sides 370, 32 290; the
    // kernel that converted gathered rows of 48 took 509)
    kp = k <= 16 ? 16 : (k <= 32 ? 32 : 64);
    if (h->num_sms <= 0) {
        int dev = 0;
        HBI_CUDA_TRY(cudaGetDevice(&dev));
        HBI_CUDA_TRY(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev));
    }
    return mr_prepare(h, kp);
}
}  // namespace
}  // namespace hbi

using namespace hbi;

extern "C" hbi_status hbi_matvec_multi(hbi_handle *h, int k, const double *d_X, double *d_Y, hbi_stream stream) {
    if (!d_X || !d_Y) { set_error("X and Y are required"); return HBI_ERR_INVALID_ARG; }
    int kp = 0;
    hbi_status st = mr_args(h, k, kp);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if ((st = mr_enqueue(h, k, kp, d_X, d_Y, s))) return st;
    HBI_CUDA_TRY(cudaStreamSynchronize(s));
    return mr_check(h);
}

extern "C" hbi_status hbi_time_multi(hbi_handle *h, int k, int n_rep, double *out3, hbi_stream stream) {
    if (!out3 || n_rep < 1) { set_error("out3 and n_rep >= 1 are required"); return HBI_ERR_INVALID_ARG; }
    int kp = 0;
    hbi_status st = mr_args(h, k, kp);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    cudaEvent_t e[4];
    for (auto &x : e) HBI_CUDA_TRY(cudaEventCreate(&x));
    double acc[3] = {0, 0, 0};
    for (int r = 0; r < n_rep && !st; ++r) {
        // the input already in xt and its scales (from the last call)
        HBI_CUDA_TRY(cudaEventRecord(e[0], s));
        st = mr_phase(h, kp, 0, s);
        if (!st) { HBI_CUDA_TRY(cudaEventRecord(e[1], s)); st = mr_phase(h, kp, 1, s); }
        if (!st) HBI_CUDA_TRY(cudaEventRecord(e[2], s));
        if (!st) HBI_CUDA_TRY(cudaEventSynchronize(e[2]));
        float a = 0, b = 0;
        if (!st) {
            HBI_CUDA_TRY(cudaEventElapsedTime(&a, e[0], e[1]));
            HBI_CUDA_TRY(cudaEventElapsedTime(&b, e[1], e[2]));
        }
        acc[0] += a; acc[1] += b; acc[2] += a + b;
    }
    for (auto &x : e) cudaEventDestroy(x);
    if (st) return st;
    for (int i = 0; i < 3; ++i) out3[i] = acc[i] / n_rep;
    return mr_check(h);
}

extern "C" hbi_status hbi_multi_stats(const hbi_handle *h, hbi_multi_stats_t *out) {
    if (!h || !out) { set_error("handle and out are required"); return HBI_ERR_INVALID_ARG; }
    if (!h->mr) { set_error("the handle was built without the multi-RHS panels"); return HBI_ERR_INVALID_ARG; }
    const MultiRhs *M = h->mr;
    out->panel_bytes = M->panel_bytes;
    out->bytes_panels_algorithmic = M->bytes_panels_alg;
    out->vector_bytes_per_rhs = M->vec_bytes_per_rhs;
    out->flops_per_rhs = M->flops_per_rhs;
    out->mma_flops_per_rhs = M->mma_flops_per_rhs;
    out->n_tasks_vt = M->n_vt;
    out->n_tasks_uy = M->n_uy;
    out->n_t = M->n_t;
    out->n_split_tiles = M->n_split;
    return HBI_OK;
}
