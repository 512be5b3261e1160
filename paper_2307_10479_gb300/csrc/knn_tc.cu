// Exact k nearest neighbours (paper Eq. 1) with the distance contraction on the 5th-generation
// tensor cores. The result equals the CUDA-core path's bit for bit: the same float32 distances
// sum_d fmaf(q_d - x_d, q_d - x_d, .) in dimension order, ties ordered by id.
//
// Per chunk of queries:
//   1. 16-bit copies of rows and queries (K padded to a multiple of 64), with float32 squared
//      norms and the norms of the rounding residuals x - h(x). The copies are float16 unless a value
//      does not fit it or bfloat16 rounds the inputs better (see choose_bf16): float16's 11 bits
//      make the window below eight times narrower than bfloat16's 8 on rows neither holds exactly.
//      Measured, 1,000 queries x 1M x 960 Gaussian-mixture rows, k = 10: with bfloat16 copies nearly
//      every query overflowed its candidate list and went to the CUDA cores (131 ms); with float16
//      copies none does (2.4 ms);
//   2. sample pass: approximate squared distances a = |q|^2 + |x|^2 - 2 h(q).h(x) of every
//      query against every s-th row (tcgen05.mma.kind::f16, float32 accumulators in tensor memory),
//      reduced to the minimum of each group of 16 or 64 sampled rows; t_s = the k-th smallest group
//      minimum. k groups hold k distinct rows with a <= t_s, so t_s is at least the k-th smallest a
//      over all rows;
//   3. filter pass: a against every row; a row is a candidate when a <= t_s + 2b, where b bounds
//      |a - e| for the float32 distance e (16-bit rounding, accumulation and norm rounding; see
//      error_bound). If e_k is the k-th smallest e, the k rows with the smallest a have e <= t + b
//      (t = k-th smallest a), so e_k <= t + b and every row with e <= e_k has a <= t + 2b <= t_s + 2b:
//      all true neighbours, ties included, are candidates;
//   4. re-rank: per query, t = the k-th smallest a among the candidates (it is the global one), the
//      rows with a <= t + 2b get e computed exactly, sorted by (e, id), the first k returned.
// A query with more candidates than the buffer holds, or fewer than k, is recomputed by the CUDA-core path; one
// whose limit says so beforehand skips the filter pass. Which calls go there whole: knn_sample.h.
//
// The distance kernel is a persistent, warp-specialised tcgen05 pipeline, one CTA per SM:
//   warp 0  TMA producer: 128 queries x 64 and 256 rows x 64 16-bit tiles (128-byte swizzle) into a
//           4-stage shared-memory ring, completion counted on the stage's mbarrier;
//   warp 1  MMA issuer: one thread issues tcgen05.mma (M = 128, N = 256, K = 16) into one of two
//           256-column tensor-memory accumulators, commits each stage back to the producer and each
//           finished tile to the epilogue;
//   warps 2-17 epilogue, eight per accumulator: tcgen05.ld of the finished one (two warps per 32-lane
//           quarter, 128 columns each), approximate distances, group minima (sample pass) or candidate
//           appends (filter pass), then the accumulator is handed back. The two groups work on
//           different tiles, so one's waits and tensor-memory loads overlap the other's
//           arithmetic: sample and filter pass of 10,000 queries x 1M x 128 take 0.130 and 2.50 ms
//           (0.139 and 2.56 ms with all 16 warps on each tile), 1.02 PFLOP/s. There the MMA thread
//           is held by the tensor pipe for 1,650 of 2,450 cycles a tile (the operand copies and reads
//           share its shared-memory bandwidth), by the epilogue for 600, by loads for 240.
// Work items are (query tile, row tile) pairs, the query tile varying fastest, so the CTAs running
// at one time read the same row tiles (each row tile leaves DRAM once, the rest are L2 hits).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "deg_internal.h"
#include "knn_sample.h"

namespace deg {
namespace {

constexpr int TM = 128, TN = 256, KC = 64;
constexpr int kStages = 4;
constexpr int kStageA = TM * KC * 2;                    // 16 KiB of queries
constexpr int kStageB = TN * KC * 2;                    // 32 KiB of rows
constexpr int kStageBytes = kStageA + kStageB;
constexpr int kSmemDyn = kStages * kStageBytes + 1024;  // + alignment slack: one CTA per SM
constexpr int kEpiWarps = 16;                           // epilogue warps: two groups, one per accumulator
constexpr int kGroupWarps = kEpiWarps / 2;              // two per lane quarter
constexpr int kEpiCols = TN * 4 / kGroupWarps;          // accumulator columns per epilogue warp
static_assert(kEpiCols == 128, "the epilogue reads two pairs of 32-column blocks per warp");
constexpr int kTcThreads = 32 * (2 + kEpiWarps);        // producer, MMA, epilogue
constexpr int kTmemCols = 2 * TN;                       // two accumulators
constexpr int kMeta = 4;                                // tiles whose norms and thresholds are staged at once
constexpr int kQueue = 64;                              // candidates an epilogue warp holds before it writes them out
constexpr int64_t kPlanRowsMax = 4096;                  // rows of a k-NN plan (inline fallback in shared memory)
constexpr int64_t kPlanScanRows = 32;                   // up to so many, a plan's k = 1 run scores every row, one a lane
constexpr int kSelThreads = 256;
constexpr int kSelWarpGroups = 1024;                    // groups a warp selects among in registers (32 a lane)
constexpr int kSelBatch = 8;                            // queries a selection block loads at once
constexpr int kRowStage = 36;                           // floats between staged rows of an exact re-scoring
constexpr unsigned long long kWaitNs = 2000000000ull;   // bounded wait on the tensor core: 2 s

// Instruction descriptor, kind::f16: D float32 (bits 4-5 = 1), A and B float16 (bits 7-9, 10-12 = 0)
// or both bfloat16 (= 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t kIdescF16 = (1u << 4) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
constexpr uint32_t kIdescBF16 = kIdescF16 | (1u << 7) | (1u << 10);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a K-major operand in the 128-byte swizzle layout that TMA
// writes (8-row groups of 128-byte rows, 1024 bytes apart): start address >> 4, leading byte
// offset 16 (unused for this layout), stride byte offset 1024, descriptor version 1 (bit 46),
// layout type 2 = 128-byte swizzle (bits 61-63). A K step of 16 elements moves the start by 32 bytes.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, int32_t x, int32_t y, uint32_t mbar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(mbar) : "memory");
}
// `bytes` (a multiple of 16) from 16-byte aligned global memory
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Waits for the given phase of the barrier; false after kWaitNs.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase) {
    const uint64_t start = global_ns();
    for (;;) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(mbar), "r"(phase) : "memory");
        if (done) return true;
        if (global_ns() - start > kWaitNs) return false;
    }
}

// Order-preserving map of a float to an unsigned key (negative approximate distances occur).
__device__ __forceinline__ uint32_t okey(float v) {
    const uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_okey(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Upper bound on |a - e| for one query against any row, with u = 2^-24:
//  - 16-bit rounding of the dot product: with q = bq + rq, x = bx + rx (b the copies),
//    |q.x - bq.bx| <= |q||rx| + |rq||x| + |rq||rx|, doubled by the factor 2 of a;
//  - float32 accumulation of the products, which float32 holds exactly (at most 22 bits): <= (K + 2) 2^-22 sum |bq_d bx_d|
//    (four times the per-addition error of a truncating adder), doubled;
//  - rounding of |q|^2, |x|^2 (K u each, relative), of their combination (2u each), and of e
//    itself ((K + 3) u relative to |q - x|^2 <= (|q| + |x|)^2): (3K + 8) u (|q| + |x|)^2;
//  - coordinates below 2^-126, flushed to zero in the copies: 2^-126 (|q| + |x|) each, doubled.
// K is the padded dimension. |x| and |rx| are replaced by their maxima over the rows; a 1%
// margin covers the float32 evaluation of the bound.
__device__ __forceinline__ float error_bound(float qn, float rq, float xmax2, float rmax, int kpad) {
    const float u = 5.9604645e-08f;
    const float grow = 1.f + (float)(kpad + 2) * u;
    const float Q = sqrtf(qn * grow) * 1.0001f, X = sqrtf(xmax2 * grow) * 1.0001f;
    const float RQ = rq * 1.001f, R = rmax * 1.001f;
    const float rounding = 2.f * (Q * R + RQ * X + RQ * R);
    const float accumulate = 2.f * (float)(kpad + 2) * 2.3841858e-07f * (Q + RQ) * (X + R);
    const float sums = (3.f * (float)kpad + 8.f) * u * (Q + X) * (Q + X);
    const float flushed = 2.f * (float)kpad * 1.1754944e-38f * (Q + X);       // coordinates below 2^-126
    return 1.01f * (rounding + accumulate + sums + flushed) + 1e-30f;
}

// t + 2b, rounded up past the float32 rounding of the sum.
__device__ __forceinline__ float window_limit(float t, float b) {
    return t + 2.f * b + (fabsf(t) + 2.f * b) * 4.7683716e-07f;
}

// The filter compares u = a - |q|^2 with T = limit - |q|^2 rounded up, so a row passes whenever a <= limit.
__device__ __forceinline__ float filter_threshold(float limit, float qn) {
    const float d = limit - qn;
    return d + fabsf(d) * 2.3841858e-07f;
}

// Statistics of a set of rows or queries (non-negative floats, so the int order of the bits is theirs):
// the largest squared norm, the largest residual norm in either format, 1 if float16 cannot hold a value.
enum { kMaxNorm, kMaxRes16, kMaxResB, kNoF16, kStats };
struct Stats {
    const float* x;   // of the rows
    const float* q;   // of the queries
};

// The 16-bit format of the copies, the same for rows and queries (the tensor core takes operands of
// one type): float16, unless some value is outside its range or not finite, or its largest
// residual exceeds what bfloat16 (half an ulp: 2^-9 of a value) can leave at most, on the rows or on
// the queries: values so small that float16 has few or no bits for them. Any choice gives exact
// results, since the bound uses the residuals of the format chosen.
__device__ __forceinline__ bool wants_bf16(const float* st) {
    return st[kNoF16] != 0.f || st[kMaxRes16] > 0.001953125f * sqrtf(st[kMaxNorm]);
}
__device__ __forceinline__ bool choose_bf16(const Stats& st) { return wants_bf16(st.x) || wants_bf16(st.q); }
// The largest row residual in the chosen format.
__device__ __forceinline__ float row_residual(const Stats& st) { return st.x[choose_bf16(st) ? kMaxResB : kMaxRes16]; }

// A 16-bit copy, as two neighbouring elements, and its decoded values. Values that a format holds
// only as subnormals are flushed here, so that the residual accounts for them whatever the tensor
// core does with subnormal operands.
__device__ __forceinline__ uint32_t to_f16x2(float x, float y, float2& back) {
    __half2 h = __floats2half2_rn(x, y);
    const uint32_t keep = __hge2_mask(__habs2(h), __halves2half2(__ushort_as_half(0x0400), __ushort_as_half(0x0400)));
    const uint32_t u = *reinterpret_cast<uint32_t*>(&h) & keep;
    h = *reinterpret_cast<const __half2*>(&u);
    back = __half22float2(h);
    return u;
}
__device__ __forceinline__ uint32_t to_bf16x2(float x, float y, float2& back) {
    const float tiny = 1.17549435e-38f;
    const __nv_bfloat162 b = __floats2bfloat162_rn(fabsf(x) < tiny ? 0.f : x, fabsf(y) < tiny ? 0.f : y);
    back = __bfloat1622float2(b);
    return *reinterpret_cast<const uint32_t*>(&b);
}

struct HalfRows {
    const float* x;          // [rows][dim]
    int64_t rows;
    int32_t dim, kpad;
    uint16_t* out16;         // [rows][kpad] copies
    uint16_t* outb;
    float* norms;            // [rows] float32 sums of squares
    float* res16;            // [rows] residual norms |x - h(x)|, or null
    float* resb;
    float* st;               // [kStats] the statistics of these rows
    Stats both;              // the call's (kIf)
};

// 16-bit copies with zero padding to kpad columns (float16 if kF16, bfloat16 if kB), norms, residual
// norms and their maxima. A residual that is not finite marks values that float16 cannot hold
// (overflow, infinities, NaN). With kIf the kernel does its work only when bfloat16 was chosen: it
// then replaces the float16 copies a first launch wrote. One warp converts kR rows at a time, four
// columns a lane (16-byte loads where the rows are aligned), so kR loads are in flight per lane: 4 for
// a base set, 1 for the few rows of a plan's queries, which need the warps. Bound by HBM: 1M x 128
// takes 125 us (6.2 TB/s; one row a warp and 4-byte loads took 175 us), 1M x 960 825 us (7.0 TB/s;
// 950 us). Residuals of both formats in one pass over a base set cost 324 and 1,801 us.
template <bool kF16, bool kB, bool kIf, int kR>
__global__ void __launch_bounds__(256) half_rows_kernel(const HalfRows A) {
    if (kIf && !choose_bf16(A.both)) return;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const bool vec = (A.dim & 3) == 0 && (reinterpret_cast<uintptr_t>(A.x) & 15) == 0;
    float mn = 0.f, m16 = 0.f, mb = 0.f;
    bool bad = false;
    for (int64_t r0 = warp * kR; r0 < A.rows; r0 += nw * kR) {
        float s[kR] = {}, e[kR] = {}, f[kR] = {};
        for (int i = 4 * lane; i < A.kpad; i += 128) {
            float4 v[kR];
#pragma unroll
            for (int j = 0; j < kR; ++j) {
                v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                const float* p = A.x + (r0 + j) * A.dim + i;
                if (r0 + j >= A.rows) continue;
                if (vec) {
                    if (i < A.dim) v[j] = __ldg(reinterpret_cast<const float4*>(p));
                } else {
                    if (i < A.dim) v[j].x = p[0];
                    if (i + 1 < A.dim) v[j].y = p[1];
                    if (i + 2 < A.dim) v[j].z = p[2];
                    if (i + 3 < A.dim) v[j].w = p[3];
                }
            }
#pragma unroll
            for (int j = 0; j < kR; ++j) {
                if (r0 + j >= A.rows) continue;
                const float4 w = v[j];
                s[j] = fmaf(w.w, w.w, fmaf(w.z, w.z, fmaf(w.y, w.y, fmaf(w.x, w.x, s[j]))));
                float2 lo, hi;
                if (kF16) {
                    uint2 h;
                    h.x = to_f16x2(w.x, w.y, lo);
                    h.y = to_f16x2(w.z, w.w, hi);
                    *reinterpret_cast<uint2*>(A.out16 + (r0 + j) * A.kpad + i) = h;
                    const float a = w.x - lo.x, b = w.y - lo.y, c = w.z - hi.x, d = w.w - hi.y;
                    e[j] = fmaf(d, d, fmaf(c, c, fmaf(b, b, fmaf(a, a, e[j]))));
                }
                if (kB) {
                    uint2 h;
                    h.x = to_bf16x2(w.x, w.y, lo);
                    h.y = to_bf16x2(w.z, w.w, hi);
                    *reinterpret_cast<uint2*>(A.outb + (r0 + j) * A.kpad + i) = h;
                    const float a = w.x - lo.x, b = w.y - lo.y, c = w.z - hi.x, d = w.w - hi.y;
                    f[j] = fmaf(d, d, fmaf(c, c, fmaf(b, b, fmaf(a, a, f[j]))));
                }
            }
        }
#pragma unroll
        for (int m = 16; m; m >>= 1)
#pragma unroll
            for (int j = 0; j < kR; ++j) {
                s[j] += __shfl_xor_sync(0xffffffffu, s[j], m);
                if (kF16) e[j] += __shfl_xor_sync(0xffffffffu, e[j], m);
                if (kB) f[j] += __shfl_xor_sync(0xffffffffu, f[j], m);
            }
#pragma unroll
        for (int j = 0; j < kR; ++j) {
            if (kF16) bad |= !(e[j] < __int_as_float(0x7f800000));
            e[j] = sqrtf(e[j]);
            f[j] = sqrtf(f[j]);
            mn = fmaxf(mn, s[j]);
            m16 = fmaxf(m16, e[j]);
            mb = fmaxf(mb, f[j]);
            if (lane == j && r0 + j < A.rows) {
                A.norms[r0 + j] = s[j];
                if (kF16 && A.res16) A.res16[r0 + j] = e[j];
                if (kB && A.resb) A.resb[r0 + j] = f[j];
            }
        }
    }
    __shared__ float red[3][8];
    bad = __syncthreads_or(bad);
    if (lane == 0) {
        red[0][threadIdx.x >> 5] = mn;
        red[1][threadIdx.x >> 5] = m16;
        red[2][threadIdx.x >> 5] = mb;
    }
    __syncthreads();
    if (threadIdx.x < 3 && (threadIdx.x == 0 || (threadIdx.x == 1 ? kF16 : kB))) {
        float m = 0.f;
        for (int i = 0; i < 8; ++i) m = fmaxf(m, red[threadIdx.x][i]);
        atomicMax(reinterpret_cast<int*>(A.st) + kMaxNorm + threadIdx.x, __float_as_int(m));
    }
    if (threadIdx.x == 0 && bad) A.st[kNoF16] = 1.f;
}

// error_bound of query q in the chosen format.
__device__ __forceinline__ float query_bound(int64_t q, const float* qn, const float* rq16, const float* rqb, const Stats& st, int kpad) {
    return error_bound(qn[q], choose_bf16(st) ? rqb[q] : rq16[q], st.x[kMaxNorm], row_residual(st), kpad);
}

// 32 consecutive accumulator columns of this warp's 32 lanes (one register per column).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr) : "memory");
}

// (u0, u1) = (x0 - 2 v0, x1 - 2 v1) in one paired float32 FMA (each lane rounded once).
__device__ __forceinline__ void xn_minus_2v(float x0, float x1, uint32_t v0, uint32_t v1, float& u0, float& u1) {
    unsigned long long vv, xx, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(vv) : "r"(v0), "r"(v1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(xx) : "f"(x0), "f"(x1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(vv), "l"(0xC0000000C0000000ull), "l"(xx));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(u0), "=f"(u1) : "l"(r));
}

// Waits for this thread's tcgen05.ld; v is tied to the wait, so the compiler treats the registers
// as written here (not at the load) and touches them only afterwards.
__device__ __forceinline__ void tmem_wait_ld(uint32_t* v) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                   "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                   "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :: "memory");
}

// min(a, b, c) in one three-input min (sm_100 and later).
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

struct TcArgs {
    int32_t q_row0;                // first query of this chunk (tensor-map row)
    int32_t nq;                    // queries in this chunk
    int32_t qblocks;               // ceil(nq / 128)
    int64_t ncols;                 // rows in this pass
    int64_t tiles;                 // ceil(ncols / 256)
    int32_t nk;                    // kpad / 64
    const float* qn;               // [ldq] squared norms of this chunk's queries (16-byte aligned)
    const float* xn;               // squared norms of this pass's rows, zero-padded to tiles * 256
    float* gmin;                   // sample pass: [groups][ldq] minima of `group` consecutive rows
    int32_t group;                 //   16 or 64
    int32_t ldq;                   //   qblocks * 128
    const float* limit;            // filter pass: [ldq] the thresholds T of filter_threshold, -inf past nq
    unsigned long long* cand;      // filter pass: [nq][cap] keys okey(a) << 32 | row
    int32_t* cnt;                  // filter pass: [nq]
    int32_t cap;
    int32_t* error;                // set to 1 when a wait ran out
    Stats st;                      // the inputs' statistics: they name the copies' format
};

// Candidates of one epilogue warp, written out together (a query's list needs a global atomic for each,
// and a warp that waits for it holds up its accumulator, and with it the MMA warp); emptied before the
// wait for a tile. Candidates are rare (10,000 queries x 1M x 128: one in every sixth 32 x 32 block), so
// what a block with one costs is mostly instruction fetches: code unrolled over the 32 columns is
// never in the instruction cache. So the lane that holds one hands its 32 values to the warp through shared memory, and a
// short loop compares them, one a lane. The filter pass took 3.75 ms with the columns unrolled and a global
// atomic at each, 5.5 ms with the columns unrolled and a shared-memory queue, 4.2 ms with this loop, 2.56 ms
// once the norms and thresholds no longer came from global memory either (kMeta).
struct Queue {
    float* slot;                   // [32] one lane's values of a half
    unsigned long long* key;       // [kQueue] okey(a) << 32 | row
    int32_t* query;                // [kQueue]
    int n;                         // candidates since the last flush; those past kQueue went straight to their lists
};
__device__ __forceinline__ void append_candidate(const TcArgs& a, int64_t q, unsigned long long key) {
    const int p = atomicAdd(a.cnt + q, 1);
    if (p < a.cap) a.cand[q * a.cap + p] = key;
}
__device__ __forceinline__ void queue_flush(Queue& Q, const TcArgs& a, int lane) {
    __syncwarp();
    for (int i = lane; i < min(Q.n, kQueue); i += 32) append_candidate(a, Q.query[i], Q.key[i]);
    Q.n = 0;
    __syncwarp();
}

// One 32-column half of an epilogue warp's accumulator block: lane = query row qrow, column j =
// row xc + 32 c + j. Per column u = |x|^2 - 2 q.x (one paired FMA; rows past the end get +inf,
// which no filter or group minimum takes); the filter pass queues the rows with u <= T (T = -inf in
// lanes without a query), the sample pass reduces to minima |q|^2 + min u: two of 16 rows, or one of
// the block's 64 carried in `run`. Minima are stored with the query index fastest, 128 bytes a warp.
template <bool kFilter>
__device__ __forceinline__ void epilogue_half(const TcArgs& a, const uint32_t* v, const float4* xs4, int c, int64_t xc,
                                              int64_t qrow, float qnorm, float T, float& run, Queue& Q, int lane) {
    const int64_t xg = xc + c * 32;
    if (xg >= a.ncols) return;                               // warp-uniform
    float u[32];
#pragma unroll
    for (int j4 = 0; j4 < 8; ++j4) {
        const float4 xv = xs4[c * 8 + j4];
        xn_minus_2v(xv.x, xv.y, v[j4 * 4], v[j4 * 4 + 1], u[j4 * 4], u[j4 * 4 + 1]);
        xn_minus_2v(xv.z, xv.w, v[j4 * 4 + 2], v[j4 * 4 + 3], u[j4 * 4 + 2], u[j4 * 4 + 3]);
    }
    if (xg + 32 > a.ncols) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (xg + j >= a.ncols) u[j] = __int_as_float(0x7f800000);
    }
    if (kFilter) {
        float m[11];
#pragma unroll
        for (int j = 0; j < 10; ++j) m[j] = min3f(u[3 * j], u[3 * j + 1], u[3 * j + 2]);
        m[10] = fminf(u[30], u[31]);
        const float lo = fminf(min3f(min3f(m[0], m[1], m[2]), min3f(m[3], m[4], m[5]), min3f(m[6], m[7], m[8])),
                               fminf(m[9], m[10]));
        unsigned hits = __ballot_sync(0xffffffffu, lo <= T);
        while (hits) {
            const int src = __ffs(hits) - 1;
            hits &= hits - 1;
            if (lane == src) {
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *reinterpret_cast<float4*>(Q.slot + j) = make_float4(u[j], u[j + 1], u[j + 2], u[j + 3]);
            }
            __syncwarp();
            const float w = Q.slot[lane];
            const float Ts = __shfl_sync(0xffffffffu, T, src), qs = __shfl_sync(0xffffffffu, qnorm, src);
            const bool hit = w <= Ts && xg + lane < a.ncols;
            const unsigned b = __ballot_sync(0xffffffffu, hit);
            if (hit) {
                const int at = Q.n + __popc(b & ((1u << lane) - 1u));
                const unsigned long long key = ((unsigned long long)okey(qs + w) << 32) | (uint32_t)(xg + lane);
                const int32_t q = (int32_t)qrow - lane + src;
                if (at < kQueue) {
                    Q.key[at] = key;
                    Q.query[at] = q;
                } else {
                    append_candidate(a, q, key);
                }
            }
            Q.n += __popc(b);
            __syncwarp();
        }
    } else {
        float g[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float* w = u + 16 * h;
            const float t0 = min3f(w[0], w[1], w[2]), t1 = min3f(w[3], w[4], w[5]), t2 = min3f(w[6], w[7], w[8]);
            const float t3 = min3f(w[9], w[10], w[11]), t4 = min3f(w[12], w[13], w[14]);
            g[h] = min3f(min3f(t0, t1, t2), fminf(t3, t4), w[15]);
        }
        if (a.group == 16) {
            a.gmin[(xg / 16) * a.ldq + qrow] = qnorm + g[0];
            if (xg + 16 < a.ncols) a.gmin[(xg / 16 + 1) * a.ldq + qrow] = qnorm + g[1];
        } else {
            run = c == 0 ? fminf(g[0], g[1]) : min3f(run, g[0], g[1]);
            if (c == 1 || xg + 32 >= a.ncols) a.gmin[(xc / 64) * a.ldq + qrow] = qnorm + run;
        }
    }
}

template <bool kFilter>
__global__ void __launch_bounds__(kTcThreads, 1) dist_tc_kernel(const __grid_constant__ CUtensorMap tq16,
                                                               const __grid_constant__ CUtensorMap tx16,
                                                               const __grid_constant__ CUtensorMap tqb,
                                                               const __grid_constant__ CUtensorMap txb, const TcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], tfull_bar[2], tempty_bar[2];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t meta_full[kMeta], meta_empty[kMeta];
    __shared__ __align__(16) float meta_xn[kMeta][TN], meta_qn[kMeta][TM], meta_t[kMeta][TM];   // a tile's norms, thresholds
    __shared__ unsigned long long queue_key[kFilter ? kEpiWarps : 1][kQueue];
    __shared__ int32_t queue_query[kFilter ? kEpiWarps : 1][kQueue];
    __shared__ __align__(16) float queue_slot[kFilter ? kEpiWarps : 1][32];
    const uint32_t ring = smem_u32(smem_raw) + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t items = (uint32_t)(a.qblocks * a.tiles);      // < 2^31: checked by the caller
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&tfull_bar[b]), 1);
            mbar_init(smem_u32(&tempty_bar[b]), kGroupWarps);
        }
        for (int m = 0; m < kMeta; ++m) {
            mbar_init(smem_u32(&meta_full[m]), 1);
            mbar_init(smem_u32(&meta_empty[m]), kGroupWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    bool failed = false;
    if (warp == 0) {
        // ---- TMA producer ----
        if (lane == 0) {
            const bool bf = choose_bf16(a.st);
            const CUtensorMap* tq = bf ? &tqb : &tq16;
            const CUtensorMap* tx = bf ? &txb : &tx16;
            asm volatile("prefetch.tensormap [%0];" ::"l"(tq) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(tx) : "memory");
            int s = 0, m = 0;
            uint32_t ph = 0, mph = 0;
            for (uint32_t w = blockIdx.x; w < items && !failed; w += gridDim.x) {
                const int32_t q0 = (int32_t)(w % (uint32_t)a.qblocks) * TM, qy = a.q_row0 + q0;
                const int32_t xy = (int32_t)(w / (uint32_t)a.qblocks) * TN;
                // the epilogue's inputs come by bulk copy too: read by its own warps they put an L2
                // round trip into every tile (10,000 x 1M x 128, filter pass: 4.2 ms that way, 2.56 ms with the copies)
                if (!mbar_wait(smem_u32(&meta_empty[m]), mph ^ 1u)) {
                    failed = true;
                    break;
                }
                const uint32_t mb = smem_u32(&meta_full[m]);
                mbar_expect_tx(mb, 4 * (TN + TM + (kFilter ? TM : 0)));
                bulk_load(smem_u32(meta_xn[m]), a.xn + xy, 4 * TN, mb);
                bulk_load(smem_u32(meta_qn[m]), a.qn + q0, 4 * TM, mb);
                if (kFilter) bulk_load(smem_u32(meta_t[m]), a.limit + q0, 4 * TM, mb);
                if (++m == kMeta) {
                    m = 0;
                    mph ^= 1u;
                }
                for (int kc = 0; kc < a.nk; ++kc) {
                    if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u)) {
                        failed = true;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full_bar[s]);
                    mbar_expect_tx(fb, kStageBytes);
                    const uint32_t dst = ring + s * kStageBytes;
                    tma_load_2d(dst, tq, kc * KC, qy, fb);
                    tma_load_2d(dst + kStageA, tx, kc * KC, xy, fb);
                    if (++s == kStages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer ----
        if (lane == 0) {
            const uint32_t idesc = choose_bf16(a.st) ? kIdescBF16 : kIdescF16;
            int s = 0, acc = 0;
            uint32_t ph = 0, aph = 0;
            for (uint32_t w = blockIdx.x; w < items && !failed; w += gridDim.x) {
                if (!mbar_wait(smem_u32(&tempty_bar[acc]), aph ^ 1u)) {
                    failed = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d = tmem + (uint32_t)(acc * TN);
                for (int kc = 0; kc < a.nk; ++kc) {
                    if (!mbar_wait(smem_u32(&full_bar[s]), ph)) {
                        failed = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = ring + s * kStageBytes, sb = sa + kStageA;
#pragma unroll
                    for (int k16 = 0; k16 < KC / 16; ++k16) {
                        const uint64_t ad = sw128_desc(sa + k16 * 32), bd = sw128_desc(sb + k16 * 32);
                        const uint32_t accumulate = (kc > 0 || k16 > 0) ? 1u : 0u;
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                     ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate) : "memory");
                    }
                    mma_commit(smem_u32(&empty_bar[s]));        // the stage is free once these MMAs finish
                    if (++s == kStages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (failed) break;
                mma_commit(smem_u32(&tfull_bar[acc]));          // the tile is ready for the epilogue
                if (++acc == 2) {
                    acc = 0;
                    aph ^= 1u;
                }
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: warps 2-9 take the tiles of accumulator 0, warps 10-17 those of accumulator 1;
        // a warp reads tensor-memory lanes 32 * (warp % 4) ... + 31 and 128 columns. Per column
        // u = |x|^2 - 2 q.x (one paired FMA) and a = |q|^2 + u: stored keys and group minima are
        // |q|^2 + u. Its rounding and that of filter_threshold are inside the error bound.
        const int group = (warp - 2) / kGroupWarps, quarter = warp & 3, cgroup = ((warp - 2) % kGroupWarps) >> 2;
        const int mine = kFilter ? warp - 2 : 0;
        Queue Q{queue_slot[mine], queue_key[mine], queue_query[mine], 0};
        const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(group * TN + cgroup * kEpiCols);
        int m = group;
        uint32_t aph = 0, mph = 0;
        for (uint32_t w = blockIdx.x + group * gridDim.x; w < items; w += 2 * gridDim.x) {
            const int64_t qrow = (int64_t)(w % (uint32_t)a.qblocks) * TM + quarter * 32 + lane;
            const int64_t xc = (int64_t)(w / (uint32_t)a.qblocks) * TN + cgroup * kEpiCols;
            if (kFilter && Q.n > kQueue / 2) queue_flush(Q, a, lane);
            const bool ok = mbar_wait(smem_u32(&meta_full[m]), mph) && mbar_wait(smem_u32(&tfull_bar[group]), aph);
            if (!__all_sync(0xffffffffu, ok)) {
                failed = true;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const float4* xs4 = reinterpret_cast<const float4*>(meta_xn[m] + cgroup * kEpiCols);
            const float qnorm = meta_qn[m][quarter * 32 + lane], T = kFilter ? meta_t[m][quarter * 32 + lane] : 0.f;
            float run = 0.f;
            // four blocks of 32 columns, one at a time: the other group's warps fill the waits
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                uint32_t v[32];
                tmem_ld32(tbase + h * 32, v);
                tmem_wait_ld(v);
                if (h == 3) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tempty_bar[group]));
                }
                epilogue_half<kFilter>(a, v, xs4 + (h & 2) * 8, h & 1, xc + (h & 2) * 32, qrow, qnorm, T, run, Q, lane);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&meta_empty[m]));
            m += 2;
            if (m >= kMeta) {
                m -= kMeta;
                mph ^= 1u;
            }
            aph ^= 1u;
        }
        if (kFilter) queue_flush(Q, a, lane);
    }
    if (failed && lane == 0) atomicExch(a.error, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// Radix select over `count` 32-bit keys: the key of rank `rank` (0-based), keys read through
// get(i); four passes of 8-bit digits. Lanes of a warp that hit the same bin add once (keys of
// one query crowd into a few bins).
template <int kThreads, typename Get>
__device__ uint32_t radix_select32(int count, uint32_t rank, Get get, uint32_t* hist, uint32_t* prefix_s, uint32_t* rank_s) {
    if (threadIdx.x == 0) {
        *prefix_s = 0;
        *rank_s = rank;
    }
    for (int pass = 0; pass < 4; ++pass) {
        for (int i = threadIdx.x; i < 256; i += kThreads) hist[i] = 0;
        __syncthreads();
        const int shift = 24 - 8 * pass;
        const uint32_t want = *prefix_s;
        const uint32_t hmask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
        for (int i0 = 0; i0 < count; i0 += kThreads) {
            const int i = i0 + (int)threadIdx.x;
            uint32_t bin = 256u;
            if (i < count) {
                const uint32_t kv = get(i);
                if ((kv & hmask) == (want & hmask)) bin = (kv >> shift) & 0xffu;
            }
            const uint32_t peers = __match_any_sync(0xffffffffu, bin);
            if (bin < 256u && (threadIdx.x & 31) == (uint32_t)(__ffs(peers) - 1)) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // the bin that holds the rank: lane l sums bins 8 l ... 8 l + 7, a warp scan finds the lane,
            // and that lane the bin (a serial walk over 256 bins took most of a pass)
            const int lane = threadIdx.x;
            const uint32_t r = *rank_s;
            uint32_t h[8], sum = 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                h[b] = hist[lane * 8 + b];
                sum += h[b];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int m = 1; m < 32; m <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, m);
                if (lane >= m) incl += t;
            }
            // past the last key (rank >= count) the last bin stands, as in a walk that ends there
            const unsigned holds = __ballot_sync(0xffffffffu, r < incl);
            const int src = holds ? __ffs(holds) - 1 : 31;
            __syncwarp();
            if (lane == src) {
                uint32_t acc = incl - sum;
                int b = 0;
                for (; b < 7; ++b) {
                    if (acc + h[b] > r) break;
                    acc += h[b];
                }
                *rank_s = r - acc;
                *prefix_s = want | ((uint32_t)(lane * 8 + b) << shift);
            }
        }
        __syncthreads();
    }
    return *prefix_s;
}

// Groups with a row within a query's limit, at most, while those rows are likely no more than its list holds: a share s
// of n rows is in a share 1 - (1 - s)^group of the groups.
int groups_in_list(int64_t ng, int group, int64_t n, int cap) {
    return n <= cap ? (int)ng : (int)(0.5 + (double)ng * (1.0 - std::pow(1.0 - (double)cap / (double)n, group)));
}

// limit[q] = the filter threshold of window_limit(k-th smallest group minimum, b_q), for the `batch`
// queries from batch * blockIdx.x; +inf when there are fewer than k groups (every row is then a
// candidate), -inf past nq. The
// block reads the minima of its queries group by group (32 bytes each: the group-major layout
// that the sample pass can store coalesced) into shared memory.
//
// A query for whose candidates the list is likely too short (the rounding window is wide for the distances: rows far
// from the origin for their spread) gets the threshold -inf and is marked as overflowed, cnt[q] = cap + 1: it
// goes to the CUDA cores anyway, and the filter pass, made for rare candidates, would spend far longer on its rows than
// they do (200 queries x 1M x 128 Gaussian-mixture rows at an offset of 300, k = 10: 45.2 ms that way).
//
// Up to kSelWarpGroups groups a warp takes a query: 32 keys a lane in registers, and the k-th smallest
// found bit by bit from the top, counting the keys below each trial value (no shared-memory histogram,
// no block barrier). More groups: the block takes one query after the other with a radix select.
// 10,000 queries, 1M rows, k = 10: 55 us (a block per query over 4,096 groups of 16: 131 us).
__global__ void __launch_bounds__(kSelThreads) sample_limit_kernel(const float* __restrict__ gmin, int ng, int ldq, int64_t nq,
                                                                  int k, int batch, const float* __restrict__ qn,
                                                                  const float* __restrict__ rq16, const float* __restrict__ rqb,
                                                                  Stats st, int32_t kpad, float* __restrict__ limit,
                                                                  int max_within, int cap, int32_t* __restrict__ cnt) {
    extern __shared__ __align__(16) uint32_t skeys[];
    __shared__ uint32_t hist[256], prefix_s, rank_s;
    __shared__ int within;
    const int64_t q0 = (int64_t)blockIdx.x * batch;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ld = ng | 1;                                   // odd: the lanes' queries fall into different banks
    if (ng >= k)
        for (int i = threadIdx.x; i < ng * batch; i += kSelThreads) {
            const int g = i / batch, j = i - g * batch;
            skeys[j * ld + g] = okey(gmin[(int64_t)g * ldq + q0 + j]);   // padded to ldq queries
        }
    __syncthreads();
    if (ng <= kSelWarpGroups) {                              // batch == kSelBatch == warps
        const int64_t q = q0 + warp;
        if (q >= nq || ng < k) {
            if (lane == 0) limit[q] = __int_as_float(q < nq ? 0x7f800000 : 0xff800000);
            return;
        }
        uint32_t v[kSelWarpGroups / 32];
#pragma unroll
        for (int i = 0; i < kSelWarpGroups / 32; ++i) v[i] = i * 32 + lane < ng ? skeys[warp * ld + i * 32 + lane] : 0xffffffffu;
        uint32_t t = 0;                                      // keys below t: at most k - 1
        for (int bit = 31; bit >= 0; --bit) {
            const uint32_t trial = t | (1u << bit);
            int c = 0;
#pragma unroll
            for (int i = 0; i < kSelWarpGroups / 32; ++i) c += v[i] < trial;
            if (__reduce_add_sync(0xffffffffu, c) < k) t = trial;
        }
        const float lim = window_limit(from_okey(t), query_bound(q, qn, rq16, rqb, st, kpad));
        const uint32_t klim = okey(lim);                     // an undefined limit counts every group: the CUDA cores too
        int c = 0;
#pragma unroll
        for (int i = 0; i < kSelWarpGroups / 32; ++i) c += v[i] <= klim;
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) {
            const bool over = c > max_within;
            limit[q] = over ? __int_as_float(0xff800000) : filter_threshold(lim, qn[q]);
            if (over) cnt[q] = cap + 1;
        }
    } else {
        for (int j = 0; j < batch; ++j) {
            const int64_t q = q0 + j;
            if (q >= nq || ng < k) {                         // block-uniform
                if (threadIdx.x == 0) limit[q] = __int_as_float(q < nq ? 0x7f800000 : 0xff800000);
                continue;
            }
            const uint32_t* keys = skeys + j * ld;
            if (threadIdx.x == 0) within = 0;                // read only after the selection's barriers
            const uint32_t tk = radix_select32<kSelThreads>(ng, (uint32_t)(k - 1), [&](int i) { return keys[i]; }, hist,
                                                            &prefix_s, &rank_s);
            const float lim = window_limit(from_okey(tk), query_bound(q, qn, rq16, rqb, st, kpad));
            const uint32_t klim = okey(lim);
            int c = 0;
            for (int i = threadIdx.x; i < ng; i += kSelThreads) c += keys[i] <= klim;
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0 && c) atomicAdd(&within, c);
            __syncthreads();
            if (threadIdx.x == 0) {
                const bool over = within > max_within;
                limit[q] = over ? __int_as_float(0xff800000) : filter_threshold(lim, qn[q]);
                if (over) cnt[q] = cap + 1;
            }
        }
    }
}

// Queries a block of sample_limit_kernel takes: kSelBatch where a warp takes one; with more groups as
// many as fit 160 KB of shared memory, and fewer while that leaves SMs idle.
int limit_batch(int64_t ng, int64_t ldq, int sms) {
    int batch = kSelBatch;
    if (ng <= kSelWarpGroups) return batch;
    while (batch > 1 && ((ng | 1) * 4 * batch > 160 * 1024 || ldq / batch < 2 * sms)) batch >>= 1;
    return batch;
}

// Exact float32 squared distance of row x, summed in dimension order (as the CUDA-core path).
__device__ __forceinline__ float exact_row_d2(const float* qv, const float* __restrict__ xf, int64_t x, int32_t dim, bool vec) {
    const float* xv = xf + x * dim;
    float e = 0.f;
    int j = 0;
    if (vec)
        for (; j < dim; j += 4) {
            const float4 r = __ldg(reinterpret_cast<const float4*>(xv + j));
            float t = qv[j] - r.x;
            e = fmaf(t, t, e);
            t = qv[j + 1] - r.y;
            e = fmaf(t, t, e);
            t = qv[j + 2] - r.z;
            e = fmaf(t, t, e);
            t = qv[j + 3] - r.w;
            e = fmaf(t, t, e);
        }
    for (; j < dim; ++j) {
        const float t = qv[j] - xv[j];
        e = fmaf(t, t, e);
    }
    return e;
}

// The same distances of 32 rows, lane l's of row x (lanes with live = false score nothing). The warp reads
// the rows together, 32 columns at a time: eight lanes a row, so every 128-byte line of a row is
// read once and in full, and eight loads a lane are in flight; the columns go through `stage` ([32][kRowStage]
// floats of shared memory, conflict-free both ways) to the lane that sums its row, in dimension
// order. A lane that walks its own row instead asks for 32 lines per load and finds them evicted
// when it comes back: 1,000 queries x 960 columns took 222 us that way, 79 us so.
__device__ __forceinline__ float exact_rows_d2(const float* qv, const float* __restrict__ xf, uint32_t x, bool live, int32_t dim,
                                               bool vec, float* stage, int lane) {
    const unsigned any = __ballot_sync(0xffffffffu, live);
    const int rows = 32 - __clz(any);                        // rows above the last live lane are not read
    float e = 0.f;
    float4 v[8];
    auto load = [&](int d0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 4 * i + (lane >> 3), d = d0 + 4 * (lane & 7);
            const uint32_t xr = __shfl_sync(0xffffffffu, x, r);
            v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r >= rows || !((any >> r) & 1u)) continue;
            const float* p = xf + (int64_t)xr * dim + d;
            if (vec) {
                if (d < dim) v[i] = __ldg(reinterpret_cast<const float4*>(p));
            } else {
                if (d < dim) v[i].x = p[0];
                if (d + 1 < dim) v[i].y = p[1];
                if (d + 2 < dim) v[i].z = p[2];
                if (d + 3 < dim) v[i].w = p[3];
            }
        }
    };
    load(0);
    for (int d0 = 0; d0 < dim; d0 += 32) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i)
            *reinterpret_cast<float4*>(stage + (4 * i + (lane >> 3)) * kRowStage + 4 * (lane & 7)) = v[i];
        __syncwarp();
        if (d0 + 32 < dim) load(d0 + 32);                    // in flight while this chunk is summed
        const int m = min(32, dim - d0);
        const float* sr = stage + lane * kRowStage;
        if (m == 32) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 r = *reinterpret_cast<const float4*>(sr + j), y = *reinterpret_cast<const float4*>(qv + d0 + j);
                float t = y.x - r.x;
                e = fmaf(t, t, e);
                t = y.y - r.y;
                e = fmaf(t, t, e);
                t = y.z - r.z;
                e = fmaf(t, t, e);
                t = y.w - r.w;
                e = fmaf(t, t, e);
            }
        } else {
            for (int j = 0; j < m; ++j) {
                const float t = qv[d0 + j] - sr[j];
                e = fmaf(t, t, e);
            }
        }
    }
    return e;
}

// Ascending block-wide bitonic sort of P keys (P a power of two) in shared memory.
template <int kThreads>
__device__ void bitonic_sort(unsigned long long* a, int P) {
    for (int size = 2; size <= P; size <<= 1)
        for (int stride = size >> 1; stride; stride >>= 1) {
            for (int t = threadIdx.x; t < P / 2; t += kThreads) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const unsigned long long u = a[lo], w = a[hi];
                if ((u > w) == up) {
                    a[lo] = w;
                    a[hi] = u;
                }
            }
            __syncthreads();
        }
}

struct RerankArgs {
    const unsigned long long* cand;   // [nq][cap] candidate keys okey(a) << 32 | row
    const int32_t* cnt;               // [nq]
    int32_t cap, k;
    const float* qf;                  // [nq][dim] float32 queries
    const float* xf;                  // [rows][dim] float32 rows
    int32_t dim;
    const float* qn;                  // [nq]
    const float* rq16;                // [nq] residual norms, float16 and bfloat16
    const float* rqb;
    Stats st;                         // the inputs' statistics
    int32_t kpad;
    int32_t* ids;                     // [nq][k]
    float* dists;                     // [nq][k]
    int32_t* ov;                      // [0] count, [1..] queries left for the CUDA-core path
    int32_t inline_n;                 // > 0: such a query is finished here, exactly, over all inline_n rows
    const int32_t* error;             // nonzero: a tensor-core wait ran out; the results are ids -1
    int32_t sel_at, score_warps;      // rerank_shape
};

// Re-rank (step 4). Dynamic shared memory (rerank_shape): the query row, `cap` 64-bit keys (cap a power
// of 2), overlaid by a row stage per scoring warp once they have been read, and the selected keys; or,
// for the inline fallback, the keys of all rows. Short lists
// (cap up to 1024, the usual case) take blocks of 128 threads, so that 8 to 12 queries share an SM and
// hide each other's barriers; long ones 512. 10,000 queries x 1M x 128, k = 10: 272 us with 512
// threads each, 110 us.
template <int kRerankThreads>
__global__ void __launch_bounds__(kRerankThreads) rerank_kernel(const RerankArgs A) {
    extern __shared__ __align__(16) unsigned long long rk[];
    const int dim4 = (A.dim + 3) & ~3;
    const int lane = threadIdx.x & 31;
    float* qv = reinterpret_cast<float*>(rk);
    unsigned long long* keys = rk + dim4 / 2;
    float* row_stage = reinterpret_cast<float*>(keys) + (threadIdx.x >> 5) * 32 * kRowStage;   // once the keys are read
    unsigned long long* sel = keys + A.sel_at;
    __shared__ uint32_t hist[256], prefix_s, rank_s;
    __shared__ int m_s;
    const int64_t q = blockIdx.x;
    const int k = A.k;
    if (A.error && *A.error) {
        for (int i = threadIdx.x; i < k; i += kRerankThreads) {
            A.ids[q * k + i] = -1;
            A.dists[q * k + i] = __int_as_float(0x7f800000);
        }
        return;
    }
    const int c = A.cnt[q];
    // recomputed by the CUDA-core path: a list too short for its candidates, or fewer than k of them
    // (infinite or undefined distances, which the filter does not order)
    if ((c > A.cap || c < k) && A.inline_n == 0) {
        if (threadIdx.x == 0) A.ov[1 + atomicAdd(A.ov, 1)] = (int32_t)q;
        return;
    }
    for (int j = threadIdx.x; j < A.dim; j += kRerankThreads) qv[j] = A.qf[q * A.dim + j];
    const bool vec = (A.dim & 3) == 0 && (reinterpret_cast<uintptr_t>(A.xf) & 15) == 0;
    if (c > A.cap) {                                     // every row, exactly
        __syncthreads();
        int P = 1;
        while (P < A.inline_n) P <<= 1;
        for (int i = threadIdx.x; i < P; i += kRerankThreads)
            keys[i] = i < A.inline_n ? ((unsigned long long)__float_as_uint(exact_row_d2(qv, A.xf, i, A.dim, vec)) << 32) | (uint32_t)i
                                     : ~0ull;
        __syncthreads();
        bitonic_sort<kRerankThreads>(keys, P);
        for (int i = threadIdx.x; i < k; i += kRerankThreads) {
            A.ids[q * k + i] = (int32_t)(uint32_t)keys[i];
            A.dists[q * k + i] = sqrtf(__uint_as_float((uint32_t)(keys[i] >> 32)));
        }
        return;
    }
    for (int i = threadIdx.x; i < c; i += kRerankThreads) keys[i] = A.cand[q * A.cap + i];
    if (threadIdx.x == 0) m_s = 0;
    __syncthreads();
    const uint32_t tk = radix_select32<kRerankThreads>(c, (uint32_t)(k - 1), [&](int i) { return (uint32_t)(keys[i] >> 32); },
                                                       hist, &prefix_s, &rank_s);
    const float lim = window_limit(from_okey(tk), query_bound(q, A.qn, A.rq16, A.rqb, A.st, A.kpad));
    for (int i = threadIdx.x; i < c; i += kRerankThreads) {
        const unsigned long long key = keys[i];
        if (!(from_okey((uint32_t)(key >> 32)) > lim)) sel[atomicAdd(&m_s, 1)] = (uint32_t)key;
    }
    __syncthreads();
    const int m = m_s;
    for (int i0 = threadIdx.x & ~31; i0 < m && (int)threadIdx.x < 32 * A.score_warps; i0 += 32 * A.score_warps) {
        const bool live = i0 + lane < m;
        const uint32_t x = live ? (uint32_t)sel[i0 + lane] : 0u;
        const float e = exact_rows_d2(qv, A.xf, x, live, A.dim, vec, row_stage, lane);
        if (live) sel[i0 + lane] = ((unsigned long long)__float_as_uint(e) << 32) | x;
    }
    __syncthreads();
    int P = 1;
    while (P < m) P <<= 1;
    for (int i = m + threadIdx.x; i < P; i += kRerankThreads) sel[i] = ~0ull;
    __syncthreads();
    bitonic_sort<kRerankThreads>(sel, P);
    for (int i = threadIdx.x; i < k; i += kRerankThreads) {
        A.ids[q * k + i] = (int32_t)(uint32_t)sel[i];
        A.dists[q * k + i] = sqrtf(__uint_as_float((uint32_t)(sel[i] >> 32)));
    }
}

// k = 1: the filter threshold of window_limit(min of the group minima, b_q). A block takes 32 queries,
// one a lane; its four warps share the groups, so that even the 64 groups of 4,096 rows are one or two
// rounds of loads (a thread per query walks them in eight). A group whose minimum is within the limit holds
// a candidate: with more such groups than a list holds (cnt given), the query takes no part in the filter pass
// and is marked as overflowed at once; the counts of the others are cleared.
constexpr int kPlanGroups = kPlanRowsMax / 64;
__global__ void __launch_bounds__(128) nearest_limit_kernel(const float* __restrict__ gmin, int ng, int ldq, int64_t nq,
                                                            const float* __restrict__ qn, const float* __restrict__ rq16,
                                                            const float* __restrict__ rqb, Stats st, int32_t kpad,
                                                            float* __restrict__ limit, int cap, int32_t* __restrict__ cnt) {
    __shared__ float part[4][32];
    __shared__ int within[4][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * 32 + lane;          // below ldq, a multiple of 128
    const float inf = __int_as_float(0x7f800000);
    float v[kPlanGroups / 4], m = inf;
#pragma unroll
    for (int i = 0; i < kPlanGroups / 4; ++i) {
        v[i] = warp + 4 * i < ng ? __ldg(gmin + (int64_t)(warp + 4 * i) * ldq + q) : inf;
        m = fminf(m, v[i]);
    }
    part[warp][lane] = m;
    __syncthreads();
    if (!cnt && warp > 0) return;
    m = fminf(fminf(part[0][lane], part[1][lane]), fminf(part[2][lane], part[3][lane]));
    const float lim = q < nq ? window_limit(m, query_bound(q, qn, rq16, rqb, st, kpad)) : -inf;
    bool over = false;
    if (cnt) {
        int c = 0;
#pragma unroll
        for (int i = 0; i < kPlanGroups / 4; ++i) c += warp + 4 * i < ng && v[i] <= lim;
        within[warp][lane] = c;
        __syncthreads();
        if (warp > 0) return;
        over = q < nq && within[0][lane] + within[1][lane] + within[2][lane] + within[3][lane] > cap;
        if (q < nq) cnt[q] = over ? cap + 1 : 0;
    }
    limit[q] = q < nq && !over ? filter_threshold(lim, qn[q]) : -inf;
}

// k = 1, one warp per query: the exact (distance, row) minimum over the candidates, or over every
// row when they overflowed; or, with `left`, the queries whose candidates overflowed or are none (an undefined
// bound) are listed there, from row0 on, for a kernel that scores all rows by tiles. All candidates are scored, so no selection is needed; a lone candidate is
// the answer as it stands where no distance is asked for (dists null). Four rows at a time are read
// together with the query, 128 columns of each by the whole warp (512 contiguous bytes), and summed by a lane each from
// shared memory, in dimension order. A lane that walked its own row took 15.5 us for 10,000 queries x 128
// columns, this 14 us (most of it
// one dependent chain: count, candidate, row, 128 FMAs). Without `left` a query without a candidate gets row -1.
// kAll: no candidates are given, every row is scored, and a query without a finite distance gets row -1.
constexpr int kFinishRows = 4, kFinishStride = 132;
template <bool kAll>
__global__ void __launch_bounds__(256) nearest_finish_kernel(const unsigned long long* __restrict__ cand,
                                                             const int32_t* __restrict__ cnt, int cap,
                                                             const float* __restrict__ qf, const float* __restrict__ xf,
                                                             int32_t dim, int64_t n, int64_t nq, int32_t* __restrict__ left,
                                                             int32_t* __restrict__ left_n, int32_t row0,
                                                             int32_t* __restrict__ ids, float* __restrict__ dists,
                                                             const int32_t* __restrict__ error) {
    __shared__ __align__(16) float stage[8][(1 + kFinishRows) * kFinishStride];
    const int lane = threadIdx.x & 31;
    const int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= nq) return;
    const int c = kAll || *error ? 0 : cnt[q];
    if (!kAll && *error) {
        if (lane == 0) {
            ids[q] = -1;
            if (dists) dists[q] = __int_as_float(0x7f800000);
        }
        return;
    }
    const float* qv = qf + q * dim;
    const bool vec = (dim & 3) == 0 && (reinterpret_cast<uintptr_t>(xf) & 15) == 0 && (reinterpret_cast<uintptr_t>(qf) & 15) == 0;
    unsigned long long best = ~0ull;
    if (left && (c > cap || c == 0)) {
        if (lane == 0) left[atomicAdd(left_n, 1)] = row0 + (int32_t)q;
        return;
    }
    if (kAll || c > cap) {
        for (int64_t x = lane; x < n; x += 32)
            best = min(best, ((unsigned long long)__float_as_uint(exact_row_d2(qv, xf, x, dim, vec)) << 32) | (uint32_t)x);
    } else if (c == 1 && !dists) {
        if (lane == 0) ids[q] = (int32_t)(uint32_t)cand[q * cap];
        return;
    } else {
        float* s = stage[threadIdx.x >> 5];
        auto load4 = [&](const float* row, int d) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (vec) {
                if (d < dim) v = __ldg(reinterpret_cast<const float4*>(row + d));
            } else {
                if (d < dim) v.x = row[d];
                if (d + 1 < dim) v.y = row[d + 1];
                if (d + 2 < dim) v.z = row[d + 2];
                if (d + 3 < dim) v.w = row[d + 3];
            }
            return v;
        };
        for (int i0 = 0; i0 < c; i0 += kFinishRows) {
            const int m = min(kFinishRows, c - i0);
            const uint32_t x = lane < m ? (uint32_t)cand[q * cap + i0 + lane] : 0u;
            float e = 0.f;
            for (int d0 = 0; d0 < dim; d0 += 128) {
                const int d = d0 + 4 * lane;
                float4 v[1 + kFinishRows];
                v[0] = load4(qv, d);
#pragma unroll
                for (int r = 0; r < kFinishRows; ++r) {
                    const uint32_t xr = __shfl_sync(0xffffffffu, x, r);
                    if (r < m) v[1 + r] = load4(xf + (int64_t)xr * dim, d);
                }
                __syncwarp();
#pragma unroll
                for (int r = 0; r <= kFinishRows; ++r)
                    if (r <= m) *reinterpret_cast<float4*>(s + r * kFinishStride + 4 * lane) = v[r];
                __syncwarp();
                if (lane < m) {
                    const float* row = s + (1 + lane) * kFinishStride;
                    const int w = min(128, dim - d0);          // columns past dim hold zeros: adding them changes nothing
#pragma unroll 8
                    for (int j = 0; j < w; j += 4) {
                        const float4 a = *reinterpret_cast<const float4*>(s + j), b = *reinterpret_cast<const float4*>(row + j);
                        float t = a.x - b.x;
                        e = fmaf(t, t, e);
                        t = a.y - b.y;
                        e = fmaf(t, t, e);
                        t = a.z - b.z;
                        e = fmaf(t, t, e);
                        t = a.w - b.w;
                        e = fmaf(t, t, e);
                    }
                }
            }
            if (lane < m) best = min(best, ((unsigned long long)__float_as_uint(e) << 32) | x);
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, best, o);
        best = min(best, t);
    }
    if (kAll && (uint32_t)(best >> 32) >= 0x7f800000u) best = ~0ull;
    if (lane == 0) {
        ids[q] = (int32_t)(uint32_t)best;
        if (dists) dists[q] = sqrtf(__uint_as_float((uint32_t)(best >> 32)));
    }
}

// Threads of rerank_kernel, where its selected keys start (in keys), the warps that score rows (all
// whose stages fit beside the rest, at least those that fit over the keys) and its shared memory.
struct RerankShape {
    int threads, sel_at, score_warps, smem;
};
RerankShape rerank_shape(int cap, int dim, int inline_n, int smem_max) {
    constexpr int stage = 32 * kRowStage * 4;
    int P = 1;
    while (P < inline_n) P <<= 1;
    RerankShape r{};
    r.threads = cap <= 1024 ? 128 : 512;
    for (r.score_warps = r.threads / 32;; --r.score_warps) {
        r.sel_at = std::max(8 * cap, r.score_warps * stage) / 8;
        r.smem = 4 * ((dim + 3) & ~3) + 8 * std::max(r.sel_at + cap, inline_n > 0 ? P : 0);
        if (r.smem <= smem_max || r.score_warps == 1 || r.score_warps * stage <= 8 * cap) return r;
    }
}
void launch_rerank(RerankArgs A, int64_t nq, const RerankShape& r, cudaStream_t st) {
    A.sel_at = r.sel_at;
    A.score_warps = r.score_warps;
    if (r.threads == 128) rerank_kernel<128><<<(unsigned)nq, 128, r.smem, st>>>(A);
    else rerank_kernel<512><<<(unsigned)nq, 512, r.smem, st>>>(A);
}

__global__ void gather_rows_kernel(const float* __restrict__ src, const int32_t* __restrict__ list, int count, int32_t dim,
                                   float* __restrict__ dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)count * dim;
         i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[(int64_t)list[i / dim] * dim + i % dim];
}

__global__ void scatter_results_kernel(const int32_t* __restrict__ gid, const float* __restrict__ gd,
                                       const int32_t* __restrict__ list, int count, int k, int32_t* __restrict__ ids,
                                       float* __restrict__ dists) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)count * k;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = list[i / k];
        ids[q * k + i % k] = gid[i];
        dists[q * k + i % k] = gd[i];
    }
}

// xs[j] = xn[j * stride] for j < ns; zero up to `padded`.
__global__ void strided_norms_kernel(const float* __restrict__ xn, int64_t stride, int64_t ns, int64_t padded,
                                     float* __restrict__ xs) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < padded; j += (int64_t)gridDim.x * blockDim.x)
        xs[j] = j < ns ? xn[j * stride] : 0.f;
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once through the runtime (no link to libcuda).
EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// 2-D map over `rows` rows of `kpad` 16-bit elements, `row_bytes` apart; box 64 x box_rows with the
// 128-byte swizzle; rows past the end read as zero.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t kpad, uint64_t row_bytes, uint32_t box_rows) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[2] = {kpad, rows};
    const cuuint64_t strides[1] = {row_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)KC, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// dst[i][0 .. dim) = src[(ids ? ids[i] : i) * stride + 0 .. dim)
__global__ void gather_plan_rows_kernel(const float* __restrict__ src, int64_t stride, const int32_t* __restrict__ ids,
                                        int64_t n, int32_t dim, float* __restrict__ dst) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * dim; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / dim;
        dst[t] = src[(ids ? (int64_t)ids[i] : i) * stride + t % dim];
    }
}

// The dynamic shared-memory limit is one process-wide setting per kernel: raise it, once, to the
// device's opt-in maximum (occupancy follows the bytes each launch asks for, not this limit).
template <typename F>
cudaError_t open_smem_limit(F* f, int optin) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    return e;
}

// rerank_max: the dynamic shared memory a block of rerank_kernel may ask for.
cudaError_t open_smem_limits(int* rerank_max) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = open_smem_limit(dist_tc_kernel<false>, optin);
    if (e == cudaSuccess) e = open_smem_limit(dist_tc_kernel<true>, optin);
    if (e == cudaSuccess) e = open_smem_limit(rerank_kernel<128>, optin);
    if (e == cudaSuccess) e = open_smem_limit(rerank_kernel<512>, optin);
    if (e == cudaSuccess) e = open_smem_limit(sample_limit_kernel, optin);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, rerank_kernel<512>);
    if (e == cudaSuccess) *rerank_max = optin - (int)fa.sharedSizeBytes;
    return e;
}

struct Scratch {
    void* p[13] = {};
    ~Scratch() {
        for (void* q : p) cudaFree(q);
    }
};

// launch_knn_exact's scratch, kept between calls: per device, grown when a call needs more, made
// again in a new context of the device (the old context's memory went with it). The lock is held
// for the whole call, which ends with its stream synchronised, so no call's kernels use a buffer
// that another call frees or grows.
struct KnnScratch {
    static constexpr int kBuffers = 13;
    std::mutex mu;
    unsigned long long ctx = 0;
    void* p[kBuffers] = {};
    size_t bytes[kBuffers] = {};
};
KnnScratch g_knn_scratch[64];

}  // namespace

int launch_knn_exact(const float* base, int64_t n, const float* queries, int64_t nq, int32_t dim, int32_t k,
                     int32_t* ids, float* dists, deg_stream_t stream, std::string* why) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (k > n) return *why = "k larger than n", (int)cudaErrorInvalidValue;
    if (nq == 0) return 0;
    if (n > INT32_MAX - TN) return *why = "n too large", (int)cudaErrorInvalidValue;   // work items fit 31 bits
    const int32_t kpad = (dim + KC - 1) / KC * KC;
    const SamplePlan plan = sample_plan(n, nq, dim, k);
    // the CUDA cores also take rows too wide for the re-rank's shared memory (its longest lists leave room for about
    // 24,000 columns, its shortest for about 52,000)
    int rerank_max = 0;
    if (const cudaError_t e = open_smem_limits(&rerank_max)) return *why = cudaGetErrorString(e), (int)e;
    const RerankShape rerank = rerank_shape(plan.cap, dim, 0, rerank_max);
    if (!plan.filter || rerank.smem > rerank_max) return launch_knn_simt(base, n, queries, nq, dim, k, ids, dists, stream, why);
    const int64_t stride = plan.stride, ns = plan.ns, ng = plan.ng;
    const int32_t group = plan.group, cap = plan.cap;
    const int max_within = groups_in_list(ng, group, n, cap);
    // queries per chunk: at most 16,384, and at most 1 GiB of group minima
    const int64_t chunk = std::min<int64_t>({(nq + TM - 1) / TM * TM, 16384, (1ll << 28) / ng / TM * TM});
    const int64_t tiles_n = (n + TN - 1) / TN, tiles_s = (ns + TN - 1) / TN;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    if (dev < 0 || dev >= 64) return *why = "device index above 63", (int)cudaErrorInvalidValue;
    KnnScratch& s = g_knn_scratch[dev];
    std::lock_guard<std::mutex> lock(s.mu);
    unsigned long long ctx = current_context_id();
    if (ctx == 0) {
        cudaFree(nullptr);                                   // makes the device's context current
        ctx = current_context_id();
    }
    if (ctx == 0 || ctx != s.ctx) {
        for (int i = 0; i < KnnScratch::kBuffers; ++i) {
            s.p[i] = nullptr;
            s.bytes[i] = 0;
        }
        s.ctx = ctx;
    }
    const size_t sizes[KnnScratch::kBuffers] = {2ull * n * kpad, 4ull * tiles_n * TN, 2ull * nq * kpad, 4ull * ((nq + TM - 1) / TM * TM), 4ull * nq,
                            4ull * nq, 8ull * kStats, 4ull * chunk * ng, 4ull * chunk, 8ull * chunk * cap, 4ull * chunk,
                            4ull * (chunk + 2), 4ull * tiles_s * TN};
    for (int i = 0; i < KnnScratch::kBuffers && e == cudaSuccess; ++i) {
        const size_t need = std::max<size_t>(sizes[i], 16);
        if (s.bytes[i] >= need) continue;
        if (s.p[i]) cudaFree(s.p[i]);
        s.p[i] = nullptr;
        s.bytes[i] = 0;
        if ((e = cudaMalloc(&s.p[i], need)) == cudaSuccess) s.bytes[i] = need;
    }
    if (e == cudaErrorMemoryAllocation) {
        // no room for the 16-bit copy of the rows: the CUDA-core path needs 2 GiB at most
        cudaGetLastError();
        for (int i = 0; i < KnnScratch::kBuffers; ++i) {
            cudaFree(s.p[i]);
            s.p[i] = nullptr;
            s.bytes[i] = 0;
        }
        return launch_knn_simt(base, n, queries, nq, dim, k, ids, dists, stream, why);
    }
    if (e != cudaSuccess) return *why = std::string("knn scratch: ") + cudaGetErrorString(e), (int)e;
    auto* xh = static_cast<uint16_t*>(s.p[0]);
    auto* xn = static_cast<float*>(s.p[1]);
    auto* qh = static_cast<uint16_t*>(s.p[2]);
    auto* qn = static_cast<float*>(s.p[3]);
    auto* qr16 = static_cast<float*>(s.p[4]);
    auto* qrb = static_cast<float*>(s.p[5]);
    auto* stats = static_cast<float*>(s.p[6]);
    auto* gmin = static_cast<float*>(s.p[7]);
    auto* limit = static_cast<float*>(s.p[8]);
    auto* cand = static_cast<unsigned long long*>(s.p[9]);
    auto* cnt = static_cast<int32_t*>(s.p[10]);
    auto* ov = static_cast<int32_t*>(s.p[11]);         // [0] overflow count, [1..chunk] queries, [chunk+1] error
    auto* xs = static_cast<float*>(s.p[12]);
    int32_t* err = ov + chunk + 1;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    CUtensorMap tq, tx_all, tx_sample;
    if (!make_map(&tq, qh, nq, kpad, 2ull * kpad, TM) || !make_map(&tx_all, xh, n, kpad, 2ull * kpad, TN) ||
        !make_map(&tx_sample, xh, ns, kpad, 2ull * kpad * stride, TN))
        return *why = "tensor map encoding failed", (int)cudaErrorInvalidValue;
    const Stats both{stats, stats + kStats};
    cudaMemsetAsync(stats, 0, 8ull * kStats, st);
    cudaMemsetAsync(xn, 0, 4ull * tiles_n * TN, st);
    const HalfRows hx{base, n, dim, kpad, xh, xh, xn, nullptr, nullptr, stats, both};
    const HalfRows hq{queries, nq, dim, kpad, qh, qh, qn, qr16, qrb, stats + kStats, both};
    auto blocks = [&](int64_t rows) { return (unsigned)std::min<int64_t>((rows + 31) / 32, (int64_t)sms * 8); };
    half_rows_kernel<true, false, false, 4><<<blocks(n), 256, 0, st>>>(hx);
    half_rows_kernel<true, false, false, 4><<<blocks(nq), 256, 0, st>>>(hq);
    half_rows_kernel<false, true, true, 4><<<blocks(n), 256, 0, st>>>(hx);
    half_rows_kernel<false, true, true, 4><<<blocks(nq), 256, 0, st>>>(hq);
    strided_norms_kernel<<<256, 256, 0, st>>>(xn, stride, ns, tiles_s * TN, xs);
    for (int64_t q0 = 0; q0 < nq && e == cudaSuccess; q0 += chunk) {
        const int64_t qc = std::min(chunk, nq - q0);
        const int32_t qblocks = (int32_t)((qc + TM - 1) / TM);
        const int batch = limit_batch(ng, qblocks * TM, sms);
        auto grid = [&](int64_t tiles) { return (unsigned)std::min<int64_t>((int64_t)qblocks * tiles, sms); };
        const TcArgs sa{(int32_t)q0, (int32_t)qc, qblocks, ns, tiles_s, kpad / KC, qn + q0, xs, gmin, group, qblocks * TM, nullptr, nullptr, nullptr, 0, err, both};
        const TcArgs fa{(int32_t)q0, (int32_t)qc, qblocks, n, tiles_n, kpad / KC, qn + q0, xn, nullptr, 0, 0, limit, cand, cnt, cap, err, both};
        cudaMemsetAsync(ov, 0, 4ull * (chunk + 2), st);
        cudaMemsetAsync(cnt, 0, 4ull * qc, st);
        dist_tc_kernel<false><<<grid(tiles_s), kTcThreads, kSmemDyn, st>>>(tq, tx_sample, tq, tx_sample, sa);
        sample_limit_kernel<<<(unsigned)(qblocks * TM / batch), kSelThreads, 4 * (int)(ng | 1) * batch, st>>>(gmin, (int)ng, qblocks * TM, qc, k, batch, qn + q0, qr16 + q0, qrb + q0, both, kpad, limit, max_within, cap, cnt);
        dist_tc_kernel<true><<<grid(tiles_n), kTcThreads, kSmemDyn, st>>>(tq, tx_all, tq, tx_all, fa);
        const RerankArgs ra{cand, cnt, cap, k, queries + q0 * dim, base, dim, qn + q0, qr16 + q0, qrb + q0, both, kpad,
                            ids + q0 * k, dists + q0 * k, ov, 0, nullptr};
        launch_rerank(ra, qc, rerank, st);
        int32_t flags[2] = {0, 0};
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        if ((e = cudaMemcpyAsync(&flags[0], ov, 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess) break;
        if ((e = cudaMemcpyAsync(&flags[1], err, 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess) break;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) break;
        if (flags[1]) return *why = "a tensor-core wait exceeded its limit", (int)cudaErrorLaunchTimeout;
        if (flags[0] > 0) {                              // too many candidates: the CUDA-core path
            const int nov = flags[0];
            Scratch g;
            if ((e = cudaMalloc(&g.p[0], 4ull * nov * dim)) != cudaSuccess || (e = cudaMalloc(&g.p[1], 4ull * nov * k)) != cudaSuccess ||
                (e = cudaMalloc(&g.p[2], 4ull * nov * k)) != cudaSuccess)
                break;
            gather_rows_kernel<<<256, 256, 0, st>>>(queries + q0 * dim, ov + 1, nov, dim, static_cast<float*>(g.p[0]));
            const int r = launch_knn_simt(base, n, static_cast<float*>(g.p[0]), nov, dim, k, static_cast<int32_t*>(g.p[1]),
                                          static_cast<float*>(g.p[2]), stream, why);
            if (r != 0) return r;
            scatter_results_kernel<<<256, 256, 0, st>>>(static_cast<int32_t*>(g.p[1]), static_cast<float*>(g.p[2]), ov + 1,
                                                        nov, k, ids + q0 * k, dists + q0 * k);
            if ((e = cudaStreamSynchronize(st)) != cudaSuccess) break;
        }
    }
    if (e != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    return 0;
}

// ---- k-NN plan over a small fixed row set (entry routing) ------------------------------------
// The same pipeline as launch_knn_exact, with the rows' 16-bit copies, norms and tensor maps made
// once, scratch kept between calls, and no host synchronisation: a query with more candidates
// than `cap` is finished exactly inside the re-rank kernel over all rows (at most kPlanRowsMax).
struct KnnPlan {
    int64_t n = 0;
    int32_t dim = 0, kpad = 0, k = 0, cap = 0, sms = 0, group = 0;
    RerankShape rerank{};
    int64_t tiles = 0, ng = 0;
    float* x32 = nullptr;             // [n][dim] contiguous float32 rows
    uint16_t* xh = nullptr;           // [n][kpad] float16, and the bfloat16 copy: a run takes the format its queries want
    uint16_t* xb = nullptr;
    float* xn = nullptr;              // [tiles * 256], zero padded
    float* xst = nullptr;             // [kStats] the rows' statistics
    CUtensorMap tx16, txb;
    int64_t cap_q = 0;                // queries the scratch below holds
    uint16_t *qh = nullptr, *qb = nullptr;
    float *qn = nullptr, *qr16 = nullptr, *qrb = nullptr, *gmin = nullptr, *limit = nullptr, *dscr = nullptr;
    unsigned long long* cand = nullptr;
    int32_t *cnt = nullptr, *flags = nullptr;   // flags: [0] error, [1] unused overflow count; then the queries' statistics
};

namespace {
void plan_free_scratch(KnnPlan* p) {
    cudaFree(p->qh);
    cudaFree(p->qb);
    cudaFree(p->qn);
    cudaFree(p->qr16);
    cudaFree(p->qrb);
    cudaFree(p->gmin);
    cudaFree(p->limit);
    cudaFree(p->dscr);
    cudaFree(p->cand);
    cudaFree(p->cnt);
    cudaFree(p->flags);
    p->qh = nullptr;
    p->qb = nullptr;
    p->qn = p->qr16 = p->qrb = p->gmin = p->limit = p->dscr = nullptr;
    p->cand = nullptr;
    p->cnt = p->flags = nullptr;
    p->cap_q = 0;
}
}  // namespace

void knn_plan_destroy(KnnPlan* p) {
    if (!p) return;
    plan_free_scratch(p);
    cudaFree(p->x32);
    cudaFree(p->xh);
    cudaFree(p->xb);
    cudaFree(p->xn);
    cudaFree(p->xst);
    delete p;
}

int knn_plan_create(KnnPlan** out, const float* rows, int64_t row_stride, const int32_t* row_ids, int64_t n, int32_t dim,
                    int32_t k, int32_t cap, deg_stream_t stream, std::string* why) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    *out = nullptr;
    if (n < 1 || n > kPlanRowsMax || k < 1 || k > n || dim < 1 || cap < 1 || (cap & (cap - 1)))
        return *why = "knn plan: bad sizes", (int)cudaErrorInvalidValue;
    KnnPlan* p = new KnnPlan;
    p->n = n;
    p->dim = dim;
    p->kpad = (dim + KC - 1) / KC * KC;
    p->k = k;
    p->cap = cap;
    p->tiles = (n + TN - 1) / TN;
    p->group = (n + 63) / 64 >= 16 * (int64_t)k || k == 1 ? 64 : 16;
    p->ng = (n + p->group - 1) / p->group;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e;
    int rerank_max = 0;
    if ((e = cudaMalloc(&p->x32, 4ull * n * dim)) != cudaSuccess || (e = cudaMalloc(&p->xh, 2ull * n * p->kpad)) != cudaSuccess ||
        (e = cudaMalloc(&p->xb, 2ull * n * p->kpad)) != cudaSuccess || (e = cudaMalloc(&p->xn, 4ull * p->tiles * TN)) != cudaSuccess ||
        (e = cudaMalloc(&p->xst, 4ull * kStats)) != cudaSuccess || (e = open_smem_limits(&rerank_max)) != cudaSuccess) {
        knn_plan_destroy(p);
        return *why = std::string("knn plan: ") + cudaGetErrorString(e), (int)e;
    }
    p->rerank = rerank_shape(cap, dim, (int)n, rerank_max);
    cudaMemsetAsync(p->xn, 0, 4ull * p->tiles * TN, st);
    cudaMemsetAsync(p->xst, 0, 4ull * kStats, st);
    gather_plan_rows_kernel<<<256, 256, 0, st>>>(rows, row_stride, row_ids, n, dim, p->x32);
    half_rows_kernel<true, true, false, 1><<<(unsigned)((n + 7) / 8), 256, 0, st>>>(
        HalfRows{p->x32, n, dim, p->kpad, p->xh, p->xb, p->xn, nullptr, nullptr, p->xst, {}});
    if (!make_map(&p->tx16, p->xh, n, p->kpad, 2ull * p->kpad, TN) || !make_map(&p->txb, p->xb, n, p->kpad, 2ull * p->kpad, TN)) {
        knn_plan_destroy(p);
        return *why = "knn plan: tensor map encoding failed", (int)cudaErrorInvalidValue;
    }
    if ((e = cudaGetLastError()) == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        knn_plan_destroy(p);
        return *why = std::string("knn plan: ") + cudaGetErrorString(e), (int)e;
    }
    *out = p;
    return 0;
}

int knn_plan_run(KnnPlan* p, const float* queries, int64_t nq, int32_t* ids, float* dists, deg_stream_t stream,
                 std::string* why) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (nq <= 0) return 0;
    if (nq > (int64_t)1 << 24) return *why = "knn plan: too many queries", (int)cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    if (nq > p->cap_q) {                                  // grow the scratch (the only allocation)
        plan_free_scratch(p);
        const int64_t c = std::max<int64_t>(1024, (nq + TM - 1) / TM * TM);
        if ((e = cudaMalloc(&p->qh, 2ull * c * p->kpad)) != cudaSuccess || (e = cudaMalloc(&p->qb, 2ull * c * p->kpad)) != cudaSuccess ||
            (e = cudaMalloc(&p->qn, 4ull * c)) != cudaSuccess || (e = cudaMalloc(&p->qr16, 4ull * c)) != cudaSuccess ||
            (e = cudaMalloc(&p->qrb, 4ull * c)) != cudaSuccess || (e = cudaMalloc(&p->gmin, 4ull * c * p->ng)) != cudaSuccess ||
            (e = cudaMalloc(&p->limit, 4ull * c)) != cudaSuccess || (e = cudaMalloc(&p->dscr, 4ull * c * p->k)) != cudaSuccess ||
            (e = cudaMalloc(&p->cand, 8ull * c * p->cap)) != cudaSuccess || (e = cudaMalloc(&p->cnt, 4ull * c)) != cudaSuccess ||
            (e = cudaMalloc(&p->flags, 4ull * (4 + kStats))) != cudaSuccess) {
            plan_free_scratch(p);
            return *why = std::string("knn plan scratch: ") + cudaGetErrorString(e), (int)e;
        }
        p->cap_q = c;
    }
    const unsigned wblocks = (unsigned)((nq + 7) / 8);   // one warp per query, 8 per block
    if (p->k == 1 && p->n <= kPlanScanRows) {
        nearest_finish_kernel<true><<<wblocks, 256, 0, st>>>(nullptr, nullptr, 0, queries, p->x32, p->dim, p->n, nq, nullptr, nullptr, 0,
                                                             ids, dists ? dists : p->dscr, p->flags);
        if ((e = cudaGetLastError()) != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
        return 0;
    }
    CUtensorMap tq16, tqb;
    if (!make_map(&tq16, p->qh, nq, p->kpad, 2ull * p->kpad, TM) || !make_map(&tqb, p->qb, nq, p->kpad, 2ull * p->kpad, TM))
        return *why = "knn plan: tensor map encoding failed", (int)cudaErrorInvalidValue;
    const int32_t qblocks = (int32_t)((nq + TM - 1) / TM);
    const unsigned grid = (unsigned)std::min<int64_t>((int64_t)qblocks * p->tiles, p->sms);
    float* qst = reinterpret_cast<float*>(p->flags + 4);
    const Stats stats{p->xst, qst};
    cudaMemsetAsync(p->flags, 0, 4ull * (4 + kStats), st);
    cudaMemsetAsync(p->cnt, 0, 4ull * nq, st);
    half_rows_kernel<true, true, false, 1><<<(unsigned)std::min<int64_t>((nq + 7) / 8, 8 * p->sms), 256, 0, st>>>(
        HalfRows{queries, nq, p->dim, p->kpad, p->qh, p->qb, p->qn, p->qr16, p->qrb, qst, {}});
    const TcArgs sa{0, (int32_t)nq, qblocks, p->n, p->tiles, p->kpad / KC, p->qn, p->xn, p->gmin, p->group, qblocks * TM, nullptr, nullptr, nullptr, 0,
                    p->flags, stats};
    const TcArgs fa{0, (int32_t)nq, qblocks, p->n, p->tiles, p->kpad / KC, p->qn, p->xn, nullptr, 0, 0, p->limit, p->cand, p->cnt,
                    p->cap, p->flags, stats};
    dist_tc_kernel<false><<<grid, kTcThreads, kSmemDyn, st>>>(tq16, p->tx16, tqb, p->txb, sa);
    if (p->k == 1)
        nearest_limit_kernel<<<(unsigned)(qblocks * TM / 32), 128, 0, st>>>(p->gmin, (int)p->ng, qblocks * TM, nq, p->qn, p->qr16, p->qrb, stats, p->kpad, p->limit, p->cap, nullptr);
    else
        sample_limit_kernel<<<(unsigned)(qblocks * TM / kSelBatch), kSelThreads, 4 * (int)(p->ng | 1) * kSelBatch, st>>>(p->gmin, (int)p->ng, qblocks * TM, nq, p->k, kSelBatch, p->qn, p->qr16, p->qrb, stats, p->kpad,
                                                                  p->limit, groups_in_list(p->ng, p->group, p->n, p->cap), p->cap, p->cnt);
    dist_tc_kernel<true><<<grid, kTcThreads, kSmemDyn, st>>>(tq16, p->tx16, tqb, p->txb, fa);
    if (p->k == 1) {
        nearest_finish_kernel<false><<<wblocks, 256, 0, st>>>(p->cand, p->cnt, p->cap, queries, p->x32, p->dim, p->n, nq, nullptr, nullptr, 0,
                                                       ids, dists ? dists : p->dscr, p->flags);
    } else {
        const RerankArgs ra{p->cand, p->cnt, p->cap, p->k, queries, p->x32, p->dim, p->qn, p->qr16, p->qrb, stats, p->kpad,
                            ids, dists ? dists : p->dscr, p->flags + 1, (int32_t)p->n, p->flags};
        launch_rerank(ra, nq, p->rerank, st);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    return 0;
}

// ---- many rows to the nearest of a few (k-means, the locality layout) ---------------------------
// The same filter with the roles of a plan turned round: the many rows are the queries, converted
// once, and the few rows change from call to call. Labels and distances equal those of the CUDA-core
// kernel (float32 sums in dimension order, ties to the lower index). Rows go through in chunks whose
// group minima and candidate lists stay in L2.
//
// Where the rows lie far from the origin for their spread, the rounding window covers more of the few rows than a
// list holds. Such rows are left to the CUDA-core kernel, by a list; and where they are more than half, of the first
// chunk (where there are more than four) or of a whole run, that kernel takes all rows from there on. It scores a row in 12 times the time
// that the filter takes (500,000 x 1,953 x 128: 12 ms, 1.1 ms), so the filter pays up to nine tenths left over; half
// leaves room for the two passes over a row that it cannot decide.
struct RowAssign {
    static constexpr int64_t kChunk = 131072;
    static constexpr int kCap = 32;           // candidates per row; a row with more is left over
    int64_t n = 0;
    int32_t dim = 0, kpad = 0, kmax = 0, sms = 0;
    bool probed = false, off = false;
    const float* x = nullptr;                 // [n][dim], the caller's
    void* p[12] = {};
    CUtensorMap tq;
};

void row_assign_destroy(RowAssign* a) {
    if (!a) return;
    for (void* q : a->p) cudaFree(q);
    delete a;
}

// *out is null (and the result 0) where the path does not apply: too little work, rows that float16 does not hold
// well, or no memory for their copy.
int row_assign_create(RowAssign** out, const float* x, int64_t n, int32_t dim, int32_t kmax, deg_stream_t stream, std::string* why) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    *out = nullptr;
    if (n < 4096 || n * (int64_t)kmax < (1ll << 22) || kmax > kPlanRowsMax || n > INT32_MAX - TM || (reinterpret_cast<uintptr_t>(x) & 15))
        return 0;
    RowAssign* a = new RowAssign;
    a->n = n;
    a->dim = dim;
    a->kpad = (dim + KC - 1) / KC * KC;
    a->kmax = kmax;
    a->x = x;
    int dev = 0, unused = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&a->sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t npad = (n + TM - 1) / TM * TM, chunk = std::min<int64_t>(RowAssign::kChunk, npad);
    const int64_t tiles = (kmax + TN - 1) / TN;
    const size_t sizes[12] = {2ull * n * a->kpad, 4ull * npad, 4ull * npad, 4ull * (2 * kStats + 4),   // rows: copy, norms, residuals; stats, error, rows left
                              4ull * kmax * dim, 2ull * kmax * a->kpad, 4ull * tiles * TN,             // the few: float32, copy, norms
                              4ull * chunk * tiles * (TN / 64), 4ull * chunk, 8ull * chunk * RowAssign::kCap, 4ull * chunk,
                              4ull * n};                                                               // rows left
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 12 && e == cudaSuccess; ++i) e = cudaMalloc(&a->p[i], sizes[i]);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        row_assign_destroy(a);
        return 0;
    }
    if (e == cudaSuccess) e = open_smem_limits(&unused);
    float* qst = static_cast<float*>(a->p[3]) + kStats;
    float h[kStats] = {};
    if (e == cudaSuccess) e = cudaMemsetAsync(a->p[3], 0, sizes[3], st);
    if (e == cudaSuccess) {
        half_rows_kernel<true, false, false, 4><<<(unsigned)std::min<int64_t>((n + 31) / 32, 8 * a->sms), 256, 0, st>>>(
            HalfRows{x, n, dim, a->kpad, static_cast<uint16_t*>(a->p[0]), nullptr, static_cast<float*>(a->p[1]),
                     static_cast<float*>(a->p[2]), nullptr, qst, {}});
        e = cudaMemcpyAsync(h, qst, sizeof h, cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    const bool bf16 = h[kNoF16] != 0.f || h[kMaxRes16] > 0.001953125f * sqrtf(h[kMaxNorm]);   // wants_bf16
    if (e != cudaSuccess || bf16 || !make_map(&a->tq, a->p[0], n, a->kpad, 2ull * a->kpad, TM)) {
        row_assign_destroy(a);
        return e != cudaSuccess ? (*why = std::string("row assignment: ") + cudaGetErrorString(e), (int)e) : 0;
    }
    *out = a;
    return 0;
}

// labels[v] = the nearest of the k rows few[(ids ? ids[i] : i) * stride ...] to row v; dists (nullable) its distance.
// *left: the rows still to do, all of them if the few do not suit float16 or the lists are too short (nothing valid
// written then). Synchronises the stream.
int row_assign_run(RowAssign* a, const float* few, int64_t stride, const int32_t* ids, int32_t k, int32_t* labels, float* dists,
                   RowsLeft* left, deg_stream_t stream, std::string* why) {
    *left = RowsLeft{a->n, nullptr};
    if (a->off) return 0;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    auto* qn = static_cast<float*>(a->p[1]);
    auto* qr = static_cast<float*>(a->p[2]);
    auto* xst = static_cast<float*>(a->p[3]);
    auto* err = reinterpret_cast<int32_t*>(xst + 2 * kStats);
    auto* c32 = static_cast<float*>(a->p[4]);
    auto* ch = static_cast<uint16_t*>(a->p[5]);
    auto* cn = static_cast<float*>(a->p[6]);
    auto* gmin = static_cast<float*>(a->p[7]);
    auto* limit = static_cast<float*>(a->p[8]);
    auto* cand = static_cast<unsigned long long*>(a->p[9]);
    auto* cnt = static_cast<int32_t*>(a->p[10]);
    auto* rest = static_cast<int32_t*>(a->p[11]);
    const Stats stats{xst, xst + kStats};
    const int64_t tiles = (k + TN - 1) / TN;
    const int32_t ng = (k + 63) / 64;
    CUtensorMap tx;
    if (!make_map(&tx, ch, k, a->kpad, 2ull * a->kpad, TN)) return *why = "tensor map encoding failed", (int)cudaErrorInvalidValue;
    cudaMemsetAsync(xst, 0, 4ull * kStats, st);
    cudaMemsetAsync(err, 0, 16, st);
    cudaMemsetAsync(cn, 0, 4ull * tiles * TN, st);
    gather_plan_rows_kernel<<<256, 256, 0, st>>>(few, stride, ids, k, a->dim, c32);
    half_rows_kernel<true, false, false, 1><<<(unsigned)((k + 7) / 8), 256, 0, st>>>(
        HalfRows{c32, k, a->dim, a->kpad, ch, nullptr, cn, nullptr, nullptr, xst, {}});
    // the state of the run after the rows so far: whether the few suit float16, the error flag and the rows left
    int32_t flags[2] = {};
    auto sync = [&](bool* suits) {
        float h[kStats] = {};
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, xst, sizeof h, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(flags, err, sizeof flags, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return *why = std::string("row assignment: ") + cudaGetErrorString(e), (int)e;
        if (flags[0]) return *why = "a tensor-core wait exceeded its limit", (int)cudaErrorLaunchTimeout;
        *suits = h[kNoF16] == 0.f && h[kMaxRes16] <= 0.001953125f * sqrtf(h[kMaxNorm]);
        return 0;
    };
    bool suits = false;
    for (int64_t q0 = 0, qc; q0 < a->n; q0 += qc) {
        const bool probe = !a->probed && q0 == 0 && a->n > 4 * RowAssign::kChunk;
        qc = std::min(RowAssign::kChunk, a->n - q0);
        const int32_t qblocks = (int32_t)((qc + TM - 1) / TM);
        const unsigned grid = (unsigned)std::min<int64_t>((int64_t)qblocks * tiles, a->sms);
        const TcArgs sa{(int32_t)q0, (int32_t)qc, qblocks, k, tiles, a->kpad / KC, qn + q0, cn, gmin, 64, qblocks * TM, nullptr, nullptr, nullptr, 0, err, stats};
        const TcArgs fa{(int32_t)q0, (int32_t)qc, qblocks, k, tiles, a->kpad / KC, qn + q0, cn, nullptr, 0, 0, limit, cand, cnt, RowAssign::kCap, err, stats};
        dist_tc_kernel<false><<<grid, kTcThreads, kSmemDyn, st>>>(a->tq, tx, a->tq, tx, sa);
        nearest_limit_kernel<<<(unsigned)(qblocks * TM / 32), 128, 0, st>>>(gmin, ng, qblocks * TM, qc, qn + q0, qr + q0, qr + q0, stats, a->kpad, limit, RowAssign::kCap, cnt);
        dist_tc_kernel<true><<<grid, kTcThreads, kSmemDyn, st>>>(a->tq, tx, a->tq, tx, fa);
        nearest_finish_kernel<false><<<(unsigned)((qc + 7) / 8), 256, 0, st>>>(cand, cnt, RowAssign::kCap, a->x + q0 * a->dim, c32, a->dim, k, qc,
                                                                       rest, err + 1, (int32_t)q0, labels + q0, dists ? dists + q0 : nullptr, err);
        if (probe) {
            if (const int r = sync(&suits)) return r;
            if (!suits) return 0;
            a->off = 2 * (int64_t)flags[1] > qc;
            if (a->off) return 0;
        }
    }
    if (const int r = sync(&suits)) return r;
    if (!suits) return 0;
    a->probed = true;
    a->off = 2 * (int64_t)flags[1] > a->n;
    *left = RowsLeft{flags[1], rest};
    return 0;
}

}  // namespace deg
