// Small batches: the search of search_impl.cuh with a block of eight warps per query.
//
// A small batch is bound by the time of one hop, not by throughput: one warp that runs a query alone on
// its SM spends 3 to 4 us a hop (7,500 cycles: about 1,000 instructions issued one after the other
// between two global round trips and an atomic's). Here a hop's work is spread over the block:
//   distances   the eight warps take the new rows in turn, all of them in flight at once; a row is summed
//               by the same lanes in the same order as in search_impl.cuh, so distances are bit-identical.
//               The adjacency rows of the new vertices are prefetched into L2 meanwhile;
//   the runner  (the last warp) then goes ahead: the next vertex to pop is the smaller of the front's head
//               and the smallest new key, whatever the merge does, so it reads that vertex's adjacency
//               row, marks its neighbours and lists the new ones while the other warps finish this hop
//               (if the radius after the hop ends the search, what it marked no longer matters);
//   the others  rank the new keys, a key a lane: warp 0 in R, warp 1 in the front of S, the rest among
//               themselves; then warp 0 merges R and warps 1 to 5 the front into their second buffers.
// Two block barriers a hop, one among the seven. The checked set C is a bitmap in shared memory (1M
// vertices: 125 KB), so test-and-set costs no L2 round trip and nothing is left to clear in device memory.
// A float32 hop takes about 3,000 cycles (1M x 128, idle SM): 1,250 for the rows, the rest for ranks and
// merge, which hide the runner's 1,000; reading adjacency rows ahead into shared memory made the first
// part 500 cycles longer and saved the runner's wait only.
//
// R, S and C hold the same sets after every hop as in the one-warp kernel (front of kFront keys,
// watermark, back pool, the same refills), so results, H, E and the peak of S are the same. A back pool that fills is
// cleared of the keys outside the radius before the hop's keys go in, in the one-warp kernel
// between them: the peak of S may differ by a few keys then, and nothing else. A query whose pool is still full
// starts again with room for all n vertices: in the second kernel, or, direct, in its own block.
// The keys that enter R, the front or S at all are each the smallest of the hop's (the tests are thresholds on the
// key), so one order among the hop's keys serves all three.
//
// Measured, 1M x 128, whole calls, the queries of one seed: one fp8 query from the learned entry points (52 hops)
// 241 -> 104 us, 64 float32 queries from the pivots, the longest of 270 hops, 1,050 -> 402 us. The longest walk sets
// both times, so other queries take 80 to 105 us and 150 to 430 us, and as much less than before. Where the line to
// the one-warp kernel lies: use_wide (search.cu).
#ifndef DEG_SEARCH_WIDE_CUH
#define DEG_SEARCH_WIDE_CUH

#include <type_traits>

#include "search_impl.cuh"

namespace deg {
namespace sk {

constexpr int kWideWarps = 8, kWideThreads = 32 * kWideWarps;
constexpr int kWords = kMaxDegree / 32;   // 32-key words of a hop's new neighbours, at most
constexpr int kWideKept = 128;            // results kept, at most
constexpr int kWideDirect = 64;           // queries that run without a cursor, at most

// Block state besides the bitmap and the query.
struct WideShared {
    uint64_t front[2][kFront];            // sorted ascending, from `f0` on
    uint64_t res[2][kWideKept];           // R, sorted ascending
    int32_t cid[2][kMaxDegree];           // the new neighbours' internal ids
    int32_t ccid[2][kMaxDegree];          //   and caller ids
    uint64_t key[kMaxDegree];             //   and search keys
    int32_t order[kMaxDegree];            //   how many of them are below each,
    int32_t rpos[kMaxDegree];             //   how many of R's keys
    int32_t fpos[kMaxDegree];             //   and of the front's
    uint32_t hist[256];                   // refill
    uint64_t red[kWideWarps];
    uint64_t next_key;                    // the runner's vertex (kEmptyKey: none in the front) and
    int32_t next_cnt;                     //   how many new neighbours it has
    int32_t again[3];                     // {state, vertices popped, new neighbours} of a pop from the front as it stands
    int32_t refilled[2];                  // front keys, back keys
    uint64_t refill_mark;
    uint64_t wmark;                       // the scalars of the search after a merge, for the runner
    int32_t rn, fn, back_n, peak, lost, trimmed;
    float r2;
    int32_t query;
    int32_t tier;                         // 1: a second pass, with room in the pool for all n vertices
    int32_t pad[3];
};

static_assert(sizeof(WideShared) % 16 == 0, "the query and the bitmap behind it are read and cleared 16 bytes at a time");

enum { kWideGo, kWideStop, kWideRefill, kWideHopLimit };

__host__ __device__ inline int64_t wide_bytes(int64_t words, int dim) {
    return (int64_t)sizeof(WideShared) + 4 * ((dim + 15) / 16 * 16) + 4 * words;
}

// The keys of cid[0 .. cnt) by all warps: Engine::distances with the rows dealt to the warps in turn.
template <class Rows, int G, int CPL>
__device__ __forceinline__ void wide_distances(const Engine<Rows, G, CPL>& eng, const Params& P, const int32_t* cid, const int32_t* ccid,
                                               uint64_t* key, int cnt, int warp, int lane) {
    constexpr int RP = 32 / G, U = G == 32 && CPL == 1 ? 4 : G >= 16 && CPL <= 2 ? 2 : 1;
    const int g = lane / G, p = lane % G;
    for (int i0 = 0; i0 + warp * RP < cnt; i0 += kWideWarps * RP * U) {
        uint4 buf[U][CPL];
        float2 sc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + (u * kWideWarps + warp) * RP + g;
            sc[u] = make_float2(1.f, 0.f);
#pragma unroll
            for (int j = 0; j < CPL; ++j) buf[u][j] = make_uint4(0, 0, 0, 0);
            if (i < cnt) {
                const int32_t id = cid[i];
                const uint8_t* row = P.rows + (int64_t)id * P.row_bytes;
                sc[u] = Rows::scale(P.norm8, id);
#pragma unroll
                for (int j = 0; j < CPL; ++j) {
                    const int c = p + G * j;
                    if (c < P.nchunk) buf[u][j] = __ldg(reinterpret_cast<const uint4*>(row) + c);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + (u * kWideWarps + warp) * RP >= cnt) break;              // warp-uniform
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int j = 0; j < CPL; ++j)
                if (p + G * j < P.nchunk) Rows::acc(buf[u][j], eng.q[j], a0, a1);
            float a = a0 + a1;
#pragma unroll
            for (int m = G / 2; m; m >>= 1) a += __shfl_xor_sync(0xffffffffu, a, m);
            const int i = i0 + (u * kWideWarps + warp) * RP + g;
            if (p == 0 && i < cnt) key[i] = make_key(Rows::fin(a, sc[u], eng.qq), ccid[i]);
        }
    }
}

// N(G, s) \ C into cid / ccid, C <- C u N; one warp. Returns their number.
__device__ __forceinline__ int wide_expand(const Params& P, uint32_t* bitmap, int32_t s, int32_t* cid, int32_t* ccid, int lane) {
    int cnt = 0;
    for (int j0 = 0; j0 < P.degree; j0 += 32) {
        const int j = j0 + lane;
        const int2 e = j < P.degree ? __ldg(P.adj + (int64_t)s * P.deg_pad + j) : make_int2(-1, -1);
        const int isnew = e.x >= 0 ? visit(bitmap, e.x) : 0;
        const unsigned nm = __ballot_sync(0xffffffffu, isnew);
        if (isnew) {
            const int at = cnt + __popc(nm & lanes_below(lane));
            cid[at] = e.x;
            ccid[at] = e.y;
        }
        cnt += __popc(nm);
    }
    return cnt;
}

// Number of keys below `key` in the ascending a[0 .. n), n <= kFront or kWideKept: three probes a step, without branches
// (four steps of independent reads instead of eight dependent ones). a[0] may be read when n = 0.
constexpr int kCountStep = kFront <= 128 && kWideKept <= 128 ? 32 : 128;   // four steps cover 4 kCountStep keys
static_assert(kFront <= 4 * kCountStep && kWideKept <= 4 * kCountStep, "the front and R fit the ranking steps");
__device__ __forceinline__ int count_below(const uint64_t* a, int n, uint64_t key) {
    int lo = 0;
#pragma unroll
    for (int step = kCountStep; step >= 2; step >>= 2) {
        int add = 0;
#pragma unroll
        for (int t = 1; t <= 3; ++t) {
            const int i = lo + t * step;
            const uint64_t v = a[i <= n ? i - 1 : 0];
            add += (i <= n) & (v < key);
        }
        lo += add * step;
    }
    const uint64_t u = a[lo < n ? lo : 0], v = a[lo + 1 < n ? lo + 1 : 0];   // at most two more
    return lo + ((lo < n) & (u < key)) + ((lo + 1 < n) & (v < key));
}

// Barrier of the warps beside the runner.
__device__ __forceinline__ void merge_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kWideThreads - 32) : "memory"); }

struct WideArgs {
    int32_t direct;                       // 1: block b runs query b, no cursor
    const unsigned long long* part;       // routing of a few queries: [nparts][nq] keys d2 << 32 | pivot, or null
    int32_t nparts;
    const int32_t* pivots;                // internal ids
    uint64_t* backs;                      // [grid][bstride] back pools
    int64_t bstride;
    int32_t bcap;                         // keys a query may hold there; direct: any number in a second pass, if it
                                          //   outgrew bcap (the pool of n + 1 keys has room for all)
    int32_t smem_max, sms;                // of the device, for the launch
};

// Blocks an SM that the registers leave room for. Float32 rows of one chunk a lane run in 80 registers, three blocks
// (the bitmap allows them up to about 500,000 vertices), the others in 128, two blocks, but for the widest fp8 rows,
// whose query alone takes 128. Stated, since one register more had the compiler take 124 and two blocks for the first
// (200k x 128, exploration k = 100, 400 queries: 375 us, 238 with three); so what a query keeps for its rare second pass is in shared memory, and read only where a pool is full.
template <class Rows, int CPL>
constexpr int wide_blocks() {
    return Rows::EPC == 4 && CPL == 1 ? 3 : Rows::EPC == 16 && CPL == 8 ? 1 : 2;
}

template <class Rows, int G, int CPL>
__global__ void __launch_bounds__(kWideThreads, wide_blocks<Rows, CPL>()) search_wide_kernel(const Params P, const WideArgs A) {
    extern __shared__ __align__(16) uint8_t smem[];
    WideShared& S = *reinterpret_cast<WideShared*>(smem);
    float* qv = reinterpret_cast<float*>(smem + sizeof(WideShared));
    const int dim16 = (P.dim + 15) / 16 * 16;
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(qv + dim16);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float inf = __int_as_float(0x7f800000);
    uint64_t* back = A.backs + (int64_t)blockIdx.x * A.bstride;
    if (tid == 0) S.tier = 0;
    for (int round = 0;; ++round) {
        if (A.direct) {
            if (round > 0 && round > S.tier) break;
        } else if (tid == 0) {
            const int t = atomicAdd(P.counters + 2, 1);
            S.query = t >= P.nq ? P.nq : P.order ? P.order[t] : t;
        }
        __syncthreads();
        const int q = A.direct ? (int)blockIdx.x : S.query;
        if (q >= P.nq) break;

        // the seed, as in run_query; or the nearest pivot from the partial minima (-1 where no distance
        // is finite, as the batch routing reports it)
        bool given = P.explore || P.seeds, internal = P.seeds_internal != 0;
        int32_t seed_in = given ? P.seeds[q] : 0;
        if (A.part) {
            uint64_t v = kEmptyKey;
            for (int b = tid; b < A.nparts; b += kWideThreads) v = min(v, (uint64_t)A.part[(int64_t)b * P.nq + q]);
            v = warp_min64(v);
            if (lane == 0) S.red[warp] = v;
            __syncthreads();
            for (int w = 0; w < kWideWarps; ++w) v = min(v, S.red[w]);
            seed_in = (uint32_t)(v >> 32) < 0x7f800000u ? A.pivots[key_id(v)] : -1;
            given = internal = true;
        }
        const bool seed_ok = !given || (seed_in >= 0 && seed_in < P.n);
        const int32_t seed = !given ? P.entry : !seed_ok ? 0 : internal ? seed_in : __ldg(P.old2new + seed_in);
        const int32_t seed_c = !given ? P.entry_caller : !seed_ok ? 0 : internal ? __ldg(P.new2old + seed_in) : seed_in;
        const float* qsrc = P.explore ? P.x32 + (int64_t)seed * P.dim_pad : P.queries + (int64_t)q * P.dim;
        for (int i = tid; i < dim16; i += kWideThreads) qv[i] = i < P.dim ? qsrc[i] : 0.f;
        uint4* b4 = reinterpret_cast<uint4*>(bitmap);
        for (int i = tid; i < (int)(P.words / 4); i += kWideThreads) b4[i] = make_uint4(0, 0, 0, 0);
        if (tid == 0) {
            S.cid[0][0] = seed;
            S.ccid[0][0] = seed_c;
        }
        __syncthreads();
        Engine<Rows, G, CPL> eng;
        eng.load_query(qv, P.dim, lane);
        wide_distances(eng, P, S.cid[0], S.ccid[0], S.key, 1, warp, lane);
        if (tid == 0) visit(bitmap, seed);
        __syncthreads();

        // every thread carries the scalars of the search; they change alike in all
        int fb = 0, f0 = 0, fn = 1, rb = 0, rn = P.explore || !seed_ok ? 0 : 1, cb = 0, cnt = 0;
        int back_n = 0, hops = 0, evals = 1, peak = 1, status = seed_ok ? DEG_OK : DEG_EINVAL;
        uint64_t wmark = kEmptyKey;
        bool trimmed = false, again = true, lost = false;
        float r2 = inf;
        if (tid == 0) {
            S.front[0][0] = S.key[0];
            S.res[0][0] = S.key[0];
        }
        if (!seed_ok) hops = evals = peak = 0;
        __syncthreads();
        while (seed_ok) {
            if (again) {
                // pop from the front as it stands: at the start, after a refill, and after a vertex
                // with no new neighbour
                if (warp == kWideWarps - 1) {
                    const Radius thr{trimmed ? r2 : inf, P.f, P.f_lo};
                    int state = kWideStop, pops = 0, c = 0;
                    for (;;) {
                        if (pops == fn) {
                            state = back_n > 0 ? kWideRefill : kWideStop;
                            break;
                        }
                        const uint64_t m = S.front[fb][f0 + pops];
                        if (!thr.admits(key_d2(m))) break;
                        if (P.max_hops && hops + pops >= P.max_hops) {
                            state = kWideHopLimit;
                            break;
                        }
                        ++pops;
                        c = wide_expand(P, bitmap, key_id(m), S.cid[cb], S.ccid[cb], lane);
                        if (c > 0) {
                            state = kWideGo;
                            break;
                        }
                    }
                    if (lane == 0) {
                        S.again[0] = state;
                        S.again[1] = pops;
                        S.again[2] = c;
                    }
                }
                __syncthreads();
                const int state = S.again[0], pops = S.again[1];
                cnt = S.again[2];
                f0 += pops;
                fn -= pops;
                hops += pops;
                if (state == kWideRefill) {
                    if (warp == 0) {
                        WarpState W;
                        W.front = S.front[0];
                        W.cid = reinterpret_cast<int32_t*>(S.hist);
                        W.back = back;
                        W.back_n = back_n;
                        W.sorted = false;
                        refill(W, Radius{trimmed ? r2 : inf, P.f, P.f_lo}, lane);
                        for (int i = W.fn + lane; i < kFront; i += 32) W.front[i] = kEmptyKey;
                        __syncwarp();
                        for (int size = 2; size <= kFront; size <<= 1)
                            for (int stride = size >> 1; stride; stride >>= 1) {
                                for (int t = lane; t < kFront / 2; t += 32) {
                                    const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                                    const bool up = (lo & size) == 0;
                                    const uint64_t a = W.front[lo], b = W.front[hi];
                                    if ((a > b) == up) { W.front[lo] = b; W.front[hi] = a; }
                                }
                                __syncwarp();
                            }
                        if (lane == 0) {
                            S.refilled[0] = W.fn;
                            S.refilled[1] = W.back_n;
                            S.refill_mark = W.wmark;
                        }
                    }
                    __syncthreads();
                    fb = f0 = 0;
                    fn = S.refilled[0];
                    back_n = S.refilled[1];
                    wmark = S.refill_mark;
                    if (fn == 0) break;
                    continue;
                }
                if (state == kWideHopLimit) status = DEG_EHOPLIMIT;
                if (state != kWideGo) break;
                again = false;
            }
            evals += cnt;

            // squared distances of the new neighbours
            if (warp == kWideWarps - 2)
                for (int i = lane; i < cnt; i += 32) {
                    const int2* row = P.adj + (int64_t)S.ccid[cb][i] * P.deg_pad;
                    for (int b = 0; b < P.deg_pad; b += 16) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + b));
                }
            wide_distances(eng, P, S.cid[cb], S.ccid[cb], S.key, cnt, warp, lane);
            __syncthreads();

            if (warp == kWideWarps - 1) {
                const uint64_t head = fn > 0 ? S.front[fb][f0] : kEmptyKey;
                uint64_t m = lane < cnt ? S.key[lane] : kEmptyKey;
                for (int i = 32 + lane; i < cnt; i += 32) m = min(m, S.key[i]);
                m = warp_min64(m);
                m = m < wmark ? min(m, head) : head;          // a new key above the watermark goes to the back pool
                const int c = m == kEmptyKey ? 0 : wide_expand(P, bitmap, key_id(m), S.cid[cb ^ 1], S.ccid[cb ^ 1], lane);
                if (lane == 0) {
                    S.next_key = m;
                    S.next_cnt = c;
                }
            } else {
                // ranks and merges, with the words of new keys known at compile time: nearly always one
                auto merge = [&](auto words) {
                    constexpr int NW = decltype(words)::value;
                    // a lane's keys (one for every 32 new neighbours)
                    uint64_t key[NW];
#pragma unroll
                    for (int w = 0; w < NW; ++w) key[w] = 32 * w + lane < cnt ? S.key[32 * w + lane] : kEmptyKey;
                    if (warp < 2) {
                        const uint64_t* a = warp == 0 ? S.res[rb] : S.front[fb] + f0;
                        int32_t* to = warp == 0 ? S.rpos : S.fpos;
                        const int n = warp == 0 ? rn : fn;
#pragma unroll
                        for (int w = 0; w < NW; ++w)
                            if (32 * w + lane < cnt) to[32 * w + lane] = count_below(a, n, key[w]);
                    } else {
#pragma unroll 2
                        for (int i = warp - 2; i < cnt; i += kWideWarps - 3) {
                            const uint64_t other = S.key[i];
                            int r = 0;
#pragma unroll
                            for (int w = 0; w < NW; ++w) r += __popc(__ballot_sync(0xffffffffu, key[w] < other));
                            if (lane == 0) S.order[i] = r;
                        }
                    }
                    merge_barrier();
                    int order[NW], rpos[NW], fpos[NW];
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        order[w] = S.order[32 * w + lane];    // undefined past cnt, and not used there
                        rpos[w] = S.rpos[32 * w + lane];
                        fpos[w] = S.fpos[32 * w + lane];
                    }

                    // R <- R u {n : d(n) <= r}, the ks smallest: a new key's merged index is rank + place; the
                    // others keep their order around them. The radius after the hop is the merged list's last key.
                    const float r2pre = trimmed ? r2 : inf;
                    int m_r = 0, at_last = 0, kn[NW];
                    uint64_t last = 0;
                    bool last_new = false;
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        const bool take = 32 * w + lane < cnt && key_d2(key[w]) <= r2pre;
                        kn[w] = take ? order[w] + rpos[w] : 0x7fffffff;
                        m_r += __popc(__ballot_sync(0xffffffffu, take));
                        at_last += __popc(__ballot_sync(0xffffffffu, kn[w] < P.ks - 1));
                        const unsigned is = __ballot_sync(0xffffffffu, kn[w] == P.ks - 1);
                        if (is) {
                            last = shfl64(key[w], __ffs(is) - 1);
                            last_new = true;
                        }
                    }
                    // old keys of slots 32 c ... 32 c + 31 of a merge in which the new keys take the indices kn
                    auto old_of = [&](int c, int& from) {
                        int below = 0;
                        unsigned word = 0;
#pragma unroll
                        for (int w = 0; w < NW; ++w) {
                            below += __popc(__ballot_sync(0xffffffffu, kn[w] < 32 * c));
                            word |= __reduce_or_sync(0xffffffffu, (kn[w] >> 5) == c ? 1u << (kn[w] & 31) : 0u);
                        }
                        from = 32 * c + lane - below - __popc(word & lanes_below(lane));
                        return ((word >> lane) & 1u) == 0;
                    };
                    const int total_r = min(rn + m_r, P.ks);
                    if (warp == 0) {
                        for (int c = 0; 32 * c < total_r; ++c) {
                            int from;
                            const bool old = old_of(c, from);
                            if (old && 32 * c + lane < total_r) S.res[rb ^ 1][32 * c + lane] = S.res[rb][from];
                        }
                    }
                    if (warp == 6) {
#pragma unroll
                        for (int w = 0; w < NW; ++w)
                            if (kn[w] < P.ks) S.res[rb ^ 1][kn[w]] = key[w];
                    }
                    if (rn + m_r > P.ks) {
                        if (!last_new) last = S.res[rb][P.ks - 1 - at_last];
                        trimmed = true;
                        r2 = key_d2(last);
                    }
                    rn = total_r;

                    // S <- S u {n : d(n) <= r (1 + eps)} for the radius after the hop
                    const Radius thr{trimmed ? r2 : inf, P.f, P.f_lo};
                    int m_f = 0, m_b = 0, at_edge = 0, kb[NW];
                    uint64_t edge = kEmptyKey;
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        const bool take = 32 * w + lane < cnt && thr.admits(key_d2(key[w])), to_f = take && key[w] < wmark;
                        kn[w] = to_f ? order[w] + fpos[w] : 0x7fffffff;
                        const unsigned mb = __ballot_sync(0xffffffffu, take && !to_f);
                        kb[w] = take && !to_f ? m_b + __popc(mb & lanes_below(lane)) : -1;
                        m_f += __popc(__ballot_sync(0xffffffffu, to_f));
                        m_b += __popc(mb);
                        if (fn + cnt > kFront) {
                            at_edge += __popc(__ballot_sync(0xffffffffu, kn[w] < kFront));
                            const unsigned is = __ballot_sync(0xffffffffu, kn[w] == kFront);
                            if (is) edge = shfl64(key[w], __ffs(is) - 1);
                        }
                    }
                    const int total_f = fn + m_f, evicted = max(0, total_f - kFront);
                    if (back_n + m_b + evicted > A.bcap && S.tier == 0) {
                        // no room: drop the back keys outside the radius; if that is not enough, the query
                        // starts again
                        merge_barrier();
                        if (warp == 0) {
                            int out = 0;
                            for (int i0 = 0; i0 < back_n; i0 += 32) {
                                const int i = i0 + lane;
                                const uint64_t v = i < back_n ? back[i] : kEmptyKey;
                                const bool keep = i < back_n && thr.admits(key_d2(v));
                                const unsigned m = __ballot_sync(0xffffffffu, keep);
                                __syncwarp();
                                if (keep) back[out + __popc(m & lanes_below(lane))] = v;
                                out += __popc(m);
                                __syncwarp();
                            }
                            if (lane == 0) S.refilled[1] = out;
                        }
                        merge_barrier();
                        back_n = S.refilled[1];
                        lost = back_n + m_b + evicted > A.bcap;
                    }
                    if (!lost) {
                        if (evicted > 0 && edge == kEmptyKey) edge = S.front[fb][f0 + kFront - at_edge];
                        if (warp >= 1 && warp <= 5)
                            for (int c = warp - 1; 32 * c < total_f; c += 5) {
                                int from;
                                const bool old = old_of(c, from);
                                const int slot = 32 * c + lane;
                                if (old && slot < total_f) {
                                    const uint64_t v = S.front[fb][f0 + from];
                                    if (slot < kFront) S.front[fb ^ 1][slot] = v;
                                    else back[back_n + m_b + slot - kFront] = v;
                                }
                            }
                        if (warp == 6) {                      // the new keys
#pragma unroll
                            for (int w = 0; w < NW; ++w) {
                                if (kn[w] < kFront) S.front[fb ^ 1][kn[w]] = key[w];
                                else if (kn[w] != 0x7fffffff) back[back_n + m_b + kn[w] - kFront] = key[w];
                                if (kb[w] >= 0) back[back_n + kb[w]] = key[w];
                            }
                        }
                        back_n += m_b + evicted;
                        fn = total_f - evicted;
                        if (evicted > 0) wmark = edge;
                        peak = max(peak, fn + back_n);
                    }
                };
                if (cnt <= 32) merge(std::integral_constant<int, 1>{});
                else merge(std::integral_constant<int, kWords>{});
                if (tid == 0) {
                    S.rn = rn;
                    S.fn = fn;
                    S.back_n = back_n;
                    S.peak = peak;
                    S.lost = lost;
                    S.wmark = wmark;
                    S.trimmed = trimmed;
                    S.r2 = r2;
                }
            }
            f0 = 0;
            fb ^= 1;
            rb ^= 1;
            cb ^= 1;
            __syncthreads();
            if (warp == kWideWarps - 1) {
                rn = S.rn;
                fn = S.fn;
                back_n = S.back_n;
                peak = S.peak;
                lost = S.lost != 0;
                wmark = S.wmark;
                trimmed = S.trimmed != 0;
                r2 = S.r2;
            }
            if (lost) break;
            const uint64_t m = S.next_key;
            again = true;
            if (m == kEmptyKey) continue;                     // the front is empty: refill, or the end
            if (!Radius{trimmed ? r2 : inf, P.f, P.f_lo}.admits(key_d2(m))) break;
            if (P.max_hops && hops >= P.max_hops) {
                status = DEG_EHOPLIMIT;
                break;
            }
            ++hops;
            f0 = 1;
            --fn;
            cnt = S.next_cnt;
            again = cnt == 0;
        }
        __syncthreads();
        if (lost) {
            if (A.direct && tid == 0) S.tier = 1;
            else if (tid == 0) P.overflow[atomicAdd(P.counters, 1)] = q;
            __syncthreads();
            continue;
        }

        // the results: re-ranked on the float32 rows if asked, then written out
        uint64_t* res = S.res[rb];
        if (P.rerank) {
            for (int i = tid; i < P.kcap; i += kWideThreads) {
                const int32_t id = i < rn ? key_id(res[i]) : 0;
                res[i] = i < rn ? make_key(exact_d2_lane(P.x32, P.dim_pad, __ldg(P.old2new + id), qv), id) : kEmptyKey;
            }
            __syncthreads();
            if (warp == 0)
                for (int size = 2; size <= P.kcap; size <<= 1)
                    for (int stride = size >> 1; stride; stride >>= 1) {
                        for (int t = lane; t < P.kcap / 2; t += 32) {
                            const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                            const bool up = (lo & size) == 0;
                            const uint64_t a = res[lo], b = res[hi];
                            if ((a > b) == up) { res[lo] = b; res[hi] = a; }
                        }
                        __syncwarp();
                    }
            __syncthreads();
        }
        for (int i = tid; i < P.k; i += kWideThreads) {
            const bool ok = i < rn;
            const uint64_t v = ok ? res[i] : kEmptyKey;
            P.ids[(int64_t)q * P.k + i] = ok ? key_id(v) : -1;
            P.dists[(int64_t)q * P.k + i] = ok ? sqrtf(key_d2(v)) : inf;
        }
        if (tid == 0) {
            if (P.status) P.status[q] = status;
            if (P.trace) {
                P.trace[4 * (int64_t)q + 0] = hops;
                P.trace[4 * (int64_t)q + 1] = evals;
                P.trace[4 * (int64_t)q + 2] = peak;
                P.trace[4 * (int64_t)q + 3] = S.tier;
            }
        }
        __syncthreads();
    }
}

// Launches the kernel on min(nq, resident blocks) blocks, with a cursor over the queries; or, direct, on a
// block per query and without the second kernel (whose pools are used).
template <class Rows, int G, int CPL>
int launch_wide(const Params& P, WideArgs A, cudaStream_t st, void* timer_start, void* timer_end, std::string* why) {
    cudaError_t e;
    const int smem = (int)wide_bytes(P.words, P.dim);
    auto k = search_wide_kernel<Rows, G, CPL>;
    if ((e = open_smem(k, A.smem_max)) != cudaSuccess)
        return *why = std::string("shared memory attribute: ") + cudaGetErrorString(e), (int)e;
    int64_t grid = P.nq;
    if (!A.direct) {
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kWideThreads, (size_t)smem)) != cudaSuccess)
            return *why = "occupancy query failed", (int)e;
        grid = std::max<int64_t>(1, std::min<int64_t>({grid, (int64_t)A.sms * per_sm, (int64_t)P.slots}));
        if ((e = cudaMemsetAsync(P.counters, 0, 4 * sizeof(int32_t), st)) != cudaSuccess) return *why = "memset", (int)e;
    }
    if (timer_start && (e = cudaEventRecord(static_cast<cudaEvent_t>(timer_start), st)) != cudaSuccess)
        return *why = "timer event", (int)e;
    k<<<(unsigned)grid, kWideThreads, smem, st>>>(P, A);
    if ((e = cudaGetLastError()) != cudaSuccess) return *why = std::string("wide kernel: ") + cudaGetErrorString(e), (int)e;
    if (!A.direct)
        if (const int r = launch_second<Rows, G, CPL>(P, st, why)) return r;
    if (timer_end && (e = cudaEventRecord(static_cast<cudaEvent_t>(timer_end), st)) != cudaSuccess)
        return *why = "timer event", (int)e;
    return 0;
}

template <class Rows>
int dispatch_wide(const Params& P, const WideArgs& A, cudaStream_t st, void* t0, void* t1, std::string* why) {
    const int nc = P.nchunk;
    if (nc <= 4) return launch_wide<Rows, 4, 1>(P, A, st, t0, t1, why);
    if (nc <= 8) return launch_wide<Rows, 8, 1>(P, A, st, t0, t1, why);
    if (nc <= 16) return launch_wide<Rows, 16, 1>(P, A, st, t0, t1, why);
    if (nc <= 32) return launch_wide<Rows, 32, 1>(P, A, st, t0, t1, why);
    if (nc <= 64) return launch_wide<Rows, 32, 2>(P, A, st, t0, t1, why);
    if (nc <= 128) return launch_wide<Rows, 32, 4>(P, A, st, t0, t1, why);
    if (nc <= 256) return launch_wide<Rows, 32, 8>(P, A, st, t0, t1, why);
    *why = "row too wide (at most 4096 bytes)";
    return (int)cudaErrorInvalidValue;
}

int dispatch_wide_f32(const Params& P, const WideArgs& A, cudaStream_t st, void* t0, void* t1, std::string* why);
int dispatch_wide_bf16(const Params& P, const WideArgs& A, cudaStream_t st, void* t0, void* t1, std::string* why);
int dispatch_wide_fp8(const Params& P, const WideArgs& A, cudaStream_t st, void* t0, void* t1, std::string* why);

}  // namespace sk
}  // namespace deg

#endif
