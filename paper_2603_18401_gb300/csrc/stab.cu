// Candidate retrieval and candidate-restricted matching.
//
//   stab_kernel       one warp per query (Sec. 4.2 "query"; Algorithm 1,
//                     Match loop).  Lane l computes the angle window of level
//                     l, the largest angular radius among that level's
//                     keypoints widened by the line's distance from the
//                     epipole, then the warp walks the concatenated windows
//                     32 keypoints at a time.  Each keypoint in a window gets
//                     the point-to-line test of Eq. 3 / Eq. 4: an FP32 test
//                     with a rigorous error bound, and, only when that is not
//                     conclusive, the FP64 expression of the brute-force
//                     definition.  Candidates are compared by descriptor
//                     (Sec. 4.3) and the warp keeps the best two by
//                     (distance, index), then applies the ratio test.
#include <math.h>

#include "egm_internal.cuh"

namespace egm {

namespace {

// ------------------------------------------------------------ descriptors

// ------------------------------------------------------------ stabbing
//
// One block takes kQB consecutive queries.  On GB300 a dependent global
// access costs about a microsecond, so the kernel is organised around the
// number of serial memory round trips per block:
//   phase 1  (2 trips)  query records and the block's pair geometry; then
//            the bucket-table loads of every window and the query
//            descriptors together.  Warp w handles queries 4w .. 4w+3,
//            lane = level; non-empty ranges are compacted into shared memory.
//   2a (1 trip)  the concatenated window elements, a contiguous chunk per
//            thread, record loads issued together; each passes the Eq. 3/4
//            test (FP32 with a rigorous bound, FP64 brute-force expression
//            when inconclusive); candidates are appended to a list with one
//            warp-aggregated atomic.
//   2a'      the list is counting-sorted by query into segments.
//   2b (1 trip per 128 candidates)  a group of G lanes per candidate
//            (G 16-byte chunks of its descriptor), four candidates per group
//            with all loads issued first; distances go to the segment.
//   2c       one warp per query reduces its segment into the query's best
//            two (distance, index) keys - a single writer, no atomics.
// Rounds of kRound elements repeat 2a-2c; the outputs follow the last round.
constexpr int kQB = kStabQB;
// the per-round segment scan gives one lane of warp 0 to each query of the block
static_assert(kQB == 32, "one lane per query in the segment scan");
constexpr int kStabThreads = 256;
constexpr int kRangesPerQuery = 2 * kLevels;
constexpr int kDescCache = 256;  // query descriptors up to this many bytes are staged in shared memory
// window elements a thread tests per batch of record loads, and candidates
// per lane group in the distance pass
constexpr int kBatch = 4;
constexpr int kU = 4;
// window elements tested per round (shared memory for occupancy)
constexpr int kRound = 1024;
constexpr int kQPerWarp = kQB / (kStabThreads / 32);

template <int kRound>
struct StabSmem {
    uint2 rng[kQB][kRangesPerQuery];  // (first sorted position, length) of each non-empty range
    QueryRec qr[kQB];
    PairGeom g;                       // geometry of the block's first pair
    PairDesc pd;                      //   and its descriptor
    unsigned long long b1[kQB], b2[kQB];
    uint32_t nrng[kQB];
    uint32_t tq[kQB];
    uint32_t eoff[kQB + 1];
    uint32_t cnt[kQB];                // candidates per query (all rounds)
    uint32_t rcnt[kQB];               // candidates per query in this round
    uint32_t roff[kQB + 1];           //   their segment offsets
    uint32_t rfill[kQB];
    uint32_t nwin, nexact, ncand;
    int32_t gpair;
    uint32_t lj[kRound];              // append list: reference index
    uint8_t lq[kRound];               //   and query slot
    uint32_t sj[kRound];              // per-query segments: reference index
    uint8_t sq[kRound];               //   and query slot
    uint32_t sd[kRound];              //   and descriptor distance
    uint32_t rmask[kQB][2];           // non-empty ranges of each query (bit k: range k)
    int32_t lv[kLevels];              // non-empty levels of the block's pair
    int32_t nlev;
    uint4 qdesc[kQB][kDescCache / 16];
};

constexpr int kKindAny = -1;  // a launch that mixes descriptor kinds

// Contribution of one 16-byte chunk to a descriptor distance.
template <int KIND>
__device__ __forceinline__ void chunk_dist(int kind, uint4 a, uint4 b, uint32_t &acc, float &facc) {
    const int k = KIND == kKindAny ? kind : KIND;
    if (k == EGM_DESC_U8_L2) {
        uint32_t d;
        d = __vabsdiffu4(a.x, b.x); acc = __dp4a(d, d, acc);
        d = __vabsdiffu4(a.y, b.y); acc = __dp4a(d, d, acc);
        d = __vabsdiffu4(a.z, b.z); acc = __dp4a(d, d, acc);
        d = __vabsdiffu4(a.w, b.w); acc = __dp4a(d, d, acc);
    } else if (k == EGM_DESC_BIN) {
        acc += __popc(a.x ^ b.x) + __popc(a.y ^ b.y) + __popc(a.z ^ b.z) + __popc(a.w ^ b.w);
    } else {
        float d;
        d = __uint_as_float(a.x) - __uint_as_float(b.x); facc = fmaf(d, d, facc);
        d = __uint_as_float(a.y) - __uint_as_float(b.y); facc = fmaf(d, d, facc);
        d = __uint_as_float(a.z) - __uint_as_float(b.z); facc = fmaf(d, d, facc);
        d = __uint_as_float(a.w) - __uint_as_float(b.w); facc = fmaf(d, d, facc);
    }
}

__device__ __forceinline__ void top2_key(unsigned long long key, unsigned long long &b1, unsigned long long &b2) {
    if (key < b1) {
        b2 = b1;
        b1 = key;
    } else if (key < b2) {
        b2 = key;
    }
}

// 16-byte asynchronous copy global -> shared (no registers held while it is
// in flight); cp_async_wait() before the data is read
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void copy16(void *dst, const void *src, int bytes, int lane) {
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst);
    for (int k = lane; k < bytes / 16; k += 32) d4[k] = __ldg(s4 + k);
}

// Matching (match: some pair has descriptors) and, when L.qcount is set, the
// candidates per query.  (Rows of the usual kinds and sizes run
// stab_pair_kernel instead, see launch_warp_per_query.)
template <int KIND>
__global__ void __launch_bounds__(kStabThreads, 4) stab_kernel(Launch L) {
    pdl_begin();
    __shared__ __align__(16) StabSmem<kRound> S;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const bool match = L.kinds != 0u;
    uint32_t nwin = 0, nexact = 0;
    if (tid == 0) { S.nwin = 0; S.nexact = 0; S.ncand = 0; }
    for (int64_t q0 = (int64_t)blockIdx.x * kQB; q0 < L.nq; q0 += (int64_t)gridDim.x * kQB) {
        const int nqb = (int)min((int64_t)kQB, L.nq - q0);
        // ---- phase 1, trip 1: query records, and the first pair's geometry and descriptor
        const int qbase = warp * kQPerWarp;
        if (lane < 3 * kQPerWarp) {
            const int ql = qbase + lane / 3;
            if (ql < nqb)
                reinterpret_cast<uint4 *>(&S.qr[ql])[lane % 3] =
                    __ldg(reinterpret_cast<const uint4 *>(L.qrec + q0 + ql) + lane % 3);
        }
        if (warp == kStabThreads / 32 - 1) {
            const int p0 = L.npairs == 1 ? 0 : L.blkpair[q0 / kQB];
            copy16(&S.g, L.geom + p0, (int)sizeof(PairGeom), lane);
            copy16(&S.pd, L.pairs + p0, (int)sizeof(PairDesc), lane);
            if (lane == 0) S.gpair = p0;
        }
        __syncthreads();
        // ---- phase 1, trip 2: windows, their bucket-table loads and the query
        // descriptors issued together.  Lanes take (query, non-empty level)
        // slots of the block's pair, so a pair with two populated levels costs
        // two lanes per query, not 32; ranges go to fixed slots 2 i, 2 i + 1 of
        // level index i (empty ones have length 0).
        if (warp == 0) {
            const uint32_t nz = __ballot_sync(0xffffffffu, S.g.cnt[lane] > 0);
            if (nz & (1u << lane)) S.lv[__popc(nz & lt)] = lane;
            if (lane == 0) S.nlev = __popc(nz);
        }
        if (tid < kQB) {
            S.tq[tid] = 0;
            S.nrng[tid] = 0;
            S.b1[tid] = ~0ull;
            S.b2[tid] = ~0ull;
            S.cnt[tid] = 0;
            S.rmask[tid][0] = S.rmask[tid][1] = 0u;
        }
        __syncthreads();
        // the query descriptors, copied to shared memory while the windows are computed
        constexpr int kStage = kQPerWarp * kDescCache / 16 / 32;
#pragma unroll
        for (int k = 0; k < kStage; k++) {
            const int idx = lane + 32 * k;
            const int ql = qbase + idx / (kDescCache / 16);
            const int c = idx % (kDescCache / 16);
            if (match && ql < nqb) {
                const int p = S.qr[ql].pair;
                const PairDesc &P = p == S.gpair ? S.pd : L.pairs[p];
                if (P.row_bytes > 0 && P.row_bytes <= kDescCache && c < (P.row_bytes >> 4))
                    cp_async16(&S.qdesc[ql][c], reinterpret_cast<const uint4 *>(P.desc1 + (q0 + ql - P.q_off) *
                                                                                         (int64_t)P.row_bytes) + c);
            }
        }
        {
            const int nlev = S.nlev;
            const int nslot = nqb * nlev;
            for (int g0 = warp * 32; g0 < nslot; g0 += kStabThreads) {
                const int sl = g0 + lane;
                WinKeys wk;
                wk.kind = 0;
                int ql = 0, li = 0;
                if (sl < nslot) {
                    ql = sl / nlev;
                    li = sl - ql * nlev;
                    if (S.qr[ql].pair == S.gpair) wk = window_keys(S.g, S.qr[ql], S.lv[li]);
                    else ql = -1;  // another pair: handled below
                }
                uint32_t a = 0, b = 0;
                if (wk.kind >= 2) {
                    const uint32_t *T = L.tab + S.pd.t_off + S.g.tab[S.lv[li]];
                    a = __ldg(T + wk.ta);
                    b = __ldg(T + wk.tb);
                }
                if (sl < nslot && ql >= 0) {
                    const Window w = window_ranges(wk, a, b);
                    S.rng[ql][2 * li] = make_uint2(w.b0, w.len0);
                    S.rng[ql][2 * li + 1] = make_uint2(w.b1, w.len1);
                    if (w.len0 + w.len1) {
                        atomicAdd(&S.tq[ql], w.len0 + w.len1);
                        const uint32_t bits = (w.len0 ? 1u : 0u) | (w.len1 ? 2u : 0u);
                        atomicOr(&S.rmask[ql][li >> 4], bits << (2 * (li & 15)));
                    }
                    if (li == 0) S.nrng[ql] = 2 * nlev;
                }
            }
            // queries of another pair than the block's first: one warp per query, lane = level
#pragma unroll 1
            for (int t = 0; t < kQPerWarp; t++) {
                const int ql = qbase + t;
                if (ql >= nqb || S.qr[ql].pair == S.gpair) continue;
                const int p = S.qr[ql].pair;
                const PairGeom &G = L.geom[p];
                const WinKeys wk = window_keys(G, S.qr[ql], lane);
                uint32_t a = 0, b = 0;
                if (wk.kind >= 2) {
                    const uint32_t *T = L.tab + L.pairs[p].t_off + G.tab[lane];
                    a = __ldg(T + wk.ta);
                    b = __ldg(T + wk.tb);
                }
                const Window w = window_ranges(wk, a, b);
                S.rng[ql][2 * lane] = make_uint2(w.b0, w.len0);
                S.rng[ql][2 * lane + 1] = make_uint2(w.b1, w.len1);
                const uint32_t bits = (w.len0 ? 1u : 0u) | (w.len1 ? 2u : 0u);
                const uint32_t lo16 = __reduce_or_sync(0xffffffffu, lane < 16 ? bits << (2 * lane) : 0u);
                const uint32_t hi16 = __reduce_or_sync(0xffffffffu, lane >= 16 ? bits << (2 * (lane - 16)) : 0u);
                if (lane == 0) { S.rmask[ql][0] = lo16; S.rmask[ql][1] = hi16; }
                uint32_t tot = w.len0 + w.len1;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
                if (lane == 0) {
                    S.tq[ql] = tot;
                    S.nrng[ql] = 2 * kLevels;
                }
            }
        }
        cp_async_wait();
        // every query of the block in the cached pair, descriptors of one kind
        // and staged: the pair's fields are block constants (the common case)
        const bool uni = __syncthreads_and(tid >= nqb || S.qr[tid].pair == S.gpair) && KIND != kKindAny &&
                         S.pd.row_bytes <= kDescCache;
        const float4 *recb = L.rec + S.pd.r_off;
        if (warp == 0) {
            uint32_t incl = S.tq[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            S.eoff[lane + 1] = incl;
            if (lane == 0) S.eoff[0] = 0;
        }
        __syncthreads();

        // ---- phase 2, in rounds of kRound window elements
        const uint32_t T = S.eoff[kQB];
        for (uint32_t base = 0; base < T; base += kRound) {
            // 2a: tests, candidates appended to the list
            if (tid < kQB) S.rcnt[tid] = 0;
            __syncthreads();
            const uint32_t Tr = min(T - base, (uint32_t)kRound);
            const uint32_t K = (Tr + kStabThreads - 1) / kStabThreads;  // the same for every thread
            uint32_t f = base + (uint32_t)tid * K;
            const uint32_t fend = min(f + K, base + Tr);
            int q = 0, k = 0;
            uint32_t rem = 0;
            // move (q, k, rem) forward to a real element: past exhausted or empty
            // ranges and past queries without elements
            auto settle = [&]() {
                while (q < kQB) {
                    // next non-empty range at or after k
                    const uint32_t m0 = k < 32 ? S.rmask[q][0] & (~0u << k) : 0u;
                    const uint32_t m1 = k >= 64 ? 0u : k <= 32 ? S.rmask[q][1] : S.rmask[q][1] & (~0u << (k - 32));
                    if (m0) k = __ffs(m0) - 1;
                    else if (m1) k = 32 + __ffs(m1) - 1;
                    else { q++; k = 0; continue; }
                    const uint32_t len = S.rng[q][k].y;
                    if (rem < len) break;
                    rem -= len;
                    k++;
                }
            };
            if (f < fend) {
#pragma unroll
                for (int st = 16; st > 0; st >>= 1)
                    if (S.eoff[q + st] <= f) q += st;
                rem = f - S.eoff[q];
                settle();
            }
            for (uint32_t kb = 0; kb < K; kb += kBatch) {
                int bq[kBatch];
                uint32_t bpos[kBatch];
                bool bv[kBatch];
#pragma unroll
                for (int t = 0; t < kBatch; t++) {
                    bv[t] = f < fend;
                    bq[t] = q;
                    bpos[t] = 0;
                    if (bv[t]) {
                        bpos[t] = S.rng[q][k].x + rem;
                        f++;
                        rem++;
                        if (f < fend) settle();
                    }
                }
                float4 rc[kBatch];
#pragma unroll
                for (int t = 0; t < kBatch; t++) {
                    if (bv[t]) {
                        if (uni) {
                            rc[t] = __ldg(recb + bpos[t]);
                        } else {
                            const int p = S.qr[bq[t]].pair;
                            const int64_t ro = p == S.gpair ? S.pd.r_off : L.pairs[p].r_off;
                            rc[t] = __ldg(L.rec + ro + bpos[t]);
                        }
                    }
                }
#pragma unroll 1
                for (int t = 0; t < kBatch; t++) {
                    // element t of the batch by register selects: a dynamic index into
                    // these arrays would place them in local memory
                    int qq = bq[0];
                    bool bvt = bv[0];
                    float4 rct = rc[0];
#pragma unroll
                    for (int u = 1; u < kBatch; u++)
                        if (t == u) {
                            qq = bq[u];
                            bvt = bv[u];
                            rct = rc[u];
                        }
                    uint32_t j = 0;
                    bool cand = false;
                    if (bvt) {
                        const QueryRec &r = S.qr[qq];
                        j = __float_as_uint(rct.w);
                        nwin++;
                        bool exact = (r.flags & kQExactOnly) != 0;
                        if (!exact) {
                            const float x = rct.x, y = rct.y, e = rct.z;
                            const float d = fabsf(fmaf(r.A, x, fmaf(r.B, y, r.C)));
                            const float Sm = fmaf(fabsf(r.A), fabsf(x), fmaf(fabsf(r.B), fabsf(y), fabsf(r.C)));
                            // FP32 rounding (16u S), the FP32 tolerance (2u eps) and the
                            // distance between this line and the brute force's FP64 line
                            const float lerr = fmaf(r.E1, fabsf(x) + fabsf(y) + 2.0f * e, r.E0);
                            const float bound = fmaf(9.6e-7f, Sm, fmaf(1.2e-7f, e, lerr + 1e-9f));
                            cand = d <= e - bound;
                            exact = !cand && !(d > e + bound);
                        }
                        if (exact) {
                            // FP32 inconclusive: the brute-force FP64 expression decides.
                            const PairDesc &P = L.pairs[r.pair];
                            cand = exact_pair(P, q0 + qq - P.q_off, j);
                            nexact++;
                        }
                    }
                    if (!match) {
                        if (cand) atomicAdd(&S.cnt[qq], 1u);
                    } else {
                        // warp-aggregated append to the round's candidate list
                        const uint32_t m = __ballot_sync(0xffffffffu, cand);
                        if (m) {
                            const int leader = __ffs(m) - 1;
                            uint32_t c0 = 0;
                            if (lane == leader) c0 = atomicAdd(&S.ncand, (uint32_t)__popc(m));
                            c0 = __shfl_sync(0xffffffffu, c0, leader);
                            if (cand) {
                                const uint32_t c = c0 + __popc(m & lt);
                                S.lj[c] = j;
                                S.lq[c] = (uint8_t)qq;
                                atomicAdd(&S.rcnt[qq], 1u);
                            }
                        }
                    }
                }
            }
            __syncthreads();
            const uint32_t nc = S.ncand;
            // the round's candidates per query (rather than one more atomic add per candidate)
            if (match && tid < kQB) S.cnt[tid] += S.rcnt[tid];
            if (match && nc > 0) {
                // 2a': segments by query
                if (warp == 0) {
                    const uint32_t v = S.rcnt[lane];
                    uint32_t incl = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += t;
                    }
                    S.roff[lane] = incl - v;
                    S.rfill[lane] = incl - v;
                    if (lane == 31) S.roff[kQB] = incl;
                }
                __syncthreads();
                for (uint32_t c = tid; c < nc; c += kStabThreads) {
                    const int qq = S.lq[c];
                    const uint32_t pos = atomicAdd(&S.rfill[qq], 1u);
                    S.sj[pos] = S.lj[c];
                    S.sq[pos] = (uint8_t)qq;
                }
                __syncthreads();
                // 2b: G lanes per candidate read its descriptor row together (one
                // cache line per group of eight 16-byte chunks), four candidates per
                // group with the loads issued first; distances go to shared memory.
                const int rb0 = KIND != kKindAny ? S.pd.row_bytes : kDescCache;
                const int chunks0 = rb0 >> 4;
                const int G = chunks0 >= 32 ? 32 : chunks0 >= 16 ? 16 : chunks0 >= 8 ? 8 : chunks0 >= 4 ? 4
                            : chunks0 >= 2 ? 2 : 1;
                const int groups = kStabThreads / G;
                const int gl = tid % G;
                constexpr int U = kU;
                if (uni && chunks0 <= G) {
                    // block constants; one chunk per lane of each candidate
                    const uint4 *d2 = reinterpret_cast<const uint4 *>(S.pd.desc2);
                    const int rb16 = chunks0;
                    for (uint32_t cb = 0; cb < nc; cb += (uint32_t)(groups * U)) {
                        uint32_t cc[U];
                        uint4 rv[U];
#pragma unroll
                        for (int u = 0; u < U; u++) {
                            cc[u] = cb + (uint32_t)(tid / G) + (uint32_t)(u * groups);
                            if (cc[u] < nc && gl < rb16) rv[u] = __ldg(d2 + (int64_t)S.sj[cc[u]] * rb16 + gl);
                        }
#pragma unroll
                        for (int u = 0; u < U; u++) {
                            uint32_t acc = 0;
                            float facc = 0.0f;
                            if (cc[u] < nc && gl < rb16) chunk_dist<KIND>(KIND, S.qdesc[S.sq[cc[u]]][gl], rv[u], acc, facc);
                            if (KIND == EGM_DESC_F32_L2) {
                                for (int o = G >> 1; o > 0; o >>= 1) facc += __shfl_xor_sync(0xffffffffu, facc, o, G);
                                acc = __float_as_uint(facc);
                            } else {
                                for (int o = G >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o, G);
                            }
                            if (gl == 0 && cc[u] < nc) S.sd[cc[u]] = acc;
                        }
                    }
                } else
                for (uint32_t cb = 0; cb < nc; cb += (uint32_t)(groups * U)) {
                    uint32_t cc[U];
                    const uint4 *rrow[U];
                    const uint4 *qrow[U];
                    int chunks[U], kinds[U];
                    bool qsm[U];
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        cc[u] = cb + (uint32_t)(tid / G) + (uint32_t)(u * groups);
                        chunks[u] = 0;
                        kinds[u] = KIND;
                        rrow[u] = qrow[u] = nullptr;
                        qsm[u] = true;
                        if (cc[u] < nc) {
                            const int qq = S.sq[cc[u]];
                            const int p = S.qr[qq].pair;
                            const PairDesc &P = p == S.gpair ? S.pd : L.pairs[p];
                            chunks[u] = P.row_bytes >> 4;
                            if (KIND == kKindAny) kinds[u] = P.kind;
                            rrow[u] = reinterpret_cast<const uint4 *>(P.desc2 + (int64_t)S.sj[cc[u]] * P.row_bytes);
                            qsm[u] = P.row_bytes <= kDescCache;
                            qrow[u] = qsm[u] ? S.qdesc[qq]
                                             : reinterpret_cast<const uint4 *>(P.desc1 + (q0 + qq - P.q_off) *
                                                                                         (int64_t)P.row_bytes);
                        }
                    }
                    uint32_t acc[U];
                    float facc[U];
#pragma unroll
                    for (int u = 0; u < U; u++) { acc[u] = 0; facc[u] = 0.0f; }
                    int maxch = 0;
#pragma unroll
                    for (int u = 0; u < U; u++) maxch = max(maxch, chunks[u]);
                    for (int ch0 = 0; ch0 < maxch; ch0 += G) {
                        const int ch = ch0 + gl;
                        uint4 rv[U];
#pragma unroll
                        for (int u = 0; u < U; u++)
                            if (ch < chunks[u]) rv[u] = __ldg(rrow[u] + ch);
#pragma unroll
                        for (int u = 0; u < U; u++)
                            if (ch < chunks[u])
                                chunk_dist<KIND>(kinds[u], qsm[u] ? qrow[u][ch] : __ldg(qrow[u] + ch), rv[u], acc[u],
                                                 facc[u]);
                    }
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const bool isf = (KIND == kKindAny ? kinds[u] : KIND) == EGM_DESC_F32_L2;
                        uint32_t v = isf ? __float_as_uint(facc[u]) : acc[u];
                        for (int o = G >> 1; o > 0; o >>= 1) {
                            if (isf) {
                                facc[u] += __shfl_xor_sync(0xffffffffu, facc[u], o, G);
                                v = __float_as_uint(facc[u]);
                            } else {
                                acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o, G);
                                v = acc[u];
                            }
                        }
                        if (gl == 0 && cc[u] < nc) S.sd[cc[u]] = v;
                    }
                }
                __syncthreads();
                // 2c: a thread per candidate, segmented best two per query within
                // the warp (a query's candidates are contiguous), merged by the
                // segment's first lane.  The merge keeps the minimum with one
                // atomicMin and offers min(the larger of the displaced and the
                // offered first, the offered second) to the second slot: every
                // value offered there is an element other than the minimum and
                // the true second is always offered, so the pair is exact under
                // any interleaving.
                for (uint32_t cb = 0; cb < nc; cb += kStabThreads) {
                    const uint32_t c = cb + (uint32_t)tid;
                    const bool valid = c < nc;
                    const int qq = valid ? (int)S.sq[c] : -1 - lane;
                    unsigned long long k1 = valid ? ((unsigned long long)S.sd[c] << 32) | S.sj[c] : ~0ull;
                    unsigned long long k2 = ~0ull;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned long long o1 = __shfl_down_sync(0xffffffffu, k1, o);
                        const unsigned long long o2 = __shfl_down_sync(0xffffffffu, k2, o);
                        const int oq = __shfl_down_sync(0xffffffffu, qq, o);
                        if (lane + o < 32 && oq == qq) {
                            const unsigned long long mx = k1 < o1 ? o1 : k1;
                            const unsigned long long mn2 = k2 < o2 ? k2 : o2;
                            k1 = k1 < o1 ? k1 : o1;
                            k2 = mx < mn2 ? mx : mn2;
                        }
                    }
                    const int pq = __shfl_up_sync(0xffffffffu, qq, 1);
                    if (valid && (lane == 0 || pq != qq)) {
                        const unsigned long long old = atomicMin(&S.b1[qq], k1);
                        const unsigned long long lose = old > k1 ? old : k1;
                        const unsigned long long offer = lose < k2 ? lose : k2;
                        if (offer != ~0ull) atomicMin(&S.b2[qq], offer);
                    }
                }
            }
            __syncthreads();
            if (tid == 0) S.ncand = 0;
        }
        if (L.counters) {
            atomicAdd(&S.nwin, nwin);
            atomicAdd(&S.nexact, nexact);
            nwin = nexact = 0;
        }
        __syncthreads();

        // ---- results
        if (tid < nqb) {
            const int64_t gq = q0 + tid;
            if (L.qcount) L.qcount[gq] = S.cnt[tid];
            const int p = S.qr[tid].pair;
            const PairDesc &P = p == S.gpair ? S.pd : L.pairs[p];
            store_match(L, gq, P, S.qr[tid].flags, S.b1[tid], S.b2[tid]);
            if (L.counters) atomicAdd(L.counters + 3, (unsigned long long)S.cnt[tid]);
        }
        __syncthreads();
    }
    if (L.counters && tid == 0) {
        atomicAdd(L.counters + 2, (unsigned long long)S.nwin);
        atomicAdd(L.counters + 4, (unsigned long long)S.nexact);
    }
}

// ------------------------------------------------------------ one pair, a warp per query
//
// The queries of one pair share nothing but the pair's tables, so in this
// variant each warp takes one query at a time and needs no block-wide
// phase: lane l computes the window of the pair's l-th populated level and
// its two ranges of sorted positions (Sec. 4.2 query, split at the seam);
// the ranges are flattened by a prefix sum over the lanes, and the warp
// tests 32 window elements per step (each lane finds its element's range by
// a five-step search over the lanes' prefix sums).  Candidates go to a small
// per-warp ring in shared memory; every 32 of them are one batch of
// descriptor distances (Sec. 4.3): G lanes read one candidate's row (16
// bytes each, coalesced), G rounds are accumulated per lane and reduced by
// a transposed butterfly (G - 1 shuffles for the G rounds), after which
// each lane holds one candidate's distance.  Each lane keeps its best two
// (distance, index) keys; four warp reductions give the query's best two.
constexpr int kPairThreads = 64;
constexpr int kPairWarps = kPairThreads / 32;
constexpr int kRing = 64;  // candidate ring per warp: 32 waiting + 32 new
constexpr int kChunkQ = 8; // queries per warp whose windows are computed in one pass

// The window of a query in one level, from the level's half-width over all
// of the pair's queries (key_window_span with the pair's extremes of the pad
// arguments and of |key|, recorded by the prep kernel): a superset of each
// query's own window, so the exact test keeps the same candidates.
//
// Where F has rank 2 to rounding, the lines pass the epipole within far less
// than a pixel and the extremes add nothing.  Where it has not (an estimate
// whose rank was not enforced), a line's distance from the epipole grows
// towards the epipole of image 1, and one query there would widen every
// window of the pair: levels that the extremes widen by more than about a
// fourth over the pair's best query take each query's own half-width instead.
// (16,384 keypoints at 2 px, epipoles inside, the smallest singular value 1e-4
// of the second: mutual match 308 us against 1,614 with the extremes, 8 pairs 414
// against 6,329, one u8 pair 250 against 889, one float pair 268 against 1,319.
// What is left is the query next to the epipole itself, whose window is the
// image: its warp walks 15,000 references alone, 135 us; without the five
// keypoints within 30 px the mutual match takes 150.  Loading its records
// several steps ahead, in a function of its own or into the L1 cache, shortens
// that walk by a quarter at most and slows every other call.)
enum : int { kWinShared = 0, kWinWhole = 1, kWinOwn = 2 };
struct LevelWin {
    float hw;      // half-width of every window in the level's key space
    int kind;      // kWinShared; kWinWhole: every window covers the whole level; kWinOwn: a half-width per query
    uint32_t s, e; // sorted positions of the level
    int sh;        // key bits below the level's buckets
};

__device__ __forceinline__ LevelWin level_win(const PairGeom &G, int lv) {
    const bool angular = G.mode == kModeAngular;
    const float a0min = __uint_as_float(G.qa0min), a0max = __uint_as_float(G.qa0max), a1max = __uint_as_float(G.qa1max);
    const KeyWin w = key_window_span(G, lv, 0.0f, 0.0f, __uint_as_float(G.qkabs), angular ? a0max : a0min, a1max, false);
    LevelWin c;
    c.hw = w.hi;
    c.kind = w.kind == 1 ? kWinWhole : kWinShared;
    // the half-width's leading term is (smax dmin + a0) / dmin, or (smax + R a1) / a0 in the parallel frame
    const float smax = __uint_as_float(G.smax[lv]), dmin = __uint_as_float(G.dmin[lv]), R = __uint_as_float(G.tmax[lv]);
    if (angular ? smax < 1.0f && a0max > 1.25f * a0min + 0.25f * (smax * dmin)
                : smax + R * a1max > 1.25f * (a0min * smax))
        c.kind = kWinOwn;
    c.s = G.start[lv];
    c.e = G.start[lv + 1];
    c.sh = kQBits - G.bits[lv];
    return c;
}

// The half-width of query r's own window in level lv, infinite where the
// window is the whole level.
__device__ __forceinline__ float own_half_width(const PairGeom &G, int lv, const QueryRec &r) {
    const KeyWin w = key_window_span(G, lv, 0.0f, 0.0f, fabsf(r.key), r.aux0, r.aux1, false);
    return w.kind == 2 ? w.hi : INFINITY;
}

// The window of query r in the lane's level lv as bucket-table indices (the
// kinds of WinKeys).
__device__ __forceinline__ WinKeys level_window(const PairGeom &G, const LevelWin &c, int lv, const QueryRec &r) {
    WinKeys k;
    k.s = c.s;
    k.e = c.e;
    k.ta = k.tb = 0u;
    k.kind = 0;
    if (r.flags & EGM_FLAG_DEGENERATE_LINE) return k;
    bool full = c.kind == kWinWhole || (r.flags & kQExactOnly) != 0;
    float hw = c.hw;
    if (c.kind == kWinOwn && !full) {
        hw = own_half_width(G, lv, r);
        full = !(hw < INFINITY);
    }
    const float lo = r.key - hw, hi = r.key + hw;
    const bool low = G.mode == kModeAngular && lo < -kHalfPiF;
    const bool high = G.mode == kModeAngular && hi >= kHalfPiF;
    if (full || (low && high)) {
        k.kind = 1;
    } else if (low || high) {
        // across the seam of the [-pi/2, pi/2) domain: [ta, end) and [start, tb)
        k.ta = qmap(low ? lo + kPiF : lo, G.kmin, G.kscale) >> c.sh;
        k.tb = (qmap(low ? hi : hi - kPiF, G.kmin, G.kscale) >> c.sh) + 1;
        k.kind = 3;
    } else {
        k.ta = qmap(lo, G.kmin, G.kscale) >> c.sh;
        k.tb = (qmap(hi, G.kmin, G.kscale) >> c.sh) + 1;
        k.kind = 2;
    }
    return k;
}

// The brute force's FP64 decision for one (query, reference) pair of a
// single-pair call, from plain pointers.
static __device__ __noinline__ bool exact_pair_p(const double *F, const double *xy1, const double *xy2,
                                                 const double *eps2, double eps_scalar, int64_t i, uint32_t j) {
    double a, b, c;
    exact_line(F, xy1[2 * i], xy1[2 * i + 1], a, b, c);
    const double eps = eps2 ? eps2[j] : eps_scalar;
    return exact_within(a, b, c, xy2[2 * (int64_t)j], xy2[2 * (int64_t)j + 1], eps);
}

// A pair as a warp works on it, in shared memory: its geometry, its populated
// levels and their windows' constants.
struct PairWork {
    PairGeom g;
    LevelWin win[kLevels];
    int32_t lv[kLevels];
};

// Loads pair geometry `src` into the warp's W; returns the populated levels.
__device__ __forceinline__ int load_pair_work(PairWork &W, const PairGeom *src, int lane) {
    __syncwarp();  // the previous pair's readers are done
    for (int k = lane; k < (int)(sizeof(PairGeom) / 16); k += 32)
        reinterpret_cast<uint4 *>(&W.g)[k] = __ldg(reinterpret_cast<const uint4 *>(src) + k);
    __syncwarp();
    const bool have = W.g.cnt[lane] > 0;
    const uint32_t nz = __ballot_sync(0xffffffffu, have);
    if (have) {
        const int idx = __popc(nz & ((1u << lane) - 1u));
        W.lv[idx] = lane;
        W.win[idx] = level_win(W.g, lane);
    }
    __syncwarp();
    return __popc(nz);
}

// G lanes read a descriptor row, C 16-byte chunks each (a row is G C 16 bytes):
// lane s of a group the chunks C s .. C s + C - 1, or, of float rows, s and
// s + G (with the butterfly below, the order of additions of one lane per
// chunk and an XOR butterfly over them, the one every form uses).
//
// ONE: the call has one pair (its plan in the launch parameters), the warps
// take strided queries.  Otherwise every warp takes runs of `run` consecutive
// queries in turn and, within a run, the queries of one pair at a time: its
// own copy of the pair's geometry, so that no block-wide phase exists either.
// (Two directions of a 16,384-keypoint pair, tolerances per keypoint: 112 us
// in blocks of 32 queries, 48 us here; one float pair of 16,384 keypoints at
// 2 px 86 -> 48 us a call, at 8 px 279 -> 74.)  Blocks per SM: 13 for one pair
// (12: 1 % slower over nine pairs, 16: 2 %), 16 for several (13: 4 % slower),
// 8 for float rows (128 registers).
template <int KIND, int G, int C, bool ONE>
__global__ void __launch_bounds__(kPairThreads, KIND == EGM_DESC_F32_L2 ? 8 : ONE ? 13 : 16)
    stab_pair_kernel(const __grid_constant__ Launch L, int64_t run) {
    static_assert(G >= 1 && G <= 16 && (G & (G - 1)) == 0, "lanes per descriptor row");
    constexpr bool kFlt = KIND == EGM_DESC_F32_L2;
    constexpr int kPerRound = 32 / G;  // candidates per round of loads
    constexpr int kRow16 = G * C;      // 16-byte chunks per row
    pdl_begin();
    __shared__ __align__(16) PairWork work[ONE ? 1 : kPairWarps];
    __shared__ int32_t snlev;
    __shared__ uint32_t ring[kPairWarps][kRing];
    // a warp's chunk of queries: their records, descriptor rows and window ranges
    __shared__ __align__(16) QueryRec qchunk[kPairWarps][kChunkQ];
    __shared__ __align__(16) uint4 dchunk[kPairWarps][kChunkQ][kRow16];
    __shared__ __align__(16) uint4 wrng[kPairWarps][kChunkQ * kLevels];
    __shared__ __align__(16) uint4 res[kPairWarps][kChunkQ];   // best two (distance, index) of each query
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t lt = (1u << lane) - 1u;
    PairWork &W = work[ONE ? 0 : warp];
    uint32_t *rg = ring[warp];
    const int sub = lane % G, grp = lane / G;
    auto chunk_of = [&](int c) { return kFlt ? sub + c * G : sub * C + c; };
    const int64_t nwarps = (int64_t)gridDim.x * kPairWarps, gw = (int64_t)blockIdx.x * kPairWarps + warp;
    uint32_t nwin = 0, ncand = 0, nexact = 0;
    int p = -1, nlev = 0;  // the pair in W and its populated levels

    // nk <= kChunkQ queries c0, c0 + step, ... of the pair PD: their records and
    // descriptor rows are copied at once, and the windows of every (query,
    // level) slot are computed in one pass over the lanes, with their table
    // loads issued together
    auto chunk = [&](const PairDesc &PD, int64_t c0, int nk, int64_t step) {
    const bool haslev = lane < nlev;
    const float4 *recb = L.rec + PD.r_off;
    const uint4 *d1 = reinterpret_cast<const uint4 *>(PD.desc1);
    const uint4 *d2 = reinterpret_cast<const uint4 *>(PD.desc2);
    for (int t = lane; t < 3 * nk; t += 32)
        cp_async16(reinterpret_cast<uint4 *>(&qchunk[warp][t / 3]) + t % 3,
                   reinterpret_cast<const uint4 *>(L.qrec + c0 + (int64_t)(t / 3) * step) + t % 3);
    for (int t = lane; t < kRow16 * nk; t += 32)
        cp_async16(&dchunk[warp][t / kRow16][t % kRow16],
                   d1 + (c0 + (int64_t)(t / kRow16) * step - PD.q_off) * kRow16 + t % kRow16);
    cp_async_wait();
    __syncwarp();
    for (int s0 = 0; s0 < nk * nlev; s0 += 32) {
        const int sl = s0 + lane;
        if (sl < nk * nlev) {
            const int k = sl / nlev, l = sl - k * nlev;
            const WinKeys wk = level_window(W.g, W.win[l], W.lv[l], qchunk[warp][k]);
            uint32_t a = 0, b = 0;
            if (wk.kind >= 2) {
                const uint32_t *Tl = L.tab + PD.t_off + W.g.tab[W.lv[l]];
                a = __ldg(Tl + wk.ta);
                b = __ldg(Tl + wk.tb);
            }
            const Window wl = window_ranges(wk, a, b);
            wrng[warp][k * kLevels + l] = make_uint4(wl.b0, wl.len0, wl.b1, wl.len1);
        }
    }
    __syncwarp();
    uint32_t mine = 0;  // lane k: the candidates of query k
    for (int k = 0; k < nk; k++) {
        const int64_t q = c0 + (int64_t)k * step;
        const QueryRec rq = qchunk[warp][k];
        uint4 qdq[C];
#pragma unroll
        for (int c = 0; c < C; c++) qdq[c] = dchunk[warp][k][chunk_of(c)];
        // the window of this lane's level as (at most) two ranges of sorted positions
        Window w;
        w.b0 = w.len0 = w.b1 = w.len1 = 0u;
        if (haslev) {
            const uint4 v = wrng[warp][k * kLevels + lane];
            w.b0 = v.x;
            w.len0 = v.y;
            w.b1 = v.z;
            w.len1 = v.w;
        }
        const uint32_t tl = w.len0 + w.len1;
        uint32_t incl = tl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const uint32_t p0 = incl - tl;  // first flattened element of this lane's ranges
        const uint32_t E = __shfl_sync(0xffffffffu, incl, 31);
        const bool exact_only = (rq.flags & kQExactOnly) != 0;
        uint32_t count = 0, done = 0;  // candidates found / already in a distance batch (warp-uniform)
        unsigned long long k1 = ~0ull, k2 = ~0ull;

        // one batch of nb <= 32 candidates from the ring, starting at `start`
        auto batch = [&](uint32_t start, uint32_t nb) {
            __syncwarp();
            uint32_t acc[G];  // distances (float rows: their bits)
#pragma unroll
            for (int u = 0; u < G; u++) acc[u] = 0u;
#pragma unroll
            for (int u = 0; u < G; u++) {
                if ((uint32_t)(u * kPerRound) >= nb) break;
                const uint32_t c = (uint32_t)(u * kPerRound + grp);
                if (c < nb) {
                    const uint32_t jj = rg[(start + c) % kRing];
                    const uint4 *row = d2 + (int64_t)jj * kRow16;
                    uint4 rv[C];
#pragma unroll
                    for (int cc = 0; cc < C; cc++) rv[cc] = __ldg(row + chunk_of(cc));
                    float f = 0.0f;
#pragma unroll
                    for (int cc = 0; cc < C; cc++) {
                        float fc = 0.0f;
                        chunk_dist<KIND>(KIND, qdq[cc], rv[cc], acc[u], fc);
                        f = cc == 0 ? fc : f + fc;
                    }
                    if (kFlt) acc[u] = __float_as_uint(f);
                }
            }
            // transposed butterfly: after the step over lane bit h a lane keeps
            // the rounds whose bit h equals its own, summed with its partner's
#pragma unroll
            for (int h = G / 2; h >= 1; h >>= 1) {
                const bool up = (sub & h) != 0;
#pragma unroll
                for (int k = 0; k < h; k++) {
                    const uint32_t send = up ? acc[k] : acc[k + h];
                    const uint32_t keep = up ? acc[k + h] : acc[k];
                    const uint32_t got = __shfl_xor_sync(0xffffffffu, send, h);
                    acc[k] = kFlt ? __float_as_uint(__uint_as_float(keep) + __uint_as_float(got)) : keep + got;
                }
            }
            // lane (grp, sub) now holds the full distance of round sub
            const uint32_t c = (uint32_t)(sub * kPerRound + grp);
            if (c < nb) top2_key(((unsigned long long)acc[0] << 32) | rg[(start + c) % kRing], k1, k2);
            __syncwarp();
        };

        for (uint32_t base = 0; base < E; base += 32) {
            const uint32_t e = base + (uint32_t)lane;
            // the lane whose ranges hold element e: the last one whose first
            // element is <= e (it has elements, since the next one starts after e)
            int o = 0;
#pragma unroll
            for (int st = 16; st > 0; st >>= 1)
                if (__shfl_sync(0xffffffffu, p0, o + st) <= e) o += st;
            const uint32_t ob0 = __shfl_sync(0xffffffffu, w.b0, o), ol0 = __shfl_sync(0xffffffffu, w.len0, o);
            const uint32_t ob1 = __shfl_sync(0xffffffffu, w.b1, o), op0 = __shfl_sync(0xffffffffu, p0, o);
            bool cand = false;
            uint32_t j = 0;
            if (e < E) {
                const uint32_t off = e - op0;
                const float4 rc = __ldg(recb + (off < ol0 ? ob0 + off : ob1 + (off - ol0)));
                j = __float_as_uint(rc.w);
                nwin++;
                bool exact = exact_only;
                if (!exact) {
                    const float x = rc.x, y = rc.y, ee = rc.z;
                    const float d = fabsf(fmaf(rq.A, x, fmaf(rq.B, y, rq.C)));
                    const float Sm = fmaf(fabsf(rq.A), fabsf(x), fmaf(fabsf(rq.B), fabsf(y), fabsf(rq.C)));
                    // FP32 rounding (16u S), the FP32 tolerance (2u eps) and the
                    // distance between this line and the brute force's FP64 line
                    const float lerr = fmaf(rq.E1, fabsf(x) + fabsf(y) + 2.0f * ee, rq.E0);
                    const float bound = fmaf(9.6e-7f, Sm, fmaf(1.2e-7f, ee, lerr + 1e-9f));
                    cand = d <= ee - bound;
                    exact = !cand && !(d > ee + bound);
                }
                if (exact) {
                    // FP32 inconclusive: the brute-force FP64 expression decides
                    cand = exact_pair_p(PD.F, PD.xy1, PD.xy2, PD.eps2, PD.eps_scalar, q - PD.q_off, j);
                    nexact++;
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, cand);
            if (cand) rg[(count + (uint32_t)__popc(m & lt)) % kRing] = j;
            count += (uint32_t)__popc(m);
            if (count - done >= 32u) {
                batch(done, 32u);
                done += 32u;
            }
        }
        if (count > done) batch(done, count - done);
        ncand += count;
        if (lane == k) mine = count;
        // the query's best two over the lanes' best two: (distance, index) minima
        const uint32_t dk1 = (uint32_t)(k1 >> 32), jk1 = (uint32_t)k1;
        const uint32_t md = __reduce_min_sync(0xffffffffu, dk1);
        const uint32_t mj = __reduce_min_sync(0xffffffffu, dk1 == md ? jk1 : 0xffffffffu);
        const unsigned long long c2 = (dk1 == md && jk1 == mj) ? k2 : k1;
        const uint32_t dk2 = (uint32_t)(c2 >> 32), jk2 = (uint32_t)c2;
        const uint32_t sd = __reduce_min_sync(0xffffffffu, dk2);
        const uint32_t sj = __reduce_min_sync(0xffffffffu, dk2 == sd ? jk2 : 0xffffffffu);
        // the query's best two wait in shared memory; lane k writes query k's
        // outputs after the chunk
        if (lane == 0) res[warp][k] = make_uint4(md, mj, sd, sj);
    }
    __syncwarp();
    if (lane < nk) {
        const uint4 rr = res[warp][lane];
        const int64_t q = c0 + (int64_t)lane * step;
        store_match_kind(L, q, KIND, qchunk[warp][lane].flags, ((unsigned long long)rr.x << 32) | rr.y,
                         ((unsigned long long)rr.z << 32) | rr.w);
        if (L.qcount) L.qcount[q] = mine;
    }
    __syncwarp();  // the chunk's buffers are read before the next chunk's copies
    };

    if (ONE) {
        if (warp == 0) {
            const int k = load_pair_work(W, L.geom, lane);
            if (lane == 0) snlev = k;
        }
        __syncthreads();
        nlev = snlev;
        for (int64_t c0 = gw; c0 < L.nq; c0 += kChunkQ * nwarps)
            chunk(L.inl, c0, (int)min((int64_t)kChunkQ, (L.nq - c0 + nwarps - 1) / nwarps), nwarps);
    } else {
        for (int64_t q0 = gw * run; q0 < L.nq; q0 += nwarps * run) {
            const int64_t qe = min(q0 + run, L.nq);
            int64_t qa = q0;
            while (qa < qe) {
                const int np = L.qrec[qa].pair;
                const PairDesc &PD = L.pairs[np];
                if (np != p) {
                    p = np;
                    nlev = load_pair_work(W, L.geom + np, lane);
                }
                // the run's queries of this pair, in chunks of about the same size
                int left = (int)(min(qe, PD.q_off + (int64_t)PD.m) - qa);
                while (left > 0) {
                    const int parts = (left + kChunkQ - 1) / kChunkQ, nk = (left + parts - 1) / parts;
                    chunk(PD, qa, nk, 1);
                    qa += nk;
                    left -= nk;
                }
            }
        }
    }
    if (L.counters) {
        const uint32_t a = __reduce_add_sync(0xffffffffu, nwin);
        const uint32_t b = __reduce_add_sync(0xffffffffu, lane == 0 ? ncand : 0u);
        const uint32_t c = __reduce_add_sync(0xffffffffu, nexact);
        if (lane == 0) {
            atomicAdd(L.counters + 2, (unsigned long long)a);
            atomicAdd(L.counters + 3, (unsigned long long)b);
            atomicAdd(L.counters + 4, (unsigned long long)c);
        }
    }
}

template <int KIND, int G, int C, bool ONE>
cudaError_t launch_pair(const Launch &L, int sms, cudaStream_t s) {
    static int per_sm = 0;
    if (per_sm == 0) {
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, stab_pair_kernel<KIND, G, C, ONE>,
                                                                      kPairThreads, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
    }
    int64_t blocks = (L.nq + kPairWarps - 1) / kPairWarps;
    blocks = std::min<int64_t>(blocks, (int64_t)per_sm * sms);
    // several pairs: runs of about 32 queries (a pair's geometry is loaded once
    // per run; shorter runs spread pairs of uneven cost over the warps), all
    // queries in one round where they are few
    const int64_t warps = blocks * kPairWarps, rounds = std::max<int64_t>(L.nq / (warps * 32), 1);
    const int64_t run = (L.nq + warps * rounds - 1) / (warps * rounds);
    return launch_pdl(stab_pair_kernel<KIND, G, C, ONE>, dim3((unsigned)blocks), dim3(kPairThreads), 0, s, L, run);
}

// Whether a launch of stab_pair_kernel covers the call (then it is enqueued):
// every pair with rows of one kind and size.  Calls of one pair: u8 and
// binary rows of 16 .. 256 bytes, a power of two, and 64- and 128-d float
// rows; calls of several pairs: the sizes they are usually made of.
bool launch_warp_per_query(const Launch &L, int sms, cudaStream_t s, cudaError_t &e) {
    constexpr int U8 = EGM_DESC_U8_L2, F32 = EGM_DESC_F32_L2, BIN = EGM_DESC_BIN;
    const bool one = L.npairs == 1 && L.inl_use != 0;
    // rows of 32 bytes and more: a lane reads 32 bytes of a row
    switch (L.kind >= 0 && L.row_bytes > 0 ? L.kind * 4096 + L.row_bytes : -1) {
        case U8 * 4096 + 128:
            e = one ? launch_pair<U8, 4, 2, true>(L, sms, s) : launch_pair<U8, 4, 2, false>(L, sms, s);
            return true;
        case BIN * 4096 + 32:
            e = one ? launch_pair<BIN, 1, 2, true>(L, sms, s) : launch_pair<BIN, 1, 2, false>(L, sms, s);
            return true;
        case F32 * 4096 + 512:
            e = one ? launch_pair<F32, 16, 2, true>(L, sms, s) : launch_pair<F32, 16, 2, false>(L, sms, s);
            return true;
        default: break;
    }
    if (!one) return false;
    switch (L.kind >= 0 && L.row_bytes > 0 ? L.kind * 4096 + L.row_bytes : -1) {
        case U8 * 4096 + 16: e = launch_pair<U8, 1, 1, true>(L, sms, s); return true;
        case U8 * 4096 + 32: e = launch_pair<U8, 1, 2, true>(L, sms, s); return true;
        case U8 * 4096 + 64: e = launch_pair<U8, 2, 2, true>(L, sms, s); return true;
        case U8 * 4096 + 256: e = launch_pair<U8, 8, 2, true>(L, sms, s); return true;
        case BIN * 4096 + 16: e = launch_pair<BIN, 1, 1, true>(L, sms, s); return true;
        case BIN * 4096 + 64: e = launch_pair<BIN, 2, 2, true>(L, sms, s); return true;
        case BIN * 4096 + 128: e = launch_pair<BIN, 4, 2, true>(L, sms, s); return true;
        case BIN * 4096 + 256: e = launch_pair<BIN, 8, 2, true>(L, sms, s); return true;
        case F32 * 4096 + 256: e = launch_pair<F32, 8, 2, true>(L, sms, s); return true;
        default: return false;
    }
}

}  // namespace

cudaError_t launch_stab(const Launch &L, int sms, cudaStream_t s) {
    if (L.nq == 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (launch_warp_per_query(L, sms, s, e)) return e;
    int64_t blocks = (L.nq + kQB - 1) / kQB;
    if (blocks > 152 * 8) blocks = 152 * 8;
    const dim3 g((unsigned)blocks), b(kStabThreads);
    const auto kernel = L.kind == EGM_DESC_U8_L2    ? stab_kernel<EGM_DESC_U8_L2>
                        : L.kind == EGM_DESC_BIN    ? stab_kernel<EGM_DESC_BIN>
                        : L.kind == EGM_DESC_F32_L2 ? stab_kernel<EGM_DESC_F32_L2>
                                                    : stab_kernel<kKindAny>;
    // One pair of more than one block per SM: after its predecessor.  Placed
    // beside that kernel's clusters, the blocks pile up on the SMs they leave free
    // (float rows of 1,024 bytes: 256 blocks 821 us a call at 50 px against 753, 100
    // and 95 at 2 px; 125 blocks 400 against 393, but 82 against 86).
    if (L.npairs > 1 || blocks <= 152) return launch_pdl(kernel, g, b, 0, s, L);
    kernel<<<g, b, 0, s>>>(L);
    return cudaGetLastError();
}

}  // namespace egm
