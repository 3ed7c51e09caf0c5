// Candidate sets in CSR form (Eq. 4: C_i for every query, ascending index).
//
// The matching kernel of the call (plain or banded) leaves the number of
// candidates of every query in L.qcount; then
//
//   offset_tiles_kernel  sums of the counts over tiles of 4096 queries
//   offsets_kernel       exclusive prefix sum into cand_offsets, the total
//                        and the check of the caller's capacity
//   rows_kernel          a warp per query finds the query's candidates again
//                        (its windows, the exact test) and writes its row
//                        once, already in ascending order
#include "egm_internal.cuh"

namespace egm {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;
static_assert(kScanTile == kCountTile, "the scratch holds one partial per tile");

// Exclusive prefix sum of v over the block and the block's total.
__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t *warp_sums, int64_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
        int64_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        warp_sums[lane] = wi - w;
        if (lane == 31) warp_sums[32] = wi;
    }
    __syncthreads();
    const int64_t r = warp_sums[warp] + incl - v;
    total = warp_sums[32];
    __syncthreads();
    return r;
}

// The counts of this thread's four queries (zero past the last query).
__device__ __forceinline__ uint4 load_counts(const Launch &L, int64_t i) {
    if (i + 4 <= L.nq) return *reinterpret_cast<const uint4 *>(L.qcount + i);
    uint4 c = make_uint4(0, 0, 0, 0);
    if (i < L.nq) c.x = L.qcount[i];
    if (i + 1 < L.nq) c.y = L.qcount[i + 1];
    if (i + 2 < L.nq) c.z = L.qcount[i + 2];
    return c;
}

__global__ void __launch_bounds__(kScanThreads) offset_tiles_kernel(Launch L) {
    pdl_begin();
    __shared__ int64_t ws[33];
    const uint4 c = load_counts(L, (int64_t)blockIdx.x * kScanTile + 4 * threadIdx.x);
    int64_t total;
    block_excl_scan((int64_t)c.x + c.y + c.z + c.w, ws, total);
    if (threadIdx.x == 0) L.scan_tmp[blockIdx.x] = total;
}

// Each block adds up the sums of the tiles before its own (they are few: one
// per 4096 queries) instead of waiting for another launch to scan them.
__global__ void __launch_bounds__(kScanThreads) offsets_kernel(Launch L) {
    pdl_begin();
    __shared__ int64_t ws[33];
    int64_t before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) before += L.scan_tmp[b];
    int64_t base;
    block_excl_scan(before, ws, base);
    const int64_t i = (int64_t)blockIdx.x * kScanTile + 4 * threadIdx.x;
    const uint4 c = load_counts(L, i);
    int64_t total;
    const int64_t e0 = base + block_excl_scan((int64_t)c.x + c.y + c.z + c.w, ws, total);
    const int64_t e[4] = {e0, e0 + c.x, e0 + c.x + c.y, e0 + c.x + c.y + c.z};
#pragma unroll
    for (int k = 0; k < 4; k++)
        if (i + k < L.nq) L.cand_offsets[i + k] = e[k];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        L.cand_offsets[L.nq] = base + total;
        *L.cand_total = base + total;
        if (base + total > L.cand_capacity) atomicOr(L.status, kStCapacity);
    }
}

// ------------------------------------------------------------ rows
constexpr int kRowWarps = 4;
constexpr int kShortRow = 64;             // longest row sorted in registers
constexpr int kStage = 768;              // row entries (16-bit, from the step's first) staged for coalesced stores
constexpr uint32_t kLaneWords = 31;       // most bitmap words a lane walks per step; odd, and 32 * 32 * 31 < 2^16
constexpr int kMaxBits = 1 << 16;         // bitmap bits per warp: longer index ranges take several passes
constexpr int kSortRow = 1024;            // longest row sorted in registers there
static_assert(kSortRow <= kMaxBits / 32, "the bitmap's memory holds the row's candidates");

// Ascending sort of K = 32 or 64 keys, one or two per lane (lane l holds keys
// l and 32 + l), by a bitonic network: the step across 32 keys pairs the
// lane's own two, the others are shuffles.
template <int K>
__device__ __forceinline__ void sort_lanes(uint32_t &a, uint32_t &b, int lane) {
#pragma unroll
    for (int k = 2; k <= K; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j == 32) {
                const uint32_t lo = min(a, b), hi = max(a, b);
                a = lo;
                b = hi;
            } else {
                const bool low = (lane & j) == 0;
                // a block of k keys is sorted upwards when bit k of its keys' numbers is 0
                const bool ua = k == K || (lane & k) == 0;
                const uint32_t oa = __shfl_xor_sync(0xffffffffu, a, j);
                a = (low == ua) ? min(a, oa) : max(a, oa);
                if (K == 64) {
                    const bool ub = k == K || (((lane + 32) & k) == 0);
                    const uint32_t ob = __shfl_xor_sync(0xffffffffu, b, j);
                    b = (low == ub) ? min(b, ob) : max(b, ob);
                }
            }
        }
    }
}

// Ascending sort of K = 128 to 1024 keys, K / 32 per lane (lane l holds
// keys l, l + 32, ...), by a bitonic network: steps across 32 keys and more pair
// a lane's own keys, the others are shuffles.  (The loops over the shuffles'
// distances are not unrolled: of 512 keys 550 instructions in the place of
// 2,900.)
template <int K>
__device__ __forceinline__ void sort_regs(uint32_t (&a)[K / 32], int lane) {
    constexpr int R = K / 32;
    auto across = [&](int j, int r, bool up) {
        const uint32_t o = __shfl_xor_sync(0xffffffffu, a[r], j);
        a[r] = ((lane & j) == 0) == up ? min(a[r], o) : max(a[r], o);
    };
#pragma unroll 1
    for (int k = 2; k <= 16; k <<= 1)
#pragma unroll 1
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < R; r++) across(j, r, (lane & k) == 0);
#pragma unroll
    for (int q = 1; q <= R; q <<= 1) {  // blocks of 32 q keys
#pragma unroll
        for (int h = q >> 1; h > 0; h >>= 1)
#pragma unroll
            for (int r = 0; r < R; r++)
                if ((r & h) == 0) {
                    const bool up = q == R || (r & q) == 0;
                    const uint32_t lo = min(a[r], a[r | h]), hi = max(a[r], a[r | h]);
                    a[r] = up ? lo : hi;
                    a[r | h] = up ? hi : lo;
                }
#pragma unroll 1
        for (int j = 16; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < R; r++) across(j, r, q == R || (r & q) == 0);
    }
}

// `have` <= K keys of `list` in ascending order to `out`; the list is zero afterwards.
template <int K>
__device__ __forceinline__ void write_sorted(uint32_t *list, uint32_t have, int32_t *out, int lane) {
    uint32_t a[K / 32];
#pragma unroll
    for (int r = 0; r < K / 32; r++) {
        a[r] = (uint32_t)(32 * r + lane) < have ? list[32 * r + lane] : ~0u;
        list[32 * r + lane] = 0u;
    }
    sort_regs<K>(a, lane);
#pragma unroll
    for (int r = 0; r < K / 32; r++)
        if ((uint32_t)(32 * r + lane) < have) out[32 * r + lane] = (int32_t)a[r];
}

// One warp per query.  The query's windows are computed by its lanes (lane =
// level) and flattened by a prefix sum; the warp tests 32 window elements per
// step.  Rows of up to 64 candidates are collected and sorted in registers.
// Longer rows are sorted by construction: each candidate sets its bit in the
// warp's bitmap over the pair's references, and the warp then walks the
// bitmap in index order, W words per lane and step, and writes the indices of
// the set bits through a staging buffer, so the row leaves in coalesced
// stores.  The work per row is its window plus n / 1024 words per lane
// whatever the row's length; there is no exchange between elements and no
// second pass over the row.  (Rows above 1024 entries used to be written
// unsorted and sorted one after the other by a single block: the rows of
// 50,000 queries of about 1,200 candidates each took 1.54 s, and the second
// pass of the matching kernel that wrote them 0.76 ms; this kernel takes
// 0.28 ms.)  It is bound by instruction issue, 72 % active: 224 M warp
// instructions.  Two things keep them few: a step whose 32 elements lie in one
// range looks up its range once for the warp (each lane for its own element:
// 279 M and 0.34 ms), and a lane's words are many, so that the lanes' numbers
// of set bits differ little (4 words per lane and step: 345 M and 0.50 ms;
// 15 words: 10 % more time on the whole call than 31).  The staging buffer is
// 16-bit and no larger than 28 resident warps per SM allow, which is also the
// registers' limit (1024 entries: 24 warps, 4 % on the whole call).
//
// Index ranges beyond kMaxBits take one pass over the windows per range, and
// medium rows there are collected and sorted in registers (LARGE: an instance
// of its own, for calls with such an image).  With one bitmap for up to 262,144
// references, whose memory left one block per SM, and every row walked from it:
// offsets and rows of 20,000 queries of 100 candidates each 429 us at 262,144
// references and 1,870 at 1,048,576, now 65 and 112; of 500 candidates 630 and
// 2,330, now 200 and 253.
template <bool LARGE>
__global__ void __launch_bounds__(kRowWarps * 32, LARGE ? 5 : 0) rows_kernel(Launch L, int words) {
    pdl_begin();
    extern __shared__ __align__(16) uint32_t rsm[];
    if (L.cand_offsets[L.nq] > L.cand_capacity) return;  // capacity error: no row is written
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t *bm = rsm + warp * (words + kStage / 2);
    uint16_t *stage = reinterpret_cast<uint16_t *>(bm + words);
    for (int k = lane; k < words; k += 32) bm[k] = 0u;
    __syncwarp();
    const int64_t nwarps = (int64_t)gridDim.x * kRowWarps;
    for (int64_t q = (int64_t)blockIdx.x * kRowWarps + warp; q < L.nq; q += nwarps) {
        const int64_t row = L.cand_offsets[q];
        const uint32_t len = (uint32_t)(L.cand_offsets[q + 1] - row);
        if (len == 0) continue;
        const QueryRec r = L.qrec[q];
        const PairDesc &P = L.pairs[r.pair];
        const PairGeom &G = L.geom[r.pair];
        const int64_t qi = q - P.q_off;
        const uint32_t n = (uint32_t)P.n;
        const float4 *recb = L.rec + P.r_off;
        const WinKeys wk = window_keys(G, r, lane);
        uint32_t ta = 0, tb = 0;
        if (wk.kind >= 2) {
            const uint32_t *T = L.tab + P.t_off + G.tab[lane];
            ta = __ldg(T + wk.ta);
            tb = __ldg(T + wk.tb);
        }
        const Window w = window_ranges(wk, ta, tb);
        const uint32_t tl = w.len0 + w.len1;
        uint32_t incl = tl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const uint32_t p0 = incl - tl;  // first flattened element of this lane's ranges
        const uint32_t E = __shfl_sync(0xffffffffu, incl, 31);
        const bool exact_only = (r.flags & kQExactOnly) != 0;
        // the pre-test bound of the banded form: k1 (|x| + |y|) + ke eps + k0
        const float k1 = 9.6e-7f * 1.00001f + r.E1;
        const float ke = 1.2e-7f + 2.0f * r.E1;
        const float k0 = fmaf(9.6e-7f, fabsf(r.C), r.E0 + 1e-9f);
        auto is_candidate = [&](const float4 &rc) {
            const float d = fabsf(fmaf(r.A, rc.x, fmaf(r.B, rc.y, r.C)));
            const float bound = fmaf(k1, fabsf(rc.x) + fabsf(rc.y), fmaf(ke, rc.z, k0));
            const bool cand = !exact_only && d <= rc.z - bound;
            // FP32 inconclusive: the brute-force FP64 expression decides
            if (exact_only || (!cand && !(d > rc.z + bound))) return exact_pair(P, qi, __float_as_uint(rc.w));
            return cand;
        };
        // every candidate of the query, 32 window elements per step: f(is candidate, index)
        auto visit = [&](auto f) {
            for (uint32_t base = 0; base < E;) {
                // the lane whose ranges hold element `base`: the last one that starts at or before it
                int o = __popc(__ballot_sync(0xffffffffu, p0 <= base)) - 1;
                uint32_t op0 = __shfl_sync(0xffffffffu, p0, o);
                uint32_t ob0 = __shfl_sync(0xffffffffu, w.b0, o), ol0 = __shfl_sync(0xffffffffu, w.len0, o);
                uint32_t ob1 = __shfl_sync(0xffffffffu, w.b1, o);
                const uint32_t off0 = base - op0;
                const uint32_t left = (off0 < ol0 ? ol0 : __shfl_sync(0xffffffffu, tl, o)) - off0;
                if (left >= 32u) {  // whole steps within one range: no element looks its own up
                    const float4 *at = recb + (off0 < ol0 ? ob0 + off0 : ob1 + (off0 - ol0)) + lane;
                    const uint32_t end = base + (left & ~31u);
                    float4 next = __ldg(at);
                    while (base < end) {
                        const float4 rc = next;
                        base += 32;
                        at += 32;
                        if (base < end) next = __ldg(at);
                        f(is_candidate(rc), __float_as_uint(rc.w));
                    }
                    continue;
                }
                const uint32_t e = base + (uint32_t)lane;
                o = 0;
#pragma unroll
                for (int st = 16; st > 0; st >>= 1)
                    if (__shfl_sync(0xffffffffu, p0, o + st) <= e) o += st;
                op0 = __shfl_sync(0xffffffffu, p0, o);
                ob0 = __shfl_sync(0xffffffffu, w.b0, o);
                ol0 = __shfl_sync(0xffffffffu, w.len0, o);
                ob1 = __shfl_sync(0xffffffffu, w.b1, o);
                bool cand = false;
                uint32_t j = 0;
                if (e < E) {
                    const uint32_t off = e - op0;
                    const float4 rc = __ldg(recb + (off < ol0 ? ob0 + off : ob1 + (off - ol0)));
                    j = __float_as_uint(rc.w);
                    cand = is_candidate(rc);
                }
                f(cand, j);
                base += 32;
            }
        };
        int32_t *out = L.cand_idx + row;
        if (len <= (uint32_t)kShortRow) {
            uint32_t *srow = bm + words;
            uint32_t count = 0;
            visit([&](bool cand, uint32_t j) {
                const uint32_t m = __ballot_sync(0xffffffffu, cand);
                const uint32_t slot = count + (uint32_t)__popc(m & lt);
                if (cand && slot < (uint32_t)kShortRow) srow[slot] = j;
                count += (uint32_t)__popc(m);
            });
            __syncwarp();
            const uint32_t have = min(count, len);
            uint32_t a = (uint32_t)lane < have ? srow[lane] : ~0u;
            uint32_t b = (uint32_t)lane + 32u < have ? srow[lane + 32] : ~0u;
            if (have <= 32u) sort_lanes<32>(a, b, lane);
            else sort_lanes<64>(a, b, lane);
            if ((uint32_t)lane < have) out[lane] = (int32_t)a;
            if ((uint32_t)lane + 32u < have) out[lane + 32] = (int32_t)b;
            __syncwarp();
            continue;
        }
        // sorted in registers; of two ranges (two passes) rows of up to 512 only: up to 1024, 189 us against 175 with the
        // passes (131,072 references, rows of about 500), of four ranges 198 against 285
        if (LARGE && n > (uint32_t)kMaxBits && len <= (n > 2u * kMaxBits ? (uint32_t)kSortRow : kSortRow / 2u)) {
            uint32_t count = 0;  // the candidates, in the bitmap's memory
            visit([&](bool cand, uint32_t j) {
                const uint32_t m = __ballot_sync(0xffffffffu, cand);
                const uint32_t slot = count + (uint32_t)__popc(m & lt);
                if (cand && slot < len) bm[slot] = j;
                count += (uint32_t)__popc(m);
            });
            __syncwarp();
            const uint32_t have = min(count, len);
            if (have <= 128u) write_sorted<128>(bm, have, out, lane);
            else if (have <= 256u) write_sorted<256>(bm, have, out, lane);
            else if (have <= 512u) write_sorted<512>(bm, have, out, lane);
            else write_sorted<kSortRow>(bm, have, out, lane);
            __syncwarp();
            continue;
        }
        const uint32_t nbits = 32u * (uint32_t)words;
        uint32_t done = 0;  // entries of the row written
        for (uint32_t j0 = 0; j0 < n; j0 += nbits) {
            visit([&](bool cand, uint32_t j) {
                const uint32_t k = j - j0;  // wraps to a large value below the range
                if (cand && k < nbits) atomicOr(&bm[k >> 5], 1u << (k & 31u));
            });
            __syncwarp();
            // the walk in equal steps: lane l takes W words from l W on.  W is odd, so the lanes'
            // words of one turn lie in different banks.
            const uint32_t used = (min(nbits, n - j0) + 31u) / 32u;
            const uint32_t steps = (used + 32u * kLaneWords - 1u) / (32u * kLaneWords);
            const uint32_t W = ((used + 32u * steps - 1u) / (32u * steps)) | 1u;
            for (uint32_t w0 = 0; w0 < used; w0 += 32u * W) {
                const uint32_t first = w0 + W * (uint32_t)lane;
                const uint32_t mine = first < used ? min(W, used - first) : 0u;
                uint32_t c = 0, full = 0;  // set bits and nonzero words of this lane
                for (uint32_t k = 0; k < mine; k++) {
                    const uint32_t v = bm[first + k];
                    c += (uint32_t)__popc(v);
                    full |= (v ? 1u : 0u) << k;
                }
                uint32_t ci = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xffffffffu, ci, o);
                    if (lane >= o) ci += x;
                }
                const uint32_t tot = __shfl_sync(0xffffffffu, ci, 31);
                if (tot == 0) continue;
                const bool staged = tot <= (uint32_t)kStage;
                uint32_t at = ci - c;
                const uint32_t end = ci;
                uint32_t v = 0, jw = 0;
                while (at < end) {
                    if (v == 0) {
                        const uint32_t k = first + (uint32_t)__ffs((int)full) - 1u;
                        full &= full - 1u;
                        v = bm[k];
                        bm[k] = 0u;
                        jw = 32u * (k - w0);
                    }
                    const uint32_t j = jw + (uint32_t)__ffs((int)v) - 1u;
                    v &= v - 1u;
                    if (staged) stage[at] = (uint16_t)j;
                    else if (done + at < len) out[done + at] = (int32_t)(j0 + 32u * w0 + j);
                    at++;
                }
                __syncwarp();
                if (staged) {
                    for (uint32_t k = (uint32_t)lane; k < tot; k += 32u)
                        if (done + k < len) out[done + k] = (int32_t)(j0 + 32u * w0 + stage[k]);
                    __syncwarp();
                }
                done += tot;
            }
            __syncwarp();
        }
    }
}

}  // namespace

cudaError_t launch_csr_offsets(const Launch &L, cudaStream_t s) {
    const unsigned nb = (unsigned)std::max<int64_t>((L.nq + kScanTile - 1) / kScanTile, 1);
    cudaError_t e = cudaSuccess;
    // a single tile has no earlier sums to add
    if (nb > 1) e = launch_pdl(offset_tiles_kernel, dim3(nb), dim3(kScanThreads), 0, s, L);
    if (e != cudaSuccess) return e;
    return launch_pdl(offsets_kernel, dim3(nb), dim3(kScanThreads), 0, s, L);
}

cudaError_t launch_csr_rows(const Launch &L, int sms, cudaStream_t s) {
    if (L.nq == 0 || L.nr == 0) return cudaSuccess;
    const int words = (int)((std::min<int64_t>(L.max_n, kMaxBits) + 31) / 32);  // the largest image of the call
    const bool large = L.max_n > kMaxBits;
    const auto kernel = large ? rows_kernel<true> : rows_kernel<false>;
    const size_t smem = sizeof(uint32_t) * kRowWarps * (size_t)(words + kStage / 2);
    // the limit is the function's on the device, shared with other contexts'
    // threads: always the largest any call needs
    constexpr int kMostSmem = (int)sizeof(uint32_t) * kRowWarps * (kMaxBits / 32 + kStage / 2);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kRowWarps * 32, smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::min<int64_t>((L.nq + kRowWarps - 1) / kRowWarps, (int64_t)std::max(per_sm, 1) * sms);
    return launch_pdl(kernel, dim3((unsigned)blocks), dim3(kRowWarps * 32), smem, s, L, words);
}

}  // namespace egm
