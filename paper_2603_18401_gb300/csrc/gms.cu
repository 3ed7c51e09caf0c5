// Grid-based motion statistics (GMS) filter of the matches of a batch of
// pairs (one pair: a batch of one): the filter
// the paper applies to its guided matches by default, with the neighbour
// threshold 6 (Sec. 5.1; Sec. 4.3 names GMS as suited to guided matching).
// GMS is from Bian et al. (CVPR 2017):
//
//   cells      image 1: floor(x * G / W1 + s) for a grid shift s in {0, 1/2}
//              (clamped to 0 .. G), image 2: floor(x * G / W2) (0 .. G - 1);
//              FP64 with one rounding per operation
//   motion     M[c][d] = matches from image-1 cell c to image-2 cell d,
//              N[c] = matches in c; d*(c) = argmax_d M[c][d] (lowest d on ties)
//   score      S(c) = sum over the 3 x 3 offsets o of M[c + o][d*(c) + o]
//   keep       d == d*(c) and S(c) > alpha * sqrt(sum_o N[c + o] / 9),
//              the union over the four shifts
//
// Rows of all pairs are concatenated (pair p's rows start at row_off[p]).
// gms_prep_kernel: one thread per row; the image-1 column and row of the grid
// with and without the half-cell shift (a byte each) and the image-2 cell.
// gms_cells_kernel: one block per (pair, shift, run of up to `span` cells of
// one image-1 grid row); its 3 x (span + 2) neighbourhood of M is a table in
// shared memory, filled from all of the pair's matches; then a warp per cell
// takes d* and S.  The decision of each cell (d* or -1) goes to a table per
// pair and shift.
// gms_sorted_kernel: the same for many pairs or fine grids, one block per
// (pair, shift): a counting sort of its matches by image-1 cell, then a warp per
// cell over the cell's own list.
// gms_flag_kernel: one thread per row sets or clears EGM_FLAG_GMS.
#include "egm_internal.cuh"

namespace egm {

namespace {

constexpr int kGmsThreads = 512;
constexpr int kGmsWarps = kGmsThreads / 32;
constexpr int kSortedThreads = 1024;  // gms_sorted_kernel
constexpr int kSortedWarps = kSortedThreads / 32;
constexpr int kGmsSmemBudget = 200 * 1024;

constexpr uint16_t kNoCell = 0xFFFF;

__device__ __forceinline__ int clamp_cell(double t, int top) {
    const double f = floor(t);
    if (!(f > 0.0)) return 0;  // also NaN
    return f >= (double)top ? top : (int)f;
}

// Cells of coordinate v: c0 = clamp(floor(v * G / size)) to 0 .. top and, for
// the shifted grid, c1 = clamp(floor(v * G / size + 1/2)), both with the FP64
// operations rounded as written.  An FP32 quotient decides when it is further
// than 1e-3 from a multiple of 1/2: it is within 1e-4 of the exact value for
// quotients up to 64, so the floors are the same; otherwise (and outside that
// range) the FP64 formula itself runs (a division on GB300's FP64 pipe).
__device__ __forceinline__ void grid_cells(double v, int G, double size, int top, int &c0, int &c1) {
    const float t = __double2float_rn(v) * (float)G / __double2float_rn(size);
    const float h = 2.0f * t, r = rintf(h);
    if (fabsf(h - r) > 2e-3f && t > 0.0f && t < 64.0f) {
        c0 = min((int)t, top);
        c1 = min((int)(t + 0.5f), top);
        return;
    }
    const double d = __ddiv_rn(__dmul_rn(v, (double)G), size);
    c0 = clamp_cell(d, top);
    c1 = clamp_cell(__dadd_rn(d, 0.5), top);
}

struct GmsArgs {
    const GmsPair *pairs;
    const int64_t *row_offs;  // npairs + 1
    int32_t npairs;
    int64_t rows;
    uint32_t require;
    int G;
    double alpha;
    GmsPair one;              // a single pair's entry (no table to read)
};

__device__ __forceinline__ int gms_pair_of(const GmsArgs &a, const int64_t *s_offs, bool cached, int64_t i) {
    if (a.npairs == 1) return 0;
    return cached ? pair_of_shared(s_offs, a.npairs, i) : pair_of(a.row_offs, a.npairs, i);
}

// cells1[i] = the image-1 cell of row i: column without and with the shift in
// bytes 0 and 1, row without and with it in bytes 2 and 3; cell2[i] = its
// image-2 cell, kNoCell where row i is not an input match
__global__ void __launch_bounds__(128) gms_prep_kernel(const __grid_constant__ GmsArgs a, uint32_t *cells1,
                                                       uint16_t *cell2) {
    pdl_begin();
    __shared__ int64_t s_offs[kSmemPairs + 1];
    const bool cached = a.npairs > 1 && load_offsets(s_offs, a.row_offs, a.npairs);
    __syncthreads();
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < a.rows;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int p = gms_pair_of(a, s_offs, cached, g);
        const GmsPair &P = a.npairs == 1 ? a.one : a.pairs[p];
        const int64_t i = g - P.row_off;
        const int32_t j = P.best[i];
        const bool in = j >= 0 && j < P.n && (P.flags[i] & a.require) == a.require;
        uint32_t c1 = 0;
        uint16_t c2 = kNoCell;
        if (in) {
            const int G = a.G;
            int x0, x1, y0, y1, dx, dy, unused;
            grid_cells(P.xy1[2 * i], G, P.w1, G, x0, x1);
            grid_cells(P.xy1[2 * i + 1], G, P.h1, G, y0, y1);
            grid_cells(P.xy2[2 * (int64_t)j], G, P.w2, G - 1, dx, unused);
            grid_cells(P.xy2[2 * (int64_t)j + 1], G, P.h2, G - 1, dy, unused);
            c1 = (uint32_t)x0 | ((uint32_t)x1 << 8) | ((uint32_t)y0 << 16) | ((uint32_t)y1 << 24);
            c2 = (uint16_t)(dy * G + dx);
        }
        cells1[g] = c1;
        cell2[g] = c2;
    }
}

// Column and row of a match's image-1 cell under shift s.
__device__ __forceinline__ int shift_x(uint32_t c, int s) { return (c >> ((s & 1) * 8)) & 0xff; }
__device__ __forceinline__ int shift_y(uint32_t c, int s) { return (c >> (16 + (s >> 1) * 8)) & 0xff; }

// Dynamic shared memory: count, start, cursor, dstar [(G + 1)^2] int32, then
// the histograms of `hw` warps, G^2 uint32 each.  Block b: pair b / 4, shift b % 4.
// dsorted: the pair and shift's image-2 cells in image-1 cell order.
__global__ void __launch_bounds__(kSortedThreads, 1) gms_sorted_kernel(const __grid_constant__ GmsArgs a, int hw,
                                                                    const uint32_t *cells1, const uint16_t *cell2,
                                                                    uint16_t *dsorted, int32_t *decision) {
    pdl_begin();
    extern __shared__ __align__(16) uint32_t gsm[];
    const int G = a.G, G1 = G + 1, C1 = G1 * G1, C2 = G * G;
    const int p = blockIdx.x >> 2, s = blockIdx.x & 3;
    const GmsPair &P = a.npairs == 1 ? a.one : a.pairs[p];
    const int64_t m = P.m, roff = P.row_off;
    const uint32_t *c1 = cells1 + roff;
    const uint16_t *c2 = cell2 + roff;
    int32_t *count = reinterpret_cast<int32_t *>(gsm), *start = count + C1, *cursor = count + 2 * C1,
            *dstar = count + 3 * C1;
    uint32_t *hist = gsm + 4 * C1;
    uint16_t *ds = dsorted + 4 * roff + (int64_t)s * m;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto cell_of = [&](uint32_t c) { return shift_y(c, s) * G1 + shift_x(c, s); };

    for (int k = threadIdx.x; k < C1; k += kSortedThreads) count[k] = 0, cursor[k] = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < m; i += kSortedThreads)
        if (c2[i] != kNoCell) atomicAdd(&count[cell_of(c1[i])], 1);
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the counts
        int carry = 0;
        for (int b = 0; b < C1; b += 32) {
            const int v = b + lane < C1 ? count[b + lane] : 0;
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            if (b + lane < C1) start[b + lane] = carry + incl - v;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < m; i += kSortedThreads) {
        const uint16_t d = c2[i];
        if (d == kNoCell) continue;
        const int c = cell_of(c1[i]);
        ds[start[c] + atomicAdd(&cursor[c], 1)] = d;
    }
    __syncthreads();

    // d*(c): the most frequent image-2 cell of c's list, the lowest on ties
    if (warp < hw) {
        uint32_t *h = hist + (size_t)warp * C2;
        for (int c = warp; c < C1; c += hw) {
            const int len = count[c];
            if (len == 0) {
                if (lane == 0) dstar[c] = -1;
                continue;
            }
            for (int b = lane; b < C2; b += 32) h[b] = 0u;
            __syncwarp();
            const uint16_t *lst = ds + start[c];
            for (int k = lane; k < len; k += 32) atomicAdd(&h[lst[k]], 1u);
            __syncwarp();
            uint32_t bc = 0;
            int bb = C2;
            for (int b = lane; b < C2; b += 32) {
                const uint32_t v = h[b];
                if (v > bc) bc = v, bb = b;  // ascending b: the first maximum of this lane
            }
            const uint32_t top = __reduce_max_sync(0xffffffffu, bc);
            const int d = (int)__reduce_min_sync(0xffffffffu, bc == top ? (uint32_t)bb : (uint32_t)C2);
            if (lane == 0) dstar[c] = d;
            __syncwarp();
        }
    }
    __syncthreads();

    // S(c) and the threshold
    int32_t *dec = decision + (int64_t)blockIdx.x * C1;
    for (int c = warp; c < C1; c += kSortedWarps) {
        const int d = dstar[c];
        int32_t res = -1;
        if (d >= 0) {
            const int cx = c % G1, cy = c / G1, dx = d % G, dy = d / G;
            uint32_t S = 0, total = 0;
            for (int o = 0; o < 9; o++) {
                const int ox = o % 3 - 1, oy = o / 3 - 1;
                const int ax = cx + ox, ay = cy + oy;
                if (ax < 0 || ax >= G1 || ay < 0 || ay >= G1) continue;
                const int ac = ay * G1 + ax;
                total += (uint32_t)count[ac];
                const int bx = dx + ox, by = dy + oy;
                if (bx < 0 || bx >= G || by < 0 || by >= G) continue;
                const uint16_t target = (uint16_t)(by * G + bx);
                const uint16_t *lst = ds + start[ac];
                uint32_t k0 = 0;
                for (int k = lane; k < count[ac]; k += 32) k0 += lst[k] == target;
                S += __reduce_add_sync(0xffffffffu, k0);
            }
            const double thr = __dmul_rn(a.alpha, __dsqrt_rn(__ddiv_rn((double)total, 9.0)));
            if ((double)S > thr) res = d;
        }
        if (lane == 0) dec[c] = res;
    }
}

// Dynamic shared memory: per cell of the block's 3 x (span + 2) neighbourhood
// its row of M (C2 = G^2 counts), then its match count and its d*.  Block:
// (run of cells in a grid row, grid row, pair * 4 + shift).
//
// One block used to take a whole (pair, shift): a counting sort of its
// matches, then 441 cells in turns, 132 us for one pair on four SMs.  A block
// per grid row reads every match of the pair (6 bytes each, from L2) and
// keeps the ones of its three grid rows, which needs no order and puts 84
// blocks on a pair: 132 -> 14.6 us (16,384 matches, 20 x 20 cells).  Where
// the pairs fill the SMs or the grid's tables fill the shared memory, reading
// every match again costs more than sorting them once: rows_take_less picks.
__global__ void __launch_bounds__(kGmsThreads) gms_cells_kernel(const __grid_constant__ GmsArgs a, int span,
                                                                const uint32_t *cells1, const uint16_t *cell2,
                                                                int32_t *decision) {
    pdl_begin();
    extern __shared__ __align__(16) uint32_t gsm[];
    const int G = a.G, G1 = G + 1, C2 = G * G, W = span + 2, nc = 3 * W;
    const int y = blockIdx.y, x0 = blockIdx.x * span, xe = min(x0 + span, G1);  // cells (x0 .. xe - 1, y)
    const int p = blockIdx.z >> 2, s = blockIdx.z & 3;
    const GmsPair &P = a.npairs == 1 ? a.one : a.pairs[p];
    const int64_t m = P.m;
    const uint32_t *c1 = cells1 + P.row_off;
    const uint16_t *c2 = cell2 + P.row_off;
    uint32_t *hist = gsm, *count = gsm + nc * C2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k < nc * (C2 + 1); k += kGmsThreads) gsm[k] = 0u;
    __syncthreads();
    // the matches of the neighbourhood's cells; four rows per thread and step,
    // loaded together
    for (int64_t i0 = 0; i0 < m; i0 += 4 * kGmsThreads) {
        uint32_t c[4];
        uint16_t d[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int64_t i = i0 + k * kGmsThreads + tid;
            d[k] = kNoCell;
            if (i < m) {
                c[k] = c1[i];
                d[k] = c2[i];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (d[k] == kNoCell) continue;
            const int dy = shift_y(c[k], s) - (y - 1), dx = shift_x(c[k], s) - (x0 - 1);
            if ((unsigned)dy < 3u && (unsigned)dx < (unsigned)W) {
                const int cell = dy * W + dx;
                atomicAdd(&hist[cell * C2 + d[k]], 1u);
                atomicAdd(&count[cell], 1u);
            }
        }
    }
    __syncthreads();
    int32_t *dec = decision + (int64_t)blockIdx.z * G1 * G1 + y * G1;
    for (int x = x0 + warp; x < xe; x += kGmsWarps) {
        const int cell = W + (x - x0 + 1);
        int32_t res = -1;
        if (count[cell] > 0) {
            // d*: the most frequent image-2 cell, the lowest on ties
            const uint32_t *h = hist + cell * C2;
            uint32_t bc = 0;
            int bb = C2;
            for (int b = lane; b < C2; b += 32) {
                const uint32_t v = h[b];
                if (v > bc) bc = v, bb = b;  // ascending b: the first maximum of this lane
            }
            const uint32_t top = __reduce_max_sync(0xffffffffu, bc);
            const int d = (int)__reduce_min_sync(0xffffffffu, bc == top ? (uint32_t)bb : (uint32_t)C2);
            // S and the neighbourhood's matches: lane o of 9 takes offset o
            const int ox = lane % 3 - 1, oy = lane / 3 - 1;
            const int ax = x + ox, ay = y + oy, bx = d % G + ox, by = d / G + oy;
            const bool in1 = lane < 9 && ax >= 0 && ax < G1 && ay >= 0 && ay < G1;
            const bool in2 = in1 && bx >= 0 && bx < G && by >= 0 && by < G;
            const int nb = in1 ? cell + oy * W + ox : cell;
            const uint32_t total = __reduce_add_sync(0xffffffffu, in1 ? count[nb] : 0u);
            const uint32_t S = __reduce_add_sync(0xffffffffu, in2 ? hist[nb * C2 + by * G + bx] : 0u);
            const double thr = __dmul_rn(a.alpha, __dsqrt_rn(__ddiv_rn((double)total, 9.0)));
            if ((double)S > thr) res = d;
        }
        if (lane == 0) dec[x] = res;
    }
}

__global__ void __launch_bounds__(128) gms_flag_kernel(const __grid_constant__ GmsArgs a, const uint32_t *cells1,
                                                       const uint16_t *cell2, const int32_t *decision) {
    pdl_begin();
    __shared__ int64_t s_offs[kSmemPairs + 1];
    const bool cached = a.npairs > 1 && load_offsets(s_offs, a.row_offs, a.npairs);
    __syncthreads();
    const int G1 = a.G + 1, C1 = G1 * G1;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < a.rows;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int p = gms_pair_of(a, s_offs, cached, g);
        const GmsPair &P = a.npairs == 1 ? a.one : a.pairs[p];
        const int64_t i = g - P.row_off;
        const uint16_t d = cell2[g];
        bool keep = false;
        if (d != kNoCell) {
            const uint32_t c = cells1[g];
            const int32_t *dec = decision + (int64_t)p * 4 * C1;
#pragma unroll
            for (int s = 0; s < 4; s++) keep |= dec[s * C1 + shift_y(c, s) * G1 + shift_x(c, s)] == d;
        }
        const uint8_t f = P.flags[i];
        P.flags[i] = (uint8_t)((f & ~EGM_FLAG_GMS) | (keep ? EGM_FLAG_GMS : 0));
    }
}

// The cells kernel's split: a grid row of cells per block where its tables fit
// the shared memory (up to 24 x 24 cells), else equal runs of cells.
struct GmsRuns {
    int runs, span;
    size_t smem;
    explicit GmsRuns(int grid) {
        const int G1 = grid + 1;
        const size_t column = (size_t)3 * (grid * grid + 1) * sizeof(uint32_t);  // tables of three cells
        const int most = std::max((int)(kGmsSmemBudget / column) - 2, 1);
        runs = (G1 + most - 1) / most;
        span = (G1 + runs - 1) / runs;
        smem = column * (size_t)(span + 2);
    }
};

// Whether the cells kernel (a block per run of a grid row, which reads every
// match of its pair) takes less time than the sorted one (a block per pair and
// shift): both in us, as rounds of resident blocks times a block's time.  A
// block of the first clears its tables and reads m matches; one of the second
// takes its populated cells in turn.  Fitted to grids of 10 to 48 cells, 500 to
// 100,000 matches and 1 to 128 pairs, where the one picked is never the slower
// one by more than 1.4 and never slower than the sorted one: 32 pairs of 16,384
// matches at 20 x 20 cells 160 against 227, at 28 x 28 470 against 264, at
// 48 x 48 2,836 against 728; one pair there 99 against 772.
bool rows_take_less(int npairs, int64_t rows, int grid) {
    const GmsRuns r(grid);
    const int G1 = grid + 1, C2 = grid * grid;
    const double m = (double)rows / npairs;
    const int per_sm = std::max(std::min((int)(227 * 1024 / (r.smem + 1024)), 4), 1);
    const double block = (3.0 + 8e-5 * (double)(r.smem / sizeof(uint32_t)) + 3e-4 * m) * (per_sm == 1 ? 1.0 : 1.35);
    const double by_rows = 4.0 * npairs * G1 * r.runs / (152.0 * per_sm) * block;
    const double cells = std::min(m, (double)G1 * G1);
    const double sorted = (30.0 + 0.19 * cells + 6e-5 * cells * C2 + 2e-3 * m) * std::max(1.0, 4.0 * npairs / 152.0);
    return by_rows < sorted;
}

}  // namespace

// scratch: pair table | row offsets | decisions 4 npairs (G + 1)^2 x 32 bit |
// image-1 cells rows x 32 bit | image-2 cells rows x 16 bit | sorted form: the
// lists of the four shifts, 4 rows x 16 bit
GmsLayout gms_layout(int npairs, int64_t rows, int grid) {
    GmsLayout l;
    l.table = 0;
    l.offs = align256(sizeof(GmsPair) * (size_t)npairs);
    l.dec = l.offs + align256(sizeof(int64_t) * (size_t)(npairs + 1));
    l.c1 = l.dec + align256((size_t)4 * npairs * (grid + 1) * (grid + 1) * sizeof(int32_t));
    l.c2 = l.c1 + align256((size_t)rows * sizeof(uint32_t));
    l.ds = l.c2 + align256((size_t)rows * sizeof(uint16_t));
    l.sorted = rows > 0 && npairs > 0 && !rows_take_less(npairs, rows, grid);
    l.total = l.ds + (l.sorted ? align256((size_t)4 * (size_t)rows * sizeof(uint16_t)) : 0);
    return l;
}

cudaError_t launch_gms(void *scratch, const GmsLayout &l, const GmsPair *one, int npairs, int64_t rows,
                       uint32_t require, int grid, double alpha, cudaStream_t st) {
    if (rows == 0 || npairs == 0) return cudaSuccess;
    char *b = static_cast<char *>(scratch);
    GmsArgs a{reinterpret_cast<const GmsPair *>(b + l.table), reinterpret_cast<const int64_t *>(b + l.offs),
              npairs, rows, require, grid, alpha, *one};
    int32_t *dec = reinterpret_cast<int32_t *>(b + l.dec);
    uint32_t *c1 = reinterpret_cast<uint32_t *>(b + l.c1);
    uint16_t *c2 = reinterpret_cast<uint16_t *>(b + l.c2);
    const int G1 = grid + 1;
    // the limits are the functions' on the device, shared with other contexts'
    // threads: always the largest any grid needs (the tables of three cells,
    // the least a block takes, fit the budget up to 48 x 48 cells)
    cudaError_t e = l.sorted ? cudaFuncSetAttribute(gms_sorted_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    kGmsSmemBudget)
                             : cudaFuncSetAttribute(gms_cells_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    kGmsSmemBudget);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::min<int64_t>((rows + 127) / 128, 152 * 16);
    if ((e = launch_pdl(gms_prep_kernel, dim3((unsigned)blocks), dim3(128), 0, st, a, c1, c2)) != cudaSuccess) return e;
    if (l.sorted) {
        const size_t fixed = (size_t)4 * G1 * G1 * sizeof(int32_t), table = (size_t)grid * grid * sizeof(uint32_t);
        const int hw = (int)std::min<size_t>(kSortedWarps, (kGmsSmemBudget - fixed) / table);
        e = launch_pdl(gms_sorted_kernel, dim3((unsigned)(4 * npairs)), dim3(kSortedThreads), fixed + hw * table, st, a, hw,
                       (const uint32_t *)c1, (const uint16_t *)c2, reinterpret_cast<uint16_t *>(b + l.ds), dec);
        if (e != cudaSuccess) return e;
    } else {
        const GmsRuns r(grid);
        // the grid's z extent is limited to 65,535: 16,383 pairs a launch
        for (int p0 = 0; p0 < npairs; p0 += 16383) {
            GmsArgs part = a;
            part.pairs += p0;
            const int np = std::min(npairs - p0, 16383);
            e = launch_pdl(gms_cells_kernel, dim3((unsigned)r.runs, (unsigned)G1, (unsigned)(4 * np)), dim3(kGmsThreads),
                           r.smem, st, part, r.span, (const uint32_t *)c1, (const uint16_t *)c2,
                           dec + (int64_t)p0 * 4 * G1 * G1);
            if (e != cudaSuccess) return e;
        }
    }
    return launch_pdl(gms_flag_kernel, dim3((unsigned)blocks), dim3(128), 0, st, a, (const uint32_t *)c1,
                      (const uint16_t *)c2, (const int32_t *)dec);
}

}  // namespace egm
