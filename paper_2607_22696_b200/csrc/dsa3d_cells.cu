// The general operator's backward on samples sorted by key cell: see dsa3d_cells.cuh.
//
//   cells_bin_kernel     sorts the samples of a query tile by key block; 18 bytes per sample
//   cells_sort_kernel    per block: its samples in the order of their cells
//   cells_dots_kernel    per block: samples by cell, 16 at a time  q . K_corner  and  dO . V_corner  (tensor cores), the
//                        trilinear value and derivatives of both per sample: eight numbers
//   cells_query_kernel   per query: alpha, delta, dS, dOffsets, the two coefficients per sample, dQ (a gather of K rows)
//   cells_sums_kernel    per block: samples by cell, 16 at a time their contributions to the eight corner rows of dK or dV
//                        (tensor cores), reduced into the fp32 accumulators
//   far_part             what falls beyond the bins (more than 12 positions from the query's tile), row by row, in
//                        CTAs of the last two block kernels
#include <cuda_bf16.h>

#include <type_traits>

#include "dsa3d_cells.cuh"
#include "dsa3d_kernels.h"

namespace dsa3d {
namespace {

using namespace cells;
using bf16 = __nv_bfloat16;

// ------------------------------------------------------------------------------------------------ binning
constexpr int kBinThreads = 512, kBinWarps = kBinThreads / 32, kCopies = 8;

// kKeep: the fractions wait in shared memory for the samples' places (windows up to kBinKeep samples: three CTAs per SM still);
// else the cells are worked out twice.  (Three CTAs against two: 403 -> 381 us for
// 566 K items, window (3,3,3); kept: 359.)
constexpr int kBinKeep = 36;
template <bool kKeep>
__device__ __forceinline__ void bin_block(const unsigned block, const float* __restrict__ offsets, const Problem& pr, const Slab& sl, unsigned inv_p,
                                          uint4* __restrict__ clear, long long clear_each, long long clear_all) {
    extern __shared__ __align__(16) unsigned char raw[];
    uint32_t* counters = reinterpret_cast<uint32_t*>(raw);                 // [kBins + 1][kCopies]: lanes of a warp mostly hit the same bin
    uint32_t* words = counters + (kBins + 1) * kCopies;                     // [kRows * P]: bin (9 bits), cell (6), rank in its counter (16)
    __shared__ uint32_t scan[kBinWarps];
    float* kept = kKeep ? reinterpret_cast<float*>(words + kRows * pr.P) : nullptr;     // [3][kRows * P]: the samples' fractions
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long tile = block;
    int r = static_cast<int>(tile % (sl.tiles_t * sl.tiles_y * sl.tiles_x));
    const int m = sl.m0 + static_cast<int>(tile / (sl.tiles_t * sl.tiles_y * sl.tiles_x));
    const int x0 = (r % sl.tiles_x) * kTileX; r /= sl.tiles_x;
    const int y0 = (r % sl.tiles_y) * 4, t0 = sl.f0 + (r / sl.tiles_y) * 4;
    const int samples = kRows * pr.P;
    if (block == 0 && tid == 0) { *sl.marked = 0; *sl.used = 0u; }
    // the block's part of the accumulators: stores in the shadow of a kernel that waits for its offsets
    const long long clear_to = min(clear_all, (block + 1ll) * clear_each);
    for (long long i = block * clear_each + tid; i < clear_to; i += kBinThreads) clear[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < (kBins + 1) * kCopies / 4; i += kBinThreads) reinterpret_cast<uint4*>(counters)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    auto row_of = [&](int s) { return static_cast<int>((static_cast<unsigned long long>(static_cast<unsigned>(s)) * inv_p) >> 24); };
    auto cell_of = [&](int s, int& n) -> Cell {
        const int row = row_of(s), p = s - row * pr.P;
        const int ty = row / kTileX, t = t0 + (ty >> 2), y = y0 + (ty & 3), x = x0 + row - ty * kTileX;
        n = (t * pr.H + y) * pr.W + x;
        if (t >= sl.f1 || y >= pr.H || x >= pr.W) { Cell c; c.it = c.iy = c.ix = 0; c.mask = 0u; c.ft = c.fy = c.fx = 0.0f; return c; }
        return make_cell(pr, t, y, x, p, offsets + ((static_cast<long long>(n) * pr.heads + m) * pr.P + p) * 3);
    };
    for (int base = 0; base < samples; base += 3 * kBinThreads) {
        uint32_t w[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {                  // three samples per thread at a time: their offsets load together
            const int s = base + i * kBinThreads + tid;
            w[i] = 0xffffffffu;
            if (s >= samples) continue;
            int n;
            const Cell c = cell_of(s, n);
            if (c.mask == 0u) continue;
            if constexpr (kKeep) { kept[s] = c.ft; kept[samples + s] = c.fy; kept[2 * samples + s] = c.fx; }
            const int rt = c.it - t0 + kReach, ry = c.iy - y0 + kReach, rx = c.ix - x0 + kReach;
            uint32_t bin = kBins, cell = 0u;
            if (static_cast<unsigned>(rt) < 4u * kBinsT && static_cast<unsigned>(ry) < 4u * kBinsY && static_cast<unsigned>(rx) < 3u * kBinsX) {
                const int bx = rx / kBlockX;
                bin = static_cast<uint32_t>(((rt >> 2) * kBinsY + (ry >> 2)) * kBinsX + bx);
                cell = static_cast<uint32_t>(((rt & 3) * 4 + (ry & 3)) * kBlockX + rx - bx * kBlockX);
            }
            w[i] = bin | (cell << 9);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int s = base + i * kBinThreads + tid;
            if (s >= samples) continue;
            if (w[i] != 0xffffffffu) w[i] |= atomicAdd(&counters[(w[i] & 511u) * kCopies + (lane & (kCopies - 1))], 1u) << 15;
            words[s] = w[i];
        }
    }
    __syncthreads();
    uint32_t c[kCopies], total = 0u;
    if (tid <= kBins) {
#pragma unroll
        for (int i = 0; i < kCopies; i += 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(&counters[tid * kCopies + i]);
            c[i] = v.x; c[i + 1] = v.y; c[i + 2] = v.z; c[i + 3] = v.w;
        }
#pragma unroll
        for (int i = 0; i < kCopies; ++i) total += c[i];
    }
    uint32_t incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane == 31) scan[warp] = incl;
    __syncthreads();
    uint32_t start = incl - total;
#pragma unroll
    for (int i = 0; i < kBinWarps; ++i) if (i < warp) start += scan[i];
    if (tid <= kBins) {
        sl.seg[tile * (kBins + 1) + tid] = start | (total << 16);
#pragma unroll
        for (int i = 0; i < kCopies; ++i) {
            const uint32_t n = c[i];
            c[i] = start;
            start += n;
        }
#pragma unroll
        for (int i = 0; i < kCopies; i += 4) *reinterpret_cast<uint4*>(&counters[tid * kCopies + i]) = make_uint4(c[i], c[i + 1], c[i + 2], c[i + 3]);
    }
    __syncthreads();
    uint4* geo = sl.geo + tile * samples;
    uint16_t* meta = sl.meta + tile * samples;
    for (int s = tid; s < samples; s += kBinThreads) {
        const uint32_t w = words[s];
        if (w == 0xffffffffu) continue;
        int n;
        float ft, fy, fx;
        if constexpr (kKeep) {
            const int row = row_of(s), ty = row / kTileX;
            n = ((t0 + (ty >> 2)) * pr.H + y0 + (ty & 3)) * pr.W + x0 + row - ty * kTileX;
            ft = kept[s]; fy = kept[samples + s]; fx = kept[2 * samples + s];
        } else {
            const Cell cl = cell_of(s, n);             // once more from the offsets, in L1 or L2 by now
            ft = cl.ft; fy = cl.fy; fx = cl.fx;
        }
        const uint32_t at = counters[(w & 511u) * kCopies + (lane & (kCopies - 1))] + (w >> 15);
        geo[at] = make_uint4(static_cast<uint32_t>(n), __float_as_uint(ft), __float_as_uint(fy), __float_as_uint(fx));
        meta[at] = static_cast<uint16_t>(static_cast<uint32_t>(s - row_of(s) * pr.P) | (((w >> 9) & 63u) << 8));
    }
}

template <bool kGated, bool kKeep>
__global__ void __launch_bounds__(kBinThreads, 3)
cells_bin_kernel(const float* __restrict__ offsets, const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned inv_p, unsigned blocks,
                 uint4* __restrict__ clear, long long clear_each, long long clear_all) {
    if constexpr (!kGated) {
        bin_block<kKeep>(blockIdx.x, offsets, pr, sl, inv_p, clear, clear_each, clear_all);
    } else {
        if (gated_off_early(pr.gate)) return;
        for (unsigned block = blockIdx.x; block < blocks; block += gridDim.x) {
            bin_block<kKeep>(block, offsets, pr, sl, inv_p, clear, clear_each, clear_all);
            __syncthreads();
        }
    }
}


// ------------------------------------------------------------------------------------------------ a block's samples
struct BlockPos { int m, t, y, x, bt, by, bx; };   // head, first cell along t, y, x; block numbers (bt from the slab's first frame)

__device__ __forceinline__ BlockPos block_pos(const Slab& sl, long long id) {
    BlockPos b;
    b.bx = static_cast<int>(id % sl.blocks_x) - 1; id /= sl.blocks_x;
    b.by = static_cast<int>(id % sl.blocks_y) - 1; id /= sl.blocks_y;
    b.bt = static_cast<int>(id % sl.blocks_t) + sl.bt0;
    b.m = sl.m0 + static_cast<int>(id / sl.blocks_t);
    b.t = sl.f0 + 4 * b.bt;
    b.y = 4 * b.by;
    b.x = kBlockX * b.bx;
    return b;
}

struct Segments {
    uint32_t first[kSegs + 1];                      // samples before the segment
    uint32_t start[kSegs];                          // its place in its tile's list
    int tile[kSegs];
    uint32_t scan[8];
};

// Finds the segments of a block (at least 256 threads, all of the CTA); returns how many samples they hold.
__device__ __forceinline__ uint32_t find_segments(const Slab& sl, const BlockPos& b, Segments& sg) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t count = 0u, start = 0u;
    int tile = 0;
    if (tid < kSegs) {
        const int bt = tid / (kBinsY * kSegsX), by = (tid / kSegsX) % kBinsY;
        const int bx = (b.bx & 1) + 2 * (tid % kSegsX);             // kReach is an even number of blocks: same parity as b.bx
        const int tt = b.bt + kReach / 4 - bt, ty = b.by + kReach / 4 - by, dx = b.bx + kReach / kBlockX - bx, tx = dx / 2;
        if (static_cast<unsigned>(tt) < static_cast<unsigned>(sl.tiles_t) && static_cast<unsigned>(ty) < static_cast<unsigned>(sl.tiles_y) &&
            dx >= 0 && tx < sl.tiles_x) {
            tile = (((b.m - sl.m0) * sl.tiles_t + tt) * sl.tiles_y + ty) * sl.tiles_x + tx;
            const uint32_t w = __ldg(sl.seg + static_cast<long long>(tile) * (kBins + 1) + (bt * kBinsY + by) * kBinsX + bx);
            start = w & 0xffffu;
            count = w >> 16;
        }
    }
    uint32_t incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += up;
    }
    if (warp < 8 && lane == 31) sg.scan[warp] = incl;
    __syncthreads();
    uint32_t before = 0u, total = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t v = sg.scan[i];
        if (i < warp) before += v;
        total += v;
    }
    if (tid < kSegs) {
        sg.first[tid] = before + incl - count;
        sg.start[tid] = start;
        sg.tile[tid] = tile;
        if (tid == kSegs - 1) sg.first[kSegs] = total;
    }
    __syncthreads();
    return total;
}

// Index, in the slab's sample lists, of the block's i-th sample.
__device__ __forceinline__ long long sample_of(const Segments& sg, uint32_t i, int samples_per_tile) {
    int lo = 0, hi = kSegs;                         // first[lo] <= i < first[hi]
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int mid = (lo + hi) >> 1;
        if (sg.first[mid] <= i) lo = mid; else hi = mid;
    }
    return static_cast<long long>(sg.tile[lo]) * samples_per_tile + sg.start[lo] + (i - sg.first[lo]);
}

// A block's samples in the order of their cells.  (A kernel of its own: it is a chain of dependent loads - segment,
// sample, place - which wants many small CTAs per SM, and both block kernels read what it leaves in one stream.)
constexpr int kSortThreads = 256, kSortKeep = 2048;
__device__ __forceinline__ void sort_block(const unsigned block, const Problem& pr, const Slab& sl) {
    __shared__ Segments sg;
    __shared__ uint32_t count[kCells], cursor[kCells], base;
    __shared__ uint32_t kept[kSortKeep];                    // place in its tile's list of the first samples
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const BlockPos b = block_pos(sl, block);
    if (tid < kCells) count[tid] = 0u;
    const uint32_t total = find_segments(sl, b, sg);
    uint32_t* first = sl.first + static_cast<long long>(block) * (kCells + 1);
    if (total == 0u) {
        if (tid <= kCells) first[tid] = 0u;
        return;
    }
    for (uint32_t i = tid; i < total; i += kSortThreads) {
        const uint32_t at = static_cast<uint32_t>(sample_of(sg, i, kRows * pr.P));
        if (i < kSortKeep) kept[i] = at;
        atomicAdd(&count[__ldg(sl.meta + at) >> 8], 1u);
    }
    if (tid == 0) base = atomicAdd(sl.used, total);
    __syncthreads();
    if (warp == 0) {
        const uint32_t c0 = lane < kCells / 2 ? count[2 * lane] : 0u, c1 = lane < kCells / 2 ? count[2 * lane + 1] : 0u;
        uint32_t inc = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(kFullMask, inc, o);
            if (lane >= o) inc += up;
        }
        if (lane < kCells / 2) {
            cursor[2 * lane] = first[2 * lane] = base + inc - c0 - c1;
            cursor[2 * lane + 1] = first[2 * lane + 1] = base + inc - c1;
        }
        if (lane == 31) first[kCells] = base + inc;
    }
    __syncthreads();
    for (uint32_t i = tid; i < total; i += kSortThreads) {
        const uint32_t at = i < kSortKeep ? kept[i] : static_cast<uint32_t>(sample_of(sg, i, kRows * pr.P));
        const uint32_t mt = __ldg(sl.meta + at);
        const uint4 u = __ldg(sl.geo + at);
        const uint32_t to = atomicAdd(&cursor[mt >> 8], 1u);
        sl.sorted[to] = make_float4(__uint_as_float(u.y), __uint_as_float(u.z), __uint_as_float(u.w), __uint_as_float(u.x));
        sl.place[to] = static_cast<uint32_t>(sample_at(sl, pr, b.m, static_cast<int>(u.x), static_cast<int>(mt & 255u)));
    }
}

template <bool kGated>
__global__ void __launch_bounds__(kSortThreads)
cells_sort_kernel(const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned blocks) {
    if constexpr (!kGated) {
        sort_block(blockIdx.x, pr, sl);
    } else {
        if (gated_off_early(pr.gate)) return;
        for (unsigned block = blockIdx.x; block < blocks; block += gridDim.x) {
            sort_block(block, pr, sl);
            __syncthreads();
        }
    }
}


// Byte of 16-byte chunk `chunk` of box row `row` in shared memory: rows of 128 bytes and more have their chunks permuted by
// the row's parity, so that the four even (or odd) chunks a quarter-warp reads of two neighbouring rows lie in different banks.
template <int D> __device__ __forceinline__ int box_byte(int row, int chunk) {
    return row * (D * 2) + ((D >= 64 ? (chunk ^ (row & 1)) : chunk) << 4);
}

// The rows of a block's box of one tensor into shared memory, zeros outside the grid.
template <int D, int NT>
__device__ __forceinline__ void load_box(unsigned char* dst, const bf16* __restrict__ src, const BlockPos& b, const Problem& pr) {
    constexpr int CH = D / 8;
    for (int i = threadIdx.x; i < kBox * CH; i += NT) {
        const int row = i / CH, chunk = i - row * CH;
        const int t = b.t + row / 20, y = b.y + (row / 4) % 5, x = b.x + row % 4;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (static_cast<unsigned>(t) < static_cast<unsigned>(pr.T) && static_cast<unsigned>(y) < static_cast<unsigned>(pr.H) && static_cast<unsigned>(x) < static_cast<unsigned>(pr.W))
            v = __ldg(reinterpret_cast<const uint4*>(src + (((static_cast<long long>(t) * pr.H + y) * pr.W + x) * pr.heads + b.m) * D) + chunk);
        *reinterpret_cast<uint4*>(dst + box_byte<D>(row, chunk)) = v;
    }
}

// ------------------------------------------------------------------------------------------------ beyond the bins
// The samples in bin kBins of every tile, a warp per sample, row by row: part `part` of `parts` (a CTA each).
// kScatter: their contributions to dK and dV, and those of marked samples of the other bins; otherwise what the
// products of cells_dots_kernel leave for the others.  There are none in nearly every call: the work rides in CTAs
// behind those of the block kernels instead of two launches of its own.
template <typename T, int D, bool kScatter>
__device__ __noinline__ void far_part(const unsigned part, const unsigned parts, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                      const T* __restrict__ dout, const float* __restrict__ offsets, float* __restrict__ acc_dk, float* __restrict__ acc_dv,
                                      const Problem& pr, const Slab& sl) {
    const int tiles = sl.heads * sl.tiles_t * sl.tiles_y * sl.tiles_x;
    constexpr int V = D / 32;                       // channels per lane
    const int lane = threadIdx.x & 31, warp = static_cast<int>(threadIdx.x >> 5), warps = static_cast<int>(blockDim.x >> 5);
    const long long tok = static_cast<long long>(pr.heads) * D;
    const int per_head = sl.tiles_t * sl.tiles_y * sl.tiles_x;
    [[maybe_unused]] const long long kv_extent = pr.N * pr.heads * D;
    const bool marked = kScatter && *sl.marked != 0;
    // a lane per tile finds those with something to do; the warps of the CTA then share a tile's samples
    const int at_once = min(32, (tiles + static_cast<int>(parts) - 1) / static_cast<int>(parts));
    for (int base = static_cast<int>(part) * at_once; base < tiles; base += static_cast<int>(parts) * at_once) {
        uint32_t mine = 0u;
        if (lane < at_once && base + lane < tiles) mine = __ldg(sl.seg + static_cast<long long>(base + lane) * (kBins + 1) + kBins);
        if (marked) mine = ((mine & 0xffffu) + (mine >> 16)) << 16;        // all samples of the tile: those beyond the bins are its last
        unsigned todo = __ballot_sync(kFullMask, (mine >> 16) != 0u);
        while (todo) {
            const int src = __ffs(static_cast<int>(todo)) - 1;
            todo &= todo - 1u;
            const uint32_t w = __shfl_sync(kFullMask, mine, src);
            const long long tile = base + src;
            const int m = sl.m0 + static_cast<int>(tile / per_head);
            const uint32_t far_from = marked ? __ldg(sl.seg + tile * (kBins + 1) + kBins) & 0xffffu : 0u;
            const long long list = tile * (kRows * pr.P) + (w & 0xffffu);
            uint32_t next = static_cast<uint32_t>(warp) * 32u;
            unsigned some = 0u;
            while (true) {
                while (some == 0u && next < (w >> 16)) {   // 32 samples at a time: which of them are beyond the bins or marked
                    const uint32_t i = next + static_cast<uint32_t>(lane);
                    bool take = i < (w >> 16);
                    if (take && marked && i < far_from)
                        take = __float_as_uint(sl.coef[sample_at(sl, pr, m, static_cast<int>(__ldg(sl.geo + list + i).x), static_cast<int>(__ldg(sl.meta + list + i) & 255u))].y) >> 31;
                    some = __ballot_sync(kFullMask, take);
                    next += static_cast<uint32_t>(warps) * 32u;
                }
                if (some == 0u) break;
                const long long at = list + next - static_cast<uint32_t>(warps) * 32u + static_cast<uint32_t>(__ffs(static_cast<int>(some)) - 1);
                some &= some - 1u;
                const int n = static_cast<int>(__ldg(sl.geo + at).x), p = static_cast<int>(__ldg(sl.meta + at) & 255u);
                const int x = n % pr.W, y = (n / pr.W) % pr.H, t = n / (pr.W * pr.H);
                const long long row = static_cast<long long>(n) * pr.heads + m;
                const Sample smp = to_sample(pr, make_cell(pr, t, y, x, p, offsets + (row * pr.P + p) * 3));
                const long long o0 = static_cast<long long>(m) * D + smp.base * tok + lane * V;
                float qv[V], dv[V];
#pragma unroll
                for (int z = 0; z < V; ++z) {
                    qv[z] = static_cast<float>(q[row * D + lane * V + z]);
                    dv[z] = static_cast<float>(dout[row * D + lane * V + z]);
                }
                const float wt[2] = {1.0f - smp.ft, smp.ft}, wy[2] = {1.0f - smp.fy, smp.fy}, wx[2] = {1.0f - smp.fx, smp.fx};
                const long long sy = static_cast<long long>(pr.W) * tok, st = static_cast<long long>(pr.H) * sy;
                const long long sidx = sample_at(sl, pr, m, n, p);
                if constexpr (kScatter) {
                    const float2 cf = sl.coef[sidx];
                    for (int j = 0; j < 8; ++j) {
                        const float wj = wt[j >> 2] * wy[(j >> 1) & 1] * wx[j & 1];
                        const long long o = o0 + (j >> 2) * st + ((j >> 1) & 1) * sy + (j & 1) * tok;
                        if (!((smp.mask >> j) & 1u) || wj == 0.0f || !DSA3D_IN_RANGE(pr, o, kv_extent, 7)) continue;
#pragma unroll
                        for (int z = 0; z < V; ++z) {
                            atomicAdd(acc_dk + o + z, wj * cf.x * qv[z]);
                            atomicAdd(acc_dv + o + z, wj * fabsf(cf.y) * dv[z]);
                        }
                    }
                } else {
                    float a[8], bb[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int ct = j >> 2, cy = (j >> 1) & 1, cx = j & 1;
                        const bool needed = wt[ct] * wy[cy] * wx[cx] != 0.0f || wy[cy] * wx[cx] != 0.0f || wt[ct] * wx[cx] != 0.0f || wt[ct] * wy[cy] != 0.0f;
                        const long long o = o0 + ct * st + cy * sy + cx * tok;
                        a[j] = bb[j] = 0.0f;
                        if (!((smp.mask >> j) & 1u) || !needed || !DSA3D_IN_RANGE(pr, o, kv_extent, 5)) continue;
#pragma unroll
                        for (int z = 0; z < V; ++z) {
                            a[j] = fmaf(qv[z], static_cast<float>(k[o + z]), a[j]);
                            bb[j] = fmaf(dv[z], static_cast<float>(v[o + z]), bb[j]);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        a[j] = group_sum<32>(a[j], kFullMask);
                        bb[j] = group_sum<32>(bb[j], kFullMask);
                    }
                    float r[8];
                    trilerp_grad(a, smp.ft, smp.fy, smp.fx, r[0], r[1], r[2], r[3]);
                    trilerp_grad(bb, smp.ft, smp.fy, smp.fx, r[4], r[5], r[6], r[7]);
                    if (lane == 0) {
#pragma unroll
                        for (int z = 0; z < 8; ++z) sl.stats[sidx * 8 + z] = r[z];
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------ dot products
constexpr int kDotThreads = 256;

template <int D> struct DotSmem {
    unsigned char box[2][kBox * D * 2];
    uint32_t first[kCells + 1], groups[64];         // groups: of 16 samples, before the cell (the rest of the 64 never reached)
};

// Value and derivatives of the trilinear interpolant of eight corner numbers, two corners (2j, 2j + 1: x pair of (ct, cy) =
// (j >> 1, j & 1)) on each of four lanes: lane j returns number j of (value, d/dt, d/dy, d/dx).  Corners whose
// weight and weight derivatives are all zero do not enter (they may hold anything).
__device__ __forceinline__ float trilerp_lanes(float s0, float s1, int j, float ft, float fy, float fx) {
    const float wt = (j & 2) ? ft : 1.0f - ft, wy = (j & 1) ? fy : 1.0f - fy;
    const bool at = wt != 0.0f, ay = wy != 0.0f, ax = fx != 0.0f;
    if (!(at || ay)) s0 = 0.0f;
    if (!((at && ay) || (ax && (at || ay)))) s1 = 0.0f;
    const float X = s1 - s0, L = fmaf(fx, X, s0), wty = wt * wy;
    const float v0 = wty * L, v1 = (j & 2) ? wy * L : -wy * L, v2 = (j & 1) ? wt * L : -wt * L, v3 = wty * X;
    const bool up = (j & 2) != 0;
    const float keep0 = up ? v2 : v0, keep1 = up ? v3 : v1, send0 = up ? v0 : v2, send1 = up ? v1 : v3;
    const float r0 = keep0 + __shfl_xor_sync(kFullMask, send0, 2), r1 = keep1 + __shfl_xor_sync(kFullMask, send1, 2);
    const bool odd = (j & 1) != 0;
    return (odd ? r1 : r0) + __shfl_xor_sync(kFullMask, odd ? r0 : r1, 1);
}

// 32 bytes of a row (16 where I = 1).  One 32-byte load where the tensor's alignment allows: a quarter-warp then reads whole 128-byte
// lines, while two 16-byte loads meet in the same banks (8 data-pipe cycles per 512 bytes against 4).
template <bool kWide, int I> __device__ __forceinline__ void load_piece(const uint4* p, uint4* r) {
    if constexpr (kWide && I > 1) {
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0].x), "=r"(r[0].y), "=r"(r[0].z), "=r"(r[0].w), "=r"(r[1].x), "=r"(r[1].y), "=r"(r[1].z), "=r"(r[1].w) : "l"(p));
    } else {
        r[0] = __ldg(p);
        if constexpr (I > 1) r[1] = __ldg(p + 1);
    }
}

// q . K and dO . V with derivatives, eight numbers per sample into stats; even warps take q . K, odd ones dO . V.
template <int D, bool kWide>
__device__ __forceinline__ void dots_block(const unsigned block, const bf16* __restrict__ q, const bf16* __restrict__ k, const bf16* __restrict__ v, const bf16* __restrict__ dout,
                  const Problem& pr, const Slab& sl) {
    constexpr int I = D / 32, W = kDotThreads / 64;
    extern __shared__ __align__(16) unsigned char raw[];
    DotSmem<D>& s = *reinterpret_cast<DotSmem<D>*>(raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g8 = lane >> 2, j = lane & 3;
    const int tensor = warp & 1;
    const uint32_t* first = sl.first + static_cast<long long>(block) * (kCells + 1);
    if (__ldg(first) == __ldg(first + kCells)) return;
    const BlockPos b = block_pos(sl, block);
    if (warp == 0) {
        const uint32_t f0 = __ldg(first + min(2 * lane, kCells)), f1 = __ldg(first + min(2 * lane + 1, kCells)), f2 = __ldg(first + min(2 * lane + 2, kCells));
        const uint32_t n0 = (f1 - f0 + 15u) >> 4, n1 = (f2 - f1 + 15u) >> 4;
        uint32_t inc = n0 + n1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(kFullMask, inc, o);
            if (lane >= o) inc += up;
        }
        if (lane <= kCells / 2) s.first[2 * lane] = f0;
        if (lane < kCells / 2) s.first[2 * lane + 1] = f1;
        s.groups[2 * lane] = inc - n0 - n1;
        s.groups[2 * lane + 1] = inc - n1;
    }
    load_box<D, kDotThreads>(s.box[0], k, b, pr);
    load_box<D, kDotThreads>(s.box[1], v, b, pr);
    __syncthreads();
    const bf16* src = (tensor ? dout : q) + static_cast<long long>(b.m) * D + j * (I > 1 ? 16 : 8);
    const unsigned char* box = s.box[tensor];
    const long long tok = static_cast<long long>(pr.heads) * D;
    const int groups = static_cast<int>(s.groups[kCells]);
    float* out = sl.stats + tensor * 4 + j;
    // what the lane needs of a group: its cell, its samples (rows g8 and g8 + 8 of the tile)
    int cell = 0;
    bool live_a = false, live_b = false;
    float4 ga = make_float4(0.0f, 0.0f, 0.0f, 0.0f), gb = ga;
    uint32_t pa = 0u, pb = 0u;
    auto fetch = [&](int g) {
        const uint32_t ug = static_cast<uint32_t>(g);
        // cells 1 .. 47 whose groups begin at or before this one
        cell = __popc(__ballot_sync(kFullMask, s.groups[lane + 1] <= ug)) + __popc(__ballot_sync(kFullMask, lane < kCells - 33 && s.groups[min(lane + 33, 63)] <= ug));
        const uint32_t f = s.first[cell] + 16u * (ug - s.groups[cell]), end = s.first[cell + 1];
        const uint32_t ia = min(f + static_cast<uint32_t>(g8), end - 1u), ib = min(f + static_cast<uint32_t>(g8) + 8u, end - 1u);   // a missing sample repeats the last one
        live_a = f + static_cast<uint32_t>(g8) < end;
        live_b = f + static_cast<uint32_t>(g8) + 8u < end;
        ga = __ldg(sl.sorted + ia);
        gb = __ldg(sl.sorted + ib);
        pa = __ldg(sl.place + ia);
        pb = __ldg(sl.place + ib);
    };
    int g = warp >> 1;
    if (g < groups) fetch(g);
    for (; g < groups; g += W) {
        const int row = box_row(cell) + box_step(g8);
        const uint4* ra_p = reinterpret_cast<const uint4*>(src + __float_as_int(ga.w) * tok);
        const uint4* rb_p = reinterpret_cast<const uint4*>(src + __float_as_int(gb.w) * tok);
        // The order of the channels inside a product is free: lane j takes bytes 32 j .. of every 128 (chunk j of
        // the 64 of a 32-channel row), whole pieces on both sides.
        uint4 ra[I], rb[I];
#pragma unroll
        for (int i = 0; i < I; i += 2) {
            load_piece<kWide, I>(ra_p + (I > 1 ? 4 * i : 0), ra + i);
            load_piece<kWide, I>(rb_p + (I > 1 ? 4 * i : 0), rb + i);
        }
        const float fa0 = ga.x, fa1 = ga.y, fa2 = ga.z, fb0 = gb.x, fb1 = gb.y, fb2 = gb.z;
        float* da = live_a ? out + static_cast<size_t>(pa) * 8 : nullptr;
        float* db = live_b ? out + static_cast<size_t>(pb) * 8 : nullptr;
        if (g + W < groups) fetch(g + W);           // the next group's samples, a group ahead of its rows
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const uint4 kb = *reinterpret_cast<const uint4*>(box + box_byte<D>(row, I > 1 ? (i >> 1) * 8 + 2 * j + (i & 1) : j));
            mma_bf16(c, ra[i].x, rb[i].x, ra[i].y, rb[i].y, kb.x, kb.y);
            mma_bf16(c, ra[i].z, rb[i].z, ra[i].w, rb[i].w, kb.z, kb.w);
        }
        const float xa = trilerp_lanes(c[0], c[1], j, fa0, fa1, fa2), xb = trilerp_lanes(c[2], c[3], j, fb0, fb1, fb2);
        if (da) *da = xa;
        if (db) *db = xb;
    }
}

template <int D, bool kWide, bool kGated>
__global__ void __launch_bounds__(kDotThreads, D == 128 ? 3 : 4)
cells_dots_kernel(const bf16* __restrict__ q, const bf16* __restrict__ k, const bf16* __restrict__ v, const bf16* __restrict__ dout,
                  const float* __restrict__ offsets, const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned blocks) {
    if constexpr (!kGated) {
        if (blockIdx.x < blocks) dots_block<D, kWide>(blockIdx.x, q, k, v, dout, pr, sl);
        else far_part<bf16, D, false>(blockIdx.x - blocks, gridDim.x - blocks, q, k, v, dout, offsets, nullptr, nullptr, pr, sl);
    } else {
        if (gated_off_early(pr.gate)) return;
        for (unsigned block = blockIdx.x; block < blocks; block += gridDim.x) {
            dots_block<D, kWide>(block, q, k, v, dout, pr, sl);
            __syncthreads();
        }
        far_part<bf16, D, false>(blockIdx.x, gridDim.x, q, k, v, dout, offsets, nullptr, nullptr, pr, sl);
    }
}


// ------------------------------------------------------------------------------------------------ per query
constexpr int kQueryWarps = 2;

// alpha from the saved lse, delta, dS, dOffsets, the two coefficients per sample (ck = scale dS, cv = alpha), and
// dQ = sum_p ck_p sum_c w_c K_c: a warp per (query, head), 32 samples at a time, a sample per lane; the K rows are summed as
// in the forward (dsa3d_gather.cuh).  A sample with anything that is not finite (its rows of q, dO, K or V, or its
// coefficients) is marked by the sign of cv: its contributions to dK and dV are formed one by one, so that they reach only
// the corners with a weight.  Windows of at most 8 (16) samples: G = 4 (2) neighbouring queries share a warp.
// Bound by the data pipe (81 %) and the issue slots (71 %), for more samples by the latency of the row loads (59 % of both): what an item
// does before its first row counts, and what it holds.  The statistics are asked for beside the offsets (backward 0.5 - 2.4 % faster), and
// windows of at most 32 samples have an instance of one round (kOne), which keeps nothing for a next one (this kernel 0.52 -> 0.40 ms on
// 141,440 items of 128 channels, 0.35 -> 0.24 of 64, where 21 CTAs fit an SM then).  Backward, window (3,3,3), 16 x 68 x 120, 16 heads: 128 channels
// 21.9 -> 20.0 ms, 64 channels 15.1 -> 13.4; (2,2,2), integer offsets, 16 x 45 x 80: 4.00 -> 3.92 ms; (3,7,7) 16.8 -> 16.3 ms (8 x 68 x 120,
// 6 heads).  (Rows of the next batch ahead of the sums, or the first rows ahead of the statistics: with one round 2 % slower, for registers.)
template <typename T, int D, int G, bool kOne>
__device__ __forceinline__ void query_block(const unsigned block, const T* __restrict__ k, const float* __restrict__ offsets, const float* __restrict__ lse, T* __restrict__ dq,
                   float* __restrict__ doffsets, const Problem& pr, const Slab& sl, unsigned blocks_per_head) {
    __shared__ GatherList lists[kQueryWarps];
    constexpr int L = 32 / G;                       // lanes per query
    constexpr int CH = GatherStep<D, T>::CH, U = GatherStep<D, T>::U, PER = U > G ? U / G : 1, ITEMS = G > U ? G / U : 1;      // subgroups per query, queries per subgroup
    constexpr int step = G == 1 ? GatherStep<D, T>::N : 4 * PER;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gl_lane = lane & (L - 1);
    GatherList& gl = lists[warp];
    const int frame = pr.H * pr.W, mh = static_cast<int>(block / blocks_per_head), per_head = frame * (sl.f1 - sl.f0);
    const int warp_first = (static_cast<int>(block - static_cast<unsigned>(mh) * blocks_per_head) * kQueryWarps + warp) * G;
    if (warp_first >= per_head) return;
    const bool active = warp_first + lane / L < per_head;        // a query past the end repeats the last one, stores off
    const int local = active ? warp_first + lane / L : per_head - 1;
    const int m = sl.m0 + mh, n = frame * sl.f0 + local;
    const int x = n % pr.W, ty = n / pr.W, y = ty % pr.H, t = ty / pr.H;
    const long long row = static_cast<long long>(n) * pr.heads + m, item = static_cast<long long>(mh) * per_head + local;
    const float scale = rsqrtf(static_cast<float>(D)), lse2 = __ldg(lse + row) * kLog2e;
    const float* off_row = offsets + row * pr.P * 3;
    const float* st_row = sl.stats + item * pr.P * 8;
    const uint32_t tok_bytes = static_cast<uint32_t>(pr.heads) * (D * static_cast<int>(sizeof(T)));
    const T* kh = k + static_cast<long long>(m) * D;
    auto sample = [&](int p, Sample& s, float4& a, float4& b) {
        s.base = 0; s.mask = 0u; s.ft = s.fy = s.fx = 0.0f;
        a = b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (p >= pr.P) return;
        // asked for beside the offsets, not behind them; what stands there for a dead sample is not used (it has g = 0)
        a = __ldg(reinterpret_cast<const float4*>(st_row + p * 8));
        b = __ldg(reinterpret_cast<const float4*>(st_row + p * 8) + 1);
        s = to_sample(pr, make_cell(pr, t, y, x, p, off_row + p * 3));
    };
    auto weight = [&](float sv) { return exp2f(fmaf(sv, scale * kLog2e, -lse2)); };
    Sample s;
    float4 a, b;
    sample(gl_lane, s, a, b);
    float delta = s.mask ? weight(a.x) * b.x : 0.0f;
    for (int p = gl_lane + L; !kOne && p < pr.P; p += L) {
        Sample s2;
        float4 a2, b2;
        sample(p, s2, a2, b2);
        if (s2.mask) delta = fmaf(weight(a2.x), b2.x, delta);
    }
    delta = group_sum<L>(delta, kFullMask);
    float acc[CH];
#pragma unroll
    for (int e = 0; e < CH; ++e) acc[e] = 0.0f;
    for (int pb = 0; kOne ? pb == 0 : pb < pr.P; pb += L) {
        const int p = pb + gl_lane;
        if (!kOne && pb > 0) sample(p, s, a, b);
        float ck = 0.0f, d0 = 0.0f, d1 = 0.0f, d2 = 0.0f;
        if (s.mask != 0u) {
            const float alpha = weight(a.x);
            ck = scale * (alpha * (b.x - delta));
            d0 = fmaf(ck, a.y, alpha * b.y);
            d1 = fmaf(ck, a.z, alpha * b.z);
            d2 = fmaf(ck, a.w, alpha * b.w);
            const bool odd = !(fabsf(a.x) < INFINITY) || !(fabsf(b.x) < INFINITY) || !(fabsf(ck) < INFINITY) || !(alpha < INFINITY);
            if (odd) *sl.marked = 1;
            if (active) sl.coef[item * pr.P + p] = make_float2(ck, __uint_as_float(__float_as_uint(alpha) | (odd ? 0x80000000u : 0u)));
        }
        if (active && p < pr.P) {
            float* d = doffsets + (row * pr.P + p) * 3;
            d[0] = d0; d[1] = d1; d[2] = d2;
        }
        const GatherPart part = gather_list<G>(gl, checked_corners(pr, weighted_corners(s.mask, s.ft, s.fy, s.fx), s.base, 4), s.base, pr, step);
        const float wt[2] = {1.0f - s.ft, s.ft}, wy[2] = {1.0f - s.fy, s.fy}, wx[2] = {1.0f - s.fx, s.fx};
        float w[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) w[c] = wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1];
        gather_weights<G>(gl, part, ck, w, step);
        __syncwarp();
        if constexpr (G == 1) {
            gather_sum<D, T>(gl, part.total, kh, tok_bytes, acc);
        } else {
            constexpr int LPR = GatherStep<D, T>::LPR;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int u = lane / LPR, it = PER > 1 ? u / PER : u * ITEMS + i;
                const int total = __shfl_sync(kFullMask, part.total, it * L);
#pragma unroll
                for (int e = 0; e < CH; ++e) acc[e] = 0.0f;
                gather_sum_item<D, PER, T>(gl, it * (kGatherRows / G), total, PER > 1 ? u % PER : 0, kh, tok_bytes, acc);
                __syncwarp();
#pragma unroll
                for (int o = LPR; o < LPR * PER; o <<= 1)
#pragma unroll
                    for (int e = 0; e < CH; ++e) acc[e] += __shfl_xor_sync(kFullMask, acc[e], o);
                if (warp_first + it < per_head && (PER == 1 || u % PER == 0))
                    Elt<T, 1>::store(dq + (static_cast<long long>(frame * sl.f0 + warp_first + it) * pr.heads + m) * D + (lane % LPR) * CH, acc);
            }
        }
        __syncwarp();
    }
    if constexpr (G == 1) {
        gather_finish<D>(acc);
        if (lane < D / CH) Elt<T, 1>::store(dq + row * D + lane * CH, acc);
    }
}

template <typename T, int D, int G, bool kOne, bool kGated>
__global__ void __launch_bounds__(kQueryWarps * 32, 16)
cells_query_kernel(const T* __restrict__ k, const float* __restrict__ offsets, const float* __restrict__ lse, T* __restrict__ dq,
                   float* __restrict__ doffsets, const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned blocks_per_head, unsigned blocks) {
    if constexpr (!kGated) {
        query_block<T, D, G, kOne>(blockIdx.x, k, offsets, lse, dq, doffsets, pr, sl, blocks_per_head);
    } else {
        if (gated_off_early(pr.gate)) return;
        for (unsigned block = blockIdx.x; block < blocks; block += gridDim.x) {
            query_block<T, D, G, kOne>(block, k, offsets, lse, dq, doffsets, pr, sl, blocks_per_head);
            __syncthreads();
        }
    }
}


// ------------------------------------------------------------------------------------------------ dK, dV
constexpr int kSumThreads = 256;

template <int D> struct SumSmem {
    static constexpr int STAGES = 2, GROUP = 16 * D * 2;
    unsigned char stage[kSumThreads / 32][STAGES][GROUP];         // a warp's ring of 16 query rows
    float4 geo[kSumThreads / 32][2][16];                          // ft, fy, fx, coefficient of a group's samples
    uint32_t first[kCells + 1];
};

__device__ __forceinline__ void red_add_v2(float* addr, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(addr), "f"(a), "f"(b) : "memory");
}

// A warp works on one tensor and runs of three cells along x: the corners of a run are 4 columns x 4 (t, y) rows of the
// accumulators, the 16 rows of the product tile, and 16 of the run's samples at a time are its depth.  A lane forms
// the weights of its (t, y) in columns g8 / 4 and g8 / 4 + 2: a sample has a weight in exactly one of the two, which goes in
// as three bf16 numbers whose sum is the fp32 weight, three products into the same sums.  (With two, 2^-17 of the weights was
// lost: where contributions cancel that shows, elsewhere the seventh digit of an error of 1.6558e-3, the outputs' rounding.
// The third costs the backward 0.7 - 2.4 %: 57.4 -> 58.5 ms for 5.5 M items of 128 channels, 29.2 -> 29.4 for 4.2 M of 64, window
// (3,3,3).)  Nothing is shared between warps: each walks through its
// groups in three steps that overlap - samples (two groups ahead), coefficients and query rows (one ahead), products.
template <int D>
__device__ __forceinline__ void sums_block(const unsigned block, const bf16* __restrict__ q, const bf16* __restrict__ dout, float* __restrict__ acc_dk, float* __restrict__ acc_dv,
                  const Problem& pr, const Slab& sl) {
    using S = SumSmem<D>;
    constexpr int STRIDE = 4;                       // the four warps of a tensor take the runs in turn
    constexpr int CPR = D / 8;                      // 16-byte chunks of a staged row, permuted by the row (SWZ)
    constexpr int LD = 16 * CPR / 32, RPI = 32 / CPR;      // fetches per lane for 16 rows; rows per fetch of the warp
    constexpr int SWZ = CPR < 8 ? CPR - 1 : 7;
    extern __shared__ __align__(16) unsigned char raw[];
    S& s = *reinterpret_cast<S*>((reinterpret_cast<uintptr_t>(raw) + 255) & ~uintptr_t(255));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g8 = lane >> 2, j = lane & 3;
    const uint32_t* first = sl.first + static_cast<long long>(block) * (kCells + 1);
    if (__ldg(first) == __ldg(first + kCells)) return;
    const BlockPos b = block_pos(sl, block);
    if (tid <= kCells) s.first[tid] = __ldg(first + tid);
    __syncthreads();
    const long long tok = static_cast<long long>(pr.heads) * D;
    const uint32_t tok_bytes = static_cast<uint32_t>(tok) * 2u;
    [[maybe_unused]] const long long kv_extent = pr.N * pr.heads * D;
    const int tensor = warp & 1, run0 = warp >> 1;
    const char* src = reinterpret_cast<const char*>((tensor ? dout : q) + static_cast<long long>(b.m) * D + (lane % CPR) * 8);
    float* acc = (tensor ? acc_dv : acc_dk) + static_cast<long long>(b.m) * D + 2 * j;
    const float* coef = reinterpret_cast<const float*>(sl.coef) + tensor;
    const float st = (g8 & 2) ? 1.0f : -1.0f, ot = (g8 & 2) ? 0.0f : 1.0f, sy = (g8 & 1) ? 1.0f : -1.0f, oy = (g8 & 1) ? 0.0f : 1.0f;
    const int col = g8 >> 2;
    const uint32_t stage0 = static_cast<uint32_t>(__cvta_generic_to_shared(s.stage[warp][0]));
    // where the lane's chunk of row i * RPI + lane / CPR goes, and where its row pointer of an ldmatrix points: the
    // chunk's permutation is an exclusive or within 256 aligned bytes
    const uint32_t put = static_cast<uint32_t>((lane / CPR) * (D * 2) + (((lane % CPR) ^ ((lane / CPR) & SWZ)) << 4));
    const uint32_t get = static_cast<uint32_t>((lane & 15) * (D * 2) + (((lane >> 4) ^ (lane & SWZ)) << 4));

    // step 1: a group's samples, lane l sample l % 16 (beyond the run its last one again)
    int run1 = run0 - STRIDE;
    uint32_t f1 = 0u, stop1 = 0u;
    float4 geo1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    uint32_t place1 = 0u;
    bool any1 = false;
    auto samples = [&]() {                          // the group at f1, or the next run's first
        while (f1 >= stop1 && run1 < kRuns - STRIDE) {
            run1 += STRIDE;
            f1 = s.first[kBlockX * run1];
            stop1 = s.first[kBlockX * run1 + kBlockX];
        }
        any1 = f1 < stop1;
        if (any1) {
            const uint32_t i = min(f1 + static_cast<uint32_t>(lane & 15), stop1 - 1u);
            geo1 = __ldg(sl.sorted + i);
            place1 = __ldg(sl.place + i);
        }
    };
    // step 2: their coefficients and query rows
    int run2 = 0;
    uint32_t f2 = 0u, stop2 = 0u;
    float4 geo2 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float coef2 = 0.0f, mark2 = 0.0f;
    bool any2 = false;
    uint32_t stage2 = stage0;
    auto rows = [&]() {
        any2 = any1;
        if (any1) {
            run2 = run1; f2 = f1; stop2 = stop1; geo2 = geo1;
            coef2 = __ldg(coef + static_cast<size_t>(place1) * 2);
            mark2 = tensor ? coef2 : __ldg(coef + static_cast<size_t>(place1) * 2 + 1);
            const uint32_t token = __float_as_uint(geo1.w);
#pragma unroll
            for (int i = 0; i < LD; ++i) {
                const uint32_t t = __shfl_sync(kFullMask, token, i * RPI + lane / CPR);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             ::"r"(stage2 + ((put ^ (((i * RPI) & SWZ) << 4)) + i * RPI * (D * 2))), "l"(src + static_cast<uint64_t>(t) * tok_bytes) : "memory");
            }
            stage2 = stage2 == stage0 + (S::STAGES - 1) * S::GROUP ? stage0 : stage2 + S::GROUP;
            f1 += 16u;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    samples();
    rows();
    samples();
    uint32_t stage3 = stage0;
    int slot = 0;
    uint32_t used_a = 0u, used_b = 0u;                 // weights the lane has put into its two rows of the run
    float c[D / 8][4];
#pragma unroll
    for (int i = 0; i < D / 8; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0.0f;
#pragma unroll 1
    while (any2) {
        // step 3: the products of the group whose rows are on their way
        const int run = run2;
        const uint32_t f = f2, stop = stop2, from1 = s.first[kBlockX * run + 1], from2 = s.first[kBlockX * run + 2];
        const bool odd = __float_as_uint(mark2) >> 31;             // marked: far_part takes it
        const unsigned odds = __ballot_sync(kFullMask, odd);
        if (lane < 16) s.geo[warp][slot][lane] = make_float4(geo2.x, geo2.y, geo2.z, (odd || f + lane >= stop) ? 0.0f : coef2);
        const uint32_t from = stage3;
        stage3 = stage3 == stage0 + (S::STAGES - 1) * S::GROUP ? stage0 : stage3 + S::GROUP;
        __syncwarp();                                  // also: everybody has read the slot that the next rows go to
        rows();
        samples();
        // weights for samples 2j, 2j + 1, 2j + 8, 2j + 9; `mine`: those that belong to column `col`, the others to col + 2
        uint32_t head[2], rest[2], last[2], mine[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float w2[2];
            mine[h] = 0u;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int i = 2 * j + e + 8 * h;
                const float4 ge = s.geo[warp][slot][i];
                const uint32_t k = f + static_cast<uint32_t>(i);
                const int d = col - (k >= from1 ? 1 : 0) - (k >= from2 ? 1 : 0);     // column - cell: -2, 0 left, -1, 1 right
                w2[e] = fmaf(ge.x, st, ot) * fmaf(ge.y, sy, oy) * ((d & 1) ? ge.z : 1.0f - ge.z) * ge.w;
                if (d >= 0) mine[h] |= 0xffffu << (16 * e);
            }
            const __nv_bfloat162 hd = __floats2bfloat162_rn(w2[0], w2[1]);
            head[h] = *reinterpret_cast<const uint32_t*>(&hd);
            w2[0] -= __uint_as_float(head[h] << 16);
            w2[1] -= __uint_as_float(head[h] & 0xffff0000u);
            const __nv_bfloat162 rs = __floats2bfloat162_rn(w2[0], w2[1]);
            rest[h] = *reinterpret_cast<const uint32_t*>(&rs);
            const __nv_bfloat162 ls = __floats2bfloat162_rn(w2[0] - __uint_as_float(rest[h] << 16), w2[1] - __uint_as_float(rest[h] & 0xffff0000u));
            last[h] = *reinterpret_cast<const uint32_t*>(&ls);
        }
        slot ^= 1;
        used_a |= (head[0] & mine[0]) | (head[1] & mine[1]);
        used_b |= (head[0] & ~mine[0]) | (head[1] & ~mine[1]);
        const uint32_t a0 = head[0] & mine[0], a1 = head[0] & ~mine[0], a2 = head[1] & mine[1], a3 = head[1] & ~mine[1];
        const uint32_t r0 = rest[0] & mine[0], r1 = rest[0] & ~mine[0], r2 = rest[1] & mine[1], r3 = rest[1] & ~mine[1];
        const uint32_t l0 = last[0] & mine[0], l1 = last[0] & ~mine[0], l2 = last[1] & mine[1], l3 = last[1] & ~mine[1];
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        if (odds) {                                    // rows of marked samples may hold anything
            for (int r = 0; r < 16; ++r)
                if ((odds >> r) & 1u)
                    for (int i = lane; i < CPR; i += 32) asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(from + r * (D * 2) + i * 16), "r"(0) : "memory");
            __syncwarp();
        }
#pragma unroll
        for (int i = 0; i < D / 16; ++i) {
            uint32_t b0r, b1r, b2r, b3r;
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(b0r), "=r"(b1r), "=r"(b2r), "=r"(b3r) : "r"((from + get) ^ (i << 5)));
            mma_bf16(c[2 * i], a0, a1, a2, a3, b0r, b1r);
            mma_bf16(c[2 * i + 1], a0, a1, a2, a3, b2r, b3r);
            mma_bf16(c[2 * i], r0, r1, r2, r3, b0r, b1r);
            mma_bf16(c[2 * i + 1], r0, r1, r2, r3, b2r, b3r);
            mma_bf16(c[2 * i], l0, l1, l2, l3, b0r, b1r);
            mma_bf16(c[2 * i + 1], l0, l1, l2, l3, b2r, b3r);
        }
        if (f + 16u >= stop) {                         // the run is complete
            const int rt = b.t + (run >> 2) + ((g8 >> 1) & 1), ry = b.y + (run & 3) + (g8 & 1), rx = b.x + col;
            // rows that no sample has a weight for (most of them when offsets are integers) are left alone
            const unsigned any_a = __ballot_sync(kFullMask, used_a != 0u) >> (lane & 28), any_b = __ballot_sync(kFullMask, used_b != 0u) >> (lane & 28);
            used_a = used_b = 0u;
            if (static_cast<unsigned>(rt) < static_cast<unsigned>(pr.T) && static_cast<unsigned>(ry) < static_cast<unsigned>(pr.H)) {
                float* to = acc + ((static_cast<long long>(rt) * pr.H + ry) * pr.W + rx) * tok;
                if ((any_a & 15u) && static_cast<unsigned>(rx) < static_cast<unsigned>(pr.W) && DSA3D_IN_RANGE(pr, to - (tensor ? acc_dv : acc_dk), kv_extent, 10)) {
#pragma unroll
                    for (int i = 0; i < D / 8; ++i) red_add_v2(to + 8 * i, c[i][0], c[i][1]);
                }
                to += 2 * tok;
                if ((any_b & 15u) && static_cast<unsigned>(rx + 2) < static_cast<unsigned>(pr.W) && DSA3D_IN_RANGE(pr, to - (tensor ? acc_dv : acc_dk), kv_extent, 10)) {
#pragma unroll
                    for (int i = 0; i < D / 8; ++i) red_add_v2(to + 8 * i, c[i][2], c[i][3]);
                }
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < D / 8; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0.0f;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

template <int D, bool kGated>
__global__ void __launch_bounds__(kSumThreads, D == 32 ? 3 : 2)
cells_sums_kernel(const bf16* __restrict__ q, const bf16* __restrict__ dout, const float* __restrict__ offsets, float* __restrict__ acc_dk,
                  float* __restrict__ acc_dv, const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned blocks) {
    if constexpr (!kGated) {
        if (blockIdx.x < blocks) sums_block<D>(blockIdx.x, q, dout, acc_dk, acc_dv, pr, sl);
        else far_part<bf16, D, true>(blockIdx.x - blocks, gridDim.x - blocks, q, static_cast<const bf16*>(nullptr), static_cast<const bf16*>(nullptr), dout, offsets, acc_dk, acc_dv, pr, sl);
    } else {
        if (gated_off_early(pr.gate)) return;
        for (unsigned block = blockIdx.x; block < blocks; block += gridDim.x) {
            sums_block<D>(block, q, dout, acc_dk, acc_dv, pr, sl);
            __syncthreads();
        }
        far_part<bf16, D, true>(blockIdx.x, gridDim.x, q, static_cast<const bf16*>(nullptr), static_cast<const bf16*>(nullptr), dout, offsets, acc_dk, acc_dv, pr, sl);
    }
}


// ------------------------------------------------------------------------------------------------ fp32 storage
// The block kernels for fp32 storage, on fp32 FMAs.  A cell's samples follow one another through a group of D / 4 lanes (16
// bytes of a row each; groups alternate between the two tensors) which holds the cell's eight corner rows - for the
// sums, their accumulators - in registers: per sample one query row is read instead of eight key rows, and a cell's rows are
// reduced into the accumulators once instead of once per sample (which bound the row kernels: 1.67 ms
// for 99840 items of 64 channels, window (3,3,3), against 1.19 ms; the issue rate bounds these: 104 and 83 instructions of a
// warp per sample).
constexpr int kF32Ahead = 4;        // samples a group has in flight

template <int D> struct F32Lanes {
    static constexpr int LPR = D / 4, U = 32 / LPR, SP = U > 1 ? U / 2 : 1;       // groups of a warp; samples it takes at a time
    int gl, tensor, sub, cell0, cell_step;
    __device__ __forceinline__ F32Lanes() {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, slot = lane / LPR;
        gl = lane % LPR;
        tensor = U > 1 ? slot & 1 : warp & 1;
        sub = slot >> 1;
        cell0 = U > 1 ? warp : warp >> 1;
        cell_step = static_cast<int>(blockDim.x) / (U > 1 ? 32 : 64);
    }
};

template <int D, int kThreads>
__global__ void __launch_bounds__(kThreads, 640 / kThreads)
cells_dots_f32_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v, const float* __restrict__ dout,
                      const float* __restrict__ offsets, const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned blocks) {
    if (gated_off_early(pr.gate)) return;
    if (blockIdx.x >= blocks) {
        far_part<float, D, false>(blockIdx.x - blocks, gridDim.x - blocks, q, k, v, dout, offsets, nullptr, nullptr, pr, sl);
        return;
    }
    using L = F32Lanes<D>;
    constexpr int LPR = L::LPR, SP = L::SP;
    const uint32_t* first = sl.first + static_cast<long long>(blockIdx.x) * (kCells + 1);
    if (__ldg(first) == __ldg(first + kCells)) return;
    const L ln;
    const BlockPos b = block_pos(sl, blockIdx.x);
    const long long tok = static_cast<long long>(pr.heads) * D, head = static_cast<long long>(b.m) * D + ln.gl * 4;
    const float* keys = (ln.tensor ? v : k) + head;
    const float* src = (ln.tensor ? dout : q) + head;
    float* out = sl.stats + ln.tensor * 4 + ((ln.gl & (LPR / 2)) ? 2 : 0) + ((ln.gl & (LPR / 4)) ? 1 : 0);
    const bool writes = (ln.gl & (LPR / 4 - 1)) == 0;
    for (int cell = ln.cell0; cell < kCells; cell += ln.cell_step) {
        const uint32_t f0 = __ldg(first + cell), f1 = __ldg(first + cell + 1);
        if (f0 == f1) continue;
        float4 rows[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int t = b.t + cell_t(cell) + (c >> 2), y = b.y + cell_y(cell) + ((c >> 1) & 1), x = b.x + cell_x(cell) + (c & 1);
            rows[c] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (static_cast<unsigned>(t) < static_cast<unsigned>(pr.T) && static_cast<unsigned>(y) < static_cast<unsigned>(pr.H) && static_cast<unsigned>(x) < static_cast<unsigned>(pr.W))
                rows[c] = __ldg(reinterpret_cast<const float4*>(keys + ((static_cast<long long>(t) * pr.H + y) * pr.W + x) * tok));
        }
        for (uint32_t f = f0; f < f1; f += SP * kF32Ahead) {
            float4 geo[kF32Ahead], r[kF32Ahead];
            uint32_t at[kF32Ahead];
#pragma unroll
            for (int i = 0; i < kF32Ahead; ++i) {
                const uint32_t s = min(f + static_cast<uint32_t>(i * SP + ln.sub), f1 - 1u);       // a missing sample repeats the last one
                geo[i] = __ldg(sl.sorted + s);
                at[i] = __ldg(sl.place + s);
            }
#pragma unroll
            for (int i = 0; i < kF32Ahead; ++i) r[i] = __ldg(reinterpret_cast<const float4*>(src + __float_as_int(geo[i].w) * tok));
#pragma unroll
            for (int i = 0; i < kF32Ahead; ++i) {
                if (f + static_cast<uint32_t>(i * SP) >= f1) break;
                const float ft = geo[i].x, fy = geo[i].y, fx = geo[i].z;
                float a[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) a[c] = fmaf(r[i].w, rows[c].w, fmaf(r[i].z, rows[c].z, fmaf(r[i].y, rows[c].y, r[i].x * rows[c].x)));
                // corners whose weight and weight derivatives are all zero do not enter (they may hold anything)
                if (ft == 0.0f || fy == 0.0f || fx == 0.0f) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (((c >> 2) && ft == 0.0f) + (((c >> 1) & 1) && fy == 0.0f) + ((c & 1) && fx == 0.0f) > 1) a[c] = 0.0f;
                }
                float n0, n1, n2, n3;
                trilerp_grad(a, ft, fy, fx, n0, n1, n2, n3);
                // four sums over the group, handing half of the numbers over at each of the first two steps
                const bool up = ln.gl & (LPR / 2), up2 = ln.gl & (LPR / 4);
                const float x0 = (up ? n2 : n0) + __shfl_xor_sync(kFullMask, up ? n0 : n2, LPR / 2);
                const float x1 = (up ? n3 : n1) + __shfl_xor_sync(kFullMask, up ? n1 : n3, LPR / 2);
                float x = (up2 ? x1 : x0) + __shfl_xor_sync(kFullMask, up2 ? x0 : x1, LPR / 4);
#pragma unroll
                for (int o = LPR / 8; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
                if (writes && f + static_cast<uint32_t>(i * SP + ln.sub) < f1) out[static_cast<size_t>(at[i]) * 8] = x;
            }
        }
    }
}

template <int D, int kThreads>
__global__ void __launch_bounds__(kThreads, 640 / kThreads)
cells_sums_f32_kernel(const float* __restrict__ q, const float* __restrict__ dout, const float* __restrict__ offsets, float* __restrict__ acc_dk,
                      float* __restrict__ acc_dv, const __grid_constant__ Problem pr, const __grid_constant__ Slab sl, unsigned blocks) {
    if (gated_off_early(pr.gate)) return;
    if (blockIdx.x >= blocks) {
        far_part<float, D, true>(blockIdx.x - blocks, gridDim.x - blocks, q, static_cast<const float*>(nullptr), static_cast<const float*>(nullptr), dout, offsets, acc_dk, acc_dv, pr, sl);
        return;
    }
    using L = F32Lanes<D>;
    constexpr int LPR = L::LPR, SP = L::SP;
    const uint32_t* first = sl.first + static_cast<long long>(blockIdx.x) * (kCells + 1);
    if (__ldg(first) == __ldg(first + kCells)) return;
    const L ln;
    const BlockPos b = block_pos(sl, blockIdx.x);
    [[maybe_unused]] const long long kv_extent = pr.N * pr.heads * D;
    const long long tok = static_cast<long long>(pr.heads) * D, head = static_cast<long long>(b.m) * D + ln.gl * 4;
    const float* src = (ln.tensor ? dout : q) + head;
    float* const base = ln.tensor ? acc_dv : acc_dk;
    for (int cell = ln.cell0; cell < kCells; cell += ln.cell_step) {
        const uint32_t f0 = __ldg(first + cell), f1 = __ldg(first + cell + 1);
        if (f0 == f1) continue;
        float acc[8][4];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.0f;
        unsigned used = 0u;                            // corners that a sample has a weight for
        for (uint32_t f = f0; f < f1; f += SP * kF32Ahead) {
            float4 geo[kF32Ahead], r[kF32Ahead];
            float2 cf[kF32Ahead];
#pragma unroll
            for (int i = 0; i < kF32Ahead; ++i) {
                const uint32_t s = min(f + static_cast<uint32_t>(i * SP + ln.sub), f1 - 1u);
                geo[i] = __ldg(sl.sorted + s);
                cf[i] = __ldg(sl.coef + __ldg(sl.place + s));
                r[i] = __ldg(reinterpret_cast<const float4*>(src + __float_as_int(geo[i].w) * tok));
            }
#pragma unroll
            for (int i = 0; i < kF32Ahead; ++i) {
                // beyond the cell, or marked (far_part takes it)
                if (f + static_cast<uint32_t>(i * SP + ln.sub) >= f1 || (__float_as_uint(cf[i].y) >> 31)) continue;
                const float ft = geo[i].x, fy = geo[i].y, fx = geo[i].z, co = ln.tensor ? cf[i].y : cf[i].x;
                used |= weighted_corners(0xffu, ft, fy, fx);
                const float wt[2] = {1.0f - ft, ft}, wy[2] = {1.0f - fy, fy}, wx[2] = {(1.0f - fx) * co, fx * co};
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float w = wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1];
                    fma2(acc[c][0], acc[c][1], w, w, r[i].x, r[i].y);
                    fma2(acc[c][2], acc[c][3], w, w, r[i].z, r[i].w);
                }
            }
        }
#pragma unroll
        for (int o = 2 * LPR; o < 32; o <<= 1) {       // groups that shared the cell's samples
            used |= __shfl_xor_sync(kFullMask, used, o);
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[c][e] += __shfl_xor_sync(kFullMask, acc[c][e], o);
        }
        if (ln.sub != 0) continue;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int t = b.t + cell_t(cell) + (c >> 2), y = b.y + cell_y(cell) + ((c >> 1) & 1), x = b.x + cell_x(cell) + (c & 1);
            if (!((used >> c) & 1u) || static_cast<unsigned>(t) >= static_cast<unsigned>(pr.T) || static_cast<unsigned>(y) >= static_cast<unsigned>(pr.H) ||
                static_cast<unsigned>(x) >= static_cast<unsigned>(pr.W))
                continue;
            float* to = base + ((static_cast<long long>(t) * pr.H + y) * pr.W + x) * tok + head;
            if (DSA3D_IN_RANGE(pr, to - base, kv_extent, 10))
                red_add_v4(to, acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
        }
    }
}

// ------------------------------------------------------------------------------------------------ host
int floor_div4(int a) { return a >= 0 ? a / 4 : -((-a + 3) / 4); }

size_t round256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

// Lays a slab's buffers out at `base` (may be NULL); returns their bytes.  They depend on how many heads and frames the slab has and
// not on where its frames lie, and fewer need no more: a slab at the video's start has only one layer of blocks below
// its tiles, one in the middle three, so room is taken for the most that any can have - three below and three above, and
// no more than blocks of four cut the cells -1 .. T - 1 into wherever they begin.
size_t lay_out(const Problem& pr, int m0, int heads, int f0, int f1, char* base, Slab& s) {
    s.m0 = m0; s.heads = heads; s.f0 = f0; s.f1 = f1;
    s.tiles_t = (f1 - f0 - 1) / 4 + 1; s.tiles_y = (pr.H + 3) / 4; s.tiles_x = (pr.W + kTileX - 1) / kTileX;
    const int lo = floor_div4(-1 - f0), hi = floor_div4(pr.T - 1 - f0);
    s.bt0 = lo < -3 ? -3 : lo;
    const int top = s.tiles_t - 1 + 3 < hi ? s.tiles_t - 1 + 3 : hi;
    s.blocks_t = top - s.bt0 + 1;
    s.blocks_y = (pr.H - 1) / 4 + 2;
    s.blocks_x = (pr.W - 1) / kBlockX + 2;
    const size_t tiles = static_cast<size_t>(heads) * s.tiles_t * s.tiles_y * s.tiles_x, samples = tiles * kRows * pr.P;
    const size_t live = static_cast<size_t>(heads) * (f1 - f0) * pr.H * pr.W * pr.P;
    if (samples >> 32) return ~static_cast<size_t>(0);          // places are 32-bit
    size_t at = 0;
    s.geo = reinterpret_cast<uint4*>(base + at); at += round256(samples * sizeof(uint4));
    s.meta = reinterpret_cast<uint16_t*>(base + at); at += round256(samples * sizeof(uint16_t));
    s.seg = reinterpret_cast<uint32_t*>(base + at); at += round256(tiles * (kBins + 1) * sizeof(uint32_t));
    const int layers = s.tiles_t + 6 < (pr.T - 1) / 4 + 2 ? s.tiles_t + 6 : (pr.T - 1) / 4 + 2;
    if (s.blocks_t > layers) return ~static_cast<size_t>(0);
    const size_t blocks = static_cast<size_t>(heads) * layers * s.blocks_y * s.blocks_x;
    s.sorted = reinterpret_cast<float4*>(base + at); at += round256(live * sizeof(float4));
    s.place = reinterpret_cast<uint32_t*>(base + at); at += round256(live * sizeof(uint32_t));
    s.first = reinterpret_cast<uint32_t*>(base + at); at += round256(blocks * (kCells + 1) * sizeof(uint32_t));
    s.stats = reinterpret_cast<float*>(base + at); at += round256(live * 8 * sizeof(float));
    s.coef = reinterpret_cast<float2*>(base + at); at += round256(live * sizeof(float2));
    s.marked = reinterpret_cast<int*>(base + at);
    s.used = reinterpret_cast<uint32_t*>(base + at + 128); at += 256;
    return at;
}

// Behind a gate that is mostly closed launching all CTAs would cost more than anything else (0.95 ms for 1.8 M of the query kernel):
// the gated instances loop over their blocks, with about as many CTAs as an SM holds (four times as many cost an
// empty chain 6 us more).
template <typename T, int D, bool kGated>
cudaError_t launch_slab(const void* q_, const void* k_, const void* v_, const float* offsets, const float* lse, const void* dout_, void* dq_,
                        float* acc_dk, float* acc_dv, float* doffsets, const Problem& pr, const Slab& s, void* clear, size_t clear_bytes, cudaStream_t stream,
                        cudaEvent_t queries_done) {
    constexpr bool kF32 = std::is_same<T, float>::value;
    const T *q = static_cast<const T*>(q_), *k = static_cast<const T*>(k_), *v = static_cast<const T*>(v_), *dout = static_cast<const T*>(dout_);
    const unsigned tiles = static_cast<unsigned>(s.heads * s.tiles_t * s.tiles_y * s.tiles_x), blocks = static_cast<unsigned>(s.heads * s.blocks_t * s.blocks_y * s.blocks_x);
    const unsigned inv_p = ((1u << 24) + static_cast<unsigned>(pr.P) - 1u) / static_cast<unsigned>(pr.P);
    auto grid = [](unsigned n, unsigned resident) { return kGated && n > 148u * resident ? 148u * resident : n; };
    cudaError_t e = cudaSuccess;
    auto big = [&](auto kern, size_t smem) {           // allows the kernel its dynamic shared memory
        if (e == cudaSuccess && smem > 48 * 1024) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        return kern;
    };
    const bool keep = pr.P <= kBinKeep;
    const size_t bin_smem = static_cast<size_t>((kBins + 1) * kCopies + kRows * pr.P * (keep ? 4 : 1)) * sizeof(uint32_t), dot_smem = kF32 ? 0 : sizeof(DotSmem<D>), sum_smem = kF32 ? 0 : sizeof(SumSmem<D>) + 256;
    const bool wide = ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(dout)) & 31u) == 0;
    // fp32: a warp takes cell after cell; CTAs of four warps while they fill the chip three times (five to an SM: the smallest
    // loss at the end of a block), beyond that many warps to a block so that each has few cells
    [[maybe_unused]] const unsigned f32_threads = blocks >= 3u * 5u * 148u ? 128u : 512u;
    auto bin = big(keep ? cells_bin_kernel<kGated, true> : cells_bin_kernel<kGated, false>, bin_smem);
    auto dots = [&] { if constexpr (kF32) return f32_threads == 128u ? cells_dots_f32_kernel<D, 128> : cells_dots_f32_kernel<D, 512>; else return big(wide ? cells_dots_kernel<D, true, kGated> : cells_dots_kernel<D, false, kGated>, dot_smem); }();
    auto sums = [&] { if constexpr (kF32) return f32_threads == 128u ? cells_sums_f32_kernel<D, 128> : cells_sums_f32_kernel<D, 512>; else return big(cells_sums_kernel<D, kGated>, sum_smem); }();
    if (e != cudaSuccess) return e;
    bool ordinary = kF32;                              // the kernel that writes the gate may be the one before
    auto launch = [&](auto kern, unsigned ctas, unsigned threads, size_t smem, const auto&... args) {
        if (e != cudaSuccess) return;
        if (kGated && !ordinary) {
            e = launch_gated(kern, dim3(ctas), threads, smem, stream, args...);
        } else {
            kern<<<ctas, threads, smem, stream>>>(args...);
            e = cudaGetLastError();
        }
    };
    const long long clear_all = static_cast<long long>(clear_bytes / 16);
    launch(bin, grid(tiles, 2), kBinThreads, bin_smem, offsets, pr, s, inv_p, tiles, static_cast<uint4*>(clear), (clear_all + tiles - 1) / tiles, clear_all);
    ordinary = false;
    launch(cells_sort_kernel<kGated>, grid(blocks, 4), kSortThreads, 0, pr, s, blocks);
    const unsigned far_parts = tiles < 148u * 4u ? tiles : 148u * 4u;
    launch(dots, grid(blocks + far_parts, kF32 ? 1u << 20 : 3u), kF32 ? f32_threads : kDotThreads, dot_smem, q, k, v, dout, offsets, pr, s, blocks);
    // As many queries per warp as have a lane for every sample.
    const int share = pr.P <= 8 ? 4 : pr.P <= 16 ? 2 : 1, per_block = kQueryWarps * share;
    const unsigned per_head = static_cast<unsigned>((static_cast<long long>(s.f1 - s.f0) * pr.H * pr.W + per_block - 1) / per_block), query_blocks = per_head * static_cast<unsigned>(s.heads);
    auto query = share == 4 ? cells_query_kernel<T, D, 4, true, kGated> : share == 2 ? cells_query_kernel<T, D, 2, true, kGated> : pr.P <= 32 ? cells_query_kernel<T, D, 1, true, kGated> : cells_query_kernel<T, D, 1, false, kGated>;
    launch(query, grid(query_blocks, 12), kQueryWarps * 32, 0, k, offsets, lse, static_cast<T*>(dq_), doffsets, pr, s, per_head, query_blocks);
    if (e == cudaSuccess && queries_done) e = cudaEventRecord(queries_done, stream);
    launch(sums, grid(blocks + far_parts, kF32 ? 1u << 20 : 2u), kF32 ? f32_threads : kSumThreads, sum_smem, q, dout, offsets, acc_dk, acc_dv, pr, s, blocks);
    return e;
}

// fp32 storage: *on_grid = 1 if most of up to 4096 samples spread over the offsets lie on grid positions, *off_grid = 1 if not.
__global__ void __launch_bounds__(1024)
cells_choose_kernel(const float* __restrict__ offsets, long long samples, int* __restrict__ on_grid, int* __restrict__ off_grid) {
    int off = 0, seen = 0;
    for (int i = 0; i < 4; ++i) {
        const long long s = (samples * (4 * static_cast<int>(threadIdx.x) + i)) >> 12;
        if (i > 0 && s == (samples * (4 * static_cast<int>(threadIdx.x) + i - 1)) >> 12) continue;
        const float a = offsets[3 * s], b = offsets[3 * s + 1], c = offsets[3 * s + 2];
        ++seen;
        off += floorf(a) != a || floorf(b) != b || floorf(c) != c;
    }
    const int votes = __syncthreads_count(2 * off > seen);
    if (threadIdx.x == 0) {
        *on_grid = 2 * votes <= 1024;
        *off_grid = 2 * votes > 1024;
    }
}
}  // namespace

cudaError_t launch_cells_choose(const float* offsets, long long samples, int* on_grid, int* off_grid, cudaStream_t stream) {
    cells_choose_kernel<<<1, 1024, 0, stream>>>(offsets, samples, on_grid, off_grid);
    return cudaGetLastError();
}

// The heads and frames of a pass over `pr`'s heads and `frames` of its frames whose buffers fit `bytes`: divided by heads first
// (they share nothing), then by frames.  Returns the bytes of the largest pass, 0 if the smallest does not fit.
static size_t divide(const Problem& pr, size_t bytes, int& heads, int& frames) {
    heads = pr.heads;
    Slab s;
    size_t need;
    while ((need = lay_out(pr, 0, heads, 0, frames, nullptr, s)) > bytes) {
        if (heads > 1) heads = (heads + 1) / 2;
        else if (frames > 4) frames = ((frames + 1) / 2 + 3) / 4 * 4;
        else return 0;
    }
    return need;
}

static int frames_in(const Problem& pr) { return static_cast<int>(pr.q_count / (static_cast<long long>(pr.H) * pr.W)); }

// Scratch the fp32 route asks for: all queries of `pr` in one pass up to 1 GiB, passes of at most that beyond.
size_t cells_scratch_bytes(const Problem& pr) {
    int heads, frames = frames_in(pr);
    return divide(pr, static_cast<size_t>(1) << 30, heads, frames);
}

int cells_passes(const Problem& pr, size_t bytes, size_t* largest) {
    *largest = 0;
    int heads, frames = pr.T;
    if (divide(pr, bytes, heads, frames) == 0) return 0;
    Slab s;
    int passes = 0;
    for (int f = 0; f < pr.T; f += frames)
        for (int m = 0; m < pr.heads; m += heads, ++passes) {
            const int f1 = f + frames < pr.T ? f + frames : pr.T, mh = m + heads < pr.heads ? heads : pr.heads - m;
            const size_t used = lay_out(pr, m, mh, f, f1, nullptr, s);
            const uint32_t* first_end = s.first + static_cast<size_t>(mh) * s.blocks_t * s.blocks_y * s.blocks_x * (kCells + 1);
            if (first_end > reinterpret_cast<const uint32_t*>(s.stats)) { *largest = ~static_cast<size_t>(0); return passes + 1; }
            if (used > *largest) *largest = used;
        }
    return passes;
}

bool cells_fit(const Problem& pr, size_t bytes) {
    int heads, frames = frames_in(pr);
    return divide(pr, bytes, heads, frames) != 0;
}

cudaError_t launch_cells_backward(const void* q, const void* k, const void* v, const float* offsets, const float* lse, const void* dout, void* dq,
                                  float* acc_dk, float* acc_dv, float* doffsets, void* scratch, size_t bytes, void* clear, size_t clear_bytes,
                                  const Problem& pr, bool bf16_storage, cudaStream_t stream, cudaEvent_t queries_done) {
    const int f_begin = static_cast<int>(pr.q_begin / (static_cast<long long>(pr.H) * pr.W)), f_end = f_begin + frames_in(pr);
    int heads, frames = f_end - f_begin;
    if (divide(pr, bytes, heads, frames) == 0) return cudaErrorInvalidValue;
    Slab s;
    for (int f = f_begin; f < f_end; f += frames)
        for (int m = 0; m < pr.heads; m += heads) {
            const int f1 = f + frames < f_end ? f + frames : f_end, mh = m + heads < pr.heads ? heads : pr.heads - m;
            if (lay_out(pr, m, mh, f, f1, static_cast<char*>(scratch), s) > bytes) return cudaErrorInvalidValue;
            auto slab = !bf16_storage ? (pr.d == 128 ? launch_slab<float, 128, true> : pr.d == 64 ? launch_slab<float, 64, true> : launch_slab<float, 32, true>)
                        : pr.d == 128 ? (pr.gate ? launch_slab<bf16, 128, true> : launch_slab<bf16, 128, false>)
                        : pr.d == 64  ? (pr.gate ? launch_slab<bf16, 64, true> : launch_slab<bf16, 64, false>)
                                      : (pr.gate ? launch_slab<bf16, 32, true> : launch_slab<bf16, 32, false>);
            const bool last = f1 == f_end && m + mh == pr.heads;
            const cudaError_t e = slab(q, k, v, offsets, lse, dout, dq, acc_dk, acc_dv, doffsets, pr, s, clear, clear_bytes, stream, last ? queries_done : nullptr);
            clear_bytes = 0;                                        // the first pass clears for all
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace dsa3d
