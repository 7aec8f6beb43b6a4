// Fixed-window forward for windows larger than 3 x 3 x 3 (the paper's own (3,7,7) of its zero-offset ablation, and (3,5,5)) as
// tile attention with both contractions on the tensor cores, one region plane at a time; and, with the box of 5 x 5 x 5
// positions that the samples can reach in the window's place, the forward for learned offsets below 1 in size.
//
// With zero offsets sample p of a query sits on the grid position query + b(p).  The halo region of a 4 x 4 x 8 query tile holds
// (4+kt-1)(4+kh-1)(8+kw-1) key rows - 840 for (3,7,7) - more than shared memory takes at once, so the tile walks
// the region's kt+3 planes (along t) twice, K planes and then V planes through one ring of buffers filled by TMA (zero rows
// outside the grid = the zero-padded key of a dead sample).  A pair of x-rows of eight queries has a table of its queries'
// window positions in shared memory (dsa3d_window_planes.cuh) and two warps (one for 64 channels):
//
//   K planes   per region row of 8 + kw - 1 positions: positions x channels x queries (m16n8k16, all channels; the warps take the
//              region rows in turn), scores of positions inside a query's window into the table;
//   softmax    four threads (two) per query, over its part of the table; lse out; each fp32 weight back into the table as a bf16
//              head and a bf16 remainder (relative error of the pair 2^-17, far inside the rounding of the output).
//              Learned offsets: every sample's logit is the trilinear combination of eight scores of the box, and the weights alpha_p *
//              w_c are summed per position of the box;
//   V planes   channels x positions x queries for head and remainder, a warp 64 channels of both x-rows.
//
// What bounds it, (3,7,7), 128 channels: chains of ldmatrix and products at 16 warps an SM, 340 clocks per query; the data pipe (ldmatrix,
// table) is busy for 60 % of them, the tensor unit for 42 % (66 products of 2.16 clocks; the first and the last region row are multiplied with both
// x-rows although one of them does not reach it).  128 registers, 4 to 12 bytes spilled at 128 channels.  A dense product of the tile's 128 queries with a
// plane (tcgen05) spends its time on moving every score plane from TMEM through shared memory into registers and on laying the weights out
// among the plane's columns.  That kernel -> this one, 64 x 45 x 80, 16 heads of 128: (3,7,7) 4.94 -> 4.38 ms, (3,5,5) 3.39 -> 3.36 ms,
// learned offsets 6.89 -> 6.69 ms; 16 x 45 x 80, 16 heads of 64: 1156 -> 869 us, 760 -> 693 us, 1494 -> 1425 us; 4 x 9 x 13, 2 heads of 64:
// 25.8 -> 20.5 us, 18.5 -> 16.4 us, 38.0 -> 35.9 us.  (Sums of even and odd chunks of channels apart, or the operands of the next region row
// ahead of the products: 2 to 4 % slower, for registers.)
//
// The last warp to leave a plane buffer issues its next load; the warps of a pair meet at a barrier of their own.  Every wait on an mbarrier
// is bounded; a wait that runs out raises the library's timeout flag, after which nobody waits or loads any more: the CTA walks
// through the rest of its work and drains its loads.
#include <cuda_bf16.h>

#include <cfloat>
#include <cmath>

#include "dsa3d_common.cuh"
#include "dsa3d_kernels.h"
#include "dsa3d_window_planes.cuh"

namespace dsa3d {
namespace {

constexpr int kPlTT = 4, kPlTY = 4, kPlTX = 8;                      // queries per tile

// BOUNDED = false: fixed window (KT, KH, KW), all offsets zero.  BOUNDED = true: learned offsets with
// |offset| < 1 on every axis; (KT, KH, KW) is then the BOX of grid positions a query's samples can touch,
// the window grown by one position on each side, and the window itself is (KT-2, KH-2, KW-2).
template <int D, int KT, int KH, int KW>
struct PlaneShape : WindowPlanes<D, KT, KH, KW> {
    using B = WindowPlanes<D, KT, KH, KW>;
    static constexpr int PARTS = B::PAIR / 16;                      // threads per query
    static constexpr int NS_RAW = (227 * 1024 - 3072 - (8 * KT + 1) * B::TABLE * 4 - B::WARPS * kPlTX * 128) / (B::NH * B::SLOT_HALF);
    static constexpr int NS = NS_RAW > 4 ? 4 : NS_RAW;
    static_assert(NS >= 2, "at least two plane buffers");
    static_assert(KT * B::TABLE * 4 >= 16 * D * 2, "a pair's query rows are staged in its table");
};

template <int D, int KT, int KH, int KW>
struct __align__(1024) PlSmem {
    using S = PlaneShape<D, KT, KH, KW>;
    unsigned char slot[S::NS][S::NH][S::SLOT_HALF];                 // ring of K or V planes
    unsigned char out[S::WARPS][kPlTX * 128];                       // a warp's results on their way out
    uint32_t table[8][KT][S::TABLE];                                // per pair: scores, then weights, of its queries' windows
    uint32_t zero[S::TABLE];                                        // weights of positions outside a query's window
    float2 part[8][2][16];                                          // maximum and sum of a warp's part of a query
    uint64_t bar_full[4];
    unsigned left[4];                                               // warps that are done with a plane buffer
    uint32_t abort;                                                 // a wait ran out somewhere: nobody waits any more
};

// Load j of tile ti (the K planes, then the V planes; j may run into the next tile) into plane buffer sl.
template <int D, int KT, int KH, int KW, typename Locate>
__device__ __forceinline__ void load_plane(PlSmem<D, KT, KH, KW>& s, const CUtensorMap& map_k, const CUtensorMap& map_v, int ti, int j, int sl, int my_tiles, Locate locate) {
    using S = PlaneShape<D, KT, KH, KW>;
    static_assert(S::NS <= 2 * S::RT, "");
    if (j >= 2 * S::RT) { j -= 2 * S::RT; ++ti; }
    if (ti >= my_tiles || *reinterpret_cast<volatile uint32_t*>(&s.abort)) return;
    int m, t0, y0, x0;
    locate(ti, m, t0, y0, x0);
    const uint32_t bar = smem_u32(&s.bar_full[sl]);
    mbar_expect_tx(bar, static_cast<uint32_t>(S::NH) * S::PS * 128u);
    for (int h = 0; h < S::NH; ++h)
        tma_load_5d(smem_u32(s.slot[sl][h]), j < S::RT ? &map_k : &map_v, bar, h * 64, m, x0 - KW / 2, y0 - KH / 2, t0 - KT / 2 + (j < S::RT ? j : j - S::RT));
}
// Gave up: loads may still be in flight towards this CTA's shared memory.
template <int D, int KT, int KH, int KW> __device__ __forceinline__ void drain_planes(PlSmem<D, KT, KH, KW>& s) {
    if (*reinterpret_cast<volatile uint32_t*>(&s.abort) && threadIdx.x == 0)
        for (int i = 0; i < PlaneShape<D, KT, KH, KW>::NS; ++i) {
            mbar_wait_limit(smem_u32(&s.bar_full[i]), 0u, 1u << 16);
            mbar_wait_limit(smem_u32(&s.bar_full[i]), 1u, 1u << 16);
        }
}

// kEdge: pairs whose x-rows both lie outside the grid do nothing but let the planes go by, and the tiles of a last, partial row of tiles
// along t come behind all others, so that no CTA is left with a full tile more than the rest (see launch_planes).
template <int D, int KT, int KH, int KW, bool BOUNDED, bool kEdge>
__global__ void __launch_bounds__(PlaneShape<D, KT, KH, KW>::THREADS, 1)
fixed_window_planes_kernel(const __nv_bfloat16* __restrict__ q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                           __nv_bfloat16* __restrict__ out, float* __restrict__ lse, int T, int H, int W, int heads, int tiles_x, int tiles_y,
                           int total, int* timeout_flag, const float* __restrict__ offsets, const int* __restrict__ gate) {
    using S = PlaneShape<D, KT, KH, KW>;
    constexpr int NH = S::NH, RT = S::RT, NS = S::NS, ROW = S::ROW, TABLE = S::TABLE, PAIR = S::PAIR, PARTS = S::PARTS;
    extern __shared__ unsigned char raw[];
    PlSmem<D, KT, KH, KW>& s = *reinterpret_cast<PlSmem<D, KT, KH, KW>*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) { mbar_init(smem_u32(&s.bar_full[i]), 1); s.left[i] = 0u; }
        s.abort = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    S::template clear_tails<NS>(s.slot);
    for (int i = tid; i < TABLE; i += S::THREADS) s.zero[i] = 0u;
    fence_async_smem();
    __syncthreads();
    volatile uint32_t* abort_flag = &s.abort;
    auto wait = [&](uint64_t* bar, uint32_t parity, int code) -> bool {
        if (*abort_flag) return false;
        if (mbar_wait(smem_u32(bar), parity)) return true;
        atomicExch(timeout_flag, code);
        *abort_flag = 1u;
        return false;
    };
    const int tiles_per_head = total / heads;                        // 32-bit throughout: the host checks the counts fit
    auto locate = [&](int ti, int& m, int& t0, int& y0, int& x0) {   // tile ti of this CTA
        const int item = static_cast<int>(blockIdx.x) + ti * static_cast<int>(gridDim.x);
        int tile = item;
        if (!(kEdge && D == 128)) { m = item / tiles_per_head; tile -= m * tiles_per_head; }
        x0 = (tile % tiles_x) * kPlTX; tile /= tiles_x;
        y0 = (tile % tiles_y) * kPlTY; tile /= tiles_y;
        if (kEdge && D == 128) { m = tile % heads; tile /= heads; }
        t0 = tile * kPlTT;
    };
    // BOUNDED: an earlier kernel on the stream left 0 in *gate if every offset is finite and below 1 in size;
    // otherwise the general kernel behind this one takes the call
    const bool open = !BOUNDED || gate == nullptr || *gate == 0;
    const int my_tiles = open && static_cast<int>(blockIdx.x) < total
                             ? (total - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x) : 0;
    auto load = [&](int ti, int j, int sl) { load_plane<D, KT, KH, KW>(s, map_k, map_v, ti, j, sl, my_tiles, locate); };
    if (tid == 0)
        for (int i = 0; i < NS; ++i) load(0, i, i);
    const int pair = warp / NH, half = warp % NH, lt = pair >> 1, ly = (pair & 1) * 2;     // query plane, first x-row, channels
    const int me = half * 32 + lane;
    // the thread's query of the softmax (x-row of the pair, x) and its part of it
    const int qr = (me >> 3) & 1, qx = me & 7, part = me >> 4;
    uint32_t* table = s.table[pair][0];
    const float lscale = rsqrtf(static_cast<float>(D)) * kLog2e;     // scores in log2 units
    int place[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) place[e] = S::weight_place(e);
    int sl = 0;
    uint32_t parity = 0u;
    auto next_slot = [&](int ti, int j) {                             // done with the plane of load j
        S::release(&s.left[sl], [&] { load(ti, j + NS, sl); });
        if (++sl == NS) { sl = 0; parity ^= 1u; }
    };
    // maximum and sum of the query's parts -> maximum, 1 / sum; every thread of the query calls it
    auto combine = [&](float& mx, float& sum) {
#pragma unroll
        for (int o = 16; o < PAIR && o < 32; o <<= 1) {
            const float m2 = __shfl_xor_sync(kFullMask, mx, o), s2 = __shfl_xor_sync(kFullMask, sum, o), m1 = fmaxf(mx, m2);
            sum = sum * exp2f(mx - m1) + s2 * exp2f(m2 - m1);
            mx = m1;
        }
        if constexpr (NH == 2) {
            if (lane < 16) s.part[pair][half][lane] = make_float2(mx, sum);
            S::pair_barrier(pair);
            const float2 o = s.part[pair][half ^ 1][lane & 15];
            const float m1 = fmaxf(mx, o.x);
            // in the same order on both sides: the parts of a query agree on its sum
            const float own = sum * exp2f(mx - m1), other = o.y * exp2f(o.x - m1);
            sum = half ? other + own : own + other;
            mx = m1;
        }
    };
    for (int ti = 0; ti < my_tiles; ++ti) {
        int m, t0, y0, x0;
        locate(ti, m, t0, y0, x0);
        if (kEdge && (t0 + lt >= T || y0 + ly >= H)) {
_Pragma("unroll 1")
            for (int pl = 0; pl < 2 * RT; ++pl) {
                wait(&s.bar_full[sl], parity, 14);
                next_slot(ti, pl);
            }
            continue;
        }
        const int qt = t0 + lt, qy = y0 + ly + qr, qxx = x0 + qx;
        const bool in_grid = qt < T && qy < H && qxx < W;
        const long long n = (static_cast<long long>(qt) * H + qy) * W + qxx;
        // samples of the thread (learned offsets): every PARTS-th of the window; their offsets are requested now
        constexpr int WT = BOUNDED ? KT - 2 : 1, WH = BOUNDED ? KH - 2 : 1, WW = BOUNDED ? KW - 2 : 1, NP = WT * WH * WW, PH = (NP + PARTS - 1) / PARTS;
        float offv[BOUNDED ? PH : 1][3];
        if constexpr (BOUNDED) {
            const float* off_row = offsets + (n * heads + m) * (NP * 3);
#pragma unroll
            for (int i = 0; i < PH; ++i) {
                const int p = i * PARTS + part;
                offv[i][0] = offv[i][1] = offv[i][2] = 0.0f;
                if (in_grid && p < NP) { offv[i][0] = __ldg(off_row + p * 3); offv[i][1] = __ldg(off_row + p * 3 + 1); offv[i][2] = __ldg(off_row + p * 3 + 2); }
            }
        }
        uint32_t qf[2][D / 16][2];
        S::operands(qf, table, q, pair, me, qt, y0 + ly, x0, m, T, H, W, heads);
        // ---- K planes: the window's scores
_Pragma("unroll 1")
        for (int pl = 0; pl < RT; ++pl) {
            wait(&s.bar_full[sl], parity, 12);
            if (pl >= lt && pl < lt + KT) S::scores(qf, s.slot[sl], ly, half, reinterpret_cast<float*>(table + (pl - lt) * TABLE), lscale);
            next_slot(ti, pl);
            if (pl == lt + KT - 1) S::pair_barrier(pair);             // the scores are in place
        }
        // ---- softmax; the table then holds weights
        // the maximum starts at the lowest finite number: a part of a query whose logits are all minus infinity (masked keys) then has a
        // sum of zero, where the difference of two infinities would make the whole query NaN
        float mx = -FLT_MAX, sum = 0.0f;
        if constexpr (!BOUNDED) {
            constexpr int ROWS = (KT * KH + PARTS - 1) / PARTS;       // kernel rows (u, v) of the thread: every PARTS-th
            float sc[ROWS][KW];
            uint32_t* mine = table + qr * ROW + qx * KW;
            auto at = [&](int i) { const int uv = i * PARTS + part, u = uv / KH; return mine + u * TABLE + (uv - u * KH) * (kPlTX * KW); };
#pragma unroll
            for (int i = 0; i < ROWS; ++i)
#pragma unroll
                for (int w = 0; w < KW; ++w) {
                    sc[i][w] = i * PARTS + part < KT * KH ? __uint_as_float(at(i)[w]) : -INFINITY;
                    mx = fmaxf(mx, sc[i][w]);
                }
#pragma unroll
            for (int i = 0; i < ROWS; ++i)
#pragma unroll
                for (int w = 0; w < KW; ++w) { sc[i][w] = exp2f(sc[i][w] - mx); sum += sc[i][w]; }
            const float own = mx;
            combine(mx, sum);
            const float inv = exp2f(own - mx) / sum;
#pragma unroll
            for (int i = 0; i < ROWS; ++i)
                if (i * PARTS + part < KT * KH)
#pragma unroll
                    for (int w = 0; w < KW; ++w) at(i)[w] = split_weight(sc[i][w] * inv);
        } else {
            float lg[PH], fr[PH][3];
            int cell[PH];
            // position of a sample relative to the box origin, exactly as the general kernel forms it:
            // float(coord + b) + offset, floor, difference - all in fp32
#pragma unroll
            for (int i = 0; i < PH; ++i) {
                const int p = i * PARTS + part, w = p % WW, v = (p / WW) % WH, u = p / (WW * WH);
                const float pt = __fadd_rn(static_cast<float>(qt + u - WT / 2), offv[i][0]), py = __fadd_rn(static_cast<float>(qy + v - WH / 2), offv[i][1]),
                            px = __fadd_rn(static_cast<float>(qxx + w - WW / 2), offv[i][2]);
                const float flt = floorf(pt), fly = floorf(py), flx = floorf(px);
                float ft = __fsub_rn(pt, flt), fy = __fsub_rn(py, fly), fx = __fsub_rn(px, flx);
                // cell index of corner (0,0,0) inside the box (origin = query - K/2).  An offset just below +1
                // can round the fp32 position up to the next integer: the sample then sits exactly on the
                // box's last position, which is written as the cell before it with fraction 1.  (The clamps
                // also keep a garbage offset from indexing outside the box.)
                int ct = max(static_cast<int>(flt) - (qt - KT / 2), 0), cy = max(static_cast<int>(fly) - (qy - KH / 2), 0), cx = max(static_cast<int>(flx) - (qxx - KW / 2), 0);
                if (ct > KT - 2) { ct = KT - 2; ft = 1.0f; }
                if (cy > KH - 2) { cy = KH - 2; fy = 1.0f; }
                if (cx > KW - 2) { cx = KW - 2; fx = 1.0f; }
                cell[i] = ct * TABLE + qr * ROW + (cy * kPlTX + qx) * KW + cx;
                fr[i][0] = ft; fr[i][1] = fy; fr[i][2] = fx;
            }
            auto corner = [](int c) { return (c >> 2) * TABLE + ((c >> 1) & 1) * (kPlTX * KW) + (c & 1); };
            const float* box = reinterpret_cast<const float*>(table);
#pragma unroll
            for (int i = 0; i < PH; ++i) {
                lg[i] = -INFINITY;
                if (i * PARTS + part < NP) {
                    const float ft = fr[i][0], fy = fr[i][1], fx = fr[i][2];
                    float a[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) a[c] = box[cell[i] + corner(c)];
                    const float x0v = fmaf(fx, a[1] - a[0], a[0]), x1v = fmaf(fx, a[3] - a[2], a[2]);
                    const float x2v = fmaf(fx, a[5] - a[4], a[4]), x3v = fmaf(fx, a[7] - a[6], a[6]);
                    const float y0v = fmaf(fy, x1v - x0v, x0v), y1v = fmaf(fy, x3v - x2v, x2v);
                    lg[i] = fmaf(ft, y1v - y0v, y0v);
                    mx = fmaxf(mx, lg[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < PH; ++i) { lg[i] = exp2f(lg[i] - mx); sum += lg[i]; }
            const float own = mx;
            combine(mx, sum);
            const float inv = exp2f(own - mx) / sum;
            S::pair_barrier(pair);                                    // every score of the pair's boxes has been read
            // the box now collects the weights: cleared, then the threads of a query add their samples one after the
            // other (plain read-add-write: no two threads at a cell at once)
            for (int i = 4 * me; i < KT * TABLE; i += 4 * PAIR) *reinterpret_cast<uint4*>(table + i) = make_uint4(0u, 0u, 0u, 0u);
            S::pair_barrier(pair);
            float* sums = reinterpret_cast<float*>(table);
#pragma unroll
            for (int turn = 0; turn < PARTS; ++turn) {
                if (turn == part) {
#pragma unroll
                    for (int i = 0; i < PH; ++i) {
                        if (i * PARTS + part >= NP) continue;
                        const float al = lg[i] * inv;
                        const float wt[2] = {1.0f - fr[i][0], fr[i][0]}, wy[2] = {1.0f - fr[i][1], fr[i][1]}, wx[2] = {1.0f - fr[i][2], fr[i][2]};
                        float old[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) old[c] = sums[cell[i] + corner(c)];
#pragma unroll
                        for (int c = 0; c < 8; ++c) sums[cell[i] + corner(c)] = old[c] + al * (wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1]);
                    }
                }
                if (turn & 1) S::pair_barrier(pair);
                else __syncwarp();
            }
            for (int i = me; i < KT * TABLE; i += PAIR) table[i] = split_weight(sums[i]);
        }
        if (part == 0 && in_grid && !*abort_flag) lse[n * heads + m] = sum > 0.0f ? (mx + log2f(sum)) * kLn2 : NAN;
        S::pair_barrier(pair);                                        // the weights are in place
        // ---- V planes: the output
        float acc[2][4][4];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) acc[r][mt][0] = acc[r][mt][1] = acc[r][mt][2] = acc[r][mt][3] = 0.0f;
_Pragma("unroll 1")
        for (int pl = 0; pl < RT; ++pl) {
            wait(&s.bar_full[sl], parity, 13);
            if (pl >= lt && pl < lt + KT) S::sums(acc, s.slot[sl][half], ly, table + (pl - lt) * TABLE, s.zero, place);
            next_slot(ti, RT + pl);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int y = y0 + ly + r;
            const bool live = qt < T && y < H && !*abort_flag;
            __nv_bfloat16* to = out + (((static_cast<long long>(qt) * H + y) * W + x0) * heads + m) * D + half * 64;
            S::results(acc[r], s.out[warp], [&](int o, int chunk, const uint4& bits) {
                if (live && x0 + o < W) *reinterpret_cast<uint4*>(to + static_cast<long long>(o) * heads * D + chunk * 8) = bits;
            });
        }
    }
    drain_planes<D, KT, KH, KW>(s);
}

bool make_plane_maps(const void* k, const void* v, const Problem& pr, int kh, int kw, CUtensorMap* mk, CUtensorMap* mv) {
    const unsigned long long d = static_cast<unsigned long long>(pr.d), hd = static_cast<unsigned long long>(pr.heads);
    const unsigned long long dims[5] = {d, hd, static_cast<unsigned long long>(pr.W), static_cast<unsigned long long>(pr.H),
                                        static_cast<unsigned long long>(pr.T)};
    const unsigned long long strides[4] = {d * 2, hd * d * 2, static_cast<unsigned long long>(pr.W) * hd * d * 2,
                                           static_cast<unsigned long long>(pr.H) * pr.W * hd * d * 2};
    const unsigned box[5] = {64, 1, static_cast<unsigned>(kPlTX + kw - 1), static_cast<unsigned>(kPlTY + kh - 1), 1};
    return encode_tensor_map_bf16(mk, k, 5, dims, strides, box, true) && encode_tensor_map_bf16(mv, v, 5, dims, strides, box, true);
}

// kEdge where a sixteenth or more of the pairs lies outside the grid: it costs four registers that 128 channels do not have (64 x 45 x 80, a
// twenty-fourth outside: (3,5,5) 1.1 % and small offsets 0.6 % slower); 64 channels take it always.
template <int D, int KT, int KH, int KW, bool BOUNDED>
cudaError_t launch_planes(const void* q, const CUtensorMap& mk, const CUtensorMap& mv, void* out, float* lse,
                          const Problem& pr, int* flag, const float* offsets, const int* gate, cudaStream_t stream) {
    using S = PlaneShape<D, KT, KH, KW>;
    const int tiles_x = (pr.W + kPlTX - 1) / kPlTX, tiles_y = (pr.H + kPlTY - 1) / kPlTY,
              tiles_t = (pr.T + kPlTT - 1) / kPlTT;
    const size_t smem = sizeof(PlSmem<D, KT, KH, KW>) + 1024;
    const long long pairs = static_cast<long long>(tiles_t) * kPlTT * tiles_y * (kPlTY / 2), live = static_cast<long long>(pr.T) * ((pr.H + 1) / 2);
    auto kern = fixed_window_planes_kernel<D, KT, KH, KW, BOUNDED, true>;
    if constexpr (D == 128)
        if (16 * (pairs - live) < pairs) kern = fixed_window_planes_kernel<D, KT, KH, KW, BOUNDED, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    const long long total = static_cast<long long>(tiles_x) * tiles_y * tiles_t * pr.heads;
    if (total * (2 * S::RT) >= (1LL << 31)) return cudaErrorInvalidValue;   // the kernel counts planes in 32 bits
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const unsigned grid = static_cast<unsigned>(total < sms ? total : sms);     // persistent: one CTA per SM
    kern<<<grid, S::THREADS, smem, stream>>>(static_cast<const __nv_bfloat16*>(q), mk, mv, static_cast<__nv_bfloat16*>(out), lse, pr.T, pr.H, pr.W,
                                             pr.heads, tiles_x, tiles_y, static_cast<int>(total), flag, offsets, gate);
    return cudaGetLastError();
}

// *gate = 1 if some offset component is NaN, infinite or not below 1 in size (plain stores of the same
// value: no ordering needed).  The caller has set *gate = 0 on the same stream.
__global__ void __launch_bounds__(256)
offsets_bound_kernel(const float4* __restrict__ off4, long long count4, const float* __restrict__ tail, int tail_count,
                     int* __restrict__ gate) {
    bool bad = false;
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < count4; i += stride) {
        const float4 o = __ldg(off4 + i);
        bad = bad || !(fabsf(o.x) < 1.0f) || !(fabsf(o.y) < 1.0f) || !(fabsf(o.z) < 1.0f) || !(fabsf(o.w) < 1.0f);
    }
    if (blockIdx.x == 0 && static_cast<int>(threadIdx.x) < tail_count) bad = bad || !(fabsf(tail[threadIdx.x]) < 1.0f);
    if (__syncthreads_or(bad) && threadIdx.x == 0) *gate = 1;
}

}  // namespace

bool try_fixed_window_forward_planes(const void* q, const void* k, const void* v, void* out, float* lse,
                                     const Problem& pr, cudaStream_t stream, cudaError_t* err) {
    *err = cudaSuccess;
    if (pr.d != 128 && pr.d != 64) return false;
    const bool w355 = pr.kt == 3 && pr.kh == 5 && pr.kw == 5, w377 = pr.kt == 3 && pr.kh == 7 && pr.kw == 7;
    if (!w355 && !w377) return false;
    const long long tiles = static_cast<long long>((pr.W + kPlTX - 1) / kPlTX) * ((pr.H + kPlTY - 1) / kPlTY) *
                            ((pr.T + kPlTT - 1) / kPlTT);
    if (tiles * pr.heads * 2 * (kPlTT + pr.kt - 1) >= (1LL << 31)) return false;     // the kernel counts planes in 32 bits
    int* flag = timeout_flag_device_address();
    CUtensorMap mk, mv;
    if (!flag || !make_plane_maps(k, v, pr, pr.kh, pr.kw, &mk, &mv)) return false;
    if (pr.d == 128)
        *err = w355 ? launch_planes<128, 3, 5, 5, false>(q, mk, mv, out, lse, pr, flag, nullptr, nullptr, stream)
                    : launch_planes<128, 3, 7, 7, false>(q, mk, mv, out, lse, pr, flag, nullptr, nullptr, stream);
    else
        *err = w355 ? launch_planes<64, 3, 5, 5, false>(q, mk, mv, out, lse, pr, flag, nullptr, nullptr, stream)
                    : launch_planes<64, 3, 7, 7, false>(q, mk, mv, out, lse, pr, flag, nullptr, nullptr, stream);
    return true;
}

bool bounded_offsets_shape_covered(const Problem& pr, bool bf16) {
    return bf16 && (pr.d == 128 || pr.d == 64) && pr.kt == 3 && pr.kh == 3 && pr.kw == 3;
}

cudaError_t launch_offsets_bound_check(const float* offsets, long long count, int* gate, cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(gate, 0, sizeof(int), stream);
    if (e != cudaSuccess) return e;
    const long long count4 = count / 4;
    long long blocks = (count4 + 255) / 256;
    if (blocks > 148LL * 8) blocks = 148LL * 8;
    if (blocks < 1) blocks = 1;
    offsets_bound_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(
        reinterpret_cast<const float4*>(offsets), count4, offsets + count4 * 4, static_cast<int>(count - count4 * 4), gate);
    return cudaGetLastError();
}

bool try_bounded_offsets_forward(const void* q, const void* k, const void* v, const float* offsets, const int* gate,
                                 void* out, float* lse, const Problem& pr, cudaStream_t stream, cudaError_t* err) {
    *err = cudaSuccess;
    if (!bounded_offsets_shape_covered(pr, true)) return false;
    const long long tiles = static_cast<long long>((pr.W + kPlTX - 1) / kPlTX) * ((pr.H + kPlTY - 1) / kPlTY) *
                            ((pr.T + kPlTT - 1) / kPlTT);
    if (tiles * pr.heads * 2 * (kPlTT + pr.kt + 2 - 1) >= (1LL << 31)) return false;
    int* flag = timeout_flag_device_address();
    CUtensorMap mk, mv;
    if (!flag || !make_plane_maps(k, v, pr, pr.kh + 2, pr.kw + 2, &mk, &mv)) return false;
    *err = pr.d == 128 ? launch_planes<128, 5, 5, 5, true>(q, mk, mv, out, lse, pr, flag, offsets, gate, stream)
                       : launch_planes<64, 5, 5, 5, true>(q, mk, mv, out, lse, pr, flag, offsets, gate, stream);
    return true;
}

}  // namespace dsa3d
