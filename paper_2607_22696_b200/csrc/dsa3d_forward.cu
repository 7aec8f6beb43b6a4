// Forward of 3D Deformable Slide Attention (Eq. 1 second term and the softmax under it).  Two kernels, both with an online
// softmax in fp32; nothing of size N*P is written.  Work items are ordered head-major, neighbours along x in one
// CTA, so that the CTAs in flight gather from one head's K / V over a few frames: L2, and L1 within a CTA, serve most rows.
//
// gather_forward_kernel (bf16): a warp owns one (token, head) item and takes its samples
// 32 at a time, one per lane.  The corner rows with a weight are listed in shared memory; q . K_corner of 16 rows is one chain
// of m16n8k16 products, a lane adds the trilinear combination of its sample's corners to a logit, the softmax runs over
// the lanes, and the V rows are summed with fp32 FMAs (dsa3d_gather.cuh).  What bounds it: the L1 data pipe (83 % busy on
// 12 x 45 x 80, 8 heads of 128: 110 KB of rows per item, 5.6 cycles per 512 bytes with the misses, 4 without).
// 32 x 45 x 80, 16 heads of 128, window (3,3,3), offsets N(0, 1.5): 11.4 -> 10.5 ms; N(0, 3): 11.7 -> 9.8; window (3,7,7) on
// 4 x 68 x 120: 18.5 -> 9.8 ms.
//
// (gather_forward_small_kernel: the same for two or four items per warp where the window is small: 32 x 45 x 80, 16 heads of 128, window
// (2,2,2): 3.83 -> 3.24 ms, integer offsets 1.25 -> 0.94 ms.)
//
// forward_kernel (fp32; bf16 with 32 channels and few samples or 128 channels in long calls, see launch_forward): one group of LPR = d / VEC lanes owns one item; each lane holds VEC consecutive channels
// (16 bytes) of every row it touches.  Per sample: the 8 corner rows of K and of V are loaded with 16-byte loads, the
// logit is the weighted sum of the corner dot products, and the output is accumulated in fp32 registers.  A sample whose 8
// corners are all inside the grid with non-zero weights (the usual case for real-valued offsets) takes a branch-free path
// that issues its 16 row loads back to back; border samples and samples on integer positions take a per-corner path that skips
// corners outside the grid and corners of weight zero.
#include <type_traits>

#include "dsa3d_common.cuh"
#include "dsa3d_gather.cuh"
#include "dsa3d_kernels.h"

namespace dsa3d {

__device__ const float kZeroOffset[3] = {0.0f, 0.0f, 0.0f};     // stands in for a NULL offsets tensor

// Two warps per CTA: a warp's slot is free again as soon as it is done (CTAs of 8 warps: 11.2 against 10.5 ms on 32 x 45 x 80,
// 16 heads of 128, offsets N(0, 1.5)).
constexpr int kFwdWarps = 2;

// One item by a warp, row by row: taken when a result is not finite, so that NaN and infinity reach exactly the
// results whose definition they enter (a product with a zero weight makes NaN of infinity).
template <int D>
__device__ __noinline__ void forward_item_plain(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v, const float* offsets,
                                                const __nv_bfloat16* addend, __nv_bfloat16* out, float* lse, const Problem& pr, int m, int t, int y, int x) {
    constexpr int V = D / 32;
    const int lane = threadIdx.x & 31;
    const long long row = ((static_cast<long long>(t) * pr.H + y) * pr.W + x) * pr.heads + m, tok = static_cast<long long>(pr.heads) * D;
    const long long sy = static_cast<long long>(pr.W) * tok, st = static_cast<long long>(pr.H) * sy;
    float acc[V], qv[V], m_run = -INFINITY, l_run = 0.0f;
    for (int i = 0; i < V; ++i) { acc[i] = 0.0f; qv[i] = __bfloat162float(q[row * D + lane * V + i]); }
    for (int p = 0; p < pr.P; ++p) {
        const Sample s = to_sample(pr, make_cell(pr, t, y, x, p, offsets ? offsets + (row * pr.P + p) * 3 : kZeroOffset));
        const unsigned mask = weighted_corners(s.mask, s.ft, s.fy, s.fx);
        const long long o0 = static_cast<long long>(m) * D + s.base * tok + lane * V;
        float sdot = 0.0f;
        for (int c = 0; c < 8; ++c) {
            if (!((mask >> c) & 1u)) continue;
            const float w = ((c & 4) ? s.ft : 1.0f - s.ft) * ((c & 2) ? s.fy : 1.0f - s.fy) * ((c & 1) ? s.fx : 1.0f - s.fx);
            float dot = 0.0f;
            for (int i = 0; i < V; ++i) dot = fmaf(qv[i], __bfloat162float(k[o0 + (c >> 2) * st + ((c >> 1) & 1) * sy + (c & 1) * tok + i]), dot);
            sdot = fmaf(w, group_sum<32>(dot, kFullMask), sdot);
        }
        const float sp = sdot * rsqrtf(static_cast<float>(D)) * kLog2e;
        if (sp > m_run) {
            const float corr = exp2f(m_run - sp);
            l_run *= corr;
            for (int i = 0; i < V; ++i) acc[i] *= corr;
            m_run = sp;
        }
        const float pe = exp2f(sp - m_run);
        l_run += pe;
        for (int c = 0; c < 8; ++c) {
            if (!((mask >> c) & 1u)) continue;
            const float w = pe * (((c & 4) ? s.ft : 1.0f - s.ft) * ((c & 2) ? s.fy : 1.0f - s.fy) * ((c & 1) ? s.fx : 1.0f - s.fx));
            for (int i = 0; i < V; ++i) acc[i] = fmaf(w, __bfloat162float(v[o0 + (c >> 2) * st + ((c >> 1) & 1) * sy + (c & 1) * tok + i]), acc[i]);
        }
    }
    for (int i = 0; i < V; ++i)
        out[row * D + lane * V + i] = __float2bfloat16_rn(acc[i] / l_run + (addend ? __bfloat162float(addend[row * D + lane * V + i]) : 0.0f));
    if (lane == 0) lse[row] = (m_run + log2f(l_run)) * kLn2;
}

// CTAs are handed to the SMs in turn: a wave's CTA numbers are permuted so that kRun consecutive blocks of items, whose samples
// share K and V rows, run on one SM (64 channels: 13.18 -> 12.95 ms for 4.2 M items; 128 channels 32.19 -> 32.06 for 5.5 M;
// runs of 8 and 16 gain less).
__device__ __forceinline__ unsigned sm_neighbours(unsigned block, unsigned blocks) {
    constexpr unsigned kSms = 148u, kRun = 4, kWave = kSms * kRun;
    const unsigned wave = block / kWave, r = block - wave * kWave;
    return (wave + 1u) * kWave <= blocks ? wave * kWave + (r % kSms) * kRun + r / kSms : block;
}

// Bound by the L1 data pipe (87 % at 128 channels, 80 % at 64).  Windows of 17 to 32 samples have an instance of one round (kOne), which
// keeps nothing for a next one: window (3,3,3), 16 x 68 x 120, 16 heads of 128, N(0, 1.5) 11.72 -> 10.92 ms, 16 x 45 x 80 integer offsets
// 1.54 -> 1.26 ms, N(0, 0.5) 5.68 -> 5.57, N(0, 3) 4.63 -> 4.24; 64 channels 6.65 -> 6.56 ms, and 6.32 with 20 CTAs per SM (48
// registers; 24 CTAs, 40 registers: 6.61; 128 channels with 18: 11.3).  With several rounds 128 channels spill 100 bytes at 64 registers.
template <int D, bool kAdd, bool kGated, bool kOne>
__global__ void __launch_bounds__(kFwdWarps * 32, D == 64 && kOne && !kGated ? 20 : 16)
gather_forward_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                      const float* __restrict__ offsets, const __nv_bfloat16* addend, __nv_bfloat16* out, float* __restrict__ lse,
                      const __grid_constant__ Problem pr, unsigned blocks_per_head, const int* __restrict__ gate) {
    if (kGated && *gate == 0) return;                    // another kernel takes this call (see launch_forward)
    __shared__ GatherList lists[kFwdWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    GatherList& gl = lists[warp];
    // One block of items per CTA; behind a gate (a small launch, see launch_gather_forward) a loop over them.  The loop costs the
    // kernel 2 - 15 %, so only the gated instance has it.
    unsigned block = kGated ? blockIdx.x : sm_neighbours(blockIdx.x, gridDim.x);
_Pragma("unroll 1")
    do {
        const int m = static_cast<int>(block / blocks_per_head);
        const long long local = static_cast<long long>(block - static_cast<unsigned>(m) * blocks_per_head) * kFwdWarps + warp;
        if (local >= pr.q_count) { if constexpr (kGated) continue; else return; }
        const int n = static_cast<int>(pr.q_begin + local);
        const int x = n % pr.W, ty = n / pr.W, y = ty % pr.H, t = ty / pr.H;
        const long long row = static_cast<long long>(n) * pr.heads + m;
        const uint32_t tok_bytes = static_cast<uint32_t>(pr.heads) * (D * 2);
        const __nv_bfloat16 *kh = k + static_cast<long long>(m) * D, *vh = v + static_cast<long long>(m) * D;
        const float lscale = rsqrtf(static_cast<float>(D)) * kLog2e;    // logits in log2 units
        constexpr int step = GatherStep<D>::N;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
        float m_run = -INFINITY, l_run = 0.0f;               // l_run: the lane's part
        for (int pb = 0; kOne ? pb == 0 : pb < pr.P; pb += 32) {
            const bool have = pb + lane < pr.P;
            Sample s;
            GatherQuery<D> qr;                               // on its way while the samples are listed
            gather_query<D>(qr, q + row * D);
            s.base = 0; s.mask = 0u; s.ft = s.fy = s.fx = 0.0f;
            if (have) s = to_sample(pr, make_cell(pr, t, y, x, pb + lane, offsets ? offsets + (row * pr.P + pb + lane) * 3 : kZeroOffset));
            const unsigned mask = checked_corners(pr, weighted_corners(s.mask, s.ft, s.fy, s.fx), s.base, 2);
            const GatherPart part = gather_list<1, (D < 128)>(gl, mask, s.base, pr, step);
            __syncwarp();
            gather_dots<D>(gl, part.total, qr, kh, tok_bytes);
            __syncwarp();
            const float wt[2] = {1.0f - s.ft, s.ft}, wy[2] = {1.0f - s.fy, s.fy}, wx[2] = {1.0f - s.fx, s.fx};
            float w[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) w[c] = wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1];
            float sp = gather_combine(gl, part, w);
            sp = have ? sp * lscale : -INFINITY;             // a dead sample stays in the softmax with logit 0
            float mx = sp;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, o));
            if (kOne) {
                m_run = mx;
            } else if (mx > m_run) {
                const float corr = exp2f(m_run - mx);
                l_run *= corr;
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] *= corr;
                m_run = mx;
            }
            const float pe = have ? exp2f(sp - m_run) : 0.0f;
            l_run += pe;
            __syncwarp();
            gather_weights(gl, part, pe, w, step);
            __syncwarp();
            gather_sum<D>(gl, part.total, vh, tok_bytes, acc);
            __syncwarp();
        }
        l_run = group_sum<32>(l_run, kFullMask);
        const float inv = 1.0f / l_run;
        bool bad = !(l_run < INFINITY);
        gather_finish<D>(acc);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            acc[e] *= inv;
            bad = bad || !(fabsf(acc[e]) < INFINITY);
        }
        if (__any_sync(kFullMask, bad)) {
            forward_item_plain<D>(q, k, v, offsets, kAdd ? addend : nullptr, out, lse, pr, m, t, y, x);
            { if constexpr (kGated) continue; else return; }
        }
        if (lane < D / 8) {
            using E = Elt<__nv_bfloat16, 1>;
            if constexpr (kAdd) {                            // first term of Eq. 1, added before the rounding
                float add[8];
                E::to_float(E::load(addend + row * D + lane * 8), add);
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] += add[e];
            }
            E::store(out + row * D + lane * 8, acc);
        }
        if (lane == 0) lse[row] = (m_run + log2f(l_run)) * kLn2;
        if constexpr (!kGated) return;
    } while ((block += gridDim.x) < blocks_per_head * static_cast<unsigned>(pr.heads));
}

// Windows of at most 8 (G = 4) or 16 (G = 2) samples: G neighbouring items share a warp, 32 / G lanes each, so that one trip
// through list, products and softmax serves them all.
template <int D, int G, bool kAdd>
__global__ void __launch_bounds__(kFwdWarps * 32, 16)
gather_forward_small_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                            const float* __restrict__ offsets, const __nv_bfloat16* addend, __nv_bfloat16* out, float* __restrict__ lse,
                            const __grid_constant__ Problem pr, unsigned blocks_per_head, const int* __restrict__ gate) {
    if (gate && *gate == 0) return;
    using E = Elt<__nv_bfloat16, 1>;
    constexpr int L = 32 / G, LPR = GatherStep<D>::LPR, U = GatherStep<D>::U;
    constexpr int PER = U > G ? U / G : 1, ITEMS = G > U ? G / U : 1;        // subgroups per item, items per subgroup
    constexpr int step = 4 * PER > 8 ? 4 * PER : 8, region = kGatherRows / G;
    static_assert(step <= L, "a lane per padding entry");
    __shared__ GatherList lists[kFwdWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, p = lane & (L - 1);
    GatherList& gl = lists[warp];
    const int m = static_cast<int>(blockIdx.x / blocks_per_head);
    const long long warp_first = (static_cast<long long>(blockIdx.x - static_cast<unsigned>(m) * blocks_per_head) * kFwdWarps + warp) * G;
    if (warp_first >= pr.q_count) return;
    const int items = static_cast<int>(min(static_cast<long long>(G), pr.q_count - warp_first));      // an item past the end repeats the last one, stores off
    const int mine = min(lane / L, items - 1), n0 = static_cast<int>(pr.q_begin + warp_first), n = n0 + mine;
    const int x = n % pr.W, ty = n / pr.W, y = ty % pr.H, t = ty / pr.H;
    const long long row = static_cast<long long>(n) * pr.heads + m, row0 = static_cast<long long>(n0) * pr.heads + m;
    const uint32_t tok_bytes = static_cast<uint32_t>(pr.heads) * (D * 2);
    const __nv_bfloat16 *kh = k + static_cast<long long>(m) * D, *vh = v + static_cast<long long>(m) * D;
    const bool have = p < pr.P;
    Sample s;
    s.base = 0; s.mask = 0u; s.ft = s.fy = s.fx = 0.0f;
    if (have) s = to_sample(pr, make_cell(pr, t, y, x, p, offsets ? offsets + (row * pr.P + p) * 3 : kZeroOffset));
    const GatherPart part = gather_list<G>(gl, checked_corners(pr, weighted_corners(s.mask, s.ft, s.fy, s.fx), s.base, 2), s.base, pr, step);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < G; i += 2) {
        const int ta = __shfl_sync(kFullMask, part.total, i * L), tb = __shfl_sync(kFullMask, part.total, (i + 1) * L);
        gather_dots_pair<D>(gl, i * region, ta, (i + 1) * region, tb, q + (row0 + static_cast<long long>(min(i, items - 1)) * pr.heads) * D,
                            q + (row0 + static_cast<long long>(min(i + 1, items - 1)) * pr.heads) * D, kh, tok_bytes);
    }
    __syncwarp();
    const float wt[2] = {1.0f - s.ft, s.ft}, wy[2] = {1.0f - s.fy, s.fy}, wx[2] = {1.0f - s.fx, s.fx};
    float w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1];
    const float sp = have ? gather_combine(gl, part, w) * (rsqrtf(static_cast<float>(D)) * kLog2e) : -INFINITY;
    float mx = sp;
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, o));
    const float pe = have ? exp2f(sp - mx) : 0.0f, l = group_sum<L>(pe, kFullMask), inv = 1.0f / l;
    __syncwarp();
    gather_weights<G>(gl, part, pe * inv, w, step);
    if (p == 0 && lane / L < items) lse[row] = (mx + log2f(l)) * kLn2;
    bool bad = !(l < INFINITY);
    const unsigned bad_l = __ballot_sync(kFullMask, bad && p == 0);
    unsigned redo = 0u;                                  // items with something that is not finite
#pragma unroll
    for (int i = 0; i < G; ++i) redo |= ((bad_l >> (i * L)) & 1u) << i;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int u = lane / LPR, it = PER > 1 ? u / PER : u * ITEMS + i;
        const int total = __shfl_sync(kFullMask, part.total, it * L);
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
        gather_sum_item<D, PER>(gl, it * region, total, PER > 1 ? u % PER : 0, vh, tok_bytes, acc);
        __syncwarp();
#pragma unroll
        for (int o = LPR; o < LPR * PER; o <<= 1)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(kFullMask, acc[e], o);
        bad = false;
#pragma unroll
        for (int e = 0; e < 8; ++e) bad = bad || !(fabsf(acc[e]) < INFINITY);
#pragma unroll
        for (int z = 0; z < G; ++z)
            if (__any_sync(kFullMask, bad && it == z)) redo |= 1u << z;
        if (it < items && (PER == 1 || u % PER == 0)) {
            const long long at = (row0 + static_cast<long long>(it) * pr.heads) * D + (lane % LPR) * 8;
            if constexpr (kAdd) {                        // first term of Eq. 1, added before the rounding
                if (!((redo >> it) & 1u)) {              // (out may be the addend: the plain path below reads it)
                    float add[8];
                    E::to_float(E::load(addend + at), add);
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[e] += add[e];
                    E::store(out + at, acc);
                }
            } else {
                E::store(out + at, acc);
            }
        }
    }
    while (redo) {
        const int it = __ffs(static_cast<int>(redo)) - 1;
        redo &= redo - 1u;
        if (it >= items) break;
        const int n2 = n0 + it;
        forward_item_plain<D>(q, k, v, offsets, kAdd ? addend : nullptr, out, lse, pr, m, n2 / pr.W / pr.H, n2 / pr.W % pr.H, n2 % pr.W);
    }
}

#ifndef DSA3D_FWD_MINBLOCKS
#define DSA3D_FWD_MINBLOCKS 3
#endif

// fp32 storage, and bf16 where launch_forward keeps it: a group of lanes per item.
template <typename T, int D, bool kAdd>
__global__ void __launch_bounds__(256, DSA3D_FWD_MINBLOCKS)
forward_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
               const float* __restrict__ offsets, const T* addend, T* out, float* __restrict__ lse,
               const Problem pr, const int* __restrict__ gate) {
    if (gate && *gate == 0) return;                      // another kernel takes this call (see launch_forward)
    using E = Elt<T, 1>;
    using Row = typename E::Row;
    constexpr int VEC = E::VEC;
    constexpr int LPR = D / VEC;
    const int lane = threadIdx.x & 31;
    const int gl = lane & (LPR - 1);
    constexpr unsigned gmask = kFullMask;
    long long item = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) / LPR;
    const long long warp_first = (static_cast<long long>(blockIdx.x) * blockDim.x + (threadIdx.x & ~31)) / LPR;
    if (warp_first >= pr.items) return;                  // whole warp past the end
    const bool active = item < pr.items;                 // a trailing group repeats the last item, stores off
    if (!active) item = pr.items - 1;

    const int m = static_cast<int>(item / pr.q_count);
    const long long n = pr.q_begin + (item - static_cast<long long>(m) * pr.q_count);
    const int x = static_cast<int>(n % pr.W);
    const int y = static_cast<int>((n / pr.W) % pr.H);
    const int t = static_cast<int>(n / (static_cast<long long>(pr.W) * pr.H));
    const long long row = (n * pr.heads + m);               // row index into [N*heads, ...]
    const int ch = gl * VEC;
    const long long tok_stride = static_cast<long long>(pr.heads) * D;
    const long long sx = tok_stride;                         // element stride between x neighbours
    const long long sy = static_cast<long long>(pr.W) * sx;      // 64-bit once, so that the pointer
    const long long st = static_cast<long long>(pr.H) * sy;      // arithmetic below needs no widening                                // < 2^31: checked by the host

    const Row qr = E::load(q + row * D + ch);
    const float lscale = rsqrtf(static_cast<float>(D)) * kLog2e;    // logits in log2 units
    const float* off_row = offsets + row * pr.P * 3;
    const T* kh = k + static_cast<long long>(m) * D + ch;    // + tok * heads * D
    const long long v_minus_k = v - k;                       // same layout: V row = K row + this
    [[maybe_unused]] const long long kv_extent = pr.N * pr.heads * D;      // elements of K (= of V): checked build

    float acc[VEC];
#pragma unroll
    for (int j = 0; j < VEC; ++j) acc[j] = 0.0f;
    float m_run = -INFINITY, l_run = 0.0f;

    for (int pb = 0; pb < pr.P; pb += LPR) {
        Sample mine;
        mine.base = 0; mine.mask = 0u; mine.ft = mine.fy = mine.fx = 0.0f;
        if (pb + gl < pr.P)
            mine = to_sample(pr, make_cell(pr, t, y, x, pb + gl, offsets ? off_row + (pb + gl) * 3 : kZeroOffset));
        const int cnt = min(LPR, pr.P - pb);
        if constexpr (LPR >= 8) {
            // Fixed-window regime: every sample of this chunk (in every group of the warp) sits
            // exactly on a grid position, so it needs one K row and one V row.  Eight samples
            // are then taken together - 16 loads in flight instead of 2 - and their eight
            // logits leave one transposed reduction.
            const bool lattice = pb + gl >= pr.P || (mine.ft == 0.0f && mine.fy == 0.0f && mine.fx == 0.0f);
            if (__all_sync(kFullMask, lattice)) {
                for (int jb = 0; jb < cnt; jb += 8) {
                    Row kk[8], vv[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int base = __shfl_sync(gmask, mine.base, jb + i, LPR);
                        const unsigned mk = __shfl_sync(gmask, mine.mask, jb + i, LPR);
                        kk[i] = E::zero();
                        vv[i] = E::zero();
                        if ((mk & 1u) && jb + i < cnt) {            // corner (0,0,0) inside the grid
                            const T* pk = kh + base * tok_stride;
                            if (DSA3D_IN_RANGE(pr, pk - k, kv_extent, 1)) {
                                kk[i] = E::load(pk);
                                vv[i] = E::load(pk + v_minus_k);
                            }
                        }
                    }
                    float dd[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) dd[i] = E::dot(qr, kk[i], 0.0f);
                    group_reduce8<LPR>(dd, gl, gmask);
                    float sp[8], mx = -INFINITY;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        sp[i] = __shfl_sync(gmask, dd[0], reduce8_lane<LPR>(i), LPR) * lscale;
                        if (jb + i >= cnt) sp[i] = -INFINITY;       // no such sample
                        mx = fmaxf(mx, sp[i]);
                    }
                    if (mx > m_run + 8.0f) {
                        const float corr = exp2f(m_run - mx);
                        l_run *= corr;
#pragma unroll
                        for (int e = 0; e < VEC; ++e) acc[e] *= corr;
                        m_run = mx;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float pe = exp2f(sp[i] - m_run);
                        l_run += pe;
                        E::axpy(pe, vv[i], acc);
                    }
                }
                continue;
            }
        }
        for (int j = 0; j < cnt; ++j) {
            const Sample s = group_bcast<LPR>(mine, j, gmask);
            const float wt[2] = {1.0f - s.ft, s.ft}, wy[2] = {1.0f - s.fy, s.fy}, wx[2] = {1.0f - s.fx, s.fx};
            float w[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) w[c] = wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1];
            // corner row pointers: (ct, cy) pairs, the cx = 1 row is one token further
            const T* kp4[4];
            kp4[0] = kh + s.base * tok_stride;
            kp4[1] = kp4[0] + sy;
            kp4[2] = kp4[0] + st;
            kp4[3] = kp4[2] + sy;
            const bool full = s.mask == 0xffu && s.ft != 0.0f && s.fy != 0.0f && s.fx != 0.0f;
            float sdot = 0.0f;
            Row vv[8];
            if (full) {
                Row kk[8];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    kk[c] = DSA3D_IN_RANGE(pr, kp4[c >> 1] + (c & 1) * sx - k, kv_extent, 2) ? E::load(kp4[c >> 1] + (c & 1) * sx) : E::zero();
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    vv[c] = DSA3D_IN_RANGE(pr, kp4[c >> 1] + (c & 1) * sx - k, kv_extent, 2) ? E::load(kp4[c >> 1] + (c & 1) * sx + v_minus_k) : E::zero();
#pragma unroll
                for (int c = 0; c < 8; ++c) sdot = fmaf(w[c], E::dot(qr, kk[c], 0.0f), sdot);
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    vv[c] = E::zero();
                    if (((s.mask >> c) & 1u) && w[c] != 0.0f && DSA3D_IN_RANGE(pr, kp4[c >> 1] + (c & 1) * sx - k, kv_extent, 3)) {
                        const T* pk = kp4[c >> 1] + (c & 1) * sx;
                        const Row kk = E::load(pk);
                        vv[c] = E::load(pk + v_minus_k);
                        sdot = fmaf(w[c], E::dot(qr, kk, 0.0f), sdot);
                    } else {
                        w[c] = 0.0f;
                    }
                }
            }
            const float sp = group_sum<LPR>(sdot, gmask) * lscale;
            // Online softmax with a lazily updated reference: the running maximum m_run only
            // moves when a logit exceeds it by more than 8 (log2 units), so exp2(sp - m_run)
            // stays below 256 and the accumulators are rescaled only a few times per query.
            if (sp > m_run + 8.0f) {
                const float corr = exp2f(m_run - sp);
                l_run *= corr;
#pragma unroll
                for (int e = 0; e < VEC; ++e) acc[e] *= corr;
                m_run = sp;
            }
            const float pe = exp2f(sp - m_run);
            l_run += pe;
#pragma unroll
            for (int c = 0; c < 8; ++c) E::axpy(pe * w[c], vv[c], acc);
        }
    }
    const float inv = 1.0f / l_run;
#pragma unroll
    for (int e = 0; e < VEC; ++e) acc[e] *= inv;
    if (active) {
        if constexpr (kAdd) {                            // first term of Eq. 1, added before the rounding
            float add[VEC];
            E::to_float(E::load(addend + row * D + ch), add);
#pragma unroll
            for (int e = 0; e < VEC; ++e) acc[e] += add[e];
        }
        E::store(out + row * D + ch, acc);
        if (gl == 0) lse[row] = (m_run + log2f(l_run)) * kLn2;
    }
}

// fp32 calls of few tokens (by_classes): the samples of an item in four classes of consecutive ones, each with sums of its own that are folded
// into the whole in order.  What bounds such a call by rows is the chain of one item, a gather and an update of the running maximum per
// sample; with a group of lanes per class (G = 4) it is a quarter as deep.  Calls with more items than that has lanes for walk the
// classes one after the other (G = 1): the same sums in the same order, whichever of the two paths below a warp takes, so that the bits of
// a head do not depend on how many heads the call has.  120 registers: with 96 or 80 the rows are no longer all asked for
// at once (window (3,3,3), 64 heads: 52 -> 62 and 89 us).  Figures: class_groups.
constexpr int kClasses = 4, kClassThreads = 128;
template <int D, bool kAdd, int G>
__global__ void __launch_bounds__(kClassThreads, 4)
forward_classes_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v, const float* __restrict__ offsets,
                       const float* addend, float* out, float* __restrict__ lse, const __grid_constant__ Problem pr) {
    using E = Elt<float, 1>;
    using Row = typename E::Row;
    constexpr int LPR = D / 4, ITEMS = kClassThreads / (G * LPR);
    const int gl = threadIdx.x % LPR, group = threadIdx.x / LPR;
    long long item = static_cast<long long>(blockIdx.x) * ITEMS + group / G;
    const bool active = item < pr.items;                 // trailing groups repeat the last item, stores off
    if (!active) item = pr.items - 1;
    const int m = static_cast<int>(item / pr.q_count), n = static_cast<int>(pr.q_begin + (item - m * pr.q_count));
    const int x = n % pr.W, ty = n / pr.W, y = ty % pr.H, t = ty / pr.H;
    const long long row = static_cast<long long>(n) * pr.heads + m;
    const long long tok = static_cast<long long>(pr.heads) * D, sy = pr.W * tok, st = pr.H * sy;
    const Row qr = E::load(q + row * D + gl * 4);
    const float* kh = k + static_cast<long long>(m) * D + gl * 4;
    const long long v_minus_k = v - k;
    [[maybe_unused]] const long long kv_extent = pr.N * pr.heads * D;
    const float lscale = rsqrtf(static_cast<float>(D)) * kLog2e;        // logits in log2 units
    // with a q that is not finite a sample without a row has the logit 0 all the same: not by the products below that take eight at once
    const bool finite = fabsf(qr.v[0] + qr.v[1] + qr.v[2] + qr.v[3]) < INFINITY;
    int size = (pr.P + kClasses - 1) / kClasses;
    if (pr.P > 16) size = (size + 7) & ~7;               // so that eight samples on the grid belong to one class
    const int span = G == 1 ? pr.P : size, begin = G == 1 ? 0 : group % G * size;
    float total[4] = {0.0f, 0.0f, 0.0f, 0.0f}, m_all = -INFINITY, l_all = 0.0f;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, m_run = -INFINITY, l_run = 0.0f;       // of the class
    auto fold = [&](const float (&a)[4], float m_part, float l_part) {
        const float mx = fmaxf(m_all, m_part), f = m_all == mx ? 1.0f : exp2f(m_all - mx), g = m_part == mx ? 1.0f : exp2f(m_part - mx);
        l_all = fmaf(l_part, g, __fmul_rn(l_all, f));
#pragma unroll
        for (int e = 0; e < 4; ++e) total[e] = fmaf(a[e], g, __fmul_rn(total[e], f));
        m_all = mx;
    };
    int left = size;                                     // samples of the class still to come (G = 1)
    auto next_class = [&](int taken) {
        if (left == 0) {
            fold(acc, m_run, l_run);
            acc[0] = acc[1] = acc[2] = acc[3] = l_run = 0.0f;
            m_run = -INFINITY;
            left = size;
        }
        left -= taken;
    };
    // the next sample's logit: its weight beside the sums so far
    auto weight = [&](float sp) {
        if (sp > m_run + 8.0f) {
            const float corr = exp2f(m_run - sp);
            l_run *= corr;
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] *= corr;
            m_run = sp;
        }
        const float pe = sp == -INFINITY ? 0.0f : exp2f(sp - m_run);
        l_run = __fadd_rn(l_run, pe);
        return pe;
    };
    for (int i0 = 0; i0 < span; i0 += LPR) {
        const int p0 = begin + i0, cnt = min(LPR, span - i0);           // (the last class may end before its samples do: no logit)
        Sample mine;
        mine.base = 0; mine.mask = 0u; mine.ft = mine.fy = mine.fx = 0.0f;
        if (gl < cnt && p0 + gl < pr.P) mine = to_sample(pr, make_cell(pr, t, y, x, p0 + gl, offsets ? offsets + (row * pr.P + p0 + gl) * 3 : kZeroOffset));
        if (__all_sync(kFullMask, finite && mine.ft == 0.0f && mine.fy == 0.0f && mine.fx == 0.0f)) {     // on the grid: a row each, eight samples at a time
            for (int jb = 0; jb < cnt; jb += 8) {
                Row kk[8], vv[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int base = __shfl_sync(kFullMask, mine.base, jb + i, LPR);
                    const unsigned mask = __shfl_sync(kFullMask, mine.mask, jb + i, LPR);
                    kk[i] = vv[i] = E::zero();
                    const float* pk = kh + base * tok;
                    if ((mask & 1u) && jb + i < cnt && DSA3D_IN_RANGE(pr, pk - k, kv_extent, 1)) {
                        kk[i] = E::load(pk);
                        vv[i] = E::load(pk + v_minus_k);
                    }
                }
                float dd[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) dd[i] = E::dot(qr, kk[i], 0.0f);
                group_reduce8<LPR>(dd, gl, kFullMask);
                float sp[8], mx = -INFINITY;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    sp[i] = __shfl_sync(kFullMask, dd[0], reduce8_lane<LPR>(i), LPR) * lscale;
                    if (jb + i >= cnt || p0 + jb + i >= pr.P) sp[i] = -INFINITY;
                    mx = fmaxf(mx, sp[i]);
                }
                const bool aligned = G != 1 || size % 8 == 0;
                if (G == 1 && aligned) next_class(8);
                // the first sample of a class sets the maximum; as a rule none of the eight moves it again
                const float first = aligned && m_run == -INFINITY && sp[0] > m_run ? sp[0] : m_run;
                if (__all_sync(kFullMask, aligned && first > -INFINITY && mx <= first + 8.0f)) {
                    m_run = first;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float pe = exp2f(sp[i] - m_run);
                        l_run = __fadd_rn(l_run, pe);
                        E::axpy(pe, vv[i], acc);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        if (jb + i >= cnt) continue;
                        if (G == 1 && !aligned) next_class(1);
                        E::axpy(weight(sp[i]), vv[i], acc);
                    }
                }
            }
            continue;
        }
        for (int j = 0; j < cnt; ++j) {
            const Sample s = group_bcast<LPR>(mine, j, kFullMask);
            const float wt[2] = {1.0f - s.ft, s.ft}, wy[2] = {1.0f - s.fy, s.fy}, wx[2] = {1.0f - s.fx, s.fx};
            const float* at = kh + s.base * tok;
            float w[8], sdot = 0.0f;
            Row kk[8], vv[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                w[c] = wt[c >> 2] * wy[(c >> 1) & 1] * wx[c & 1];
                kk[c] = vv[c] = E::zero();
                const float* pk = at + (c >> 2) * st + ((c >> 1) & 1) * sy + (c & 1) * tok;
                if (((s.mask >> c) & 1u) && w[c] != 0.0f && DSA3D_IN_RANGE(pr, pk - k, kv_extent, 3)) {
                    kk[c] = E::load(pk);
                    vv[c] = E::load(pk + v_minus_k);
                } else {
                    w[c] = 0.0f;
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (w[c] != 0.0f) sdot = fmaf(w[c], E::dot(qr, kk[c], 0.0f), sdot);
            const float sp = group_sum<LPR>(sdot, kFullMask) * lscale;
            if (G == 1) next_class(1);
            const float pe = weight(p0 + j < pr.P ? sp : -INFINITY);
#pragma unroll
            for (int c = 0; c < 8; ++c) E::axpy(pe * w[c], vv[c], acc);
        }
    }
    if constexpr (G == 1) {
        fold(acc, m_run, l_run);
    } else {
        __shared__ float4 part[ITEMS][kClasses][LPR];
        __shared__ float2 stat[ITEMS][kClasses];
        part[group / G][group % G][gl] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        if (gl == 0) stat[group / G][group % G] = make_float2(m_run, l_run);
        __syncthreads();
        if (group % G != 0) return;
#pragma unroll
        for (int c = 0; c < kClasses; ++c) {
            const float4 a = part[group / G][c][gl];
            const float2 s = stat[group / G][c];
            fold({a.x, a.y, a.z, a.w}, s.x, s.y);
        }
    }
    if (!active) return;
    const float inv = 1.0f / l_all;
#pragma unroll
    for (int e = 0; e < 4; ++e) total[e] = __fmul_rn(total[e], inv);
    if constexpr (kAdd) {
        float add[4];
        E::to_float(E::load(addend + row * D + gl * 4), add);
#pragma unroll
        for (int e = 0; e < 4; ++e) total[e] = __fadd_rn(total[e], add[e]);
    }
    E::store(out + row * D + gl * 4, total);
    if (gl == 0) lse[row] = (m_all + log2f(l_all)) * kLn2;
}

template <int D, bool kAdd, int G>
static cudaError_t launch_forward_classes(const void* q, const void* k, const void* v, const float* offsets, const void* addend, void* out, float* lse, const Problem& pr, cudaStream_t stream) {
    constexpr int items = kClassThreads / (G * (D / 4));
    forward_classes_kernel<D, kAdd, G><<<static_cast<unsigned>((pr.items + items - 1) / items), kClassThreads, 0, stream>>>(
        static_cast<const float*>(q), static_cast<const float*>(k), static_cast<const float*>(v), offsets, static_cast<const float*>(addend), static_cast<float*>(out), lse, pr);
    return cudaGetLastError();
}

template <int D>
static cudaError_t launch_gather_forward(const void* q, const void* k, const void* v, const float* offsets, const void* addend, void* out,
                                         float* lse, const Problem& pr, cudaStream_t stream, const int* gate) {
    using T = __nv_bfloat16;
    // as many items per warp as have a lane for every sample
    const int share = pr.P <= 8 ? 4 : pr.P <= 16 ? 2 : 1;
    const long long per_head = (pr.q_count + kFwdWarps * share - 1) / (kFwdWarps * share);
    // behind a gate that is mostly closed, a CTA per two items would cost more to launch than to run (0.95 ms for 3.7 M items)
    const long long all = per_head * pr.heads;
    const unsigned blocks = static_cast<unsigned>(gate && share == 1 && all > 148 * 16 ? 148 * 16 : all);
    if (share > 1) {
        auto kern = share == 4 ? (addend ? gather_forward_small_kernel<D, 4, true> : gather_forward_small_kernel<D, 4, false>)
                               : (addend ? gather_forward_small_kernel<D, 2, true> : gather_forward_small_kernel<D, 2, false>);
        kern<<<blocks, kFwdWarps * 32, 0, stream>>>(static_cast<const T*>(q), static_cast<const T*>(k), static_cast<const T*>(v), offsets,
                                                    static_cast<const T*>(addend), static_cast<T*>(out), lse, pr, static_cast<unsigned>(per_head), gate);
        return cudaGetLastError();
    }
    if (gate)
        gather_forward_kernel<D, false, true, false><<<blocks, kFwdWarps * 32, 0, stream>>>(
            static_cast<const T*>(q), static_cast<const T*>(k), static_cast<const T*>(v), offsets, nullptr, static_cast<T*>(out), lse, pr,
            static_cast<unsigned>(per_head), gate);
    else {
        auto kern = addend ? gather_forward_kernel<D, true, false, false> : gather_forward_kernel<D, false, false, false>;
        if constexpr (D > 32)                            // (32 channels come here with more samples only)
            if (pr.P <= 32) kern = addend ? gather_forward_kernel<D, true, false, true> : gather_forward_kernel<D, false, false, true>;
        kern<<<blocks, kFwdWarps * 32, 0, stream>>>(static_cast<const T*>(q), static_cast<const T*>(k), static_cast<const T*>(v), offsets, static_cast<const T*>(addend),
                                                    static_cast<T*>(out), lse, pr, static_cast<unsigned>(per_head), gate);
    }
    return cudaGetLastError();
}

template <typename T, int D>
static cudaError_t launch_forward_t(const void* q, const void* k, const void* v, const float* offsets,
                                    const void* addend, void* out, float* lse, const Problem& pr,
                                    cudaStream_t stream, const int* gate) {
    constexpr int LPR = D / Elt<T, 1>::VEC;
    constexpr int threads = 256;
    if constexpr (std::is_same<T, float>::value) {
        if (!gate && by_classes(pr)) {
            if (class_groups(pr) == 1) return addend ? launch_forward_classes<D, true, 1>(q, k, v, offsets, addend, out, lse, pr, stream) : launch_forward_classes<D, false, 1>(q, k, v, offsets, addend, out, lse, pr, stream);
            return addend ? launch_forward_classes<D, true, kClasses>(q, k, v, offsets, addend, out, lse, pr, stream) : launch_forward_classes<D, false, kClasses>(q, k, v, offsets, addend, out, lse, pr, stream);
        }
    }
    const long long groups_per_block = threads / LPR;
    const long long blocks = (pr.items + groups_per_block - 1) / groups_per_block;
    if (addend)
        forward_kernel<T, D, true><<<static_cast<unsigned>(blocks), threads, 0, stream>>>(
            static_cast<const T*>(q), static_cast<const T*>(k), static_cast<const T*>(v), offsets,
            static_cast<const T*>(addend), static_cast<T*>(out), lse, pr, gate);
    else
        forward_kernel<T, D, false><<<static_cast<unsigned>(blocks), threads, 0, stream>>>(
            static_cast<const T*>(q), static_cast<const T*>(k), static_cast<const T*>(v), offsets, nullptr,
            static_cast<T*>(out), lse, pr, gate);
    return cudaGetLastError();
}

// Calls from this many samples on last long enough for the card's power limit to set the clock.
constexpr long long kPowerLimitedSamples = 300000000;

cudaError_t launch_forward(const void* q, const void* k, const void* v, const float* offsets, const void* addend,
                           void* out, float* lse, const Problem& pr, bool bf16, cudaStream_t stream, const int* gate) {
    // Which bf16 calls a warp per item serves, and which the rows of forward_kernel (time by rows over time by a warp per item):
    // 32 channels, up to 32 samples: the row traffic is too small to pay for the list (0.94 - 0.97); more samples 1.9 - 2.9.
    // 64 channels, window (3,3,3): 1.14 - 1.36 on 8 x 45 x 80, 16 heads, 1.03 - 1.14 on 16 x 68 x 120, 32 heads, 0.97 - 1.03 on
    // 64 x 68 x 120, the larger the offsets the more; integer offsets 1.03 - 0.85.
    // 128 channels: window (2,2,2) 1.4, (3,3,3) 1.03 - 1.17 on 32 x 45 x 80, 16 heads, at the full clock, before the
    // instance of one round that is 2 - 8 % faster.  But it draws more power, and
    // in calls of 0.1 s and more the clock follows: forward of 128 x 68 x 120, 16 heads, by rows 98, 105 and 116 ms for offsets N(0, 0.5),
    // N(0, 2) and N(0, 3), by a warp per item 105, 102 and 111 (training steps 1.03, 0.993 and 0.98 of those by rows), so windows of 17 to 32
    // samples go by rows from kPowerLimitedSamples on.  More samples 1.0 - 1.9 (147: 9.8 against 18.5 ms).
    switch (bf16 ? pr.d : -pr.d) {
        case 32:
            return pr.P <= 32 ? launch_forward_t<__nv_bfloat16, 32>(q, k, v, offsets, addend, out, lse, pr, stream, gate)
                              : launch_gather_forward<32>(q, k, v, offsets, addend, out, lse, pr, stream, gate);
        case 64: return launch_gather_forward<64>(q, k, v, offsets, addend, out, lse, pr, stream, gate);
        case 128:
            return pr.P > 16 && pr.P <= 32 && pr.items * pr.P >= kPowerLimitedSamples && !gate
                       ? launch_forward_t<__nv_bfloat16, 128>(q, k, v, offsets, addend, out, lse, pr, stream, gate)
                       : launch_gather_forward<128>(q, k, v, offsets, addend, out, lse, pr, stream, gate);
        case -32: return launch_forward_t<float, 32>(q, k, v, offsets, addend, out, lse, pr, stream, gate);
        case -64: return launch_forward_t<float, 64>(q, k, v, offsets, addend, out, lse, pr, stream, gate);
        case -128: return launch_forward_t<float, 128>(q, k, v, offsets, addend, out, lse, pr, stream, gate);
    }
    return cudaErrorInvalidValue;
}

}  // namespace dsa3d
