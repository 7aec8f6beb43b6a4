// Shared device helpers of the 3D-DSA kernels: problem description, element access for
// fp32 / bf16 storage, sample geometry (Formulation: position = token coordinate + window
// displacement + learned offset; trilinear corners with zero padding) and group shuffles.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dsa3d {

// One contribution to dK/dV as the tile kernel bins it: byte offset of the query's q/dO row
// pair in shared memory and the two coefficients (w_c * ck_p, w_c * cv_p).
using TileEntry = uint4;            // {offset, fp32 wk, fp32 wv, unused}

struct Problem {
    int T, H, W, heads, d;
    int kt, kh, kw, P;
    // ceil(2^20 / kw) and ceil(2^20 / kh): p / kw = (p * inv_kw) >> 20 exactly for p < 2^8 (P <= 256), so that
    // a sample's window cell needs no integer division
    unsigned inv_kw, inv_kh;
    long long N;       // T*H*W
    long long items;   // work items of this launch: one per (query token, head) = q_count*heads
    // Query tokens [q_begin, q_begin + q_count) are processed (the whole grid unless a caller
    // works through the video in slabs of frames); K and V always cover the whole grid.
    long long q_begin, q_count;
    // Query tiling of the backward scatter (tile_t < 1: no tiling, every dK/dV contribution
    // goes straight to the global accumulators).  A corner is "in the halo" of a query when
    // it lies within `halo` grid cells of the query's tile on every axis.
    int tile_t, tile_y, tile_x, halo;
    int tiles_t, tiles_y, tiles_x;
    int tt_begin, tt_count;   // tile rows along t that the tile kernel visits (all: 0, tiles_t)
    // Checked build (-DDSA3D_DEBUG) only: device word that receives the first out-of-range index a
    // kernel was about to use (0 = none); NULL otherwise.
    unsigned long long* debug_word;
    // Backward behind a check of the offsets (dsa3d_backward_bounded_offsets): the general kernels run only
    // if this device word is non-zero (the check found offsets its tile kernels do not cover); NULL: always.
    const int* gate;
};

// The start of a kernel launched by launch_gated: true when it has nothing to do.  Its CTAs may be put in place while the
// kernel before it still runs; they wait here until that has completed and its memory is visible.  Of a chain of kernels that
// find their gate closed only 1 of 4 us each is left.  (When it is open the next kernel is not let in early: its waiting
// CTAs cost the running one 9 %.)  The gate is final long before: ordinary launches lie between the check that writes it
// and the chain.  Nothing else is read before the wait, and the loads behind it stand behind the branch on the gate.
__device__ __forceinline__ bool gated_off_early(const int* gate) {
    const bool off = *reinterpret_cast<const volatile int*>(gate) == 0;
    if (off) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return off;
}
template <typename... P, typename... A>
cudaError_t launch_gated(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, const A&... args) {
    cudaLaunchAttribute early;
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config = {};
    config.gridDim = grid; config.blockDim = dim3(threads); config.dynamicSmemBytes = smem; config.stream = stream;
    config.attrs = &early; config.numAttrs = 1;
    return cudaLaunchKernelEx(&config, kern, static_cast<P>(args)...);
}

// True when a gated general kernel has nothing to do (see Problem::gate).
__device__ __forceinline__ bool gated_off(const Problem& pr) { return pr.gate != nullptr && *pr.gate == 0; }

// Checked build: every row a gather reads and every row or bin a scatter writes is tested against its
// tensor's extent first; a violation is recorded (first one wins: code in the top 8 bits, the offending
// element offset in the rest) and the access is skipped - nothing traps.  In the normal build the
// tests compile to `true`.
#ifdef DSA3D_DEBUG
__device__ __forceinline__ bool debug_in_range(const Problem& pr, long long offset, long long extent, int code) {
    if (offset >= 0 && offset < extent) return true;
    if (pr.debug_word)
        atomicCAS(pr.debug_word, 0ull, (static_cast<unsigned long long>(code) << 56) |
                                           (static_cast<unsigned long long>(offset) & ((1ull << 56) - 1)));
    return false;
}
#define DSA3D_IN_RANGE(pr, offset, extent, code) dsa3d::debug_in_range((pr), (offset), (extent), (code))
#else
#define DSA3D_IN_RANGE(pr, offset, extent, code) true
#endif

// ---------------------------------------------------------------------------------------
// Element access.  A lane handles NV consecutive 16-byte vectors of a row (8 bf16 or 4 fp32
// channels each).
// `Row` keeps that vector in its storage form.  For bf16 the dot products (both factors
// bf16) use the sm_100 mixed-precision instruction fma.rn.f32.bf16 (exact fp32 product,
// fp32 accumulate), which needs no unpacking; `axpy` (fp32 coefficient) widens the row.
// ---------------------------------------------------------------------------------------
// Two independent fp32 FMAs in one instruction (sm_100 fma.rn.f32x2): a0 += x0*y0, a1 += x1*y1,
// each rounded exactly as fmaf would.  Pays where a loop is bound by issue slots and most of its
// instructions are FMAs.
__device__ __forceinline__ void fma2(float& a0, float& a1, float x0, float x1, float y0, float y1) {
    unsigned long long acc, x, y;
    asm("mov.b64 %0, {%1, %2};" : "=l"(acc) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(x0), "f"(x1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(y0), "f"(y1));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(x), "l"(y));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a0), "=f"(a1) : "l"(acc));
}

// The 128-channel backward gather (two 16-byte vectors per lane) uses the packed FMA in its row
// scalings (2.9 % faster); the forward and the narrower kernels measured no gain and keep fmaf.
constexpr bool kPackedAxpy = true;

template <typename T, int NV> struct Elt;       // NV = 16-byte vectors per lane (1 or 2)

template <int NV> struct Elt<float, NV> {
    static constexpr int VEC = 4 * NV;
    struct Row { float v[VEC]; };
    static __device__ __forceinline__ Row load(const float* p) {
        Row r;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p) + i);
            r.v[4 * i] = x.x; r.v[4 * i + 1] = x.y; r.v[4 * i + 2] = x.z; r.v[4 * i + 3] = x.w;
        }
        return r;
    }
    static __device__ __forceinline__ Row zero() {
        Row r;
#pragma unroll
        for (int e = 0; e < VEC; ++e) r.v[e] = 0.0f;
        return r;
    }
    static __device__ __forceinline__ float dot(const Row& a, const Row& b, float acc) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc = fmaf(a.v[e], b.v[e], acc);
        return acc;
    }
    static __device__ __forceinline__ void axpy(float c, const Row& x, float (&acc)[VEC]) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc[e] = fmaf(c, x.v[e], acc[e]);
    }
    static __device__ __forceinline__ void axpy_paired(float c, const Row& x, float (&acc)[VEC]) { axpy(c, x, acc); }
    static __device__ __forceinline__ void to_float(const Row& x, float (&f)[VEC]) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) f[e] = x.v[e];
    }
    static __device__ __forceinline__ void store(float* p, const float (&x)[VEC]) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
            reinterpret_cast<float4*>(p)[i] = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
    }
};

__device__ __forceinline__ float fma_bf16(unsigned short a, unsigned short b, float c) {
    float d;
    asm("fma.rn.f32.bf16 %0, %1, %2, %3;" : "=f"(d) : "h"(a), "h"(b), "f"(c));
    return d;
}

__device__ __forceinline__ void split_b32(uint32_t r, unsigned short& lo, unsigned short& hi) {
    asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(r));
}

template <int NV> struct Elt<__nv_bfloat16, NV> {
    static constexpr int VEC = 8 * NV;
    static constexpr int NW = 4 * NV;            // 32-bit words per lane
    struct Row { uint32_t w[NW]; };
    static __device__ __forceinline__ Row load(const __nv_bfloat16* p) {
        Row r;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const uint4 x = __ldg(reinterpret_cast<const uint4*>(p) + i);
            r.w[4 * i] = x.x; r.w[4 * i + 1] = x.y; r.w[4 * i + 2] = x.z; r.w[4 * i + 3] = x.w;
        }
        return r;
    }
    static __device__ __forceinline__ Row zero() {
        Row r;
#pragma unroll
        for (int i = 0; i < NW; ++i) r.w[i] = 0u;
        return r;
    }
    static __device__ __forceinline__ float dot(const Row& a, const Row& b, float acc) {
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            unsigned short al, ah, bl, bh;
            split_b32(a.w[i], al, ah);
            split_b32(b.w[i], bl, bh);
            acc = fma_bf16(al, bl, acc);
            acc = fma_bf16(ah, bh, acc);
        }
        return acc;
    }
    // acc += c * x with an fp32 coefficient: the bf16 values are widened (one shift or mask
    // each) and multiplied in fp32, so the coefficient keeps all its bits.  (Rounding the
    // coefficient to bf16 and using the mixed instruction was measured 12 % faster overall, but
    // its error reaches the 2e-2 bound on rare elements of very large tensors.)
    static __device__ __forceinline__ void axpy(float c, const Row& x, float (&acc)[VEC]) {
        if constexpr (NV == 2 && kPackedAxpy) {
#pragma unroll
            for (int i = 0; i < NW; ++i)
                fma2(acc[2 * i], acc[2 * i + 1], c, c, __uint_as_float(x.w[i] << 16), __uint_as_float(x.w[i] & 0xffff0000u));
        } else {
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                acc[2 * i] = fmaf(c, __uint_as_float(x.w[i] << 16), acc[2 * i]);
                acc[2 * i + 1] = fmaf(c, __uint_as_float(x.w[i] & 0xffff0000u), acc[2 * i + 1]);
            }
        }
    }
    // The same with two FMAs per instruction whatever the lane width (for loops that are bound by issue slots).
    static __device__ __forceinline__ void axpy_paired(float c, const Row& x, float (&acc)[VEC]) {
#pragma unroll
        for (int i = 0; i < NW; ++i)
            fma2(acc[2 * i], acc[2 * i + 1], c, c, __uint_as_float(x.w[i] << 16), __uint_as_float(x.w[i] & 0xffff0000u));
    }
    static __device__ __forceinline__ void to_float(const Row& x, float (&f)[VEC]) {
#pragma unroll
        for (int i = 0; i < NW; ++i) {          // bf16 is the upper half of an fp32
            f[2 * i] = __uint_as_float(x.w[i] << 16);
            f[2 * i + 1] = __uint_as_float(x.w[i] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, const float (&x)[VEC]) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(x[8 * i + 2 * j], x[8 * i + 2 * j + 1]);   // RNE
                w[j] = *reinterpret_cast<const uint32_t*>(&h);
            }
            reinterpret_cast<uint4*>(p)[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
};

// ---------------------------------------------------------------------------------------
// Sample geometry.  (it, iy, ix) is corner (0,0,0) of the cell (a component may be -1;
// only corners flagged in `mask` are ever dereferenced), bit c = ct*4 + cy*2 + cx of
// `mask` says corner c lies inside the grid, f* are the fractional parts.  A sample with a
// NaN position or one at < -1 or >= size on any axis has mask 0.  The position is
// float(coord + b) + offset with one fp32 rounding, then floorf, then the fp32 difference:
// the same sequence on every path so that the integer cell decision never depends on who
// computes it.
// ---------------------------------------------------------------------------------------
struct Cell {
    int it, iy, ix;
    unsigned mask;
    float ft, fy, fx;
};

// What a lane needs to process a sample somebody else located: linear index of corner
// (0,0,0), corner mask, fractional parts.
struct Sample {
    int base;
    unsigned mask;
    float ft, fy, fx;
};

__device__ __forceinline__ bool axis_cell(int coord_plus_b, float off, int size, int& i0, float& f) {
    const float pi = __fadd_rn(static_cast<float>(coord_plus_b), off);
    if (!(pi >= -1.0f) || !(pi < static_cast<float>(size))) return false;
    const float fl = floorf(pi);
    i0 = static_cast<int>(fl);
    f = __fsub_rn(pi, fl);
    return true;
}

// Bit c of the result is set when corner c = (ct, cy, cx) has lo <= i0 + c < hi on every axis,
// where the test per axis is written as an unsigned range check on (i0 - lo).
__device__ __forceinline__ unsigned corner_mask(int rt, int ry, int rx, int et, int ey, int ex) {
    const unsigned t0 = static_cast<unsigned>(rt) < static_cast<unsigned>(et);
    const unsigned t1 = static_cast<unsigned>(rt + 1) < static_cast<unsigned>(et);
    const unsigned y0 = static_cast<unsigned>(ry) < static_cast<unsigned>(ey);
    const unsigned y1 = static_cast<unsigned>(ry + 1) < static_cast<unsigned>(ey);
    const unsigned x0 = static_cast<unsigned>(rx) < static_cast<unsigned>(ex);
    const unsigned x1 = static_cast<unsigned>(rx + 1) < static_cast<unsigned>(ex);
    const unsigned yx = (y0 & x0) | ((y0 & x1) << 1) | ((y1 & x0) << 2) | ((y1 & x1) << 3);
    return (t0 ? yx : 0u) | (t1 ? (yx << 4) : 0u);
}

// The same from the three offset components already loaded.
__device__ __forceinline__ Cell make_cell_values(const Problem& pr, int t, int y, int x, int p, float ot, float oy,
                                                 float ox) {
    const int pk = static_cast<int>((static_cast<unsigned>(p) * pr.inv_kw) >> 20);      // p / kw
    const int w = p - pk * pr.kw;
    const int u = static_cast<int>((static_cast<unsigned>(pk) * pr.inv_kh) >> 20);     // p / (kw * kh)
    const int v = pk - u * pr.kh;
    Cell c;
    c.it = c.iy = c.ix = 0;
    c.mask = 0u;
    c.ft = c.fy = c.fx = 0.0f;
    int it, iy, ix;
    float ft, fy, fx;
    if (!axis_cell(t + u - pr.kt / 2, ot, pr.T, it, ft)) return c;
    if (!axis_cell(y + v - pr.kh / 2, oy, pr.H, iy, fy)) return c;
    if (!axis_cell(x + w - pr.kw / 2, ox, pr.W, ix, fx)) return c;
    c.it = it; c.iy = iy; c.ix = ix;
    c.ft = ft; c.fy = fy; c.fx = fx;
    c.mask = corner_mask(it, iy, ix, pr.T, pr.H, pr.W);
    return c;
}

__device__ __forceinline__ Cell make_cell(const Problem& pr, int t, int y, int x, int p,
                                          const float* __restrict__ off3) {
    const int pk = static_cast<int>((static_cast<unsigned>(p) * pr.inv_kw) >> 20);      // p / kw
    const int w = p - pk * pr.kw;
    const int u = static_cast<int>((static_cast<unsigned>(pk) * pr.inv_kh) >> 20);     // p / (kw * kh)
    const int v = pk - u * pr.kh;
    Cell c;
    c.it = c.iy = c.ix = 0;
    c.mask = 0u;
    c.ft = c.fy = c.fx = 0.0f;
    int it, iy, ix;
    float ft, fy, fx;
    const float ot = __ldg(off3), oy = __ldg(off3 + 1), ox = __ldg(off3 + 2);
    if (!axis_cell(t + u - pr.kt / 2, ot, pr.T, it, ft)) return c;
    if (!axis_cell(y + v - pr.kh / 2, oy, pr.H, iy, fy)) return c;
    if (!axis_cell(x + w - pr.kw / 2, ox, pr.W, ix, fx)) return c;
    c.it = it; c.iy = iy; c.ix = ix;
    c.ft = ft; c.fy = fy; c.fx = fx;
    c.mask = corner_mask(it, iy, ix, pr.T, pr.H, pr.W);
    return c;
}

__device__ __forceinline__ Sample to_sample(const Problem& pr, const Cell& c) {
    Sample s;
    s.base = (c.it * pr.H + c.iy) * pr.W + c.ix;
    s.mask = c.mask;
    s.ft = c.ft; s.fy = c.fy; s.fx = c.fx;
    return s;
}

// Corners of `c` that lie in the halo box of the tile containing query (t, y, x).
__device__ __forceinline__ unsigned halo_corner_mask(const Problem& pr, const Cell& c, int t, int y, int x) {
    if (pr.tile_t < 1) return 0u;
    const int lo_t = (t / pr.tile_t) * pr.tile_t - pr.halo;
    const int lo_y = (y / pr.tile_y) * pr.tile_y - pr.halo;
    const int lo_x = (x / pr.tile_x) * pr.tile_x - pr.halo;
    return corner_mask(c.it - lo_t, c.iy - lo_y, c.ix - lo_x, pr.tile_t + 2 * pr.halo,
                       pr.tile_y + 2 * pr.halo, pr.tile_x + 2 * pr.halo);
}

// Shuffles inside a group of LPR consecutive lanes (LPR a power of two <= 32).
template <int LPR> __device__ __forceinline__ unsigned group_mask(int lane) {
    if constexpr (LPR == 32) {
        return 0xffffffffu;
    } else {
        return ((1u << LPR) - 1u) << (lane & ~(LPR - 1));
    }
}

// All shuffles below name the full warp: the kernels keep every lane of a warp alive and
// on the same control path at each shuffle (a group past the end of the problem repeats
// the last item with its stores switched off), so no per-group mask is needed.
constexpr unsigned kFullMask = 0xffffffffu;

template <int LPR> __device__ __forceinline__ float group_sum(float v, unsigned gmask) {
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gmask, v, o, LPR);
    return v;
}

// Sum 8 per-lane numbers over the group so that every sum ends up on some lane, with a
// quarter of the shuffles a butterfly per value would take: at each of the first three
// xor distances a lane hands half of its values to its partner and keeps the other half.
// On return v[0] of lane gl holds the complete sum number reduce8_index<LPR>(gl).
// (LPR >= 8; narrower groups use group_sum.)
template <int LPR> __device__ __forceinline__ int reduce8_index(int gl) {
    return (((gl / (LPR / 2)) & 1) << 2) | (((gl / (LPR / 4)) & 1) << 1) | ((gl / (LPR / 8)) & 1);
}
template <int LPR> __device__ __forceinline__ int reduce8_lane(int index) {     // a lane holding sum `index`
    return ((index >> 2) & 1) * (LPR / 2) + ((index >> 1) & 1) * (LPR / 4) + (index & 1) * (LPR / 8);
}
template <int LPR> __device__ __forceinline__ void group_reduce8(float (&v)[8], int gl, unsigned gmask) {
    static_assert(LPR >= 8, "needs three halving steps");
    int n = 8;
#pragma unroll
    for (int d = LPR / 2; d >= LPR / 8; d >>= 1) {
        const bool upper = (gl & d) != 0;
        n >>= 1;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < n) {
                const float send = upper ? v[i] : v[i + n];
                const float keep = upper ? v[i + n] : v[i];
                v[i] = keep + __shfl_xor_sync(gmask, send, d, LPR);
            }
        }
    }
#pragma unroll
    for (int d = LPR / 16; d > 0; d >>= 1) v[0] += __shfl_xor_sync(gmask, v[0], d, LPR);
}

// Value and the three partial derivatives (along t, y, x) of the trilinear interpolant of
// eight corner numbers a[c], c = ct*4 + cy*2 + cx, at fractional position (ft, fy, fx):
// value = sum_c w_c a_c, d/da = sum_c (dw_c/da) a_c.  Corners outside the grid enter as 0.
__device__ __forceinline__ void trilerp_grad(const float (&a)[8], float ft, float fy, float fx, float& val,
                                             float& dt, float& dy, float& dx) {
    float L[4], X[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        X[i] = a[2 * i + 1] - a[2 * i];
        L[i] = fmaf(fx, X[i], a[2 * i]);
    }
    float M[2], Y[2], Xy[2];
#pragma unroll
    for (int ct = 0; ct < 2; ++ct) {
        Y[ct] = L[2 * ct + 1] - L[2 * ct];
        M[ct] = fmaf(fy, Y[ct], L[2 * ct]);
        Xy[ct] = fmaf(fy, X[2 * ct + 1] - X[2 * ct], X[2 * ct]);
    }
    dt = M[1] - M[0];
    val = fmaf(ft, dt, M[0]);
    dy = fmaf(ft, Y[1] - Y[0], Y[0]);
    dx = fmaf(ft, Xy[1] - Xy[0], Xy[0]);
}

template <int LPR> __device__ __forceinline__ Sample group_bcast(const Sample& s, int src, unsigned gmask) {
    Sample r;
    r.base = __shfl_sync(gmask, s.base, src, LPR);
    r.mask = __shfl_sync(gmask, s.mask, src, LPR);
    r.ft = __shfl_sync(gmask, s.ft, src, LPR);
    r.fy = __shfl_sync(gmask, s.fy, src, LPR);
    r.fx = __shfl_sync(gmask, s.fx, src, LPR);
    return r;
}

// One 16-byte fp32 reduction into global memory (the dK/dV accumulators).
__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

// Forward of fp32 calls: up to this many lanes of a head's tokens, d / 4 each, by classes of samples (forward_classes_kernel), whose sums are
// in another order than those of the rows: the line does not look at the heads, so that a shard of them gives the bits of the whole.
constexpr long long kClassLanes = 148 * 16;
__host__ __device__ inline bool by_classes(const Problem& pr) { return pr.N * (pr.d / 4) <= kClassLanes && pr.P > 1; }

// There: groups of lanes per item, one per class or one for all, the same bits.  Just below that line (256, 144 and 72 tokens of 32, 64 and 128
// channels), us by rows | four groups | one, N(0, 1) and integer offsets:
//     heads            2                    8                    16                   32                   64
//     32, (2,2,2)     9.2|3.7| 6.6         9.4| 5.2| 6.9        9.6| 8.6| 8.1       12.2|14.4|11.4       23.6|26.4|18.7
//         integer     3.4|3.1| 3.7         3.6| 4.2| 3.9        3.7| 6.3| 4.2        4.4|11.0| 4.8        7.1|20.0| 8.1
//     32, (3,3,3)    23.0|6.8|17.2        23.5|11.4|17.2       23.7|18.7|20.6       32.4|34.5|31.2       59.7|65.3|52.3
//         integer     7.5|3.4| 7.1         7.6| 4.4| 7.4        7.7| 7.0| 7.7        9.5|11.6| 9.7       16.4|21.0|16.5
//     32, (3,7,7)   101.4|23.7|75.4      100.2|44.8|75.6      101.3|75.4|94.8      148.1|144.5|152.2    277.5|280.0|256.1
//         integer    25.6|8.0|24.3        25.9|11.4|24.6       26.1|19.0|26.9       33.3|35.2|36.6       61.6|66.4|61.8
//     64, (3,3,3)    19.2|6.6|15.6        19.2|10.7|15.8       19.8|19.3|18.9       27.1|35.5|29.0       50.1|67.2|54.9
//         integer     6.4|3.3| 5.7         6.6| 4.2| 5.8        6.7| 6.9| 6.7        8.4|12.3| 8.9       14.5|22.3|15.8
//     128, (3,3,3)   17.2|7.4|14.7        17.0|10.6|15.0       17.3|19.1|17.7       24.4|35.3|27.6       44.8|66.1|51.8
//         integer     5.8|3.3| 5.6         5.9| 4.2| 5.5        5.9| 7.0| 6.3        7.8|12.1| 8.6       13.3|21.9|15.4
// (What is left slower than by rows: more than 16 heads, on integer offsets 2 - 15 %, 26 % for (2,2,2); real-valued ones of 64 and 128
// channels 7 - 14 %.)
__host__ __device__ inline int class_groups(const Problem& pr) {
    return pr.items * (pr.d / 4) <= 148ll * (pr.P <= 32 ? 128 : 256) ? 4 : 1;
}

// Backward of fp32 calls: up to this many lanes a CTA per item (backward_split_kernel), the same bits.  By rows | a CTA per item, as above:
//     heads            2                    8                    16
//     32, (2,2,2)    21.5| 7.7            22.2|15.6            23.0|25.5              integer  11.8| 6.9     12.2|13.5     12.3|21.8
//     32, (3,3,3)    55.6|12.5            56.4|27.0            57.8|45.4                       28.0| 8.7     28.7|19.8     29.0|34.1
//     32, (3,7,7)   281.3|35.8           307.8|93.7           348.8|180.0                     133.6|24.6    137.7|68.4    154.8|127.6
//     64, (3,3,3)    44.8|14.1            45.8|27.1            48.4|44.9                       25.5|11.1     25.8|21.4     26.2|36.6
//     64, (3,7,7)   235.0|44.8           243.5|104.7          271.2|176.1                     115.5|33.1    118.1|76.3    131.8|142.1
//     128, (3,3,3)   38.2|16.8            39.0|24.1            45.0|41.2                       21.9|14.2     22.4|18.6     22.6|31.1
//     128, (3,7,7)  154.2|51.2           155.3|92.7           176.2|168.5                      89.5|46.8     90.2|74.5     91.0|135.1
__host__ __device__ inline bool split_backward(const Problem& pr) {
    const int per_sm = pr.d == 128 ? 128 : pr.P > 64 ? 224 : pr.d == 64 ? 128 : pr.P > 16 ? 168 : 96;
    return pr.items * (pr.d / 4) <= 148ll * per_sm && pr.P > 1;
}

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

}  // namespace dsa3d
