// Dot products and weighted sums of gathered rows (bf16 storage), a warp per (token, head): the corner rows of a query's samples
// are listed in shared memory - only the corners inside the grid with a weight, so that border samples, dead samples and
// samples on grid positions cost what they need.
//
//   gather_dots   16 rows at a time on the tensor cores (m16n8k16: rows x channels as A, q as B).  Row g of a tile is read by
//                 lanes (g, 0 .. 3), 16 bytes each at a time, and odd rows take the 64-byte halves of every 128 bytes in the
//                 other order: rows start at the same bank, and the two rows a quarter-warp reads would meet in it
//                 (measured 8.0 data-pipe cycles per 512 bytes against 4.06).  B holds q in the order of the even rows
//                 in its even columns, in that of the odd rows in its odd ones.
//   gather_sum    D / 8 lanes per row, fp32 FMAs.  (As products - rows turned by movmatrix, weights as bf16 head and remainder - the
//                 same sums need fewer instructions but half as many data-pipe cycles again, which is what bounds: 14.8
//                 against 11.2 ms for the forward on 32 x 45 x 80, 16 heads of 128.)
#pragma once
#include "dsa3d_common.cuh"

namespace dsa3d {

constexpr int kGatherRows = 32 * 8;                // a round: 32 samples, a sample per lane

struct __align__(16) GatherList {
    uint32_t token[kGatherRows];
    float value[kGatherRows];                      // dot products, then weights
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The corners of a sample that have a weight.
__device__ __forceinline__ unsigned weighted_corners(unsigned mask, float ft, float fy, float fx) {
    if (ft == 0.0f) mask &= 0x0fu;
    if (fy == 0.0f) mask &= 0x33u;
    if (fx == 0.0f) mask &= 0x55u;
    return mask;
}

// Checked build: the corners of `mask` whose rows lie inside the tensor.
__device__ __forceinline__ unsigned checked_corners(const Problem& pr, unsigned mask, int base, [[maybe_unused]] int code) {
#ifdef DSA3D_DEBUG
    for (int c = 0; c < 8; ++c)
        if (((mask >> c) & 1u) && !DSA3D_IN_RANGE(pr, (base + (static_cast<long long>(c >> 2) * pr.H + ((c >> 1) & 1)) * pr.W + (c & 1)) * pr.heads * pr.d, pr.N * pr.heads * pr.d, code))
            mask &= ~(1u << c);
#endif
    return mask;
}

// A lane's part of the list.  `whole`: every sample of the warp has all eight corners or none, so a lane's entries are
// two aligned 16-byte pieces.  `single`: corner (0,0,0) alone or none (integer offsets), no scan and no loop over corners
// (window (2,2,2), 3.7 M items of 128 channels: forward 1.87 -> 1.74 ms, per query 1.53 -> 1.38; kSingle off where its
// registers cost the other offsets more, the forward at 128 channels, 2 %).
struct GatherPart { int first, total; unsigned mask; bool whole, single; };

// G items of 32 / G samples share a warp: item i has entries i * kGatherRows / G on.  Lists the corners `mask` of every lane's sample
// (corner (0,0,0) at linear index `base`), each item's padded to a multiple of `step` (<= 32 / G) with its last row;
// `total`: entries of the lane's item.
template <int G = 1, bool kSingle = true>
__device__ __forceinline__ GatherPart gather_list(GatherList& gl, unsigned mask, int base, const Problem& pr, int step) {
    constexpr int L = 32 / G;
    const int lane = threadIdx.x & 31, n = __popc(mask), sy = pr.W, st = pr.H * pr.W;
    const int lane0 = lane & ~(L - 1), region = (lane / L) * (kGatherRows / G);
    GatherPart part;
    part.mask = mask;
    part.whole = __all_sync(kFullMask, n == 8 || n == 0);
    part.single = kSingle && __all_sync(kFullMask, mask <= 1u);
    const unsigned have = (__ballot_sync(kFullMask, n > 0) >> lane0) & (L == 32 ? 0xffffffffu : (1u << L) - 1u);
    int last = 0;
    if (part.single) {
        part.first = region + __popc(have & ((1u << (lane - lane0)) - 1u));
        part.total = __popc(have);
        last = base;
        if (n) gl.token[part.first] = static_cast<uint32_t>(base);
    } else if (part.whole) {
        part.first = region + 8 * __popc(have & ((1u << (lane - lane0)) - 1u));
        part.total = 8 * __popc(have);
        last = base + st + sy + 1;
        if (n) {
            uint4* to = reinterpret_cast<uint4*>(gl.token + part.first);
            to[0] = make_uint4(base, base + 1, base + sy, base + sy + 1);
            to[1] = make_uint4(base + st, base + st + 1, base + st + sy, last);
        }
    } else {
        int incl = n;
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            const int up = __shfl_up_sync(kFullMask, incl, o, L);
            if (lane - lane0 >= o) incl += up;
        }
        part.total = __shfl_sync(kFullMask, incl, L - 1, L);
        part.first = region + incl - n;
        int at = part.first;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if ((mask >> c) & 1u) {
                last = base + (c >> 2) * st + ((c >> 1) & 1) * sy + (c & 1);
                gl.token[at++] = static_cast<uint32_t>(last);
            }
    }
    last = __shfl_sync(kFullMask, last, have ? 31 - __clz(static_cast<int>(have)) : 0, L);
    const int pad = part.total + lane - lane0;
    if (pad < (part.total + step - 1) / step * step) gl.token[region + pad] = static_cast<uint32_t>(last);
    return part;
}

// Sum of w[c] * value over the lane's entries; the lane's entries set to s * w[c], zero in the padding.
__device__ __forceinline__ float gather_combine(const GatherList& gl, const GatherPart& part, const float (&w)[8]) {
    float sum = 0.0f;
    if (part.single) {
        if (part.mask) sum = w[0] * gl.value[part.first];
    } else if (part.whole) {
        if (part.mask) {
            const float4 a = *reinterpret_cast<const float4*>(gl.value + part.first), b = *reinterpret_cast<const float4*>(gl.value + part.first + 4);
            sum = fmaf(w[7], b.w, fmaf(w[6], b.z, fmaf(w[5], b.y, fmaf(w[4], b.x, fmaf(w[3], a.w, fmaf(w[2], a.z, fmaf(w[1], a.y, w[0] * a.x)))))));
        }
    } else {
        int at = part.first;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if ((part.mask >> c) & 1u) sum = fmaf(w[c], gl.value[at++], sum);
    }
    return sum;
}
template <int G = 1>
__device__ __forceinline__ void gather_weights(GatherList& gl, const GatherPart& part, float s, const float (&w)[8], int step) {
    if (part.single) {
        if (part.mask) gl.value[part.first] = s * w[0];
    } else if (part.whole) {
        if (part.mask) {
            float4* to = reinterpret_cast<float4*>(gl.value + part.first);
            to[0] = make_float4(s * w[0], s * w[1], s * w[2], s * w[3]);
            to[1] = make_float4(s * w[4], s * w[5], s * w[6], s * w[7]);
        }
    } else {
        int at = part.first;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if ((part.mask >> c) & 1u) gl.value[at++] = s * w[c];
    }
    constexpr int L = 32 / G;
    const int lane = threadIdx.x & 31, pad = part.total + (lane & (L - 1));
    if (pad < (part.total + step - 1) / step * step) gl.value[(lane / L) * (kGatherRows / G) + pad] = 0.0f;
}

// 16 rows: those of entries s + g (a) and s + 8 + g (b).
template <int D> struct GatherRows { static constexpr int I = D / 32; uint4 a[I], b[I]; };
template <int D>
__device__ __forceinline__ void gather_load(GatherRows<D>& r, const GatherList& gl, int s, const char* src, uint32_t tok_bytes) {
    constexpr int I = GatherRows<D>::I;
    const int g = (threadIdx.x & 31) >> 2;
    const uint32_t odd = I > 1 ? (g & 1) * 64u : 0u;
    const char* pa = src + static_cast<uint64_t>(gl.token[s + g]) * tok_bytes + odd;
    const char* pb = src + static_cast<uint64_t>(gl.token[s + g + 8]) * tok_bytes + odd;
    const int other = I > 1 ? ((g & 1) ? -64 : 64) : 0;       // from the first to the second half of 128 bytes
#pragma unroll
    for (int i = 0; i < I; ++i) {
        r.a[i] = __ldg(reinterpret_cast<const uint4*>(pa + (i >> 1) * 128 + ((i & 1) ? other : 0)));
        r.b[i] = __ldg(reinterpret_cast<const uint4*>(pb + (i >> 1) * 128 + ((i & 1) ? other : 0)));
    }
}

// gl.value[i] = q . row i for the listed rows.  `rows`: the head's first row, `q`: the query's.
template <int D> struct GatherQuery { uint4 v[D / 32]; };
template <int D> __device__ __forceinline__ void gather_query(GatherQuery<D>& qr, const __nv_bfloat16* __restrict__ q) {
    constexpr int I = D / 32;
    const int lane = threadIdx.x & 31, g = lane >> 2, j = lane & 3;
#pragma unroll
    for (int i = 0; i < I; ++i) qr.v[i] = __ldg(reinterpret_cast<const uint4*>(q) + 4 * (I > 1 ? i ^ (g & 1) : i) + j);
}
template <int D>
__device__ __forceinline__ void gather_dots(GatherList& gl, int total, const GatherQuery<D>& qr, const __nv_bfloat16* __restrict__ rows, uint32_t tok_bytes) {
    constexpr int I = D / 32;
    const int lane = threadIdx.x & 31, g = lane >> 2, j = lane & 3;
    const uint4 (&qv)[I] = qr.v;
    const char* src = reinterpret_cast<const char*>(rows) + j * 16;
    _Pragma("unroll 1")
    for (int s = 0; s < total; s += 16) {
        GatherRows<D> r;
        gather_load<D>(r, gl, s, src, tok_bytes);
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < I; ++i) {
            mma_bf16(c, r.a[i].x, r.b[i].x, r.a[i].y, r.b[i].y, qv[i].x, qv[i].y);
            mma_bf16(c, r.a[i].z, r.b[i].z, r.a[i].w, r.b[i].w, qv[i].z, qv[i].w);
        }
        // all even columns are equal, and all odd ones: the four lanes of a row hold the same numbers
        const float da = (g & 1) ? c[1] : c[0], db = (g & 1) ? c[3] : c[2];
        if (j < 2) gl.value[s + 8 * j + g] = j ? db : da;
    }
}

// The same for two items that share the warp: rows of the entries from `ra` on against query `qa`, from `rb` on against `qb`, eight
// of each at a time (lists padded to a multiple of 8).
template <int D>
__device__ __forceinline__ void gather_dots_pair(GatherList& gl, int ra, int ta, int rb, int tb, const __nv_bfloat16* __restrict__ qa,
                                                 const __nv_bfloat16* __restrict__ qb, const __nv_bfloat16* __restrict__ rows, uint32_t tok_bytes) {
    constexpr int I = D / 32;
    const int lane = threadIdx.x & 31, g = lane >> 2, j = lane & 3;
    GatherQuery<D> qr;                                 // columns 0, 1 (4, 5) the first query, 2, 3 the second
    gather_query<D>(qr, (g & 2) ? qb : qa);
    const char* src = reinterpret_cast<const char*>(rows) + j * 16;
    const uint32_t odd = I > 1 ? (g & 1) * 64u : 0u;
    const int other = I > 1 ? ((g & 1) ? -64 : 64) : 0;
    for (int s = 0; s < max(ta, tb); s += 8) {
        const char* pa = src + static_cast<uint64_t>(gl.token[(s < ta ? ra : rb) + s + g]) * tok_bytes + odd;     // a list that is at its end repeats the other's rows
        const char* pb = src + static_cast<uint64_t>(gl.token[(s < tb ? rb : ra) + s + g]) * tok_bytes + odd;
        uint4 a[I], b[I];
#pragma unroll
        for (int i = 0; i < I; ++i) {
            a[i] = __ldg(reinterpret_cast<const uint4*>(pa + (i >> 1) * 128 + ((i & 1) ? other : 0)));
            b[i] = __ldg(reinterpret_cast<const uint4*>(pb + (i >> 1) * 128 + ((i & 1) ? other : 0)));
        }
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < I; ++i) {
            mma_bf16(c, a[i].x, b[i].x, a[i].y, b[i].y, qr.v[i].x, qr.v[i].y);
            mma_bf16(c, a[i].z, b[i].z, a[i].w, b[i].w, qr.v[i].z, qr.v[i].w);
        }
        if (j == 0 && s < ta) gl.value[ra + s + g] = (g & 1) ? c[1] : c[0];
        if (j == 1 && s < tb) gl.value[rb + s + g] = (g & 1) ? c[3] : c[2];
    }
}

// acc += sum of value[i] * row i: 16 bytes of a row per lane (LPR lanes per row, CH channels each); the subgroups of a warp take four
// rows each in turn and their sums are added up by gather_finish.  The list is padded to a multiple of GatherStep::N.
template <int D, typename T = __nv_bfloat16> struct GatherStep {
    static constexpr int CH = 16 / static_cast<int>(sizeof(T)), LPR = D / CH, U = 32 / LPR, N = LPR >= 16 ? 8 * U : 4 * U;
};
template <int D, typename T = __nv_bfloat16>
__device__ __forceinline__ void gather_sum(const GatherList& gl, int total, const T* __restrict__ rows, uint32_t tok_bytes, float (&acc)[16 / sizeof(T)]) {
    using E = Elt<T, 1>;
    constexpr int LPR = GatherStep<D, T>::LPR, U = GatherStep<D, T>::U, B = GatherStep<D, T>::N / (4 * U);    // B batches of four rows in flight
    const int lane = threadIdx.x & 31;
    const char* src = reinterpret_cast<const char*>(rows) + (lane % LPR) * 16;
    const int u4 = (lane / LPR) * 4;
_Pragma("unroll 1")
    for (int s = 0; s < total; s += GatherStep<D, T>::N) {
        typename E::Row r[4 * B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const uint4 t = *reinterpret_cast<const uint4*>(gl.token + s + b * 4 * U + u4);
            const uint32_t tk[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) r[4 * b + i] = E::load(reinterpret_cast<const T*>(src + static_cast<uint64_t>(tk[i]) * tok_bytes));
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const float4 w = *reinterpret_cast<const float4*>(gl.value + s + b * 4 * U + u4);
            E::axpy_paired(w.x, r[4 * b], acc);
            E::axpy_paired(w.y, r[4 * b + 1], acc);
            E::axpy_paired(w.z, r[4 * b + 2], acc);
            E::axpy_paired(w.w, r[4 * b + 3], acc);
        }
    }
}

// The same for the item whose entries start at `region` by PER neighbouring subgroups of the warp (`sub`: which of them this is); the
// list is padded to a multiple of 4 * PER.
template <int D, int PER, typename T = __nv_bfloat16>
__device__ __forceinline__ void gather_sum_item(const GatherList& gl, int region, int total, int sub, const T* __restrict__ rows, uint32_t tok_bytes,
                                                float (&acc)[16 / sizeof(T)]) {
    using E = Elt<T, 1>;
    const char* src = reinterpret_cast<const char*>(rows) + ((threadIdx.x & 31) % GatherStep<D, T>::LPR) * 16;
    for (int s = region + sub * 4; s < region + total; s += 4 * PER) {
        const uint4 t = *reinterpret_cast<const uint4*>(gl.token + s);
        const uint32_t tk[4] = {t.x, t.y, t.z, t.w};
        typename E::Row r[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) r[i] = E::load(reinterpret_cast<const T*>(src + static_cast<uint64_t>(tk[i]) * tok_bytes));
        const float4 w = *reinterpret_cast<const float4*>(gl.value + s);
        E::axpy_paired(w.x, r[0], acc);
        E::axpy_paired(w.y, r[1], acc);
        E::axpy_paired(w.z, r[2], acc);
        E::axpy_paired(w.w, r[3], acc);
    }
}

// Adds the subgroups' sums up: every lane then holds the whole sums of its channels.
template <int D, int CH> __device__ __forceinline__ void gather_finish(float (&acc)[CH]) {
#pragma unroll
    for (int o = D / CH; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < CH; ++e) acc[e] += __shfl_xor_sync(kFullMask, acc[e], o);
}

}  // namespace dsa3d
