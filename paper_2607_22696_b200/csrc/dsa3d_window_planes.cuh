// Tiles of 4 x 4 x 8 queries of a fixed window whose halo region is walked one plane (along t) at a time: the pieces of
// dsa3d_fixed_window_planes.cu.
//
// Eight x-row pairs (two x-rows of eight outputs, neighbours along y) per tile, a warp per pair and 64 channels.  A product
// (m16n8k16) has one region row, 8 + kw - 1 positions padded to 16, on one side and the eight outputs of an x-row on the other.  What an
// output has to do with a position (its score, its weight) lies in the pair's table in shared memory, [x-row][v][output][w]: an
// output reaches kw positions of a region row, at the others it has no score to keep and a weight of zero, read from a
// place that holds zeros.
#pragma once
#include <cuda_bf16.h>

#include "dsa3d_common.cuh"
#include "dsa3d_gather.cuh"
#include "dsa3d_tcgen05.cuh"

namespace dsa3d {

template <int D, int KT, int KH, int KW>
struct WindowPlanes {
    static constexpr int TT = 4, TY = 4, TX = 8;
    static constexpr int NH = D / 64;                               // 64-channel halves of a row
    static constexpr int RT = TT + KT - 1, RY = TY + KH - 1, RX = TX + KW - 1;
    static constexpr int PS = RY * RX;                              // rows of one region plane
    static constexpr int PSP = ((RY - 1) * RX + 16 + 7) / 8 * 8;    // the last region row's 16 positions end inside its buffer
    static constexpr int WARPS = 8 * NH, THREADS = WARPS * 32;
    static constexpr int SLOT_HALF = PSP * 128;                     // one 64-channel half of a plane buffer: rows of 128 bytes, 128-byte swizzle
    static constexpr int ROW = KH * TX * KW, TABLE = 2 * ROW;       // words of an x-row, of a pair, for one kernel plane
    static constexpr int PAIR = 32 * NH;                            // threads that share a table
    static_assert(PSP >= PS && RX <= 16 && SLOT_HALF % 1024 == 0, "plane buffers keep the 1024-byte alignment of the swizzle");

    // Zeroes the rows of the plane buffers that no load writes: they are multiplied by zeros and must not hold anything non-finite.
    template <int NS> static __device__ __forceinline__ void clear_tails(unsigned char (&slot)[NS][NH][SLOT_HALF]) {
        for (int i = threadIdx.x; i < NS * NH * (PSP - PS) * 8; i += THREADS) {
            const int chunk = i & 7, row = PS + (i >> 3) % (PSP - PS), which = (i >> 3) / (PSP - PS);
            *reinterpret_cast<uint4*>(&slot[which / NH][which % NH][row * 128 + chunk * 16]) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    // The calling warp is done with a plane buffer that all warps read in turn (`left`: how many have, zero at the start).  The last one
    // refills it: a thread that does nothing but load would cost the others a quarter of their registers, which are given out by
    // four warps at a time.
    template <typename Refill> static __device__ __forceinline__ void release(unsigned* left, Refill refill) {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) {
            __threadfence_block();
            if (atomicAdd(left, 1u) == WARPS - 1u) {
                *left = 0u;
                __threadfence_block();
                refill();
            }
        }
    }
    // The pair's threads have all come here.
    static __device__ __forceinline__ void pair_barrier(int pair) { asm volatile("bar.sync %0, %1;" ::"r"(pair + 1), "n"(PAIR) : "memory"); }

    // Place in the table of the lane's e-th position (2 j, 2 j + 1, 2 j + 8, 2 j + 9) of a region row for output lane / 4; -1: outside its window.
    static __device__ __forceinline__ int weight_place(int e) {
        const int g = (threadIdx.x & 31) >> 2, w = 2 * (threadIdx.x & 3) + (e & 1) + 8 * (e >> 1) - g;
        return w >= 0 && w < KW ? g * KW + w : -1;
    }

    // A pair's sixteen rows (queries, or their dO) as operands of `scores`, by way of the pair's table (16 * D * 2 bytes of it, chunks
    // permuted by the row); zeros for outputs outside the grid.  The pair's threads call it together when nothing in the table is needed
    // any more; it may be written again when it returns.
    static __device__ __forceinline__ void operands(uint32_t (&op)[2][D / 16][2], uint32_t* table, const __nv_bfloat16* __restrict__ rows, int pair, int me,
                                                    int t, int y0, int x0, int m, int T, int H, int W, int heads) {
        constexpr int CPR = D / 8;
        const int lane = threadIdx.x & 31;
        unsigned char* stage = reinterpret_cast<unsigned char*>(table);
        pair_barrier(pair);
#pragma unroll
        for (int i = me; i < 16 * CPR; i += PAIR) {
            const int row = i / CPR, chunk = i % CPR, y = y0 + (row >> 3), x = x0 + (row & 7);
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (t < T && y < H && x < W) v = __ldg(reinterpret_cast<const uint4*>(rows + (((static_cast<long long>(t) * H + y) * W + x) * heads + m) * D) + chunk);
            *reinterpret_cast<uint4*>(stage + row * (D * 2) + ((chunk ^ (row & 7)) << 4)) = v;
        }
        pair_barrier(pair);
        const int row = (lane & 7) + ((lane >> 4) << 3);
        const uint32_t at = smem_u32(stage) + row * (D * 2);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(op[0][ks][0]), "=r"(op[0][ks][1]), "=r"(op[1][ks][0]), "=r"(op[1][ks][1]) : "r"(at + (((2 * ks + ((lane >> 3) & 1)) ^ (row & 7)) << 4)));
        pair_barrier(pair);
    }

    // Scores (times `scale`) of the pair's rows with a region plane into the table of its kernel plane, every NH-th region row by this warp.
    static __device__ __forceinline__ void scores(const uint32_t (&op)[2][D / 16][2], const unsigned char (&plane)[NH][SLOT_HALF], int ly, int half, float* table, float scale) {
        const int lane = threadIdx.x & 31, g8 = lane >> 2, j4 = lane & 3;
_Pragma("unroll 1")
        for (int rr = half; rr <= KH; rr += NH) {              // row rr of the first x-row's window, rr - 1 of the second's
            float c[2][4];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int e = 0; e < 4; ++e) c[r][e] = 0.0f;
            const int row = (ly + rr) * RX + (lane & 15);
            const uint32_t at = smem_u32(plane[0]) + row * 128;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                uint32_t a0, a1, a2, a3;
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                             : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3) : "r"(at + (ks >> 2) * SLOT_HALF + (((2 * (ks & 3) + (lane >> 4)) ^ (row & 7)) << 4)));
                mma_bf16(c[0], a0, a1, a2, a3, op[0][ks][0], op[0][ks][1]);
                mma_bf16(c[1], a0, a1, a2, a3, op[1][ks][0], op[1][ks][1]);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int v = rr - r;
                if (v < 0 || v >= KH) continue;
                float* to = table + r * ROW + v * (TX * KW);
#pragma unroll
                for (int e = 0; e < 4; ++e) {                  // position g8 (+ 8) of the region row, output 2 j4 (+ 1)
                    const int x = 2 * j4 + (e & 1), w = g8 + 8 * (e >> 1) - x;
                    if (w >= 0 && w < KW) to[x * KW + w] = c[r][e] * scale;
                }
            }
        }
    }

    // acc[r] += rows of a region plane (64 channels at `plane`) . weights of x-row r, each weight a word of bf16 head | bf16 remainder
    // << 16; `ly`: the pair's first x-row, `table`: its words for this kernel plane.
    static __device__ __forceinline__ void sums(float (&acc)[2][4][4], const unsigned char* plane, int ly, const uint32_t* table, const uint32_t* zero, const int (&place)[4]) {
        const int lane = threadIdx.x & 31;
        const uint32_t* word[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) word[e] = place[e] >= 0 ? table + place[e] : zero;
        const uint32_t xs = smem_u32(plane);
        const int row0 = ly * RX + (lane & 7) + ((lane >> 4) << 3);
#pragma unroll
        for (int rr = 0; rr <= KH; ++rr) {
            uint32_t a[4][4];
            const int row = row0 + rr * RX;
            const uint32_t at = xs + row * 128 + ((((lane >> 3) & 1) ^ (row & 7)) << 4);
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                             : "=r"(a[mt][0]), "=r"(a[mt][1]), "=r"(a[mt][2]), "=r"(a[mt][3]) : "r"(at ^ (mt << 5)));
            uint32_t b[2][2][2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (rr - r < 0 || rr - r >= KH) continue;
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) w[e] = word[e][r * ROW + (rr - r) * (TX * KW)];
                b[0][r][0] = __byte_perm(w[0], w[1], 0x5410); b[0][r][1] = __byte_perm(w[2], w[3], 0x5410);
                b[1][r][0] = __byte_perm(w[0], w[1], 0x7632); b[1][r][1] = __byte_perm(w[2], w[3], 0x7632);
            }
#pragma unroll
            for (int z = 0; z < 2; ++z)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (rr - r < 0 || rr - r >= KH) continue;
#pragma unroll
                    for (int mt = 0; mt < 4; ++mt) mma_bf16(acc[r][mt], a[mt][0], a[mt][1], a[mt][2], a[mt][3], b[z][r][0], b[z][r][1]);
                }
        }
    }

    // The eight outputs of an x-row, 64 channels, rounded to bf16: channels x outputs turned into outputs x channels in `mine` (1 KB of
    // the warp's, chunks permuted by the output), then write(output, 16-byte chunk, bits).
    template <typename Write> static __device__ __forceinline__ void results(const float (&acc)[4][4], unsigned char* mine, Write write) {
        const int lane = threadIdx.x & 31;
        const uint32_t to = smem_u32(mine) + (lane & 7) * 128;
#pragma unroll
        for (int mt = 0; mt < 4; mt += 2) {
            uint32_t v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(acc[mt + (e >> 1)][2 * (e & 1)], acc[mt + (e >> 1)][2 * (e & 1) + 1]);
                v[e] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                         ::"r"(to + (((2 * mt + (lane >> 3)) ^ (lane & 7)) << 4)), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
        }
        __syncwarp();
#pragma unroll
        for (int i = lane; i < TX * 8; i += 32) write(i >> 3, i & 7, *reinterpret_cast<const uint4*>(mine + (i >> 3) * 128 + (((i & 7) ^ (i >> 3)) << 4)));
        __syncwarp();
    }
};

// An fp32 weight as two bf16 numbers whose sum is the weight to 2^-17 relative: head in the low half of the word, remainder in the high half.
__device__ __forceinline__ uint32_t split_weight(float w) {
    const __nv_bfloat16 head = __float2bfloat16_rn(w), rest = __float2bfloat16_rn(w - __bfloat162float(head));
    return static_cast<uint32_t>(__bfloat16_as_ushort(head)) | (static_cast<uint32_t>(__bfloat16_as_ushort(rest)) << 16);
}

}  // namespace dsa3d
