// FP32 products on the half-precision tensor-core instructions (mma.sync.m16n8k16, FP32
// accumulate): every operand is the sum of two or three half-precision pieces and the products
// of the pieces that matter are accumulated. On this chip m16n8k16 issues as often as the TF32
// m16n8k8 (one per 8.3 cycles per scheduler, measured) with twice the inner width, so pieces of
// 16 bits do a split product in at most the instructions TF32 pieces take.
//
//   Bf16x3 : x = h + m + l in bfloat16, exact (8 + 8 + 8 bits, the exponent range of FP32). Six
//            products (hh, hm, mh, mm, hl, lh); what is dropped is below 2^-26 of a term.
//   Fp16x2 : x = h + l in half precision. Three products (hh, hl, lh); ll is below 2^-24 of a term,
//            as in a TF32 head + tail split. Half the instructions of Bf16x3, but five exponent bits:
//            a row of activations (and a warp's block of weights) is multiplied by a power of two
//            that puts a bound of its entries at 2^15. Entries down to 2^-17 of the bound are then
//            within 2^-24 of themselves (half an ulp of FP32), smaller ones within 2^-40 of the
//            bound. A layer's bound is that of its input times prod(norm + 1) of the layers between,
//            2^3 to 2^5 a layer above what comes out: entries below 2^-5 to 2^-8 of a row's largest
//            lose bits in f's second product, a hundredth of the rounding of a row's largest entry.
//
// The product is computed transposed: the instruction's 16 rows are 16 output columns of a layer
// (weights, A fragments, in registers), its 8 columns a tile's 8 data rows (B fragments, read with
// ldmatrix from a row-major tile of 16-bit pieces); results go back into such a tile with stmatrix.trans.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "kernels.cuh"

namespace placeto {
namespace split {

struct Bf16x3 {
    static constexpr int kPieces = 3;
    static constexpr bool kScaled = false;
    // two values -> their pieces, each pair packed into 32 bits (first value in the low half)
    __device__ static __forceinline__ void pieces(float x, float y, unsigned (&p)[3]) {
        p[0] = pack(x, y);
        x -= __uint_as_float(p[0] << 16);
        y -= __uint_as_float(p[0] & 0xffff0000u);
        p[1] = pack(x, y);
        x -= __uint_as_float(p[1] << 16);
        y -= __uint_as_float(p[1] & 0xffff0000u);
        p[2] = pack(x, y);
    }
    __device__ static __forceinline__ unsigned pack(float lo, float hi) {
        unsigned d;
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
        return d;
    }
    __device__ static __forceinline__ void mma(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
        // volatile: the accumulator chains stay interleaved as written
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    }
    __device__ static __forceinline__ void mma_zero(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
    }
};

struct Fp16x2 {
    static constexpr int kPieces = 2;
    static constexpr bool kScaled = true;
    __device__ static __forceinline__ void pieces(float x, float y, unsigned (&p)[2]) {
        const __half2 h = __floats2half2_rn(x, y);
        const float2 f = __half22float2(h);
        const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
        p[0] = *reinterpret_cast<const unsigned *>(&h);
        p[1] = *reinterpret_cast<const unsigned *>(&l);
    }
    __device__ static __forceinline__ void mma(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    }
    __device__ static __forceinline__ void mma_zero(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
    }
};

// The power of two that brings numbers of magnitude at most `bound` below 2^15. Bounds below 2^-97 are taken as
// 2^-97, so that it and its inverse stay normal numbers.
__device__ __forceinline__ float scale_up(float bound) {
    return __uint_as_float((268u - min(max(__float_as_uint(bound) >> 23 & 0xffu, 30u), 250u)) << 23);
}
// 1 / p for a power of two (both normal)
__device__ __forceinline__ float inverse_pow2(float p) { return __uint_as_float(0x7f000000u - __float_as_uint(p)); }
// the smallest power of two that is at least x (x >= 1, finite)
__device__ __forceinline__ float pow2_above(float x) {
    const unsigned b = __float_as_uint(x);
    return __uint_as_float((b & 0x7fffffu) ? (b & 0x7f800000u) + 0x800000u : b);
}

// One warp's 16 output columns [c0, c0 + 16) of a matrix as A fragments of the transposed product: for
// k-step ks, with g = lane / 4 and t = lane % 4, register i holds the k = 16 ks + 2t + 8 (i / 2) (and
// the next) entries of column c0 + g + 8 (i % 2). `inv` undoes the block's scale.
template <typename SP, int KS>
struct Weights {
    unsigned a[SP::kPieces][KS][4];
    float inv;
    // `at(k, c)`: the entry at inner index k of output column c. Returns the largest sum of magnitudes over
    // a column of the block (only where SP scales): |out| <= that * max |in|.
    template <typename At>
    __device__ __forceinline__ float load(int c0, int lane, At at) {
        const int g = lane >> 2, t = lane & 3;
        float raw[KS][4][2];
        float top = 0.f, sum[2] = {0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    raw[ks][i][j] = at(16 * ks + 2 * t + 8 * (i >> 1) + j, c0 + g + 8 * (i & 1));
                    top = fmaxf(top, fabsf(raw[ks][i][j]));
                    sum[i & 1] += fabsf(raw[ks][i][j]);
                }
        float up = 1.f, norm = 0.f;
        inv = 1.f;
        if (SP::kScaled) {
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
                sum[1] += __shfl_xor_sync(0xffffffffu, sum[1], o);
            }
            norm = fmaxf(sum[0], sum[1]);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
                norm = fmaxf(norm, __shfl_xor_sync(0xffffffffu, norm, o));
            }
            up = scale_up(top);
            inv = inverse_pow2(up);
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                unsigned p[SP::kPieces];
                SP::pieces(raw[ks][i][0] * up, raw[ks][i][1] * up, p);
#pragma unroll
                for (int q = 0; q < SP::kPieces; ++q) a[q][ks][i] = p[q];
            }
        return norm;
    }
};

// Four (two) 8 x 8 blocks of 16-bit words: lane i gives the address of row i % 8 of block i / 8 and receives,
// from block j, the words 2 (lane % 4) and the next of row lane / 4. OFF: a byte offset known at compile time
// (no address arithmetic per instruction).
template <int OFF>
__device__ __forceinline__ void ldmatrix4(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4+%5];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr), "n"(OFF)
                 : "memory");
}
template <int OFF>
__device__ __forceinline__ void ldmatrix2(unsigned (&r)[2], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2+%3];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(addr), "n"(OFF)
                 : "memory");
}
// The reverse, transposed: from lane's word pair (row lane / 4, columns 2 (lane % 4) ...) of block j, word r of
// memory row c is row r, column c of the block.
__device__ __forceinline__ void stmatrix4_trans(unsigned addr, unsigned a, unsigned b, unsigned c, unsigned d) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ void stmatrix2_trans(unsigned addr, unsigned a, unsigned b) {
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

template <typename SP, bool kFirst>
__device__ __forceinline__ void chain(float (&d)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
    if constexpr (kFirst) SP::mma_zero(d, a, b[0], b[1]);
    else SP::mma(d, a, b[0], b[1]);
}
// A tile: 8 rows of `stride` bytes per piece (16 mod 128 or an equivalent that spreads eight rows' 16-byte
// chunks over the banks), the pieces PIECE bytes apart. Sums KS k-steps of 16 of NT tiles into `out`. Three
// accumulator chains per tile, interleaved, so that a dependent instruction (21 cycles) finds the pipe free: the
// large products (hh) of either half of the k-steps after some of the small ones, the other small ones alone. The
// tensor core's own accumulation truncates, so the halves are added up outside. (k-steps in the order in which the
// fragments arrive, or the chains dealt strictly in turn: 4 to 10 % slower in the sweep kernel.)
template <typename SP, int KS, int NT, int OFF, int PIECE>
__device__ __forceinline__ void tile_mma(const Weights<SP, KS> &w, const unsigned (&tile)[NT], float (&out)[NT][4]) {
    constexpr int NP = SP::kPieces;
    static_assert(KS == 1 || KS == 2 || KS == 4, "one k-step or whole pairs");
    constexpr int KH = KS > 1 ? KS / 2 : 1;          // k-steps of chains A and B
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        unsigned b[NP][KS][2];
        auto load = [&](auto piece, auto pair) {
            constexpr int q = decltype(piece)::value, kp = decltype(pair)::value;
            if constexpr (q < NP && 2 * kp < KS) {
                if constexpr (KS == 1) {
                    ldmatrix2<OFF + q * PIECE>(b[q][0], tile[nt]);
                } else {
                    unsigned r[4];
                    ldmatrix4<OFF + q * PIECE + 64 * kp>(r, tile[nt]);
                    b[q][2 * kp][0] = r[0]; b[q][2 * kp][1] = r[1];
                    b[q][2 * kp + 1][0] = r[2]; b[q][2 * kp + 1][1] = r[3];
                }
            }
        };
        typedef std::integral_constant<int, 0> c0;
        typedef std::integral_constant<int, 1> c1;
        typedef std::integral_constant<int, 2> c2;
        load(c0(), c0()); load(c1(), c0()); load(c2(), c0());
        load(c0(), c1()); load(c1(), c1()); load(c2(), c1());
        float A[4], Bc[4], C[4];
        if constexpr (KS == 1) {
            if constexpr (NP == 2) {
                chain<SP, true>(A, w.a[0][0], b[1][0]);
                chain<SP, true>(C, w.a[1][0], b[0][0]);
                chain<SP, false>(A, w.a[0][0], b[0][0]);
#pragma unroll
                for (int c = 0; c < 4; ++c) out[nt][c] = A[c] + C[c];
            } else {
                chain<SP, true>(A, w.a[2][0], b[0][0]);
                chain<SP, true>(Bc, w.a[0][0], b[2][0]);
                chain<SP, true>(C, w.a[0][0], b[1][0]);
                chain<SP, false>(A, w.a[1][0], b[1][0]);
                chain<SP, false>(C, w.a[1][0], b[0][0]);
                chain<SP, false>(A, w.a[0][0], b[0][0]);
#pragma unroll
                for (int c = 0; c < 4; ++c) out[nt][c] = A[c] + (Bc[c] + C[c]);
            }
        } else {
#pragma unroll
            for (int ks = 0; ks < KH; ++ks) {
                auto small = [&](auto first) {
                    constexpr bool z = decltype(first)::value;
                    chain<SP, z>(A, w.a[NP == 2 ? 0 : 2][ks], b[NP == 2 ? 1 : 0][ks]);
                    chain<SP, z>(Bc, w.a[NP == 2 ? 0 : 2][KH + ks], b[NP == 2 ? 1 : 0][KH + ks]);
                    chain<SP, z>(C, w.a[NP == 2 ? 1 : 0][ks], b[NP == 2 ? 0 : 1][ks]);
                    if constexpr (NP == 3) {
                        chain<SP, false>(A, w.a[0][ks], b[2][ks]);
                        chain<SP, false>(Bc, w.a[0][KH + ks], b[2][KH + ks]);
                        chain<SP, false>(C, w.a[1][ks], b[0][ks]);
                        chain<SP, false>(A, w.a[1][ks], b[1][ks]);
                        chain<SP, false>(Bc, w.a[1][KH + ks], b[1][KH + ks]);
                        chain<SP, false>(C, w.a[0][KH + ks], b[1][KH + ks]);
                    }
                    chain<SP, false>(C, w.a[1][KH + ks], b[0][KH + ks]);
                };
                if (ks == 0) small(std::true_type());
                else small(std::false_type());
            }
#pragma unroll
            for (int ks = 0; ks < KH; ++ks) {
                chain<SP, false>(A, w.a[0][ks], b[0][ks]);
                chain<SP, false>(Bc, w.a[0][KH + ks], b[0][KH + ks]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) out[nt][c] = (A[c] + Bc[c]) + C[c];
        }
    }
}
// this lane's ldmatrix offset in a tile piece (row lane % 8, block lane / 8)
__device__ __forceinline__ unsigned ld_offset(int lane, int stride) { return (lane & 7) * stride + 16 * (lane >> 3); }
// and its stmatrix offset for a block of 16 columns from c0: row lane % 8, columns c0 + 8 (lane / 8 % 2) ...
__device__ __forceinline__ unsigned st_offset(int lane, int stride, int c0) { return (lane & 7) * stride + 2 * (c0 + 8 * (lane >> 3 & 1)); }

// v[0], v[1]: column g of rows 2t, 2t + 1; v[2], v[3]: column g + 8 (the accumulator layout), split and stored
// into a tile; `at` is the tile's address plus st_offset.
template <typename SP>
__device__ __forceinline__ void store_tile(unsigned at, unsigned piece_bytes, int lane, const float (&v)[4]) {
    unsigned a[SP::kPieces], b[SP::kPieces];
    SP::pieces(v[0], v[1], a);
    SP::pieces(v[2], v[3], b);
    stmatrix4_trans(at + (lane >= 16 ? piece_bytes : 0u), a[0], b[0], a[1], b[1]);
    if constexpr (SP::kPieces == 3) stmatrix2_trans(at + 2 * piece_bytes, a[2], b[2]);
}
// four adjacent columns of a row, split and stored at `p` (the first piece; 8-byte aligned)
template <typename SP>
__device__ __forceinline__ void store_row4(unsigned char *p, unsigned piece_bytes, float4 v) {
    unsigned a[SP::kPieces], b[SP::kPieces];
    SP::pieces(v.x, v.y, a);
    SP::pieces(v.z, v.w, b);
#pragma unroll
    for (int q = 0; q < SP::kPieces; ++q) *reinterpret_cast<uint2 *>(p + q * piece_bytes) = make_uint2(a[q], b[q]);
}

// barrier of one group of warps (id 1 .. 15)
template <int kCount>
__device__ __forceinline__ void group_sync(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kCount) : "memory");
}

}  // namespace split
}  // namespace placeto
