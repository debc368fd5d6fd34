// Warp-level tensor-core pieces (mma.sync, fragments in registers) and the swizzled shared-memory tiles they read.
//
// Fragment conventions (lane = 4 g + c, g = 0 .. 7, c = 0 .. 3), for D[16 x 8] += A[16 x 16] B[16 x 8]:
//   A: a0 (row g, k 2c, 2c+1), a1 (row g + 8, same k), a2 (row g, k 2c + 8, 2c + 9), a3 (row g + 8, k 2c + 8, 2c + 9)
//   B: b0 (k 2c, 2c+1; column g), b1 (k 2c + 8, 2c + 9; column g)
//   D: d0, d1 (row g, columns 2c, 2c+1), d2, d3 (row g + 8, same columns)
// so the D fragment of one product, packed to bf16, is the A fragment of the next.
#pragma once
#include <cuda_bf16.h>

#include "ptx.cuh"

namespace vig {
namespace wmma16 {

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0));
}
// D = A B
__device__ __forceinline__ void mma_k16_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// D = A B + (lo, hi) in the even, odd columns of every row.
__device__ __forceinline__ void mma_k16_from(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1, float lo,
                                             float hi) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(lo), "f"(hi));
}
// Transpose of the 8 x 8 matrix of bf16 of which a warp holds one row per four lanes.
__device__ __forceinline__ uint32_t movmatrix(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

__device__ __forceinline__ void ldsm(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
// A [rows][RB bytes] bf16 tile in shared memory under the TMA swizzle of span RB, seen by one lane of an ldmatrix /
// stmatrix of four 8 x 8 matrices: rows row0 .. row0 + 15, 16-byte column pieces 2 n and 2 n + 1.  The operands of an mma
// are consecutive registers, so the order of the four matrices is chosen for the use (moves otherwise cost as many
// instructions as the products):
//   load        as A operand: a0 .. a3 of K step n
//   load_b      as B operand with the tile's rows as columns: rows 0-7 take (r[0], r[1]), rows 8-15 (r[2], r[3])
//   load_trans  as B operand that contracts over the rows: columns of piece 2n take (r[0], r[1]), of piece 2n + 1 (r[2], r[3])
//   (with off_b and a transposing load: A operand with the tile's columns as rows, a0 .. a3)
template <int RB>
struct Tile {
    uint32_t off[RB / 32], off_b[RB / 32];   // this lane's row of the sixteen and its swizzled piece, per n, in either order
    __device__ __forceinline__ explicit Tile(int lane) {
        auto at = [](int r, int h, int n) {
            const uint32_t sw = RB == 128 ? (uint32_t)((h ^ (r & 7)) << 4) : (uint32_t)((h ^ ((r >> 1) & 3)) << 4);
            return (uint32_t)r * RB + (sw ^ (uint32_t)(n << 5));
        };
#pragma unroll
        for (int n = 0; n < RB / 32; ++n) {
            off[n] = at(lane & 15, lane >> 4, n);
            off_b[n] = at((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1, n);
        }
    }
    __device__ __forceinline__ uint32_t at(uint32_t tile, int row0, int n) const { return tile + (uint32_t)row0 * RB + off[n]; }
    __device__ __forceinline__ void load(uint32_t tile, int row0, int n, uint32_t (&r)[4]) const { ldsm(at(tile, row0, n), r); }
    __device__ __forceinline__ void load_b(uint32_t tile, int row0, int n, uint32_t (&r)[4]) const { ldsm(tile + (uint32_t)row0 * RB + off_b[n], r); }
    __device__ __forceinline__ void load_trans(uint32_t tile, int row0, int n, uint32_t (&r)[4]) const { ldsm_trans(at(tile, row0, n), r); }
    __device__ __forceinline__ void store(uint32_t tile, int row0, int n, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) const {
        asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(at(tile, row0, n)), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
                     : "memory");
    }
};

// A fragment (a0 = a3) of the diagonal 8 x 8 blocks of the lower triangle of ones, with or without the diagonal; a1 of the
// 16 x 16 triangle is kOnes, a2 zero.
__device__ __forceinline__ uint32_t triangle(int g, int c, bool diagonal) {
    const int lim = diagonal ? g : g - 1;
    return (2 * c <= lim ? 0x3F80u : 0u) | (2 * c + 1 <= lim ? 0x3F800000u : 0u);
}
constexpr uint32_t kOnes = 0x3F803F80u;

// A 16 x 16 tile of scores on the diagonal, packed as A operand (p[0]: rows g, columns 2c, 2c+1; p[1]: rows g + 8; p[2], p[3]:
// columns + 8): left keeps the columns up to the row, else those from the row on.
struct DiagonalMask {
    uint32_t l, r;
    __device__ __forceinline__ DiagonalMask(int g, int c) {
        l = (2 * c <= g ? 0xFFFFu : 0u) | (2 * c + 1 <= g ? 0xFFFF0000u : 0u);
        r = (2 * c >= g ? 0xFFFFu : 0u) | (2 * c + 1 >= g ? 0xFFFF0000u : 0u);
    }
    __device__ __forceinline__ void apply(uint32_t (&p)[4], bool left) const {
        p[0] &= left ? l : r;
        p[3] &= left ? l : r;
        if (left) p[2] = 0u;
        else p[1] = 0u;
    }
};

// 1 / x for two packed positive, normal bf16 values without the special-function unit and without leaving the packed
// format: a bit-level first guess per half (one 32-bit subtraction: neither half borrows) and one Newton step r (2 - x r) in
// bf16x2 arithmetic.  Relative error at most 0.63 % (root mean square 0.27 %, the same as rounding an exact reciprocal to
// bf16 after a first guess of this kind); the result only scales bf16 operands, whose own rounding unit is 0.39 %, and it
// is the reciprocal of the very factor the other operand is scaled by.
__device__ __forceinline__ uint32_t rcp_bf16x2(uint32_t x) {
    const uint32_t r0 = 0x7EF27EF2u - x;
    const __nv_bfloat162 xb = *reinterpret_cast<const __nv_bfloat162*>(&x), rb = *reinterpret_cast<const __nv_bfloat162*>(&r0);
    const __nv_bfloat162 r1 = __hmul2(rb, __hfma2(__hneg2(xb), rb, __float2bfloat162_rn(2.0f)));
    return *reinterpret_cast<const uint32_t*>(&r1);
}

// Two bf16 as two fp32 (a bf16 is the upper half of its fp32), and two fp32 rounded to two bf16.
__device__ __forceinline__ f32x2 widen(uint32_t x) { return pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
__device__ __forceinline__ uint32_t pack_f32x2(f32x2 x) {
    float x0, x1;
    unpack2(x, x0, x1);
    return pack_bf16(x0, x1);
}

// log2 alpha = logsigmoid(g) / (tau ln 2) (Eq. 5 line 1, in base 2 so that the operand scaling needs no further
// multiplication) of two gate logits, evaluated in fp32 as (min(g, 0) log2(e) - log2(1 + e)) / tau with e = e^{-|g|} in (0, 1]
// from the special-function unit and log2(1 + e) = e p(e), on the FMA pipe, two values per instruction.
// LONG: p of degree five with the least relative error on [0, 1] (8.4e-6; 1.1e-5 over all bf16 logits as evaluated): an open
// gate's log alpha is e itself, and what p is off there does not average out over thousands of tokens as the bf16 rounding
// that follows does.  The cubic is off by 1e-4 at most, 0.25 % of e for open gates: units of up to 256 tokens, where it does
// not show in the result (4.6e-3 off in 2-norm with either), take it.  The two further terms cost 1 % of a call of 32 x 4096
// tokens (24, 48).
template <bool LONG>
__device__ __forceinline__ uint32_t log2_alpha_pair(uint32_t g, float inv_tau) {
    const float g0 = __uint_as_float(g << 16), g1 = __uint_as_float(g & 0xffff0000u);
    const f32x2 e = pack2(ex2(-fabsf(g0) * kLog2e), ex2(-fabsf(g1) * kLog2e));
    f32x2 p;
    if constexpr (LONG) {
        p = pack2(-0.034435905516147614f, -0.034435905516147614f);
        p = ffma2(p, e, pack2(0.1460328847169876f, 0.1460328847169876f));
        p = ffma2(p, e, pack2(-0.3030362129211426f, -0.3030362129211426f));
        p = ffma2(p, e, pack2(0.4691740572452545f, 0.4691740572452545f));
        p = ffma2(p, e, pack2(-0.7204261422157288f, -0.7204261422157288f));
        p = ffma2(p, e, pack2(1.4426828622817993f, 1.4426828622817993f));
    } else {
        p = pack2(-0.08476800471544266f, -0.08476800471544266f);
        p = ffma2(p, e, pack2(0.3255951702594757f, 0.3255951702594757f));
        p = ffma2(p, e, pack2(-0.6799444556236267f, -0.6799444556236267f));
        p = ffma2(p, e, pack2(1.4390150308609009f, 1.4390150308609009f));
    }
    const f32x2 minus = ffma2(p, e, fmul2(pack2(fminf(g0, 0.f), fminf(g1, 0.f)), pack2(-kLog2e, -kLog2e)));
    return pack_f32x2(fmul2(minus, pack2(-inv_tau, -inv_tau)));
}

// This lane's pairs of key dimensions of a row of DK bf16, straight from global memory.  Which dimensions pair j of lane c
// holds only has to be the same in both operands of a contraction; it is chosen so that a warp reads its rows in whole
// pieces, contiguous across the four lanes of a row:
//   DK = 32: dims 8c + 2j, +1;   DK = 24: dims 4c + 2j, +1 (j = 0, 1) and 16 + 2c, +1 (j = 2);   DK = 16: dims 4c + 2j, +1
// Ordinary loads, not those of the read-only path: this kernel may have started while the one that writes the row still ran
// (programmatic dependent launch), so the row is not read-only for the kernel's lifetime and the load must stay behind
// pdl_wait().  AHEAD: loads ahead of it, of rows that are known to be complete, from L2 (see pdl_wait).
template <int DK, bool AHEAD = false>
__device__ __forceinline__ void load_pairs(const __nv_bfloat16* row, int c, uint32_t (&r)[DK / 8]) {
    const char* p = reinterpret_cast<const char*>(row);
    if constexpr (DK == 32) {
        const uint4 x = AHEAD ? ld_gpu16(p + 16 * c) : *reinterpret_cast<const uint4*>(p + 16 * c);
        r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
    } else {
        const uint2 x = AHEAD ? ld_gpu8(p + 8 * c) : *reinterpret_cast<const uint2*>(p + 8 * c);
        r[0] = x.x; r[1] = x.y;
        if constexpr (DK == 24) r[2] = AHEAD ? ld_gpu4(p + 32 + 4 * c) : *reinterpret_cast<const uint32_t*>(p + 32 + 4 * c);
    }
}

// Lane c of a group of four holds words (c, 0 .. 3); afterwards words (0 .. 3, c).
__device__ __forceinline__ void transpose4(uint32_t (&x)[4], int c) {
#pragma unroll
    for (int p = 0; p < 4; p += 2) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, (c & 1) ? x[p] : x[p + 1], 1);
        if (c & 1) x[p] = y;
        else x[p + 1] = y;
    }
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, (c & 2) ? x[p] : x[p + 2], 2);
        if (c & 2) x[p] = y;
        else x[p + 2] = y;
    }
}

// x = hi + lo with two bf16 each: sixteen significant bits of an fp32 value as two tensor-core operands.
__device__ __forceinline__ void split_bf16(f32x2 x, uint32_t& hi, uint32_t& lo) {
    float x0, x1;
    unpack2(x, x0, x1);
    hi = pack_bf16(x0, x1);
    unpack2(ffma2(pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), pack2(-1.f, -1.f), x), x0, x1);
    lo = pack_bf16(x0, x1);
}

}  // namespace wmma16
}  // namespace vig
