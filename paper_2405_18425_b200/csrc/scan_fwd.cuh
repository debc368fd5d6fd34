// BiGLA forward (paper Eq. 6) step by step in fp32 on the CUDA cores: the fp32 entry point, the bf16 head sizes the
// tensor-core kernels do not cover, and (adjoint) the gradient with respect to v of units beyond the range of the factorised tiles.  No factorised gates, so any decay is in range.
//
// Column j of the state depends on column j of v alone, so a block takes sixteen value columns of one unit, and its warps
// take the sequence in segments that are walked at the same time: every warp first finds, in one ascending pass, what its
// tokens add to either state and by how much they shrink what enters it; each then folds the segments before it (forward)
// and after it (backward) and walks its tokens up and down from those states.  What bounds it is the chain of tokens a
// warp walks (about 50 instructions each), so few units are cut into many segments; enough units to fill the chip are
// walked whole, without the first pass.  48 units of 196 tokens, 32 x 64, fp32: 31 us; one block of 128 threads per unit,
// one direction after the other, took 256 us.
//
// Lane (rg, cp) keeps rows [rg RPL, rg RPL + RPL) of columns 2 cp, 2 cp + 1 as packed pairs of rows, so that the rows of q,
// k and the gates come from shared memory as the operands they are.  Tokens are staged TG at a time by the warp that walks
// them, the next TG on their way in registers meanwhile; no barrier but the two around the fold.
#pragma once
#include "ptx.cuh"
#include "recurrence.cuh"

namespace vig {
namespace scan {

constexpr int TG = 4;       // tokens staged at once
constexpr int kCols = 16;   // value columns of a block of two columns a lane

template <typename T>
struct ScanArgs {
    const T *q, *k, *v, *gf, *gb;   // log gates of the two directions; the gate of token t is element t + sf (t + sb), 0 outside
    T* out;
    int L, dk, dv, seg_len, sf, sb;
};

constexpr int scan_max_warps(int rpl) { return rpl <= 16 ? 8 : 1; }   // segments per block (32 rows a lane: no registers for the first pass)
// Segments of calls whose blocks have an SM each: twice as many, of twelve tokens at least (a segment costs every other one a fold step).
// Up to 1200 tokens: beyond that they are less exact (error against 64 bits, sixteen to eight, gate logits around -1 / 0 / 2:
// 1.00 / 1.00 / 0.98 at 1200 tokens, 1.013 / 1.003 / 0.99 at 2048, 1.02 / 1.01 / 0.99 at 3000), if faster (training step of 12 units of
// 1100, 24 x 48: 258 us, 326 with eight).
constexpr int kManyWarps = 16, kManyTokens = 1200;
inline int many_segments(int L) { return L / 12 < 8 ? 8 : (L / 12 < kManyWarps ? L / 12 : kManyWarps); }
constexpr size_t scan_stage_floats(int rpl, int cpl = 2) { return (size_t)TG * (3 * 4 * rpl + 8 * cpl); }
constexpr size_t scan_fold_floats(int rpl, int cpl = 2) { return (size_t)2 * 4 * rpl * (8 * cpl + 1); }

// One slab of 8 CPL value columns of one unit by the first nw warps of a block (this one is number w), a segment of
// a.seg_len tokens each: nw of them cover the sequence.  Every thread of the block calls it: block barriers inside.
template <typename T, int RPL, bool VEC, int CPL = 2>
__device__ __forceinline__ void scan_fwd_slab(const ScanArgs<T>& a, size_t unit, int slab, int w, int nw, float* sc_smem) {
    constexpr int DKP = 4 * RPL, R2 = RPL / 2, HC = (RPL + 7) / 8, kWide = 8 * CPL, kPieces = TG * kWide / 4;   // 4-column pieces of v in a group
    const int lane = threadIdx.x & 31;
    const int cp = lane & 7, rg = lane >> 3;
    const bool on = w < nw;
    const int L = a.L, dk = a.dk, dv = a.dv;
    const size_t ok = unit * L * dk, ov = unit * L * dv;
    const int col0 = slab * kWide;
    const int s0 = w * a.seg_len, s1 = min(L, s0 + a.seg_len);
    float* xs = sc_smem + w * scan_stage_floats(RPL, CPL);   // [TG][DKP]: q (walks) or the gates of the backward direction (first pass)
    float* ks = xs + TG * DKP;
    float* as = ks + TG * DKP;
    float* vs = as + TG * DKP;                          // [TG][8 CPL]

    // the next TG tokens of a walk (t = base + step n) on their way, four key dimensions (value columns) of a token per lane
    using P = Piece<T, VEC>;
    P rx[HC], rk[HC], ra[HC], rv;
    auto fetch = [&](int base, int step, const T* x, int sx, const T* ga, int sa) {
#pragma unroll
        for (int h = 0; h < HC; ++h) {
            const int y = lane + 32 * h, t = base + step * (y / RPL), d = 4 * (y % RPL);   // (RPL = 4: the upper half of the warp has nothing to do)
            const int n = t >= s0 && t < s1 && y < TG * RPL ? dk - d : 0;
            rx[h].load(x + (ptrdiff_t)(t + sx) * dk + d, t + sx >= 0 && t + sx < L ? n : 0);
            rk[h].load(a.k + ok + (ptrdiff_t)t * dk + d, n);
            ra[h].load(ga + (ptrdiff_t)(t + sa) * dk + d, t + sa >= 0 && t + sa < L ? n : 0);
        }
        const int t = base + step * (lane / (kWide / 4)), j = col0 + 4 * (lane % (kWide / 4));
        rv.load(a.v + ov + (ptrdiff_t)t * dv + j, lane < kPieces && t >= s0 && t < s1 ? dv - j : 0);
    };
    // ... and into shared memory (tokens outside the segment: k = q = 0, gate 1)
    auto commit = [&](bool x_is_gate) {
        __syncwarp();
#pragma unroll
        for (int h = 0; h < HC; ++h) {
            const int y = lane + 32 * h;
            if (RPL >= 8 || y < TG * RPL) {   // (the pieces of a token are consecutive: y is also the place)
                float4 x = rx[h].get(), g = ra[h].get();
                if (x_is_gate) x = make_float4(expf(x.x), expf(x.y), expf(x.z), expf(x.w));
                reinterpret_cast<float4*>(xs)[y] = x;
                reinterpret_cast<float4*>(ks)[y] = rk[h].get();
                reinterpret_cast<float4*>(as)[y] = make_float4(expf(g.x), expf(g.y), expf(g.z), expf(g.w));
            }
        }
        if (lane < kPieces) reinterpret_cast<float4*>(vs)[lane] = rv.get();
        __syncwarp();
    };
    auto rows = [&](const float* p, int n, f32x2 (&r)[R2]) {
        const ulonglong2* s = reinterpret_cast<const ulonglong2*>(p + n * DKP + rg * RPL);
#pragma unroll
        for (int x = 0; x < R2 / 2; ++x) {
            const ulonglong2 u = s[x];
            r[2 * x] = u.x;
            r[2 * x + 1] = u.y;
        }
    };
    // column h of this lane: two of them side by side, more of them eight apart (the eight lanes of a row group read whole lines)
    auto column = [&](int h) { return CPL == 2 ? 2 * cp + h : 8 * h + cp; };
    auto cols = [&](int n, f32x2 (&v2)[CPL]) {
        if constexpr (CPL == 2) {
            const float2 v = *reinterpret_cast<const float2*>(vs + n * kWide + 2 * cp);
            v2[0] = pack2(v.x, v.x);
            v2[1] = pack2(v.y, v.y);
        } else {
#pragma unroll
            for (int h = 0; h < CPL; ++h) {
                const float v = vs[n * kWide + column(h)];
                v2[h] = pack2(v, v);
            }
        }
    };

    f32x2 S[R2][CPL], X[R2][CPL];   // the states that enter the segment from the left and from the right
#pragma unroll
    for (int r = 0; r < R2; ++r)
#pragma unroll
        for (int h = 0; h < CPL; ++h) S[r][h] = X[r][h] = 0ull;   // (+0, +0)
    if (scan_max_warps(RPL) > 1 && nw > 1) {
        // ---- first pass: forward state left behind (S) and its decay (D); backward state at the first token (X), the running
        // product of the backward gates (P) turning the recurrence into a sum that also runs upwards ----
        f32x2 D[R2], P[R2];
        const f32x2 one = pack2(1.f, 1.f);
#pragma unroll
        for (int r = 0; r < R2; ++r) D[r] = P[r] = one;
        if (on) fetch(s0, 1, a.gb + ok, a.sb, a.gf + ok, a.sf);
        for (int t0 = s0; on && t0 < s1; t0 += TG) {
            commit(true);
            if (t0 + TG < s1) fetch(t0 + TG, 1, a.gb + ok, a.sb, a.gf + ok, a.sf);
#pragma unroll
            for (int n = 0; n < TG; ++n) {
                f32x2 kk[R2], af[R2], ab[R2], v2[CPL];
                rows(ks, n, kk);
                rows(as, n, af);
                rows(xs, n, ab);
                cols(n, v2);
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    const f32x2 pk = fmul2(P[r], kk[r]);
#pragma unroll
                    for (int h = 0; h < CPL; ++h) {
                        S[r][h] = ffma2(af[r], S[r][h], fmul2(kk[r], v2[h]));
                        X[r][h] = ffma2(pk, v2[h], X[r][h]);
                    }
                    D[r] = fmul2(D[r], af[r]);
                    P[r] = fmul2(P[r], ab[r]);
                }
            }
        }
        __syncthreads();   // the fold area lies over the staging
        f32x2* st = reinterpret_cast<f32x2*>(sc_smem);                                   // [warp][dir][R2][CPL][lane]
        f32x2* dec = reinterpret_cast<f32x2*>(sc_smem + (size_t)nw * 2 * DKP * kWide);   // [warp][dir][DKP / 2]
#pragma unroll
        for (int r = 0; r < R2; ++r) {
#pragma unroll
            for (int h = 0; h < CPL; ++h) {
                if (on) {
                    st[(((w * 2) * R2 + r) * CPL + h) * 32 + lane] = S[r][h];
                    st[(((w * 2 + 1) * R2 + r) * CPL + h) * 32 + lane] = X[r][h];
                }
                S[r][h] = X[r][h] = 0ull;
            }
            if (on && cp == 0) {
                dec[(w * 2) * (DKP / 2) + rg * R2 + r] = D[r];
                dec[(w * 2 + 1) * (DKP / 2) + rg * R2 + r] = P[r];
            }
        }
        __syncthreads();
        auto fold = [&](int s, int dir, f32x2 (&to)[R2][CPL]) {
#pragma unroll
            for (int r = 0; r < R2; ++r) {
                const f32x2 d = dec[(s * 2 + dir) * (DKP / 2) + rg * R2 + r];
#pragma unroll
                for (int h = 0; h < CPL; ++h) to[r][h] = ffma2(d, to[r][h], st[(((s * 2 + dir) * R2 + r) * CPL + h) * 32 + lane]);
            }
        };
        for (int s = 0; s < w && on; ++s) fold(s, 0, S);
        for (int s = nw - 1; s > w; --s) fold(s, 1, X);
        __syncthreads();
    }
    if (!on) return;

    // ---- the walks: up (o> into `out`), then down ((o> + o<) / 2); the same lane writes and reads back an element ----
#pragma unroll 1
    for (int walk = 0; walk < 2; ++walk) {
        const int step = walk == 0 ? 1 : -1;
        const T* ga = (walk == 0 ? a.gf : a.gb) + ok;
        const int sa = walk == 0 ? a.sf : a.sb, first = walk == 0 ? s0 : s1 - 1;
        if (walk == 1) {
#pragma unroll
            for (int r = 0; r < R2; ++r)
#pragma unroll
                for (int h = 0; h < CPL; ++h) S[r][h] = X[r][h];
        }
        fetch(first, step, a.q + ok, 0, ga, sa);
        for (int m = 0; m < s1 - s0; m += TG) {
            const int base = first + step * m;
            commit(false);
            if (m + TG < s1 - s0) fetch(base + step * TG, step, a.q + ok, 0, ga, sa);
            T up[CPL];
            if (walk == 1) {
#pragma unroll
                for (int h = 0; h < CPL; ++h) {
                    const int t = base - rg, j = col0 + column(h);
                    up[h] = t >= s0 && j < dv ? a.out[ov + (size_t)t * dv + j] : T(0.f);
                }
            }
            float o[4][CPL];
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                f32x2 qq[R2], kk[R2], af[R2], v2[CPL], acc[CPL];
                rows(xs, n, qq);
                rows(ks, n, kk);
                rows(as, n, af);
                cols(n, v2);
#pragma unroll
                for (int h = 0; h < CPL; ++h) acc[h] = 0ull;
#pragma unroll
                for (int r = 0; r < R2; ++r) {
#pragma unroll
                    for (int h = 0; h < CPL; ++h) {
                        S[r][h] = ffma2(af[r], S[r][h], fmul2(kk[r], v2[h]));   // S_t = G_t . S_prev + k_t^T v_t
                        acc[h] = ffma2(qq[r], S[r][h], acc[h]);                 // o_t = q_t S_t
                    }
                }
#pragma unroll
                for (int h = 0; h < CPL; ++h) o[n][h] = sum2(acc[h]);
            }
            // sums over the four row groups, token n to the lanes of row group n
            float h2[2][CPL], o1[CPL];
            const bool hi = rg & 2, odd = rg & 1;
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int h = 0; h < CPL; ++h) h2[n][h] = (hi ? o[n + 2][h] : o[n][h]) + __shfl_xor_sync(0xffffffffu, hi ? o[n][h] : o[n + 2][h], 16);
#pragma unroll
            for (int h = 0; h < CPL; ++h) o1[h] = (odd ? h2[1][h] : h2[0][h]) + __shfl_xor_sync(0xffffffffu, odd ? h2[0][h] : h2[1][h], 8);
            const int t = base + step * rg;
            if (t >= s0 && t < s1) {
#pragma unroll
                for (int h = 0; h < CPL; ++h) {
                    const int j = col0 + column(h);
                    if (j < dv) rec_store(a.out + ov + (size_t)t * dv + j, walk == 0 ? o1[h] : 0.5f * (rec_to_float(up[h]) + o1[h]));
                }
            }
        }
    }
}

}  // namespace scan
}  // namespace vig
