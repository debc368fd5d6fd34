// Gradient of the BiGLA forward pass (paper Eq. 6) with respect to q, k and the two log gates, by the reverse-mode adjoint
// of the two recurrences, in fp32 on the CUDA cores; the gradient with respect to v is a forward pass on swapped operands
// with the gates moved by one token, which the caller launches.
//
// With g = dLoss/d_out, a> = exp(log alpha>), a< = exp(log alpha<), per unit and token t:
//   S>_t = a>_t S>_{t-1} + k_t^T v_t            (Eq. 6)            dq>_t = S>_t g_t^T / 2
//   Z>_t = a>_{t+1} Z>_{t+1} + q_t^T g_t / 2    (adjoint of S>_t)   dk>_t = Z>_t v_t^T
//   S<_t = a<_t S<_{t+1} + k_t^T v_t            (Eq. 6)            dq<_t = S<_t g_t^T / 2
//   Z<_t = a<_{t-1} Z<_{t-1} + q_t^T g_t / 2    (adjoint of S<_t)   dk<_t = Z<_t v_t^T
//   dq = dq> + dq<,  dk = dk> + dk<,  E> = q dq> - k dk>,  E< = q dq< - k dk< (element-wise)
//   dlog alpha>_t = sum_{m >= t} E>_m,   dlog alpha<_t = - sum_{m > t} E<_m
// (the log gates enter only through sums of gates between a key and a query; each direction is unchanged by q -> q / c,
// k -> c k per key dimension, so sum_m E_m = 0).  Over the tokens after a border these sums are the row sums of S o Z of the
// two states that meet there: pairs of tokens on the same side cancel.
//
// Row i of every state depends on key dimension i alone, so a block takes eight key dimensions of one unit and its warps
// take the sequence in segments walked at the same time: one ascending pass for what a segment adds to the four states and
// by how much it shrinks what enters them, a fold over the segments, then the walk up (S>, Z<: dq>, dk< to scratch) and the
// walk down (S<, Z>: everything else).  Nothing passes between blocks, and the call is one launch.  48 units of 196 tokens,
// 32 x 64, fp32: 50 us; 100 us as four launches (summary, fold, walks, sums put together) of four warps per segment.
#pragma once
#include "scan_fwd.cuh"

namespace vig {
namespace scan {

constexpr int kRows = 8;    // key dimensions of a block

template <typename T>
struct ScanBwdArgs {
    const T *q, *k, *v, *la_f, *la_b, *g;
    T *dq, *dkey, *dla_f, *dla_b;
    int L, dk, dv, seg_len;
};

// Threads of a row: four, CN columns each.
constexpr int bwd_max_warps(int cn) { return cn <= 16 ? 8 : 4; }   // segments per block
constexpr size_t bwd_stage_floats(int cn) { return (size_t)TG * (4 * kRows + 8 * (cn + 4)); }   // row records, v and d_out (groups of CN + 4: no bank conflicts)
constexpr size_t bwd_fold_floats(int cn) { return (size_t)4 * kRows * 4 * cn + 4 * kRows; }

// Where dq>, dk< of an element stay between the walks: scratch, [unit][L][dk].
struct FloatPairs {
    float2* p;
    __device__ __forceinline__ void put(size_t e, float2 x) const { p[e] = x; }
    __device__ __forceinline__ float2 get(size_t e) const { return p[e]; }
};

// One slab of eight key dimensions of one unit by the first nw warps of a block (this one is number w), a segment of a.seg_len
// tokens each: nw of them cover the sequence.  Every thread of the block calls it: block barriers inside.
template <typename T, int CN, bool VEC, typename Pairs>
__device__ __forceinline__ void scan_bwd_slab(const ScanBwdArgs<T>& a, const Pairs& pairs, size_t unit, int slab, int w, int nw, float* sb_smem) {
    constexpr int DVP = 4 * CN, VC = TG * CN / 32 + (TG * CN % 32 != 0), C2 = CN / 2, kPitch = 4 * (CN + 4);
    const int lane = threadIdx.x & 31;
    const int i = lane >> 2, cg = lane & 3;
    const bool on = w < nw;
    const int L = a.L, dk = a.dk, dv = a.dv;
    const size_t ok = unit * L * dk, ov = unit * L * dv;
    const int row0 = slab * kRows, row = row0 + i;
    const int s0 = w * a.seg_len, s1 = min(L, s0 + a.seg_len);
    float4* rec = reinterpret_cast<float4*>(sb_smem + w * bwd_stage_floats(CN));   // [TG][8]: k, q, decay of S, decay of Z
    float* vs = reinterpret_cast<float*>(rec + TG * kRows);                        // [TG][4 (CN + 4)]
    float* gs = vs + TG * kPitch;
    ulonglong2* st = reinterpret_cast<ulonglong2*>(sb_smem + nw * bwd_stage_floats(CN));   // [warp][kind][CN / 4][lane]
    float* dec = sb_smem + nw * bwd_stage_floats(CN) + (size_t)nw * 4 * kRows * DVP;       // [warp][kind][8]

    // the next TG tokens of a walk (t = base + step n) on their way; Z decays by the other direction's gate of the token before
    T rk, rq, rs, rz;
    Piece<T, VEC> rv[VC], rg[VC];
    auto fetch = [&](int base, int step, const T* las, const T* laz) {
        const int t = base + step * (lane >> 3), r = row0 + (lane & 7), tz = t - step;
        const bool in = t >= s0 && t < s1 && r < dk;
        const size_t e = ok + (size_t)t * dk + r;
        rk = in ? a.k[e] : T(0.f);
        rq = in ? a.q[e] : T(0.f);
        rs = in ? las[e] : T(0.f);
        rz = in && tz >= 0 && tz < L ? laz[ok + (size_t)tz * dk + r] : T(0.f);
#pragma unroll
        for (int m = 0; m < VC; ++m) {
            const int x = lane + 32 * m, tv = base + step * (x / CN), j = 4 * (x % CN);   // four columns of a token
            const int n = x < TG * CN && tv >= s0 && tv < s1 ? dv - j : 0;
            rv[m].load(a.v + ov + (ptrdiff_t)tv * dv + j, n);
            rg[m].load(a.g + ov + (ptrdiff_t)tv * dv + j, n);
        }
    };
    auto commit = [&]() {   // tokens outside the segment: k = q = v = g = 0, gates 1
        __syncwarp();
        rec[lane] = make_float4(rec_to_float(rk), rec_to_float(rq), expf(rec_to_float(rs)), expf(rec_to_float(rz)));
#pragma unroll
        for (int m = 0; m < VC; ++m) {
            const int x = lane + 32 * m, j = 4 * (x % CN), at = x / CN * kPitch + j / CN * (CN + 4) + j % CN;
            if (TG * CN % 32 == 0 || x < TG * CN) {
                *reinterpret_cast<float4*>(vs + at) = rv[m].get();
                *reinterpret_cast<float4*>(gs + at) = rg[m].get();
            }
        }
        __syncwarp();
    };
    f32x2 S[C2], Z[C2];
#pragma unroll
    for (int c = 0; c < C2; ++c) S[c] = Z[c] = 0ull;   // (+0, +0)

    const bool split = nw > 1;
    if (split && on) {
        // ---- first pass: S>, Z< left behind; S<, Z> at the first token, running products (ps, pz) of the gates turning their
        // recurrences into sums that also run upwards ----
        f32x2 R[C2], Y[C2];
#pragma unroll
        for (int c = 0; c < C2; ++c) R[c] = Y[c] = 0ull;
        float ds = 1.f, dz = 1.f, ps = 1.f, pz = 1.f;
        fetch(s0, 1, a.la_f, a.la_b);
        for (int t0 = s0; t0 < s1; t0 += TG) {
            commit();
            if (t0 + TG < s1) fetch(t0 + TG, 1, a.la_f, a.la_b);
#pragma unroll
            for (int n = 0; n < TG; ++n) {
                const float4 r4 = rec[n * kRows + i];
                const float hq = 0.5f * r4.y;
                ds *= r4.z;
                dz *= r4.w;
                if (n > 0 || t0 > s0) {
                    ps *= r4.z;
                    pz *= r4.w;
                }
                const f32x2 ds2 = pack2(r4.z, r4.z), dz2 = pack2(r4.w, r4.w), k2 = pack2(r4.x, r4.x), q2 = pack2(hq, hq);
                const f32x2 pk2 = pack2(pz * r4.x, pz * r4.x), pq2 = pack2(ps * hq, ps * hq);
                const ulonglong2* vp = reinterpret_cast<const ulonglong2*>(vs + n * kPitch + cg * (CN + 4));
                const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(gs + n * kPitch + cg * (CN + 4));
#pragma unroll
                for (int c4 = 0; c4 < CN / 4; ++c4) {
                    const ulonglong2 v2 = vp[c4], g2 = gp[c4];
                    const f32x2 vq[2] = {v2.x, v2.y}, gq[2] = {g2.x, g2.y};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int c = 2 * c4 + h;
                        S[c] = ffma2(ds2, S[c], fmul2(k2, vq[h]));
                        Z[c] = ffma2(dz2, Z[c], fmul2(q2, gq[h]));
                        R[c] = ffma2(pk2, vq[h], R[c]);
                        Y[c] = ffma2(pq2, gq[h], Y[c]);
                    }
                }
            }
        }
        // the decays of what enters from the right take the gate at the border as well
        pz *= row < dk ? expf(rec_to_float(a.la_b[ok + (size_t)(s1 - 1) * dk + row])) : 1.f;
        ps *= row < dk && s1 < L ? expf(rec_to_float(a.la_f[ok + (size_t)s1 * dk + row])) : 1.f;
#pragma unroll
        for (int x = 0; x < CN / 4; ++x) {
            st[((w * 4 + 0) * (CN / 4) + x) * 32 + lane] = make_ulonglong2(S[2 * x], S[2 * x + 1]);
            st[((w * 4 + 1) * (CN / 4) + x) * 32 + lane] = make_ulonglong2(Z[2 * x], Z[2 * x + 1]);
            st[((w * 4 + 2) * (CN / 4) + x) * 32 + lane] = make_ulonglong2(R[2 * x], R[2 * x + 1]);
            st[((w * 4 + 3) * (CN / 4) + x) * 32 + lane] = make_ulonglong2(Y[2 * x], Y[2 * x + 1]);
        }
        if (cg == 0) {
            dec[(w * 4 + 0) * kRows + i] = ds;
            dec[(w * 4 + 1) * kRows + i] = dz;
            dec[(w * 4 + 2) * kRows + i] = pz;
            dec[(w * 4 + 3) * kRows + i] = ps;
        }
    }
    if (split) __syncthreads();
    if (!on) return;
    // the state of kind `kind` (S>, Z<, S<, Z>) that enters this segment
    auto enter = [&](int kind, f32x2 (&to)[C2]) {
#pragma unroll
        for (int c = 0; c < C2; ++c) to[c] = 0ull;
        if (!split) return;
        for (int s = kind < 2 ? 0 : nw - 1; s != w; s += kind < 2 ? 1 : -1) {
            const float d = dec[(s * 4 + kind) * kRows + i];
            const f32x2 d2 = pack2(d, d);
#pragma unroll
            for (int x = 0; x < CN / 4; ++x) {
                const ulonglong2 e = st[((s * 4 + kind) * (CN / 4) + x) * 32 + lane];
                to[2 * x] = ffma2(d2, to[2 * x], e.x);
                to[2 * x + 1] = ffma2(d2, to[2 * x + 1], e.y);
            }
        }
    };
    enter(0, S);
    enter(1, Z);

    float run_f = 0.f, run_b = 0.f;   // sums of E> and E< over the tokens walked down so far
#pragma unroll 1
    for (int walk = 0; walk < 2; ++walk) {
        const int step = walk == 0 ? 1 : -1, first = walk == 0 ? s0 : s1 - 1;
        const T* las = walk == 0 ? a.la_f : a.la_b;
        const T* laz = walk == 0 ? a.la_b : a.la_f;
        fetch(first, step, las, laz);
        if (walk == 1) {
            // S>, Z< of the last token meet the states from the right
            f32x2 X[C2], sb = 0ull, sf = 0ull;
            enter(2, X);
#pragma unroll
            for (int c = 0; c < C2; ++c) {
                sb = ffma2(Z[c], X[c], sb);
                Z[c] = X[c];
            }
            enter(3, X);
#pragma unroll
            for (int c = 0; c < C2; ++c) {
                sf = ffma2(S[c], X[c], sf);
                S[c] = Z[c];
                Z[c] = X[c];
            }
            if (split) {
                float f = sum2(sf), b = sum2(sb);
                f += __shfl_xor_sync(0xffffffffu, f, 1);
                b += __shfl_xor_sync(0xffffffffu, b, 1);
                f += __shfl_xor_sync(0xffffffffu, f, 2);
                b += __shfl_xor_sync(0xffffffffu, b, 2);
                run_f = row < dk && s1 < L ? f * expf(rec_to_float(a.la_f[ok + (size_t)s1 * dk + row])) : 0.f;
                run_b = row < dk ? -b * expf(rec_to_float(a.la_b[ok + (size_t)(s1 - 1) * dk + row])) : 0.f;
            }
        }
        for (int m = 0; m < s1 - s0; m += TG) {
            const int base = first + step * m;
            commit();
            if (m + TG < s1 - s0) fetch(base + step * TG, step, las, laz);
            // this lane finishes token cg of the four: dq>, dk< of the ascending walk
            const int t = base + step * cg;
            const bool mine = t >= s0 && t < s1 && row < dk;
            const size_t e = ok + (size_t)t * dk + row;
            float2 x2 = make_float2(0.f, 0.f);
            if (walk == 1 && mine) x2 = pairs.get(e);
            float y[TG][2];
#pragma unroll
            for (int n = 0; n < TG; ++n) {
                const float4 r4 = rec[n * kRows + i];
                const float hq = 0.5f * r4.y;
                const f32x2 ds2 = pack2(r4.z, r4.z), dz2 = pack2(r4.w, r4.w), k2 = pack2(r4.x, r4.x), q2 = pack2(hq, hq);
                const ulonglong2* vp = reinterpret_cast<const ulonglong2*>(vs + n * kPitch + cg * (CN + 4));
                const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(gs + n * kPitch + cg * (CN + 4));
                f32x2 aq[2] = {0ull, 0ull}, ak[2] = {0ull, 0ull};
#pragma unroll
                for (int c4 = 0; c4 < CN / 4; ++c4) {
                    const ulonglong2 v2 = vp[c4], g2 = gp[c4];
                    const f32x2 vq[2] = {v2.x, v2.y}, gq[2] = {g2.x, g2.y};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int c = 2 * c4 + h;
                        S[c] = ffma2(ds2, S[c], fmul2(k2, vq[h]));   // S_t = a S + k^T v
                        aq[h] = ffma2(S[c], gq[h], aq[h]);           // S_t g^T
                        Z[c] = ffma2(dz2, Z[c], fmul2(q2, gq[h]));   // Z_t = a' Z + q^T g / 2
                        ak[h] = ffma2(Z[c], vq[h], ak[h]);           // Z_t v^T
                    }
                }
                y[n][0] = sum2(fadd2(aq[0], aq[1]));
                y[n][1] = sum2(fadd2(ak[0], ak[1]));
            }
            // sums over the four lanes of a row, token n to lane n
            float h2[2][2], acc[2];
            const bool hi = cg & 2, odd = cg & 1;
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int h = 0; h < 2; ++h) h2[n][h] = (hi ? y[n + 2][h] : y[n][h]) + __shfl_xor_sync(0xffffffffu, hi ? y[n][h] : y[n + 2][h], 2);
#pragma unroll
            for (int h = 0; h < 2; ++h) acc[h] = (odd ? h2[1][h] : h2[0][h]) + __shfl_xor_sync(0xffffffffu, odd ? h2[0][h] : h2[1][h], 1);
            const float accq = 0.5f * acc[0], acck = acc[1];
            if (walk == 0) {
                if (mine) pairs.put(e, make_float2(accq, acck));   // (the same lane reads it back)
            } else {   // accq = dq<_t, acck = dk>_t
                const float4 r4 = rec[cg * kRows + i];
                const float ef = r4.y * x2.x - r4.x * acck, eb = r4.y * accq - r4.x * x2.y;
                float f = ef, b = eb;   // inclusive sums over the four tokens
#pragma unroll
                for (int d = 1; d <= 2; d <<= 1) {
                    const float fu = __shfl_up_sync(0xffffffffu, f, d, 4), bu = __shfl_up_sync(0xffffffffu, b, d, 4);
                    if (cg >= d) {
                        f += fu;
                        b += bu;
                    }
                }
                if (mine) {
                    rec_store(a.dq + e, x2.x + accq);
                    rec_store(a.dkey + e, acck + x2.y);
                    rec_store(a.dla_f + e, run_f + f);
                    rec_store(a.dla_b + e, -(run_b + (b - eb)));
                }
                run_f += __shfl_sync(0xffffffffu, f, 3, 4);
                run_b += __shfl_sync(0xffffffffu, b, 3, 4);
            }
        }
    }
}

}  // namespace scan
}  // namespace vig
