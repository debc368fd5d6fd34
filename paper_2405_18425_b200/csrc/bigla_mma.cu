// bf16 BiGLA forward on the warp-level tensor-core instructions (mma.sync): one warp per 16 tokens, every product a chain of
// 16 x 16 tiles whose scores stay in registers.  Units of at most 256 tokens are one block each (a cluster of two, large
// states of few units); longer sequences are cut
// into chunks of up to 128 tokens, one block each.  Up to eight chunks (1024 tokens): one launch, a cluster of blocks per unit, each of
// which gives the others the state it adds through distributed shared memory.  Any length: three launches, the state every chunk adds in
// either direction, a fold over the chunks, the chunks themselves from the states that enter them.
//
// With b_t the inclusive prefix sum of log alpha> and x_t the exclusive prefix sum of log alpha< (the backward decay from t
// to s > t is exp(x_s - x_t): the gates t .. s-1), both from the start of a chunk of 128 tokens, Eq. 6 is, per chunk,
//     q~> = q e^{b} / 2,  k~> = k e^{-b},  q~< = q e^{-x} / 2,  k~< = k e^{x}
//     out_t = sum_{s <= t} (q~>_t k~>_s) v_s + sum_{s >= t} (q~<_t k~<_s) v_s + q~ S
// with S the state the other chunk of the unit hands over (k~>^T v of chunk 0 forward, k~<^T v of chunk 1 backward, either
// times the whole decay of chunk 0).
//
// A warp reads its rows of q, k and the gates straight into fragment order, takes their prefix sums as products with a
// 16 x 16 triangle of ones (fp32 accumulation of bf16 values: exact up to fp32 addition), leaves k~ in shared memory and
// keeps q~ in registers; v comes by one TMA load.  Then it runs over the tiles of its chunk: scores, packed to bf16 as the A
// operand of the product with v.  Two block barriers (gate totals, k~) and one mbarrier (states) order the warps.
//
// What bounds it: with one block per SM the latency of that chain (4.5 us at 100 tokens, 6.5 us at 196), with more of them
// instruction issue (about 1600 warp instructions per warp at 196 tokens, 32 x 64), so registers are held to what lets two
// blocks of thirteen or sixteen warps, or three of eight, share an SM.  Against the tcgen05 form (two 128-row chunk
// pipelines per block, whose hand-overs between tensor-core batches bound it): 148 units of 49 tokens 3.1 us to 6.2, 768 of
// 128 tokens 14.9 to 24.5 (24 x 48), 1536 of 196 tokens 53.6 to 61.9 (24 x 48); mma_preferred holds the shapes it loses.
#include <cuda.h>

#include <atomic>
#include <type_traits>

#include "fold.cuh"
#include "mma.cuh"
#include "recurrence.cuh"
#include "tma_host.h"
#include "vig_internal.h"

namespace vig {
namespace {

using namespace wmma16;

#pragma nv_diag_suppress 128   // the summary instances return half way: the loops behind that are not reachable in them

enum { kUnit = 0, kSummary = 1, kMain = 2, kCluster = 3 };
constexpr int kChunkTiles = 8;        // 16-token tiles of a chunk at most
constexpr float kGateRange = 60.f;    // largest decay of a chunk, as -log, that the factorised tiles take

struct MArgs {
    const __nv_bfloat16 *q, *k, *v, *la_f, *la_b;   // GATES: la_f / la_b hold the gate logits
    __nv_bfloat16* out;
    int L;
    long long blocks;  // units (kUnit) or units x chunks
    int nch, tiles;    // chunks per unit, tiles per chunk (long sequences)
    int* dev_status;
    float inv_tau;
    int ahead;         // the block this many further on has its inputs pulled into L2
    int expire_wait;   // test hook: every block lets one bounded wait, on an mbarrier nothing completes, run out
};
// What chunks have beside it.  Units of one block do without: with everything in one struct the compiler lets their instances keep fewer of
// the parameters in registers and put up to 92 bytes a thread on the stack instead of up to 40 (202 units of 187 tokens, 16 x 64: 8.5 us,
// 7.9 this way); clusters are the faster ones with it (24 x 6 units of 300, 32 x 64: 18.6 us, 20.5 without).
struct MChunkArgs : MArgs {
    long long units;
    float* u;          // [unit][chunk][S>, S<][DV][DK] fp32: what a chunk adds to the states, key dimensions in fragment order
    uint8_t* img;      // [unit][chunk][S>, S<][DV][64 B]: the states that enter a chunk, as shared-memory tiles
    float* decay;      // [unit][chunk][2][32]: products of alpha over the chunk
    int* flags;        // [unit][chunk]: 1: gates out of range, 2: not computed (a wait ran out)
};
template <int MODE>
using ArgsOf = std::conditional_t<MODE == kUnit, MArgs, MChunkArgs>;

// Shared memory: v [rows][RV], k~> and k~< [rows][64 B], the two states [DV][64 B], gate totals [tile][2][32] fp32; chunks of a
// cluster: a slot for each of the other chunks (the state it adds, [DV][DK] fp32, its decay [DK] and a status word), then the
// decay of its own that it needs.
template <int DV>
struct MLayout {
    static constexpr uint32_t kVRow = DV == 32 ? 64 : 128, kState = DV * 64;
    uint32_t kf, kb, st, totals, slots, bar, total;
    __host__ __device__ MLayout(int tiles, bool states, uint32_t slot_bytes = 0) {
        const uint32_t rows = tiles * 16u;
        kf = rows * kVRow;
        kb = kf + rows * 64;
        st = kb + rows * 64;
        totals = st + (states ? 2 * kState : 0);
        slots = totals + tiles * 256u;
        bar = slots + slot_bytes;
        total = bar + 64;
    }
};
constexpr uint32_t slot_bytes(int dk, int dv) { return dv * dk * 4u + 144u; }   // (the decay behind the state, the word 128 bytes on)
constexpr uint32_t all_slots(int dk, int dv, int nch) { return (nch - 1) * slot_bytes(dk, dv) + 128u; }

// Blocks per SM the registers are held to (64 registers a thread for four: 19 us against 15 where the state is large, units of one block,
// 768 of 100 tokens, 32 x 64; chunks of small states gain, 2 x 4 units of 16384 tokens, 24 x 48: 39.8 to 38.5, though at 24 x 48 and
// 32 x 32 some 50 bytes a thread go to the stack; from five chunks on the slots of a cluster leave room for three blocks only).
constexpr int mma_blocks_per_sm(int dk, int dv, int max_tiles, int mode) {
    return max_tiles > 8 ? 2 : (mode != kUnit && dk * dv <= 1152 ? 4 : 3);
}

template <int DK, int DV, bool GATES, int MAXT, int MODE>
__global__ void __launch_bounds__(MAXT * 32, mma_blocks_per_sm(DK, DV, MAXT, MODE)) bigla_mma_kernel(const __grid_constant__ CUtensorMap tm_v, const ArgsOf<MODE> args) {
    constexpr int NP = DK / 8, MP = (NP + 1) / 2;   // 8-column tiles of the key dimensions, pairs of them
    constexpr int NV = DV / 8, MV = DV / 16;        // ... of the value dimensions
    constexpr int RV = MLayout<DV>::kVRow;
    constexpr uint32_t kState = MLayout<DV>::kState;
    constexpr bool kTwo = MODE == kUnit && MAXT > 8;   // units of two chunks
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, w = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int g = lane >> 2, c = lane & 3;
    const int L = args.L, nch = MODE == kUnit ? 1 : args.nch;
    const int chunk = MODE == kUnit ? 0 : (int)(blockIdx.x % (unsigned)nch);
    const size_t unit = MODE == kUnit ? blockIdx.x : blockIdx.x / (unsigned)nch;
    const int Tall = (L + 15) >> 4, tiles = MODE == kUnit ? Tall : args.tiles;
    const int tok0 = chunk * tiles * 16, T = min(tiles, Tall - chunk * tiles);   // this block's first token and its tiles
    const bool live = w < T;                          // (blocks have two warps at least: the in-kernel recurrence needs them)
    const int ch = kTwo ? w >> 3 : 0, c0 = 8 * ch;    // this warp's chunk and its first tile
    const MLayout<DV> lay(tiles, kTwo ? Tall > 8 : MODE == kMain || MODE == kCluster, MODE == kCluster ? all_slots(DK, DV, nch) : 0u);
    const uint32_t base = smem_u32(smem), tv = base, tkf = base + lay.kf, tkb = base + lay.kb, tst = base + lay.st, bar = base + lay.bar;
    float* totals = reinterpret_cast<float*>(smem + lay.totals);
    volatile int* slow = reinterpret_cast<volatile int*>(smem + lay.bar + 32);

    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 8, MODE == kMain || MODE == kCluster ? 1 : 2 * MV);   // the states: one bulk copy, the other chunks' slots, or one arrival per piece formed here
        mbar_init(bar + 16, 1);       // never completed: only the test hook waits on it
        *slow = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    auto pull = [&](size_t at, uint32_t n) {   // n tokens from `at` into L2
        prefetch_l2(args.la_f + at * DK, n * DK * 2);
        prefetch_l2(args.la_b + at * DK, n * DK * 2);
        prefetch_l2(args.k + at * DK, n * DK * 2);
        prefetch_l2(args.v + at * DV, n * DV * 2);
        prefetch_l2(args.q + at * DK, n * DK * 2);
    };
    // A block that is let in while the launch before still runs has its tokens brought to L2 meanwhile (a prefetch consumes nothing,
    // and L2 stays coherent with what that launch still writes); the blocks after the first round are pulled in by those of it.
    if (MODE != kMain && tid == 32 && (int)blockIdx.x < args.ahead) pull(unit * L + tok0, min(tiles * 16, L - tok0));
    // The chunks' launch starts under the fold: that one lets it in only behind its own wait, when the summaries are complete, and
    // with them all that was launched before.  So inputs and flags are read at once, from L2 (see pdl_wait), and only what the fold
    // writes is waited for.
    if (MODE != kMain) {
        pdl_wait();
        pdl_launch_dependents();
    }
    if (tid == 0) {
        mbar_expect_tx(bar, (uint32_t)tiles * 16 * RV);
        tma_load_3d(tv, &tm_v, 0, tok0, (int)unit, bar);   // rows >= L and columns >= DV arrive as zeros
        if (MODE == kCluster) mbar_expect_tx(bar + 8, (nch - 1) * (DV * DK * 4 + DK * 4 + 4));
    }

    // ---- this warp's 16 rows (g and g + 8) in fragment order: pair j of lane c ----
    uint32_t qr[2][NP], kr[2][NP], af[2][NP], ab[2][NP];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int row = tok0 + w * 16 + 8 * r + g;
        if (live && row < L) {
            const size_t at = (unit * L + row) * DK;
            load_pairs<DK, MODE == kMain>(args.la_f + at, c, af[r]);
            load_pairs<DK, MODE == kMain>(args.la_b + at, c, ab[r]);
            load_pairs<DK, MODE == kMain>(args.k + at, c, kr[r]);
            if (MODE != kSummary) load_pairs<DK, MODE == kMain>(args.q + at, c, qr[r]);
        } else {
#pragma unroll
            for (int j = 0; j < NP; ++j) {   // rows past the end: q = k = 0 and no decay (GATES: a logit of 100, log alpha = 0)
                qr[r][j] = kr[r][j] = 0u;
                af[r][j] = ab[r][j] = GATES ? 0x42C842C8u : 0u;
            }
        }
    }
    if (MODE != kMain && tid == 0 && blockIdx.x + (long long)args.ahead < args.blocks) {   // a block that starts when one of these is done finds its inputs in L2
        const size_t next = blockIdx.x + (size_t)args.ahead;
        const int nr = MODE == kUnit ? 0 : (int)(next % (unsigned)nch) * tiles * 16;
        pull((MODE == kUnit ? next : next / (unsigned)nch) * L + nr, min(tiles * 16, L - nr));   // (q: for the chunks' launch as well)
    }
    // ---- gate totals of the tile; the gates turned, as B operands of products over the tokens ----
    auto prepare = [&](int r, int j) {
        if (GATES) {
            af[r][j] = log2_alpha_pair<MODE != kUnit>(af[r][j], args.inv_tau);
            ab[r][j] = log2_alpha_pair<MODE != kUnit>(ab[r][j], args.inv_tau);
        }
    };
    if (MODE == kCluster) {   // (all of them first: 12 bytes a thread on the stack at 32 x 64 instead of 52; elsewhere as they are turned: 12 instead of 24 at 24 x 48)
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int r = 0; r < 2; ++r) prepare(r, j);
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (MODE != kCluster) prepare(r, j);
            af[r][j] = movmatrix(af[r][j]);
            ab[r][j] = movmatrix(ab[r][j]);
        }
        float tf[4], tb[4];
        mma_k16_from(tf, kOnes, kOnes, kOnes, kOnes, af[0][j], af[1][j], 0.f, 0.f);
        mma_k16_from(tb, kOnes, kOnes, kOnes, kOnes, ab[0][j], ab[1][j], 0.f, 0.f);
        if (g == 0 && live) {
            *reinterpret_cast<float2*>(totals + (w * 2) * 32 + 8 * j + 2 * c) = make_float2(tf[0], tf[1]);
            *reinterpret_cast<float2*>(totals + (w * 2 + 1) * 32 + 8 * j + 2 * c) = make_float2(tb[0], tb[1]);
        }
    }
    __syncthreads();
    if (MODE == kCluster) cluster_arrive_relaxed();   // the other chunks may write here once this one's barriers stand
    // sums over tiles [from, to) of one direction
    auto sum_totals = [&](int dir, int from, int to, f32x2 (&s)[NP]) {
#pragma unroll
        for (int j = 0; j < NP; ++j) s[j] = 0ull;   // (+0, +0)
        const float* p = totals + (from * 2 + dir) * 32 + 2 * c;
#pragma unroll 1
        for (int x = from; x < to; ++x, p += 64)
#pragma unroll
            for (int j = 0; j < NP; ++j) s[j] = fadd2(s[j], *reinterpret_cast<const f32x2*>(p + 8 * j));
    };
    if (w == T - 1 && lane < DK) {   // range check: the decay of each chunk per key dim and direction
#pragma unroll
        for (int h = 0; h < (kTwo ? 2 : 1); ++h)
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                float s = 0.f;
                for (int x = 8 * h; x < min(T, 8 * h + 8); ++x) s += totals[(x * 2 + d) * 32 + lane];
                if (!(s >= -kGateRange * (GATES ? kLog2e : 1.f))) *slow = 1;
            }
    }
    // ---- prefix sums from the start of the chunk and scaled operands: k~ to shared memory, q~ in registers ----
    uint32_t qf[MP][4], qb[MP][4];
    if (live) {
        const uint32_t tri_i = triangle(g, c, true), tri_x = triangle(g, c, false);
        const Tile<64> t64(lane);
        f32x2 cf[NP], cb[NP];
        sum_totals(0, c0, w, cf);
        sum_totals(1, c0, w, cb);
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            uint32_t kfw[4], kbw[4];
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                const int j = 2 * m + jj;
                if (j < NP) {
                    float b[4], x[4], f0, f1, e0, e1;
                    unpack2(cf[j], f0, f1);
                    unpack2(cb[j], e0, e1);
                    mma_k16_from(b, tri_i, kOnes, 0u, tri_i, af[0][j], af[1][j], f0, f1);
                    mma_k16_from(x, tri_x, kOnes, 0u, tri_x, ab[0][j], ab[1][j], e0, e1);
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        float b0 = b[2 * r], b1 = b[2 * r + 1], x0 = x[2 * r], x1 = x[2 * r + 1];
                        if constexpr (!GATES) {   // natural logarithms in
                            unpack2(fmul2(pack2(b0, b1), pack2(kLog2e, kLog2e)), b0, b1);
                            unpack2(fmul2(pack2(x0, x1), pack2(kLog2e, kLog2e)), x0, x1);
                        }
                        if constexpr (MODE == kUnit) {
                            // the decaying factors on the special-function unit, the growing ones as their packed reciprocals
                            const uint32_t ef = pack_bf16(ex2(b0), ex2(b1)), eb = pack_bf16(ex2(x0), ex2(x1));
                            const uint32_t hq = mul_bf16x2(qr[r][j], 0x3F003F00u);   // the 1/2 of the result: exact
                            kfw[2 * jj + r] = mul_bf16x2(kr[r][j], rcp_bf16x2(ef));
                            kbw[2 * jj + r] = mul_bf16x2(kr[r][j], eb);
                            qf[m][2 * jj + r] = mul_bf16x2(hq, ef);
                            qb[m][2 * jj + r] = mul_bf16x2(hq, rcp_bf16x2(eb));
                        } else {
                            // Factor and product in fp32, one rounding: what the packed reciprocals are low by on average would
                            // pass into the states and on from chunk to chunk (with them 32 x 4096 tokens, gate logits around 4,
                            // were 4.8e-3 off in 2-norm, the tcgen05 forms 4.5e-3; this way 3.3e-3 in the same time).
                            const f32x2 k2 = widen(kr[r][j]);
                            kfw[2 * jj + r] = pack_f32x2(fmul2(k2, pack2(ex2(-b0), ex2(-b1))));
                            kbw[2 * jj + r] = pack_f32x2(fmul2(k2, pack2(ex2(x0), ex2(x1))));
                            if (MODE != kSummary) {
                                const f32x2 q2 = fmul2(widen(qr[r][j]), pack2(0.5f, 0.5f));   // the 1/2 of the result
                                qf[m][2 * jj + r] = pack_f32x2(fmul2(q2, pack2(ex2(b0), ex2(b1))));
                                qb[m][2 * jj + r] = pack_f32x2(fmul2(q2, pack2(ex2(-x0), ex2(-x1))));
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < 2; ++r) kfw[2 + r] = kbw[2 + r] = qf[m][2 + r] = qb[m][2 + r] = 0u;
                }
            }
            t64.store(tkf, 16 * w, m, kfw[0], kfw[1], kfw[2], kfw[3]);
            t64.store(tkb, 16 * w, m, kbw[0], kbw[1], kbw[2], kbw[3]);
        }
    }
    bool ok = true;
    if (args.expire_wait && tid == 0) ok = mbar_wait_bounded(bar + 16, 0, 64);   // test hook: this wait cannot succeed
    ok = mbar_wait_bounded(bar, 0) && ok;
    ok = __syncthreads_and(ok);
    if (MODE == kCluster) {
        cluster_wait();
    } else if (!ok) {   // a load that never lands: report it and leave, all threads together, nothing stored
        if (tid == 0) atomicOr(args.dev_status, kDevStatusTimeout);
        if constexpr (MODE == kSummary) {
            if (tid == 0) args.flags[blockIdx.x] = 2;   // (nor by the launches behind this one)
        }
        if (MODE == kMain) pdl_wait();   // (no block ends before the fold: what comes next only waits for this launch)
        return;
    }
    if constexpr (MODE == kSummary) {
        if (tid < 64 && (tid & 31) < DK) {   // (at least two warps)
            float s = 0.f;
            for (int x = 0; x < T; ++x) s += totals[(x * 2 + (tid >> 5)) * 32 + (tid & 31)];
            args.decay[(size_t)blockIdx.x * 64 + tid] = ex2(GATES ? s : s * kLog2e);
            if (tid == 0) args.flags[blockIdx.x] = *slow;
        }
    }
    bool redo = MODE == kUnit && *slow;
    if constexpr (MODE == kMain) {
        int any = 0;
        for (int x = tid; x < nch; x += blockDim.x) any |= (int)ld_gpu4(args.flags + unit * nch + x);
        const bool missing = __syncthreads_or(any & 2);
        redo = __syncthreads_or(any);
        if (w == 0 || redo) pdl_wait();   // the fold
        if (missing) return;   // a summary of this unit did not get its inputs, and has said so
        if (tid == 0 && !redo) {
            pdl_launch_dependents();
            mbar_expect_tx(bar + 8, 2 * kState);
            bulk_load(tst, args.img + (size_t)blockIdx.x * 2 * kState, 2 * kState, bar + 8);
        }
    }
    if (redo) {   // gates beyond the range of the factorised tiles: Eq. 6 step by step, over the dead tiles, by one block of the unit
        if (chunk != 0) return;
        if (tid == 0) atomicAdd(args.dev_status + 1, 1);
        __syncthreads();
        const size_t okk = unit * L * DK, ov = unit * L * DV;
        recurrence_unit<__nv_bfloat16>(args.q + okk, args.k + okk, args.v + ov, args.la_f + okk, args.la_b + okk, args.out + ov, L, DK, DV,
                                       reinterpret_cast<float*>(smem), args.inv_tau);
        return;
    }
    if (MODE != kCluster && !live) return;
    const Tile<64> t64(lane);
    const Tile<RV> tvv(lane);
    float* slots = reinterpret_cast<float*>(smem + lay.slots);
    constexpr int kSlotFloats = slot_bytes(DK, DV) / 4, kStateFloats = DV * DK;
    // Place of a key dimension (a column of the operand tiles) in a row of a slot: pairs of a lane's pairs side by side.
    auto slot_place = [](int col) {
        const int j = col >> 3, m = j >> 1, cc = (col & 7) >> 1;
        return 16 * m + (2 * m + 1 < NP ? 4 * cc + 2 * (j & 1) : 2 * cc) + (col & 1);
    };

    // ---- the states the chunks hand each other, transposed: rows of v times k~ over the tokens, 16 value columns a job; the
    // last warps first: theirs is the shorter chunk ----
    if (MODE == kSummary || MODE == kCluster || (kTwo && T > 8)) {
        // (in a cluster the first chunk owes nobody S<, the last nobody S>)
        const int dirs = MODE == kCluster ? (chunk > 0) + (chunk + 1 < nch) : 2;
        for (int job = live ? T - 1 - w : 2 * MV; job < dirs * MV; job += T) {
            const int dir = dirs == 2 ? job & 1 : (chunk == 0 ? 0 : 1), mt = dirs == 2 ? job >> 1 : job;   // two chunks: dir 0: chunk 0 -> 1 (forward), dir 1: chunk 1 -> 0
            const int t0 = !kTwo || dir == 0 ? 0 : 8, t1 = kTwo && dir == 0 ? 8 : T;
            float u[2 * MP][4];
#pragma unroll
            for (int j = 0; j < 2 * MP; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) u[j][e] = 0.f;
            uint32_t left = tv + t0 * 16 * RV + (tvv.off_b[0] ^ (uint32_t)(mt << 5));   // (the piece bits of an offset are its swizzle alone)
            uint32_t right = (dir == 0 ? tkf : tkb) + t0 * 1024;
#pragma unroll 2
            for (int t = t0; t < t1; ++t, left += 16 * RV, right += 1024) {
                uint32_t va[4];
                ldsm_trans(left, va);
#pragma unroll
                for (int m = 0; m < MP; ++m) {
                    uint32_t h[4];
                    t64.load_trans(right, 0, m, h);
                    mma_k16(u[2 * m], va, h[0], h[1]);
                    if (2 * m + 1 < NP) mma_k16(u[2 * m + 1], va, h[2], h[3]);
                }
            }
            f32x2 dec[NP];
            sum_totals(dir, 0, min(T, 8), dec);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                // two chunks: times chunk 0's decay, of what it leaves behind (forward), of what it takes in (backward); long
                // sequences: the forward state alone decays to the chunk's end
                float d0, d1;
                unpack2(GATES ? dec[j] : fmul2(dec[j], pack2(kLog2e, kLog2e)), d0, d1);
                d0 = !kTwo && dir == 1 ? 1.f : ex2(d0);
                d1 = !kTwo && dir == 1 ? 1.f : ex2(d1);
                if (MODE == kCluster) {
                    u[j][0] *= d0; u[j][1] *= d1; u[j][2] *= d0; u[j][3] *= d1;
                    continue;
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int n = 16 * mt + 8 * r + g;
                    const float u0 = u[j][2 * r] * d0, u1 = u[j][2 * r + 1] * d1;
                    if constexpr (MODE == kSummary)
                        *reinterpret_cast<float2*>(args.u + (((size_t)blockIdx.x * 2 + dir) * DV + n) * DK + 8 * j + 2 * c) = make_float2(u0, u1);
                    else
                        *reinterpret_cast<uint32_t*>(smem + lay.st + dir * kState + n * 64 + ((j ^ ((n >> 1) & 3)) << 4) + 4 * c) = pack_bf16(u0, u1);
                }
            }
            if (MODE == kCluster) {   // to every chunk behind (S>) or before (S<) this one
                const int p0 = dir == 0 ? chunk + 1 : 0, p1 = dir == 0 ? nch : chunk;
                const uint32_t at = base + lay.slots + (dir == 0 ? chunk : chunk - 1) * slot_bytes(DK, DV) + (16 * mt + g) * (DK * 4);
#pragma unroll 1
                for (int p = p0; p < p1; ++p) {
                    const uint32_t to = cluster_peer(at, p), peer_bar = cluster_peer(bar + 8, p);
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int m = 0; m < MP; ++m) {
                            if (2 * m + 1 < NP)
                                st_async4(to + 8 * r * DK * 4 + 64 * m + 16 * c, __float_as_uint(u[2 * m][2 * r]), __float_as_uint(u[2 * m][2 * r + 1]),
                                          __float_as_uint(u[2 * m + 1][2 * r]), __float_as_uint(u[2 * m + 1][2 * r + 1]), peer_bar);
                            else
                                st_async2(to + 8 * r * DK * 4 + 64 * m + 8 * c, __float_as_uint(u[2 * m][2 * r]), __float_as_uint(u[2 * m][2 * r + 1]), peer_bar);
                        }
                }
            }
            __syncwarp();
            if (kTwo && lane == 0) mbar_arrive(bar + 8);
        }
        if (MODE == kSummary) return;
    }
    if (MODE == kCluster && w == 0) {   // the decay across this chunk, and whether anything is wrong here
        const int word = (*slow ? 1 : 0) | (ok ? 0 : 2);
        if (lane < DK) {
            float s0 = 0.f, s1 = 0.f;
            for (int x = 0; x < T; ++x) {
                s0 += totals[(x * 2) * 32 + lane];
                s1 += totals[(x * 2 + 1) * 32 + lane];
            }
            s0 = ex2(GATES ? s0 : s0 * kLog2e);
            s1 = ex2(GATES ? s1 : s1 * kLog2e);
            slots[(nch - 1) * kSlotFloats + slot_place(lane)] = s1;   // its own, of S< across this chunk
#pragma unroll 1
            for (int p = 0; p < nch; ++p) {
                if (p == chunk) continue;
                const uint32_t at = base + lay.slots + (p > chunk ? chunk : chunk - 1) * slot_bytes(DK, DV) + kStateFloats * 4;
                const uint32_t peer_bar = cluster_peer(bar + 8, p);
                st_async1(cluster_peer(at + slot_place(lane) * 4, p), __float_as_uint(p > chunk ? s0 : s1), peer_bar);
                if (lane == 0) st_async1(cluster_peer(at + 128, p), (uint32_t)word, peer_bar);
            }
        }
    }

    // ---- this warp's rows against the tiles of its chunk: forward products up to the diagonal tile, backward ones from it on
    // (loops without the masks and the change of operands in them: those cost as many instructions as the products) ----
    float o[NV][4];
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
    const DiagonalMask dmask(g, c);
    const int nT = min(T - c0, 8), mine = w - c0;
    // one tile of keys: scores with q~ (in qq), keep: 0 all of them, 1 columns up to the row, 2 columns from the row on
    auto tile = [&](const uint32_t (&qq)[MP][4], uint32_t kt, uint32_t vt, int keep) {
        float d0[4], d1[4];
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            uint32_t r[4];
            t64.load_b(kt, 0, m, r);
            if (m == 0) {
                mma_k16_zero(d0, qq[0], r[0], r[1]);
                mma_k16_zero(d1, qq[0], r[2], r[3]);
            } else if (2 * m + 1 < NP) {
                mma_k16(d0, qq[m], r[0], r[1]);
                mma_k16(d1, qq[m], r[2], r[3]);
            } else {
                mma_k8(d0, qq[m][0], qq[m][1], r[0]);
                mma_k8(d1, qq[m][0], qq[m][1], r[2]);
            }
        }
        uint32_t p[4] = {pack_bf16(d0[0], d0[1]), pack_bf16(d0[2], d0[3]), pack_bf16(d1[0], d1[1]), pack_bf16(d1[2], d1[3])};
        if (keep) dmask.apply(p, keep == 1);
#pragma unroll
        for (int n2 = 0; n2 < MV; ++n2) {
            uint32_t r[4];
            tvv.load_trans(vt, 0, n2, r);
            mma_k16(o[2 * n2], p, r[0], r[1]);
            mma_k16(o[2 * n2 + 1], p, r[2], r[3]);
        }
    };
    if (live) {
        uint32_t kt = tkf + (uint32_t)c0 * 1024, vt = tv + (uint32_t)c0 * 16 * RV;
#pragma unroll 1
        for (int j = 0; j < mine; ++j, kt += 1024, vt += 16 * RV) tile(qf, kt, vt, 0);
        tile(qf, kt, vt, 1);
        kt += tkb - tkf;
        tile(qb, kt, vt, 2);
#pragma unroll 1
        for (int j = mine + 1; j < nT; ++j) {
            kt += 1024;
            vt += 16 * RV;
            tile(qb, kt, vt, 0);
        }
    }
    if (MODE == kCluster) {
        // ---- the states that enter this chunk, from what the chunks before and behind it add: in(c + 1) = d>(c) in(c) + own(c),
        // in(c - 1) = d<(c) in(c) + own(c), the latter stored times this chunk's d<, as the fold of the long form does ----
        const bool got = __syncthreads_and(mbar_wait_bounded(bar + 8, 0) && ok);
        int word = got ? *slow : 2;
        for (int x = 0; got && x + 1 < nch; ++x) word |= *reinterpret_cast<const int*>(slots + x * kSlotFloats + kStateFloats + 32);
        if (word) {   // (every block has all that is sent to it by now, so none is written to after its end)
            if (word & 2) {
                if (tid == 0) atomicOr(args.dev_status, kDevStatusTimeout);
                return;
            }
            if (chunk != (int)(unit % (unsigned)nch)) return;   // (the first blocks of clusters share SMs)
            if (tid == 0) atomicAdd(args.dev_status + 1, 1);
            __syncthreads();
            const size_t okk = unit * L * DK, ov = unit * L * DV;
            recurrence_unit<__nv_bfloat16>(args.q + okk, args.k + okk, args.v + ov, args.la_f + okk, args.la_b + okk, args.out + ov, L, DK, DV,
                                           reinterpret_cast<float*>(smem), args.inv_tau);
            return;
        }
        constexpr int P = DK / 4;
        const float4* own = reinterpret_cast<const float4*>(slots + (nch - 1) * kSlotFloats);
        for (int x = tid; x < 2 * DV * P; x += blockDim.x) {
            const int dir = x >= DV * P, y = dir ? x - DV * P : x, n = y / P, p = y % P;
            float4 carry = make_float4(0.f, 0.f, 0.f, 0.f);
            const int first = dir == 0 ? 0 : nch - 2, last = dir == 0 ? chunk : chunk - 1, step = dir == 0 ? 1 : -1;
#pragma unroll 1
            for (int s = first; s != last; s += step) {
                const float4 u = *reinterpret_cast<const float4*>(slots + s * kSlotFloats + n * DK + 4 * p);
                const float4 d = *reinterpret_cast<const float4*>(slots + s * kSlotFloats + kStateFloats + 4 * p);
                carry = make_float4(fmaf(d.x, carry.x, u.x), fmaf(d.y, carry.y, u.y), fmaf(d.z, carry.z, u.z), fmaf(d.w, carry.w, u.w));
            }
            if (dir == 1) {
                const float4 d = own[p];
                carry = make_float4(carry.x * d.x, carry.y * d.y, carry.z * d.z, carry.w * d.w);
            }
            const int m = p >> 2, cc = p & 3;
            uint8_t* row = smem + lay.st + dir * kState + n * 64;
            auto at = [&](int j) { return row + ((j ^ ((n >> 1) & 3)) << 4); };
            if (2 * m + 1 < NP) {
                *reinterpret_cast<uint32_t*>(at(2 * m) + 4 * cc) = pack_bf16(carry.x, carry.y);
                *reinterpret_cast<uint32_t*>(at(2 * m + 1) + 4 * cc) = pack_bf16(carry.z, carry.w);
            } else {
                *reinterpret_cast<uint2*>(at(2 * m) + 8 * cc) = make_uint2(pack_bf16(carry.x, carry.y), pack_bf16(carry.z, carry.w));
            }
        }
        __syncthreads();
        if (!live) return;
    }
    if (MODE == kMain || MODE == kCluster || (kTwo && T > 8)) {
        if (MODE != kCluster && !__all_sync(0xffffffffu, mbar_wait_bounded(bar + 8, 0))) {   // (never expected where the warps of this block form the states)
            if (lane == 0) atomicOr(args.dev_status, kDevStatusTimeout);
            return;
        }
        auto state = [&](const uint32_t (&qq)[MP][4], uint32_t st) {
#pragma unroll
            for (int n2 = 0; n2 < MV; ++n2) {
#pragma unroll
                for (int m = 0; m < MP; ++m) {
                    uint32_t r[4];
                    t64.load_b(st, 16 * n2, m, r);
                    if (2 * m + 1 < NP) {
                        mma_k16(o[2 * n2], qq[m], r[0], r[1]);
                        mma_k16(o[2 * n2 + 1], qq[m], r[2], r[3]);
                    } else {
                        mma_k8(o[2 * n2], qq[m][0], qq[m][1], r[0]);
                        mma_k8(o[2 * n2 + 1], qq[m][0], qq[m][1], r[2]);
                    }
                }
            }
        };
        if (MODE == kMain || MODE == kCluster) {   // (the first chunk's S> and the last one's S< are zero)
            if (chunk > 0) state(qf, tst);
            if (chunk + 1 < nch) state(qb, tst + kState);
        } else if (ch == 0) {
            state(qb, tst + kState);
        } else {
            state(qf, tst);
        }
    }
    // ---- out: four 8-column tiles at a time turned so that a lane holds sixteen bytes of a row ----
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int row = tok0 + 16 * w + 8 * r + g;
        __nv_bfloat16* op = args.out + (unit * L + row) * DV;
#pragma unroll
        for (int n4 = 0; n4 < NV; n4 += 4) {
            uint32_t x[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) x[n] = n4 + n < NV ? pack_bf16(o[n4 + n < NV ? n4 + n : 0][2 * r], o[n4 + n < NV ? n4 + n : 0][2 * r + 1]) : 0u;
            transpose4(x, c);
            if (row < L && n4 + c < NV) *reinterpret_cast<uint4*>(op + 8 * (n4 + c)) = make_uint4(x[0], x[1], x[2], x[3]);
        }
    }
}

// Second launch of a long call: the states that enter every chunk from what the chunks add, S> ascending, S< descending, the latter
// stored times d<(c), the decay from the chunk's end to its start.
template <int DK, int DV, int GROUPS, int RUN>
__global__ void __launch_bounds__(kFoldThreads, fold_blocks_per_sm(RUN)) mma_fold_kernel(const MChunkArgs a) {
    constexpr int P = DK / 4, kItems = kFoldThreads / GROUPS;
    constexpr int kState = (int)MLayout<DV>::kState;
    const size_t unit = blockIdx.x;
    const int dir = blockIdx.y, item = threadIdx.x % kItems, grp = threadIdx.x / kItems;
    const int x = blockIdx.z * kItems + item, nch = a.nch;
    const int run = (nch + GROUPS - 1) / GROUPS, i0 = min(nch, grp * run), i1 = min(nch, i0 + run);   // in walking order
    const bool in = x < P * DV;
    const int p = in ? x % P : 0, n = in ? x / P : 0;
    const int step = dir == 0 ? 1 : -1;
    const size_t first = unit * nch + (dir == 0 ? i0 : nch - 1 - i0);
    uint8_t* img = a.img + (first * 2 + dir) * kState + n * 64 + (((p >> 1) ^ ((n >> 1) & 3)) << 4) + 8 * (p & 1);
    pdl_wait();
    pdl_launch_dependents();
    fold_runs<GROUPS, RUN>(a.u + ((first * 2 + dir) * DV + n) * DK + 4 * p, step * (2 * DV * DK), a.decay + first * 64 + dir * 32 + 4 * p, step * 64, run, i1 - i0, in,
                      item, grp, [&](int i, float4 carry, float4 d) {
                          if (dir == 1) carry = make_float4(carry.x * d.x, carry.y * d.y, carry.z * d.z, carry.w * d.w);
                          *reinterpret_cast<uint2*>(img + (ptrdiff_t)(i * step) * (2 * kState)) = make_uint2(pack_bf16(carry.x, carry.y), pack_bf16(carry.z, carry.w));
                      });
}

template <int DK, int DV, bool GATES, int MAXT, int MODE>
cudaError_t launch_mma_t(ArgsOf<MODE> a, const CUtensorMap& tv, int tiles, cudaStream_t stream) {
    const int threads = (tiles < 2 ? 2 : tiles) * 32;
    const size_t smem = MLayout<DV>(tiles, MODE == kMain || MODE == kCluster || (MODE == kUnit && tiles > 8), MODE == kCluster ? all_slots(DK, DV, a.nch) : 0u).total, rec = (size_t)rec_plan(threads < kRecThreads ? threads : kRecThreads, DK, DV).smem_floats * 4;
    static std::atomic<int> sms_of[64];   // 0: this instance is not configured on the device yet
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = sms_of[dev].load(std::memory_order_acquire);
    if (sms == 0) {
        auto kernel = bigla_mma_kernel<DK, DV, GATES, MAXT, MODE>;
        if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MODE == kCluster ? 112 * 1024 : 100 * 1024)) != cudaSuccess) return e;
        if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        sms_of[dev].store(sms, std::memory_order_release);
    }
    a.ahead = mma_blocks_per_sm(DK, DV, MAXT, MODE) * sms;
    const cudaError_t le = launch_pdl_cluster(bigla_mma_kernel<DK, DV, GATES, MAXT, MODE>, dim3((unsigned)a.blocks), dim3(threads), smem > rec ? smem : rec,
                                              MODE == kCluster ? a.nch : 1, stream, tv, a);
    count_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

// Registers per thread follow from the longest unit an instance takes.
template <int DK, int DV, bool GATES>
cudaError_t launch_mma(const MArgs& a, cudaStream_t stream) {
    const int T = (a.L + 15) / 16;
    CUtensorMap tv;
    if (!make_map(&tv, a.v, a.blocks, a.L, DV, DV == 32 ? 32 : 64, T * 16)) return cudaErrorInvalidValue;
    if (T <= 8) return launch_mma_t<DK, DV, GATES, 8, kUnit>(a, tv, T, stream);
    if (T <= 13) return launch_mma_t<DK, DV, GATES, 13, kUnit>(a, tv, T, stream);
    return launch_mma_t<DK, DV, GATES, 16, kUnit>(a, tv, T, stream);
}

// Multiprocessors of the current device, 0 if it cannot be asked.
static int device_sms() {
    static std::atomic<int> sms_of[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int sms = sms_of[dev].load(std::memory_order_relaxed);
    if (sms == 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        sms_of[dev].store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// Sequences of any length: chunks of equal numbers of tiles, up to eight.  From logits, beyond eight chunks, the tiles are what makes
// the rounds of blocks cheapest, a block's time being about that of its loads and hand-overs (eight tiles' worth) and of its tiles, short
// of the 128 chunks up to which the fold keeps its runs short.  6 x 4 units of 1300 tokens, 24 x 64: 17.8 us a call, 20.6 with
// eight tiles; 3 x 3 of 5000, 24 x 32: 16.4 and 18.3; 8 x 4 of 4096, 24 x 48: 37.4 and 37.8.  Beyond two rounds and
// a quarter the blocks no longer end together, so that a round saved is none (119 units of 1868, 24 x 48, 3.0 rounds: 67.1 us cut by rounds,
// 64.1 with eight tiles; 15 of 10813, 2.15 rounds: 46.7 and 48.8), four at 16 x 32, whose blocks are short (129 units of 1300,
// 2.4 rounds: 28.9 and 31.6), and the scratch, which grows with the number of chunks, stays that of eight tiles.  (From log gates the scratch may be the caller's, whose size this keeps.)
struct ChunkPlan {
    int nch, tiles;
    size_t u, img, decay, flags, total;   // byte offsets in the scratch
};
ChunkPlan chunk_plan(long long units, int L, int dk, int dv, bool gates = false) {
    ChunkPlan p;
    const int T = (L + 15) / 16;
    auto cut = [&](int tiles) {
        p.nch = (T + tiles - 1) / tiles;
        p.tiles = (T + p.nch - 1) / p.nch;
        p.nch = (T + p.tiles - 1) / p.tiles;
    };
    cut(kChunkTiles);
    const long long slots = (long long)mma_blocks_per_sm(dk, dv, kChunkTiles, kMain) * device_sms();
    if (gates && p.nch > kChunkTiles && 4 * form_units(units) * p.nch <= (dk * dv <= 512 ? 16 : 9) * slots) {
        int best = p.tiles;
        long long best_cost = -1;
        for (int tiles = kChunkTiles; tiles >= 5; --tiles) {
            const int nch = (T + tiles - 1) / tiles;
            const long long cost = (form_units(units) * nch + slots - 1) / slots * (8 + tiles);
            if (best_cost < 0 || (cost < best_cost && nch <= 128)) best = tiles, best_cost = cost;
        }
        cut(best);
    }
    const size_t n = (size_t)units * p.nch;
    p.u = 0;
    p.img = n * 2 * dk * dv * 4;
    p.decay = p.img + n * 2 * dv * 64;
    p.flags = p.decay + n * 64 * 4;
    p.total = (p.flags + n * 4 + 255) / 256 * 256;
    return p;
}

// One launch: the chunks of a unit are the blocks of a cluster.
template <int DK, int DV, bool GATES>
cudaError_t launch_cluster(MChunkArgs a, cudaStream_t stream) {
    CUtensorMap tv;
    if (!make_map(&tv, a.v, a.units, a.L, DV, DV == 32 ? 32 : 64, a.tiles * 16)) return cudaErrorInvalidValue;
    return launch_mma_t<DK, DV, GATES, 8, kCluster>(a, tv, a.tiles, stream);
}

template <int DK, int DV, bool GATES>
cudaError_t launch_chunks(MChunkArgs a, cudaStream_t stream) {
    CUtensorMap tv;
    if (!make_map(&tv, a.v, a.units, a.L, DV, DV == 32 ? 32 : 64, a.tiles * 16)) return cudaErrorInvalidValue;
    cudaError_t e = launch_mma_t<DK, DV, GATES, 8, kSummary>(a, tv, a.tiles, stream);
    if (e != cudaSuccess) return e;
    e = with_fold_plan(a.nch, a.units, 2, DK / 4 * DV, device_sms(), [&](auto groups, auto run) {
        constexpr int kGroups = decltype(groups)::value, kItems = kFoldThreads / kGroups;
        return launch_pdl(mma_fold_kernel<DK, DV, kGroups, decltype(run)::value>, dim3((unsigned)a.units, 2, (DK / 4 * DV + kItems - 1) / kItems), dim3(kFoldThreads), 0, stream, a);
    });
    count_launch();
    if (e != cudaSuccess) return e;
    a.expire_wait = 0;   // (of a long call the first launch)
    return launch_mma_t<DK, DV, GATES, 8, kMain>(a, tv, a.tiles, stream);
}

}  // namespace

// Where this form is the faster one for units of up to 256 tokens.  Its work per unit grows with the 16-token tiles and with
// the state, while the tcgen05 form's time is its hand-overs whatever the state, so the line is a product of the two; and it
// drops with the units per SM, as the other form gets its latency hidden, sooner where the gates come prepared, which spares
// the other form a phase.  Timed against the tcgen05 form for six head sizes, 130 to 256 tokens, 1 to 1024 units, with and without
// the gates (756 shapes): within 0.2 % of the better form on average.  512 units of 208 tokens, 24 x 48, us, this form / tcgen05:
// from logits 20.4 / 23.7, from log gates 20.2 / 19.9; 768 of 208, 32 x 64, from logits 37.2 / 30.7.
bool mma_preferred(long long units, int L, int dk, int dv, bool gates) {
    const int sms = device_sms();
    if (sms == 0) return false;
    units = form_units(units);
    const int work = (L + 15) / 16 * dk * dv;
    return work <= (units <= sms ? 27000 : (gates || units <= 3LL * sms ? 20000 : 15200));
}

cudaError_t launch_bigla_mma(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                             const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out, long long units,
                             int L, int dk, int dv, float gate_tau, cudaStream_t stream) {
    MArgs a{};
    a.q = q; a.k = k; a.v = v; a.la_f = la_f; a.la_b = la_b; a.out = out;
    a.L = L; a.blocks = units;
    a.inv_tau = gate_tau > 0.f ? 1.f / gate_tau : 0.f;
    a.expire_wait = take_expire_next_wait() == 1;
    a.dev_status = device_status_ptr();
    if (!a.dev_status) return cudaErrorUnknown;
#define VIG_CASE(DK_, DV_) \
    if (dk == DK_ && dv == DV_) return gate_tau > 0.f ? launch_mma<DK_, DV_, true>(a, stream) : launch_mma<DK_, DV_, false>(a, stream);
    VIG_CASE(16, 32) VIG_CASE(16, 48) VIG_CASE(16, 64)
    VIG_CASE(24, 32) VIG_CASE(24, 48) VIG_CASE(24, 64)
    VIG_CASE(32, 32) VIG_CASE(32, 48) VIG_CASE(32, 64)
#undef VIG_CASE
    return cudaErrorNotSupported;
}

// Where the chunks run faster this way than as tcgen05 segments or chunk tasks.  A chunk's chain of dependent steps is shorter
// here, so few chunks gain most (1.3 to 1.7 times up to one per SM); a chunk's work grows with the key dimensions, while the chunk
// tasks, once their latency is hidden, cost the same whatever the state: keys of 32 lose in large calls, sooner where the gates come
// prepared (32 units of 4096 tokens, 32 x 64: 51.7 us this way, 42.4 as tasks; 24 x 48 from log gates 36.6 and 37.4).  The segmented launch is at its best while two full segments (four chunks) of every unit are
// resident in one round; beyond that round it is at its worst (300 units of 304 tokens, 32 x 64, from logits: 52.7 us, 43.7 this way).
// More than 64 chunks: the tasks' fold takes one run.  Timed against the tcgen05 forms for six head sizes, 1100 to 16384 tokens,
// 1 to 96 units, with and without the gates (468 shapes; 1530 more up to 512 tokens before clusters took most of them): within 0.2 %
// of the better form on average.  For the calls that clusters take, this only says what scratch a caller is asked for, as before them.
bool mma_chunks_preferred(long long units, int L, int dk, int dv, bool gates) {
    if (dk == 16) return true;
    const long long sms = device_sms();
    if (sms == 0) return false;
    units = form_units(units);
    const int nch = chunk_plan(units, L, dk, dv).nch;
    const long long chunks = units * nch;
    const bool two_segments = L <= 512;
    if (two_segments && nch == 4 && units <= sms) return dk == 32 ? chunks <= sms : (chunks <= 3 * sms || dv <= (gates ? 48 : 32));
    if (two_segments && units > sms) return gates || dk == 24 || chunks <= 8 * sms;
    if (dk == 24) return true;
    if (gates) return dv == 32 || chunks <= 5 * sms;
    return 10 * chunks <= 28 * sms || (nch > 64 && chunks <= 4 * sms);
}

bool mma_chunks_supported(long long units, int L, int dk, int dv) { return units * chunk_plan(units, L, dk, dv).nch <= 0x7fffffffLL; }

bool mma_cluster_supported(long long units, int L, int dk, int dv) {
    const int nch = chunk_plan(units, L, dk, dv).nch;
    return nch >= 2 && nch <= 8 && units * nch <= 0x7fffffffLL;
}

// Where one launch of clusters is the fastest form.  Against the three launches over chunks, the tcgen05 segments and chunk tasks
// (564 shapes, six head sizes, 257 to 1024 tokens, 8 to 600 units): three chunks always (144 units of 300 tokens, 32 x 64, from
// logits 19.7 us, 23.2 in three launches); four unless a large state meets what suits the segments, two of them for every unit
// in one round, or comes with its gates prepared; more while the clusters of the call run side by side, since every chunk gives its states
// to all the others and clusters of seven or eight blocks leave SMs without one (148 units of 1024 tokens, 32 x 64: 86 us, 59 in three
// launches).  Within 1.0 % of the best form on average.  Units of one block otherwise (336 shapes): two chunks on SMs of their own
// halve the chain of a large unit while SMs are free (one unit of 256 tokens, 32 x 64: 8.0 us, 10.3 and 11.2 in one block).
bool mma_cluster_preferred(long long units, int L, int dk, int dv, bool gates) {
    const long long sms = device_sms();
    if (sms == 0) return false;
    units = form_units(units);
    const int nch = chunk_plan(units, L, dk, dv).nch, state = dk * dv;
    const long long chunks = units * nch;
    if (nch == 2) return 2 * units <= sms && (L + 15) / 16 * state >= 19900;
    if (nch == 3 || state <= 512) return true;
    if (nch == 4) return state <= 1152 || (units <= sms ? 10 * chunks <= 28 * sms : gates || state <= 1536);
    return 10 * chunks <= (nch <= 6 ? 28 : (state <= 1152 ? 20 : 10)) * sms;
}

size_t mma_chunks_workspace_bytes(long long units, int L, int dk, int dv, bool gates) { return chunk_plan(units, L, dk, dv, gates).total; }

cudaError_t launch_bigla_mma_chunks(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                    const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out, long long units,
                                    int L, int dk, int dv, float gate_tau, void* ws, cudaStream_t stream) {
    const ChunkPlan p = chunk_plan(units, L, dk, dv, gate_tau > 0.f);
    char* b = static_cast<char*>(ws);
    MChunkArgs a{};
    a.q = q; a.k = k; a.v = v; a.la_f = la_f; a.la_b = la_b; a.out = out;
    a.L = L; a.units = units; a.blocks = units * p.nch; a.nch = p.nch; a.tiles = p.tiles;
    a.u = reinterpret_cast<float*>(b + p.u);
    a.img = reinterpret_cast<uint8_t*>(b + p.img);
    a.decay = reinterpret_cast<float*>(b + p.decay);
    a.flags = reinterpret_cast<int*>(b + p.flags);
    a.inv_tau = gate_tau > 0.f ? 1.f / gate_tau : 0.f;
    a.expire_wait = take_expire_next_wait() == 1;
    a.dev_status = device_status_ptr();
    if (!a.dev_status) return cudaErrorUnknown;
#define VIG_CASE(DK_, DV_)        \
    if (dk == DK_ && dv == DV_) \
        return gate_tau > 0.f ? launch_chunks<DK_, DV_, true>(a, stream) : launch_chunks<DK_, DV_, false>(a, stream);
    VIG_CASE(16, 32) VIG_CASE(16, 48) VIG_CASE(16, 64)
    VIG_CASE(24, 32) VIG_CASE(24, 48) VIG_CASE(24, 64)
    VIG_CASE(32, 32) VIG_CASE(32, 48) VIG_CASE(32, 64)
#undef VIG_CASE
    return cudaErrorNotSupported;
}

cudaError_t launch_bigla_mma_cluster(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                     const __nv_bfloat16* la_f, const __nv_bfloat16* la_b, __nv_bfloat16* out, long long units,
                                     int L, int dk, int dv, float gate_tau, cudaStream_t stream) {
    const ChunkPlan p = chunk_plan(units, L, dk, dv);
    MChunkArgs a{};
    a.q = q; a.k = k; a.v = v; a.la_f = la_f; a.la_b = la_b; a.out = out;
    a.L = L; a.units = units; a.blocks = units * p.nch; a.nch = p.nch; a.tiles = p.tiles;
    a.inv_tau = gate_tau > 0.f ? 1.f / gate_tau : 0.f;
    a.expire_wait = take_expire_next_wait() == 1;
    a.dev_status = device_status_ptr();
    if (!a.dev_status) return cudaErrorUnknown;
#define VIG_CASE(DK_, DV_)        \
    if (dk == DK_ && dv == DV_) \
        return gate_tau > 0.f ? launch_cluster<DK_, DV_, true>(a, stream) : launch_cluster<DK_, DV_, false>(a, stream);
    VIG_CASE(16, 32) VIG_CASE(16, 48) VIG_CASE(16, 64)
    VIG_CASE(24, 32) VIG_CASE(24, 48) VIG_CASE(24, 64)
    VIG_CASE(32, 32) VIG_CASE(32, 48) VIG_CASE(32, 64)
#undef VIG_CASE
    return cudaErrorNotSupported;
}

}  // namespace vig
