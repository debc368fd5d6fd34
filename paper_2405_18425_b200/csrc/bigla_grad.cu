// Gradient of the bf16 BiGLA forward pass (paper Eq. 6) on the tensor cores, for the head sizes of the paper's models.
//
// Per unit, with g = dLoss/d_out, b_t the inclusive prefix sums of log alpha> and x_t the exclusive ones of log alpha<,
//     q~> = q e^{b},  k~> = k e^{-b},  q~< = q e^{-x},  k~< = k e^{x},   D_ts = g_t . v_s
//     dq_t = 1/2 [ e^{b_t} sum_{s <= t} D_ts k~>_s  +  e^{-x_t} sum_{s >= t} D_ts k~<_s ]
//     dk_s = 1/2 [ e^{-b_s} sum_{t >= s} D_ts q~>_t  +  e^{x_s} sum_{t <= s} D_ts q~<_t ]
//     dv_s = 1/2 [ sum_{t >= s} (q~>_t . k~>_s) g_t  +  sum_{t <= s} (q~<_t . k~<_s) g_t ]
//     dlog alpha>_t = sum_{m >= t} E>_m,   dlog alpha<_t = - sum_{m > t} E<_m,   E = q dq - k dk per direction.
// A sequence is cut into chunks; what lies outside a chunk enters through four dk x dv states at its borders,
//     S> = sum_{s before} e^{b_end - b_s} k_s^T v_s      Z< = sum_{t before} e^{x_end - x_t} q_t^T g_t     (from the left)
//     S< = sum_{s after} e^{x_s} k_s^T v_s               Z> = sum_{t after} e^{b_t} q_t^T g_t              (from the right)
// and the sums of E over the tokens after a chunk come from there too (from the other block of a pair, or as the row sums
// of S o Z of the two states that meet at the chunk's right border).
//
// One block per chunk, one warp per 16 tokens, every product a chain of 16 x 16 tiles whose scores stay in registers: a
// warp holds its tokens' rows of g, v or k~ as A fragments, runs over the chunk's tiles in shared memory, and feeds the
// scores straight back as the A operand of the second product.  D, k~, q~ and the states of the dq / dk products are
// taken as sums of two bf16 (sixteen significant bits, three products each, fp32 accumulation; g and v are bf16 as
// given), so that dq, dk and the gate gradients carry no rounding above the 2^-17 level before they are stored; dv takes
// one bf16 per operand like the forward pass.
//
//   kSingle   units of one chunk
//   kPair     two chunks: two blocks of a cluster hand each other the border states through distributed shared memory
//   kSummary, (fold), kMain   any length: the chunks' own states to scratch, folded over the sequence, then the chunks
#include <cuda.h>

#include <atomic>

#include "fold.cuh"
#include "mma.cuh"
#include "scan_bwd.cuh"
#include "tma_host.h"
#include "vig_internal.h"

namespace vig {
namespace {

using namespace wmma16;

enum { kSingle = 0, kPair = 1, kMain = 2, kSummary = 3 };
constexpr float kGateRange = 60.f;   // largest decay of a chunk, as -log, that the factorised tiles take

// Tiles (of 16 tokens) per block: with two blocks per SM, shared memory (768 B a token, 8 KB a state) takes eight tiles
// without states, seven with two states, six with four.
constexpr int max_tiles(int mode) { return mode == kSingle ? 8 : (mode == kPair ? 7 : 6); }
// Warps per block: one per tile; eight where the chunk's own states are formed (eight or sixteen equal jobs).
constexpr int grad_warps(int mode, int tiles) { return mode == kPair || mode == kSummary ? 8 : tiles; }

struct GArgs {
    const __nv_bfloat16 *q, *k, *v, *la_f, *la_b, *g;
    __nv_bfloat16 *dq, *dk, *dv, *dla_f, *dla_b;
    int L, nch, tiles;      // tokens, chunks per unit, tiles per chunk
    float* u;               // [unit][chunk][kind][DV][DK] fp32: the chunks' own states (kinds S>, Z<, S<, Z>)
    uint8_t* img;           // [unit][chunk][kind][hi, lo][DV][64 B]: the states entering a chunk, as shared-memory tiles
    float* decay;           // [unit][chunk][2][32]: products of alpha>, alpha< over the chunk
    int* flags;             // [unit][chunk]: 1: gates out of range, 2: not computed (a wait ran out)
    long long chunks;       // of the call
    int ahead;              // the chunk this many blocks on is pulled into L2
    int* dev_status;
    int expire_wait;        // test hook, 1: every block lets one bounded wait, on an mbarrier nothing completes, run out; 2: a pair's left block its last
};

// Operand tiles [rows][32] bf16 (64-byte rows), in this order behind the v and g tiles.  As loaded: q in kQf, k in kKf,
// log alpha> in kQb, log alpha< in kKb.
enum { kKf = 0, kKb = 2, kQf = 4, kQb = 6 };   // hi; lo = + 1
template <int DV>
struct GLayout {
    static constexpr uint32_t kVRow = DV == 32 ? 64 : 128, kState = DV * 64;   // bytes of a state tile (hi or lo)
    uint32_t g, op, op_bytes, st, totals, ends, part, bar, total;
    __host__ __device__ GLayout(int tiles, int mode) {
        const uint32_t rows = tiles * 16u, warps = grad_warps(mode, tiles);
        g = rows * kVRow;
        op = 2 * g;
        op_bytes = rows * 64;
        st = op + 8 * op_bytes;
        totals = st + (mode == kPair ? 2u : (mode == kMain ? 4u : 0u)) * 2 * kState;   // [tile][2][32] fp32
        ends = totals + tiles * 256u;                                                // [2][32] fp32
        part = ends + 256;                                                           // [warp][2][32] fp32
        bar = part + (mode == kSummary ? 0u : warps * 256u);
        total = bar + 64;
    }
};

// dq>, dk< of an element between the walks of gradient_by_walks, as fp32 in two bf16 result buffers each (written over at the end).
struct ResultPairs {
    __nv_bfloat16 *dq, *dk, *dla_f, *dla_b;
    static __device__ __forceinline__ void put_halves(__nv_bfloat16* hi, __nv_bfloat16* lo, float x) {
        *reinterpret_cast<unsigned short*>(hi) = (unsigned short)(__float_as_uint(x) >> 16);
        *reinterpret_cast<unsigned short*>(lo) = (unsigned short)(__float_as_uint(x) & 0xffffu);
    }
    static __device__ __forceinline__ float get_halves(const __nv_bfloat16* hi, const __nv_bfloat16* lo) {
        return __uint_as_float(((uint32_t)*reinterpret_cast<const unsigned short*>(hi) << 16) | *reinterpret_cast<const unsigned short*>(lo));
    }
    __device__ __forceinline__ void put(size_t e, float2 x) const {
        put_halves(dq + e, dk + e, x.x);
        put_halves(dla_f + e, dla_b + e, x.y);
    }
    __device__ __forceinline__ float2 get(size_t e) const { return make_float2(get_halves(dq + e, dk + e), get_halves(dla_f + e, dla_b + e)); }
};
struct WalkArgs {
    scan::ScanBwdArgs<__nv_bfloat16> bwd;
    scan::ScanArgs<__nv_bfloat16> fwd;
    ResultPairs pairs;
};

// A unit whose gates leave the range of the factorised tiles: the fp32 walks of any decay (scan_bwd.cuh for dq, dk and the gate
// gradients, scan_fwd.cuh on (k, q, d_out) for dv), a sequence cut into as many segments as the block has warps, or room for in
// the shared memory of its dead tiles.  The unit's slabs of eight key dimensions and of sixteen value columns are dealt out
// over its blocks.  Every thread of the block calls it.  768 such units of 196 tokens (32, 64): 10.9 ms with one key dimension
// or value column a warp, serial over the tokens.
template <int DK, int DV>
__device__ __noinline__ void gradient_by_walks(WalkArgs x, size_t unit, int block, int blocks, float* smem, uint32_t smem_bytes) {
    constexpr int kBwdSlabs = DK / scan::kRows, kSlabs = kBwdSlabs + DV / scan::kCols, RPL = DK <= 16 ? 4 : 8;
    constexpr size_t kBwd = scan::bwd_stage_floats(DV / 4) + scan::bwd_fold_floats(DV / 4);
    constexpr size_t kFwd = scan::scan_stage_floats(RPL) > scan::scan_fold_floats(RPL) ? scan::scan_stage_floats(RPL) : scan::scan_fold_floats(RPL);
    constexpr int kPerWarp = (int)(4 * (kBwd > kFwd ? kBwd : kFwd));
    const int L = x.bwd.L, w = threadIdx.x >> 5;
    int nw = max(1, min(min((int)blockDim.x >> 5, scan::bwd_max_warps(DV / 4)), (int)smem_bytes / kPerWarp));
    x.bwd.seg_len = x.fwd.seg_len = ((L + nw - 1) / nw + scan::TG - 1) / scan::TG * scan::TG;
    nw = (L + x.bwd.seg_len - 1) / x.bwd.seg_len;
    for (int slab = block; slab < kSlabs; slab += blocks) {
        __syncthreads();   // the tiles, or the slab before
        if (slab < kBwdSlabs) scan::scan_bwd_slab<__nv_bfloat16, DV / 4, true>(x.bwd, x.pairs, unit, slab, w, nw, smem);
        else scan::scan_fwd_slab<__nv_bfloat16, RPL, true>(x.fwd, unit, slab - kBwdSlabs, w, nw, smem);
    }
}

template <int DK, int DV, int MODE>
__global__ void __launch_bounds__(grad_warps(MODE, max_tiles(MODE)) * 32, 2)
bigla_grad_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_f,
                  const __grid_constant__ CUtensorMap tm_b, const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_g,
                  const GArgs a) {
    constexpr int NP = DK / 8, MP = (NP + 1) / 2;   // 8-column tiles of the key dimensions, pairs of them
    constexpr int NV = DV / 8, MV = DV / 16;        // ... of the value dimensions
    constexpr int RV = GLayout<DV>::kVRow;
    constexpr uint32_t kState = GLayout<DV>::kState;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, w = __shfl_sync(0xffffffffu, tid >> 5, 0), nw = blockDim.x >> 5;
    const int g = lane >> 2, c = lane & 3;
    const int L = a.L, T = (L + 15) >> 4, tiles = a.tiles;
    const int nch = MODE == kSingle ? 1 : a.nch;
    const int chunk = (int)(blockIdx.x % (unsigned)nch);
    const size_t unit = blockIdx.x / (unsigned)nch;
    const int row0 = chunk * tiles * 16, nT = min(tiles, T - chunk * tiles);   // this chunk's first token and live tiles
    // Tile of this warp (idle beyond the live ones).  Odd chunks leave the first warps idle, even ones the last, so that the
    // tiles of two resident blocks spread over the SM's four schedulers.
    const int wt = (chunk & 1) ? w - (nw - nT) : w;
    const bool live = wt >= 0 && wt < nT;
    const GLayout<DV> lay(tiles, MODE);
    const uint32_t base = smem_u32(smem), tv = base, tg = base + lay.g, top = base + lay.op, tst = base + lay.st;
    const uint32_t bar = base + lay.bar;   // q, k, gates landed; + 40: v, g landed; + 8: states landed; + 24: never completed, for the test hook; + 32: a pair's sums of E landed
    auto op = [&](int o) { return top + (uint32_t)o * lay.op_bytes; };
    float* totals = reinterpret_cast<float*>(smem + lay.totals);
    float* ends = reinterpret_cast<float*>(smem + lay.ends);
    float* part = reinterpret_cast<float*>(smem + lay.part);
    volatile int* state_word = reinterpret_cast<volatile int*>(smem + lay.bar + 16);   // [0]: gates out of range here;  [1]: in the other block of a pair
    const Tile<64> t64(lane);
    const Tile<RV> tvv(lane);

    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 8, 1);
        mbar_init(bar + 24, 1);
        mbar_init(bar + 32, 1);
        mbar_init(bar + 40, 1);
        state_word[0] = 0;   // (the other word is written by the other block alone, and read once that has landed)
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    auto walk_args = [&] {   // the adjoint walk for dv: (k, q, d_out), the gates exchanged and moved by one token
        return WalkArgs{{a.q, a.k, a.v, a.la_f, a.la_b, a.g, a.dq, a.dk, a.dla_f, a.dla_b, a.L, DK, DV, 0},
                        {a.k, a.q, a.g, a.la_b, a.la_f, a.dv, a.L, DK, DV, 0, -1, 1},
                        {a.dq, a.dk, a.dla_f, a.dla_b}};
    };
    auto pull = [&](long long block) {   // the tokens of a block into L2
        const long long nu = block / nch;
        const int nr = (int)(block % nch) * tiles * 16;
        const size_t at = (size_t)nu * L + nr;
        const uint32_t n = min(tiles * 16, L - nr);
        prefetch_l2(a.la_f + at * DK, n * DK * 2);
        prefetch_l2(a.la_b + at * DK, n * DK * 2);
        prefetch_l2(a.q + at * DK, n * DK * 2);
        prefetch_l2(a.k + at * DK, n * DK * 2);
        prefetch_l2(a.v + at * DV, n * DV * 2);
        prefetch_l2(a.g + at * DV, n * DV * 2);
    };
    // ... and those of the first round while the launch before still runs: a prefetch consumes nothing, and L2 stays coherent with
    // what that launch still writes.
    if (MODE != kMain && tid == 0 && (long long)blockIdx.x < a.ahead) pull(blockIdx.x);
    // The chunks' launch starts under the fold: that one lets it in only behind its own wait, when the summaries are complete, and
    // with them all that was launched before.  So inputs and flags are read at once, from L2 (see pdl_wait), and only what the fold
    // writes is waited for.
    if (MODE != kMain) {
        pdl_wait();
        pdl_launch_dependents();
    }
    if (tid == 0) {
        mbar_expect_tx(bar, 4 * lay.op_bytes);   // (v and g, which nothing needs before the operands are scaled, behind a barrier of their own)
        tma_load_3d(op(kQb), &tm_f, 0, row0, (int)unit, bar);
        tma_load_3d(op(kKb), &tm_b, 0, row0, (int)unit, bar);
        tma_load_3d(op(kQf), &tm_q, 0, row0, (int)unit, bar);
        tma_load_3d(op(kKf), &tm_k, 0, row0, (int)unit, bar);
        mbar_expect_tx(bar + 40, 2 * lay.g);
        tma_load_3d(tv, &tm_v, 0, row0, (int)unit, bar + 40);
        tma_load_3d(tg, &tm_g, 0, row0, (int)unit, bar + 40);
        if (MODE == kPair) {   // two states and a word from the other block; from the right one also its sums of E
            mbar_expect_tx(bar + 8, 4 * DV * NP * 16 + 4);
            mbar_expect_tx(bar + 32, 2 * DK * 4);
        }
        const long long next = (long long)blockIdx.x + a.ahead;
        if (next < a.chunks) pull(next);   // a block that starts when one of these is done finds its tokens in L2
    }
    __syncthreads();
    if (MODE == kPair) cluster_arrive_relaxed();   // the other block may be written to once it runs (nothing of its own goes where that lands)
    bool ok = true;
    if (a.expire_wait == 1 && tid == 0) ok = mbar_wait_bounded(bar + 24, 0, 64);   // test hook: this wait cannot succeed
    ok = mbar_wait_bounded(bar, 0) && ok;

    // ---- this warp's 16 rows; the gate tiles turned, as B operands of products over the tokens ----
    uint32_t qa[MP][4], ka[MP][4], fa[MP][4], ba[MP][4];
    if (live) {
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            t64.load_trans(op(kQb), 16 * wt, m, fa[m]);
            t64.load_trans(op(kKb), 16 * wt, m, ba[m]);
            t64.load(op(kQf), 16 * wt, m, qa[m]);
            t64.load(op(kKf), 16 * wt, m, ka[m]);
        }
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            float tf[4], tb[4];
            mma_k16_from(tf, kOnes, kOnes, kOnes, kOnes, fa[j >> 1][2 * (j & 1)], fa[j >> 1][2 * (j & 1) + 1], 0.f, 0.f);
            mma_k16_from(tb, kOnes, kOnes, kOnes, kOnes, ba[j >> 1][2 * (j & 1)], ba[j >> 1][2 * (j & 1) + 1], 0.f, 0.f);
            if (g == 0) {
                *reinterpret_cast<float2*>(totals + (wt * 2) * 32 + 8 * j + 2 * c) = make_float2(tf[0], tf[1]);
                *reinterpret_cast<float2*>(totals + (wt * 2 + 1) * 32 + 8 * j + 2 * c) = make_float2(tb[0], tb[1]);
            }
        }
    }
    __syncthreads();
    // running sums over the tiles, in place: what comes before each tile; at the end the chunk's totals and the range check
    for (int d = w; d < 2; d += nw < 2 ? 1 : nw) {   // (a block of one warp: both directions by it)
        if (lane < DK) {
            float s = 0.f;
            for (int x = 0; x < nT; ++x) {
                const float t = totals[(x * 2 + d) * 32 + lane];
                totals[(x * 2 + d) * 32 + lane] = s;
                s += t;
            }
            ends[d * 32 + lane] = s;
            if (!(s >= -kGateRange)) state_word[0] = 1;
        }
    }
    __syncthreads();
    auto carry = [&](int d, int j) { return *reinterpret_cast<const float2*>(totals + (wt * 2 + d) * 32 + 8 * j + 2 * c); };
    const uint32_t tri_i = triangle(g, c, true), tri_x = triangle(g, c, false);
    // ---- scaled operands in two bf16 each, over the loaded tiles (a warp only touches its own rows) ----
    if (live) {
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            uint32_t kfh[4], kfl[4], kbh[4], kbl[4], qfh[4], qfl[4], qbh[4], qbl[4];
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                const int j = 2 * m + jj;
                if (j < NP) {
                    float b[4], x[4];
                    const float2 cf = carry(0, j), cb = carry(1, j);
                    mma_k16_from(b, tri_i, kOnes, 0u, tri_i, fa[m][2 * jj], fa[m][2 * jj + 1], cf.x, cf.y);
                    mma_k16_from(x, tri_x, kOnes, 0u, tri_x, ba[m][2 * jj], ba[m][2 * jj + 1], cb.x, cb.y);
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const uint32_t qw = qa[m][2 * jj + r], kw = ka[m][2 * jj + r];
                        const f32x2 q2 = pack2(__uint_as_float(qw << 16), __uint_as_float(qw & 0xffff0000u));
                        const f32x2 k2 = pack2(__uint_as_float(kw << 16), __uint_as_float(kw & 0xffff0000u));
                        float b0, b1, x0, x1;
                        unpack2(fmul2(pack2(b[2 * r], b[2 * r + 1]), pack2(kLog2e, kLog2e)), b0, b1);
                        unpack2(fmul2(pack2(x[2 * r], x[2 * r + 1]), pack2(kLog2e, kLog2e)), x0, x1);
                        split_bf16(fmul2(q2, pack2(ex2(b0), ex2(b1))), qfh[2 * jj + r], qfl[2 * jj + r]);
                        split_bf16(fmul2(k2, pack2(ex2(-b0), ex2(-b1))), kfh[2 * jj + r], kfl[2 * jj + r]);
                        split_bf16(fmul2(q2, pack2(ex2(-x0), ex2(-x1))), qbh[2 * jj + r], qbl[2 * jj + r]);
                        split_bf16(fmul2(k2, pack2(ex2(x0), ex2(x1))), kbh[2 * jj + r], kbl[2 * jj + r]);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < 2; ++r) qfh[2 + r] = qfl[2 + r] = kfh[2 + r] = kfl[2 + r] = qbh[2 + r] = qbl[2 + r] = kbh[2 + r] = kbl[2 + r] = 0u;
                }
            }
            t64.store(op(kKf), 16 * wt, m, kfh[0], kfh[1], kfh[2], kfh[3]);
            t64.store(op(kKf + 1), 16 * wt, m, kfl[0], kfl[1], kfl[2], kfl[3]);
            t64.store(op(kKb), 16 * wt, m, kbh[0], kbh[1], kbh[2], kbh[3]);
            t64.store(op(kKb + 1), 16 * wt, m, kbl[0], kbl[1], kbl[2], kbl[3]);
            t64.store(op(kQf), 16 * wt, m, qfh[0], qfh[1], qfh[2], qfh[3]);
            t64.store(op(kQf + 1), 16 * wt, m, qfl[0], qfl[1], qfl[2], qfl[3]);
            t64.store(op(kQb), 16 * wt, m, qbh[0], qbh[1], qbh[2], qbh[3]);
            t64.store(op(kQb + 1), 16 * wt, m, qbl[0], qbl[1], qbl[2], qbl[3]);
        }
    }
    ok = mbar_wait_bounded(bar + 40, 0) && ok;
    ok = __syncthreads_and(ok);
    if (MODE == kPair) {
        cluster_wait();
    } else if (!ok) {   // a load that never lands: report it and leave, all threads together, nothing stored
        if (tid == 0) atomicOr(a.dev_status, kDevStatusTimeout);
        if (MODE == kSummary && tid == 0) a.flags[unit * nch + chunk] = 2;   // (nor by the launches behind this one)
        if (MODE == kMain) pdl_wait();   // (no block ends before the fold: what comes next only waits for this launch)
        return;
    }

    // ---- the chunk's own states, transposed: rows of v or g times the scaled operands, 16 value columns a job ----
    if (MODE == kPair || MODE == kSummary) {
        constexpr int NK = MODE == kPair ? 2 : 4;   // states of this chunk
        for (int job = w; job < NK * MV; job += nw) {
            const int mt = job / NK;   // 16 value columns
            // kinds S>, Z<, S<, Z>; the left chunk of a pair owes the right one S> and Z<, the right one the left one S< and Z>
            const int kind = MODE == kPair ? (chunk == 0 ? 0 : 2) + job % NK : job % NK;
            const int o = kind == 0 ? kKf : (kind == 1 ? kQb : (kind == 2 ? kKb : kQf));
            float u[2 * MP][4];
#pragma unroll
            for (int j = 0; j < 2 * MP; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) u[j][e] = 0.f;
            uint32_t left = ((kind & 1) ? tg : tv) + (tvv.off_b[0] ^ (uint32_t)(mt << 5)), right = op(o);   // (the piece bits of an offset are its swizzle alone)
#pragma unroll 2
            for (int t = 0; t < nT; ++t, left += 16 * RV, right += 1024) {
                uint32_t va[4];
                ldsm_trans(left, va);
#pragma unroll
                for (int m = 0; m < MP; ++m) {
                    uint32_t h[4], l[4];
                    t64.load_trans(right, 0, m, h);
                    t64.load_trans(right + lay.op_bytes, 0, m, l);
                    mma_k16(u[2 * m], va, h[0], h[1]);
                    mma_k16(u[2 * m + 1], va, h[2], h[3]);   // (an odd last tile of key dimensions is computed on padding and dropped)
                    mma_k16(u[2 * m], va, l[0], l[1]);
                    mma_k16(u[2 * m + 1], va, l[2], l[3]);
                }
            }
            if (kind < 2) {   // from the chunk's start to its end
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 e = *reinterpret_cast<const float2*>(ends + kind * 32 + 8 * j + 2 * c);
                    const float d0 = ex2(e.x * kLog2e), d1 = ex2(e.y * kLog2e);
                    u[j][0] *= d0; u[j][1] *= d1; u[j][2] *= d0; u[j][3] *= d1;
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int n = 16 * mt + 8 * r + g;
                if (MODE == kSummary) {
#pragma unroll
                    for (int j = 0; j < NP; ++j)
                        *reinterpret_cast<float2*>(a.u + (((unit * nch + chunk) * 4 + kind) * DV + n) * DK + 8 * j + 2 * c) =
                            make_float2(u[j][2 * r], u[j][2 * r + 1]);
                } else {   // as whole 16-byte pieces of the other block's state tiles
                    uint32_t hi[4] = {0u, 0u, 0u, 0u}, lo[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int j = 0; j < NP; ++j) split_bf16(pack2(u[j][2 * r], u[j][2 * r + 1]), hi[j], lo[j]);
                    transpose4(hi, c);
                    transpose4(lo, c);
                    if (c < NP) {
                        const uint32_t at = cluster_peer(tst + (uint32_t)(kind & 1) * 2 * kState + n * 64 + ((c ^ ((n >> 1) & 3)) << 4), 1 - chunk);
                        const uint32_t peer_bar = cluster_peer(bar + 8, 1 - chunk);
                        st_async4(at, hi[0], hi[1], hi[2], hi[3], peer_bar);
                        st_async4(at + kState, lo[0], lo[1], lo[2], lo[3], peer_bar);
                    }
                }
            }
        }
        if (MODE == kSummary) {
            for (int x = tid; x < 64; x += nw * 32)
                if ((x & 31) < DK) a.decay[(unit * nch + chunk) * 64 + x] = ex2(ends[x] * kLog2e);
            if (tid == 0) a.flags[unit * nch + chunk] = state_word[0];
            return;
        }
        if (tid == 0) st_async1(cluster_peer(bar + 16 + 4, 1 - chunk), (uint32_t)(state_word[0] | (ok ? 0 : 2)), cluster_peer(bar + 8, 1 - chunk));
    }
    if (MODE == kMain) {
        int slow = 0;
        for (int x = tid; x < nch; x += blockDim.x) slow |= (int)ld_gpu4(a.flags + unit * nch + x);
        const bool missing = __syncthreads_or(slow & 2);
        if (__syncthreads_or(slow)) {
            pdl_wait();
            if (missing) return;             // a summary of this unit did not get its inputs, and has said so
            if (chunk == 0 && tid == 0) atomicAdd(a.dev_status + 1, 1);
            gradient_by_walks<DK, DV>(walk_args(), unit, chunk, nch, reinterpret_cast<float*>(smem), lay.bar);
            return;
        }
        if (w == 0) pdl_wait();   // the fold
        if (tid == 0) {
            pdl_launch_dependents();
            mbar_expect_tx(bar + 8, 8 * kState);
            bulk_load(tst, a.img + (unit * nch + chunk) * 8 * kState, 8 * kState, bar + 8);
        }
    }
    if (MODE == kSingle && state_word[0]) {
        if (tid == 0) atomicAdd(a.dev_status + 1, 1);
        gradient_by_walks<DK, DV>(walk_args(), unit, 0, 1, reinterpret_cast<float*>(smem), lay.bar);
        return;
    }

    const DiagonalMask dmask(g, c);
    // Every sum below runs over the tiles up to the warp's own (the left side) and from it on (the right side): a loop, the
    // two halves of the diagonal tile, a loop, so that no loop carries the masks or a change of operands (as one loop over
    // nT + 1 steps with both inside, the moves and selects of a step were as many as its products: 43 M warp instructions
    // at 768 units of 196 tokens, 32 x 64, against 37 M).

    // ---- dq, dk: the scores D = g v^T (this warp's tokens as queries), then D^T (as keys), split, times the scaled operands ----
    float sum[2][2][NP][4];   // [dq, dk][left, right side], not yet scaled
    if (live) {
        uint32_t ra[MV][4];
        // scores of this warp's rows against a tile of rows, split, times that tile's operand pair; keep: 0 all scores, 1 left, 2 right
        auto tile = [&](uint32_t s_tile, uint32_t o_tile, float (&acc)[NP][4], int keep) {
            float d0[4], d1[4];
#pragma unroll
            for (int m = 0; m < MV; ++m) {
                uint32_t r[4];
                tvv.load_b(s_tile, 0, m, r);
                if (m == 0) {
                    mma_k16_zero(d0, ra[0], r[0], r[1]);
                    mma_k16_zero(d1, ra[0], r[2], r[3]);
                } else {
                    mma_k16(d0, ra[m], r[0], r[1]);
                    mma_k16(d1, ra[m], r[2], r[3]);
                }
            }
            uint32_t ah[4], al[4];
            split_bf16(pack2(d0[0], d0[1]), ah[0], al[0]);
            split_bf16(pack2(d0[2], d0[3]), ah[1], al[1]);
            split_bf16(pack2(d1[0], d1[1]), ah[2], al[2]);
            split_bf16(pack2(d1[2], d1[3]), ah[3], al[3]);
            if (keep) {
                dmask.apply(ah, keep == 1);
                dmask.apply(al, keep == 1);
            }
#pragma unroll
            for (int m = 0; m < MP; ++m) {
                uint32_t h[4], l[4];
                t64.load_trans(o_tile, 0, m, h);
                t64.load_trans(o_tile + lay.op_bytes, 0, m, l);
                mma_k16(acc[2 * m], ah, h[0], h[1]);
                if (2 * m + 1 < NP) mma_k16(acc[2 * m + 1 < NP ? 2 * m + 1 : 0], ah, h[2], h[3]);
                mma_k16(acc[2 * m], al, h[0], h[1]);
                if (2 * m + 1 < NP) mma_k16(acc[2 * m + 1 < NP ? 2 * m + 1 : 0], al, h[2], h[3]);
                mma_k16(acc[2 * m], ah, l[0], l[1]);
                if (2 * m + 1 < NP) mma_k16(acc[2 * m + 1 < NP ? 2 * m + 1 : 0], ah, l[2], l[3]);
            }
        };
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            // dq: g rows against v tiles, k~> left, k~< right;  dk: v rows against g tiles, q~< left, q~> right
#pragma unroll
            for (int m = 0; m < MV; ++m) tvv.load(pass == 0 ? tg : tv, 16 * wt, m, ra[m]);
#pragma unroll
            for (int side = 0; side < 2; ++side)
#pragma unroll
                for (int j = 0; j < NP; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) sum[pass][side][j][e] = 0.f;
            uint32_t s_tile = pass == 0 ? tv : tg, o_tile = op(pass == 0 ? kKf : kQb);
#pragma unroll 1
            for (int j = 0; j < wt; ++j, s_tile += 16 * RV, o_tile += 1024) tile(s_tile, o_tile, sum[pass][0], 0);
            tile(s_tile, o_tile, sum[pass][0], 1);
            o_tile = op(pass == 0 ? kKb : kQf) + wt * 1024;
            tile(s_tile, o_tile, sum[pass][1], 2);
#pragma unroll 1
            for (int j = wt + 1; j < nT; ++j) {
                s_tile += 16 * RV;
                o_tile += 1024;
                tile(s_tile, o_tile, sum[pass][1], 0);
            }
        }
    }

    // ---- the states at the chunk's borders ----
    const bool has_left = MODE == kMain ? chunk > 0 : (MODE == kPair && chunk == 1);
    const bool has_right = MODE == kMain ? chunk + 1 < nch : (MODE == kPair && chunk == 0);
    // S> and Z< from the left, S< and Z> from the right, hi and lo tiles each; a block of a pair has two of them
    const uint32_t st_left = tst, st_right = tst + (MODE == kMain ? 4 : 0) * kState;
    if (MODE == kPair) {
        const int here = __syncthreads_or(!(mbar_wait_bounded(bar + 8, 0) && ok)) ? 2 : 0;
        const int word = here ? here : state_word[0] | state_word[1];
        if (word) {
            if (word & 2) {
                if (chunk == 0 && ok && here) mbar_wait_bounded(bar + 32, 0);   // (the other block does not know and may send its sums)
                if (tid == 0) atomicOr(a.dev_status, kDevStatusTimeout);
                return;
            }
            if (chunk == 0 && tid == 0) atomicAdd(a.dev_status + 1, 1);
            gradient_by_walks<DK, DV>(walk_args(), unit, chunk, nch, reinterpret_cast<float*>(smem), lay.bar);
            return;
        }
    }
    if (MODE == kMain) {
        ok = __syncthreads_and(mbar_wait_bounded(bar + 8, 0));
        if (!ok) {
            if (tid == 0) atomicOr(a.dev_status, kDevStatusTimeout);
            return;
        }
    }
    if (MODE != kSingle && live) {   // what the border states add to the sums
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            uint32_t ra[MV][4];
#pragma unroll
            for (int m = 0; m < MV; ++m) tvv.load(pass == 0 ? tg : tv, 16 * wt, m, ra[m]);
            auto state_product = [&](uint32_t st, float (&acc)[NP][4]) {
#pragma unroll
                for (int kk = 0; kk < MV; ++kk) {
#pragma unroll
                    for (int m = 0; m < MP; ++m) {
                        uint32_t h[4], l[4];
                        t64.load_trans(st, 16 * kk, m, h);
                        t64.load_trans(st + kState, 16 * kk, m, l);
                        mma_k16(acc[2 * m], ra[kk], h[0], h[1]);
                        if (2 * m + 1 < NP) mma_k16(acc[2 * m + 1 < NP ? 2 * m + 1 : 0], ra[kk], h[2], h[3]);
                        mma_k16(acc[2 * m], ra[kk], l[0], l[1]);
                        if (2 * m + 1 < NP) mma_k16(acc[2 * m + 1 < NP ? 2 * m + 1 : 0], ra[kk], l[2], l[3]);
                    }
                }
            };
            if (has_left) state_product(st_left + (pass == 0 ? 0 : 2) * kState, sum[pass][0]);
            if (has_right) {   // times the chunk's own decay, from its end to its start: log alpha< for S<, log alpha> for Z>
                float acc[NP][4];
#pragma unroll
                for (int j = 0; j < NP; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
                state_product(st_right + (pass == 0 ? 0 : 2) * kState, acc);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 e = *reinterpret_cast<const float2*>(ends + (pass == 0 ? 32 : 0) + 8 * j + 2 * c);
                    const float f0 = ex2(e.x * kLog2e), f1 = ex2(e.y * kLog2e);
                    float (&to)[4] = sum[pass][1][j];
                    to[0] = fmaf(f0, acc[j][0], to[0]); to[1] = fmaf(f1, acc[j][1], to[1]);
                    to[2] = fmaf(f0, acc[j][2], to[2]); to[3] = fmaf(f1, acc[j][3], to[3]);
                }
            }
        }
    }
    // ---- dq, dk and E (q, k and the gates are read once more, from L2: keeping them costs the registers of the passes) ----
    float ef_[NP][4], eb_[NP][4];
    if (live) {
        const size_t at = (unit * L + row0 + 16 * wt + g) * DK + 2 * c;
        const bool in0 = row0 + 16 * wt + g < L, in1 = row0 + 16 * wt + 8 + g < L;
        auto word = [&](const __nv_bfloat16* p, int j, int r) {
            return (r ? in1 : in0) ? *reinterpret_cast<const uint32_t*>(p + at + 8 * r * DK + 8 * j) : 0u;
        };
        uint32_t lf[NP][2], lb[NP][2], qw[NP][2], kw[NP][2];
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                lf[j][r] = word(a.la_f, j, r);
                lb[j][r] = word(a.la_b, j, r);
                qw[j][r] = word(a.q, j, r);
                kw[j][r] = word(a.k, j, r);
            }
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            float b[4], x[4];
            const float2 cf = carry(0, j), cb = carry(1, j);
            mma_k16_from(b, tri_i, kOnes, 0u, tri_i, movmatrix(lf[j][0]), movmatrix(lf[j][1]), cf.x, cf.y);
            mma_k16_from(x, tri_x, kOnes, 0u, tri_x, movmatrix(lb[j][0]), movmatrix(lb[j][1]), cb.x, cb.y);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float b0, b1, x0, x1;
                unpack2(fmul2(pack2(b[2 * r], b[2 * r + 1]), pack2(kLog2e, kLog2e)), b0, b1);
                unpack2(fmul2(pack2(x[2 * r], x[2 * r + 1]), pack2(kLog2e, kLog2e)), x0, x1);
                // left side of dq and right side of dk are the forward direction
                const f32x2 qf = fmul2(pack2(sum[0][0][j][2 * r], sum[0][0][j][2 * r + 1]), pack2(ex2(b0), ex2(b1)));
                const f32x2 qb = fmul2(pack2(sum[0][1][j][2 * r], sum[0][1][j][2 * r + 1]), pack2(ex2(-x0), ex2(-x1)));
                const f32x2 kb = fmul2(pack2(sum[1][0][j][2 * r], sum[1][0][j][2 * r + 1]), pack2(ex2(x0), ex2(x1)));
                const f32x2 kf = fmul2(pack2(sum[1][1][j][2 * r], sum[1][1][j][2 * r + 1]), pack2(ex2(-b0), ex2(-b1)));
                const f32x2 q2 = pack2(__uint_as_float(qw[j][r] << 16), __uint_as_float(qw[j][r] & 0xffff0000u));
                const f32x2 k2 = pack2(__uint_as_float(kw[j][r] << 16) * -1.f, __uint_as_float(kw[j][r] & 0xffff0000u) * -1.f);
                float s0, s1;
                if (r ? in1 : in0) {
                    unpack2(fadd2(qf, qb), s0, s1);
                    *reinterpret_cast<uint32_t*>(a.dq + at + 8 * r * DK + 8 * j) = mul_bf16x2(pack_bf16(s0, s1), 0x3F003F00u);   // x 1/2: exact
                    unpack2(fadd2(kf, kb), s0, s1);
                    *reinterpret_cast<uint32_t*>(a.dk + at + 8 * r * DK + 8 * j) = mul_bf16x2(pack_bf16(s0, s1), 0x3F003F00u);
                }
                unpack2(ffma2(q2, qf, fmul2(k2, kf)), ef_[j][2 * r], ef_[j][2 * r + 1]);
                unpack2(ffma2(q2, qb, fmul2(k2, kb)), eb_[j][2 * r], eb_[j][2 * r + 1]);
            }
        }
    }
    // ---- dv: keys of this warp against queries before (<) and after (>) ----
    float o[NV][4];
#pragma unroll
    for (int n = 0; n < NV; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
    if (live) {
        uint32_t kk[MP][4];
        auto own_keys = [&](int which) {
#pragma unroll
            for (int m = 0; m < MP; ++m) t64.load(op(which), 16 * wt, m, kk[m]);
        };
        auto tile = [&](uint32_t q_tile, uint32_t g_tile, int keep) {
            float d0[4], d1[4];
#pragma unroll
            for (int m = 0; m < MP; ++m) {
                uint32_t r[4];
                t64.load_b(q_tile, 0, m, r);
                if (m == 0) {
                    mma_k16_zero(d0, kk[0], r[0], r[1]);
                    mma_k16_zero(d1, kk[0], r[2], r[3]);
                } else if (2 * m + 1 < NP) {
                    mma_k16(d0, kk[m], r[0], r[1]);
                    mma_k16(d1, kk[m], r[2], r[3]);
                } else {
                    mma_k8(d0, kk[m][0], kk[m][1], r[0]);
                    mma_k8(d1, kk[m][0], kk[m][1], r[2]);
                }
            }
            uint32_t p[4] = {pack_bf16(d0[0], d0[1]), pack_bf16(d0[2], d0[3]), pack_bf16(d1[0], d1[1]), pack_bf16(d1[2], d1[3])};
            if (keep) dmask.apply(p, keep == 1);
#pragma unroll
            for (int n2 = 0; n2 < MV; ++n2) {
                uint32_t r[4];
                tvv.load_trans(g_tile, 0, n2, r);
                mma_k16(o[2 * n2], p, r[0], r[1]);
                mma_k16(o[2 * n2 + 1], p, r[2], r[3]);
            }
        };
        own_keys(kKb);
        uint32_t q_tile = op(kQb), g_tile = tg;
#pragma unroll 1
        for (int j = 0; j < wt; ++j, q_tile += 1024, g_tile += 16 * RV) tile(q_tile, g_tile, 0);
        tile(q_tile, g_tile, 1);
        own_keys(kKf);
        q_tile = op(kQf) + wt * 1024;
        tile(q_tile, g_tile, 2);
#pragma unroll 1
        for (int j = wt + 1; j < nT; ++j) {
            q_tile += 1024;
            g_tile += 16 * RV;
            tile(q_tile, g_tile, 0);
        }
        if (MODE != kSingle) {   // dv from the border states, one bf16 per operand
#pragma unroll 1
            for (int side = 0; side < 2; ++side) {
                if (!(side == 0 ? has_left : has_right)) continue;
                const uint32_t st = (side == 0 ? st_left : st_right) + 2 * kState;   // Z< or Z>
#pragma unroll
                for (int m = 0; m < MP; ++m) {
                    t64.load(op(side == 0 ? kKb : kKf), 16 * wt, m, kk[m]);
                    if (side == 1) {   // from the chunk's end to its start
#pragma unroll
                        for (int jj = 0; jj < 2; ++jj) {
                            const float2 e = *reinterpret_cast<const float2*>(ends + 8 * (2 * m + jj < NP ? 2 * m + jj : 0) + 2 * c);
                            const uint32_t d = pack_bf16(ex2(e.x * kLog2e), ex2(e.y * kLog2e));
                            kk[m][2 * jj] = mul_bf16x2(kk[m][2 * jj], d);
                            kk[m][2 * jj + 1] = mul_bf16x2(kk[m][2 * jj + 1], d);
                        }
                    }
                }
#pragma unroll
                for (int n2 = 0; n2 < MV; ++n2) {
#pragma unroll
                    for (int m = 0; m < MP; ++m) {
                        uint32_t r[4];
                        t64.load_b(st, 16 * n2, m, r);
                        if (2 * m + 1 < NP) {
                            mma_k16(o[2 * n2], kk[m], r[0], r[1]);
                            mma_k16(o[2 * n2 + 1], kk[m], r[2], r[3]);
                        } else {
                            mma_k8(o[2 * n2], kk[m][0], kk[m][1], r[0]);
                            mma_k8(o[2 * n2 + 1], kk[m][0], kk[m][1], r[2]);
                        }
                    }
                }
            }
        }
        __nv_bfloat16* op_ = a.dv + (unit * L + row0) * DV;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = 16 * wt + 8 * r + g;
            if (row0 + row < L) {
                uint32_t* rp = reinterpret_cast<uint32_t*>(op_ + (size_t)row * DV + 2 * c);
#pragma unroll
                for (int n = 0; n < NV; ++n) rp[4 * n] = mul_bf16x2(pack_bf16(o[n][2 * r], o[n][2 * r + 1]), 0x3F003F00u);
            }
        }
    }
    if (MODE == kMain && has_right) {
        // Row sums of S> o Z> and of Z< o S< at the right border: what the tokens after the chunk add to its gate gradients.
        const int j = tid & 3;
        float pf[8], pb[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) pf[e] = pb[e] = 0.f;
        if (j < NP) {
#pragma unroll 1
            for (int n = tid >> 2; n < DV; n += nw * 8) {
                const uint32_t off = n * 64 + ((j ^ ((n >> 1) & 3)) << 4);
#pragma unroll
                for (int x = 0; x < 2; ++x) {   // x = 0: S> of the chunk on the right with Z> here;  1: Z< there with S< here
                    const uint8_t* p = a.img + (unit * nch + chunk + 1) * 8 * kState + off + 2 * x * kState;
                    const uint4 fh = *reinterpret_cast<const uint4*>(p), fl = *reinterpret_cast<const uint4*>(p + kState);
                    const uint8_t* own = smem + (st_right - base) + (x == 0 ? 2 : 0) * kState + off;
                    const uint4 oh = *reinterpret_cast<const uint4*>(own), ol = *reinterpret_cast<const uint4*>(own + kState);
                    const uint32_t fhw[4] = {fh.x, fh.y, fh.z, fh.w}, flw[4] = {fl.x, fl.y, fl.z, fl.w};
                    const uint32_t ohw[4] = {oh.x, oh.y, oh.z, oh.w}, olw[4] = {ol.x, ol.y, ol.z, ol.w};
                    float (&acc)[8] = x == 0 ? pf : pb;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        acc[2 * e] = fmaf(__uint_as_float(fhw[e] << 16) + __uint_as_float(flw[e] << 16),
                                          __uint_as_float(ohw[e] << 16) + __uint_as_float(olw[e] << 16), acc[2 * e]);
                        acc[2 * e + 1] = fmaf(__uint_as_float(fhw[e] & 0xffff0000u) + __uint_as_float(flw[e] & 0xffff0000u),
                                              __uint_as_float(ohw[e] & 0xffff0000u) + __uint_as_float(olw[e] & 0xffff0000u), acc[2 * e + 1]);
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
#pragma unroll
            for (int m = 4; m <= 16; m <<= 1) {
                pf[e] += __shfl_xor_sync(0xffffffffu, pf[e], m);
                pb[e] += __shfl_xor_sync(0xffffffffu, pb[e], m);
            }
        }
        if (lane < NP) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                part[(w * 2) * 32 + 8 * lane + e] = pf[e];
                part[(w * 2 + 1) * 32 + 8 * lane + e] = pb[e];
            }
        }
    }
    __syncthreads();   // every warp is done with the operand tiles
    // ---- suffix sums of E: within the warp's tile, one pair of key dimensions of one direction per lane, then over the tiles
    // and the border ----
    constexpr int kPitch = 40;   // floats: eight rows apart in different banks
    float* e_w = reinterpret_cast<float*>(smem + lay.op) + wt * 2 * 16 * kPitch;
    const int dir = lane >> 4, dp = lane & 15;
    const bool scan = live && dp < DK / 2;
    f32x2 es[16];
    if (live) {
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                *reinterpret_cast<float2*>(e_w + (8 * r + g) * kPitch + 8 * j + 2 * c) = make_float2(ef_[j][2 * r], ef_[j][2 * r + 1]);
                *reinterpret_cast<float2*>(e_w + (16 + 8 * r + g) * kPitch + 8 * j + 2 * c) = make_float2(eb_[j][2 * r], eb_[j][2 * r + 1]);
            }
        __syncwarp();
        if (scan) {
            const float* src = e_w + dir * 16 * kPitch + 2 * dp;
            f32x2 run = 0ull;   // (+0, +0)
#pragma unroll
            for (int t = 15; t >= 0; --t) {   // > takes its own token, < does not (the rows past the end hold zeros)
                const f32x2 e = *reinterpret_cast<const f32x2*>(src + t * kPitch);
                const f32x2 next = fadd2(run, e);
                es[t] = dir == 0 ? next : run;
                run = next;
            }
            *reinterpret_cast<f32x2*>(totals + (wt * 2 + dir) * 32 + 2 * dp) = run;
        }
    }
    __syncthreads();
    if (MODE == kPair) {   // the right chunk's sums are what the left one's gate gradients lack
        if (chunk == 1) {
            if (w == 0 && dp < DK / 2) {
                f32x2 all = 0ull;
                for (int x = nT - 1; x >= 0; --x) all = fadd2(all, *reinterpret_cast<const f32x2*>(totals + (x * 2 + dir) * 32 + 2 * dp));
                float s0, s1;
                unpack2(all, s0, s1);
                const uint32_t at = cluster_peer(smem_u32(part) + (dir * 32 + 2 * dp) * 4, 0), peer_bar = cluster_peer(bar + 32, 0);
                st_async1(at, __float_as_uint(s0), peer_bar);
                st_async1(at + 4, __float_as_uint(s1), peer_bar);
            }
        } else if (!__syncthreads_and(mbar_wait_bounded(bar + 32, 0) && a.expire_wait != 2)) {   // no gate gradients from sums that are not there
            if (tid == 0) atomicOr(a.dev_status, kDevStatusTimeout);
            return;
        }
    }
    if (scan) {
        f32x2 rest = 0ull;
        if (MODE != kSingle && has_right) {
            if (MODE == kPair) {
                rest = *reinterpret_cast<const f32x2*>(part + dir * 32 + 2 * dp);
            } else {
                for (int x = 0; x < nw; ++x) rest = fadd2(rest, *reinterpret_cast<const f32x2*>(part + (x * 2 + dir) * 32 + 2 * dp));
                if (dir == 1) rest = fmul2(rest, pack2(-1.f, -1.f));   // (the sum of E< over the tokens after the chunk is minus the border's)
            }
        }
        for (int x = nT - 1; x > wt; --x) rest = fadd2(rest, *reinterpret_cast<const f32x2*>(totals + (x * 2 + dir) * 32 + 2 * dp));
        const uint32_t half = dir == 0 ? 0x3F003F00u : 0xBF00BF00u;   // x 1/2, and the sign of the < direction
        __nv_bfloat16* dst = (dir == 0 ? a.dla_f : a.dla_b) + (unit * L + row0 + 16 * wt) * DK + 2 * dp;
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            float s0, s1;
            unpack2(fadd2(es[t], rest), s0, s1);
            if (row0 + 16 * wt + t < L) *reinterpret_cast<uint32_t*>(dst + t * DK) = mul_bf16x2(pack_bf16(s0, s1), half);
        }
    }
}

// Second launch of a long call: the states entering every chunk, from the chunks' own: S> and Z< ascending, S< and Z> descending.
template <int DK, int DV, int GROUPS, int RUN>
__global__ void __launch_bounds__(kFoldThreads, fold_blocks_per_sm(RUN)) grad_fold_kernel(const GArgs a) {
    constexpr int P = DK / 4, kItems = kFoldThreads / GROUPS;
    constexpr int kState = (int)GLayout<DV>::kState;
    const size_t unit = blockIdx.x;
    const int kind = blockIdx.y, dir = (kind == 0 || kind == 3) ? 0 : 1;   // S>, Z> decay by log alpha>
    const bool up = kind < 2;
    const int item = threadIdx.x % kItems, grp = threadIdx.x / kItems, x = blockIdx.z * kItems + item, nch = a.nch;
    const int run = (nch + GROUPS - 1) / GROUPS, i0 = min(nch, grp * run), i1 = min(nch, i0 + run);   // in walking order
    const bool in = x < P * DV;
    const int p = in ? x % P : 0, n = in ? x / P : 0;
    const int step = up ? 1 : -1;
    const size_t first = unit * nch + (up ? i0 : nch - 1 - i0);
    uint8_t* img = a.img + (first * 4 + kind) * 2 * kState + n * 64 + (((p >> 1) ^ ((n >> 1) & 3)) << 4) + 8 * (p & 1);
    pdl_wait();
    pdl_launch_dependents();
    fold_runs<GROUPS, RUN>(a.u + ((first * 4 + kind) * DV + n) * DK + 4 * p, step * (4 * DV * DK), a.decay + first * 64 + dir * 32 + 4 * p, step * 64, run, i1 - i0, in,
                      item, grp, [&](int i, float4 carry, float4) {
                          uint2 hi, lo;
                          split_bf16(pack2(carry.x, carry.y), hi.x, lo.x);
                          split_bf16(pack2(carry.z, carry.w), hi.y, lo.y);
                          uint8_t* to = img + (ptrdiff_t)(i * step) * (8 * kState);
                          *reinterpret_cast<uint2*>(to) = hi;
                          *reinterpret_cast<uint2*>(to + kState) = lo;
                      });
}

// How a sequence is cut: one chunk of up to eight tiles, two of up to seven, else chunks of six.
struct GPlan {
    int mode, tiles, nch;
};
GPlan grad_plan(int L) {
    const int T = (L + 15) / 16;
    if (T <= max_tiles(kSingle)) return {kSingle, T, 1};
    if (T <= 2 * max_tiles(kPair)) return {kPair, (T + 1) / 2, 2};
    return {kMain, max_tiles(kMain), (T + max_tiles(kMain) - 1) / max_tiles(kMain)};
}
struct GScratch {
    size_t u, img, decay, flags, total;   // byte offsets
};
GScratch grad_scratch(const GPlan& p, long long units, int dk, int dv) {
    GScratch s{};
    if (p.mode != kMain) return s;
    const size_t n = (size_t)units * p.nch;
    s.u = 0;
    s.img = n * 4 * dk * dv * 4;
    s.decay = s.img + n * 8 * dv * 64;
    s.flags = s.decay + n * 64 * 4;
    s.total = (s.flags + n * 4 + 255) / 256 * 256;
    return s;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_grad(void (*kernel)(KArgs...), unsigned grid, int threads, size_t smem, bool pair, cudaStream_t stream, Args&&... args) {
    count_launch();
    return launch_pdl_cluster(kernel, dim3(grid), dim3(threads), smem, pair ? 2 : 1, stream, static_cast<KArgs>(args)...);
}

template <int DK, int DV>
cudaError_t launch_grad_t(GArgs a, const GPlan& p, long long units, cudaStream_t stream) {
    const int rows = p.tiles * 16, vrow = DV == 32 ? 32 : 64;
    CUtensorMap tq, tk, tf, tb, tv, tg;
    if (!make_map(&tq, a.q, units, a.L, DK, 32, rows) || !make_map(&tk, a.k, units, a.L, DK, 32, rows) ||
        !make_map(&tf, a.la_f, units, a.L, DK, 32, rows) || !make_map(&tb, a.la_b, units, a.L, DK, 32, rows) ||
        !make_map(&tv, a.v, units, a.L, DV, vrow, rows) || !make_map(&tg, a.g, units, a.L, DV, vrow, rows))
        return cudaErrorInvalidValue;
    static std::atomic<int> sms_of[64];   // 0: the instances of this device are not configured yet
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = sms_of[dev].load(std::memory_order_acquire);
    if (sms == 0) {
        auto opt_in = [&](auto kernel, int mode) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GLayout<DV>(max_tiles(mode), mode).total);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        };
        opt_in(bigla_grad_kernel<DK, DV, kSingle>, kSingle);
        opt_in(bigla_grad_kernel<DK, DV, kPair>, kPair);
        opt_in(bigla_grad_kernel<DK, DV, kMain>, kMain);
        opt_in(bigla_grad_kernel<DK, DV, kSummary>, kSummary);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        sms_of[dev].store(sms, std::memory_order_release);
    }
    // Two blocks per SM.  The summary launch of a long call fits three where they have one warp per tile: worth the uneven share of its
    // jobs in the larger calls (training step of 8 x 4 units of 4096 tokens, 24 x 48: 159.5 to 154.3 us; 24 x 6 of 300, 32 x 64: 80.8 to 82.5).
    const bool three = p.mode == kMain && units * p.nch > 4LL * sms && DK * DV > 512;
    a.ahead = (three ? 3 : 2) * sms;
    const unsigned grid = (unsigned)(units * p.nch);
    auto threads = [&](int mode) { return 32 * grad_warps(mode, p.tiles); };
    if (p.mode == kSingle)
        e = launch_grad(bigla_grad_kernel<DK, DV, kSingle>, grid, threads(kSingle), GLayout<DV>(p.tiles, kSingle).total, false, stream, tq, tk, tf, tb, tv, tg, a);
    else if (p.mode == kPair)
        e = launch_grad(bigla_grad_kernel<DK, DV, kPair>, grid, threads(kPair), GLayout<DV>(p.tiles, kPair).total, true, stream, tq, tk, tf, tb, tv, tg, a);
    else {
        e = launch_grad(bigla_grad_kernel<DK, DV, kSummary>, grid, three ? 32 * p.tiles : threads(kSummary), GLayout<DV>(p.tiles, kSummary).total, false, stream, tq, tk, tf, tb, tv, tg, a);
        if (e == cudaSuccess) {
            count_launch();
            e = with_fold_plan(p.nch, units, 4, DK / 4 * DV, sms, [&](auto groups, auto run) {
                constexpr int kGroups = decltype(groups)::value, kItems = kFoldThreads / kGroups;
                return launch_pdl(grad_fold_kernel<DK, DV, kGroups, decltype(run)::value>, dim3((unsigned)units, 4, (DK / 4 * DV + kItems - 1) / kItems), dim3(kFoldThreads), 0, stream, a);
            });
        }
        a.expire_wait = 0;   // (of a long call the first launch)
        a.ahead = 2 * sms;
        if (e == cudaSuccess)
            e = launch_grad(bigla_grad_kernel<DK, DV, kMain>, grid, threads(kMain), GLayout<DV>(p.tiles, kMain).total, false, stream, tq, tk, tf, tb, tv, tg, a);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

bool grad_supported(long long units, int L, int dk, int dv) {
    // fewer tokens than one tile: the walks, which pad nothing
    return (dk == 16 || dk == 24 || dk == 32) && (dv == 32 || dv == 48 || dv == 64) && L >= 16 && units * grad_plan(L).nch <= 0x7fffffffLL;
}

size_t grad_scratch_bytes(long long units, int L, int dk, int dv) { return grad_scratch(grad_plan(L), units, dk, dv).total; }

cudaError_t launch_bigla_grad(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v, const __nv_bfloat16* la_f,
                              const __nv_bfloat16* la_b, const __nv_bfloat16* d_out, __nv_bfloat16* dq, __nv_bfloat16* dk_out,
                              __nv_bfloat16* dv_out, __nv_bfloat16* dla_f, __nv_bfloat16* dla_b, void* scratch, long long units, int L, int dk,
                              int dv, cudaStream_t stream) {
    const GPlan p = grad_plan(L);
    const GScratch s = grad_scratch(p, units, dk, dv);
    char* b = static_cast<char*>(scratch);
    GArgs a{q, k, v, la_f, la_b, d_out, dq, dk_out, dv_out, dla_f, dla_b, L, p.nch, p.tiles,
            reinterpret_cast<float*>(b + s.u), reinterpret_cast<uint8_t*>(b + s.img), reinterpret_cast<float*>(b + s.decay),
            reinterpret_cast<int*>(b + s.flags), units * p.nch, 0, device_status_ptr(), take_expire_next_wait()};
    if (!a.dev_status) return cudaErrorUnknown;
#define VIG_CASE(DK_, DV_) \
    if (dk == DK_ && dv == DV_) return launch_grad_t<DK_, DV_>(a, p, units, stream);
    VIG_CASE(16, 32) VIG_CASE(16, 48) VIG_CASE(16, 64)
    VIG_CASE(24, 32) VIG_CASE(24, 48) VIG_CASE(24, 64)
    VIG_CASE(32, 32) VIG_CASE(32, 48) VIG_CASE(32, 64)
#undef VIG_CASE
    return cudaErrorNotSupported;
}

}  // namespace vig
