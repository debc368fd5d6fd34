// Fold over the chunks of a sequence: the states that enter every chunk from what the chunks add, in(c + 1) = d(c) in(c) + own(c) in
// walking order, element by element of the state.
//
// A thread takes four key dimensions of one value column over a run of chunks, GROUPS runs side by side: what a run adds and by how
// much it decays, then the carry of the runs before it, then the states.  A run of up to RUN chunks is read once and kept in
// registers (but for 20 to 92 bytes that the blocks an SM is to hold leave to the stack, several runs side by side), a longer one twice, a
// batch at a time.  What bounds the launch is how many of its loads are in flight; and until its last
// block has started, the launch behind it, which runs under it, does not (8 x 4 units of 4096 tokens, 24 x 48: blocks of 100 registers
// in two rounds, each run read twice, 39.9 us a call; this way 37.7).
#pragma once
#include <cuda_runtime.h>
#include <type_traits>

namespace vig {

constexpr int kFoldThreads = 256;
constexpr int fold_blocks_per_sm(int run) { return run <= 4 ? 4 : 2; }   // what the registers of a run leave room for

// emit(i, carry, decay): the state that enters chunk i of this thread's run, and that chunk's decay.  Every thread of the block calls it.
template <int GROUPS, int RUN, typename Emit>
__device__ __forceinline__ void fold_runs(const float* own0, int own_step, const float* dec0, int dec_step, int run, int len, bool in, int item,
                                          int grp, const Emit& emit) {
    constexpr int kItems = kFoldThreads / GROUPS;
    __shared__ float4 s_state[GROUPS][kItems], s_decay[GROUPS][kItems];
    float4 own[RUN], d[RUN], carry = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int b0) {
#pragma unroll
        for (int b = 0; b < RUN; ++b) {
            if (b0 + b < len) {
                own[b] = *reinterpret_cast<const float4*>(own0 + (b0 + b) * own_step);
                d[b] = *reinterpret_cast<const float4*>(dec0 + (b0 + b) * dec_step);
            }
        }
    };
    auto step = [&](int b) {
        carry = make_float4(fmaf(d[b].x, carry.x, own[b].x), fmaf(d[b].y, carry.y, own[b].y), fmaf(d[b].z, carry.z, own[b].z), fmaf(d[b].w, carry.w, own[b].w));
    };
    const bool once = GROUPS > 1 && run <= RUN;
    if (in && once) fetch(0);
    if (GROUPS > 1) {
        float4 all = make_float4(1.f, 1.f, 1.f, 1.f);
        if (in) {
            for (int b0 = 0; b0 < len; b0 += RUN) {
                if (!once) fetch(b0);
#pragma unroll
                for (int b = 0; b < RUN; ++b) {
                    if (b0 + b < len) {
                        all = make_float4(all.x * d[b].x, all.y * d[b].y, all.z * d[b].z, all.w * d[b].w);
                        step(b);
                    }
                }
            }
        }
        s_state[grp][item] = carry;
        s_decay[grp][item] = all;
        __syncthreads();
        carry = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int y = 0; y < grp; ++y) {
            const float4 u = s_state[y][item], e = s_decay[y][item];
            carry = make_float4(fmaf(e.x, carry.x, u.x), fmaf(e.y, carry.y, u.y), fmaf(e.z, carry.z, u.z), fmaf(e.w, carry.w, u.w));
        }
    }
    if (in) {
        for (int b0 = 0; b0 < len; b0 += RUN) {
            if (!once) fetch(b0);
#pragma unroll
            for (int b = 0; b < RUN; ++b) {
                if (b0 + b < len) {
                    emit(b0 + b, carry, d[b]);
                    step(b);
                }
            }
        }
    }
}

// Runs side by side and chunks of a run for a sequence of nch chunks, and the launch: f(groups, run), compile-time numbers.  Few blocks
// where they do: the launch behind this one shares the chip with it (13 chunks of 16 units, 24 x 48, in four runs of 160 blocks instead
// of one of 64: 17.2 us a call instead of 14.1).  So up to 128 chunks in eight longer runs, read twice, where that gives every block of
// both launches an SM of its own and sixteen do not: the chunks' blocks would come to stand two on an SM beside idle ones.
// states, pieces: of a unit; a piece is four key dimensions of a value column.
template <typename F>
cudaError_t with_fold_plan(int nch, long long units, int states, int pieces, int sms, const F& f) {
    using std::integral_constant;
    auto apart = [&](int groups) {
        const int items = kFoldThreads / groups;
        return units * (states * ((pieces + items - 1) / items) + nch) <= sms;
    };
    if (nch <= 4) return f(integral_constant<int, 1>{}, integral_constant<int, 4>{});
    if (nch <= 24) return f(integral_constant<int, 1>{}, integral_constant<int, 8>{});
    if (nch <= 32) return f(integral_constant<int, 8>{}, integral_constant<int, 4>{});
    if (nch <= 64 || (nch <= 128 && apart(8) && !apart(16))) return f(integral_constant<int, 8>{}, integral_constant<int, 8>{});
    if (nch <= 128) return f(integral_constant<int, 16>{}, integral_constant<int, 8>{});
    return f(integral_constant<int, 32>{}, integral_constant<int, 8>{});
}

}  // namespace vig
