// Slice products of one K block of a split contraction, as tcgen05 MMAs (see mixed.cu).
#pragma once

#include "mixed.cuh"
#include "mma_schedule.h"
#include "tc_ptx.cuh"

namespace vfmm {

// All slice products (i, j), i + j <= S + 1, of one K block (mma_schedule.h): accumulator acc_of(i, j); on
// the first K block of a drain group the first product into each accumulator overwrites it (with
// S >= kMinSlices every accumulator gets one from slice 1 of A).
//
// One MMA with an N of up to 256 does several products of one A tile: 8 instead of 21 MMAs per 16 K values
// at S = 6, N = 64, each near the tensor pipe's rate (128 cycles at N = 256, where N = 64 alone takes 36
// and, with the stage's loads going on, 47).
template <bool kFirst, int S, int N>
__device__ __forceinline__ void issue_unit(uint32_t tmem, uint64_t ad0, uint64_t bd0) {
    constexpr uint32_t A_SLICE = kTileM * 64, B_SLICE = N * 64;
    static_assert(S >= kMinSlices && S <= kSlices && mma_schedule_ok(S, N), "slice count");
#pragma unroll
    for (int i = 1; i <= S; ++i)
#pragma unroll
        for (int ks = 0; ks < kKBlock / 16; ++ks) {
            // every MMA of one A tile in a row: it is read from shared memory once
            const uint64_t ad = ad0 + (((i - 1) * A_SLICE + ks * 32) >> 4);
            const int total = mma_count(S, N, i);
#pragma unroll
            for (int q = 0; q < total; ++q) {
                const MmaStep m = mma_step(S, N, i, q);
                const uint64_t bd = bd0 + (((m.j - 1) * B_SLICE + ks * 32) >> 4);
                const uint32_t d = tmem + acc_of(i, m.j) * N, idesc = tc::idesc_bf16_f32(kTileM, m.w * N);
                const uint32_t accum = (kFirst && i == 1 && ks == 0 && m.j <= kNumAcc) ? 0u : 1u;
                if (total == 1) tc::umma_bf16<tc::CollectA::kDiscard>(d, ad, bd, idesc, accum);
                else if (q == 0) tc::umma_bf16<tc::CollectA::kFill>(d, ad, bd, idesc, accum);
                else if (q < total - 1) tc::umma_bf16<tc::CollectA::kUse>(d, ad, bd, idesc, accum);
                else tc::umma_bf16<tc::CollectA::kLastUse>(d, ad, bd, idesc, accum);
            }
        }
}

}  // namespace vfmm
