// Slice products of one K block of a split contraction, as tcgen05 MMAs (see mixed.cu).
#pragma once

#include <type_traits>

#include "mixed.cuh"
#include "tc_ptx.cuh"

namespace vfmm {

// Accumulator of slice product (i, j): its diagonal i + j - 2; diagonals >= kNumAcc - 1 share the last.
__host__ __device__ constexpr int acc_of(int i, int j) { return (i + j - 2) < (kNumAcc - 1) ? (i + j - 2) : (kNumAcc - 1); }

// All slice products (i, j), i + j <= S + 1, of one K block: accumulator acc_of(i, j); on the
// first K block of a configuration the first product into each accumulator overwrites it (with
// S >= kMinSlices every accumulator gets one from slice 1 of A).
//
// Slices j, j + 1, ... of B are consecutive rows in shared memory and their accumulators (diagonals)
// consecutive columns in TMEM, so one MMA with an N of up to 256 does several products of one A tile:
// 8 instead of 21 MMAs per 16 K values at S = 6, N = 64, each near the tensor pipe's rate (128 cycles at
// N = 256, where N = 64 alone takes 36 and, with the stage's loads going on, 47).
template <bool kFirst, int S, int N>
__device__ __forceinline__ void issue_unit(uint32_t tmem, uint64_t ad0, uint64_t bd0) {
    constexpr uint32_t A_SLICE = kTileM * 64, B_SLICE = N * 64;
    constexpr int kWide = 256 / N;  // slices of B in one MMA
    static_assert(S >= kMinSlices && S <= kSlices, "slice count");
#pragma unroll
    for (int i = 1; i <= S; ++i)
#pragma unroll
        for (int ks = 0; ks < kKBlock / 16; ++ks) {
            // every MMA of one A tile in a row: it is read from shared memory once
            const uint64_t ad = ad0 + (((i - 1) * A_SLICE + ks * 32) >> 4);
            const int n = S + 1 - i;
            const int run = n < kNumAcc + 1 - i ? n : kNumAcc + 1 - i;  // products with an accumulator each
            const int parts = (run + kWide - 1) / kWide, total = parts + n - run;
            int done = 0;
            auto mma = [&](int j, auto width) {
                constexpr int w = decltype(width)::value;
                const uint64_t bd = bd0 + (((j - 1) * B_SLICE + ks * 32) >> 4);
                const uint32_t d = tmem + acc_of(i, j) * N, idesc = tc::idesc_bf16_f32(kTileM, w * N);
                const uint32_t accum = (kFirst && i == 1 && ks == 0 && j <= kNumAcc) ? 0u : 1u;
                if (total == 1) tc::umma_bf16<tc::CollectA::kDiscard>(d, ad, bd, idesc, accum);
                else if (done == 0) tc::umma_bf16<tc::CollectA::kFill>(d, ad, bd, idesc, accum);
                else if (done < total - 1) tc::umma_bf16<tc::CollectA::kUse>(d, ad, bd, idesc, accum);
                else tc::umma_bf16<tc::CollectA::kLastUse>(d, ad, bd, idesc, accum);
                ++done;
            };
            // the run in parts of equal width (the first ones one wider where it does not divide)
#pragma unroll
            for (int p = 0, j = 1; p < parts; ++p) {
                const int w = run / parts + (p < run % parts ? 1 : 0);
                if (w == 1) mma(j, std::integral_constant<int, 1>{});
                if constexpr (kWide >= 2) if (w == 2) mma(j, std::integral_constant<int, 2>{});
                if constexpr (kWide >= 3) if (w == 3) mma(j, std::integral_constant<int, 3>{});
                if constexpr (kWide >= 4) if (w == 4) mma(j, std::integral_constant<int, 4>{});
                if constexpr (kWide >= 5) if (w == 5) mma(j, std::integral_constant<int, 5>{});
                j += w;
            }
#pragma unroll
            for (int j = run + 1; j <= n; ++j) mma(j, std::integral_constant<int, 1>{});
        }
}

}  // namespace vfmm
