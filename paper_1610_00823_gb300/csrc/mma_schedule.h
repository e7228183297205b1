// Which slice products the MMAs of one K block of a split contraction do, in issue order. Plain C++: the
// kernels unroll it and the host checks it.
//
// Slice i of A meets slices j = 1 .. S + 1 - i of B, product (i, j) going to accumulator acc_of(i, j), its
// diagonal. Slices of B are consecutive rows in shared memory and diagonals consecutive columns in TMEM, so
// one MMA does up to 256 / N products whose accumulators are distinct: a run of them from j = 1, cut
// into parts of nearly equal width (the first ones one wider where it does not divide). Products on
// diagonals that share the last accumulator beyond its first take an MMA each.
#pragma once

namespace vfmm {

constexpr int kSlices = 8;     // BF16 slice slots per operand (balanced base-128 digits, 56 bits)
constexpr int kMinSlices = 6;  // fewest slices a contraction may take (every accumulator gets a product)
constexpr int kNumAcc = 6;     // TMEM accumulators (diagonals 0..4 exact, 5+ shared)

// Accumulator of slice product (i, j): its diagonal i + j - 2; diagonals >= kNumAcc - 1 share the last.
constexpr int acc_of(int i, int j) { return i + j - 2 < kNumAcc - 1 ? i + j - 2 : kNumAcc - 1; }

// Products of slice i of A with an accumulator each: none where i alone is past the last diagonal (i > kNumAcc).
constexpr int mma_run(int S, int i) {
    const int n = S + 1 - i, own = kNumAcc + 1 - i;
    return n < own ? n : (own > 0 ? own : 0);
}
constexpr int mma_parts(int S, int N, int i) { return (mma_run(S, i) + 256 / N - 1) / (256 / N); }
// MMAs of slice i of A (per 16 K values).
constexpr int mma_count(int S, int N, int i) { return mma_parts(S, N, i) + S + 1 - i - mma_run(S, i); }

struct MmaStep {
    int j, w;  // products (i, j) .. (i, j + w - 1) in one MMA of width w * N
};
constexpr MmaStep mma_step(int S, int N, int i, int q) {
    const int run = mma_run(S, i), parts = mma_parts(S, N, i);
    if (q >= parts) return MmaStep{run + 1 + q - parts, 1};
    const int rem = run % parts;
    return MmaStep{1 + q * (run / parts) + (q < rem ? q : rem), run / parts + (q < rem ? 1 : 0)};
}

// Every product i + j <= S + 1 once and no other, wide MMAs within 256 columns and on distinct
// accumulators, and the first slice of A writing every accumulator (its MMAs overwrite on a first K block).
constexpr bool mma_schedule_ok(int S, int N) {
    for (int i = 1; i <= S; ++i) {
        int next = 1;
        for (int q = 0; q < mma_count(S, N, i); ++q) {
            const MmaStep m = mma_step(S, N, i, q);
            if (m.j != next || m.w < 1 || m.w * N > 256) return false;
            if (acc_of(i, m.j + m.w - 1) != acc_of(i, m.j) + m.w - 1) return false;
            next += m.w;
        }
        if (next != S + 2 - i) return false;
    }
    return S >= kNumAcc;
}
static_assert(mma_schedule_ok(6, 48) && mma_schedule_ok(6, 64) && mma_schedule_ok(6, 80), "schedule, S = 6");
static_assert(mma_schedule_ok(7, 48) && mma_schedule_ok(7, 64) && mma_schedule_ok(7, 80), "schedule, S = 7");
static_assert(mma_schedule_ok(8, 48) && mma_schedule_ok(8, 64) && mma_schedule_ok(8, 80), "schedule, S = 8");

}  // namespace vfmm
