// Plain arithmetic that kernels and launchers share and that a test can compile and check on its own: no CUDA in here.
#pragma once

#ifdef __CUDACC__
#define FC_RULE __host__ __device__ constexpr
#else
#define FC_RULE constexpr
#endif

namespace fc {

// How often slot `slot` of a ring of `slots` buffers has been asked for when `requested` boxes were requested in order.
// The barrier of a slot completes one phase per request, so the last one is phase ring_uses - 1.
FC_RULE int ring_uses(long long requested, int slot, int slots) {
    return requested > slot ? (int)((requested - slot + slots - 1) / slots) : 0;
}

// ---- tensor-core contraction: CTAs per SM and shared memory of one ----------
constexpr int TC_BM = 128, TC_BN = 128, TC_BK = 32, TC_STAGES = 3;
constexpr unsigned TC_TILE_BYTES = TC_BM * TC_BK * 4;               // one 128 x 32 fp32 box: 16 KB
constexpr unsigned TC_STAGE_BYTES = 4 * TC_TILE_BYTES;              // A_re, A_im, B_re, B_im
constexpr unsigned TC_EPI_BUF_BYTES = 32 * 128;                     // 32 rows x 32 fp32, one TMA store box
constexpr unsigned TC_EPI_BYTES = 4 * 2 * TC_EPI_BUF_BYTES;         // 4 warps x 2 buffers
// Narrow matrices leave room for more stages than three, but more than four do not pay (S64 f64 f'128,
// n = 64: 62 us with three, 59 with four, 65 with six).
constexpr int TC_MAX_STAGES = 4;
constexpr unsigned TC_FIXED_BYTES = 1024 + 512;                     // alignment of the ring; barriers
constexpr unsigned SM_SHARED_BYTES = 228 * 1024, CTA_RESERVED_BYTES = 1024;     // of an SM; per CTA, by the system

struct TcShare {
    int per_sm, stages;
    unsigned ring_bytes, epi_bytes, smem;
    unsigned acc_cols;          // TMEM columns from one accumulator to the next
};
// The tiles of narrow matrices (N <= 64) are short chains of a load, a few MMAs and a store, which one CTA's ring and two
// accumulators do not hide.  Where the accumulators leave tensor memory for more CTAs (N <= 64: two, N <= 32: four) as
// many run as find two stages of the ring in shared memory (three, where N > 32 and the sum is longer than a stage: M, N, K = 64,
// 64, 64 over the bins of n = 64 38.6 us with four stages in one CTA, 41.5 with two in each of two), and as there are tiles for.  M, N, K = 55, 12, 15 over the
// bins of n = 64 18.7 -> 12.8 us, 18, 6, 33 21.0 -> 12.9, 19, 34, 4 22.8 -> 16.0, n = 128: 9, 18, 20 55.6 -> 27, 40, 20, 60
// 88 -> 58-67, 96, 3, 128 158 -> 132-140; 300, 20, 20 (n = 64) unchanged.
// * Tiles for one CTA per SM or fewer: as many stages as one CTA can have, because a long sum lives on the loads in flight
//   (M, N, K = 45, 10, 2001, n = 16: 47.6 us with four stages, 62.0 with the three of a shared SM).
// * No more CTAs fit than find tensor memory, and with several per SM no more than planned: the shared memory is padded.
//   One more would wait until another has done all its tiles, while SMs that the previous kernel still holds get none
//   (a dependent's CTAs are placed early): fprop of S4 f1 f'39 60 x 23, n = 64, 38.2 us without the padding, 27.7 with it,
//   36.2 with one CTA per SM.
// rows_a, rows_b: rows of a stage's boxes.
FC_RULE TcShare tc_share(int rows_a, int rows_b, int N, int k_blocks, long long tiles, int sms) {
    const unsigned stage = 256u * (unsigned)(rows_a + rows_b);
    const int most = N > 64 ? 1 : (N > 32 ? 2 : 4);             // by tensor memory
    TcShare s{1, 0, TC_STAGES * TC_STAGE_BYTES, TC_EPI_BYTES, 0, (unsigned)TC_BN};
    if (most > 1) {
        // the staging tiles of the warps that have rows; at least 16 KB, because an MMA reads 128 rows of A whatever rows_a
        // is, and what lies behind the last stage's has to be shared memory of this CTA
        const unsigned warps = (unsigned)((rows_a + 31) / 32);
        s.epi_bytes = (warps < 2 ? 2 : warps) * 2 * TC_EPI_BUF_BYTES;
        s.acc_cols = 128 / (unsigned)most;
        const unsigned fixed = TC_FIXED_BYTES + s.epi_bytes, needed = N > 32 && k_blocks > 1 ? 3 : 2;
        for (int c = most; c >= 1; --c) {
            const unsigned room = (SM_SHARED_BYTES - 1024) / (unsigned)c / 1024 * 1024 - (c > 1 ? CTA_RESERVED_BYTES : 0);
            if (c > 1 && (tiles <= (long long)(c - 1) * sms || room < fixed + needed * stage)) continue;
            s.per_sm = c;
            s.ring_bytes = (room - fixed) / 1024 * 1024;
            break;
        }
    }
    const int fit = (int)(s.ring_bytes / stage);
    s.stages = fit < TC_MAX_STAGES ? fit : TC_MAX_STAGES;
    if (most > 1) s.ring_bytes = (unsigned)s.stages * stage;
    s.smem = TC_FIXED_BYTES + s.ring_bytes + s.epi_bytes;
    const int fits = s.per_sm > 1 ? s.per_sm : most;            // CTAs that may share an SM
    const unsigned least = SM_SHARED_BYTES / (unsigned)(fits + 1) / 1024 * 1024 + 1024 - CTA_RESERVED_BYTES;
    if (most > 1 && s.smem < least) s.smem = least;
    return s;
}

}  // namespace fc
