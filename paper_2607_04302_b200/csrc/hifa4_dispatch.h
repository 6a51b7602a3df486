// Which attention kernel is the faster one for a problem: rules on sizes only (host code without CUDA, so that
// tests/test_dispatch_rules.py can hold them against a table of measured times).
//   blocks  128-row query blocks of all heads and batch elements
//   pairs   CTAs of the two-block kernel: blocks are paired inside a unit (the query heads of a KV head; single query heads
//           under a custom head map), so an odd number of blocks per unit leaves one half of a pair empty
// Times: B200, both sides forced and run in turn; graphs of repeated calls (no host time), from N = 4096 up sustained runs.
#pragma once

namespace hifa4 {

// The 64-key kernel with four groups of softmax warps and one block per SM against two groups and two blocks per SM (d = 64
// and 128).  Where every block has an SM to itself, four groups win once a row has work for them all (d = 64: 96 blocks, N = 256
// 6.5 against 6.1 us, N = 512 8.2 against 8.4, N = 1024 12.1 against 13.2; d = 128: one block, N = 64 4.7 against 4.4, N = 128 5.9
// against 5.9; 96 blocks, N = 1024 15.8 against 15.9).  With more blocks than SMs the last ones run alone, and under a causal mask
// those are the short ones: how many pay grows with the rows (d = 128: 152 blocks of N = 128 11.6 against 9.1 us, 192 of N = 384 13.6
// against 11.7; of their time with an earlier quantizer of P: 160 of N = 640 0.92 and 190 1.04, 192 of N = 768 0.98 and 210 1.05,
// 224 of N = 1024 0.99 and 256 1.02, 256 of N = 2048 0.96, d = 64 0.88).  Not causal: never (d = 64: 160 blocks of N = 1024 22.2
// against 19.8 us, 256 of N = 2048 37.9 against 35.5).
inline bool four_groups_faster(int d, int N, bool causal, long long blocks, int sms)
{
    if (blocks <= sms) return N >= (d == 64 ? 320 : 128);
    const int slack = N - 512 < 768 ? N - 512 : 768;
    return causal && slack > 0 && 1024 * (blocks - sms) <= (long long)sms * slack;
}

// The two-block kernel (d = 128) against the 64-key kernel, or against the 128-key kernel where Bc = 128.  The lines were fitted to
// 2196 sizes (N = 64 to 8192, 100 to 2400 blocks, causal and not, with and without Q-Mean) and held against 1142 others: over all of
// them the side chosen is 0.2 % off the faster one on the average and at most 10 % off, but for N = 64, 576 blocks in 384 pairs (12.6
// against 10.9 us).
// Blocks of equal length, and short causal rows, come in waves: fixed parts (set-up, fill, epilogue) plus waves * tiles, in units of
// a 64-key tile.  A pair per SM takes a little less than two blocks on an SM (0.915 of it, with Q-Mean 1.02) and pays set-up and
// fill once instead of once per wave; a last wave of at most one block per SM counts 0.44 in the 64-key kernel, which then runs those
// blocks with an SM each (N = 2304, 288 blocks: 46.7 against 53.2 us; N = 1024, 224 blocks 24.7 against 28.3; N = 4096, 1024 blocks, 3.44
// waves against 4, 297 against 281; N = 8192, 2048 blocks 1016 against 1064; N = 64, 224 blocks 8.5 against 6.1).  The 128-key kernel runs
// one block per SM; a wave of pairs takes 1.72 of its waves, with Q-Mean 1.63 (N = 896, 672 blocks: 62 against 71; N = 1152, 288 blocks
// 41.5 against 34.0; with Q-Mean N = 1280, 960 blocks 124 against 163).
// Longer causal rows differ, the heaviest start first and fill one another's gaps: there a number of pairs per SM decides, which
// grows with the rows because a lone last pair takes the longer (two-block against 64-key kernel: N = 512, 384 blocks 16.4
// against 19.5; N = 1152, 432 blocks 26.6 against 30.8; N = 1024, 320 blocks 23.2 against 20.9; N = 4096, 512 blocks 0.85 of the
// time, 384 blocks 1.17; against the 128-key kernel: N = 256, 320 blocks 16.2 against 18.5; N = 512, 448 blocks 22.8 against 27.0;
// N = 1024, 320 blocks 30.0 against 28.2; N = 4096, 448 blocks with Q-Mean 0.95).
inline bool two_blocks_faster(int Bc, int N, bool causal, bool qmean, long long blocks, long long pairs, int sms)
{
    const double waves = (double)((pairs + sms - 1) / sms), pairs_per_sm = (double)((blocks + 1) / 2) / sms;
    if (Bc == 128) {
        if (causal && N > 128) {
            const double line = 0.6 + (N - 256) / 1000.0, cap = qmean ? 1.37 : 1.5;
            return pairs_per_sm >= (line < cap ? line : cap);
        }
        const int tiles = (N + 127) / 128 * 2;
        return 2.9 + (qmean ? 1.63 : 1.72) * waves * tiles <= (double)((blocks + sms - 1) / sms) * (tiles + (qmean ? 2.0 : 1.5));
    }
    if (causal && N > 320) {
        const double line = 1.05 + (N - 512) / 4200.0;
        return pairs_per_sm >= (line < 1.42 ? line : 1.42);
    }
    const int tiles = (N + 63) / 64;
    const long long full = blocks / (2 * sms), rest = blocks % (2 * sms);
    const double low = causal ? 0.74 : 0.44, waves64 = (double)full + (rest == 0 ? 0.0 : rest <= sms ? low : 1.0);
    if (causal) return 2.2 + 0.74 * waves * tiles <= waves64 * (tiles + 0.75);
    return 3.1 + (qmean ? 1.02 : 0.915) * waves * (tiles + 1.3) <= waves64 * (tiles + 4.0);
}

}  // namespace hifa4
