// Which attention kernel is the faster one for a problem: rules on sizes only (host code without CUDA, so that
// tests/test_dispatch_rules.py can hold them against a table of measured times).
//   blocks  128-row query blocks of all heads and batch elements
//   pairs   CTAs of the two-block kernel: blocks are paired inside a unit (the query heads of a KV head; single query heads
//           under a custom head map), so an odd number of blocks per unit leaves one half of a pair empty
// Times: B200, both sides forced; graphs of repeated calls (no host time), from N = 4096 up sustained runs.
#pragma once

namespace hifa4 {

// The 64-key kernel with four groups of softmax warps and one block per SM against two groups and two blocks per SM (d = 64
// and 128).  Where every block has an SM to itself, four groups win once a row has work for them all (130 blocks, d = 64: N =
// 128 5.8 against 5.4 us, N = 256 7.0 against 6.7, N = 512 8.9 against 9.4, N = 2048 21 against 25; d = 128: N = 64 5.5 against
// 5.2, N = 128 6.5 against 6.7).  With more blocks than SMs the last ones run alone, and under a causal mask those are the short
// ones: how many pay grows with the rows (d = 128: 152 blocks of N = 128 12.0 against 9.4 us, 192 of N = 384 14.2 against 12.3, 160
// of N = 640 0.92 of the time and 190 1.04, 192 of N = 768 0.98 and 210 1.05, 224 of N = 1024 0.99 and 256 1.02, 256 of N = 2048
// 0.96, d = 64 0.88).  Not causal: never (256 blocks of N = 2048 1.16, d = 64 1.03).
inline bool four_groups_faster(int d, int N, bool causal, long long blocks, int sms)
{
    if (blocks <= sms) return N >= (d == 64 ? 320 : 128);
    const int slack = N - 512 < 768 ? N - 512 : 768;
    return causal && slack > 0 && 1024 * (blocks - sms) <= (long long)sms * slack;
}

// The two-block kernel (d = 128) against the 64-key kernel, or against the 128-key kernel where Bc = 128.
// Blocks of equal length come in waves.  A pair per SM takes as long as two blocks on an SM, and the persistent CTAs pay set-up
// and fill once instead of once per wave: in units of a 64-key tile, 3 + waves * tiles against waves * (tiles + 1.5), a last
// wave of at most one block per SM counting 0.67.  Over 520 non-causal sizes (N = 64 to 2048, 160 to 1200 blocks) that picks
// the faster side or one within 7 % of it, 0.2 % off on the average (N = 64, 8 / 8 heads, 224 blocks: 9.3 against 6.5 us; N =
// 384, 12 / 4, 288 blocks 21.5 against 15.1, 900 blocks 42.6 against 44.6; N = 1152, 8 / 8, 288 blocks 38 against 30; N = 4096, 32
// heads, 323 against 310; N = 8192, 32 heads 1149 against 1165).  The 128-key kernel runs one block per SM, a wave of pairs
// takes 1.9 of its waves, 1.7 with Q-Mean: 3 + 1.9 * waves * tiles against waves * (tiles + 2) (N = 1152, 8 / 8, 288 blocks: 48
// against 36; N = 1280, 960 blocks 126 against 125, with Q-Mean 143 against 153).
// Causal blocks differ, the heaviest start first and fill one another's gaps: there the two-block kernel wins from 1.5 pairs per
// SM up (N = 1024, 8 / 8 heads: 320 blocks 26.6 against 22.2, 512 blocks 32.8 against 33.4, 768 blocks 45.9 against 48.8; N =
// 4096, 32 heads 166 against 168), 1.6 against the 128-key kernel (N = 1024, 8 / 8: 448 blocks 33.5 against 36.8).  Rows too
// short to differ much (N up to 256; 128) go by waves as above; N = 320, whose last block is half empty, from 2.5 pairs per SM
// (14 / 2 heads, 588 blocks 24.7 against 20.5, 756 blocks 0.96 of the time).
inline bool two_blocks_faster(int Bc, int N, bool causal, bool qmean, long long blocks, long long pairs, int sms)
{
    const long long waves = (pairs + sms - 1) / sms;
    if (Bc == 128) {
        if (causal && N > 128) return 5 * ((blocks + 1) / 2) >= 8LL * sms;
        const int tiles = (N + 127) / 128 * 2;
        return 3.0 + (qmean ? 1.7 : 1.9) * (double)waves * tiles <= (double)((blocks + sms - 1) / sms) * (tiles + 2);
    }
    if (causal && N > 320) return 2 * ((blocks + 1) / 2) >= 3LL * sms;
    if (causal && N > 256) return 2 * pairs >= 5LL * sms;
    const int tiles = (N + 63) / 64;
    const long long full = blocks / (2 * sms), rest = blocks % (2 * sms);
    const double waves64 = (double)full + (rest == 0 ? 0.0 : rest <= sms ? 0.67 : 1.0);
    return 3.0 + (double)waves * tiles <= waves64 * (tiles + 1.5);
}

}  // namespace hifa4
