// Which attention kernel is the faster one for a problem: rules on sizes only (host code without CUDA, so that
// tests/test_dispatch_rules.py can hold them against a table of measured times).
//   blocks  128-row query blocks of all heads and batch elements
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

}  // namespace hifa4
