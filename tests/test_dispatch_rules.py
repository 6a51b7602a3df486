"""The rules that choose between attention kernels (hifa4_dispatch.h, host code without CUDA) against measured times of both
sides (B200, us; graphs of repeated calls, from N = 4096 up sustained runs): the kernel chosen is never slower than the other
by more than 8 %.  Rows lie on both sides of every line and where an earlier form of the rules chose the slower kernel by 10
to 45 %."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 148

# d, N, causal, blocks, two groups of softmax warps, four groups
GROUPS = [
    (64, 64, True, 192, 5.87, 8.48), (64, 64, False, 130, 4.00, 4.52), (64, 128, True, 192, 7.85, 10.62), (64, 256, True, 96, 6.64, 6.90),
    (64, 320, True, 192, 8.53, 11.82), (64, 384, True, 153, 9.22, 10.52), (64, 512, True, 192, 10.24, 12.18), (64, 512, False, 96, 9.26, 8.83),
    (64, 1024, False, 96, 14.54, 12.97), (64, 1024, False, 160, 22.45, 24.62), (64, 2048, False, 256, 40.08, 41.34),
    (128, 64, False, 1, 4.55, 4.80), (128, 64, True, 192, 6.73, 9.75), (128, 128, False, 1, 6.24, 6.04), (128, 128, True, 152, 9.39, 11.98),
    (128, 192, True, 192, 9.52, 12.66), (128, 256, True, 192, 10.69, 13.02), (128, 320, True, 192, 10.56, 14.06), (128, 384, True, 192, 12.28, 14.18),
    (128, 512, False, 96, 11.17, 10.93), (128, 1024, False, 96, 17.12, 16.62),
]


# Bc, N, causal, blocks, pairs launched, 64-key (Bc = 128: 128-key) kernel, two-block kernel
PAIRS = [
    (64, 64, False, 160, 160, 6.13, 8.93), (64, 64, False, 224, 224, 6.49, 9.27), (64, 64, False, 294, 168, 6.60, 10.10),
    (64, 64, True, 448, 448, 11.47, 14.89), (64, 64, True, 1200, 1200, 25.21, 30.06), (64, 64, False, 1200, 600, 23.25, 21.19),
    (64, 128, False, 156, 104, 9.06, 9.73), (64, 128, False, 294, 168, 9.43, 13.34), (64, 128, False, 1200, 600, 37.61, 31.08),
    (64, 128, True, 520, 520, 17.43, 20.39), (64, 320, False, 288, 160, 13.66, 19.46), (64, 320, True, 588, 308, 20.45, 24.74),
    (64, 320, True, 528, 352, 20.19, 22.98), (64, 320, True, 1200, 600, 41.99, 38.32), (64, 384, False, 288, 192, 15.04, 21.61),
    (64, 384, False, 900, 500, 44.60, 42.57), (64, 384, False, 588, 308, 27.10, 32.05), (64, 384, True, 1200, 800, 53.69, 47.12),
    (64, 640, False, 520, 312, 36.93, 41.15), (64, 1024, True, 320, 160, 22.15, 26.58), (64, 1024, True, 576, 288, 35.15, 33.24),
    (64, 1152, False, 288, 160, 29.77, 38.40), (64, 1152, False, 576, 320, 56.07, 64.35), (64, 1152, False, 864, 480, 83.32, 95.13),
    (64, 4096, False, 1024, 512, 310.0, 322.9), (64, 8192, False, 1024, 512, 585.9, 615.7), (64, 8192, False, 2048, 1024, 1165.3, 1149.3),
    (64, 4096, True, 1024, 512, 168.0, 165.7),
    (128, 64, False, 448, 448, 18.46, 20.73), (128, 64, True, 1200, 1200, 36.83, 43.12), (128, 64, False, 608, 304, 22.01, 20.67),
    (128, 128, False, 294, 168, 12.89, 14.41), (128, 128, False, 602, 344, 25.19, 20.67), (128, 128, True, 448, 224, 21.83, 17.08),
    (128, 320, False, 288, 192, 19.42, 25.27), (128, 320, False, 588, 308, 33.07, 37.19), (128, 320, False, 600, 400, 41.08, 37.40),
    (128, 1024, True, 320, 160, 29.10, 32.02), (128, 1024, False, 320, 160, 47.74, 56.95), (128, 1024, True, 576, 288, 43.87, 39.96),
    (128, 1152, False, 288, 160, 36.27, 47.64), (128, 1152, False, 576, 320, 70.01, 80.49), (128, 2048, False, 256, 128, 56.10, 58.50),
    (128, 768, False, 396, 198, 39.20, 47.68), (128, 1280, False, 1500, 750, 198.12, 178.88), (128, 2048, False, 736, 368, 132.83, 146.38),
]
PAIRS_QMEAN = [
    (64, 768, False, 300, 150, 35.62, 43.11), (64, 768, False, 456, 228, 45.43, 44.25), (64, 2048, False, 896, 448, 165.25, 188.78),
    (128, 768, False, 396, 198, 46.68, 54.34), (128, 768, False, 1044, 522, 114.71, 97.23), (128, 1280, False, 960, 480, 153.08, 143.45),
    (128, 2048, False, 384, 192, 101.38, 114.06), (128, 2048, False, 608, 304, 166.23, 163.58),
]


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    (d / "shim.cpp").write_text(
        '#include "%s"\n' % os.path.join(ROOT, "paper_2607_04302_b200", "csrc", "hifa4_dispatch.h") +
        'extern "C" int four_groups(int d, int N, int causal, long long blocks, int sms)\n'
        '{ return hifa4::four_groups_faster(d, N, causal != 0, blocks, sms); }\n'
        'extern "C" int two_blocks(int Bc, int N, int causal, int qmean, long long blocks, long long pairs, int sms)\n'
        '{ return hifa4::two_blocks_faster(Bc, N, causal != 0, qmean != 0, blocks, pairs, sms); }\n')
    so = str(d / "shim.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", str(d / "shim.cpp"), "-o", so])
    lib, ll = ctypes.CDLL(so), ctypes.c_longlong
    lib.four_groups.argtypes = [ctypes.c_int] * 3 + [ll, ctypes.c_int]
    lib.two_blocks.argtypes = [ctypes.c_int] * 4 + [ll, ll, ctypes.c_int]
    return lib


def test_four_groups_rule(rules):
    for d, N, causal, blocks, two, four in GROUPS:
        chosen = four if rules.four_groups(d, N, int(causal), blocks, SMS) else two
        assert chosen <= 1.08 * min(two, four), (d, N, causal, blocks)


def test_two_block_rule(rules):
    for qmean, rows in ((0, PAIRS), (1, PAIRS_QMEAN)):
        for Bc, N, causal, blocks, pairs, one, two in rows:
            chosen = two if rules.two_blocks(Bc, N, int(causal), qmean, blocks, pairs, SMS) else one
            assert chosen <= 1.08 * min(one, two), (Bc, N, causal, qmean, blocks, pairs)


def test_the_cases_of_the_gpu_tests_reach_the_kernels_they_name(rules):
    """Sizes of the tests that compare kernels with one another, on a B200's 148 SMs."""
    from tests import test_gpu_attention_groups as groups
    from tests import test_gpu_attention_pair as pair

    def takes_pairs(Bc, B, Hq, Hkv, N, causal, qmean, head_map):
        G = 1 if head_map else Hq // Hkv
        unit, units = (N + 127) // 128 * G, Hq // G * B
        return rules.two_blocks(Bc, N, int(causal), int(qmean), unit * units, (unit + 1) // 2 * units, SMS)

    def params(test, first):
        return next(m.args[1] for m in test.pytestmark if m.name == "parametrize" and m.args[0].startswith(first))

    for name, (B, Hq, Hkv, N, causal, qmean, head_map) in pair.CASES.items():
        assert takes_pairs(64, B, Hq, Hkv, N, causal, qmean, head_map), name
    for B, Hq, Hkv, N, causal, qmean, head_map in params(pair.test_two_block_kernel_with_128_key_tiles, "B,"):
        assert takes_pairs(128, B, Hq, Hkv, N, causal, qmean, head_map), (B, Hq, N)
    seen = set()
    for B, Hq, Hkv, N, causal, _, _ in params(groups.test_four_groups_are_bit_identical_to_two, "B,"):
        for d in (64, 128):
            if rules.four_groups(d, N, int(causal), (N + 127) // 128 * Hq * B, SMS):
                seen.add((d, (N + 63) // 64 % 4))
    assert seen == {(d, r) for d in (64, 128) for r in range(4)}            # every remainder of tiles by groups


def test_bench_names_the_kernel_that_runs(rules):
    import bench
    from paper_2607_04302_b200 import synth
    for Bc in (64, 128):
        for N in (64, 128, 256, 320, 384, 1024, 1152, 4096):
            for B, Hq, Hkv in ((1, 1, 1), (1, 32, 8), (4, 28, 4), (8, 8, 8), (20, 8, 8)):
                for causal in (True, False):
                    for qmean in (False, True):
                        cfg = synth.config("C2", B=B, Hq=Hq, Hkv=Hkv, N=N, causal=causal, Bc=Bc)
                        unit, units = (N + 127) // 128 * (Hq // Hkv), Hkv * B
                        want = rules.two_blocks(Bc, N, int(causal), int(qmean), unit * units, (unit + 1) // 2 * units, SMS)
                        assert bench.two_blocks_chosen(cfg, SMS, qmean) == bool(want), (Bc, N, B, Hq, Hkv, causal, qmean)
    assert bench.attention_kernel(synth.config("C2")) == "attention_fwd_pair_kernel<0, 0>"
    assert bench.attention_kernel(synth.config("C4")) == "attention_fwd_cta2_kernel<0>"
    assert bench.attention_kernel(synth.config("C1")) == "attention_fwd_ws64_kernel<128>"
