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
    (64, 64, True, 192, 5.51, 8.19), (64, 64, False, 130, 3.87, 4.25), (64, 128, True, 192, 7.37, 10.00),
    (64, 256, True, 96, 6.13, 6.46), (64, 320, True, 192, 7.92, 11.18), (64, 384, True, 153, 8.53, 9.93),
    (64, 512, True, 192, 9.49, 11.53), (64, 512, False, 96, 8.40, 8.19), (64, 1024, False, 96, 13.24, 12.14),
    (64, 1024, False, 160, 19.81, 22.20), (64, 2048, False, 256, 35.53, 37.94), (128, 64, False, 1, 4.40, 4.71),
    (128, 64, True, 192, 6.34, 9.38), (128, 128, False, 1, 5.94, 5.94), (128, 128, True, 152, 9.06, 11.59),
    (128, 192, True, 192, 8.94, 12.16), (128, 256, True, 192, 10.05, 12.51), (128, 320, True, 192, 9.86, 13.41),
    (128, 384, True, 192, 11.70, 13.64), (128, 512, False, 96, 10.34, 10.25), (128, 1024, False, 96, 15.92, 15.76),
]


# Bc, N, causal, blocks, pairs launched, 64-key (Bc = 128: 128-key) kernel, two-block kernel
PAIRS = [
    (64, 64, False, 160, 160, 5.86, 8.23), (64, 64, False, 224, 224, 6.05, 8.45), (64, 64, False, 294, 168, 6.29, 9.32),
    (64, 64, True, 448, 448, 10.87, 13.50), (64, 64, True, 1200, 1200, 24.01, 26.20),
    (64, 64, False, 1200, 600, 22.08, 18.85), (64, 128, False, 156, 104, 8.58, 8.86),
    (64, 128, False, 294, 168, 8.98, 12.21), (64, 128, False, 1200, 600, 37.11, 29.52),
    (64, 128, True, 520, 520, 16.99, 18.62), (64, 320, False, 288, 160, 13.06, 17.30),
    (64, 320, True, 588, 308, 19.75, 22.34), (64, 320, True, 528, 352, 19.62, 19.36),
    (64, 320, True, 1200, 600, 40.34, 34.18), (64, 384, False, 288, 192, 13.79, 18.50),
    (64, 384, False, 900, 500, 42.93, 37.83), (64, 384, False, 588, 308, 26.03, 28.37),
    (64, 384, True, 1200, 800, 52.38, 42.67), (64, 640, False, 520, 312, 33.29, 33.15),
    (64, 1024, True, 320, 160, 20.87, 23.16), (64, 1024, True, 576, 288, 33.23, 29.72),
    (64, 1152, False, 288, 160, 26.50, 29.93), (64, 1152, False, 576, 320, 52.32, 54.53),
    (64, 1152, False, 864, 480, 83.17, 87.40), (64, 4096, False, 1024, 512, 281.4, 296.9),
    (64, 8192, False, 1024, 512, 525.4, 570.5), (64, 8192, False, 2048, 1024, 1063.9, 1016.4),
    (64, 4096, True, 1024, 512, 167.5, 157.2), (128, 64, False, 448, 448, 18.14, 19.40),
    (128, 64, True, 1200, 1200, 35.50, 39.50), (128, 64, False, 608, 304, 21.22, 19.56),
    (128, 128, False, 294, 168, 12.41, 13.98), (128, 128, False, 602, 344, 24.28, 19.91),
    (128, 128, True, 448, 224, 21.02, 16.54), (128, 320, False, 288, 192, 18.32, 23.45),
    (128, 320, False, 588, 308, 31.75, 35.02), (128, 320, False, 600, 400, 38.69, 34.58),
    (128, 1024, True, 320, 160, 28.15, 30.02), (128, 1024, False, 320, 160, 44.26, 48.44),
    (128, 1024, True, 576, 288, 42.54, 37.02), (128, 1152, False, 288, 160, 33.98, 41.53),
    (128, 1152, False, 576, 320, 65.40, 69.86), (128, 2048, False, 256, 128, 51.95, 54.08),
    (128, 768, False, 396, 198, 37.00, 43.57), (128, 1280, False, 1500, 750, 207.7, 168.9),
    (128, 2048, False, 736, 368, 128.3, 128.2),
    # sizes that an earlier form of the rule, fitted to earlier kernels, sent to the slower side
    (64, 320, False, 2304, 1536, 83.79, 73.79), (64, 1024, False, 224, 112, 28.29, 24.68),
    (64, 2304, False, 288, 144, 53.22, 46.70), (64, 1152, False, 1512, 768, 153.5, 137.3),
    (64, 384, True, 384, 192, 18.98, 16.97), (64, 512, True, 384, 192, 19.54, 16.38),
    (64, 768, True, 420, 210, 25.24, 21.33), (64, 1152, True, 432, 224, 30.79, 26.58),
    (64, 1664, True, 416, 224, 40.39, 35.43), (128, 320, False, 2304, 1536, 124.6, 105.8),
    (128, 384, False, 768, 512, 50.16, 43.77), (128, 896, False, 672, 384, 71.48, 62.15),
    (128, 1152, False, 1440, 800, 162.7, 144.7), (128, 192, True, 256, 128, 14.64, 12.37),
    (128, 256, True, 320, 160, 18.50, 16.21), (128, 384, True, 360, 192, 22.02, 18.25),
    (128, 512, True, 448, 224, 26.99, 22.83), (128, 896, True, 448, 224, 32.41, 28.88),
]
PAIRS_QMEAN = [
    (64, 768, False, 300, 150, 31.46, 36.61), (64, 768, False, 456, 228, 40.19, 38.34),
    (64, 2048, False, 896, 448, 149.7, 161.8), (128, 768, False, 396, 198, 47.04, 47.78),
    (128, 768, False, 1044, 522, 124.2, 84.50), (128, 1280, False, 960, 480, 163.4, 124.2),
    (128, 2048, False, 384, 192, 96.13, 94.92), (128, 2048, False, 608, 304, 158.9, 138.7),
    (64, 384, True, 360, 192, 20.66, 17.20), (64, 512, True, 384, 192, 21.67, 18.87),
    (64, 1152, True, 432, 216, 33.99, 30.24), (128, 320, False, 1152, 768, 78.44, 66.43),
    (128, 256, True, 208, 104, 16.42, 12.53), (128, 320, True, 330, 176, 21.69, 17.69),
    (128, 384, True, 384, 192, 25.06, 21.20), (128, 768, True, 360, 180, 31.96, 28.15),
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
    from tests.test_gpu_attention import RAW_CASES
    for B, Hq, Hkv, N in RAW_CASES:
        assert not takes_pairs(64, B, Hq, Hkv, N, False, False, None), (B, Hq, N)
    assert [B * Hq * N >= 131072 for B, Hq, _, N in RAW_CASES] == [True, False]
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
