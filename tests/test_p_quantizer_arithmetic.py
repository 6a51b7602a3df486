"""The packed FP16 arithmetic of the in-register quantizer of P (hifa4_attention.cuh), restated in numpy: on every
finite non-negative FP16 value of P (above 1 too: the running maximum may have been rounded down) under every E6M2 scale a
group maximum can select and every shift, the element code is the round-to-nearest-even of the exact quotient, the shift
thresholds are exact and the BF16 FMA returns code * step."""
import numpy as np
import pytest

P = np.arange(0, 0x7C00, dtype=np.uint16).view(np.float16).astype(np.float64)
HI = (0x3C00, 0x3A66, 0x3955, 0x3892)              # RN16(4 / (4 + M))


def f16(bits):
    return float(np.array(bits, dtype=np.uint16).view(np.float16))


def rn16(x):
    return x.astype(np.float16).astype(np.float64)


def bits16(x):
    return x.astype(np.float16).view(np.uint16).astype(int)


def e6m2_code(a):                                  # smallest E6M2 value with 7 S >= a
    codes = np.arange(256)
    s = 2.0 ** (codes // 4 - 48.0) * (1 + codes % 4 / 4)
    return int(np.searchsorted(7 * s, a, side="left"))


GROUPS = sorted({(e6m2_code(a), 0 if a >= 2.0 ** -12 else 12) for a in P[1:]})


@pytest.mark.parametrize("M", range(4))
def test_packed_fp16_quantizer_is_exact(M):
    seen = 0
    for code, s in GROUPS:
        if code & 3 != M:
            continue
        e = code >> 2
        S = 2.0 ** (e - 48) * (1 + M / 4)
        p = P[P <= min(65504.0 if s == 0 else 2.0 ** -12 * (1 - 2.0 ** -11), 7 * S)]
        hi_bits = HI[M] + ((49 - e - s) << 10)
        hi = f16(hi_bits)
        lo = float(rn16(np.float64(hi * 2.0 ** -12))) if M else 0.0
        assert np.isfinite(hi) and hi_bits >> 10 > 0
        q = rn16(p * hi + rn16(p * lo))            # exact in double before the one rounding of the FMA
        need = np.maximum(bits16(q) + 1023 - (0x4300 - (s << 10)), 0) >> 10
        assert (need == (p > 1.75 * S).astype(int) + (p > 3.5 * S)).all()
        for k in range(3):
            step, ok = S * 2 ** k / 4, p <= 1.75 * S * 2 ** k
            pp = p[ok]
            magic_bits = (0x6200 - (s << 10)) | (k << 10)
            y = bits16(rn16(q[ok] + f16(magic_bits)))
            j = np.floor(pp / step)                # exact floor of the quotient, then ties to even
            j = np.where(j * step > pp, j - 1, np.where((j + 1) * step <= pp, j + 1, j))
            r = 2 * pp - (2 * j + 1) * step
            want = np.where(r > 0, j + 1, np.where(r < 0, j, j + j % 2))
            assert (y - magic_bits == want).all()
            kk = k << 10
            c_bits = (((e + (111 if s else 15)) << 7) | (M << 5)) + (kk >> 3) - kk
            n_bits = (0x8000 | ((e + 84) << 7) | (M << 5)) + (kk >> 3)
            c = 2.0 ** ((c_bits >> 7) - 127) * (1 + (c_bits & 127) / 128)
            n = 2.0 ** (((n_bits & 0x7FFF) >> 7) - 127) * (1 + (n_bits & 127) / 128)
            assert 0 < c_bits >> 7 < 255 and n_bits >> 15 == 1
            y_bf16 = 2.0 ** ((y >> 7) - 127) * (1 + (y & 127) / 128)
            assert (y_bf16 * c - n == want * step).all()
            seen += len(pp)
    assert seen > 100000
