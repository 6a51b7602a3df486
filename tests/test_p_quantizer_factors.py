"""The packed FP16 arithmetic of the in-register quantizer of P with two FP16 factors (hifa4_attention.cuh), restated in numpy
down to the packed integer constants: on every finite non-negative FP16 value of P under every E6M2 scale a group maximum can
select and every shift, the scale and the subgroup shifts are those of exact arithmetic, the element code is the
round-to-nearest-even of the exact quotient and the BF16 FMA returns code * step."""
import numpy as np
import pytest

P16 = np.arange(0, 0x7C00, dtype=np.uint16).view(np.float16)
P = P16.astype(np.float64)
F1 = (0x3C00, 0x3C92, 0x3F38, 0x3E30)
F2 = (0x4000, 0x3D9A, 0x39E9, 0x39E9)
TADD = (0x24FF, 0x22FF, 0x1F42, 0x1F42)


def f16(bits):
    return float(np.array(bits, dtype=np.uint16).view(np.float16))


def rn16(x):
    return x.astype(np.float16).astype(np.float64)


def bits16(x):
    return x.astype(np.float16).view(np.uint16).astype(np.int64)


def e6m2_code(a):                                  # smallest E6M2 value with 7 S >= a
    codes = np.arange(256)
    s = 2.0 ** (codes // 4 - 48.0) * (1 + codes % 4 / 4)
    return np.searchsorted(7 * s, a, side="left")


def scale_bits(a16):                               # upper bits of S as a float, FP32 arithmetic of the kernel
    seventh = np.array(0x3E124924, dtype=np.uint32).view(np.float32)
    return ((a16.astype(np.float32) * seventh).view(np.uint32).astype(np.int64) + 0x1FFFFF) >> 21


def dup(h):
    return h * 0x10001


def halves(w):
    return w & 0xFFFF, (w >> 16) & 0xFFFF


def bf16(bits):
    return 2.0 ** (((bits & 0x7FFF) >> 7) - 127) * (1 + (bits & 127) / 128)


def test_scale_of_every_group_maximum():
    assert (scale_bits(P16[1:]) - 4 * 79 == e6m2_code(P[1:])).all()


GROUPS = sorted({(int(t), 0 if a >= 2.0 ** -12 else 1) for t, a in zip(scale_bits(P16[1:]), P[1:])})


@pytest.mark.parametrize("M", range(4))
def test_two_factor_quantizer_is_exact(M):
    seen = 0
    for t, small in GROUPS:
        if t & 3 != M:
            continue
        S = 2.0 ** ((t >> 2) - 127) * (1 + M / 4)
        top = 0x30003000 if small else 0
        f1 = (dup(F1[M]) + (127 - (t >> 2)) * 0x04000400 - top) & 0xFFFFFFFF
        f2, tadd = dup(F2[M]) + top, dup(TADD[M]) + top
        n0 = (t * 0x00200020 + 0x76807680) & 0xFFFFFFFF
        for w in (f1, f2, tadd, n0):
            assert w & 0xFFFF == w >> 16
        c1, c2 = f16(f1 & 0xFFFF), f16(f2 & 0xFFFF)
        assert 2.0 ** -14 <= c1 < 65536 and np.isfinite(c2)
        p = P[P <= min(65504.0 if not small else 2.0 ** -12 * (1 - 2.0 ** -11), 7 * S)]
        q = rn16(p * c1)
        assert np.isfinite(q).all()

        def magic_of(b):                           # largest q of the subgroup (or half of the other's) -> magic constant
            return np.maximum(b + (tadd & 0xFFFF), 0x6000) & 0xFC00

        need = (p > 1.75 * S).astype(int) + (p > 3.5 * S)
        assert bits16(q).max() + (tadd & 0xFFFF) < 0x8000
        assert (magic_of(bits16(q)) == 0x6000 + (need << 10)).all()
        assert (magic_of(bits16(q) - 1024) == 0x6000 + (np.maximum(need - 1, 0) << 10)).all()
        for k0 in range(3):
            for k1 in range(3):                    # packed integer constants: no carry between the halves
                magic = (0x6000 + (k0 << 10)) | ((0x6000 + (k1 << 10)) << 16)
                n = (n0 + (magic >> 3)) & 0xFFFFFFFF
                c = (n - magic - 0x40804080) & 0xFFFFFFFF
                for k, nk, ck in zip((k0, k1), halves(n), halves(c)):
                    assert nk >> 15 == 1 and bf16(nk) == S * 2 ** k / 4 * 128
                    assert 0 < ck >> 7 < 255 and bf16(ck) == S * 2 ** k / 4 * 128 * 2.0 ** -(65 + 8 * k)
        for k in range(3):
            step, ok = S * 2 ** k / 4, p <= 1.75 * S * 2 ** k
            pp, magic = p[ok], 0x6000 + (k << 10)
            y = bits16(rn16(q[ok] * c2 + f16(magic)))      # exact in double before the one rounding of the FMA
            j = np.floor(pp / step)                # exact floor of the quotient, then ties to even
            j = np.where(j * step > pp, j - 1, np.where((j + 1) * step <= pp, j + 1, j))
            r = 2 * pp - (2 * j + 1) * step
            want = np.where(r > 0, j + 1, np.where(r < 0, j, j + j % 2))
            assert (y - magic == want).all()
            c, n = bf16(halves(n0 + (dup(magic) >> 3))[0] - magic - 0x4080), S * 2 ** k / 4 * 128
            assert (bf16(y) * c - n == want * step).all()
            seen += len(pp)
    assert seen > 100000
