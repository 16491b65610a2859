"""INT8 weight carriers where the precision of 127 q decides them: shapes for which the fp32 product 127 q is exactly half way
between two integers although the product in more bits is not.  The format rounds twice (to fp32, then to an integer); a
kernel that forms product and rounding in one step is off by one there, some 2e-7 of all table entries.  The shapes
come from a random search over binary16 pairs (a, b) whose level curve rises by more than 0.01 everywhere."""
import numpy as np
import pytest

import datagen
import oracle

# width: (magnitude, a, b) with a and b as binary16 bit patterns
TIES = {
    3: [(2, 0x3417, 0xa02a), (2, 0x33d8, 0x24a3), (1, 0x3c70, 0x1d8b), (2, 0x33c9, 0x25cf), (2, 0x3436, 0xa6ed), (2, 0x3412, 0x9d34)],
    4: [(3, 0x3d6d, 0xab5b), (3, 0x3d58, 0x2194), (4, 0x376c, 0x1f99), (5, 0x3398, 0xb655), (5, 0x32ee, 0xb589), (5, 0x3334, 0xb5dd)],
    5: [(3, 0x3cab, 0x1f12), (6, 0x3c29, 0x91be), (8, 0x3335, 0x37e5), (9, 0x37ee, 0x36e9), (9, 0x3ab5, 0xb7b7), (9, 0x3c2b, 0x230f)],
    6: [(5, 0x3d13, 0xafe5), (7, 0x3b9e, 0xb196), (7, 0x3ab0, 0x374d), (7, 0x3bdd, 0xb577), (7, 0x3c07, 0xb78b), (7, 0x3916, 0xaabe)],
    7: [(9, 0x3cbf, 0x24db), (9, 0x3cc4, 0xa525), (10, 0x3cf4, 0x33d5), (14, 0x3d39, 0x240e), (16, 0x3c2d, 0xa2b3), (17, 0x38f1, 0x2b2c)],
    8: [(14, 0x3d49, 0x2947), (18, 0x3bbb, 0x37ff), (18, 0x3c57, 0xb74c), (18, 0x3c69, 0xb8c8), (20, 0x3be5, 0xbac3), (20, 0x3ba9, 0xb90a)],
}


def half(bits):
    return np.uint16(bits).view(np.float16)


@pytest.mark.parametrize("B", sorted(TIES))
def test_the_shapes_tell_one_rounding_from_two(B):
    for i, a, b in TIES[B]:
        assert oracle.shape_margin(float(half(a)), float(half(b))) > 0.0
        af, bf, t = np.float32(half(a)), np.float32(half(b)), np.float32(i) / np.float32((1 << (B - 1)) - 1)
        c = (np.float32(1) - af) - bf
        fma = lambda x, y: np.float32(np.float64(t) * np.float64(x) + np.float64(y))
        q = t * fma(fma(c, bf), af)
        assert float(np.float32(127) * q) % 1.0 == 0.5 and (127.0 * float(q)) % 1.0 != 0.5
        twice, once = np.rint(np.float32(127) * q), np.rint(127.0 * float(q))
        assert int(oracle.carriers(B, a, b)[i]) == twice != once


@pytest.mark.gpu
@pytest.mark.parametrize("M", [8, 16, 64, 256])   # the INT8 mma.sync kernel and the tcgen05 one
@pytest.mark.parametrize("G", [32, 128])
@pytest.mark.parametrize("B", sorted(TIES))
def test_carriers_of_the_products(B, G, M):
    from test_gpu_exact import a8_exact   # every bit of the result
    from util import Case
    N, K = 24, 256   # a row is one magnitude of one shape, of either sign
    mag, a, b = (np.array([TIES[B][n % 6][j] for n in range(N)]) for j in range(3))
    k = np.where((np.arange(K) + np.arange(N)[:, None]) % 2, mag[:, None], -mag[:, None]).astype(np.int8)
    shape = lambda v: np.repeat(v.astype(np.uint16).view(np.float16)[:, None], K // G, axis=1)
    case = Case(k, np.full((N, K // G), 127.0, np.float32), shape(a), shape(b), B, G)
    x = np.zeros((M, K), np.float32)
    x[np.arange(M), np.arange(M) * 37 % K] = 127.0
    a8_exact(case, datagen.to_bf16_bits(x))
