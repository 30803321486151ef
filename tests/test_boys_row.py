"""Integer logic of the FP64 Boys table's row index (boys_row in eri_common.cuh), emulated on the CPU: the row
and its grid point come from the high word of T; |T - T_k| stays within the Taylor expansion's range and the
row is the one that holds T_k's coefficients (k/512 below 64, 4,096 rows per binade above)."""
import struct

import numpy as np

SUB, ROWS_A = 12, 64 * 512 + 1
HI_B = 0x40500000


def boys_row(T):
    bits = struct.unpack("<q", struct.pack("<d", T))[0]
    h = bits >> 32
    regb = h >= HI_B
    s = 20 - SUB if regb else min(11 + 1023 - (h >> 20), 20)
    half = 1 << (s - 1)
    hr = (h + half) & ~((1 << s) - 1)
    k = ((h & 0xfffff) + 0x100000 + half) >> s
    if h < 0x3F600000:
        k = int(h >= 0x3F500000)
        hr = 0x3F600000 if k else 0
    if regb:
        k = (hr >> (20 - SUB)) - (HI_B >> (20 - SUB)) + ROWS_A
    return k, struct.unpack("<d", struct.pack("<q", hr << 32))[0]


def test_row_and_grid_point():
    rng = np.random.default_rng(0)
    Ts = list(rng.uniform(0, 64, 3000)) + list(10.0 ** rng.uniform(-320, 0, 500)) + list(10.0 ** rng.uniform(1.8, 9.3, 3000))
    Ts += [0.0, 5e-324, 2.0 ** -10, np.nextafter(2.0 ** -10, 0), 2.0 ** -9, np.nextafter(2.0 ** -9, 0), 63.999999999, 64.0,
           np.nextafter(64.0, 0), 127.99999999, 2.0 ** 31 - 1e-3] + [k / 512 + x for k in range(1, 50) for x in (1 / 1024, -1 / 1024)]
    for T in Ts:
        k, Tk = boys_row(float(T))
        if T < 64.0:
            assert 0 <= k < ROWS_A and Tk == k / 512.0 and abs(T - Tk) <= (1 + 1e-5) / 1024
        else:
            r = k - ROWS_A
            e, i = 6 + (r >> SUB), r & ((1 << SUB) - 1)
            assert 6 <= e <= 31 and Tk == 2.0 ** e * (1 + i / 4096) and abs(T - Tk) <= (1 + 1e-5) * T / 8192
