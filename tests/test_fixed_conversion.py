"""The conversion of doubles to fixed point (csrc/fixed.cuh: from_double and from_double_any), restated on the bits, over
the shifts that its callers form (CPU): the moments' 57 + 1022 - eb for a batch's largest field eb in 200 .. 1800, the
rows' 60 + e for any step of the table, the descriptors' 57 or 60 places."""
import struct

import numpy as np
import pytest


def _hi(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0] >> 32


def from_double(x, sh):
    b = struct.unpack("<Q", struct.pack("<d", x))[0]
    moved = ((((b >> 32) + (sh << 20)) & 0xffffffff) << 32) | (b & 0xffffffff)
    d = struct.unpack("<d", struct.pack("<Q", moved))[0]
    if np.isnan(d) or abs(d) >= 2.0 ** 63:  # the conversion saturates (a NaN: its lowest value)
        return -(1 << 63) if np.isnan(d) or d < 0 else (1 << 63) - 1
    return int(np.rint(d)) if abs(d) < 2.0 ** 52 else int(d)


def from_double_any(x, sh):
    return from_double(x, sh) if ((_hi(x) >> 20) & 0x7ff) + sh > 0 else 0


SMALL = [0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1022, -2.0 ** -1022, -1e-300]


@pytest.mark.parametrize("eb", [200, 900, 1078, 1079, 1080, 1200, 1500, 1800])
def test_small_values_beside_the_largest(eb):
    sh = 57 + 1022 - eb  # the moments' (negative from 2^57 up)
    top = 2.0 ** (eb - 1023)
    conv = from_double if sh >= 0 else from_double_any
    for x in SMALL + [top, -top, np.nextafter(2 * top, 0), top * 2.0 ** -57, -top * 2.0 ** -58, 1.0, -1.0]:
        if abs(x) >= 2 * top:
            continue
        want = int(np.rint(np.longdouble(x) * np.longdouble(2) ** sh))
        assert conv(x, sh) == want, (x, sh)


@pytest.mark.parametrize("e", [-200, -62, -61, -60, 0, 7, 300])
def test_offsets_of_any_step(e):
    for x in [0.0, -0.0, 2.0 ** -e * 0.9, -(2.0 ** -e) * 1e-9]:
        assert from_double_any(x, 60 + e) == int(np.rint(np.longdouble(x) * np.longdouble(2) ** (60 + e)))


def test_why_the_shift_must_not_be_negative():
    assert from_double(-0.0, -1) == (1 << 63) - 1 and from_double(0.0, -1) == -(1 << 63)
