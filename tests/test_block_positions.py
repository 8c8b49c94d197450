"""The position of a block of the symmetric backprojection, formed in 2^-31 bins from the tile's
base and 32-bit C and S as the kernel does, lies within 2^-32 bins of the exact one of the
fixed-point geometry (15 units of 2^-31 on the axis, where C = 2^32), over the whole range of C and
S (2^31 <= C <= 2^32, S <= C) and every block of a tile, and stays in the staged window."""
import pytest


def position(base, C, S, it, jt):
    """bin and fraction in 2^-31 bins, with the kernel's 64- and 32-bit words."""
    P = (base >> 1) + (it >> 1) * min(C, 2 ** 32 - 1) + (jt >> 1) * S
    assert 0 <= P < 2 ** 64 and S < 2 ** 32
    return P >> 31, P & 0x7FFFFFFF


@pytest.mark.parametrize("C,S", [(2 ** 32, 0), (2 ** 32 - 1, 1), (2 ** 31, 2 ** 31), (2 ** 31 + 1, 12345), (3037000500, 3037000499),
                                 (4294967293, 123456789), (3221225473, 2863311529)])
@pytest.mark.parametrize("base", [2 * 2 ** 32, 2 * 2 ** 32 + 1, 3 * 2 ** 32 + 4294967295, 2 * 2 ** 32 + 2147483649])
def test_positions(C, S, base):
    for it in range(0, 32, 2):
        for jt in range(0, 32, 4):
            want = base + it * C + jt * S                 # in 2^-32 bins
            b, f = position(base, C, S, it, jt)
            assert b >= 2
            err = want - 2 * (b * 2 ** 31 + f)
            assert 0 <= err <= (1 if C < 2 ** 32 else 31)
