"""The symmetric projectors' index maps and block arithmetic, emulated on the CPU with the
kernels' integers: every window of staged bins lies inside its padded row and every access
inside its window, and the per-block sums give the linear interpolation of each pixel."""
import numpy as np
import pytest


def jobs_of(n, M, thetas, ratio=1.0):
    """Canonical jobs (A, B, Op) of the fixed-point geometry, F = 32."""
    out = []
    for th in thetas:
        c, s = abs(np.cos(th)) * ratio, abs(np.sin(th)) * ratio
        A, B = int(round(max(c, s) * 2 ** 32)), int(round(min(c, s) * 2 ** 32))
        out.append((A, B, ((M - 1) * 2 ** 32 - (n - 1) * (A + B)) >> 1))
    return sorted(out, key=lambda j: j[1] / j[0])


GEOMETRIES = [(1, 1, 1.0), (7, 3, 1.0), (33, 47, 1.0), (64, 95, 1.0), (100, 60, 0.41), (129, 500, 0.8)]
THETAS = np.concatenate([[0.0, 1e-9, np.pi / 4, np.arctan(1 / 3), np.arctan(0.5), np.arctan(2 / 3)],
                         np.linspace(0.01, 0.785, 9)])


@pytest.mark.parametrize("n,M,ratio", GEOMETRIES)
@pytest.mark.parametrize("nc", [4, 2])
def test_backprojection_windows_and_blocks(n, M, ratio, nc):
    jobs = jobs_of(n, M, THETAS, ratio)
    al = 4 // nc
    win = (max((30 * A + 28 * B) >> 32 for A, B, _ in jobs) + 7 + 2 * (al - 1)) // al * al
    far = (n + 31) // 32 * 32 - 32
    lo, hi = 0, M
    for A, B, Op in jobs:
        P = Op + ((A + 3 * B) >> 1)
        lo = min(lo, (P >> 32) - 2)
        hi = max(hi, ((P + far * (A + B)) >> 32) - 2 + win)
    pad = (-lo + 4 + 3) & ~3
    pitch = (pad + hi + 3) & ~3
    rng = np.random.default_rng(3)
    it, jt = np.meshgrid(np.arange(0, 32, 2), np.arange(0, 32, 4), indexing="ij")
    for A, B, Op in jobs:
        g = rng.standard_normal(M)
        bar = np.zeros(pitch)
        bar[pad:pad + M] = g
        c, s = A / 2 ** 32, B / 2 ** 32
        e = [0.5 * c + 1.5 * s, 0.5 * c + 0.5 * s, 0.5 * c - 0.5 * s, 0.5 * c - 1.5 * s]
        flat = 3 * B <= A
        for i0 in range(0, n, 32):
            for j0 in range(0, n, 32):
                P = i0 * A + j0 * B + Op + ((A + 3 * B) >> 1)
                first = ((P >> 32) - 2 + pad) & ~(al - 1)
                assert 0 <= first and first + win <= pitch
                base = (P - ((first - pad) << 32)) >> 1
                q = base + it.astype(object) * (A >> 1) + jt.astype(object) * (B >> 1)
                b = (q >> 31).astype(int)
                f = (q & 0x7FFFFFFF).astype(float) / 2 ** 31
                assert b.min() - 2 >= 0 and b.max() + 3 < win
                v = {k: bar[first + b + k] for k in range(-2, 4)}
                d = {k: v[k + 1] - v[k] for k in range(-2, 3)}
                dr, dl, dr2, dl2 = d[1] - d[0], d[0] - d[-1], d[2] - d[1], d[-1] - d[-2]
                pos = lambda x: np.maximum(x, 0.0)  # noqa: E731
                for k in range(4):
                    kr, kl = pos(f + e[k] - 1) * dr, pos(e[k] - f) * dl
                    if not flat and k == 0:
                        kr, kl = kr + pos(f + e[0] - 2) * dr2, kl + pos(e[0] - f - 1) * dl2
                    if not flat and k == 3:
                        kr, kl = pos(-e[3] - f) * dl, pos(f - e[3] - 1) * dr
                    for sign, row, col, knot in ((1, 1, 3 - k, kr), (-1, 0, k, kl)):
                        got = v[0] + f * d[0] + sign * e[k] * d[0] + knot
                        i, j = i0 + it + row, j0 + jt + col
                        p = (i * c + j * s + Op / 2 ** 32)
                        kk = np.floor(p).astype(int)
                        w = p - kk
                        ext = np.zeros(M + 2)
                        ext[1:-1] = g
                        at = lambda x: np.where((x >= 0) & (x < M), ext[np.clip(x, -1, M) + 1], 0.0)  # noqa: E731
                        inside = (i < n) & (j < n)
                        want = (1 - w) * at(kk) + w * at(kk + 1)
                        assert np.abs((got - want)[inside]).max(initial=0.0) < 1e-6
