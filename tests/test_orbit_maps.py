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
def test_backprojection_windows_and_blocks(n, M, ratio):
    jobs = jobs_of(n, M, THETAS, ratio)
    al = 2
    win = (max((30 * A + 28 * B) >> 32 for A, B, _ in jobs) + 9) & ~1
    assert win <= 52
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


def rows_out(Q0, binv, qlo, qhi, n):
    f32 = np.float32
    if binv != 0:
        m1, m2 = f32((Q0 - f32(qhi)) * binv), f32((Q0 - f32(qlo)) * binv)
        a0, a1 = max(0.0, np.floor(min(m1, m2))), min(n - 1.0, np.ceil(max(m1, m2)))
        return (int(a0), int(a1)) if a0 <= a1 else (n, -1)
    return (0, n - 1) if qlo < Q0 < qhi else (n, -1)


@pytest.mark.parametrize("n,M,ratio", GEOMETRIES + [(40, 300000, 1.0)])
@pytest.mark.parametrize("segs", [1, 4])
def test_forward_rows_pads_and_slot_sums(n, M, ratio, segs):
    lanes, pad, one = 64, 72, 2 ** 32
    f32 = np.float32
    u = np.random.default_rng(5).standard_normal((n, n))            # ubar[m][q], one channel
    qq, mm = np.meshgrid(np.arange(n), np.arange(n))
    for A, B, Op in jobs_of(n, M, THETAS, ratio):
        want = np.zeros(M + 2)
        p = (qq * A + mm * B + Op) / one
        k = np.floor(p).astype(int)
        for kk, w in ((k, 1 - (p - k)), (k + 1, p - k)):
            np.add.at(want, np.where((kk >= 0) & (kk < M), kk + 1, 0), w * u)
        nb = ((lanes * A) >> 32) - 1
        assert nb >= 1
        centre = np.array([-((-q * A) >> 32) for q in range(lanes)])
        phi = np.array([q * A / one for q in range(lanes)]) - centre
        chunks = range((M + nb - 1) // nb)
        for bx in (chunks if M < 1000 else [0, len(chunks) // 2 - 1, len(chunks) // 2, len(chunks) - 1]):
            kb, S, X, P = bx * nb, np.zeros(lanes), np.zeros(lanes), np.zeros(lanes)
            K0 = (kb - 1) * one
            Q0 = f32(K0 - Op) * f32(f32(one / A) * f32(2.0 ** -32))
            lo, hi = rows_out(Q0, f32(A / B) if B / A > 1e-9 else f32(0), -lanes - 1, n + 1, n)
            per = (hi - lo + segs) // segs
            for seg in range(segs):
                mlo = lo + seg * per
                mhi = min(hi, mlo + per - 1)
                if mlo > mhi:
                    continue
                q = int(np.ceil(Q0 - f32(mlo) * (f32(B) / f32(A))))
                x = q * A + mlo * B + Op - K0
                while x < 0:
                    x, q = x + A, q + 1
                while x >= A:
                    x, q = x - A, q - 1
                bound = min(A - B, one - 1)
                r = min(x, one - 2) if B == 0 else x
                for m in range(mlo, mhi + 1):
                    assert -pad <= q and q + lanes - 1 < n + pad
                    assert 0 <= r < A and abs(q * A + m * B + Op - K0 - r) <= (B == 0)
                    at = np.arange(q, q + lanes)
                    v = np.where((at >= 0) & (at < n), u[m, np.clip(at, 0, n - 1)], 0.0)
                    z = r / one + phi
                    assert np.abs(z).max() <= 1
                    S, X, P = S + v, X + r / one * v, P + np.clip(z, 0, 1) * v
                    step = r >= bound
                    r = (r + (B - A if step else B)) % one
                    q -= step
            N = P - X - phi * S
            got = [P[centre == b].sum() + (S - P - N)[centre == b + 1].sum() + N[centre == b + 2].sum()
                   for b in range(min(nb, M - kb))]
            ref = want[1:-1][kb:min(kb + nb, M)]
            assert np.abs(np.array(got) - ref).max(initial=0.0) < 1e-4 * max(1.0, np.abs(want[1:-1]).max())
