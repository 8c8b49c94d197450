// The discrete Radon transform R_h and its adjoint R_h^* (linear backprojection)
// of Sec. 3.1, as an exact transpose pair of gather kernels for sm_103a.
//
//  * R_h^* (pixel-driven): a CTA owns a 32 x 32 tile of pixels and one group of
//    angles; per chunk of 32 angles it stages, for every angle, the tile's
//    detector footprint into shared memory as interpolation-ready pairs, then each
//    thread walks its 8 pixels' exact fixed-point detector coordinate P and spends
//    one shared-memory load and one FMA per (pixel, angle).  With several angle
//    groups the groups' partial images are summed by a small epilogue kernel
//    (enough CTAs to fill 152 SMs at n = 512).  No atomics.
//  * R_h (ray-driven): one lane per detector interval [k, k+1) of one angle
//    marches across the image rows, tracking exactly (integer arithmetic) the
//    first pixel whose coordinate falls in its interval; it accumulates
//    sum u and sum frac*u over the pixels of its interval, and the two neighbouring
//    intervals' sums are combined with one warp shuffle:
//        g_k = sum_{floor p = k} (1 - frac) u  +  sum_{floor p = k-1} frac u.
//    A CTA takes 4 adjacent angles (one warp each) over 31 bins; the rows on which
//    every lane of a warp stays inside the image run without bounds checks.
//    No atomics; each output bin is written once.
// Both kernels derive each weight from the same integer P (see ctr_internal.cuh),
// so they are transposes of one matrix.  Plans whose angles are symmetric images of
// one another take the kernels of orbit.cuh (FP64: orbit64.cuh) instead, which start from the same
// integers; in FP32 they round their weights apart, so that the pair is adjoint up to FP32 rounding.
#include <algorithm>
#include <type_traits>

#include "ctr_internal.cuh"

namespace ctr {

namespace {

// CTA barrier of a stage body.  NAMED: the body runs on the first 128 threads of a larger
// CTA (the persistent batched iteration) and synchronises them with named barrier 1.
template <bool NAMED>
__device__ __forceinline__ void body_sync()
{
    if constexpr (NAMED) asm volatile("bar.sync 1, 128;" ::: "memory");
    else __syncthreads();
}

#ifndef CTR_BP_TY
#define CTR_BP_TY 4
#endif
#ifndef CTR_BP_R
#define CTR_BP_R 8
#endif
#ifndef CTR_BP_ACH
#define CTR_BP_ACH 32
#endif
constexpr int BP_TJ = 32;          // tile width along j (one warp)
constexpr int BP_TY = CTR_BP_TY;   // warps per CTA
constexpr int BP_R = CTR_BP_R;     // pixels per thread (rows i0 + ty + BP_TY r)
constexpr int BP_TI = BP_TY * BP_R;
constexpr int BP_ACH = CTR_BP_ACH; // angles per staged chunk

template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

// operand loads: FP32/FP64 as stored, bfloat16 widened to FP32
__device__ __forceinline__ float ldv(const float *p) { return *p; }
__device__ __forceinline__ double ldv(const double *p) { return *p; }
__device__ __forceinline__ float ldv(const __nv_bfloat16 *p) { return __bfloat162float(*p); }

// floor(p) = P >> F; the FP32 path has F = 32, so it is the high word.
template <typename T>
__device__ __forceinline__ int bin_of(long long P, int F)
{
    if constexpr (sizeof(T) == 4) return (int)(P >> 32);
    else return (int)(P >> F);
}

#ifndef CTR_FWD_UNROLL
#define CTR_FWD_UNROLL 8
#endif
constexpr int FWD_UNROLL = CTR_FWD_UNROLL;   // rows per unrolled step of the ray march

// x / d for x, d >= 0 with x d < 2^32 as the high word of x m, m = floor((2^32 - 1) / d) + 1
// (then m - 2^32 / d < 1 and the error x (m - 2^32/d) / 2^32 stays below 1/d, so the floor is
// exact).  The staging loops divide element indices by a row width once per copied element;
// a runtime integer division costs an instruction sequence, this one multiply.
__device__ __forceinline__ unsigned udiv_magic(unsigned d) { return d <= 1 ? 0u : 0xFFFFFFFFu / d + 1u; }
__device__ __forceinline__ int udiv_fast(int x, int d, unsigned m) { return d <= 1 ? x : (int)__umulhi((unsigned)x, m); }

// 1 + frac(p) in [1, 2) from the low 32 bits of P (F = 32): the top 23 fraction
// bits become the mantissa of a float, so the weight is exact and identical in
// both projectors.
__device__ __forceinline__ float one_plus_frac32(long long P)
{
    return __uint_as_float((((unsigned)(unsigned long long)P) >> 9) | 0x3F800000u);
}

__device__ __forceinline__ float one_plus_frac32u(unsigned lo)
{
    return __uint_as_float((lo >> 9) | 0x3F800000u);
}

__device__ __forceinline__ float2 make_stage(float g0, float g1)
{
    const float d = g1 - g0;
    return make_float2(g0 - d, d);     // value = (g0 - d) + (1 + frac) d
}
__device__ __forceinline__ double2 make_stage(double g0, double g1)
{
    return make_double2(g0, g1 - g0);  // value = g0 + frac d
}

__device__ __forceinline__ float interp(float acc, float2 pr, long long P, int, double)
{
    return fmaf(one_plus_frac32(P), pr.y, acc + pr.x);
}
__device__ __forceinline__ double interp(double acc, double2 pr, long long P, int F, double inv2F)
{
    const unsigned long long mask = (1ull << F) - 1ull;
    const double a = (double)((unsigned long long)P & mask) * inv2F;
    return acc + fma(a, pr.y, pr.x);
}

template <typename T>
__device__ __forceinline__ void bp_epilogue(const BackprojEpi<T> &epi, int n, int i, int j, T acc)
{
    const size_t o = (size_t)i * n + j;
    const T old = epi.bar_out ? epi.ub[o] : T(0);      // read before out (may alias ub) is written
    const T v = bp_epilogue_value(epi, n, i, j, acc);
    if (epi.bar_out) epi.bar_out[o] = T(2) * v - old;
    if (epi.complex_out) {
        epi.out[2 * o] = v;
        epi.out[2 * o + 1] = T(0);
    } else {
        epi.out[o] = v;
    }
}

// One CTA of the backprojection: tile (bx, by), angle group bz.
// part == nullptr: apply the epilogue directly (one angle group).  Otherwise write
// this group's partial sums to part[bz][n][n].
template <typename T, typename S, bool NAMED = false>
__device__ __forceinline__ void bp_body(const S *g, int n, int N, int M, int F, int wstride,
                                        int angles_per_group, const AngleGeom *__restrict__ geom,
                                        const BackprojEpi<T> &epi, T *part, int bx, int by, int bz)
{
    using T2 = typename Pair<T>::type;
    constexpr int NT = 32 * BP_TY;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T2 *stage = reinterpret_cast<T2 *>(smem_raw);
    long long *sPb = reinterpret_cast<long long *>(stage + BP_ACH * wstride);
    long long *sC = sPb + BP_ACH;
    long long *sS = sC + BP_ACH;
    int *sK = reinterpret_cast<int *>(sS + BP_ACH);

    const int tx = threadIdx.x & 31;
    const int ty = threadIdx.x >> 5;
    const int i0 = by * BP_TI;
    const int j0 = bx * BP_TJ;
    const int la = bz * angles_per_group;
    const int lb = min(N, la + angles_per_group);
    const double inv2F = ldexp(1.0, -F);

    T acc[BP_R];
#pragma unroll
    for (int r = 0; r < BP_R; ++r) acc[r] = T(0);

    for (int l0 = la; l0 < lb; l0 += BP_ACH) {
        const int na = min(BP_ACH, lb - l0);
        body_sync<NAMED>();
        if (threadIdx.x < na) {
            const AngleGeom ag = geom[l0 + threadIdx.x];
            const long long P00 = (long long)i0 * ag.C + (long long)j0 * ag.S + ag.O;
            const long long P10 = P00 + (long long)(BP_TI - 1) * ag.C;
            const long long P01 = P00 + (long long)(BP_TJ - 1) * ag.S;
            const long long P11 = P10 + (long long)(BP_TJ - 1) * ag.S;
            const long long pmin = min(min(P00, P10), min(P01, P11));
            const long long kmin = pmin >> F;   // arithmetic shift: floor
            sK[threadIdx.x] = (int)kmin;
            sPb[threadIdx.x] = P00 - (kmin << F);
            sC[threadIdx.x] = ag.C;
            sS[threadIdx.x] = ag.S;
        }
        body_sync<NAMED>();
        const unsigned mw = udiv_magic((unsigned)wstride);
        for (int e = threadIdx.x; e < na * wstride; e += NT) {
            const int a = udiv_fast(e, wstride, mw);
            const int k = sK[a] + (e - a * wstride);
            const S *row = g + (size_t)(l0 + a) * M;
            const T g0 = (k >= 0 && k < M) ? (T)ldv(row + k) : T(0);
            const T g1 = (k + 1 >= 0 && k + 1 < M) ? (T)ldv(row + k + 1) : T(0);
            stage[e] = make_stage(g0, g1);
        }
        body_sync<NAMED>();
#pragma unroll 2
        for (int a = 0; a < na; ++a) {
            const long long C = sC[a];
            long long P = sPb[a] + (long long)ty * C + (long long)tx * sS[a];
            const long long D = C * BP_TY;
            const T2 *row = stage + a * wstride;
#pragma unroll
            for (int r = 0; r < BP_R; ++r) {
                acc[r] = interp(acc[r], row[bin_of<T>(P, F)], P, F, inv2F);
                P += D;
            }
        }
    }

    const int j = j0 + tx;
#pragma unroll
    for (int r = 0; r < BP_R; ++r) {
        const int i = i0 + ty + BP_TY * r;
        if (i < n && j < n) {
            if (part) part[((size_t)bz * n + i) * n + j] = acc[r];
            else bp_epilogue(epi, n, i, j, acc[r]);
        }
    }
}

template <typename T, typename S>
__global__ void __launch_bounds__(32 * BP_TY)
k_backproject(const S *__restrict__ g, int n, int N, int M, int F, int wstride, int angles_per_group,
              const AngleGeom *__restrict__ geom, BackprojEpi<T> epi, T *__restrict__ part)
{
    bp_body<T, S>(g, n, N, M, F, wstride, angles_per_group, geom, epi, part, blockIdx.x, blockIdx.y, blockIdx.z);
}

// Sum of the angle groups' partial images, then the backprojection epilogue
// (block b of nb, grid-stride over the n*n pixels).
template <typename T>
__device__ __forceinline__ void bp_reduce_body(const T *__restrict__ part, int groups, int n,
                                               const BackprojEpi<T> &epi, int b, int nb)
{
    const size_t nn = (size_t)n * n;
    for (size_t e = b * (size_t)blockDim.x + threadIdx.x; e < nn; e += (size_t)nb * blockDim.x) {
        T s = part[e];
        for (int z = 1; z < groups; ++z) s += part[(size_t)z * nn + e];
        bp_epilogue(epi, n, pix_i(e, n), pix_j(e, n), s);
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_bp_reduce(const T *__restrict__ part, int groups, int n, BackprojEpi<T> epi)
{
    bp_reduce_body<T>(part, groups, n, epi, blockIdx.x, gridDim.x);
}

__device__ __forceinline__ long long ceil_div_ll(long long a, long long b)
{
    // b > 0
    long long q = a / b;
    if (q * b < a) ++q;
    return q;
}

__device__ __forceinline__ void acc_sample(float &Su, float &Sf, float v, long long P, int, double)
{
    Su += v;
    Sf = fmaf(one_plus_frac32(P), v, Sf);     // sum (1 + frac) u
}
__device__ __forceinline__ void acc_sample(double &Su, double &Sf, double v, long long P, int F, double inv2F)
{
    const unsigned long long mask = (1ull << F) - 1ull;
    Su += v;
    Sf = fma((double)((unsigned long long)P & mask) * inv2F, v, Sf);   // sum frac u
}

// The data resolvent (id + s dg_r^*)^{-1}(z) = z - s clip(q, lo, hi), q = (z + w a)/(s + w),
// written as w (z - s a)/(s + w) + s (q - clip(q)): for w = 0 and q inside the box it is
// exactly 0 (the one-sided trace constraint then keeps its dual in the conjugate's domain).
template <typename T>
__device__ __forceinline__ T data_resolvent(T z, T s, T w, T a, T lo, T hi)
{
    const T q = (z + w * a) / (s + w);
    return w * (z - s * a) / (s + w) + s * (q - fmin(fmax(q, lo), hi));
}

// The next iteration's backprojection operand: in orbit layout (ydst; rounded through
// bfloat16 for a BF16 plan), in bfloat16, or as it is.
template <typename T>
__device__ __forceinline__ void store_y1(const ForwardEpi<T> &epi, size_t r, T y, T *ydst)
{
    if constexpr (sizeof(T) == 4) {
        if (ydst) *ydst = epi.yround ? __bfloat162float(__float2bfloat16_rn(y)) : y;
        else if (epi.y1h) epi.y1h[r] = __float2bfloat16_rn(y);
        else epi.y1[r] = y;
    } else {
        epi.y1[r] = y;
    }
}

template <typename T>
__device__ __forceinline__ void forward_epilogue(const ForwardEpi<T> &epi, size_t r, T val, T *ydst = nullptr)
{
    if (epi.mode == 0) {
        epi.g[r] = val * epi.scale;
        return;
    }
    if (epi.mode == 2) {
        // Alg. 1: v = (id + tau dG1^*)^{-1}(v + tau Rt u_bar), tau carried in epi.sigma
        const T z = epi.v1b[r] + epi.sigma * (val * epi.scale);
        epi.v1b[r] = data_resolvent(z, epi.sigma, epi.dw[r], epi.da[r], epi.dlo[r], epi.dhi[r]);
        return;
    }
    if (epi.mode == 3) {
        // Alg. 3: the next iteration backprojects the residual Rt u_new - ft
        const T Ru = val * epi.scale;
        const T y = Ru - epi.da[r];
        epi.Ru[r] = Ru;
        store_y1(epi, r, y, ydst);
        if (epi.t1) epi.t1[r] = y;
        return;
    }
    // Alg. 4: v1 = v1b + sigma Rt u_new; t = (id + sigma dG1^*)^{-1}(2 v1 - v1b);
    // v1b <- v1b + t - v1; and the next iteration's y1 = v1b + sigma Rt u_new.
    const T sigma = epi.sigma;
    const T Ru = val * epi.scale;
    const T vb = epi.v1b[r];
    const T v1 = vb + sigma * Ru;
    const T z = T(2) * v1 - vb;
    const T t = data_resolvent(z, sigma, epi.dw[r], epi.da[r], epi.dlo[r], epi.dhi[r]);
    const T vbn = vb + t - v1;
    epi.Ru[r] = Ru;
    epi.v1b[r] = vbn;
    store_y1(epi, r, vbn + sigma * Ru, ydst);
    if (epi.t1) epi.t1[r] = t;
}

// The same epilogue (modes 1 and 2) on operands fetched ahead: vb = v1b[r], w, a, lo, hi.
__device__ __forceinline__ void forward_epilogue_pre(const ForwardEpi<float> &epi, size_t r, float val, float vb,
                                                     float w, float a, float lo, float hi, float *ydst)
{
    const float sigma = epi.sigma;
    if (epi.mode == 2) {
        const float z = vb + sigma * (val * epi.scale);
        epi.v1b[r] = data_resolvent(z, sigma, w, a, lo, hi);
        return;
    }
    const float Ru = val * epi.scale;
    const float v1 = vb + sigma * Ru;
    const float z = 2.f * v1 - vb;
    const float t = data_resolvent(z, sigma, w, a, lo, hi);
    const float vbn = vb + t - v1;
    epi.Ru[r] = Ru;
    epi.v1b[r] = vbn;
    store_y1(epi, r, vbn + sigma * Ru, ydst);
    if (epi.t1) epi.t1[r] = t;
}

// One row of the march: the NC candidate pixels q, q+1, ... of the lane's interval.
// EXACT1: the first candidate is always inside the interval (A <= 2^F, i.e. h <= ds).
template <typename T, typename S, int NC, bool EXACT1>
__device__ __forceinline__ void march_row(const S *rowp, int dq, int n, int k, int F, double inv2F,
                                          long long Pa, int q, long long A, T &Su, T &Sf)
{
    {
        bool ok = (unsigned)q < (unsigned)n;
        if (!EXACT1) ok = ok && bin_of<T>(Pa, F) == k;
        const T v = ok ? (T)ldv(rowp + dq * q) : T(0);
        acc_sample(Su, Sf, v, Pa, F, inv2F);
    }
    long long P = Pa;
#pragma unroll
    for (int c = 1; c < NC; ++c) {
        P += A;
        const int qq = q + c;
        const bool ok = bin_of<T>(P, F) == k && (unsigned)qq < (unsigned)n;
        if (__any_sync(0xffffffffu, ok)) {
            const T v = ok ? (T)ldv(rowp + dq * qq) : T(0);
            acc_sample(Su, Sf, v, P, F, inv2F);
        }
    }
}

constexpr int FWD_AW = 4;                     // adjacent angles per CTA, one warp each
constexpr int FWD_THREADS = 32 * FWD_AW;

// FP32 ray march over `rows` rows (F = 32, 2^31 <= A <= 2^32).  State: r = P(q_a) - k 2^32
// in [0, A) (the fixed-point fraction of the interval's first pixel q_a), off = element
// offset of pixel (m, q_a), and q_a itself where CHECK.  The second pixel q_a + 1 lies in
// the interval iff r + A < 2^32, i.e. r < lim.  Next row: P += B; B > 0 (BPOS) steps
// q_a back when r >= thr = A - B, B <= 0 steps it forward when r < thr = |B|.
// CHECK = false: every lane's q_a and q_a + 1 are inside [0, n) on these rows.
template <int DQ, bool BPOS, bool CHECK, typename S>
__device__ __forceinline__ void march32(const S *base, int n, int rows, unsigned &r, int &q, int &off,
                                        unsigned A32, unsigned lim, unsigned B32, unsigned thr, float &Su, float &Sf)
{
#pragma unroll FWD_UNROLL
    for (int rr = 0; rr < rows; ++rr) {
        float v1, v2;
        if constexpr (CHECK) {
            v1 = ((unsigned)q < (unsigned)n) ? ldv(base + off) : 0.f;
            v2 = (r < lim && (unsigned)(q + 1) < (unsigned)n) ? ldv(base + off + DQ) : 0.f;
        } else {
            v1 = ldv(base + off);
            v2 = r < lim ? ldv(base + off + DQ) : 0.f;
        }
        Su += v1 + v2;
        Sf = fmaf(one_plus_frac32u(r), v1, Sf);
        Sf = fmaf(one_plus_frac32u(r + A32), v2, Sf);
        if constexpr (BPOS) {
            const bool s = r >= thr;
            r += s ? B32 - A32 : B32;
            off += s ? n - DQ : n;
            if constexpr (CHECK) q -= s ? 1 : 0;
        } else {
            const bool s = r < thr;
            r += s ? A32 - thr : 0u - thr;
            off += s ? n + DQ : n;
            if constexpr (CHECK) q += s ? 1 : 0;
        }
    }
}

// The FP32 march of one lane over rows [mlo, mhi] of the warp, without bounds checks on
// the warp's interior rows [ilo, ihi] (mlo <= ilo, ihi <= mhi; ilo > ihi: none).
template <int DQ, bool BPOS, typename S>
__device__ __forceinline__ void march32_rows(const S *base, int n, long long K, const AngleMarch &am,
                                             int mlo, int mhi, int ilo, int ihi, float &Su, float &Sf)
{
    const long long A = am.A, B = am.B;
    const long long qa = ceil_div_ll(K - (long long)mlo * B - am.Op, A);
    unsigned r = (unsigned)(qa * A + (long long)mlo * B + am.Op - K);
    int q = (int)qa;
    int off = mlo * n + DQ * q;
    const unsigned A32 = (unsigned)A;             // A = 2^32 wraps to 0 (then B = 0)
    const unsigned lim = (unsigned)((1ll << 32) - A);
    const unsigned B32 = (unsigned)B;
    const unsigned thr = BPOS ? (unsigned)(A - B) : (unsigned)(-B);
    if (ilo > ihi) {
        march32<DQ, BPOS, true>(base, n, mhi - mlo + 1, r, q, off, A32, lim, B32, thr, Su, Sf);
        return;
    }
    march32<DQ, BPOS, true>(base, n, ilo - mlo, r, q, off, A32, lim, B32, thr, Su, Sf);
    march32<DQ, BPOS, false>(base, n, ihi - ilo + 1, r, q, off, A32, lim, B32, thr, Su, Sf);
    q = DQ * (off - (ihi + 1) * n);               // off = m n + DQ q
    march32<DQ, BPOS, true>(base, n, mhi - ihi, r, q, off, A32, lim, B32, thr, Su, Sf);
}

// Sum u and sum frac u (FP64) or sum (1 + frac) u (generic FP32) over the pixels of rows
// m0 .. m0 + rows - 1 whose detector coordinate lies in the lane's interval [k, k+1).
template <typename T, typename S, int NC, bool EXACT1>
__device__ __forceinline__ void fwd_march(const S *base, int dq, int n, int k, int F,
                                          const AngleMarch &am, int m0, int rows, T &Su, T &Sf)
{
    const double inv2F = ldexp(1.0, -F);
    const long long K = (long long)k << F;
    const long long A = am.A, B = am.B;
    long long qa = ceil_div_ll(K - (long long)m0 * B - am.Op, A);
    long long Pa = qa * A + (long long)m0 * B + am.Op;   // in [K, K + A)
    int q = (int)qa;
    const S *rowp = base + (size_t)m0 * n;
    // next row: restore P(q_a) in [K, K + A) (|B| <= A: at most one step)
    if (B >= 0) {
        const long long KA = K + A;
#pragma unroll 2
        for (int r = 0; r < rows; ++r) {
            march_row<T, S, NC, EXACT1>(rowp, dq, n, k, F, inv2F, Pa, q, A, Su, Sf);
            Pa += B;
            if (Pa >= KA) { Pa -= A; --q; }
            rowp += n;
        }
    } else {
#pragma unroll 2
        for (int r = 0; r < rows; ++r) {
            march_row<T, S, NC, EXACT1>(rowp, dq, n, k, F, inv2F, Pa, q, A, Su, Sf);
            Pa += B;
            if (Pa < K) { Pa += A; ++q; }
            rowp += n;
        }
    }
}

// Rows m of [0, n) on which q*(m) = Q0 - m b lies in [qlo, qhi] (FP32; the callers'
// margins of half a pixel or more absorb its rounding).  OUTER rounds the range out
// (rows that may touch), otherwise in (rows that surely lie inside).  lo > hi: none.
template <bool OUTER>
__device__ __forceinline__ void rows_in(float Q0, float binv, float qlo, float qhi, int n, int &lo, int &hi)
{
    lo = n;
    hi = -1;
    if (qlo > qhi) return;
    if (binv != 0.f) {
        const float m1 = (Q0 - qhi) * binv, m2 = (Q0 - qlo) * binv;
        float a0 = fminf(m1, m2), a1 = fmaxf(m1, m2);
        a0 = fmaxf(0.f, OUTER ? floorf(a0) : ceilf(a0));
        a1 = fminf((float)(n - 1), OUTER ? ceilf(a1) : floorf(a1));
        if (a0 <= a1) {
            lo = (int)a0;
            hi = (int)a1;
        }
    } else if (Q0 > qlo && Q0 < qhi) {            // rays parallel to the march axis
        lo = 0;
        hi = n - 1;
    }
}

// One CTA of the forward projector: warp w takes angle by*FWD_AW + w and bins
// bx*31 + [0, 31).  The angles are adjacent, so their rays nearly coincide and the
// image rows they read are shared in L1.
template <typename T, typename S, int NC, bool EXACT1>
__device__ __forceinline__ void fwd_body(const S *u, const S *uT, int n, int N, int M, int F,
                                         const AngleMarch *__restrict__ march, const ForwardEpi<T> &epi, int bx, int by)
{
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int l = by * FWD_AW + warp;
    const int kb = bx * 31;                           // first output bin of this warp
    const int k = kb + lane - 1;                      // this lane's interval [k, k+1)
    if (l >= N || kb >= M) return;                    // warp-uniform
    const AngleMarch am = march[l];
    // pixel (m, q) of the march is at base[m*n + dq*q]
    const S *base = (am.layout ? u : uT) + (am.flip ? (n - 1) : 0);
    // q*(m) = Q0 - m b: the real pick coordinate where P(q, m) = k 2^F
    const float Q0 = (float)k * am.kA - am.oA;
    int mlo, mhi;                                     // rows where the lane's pixel run may be inside [0, n)
    rows_in<true>(Q0, am.binv, -(float)NC - 1.f, (float)n + 1.f, n, mlo, mhi);
    const int mlo_w = __reduce_min_sync(0xffffffffu, mlo);
    const int mhi_w = __reduce_max_sync(0xffffffffu, mhi);
    T Su = T(0), Sf = T(0);
    if (mlo_w <= mhi_w) {
        if constexpr (sizeof(T) == 4 && EXACT1 && NC == 2) {
            // interior rows: q_a in [1, n - 3] for every lane, no bounds checks needed
            int ilo, ihi;
            rows_in<false>(Q0, am.binv, 0.5f, (float)n - 3.5f, n, ilo, ihi);
            const int ilo_w = max(__reduce_max_sync(0xffffffffu, ilo), mlo_w);
            const int ihi_w = min(__reduce_min_sync(0xffffffffu, ihi), mhi_w);
            const long long K = (long long)k << 32;
            if (am.B > 0) {                           // B = 0 takes the B < 0 march (thr = 0: never steps)
                if (am.flip) march32_rows<-1, true>(base, n, K, am, mlo_w, mhi_w, ilo_w, ihi_w, Su, Sf);
                else march32_rows<1, true>(base, n, K, am, mlo_w, mhi_w, ilo_w, ihi_w, Su, Sf);
            } else {
                if (am.flip) march32_rows<-1, false>(base, n, K, am, mlo_w, mhi_w, ilo_w, ihi_w, Su, Sf);
                else march32_rows<1, false>(base, n, K, am, mlo_w, mhi_w, ilo_w, ihi_w, Su, Sf);
            }
        } else {
            fwd_march<T, S, NC, EXACT1>(base, am.flip ? -1 : 1, n, k, F, am, mlo_w, mhi_w - mlo_w + 1, Su, Sf);
        }
    }
    T Bk, Ak;
    if constexpr (sizeof(T) == 4) { Bk = Sf - Su; Ak = Su - Bk; }
    else { Bk = Sf; Ak = Su - Sf; }
    const T Bprev = __shfl_up_sync(0xffffffffu, Bk, 1);
    if (lane >= 1 && k < M) forward_epilogue(epi, (size_t)l * M + k, Ak + Bprev);
}

template <typename T, typename S, int NC, bool EXACT1>
__global__ void __launch_bounds__(FWD_THREADS)
k_forward(const S *__restrict__ u, const S *__restrict__ uT, int n, int N, int M, int F,
          const AngleMarch *__restrict__ march, ForwardEpi<T> epi)
{
    fwd_body<T, S, NC, EXACT1>(u, uT, n, N, M, F, march, epi, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Symmetric forward path (OrbitJob): one canonical ray march per job serves the
// job's up to four angles, reading the four channels of the orbit image at once.
// ---------------------------------------------------------------------------

// The orbit image: channel v of the canonical march pixel (q, m) is u(T_v^{-1}(q, m)),
//     ubar[m][q] = (u[q][m], u[n-1-q][m], u[m][q], u[n-1-m][q]),
// FP32 (a BF16 plan's operand is widened here).  Rows of
// orbit_pitch pixels, pixel 0 at ORBIT_PAD; the pads keep the zeros they got when the plan was
// made.  Two planes (float2): channels {0, 1}, then {2, 3}.
__device__ __forceinline__ void orbit_store(float *ubar, size_t plane, size_t o, float a, float b, float c,
                                            float d)
{
    reinterpret_cast<float2 *>(ubar)[o] = make_float2(a, b);
    reinterpret_cast<float2 *>(ubar)[plane + o] = make_float2(c, d);
}

// 32 x 32 tiles: four coalesced tile loads (two of them transposed through shared
// memory), one coalesced record store per pixel.
template <typename S>
__device__ __forceinline__ void orbit_image_body(const S *u, float *ubar, int n, int bx, int by)
{
    __shared__ float tA[32][33], tB[32][33], tC[32][33], tD[32][33];
    const size_t pitch = orbit_pitch(n), plane = pitch * n;
    ubar += 2 * ORBIT_PAD;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int q0 = bx * 32, m0 = by * 32;
    for (int r = ty; r < 32; r += 8) {
        const int mr = m0 + r, qc = q0 + tx;          // tiles A, B: rows m, columns q
        if (mr < n && qc < n) {
            tA[r][tx] = ldv(u + (size_t)mr * n + qc);
            tB[r][tx] = ldv(u + (size_t)(n - 1 - mr) * n + qc);
        }
        const int qr = q0 + r, mc = m0 + tx;          // tiles C, D: rows q, columns m
        if (qr < n && mc < n) {
            tC[r][tx] = ldv(u + (size_t)qr * n + mc);
            tD[r][tx] = ldv(u + (size_t)(n - 1 - qr) * n + mc);
        }
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int m = m0 + r, q = q0 + tx;
        if (m < n && q < n)
            orbit_store(ubar, plane, (size_t)m * pitch + q, tC[tx][r], tD[tx][r], tA[r][tx], tB[r][tx]);
    }
}

template <typename S>
__global__ void __launch_bounds__(256)
k_orbit_image(const S *u, float *ubar, int n)
{
    pdl_wait();
    pdl_trigger();
    orbit_image_body<S>(u, ubar, n, blockIdx.x, blockIdx.y);
}

// The orbit image and, for the pixels (m, q) of the CTA's tile, the TV dual step of
// Alg. 4 (both read u; each pixel's TV step runs exactly once over the grid).  The TV
// operands (bar v2, and bar u for Alg. 5) are fetched before the tile barrier, and u with
// its forward neighbours comes from tile A (rows m, columns q, plus a one-pixel halo), so
// the kernel waits on global memory once; the arithmetic is that of tv_dual_at.
__global__ void __launch_bounds__(256)
k_orbit_image_tv(const float *u, float *ubar, int n, TvDualJob<float> tv)
{
    pdl_wait();
    pdl_trigger();
    __shared__ float tA[33][33], tB[32][33], tC[32][33], tD[32][33];
    const size_t pitch = orbit_pitch(n), plane = pitch * n;
    ubar += 2 * ORBIT_PAD;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int q0 = blockIdx.x * 32, m0 = blockIdx.y * 32;
    const size_t nn = (size_t)n * n;
    float vbx[4], vby[4], ubv[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int m = m0 + ty + 8 * k, q = q0 + tx;
        vbx[k] = vby[k] = ubv[k] = 0.f;
        if (m < n && q < n) {
            const size_t e = (size_t)m * n + q;
            vbx[k] = tv.v2b[e];
            vby[k] = tv.v2b[e + nn];
            if (tv.ub) ubv[k] = tv.ub[e];
        }
    }
    for (int r = ty; r < 32; r += 8) {
        const int mr = m0 + r, qc = q0 + tx;          // tiles A, B: rows m, columns q
        if (mr < n && qc < n) {
            tA[r][tx] = u[(size_t)mr * n + qc];
            tB[r][tx] = u[(size_t)(n - 1 - mr) * n + qc];
        }
        const int qr = q0 + r, mc = m0 + tx;          // tiles C, D: rows q, columns m
        if (qr < n && mc < n) {
            tC[r][tx] = u[(size_t)qr * n + mc];
            tD[r][tx] = u[(size_t)(n - 1 - qr) * n + mc];
        }
    }
    if (ty == 0 && m0 + 32 < n && q0 + tx < n) tA[32][tx] = u[(size_t)(m0 + 32) * n + q0 + tx];   // halo row
    if (ty == 1 && q0 + 32 < n && m0 + tx < n) tA[tx][32] = u[(size_t)(m0 + tx) * n + q0 + 32];   // halo column
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int m = m0 + r, q = q0 + tx;
        if (m < n && q < n)
            orbit_store(ubar, plane, (size_t)m * pitch + q, tC[tx][r], tD[tx][r], tA[r][tx], tB[r][tx]);
    }
    const float st = tv.sigma * tv.tau;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = ty + 8 * k, m = m0 + r, q = q0 + tx;
        if (m >= n || q >= n) continue;
        const size_t e = (size_t)m * n + q;
        const float c = tA[r][tx];
        const float gx = (m < n - 1) ? (tA[r + 1][tx] - c) * tv.inv_h : 0.f;
        const float gy = (q < n - 1) ? (tA[r][tx + 1] - c) * tv.inv_h : 0.f;
        const float bx = vbx[k], by = vby[k];
        const float vx = bx + st * gx, vy = by + st * gy;
        const float zx = 2.f * vx - bx, zy = 2.f * vy - by;
        float tx2 = 0.f, ty2 = 0.f;
        if (tv.lam > 0.f) {
            const float den = fmax(1.f, tv.tau * sqrt(zx * zx + zy * zy) / tv.lam);
            tx2 = zx / den;
            ty2 = zy / den;
        }
        const float nbx = bx + tx2 - vx, nby = by + ty2 - vy;
        tv.v2b[e] = nbx;
        tv.v2b[e + nn] = nby;
        tv.y2[e] = nbx + st * gx;
        tv.y2[e + nn] = nby + st * gy;
        if (tv.t2) {
            tv.t2[e] = tx2;
            tv.t2[e + nn] = ty2;
        }
        if (tv.ub) tv.ub[e] = ubv[k] + fmax(2.f * c - ubv[k], 0.f) - c;
    }
}

// Asynchronous copies global -> shared (cp.async): commit, and wait on this thread's groups.
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Paired FP32 arithmetic (add / sub / fma on two lanes of a 64-bit register pair, one
// instruction for two values; each lane rounds exactly as the scalar instruction).
#ifndef CTR_F32X2
#define CTR_F32X2 1
#endif
__device__ __forceinline__ float2 fadd2(float2 a, float2 b)
{
#if CTR_F32X2
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__device__ __forceinline__ float2 fsub2(float2 a, float2 b)
{
#if CTR_F32X2
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
#else
    return make_float2(a.x - b.x, a.y - b.y);
#endif
}
// a * b + c per lane
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c)
{
#if CTR_F32X2
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}

#include "orbit.cuh"
#include "orbit64.cuh"

// The fold of the symmetric backprojection's partial planes, then the
// backprojection epilogue (grid-stride over the pixels).
template <typename T>
__global__ void __launch_bounds__(256)
k_bp_fold(const T *part, int groups, int n, BackprojEpi<T> epi)
{
    pdl_wait();
    pdl_trigger();
    const size_t nn = (size_t)n * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int i = pix_i(e, n), j = pix_j(e, n);
        bp_epilogue(epi, n, i, j, orbit_fold<T>(part, groups, n, i, j));
    }
}

// Batched stages: block b of the launch belongs to the slice s with
// prefix[s] <= b < prefix[s+1]; the slice's parameters come from its SliceDesc.
__device__ __forceinline__ int find_slice(const int *__restrict__ prefix, int ns, int b)
{
    int lo = 0, hi = ns - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(32 * BP_TY)
k_backproject_batch(const SliceDesc *__restrict__ sd, const int *__restrict__ prefix, int ns)
{
    const int s = find_slice(prefix, ns, blockIdx.x);
    const SliceDesc &d = sd[s];
    const int local = blockIdx.x - prefix[s];
    const int bx = local % d.bp_tiles_x, rest = local / d.bp_tiles_x;
    const int by = rest % d.bp_tiles_y, bz = rest / d.bp_tiles_y;
    bp_body<float, float>(d.y1, d.n, d.N, d.M, 32, d.wstride, d.per_group, d.geom, d.bpe,
                          d.bp_groups > 1 ? d.bp_part : nullptr, bx, by, bz);
}

__device__ __forceinline__ ObpArgs obp_args(const SliceDesc &d)
{
    return ObpArgs{d.ybar, d.jobs, d.bp_part, d.n, d.bar_pitch, d.bar_pad, d.obp_win, d.bp_groups,
                   {d.job_list[0], d.job_list[1], d.job_list[2]}};
}

__global__ void __launch_bounds__(OBP_THREADS, 4)
k_backproject_orbit_batch(const SliceDesc *__restrict__ sd, const int *__restrict__ prefix, int ns)
{
    const int s = find_slice(prefix, ns, blockIdx.x);
    const SliceDesc &d = sd[s];
    const int local = blockIdx.x - prefix[s];
    const int bx = local % d.bp_tiles_x, rest = local / d.bp_tiles_x;
    const int by = rest % d.bp_tiles_y, bz = rest / d.bp_tiles_y;
    if (d.pair_jobs) obp_body<2, false>(obp_args(d), bx, by, bz);
    else obp_body<4, false>(obp_args(d), bx, by, bz);
}

__global__ void __launch_bounds__(256)
k_orbit_image_batch(const SliceDesc *__restrict__ sd, const int *__restrict__ prefix, int ns)
{
    const int s = find_slice(prefix, ns, blockIdx.x);
    const SliceDesc &d = sd[s];
    const int local = blockIdx.x - prefix[s], tiles = (d.n + 31) / 32;
    orbit_image_body<float>(d.u, d.ubar, d.n, local % tiles, local / tiles);
}

__device__ __forceinline__ OfwArgs ofw_args(const SliceDesc &d)
{
    return OfwArgs{d.ubar, d.jobs, d.n, d.M, d.n_jobs, d.job_list[1]};
}

__global__ void __launch_bounds__(OFW_THREADS, 6)
k_forward_orbit_batch(const SliceDesc *__restrict__ sd, const int *__restrict__ prefix, int ns)
{
    const int s = find_slice(prefix, ns, blockIdx.x);
    const SliceDesc &d = sd[s];
    const int local = blockIdx.x - prefix[s];
    if (d.pair_jobs)
        ofw_body<2, OFW_JOBS, OFW_SEGS, false>(ofw_args(d), d.fwe, local % d.fwd_chunks, local / d.fwd_chunks);
    else ofw_body<4, OFW_JOBS, OFW_SEGS, false>(ofw_args(d), d.fwe, local % d.fwd_chunks, local / d.fwd_chunks);
}

__global__ void __launch_bounds__(FWD_THREADS)
k_forward_batch(const SliceDesc *__restrict__ sd, const int *__restrict__ prefix, int ns)
{
    const int s = find_slice(prefix, ns, blockIdx.x);
    const SliceDesc &d = sd[s];
    const int local = blockIdx.x - prefix[s];
    fwd_body<float, float, 2, true>(d.u, d.uT, d.n, d.N, d.M, 32, d.march, d.fwe, local % d.fwd_chunks,
                                    local / d.fwd_chunks);
}

template <typename T>
__global__ void __launch_bounds__(256) k_transpose(const T *__restrict__ in, T *__restrict__ out, int n)
{
    __shared__ T tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = by + r, j = bx + threadIdx.x;
        if (i < n && j < n) tile[r][threadIdx.x] = in[(size_t)i * n + j];
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = bx + r, j = by + threadIdx.x;
        if (i < n && j < n) out[(size_t)i * n + j] = tile[threadIdx.x][r];
    }
}

template <typename T>
size_t bp_smem(const ctr_plan *p)
{
    using T2 = typename Pair<T>::type;
    return sizeof(T2) * BP_ACH * p->wstride + 3 * sizeof(long long) * BP_ACH + sizeof(int) * BP_ACH;
}

template <typename T, typename S, int NC, bool EXACT1>
void launch_fwd_cfg(const ctr_plan *p, dim3 grid, const S *u, const S *uT, const ForwardEpi<T> &epi, cudaStream_t s)
{
    k_forward<T, S, NC, EXACT1><<<grid, FWD_THREADS, 0, s>>>(u, uT, p->n, p->N, p->M, p->F, p->d_march, epi);
}

// g (N x M) into orbit layout (bar)
template <typename S>
ctr_status launch_orbit_sino(const ctr_plan *p, const S *g, float *bar, cudaStream_t s)
{
    p->launches++;
    const dim3 grid((p->M + 255) / 256, p->n_jobs);
    auto kern = p->pair_jobs ? k_orbit_sino<S, 2> : k_orbit_sino<S, 4>;
    launch_pdl(p->pdl != 0, kern, grid, dim3(256), 0, s, g, p->M, p->job_list[1], p->bar_pitch, p->bar_pad,
               (const OrbitJob *)p->d_jobs, bar);
    CTR_CHECK_LAUNCH("k_orbit_sino");
    return CTR_OK;
}

template <typename T, typename S>
ctr_status bp_impl(const ctr_plan *p, const S *g, const BackprojEpi<T> &epi, cudaStream_t s, bool defer_reduce)
{
    if constexpr (sizeof(T) == 4) {
        if (p->orbit) {
            const int G = p->obp_groups;
            const dim3 grid((p->n + 31) / 32, (p->n + 31) / 32, G);
            float *part = (float *)p->obp_part;
            const float *bar = (const float *)p->ybar;
            const bool plain = (const void *)g != p->ybar;                 // an operand in sinogram layout
            // small calls are bound by their launches: the kernel stages the rows themselves
            const bool direct = std::is_same<S, float>::value && plain && p->n <= obp_direct_n(p->pair_jobs != 0);
            if (plain && !direct) {
                ctr_status st = launch_orbit_sino<S>(p, g, (float *)p->gbar, s);
                if (st != CTR_OK) return st;
                bar = (const float *)p->gbar;
            }
            p->launches++;
            auto kern = p->pair_jobs ? (defer_reduce ? k_backproject_orbit<2, false> : k_backproject_orbit<2, true>)
                                     : (defer_reduce ? k_backproject_orbit<4, false> : k_backproject_orbit<4, true>);
            ObpArgs args = obp_args(p, bar);
            if (direct) args.g = (const float *)g;
            launch_pdl(p->pdl != 0, kern, grid, dim3(OBP_THREADS), obp_smem(p->pair_jobs ? 2 : 4), s,
                       args);
            CTR_CHECK_LAUNCH("k_backproject_orbit");
            if (!defer_reduce) {
                const size_t nn = (size_t)p->n * p->n;
                int blocks = (int)((nn + 255) / 256);
                if (blocks > 4096) blocks = 4096;
                p->launches++;
                launch_pdl(p->pdl != 0, k_bp_fold<float>, dim3(blocks), dim3(256), 0, s, (const float *)part, G, p->n, epi);
                CTR_CHECK_LAUNCH("k_bp_fold");
            }
            return CTR_OK;
        }
    }
    if constexpr (std::is_same<T, double>::value) {
        if (p->sym64) {
            ctr_status st = launch_backproject_sym64(p, g, s);
            if (st != CTR_OK || defer_reduce) return st;
            const size_t nn = (size_t)p->n * p->n;
            p->launches++;
            launch_pdl(p->pdl != 0, k_bp_fold<double>, dim3((unsigned)std::min<size_t>((nn + 127) / 128, 4096)), dim3(128), 0,
                       s, (const double *)p->bp_part, p->bp_groups, p->n, epi);
            CTR_CHECK_LAUNCH("k_bp_fold");
            return CTR_OK;
        }
    }
    const int G = p->bp_groups;
    const int per = (p->N + G - 1) / G;
    dim3 grid((p->n + BP_TJ - 1) / BP_TJ, (p->n + BP_TI - 1) / BP_TI, G);
    T *part = G > 1 ? (T *)p->bp_part : nullptr;
    p->launches++;
    k_backproject<T, S><<<grid, 32 * BP_TY, bp_smem<T>(p), s>>>(g, p->n, p->N, p->M, p->F, p->wstride, per,
                                                                 p->d_geom, epi, part);
    CTR_CHECK_LAUNCH("k_backproject");
    if (G > 1 && !defer_reduce) {
        const size_t nn = (size_t)p->n * p->n;
        int blocks = (int)((nn + 255) / 256);
        if (blocks > 4096) blocks = 4096;
        p->launches++;
        k_bp_reduce<T><<<blocks, 256, 0, s>>>(part, G, p->n, epi);
        CTR_CHECK_LAUNCH("k_bp_reduce");
    }
    return CTR_OK;
}

template <typename T, typename S>
ctr_status fwd_impl(const ctr_plan *p, const S *u, const S *uT, const ForwardEpi<T> &epi, cudaStream_t s,
                    const TvDualJob<T> *tv = nullptr)
{
    const bool exact1 = p->h <= p->ds;
    if constexpr (sizeof(T) == 4) {
        if (p->orbit) {
            float *ub = (float *)p->ubar;
            p->launches++;
            const dim3 og((p->n + 31) / 32, (p->n + 31) / 32);
            if constexpr (std::is_same<S, float>::value) {
                if (tv) launch_pdl(p->pdl != 0, k_orbit_image_tv, og, dim3(256), 0, s, u, ub,
                                   p->n, *tv);
                else launch_pdl(p->pdl != 0, k_orbit_image<S>, og, dim3(256), 0, s, u, ub, p->n);
            } else {
                launch_pdl(p->pdl != 0, k_orbit_image<S>, og, dim3(256), 0, s, u, ub, p->n);
            }
            CTR_CHECK_LAUNCH("k_orbit_image");
            p->launches++;
            launch_forward_orbit(p, ub, epi, s);
            CTR_CHECK_LAUNCH("k_forward_orbit");
            return CTR_OK;
        }
    }
    if constexpr (std::is_same<T, double>::value)
        if (p->sym64) return launch_forward_sym64(p, u, epi, s);
    p->launches++;
    dim3 grid(fwd_grid_x(p->M), fwd_grid_y(p->N));
    switch (p->ncand * 2 + (exact1 ? 1 : 0)) {
    case 2: launch_fwd_cfg<T, S, 1, false>(p, grid, u, uT, epi, s); break;
    case 3: launch_fwd_cfg<T, S, 1, true>(p, grid, u, uT, epi, s); break;
    case 4: launch_fwd_cfg<T, S, 2, false>(p, grid, u, uT, epi, s); break;
    case 5: launch_fwd_cfg<T, S, 2, true>(p, grid, u, uT, epi, s); break;
    case 6: launch_fwd_cfg<T, S, 3, false>(p, grid, u, uT, epi, s); break;
    case 7: launch_fwd_cfg<T, S, 3, true>(p, grid, u, uT, epi, s); break;
    case 8: launch_fwd_cfg<T, S, 4, false>(p, grid, u, uT, epi, s); break;
    case 9: launch_fwd_cfg<T, S, 4, true>(p, grid, u, uT, epi, s); break;
    default: return fail(CTR_EUNSUPPORTED, "forward projector: too many pixels per detector interval");
    }
    CTR_CHECK_LAUNCH("k_forward");
    return CTR_OK;
}

}  // namespace

template <typename T>
ctr_status configure_radon(const ctr_plan *p)
{
    const size_t smem = bp_smem<T>(p);
    ctr_status st = raise_smem_limit(k_backproject<T, T>, smem);
    if (st == CTR_OK && p->orbit)
        st = p->pair_jobs ? raise_smem_limit(k_backproject_orbit<2, false>, obp_smem(2), true)
                          : raise_smem_limit(k_backproject_orbit<4, false>, obp_smem(4), true);
    if (st == CTR_OK && p->orbit)
        st = p->pair_jobs ? raise_smem_limit(k_backproject_orbit<2, true>, obp_smem(2), true)
                          : raise_smem_limit(k_backproject_orbit<4, true>, obp_smem(4), true);
    if constexpr (sizeof(T) == 4)
        if (st == CTR_OK) st = raise_smem_limit(k_backproject<float, __nv_bfloat16>, smem);
    return st;
}

ctr_status launch_backproject_bf16(const ctr_plan *p, const __nv_bfloat16 *g, const BackprojEpi<float> &epi,
                                   cudaStream_t s, bool defer_reduce)
{
    return bp_impl<float, __nv_bfloat16>(p, g, epi, s, defer_reduce);
}

ctr_status launch_forward_bf16(const ctr_plan *p, const __nv_bfloat16 *u, const __nv_bfloat16 *uT,
                               const ForwardEpi<float> &epi, cudaStream_t s)
{
    return fwd_impl<float, __nv_bfloat16>(p, u, uT, epi, s);
}

template <typename T>
ctr_status launch_backproject(const ctr_plan *p, const T *g, const BackprojEpi<T> &epi, cudaStream_t s,
                              bool defer_reduce)
{
    return bp_impl<T, T>(p, g, epi, s, defer_reduce);
}

template <typename T>
ctr_status launch_forward(const ctr_plan *p, const T *u, const T *uT, const ForwardEpi<T> &epi, cudaStream_t s,
                          const TvDualJob<T> *tv)
{
    return fwd_impl<T, T>(p, u, uT, epi, s, tv);
}

template <typename T>
ctr_status launch_transpose(const ctr_plan *p, const T *in, T *out, cudaStream_t s)
{
    dim3 grid((p->n + 31) / 32, (p->n + 31) / 32);
    p->launches++;
    k_transpose<T><<<grid, dim3(32, 8), 0, s>>>(in, out, p->n);
    CTR_CHECK_LAUNCH("k_transpose");
    return CTR_OK;
}

int backproject_tile_rows() { return BP_TI; }

template <typename T>
bool bp_deferred(const ctr_plan *p)
{
    return p->bp_groups > 1 || (sizeof(T) == 4 && p->orbit) || p->sym64;
}
template bool bp_deferred<float>(const ctr_plan *);
template bool bp_deferred<double>(const ctr_plan *);

int fwd_grid_x(int M) { return (M + 30) / 31; }

int fwd_shape(const ctr_plan *p) { return ofw_shape(p); }

int ofw_batch_groups(const ctr_plan *p) { return ofw_groups(p, OFW_JOBS); }

size_t sym64_image_bytes(int n) { return 2 * sizeof(double2) * (size_t)n * f64_pitch(n); }

int orbit_fwd_chunks(const std::vector<OrbitJob> &jobs, int M, int F)
{
    const int lanes = F == 32 ? OFW_LANES : F64_LANES;
    int most = 1;
    for (const OrbitJob &j : jobs) {
        const int nb = (int)((lanes * j.am.A) >> F) - 1;
        most = std::max(most, (M + nb - 1) / nb);
    }
    return most;
}
int fwd_grid_y(int N) { return (N + FWD_AW - 1) / FWD_AW; }

size_t obp_smem_bytes(const ctr_plan *p) { return obp_smem(p->pair_jobs ? 2 : 4); }

int obp_window(const std::vector<OrbitJob> &jobs)
{
    // bins of a tile's block centres (30 C + 28 S), two on the left and three on the right,
    // and what the 16-byte alignment of the first bin adds
    long long w = 0;
    for (const OrbitJob &j : jobs) w = std::max(w, (30 * j.am.A + 28 * j.am.B) >> 32);
    return std::min(OBP_WIN, ((int)w + 9) & ~1);
}

template <typename T>
ctr_status launch_orbit_bar(const ctr_plan *p, const T *g, cudaStream_t s)
{
    return launch_orbit_sino<T>(p, g, (float *)p->ybar, s);
}
template ctr_status launch_orbit_bar<float>(const ctr_plan *, const float *, cudaStream_t);
template ctr_status launch_orbit_bar<__nv_bfloat16>(const ctr_plan *, const __nv_bfloat16 *, cudaStream_t);

size_t bp_smem_bytes(int wstride)
{
    return sizeof(float2) * BP_ACH * wstride + 3 * sizeof(long long) * BP_ACH + sizeof(int) * BP_ACH;
}

void bp_tiles(int n, int &tx, int &ty)
{
    tx = (n + BP_TJ - 1) / BP_TJ;
    ty = (n + BP_TI - 1) / BP_TI;
}

ctr_status configure_batch_radon(size_t bp_smem, size_t obp_smem_max)
{
    ctr_status st = raise_smem_limit(k_backproject_batch, bp_smem);
    if (st == CTR_OK) st = raise_smem_limit(k_backproject_orbit_batch, obp_smem_max, true);
    return st;
}

// One batched projector stage over all slices (blocks = total CTAs of the stage).
ctr_status launch_batch_radon(int stage, const SliceDesc *sd, const int *prefix, int ns, int blocks, size_t smem,
                              cudaStream_t s)
{
    if (blocks <= 0) return CTR_OK;
    switch (stage) {
    case BS_BP: k_backproject_batch<<<blocks, 32 * BP_TY, smem, s>>>(sd, prefix, ns); break;
    case BS_BP_SYM: k_backproject_orbit_batch<<<blocks, OBP_THREADS, smem, s>>>(sd, prefix, ns); break;
    case BS_ORBIT: k_orbit_image_batch<<<blocks, 256, 0, s>>>(sd, prefix, ns); break;
    case BS_FWD_SYM: k_forward_orbit_batch<<<blocks, OFW_THREADS, 0, s>>>(sd, prefix, ns); break;
    case BS_FWD: k_forward_batch<<<blocks, FWD_THREADS, 0, s>>>(sd, prefix, ns); break;
    default: return fail(CTR_EINVAL, "not a projector stage");
    }
    CTR_CHECK_LAUNCH("batched projector stage");
    return CTR_OK;
}

template ctr_status launch_backproject<float>(const ctr_plan *, const float *, const BackprojEpi<float> &, cudaStream_t,
                                             bool);
template ctr_status launch_backproject<double>(const ctr_plan *, const double *, const BackprojEpi<double> &,
                                              cudaStream_t, bool);
template ctr_status launch_forward<float>(const ctr_plan *, const float *, const float *, const ForwardEpi<float> &,
                                         cudaStream_t, const TvDualJob<float> *);
template ctr_status launch_forward<double>(const ctr_plan *, const double *, const double *,
                                          const ForwardEpi<double> &, cudaStream_t, const TvDualJob<double> *);
template ctr_status configure_radon<float>(const ctr_plan *);
template ctr_status configure_radon<double>(const ctr_plan *);
template ctr_status launch_transpose<float>(const ctr_plan *, const float *, float *, cudaStream_t);
template ctr_status launch_transpose<double>(const ctr_plan *, const double *, double *, cudaStream_t);
template ctr_status launch_transpose<__nv_bfloat16>(const ctr_plan *, const __nv_bfloat16 *, __nv_bfloat16 *, cudaStream_t);

}  // namespace ctr
