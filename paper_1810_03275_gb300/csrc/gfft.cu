// The preconditioner's passes for FP32 images of n = L V pixels (L, V <= 32, 2^a 3^b): one warp
// per transform in two register-resident stages, for the sizes that are not 32 V with V a power
// of two (fft.cu has those).  Same real-input form, buffers and epilogues as fft.cu's passes.
//
//   x[l + L m] -> DFT_V over m in lane l's registers -> times W_n^{l k1}, through shared memory
//   -> DFT_L over l in lane k1's registers -> X[k1 + V k2]; the inverse runs the steps backwards.
//
// What bounds these sizes is latency, not bytes (384^2: 0.6 MB a pass).  The CTA-level passes
// give a transform to 256 threads, of which a radix-8 stage of 768 points keeps 96 busy, with a
// barrier after each of four or five stages and the same again for the inverse.  Here a transform
// waits once each way, for its transposition through shared memory (rows padded to an odd length:
// both directions are free of bank conflicts), and every butterfly is in registers.
// An iteration of Alg. 4 (n / 2 views), CTA-level -> two-stage, us: 64^2 24.6 -> 18.4,
// 128^2 30.6 -> 23.8, 216^2 38.1 -> 30.1, 384^2 54.3 -> 44.2, 432^2 61.1 -> 48.8,
// 576^2 79.8 -> 73.6, 648^2 103 -> 91, 768^2 136.9 -> 135.9, 864^2 172 -> 170 (there the projectors
// hide it); M^{-1} y alone 768^2 33.1 -> 25 (launched by the host: 22 to 27), 864^2 37.4 -> 33.0.
// Error against 64 bits 1.9e-7 .. 2.8e-7 in both.
#include "ctr_internal.cuh"

namespace ctr {
namespace {

// cos and sin of 2 pi t / N, t = 0 .. N - 1, by their power series
constexpr double series(double x, bool sine)
{
    double term = sine ? x : 1.0, sum = term;
    for (int k = 1; k < 24; ++k) {
        const int a = 2 * k + (sine ? 1 : 0);
        term *= -x * x / ((a - 1.0) * a);
        sum += term;
    }
    return sum;
}
template <int N> struct Roots {
    float c[N], s[N];
    constexpr Roots() : c(), s()
    {
        for (int t = 0; t < N; ++t) {
            const double x = 6.283185307179586476925 * (2 * t < N ? t : t - N) / N;   // |x| <= pi
            c[t] = (float)series(x, false);
            s[t] = (float)series(x, true);
        }
        c[0] = 1.f;
        s[0] = 0.f;
        if (N % 2 == 0) { c[N / 2] = -1.f; s[N / 2] = 0.f; }
        if (N % 4 == 0) { c[N / 4] = c[3 * N / 4] = 0.f; s[N / 4] = 1.f; s[3 * N / 4] = -1.f; }
    }
};

// d e^{S 2 pi i t / N}, t a constant once the loops are unrolled
template <int N, int S>
__device__ __forceinline__ float2 rot(float2 d, int t)
{
    constexpr Roots<N> R{};
    t %= N;
    if (t == 0) return d;
    if (2 * t == N) return make_float2(-d.x, -d.y);
    if (4 * t == N) return S > 0 ? make_float2(-d.y, d.x) : make_float2(d.y, -d.x);
    if (4 * t == 3 * N) return S > 0 ? make_float2(d.y, -d.x) : make_float2(-d.y, d.x);
    const float c = R.c[t], s = (float)S * R.s[t];
    return make_float2(d.x * c - d.y * s, d.x * s + d.y * c);
}

__device__ __forceinline__ float2 add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// N-point DFT with sign S in registers, natural order in and out: R sub-transforms of the
// inputs r, r + R, ..., twiddled and combined.
template <int N, int S>
__device__ __forceinline__ void dft(float2 (&v)[N])
{
    if constexpr (N == 1) {
        return;
    } else if constexpr (N == 2) {
        const float2 a = v[0], b = v[1];
        v[0] = add(a, b);
        v[1] = sub(a, b);
    } else if constexpr (N == 3) {
        constexpr float h = 0.86602540378443864676f;
        const float2 a = v[0], t = add(v[1], v[2]), d = sub(v[1], v[2]);
        const float2 m = make_float2(fmaf(-0.5f, t.x, a.x), fmaf(-0.5f, t.y, a.y));
        const float2 e = make_float2(-S * h * d.y, S * h * d.x);
        v[0] = add(a, t);
        v[1] = add(m, e);
        v[2] = sub(m, e);
    } else if constexpr (N == 4) {
        const float2 a = add(v[0], v[2]), b = sub(v[0], v[2]), c = add(v[1], v[3]);
        const float2 d = rot<4, S>(sub(v[1], v[3]), 1);
        v[0] = add(a, c);
        v[1] = add(b, d);
        v[2] = sub(a, c);
        v[3] = sub(b, d);
    } else {
        constexpr int R = N % 3 == 0 ? 3 : N % 4 == 0 ? 4 : 2, M = N / R;
        float2 y[R][M];
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int m = 0; m < M; ++m) y[r][m] = v[r + R * m];
            dft<M, S>(y[r]);
        }
#pragma unroll
        for (int k = 0; k < M; ++k) {
            float2 t[R];
#pragma unroll
            for (int r = 0; r < R; ++r) t[r] = rot<N, S>(y[r][k], r * k);
            dft<R, S>(t);
#pragma unroll
            for (int j = 0; j < R; ++j) v[k + M * j] = t[j];
        }
    }
}

template <int L, int V> struct Two {
    static constexpr int n = L * V, H = n / 2 + 1, P = L | 1;   // padded row of the transposition
    static constexpr int buf = V * P;
};

__device__ __forceinline__ float2 twiddle(float2 a, float2 w) { return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x); }

// v[m] = x[lane + L m] (lane < L) in, w[k2] = X[lane + V k2] (lane < V) out
template <int L, int V>
__device__ __forceinline__ void two_fwd(float2 (&v)[V], float2 (&w)[L], int lane, float2 *buf, const float2 *tw)
{
    using T = Two<L, V>;
    if (lane < L) {
        dft<V, -1>(v);
#pragma unroll
        for (int k = 0; k < V; ++k) buf[k * T::P + lane] = k ? twiddle(v[k], tw[lane * k]) : v[k];
    }
    __syncwarp();
    if (lane < V) {
#pragma unroll
        for (int l = 0; l < L; ++l) w[l] = buf[lane * T::P + l];
        dft<L, -1>(w);
    }
    __syncwarp();
}

// the steps backwards, unnormalised: w[k2] = X[lane + V k2] in, v[m] = x[lane + L m] out
template <int L, int V>
__device__ __forceinline__ void two_inv(float2 (&w)[L], float2 (&v)[V], int lane, float2 *buf, const float2 *tw)
{
    using T = Two<L, V>;
    if (lane < V) {
        dft<L, +1>(w);
#pragma unroll
        for (int l = 0; l < L; ++l) {
            float2 t = tw[l * lane];
            t.y = -t.y;
            buf[lane * T::P + l] = l ? twiddle(w[l], t) : w[l];
        }
    }
    __syncwarp();
    if (lane < L) {
#pragma unroll
        for (int k = 0; k < V; ++k) v[k] = buf[k * T::P + lane];
        dft<V, +1>(v);
    }
}

template <int N>
__device__ __forceinline__ void stage(float2 *s_tw, const float2 *__restrict__ tw)
{
    for (int t = threadIdx.x; t < N; t += blockDim.x) s_tw[t] = __ldg(tw + t);
}

// (2 and 1 warps per CTA: 384^2 43.8 -> 51.3 us per iteration, 576^2 73.5 -> 85.0; 2 and 4 the same)
constexpr int ROWS_THREADS = 256, COL_WARPS = 4, INV_WARPS = 2;

// Forward row pass, one row pair per CTA: all threads form the real inputs (the fold of the
// backprojection's partial planes and the step-A epilogue, or a real image), one warp transforms
// z = x_a + i x_b and writes X_a(k), X_b(k), k <= n / 2.
template <int L, int V>
__global__ void __launch_bounds__(ROWS_THREADS)
k_gfft_rows_fwd(const float *in_real, const float *part, int groups, BackprojEpi<float> epi,
                float2 *cbuf, const float2 *__restrict__ tw)
{
    using T = Two<L, V>;
    constexpr int n = T::n, H = T::H;
    __shared__ __align__(16) float s_in[2 * n];
    __shared__ float2 s_buf[T::buf], s_tw[n];
    const int ra = 2 * blockIdx.x;
    stage<n>(s_tw, tw);
    pdl_wait();
    pdl_trigger();
    if (part) {
        for (int e4 = threadIdx.x; e4 < n / 2; e4 += ROWS_THREADS) {
            const int row = ra + (4 * e4 >= n ? 1 : 0), col = 4 * e4 - (4 * e4 >= n ? n : 0);
            const float4 acc = orbit_fold4(part, groups, n, row, col);
            float *dst = s_in + 4 * e4;
            dst[0] = bp_epilogue_value(epi, n, row, col, acc.x);
            dst[1] = bp_epilogue_value(epi, n, row, col + 1, acc.y);
            dst[2] = bp_epilogue_value(epi, n, row, col + 2, acc.z);
            dst[3] = bp_epilogue_value(epi, n, row, col + 3, acc.w);
        }
    } else {
        const float4 *src = reinterpret_cast<const float4 *>(in_real + (size_t)ra * n);
        for (int e4 = threadIdx.x; e4 < n / 2; e4 += ROWS_THREADS) reinterpret_cast<float4 *>(s_in)[e4] = src[e4];
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    float2 v[V], w[L];
    if (lane < L) {
#pragma unroll
        for (int m = 0; m < V; ++m) v[m] = make_float2(s_in[lane + L * m], s_in[n + lane + L * m]);
    }
    two_fwd<L, V>(v, w, lane, s_buf, s_tw);
    if (lane < V) {
#pragma unroll
        for (int k = 0; k < L; ++k) s_buf[lane + V * k] = w[k];           // natural order
    }
    __syncwarp();
    float2 *xa_row = cbuf + (size_t)ra * H, *xb_row = xa_row + H;
    for (int k = lane; k < H; k += 32) {
        const float2 z = s_buf[k], zm = s_buf[k == 0 ? 0 : n - k];
        xa_row[k] = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
        xb_row[k] = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
    }
}

// Column pass: one warp per stored column, forward, times the real symbol, inverse.
template <int L, int V>
__global__ void __launch_bounds__(32 * COL_WARPS)
k_gfft_cols(float2 *cbuf, const float *__restrict__ sym, const float2 *__restrict__ tw)
{
    using T = Two<L, V>;
    constexpr int n = T::n, H = T::H;
    __shared__ float2 s_buf[COL_WARPS][T::buf], s_tw[n];
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31, c = blockIdx.x * COL_WARPS + q;
    stage<n>(s_tw, tw);
    pdl_wait();
    pdl_trigger();
    float2 v[V], w[L];
    float sy[L];
    const bool live = c < H;
    if (live && lane < L) {
#pragma unroll
        for (int m = 0; m < V; ++m) v[m] = cbuf[(size_t)(lane + L * m) * H + c];
    }
    if (live && lane < V) {
#pragma unroll
        for (int k = 0; k < L; ++k) sy[k] = __ldg(sym + (size_t)(lane + V * k) * n + c);
    }
    __syncthreads();
    if (!live) return;
    two_fwd<L, V>(v, w, lane, s_buf[q], s_tw);
    if (lane < V) {
#pragma unroll
        for (int k = 0; k < L; ++k) {
            w[k].x *= sy[k];
            w[k].y *= sy[k];
        }
    }
    two_inv<L, V>(w, v, lane, s_buf[q], s_tw);
    if (lane < L) {
#pragma unroll
        for (int m = 0; m < V; ++m) cbuf[(size_t)(lane + L * m) * H + c] = v[m];
    }
}

// Inverse row pass: one warp per row pair, Z = X_a + i X_b, real part -> row 2c, imaginary part
// -> row 2c + 1 (mode 0: out = v; mode 1: out += v; dout = v).
template <int L, int V>
__global__ void __launch_bounds__(32 * INV_WARPS)
k_gfft_rows_inv(const float2 *cbuf, const float2 *__restrict__ tw, float *out, int mode, float *dout)
{
    using T = Two<L, V>;
    constexpr int n = T::n, H = T::H;
    __shared__ float2 s_buf[INV_WARPS][T::buf], s_tw[n];
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31, ra = 2 * (blockIdx.x * INV_WARPS + q);
    stage<n>(s_tw, tw);
    pdl_wait();
    pdl_trigger();
    const bool live = ra < n;
    const float2 *xa_row = cbuf + (size_t)ra * H, *xb_row = xa_row + H;
    const size_t ga = (size_t)ra * n, gb = ga + n;
    float2 w[L], v[V];
    float pa[V], pb[V];
    if (live && lane < V) {
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const int k = lane + V * i;
            const bool lo = k <= n / 2;
            float2 xa = xa_row[lo ? k : n - k], xb = xb_row[lo ? k : n - k];
            if (!lo) {
                xa.y = -xa.y;
                xb.y = -xb.y;
            }
            w[i] = make_float2(xa.x - xb.y, xa.y + xb.x);
        }
    }
    if (live && lane < L) {
#pragma unroll
        for (int m = 0; m < V; ++m) {
            pa[m] = mode == 1 ? out[ga + lane + L * m] : 0.f;
            pb[m] = mode == 1 ? out[gb + lane + L * m] : 0.f;
        }
    }
    __syncthreads();
    if (!live) return;
    two_inv<L, V>(w, v, lane, s_buf[q], s_tw);
    if (lane >= L) return;
#pragma unroll
    for (int m = 0; m < V; ++m) {
        const int j = lane + L * m;
        if (dout) {
            dout[ga + j] = v[m].x;
            dout[gb + j] = v[m].y;
        }
        out[ga + j] = v[m].x + pa[m];
        out[gb + j] = v[m].y + pb[m];
    }
}

template <int L, int V>
ctr_status launch_two(bool pdl, const float *in_real, const float *part, int groups, const BackprojEpi<float> &epi, float2 *cb,
                      const float *sym, const float2 *tw, float *out, int mode, float *dout, cudaStream_t s)
{
    using T = Two<L, V>;
    launch_pdl(pdl, k_gfft_rows_fwd<L, V>, dim3(T::n / 2), dim3(ROWS_THREADS), 0, s, in_real, part, groups, epi, cb, tw);
    CTR_CHECK_LAUNCH("k_gfft_rows_fwd");
    launch_pdl(pdl, k_gfft_cols<L, V>, dim3((T::H + COL_WARPS - 1) / COL_WARPS), dim3(32 * COL_WARPS), 0, s, cb, sym, tw);
    CTR_CHECK_LAUNCH("k_gfft_cols");
    launch_pdl(pdl, k_gfft_rows_inv<L, V>, dim3((T::n / 2 + INV_WARPS - 1) / INV_WARPS), dim3(32 * INV_WARPS), 0, s,
               (const float2 *)cb, tw, out, mode, dout);
    CTR_CHECK_LAUNCH("k_gfft_rows_inv");
    return CTR_OK;
}

}  // namespace

// Every n = 2^a 3^b from 64 to 864 that is a multiple of 4 (16-byte rows), but for 256 and 512,
// which fft.cu's warp-level passes take.  Smaller and larger sizes and the odd multiples of 2
// keep the CTA-level passes; n = 972 has no factorisation with both factors within a warp.
#define CTR_GFFT_SIZES(X)                                                                                     \
    X(8, 8) X(9, 8) X(12, 8) X(12, 9) X(16, 8) X(12, 12) X(16, 12) X(18, 12) X(18, 16) X(18, 18) X(24, 16) \
    X(24, 18) X(24, 24) X(27, 24) X(32, 24) X(32, 27)

bool gfft_supported(int n)
{
#define CTR_GFFT_HAS(L, V) if (n == L * V) return true;
    CTR_GFFT_SIZES(CTR_GFFT_HAS)
    return false;
}

ctr_status launch_gfft(bool pdl, int n, const float *in_real, const float *part, int groups, const BackprojEpi<float> &epi,
                       float2 *cb, const float *sym, const float2 *tw, float *out, int mode, float *dout,
                       cudaStream_t s)
{
#define CTR_GFFT_RUN(L, V) \
    if (n == L * V) return launch_two<L, V>(pdl, in_real, part, groups, epi, cb, sym, tw, out, mode, dout, s);
    CTR_GFFT_SIZES(CTR_GFFT_RUN)
    return fail(CTR_EUNSUPPORTED, "no two-stage transform of this size");
}

}  // namespace ctr
