// The symmetric path of FP64 plans (OrbitJob in units of 2^-F bins, F <= 51): included by
// radon.cu, inside its unnamed namespace.
//
// GB300 has two FP64 lanes per SM and cycle, so the FP64 operations per sample are what counts.
// The per-angle kernels spend four or more on each (pixel, angle) -- the conversion of the
// fraction, its scaling, the interpolation, the sum -- and twice that where the forward
// projector tests two candidate pixels.  Here a job's weight is formed once for its NC angles,
// from the integer's own bits (no FP64 operation), and a sample costs two operations in R_h^*
// and three in R_h.  256^2 / 360 views, R_h + R_h^*: 645 us with the per-angle kernels, 376 us
// (FP64 pipe: 87 of 117 us in R_h^*, about 150 of 230 in R_h with the slots beside the image).

// frac(p) in [0, 1) from P mod 2^F
__device__ __forceinline__ double frac64(unsigned long long P, int F)
{
    return __longlong_as_double((long long)(((P << (64 - F)) >> 12) | 0x3FF0000000000000ull)) - 1.0;
}

// ---------------------------------------------------------------------------
// R_h^*: a CTA of 64 threads owns a 16 x 16 tile of canonical pixels and one group of jobs;
// each thread owns 4 pixels (rows i0 + ty + 4 r).  The NC channels' (g_b, g_{b+1} - g_b) of the
// tile's bins are staged in shared memory per chunk of jobs.  Small tiles, because a small
// image has to be spread over 152 SMs: 64^2 / 90 views 64 us on 8 CTAs, 10 us on 128.
// ---------------------------------------------------------------------------
constexpr int S64_TILE = 16, S64_THREADS = 64, S64_R = 4, S64_JCH = 8;
constexpr int S64_WIN = 26;   // staged bins per job: 15 (C + S) <= 21.3, and the rounding of both ends

struct Sym64Args {
    const OrbitJob *jobs;
    int n, M, F, groups;
    int list[3];            // first job of each list, and the end (NC = 4: one list)
};

template <int NC>
__global__ void __launch_bounds__(S64_THREADS)
k_backproject_sym64(const double *g, Sym64Args a, double *__restrict__ part)
{
    __shared__ double2 s_bin[S64_JCH][NC][S64_WIN];
    __shared__ long long s_P[S64_JCH], s_C[S64_JCH], s_S[S64_JCH];
    __shared__ int s_k[S64_JCH];
    __shared__ int s_l[S64_JCH][NC];
    pdl_wait();
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int i0 = blockIdx.y * S64_TILE, j0 = blockIdx.x * S64_TILE, n = a.n;
    const size_t nn = (size_t)n * n;
    double *pg = part + (size_t)blockIdx.z * 4 * nn;
#pragma unroll 1
    for (int li = 0; li < 4 / NC; ++li) {
        const int first = li == 0 ? a.list[0] : a.list[1], len = (li == 0 ? a.list[1] : a.list[2]) - first;
        const int per = (len + a.groups - 1) / a.groups;
        const int la = first + min(len, (int)blockIdx.z * per), lb = first + min(len, ((int)blockIdx.z + 1) * per);
        double acc[S64_R][NC];
#pragma unroll
        for (int r = 0; r < S64_R; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[r][c] = 0.0;
        for (int c0 = la; c0 < lb; c0 += S64_JCH) {
            const int na = min(S64_JCH, lb - c0);
            __syncthreads();
            if (tid < na) {
                const AngleMarch am = a.jobs[c0 + tid].am;
                const long long P = (long long)i0 * am.A + (long long)j0 * am.B + am.Op, k = P >> a.F;   // A, B >= 0
                s_P[tid] = P - (k << a.F);
                s_k[tid] = (int)k;
                s_C[tid] = am.A;
                s_S[tid] = am.B;
            }
            if (tid < na * NC) s_l[tid / NC][tid % NC] = a.jobs[c0 + tid / NC].l[li * NC + tid % NC];
            __syncthreads();
            for (int e = tid; e < na * NC * S64_WIN; e += S64_THREADS) {
                const int w = e % S64_WIN, jc = e / S64_WIN, jt = jc / NC, c = jc - jt * NC;
                const int l = s_l[jt][c], k = s_k[jt] + w;
                const double *row = g + (size_t)(l < 0 ? 0 : l) * a.M;
                const double g0 = l >= 0 && k >= 0 && k < a.M ? row[k] : 0.0;
                const double g1 = l >= 0 && k + 1 >= 0 && k + 1 < a.M ? row[k + 1] : 0.0;
                s_bin[jt][c][w] = make_double2(g0, g1 - g0);
            }
            __syncthreads();
            for (int t = 0; t < na; ++t) {
                const long long C = s_C[t];
                long long P = s_P[t] + (long long)ty * C + (long long)tx * s_S[t];
#pragma unroll
                for (int r = 0; r < S64_R; ++r) {
                    const int b = (int)(P >> a.F);
                    const double f = frac64((unsigned long long)P, a.F);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const double2 q = s_bin[t][c][b];
                        acc[r][c] += fma(f, q.y, q.x);
                    }
                    P += 4 * C;
                }
            }
        }
        // partial planes [group][v] in the layout of orbit_fold: 0 and 1 as they are, 2 and 3 transposed
#pragma unroll
        for (int r = 0; r < S64_R; ++r) {
            const int i = i0 + ty + 4 * r, j = j0 + tx;
            if (i >= n || j >= n) continue;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int v = li * NC + c;
                pg[(size_t)v * nn + (v < 2 ? (size_t)i * n + j : (size_t)j * n + i)] = acc[r][c];
            }
        }
    }
    pdl_trigger();
}

// ---------------------------------------------------------------------------
// R_h: the slot form of orbit.cuh with 32 slots per warp (one per lane), one job per CTA and
// four warps that split its rows.  z is formed from x's bits and one addition; max(z, 0) and
// max(-z, 0) by masking on the sign bit.
// ---------------------------------------------------------------------------
constexpr int F64_LANES = 32, F64_PAD = F64_LANES + 8, F64_SEGS = 4;
constexpr int f64_pitch(int n) { return n + 2 * F64_PAD; }

__global__ void __launch_bounds__(256)
k_orbit_image64(const double *u, double *ubar, int n)
{
    __shared__ double tC[32][33], tD[32][33];
    pdl_wait();
    pdl_trigger();
    const int pitch = n + 2 * F64_PAD;
    const size_t plane = (size_t)pitch * n;
    double2 *ub = reinterpret_cast<double2 *>(ubar) + F64_PAD;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, q0 = blockIdx.x * 32, m0 = blockIdx.y * 32;
    for (int r = ty; r < 32; r += 8) {
        const int qr = q0 + r, mc = m0 + tx;          // rows q, columns m, transposed below
        if (qr < n && mc < n) {
            tC[r][tx] = u[(size_t)qr * n + mc];
            tD[r][tx] = u[(size_t)(n - 1 - qr) * n + mc];
        }
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int m = m0 + r, q = q0 + tx;
        if (m >= n || q >= n) continue;
        const size_t o = (size_t)m * pitch + q;
        ub[o] = make_double2(tC[tx][r], tD[tx][r]);
        ub[plane + o] = make_double2(u[(size_t)m * n + q], u[(size_t)(n - 1 - m) * n + q]);
    }
}

__device__ __forceinline__ double pos64(double z)
{
    const long long b = __double_as_longlong(z);
    return __longlong_as_double(b & ~(b >> 63));
}

// (ALONE: the instances of plain projections, mode 0.  A solver's carry no call of bin_alone: the
// preconditioner spreads such values anyway, and 64^2 / 90 views lose 5 % of an iteration to it)
template <int NC, bool ALONE>
__global__ void __launch_bounds__(32 * F64_SEGS)
k_forward_sym64(const double *ubar, Sym64Args a, ForwardEpi<double> epi)
{
    constexpr int LN = F64_LANES, NT = 32 * F64_SEGS;
    __shared__ double s_part[F64_SEGS][NC][3 * LN];   // the slots' sums for bins c, c + 1, c - 1
    __shared__ int s_first[LN + 4];
    pdl_wait();
    const int seg = threadIdx.x >> 5, lane = threadIdx.x & 31, jb = blockIdx.y, F = a.F;
    const int half = NC == 4 || jb < a.list[1] ? 0 : 2;
    const long long one = 1ll << F;
    const AngleMarch am = a.jobs[jb].am;
    const long long A = am.A, B = am.B;
    const int nb = (int)((LN * A) >> F) - 1, kb = blockIdx.x * nb;
    if (kb >= a.M) return;                            // CTA-uniform
    const long long K0 = (long long)(kb - 1) << F;
    const float ulp = __int_as_float((127 - F) << 23);                       // 2^-F
    const float Q0 = (float)(K0 - am.Op) * ulp * am.kA;
    int mlo, mhi;
    rows_in<true>(Q0, am.binv, -(float)LN - 1.f, (float)a.n + 1.f, a.n, mlo, mhi);
    if (mlo <= mhi) {
        const int per = (mhi - mlo + F64_SEGS) / F64_SEGS;
        mlo += seg * per;
        mhi = min(mhi, mlo + per - 1);
    }
    double S[NC], Pp[NC], Nn[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) S[c] = Pp[c] = Nn[c] = 0.0;
    if (mlo <= mhi) {
        int q = (int)ceilf(Q0 - (float)mlo * ((float)B / (float)A));
        long long x = (long long)q * A + (long long)mlo * B + am.Op - K0;
        while (x < 0) { x += A; ++q; }                // (the estimate is off by one at most)
        while (x >= A) { x -= A; --q; }
        const long long bound = A - B;                // x + B >= A: the next row's first pixel moves left
        const long long y = (long long)lane * A, c = (y + one - 1) >> F;
        const double phi1 = (double)(y - (c << F)) * ldexp(1.0, -F) - 1.0;   // phi - 1, added to 1 + x
        const int pitch = a.n + 2 * F64_PAD;
        const size_t plane = (size_t)pitch * a.n;
        const double2 *ub = reinterpret_cast<const double2 *>(ubar) + (half ? plane : 0) + F64_PAD + lane;
        int off = mlo * pitch + q;
#pragma unroll 4
        for (int m = mlo; m <= mhi; ++m) {
            double v[NC];
#pragma unroll
            for (int h = 0; h < NC / 2; ++h) {
                const double2 w = ub[h * plane + off];
                v[2 * h] = w.x;
                v[2 * h + 1] = w.y;
            }
            // x = 2^F only for x in [0, A), A <= 2^F: 1 + x is a double's mantissa
            const double z = __longlong_as_double((long long)(((unsigned long long)x << (52 - F)) | 0x3FF0000000000000ull)) + phi1;
            const double wp = pos64(z), wn = pos64(-z);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                S[k] += v[k];
                Pp[k] = fma(wp, v[k], Pp[k]);
                Nn[k] = fma(wn, v[k], Nn[k]);
            }
            const bool step = x >= bound;
            x += step ? B - A : B;
            off += step ? pitch - 1 : pitch;
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        double *q = s_part[seg][c] + lane;
        q[0] = S[c] - Pp[c] - Nn[c];
        q[LN] = Pp[c];
        q[2 * LN] = Nn[c];
    }
    if (seg == 0) {
        for (int e = lane; e < LN + 4; e += 32) s_first[e] = LN;
        __syncwarp();
        const int c = (int)((lane * A + one - 1) >> F), cp = (int)(((lane - 1) * A + one - 1) >> F);
        if (lane == 0 || c > cp) s_first[c] = lane;   // A <= 1: no centre is skipped
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NC * 3 * LN; e += NT) {
        const int c = e / (3 * LN), q = e - c * (3 * LN);
        double v = s_part[0][c][q];
#pragma unroll
        for (int z = 1; z < F64_SEGS; ++z) v += s_part[z][c][q];
        s_part[0][c][q] = v;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < NC * LN; it += NT) {
        const int c = it / LN, b = it % LN, k = kb + b, l = a.jobs[jb].l[half + c];
        if (b >= nb || k >= a.M || l < 0) continue;
        const double *acc = s_part[0][c];
        double g = 0.0;
        for (int q = s_first[b]; q < s_first[b + 1]; ++q) g += acc[LN + q];
        for (int q = s_first[b + 1]; q < s_first[b + 2]; ++q) g += acc[q];
        for (int q = s_first[b + 2]; q < s_first[b + 3]; ++q) g += acc[2 * LN + q];
        if constexpr (ALONE)
            if (!isfinite(g)) {                       // three bins per slot: see bin_alone
                const int pitch = f64_pitch(a.n), v = half + c;
                const double *pix = ubar + 2 * ((size_t)(v >> 1) * pitch * a.n + F64_PAD) + (v & 1);
                g = bin_alone<double>(pix, pitch, a.n, a.jobs[jb].am.A, a.jobs[jb].am.B, a.jobs[jb].am.Op, F, k);
            }
        forward_epilogue<double>(epi, (size_t)l * a.M + k, g);
    }
    pdl_trigger();
}

Sym64Args sym64_args(const ctr_plan *p)
{
    return Sym64Args{p->d_jobs, p->n, p->M, p->F, p->bp_groups, {p->job_list[0], p->job_list[1], p->job_list[2]}};
}

ctr_status launch_backproject_sym64(const ctr_plan *p, const double *g, cudaStream_t s)
{
    p->launches++;
    const int tiles = (p->n + S64_TILE - 1) / S64_TILE;
    const dim3 grid(tiles, tiles, p->bp_groups);
    // launched early, several CTAs per SM would crowd on those SMs that the kernel ahead leaves
    // first, and FP64 work does not move (128^2: 144 us an iteration against 118)
    launch_pdl(p->pdl != 0 && grid.x * grid.y * grid.z <= 152, p->pair_jobs ? k_backproject_sym64<2> : k_backproject_sym64<4>, grid, dim3(S64_THREADS), 0, s, g,
               sym64_args(p), (double *)p->bp_part);
    CTR_CHECK_LAUNCH("k_backproject_sym64");
    return CTR_OK;
}

ctr_status launch_forward_sym64(const ctr_plan *p, const double *u, const ForwardEpi<double> &epi, cudaStream_t s)
{
    p->launches += 2;
    const dim3 tiles((p->n + 31) / 32, (p->n + 31) / 32);
    launch_pdl(p->pdl != 0, k_orbit_image64, tiles, dim3(256), 0, s, u, (double *)p->ubar, p->n);
    CTR_CHECK_LAUNCH("k_orbit_image64");
    const dim3 grid(p->fwd_chunks, p->n_jobs);
    auto kern = p->pair_jobs ? (epi.mode == 0 ? k_forward_sym64<2, true> : k_forward_sym64<2, false>)
                             : (epi.mode == 0 ? k_forward_sym64<4, true> : k_forward_sym64<4, false>);
    launch_pdl(p->pdl != 0 && grid.x * grid.y <= 152, kern, grid, dim3(32 * F64_SEGS), 0, s, (const double *)p->ubar,
               sym64_args(p), epi);
    CTR_CHECK_LAUNCH("k_forward_sym64");
    return CTR_OK;
}
