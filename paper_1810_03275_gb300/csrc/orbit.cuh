// Kernels of the projectors' symmetric path (OrbitJob): included by radon.cu, inside its
// unnamed namespace.
//
// Both operands are kept in planes of two channels (float2): channels {0, 1} and {2, 3} of a job.
// On GB300 an 8-byte shared-memory or L1 load of a warp's 32 distinct records takes 2 cycles of
// an SM, a 16-byte one takes 8 (measured; 64 bytes per cycle instead of 128), so two planes cost
// half of what one array of float4 does.  NC = 4: plans whose jobs hold up to four angles, both
// planes read together.  NC = 2: pair plans (odd view counts), each job has one plane; the jobs of
// channels {0, 1} come first, then those of {2, 3}.
//
// The sinogram operand of the backprojection lives in *orbit layout*: NC / 2 rows per job, bin by
// bin, zero-padded on both sides far enough that every tile's window of bins lies inside the row.

// NC channel values and their packed arithmetic.
template <int NC> struct Vec;
template <> struct Vec<4> {
    float2 a, b;
};
template <> struct Vec<2> {
    float2 a;
};
__device__ __forceinline__ Vec<4> vzero(Vec<4> *) { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ Vec<2> vzero(Vec<2> *) { return {make_float2(0.f, 0.f)}; }
// the record at p in the first plane, `plane` records further in the second
template <int NC> __device__ __forceinline__ Vec<NC> vload(const float2 *p, int plane)
{
    if constexpr (NC == 4) return {p[0], p[plane]};
    else return {p[0]};
}
__device__ __forceinline__ Vec<4> vadd(Vec<4> x, Vec<4> y) { return {fadd2(x.a, y.a), fadd2(x.b, y.b)}; }
__device__ __forceinline__ Vec<2> vadd(Vec<2> x, Vec<2> y) { return {fadd2(x.a, y.a)}; }
__device__ __forceinline__ Vec<4> vsub(Vec<4> x, Vec<4> y) { return {fsub2(x.a, y.a), fsub2(x.b, y.b)}; }
__device__ __forceinline__ Vec<2> vsub(Vec<2> x, Vec<2> y) { return {fsub2(x.a, y.a)}; }
// w x + y
__device__ __forceinline__ Vec<4> vfma(float w, Vec<4> x, Vec<4> y)
{
    const float2 w2 = make_float2(w, w);
    return {ffma2(w2, x.a, y.a), ffma2(w2, x.b, y.b)};
}
__device__ __forceinline__ Vec<2> vfma(float w, Vec<2> x, Vec<2> y)
{
    return {ffma2(make_float2(w, w), x.a, y.a)};
}
__device__ __forceinline__ float2 vplane(const Vec<4> &v, int h) { return h == 0 ? v.a : v.b; }
__device__ __forceinline__ float2 vplane(const Vec<2> &v, int) { return v.a; }
__device__ __forceinline__ float vget(const Vec<4> &v, int c) { return c == 0 ? v.a.x : c == 1 ? v.a.y : c == 2 ? v.b.x : v.b.y; }
__device__ __forceinline__ float vget(const Vec<2> &v, int c) { return c == 0 ? v.a.x : v.a.y; }

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool valid)   // zero where not valid
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// ---------------------------------------------------------------------------
// g (N x M, FP32 or bfloat16) into orbit layout: one thread per (job, bin).  The pads and the
// channels without an angle keep the zeros they got when the plan was made.
// ---------------------------------------------------------------------------
template <typename S, int NC>
__global__ void __launch_bounds__(256)
k_orbit_sino(const S *g, int M, int list1, int pitch, int pad,
             const OrbitJob *__restrict__ jobs, float *__restrict__ bar)
{
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * 256 + threadIdx.x;
    const int j = blockIdx.y;
    if (k >= M) return;
    const int4 ls = *reinterpret_cast<const int4 *>(jobs[j].l);
    const int half = NC == 4 || j < list1 ? 0 : 2;
    const int l[4] = {ls.x, ls.y, ls.z, ls.w};
    float2 *row = reinterpret_cast<float2 *>(bar) + (size_t)j * (NC / 2) * pitch + pad + k;
#pragma unroll
    for (int h = 0; h < NC / 2; ++h) {
        const int la = half ? l[2] : l[2 * h], lb = half ? l[3] : l[2 * h + 1];
        row[(size_t)h * pitch] = make_float2(la >= 0 ? ldv(g + (size_t)la * M + k) : 0.f,
                                             lb >= 0 ? ldv(g + (size_t)lb * M + k) : 0.f);
    }
}

// ---------------------------------------------------------------------------
// Symmetric backprojection.  A CTA of 4 warps owns a 32 x 32 tile of canonical pixels and
// one group of jobs; every thread owns a block of 2 (along i) x 4 (along j) pixels.
//
// Along such a block the detector coordinate moves by at most about two bins, so the block's
// eight linear interpolations of one job are one piecewise-linear function with few knots:
// with f in [0, 1) the block centre's position in its bin b, a pixel at offset o from the
// centre (o = +-C/2 + {-3, -1, 1, 3} S/2) takes
//     g_b + (f + o) d_b + max(f + o - 1, 0) (d_{b+1} - d_b) + max(-f - o, 0) (d_b - d_{b-1}),
// d_b = g_{b+1} - g_b (and the next knot on either side where o can pass it).  The first two
// terms are linear in o, so their sums over the jobs are kept once per block (A, and L0, L3
// for two of the offsets); a pixel adds only its knot, and half of the pixels meet only the
// right knot, half only the left.  Per block, job and channel that is 12 fused multiply-adds
// and 5 differences for 8 pixels, and 4 shared-memory bins, where an interpolation per pixel
// takes 24 operations and 16 bins.  One R_h^* call, 500^2 / 725 views (pair jobs): 85.6 us with an
// interpolation per pixel, 39.7 us; 2048^2 / 2048 views: 2280 us, 980 us
// (951 of 975 us this kernel: shared-memory pipe 76 % of its peak, FMA pipe 70 %, issue 62 %, and
// the packed fma.f32x2 on three distinct register pairs issues every third cycle: about 130 of
// the 141 cycles a warp and job take on a scheduler).
//
// offsets e0 = (C + 3S)/2, e1 = (C + S)/2, e2 = (C - S)/2, e3 = (C - 3S)/2: pixel (1, 3 - k)
// sits at +e_k and pixel (0, k) at -e_k.  Jobs with 3 S <= C ("flat") have 0 <= e_k < 1:
// four bins b - 1 .. b + 2.  The others have e3 < 0 (those two pixels swap knots) and e0 up
// to 1.42 (two more knots, bins b - 2 .. b + 3).  The jobs of a list are sorted by S / C, so
// each chunk is a run of flat jobs and a run of steep ones.
//
// A pixel's terms of bins that it does not interpolate from cancel only up to rounding: a bin leaves
// up to 2^-22 of its value (as much as a weight's own rounding) in the other pixels of the blocks
// whose bins b - 2 .. b + 3 hold it.
//
// Bank conflicts: an 8-byte load is served sixteen lanes at a time; they hold 8 x 2 blocks,
// whose bins span 14 C + 4 S <= 14.6 plus one: distinct or equal modulo sixteen.
// ---------------------------------------------------------------------------
constexpr int OBP_THREADS = 128;
constexpr int OBP_JCH = 16;    // jobs per staged chunk (two buffers)
constexpr int OBP_TJ = 128;    // jobs per table block (one per thread)

// Up to this image size a call stages the sinogram's rows itself instead of having them brought
// into orbit layout by a kernel of their own (one R_h^* call, 64^2 / 90 views: 12.9 us with it, 9.8
// without; 256^2 / 360: 14.0, 13.4; 384^2 / 480: 19.5, 20.2; pair jobs 256^2 / 361: 14.5, 15.2)
constexpr int obp_direct_n(bool pairs) { return pairs ? 192 : 256; }
constexpr int OBP_WIN = 52;    // bins per staged row (obp_window's most: floor(30 C + 28 S) <= 41, + 9)

// One CTA's inputs (also built from a SliceDesc by the batched stage).
struct ObpArgs {
    const float *bar;       // sinogram in orbit layout
    const OrbitJob *jobs;
    float *part;            // partial planes [group][v][row][col]
    int n, pitch, pad, win; // row pitch and left pad in bins; staged bins per row
    int groups;
    int list[3];            // first job of each list, and the end (NC = 4: one list)
    const float *g;         // if set: the sinogram itself (N x M), staged from its rows instead of bar
    int M;
};

struct ObpTables {
    uint4 *pos;    // {low, high word of the centre of the tile's first block in 2^-31 bins, C, S in 2^-32 bins}
    float4 *e;     // e0 .. e3
    long long *row;   // first staged bin (element of the orbit layout; of the detector with ObpArgs::g)
    int *flat;     // number of flat jobs of the table block
};

template <int NC, bool STEEP>
__device__ __forceinline__ void obp_job(const float2 *__restrict__ row, uint4 tp, float4 e, int it, int jt,
                                        Vec<NC> &A, Vec<NC> &L0, Vec<NC> &L3, Vec<NC> (&KR)[4], Vec<NC> (&KL)[4])
{
    using V = Vec<NC>;
    // it and jt are even: their halves times C and S count 2^-31 bins
    const unsigned long long P = (((unsigned long long)tp.y << 32) | tp.x) + (unsigned long long)(it >> 1) * tp.z +
                                 (unsigned long long)(jt >> 1) * tp.w;
    const int b = (int)(P >> 31);
    const float f = (float)((unsigned)P & 0x7FFFFFFFu) * 4.656612873077393e-10f;   // 2^-31
    const float fm = f - 1.f;
    const float2 *q = row + b;
    const V g0 = vload<NC>(q, OBP_WIN), g1 = vload<NC>(q + 1, OBP_WIN);
    const V gm = vload<NC>(q - 1, OBP_WIN), g2 = vload<NC>(q + 2, OBP_WIN);
    const V d0 = vsub(g1, g0), d1 = vsub(g2, g1), dm = vsub(g0, gm);
    const V dr = vsub(d1, d0), dl = vsub(d0, dm);
    A = vadd(A, vfma(f, d0, g0));
    L0 = vfma(e.x, d0, L0);
    L3 = vfma(e.w, d0, L3);
    KR[1] = vfma(__saturatef(fm + e.y), dr, KR[1]);
    KL[1] = vfma(__saturatef(e.y - f), dl, KL[1]);
    KR[2] = vfma(__saturatef(fm + e.z), dr, KR[2]);
    KL[2] = vfma(__saturatef(e.z - f), dl, KL[2]);
    if constexpr (!STEEP) {
        KR[0] = vfma(__saturatef(fm + e.x), dr, KR[0]);
        KL[0] = vfma(__saturatef(e.x - f), dl, KL[0]);
        KR[3] = vfma(__saturatef(fm + e.w), dr, KR[3]);
        KL[3] = vfma(__saturatef(e.w - f), dl, KL[3]);
    } else {
        const V g3 = vload<NC>(q + 3, OBP_WIN), gn = vload<NC>(q - 2, OBP_WIN);
        const V dr2 = vsub(vsub(g3, g2), d1), dl2 = vsub(dm, vsub(gm, gn));
        const float wr = fm + e.x, wl = e.x - f;
        KR[0] = vfma(fmaxf(wr, 0.f), dr, KR[0]);
        KL[0] = vfma(fmaxf(wl, 0.f), dl, KL[0]);
        KR[0] = vfma(__saturatef(wr - 1.f), dr2, KR[0]);
        KL[0] = vfma(__saturatef(wl - 1.f), dl2, KL[0]);
        KR[3] = vfma(__saturatef(-e.w - f), dl, KR[3]);
        KL[3] = vfma(__saturatef(fm - e.w), dr, KL[3]);
    }
}

// One pixel of R_h^* over the jobs [la, lb), channel v, from the two bins beside its coordinate in
// each: where the block form gives a value that is not finite.  A block's pixels share four or six
// bins and their differences, so that a NaN or an infinite bin, or differences that overflow, would
// reach pixels that do not interpolate from it.
template <int NC>
__device__ __noinline__ float pixel_alone(const float *bar, const float *g, const OrbitJob *jobs, int M, int pitch, int pad,
                                          int la, int lb, int v, int i, int j)
{
    float acc = 0.f;
    for (int t = la; t < lb; ++t) {
        const AngleMarch am = jobs[t].am;
        const long long P = (long long)i * am.A + (long long)j * am.B + am.Op;
        const int k = (int)(P >> 32), l = jobs[t].l[v];
        if (l < 0) continue;
        const size_t plane = (size_t)t * (NC / 2) + (NC == 4 ? v >> 1 : 0);
        const float *row = g ? g + (size_t)l * M : bar + 2 * (plane * pitch + pad) + (v & 1);
        const int step = g ? 1 : 2;
        const float g0 = (unsigned)k < (unsigned)M ? row[(long long)step * k] : 0.f;
        const float g1 = (unsigned)(k + 1) < (unsigned)M ? row[(long long)step * (k + 1)] : 0.f;
        acc = interp(acc, make_stage(g0, g1), P, 32, 0.0);
    }
    return acc;
}

// ALONE: a plain backprojection; a solver's preconditioner spreads values that are not finite anyway.
template <int NC, bool NAMED, bool ALONE = false>
__device__ __forceinline__ void obp_body(const ObpArgs &a, int bx, int by, int bz)
{
    using V = Vec<NC>;
    constexpr int JROW = NC / 2 * OBP_WIN;                                 // staged records per job
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *buf = reinterpret_cast<float2 *>(smem_raw);                    // [2][OBP_JCH][NC / 2][OBP_WIN]
    ObpTables tb;
    tb.pos = reinterpret_cast<uint4 *>(buf + 2 * OBP_JCH * JROW);
    tb.e = reinterpret_cast<float4 *>(tb.pos + OBP_TJ);
    tb.row = reinterpret_cast<long long *>(tb.e + OBP_TJ);
    tb.flat = reinterpret_cast<int *>(tb.row + OBP_TJ);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = by * 32, j0 = bx * 32;
    // warp: 16 x 16 pixels; sixteen lanes: 16 x 8 pixels
    const int it = (warp & 1) * 16 + (lane & 7) * 2;
    const int jt = (warp >> 1) * 16 + (lane >> 3) * 4;
    const size_t nn = (size_t)a.n * a.n;
    float *pg = a.part + (size_t)bz * 4 * nn;
#pragma unroll 1
    for (int li = 0; li < 4 / NC; ++li) {
        const int first_job = li == 0 ? a.list[0] : a.list[1];
        const int len = (li == 0 ? a.list[1] : a.list[2]) - first_job;
        const int per = (len + a.groups - 1) / a.groups;
        const int la = first_job + min(len, bz * per), lb = first_job + min(len, (bz + 1) * per);
        V A, L0, L3, KR[4], KL[4];
        A = L0 = L3 = vzero((V *)nullptr);
#pragma unroll
        for (int k = 0; k < 4; ++k) KR[k] = KL[k] = A;
#pragma unroll 1
        for (int t0 = la; t0 < lb; t0 += OBP_TJ) {
            const int nt = min(OBP_TJ, lb - t0);
            body_sync<NAMED>();                                            // the tables and buffers are free
            if (tid < nt) {
                const AngleMarch am = a.jobs[t0 + tid].am;                 // canonical P(i, j) = i A + j B + Op
                const long long C = am.A, S = am.B;
                const long long P = (long long)i0 * C + (long long)j0 * S + am.Op + ((C + 3 * S) >> 1);
                const int first = (int)((P >> 32) - 2 + a.pad) & ~1;                // 16-byte aligned
                const unsigned long long base = (unsigned long long)(P - ((long long)(first - a.pad) << 32)) >> 1;
                // (C = 2^32, S = 0 of the axis: one unit less, 15 units of 2^-31 bins over the tile; the first
                // block keeps its bin)
                tb.pos[tid] = make_uint4((unsigned)base, (unsigned)(base >> 32), (unsigned)min(C, 0xFFFFFFFFll), (unsigned)S);
                const float c = (float)C * 2.3283064365386963e-10f, s = (float)S * 2.3283064365386963e-10f;   // 2^-32
                const bool flat = 3 * S <= C;
                // (e3 = 0 up to rounding either way: both forms of the job then agree)
                tb.e[tid] = make_float4(0.5f * c + 1.5f * s, 0.5f * c + 0.5f * s, 0.5f * c - 0.5f * s, 0.5f * c - 1.5f * s);
                tb.row[tid] = a.g ? first - a.pad : (long long)(t0 + tid) * (NC / 2) * a.pitch + first;
                if (tid == 0 && !flat) *tb.flat = 0;
                if (flat) {                                                // sorted by S / C: the last flat job
                    bool next = false;
                    if (tid + 1 < nt) {
                        const AngleMarch nx = a.jobs[t0 + tid + 1].am;
                        next = 3 * nx.B <= nx.A;
                    }
                    if (!next) *tb.flat = tid + 1;
                }
            }
            body_sync<NAMED>();
            const int flat = *tb.flat;
            const int nch = (nt + OBP_JCH - 1) / OBP_JCH;
            const float2 *bar = reinterpret_cast<const float2 *>(a.bar) + 2 * lane;
            auto prefetch = [&](int ch) {                                  // 16 bytes per lane: win <= 64
                const int a0 = ch * OBP_JCH, na = min(OBP_JCH, nt - a0);
                if (a.g) {                                                 // four bytes per lane, zeros off the detector
                    float *dst = reinterpret_cast<float *>(buf + (ch & 1) * (OBP_JCH * JROW));
                    for (int t = warp; t < na; t += OBP_THREADS / 32) {
                        const int4 ls = *reinterpret_cast<const int4 *>(a.jobs[t0 + a0 + t].l);
                        const int l4[4] = {ls.x, ls.y, ls.z, ls.w};
                        const int k0 = (int)tb.row[a0 + t];
                        for (int w = lane; w < a.win; w += 32)
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                const int l = NC == 4 || li == 0 ? l4[c] : l4[2 + (c & 1)];
                                const bool ok = l >= 0 && (unsigned)(k0 + w) < (unsigned)a.M;
                                cp_async4(dst + 2 * (t * JROW + (c >> 1) * OBP_WIN + w) + (c & 1),
                                          ok ? a.g + (size_t)l * a.M + k0 + w : a.g, ok);
                            }
                    }
                    return;
                }
                float2 *dst = buf + (ch & 1) * (OBP_JCH * JROW) + 2 * lane;
                if (2 * lane < a.win)
                    for (int t = warp; t < na; t += OBP_THREADS / 32) {
                        const float2 *src = bar + tb.row[a0 + t];
                        cp_async16(dst + t * JROW, src);
                        if constexpr (NC == 4) cp_async16(dst + t * JROW + OBP_WIN, src + a.pitch);
                    }
            };
            prefetch(0);
            cp_async_commit();
#pragma unroll 1
            for (int ch = 0; ch < nch; ++ch) {
                if (ch + 1 < nch) prefetch(ch + 1);
                cp_async_commit();
                cp_async_wait<1>();                                        // this thread's copies of chunk ch
                body_sync<NAMED>();                                        // everyone's
                const int a0 = ch * OBP_JCH, na = min(OBP_JCH, nt - a0);
                const float2 *rows = buf + (ch & 1) * (OBP_JCH * JROW);
                const int nf = min(max(flat - a0, 0), na);
#pragma unroll 2
                for (int t = 0; t < nf; ++t)
                    obp_job<NC, false>(rows + t * JROW, tb.pos[a0 + t], tb.e[a0 + t], it, jt, A, L0, L3, KR, KL);
#pragma unroll 2
                for (int t = nf; t < na; ++t)
                    obp_job<NC, true>(rows + t * JROW, tb.pos[a0 + t], tb.e[a0 + t], it, jt, A, L0, L3, KR, KL);
                body_sync<NAMED>();                                        // buffer ch & 1 is refilled next
            }
            cp_async_wait<0>();
        }
        // the block's pixels: (1, 3 - k) = A + L_k + KR_k, (0, k) = A - L_k + KL_k, L_k linear in e_k
        const V zero = vzero((V *)nullptr);
        const V L1 = vfma(2.f / 3.f, L0, vfma(1.f / 3.f, L3, zero)), L2 = vfma(1.f / 3.f, L0, vfma(2.f / 3.f, L3, zero));
        const V L[4] = {L0, L1, L2, L3};
        V px[2][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            px[1][3 - k] = vadd(vadd(A, L[k]), KR[k]);
            px[0][k] = vadd(vsub(A, L[k]), KL[k]);
        }
        const int i = i0 + it, j = j0 + jt;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int v = li * NC + c;
            float *pl = pg + (size_t)v * nn;
            if (v < 2) {                                                   // rows i: four adjacent columns
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (i + r >= a.n) continue;
                    float *q = pl + (size_t)(i + r) * a.n + j;
                    if ((a.n & 3) == 0 && j < a.n) {
                        *reinterpret_cast<float4 *>(q) = make_float4(vget(px[r][0], c), vget(px[r][1], c),
                                                                     vget(px[r][2], c), vget(px[r][3], c));
                    } else {
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            if (j + m < a.n) q[m] = vget(px[r][m], c);
                    }
                }
            } else {                                                       // transposed planes: rows j
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (j + m >= a.n) continue;
                    float *q = pl + (size_t)(j + m) * a.n + i;
                    if ((a.n & 1) == 0 && i < a.n) {
                        *reinterpret_cast<float2 *>(q) = make_float2(vget(px[0][m], c), vget(px[1][m], c));
                    } else {
                        if (i < a.n) q[0] = vget(px[0][m], c);
                        if (i + 1 < a.n) q[1] = vget(px[1][m], c);
                    }
                }
            }
        }
        if constexpr (ALONE) {
            V sum = px[0][0];                                              // (not finite if one of them is not)
#pragma unroll
            for (int e = 1; e < 8; ++e) sum = vadd(sum, px[e >> 2][e & 3]);
            bool finite = true;
#pragma unroll
            for (int c = 0; c < NC; ++c) finite = finite && isfinite(vget(sum, c));
            if (finite) continue;
#pragma unroll 1
            for (int e = 0; e < 8 * NC; ++e) {
                const int v = li * NC + (e >> 3), ii = i + ((e >> 2) & 1), jj = j + (e & 3);
                if (ii < a.n && jj < a.n)
                    pg[(size_t)v * nn + (v < 2 ? (size_t)ii * a.n + jj : (size_t)jj * a.n + ii)] =
                        pixel_alone<NC>(a.bar, a.g, a.jobs, a.M, a.pitch, a.pad, la, lb, v, ii, jj);
            }
        }
    }
}

template <int NC, bool ALONE>
__global__ void __launch_bounds__(OBP_THREADS, 5) k_backproject_orbit(ObpArgs a)
{
    pdl_wait();
    obp_body<NC, false, ALONE>(a, blockIdx.x, blockIdx.y, blockIdx.z);
    pdl_trigger();
}

size_t obp_smem(int nc)
{
    return (size_t)2 * OBP_JCH * OBP_WIN * nc * sizeof(float) + OBP_TJ * (sizeof(uint4) + sizeof(float4) + sizeof(long long)) + 16;
}

// the plan's launch arguments
ObpArgs obp_args(const ctr_plan *p, const float *bar)
{
    ObpArgs a{};
    a.bar = bar;
    a.jobs = p->d_jobs;
    a.part = (float *)p->obp_part;
    a.n = p->n;
    a.pitch = p->bar_pitch;
    a.pad = p->bar_pad;
    a.win = p->obp_win;
    a.groups = p->obp_groups;
    a.M = p->M;
    for (int k = 0; k < 3; ++k) a.list[k] = p->job_list[k];
    return a;
}

// R_h at bin k for one channel of the orbit image, from the pixels whose coordinate lies in
// [k, k + 1) and [k - 1, k) alone (pix: the channel of pixel (0, 0); P in 2^-F bins): where the slot
// form gives a value that is not finite.  It meets three bins per slot, so that a NaN or an infinity
// would reach a bin beside the two that its pixel touches (0 times infinity), and infinities of
// both signs could meet in a bin that neither touches.
template <typename T>
__device__ __noinline__ T bin_alone(const T *pix, int pitch, int n, long long A, long long B, long long Op, int F, int k)
{
    const double inv2F = ldexp(1.0, -F);
    T g = T(0);
    for (int iv = 0; iv < 2; ++iv) {
        const long long K = (long long)(k - iv) << F;
        long long q = ceil_div_ll(K - Op, A), P = q * A + Op - K;            // the row's first pixel, P in [0, A)
        T Su = T(0), Sf = T(0);
        for (int m = 0; m < n; ++m) {
            for (int c = 0; c < 2; ++c)
                if (P + c * A < (1ll << F) && q + c >= 0 && q + c < n)
                    acc_sample(Su, Sf, pix[2 * ((long long)m * pitch + q + c)], P + c * A, F, inv2F);
            P += B;                                                          // 0 <= B <= A: one step at most
            if (P >= A) { P -= A; --q; }
        }
        const T Bk = sizeof(T) == 4 ? Sf - Su : Sf;                          // (FP32 sums 1 + frac)
        g += iv == 0 ? Su - Bk : Bk;
    }
    return g;
}

// ---------------------------------------------------------------------------
// Symmetric forward projector.  A warp follows one job's rays down the image rows: lane l
// carries the pixels q0(m) + l and q0(m) + l + 32, where q0(m) is the first pixel of row m
// whose coordinate is at least K0 = kb - 1 (the bin before the CTA's first).  P(q0(m), m) - K0
// = x(m) lies in [0, A) on every row, so pixel slot s (0 <= s < 64) stays within one step
// A <= 1 of s A + K0 and meets three bins only: its centre c = ceil(s A) and the two beside
// it.  With z = x + s A - c in (-1, 1) a pixel adds max(z, 0) u to bin c + 1, max(-z, 0) u to
// bin c - 1 and the rest to bin c; the lane sums u, max(z, 0) u and max(-z, 0) u.  Rounding x
// and s A - c is monotone and alike for both signs, so neither weight is positive where the exact
// one is 0: a bin that no pixel touches comes out as exactly 0 (metal traces rely on it).
// Each pixel of a row is read once by one lane, and x(m) is the same for the whole warp: per
// slot 3 multiply-adds per channel and two for the weights, per row one conversion.
// (Marching one bin per lane instead reads two pixels per row, half of the second ones for
// nothing, and does 4 multiply-adds.)
//
// Every job reads the whole orbit image (760 MB in all at 512^2 and 720 views): a CTA takes
// JOBS adjacent jobs, whose rays nearly coincide, so that they share its lines in L1, and SEGS
// warps per job that split its rows.  The image rows carry zeros on both sides, so no load is
// tested.  A chunk of bins is as wide as the slots cover, [kb, kb + nb), nb = floor(64 A) - 1;
// at the end the slots' three sums are gathered per bin through shared memory, in a fixed order,
// and all of a job's warps share the epilogue.  One R_h call, 512^2 / 720 views: 69.9 us with the
// march per bin, 56.1 us; 2048^2 / 2048 views: 2240 us, 1588 us (with max(-z, 0) u formed at the end from
// u and x u, which left rounding in untouched bins: 54.8 and 1537).  At 2048^2 the L1 pipe is at 67 %
// of its peak, FMA at 62 %, issue 55 %, with 37 % of the warp slots at 80 registers; at 512^2 53, 48 and
// 46 %: load latency.  An 8-byte load of 32 pixels at an unaligned offset takes up to 3 wavefronts.
// Tried and slower: float4 records (512^2 59.8 us when planes took 57.7), the rows staged in shared
// memory by cp.async (86: the copies cost as much as the loads), 32 warps a SM at 64 registers, an L1
// prefetch 12 to 32 rows ahead (no change).
// ---------------------------------------------------------------------------
constexpr int OFW_JOBS = 2, OFW_SEGS = 2, OFW_THREADS = 32 * OFW_JOBS * OFW_SEGS;   // of the batched stage

struct OfwArgs {
    const float *ubar;      // orbit image
    const OrbitJob *jobs;
    int n, M, n_jobs, list1;
};

// ALONE: plain projections (mode 0); a solver's preconditioner spreads such values anyway.
template <int NC, int JOBS, int SEGS, bool NAMED, bool ALONE = false>
__device__ __forceinline__ void ofw_body(const OfwArgs &a, const ForwardEpi<float> &epi, int bx, int by)
{
    using V = Vec<NC>;
    constexpr int STRIPS = OFW_LANES / 32, LN = OFW_LANES;
    constexpr int H = NC / 2, NT = 32 * SEGS;
    __shared__ float2 s_part[JOBS][SEGS][H][3 * LN];   // per plane: the slots' sums for bins c, c + 1, c - 1
    __shared__ int s_first[JOBS][LN + 4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = warp % JOBS, seg = warp / JOBS;
    // the CTA's jobs: groups of JOBS within each list
    const int g0 = (a.list1 + JOBS - 1) / JOBS;
    const int j0 = by < g0 ? by * JOBS : a.list1 + (by - g0) * JOBS;
    const int nj = min(JOBS, (by < g0 ? a.list1 : a.n_jobs) - j0), jb = j0 + slot;
    const int half = NC == 4 || by < g0 ? 0 : 2;      // (pair plans: the list's channels)
    // chunk width: the narrowest of the CTA's jobs, so that their bins coincide
    long long amin = 1ll << 32;
#pragma unroll
    for (int q = 0; q < JOBS; ++q)
        if (q < nj) amin = min(amin, a.jobs[j0 + q].am.A);
    const int nb = (int)((LN * amin) >> 32) - 1;
    const int kb = bx * nb;
    if (kb >= a.M) return;                            // CTA-uniform
    const bool active = slot < nj;                    // warp-uniform
    V S[STRIPS], Pp[STRIPS], Nn[STRIPS];              // sums of u, max(z, 0) u and max(-z, 0) u
#pragma unroll
    for (int t = 0; t < STRIPS; ++t) S[t] = Nn[t] = Pp[t] = vzero((V *)nullptr);
    const AngleMarch am = a.jobs[active ? jb : j0].am;
    const long long A = am.A, B = am.B, K0 = (long long)(kb - 1) << 32;
    // rows on which a slot may lie in the image, rounded out: q0(m) stays within [-66, n + 3]
    // there, inside the pads (the estimate is off by far less than a pixel: |Q0| < 2^14 wherever
    // a row meets the image)
    const float Q0 = (float)(K0 - am.Op) * (am.kA * 2.3283064365386963e-10f);
    int mlo, mhi;
    rows_in<true>(Q0, am.binv, -(float)LN - 1.f, (float)a.n + 1.f, a.n, mlo, mhi);
    if (SEGS > 1 && mlo <= mhi) {                     // this warp's part of the rows
        const int per = (mhi - mlo + SEGS) / SEGS;
        mlo += seg * per;
        mhi = min(mhi, mlo + per - 1);
    }
    if (active && mlo <= mhi) {
        int q = (int)ceilf(Q0 - (float)mlo * ((float)B / (float)A));
        long long x = (long long)q * A + (long long)mlo * B + am.Op - K0;
        while (x < 0) { x += A; ++q; }                // (the estimate is off by one at most)
        while (x >= A) { x -= A; --q; }
        // x + B >= A: the next row's first pixel moves left.  The bound A - B is 2^32 only for
        // A = 2^32, B = 0, where x never moves: bound and x are kept one unit lower there
        const unsigned bound = (unsigned)min(A - B, 0xFFFFFFFFll);
        unsigned r = B == 0 ? min((unsigned)x, 0xFFFFFFFEu) : (unsigned)x;
        const unsigned B32 = (unsigned)B, BA32 = (unsigned)(B - A);
        float phi[STRIPS];
#pragma unroll
        for (int t = 0; t < STRIPS; ++t) {
            const long long y = (long long)(lane + 32 * t) * A;
            phi[t] = -(float)(unsigned)(-y) * 2.3283064365386963e-10f;   // y - ceil(y), y in 2^-32 bins
        }
        const int pitch = orbit_pitch(a.n), plane = pitch * a.n;
        const float2 *ub = reinterpret_cast<const float2 *>(a.ubar) + (half ? plane : 0) + ORBIT_PAD + lane;
        const float2 *ub2 = ub + plane;
        int off = mlo * pitch + q;
#pragma unroll 8
        for (int m = mlo; m <= mhi; ++m) {
            V v[STRIPS];
#pragma unroll
            for (int t = 0; t < STRIPS; ++t) {
                v[t].a = ub[off + 32 * t];
                if constexpr (NC == 4) v[t].b = ub2[off + 32 * t];
            }
            const float xf = (float)r;                // x, in 2^-32 bins
#pragma unroll
            for (int t = 0; t < STRIPS; ++t) {
                S[t] = vadd(S[t], v[t]);
                Pp[t] = vfma(__saturatef(fmaf(xf, 2.3283064365386963e-10f, phi[t])), v[t], Pp[t]);
                Nn[t] = vfma(__saturatef(fmaf(xf, -2.3283064365386963e-10f, -phi[t])), v[t], Nn[t]);
            }
            const bool step = r >= bound;
            r += step ? BA32 : B32;
            off += step ? pitch - 1 : pitch;
        }
    }
#pragma unroll
    for (int t = 0; t < STRIPS; ++t) {
        const V mid = vsub(S[t], vadd(Pp[t], Nn[t]));
#pragma unroll
        for (int h = 0; h < H; ++h) {
            float2 *q = s_part[slot][seg][h] + lane + 32 * t;
            q[0] = vplane(mid, h);
            q[LN] = vplane(Pp[t], h);
            q[2 * LN] = vplane(Nn[t], h);
        }
    }
    // the slots of centre v are first[v] .. first[v + 1] - 1
    int *first = s_first[slot];
    if (seg == 0) {
        for (int e = lane; e < LN + 4; e += 32) first[e] = LN;
        __syncwarp();
#pragma unroll
        for (int t = 0; t < STRIPS; ++t) {
            const int q = lane + 32 * t;
            const int c = (int)((q * A + 0xFFFFFFFFll) >> 32), cp = (int)(((q - 1) * A + 0xFFFFFFFFll) >> 32);
            if (q == 0 || c > cp) first[c] = q;       // A <= 1: no centre is skipped
        }
    }
    // from here on the job's NT threads share its bins: one bin and plane each
    const int tj = seg * 32 + lane;
    constexpr int ITEMS = (LN * H + NT - 1) / NT;
    const bool pre = epi.mode == 1 || epi.mode == 2;
    float ops[2][5];                                  // the first item's operands, on their way meanwhile
    auto fetch = [&](int it) {
        const int b = it % LN, h = it / LN, k = kb + b;
        const bool ok = active && it < LN * H && b < nb && k < a.M;
        const float *src[5] = {epi.v1b, epi.dw, epi.da, epi.dlo, epi.dhi};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int l = ok ? a.jobs[jb].l[half + 2 * h + c] : -1;
#pragma unroll
            for (int o = 0; o < 5; ++o) ops[c][o] = l >= 0 ? src[o][(size_t)l * a.M + k] : 0.f;
        }
    };
    if (pre) fetch(tj);
    body_sync<NAMED>();
    if constexpr (SEGS > 1) {
        for (int e = tj; e < 3 * LN * H; e += NT) {
            const int h = e / (3 * LN), q = e - h * (3 * LN);
            float2 v = s_part[slot][0][h][q];
#pragma unroll
            for (int z = 1; z < SEGS; ++z) v = fadd2(v, s_part[slot][z][h][q]);
            s_part[slot][0][h][q] = v;
        }
        body_sync<NAMED>();
    }
    if (!active) return;
    unsigned again = 0;                               // values to form from their own pixels: see bin_alone
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int it = tj + i * NT, b = it % LN, h = it / LN, k = kb + b;
        if (i > 0 && pre) fetch(it);
        if (it >= LN * H || b >= nb || k >= a.M) continue;
        // bin kb + b is centre c = b + 1
        const float2 *acc = s_part[slot][0][h];
        float2 g = make_float2(0.f, 0.f);
        const int q0 = first[b], q1 = first[b + 1], q2 = first[b + 2], q3 = first[b + 3];
        for (int q = q0; q < q1; ++q) g = fadd2(g, acc[LN + q]);
        for (int q = q1; q < q2; ++q) g = fadd2(g, acc[q]);
        for (int q = q2; q < q3; ++q) g = fadd2(g, acc[2 * LN + q]);
        float y[2] = {0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int l = a.jobs[jb].l[half + 2 * h + c];
            if (l < 0) continue;
            float *yd = epi.ybar ? &y[c] : nullptr;
            const float val = c == 0 ? g.x : g.y;
            if (ALONE && !isfinite(val)) again |= 1u << (2 * i + c);
            if (pre)
                forward_epilogue_pre(epi, (size_t)l * a.M + k, val, ops[c][0], ops[c][1], ops[c][2], ops[c][3], ops[c][4], yd);
            else forward_epilogue(epi, (size_t)l * a.M + k, val, yd);
        }
        if (epi.ybar)
            reinterpret_cast<float2 *>(epi.ybar)[((size_t)jb * H + h) * epi.ypitch + epi.ypad + k] = make_float2(y[0], y[1]);
    }
    if constexpr (ALONE) {
        if (again == 0) return;
        const int pitch = orbit_pitch(a.n);
        for (int e = 0; e < 2 * ITEMS; ++e) {
            if (!(again >> e & 1)) continue;
            const int it = tj + (e >> 1) * NT, k = kb + it % LN, v = half + 2 * (it / LN) + (e & 1);
            const float *pix = a.ubar + 2 * ((size_t)(v >> 1) * pitch * a.n + ORBIT_PAD) + (v & 1);
            const OrbitJob &job = a.jobs[jb];
            epi.g[(size_t)job.l[v] * a.M + k] =
                epi.scale * bin_alone<float>(pix, pitch, a.n, job.am.A, job.am.B, job.am.Op, 32, k);
        }
    }
}

// (instances of their own for plain projections: without bin_alone a solver's save 0.5 % of an
// iteration at 512^2)
template <int NC, int JOBS, int SEGS, bool ALONE>
__global__ void __launch_bounds__(32 * JOBS * SEGS, 24 / (JOBS * SEGS))
k_forward_orbit(OfwArgs a, ForwardEpi<float> epi)
{
    pdl_wait();
    // chunks from the detector's middle outwards: the long rays first, the short ones fill the tail
    const int c = blockIdx.z * gridDim.y + blockIdx.y, mid = (gridDim.y * gridDim.z - 1) / 2;
    ofw_body<NC, JOBS, SEGS, false, ALONE>(a, epi, c & 1 ? mid + (c + 1) / 2 : mid - c / 2, blockIdx.x);
    pdl_trigger();
}

// CTA rows of the job lists in groups of `jobs`
int ofw_groups(const ctr_plan *p, int jobs)
{
    return (p->job_list[1] + jobs - 1) / jobs + (p->n_jobs - p->job_list[1] + jobs - 1) / jobs;
}

template <int JOBS, int SEGS>
void launch_forward_orbit_shape(const ctr_plan *p, const float *ub, const ForwardEpi<float> &epi, cudaStream_t s)
{
    // (chunks beyond a grid's 65535 rows, detectors of some millions of bins, go on in z; what is
    // left over there lies beyond the detector)
    const int z = (p->fwd_chunks + 65534) / 65535;
    const dim3 grid(ofw_groups(p, JOBS), (p->fwd_chunks + z - 1) / z, z);
    auto kern = p->pair_jobs
                    ? (epi.mode == 0 ? k_forward_orbit<2, JOBS, SEGS, true> : k_forward_orbit<2, JOBS, SEGS, false>)
                    : (epi.mode == 0 ? k_forward_orbit<4, JOBS, SEGS, true> : k_forward_orbit<4, JOBS, SEGS, false>);
    launch_pdl(p->pdl != 0, kern, grid, dim3(32 * JOBS * SEGS), 0, s,
               OfwArgs{ub, p->d_jobs, p->n, p->M, p->n_jobs, p->job_list[1]}, epi);
}

// The launch shape (jobs * 16 + segments): the one ctr_plan_set_fwd_shape set, else the one
// measured best for the number of (job, chunk) pairs there are: with many, two
// adjacent jobs share their image lines in L1 (four-channel jobs 2048^2: (2, 4) 1588 us, (1, 4)
// 1798; 1024^2 / 1440: 309 and 336; 512^2 with 3077 pairs: 56 either way.  Pair jobs 2048^2 / 2047 views:
// (2, 2) 1965, (1, 4) 2000; 500^2 / 725 with 6171 pairs: 62.1 and 61.4); with few, splitting rows over
// four warps matters more (256^2: (1, 4) 17.5, (2, 2) 25.7).
int ofw_shape(const ctr_plan *p)
{
    if (p->fwd_slots > 0) return p->fwd_slots * 16 + p->fwd_segs;
    const long long pairs = (long long)p->n_jobs * p->fwd_chunks;
    if (p->pair_jobs) return pairs >= 8000 ? 2 * 16 + 2 : 1 * 16 + 4;
    return pairs >= 4000 ? 2 * 16 + 4 : 1 * 16 + 4;
}

void launch_forward_orbit(const ctr_plan *p, const float *ub, const ForwardEpi<float> &epi, cudaStream_t s)
{
    switch (ofw_shape(p)) {
    case 1 * 16 + 2: launch_forward_orbit_shape<1, 2>(p, ub, epi, s); break;
    case 1 * 16 + 8: launch_forward_orbit_shape<1, 8>(p, ub, epi, s); break;
    case 2 * 16 + 2: launch_forward_orbit_shape<2, 2>(p, ub, epi, s); break;
    case 2 * 16 + 4: launch_forward_orbit_shape<2, 4>(p, ub, epi, s); break;
    case 4 * 16 + 2: launch_forward_orbit_shape<4, 2>(p, ub, epi, s); break;
    case 4 * 16 + 1: launch_forward_orbit_shape<4, 1>(p, ub, epi, s); break;
    default: launch_forward_orbit_shape<1, 4>(p, ub, epi, s); break;
    }
}
