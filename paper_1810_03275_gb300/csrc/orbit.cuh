// Kernels of the projectors' symmetric path (OrbitJob): included by radon.cu, inside its
// unnamed namespace.
//
// The sinogram operand of the backprojection lives in *orbit layout*: row j holds, for every
// detector bin, the NC live channels of job j side by side, zero-padded on both sides far
// enough that every tile's window of bins lies inside the row.  NC = 4 for plans whose jobs
// hold up to four angles, 2 for plans of pair jobs (odd view counts; the jobs of channels
// {0, 1} first, then those of {2, 3}).

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
__device__ __forceinline__ Vec<4> vload(const Vec<4> *p)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ Vec<2> vload(const Vec<2> *p) { return {*reinterpret_cast<const float2 *>(p)}; }
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
__device__ __forceinline__ float vget(const Vec<4> &v, int c) { return c == 0 ? v.a.x : c == 1 ? v.a.y : c == 2 ? v.b.x : v.b.y; }
__device__ __forceinline__ float vget(const Vec<2> &v, int c) { return c == 0 ? v.a.x : v.a.y; }

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
k_orbit_sino(const S *__restrict__ g, int M, int n_jobs, int list1, int pitch, int pad,
             const OrbitJob *__restrict__ jobs, float *__restrict__ bar)
{
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * 256 + threadIdx.x;
    const int j = blockIdx.y;
    if (k >= M) return;
    const int4 ls = *reinterpret_cast<const int4 *>(jobs[j].l);
    const size_t o = (size_t)j * pitch + pad + k;
    if constexpr (NC == 4) {
        float4 v;
        v.x = ls.x >= 0 ? ldv(g + (size_t)ls.x * M + k) : 0.f;
        v.y = ls.y >= 0 ? ldv(g + (size_t)ls.y * M + k) : 0.f;
        v.z = ls.z >= 0 ? ldv(g + (size_t)ls.z * M + k) : 0.f;
        v.w = ls.w >= 0 ? ldv(g + (size_t)ls.w * M + k) : 0.f;
        reinterpret_cast<float4 *>(bar)[o] = v;
    } else {
        const int la = j < list1 ? ls.x : ls.z, lb = j < list1 ? ls.y : ls.w;
        float2 v;
        v.x = la >= 0 ? ldv(g + (size_t)la * M + k) : 0.f;
        v.y = lb >= 0 ? ldv(g + (size_t)lb * M + k) : 0.f;
        reinterpret_cast<float2 *>(bar)[o] = v;
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
// and 5 differences for 8 pixels, and 4 shared-memory bins instead of 16, where an
// interpolation per pixel takes 24 operations: the shared-memory pipe bounded that form
// (l1tex 88 %, 8 wavefronts per pixel and warp), the FP32 pipe bounds this one.
//
// offsets e0 = (C + 3S)/2, e1 = (C + S)/2, e2 = (C - S)/2, e3 = (C - 3S)/2: pixel (1, 3 - k)
// sits at +e_k and pixel (0, k) at -e_k.  Jobs with 3 S <= C ("flat") have 0 <= e_k < 1:
// four bins b - 1 .. b + 2.  The others have e3 < 0 (those two pixels swap knots) and e0 up
// to 1.42 (two more knots, bins b - 2 .. b + 3).  The jobs of a list are sorted by S / C, so
// each chunk is a run of flat jobs and a run of steep ones.
//
// Bank conflicts: a 16-byte load is served eight lanes at a time; eight lanes hold 4 x 2
// blocks, whose bins span 6 C + 4 S <= 7.2 plus one: distinct or equal modulo eight.
// ---------------------------------------------------------------------------
constexpr int OBP_THREADS = 128;
constexpr int OBP_JCH = 16;    // jobs per staged chunk (two buffers)
constexpr int OBP_TJ = 128;    // jobs per table block (one per thread)

template <int NC> constexpr int obp_align() { return 4 / NC; }   // bins per 16 bytes

// One CTA's inputs (also built from a SliceDesc by the batched stage).
struct ObpArgs {
    const float *bar;       // sinogram in orbit layout
    const OrbitJob *jobs;
    float *part;            // partial planes [group][v][row][col]
    int n, pitch, pad, win; // row pitch and left pad in bins; staged bins per job
    int groups;
    int list[3];            // first job of each list, and the end (NC = 4: one list)
};

struct ObpTables {
    uint4 *pos;    // {low, high word of the centre of the tile's first block in 2^-31 bins, C, S in 2^-31 bins}
    float4 *e;     // e0 .. e3
    long long *row;   // first staged bin (element of the orbit layout)
    int *flat;     // number of flat jobs of the table block
};

template <int NC, bool STEEP>
__device__ __forceinline__ void obp_job(const Vec<NC> *__restrict__ row, uint4 tp, float4 e, int it, int jt,
                                        Vec<NC> &A, Vec<NC> &L0, Vec<NC> &L3, Vec<NC> (&KR)[4], Vec<NC> (&KL)[4])
{
    using V = Vec<NC>;
    const unsigned long long P = (((unsigned long long)tp.y << 32) | tp.x) + (unsigned long long)it * tp.z +
                                 (unsigned long long)jt * tp.w;
    const int b = (int)(P >> 31);
    const float f = (float)((unsigned)P & 0x7FFFFFFFu) * 4.656612873077393e-10f;   // 2^-31
    const float fm = f - 1.f;
    const V *q = row + b;
    const V g0 = vload(q), g1 = vload(q + 1), gm = vload(q - 1), g2 = vload(q + 2);
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
        const V g3 = vload(q + 3), gn = vload(q - 2);
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

template <int NC, bool NAMED>
__device__ __forceinline__ void obp_body(const ObpArgs &a, int bx, int by, int bz)
{
    using V = Vec<NC>;
    constexpr int AL = obp_align<NC>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *buf = reinterpret_cast<V *>(smem_raw);                              // [2][OBP_JCH][win]
    ObpTables tb;
    tb.pos = reinterpret_cast<uint4 *>(buf + 2 * OBP_JCH * a.win);
    tb.e = reinterpret_cast<float4 *>(tb.pos + OBP_TJ);
    tb.row = reinterpret_cast<long long *>(tb.e + OBP_TJ);
    tb.flat = reinterpret_cast<int *>(tb.row + OBP_TJ);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = by * 32, j0 = bx * 32;
    // warp: 16 x 16 pixels; eight lanes: 8 x 8 pixels
    const int it = (warp & 1) * 16 + ((lane >> 3) & 1) * 8 + (lane & 3) * 2;
    const int jt = (warp >> 1) * 16 + (lane >> 4) * 8 + ((lane >> 2) & 1) * 4;
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
                const int first = (int)((P >> 32) - 2 + a.pad) & ~(AL - 1);
                const unsigned long long base = (unsigned long long)(P - ((long long)(first - a.pad) << 32)) >> 1;
                tb.pos[tid] = make_uint4((unsigned)base, (unsigned)(base >> 32), (unsigned)(C >> 1), (unsigned)(S >> 1));
                const float c = (float)C * 2.3283064365386963e-10f, s = (float)S * 2.3283064365386963e-10f;   // 2^-32
                const bool flat = 3 * S <= C;
                // (e3 = 0 up to rounding either way: both forms of the job then agree)
                tb.e[tid] = make_float4(0.5f * c + 1.5f * s, 0.5f * c + 0.5f * s, 0.5f * c - 0.5f * s, 0.5f * c - 1.5f * s);
                tb.row[tid] = (long long)(t0 + tid) * a.pitch + first;
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
            const int units = a.win / AL;                                  // 16-byte units per job
            auto prefetch = [&](int ch) {
                const int a0 = ch * OBP_JCH, na = min(OBP_JCH, nt - a0);
                V *dst = buf + (size_t)(ch & 1) * OBP_JCH * a.win;
                for (int t = warp; t < na; t += OBP_THREADS / 32) {
                    const float *src = a.bar + (size_t)tb.row[a0 + t] * NC;
                    float *d = reinterpret_cast<float *>(dst + t * a.win);
                    for (int w = lane; w < units; w += 32) cp_async16(d + 4 * w, src + 4 * w);
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
                const V *rows = buf + (size_t)(ch & 1) * OBP_JCH * a.win;
                const int nf = min(max(flat - a0, 0), na);
#pragma unroll 2
                for (int t = 0; t < nf; ++t)
                    obp_job<NC, false>(rows + t * a.win, tb.pos[a0 + t], tb.e[a0 + t], it, jt, A, L0, L3, KR, KL);
#pragma unroll 2
                for (int t = nf; t < na; ++t)
                    obp_job<NC, true>(rows + t * a.win, tb.pos[a0 + t], tb.e[a0 + t], it, jt, A, L0, L3, KR, KL);
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
    }
}

template <int NC>
__global__ void __launch_bounds__(OBP_THREADS, 4) k_backproject_orbit(ObpArgs a)
{
    pdl_wait();
    pdl_trigger();
    obp_body<NC, false>(a, blockIdx.x, blockIdx.y, blockIdx.z);
}

size_t obp_smem(int win, int nc)
{
    return (size_t)2 * OBP_JCH * win * nc * sizeof(float) + OBP_TJ * (sizeof(uint4) + sizeof(float4) + sizeof(long long)) + 16;
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
    for (int k = 0; k < 3; ++k) a.list[k] = p->job_list[k];
    return a;
}
