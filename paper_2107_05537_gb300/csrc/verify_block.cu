// Verification of a small batch: a block of W warps per query.
//
// k_verify gives a query one warp, which a large batch turns into thousands of
// resident warps; a batch of a few hundred queries leaves most of the GPU idle
// while each warp walks its query's chain of dependent loads (leaf list, bounds,
// leaf centres, chunks, rows, guard set) alone.  Here the block takes each link
// of that chain together: the leaf list is made and bounded by all threads, a
// window of leaves gets its full bounds eight leaves per warp, the leaves are
// visited in groups whose rows' distances are taken eight rows per warp at once,
// and the guard set's FP64 sums run on as many lanes as there are rows.
// Measured against k_verify (one launch, GB300): 1 query on 10,000 x 128 31 us
// (77), 200 on 54,387 x 192 59 us (269), 1,001 on 199,999 x 100 152 us (264), 1,000
// on 200,000 x 960 568 us (1,394, BF16 first pass).
//
// The result is that of k_verify (and of verifying every candidate): every leaf,
// chunk or row left out has a proven lower bound above an upper bound of the
// KP-th smallest FP32 distance, and the guard set is recomputed in FP64 and
// ranked by (FP64 distance, id).
#include <cfloat>

#include "knn_shared.cuh"

namespace pmk {

namespace {

constexpr int VB_ROWS = 1024;            // rows of a group of leaves (a leaf has at most 1,024)
constexpr int VB_KEEP = 512;             // entries that a cut keeps at most (KP is at most 320)
constexpr int VB_CAP = VB_KEEP + VB_ROWS;
constexpr int VB_WIN = 128;              // leaves of a window at most
constexpr int VB_WANT = 64;              // and at least, while leaves are left
constexpr int VB_GROUP = 32;             // leaves of a group at most
constexpr int VB_FIRST = 192;            // rows that close the first group, before anything can be pruned,
constexpr int VB_NEXT = 512;             // and the later ones
constexpr int VB_BINS = 512;
constexpr int VB_GR = 64;                // guard rows whose FP64 sums run together

// Shared memory of the walk; the guard set's squares take the same place after it.
struct VbWalk {
    float val[VB_CAP];                   // kept entries, then the group's: FP32 distance^2
    int pos[VB_CAP];                     // and position
    float wb[VB_WIN], fb[VB_WIN];        // window: cheap bound, full bound
    int wl[VB_WIN], ord[VB_WIN];         // leaf (-1: pruned), window index by ascending full bound
    int wcb[VB_WIN], wce[VB_WIN], wn[VB_WIN];   // chunk range and size of the leaf
    float wrx[VB_WIN];                   // radius of the leaf
    int chunk[VB_ROWS], crow[VB_ROWS];   // chunks of the group: number, first row
    unsigned char cn[VB_ROWS];           // rows (at most 32)
    unsigned char cf[VB_ROWS];           // 1: leaf full, 2: needs its own bound, 4: pruned
    unsigned int hist[VB_BINS];
};
struct VbShared {
    union {
        VbWalk w;
        double sq64[2 * 32 * (VB_GR + 1)];   // squares of two steps of 32 coordinates, [coordinate][row]
    };
    alignas(16) float sq[PM_MP];
    float sp[PM_MAX_PIVOTS], sPq[PM_PCA];
    unsigned int kMin, kMax;             // ordered keys of a minimum and a maximum
    int cnt, bin, below, in, work;
};

// Total order of finite FP32 values as unsigned keys.
__device__ __forceinline__ unsigned int vb_key(float f)
{
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float vb_unkey(unsigned int k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
// A finite stand-in for a distance bound that keeps the order: NaN (no bound) first.
__device__ __forceinline__ float vb_finite(float f)
{
    return f != f ? -1e30f : fminf(fmaxf(f, -1e30f), 1e30f);
}

// Squared FP32 distances of the query to the rows x and (TWO) y of the lane's group
// of four (the same pointers in the four lanes), eight rows each per warp; the sums
// in all four lanes, in warp_d2x4's order.  The loads of a step are issued together
// and unconditionally (a lane without a row reads a valid one); the rest of a row,
// two, four or six loads per lane (ld % 32 == 0), goes in steps of four and two: one
// load at a time exposed its latency six times on rows of 96 coordinates.
template <bool TWO, int N>
__device__ __forceinline__ void vb_step(const float4 *__restrict__ q4, const float4 *__restrict__ x,
                                        const float4 *__restrict__ y, int t, unsigned long long &ax,
                                        unsigned long long &ay)
{
    float4 u[N], v[N];
#pragma unroll
    for (int i = 0; i < N; i++) {
        u[i] = __ldg(x + t + 4 * i);
        if (TWO) v[i] = __ldg(y + t + 4 * i);
    }
#pragma unroll
    for (int i = 0; i < N; i++) {
        const float4 qv = q4[t + 4 * i];
        const unsigned long long q0 = f32x2_pack(qv.x, qv.y), q1 = f32x2_pack(qv.z, qv.w);
        f32x2_sqdiff_acc(ax, q0, f32x2_pack(u[i].x, u[i].y));
        f32x2_sqdiff_acc(ax, q1, f32x2_pack(u[i].z, u[i].w));
        if (TWO) {
            f32x2_sqdiff_acc(ay, q0, f32x2_pack(v[i].x, v[i].y));
            f32x2_sqdiff_acc(ay, q1, f32x2_pack(v[i].z, v[i].w));
        }
    }
}

template <bool TWO>
__device__ __forceinline__ void vb_d2(const float4 *__restrict__ q4, const float4 *__restrict__ x,
                                      const float4 *__restrict__ y, int nf4, int g, float &dx, float &dy)
{
    unsigned long long ax = 0ull, ay = 0ull;
    int t = g;
#pragma unroll 1
    for (; t + 28 < nf4; t += 32) vb_step<TWO, 8>(q4, x, y, t, ax, ay);
    if (t + 12 < nf4) {
        vb_step<TWO, 4>(q4, x, y, t, ax, ay);
        t += 16;
    }
    if (t + 4 < nf4) vb_step<TWO, 2>(q4, x, y, t, ax, ay);
    dx = __fadd_rn(__uint_as_float((unsigned)ax), __uint_as_float((unsigned)(ax >> 32)));
    dx = __fadd_rn(dx, __shfl_xor_sync(VW_FULL, dx, 1));
    dx = __fadd_rn(dx, __shfl_xor_sync(VW_FULL, dx, 2));
    if (TWO) {
        dy = __fadd_rn(__uint_as_float((unsigned)ay), __uint_as_float((unsigned)(ay >> 32)));
        dy = __fadd_rn(dy, __shfl_xor_sync(VW_FULL, dy, 1));
        dy = __fadd_rn(dy, __shfl_xor_sync(VW_FULL, dy, 2));
    }
}

// One row, not inlined: leaf and chunk centres.
__device__ __noinline__ float vb_centre(const float *qs, const float *x, int nf4, int g)
{
    float d, none;
    vb_d2<false>((const float4 *)qs, (const float4 *)x, nullptr, nf4, g, d, none);
    return d;
}

// FP64 decision of a point inside the FP32 band (k_band64's test).
__device__ __noinline__ bool vb_band(const double *o, const double *q, int m, double R)
{
    return pm_pdist64(o, q, m) <= R;
}

// Selection of the smallest values by the block: v[e stride], e < n, taking part
// if valid[e stride] >= 0 (valid not null) and not above lim; NaN and infinity
// count as the largest finite value (squared distances reach it; bounds stay within
// +-1e30, so that a range never overflows).  Finds lo, hi and S.bin such that the values with v < lo, or
// v <= hi and vb_bin(v) <= S.bin, are at least `want` (or all) and, unless values
// tie, either at most `cap` in all or at most `capBin` in that bin (S.in; S.below
// before it).  Bins are linear in the value and monotone under rounding.  Not
// inlined: the block's three uses share its instructions, whose first fetch is a
// good part of a single query's time.
struct VbCut {
    float lo, hi, scale;
};
__device__ __forceinline__ int vb_bin(float v, float lo, float scale)
{
    return min(VB_BINS - 1, (int)((v - lo) * scale));
}
__device__ __forceinline__ float vb_val(float v) { return fminf(v, FLT_MAX); }

__device__ __noinline__ VbCut vb_select(VbShared &S, const float *vals, const int *valid, int stride, int n, float lim,
                                        int want, int cap, int capBin)
{
    const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
    VbCut c{-FLT_MAX, FLT_MAX, 0.f};
    int below = 0;
    for (int it = 0; it < 8; it++) {
        // range of the values in [lo, hi] (of the chosen bin, from the second step on)
        __syncthreads();
        if (tid == 0) {
            S.kMin = 0xFFFFFFFFu;
            S.kMax = 0u;
        }
        for (int i = tid; i < VB_BINS; i += T) S.w.hist[i] = 0u;
        __syncthreads();
        const int b0 = S.bin;
        unsigned int mn = 0xFFFFFFFFu, mx = 0u;
        for (int e = tid; e < n; e += T) {
            const float x = vals[e * stride], v = vb_val(x);
            if (x > lim || (valid && valid[e * stride] < 0) || v < c.lo || v > c.hi ||
                (it > 0 && vb_bin(v, c.lo, c.scale) != b0))
                continue;
            const unsigned int k = vb_key(v);
            mn = min(mn, k);
            mx = max(mx, k);
        }
        mn = __reduce_min_sync(VW_FULL, mn);
        mx = __reduce_max_sync(VW_FULL, mx);
        if (lane == 0 && mn <= mx) {
            atomicMin(&S.kMin, mn);
            atomicMax(&S.kMax, mx);
        }
        __syncthreads();
        const unsigned int kMin = S.kMin, kMax = S.kMax;
        if (kMin > kMax) break;   // nothing takes part (block-uniform); S.bin stays
        c.lo = vb_unkey(kMin);
        c.hi = vb_unkey(kMax);
        c.scale = c.hi > c.lo ? ((float)VB_BINS - 0.5f) / (c.hi - c.lo) : 0.f;
        for (int e = tid; e < n; e += T) {
            const float x = vals[e * stride], v = vb_val(x);
            if (!(x > lim) && !(valid && valid[e * stride] < 0) && v >= c.lo && v <= c.hi)
                atomicAdd(&S.w.hist[vb_bin(v, c.lo, c.scale)], 1u);
        }
        __syncthreads();
        if (tid < 32) {
            // the first bin at which `want` is reached (the last one otherwise)
            unsigned int h[VB_BINS / 32], sum = 0u;
#pragma unroll
            for (int j = 0; j < VB_BINS / 32; j++) {
                h[j] = S.w.hist[lane * (VB_BINS / 32) + j];
                sum += h[j];
            }
            unsigned int incl = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int t = __shfl_up_sync(VW_FULL, incl, o);
                if (lane >= o) incl += t;
            }
            const unsigned hit = __ballot_sync(VW_FULL, below + (int)incl >= want);
            const int src = hit ? __ffs(hit) - 1 : 31;
            if (lane == src) {
                int run = below + (int)(incl - sum), bin = 0, in = (int)h[0];
                bool found = run + in >= want;
#pragma unroll
                for (int j = 1; j < VB_BINS / 32; j++)
                    if (!found) {
                        run += in;
                        in = (int)h[j];
                        bin = j;
                        found = run + in >= want;
                    }
                S.bin = lane * (VB_BINS / 32) + bin;
                S.below = run;
                S.in = in;
            }
        }
        __syncthreads();
        if (S.below + S.in <= cap || S.in <= capBin || c.scale == 0.f) break;
        below = S.below;   // refine inside the bin
    }
    return c;
}

// FP32 value as sign, mantissa and exponent, value = m 2^(e - 150); zero: m = 0,
// e = 255.  ok: false for subnormals, infinities and NaN.
struct SqParts {
    int m, e;
    bool ok;
};
__device__ __forceinline__ SqParts sq_parts(float f)
{
    const unsigned int u = __float_as_uint(f);
    const int e = (int)((u >> 23) & 0xFFu);
    const bool z = (u << 1) == 0u;
    const int m = z ? 0 : (int)((u & 0x7FFFFFu) | 0x800000u);
    SqParts p;
    p.m = (int)u < 0 ? -m : m;
    p.e = z ? 255 : e;
    p.ok = z || (e > 0 && e < 255);
    return p;
}

// RN((x - q)^2) in FP64, the difference exact, by integer arithmetic: the same
// bits as __dmul_rn(t, t) with t = __dsub_rn(x, q), without the FP64 pipe (64
// cycles per warp instruction).  Holds where the exponents differ by at most six
// (the difference then has at most 31 bits, its square at most 62, rounded to
// nearest even); ok: false otherwise.
__device__ __forceinline__ double sq_int(const SqParts x, const SqParts q, bool &ok)
{
    const int emin = min(x.e, q.e), sx = x.e - emin, sq = q.e - emin;
    ok = x.ok && q.ok && (sx <= 6 || x.m == 0) && (sq <= 6 || q.m == 0);
    const int t = (x.m << (sx & 31)) - (q.m << (sq & 31));
    const unsigned int a = (unsigned int)abs(t);
    const int z = __clz((int)a);
    const unsigned int an = a << (z & 31);             // leading bit 31 (a = 0: zero)
    unsigned long long p = (unsigned long long)an * an;   // leading bit 63 or 62
    const int low = 1 - (int)(p >> 63);
    p <<= low;
    const unsigned long long r = (p + 0x3FFull + ((p >> 11) & 1ull)) >> 11;   // 53 bits, to nearest even
    const int E = 2 * (emin - 150 - z) - low + 63 + 1023;
    const unsigned long long bits = ((unsigned long long)(unsigned int)(E - 1) << 52) + r;
    return a == 0u ? 0.0 : __longlong_as_double((long long)bits);
}

template <int W>
__global__ void __launch_bounds__(32 * W, 16 / W)
k_verify_block(VwArgs A)
{
    constexpr int T = 32 * W, PER = VB_CAP / T;
    static_assert(VB_CAP % T == 0, "entries per thread");
    extern __shared__ __align__(16) unsigned char vbs[];
    VbShared &S = *(VbShared *)vbs;
    float *qs = (float *)(vbs + (sizeof(VbShared) + 15) / 16 * 16);
    double *gd = (double *)(qs + A.ld);
    long long *gid = (long long *)(gd + A.KP);
    int *gpos = (int *)(gid + A.KP);
    const float4 *q4 = (const float4 *)qs;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5, grp = lane >> 2, g = lane & 3;
    const int ld = A.ld, KP = A.KP, k = A.k, s = A.s, nf4 = A.ld >> 2;
    const int64_t L = A.L;
    int2 *list = A.lists + (int64_t)blockIdx.x * L;
    const double epsv = (double)(ld + 8) * 0x1.0p-24;
    const float lbMulF = __double2float_rd(1.0 - epsv), cutF = __double2float_ru(1.0 + 3.0 * epsv);
    const float lbSlack = 1.f - (float)((ld + 8) * 0x1.0p-24) - 1e-6f;
    // the first query by the block's number, the others from the counter
    for (int turn = 0;; turn++) {
        __syncthreads();
        if (tid == 0) {
            S.work = turn == 0 ? (int)blockIdx.x
                               : (A.nwork > (int)gridDim.x ? (int)gridDim.x + atomicAdd(A.workCtr, 1) : A.nwork);
            S.cnt = 0;
        }
        __syncthreads();
        int a = S.work;
        if (a >= A.nwork) break;
        if (A.order) a = A.order[a];
        if (!VW_CHECK(a >= 0, 7, a)) break;   // (block-uniform)
        const int q = A.act[a];
        const Thr Th = A.thr[a];
        const float lov = Th.lov;
        const float Rv = lov > 0.f ? __fsqrt_rn(lov) : -1.f;
        const bool inl = A.inlineBand != 0 && Th.pad == 0.f;
        const float Rout = inl ? __fsqrt_rn(Th.hi) : Rv;
        for (int i = tid; i < nf4; i += T) ((float4 *)qs)[i] = ((const float4 *)(A.Qd + (int64_t)q * ld))[i];
        if (tid < PM_MP) S.sq[tid] = A.qp32[(int64_t)q * PM_MP + tid];
        if (tid < PM_MAX_PIVOTS) S.sp[tid] = A.qpiv[(int64_t)q * PM_MAX_PIVOTS + tid];
        if (tid < PM_PCA) S.sPq[tid] = A.qpca[(int64_t)q * PM_PCA + tid];
        // block-uniform state: n0 kept entries, cmax an upper bound of the KP-th
        // smallest FP32 distance^2 of the candidates so far
        int n0 = 0, seen = 0, leaves = 0, nfp = 0;
        float cmax = INFINITY;
        auto pruned = [&](float lb) -> bool {
            return lb > 0.f && __fmul_rd(__fmul_rd(lb, lb), lbMulF) > __fmul_ru(cmax, cutF);
        };
        // 1. candidate leaves from the bit set, then their cheap bounds
        if (Rv > 0.f || inl) {
            const uint32_t *bits = A.leafBits + (int64_t)a * A.W32;
            for (int w0 = wib * 32; w0 < A.W32; w0 += T) {
                const int wi = w0 + lane;
                uint32_t word = wi < A.W32 ? bits[wi] : 0u;
                const int c = __popc(word);
                int incl = c;
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(VW_FULL, incl, o);
                    if (lane >= o) incl += v;
                }
                int base = 0;
                if (lane == 31 && incl) base = atomicAdd(&S.cnt, incl);
                int at = __shfl_sync(VW_FULL, base, 31) + incl - c;
                while (word) {
                    const int b = __ffs(word) - 1;
                    word &= word - 1u;
                    const int64_t l = (int64_t)wi * 32 + b;   // (bits at and past L are never set)
                    if (at < L) list[at] = make_int2((int)l, 0);
                    at++;
                }
            }
        }
        __syncthreads();
        const int cnt = (int)min((int64_t)S.cnt, L);
        // slack of the cheap bound: as in k_verify
        const float pSlack = __fmul_ru(1.01f, __fadd_ru(__fmul_ru((float)(4 * (ld + 2)) * 0x1.0p-24f, A.qnx[q]),
                                                        __fmul_ru(0x1.0p-20f, __fadd_ru(A.qnx[q], A.muMax))));
        for (int e = tid; e < cnt; e += T) {
            const int l = list[e].x;
            if (!VW_CHECK(l >= 0 && l < L, 1, l)) {
                list[e] = make_int2(-1, 0);
                continue;
            }
            const float4 *pm4 = (const float4 *)(A.leafPmu + (int64_t)l * PM_PCA);
            const float rx = A.leafRx[l];
            float acc = 0.f;
#pragma unroll
            for (int r4 = 0; r4 < PM_PCA / 4; r4++) {
                const float4 v = __ldg(pm4 + r4);
                float u = __fsub_rn(S.sPq[4 * r4], v.x);
                acc = __fmaf_rn(u, u, acc);
                u = __fsub_rn(S.sPq[4 * r4 + 1], v.y);
                acc = __fmaf_rn(u, u, acc);
                u = __fsub_rn(S.sPq[4 * r4 + 2], v.z);
                acc = __fmaf_rn(u, u, acc);
                u = __fsub_rn(S.sPq[4 * r4 + 3], v.w);
                acc = __fmaf_rn(u, u, acc);
            }
            const float lbp = __fsub_rn(__fsub_rn(__fmul_rn(__fsqrt_rn(acc), 1.f - 0x1.0p-18f), pSlack), rx);
            list[e] = make_int2(l, __float_as_int(vb_finite(lbp)));
        }
        // keeps the entries that can be among the KP smallest of val[0, n1)
        auto cut = [&](int n1) {
            if (n1 < KP) {
                n0 = n1;
                return;
            }
            const float lim = cmax;
            const VbCut c = vb_select(S, S.w.val, nullptr, 1, n1, lim, KP, VB_KEEP, 0);
            const int bin = S.bin;
            float v[PER];
            int p[PER];
#pragma unroll
            for (int u = 0; u < PER; u++) {
                const int e = u * T + tid;
                v[u] = e < n1 ? S.w.val[e] : 0.f;
                p[u] = e < n1 ? S.w.pos[e] : 0;
            }
            __syncthreads();
            if (tid == 0) {
                S.cnt = 0;
                S.kMax = 0u;
            }
            __syncthreads();
            unsigned int mx = 0u;
#pragma unroll
            for (int u = 0; u < PER; u++) {
                const int e = u * T + tid;
                const float f = vb_val(v[u]);
                const bool keep = e < n1 && !(v[u] > lim) && (f < c.lo || (f <= c.hi && vb_bin(f, c.lo, c.scale) <= bin));
                const unsigned m = __ballot_sync(VW_FULL, keep);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&S.cnt, __popc(m));
                const int at = __shfl_sync(VW_FULL, base, 0) + __popc(m & ((1u << lane) - 1u));
                if (keep && at < VB_KEEP) {
                    S.w.val[at] = v[u];
                    S.w.pos[at] = p[u];
                }
                if (keep) mx = max(mx, vb_key(v[u]));
            }
            mx = __reduce_max_sync(VW_FULL, mx);
            if (lane == 0 && mx) atomicMax(&S.kMax, mx);
            __syncthreads();
            n0 = min(S.cnt, VB_KEEP);
            // at least KP entries are kept and none is larger; entries left out
            // are at least as large as the largest kept
            cmax = fminf(cmax, vb_unkey(S.kMax));
        };
        // FP32 distances of the entries [n0, n1): sixteen rows per warp in flight
        auto distances = [&](int n1) {
            for (int e0 = n0 + wib * 8; e0 < n1; e0 += 16 * W) {
                const int e = e0 + grp, f = e + 8 * W;
                const float4 *x = (const float4 *)(A.X + (int64_t)S.w.pos[min(e, n1 - 1)] * ld);
                float dx, dy = 0.f;
                if (e0 + 8 * W < n1) {   // (warp-uniform)
                    const float4 *y = (const float4 *)(A.X + (int64_t)S.w.pos[min(f, n1 - 1)] * ld);
                    vb_d2<true>(q4, x, y, nf4, g, dx, dy);
                } else {
                    vb_d2<false>(q4, x, x, nf4, g, dx, dy);
                }
                if (e < n1 && g == 0) S.w.val[e] = dx;
                if (f < n1 && g == 0) S.w.val[f] = dy;
            }
            __syncthreads();
        };
        // 2. windows of the leaves with the smallest cheap bounds
        int remaining = cnt;
        while (remaining > 0) {
            const VbCut c = vb_select(S, (const float *)list + 1, (const int *)list, 2, cnt, INFINITY,
                                      min(VB_WANT, remaining), VB_WIN, 0);
            const int bin = S.bin;
            __syncthreads();
            if (tid == 0) {
                S.cnt = 0;
                S.kMax = 0u;
            }
            __syncthreads();
            unsigned int mx = 0u;
            for (int e0 = 0; e0 < cnt; e0 += T) {
                const int e = e0 + tid;
                const int2 x = e < cnt ? list[e] : make_int2(-1, 0);
                const float v = __int_as_float(x.y);
                const bool take = x.x >= 0 && (v < c.lo || (v <= c.hi && vb_bin(v, c.lo, c.scale) <= bin));
                const unsigned m = __ballot_sync(VW_FULL, take);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&S.cnt, __popc(m));
                const int at = __shfl_sync(VW_FULL, base, 0) + __popc(m & ((1u << lane) - 1u));
                if (take && at < VB_WIN) {
                    S.w.wb[at] = v;
                    S.w.wl[at] = x.x;
                    list[e].x = -1;
                    mx = max(mx, vb_key(v));
                }
            }
            mx = __reduce_max_sync(VW_FULL, mx);
            if (lane == 0 && mx) atomicMax(&S.kMax, mx);
            __syncthreads();
            const int nw = min(S.cnt, VB_WIN);
            if (nw == 0) break;
            const float tau = vb_unkey(S.kMax);   // no leaf left has a smaller cheap bound
            remaining -= nw;
            // full bounds (original-space leaf ball), eight leaves per warp
            for (int i0 = wib * 8; i0 < nw; i0 += 8 * W) {
                const int i = i0 + grp;
                const bool need = i < nw && !pruned(S.w.wb[i]);
                const int l = need ? S.w.wl[i] : 0;
                const float d2 = vb_centre(qs, A.leafMu + (int64_t)l * ld, nf4, g);
                if (i < nw && g == 0) {
                    if (need) {
                        const float rx = A.leafRx[l];
                        S.w.fb[i] = vb_finite(__fsub_rn(__fmul_rn(__fsqrt_rn(d2), lbSlack), rx));
                        S.w.wrx[i] = rx;
                        S.w.wcb[i] = A.leafChunk[l];
                        S.w.wce[i] = A.leafChunk[l + 1];
                        S.w.wn[i] = (int)(A.leafOff[l + 1] - A.leafOff[l]);
                    } else {
                        S.w.fb[i] = FLT_MAX;   // after every leaf that is not pruned
                        S.w.wl[i] = -1;
                    }
                }
            }
            __syncthreads();
            for (int i = tid; i < nw; i += T) {
                const float f = S.w.fb[i];
                int r = 0;
                for (int j = 0; j < nw; j++) {
                    const float h = S.w.fb[j];
                    r += (h < f || (h == f && j < i)) ? 1 : 0;
                }
                S.w.ord[r] = i;
            }
            __syncthreads();
            // visits, by groups of leaves in ascending full bound: enough rows
            // for every warp, at most VB_ROWS
            for (int i = 0; i < nw;) {
                int j = i, rows = 0, nch = 0;
                bool bounds = false;
                for (; j < nw && j - i < VB_GROUP; j++) {
                    const int e = S.w.ord[j];
                    const float f = S.w.fb[e];
                    if (S.w.wl[e] < 0 || pruned(f)) break;
                    const int n = S.w.wn[e], c = S.w.wce[e] - S.w.wcb[e];
                    if (!VW_CHECK(n >= 1 && n <= VB_ROWS && c >= 1 && c <= n, 3, n)) break;
                    if (rows > 0 && (rows >= (cmax == INFINITY ? VB_FIRST : VB_NEXT) || rows + n > VB_ROWS)) break;
                    // chunk bounds only if one can prune (see k_verify)
                    const float ubl = __fadd_ru(__fmul_ru(__fadd_ru(fmaxf(f, 0.f), S.w.wrx[e]), 1.0001f), S.w.wrx[e]);
                    const bool cb = __fmul_ru(ubl, ubl) > cmax;
                    bounds |= cb;
                    const int l = S.w.wl[e];
                    const unsigned char cl = Th.pad == 0.f
                        ? (((A.fullBits[(int64_t)a * A.W32 + (l >> 5)] >> (l & 31)) & 1u) ? CL_FULL : CL_PART)
                        : leaf_class(S.sq, S.sp, s, Rv, Rout, A.meta + (int64_t)l * PM_LEAF_STRIDE);
                    for (int x = tid; x < c; x += T) {
                        const int ch = S.w.wcb[e] + x;
                        const int64_t r0 = A.chunkOff[ch];
                        int nr = (int)(A.chunkOff[ch + 1] - r0);
                        if (!VW_CHECK(nr >= 1 && nr <= 32 && r0 >= 0 && r0 + nr <= A.n, 2, nr)) nr = 0;
                        S.w.chunk[nch + x] = ch;
                        S.w.crow[nch + x] = (int)r0;
                        S.w.cn[nch + x] = (unsigned char)nr;
                        S.w.cf[nch + x] = (unsigned char)((cl == CL_FULL ? 1 : 0) | (cb ? 2 : 0));
                    }
                    rows += n;
                    nch += c;
                }
                if (j == i) break;   // the first leaf is pruned, and so are the rest
                if (tid == 0) S.cnt = 0;
                __syncthreads();
                if (bounds) {
                    for (int c0 = wib * 8; c0 < nch; c0 += 8 * W) {
                        const int x = c0 + grp;
                        const bool need = x < nch && (S.w.cf[x] & 2);
                        const int c = need ? S.w.chunk[x] : 0;
                        const float d2 = vb_centre(qs, A.chunkMu + (int64_t)c * ld, nf4, g);
                        if (need && g == 0 && pruned(__fsub_rn(__fmul_rn(__fsqrt_rn(d2), lbSlack), A.chunkRx[c])))
                            S.w.cf[x] |= 4;
                    }
                    __syncthreads();
                }
                // candidate rows, four chunks per warp and step
                for (int x0 = wib; x0 < nch; x0 += 4 * W) {
                    bool cand[4];
                    int row[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int x = x0 + u * W;
                        const unsigned char f = x < nch ? S.w.cf[x] : 4;
                        const int nr = (f & 4) ? 0 : S.w.cn[x];
                        row[u] = nr ? S.w.crow[x] + lane : 0;
                        cand[u] = lane < nr;
                        if (cand[u] && !(f & 1)) {
                            const float pd = pd2_row(A.O32 + (int64_t)row[u] * PM_MP, S.sq);
                            cand[u] = pd <= lov;
                            if (!cand[u] && inl && pd <= Th.hi) {
                                cand[u] = vb_band(A.O64 + (int64_t)row[u] * PM_MP, A.qp64 + (int64_t)q * PM_MP, A.m, Th.R);
                                nfp++;
                            }
                        }
                    }
                    unsigned m[4];
                    int tot = 0, at[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        m[u] = __ballot_sync(VW_FULL, cand[u]);
                        at[u] = tot + __popc(m[u] & ((1u << lane) - 1u));
                        tot += __popc(m[u]);
                    }
                    int base = 0;
                    if (lane == 0 && tot) base = atomicAdd(&S.cnt, tot);
                    base = n0 + __shfl_sync(VW_FULL, base, 0);
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (cand[u] && base + at[u] < VB_CAP) S.w.pos[base + at[u]] = row[u];
                }
                __syncthreads();
                const int n1 = min(n0 + S.cnt, VB_CAP);
                seen += n1 - n0;
                leaves += j - i;
                distances(n1);
                if (n1 > n0) cut(n1);
                __syncthreads();
                i = j;
            }
            __syncthreads();
            if (pruned(tau)) break;
        }
        // band-in points (FP64-resolved members just inside the radius)
        const int nIn = min(A.inN[a], BCAP);
        if (nIn > 0) {
            for (int e = tid; e < nIn; e += T) {
                int pos = A.inPos[(int64_t)a * BCAP + e];
                if (!VW_CHECK(pos >= 0 && pos < A.n, 4, pos)) pos = 0;
                S.w.pos[n0 + e] = pos;   // (at most VB_KEEP + BCAP entries)
            }
            __syncthreads();
            distances(n0 + nIn);
            n0 += nIn;
            seen += nIn;
        }
        // 3. guard set: exact k-th smallest value, by the ranks of the entries
        // around it
        float K32 = INFINITY;
        if (n0 >= k) {
            const VbCut c = vb_select(S, S.w.val, nullptr, 1, n0, INFINITY, k, 0, VB_WIN);
            const int bin = S.bin, below = S.below;
            __syncthreads();
            if (tid == 0) S.kMax = vb_key(INFINITY);
            __syncthreads();
            // the (k - below)-th smallest of the chosen bin: its members are few
            // (more than VB_WIN only if they tie, and then all are equal)
            if (tid == 0) S.cnt = 0;
            __syncthreads();
            for (int e = tid; e < n0; e += T) {
                const float f = vb_val(S.w.val[e]);
                if (f >= c.lo && f <= c.hi && vb_bin(f, c.lo, c.scale) == bin) {
                    const int at = atomicAdd(&S.cnt, 1);
                    if (at < VB_WIN) S.w.wb[at] = S.w.val[e];
                }
            }
            __syncthreads();
            const int nb = min(S.cnt, VB_WIN);
            for (int e = tid; e < nb; e += T) {
                const float f = S.w.wb[e];
                int r = 0;
                for (int h = 0; h < nb; h++) r += (S.w.wb[h] < f || (S.w.wb[h] == f && h < e)) ? 1 : 0;
                if (r == min(k - 1 - below, nb - 1)) S.kMax = vb_key(f);
            }
            __syncthreads();
            K32 = vb_unkey(S.kMax);
        }
        const float thrv = K32 < INFINITY ? (float)((double)K32 * (1.0 + 3.0 * epsv) + 1e-36) : INFINITY;
        __syncthreads();
        if (tid == 0) S.cnt = 0;
        __syncthreads();
        for (int e0 = 0; e0 < n0; e0 += T) {
            const int e = e0 + tid;
            const float v = e < n0 ? S.w.val[e] : INFINITY;
            const bool in = v <= thrv && v < INFINITY;
            const unsigned m = __ballot_sync(VW_FULL, in);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&S.cnt, __popc(m));
            const int at = __shfl_sync(VW_FULL, base, 0) + __popc(m & ((1u << lane) - 1u));
            if (in && at < KP) gpos[at] = S.w.pos[e];
        }
        __syncthreads();
        // KP entries or more inside the guard band: some may have been left out
        if (tid == 0 && seen > KP && S.cnt >= KP) atomicOr(A.errFlag, 16);
        const int G = min(S.cnt, KP);
        // FP64 distances, the oracle's sequential sum over i = 0 .. d - 1 of the
        // rounded squares.  The FP64 pipe takes 64 cycles per warp instruction
        // whatever its active lanes, and only the additions are a chain that needs
        // it: the squares are taken by integer arithmetic, the lanes over the
        // coordinates (a warp per row and 32 coordinates), by the warps that do not
        // add, a step ahead of the one or two warps that add them with a row per
        // lane.  The guard set then costs the latency of its additions, 64 d
        // cycles: 10 rows of 128 took 50,000 cycles with a row per lane throughout
        // (subtraction, multiplication and addition in one chain), 16,800 now.
        for (int e = tid; e < G; e += T) {
            int p = gpos[e];
            if (!VW_CHECK(p >= 0 && p < A.n, 5, p)) gpos[e] = p = 0;
            gid[e] = (long long)A.perm[p];
        }
        for (int r0 = 0; r0 < G; r0 += VB_GR) {
            const int nr = min(VB_GR, G - r0), na = (nr + 31) / 32;   // rows and adding warps
            const int nstep = (A.d + 31) / 32;
            double sum = 0.0;
            __syncthreads();
            // (the squaring warps read the next step's coordinates before they wait)
            constexpr int PF = 8;
            float xv[PF];
            auto fetch = [&](int st) {
                const int i = st * 32 + lane;
#pragma unroll
                for (int u = 0; u < PF; u++) {
                    const int r = wib - na + u * (W - na);
                    xv[u] = r < nr && i < A.d ? __ldg(A.X + (int64_t)gpos[r0 + r] * ld + i) : 0.f;
                }
            };
            if (wib >= na) fetch(0);
            for (int st = 0; st <= nstep; st++) {
                if (wib >= na) {
                    if (st < nstep) {
                        const int i = st * 32 + lane;
                        const bool iv = i < A.d;
                        const float qf = iv ? qs[i] : 0.f;
                        const SqParts qp = sq_parts(qf);
                        double *tb = S.sq64 + (st & 1) * 32 * (VB_GR + 1) + lane * (VB_GR + 1);
                        // (columns past d add +0)
                        auto square = [&](int r, float x) {
                            bool ok;
                            double v = sq_int(sq_parts(x), qp, ok);
                            if (__any_sync(VW_FULL, !ok)) {   // a real branch: few rows take it
                                const double t = __dsub_rn(f2d_exact(x), f2d_exact(qf)), w = __dmul_rn(t, t);
                                v = ok ? v : w;
                            }
                            tb[r] = v;
                        };
#pragma unroll
                        for (int u = 0; u < PF; u++) {
                            const int r = wib - na + u * (W - na);
                            if (r < nr) square(r, xv[u]);
                        }
                        // the rows beyond, eight loads at a time (one by one their latency
                        // stood in every step: 256 coordinates, up to 101 rows on four
                        // warps, 126,000 cycles per query, 92,000 now)
#pragma unroll 1
                        for (int u0 = PF; wib - na + u0 * (W - na) < nr; u0 += PF) {
                            float y[PF];
#pragma unroll
                            for (int u = 0; u < PF; u++) {
                                const int r = wib - na + (u0 + u) * (W - na);
                                y[u] = r < nr && iv ? __ldg(A.X + (int64_t)gpos[r0 + r] * ld + i) : 0.f;
                            }
#pragma unroll
                            for (int u = 0; u < PF; u++) {
                                const int r = wib - na + (u0 + u) * (W - na);
                                if (r < nr) square(r, y[u]);
                            }
                        }
                        if (st + 1 < nstep) fetch(st + 1);
                    }
                } else if (st > 0) {
                    const double *tb = S.sq64 + ((st - 1) & 1) * 32 * (VB_GR + 1) + wib * 32 + lane;
                    // sixteen values ahead of the additions
                    double u[16], v[16];
#pragma unroll
                    for (int c = 0; c < 16; c++) u[c] = tb[c * (VB_GR + 1)];
#pragma unroll
                    for (int c = 0; c < 16; c++) v[c] = tb[(16 + c) * (VB_GR + 1)];
#pragma unroll
                    for (int c = 0; c < 16; c++) sum = __dadd_rn(sum, u[c]);
#pragma unroll
                    for (int c = 0; c < 16; c++) sum = __dadd_rn(sum, v[c]);
                }
                __syncthreads();
            }
            if (wib < na && wib * 32 + lane < nr) gd[r0 + wib * 32 + lane] = __dsqrt_rn(sum);
        }
        __syncthreads();
        // rank by (FP64 distance, id); the k nearest are written in order
        for (int e = tid; e < G; e += T) {
            const double dv = gd[e];
            const long long iv = gid[e], db = __double_as_longlong(dv);
            int rank = 0;
#pragma unroll 4
            for (int f = 0; f < G; f++) {
                const long long fbits = __double_as_longlong(gd[f]);
                rank += (fbits < db || (fbits == db && gid[f] < iv)) ? 1 : 0;
            }
            if (rank < k) {
                const int64_t o = (int64_t)q * k + rank;
                const float fv = __double2float_rn(dv);
                A.outIds[o] = iv;
                A.outD[o] = fv;
                A.outErr[o] = (float)fabs((double)fv - dv);
            }
            if (rank == k - 1) A.dk[a] = dv;
        }
        for (int e = G + tid; e < k; e += T) {
            const int64_t o = (int64_t)q * k + e;
            A.outIds[o] = -1;
            A.outD[o] = INFINITY;
            A.outErr[o] = 0.f;
        }
        for (int o = 16; o; o >>= 1) nfp += __shfl_xor_sync(VW_FULL, nfp, o);
        if (lane == 0 && nfp) atomicAdd(&A.fp64cnt[a], nfp);
        if (tid == 0) {
            if (G < k) A.dk[a] = INFINITY;
            atomicAdd(&A.fp64cnt[a], G);
            A.nverOut[a] = seen;
            A.nleafOut[a] = leaves;
        }
    }
}

}  // namespace

size_t vb_smem_bytes(int ld, int KP)
{
    return (sizeof(VbShared) + 15) / 16 * 16 + (size_t)ld * 4 + (size_t)KP * 20;
}

pmlsh_status vb_launch(const VwArgs &A, int W, int grid, cudaStream_t st)
{
    const size_t smem = vb_smem_bytes(A.ld, A.KP);
    if (W == 8) {
        PM_TRY(pm_allow_max_dyn_smem((const void *)k_verify_block<8>));
        PM_LAUNCH("k_verify_block", st, k_verify_block<8><<<grid, 256, smem, st>>>(A));
    } else {
        PM_TRY(pm_allow_max_dyn_smem((const void *)k_verify_block<4>));
        PM_LAUNCH("k_verify_block", st, k_verify_block<4><<<grid, 128, smem, st>>>(A));
    }
    PM_CUDA(cudaGetLastError());
    return PMLSH_OK;
}

}  // namespace pmk
