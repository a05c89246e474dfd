// (c,k)-ACP query path: Algorithm 4 (radius filtering) with FindLCA
// (Algorithm 5) over the index's leaf hierarchy.
//
//   k_cp_selfjoin   every pair inside each leaf: FP32 squared distance
//   k_node_box,     node balls (Sec. 4.1) in FP64, bounding-box midpoint and
//   k_node_radius   largest distance, the same arithmetic as the oracle
//   [host]          FindLCA: maximal inner nodes with radius < R = gamma t ub,
//                   sorted by (radius, node id)
//   k_cp_tiles      cross-leaf pairs of nodes' subtrees with projected distance
//                   < t ub (FP32 with a proven band, FP64 inside it)
//   k_cp_replay     the nodes of a batch in order, for one value of ub
//   k_pair_*        exact top-k merges: radix select of an FP32 threshold,
//                   guard set, FP64 distances, sort by (dist, i, j)
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "pmlsh_impl.h"

namespace {

constexpr int PAIR_SORT_CAP = 4096;   // guard entries merged in one block

struct PairCand {
    float key;      // FP32 squared distance (original or projected space)
    int32_t a, b;   // leaf-order positions, a < b in position order
};

// All pairs inside leaf l, FP32 squared distance by direct difference
// (sequential over the row).  One block per leaf.
__global__ void k_cp_selfjoin(const float *__restrict__ X, int ld, const int64_t *__restrict__ off,
                              const int64_t *__restrict__ pairOff, PairCand *__restrict__ out)
{
    const int64_t l = blockIdx.x;
    const int64_t p0 = off[l], s = off[l + 1] - p0;
    const int64_t np = s * (s - 1) / 2;
    for (int64_t e = threadIdx.x; e < np; e += blockDim.x) {
        // e -> (i, j), i < j, row-major over the upper triangle: row i starts
        // at C(i) = i (2 s - i - 1) / 2; i from the root of C(i) = e in FP64,
        // then integer corrections (at most a step or two)
        const double b2 = 2.0 * (double)s - 1.0;
        int64_t i = (int64_t)((b2 - sqrt(fmax(0.0, b2 * b2 - 8.0 * (double)e))) * 0.5);
        i = i < 0 ? 0 : (i > s - 2 ? s - 2 : i);
        while (i > 0 && i * (2 * s - i - 1) / 2 > e) i--;
        while (i < s - 2 && (i + 1) * (2 * s - i - 2) / 2 <= e) i++;
        const int64_t j = i + 1 + (e - i * (2 * s - i - 1) / 2);
        const float *x = X + (p0 + i) * ld, *y = X + (p0 + j) * ld;
        float acc = 0.f;
        for (int c = 0; c < ld; c++) {
            float t = __fsub_rn(x[c], y[c]);
            acc = __fmaf_rn(t, t, acc);
        }
        PairCand pc;
        pc.key = acc;
        pc.a = (int32_t)(p0 + i);
        pc.b = (int32_t)(p0 + j);
        out[pairOff[l] + e] = pc;
    }
}

// Node balls in FP64 (Sec. 4.1): centre = midpoint of the bounding box of the
// node's projected points, radius = largest FP64 distance to it.  A node is
// cut into slices of NB_SLICE positions, a warp per slice: k_node_box takes the
// bounding boxes (minima and maxima of order-preserving integer keys, which
// leave the FP64 pipe to the distances), k_node_radius the largest distance;
// the slices of a node meet in integer atomics, so no order matters.  Bound by
// the FP64 pipe, two operations per SM and clock here: n depth 45 operations,
// which slices spread evenly; a block per node left the root's 100,000 points
// to one SM (77,000 nodes: 5.5 ms, in slices 0.3 ms).
constexpr int NB_SLICE = 256;
struct NodeSlice {
    int64_t lo, hi;
    int32_t node;
    int32_t pad;
};

__device__ __forceinline__ long long nb_key(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double nb_unkey(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

// box [node][2][PM_MP]: keys of the minima and maxima
__global__ void k_node_box_init(long long *__restrict__ box, unsigned long long *__restrict__ rad, int64_t nodes)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < nodes * 2 * PM_MP) box[i] = (i / PM_MP) % 2 == 0 ? 0x7fffffffffffffffLL : (long long)0x8000000000000000ULL;
    if (i < nodes) rad[i] = 0ull;
}

__global__ void __launch_bounds__(256)
k_node_box(const double *__restrict__ O64, const NodeSlice *__restrict__ sl, int64_t ns, long long *__restrict__ box)
{
    const int lane = threadIdx.x & 31, j = lane & 7;
    const int64_t i = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= ns) return;   // warp-uniform
    const NodeSlice S = sl[i];
    // eight lanes per point, two coordinates per lane
    long long mn0 = 0x7fffffffffffffffLL, mn1 = mn0, mx0 = (long long)0x8000000000000000ULL, mx1 = mx0;
#pragma unroll 4
    for (int64_t p = S.lo + (lane >> 3); p < S.hi; p += 4) {
        const double2 v = __ldg((const double2 *)(O64 + p * PM_MP) + j);
        const long long k0 = nb_key(v.x), k1 = nb_key(v.y);
        mn0 = k0 < mn0 ? k0 : mn0;
        mx0 = k0 > mx0 ? k0 : mx0;
        mn1 = k1 < mn1 ? k1 : mn1;
        mx1 = k1 > mx1 ? k1 : mx1;
    }
    for (int o = 8; o < 32; o <<= 1) {
        const long long a = __shfl_xor_sync(0xffffffffu, mn0, o), b = __shfl_xor_sync(0xffffffffu, mn1, o);
        const long long c = __shfl_xor_sync(0xffffffffu, mx0, o), d = __shfl_xor_sync(0xffffffffu, mx1, o);
        mn0 = a < mn0 ? a : mn0;
        mn1 = b < mn1 ? b : mn1;
        mx0 = c > mx0 ? c : mx0;
        mx1 = d > mx1 ? d : mx1;
    }
    if (lane < 8) {
        long long *B = box + (int64_t)S.node * 2 * PM_MP;
        atomicMin(B + 2 * j, mn0);
        atomicMin(B + 2 * j + 1, mn1);
        atomicMax(B + PM_MP + 2 * j, mx0);
        atomicMax(B + PM_MP + 2 * j + 1, mx1);
    }
}

__global__ void __launch_bounds__(256)
k_node_radius(const double *__restrict__ O64, const NodeSlice *__restrict__ sl, int64_t ns,
              const long long *__restrict__ box, int m, unsigned long long *__restrict__ rad)
{
    __shared__ double sC[8][PM_MP];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)(blockDim.x >> 5) + w;
    if (i >= ns) return;   // warp-uniform
    const NodeSlice S = sl[i];
    const long long *B = box + (int64_t)S.node * 2 * PM_MP;
    if (lane < PM_MP) sC[w][lane] = lane < m ? __dmul_rn(0.5, __dadd_rn(nb_unkey(B[lane]), nb_unkey(B[PM_MP + lane]))) : 0.0;
    __syncwarp();
    double r = 0.0;
    for (int64_t p = S.lo + lane; p < S.hi; p += 32) r = fmax(r, pm_pdist64(O64 + p * PM_MP, sC[w], m));
    // distances are >= +0: their bits order like them
    unsigned long long rb = (unsigned long long)__double_as_longlong(r);
    for (int o = 16; o; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, rb, o);
        rb = x > rb ? x : rb;
    }
    if (lane == 0) atomicMax(rad + S.node, rb);
}

// Sec. 6.3, setting of gamma: for every pair (a, b), a < b, of the n
// positions of a layout, R / ||o_a', o_b'|| with R the radius of their lowest
// common node (descending from the root while both leaves lie in one child;
// the leaf itself for two points of one leaf), FP64 projected distance with
// the oracle's arithmetic and a correctly rounded quotient; 0 / 0 -> 0,
// R / 0 -> +inf.  Block a writes pairs (a, b) at a n - a (a + 1) / 2 + b - a - 1.
__global__ void k_gamma_ratio(const double *__restrict__ O64, int64_t n, int m, const int32_t *__restrict__ leafOf,
                              const int64_t *__restrict__ node /*[N][4]: left, right, leaf lo, leaf hi*/,
                              const double *__restrict__ rad, double *__restrict__ out, int *__restrict__ err)
{
    const int64_t a = blockIdx.x;
    const int64_t base = a * n - a * (a + 1) / 2 - a - 1;
    const int64_t la = leafOf[a];
    for (int64_t b = a + 1 + threadIdx.x; b < n; b += blockDim.x) {
        const int64_t lb = leafOf[b];
        int64_t e = 0;
        int depth = 0;
        for (; depth < 4096; depth++) {
            const int64_t x = node[e * 4], y = node[e * 4 + 1];
            if (x < 0) break;
            if (la >= node[x * 4 + 2] && la < node[x * 4 + 3] && lb >= node[x * 4 + 2] && lb < node[x * 4 + 3])
                e = x;
            else if (la >= node[y * 4 + 2] && la < node[y * 4 + 3] && lb >= node[y * 4 + 2] && lb < node[y * 4 + 3])
                e = y;
            else
                break;
        }
        if (depth == 4096) atomicOr(err, 1);
        const double R = rad[e];
        const double dv = pm_pdist64(O64 + a * PM_MP, O64 + b * PM_MP, m);
        out[base + b] = dv > 0.0 ? __ddiv_rn(R, dv) : (R > 0.0 ? (double)INFINITY : 0.0);
    }
}

// The same ratios in FP32, to find the few whose FP64 value can be the wanted rank.
// Block a walks to its leaf once and keeps the ranges and radii of the nodes on the
// way in shared memory: the lowest common node of (a, b), b > a, is the deepest one
// that ends beyond b's leaf (k_gamma_ratio descends from the root for every pair and
// divides in FP64: 50 M pairs 5.9 ms, here 0.85 ms for both passes).
// LIST = false: v [pair] = R / d' approximately.  LIST = true, for a window [P, Q]:
// with |sqrt(d'^2_32) - d'_64| <= eps = e0 + 2^-19 d' the ratio lies in
// [R / (d' + eps), R / (d' - eps)]; pairs that lie below P by that are counted, those
// above Q dropped, the rest listed with their node.  err bit 2: a path of more than
// GP_DEPTH nodes.
constexpr int GP_DEPTH = 1024;
struct GammaPair {
    int32_t a, b, node;
};
template <bool LIST>
__global__ void __launch_bounds__(256)
k_gamma_scan(const float *__restrict__ O32, int64_t n, const int32_t *__restrict__ leafOf,
             const int64_t *__restrict__ node, const double *__restrict__ rad, float *__restrict__ v, float e0, float P,
             float Q, unsigned long long *__restrict__ below, unsigned long long *__restrict__ nList,
             unsigned long long cap, GammaPair *__restrict__ list, int *__restrict__ err)
{
    __shared__ int sEnd[GP_DEPTH], sNode[GP_DEPTH];
    __shared__ float2 sR[GP_DEPTH];   // the radius rounded down and up
    __shared__ int sDepth;
    const int64_t a = blockIdx.x;
    const int lane = threadIdx.x & 31;
    const int la = leafOf[a];
    if (threadIdx.x == 0) {
        int64_t e = 0;
        int depth = 0;
        for (; depth < GP_DEPTH; depth++) {
            sNode[depth] = (int)e;
            sEnd[depth] = (int)node[e * 4 + 3];
            const int64_t x = node[e * 4], y = node[e * 4 + 1];
            if (x < 0) break;
            e = la < node[x * 4 + 3] ? x : y;
        }
        if (depth == GP_DEPTH) atomicOr(err, 2);
        sDepth = depth == GP_DEPTH ? GP_DEPTH - 1 : depth;   // the leaf's place
    }
    __syncthreads();
    const int depth = sDepth;
    for (int i = threadIdx.x; i <= depth; i += blockDim.x) {
        const double r = rad[sNode[i]];
        sR[i] = make_float2(__double2float_rd(r), __double2float_ru(r));
    }
    float oa[PM_MP];
#pragma unroll
    for (int j = 0; j < PM_MP; j++) oa[j] = O32[a * PM_MP + j];
    __syncthreads();
    const int64_t base = a * n - a * (a + 1) / 2 - a - 1;
    unsigned long long mine = 0;
    for (int64_t b0 = a + 1; b0 < n; b0 += blockDim.x) {
        const int64_t b = b0 + threadIdx.x;
        const bool ok = b < n;
        float d = 0.f;
        float2 R = make_float2(0.f, 0.f);
        int at = 0;
        if (ok) {
            const int lb = leafOf[b];
            // ends fall along the path: the last one beyond lb
            int lo = 0, hi = depth;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (sEnd[mid] > lb) lo = mid;
                else hi = mid - 1;
            }
            at = lo;
            R = sR[lo];
            float o[PM_MP];
#pragma unroll
            for (int j4 = 0; j4 < PM_MP / 4; j4++) {
                const float4 x = __ldg((const float4 *)(O32 + b * PM_MP) + j4);
                o[4 * j4] = x.x;
                o[4 * j4 + 1] = x.y;
                o[4 * j4 + 2] = x.z;
                o[4 * j4 + 3] = x.w;
            }
            d = __fsqrt_rn(pm_pd2_32(oa, o));
        }
        if (!LIST) {
            if (ok) v[base + b] = d > 0.f ? __fdividef(R.y, d) : (R.y > 0.f ? INFINITY : 0.f);
        } else {
            const float eps = __fmaf_ru(0x1.0p-19f, d, e0);
            // a radius of 0 gives the ratio 0 at any distance
            const bool under = R.y == 0.f ? P > 0.f : R.y < __fmul_rd(P, __fsub_rd(d, eps));
            const bool over = R.x > __fmul_ru(Q, __fadd_ru(d, eps));
            mine += ok && under ? 1 : 0;
            if (ok && !under && !over) {
                const unsigned long long slot = atomicAdd(nList, 1ull);
                if (slot < cap) {
                    GammaPair g;
                    g.a = (int32_t)a;
                    g.b = (int32_t)b;
                    g.node = sNode[at];
                    list[slot] = g;
                }
            }
        }
    }
    if (LIST) {
        for (int o = 16; o; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
        if (lane == 0 && mine) atomicAdd(below, mine);
    }
}

// Exact ratios of the listed pairs (k_gamma_ratio's arithmetic).
__global__ void __launch_bounds__(32)
k_gamma_exact(const double *__restrict__ O64, int m, const GammaPair *__restrict__ list,
              const unsigned long long *__restrict__ nList, unsigned long long cap, const double *__restrict__ rad,
              double *__restrict__ out)
{
    const unsigned long long n = *nList < cap ? *nList : cap, e = blockIdx.x * 32ull + threadIdx.x;
    if (e >= n) return;
    const GammaPair g = list[e];
    const double R = rad[g.node];
    const double dv = pm_pdist64(O64 + (int64_t)g.a * PM_MP, O64 + (int64_t)g.b * PM_MP, m);
    out[e] = dv > 0.0 ? __ddiv_rn(R, dv) : (R > 0.0 ? (double)INFINITY : 0.0);
}

// Histogram of w bits at `shift` of non-negative FP32 keys (their bits order like
// them) that share the bits above.
__global__ void __launch_bounds__(256)
k_gamma_hist32(const float *__restrict__ v, int64_t N, int shift, int w, unsigned int hiMask, unsigned int prefix,
               unsigned int *__restrict__ hist)
{
    __shared__ unsigned int h[2048];
    for (int i = threadIdx.x; i < (1 << w); i += blockDim.x) h[i] = 0u;
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const unsigned int k = __float_as_uint(v[e]);
        if ((k & hiMask) == prefix) atomicAdd(&h[(k >> shift) & ((1u << w) - 1u)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (1 << w); i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// 256-bin histogram of 8 bits at `shift` of the keys whose bits above them
// equal `prefix` (non-negative doubles and +inf order like their bits).
__global__ void k_gamma_hist(const unsigned long long *__restrict__ v, int64_t N, int shift,
                             unsigned long long hiMask, unsigned long long prefix, unsigned int *__restrict__ hist)
{
    __shared__ unsigned int h[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0u;
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long k = v[e];
        if ((k & hiMask) == prefix) atomicAdd(&h[(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Rows X[pos[i]] (leaf-order copy, row length ld) -> S[i] (row length d).
__global__ void k_gather_rows(const float *__restrict__ X, int ld, int d, const int64_t *__restrict__ pos,
                              int64_t ns, float *__restrict__ S)
{
    const int64_t i = blockIdx.x;
    if (i >= ns) return;
    const float *x = X + pos[i] * ld;
    for (int j = threadIdx.x; j < d; j += blockDim.x) S[i * d + j] = x[j];
}

// Cross-leaf pairs (a, b), a < b, of node subtrees whose FP32 projected
// squared distance is at most hiT, by tiles of CT x CT positions: a listed
// tile (`tiles`), or, without a list, the tiles of the one node [lo, hi) by
// the grid (x: columns, y: rows).  exact: only the pairs with FP64 projected
// distance < Rt (strict, Algorithm 4): |sqrt(d'^2_32) - d'_64| <= eps, so
// d'^2_32 < loT is surely in, > hiT surely out, and the rest is decided in
// FP64 (counted in fp64n); else the superset up to hiT, with the tile's node
// number beside each pair.
// Bound by instruction issue (about 45 per pair).  A thread holds one row and
// takes 16 columns out of shared memory; the kept pairs of a warp are counted
// first and take one atomic on the output counter.  A thread per row walking
// the whole node left most of the GPU idle: 1,265 nodes of 79 points on average
// took 94 ms in 1,265 launches, 0.08 ms in two tiled ones.
constexpr int CT = 64;
struct PairTile {
    int32_t a0, b0;   // first row and column position (b0 >= a0)
    int32_t hi;       // end of the node's positions
    int32_t node;     // number of the node in its batch
};

__global__ void __launch_bounds__(256)
k_cp_tiles(const float *__restrict__ O32, const double *__restrict__ O64, int m, const int32_t *__restrict__ leafOf,
           const PairTile *__restrict__ tiles, int64_t lo, int64_t hi, int exact, float loT, float hiT, double Rt,
           PairCand *__restrict__ out, int32_t *__restrict__ outNode, unsigned long long *cnt, unsigned long long cap,
           unsigned long long *fp64n)
{
    constexpr int NC = CT * CT / 256;   // columns per thread
    __shared__ float4 sO[CT][PM_MP / 4];
    __shared__ int sLeaf[CT];
    const int t = threadIdx.x, lane = t & 31, r = t & (CT - 1), part = t / CT;
    const int64_t rows = tiles ? 1 : (hi - lo + CT - 1) / CT;
    for (int64_t ty = blockIdx.y; ty < rows; ty += gridDim.y) {
        int64_t a0, b0, end;
        int node = 0;
        if (tiles) {
            const PairTile T = tiles[blockIdx.x];
            a0 = T.a0;
            b0 = T.b0;
            end = T.hi;
            node = T.node;
        } else {
            a0 = lo + ty * CT;
            b0 = lo + (int64_t)blockIdx.x * CT;
            end = hi;
            if (b0 < a0) continue;   // block-uniform
        }
        __syncthreads();
        {
            // CT columns of four float4 each: one per thread
            const int64_t b = b0 + (t >> 2);
            sO[t >> 2][t & 3] = b < end ? ((const float4 *)(O32 + b * PM_MP))[t & 3] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (t < CT) sLeaf[t] = b0 + t < end ? leafOf[b0 + t] : -1;
        }
        __syncthreads();
        const int64_t a = a0 + r;
        const bool av = a < end;
        float oa[PM_MP];
#pragma unroll
        for (int j4 = 0; j4 < PM_MP / 4; j4++) {
            const float4 v = av ? ((const float4 *)(O32 + a * PM_MP))[j4] : make_float4(0.f, 0.f, 0.f, 0.f);
            oa[4 * j4] = v.x;
            oa[4 * j4 + 1] = v.y;
            oa[4 * j4 + 2] = v.z;
            oa[4 * j4 + 3] = v.w;
        }
        const int la = av ? leafOf[a] : -1;
        float v[NC];
        unsigned keep = 0u;
#pragma unroll
        for (int c = 0; c < NC; c++) {
            const int cc = part * NC + c;
            v[c] = pm_pd2_32(oa, (const float *)sO[cc]);
            const int64_t b = b0 + cc;
            const int lb = sLeaf[cc];
            if (av && b > a && b < end && lb != la && v[c] <= hiT) keep |= 1u << c;
        }
        if (exact) {
#pragma unroll
            for (int c = 0; c < NC; c++)
                if (((keep >> c) & 1u) && !(v[c] < loT)) {
                    atomicAdd(fp64n, 1ull);
                    if (!(pm_pdist64(O64 + a * PM_MP, O64 + (b0 + part * NC + c) * PM_MP, m) < Rt)) keep &= ~(1u << c);
                }
        }
        const int mine = __popc(keep);
        int incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long base = 0;
        if (lane == 0 && total) base = atomicAdd(cnt, (unsigned long long)total);
        base = __shfl_sync(0xffffffffu, base, 0) + (unsigned long long)(incl - mine);
#pragma unroll
        for (int c = 0; c < NC; c++)
            if ((keep >> c) & 1u) {
                if (base < cap) {
                    PairCand pc;
                    pc.key = v[c];
                    pc.a = (int32_t)a;
                    pc.b = (int32_t)(b0 + part * NC + c);
                    out[base] = pc;
                    if (outNode) outNode[base] = node;
                }
                base++;
            }
    }
}

// Original-space FP32 squared distances of candidate pairs, into dst [n] or, if
// that is null, over the pairs' keys.
// Bound by the L2 reads of the two rows (8 ld bytes per pair, 24 ld^-1 flops
// per byte): eight lanes take a pair, so that every load instruction of the
// warp covers whole 128-byte lines of four pairs' rows, and four loads of each
// row are in flight per lane; consecutive pairs share rows, which L1 then
// holds.  The partial sums are added by a butterfly: the guard band of the
// selection, (ld + 8) 2^-24, holds for any order of the ld non-negative terms.
// Measured on 8.64 M pairs of 784 coordinates: 3.5 ms (15.6 TB/s of row reads
// out of L1 and L2) against 36.3 ms for a thread per pair with scalar loads.
// Requires ld % 32 == 0 (rows padded with zeros).
__global__ void __launch_bounds__(256)
k_pair_dist32(const float *__restrict__ X, int ld, PairCand *__restrict__ p, int64_t n, float *__restrict__ dst)
{
    const int lane = threadIdx.x & 31, grp = lane >> 3, g = lane & 7, nf4 = ld >> 2;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t e0 = (blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)) * 4; e0 < n; e0 += warps * 4) {
        const int64_t e = e0 + grp;
        float acc = 0.f;
        if (e < n) {
            const float4 *x = (const float4 *)(X + (int64_t)p[e].a * ld), *y = (const float4 *)(X + (int64_t)p[e].b * ld);
            float acc1 = 0.f;
            auto add = [&](const float4 u, const float4 v) {
                float t = __fsub_rn(u.x, v.x);
                acc = __fmaf_rn(t, t, acc);
                t = __fsub_rn(u.y, v.y);
                acc1 = __fmaf_rn(t, t, acc1);
                t = __fsub_rn(u.z, v.z);
                acc = __fmaf_rn(t, t, acc);
                t = __fsub_rn(u.w, v.w);
                acc1 = __fmaf_rn(t, t, acc1);
            };
            int c = g;
            for (; c + 24 < nf4; c += 32) {
                float4 u[4], v[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    u[i] = __ldg(x + c + 8 * i);
                    v[i] = __ldg(y + c + 8 * i);
                }
#pragma unroll
                for (int i = 0; i < 4; i++) add(u[i], v[i]);
            }
            for (; c < nf4; c += 8) add(__ldg(x + c), __ldg(y + c));
            acc = __fadd_rn(acc, acc1);
        }
        acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, 1));
        acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, 2));
        acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, 4));
        if (e < n && g == 0) {
            if (dst) dst[e] = acc;
            else p[e].key = acc;
        }
    }
}

// Launches k_pair_dist32: four pairs per warp and step, up to eight 256-thread
// blocks per SM.
void launch_pair_dist32(const pmlsh_index *ix, PairCand *p, int64_t n, cudaStream_t st, float *dst = nullptr)
{
    const unsigned grid = (unsigned)std::min<int64_t>((n + 31) / 32, 8 * 152);
    PM_LAUNCH("k_pair_dist32", st, k_pair_dist32<<<grid, 256, 0, st>>>(ix->X, ix->ld, p, n, dst));
}

// Histogram of key bits [sh, sh+w) among keys whose bits above sh+w equal
// `prefix` (radix select pass over a global buffer).
__global__ void k_pair_hist(const PairCand *__restrict__ p, int64_t n, int sh, int w, unsigned int hiMask,
                            unsigned int prefix, unsigned int *__restrict__ hist)
{
    __shared__ unsigned int h[2048];
    for (int i = threadIdx.x; i < (1 << w); i += blockDim.x) h[i] = 0;
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        unsigned int k = __float_as_uint(p[e].key);
        if ((k & hiMask) == (prefix & hiMask)) atomicAdd(&h[(k >> sh) & ((1u << w) - 1)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (1 << w); i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Entries with key <= thr, appended to `out` with FP64 distance (original or
// projected space) and original ids (i < j).
struct PairExact {
    double dist;
    int64_t i, j;
    int32_t a, b;   // positions
};

// (the entries' positions first, so that their FP64 sums fill whole warps: a warp's
// FP64 instruction takes as long for one entry as for 32)
__global__ void __launch_bounds__(256)
k_pair_pick(const PairCand *__restrict__ p, int64_t n, float thr, PairExact *__restrict__ out, unsigned long long *cnt,
            unsigned long long cap)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const PairCand c = p[e];
        if (!(c.key <= thr)) continue;
        const unsigned long long slot = atomicAdd(cnt, 1ull);
        if (slot >= cap) continue;
        out[slot].a = c.a;
        out[slot].b = c.b;
    }
}

__global__ void __launch_bounds__(32)
k_pair_exact(const float *__restrict__ X, int ld, int d, const double *__restrict__ O64, int m, int useProj,
             const int32_t *__restrict__ perm, PairExact *__restrict__ v, const unsigned long long *cnt,
             unsigned long long cap)
{
    const unsigned long long n = *cnt < cap ? *cnt : cap, e = blockIdx.x * 32ull + threadIdx.x;
    if (e >= n) return;
    PairExact x = v[e];
    x.dist = useProj ? pm_pdist64(O64 + (int64_t)x.a * PM_MP, O64 + (int64_t)x.b * PM_MP, m)
                     : pm_dist64(X + (int64_t)x.a * ld, X + (int64_t)x.b * ld, d);
    const int64_t ia = perm[x.a], ib = perm[x.b];
    x.i = ia < ib ? ia : ib;
    x.j = ia < ib ? ib : ia;
    v[e] = x;
}

__host__ __device__ __forceinline__ bool pe_less(const PairExact &x, const PairExact &y)
{
    if (x.dist != y.dist) return x.dist < y.dist;
    if (x.i != y.i) return x.i < y.i;
    return x.j < y.j;
}

// A batch of nodes [from, to) replayed for one value of ub: per node the
// candidates with FP64 projected distance < Rt (FP32 band as in k_cp_tiles) and
// the FP64 decisions taken, and, with FP64 distances, those that may enter the
// top-k (FP32 squared distance <= thr).  Entries of one node are mostly
// neighbours: lanes with the same node add once.
struct NodeExact {
    PairExact x;
    int32_t node;
    int32_t pad;
};

__global__ void __launch_bounds__(256)
k_cp_replay(const PairCand *__restrict__ cand, const int32_t *__restrict__ node, const float *__restrict__ d32,
            int64_t n, int from, int to, float loT, float hiT, double Rt, float thr, const float *__restrict__ X, int ld,
            int d, const double *__restrict__ O64, int m, const int32_t *__restrict__ perm, int *__restrict__ nodeCnt,
            int *__restrict__ nodeFp, NodeExact *__restrict__ out, unsigned long long *nOut, unsigned long long cap)
{
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    // (the last round is entered by whole warps)
    for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); e0 < n; e0 += step) {
        const int64_t e = e0 + lane;
        const int nd = e < n ? node[e] : -1;
        bool in = false, fp = false;
        PairCand c;
        if (nd >= from && nd < to) {
            c = cand[e];
            in = c.key < loT;
            if (!in && c.key <= hiT) {
                fp = true;
                in = pm_pdist64(O64 + (int64_t)c.a * PM_MP, O64 + (int64_t)c.b * PM_MP, m) < Rt;
            }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, nd);
        const unsigned ins = __ballot_sync(0xffffffffu, in) & peers, fps = __ballot_sync(0xffffffffu, fp) & peers;
        if (lane == __ffs(peers) - 1) {
            if (ins) atomicAdd(&nodeCnt[nd], __popc(ins));
            if (fps) atomicAdd(&nodeFp[nd], __popc(fps));
        }
        if (in && d32[e] <= thr) {
            const unsigned long long slot = atomicAdd(nOut, 1ull);
            if (slot < cap) {
                NodeExact y;
                y.x.dist = pm_dist64(X + (int64_t)c.a * ld, X + (int64_t)c.b * ld, d);
                const int64_t ia = perm[c.a], ib = perm[c.b];
                y.x.i = ia < ib ? ia : ib;
                y.x.j = ia < ib ? ib : ia;
                y.x.a = c.a;
                y.x.b = c.b;
                y.node = nd;
                y.pad = 0;
                out[slot] = y;
            }
        }
    }
}

// One block: sorts n (<= PAIR_SORT_CAP) entries by (dist, i, j) in place.
__global__ void k_pair_sort(PairExact *__restrict__ v, int n)
{
    extern __shared__ __align__(16) unsigned char psm[];
    PairExact *s = (PairExact *)psm;
    int P = 1;
    while (P < n) P <<= 1;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        if (i < n) s[i] = v[i];
        else { s[i].dist = INFINITY; s[i].i = 0x7fffffffffffffffLL; s[i].j = 0x7fffffffffffffffLL; s[i].a = s[i].b = -1; }
    }
    __syncthreads();
    for (int k2 = 2; k2 <= P; k2 <<= 1)
        for (int j = k2 >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < P; i += blockDim.x) {
                int ixj = i ^ j;
                if (ixj > i) {
                    bool up = (i & k2) == 0;
                    if (pe_less(s[ixj], s[i]) == up) {
                        PairExact t = s[i]; s[i] = s[ixj]; s[ixj] = t;
                    }
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] = s[i];
}


// ------------------------------------------- Algorithm 3 (branch and bound)

// All pairs inside leaf l keyed by their FP32 projected squared distance.
// One block per leaf.
__global__ void k_bnb_selfjoin(const float *__restrict__ O32, const int64_t *__restrict__ off,
                               const int64_t *__restrict__ pairOff, PairCand *__restrict__ out)
{
    const int64_t l = blockIdx.x;
    const int64_t p0 = off[l], s = off[l + 1] - p0;
    const int64_t np = s * (s - 1) / 2;
    for (int64_t e = threadIdx.x; e < np; e += blockDim.x) {
        int64_t i = 0, rem = e;
        while (rem >= s - 1 - i) { rem -= s - 1 - i; i++; }
        const int64_t j = i + 1 + rem;
        PairCand pc;
        pc.key = pm_pd2_32(O32 + (p0 + i) * PM_MP, O32 + (p0 + j) * PM_MP);
        pc.a = (int32_t)(p0 + i);
        pc.b = (int32_t)(p0 + j);
        out[pairOff[l] + e] = pc;
    }
}

struct LeafPair {
    float md;      // lower bound of the projected distance of any pair in l1 x l2
    int32_t l1, l2;
};

// Mindist of Sec. 6.1 for leaf pairs (l1, l2), l1 < l2: the larger of
// ||RO1, RO2|| - r1 - r2 and the gaps between the pivot rings, from the leaf
// entries (FP32, rounded so that it stays a lower bound).  Pairs with Mindist in
// (dLo, dT] are listed, up to cap, and counted.  Bound by FP32 issue,
// about 70 instructions per pair: a block takes 128 leaves l1, a record per thread
// in registers, and reads its share of the l2 records (grid.y slices) through shared
// memory, 32 at a time, instead of each thread reading every 160-byte record from
// L2; the listed pairs of a warp take one atomic.  22,125 leaves (245 M pairs):
// 1.2 ms, 9.1 before.
constexpr int BM_T = 128;
__global__ void __launch_bounds__(BM_T)
k_bnb_mindist(const float *__restrict__ meta, int s, int64_t L, float dLo, float dT, LeafPair *__restrict__ out,
              unsigned long long *cnt, unsigned long long cap)
{
    __shared__ __align__(16) float sM[32][PM_LEAF_STRIDE];
    const int t = threadIdx.x, lane = t & 31;
    const int64_t a0 = (int64_t)blockIdx.x * BM_T, l1 = a0 + t;
    const bool v1 = l1 < L;
    float o[PM_MP], hn[PM_MAX_PIVOTS], hx[PM_MAX_PIVOTS];
    const float *M1 = meta + (v1 ? l1 : 0) * PM_LEAF_STRIDE;
#pragma unroll
    for (int j = 0; j < PM_MP; j++) o[j] = M1[j];
    const float r1 = M1[16];
#pragma unroll
    for (int i = 0; i < PM_MAX_PIVOTS; i++) {
        // pivots beyond s give no gap
        hn[i] = i < s ? M1[24 + i] : -INFINITY;
        hx[i] = i < s ? M1[32 + i] : INFINITY;
    }
    // l2 tiles of 32 from the block's first possible one
    const int64_t t0 = (a0 + 1) / 32, nT = (L + 31) / 32;
    for (int64_t tile = t0 + blockIdx.y; tile < nT; tile += gridDim.y) {
        const int64_t b0 = tile * 32;
        const int nb = L - b0 < 32 ? (int)(L - b0) : 32;
        __syncthreads();
        for (int e = t; e < nb * (PM_LEAF_STRIDE / 4); e += BM_T)
            ((float4 *)&sM[0][0])[e] = __ldg((const float4 *)(meta + b0 * PM_LEAF_STRIDE) + e);
        __syncthreads();
        for (int c = 0; c < nb; c++) {
            const float *M2 = sM[c];
            const float dc = __fsqrt_rn(pm_pd2_32(o, M2));
            float md = __fsub_rn(__fsub_rn(__fmul_rn(dc, 1.f - 1e-5f), r1), M2[16]);
#pragma unroll
            for (int i = 0; i < PM_MAX_PIVOTS; i++) {
                if (i < s) {
                    // rings [min, max] of the two leaves (already widened outwards)
                    md = fmaxf(md, __fsub_rn(M2[24 + i], hx[i]));
                    md = fmaxf(md, __fsub_rn(hn[i], M2[32 + i]));
                }
            }
            const bool in = v1 && b0 + c > l1 && md > dLo && md <= dT;
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (m == 0u) continue;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(cnt, (unsigned long long)__popc(m));
            base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
            if (in && base < cap) {
                LeafPair lp;
                lp.md = md;
                lp.l1 = (int32_t)l1;
                lp.l2 = (int32_t)(b0 + c);
                out[base] = lp;
            }
        }
    }
}

// Listed leaf pairs in ascending (Mindist, l1, l2) on the device: a 64-bit
// key per pair, the order-preserving bits of Mindist (+0 and -0 taken as
// one) above the pair's rank in (l1, l2) order, l1 (2L - l1 - 1) / 2 +
// l2 - l1 - 1 (below 2^32 when L(L - 1)/2 is), sorted by a stable LSD radix
// sort of 8-bit digits and decoded back.
constexpr int RS_THREADS = 256, RS_ITEMS = 32;   // keys per block and pass: 8,192
constexpr int64_t LP_GPU_MAX_L = 92682;         // L (L - 1) / 2 < 2^32

__device__ __forceinline__ int64_t lp_rank_base(int64_t l1, int64_t L) { return l1 * (2 * L - l1 - 1) / 2; }

__global__ void k_lp_key(const LeafPair *__restrict__ lp, int64_t n, int64_t L, unsigned long long *__restrict__ key)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const LeafPair x = lp[e];
    const unsigned int u = __float_as_uint(__fadd_rn(x.md, 0.f));
    const unsigned int ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    const int64_t rk = lp_rank_base(x.l1, L) + (x.l2 - x.l1 - 1);
    key[e] = ((unsigned long long)ord << 32) | (unsigned long long)(uint32_t)rk;
}

// digit counts of each block's keys, digit-major: hist[d * nb + block]
__global__ void __launch_bounds__(RS_THREADS)
k_rs_hist(const unsigned long long *__restrict__ key, int64_t n, int shift, unsigned int *__restrict__ hist, int nb)
{
    __shared__ unsigned int h[256];
    h[threadIdx.x] = 0u;
    __syncthreads();
    const int64_t b0 = (int64_t)blockIdx.x * RS_THREADS * RS_ITEMS;
    const int64_t b1 = b0 + (int64_t)RS_THREADS * RS_ITEMS < n ? b0 + (int64_t)RS_THREADS * RS_ITEMS : n;
    for (int64_t e = b0 + threadIdx.x; e < b1; e += RS_THREADS) atomicAdd(&h[(unsigned)(key[e] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(int64_t)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

// exclusive prefix sums of each digit's row h[d nb, (d + 1) nb) in place, a block
// per digit, and the rows' totals
__global__ void __launch_bounds__(256) k_rs_scan(unsigned int *__restrict__ h, int nb, unsigned int *__restrict__ total)
{
    __shared__ unsigned int ws[8];
    unsigned int *row = h + (int64_t)blockIdx.x * nb;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned int carry = 0u;
    for (int i0 = 0; i0 < nb; i0 += 256) {
        const unsigned int v = i0 + t < nb ? row[i0 + t] : 0u;
        unsigned int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) ws[w] = incl;
        __syncthreads();
        unsigned int before = 0u, all = 0u;
        for (int i = 0; i < 8; i++) {
            before += i < w ? ws[i] : 0u;
            all += ws[i];
        }
        if (i0 + t < nb) row[i0 + t] = carry + before + incl - v;
        carry += all;
        __syncthreads();
    }
    if (t == 0) total[blockIdx.x] = carry;
}

// stable scatter by one digit: each block walks its keys in order, 256 per
// round; a key's place is its digit's running base plus the keys of that
// digit before it in the round (earlier warps, then earlier lanes)
__global__ void __launch_bounds__(RS_THREADS)
k_rs_scatter(const unsigned long long *__restrict__ in, unsigned long long *__restrict__ out, int64_t n, int shift,
             const unsigned int *__restrict__ off, const unsigned int *__restrict__ total, int nb)
{
    constexpr int NW = RS_THREADS / 32;
    __shared__ unsigned int base[256];
    __shared__ unsigned int wc[NW][256];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    {
        // a digit's first place: the totals of the digits before it
        const unsigned int v = total[t];
        unsigned int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) wc[0][w] = incl;
        __syncthreads();
        unsigned int before = 0u;
        for (int i = 0; i < w; i++) before += wc[0][i];
        __syncthreads();
        base[t] = off[(int64_t)t * nb + blockIdx.x] + before + incl - v;
    }
    const int64_t b0 = (int64_t)blockIdx.x * RS_THREADS * RS_ITEMS;
    for (int r = 0; r < RS_ITEMS; r++) {
        for (int j = 0; j < NW; j++) wc[j][t] = 0u;
        __syncthreads();
        const int64_t e = b0 + (int64_t)r * RS_THREADS + t;
        const bool valid = e < n;
        const unsigned long long k = valid ? in[e] : 0ull;
        const unsigned int d = valid ? ((unsigned)(k >> shift) & 255u) : 256u;
        const unsigned int peers = __match_any_sync(0xffffffffu, d);
        const int rankW = __popc(peers & ((1u << lane) - 1u));
        if (valid && rankW == 0) wc[w][d] = (unsigned)__popc(peers);
        __syncthreads();
        if (valid) {
            unsigned int pos = base[d] + (unsigned)rankW;
            for (int j = 0; j < w; j++) pos += wc[j][d];
            out[pos] = k;
        }
        __syncthreads();
        unsigned int add = 0u;
        for (int j = 0; j < NW; j++) add += wc[j][t];
        base[t] += add;
        __syncthreads();
    }
}

// keys back to leaf pairs; flags a key out of order (bit 1) or a rank that
// does not decode to l1 < l2 < L (bit 2)
__global__ void k_lp_decode(const unsigned long long *__restrict__ key, int64_t n, int64_t L,
                            LeafPair *__restrict__ out, int *__restrict__ bad)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n) return;
    const unsigned long long k = key[e];
    if (e > 0 && key[e - 1] > k) atomicOr(bad, 1);
    const unsigned int ord = (unsigned int)(k >> 32);
    const unsigned int u = (ord & 0x80000000u) ? (ord & 0x7fffffffu) : ~ord;
    const int64_t rk = (int64_t)(k & 0xffffffffull);
    // l1: the largest l with lp_rank_base(l) <= rk (root of the quadratic,
    // then at most a few steps of correction)
    const double A = 2.0 * (double)L - 1.0;
    const double disc = A * A - 8.0 * (double)rk;
    int64_t l1 = (int64_t)floor((A - sqrt(disc > 0.0 ? disc : 0.0)) * 0.5);
    l1 = l1 < 0 ? 0 : (l1 > L - 2 ? L - 2 : l1);
    for (int it = 0; it < 4 && l1 + 1 <= L - 2 && lp_rank_base(l1 + 1, L) <= rk; it++) l1++;
    for (int it = 0; it < 4 && l1 > 0 && lp_rank_base(l1, L) > rk; it++) l1--;
    const int64_t l2 = rk - lp_rank_base(l1, L) + l1 + 1;
    LeafPair x;
    x.md = __uint_as_float(u);
    x.l1 = (int32_t)l1;
    x.l2 = (int32_t)l2;
    if (!(l1 >= 0 && l1 < l2 && l2 < L)) {
        atomicOr(bad, 2);
        x.l1 = 0;
        x.l2 = 1;
    }
    out[e] = x;
}

// State of the T-cut on the device: the selection's progress, the band of its last
// key, and the bound dT of the T-th projected distance that the search stops at.
struct CutState {
    unsigned long long need;      // rank left inside the selected prefix
    unsigned long long nBelow, nBand;   // counters of the last split
    unsigned long long fp64;      // band entries of all cuts
    unsigned int prefix;          // bits of the T-th key found so far
    int err;                      // 1: a band did not fit or did not hold the cut
    float lo, hi;                 // FP32 band of the T-th key
    int below;                    // keys below lo exist (its distance is above the error)
    int pad;
    double dT;                    // upper bound of the T-th projected distance
};
// What the next batch of listed leaf pairs takes.
struct BatchPlan {
    long long end, tot;           // leaf pairs [next, end), their cross pairs
    unsigned long long fp64;
    double dT;
    int err, stop;                // stop: the first pair's Mindist exceeds dT
};

// Sizes na nb of the listed leaf pairs, and per block of 1,024 their sum.
__global__ void __launch_bounds__(1024)
k_lp_size(const LeafPair *__restrict__ lp, int64_t n, const int64_t *__restrict__ off, int64_t *__restrict__ pre,
          int64_t *__restrict__ blk)
{
    __shared__ int64_t ws[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int64_t e = blockIdx.x * 1024ll + t;
    int64_t v = 0;
    if (e < n) {
        const LeafPair x = lp[e];
        v = (off[x.l1 + 1] - off[x.l1]) * (off[x.l2 + 1] - off[x.l2]);
    }
    int64_t incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    if (w == 0) {
        int64_t x = ws[lane], xi = x;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += y;
        }
        ws[lane] = xi - x;
        if (lane == 31) blk[blockIdx.x] = xi;
    }
    __syncthreads();
    if (e < n) pre[e] = ws[w] + incl - v;   // exclusive, inside the block
}
// exclusive prefix sums of blk [nb] in place, one block
__global__ void __launch_bounds__(1024) k_lp_scan(int64_t *__restrict__ blk, int nb)
{
    __shared__ int64_t ws[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int64_t carry = 0;
    for (int i0 = 0; i0 < nb; i0 += 1024) {
        const int64_t v = i0 + t < nb ? blk[i0 + t] : 0;
        int64_t incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) ws[w] = incl;
        __syncthreads();
        int64_t before = 0, all = 0;
        for (int i = 0; i < 32; i++) {
            before += i < w ? ws[i] : 0;
            all += ws[i];
        }
        if (i0 + t < nb) blk[i0 + t] = carry + before + incl - v;
        carry += all;
        __syncthreads();
    }
}

// The batch that starts at listed pair `next`: at most maxPairs leaf pairs, Mindist
// <= dT, and (beyond the first) at most cap cross pairs.  One warp: 32-way searches.
__global__ void __launch_bounds__(32)
k_bnb_plan(const LeafPair *__restrict__ lp, const int64_t *__restrict__ pre, const int64_t *__restrict__ blk,
           const int64_t *__restrict__ off, int64_t n, int64_t next, int64_t maxPairs, int64_t cap,
           const CutState *__restrict__ st, BatchPlan *__restrict__ out)
{
    const int lane = threadIdx.x;
    const double dT = st->dT;
    auto at = [&](int64_t e) { return pre[e] + blk[e >> 10]; };
    auto size = [&](int64_t e) {
        const LeafPair x = lp[e];
        return (off[x.l1 + 1] - off[x.l1]) * (off[x.l2 + 1] - off[x.l2]);
    };
    const int64_t base = at(next);
    // first index in [next, hi) that a batch may not hold (ok is true, then false)
    int64_t lo = next, hi = next + maxPairs < n ? next + maxPairs : n;
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) / 32, e = lo + lane * step;
        bool ok = false;
        if (e < hi) ok = (double)lp[e].md <= dT && (e == next || at(e) - base + size(e) <= cap);
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        const int k = m == 0xffffffffu ? 32 : __ffs(~m) - 1;   // probes 0 .. k - 1 hold
        if (k == 0) {
            hi = lo;
        } else {
            const int64_t nlo = lo + (k - 1) * step + 1, nhi = k < 32 ? lo + k * step : hi;
            lo = nlo;
            hi = nhi < hi ? nhi : hi;
        }
    }
    if (lane == 0) {
        BatchPlan p;
        p.end = lo;
        p.tot = lo > next ? at(lo - 1) - base + size(lo - 1) : 0;
        p.fp64 = st->fp64;
        p.dT = dT;
        p.err = st->err;
        p.stop = !((double)lp[next].md <= dT);
        *out = p;
    }
}

// Every cross pair of the listed leaf pairs [first, end), keyed by the FP32 projected
// squared distance, appended behind cnt.  A warp per leaf pair.  cut: after a first
// cut, pairs beyond the last one's band (key > hi) cannot be among the T nearest.
__global__ void __launch_bounds__(256)
k_bnb_cross(const float *__restrict__ O32, const int64_t *__restrict__ off, const LeafPair *__restrict__ lp,
            int64_t first, int64_t end, int cut, const CutState *__restrict__ st, PairCand *__restrict__ out,
            unsigned long long *cnt)
{
    const int lane = threadIdx.x & 31;
    const int64_t l = first + blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (l >= end) return;   // warp-uniform
    const float hi = cut ? st->hi : INFINITY;
    const LeafPair pr = lp[l];
    const int64_t a0 = off[pr.l1], na = off[pr.l1 + 1] - a0;
    const int64_t b0 = off[pr.l2], nb = off[pr.l2 + 1] - b0;
    for (int64_t e0 = 0; e0 < na * nb; e0 += 32) {
        const int64_t e = e0 + lane;
        PairCand pc;
        pc.key = INFINITY;
        bool in = e < na * nb;
        if (in) {
            const int64_t ia = e / nb, ib = e - ia * nb;
            pc.key = pm_pd2_32(O32 + (a0 + ia) * PM_MP, O32 + (b0 + ib) * PM_MP);
            pc.a = (int32_t)(a0 + ia);
            pc.b = (int32_t)(b0 + ib);
            in = !cut || pc.key <= hi;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (m == 0u) continue;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(cnt, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
        if (in) out[base] = pc;
    }
}

// The T-th smallest FP32 key of p[0, *n) by three histogram passes of 11, 11 and 10
// bits, on the device: k_cut_hist counts the keys that share the prefix, k_cut_bin
// extends it (and, after the last pass, forms the FP32 band that the FP64 distance
// of the T-th pair can lie in).
__global__ void __launch_bounds__(256)
k_cut_hist(const PairCand *__restrict__ p, const unsigned long long *__restrict__ np, int pass,
           const CutState *__restrict__ st, unsigned int *__restrict__ hist)
{
    __shared__ unsigned int h[2048];
    const int sh = pass == 0 ? 21 : (pass == 1 ? 10 : 0), w = pass == 2 ? 10 : 11;
    const unsigned int hiMask = pass == 0 ? 0u : (0xffffffffu << (sh + w)), prefix = pass == 0 ? 0u : st->prefix;
    for (int i = threadIdx.x; i < (1 << w); i += blockDim.x) h[i] = 0;
    __syncthreads();
    const int64_t n = (int64_t)*np;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const unsigned int k = __float_as_uint(p[e].key);
        if ((k & hiMask) == (prefix & hiMask)) atomicAdd(&h[(k >> sh) & ((1u << w) - 1)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (1 << w); i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

__global__ void __launch_bounds__(1024)
k_cut_bin(unsigned int *__restrict__ hist, int pass, unsigned long long T, double maxNorm, CutState *__restrict__ st)
{
    __shared__ unsigned long long ws[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int sh = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
    const unsigned long long need = pass == 0 ? T : st->need;
    const unsigned int prefix = pass == 0 ? 0u : st->prefix;
    const unsigned int h0 = hist[2 * t], h1 = hist[2 * t + 1];   // (the last pass's upper half is zero)
    unsigned long long incl = (unsigned long long)h0 + h1;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) ws[w] = incl;
    hist[2 * t] = 0u;   // for the next pass
    hist[2 * t + 1] = 0u;
    __syncthreads();
    unsigned long long before = 0;
    for (int i = 0; i < w; i++) before += ws[i];
    const unsigned long long ex = before + incl - h0 - h1;
    if (ex < need && need <= ex + h0 + h1) {
        const bool first = need <= ex + h0;
        const unsigned int pf = prefix | ((unsigned int)(first ? 2 * t : 2 * t + 1) << sh);
        st->prefix = pf;
        st->need = need - ex - (first ? 0u : h0);
        if (pass == 2) {
            const double tau = __dsqrt_rn((double)__uint_as_float(pf));
            const double eps = __dadd_rn(__dadd_rn(__dmul_rn(0x1.0p-22, maxNorm), __dmul_rn(0x1.0p-19, tau)), 1e-300);
            const double loD = __dsub_rn(tau, __dmul_rn(2.0, eps)), hiD = __dadd_rn(tau, __dmul_rn(2.0, eps));
            st->below = loD > 0.0;
            st->lo = loD > 0.0 ? __double2float_rd(__dmul_rn(loD, loD)) : 0.f;
            st->hi = __double2float_ru(__dmul_rn(hiD, hiD));
            st->nBelow = 0;
            st->nBand = 0;
            st->dT = fmin(st->dT, __dadd_rn(tau, eps));
        }
    }
}

// Keys below the band go to out in order, 2,048 pairs per block and step with one
// atomic; keys inside it to the band list (their FP64 distances follow packed, in
// k_cut_band).  Bound by HBM, 24 bytes per kept pair: 8.6 M pairs 35 us; one atomic
// per kept pair and a copy back took 235.
__global__ void __launch_bounds__(256)
k_cut_split(const PairCand *__restrict__ p, const unsigned long long *__restrict__ np, PairCand *__restrict__ out,
            PairExact *__restrict__ band, unsigned long long cap, CutState *__restrict__ st)
{
    constexpr int PER = 8;
    __shared__ unsigned int cw[PER * 8];   // kept pairs per step of 256 and warp, then their places
    __shared__ unsigned long long sBase;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const float lo = st->lo, hi = st->hi;
    const bool below = st->below != 0;
    const int64_t n = (int64_t)*np;
    for (int64_t b0 = blockIdx.x * (int64_t)(256 * PER); b0 < n; b0 += (int64_t)gridDim.x * 256 * PER) {
        PairCand c[PER];
        unsigned int m[PER];
#pragma unroll
        for (int u = 0; u < PER; u++) {
            const int64_t e = b0 + u * 256 + t;
            c[u].key = INFINITY;
            if (e < n) c[u] = p[e];
        }
#pragma unroll
        for (int u = 0; u < PER; u++) {
            const bool v = b0 + u * 256 + t < n;
            m[u] = __ballot_sync(0xffffffffu, v && below && c[u].key < lo);
            if (lane == 0) cw[u * 8 + w] = __popc(m[u]);
            if (v && (!below || c[u].key >= lo) && c[u].key <= hi) {
                const unsigned long long slot = atomicAdd(&st->nBand, 1ull);
                if (slot < cap) {
                    band[slot].a = c[u].a;
                    band[slot].b = c[u].b;
                }
            }
        }
        __syncthreads();
        if (w == 0) {
            const unsigned int x = cw[lane], y = cw[32 + lane];
            unsigned int ix = x, iy = y;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int p0 = __shfl_up_sync(0xffffffffu, ix, o), p1 = __shfl_up_sync(0xffffffffu, iy, o);
                if (lane >= o) {
                    ix += p0;
                    iy += p1;
                }
            }
            const unsigned int half = __shfl_sync(0xffffffffu, ix, 31), all = half + __shfl_sync(0xffffffffu, iy, 31);
            cw[lane] = ix - x;
            cw[32 + lane] = half + iy - y;
            if (lane == 0) sBase = all ? atomicAdd(&st->nBelow, (unsigned long long)all) : 0ull;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; u++)
            if ((m[u] >> lane) & 1u) out[sBase + cw[u * 8 + w] + __popc(m[u] & ((1u << lane) - 1u))] = c[u];
        __syncthreads();
    }
}

// FP64 projected distances and ids of the band's pairs, 32 per warp.
__global__ void __launch_bounds__(32)
k_cut_band(PairExact *__restrict__ band, unsigned long long cap, const double *__restrict__ O64, int m,
           const int32_t *__restrict__ perm, const CutState *__restrict__ st)
{
    const unsigned long long n = st->nBand < cap ? st->nBand : cap, e = blockIdx.x * 32ull + threadIdx.x;
    if (e >= n) return;
    PairExact x = band[e];
    x.dist = pm_pdist64(O64 + (int64_t)x.a * PM_MP, O64 + (int64_t)x.b * PM_MP, m);
    const int64_t ia = perm[x.a], ib = perm[x.b];
    x.i = ia < ib ? ia : ib;
    x.j = ia < ib ? ib : ia;
    band[e] = x;
}

// The band's first T - nBelow entries by (FP64 projected distance, i, j) join out,
// each placed by its rank among them; *np becomes T.
__global__ void __launch_bounds__(128)
k_cut_fill(const PairExact *__restrict__ band, unsigned long long cap, unsigned long long T, PairCand *__restrict__ out,
           unsigned long long *__restrict__ np, CutState *__restrict__ st)
{
    __shared__ ulonglong2 s[128];   // distance bits (>= +0: they order like it), ids i 2^32 + j
    const unsigned long long nBand = st->nBand, nBelow = st->nBelow;
    if (nBand > cap || nBelow > T || nBelow + nBand < T) {
        if (blockIdx.x == 0 && threadIdx.x == 0) st->err = 1;
        return;   // (uniform over the grid)
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->fp64 += nBand;
        *np = T;
    }
    const unsigned long long need = T - nBelow, e = blockIdx.x * 128ull + threadIdx.x;
    if (blockIdx.x * 128ull >= nBand) return;   // block-uniform
    auto key = [](const PairExact &x) {
        return make_ulonglong2((unsigned long long)__double_as_longlong(x.dist),
                               ((unsigned long long)x.i << 32) | (unsigned long long)x.j);
    };
    const bool v = e < nBand;
    const PairExact x = band[v ? e : 0];
    const ulonglong2 kx = key(x);
    unsigned int rank = 0;
    for (unsigned long long f0 = 0; f0 < nBand; f0 += 128) {
        __syncthreads();
        s[threadIdx.x] = f0 + threadIdx.x < nBand ? key(band[f0 + threadIdx.x]) : make_ulonglong2(~0ull, ~0ull);
        __syncthreads();
#pragma unroll 4
        for (int f = 0; f < 128; f++) rank += s[f].x < kx.x || (s[f].x == kx.x && s[f].y < kx.y) ? 1 : 0;
    }
    if (v && rank < need) {
        PairCand pc;
        pc.key = 0.f;
        pc.a = x.a;
        pc.b = x.b;
        out[nBelow + rank] = pc;
    }
}

template <class T> pmlsh_status dalloc(T **p, size_t count)
{
    PM_CUDA(cudaMalloc((void **)p, std::max<size_t>(1, count) * sizeof(T)));
    return PMLSH_OK;
}

struct DevPtrs {
    std::vector<void *> ps;
    ~DevPtrs() { for (void *p : ps) cudaFree(p); }
    template <class T> pmlsh_status get(T **p, size_t n)
    {
        PM_TRY(dalloc(p, n));
        ps.push_back(*p);
        return PMLSH_OK;
    }
};

// FP64 ball radii of the index's nodes into dRad [N] (device); innerOnly: the
// leaf nodes' entries are left at 0.
pmlsh_status node_radii(const pmlsh_index *ix, bool innerOnly, DevPtrs &mem, double **dRad, cudaStream_t st)
{
    const int64_t N = (int64_t)ix->nodeLo.size();
    std::vector<NodeSlice> sl;
    sl.reserve((size_t)N);
    for (int64_t e = 0; e < N; e++) {
        if (innerOnly && ix->nodeLeft[e] < 0) continue;
        const int64_t lo = ix->leafOffH[ix->nodeLo[e]], hi = ix->leafOffH[ix->nodeHi[e]];
        for (int64_t a = lo; a < hi; a += NB_SLICE) sl.push_back(NodeSlice{a, std::min(hi, a + NB_SLICE), (int32_t)e, 0});
    }
    const int64_t ns = (int64_t)sl.size();
    NodeSlice *dSl;
    long long *box;
    PM_TRY(mem.get(&dSl, (size_t)ns));
    PM_TRY(mem.get(&box, (size_t)N * 2 * PM_MP));
    PM_TRY(mem.get(dRad, (size_t)N));
    PM_CUDA(cudaMemcpyAsync(dSl, sl.data(), (size_t)ns * sizeof(NodeSlice), cudaMemcpyHostToDevice, st));
    PM_LAUNCH("k_node_box_init", st, k_node_box_init<<<(unsigned)((N * 2 * PM_MP + 255) / 256), 256, 0, st>>>(
        box, (unsigned long long *)*dRad, N));
    if (ns > 0) {
        const unsigned g = (unsigned)((ns + 7) / 8);
        PM_LAUNCH("k_node_box", st, k_node_box<<<g, 256, 0, st>>>(ix->O64, dSl, ns, box));
        PM_LAUNCH("k_node_radius", st, k_node_radius<<<g, 256, 0, st>>>(ix->O64, dSl, ns, box, ix->m,
                                                                        (unsigned long long *)*dRad));
    }
    PM_CUDA(cudaGetLastError());
    return PMLSH_OK;
}

// Radix select over a device pair buffer: the rank-th smallest FP32 key
// (1-based).  Three passes of 11/11/10 bits.
pmlsh_status pair_kth(const PairCand *p, int64_t n, int64_t rank, unsigned int *hist, float *out, cudaStream_t st)
{
    unsigned int prefix = 0;
    int64_t need = rank;
    const int shifts[3] = {21, 10, 0}, widths[3] = {11, 11, 10};
    std::vector<unsigned int> hh(2048);
    for (int pass = 0; pass < 3; pass++) {
        const int sh = shifts[pass], w = widths[pass];
        const unsigned int hiMask = pass == 0 ? 0u : (0xffffffffu << (sh + w));
        PM_CUDA(cudaMemsetAsync(hist, 0, sizeof(unsigned int) * 2048, st));
        int grid = (int)std::min<int64_t>(1024, (n + 255) / 256);
        PM_LAUNCH("k_pair_hist", st, k_pair_hist<<<std::max(1, grid), 256, 0, st>>>(p, n, sh, w, hiMask, prefix, hist));
        PM_CUDA(cudaMemcpyAsync(hh.data(), hist, sizeof(unsigned int) * (1u << w), cudaMemcpyDeviceToHost, st));
        PM_CUDA(cudaStreamSynchronize(st));
        int64_t acc = 0;
        int bin = 0;
        for (; bin < (1 << w); bin++) {
            if (acc + (int64_t)hh[bin] >= need) break;
            acc += hh[bin];
        }
        need -= acc;
        prefix |= (unsigned int)bin << sh;
    }
    float f;
    std::memcpy(&f, &prefix, sizeof(f));
    *out = f;
    return PMLSH_OK;
}

// Entries of p[0, n) with key <= thr into out (at most cap, counted in cnt) with
// their FP64 distance (original space, or projected) and ids.
void launch_pair_collect(const pmlsh_index *ix, const PairCand *p, int64_t n, float thr, int useProj, PairExact *out,
                         unsigned long long *cnt, unsigned long long cap, cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 16 * 152);
    PM_LAUNCH("k_pair_pick", st, k_pair_pick<<<grid, 256, 0, st>>>(p, n, thr, out, cnt, cap));
    PM_LAUNCH("k_pair_exact", st, k_pair_exact<<<(unsigned)((cap + 31) / 32), 32, 0, st>>>(
        ix->X, ix->ld, ix->d, ix->O64, ix->m, useProj, ix->perm, out, cnt, cap));
}

// Exact top-k merge: the current list `top` (sorted by (dist, i, j), FP64
// distances, size kc <= k) and the candidate buffer p[0, n) with FP32
// original-space squared distances.  A candidate can enter only if its FP32
// value is <= min(K32 (1 + 3 eps_v), D_k^2 (1 + 3 eps_v)) (K32: k-th smallest
// FP32 candidate value, D_k: current k-th distance); those are recomputed in
// FP64 and sorted with the current list.
struct TopK {
    std::vector<PairExact> v;   // host copy, sorted
};

pmlsh_status pair_merge(TopK &top, int k, const PairCand *p, int64_t n, const pmlsh_index *ix, unsigned int *hist,
                        PairExact *scratch, unsigned long long *cnt, cudaStream_t st)
{
    if (n <= 0) return PMLSH_OK;
    const double epsv = (double)(ix->ld + 8) * 0x1.0p-24;
    double thr = INFINITY;
    if (n >= k) {
        float K32;
        PM_TRY(pair_kth(p, n, k, hist, &K32, st));
        thr = (double)K32 * (1.0 + 3.0 * epsv) + 1e-36;
    }
    if ((int)top.v.size() >= k) {
        double Dk = top.v[k - 1].dist;
        thr = std::min(thr, Dk * Dk * (1.0 + 3.0 * epsv) + 1e-36);
    }
    float thr32 = std::isinf(thr) ? INFINITY : (float)thr;
    if (!std::isinf(thr) && (double)thr32 < thr) thr32 = nextafterf(thr32, INFINITY);
    PM_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st));
    const unsigned long long cap = PAIR_SORT_CAP - (unsigned long long)top.v.size();
    launch_pair_collect(ix, p, n, thr32, 0, scratch + top.v.size(), cnt, cap, st);
    PM_CUDA(cudaGetLastError());
    unsigned long long got = 0;
    PM_CUDA(cudaMemcpyAsync(&got, cnt, sizeof(got), cudaMemcpyDeviceToHost, st));
    PM_CUDA(cudaStreamSynchronize(st));
    if (got > cap) {
        pm_set_error("closest pairs: %llu candidates tied inside the FP32 guard band (capacity %llu)", got, cap);
        return PMLSH_EINTERNAL;
    }
    const int tot = (int)(top.v.size() + got);
    if (!top.v.empty())
        PM_CUDA(cudaMemcpyAsync(scratch, top.v.data(), top.v.size() * sizeof(PairExact), cudaMemcpyHostToDevice, st));
    int P = 1;
    while (P < tot) P <<= 1;
    PM_LAUNCH("k_pair_sort", st, k_pair_sort<<<1, 1024, (size_t)P * sizeof(PairExact), st>>>(scratch, tot));
    PM_CUDA(cudaGetLastError());
    const int keep = std::min(tot, k);
    top.v.resize(keep);
    PM_CUDA(cudaMemcpyAsync(top.v.data(), scratch, keep * sizeof(PairExact), cudaMemcpyDeviceToHost, st));
    PM_CUDA(cudaStreamSynchronize(st));
    return PMLSH_OK;
}

// Keeps the `need` candidates with the smallest (FP64 projected distance,
// i, j) of p[0, n) (the count > T cut of Algorithm 4).
pmlsh_status pair_truncate(PairCand *p, int64_t n, int64_t need, const pmlsh_index *ix, unsigned int *hist,
                           PairExact *scratch, unsigned long long *cnt, int64_t *nOut, cudaStream_t st)
{
    if (need >= n) { *nOut = n; return PMLSH_OK; }
    if (need <= 0) { *nOut = 0; return PMLSH_OK; }
    // FP32 projected keys: |sqrt(key) - d'_64| <= eps(d'); select the need-th
    // and resolve the band around it in FP64
    float K;
    PM_TRY(pair_kth(p, n, need, hist, &K, st));
    const double tau = std::sqrt((double)K);
    const double eps = 0x1.0p-22 * ix->maxNorm + 0x1.0p-19 * tau + 1e-300;
    const float hiK = (float)((tau + 2 * eps) * (tau + 2 * eps));
    PM_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st));
    launch_pair_collect(ix, p, n, nextafterf(hiK, INFINITY), 1, scratch, cnt, PAIR_SORT_CAP, st);
    unsigned long long got = 0;
    PM_CUDA(cudaMemcpyAsync(&got, cnt, sizeof(got), cudaMemcpyDeviceToHost, st));
    PM_CUDA(cudaStreamSynchronize(st));
    if (got > PAIR_SORT_CAP) {
        pm_set_error("closest pairs: %llu candidates tied at the count > T cut (capacity %d)", got, PAIR_SORT_CAP);
        return PMLSH_EINTERNAL;
    }
    int P = 1;
    while (P < (int)got) P <<= 1;
    PM_LAUNCH("k_pair_sort", st, k_pair_sort<<<1, 1024, (size_t)P * sizeof(PairExact), st>>>(scratch, (int)got));
    std::vector<PairExact> v(got);
    PM_CUDA(cudaMemcpyAsync(v.data(), scratch, got * sizeof(PairExact), cudaMemcpyDeviceToHost, st));
    PM_CUDA(cudaStreamSynchronize(st));
    const int64_t keep = std::min<int64_t>(need, (int64_t)got);
    std::vector<PairCand> kept(keep);
    for (int64_t e = 0; e < keep; e++) {
        kept[e].key = 0.f;
        kept[e].a = v[e].a;
        kept[e].b = v[e].b;
    }
    PM_CUDA(cudaMemcpyAsync(p, kept.data(), keep * sizeof(PairCand), cudaMemcpyHostToDevice, st));
    PM_CUDA(cudaStreamSynchronize(st));
    *nOut = keep;
    return PMLSH_OK;
}


}  // namespace

// gamma of Sec. 6.3 over all pairs of the index `lx` (its own layout).
static pmlsh_status gamma_of_layout(const pmlsh_index *lx, double pr, double *gamma, cudaStream_t st)
{
    const int64_t n = lx->n, L = lx->L, N = (int64_t)lx->nodeLo.size();
    const int64_t npairs = n * (n - 1) / 2;
    DevPtrs mem;
    // node balls (FP64, the oracle's arithmetic)
    std::vector<int64_t> nodeH((size_t)N * 4);
    for (int64_t e = 0; e < N; e++) {
        nodeH[e * 4] = lx->nodeLeft[e];
        nodeH[e * 4 + 1] = lx->nodeRight[e];
        nodeH[e * 4 + 2] = lx->nodeLo[e];
        nodeH[e * 4 + 3] = lx->nodeHi[e];
    }
    std::vector<int32_t> lof(n);
    for (int64_t l = 0; l < L; l++)
        for (int64_t p = lx->leafOffH[l]; p < lx->leafOffH[l + 1]; p++) lof[p] = (int32_t)l;
    int64_t *dNode;
    double *dRad, *ratio;
    int32_t *dLeafOf;
    unsigned int *hist;
    int *err;
    PM_TRY(mem.get(&dNode, (size_t)N * 4));
    PM_TRY(mem.get(&dLeafOf, n));
    PM_TRY(mem.get(&hist, 2048));
    PM_TRY(mem.get(&err, 1));
    PM_CUDA(cudaMemcpyAsync(dNode, nodeH.data(), N * 4 * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    PM_CUDA(cudaMemcpyAsync(dLeafOf, lof.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    PM_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
    PM_TRY(node_radii(lx, false, mem, &dRad, st));
    int64_t rank = (int64_t)std::ceil(pr * (double)npairs - 1e-9);
    rank = std::max<int64_t>(1, std::min<int64_t>(npairs, rank));
    // 1. the ranked ratio in FP32, then the FP64 values of the pairs around it.  It
    // stands if the rank falls among those and its value inside their window: every
    // pair counted below is smaller, every one left out larger.
    {
        constexpr unsigned long long GL = 1ull << 16;
        float *v;
        unsigned long long *ctr;
        GammaPair *list;
        double *ex;
        PM_TRY(mem.get(&v, (size_t)npairs));
        PM_TRY(mem.get(&ctr, 2));
        PM_TRY(mem.get(&list, (size_t)GL));
        PM_TRY(mem.get(&ex, (size_t)GL));
        PM_LAUNCH("k_gamma_scan", st, k_gamma_scan<false><<<(unsigned)(n - 1), 256, 0, st>>>(
            lx->O32, n, dLeafOf, dNode, dRad, v, 0.f, 0.f, 0.f, nullptr, nullptr, 0, nullptr, err));
        PM_CUDA(cudaGetLastError());
        unsigned int prefix = 0;
        int64_t need = rank;
        const int shifts[3] = {21, 10, 0}, widths[3] = {11, 11, 10};
        std::vector<unsigned int> hh(2048);
        const int grid = (int)std::min<int64_t>(16 * 152, (npairs + 255) / 256);
        for (int pass = 0; pass < 3; pass++) {
            const unsigned int hiMask = pass == 0 ? 0u : (0xffffffffu << (shifts[pass] + widths[pass]));
            PM_CUDA(cudaMemsetAsync(hist, 0, 2048 * sizeof(unsigned int), st));
            PM_LAUNCH("k_gamma_hist32", st, k_gamma_hist32<<<grid, 256, 0, st>>>(v, npairs, shifts[pass], widths[pass],
                                                                                hiMask, prefix, hist));
            PM_CUDA(cudaMemcpyAsync(hh.data(), hist, sizeof(unsigned int) << widths[pass], cudaMemcpyDeviceToHost, st));
            PM_CUDA(cudaStreamSynchronize(st));
            int bin = 0;
            while (bin < (1 << widths[pass]) - 1 && need > (int64_t)hh[bin]) need -= hh[bin++];
            prefix |= (unsigned int)bin << shifts[pass];
        }
        float K;
        std::memcpy(&K, &prefix, sizeof(K));
        int herr = 0;
        PM_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
        PM_CUDA(cudaStreamSynchronize(st));
        if (herr == 0 && K > 0.f && K < 1e30f) {
            const float Pw = K * (1.f - 0x1.0p-16f), Qw = K * (1.f + 0x1.0p-16f);
            const float e0 = nextafterf((float)(0x1.0p-22 * lx->maxNorm), INFINITY) + 1e-30f;
            PM_CUDA(cudaMemsetAsync(ctr, 0, 2 * sizeof(unsigned long long), st));
            PM_LAUNCH("k_gamma_scan", st, k_gamma_scan<true><<<(unsigned)(n - 1), 256, 0, st>>>(
                lx->O32, n, dLeafOf, dNode, dRad, nullptr, e0, Pw, Qw, ctr, ctr + 1, GL, list, err));
            PM_LAUNCH("k_gamma_exact", st, k_gamma_exact<<<(unsigned)(GL / 32), 32, 0, st>>>(lx->O64, lx->m, list, ctr + 1,
                                                                                            GL, dRad, ex));
            PM_CUDA(cudaGetLastError());
            unsigned long long hc[2];
            PM_CUDA(cudaMemcpyAsync(hc, ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
            PM_CUDA(cudaStreamSynchronize(st));
            const int64_t r = rank - (int64_t)hc[0];
            if (hc[1] <= GL && r >= 1 && r <= (int64_t)hc[1]) {
                std::vector<double> x((size_t)hc[1]);
                PM_CUDA(cudaMemcpyAsync(x.data(), ex, x.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
                PM_CUDA(cudaStreamSynchronize(st));
                std::nth_element(x.begin(), x.begin() + (r - 1), x.end());
                const double g = x[r - 1];
                if (g >= (double)Pw && g <= (double)Qw) {
                    *gamma = g;
                    return PMLSH_OK;
                }
            }
        }
        PM_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
    }
    // 2. otherwise (many equal ratios, or none finite) every ratio in FP64
    PM_TRY(mem.get(&ratio, (size_t)npairs));
    PM_LAUNCH("k_gamma_ratio", st, k_gamma_ratio<<<(unsigned)(n - 1), 256, 0, st>>>(lx->O64, n, lx->m, dLeafOf, dNode,
                                                                                     dRad, ratio, err));
    PM_CUDA(cudaGetLastError());
    // exact rank-th smallest ratio: radix select, 8 passes of 8 bits
    unsigned long long prefix = 0, hiMask = 0;
    unsigned int hh[256];
    const int grid = (int)std::min<int64_t>(4096, (npairs + 255) / 256);
    for (int shift = 56; shift >= 0; shift -= 8) {
        PM_CUDA(cudaMemsetAsync(hist, 0, 256 * sizeof(unsigned int), st));
        PM_LAUNCH("k_gamma_hist", st, k_gamma_hist<<<grid, 256, 0, st>>>((const unsigned long long *)ratio, npairs,
                                                                           shift, hiMask, prefix, hist));
        PM_CUDA(cudaMemcpyAsync(hh, hist, sizeof(hh), cudaMemcpyDeviceToHost, st));
        PM_CUDA(cudaStreamSynchronize(st));
        int dg = 0;
        int64_t below = 0;
        while (dg < 255 && below + (int64_t)hh[dg] < rank) below += hh[dg++];
        rank -= below;
        prefix |= (unsigned long long)dg << shift;
        hiMask |= 0xFFull << shift;
    }
    int herr = 0;
    PM_CUDA(cudaMemcpy(&herr, err, sizeof(int), cudaMemcpyDeviceToHost));
    if (herr) {
        pm_set_error("gamma calibration: the hierarchy is deeper than 4096 levels");
        return PMLSH_EINTERNAL;
    }
    double g;
    std::memcpy(&g, &prefix, sizeof(g));
    *gamma = g;
    return PMLSH_OK;
}

pmlsh_status pm_gamma_calibrate(pmlsh_index *ix, double pr, int64_t nsample, uint64_t seed, double *gamma,
                                cudaStream_t st)
{
    const int64_t n = ix->n;
    if (nsample >= n) return gamma_of_layout(ix, pr, gamma, st);
    // the sample: partial Fisher-Yates shuffle of 0..n-1 driven by the
    // counter-based stream `seed`, the first nsample ids sorted
    std::vector<int64_t> ids(n);
    for (int64_t i = 0; i < n; i++) ids[i] = i;
    for (int64_t i = 0; i < nsample; i++) {
        const int64_t j = i + (int64_t)(pm_splitmix64(seed, (uint64_t)i) % (uint64_t)(n - i));
        std::swap(ids[i], ids[j]);
    }
    ids.resize(nsample);
    std::sort(ids.begin(), ids.end());
    // their rows (original order) from the leaf-order copy of X
    std::vector<int64_t> inv(n), pos(nsample);
    for (int64_t p = 0; p < n; p++) inv[ix->permH[p]] = p;
    for (int64_t i = 0; i < nsample; i++) pos[i] = inv[ids[i]];
    DevPtrs mem;
    int64_t *dPos;
    float *S;
    PM_TRY(mem.get(&dPos, nsample));
    PM_TRY(mem.get(&S, (size_t)nsample * ix->d));
    PM_CUDA(cudaMemcpyAsync(dPos, pos.data(), nsample * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    PM_LAUNCH("k_gather_rows", st, k_gather_rows<<<(unsigned)nsample, 128, 0, st>>>(ix->X, ix->ld, ix->d, dPos, nsample, S));
    PM_CUDA(cudaGetLastError());
    // the layout of the sample: the same build with the same projection,
    // pivot count and leaf capacity
    pmlsh_build_opts bo;
    pmlsh_build_opts_default(&bo);
    bo.m = ix->m;
    bo.s = ix->s;
    bo.leaf_size = ix->M;
    bo.seed = ix->seed;
    bo.proj = ix->A_host.data();
    bo.bf16_shadow = 0;
    // (only its hierarchy and projected points: what queries read of an index,
    // the principal directions of its leaf centres above all, took 75 of the
    // 100 ms of a calibration on 100,000 x 512)
    pmlsh_index sub;
    sub.n = nsample;
    sub.d = ix->d;
    sub.ld = ix->ld;
    sub.m = bo.m;
    sub.s = (int)std::min<int64_t>(bo.s, (nsample + bo.leaf_size - 1) / bo.leaf_size);
    sub.M = bo.leaf_size;
    sub.seed = bo.seed;
    pmlsh_status s = pm_build_index(&sub, S, true, &bo, st, true);
    if (s == PMLSH_OK) s = gamma_of_layout(&sub, pr, gamma, st);
    pm_free_index(&sub);
    return s;
}

pmlsh_status pm_closest_pair(pmlsh_index *ix, const pmlsh_cp_opts *o, int64_t *out_pairs, float *out_dists,
                             pmlsh_cp_stats *stats, cudaStream_t st)
{
    const int64_t n = ix->n, L = ix->L;
    const int k = o->k;
    const double t = o->t > 0.0 ? o->t : std::sqrt(pm_chi2_upper_quantile(o->alpha1, ix->m));
    double gamma = o->gamma;
    if (!(gamma > 0.0)) PM_TRY(pm_gamma_calibrate(ix, 0.85, 10000, ix->seed + 7, &gamma, st));
    const int64_t T = o->T > 0 ? o->T : (int64_t)std::ceil(o->alpha2 * (double)n * (double)(n - 1) - 1e-9) + k;
    DevPtrs mem;
    // 1. self-join of every leaf
    std::vector<int64_t> pairOff(L + 1, 0);
    for (int64_t l = 0; l < L; l++) {
        int64_t s = ix->leafOffH[l + 1] - ix->leafOffH[l];
        pairOff[l + 1] = pairOff[l] + s * (s - 1) / 2;
    }
    const int64_t nSelf = pairOff[L];
    int64_t *dPairOff;
    PairCand *pairs;
    unsigned int *hist;
    PairExact *scratch;
    unsigned long long *cnt;
    PM_TRY(mem.get(&dPairOff, L + 1));
    PM_TRY(mem.get(&pairs, (size_t)std::max<int64_t>(nSelf, 1)));
    PM_TRY(mem.get(&hist, 2048));
    PM_TRY(mem.get(&scratch, PAIR_SORT_CAP));
    PM_TRY(mem.get(&cnt, 4));
    PM_CUDA(cudaMemcpyAsync(dPairOff, pairOff.data(), (L + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    PM_TRY(pm_allow_max_dyn_smem((const void *)k_pair_sort));
    if (nSelf > 0) {
        PM_LAUNCH("k_cp_selfjoin", st, k_cp_selfjoin<<<(unsigned)L, 128, 0, st>>>(ix->X, ix->ld, ix->leafOff, dPairOff, pairs));
        PM_CUDA(cudaGetLastError());
    }
    TopK top;
    PM_TRY(pair_merge(top, k, pairs, nSelf, ix, hist, scratch, cnt, st));
    int64_t count = nSelf;
    double ub = (int)top.v.size() >= k ? top.v[k - 1].dist : INFINITY;
    const double ubSelf = ub;
    const double R = gamma * t * ub;
    // 2. node balls (FP64) and FindLCA (Algorithm 5) over the hierarchy
    const int64_t N = (int64_t)ix->nodeLo.size();
    std::vector<int64_t> pLo(N), pHi(N);
    for (int64_t e = 0; e < N; e++) {
        pLo[e] = ix->leafOffH[ix->nodeLo[e]];
        pHi[e] = ix->leafOffH[ix->nodeHi[e]];
    }
    double *dRad;
    PM_TRY(node_radii(ix, true, mem, &dRad, st));
    std::vector<double> rad(N);
    PM_CUDA(cudaMemcpyAsync(rad.data(), dRad, N * sizeof(double), cudaMemcpyDeviceToHost, st));
    PM_CUDA(cudaStreamSynchronize(st));
    std::vector<int64_t> A;
    {
        std::vector<int64_t> stack{0};
        while (!stack.empty()) {
            int64_t e = stack.back();
            stack.pop_back();
            if (ix->nodeLeft[e] < 0) continue;             // leaf nodes are never inserted
            if (rad[e] < R) { A.push_back(e); continue; }
            stack.push_back(ix->nodeRight[e]);             // visit left first (order is irrelevant:
            stack.push_back(ix->nodeLeft[e]);              // A is sorted below)
        }
        std::sort(A.begin(), A.end(), [&rad](int64_t x, int64_t y) { return rad[x] < rad[y] || (rad[x] == rad[y] && x < y); });
    }
    // leaf of each position
    int32_t *dLeafOf;
    PM_TRY(mem.get(&dLeafOf, n));
    {
        std::vector<int32_t> lof(n);
        for (int64_t l = 0; l < L; l++)
            for (int64_t p = ix->leafOffH[l]; p < ix->leafOffH[l + 1]; p++) lof[p] = (int32_t)l;
        PM_CUDA(cudaMemcpyAsync(dLeafOf, lof.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    }
    // 3. nodes in ascending radius while count <= T.  A node's filter depends on
    // ub as the nodes before it leave it, but ub changes at a few nodes only
    // (tens of thousands of candidates per change), so nodes are taken in
    // batches: the candidates of every node of a batch are listed for the ub at
    // its start (a superset for each later, smaller ub) with their distances,
    // and the nodes are replayed in order from per-node counts and the few
    // candidates that may enter the top-k; where ub falls, the rest of the batch
    // is counted again for the new ub.  On 100,000 x 512 (1,265 nodes, 2.2 M
    // candidates) node by node took 245 ms, most of it 1,265 rounds of five host
    // synchronisations; two batches and 13 replays take 4 ms.
    int64_t nodesDone = 0, fp64 = 0;
    PairCand *cand = nullptr;
    size_t candCap = 0;
    struct Cut { float lo, hi; };
    auto cut_of = [&](double Rt) -> Cut {
        Cut c{INFINITY, INFINITY};   // infinite ub: every pair is a candidate
        if (!std::isinf(Rt)) {
            const double eps = 0x1.0p-22 * ix->maxNorm + 0x1.0p-19 * Rt + 1e-300;
            c.lo = Rt - eps > 0 ? (float)((Rt - eps) * (Rt - eps)) : -1.f;
            if ((double)c.lo > (Rt - eps) * (Rt - eps)) c.lo = nextafterf(c.lo, -INFINITY);
            c.hi = (float)((Rt + eps) * (Rt + eps));
            if ((double)c.hi < (Rt + eps) * (Rt + eps)) c.hi = nextafterf(c.hi, INFINITY);
        }
        return c;
    };
    // one node by itself: a node that crosses count > T, one met while ub is
    // infinite, or one with more candidates than a batch takes
    auto single = [&](size_t ai) -> pmlsh_status {
        const int64_t lo = pLo[A[ai]], hi = pHi[A[ai]];
        const double Rt = t * ub;
        const Cut c = cut_of(Rt);
        const int64_t nt = (hi - lo + CT - 1) / CT;
        int64_t ncand = 0;
        for (int attempt = 0; attempt < 2; attempt++) {
            if (!cand) {
                candCap = std::max<size_t>(candCap, (size_t)1 << 20);
                PM_TRY(mem.get(&cand, candCap));
            }
            PM_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), st));
            PM_LAUNCH("k_cp_tiles", st, k_cp_tiles<<<dim3((unsigned)nt, (unsigned)std::min<int64_t>(nt, 65535)), 256, 0, st>>>(
                ix->O32, ix->O64, ix->m, dLeafOf, nullptr, lo, hi, 1, c.lo, c.hi, Rt, cand, nullptr, cnt, candCap,
                cnt + 1));
            PM_CUDA(cudaGetLastError());
            unsigned long long hc[2];
            PM_CUDA(cudaMemcpyAsync(hc, cnt, sizeof(hc), cudaMemcpyDeviceToHost, st));
            PM_CUDA(cudaStreamSynchronize(st));
            if (hc[0] <= candCap) {
                ncand = (int64_t)hc[0];
                fp64 += (int64_t)hc[1];
                break;
            }
            // grow and redo this node
            candCap = (size_t)hc[0];
            cand = nullptr;
            if (attempt == 1) {
                pm_set_error("closest pairs: candidate buffer growth failed");
                return PMLSH_EINTERNAL;
            }
        }
        int64_t keep = ncand;
        if (count + ncand > T) PM_TRY(pair_truncate(cand, ncand, T + 1 - count, ix, hist, scratch, cnt, &keep, st));
        if (keep > 0) {
            launch_pair_dist32(ix, cand, keep, st);
            PM_TRY(pair_merge(top, k, cand, keep, ix, hist, scratch, cnt, st));
        }
        count += keep;
        ub = (int)top.v.size() >= k ? top.v[k - 1].dist : INFINITY;
        nodesDone++;
        return PMLSH_OK;
    };
    // batches: up to CB_CAND candidates (20 bytes each), CB_TILES tiles
    constexpr unsigned long long CB_CAND = 1ull << 22;
    constexpr size_t CB_TILES = (size_t)1 << 16, CB_NODES = (size_t)1 << 14;
    PairCand *bCand = nullptr;
    int32_t *bNode = nullptr;
    float *bD32 = nullptr;
    PairTile *bTiles = nullptr;
    int *bCnt = nullptr;          // nodeCnt [CB_NODES], nodeFp [CB_NODES], then two 64-bit counters
    NodeExact *bEx = nullptr;
    std::vector<PairTile> tiles;
    std::vector<int> cntH(2 * CB_NODES + 4);
    std::vector<NodeExact> exH;
    const double epsv = (double)(ix->ld + 8) * 0x1.0p-24;
    size_t tileBudget = 512, grow = 8;   // tiles of a batch: few at first, which lower ub for the rest
    for (size_t ai = 0; ai < A.size() && count <= T;) {
        if ((int)top.v.size() < k) {
            PM_TRY(single(ai++));
            continue;
        }
        tiles.clear();
        size_t aj = ai;
        for (; aj < A.size() && aj - ai < CB_NODES; aj++) {
            const int64_t lo = pLo[A[aj]], hi = pHi[A[aj]], nt = (hi - lo + CT - 1) / CT;
            const size_t add = (size_t)(nt * (nt + 1) / 2);
            if (tiles.size() + add > (aj == ai ? CB_TILES : tileBudget)) break;
            for (int64_t y = 0; y < nt; y++)
                for (int64_t x = y; x < nt; x++)
                    tiles.push_back(PairTile{(int32_t)(lo + y * CT), (int32_t)(lo + x * CT), (int32_t)hi, (int32_t)(aj - ai)});
        }
        if (aj == ai) {   // one node of more tiles than a batch holds
            PM_TRY(single(ai++));
            continue;
        }
        if (!bCand) {
            PM_TRY(mem.get(&bCand, (size_t)CB_CAND));
            PM_TRY(mem.get(&bNode, (size_t)CB_CAND));
            PM_TRY(mem.get(&bD32, (size_t)CB_CAND));
            PM_TRY(mem.get(&bTiles, CB_TILES));
            PM_TRY(mem.get(&bCnt, 2 * CB_NODES + 4));
            PM_TRY(mem.get(&bEx, PAIR_SORT_CAP));
        }
        const int nb = (int)(aj - ai);
        unsigned long long *bN = (unsigned long long *)(bCnt + 2 * nb);   // candidates, top-k entrants
        const Cut c0 = cut_of(t * ub);
        PM_CUDA(cudaMemcpyAsync(bTiles, tiles.data(), tiles.size() * sizeof(PairTile), cudaMemcpyHostToDevice, st));
        PM_CUDA(cudaMemsetAsync(bN, 0, sizeof(unsigned long long), st));
        PM_LAUNCH("k_cp_tiles", st, k_cp_tiles<<<(unsigned)tiles.size(), 256, 0, st>>>(
            ix->O32, ix->O64, ix->m, dLeafOf, bTiles, 0, 0, 0, c0.lo, c0.hi, 0.0, bCand, bNode, bN, CB_CAND, cnt));
        PM_CUDA(cudaGetLastError());
        unsigned long long nC = 0;
        PM_CUDA(cudaMemcpyAsync(&nC, bN, sizeof(nC), cudaMemcpyDeviceToHost, st));
        PM_CUDA(cudaStreamSynchronize(st));
        if (nC > CB_CAND) {
            if (nb == 1) PM_TRY(single(ai++));
            tileBudget = std::max<size_t>(1, std::min(tileBudget, tiles.size()) / 4);
            grow = 2;
            continue;
        }
        if (nC > 0) launch_pair_dist32(ix, bCand, (int64_t)nC, st, bD32);
        PM_CUDA(cudaGetLastError());
        const unsigned rgrid = (unsigned)std::max<unsigned long long>(1, std::min<unsigned long long>((nC + 255) / 256, 8 * 152));
        int to = nb;
        bool alone = false;   // the node at ai is taken by itself next
        for (size_t base = ai; ai < aj && !alone;) {
            // replay nodes [from, to) of the batch for this ub
            const int from = (int)(ai - base);
            const double Rt = t * ub, thr = ub * ub * (1.0 + 3.0 * epsv) + 1e-36;
            const Cut c = cut_of(Rt);
            float thr32 = (float)thr;
            if ((double)thr32 < thr) thr32 = nextafterf(thr32, INFINITY);
            PM_CUDA(cudaMemsetAsync(bCnt, 0, (size_t)(2 * nb + 4) * sizeof(int), st));
            if (nC > 0)
                PM_LAUNCH("k_cp_replay", st, k_cp_replay<<<rgrid, 256, 0, st>>>(
                    bCand, bNode, bD32, (int64_t)nC, from, to, c.lo, c.hi, Rt, thr32, ix->X, ix->ld, ix->d, ix->O64,
                    ix->m, ix->perm, bCnt, bCnt + nb, bEx, bN + 1, PAIR_SORT_CAP));
            PM_CUDA(cudaGetLastError());
            PM_CUDA(cudaMemcpyAsync(cntH.data(), bCnt, (size_t)(2 * nb + 4) * sizeof(int), cudaMemcpyDeviceToHost, st));
            PM_CUDA(cudaStreamSynchronize(st));
            unsigned long long nX;
            std::memcpy(&nX, cntH.data() + 2 * nb + 2, sizeof(nX));
            if (nX > PAIR_SORT_CAP) {
                // more than the list holds: fewer nodes, down to one by itself
                if (to - from == 1) alone = true;
                else to = from + (to - from) / 2;
                continue;
            }
            exH.resize((size_t)nX);
            if (nX > 0) {
                PM_CUDA(cudaMemcpyAsync(exH.data(), bEx, (size_t)nX * sizeof(NodeExact), cudaMemcpyDeviceToHost, st));
                PM_CUDA(cudaStreamSynchronize(st));
                std::sort(exH.begin(), exH.end(), [](const NodeExact &x, const NodeExact &y) {
                    return x.node != y.node ? x.node < y.node : pe_less(x.x, y.x);
                });
            }
            bool moved = false;
            size_t x0 = 0;
            for (int i = from; i < to && !moved && !alone; i++) {
                if (count + cntH[i] > T) {
                    alone = true;   // the cut inside a node (or, at count > T, the end)
                    break;
                }
                size_t x1 = x0;
                while (x1 < exH.size() && exH[x1].node == i) x1++;
                if (x1 > x0) {
                    for (size_t x = x0; x < x1; x++) top.v.push_back(exH[x].x);
                    std::sort(top.v.begin(), top.v.end(), pe_less);
                    top.v.resize(k);
                    moved = top.v[k - 1].dist < ub;
                    ub = top.v[k - 1].dist;
                }
                x0 = x1;
                count += cntH[i];
                fp64 += cntH[nb + i];
                nodesDone++;
                ai++;
            }
            if (!moved && !alone) to = nb;
        }
        if (alone && count <= T) PM_TRY(single(ai++));
        tileBudget = std::min(CB_TILES, tileBudget * grow);
    }
    // results
    std::vector<int64_t> op((size_t)2 * k, -1);
    std::vector<float> od(k, INFINITY);
    for (int e = 0; e < k && e < (int)top.v.size(); e++) {
        op[2 * e] = top.v[e].i;
        op[2 * e + 1] = top.v[e].j;
        od[e] = (float)top.v[e].dist;
    }
    PM_CUDA(cudaMemcpy(out_pairs, op.data(), op.size() * sizeof(int64_t),
                       pm_is_device_ptr(out_pairs) ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost));
    PM_CUDA(cudaMemcpy(out_dists, od.data(), od.size() * sizeof(float),
                       pm_is_device_ptr(out_dists) ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost));
    if (stats) {
        stats->count = count;
        stats->ub_self = ubSelf;
        stats->lca_nodes = (int64_t)A.size();
        stats->nodes_done = nodesDone;
        stats->self_pairs = nSelf;
        stats->fp64_checks = fp64;
        stats->t = t;
        stats->T = T;
        stats->gamma = gamma;
    }
    return PMLSH_OK;
}

// Algorithm 3 (Sec. 6.1): the T pairs nearest in the projected space, found
// by branch and bound over leaf pairs, verified, cut to the k nearest.
//   1. every leaf's self-join, keyed by projected distance; if it yields T
//      pairs, the T-th of them bounds d_T from above;
//   2. Mindist of every leaf pair (a flat stand-in for the priority queue
//      over node pairs: with a lower bound per leaf pair the same pairs are
//      examined), the pairs with Mindist <= that bound taken in ascending
//      (Mindist, l1, l2);
//   3. their cross pairs in batches; after each batch the candidates are cut
//      to the exact T nearest (FP64-resolved band at the cut) and the search
//      stops at the first leaf pair whose Mindist exceeds the T-th distance;
//   4. the T pairs verified in the original space, exact top-k.
// The result equals the oracle's: the T pairs with the smallest (FP64
// projected distance, i, j), then the k smallest (FP64 distance, i, j).
pmlsh_status pm_closest_pair_bnb(pmlsh_index *ix, const pmlsh_cp_opts *o, int64_t *out_pairs, float *out_dists,
                                 pmlsh_cp_stats *stats, cudaStream_t st)
{
    const int64_t n = ix->n, L = ix->L;
    const int k = o->k;
    const int64_t P = n * (n - 1) / 2;
    int64_t T = o->T > 0 ? o->T : (int64_t)std::ceil(o->alpha2 * (double)n * (double)(n - 1) - 1e-9) + k;
    T = std::min(std::max<int64_t>(T, k), P);
    DevPtrs mem;
    unsigned int *hist;
    PairExact *scratch;
    unsigned long long *cnt;
    CutState *state;
    BatchPlan *planD;
    PM_TRY(mem.get(&hist, 2048));
    PM_TRY(mem.get(&scratch, PAIR_SORT_CAP));
    PM_TRY(mem.get(&cnt, 4));
    PM_TRY(mem.get(&state, 1));
    PM_TRY(mem.get(&planD, 1));
    PM_TRY(pm_allow_max_dyn_smem((const void *)k_pair_sort));
    // 1. self-joins
    std::vector<int64_t> pairOff(L + 1, 0);
    for (int64_t l = 0; l < L; l++) {
        const int64_t s = ix->leafOffH[l + 1] - ix->leafOffH[l];
        pairOff[l + 1] = pairOff[l] + s * (s - 1) / 2;
    }
    const int64_t nSelf = pairOff[L];
    // two candidate buffers, each up to T kept pairs followed by a batch: a cut
    // reads one and writes the other.  cnt[0]: pairs in the current one.
    const int64_t batchCap = std::max<int64_t>((int64_t)1 << 24, nSelf);
    PairCand *buf, *other;
    int64_t *dPairOff;
    PM_TRY(mem.get(&buf, (size_t)(T + batchCap)));
    PM_TRY(mem.get(&other, (size_t)(T + batchCap)));
    PM_TRY(mem.get(&dPairOff, L + 1));
    PM_CUDA(cudaMemcpyAsync(dPairOff, pairOff.data(), (L + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    if (nSelf > 0)
        PM_LAUNCH("k_bnb_selfjoin", st, k_bnb_selfjoin<<<(unsigned)L, 128, 0, st>>>(ix->O32, ix->leafOff, dPairOff, buf));
    PM_CUDA(cudaGetLastError());
    CutState state0;
    std::memset(&state0, 0, sizeof(state0));
    state0.dT = INFINITY;
    const unsigned long long nSelfU = (unsigned long long)nSelf;
    PM_CUDA(cudaMemcpyAsync(state, &state0, sizeof(state0), cudaMemcpyHostToDevice, st));
    PM_CUDA(cudaMemcpyAsync(cnt, &nSelfU, sizeof(nSelfU), cudaMemcpyHostToDevice, st));
    PM_CUDA(cudaMemsetAsync(hist, 0, 2048 * sizeof(unsigned int), st));
    int64_t nBuf = nSelf, fp64 = 0;   // (the pairs in buf before any that a cut's band left out)
    double dT = INFINITY;   // upper bound of the T-th projected distance
    bool cutDone = false;
    // the T pairs of buf with the smallest (FP64 projected distance, i, j), entirely
    // on the device (its bound dT and errors are read with the next batch's plan)
    auto cut = [&]() -> pmlsh_status {
        if (nBuf <= T) return PMLSH_OK;
        const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(8 * 152, (nBuf + 2047) / 2048));
        for (int pass = 0; pass < 3; pass++) {
            PM_LAUNCH("k_cut_hist", st, k_cut_hist<<<g, 256, 0, st>>>(buf, cnt, pass, state, hist));
            PM_LAUNCH("k_cut_bin", st, k_cut_bin<<<1, 1024, 0, st>>>(hist, pass, (unsigned long long)T, ix->maxNorm, state));
        }
        PM_LAUNCH("k_cut_split", st, k_cut_split<<<g, 256, 0, st>>>(buf, cnt, other, scratch, PAIR_SORT_CAP, state));
        PM_LAUNCH("k_cut_band", st, k_cut_band<<<PAIR_SORT_CAP / 32, 32, 0, st>>>(scratch, PAIR_SORT_CAP, ix->O64, ix->m,
                                                                                 ix->perm, state));
        PM_LAUNCH("k_cut_fill", st, k_cut_fill<<<PAIR_SORT_CAP / 128, 128, 0, st>>>(scratch, PAIR_SORT_CAP,
                                                                    (unsigned long long)T, other, cnt, state));
        PM_CUDA(cudaGetLastError());
        std::swap(buf, other);
        nBuf = T;
        cutDone = true;
        return PMLSH_OK;
    };
    // the device's dT, band decisions and errors
    auto read_state = [&]() -> pmlsh_status {
        CutState h;
        PM_CUDA(cudaMemcpyAsync(&h, state, sizeof(h), cudaMemcpyDeviceToHost, st));
        PM_CUDA(cudaStreamSynchronize(st));
        dT = h.dT;
        fp64 = (int64_t)h.fp64;
        if (h.err) {
            pm_set_error("closest pairs: %lld candidates inside the FP32 band at the T-th projected distance "
                         "(capacity %d)", (long long)h.nBand, PAIR_SORT_CAP);
            return PMLSH_EINTERNAL;
        }
        return PMLSH_OK;
    };
    PM_TRY(cut());
    PM_TRY(read_state());
    // 2./3. leaf pairs in bands of Mindist, (lo, hi]: each band's pairs in
    // ascending (Mindist, l1, l2), cut to the T nearest after each batch;
    // the search ends at the first leaf pair whose Mindist exceeds the T-th
    // projected distance (dT), and once a band's upper end reaches dT no
    // later band holds such a pair.  The first band ends at a generous
    // quantile of a sample of projected pair distances (near the T-th
    // distance), so that the leaf pairs listed stay few; each further band
    // quadruples the quantile.
    std::vector<double> F;
    PM_TRY(pm_distance_sample(ix, (int64_t)1 << 16, ix->seed + 8, F, st, false));
    const double pT = (double)T / (double)P;
    double pBand = std::min(1.0, 4.0 * pT + 64.0 / (double)F.size());
    auto quantile = [&](double p) -> double {
        if (p >= 1.0 || F.empty()) return INFINITY;
        const int64_t r = std::min<int64_t>((int64_t)F.size() - 1, (int64_t)std::ceil(p * (double)F.size()));
        std::nth_element(F.begin(), F.begin() + r, F.end());
        return F[r];
    };
    double bandHi = quantile(pBand);
    float lo32 = -INFINITY;   // FP32 end of the previous band: bands are disjoint in FP32
    const int64_t lpBatch = (int64_t)1 << 16;
    // per listed leaf pair: the pair, two sort keys, the prefix of the cross pairs
    LeafPair *dlp = nullptr;
    unsigned long long *keyA = nullptr, *keyB = nullptr;
    unsigned int *rsHist = nullptr;
    int64_t *pre = nullptr, *blk = nullptr;
    unsigned long long lpCap = 0, keyCap = 0;
    const dim3 mdGrid((unsigned)((L + BM_T - 1) / BM_T),
                      (unsigned)std::max<int64_t>(1, std::min<int64_t>(64, 16 * 152 / ((L + BM_T - 1) / BM_T))));
    int64_t examined = 0, listed = 0;
    for (;;) {
        const double hiCut = std::min(bandHi, dT);
        // the band is (lo32, hi32] in FP32 Mindist, hi32 >= hiCut
        const float hi32 = std::isinf(hiCut) ? INFINITY : nextafterf((float)hiCut, INFINITY);
        // listed up to the buffer's size, and again into one of the band's size if
        // that was too short (a list for every leaf pair took 12 bytes times
        // L (L - 1) / 2)
        unsigned long long nlp = 0;
        for (int attempt = 0; L > 1 && attempt < 2; attempt++) {
            if (!dlp || attempt == 1) {
                lpCap = attempt == 1 ? nlp : (unsigned long long)std::min<int64_t>(L * (L - 1) / 2, (int64_t)1 << 23);
                PM_TRY(mem.get(&dlp, (size_t)lpCap));
            }
            PM_CUDA(cudaMemsetAsync(cnt + 1, 0, sizeof(unsigned long long), st));
            PM_LAUNCH("k_bnb_mindist", st, k_bnb_mindist<<<mdGrid, BM_T, 0, st>>>(ix->leafMeta, ix->s, L, lo32, hi32,
                                                                                  dlp, cnt + 1, lpCap));
            PM_CUDA(cudaGetLastError());
            PM_CUDA(cudaMemcpyAsync(&nlp, cnt + 1, sizeof(nlp), cudaMemcpyDeviceToHost, st));
            PM_CUDA(cudaStreamSynchronize(st));
            if (nlp <= lpCap) break;
        }
        const int64_t nl = (int64_t)nlp;
        const bool gpuSort = L <= LP_GPU_MAX_L;
        if (nlp > keyCap) {
            PM_TRY(mem.get(&pre, (size_t)nlp));
            PM_TRY(mem.get(&blk, (size_t)(nl + 1023) / 1024));
            if (gpuSort) {
                PM_TRY(mem.get(&keyA, (size_t)nlp));
                PM_TRY(mem.get(&keyB, (size_t)nlp));
                PM_TRY(mem.get(&rsHist, (size_t)256 * ((nlp + RS_THREADS * RS_ITEMS - 1) / (RS_THREADS * RS_ITEMS)) + 256));
            }
            keyCap = nlp;
        }
        if (nl > 0) {
            if (gpuSort) {
                // ascending (Mindist, l1, l2) by the device radix sort
                const int nb = (int)((nl + RS_THREADS * RS_ITEMS - 1) / (RS_THREADS * RS_ITEMS));
                const unsigned g = (unsigned)((nl + 255) / 256);
                unsigned int *total = rsHist + (size_t)256 * nb;
                PM_LAUNCH("k_lp_key", st, k_lp_key<<<g, 256, 0, st>>>(dlp, nl, L, keyA));
                unsigned long long *src = keyA, *dst = keyB;
                for (int shift = 0; shift < 64; shift += 8) {
                    // (digits of the pair's rank that no rank reaches)
                    if (shift < 32 && (uint64_t)(L * (L - 1) / 2) <= ((uint64_t)1 << shift)) continue;
                    PM_LAUNCH("k_rs_hist", st, k_rs_hist<<<(unsigned)nb, RS_THREADS, 0, st>>>(src, nl, shift, rsHist, nb));
                    PM_LAUNCH("k_rs_scan", st, k_rs_scan<<<256, 256, 0, st>>>(rsHist, nb, total));
                    PM_LAUNCH("k_rs_scatter", st, k_rs_scatter<<<(unsigned)nb, RS_THREADS, 0, st>>>(src, dst, nl, shift,
                                                                                                  rsHist, total, nb));
                    std::swap(src, dst);
                }
                PM_CUDA(cudaMemsetAsync(cnt + 3, 0, sizeof(unsigned long long), st));
                PM_LAUNCH("k_lp_decode", st, k_lp_decode<<<g, 256, 0, st>>>(src, nl, L, dlp, (int *)(cnt + 3)));
                PM_CUDA(cudaGetLastError());
                unsigned long long badH = 0;
                PM_CUDA(cudaMemcpyAsync(&badH, cnt + 3, sizeof(badH), cudaMemcpyDeviceToHost, st));
                PM_CUDA(cudaStreamSynchronize(st));
                if (badH != 0) {
                    pm_set_error("closest pairs: the device sort of %llu leaf pairs failed its check (%llu)", nlp, badH);
                    return PMLSH_EINTERNAL;
                }
            } else {
                std::vector<LeafPair> lps(nlp);
                PM_CUDA(cudaMemcpyAsync(lps.data(), dlp, nlp * sizeof(LeafPair), cudaMemcpyDeviceToHost, st));
                PM_CUDA(cudaStreamSynchronize(st));
                std::sort(lps.begin(), lps.end(), [](const LeafPair &x, const LeafPair &y) {
                    if (x.md != y.md) return x.md < y.md;
                    if (x.l1 != y.l1) return x.l1 < y.l1;
                    return x.l2 < y.l2;
                });
                PM_CUDA(cudaMemcpyAsync(dlp, lps.data(), nlp * sizeof(LeafPair), cudaMemcpyHostToDevice, st));
                PM_CUDA(cudaStreamSynchronize(st));
            }
            PM_LAUNCH("k_lp_size", st, k_lp_size<<<(unsigned)((nl + 1023) / 1024), 1024, 0, st>>>(dlp, nl, ix->leafOff, pre, blk));
            PM_LAUNCH("k_lp_scan", st, k_lp_scan<<<1, 1024, 0, st>>>(blk, (int)((nl + 1023) / 1024)));
            PM_CUDA(cudaGetLastError());
        }
        listed += nl;
        bool stop = false;
        for (int64_t next = 0; next < nl;) {
            // the next batch (one read of the device's decisions)
            BatchPlan plan;
            PM_LAUNCH("k_bnb_plan", st, k_bnb_plan<<<1, 32, 0, st>>>(dlp, pre, blk, ix->leafOff, nl, next, lpBatch,
                                                                     batchCap, state, planD));
            PM_CUDA(cudaMemcpyAsync(&plan, planD, sizeof(plan), cudaMemcpyDeviceToHost, st));
            PM_CUDA(cudaStreamSynchronize(st));
            dT = plan.dT;
            if (plan.err) return read_state();
            if (plan.stop) { stop = true; break; }   // no pair under it can beat the T-th
            if (plan.tot > batchCap) {
                pm_set_error("closest pairs: one leaf pair holds more pairs than the batch capacity");
                return PMLSH_EINTERNAL;
            }
            PM_LAUNCH("k_bnb_cross", st, k_bnb_cross<<<(unsigned)((plan.end - next + 7) / 8), 256, 0, st>>>(
                ix->O32, ix->leafOff, dlp, next, plan.end, cutDone ? 1 : 0, state, buf, cnt));
            PM_CUDA(cudaGetLastError());
            nBuf += plan.tot;
            examined += plan.end - next;
            next = plan.end;
            PM_TRY(cut());
        }
        PM_TRY(read_state());
        // done when this band reached dT (every later pair has Mindist > dT)
        // or covered everything
        if (stop || std::isinf(bandHi) || dT <= bandHi) break;
        lo32 = hi32;
        pBand = std::min(1.0, pBand * 4.0);
        bandHi = std::max(quantile(pBand), (double)hi32);
    }
    // 4. verification and the exact top-k
    if (nBuf > 0)
        launch_pair_dist32(ix, buf, nBuf, st);
    TopK top;
    PM_TRY(pair_merge(top, k, buf, nBuf, ix, hist, scratch, cnt, st));
    std::vector<int64_t> op((size_t)2 * k, -1);
    std::vector<float> od(k, INFINITY);
    for (int e = 0; e < k && e < (int)top.v.size(); e++) {
        op[2 * e] = top.v[e].i;
        op[2 * e + 1] = top.v[e].j;
        od[e] = (float)top.v[e].dist;
    }
    PM_CUDA(cudaMemcpy(out_pairs, op.data(), op.size() * sizeof(int64_t),
                       pm_is_device_ptr(out_pairs) ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost));
    PM_CUDA(cudaMemcpy(out_dists, od.data(), od.size() * sizeof(float),
                       pm_is_device_ptr(out_dists) ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost));
    if (stats) {
        stats->count = nBuf;
        stats->ub_self = INFINITY;
        stats->lca_nodes = listed;
        stats->nodes_done = examined;
        stats->self_pairs = nSelf;
        stats->fp64_checks = fp64;
        stats->t = 0.0;
        stats->T = T;
        stats->gamma = o->gamma;
    }
    return PMLSH_OK;
}
