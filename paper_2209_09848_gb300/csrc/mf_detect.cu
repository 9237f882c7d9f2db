// Score normalisation and candidate extraction (Section 3.3 of Ganapathi
// 2022): each pixel's best score in units of the standard deviation of the
// scores in the square centred on it, candidates above a threshold, and one
// detection per group of touching candidates.
//
// Data path, all on the caller's stream, P = H x W pixels:
//   k_det_cols     thread per (column, chunk of rows): sliding sums over the
//                  window's rows of the valid scores, their squares and the
//                  valid count (FP64, FP64, int32 per pixel);
//   k_det_rows     block per (row, tile of columns): the tile's column sums
//                  plus halo in shared memory, prefix sums along the row,
//                  window sums as prefix differences, then z, the candidate
//                  flag, the union-find parent (itself for a candidate, -1
//                  otherwise) and the list of candidates;
//   k_det_union    thread per candidate: union with the candidate neighbours
//                  above it and to its left (lock-free union-find in which a
//                  root only ever hangs below a smaller index, so every
//                  component ends rooted at its smallest flat index);
//   k_det_peak_z   every candidate points at its root; per component the
//                  largest z (atomicMax on order-preserving FP64 bits) and the
//                  pixel count;
//   k_det_peak_at  the smallest index attaining that z;
//   k_det_mark     per root: the peak's FP32 z and index as a selection key;
//   top-k select   the shared selection over those keys (z desc, index asc);
//   k_det_emit     one record per selected detection (its window's mean and
//                  sigma summed again) and the counts.
// Every reduction is an integer atomic or a fixed-order sum, so reruns are
// bit-identical.
//
// FP64 operations -- arithmetic, comparisons and conversions alike -- issue
// once per 64 cycles and scheduler on this GPU and bound the first two kernels,
// so they are counted: conversions go by bits (widen), and k_det_rows keeps
// FP64 for the sums and the cancelling n s - s1 and n s2 - s1^2, forms z from
// them in pairs of FP32 numbers, and takes the FP64 formula only for pixels at
// or above the threshold (or a window near the degenerate limit).

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "mf_device.cuh"
#include "mf_internal.h"

namespace mf {
namespace {

using dev::launch_dependents;
using dev::sel_key;
using dev::wait_previous;
using dev::widen;

constexpr int kRowTile = 2048;  // output columns per k_det_rows block at most
constexpr int kRowThreads = 256;
constexpr int kUnionBudget = 1 << 20;  // iterations of one find or merge loop

struct DetectLayout {
    size_t c1, c2, cn, zd, zmax, parent, peak, npix, cand, sel_base, total;
    SelectLayout sel;
};

DetectLayout detect_layout(int64_t P, int32_t max_out) {
    DetectLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = (off + bytes + 255) / 256 * 256;
        return o;
    };
    L.c1 = take((size_t)P * 8);
    L.c2 = take((size_t)P * 8);
    L.cn = take((size_t)P * 4);
    L.zd = take((size_t)P * 8);    // this and the next five: at candidates only (parent everywhere)
    L.zmax = take((size_t)P * 8);
    L.parent = take((size_t)P * 4);
    L.peak = take((size_t)P * 4);
    L.npix = take((size_t)P * 4);
    L.cand = take((size_t)P * 4);  // the candidates' flat indices, in no order
    L.sel_base = off;
    L.sel = select_layout(P, max_out > 0 ? max_out : 1);
    L.total = L.sel_base + L.sel.total;
    return L;
}

// Unbiased exponent of x, by bits (1024: not finite; -1023: 0 or subnormal).
__device__ __forceinline__ int exponent(double x) { return (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7FFu) - 1023; }

// A sum from which more than 2^kSpoil times its size has been taken has lost
// that many of its 53 bits; beyond this it is formed again.
constexpr int kSpoil = 20;

__device__ __forceinline__ unsigned long long ord_bits(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}

// Vertical window sums: for output row y the rows y - R .. y + R clipped to
// the image.  A thread owns one column of a chunk of output rows: it sums its
// first row's window directly, then each step adds the row entering the window
// and drops the row leaving it: 4 FP64 operations a pixel plus 2 (2 R + 1) per
// chunk.  The chunks are as long as two blocks of four warps per SM allow
// (2048^2, window 255: 108 rows; one block per SM does fewer sums but leaves
// the pipe idle behind the loads, 132 us).  The count goes by bit masks.
// Both kernels of the stage, 2048^2 with window 255: 567 -> 236 us.
//
// A score that leaves a window leaves the rounding errors it caused behind: one
// that is not finite, or whose square is 2^kSpoil times what remains, would
// spoil its column down to the chunk's end.  Such a window is summed directly
// (found by exponents, in integers: the FP64 pipe sets the pace), and an empty
// one is exactly zero.
__global__ void __launch_bounds__(128) k_det_cols(const float *__restrict__ s, const int32_t *__restrict__ am, int H,
                                                  int W, int R, int chunk, double *__restrict__ c1,
                                                  double *__restrict__ c2, int *__restrict__ cn, SelState *st) {
    launch_dependents();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *st = SelState{};  // the next kernel's counters
    constexpr int U = 8;  // rows whose loads are in flight together
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= W) return;
    const int y0 = blockIdx.y * chunk, y1 = min(H, y0 + chunk);
    double a1 = 0.0, a2 = 0.0;
    int an = 0;
    // the valid scores of rows y .. y + U - 1 that lie in lo .. hi - 1, 0
    // elsewhere, and a bit for each that counts (score and flag are loaded at
    // once: a score load that waits for its flag would stall the warp)
    auto fetch = [&](int y, int lo, int hi, float (&v)[U]) {
        unsigned int bits = 0;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const bool in = y + u >= lo && y + u < hi;
            const size_t i = (size_t)(in ? y + u : 0) * W + x;
            const int k = am[i];
            const float f = s[i];
            const bool ok = in && k >= 0;
            v[u] = ok ? f : 0.f;
            bits |= (unsigned int)ok << u;
        }
        return bits;
    };
    // the rows of the next step are on their way while this one's are summed
    float vi[U], vo[U], wi[U], wo[U];
    const int first = max(0, y0 - R - 1), upto = min(H, y0 + R);
    unsigned int ni, no, mi = fetch(first, first, upto, wi), mo;
    for (int y = first; y < upto; y += U) {
        ni = mi;
#pragma unroll
        for (int u = 0; u < U; u++) vi[u] = wi[u];
        mi = fetch(y + U, first, upto, wi);
        an += __popc(ni);
#pragma unroll
        for (int u = 0; u < U; u++) {
            const double d = widen(vi[u]);
            a1 += d;
            a2 = fma(d, d, a2);
        }
    }
    mi = fetch(y0 + R, 0, H, wi);
    mo = fetch(y0 - R - 1, 0, H, wo);
    for (int y = y0; y < y1; y += U) {
        ni = mi;
        no = mo;
#pragma unroll
        for (int u = 0; u < U; u++) {
            vi[u] = wi[u];
            vo[u] = wo[u];
        }
        mi = fetch(y + U + R, 0, H, wi);
        mo = fetch(y + U - R - 1, 0, H, wo);
        unsigned int spoilt = 0;  // a bit per row
#pragma unroll
        for (int u = 0; u < U; u++) {
            const double di = widen(vi[u]), dn = widen(vo[u]);
            a1 += di;
            a2 = fma(di, di, a2);
            a1 -= dn;
            a2 = fma(-dn, dn, a2);
            an += (int)((ni >> u) & 1u) - (int)((no >> u) & 1u);
            a1 = an == 0 ? 0.0 : a1;
            a2 = an == 0 ? 0.0 : a2;
            const int ev = (int)((__float_as_uint(vo[u]) >> 23) & 0xFFu);
            spoilt |= (unsigned int)(an != 0 && ev != 0 &&
                                     (ev == 255 || 2 * (ev - 127) - exponent(a2) > kSpoil)) << u;
            if (y + u < y1) {
                const size_t i = (size_t)(y + u) * W + x;
                c1[i] = a1;
                c2[i] = a2;
                cn[i] = an;
            }
        }
        if (spoilt) {  // from the first such window on, row by row
            auto one = [&](int q) {
                const bool in = q >= 0 && q < H;
                const size_t i = (size_t)(in ? q : 0) * W + x;
                return in && am[i] >= 0 ? widen(s[i]) : 0.0;
            };
            for (int u = __ffs(spoilt) - 1; u < U && y + u < y1; u++) {
                if ((spoilt >> u) & 1u) {
                    const int lo = max(0, y + u - R), hi = min(H, y + u + R + 1);
                    a1 = 0.0;
                    a2 = 0.0;
                    for (int q = lo; q < hi; q += U) {
                        fetch(q, lo, hi, vi);
#pragma unroll
                        for (int j = 0; j < U; j++) {
                            const double d = widen(vi[j]);
                            a1 += d;
                            a2 = fma(d, d, a2);
                        }
                    }
                } else {
                    const double di = one(y + u + R), dn = one(y + u - R - 1);
                    a1 += di;
                    a2 = fma(di, di, a2);
                    a1 -= dn;
                    a2 = fma(-dn, dn, a2);
                }
                const size_t i = (size_t)(y + u) * W + x;
                if (cn[i] == 0) {
                    a1 = 0.0;
                    a2 = 0.0;
                }
                c1[i] = a1;
                c2[i] = a2;
            }
        }
    }
}

// Exclusive scan of one value over the block (fixed order: the warp's
// shuffles, then the warps' totals in order).
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T *warp_tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T ti = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : T(0);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const T o = __shfl_up_sync(0xffffffffu, ti, d);
            if (lane >= d) ti += o;
        }
        ti = __shfl_up_sync(0xffffffffu, ti, 1);
        if (lane < (int)(blockDim.x >> 5)) warp_tot[lane] = lane ? ti : T(0);  // exclusive offsets of the warps
    }
    __syncthreads();
    // the sums in front, never a sum less its last: a large value would take them along
    const T before = __shfl_up_sync(0xffffffffu, inc, 1);
    const T r = lane ? warp_tot[warp] + before : warp_tot[warp];
    __syncthreads();  // warp_tot may be reused
    return r;
}

// x = hi + lo to 2^-47 relative, by bits; false where a part could leave the
// range of normal FP32 numbers.
__device__ __forceinline__ bool split(double x, float &hi, float &lo) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const int e = (int)((h >> 20) & 0x7FFu) - 1023;
    const bool zero = ((h << 1) | l) == 0u;
    hi = zero ? 0.f
              : __uint_as_float((h & 0x80000000u) | (uint32_t)(e + 127) << 23 | ((h & 0xFFFFFu) << 3) | (l >> 29));
    const float m = (float)(l & 0x1FFFFFFFu) * __uint_as_float((uint32_t)(e + 127 - 52) << 23);
    lo = zero ? 0.f : ((h & 0x80000000u) ? -m : m);
    return zero || (e >= -60 && e <= 60);
}

// The FP64 statistics of one window: mean and variance of n values from their
// sum and the sum of their squares.
__device__ __forceinline__ void window_stats(double s1, double s2, int n, double &mean, double &var) {
    mean = 0.0;
    var = 0.0;
    if (n > 0) {
        const double inv_n = 1.0 / n;
        mean = s1 * inv_n;
        var = fmax(s2 * inv_n - mean * mean, 0.0);
    }
}

// Horizontal window sums, z and the candidate flag for the columns x0 .. x0 +
// tile - 1 of row y.  Shared entry j holds column lo + j, lo = x0 - R - 1 (0
// outside the image); after the prefix scan the window [x - R, x + R] of
// column x = x0 + t is entries t + 1 .. t + 2R + 1.  A window behind column sums
// so large that their prefix has swallowed it, or not finite, is summed directly
// from the column sums.
__global__ void __launch_bounds__(kRowThreads) k_det_rows(
    const float *__restrict__ s, const int32_t *__restrict__ am, const double *c1,
    const double *c2, const int *cn, int H, int W, int R, int tile, double thr,
    float thr_low, int submean, float *__restrict__ z_out, double *__restrict__ zd,
    unsigned long long *__restrict__ zmax, unsigned int *__restrict__ peak, int *__restrict__ npix,
    int *__restrict__ parent, int *__restrict__ cand, SelState *st) {
    launch_dependents();
    wait_previous();
    extern __shared__ double sm[];
    __shared__ double wt1[kRowThreads / 32], wt2[kRowThreads / 32];
    __shared__ int wtn[kRowThreads / 32], hi_exp[kRowThreads / 32], lo_exp[kRowThreads / 32];
    const int tiles = (W + tile - 1) / tile;
    const int y = (int)(blockIdx.x / tiles);
    const int x0 = (int)(blockIdx.x % tiles) * tile;
    const int lo = x0 - R - 1;
    const int L = tile + 2 * R + 1;
    double *p1 = sm;
    double *p2 = sm + L;
    int *pn = reinterpret_cast<int *>(sm + 2 * L);
    const size_t row = (size_t)y * W;
    int e_hi = -1024, e_lo = 1024;  // exponents of the tile's column sums of squares, zeros left out
    for (int j = threadIdx.x; j < L; j += blockDim.x) {
        const int x = lo + j;
        const bool in = x >= 0 && x < W;
        p1[j] = in ? c1[row + x] : 0.0;
        const double q = in ? c2[row + x] : 0.0;
        p2[j] = q;
        pn[j] = in ? cn[row + x] : 0;
        const int e = exponent(q);
        if (e > -1023) {
            e_hi = max(e_hi, e);
            e_lo = min(e_lo, e);
        }
    }
    const int lane = threadIdx.x & 31;
    e_hi = __reduce_max_sync(0xffffffffu, e_hi);
    e_lo = __reduce_min_sync(0xffffffffu, e_lo);
    if (lane == 0) {
        hi_exp[threadIdx.x >> 5] = e_hi;
        lo_exp[threadIdx.x >> 5] = e_lo;
    }
    __syncthreads();
    const int per = ((L + blockDim.x - 1) / blockDim.x) | 1;  // odd: neighbouring threads on other banks
    const int j0 = min(L, (int)threadIdx.x * per), j1 = min(L, j0 + per);
    double r1 = 0.0, r2 = 0.0;
    int rn = 0;
    for (int j = j0; j < j1; j++) {
        r1 += p1[j];
        p1[j] = r1;
        r2 += p2[j];
        p2[j] = r2;
        rn += pn[j];
        pn[j] = rn;
    }
    const double o1 = block_exclusive_scan(r1, wt1);
    const double o2 = block_exclusive_scan(r2, wt2);
    const int on = block_exclusive_scan(rn, wtn);
    for (int j = j0; j < j1; j++) {
        p1[j] += o1;
        p2[j] += o2;
        pn[j] += on;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kRowThreads / 32; w++) {
        e_hi = max(e_hi, hi_exp[w]);
        e_lo = min(e_lo, lo_exp[w]);
    }
    // Can a window sum have lost the bits that kSpoil allows?  Only if column
    // sums differ by more than the 2^13 that a prefix of 4095 adds.  Has one?
    // Then each thread sums the window of its first pixel directly, slides it
    // over its others and starts again where a column that dwarfs it leaves:
    // results do not depend on the tile.  (One spike of 1e15 in 500 x 2100,
    // window 127: 314 us; clean maps as without the check.)
    bool slid = false;
    if (e_hi - e_lo > kSpoil - 13) {
        bool lost = false;
        for (int t = threadIdx.x; t < tile; t += blockDim.x) {
            const double before = p2[t], upto = p2[t + 2 * R + 1];
            lost = lost || (pn[t + 2 * R + 1] - pn[t] >= 2 &&
                            (exponent(upto) == 1024 || exponent(before) - exponent(upto - before) > kSpoil));
        }
        slid = __syncthreads_or(lost);
    }
    if (slid) {
        const int own = (tile + blockDim.x - 1) / blockDim.x, first = (int)threadIdx.x * own;
        double s1 = 0.0, s2 = 0.0;
        for (int t = first; t < min(tile, first + own) && x0 + t < W; t++) {
            const int x = x0 + t;
            bool direct = t == first;
            if (!direct) {
                const double out = x - R - 1 >= 0 ? c2[row + x - R - 1] : 0.0;
                s1 += x + R < W ? c1[row + x + R] : 0.0;
                s2 += x + R < W ? c2[row + x + R] : 0.0;
                s1 -= x - R - 1 >= 0 ? c1[row + x - R - 1] : 0.0;
                s2 -= out;
                direct = exponent(out) > -1023 && (exponent(out) == 1024 || exponent(out) - exponent(s2) > kSpoil);
            }
            if (direct) {
                s1 = 0.0;
                s2 = 0.0;
                for (int q = max(0, x - R); q <= min(W - 1, x + R); q++) {
                    s1 += c1[row + q];
                    s2 += c2[row + q];
                }
            }
            p1[t] = s1;
            p2[t] = s2;
        }
        __syncthreads();
    }
    for (int t0 = threadIdx.x & ~31; t0 < tile; t0 += blockDim.x) {  // whole warps: they add to the list together
        const int t = t0 + lane, x = x0 + t;
        const bool in = t < tile && x < W;
        const size_t i = row + (in ? x : 0);
        bool flag = false;
        double z = 0.0;
        if (in) {
            const bool valid = am[i] >= 0;
            float zf = 0.f;
            if (valid) {
                const int n = pn[t + 2 * R + 1] - pn[t];
                const double s1 = slid ? p1[t] : p1[t + 2 * R + 1] - p1[t];
                const double s2 = slid ? p2[t] : p2[t + 2 * R + 1] - p2[t];
                // u = n (s - mean) or n s, v = n^2 var: z = u / sqrt(v)
                const float nf = (float)n;  // n < 2^24
                const double nd = widen(nf), sd = widen(s[i]);
                const double u = submean ? fma(nd, sd, -s1) : nd * sd;
                const double v = fma(nd, s2, -(s1 * s1));
                float uh, ul, vh, vl, qh, ql;
                bool plain = split(u, uh, ul);
                plain = split(v, vh, vl) && plain;
                plain = split(s2, qh, ql) && plain;
                plain = plain && n >= 2 && vh > 1e-10f * (nf * qh);  // far from a constant window
                if (plain) {
                    // 1 / sqrt(v) = y (1 + e / 2), e = 1 - v y^2 in two FP32 parts
                    const float y1 = rsqrtf(vh);
                    const float p = vh * y1, pe = fmaf(vh, y1, -p);
                    float e = fmaf(-p, y1, 1.f);
                    e = fmaf(-pe, y1, e);
                    e = fmaf(-vl * y1, y1, e);
                    const float yl = 0.5f * e * y1;
                    const float zh = uh * y1;
                    float ze = fmaf(uh, y1, -zh);
                    ze = fmaf(uh, yl, ze);
                    ze = fmaf(ul, y1, ze);
                    zf = zh + ze;
                }
                if (!plain || !(zf < thr_low)) {
                    double mean, var;
                    window_stats(s1, s2, n, mean, var);
                    if (n >= 2 && var > 1e-12 * (mean * mean + var)) {
                        z = ((double)s[i] - (submean ? mean : 0.0)) * rsqrt(var);
                        flag = z > thr;
                    }
                    zf = (float)z;
                }
            }
            if (z_out) z_out[i] = zf;
            parent[i] = flag ? (int)i : -1;
            if (flag) {
                zd[i] = z;
                zmax[i] = 0ull;
                peak[i] = 0xFFFFFFFFu;
                npix[i] = 0;
            }
        }
        const unsigned int m = __ballot_sync(0xffffffffu, flag);
        if (m) {
            unsigned int at = 0;
            if (lane == 0) at = atomicAdd(&st->ticket, (unsigned int)__popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (flag) cand[at + __popc(m & ((1u << lane) - 1u))] = (int)i;
        }
    }
}

__device__ __forceinline__ int uf_find(const int *parent, int x, int *status) {
    for (int it = 0; it < kUnionBudget; it++) {
        const int p = *(const volatile int *)(parent + x);
        if (p == x) return x;
        x = p;
    }
    atomicCAS(status, 0, 3);
    return x;
}

// Join the components of candidates a and b: the larger root is hung below
// the smaller one; if it stopped being a root meanwhile, retry from its new
// parent (the pixel keeps a parent in the same component either way).
__device__ __forceinline__ void uf_merge(int *parent, int a, int b, int *status) {
    for (int it = 0; it < kUnionBudget; it++) {
        a = uf_find(parent, a, status);
        b = uf_find(parent, b, status);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(parent + a, b);
        if (old == a) return;
        a = old;
    }
    atomicCAS(status, 0, 3);
}

// The kernels below walk the list of candidates, st->ticket of them.  From the
// column sums on, each kernel of a detection starts early (see launch_after) and
// waits for the one before it at its top: a few microseconds of work each, so
// that the gap between two launches would be most of their time (2048^2, window
// 255: 311 -> 296 us; 301 x 277, window 63: 120 -> 111).  What earlier
// kernels wrote is read through pointers that are not __restrict__ (loads of
// const __restrict__ data need not stay behind the wait).
__global__ void k_det_union(int *__restrict__ parent, const int *cand, const SelState *st, int W,
                            int *status) {
    launch_dependents();
    wait_previous();
    const unsigned int n = st->ticket;
    for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int i = cand[j];
        const int y = i / W, x = i % W;
        if (x > 0 && parent[i - 1] >= 0) uf_merge(parent, i, i - 1, status);
        if (y > 0) {
            const int up = i - W;
            if (x > 0 && parent[up - 1] >= 0) uf_merge(parent, i, up - 1, status);
            if (parent[up] >= 0) uf_merge(parent, i, up, status);
            if (x + 1 < W && parent[up + 1] >= 0) uf_merge(parent, i, up + 1, status);
        }
    }
}

__global__ void k_det_peak_z(int *parent, const int *cand, const SelState *st,
                             const double *zd, unsigned long long *__restrict__ zmax,
                             int *__restrict__ npix, int *status) {
    launch_dependents();
    wait_previous();
    const unsigned int n = st->ticket;
    for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int i = cand[j];
        const int r = uf_find(parent, i, status);
        parent[i] = r;  // others that pass through i meet an ancestor either way
        atomicMax(zmax + r, ord_bits(zd[i]));
        atomicAdd(npix + r, 1);
    }
}

__global__ void k_det_peak_at(const int *parent, const int *cand, const SelState *st,
                              const double *zd, const unsigned long long *zmax,
                              unsigned int *__restrict__ peak) {
    launch_dependents();
    wait_previous();
    const unsigned int n = st->ticket;
    for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int i = cand[j], r = parent[i];
        if (ord_bits(zd[i]) == zmax[r]) atomicMin(peak + r, (unsigned int)i);
    }
}

__global__ void k_det_mark(const int *parent, const int *cand, SelState *st,
                           const double *zd, const unsigned int *peak,
                           unsigned long long *__restrict__ keys) {
    launch_dependents();
    wait_previous();
    const unsigned int n = st->ticket;
    const unsigned int lane = threadIdx.x & 31;
    for (unsigned int j0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); j0 < n; j0 += gridDim.x * blockDim.x) {
        const int i = j0 + lane < n ? cand[j0 + lane] : -1;
        const bool root = i >= 0 && parent[i] == i;
        const unsigned int m = __ballot_sync(0xffffffffu, root);
        if (m == 0) continue;
        unsigned int at = 0;
        if (lane == 0) at = atomicAdd(&st->list, (unsigned int)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (root) {
            const unsigned int pk = peak[i];
            keys[at + __popc(m & ((1u << lane) - 1u))] = sel_key((float)zd[pk], pk);
        }
    }
}

// A warp per detection; its lanes sum the peak's window again from the column
// sums of the peak's row.
__global__ void __launch_bounds__(256) k_det_emit(
    const unsigned long long *top, const SelState *st, int max_out, const int *parent,
    const float *__restrict__ s, const int32_t *__restrict__ am, const double *zd,
    const double *c1, const double *c2, const int *cn,
    const int *npix, int W, int R, mf_detection *__restrict__ out, int32_t *__restrict__ n_out) {
    wait_previous();
    const int n = max_out > 0 ? (int)st->count : 0;
    const int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        n_out[0] = (int32_t)st->list;
        n_out[1] = n;
    }
    if (i >= n) return;
    const int p = (int)(0xFFFFFFFFu - (unsigned int)(top[i] & 0xFFFFFFFFull));
    const int y = p / W, x = p % W;
    double s1 = 0.0, s2 = 0.0;
    int cnt = 0;
    for (int q = max(0, x - R) + lane; q <= min(W - 1, x + R); q += 32) {
        const size_t at = (size_t)y * W + q;
        s1 += c1[at];
        s2 += c2[at];
        cnt += cn[at];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (lane != 0) return;
    double mean, var;
    window_stats(s1, s2, cnt, mean, var);
    mf_detection d;
    d.y = y;
    d.x = x;
    d.k = am[p];
    d.npix = npix[parent[p]];
    d.z = zd[p];
    d.mean = mean;
    d.sigma = sqrt(var);
    d.snr = s[p];
    d.reserved = 0;
    out[i] = d;
}

int grid_for(int64_t n, int threads) {
    const int64_t b = (n + threads - 1) / threads;
    return (int)(b < 152 * 8 ? (b < 1 ? 1 : b) : 152 * 8);
}

struct Scope {
    ProfToken t;
    Scope(int kid, cudaStream_t s) : t(prof_begin(kid, s)) {}
    ~Scope() { prof_end(t); }
};

}  // namespace

size_t detect_workspace(int64_t H, int64_t W, int32_t max_out) { return detect_layout(H * W, max_out).total; }

int launch_detect(const DetectArgs &a, char *err, size_t errlen) {
    cudaStream_t stream = (cudaStream_t)a.stream;
    const int H = (int)a.H, W = (int)a.W;
    const int64_t P = a.H * a.W;
    const int R = a.window / 2;
    const DetectLayout L = detect_layout(P, a.max_out);
    char *ws = a.ws;
    double *c1 = reinterpret_cast<double *>(ws + L.c1);
    double *c2 = reinterpret_cast<double *>(ws + L.c2);
    int *cn = reinterpret_cast<int *>(ws + L.cn);
    double *zd = reinterpret_cast<double *>(ws + L.zd);
    unsigned long long *zmax = reinterpret_cast<unsigned long long *>(ws + L.zmax);
    int *parent = reinterpret_cast<int *>(ws + L.parent);
    unsigned int *peak = reinterpret_cast<unsigned int *>(ws + L.peak);
    int *npix = reinterpret_cast<int *>(ws + L.npix);
    int *cand = reinterpret_cast<int *>(ws + L.cand);
    char *sws = ws + L.sel_base;
    SelState *st = reinterpret_cast<SelState *>(sws + L.sel.st_off);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(sws + L.sel.keys_off);
    const unsigned long long *top = reinterpret_cast<const unsigned long long *>(sws + L.sel.top_off);
    int *status = status_word(err, errlen);
    if (!status) return (int)cudaErrorUnknown;
    cudaError_t e = cudaSuccess;
#define DET_CHECK(what)                                                          \
    do {                                                                         \
        if (e == cudaSuccess) e = cudaGetLastError();                            \
        if (e != cudaSuccess) {                                                  \
            snprintf(err, errlen, "%s: %s", what, cudaGetErrorString(e));        \
            return (int)e;                                                       \
        }                                                                        \
    } while (0)
    {
        // two blocks of four warps per SM, but no chunk shorter than 8 rows
        const int nbx = (W + 127) / 128, chunks = std::max(1, 2 * 152 / nbx);
        const int chunk = std::max({8, (H + chunks - 1) / chunks, (H + 65534) / 65535});
        const dim3 grid((unsigned)nbx, (unsigned)((H + chunk - 1) / chunk));
        Scope sc(kKDetStats, stream);
        k_det_cols<<<grid, 128, 0, stream>>>(a.snr_max, a.argmax, H, W, R, chunk, c1, c2, cn, st);
    }
    DET_CHECK("k_det_cols");
    {
        const int tile = std::min(kRowTile, (W + 31) / 32 * 32);
        const size_t smem = (size_t)(tile + 2 * R + 1) * (8 + 8 + 4);
        e = cudaFuncSetAttribute(k_det_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAllowStatic);
        if (e != cudaSuccess) {
            snprintf(err, errlen, "cudaFuncSetAttribute(k_det_rows): %s", cudaGetErrorString(e));
            return (int)e;
        }
        // below this an FP32 z (the pairs' error, as it stands in z_out, is under
        // 1e-6 of it) cannot belong to a candidate
        const double low = a.threshold - 1e-5 * std::max(1.0, std::fabs(a.threshold));
        const float thr_low = (float)std::max(-3e38, std::min(3e38, low));
        Scope sc(kKDetStats, stream);
        const unsigned grid = (unsigned)(((W + tile - 1) / tile) * (int64_t)H);
        e = launch_after(true, k_det_rows, dim3(grid), dim3(kRowThreads), smem, stream, a.snr_max, a.argmax, c1, c2, cn,
                         H, W, R, tile, a.threshold, thr_low, a.subtract_mean, a.z_out, zd, zmax, peak, npix, parent,
                         cand, st);
    }
    DET_CHECK("k_det_rows");
    {
        Scope sc(kKDetComponents, stream);
        const int g = grid_for(P, 256);
        const auto next = [&](auto kern, auto... args) {
            if (e == cudaSuccess) e = launch_after(true, kern, dim3((unsigned)g), dim3(256), 0, stream, args...);
        };
        next(k_det_union, parent, cand, st, W, status);
        next(k_det_peak_z, parent, cand, st, zd, zmax, npix, status);
        next(k_det_peak_at, parent, cand, st, zd, zmax, peak);
        next(k_det_mark, parent, cand, st, zd, peak, keys);
    }
    DET_CHECK("k_det components");
    if (a.max_out > 0) {
        const int rc = launch_select_list(P, a.max_out, 0, sws, L.sel, stream, err, errlen);
        if (rc) return rc;
    }
    {
        Scope sc(kKDetEmit, stream);
        const int n = a.max_out > 0 ? a.max_out : 1;
        e = launch_after(true, k_det_emit, dim3((unsigned)(n + 7) / 8), dim3(256), 0, stream, top, st, a.max_out, parent,
                         a.snr_max, a.argmax, zd, c1, c2, cn, npix, W, R, a.out, a.n_out);
    }
    DET_CHECK("k_det_emit");
#undef DET_CHECK
    return 0;
}

}  // namespace mf
