// Top-k selection of scores (Section 3.3: the candidates of a search and its
// detections, best first).  Every entry has a unique 64-bit key, (order-
// preserving score bits << 32) | (0xFFFFFFFF - flat index): descending key =
// score descending, then flat index ascending.
//
//   k_sel_hist    counts a map's keys by their top 15 bits, a whole histogram
//                 in each block's shared memory (one shared add per pixel);
//                 the last block to finish finds the bin that holds the
//                 k_top-th largest key;
//   k_sel_gather  the map's keys from that bin upwards into a list: the top
//                 k_top and the rest of one bin (for a score map, about a
//                 thousand more);
//   k_sel_refine  only for a list longer than the ranking takes (massive
//                 ties, a list of very many detections): radix select of the
//                 remaining bits over the list by one cluster, whose eight
//                 CTAs meet at the cluster's own barrier; otherwise it returns
//                 at once;
//   k_sel_rank    a key's place is the number of larger keys: counted for 32
//                 keys per block, the first k_top written in order.
// Keys are unique, so the result does not depend on the list's order.
//
// Bound by the two passes over the map and the launches: 1024^2, k_top 4096:
// 45 us (hist 15, gather 5, refine 2 unused, rank 13) against 409 us for four
// rounds of global 16-bit histograms over a P-long key array, a one-block pick
// each (40 us: strided reads) and a one-block bitonic sort (51 us).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>

#include "mf_device.cuh"
#include "mf_internal.h"

namespace mf {
namespace {

using dev::launch_dependents;
using dev::sel_key;
using dev::wait_previous;

constexpr int kBins = 1 << kSelFirstBits;  // of the first histogram
constexpr int kBinShift = 64 - kSelFirstBits;
constexpr int kThreads = 1024;
constexpr int kCluster = 8;

// For one block of kThreads: the bin of hist[0 .. n) (n a multiple of 1024) at
// which the count from the top reaches `need` (1 .. total), and the count
// above it.  Thread 0 holds the answer in *bin, *above; returns the total.
// The histogram was built by other blocks: read past the L1 cache.
__device__ unsigned int block_pick(const unsigned int *hist, int n, unsigned int need_max, unsigned int *bin,
                                   unsigned int *above, unsigned int *need_out) {
    __shared__ unsigned int wsum[32], wexcl[32];
    __shared__ unsigned int total, s_need, s_bin, s_above;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int seg = n / 32;  // bins of a warp, from the top
    const unsigned int *h = hist + n - (size_t)(warp + 1) * seg;
    unsigned int sum = 0;
    for (int j = 4 * lane; j < seg; j += 128) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(h + j));
        sum += v.x + v.y + v.z + v.w;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) wsum[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        unsigned int inc = wsum[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned int o = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += o;
        }
        wexcl[lane] = inc - wsum[lane];
        if (lane == 31) {
            total = inc;
            s_need = inc < need_max ? inc : need_max;
            s_bin = 0;
            s_above = 0;
        }
    }
    __syncthreads();
    const unsigned int need = s_need;
    if (need > 0 && wexcl[warp] < need && wexcl[warp] + wsum[warp] >= need) {
        // this warp's bins: 32 lanes of seg / 32, lane 0 the topmost
        const int per = seg / 32;
        const unsigned int *hl = h + seg - (size_t)(lane + 1) * per;
        unsigned int mine = 0;
        for (int j = 0; j < per; j++) mine += __ldcg(hl + j);
        unsigned int inc = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned int o = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += o;
        }
        unsigned int acc = wexcl[warp] + inc - mine;
        if (acc < need && acc + mine >= need) {
            int j = per - 1;
            for (; j > 0; j--) {
                const unsigned int c = __ldcg(hl + j);
                if (acc + c >= need) break;
                acc += c;
            }
            s_bin = (unsigned int)(hl + j - hist);
            s_above = acc;
        }
    }
    __syncthreads();
    *bin = s_bin;
    *above = s_above;
    *need_out = need;
    const unsigned int t = total;
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(kThreads) k_sel_hist(const float *__restrict__ score,
                                                       const int32_t *__restrict__ valid, int64_t P,
                                                       unsigned int *__restrict__ hist, SelState *st,
                                                       unsigned int k_top) {
    launch_dependents();
    extern __shared__ unsigned int bins[];
    for (int j = threadIdx.x; j < kBins; j += kThreads) bins[j] = 0u;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < P; i += 4 * stride) {
        float s[4];
        int32_t v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int64_t q = i + u * stride;
            v[u] = q < P ? valid[q] : -1;
            s[u] = q < P ? score[q] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (v[u] >= 0) atomicAdd(&bins[sel_key(s[u], 0u) >> kBinShift], 1u);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kBins; j += kThreads)
        if (bins[j]) atomicAdd(&hist[j], bins[j]);
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) + 1 == gridDim.x;
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned int bin, above, need;
    block_pick(hist, kBins, k_top, &bin, &above, &need);
    if (threadIdx.x == 0) {
        st->prefix = need ? (unsigned long long)bin << kBinShift : ~0ull;
        st->need = need - above;
    }
}

__global__ void __launch_bounds__(256) k_sel_gather(const float *__restrict__ score,
                                                    const int32_t *__restrict__ valid, int64_t P,
                                                    unsigned long long *__restrict__ list, SelState *st) {
    launch_dependents();
    wait_previous();
    const unsigned long long from = st->prefix;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < P; base += 4 * stride) {
        float s[4];
        int32_t v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int64_t q = base + lane + u * stride;
            v[u] = q < P ? valid[q] : -1;
            s[u] = q < P ? score[q] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const unsigned long long key = sel_key(s[u], (uint32_t)(base + lane + u * stride));
            const bool take = v[u] >= 0 && key >= from;
            const unsigned int m = __ballot_sync(0xffffffffu, take);
            if (m == 0) continue;
            unsigned int at = 0;
            if (lane == 0) at = atomicAdd(&st->list, (unsigned int)__popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (take) list[at + __popc(m & ((1u << lane) - 1u))] = key;
        }
    }
}

// fixed_bits: key bits already fixed by st->prefix (with st->need keys wanted
// among those that share them); 0: none, the k_top-th of the whole list is
// wanted.
__global__ void __cluster_dims__(kCluster) __launch_bounds__(kThreads)
    k_sel_refine(const unsigned long long *list, unsigned int *hist, SelState *st, unsigned int k_top,
                 unsigned int limit, int fixed_bits) {
    launch_dependents();
    wait_previous();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const unsigned int n = st->list;
    if (n <= limit) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->n = n;
            st->refined = 0u;
            st->count = n < k_top ? n : k_top;
        }
        return;  // the same for every CTA of the cluster
    }
    const unsigned int gtid = blockIdx.x * kThreads + threadIdx.x, gsize = kCluster * kThreads;
    unsigned long long prefix = fixed_bits ? st->prefix : 0ull;
    unsigned int need = fixed_bits ? st->need : k_top;  // n > limit > k_top
    for (int lo = 64 - fixed_bits; lo > 0;) {
        const int width = lo < 16 ? lo : 16;
        for (unsigned int j = gtid; j < 65536u; j += gsize) hist[j] = 0u;
        __threadfence();
        cl.sync();
        for (unsigned int i = gtid; i < (n + 31u) / 32u * 32u; i += gsize) {
            const unsigned long long key = i < n ? list[i] : 0ull;
            const bool in = i < n && (lo == 64 || (key >> (lo & 63)) == (prefix >> (lo & 63)));
            const unsigned int bin = in ? (unsigned int)(key >> (lo - width)) & ((1u << width) - 1u) : 0xFFFFFFFFu;
            const unsigned int same = __match_any_sync(0xffffffffu, bin);
            if (in && (threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&hist[bin], (unsigned int)__popc(same));
        }
        __threadfence();
        cl.sync();
        unsigned int bin, above, wanted;
        block_pick(hist, 65536, need, &bin, &above, &wanted);  // every CTA for itself
        const unsigned int here = __ldcg(hist + bin);
        prefix |= (unsigned long long)bin << (lo - width);
        need -= above;
        lo -= width;
        cl.sync();  // every CTA has read the histogram
        if (here == need) break;  // the whole bin is wanted: keys from prefix upwards
    }
    // the k_top keys at or above the prefix, into the histogram's space
    unsigned long long *out = reinterpret_cast<unsigned long long *>(hist);
    for (unsigned int i = gtid; i < n; i += gsize) {
        const unsigned long long key = list[i];
        if (key >= prefix) {
            const unsigned int at = atomicAdd(&st->n, 1u);
            if (at < k_top) out[at] = key;
        }
    }
    if (gtid == 0) {
        st->refined = 1u;
        st->count = k_top;
    }
}

__global__ void __launch_bounds__(256) k_sel_rank(const unsigned long long *list,
                                                  const unsigned long long *refined, const SelState *st,
                                                  unsigned int k_top, unsigned long long *__restrict__ top) {
    launch_dependents();
    wait_previous();
    constexpr unsigned int kTile = 2048;  // keys staged at a time
    __shared__ __align__(16) unsigned long long tile[kTile];
    __shared__ unsigned int part[8][32];
    const unsigned int n = st->n, first = blockIdx.x * 32u;
    if (first >= n) return;
    const unsigned long long *src = st->refined ? refined : list;
    const unsigned int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long mine = first + lane < n ? src[first + lane] : ~0ull;
    unsigned int larger = 0;
    for (unsigned int t = 0; t < n; t += kTile) {
        __syncthreads();
#pragma unroll
        for (unsigned int j = 0; j < kTile; j += 256) {
            const unsigned int q = t + j + threadIdx.x;
            tile[j + threadIdx.x] = q < n ? src[q] : 0ull;  // 0 is below every key
        }
        __syncthreads();
        const ulonglong2 *two = reinterpret_cast<const ulonglong2 *>(tile) + warp * (kTile / 16);
#pragma unroll 8
        for (unsigned int j = 0; j < kTile / 16; j++) {  // the warp's eighth, two keys per read
            const ulonglong2 o = two[j];
            larger += (o.x > mine) + (o.y > mine);
        }
    }
    part[warp][lane] = larger;
    __syncthreads();
    if (warp == 0 && first + lane < n) {
        unsigned int rank = 0;
#pragma unroll
        for (int w = 0; w < 8; w++) rank += part[w][lane];
        if (rank < k_top) top[rank] = mine;
    }
}

struct Scope {
    ProfToken t;
    Scope(int kid, cudaStream_t s) : t(prof_begin(kid, s)) {}
    ~Scope() { prof_end(t); }
};

#define SEL_CHECK(what)                                                   \
    do {                                                                  \
        if (e == cudaSuccess) e = cudaGetLastError();                     \
        if (e != cudaSuccess) {                                           \
            snprintf(err, errlen, "%s: %s", what, cudaGetErrorString(e)); \
            return (int)e;                                                \
        }                                                                 \
    } while (0)

}  // namespace

SelectLayout select_layout(int64_t P, int32_t k_top) {
    SelectLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = (off + bytes + 255) / 256 * 256;
        return o;
    };
    L.keys_off = take((size_t)P * sizeof(unsigned long long));
    L.hist_off = take(65536 * sizeof(unsigned int));
    L.st_off = take(sizeof(SelState));
    L.top_off = take((size_t)k_top * sizeof(unsigned long long));
    L.total = off;
    return L;
}

// Keys a list may hold for the ranking to count them all: beyond the k_top,
// the rest of one bin of the first histogram.  The ranking grows with the
// square of the list, so a longer list is cut to k_top first.
static unsigned int rank_limit(int32_t k_top) { return (unsigned int)k_top + 8192u; }

int launch_select_list(int64_t P, int32_t k_top, int fixed_bits, char *ws, const SelectLayout &L, void *stream_,
                       char *err, size_t errlen) {
    cudaStream_t stream = (cudaStream_t)stream_;
    unsigned long long *list = reinterpret_cast<unsigned long long *>(ws + L.keys_off);
    unsigned int *hist = reinterpret_cast<unsigned int *>(ws + L.hist_off);
    SelState *st = reinterpret_cast<SelState *>(ws + L.st_off);
    unsigned long long *top = reinterpret_cast<unsigned long long *>(ws + L.top_off);
    const unsigned int limit = rank_limit(k_top);
    cudaError_t e = cudaSuccess;
    {
        Scope sc(kKCompact, stream);
        e = launch_after(true, k_sel_refine, dim3(kCluster), dim3(kThreads), 0, stream, list, hist, st, (unsigned)k_top,
                         limit, fixed_bits);
    }
    SEL_CHECK("k_sel_refine");
    {
        const int64_t most = P < (int64_t)limit ? P : (int64_t)limit;
        Scope sc(kKSort, stream);
        e = launch_after(true, k_sel_rank, dim3((unsigned)((most + 31) / 32)), dim3(256), 0, stream, list,
                         reinterpret_cast<const unsigned long long *>(hist), st, (unsigned)k_top, top);
    }
    SEL_CHECK("k_sel_rank");
    return 0;
}

int launch_select(const float *score, const int32_t *valid, int64_t P, int32_t k_top, char *ws,
                  const SelectLayout &L, void *stream_, char *err, size_t errlen) {
    cudaStream_t stream = (cudaStream_t)stream_;
    if (k_top > kMaxTop) {
        snprintf(err, errlen, "k_top above %d", kMaxTop);
        return (int)cudaErrorInvalidValue;
    }
    unsigned long long *list = reinterpret_cast<unsigned long long *>(ws + L.keys_off);
    unsigned int *hist = reinterpret_cast<unsigned int *>(ws + L.hist_off);
    SelState *st = reinterpret_cast<SelState *>(ws + L.st_off);
    cudaError_t e = cudaMemsetAsync(ws + L.hist_off, 0, L.top_off - L.hist_off, stream);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sel_hist, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kBins * sizeof(unsigned int)));
    if (e != cudaSuccess) {
        snprintf(err, errlen, "top-k set-up: %s", cudaGetErrorString(e));
        return (int)e;
    }
    auto blocks = [&](int64_t per, int64_t most) {
        const int64_t b = (P + per - 1) / per;
        return (unsigned)(b < most ? b : most);
    };
    {
        Scope sc(kKSelect, stream);
        k_sel_hist<<<blocks(4 * kThreads, 152), kThreads, kBins * sizeof(unsigned int), stream>>>(
            score, valid, P, hist, st, (unsigned)k_top);
    }
    SEL_CHECK("k_sel_hist");
    {
        Scope sc(kKSelect, stream);
        e = launch_after(true, k_sel_gather, dim3(blocks(4 * 256, 152 * 8)), dim3(256), 0, stream, score, valid, P,
                         list, st);
    }
    SEL_CHECK("k_sel_gather");
    return launch_select_list(P, k_top, kSelFirstBits, ws, L, stream, err, errlen);
}

}  // namespace mf
