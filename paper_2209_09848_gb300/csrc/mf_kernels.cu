// Device side of libmf: the matched-filter search of Ganapathi (2022),
// Section 3.2 (Eq. 5 and the maximum over the filter bank), for sm_103a.
//
// Kernels, in launch order (of a factored search, whose numerator is in
// mf_factored.cu: the denominator after it):
//   k_lambda       inverse variance lambda = (1 - m) / sigma^2 into a zero-
//                  padded image (Section 3.2 noise model; clipped pixels and
//                  pixels outside the frame weigh 0);
//   k_weight       y_t = lambda * r_t, the inverse-variance weighted stack;
//   k_denominator  D_k(p) = sum_t sum_ab W^2 lambda, from runs of frames with
//                  a constant base shift, FP32 products accumulated in FP64;
//                  stores 1 / sqrt(D);
//   k_numerator    N_k(p) = sum_t sum_ab W y_t, the gather stencil: frame
//                  windows staged in shared memory by TMA and reused by the
//                  2 to 16 trajectories of a CTA, 25 FP32 FMAs per
//                  (trajectory, pixel, frame); epilogue forms SNR, reduces the
//                  max / argmax over the CTA's trajectories and merges it into
//                  a per-pixel 64-bit key with atomicMax;
//   k_finalize     key -> (snr_max, argmax).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdio>
#include <type_traits>
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "mf_device.cuh"
#include "mf_internal.h"

namespace mf {

// Device status word: 0, or the code of a bounded wait that gave up.
__device__ int g_status;

namespace {

using namespace dev;

// A bounded wait that records a failure in the device-wide word (the search
// kernels record theirs in their own search's status slot instead).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int code) {
    return dev::mbar_wait(bar, parity, code, &g_status);
}

template <typename T>
__device__ __forceinline__ float to_f32(T v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ float to_f32<__half>(__half v) { return __half2float(v); }

// ------------------------------------------------------------- lambda ---

// Also the search's status area (16 bytes): LMAX (cleared before): the largest
// lambda, into its third word (lambda >= 0, so the float bits order as unsigned
// integers); otherwise it is cleared here (a fill of its own would be one more
// operation in the stream).
template <bool LMAX>
__global__ void k_lambda(const float *__restrict__ sigma, const uint8_t *__restrict__ mask, int64_t H,
                         int64_t W, int64_t pad, int64_t lw, int64_t lh, float *__restrict__ lam,
                         unsigned int *status_area) {
    launch_dependents();
    if (!LMAX && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 4) status_area[threadIdx.x] = 0u;
    float vmax = 0.f;
    for (int64_t row = blockIdx.y; row < lh; row += gridDim.y)
        for (int64_t col = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; col < lw;
             col += (int64_t)gridDim.x * blockDim.x) {
            const int64_t yy = row - pad, xx = col - pad;
            float v = 0.f;
            if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
                const int64_t q = yy * W + xx;
                const float s = sigma[q];
                const bool m = mask ? (mask[q] != 0) : false;
                if (!m && s > 0.f && isfinite(s)) v = (float)(1.0 / ((double)s * (double)s));
            }
            lam[row * lw + col] = v;
            vmax = fmaxf(vmax, v);
        }
    if constexpr (LMAX) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if ((threadIdx.x & 31) == 0 && vmax > 0.f) atomicMax(status_area + 2, __float_as_uint(vmax));
    }
}

// ------------------------------------------------------------- weight ---

// y_t = lambda * (scale_t * r_t) in FP32; stored as FP32 (TOut = float) or
// in the stack's own 16-bit type (TOut = TIn): bf16 as is (beta_t = 1), fp16
// times 1 / beta_t, beta_t the power of two at or above lambda_max * scale_t,
// (of |scale_t|), so that no value overflows (|stored r| <= 65504) and the
// scaling is exact.
// The thread of (frame t, row 0, first column quad) writes beta[t].
__device__ __forceinline__ float fp16_frame_beta(float lmax, float sc, float *inv) {
    const float x = lmax * sc;
    if (!(x > 0.f)) {
        *inv = 1.f;
        return 1.f;
    }
    // x = 1.m * 2^(e - 127) <= 2^(e - 126): beta = 2^(e - 126), from the bits
    const int e = min((int)((__float_as_uint(x) >> 23) & 0xFFu), 253);
    *inv = __uint_as_float((uint32_t)(253 - e) << 23);  // 2^(126 - e)
    return __uint_as_float((uint32_t)(e + 1) << 23);    // 2^(e - 126)
}

template <typename T>
__device__ __forceinline__ T from_f32(float v);
template <>
__device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ __half from_f32<__half>(float v) { return __float2half_rn(v); }

// Four consecutive stack values as FP32, from one 128-bit (FP32) or 64-bit
// (16-bit types) read: p is aligned to four elements.
template <typename T>
__device__ __forceinline__ void load4_f32(const T *p, float v[4]) {
    if constexpr (sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const uint2 q = *reinterpret_cast<const uint2 *>(p);
        const T *e = reinterpret_cast<const T *>(&q);
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] = to_f32(e[j]);
    }
}

// y_t = lambda * (scale_t * r_t) (16-bit outputs of an fp16 stack also times
// 2^-e_t, exact).  A warp takes one (frame, row) at a time, so the row's
// index split is made once per row; lanes walk the row four values each,
// reading lambda and writing y with aligned vector accesses and the stack
// with them too when its rows allow (VR: aligned base, strides multiples of
// four elements).
template <typename TIn, typename TOut, bool VR>
__global__ void k_weight(const TIn *__restrict__ r, int64_t fstride, int64_t rstride,
                         const float *__restrict__ scale, const float *__restrict__ lam, int64_t pad, int64_t lw,
                         TOut *__restrict__ y, int64_t T, int64_t H, int64_t W, int64_t yp,
                         const unsigned int *lmax_bits, float *__restrict__ beta) {
    constexpr bool kHalfScaled = std::is_same<TOut, __half>::value;
    // in this order: a general search's k_den_box starts from here and reads
    // lambda, this kernel's input, without a wait of its own
    wait_previous();
    launch_dependents();
    const float lmax = kHalfScaled ? __uint_as_float(*lmax_bits) : 0.f;
    const int64_t wq = (W + 3) / 4, rows = T * H;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t ri = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); ri < rows; ri += nwarps) {
        const int64_t t = ri / H, yy = ri - t * H;
        const float sc = scale ? scale[t] : 1.f;
        float inv = 1.f, bt = 1.f;
        if (kHalfScaled) bt = fp16_frame_beta(lmax, fabsf(sc), &inv);
        if (beta && yy == 0 && lane == 0) beta[t] = bt;
        const float *lrow = lam + (yy + pad) * lw + pad;  // padded: columns W .. W + 3 exist
        const TIn *rrow = r + t * fstride + yy * rstride;
        TOut *yrow = y + ri * yp;
        // two chunks of four pixels a lane, their loads before their stores (1000
        // x 2048^2 frames: 5.42 ms, one after the other 5.85, four chunks 5.36;
        // 600 x 512^2 bf16: 0.17 ms, four chunks 0.20)
        constexpr int NC = 2;
        for (int64_t xb = lane; xb < wq; xb += 32 * NC) {
            float4 l4[NC] = {};
            float v[NC][4] = {};
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const int64_t x0 = (xb + 32 * c) * 4;
                if (x0 >= W) continue;
                load_awaited(l4[c], reinterpret_cast<const float4 *>(lrow + x0));
                if (VR && x0 + 4 <= W) {
                    load4_f32(rrow + x0, v[c]);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; j++) v[c][j] = x0 + j < W ? to_f32(rrow[x0 + j]) : 0.f;
                }
            }
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const int64_t x0 = (xb + 32 * c) * 4;
                if (x0 >= W) continue;
                const float l[4] = {l4[c].x, l4[c].y, l4[c].z, l4[c].w};
                float o[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    o[j] = (x0 + j < W) ? l[j] * (sc * v[c][j]) : 0.f;
                    if (kHalfScaled) o[j] *= inv;  // a power of two: exact
                }
                TOut *dst = yrow + x0;
                if (std::is_same<TOut, float>::value) {
                    *reinterpret_cast<float4 *>(dst) = make_float4(o[0], o[1], o[2], o[3]);
                } else {
                    TOut q[4] = {from_f32<TOut>(o[0]), from_f32<TOut>(o[1]), from_f32<TOut>(o[2]),
                                 from_f32<TOut>(o[3])};
                    *reinterpret_cast<uint2 *>(dst) = *reinterpret_cast<const uint2 *>(q);
                }
            }
        }
    }
}

// -------------------------------------------------------- denominator ---

// D_k(p) = sum_u G_k(u) lambda(p + u) over the rows (runs) of the collapsed
// kernel G_k.  A thread owns 8 consecutive start pixels of one row, a warp 256
// of them, a CTA 8 rows; blockIdx.y walks the trajectories.  For each run the
// thread slides an 8-wide register window along the lambda row (one aligned
// float4 per 4 taps), so every loaded value feeds 8 FMAs.  Products and
// partial sums are FP32 over at most kDenTaps taps; the partials are added in
// FP64.  The result is stored as 1 / sqrt(D) (0 where D = 0).
__global__ void __launch_bounds__(256) k_denominator(const float *__restrict__ lam, int64_t lw, int64_t pad,
                                                     const RunRec *__restrict__ runs,
                                                     const int32_t *__restrict__ run_off,
                                                     const float *__restrict__ wts, int K, int64_t H, int64_t W,
                                                     int nbx, float *__restrict__ isd) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t py = (int64_t)(blockIdx.x / nbx) * 8 + warp;
    const int64_t px0 = (int64_t)(blockIdx.x % nbx) * kDenCols + 8 * lane;
    const int64_t P = H * W;
    for (int k = blockIdx.y; k < K; k += gridDim.y) {
        double d[8];
        float a[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {
            d[c] = 0.0;
            a[c] = 0.f;
        }
        int taps = 0;
        const int r0 = run_off[k], r1 = run_off[k + 1];
        for (int r = r0; r < r1; r++) {
            const RunRec rr = runs[r];
            const float4 *row = reinterpret_cast<const float4 *>(lam + (py + rr.dy + pad) * lw + px0 + rr.x0 + pad);
            const float4 *wp = reinterpret_cast<const float4 *>(wts + rr.woff);
            // 12-value window of lambda in three float4 slots that rotate:
            // chunk ch (4 taps) uses slot ch mod 3 onwards and, before its
            // FMAs, loads the slot two ahead; unrolled by 3 so that every
            // register index is static
            float v[12];
            {
                const float4 p0 = __ldg(row), p1 = __ldg(row + 1);
                v[0] = p0.x; v[1] = p0.y; v[2] = p0.z; v[3] = p0.w;
                v[4] = p1.x; v[5] = p1.y; v[6] = p1.z; v[7] = p1.w;
            }
            for (int ch = 0; ch < rr.nch; ch += 3) {
#pragma unroll
                for (int u = 0; u < 3; u++) {
                    if (ch + u < rr.nch) {
                        const float4 pn = __ldg(row + ch + u + 2);
                        const int ns = ((u + 2) % 3) * 4;  // slot receiving columns 4 (ch + u + 2) ..
                        v[ns] = pn.x; v[ns + 1] = pn.y; v[ns + 2] = pn.z; v[ns + 3] = pn.w;
                        const float4 w4 = __ldg(wp + ch + u);
                        const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                        for (int i = 0; i < 4; i++)
#pragma unroll
                            for (int c = 0; c < 8; c++) a[c] = fmaf(w[i], v[(4 * u + i + c) % 12], a[c]);
                    }
                }
            }
            taps += rr.nch * 4;
            if (taps >= kDenTaps) {
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    d[c] += (double)a[c];
                    a[c] = 0.f;
                }
                taps = 0;
            }
        }
        if (py < H) {
#pragma unroll
            for (int c = 0; c < 8; c++) {
                const double dd = d[c] + (double)a[c];
                const int64_t px = px0 + c;
                if (px < W) isd[(int64_t)k * P + py * W + px] = dd > 0.0 ? rsqrtf((float)dd) : 0.f;
            }
        }
    }
}

// One run of N chunks (4 taps each) for NO start pixels: every index is known
// at compile time.
template <int N, int NO>
__device__ __forceinline__ void den_run(const float4 *row, const float4 *wp, float (&a)[NO]) {
    float v[4 * (N + NO / 4)];
#pragma unroll
    for (int q = 0; q < N + NO / 4; q++) {
        const float4 x = row[q];
        v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
    }
#pragma unroll
    for (int ch = 0; ch < N; ch++) {
        const float4 w4 = wp[ch];
        const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int c = 0; c < NO; c++) a[c] = fmaf(w[i], v[4 * ch + i + c], a[c]);
    }
}

// The same sums from a staged box.  A CTA owns `th` rows x C start pixels of
// one trajectory k: it copies the lambda box its start pixels reach through G_k
// (rows dy0 .., columns x0 .. of the box, plus the tile), G_k's weights and its
// runs into shared memory.  A thread then owns NO consecutive start pixels of
// one tile row and slides an NO-wide register window along each run, so that
// every 128-bit read of lambda feeds 4 NO FMAs.  A warp covers 8 rows x 4 NO
// columns: the 8 threads of a quarter warp hold the same columns of 8
// consecutive rows, which an odd row pitch (in 16-byte chunks) puts in 8
// distinct bank groups, so the reads are conflict-free at plain row-major
// addresses (base + chunk, no per-read index arithmetic).  Same FP32 products,
// same FP64 accumulation as k_denominator; the partials are widened by bits (a
// conversion would cost a second FP64 operation each).
template <int NO, int C>
__global__ void __launch_bounds__(32 * C / NO, 256 / C) k_den_box(
    const float *__restrict__ lam, int64_t lw, int64_t lh, int64_t pad, const RunRec *__restrict__ runs,
    const int32_t *__restrict__ run_off, const float *__restrict__ wts, const DenBox *__restrict__ boxes, int K,
    int64_t H, int64_t W, int nbx, int th, float *__restrict__ isd) {
    static_assert(NO % 4 == 0 && C % (4 * NO) == 0, "whole chunks, whole warps per 8 rows");
    constexpr int WR = C / (4 * NO);  // warps per 8 tile rows
    extern __shared__ __align__(16) float4 dsm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tile row y and first column xs of this thread's NO start pixels
    const int y = 8 * (warp / WR) + (lane & 7), xs = 4 * NO * (warp % WR) + NO * (lane >> 3);
    const int64_t py = (int64_t)(blockIdx.x / nbx) * th + y;
    const int64_t px0 = (int64_t)(blockIdx.x % nbx) * C;
    const int64_t P = H * W;
    const bool vec = (W & 3) == 0;  // rows (and planes) start on 16-byte boundaries
    for (int k = blockIdx.y; k < K; k += gridDim.y) {
        const DenBox bx = boxes[k];
        const int R = th + bx.rows - 1, NC = (C + bx.cols) / 4, PC = den_pitch(bx.cols, C);
        const int r0 = run_off[k], nr = run_off[k + 1] - r0;
        float4 *wsm = dsm + (size_t)R * PC;                           // weights after the box
        RunRec *rsm = reinterpret_cast<RunRec *>(wsm + bx.nw / 4);    // then the runs
        __syncthreads();                                               // the previous trajectory's reads are done
        // lambda rows py0 + dy0 .. of the padded image (zero beyond its last row)
        const int64_t gy0 = py - y + bx.dy0 + pad, gx0 = px0 + bx.x0 + pad;
        for (int i = threadIdx.x; i < R * NC; i += blockDim.x) {
            const int r = i / NC, j = i % NC;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gy0 + r < lh) v = __ldg(reinterpret_cast<const float4 *>(lam + (gy0 + r) * lw + gx0) + j);
            dsm[(size_t)r * PC + j] = v;
        }
        for (int i = threadIdx.x; i < bx.nw / 4; i += blockDim.x)
            wsm[i] = __ldg(reinterpret_cast<const float4 *>(wts + bx.w0) + i);
        // a run's first chunk and weights relative to the box
        for (int i = threadIdx.x; i < nr; i += blockDim.x) {
            RunRec rr = runs[r0 + i];
            rr.dy = (rr.dy - bx.dy0) * PC + (rr.x0 - bx.x0) / 4;
            rr.woff = (rr.woff - bx.w0) / 4;
            rsm[i] = rr;
        }
        __syncthreads();
        if (py >= H || px0 + xs >= W) continue;
        double d[NO];
        float a[NO];
#pragma unroll
        for (int c = 0; c < NO; c++) {
            d[c] = 0.0;
            a[c] = 0.f;
        }
        const float4 *mine = dsm + y * PC + xs / 4;
        int taps = 0;
        for (int r = 0; r < nr; r++) {
            const RunRec rr = rsm[r];
            const float4 *row = mine + rr.dy, *wp = wsm + rr.woff;
            // a slow mover's runs have two to four chunks
            switch (rr.nch) {
                case 1: den_run<1, NO>(row, wp, a); break;
                case 2: den_run<2, NO>(row, wp, a); break;
                case 3: den_run<3, NO>(row, wp, a); break;
                case 4: den_run<4, NO>(row, wp, a); break;
                case 5: den_run<5, NO>(row, wp, a); break;
                default: {
                    int ch = 0;
                    for (; ch + 4 <= rr.nch; ch += 4) den_run<4, NO>(row + ch, wp + ch, a);
                    for (; ch < rr.nch; ch++) den_run<1, NO>(row + ch, wp + ch, a);
                }
            }
            taps += rr.nch * 4;
            if (taps >= kDenTaps) {
#pragma unroll
                for (int c = 0; c < NO; c++) {
                    d[c] += widen(a[c]);
                    a[c] = 0.f;
                }
                taps = 0;
            }
        }
        float o[NO];
#pragma unroll
        for (int c = 0; c < NO; c++) {
            const double dd = d[c] + widen(a[c]);
            const long long bits = __double_as_longlong(dd);  // dd > 0, by its bits (NaN is not)
            o[c] = bits > 0 && bits <= 0x7FF0000000000000ll ? rsqrtf((float)dd) : 0.f;
        }
        const int64_t px = px0 + xs;
        float *dst = isd + (int64_t)k * P + py * W + px;
        if (vec && px + NO <= W) {
#pragma unroll
            for (int q = 0; q < NO / 4; q++)
                reinterpret_cast<float4 *>(dst)[q] = make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
        } else {
#pragma unroll
            for (int c = 0; c < NO; c++)
                if (px + c < W) dst[c] = o[c];
        }
    }
    // started early, it ends after the kernel before it: what follows may read
    // what both wrote
    launch_dependents();
    if (blockIdx.x == 0 && blockIdx.y == 0) wait_previous();
}

// ---------------------------------------------------------- numerator ---

struct NumParams {
    const unsigned char *blocks;  // [G][T] frame blocks
    const FrameHdr *hdr;          // [G][T]
    const float *isd;             // [K][H][W]
    unsigned long long *keys;     // [H][W]
    float *snr_all;               // [K][H][W] or null
    int *status;                  // the search's status slot
    int T, G;
    int64_t H, W;
    int tiles_x;
    int S, BH;
    int lockstep;  // 1: CTA barrier after every frame; 0: the last warp out refills the stage
};

// Column skew of lane row-group ty for window loads of VEC floats: it keeps
// the lanes of every shared-memory wavefront on distinct banks (pitch a
// multiple of 32 words) and is a multiple of VEC, so a lane's row segment
// starts VEC-aligned whenever the warp's window offset is.
template <int VEC>
__device__ __forceinline__ int lane_skew(int ty) {
    return VEC == 1 ? ty : (VEC == 2 ? 2 * (ty & 3) : 4 * (ty & 1));
}

// The 4 x 8 block of one lane for one (trajectory, frame): 8 window rows of
// 12 values each, 25 FMAs per output.  `base` is the lane's first window value
// minus M (so VEC-aligned); M = window offset mod VEC is a compile-time
// constant of the variant, so the row segment is read with aligned VEC-wide
// loads and the register selection costs nothing.
template <int VEC, int M>
__device__ __forceinline__ void stencil_4x8(const float *__restrict__ base, int S, const float (&w)[28],
                                            float (&blk)[kMicroRows][kMicroCols]) {
    constexpr int NV = (kMicroCols + 4 + M + VEC - 1) / VEC;  // vector loads per row
#pragma unroll
    for (int i = 0; i < kMicroRows + 4; i++) {
        float f[NV * VEC];
        const float *rp = base + i * S;
#pragma unroll
        for (int q = 0; q < NV; q++) {
            if (VEC == 4) {
                const float4 x = reinterpret_cast<const float4 *>(rp)[q];
                f[4 * q] = x.x;
                f[4 * q + 1] = x.y;
                f[4 * q + 2] = x.z;
                f[4 * q + 3] = x.w;
            } else if (VEC == 2) {
                const float2 x = reinterpret_cast<const float2 *>(rp)[q];
                f[2 * q] = x.x;
                f[2 * q + 1] = x.y;
            } else {
                f[q] = rp[q];
            }
        }
#pragma unroll
        for (int r = 0; r < kMicroRows; r++) {
            const int a = i - r;
            if (a < 0 || a > 4) continue;
#pragma unroll
            for (int c = 0; c < kMicroCols; c++)
#pragma unroll
                for (int b = 0; b < 5; b++) blk[r][c] = fmaf(w[a * 5 + b], f[M + c + b], blk[r][c]);
        }
    }
}

template <int VEC>
__device__ __forceinline__ void stencil_dispatch(const float *__restrict__ base, int m, int S, const float (&w)[28],
                                                 float (&blk)[kMicroRows][kMicroCols]) {
    if (VEC == 1) {
        stencil_4x8<1, 0>(base, S, w, blk);
    } else if (VEC == 2) {
        if (m == 0) stencil_4x8<2, 0>(base, S, w, blk);
        else stencil_4x8<2, 1>(base - 1, S, w, blk);
    } else {
        switch (m) {
            case 0: stencil_4x8<4, 0>(base, S, w, blk); break;
            case 1: stencil_4x8<4, 1>(base - 1, S, w, blk); break;
            case 2: stencil_4x8<4, 2>(base - 2, S, w, blk); break;
            default: stencil_4x8<4, 3>(base - 3, S, w, blk); break;
        }
    }
}

// One CTA: an output tile of (32 TYS) x (32 TXS) start pixels for KT
// trajectories, one (trajectory, sub-tile) pair per warp, kWarps warps or half
// of them (see numerator_halves).
// The work of one CTA on one (output tile, trajectory group): returns false
// if it gave up (a bounded wait ran out; the device status word says why).
// `smem` is the CTA's 1024-aligned dynamic shared memory, derived from the
// extern array so that its loads stay shared-memory loads.
template <int KT, int TXS, int TYS, int VEC>
__device__ __forceinline__ bool numerator_tile(const CUtensorMap *ymap, const NumParams &p, int g, int tile,
                                               unsigned char *smem) {
    constexpr int NW = KT * TXS * TYS;
    static_assert(NW == kWarps || NW == kWarps / 2, "one warp per (trajectory, sub-tile)");
    constexpr int NS = kStages;
    constexpr int TH = kTile * TYS, TW = kTile * TXS;
    constexpr uint32_t kBlockBytes = (uint32_t)(sizeof(FrameHdr) + KT * sizeof(SlotRec));
    constexpr int R = kRecordChunk;  // frames per record chunk
    static_assert(R >= NS, "a record chunk must outlive the frames in flight");
    const int win_floats = p.BH * p.S;
    float *win = reinterpret_cast<float *>(smem);
    unsigned char *fb = smem + (size_t)NS * win_floats * sizeof(float);  // NS frame blocks
    uint64_t *bars = reinterpret_cast<uint64_t *>(fb + 2 * R * kBlockBytes);  // fb: 2 chunks of R blocks
    int *cnt = reinterpret_cast<int *>(bars + NS);
    int *last_issued = cnt + NS;
    int *bad_flag = last_issued + NS;
    unsigned long long *red = reinterpret_cast<unsigned long long *>(smem);  // epilogue reuses the windows

    const int tile_y0 = (tile / p.tiles_x) * TH;
    const int tile_x0 = (tile % p.tiles_x) * TW + kTileOriginX;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = warp % KT, sub = warp / KT;
    const int stx = sub % TXS, sty = sub / TXS;
    const int tx = lane & 3, ty = lane >> 2;
    const int skew = lane_skew<VEC>(ty);
    const unsigned char *gblocks = p.blocks + (size_t)g * p.T * kBlockBytes;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; s++) {
            mbar_init(smem_u32(&bars[s]), 1);
            cnt[s] = 0;
            last_issued[s] = -1;
        }
        *bad_flag = dev::status_now(p.status);  // an earlier CTA of this search gave up: do not start
        fence_barrier_init();
    }
    __syncthreads();
    if (*bad_flag != 0) return false;  // same value for every thread of the CTA

    // Load frame f into stage s: the rows the group's window needs at frame f
    // (TMA, zero fill outside the frame) and the frame's slot records.
    auto issue = [&](int f, int s, FrameHdr h) {
        // one box of the whole window (BH x S): every TMA operation costs the
        // CTA's shared-memory pipeline more than the rows it would save
        const uint32_t bar = smem_u32(&bars[s]);
        // the first frame of a chunk also brings the records of the chunk's
        // frames (its buffer last held chunk f / R - 2, long released)
        const int nrec = (f % R == 0) ? min(R, p.T - f) : 0;
        mbar_expect_tx(bar, (uint32_t)win_floats * 4 + (uint32_t)nrec * kBlockBytes);
        tma_load_3d(smem_u32(win + (size_t)s * win_floats), ymap, tile_x0 + h.rox, tile_y0 + h.roy, f, bar);
        if (nrec)
            bulk_load(smem_u32(fb + ((f / R) & 1) * R * kBlockBytes), gblocks + (size_t)f * kBlockBytes,
                      (uint32_t)nrec * kBlockBytes, bar);
        last_issued[s] = f;
    };
    if (threadIdx.x == 0) {
        fence_proxy_async();  // earlier generic writes to these buffers precede the copies
        for (int s = 0; s < NS && s < p.T; s++) issue(s, s, p.hdr[(size_t)g * p.T + s]);
    }

    // A warp whose sub-tile lies entirely outside the image only keeps pace.
    const int sub_y0 = tile_y0 + kTile * sty, sub_x0 = tile_x0 + kTile * stx;
    const bool inside = sub_y0 < p.H && sub_x0 + kTile + 7 > 0 && sub_x0 < p.W;

    float acc[kMicroRows][kMicroCols], blk[kMicroRows][kMicroCols];
#pragma unroll
    for (int r = 0; r < kMicroRows; r++)
#pragma unroll
        for (int c = 0; c < kMicroCols; c++) {
            acc[r][c] = 0.f;
            blk[r][c] = 0.f;
        }
    int kk = -1;
    bool bad = false;
    bool next_ready = false;  // frame t's data already seen complete during frame t - 1
    // lane's offset in a window; stage and barrier phase advance incrementally
    const int lane_off = (kTile * sty + kMicroRows * ty) * p.S + kTile * stx + kMicroCols * tx + skew;
    int s = 0;
    uint32_t par = 0;
    for (int t = 0; t < p.T; t++) {
        const int s1 = (s + 1 == NS) ? 0 : s + 1;            // stage and phase of frame t + 1
        const uint32_t par1 = (s + 1 == NS) ? (par ^ 1u) : par;
        const bool ready = next_ready || dev::mbar_wait(smem_u32(&bars[s]), par, 1, p.status);
        if (!ready && !p.lockstep) {
            bad = true;
            break;
        }
        const unsigned char *fblk = fb + (((t / R) & 1) * R + t % R) * kBlockBytes;  // frame t's block
        const SlotRec *rec = reinterpret_cast<const SlotRec *>(fblk + sizeof(FrameHdr)) + slot;
        kk = rec->k;
        // Look at the next frame's barrier now: the check's latency then hides
        // behind this frame's arithmetic instead of stalling the next frame.
        next_ready = !p.lockstep && t + 1 < p.T && mbar_test_wait(smem_u32(&bars[s1]), par1);
        if (ready && kk >= 0 && inside) {
            float w[28];
            const float4 *w4 = reinterpret_cast<const float4 *>(rec->taps);
#pragma unroll
            for (int i = 0; i < 7; i++) {
                const float4 v = w4[i];
                w[4 * i + 0] = v.x;
                w[4 * i + 1] = v.y;
                w[4 * i + 2] = v.z;
                w[4 * i + 3] = v.w;
            }
            const int offy = __float_as_int(w[25]);
            const int offx = __float_as_int(w[26]);
            const float *base = win + (size_t)s * win_floats + offy * p.S + offx + lane_off;
            stencil_dispatch<VEC>(base, offx & (VEC - 1), p.S, w, blk);
        }
        if ((t + 1) % kFrameBlock == 0) {
#pragma unroll
            for (int r = 0; r < kMicroRows; r++)
#pragma unroll
                for (int c = 0; c < kMicroCols; c++) {
                    acc[r][c] += blk[r][c];
                    blk[r][c] = 0.f;
                }
        }
        if (p.lockstep) {
            // every warp is done with stage s: refill it with frame t + NS
            if (__syncthreads_or(!ready)) {
                bad = true;
                break;
            }
            if (threadIdx.x == 0 && t + NS < p.T) {
                const FrameHdr h = *reinterpret_cast<const FrameHdr *>(fblk);
                fence_proxy_async();
                issue(t + NS, s, h);
            }
            s = s1;
            par = par1;
            continue;
        }
        // Release stage s; the last warp to release it loads frame t + NS.
        __syncwarp();
        if (lane == 0) {
            __threadfence_block();
            const int prev = atomicAdd(&cnt[s], 1);
            if (prev == NW - 1) {
                cnt[s] = 0;
                if (t + NS < p.T) {
                    const FrameHdr h = *reinterpret_cast<const FrameHdr *>(fblk);
                    fence_proxy_async();
                    issue(t + NS, s, h);
                }
            }
        }
        s = s1;
        par = par1;
    }
    if (bad) atomicExch(bad_flag, 1);
    __syncthreads();
    if (*bad_flag) {
        // Let any copy still in flight land before the CTA's shared memory goes away.
        if (threadIdx.x == 0) {
            for (int s = 0; s < NS; s++) {
                const int f = last_issued[s];
                if (f >= 0) dev::mbar_wait(smem_u32(&bars[s]), (uint32_t)((f / NS) & 1), 2, p.status);
            }
        }
        return false;
    }

    // Epilogue: every issued frame has been consumed, so the windows are free
    // for the tile of packed (SNR, k) keys.
    for (int i = threadIdx.x; i < TH * TW; i += blockDim.x) red[i] = 0ull;
    __syncthreads();
    const int64_t P = p.H * p.W;
#pragma unroll
    for (int r = 0; r < kMicroRows; r++)
#pragma unroll
        for (int c = 0; c < kMicroCols; c++) {
            const float n = acc[r][c] + blk[r][c];
            const int64_t py = sub_y0 + kMicroRows * ty + r;
            const int64_t px = sub_x0 + kMicroCols * tx + skew + c;
            if (kk >= 0 && py < p.H && px >= 0 && px < p.W) {
                const int64_t q = py * p.W + px;
                const float isd = p.isd[(int64_t)kk * P + q];
                const float snr = n * isd;
                if (p.snr_all) p.snr_all[(int64_t)kk * P + q] = isd > 0.f ? snr : 0.f;
                if (isd > 0.f)
                    atomicMax(&red[(kTile * sty + kMicroRows * ty + r) * TW + kTile * stx + kMicroCols * tx + c],
                              pack_key(snr, kk));
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < TH * TW; i += blockDim.x) {
        const unsigned long long key = red[i];
        if (key == 0ull) continue;
        const int ly = i / TW, lx = i % TW;
        const int64_t py = tile_y0 + ly;
        const int64_t px = tile_x0 + lx + lane_skew<VEC>((ly / kMicroRows) % 8);
        atomicMax(&p.keys[py * p.W + px], key);
    }
    // the barriers may be initialised again for this CTA's next tile
    if (threadIdx.x == 0)
        for (int s = 0; s < NS; s++) mbar_inval(smem_u32(&bars[s]));
    return true;
}

template <int KT, int TXS, int TYS, int VEC>
__global__ void __launch_bounds__(KT * TXS * TYS * 32, kWarps / (KT * TXS * TYS))
    k_numerator(const __grid_constant__ CUtensorMap ymap, const NumParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    numerator_tile<KT, TXS, TYS, VEC>(&ymap, p, (int)(blockIdx.x % (unsigned)p.G),
                                      (int)(blockIdx.x / (unsigned)p.G), smem);
}

// One item of a batched search: its numerator parameters, tile count and the
// first entry of its CTA work in the batch-wide work list.
struct BatchItem {
    NumParams p;
    int tiles_y;
    int pad;
    long long cta_begin;
};

// Persistent numerator over a batch of searches: one CTA per SM takes
// (item, tile, group) work entries from a global counter until the list is
// exhausted, running the same per-tile code as k_numerator.
template <int KT, int TXS, int TYS, int VEC>
__global__ void __launch_bounds__(kWarps * 32, 1) k_numerator_batch(const CUtensorMap *__restrict__ maps,
                                                                    const BatchItem *__restrict__ items, int n_items,
                                                                    long long total,
                                                                    unsigned long long *counter) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ long long work;
    __shared__ int item;
    for (;;) {
        if (threadIdx.x == 0) {
            const long long w = (long long)atomicAdd(counter, 1ull);
            int lo = 0, hi = n_items - 1;  // last item whose cta_begin <= w
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (items[mid].cta_begin <= w) lo = mid;
                else hi = mid - 1;
            }
            work = w;
            item = lo;
        }
        __syncthreads();
        const long long w = work;
        const int i = item;
        __syncthreads();
        if (w >= total) break;
        const NumParams &p = items[i].p;
        const long long local = w - items[i].cta_begin;
        if (!numerator_tile<KT, TXS, TYS, VEC>(maps + i, p, (int)(local % p.G), (int)(local / p.G), smem)) break;
        __syncthreads();
    }
}

// ----------------------------------------------------------- finalize ---

__global__ void k_finalize(const unsigned long long *__restrict__ keys, int64_t P, float *__restrict__ snr_max,
                           int32_t *__restrict__ argmax, const int *slot, int *global_status) {
    // a failure of this search also goes into the device-wide word
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int s = *(const volatile int *)slot;
        if (s != 0) atomicCAS(global_status, 0, s);
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long key = keys[i];
        if (key == 0ull) {
            snr_max[i] = 0.f;
            argmax[i] = -1;
        } else {
            uint32_t b = (uint32_t)(key >> 32);
            b = (b & 0x80000000u) ? (b & 0x7FFFFFFFu) : ~b;
            snr_max[i] = __uint_as_float(b);
            argmax[i] = (int32_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
        }
    }
}

// --------------------------------------------------------------- host ---

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

int get_encode(char *err, size_t errlen) {
    std::call_once(g_encode_once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    if (!g_encode) {
        snprintf(err, errlen, "cuTensorMapEncodeTiled is not available from the driver");
        return (int)cudaErrorNotSupported;
    }
    return 0;
}

int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 64) b = 152 * 64;
    if (b < 1) b = 1;
    return (int)b;
}


#define MF_CHECK_LAUNCH(what)                                                             \
    do {                                                                                  \
        cudaError_t e_ = cudaGetLastError();                                              \
        if (e_ != cudaSuccess) {                                                          \
            snprintf(err, errlen, "%s: %s", what, cudaGetErrorString(e_));                \
            return (int)e_;                                                               \
        }                                                                                 \
    } while (0)

// ---------------------------------------------------------- profiling ---

// k_select: k_sel_hist and k_sel_gather; k_compact: k_sel_refine; k_sort:
// k_sel_rank (names that callers of mf_profile_read know).
const char *kKernelNames[kKernelCount] = {"k_lambda",    "k_weight",      "k_denominator", "k_numerator",
                                          "k_finalize",  "k_select",      "k_rescore",     "k_compact",
                                          "k_sort",      "k_det_stats",   "k_det_cc",      "k_det_emit",
                                          "k_refit"};

struct ProfPending {
    int kid;
    cudaEvent_t a, b;
};

std::mutex g_prof_mu;
bool g_prof_on = false;
std::vector<ProfPending> g_pending;
double g_prof_ms[kKernelCount];
long long g_prof_count[kKernelCount];

// Bracket one launch: call with stage 0 before and stage 1 after it.
struct LaunchScope {
    int kid;
    cudaStream_t st;
    cudaEvent_t a = nullptr, b = nullptr;
    LaunchScope(int k, cudaStream_t s) : kid(k), st(s) {
        std::lock_guard<std::mutex> lk(g_prof_mu);
        g_prof_count[kid]++;
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) cs = cudaStreamCaptureStatusActive;
        if (g_prof_on && cs == cudaStreamCaptureStatusNone && cudaEventCreate(&a) == cudaSuccess &&
            cudaEventCreate(&b) == cudaSuccess)
            cudaEventRecord(a, st);
    }
    ~LaunchScope() {
        if (a && b) {
            cudaEventRecord(b, st);
            std::lock_guard<std::mutex> lk(g_prof_mu);
            g_pending.push_back({kid, a, b});
        }
    }
};

}  // namespace

ProfToken prof_begin(int kid, void *stream) {
    LaunchScope *ls = new LaunchScope(kid, (cudaStream_t)stream);
    return ProfToken{ls};
}

void prof_end(const ProfToken &t) { delete static_cast<LaunchScope *>(t.scope); }

int profile_enable(int on) {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    g_prof_on = on != 0;
    return 0;
}

int profile_read(mf_profile *out, int reset) {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    for (auto &p : g_pending) {
        float ms = 0.f;
        if (cudaEventSynchronize(p.b) == cudaSuccess && cudaEventElapsedTime(&ms, p.a, p.b) == cudaSuccess)
            g_prof_ms[p.kid] += ms;
        cudaEventDestroy(p.a);
        cudaEventDestroy(p.b);
    }
    g_pending.clear();
    std::memset(out, 0, sizeof *out);
    for (int i = 0; i < kKernelCount && i < 16; i++) {
        std::snprintf(out->k[i].name, sizeof out->k[i].name, "%s", kKernelNames[i]);
        out->k[i].launches = g_prof_count[i];
        out->k[i].ms = g_prof_ms[i];
        out->launches += g_prof_count[i];
    }
    out->n = kKernelCount;
    if (reset) {
        for (int i = 0; i < kKernelCount; i++) {
            g_prof_ms[i] = 0.0;
            g_prof_count[i] = 0;
        }
    }
    return 0;
}

namespace {

// Columns of a staged-denominator tile for images W wide: the widest of 256,
// 128, 64, 32 unless a narrower one wastes less.  A tile's cost is its start
// pixels (those past W too) times G_k's taps, plus the lambda values it stages
// (about 6 FMAs' worth each); the narrower the tile, the more of these per
// start pixel.  301 x 277, 54 trajectories, 231 taps each: 217 us with 256
// columns (512 of them for 277), 99 with 32 (the loop by chunk counts and the
// halved FP64 work included: 2048^2, 100 trajectories, 256 columns as before,
// 17.2 -> 16.1 ms).
int den_tile_cols(const mf_prf_table &tab, int64_t W) {
    const double taps = (double)tab.g_nnz / tab.K;
    int best = 256;
    double least = 0.0;
    for (int C = 256; C >= 32; C /= 2) {
        const double stage = (1.0 + (double)tab.den_cols / C) * (1.0 + (double)tab.den_rows / tab.den_th);
        const double cost = (double)((W + C - 1) / C * C) * (taps + 6.0 * stage);
        if (C == 256 || cost < least) {
            best = C;
            least = cost;
        }
    }
    return best;
}

// Inverse variance and weighted stack; `early`: the second as a programmatic
// dependent of the first (not in a batch, whose side streams fill the device
// already: its waiting CTAs would take the other searches' places).
int enqueue_pre(const SearchArgs &a, bool early, cudaStream_t stream, char *err, size_t errlen) {
    const mf_stack &st = *a.stack;
    const WorkspaceLayout &L = a.L;
    const int64_t T = st.T, H = st.H, W = st.W;
    float *lam = reinterpret_cast<float *>(a.ws + L.lam_off);
    void *y = a.ws + L.y_off;
    float *beta = reinterpret_cast<float *>(a.ws + L.beta_off);
    unsigned int *lmax = reinterpret_cast<unsigned int *>(a.ws + L.status_off + 8);
    // the search's status slot and the lambda maximum start clear (the
    // kernels after this in stream order write the slot only on a failure);
    // only fp16 weighted stacks need the maximum
    unsigned int *area = reinterpret_cast<unsigned int *>(a.ws + L.status_off);
    const bool need_max = st.dtype == MF_F16 && L.ybytes == 2;
    if (need_max) {
        const cudaError_t e0 = cudaMemsetAsync(area, 0, 16, stream);
        if (e0 != cudaSuccess) {
            snprintf(err, errlen, "cudaMemsetAsync: %s", cudaGetErrorString(e0));
            return (int)e0;
        }
    }
    {
        LaunchScope ls(kKLambda, stream);
        // rows and columns by grid dimension (no 64-bit division per pixel); a
        // few blocks per SM, since with the maximum every warp ends in an atomic
        // (2048^2: 78 us with 32 per SM, 88 with 16)
        const int64_t gx = (L.lam_w + 127) / 128, gy = std::max<int64_t>(1, std::min(L.lam_h, 152 * 32 / gx));
        const dim3 grid((unsigned)std::min<int64_t>(gx, 65535), (unsigned)gy);
        (need_max ? k_lambda<true> : k_lambda<false>)<<<grid, 128, 0, stream>>>(a.sigma, a.mask, H, W, L.pad, L.lam_w,
                                                                               L.lam_h, lam, area);
    }
    MF_CHECK_LAUNCH("k_lambda");

    const int64_t fs = st.frame_stride, rs = st.row_stride;
    cudaError_t we = cudaSuccess;
    {
        LaunchScope ls(kKWeight, stream);
        const int gw = grid_for(T * H * 32, 256);  // a warp per (frame, row)
        const bool y16 = L.ybytes == 2;
        const size_t esz = st.dtype == MF_F32 ? 4 : 2;
        // vector reads of the stack: aligned base, rows and frames on multiples of four elements
        const bool vr = ((uintptr_t)st.data % (4 * esz)) == 0 && fs % 4 == 0 && rs % 4 == 0;
        auto go = [&](auto tin, auto tout, auto vrc) {
            using TI = decltype(tin);
            using TO = decltype(tout);
            we = launch_after(early, k_weight<TI, TO, decltype(vrc)::value>, dim3(gw), dim3(256), 0, stream,
                              (const TI *)st.data, fs, rs, st.frame_scale, (const float *)lam, L.pad, L.lam_w, (TO *)y,
                              T, H, W, L.y_pitch, (const unsigned int *)lmax, beta);
        };
        auto go2 = [&](auto tin, auto tout) {
            if (vr) go(tin, tout, std::true_type{});
            else go(tin, tout, std::false_type{});
        };
        if (st.dtype == MF_F32) go2(float{}, float{});
        else if (st.dtype == MF_BF16 && y16) go2(__nv_bfloat16{}, __nv_bfloat16{});
        else if (st.dtype == MF_BF16) go2(__nv_bfloat16{}, float{});
        else if (y16) go2(__half{}, __half{});
        else go2(__half{}, float{});
    }
    if (we != cudaSuccess) {
        snprintf(err, errlen, "k_weight: %s", cudaGetErrorString(we));
        return (int)we;
    }
    return 0;
}

// The denominator; `early`: k_den_box as a programmatic dependent of the kernel
// before it, the numerator's last launch of a factored search, the weighting of
// a general one (whose keys hold final SNR).  It reads lambda, through the L1
// cache and without a wait: lambda's writer k_lambda, a launch in full order,
// has completed before k_weight lets anything start (its wait stands before its
// launch_dependents, and segment 0's of the numerator likewise), and no kernel
// since has put lambda into an L1 cache.  A kernel put between them, or a
// k_lambda started early, would have to keep that.  In a factored search the
// denominator so takes the SMs that the numerator's last CTAs leave (1 / sqrt(D)
// is needed only at the finalisation): with every kernel started early, 333
// frames of 301 x 277 pixels and 54 trajectories take 707 us instead of 783, 32
// frames of 128 x 128 and 16 trajectories 43.5 instead of 47.2.  (For the
// general numerator also a cleared key buffer.)
int enqueue_den(const SearchArgs &a, bool early, cudaStream_t stream, char *err, size_t errlen) {
    const mf_prf_table &tab = *a.tab;
    const WorkspaceLayout &L = a.L;
    const int64_t H = a.stack->H, W = a.stack->W, P = H * W;
    const float *lam = reinterpret_cast<const float *>(a.ws + L.lam_off);
    float *isd = reinterpret_cast<float *>(a.ws + L.isd_off);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(a.ws + L.keys_off);
    if (tab.den_th > 0) {
        // staged: one CTA per (tile of den_th x C start pixels, trajectory)
        const int th = tab.den_th, C = den_tile_cols(tab, W);
        const size_t smem = den_box_smem(th, tab.den_rows, tab.den_cols, tab.den_nw, tab.den_nr, C);
        const auto kern = C == 256   ? k_den_box<kDenOut, 256>
                          : C == 128 ? k_den_box<kDenOut, 128>
                          : C == 64  ? k_den_box<kDenOut, 64>
                                     : k_den_box<kDenOut, 32>;
        const int nbx = (int)((W + C - 1) / C);
        const int nby = (int)((H + th - 1) / th);
        dim3 grid((unsigned)(nbx * nby), (unsigned)std::min(tab.K, 65535));
        cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAllow);
        if (ea != cudaSuccess) {
            snprintf(err, errlen, "cudaFuncSetAttribute(k_den_box): %s", cudaGetErrorString(ea));
            return (int)ea;
        }
        LaunchScope ls(kKDenominator, stream);
        const dim3 block((unsigned)(th * C / kDenOut));
        const RunRec *runs = tab.d_runs;
        const int32_t *run_off = tab.d_run_off;
        const float *wts = tab.d_wts;
        const DenBox *boxes = tab.d_boxes;
        const cudaError_t el = launch_after(early, kern, grid, block, smem, stream, lam, L.lam_w, L.lam_h, L.pad, runs,
                                            run_off, wts, boxes, tab.K, H, W, nbx, th, isd);
        if (el != cudaSuccess) {
            snprintf(err, errlen, "k_den_box: %s", cudaGetErrorString(el));
            return (int)el;
        }
    } else {
        const int nbx = (int)((W + kDenCols - 1) / kDenCols);
        const int nby = (int)((H + 7) / 8);
        dim3 grid((unsigned)(nbx * nby), (unsigned)std::min(tab.K, 65535));
        LaunchScope ls(kKDenominator, stream);
        k_denominator<<<grid, 256, 0, stream>>>(lam, L.lam_w, L.pad, tab.d_runs, tab.d_run_off, tab.d_wts, tab.K, H,
                                                W, nbx, isd);
        MF_CHECK_LAUNCH("k_denominator");
    }
    // the general numerator merges its maxima into cleared keys; the factored
    // one has none
    const cudaError_t e = tab.plan.kernel == 2
                              ? cudaSuccess
                              : cudaMemsetAsync(keys, 0, (size_t)P * sizeof(unsigned long long), stream);
    if (e != cudaSuccess) {
        snprintf(err, errlen, "cudaMemsetAsync: %s", cudaGetErrorString(e));
        return (int)e;
    }
    return 0;
}

// Tile and staged window of the general numerator's CTAs.
struct NumGeometry {
    int tw, th, S, BH;
};

// The plan's, or (half) the same groups on tiles of half the sub-tiles: a window
// shrinks with its tile, which is a whole number of 32-column sub-tiles or of
// 32 rows smaller.
NumGeometry numerator_geometry(const Plan &pl, bool half) {
    NumGeometry g = {pl.tile_w(), pl.tile_h(), pl.S, pl.BH};
    if (half) {
        const int cut = kShapes[pl.shape].txs == kShapes[pl.shape].tys ? g.th / 2 : 0;  // 2 x 2: 2 x 1
        if (cut) {
            g.th -= cut;
            g.BH -= cut;
        } else {
            g.S -= g.tw / 2;
            g.tw /= 2;
        }
    }
    return g;
}

long long numerator_ctas(const Plan &pl, const NumGeometry &g, int64_t H, int64_t W) {
    return (long long)pl.G * ((W - kTileOriginX + g.tw - 1) / g.tw) * ((H + g.th - 1) / g.th);
}

// Two CTAs of 8 warps on an SM instead of one of 16: they wait for their frames
// apart and fill the last wave better, and every sum is the same.  60 frames x 24
// trajectories (groups of 8): 128^2 153 -> 92 us, 500 x 421 450 -> 384, 1024^2
// 1653 -> 1555, 2048^2 6258 -> 6025; 300 x 1000^2 x 4 (groups of 2) 2783 -> 1621.
// Not where all CTAs of 16 warps run at once and those of 8 would not, one to an
// SM: the same two halves on the fullest SM with more halo to load (256^2: 154
// and 156 us); nor where two windows do not fit on an SM.
bool numerator_halves(const Plan &pl, int64_t H, int64_t W) {
    if (kShapes[pl.shape].txs * kShapes[pl.shape].tys < 2) return false;
    const NumGeometry g = numerator_geometry(pl, true);
    if (numerator_smem_bytes(g.S, g.BH, pl.kt()) > (size_t)kSmemBudget / 2) return false;
    const long long full = numerator_ctas(pl, numerator_geometry(pl, false), H, W);
    return full > 152 || numerator_ctas(pl, g, H, W) <= 152;
}

// Tensor map over the weighted stack and the numerator's parameters.
int numerator_params(const SearchArgs &a, const NumGeometry &geo, CUtensorMap *map, NumParams *np, int *tiles_y,
                     char *err, size_t errlen) {
    const mf_stack &st = *a.stack;
    const mf_prf_table &tab = *a.tab;
    const Plan &pl = tab.plan;
    const WorkspaceLayout &L = a.L;
    const int64_t T = st.T, H = st.H, W = st.W;
    int rc = get_encode(err, errlen);
    if (rc) return rc;
    float *y = reinterpret_cast<float *>(a.ws + L.y_off);
    cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)T};
    cuuint64_t strides[2] = {(cuuint64_t)L.y_pitch * 4, (cuuint64_t)(H * L.y_pitch * 4)};
    cuuint32_t box[3] = {(cuuint32_t)geo.S, (cuuint32_t)geo.BH, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult cr = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, y, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) {
        snprintf(err, errlen, "cuTensorMapEncodeTiled failed (%d)", (int)cr);
        return (int)cudaErrorInvalidValue;
    }
    np->blocks = tab.d_blocks;
    np->hdr = tab.d_hdr;
    np->isd = reinterpret_cast<float *>(a.ws + L.isd_off);
    np->keys = reinterpret_cast<unsigned long long *>(a.ws + L.keys_off);
    np->snr_all = a.snr_all;
    np->status = reinterpret_cast<int *>(a.ws + L.status_off);
    np->T = (int)T;
    np->G = pl.G;
    np->H = H;
    np->W = W;
    np->tiles_x = (int)((W - kTileOriginX + geo.tw - 1) / geo.tw);
    np->S = geo.S;
    np->BH = geo.BH;
    np->lockstep = pl.lockstep;
    *tiles_y = (int)((H + geo.th - 1) / geo.th);
    return 0;
}

// Tensor map and parameters of the factored numerator with tiles of `th` rows
// (the plan's, or fewer).
int fac_params(const SearchArgs &a, int th, CUtensorMap *map, FacParams *fp, char *err, size_t errlen) {
    const mf_stack &st = *a.stack;
    const mf_prf_table &tab = *a.tab;
    const Plan &pl = tab.plan;
    const WorkspaceLayout &L = a.L;
    const int64_t T = st.T, H = st.H, W = st.W;
    int rc = get_encode(err, errlen);
    if (rc) return rc;
    int *status = reinterpret_cast<int *>(a.ws + L.status_off);
    void *y = a.ws + L.y_off;
    const bool y16 = L.ybytes == 2;
    cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)T};
    cuuint64_t strides[2] = {(cuuint64_t)L.y_pitch * L.ybytes, (cuuint64_t)(H * L.y_pitch * L.ybytes)};
    cuuint32_t box[3] = {(cuuint32_t)(y16 ? fac_rpitch16(pl.f_tw) : fac_rpitch(pl.f_tw)),
                         (cuuint32_t)(pl.f_bh - (pl.f_th - th)), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    const CUtensorMapDataType ty = !y16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                        : (st.dtype == MF_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                               : CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
    CUresult cr = g_encode(map, ty, 3, y, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS) {
        snprintf(err, errlen, "cuTensorMapEncodeTiled failed (%d)", (int)cr);
        return (int)cudaErrorInvalidValue;
    }
    fp->blocks = tab.d_blocks;
    fp->hdr = tab.d_hdr;
    fp->members = tab.d_members;
    fp->segs = tab.d_segs;
    fp->refs = tab.d_refs;
    fp->plane = reinterpret_cast<float *>(a.ws + L.planes_off);
    fp->status = status;
    // fp16 weighted stacks carry a power-of-two scale per frame; bf16 ones none
    fp->beta = (y16 && st.dtype == MF_F16) ? reinterpret_cast<const float *>(a.ws + L.beta_off) : nullptr;
    fp->T = (int)T;
    fp->G = pl.G;
    fp->kt = pl.f_kt;
    fp->npl = pl.f_planes;
    fp->th = th;
    fp->dth = pl.f_th - th;
    fp->bh = pl.f_bh - fp->dth;
    fp->ns = pl.f_ns;
    fp->S = pl.f_seg;
    fp->seg = 0;
    fp->K = tab.K;
    fp->warps = pl.warps_at(th);
    fp->H = H;
    fp->W = W;
    fp->tiles_x = (int)((W + pl.f_tw - 1) / pl.f_tw);
    return 0;
}

typedef void (*NumKernel)(const CUtensorMap, const NumParams);
typedef void (*NumBatchKernel)(const CUtensorMap *, const BatchItem *, int, long long, unsigned long long *);

NumKernel pick_numerator(int shape, int vec, bool half) {
#define MF_PICK(V)                                       \
    switch (shape + (half ? kNumShapes : 0)) {           \
        case kNumShapes + 1: return k_numerator<8, 1, 1, V>; \
        case kNumShapes + 2: return k_numerator<4, 2, 1, V>; \
        case kNumShapes + 3: return k_numerator<2, 2, 2, V>; \
        case 0: return k_numerator<16, 1, 1, V>;         \
        case 1: return k_numerator<8, 2, 1, V>;          \
        case 2: return k_numerator<4, 2, 2, V>;          \
        default: return k_numerator<2, 4, 2, V>;         \
    }
    if (vec == 4) {
        MF_PICK(4)
    } else if (vec == 2) {
        MF_PICK(2)
    } else {
        MF_PICK(1)
    }
#undef MF_PICK
}

NumBatchKernel pick_numerator_batch(int shape) {
    switch (shape) {
        case 0: return k_numerator_batch<16, 1, 1, 2>;
        case 1: return k_numerator_batch<8, 2, 1, 2>;
        case 2: return k_numerator_batch<4, 2, 2, 2>;
        default: return k_numerator_batch<2, 4, 2, 2>;
    }
}

int enqueue_finalize(const SearchArgs &a, bool early, cudaStream_t stream, char *err, size_t errlen) {
    const int64_t P = a.stack->H * a.stack->W;
    const int *slot = reinterpret_cast<const int *>(a.ws + a.L.status_off);
    int *gstatus = status_word(err, errlen);
    if (!gstatus) return (int)cudaErrorInvalidSymbol;
    if (a.tab->plan.kernel == 2) {
        LaunchScope ls(kKFinalize, stream);
        return fac_finalize_enqueue(reinterpret_cast<const float *>(a.ws + a.L.planes_off),
                                    reinterpret_cast<const float *>(a.ws + a.L.isd_off), a.tab->K, P, a.snr_max,
                                    a.argmax, a.snr_all, slot, gstatus, early, stream, err, errlen);
    }
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(a.ws + a.L.keys_off);
    {
        LaunchScope ls(kKFinalize, stream);
        k_finalize<<<grid_for(P, 256), 256, 0, stream>>>(keys, P, a.snr_max, a.argmax, slot, gstatus);
    }
    MF_CHECK_LAUNCH("k_finalize");
    return 0;
}

}  // namespace

int launch_search(const SearchArgs &a, char *err, size_t errlen) {
    cudaStream_t stream = (cudaStream_t)a.stream;
    const Plan &pl = a.tab->plan;
    int rc = enqueue_pre(a, true, stream, err, errlen);
    if (rc) return rc;
    const bool early_den = pl.kernel == 2 && a.tab->den_th > 0;
    if (!early_den && (rc = enqueue_den(a, true, stream, err, errlen))) return rc;
    CUtensorMap map;
    if (pl.kernel == 2) {
        FacParams fp;
        const int th = fac_tile_rows(*a.tab, a.stack->H, a.stack->W);
        rc = fac_params(a, th, &map, &fp, err, errlen);
        if (rc) return rc;
        // one launch per time segment, in order: segment 0 stores the
        // numerator plane, the later ones add to it
        for (int j = 0; j < pl.f_seg; j++) {
            fp.seg = j;
            LaunchScope ls(kKNumerator, stream);
            rc = fac_enqueue(&map, fp, pl.f_tw, pl.f_taps, a.L.ybytes == 2 ? a.stack->dtype : MF_F32,
                             (fp.warps + 3) / 4 * 4, pl.smem_at(th), fac_ctas(*a.tab, a.stack->H, a.stack->W, j, th),
                             stream, err, errlen);
            if (rc) return rc;
        }
        if (early_den && (rc = enqueue_den(a, true, stream, err, errlen))) return rc;
        return enqueue_finalize(a, true, stream, err, errlen);
    }
    NumParams np;
    int tiles_y = 0;
    const bool half = numerator_halves(pl, a.stack->H, a.stack->W);
    const NumGeometry geo = numerator_geometry(pl, half);
    rc = numerator_params(a, geo, &map, &np, &tiles_y, err, errlen);
    if (rc) return rc;
    {
        const size_t smem = numerator_smem_bytes(geo.S, geo.BH, pl.kt());
        NumKernel kern = pick_numerator(pl.shape, pl.vec, half);
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAllow);
        if (e != cudaSuccess) {
            snprintf(err, errlen, "cudaFuncSetAttribute(smem=%zu): %s", smem, cudaGetErrorString(e));
            return (int)e;
        }
        const long long nblocks = numerator_ctas(pl, geo, a.stack->H, a.stack->W);
        LaunchScope ls(kKNumerator, stream);
        kern<<<(unsigned)nblocks, (half ? kWarps / 2 : kWarps) * 32, smem, stream>>>(map, np);
        MF_CHECK_LAUNCH("k_numerator");
    }
    return enqueue_finalize(a, true, stream, err, errlen);
}

// ------------------------------------------------------------ batching ---
//
// A batch of searches (uneven cutouts, each with its own filter bank) runs as
// per-item preparation kernels spread over side streams, one persistent
// numerator launch per CTA shape in the batch (usually one), and per-item
// finalisation.  The descriptors the persistent kernel reads (tensor maps,
// parameters, work-list offsets) live in device memory owned by the batch.

struct BatchDevice {
    struct Group {
        int shape = 0;
        int first = 0, count = 0;  // range in the device arrays
        long long total = 0;       // CTA work entries
        size_t smem = 0;
    };
    std::vector<Group> groups;
    std::vector<int> order;  // device-array position -> item
    // searches with a factored numerator: one persistent launch per tile
    // width, with as many warps and as much shared memory as its largest
    // layout needs
    struct FacGroup {
        int chain = 0;             // (tile width, element type): chains are independent of each other
        int tw = 32;
        int etype = MF_F32;        // element type of the weighted stacks
        int seg = 0;               // time segment (groups run in segment order)
        int first = 0, count = 0;  // range in d_fmaps and h_fitems
        long long total = 0;       // CTA work entries
        size_t smem = 0;
        int warps = 0;
    };
    std::vector<FacGroup> fac;
    std::vector<int> item_chain;  // the chain of each search, -1: general numerator
    CUtensorMap *d_fmaps = nullptr;
    std::vector<FacBatchItem> h_fitems;  // passed by value to each launch
    unsigned long long *d_fcounters = nullptr;  // one per group
    CUtensorMap *d_maps = nullptr;
    BatchItem *d_items = nullptr;
    unsigned long long *d_counters = nullptr;
    static constexpr int kSide = 4;
    cudaStream_t side[kSide] = {};
    cudaEvent_t fork = nullptr, join[kSide] = {};
    int sms = 0;
};

void batch_free(BatchDevice *b) {
    if (!b) return;
    cudaFree(b->d_maps);
    cudaFree(b->d_items);
    cudaFree(b->d_counters);
    cudaFree(b->d_fmaps);
    cudaFree(b->d_fcounters);
    for (int i = 0; i < BatchDevice::kSide; i++) {
        if (b->side[i]) cudaStreamDestroy(b->side[i]);
        if (b->join[i]) cudaEventDestroy(b->join[i]);
    }
    if (b->fork) cudaEventDestroy(b->fork);
    delete b;
}

int batch_build(const SearchArgs *items, int n, BatchDevice **out, char *err, size_t errlen) {
    auto *b = new BatchDevice;
    std::vector<CUtensorMap> maps;
    std::vector<BatchItem> bitems;
    for (int shape = 0; shape < kNumShapes; shape++) {
        BatchDevice::Group grp;
        grp.shape = shape;
        grp.first = (int)bitems.size();
        for (int i = 0; i < n; i++) {
            const Plan &pl = items[i].tab->plan;
            if (pl.kernel != 1 || pl.shape != shape) continue;
            CUtensorMap m;
            BatchItem bi;
            std::memset(&bi, 0, sizeof bi);
            int rc = numerator_params(items[i], numerator_geometry(items[i].tab->plan, false), &m, &bi.p, &bi.tiles_y, err, errlen);
            if (rc) {
                batch_free(b);
                return rc;
            }
            bi.cta_begin = grp.total;
            grp.total += (long long)pl.G * bi.p.tiles_x * bi.tiles_y;
            grp.smem = std::max(grp.smem, numerator_smem_bytes(pl.S, pl.BH, pl.kt()));
            maps.push_back(m);
            bitems.push_back(bi);
            b->order.push_back(i);
        }
        grp.count = (int)bitems.size() - grp.first;
        if (grp.count > 0) b->groups.push_back(grp);
    }
    std::vector<CUtensorMap> fmaps;
    std::vector<FacBatchItem> fitems;
    int max_seg = 0;
    for (int i = 0; i < n; i++)
        if (items[i].tab->plan.kernel == 2) max_seg = std::max(max_seg, items[i].tab->plan.f_seg);
    // searches whose work entries take longest first, so that a launch ends on
    // short ones (an entry's time goes with its frames and its warps' rows)
    std::vector<int> by_time(n);
    for (int i = 0; i < n; i++) by_time[i] = i;
    auto entry = [&](int i) {
        const Plan &pl = items[i].tab->plan;
        return pl.kernel == 2 ? (double)items[i].stack->T / pl.f_seg * (pl.warps() + 8) : 0.0;
    };
    std::stable_sort(by_time.begin(), by_time.end(), [&](int x, int y) { return entry(x) > entry(y); });
    b->item_chain.assign(n, -1);
    // one persistent launch per (segment, tile width, element type of the
    // weighted stack)
    for (int j = 0; j < max_seg; j++) {
        for (int tw : {32, 64})
        for (int et : {(int)MF_F32, (int)MF_BF16, (int)MF_F16}) {
            BatchDevice::FacGroup grp;
            grp.chain = (tw == 64 ? 3 : 0) + et;
            grp.tw = tw;
            grp.etype = et;
            grp.seg = j;
            grp.first = (int)fitems.size();
            for (const int i : by_time) {
                const Plan &pl = items[i].tab->plan;
                const int item_et = items[i].L.ybytes == 2 ? items[i].stack->dtype : MF_F32;
                if (pl.kernel != 2 || pl.f_tw != tw || item_et != et || j >= pl.f_seg) continue;
                CUtensorMap m;
                FacBatchItem fi;
                std::memset(&fi, 0, sizeof fi);
                int rc = fac_params(items[i], pl.f_th, &m, &fi.p, err, errlen);
                if (rc) {
                    batch_free(b);
                    return rc;
                }
                b->item_chain[i] = grp.chain;
                fi.p.seg = j;
                fi.cta_begin = grp.total;
                grp.total += fac_ctas(*items[i].tab, items[i].stack->H, items[i].stack->W, j, pl.f_th);
                grp.smem = std::max(grp.smem, pl.smem());
                grp.warps = std::max(grp.warps, pl.launch_warps());
                fmaps.push_back(m);
                fitems.push_back(fi);
                if ((int)fitems.size() - grp.first == kFacBatchArgItems) {
                    // a launch takes at most kFacBatchArgItems searches: the
                    // rest of this segment goes to the next launch
                    grp.count = kFacBatchArgItems;
                    b->fac.push_back(grp);
                    grp.first = (int)fitems.size();
                    grp.total = 0;
                    grp.smem = 0;
                    grp.warps = 0;
                }
            }
            grp.count = (int)fitems.size() - grp.first;
            if (grp.count > 0) b->fac.push_back(grp);
        }
    }
    cudaError_t e = cudaSuccess;
    if (!fitems.empty()) e = cudaMalloc((void **)&b->d_fmaps, fmaps.size() * sizeof(CUtensorMap));
    if (e == cudaSuccess && !fitems.empty())
        e = cudaMalloc((void **)&b->d_fcounters, b->fac.size() * sizeof(unsigned long long));
    if (e == cudaSuccess && !fitems.empty())
        e = cudaMemcpy(b->d_fmaps, fmaps.data(), fmaps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
    b->h_fitems = fitems;
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && !maps.empty()) e = cudaMalloc((void **)&b->d_maps, maps.size() * sizeof(CUtensorMap));
    if (e == cudaSuccess && !bitems.empty()) e = cudaMalloc((void **)&b->d_items, bitems.size() * sizeof(BatchItem));
    if (e == cudaSuccess) e = cudaMalloc((void **)&b->d_counters, kNumShapes * sizeof(unsigned long long));
    if (e == cudaSuccess && !maps.empty())
        e = cudaMemcpy(b->d_maps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !bitems.empty())
        e = cudaMemcpy(b->d_items, bitems.data(), bitems.size() * sizeof(BatchItem), cudaMemcpyHostToDevice);
    for (int i = 0; i < BatchDevice::kSide && e == cudaSuccess; i++) {
        e = cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->join[i], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
    for (const auto &grp : b->groups) {
        if (e != cudaSuccess) break;
        e = cudaFuncSetAttribute(pick_numerator_batch(grp.shape), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemAllow);
    }
    if (e != cudaSuccess) {
        snprintf(err, errlen, "batch set-up: %s", cudaGetErrorString(e));
        batch_free(b);
        return (int)e;
    }
    for (const auto &grp : b->fac) {
        const int rc = fac_batch_attr(grp.tw, grp.etype, err, errlen);
        if (rc) {
            batch_free(b);
            return rc;
        }
    }
    *out = b;
    return 0;
}

int batch_enqueue(BatchDevice *b, const SearchArgs *items, int n, void *stream_v, char *err, size_t errlen) {
    cudaStream_t stream = (cudaStream_t)stream_v;
    cudaError_t e = cudaEventRecord(b->fork, stream);
    for (int s = 0; s < BatchDevice::kSide && e == cudaSuccess; s++) e = cudaStreamWaitEvent(b->side[s], b->fork, 0);
    if (e != cudaSuccess) {
        snprintf(err, errlen, "batch fork: %s", cudaGetErrorString(e));
        return (int)e;
    }
    for (int i = 0; i < n; i++) {
        int rc = enqueue_pre(items[i], false, b->side[i % BatchDevice::kSide], err, errlen);
        if (!rc) rc = enqueue_den(items[i], false, b->side[i % BatchDevice::kSide], err, errlen);
        if (rc) return rc;
    }
    for (int s = 0; s < BatchDevice::kSide && e == cudaSuccess; s++) {
        e = cudaEventRecord(b->join[s], b->side[s]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, b->join[s], 0);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(b->d_counters, 0, kNumShapes * sizeof(unsigned long long), stream);
    if (e != cudaSuccess) {
        snprintf(err, errlen, "batch join: %s", cudaGetErrorString(e));
        return (int)e;
    }
    if (!b->fac.empty()) {
        e = cudaMemsetAsync(b->d_fcounters, 0, b->fac.size() * sizeof(unsigned long long), stream);
        if (e != cudaSuccess) {
            snprintf(err, errlen, "batch counters: %s", cudaGetErrorString(e));
            return (int)e;
        }
    }
    // Factored searches: the launches of one tile width and element type follow
    // each other (segments in order, then the finalisation), those of different
    // ones run side by side, so that one chain's next CTAs take the SMs that the
    // last work entries of another leave.  General ones stay on `stream`.
    e = cudaEventRecord(b->fork, stream);
    for (int s = 0; s < BatchDevice::kSide && e == cudaSuccess; s++) e = cudaStreamWaitEvent(b->side[s], b->fork, 0);
    if (e != cudaSuccess) {
        snprintf(err, errlen, "batch fork: %s", cudaGetErrorString(e));
        return (int)e;
    }
    auto lane = [&](int chain) { return chain < 0 ? stream : b->side[chain % BatchDevice::kSide]; };
    for (const auto &grp : b->groups) {
        const int grid = (int)std::min<long long>(grp.total, (long long)b->sms);
        LaunchScope ls(kKNumerator, stream);
        pick_numerator_batch(grp.shape)<<<grid, kWarps * 32, grp.smem, stream>>>(
            b->d_maps + grp.first, b->d_items + grp.first, grp.count, grp.total, b->d_counters + grp.shape);
        MF_CHECK_LAUNCH("k_numerator_batch");
    }
    for (size_t gi = 0; gi < b->fac.size(); gi++) {
        const auto &grp = b->fac[gi];
        const int grid = (int)std::min<long long>(grp.total, (long long)b->sms);
        LaunchScope ls(kKNumerator, lane(grp.chain));
        int rc = fac_batch_enqueue(b->d_fmaps + grp.first, b->h_fitems.data() + grp.first, grp.count, grp.total,
                                   b->d_fcounters + gi, grp.tw, grp.etype, grp.warps, grp.smem, grid,
                                   lane(grp.chain), err, errlen);
        if (rc) return rc;
    }
    for (int i = 0; i < n; i++) {
        int rc = enqueue_finalize(items[i], false, lane(b->item_chain[i]), err, errlen);
        if (rc) return rc;
    }
    for (int s = 0; s < BatchDevice::kSide && e == cudaSuccess; s++) {
        e = cudaEventRecord(b->join[s], b->side[s]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, b->join[s], 0);
    }
    if (e != cudaSuccess) {
        snprintf(err, errlen, "batch join: %s", cudaGetErrorString(e));
        return (int)e;
    }
    return 0;
}

// ------------------------------------------------------------ rescore ---
//
// Candidate list (Section 3.3: scores above a threshold are candidates) and
// FP64 re-score: the k_top best start pixels (mf_select.cu), then N and D of
// each in FP64 from the master stack.

namespace {

// FP64 inverse variance of every pixel for the re-score: 1 / (s * s) from
// the FP32 noise value s in FP64, 0 where the pixel is masked or s is not a
// usable noise value (s <= 0 or not finite; a finite FP32 s never makes the
// FP64 quotient 0).  Computed once per re-score instead of per tap.
__global__ void k_lambda64(const float *__restrict__ sigma, const uint8_t *__restrict__ mask, int64_t P,
                           double *__restrict__ lam64) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
        const double s = (double)sigma[i];
        lam64[i] = ((mask && mask[i]) || !(s > 0.0) || !isfinite(s)) ? 0.0 : 1.0 / (s * s);
    }
}

// One candidate per `wpc` warps (1, 2, 4 or 8: a block holds whole
// candidates), each taking a share of the frames.
//
// N: lanes 0 .. 24 are the footprint's taps; per frame a warp reads the 25
// FP64 taps (200 consecutive bytes) and the five rows of five stack values,
// and adds w (s r) into a sum per tap; the sums meet lambda only when the
// trajectory's base pixel changes (a slow mover stays on a pixel for tens of
// frames), so a frame costs one FP64 FMA.  Of a trajectory that leaves the
// image, only the frames from the first to the last that reach it are walked
// (a check in the loop itself would put the shifts' latency before the taps':
// 1398 us instead of 621).
//
// D: lambda does not depend on the frame, so D is the collapsed kernel G_k
// (FP64, a few hundred taps) against lambda, half a warp per run of it, four
// runs' loads in flight, only the runs whose rows lie on the image.  TAPD: D
// from the taps, a second sum beside N's, for tables where a G_k has more
// steps of 16 columns than the 4 T that this costs at most (footprints that
// hardly overlap: 300 frames at 5 pixels per frame, 16384 candidates, 524 us
// against 584; shifts that jump, whose runs are mostly gaps).
//
// Bound: the FP64 pipe (one warp instruction per 64 cycles and scheduler) and
// the scattered reads.  4096 candidates of 1000 frames of 1024^2, whole call:
// lanes over frames (25 taps of four FP64 operations and a conversion each for
// N and D, 75 scattered reads per 32 frames) 2016 us, this form 621; 16384 of
// 512^2 at 3 pixels per frame, mostly off the image: 1620 and 1004 (every frame
// and run walked: 3361).  Four frames in flight and 32 warps per SM, so that
// 4096 candidates run at once; eight frames and 16 warps: a fifth slower.
template <typename TIn, bool TAPD>
__global__ void __launch_bounds__(256, 4) k_rescore(
    const TIn *__restrict__ r, int64_t fstride, int64_t rstride, const float *__restrict__ scale,
    const double *__restrict__ lam64, const double *__restrict__ taps64, const int2 *__restrict__ shifts,
    const RunRec *__restrict__ runs, const int32_t *__restrict__ run_off, const double *__restrict__ wts64,
    const DenBox *__restrict__ boxes, const float *__restrict__ snr_max, const int32_t *__restrict__ argmax,
    const unsigned long long *__restrict__ keys, const SelState *st, int wpc, int T, int64_t H, int64_t W,
    mf_candidate *__restrict__ out, int32_t *__restrict__ n_out) {
    constexpr int U = 4;  // frames whose loads are in flight together
    __shared__ double part_n[8], part_d[8];
    const unsigned int n = st->count;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned int cand = (blockIdx.x * 8u + warp) / (unsigned)wpc;
    const int part = warp % wpc;
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_out = (int32_t)n;
    const bool on = cand < n;
    double num = 0.0, den = 0.0;
    int64_t idx = 0;
    int k = 0;
    if (on) {
        idx = (int64_t)(0xFFFFFFFFu - (uint32_t)(keys[cand] & 0xFFFFFFFFull));
        k = argmax[idx];
        const int Hi = (int)H, Wi = (int)W;  // at most 2^20
        const int py = (int)(idx / W), px = (int)(idx % W);
        const int b = lane / 5 - 2, a = lane % 5 - 2;
        int t0 = (int)((int64_t)T * part / wpc), t1 = (int)((int64_t)T * (part + 1) / wpc);
        const size_t kt = (size_t)k * T;
        // rows and columns that G_k reaches; where the image does not hold them
        // all, only the frames from the first to the last that reach it count
        const DenBox box = boxes[k];
        const bool rows_in = py + box.dy0 >= 0 && py + box.dy0 + box.rows <= Hi;
        if (!rows_in || px + box.x0 < 0 || px + box.x0 + box.cols > Wi) {
            int first = t1, last = t0;
            for (int t = t0; t < t1; t += 128) {
                int2 s[4];
#pragma unroll
                for (int u = 0; u < 4; u++) s[u] = shifts[kt + min(t + 32 * u + lane, t1 - 1)];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const unsigned int m = __ballot_sync(0xffffffffu, t + 32 * u + lane < t1 &&
                                                                          (unsigned)(py + s[u].y + 2) < (unsigned)(Hi + 4) &&
                                                                          (unsigned)(px + s[u].x + 2) < (unsigned)(Wi + 4));
                    if (m) {
                        first = min(first, t + 32 * u + __ffs(m) - 1);
                        last = t + 32 * u + 32 - __clz(m);
                    }
                }
            }
            t0 = first;
            t1 = last;
        }
        int2 base = make_int2(INT_MIN, INT_MIN);
        double lam = 0.0, acc = 0.0, acc2 = 0.0;
        const TIn *src = r;
        bool use = false;
        for (int t = t0; t < t1; t += U) {
            int2 s[U];
            double w[U];
            float v[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int q = min(t + u, t1 - 1);
                s[u] = shifts[kt + q];
                w[u] = lane < 25 && t + u < t1 ? taps64[(kt + q) * 25 + lane] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int qy = py + s[u].y + b, qx = px + s[u].x + a;
                const bool in = lane < 25 && t + u < t1 && (unsigned)qy < (unsigned)Hi && (unsigned)qx < (unsigned)Wi;
                v[u] = in ? to_f32(src[(t + u) * fstride + qy * rstride + qx]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (s[u].x != base.x || s[u].y != base.y) {  // the same for the whole warp
                    num = fma(lam, acc, num);
                    acc = 0.0;
                    if constexpr (TAPD) {
                        den = fma(lam, acc2, den);
                        acc2 = 0.0;
                    }
                    base = s[u];
                    const int qy = py + base.y + b, qx = px + base.x + a;
                    const bool in = lane < 25 && (unsigned)qy < (unsigned)Hi && (unsigned)qx < (unsigned)Wi;
                    lam = in ? lam64[qy * W + qx] : 0.0;
                    // else off the image, masked, or no usable noise value:
                    // neither the stack's value nor the frame's scale matters
                    use = (__double2hiint(lam) | __double2loint(lam)) != 0;
                }
                const double x = widen(use ? v[u] : 0.f);
                if (scale) acc = fma(w[u], use ? (double)scale[min(t + u, t1 - 1)] * x : 0.0, acc);
                else acc = fma(w[u], x, acc);
                if constexpr (TAPD) acc2 = fma(w[u], w[u], acc2);
            }
        }
        num = fma(lam, acc, num);
        if constexpr (TAPD) den = fma(lam, acc2, den);
        // D: runs of G_k by half warps, the loads of four before their sums
        if constexpr (!TAPD) {
            constexpr int R = 4;
            int r0 = run_off[k], r1 = run_off[k + 1];
            if (!rows_in) {  // runs ascend in dy: the first and the end of those on the image
                for (int end = r1; r0 < end;) {
                    const int mid = (r0 + end) >> 1;
                    if (py + runs[mid].dy < 0) r0 = mid + 1;
                    else end = mid;
                }
                for (int from = r0; from < r1;) {
                    const int mid = (from + r1) >> 1;
                    if (py + runs[mid].dy < Hi) from = mid + 1;
                    else r1 = mid;
                }
            }
            const int half = lane & 15;
            for (int q = r0 + 2 * part + (lane >> 4); q < r1; q += 2 * wpc * R) {
                double g[R], l[R];
                unsigned int longer = 0;  // a bit per run of more than 16 columns
#pragma unroll
                for (int j = 0; j < R; j++) {
                    const int at = q + 2 * wpc * j;
                    const RunRec rr = runs[min(at, r1 - 1)];
                    const int y = py + rr.dy, x = px + rr.x0 + half;
                    const bool row = at < r1;
                    const bool in = row && half < 4 * rr.nch && (unsigned)x < (unsigned)Wi;
                    g[j] = in ? wts64[rr.woff + half] : 0.0;
                    l[j] = in ? lam64[y * W + x] : 0.0;
                    longer |= (unsigned int)(row && rr.nch > 4) << j;
                }
#pragma unroll
                for (int j = 0; j < R; j++) den = fma(g[j], l[j], den);
                for (int j = 0; longer; j++, longer >>= 1) {
                    if (!(longer & 1u)) continue;
                    const RunRec rr = runs[q + 2 * wpc * j];
                    for (int c = half + 16; c < 4 * rr.nch; c += 16) {
                        const int x = px + rr.x0 + c;
                        if ((unsigned)x < (unsigned)Wi) den = fma(wts64[rr.woff + c], lam64[(py + rr.dy) * W + x], den);
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            num += __shfl_xor_sync(0xffffffffu, num, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
    }
    if (wpc > 1) {
        if (lane == 0) {
            part_n[warp] = num;
            part_d[warp] = den;
        }
        __syncthreads();
        if (part != 0) return;
        for (int w = 1; w < wpc; w++) {
            num += part_n[warp + w];
            den += part_d[warp + w];
        }
    }
    if (on && lane == 0) {
        mf_candidate c;
        c.y = (int32_t)(idx / W);
        c.x = (int32_t)(idx % W);
        c.k = k;
        c.reserved = 0;
        c.snr = den > 0.0 ? num / sqrt(den) : 0.0;
        c.flux = den > 0.0 ? num / den : 0.0;
        c.snr_search = snr_max[idx];
        c.reserved2 = 0.f;
        out[cand] = c;
    }
}

}  // namespace

size_t rescore_workspace(int64_t H, int64_t W, int32_t k_top) { return select_layout(H * W, k_top).total; }

int launch_rescore(const RescoreArgs &a, char *err, size_t errlen) {
    const mf_stack &st = *a.stack;
    const mf_prf_table &tab = *a.tab;
    cudaStream_t stream = (cudaStream_t)a.stream;
    const int64_t H = st.H, W = st.W, P = H * W;
    const SelectLayout L = select_layout(P, a.k_top);
    SelState *sst = reinterpret_cast<SelState *>(a.ws + L.st_off);
    unsigned long long *top = reinterpret_cast<unsigned long long *>(a.ws + L.top_off);
    int rc = launch_select(a.snr_max, a.argmax, P, a.k_top, a.ws, L, stream, err, errlen);
    if (rc) return rc;
    // the selection is done with the per-pixel keys: their space holds the
    // FP64 inverse variance (P doubles) the re-score reads (both launches
    // count as the re-score)
    static_assert(sizeof(double) == sizeof(unsigned long long), "one double per key");
    double *lam64 = reinterpret_cast<double *>(a.ws + L.keys_off);
    {
        LaunchScope ls(kKRescore, stream);
        k_lambda64<<<grid_for(P, 256), 256, 0, stream>>>(a.sigma, a.mask, P, lam64);
    }
    MF_CHECK_LAUNCH("k_lambda64");
    {
        // enough warps to fill the chip (24 per SM) when candidates are few
        int wpc = 1;
        while (wpc < 8 && (int64_t)a.k_top * wpc < 152 * 24) wpc *= 2;
        const unsigned blocks = (unsigned)(((int64_t)a.k_top * wpc + 7) / 8);
        LaunchScope ls(kKRescore, stream);
        auto go = [&](auto t) {
            using TI = decltype(t);
            const auto kern = tab.den_steps > 4LL * tab.T ? k_rescore<TI, true> : k_rescore<TI, false>;
            kern<<<blocks, 256, 0, stream>>>(
                (const TI *)st.data, st.frame_stride, st.row_stride, st.frame_scale, lam64, tab.d_taps64,
                reinterpret_cast<const int2 *>(tab.d_shifts), tab.d_runs, tab.d_run_off, tab.d_wts64, tab.d_boxes,
                a.snr_max,
                a.argmax, top, sst, wpc, tab.T, H, W, a.out, a.n_out);
        };
        if (st.dtype == MF_F32) go(float{});
        else if (st.dtype == MF_BF16) go(__nv_bfloat16{});
        else go(__half{});
    }
    MF_CHECK_LAUNCH("k_rescore");
    return 0;
}

namespace {

// One CTA whose thread 0 waits on an mbarrier that nothing arrives at, with
// the same bounded wait as every kernel of the library: the wait gives up,
// records `code` in the status word (and in a search's status slot, if one is
// given) and returns, and the CTA exits.  It exercises the failure path of
// the search kernels on purpose; nothing faults, traps or hangs.
__global__ void k_wait_probe(int code, int *slot) {
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait(smem_u32(&bar), 0u, code) && slot) atomicCAS(slot, 0, code);
    __syncthreads();
    if (threadIdx.x == 0) mbar_inval(smem_u32(&bar));
}

}  // namespace

int launch_wait_probe(void *stream, int *slot, char *err, size_t errlen) {
    k_wait_probe<<<1, 32, 0, (cudaStream_t)stream>>>(kWaitProbeCode, slot);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        snprintf(err, errlen, "k_wait_probe: %s", cudaGetErrorString(e));
        return (int)e;
    }
    return 0;
}

int *status_word(char *err, size_t errlen) {
    static std::mutex mu;
    static std::vector<int *> addr;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        snprintf(err, errlen, "cudaGetDevice: %s", cudaGetErrorString(e));
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(mu);
    if ((int)addr.size() <= dev) addr.resize(dev + 1, nullptr);
    if (!addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_status);
        if (e != cudaSuccess) {
            snprintf(err, errlen, "cudaGetSymbolAddress(status word): %s", cudaGetErrorString(e));
            return nullptr;
        }
        addr[dev] = static_cast<int *>(p);
    }
    return addr[dev];
}

int read_device_status(int *status) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return (int)e;
    int v = 0, zero = 0;
    e = cudaMemcpyFromSymbol(&v, g_status, sizeof(int));
    if (e != cudaSuccess) return (int)e;
    e = cudaMemcpyToSymbol(g_status, &zero, sizeof(int));
    if (e != cudaSuccess) return (int)e;
    *status = v;
    return 0;
}

}  // namespace mf
