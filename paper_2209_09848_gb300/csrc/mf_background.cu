// Per-pixel background re-fit (Section 3.1 of Ganapathi 2022): with the
// low-resolution scattered light fixed, every pixel's time series is
// regressed on the same six jitter basis values under the Huber loss,
// reached by least-squares steps on clipped residuals.
//
// The host turns the basis Phi [T][6] into an orthonormal one, Q = Phi R^-1
// (G = Phi^T Phi = R^T R, FP64 Cholesky), so the shared Gram inverse becomes
// the identity and each step is beta_Q <- beta_Q + Q^T psi(y - Q beta_Q):
// the same iterates as beta <- beta + G^-1 Phi^T psi(y - Phi beta) with
// beta = R^-1 beta_Q, but with well-scaled FP32 arithmetic.
//
// k_refit_resident (up to kRefitMaxResident frames): a CTA keeps the whole
// series of its pixels in shared memory, so HBM sees each frame value once in and
// each residual once out (8 bytes per pixel and frame instead of (iterations
// + 4) x 4).  k_refit (longer series): one thread per pixel re-reads its
// series from memory on every pass.

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>

#include "mf_device.cuh"
#include "mf_internal.h"

namespace mf {
namespace {

constexpr int kRefitThreads = 256;
constexpr int kRefitChunk = 256;  // frames of Q staged in shared memory
constexpr int kRefitBlock = 32;   // frames per FP32 partial sum
constexpr int kRefitUnroll = 8;   // frames whose loads are in flight together

using dev::widen;

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// The resident form.  A CTA of NW warps keeps the series of 4 QUADS pixels and
// the basis in shared memory; thread = (four pixels, frame group), group g of
// the G = 32 NW / QUADS owning frames g, g + G, g + 2 G ..: only that thread
// touches its values, so the passes over the frames need no barrier.
//
// Values are held as v_t = y_t - y0, y0 the median of three frames, or 0 where
// that is within 2 delta of 0 (the constant is in the basis' span, so the fit of
// v has the residuals of the fit of y, and y0 returns in the constant
// coefficient): all FP32 arithmetic sees noise-sized numbers.  One frame alone
// would not do: an outlier there would be every value's size.  Largest error of
// the other frames' residuals against FP64, in sigma (y itself held, y0 = y_0,
// and as it is): T = 600 on a background of 100 sigma 2.8e-5, 9.2e-7, 4.7e-7,
// on none 3.9e-7, 9.0e-7, 4.2e-7; T = 1500 on none, 300 sigma off in frame 0,
// 2.4e-7, 3.3e-5, 8.0e-7.  A
// clipped step is, per frame, e = v - Q beta, the clip and the sums Q^T psi(e):
// 12 FMAs per pixel, packed over pairs of frames (the basis pairs are read as
// they lie; beta stands twice in registers), two frames by four pixels at a
// time: 48 packed FMAs to five 128-bit reads of shared memory.  A basis read
// fills 32 lanes' registers whatever its addresses, which is why a thread has
// four pixels: with one, those reads set the pace.  Partial sums: even and odd
// frames of a thread, groups of a warp (halving exchanges), warps in order --
// all fixed, so reruns are bit-identical.  Frames past T have zero basis rows
// and values.
//
// Bound: the FP32 pipe.  The loop over the frames alone (residual, clip, sums)
// measures 38 SM cycles per warp and pair of frames -- packed or scalar FMAs
// with three register operands run at three quarters of the pipe's rate here,
// and the clip's min / max are half rate -- and the whole step 50, the rest
// being the exchanges, the barrier and three warps a scheduler to cover them.
// 1000 x 2048^2, 10 steps: 63.7 -> 41.8 ms; 203 x 317 x 411: 488 -> 289 us.
// Rows of 16 pixels (two whole sectors) because 32-pixel rows leave one CTA an
// SM and 8-pixel rows double the requests (the load alone: 3.3 against 6.5 ms
// at 1000 x 1024^2).  Values in registers (24 frames a thread, T = 1000): 38.9
// ms, but 405 us on the cutout; 24 warps with one frame at a time: 40.5 ms,
// 317 us.
constexpr int kResWarps = 12;  // resident warps per SM (168 registers a thread)

// One exchange of a halving sum: of 2 N values a lane keeps N (the upper ones
// if its bit m is set), each with the partner lane's added, in x[0 .. N - 1];
// returns where they stood.
template <int N>
__device__ __forceinline__ int halve(float (&x)[24], int lane, int m) {
    const bool up = (lane & m) != 0;
#pragma unroll
    for (int i = 0; i < N; i++) {
        const float give = up ? x[i] : x[i + N], keep = up ? x[i + N] : x[i];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
    return up ? N : 0;
}

// Pixel coordinate i of an axis of `size` pixels on the n-point scattered-light
// grid (pixel centres aligned, clamped at the edge).
__device__ __forceinline__ float grid_coord(int i, int n, int size) {
    return fminf(fmaxf(((float)i + 0.5f) * (float)n / (float)size - 0.5f, 0.f), (float)(n - 1));
}

__device__ __forceinline__ void cp_async16(float4 *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool live) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(live ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int NW, int QUADS, bool VEC>
__global__ void __launch_bounds__(32 * NW, kResWarps / NW) k_refit_resident(
    const float *data, int T, int H, int W, const float *__restrict__ scatter, int n, const float *__restrict__ Q,
    const double *__restrict__ Rinv, int iterations, float delta, int np, float *resid, float *__restrict__ coef) {
    constexpr int NT = 32 * NW, PX = 4 * QUADS, G = NT / QUADS;
    constexpr int NX = QUADS == 16 ? 12 : QUADS == 8 ? 6 : 3;  // sums a lane keeps of its quad's 24
    static_assert(QUADS == 2 || QUADS == 4 || QUADS == 8 || QUADS == 16, "the exchanges below");
    // [2 np][NT]: a thread's frame f at [f][tid] as loaded (four pixels); after
    // the first pass its pair i holds pixels 0, 1 of frames 2 i, 2 i + 1 at
    // [2 i] and pixels 2, 3 at [2 i + 1], each pixel's two values together
    extern __shared__ float4 vs[];
    float4 *qs = vs + (size_t)2 * np * NT;  // [np][G][3]: (q_k, q_k) of the pair's two frames, k = 0 .. 5
    __shared__ float red[2][NW][QUADS][24];
    __shared__ double rsh[36];            // R^-1
    __shared__ float4 bsh[NW][QUADS][6];  // -beta of the quad's four pixels per basis vector (a copy per warp)
    const int64_t P = (int64_t)H * W;
    const int tid = threadIdx.x, quad = tid % QUADS, grp = tid / QUADS, warp = tid >> 5, lane = tid & 31;
    const int cnt = grp < T ? (T - grp + G - 1) / G : 0;  // frames of this thread
    for (int j = tid; j < 2 * np * G; j += NT) {
        const int f = j / G, g = j - f * G, t = g + G * f;
        float *dst = reinterpret_cast<float *>(qs + ((size_t)(f >> 1) * G + g) * 3) + (f & 1);
#pragma unroll
        for (int k = 0; k < 6; k++) dst[2 * k] = t < T ? Q[(size_t)t * kRefitBasisPitch + k] : 0.f;
    }
    for (int j = tid; j < 36; j += NT) rsh[j] = Rinv[j];
    __syncthreads();
    const int64_t nblk = (P + PX - 1) / PX;
    const size_t nn = (size_t)n * n;
    const float near = isfinite(delta) ? 2.f * delta : 0.f;  // an origin of the noise's size gains nothing
    const int og = (lane / QUADS) % 3;  // this lane's frame of the origin
    // pixel j of this thread: four consecutive ones for 128-bit accesses, else
    // QUADS apart (each access of a warp covers consecutive pixels)
    const int first = VEC ? 4 * quad : quad;
    constexpr int STEP = VEC ? 1 : QUADS;
    float4 *vt = vs + tid;
    const float4 *qt = qs + 3 * grp;
    // The buffer of the next exchange between the warps.  It alternates through
    // the pixel blocks too (the step's parity would start each block with the
    // buffer that the last step of an even number of them has just used): a
    // warp writes a buffer again only past the barrier of the exchange in
    // between, which every warp reaches after its reads of this one.
    int buf = 0;
    for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        const int64_t p = blk * PX + first;
        const bool live[4] = {p < P, p + STEP < P, p + 2 * STEP < P, p + 3 * STEP < P};
        {
            const float *src = data + (size_t)grp * P + p;
            for (int f = 0; f < 2 * np; f++, src += (size_t)G * P) {
                if (f < cnt && live[0]) {
                    if constexpr (VEC) {
                        cp_async16(vt + NT * f, src);  // P is a multiple of 4: all or none live
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            cp_async4(reinterpret_cast<float *>(vt + NT * f) + j, live[j] ? src + j * STEP : src, live[j]);
                    }
                }
            }
        }
        // the values' origin: the median of three frames, one in each group of a
        // warp (behind the series: in front of it 20.90 -> 21.05 ms at 1000 x
        // 1024 x 2048)
        constexpr int NO = QUADS == 16 ? 3 : 1;  // frames a lane loads (a warp of two groups has none for the third)
        const int of[3] = {NO == 3 || og == 0 ? 0 : og == 1 ? T / 2 : T - 1, T / 2, T - 1};
        float o[NO][4];
#pragma unroll
        for (int i = 0; i < NO; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) o[i][j] = data[(size_t)of[i] * P + (live[j] ? p + j * STEP : 0)];
        // the pixels' places on the scattered-light grid; pixels of one cell
        // share its corners
        float fy[4], fx[4];
        int o00[4], di[4], dj[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t pj = live[j] ? p + j * STEP : 0;
            const int r = (int)(pj / W), c = (int)(pj - (int64_t)r * W);
            const float u = grid_coord(r, n, H), w = grid_coord(c, n, W);
            const int i0 = (int)floorf(u), j0 = (int)floorf(w);
            fy[j] = u - (float)i0;
            fx[j] = w - (float)j0;
            o00[j] = i0 * n + j0;
            di[j] = i0 + 1 < n ? n : 0;
            dj[j] = j0 + 1 < n ? 1 : 0;
        }
        const bool one = o00[0] == o00[1] && o00[0] == o00[2] && o00[0] == o00[3];
        auto light = [&](const float *S, float *o) {
            float a = S[o00[0]], b = S[o00[0] + dj[0]] - a, c = S[o00[0] + di[0]], d = S[o00[0] + di[0] + dj[0]] - c;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (j > 0 && !one) {
                    const float *s = S + o00[j];
                    a = s[0];
                    b = s[dj[j]] - a;
                    c = s[di[j]];
                    d = s[di[j] + dj[j]] - c;
                }
                const float top = fmaf(fx[j], b, a), bot = fmaf(fx[j], d, c);
                o[j] -= fmaf(fy[j], bot - top, top);
            }
        };
        if (scatter)
#pragma unroll
            for (int i = 0; i < NO; i++) light(scatter + (size_t)of[i] * nn, o[i]);
        float y0[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float u, v, w;
            if constexpr (NO == 3) {
                u = o[0][j];
                v = o[1][j];
                w = o[2][j];
            } else {
                u = __shfl_sync(0xffffffffu, o[0][j], quad);
                v = __shfl_sync(0xffffffffu, o[0][j], quad + QUADS);
                w = __shfl_sync(0xffffffffu, o[0][j], quad + 2 * QUADS);
            }
            y0[j] = fmaxf(fminf(u, v), fminf(fmaxf(u, v), w));
            if (fabsf(y0[j]) <= near) y0[j] = 0.f;
        }
        cp_async_wait();
        float2 s[6][4], nb[6][4];  // sums (even, odd frames) and -beta (twice) of the four pixels
        auto sums = [&](const float2 (&q)[6], const float2 (&e)[4]) {
#pragma unroll
            for (int k = 0; k < 6; k++)
#pragma unroll
                for (int j = 0; j < 4; j++) s[k][j] = __ffma2_rn(q[k], e[j], s[k][j]);
        };
        auto basis = [&](int i, float2 (&q)[6]) {
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float4 a = qt[(size_t)i * G * 3 + c];
                q[2 * c] = make_float2(a.x, a.y);
                q[2 * c + 1] = make_float2(a.z, a.w);
            }
        };
        auto values = [&](int i, float2 (&e)[4]) {
            const float4 a = vt[NT * 2 * i], b = vt[NT * (2 * i + 1)];
            e[0] = make_float2(a.x, a.y);
            e[1] = make_float2(a.z, a.w);
            e[2] = make_float2(b.x, b.y);
            e[3] = make_float2(b.z, b.w);
        };
        // e = v - Q beta of pair i
        auto residual = [&](int i, const float2 (&q)[6], float2 (&e)[4]) {
            values(i, e);
#pragma unroll
            for (int k = 0; k < 6; k++)
#pragma unroll
                for (int j = 0; j < 4; j++) e[j] = __ffma2_rn(q[k], nb[k][j], e[j]);
        };
        auto clear = [&]() {
#pragma unroll
            for (int k = 0; k < 6; k++)
#pragma unroll
                for (int j = 0; j < 4; j++) s[k][j] = make_float2(0.f, 0.f);
        };
        // least squares: beta = Q^T v, with v formed on the way
        clear();
        for (int i = 0; i < np; i++) {
            float v[2][4];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int f = 2 * i + h;
                const bool on = f < cnt && live[0];
                const float4 d = vt[NT * f];
                v[h][0] = d.x; v[h][1] = d.y; v[h][2] = d.z; v[h][3] = d.w;
                if (scatter && on) light(scatter + (size_t)(grp + G * f) * nn, v[h]);
#pragma unroll
                for (int j = 0; j < 4; j++) v[h][j] = on ? v[h][j] - y0[j] : 0.f;
            }
            vt[NT * 2 * i] = make_float4(v[0][0], v[1][0], v[0][1], v[1][1]);
            vt[NT * (2 * i + 1)] = make_float4(v[0][2], v[1][2], v[0][3], v[1][3]);
            float2 q[6];
            basis(i, q);
            const float2 e[4] = {{v[0][0], v[1][0]}, {v[0][1], v[1][1]}, {v[0][2], v[1][2]}, {v[0][3], v[1][3]}};
            sums(q, e);
        }
        float own[NX];  // -beta of the values this lane sums
#pragma unroll
        for (int i = 0; i < NX; i++) own[i] = 0.f;
        for (int step = 0;; step++) {
            float x[24];
#pragma unroll
            for (int k = 0; k < 6; k++)
#pragma unroll
                for (int j = 0; j < 4; j++) x[4 * k + j] = s[k][j].x + s[k][j].y;
            // sums over the warp's groups: each exchange halves the values a
            // lane keeps, the last one plain; a lane ends with NX of its
            // quad's 24
            int pos = halve<12>(x, lane, 16);
            if constexpr (QUADS <= 8) pos += halve<6>(x, lane, 8);
            if constexpr (QUADS <= 4) pos += halve<3>(x, lane, 4);
            if constexpr (QUADS == 2) {
#pragma unroll
                for (int i = 0; i < NX; i++) x[i] += __shfl_xor_sync(0xffffffffu, x[i], 2);
            }
            if constexpr (NW > 1) {  // and over the warps, in order, by every warp for itself
                float *mine = &red[buf][warp][quad][pos];
                if (QUADS != 2 || (lane & 2) == 0) {
#pragma unroll
                    for (int i = 0; i < NX; i++) mine[i] = x[i];
                }
                __syncthreads();
#pragma unroll
                for (int i = 0; i < NX; i++) x[i] = red[buf][0][quad][pos + i];
#pragma unroll
                for (int r = 1; r < NW; r++)
#pragma unroll
                    for (int i = 0; i < NX; i++) x[i] += red[buf][r][quad][pos + i];
                buf ^= 1;
            }
            float *mine = reinterpret_cast<float *>(&bsh[warp][quad][0]) + pos;
            __syncwarp();  // every lane has read the previous beta
#pragma unroll
            for (int i = 0; i < NX; i++) {
                own[i] -= x[i];
                mine[i] = own[i];
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 6; k++) {
                const float4 b = bsh[warp][quad][k];
                nb[k][0] = make_float2(b.x, b.x);
                nb[k][1] = make_float2(b.y, b.y);
                nb[k][2] = make_float2(b.z, b.z);
                nb[k][3] = make_float2(b.w, b.w);
            }
            if (step == iterations) break;
            clear();
#pragma unroll 2
            for (int i = 0; i < np; i++) {
                float2 q[6], e[4];
                basis(i, q);
                residual(i, q, e);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    e[j].x = fminf(fmaxf(e[j].x, -delta), delta);
                    e[j].y = fminf(fmaxf(e[j].y, -delta), delta);
                }
                sums(q, e);
            }
        }
        if (live[0]) {
            float *dst = resid + (size_t)grp * P + p;
            for (int i = 0; i < np; i++) {
                // the fit by itself first: its terms are smaller than the
                // values, and so is what their sum's roundings leave
                float2 q[6], e[4], m[4];
                basis(i, q);
                values(i, e);
#pragma unroll
                for (int j = 0; j < 4; j++) m[j] = __fmul2_rn(q[0], nb[0][j]);
#pragma unroll
                for (int k = 1; k < 6; k++)
#pragma unroll
                    for (int j = 0; j < 4; j++) m[j] = __ffma2_rn(q[k], nb[k][j], m[j]);
#pragma unroll
                for (int j = 0; j < 4; j++) e[j] = __fadd2_rn(e[j], m[j]);
#pragma unroll
                for (int h = 0; h < 2; h++, dst += (size_t)G * P) {
                    if (2 * i + h >= cnt) break;
                    float o[4];
#pragma unroll
                    for (int j = 0; j < 4; j++) o[j] = h ? e[j].y : e[j].x;
                    if constexpr (VEC) {
                        *reinterpret_cast<float4 *>(dst) = make_float4(o[0], o[1], o[2], o[3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            if (live[j]) dst[j * STEP] = o[j];
                    }
                }
            }
        }
        // coefficients in the basis (1, x, y, x^2, y^2, x y): R^-1 beta (R^-1
        // upper triangular), plus y0 in the constant.  A pixel's rows i and 5 - i
        // of R^-1 are one task, 12 a quad, dealt to the groups; FP32 values widened
        // by bits: FP64 operations set the pace of short series (1024^2, 6 frames,
        // no steps, 16 pixels a warp: six groups with a row of four pixels each
        // 282 us, the tasks 182)
        if (coef) {
            for (int task = grp; task < 12; task += G) {
                const int i = task % 3, j = task / 3;
                const int64_t pj = p + j * STEP;
                if (pj >= P) continue;
                const float *b = reinterpret_cast<const float *>(&bsh[warp][quad][0]) + j;  // -beta_k at b[4 k]
                const float origin = j == 0 ? y0[0] : j == 1 ? y0[1] : j == 2 ? y0[2] : y0[3];
                double lo = i == 0 ? widen(origin) : 0.0, hi = 0.0;
#pragma unroll
                for (int k = 0; k < 6; k++) {
                    const double v = widen(b[4 * k]);
                    if (k > 1 || k >= i) lo -= rsh[i * 6 + k] * v;
                    if (k > 4 || (k > 2 && k >= 5 - i)) hi -= rsh[(5 - i) * 6 + k] * v;
                }
                coef[(size_t)pj * 6 + i] = (float)lo;
                coef[(size_t)pj * 6 + 5 - i] = (float)hi;
            }
        }
    }
}

__global__ void __launch_bounds__(kRefitThreads) k_refit(const float *data, int T, int H, int W,
                                                         const float *__restrict__ scatter, int n,
                                                         const float4 *__restrict__ Q,
                                                         const double *__restrict__ Rinv,
                                                         const double *__restrict__ q1, int iterations, float delta,
                                                         float *resid, float *__restrict__ coef) {
    __shared__ float4 qs[kRefitChunk * 2];
    const int64_t P = (int64_t)H * W;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = p < P;
    // bilinear weights of this pixel on the scattered-light grid
    int o00 = 0, o01 = 0, o10 = 0, o11 = 0;
    float fy = 0.f, fx = 0.f;
    if (scatter && live) {
        const int i = (int)(p / W), j = (int)(p % W);
        const float u = fminf(fmaxf(((float)i + 0.5f) * (float)n / (float)H - 0.5f, 0.f), (float)(n - 1));
        const float v = fminf(fmaxf(((float)j + 0.5f) * (float)n / (float)W - 0.5f, 0.f), (float)(n - 1));
        const int i0 = (int)floorf(u), j0 = (int)floorf(v);
        const int i1 = min(i0 + 1, n - 1), j1 = min(j0 + 1, n - 1);
        fy = u - (float)i0;
        fx = v - (float)j0;
        o00 = i0 * n + j0;
        o01 = i0 * n + j1;
        o10 = i1 * n + j0;
        o11 = i1 * n + j1;
    }
    float beta[6], acc[6], part[6];
#pragma unroll
    for (int k = 0; k < 6; k++) beta[k] = 0.f;
    float y0 = 0.f;
    // pass 0: least-squares start; passes 1 .. iterations: clipped steps;
    // pass iterations + 1: residuals
    for (int pass = 0; pass <= iterations + 1; pass++) {
        const bool last = pass == iterations + 1;
#pragma unroll
        for (int k = 0; k < 6; k++) {
            acc[k] = 0.f;
            part[k] = 0.f;
        }
        for (int c0 = 0; c0 < T; c0 += kRefitChunk) {
            const int cn = min(kRefitChunk, T - c0);
            __syncthreads();
            for (int q = threadIdx.x; q < 2 * cn; q += blockDim.x) qs[q] = Q[(size_t)c0 * 2 + q];
            __syncthreads();
            if (!live) continue;
            // eight frames at a time: their loads are issued before any use
            for (int tt0 = 0; tt0 < cn; tt0 += kRefitUnroll) {
                float v[kRefitUnroll];
                const float *src = pass == 0 ? data : resid;
#pragma unroll
                for (int u = 0; u < kRefitUnroll; u++)
                    v[u] = tt0 + u < cn ? src[(size_t)(c0 + tt0 + u) * P + p] : 0.f;
#pragma unroll
                for (int u = 0; u < kRefitUnroll; u++) {
                    const int tt = tt0 + u;
                    if (tt >= cn) break;
                    const int t = c0 + tt;
                    const size_t idx = (size_t)t * P + p;
                    const float4 qa = qs[2 * tt], qb = qs[2 * tt + 1];
                    const float qv[6] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y};
                    float val;
                    if (pass == 0) {
                        float y = v[u];
                        if (scatter) {
                            const float *S = scatter + (size_t)t * n * n;
                            const float top = S[o00] * (1.f - fx) + S[o01] * fx;
                            const float bot = S[o10] * (1.f - fx) + S[o11] * fx;
                            y -= top * (1.f - fy) + bot * fy;
                        }
                        resid[idx] = y;
                        if (t == 0) y0 = y;
                        val = y - y0;
                    } else {
                        float fit = 0.f;
#pragma unroll
                        for (int k = 0; k < 6; k++) fit = fmaf(qv[k], beta[k], fit);
                        const float e = v[u] - fit;
                        if (last) {
                            resid[idx] = e;
                            continue;
                        }
                        val = fminf(fmaxf(e, -delta), delta);
                    }
#pragma unroll
                    for (int k = 0; k < 6; k++) part[k] = fmaf(qv[k], val, part[k]);
                    if ((t + 1) % kRefitBlock == 0) {
#pragma unroll
                        for (int k = 0; k < 6; k++) {
                            acc[k] += part[k];
                            part[k] = 0.f;
                        }
                    }
                }
            }
        }
        if (last) break;
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const float s = acc[k] + part[k];
            beta[k] = pass == 0 ? s + y0 * (float)q1[k] : beta[k] + s;
        }
    }
    if (coef && live) {
        // coefficients in the basis (1, x, y, x^2, y^2, x y): beta = R^-1 beta_Q
#pragma unroll
        for (int i = 0; i < 6; i++) {
            double c = 0.0;
#pragma unroll
            for (int k = 0; k < 6; k++) c += Rinv[i * 6 + k] * (double)beta[k];
            coef[(size_t)p * 6 + i] = (float)c;
        }
    }
}

}  // namespace

size_t refit_q_off() { return 0; }
size_t refit_rinv_off(int64_t T) { return align256((size_t)T * kRefitBasisPitch * sizeof(float)); }
size_t refit_q1_off(int64_t T) { return refit_rinv_off(T) + align256(36 * sizeof(double)); }
size_t refit_workspace(int64_t T) { return refit_q1_off(T) + align256(6 * sizeof(double)); }

namespace {

typedef void (*ResidentKernel)(const float *, int, int, int, const float *, int, const float *, const double *, int,
                               float, int, float *, float *);
struct Resident {
    int nw, quads;  // warps and pixel quads of a CTA
    ResidentKernel kern;
};

template <int NW, int QUADS>
Resident resident(bool vec) {
    return {NW, QUADS, vec ? k_refit_resident<NW, QUADS, true> : k_refit_resident<NW, QUADS, false>};
}

// The fewest warps (frames of a thread up to 22, or 24 at the longest) whose
// CTAs of 12 warps fit an SM's shared memory: longer runs per thread mean fewer
// sums to exchange (T = 203: 2 warps 285 us, 8 warps 317 us).  Past 1152 frames
// two such CTAs no longer fit with 16 pixels.
//
// Short series: a block costs its exchanges and latencies whatever its frames,
// so a warp takes 32 or 64 pixels instead of 16 where the image still gives
// every CTA a block.  1024^2, 4 and 10 steps, 16 / 32 / 64 pixels: 6 frames
// 256, 169, 136 and 376, 233, 174 us; 32 frames 327, 255, 230 and 488, 379,
// 334; 48 frames 393, 313, 299 and 596, 482, 447; 96 frames 601, 523 and 928,
// 818.  64^2, 16 / 32 pixels: 32 frames 52, 45 and 52, 49; 96 frames 56, 56 and
// 60, 63.
Resident pick_resident(int64_t T, int64_t P, bool vec) {
    constexpr int64_t ctas = 152 * kResWarps;  // of one warp, at once
    if (T <= 32 && P >= 64 * ctas) return resident<1, 16>(vec);
    if (T <= 48 || (T <= 96 && P >= 32 * ctas)) return resident<1, 8>(vec);
    if (T <= 176) return resident<1, 4>(vec);
    if (T <= 352) return resident<2, 4>(vec);
    if (T <= 528) return resident<3, 4>(vec);
    if (T <= 768) return resident<4, 4>(vec);
    if (T <= 1152) return resident<6, 4>(vec);
    return resident<6, 2>(vec);
}

}  // namespace

int launch_refit(const RefitArgs &a, char *err, size_t errlen) {
    cudaStream_t stream = (cudaStream_t)a.stream;
    const int64_t P = a.H * a.W;
    const float4 *Q = reinterpret_cast<const float4 *>(a.ws + refit_q_off());
    const double *Rinv = reinterpret_cast<const double *>(a.ws + refit_rinv_off(a.T));
    const double *q1 = reinterpret_cast<const double *>(a.ws + refit_q1_off(a.T));
    cudaError_t e = cudaSuccess;
    if (a.T <= kRefitMaxResident) {
        const bool vec = P % 4 == 0 && (uintptr_t)a.data % 16 == 0 && (uintptr_t)a.resid % 16 == 0;
        const Resident r = pick_resident(a.T, P, vec);
        const int groups = 32 * r.nw / r.quads, np = (int)((a.T + 2 * groups - 1) / (2 * groups));
        const size_t smem = (size_t)np * (2 * 32 * r.nw + 3 * groups) * sizeof(float4);
        e = cudaFuncSetAttribute(r.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAllowStatic);
        if (e == cudaSuccess) {
            const int64_t nblk = (P + 4 * r.quads - 1) / (4 * r.quads), ctas = (int64_t)152 * (kResWarps / r.nw);
            const ProfToken tok = prof_begin(kKRefit, stream);
            r.kern<<<(unsigned)(nblk < ctas ? nblk : ctas), 32 * r.nw, smem, stream>>>(
                a.data, (int)a.T, (int)a.H, (int)a.W, a.scatter, a.n, reinterpret_cast<const float *>(Q), Rinv,
                a.iterations, a.delta, np, a.resid, a.coef);
            prof_end(tok);
            e = cudaGetLastError();
        }
    } else {
        const ProfToken tok = prof_begin(kKRefit, stream);
        k_refit<<<(unsigned)((P + kRefitThreads - 1) / kRefitThreads), kRefitThreads, 0, stream>>>(
            a.data, (int)a.T, (int)a.H, (int)a.W, a.scatter, a.n, Q, Rinv, q1, a.iterations, a.delta, a.resid,
            a.coef);
        prof_end(tok);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        snprintf(err, errlen, "k_refit: %s", cudaGetErrorString(e));
        return (int)e;
    }
    return 0;
}

}  // namespace mf
