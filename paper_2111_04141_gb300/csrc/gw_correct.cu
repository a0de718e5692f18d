// Correction Step (Section 2.3, Algorithm convgridding; Section 3.3.8) and the
// centre/corner origin shift used around the FFT (Section 3.3.6).
//
//   correct: image[pol][i][j] *= s(i, j) h(m_i) h(l_j), s = (-1)^(i+j) when the
//            image comes from (or goes to) an FFT of a shifted grid, else 1.
//   shift:   grid[pol][kv][ku] *= (-1)^(kv+ku).
//   finish:  the correction of an image whose grid was not shifted, with the
//            normalisation: the shift's factor (-1)^(kv+ku) is the circular
//            shift by N/2 of the transform, done as a swap of quadrants.
//   fold:    grid += err, err = 0 (ends a compensated gridding sequence).
// For even N, (-1)^(k) before and (-1)^(i) after an unnormalised FFT turn it
// into the transform with both origins at pixel N/2.
#include <cmath>
#include <type_traits>

#include "gw_internal.cuh"

namespace gw {

namespace {

__global__ void k_correct(float2* __restrict__ img, const float* __restrict__ h, int N, int npol,
                          int shift) {
    const int64_t n = (int64_t)N * N;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / N), j = (int)(e - (int64_t)i * N);
        float m = __ldg(h + i) * __ldg(h + j);
        if (shift && ((i + j) & 1)) m = -m;
        for (int p = 0; p < npol; ++p) {
            float2 v = img[(int64_t)p * n + e];
            v.x *= m;
            v.y *= m;
            img[(int64_t)p * n + e] = v;
        }
    }
}

// image[p][i][j] = image[p][i + N/2][j + N/2] (mod N) s(i, j) h(m_i) h(l_j) scale[p]:
// a thread swaps two pixels half the image apart (V of them side by side).
// One pass over the image where shift, correction and normalisation each made
// one: HBM bound, 4096^2 x 4 (0.54 GB read and written) in 0.20 ms, 5.4 TB/s.
template <int V>
__global__ void __launch_bounds__(256) k_finish(float2* __restrict__ img, const float* __restrict__ h,
                                                int N, float scale,
                                                const float* __restrict__ scale_dev) {
    using T = std::conditional_t<V == 2, float4, float2>;
    const int half = N / 2, p = blockIdx.z;
    const float sc = scale_dev ? scale * __ldg(scale_dev + p) : scale;
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    if (j >= N) return;
    const int j2 = j < half ? j + half : j - half;
    float a[V], b[V];                    // column factors of both pixels
#pragma unroll
    for (int k = 0; k < V; ++k) {
        a[k] = __ldg(h + j + k);
        b[k] = __ldg(h + j2 + k);
    }
    float2* const plane = img + (int64_t)p * N * N;
    for (int i = blockIdx.y; i < half; i += gridDim.y) {
        T* const q0 = reinterpret_cast<T*>(plane + (int64_t)i * N + j);
        T* const q1 = reinterpret_cast<T*>(plane + (int64_t)(i + half) * N + j2);
        T x[2] = {*q0, *q1};
        float2* const v0 = reinterpret_cast<float2*>(&x[0]);
        float2* const v1 = reinterpret_cast<float2*>(&x[1]);
        const float h0 = __ldg(h + i), h1 = __ldg(h + i + half);
#pragma unroll
        for (int k = 0; k < V; ++k) {
            // s is the same for both: they are N apart in i + j
            const float m0 = ((i + j + k) & 1) ? -h0 * a[k] : h0 * a[k];
            const float m1 = ((i + j + k) & 1) ? -h1 * b[k] : h1 * b[k];
            const float2 t = v0[k];
            // the scale last: it is 1e30 where every weight is 0
            v0[k] = make_float2(v1[k].x * m0 * sc, v1[k].y * m0 * sc);
            v1[k] = make_float2(t.x * m1 * sc, t.y * m1 * sc);
        }
        *q0 = x[0];
        *q1 = x[1];
    }
}

__global__ void k_shift(float2* __restrict__ g, int N, int npol) {
    const int64_t n = (int64_t)N * N;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / N), j = (int)(e - (int64_t)i * N);
        if (!((i + j) & 1)) continue;
        for (int p = 0; p < npol; ++p) {
            float2 v = g[(int64_t)p * n + e];
            g[(int64_t)p * n + e] = make_float2(-v.x, -v.y);
        }
    }
}

__global__ void k_fold(float2* __restrict__ g, float2* __restrict__ err, int64_t n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const float2 d = err[e];
        if (d.x == 0.f && d.y == 0.f) continue;
        float2 v = g[e];
        v.x += d.x;
        v.y += d.y;
        g[e] = v;
        err[e] = make_float2(0.f, 0.f);
    }
}

__global__ void k_zero_vis(uint32_t* __restrict__ v, int64_t n_max, int words, DevCount dc) {
    const int64_t n = dc.clamp(n_max) * words;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        v[e] = 0u;
}

// exp(+j pi a) for a phase a in units of pi: a is reduced to [-1, 1] in FP64
// (exact for the |a| of any w-screen), then evaluated in FP32.
__device__ __forceinline__ void screen_pi(double a, float& s, float& c) {
    const double r = a - 2.0 * rint(0.5 * a);
    sincospif((float)r, &s, &c);
}

// Phase t = w (n - 1) in turns, reduced modulo 1 in fixed point: with |t| below
// 2^18, t 2^32 + 1.5 x 2^52 (one FP64 operation) holds t's multiple of 2^-32 in
// its low word, which is t modulo 1 as it stands.  Taken below kPhaseTurns, where
// the error of n - 1 (2e-14) is 3e-8 of a radian at most, half of the rounding of
// the FP32 screen.  Relative errors of the sum against 64 bits, phases reduced in
// FP64 / here, e-7: 16 layers of 1024^2, w to 1e3 2.322 / 2.322, to 2.5e5 2.300 / 2.301;
// 32 layers, to 2.6e5, corners beyond the horizon 2.511 / 2.512; 7 layers of 2048^2, to
// 2e4 1.900 / 1.903.  (Multiples of 2^-30 gave 2.327, 2.305, 2.517 and 1.914.)
constexpr double kPhaseScale = 4294967296.0;         // 2^32
constexpr double kPhaseTurns = 262144.0;             // 2^18
__device__ __forceinline__ void screen_fixed(double w32, double nm1, float& s, float& c) {
    const int q = __double2loint(__fma_rn(w32, nm1, 6755399441055744.0));
    sincospif((float)q * 4.656612873077393e-10f, &s, &c);          // 2^-31 half turns
}

// Sum of the layer images times their w-screens exp(+j 2 pi w_l (n - 1)),
// w_l = wmin + l dw (w-stacking, Section 1.7.1).  n - 1 and the phases are
// formed in FP64 (w (n - 1) reaches hundreds of radians); the screens follow
// a rotation recursion in FP32 from an anchor recomputed every 8 layers, and
// the sum is FP32.  The layer images are the inverse transforms of the
// unshifted layer grids: the centring factor (-1)^(u + v) of the grid is the
// circular shift by N/2 of its transform, applied here in the read (N is
// even).  The layers are read once, coalesced.
//
// FIXED: FP64 operations bound the kernel, not the layers it reads, so n - 1 =
// sqrt(1 - r^2) - 1 is an FP32 square root and one Newton step (error below
// 2e-14), and every phase one FP64 operation (screen_fixed).  Otherwise (w of
// 2^18 wavelengths and more) the phases are reduced in FP64.  16 layers of
// 2048^2 x 1: 521 us reduced in FP64, 270 us fixed.
//
// The four pixels (+-i, +-j) from the image's centre have the same screens: a
// thread serves all four (their transform rows are i and N - i), so the
// phases and the recursion are formed once for them.  The same 16 layers: 270
// us with a thread a pixel, 104 us here (0.54 GB read, 5.2 TB/s: HBM bound).
template <bool FIXED, int NPOL>
__global__ void __launch_bounds__(256) k_wstack_combine(const float2* __restrict__ layers,
                                                        int nlayers, double wmin, double dw, int N,
                                                        double cell, float2* __restrict__ image) {
    const int64_t n = (int64_t)N * N;
    const int half = N / 2, side = half + 1;
    const double c2 = cell * cell;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < side * side;
         e += gridDim.x * blockDim.x) {
        const int i = e / side, j = e - i * side;     // offsets from the centre, 0 .. N/2
        // the pixels in the unshifted transform; 0 and N/2 have no mirror
        const bool mi = i > 0 && i < half, mj = j > 0 && j < half;
        const bool on[4] = {true, mj, mi, mi && mj};
        const int rows[2] = {i, mi ? N - i : i}, cols[2] = {j, mj ? N - j : j};
        int es[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) es[q] = rows[q >> 1] * N + cols[q & 1];
        double nm1;
        if constexpr (FIXED) {
            // r^2 = cell^2 (l^2 + m^2), the sum of squares an exact integer
            const double a = __fma_rn(-c2, (double)(i * i + j * j), 1.0);
            nm1 = 0.0;
            if (a > 0.0) {
                const float s0 = sqrtf((float)a);
                const double sd = (double)s0;
                const float corr = __fdividef((float)__fma_rn(-sd, sd, a), 2.f * s0);
                nm1 = (sd - 1.0) + (double)corr;
            }
        } else {
            const double l = j * cell, m = i * cell;
            const double r2 = l * l + m * m;
            nm1 = r2 < 1.0 ? -r2 / (1.0 + sqrt(1.0 - r2)) : 0.0;
        }
        float s1, c1;                                 // one layer step
        if constexpr (FIXED)
            screen_fixed(dw * kPhaseScale, nm1, s1, c1);
        else
            screen_pi(2.0 * dw * nm1, s1, c1);
        float acc[4][NPOL][2] = {};
        float cr = 1.f, ci = 0.f;
        const float2* layer = layers;
        for (int L = 0; L < nlayers; ++L, layer += NPOL * n) {
            float2 v[4][NPOL];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < NPOL; ++p) v[q][p] = __ldcs(layer + p * n + es[q]);
            if ((L & 7) == 0) {
                if constexpr (FIXED)
                    screen_fixed((wmin + L * dw) * kPhaseScale, nm1, ci, cr);
                else
                    screen_pi(2.0 * (wmin + L * dw) * nm1, ci, cr);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int p = 0; p < NPOL; ++p) {
                    acc[q][p][0] = fmaf(v[q][p].x, cr, fmaf(-v[q][p].y, ci, acc[q][p][0]));
                    acc[q][p][1] = fmaf(v[q][p].x, ci, fmaf(v[q][p].y, cr, acc[q][p][1]));
                }
            const float nr = cr * c1 - ci * s1, ni = cr * s1 + ci * c1;
            cr = nr;
            ci = ni;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (!on[q]) continue;
            const int r = rows[q >> 1], c = cols[q & 1];
            const int64_t px = (int64_t)(r < half ? r + half : r - half) * N +
                               (c < half ? c + half : c - half);
#pragma unroll
            for (int p = 0; p < NPOL; ++p) {
                float2 o = image[p * n + px];
                o.x += acc[q][p][0];
                o.y += acc[q][p][1];
                image[p * n + px] = o;
            }
        }
    }
}

unsigned blocks_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    if (b > current_sm_count() * 32) b = current_sm_count() * 32;
    return (unsigned)std::max<int64_t>(b, 1);
}

}  // namespace

void launch_correct(float2* image, const float* h, int N, int npol, int mode, cudaStream_t s) {
    k_correct<<<blocks_for((int64_t)N * N), 256, 0, s>>>(image, h, N, npol, mode != 0);
    note_launch();
}

void launch_finish(float2* image, const float* h, int N, int npol, float scale,
                   const float* scale_dev, cudaStream_t s) {
    // pairs of pixels where both halves of a row start on 16 bytes
    const bool wide = N % 4 == 0 && reinterpret_cast<uintptr_t>(image) % 16 == 0;
    const int per = 256 * (wide ? 2 : 1), cols = (N + per - 1) / per;
    const int rows = std::min(N / 2, std::max(1, current_sm_count() * 32 / (cols * npol)));
    const dim3 grid((unsigned)cols, (unsigned)rows, (unsigned)npol);
    if (wide)
        k_finish<2><<<grid, 256, 0, s>>>(image, h, N, scale, scale_dev);
    else
        k_finish<1><<<grid, 256, 0, s>>>(image, h, N, scale, scale_dev);
    note_launch();
}

void launch_shift(float2* grid, int N, int npol, cudaStream_t s) {
    k_shift<<<blocks_for((int64_t)N * N), 256, 0, s>>>(grid, N, npol);
    note_launch();
}

void launch_zero_vis(void* vis, int kind, int64_t n_max, int npol, DevCount dc, cudaStream_t s) {
    const int words = npol * dtype_bytes(kind) / 4;
    k_zero_vis<<<blocks_for(n_max * words), 256, 0, s>>>(static_cast<uint32_t*>(vis), n_max, words,
                                                        dc);
    note_launch();
}

void launch_wstack_combine(const float2* layers, int nlayers, double wmin, double dw, int N,
                           int npol, double cell, float2* image, cudaStream_t s) {
    // |n - 1| <= 1; the sum of squares of pixel offsets fits 31 bits for any N
    const double w = std::max(std::abs(wmin), std::abs(wmin + (nlayers - 1) * dw));
    const unsigned blocks = blocks_for((int64_t)(N / 2 + 1) * (N / 2 + 1));
    const bool fixed = std::max(w, std::abs(dw)) < kPhaseTurns;
    auto go = [&](auto f, auto g) {
        (fixed ? f : g)<<<blocks, 256, 0, s>>>(layers, nlayers, wmin, dw, N, cell, image);
    };
    switch (npol) {
        case 1: go(k_wstack_combine<true, 1>, k_wstack_combine<false, 1>); break;
        case 2: go(k_wstack_combine<true, 2>, k_wstack_combine<false, 2>); break;
        case 3: go(k_wstack_combine<true, 3>, k_wstack_combine<false, 3>); break;
        default: go(k_wstack_combine<true, 4>, k_wstack_combine<false, 4>); break;
    }
    note_launch();
}

void launch_fold(float2* grid, float2* err, int64_t n, cudaStream_t s) {
    k_fold<<<blocks_for(n), 256, 0, s>>>(grid, err, n);
    note_launch();
}

}  // namespace gw
