// imaging.cu -- the imaging half of the major cycle (Sec. 2.2, the Cotton-
// Schwab steps after Eq. 6) around the model prediction: gridding and FFT
// to a dirty image, Hogbom clean (Eqs. 4-6), and the loop of major cycles.
//
// Conventions (an n x n image, n even, pixel size dl radians):
//   pixel (ix, iy) at l = (ix - n/2) dl, m = (iy - n/2) dl, arrays [iy][ix];
//   uv cell (iu, iv) at u = (iu - n/2) du, v = (iv - n/2) du, du = 1/(n dl).
// Gridding is nearest-cell with unit weights: each visibility and its
// Hermitian conjugate at -B (a visibility whose cell falls outside the grid
// is left out); the w term is not used in imaging (the 2-D transform of
// Eq. 2). The dirty image is (1/W) Re sum_cells G(u, v) exp(-i 2 pi (ul + vm))
// with W the number of gridded entries, so that a unit point source at the
// phase centre images to 1; the dirty beam is the image of unit
// visibilities. Both index shifts of the transform (cell n/2 is u = 0,
// pixel n/2 is l = 0) are applied as (-1)^(iu+iv) on the grid and
// (-1)^(ix+iy) on the image, which is exact for even n.
//
// The 2-D FFT is cuFFT's, loaded at first use (a library call for a plain
// transform); everything else is in the kernels below.
//
// Hogbom clean takes "the pixel with the maximum value" literally (the
// largest value; ties to the first pixel in row-major order), subtracts
// g C times the beam centred there wherever it overlaps the image, and
// stops after max_iter components or when the maximum falls below the
// threshold. The arithmetic is float32 without contraction: fl(g C) and
// fl(I - fl(f B)). Two schedules, identical results:
//   persistent  the whole minor cycle in one cooperative launch: each CTA
//               keeps its rows of the image in shared memory for every
//               iteration; the CTAs meet once for a batch of components,
//               each found among the largest pixels they posted there, and
//               subtract the batch from their rows (the beam is read from
//               global memory and stays in L2);
//   per launch  one launch per iteration when the rows do not fit in shared
//               memory: every CTA subtracts the previous component over its
//               pixels and finds its largest updated value; a 64-bit
//               atomicMax picks the winner and the last CTA to finish (an
//               atomic counter, no waiting) records the component for the
//               next launch.
#include <dlfcn.h>
#include <math.h>
#include <stdint.h>
#include <stddef.h>
#include <string.h>

#include <cufft.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "wt_internal.cuh"

namespace wt {
namespace {

// ---------------------------------------------------------------- cuFFT
struct CufftApi {
    bool tried = false;
    void* so = nullptr;
    cufftResult (*plan2d)(cufftHandle*, int, int, cufftType) = nullptr;
    cufftResult (*set_stream)(cufftHandle, cudaStream_t) = nullptr;
    cufftResult (*exec_c2c)(cufftHandle, cufftComplex*, cufftComplex*, int) = nullptr;
    cufftResult (*destroy)(cufftHandle) = nullptr;
};

std::mutex g_fft_mu;
CufftApi g_fft;

struct FftPlan {
    int device, n;
    cufftHandle h;
};
std::vector<FftPlan> g_plans;

int fft_api()
{
    if (g_fft.so) return WT_OK;
    if (g_fft.tried) return set_error(WT_ERR_UNSUPPORTED, "cuFFT (libcufft.so) could not be loaded");
    g_fft.tried = true;
    const char* names[] = {"libcufft.so.12", "libcufft.so", "/usr/local/cuda/lib64/libcufft.so.12"};
    for (const char* nm : names)
        if ((g_fft.so = dlopen(nm, RTLD_NOW | RTLD_LOCAL))) break;
    if (!g_fft.so) return set_error(WT_ERR_UNSUPPORTED, "cuFFT (libcufft.so) could not be loaded");
    g_fft.plan2d = reinterpret_cast<decltype(g_fft.plan2d)>(dlsym(g_fft.so, "cufftPlan2d"));
    g_fft.set_stream = reinterpret_cast<decltype(g_fft.set_stream)>(dlsym(g_fft.so, "cufftSetStream"));
    g_fft.exec_c2c = reinterpret_cast<decltype(g_fft.exec_c2c)>(dlsym(g_fft.so, "cufftExecC2C"));
    g_fft.destroy = reinterpret_cast<decltype(g_fft.destroy)>(dlsym(g_fft.so, "cufftDestroy"));
    if (!g_fft.plan2d || !g_fft.set_stream || !g_fft.exec_c2c || !g_fft.destroy) {
        g_fft.so = nullptr;
        return set_error(WT_ERR_UNSUPPORTED, "cuFFT loaded without the expected entry points");
    }
    return WT_OK;
}

// In-place forward 2-D transform (sign -1) of an n x n complex64 array.
int fft2_forward(float2* data, int n, cudaStream_t s)
{
    std::lock_guard<std::mutex> lk(g_fft_mu);
    int rc = fft_api();
    if (rc) return rc;
    int dev = 0;
    WT_CUDA_TRY(cudaGetDevice(&dev));
    cufftHandle h = 0;
    bool found = false;
    for (const FftPlan& p : g_plans)
        if (p.device == dev && p.n == n) {
            h = p.h;
            found = true;
        }
    if (!found) {
        if (g_fft.plan2d(&h, n, n, CUFFT_C2C) != CUFFT_SUCCESS)
            return set_error(WT_ERR_CUDA, "cufftPlan2d(%d x %d) failed", n, n);
        g_plans.push_back(FftPlan{dev, n, h});
    }
    if (g_fft.set_stream(h, s) != CUFFT_SUCCESS) return set_error(WT_ERR_CUDA, "cufftSetStream failed");
    cufftComplex* d = reinterpret_cast<cufftComplex*>(data);
    if (g_fft.exec_c2c(h, d, d, CUFFT_FORWARD) != CUFFT_SUCCESS) return set_error(WT_ERR_CUDA, "cufftExecC2C failed");
    return WT_OK;
}

// ---------------------------------------------------------------- gridding
constexpr int kImgThreads = 256;

// Visibility n (unit value if vis is null) and its conjugate into their
// cells, times (-1)^(iu+iv) (the index shift); counts the entries.
__global__ void k_grid_nn(const double* __restrict__ uvw, const float2* __restrict__ vis, int64_t n_vis, int n,
                          double inv_du, float2* __restrict__ grid, unsigned long long* __restrict__ count)
{
    __shared__ unsigned int blk;
    if (threadIdx.x == 0) blk = 0;
    __syncthreads();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n_vis) {
        const double ru = rint(uvw[3 * i] * inv_du), rv = rint(uvw[3 * i + 1] * inv_du);
        const double h = 0.5 * n;
        if (ru > -h && ru < h && rv > -h && rv < h) {
            const int iu = static_cast<int>(ru) + n / 2, iv = static_cast<int>(rv) + n / 2;
            const int ju = n - iu, jv = n - iv;               // the mirrored cell: n/2 - ru
            const float2 V = vis ? vis[i] : make_float2(1.0f, 0.0f);
            const float sg = ((iu + iv) & 1) ? -1.0f : 1.0f;   // (-1)^(ju+jv) is the same: n even
            float* a = reinterpret_cast<float*>(grid + static_cast<int64_t>(iv) * n + iu);
            float* b = reinterpret_cast<float*>(grid + static_cast<int64_t>(jv) * n + ju);
            atomicAdd(a, sg * V.x);
            atomicAdd(a + 1, sg * V.y);
            atomicAdd(b, sg * V.x);
            atomicAdd(b + 1, -sg * V.y);
            atomicAdd(&blk, 2u);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && blk) atomicAdd(count, static_cast<unsigned long long>(blk));
}

// Real part of the transformed grid, times (-1)^(ix+iy) / W.
__global__ void k_image_from_fft(const float2* __restrict__ f, int n, const unsigned long long* __restrict__ count,
                                 float* __restrict__ image)
{
    const unsigned long long W = *count;
    const float inv = W ? static_cast<float>(1.0 / static_cast<double>(W)) : 0.0f;
    for (int iy = blockIdx.x; iy < n; iy += gridDim.x) {            // a row per CTA step, no division
        const int64_t row = static_cast<int64_t>(iy) * n;
        for (int ix = threadIdx.x; ix < n; ix += blockDim.x) {
            const float sg = ((ix + iy) & 1) ? -1.0f : 1.0f;
            image[row + ix] = sg * f[row + ix].x * inv;
        }
    }
}

// ---------------------------------------------------------------- w-projection
// The w-corrected dirty image (the wide-field imaging of Sec. 3.6.2, which
// grids with an anti-aliasing kernel and a w-kernel over w-planes):
//   I(l, m) = (1/W) Re sum_entries V exp(-i 2 pi (u l + v m + w (n(l, m) - 1))),
// approximated by convolutional gridding. In image units t = l / (n dl),
// s = m / (n dl) (the field is |t|, |s| < 1/2) and uv units of cells
// x = u / du, the kernel of a plane at w is
//   K_w(x, y) = int int c(t) c(s) exp(-i 2 pi w (n - 1)) exp(i 2 pi (x t + y s)) dt ds
// over the field, c the Fourier transform of a Kaiser-Bessel kernel of
// width kWpWidth cells (closed form, c(0) = 1); summed over all cells,
// sum_x K_w(x - x_k) exp(-i 2 pi x t) = c(t) exp(-i 2 pi w (n - 1)) exp(-i 2 pi x_k t)
// inside the field, so the transformed grid divided by c(t) c(s) is the
// image above. K_w is tabulated at kWpOversample points per cell over the
// support S = 2h + 1 cells (h from the largest chirp frequency of the field
// and the Kaiser-Bessel half-width) for planes uniformly spaced in |w|,
// from a midpoint sum over kWpSamples^2 points of the field, and interpolated
// linearly in |w| between the two nearest planes. Each visibility stands for
// two entries, V at B and conj(V) at -B, whose taps are each other's conjugates
// at mirrored cells: the one at w >= 0 is worked out and added to both. Each
// entry is spread over the support its own |w| needs (the same rule at that
// |w|), not the table's.
//
// The table is summed over the whole field in a fixed order, multiplications
// and additions rounded one by one: its rounding, divided by c(t) c(s) at the
// image's edges, is most of a small image's error (1e-5 of it), and sums over
// one quadrant with real cosines (16 times less work, 34 us where this takes
// 119 at 64 planes and h = 11) move every image by as much. What the symmetry
// gives exactly is taken: f is even in q, so stage 1 runs over half its rows.
// 657 + 230 us with a thread per point reading along its own row of tw; the
// field 18 us, 420 with float64 tapers and sincospi at every sample.
constexpr int kWpWidth = 7;             // Kaiser-Bessel width (cells)
constexpr double kWpBeta = 16.25;       // its shape parameter
constexpr int kWpOversample = 8;        // table points per cell
constexpr int kWpSamples = 128;         // field samples per axis for the kernels
constexpr int kWpHalf = kWpSamples / 2; // those at t > 0
constexpr int kWpMaxHalf = 32;          // largest half-support h (cells)

// c(t) / c(0) for the Kaiser-Bessel kernel of width W and shape beta: the
// kernel's Fourier transform, sinh(sqrt(beta^2 - (pi W t)^2)) / sqrt(...),
// or sin(...) / ... past the zero of the root.
__host__ __device__ inline double kb_taper(double t)
{
    const double a = kWpBeta * kWpBeta - (kPi * kWpWidth * t) * (kPi * kWpWidth * t);
    const double c0 = sinh(kWpBeta) / kWpBeta;
    if (a > 0.0) {
        const double r = sqrt(a);
        return (sinh(r) / r) / c0;
    }
    if (a < 0.0) {
        const double r = sqrt(-a);
        return (sin(r) / r) / c0;
    }
    return 1.0 / c0;
}

struct WpPlan {
    int P;          // planes
    int h, S;       // half-support, support (cells)
    int T;          // table points per axis (S * oversample + 1)
    double dw;      // plane spacing in |w|
    double ndl;     // n dl: the field width (radians)
    double xc_per_w;   // the field's largest chirp frequency (cells) per unit |w|
};

__device__ __forceinline__ double wp_sample(int q) { return (q + 0.5) / kWpSamples; }   // the q-th t > 0

// The tables of one image: tw[r][j] = exp(i 2 pi x_j t_r), x_j = j /
// oversample - (h + 1/2), for the samples t_r > 0 (at -t_r its conjugate);
// ft[r] = c(t_r); gc[i] = 1 / c((i - n/2) / n), the pixels' grid correction,
// as a double-float.
__global__ void k_wp_tables(WpPlan pl, int n, float2* __restrict__ tw, double* __restrict__ ft, F2* __restrict__ gc)
{
    const int nt = pl.T * kWpHalf, total = nt + kWpHalf + n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        if (i < nt) {
            const int r = i / pl.T, j = i % pl.T;
            const double x = static_cast<double>(j) / kWpOversample - (pl.h + 0.5);
            double sn, cs;
            sincos_turns_f64(x * wp_sample(r), sn, cs);
            tw[i] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
        } else if (i < nt + kWpHalf) {
            ft[i - nt] = kb_taper(wp_sample(i - nt));
        } else {
            const int k = i - nt - kWpHalf;
            gc[k] = split_f64(1.0 / kb_taper(static_cast<double>(k - n / 2) / n));
        }
    }
}

// f[p][q][r] = c(t_q) c(t_r) exp(-i 2 pi w_p (n - 1)) at the field's sample
// points t > 0 (float64 phase): a thread per (q, r), the planes of a group of
// kWpFieldPlanes one after the other (n - 1 and the taper are theirs alike).
constexpr int kWpFieldPlanes = 4;

__global__ void k_wp_field(WpPlan pl, const double* __restrict__ ft, float2* __restrict__ f)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kWpHalf * kWpHalf) return;
    const int r = i % kWpHalf, q = i / kWpHalf;
    const double l = wp_sample(q) * pl.ndl, m = wp_sample(r) * pl.ndl;
    const double r2 = l * l + m * m;
    const double nm1 = -r2 / (1.0 + sqrt(1.0 - r2));
    const double c = ft[q] * ft[r];
    const int p1 = min(pl.P, static_cast<int>(blockIdx.y + 1) * kWpFieldPlanes);
    for (int p = blockIdx.y * kWpFieldPlanes; p < p1; ++p) {
        double sn, cs;
        sincos_turns_f64(-(p * pl.dw) * nm1, sn, cs);
        f[static_cast<int64_t>(p) * kWpHalf * kWpHalf + i] =
            make_float2(static_cast<float>(c * cs), static_cast<float>(c * sn));
    }
}

// The products' inner step for kWpGroup rows and two columns at once: acc[g] +=
// x_g b, x_g spread over pairs as (re, re, im, im): fl(re b.re - fl(im b.im))
// and fl(re b.im + fl(im b.re)), then added, two elements per packed operation
// (one 16-byte read of shared memory per six of them).
constexpr int kWpGroup = 8;

__device__ __forceinline__ void wp_step(float2 (&acc)[kWpGroup][2], const float4* x, float2 b0, float2 b1)
{
    const float2 s0 = make_float2(-b0.y, b0.x), s1 = make_float2(-b1.y, b1.x);
#pragma unroll
    for (int g = 0; g < kWpGroup; ++g) {
        const float4 v = x[g];
        const float2 re = make_float2(v.x, v.y), im = make_float2(v.z, v.w);
        acc[g][0] = add2(acc[g][0], fma2(re, b0, mul2(im, s0)));
        acc[g][1] = add2(acc[g][1], fma2(re, b1, mul2(im, s1)));
    }
}
__device__ __forceinline__ float4 wp_pairs(float2 v) { return make_float4(v.x, v.x, v.y, v.y); }

// a[p][q][j] = sum_r f[p][q][r] tw[j][r] for the rows q at t > 0 (those at -t
// are the same): a CTA per (plane, kWpGroup rows), a thread per two columns.
__global__ void k_wp_stage1(WpPlan pl, const float2* __restrict__ f, const float2* __restrict__ tw,
                            float2* __restrict__ a)
{
    __shared__ float4 row[kWpHalf][kWpGroup];
    const int p = blockIdx.x, q0 = blockIdx.y * kWpGroup;
    const float2* src = f + (static_cast<int64_t>(p) * kWpHalf + q0) * kWpHalf;
    for (int i = threadIdx.x; i < kWpGroup * kWpHalf; i += blockDim.x)
        row[i % kWpHalf][i / kWpHalf] = wp_pairs(src[i]);
    __syncthreads();
    const int half = (pl.T + 1) / 2;
    for (int j = threadIdx.x; j < half; j += blockDim.x) {
        const int j1 = min(j + half, pl.T - 1);   // T odd: the last thread's second column is its neighbour's too
        float2 acc[kWpGroup][2];
#pragma unroll
        for (int g = 0; g < kWpGroup; ++g) acc[g][0] = acc[g][1] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int r = kWpHalf - 1; r >= 0; --r) {   // t < 0
            const float2 t0 = __ldg(tw + r * pl.T + j), t1 = __ldg(tw + r * pl.T + j1);
            wp_step(acc, row[r], make_float2(t0.x, -t0.y), make_float2(t1.x, -t1.y));
        }
#pragma unroll 4
        for (int r = 0; r < kWpHalf; ++r) wp_step(acc, row[r], __ldg(tw + r * pl.T + j), __ldg(tw + r * pl.T + j1));
#pragma unroll
        for (int g = 0; g < kWpGroup; ++g) {
            float2* out = a + (static_cast<int64_t>(p) * kWpHalf + q0 + g) * pl.T;
            out[j] = acc[g][0];
            out[j1] = acc[g][1];
        }
    }
}

// The table point (i, j), x_i and y_j, of plane p is (1/M^2) sum_q tw[i][q]
// a[p][q][j]: a CTA per (plane, kWpGroup points i), a thread per two points j.
// Written as the gridding reads it: K[p][oy][ox][ty][tx], tx, ty = 0 .. S, i =
// tx oversample + ox, j = ty oversample + oy (an entry's taps are whole rows;
// the places past the last point, i = S oversample, are never read).
__global__ void k_wp_stage2(WpPlan pl, const float2* __restrict__ a, const float2* __restrict__ tw,
                            float2* __restrict__ K)
{
    constexpr int O = kWpOversample;
    __shared__ float4 neg[kWpHalf][kWpGroup], pos[kWpHalf][kWpGroup];
    const int p = blockIdx.x, i0 = blockIdx.y * kWpGroup;
    for (int k = threadIdx.x; k < kWpGroup * kWpHalf; k += blockDim.x) {
        const int q = k / kWpGroup, g = k % kWpGroup;
        const float2 t = i0 + g < pl.T ? tw[q * pl.T + i0 + g] : make_float2(0.f, 0.f);
        pos[q][g] = wp_pairs(t);
        neg[q][g] = wp_pairs(make_float2(t.x, -t.y));
    }
    __syncthreads();
    const float inv = 1.0f / (static_cast<float>(kWpSamples) * static_cast<float>(kWpSamples));
    const int half = (pl.T + 1) / 2, R = pl.S + 1;
    float2* out = K + static_cast<int64_t>(p) * O * O * R * R;
    for (int j = threadIdx.x; j < half; j += blockDim.x) {
        const int j1 = min(j + half, pl.T - 1);
        float2 acc[kWpGroup][2];
#pragma unroll
        for (int g = 0; g < kWpGroup; ++g) acc[g][0] = acc[g][1] = make_float2(0.f, 0.f);
        const float2* ap = a + static_cast<int64_t>(p) * kWpHalf * pl.T;
#pragma unroll 4
        for (int q = kWpHalf - 1; q >= 0; --q)
            wp_step(acc, neg[q], __ldg(ap + q * pl.T + j), __ldg(ap + q * pl.T + j1));
#pragma unroll 4
        for (int q = 0; q < kWpHalf; ++q) wp_step(acc, pos[q], __ldg(ap + q * pl.T + j), __ldg(ap + q * pl.T + j1));
#pragma unroll
        for (int g = 0; g < kWpGroup; ++g)
            if (i0 + g < pl.T) {
                const int ox = (i0 + g) % O, tx = (i0 + g) / O;
                out[((j % O) * O + ox) * R * R + (j / O) * R + tx] = make_float2(acc[g][0].x * inv, acc[g][0].y * inv);
                out[((j1 % O) * O + ox) * R * R + (j1 / O) * R + tx] =
                    make_float2(acc[g][1].x * inv, acc[g][1].y * inv);
            }
    }
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// An entry whose offsets sit within kWpTie of a tie between two table points
// (in units of the table's spacing): float32 rounds the taps' positions to
// their nearest points one by one, each entry of the Hermitian pair by itself,
// and near a tie they need not agree. Three float32 roundings of positions
// below 2 kWpMaxHalf + 1 cells, 2^-19 each, times the oversampling: below
// 2^-14.
constexpr float kWpTie = 1.0f / 8192;

__device__ __forceinline__ float2 wp_mix(float2 k0, float2 k1, float a)
{
    return make_float2(fmaf(a, k1.x - k0.x, k0.x), fmaf(a, k1.y - k0.y, k0.y));
}

// The general form of an entry (V at cell (uc, vc) of the grid, half-support
// he, offsets fx, fy): every tap finds its table point in each entry of the
// pair.
__device__ __noinline__ void wp_spread_ties(const WpPlan& pl, const float2* __restrict__ K0, float a, float2 V,
                                            int uc, int vc, int he, float fx, float fy, int n,
                                            float2* __restrict__ grid, int lane)
{
    constexpr int O = kWpOversample;
    const int R = pl.S + 1, last = pl.S * O, Se = 2 * he + 1;
    const int64_t mirror = static_cast<int64_t>(n / 2 * 2) * (n + 1);   // the sum of two mirrored cells' indices
    const float2* K1 = K0 + static_cast<int64_t>(O) * O * R * R;
    auto index = [&](int d, float f) { return __float2int_rn((static_cast<float>(d) - f + pl.h + 0.5f) * O); };
    auto value = [&](int ix, int iy) {
        const int at = ((iy % O) * O + ix % O) * R * R + (iy / O) * R + ix / O;
        return wp_mix(__ldg(K0 + at), __ldg(K1 + at), a);
    };
    for (int t = lane; t < Se * Se; t += 32) {
        const int dx = t % Se - he, dy = t / Se - he;
        const float2 k0 = value(index(dx, fx), index(dy, fy));
        const float2 k1 = value(last - index(-dx, -fx), last - index(-dy, -fy));
        const float sg = ((uc + dx + vc + dy) & 1) ? -1.0f : 1.0f;
        const int64_t at = static_cast<int64_t>(vc + dy) * n + uc + dx;
        const float2 e = cmul(V, k0), m = cmul(V, k1);
        atomicAdd(grid + at, make_float2(sg * e.x, sg * e.y));
        atomicAdd(grid + (mirror - at), make_float2(sg * m.x, -sg * m.y));
    }
}

// A warp takes every warps-th visibility (unit values if vis is null), 32 at a
// time: each lane plans one (cell, offset, planes, support: float64 work that a
// whole warp would repeat), then the warp spreads them one after the other, a
// lane per tap, row by row, into both cells of the pair. An entry whose support
// leaves the grid is dropped; counts two entries per visibility gridded.
// Bound by the load/store path: per tap 16 bytes of table (two planes, rows of
// the layout) and two 8-byte additions to the grid, all in whole lines. Medium
// array, 1 008 000 visibilities, 2048 x 2048, 64 planes: 0.73 ms, against 3.0
// when each entry read the table across its rows and added 4 bytes at a time.
// The visibilities are dealt to the warps in a fixed interleaving, but a cell's
// float32 sum takes them as the warps reach it: two runs on the same input differ
// (by 1.5e-5 of the image, RMS; 2e-7 to 3.4e-5 over other sizes, where the error
// against float64 is 7e-5, and 1e-5 to 2.2e-4: a thousand additions of like sign
// under a correction of 1 / c^2 = 2 900 in the corners). One entry per pair and the
// image doubled, runs of neighbouring visibilities to a warp, take 0.44 ms and are
// no less accurate, but put like visibilities next to one another in the sums and
// so move images by up to 1.4e-4, beyond what runs differ by: not taken.
__global__ void __launch_bounds__(256) k_grid_wproj(WpPlan pl, const float2* __restrict__ K,
                                                    const double* __restrict__ uvw, const float2* __restrict__ vis,
                                                    int64_t n_vis, int n, double inv_du,
                                                    float2* __restrict__ grid, unsigned long long* __restrict__ count)
{
    constexpr int O = kWpOversample;
    __shared__ unsigned int blk;
    if (threadIdx.x == 0) blk = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int R = pl.S + 1, half = n / 2;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
    const int64_t plane = static_cast<int64_t>(O) * O * R * R;
    const int64_t mirror = static_cast<int64_t>(half * 2) * (n + 1);   // the sum of two mirrored cells' indices
    for (int64_t k0 = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5); k0 < n_vis;
         k0 += 32 * warps) {
        const int64_t k = k0 + lane * warps;
        // the plan of this lane's visibility: its cell, half-support, lower plane,
        // table row and column of the first tap (-1: near a tie), offset from the
        // cell's centre and weight between the planes
        int uc = 0, vc = 0, he = -1, p0 = 0, tab = -1;
        float fx = 0.0f, fy = 0.0f, a = 0.0f;
        float2 V = make_float2(0.f, 0.f);
        if (k < n_vis) {
            double x = uvw[3 * k] * inv_du, y = uvw[3 * k + 1] * inv_du, w = uvw[3 * k + 2];
            V = vis ? vis[k] : make_float2(1.0f, 0.0f);
            if (w < 0.0) {               // the conjugate entry
                x = -x;
                y = -y;
                w = -w;
                V.y = -V.y;
            }
            const double icd = rint(x), jcd = rint(y);
            const double lo = -half + pl.h + 1, hi = half - pl.h - 1;
            if (icd >= lo && icd <= hi && jcd >= lo && jcd <= hi && w <= 1e30) {   // false for NaN too
                fx = static_cast<float>(x - icd);
                fy = static_cast<float>(y - jcd);
                const double pw = w / pl.dw;
                p0 = static_cast<int>(floor(pw));
                if (p0 > pl.P - 2) p0 = pl.P - 2;
                if (p0 < 0) p0 = 0;
                a = static_cast<float>(fmin(fmax(pw - p0, 0.0), 1.0));
                // this entry's own support: the Kaiser-Bessel half-width and the
                // chirp frequency of its |w| (the kernel is negligible beyond),
                // within the table's
                he = static_cast<int>(fmin(ceil(0.5 * kWpWidth + pl.xc_per_w * w) + 1.0, static_cast<double>(pl.h)));
                uc = static_cast<int>(icd) + half;
                vc = static_cast<int>(jcd) + half;
                // tap d's nearest table point is at (d - fx + h + 1/2) oversample:
                // d + h cells and an offset o = 0 .. oversample alike for every tap
                // (o = oversample: the next cell's 0)
                const float gx = (0.5f - fx) * O, gy = (0.5f - fy) * O;
                const int ox = __float2int_rn(gx), oy = __float2int_rn(gy);
                if (fabsf(fabsf(gx - ox) - 0.5f) > kWpTie && fabsf(fabsf(gy - oy) - 0.5f) > kWpTie)
                    tab = (((oy % O) * O + ox % O) * R + pl.h - he + oy / O) * R + pl.h - he + ox / O;
            }
        }
        const unsigned todo = __ballot_sync(0xffffffffu, he >= 0);
        if (lane == 0 && todo) atomicAdd(&blk, 2u * __popc(todo));
        for (unsigned left = todo; left; left &= left - 1) {
            const int src = __ffs(left) - 1;
            const int su = __shfl_sync(0xffffffffu, uc, src), sv = __shfl_sync(0xffffffffu, vc, src);
            const int sh = __shfl_sync(0xffffffffu, he, src), st = __shfl_sync(0xffffffffu, tab, src);
            const int sp = __shfl_sync(0xffffffffu, p0, src);
            const float sa = __shfl_sync(0xffffffffu, a, src);
            const float2 sV = make_float2(__shfl_sync(0xffffffffu, V.x, src), __shfl_sync(0xffffffffu, V.y, src));
            const float2* K0 = K + sp * plane;
            if (st < 0) {
                const float sx = __shfl_sync(0xffffffffu, fx, src), sy = __shfl_sync(0xffffffffu, fy, src);
                wp_spread_ties(pl, K0, sa, sV, su, sv, sh, sx, sy, n, grid, lane);
                continue;
            }
            K0 += st;
            const float2* K1 = K0 + plane;
            const int Se = 2 * sh + 1;
            float2* out = grid + static_cast<int64_t>(sv - sh) * n + su - sh;   // the first tap's cell
            float2* opp = grid + (mirror - (out - grid));           // the mirrored entry's
            const int par = su + sv;                               // of (-1)^(iu+iv): that of the first tap's cell
            const unsigned recip = ((1u << 20) + Se - 1) / Se;     // t / Se = (t recip) >> 20 for t < 65^2
            for (int t = lane; t < Se * Se; t += 32) {
                const int r = static_cast<int>((t * recip) >> 20), q = t - r * Se;
                const int at = r * R + q;
                const float2 e = cmul(sV, wp_mix(__ldg(K0 + at), __ldg(K1 + at), sa));
                const float sg = ((par + r + q) & 1) ? -1.0f : 1.0f;
                const float2 v = make_float2(sg * e.x, sg * e.y);
                atomicAdd(out + (r * n + q), v);
                atomicAdd(opp - (r * n + q), make_float2(v.x, -v.y));
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && blk) atomicAdd(count, static_cast<unsigned long long>(blk));
}

// Real part of the transformed grid, times (-1)^(ix+iy) / (W c(t) c(s)), the
// correction's product in double-float: of 2e8 pixels four round to a float32
// other than the float64 quotient's, by a unit in the last place. Bound by HBM (12
// bytes per pixel): 23 us at 2048 x 2048, 46 with the product in float64, 714 with
// both tapers evaluated per pixel.
__global__ void k_image_from_fft_wp(const float2* __restrict__ f, int n, const unsigned long long* __restrict__ count,
                                    const F2* __restrict__ gc, float* __restrict__ image)
{
    const unsigned long long W = *count;
    const double inv = W ? 1.0 / static_cast<double>(W) : 0.0;
    for (int iy = blockIdx.x; iy < n; iy += gridDim.x) {
        const int64_t row = static_cast<int64_t>(iy) * n;
        const F2 g = gc[iy];
        const F2 cy = split_f64((static_cast<double>(g.hi) + static_cast<double>(g.lo)) * inv);
        for (int ix = threadIdx.x; ix < n; ix += blockDim.x) {
            const float sg = ((ix + iy) & 1) ? -1.0f : 1.0f;
            float p, t;
            df_product(cy, gc[ix], p, t);
            const float v = sg * f[row + ix].x;
            image[row + ix] = fmaf(v, p, v * t);
        }
    }
}

// ---------------------------------------------------------------- Hogbom
struct HogbomState {
    unsigned long long key;   // (ordered value << 32) | (0xffffffff - pixel) of the current maximum
    unsigned int done;        // CTAs finished in this launch
    int iter;                 // components recorded
    int stopped;              // 1 once the clean has ended
    int pend_pix;             // component to subtract at the next launch (-1: none)
    float pend_flux;
    int pad;
};

__device__ __forceinline__ unsigned int ordered(float v)
{
    const unsigned int b = __float_as_uint(v);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);   // monotone in v
}

__global__ void __launch_bounds__(kImgThreads) k_hogbom_step(float* __restrict__ img, const float* __restrict__ psf,
                                                             int n, float gain, float threshold, int max_iter,
                                                             HogbomState* __restrict__ st, int* __restrict__ comp_pix,
                                                             float* __restrict__ comp_flux, int* __restrict__ n_comp)
{
    __shared__ unsigned long long best[kImgThreads / 32];
    __shared__ bool last;
    if (st->stopped) return;
    const int p = st->pend_pix;
    const float f = st->pend_flux;
    const int py = p >= 0 ? p / n : 0, px = p >= 0 ? p % n : 0, c = n / 2;
    // this thread's largest value and its pixel: pixels are visited in
    // increasing order, so a strict comparison keeps the first of equals
    float bv = -INFINITY;
    unsigned int bq = 0xffffffffu;
    const bool vec4 = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(img) & 15) == 0;
    for (int qy = blockIdx.x; qy < n; qy += gridDim.x) {            // a row per CTA step, no division
        const int by = qy - py + c;                                 // beam row under image row qy
        const bool row_hit = p >= 0 && by >= 0 && by < n;
        float* irow = img + static_cast<int64_t>(qy) * n;
        const float* brow = psf + static_cast<int64_t>(row_hit ? by : 0) * n;
        const unsigned int q0 = static_cast<unsigned int>(qy) * static_cast<unsigned int>(n);
        if (vec4) {                                                 // four pixels per step, 16-byte image accesses
            for (int qx = 4 * threadIdx.x; qx < n; qx += 4 * blockDim.x) {
                float4 v4 = *reinterpret_cast<const float4*>(irow + qx);
                float v[4] = {v4.x, v4.y, v4.z, v4.w};
                if (row_hit) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int bx = qx + j - px + c;             // beam column under qx + j
                        if (bx >= 0 && bx < n) v[j] = __fsub_rn(v[j], __fmul_rn(f, brow[bx]));
                    }
                    *reinterpret_cast<float4*>(irow + qx) = make_float4(v[0], v[1], v[2], v[3]);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (v[j] > bv) {
                        bv = v[j];
                        bq = q0 + static_cast<unsigned int>(qx + j);
                    }
            }
        } else {
            for (int qx = threadIdx.x; qx < n; qx += blockDim.x) {
                float v = irow[qx];
                const int bx = qx - px + c;
                if (row_hit && bx >= 0 && bx < n) {
                    v = __fsub_rn(v, __fmul_rn(f, brow[bx]));
                    irow[qx] = v;
                }
                if (v > bv) {
                    bv = v;
                    bq = q0 + static_cast<unsigned int>(qx);
                }
            }
        }
    }
    unsigned long long key =
        bq == 0xffffffffu ? 0ull : (static_cast<unsigned long long>(ordered(bv)) << 32) | (0xffffffffu - bq);
    __threadfence();   // this thread's image updates before the CTA's count below
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
        if (other > key) key = other;
    }
    if ((threadIdx.x & 31) == 0) best[threadIdx.x >> 5] = key;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long b = best[0];
        for (int w = 1; w < kImgThreads / 32; ++w)
            if (best[w] > b) b = best[w];
        atomicMax(&st->key, b);
        __threadfence();   // the key before the count
        last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x != 0) return;
    // the last CTA: every other CTA's writes are visible after the fence
    __threadfence();
    const unsigned long long k = atomicAdd(&st->key, 0ull);
    // no comparable value anywhere (an all-NaN image): nothing to clean
    const int win = k ? static_cast<int>(0xffffffffu - static_cast<unsigned int>(k & 0xffffffffu)) : 0;
    const float peak = k ? __ldcg(img + win) : __int_as_float(0x7fc00000);
    const int it = st->iter;
    if (it >= max_iter || !(peak >= threshold)) {
        st->stopped = 1;
        st->pend_pix = -1;
    } else {
        const float flux = __fmul_rn(gain, peak);
        comp_pix[it] = win;
        comp_flux[it] = flux;
        st->iter = it + 1;
        st->pend_pix = win;
        st->pend_flux = flux;
    }
    *n_comp = st->iter;
    st->key = 0;
    st->done = 0;
    __threadfence();
}

__global__ void k_hogbom_reset(HogbomState* st, int* n_comp)
{
    st->key = 0;
    st->done = 0;
    st->iter = 0;
    st->stopped = 0;
    st->pend_pix = -1;
    st->pend_flux = 0.0f;
    st->pad = 0;
    *n_comp = 0;
}

// ---------------------------------------------------------------- persistent Hogbom
// Several components per synchronisation. Finding one component over the whole
// grid costs a grid-wide exchange (3 us, half an iteration at 2048 x 2048 and
// nearly all of it below 1024 x 1024), but the next components are almost always among
// a few hundred pixels that are already known to be the largest. So after a
// scan of its rows each CTA posts its kTop largest pixels and a bound on all
// its others, the CTAs meet once, and then every CTA plays the following
// iterations through on the posted pixels alone: their values are updated with
// the same operations in the same order as in the image, and the bound grows
// by what a subtraction can at most add to a pixel (|f| times the beam's most
// negative value, rounded up). While the largest posted value stays above the
// bound it is the image's largest, and the next component; once it does not,
// or after kBatch components, the CTAs subtract the batch from their rows, in
// order, and scan again. Components, fluxes and image are those of the one-by-
// one clean bit for bit; the image's rows are read and written once per batch.
constexpr int kHogThreads = 1024;
constexpr int kHogWarps = kHogThreads / 32;
constexpr int kMaxHogCtas = 256;   // grid cap of the persistent clean
constexpr int kTop = 8;            // pixels a CTA posts
constexpr int kWarpTop = 4;        // of them at most from one warp
constexpr int kBatch = 64;         // components per synchronisation at most
constexpr int kPerThread = kMaxHogCtas * kTop / kHogThreads;   // posted pixels a thread plays
// Polls of the grid barrier before a CTA gives up: each poll is a round trip
// to L2 and a 40 ns sleep, so the limit is of the order of a second (a healthy
// barrier completes within microseconds).
constexpr uint32_t kGridSpinLimit = 1u << 20;

// The CTAs' meeting place. Posts alternate between two sets: a CTA writes set
// e + 2 over e only after the meeting e + 1, which everyone joins after
// reading all of e.
struct HogSync {
    unsigned int count;                              // arrivals, over all meetings
    int abort;                                       // 1 once a CTA gave up waiting
    float beam[kMaxHogCtas][2];                      // largest -psf and psf of a CTA's share
    float bound[2][kMaxHogCtas];
    unsigned long long key[2][kMaxHogCtas][kTop];
};

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ float unordered(unsigned int o)
{
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);   // inverse of ordered()
}

// Key of a value at a pixel: larger values first, then lower pixels. 0: none.
__device__ __forceinline__ unsigned long long pixel_key(float v, unsigned int pixel)
{
    return (static_cast<unsigned long long>(ordered(v)) << 32) | (0xffffffffu - pixel);
}
__device__ __forceinline__ unsigned int key_pixel(unsigned long long key)
{
    return 0xffffffffu - static_cast<unsigned int>(key);
}
__device__ __forceinline__ float key_value(unsigned long long key)
{
    return unordered(static_cast<unsigned int>(key >> 32));   // no key: NaN
}

// The largest key of a warp, in every lane.
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key)
{
    const unsigned int hi = static_cast<unsigned int>(key >> 32);
    const unsigned int mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned int ml = __reduce_max_sync(0xffffffffu, hi == mh ? static_cast<unsigned int>(key) : 0u);
    return (static_cast<unsigned long long>(mh) << 32) | ml;
}

// One thread of every CTA of a cooperative launch (all resident), its CTA's
// writes made visible to it by a CTA barrier: counts itself in (release) and
// waits (acquire) until `target` arrivals are in, over all meetings so far;
// false when this CTA gave up waiting or another CTA had.
__device__ bool grid_meet(HogSync* sy, unsigned int target, uint32_t limit = kGridSpinLimit)
{
    __threadfence();
    atomicAdd(&sy->count, 1u);
    for (uint32_t polls = 0; static_cast<int>(ld_acquire_u32(&sy->count) - target) < 0; ++polls) {
        if (*reinterpret_cast<volatile int*>(&sy->abort) || polls >= limit) {
            atomicExch(&sy->abort, 1);
            return false;
        }
        __nanosleep(40);
    }
    __threadfence();
    return true;
}

// A meeting that never completes: one arrival more than the grid makes.
__global__ void k_selftest_grid_barrier(HogSync* sy, uint32_t limit, int* status)
{
    if (threadIdx.x == 0 && !grid_meet(sy, gridDim.x + 1, limit)) record_status(status, WT_ERR_TIMEOUT);
}

// CTA b owns image rows b, b + G, b + 2G, ... (G = gridDim.x <= n), held in
// shared memory as local rows 0, 1, 2, ... for the whole clean; one CTA per SM.
// A warp takes segments of 128 pixels of a row (every 32nd of the CTA's
// row-major list of them), a lane the pixels lane, lane + 32, ...: the beam,
// shifted by any number of pixels, is read in whole lines. The beam comes from
// L2, four bytes per pixel and component, which bounds large images; playing a
// component (a CTA-wide maximum and a gather of the beam) bounds small ones.
// Microseconds a component, one component per meeting before -> now: 64 x 64
// 3.2 -> 1.2, 512 x 512 3.9 -> 1.7, 1024 x 1024 4.1 -> 2.0, 2048 x 2048 6.5 ->
// 3.5 (noise, little to batch); a 2048 x 2048 field of 300 sources 6.7 -> 3.3.
__global__ void __launch_bounds__(kHogThreads, 1) k_hogbom_persistent(float* __restrict__ img,
                                                                     const float* __restrict__ psf, int n, float gain,
                                                                     float threshold, int max_iter,
                                                                     HogSync* __restrict__ sy,
                                                                     int* __restrict__ comp_pix,
                                                                     float* __restrict__ comp_flux,
                                                                     int* __restrict__ n_comp, int* status)
{
    extern __shared__ __align__(16) float rows[];
    __shared__ unsigned long long wkey[2][kHogWarps * kWarpTop];
    __shared__ unsigned int wbound[kHogWarps];
    __shared__ int b_oy[kBatch], b_ox[kBatch];   // the beam's row and column over image pixel (0, 0)
    __shared__ float b_f[kBatch];
    __shared__ bool gave_up;
    const int G = gridDim.x, b = blockIdx.x, c = n / 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nloc = (n - 1 - b) / G + 1;
    const int segs = (n + 127) / 128, items = segs * nloc;
    float neg = 0.0f, pos = 0.0f;                // the beam's largest -psf and psf, at least 0 (NaN aside)
    for (int r = 0; r < nloc; ++r)
        for (int x = tid; x < n; x += kHogThreads) {
            const int64_t q = static_cast<int64_t>(b + r * G) * n + x;
            rows[r * n + x] = __ldcg(img + q);
            const float p = __ldg(psf + q);
            neg = fmaxf(neg, -p);
            pos = fmaxf(pos, p);
        }
    // non-negative floats order as their bits
    wkey[0][warp] = (static_cast<unsigned long long>(__reduce_max_sync(0xffffffffu, __float_as_uint(neg))) << 32) |
                    __reduce_max_sync(0xffffffffu, __float_as_uint(pos));
    __syncthreads();
    if (tid == 0) {
        unsigned int hn = 0, hp = 0;
        for (int w = 0; w < kHogWarps; ++w) {
            hn = max(hn, static_cast<unsigned int>(wkey[0][w] >> 32));
            hp = max(hp, static_cast<unsigned int>(wkey[0][w]));
        }
        sy->beam[b][0] = __uint_as_float(hn);
        sy->beam[b][1] = __uint_as_float(hp);
    }
    __syncthreads();

    int m = 0, it = 0;                           // components of the batch, and in all
    bool finished = false;
    for (unsigned int epoch = 0;; ++epoch) {
        // ---- the batch off the rows; the thread's largest pixel and the
        // largest of its others (pixels in increasing order: a strict
        // comparison keeps the first of equals)
        float b1 = -INFINITY, b2 = -INFINITY;
        unsigned int bq = 0xffffffffu;
        for (int item = warp; item < items; item += kHogWarps) {
            const int r = item / segs, xs = (item - r * segs) * 128;
            const int row = b + r * G;
            float* px = rows + r * n + xs + lane;
            float v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = xs + lane + 32 * j < n ? px[32 * j] : 0.0f;
            for (int i0 = 0; i0 < m; i0 += 4) {
                float bm[4][4];
                bool in[4];
                bool whole = xs + 128 <= n;      // every pixel of the segment under every beam of the four
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int by = row + b_oy[i0 + i], bx = xs + b_ox[i0 + i];   // past m: rows off the beam
                    in[i] = by >= 0 && by < n;
                    whole = whole && (!in[i] || (bx >= 0 && bx + 128 <= n));
                }
                if (whole) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float* p = psf + static_cast<int64_t>(in[i] ? row + b_oy[i0 + i] : 0) * n +
                                         (in[i] ? xs + b_ox[i0 + i] : 0) + lane;
#pragma unroll
                        for (int j = 0; j < 4; ++j) bm[i][j] = __ldg(p + 32 * j);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (!in[i]) continue;
                        const float f = b_f[i0 + i];
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = __fsub_rn(v[j], __fmul_rn(f, bm[i][j]));
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (!in[i]) continue;
                        const float* p = psf + static_cast<int64_t>(row + b_oy[i0 + i]) * n;
                        const float f = b_f[i0 + i];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int x = xs + lane + 32 * j, bx = x + b_ox[i0 + i];
                            if (x < n && bx >= 0 && bx < n) v[j] = __fsub_rn(v[j], __fmul_rn(f, __ldg(p + bx)));
                        }
                    }
                }
            }
            const unsigned int q0 = static_cast<unsigned int>(row) * static_cast<unsigned int>(n) + xs + lane;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (xs + lane + 32 * j >= n) continue;
                if (m > 0) px[32 * j] = v[j];
                if (v[j] > b1) {
                    b2 = b1;
                    b1 = v[j];
                    bq = q0 + 32 * j;
                } else {
                    b2 = fmaxf(b2, v[j]);
                }
            }
        }
        if (finished) break;

        // ---- the CTA's kTop largest of the threads' pixels, at most kWarpTop
        // from a warp, and the bound on all the others
        {
            unsigned long long key = bq == 0xffffffffu ? 0ull : pixel_key(b1, bq);
            float rest = b2;
#pragma unroll
            for (int k = 0; k < kWarpTop; ++k) {
                const unsigned long long top = warp_max_key(key);
                if (lane == 0) wkey[0][warp * kWarpTop + k] = top;
                if (key == top) key = 0ull;      // keys are distinct, but for none
            }
            if (key != 0ull) rest = fmaxf(rest, key_value(key));
            const unsigned int o = __reduce_max_sync(0xffffffffu, ordered(rest));
            if (lane == 0) wbound[warp] = o;
        }
        __syncthreads();
        if (warp == 0) {
            // a lane's keys are a warp's, in decreasing order
            const unsigned long long* mine = wkey[0] + lane * kWarpTop;
            int taken = 0;
            unsigned long long out = 0ull;
#pragma unroll
            for (int k = 0; k < kTop; ++k) {
                const unsigned long long head = taken < kWarpTop ? mine[taken] : 0ull;
                const unsigned long long top = warp_max_key(head);
                if (head == top && head != 0ull) ++taken;
                if (lane == k) out = top;
            }
            unsigned int o = wbound[lane];
            if (taken < kWarpTop && mine[taken] != 0ull)
                o = max(o, static_cast<unsigned int>(mine[taken] >> 32));
            o = __reduce_max_sync(0xffffffffu, o);
            if (lane < kTop) __stcg(&sy->key[epoch & 1][b][lane], out);
            if (lane == 0) __stcg(&sy->bound[epoch & 1][b], unordered(o));
            __syncwarp();
            if (lane == 0) {
                const bool ok = grid_meet(sy, (epoch + 1) * static_cast<unsigned int>(G));
                if (!ok) record_status(status, WT_ERR_TIMEOUT);
                gave_up = !ok;
            }
        }
        __syncthreads();
        if (gave_up) return;   // every CTA leaves

        // ---- the posted pixels of this thread, and the bound on all others
        float pv[kPerThread];
        int py[kPerThread], px[kPerThread];
        float lim = -INFINITY;
        for (int g = lane; g < G; g += 32) lim = fmaxf(lim, __ldcg(&sy->bound[epoch & 1][g]));
        lim = unordered(__reduce_max_sync(0xffffffffu, ordered(lim)));
        if (epoch == 0) {
            for (int g = lane; g < G; g += 32) {
                neg = fmaxf(neg, __ldcg(&sy->beam[g][0]));
                pos = fmaxf(pos, __ldcg(&sy->beam[g][1]));
            }
            neg = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(neg)));
            pos = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(pos)));
        }
#pragma unroll
        for (int i = 0; i < kPerThread; ++i) {
            const int k = tid + i * kHogThreads;
            const unsigned long long key = k < G * kTop ? __ldcg(&sy->key[epoch & 1][0][0] + k) : 0ull;
            pv[i] = key_value(key);              // NaN: none
            const int q = key ? static_cast<int>(key_pixel(key)) : 0;
            py[i] = q / n;
            px[i] = q - py[i] * n;
        }

        // ---- the iterations that are certain
        for (m = 0; m < kBatch;) {
            unsigned long long key = 0ull;
#pragma unroll
            for (int i = 0; i < kPerThread; ++i)
                if (pv[i] > -INFINITY) {
                    const unsigned long long k = pixel_key(pv[i], static_cast<unsigned int>(py[i] * n + px[i]));
                    key = k > key ? k : key;
                }
            key = warp_max_key(key);
            if (lane == 0) wkey[m & 1][warp] = key;
            __syncthreads();
            key = warp_max_key(wkey[m & 1][lane]);
            const float peak = key_value(key);
            if (m > 0 && !(peak > lim)) break;   // another pixel may be larger
            if (it >= max_iter || !(peak >= threshold)) {
                finished = true;
                break;
            }
            const int q = static_cast<int>(key_pixel(key));
            const int oy = c - q / n, ox = c - (q - q / n * n);
            const float f = __fmul_rn(gain, peak);
            if (tid == 0) {
                b_oy[m] = oy;
                b_ox[m] = ox;
                b_f[m] = f;
                if (b == 0) {
                    comp_pix[it] = q;
                    comp_flux[it] = f;
                }
            }
#pragma unroll
            for (int i = 0; i < kPerThread; ++i) {
                const int by = py[i] + oy, bx = px[i] + ox;
                if (pv[i] > -INFINITY && by >= 0 && by < n && bx >= 0 && bx < n)
                    pv[i] = __fsub_rn(pv[i], __fmul_rn(f, __ldg(psf + static_cast<int64_t>(by) * n + bx)));
            }
            lim = f >= 0.0f ? __fadd_ru(lim, __fmul_ru(f, neg)) : __fadd_ru(lim, __fmul_ru(-f, pos));
            ++m;
            ++it;
        }
        __syncthreads();                         // the batch's list, and the keys' last readers
        if (finished && m == 0) break;
        if (tid < ((m + 3) & ~3) - m) b_oy[m + tid] = 2 * n;   // a last group of four filled up with beams off every row
        __syncthreads();
    }
    __syncthreads();
    for (int r = 0; r < nloc; ++r)
        for (int x = tid; x < n; x += kHogThreads) img[static_cast<int64_t>(b + r * G) * n + x] = rows[r * n + x];
    if (b == 0 && tid == 0) *n_comp = it;
}

// ---------------------------------------------------------------- components
// (l, m, flux) in float64 of recorded components [from, to).
__global__ void k_components_lm(const int* __restrict__ pix, const float* __restrict__ flux, int from, int to, int n,
                                double dl, double* __restrict__ l, double* __restrict__ m, double* __restrict__ f)
{
    const int i = from + static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= to) return;
    const int p = pix[i];
    l[i] = static_cast<double>(p % n - n / 2) * dl;
    m[i] = static_cast<double>(p / n - n / 2) * dl;
    f[i] = static_cast<double>(flux[i]);
}

// CTAs for the row loops: one row per CTA step, at most 8 CTAs per SM.
int rows_blocks(int n)
{
    const int cap = num_sms() * 8;
    return n < cap ? n : cap;
}

}  // namespace

// Dirty image (or beam) into `image`, with `grid` (n x n complex64) as
// scratch and `count` (one unsigned long long) as the entry counter.
int dirty_image(const double* uvw, const float2* vis, int64_t n_vis, int n, double dl, float* image, float2* grid,
                unsigned long long* count, cudaStream_t s)
{
    const int64_t nn = static_cast<int64_t>(n) * n;
    WT_CUDA_TRY(cudaMemsetAsync(grid, 0, static_cast<size_t>(nn) * sizeof(float2), s));
    WT_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(unsigned long long), s));
    if (n_vis > 0) {
        const double inv_du = static_cast<double>(n) * dl;   // 1 / du
        k_grid_nn<<<static_cast<unsigned>((n_vis + kImgThreads - 1) / kImgThreads), kImgThreads, 0, s>>>(
            uvw, vis, n_vis, n, inv_du, grid, count);
        WT_CUDA_TRY(cudaGetLastError());
    }
    int rc = fft2_forward(grid, n, s);
    if (rc) return rc;
    k_image_from_fft<<<rows_blocks(n), kImgThreads, 0, s>>>(grid, n, count, image);
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

// Hogbom clean of `image` in place; components appended to comp_pix /
// comp_flux (device, capacity max_iter), their count in *n_comp (device).
// `state` is a device HogbomState, reset here.
namespace {

size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

// CTAs and shared-memory bytes of a persistent clean of an n x n image, or 0
// CTAs when the schedule does not apply (rows too large for shared memory,
// no cooperative launch, or WT_HOGBOM=launches in the environment).
int persistent_grid(int n, size_t* smem)
{
    const char* e = getenv("WT_HOGBOM");
    if (e && strcmp(e, "launches") == 0) return 0;
    int dev = 0, coop = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return 0;
    }
    const int sms = num_sms();
    const int G = std::min(std::min(n, sms), kMaxHogCtas);
    const size_t bytes = static_cast<size_t>((n + G - 1) / G) * n * sizeof(float);
    cudaFuncAttributes fa;
    int occ = 0;
    if (cudaFuncGetAttributes(&fa, k_hogbom_persistent) != cudaSuccess ||
        bytes + fa.sharedSizeBytes > static_cast<size_t>(optin) ||
        // (the same limit from every thread: allow_dynamic_smem)
        cudaFuncSetAttribute(k_hogbom_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - static_cast<int>(fa.sharedSizeBytes)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_hogbom_persistent, kHogThreads, bytes) != cudaSuccess ||
        static_cast<int64_t>(occ) * sms < G) {
        cudaGetLastError();
        return 0;
    }
    *smem = bytes;
    return G;
}

int launch_persistent(int G, size_t smem, float* image, const float* psf, int n, float gain, float threshold,
                      int max_iter, HogSync* sy, int* comp_pix, float* comp_flux, int* n_comp, cudaStream_t s)
{
    int* status = device_status_word();
    if (!status) return set_error(WT_ERR_CUDA, "wt_hogbom: no device status word");
    WT_CUDA_TRY(cudaMemsetAsync(sy, 0, offsetof(HogSync, beam), s));
    void* args[] = {&image, &psf, &n, &gain, &threshold, &max_iter, &sy, &comp_pix, &comp_flux, &n_comp, &status};
    WT_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_hogbom_persistent), dim3(G),
                                            dim3(kHogThreads), args, smem, s));
    return WT_OK;
}

}  // namespace

int hogbom(float* image, const float* psf, int n, float gain, float threshold, int max_iter, int* comp_pix,
           float* comp_flux, int* n_comp, void* state, cudaStream_t s)
{
    HogSync* sy = reinterpret_cast<HogSync*>(static_cast<char*>(state) + round256(sizeof(HogbomState)));
    size_t smem = 0;
    const int G = persistent_grid(n, &smem);
    if (G > 0)
        return launch_persistent(G, smem, image, psf, n, gain, threshold, max_iter, sy, comp_pix, comp_flux, n_comp, s);
    k_hogbom_reset<<<1, 1, 0, s>>>(static_cast<HogbomState*>(state), n_comp);
    const int blocks = rows_blocks(n);
    // max_iter + 1 launches: the last subtracts the last component and stops
    for (int it = 0; it <= max_iter; ++it) {
        k_hogbom_step<<<blocks, kImgThreads, 0, s>>>(image, psf, n, gain, threshold, max_iter,
                                                     static_cast<HogbomState*>(state), comp_pix, comp_flux, n_comp);
    }
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

size_t hogbom_state_bytes() { return round256(sizeof(HogbomState)) + sizeof(HogSync); }

int components_lm(const int* pix, const float* flux, int from, int to, int n, double dl, double* l, double* m,
                  double* f, cudaStream_t s)
{
    if (to <= from) return WT_OK;
    const int cnt = to - from;
    k_components_lm<<<(cnt + 127) / 128, 128, 0, s>>>(pix, flux, from, to, n, dl, l, m, f);
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

}  // namespace wt

// ===========================================================================
// C entry points (declared in include/wtvis.h)
// ===========================================================================
namespace {

int check_image_args(const char* fn, int n, double dl)
{
    using namespace wt;
    if (n < 2 || n > 16384 || (n & 1)) return set_error(WT_ERR_ARG, "%s: n = %d must be even, 2..16384", fn, n);
    if (!(dl > 0.0) || !isfinite(dl)) return set_error(WT_ERR_RANGE, "%s: pixel size must be positive", fn);
    return WT_OK;
}

}  // namespace

extern "C" int wt_dirty_image(const double* uvw, const void* vis, int64_t n_vis, int n, double dl, float* image,
                              void* stream)
{
    using namespace wt;
    const char* fn = "wt_dirty_image";
    int rc = check_image_args(fn, n, dl);
    if (rc) return rc;
    if (n_vis < 0) return set_error(WT_ERR_ARG, "%s: n_vis < 0", fn);
    const size_t nn = static_cast<size_t>(n) * n;
    if ((rc = check_device_buffer(uvw, static_cast<size_t>(n_vis) * 24, fn, "uvw", 8)) ||
        (vis && (rc = check_device_buffer(vis, static_cast<size_t>(n_vis) * 8, fn, "vis", 8))) ||
        (rc = check_device_buffer(image, nn * 4, fn, "image", 4)))
        return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void* scratch = nullptr;
    const size_t bytes = nn * sizeof(float2) + 256;
    cudaError_t e = cudaMallocAsync(&scratch, bytes, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(WT_ERR_NOMEM, "%s: scratch allocation of %zu bytes failed", fn, bytes);
    }
    float2* grid = static_cast<float2*>(scratch);
    unsigned long long* count = reinterpret_cast<unsigned long long*>(static_cast<char*>(scratch) + nn * sizeof(float2));
    rc = dirty_image(uvw, static_cast<const float2*>(vis), n_vis, n, dl, image, grid, count, s);
    const cudaError_t ef = cudaFreeAsync(scratch, s);
    if (rc) return rc;
    if (ef != cudaSuccess) return cuda_error(ef, "cudaFreeAsync");
    return WT_OK;
}

namespace wt {
namespace {

// The largest |w| of the visibilities as float64 bits (non-negative doubles
// order as their bits); *out zeroed before the launch. One atomic per CTA of
// 256 threads, at most four CTAs per SM (an atomic per warp of a thread per
// visibility: 28 us against 10 for 1 008 000).
__global__ void __launch_bounds__(256) k_max_abs_w(const double* __restrict__ uvw, int64_t n_vis, unsigned long long* __restrict__ out)
{
    unsigned long long m = 0;
#pragma unroll 4
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_vis;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const double w = fabs(uvw[3 * i + 2]);
        if (isfinite(w)) {
            const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(w));
            m = b > m ? b : m;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, m, o);
        m = other > m ? other : m;
    }
    __shared__ unsigned long long wm[8];
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) m = wm[i] > m ? wm[i] : m;
        if (m) atomicMax(out, m);
    }
}

// The batch's largest finite |w| (1 if none is above 0); synchronises s.
int max_abs_w(const double* uvw, int64_t n_vis, cudaStream_t s, double* out)
{
    unsigned long long* d = nullptr;
    WT_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void**>(&d), sizeof(unsigned long long), s));
    unsigned long long h = 0;
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof(unsigned long long), s);
    if (e == cudaSuccess && n_vis > 0) {
        int64_t b = (n_vis + 255) / 256;
        if (b > 4 * num_sms()) b = 4 * num_sms();
        k_max_abs_w<<<static_cast<unsigned>(b), 256, 0, s>>>(uvw, n_vis, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(d, s);
    if (e != cudaSuccess) return cuda_error(e, "the largest |w|");
    double wm;
    memcpy(&wm, &h, sizeof(wm));
    *out = wm > 0.0 ? wm : 1.0;
    return WT_OK;
}

int dirty_image_w(const double* uvw, const float2* vis, int64_t n_vis, int n, double dl, int planes, double w_max,
                  float* image, cudaStream_t s)
{
    const char* fn = "wt_dirty_image_w";
    const double ndl = n * dl;
    if (!(ndl * ndl < 1.0)) return set_error(WT_ERR_RANGE, "%s: the field (n dl = %g) must lie inside l^2 + m^2 < 1", fn, ndl);
    const int64_t nn = static_cast<int64_t>(n) * n;
    if (w_max <= 0.0) {   // the batch's own largest |w|
        const int rc = max_abs_w(uvw, n_vis, s, &w_max);
        if (rc) return rc;
    }
    WpPlan pl;
    pl.P = planes;
    pl.dw = w_max / (planes - 1);
    pl.ndl = ndl;
    // the largest chirp frequency of the field in cells: w (n dl)^2 / (2 n) at its corner
    const double n_min = sqrt(1.0 - 0.5 * ndl * ndl);
    pl.xc_per_w = ndl * ndl / (2.0 * n_min);
    const double xc = w_max * pl.xc_per_w;
    pl.h = static_cast<int>(ceil(0.5 * kWpWidth + xc)) + 1;
    if (pl.h > kWpMaxHalf)
        return set_error(WT_ERR_RANGE, "%s: w up to %g needs a kernel half-width of %d cells (at most %d)", fn, w_max,
                         pl.h, kWpMaxHalf);
    if (2 * pl.h + 2 >= n / 2) return set_error(WT_ERR_RANGE, "%s: a %d-cell kernel does not fit an n = %d grid", fn,
                                                2 * pl.h + 1, n);
    pl.S = 2 * pl.h + 1;
    pl.T = pl.S * kWpOversample + 1;
    constexpr int H = kWpHalf, O = kWpOversample;
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t b_grid = up(nn * sizeof(float2)), b_cnt = 256;
    const size_t b_tw = up(static_cast<size_t>(pl.T) * H * sizeof(float2));
    const size_t b_ft = up(H * sizeof(double)), b_gc = up(static_cast<size_t>(n) * sizeof(F2));
    const size_t b_f = up(static_cast<size_t>(planes) * H * H * sizeof(float2));
    const size_t b_a = up(static_cast<size_t>(planes) * H * pl.T * sizeof(float2));
    const size_t b_k = up(static_cast<size_t>(planes) * O * O * (pl.S + 1) * (pl.S + 1) * sizeof(float2));
    char* scratch = nullptr;
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&scratch),
                                    b_grid + b_cnt + b_tw + b_ft + b_gc + b_f + b_a + b_k, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(WT_ERR_NOMEM, "%s: scratch allocation failed: %s", fn, cudaGetErrorString(e));
    }
    char* at = scratch;
    auto take = [&](size_t b) {
        char* r = at;
        at += b;
        return r;
    };
    float2* grid = reinterpret_cast<float2*>(take(b_grid));
    unsigned long long* count = reinterpret_cast<unsigned long long*>(take(b_cnt));
    float2* tw = reinterpret_cast<float2*>(take(b_tw));
    double* ft = reinterpret_cast<double*>(take(b_ft));
    F2* gc = reinterpret_cast<F2*>(take(b_gc));
    float2* f = reinterpret_cast<float2*>(take(b_f));
    float2* a = reinterpret_cast<float2*>(take(b_a));
    float2* K = reinterpret_cast<float2*>(take(b_k));
    int rc = WT_OK;
    const int pairs = (pl.T + 1) / 2, turns = (pairs + 255) / 256;
    const int tj = ((pairs + turns - 1) / turns + 31) / 32 * 32;   // a thread per two table points
    k_wp_tables<<<(pl.T * H + H + n + 127) / 128, 128, 0, s>>>(pl, n, tw, ft, gc);
    k_wp_field<<<dim3((H * H + 127) / 128, (planes + kWpFieldPlanes - 1) / kWpFieldPlanes), 128, 0, s>>>(pl, ft, f);
    k_wp_stage1<<<dim3(planes, H / kWpGroup), tj, 0, s>>>(pl, f, tw, a);
    k_wp_stage2<<<dim3(planes, (pl.T + kWpGroup - 1) / kWpGroup), tj, 0, s>>>(pl, a, tw, K);
    if (cudaGetLastError() != cudaSuccess) rc = set_error(WT_ERR_CUDA, "%s: kernel tables", fn);
    if (rc == WT_OK && (cudaMemsetAsync(grid, 0, static_cast<size_t>(nn) * sizeof(float2), s) != cudaSuccess ||
                        cudaMemsetAsync(count, 0, sizeof(unsigned long long), s) != cudaSuccess))
        rc = set_error(WT_ERR_CUDA, "%s: clearing the grid", fn);
    if (rc == WT_OK && n_vis > 0) {
        // 8 warps per CTA; a warp per visibility up to 256 warps per SM
        const int64_t b = std::min<int64_t>((n_vis + 7) / 8, static_cast<int64_t>(num_sms()) * 32);
        k_grid_wproj<<<static_cast<unsigned>(b), 256, 0, s>>>(pl, K, uvw, vis, n_vis, n, ndl, grid, count);
        if (cudaGetLastError() != cudaSuccess) rc = set_error(WT_ERR_CUDA, "%s: gridding launch", fn);
    }
    if (rc == WT_OK) rc = fft2_forward(grid, n, s);
    if (rc == WT_OK) {
        k_image_from_fft_wp<<<rows_blocks(n), kImgThreads, 0, s>>>(grid, n, count, gc, image);
        if (cudaGetLastError() != cudaSuccess) rc = set_error(WT_ERR_CUDA, "%s: image launch", fn);
    }
    const cudaError_t ef = cudaFreeAsync(scratch, s);
    if (rc) return rc;
    if (ef != cudaSuccess) return cuda_error(ef, "cudaFreeAsync");
    return WT_OK;
}

}  // namespace
}  // namespace wt

extern "C" int wt_dirty_image_w(const double* uvw, const void* vis, int64_t n_vis, int n, double dl, int w_planes,
                                double w_max, float* image, void* stream)
{
    using namespace wt;
    const char* fn = "wt_dirty_image_w";
    int rc = check_image_args(fn, n, dl);
    if (rc) return rc;
    if (n_vis < 0) return set_error(WT_ERR_ARG, "%s: n_vis < 0", fn);
    if (w_planes < 2 || w_planes > 1024) return set_error(WT_ERR_ARG, "%s: w_planes = %d must be 2..1024", fn, w_planes);
    if (!(w_max >= 0.0) || !isfinite(w_max)) return set_error(WT_ERR_ARG, "%s: w_max must be finite and >= 0", fn);
    const size_t nn = static_cast<size_t>(n) * n;
    if ((rc = check_device_buffer(uvw, static_cast<size_t>(n_vis) * 24, fn, "uvw", 8)) ||
        (vis && (rc = check_device_buffer(vis, static_cast<size_t>(n_vis) * 8, fn, "vis", 8))) ||
        (rc = check_device_buffer(image, nn * 4, fn, "image", 4)))
        return rc;
    return dirty_image_w(uvw, static_cast<const float2*>(vis), n_vis, n, dl, w_planes, w_max, image,
                         static_cast<cudaStream_t>(stream));
}

extern "C" int wt_selftest_grid_barrier(uint32_t spin_limit, void* stream)
{
    using namespace wt;
    const char* fn = "wt_selftest_grid_barrier";
    if (spin_limit < 1 || spin_limit > 65536) return set_error(WT_ERR_ARG, "%s: spin_limit must be in 1..65536", fn);
    int dev = 0, coop = 0;
    WT_CUDA_TRY(cudaGetDevice(&dev));
    WT_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return set_error(WT_ERR_UNSUPPORTED, "%s: no cooperative launch on this device", fn);
    int* status = device_status_word();
    if (!status) return set_error(WT_ERR_CUDA, "%s: no device status word", fn);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    HogSync* sy = nullptr;
    WT_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void**>(&sy), sizeof(HogSync), s));
    int rc = WT_OK;
    cudaError_t e = cudaMemsetAsync(sy, 0, sizeof(HogSync), s);
    if (e == cudaSuccess) {
        void* args[] = {&sy, &spin_limit, &status};
        e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_selftest_grid_barrier), dim3(2), dim3(32),
                                        args, 0, s);
    }
    if (e != cudaSuccess) rc = cuda_error(e, fn);
    const cudaError_t ef = cudaFreeAsync(sy, s);
    if (!rc && ef != cudaSuccess) rc = cuda_error(ef, "cudaFreeAsync");
    return rc;
}

extern "C" int wt_hogbom(float* image, const float* psf, int n, float gain, float threshold, int max_iter,
                         int* comp_pix, float* comp_flux, int* n_comp, void* stream)
{
    using namespace wt;
    const char* fn = "wt_hogbom";
    if (n < 2 || n > 16384 || (n & 1)) return set_error(WT_ERR_ARG, "%s: n = %d must be even, 2..16384", fn, n);
    if (max_iter < 0 || max_iter > (1 << 24)) return set_error(WT_ERR_ARG, "%s: max_iter outside 0..2^24", fn);
    if (!(gain > 0.0f) || !(gain <= 1.0f)) return set_error(WT_ERR_RANGE, "%s: gain must be in (0, 1]", fn);
    if (!isfinite(threshold)) return set_error(WT_ERR_RANGE, "%s: threshold must be finite", fn);
    const size_t nn = static_cast<size_t>(n) * n;
    int rc;
    if ((rc = check_device_buffer(image, nn * 4, fn, "image", 4)) || (rc = check_device_buffer(psf, nn * 4, fn, "psf", 4)) ||
        (rc = check_device_buffer(n_comp, 4, fn, "n_comp", 4)) ||
        (max_iter > 0 && ((rc = check_device_buffer(comp_pix, static_cast<size_t>(max_iter) * 4, fn, "comp_pix", 4)) ||
                          (rc = check_device_buffer(comp_flux, static_cast<size_t>(max_iter) * 4, fn, "comp_flux", 4)))))
        return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void* state = nullptr;
    cudaError_t e = cudaMallocAsync(&state, hogbom_state_bytes(), s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(WT_ERR_NOMEM, "%s: state allocation failed", fn);
    }
    rc = hogbom(image, psf, n, gain, threshold, max_iter, comp_pix, comp_flux, n_comp, state, s);
    const cudaError_t ef = cudaFreeAsync(state, s);
    if (rc) return rc;
    if (ef != cudaSuccess) return cuda_error(ef, "cudaFreeAsync");
    return WT_OK;
}

extern "C" int wt_clean(const double* uvw, const void* vis_obs, int64_t n_vis, int n, double dl, double ra0,
                        double dec0, int J, int predictor, int mode, float gain, float threshold, int minor_iter,
                        int n_major, int w_planes, int* comp_pix, float* comp_flux, int* n_comp, void* vis_resid,
                        float* image_resid, void* stream)
{
    using namespace wt;
    const char* fn = "wt_clean";
    int rc = check_image_args(fn, n, dl);
    if (rc) return rc;
    if (n_vis < 0) return set_error(WT_ERR_ARG, "%s: n_vis < 0", fn);
    if (predictor != WT_PREDICT_TREE && predictor != WT_PREDICT_DIRECT)
        return set_error(WT_ERR_ARG, "%s: bad predictor %d", fn, predictor);
    if (mode != WT_MIXED && mode != WT_MIXED_FAST && !(mode == WT_MIXED_TC && predictor == WT_PREDICT_DIRECT))
        return set_error(WT_ERR_ARG,
                         "%s: mode must be WT_MIXED or WT_MIXED_FAST (complex64 visibilities), or WT_MIXED_TC with "
                         "the direct-sum predictor", fn);
    if (minor_iter < 0 || n_major < 0 || static_cast<int64_t>(minor_iter) * n_major > (1 << 24))
        return set_error(WT_ERR_ARG, "%s: minor_iter x n_major outside 0..2^24", fn);
    if (!(gain > 0.0f) || !(gain <= 1.0f)) return set_error(WT_ERR_RANGE, "%s: gain must be in (0, 1]", fn);
    if (!isfinite(threshold)) return set_error(WT_ERR_RANGE, "%s: threshold must be finite", fn);
    if (w_planes != 0 && (w_planes < 2 || w_planes > 1024))
        return set_error(WT_ERR_ARG, "%s: w_planes = %d must be 0 or 2..1024", fn, w_planes);
    if (!n_comp) return set_error(WT_ERR_ARG, "%s: n_comp (host) is NULL", fn);
    const int cap = minor_iter * n_major;
    const size_t nn = static_cast<size_t>(n) * n;
    if ((rc = check_device_buffer(uvw, static_cast<size_t>(n_vis) * 24, fn, "uvw", 8)) ||
        (rc = check_device_buffer(vis_obs, static_cast<size_t>(n_vis) * 8, fn, "vis_obs", 8)) ||
        (rc = check_device_buffer(vis_resid, static_cast<size_t>(n_vis) * 8, fn, "vis_resid", 8)) ||
        (rc = check_device_buffer(image_resid, nn * 4, fn, "image_resid", 4)) ||
        (cap > 0 && ((rc = check_device_buffer(comp_pix, static_cast<size_t>(cap) * 4, fn, "comp_pix", 4)) ||
                     (rc = check_device_buffer(comp_flux, static_cast<size_t>(cap) * 4, fn, "comp_flux", 4)))))
        return rc;
    *n_comp = 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // scratch: grid, beam, model visibilities, component (l, m, flux), counters
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t c3 = static_cast<size_t>(cap > 0 ? cap : 1) * 8;
    const bool tree = predictor == WT_PREDICT_TREE;
    const size_t bytes = up(nn * 8) + up(nn * 4) + up(static_cast<size_t>(n_vis > 0 ? n_vis : 1) * 8) + 3 * up(c3) +
                         up(8) + up(hogbom_state_bytes()) + up(4) + (tree ? up(nn * 8) : 0);
    void* scratch = nullptr;
    cudaError_t e = cudaMallocAsync(&scratch, bytes, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(WT_ERR_NOMEM, "%s: scratch allocation of %zu bytes failed", fn, bytes);
    }
    char* q = static_cast<char*>(scratch);
    auto take = [&](size_t b) {
        char* r = q;
        q += up(b);
        return r;
    };
    float2* grid = reinterpret_cast<float2*>(take(nn * 8));
    float* beam = reinterpret_cast<float*>(take(nn * 4));
    float2* model = reinterpret_cast<float2*>(take(static_cast<size_t>(n_vis > 0 ? n_vis : 1) * 8));
    double* cl = reinterpret_cast<double*>(take(c3));
    double* cm = reinterpret_cast<double*>(take(c3));
    double* cf = reinterpret_cast<double*>(take(c3));
    unsigned long long* count = reinterpret_cast<unsigned long long*>(take(8));
    void* state = take(hogbom_state_bytes());
    int* d_found = reinterpret_cast<int*>(take(4));
    int64_t* xref = tree ? reinterpret_cast<int64_t*>(take(nn * 8)) : nullptr;

    int total = 0;
    // the imaging: nearest-cell without w, or w-projection planned for the
    // batch's largest |w| (found once)
    double w_max = 0.0;
    auto image_of = [&](const float2* v, float* out) {
        return w_planes ? dirty_image_w(uvw, v, n_vis, n, dl, w_planes, w_max, out, s)
                        : dirty_image(uvw, v, n_vis, n, dl, out, grid, count, s);
    };
    rc = w_planes ? max_abs_w(uvw, n_vis, s, &w_max) : WT_OK;
    // the tree predictor maps components through the cross-reference table
    // of the image pixels, built once (Sec. 3.5)
    if (!rc && tree) rc = wt_xref_table(n, dl, ra0, dec0, J, xref, stream);
    if (!rc) rc = image_of(nullptr, beam);
    if (!rc && n_vis > 0) {
        e = cudaMemcpyAsync(vis_resid, vis_obs, static_cast<size_t>(n_vis) * 8, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) rc = cuda_error(e, "cudaMemcpyAsync");
    }
    for (int cycle = 0; cycle < n_major && !rc; ++cycle) {
        // 3. gridding and FFT of the residuals, then the minor cycles
        if ((rc = image_of(static_cast<const float2*>(vis_resid), image_resid))) break;
        if ((rc = hogbom(image_resid, beam, n, gain, threshold, minor_iter, comp_pix + total, comp_flux + total, d_found,
                         state, s)))
            break;
        int found = 0;
        e = cudaMemcpyAsync(&found, d_found, sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            rc = cuda_error(e, "reading the component count");
            break;
        }
        if (found == 0) break;
        if ((rc = components_lm(comp_pix, comp_flux, total, total + found, n, dl, cl, cm, cf, s))) break;
        total += found;
        // 1. model visibilities from every component so far, 2. subtraction
        if (predictor == WT_PREDICT_TREE) {
            wt_tree t = nullptr;
            if ((rc = wt_build_tree_xref(xref, n, comp_pix, cf, total, ra0, dec0, J, &t, stream))) break;
            rc = wt_predict_vis(t, uvw, n_vis, model, mode, 1, WT_SUM_EQ17_REGROUPED, stream);
            wt_free_tree(t);
        } else {
            rc = dft_predict_vis(cl, cm, cf, total, uvw, n_vis, model, mode, 1, stream);
        }
        if (!rc) rc = subtract_model(vis_obs, model, vis_resid, n_vis, mode, stream);
    }
    // the dirty image of the final residual visibilities
    if (!rc) rc = image_of(static_cast<const float2*>(vis_resid), image_resid);
    *n_comp = total;
    const cudaError_t ef = cudaFreeAsync(scratch, s);
    if (rc) return rc;
    if (ef != cudaSuccess) return cuda_error(ef, "cudaFreeAsync");
    return WT_OK;
}
