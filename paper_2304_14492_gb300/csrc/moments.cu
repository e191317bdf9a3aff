// Moments (Eq. 1): bilinear polar resampling (Sec. 2.5) fused with a real FFT of
// every ring (the e^{-j m theta} factor), then the radial projection with the
// (n+1)/pi weight, and the Neumann factor of Eq. 14-15.
#include <cuda_bf16.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "ring_fft.cuh"
#include "zm_internal.cuh"

namespace zm {

int launch_projection_tc(zm_plan_t p, const float* F, int batch, float* out, unsigned flags, cudaStream_t st);

// ============================================================== K-b
constexpr int KB_MAX_IMG = 128;

struct KbParams {
    int n_rho, n_max, batch_total, b_off;
    int nb;                // images in this launch
    uint8_t* Fblk;         // bf16 hi / lo operand blocks of F (R = 8 or 4), or NULL
    size_t fblk_half;      // bytes of one half
    int n_chunks;          // 64-node chunks of the radial index
    const float* rho32;    // [n_rho]
    const float2* cs;      // [N] (cos theta_k, sin theta_k)
    const float2* tw;      // [N] e^{-2 pi i j / N}
    float* F;              // [n_max+1][batch_total][2][n_rho]
    float* fhat_out;       // [batch_total][n_rho][N] or NULL
    const float* fhat_in;  // [batch_total][n_rho][N] (polar input mode)
    int discard_in;        // fhat_in is the plan's scratch: its L2 lines are dropped once read
    int release;           // the next kernel may start early (k_ring_spectra)
    GeoImage img[KB_MAX_IMG];
};

// KB_TILED: polar samples that the tile resampler has just written (1024 angles)
enum { KB_GATHER = 0, KB_POLAR = 1, KB_RESAMPLE = 2, KB_TILED = 3 };

// Bilinear value at pixel coordinates (X, Y); neighbours outside the image are 0.
__device__ __forceinline__ float bilinear(const GeoImage& im, float X, float Y) {
    const float xf = floorf(X), yf = floorf(Y);
    const float fx = X - xf, fy = Y - yf;
    const int x0 = (int)fminf(fmaxf(xf, -2.f), (float)im.w + 1.f);
    const int y0 = (int)fminf(fmaxf(yf, -2.f), (float)im.h + 1.f);
    const float* d = im.data;
    const bool xa = (unsigned)x0 < (unsigned)im.w, xb = (unsigned)(x0 + 1) < (unsigned)im.w;
    const bool ya = (unsigned)y0 < (unsigned)im.h, yb = (unsigned)(y0 + 1) < (unsigned)im.h;
    const float* r0 = d + (long long)y0 * im.pitch;
    const float* r1 = r0 + im.pitch;
    const float p00 = (xa && ya) ? __ldg(r0 + x0) : 0.f;
    const float p01 = (xb && ya) ? __ldg(r0 + x0 + 1) : 0.f;
    const float p10 = (xa && yb) ? __ldg(r1 + x0) : 0.f;
    const float p11 = (xb && yb) ? __ldg(r1 + x0 + 1) : 0.f;
    const float top = fmaf(fx, p01 - p00, p00);
    const float bot = fmaf(fx, p11 - p10, p10);
    return fmaf(fy, bot - top, top);
}

// The same value, bit for bit, where the whole stencil is known to lie in an
// image of less than 2^31 elements and 2^22 columns and rows: the floor is a
// rounded-down addition of 2^23 (its low bits are the integer), one 32-bit
// offset addresses all four pixels, and nothing is clamped or tested (22
// instructions a sample where the general form takes about 50).
__device__ __forceinline__ float bilinear_inside(const float* d, int pitch, float X, float Y) {
    const float tx = __fadd_rd(X, 8388608.f), ty = __fadd_rd(Y, 8388608.f);
    const float fx = X - (tx - 8388608.f), fy = Y - (ty - 8388608.f);
    const int o = (__float_as_int(ty) - 0x4b000000) * pitch + (__float_as_int(tx) - 0x4b000000);
    const float* r0 = d + o;
    const float* r1 = r0 + pitch;
    const float p00 = __ldg(r0), p01 = __ldg(r0 + 1), p10 = __ldg(r1), p11 = __ldg(r1 + 1);
    const float top = fmaf(fx, p01 - p00, p00);
    const float bot = fmaf(fx, p11 - p10, p10);
    return fmaf(fy, bot - top, top);
}

// Every stencil of the ring of radius rad lies inside the image, with a pixel
// to spare for the rounding of the sample coordinates (below 2^22 they are off
// by less than that).
__device__ __forceinline__ bool ring_inside(const GeoImage& im, float rad) {
    return im.w < (1 << 22) && im.h < (1 << 22) && (long long)im.h * im.pitch < (1ll << 31) && im.cx - rad >= 1.f &&
           im.cx + rad <= (float)(im.w - 3) && im.cy - rad >= 1.f && im.cy + rad <= (float)(im.h - 3);
}

// One CTA = R consecutive rings of one image at a time, one warp per ring
// (R = blockDim/32); the grid is persistent and each CTA walks ring blocks
// (image, block) after loading the FFT twiddles once.
// Phase 1: each warp's samples straight into its FFT registers: bilinear gather
// (a lane takes the two angles of a packed point, so nothing passes through
// shared memory and no barrier separates the warps), or the polar input.  Phase
// 2: per warp, the N-point real FFT of its ring as an N/2-point complex FFT
// plus the split
//   F_m = (Z_m + conj Z_{M-m})/2 + e^{-2 pi i m/N} (Z_m - conj Z_{M-m})/(2i),
// for m = 0..n_max.  Phase 3: F[m][b][re/im][i0..i0+R) written as segments.
//
// Residency: four CTAs per SM up to 512 angles.  At 1024 the 64 registers that
// leaves cost the gather its loads in flight and, with 32 rings at once, its hits
// in L1: 8 images of 2161 x 2161 on 1024 x 1024 took 248 us, with two CTAs 67.
// So do a caller's polar samples (16 images of 1024 x 1024 samples 42.1 us a call
// with the projection, FP32; with four CTAs 44.6), but not what the tile resampler
// leaves: there the wider CTAs, launched while it runs, take its place (FP32 spectra
// of two 1024 x 1024 images on 1024 x 1024: 23.7 us a call, with four CTAs 17.5; from
// eight such images on two are ahead again, 41.2 and 43.3).
constexpr int kb_ctas(int logn, int mode) {
    return logn >= 11 || (logn == 10 && mode != KB_RESAMPLE && mode != KB_TILED) ? 2 : 4;
}
constexpr long long TILED_SAMPLES = 3ll << 21;    // calls of more samples take KB_POLAR after the tiles

template <int LOGN, int MODE>
__global__ void __launch_bounds__(256, kb_ctas(LOGN, MODE)) k_ring_spectra(const __grid_constant__ KbParams p) {
    using FFT = RingFFT<LOGN>;
    constexpr int N = FFT::N;
    constexpr int ROW = FFT::ROW_FLOATS;
    constexpr bool POLAR = MODE == KB_POLAR || MODE == KB_TILED;
    extern __shared__ __align__(16) float smem[];
    const int R = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_rho = p.n_rho;
    const int n_max = p.n_max;
    float* rings = smem;
    float* Fs = smem + R * ROW;                  // [2][n_max+1][R]
    float2* twt = reinterpret_cast<float2*>(smem + ((R * ROW + 2 * (n_max + 1) * R + 1) & ~1));
    float2* twm = twt + FFT::TW_FLOAT2;            // e^{-2 pi i m / N}, m <= n_max
    if (MODE != KB_RESAMPLE) {
        FFT::load_twiddles(twt, p.tw);
        for (int m = threadIdx.x; m <= n_max; m += blockDim.x) twm[m] = __ldg(&p.tw[m]);
    }
    // with operand blocks, ring blocks run up to the last 64-node chunk (rings
    // past n_rho are zero), so that every block of the chunk is written
    const int n_rb = p.Fblk ? p.n_chunks * (64 / R) : (n_rho + R - 1) / R;
    const int n_items = n_rb * p.nb;
    // polar input: this warp's ring of a ring block straight into the FFT
    // registers (lane t holds z[t + L s]); the next block's ring is loaded as
    // soon as the current FFT has left the registers
    float2 v[FFT::Q];
    auto load_ring = [&](int item) {
        const int bl = item / n_rb;
        const int i = (item - bl * n_rb) * R + warp;
        const bool live = lane < FFT::L && i < n_rho;
        const float* src = p.fhat_in + ((size_t)(p.b_off + bl) * n_rho + (live ? i : 0)) * N;
        if ((reinterpret_cast<uintptr_t>(p.fhat_in) & 7) == 0) {
            const float2* z = reinterpret_cast<const float2*>(src);
#pragma unroll
            for (int s = 0; s < FFT::Q; ++s) v[s] = live ? __ldg(&z[lane + FFT::L * s]) : make_float2(0.f, 0.f);
        } else {
#pragma unroll
            for (int s = 0; s < FFT::Q; ++s) {
                const int j = lane + FFT::L * s;
                v[s] = live ? make_float2(__ldg(src + 2 * j), __ldg(src + 2 * j + 1)) : make_float2(0.f, 0.f);
            }
        }
    };
    griddep_wait();                // the images or polar samples are written, the spectra are free
    if (p.release) griddep_launch();
    if (POLAR && (int)blockIdx.x < n_items) load_ring(blockIdx.x);
    bool ready = false;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int bl = item / n_rb;
        const int i0 = (item - bl * n_rb) * R;
        const int b = p.b_off + bl;
        if (MODE == KB_RESAMPLE) {
            const GeoImage im = p.img[bl];
#pragma unroll 4
            for (int idx = threadIdx.x; idx < R * N; idx += blockDim.x) {
                const int r = idx >> LOGN, k = idx & (N - 1);
                const int i = i0 + r;
                if (i < n_rho) {
                    const float rad = im.r * __ldg(&p.rho32[i]);
                    const float2 c = __ldg(&p.cs[k]);
                    p.fhat_out[((size_t)b * n_rho + i) * N + k] =
                        bilinear(im, fmaf(rad, c.x, im.cx), fmaf(-rad, c.y, im.cy));
                }
            }
            continue;
        }
        if (MODE == KB_GATHER) {
            const GeoImage& im = p.img[bl];
            const int i = i0 + warp;
#pragma unroll
            for (int s = 0; s < FFT::Q; ++s) v[s] = make_float2(0.f, 0.f);
            if (i < n_rho && lane < FFT::L) {
                const float rad = im.r * __ldg(&p.rho32[i]);
                const float4* cs2 = reinterpret_cast<const float4*>(p.cs);      // two angles
                if (ring_inside(im, rad)) {
                    const float* d = im.data;
                    const int pitch = (int)im.pitch;
                    const float cx = im.cx, cy = im.cy;
#pragma unroll
                    for (int s = 0; s < FFT::Q; ++s) {
                        const float4 c = __ldg(&cs2[lane + FFT::L * s]);
                        v[s].x = bilinear_inside(d, pitch, fmaf(rad, c.x, cx), fmaf(-rad, c.y, cy));
                        v[s].y = bilinear_inside(d, pitch, fmaf(rad, c.z, cx), fmaf(-rad, c.w, cy));
                    }
                } else {
#pragma unroll
                    for (int s = 0; s < FFT::Q; ++s) {
                        const float4 c = __ldg(&cs2[lane + FFT::L * s]);
                        v[s].x = bilinear(im, fmaf(rad, c.x, im.cx), fmaf(-rad, c.y, im.cy));
                        v[s].y = bilinear(im, fmaf(rad, c.z, im.cx), fmaf(-rad, c.w, im.cy));
                    }
                }
                if (p.fhat_out) {
                    float* dst = p.fhat_out + ((size_t)b * n_rho + i) * N;
#pragma unroll
                    for (int s = 0; s < FFT::Q; ++s) {
                        dst[2 * (lane + FFT::L * s)] = v[s].x;
                        dst[2 * (lane + FFT::L * s) + 1] = v[s].y;
                    }
                }
            }
        }
        if (!ready) {
            __syncthreads();                           // the twiddles
            ready = true;
        }

        {
            float* row = rings + warp * ROW;
            float2* X = reinterpret_cast<float2*>(row);
            FFT::fwd(v, lane, twt, X);                 // the row doubles as the transpose buffer
            if (lane < FFT::L) {
#pragma unroll
                for (int r = 0; r < FFT::Q; ++r) X[FFT::pad(FFT::fwd_index(r, lane))] = v[r];
            }
            __syncwarp();
            if (POLAR && item + (int)gridDim.x < n_items) load_ring(item + gridDim.x);
            for (int m = lane; m <= n_max; m += 32) {
                const float2 A = X[FFT::pad(m)];
                const float2 B = cconj(X[FFT::pad((FFT::M - m) & (FFT::M - 1))]);
                const float2 E = cscale(cadd(A, B), 0.5f);
                const float2 D = csub(A, B);
                const float2 O = make_float2(0.5f * D.y, -0.5f * D.x);
                const float2 Fm = cadd(E, cmul(twm[m], O));
                Fs[m * R + warp] = Fm.x;
                Fs[((n_max + 1) + m) * R + warp] = Fm.y;
            }
        }
        __syncthreads();
        const int nm1 = n_max + 1;
        if (p.Fblk) {
            // 8 rings = one 16-byte row per (m, re/im): bf16 hi and lo halves
            // (R = 4: half a row)
            const int ncol = 2 * p.batch_total;
            // (re and im of an order are the halves of one 32-byte sector:
            // adjacent threads, so that no sector is written in two pieces)
            for (int e = threadIdx.x; e < 2 * nm1; e += blockDim.x) {
                const int c = e & 1, m = e >> 1;
                const float* src = Fs + (size_t)(c * nm1 + m) * R;
                uint32_t h[4], l[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (2 * q >= R) break;
                    const __nv_bfloat16 h0 = __float2bfloat16_rn(src[2 * q]), h1 = __float2bfloat16_rn(src[2 * q + 1]);
                    const __nv_bfloat16 l0 = __float2bfloat16_rn(src[2 * q] - __bfloat162float(h0));
                    const __nv_bfloat16 l1 = __float2bfloat16_rn(src[2 * q + 1] - __bfloat162float(h1));
                    h[q] = __bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                    l[q] = __bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                }
                const size_t o = fblk_row(m, i0 & ~7, 2 * b + c, p.n_chunks, ncol) + 2 * (i0 & 7);
                if (R == 8) {
                    *reinterpret_cast<uint4*>(p.Fblk + o) = make_uint4(h[0], h[1], h[2], h[3]);
                    *reinterpret_cast<uint4*>(p.Fblk + p.fblk_half + o) = make_uint4(l[0], l[1], l[2], l[3]);
                } else {
                    *reinterpret_cast<uint2*>(p.Fblk + o) = make_uint2(h[0], h[1]);
                    *reinterpret_cast<uint2*>(p.Fblk + p.fblk_half + o) = make_uint2(l[0], l[1]);
                }
            }
        } else {
            const int lgR = __ffs(R) - 1;                 // R is a power of two
            const int tot = 2 * nm1 * R;
            for (int e = threadIdx.x; e < tot; e += blockDim.x) {
                const int r = e & (R - 1);
                const int cm = e >> lgR;
                const int c = cm >= nm1 ? 1 : 0;
                const int m = cm - c * nm1;
                const int i = i0 + r;
                if (i < n_rho) p.F[(((size_t)m * p.batch_total + b) * 2 + c) * n_rho + i] = Fs[e];
            }
        }
        __syncthreads();   // rings and Fs are refilled for the next block
    }
}

// Polar samples -> ring spectra as bf16 operand blocks (the blocked
// projection's F), one item = a block of 8 rings of IPI images (4: one 8-column
// group of the blocks).  Warp w transforms ring i0 + w of the images in turn
// (the next ring's samples are loaded as soon as the current FFT has left the
// registers), splits each into F_m, m <= n_max, and stages them as
// Fs[image][re/im][ring][m]; then 2 IPI consecutive threads write 32 IPI
// consecutive bytes (a full line at 4) per order and half.
// IPI is picked by launch_blk_t: small batches spread over the SMs and transform
// no absent images (one 4K frame, tiles + FFT + projection: 23.9 us a call with
// four, 19.4 with one), and the last round of items is not nearly empty (16 4K
// frames are 512 items of four images on 456 slots: 87.3 us, with two 86.7).
// Occupancy: three CTAs per SM at N = 1024 (shared memory, 69 KB each), so the
// register bound is set for three (77 registers; at 64 for four the kernel was
// 0.7 us per batch of 16 4K frames slower).
template <int LOGN, int IPI>
__global__ void __launch_bounds__(256, (LOGN >= 11 ? 2 : (LOGN == 10 ? 3 : 4)))
    k_ring_blk(const __grid_constant__ KbParams p) {
    using FFT = RingFFT<LOGN>;
    constexpr int N = FFT::N;
    constexpr int ROW = FFT::ROW_FLOATS;
    constexpr int R = 8;                           // rings per block = warps
    extern __shared__ __align__(16) float smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_rho = p.n_rho, n_max = p.n_max, nm1 = n_max + 1;
    float* rows = smem;                                       // [R][ROW]
    float* Fs = smem + R * ROW;                               // [IPI][2][R][nm1]
    float2* twt = reinterpret_cast<float2*>(smem + ((R * ROW + 16 * IPI * nm1 + 3) & ~3));
    float2* twm = twt + FFT::TW_FLOAT2;                       // e^{-2 pi i m / N}, m <= n_max
    FFT::load_twiddles(twt, p.tw);
    for (int m = threadIdx.x; m <= n_max; m += blockDim.x) twm[m] = __ldg(&p.tw[m]);
    const int n_rb = p.n_chunks * (64 / R);
    const int g0 = p.b_off / IPI, g1 = (p.b_off + p.nb - 1) / IPI;
    const int ng = g1 - g0 + 1;
    const int n_items = n_rb * ng;
    const int ncol = 2 * p.batch_total;
    auto in_run = [&](int b) { return b >= p.b_off && b < p.b_off + p.nb; };
    float2 v[FFT::Q];
    // the ring of (item, q) for this warp
    auto load_ring = [&](int item, int q) {
        const int gi = item / n_rb;
        const int i = (item - gi * n_rb) * R + warp;
        const int b = (g0 + gi) * IPI + q;
        const bool live = lane < FFT::L && i < n_rho && in_run(b);
        const float* src = p.fhat_in + ((size_t)(live ? b : 0) * n_rho + (live ? i : 0)) * N;
        if ((reinterpret_cast<uintptr_t>(p.fhat_in) & 7) == 0) {
            const float2* z = reinterpret_cast<const float2*>(src);
#pragma unroll
            for (int s2 = 0; s2 < FFT::Q; ++s2) v[s2] = live ? __ldg(&z[lane + FFT::L * s2]) : make_float2(0.f, 0.f);
        } else {
#pragma unroll
            for (int s2 = 0; s2 < FFT::Q; ++s2) {
                const int j = lane + FFT::L * s2;
                v[s2] = live ? make_float2(__ldg(src + 2 * j), __ldg(src + 2 * j + 1)) : make_float2(0.f, 0.f);
            }
        }
    };
    griddep_wait();                                           // the polar samples are written
    griddep_launch();
    if ((int)blockIdx.x < n_items) load_ring(blockIdx.x, 0);
    __syncthreads();                                          // twiddles
    float* row = rows + warp * ROW;
    float2* X = reinterpret_cast<float2*>(row);
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int gi = item / n_rb;
        const int rb = item - gi * n_rb;
        const int i0 = rb * R;
        for (int q = 0; q < IPI; ++q) {
            FFT::fwd(v, lane, twt, X);
            if constexpr (N >= 32) {
                // the ring's samples are in the registers now: when they are the
                // plan's scratch, their L2 lines are invalidated without a write
                // back (every line of a ring row belongs to that ring alone)
                const int b = (g0 + gi) * IPI + q;
                if (p.discard_in && i0 + warp < n_rho && in_run(b)) {
                    const char* base = reinterpret_cast<const char*>(p.fhat_in + ((size_t)b * n_rho + i0 + warp) * N);
                    for (int l = lane; l < N / 32; l += 32)
                        asm volatile("discard.global.L2 [%0], 128;" ::"l"(base + 128 * l) : "memory");
                }
            }
            if (lane < FFT::L) {
#pragma unroll
                for (int r = 0; r < FFT::Q; ++r) X[FFT::pad(FFT::fwd_index(r, lane))] = v[r];
            }
            __syncwarp();
            // the next ring into the registers while this one is split
            if (q < IPI - 1) load_ring(item, q + 1);
            else if (item + (int)gridDim.x < n_items) load_ring(item + gridDim.x, 0);
            float* fre = Fs + ((q * 2 + 0) * R + warp) * nm1;
            float* fim = Fs + ((q * 2 + 1) * R + warp) * nm1;
            for (int m = lane; m <= n_max; m += 32) {
                const float2 A = X[FFT::pad(m)];
                const float2 Bc = cconj(X[FFT::pad((FFT::M - m) & (FFT::M - 1))]);
                const float2 E = cscale(cadd(A, Bc), 0.5f);
                const float2 D = csub(A, Bc);
                const float2 O = make_float2(0.5f * D.y, -0.5f * D.x);
                const float2 Fm = cadd(E, cmul(twm[m], O));
                fre[m] = Fm.x;
                fim[m] = Fm.y;
            }
            __syncwarp();                                     // X is rewritten by the next FFT
        }
        __syncthreads();
        // (m, column) -> one 16-byte row of 8 rings; columns of images outside
        // this run (or past the batch) are left to their own launch
        for (int e = threadIdx.x; e < 2 * IPI * nm1; e += blockDim.x) {
            const int m = e / (2 * IPI), q = (e % (2 * IPI)) >> 1, c = e & 1;
            const int b = (g0 + gi) * IPI + q;
            if (!in_run(b)) continue;
            const float* src = Fs + ((q * 2 + c) * R) * nm1 + m;
            uint32_t h[4], l[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float x0 = src[(2 * k) * nm1], x1 = src[(2 * k + 1) * nm1];
                const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
                const __nv_bfloat16 l0 = __float2bfloat16_rn(x0 - __bfloat162float(h0));
                const __nv_bfloat16 l1 = __float2bfloat16_rn(x1 - __bfloat162float(h1));
                h[k] = __bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                l[k] = __bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
            const size_t o = fblk_row(m, i0, 2 * b + c, p.n_chunks, ncol);
            *reinterpret_cast<uint4*>(p.Fblk + o) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(p.Fblk + p.fblk_half + o) = make_uint4(l[0], l[1], l[2], l[3]);
        }
        __syncthreads();                                      // Fs is refilled for the next item
    }
}

template <int LOGN, int IPI>
static int blk_slots(const KbParams& kp, size_t* smem) {
    using FFT = RingFFT<LOGN>;
    *smem = sizeof(float) * (((size_t)8 * FFT::ROW_FLOATS + 16 * IPI * (kp.n_max + 1) + 3) & ~(size_t)3) +
            sizeof(float2) * ((size_t)FFT::TW_FLOAT2 + kp.n_max + 1);
    int dev = 0;
    cudaGetDevice(&dev);
    static std::mutex mu;
    static std::map<std::pair<int, size_t>, int> resident;     // (device, smem) -> CTAs on the device
    static SharedMemoryLimit limit;
    std::lock_guard<std::mutex> lk(mu);
    auto it = resident.find({dev, *smem});
    if (it != resident.end()) return it->second;
    const cudaError_t e = allow_smem(limit, k_ring_blk<LOGN, IPI>, dev, *smem);
    if (e != cudaSuccess) {
        cuda_error(e, "cudaFuncSetAttribute(k_ring_blk)");
        return 0;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ring_blk<LOGN, IPI>, 256, *smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    return resident[{dev, *smem}] = per_sm * num_sms(dev);
}

template <int LOGN>
static int launch_blk_t(const KbParams& kp, int nb, cudaStream_t st) {
    KbParams& k = const_cast<KbParams&>(kp);
    k.nb = nb;
    size_t smem[3];
    const int slots[3] = {blk_slots<LOGN, 1>(kp, &smem[0]), blk_slots<LOGN, 2>(kp, &smem[1]),
                          blk_slots<LOGN, 4>(kp, &smem[2])};
    if (!slots[0] || !slots[1] || !slots[2]) return ZM_ECUDA;
    // rounds of items (past the first, the CTAs drift apart: half a round of
    // tail) times an item's rings per warp, its barriers and stores counted as
    // half a ring.  Items of four stay where they fill the device well past once
    // (24 images: within 3 % either way), and a pair of images stays together
    // (its 64-byte pieces: 512 x 256 grid 13.5 us a call, apart 16.6)
    int best = 2;
    long long items[3];
    double cost[3];
    for (int j = 2; j >= 0; --j) {
        const int ipi = 1 << j;
        items[j] = (long long)kp.n_chunks * 8 * ((kp.b_off + nb - 1) / ipi - kp.b_off / ipi + 1);
        const double rounds = items[j] > slots[j] ? (double)items[j] / slots[j] + 0.5 : 1.0;
        cost[j] = rounds * (ipi + 0.5);
        if (items[2] < 1.25 * slots[2] && !(j == 0 && nb == 2) && cost[j] < cost[best]) best = j;
    }
    const int grid = (int)std::min<long long>(items[best], slots[best]);
    auto kernel = best == 0 ? k_ring_blk<LOGN, 1> : (best == 1 ? k_ring_blk<LOGN, 2> : k_ring_blk<LOGN, 4>);
    ZM_LAUNCH_PDL("k_ring_blk", kernel, dim3(grid), dim3(256), smem[best], st, kp);
    return ZM_OK;
}

static int launch_blk(int logn, const KbParams& kp, int nb, cudaStream_t st) {
    switch (logn) {
        case 3: return launch_blk_t<3>(kp, nb, st);
        case 4: return launch_blk_t<4>(kp, nb, st);
        case 5: return launch_blk_t<5>(kp, nb, st);
        case 6: return launch_blk_t<6>(kp, nb, st);
        case 7: return launch_blk_t<7>(kp, nb, st);
        case 8: return launch_blk_t<8>(kp, nb, st);
        case 9: return launch_blk_t<9>(kp, nb, st);
        case 10: return launch_blk_t<10>(kp, nb, st);
        case 11: return launch_blk_t<11>(kp, nb, st);
        default: return set_error(ZM_EUNSUPPORTED, "n_theta 2^%d", logn);
    }
}

template <int LOGN, int MODE>
static int launch_kb_t(const KbParams& kp, int R, int nb, cudaStream_t st, bool early = true) {
    using FFT = RingFFT<LOGN>;
    const size_t smem = sizeof(float) * ((size_t)R * FFT::ROW_FLOATS +
                                         (MODE == KB_RESAMPLE ? 0 : (size_t)2 * (kp.n_max + 1) * R + 2)) +
                        (MODE == KB_RESAMPLE ? 0 : sizeof(float2) * ((size_t)FFT::TW_FLOAT2 + kp.n_max + 1));
    int dev = 0;
    cudaGetDevice(&dev);
    static SharedMemoryLimit limit;
    ZM_CUDA_TRY(allow_smem(limit, k_ring_spectra<LOGN, MODE>, dev, smem));
    static std::mutex mu;
    static std::map<std::pair<int, size_t>, int> resident;   // (R, smem) -> CTAs per SM
    int per_sm = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = resident.find({R, smem});
        if (it != resident.end()) {
            per_sm = it->second;
        } else {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ring_spectra<LOGN, MODE>, R * 32, smem) !=
                    cudaSuccess ||
                per_sm < 1)
                per_sm = 1;
            resident[{R, smem}] = per_sm;
        }
    }
    KbParams& k = const_cast<KbParams&>(kp);
    k.nb = nb;
    const long long items = (long long)(kp.Fblk ? kp.n_chunks * (64 / R) : (kp.n_rho + R - 1) / R) * nb;
    const int grid = (int)std::min<long long>(items, (long long)per_sm * num_sms(dev));
    if (!early) {
        k_ring_spectra<LOGN, MODE><<<grid, R * 32, smem, st>>>(kp);
        ZM_LAUNCH_CHECK("k_ring_spectra");
        return ZM_OK;
    }
    ZM_LAUNCH_PDL("k_ring_spectra", (k_ring_spectra<LOGN, MODE>), dim3(grid), dim3(R * 32), smem, st, kp);
    return ZM_OK;
}

template <int MODE>
static int launch_kb_mode(int logn, const KbParams& kp, int R, int nb, cudaStream_t st, bool early = true) {
    switch (logn) {
        case 3: return launch_kb_t<3, MODE>(kp, R, nb, st, early);
        case 4: return launch_kb_t<4, MODE>(kp, R, nb, st, early);
        case 5: return launch_kb_t<5, MODE>(kp, R, nb, st, early);
        case 6: return launch_kb_t<6, MODE>(kp, R, nb, st, early);
        case 7: return launch_kb_t<7, MODE>(kp, R, nb, st, early);
        case 8: return launch_kb_t<8, MODE>(kp, R, nb, st, early);
        case 9: return launch_kb_t<9, MODE>(kp, R, nb, st, early);
        case 10: return launch_kb_t<10, MODE>(kp, R, nb, st, early);
        case 11: return launch_kb_t<11, MODE>(kp, R, nb, st, early);
        default: return set_error(ZM_EUNSUPPORTED, "n_theta 2^%d", logn);
    }
}

// ============================================================== driver
static int pick_rings(zm_plan_t p, int batch, bool tiled) {
    if (p->tune_rings == 2 || p->tune_rings == 4 || p->tune_rings == 8) return p->tune_rings;
    int R = 8;
    const int want = 2 * num_sms(p->device);
    // two rings to a CTA spread small calls over the SMs; rings of 512 angles and
    // more keep four (their twiddle tables are loaded by every CTA: one 2160 x
    // 2160 image on 1024 x 1024, gathered, FP32, 20.8 us against 23.7 with two), but of
    // 1024 angles after the tiles only where the rings are few (the same call by the
    // tiles 21.6 us with four, 19.7 with two)
    const bool many = tiled && p->n_theta == 1024 && (long long)p->n_rho * batch > want;
    const int least = p->n_theta >= 512 && !many ? 4 : 2;
    while (R > least && ((p->n_rho + R - 1) / R) * batch < want) R >>= 1;
    return R;
}

// Fused gather kernel on images [b0, b0 + nb) (any alignment): writes F and,
// when fhat_out is set, the polar samples.
static int launch_gather(zm_plan_t p, const zm_image_t* imgs, int b0, int nb, int batch, float* F, float* fhat_out,
                         bool resample_only, uint8_t* Fblk, cudaStream_t st) {
    // operand blocks take whole rows of 8 rings; calls of few blocks are spread
    // over twice the CTAs instead (us a call, not captured, with 8 / 4 rings: one 256 x 256 image
    // on 128 x 256 8.3 / 7.5, on 64 x 1024 11.7 / 9.3; one 1024 x 1024 on 512 x
    // 1024 19.2 / 16.1; beyond, the half rows cost more: four 256 x 256 images on
    // 128 x 128 7.1 / 7.4)
    const long long blocks = 8ll * p->n_chunks * batch;
    const int R = Fblk ? (blocks <= (p->n_theta >= 1024 ? 64 : 32) ? 4 : 8) : pick_rings(p, batch, false);
    static thread_local KbParams kp;
    kp.Fblk = resample_only ? nullptr : Fblk;
    kp.fblk_half = fblk_half_bytes(p->n_max, p->n_chunks, 2 * batch);
    kp.n_chunks = p->n_chunks;
    kp.n_rho = p->n_rho;
    kp.n_max = p->n_max;
    kp.batch_total = batch;
    kp.rho32 = p->rho32;
    kp.cs = p->cs;
    kp.tw = p->tw;
    kp.F = F;
    kp.fhat_out = fhat_out;
    kp.fhat_in = nullptr;
    kp.discard_in = 0;
    kp.release = 1;
    for (int c0 = b0; c0 < b0 + nb; c0 += KB_MAX_IMG) {
        const int nc = std::min(KB_MAX_IMG, b0 + nb - c0);
        kp.b_off = c0;
        for (int j = 0; j < nc; ++j) kp.img[j] = resolve(imgs[c0 + j]);
        // A large gather is not launched early: it lives on L1, and CTAs that come in
        // while the previous call's projection holds the SM's shared memory keep that
        // split for their lifetime (zm_moments captured, with the early launch / without,
        // us: 40 images of 1024 x 1024 on 512 x 256, bf16x3 149 / 54, fp16x3 151 / 69; 40 of
        // 512 x 512 on 256 x 256, bf16x3 45 / 29; 1024 x 1024 on 512 x 1024, two images 26 /
        // 17; half a million samples up to 30 % the same way, though calls of that size that
        // are not captured gain as much).  The FP32 projection of few orders holds less of
        // it: twice the samples up to order 64 and 256 angles (half a million: captured
        // 0.88 to 1.05 of the time, else 0.74 to 0.93; order 100: 1.23 and 1.04).
        const long long limit =
            p->prec == PREC_FP32 && p->n_theta <= 256 && p->n_max <= 64 ? 2 * GATHER_PDL_SAMPLES : GATHER_PDL_SAMPLES;
        const long long samples = (long long)nc * p->n_rho * p->n_theta;
        const bool early = samples <= limit;
        const int s = resample_only
                          ? launch_kb_mode<KB_RESAMPLE>(p->log_theta, kp, R, nc, st, samples <= 8 * GATHER_PDL_SAMPLES)
                          : launch_kb_mode<KB_GATHER>(p->log_theta, kp, R, nc, st, early);
        if (s != ZM_OK) return s;
    }
    return ZM_OK;
}

// Angular transform of given polar samples fhat[b][i][k] -> F (or the
// operand blocks Fblk) for images [b0, b0 + nb) of a batch of `batch`: the
// tensor-core DFT where the plan allows it, else the ring FFT.  tiled: the tile
// resampler has just written them; scratch: into the plan's workspace.
static int launch_polar_fft(zm_plan_t p, const float* fhat, int b0, int nb, int batch, float* F, uint8_t* Fblk,
                            cudaStream_t st, bool tiled = false, bool scratch = false) {
    if (Fblk && polar_dft_eligible(p, fhat)) return launch_polar_dft(p, fhat, b0, nb, batch, Fblk, st);
    const int R = Fblk ? 8 : pick_rings(p, batch, tiled);
    static thread_local KbParams kp;
    kp.Fblk = Fblk;
    kp.fblk_half = fblk_half_bytes(p->n_max, p->n_chunks, 2 * batch);
    kp.n_chunks = p->n_chunks;
    kp.n_rho = p->n_rho;
    kp.n_max = p->n_max;
    kp.batch_total = batch;
    kp.rho32 = p->rho32;
    kp.cs = p->cs;
    kp.tw = p->tw;
    kp.F = F;
    kp.fhat_out = nullptr;
    kp.fhat_in = fhat;
    kp.discard_in = scratch && Fblk && ((uintptr_t)fhat & 127u) == 0 ? 1 : 0;
    // spectra for the caller: what follows is the next call's tile resampler, which
    // would take the SMs from rings still to come (four 596 x 1152 images on 282 x 512,
    // captured: 15.0 us a call with, 10.5 without)
    kp.release = Fblk || F == (const float*)p->ws_F.ptr || !tiled ? 1 : 0;
    for (int c0 = b0; c0 < b0 + nb; c0 += 65535) {
        const int nc = std::min(65535, b0 + nb - c0);
        kp.b_off = c0;
        const bool narrow = tiled && p->log_theta == 10 && (long long)nc * p->n_rho * p->n_theta <= TILED_SAMPLES;
        const int s = Fblk     ? launch_blk(p->log_theta, kp, nc, st)
                      : narrow ? launch_kb_t<10, KB_TILED>(kp, R, nc, st)
                               : launch_kb_mode<KB_POLAR>(p->log_theta, kp, R, nc, st);
        if (s != ZM_OK) return s;
    }
    return ZM_OK;
}

// Where the gather kernel is the fastest of the three by default.  Its rings of
// up to 256 angles leave a lane eight samples, whose loads are all in flight;
// images come from L1 and L2, and no plan of tiles or stages stands before the
// first pixel.  Measured per zm_moments call, captured and back to back (gather /
// staged up to 2^17 samples an image, tiles above; us, bf16x3 unless said, sizes as
// image side on N_rho x N_theta):
//  256 angles: 256 on 128 x 256, 16 images 11.6 / 13.8; 700 on 350 x 256, 6 images
//   12.8 / 17.4, 16 images 20.7 / 21.9; 1024 on 512 x 256, 6 images 15.7 / 19.5, 12
//   images 22.5 / 25.1; 2160 on 1080 x 256, 4 images 21.9 / 27.6.  Only on grids of up
//   to 2^16 samples and from about a million samples a call is the staged kernel ahead:
//   512 on 256 x 256, order 50, 12 images 14.8 / 16.1, 16 images 17.1 / 16.2, 24 images
//   21.6 / 22.5; 512 x 440 on 239 x 256, order 87 (more operand blocks to write), 20
//   images 22.1 / 17.8, 40 images 32.7 / 29.8; with the fp16 projection already from
//   half a million, 872 x 268 on 145 x 256, 18 images 22.5 / 21.4.  Its rows do not fit the stages where
//   the disk is large for the grid, which leaves the tiles: 1024 on 250 x 256, 16
//   images 21.8 / 23.9, 40 images 48.5 / 42.1.
//  512 angles (16 samples a lane), grids of up to 2^17 samples: FP32 rows up to 1.5
//   million a call (512 on 256 x 512, 8 images 16.3 / 19.3, 16 images 23.6 / 21.4), operand
//   blocks up to half a million (256 on 128 x 512, 8 images 13.6 / 14.8, 16 images 17.9
//   / 15.8; 528 x 168 on 98 x 512, order 232, 20 images 22.2 / 16.9), or as far where the
//   disk is large for the grid (512 on 64 x 512, 24 images 18.5 / 23.0).
//  1024 angles.  Grids of up to 2^17 samples would be staged, which is far slower
//   there: up to 1.5 million a call (512 on 128 x 1024, 12 images 22.6 / 25.3, FP32
//   20.5 / 25.7).  Larger grids have the tiles, and the form the spectra are wanted in
//   decides.  Operand blocks: up to 1.25 million (512 on 256 x 1024, 4 images 21.7 /
//   23.2, 6 images 28.6 / 27.8; 1024 on 512 x 1024, 2 images 17.1 / 22.7, 3 images 23.5
//   / 22.8; 2160 on 1024 x 1024, 1 image 19.7 / 19.8).  FP32 rows, whose ring FFT
//   after the tiles is cheaper: below a million (512 on 256 x 1024, 3 images 15.9 / 20.4;
//   1024 on 512 x 1024, 1 image 12.9 / 15.1, 3 images 20.7 / 19.2; 2160 on 1024 x 1024,
//   1 image 21.3 / 18.9).
// A plan told to fuse or not to (ZM_FUSED), or to use a tensor-core transform, does
// that.
static bool gather_by_default(zm_plan_t p, const zm_image_t& im, int batch, bool operand_blocks) {
    if (p->fused_mode != 0 || p->dft_mode > 0 || p->pdft_mode > 0) return false;
    const long long samples = (long long)p->n_rho * p->n_theta, call = samples * batch;
    const GeoImage g = resolve(im);
    const double area = 4.0 * g.r * g.r;                 // of the disk's square, in pixels
    if (p->n_theta < 256) return true;
    if (p->n_theta == 256) {
        if (samples > 1 << 16) return true;
        if (area > 12 * samples) return call <= 1ll << 21;
        return call <= (p->prec == PREC_FP16X3 ? 1ll << 19 : 7ll << 17) ||
               call > (operand_blocks && p->n_max > 64 ? 5ll << 19 : 3ll << 19);
    }
    if (p->n_theta == 512)
        return samples <= FUSED_AUTO_SAMPLES && call <= (operand_blocks && area <= 4 * samples ? 1ll << 19 : 3ll << 19);
    if (p->n_theta > 1024) return false;
    if (samples <= FUSED_AUTO_SAMPLES) return call <= 3ll << 19;
    return operand_blocks ? call <= 5ll << 18 : call < 1ll << 20;
}

// Ring spectra of a batch.  Polar input: FFT only.  Images: runs of one
// geometry go through the tensor-core DFT kernel when the plan asks for it
// (dft_mode, off by default) and the spectra are wanted as operand blocks
// only (no polar samples out), else through the fused kernel when its fused_mode allows (resampling
// and ring FFT in one pass, polar samples written only to the caller's
// fhat_out), unless the gather kernel is faster there (gather_by_default);
// other runs of TMA-eligible images go through the tile resampler into the
// polar buffer (the caller's fhat_out, else the plan workspace) and then the
// ring FFT; the rest take the gather kernel.
int launch_spectra(zm_plan_t p, const zm_image_t* imgs, const float* fhat_in, int batch, float* F,
                   float* fhat_out, bool resample_only, cudaStream_t st, uint8_t* Fblk) {
    if (fhat_in) return launch_polar_fft(p, fhat_in, 0, batch, batch, F, Fblk, st);
    const bool fuse = p->fused_mode > 0 ||
                      (p->fused_mode == 0 && (long long)p->n_rho * p->n_theta <= FUSED_AUTO_SAMPLES);
    const bool gather = p->tune_gather == 1 || (p->tune_gather == 0 && !resample_only &&
                                                gather_by_default(p, imgs[0], batch, Fblk != nullptr));
    const bool dft = Fblk && !fhat_out && !resample_only && !gather && p->dft_mode > 0;
    auto use_dft = [&](int b) { return dft && dft_eligible(p, imgs[b]); };
    auto use_fused = [&](int b) { return fuse && !resample_only && !gather && fused_eligible(p, imgs[b]); };
    auto use_tma = [&](int b) { return !gather && tma_eligible(imgs[b]); };
    float* fh = fhat_out;
    int b = 0;
    while (b < batch) {
        int e = b + 1;
        int s;
        if (use_dft(b)) {
            while (e < batch && use_dft(e) && same_geometry(imgs[b], imgs[e])) ++e;
            s = launch_ring_dft(p, imgs, b, e - b, batch, Fblk, st);
            if (s == ZM_OK) {
                b = e;
                continue;
            }
            if (s != ZM_EUNSUPPORTED) return s;
            e = b + 1;                       // a geometry whose stages the buffers cannot hold
        }
        if (use_fused(b)) {
            while (e < batch && use_fused(e) && same_geometry(imgs[b], imgs[e])) ++e;
            s = launch_ring_fused(p, imgs, b, e - b, batch, F, Fblk, fhat_out, st);
            if (s == ZM_OK) {
                b = e;
                continue;
            }
            if (s != ZM_EUNSUPPORTED) return s;
            e = b + 1;                       // a geometry the stage buffers cannot hold
        }
        if (use_tma(b)) {
            while (e < batch && use_tma(e) && same_geometry(imgs[b], imgs[e])) ++e;
            if (!fh) {
                s = p->ws_fhat.grow(sizeof(float) * (size_t)batch * p->n_rho * p->n_theta);
                if (s != ZM_OK) return s;
                fh = (float*)p->ws_fhat.ptr;
            }
            // the plan's scratch (no caller buffer): the samples are kept in L2
            // for the ring FFT, which drops them once read (not for the opt-in
            // tensor-core DFT, which does not)
            const bool scratch = fh != fhat_out && !resample_only;
            const bool keep = scratch && !(Fblk && polar_dft_eligible(p, fh));
            s = launch_resample_tiles(p, imgs, b, e - b, fh, st, keep);
            if (s == ZM_OK && !resample_only) s = launch_polar_fft(p, fh, b, e - b, batch, F, Fblk, st, true, scratch);
        } else {
            while (e < batch && !use_tma(e)) ++e;
            s = launch_gather(p, imgs, b, e - b, batch, F, fhat_out, resample_only, Fblk, st);
        }
        if (s != ZM_OK) return s;
        b = e;
    }
    return ZM_OK;
}

int launch_projection(zm_plan_t p, const float* F, int batch, float* out, unsigned flags, cudaStream_t st) {
    if (p->prec == PREC_FP32) return launch_projection_fp32(p, F, batch, out, flags, st);
    return launch_projection_tc(p, F, batch, out, flags, st);
}

// Stage 1 of the moments: ring spectra of a batch (images, or polar samples
// when fhat_in is set) into the plan's workspace, in the form its projection
// reads (bf16 operand blocks for the blocked tensor-core projection, FP32
// rows otherwise).
int launch_stage_spectra(zm_plan_t p, const zm_image_t* imgs, const float* fhat_in, int batch, float* fhat_out,
                         cudaStream_t st) {
    if (blocked_projection(p)) {
        const size_t half = fblk_half_bytes(p->n_max, p->n_chunks, 2 * batch);
        const int s = p->ws_Fblk.grow(2 * half);
        if (s != ZM_OK) return s;
        return launch_spectra(p, imgs, fhat_in, batch, nullptr, fhat_out, false, st, (uint8_t*)p->ws_Fblk.ptr);
    }
    const int s = p->ws_F.grow(sizeof(float) * (size_t)(p->n_max + 1) * batch * 2 * p->n_rho);
    if (s != ZM_OK) return s;
    return launch_spectra(p, imgs, fhat_in, batch, (float*)p->ws_F.ptr, fhat_out, false, st);
}

// Stage 2: the radial projection of the spectra stage 1 left in the workspace
// (consume: no later call reads them, so the blocked form drops them from L2).
int launch_stage_project(zm_plan_t p, int batch, float* out, unsigned flags, cudaStream_t st, bool consume) {
    if (blocked_projection(p))
        return launch_projection_blocked(p, (const uint8_t*)p->ws_Fblk.ptr, batch, out, flags, st, consume);
    return launch_projection(p, (const float*)p->ws_F.ptr, batch, out, flags, st);
}

int launch_moments(zm_plan_t p, const zm_image_t* imgs, const float* fhat_in, int batch, float* out,
                   float* fhat_out, unsigned flags, cudaStream_t st) {
    const int s = launch_stage_spectra(p, imgs, fhat_in, batch, fhat_out, st);
    return s != ZM_OK ? s : launch_stage_project(p, batch, out, flags, st, true);
}

}  // namespace zm

using namespace zm;

static int moments_common(zm_plan_t plan, const zm_image_t* imgs, const float* fhat_in, int batch, float* out,
                          float* fhat_out, unsigned flags, void* stream) {
    if (!plan) return set_error(ZM_EINVAL, "plan is NULL");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1 (got %d)", batch);
    if (!out) return set_error(ZM_EINVAL, "output pointer is NULL");
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    if (!fhat_in) {
        const int s = check_images(imgs, batch);
        if (s != ZM_OK) return s;
    }
    DeviceGuard g(plan->device);
    if (!g.ok) return set_error(ZM_ECUDA, "cannot select device %d", plan->device);
    return launch_moments(plan, imgs, fhat_in, batch, out, fhat_out, flags, (cudaStream_t)stream);
}

extern "C" int zm_moments(zm_plan_t plan, const zm_image_t* imgs, int batch, float* out, unsigned flags,
                          void* stream) {
    return moments_common(plan, imgs, nullptr, batch, out, nullptr, flags, stream);
}

extern "C" int zm_moments_ex(zm_plan_t plan, const zm_image_t* imgs, int batch, float* out, float* fhat,
                             unsigned flags, void* stream) {
    return moments_common(plan, imgs, nullptr, batch, out, fhat, flags, stream);
}

extern "C" int zm_moments_polar(zm_plan_t plan, const float* fhat, int batch, float* out, unsigned flags,
                                void* stream) {
    if (!fhat) return set_error(ZM_EINVAL, "fhat is NULL");
    return moments_common(plan, nullptr, fhat, batch, out, nullptr, flags, stream);
}

extern "C" int zm_resample(zm_plan_t plan, const zm_image_t* imgs, int batch, float* fhat, void* stream) {
    if (!plan) return set_error(ZM_EINVAL, "plan is NULL");
    if (!fhat) return set_error(ZM_EINVAL, "fhat is NULL");
    const int s = check_images(imgs, batch);
    if (s != ZM_OK) return s;
    DeviceGuard g(plan->device);
    return launch_spectra(plan, imgs, nullptr, batch, nullptr, fhat, true, (cudaStream_t)stream);
}

extern "C" int zm_ring_spectra(zm_plan_t plan, const zm_image_t* imgs, int batch, float* spectra, float* fhat,
                               void* stream) {
    if (!plan) return set_error(ZM_EINVAL, "plan is NULL");
    if (!spectra) return set_error(ZM_EINVAL, "spectra is NULL");
    const int s = check_images(imgs, batch);
    if (s != ZM_OK) return s;
    DeviceGuard g(plan->device);
    return launch_spectra(plan, imgs, nullptr, batch, spectra, fhat, false, (cudaStream_t)stream);
}

extern "C" int zm_project(zm_plan_t plan, const float* spectra, int batch, float* out, unsigned flags,
                          void* stream) {
    if (!plan || !spectra || !out) return set_error(ZM_EINVAL, "NULL argument");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1 (got %d)", batch);
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    DeviceGuard g(plan->device);
    return launch_projection(plan, spectra, batch, out, flags, (cudaStream_t)stream);
}

extern "C" int zm_stage_spectra(zm_plan_t plan, const zm_image_t* imgs, int batch, void* stream) {
    if (!plan) return set_error(ZM_EINVAL, "plan is NULL");
    const int s = check_images(imgs, batch);
    if (s != ZM_OK) return s;
    DeviceGuard g(plan->device);
    if (!g.ok) return set_error(ZM_ECUDA, "cannot select device %d", plan->device);
    const int r = launch_stage_spectra(plan, imgs, nullptr, batch, nullptr, (cudaStream_t)stream);
    plan->staged_batch = (r == ZM_OK) ? batch : 0;
    return r;
}

extern "C" int zm_stage_project(zm_plan_t plan, int batch, float* out, unsigned flags, void* stream) {
    if (!plan || !out) return set_error(ZM_EINVAL, "NULL argument");
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    if (batch < 1 || batch != plan->staged_batch)
        return set_error(ZM_EINVAL, "zm_stage_project: batch %d, but the plan holds spectra of %d images", batch,
                         plan->staged_batch);
    DeviceGuard g(plan->device);
    if (!g.ok) return set_error(ZM_ECUDA, "cannot select device %d", plan->device);
    return launch_stage_project(plan, batch, out, flags, (cudaStream_t)stream);
}

extern "C" int zm_plan_reserve(zm_plan_t plan, int batch) {
    if (!plan) return set_error(ZM_EINVAL, "plan is NULL");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1");
    DeviceGuard g(plan->device);
    const size_t nb = (size_t)batch;
    int s = plan->ws_F.grow(sizeof(float) * (size_t)(plan->n_max + 1) * nb * 2 * plan->n_rho);
    // polar samples of the tile resampler
    if (s == ZM_OK) s = plan->ws_fhat.grow(sizeof(float) * nb * plan->n_rho * plan->n_theta);
    // partial sums of the split-K tensor-core projection: never more than one slice per 32 nodes
    const size_t S = (size_t)(plan->n_rho + 31) / 32;
    if (s == ZM_OK && plan->prec != PREC_FP32) s = plan->ws_part.grow(sizeof(float) * S * plan->P * 2 * nb);
    if (s == ZM_OK) s = plan->ws_G.grow(sizeof(float) * g_floats(batch, plan->n_rho, plan->n_max));
    // reductions: a record per block of an image (pixel errors) or per ring (fused errors)
    const size_t rec = std::max<size_t>(RED_MAX_PARTS, (size_t)plan->n_rho);
    if (s == ZM_OK) s = plan->ws_red.grow(sizeof(double) * nb * rec * 4);
    if (s == ZM_OK) s = plan->ws_scale.grow(sizeof(float) * 2 * nb);
    if (s == ZM_OK && blocked_projection(plan))
        s = plan->ws_Fblk.grow(2 * fblk_half_bytes(plan->n_max, plan->n_chunks, 2 * batch));
    return s;
}
