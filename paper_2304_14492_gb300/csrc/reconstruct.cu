// Reconstruction (Eq. 9) as the transpose of the moment path: a radial
// contraction G_m(rho_i) = c_m sum_n Z_nm R_nm(rho_i), an inverse real FFT per
// ring, and optional interpolation onto pixels; the reconstruction errors of
// Eq. 10 and Eq. 13 and the min-max normalisation of Sec. 3 / Table I.
#include <algorithm>
#include <map>
#include <mutex>

#include "packed.cuh"
#include "ring_fft.cuh"
#include "zm_internal.cuh"

namespace zm {

constexpr float kTwoPi = 6.28318530717958647692f;

// ============================================================== radial part
// G(b, i, m, re/im) = c_m sum_{n = m, m+2, ..} R_nm(rho_i) Z_nm (layout g_index), with
// c_m = 2/eps_m (c_0 = 1, c_m = 2) for the literal Eq. 9 and c_m = 1 for the
// half sum over the stored m >= 0.
//
// Bound by reading the table once per RB images.  One CTA = 128 nodes, one m
// and RB images (the fewest of 1, 2, 4 that hold the batch, or four); its eight warps
// take every eighth order, so the longest chain is K_m / 8 steps and the few
// heavy m do not outlast the rest, and their sums meet in shared memory in a
// fixed order.  Each warp streams its own orders' rows through a ring of three
// stages (cp.async, twelve rows in flight, the first ones on their way before
// the moments are read); a lane multiplies two pairs of nodes (fma.rn.f32x2)
// with moments staged twice each, so nothing is shuffled into pairs.  4 images,
// n_max 500, 512 nodes (129 MB of table), cold: 68 us for a thread per node
// with all K_m orders and eight image slots; 52 us with eight row loads held in
// registers (104 of them, two CTAs per SM); 41 us like this.
constexpr int RR_NODES = 128, RR_WARPS = 8, RR_U = 4, RR_STAGES = 3;
constexpr int RR_RING = RR_STAGES * RR_U * RR_NODES;      // floats of a warp's ring

// V: floats per copy (4, or 1 where rows are not 16-byte aligned).
template <int RB, int V>
__global__ void __launch_bounds__(32 * RR_WARPS, 3)
k_recon_radial(const float* __restrict__ R32m, const float2* __restrict__ Z, const int* __restrict__ mrow,
               int n_max, int n_rho, int P, int batch, int neumann, float* __restrict__ G) {
    extern __shared__ __align__(16) float rr_sm[];        // the rings, then the moments [RB][Km] (twice each)
    const int i0 = blockIdx.x * RR_NODES;
    const int m = blockIdx.y;
    const int b0 = blockIdx.z * RB;
    const int nb = min(RB, batch - b0);
    const int Km = (n_max - m) / 2 + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* ring = rr_sm + warp * RR_RING;
    float4* zs4 = reinterpret_cast<float4*>(rr_sm + max(RR_WARPS * RR_RING, RR_WARPS * RB * 2 * RR_NODES));
    const uint32_t ring_a = static_cast<uint32_t>(__cvta_generic_to_shared(ring));
    const float* Rm = R32m + (size_t)mrow[m] * n_rho + i0;
    auto issue = [&](int c, int st) {
#pragma unroll
        for (int u = 0; u < RR_U; ++u) {
            const int j = warp + RR_WARPS * (RR_U * c + u);
            if (j >= Km) break;
            const float* src = Rm + (size_t)j * n_rho;
            const uint32_t dst = ring_a + 4u * (st * RR_U + u) * RR_NODES;
            if (V == 4) {
                const int on = i0 + 4 * lane < n_rho;     // else zero-filled
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + 16u * lane),
                             "l"(on ? src + 4 * lane : Rm), "r"(on ? 16 : 0) : "memory");
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int on = i0 + lane + 32 * e < n_rho;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4u * (lane + 32 * e)),
                                 "l"(on ? src + lane + 32 * e : Rm), "r"(on ? 4 : 0) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int c = 0; c < RR_STAGES; ++c) issue(c, c);      // the table is the plan's
    griddep_wait();                    // the moments are written, G is free
    griddep_launch();
    for (int t = threadIdx.x; t < RB * Km; t += blockDim.x) {
        const int bb = t / Km, j = t - bb * Km;
        const float2 z = (bb < nb) ? __ldg(&Z[(size_t)(b0 + bb) * P + moment_index(m + 2 * j, m)]) : make_float2(0.f, 0.f);
        zs4[t] = make_float4(z.x, z.x, z.y, z.y);
    }
    __syncthreads();
    f32x2 re[RB][2], im[RB][2];
#pragma unroll
    for (int bb = 0; bb < RB; ++bb) re[bb][0] = re[bb][1] = im[bb][0] = im[bb][1] = 0;
    const ulonglong2* zs = reinterpret_cast<const ulonglong2*>(zs4);
    int st = 0;
    for (int c = 0; warp + RR_WARPS * RR_U * c < Km; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(RR_STAGES - 1) : "memory");
        __syncwarp();
#pragma unroll
        for (int u = 0; u < RR_U; ++u) {
            const int j = warp + RR_WARPS * (RR_U * c + u);
            if (j >= Km) break;
            const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(ring + (st * RR_U + u) * RR_NODES + 4 * lane);
#pragma unroll
            for (int bb = 0; bb < RB; ++bb) {
                const ulonglong2 z = zs[bb * Km + j];
                re[bb][0] = fma2(r.x, z.x, re[bb][0]);
                re[bb][1] = fma2(r.y, z.x, re[bb][1]);
                im[bb][0] = fma2(r.x, z.y, im[bb][0]);
                im[bb][1] = fma2(r.y, z.y, im[bb][1]);
            }
        }
        __syncwarp();
        issue(c + RR_STAGES, st);
        st = st + 1 < RR_STAGES ? st + 1 : 0;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                   // every ring is read: their place takes the sums
    // sums [warp][image][re/im][node]
    constexpr int OUT = RB * 2 * RR_NODES;
#pragma unroll
    for (int bb = 0; bb < RB; ++bb)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float2 a = unpack2(c ? im[bb][0] : re[bb][0]), b = unpack2(c ? im[bb][1] : re[bb][1]);
            *reinterpret_cast<float4*>(rr_sm + warp * OUT + (bb * 2 + c) * RR_NODES + 4 * lane) =
                make_float4(a.x, a.y, b.x, b.y);
        }
    __syncthreads();
    const float cm = (neumann && m > 0) ? 2.f : 1.f;
    const int nrb = (n_rho + 7) / 8;
    const int parts = min(RR_WARPS, Km);
    for (int e = threadIdx.x; e < OUT; e += blockDim.x) {
        const int i = i0 + (e & (RR_NODES - 1)), bc = e / RR_NODES;
        if (i >= n_rho || (bc >> 1) >= nb) continue;
        float v = 0.f;
        for (int w = 0; w < parts; ++w) v += rr_sm[w * OUT + e];
        G[g_index(b0 + (bc >> 1), i, m, bc & 1, nrb, n_max + 1)] = cm * v;
    }
}

// The same sums for larger batches (launch_radial).  Splitting K_m over warps costs a pass
// over all sums per eight images, which outweighs the sums themselves once the
// images fill the device, so here a warp keeps all orders of 64 nodes and 8 images:
// a lane has 8 nodes of one ring block (its share of G is one run of 64 bytes per
// image, written a 32-byte sector at a time) and 2 images as (re, im) pairs, 16 packed
// multiply-adds an order for three 16-byte shared-memory loads.  The CTA's warps are
// IG groups of images by NG of nodes; rows come in chunks of eight orders through
// three stages (cp.async), the moments of the next chunk are loaded while one is
// multiplied.  A chunk's sums are taken apart and then added, so that no sum is a
// longer chain than in k_recon_radial (8 + K_m / 8 additions).  Bound by shared-memory
// bandwidth and FP32 issue.  zm_reconstruct, us a call, with the sums split over
// warps for eight images / like this: n_max 60 on 256 nodes, 64 images 24.3 / 15.4; 127
// on 512, 16 images 30.0 / 22.4, 128 images 204 / 125; 300 on 512, 8 images 38.5 / 30.4,
// 128 images 568 / 327; 1000 on 256, 16 images 381 / 159 (a thread per node before
// either: 16.9, 23.9, 131, 42.8, 390, 359).
constexpr int RW_KC = 8, RW_STAGES = 3;

template <int IG, int NG, int V>
__global__ void __launch_bounds__(32 * IG * NG, 16 / (IG * NG))
k_recon_radial_wide(const float* __restrict__ R32m, const float2* __restrict__ Z, const int* __restrict__ mrow,
                    int n_max, int n_rho, int P, int batch, int neumann, float* __restrict__ G) {
    constexpr int NODES = 64 * NG, IMGS = 8 * IG, THREADS = 32 * IG * NG;
    __shared__ __align__(16) float rows[RW_STAGES][RW_KC][NODES];
    __shared__ __align__(16) float2 zs[2][RW_KC][IMGS];
    const int i0 = blockIdx.x * NODES, m = blockIdx.y, b0 = blockIdx.z * IMGS;
    const int Km = (n_max - m) / 2 + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ig = warp % IG, nh = warp / IG;         // the warp's images and nodes
    const int ng = lane & 7, cg = lane >> 3;          // the lane's ring block and pair of images
    const float* Rm = R32m + (size_t)mrow[m] * n_rho + i0;
    const uint32_t rows_a = static_cast<uint32_t>(__cvta_generic_to_shared(&rows[0][0][0]));
    // 16-byte words of a row: within 64 nodes the even ones first, then the odd
    // ones, so that the eight lanes of a phase read 128 consecutive bytes
    auto place = [](int q) { return (q & ~15) + ((q & 1) << 3) + ((q & 15) >> 1); };
    // chunks are taken from the high orders down, whose moments are the smaller ones
    // wherever they fall off; orders past K_m in the first are zero rows and moments
    auto issue = [&](int j0, int st) {
        if (j0 >= 0) {
            for (int e = threadIdx.x; e < RW_KC * NODES / V; e += THREADS) {
                const int k = e / (NODES / V), x = (e % (NODES / V)) * V;
                const int on = j0 + k < Km && i0 + x < n_rho;         // else zero-filled
                const float* src = on ? Rm + (size_t)(j0 + k) * n_rho + x : Rm;
                const uint32_t dst = rows_a + 4u * ((st * RW_KC + k) * NODES + 4 * place(x >> 2) + (x & 3));
                if (V == 4)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0)
                                 : "memory");
                else
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(on ? 4 : 0)
                                 : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // one moment per thread and chunk: order t / IMGS of the chunk, image t mod IMGS
    const int zk = threadIdx.x / IMGS, zb = threadIdx.x % IMGS;
    const bool zlive = zk < RW_KC && b0 + zb < batch;
    const float2* Zb = Z + (size_t)min(b0 + zb, batch - 1) * P;
    auto moment = [&](int j0) {
        return zlive && j0 >= 0 && j0 + zk < Km ? __ldg(Zb + moment_index(m + 2 * (j0 + zk), m)) : make_float2(0.f, 0.f);
    };
    int j0 = ((Km + RW_KC - 1) / RW_KC - 1) * RW_KC;
    issue(j0, 0);                      // the table is the plan's
    issue(j0 - RW_KC, 1);
    griddep_wait();                    // the moments are written, G is free
    griddep_launch();
    float2 zn = moment(j0);
    if (zk < RW_KC) zs[0][zk][zb] = zn;
    zn = moment(j0 - RW_KC);
    const bool busy = b0 + ig * 8 < batch && i0 + nh * 64 < n_rho;
    f32x2 tot[8][2];
#pragma unroll
    for (int r = 0; r < 8; ++r) tot[r][0] = tot[r][1] = 0;
    int st = 0, zbuf = 0;
    for (; j0 >= 0; j0 -= RW_KC) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();               // this chunk is here; the last one is read
        issue(j0 - 2 * RW_KC, st + 2 < RW_STAGES ? st + 2 : st + 2 - RW_STAGES);
        if (zk < RW_KC) zs[zbuf ^ 1][zk][zb] = zn;
        zn = moment(j0 - 2 * RW_KC);
        if (busy) {
            const float* rk = &rows[st][0][nh * 64 + 4 * ng];
            const float2* zr = &zs[zbuf][0][ig * 8 + cg * 2];
            f32x2 acc[8][2];
#pragma unroll
            for (int k = 0; k < RW_KC; ++k) {
                const float4 a = *reinterpret_cast<const float4*>(rk + k * NODES);
                const float4 b = *reinterpret_cast<const float4*>(rk + k * NODES + 32);
                const ulonglong2 z = *reinterpret_cast<const ulonglong2*>(zr + k * IMGS);
                const float r8[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const f32x2 rr = pack2(r8[r], r8[r]);
                    acc[r][0] = k ? fma2(rr, z.x, acc[r][0]) : mul2(rr, z.x);
                    acc[r][1] = k ? fma2(rr, z.y, acc[r][1]) : mul2(rr, z.y);
                }
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                tot[r][0] = add2(tot[r][0], acc[r][0]);
                tot[r][1] = add2(tot[r][1], acc[r][1]);
            }
        }
        st = st + 1 < RW_STAGES ? st + 1 : 0;
        zbuf ^= 1;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int i = i0 + nh * 64 + ng * 8;
    if (!busy || i >= n_rho) return;
    const float cm = (neumann && m > 0) ? 2.f : 1.f;
    const int nrb = (n_rho + 7) / 8;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int b = b0 + ig * 8 + cg * 2 + e;
        if (b >= batch) break;
        float re[8], im[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float2 v = unpack2(tot[r][e]);
            re[r] = cm * v.x;
            im[r] = cm * v.y;
        }
        // all 8 rings of the block (those past n_rho are zero and not read), a whole
        // 32-byte sector at a time
        float* g = G + g_index(b, i, m, 0, nrb, n_max + 1);
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(g), "f"(re[0]), "f"(re[1]),
                     "f"(re[2]), "f"(re[3]), "f"(re[4]), "f"(re[5]), "f"(re[6]), "f"(re[7]) : "memory");
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(g + 8), "f"(im[0]), "f"(im[1]),
                     "f"(im[2]), "f"(im[3]), "f"(im[4]), "f"(im[5]), "f"(im[6]), "f"(im[7]) : "memory");
    }
}

// ============================================================== ring inverse FFT
// f~_k = Re sum_{m=0}^{n_max} G_m e^{2 pi i m k / N}.  With the Hermitian
// spectrum S (S_0 = 2 Re G_0, S_m = G_m, S_{N-m} = conj G_m) and
// x_k = sum_m S_m e^{2 pi i m k/N} = 2 f~_k, the packed z_j = x_{2j} + i x_{2j+1}
// is the M-point inverse DFT of
//   C_m = (S_m + conj S_{M-m}) + i e^{2 pi i m/N} (S_m - conj S_{M-m}).
// One warp per ring: C is formed straight from G in shared memory in the
// order the inverse FFT wants, and its output is already in natural order
// across lanes, so f~ is written (and the reference read) with coalesced
// accesses from registers.  The grid is persistent: each CTA loads the
// twiddles once and takes blocks of R rings (b, rb): first item blockIdx.x,
// then items claimed from the counter work[0] (dynamic, so that the CTAs
// finish within about one item of each other); the last CTA to finish sets
// work[0..1] back to 0 for the next launch.
// With ERR, each warp also accumulates, against the reference polar samples
// `ref`, sum (ref - f~)^2, sum ref^2 and max ref of its ring into one record
// part[b][i] = (sd, sf, max, 0) (Eq. 10 / Eq. 13 on the polar nodes); `out`
// may then be NULL.
template <int LOGN, bool ERR>
__global__ void __launch_bounds__(256, (LOGN >= 11 ? 2 : 4))
k_recon_ifft(const float* __restrict__ G, const float2* __restrict__ tw, int n_max, int n_rho, int batch,
             float* __restrict__ out, const float* __restrict__ ref, float4* __restrict__ part,
             int* __restrict__ work) {
    using FFT = RingFFT<LOGN>;
    constexpr int N = FFT::N;
    constexpr int M = FFT::M;
    constexpr int L = FFT::L;
    constexpr int Q = FFT::Q;
    extern __shared__ __align__(16) float2 Gs[];              // [R][n_max+1]
    const int R = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nm1 = n_max + 1;
    float2* twt = Gs + R * nm1;                                   // warp-FFT twiddles
    float2* twm = twt + FFT::TW_FLOAT2;                           // e^{-2 pi i m / N}, m < M
    float2* tbuf = twm + M + warp * FFT::TBUF;                    // per-warp transpose buffer
    FFT::load_twiddles(twt, tw);
    for (int m = threadIdx.x; m < M; m += blockDim.x) twm[m] = __ldg(&tw[m]);
    griddep_wait();                    // G (and the reference samples) are written, out is free
    griddep_launch();
    // persistent: the CTA takes ring blocks (b, rb) = item / n_rb, item mod n_rb
    __shared__ int next_item[2];
    int turn = 0;
    const int n_rb = (n_rho + R - 1) / R;
    const int n_items = n_rb * batch;
    for (int item = blockIdx.x; item < n_items;) {
        const int b = item / n_rb, rb = item - b * n_rb;
        const int i0 = rb * R;
        // this block's G is one contiguous run of nm1 x 16 floats (g_index)
        // the next item is claimed, and the reference rows are asked into L2,
        // while this one is transformed
        int claim = 0;
        if (threadIdx.x == 0) claim = (int)gridDim.x + atomicAdd(&work[0], 1);
        if (ERR && i0 + warp < n_rho) {
            const char* rr = reinterpret_cast<const char*>(ref + ((size_t)b * n_rho + i0 + warp) * N);
            for (int l = lane; l * 32 < N; l += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(rr + 128 * l));
        }
        const float4* gb = reinterpret_cast<const float4*>(G + g_index(b, i0, 0, 0, n_rb, nm1));
        float* gsf = reinterpret_cast<float*>(Gs);
        for (int e = threadIdx.x; e < nm1 * 4; e += blockDim.x) {
            const float4 q4 = __ldg(&gb[e]);
            const int m = e >> 2, c = (e >> 1) & 1, r0 = (e & 1) * 4;
            gsf[2 * ((r0 + 0) * nm1 + m) + c] = q4.x;
            gsf[2 * ((r0 + 1) * nm1 + m) + c] = q4.y;
            gsf[2 * ((r0 + 2) * nm1 + m) + c] = q4.z;
            gsf[2 * ((r0 + 3) * nm1 + m) + c] = q4.w;
        }
        __syncthreads();
        const float2* Gr = Gs + warp * nm1;
        float2 v[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const int m = FFT::inv_index(a, lane);
            float2 Sm = make_float2(0.f, 0.f), T = make_float2(0.f, 0.f);
            if (m <= n_max) Sm = (m == 0) ? make_float2(2.f * Gr[0].x, 0.f) : Gr[m];
            const int q = M - m;
            if (q >= 1 && q <= n_max) T = cconj(Gr[q]);
            const float2 w = twm[m];                         // e^{-2 pi i m/N}
            const float2 ie = make_float2(w.y, w.x);         // i e^{+2 pi i m/N} = i conj(w)
            const float2 C = cadd(cadd(Sm, T), cmul(ie, csub(Sm, T)));
            v[a] = (lane < L) ? C : make_float2(0.f, 0.f);
        }
        FFT::inv(v, lane, twt, tbuf);
        const int i = i0 + warp;
        float sd = 0.f, sf = 0.f, mx = -INFINITY;
        if (i < n_rho && lane < L) {
            const size_t row = ((size_t)b * n_rho + i) * N;
            float2* o = out ? reinterpret_cast<float2*>(out + row) : nullptr;
            if (ERR && FFT::TBUF >= Q * 32) {
                // f~ goes out and into this warp's transpose buffer (free after
                // the inverse FFT), so that all Q reference loads can be in
                // flight at once without holding f~ in registers
                const float2* rf = reinterpret_cast<const float2*>(ref + row);
#pragma unroll
                for (int r = 0; r < Q; ++r) {
                    const float2 x = make_float2(0.5f * v[r].x, 0.5f * v[r].y);
                    if (o) __stcs(&o[lane + L * brev_c<FFT::LOGQ>(r)], x);   // output, not read again here
                    tbuf[r * 32 + lane] = x;
                }
                float2 f[Q];
#pragma unroll
                for (int r = 0; r < Q; ++r) f[r] = __ldcs(&rf[lane + L * brev_c<FFT::LOGQ>(r)]);   // last use
#pragma unroll
                for (int r = 0; r < Q; ++r) {
                    const float2 x = tbuf[r * 32 + lane];
                    const float d0 = f[r].x - x.x, d1 = f[r].y - x.y;
                    sd = fmaf(d0, d0, fmaf(d1, d1, sd));
                    sf = fmaf(f[r].x, f[r].x, fmaf(f[r].y, f[r].y, sf));
                    mx = fmaxf(mx, fmaxf(f[r].x, f[r].y));
                }
            } else if (ERR) {
                const float2* rf = reinterpret_cast<const float2*>(ref + row);
                // groups of four loads in flight, consumed as they arrive (few live registers)
#pragma unroll
                for (int r0 = 0; r0 < Q; r0 += 4) {
                    float2 f[4];
#pragma unroll
                    for (int u = 0; u < 4 && r0 + u < Q; ++u) f[u] = __ldg(&rf[lane + L * brev_c<FFT::LOGQ>(r0 + u)]);
#pragma unroll
                    for (int u = 0; u < 4 && r0 + u < Q; ++u) {
                        const int r = r0 + u;
                        const float2 x = make_float2(0.5f * v[r].x, 0.5f * v[r].y);
                        if (o) o[lane + L * brev_c<FFT::LOGQ>(r)] = x;
                        const float d0 = f[u].x - x.x, d1 = f[u].y - x.y;
                        sd = fmaf(d0, d0, fmaf(d1, d1, sd));
                        sf = fmaf(f[u].x, f[u].x, fmaf(f[u].y, f[u].y, sf));
                        mx = fmaxf(mx, fmaxf(f[u].x, f[u].y));
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < Q; ++r)
                    o[lane + L * brev_c<FFT::LOGQ>(r)] = make_float2(0.5f * v[r].x, 0.5f * v[r].y);
            }
        }
        if (ERR) {
            for (int o2 = 16; o2; o2 >>= 1) {
                sd += __shfl_xor_sync(0xffffffffu, sd, o2);
                sf += __shfl_xor_sync(0xffffffffu, sf, o2);
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o2));
            }
            if (lane == 0 && i < n_rho) part[(size_t)b * n_rho + i] = make_float4(sd, sf, mx, 0.f);
        }
        if (threadIdx.x == 0) next_item[turn] = claim;
        __syncthreads();   // Gs is refilled for the next ring block; next_item is set
        item = next_item[turn];
        turn ^= 1;         // rewritten only after the barrier above of the next block
    }
    // the last CTA out resets the counter (every CTA's last claim precedes its
    // arrival here)
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&work[1], 1) == (int)gridDim.x - 1) {
            work[0] = 0;
            work[1] = 0;
            __threadfence();
        }
    }
}

// Resident CTAs per SM of a kernel at a dynamic shared-memory size (cached).
template <typename K>
static int resident_blocks(K kernel, int threads, size_t smem) {
    static std::mutex mu;
    static std::map<std::pair<const void*, size_t>, int> cache;
    std::lock_guard<std::mutex> lk(mu);
    auto key = std::make_pair(reinterpret_cast<const void*>(kernel), smem);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) n = 1;
    cache[key] = n;
    return n;
}

template <int LOGN, bool ERR>
static int launch_ifft_t(const float* G, const float2* tw, int n_max, int n_rho, int batch, float* out,
                         const float* ref, float4* part, int* work, int sms, cudaStream_t st) {
    using FFT = RingFFT<LOGN>;
    const int R = 8;
    const size_t smem = sizeof(float2) * ((size_t)R * (n_max + 1) + FFT::TW_FLOAT2 + FFT::M + (size_t)R * FFT::TBUF);
    int dev = 0;
    cudaGetDevice(&dev);
    static SharedMemoryLimit limit;
    ZM_CUDA_TRY(allow_smem(limit, k_recon_ifft<LOGN, ERR>, dev, smem));
    const long long items = (long long)((n_rho + R - 1) / R) * batch;
    const int slots = sms * resident_blocks(k_recon_ifft<LOGN, ERR>, R * 32, smem);
    const int grid = (int)std::min<long long>(items, slots);
    ZM_LAUNCH_PDL("k_recon_ifft", (k_recon_ifft<LOGN, ERR>), dim3(grid), dim3(R * 32), smem, st, G, tw, n_max, n_rho,
                  batch, out, ref, part, work);
    return ZM_OK;
}

template <bool ERR>
static int launch_ifft(zm_plan_t p, const float* G, int batch, float* out, const float* ref, float4* part,
                       cudaStream_t st) {
    static int sms_cache[64] = {0};
    const int dev = p->device;
    int sms = (dev >= 0 && dev < 64) ? sms_cache[dev] : 0;
    if (!sms) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
        if (dev >= 0 && dev < 64) sms_cache[dev] = sms;
    }
    switch (p->log_theta) {
        case 3: return launch_ifft_t<3, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 4: return launch_ifft_t<4, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 5: return launch_ifft_t<5, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 6: return launch_ifft_t<6, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 7: return launch_ifft_t<7, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 8: return launch_ifft_t<8, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 9: return launch_ifft_t<9, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 10: return launch_ifft_t<10, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        case 11: return launch_ifft_t<11, ERR>(G, p->tw, p->n_max, p->n_rho, batch, out, ref, part, p->work, sms, st);
        default: return set_error(ZM_EUNSUPPORTED, "n_theta 2^%d", p->log_theta);
    }
}

template <int IG, int NG, int V>
static int launch_radial_wide_t(zm_plan_t p, const float* moments, int batch, unsigned flags, float* G,
                                cudaStream_t st) {
    constexpr int NODES = 64 * NG, IMGS = 8 * IG;
    const int nz = (batch + IMGS - 1) / IMGS;
    for (int z0 = 0; z0 < nz; z0 += 65535) {
        const int nzc = std::min(65535, nz - z0);
        const int b0 = z0 * IMGS;
        const int nbc = std::min(batch - b0, nzc * IMGS);
        ZM_LAUNCH_PDL("k_recon_radial_wide", (k_recon_radial_wide<IG, NG, V>),
                      dim3((p->n_rho + NODES - 1) / NODES, p->n_max + 1, nzc), dim3(32 * IG * NG), 0, st, (const float*)p->R32m,
                      (const float2*)moments + (size_t)b0 * p->P, (const int*)p->mrow, p->n_max, p->n_rho, p->P, nbc,
                      (flags & ZM_NEUMANN) ? 1 : 0, G + g_floats(b0, p->n_rho, p->n_max));
    }
    return ZM_OK;
}

template <int RB, int V>
static int launch_radial_t(zm_plan_t p, const float* moments, int batch, unsigned flags, float* G, cudaStream_t st) {
    const size_t smem = sizeof(float) * RR_WARPS * std::max(RR_RING, RB * 2 * RR_NODES) +
                        sizeof(float4) * RB * (size_t)(p->n_max / 2 + 1);
    const int dev = p->device;
    static SharedMemoryLimit limit;
    ZM_CUDA_TRY(allow_smem(limit, k_recon_radial<RB, V>, dev, smem));
    const int nz = (batch + RB - 1) / RB;
    for (int z0 = 0; z0 < nz; z0 += 65535) {
        const int nzc = std::min(65535, nz - z0);
        const int b0 = z0 * RB;
        const int nbc = std::min(batch - b0, nzc * RB);
        ZM_LAUNCH_PDL("k_recon_radial", (k_recon_radial<RB, V>),
                      dim3((p->n_rho + RR_NODES - 1) / RR_NODES, p->n_max + 1, nzc), dim3(32 * RR_WARPS), smem, st,
                      (const float*)p->R32m, (const float2*)moments + (size_t)b0 * p->P, (const int*)p->mrow, p->n_max,
                      p->n_rho, p->P, nbc, (flags & ZM_NEUMANN) ? 1 : 0, G + g_floats(b0, p->n_rho, p->n_max));
    }
    return ZM_OK;
}

static int launch_radial(zm_plan_t p, const float* moments, int batch, unsigned flags, cudaStream_t st,
                         float** G_out) {
    const int s = p->ws_G.grow(sizeof(float) * g_floats(batch, p->n_rho, p->n_max));
    if (s != ZM_OK) return s;
    float* G = (float*)p->ws_G.ptr;
    if (p->Rblk) {
        *G_out = G;
        return launch_radial_tc(p, moments, batch, flags, G, st);
    }
    const bool vec = (p->n_rho & 3) == 0;
    // More than four images: all orders in a warp, but past order 128 only once CTAs
    // that split them would go several times around the device; 256 nodes to a CTA, or 128 where the grid has no more or rows are copied float
    // by float.  zm_reconstruct, us a call, split / whole: n_max 200 on 128 nodes, 8
    // images 14.6 / 18.9, on 512 nodes 24.5 / 22.5, 12 images 33.7 / 25.8; 300 on 64
    // nodes, 11 images 17.6 / 23.2, on 512, 8 images 36.8 / 30.4; 100 on 256, 24 images
    // 19.2 / 15.0; 30 on 256, 8 images 6.2 / 5.4; 108 on 77 nodes, 8 images 8.0 / 9.5, but
    // 12.3 / 9.9 between the inverse transforms of 1024 angles.
    const long long split = (long long)((p->n_rho + RR_NODES - 1) / RR_NODES) * (p->n_max + 1) * ((batch + 3) / 4);
    const bool whole = batch > 4 && (p->n_max <= 128 || split > std::min(8 * p->n_max, 2400));
    const int st_ = batch == 1 ? (vec ? launch_radial_t<1, 4> : launch_radial_t<1, 1>)(p, moments, batch, flags, G, st)
                    : batch == 2 ? (vec ? launch_radial_t<2, 4> : launch_radial_t<2, 1>)(p, moments, batch, flags, G, st)
                    : !whole     ? (vec ? launch_radial_t<4, 4> : launch_radial_t<4, 1>)(p, moments, batch, flags, G, st)
                    : vec && p->n_rho > 256 ? launch_radial_wide_t<2, 4, 4>(p, moments, batch, flags, G, st)
                    : vec ? launch_radial_wide_t<2, 2, 4>(p, moments, batch, flags, G, st)
                          : launch_radial_wide_t<2, 2, 1>(p, moments, batch, flags, G, st);
    if (st_ != ZM_OK) return st_;
    *G_out = G;
    return ZM_OK;
}

int launch_reconstruct(zm_plan_t p, const float* moments, int batch, float* out, unsigned flags,
                       cudaStream_t st) {
    float* G = nullptr;
    const int s = launch_radial(p, moments, batch, flags, st, &G);
    if (s != ZM_OK) return s;
    return launch_ifft<false>(p, G, batch, out, nullptr, nullptr, st);
}

constexpr int RR_THREADS = 1024;
__global__ void k_reduce_records(const float4* __restrict__ part, int nrec, double count, double* __restrict__ out);

int launch_reconstruct_errors(zm_plan_t p, const float* moments, int batch, float* out, const float* fhat,
                              double* err, unsigned flags, cudaStream_t st) {
    float* G = nullptr;
    int s = launch_radial(p, moments, batch, flags, st, &G);
    if (s != ZM_OK) return s;
    const int nrec = p->n_rho;                 // one record per ring
    s = p->ws_red.grow(sizeof(float4) * (size_t)batch * nrec);
    if (s != ZM_OK) return s;
    float4* part = (float4*)p->ws_red.ptr;
    s = launch_ifft<true>(p, G, batch, out, fhat, part, st);
    if (s != ZM_OK) return s;
    const double count = (double)p->n_rho * (double)p->n_theta;
    ZM_LAUNCH_PDL("k_reduce_records", k_reduce_records, dim3(batch), dim3(RR_THREADS), 0, st, (const float4*)part,
                  nrec, count, err);
    return ZM_OK;
}

// ============================================================== pixels
struct CanvasDesc {
    float* data;
    long long pitch;
    int h, w;
    float cx, cy, r;
};

// Pixel centre (x, y) -> (rho, theta) in the disk's frame; same float
// arithmetic everywhere a disk membership is decided.
__device__ __forceinline__ float pixel_rho(float x, float y, float cx, float cy, float r, float* dx, float* dy) {
    *dx = x - cx;
    *dy = cy - y;
    return sqrtf((*dx) * (*dx) + (*dy) * (*dy)) / r;
}

// Canvases of one launch in groups of one geometry: the images of a group share
// every pixel's place on the polar grid.
struct CartGroup {
    int first, count;
};
struct CartParams {
    int n_rho, n_theta, b_off;
    int gauss;              // Gauss-Legendre nodes (else the midpoint rule)
    const float* rho32;
    const float* polar;     // [batch][n_rho][n_theta]
    CartGroup grp[KD_MAX_IMG];
    CanvasDesc cv[KD_MAX_IMG];
};

// The last node <= rho, or -1: a guess from the nodes' closed form (exact to
// about one node; Gauss-Legendre nodes lie near (1 - cos(pi (i + 3/4) / (n + 1/2))) / 2),
// moved until the table itself confirms it.  The arc cosine of 1 - 2 rho is only
// that guess: Abramowitz and Stegun 4.4.45, off by 6.8e-5 at most (asinf took 4 us
// more of a 4K frame).
__device__ __forceinline__ int last_node(const float* __restrict__ rho32, int n_rho, int gauss, float rho) {
    float x;
    if (gauss) {
        const float c = fabsf(1.f - 2.f * rho);
        const float t = sqrtf(fmaxf(1.f - c, 0.f)) * fmaf(fmaf(fmaf(-0.0187293f, c, 0.0742610f), c, -0.2121144f), c, 1.5707288f);
        x = ((float)n_rho + 0.5f) * (1.f / 3.14159265f) * (rho <= 0.5f ? t : 3.14159265f - t) - 0.75f;
    } else {
        x = rho * (float)n_rho - 0.5f;
    }
    int g = min(max((int)floorf(x), 0), n_rho - 1);
    while (g + 1 < n_rho && __ldg(&rho32[g + 1]) <= rho) ++g;
    while (g >= 0 && __ldg(&rho32[g]) > rho) --g;
    return g;
}

// Polar reconstruction -> pixels, one pixel per thread, a warp on an 8 x 4 tile:
// the bilinear corners of a compact tile fall on few 128-byte lines wherever it
// lies on the disk (a 32 x 1 run along a radius touches a line per pixel), and
// stores still fill whole 32-byte sectors.  The place of a pixel on the grid
// (square root, division, atan2, node lookup: about 100 instructions) is
// computed once and used for every image of the group.  Bound by the latency
// and the L1 wavefronts of the corner loads: with four pixels a thread and 24
// warps per SM three 3840 x 2160 bands took 67 us, with one and 64 warps 59 (warm;
// with the place per image and a ten-step search over the nodes 133, cold).  ONE:
// every group is one canvas, without the loop over images (one 4K canvas on 64 x 64
// Gauss nodes 51.4 us a call with it, 44.5 without; a thread per pixel and image 43.7).
constexpr int PTC_GROUP = 4;
template <bool ONE>
__global__ void __launch_bounds__(256) k_polar_to_cart(const __grid_constant__ CartParams p) {
    const CartGroup g = p.grp[blockIdx.z];
    const CanvasDesc c = p.cv[g.first];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int y = blockIdx.y * 32 + warp * 4 + (lane >> 3);
    const int x = blockIdx.x * 8 + (lane & 7);
    if (y >= c.h || x >= c.w) return;
    const int n_rho = p.n_rho, N = p.n_theta;
    // the corners' offsets (o0 < 0: outside the disk) and the two fractions
    int o0 = -1, o1 = 0, dk = 0;
    float s = 0.f, t = 0.f;
    float dx, dy;
    const float rho = pixel_rho((float)x, (float)y, c.cx, c.cy, c.r, &dx, &dy);
    if (rho <= 1.f) {
        float th = atan2f(dy, dx);
        if (th < 0.f) th += kTwoPi;
        const int lo = last_node(p.rho32, n_rho, p.gauss, rho);
        const int i1 = min(lo + 1, n_rho - 1), i0 = max(lo, 0);
        const float r0 = __ldg(&p.rho32[i0]), r1 = __ldg(&p.rho32[i1]);
        const float span = r1 - r0;
        t = fminf(fmaxf(span > 0.f ? (rho - r0) / span : 0.f, 0.f), 1.f);
        const float v = th * (float)N / kTwoPi;
        const float kf = floorf(v);
        s = v - kf;
        const int k0 = ((int)kf) & (N - 1);
        dk = ((k0 + 1) & (N - 1)) - k0;
        o0 = i0 * N + k0;
        o1 = i1 * N + k0;
    }
    const size_t img = (size_t)n_rho * N;
    const float* pb = p.polar + (size_t)(p.b_off + g.first) * img;
    auto value = [&](const float* pb) {
        if (o0 < 0) return 0.f;
        const float a0 = __ldg(pb + o0), a1 = __ldg(pb + o0 + dk), b0 = __ldg(pb + o1), b1 = __ldg(pb + o1 + dk);
        const float ra = fmaf(s, a1 - a0, a0), rb = fmaf(s, b1 - b0, b0);
        return fmaf(t, rb - ra, ra);
    };
    if constexpr (ONE) {
        c.data[(size_t)y * c.pitch + x] = value(pb);
    } else {
#pragma unroll 1
        for (int q = 0; q < g.count; ++q, pb += img)
            p.cv[g.first + q].data[(size_t)y * p.cv[g.first + q].pitch + x] = value(pb);
    }
}

static CanvasDesc resolve_canvas(const zm_canvas_t& cv) {
    zm_image_t im{cv.data, cv.height, cv.width, cv.pitch, cv.cx, cv.cy, cv.radius};
    const GeoImage g = resolve(im);
    return CanvasDesc{cv.data, g.pitch, g.h, g.w, g.cx, g.cy, g.r};
}

static bool same_disk(const CanvasDesc& a, const CanvasDesc& b) {
    return a.h == b.h && a.w == b.w && a.cx == b.cx && a.cy == b.cy && a.r == b.r;
}

int launch_polar_to_cart(zm_plan_t p, const float* polar, int batch, const zm_canvas_t* cv, cudaStream_t st) {
    static thread_local CartParams cp;
    cp.n_rho = p->n_rho;
    cp.n_theta = p->n_theta;
    cp.gauss = (p->flags & ZM_GRID_GAUSS) ? 1 : 0;
    cp.rho32 = p->rho32;
    cp.polar = polar;
    for (int b0 = 0; b0 < batch; b0 += KD_MAX_IMG) {
        const int nb = std::min(KD_MAX_IMG, batch - b0);
        cp.b_off = b0;
        int hmax = 1, wmax = 1, groups = 0;
        for (int j = 0; j < nb; ++j) {
            cp.cv[j] = resolve_canvas(cv[b0 + j]);
            hmax = std::max(hmax, cp.cv[j].h);
            wmax = std::max(wmax, cp.cv[j].w);
            // up to four images a group: enough to spread the geometry's cost,
            // and batches of small frames still fill the device
            if (groups && cp.grp[groups - 1].count < PTC_GROUP && same_disk(cp.cv[cp.grp[groups - 1].first], cp.cv[j]))
                ++cp.grp[groups - 1].count;
            else
                cp.grp[groups++] = CartGroup{j, 1};
        }
        auto kernel = groups == nb ? k_polar_to_cart<true> : k_polar_to_cart<false>;
        kernel<<<dim3((wmax + 7) / 8, (hmax + 31) / 32, groups), 256, 0, st>>>(cp);
        ZM_LAUNCH_CHECK("k_polar_to_cart");
    }
    return ZM_OK;
}

// ============================================================== reductions
constexpr int RED_THREADS = 256;
constexpr int RED_WARPS = RED_THREADS / 32;
constexpr int RED_PER_SM = 6;            // resident blocks per SM the registers allow
constexpr int RED_SEG = 2048;            // polar nodes a warp takes at a time
constexpr int RED_PARTS = 32;            // parts a block keeps in shared memory

enum { RED_DISK_ERRORS = 0, RED_POLAR_ERRORS = 1, RED_DISK_MINMAX = 2 };

struct RedParams {
    int n_nodes, b_off;
    int share;                // blocks an image may take (part_blocks)
    int release;              // the next kernel may start early
    const float* fhat;        // polar errors
    const float* frec;
    double* part;             // [image of the launch][RED_MAX_PARTS][4]
    int* done;                // [image of the launch] blocks finished, 0 between launches
    double* out;              // error modes: [batch][4]
    float* mm;                // min / max: [batch][2]
    CanvasDesc ref[KD_MAX_IMG];
    CanvasDesc tst[KD_MAX_IMG];
};

// The columns [*xa, *xb) of row y whose centres lie in the disk (empty: 0, 0).
// Membership is pixel_rho() <= 1 as everywhere (a not-a-number counts as
// inside, as a per-pixel "> 1" test has it).  |dx| grows away from the column
// nearest the centre and every float operation of pixel_rho() is monotone, so
// the columns are one run around it; its ends are guessed from the circle and
// moved until the test itself confirms them.
__device__ __forceinline__ void disk_span(const CanvasDesc& c, int y, int* xa, int* xb) {
    auto inside = [&](int x) {
        float dx, dy;
        return !(pixel_rho((float)x, (float)y, c.cx, c.cy, c.r, &dx, &dy) > 1.f);
    };
    *xa = *xb = 0;
    const int last = c.w - 1;
    const int xm = min((int)fminf(fmaxf(rintf(c.cx), 0.f), (float)last), last);
    if (!inside(xm)) return;
    const float dy = c.cy - (float)y;
    const float hw = sqrtf(fmaxf(c.r * c.r - dy * dy, 0.f));
    int a = min((int)fminf(fmaxf(ceilf(c.cx - hw), 0.f), (float)xm), xm);
    int b = max(min((int)fminf(fmaxf(floorf(c.cx + hw), (float)xm), (float)last), last), xm);
    while (a > 0 && inside(a - 1)) --a;
    while (a < xm && !inside(a)) ++a;
    while (b < last && inside(b + 1)) ++b;
    while (b > xm && !inside(b)) --b;
    *xa = a;
    *xb = b + 1;
}

// Columns of a row as 16-byte words: [*va, *vb) relative to `row` is the
// aligned middle of [xa, xb); up to three columns are left on either side.
__device__ __forceinline__ void vector_span(const float* row, int xa, int xb, int* va, int* vb) {
    const int phase = (int)((reinterpret_cast<uintptr_t>(row) >> 2) & 3);
    const int a = xa + ((4 - ((xa + phase) & 3)) & 3);
    const int n = xb > a ? (xb - a) & ~3 : 0;
    *va = n ? a : xa;
    *vb = n ? a + n : xa;
}

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_min(float v) {
    for (int o = 16; o; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Parts an image of so many rows is summed in, one record each: a row per warp up
// to RED_MAX_PARTS parts.  The image's own rows alone decide, so that the order of
// its sums, and with it every bit of them, does not depend on the images it shares
// a launch with.
__host__ __device__ __forceinline__ int row_parts(int rows) {
    const int n = (rows + RED_WARPS - 1) / RED_WARPS;
    return n < 1 ? 1 : (n < RED_MAX_PARTS ? n : RED_MAX_PARTS);
}

// Blocks that take an image's parts in turn: all that are resident at once, shared
// by the images of the launch (a block more for every part costs its own latency:
// 8 images of 4000 x 64, 25 us against 11), with RED_PARTS parts at most for one.
__host__ __device__ __forceinline__ int part_blocks(int parts, int share) {
    const int least = (parts + RED_PARTS - 1) / RED_PARTS;
    const int n = share > least ? share : least;
    return n < parts ? n : parts;
}

// Sums over the disk's pixels or the polar nodes: (sum (f - g)^2, sum f^2,
// max f, count) for the error modes, (min, max) for the min / max mode.  A warp
// takes whole rows (runs of RED_SEG nodes), of which it reads only the disk's
// columns, four 16-byte loads in flight per lane, with no test per pixel: bound
// by memory.  Two 16-byte words are summed as a tree before they join a lane's
// FP32 partial (a row of 3840 is 15 steps of it, pixel by pixel it was 120), each
// part (row_parts) is a double record, and an image's last block to finish adds its
// records in a fixed order and writes the result, so there is no second launch.
// Three 3840 x 2160 bands: min / max 151 + 5 us -> 19 us, errors 166 + 5 us -> 28 us
// (both cold, serialised; 44 and 88 MB read).  Before, 64 blocks an image tested
// every pixel with a square root and a division and had one load in flight.  A flat
// 4K image in a launch of 128 is off by 1.2e-7 (by lanes that ran on over an
// image's share of the device's blocks 2.0e-5; worst of three, emulated).
template <int MODE>
__global__ void __launch_bounds__(RED_THREADS, RED_PER_SM) k_reduce(const __grid_constant__ RedParams p) {
    constexpr int U = MODE == RED_DISK_MINMAX ? 4 : 2;     // 16-byte loads in flight per lane and image
    const int bl = blockIdx.y;
    const int b = p.b_off + bl;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    float s0 = 0.f, s1 = 0.f, mx = -INFINITY, mn = INFINITY;
    long long cnt = 0;
    auto add = [&](float f, float g) {
        if (MODE != RED_DISK_MINMAX) {
            const float d = f - g;
            s0 = fmaf(d, d, s0);
            s1 = fmaf(f, f, s1);
        } else {
            mn = fminf(mn, f);
        }
        mx = fmaxf(mx, f);
    };
    // the sums of a 16-byte word, (f - g)^2 and f^2, as trees
    auto word = [&](const float4& f, const float4& g, float* d2, float* f2) {
        const float dx = f.x - g.x, dy = f.y - g.y, dz = f.z - g.z, dw = f.w - g.w;
        *d2 = fmaf(dy, dy, dx * dx) + fmaf(dw, dw, dz * dz);
        *f2 = fmaf(f.y, f.y, f.x * f.x) + fmaf(f.w, f.w, f.z * f.z);
        mx = fmaxf(fmaxf(mx, fmaxf(f.x, f.y)), fmaxf(f.z, f.w));
    };
    const CanvasDesc& c = p.ref[bl];
    const CanvasDesc& t = p.tst[bl];
    const int rows = MODE == RED_POLAR_ERRORS ? (p.n_nodes + RED_SEG - 1) / RED_SEG : c.h;
    // (minima and maxima are the same in any order: no more parts than blocks)
    const int parts = MODE == RED_DISK_MINMAX ? min(row_parts(rows), p.share) : row_parts(rows);
    const int blocks = part_blocks(parts, p.share);
    if ((int)blockIdx.x >= blocks) return;       // the launch holds a taller image
    // this block takes the parts blockIdx.x, + blocks, ..; a warp has the rows
    // part * RED_WARPS + w, + parts * RED_WARPS, .. of each
    const int mine = (parts - 1 - (int)blockIdx.x) / blocks + 1;
    const int per = (rows + parts * RED_WARPS - 1) / (parts * RED_WARPS);
    auto row_of = [&](int q) {
        const int v = q / per;
        return ((long long)blockIdx.x + (long long)v * blocks) * RED_WARPS + w + (long long)(q - v * per) * parts * RED_WARPS;
    };
    __shared__ float sh[2][RED_PARTS][RED_WARPS];
    __shared__ float shm[2][RED_WARPS];
    __shared__ long long shc[RED_WARPS];
    __shared__ int is_last;
    int left = per, part = 0;                    // rows left of the part in hand
    const int total = mine * per;
    long long first = blockIdx.x * RED_WARPS + w, yl = first;
    for (int q0 = 0; q0 < total; q0 += 32) {
        // lane l: the span of the l-th of this warp's next 32 rows
        int sa = 0, sb = 0;
        if (MODE != RED_POLAR_ERRORS) {
            if (q0 + l < total && row_of(q0 + l) < rows) disk_span(c, (int)row_of(q0 + l), &sa, &sb);
        }
        if (q0 == 0) {                           // the images are written, the records are free
            griddep_wait();
            if (p.release) griddep_launch();
        }
        for (int q = 0; q < 32 && q0 + q < total; ++q) {
            const int y = (int)yl;               // = row_of(q0 + q)
            int xa, xb;
            const float *f, *g;
            if (MODE == RED_POLAR_ERRORS) {
                xa = 0;
                xb = min(RED_SEG, p.n_nodes - y * RED_SEG);
                f = p.fhat + (size_t)b * p.n_nodes + (size_t)y * RED_SEG;
                g = p.frec + (size_t)b * p.n_nodes + (size_t)y * RED_SEG;
            } else {
                xa = __shfl_sync(0xffffffffu, sa, q);
                xb = __shfl_sync(0xffffffffu, sb, q);
                f = c.data + (long long)y * c.pitch;
                g = MODE == RED_DISK_ERRORS ? t.data + (long long)y * t.pitch : f;
            }
            if (xa < xb) {
                cnt += xb - xa;
                int va, vb;
                vector_span(f, xa, xb, &va, &vb);
                // the columns outside the aligned middle: lane by lane
                for (int x = xa + l; x < va; x += 32) add(__ldg(f + x), MODE != RED_DISK_MINMAX ? __ldg(g + x) : 0.f);
                for (int x = vb + l; x < xb; x += 32) add(__ldg(f + x), MODE != RED_DISK_MINMAX ? __ldg(g + x) : 0.f);
                const bool gvec = ((reinterpret_cast<uintptr_t>(g + va)) & 15) == 0;
                const int nv = (vb - va) >> 2;
                for (int v0 = l; v0 < nv; v0 += 32 * U) {
                    float4 fv[U], gv[U];
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (v0 + 32 * u < nv) fv[u] = __ldg(reinterpret_cast<const float4*>(f + va) + v0 + 32 * u);
#pragma unroll
                    for (int u = 0; u < U; ++u) gv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (MODE != RED_DISK_MINMAX) {
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (v0 + 32 * u < nv) {
                                const float* gp = g + va + 4 * (v0 + 32 * u);
                                if (gvec) gv[u] = __ldg(reinterpret_cast<const float4*>(gp));
                                else gv[u] = make_float4(__ldg(gp), __ldg(gp + 1), __ldg(gp + 2), __ldg(gp + 3));
                            }
                    }
                    if (MODE == RED_DISK_MINMAX) {
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (v0 + 32 * u < nv) {
                                mn = fminf(fminf(mn, fminf(fv[u].x, fv[u].y)), fminf(fv[u].z, fv[u].w));
                                mx = fmaxf(fmaxf(mx, fmaxf(fv[u].x, fv[u].y)), fmaxf(fv[u].z, fv[u].w));
                            }
                    } else {
                        float d2[2], f2[2];
                        word(fv[0], gv[0], &d2[0], &f2[0]);
                        if (v0 + 32 < nv) {
                            word(fv[1], gv[1], &d2[1], &f2[1]);
                            d2[0] += d2[1];
                            f2[0] += f2[1];
                        }
                        s0 += d2[0];
                        s1 += f2[0];
                    }
                }
            }
            if (--left) {
                yl += (long long)parts * RED_WARPS;
                continue;
            }
            // the part's rows are done: its sums over the warp, both in one tree
            if (MODE != RED_DISK_MINMAX) {
                float v = (l & 16) ? s1 : s0;
                v += __shfl_xor_sync(0xffffffffu, (l & 16) ? s0 : s1, 16);
                for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if ((l & 15) == 0) sh[l >> 4][part][w] = v;
                s0 = s1 = 0.f;
            }
            left = per;
            ++part;
            first += (long long)blocks * RED_WARPS;
            yl = first;
        }
    }
    // maximum, minimum and count go with the block's first part
    mx = warp_max(mx);
    if (MODE == RED_DISK_MINMAX) mn = warp_min(mn);
    if (l == 0) {
        shm[0][w] = mx;
        shm[1][w] = mn;
        shc[w] = cnt;
    }
    __syncthreads();
    if (threadIdx.x < mine) {
        const int v = threadIdx.x;
        double a = 0, c1 = MODE == RED_DISK_MINMAX ? (double)INFINITY : 0;
        float m2 = -INFINITY;
        long long n = 0;
        for (int j = 0; j < RED_WARPS; ++j) {
            if (MODE != RED_DISK_MINMAX) {
                a += sh[0][v][j];
                c1 += sh[1][v][j];
            }
            if (v == 0) {
                if (MODE == RED_DISK_MINMAX) c1 = fmin(c1, (double)shm[1][j]);
                m2 = fmaxf(m2, shm[0][j]);
                n += shc[j];
            }
        }
        double* o = p.part + ((size_t)bl * RED_MAX_PARTS + blockIdx.x + (size_t)v * blocks) * 4;
        *reinterpret_cast<double2*>(o) = make_double2(a, c1);
        *reinterpret_cast<double2*>(o + 2) = make_double2((double)m2, (double)n);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(p.done + bl, 1) == blocks - 1;
    __syncthreads();
    if (!is_last || w) return;
    // out = (eps_1, eps, f_max, count), mm = (min, max): lanes over the image's
    // records, then a shuffle tree.  Every image has its own last block: one for
    // all of a launch's images took 128 of them in turn (64 x 64 pixels each: 72 us a
    // call, now 10).
    __threadfence();
    double sd = 0, sf = 0, n = 0, dmx = -INFINITY, dmn = INFINITY;
    const double2* rec = reinterpret_cast<const double2*>(p.part) + (size_t)bl * RED_MAX_PARTS * 2;
    for (int e0 = l; e0 < parts; e0 += 128) {       // four records in flight per lane
        double2 ra[4], rb[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool on = e0 + 32 * u < parts;
            ra[u] = on ? __ldcg(rec + 2 * (e0 + 32 * u))
                       : make_double2(0, MODE == RED_DISK_MINMAX ? (double)INFINITY : 0);
            rb[u] = on ? __ldcg(rec + 2 * (e0 + 32 * u) + 1) : make_double2(-(double)INFINITY, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (MODE == RED_DISK_MINMAX) {
                dmn = fmin(dmn, ra[u].y);
            } else {
                sd += ra[u].x;
                sf += ra[u].y;
                n += rb[u].y;
            }
            dmx = fmax(dmx, rb[u].x);
        }
    }
    for (int o = 16; o; o >>= 1) {
        if (MODE == RED_DISK_MINMAX) {
            dmn = fmin(dmn, __shfl_xor_sync(0xffffffffu, dmn, o));
        } else {
            sd += __shfl_xor_sync(0xffffffffu, sd, o);
            sf += __shfl_xor_sync(0xffffffffu, sf, o);
            n += __shfl_xor_sync(0xffffffffu, n, o);
        }
        dmx = fmax(dmx, __shfl_xor_sync(0xffffffffu, dmx, o));
    }
    if (l) return;
    p.done[bl] = 0;
    const size_t bj = (size_t)b;
    if (MODE == RED_DISK_MINMAX) {
        p.mm[2 * bj] = (float)dmn;
        p.mm[2 * bj + 1] = (float)dmx;
    } else {
        p.out[4 * bj + 0] = sd / sf;
        p.out[4 * bj + 1] = sd / (dmx * dmx * n);
        p.out[4 * bj + 2] = dmx;
        p.out[4 * bj + 3] = n;
    }
}

// out[b] = (eps_1, eps, f_max, count) from the nrec ring records (sd, sf,
// max, 0) of image b; count = N_rho N_theta nodes.  One block per image.  The
// sums stay in FP32 up to the 32 warp partials (sequential per thread, then
// the warp's shuffle tree), which are combined in FP64 by warp 0: GB300 runs
// FP64 at a small fraction of its FP32 rate, so only those few additions and
// the two ratios are done in FP64.  Summation order is fixed: deterministic.
// With the per-ring sums also in FP32 (32 terms per lane, then two shuffle
// trees), the worst-case relative rounding error of each sum is below 50
// units of FP32 rounding (3e-6) at N_rho = N_theta = 1024.
__global__ void __launch_bounds__(RR_THREADS)
k_reduce_records(const float4* __restrict__ part, int nrec, double count, double* __restrict__ out) {
    griddep_wait();                    // the records are written
    griddep_launch();
    __shared__ float red[32][3];
    const int b = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float sd = 0.f, sf = 0.f, mx = -INFINITY;
    const float4* rec = part + (size_t)b * nrec;
    for (int j = threadIdx.x; j < nrec; j += blockDim.x) {
        const float4 a = __ldg(&rec[j]);
        sd += a.x;
        sf += a.y;
        mx = fmaxf(mx, a.z);
    }
    for (int o = 16; o; o >>= 1) {
        sd += __shfl_xor_sync(0xffffffffu, sd, o);
        sf += __shfl_xor_sync(0xffffffffu, sf, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
        red[warp][0] = sd;
        red[warp][1] = sf;
        red[warp][2] = mx;
    }
    __syncthreads();
    if (warp != 0) return;
    const int nw = (int)(blockDim.x >> 5);
    double dsd = lane < nw ? (double)red[lane][0] : 0.0;
    double dsf = lane < nw ? (double)red[lane][1] : 0.0;
    mx = lane < nw ? red[lane][2] : -INFINITY;
    for (int o = 16; o; o >>= 1) {
        dsd += __shfl_xor_sync(0xffffffffu, dsd, o);
        dsf += __shfl_xor_sync(0xffffffffu, dsf, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
        const double dmx = (double)mx;
        out[4 * b + 0] = dsd / dsf;
        out[4 * b + 1] = dsd / (dmx * dmx * count);
        out[4 * b + 2] = dmx;
        out[4 * b + 3] = count;
    }
}

template <int MODE>
static int run_reduce(zm_plan_t p, const zm_image_t* ref, const zm_image_t* tst, const float* fhat,
                      const float* frec, int batch, double* out, float* mm, cudaStream_t st, bool release = true) {
    static thread_local RedParams rp;
    rp.release = release ? 1 : 0;
    rp.n_nodes = p->n_rho * p->n_theta;
    rp.fhat = fhat;
    rp.frec = frec;
    rp.out = out;
    rp.mm = mm;
    rp.done = p->work + 2;
    int s = p->ws_red.grow(sizeof(double) * 4 * RED_MAX_PARTS * (size_t)std::min(batch, KD_MAX_IMG));
    if (s != ZM_OK) return s;
    for (int b0 = 0; b0 < batch; b0 += KD_MAX_IMG) {
        const int nb = std::min(KD_MAX_IMG, batch - b0);
        rp.b_off = b0;
        int rows = MODE == RED_POLAR_ERRORS ? (rp.n_nodes + RED_SEG - 1) / RED_SEG : 1;
        if (MODE != RED_POLAR_ERRORS) {
            for (int j = 0; j < nb; ++j) {
                const GeoImage g = resolve(ref[b0 + j]);
                rp.ref[j] = CanvasDesc{const_cast<float*>(g.data), g.pitch, g.h, g.w, g.cx, g.cy, g.r};
                rows = std::max(rows, g.h);
                if (MODE == RED_DISK_ERRORS) {
                    const GeoImage t = resolve(tst[b0 + j]);
                    rp.tst[j] = CanvasDesc{const_cast<float*>(t.data), t.pitch, t.h, t.w, t.cx, t.cy, t.r};
                }
            }
        }
        rp.part = (double*)p->ws_red.ptr;         // each launch finishes its own images
        rp.share = std::max(1, RED_PER_SM * num_sms(p->device) / nb);
        const int blocks = part_blocks(row_parts(rows), rp.share);
        ZM_LAUNCH_PDL("k_reduce", k_reduce<MODE>, dim3(blocks, nb), dim3(RED_THREADS), 0, st, rp);
    }
    return ZM_OK;
}

int launch_errors(zm_plan_t p, const zm_image_t* ref, const zm_image_t* test, const float* fhat,
                  const float* frec, int batch, double* out, cudaStream_t st) {
    if (fhat) return run_reduce<RED_POLAR_ERRORS>(p, nullptr, nullptr, fhat, frec, batch, out, nullptr, st);
    return run_reduce<RED_DISK_ERRORS>(p, ref, test, nullptr, nullptr, batch, out, nullptr, st);
}

int launch_disk_minmax(zm_plan_t p, const zm_image_t* imgs, int batch, float* out, cudaStream_t st) {
    return run_reduce<RED_DISK_MINMAX>(p, imgs, nullptr, nullptr, nullptr, batch, nullptr, out, st);
}

struct NormParams {
    const float* mm;          // [batch][2] canvas min / max
    const float* target;      // [batch][2] wanted min / max
    int b_off;
    CanvasDesc cv[KD_MAX_IMG];
};

// Blocks per image of k_minmax_apply: a row per warp where the device holds that
// many at once (a second row for a few of the warps would double the time), at
// least one block an image.
static int apply_blocks(zm_plan_t p, int rows, int nb) {
    return std::min(row_parts(rows), std::max(1, RED_PER_SM * num_sms(p->device) / nb));
}

// Rows as in k_reduce: a warp per row, only the disk's columns, 16-byte loads
// and stores, the scale once per warp (three 3840 x 2160 bands: 62 us with a
// thread and a membership test per pixel, now 15 us, cold; 88 MB moved).
__global__ void __launch_bounds__(RED_THREADS) k_minmax_apply(const __grid_constant__ NormParams p) {
    const CanvasDesc& c = p.cv[blockIdx.y];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int b = p.b_off + blockIdx.y;
    griddep_wait();                    // the canvases and their min / max are written
    griddep_launch();
    const float gmin = p.mm[2 * b], gmax = p.mm[2 * b + 1];
    const float lo = p.target[2 * b], hi = p.target[2 * b + 1];
    const float scale = gmax > gmin ? (hi - lo) / (gmax - gmin) : 0.f;
    auto map = [&](float v) { return fmaf(v - gmin, scale, lo); };
    for (long long yl = blockIdx.x * RED_WARPS + w; yl < c.h; yl += gridDim.x * RED_WARPS) {
        const int y = (int)yl;
        int xa, xb, va, vb;
        disk_span(c, y, &xa, &xb);
        if (xa >= xb) continue;
        float* row = c.data + (long long)y * c.pitch;
        vector_span(row, xa, xb, &va, &vb);
        for (int x = xa + l; x < va; x += 32) row[x] = map(row[x]);
        for (int x = vb + l; x < xb; x += 32) row[x] = map(row[x]);
        float4* px = reinterpret_cast<float4*>(row + va);
        const int nv = (vb - va) >> 2;
        for (int v0 = l; v0 < nv; v0 += 128) {
            float4 f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (v0 + 32 * u < nv) f[u] = px[v0 + 32 * u];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (v0 + 32 * u < nv) px[v0 + 32 * u] = make_float4(map(f[u].x), map(f[u].y), map(f[u].z), map(f[u].w));
        }
    }
}

int launch_minmax_normalize(zm_plan_t p, const zm_canvas_t* cv, int batch, const float* target, cudaStream_t st) {
    int s = p->ws_scale.grow(sizeof(float) * 2 * (size_t)batch);
    if (s != ZM_OK) return s;
    std::vector<zm_image_t> ims(batch);
    for (int b = 0; b < batch; ++b)
        ims[b] = zm_image_t{cv[b].data, cv[b].height, cv[b].width, cv[b].pitch, cv[b].cx, cv[b].cy, cv[b].radius};
    float* mm = (float*)p->ws_scale.ptr;
    // (k_minmax_apply started early gains nothing here and holds back what follows it:
    // min / max, decode, normalise and score three bands of 886 x 1226 53.4 us, so 50.4)
    s = run_reduce<RED_DISK_MINMAX>(p, ims.data(), nullptr, nullptr, nullptr, batch, nullptr, mm, st, false);
    if (s != ZM_OK) return s;
    static thread_local NormParams np;
    np.mm = mm;
    np.target = target;
    for (int b0 = 0; b0 < batch; b0 += KD_MAX_IMG) {
        const int nb = std::min(KD_MAX_IMG, batch - b0);
        np.b_off = b0;
        int hmax = 1;
        for (int j = 0; j < nb; ++j) {
            np.cv[j] = resolve_canvas(cv[b0 + j]);
            hmax = std::max(hmax, np.cv[j].h);
        }
        ZM_LAUNCH_PDL("k_minmax_apply", k_minmax_apply, dim3(apply_blocks(p, hmax, nb), nb), dim3(RED_THREADS), 0, st, np);
    }
    return ZM_OK;
}

}  // namespace zm

using namespace zm;

static int check_canvases(const zm_canvas_t* cv, int batch) {
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1");
    if (!cv) return set_error(ZM_EINVAL, "canvas array is NULL");
    for (int b = 0; b < batch; ++b) {
        if (!cv[b].data) return set_error(ZM_EINVAL, "canvas %d: data is NULL", b);
        if (cv[b].height < 1 || cv[b].width < 1 || cv[b].pitch < cv[b].width)
            return set_error(ZM_EINVAL, "canvas %d: bad size / pitch", b);
    }
    return ZM_OK;
}

// moments are read, and polar rows written, as float2
static bool aligned8(const void* p) { return ((uintptr_t)p & 7u) == 0; }

extern "C" int zm_reconstruct(zm_plan_t plan, const float* moments, int batch, float* out, unsigned flags,
                              void* stream) {
    if (!plan || !moments || !out) return set_error(ZM_EINVAL, "NULL argument");
    if (!aligned8(moments) || !aligned8(out)) return set_error(ZM_EINVAL, "moments / out must be 8-byte aligned");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1");
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    DeviceGuard g(plan->device);
    return launch_reconstruct(plan, moments, batch, out, flags, (cudaStream_t)stream);
}

extern "C" int zm_reconstruct_errors(zm_plan_t plan, const float* moments, int batch, float* out,
                                     const float* fhat, double* err, unsigned flags, void* stream) {
    if (!plan || !moments || !fhat || !err) return set_error(ZM_EINVAL, "NULL argument");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1");
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    if (!aligned8(moments) || !aligned8(fhat) || (out && !aligned8(out)))
        return set_error(ZM_EINVAL, "moments / fhat / out must be 8-byte aligned");
    DeviceGuard g(plan->device);
    return launch_reconstruct_errors(plan, moments, batch, out, fhat, err, flags, (cudaStream_t)stream);
}

extern "C" int zm_reconstruct_cartesian(zm_plan_t plan, const float* moments, int batch,
                                        const zm_canvas_t* canvases, float* polar_tmp, unsigned flags,
                                        void* stream) {
    if (!plan || !moments || !polar_tmp) return set_error(ZM_EINVAL, "NULL argument");
    if (!aligned8(moments) || !aligned8(polar_tmp))
        return set_error(ZM_EINVAL, "moments / polar_tmp must be 8-byte aligned");
    int s = check_canvases(canvases, batch);
    if (s != ZM_OK) return s;
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    DeviceGuard g(plan->device);
    s = launch_reconstruct(plan, moments, batch, polar_tmp, flags, (cudaStream_t)stream);
    if (s != ZM_OK) return s;
    return launch_polar_to_cart(plan, polar_tmp, batch, canvases, (cudaStream_t)stream);
}

extern "C" int zm_errors(zm_plan_t plan, const zm_image_t* ref, const zm_image_t* test, int batch, double* out,
                         void* stream) {
    if (!plan || !out) return set_error(ZM_EINVAL, "NULL argument");
    int s = check_images(ref, batch);
    if (s == ZM_OK) s = check_images(test, batch);
    if (s != ZM_OK) return s;
    for (int b = 0; b < batch; ++b)
        if (ref[b].height != test[b].height || ref[b].width != test[b].width)
            return set_error(ZM_EINVAL, "image %d: reference and test sizes differ", b);
    DeviceGuard g(plan->device);
    return launch_errors(plan, ref, test, nullptr, nullptr, batch, out, (cudaStream_t)stream);
}

extern "C" int zm_errors_polar(zm_plan_t plan, const float* fhat, const float* frec, int batch, double* out,
                               void* stream) {
    if (!plan || !fhat || !frec || !out) return set_error(ZM_EINVAL, "NULL argument");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1");
    DeviceGuard g(plan->device);
    return launch_errors(plan, nullptr, nullptr, fhat, frec, batch, out, (cudaStream_t)stream);
}

extern "C" int zm_disk_minmax(zm_plan_t plan, const zm_image_t* imgs, int batch, float* out, void* stream) {
    if (!plan || !out) return set_error(ZM_EINVAL, "NULL argument");
    const int s = check_images(imgs, batch);
    if (s != ZM_OK) return s;
    DeviceGuard g(plan->device);
    return launch_disk_minmax(plan, imgs, batch, out, (cudaStream_t)stream);
}

extern "C" int zm_minmax_normalize(zm_plan_t plan, const zm_canvas_t* canvases, int batch, const float* target,
                                   void* stream) {
    if (!plan || !target) return set_error(ZM_EINVAL, "NULL argument");
    const int s = check_canvases(canvases, batch);
    if (s != ZM_OK) return s;
    DeviceGuard g(plan->device);
    return launch_minmax_normalize(plan, canvases, batch, target, (cudaStream_t)stream);
}
