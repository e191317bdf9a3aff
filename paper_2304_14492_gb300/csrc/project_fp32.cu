// Radial projection of Eq. 1 in FP32 on the CUDA cores.
//
// For each m the (K_m x N_rho) x (N_rho x 2B) product
//   D[n][col] = sum_i A[row(m, n)][i] F[m][col][i],   col = 2b + re/im,
// with both operands contiguous in the radial index i.  One CTA = one m, up to
// 32 orders (the K_m orders cut into equal runs), TN columns and all of i: its
// warps share the output tile and take 32-node chunks of i in turn, each
// staging its own chunks (cp.async, two deep, no barrier between warps); the
// warps' partial tiles are added in shared memory in a fixed order and written
// as moments, with the Neumann factor.  So there are no partial sums in device
// memory, no second launch and no workspace.
//
// A lane holds 8 x TN / 8 outputs and multiplies packed pairs of nodes
// (fma.rn.f32x2: even and odd nodes accumulate apart), so a 16-byte
// shared-memory load feeds two instructions per output and the two operands of
// 64 of them cost 12 loads at TN = 32.  Bound: FP32 issue and the copies'
// latency.  16 images of n_max 200 on 512 nodes (334 MFLOP, 34 MB): 58 + 9.5 us
// for a 2 x 4 tile per thread with scalar loads, barriers around every chunk
// and a split over i reduced by a second kernel; now 16 us (cold, serialised).
#include <algorithm>

#include "packed.cuh"
#include "tc_common.cuh"
#include "zm_internal.cuh"

namespace zm {

constexpr int PF_ROWS = 32;              // orders per CTA
constexpr int PF_K = 32;                 // nodes per chunk
constexpr int PF_PITCH = PF_K + 4;       // floats per staged row: 16-byte rows on different banks

struct PfParams {
    const float* A;                      // [P][n_rho], m-major rows
    const float* F;                      // [n_max + 1][ncol][n_rho]
    const int* mrow;
    float* out;                          // [batch][P][2]
    int n_max, n_rho, ncol, P, neumann;
};

template <int BYTES>
__device__ __forceinline__ void pf_copy(uint32_t dst, const float* src, bool on) {
    const int n = on ? BYTES : 0;        // 0: zero-filled
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// rows x 32 nodes from k0 of a row-major operand into this warp's buffer;
// rows past `live` and nodes past n_rho are zero
template <int V>
__device__ __forceinline__ void pf_stage(uint32_t dst, const float* src, int rows, int live, int k0, int n_rho,
                                         int lane) {
    constexpr int PER = PF_K / V;
    for (int e = lane; e < rows * PER; e += 32) {
        const int r = e / PER, k = (e % PER) * V;
        const bool on = r < live && k0 + k < n_rho;
        pf_copy<4 * V>(dst + 4u * (r * PF_PITCH + k), on ? src + (size_t)r * n_rho + k0 + k : src, on);
    }
}

// acc[j][c] += sum over a staged chunk of A[rg + 4 j][.] F[cg + 8 c][.]
template <int TM, int TC>
__device__ __forceinline__ void pf_chunk(const float* a, const float* f, int rg, int cg,
                                         f32x2 (&acc)[8][TC]) {
#pragma unroll 2
    for (int k = 0; k < PF_K; k += 4) {
        ulonglong2 av[TM], fv[TC];
#pragma unroll
        for (int j = 0; j < TM; ++j)
            av[j] = *reinterpret_cast<const ulonglong2*>(a + (rg + 4 * j) * PF_PITCH + k);
#pragma unroll
        for (int c = 0; c < TC; ++c)
            fv[c] = *reinterpret_cast<const ulonglong2*>(f + (cg + 8 * c) * PF_PITCH + k);
#pragma unroll
        for (int j = 0; j < TM; ++j)
#pragma unroll
            for (int c = 0; c < TC; ++c) {
                acc[j][c] = fma2(av[j].x, fv[c].x, acc[j][c]);
                acc[j][c] = fma2(av[j].y, fv[c].y, acc[j][c]);
            }
    }
}

// V: floats per copy (4 where rows start on 16-byte boundaries, else 1).
template <int TN, int V>
__global__ void __launch_bounds__(256) k_project_fp32(const __grid_constant__ PfParams p) {
    constexpr int TC = TN / 8;
    constexpr int BUF = (PF_ROWS + TN) * PF_PITCH;         // floats of one stage
    constexpr int RP = TN + 1;                              // pitch of a partial tile
    static_assert(PF_ROWS * RP <= 2 * BUF, "a partial tile reuses its warp's stages");
    extern __shared__ __align__(16) float pf_sm[];
    const int m = blockIdx.z;
    const int Km = (p.n_max - m) / 2 + 1;
    const int tiles = (Km + PF_ROWS - 1) / PF_ROWS;
    if ((int)blockIdx.y >= tiles) return;
    const int per = (Km + tiles - 1) / tiles;               // equal runs of orders
    const int j0 = blockIdx.y * per, live = min(per, Km - j0);
    const int col0 = blockIdx.x * TN, cols = min(TN, p.ncol - col0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int rg = lane >> 3, cg = lane & 7;
    const int nj = (live + 3) >> 2;                         // rows per lane in use
    const int srow = nj > 4 ? 32 : (nj > 2 ? 16 : 8);       // rows staged
    float* buf = pf_sm + warp * 2 * BUF;
    const uint32_t buf_a = smem_u32(buf);
    const float* A = p.A + (size_t)(p.mrow[m] + j0) * p.n_rho;
    const float* F = p.F + ((size_t)m * p.ncol + col0) * p.n_rho;
    const int chunks = (p.n_rho + PF_K - 1) / PF_K;
    f32x2 acc[8][TC];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int c = 0; c < TC; ++c) acc[j][c] = 0;
    auto stage_a = [&](int ch, int s) {
        if (ch < chunks) pf_stage<V>(buf_a + 4u * s * BUF, A, srow, live, ch * PF_K, p.n_rho, lane);
    };
    auto stage_f = [&](int ch, int s) {
        if (ch < chunks)
            pf_stage<V>(buf_a + 4u * (s * BUF + PF_ROWS * PF_PITCH), F, TN, cols, ch * PF_K, p.n_rho, lane);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the weights are the plan's: their first chunks are on the way before the
    // spectra are known to be written
    stage_a(warp, 0);
    stage_a(warp + W, 1);
    griddep_wait();
    griddep_launch();
    stage_f(warp, 0);
    stage_f(warp + W, 1);
    int s = 0;
    for (int ch = warp; ch < chunks; ch += W, s ^= 1) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const float* a = buf + s * BUF;
        const float* f = a + PF_ROWS * PF_PITCH;
        if (nj > 4) pf_chunk<8, TC>(a, f, rg, cg, acc);
        else if (nj > 2) pf_chunk<4, TC>(a, f, rg, cg, acc);
        else pf_chunk<2, TC>(a, f, rg, cg, acc);
        __syncwarp();
        stage_a(ch + 2 * W, s);
        stage_f(ch + 2 * W, s);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int c = 0; c < TC; ++c) {
            const float2 v = unpack2(acc[j][c]);
            if (j < nj) buf[(rg + 4 * j) * RP + cg + 8 * c] = v.x + v.y;
        }
    __syncthreads();
    const int parts = min(W, chunks);
    for (int e = threadIdx.x; e < live * cols; e += blockDim.x) {
        const int row = e / cols, col = e - row * cols;
        float sum = 0.f;
        for (int w = 0; w < parts; ++w) sum += pf_sm[w * 2 * BUF + row * RP + col];
        const int gcol = col0 + col, n = m + 2 * (j0 + row);
        const float f = (p.neumann && m == 0) ? 0.5f : 1.f;
        p.out[((size_t)(gcol >> 1) * p.P + moment_index(n, m)) * 2 + (gcol & 1)] = sum * f;
    }
}

template <int TN, int V>
static int launch_pf(const PfParams& pp, int dev, cudaStream_t st) {
    const int tiles = (pp.n_max / 2 + 1 + PF_ROWS - 1) / PF_ROWS;
    const int ctiles = (pp.ncol + TN - 1) / TN;
    // eight warps per CTA where that is needed to fill the SMs, else four (the
    // shared memory then holds three CTAs of 32 columns per SM)
    const int W = (long long)(pp.n_max + 1) * tiles * ctiles <= 2 * num_sms(dev) ? 8 : 4;
    const size_t smem = sizeof(float) * W * 2 * (PF_ROWS + TN) * PF_PITCH;
    static SharedMemoryLimit limit;
    ZM_CUDA_TRY(allow_smem(limit, k_project_fp32<TN, V>, dev, smem));
    ZM_LAUNCH_PDL("k_project_fp32", (k_project_fp32<TN, V>), dim3(ctiles, tiles, pp.n_max + 1), dim3(32 * W), smem, st,
                  pp);
    return ZM_OK;
}

int launch_projection_fp32(zm_plan_t p, const float* F, int batch, float* out, unsigned flags, cudaStream_t st) {
    PfParams pp;
    pp.A = p->A32;
    pp.F = F;
    pp.mrow = p->mrow;
    pp.out = out;
    pp.n_max = p->n_max;
    pp.n_rho = p->n_rho;
    pp.ncol = 2 * batch;
    pp.P = p->P;
    pp.neumann = (flags & ZM_NEUMANN) ? 1 : 0;
    const bool vec = (p->n_rho & 3) == 0 && (reinterpret_cast<uintptr_t>(F) & 15) == 0;
    // columns per CTA: the fewest that hold the batch, up to 32 (a wider tile
    // reads the weights once for more images)
    if (pp.ncol <= 8) return vec ? launch_pf<8, 4>(pp, p->device, st) : launch_pf<8, 1>(pp, p->device, st);
    if (pp.ncol <= 16) return vec ? launch_pf<16, 4>(pp, p->device, st) : launch_pf<16, 1>(pp, p->device, st);
    return vec ? launch_pf<32, 4>(pp, p->device, st) : launch_pf<32, 1>(pp, p->device, st);
}

}  // namespace zm
