// Zernike moments by Cartesian summation (Eq. 3-6): the moment integral as a
// sum over the pixels whose centres lie in the unit disk, each weighted by
// its area Delta^2 = 1/r^2 (disk radius r in pixels; Eq. 5's first-order
// approximation, with the prefactor of Eq. 3-5: Eq. 6 prints 1/(pi N^2) where
// Delta = 2/N of Eq. 5 gives 4/N^2 for an N x N image):
//
//   Z_nm = (n + 1) / (pi r^2) sum_{x^2 + y^2 <= 1} f(x, y) R_nm(rho) e^{-j m theta}.
//
// 8-point symmetry (the paper's Fig. 5 timings use it): when the disk centre
// sits at the same offset (0 or 1/2) from the pixel grid in x and y, the
// pixel centres come in orbits of (+-u, +-v), (+-v, +-u) that share rho.  One
// thread takes one representative u >= v >= 0, reads the eight pixels, folds
// them with the factors (-1)^m, (+-j)^m their angles give relative to
// theta_0 = atan2(v, u), and evaluates R_nm(rho) and e^{-j m theta_0} once.
// Other geometries take one thread per pixel.
//
// R_nm(rho) e^{-j m theta} = P_s^{(0,m)}(2 rho^2 - 1) (x - j y)^m, s = (n - m)/2:
// the Jacobi three-term recurrence for P (coefficients per block in shared
// memory; the per-pixel radii are not on any grid, so the Eq. 7 table of the
// polar path does not apply, and the recurrence is stable on [0, 1]) and the
// complex power by repeated squaring (m is the same in every thread).
//
// The kernel is bound by instruction issue, most of it the recurrence, so that
// is cut to the least: P_s is scaled (P_s = +-lambda_s Q_s) so that a step is
// Q_{s+1} = (a_s x + b_s) Q_s + Q_{s-1}, two multiply-adds; a thread takes two
// orbits as one packed pair (fma.rn.f32x2), and a step's coefficients, each
// stored twice, are one 16-byte shared-memory load: three instructions per
// step for two orbits, where an unscaled step took six for one.  One moment
// (100, 36) of a 4000 x 4000 frame: 39 us -> 25 us (cold; 50 MB read).
//
// Sums: FP32 per thread and per block (shuffle tree), FP64 over the blocks in
// a fixed order (deterministic).
#include <algorithm>
#include <cmath>

#include "packed.cuh"
#include "zm_internal.cuh"

namespace zm {

constexpr int CS_MAXP = 4;              // (n, m) pairs per pass
constexpr int CS_MAXS = 512;            // recurrence steps: (n - m) / 2 < 512
constexpr int CS_MAXI = 8;              // images per pass
constexpr int CS_TX = 32, CS_TY = 8;    // threads of a block
constexpr int CS_TC = 2 * CS_TY;        // its tile: CS_TX x CS_TC representatives (or pixels), two per thread
constexpr int CS_THREADS = CS_TX * CS_TY;
constexpr int CS_ROWS = 1024;           // tile rows listed in shared memory (radius up to 16 K pixels)
constexpr float CS_LAMBDA0 = 1024.f;    // scale of P_0: keeps every Q_s below P_s (lambda_s > 1 up to CS_MAXS)

struct CsImage {
    const float* data;
    long long pitch;
    int h, w;
    float cx, cy, r;
    int fold;               // 8-point symmetry: cx, cy on the same offset (0 or 1/2) from the grid
    int amax;               // fold: largest representative index a (a + half <= r)
    int half;               // fold: 1 if that offset is 1/2
    int ox, oy;             // fold: column of offset +u is ox + a, row of offset +v is oy - c
    int tx, tiles;          // tiles per row, tiles in all
};

struct CsParams {
    int np;
    int n[CS_MAXP], m[CS_MAXP];
    int guard[CS_MAXP];     // P_s can leave FP32's range near the centre (see guarded_radial)
    CsImage im[CS_MAXI];
    double* part;           // [image][gridDim.x][np][2]
};

__device__ __forceinline__ float pix(const CsImage& g, int col, int row) {
    return ((unsigned)col < (unsigned)g.w && (unsigned)row < (unsigned)g.h)
               ? __ldg(g.data + (long long)row * g.pitch + col)
               : 0.f;
}

// (x - j y)^m by repeated squaring from the highest bit of m, of two points at once
__device__ __forceinline__ void cpow_conj(f32x2 x, f32x2 y, int m, f32x2* re, f32x2* im) {
    f32x2 wr = pack2(1.f, 1.f), wi = 0;
    if (m > 0) {
        const f32x2 ny = neg2(y);
        wr = x;
        wi = ny;
        for (int e = 30 - __clz(m); e >= 0; --e) {
            const f32x2 u = mul2(wr, wi);
            wr = fma2(wr, wr, neg2(mul2(wi, wi)));
            wi = add2(u, u);
            if ((m >> e) & 1) {
                const f32x2 t = fma2(wr, x, mul2(wi, y));
                wi = fma2(wr, ny, mul2(wi, x));
                wr = t;
            }
        }
    }
    *re = wr;
    *im = wi;
}

// (A_s, B_s, C_s) of P_{s+1} = (A_s x + B_s) P_s - C_s P_{s-1}, the Jacobi
// polynomials P^{(0, beta)} with beta = m (P_0 = 1, P_{-1} = 0)
__device__ __forceinline__ float3 jacobi_coef(int s, int m) {
    const float b = (float)m, sf = (float)s;
    if (s == 0) return make_float3(0.5f * (b + 2.f), -0.5f * b, 0.f);
    const float a = 2.f * sf + b;
    const float d = 2.f * (sf + 1.f) * (sf + b + 1.f);
    return make_float3((a + 1.f) * (a + 2.f) / d, -(a + 1.f) * b * b / (d * a),
                       2.f * sf * (sf + b) * (a + 2.f) / (d * a));
}

// The scaled recurrence of pair (n, m): with lambda_{s+1} = C_s lambda_{s-1}
// (lambda_0 = lambda_1 = CS_LAMBDA0) and P_s = sigma_s lambda_s Q_s, sigma =
// +, +, -, -, repeating,
//   Q_{s+1} = (a_s x + b_s) Q_s + Q_{s-1},  (a_s, b_s) = (-1)^s lambda_s / lambda_{s+1} (A_s, B_s).
// coef[s] = (a_s, a_s, b_s, b_s); returns through *last the factor P_S / Q_S.
// Called by the whole block, `lam` holds CS_MAXS + 1 floats; ends in a barrier.
__device__ void scaled_recurrence(int n, int m, int tid, float4* coef, float* lam, float* last) {
    const int S = (n - m) / 2;
    for (int s = tid; s <= S; s += CS_THREADS) lam[s] = s < 2 ? CS_LAMBDA0 : jacobi_coef(s - 1, m).z;
    __syncthreads();
    if (tid < 2)                           // the even and the odd chain
        for (int s = tid + 2; s <= S; s += 2) lam[s] *= lam[s - 2];
    __syncthreads();
    for (int s = tid; s < S; s += CS_THREADS) {
        const float3 q = jacobi_coef(s, m);
        const float f = ((s & 1) ? -lam[s] : lam[s]) / lam[s + 1];
        coef[s] = make_float4(f * q.x, f * q.x, f * q.y, f * q.y);
    }
    if (tid == 0) *last = (S & 2) ? -lam[S] : lam[S];
    __syncthreads();
}

// Tiles of row c0 of a folded image that hold representatives: columns
// [c0 / CS_TX, ...) up to the last one with a corner inside the disk.
__device__ __forceinline__ int live_tiles(const CsImage& g, int row) {
    const float h = g.half ? 0.5f : 0.f;
    const int c0 = row * CS_TC, t0 = c0 / CS_TX;
    const float y = (float)c0 + h;
    auto on = [&](int tx) {
        const int a0 = tx * CS_TX;
        return a0 <= g.amax && ((float)a0 + h) * ((float)a0 + h) + y * y <= g.r * g.r;
    };
    int t1 = (int)((sqrtf(fmaxf(g.r * g.r - y * y, 0.f)) - h) / (float)CS_TX);     // guess of the last one
    t1 = min(max(t1, t0 - 1), g.tx - 1);
    while (t1 >= t0 && !on(t1)) --t1;
    while (t1 + 1 < g.tx && on(t1 + 1)) ++t1;
    return max(t1 - t0 + 1, 0);
}

// |P_s| reaches C(s + m, s) at the centre, where rho^m is small: past FP32's
// range (log2 C > 120) the plain product would be inf * 0.  Here rho^m goes
// into the recurrence piece by piece, whenever Q has grown, so that nothing
// overflows and only what is truly negligible underflows.  Returns rho^m Q_S;
// the angle's unit factor is left to the caller.
__device__ __noinline__ float guarded_radial(float rho2, int m, int S, const float4* coef) {
    const float rho = sqrtf(rho2);
    auto rpow = [&](int e) {
        float w = 1.f;
        for (float b = rho; e; e >>= 1, b *= b)
            if (e & 1) w *= b;
        return w;
    };
    const int piece = (m + 15) / 16;
    const float w = rpow(piece);
    int left = m;
    const float xx = fmaf(2.f, rho2, -1.f);
    float Q0 = 1.f / CS_LAMBDA0, Q1 = 0.f;
    for (int s = 0; s < S; ++s) {
        const float4 q = coef[s];
        const float Q2 = fmaf(fmaf(q.x, xx, q.z), Q0, Q1);
        Q1 = Q0;
        Q0 = Q2;
        // a step grows Q by less than 2^11 (2 (s + m) + 2 at s = 0)
        while (fmaxf(fabsf(Q0), fabsf(Q1)) > 1.125899907e15f && left >= piece) {    // 2^50
            Q0 *= w;
            Q1 *= w;
            left -= piece;
        }
    }
    for (; left >= piece; left -= piece) Q0 *= w;
    return Q0 * rpow(left);
}

// blockIdx.y = image; the block walks that image's tiles with stride gridDim.x.
// NP = pairs carried per thread (p.np <= NP): fewer accumulators, fewer
// registers, more resident blocks for single moments.  FAST: every image of the
// launch folds, holds all pixels of its orbits and has 32-bit offsets, so no
// pixel is tested against the image and an address is one addition.
template <int NP, bool FAST>
__global__ void __launch_bounds__(CS_THREADS, (NP <= 2 ? (FAST ? 5 : 4) : 3))
    k_cartesian(const __grid_constant__ CsParams p) {
    __shared__ float4 coef[NP][CS_MAXS];
    __shared__ float lam_s[CS_MAXS + 1];
    __shared__ int pre[FAST ? CS_ROWS + 1 : 1];    // live tiles before each tile row
    __shared__ float last_s[NP];
    __shared__ float red[CS_THREADS / 32][NP][2];
    __shared__ float tq[4][CS_TX][CS_TC + 1];      // transposed orbit points of a tile, [point][a][c]
    const int tid = threadIdx.y * CS_TX + threadIdx.x;
    const CsImage& g = p.im[blockIdx.y];
    // FAST: the live tiles in order, so that every block gets the same number
    // (a third of the rectangle's are; handing out the rectangle left some
    // blocks with twice the others' work)
    const int rows = FAST ? g.tiles / g.tx : 0;
    if (FAST)
        for (int r = tid; r < rows; r += CS_THREADS) pre[r + 1] = live_tiles(g, r);
    for (int k = 0; k < p.np; ++k) scaled_recurrence(p.n[k], p.m[k], tid, coef[k], lam_s, &last_s[k]);
    if (FAST) {
        // inclusive scan of the row counts by the first warp
        if (tid < 32) {
            int carry = 0;
            for (int r0 = 0; r0 < rows; r0 += 32) {
                int v = r0 + tid < rows ? pre[r0 + tid + 1] : 0;
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, v, o);
                    if (tid >= o) v += u;
                }
                v += carry;
                if (r0 + tid < rows) pre[r0 + tid + 1] = v;
                carry = __shfl_sync(0xffffffffu, v, 31);
            }
            if (tid == 0) pre[0] = 0;
        }
        __syncthreads();
    }
    const int tiles = FAST ? pre[rows] : g.tiles;
    griddep_wait();                        // the images are written, the partials are free
    griddep_launch();
    const bool fold = FAST || g.fold;
    const int pitch = (int)g.pitch;        // FAST only
    f32x2 acc[NP][2];
#pragma unroll
    for (int k = 0; k < NP; ++k) acc[k][0] = acc[k][1] = 0;
    const float inv_r = 1.f / g.r;

    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        int tyi, txi;
        if (FAST) {
            int lo = 0, hi = rows;          // the last row with pre[row] <= t
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (pre[mid] <= t) lo = mid;
                else hi = mid;
            }
            tyi = lo;
            txi = t - pre[lo] + lo * CS_TC / CS_TX;
        } else {
            tyi = t / g.tx;
            txi = t - tyi * g.tx;
        }
        const int a0 = txi * CS_TX, c0 = tyi * CS_TC;
        const int a = a0 + threadIdx.x;
        // two points per thread: rows c and c + CS_TY of the tile; dead ones
        // sit at (1, 0), where every P_s is 1, with zero pixels
        float f8[2][8], xr[2], yr[2], wgt[2];
        bool live[2];
        if (fold) {
            // tiles wholly below the diagonal or outside the disk (block-uniform)
            const float h = g.half ? 0.5f : 0.f;
            if (!FAST && (a0 + CS_TX - 1 < c0 || a0 > g.amax)) continue;
            if (!FAST && ((float)a0 + h) * ((float)a0 + h) + ((float)c0 + h) * ((float)c0 + h) > g.r * g.r) continue;
            // the representatives (u, v) = (a + h, c + h), u >= v >= 0; their
            // points (+-u, +-v): columns of +-u, rows of +-v (offset -w lies
            // at column ox - w - half, row oy + w + half); issued with the
            // tile's staging loads below, so that one memory latency covers both
            const float x = (float)a + h;
            const int cpu = g.ox + a, cmu = g.ox - a - g.half;
            // repeated points: each distinct pixel of an orbit appears twice
            // (v = 0 or u = v) or eight times (the centre); only tiles on the
            // axis or the diagonal hold such orbits
            const bool edge = c0 == 0 || a0 < c0 + CS_TC;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int c = c0 + threadIdx.y + CS_TY * o;
                const float y = (float)c + h;
                live[o] = a >= c && a <= g.amax && x * x + y * y <= g.r * g.r;
                const int rpv = g.oy - c, rmv = g.oy + c + g.half;
#pragma unroll
                for (int e = 0; e < 8; ++e) f8[o][e] = 0.f;
                if (FAST) {
                    if (live[o]) {
                        const int pp = rpv * pitch + cpu, mp = pp - (2 * a + g.half), dv = (2 * c + g.half) * pitch;
                        f8[o][0] = __ldg(g.data + pp);
                        f8[o][1] = __ldg(g.data + mp);
                        f8[o][2] = __ldg(g.data + (mp + dv));
                        f8[o][3] = __ldg(g.data + (pp + dv));
                    }
                } else if (live[o]) {
                    f8[o][0] = pix(g, cpu, rpv);      // ( u,  v)  angle theta_0
                    f8[o][1] = pix(g, cmu, rpv);      // (-u,  v)  pi - theta_0
                    f8[o][2] = pix(g, cmu, rmv);      // (-u, -v)  pi + theta_0
                    f8[o][3] = pix(g, cpu, rmv);      // ( u, -v)  -theta_0
                }
                wgt[o] = !edge ? 1.f : ((x == 0.f) ? 0.125f : ((y == 0.f || x == y) ? 0.5f : 1.f));
                xr[o] = live[o] ? x * inv_r : 1.f;
                yr[o] = live[o] ? y * inv_r : 0.f;
            }
            // the points (+-v, +-u) of the tile lie in 32 rows (one per a) x 16
            // columns (one per c): stage them through shared memory, sixteen
            // lanes per row, so that the loads read whole 64-byte segments
            __syncthreads();                       // tq of the previous tile is read
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int rr = (tid >> 4) + 16 * o, cc = tid & 15;  // a = a0 + rr, c = c0 + cc
                const int ra = a0 + rr, cb = c0 + cc;
                const int cpv_ = g.ox + cb, cmv_ = g.ox - cb - g.half;
                const int rpu_ = g.oy - ra, rmu_ = g.oy + ra + g.half;
                if (FAST) {
                    // every pixel of an orbit with a, c <= amax is in the image
                    const bool on = ra <= g.amax && cb <= g.amax;
                    const int pp = rpu_ * pitch + cpv_, mp = pp - (2 * cb + g.half), du = (2 * ra + g.half) * pitch;
                    tq[0][rr][cc] = on ? __ldg(g.data + pp) : 0.f;
                    tq[1][rr][cc] = on ? __ldg(g.data + mp) : 0.f;
                    tq[2][rr][cc] = on ? __ldg(g.data + (mp + du)) : 0.f;
                    tq[3][rr][cc] = on ? __ldg(g.data + (pp + du)) : 0.f;
                } else {
                    tq[0][rr][cc] = pix(g, cpv_, rpu_);   // ( v,  u)
                    tq[1][rr][cc] = pix(g, cmv_, rpu_);   // (-v,  u)
                    tq[2][rr][cc] = pix(g, cmv_, rmu_);   // (-v, -u)
                    tq[3][rr][cc] = pix(g, cpv_, rmu_);   // ( v, -u)
                }
            }
            __syncthreads();
            if (!live[0] && !live[1]) continue;
#pragma unroll
            for (int o = 0; o < 2; ++o)
                if (live[o]) {
                    const int cc = threadIdx.y + CS_TY * o;
                    f8[o][4] = tq[0][threadIdx.x][cc];  // ( v,  u)  pi/2 - theta_0
                    f8[o][5] = tq[1][threadIdx.x][cc];  // (-v,  u)  pi/2 + theta_0
                    f8[o][6] = tq[2][threadIdx.x][cc];  // (-v, -u)  -pi/2 - theta_0
                    f8[o][7] = tq[3][threadIdx.x][cc];  // ( v, -u)  -pi/2 + theta_0
                }
        } else {
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int c = c0 + threadIdx.y + CS_TY * o;
                const float x = (float)a - g.cx, y = g.cy - (float)c;
                live[o] = a < g.w && c < g.h && !(x * x + y * y > g.r * g.r);
                f8[o][0] = live[o] ? __ldg(g.data + (long long)c * g.pitch + a) : 0.f;
                wgt[o] = 1.f;
                xr[o] = live[o] ? x * inv_r : 1.f;
                yr[o] = live[o] ? y * inv_r : 0.f;
            }
            if (!live[0] && !live[1]) continue;
        }
        const f32x2 X = pack2(xr[0], xr[1]), Y = pack2(yr[0], yr[1]), wg = pack2(wgt[0], wgt[1]);
        const f32x2 rho2 = fma2(X, X, mul2(Y, Y));
        const f32x2 xx = fma2(pack2(2.f, 2.f), rho2, pack2(-1.f, -1.f));
        f32x2 F[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) F[e] = (fold || e == 0) ? pack2(f8[0][e], f8[1][e]) : 0;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            if (k >= p.np) break;
            const int m = p.m[k], S = (p.n[k] - m) / 2;
            f32x2 Q0, cs, nsn;             // rho^m e^{-j m theta_0} = (x - j y)^m = cs - j sn
            if (p.guard[k]) {
                const float2 r2 = unpack2(rho2);
                Q0 = pack2(guarded_radial(r2.x, m, S, coef[k]), guarded_radial(r2.y, m, S, coef[k]));
                const float i0 = r2.x > 0.f ? 1.f / sqrtf(r2.x) : 0.f, i1 = r2.y > 0.f ? 1.f / sqrtf(r2.y) : 0.f;
                const f32x2 inv = pack2(i0, i1);
                cpow_conj(mul2(X, inv), mul2(Y, inv), m, &cs, &nsn);
            } else {
                f32x2 Q1 = 0;
                Q0 = pack2(1.f / CS_LAMBDA0, 1.f / CS_LAMBDA0);
                const ulonglong2* cf = reinterpret_cast<const ulonglong2*>(coef[k]);
#pragma unroll 4
                for (int s = 0; s < S; ++s) {
                    const ulonglong2 q = cf[s];
                    const f32x2 Q2 = fma2(fma2(q.x, xx, q.y), Q0, Q1);
                    Q1 = Q0;
                    Q0 = Q2;
                }
                cpow_conj(X, Y, m, &cs, &nsn);
            }
            const f32x2 sn = neg2(nsn);
            const f32x2 R = mul2(mul2(Q0, pack2(last_s[k], last_s[k])), wg);
            f32x2 re, im;
            if (fold) {
                // sum_8 f e^{-j m theta} = E A + conj(E) B with E = e^{-j m theta_0},
                //   A = f(u,v) + (-1)^m f(-u,-v) + (-j)^m f(-v,u) + j^m f(v,-u)
                //   B = f(u,-v) + (-1)^m f(-u,v) + (-j)^m f(v,u) + j^m f(-v,-u)
                if (m & 1) {
                    // m = 1 mod 4; the imaginary parts change sign for m = 3 mod 4
                    const f32x2 Ar = sub2(F[0], F[2]), Br = sub2(F[3], F[1]);
                    f32x2 Ai = sub2(F[7], F[5]), Bi = sub2(F[6], F[4]);
                    if (m & 2) {
                        Ai = neg2(Ai);
                        Bi = neg2(Bi);
                    }
                    re = fma2(cs, add2(Ar, Br), mul2(sn, sub2(Ai, Bi)));
                    im = fma2(cs, add2(Ai, Bi), mul2(sn, sub2(Br, Ar)));
                } else {
                    f32x2 A2 = add2(F[5], F[7]), B2 = add2(F[4], F[6]);
                    if (m & 2) {
                        A2 = neg2(A2);
                        B2 = neg2(B2);
                    }
                    const f32x2 Ar = add2(add2(F[0], F[2]), A2), Br = add2(add2(F[3], F[1]), B2);
                    re = mul2(cs, add2(Ar, Br));
                    im = mul2(sn, sub2(Br, Ar));
                }
            } else {
                re = mul2(F[0], cs);
                im = mul2(F[0], nsn);
            }
            acc[k][0] = fma2(R, re, acc[k][0]);
            acc[k][1] = fma2(R, im, acc[k][1]);
        }
    }
    // block sums (shuffle tree, then the warps in order)
    const int warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const float2 u0 = unpack2(acc[k][0]), u1 = unpack2(acc[k][1]);
        float v0 = u0.x + u0.y, v1 = u1.x + u1.y;
        for (int o = 16; o; o >>= 1) {
            v0 += __shfl_xor_sync(0xffffffffu, v0, o);
            v1 += __shfl_xor_sync(0xffffffffu, v1, o);
        }
        if (lane == 0) {
            red[warp][k][0] = v0;
            red[warp][k][1] = v1;
        }
    }
    __syncthreads();
    if (tid < 2 * p.np) {
        const int k = tid >> 1, c = tid & 1;
        float s = 0.f;
        for (int w = 0; w < CS_THREADS / 32; ++w) s += red[w][k][c];
        p.part[(((size_t)blockIdx.y * gridDim.x + blockIdx.x) * p.np + k) * 2 + c] = (double)s;
    }
}

struct CsFinal {
    int blocks, nimg, np;
    float scale[CS_MAXI][CS_MAXP];
    float* out;             // image b, pair k at out[b * stride + (k0 + k) * 2]
    int stride, k0;
};

// out = (n + 1) / (pi r^2) (/ eps_m with Neumann) x the FP64 sum of the block
// partials: one warp per output value, lanes over the blocks with stride 32,
// then the shuffle tree (fixed order)
__global__ void k_cartesian_final(const double* __restrict__ part, const __grid_constant__ CsFinal f) {
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    griddep_wait();                        // the partials are written
    griddep_launch();
    if (e >= f.nimg * f.np * 2) return;
    const int c = e & 1, bk = e >> 1;
    const int b = bk / f.np, k = bk - b * f.np;
    double s = 0.0;
#pragma unroll 8
    for (int j = lane; j < f.blocks; j += 32) s += part[(((size_t)b * f.blocks + j) * f.np + k) * 2 + c];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) f.out[(size_t)b * f.stride + (size_t)(f.k0 + k) * 2 + c] = (float)(s * (double)f.scale[b][k]);
}

// blocks of k_cartesian<NP, FAST> that are resident at once on the device (cached)
template <int NP, bool FAST>
static int cs_blocks_t(int dev) {
    static int cached[64] = {0};
    if (dev >= 0 && dev < 64 && cached[dev]) return cached[dev];
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cartesian<NP, FAST>, CS_THREADS, 0) != cudaSuccess ||
        per < 1)
        per = 1;
    const int n = per * num_sms(dev);
    if (dev >= 0 && dev < 64) cached[dev] = n;
    return n;
}
static int cs_blocks(int dev, int np, bool fast) {
    if (np == 1) return fast ? cs_blocks_t<1, true>(dev) : cs_blocks_t<1, false>(dev);
    if (np == 2) return fast ? cs_blocks_t<2, true>(dev) : cs_blocks_t<2, false>(dev);
    return fast ? cs_blocks_t<CS_MAXP, true>(dev) : cs_blocks_t<CS_MAXP, false>(dev);
}
static int cs_blocks_max(int dev) {
    int n = 0;
    for (int np : {1, 2, CS_MAXP}) n = std::max(n, std::max(cs_blocks(dev, np, true), cs_blocks(dev, np, false)));
    return n;
}

}  // namespace zm

using namespace zm;

extern "C" int zm_cartesian_work_bytes(int batch, int count, unsigned long long* bytes) {
    if (!bytes || batch < 1 || count < 1) return set_error(ZM_EINVAL, "bad arguments");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
    // the block partials of one pass: CS_MAXI images x blocks x CS_MAXP pairs
    *bytes = (unsigned long long)CS_MAXI * cs_blocks_max(dev) * CS_MAXP * 2 * sizeof(double);
    return ZM_OK;
}

extern "C" int zm_cartesian_moments(const zm_image_t* imgs, int batch, const int* nm, int count, float* out,
                                    void* work, unsigned long long work_bytes, unsigned flags, void* stream) {
    if (!nm || !out || !work || count < 1) return set_error(ZM_EINVAL, "NULL argument or count < 1");
    int s = check_images(imgs, batch);
    if (s != ZM_OK) return s;
    for (int k = 0; k < count; ++k) {
        const int n = nm[2 * k], m = nm[2 * k + 1];
        if (n < 0 || m < 0 || m > n || ((n - m) & 1) || (n - m) / 2 >= CS_MAXS)
            return set_error(ZM_EINVAL, "pair %d: (n, m) = (%d, %d) is not a stored moment of order < %d", k, n, m,
                             2 * CS_MAXS);
    }
    unsigned long long need = 0;
    s = zm_cartesian_work_bytes(batch, count, &need);
    if (s != ZM_OK) return s;
    if (work_bytes < need) return set_error(ZM_EINVAL, "work holds %llu bytes, %llu needed", work_bytes, need);
    if ((reinterpret_cast<uintptr_t>(work) & 7u) != 0) return set_error(ZM_EINVAL, "work must be 8-byte aligned");
    int dev = 0;
    ZM_CUDA_TRY(cudaGetDevice(&dev));
    cudaStream_t st = (cudaStream_t)stream;
    double* part = (double*)work;
    for (int b0 = 0; b0 < batch; b0 += CS_MAXI) {
        const int nb = std::min(CS_MAXI, batch - b0);
        CsParams p;
        int max_tiles = 1;
        bool fast = true;
        for (int j = 0; j < nb; ++j) {
            const GeoImage g = resolve(imgs[b0 + j]);
            CsImage& ci = p.im[j];
            ci.data = g.data;
            ci.pitch = g.pitch;
            ci.h = g.h;
            ci.w = g.w;
            ci.cx = g.cx;
            ci.cy = g.cy;
            ci.r = g.r;
            const float fx = g.cx - std::floor(g.cx), fy = g.cy - std::floor(g.cy);
            ci.fold = (fx == fy && (fx == 0.f || fx == 0.5f)) ? 1 : 0;
            ci.half = (fx == 0.5f) ? 1 : 0;
            // offset +u = a + half sits at column floor(cx) + half + a, offset
            // +v = c + half at row floor(cy) - c
            ci.ox = (int)std::floor(g.cx) + ci.half;
            ci.oy = (int)std::floor(g.cy);
            // orbit offsets a + half <= r: a <= amax (exact, in double)
            ci.amax = (int)std::floor((double)g.r - 0.5 * ci.half);
            const int am = ci.amax;
            fast = fast && (ci.fold && (double)g.h * (double)g.pitch < 2147483648.0 && ci.ox - am - ci.half >= 0 && ci.ox + am < g.w && ci.oy - am >= 0 &&
                         ci.oy + am + ci.half < g.h);
            int tx, ty;
            if (ci.fold) {
                const int reps = (int)std::ceil(g.r) + 1;
                tx = (reps + CS_TX - 1) / CS_TX;
                ty = (reps + CS_TC - 1) / CS_TC;
            } else {
                tx = (g.w + CS_TX - 1) / CS_TX;
                ty = (g.h + CS_TC - 1) / CS_TC;
            }
            ci.tx = tx;
            ci.tiles = tx * ty;
            fast = fast && ty <= CS_ROWS;
            max_tiles = std::max(max_tiles, ci.tiles);
        }
        for (int k0 = 0; k0 < count; k0 += CS_MAXP) {
            const int np = std::min(CS_MAXP, count - k0);
            const int NP = np == 1 ? 1 : (np == 2 ? 2 : CS_MAXP);
            // as many blocks as fit on the device at once, shared by the images
            const int grid = std::min(max_tiles, std::max(1, cs_blocks(dev, NP, fast) / nb));
            p.np = np;
            CsFinal f;
            for (int k = 0; k < np; ++k) {
                p.n[k] = nm[2 * (k0 + k)];
                p.m[k] = nm[2 * (k0 + k) + 1];
                const double sm = (p.n[k] + p.m[k]) / 2, ss = (p.n[k] - p.m[k]) / 2;
                p.guard[k] = (std::lgamma(sm + 1.0) - std::lgamma(ss + 1.0) - std::lgamma(p.m[k] + 1.0)) > 120.0 * 0.6931;
                for (int j = 0; j < nb; ++j) {
                    const double eps = ((flags & ZM_NEUMANN) && p.m[k] == 0) ? 2.0 : 1.0;
                    const double r = p.im[j].r;
                    f.scale[j][k] = (float)((p.n[k] + 1) / (3.14159265358979323846 * r * r) / eps);
                }
            }
            p.part = part;
            const dim3 gd(grid, nb), bd(CS_TX, CS_TY);
            auto kernel = NP == 1   ? (fast ? k_cartesian<1, true> : k_cartesian<1, false>)
                          : NP == 2 ? (fast ? k_cartesian<2, true> : k_cartesian<2, false>)
                                    : (fast ? k_cartesian<CS_MAXP, true> : k_cartesian<CS_MAXP, false>);
            ZM_LAUNCH_PDL("k_cartesian", kernel, gd, bd, 0, st, p);
            f.blocks = grid;
            f.nimg = nb;
            f.np = np;
            f.out = out + (size_t)b0 * count * 2;
            f.stride = count * 2;
            f.k0 = k0;
            const int tot = nb * np * 2;                         // one warp each
            ZM_LAUNCH_PDL("k_cartesian_final", k_cartesian_final, dim3((tot + 3) / 4), dim3(128), 0, st,
                          (const double*)part, f);
        }
    }
    return ZM_OK;
}
