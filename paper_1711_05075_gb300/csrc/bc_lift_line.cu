// The lifted correlation's 4D NUFFT (bc_lift_nufft.cu) for shapes whose support
// box is narrower than the period on every axis: spreading into row pairs, the z
// and y transforms of every (r, x) plane in one launch (k_zy, bc_front.cu), the x
// transforms on warp-private lines, and one pass for the r transforms of both
// spectra, the collapse and the inverse x transform.
//
// Box element i of an axis sits at position i of its line; with the lowest cells
// lo_A, lo_B of the two boxes the product of the spectra is then off by
//     exp(2 pi i (m . (lo_B - lo_A) / n + m_r (lo_rB - lo_rA) / n_r)),
// whose spatial part the last pass applies per mode and whose r part is folded
// into the sections' phases.  (The half-period shift of the coordinates cancels.)
//
// A call at N = 128, N_r = 32 with 5,000 + 5,000 knots: 0.74 ms, against
// 1.95 ms of the passes in bc_lift_nufft.cu (spreading 33 us a shape, z and y
// 108, x 55, the last pass 206: instruction bound).
#include <algorithm>
#include <climits>

#include "bc_lift4.h"
#include "bc_passes.cuh"
#include "bc_umma.cuh"
#include "bc_wfft.cuh"

namespace bc {

namespace {

constexpr int LW8 = 8; // window width

// 4W window weights by the lanes; then a lane owns one 16-byte piece of the (y, z)
// cross-section -- a row pair and two z cells -- for all W x W cells along r and x.
__global__ void __launch_bounds__(256)
k_lx_spread(const float4 *__restrict__ knots, int n, Lift4Rot rot, int mirror, int ns, int nr, double inv_p, double inv_pr,
            Lift4Box bx, const float *__restrict__ consts, float *G)
{
    constexpr int W = LW8, C = W / 2 + 1;
    __shared__ float wts[8][4][W + 4]; // [axis][1 + offset], zero at both ends
    __shared__ int e0s[8][4];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, a = lane / W, t = lane - a * W;
    float kc[KB_NC];
    kb_load(consts, t, kc);
    for (int k = lane; k < 4 * (W + 4); k += 32) (&wts[wib][0][0])[k] = 0.f;
    __syncwarp();
    const int np = bx.b[1] >> 1, bz = bx.b[2];
    const long long xs = (long long)np * bz * 2, rs = xs * bx.b[0];
    const int pr = lane / C, zc = lane - pr * C;
    for (int i = blockIdx.x * 8 + wib; i < n; i += gridDim.x * 8) {
        const float4 c = knots[i];
        const double u = lift4_coord(c, a, rot.R, mirror, ns, nr, inv_p, inv_pr);
        const int g0 = (int)ceil(u - 0.5 * W);
        wts[wib][a][1 + t] = kb_poly(kc, (float)(u - g0 - (0.5 * W - 1.0)));
        if (t == 0) e0s[wib][a] = g0 - bx.lo[a];
        __syncwarp();
        const int ex = e0s[wib][0], ey = e0s[wib][1], ez = e0s[wib][2], er = e0s[wib][3], oy = ey & 1, oz = ez & 1;
        if (lane < C * C && 2 * pr - oy < W && 2 * zc - oz < W) {
            const float *wy = &wts[wib][1][1 + 2 * pr - oy], *wz = &wts[wib][2][1 + 2 * zc - oz];
            const float4 f = make_float4(wy[0] * wz[0], wy[1] * wz[0], wy[0] * wz[1], wy[1] * wz[1]);
            float *cr = G + er * rs + ex * xs + ((long long)((ey >> 1) + pr) * bz + 2 * ((ez >> 1) + zc)) * 2;
            for (int tr = 0; tr < W; tr++, cr += rs) {
                const float wr = wts[wib][3][1 + tr];
                float *cell = cr;
#pragma unroll
                for (int tx = 0; tx < W; tx++, cell += xs) {
                    const float w = wr * wts[wib][0][1 + tx];
                    atomicAdd(reinterpret_cast<float4 *>(cell), make_float4(w * f.x, w * f.y, w * f.z, w * f.w));
                }
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ x
// Item: (i_r, m_z, XL consecutive j_y): the b0 rows of 64 bytes of a y1 block by one
// bulk copy, two items ahead; every warp transforms its lines and stores the N modes
// of each, X1[m_z][j_y][i_r][j_x].
template <int NF>
struct LX {
    static constexpr int LW = wf_full(NF), WARPS = XL / LW, THREADS = WARPS * 32, STAGES = 3;
    static size_t smem(int b0) { return 8 * ((size_t)XL * WF<NF>::ES) + (size_t)STAGES * b0 * XL * 8 + 64; }
};

template <int NF>
__global__ void __launch_bounds__(LX<NF>::THREADS, 512 / LX<NF>::THREADS)
k_lx_x(const float2 *__restrict__ y1, int b0, int bR, const float2 *__restrict__ tw, float2 *X1, int *err)
{
    using F = WF<NF>;
    constexpr int R0 = F::R0, N = F::N, H = F::H, LW = F::LW, nch = N / XL, STAGES = LX<NF>::STAGES;
    extern __shared__ float4 sm4[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2 *E = reinterpret_cast<float2 *>(sm4) + warp * F::EW;
    float2 *ring = reinterpret_cast<float2 *>(sm4) + XL * F::ES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + (size_t)STAGES * b0 * XL);
    volatile int *stop = reinterpret_cast<volatile int *>(bars + STAGES);
    const uint32_t FULL = smem_addr(bars), bytes = (uint32_t)b0 * XL * 8;
    if (threadIdx.x == 0) {
        for (int k = 0; k < STAGES; k++) mbar_init(FULL + 8 * k, 1);
        *stop = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    float2 w[16];
    wf_twiddles<NF>(tw, lane, w);
    __syncthreads();
    const int items = bR * H * nch, s = lane / R0, j = lane - s * R0, qx = (b0 + 63) >> 6;
    int issued = 0; // thread 0: copies issued
    auto fetch = [&](int it, int st) {
        if (it >= items) return;
        issued++;
        mbar_expect_tx(FULL + 8 * st, bytes);
        bulk_g2s(smem_addr(ring + (size_t)st * b0 * XL), y1 + (long long)it * b0 * XL, bytes, FULL + 8 * st);
    };
    if (threadIdx.x == 0)
        for (int k = 0; k < STAGES - 1; k++) fetch((int)blockIdx.x + k * (int)gridDim.x, k);
    int st = 0, par = 0;
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        // the stage of the previous item is free (the barrier that ended it)
        if (threadIdx.x == 0) fetch(it + (STAGES - 1) * (int)gridDim.x, (st + STAGES - 1) % STAGES);
        if (!__syncthreads_and(umma_wait(FULL + 8 * st, par, stop, err, LIFT_ERR_LINE))) break;
        const float2 *T = ring + (size_t)st * b0 * XL;
        const int ir = it / (H * nch), rem = it - ir * H * nch, mz = rem / nch, jy0 = (rem - mz * nch) * XL;
        wf_first_any<NF>(E, lane, qx, [&](int sl, int ix, bool inside) {
            return inside || ix < b0 ? T[ix * XL + xl_place(warp * LW + sl, ix)] : make_float2(0.f, 0.f);
        });
        __syncwarp();
        float2 o[16];
        wf_last<NF>(E, lane, w, o);
        if (lane < F::LIVE) {
            float2 *dst = X1 + (((long long)mz * N + jy0 + warp * LW + s) * bR + ir) * N + j;
#pragma unroll
            for (int r = 0; r < 8; r++) dst[R0 * r] = o[r < 4 ? r : r + 8];
        }
        if (++st == STAGES) {
            st = 0;
            par ^= 1;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) // after an expired wait, copies still in flight land (bounded)
        for (int k = max(0, issued - STAGES); k < issued; k++) {
            const uint64_t t0 = global_ns();
            while (!mbar_test(FULL + 8 * (k % STAGES), (k / STAGES) & 1) && global_ns() - t0 < UMMA_WAIT_NS) {
            }
        }
}

// ------------------------------------------------------------------ r, collapse, inverse x
// W[m_z][|m_y|][k][|m_x|] = cone(|m|^2, k)^2 (D_x D_y D_z D_r)^2 / 4 (the 4: both spectra
// carry k_zy's factor 2), k the kept modes of r in FFT order, zero on the lower-edge one.
__global__ void k_lx_weights(int N, int Nr, const float *__restrict__ dxs, const float *__restrict__ drr,
                             const float2 *__restrict__ cone, float2 *w)
{
    const int A = N / 2 + 1;
    const long long total = (long long)(N / 2) * A * Nr * A;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int mx = (int)(e % A), k = (int)((e / A) % Nr), my = (int)((e / ((long long)A * Nr)) % A);
        const int mz = (int)(e / ((long long)A * Nr * A));
        const float2 f = cone[(long long)(mx * mx + my * my + mz * mz) * Nr + k];
        const double d = (double)dxs[mx] * dxs[my] * dxs[mz] * drr[k], s = k == Nr / 2 ? 0.0 : 0.25 * d * d;
        w[e] = make_float2((float)(((double)f.x * f.x - (double)f.y * f.y) * s), (float)(2.0 * f.x * f.y * s));
    }
}

// The kept outputs k1 + R1 k2, k2 = 0, 1, 6, 7 of the length 8 R1 transform of x[i] =
// T[i N], i < b, at one k1: over i = j + 8 r first (exp(-2 pi i r k1 / R1)), the
// twiddles wj[j] = exp(-2 pi i j k1 / (8 R1)), then the radix-8 over j.  wr: exp(-2 pi i
// k / (8 R1)).  Every value read is the same for the whole warp or one per lane.
template <int N, int R1>
__device__ __forceinline__ void lx_quarter(const float2 *T, int b, int k1, const float2 *wr, const float2 (&wj)[8],
                                           float2 (&o)[4])
{
    float2 t[8];
#pragma unroll
    for (int j = 0; j < 8; j++) t[j] = j < b ? T[j * N] : make_float2(0.f, 0.f);
    for (int r = 1; 8 * r < b; r++) {
        const float2 w = wr[(8 * r * k1) & (8 * R1 - 1)];
        const float2 *Tr = T + 8 * r * N;
        const int left = b - 8 * r;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            if (j >= left) break;
            const float2 x = Tr[j * N];
            t[j].x = fmaf(x.x, w.x, fmaf(-x.y, w.y, t[j].x));
            t[j].y = fmaf(x.x, w.y, fmaf(x.y, w.x, t[j].y));
        }
    }
#pragma unroll
    for (int j = 1; j < 8; j++) t[j] = cmul(t[j], wj[j]);
    dft_small<8, false>(t);
    o[0] = t[0];
    o[1] = t[1];
    o[2] = t[6];
    o[3] = t[7];
}

// Item: (m_z, XL consecutive j_y); two threads per j_x, each half of the k1.  Per j_y
// the planes A[i_r][j_x] and B[i_r][j_x] (one bulk copy each, the next j_y's ahead);
// the threads transform their mode along r, four outputs at a time, and sum over the
// kept modes
//     G_A conj(G_B) W exp(2 pi i m_r (r_s / P_r + (lo_rB - lo_rA) / n_r))   per section s,
// then the spatial phase, sign and scale follow (zero on the Nyquist planes).  The
// item's XL lines along x are inverse transformed by the warps and leave as
// h[s][k_x][m_z][j_y].
__host__ __device__ constexpr int rx_line(int N) { return (N / 8 * WI_ROW > N ? N / 8 * WI_ROW : N) | 1; } // a line's values or exchange tile
__host__ __device__ constexpr size_t rx_smem(int N, int NRK, int NS, int bA, int bB)
{
    return 8 * ((size_t)NS * XL * rx_line(N) * 2 + N + NS * NRK + 2 * NRK + 2 * (size_t)(bA + bB) * N) + 64;
}

template <int N, int NRK, int NS> // NRK: kept modes along r (N_r)
__global__ void __launch_bounds__(2 * N, N == 32 ? 8 : 2)
k_lx_rx(const float2 *__restrict__ XA, const float2 *__restrict__ XB, int bA, int bB, int4 dlo, const float2 *__restrict__ wts,
        const float *__restrict__ slices, int nslices, double period_r, float scale, const float2 *__restrict__ tws,
        const float2 *__restrict__ twr, float2 *h, int *err)
{
    constexpr int R0 = N / 8, NR = 2 * NRK, R1 = NR / 8, H = N / 2, A = H + 1, nch = N / XL, n = 2 * N, LINE = rx_line(N);
    extern __shared__ float4 sm4[];
    float2 *lines = reinterpret_cast<float2 *>(sm4); // [NS][XL][LINE]: modes, then the transformed lines
    float2 *ex = lines + NS * XL * LINE;             // [NS][XL][LINE]: partial sums, exchange tiles
    float2 *twN = ex + NS * XL * LINE;               // exp(-2 pi i k / N)
    float2 *ph = twN + N;                            // [NS][NRK]
    float2 *wr = ph + NS * NRK;                      // exp(-2 pi i k / n_r), k < n_r
    float2 *stg = wr + NR;                           // two stages of A and B planes
    const int sf2 = (bA + bB) * N;
    uint64_t *bars = reinterpret_cast<uint64_t *>(stg + 2 * (size_t)sf2);
    volatile int *stop = reinterpret_cast<volatile int *>(bars + 2);
    const uint32_t FULL = smem_addr(bars);
    const int grp = threadIdx.x / N, jx = threadIdx.x - grp * N, mx = jx < H ? jx : jx - N, ax = mx < 0 ? -mx : mx;
    if (threadIdx.x == 0) {
        mbar_init(FULL, 1);
        mbar_init(FULL + 8, 1);
        *stop = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (grp == 0) twN[jx] = tws[2 * jx];
    for (int k = threadIdx.x; k < NR; k += 2 * N) wr[k] = twr[k];
    for (int e = threadIdx.x; e < NS * NRK; e += 2 * N) {
        const int s = e / NRK, k = e - s * NRK, m = k < NRK / 2 ? k : k - NRK;
        float2 v = make_float2(0.f, 0.f);
        if (s < nslices) {
            double arg = m * ((double)slices[s] / period_r + (double)dlo.w / NR), sn, cs;
            arg -= rint(arg);
            sincospi(2.0 * arg, &sn, &cs);
            v = make_float2((float)cs, (float)sn);
        }
        ph[e] = v;
    }
    __syncthreads();
    const int items = H * nch, total = ((items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x) * XL;
    // unit u of the block: item blockIdx + (u / XL) gridDim, its j_y number u mod XL
    int issued = 0; // thread 0: units fetched
    auto fetch = [&](int u) {
        if (u >= total) return;
        issued++;
        const int it = blockIdx.x + (u / XL) * gridDim.x, mz = it / nch, jy = (it - mz * nch) * XL + u % XL, st = u & 1;
        const long long row = (long long)mz * N + jy;
        mbar_expect_tx(FULL + 8 * st, (uint32_t)sf2 * 8);
        bulk_g2s(smem_addr(stg + (size_t)st * sf2), XA + row * bA * N, (uint32_t)bA * N * 8, FULL + 8 * st);
        bulk_g2s(smem_addr(stg + (size_t)st * sf2 + bA * N), XB + row * bB * N, (uint32_t)bB * N * 8, FULL + 8 * st);
    };
    if (threadIdx.x == 0) fetch(0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int u = 0; u < total; u++) {
        const int it = blockIdx.x + (u / XL) * gridDim.x, mz = it / nch, c = u % XL, jy = (it - mz * nch) * XL + c;
        if (threadIdx.x == 0) fetch(u + 1); // its stage was read before the barrier inside unit u - 1
        if (!__syncthreads_and(umma_wait(FULL + 8 * (u & 1), (u >> 1) & 1, stop, err, LIFT_ERR_LINE))) break;
        const float2 *TA = stg + (size_t)(u & 1) * sf2 + jx, *TB_ = TA + bA * N;
        const int my = jy < H ? jy : jy - N;
        const float2 *wt = wts + ((long long)mz * A + (my < 0 ? -my : my)) * NRK * A + ax;
        float2 acc[NS];
#pragma unroll
        for (int s = 0; s < NS; s++) acc[s] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int k1 = grp; k1 < R1; k1 += 2) {
            float2 wv[4], lj[8], ga[4], gb[4];
#pragma unroll
            for (int q = 0; q < 4; q++) wv[q] = __ldg(wt + (k1 + R1 * q) * A); // kept mode k1 + R1 q in FFT order
#pragma unroll
            for (int j = 1; j < 8; j++) lj[j] = wr[(j * k1) & (NR - 1)];
            lx_quarter<N, R1>(TA, bA, k1, wr, lj, ga);
            lx_quarter<N, R1>(TB_, bB, k1, wr, lj, gb);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float2 p = cmul(cmulc(ga[q], gb[q]), wv[q]);
#pragma unroll
                for (int s = 0; s < NS; s++) acc[s] = cadd(acc[s], cmul(p, ph[s * NRK + k1 + R1 * q]));
            }
        }
        // the second half's sums join the first's (two places in turn: a thread of it may be
        // in the next unit while the first half still reads)
        float2 *half = ex + (u & 1) * LINE + jx;
        if (grp) {
#pragma unroll
            for (int s = 0; s < NS; s++) half[s * XL * LINE] = acc[s];
        }
        __syncthreads();
        if (grp == 0) {
            // exp(2 pi i m . (lo_B - lo_A) / n), (-1)^(m_x + m_y + m_z), scale
            const int k = (mx * dlo.x + my * dlo.y + mz * dlo.z) % n;
            const float2 sp = tws[k <= 0 ? -k : n - k];
            const float sg = (jx == H || jy == H) ? 0.f : ((mx + my + mz) & 1) ? -scale : scale;
#pragma unroll
            for (int s = 0; s < NS; s++)
                lines[(s * XL + c) * LINE + jx] = cscale(cmul(cadd(acc[s], half[s * XL * LINE]), sp), sg);
        }
        if (c == XL - 1) { // the item's lines are complete
            __syncthreads();
            const int nl = nslices * XL;
            // a warp takes four lines at a time: R0 first-stage butterflies each, then 8
            for (int l0 = 4 * warp; l0 < nl; l0 += 4 * (2 * N / 32)) {
                for (int e = lane; e < 4 * R0; e += 32) {
                    const int l = l0 + e / R0, j = e % R0;
                    float2 v[8];
#pragma unroll
                    for (int r = 0; r < 8; r++) v[r] = lines[l * LINE + j + R0 * r];
                    wi_first<R0>(v, ex + l * LINE, j);
                }
                __syncwarp();
                const int l = l0 + (lane >> 3), jj = lane & 7;
                float2 o[R0];
                wi_last<R0>(ex + l * LINE, jj, twN, o);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < R0; r++) lines[l * LINE + jj + 8 * r] = o[r];
            }
            __syncthreads();
            const int jy0 = jy - (XL - 1);
            for (int e = threadIdx.x; e < nl * N; e += 2 * N) {
                const int cc = e % XL, kx = (e / XL) % N, s = e / (XL * N);
                h[((long long)s * N + kx) * H * N + (long long)mz * N + jy0 + cc] = lines[(s * XL + cc) * LINE + kx];
            }
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) // after an expired wait, copies still in flight land (bounded)
        for (int k = max(0, issued - 2); k < issued; k++) {
            const uint64_t t0 = global_ns();
            while (!mbar_test(FULL + 8 * (k & 1), (k >> 1) & 1) && global_ns() - t0 < UMMA_WAIT_NS) {
            }
        }
}

constexpr size_t LX_SMEM = 220 * 1024; // of k_lx_rx, at most (lift4_line_fits)

template <int NF>
cudaError_t lx_x(const float2 *y1, int b0, int bR, const float2 *tw, float2 *X1, int *err, int nsm, cudaStream_t s)
{
    const size_t smem = LX<NF>::smem(b0);
    cudaError_t e = set_smem(k_lx_x<NF>, LX<NF>::smem(NF)); // b0 < NF
    if (e != cudaSuccess) return e;
    k_lx_x<NF><<<resident_blocks(k_lx_x<NF>, smem, nsm, LX<NF>::THREADS), LX<NF>::THREADS, smem, s>>>(y1, b0, bR, tw, X1, err);
    return cudaGetLastError();
}

template <int N, int NRK, int NS>
cudaError_t lx_rx(const float2 *XA, const float2 *XB, int bA, int bB, int4 dlo, const Lift4Tables &t, const float *slices,
                  int nslices, double period_r, float scale, float2 *h, int *err, int nsm, cudaStream_t s)
{
    const size_t smem = rx_smem(N, NRK, NS, bA, bB);
    cudaError_t e = set_smem(k_lx_rx<N, NRK, NS>, LX_SMEM);
    if (e != cudaSuccess) return e;
    k_lx_rx<N, NRK, NS><<<resident_blocks(k_lx_rx<N, NRK, NS>, smem, nsm, 2 * N), 2 * N, smem, s>>>(
        XA, XB, bA, bB, dlo, t.wts, slices, nslices, period_r, scale, t.tw_s, t.tw_r, h, err);
    return cudaGetLastError();
}

// sections beyond four take several passes over the spectra (each at most LX_NS sections)
constexpr int LX_NS = 4;

template <int N, int NRK>
cudaError_t lx_rx_ns(const float2 *XA, const float2 *XB, int bA, int bB, int4 dlo, const Lift4Tables &t, const float *slices,
                     int nslices, double period_r, float scale, float2 *h, int *err, int nsm, cudaStream_t s)
{
    for (int s0 = 0; s0 < nslices; s0 += LX_NS) {
        const int ns = std::min(LX_NS, nslices - s0);
        float2 *hs = h + (size_t)s0 * N * N * (N / 2);
        cudaError_t e = ns == 1 ? lx_rx<N, NRK, 1>(XA, XB, bA, bB, dlo, t, slices + s0, ns, period_r, scale, hs, err, nsm, s)
                                : lx_rx<N, NRK, LX_NS>(XA, XB, bA, bB, dlo, t, slices + s0, ns, period_r, scale, hs, err, nsm, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int N>
cudaError_t lx_rx_nr(int Nr, const float2 *XA, const float2 *XB, int bA, int bB, int4 dlo, const Lift4Tables &t,
                     const float *slices, int nslices, double period_r, float scale, float2 *h, int *err, int nsm, cudaStream_t s)
{
    switch (Nr) {
    case 16: return lx_rx_ns<N, 16>(XA, XB, bA, bB, dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    case 32: return lx_rx_ns<N, 32>(XA, XB, bA, bB, dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    case 64: return lx_rx_ns<N, 64>(XA, XB, bA, bB, dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace

size_t lift4_weight_bytes(int N, int Nr)
{
    return sizeof(float2) * (size_t)(N / 2) * (N / 2 + 1) * Nr * (N / 2 + 1);
}

cudaError_t lift4_build_weights(const Lift4Tables &t, int N, int Nr, const float2 *cone, cudaStream_t s)
{
    k_lx_weights<<<4096, 256, 0, s>>>(N, Nr, t.deconv_s, t.deconv_r, cone, t.wts);
    return cudaGetLastError();
}

// Whether boxes narrower than the period take these passes: the last one's shared memory
// holds two stages of both shapes' planes of one (m_z, j_y), and the passes are the faster
// ones.  They save on the transforms of the box (bX bY z lines, bX N/2 y lines and N N/2 x
// lines per cell along r), but repeat the r transforms for every LX_NS sections.
//  - Fewer items of the last pass than SMs (N = 32): a call waits for one block's chain,
//    which grows with N_r and the repetitions.  300 + 300 knots: N_r = 16, 12 sections 215
//    us (general passes 231), 16 sections 239 (243); N_r = 32, 4 sections 190 (221), 5
//    sections 233 (224), 16 sections 341 (258); N_r = 64, 1 section 264 (223).
//  - Otherwise the repetitions are weighed against the lines saved (measured at N = 64, 96
//    and 128 on boxes of a ninth and half of the period, line form / general in ms at N =
//    128, N_r = 64, half: 5 sections 2.30 / 3.03, 9 sections 3.17 / 3.42, 13 sections 4.05 /
//    3.55; ninth: 4 sections 1.19 / 1.94, 5 sections 2.00 / 2.07, 9 sections 2.88 / 2.46; at
//    N_r = 32, ninth, 16 sections 1.61 / 1.83).
bool lift4_line_fits(int N, int Nr, const Lift4Box &ba, const Lift4Box &bb, int nslices, int nsm)
{
    if (rx_smem(N, Nr, nslices > 1 ? LX_NS : 1, ba.b[3], bb.b[3]) > LX_SMEM) return false;
    const int turns = (nslices + LX_NS - 1) / LX_NS;
    if (N / 2 * (N / XL) < nsm) return turns * Nr <= 48;
    auto lines = [&](const Lift4Box &b) { return (double)b.b[0] * (b.b[1] + N / 2) + (double)N * (N / 2); };
    return 0.5 * (lines(ba) + lines(bb)) >= (turns - 1) * (double)Nr * Nr / 4300.0 * N * N;
}

cudaError_t lift4_line_spectrum(const Lift4Tables &t, int N, int Nr, const float4 *knots, int n, const Lift4Rot &rot,
                                int mirror, double ip, double ipr, const Lift4Box &bx, const InstPlan *dplan,
                                const InstDesc *dinst, float *G, size_t clean, float2 *y1, float2 *X1, int *err, int nsm, cudaStream_t s)
{
    const size_t cells = lift4_cells(bx);
    cudaError_t e;
    if (cells > clean && (e = cudaMemsetAsync(G + clean, 0, sizeof(float) * (cells - clean), s)) != cudaSuccess) return e;
    k_lx_spread<<<std::min((n + 7) / 8, 65535), 256, 0, s>>>(knots, n, rot, mirror, 2 * N, 2 * Nr, ip, ipr, bx, t.consts, G);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    Geometry g{};
    g.N = N;
    g.n = 2 * N;
    g.L = bx.b[3];
    Tables tb{};
    tb.tw_n = t.tw_s;
    if ((e = launch_zy(g, tb, dinst, 1, dplan, G, y1, bx.b[1], nsm, s, clean == 0)) != cudaSuccess) return e;
    switch (N) {
    case 32: return lx_x<64>(y1, bx.b[0], bx.b[3], t.tw_s, X1, err, nsm, s);
    case 64: return lx_x<128>(y1, bx.b[0], bx.b[3], t.tw_s, X1, err, nsm, s);
    case 96: return lx_x<192>(y1, bx.b[0], bx.b[3], t.tw_s, X1, err, nsm, s);
    case 128: return lx_x<256>(y1, bx.b[0], bx.b[3], t.tw_s, X1, err, nsm, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t lift4_line_collapse(const Lift4Tables &t, int N, int Nr, const float2 *XA, const float2 *XB, const Lift4Box &ba,
                                const Lift4Box &bb, const float *slices, int nslices, double period_r, float scale, float2 *h,
                                int *err, int nsm, cudaStream_t s)
{
    const int4 dlo = make_int4(bb.lo[0] - ba.lo[0], bb.lo[1] - ba.lo[1], bb.lo[2] - ba.lo[2], bb.lo[3] - ba.lo[3]);
    switch (N) {
    case 32: return lx_rx_nr<32>(Nr, XA, XB, ba.b[3], bb.b[3], dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    case 64: return lx_rx_nr<64>(Nr, XA, XB, ba.b[3], bb.b[3], dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    case 96: return lx_rx_nr<96>(Nr, XA, XB, ba.b[3], bb.b[3], dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    case 128: return lx_rx_nr<128>(Nr, XA, XB, ba.b[3], bb.b[3], dlo, t, slices, nslices, period_r, scale, h, err, nsm, s);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace bc
