// Single-configuration queries (Sec. 4.1, Eq. (single)): the correlation at
// arbitrary translations from a truncated set of modes of its spectrum,
//     g(R, t) = P^-3 sum_{m in M'} w_m Re( g^(m) exp(2 pi i m.t / P) ),
// with g^(m) = f^_A(m) conj(f^_RB(m)) (Eq. (ccghat)), M' the first m' modes of
// the canonical half space ordered outward from the origin, and w_m = 1 for
// m = 0, 2 otherwise (each mode stands for itself and its conjugate -m).
#include <algorithm>
#include <cstdint>

#include "bc_passes.cuh"

namespace bc {

// g^ at the listed modes from two half spectra F[jx][jy][mz] (line: F[mz][jy][jx];
// jx, jy in FFT order, mz in [0, N/2)); mode i = (m_x, m_y, m_z, w).
__global__ void k_query_gather(const float2 *__restrict__ fa, const float2 *__restrict__ fb, const int4 *__restrict__ modes,
                               int count, int N, bool line_a, bool line_b, float2 *ghat)
{
    const int H = N / 2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const int4 m = modes[i];
        const int jx = m.x < 0 ? m.x + N : m.x, jy = m.y < 0 ? m.y + N : m.y;
        const long long o = ((long long)jx * N + jy) * H + m.z, ol = ((long long)m.z * N + jy) * N + jx;
        const float2 a = fa[line_a ? ol : o], b = fb[line_b ? ol : o];
        ghat[i] = cmulc(a, b);
    }
}

// The records of k_query_lines: value e of all records is the weighted g^ of mode src[e]
// (zero for -1); their heads follow the indices.
__global__ void k_query_records(const float2 *__restrict__ ghat, const int4 *__restrict__ modes, const int *__restrict__ src,
                                int ngroups, float2 *out)
{
    constexpr int PER = QL_HEAD + QL_VALUES;
    const float2 *heads = reinterpret_cast<const float2 *>(src + (size_t)ngroups * QL_VALUES);
    const int total = ngroups * PER;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int g = e / PER, k = e - g * PER;
        float2 v;
        if (k < QL_HEAD) {
            v = heads[g * QL_HEAD + k];
        } else {
            const int i = src[g * QL_VALUES + k - QL_HEAD];
            v = i < 0 ? make_float2(0.f, 0.f) : ghat[i];
            const float w = i < 0 ? 0.f : (float)modes[i].w;
            v = make_float2(w * v.x, w * v.y);
        }
        out[e] = v;
    }
}

cudaError_t launch_query_records(const float2 *ghat, const int4 *modes, const int *src, int ngroups, QlGroup *out,
                                 cudaStream_t s)
{
    if (ngroups <= 0) return cudaSuccess;
    const int total = ngroups * (QL_HEAD + QL_VALUES);
    k_query_records<<<std::min((total + 255) / 256, 4096), 256, 0, s>>>(ghat, modes, src, ngroups, reinterpret_cast<float2 *>(out));
    return cudaGetLastError();
}

cudaError_t launch_query_gather(const float2 *fa, const float2 *fb, const int4 *modes, int count, int N, bool line_a,
                                bool line_b, float2 *ghat, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    int blocks = (count + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_query_gather<<<blocks, 256, 0, s>>>(fa, fb, modes, count, N, line_a, line_b, ghat);
    return cudaGetLastError();
}

// One block per query point.  The block first tabulates exp(2 pi i k t_a / P)
// for k in (-N/2, N/2) on each axis: the argument k t_a / P is formed and
// reduced to [-1/2, 1/2] in FP64, then sincospi runs in FP32 on the reduced
// value (|error| ~ 1e-7, independent of k and t).  Each thread then sums its
// share of the modes, w Re(g^ E_x E_y E_z), and the block reduces.
constexpr int QUERY_THREADS = 256;

__global__ void __launch_bounds__(QUERY_THREADS)
k_query_eval(const float2 *__restrict__ ghat, const int4 *__restrict__ modes, int count, int N, double inv_period,
             float scale, const float *__restrict__ t, int npts, float *g)
{
    extern __shared__ float2 E[]; // [3][N], index k + N/2
    __shared__ float red[QUERY_THREADS / 32];
    const int half = N / 2;
    for (int p = blockIdx.x; p < npts; p += gridDim.x) {
        for (int e = threadIdx.x; e < 3 * N; e += blockDim.x) {
            const int a = e / N, k = e - a * N - half;
            const double x = (double)k * (double)t[3 * p + a] * inv_period;
            const float r = (float)(x - rint(x));
            float sn, cs;
            sincospif(2.0f * r, &sn, &cs);
            E[e] = make_float2(cs, sn);
        }
        __syncthreads();
        float acc = 0.f;
        for (int i = threadIdx.x; i < count; i += blockDim.x) {
            const int4 m = modes[i];
            const float2 ph = cmul(cmul(E[m.x + half], E[N + m.y + half]), E[2 * N + m.z + half]);
            const float2 v = ghat[i];
            acc = fmaf((float)m.w, fmaf(v.x, ph.x, -v.y * ph.y), acc);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            float s = 0.f;
            for (int w = 0; w < QUERY_THREADS / 32; w++) s += red[w];
            g[p] = s * scale;
        }
        __syncthreads();
    }
}

// Many points: a warp takes 32 points (one per lane) and a share of the modes,
// ordered by columns (m_x, m_y) of consecutive m_z:
//     sum over columns of Re( E_x E_y sum_{m_z} w g^ E_z[m_z] ),
// so a mode costs four FMAs and a share of one table load (k_query_eval: three
// scattered table loads, two complex products and 24 bytes of mode data per point
// and mode).  Columns come in groups of four and at most QL_ROWS m_z, one 512-byte
// record each (QlGroup), so one E_z serves four modes and g^ is read as two
// 16-byte values, the same for every lane; a warp copies its records QL_RING
// groups ahead (without the ring every group waited on device memory: 20.6 us at
// 4,096 modes and points, 14.4 with it, k_query_eval 31).  Bound by instruction
// issue: one block of 16 warps per SM at 4,096 points.  The tables [axis][|m|][lane] hold the same
// values as k_query_eval's; a negative component takes the conjugate.
constexpr int QL_WARPS = 16, QL_RING = 4, QL_MAX_M = 128; // N <= 256: components below 128

__global__ void __launch_bounds__(QL_WARPS * 32)
k_query_lines(const QlGroup *__restrict__ groups, int ngroups, int M, double inv_period, float scale,
              const float *__restrict__ t, int npts, float *g)
{
    extern __shared__ float4 qlsm[]; // rings, then the tables [3][M][32]
    __shared__ float red[QL_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    QlGroup *ring = reinterpret_cast<QlGroup *>(qlsm) + warp * QL_RING;
    float2 *E = reinterpret_cast<float2 *>(reinterpret_cast<QlGroup *>(qlsm) + QL_WARPS * QL_RING);
    auto fetch = [&](int q, int slot) {
        if (q < ngroups)
            cp_async16(reinterpret_cast<char *>(ring + slot) + 16 * lane, reinterpret_cast<const char *>(groups + q) + 16 * lane,
                       true);
        cp_async_commit();
    };
#pragma unroll
    for (int k = 0; k < QL_RING - 1; k++) fetch(warp + k * QL_WARPS, k);
    const int p = blockIdx.x * 32 + lane;
    for (int e = warp; e < 3 * M; e += QL_WARPS) {
        const int a = e / M, k = e - a * M;
        const double x = (double)k * (double)(p < npts ? t[3 * p + a] : 0.f) * inv_period;
        const float r = (float)(x - rint(x));
        float sn, cs;
        sincospif(2.0f * r, &sn, &cs);
        E[e * 32 + lane] = make_float2(cs, sn);
    }
    __syncthreads();
    const float2 *Ex = E + lane, *Ey = Ex + M * 32, *Ez = Ey + M * 32;
    float sum = 0.f;
    int slot = 0;
    for (int q = warp; q < ngroups; q += QL_WARPS) {
        // the slot of the previous group is free (every lane has passed the barrier below since)
        fetch(q + (QL_RING - 1) * QL_WARPS, (slot + QL_RING - 1) % QL_RING);
        asm volatile("cp.async.wait_group %0;" ::"n"(QL_RING - 1) : "memory");
        __syncwarp();
        const QlGroup &gr = ring[slot];
        const float2 *ez = Ez + gr.z0 * 32;
        const int rows = gr.rows;
        float2 acc[4];
#pragma unroll
        for (int c = 0; c < 4; c++) acc[c] = make_float2(0.f, 0.f);
#pragma unroll 5
        for (int z = 0; z < rows; z++) {
            const float2 e = ez[z * 32];
            const float4 u = *reinterpret_cast<const float4 *>(&gr.v[z][0]), w = *reinterpret_cast<const float4 *>(&gr.v[z][2]);
            const float2 m[4] = {{u.x, u.y}, {u.z, u.w}, {w.x, w.y}, {w.z, w.w}};
#pragma unroll
            for (int c = 0; c < 4; c++) {
                acc[c].x = fmaf(m[c].x, e.x, fmaf(-m[c].y, e.y, acc[c].x));
                acc[c].y = fmaf(m[c].x, e.y, fmaf(m[c].y, e.x, acc[c].y));
            }
        }
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const int mx = gr.mx[c], my = gr.my[c];
            float2 ex = Ex[abs(mx) * 32], ey = Ey[abs(my) * 32];
            if (mx < 0) ex.y = -ex.y;
            if (my < 0) ey.y = -ey.y;
            const float2 ph = cmul(ex, ey);
            sum += fmaf(acc[c].x, ph.x, -acc[c].y * ph.y);
        }
        slot = (slot + 1) % QL_RING;
        __syncwarp();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    red[warp][lane] = sum;
    __syncthreads();
    if (warp == 0 && p < npts) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < QL_WARPS; w++) s += red[w][lane];
        g[p] = s * scale;
    }
}

cudaError_t launch_query_lines(const QlGroup *groups, int ngroups, int M, double period, const float *t, int npts, float *g,
                               cudaStream_t s)
{
    auto bytes = [](int m) { return sizeof(QlGroup) * QL_WARPS * QL_RING + sizeof(float2) * 3 * (size_t)m * 32; };
    const size_t smem = bytes(M);
    cudaError_t e = set_smem(k_query_lines, bytes(QL_MAX_M));
    if (e != cudaSuccess) return e;
    k_query_lines<<<(npts + 31) / 32, QL_WARPS * 32, smem, s>>>(groups, ngroups, M, 1.0 / period,
                                                                 (float)(1.0 / (period * period * period)), t, npts, g);
    return cudaGetLastError();
}

cudaError_t launch_query_eval(const float2 *ghat, const int4 *modes, int count, int N, double period, const float *t,
                              int npts, float *g, cudaStream_t s)
{
    if (npts <= 0) return cudaSuccess;
    const int blocks = npts < 65535 ? npts : 65535;
    const float scale = (float)(1.0 / (period * period * period));
    k_query_eval<<<blocks, QUERY_THREADS, sizeof(float2) * 3 * N, s>>>(ghat, modes, count, N, 1.0 / period, scale, t,
                                                                        npts, g);
    return cudaGetLastError();
}

} // namespace bc
