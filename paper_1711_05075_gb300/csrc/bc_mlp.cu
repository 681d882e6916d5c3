// Learned rotation proposal: a three-layer perceptron that maps a rotation and
// low-order Fourier-moment magnitudes of the two shapes to a predicted
// correlation peak, so that only the best-ranked rotations get full
// correlations.  The paper has no counterpart; the network follows the usual
// definitions (ReLU layers, mean squared error, Adam with bias correction --
// Kingma & Ba, 2015).
//
//   x  = [q (unit, w >= 0); f_A[0..63]; f_B[0..63]]          (132 features)
//   h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), y = w3 . h2 + b3
//
// Precision: FP32 master weights and Adam moments; every product reads its
// operands rounded to BF16 (weights, inputs, hidden activations, hidden
// gradients) and accumulates in FP32 on the tensor cores (tcgen05.mma
// kind::f16, BF16 x BF16 -> FP32 in tensor memory).  All reductions run in a fixed order, so training is
// deterministic for a fixed launch configuration.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include <cuda_bf16.h>

#include "../../include/ballcorr.h"
#include "bc_internal.h"
#include "bc_umma.cuh"

using namespace bc;

namespace {

constexpr int KIN = BC_MLP_IN;   // 132 input features
constexpr int KPAD = 144;        // padded to a multiple of 16 for the tensor-core K steps

struct Offsets {
    long long W1, b1, W2, b2, w3, b3, total;
};

Offsets offsets(int H)
{
    Offsets o;
    o.W1 = 0;
    o.b1 = o.W1 + (long long)H * KIN;
    o.W2 = o.b1 + H;
    o.b2 = o.W2 + (long long)H * H;
    o.w3 = o.b2 + H;
    o.b3 = o.w3 + H;
    o.total = o.b3 + 1;
    return o;
}

// ------------------------------------------------------------------ BF16 GEMM
// C[m][n] = sum_k A[m][k] B[k][n] (+ bias[n]) (relu), operands FP32 in global
// memory addressed through strides, rounded to BF16 when staged in shared
// memory, products on the 5th-generation tensor cores
// (tcgen05.mma.cta_group::1.kind::f16: A and B BF16, D FP32 in tensor memory;
// M = 128, N = the tile width, K = 16 per instruction).
//
// One block of 256 threads computes a 128 x nt tile of C (nt = 64, 128 or 256
// columns, chosen per call so that the grid covers the SMs).  Per K step of 64
// the threads round the A (128 x 64) and B (nt x 64) tiles to BF16 and store
// them K-major in the 128-byte-swizzled layout (row r's 16-byte chunk j at
// chunk j xor (r mod 8), 8-row groups 1024 bytes apart); one thread issues the
// step's four MMAs and commits them to the buffer's barrier while the block
// converts the next step into the other buffer.  After the last step the warps
// drain the accumulator (warp w reads lanes 32 (w mod 4) .. + 31, every other
// 16-column chunk), add the bias, apply the ReLU and store.  Every wait is
// bounded (bit 32 of the context's error word on expiry).
struct GemmArgs {
    const float *A;
    long long sAm, sAk;
    const float *B;
    long long sBk, sBn;
    float *C;
    long long sCm, sCn;
    int M, N, K;
    const float *bias;
    int relu;
    int kchunk = 0;     // split K: slice z of the grid sums k in [z kchunk, (z + 1) kchunk) (0: all of K)
    long long sCz = 0;  // and writes its partial product at C + z sCz
    int *err = nullptr; // status word for an expired tensor-core wait (required)
    int nt = 256;       // tile width (64, 128 or 256; set by the launchers)
    int bone = -1;      // >= 0: B's row bone is 1 for every k (C's column bone = the row sums of A); B has rows [0, bone)
    const float *mask = nullptr; // C = bf16(x) where mask > 0, else 0 (mask addressed like C; no bias, ReLU or split K)
};

constexpr int GU_THREADS = 256, GU_K = 64;
constexpr int GU_A_BYTES = 128 * 128; // 128 rows of 64 BF16
constexpr int GU_ERR = 32;

int gu_smem(int nt) { return 1024 + 2 * (GU_A_BYTES + nt * 128) + 64; }

__host__ __device__ constexpr uint32_t umma_idesc_bf16(int n)
{
    // D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9 = 1, 10-12 = 1), both K-major,
    // N >> 3 at bit 17, M >> 4 at bit 24 (M = 128)
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
                 : "memory");
}

__device__ __forceinline__ uint32_t bf2(float a, float b)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}

// the 16-byte chunk j (values 8 j .. 8 j + 7 along k) of row r of a swizzled tile
__device__ __forceinline__ void st_chunk(uint8_t *dst, int r, int j, float a0, float a1, float a2, float a3, float a4,
                                         float a5, float a6, float a7)
{
    *reinterpret_cast<uint4 *>(dst + r * 128 + ((j ^ (r & 7)) << 4)) =
        make_uint4(bf2(a0, a1), bf2(a2, a3), bf2(a4, a5), bf2(a6, a7));
}

// rows x 64 values of a strided FP32 matrix, rounded to BF16 into the swizzled
// tile at `dst`: element (r, k) = src[(r0 + r) sR + (k0 + k) sK], zero unless
// r0 + r < rlim and k0 + k < klim, except row r0 + r = rone (if any), which is
// 1 for every k0 + k < klim.  The global loads stay coalesced, with
// several in flight per thread:
//  - rows contiguous (sR = 1, 16-byte aligned groups of 4 rows): a thread takes
//    4 rows x 8 k as eight float4 loads, neighbouring threads neighbouring rows;
//  - otherwise pieces of 8 consecutive k of one row (two float4 loads when k is
//    contiguous and aligned, else 8 scalar loads), neighbouring threads
//    neighbouring pieces of a row.
__device__ __forceinline__ void gu_tile(uint8_t *dst, const float *__restrict__ src, long long sR, long long sK, int r0,
                                        int rows, int rlim, int k0, int klim, int rone)
{
    const bool aligned = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
    if (sR == 1 && aligned && (sK & 3) == 0 && (r0 & 3) == 0) {
        const int groups = rows >> 2, items = groups * 8;
        for (int c = threadIdx.x; c < items; c += GU_THREADS) {
            const int gi = c % groups, j = c / groups;
            const int gr = r0 + 4 * gi;
            float4 w[8];
#pragma unroll
            for (int kk = 0; kk < 8; kk++) {
                const int k = k0 + 8 * j + kk;
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                if (k < klim) {
                    const float *p = src + gr + (long long)k * sK;
                    if (gr + 3 < rlim) {
                        x = __ldg(reinterpret_cast<const float4 *>(p));
                    } else {
                        x.x = gr < rlim ? p[0] : (gr == rone ? 1.f : 0.f);
                        x.y = gr + 1 < rlim ? p[1] : (gr + 1 == rone ? 1.f : 0.f);
                        x.z = gr + 2 < rlim ? p[2] : (gr + 2 == rone ? 1.f : 0.f);
                        x.w = gr + 3 == rone ? 1.f : 0.f;
                    }
                }
                w[kk] = x;
            }
            st_chunk(dst, 4 * gi, j, w[0].x, w[1].x, w[2].x, w[3].x, w[4].x, w[5].x, w[6].x, w[7].x);
            st_chunk(dst, 4 * gi + 1, j, w[0].y, w[1].y, w[2].y, w[3].y, w[4].y, w[5].y, w[6].y, w[7].y);
            st_chunk(dst, 4 * gi + 2, j, w[0].z, w[1].z, w[2].z, w[3].z, w[4].z, w[5].z, w[6].z, w[7].z);
            st_chunk(dst, 4 * gi + 3, j, w[0].w, w[1].w, w[2].w, w[3].w, w[4].w, w[5].w, w[6].w, w[7].w);
        }
        return;
    }
    const bool kvec = aligned && sK == 1 && (sR & 3) == 0;
    const int items = rows * 8;
    for (int c0 = threadIdx.x; c0 < items; c0 += 4 * GU_THREADS) {
        float x[4][8];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int c = c0 + u * GU_THREADS;
            const int gr = r0 + (c >> 3), k = k0 + 8 * (c & 7);
            const float *p = src + (long long)gr * sR + (long long)k * sK;
            if (c < items && gr < rlim && kvec && k + 8 <= klim) {
                const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
                const float4 b = __ldg(reinterpret_cast<const float4 *>(p + 4));
                x[u][0] = a.x, x[u][1] = a.y, x[u][2] = a.z, x[u][3] = a.w;
                x[u][4] = b.x, x[u][5] = b.y, x[u][6] = b.z, x[u][7] = b.w;
            } else {
#pragma unroll
                for (int kk = 0; kk < 8; kk++)
                    x[u][kk] = (c < items && k + kk < klim) ? (gr < rlim ? p[kk * sK] : (gr == rone ? 1.f : 0.f)) : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int c = c0 + u * GU_THREADS;
            if (c < items)
                st_chunk(dst, c >> 3, c & 7, x[u][0], x[u][1], x[u][2], x[u][3], x[u][4], x[u][5], x[u][6], x[u][7]);
        }
    }
}

__global__ void __launch_bounds__(GU_THREADS, 3) k_gemm_umma(GemmArgs g, int err_bit)
{
    int *err = g.err;
    const int nt = g.nt, buf = GU_A_BYTES + nt * 128;
    extern __shared__ uint8_t gu_raw[];
    const uint32_t raw = smem_addr(gu_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gb = gu_raw + (base - raw);
    // [A 0 | B 0 | A 1 | B 1] [barriers: done[0], done[1]] [tensor-memory slot] [stop]
    uint64_t *bars = reinterpret_cast<uint64_t *>(gb + 2 * buf);
    uint32_t *slot = reinterpret_cast<uint32_t *>(bars + 2);
    volatile int *stop = reinterpret_cast<volatile int *>(slot + 1);
    const uint32_t bar0 = smem_addr(bars);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * 128, n0 = blockIdx.x * nt;
    const int ncols = min(nt, g.N - n0);
    const int NT = (ncols + 15) & ~15;
    const uint32_t idesc = umma_idesc_bf16(NT);
    const int kb = g.kchunk ? (int)blockIdx.z * g.kchunk : 0;
    const int ke = g.kchunk ? min(g.K, kb + g.kchunk) : g.K;
    const int steps = ke > kb ? (ke - kb + GU_K - 1) / GU_K : 0;
    if (threadIdx.x == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        *stop = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(nt)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    bool ok = true;
    int issued = 0; // steps whose MMAs were issued (the same count in every thread)
    for (int st = 0; st < steps && ok; st++) {
        const int b = st & 1;
        // buffer b was last read by the MMAs of step st - 2
        if (st >= 2) ok = umma_wait(bar0 + 8 * b, ((st - 2) >> 1) & 1, stop, err, err_bit);
        ok = __syncthreads_and(ok);
        if (!ok) break;
        uint8_t *ta = gb + b * buf, *tbt = ta + GU_A_BYTES;
        const int k0 = kb + st * GU_K;
        gu_tile(ta, g.A, g.sAm, g.sAk, m0, 128, g.M, k0, ke, -1);
        gu_tile(tbt, g.B, g.sBn, g.sBk, n0, NT, g.bone >= 0 ? g.bone : g.N, k0, ke, g.bone);
        fence_proxy_async_smem(); // the tile stores are visible to the tensor core's reads
        __syncthreads();
        if (threadIdx.x == 0) {
            tc_fence_after();
            const uint32_t a = base + b * buf, bb = a + GU_A_BYTES;
#pragma unroll
            for (int k = 0; k < GU_K / 16; k++) // K = 16 BF16 (32 bytes) per MMA
                umma_bf16(tmem, umma_desc_sw128(a + 32 * k), umma_desc_sw128(bb + 32 * k), idesc,
                          (st > 0 || k > 0) ? 1 : 0);
            umma_commit(bar0 + 8 * b);
        }
        issued = st + 1;
    }
    // the last step's MMAs (all earlier ones complete before it)
    if (ok && steps > 0) ok = umma_wait(bar0 + 8 * ((steps - 1) & 1), ((steps - 1) >> 1) & 1, stop, err, err_bit);
    ok = __syncthreads_and(ok);
    tc_fence_after();
    if (ok) {
        const int qd = warp & 3, half = warp >> 2;
        const int row = m0 + 32 * qd + lane;
        float *cz = g.C + blockIdx.z * g.sCz;
        const bool vec = g.sCn == 1 && (g.sCm & 3) == 0 && (reinterpret_cast<uintptr_t>(cz) & 15) == 0;
        float *crow = cz + (long long)row * g.sCm;
        for (int c0 = 16 * half; c0 < NT; c0 += 32) {
            uint32_t v[16];
            if (steps > 0) {
                tmem_ld16(tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)c0, v);
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) v[j] = 0u;
            }
            if (row < g.M) {
                float x[16], mk[16];
                if (g.mask) {
                    const float *mr = g.mask + (long long)row * g.sCm;
                    if (vec && c0 + 16 <= ncols) {
#pragma unroll
                        for (int q = 0; q < 4; q++) {
                            const float4 m4 = __ldg(reinterpret_cast<const float4 *>(mr + n0 + c0) + q);
                            mk[4 * q] = m4.x, mk[4 * q + 1] = m4.y, mk[4 * q + 2] = m4.z, mk[4 * q + 3] = m4.w;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) mk[j] = c0 + j < ncols ? mr[(long long)(n0 + c0 + j) * g.sCn] : 0.f;
                    }
                }
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    x[j] = __uint_as_float(v[j]);
                    if (g.bias && c0 + j < ncols) x[j] += g.bias[n0 + c0 + j];
                    if (g.relu) x[j] = fmaxf(x[j], 0.f);
                    if (g.mask) x[j] = mk[j] > 0.f ? __bfloat162float(__float2bfloat16_rn(x[j])) : 0.f;
                }
                if (vec && c0 + 16 <= ncols) {
                    float4 *o = reinterpret_cast<float4 *>(crow + n0 + c0);
#pragma unroll
                    for (int q = 0; q < 4; q++) o[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; j++)
                        if (c0 + j < ncols) crow[(long long)(n0 + c0 + j) * g.sCn] = x[j];
                }
            }
        }
    } else if (threadIdx.x == 0) {
        // a wait expired: let the MMAs already issued finish (bounded) before the memory goes;
        // the last commit to buffer b was step s (s < issued, s = b mod 2), phase s >> 1
        for (int b = 0; b < 2; b++) {
            const int s = ((issued - 1) & 1) == b ? issued - 1 : issued - 2;
            if (s < 0) continue;
            const uint64_t t0 = global_ns();
            while (!mbar_test(bar0 + 8 * b, (s >> 1) & 1) && global_ns() - t0 < UMMA_WAIT_NS) {
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(nt) : "memory");
    }
}

int gu_nsm()
{
    static int n = 0;
    if (n <= 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            n <= 0)
            n = 152;
    }
    return n;
}

// the widest tile whose grid (with nz slices of K) still gives every SM a block
int gu_pick_nt(int M, int N, int nz)
{
    const long long mt = (M + 127) / 128;
    for (int nt = 256; nt > 64; nt >>= 1)
        if ((long long)((N + nt - 1) / nt) * mt * nz >= gu_nsm()) return nt;
    return 64;
}

cudaError_t gu_launch(const GemmArgs &a, int nz, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_gemm_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, gu_smem(256));
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 grid((a.N + a.nt - 1) / a.nt, (a.M + 127) / 128, nz);
    k_gemm_umma<<<grid, GU_THREADS, gu_smem(a.nt), s>>>(a, GU_ERR);
    return cudaGetLastError();
}

cudaError_t gemm(GemmArgs a, cudaStream_t s)
{
    if (a.M <= 0 || a.N <= 0) return cudaSuccess;
    a.nt = gu_pick_nt(a.M, a.N, 1);
    return gu_launch(a, 1, s);
}

// out[m][n] = sum_z part[z][m][n], z in increasing order (M x N partials, rows
// `ld` floats apart); with `ocol`, column N - 1 goes to ocol[m] instead
__global__ void k_sum_partials(const float *__restrict__ part, int nz, int M, int N, int ld, float *out,
                               long long sOm, float *ocol)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)M * N) return;
    const long long m = e / N, nn = e - m * N;
    float s = 0.f;
    for (int z = 0; z < nz; z++) s += part[(z * (long long)M + m) * ld + nn];
    if (ocol && nn == N - 1) ocol[m] = s;
    else out[m * sOm + nn] = s;
}

// A weight gradient C = A B with a long K (the batch): K split into slices whose
// partial products land in `part` and are then summed in a fixed order, so the
// result does not depend on scheduling.  C is M x N with row stride sCm; with
// `ocol` (and a.bone = N - 1), C's last column -- the row sums of A -- goes to
// ocol instead.
cudaError_t gemm_splitk(GemmArgs a, float *part, long long part_floats, cudaStream_t s, float *ocol = nullptr)
{
    if (a.M <= 0 || a.N <= 0) return cudaSuccess;
    const int ld = (a.N + 3) & ~3; // partial rows padded to 16 bytes (vector stores)
    const long long mn = (long long)a.M * ld;
    const long long nzmax = std::max(1LL, std::min({32LL, part_floats / mn, (long long)(a.K + GU_K - 1) / GU_K}));
    a.nt = gu_pick_nt(a.M, a.N, (int)nzmax);
    const long long tiles = (long long)((a.N + a.nt - 1) / a.nt) * ((a.M + 127) / 128);
    int nz = (int)std::max(1LL, std::min(nzmax, (2LL * gu_nsm() + tiles - 1) / tiles)); // about two blocks per SM
    int kchunk = 0;
    if (a.K > 0) {
        kchunk = ((a.K + nz - 1) / nz + GU_K - 1) / GU_K * GU_K;
        nz = (a.K + kchunk - 1) / kchunk;
    } else {
        nz = 1;
    }
    float *C = a.C;
    const long long sCm = a.sCm;
    a.C = part;
    a.sCm = ld;
    a.sCn = 1;
    a.kchunk = kchunk;
    a.sCz = mn;
    cudaError_t e = gu_launch(a, nz, s);
    if (e != cudaSuccess) return e;
    const long long tot = (long long)a.M * a.N;
    k_sum_partials<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(part, nz, a.M, a.N, ld, C, sCm, ocol);
    return cudaGetLastError();
}

__device__ __forceinline__ float rbf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// y[b] = sum_j bf16(h2[b][j]) bf16(w3[j]) + b3 (one warp per row, fixed order)
__global__ void k_head(const float *__restrict__ h2, const float *__restrict__ w3, const float *__restrict__ b3, int n,
                       int H, float *y)
{
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= n) return;
    float s = 0.f;
    for (int j = lane; j < H; j += 32) s = fmaf(rbf(h2[(long long)row * H + j]), rbf(w3[j]), s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) y[row] = s + b3[0];
}

// The training head, for a batch of n rows:
//   y[b]   = sum_j bf16(h2[b][j]) bf16(w3[j]) + b3            (the sum of k_head, same order)
//   gy[b]  = 2 (y[b] - t[b]) / n                              (d loss / d y, mean squared error)
//   dh2[b][j] = bf16(gy[b] bf16(w3[j])) where h2[b][j] > 0, else 0
// and the sums over the batch dw3[j] = sum_b gy[b] bf16(h2[b][j]), db2[j] =
// sum_b dh2[b][j], db3 = sum_b gy[b].  k_head_train: one warp per row (lane l
// holds columns l + 32 i, the next row's loads issued before the current row's
// arithmetic); block c sums its rows, warp by warp in order, into
// part[c][0, 2H].  k_head_sums: one warp per entry adds the blocks' rows in a
// fixed order (lane l the blocks l, l + 32, ..., then a fixed shuffle tree).
constexpr int HT_THREADS = 256;

template <int NC>
__global__ void __launch_bounds__(HT_THREADS) k_head_train(const float *__restrict__ h2, const float *__restrict__ w3,
                                                           const float *__restrict__ b3, const float *__restrict__ t,
                                                           int n, int H, int rows_per_block, float *y, float *gy,
                                                           float *dh2, float *part)
{
    extern __shared__ float ht_s[]; // 2H + 1 block sums
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = HT_THREADS / 32;
    const int r0 = blockIdx.x * rows_per_block, r1 = min(n, r0 + rows_per_block);
    float w3r[NC], aw[NC], ab[NC], v[NC], a3 = 0.f;
#pragma unroll
    for (int i = 0; i < NC; i++) {
        const int j = lane + 32 * i;
        w3r[i] = j < H ? rbf(w3[j]) : 0.f;
        aw[i] = ab[i] = 0.f;
    }
    int r = r0 + warp;
    if (r < r1) {
#pragma unroll
        for (int i = 0; i < NC; i++) v[i] = lane + 32 * i < H ? h2[(long long)r * H + lane + 32 * i] : 0.f;
    }
    for (; r < r1; r += nw) {
        float vn[NC];
        const int rn = r + nw;
#pragma unroll
        for (int i = 0; i < NC; i++) vn[i] = (rn < r1 && lane + 32 * i < H) ? h2[(long long)rn * H + lane + 32 * i] : 0.f;
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < NC; i++)
            if (lane + 32 * i < H) sum = fmaf(rbf(v[i]), w3r[i], sum);
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const float yr = sum + b3[0];
        const float g = 2.f * (yr - t[r]) / (float)n;
        if (lane == 0) {
            y[r] = yr;
            gy[r] = g;
        }
        float *dr = dh2 + (long long)r * H;
#pragma unroll
        for (int i = 0; i < NC; i++) {
            const int j = lane + 32 * i;
            if (j < H) {
                const float d = v[i] > 0.f ? rbf(g * w3r[i]) : 0.f;
                dr[j] = d;
                aw[i] = fmaf(g, rbf(v[i]), aw[i]);
                ab[i] += d;
            }
            v[i] = vn[i];
        }
        a3 += g;
    }
    // block sums, warp 0 first
    for (int w = 0; w < nw; w++) {
        if (warp == w) {
#pragma unroll
            for (int i = 0; i < NC; i++) {
                const int j = lane + 32 * i;
                if (j < H) {
                    ht_s[j] = w ? ht_s[j] + aw[i] : aw[i];
                    ht_s[H + j] = w ? ht_s[H + j] + ab[i] : ab[i];
                }
            }
            if (lane == 0) ht_s[2 * H] = w ? ht_s[2 * H] + a3 : a3;
        }
        __syncthreads();
    }
    const int W = 2 * H + 1;
    for (int e = threadIdx.x; e < W; e += HT_THREADS) part[(long long)blockIdx.x * W + e] = ht_s[e];
}

__global__ void k_head_sums(const float *__restrict__ part, int nb, int H, float *dw3, float *db2, float *db3)
{
    const int W = 2 * H + 1;
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (e >= W) return;
    float sum = 0.f;
    for (int c = lane; c < nb; c += 32) sum += part[(long long)c * W + e];
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) {
        if (e < H) dw3[e] = sum;
        else if (e < 2 * H) db2[e - H] = sum;
        else db3[0] = sum;
    }
}

constexpr int HT_MAX_BLOCKS = 1024;

cudaError_t head_train(const float *h2, const float *w3, const float *b3, const float *t, int n, int H, float *y,
                       float *gy, float *dh2, float *part, long long part_floats, float *dw3, float *db2, float *db3,
                       cudaStream_t s)
{
    const long long W = 2LL * H + 1;
    // about four rows per warp
    int blocks = (int)std::min<long long>({(long long)(n + 31) / 32, (long long)HT_MAX_BLOCKS, part_floats / W});
    blocks = std::max(blocks, 1);
    const int rpb = (n + blocks - 1) / blocks;
    blocks = (n + rpb - 1) / rpb;
    const size_t smem = sizeof(float) * (size_t)W;
    const int nc = (H + 31) / 32;
#define HT_LAUNCH(NC) k_head_train<NC><<<blocks, HT_THREADS, smem, s>>>(h2, w3, b3, t, n, H, rpb, y, gy, dh2, part)
    if (nc <= 1) HT_LAUNCH(1);
    else if (nc <= 2) HT_LAUNCH(2);
    else if (nc <= 4) HT_LAUNCH(4);
    else if (nc <= 8) HT_LAUNCH(8);
    else if (nc <= 16) HT_LAUNCH(16);
    else HT_LAUNCH(32);
#undef HT_LAUNCH
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_head_sums<<<(unsigned)((W + 7) / 8), 256, 0, s>>>(part, blocks, H, dw3, db2, db3);
    return cudaGetLastError();
}

// batch row k = row perm(b0 + k) of X (KPAD floats) and t, perm(i) = (a i + c) mod n
__global__ void k_gather_batch(const float *__restrict__ X, const float *__restrict__ t, int n, long long a,
                               long long c, int b0, int nb, float *Xb, float *tb)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)nb * KPAD) return;
    const int k = (int)(e / KPAD), col = (int)(e - (long long)k * KPAD);
    const long long src = (a * (long long)(b0 + k) + c) % n;
    Xb[e] = X[src * KPAD + col];
    if (col == 0) tb[k] = t[src];
}

// the same with one float4 per thread (X 16-byte aligned; rows are KPAD = 36 float4)
__global__ void k_gather_batch4(const float4 *__restrict__ X, const float *__restrict__ t, int n, long long a,
                                long long c, int b0, int nb, float4 *Xb, float *tb)
{
    constexpr int R4 = KPAD / 4;
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)nb * R4) return;
    const int k = (int)(e / R4), col = (int)(e - (long long)k * R4);
    const long long src = (a * (long long)(b0 + k) + c) % n;
    Xb[e] = X[src * R4 + col];
    if (col == 0) tb[k] = t[src];
}

// mean of d[b]^2 with d = y - t, one block, fixed order
__global__ void k_loss(const float *__restrict__ y, const float *__restrict__ t, int n, float *loss)
{
    __shared__ float part[256];
    float s = 0.f;
    for (int b = threadIdx.x; b < n; b += 256) {
        const float d = y[b] - t[b];
        s = fmaf(d, d, s);
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = part[0] / (float)n;
}

// x[r] = [q_r / |q_r| with w >= 0; fa; fb; zeros to KPAD]; err |= 4 on a zero quaternion
// Row r: [q_r / |q_r| (w >= 0); fa; fb + r ldb] (ldb = 0: the same fb for every row).
__global__ void k_features(const float *__restrict__ q, int n, const float *__restrict__ fa,
                           const float *__restrict__ fb, long long ldb, float *X, int *err)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * KPAD) return;
    const int r = (int)(e / KPAD), c = (int)(e - (long long)r * KPAD);
    float v = 0.f;
    if (c < 4) {
        const float w = q[4 * r], x = q[4 * r + 1], y = q[4 * r + 2], z = q[4 * r + 3];
        const float n2 = w * w + x * x + y * y + z * z;
        if (!(n2 > 0.f)) {
            if (c == 0) atomicOr(err, 4);
            v = 0.f;
        } else {
            const float s = (w < 0.f ? -1.f : 1.f) / sqrtf(n2);
            v = q[4 * r + c] * s;
        }
    } else if (c < 68) {
        v = fa[c - 4];
    } else if (c < KIN) {
        v = fb[r * ldb + c - 68];
    }
    X[e] = v;
}

// ------------------------------------------------------------------ top-k
// One block sorts up to 16384 keys (score mapped to an order-preserving
// integer in the high half, the complement of the index in the low half) with
// a bitonic network in shared memory, descending; the first k indices are the
// k best scores, ties to the lowest index.

__global__ void __launch_bounds__(1024) k_topk(const float *__restrict__ s, int n, int P, int k, int *idx)
{
    extern __shared__ unsigned long long key[];
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        unsigned long long v = 0ull;
        if (i < n) {
            unsigned u = __float_as_uint(s[i]);
            u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
            v = ((unsigned long long)u << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)i);
        }
        key[i] = v;
    }
    __syncthreads();
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < P / 2; i += blockDim.x) {
                const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                const bool desc = ((lo & size) == 0);
                const unsigned long long a = key[lo], b = key[hi];
                if ((a < b) == desc) {
                    key[lo] = b;
                    key[hi] = a;
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < k; i += blockDim.x) idx[i] = (int)(0xFFFFFFFFu - (unsigned)(key[i] & 0xFFFFFFFFull));
}

__global__ void k_gather_quats(const float *__restrict__ q, const int *__restrict__ idx, int k, float *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 4 * k) out[i] = q[4 * (long long)idx[i >> 2] + (i & 3)];
}

// out_i = s * q_i (Hamilton product: rotation by q_i, then by s), quaternions (w, x, y, z)
__global__ void k_compose_quats(float4 sq, const float *__restrict__ q, int n, float *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float w2 = q[4 * (long long)i], x2 = q[4 * (long long)i + 1], y2 = q[4 * (long long)i + 2],
                z2 = q[4 * (long long)i + 3];
    const float w1 = sq.x, x1 = sq.y, y1 = sq.z, z1 = sq.w;
    float *o = out + 4 * (long long)i;
    o[0] = w1 * w2 - x1 * x2 - y1 * y2 - z1 * z2;
    o[1] = w1 * x2 + x1 * w2 + y1 * z2 - z1 * y2;
    o[2] = w1 * y2 - x1 * z2 + y1 * w2 + z1 * x2;
    o[3] = w1 * z2 + x1 * y2 - y1 * x2 + z1 * w2;
}

// y = alpha y + beta x
__global__ void k_axpby(float *y, const float *__restrict__ x, int n, float alpha, float beta)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = alpha * y[i] + beta * x[i];
}

// ------------------------------------------------------------------ fused forward pass
// Both hidden layers and the output of 128 rows in one block (hidden <= FW_MAXH):
//   h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), y = w3 . h2 + b3.
// The weights come as BF16 blocks already in the tensor core's swizzled layout
// (k_pack_weights, then kept by k_adam) by bulk copies: W1's three K blocks
// of 64 and the first of W2 at the start, W2's other blocks into W1's place once
// the first product is done.  The rows of X are rounded to BF16 by the threads; h1
// goes from tensor memory through the bias and the ReLU straight into the second
// product's operand tile.  Same operands, same order of accumulation as
// k_gemm_umma.  16,384 rows at 256 hidden: 47 us in three launches -> 12.3 us,
// most of it the latency of its chain (weights, two products, two epilogues).
constexpr int FW_MAXH = 256, FW_SLOTS = 4;

int fw_hp(int H) { return (H + 63) & ~63; }
int fw_smem(int H) { return 1024 + 4 * GU_A_BYTES + FW_SLOTS * H * 128 + 4 * (128 + 3 * FW_MAXH) + 128; }

// W1p[3][H][64], W2p[hp / 64][H][64] and W2T (row h_in, column h_out) BF16, rows of 128
// bytes swizzled as st_chunk does, zero beyond K
__global__ void k_pack_weights(const float *__restrict__ W1, const float *__restrict__ W2, int H, int hp, uint8_t *W1p,
                               uint8_t *W2p, uint8_t *W2T)
{
    const int n1 = 3 * H * 8, n2 = hp / 64 * H * 8, n3 = n2;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n1 + n2 + n3; e += gridDim.x * blockDim.x) {
        float x[8];
        if (e < n1 + n2) {
            const bool first = e < n1;
            const int q = first ? e : e - n1, j = q & 7, r = (q >> 3) % H, kb = (q >> 3) / H;
            const int K = first ? KIN : H, k0 = 64 * kb + 8 * j;
            const float *src = (first ? W1 : W2) + (long long)r * K;
#pragma unroll
            for (int k = 0; k < 8; k++) x[k] = k0 + k < K ? src[k0 + k] : 0.f;
            st_chunk((first ? W1p : W2p) + (size_t)kb * H * 128, r, j, x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
        } else { // neighbouring threads: neighbouring h_in
            const int q = e - n1 - n2, r = q % H, j = (q / H) & 7, kb = q / H / 8, k0 = 64 * kb + 8 * j;
#pragma unroll
            for (int k = 0; k < 8; k++) x[k] = k0 + k < H ? W2[(long long)(k0 + k) * H + r] : 0.f;
            st_chunk(W2T + (size_t)kb * H * 128, r, j, x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
        }
    }
}

// entry (r, k) of such blocks
__device__ __forceinline__ void st_packed(uint8_t *blocks, int H, int r, int k, float x)
{
    *reinterpret_cast<__nv_bfloat16 *>(blocks + (size_t)(k >> 6) * H * 128 + r * 128 + ((((k >> 3) & 7) ^ (r & 7)) << 4) +
                                       2 * (k & 7)) = __float2bfloat16_rn(x);
}

// Adam with bias correction on every parameter.  Where the fused passes are used it
// writes W1 and W2 into their BF16 blocks too, so that these always hold the parameters,
// also when launches are replayed from a graph.
__global__ void k_adam(float *p, float *m, float *v, const float *__restrict__ g, long long total, float lr, float b1,
                       float b2, float eps, float c1, float c2, int H, long long oW2, uint8_t *W1p, uint8_t *W2p, uint8_t *W2T)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.f - b1) * gg;
    const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    const float x = p[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    p[e] = x;
    if (!W1p) return;
    if (e < (long long)H * KIN) { // W1 comes first
        const int r = (int)e / KIN;
        st_packed(W1p, H, r, (int)e - r * KIN, x);
    } else if (e >= oW2 && e < oW2 + (long long)H * H) {
        const int q = (int)(e - oW2), r = q / H, c = q - r * H;
        st_packed(W2p, H, r, c, x);
        st_packed(W2T, H, c, r, x);
    }
}

__global__ void __launch_bounds__(GU_THREADS, 1)
k_mlp_forward(const float *__restrict__ X, int n, int H, int hp, int tcols, const uint8_t *__restrict__ W1p,
              const uint8_t *__restrict__ W2p, const float *__restrict__ b1, const float *__restrict__ b2,
              const float *__restrict__ w3, const float *__restrict__ b3, float *y, int *err)
{
    extern __shared__ uint8_t gu_raw[];
    const uint32_t raw = smem_addr(gu_raw), base = (raw + 1023u) & ~1023u;
    uint8_t *ga = gu_raw + (base - raw); // operand rows: four K blocks of 128 rows
    const uint32_t slot0 = base + 4 * GU_A_BYTES, sbytes = (uint32_t)H * 128;
    float *ys = reinterpret_cast<float *>(ga + 4 * GU_A_BYTES + FW_SLOTS * sbytes);
    float *b1s = ys + 128, *b2s = b1s + FW_MAXH, *w3s = b2s + FW_MAXH; // biases, w3 rounded to BF16
    uint64_t *bars = reinterpret_cast<uint64_t *>(w3s + FW_MAXH);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 6);
    volatile int *stop = reinterpret_cast<volatile int *>(tslot + 1);
    const uint32_t WB = smem_addr(bars), MD = WB + 8 * FW_SLOTS; // weights in slot k; product 1, 2 done
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, m0 = blockIdx.x * 128, kb2 = hp / 64;
    if (threadIdx.x == 0) {
        for (int k = 0; k < FW_SLOTS + 2; k++) mbar_init(WB + 8 * k, 1);
        *stop = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int k = 0; k < FW_SLOTS; k++) {
            mbar_expect_tx(WB + 8 * k, sbytes);
            bulk_g2s(slot0 + k * sbytes, k < 3 ? W1p + (size_t)k * sbytes : W2p, sbytes, WB + 8 * k);
        }
    }
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)), "r"(tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int c = threadIdx.x; c < H; c += GU_THREADS) {
        b1s[c] = b1[c];
        b2s[c] = b2[c];
        w3s[c] = rbf(w3[c]);
    }
#pragma unroll 1
    for (int kb = 0; kb < 3; kb++) gu_tile(ga + kb * GU_A_BYTES, X, KPAD, 1, m0, 128, n, 64 * kb, KIN, -1);
    fence_proxy_async_smem(); // the tile stores are visible to the tensor core's reads
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot, idesc = umma_idesc_bf16(H), d2 = tmem + (uint32_t)(tcols / 2);
    bool ok = true, loads2 = false, mma2 = false;
    if (threadIdx.x == 0) {
        for (int kb = 0; kb < 3 && ok; kb++) {
            ok = umma_wait(WB + 8 * kb, 0, stop, err, GU_ERR);
            if (!ok) break;
            const uint32_t a = base + kb * GU_A_BYTES, b = slot0 + kb * sbytes;
            for (int k = 0; k < (kb < 2 ? 4 : 1); k++) // K = 16 per MMA: 144 of the 192 columns
                umma_bf16(tmem, umma_desc_sw128(a + 32 * k), umma_desc_sw128(b + 32 * k), idesc, kb + k > 0);
        }
        umma_commit(MD);
    }
    ok = __syncthreads_and(umma_wait(MD, 0, stop, err, GU_ERR) && ok);
    if (ok) {
        tc_fence_after();
        if (threadIdx.x == 0 && kb2 > 1) { // W1 is used: W2's other blocks take its slots
            for (int k = 0; k < kb2 - 1; k++) {
                mbar_expect_tx(WB + 8 * k, sbytes);
                bulk_g2s(slot0 + k * sbytes, W2p + (size_t)(k + 1) * sbytes, sbytes, WB + 8 * k);
            }
        }
        loads2 = true;
        const int q = warp & 3, half = warp >> 2, r = 32 * q + lane, row = m0 + r;
#pragma unroll 1
        for (int c0 = 16 * half; c0 < hp; c0 += 32) {
            float x[16];
            if (c0 < H) {
                uint32_t v[16];
                tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, v);
#pragma unroll
                for (int j = 0; j < 16; j++) x[j] = fmaxf(__uint_as_float(v[j]) + b1s[c0 + j], 0.f);
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) x[j] = 0.f;
            }
            uint8_t *t = ga + (c0 >> 6) * GU_A_BYTES;
            const int j0 = (c0 & 63) >> 3;
            st_chunk(t, r, j0, x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
            st_chunk(t, r, j0 + 1, x[8], x[9], x[10], x[11], x[12], x[13], x[14], x[15]);
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (threadIdx.x == 0) {
            for (int kb = 0; kb < kb2 && ok; kb++) {
                const int sl = kb == 0 ? 3 : kb - 1;
                ok = umma_wait(WB + 8 * sl, kb == 0 ? 0 : 1, stop, err, GU_ERR);
                if (!ok) break;
                const uint32_t a = base + kb * GU_A_BYTES, b = slot0 + sl * sbytes;
                for (int k = 0; k < min(4, (H - 64 * kb) / 16); k++)
                    umma_bf16(d2, umma_desc_sw128(a + 32 * k), umma_desc_sw128(b + 32 * k), idesc, kb + k > 0);
            }
            umma_commit(MD + 8);
        }
        mma2 = true;
        ok = __syncthreads_and(umma_wait(MD + 8, 0, stop, err, GU_ERR) && ok);
        if (ok) {
            tc_fence_after();
            float s = 0.f;
#pragma unroll 1
            for (int c0 = 16 * half; c0 < H; c0 += 32) {
                uint32_t v[16];
                tmem_ld16(d2 + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, v);
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const float x = fmaxf(__uint_as_float(v[j]) + b2s[c0 + j], 0.f);
                    s = fmaf(rbf(x), w3s[c0 + j], s);
                }
            }
            if (half == 1) ys[r] = s;
            __syncthreads();
            if (half == 0 && row < n) y[row] = s + ys[r] + b3[0];
        }
    }
    if (!ok && threadIdx.x == 0) {
        // a wait expired: copies and MMAs in flight finish (bounded) before the memory goes
        auto drain = [&](uint32_t bar, uint32_t par) {
            const uint64_t t0 = global_ns();
            while (!mbar_test(bar, par) && global_ns() - t0 < UMMA_WAIT_NS) {
            }
        };
        for (int k = 0; k < FW_SLOTS; k++) drain(WB + 8 * k, loads2 && k < kb2 - 1 ? 1 : 0);
        drain(MD, 0);
        if (mma2) drain(MD + 8, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
    }
}

// ------------------------------------------------------------------ fused training pass
// Forward pass, loss and every gradient of 128 rows in one block (hidden <=
// FW_MAXH), the sums over the batch left as one partial per block, added in block
// order by k_train_sums:
//   products (tcgen05, BF16 operands, FP32 in tensor memory):
//     1  h1 pre = X W1^T            columns [0, H)
//     2  h2 pre = h1 W2^T           columns [T, T + H), T = half of the tensor memory taken
//     3  dW2^T  = h1^T dh2          both accumulators: rows h_in 0 .. 127 and 128 .. 255
//     4  dh1 pre = dh2 W2           columns [0, H)
//     5  [dW1 | db1]^T = [X | 1]^T dh1   rows 0 .. 127 at column T, 128 .. 143 at column 0
//   3 and 5 sum over the rows, so they read the same operand tiles transposed
//   (the tiles' 128-byte rows are 64 consecutive columns of one batch row: the
//   MN-major form of the same swizzle, K groups of 8 rows 1024 bytes apart, the
//   next 64 columns 16 KB on).  Transposed, the lanes of a warp hold consecutive
//   weights of one output unit and every store is one 128-byte run (a lane per
//   output unit: 64 us instead of 53 for the whole pass).
// Tiles: X | 1 (3 K blocks), h1 and later dh1 (4), dh2 (4), 16 KB each; the weights'
// K blocks come by bulk copies into a 32 KB slot of their own and into the tiles
// that are not in use: W1, then W2 around the dh2 tile, W2^T around the h1 tile
// (its ReLU mask is kept as bits).  Before it took five products and five other
// launches with every operand through FP32 device memory: 117.6 us for 8,192 rows,
// H = 256, now 43.  What is left is the latency of one block's chain (five products,
// five epilogues) on 64 of the 152 SMs.
constexpr int TR_TILES = 11; // 16 KB tiles: X 0-2, h 3-6, d 7-10
constexpr int TR_MAX_ROWS = 1 << 15; // partials of 400 KB per 128 rows at H = 256

int tr_smem(int H)
{
    return 1024 + TR_TILES * GU_A_BYTES + H * 128 + 4 * (2 * 128 + 8 * 2 * 128 + 8 + 3 * FW_MAXH) + 2 * 8 * GU_THREADS + 128;
}
// a block's partial: dW2 [H][H], [dW1 | db1] [H][144], db2 [H], dw3 [H], db3, loss (padded to 16 floats)
__host__ __device__ constexpr long long tr_part(int H) { return (long long)H * H + 144LL * H + 2 * H + 16; }

// descriptor of a tile read transposed: 64-column blocks GU_A_BYTES apart, groups of 8 rows 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(GU_A_BYTES >> 4) << 16; // leading byte offset
    d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// 16 columns' sums over the warp's 32 lanes: lane l returns the sum of column l / 2 mod 16
__device__ __forceinline__ float warp_colsum16(float (&x)[16], int lane)
{
#pragma unroll
    for (int o = 16, half = 8; o > 1; o >>= 1, half >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < half; j++) {
            const float keep = up ? x[j + half] : x[j], send = up ? x[j] : x[j + half];
            x[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
}

__global__ void __launch_bounds__(GU_THREADS, 1)
k_mlp_train(const float *__restrict__ X, const float *__restrict__ t, int n, int H, int hp, int tcols,
            const uint8_t *__restrict__ W1p, const uint8_t *__restrict__ W2p, const uint8_t *__restrict__ W2T,
            const float *__restrict__ b1, const float *__restrict__ b2, const float *__restrict__ w3,
            const float *__restrict__ b3, float *y, float *part, int *err)
{
    extern __shared__ uint8_t gu_raw[];
    const uint32_t raw = smem_addr(gu_raw), base = (raw + 1023u) & ~1023u;
    uint8_t *ga = gu_raw + (base - raw);
    uint8_t *hT = ga + 3 * GU_A_BYTES, *dT = ga + 7 * GU_A_BYTES;
    const uint32_t xa = base, ha = base + 3 * GU_A_BYTES, da = base + 7 * GU_A_BYTES, s0 = base + TR_TILES * GU_A_BYTES;
    const uint32_t sbytes = (uint32_t)H * 128;
    float *ys = reinterpret_cast<float *>(ga + TR_TILES * GU_A_BYTES + sbytes); // y halves [2][128]
    float *cs = ys + 2 * 128;                                                   // column sums [warp][dw3, db2][128]
    float *rs = cs + 8 * 2 * 128;                                               // row sums [4][db3, loss]
    float *b1s = rs + 8, *b2s = b1s + FW_MAXH, *w3s = b2s + FW_MAXH;            // biases, w3 rounded to BF16
    // h1 > 0 at the thread's columns 16 half + 32 i + j: bit j of ms[256 i + thread]
    uint16_t *ms = reinterpret_cast<uint16_t *>(w3s + FW_MAXH);
    uint64_t *bars = reinterpret_cast<uint64_t *>(ms + 8 * GU_THREADS);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 8);
    volatile int *stop = reinterpret_cast<volatile int *>(tslot + 1);
    // weights landed in slot 0, 1, 2 (their phase counts the loads); a product's MMAs done; slot 0 read
    const uint32_t WB = smem_addr(bars), MD = WB + 24, SF = WB + 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, m0 = blockIdx.x * 128, kb2 = hp / 64;
    const int q = warp & 3, half = warp >> 2, r = 32 * q + lane, row = m0 + r;
    const bool in = row < n;
    float *P = part + (long long)blockIdx.x * tr_part(H);
    const uint32_t slot1[3] = {s0, da, da + sbytes}, slot2[3] = {s0, ha, ha + sbytes}; // two blocks fit a 64 KB tile group
    uint32_t loads[3] = {0, 0, 0}; // thread 0: loads issued per slot
    bool copies = false;
    auto load = [&](int sl, uint32_t dst, const uint8_t *src) {
        mbar_expect_tx(WB + 8 * sl, sbytes);
        bulk_g2s(dst, src, sbytes, WB + 8 * sl);
        loads[sl]++;
        copies = true;
    };
    auto landed = [&](int sl) { return umma_wait(WB + 8 * sl, (loads[sl] - 1) & 1, stop, err, GU_ERR); };
    if (threadIdx.x == 0) {
        for (int k = 0; k < 3; k++) mbar_init(WB + 8 * k, 1);
        mbar_init(MD, 1);
        mbar_init(SF, 1);
        *stop = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int k = 0; k < 3; k++) load(k, slot1[k], W1p + (size_t)k * sbytes);
    }
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)), "r"(tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int c = threadIdx.x; c < H; c += GU_THREADS) {
        b1s[c] = b1[c];
        b2s[c] = b2[c];
        w3s[c] = rbf(w3[c]);
    }
#pragma unroll 1
    for (int kb = 0; kb < 3; kb++) gu_tile(ga + kb * GU_A_BYTES, X, KPAD, 1, m0, 128, n, 64 * kb, KIN, -1);
    __syncthreads();
    // column 132 of the tile: 1 (W1's column 132 is zero there), for db1
    if (threadIdx.x < 128 && m0 + (int)threadIdx.x < n) {
        const int rr = threadIdx.x, k = KIN - 128; // value 4 of chunk 0 of the third block
        *reinterpret_cast<__nv_bfloat16 *>(ga + 2 * GU_A_BYTES + rr * 128 + (((k >> 3) ^ (rr & 7)) << 4) + 2 * (k & 7)) =
            __float2bfloat16_rn(1.f);
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot, T = (uint32_t)(tcols / 2), lanes = (uint32_t)(32 * q) << 16;
    const uint32_t idesc = umma_idesc_bf16(H), mn = (1u << 15) | (1u << 16); // both operands MN-major
    uint32_t md = 0; // products waited for
    bool ok = true, issued = false;
    // waits (all threads) for the product thread 0 just committed
    auto product_done = [&]() {
        issued = true;
        ok = __syncthreads_and(umma_wait(MD, md & 1, stop, err, GU_ERR) && ok);
        md++;
        tc_fence_after();
        return ok;
    };
    // the threads' tile stores and tensor-memory reads precede the next product
    auto publish = [&]() {
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };
    // thread 0: D[128 rows][H] = A tiles (K-major) x weight blocks; block 3 follows block 0 in slot 0
    uint32_t sf = 0; // times slot 0 was handed on
    auto weight_product = [&](uint32_t d, uint32_t a, const uint32_t *slots, const uint8_t *src, int nkb, int K) {
        for (int kb = 0; kb < nkb && ok; kb++) {
            const int sl = kb % 3;
            if (kb == 3) {
                ok = umma_wait(SF, sf & 1, stop, err, GU_ERR);
                sf++;
                if (ok) load(0, slots[0], src + (size_t)3 * sbytes);
            }
            ok = ok && landed(sl);
            if (!ok) break;
            const int steps = min(4, (K - 64 * kb + 15) / 16);
            for (int k = 0; k < steps; k++)
                umma_bf16(d, umma_desc_sw128(a + kb * GU_A_BYTES + 32 * k), umma_desc_sw128(slots[sl] + 32 * k), idesc, kb + k > 0);
            if (kb == 0 && nkb > 3) umma_commit(SF);
        }
    };
    // the epilogue loops stay rolled: each runs once per block, and unrolled code waited on
    // instruction fetches (3.6 of the stall cycles per issued instruction)
    do {
        // ---- 1: h1
        if (threadIdx.x == 0) {
            weight_product(tmem, xa, slot1, W1p, 3, 144);
            umma_commit(MD);
        }
        if (!product_done()) break;
        if (threadIdx.x == 0)
            for (int k = 0; k < min(3, kb2); k++) load(k, slot1[k], W2p + (size_t)k * sbytes);
#pragma unroll 1
        for (int i = 0; i < 8; i++) {
            const int c0 = 16 * half + 32 * i;
            if (c0 < hp) {
                float x[16];
                if (c0 < H) {
                    uint32_t v[16], mask = 0;
                    tmem_ld16(tmem + lanes + (uint32_t)c0, v);
#pragma unroll
                    for (int j = 0; j < 16; j++) {
                        x[j] = fmaxf(__uint_as_float(v[j]) + b1s[c0 + j], 0.f);
                        if (x[j] > 0.f) mask |= 1u << j;
                    }
                    ms[GU_THREADS * i + threadIdx.x] = (uint16_t)mask;
                } else {
#pragma unroll
                    for (int j = 0; j < 16; j++) x[j] = 0.f;
                }
                uint8_t *h = hT + (c0 >> 6) * GU_A_BYTES;
                const int j0 = (c0 & 63) >> 3;
                st_chunk(h, r, j0, x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
                st_chunk(h, r, j0 + 1, x[8], x[9], x[10], x[11], x[12], x[13], x[14], x[15]);
            }
        }
        publish();
        // ---- 2: h2, y, dh2
        if (threadIdx.x == 0) {
            weight_product(tmem + T, ha, slot1, W2p, kb2, H);
            umma_commit(MD);
        }
        if (!product_done()) break;
        if (threadIdx.x == 0) load(0, s0, W2T);
        float s = 0.f;
#pragma unroll 1
        for (int c0 = 16 * half; c0 < H; c0 += 32) {
            uint32_t v[16];
            tmem_ld16(tmem + T + lanes + (uint32_t)c0, v);
#pragma unroll
            for (int j = 0; j < 16; j++) s = fmaf(rbf(fmaxf(__uint_as_float(v[j]) + b2s[c0 + j], 0.f)), w3s[c0 + j], s);
        }
        ys[half * 128 + r] = s;
        __syncthreads();
        const float yr = ys[r] + ys[128 + r] + b3[0];
        const float dy = in ? yr - t[row] : 0.f, gy = 2.f * dy / (float)n;
        if (half == 0 && in) y[row] = yr;
        if (half == 0) {
            float a = gy, b = dy * dy;
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_xor_sync(0xffffffffu, a, o);
                b += __shfl_xor_sync(0xffffffffu, b, o);
            }
            if (lane == 0) {
                rs[2 * q] = a;
                rs[2 * q + 1] = b;
            }
        }
#pragma unroll 1
        for (int i = 0; i < 8; i++) {
            const int c0 = 16 * half + 32 * i;
            if (c0 >= hp) continue;
            float dw[16], db[16];
            if (c0 < H) {
                uint32_t v[16];
                tmem_ld16(tmem + T + lanes + (uint32_t)c0, v);
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const float x = fmaxf(__uint_as_float(v[j]) + b2s[c0 + j], 0.f);
                    dw[j] = gy * rbf(x);
                    db[j] = x > 0.f ? rbf(gy * w3s[c0 + j]) : 0.f;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) dw[j] = db[j] = 0.f;
            }
            uint8_t *h = dT + (c0 >> 6) * GU_A_BYTES;
            const int j0 = (c0 & 63) >> 3;
            st_chunk(h, r, j0, db[0], db[1], db[2], db[3], db[4], db[5], db[6], db[7]);
            st_chunk(h, r, j0 + 1, db[8], db[9], db[10], db[11], db[12], db[13], db[14], db[15]);
            const float sw = warp_colsum16(dw, lane), sb = warp_colsum16(db, lane);
            if ((lane & 1) == 0) { // the warp's columns 16 i .. 16 i + 15 of its half
                cs[(2 * warp) * 128 + 16 * i + (lane >> 1)] = sw;
                cs[(2 * warp + 1) * 128 + 16 * i + (lane >> 1)] = sb;
            }
        }
        publish();
        // ---- 3: dW2
        const int halves = H > 128 ? 2 : 1;
        if (threadIdx.x == 0) {
            for (int m = 0; m < halves; m++)
                for (int k = 0; k < 8; k++)
                    umma_bf16(tmem + (m ? T : 0), umma_desc_mn(ha + 2 * m * GU_A_BYTES + 2048 * k), umma_desc_mn(da + 2048 * k),
                              idesc | mn, k > 0);
            umma_commit(MD);
        }
        {   // meanwhile the column and row sums of the four row quarters
            float *pc = P + (long long)H * H + 144LL * H;
            for (int c = threadIdx.x; c < H; c += GU_THREADS) {
                const int hf = (c >> 4) & 1, at = 16 * (c >> 5) + (c & 15);
                float w = 0.f, b = 0.f;
                for (int k = 0; k < 4; k++) {
                    w += cs[2 * (4 * hf + k) * 128 + at];
                    b += cs[(2 * (4 * hf + k) + 1) * 128 + at];
                }
                pc[c] = b;
                pc[H + c] = w;
            }
            if (threadIdx.x == 0) {
                pc[2 * H] = rs[0] + rs[2] + rs[4] + rs[6];
                pc[2 * H + 1] = rs[1] + rs[3] + rs[5] + rs[7];
            }
        }
        if (!product_done()) break;
        if (threadIdx.x == 0)
            for (int k = 1; k < min(3, kb2); k++) load(k, slot2[k], W2T + (size_t)k * sbytes);
        for (int m = 0; m < halves; m++) {
            const int hi = 128 * m + r;
#pragma unroll 1
            for (int c0 = 16 * half; c0 < H; c0 += 32) {
                uint32_t v[16];
                tmem_ld16(tmem + (m ? T : 0) + lanes + (uint32_t)c0, v);
                if (hi < H) {
#pragma unroll
                    for (int k = 0; k < 16; k++) P[(c0 + k) * H + hi] = __uint_as_float(v[k]);
                }
            }
        }
        publish();
        // ---- 4: dh1
        if (threadIdx.x == 0) {
            weight_product(tmem, da, slot2, W2T, kb2, H);
            umma_commit(MD);
        }
        if (!product_done()) break;
#pragma unroll 1
        for (int i = 0; i < 8; i++) {
            const int c0 = 16 * half + 32 * i;
            if (c0 >= hp) continue;
            float x[16];
            if (c0 < H) {
                uint32_t v[16];
                const uint32_t mask = ms[GU_THREADS * i + threadIdx.x];
                tmem_ld16(tmem + lanes + (uint32_t)c0, v);
#pragma unroll
                for (int j = 0; j < 16; j++) x[j] = (mask >> j) & 1 ? __uint_as_float(v[j]) : 0.f;
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) x[j] = 0.f;
            }
            uint8_t *h = hT + (c0 >> 6) * GU_A_BYTES;
            const int j0 = (c0 & 63) >> 3;
            st_chunk(h, r, j0, x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
            st_chunk(h, r, j0 + 1, x[8], x[9], x[10], x[11], x[12], x[13], x[14], x[15]);
        }
        publish();
        // ---- 5: [dW1 | db1]
        if (threadIdx.x == 0) {
            for (int m = 0; m < 2; m++) // rows 144 .. 255 are whatever lies beyond the X tiles: not stored
                for (int k = 0; k < 8; k++)
                    umma_bf16(tmem + (m ? 0 : T), umma_desc_mn(xa + 2 * m * GU_A_BYTES + 2048 * k), umma_desc_mn(ha + 2048 * k),
                              idesc | mn, k > 0);
            umma_commit(MD);
        }
        if (!product_done()) break;
        for (int m = 0; m < (q == 0 ? 2 : 1); m++) {
            const int k0 = 128 * m + r;
#pragma unroll 1
            for (int c0 = 16 * half; c0 < H; c0 += 32) {
                uint32_t v[16];
                tmem_ld16(tmem + (m ? 0 : T) + lanes + (uint32_t)c0, v);
                if (k0 < 144) {
                    float *o = P + H * H + k0;
#pragma unroll
                    for (int k = 0; k < 16; k++) o[(c0 + k) * 144] = __uint_as_float(v[k]);
                }
            }
        }
    } while (false);
    if (!ok && threadIdx.x == 0) {
        // a wait expired: copies and MMAs in flight finish (bounded) before the memory goes
        auto drain = [&](uint32_t bar, uint32_t par) {
            const uint64_t t0 = global_ns();
            while (!mbar_test(bar, par) && global_ns() - t0 < UMMA_WAIT_NS) {
            }
        };
        if (copies)
            for (int k = 0; k < 3; k++)
                if (loads[k]) drain(WB + 8 * k, (loads[k] - 1) & 1);
        if (issued) drain(MD, (md - 1) & 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
    }
}

// grads (parameter layout) and the loss from the blocks' partials: a warp takes every
// fourth block's 32 consecutive values in order, the four warps' sums are added in order
constexpr int TS_SLICES = 4;

__global__ void __launch_bounds__(32 * TS_SLICES)
k_train_sums(const float *__restrict__ part, int nb, int H, long long stride, Offsets o, int n, float *g, float *loss)
{
    __shared__ float red[TS_SLICES][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const long long w1 = (long long)H * H, v = w1 + 144LL * H, total = v + 2 * H + 2;
    const long long e = (long long)blockIdx.x * 32 + lane;
    float s = 0.f;
    if (e < total) {
#pragma unroll 8
        for (int b = slice; b < nb; b += TS_SLICES) s += part[b * stride + e];
    }
    red[slice][lane] = s;
    __syncthreads();
    if (slice || e >= total) return;
#pragma unroll
    for (int k = 1; k < TS_SLICES; k++) s += red[k][lane];
    if (e < w1) {
        g[o.W2 + e] = s;
    } else if (e < v) {
        const int r = (int)((e - w1) / 144), c = (int)((e - w1) % 144);
        if (c < KIN) g[o.W1 + (long long)r * KIN + c] = s;
        else if (c == KIN) g[o.b1 + r] = s;
    } else if (e < v + H) {
        g[o.b2 + (e - v)] = s;
    } else if (e < v + 2 * H) {
        g[o.w3 + (e - v - H)] = s;
    } else if (e == v + 2 * H) {
        g[o.b3] = s;
    } else if (loss) {
        *loss = s / (float)n;
    }
}

} // namespace

// ------------------------------------------------------------------ network object
struct bc_mlp_s {
    bc_ctx_t ctx = nullptr;
    int H = 0;
    Offsets off{};
    float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr; // params, Adam moments, gradients
    long long step = 0;
    // activations for the current batch capacity
    int cap = 0, ycap = 0;
    float *h1 = nullptr, *h2 = nullptr, *y = nullptr, *gy = nullptr, *dh2 = nullptr, *dh1 = nullptr;
    float *part = nullptr;        // split-K and column-sum partials
    long long part_floats = 0;
    float *xb = nullptr, *tb = nullptr; // a gathered training batch (bc_mlp_train)
    int xb_cap = 0;
    float *loss = nullptr;
    uint8_t *wp = nullptr;        // BF16 weights in the fused forward pass's layout (hidden <= FW_MAXH)
    int rotated_moments = 0;      // the ligand features are the moments of the rotated ligand (bc_mlp_set_features)
};

namespace {

bc_status mfail(bc_status s, const std::string &msg)
{
    set_last_error(msg);
    return s;
}

bc_status mcuda(cudaError_t e, const char *where)
{
    set_last_error(std::string(where) + ": " + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? BC_ERR_OOM : BC_ERR_CUDA;
}

#define MCK(call)                                                                                        \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) return mcuda(e_, #call);                                                  \
    } while (0)

template <typename T>
cudaError_t regrow(T *&p, size_t count)
{
    if (p) cudaFree(p);
    p = nullptr;
    return cudaMalloc(&p, sizeof(T) * count);
}

// Buffers of a training pass of n rows: the fused one keeps its layers on chip and
// needs y and the partials only.
bc_status ensure_batch(bc_mlp_t net, int n)
{
    const size_t H = net->H, cap = (size_t)n + n / 4 + 64;
    const bool fused = net->wp && n <= TR_MAX_ROWS;
    if (!net->g) MCK(cudaMalloc(&net->g, sizeof(float) * (size_t)net->off.total));
    if (n > net->ycap) {
        net->ycap = 0;
        MCK(regrow(net->y, cap));
        net->ycap = (int)cap;
    }
    // the fused pass's partials; or up to 32 split-K slices of the largest weight
    // gradient (H x (H + 1) or H x 133, the last column the bias gradient), and the
    // training head's block sums
    const long long need = fused ? (long long)((n + 127) / 128) * tr_part((int)H)
                                 : std::max(32LL * (long long)H * (std::max<long long>((long long)H, KIN) + 1),
                                            (long long)HT_MAX_BLOCKS * (2LL * (long long)H + 1));
    if (need > net->part_floats) {
        net->part_floats = 0;
        MCK(regrow(net->part, (size_t)need));
        net->part_floats = need;
    }
    if (fused || n <= net->cap) return BC_OK;
    net->cap = 0;
    for (float **b : {&net->h1, &net->h2, &net->dh2, &net->dh1}) MCK(regrow(*b, cap * H));
    MCK(regrow(net->gy, cap));
    net->cap = (int)cap;
    return BC_OK;
}

// The BF16 weight blocks of the fused passes, in one buffer.
struct Packed {
    uint8_t *W1 = nullptr, *W2 = nullptr, *W2T = nullptr;
    explicit Packed(bc_mlp_t net)
    {
        if (!net->wp) return;
        const size_t H = net->H, hp = fw_hp(net->H);
        W1 = net->wp;
        W2 = W1 + 3 * H * 128;
        W2T = W2 + hp / 64 * H * 128;
    }
};

// All of them from the parameters.
cudaError_t pack_weights(bc_mlp_t net, cudaStream_t s)
{
    if (!net->wp) return cudaSuccess;
    const int H = net->H, hp = fw_hp(H), items = (3 + 2 * hp / 64) * H * 8;
    const Packed w(net);
    k_pack_weights<<<(items + 255) / 256, 256, 0, s>>>(net->p + net->off.W1, net->p + net->off.W2, H, hp, w.W1, w.W2, w.W2T);
    return cudaGetLastError();
}

// One Adam step with the gradients in net->g.
cudaError_t adam(bc_mlp_t net, float lr, cudaStream_t s)
{
    net->step++;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)net->step));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)net->step));
    const long long total = net->off.total;
    const Packed w(net);
    k_adam<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(net->p, net->m, net->v, net->g, total, lr, b1, b2, eps, c1, c2,
                                                          net->H, net->off.W2, w.W1, w.W2, w.W2T);
    return cudaGetLastError();
}

// The fused forward pass: y of n rows.
bc_status fused_forward(bc_mlp_t net, const float *X, int n, float *y, cudaStream_t s)
{
    const int H = net->H, hp = fw_hp(H);
    const Offsets &o = net->off;
    const Packed w(net);
    int tcols = 32; // two accumulators of H columns
    while (tcols < 2 * H) tcols <<= 1;
    k_mlp_forward<<<(n + 127) / 128, GU_THREADS, fw_smem(H), s>>>(X, n, H, hp, tcols, w.W1, w.W2, net->p + o.b1, net->p + o.b2,
                                                                  net->p + o.w3, net->p + o.b3, y, ctx_err(net->ctx));
    MCK(cudaGetLastError());
    return BC_OK;
}

// The fused training pass: y, the gradients into g and the loss (may be null).
bc_status fused_train(bc_mlp_t net, const float *X, const float *t, int n, float *g, float *loss, cudaStream_t s)
{
    const int H = net->H, hp = fw_hp(H), blocks = (n + 127) / 128;
    const Offsets &o = net->off;
    const Packed w(net);
    k_mlp_train<<<blocks, GU_THREADS, tr_smem(H), s>>>(X, t, n, H, hp, 512, w.W1, w.W2, w.W2T, net->p + o.b1, net->p + o.b2,
                                                       net->p + o.w3, net->p + o.b3, net->y, net->part, ctx_err(net->ctx));
    MCK(cudaGetLastError());
    const long long total = (long long)H * H + 144LL * H + 2 * H + 2;
    k_train_sums<<<(unsigned)((total + 31) / 32), 32 * TS_SLICES, 0, s>>>(net->part, blocks, H, tr_part(H), o, n, g, loss);
    MCK(cudaGetLastError());
    return BC_OK;
}

// the hidden layers into net->h1, net->h2
bc_status hidden_layers(bc_mlp_t net, const float *X, int n, cudaStream_t s)
{
    const int H = net->H;
    const Offsets &o = net->off;
    GemmArgs a1{X, KPAD, 1, net->p + o.W1, 1, KIN, net->h1, H, 1, n, H, KPAD, net->p + o.b1, 1};
    // W1 is stored [H][132]; rows of X are padded to 144 with zeros, so K runs to 144 and
    // B(k, n) = W1[n][k] must be zero for k >= 132: bound K by 132 instead.
    a1.K = KIN;
    a1.err = ctx_err(net->ctx);
    MCK(gemm(a1, s));
    GemmArgs a2{net->h1, H, 1, net->p + o.W2, 1, H, net->h2, H, 1, n, H, H, net->p + o.b2, 1};
    a2.err = ctx_err(net->ctx);
    MCK(gemm(a2, s));
    return BC_OK;
}

// forward pass into net->h1, net->h2, y
bc_status forward(bc_mlp_t net, const float *X, int n, float *y, cudaStream_t s)
{
    if (net->wp) return fused_forward(net, X, n, y, s);
    if (bc_status st = hidden_layers(net, X, n, s)) return st;
    const Offsets &o = net->off;
    k_head<<<(n + 7) / 8, 256, 0, s>>>(net->h2, net->p + o.w3, net->p + o.b3, n, net->H, y);
    MCK(cudaGetLastError());
    return BC_OK;
}

// forward pass (net->y), the gradients of the mean squared error into net->g -- or,
// where given, into `grads` -- and the error itself into loss (may be null)
bc_status forward_backward(bc_mlp_t net, const float *X, const float *t, int n, float *grads, float *loss, cudaStream_t s)
{
    if (net->wp && n <= TR_MAX_ROWS) return fused_train(net, X, t, n, grads ? grads : net->g, loss, s);
    if (bc_status st = hidden_layers(net, X, n, s)) return st;
    const int H = net->H;
    const Offsets &o = net->off;
    // y, gy, dh2 and the sums over the batch: dw3, db2, db3
    MCK(head_train(net->h2, net->p + o.w3, net->p + o.b3, t, n, H, net->y, net->gy, net->dh2, net->part,
                   net->part_floats, net->g + o.w3, net->g + o.b2, net->g + o.b3, s));
    // dW2 = dh2^T h1  (M = H out, N = H in, K = n)
    GemmArgs w2{net->dh2, 1, H, net->h1, H, 1, net->g + o.W2, H, 1, H, H, n, nullptr, 0};
    w2.err = ctx_err(net->ctx);
    MCK(gemm_splitk(w2, net->part, net->part_floats, s));
    // dh1 = bf16(dh2 W2) where h1 > 0, else 0  (M = n, N = H in, K = H out)
    GemmArgs d1{net->dh2, H, 1, net->p + o.W2, H, 1, net->dh1, H, 1, n, H, H, nullptr, 0};
    d1.err = ctx_err(net->ctx);
    d1.mask = net->h1;
    MCK(gemm(d1, s));
    // [dW1 | db1] = dh1^T [X | 1]  (M = H, N = 132 + 1, K = n): the column of ones gives db1 = sum_b dh1[b]
    GemmArgs w1{net->dh1, 1, H, X, KPAD, 1, net->g + o.W1, KIN, 1, H, KIN + 1, n, nullptr, 0};
    w1.err = ctx_err(net->ctx);
    w1.bone = KIN;
    MCK(gemm_splitk(w1, net->part, net->part_floats, s, net->g + o.b1));
    if (loss) {
        k_loss<<<1, 256, 0, s>>>(net->y, t, n, loss);
        MCK(cudaGetLastError());
    }
    if (grads) MCK(cudaMemcpyAsync(grads, net->g, sizeof(float) * (size_t)net->off.total, cudaMemcpyDeviceToDevice, s));
    return BC_OK;
}

} // namespace

cudaError_t bc::launch_topk(const float *scores, int n, int k, int *idx, cudaStream_t s)
{
    int P = 1;
    while (P < n) P <<= 1;
    if (P < 2) P = 2;
    const size_t smem = sizeof(unsigned long long) * P;
    cudaError_t e = cudaFuncSetAttribute(k_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_topk<<<1, 1024, smem, s>>>(scores, n, P, k, idx);
    return cudaGetLastError();
}

__global__ void k_moments(const float2 *__restrict__ F, const int *__restrict__ modes, int count, int N, int H, bool line,
                          float *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int mx = modes[3 * i], my = modes[3 * i + 1], mz = modes[3 * i + 2];
    const int jx = mx < 0 ? mx + N : mx, jy = my < 0 ? my + N : my;
    const float2 v = F[line ? ((long long)mz * N + jy) * N + jx : ((long long)jx * N + jy) * H + mz];
    out[i] = sqrtf(v.x * v.x + v.y * v.y) / F[0].x;
}

cudaError_t bc::launch_moments(const float2 *F, const int *modes, int count, int N, int H, bool line, float *out,
                               cudaStream_t s)
{
    k_moments<<<(count + 63) / 64, 64, 0, s>>>(F, modes, count, N, H, line, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ moments of a rotated shape
// m_{R S}[i] = |f^_S(R^T m_i)| / f^_S(0) (the moments of S turned by R) by direct
// sums over the knots, f^_S(k) = sum_i h^(rho_{l_i}, |k|) exp(-2 pi i k . c_i / P)
// (Eq. (fballhat) without spreading: the band-limited spectrum at off-grid
// frequencies), for many rotations.  The mode table is compiled in (the 64 lowest
// modes are the same for every N >= 8: |m|^2 <= 9, so no component exceeds 3 and
// two or three nonzero ones are at most 2); the context checks it against the one
// it builds.
//
// With c_a, s_a = cos, sin of m_a 2 pi (R c)_a / P, the phase of a mode is
// prod_a (c_a - i s_a), so the modes (+-m_x, +-m_y, +-m_z) are signed sums of the
// 2^d real sums over the knots of h^ prod_a (c_a or s_a), d the number of nonzero
// components.  Those 122 sums are what a thread accumulates: one FMA per sum and
// knot, the products of two axes shared by the modes of the third -- a mode
// costs 2 FMAs per knot instead of up to two complex products and two FMAs (4,096
// rotations of 5,000 knots: 437 -> 223 us, bound by instruction issue; 167
// registers, three blocks per SM).  One block per rotation, thread j takes the knots j, j + 128, ...; the sums of a
// warp are reduced by exchanging halves (each of the five steps halves the
// values a lane holds), the four warps in a fixed order.
constexpr int MR_THREADS = 128, MR_SHELLS = 10, MR_SUMS = 128;
// accumulators: [0] h^(rho, 0); axis a, m = 1 .. 3: 1 + 6 a + 2 (m - 1) + (c, s);
// axes (0, 1), (0, 2), (1, 2), m, m' = 1, 2: 19 + 16 pair + 8 (m - 1) + 4 (m' - 1) + (cc, cs, sc, ss);
// three axes, triple t: 67 + 8 t + (ccc, ccs, csc, css, scc, scs, ssc, sss)
constexpr int MR_ONE = 1, MR_TWO = 19, MR_THREE = 67;
// the triples (m_x, m_y, m_z) of |m|^2 <= 9: 111, 112, 121, 211, 122, 212, 221
__host__ __device__ constexpr int mr_triple(int mx, int my, int mz)
{
    return mx * my * mz == 1 ? 0 : mx * my * mz == 2 ? (mz == 2 ? 1 : my == 2 ? 2 : 3) : mx == 1 ? 4 : my == 1 ? 5 : 6;
}

// components of mode i offset by 'D' ('A' = -3 .. 'G' = +3), in the order of the table
__host__ __device__ constexpr int mr_mode(int i, int a)
{
    return "CDDDCDDDEDEDEDDCCDCDECEDDCEDEEECDEDEEEDCCECEEECEEEEBDDDBDDDFDFDFDDBCDBDEBEDCBDCDFCFDDBEDCFDEFDFEEBDEDFEFDFCDFDEF"
           "EDBCEBEECBECCFCEFCFEEBEECFEEFEFEFCEFEEBBDBDFBFDDBFDFFFBDFDFFFDADDBBEBCFBEFBFECBF"[3 * i + a] -
           'D';
}

__host__ __device__ constexpr bool mr_covered(int i)
{
    const int x = mr_mode(i, 0), y = mr_mode(i, 1), z = mr_mode(i, 2);
    return x * x + y * y + z * z < MR_SHELLS && x * x + y * y + z * z > 0;
}
template <int... I>
__host__ __device__ constexpr bool mr_all_covered(std::integer_sequence<int, I...>) { return (mr_covered(I) && ...); }
static_assert(mr_all_covered(std::make_integer_sequence<int, BC_MOMENTS>{}), "the moment modes lie in |m|^2 <= 9");

__global__ void __launch_bounds__(MR_THREADS, 3) k_moments_rot(const float4 *__restrict__ knots, int nk,
                                                               const float *__restrict__ quats,
                                                               const float *__restrict__ ballft, int qstride, int L,
                                                               float two_over_P, float *out, int *err)
{
    __shared__ float wq_all[BC_MAX_LEVELS * MR_SHELLS];
    __shared__ float red[MR_THREADS / 32][MR_SUMS];
    const int r = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < L * MR_SHELLS; e += MR_THREADS) {
        const int l = e / MR_SHELLS, q = e - l * MR_SHELLS;
        wq_all[e] = q < qstride ? ballft[(long long)l * qstride + q] : 0.f;
    }
    float qw = quats[4 * r], qx = quats[4 * r + 1], qy = quats[4 * r + 2], qz = quats[4 * r + 3];
    const float nq = qw * qw + qx * qx + qy * qy + qz * qz;
    if (!(nq > 0.f)) {
        if (threadIdx.x == 0) atomicOr(err, 4);
        qw = 1.f, qx = qy = qz = 0.f;
    } else {
        const float s = rsqrtf(nq);
        qw *= s, qx *= s, qy *= s, qz *= s;
    }
    const float R[9] = {1.f - 2.f * (qy * qy + qz * qz), 2.f * (qx * qy - qw * qz), 2.f * (qx * qz + qw * qy),
                        2.f * (qx * qy + qw * qz), 1.f - 2.f * (qx * qx + qz * qz), 2.f * (qy * qz - qw * qx),
                        2.f * (qx * qz - qw * qy), 2.f * (qy * qz + qw * qx), 1.f - 2.f * (qx * qx + qy * qy)};
    __syncthreads();
    float acc[MR_SUMS];
#pragma unroll
    for (int j = 0; j < MR_SUMS; j++) acc[j] = 0.f;
    for (int i = threadIdx.x; i < nk; i += MR_THREADS) {
        const float4 k = knots[i];
        const float *wq = wq_all + __float_as_int(k.w) * MR_SHELLS; // h^(rho_l, 2 pi sqrt(q) / P), q = |m|^2
        float c[3][4], s[3][4]; // cos, sin of m theta_a
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const float p = fmaf(R[3 * a], k.x, fmaf(R[3 * a + 1], k.y, R[3 * a + 2] * k.z));
            sincospif(two_over_P * p, &s[a][1], &c[a][1]);
            s[a][2] = 2.f * s[a][1] * c[a][1];
            c[a][2] = fmaf(c[a][1], c[a][1], -s[a][1] * s[a][1]);
            s[a][3] = fmaf(s[a][2], c[a][1], c[a][2] * s[a][1]);
            c[a][3] = fmaf(c[a][2], c[a][1], -s[a][2] * s[a][1]);
        }
        acc[0] += wq[0];
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int m = 1; m <= 3; m++) {
                float *o = acc + MR_ONE + 6 * a + 2 * (m - 1);
                o[0] = fmaf(wq[m * m], c[a][m], o[0]);
                o[1] = fmaf(wq[m * m], s[a][m], o[1]);
            }
#pragma unroll
        for (int pr = 0; pr < 3; pr++) {
            const int a = pr == 2 ? 1 : 0, b = pr == 0 ? 1 : 2;
#pragma unroll
            for (int m = 1; m <= 2; m++)
#pragma unroll
                for (int n = 1; n <= 2; n++) {
                    const float cc = c[a][m] * c[b][n], cs = c[a][m] * s[b][n], sc = s[a][m] * c[b][n], ss = s[a][m] * s[b][n];
                    const float w = wq[m * m + n * n];
                    float *o = acc + MR_TWO + 16 * pr + 8 * (m - 1) + 4 * (n - 1);
                    o[0] = fmaf(w, cc, o[0]);
                    o[1] = fmaf(w, cs, o[1]);
                    o[2] = fmaf(w, sc, o[2]);
                    o[3] = fmaf(w, ss, o[3]);
                    if (pr == 0)
#pragma unroll
                        for (int u = 1; u <= 2; u++) {
                            if (m * m + n * n + u * u > 9) continue; // 222
                            const float v = wq[m * m + n * n + u * u], wc = v * c[2][u], ws = v * s[2][u];
                            float *t = acc + MR_THREE + 8 * mr_triple(m, n, u);
                            t[0] = fmaf(cc, wc, t[0]);
                            t[1] = fmaf(cc, ws, t[1]);
                            t[2] = fmaf(cs, wc, t[2]);
                            t[3] = fmaf(cs, ws, t[3]);
                            t[4] = fmaf(sc, wc, t[4]);
                            t[5] = fmaf(sc, ws, t[5]);
                            t[6] = fmaf(ss, wc, t[6]);
                            t[7] = fmaf(ss, ws, t[7]);
                        }
                }
        }
    }
    // lane l ends with the warp's sums 4 l .. 4 l + 3
#pragma unroll
    for (int o = 16, half = MR_SUMS / 2; o > 0; o >>= 1, half >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < half; j++) {
            const float keep = up ? acc[j + half] : acc[j], send = up ? acc[j] : acc[j + half];
            acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int j = 0; j < 4; j++) red[warp][4 * lane + j] = acc[j];
    __syncthreads();
    float sum = red[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < MR_THREADS / 32; w++) sum += red[w][threadIdx.x];
    __syncthreads();
    float *S = red[0];
    S[threadIdx.x] = sum;
    __syncthreads();
    if (threadIdx.x < BC_MOMENTS) {
        const int i = threadIdx.x, m[3] = {mr_mode(i, 0), mr_mode(i, 1), mr_mode(i, 2)};
        const int x = abs(m[0]), y = abs(m[1]), z = abs(m[2]);
        const float gx = m[0] < 0 ? -1.f : 1.f, gy = m[1] < 0 ? -1.f : 1.f, gz = m[2] < 0 ? -1.f : 1.f; // sines' signs
        float re, im; // |f^| does not depend on the sign of the imaginary part
        if (x && y && z) {
            const float *t = S + MR_THREE + 8 * mr_triple(x, y, z);
            re = t[0] - gy * gz * t[3] - gx * gz * t[5] - gx * gy * t[6];
            im = gz * t[1] + gy * t[2] + gx * t[4] - gx * gy * gz * t[7];
        } else if ((x && y) || (x && z) || (y && z)) {
            const int pr = x && y ? 0 : x ? 1 : 2, a = pr == 2 ? y : x, b = pr == 0 ? y : z;
            const float ga = pr == 2 ? gy : gx, gb = pr == 0 ? gy : gz;
            const float *t = S + MR_TWO + 16 * pr + 8 * (a - 1) + 4 * (b - 1);
            re = t[0] - ga * gb * t[3];
            im = gb * t[1] + ga * t[2];
        } else {
            const float *t = S + MR_ONE + (x ? 0 : y ? 6 : 12) + 2 * (x + y + z - 1);
            re = t[0];
            im = t[1];
        }
        out[(long long)r * BC_MOMENTS + i] = sqrtf(re * re + im * im) / S[0];
    }
}

cudaError_t bc::launch_moments_rot(const float4 *knots, int nk, const float *quats, int n, const float *ballft,
                                   int qstride, int L, float two_over_P, float *out, int *err, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_moments_rot<<<n, MR_THREADS, 0, s>>>(knots, nk, quats, ballft, qstride, L, two_over_P, out, err);
    return cudaGetLastError();
}

bool bc::moments_rot_table_matches(const int *tab)
{
    for (int i = 0; i < BC_MOMENTS; i++)
        for (int a = 0; a < 3; a++)
            if (tab[3 * i + a] != mr_mode(i, a)) return false;
    return true;
}

cudaError_t bc::launch_gather_quats(const float *q, const int *idx, int k, float *out, cudaStream_t s)
{
    if (k <= 0) return cudaSuccess;
    k_gather_quats<<<(4 * k + 255) / 256, 256, 0, s>>>(q, idx, k, out);
    return cudaGetLastError();
}

cudaError_t bc::launch_compose_quats(const float *sq, const float *q, int n, float *out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_compose_quats<<<(n + 255) / 256, 256, 0, s>>>(make_float4(sq[0], sq[1], sq[2], sq[3]), q, n, out);
    return cudaGetLastError();
}

cudaError_t bc::launch_axpby(float *y, const float *x, int n, float alpha, float beta, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_axpby<<<(n + 255) / 256, 256, 0, s>>>(y, x, n, alpha, beta);
    return cudaGetLastError();
}

void bc::mlp_orphan(bc_mlp_s *net)
{
    // p heads the allocation that also holds m, loss that of wp
    float *bufs[] = {net->p, net->v, net->g, net->loss, net->h1, net->h2, net->y, net->gy, net->dh2, net->dh1, net->part, net->xb, net->tb};
    for (float *b : bufs)
        if (b) cudaFree(b);
    net->p = net->m = net->v = net->g = net->h1 = net->h2 = net->y = net->gy = net->dh2 = net->dh1 = net->loss = nullptr;
    net->part = net->xb = net->tb = nullptr;
    net->wp = nullptr;
    net->cap = net->ycap = net->xb_cap = 0;
    net->part_floats = 0;
    net->ctx = nullptr;
}

extern "C" {

bc_status bc_mlp_create(bc_ctx_t ctx, int hidden, const float *init, bc_mlp_t *out)
{
    try {
        if (!ctx || !init || !out) return mfail(BC_ERR_ARG, "bc_mlp_create: null argument");
        *out = nullptr;
        if (hidden < 16 || hidden > 1024 || hidden % 16) return mfail(BC_ERR_ARG, "bc_mlp_create: hidden must be a multiple of 16 in [16, 1024]");
        bc_mlp_t net = new (std::nothrow) bc_mlp_s();
        if (!net) return mfail(BC_ERR_OOM, "bc_mlp_create: host allocation failed");
        net->ctx = ctx;
        net->H = hidden;
        net->off = offsets(hidden);
        const size_t bytes = sizeof(float) * (size_t)net->off.total;
        cudaStream_t s = ctx_stream(ctx);
        cudaError_t e;
        // parameters and first moments; second moments; the loss word and the BF16 weight blocks.
        // (At H = 256 these stay below the 2 MB that cudaMalloc maps at a time; with the
        // gradients, which come with the first training pass, a network took 160 us, not 40.)
        const size_t row = (size_t)((net->off.total + 63) & ~63LL), fused = hidden <= FW_MAXH;
        const size_t wbytes = fused ? (size_t)(3 + 2 * (fw_hp(hidden) / 64)) * hidden * 128 : 0;
        if ((e = cudaMalloc(&net->p, sizeof(float) * 2 * row)) != cudaSuccess ||
            (e = cudaMalloc(&net->v, bytes)) != cudaSuccess ||
            (e = cudaMalloc(&net->loss, sizeof(float) * 64 + wbytes)) != cudaSuccess) {
            bc_mlp_destroy(net);
            return mcuda(e, "bc_mlp_create: cudaMalloc");
        }
        net->m = net->p + row;
        if (fused) {
            net->wp = reinterpret_cast<uint8_t *>(net->loss + 64);
            if ((e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, fw_smem(FW_MAXH))) != cudaSuccess ||
                (e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, tr_smem(FW_MAXH))) != cudaSuccess) {
                bc_mlp_destroy(net);
                return mcuda(e, "bc_mlp_create: fused passes");
            }
        }
        if ((e = cudaMemcpyAsync(net->p, init, bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
            (e = cudaMemsetAsync(net->m, 0, bytes, s)) != cudaSuccess || (e = cudaMemsetAsync(net->v, 0, bytes, s)) != cudaSuccess ||
            (e = pack_weights(net, s)) != cudaSuccess || (e = cudaStreamSynchronize(s)) != cudaSuccess) {
            bc_mlp_destroy(net);
            return mcuda(e, "bc_mlp_create: upload");
        }
        ctx_register_mlp(ctx, net);
        *out = net;
        return BC_OK;
    } catch (...) {
        return mfail(BC_ERR_INTERNAL, "bc_mlp_create: unexpected exception");
    }
}

bc_status bc_mlp_destroy(bc_mlp_t net)
{
    if (!net) return BC_OK;
    if (net->ctx) {
        cudaStreamSynchronize(ctx_stream(net->ctx));
        ctx_unregister_mlp(net->ctx, net);
        mlp_orphan(net);
    }
    delete net;
    return BC_OK;
}

long long bc_mlp_param_count(int hidden) { return offsets(hidden).total; }

static bc_status features_impl(bc_mlp_t net, const float *quats, int n, const float *fa, const float *fb,
                               long long ldb, float *X, const char *who)
{
    if (!net || !quats || !fa || !fb || !X || n < 1) return mfail(BC_ERR_ARG, std::string(who) + ": bad arguments");
    if (!net->ctx) return mfail(BC_ERR_ARG, std::string(who) + ": the network's context was destroyed");
    const long long total = (long long)n * KPAD;
    k_features<<<(unsigned)((total + 255) / 256), 256, 0, ctx_stream(net->ctx)>>>(quats, n, fa, fb, ldb, X,
                                                                                  ctx_err(net->ctx));
    MCK(cudaGetLastError());
    return BC_OK;
}

bc_status bc_mlp_features(bc_mlp_t net, const float *quats, int n, const float *fa, const float *fb, float *X)
{
    return features_impl(net, quats, n, fa, fb, 0, X, "bc_mlp_features");
}

bc_status bc_mlp_features_rows(bc_mlp_t net, const float *quats, int n, const float *fa, const float *fb_rows, float *X)
{
    return features_impl(net, quats, n, fa, fb_rows, BC_MOMENTS, X, "bc_mlp_features_rows");
}

bc_status bc_mlp_set_features(bc_mlp_t net, int rotated_moments)
{
    if (!net || (rotated_moments != 0 && rotated_moments != 1))
        return mfail(BC_ERR_ARG, "bc_mlp_set_features: null network, or rotated_moments not 0 or 1");
    net->rotated_moments = rotated_moments;
    return BC_OK;
}

int bc_mlp_rotated_moments(bc_mlp_t net) { return net ? net->rotated_moments : 0; }

bc_status bc_mlp_predict(bc_mlp_t net, const float *X, int n, float *y)
{
    try {
        if (!net || !X || !y || n < 1) return mfail(BC_ERR_ARG, "bc_mlp_predict: bad arguments");
        if (!net->ctx) return mfail(BC_ERR_ARG, "bc_mlp_predict: the network's context was destroyed");
        if (!net->wp) // the fused pass needs no buffers
            if (bc_status st = ensure_batch(net, n)) return st;
        return forward(net, X, n, y, ctx_stream(net->ctx));
    } catch (...) {
        return mfail(BC_ERR_INTERNAL, "bc_mlp_predict: unexpected exception");
    }
}

bc_status bc_mlp_grads(bc_mlp_t net, const float *X, const float *t, int n, float *grads, float *loss)
{
    try {
        if (!net || !X || !t || n < 1) return mfail(BC_ERR_ARG, "bc_mlp_grads: bad arguments");
        if (!net->ctx) return mfail(BC_ERR_ARG, "bc_mlp_grads: the network's context was destroyed");
        if (bc_status st = ensure_batch(net, n)) return st;
        cudaStream_t s = ctx_stream(net->ctx);
        if (bc_status st = forward_backward(net, X, t, n, grads, loss, s)) return st;
        return BC_OK;
    } catch (...) {
        return mfail(BC_ERR_INTERNAL, "bc_mlp_grads: unexpected exception");
    }
}

bc_status bc_mlp_train_step(bc_mlp_t net, const float *X, const float *t, int n, float lr, float *loss)
{
    try {
        if (!net || !X || !t || n < 1 || !(lr > 0.f)) return mfail(BC_ERR_ARG, "bc_mlp_train_step: bad arguments");
        if (bc_status st = bc_mlp_grads(net, X, t, n, nullptr, loss)) return st;
        MCK(adam(net, lr, ctx_stream(net->ctx)));
        return BC_OK;
    } catch (...) {
        return mfail(BC_ERR_INTERNAL, "bc_mlp_train_step: unexpected exception");
    }
}

// Pseudo-random order of epoch `e`: perm(i) = (a i + c) mod n with a coprime
// to n, both drawn from splitmix64 of (seed, e) -- a bijection of [0, n).
static void epoch_order(unsigned long long seed, int e, int n, long long *a, long long *c)
{
    auto mix = [](unsigned long long z) {
        z += 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    auto gcd = [](long long x, long long y) {
        while (y) {
            const long long t = x % y;
            x = y;
            y = t;
        }
        return x;
    };
    long long aa = (long long)(mix(seed * 0x100000001B3ull + 2ull * (unsigned)e) % (unsigned long long)n);
    if (aa == 0) aa = 1;
    while (gcd(aa, n) != 1) aa = aa + 1 < n ? aa + 1 : 1;
    *a = aa;
    *c = (long long)(mix(seed * 0x100000001B3ull + 2ull * (unsigned)e + 1ull) % (unsigned long long)n);
}

bc_status bc_mlp_train(bc_mlp_t net, const float *X, const float *t, int n, int batch, int epochs, float lr,
                       unsigned long long seed, float *loss)
{
    try {
        if (!net || !X || !t || n < 1 || batch < 1 || batch > n || epochs < 1 || !(lr > 0.f))
            return mfail(BC_ERR_ARG, "bc_mlp_train: bad arguments");
        if (!net->ctx) return mfail(BC_ERR_ARG, "bc_mlp_train: the network's context was destroyed");
        if (bc_status st = ensure_batch(net, batch)) return st;
        cudaStream_t s = ctx_stream(net->ctx);
        if (batch > net->xb_cap) {
            if (net->xb) cudaFree(net->xb);
            if (net->tb) cudaFree(net->tb);
            net->xb = net->tb = nullptr;
            net->xb_cap = 0;
            MCK(cudaMalloc(&net->xb, sizeof(float) * (size_t)batch * KPAD));
            MCK(cudaMalloc(&net->tb, sizeof(float) * (size_t)batch));
            net->xb_cap = batch;
        }
        const int steps = n / batch;
        const bool x16 = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
        for (int e = 0; e < epochs; e++) {
            long long a = 1, c = 0;
            epoch_order(seed, e, n, &a, &c);
            const float lr_e = (float)(lr * 0.5 * (1.0 + std::cos(M_PI * e / epochs)));
            for (int st = 0; st < steps; st++) {
                if (x16) {
                    const long long tot = (long long)batch * (KPAD / 4);
                    k_gather_batch4<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(
                        reinterpret_cast<const float4 *>(X), t, n, a, c, st * batch, batch,
                        reinterpret_cast<float4 *>(net->xb), net->tb);
                } else {
                    const long long tot = (long long)batch * KPAD;
                    k_gather_batch<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(X, t, n, a, c, st * batch, batch,
                                                                                 net->xb, net->tb);
                }
                MCK(cudaGetLastError());
                if (bc_status r = forward_backward(net, net->xb, net->tb, batch, nullptr, nullptr, s)) return r;
                MCK(adam(net, lr_e, s));
            }
        }
        if (loss) {
            // the loss of the last batch at the parameters it was taken with
            k_loss<<<1, 256, 0, s>>>(net->y, net->tb, batch, loss);
            MCK(cudaGetLastError());
        }
        return BC_OK;
    } catch (...) {
        return mfail(BC_ERR_INTERNAL, "bc_mlp_train: unexpected exception");
    }
}

bc_status bc_mlp_state(bc_mlp_t net, float *params, float *m, float *v, long long *step, int get)
{
    if (!net || !net->ctx) return mfail(BC_ERR_ARG, "bc_mlp_state: null network or destroyed context");
    cudaStream_t s = ctx_stream(net->ctx);
    const size_t bytes = sizeof(float) * (size_t)net->off.total;
    float *host[3] = {params, m, v};
    float *dev[3] = {net->p, net->m, net->v};
    for (int i = 0; i < 3; i++) {
        if (!host[i]) continue;
        if (get) MCK(cudaMemcpyAsync(host[i], dev[i], bytes, cudaMemcpyDeviceToHost, s));
        else MCK(cudaMemcpyAsync(dev[i], host[i], bytes, cudaMemcpyHostToDevice, s));
        if (!get && i == 0) MCK(pack_weights(net, s));
    }
    MCK(cudaStreamSynchronize(s));
    if (step) {
        if (get) *step = net->step;
        else net->step = *step;
    }
    return BC_OK;
}

} // extern "C"
