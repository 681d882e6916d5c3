// Back half of a correlation pass whose front half ran in bc_front.cu: the x
// transforms with the window deconvolution, ball transforms and level sum of
// Eq. (fballhat), the conjugate product of Eq. (ccghat) and the inverse x
// transform (k_xw); the inverse y and z transforms of whole planes (k_iyz).
// Every line of a transform stays inside one warp (bc_wfft.cuh).
#include <algorithm>

#include "bc_passes.cuh"
#include "bc_umma.cuh"
#include "bc_wfft.cuh"

namespace bc {

// ------------------------------------------------------------------ level weights
// wl[((m_z N/XL + ch) L + l) XL + c][a], a = |m_x| in [0, N/2], j_y = XL ch + c:
// ballft_l(a^2 + m_y^2 + m_z^2) D(a) D(m_y) D(m_z).  One (item, level) is one
// contiguous run of XL (N/2 + 1) floats, fetched with the level's rows.
__global__ void k_build_wl(int N, int L, int qmax, const float *__restrict__ deconv, const float *__restrict__ ballft,
                           float *wl)
{
    const int A = N / 2 + 1, nch = N / XL;
    const long long total = (long long)(N / 2) * nch * L * XL * A, Q = qmax + 1;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int a = (int)(e % A), c = (int)((e / A) % XL), l = (int)((e / ((long long)A * XL)) % L);
        const long long item = e / ((long long)A * XL * L);
        const int ch = (int)(item % nch), mz = (int)(item / nch), jy = ch * XL + c, my = mode_of(jy, N);
        wl[e] = ballft[l * Q + a * a + my * my + mz * mz] * (deconv[a] * deconv[jy] * deconv[mz]);
    }
}

size_t wl_floats(const Geometry &g) { return (size_t)(g.N / 2) * (g.N / XL) * g.L * XL * (g.N / 2 + 1); }

cudaError_t launch_build_wl(const Geometry &g, const float *deconv, const float *ballft, float *wl, cudaStream_t s)
{
    k_build_wl<<<1024, 256, 0, s>>>(g.N, g.L, 3 * (g.N / 2) * (g.N / 2), deconv, ballft, wl);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ x pass
// Item: (m_z, XL consecutive j_y) of a pair: XL lines along x for every level of
// both instances.  A phase (instance, level) is one bulk copy of the item's b0
// rows of 64 bytes (contiguous in y1) and one of its level weights into a ring
// stage; thread 0 issues them XW_STAGES - 1 phases ahead, across items, and every
// warp runs its lines at its own pace: it waits for the stage, transforms,
// adds weight x mode to its level sum in registers and releases the stage.  After
// an instance's last level the sum takes the phase of the box origins.  A lane
// ends up with modes j + R0 r (8 per line) of both spectra, which are the first-
// stage inputs of the inverse transform, so the conjugate product needs no
// exchange.  With pr.a < 0 the spectrum of A comes from fa (layout
// [m_z][j_y][j_x]); with pr.b < 0 it is written there and nothing else happens.
// Output h[k_x][m_z][j_y].  Every wait is bounded (bit 8 of the error word); a warp
// whose wait expired leaves the walk, but takes part in the block's barriers of the
// rest of it (going on through the walk instead cost a percent of every call).
// EXPIRE (the self-test): the second phase's wait of warp 0 counts as expired.
// Bound by instructions and latency (issue 57%, 128 registers).  20,000 + 20,000
// balls, N = 128, L = 4: 37.3 us (k_fft_x 38.7 us); the walk's state in every thread's
// registers instead of shared memory 44.5 us.  Items of 8 lines, not 16: the same time
// at that size, more items for small grids.
constexpr int XW_STAGES = 3, XW_ERR = 8, XW_RW = 6;

template <int NF, int LW>
struct XW {
    static constexpr int WARPS = XL / LW, THREADS = WARPS * 32;
    static constexpr int A = NF / 4 + 1, WBYTES = XL * A * 4;
    static constexpr int EL = WF<NF>::ES > WF<NF>::R0 * WI_ROW ? WF<NF>::ES : WF<NF>::R0 * WI_ROW; // per line
    static constexpr int OUT = WF<NF>::N * XL;                                                     // output tile
    static constexpr int EALL = XL * EL > OUT ? XL * EL : OUT; // exchange tiles; the output tile shares them
    __host__ __device__ static constexpr size_t stage_bytes(int cap) { return (size_t)cap * XL * 8 + WBYTES; }
    __host__ __device__ static constexpr size_t smem(int cap)
    {
        return 8 * ((size_t)EALL + NF + WF<NF>::N + (15 - XW_RW) * 16) + XW_STAGES * stage_bytes(cap) + 128;
    }
    static_assert(WBYTES % 16 == 0, "bulk copies");
};

// The copy thread's place in the block's sequence of phases (pairs in order, the
// block's items of a pair, A if computed, then B, the levels of each), kept in
// shared memory: only thread 0 uses it, and its registers are every thread's.
struct XwCopies {
    const float2 *src; // the next phase's rows, and the step to the next level's
    const float *wsrc; // its weights
    long long lstride;
    uint32_t bytes;
    int left;          // levels left of this instance
    int pi, it, b, rot; // pair, item, whether B is next
    int issued, st, par;
    bool done;
};

template <int NF, int LW, bool EXPIRE = false>
__global__ void __launch_bounds__(XW<NF, LW>::THREADS, 512 / XW<NF, LW>::THREADS)
k_xw(Geometry g, Tables tb, const InstDesc *__restrict__ inst, const InstPlan *__restrict__ plan,
     const PairDesc *__restrict__ pairs, int npairs, const float2 *__restrict__ y1, const float2 *__restrict__ fa_cache,
     float2 *fa_out, float2 *h, int *err, int cap)
{
    using F = WF<NF, LW>;
    using X = XW<NF, LW>;
    constexpr int R0 = F::R0, N = F::N, H = F::H, A = X::A, nch = N / XL, items = H * nch;
    extern __shared__ float4 sm4[];
    __shared__ XwCopies cp;
    float2 *Eall = reinterpret_cast<float2 *>(sm4), *twF = Eall + X::EALL, *twN = twF + NF, *twL = twN + N;
    uint8_t *ring = reinterpret_cast<uint8_t *>(twL + (15 - XW_RW) * 16);
    const int sbytes = (int)X::stage_bytes(cap);
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + XW_STAGES * sbytes);
    volatile int *stop = reinterpret_cast<volatile int *>(bars + 2 * XW_STAGES);
    const uint32_t FULL = smem_addr(bars), EMPTY = FULL + 8 * XW_STAGES;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, L = g.L;
    if (threadIdx.x == 0) {
        for (int k = 0; k < XW_STAGES; k++) {
            mbar_init(FULL + 8 * k, 1);
            mbar_init(EMPTY + 8 * k, X::WARPS);
        }
        *stop = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int k = threadIdx.x; k < NF; k += X::THREADS) twF[k] = tb.tw_n[k];
    for (int k = threadIdx.x; k < N; k += X::THREADS) twN[k] = tb.tw_N[k];
    float2 w[XW_RW + 1];
    wf_twiddles<NF, XW_RW>(tb.tw_n, lane, w);
    wf_twiddle_table<NF, XW_RW>(tb.tw_n, twL);
    __syncthreads();
    pdl_signal();
    pdl_wait(); // earlier passes' outputs are read from here on
    float2 *E = Eall + warp * LW * X::EL;
    const int s = lane / R0, j = lane - s * R0; // last stage: line and butterfly
    const bool live = lane < F::LIVE;
    const int c = warp * LW + (live ? s : 0); // the lane's line of the item
    // thread 0: the next instance (B of this item, or the next item) becomes the copies' source
    auto next_source = [&]() {
        for (;;) {
            if (cp.it >= items) { // the next pair with an item for this block
                if (++cp.pi >= npairs) {
                    cp.done = true;
                    return;
                }
                cp.it = ((int)blockIdx.x - cp.rot + (int)gridDim.x) % (int)gridDim.x;
                cp.rot = (cp.rot + items) % (int)gridDim.x;
                cp.b = 0;
                continue;
            }
            const int si = cp.b ? pairs[cp.pi].b : pairs[cp.pi].a, it = cp.it;
            if (cp.b) {
                cp.b = 0;
                cp.it = it + (int)gridDim.x;
            } else {
                cp.b = 1;
            }
            if (si < 0) continue;
            const int b0 = plan[si].b[0];
            cp.src = y1 + inst[si].y1_off + (long long)it * b0 * XL;
            cp.lstride = (long long)items * b0 * XL;
            cp.bytes = (uint32_t)b0 * XL * 8;
            cp.wsrc = tb.wl + (long long)it * L * XL * A;
            cp.left = L;
            return;
        }
    };
    // thread 0: copies phases ahead of phase `used`, as far as the ring has room
    auto issue = [&](int used) {
        while (cp.issued < used + XW_STAGES && !cp.done) {
            // a phase that is not needed yet waits for a later call rather than hold this warp up
            if (cp.issued > used ? !mbar_poll(EMPTY + 8 * cp.st, cp.par ^ 1)
                                 : !umma_wait(EMPTY + 8 * cp.st, cp.par ^ 1, stop, err, XW_ERR))
                return;
            const uint32_t dst = smem_addr(ring) + cp.st * sbytes, bar = FULL + 8 * cp.st;
            mbar_expect_tx(bar, cp.bytes + X::WBYTES);
            if (cp.bytes) bulk_g2s(dst + X::WBYTES, cp.src, cp.bytes, bar);
            bulk_g2s(dst, cp.wsrc, X::WBYTES, bar);
            cp.src += cp.lstride;
            cp.wsrc += XL * A;
            cp.issued++;
            if (++cp.st == XW_STAGES) {
                cp.st = 0;
                cp.par ^= 1;
            }
            if (--cp.left == 0) next_source();
        }
    };
    if (threadIdx.x == 0) {
        cp.pi = -1;
        cp.it = items;
        cp.b = cp.rot = cp.issued = cp.st = cp.par = 0;
        cp.done = false;
        next_source();
        issue(0);
    }
    int used = 0, st = 0, par = 0, pi = 0, it = 0;
    bool ok = true;
    RotStart rs;
    for (; pi < npairs; pi++) {
        const PairDesc pr = pairs[pi];
        for (it = rs.first(); it < items; it += gridDim.x) {
            const int mz = it / nch, ch = it - mz * nch, jy = ch * XL + c, my = mode_of(jy, N);
            float2 FA[8], S[8];
            if (pr.a < 0) {
#pragma unroll
                for (int r = 0; r < 8; r++) FA[r] = fa_cache[(mz * N + jy) * N + (live ? j + R0 * r : 0)];
            }
            for (int half = pr.a < 0 ? 1 : 0; half < (pr.b < 0 ? 1 : 2); half++) {
                const InstPlan *p = plan + (half ? pr.b : pr.a);
                const int b0 = p->b[0], qx = (b0 + 63) >> 6;
#pragma unroll
                for (int r = 0; r < 8; r++) S[r] = make_float2(0.f, 0.f);
                for (int l = 0; l < L; l++, used++) {
                    if (threadIdx.x == 0) issue(used);
                    __syncwarp();
                    ok = __all_sync(0xffffffffu, umma_wait(FULL + 8 * st, par, stop, err, XW_ERR));
                    if constexpr (EXPIRE) {
                        if (warp == 0 && used == 1) {
                            ok = false;
                            if (lane == 0) {
                                atomicOr(err, XW_ERR);
                                *stop = 1;
                            }
                        }
                    }
                    if (!ok) break;
                    const float *wt = reinterpret_cast<const float *>(ring + st * sbytes) + c * A;
                    const float2 *T = reinterpret_cast<const float2 *>(ring + st * sbytes + X::WBYTES);
                    wf_first_any<NF, LW>(E, lane, qx, [&](int sl, int ix, bool inside) {
                        return inside || ix < b0 ? T[ix * XL + xl_place(warp * LW + sl, ix)] : make_float2(0.f, 0.f);
                    });
                    __syncwarp();
                    float2 o[16];
                    wf_last<NF, XW_RW, LW>(E, lane, w, o, twL);
#pragma unroll
                    for (int r = 0; r < 8; r++) { // mode j + R0 r (r < 4) or j + R0 r - N
                        const float m = wt[live ? (r < 4 ? j + R0 * r : N - (j + R0 * r)) : 0];
                        const float2 v = o[r < 4 ? r : r + 8];
                        S[r] = make_float2(fmaf(m, v.x, S[r].x), fmaf(m, v.y, S[r].y));
                    }
                    __syncwarp(); // every lane has read the stage and E
                    if (lane == 0) mbar_arrive(EMPTY + 8 * st);
                    if (++st == XW_STAGES) {
                        st = 0;
                        par ^= 1;
                    }
                }
                if (!ok) break;
                // this instance's level sum is complete: the box origins' phase
                const int px = p->pos0[0], base = (my + NF) * p->pos0[1] + mz * p->pos0[2];
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    const int mx = r < 4 ? j + R0 * r : j + R0 * r - N;
                    const float2 v = cscale(cmul(S[r], twF[((mx + NF) * px + base) % NF]), 0.5f);
                    if (half) S[r] = v;
                    else FA[r] = v;
                }
            }
            if (!ok) break;
            if (pr.b < 0) {
                if (live) {
#pragma unroll
                    for (int r = 0; r < 8; r++) fa_out[(mz * N + jy) * N + j + R0 * r] = FA[r];
                }
                continue;
            }
            // g' = P^-3 (-1)^(m_x + m_y + m_z) F_A conj(F_B), zero on the Nyquist planes
#pragma unroll
            for (int r = 0; r < 8; r++) {
                const int mx = r < 4 ? j + R0 * r : j + R0 * r - N;
                const float2 v = cscale(cmulc(FA[r], S[r]), ((mx + my + mz) & 1) ? -g.inv_P3 : g.inv_P3);
                S[r] = (jy == N / 2 || mx == -(N / 2)) ? make_float2(0.f, 0.f) : v;
            }
            if (live) wi_first<R0>(S, E + s * X::EL, j);
            __syncwarp();
            // last stage: lane -> (line, butterfly) = (lane / 8, lane mod 8), LW lines
            constexpr int IT2 = (LW * 8 + 31) / 32;
            float2 u[IT2][R0];
#pragma unroll
            for (int q = 0; q < IT2; q++) {
                const int sl = (lane >> 3) + 4 * q;
                if (sl < LW) wi_last<R0>(E + sl * X::EL, lane & 7, twN, u[q]);
            }
            __syncthreads(); // the exchange tiles become the output tile [k_x][place of the line]
#pragma unroll
            for (int q = 0; q < IT2; q++) {
                const int sl = (lane >> 3) + 4 * q;
                if (sl < LW) {
#pragma unroll
                    for (int r = 0; r < R0; r++) {
                        const int kx = (lane & 7) + 8 * r;
                        Eall[kx * XL + xl_place(warp * LW + sl, kx)] = u[q][r];
                    }
                }
            }
            __syncthreads();
            float2 *Hp = h + pr.h_off + (long long)mz * N + ch * XL;
#pragma unroll
            for (int e0 = 0; e0 < N * XL; e0 += X::THREADS) {
                const int e = e0 + threadIdx.x, kx = e / XL, cc = e % XL;
                Hp[kx * (H * N) + cc] = Eall[kx * XL + xl_place(cc, kx)];
            }
            __syncthreads();
        }
        if (!ok) break;
        rs.rot += items;
    }
    if (!ok) { // the walk from this item on, three barriers per item with an output (matched by number)
        for (bool here = true; pi < npairs; pi++, here = false) {
            if (!here) it = rs.first();
            for (const bool barriers = pairs[pi].b >= 0; it < items; it += gridDim.x)
                for (int k = 0; barriers && k < 3; k++) asm volatile("barrier.cta.sync 0;" ::: "memory");
            rs.rot += items;
        }
    }
    // the copies in flight land before the block's shared memory goes (a wait that
    // expired leaves some; otherwise all are complete)
    if (threadIdx.x == 0)
        for (int k = cp.issued - XW_STAGES < 0 ? 0 : cp.issued - XW_STAGES; k < cp.issued; k++) {
            const uint64_t t0 = global_ns();
            while (!mbar_test(FULL + 8 * (k % XW_STAGES), (k / XW_STAGES) & 1) && global_ns() - t0 < UMMA_WAIT_NS) {
            }
        }
}

// ------------------------------------------------------------------ inverse y and z
// One block per plane k_x: inverse y of its N/2 lines h[k_x][m_z][.] (read once,
// straight into first-stage registers), kept in shared memory as S[m_z][k_y];
// then the complex-to-real inverse z of row pairs, Z_k = A_k + i B_k (A_{N-k} =
// conj A_k, A_0 taken real, the m_z = N/2 term zero), whose pair (A_k, B_k) is
// one 16-byte load; finished rows leave through the warp's exchange tile so that
// each store covers whole rows.  With `keys` the block folds its largest value
// (lowest index on ties) into the pair's peak key.
// N = 128: 9.5 us, against 6.1 + 10.4 us of k_ifft_y and k_ifft_z.
template <int NI>
struct IYZ {
    static constexpr int R0 = NI / 8, H = NI / 2, LW = 4;   // lines of a warp per step
    static constexpr int THREADS = NI == 128 ? 512 : 256, WARPS = THREADS / 32;
    static constexpr int SS = NI + 2;                        // twice an odd number
    static constexpr int EL = R0 * WI_ROW;                   // exchange tile of a line
    static constexpr int FS = NI + 4;                        // finished rows: four row pairs on different banks
    static constexpr size_t smem = sizeof(float2) * ((size_t)H * SS + (size_t)WARPS * LW * EL + NI);
    static_assert(EL * 8 >= 2 * FS * 4, "two finished rows fit a line's exchange tile");
};

template <int NI>
__global__ void __launch_bounds__(IYZ<NI>::THREADS, NI == 128 ? 1 : 2)
k_iyz(Geometry g, Tables tb, const PairDesc *__restrict__ pairs, int npairs, const float2 *__restrict__ h, float *out,
      unsigned long long *keys)
{
    using I = IYZ<NI>;
    constexpr int R0 = I::R0, H = I::H, N = NI, LW = I::LW, SS = I::SS;
    __shared__ unsigned long long red[I::WARPS];
    extern __shared__ float4 sm4[];
    float2 *S = reinterpret_cast<float2 *>(sm4), *twN = S + H * SS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2 *E = twN + N + warp * LW * I::EL;
    for (int k = threadIdx.x; k < N; k += I::THREADS) twN[k] = tb.tw_N[k];
    pdl_signal();
    pdl_wait(); // earlier passes' outputs are read from here on
    __syncthreads();
    constexpr int IT = (LW * R0 + 31) / 32;
    const int sl = lane >> 3, jj = lane & 7; // last stage: line and butterfly
    const bool vec = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    const int units = npairs * N;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
        const int pi = u / N, kx = u - pi * N;
        const PairDesc pr = pairs[pi];
        if (pr.b < 0) continue; // uniform per pair
        const float2 *src = h + pr.h_off + (long long)kx * H * N;
        for (int m0 = warp * LW; m0 < H; m0 += I::WARPS * LW) {
#pragma unroll
            for (int it = 0; it < IT; it++) {
                const int idx = lane + 32 * it, l = idx / R0, j = idx - l * R0;
                if (l < LW) {
                    float2 v[8];
#pragma unroll
                    for (int r = 0; r < 8; r++) v[r] = src[(long long)(m0 + l) * N + j + R0 * r];
                    wi_first<R0>(v, E + l * I::EL, j);
                }
            }
            __syncwarp();
            float2 o[R0];
            wi_last<R0>(E + sl * I::EL, jj, twN, o);
#pragma unroll
            for (int r = 0; r < R0; r++) S[(m0 + sl) * SS + jj + 8 * r] = o[r];
            __syncwarp();
        }
        __syncthreads();
        unsigned long long best = 0ull;
        for (int q0 = warp * LW; q0 < N / 2; q0 += I::WARPS * LW) {
#pragma unroll
            for (int it = 0; it < IT; it++) {
                const int idx = lane + 32 * it, l = idx / R0, j = idx - l * R0;
                if (l < LW) {
                    float2 v[8];
#pragma unroll
                    for (int r = 0; r < 8; r++) {
                        const int k = r < 4 ? j + R0 * r : N - (j + R0 * r); // |m_z|; N/2 for j = 0, r = 4
                        float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (k < H) ab = *reinterpret_cast<const float4 *>(S + k * SS + 2 * (q0 + l));
                        if (r == 0 && j == 0) v[r] = make_float2(ab.x, ab.z);
                        else if (r < 4) v[r] = make_float2(ab.x - ab.w, ab.y + ab.z);
                        else v[r] = make_float2(ab.x + ab.w, ab.z - ab.y);
                    }
                    wi_first<R0>(v, E + l * I::EL, j);
                }
            }
            __syncwarp();
            float2 o[R0];
            wi_last<R0>(E + sl * I::EL, jj, twN, o);
            const int ky = 2 * (q0 + sl);
            if (keys) {
#pragma unroll
                for (int r = 0; r < R0; r++) {
                    const unsigned at = (unsigned)((kx * N + ky) * N + jj + 8 * r);
                    const unsigned long long k0 = peak_key(o[r].x, at), k1 = peak_key(o[r].y, at + N);
                    best = k0 > best ? k0 : best;
                    best = k1 > best ? k1 : best;
                }
            }
            __syncwarp(); // E is read: it takes the finished rows
            if (out) {
                float *f = reinterpret_cast<float *>(E);
#pragma unroll
                for (int r = 0; r < R0; r++) {
                    f[(2 * sl) * I::FS + jj + 8 * r] = o[r].x;
                    f[(2 * sl + 1) * I::FS + jj + 8 * r] = o[r].y;
                }
                __syncwarp();
                float4 *dst = reinterpret_cast<float4 *>(out + pr.out_off + ((long long)kx * N + 2 * q0) * N);
#pragma unroll
                for (int e0 = 0; e0 < 2 * LW * N / 4; e0 += 32) {
                    const int row = (e0 + lane) / (N / 4), at = (e0 + lane) % (N / 4);
                    const float4 x = *reinterpret_cast<const float4 *>(f + row * I::FS + 4 * at);
                    if (vec) {
                        dst[e0 + lane] = x;
                    } else { // a caller's grid on a 4-byte boundary only
                        float *d = reinterpret_cast<float *>(dst + e0 + lane);
                        d[0] = x.x, d[1] = x.y, d[2] = x.z, d[3] = x.w;
                    }
                }
                __syncwarp();
            }
        }
        if (keys) {
            for (int o2 = 16; o2 > 0; o2 >>= 1) {
                const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o2);
                best = other > best ? other : best;
            }
            if (lane == 0) red[warp] = best;
        }
        __syncthreads(); // S and the warps' maxima are complete
        if (keys && threadIdx.x == 0) {
            for (int k = 1; k < I::WARPS; k++) best = red[k] > best ? red[k] : best;
            atomicMax(keys + pr.key, best);
        }
    }
}

// ------------------------------------------------------------------ launchers
template <int NF, int LW>
static cudaError_t xw_t(const Geometry &g, const Tables &t, const InstDesc *inst, const InstPlan *plan,
                        const PairDesc *pairs, int npairs, const float2 *y1, const float2 *fa_cache, float2 *fa_out,
                        float2 *h, int cap, int *err, int nsm, cudaStream_t s)
{
    // where every item has an SM to itself, idle lanes cost nothing and the shorter steps
    // of two lines per warp shorten the pass (a pair at N = 32 22.6 us, with eight lines
    // 25.3).  Up to four items per SM (256 or 448
    // items) the fewer warps are the faster ones: a score at N = 64 with 5 rotations 69.9
    // us with two lines per warp, 67.7 with four; 7 rotations at N = 32 32.5 and 31.0;
    // only a single pair at N = 64 (256 items) gains from two: 38.7 against 39.2
    if constexpr (LW > 2)
        if ((long long)npairs * WF<NF>::H * (WF<NF>::N / XL) <= nsm)
            return xw_t<NF, 2>(g, t, inst, plan, pairs, npairs, y1, fa_cache, fa_out, h, cap, err, nsm, s);
    using X = XW<NF, LW>;
    const size_t smem = X::smem(cap);
    cudaError_t e = set_smem(k_xw<NF, LW>, X::smem(NF)); // cap <= NF
    if (e != cudaSuccess) return e;
    return launch_k(k_xw<NF, LW>, resident_blocks(k_xw<NF, LW>, smem, nsm, X::THREADS), X::THREADS, smem, s, g.pdl != 0, g,
                    t, inst, plan, pairs, npairs, y1, fa_cache, fa_out, h, err, cap);
}

cudaError_t launch_xw(const Geometry &g, const Tables &t, const InstDesc *inst, const InstPlan *plan,
                      const PairDesc *pairs, int npairs, const float2 *y1, const float2 *fa_cache, float2 *fa_out,
                      float2 *h, int cap, int *err, int nsm, cudaStream_t s)
{
    switch (g.n) {
    case 64: return xw_t<64, wf_full(64)>(g, t, inst, plan, pairs, npairs, y1, fa_cache, fa_out, h, cap, err, nsm, s);
    case 128: return xw_t<128, wf_full(128)>(g, t, inst, plan, pairs, npairs, y1, fa_cache, fa_out, h, cap, err, nsm, s);
    case 192: return xw_t<192, wf_full(192)>(g, t, inst, plan, pairs, npairs, y1, fa_cache, fa_out, h, cap, err, nsm, s);
    case 256: return xw_t<256, wf_full(256)>(g, t, inst, plan, pairs, npairs, y1, fa_cache, fa_out, h, cap, err, nsm, s);
    default: return cudaErrorInvalidValue;
    }
}

// One pair of empty shapes at N = 32 whose first warp gives up at its second phase:
// the kernel ends by itself and sets bit 8 of *err.
size_t xw_selftest_bytes() { return 1024 + sizeof(float2) * 32 * 32 * 16; }

cudaError_t launch_xw_selftest(void *zeroed, int *err, cudaStream_t s)
{
    constexpr int NF = 64, LW = 2;
    using X = XW<NF, LW>;
    char *p = (char *)zeroed; // two instances, plans and a pair, all zero; tables and output
    static_assert(2 * sizeof(InstDesc) + 2 * sizeof(InstPlan) + sizeof(PairDesc) <= 1024, "descriptors");
    const InstDesc *inst = (const InstDesc *)p;
    const InstPlan *plan = (const InstPlan *)(inst + 2);
    const PairDesc *pair = (const PairDesc *)(plan + 2);
    float2 *rest = (float2 *)(p + 1024);
    Geometry g{};
    g.N = 32, g.n = 64, g.H = 16, g.L = 2;
    Tables t{};
    t.tw_n = t.tw_N = rest;
    t.wl = (const float *)rest; // (N/2) (N/8) L 8 (N/2 + 1) floats: less than the output
    static_assert(sizeof(float) * 16 * 4 * 2 * 8 * 17 <= sizeof(float2) * 32 * 32 * 16, "level weights");
    const size_t smem = X::smem(0);
    cudaError_t e = set_smem(k_xw<NF, LW, true>, smem);
    if (e != cudaSuccess) return e;
    k_xw<NF, LW, true><<<2, X::THREADS, smem, s>>>(g, t, inst, plan, pair, 1, nullptr, nullptr, nullptr, rest, err, 0);
    return cudaGetLastError();
}

template <int NI>
static cudaError_t iyz_t(const Geometry &g, const Tables &t, const PairDesc *pairs, int npairs, const float2 *h,
                         float *out, unsigned long long *keys, int nsm, cudaStream_t s)
{
    const size_t smem = IYZ<NI>::smem;
    cudaError_t e = set_smem(k_iyz<NI>, smem);
    if (e != cudaSuccess) return e;
    const int blocks = std::min(resident_blocks(k_iyz<NI>, smem, nsm, IYZ<NI>::THREADS), npairs * NI);
    return launch_k(k_iyz<NI>, blocks, IYZ<NI>::THREADS, smem, s, g.pdl != 0, g, t, pairs, npairs, h, out, keys);
}

cudaError_t launch_iyz(const Geometry &g, const Tables &t, const PairDesc *pairs, int npairs, const float2 *h,
                       float *out, unsigned long long *keys, int nsm, cudaStream_t s)
{
    switch (g.N) {
    case 32: return iyz_t<32>(g, t, pairs, npairs, h, out, keys, nsm, s);
    case 64: return iyz_t<64>(g, t, pairs, npairs, h, out, keys, nsm, s);
    case 96: return iyz_t<96>(g, t, pairs, npairs, h, out, keys, nsm, s);
    case 128: return iyz_t<128>(g, t, pairs, npairs, h, out, keys, nsm, s);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace bc
