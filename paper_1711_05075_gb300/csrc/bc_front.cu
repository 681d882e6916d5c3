// Front half of a correlation pass for shapes that fit inside one period
// (front_fits): spreading into row-pair boxes, and the z and y transforms in one
// launch.  Boxes are stored as row pairs, [level][ix][iy / 2][iz][iy mod 2]: a
// pair is the complex z line the transform wants, contiguous along z.  The y and
// z extents are even (plan_instance).
#include <algorithm>

#include "bc_passes.cuh"
#include "bc_wfft.cuh"

namespace bc {

// ------------------------------------------------------------------ spread
// One warp per knot.  A lane owns one 16-byte piece of the stencil's (y, z)
// cross-section -- a row pair and two z cells -- for all W cells along x: it forms
// the piece's four products w_y w_z once, then per x cell multiplies by w_x, adds
// with one 16-byte vector atomic and steps to the next x plane.  A stencil of W
// cells reaches at most C = W / 2 + 1 row pairs and as many z pieces; where C^2
// <= 16 the two half-warps take alternate x cells, and for W = 10 (36 pieces) the
// lanes go round twice.  Weights outside the stencil are zero.
// Bound by the L2 reductions (52% of L2 throughput): 236 instructions a knot against
// 567 of k_spread took 40,000 knots of an N = 128 pair (W = 8) from 31.3 to 25.3 us.
// Gathering instead (bins of 8^3 cells, register sums) took 64 us and 16 for the bins.
constexpr int RP_WARPS = 8;

template <int W>
__global__ void __launch_bounds__(RP_WARPS * 32)
k_spread_rp(const float *__restrict__ consts, const InstDesc *__restrict__ inst, const float4 *__restrict__ ku,
            const InstPlan *__restrict__ plan, float *grid, int total)
{
    constexpr int C = W / 2 + 1, HALVES = C * C <= 16 ? 2 : 1;
    __shared__ float wts[RP_WARPS][3][W + 4]; // [axis][1 + offset], zero at both ends
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    constexpr float halfW = 0.5f * (float)W, xoff = 0.5f * (float)W - 1.f;
    const int wa = lane / W, wt = lane - wa * W;
    float kc[KB_NC];
    kb_load(consts, lane < 3 * W ? wt : 0, kc);
    for (int k = lane; k < 3 * (W + 4); k += 32) (&wts[wib][0][0])[k] = 0.f;
    const int sub = HALVES == 2 ? lane & 15 : lane, x0 = HALVES == 2 ? lane >> 4 : 0;
    pdl_signal();
    pdl_wait(); // earlier passes' outputs are read from here on
    __syncwarp();
    for (int k = blockIdx.x * RP_WARPS + wib; k < total; k += gridDim.x * RP_WARPS) {
        const float4 v = ku[k];
        const int tag = __float_as_int(v.w), level = tag & 15, i = tag >> 4;
        const InstPlan *p = plan + i;
        const int b0 = p->b[0], bz = p->b[2], np = p->b[1] >> 1;
        const int lx = p->lo[0], ly = p->lo[1], lz = p->lo[2];
        if (b0 == 0) continue;
        const int gx = (int)ceilf(v.x - halfW), gy = (int)ceilf(v.y - halfW), gz = (int)ceilf(v.z - halfW);
        if (lane < 3 * W) {
            const float u = wa == 0 ? v.x : wa == 1 ? v.y : v.z;
            const int gg = wa == 0 ? gx : wa == 1 ? gy : gz;
            wts[wib][wa][1 + wt] = kb_poly(kc, (u - (float)gg) - xoff);
        }
        __syncwarp();
        const int iy0 = gy - ly, iz0 = gz - lz, oy = iy0 & 1, oz = iz0 & 1; // iy0, iz0 >= 0
        const int xs = np * bz * 2; // floats of an x plane
        float *G = grid + inst[i].grid_off + (long long)(level * b0 + gx - lx + x0) * xs + (iy0 >> 1) * bz * 2 + (iz0 >> 1) * 4;
#pragma unroll
        for (int t0 = 0; t0 < C * C; t0 += 32) {
            const int t = t0 + sub, pr = t / C, zc = t - pr * C;
            // piece (pr, zc): rows 2 pr - oy, 2 pr - oy + 1 and cells 2 zc - oz, 2 zc - oz + 1 of the stencil
            if (t < C * C && 2 * pr - oy < W && 2 * zc - oz < W) {
                const float *wy = &wts[wib][1][1 + 2 * pr - oy], *wz = &wts[wib][2][1 + 2 * zc - oz];
                const float y0 = wy[0], y1 = wy[1], z0 = wz[0], z1 = wz[1];
                const float4 f = make_float4(y0 * z0, y1 * z0, y0 * z1, y1 * z1);
                float *cell = G + pr * bz * 2 + zc * 4;
#pragma unroll
                for (int dx = 0; dx < W; dx += HALVES) {
                    if (W % HALVES == 0 || dx + x0 < W) {
                        const float wx = wts[wib][0][1 + dx + x0];
                        atomicAdd(reinterpret_cast<float4 *>(cell), make_float4(wx * f.x, wx * f.y, wx * f.z, wx * f.w));
                    }
                    cell += HALVES * xs;
                }
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ z and y
// One block per (level, x) plane of a box; the z-transformed plane stays in
// shared memory (k_fft_z and k_fft_y write it to device memory and read it
// back).  Rows are placed at position 0 of their lines; the x pass puts the box
// origins of all three axes back with one phase per mode and instance, so an
// axis of b cells reaches only the first ceil(b / 16) inputs of each butterfly.
// A z line is a row pair (row 2q real, row 2q + 1 imaginary part); with Z its
// transform, the lane that holds Z_k, k = j + R0 r < N/2, gets Z_{n-k} from lane
// (R0 - j) mod R0 and stores
//     2 A_k = Z_k + conj Z_{n-k},   2 B_k = -i (Z_k - conj Z_{n-k})
// as one 16-byte value P[k][2q], P[k][2q + 1]; the x pass takes the factor 2 out.
// Output: y1 blocks [level][m_z][j_y / XL][ix][XL], the value of j_y at place
// xl_place(j_y, ix) of its row.
// Bound by instructions and the latency between them (issue 63%, 127 registers, two
// blocks per SM).  20,000 + 20,000 balls, N = 128: 46.9 us against 39.9 + 31.5 us of
// the tensor-core z pass and the staged y pass, whose rows crossed device memory
// twice; with block barriers in place of the warps' own tiles 85 us.  Two lines per warp
// in place of all it can take, for grids whose planes are all resident at once, gain
// nothing (128 + 128 balls at N = 32, two levels: a correlation 22.6 us either way) or
// cost (2,000 + 2,000, one level: 22.6 against 20.7).
constexpr int ZY_WARPS = 8;

template <int NF>
__global__ void __launch_bounds__(ZY_WARPS * 32, 2)
k_zy(Geometry g, Tables tb, const InstDesc *__restrict__ inst, int ninst, const InstPlan *__restrict__ plan,
     float *grid, float2 *y1, int PS, bool clear)
{
    using F = WF<NF>;
    constexpr int R0 = F::R0, H = F::H, N = F::N, LW = F::LW;
    extern __shared__ float4 sm4[];
    float2 *P = reinterpret_cast<float2 *>(sm4); // [H][PS]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2 *E = P + H * PS + warp * F::EW;
    const int s = lane / R0, j = lane - s * R0; // last stage: line and butterfly
    const int mate = s * R0 + (R0 - j) % R0;    // the lane that holds the modes n - k of this lane's k
    float2 w[16];
    wf_twiddles<NF>(tb.tw_n, lane, w);
    pdl_signal();
    pdl_wait(); // earlier passes' outputs are read from here on
    const int L = g.L;
    RotStart rs;
    for (int i = 0; i < ninst; i++) {
        const InstPlan p = plan[i];
        if (p.b[0] == 0) continue;
        const int b0 = p.b[0], b1 = p.b[1], bz = p.b[2], np = b1 >> 1;
        const int qz = (bz + 63) >> 6, qy = (b1 + 63) >> 6; // nonzero groups of four inputs
        const int planes = L * b0;
        const InstDesc d = inst[i];
        for (int it = rs.first(); it < planes; it += gridDim.x) {
            float2 *G2 = reinterpret_cast<float2 *>(grid + d.grid_off) + (long long)it * np * bz;
            for (int q0 = warp * LW; q0 < np; q0 += ZY_WARPS * LW) {
                wf_first_any<NF>(E, lane, qz, [&](int sl, int iz, bool inside) {
                    return (inside || iz < bz) && q0 + sl < np ? G2[(q0 + sl) * bz + iz] : make_float2(0.f, 0.f);
                });
                __syncwarp();
                float2 o[16], m[4];
                wf_last<NF>(E, lane, w, o);
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    m[r].x = __shfl_sync(0xffffffffu, o[15 - r].x, mate & 31);
                    m[r].y = __shfl_sync(0xffffffffu, o[15 - r].y, mate & 31);
                }
                if (j == 0) { // n - R0 r = R0 (16 - r)
                    m[0] = o[0];
                    m[1] = o[15];
                    m[2] = o[14];
                    m[3] = o[13];
                }
                const int q = q0 + s;
                if (lane < F::LIVE && q < np) {
#pragma unroll
                    for (int r = 0; r < 4; r++)
                        *reinterpret_cast<float4 *>(P + (j + R0 * r) * PS + 2 * q) =
                            make_float4(o[r].x + m[r].x, o[r].y - m[r].y, o[r].y + m[r].y, m[r].x - o[r].x);
                }
                __syncwarp();
            }
            __syncthreads();
            // the plane is read: clear it, if asked (one contiguous run; a store beside each load
            // of the same cell took 148 us instead of 47)
            float4 *G4 = reinterpret_cast<float4 *>(G2);
            for (int e = threadIdx.x; clear && e < np * bz / 2; e += ZY_WARPS * 32) G4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int l = it / b0, ix = it - l * b0;
            float2 *Y = y1 + d.y1_off + ((long long)l * H * (N / XL) * b0 + ix) * XL;
            for (int k0 = warp * LW; k0 < H; k0 += ZY_WARPS * LW) {
                wf_first_any<NF>(E, lane, qy, [&](int sl, int iy, bool inside) {
                    return inside || iy < b1 ? P[(k0 + sl) * PS + iy] : make_float2(0.f, 0.f);
                });
                __syncwarp();
                float2 o[16];
                wf_last<NF>(E, lane, w, o);
                if (lane < F::LIVE) {
                    float2 *Yk = Y + (long long)(k0 + s) * N * b0;
#pragma unroll
                    for (int r = 0; r < 16; r++) {
                        if (r >= 4 && r < 12) continue;
                        const int jy = r < 4 ? j + R0 * r : j + R0 * r - N;
                        Yk[(jy / XL) * b0 * XL + xl_place(jy, ix)] = jy == N / 2 ? make_float2(0.f, 0.f) : o[r];
                    }
                }
                __syncwarp();
            }
            __syncthreads(); // the plane is read: the next one may overwrite it
        }
        rs.rot += planes;
    }
}

// ------------------------------------------------------------------ launchers
bool supported_front(const Geometry &g)
{
    return g.prec == 0 && g.n == 2 * g.N && (g.N == 32 || g.N == 64 || g.N == 96 || g.N == 128);
}

// columns of k_zy's plane tile: at least the (even) rows of a plane, and twice an odd
// number (16-byte stores of neighbouring modes on different banks)
static int zy_ps(int cap)
{
    const int h = (cap + 2) / 2;
    return 2 * (h | 1);
}

template <int NF>
static size_t zy_smem(int cap)
{
    return sizeof(float2) * ((size_t)WF<NF>::H * zy_ps(cap) + (size_t)ZY_WARPS * WF<NF>::EW);
}

bool front_fits(const Geometry &g, int cap) { return supported_front(g) && cap + 2 <= g.n; }

template <int W>
static cudaError_t spread_rp_t(const Geometry &g, const Tables &t, const InstDesc *inst, int total_knots, const float4 *ku,
                               const InstPlan *plan, float *grid, cudaStream_t s)
{
    const int blocks = std::min((total_knots + RP_WARPS - 1) / RP_WARPS, 65535);
    return launch_k(k_spread_rp<W>, blocks, RP_WARPS * 32, 0, s, g.pdl != 0, t.consts, inst, ku, plan, grid, total_knots);
}

cudaError_t launch_spread_rp(const Geometry &g, const Tables &t, const InstDesc *inst, int total_knots, const float4 *ku,
                             const InstPlan *plan, float *grid, cudaStream_t s)
{
    if (total_knots <= 0) return cudaSuccess;
    switch (g.W) {
    case 2: return spread_rp_t<2>(g, t, inst, total_knots, ku, plan, grid, s);
    case 3: return spread_rp_t<3>(g, t, inst, total_knots, ku, plan, grid, s);
    case 4: return spread_rp_t<4>(g, t, inst, total_knots, ku, plan, grid, s);
    case 5: return spread_rp_t<5>(g, t, inst, total_knots, ku, plan, grid, s);
    case 6: return spread_rp_t<6>(g, t, inst, total_knots, ku, plan, grid, s);
    case 7: return spread_rp_t<7>(g, t, inst, total_knots, ku, plan, grid, s);
    case 8: return spread_rp_t<8>(g, t, inst, total_knots, ku, plan, grid, s);
    case 9: return spread_rp_t<9>(g, t, inst, total_knots, ku, plan, grid, s);
    case 10: return spread_rp_t<10>(g, t, inst, total_knots, ku, plan, grid, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int NF>
static cudaError_t zy_t(const Geometry &g, const Tables &t, const InstDesc *inst, int ninst, const InstPlan *plan,
                        float *grid, float2 *y1, int cap, int nsm, cudaStream_t s, bool clear)
{
    const size_t smem = zy_smem<NF>(cap);
    cudaError_t e = set_smem(k_zy<NF>, zy_smem<NF>(NF)); // cap <= NF
    if (e != cudaSuccess) return e;
    return launch_k(k_zy<NF>, resident_blocks(k_zy<NF>, smem, nsm, ZY_WARPS * 32), ZY_WARPS * 32, smem, s,
                    g.pdl != 0, g, t, inst, ninst, plan, grid, y1, zy_ps(cap), clear);
}

cudaError_t launch_zy(const Geometry &g, const Tables &t, const InstDesc *inst, int ninst, const InstPlan *plan,
                      float *grid, float2 *y1, int cap, int nsm, cudaStream_t s, bool clear)
{
    switch (g.n) {
    case 64: return zy_t<64>(g, t, inst, ninst, plan, grid, y1, cap, nsm, s, clear);
    case 128: return zy_t<128>(g, t, inst, ninst, plan, grid, y1, cap, nsm, s, clear);
    case 192: return zy_t<192>(g, t, inst, ninst, plan, grid, y1, cap, nsm, s, clear);
    case 256: return zy_t<256>(g, t, inst, ninst, plan, grid, y1, cap, nsm, s, clear);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace bc
