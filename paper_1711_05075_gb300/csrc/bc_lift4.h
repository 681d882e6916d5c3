// Lifted spectrum by a 4D type-1 NUFFT (bc_lift_nufft.cu), for the lifted
// correlation (bc_lift.cu).  Not part of the public interface.
#pragma once
#include <cstddef>
#include <string>
#include <cuda_runtime.h>

#include "bc_internal.h"

namespace bc {

// Bits of a lifted call's error word: what a bounded wait that expired was for.
enum {
    // the tensor-core contraction (bc_lift_umma.cuh)
    LIFT_ERR_COPY = 1,        // a free stage for the next copies
    LIFT_ERR_ACCUMULATOR = 2, // a free accumulator
    LIFT_ERR_STAGE = 4,       // a stage's copies
    LIFT_ERR_DRAIN = 8,       // a unit's products
    // the 4D NUFFT's line passes (bc_lift_line.cu)
    LIFT_ERR_LINE = 16        // their copies
};
inline std::string lift_stall_message(int word)
{
    const std::string incomplete = "; the spectrum is incomplete";
    if (word & LIFT_ERR_LINE) return "a pass of the 4D NUFFT stalled (a bounded wait for its copies expired)" + incomplete;
    return "tensor-core contraction stalled (waits " + std::to_string(word) + ": 1 copy, 2 accumulator, 4 stage, 8 drain)" + incomplete;
}

struct Lift4Rot {
    double R[9];
};

// Support box on the (2N)^3 x 2 N_r grid: per axis (x, y, z, r) the first cell lo and
// the extent b.
struct Lift4Box {
    int lo[4], b[4];
};

#ifdef __CUDACC__
// Fine-grid coordinate of knot c on axis a (0, 1, 2: rotated x, y, z; 3: r,
// mirrored for B), half a period on.  Every product and sum is spelled out: the box
// search and the spreading must get the same bits, or a knot on a cell's edge could lie
// one cell outside its box (left to the compiler, each kernel contracts them its own way).
__device__ __forceinline__ double lift4_coord(const float4 &c, int a, const double (&R)[9], int mirror, int ns, int nr,
                                              double inv_p, double inv_pr)
{
    double v;
    if (a < 3) v = __fma_rn(__fma_rn(R[3 * a + 2], c.z, __fma_rn(R[3 * a + 1], c.y, __dmul_rn(R[3 * a], c.x))), inv_p, 0.5);
    else v = __fma_rn(mirror ? -(double)c.w : (double)c.w, inv_pr, 0.5);
    return __dmul_rn(__dsub_rn(v, floor(v)), a < 3 ? ns : nr);
}
#endif

// Tables built by
// launch_build_tables for the spatial axes (N modes, n = 2N) and the lifted
// axis (N_r modes, n_r = 2 N_r), window width 8.
struct Lift4Tables {
    float *deconv_s = nullptr, *deconv_r = nullptr; // 1 / phi^ in FFT order: N, N_r entries
    float2 *tw_s = nullptr, *tw_r = nullptr;        // exp(-2 pi i k / n), k < n; the same for n_r
    float *consts = nullptr;                        // window polynomials (Tables::consts layout)
    // LIFT4_BOX_BYTES of device memory -- the two shapes' support boxes, 8 words each, then
    // their plans and descriptors for k_zy -- and the page-locked host copy
    int *dbox = nullptr;
    int *hbox = nullptr;
    float2 *wts = nullptr; // the line passes' mode weights, built by the first call that takes them (lift4_pair)
};
constexpr size_t LIFT4_BOX_BYTES = 1024;

size_t lift4_ws_bytes(int N, int Nr);
// h[s][j_x][j_y][m_z] (N^2 x N/2 complex per section, the collapse of the
// lifted correlation, as k_lift_collapse forms it from the two spectra) of the
// knots kA (unrotated) and kB (rotated by RB, row major, and mirrored in r),
// both spectra by the 4D NUFFT; cone = the cone transform table
// ((3 (N/2)^2 + 1) x N_r), slices = device sections, scale = P^-3 P_r^-1; ws of
// lift4_ws_bytes(N, Nr) bytes.  Synchronises s once (to size the support boxes).
// With *line set on return h is [s][k_x][m_z][j_y] instead, the inverse transform
// along x done (what launch_iyz takes); *err gets LIFT_ERR_LINE if a bounded wait expired.
// lift4_boxes first: it enqueues the search for the two shapes' support boxes.
cudaError_t lift4_boxes(const Lift4Tables &t, int N, int Nr, const float4 *kA, int nA, const float4 *kB, int nB,
                        const double (&RB)[9], double period, double period_r, int nsm, cudaStream_t s);
cudaError_t lift4_pair(Lift4Tables &t, int N, int Nr, const float4 *kA, int nA, const float4 *kB, int nB,
                       const double (&RB)[9], double period, double period_r, const float2 *cone, const float *slices,
                       int nslices, float scale, void *ws, float2 *h, bool *line, int *err, int nsm, cudaStream_t s);

// The passes for boxes narrower than the period on every axis (bc_lift_line.cu).
size_t lift4_weight_bytes(int N, int Nr);
cudaError_t lift4_build_weights(const Lift4Tables &t, int N, int Nr, const float2 *cone, cudaStream_t s);
bool lift4_line_fits(int N, int Nr, const Lift4Box &ba, const Lift4Box &bb, int nslices, int nsm);
inline size_t lift4_cells(const Lift4Box &b) { return (size_t)b.b[3] * b.b[0] * b.b[1] * b.b[2]; }
// x planes X1[m_z][j_y][i_r][j_x] of n knots; G: the box grid, whose first `clean` cells are
// zero (with none, the passes leave the box's cells zero behind them; else they don't); y1: scratch
cudaError_t lift4_line_spectrum(const Lift4Tables &t, int N, int Nr, const float4 *knots, int n, const Lift4Rot &rot,
                                int mirror, double ip, double ipr, const Lift4Box &bx, const InstPlan *dplan,
                                const InstDesc *dinst, float *G, size_t clean, float2 *y1, float2 *X1, int *err, int nsm, cudaStream_t s);
cudaError_t lift4_line_collapse(const Lift4Tables &t, int N, int Nr, const float2 *XA, const float2 *XB, const Lift4Box &ba,
                                const Lift4Box &bb, const float *slices, int nslices, double period_r, float scale, float2 *h,
                                int *err, int nsm, cudaStream_t s);

} // namespace bc
