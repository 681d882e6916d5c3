// Warp-synchronous 1D FFTs in two radix stages (FP32), for the passes that keep
// every line of a transform inside one warp (bc_front.cu, bc_line.cu,
// bc_lift_line.cu).
//
// Forward, length NF = R0 . 16 (64 = 4.16, 128 = 8.16, 192 = 12.16, 256 =
// 16.16): 16 first-stage butterflies of radix R0 on the inputs j + 16 r, then
// R0 butterflies of radix 16 on the elements j + R0 r, outputs j + R0 r.  The
// kept modes m in [-N/2, N/2), N = NF / 2, are exactly the outputs r < 4 and
// r >= 12.  Inverse, length N = 8 . R0: R0 first-stage butterflies of radix 8 on
// the inputs j + R0 r -- the modes a thread holds after the forward transform --
// then 8 butterflies of radix R0.  A warp transforms WF::LW lines at a time;
// lane -> (line, butterfly) is fixed per stage, so the last stage's twiddles
// are constants of the thread and stay in registers.
//
// Between the stages a line goes through a shared-memory exchange tile of the
// warp's own (rows = first-stage butterflies, padded to an odd number of complex
// values, so both the row-wise stores and the column-wise loads are free of bank
// conflicts); __syncwarp is the only barrier.
#pragma once
#include <utility>

#include "bc_device.cuh"

namespace bc {

constexpr int XL = 8; // lines (consecutive j_y of one m_z) of an x-pass item: 64-byte rows of y1

// place of line j_y (mod XL) in row ix of an item: a line read along ix out of
// shared memory, 64 bytes a row, falls on all banks
__device__ __forceinline__ int xl_place(int jy, int ix) { return (jy ^ (ix >> 1)) & (XL - 1); }

// lines of a warp whose last stage has a butterfly for every lane (24 of 32 at NF = 192)
constexpr int wf_full(int NF) { return NF == 192 ? 2 : 512 / NF; }

template <int NF, int LW_ = wf_full(NF)>
struct WF {
    static constexpr int R0 = NF / 16, Q = R0 / 4, N = NF / 2, H = NF / 4;
    static constexpr int LW = LW_;                      // lines of a warp (fewer: idle lanes, shorter steps)
    static constexpr int IT = LW * 16 / 32;             // first-stage butterflies per lane
    static constexpr int LIVE = LW * R0;                // lanes with a last-stage butterfly
    static constexpr int ES = 16 * (R0 + 1);            // exchange tile of a line (complex values)
    static constexpr int EW = LW * ES;                  // and of a warp
    static_assert(R0 == 4 || R0 == 8 || R0 == 12 || R0 == 16, "NF = 64, 128, 192 or 256");
    static_assert(LW >= 2 && LW <= wf_full(NF), "lines of a warp");
};

// x exp(-+2 pi i E / M) for the inner twiddles of the radix-8, -12 and -16 stages.
template <int M, int E, bool INV>
__device__ __forceinline__ float2 tw_in(float2 x)
{
    constexpr int e = E % M;
    if constexpr (M == 16) {
        return tw16_mul<e, INV>(x);
    } else if constexpr (e == 0) {
        return x;
    } else if constexpr (4 * e == M) {
        return mul_mi<INV>(x);
    } else if constexpr (2 * e == M) {
        return make_float2(-x.x, -x.y);
    } else if constexpr (M == 8) {
        constexpr float h = 0.70710678118654752440f;
        static_assert(e == 1 || e == 3, "radix-8 twiddle");
        if constexpr (e == 1)
            return INV ? make_float2(h * (x.x - x.y), h * (x.x + x.y)) : make_float2(h * (x.x + x.y), h * (x.y - x.x));
        else
            return INV ? make_float2(-h * (x.x + x.y), h * (x.x - x.y)) : make_float2(h * (x.y - x.x), -h * (x.x + x.y));
    } else {
        constexpr float s3 = 0.86602540378443864676f, sg = INV ? -1.f : 1.f;
        static_assert(M == 12 && (e == 1 || e == 2 || e == 4), "radix-12 twiddle");
        return e == 1 ? cmul(x, make_float2(s3, -0.5f * sg))
                      : e == 2 ? cmul(x, make_float2(0.5f, -s3 * sg)) : cmul(x, make_float2(-0.5f, -s3 * sg));
    }
}

// Q-point DFT of which only the first QN inputs are nonzero.
template <int Q, int QN, bool INV>
__device__ __forceinline__ void dft_head(float2 (&t)[Q])
{
    if constexpr (QN == 1) {
#pragma unroll
        for (int k = 1; k < Q; k++) t[k] = t[0];
    } else if constexpr (Q == 4 && QN == 2) {
        const float2 a = t[0], b = t[1], c = mul_mi<INV>(b);
        t[0] = cadd(a, b);
        t[1] = cadd(a, c);
        t[2] = csub(a, b);
        t[3] = csub(a, c);
    } else if constexpr (Q == 4 && QN == 3) {
        const float2 a0 = cadd(t[0], t[2]), a1 = csub(t[0], t[2]), b = t[1], c = mul_mi<INV>(b);
        t[0] = cadd(a0, b);
        t[1] = cadd(a1, c);
        t[2] = csub(a0, b);
        t[3] = csub(a1, c);
    } else if constexpr (Q == 3 && QN == 2) {
        constexpr float s = INV ? -0.86602540378443864676f : 0.86602540378443864676f;
        const float2 a = t[0], b = t[1];
        const float2 m = make_float2(fmaf(-0.5f, b.x, a.x), fmaf(-0.5f, b.y, a.y));
        t[0] = cadd(a, b);
        t[1] = make_float2(fmaf(s, b.y, m.x), fmaf(-s, b.x, m.y));
        t[2] = make_float2(fmaf(-s, b.y, m.x), fmaf(s, b.x, m.y));
    } else {
        dft_small<Q, INV>(t);
    }
}

template <int Q, int N2, bool INV, int... K1>
__device__ __forceinline__ void dft4q_tw(float2 (&t)[Q], std::integer_sequence<int, K1...>)
{
    ((t[K1] = tw_in<4 * Q, N2 * K1, INV>(t[K1])), ...);
}

template <int Q, int QN, int N2, bool INV>
__device__ __forceinline__ void dft4q_col(const float2 (&v)[4 * Q], float2 (&y)[4][Q])
{
    float2 t[Q];
#pragma unroll
    for (int n1 = 0; n1 < Q; n1++) t[n1] = n1 < QN ? v[4 * n1 + N2] : make_float2(0.f, 0.f);
    dft_head<Q, QN, INV>(t);
    if constexpr (N2 > 0 && Q > 1) dft4q_tw<Q, N2, INV>(t, std::make_integer_sequence<int, Q>{});
#pragma unroll
    for (int k1 = 0; k1 < Q; k1++) y[N2][k1] = t[k1];
}

// DFT of 4Q points whose inputs n >= 4 QN are zero (they are not read): n =
// 4 n1 + n2, k = k1 + Q k2; Q-point DFTs over n1, twiddles exp(-+2 pi i n2 k1 /
// 4Q), 4-point DFTs over n2.
template <int Q, int QN, bool INV>
__device__ __forceinline__ void dft4q(float2 (&v)[4 * Q])
{
    float2 y[4][Q];
    dft4q_col<Q, QN, 0, INV>(v, y);
    dft4q_col<Q, QN, 1, INV>(v, y);
    dft4q_col<Q, QN, 2, INV>(v, y);
    dft4q_col<Q, QN, 3, INV>(v, y);
#pragma unroll
    for (int k1 = 0; k1 < Q; k1++) {
        float2 t[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
        dft_small<4, INV>(t);
#pragma unroll
        for (int k2 = 0; k2 < 4; k2++) v[k1 + Q * k2] = t[k2];
    }
}

// Forward transform of the warp's LW lines.  src(s, pos, inside): input `pos` of
// line s, pos < 64 QN; `inside` (a constant): pos is below 64 (QN - 1) and so
// within the line's data, else src returns zero beyond them.  E: the warp's exchange tile (EW complex values); w:
// the lane's twiddles (wf_twiddles).  On return o[r], lanes < LIVE, is the
// output j + R0 r of line s, (s, j) = (lane / R0, lane % R0); only r < 4 and
// r >= 12 are meant to be used (the others are not computed).  The caller adds
// a __syncwarp before E is written again.
template <int NF, int QN, int LW, class Src>
__device__ __forceinline__ void wf_first(float2 *E, int lane, Src src)
{
    using F = WF<NF, LW>;
    constexpr int Q = F::Q, RN = QN * 4;
#pragma unroll
    for (int it = 0; it < F::IT; it++) {
        const int idx = lane + 32 * it, s = idx >> 4, j = idx & 15;
        float2 v[F::R0];
#pragma unroll
        for (int r = 0; r < RN; r++) v[r] = src(s, j + 16 * r, r < RN - 4);
        dft4q<Q, QN, false>(v);
        float2 *e = E + s * F::ES + j * (F::R0 + 1);
#pragma unroll
        for (int k = 0; k < F::R0; k++) e[k] = v[k];
    }
}

// qn: groups of 64 inputs that may be nonzero (uniform over the warp)
template <int NF, int LW = wf_full(NF), class Src>
__device__ __forceinline__ void wf_first_any(float2 *E, int lane, int qn, Src src)
{
    constexpr int Q = WF<NF>::Q;
    if (qn <= 1) wf_first<NF, 1, LW>(E, lane, src);
    else if (Q >= 2 && qn == 2) wf_first<NF, (Q >= 2 ? 2 : 1), LW>(E, lane, src);
    else if (Q >= 3 && qn == 3) wf_first<NF, (Q >= 3 ? 3 : 1), LW>(E, lane, src);
    else wf_first<NF, Q, LW>(E, lane, src);
}

// The lane's twiddles exp(-2 pi i r j / NF), j = lane mod R0, r = 1 .. 15: the first
// RW in registers, the others in a table of 16 per r, t[(r - RW - 1) 16 + j]
// (wf_twiddle_table), where registers are short.
template <int NF, int RW = 15, int LW = wf_full(NF)>
__device__ __forceinline__ void wf_last(const float2 *E, int lane, const float2 (&w)[RW + 1], float2 (&o)[16],
                                        const float2 *t = nullptr)
{
    using F = WF<NF, LW>;
    const int s = lane / F::R0, j = lane - s * F::R0;
    const float2 *e = E + (F::LIVE == 32 || lane < F::LIVE ? s : 0) * F::ES + j;
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const float2 x = e[r * (F::R0 + 1)];
        o[r] = r == 0 ? x : cmul(x, r <= RW ? w[r <= RW ? r : 0] : t[(r - RW - 1) * 16 + j]);
    }
    dft_small<16, false>(o);
}

template <int NF, int RW = 15>
__device__ __forceinline__ void wf_twiddles(const float2 *__restrict__ tw, int lane, float2 (&w)[RW + 1])
{
#pragma unroll
    for (int r = 1; r <= RW; r++) w[r] = tw[r * (lane % WF<NF>::R0)];
}

template <int NF, int RW>
__device__ __forceinline__ void wf_twiddle_table(const float2 *__restrict__ tw, float2 *t)
{
    for (int k = threadIdx.x; k < (15 - RW) * 16; k += blockDim.x) t[k] = tw[(k / 16 + RW + 1) * ((k % 16) % WF<NF>::R0)];
}

// Inverse transform, length N = 8 R0, first stage of one butterfly j < R0:
// inputs v[r] = element j + R0 r; its row of 8 goes to e (row stride 9).
constexpr int WI_ROW = 9;
template <int R0>
__device__ __forceinline__ void wi_first(float2 (&v)[8], float2 *line, int j)
{
    dft_small<8, true>(v);
    float2 *e = line + j * WI_ROW;
#pragma unroll
    for (int k = 0; k < 8; k++) e[k] = v[k];
}

// Last stage, butterfly jj < 8 of a line: o[r] = output jj + 8 r, r < R0.  twN:
// exp(-2 pi i k / N), k < N.
template <int R0>
__device__ __forceinline__ void wi_last(const float2 *line, int jj, const float2 *twN, float2 (&o)[R0])
{
#pragma unroll
    for (int r = 0; r < R0; r++) {
        const float2 x = line[r * WI_ROW + jj];
        o[r] = r == 0 ? x : cmulc(x, twN[r * jj]);
    }
    dft4q<R0 / 4, R0 / 4, true>(o);
}

} // namespace bc
