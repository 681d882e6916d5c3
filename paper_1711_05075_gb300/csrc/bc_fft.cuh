// Batched one-dimensional FFTs in shared memory (FP32), used by every
// transform pass of the correlation.
//
// Algorithm: the self-sorting Stockham formulation of the Cooley-Tukey FFT
// (T. G. Stockham, 1966; as arranged for GPUs by Govindaraju et al.,
// "High performance discrete Fourier transforms on graphics processors",
// SC 2008).  A length-NF transform runs as a sequence of radix-R stages; with
// Ns the product of the radices already applied, butterfly j of a stage reads
// x[j + r NF/R] (r < R), multiplies input r by w^(r (j mod Ns) NF/(Ns R)),
// applies an R-point DFT and writes y[(j div Ns) Ns R + (j mod Ns) + r Ns].
// Output is in natural order after the last stage; stages ping-pong between
// two shared-memory tiles.  Radix schedules: 32 = 4.8, 64 = 8.8,
// 96 = 3.4.8, 128 = 8.16, 192 = 3.8.8, 256 = 16.16, 512 = 8.8.8.
//
// Direction: forward uses exp(-2 pi i jk/NF), inverse exp(+2 pi i jk/NF); no
// scaling.  The twiddle table holds exp(-2 pi i k/NF), k < NF, rounded once
// from FP64; the inverse conjugates it.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

namespace bc {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }

// multiply by -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 mul_mi(float2 a)
{
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// x * exp(-+2 pi i E / 16) for the exponents a radix-16 butterfly uses
// (E = n2 k1, n2, k1 < 4).  E = 0 and 4 are exact (identity, -+i); E = 2 and 6
// take two adds and two multiplies by sqrt(1/2); the rest a complex multiply.
template <int E, bool INV>
__device__ __forceinline__ float2 tw16_mul(float2 x)
{
    const float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f, h = 0.70710678118654752440f;
    const float sg = INV ? -1.f : 1.f; // imaginary part of the twiddle flips for the inverse
    if constexpr (E == 0) {
        return x;
    } else if constexpr (E == 4) {
        return mul_mi<INV>(x);
    } else if constexpr (E == 2) { // (1 -+ i) h
        return INV ? make_float2(h * (x.x - x.y), h * (x.x + x.y)) : make_float2(h * (x.x + x.y), h * (x.y - x.x));
    } else if constexpr (E == 6) { // (-1 -+ i) h
        return INV ? make_float2(-h * (x.x + x.y), h * (x.x - x.y)) : make_float2(h * (x.y - x.x), -h * (x.x + x.y));
    } else if constexpr (E == 1) {
        return cmul(x, make_float2(c1, -sg * s1));
    } else if constexpr (E == 3) {
        return cmul(x, make_float2(s1, -sg * c1));
    } else {
        static_assert(E == 9, "radix-16 twiddle exponent");
        return cmul(x, make_float2(-c1, sg * s1));
    }
}

template <int N2, int K1, bool INV>
__device__ __forceinline__ float2 tw16_apply(float2 x) { return tw16_mul<N2 * K1, INV>(x); }

template <int R, bool INV>
__device__ __forceinline__ void dft_small(float2 *v)
{
    if constexpr (R == 2) {
        float2 t = v[0];
        v[0] = cadd(t, v[1]);
        v[1] = csub(t, v[1]);
    } else if constexpr (R == 3) {
        // exp(-+2 pi i/3) = -1/2 -+ i sqrt(3)/2
        const float s = INV ? 0.86602540378443864676f : -0.86602540378443864676f;
        float2 t1 = cadd(v[1], v[2]);
        float2 t2 = csub(v[1], v[2]);
        float2 m = make_float2(fmaf(-0.5f, t1.x, v[0].x), fmaf(-0.5f, t1.y, v[0].y));
        float2 r = make_float2(-s * t2.y, s * t2.x); // i s t2
        v[0] = cadd(v[0], t1);
        v[1] = cadd(m, r);
        v[2] = csub(m, r);
    } else if constexpr (R == 4) {
        float2 a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
        float2 b0 = cadd(v[1], v[3]), b1 = mul_mi<INV>(csub(v[1], v[3]));
        v[0] = cadd(a0, b0);
        v[2] = csub(a0, b0);
        v[1] = cadd(a1, b1);
        v[3] = csub(a1, b1);
    } else if constexpr (R == 16) {
        // 16 = 4 x 4: index n = 4 n1 + n2, k = k1 + 4 k2; 4-point DFTs over n1,
        // twiddles exp(-+2 pi i n2 k1 / 16), then 4-point DFTs over n2.
        float2 y[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; n2++) {
            float2 t[4] = {v[n2], v[4 + n2], v[8 + n2], v[12 + n2]};
            dft_small<4, INV>(t);
#pragma unroll
            for (int k1 = 0; k1 < 4; k1++) y[n2][k1] = t[k1];
        }
        y[1][1] = tw16_apply<1, 1, INV>(y[1][1]);
        y[1][2] = tw16_apply<1, 2, INV>(y[1][2]);
        y[1][3] = tw16_apply<1, 3, INV>(y[1][3]);
        y[2][1] = tw16_apply<2, 1, INV>(y[2][1]);
        y[2][2] = tw16_apply<2, 2, INV>(y[2][2]);
        y[2][3] = tw16_apply<2, 3, INV>(y[2][3]);
        y[3][1] = tw16_apply<3, 1, INV>(y[3][1]);
        y[3][2] = tw16_apply<3, 2, INV>(y[3][2]);
        y[3][3] = tw16_apply<3, 3, INV>(y[3][3]);
#pragma unroll
        for (int k1 = 0; k1 < 4; k1++) {
            float2 t[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
            dft_small<4, INV>(t);
#pragma unroll
            for (int k2 = 0; k2 < 4; k2++) v[k1 + 4 * k2] = t[k2];
        }
    } else if constexpr (R == 8) {
        const float h = 0.70710678118654752440f;
        float2 a[4], b[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            a[k] = cadd(v[k], v[k + 4]);
            b[k] = csub(v[k], v[k + 4]);
        }
        // b[k] *= exp(-+2 pi i k / 8)
        b[1] = INV ? make_float2(h * (b[1].x - b[1].y), h * (b[1].x + b[1].y))
                   : make_float2(h * (b[1].x + b[1].y), h * (b[1].y - b[1].x));
        b[2] = mul_mi<INV>(b[2]);
        b[3] = INV ? make_float2(-h * (b[3].x + b[3].y), h * (b[3].x - b[3].y))
                   : make_float2(h * (b[3].y - b[3].x), -h * (b[3].x + b[3].y));
        dft_small<4, INV>(a);
        dft_small<4, INV>(b);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            v[2 * k] = a[k];
            v[2 * k + 1] = b[k];
        }
    }
}

// Radix schedules: S = 0 the default of each size, S = 1 an alternative for
// the forward passes (chosen by measurement; every last stage has a radix
// divisible by 4, which the pruned x pass needs).
template <int NF, int S = 0>
struct Radix;
template <> struct Radix<32, 0>  { static constexpr int r0 = 4, r1 = 8, r2 = 1; };
template <> struct Radix<64, 0>  { static constexpr int r0 = 8, r1 = 8, r2 = 1; };
template <> struct Radix<96, 0>  { static constexpr int r0 = 3, r1 = 4, r2 = 8; };
template <> struct Radix<128, 0> { static constexpr int r0 = 8, r1 = 16, r2 = 1; };
template <> struct Radix<192, 0> { static constexpr int r0 = 3, r1 = 8, r2 = 8; };
template <> struct Radix<256, 0> { static constexpr int r0 = 16, r1 = 16, r2 = 1; };
template <> struct Radix<512, 0> { static constexpr int r0 = 8, r1 = 8, r2 = 8; };
template <> struct Radix<64, 1>  { static constexpr int r0 = 4, r1 = 16, r2 = 1; };
template <> struct Radix<128, 1> { static constexpr int r0 = 16, r1 = 8, r2 = 1; };
template <> struct Radix<192, 1> { static constexpr int r0 = 3, r1 = 4, r2 = 16; };
template <> struct Radix<256, 1> { static constexpr int r0 = 4, r1 = 8, r2 = 8; };
template <> struct Radix<512, 1> { static constexpr int r0 = 8, r1 = 4, r2 = 16; };

// Schedule of the split-precision passes: the default of each length, except
// 256, whose default (16.16) has no radix-8 stage for the tensor cores.
template <int NF>
struct SplitSched {
    static constexpr int S = NF == 256 ? 1 : 0;
};

// Column order of a tile row.  Natural: value c of row pos at column c.  Swz: at
// column c ^ f(pos), f from the row's place in the strides of the tensor-core
// stage that reads the tile (A, 0: none) and of the one that writes it (B, 0:
// none).  Those stages touch 4 rows A (B) apart with the lanes of one access, 8
// (read) and 4 (written) columns of each, and whole rows are a multiple of the
// 32 banks: unswizzled, the 4 rows fall on the same banks (a split correlation
// at N = 128, L = 4, 20,000 + 20,000 balls: 579 us, swizzled 527).
struct Natural {
    static __device__ __forceinline__ int at(int, int c) { return c; }
};
template <int A, int B>
struct Swz {
    static __device__ __forceinline__ int at(int pos, int c)
    {
        if constexpr (A > 0) c ^= ((pos / A) & 3) << 2;
        if constexpr (B > 0) {
            const int x = pos / B;
            c ^= (x & 1) | ((x & 2) << 2);
        }
        return c;
    }
};

// ---------------------------------------------------------------------------
// Interleaved tiles: C lines stored as x[pos * C + c].  Consecutive threads take
// consecutive lines c of the same butterfly, so every shared-memory access of
// a stage is a run of C consecutive complex values (no bank conflicts), and a
// tile row of C values is one 8C-byte run in global memory as well.
template <int NF, int R, int NS, bool INV, int C, int NT, class In = Natural, class Out = Natural>
__device__ __forceinline__ void il_stage(const float2 *__restrict__ in, float2 *__restrict__ out,
                                         const float2 *__restrict__ tw)
{
    constexpr int NB = NF / R;
    constexpr int TOT = NB * C;
    constexpr int IT = (TOT + NT - 1) / NT;
#pragma unroll
    for (int it = 0; it < IT; it++) {
        const int idx = (int)threadIdx.x + it * NT;
        if ((TOT % NT) != 0 && idx >= TOT) break;
        const int c = idx % C, j = idx / C;
        const int k = j % NS;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) {
            float2 x = in[(j + r * NB) * C + In::at(j + r * NB, c)];
            if (NS > 1 && r > 0) {
                float2 w = tw[r * k * (NF / (NS * R))];
                if (INV) w.y = -w.y;
                x = cmul(x, w);
            }
            v[r] = x;
        }
        dft_small<R, INV>(v);
        const int base = (j / NS) * NS * R + k;
#pragma unroll
        for (int r = 0; r < R; r++) out[(base + r * NS) * C + Out::at(base + r * NS, c)] = v[r];
    }
}

// Transforms the C interleaved lines of tile `a` (b: scratch tile); all NT
// threads of the block must call it.  Returns the tile holding the result;
// ends with a block barrier.
template <int NF, bool INV, int C, int NT>
__device__ __forceinline__ float2 *il_fft(float2 *a, float2 *b, const float2 *tw)
{
    using RR = Radix<NF>;
    il_stage<NF, RR::r0, 1, INV, C, NT>(a, b, tw);
    __syncthreads();
    il_stage<NF, RR::r1, RR::r0, INV, C, NT>(b, a, tw);
    __syncthreads();
    if constexpr (RR::r2 > 1) {
        il_stage<NF, RR::r2, RR::r0 * RR::r1, INV, C, NT>(a, b, tw);
        __syncthreads();
        return b;
    } else {
        return a;
    }
}

// ---------------------------------------------------------------------------
// Register-resident first and last stages.  A transform of C interleaved lines
// runs as: first stage (inputs held in registers, loaded straight from global
// memory by the caller) -> shared tile -> middle stage (only for three-stage
// schedules, shared -> shared) -> last stage (shared -> registers -> a sink
// functor).  Shared memory then carries each value once per exchange instead
// of once per stage plus a gather and a scatter.

// Inputs of the first stage owned by the calling thread: butterfly (c, j) of
// iteration `it` needs positions j + r NF/R, r < R.
template <int NF, int R, int C, int NT>
struct FirstInputs {
    static constexpr int NB = NF / R, TOT = NB * C, IT = (TOT + NT - 1) / NT;
    float2 v[IT][R];
    // src(c, pos) -> float2: value of line c at position pos (issue the loads only).
    template <class Src>
    __device__ __forceinline__ void load(Src src)
    {
#pragma unroll
        for (int it = 0; it < IT; it++) {
            const int idx = (int)threadIdx.x + it * NT;
            const int c = idx % C, j = idx / C;
#pragma unroll
            for (int r = 0; r < R; r++)
                v[it][r] = ((TOT % NT) == 0 || idx < TOT) ? src(c, j + r * NB) : make_float2(0.f, 0.f);
        }
    }
    // Writes the loaded values to their positions of a tile in column order `Out`.
    template <class Out = Natural>
    __device__ __forceinline__ void scatter(float2 *tile) const
    {
#pragma unroll
        for (int it = 0; it < IT; it++) {
            const int idx = (int)threadIdx.x + it * NT;
            if ((TOT % NT) != 0 && idx >= TOT) break;
            const int c = idx % C, j = idx / C;
#pragma unroll
            for (int r = 0; r < R; r++) tile[(j + r * NB) * C + Out::at(j + r * NB, c)] = v[it][r];
        }
    }
    // visit(c, pos) for every position load() read.
    template <class Vis>
    __device__ __forceinline__ void for_each(Vis visit) const
    {
#pragma unroll
        for (int it = 0; it < IT; it++) {
            const int idx = (int)threadIdx.x + it * NT;
            if ((TOT % NT) != 0 && idx >= TOT) break;
            const int c = idx % C, j = idx / C;
#pragma unroll
            for (int r = 0; r < R; r++) visit(c, j + r * NB);
        }
    }
};

// First stage (Ns = 1, no twiddles): registers -> out, column order `Out`.
template <int NF, int R, bool INV, int C, int NT, class Out = Natural>
__device__ __forceinline__ void rr_first(const FirstInputs<NF, R, C, NT> &in, float2 *__restrict__ out)
{
    using FI = FirstInputs<NF, R, C, NT>;
#pragma unroll
    for (int it = 0; it < FI::IT; it++) {
        const int idx = (int)threadIdx.x + it * NT;
        if ((FI::TOT % NT) != 0 && idx >= FI::TOT) break;
        const int c = idx % C, j = idx / C;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = in.v[it][r];
        dft_small<R, INV>(v);
#pragma unroll
        for (int r = 0; r < R; r++) out[(j * R + r) * C + Out::at(j * R + r, c)] = v[r];
    }
}

// Last stage: in[pos * C + c] -> registers -> sink(it, r, c, pos, value), where
// the output position is pos = j + r NS for butterfly j (< NS) of iteration it.
template <int NF, int R, int NS, bool INV, int C, int NT, class Sink>
__device__ __forceinline__ void rr_last(const float2 *__restrict__ in, const float2 *__restrict__ tw, Sink sink)
{
    constexpr int NB = NF / R;
    static_assert(NB == NS, "last stage");
    constexpr int TOT = NB * C;
    constexpr int IT = (TOT + NT - 1) / NT;
#pragma unroll
    for (int it = 0; it < IT; it++) {
        const int idx = (int)threadIdx.x + it * NT;
        if ((TOT % NT) != 0 && idx >= TOT) break;
        const int c = idx % C, j = idx / C;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) {
            float2 x = in[(j + r * NB) * C + c];
            if (r > 0) {
                float2 w = tw[r * j * (NF / (NS * R))];
                if (INV) w.y = -w.y;
                x = cmul(x, w);
            }
            v[r] = x;
        }
        dft_small<R, INV>(v);
#pragma unroll
        for (int r = 0; r < R; r++) sink(it, r, c, j + r * NS, v[r]);
    }
}

// Radix of the last stage of a schedule and its output stride.
template <int NF, int S = 0>
struct LastStage {
    static constexpr int R = Radix<NF, S>::r2 > 1 ? Radix<NF, S>::r2 : Radix<NF, S>::r1;
    static constexpr int NS = NF / R;
};

// Outputs of the last stage that a pass keeps: modes [-NF/4, NF/4), the first and
// last quarter of r.  Known when compiled, so the others are not computed.
template <int NF, int S>
__device__ __forceinline__ constexpr bool kept_out(int r)
{
    static_assert(LastStage<NF, S>::R % 4 == 0, "last stage");
    return r < LastStage<NF, S>::R / 4 || r >= LastStage<NF, S>::R / 4 * 3;
}

// The middle (three-stage schedules) and last stages after rr_first has
// written tile s0; s1 is scratch for three-stage schedules.  All threads call
// it; the caller adds a barrier before s0/s1 are written again.
template <int NF, bool INV, int C, int NT, int S = 0, class Sink>
__device__ __forceinline__ void rr_rest(float2 *s0, float2 *s1, const float2 *tw, Sink sink)
{
    using R = Radix<NF, S>;
    if constexpr (R::r2 > 1) {
        il_stage<NF, R::r1, R::r0, INV, C, NT>(s0, s1, tw);
        __syncthreads();
        rr_last<NF, R::r2, R::r0 * R::r1, INV, C, NT>(s1, tw, sink);
    } else {
        rr_last<NF, R::r1, R::r0, INV, C, NT>(s0, tw, sink);
    }
}

// ---------------------------------------------------------------------------
// Split-precision radix-8 stage on the tensor cores.  The 8-point DFT of a
// butterfly is y = F x with F[r'][r] = exp(-+2 pi i r r' / 8); with complex
// numbers as (re, im) pairs it is a 16 x 16 real matrix acting on a 16-vector,
// so one mma.m16n8k16 (A = F, B = the inputs of 8 butterflies, one per column)
// transforms 8 butterflies.  Both F and the twiddled inputs are split into
// BF16 hi + lo parts (hi = bf16(v), lo = bf16(v - hi)); the product is formed
// as F_hi x_hi + F_hi x_lo + F_lo x_hi with FP32 accumulation (the lo x lo term,
// of relative size 2^-18 at most, is dropped).  Lane (g, t) of a warp loads inputs
// r = t and r = t + 4 of butterfly g of the group (the B fragment layout) and
// receives output components g and g + 8 of butterflies 2t and 2t + 1.
//
// Bound by issued instructions, so the stage spends few beside the products: F is
// built from one entry, each complex value is split with two conversions, no lane
// branches, two groups are in flight, a FP32 first stage runs on the registers
// that hold its inputs, and the z pass unpacks straight from the result tile.
// Split correlation at N = 128, L = 4, 20,000 + 20,000 balls: 527 us -> 273.
//
// The lane's words of F as a pair (hi, lo), of which the entry (r', r) = (g / 2,
// t) is computed: 4 more on r' or on r turns the angle by pi times t or r', so the
// other three words are that one with its signs flipped or not.
template <bool INV>
__device__ __forceinline__ void dft8_words(int g, int t, unsigned (&hi)[4], unsigned (&lo)[4])
{
    // rows p = 0: (cos, sin), p = 1: (-sin, cos) of e pi / 4 (sin negated for the inverse)
    const int e = ((g >> 1) * t) & 7;
    const bool odd = e & 1;
    const unsigned H = odd ? 0x3f35u : 0x3f80u, L = odd ? 0x389eu : 0u; // sqrt(1/2) or 1 as bf16 hi, lo
    const bool c0 = (e & 3) == 2, s0 = (e & 3) == 0;             // the entries that are zero
    const unsigned cn = (e + 2) & 4 ? 0x8000u : 0u, sn = ((e & 4) != 0) != INV ? 0x8000u : 0u;
    const unsigned ch = c0 ? 0u : H ^ cn, cl = c0 || !L ? 0u : L ^ cn;
    const unsigned sh = s0 ? 0u : H ^ sn, sl = s0 || !L ? 0u : L ^ sn;
    const bool p = g & 1;
    const unsigned h = p ? (sh ^ 0x8000u) | ch << 16 : ch | sh << 16;
    const unsigned l = p ? (sl ^ 0x8000u) | cl << 16 : cl | sl << 16;
    const unsigned mt = t & 1 ? 0x80008000u : 0u, mr = g & 2 ? 0x80008000u : 0u;
    hi[0] = h, hi[1] = h ^ mt, hi[2] = h ^ mr, hi[3] = h ^ mt ^ mr;
    lo[0] = l, lo[1] = l ^ mt, lo[2] = l ^ mr, lo[3] = l ^ mt ^ mr;
}

// (v.x, v.y) as packed bf16 hi and lo parts, x in the lower half
__device__ __forceinline__ void split_bf16x2(float2 v, unsigned &hi, unsigned &lo)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
    hi = *reinterpret_cast<const unsigned *>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(v.x - __uint_as_float(hi << 16), v.y - __uint_as_float(hi & 0xffff0000u));
    lo = *reinterpret_cast<const unsigned *>(&l);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int NF, int NS, bool INV, int C, int NT, int U, class In, class Out>
__device__ __forceinline__ void tc_stage8(const float2 *__restrict__ in, float2 *__restrict__ out,
                                          const float2 *__restrict__ tw)
{
    constexpr int R = 8, NB = NF / R, TOT = NB * C, GROUPS = TOT / 8;
    static_assert(C == 16 && (NT / 32) % 2 == 0 && GROUPS % (NT / 32) == 0, "a group: half a row of butterflies; a warp keeps its half");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3, c0 = (warp & 1) * 8;
    unsigned ahi[4], alo[4];
    dft8_words<INV>(g, t, ahi, alo);
    float *outf = reinterpret_cast<float *>(out);
#pragma unroll U
    for (int i = 0; i < GROUPS / (NT / 32); i++) {
        const int grp = warp + i * (NT / 32);
        // inputs r = t and r = t + 4 of butterfly (j, c)
        const int c = c0 + g, j = grp >> 1, k = j % NS;
        float2 x0 = in[(j + t * NB) * C + In::at(j + t * NB, c)];
        float2 x1 = in[(j + (t + 4) * NB) * C + In::at(j + (t + 4) * NB, c)];
        if (NS > 1) { // (no branch for t = 0: its twiddle is 1)
            float2 w0 = tw[t * k * (NF / (NS * R))], w1 = tw[(t + 4) * k * (NF / (NS * R))];
            if (INV) w0.y = -w0.y, w1.y = -w1.y;
            x0 = cmul(x0, w0);
            x1 = cmul(x1, w1);
        }
        unsigned bh0, bl0, bh1, bl1;
        split_bf16x2(x0, bh0, bl0);
        split_bf16x2(x1, bh1, bl1);
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(d, ahi, bh0, bh1);
        mma_bf16(d, ahi, bl0, bl1);
        mma_bf16(d, alo, bh0, bh1);
        // d[0] = C[g][2t], d[1] = C[g][2t+1], d[2] = C[g+8][2t], d[3] = C[g+8][2t+1]
        const int p = g & 1, lo = (j / NS) * NS * R + k + (g >> 1) * NS, hi = lo + 4 * NS;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int cc = c0 + 2 * t + u;
            outf[(lo * C + Out::at(lo, cc)) * 2 + p] = d[u];
            outf[(hi * C + Out::at(hi, cc)) * 2 + p] = d[2 + u];
        }
    }
}

// A stage of the split-precision schedule: tensor-core DFT for radix 8, FP32 otherwise.
template <int NF, int R, int NS, bool INV, int C, int NT, int U, class In, class Out>
__device__ __forceinline__ void sp_stage(const float2 *in, float2 *out, const float2 *tw)
{
    if constexpr (R == 8) tc_stage8<NF, NS, INV, C, NT, U, In, Out>(in, out, tw);
    else il_stage<NF, R, NS, INV, C, NT, In, Out>(in, out, tw);
}

// Column orders of the tiles of a split-precision transform: its input, after
// the first, the second and the last stage.
template <int NF, int S>
struct SplitTiles {
    using R = Radix<NF, S>;
    static constexpr int NB = NF / 8;
    using Input = Swz<R::r0 == 8 ? NB : 0, 0>;
    using T1 = Swz<R::r1 == 8 ? NB : 0, R::r0 == 8 ? 1 : 0>;
    using T2 = Swz<R::r2 == 8 ? NB : 0, R::r1 == 8 ? R::r0 : 0>;
    using T3 = Swz<0, R::r2 == 8 ? R::r0 * R::r1 : 0>;
    using Result = std::conditional_t<(R::r2 > 1), T3, T2>;
};

// Groups that a warp has in flight in a tensor-core stage: all eight at 256 points,
// where their addresses and twiddles become constants of the loop (a split
// correlation at N = 128: 283 us with two, 273 with all in the z and y passes);
// elsewhere, and in the x pass, all of them spill.
__host__ __device__ constexpr int split_unroll(int NF) { return NF == 256 ? 8 : 2; }

// Split-precision transform of C interleaved lines whose inputs, in registers,
// sp_first has left in s1 as the outputs of an FP32 first stage (radix 3 or 4),
// or in s0 for a tensor-core one (radix 8).  sp_stages: the stages; returns the
// tile that holds the result, column order SplitTiles::Result, once the caller
// has added a barrier.  sp_all: the same, then
// sink(it, r, c, pos, value) in the thread mapping of rr_last for radix
// schedule S.  All threads call them; the caller adds a barrier after sp_first
// and before s0/s1 are written again.
template <int NF, int C, int NT, int S>
__device__ __forceinline__ void sp_first(const FirstInputs<NF, Radix<NF, S>::r0, C, NT> &in, float2 *s0, float2 *s1)
{
    using ST = SplitTiles<NF, S>;
    if constexpr (Radix<NF, S>::r0 == 8) in.template scatter<typename ST::Input>(s0);
    else rr_first<NF, Radix<NF, S>::r0, false, C, NT, typename ST::T1>(in, s1);
}

template <int NF, bool INV, int C, int NT, int S, int U = split_unroll(NF)>
__device__ __forceinline__ float2 *sp_stages(float2 *s0, float2 *s1, const float2 *tw)
{
    using R = Radix<NF, S>;
    using ST = SplitTiles<NF, S>;
    if constexpr (R::r0 == 8) {
        sp_stage<NF, R::r0, 1, INV, C, NT, U, typename ST::Input, typename ST::T1>(s0, s1, tw);
        __syncthreads();
    }
    sp_stage<NF, R::r1, R::r0, INV, C, NT, U, typename ST::T1, typename ST::T2>(s1, s0, tw);
    if constexpr (R::r2 > 1) {
        __syncthreads();
        sp_stage<NF, R::r2, R::r0 * R::r1, INV, C, NT, U, typename ST::T2, typename ST::T3>(s0, s1, tw);
        return s1;
    }
    return s0;
}

template <int NF, bool INV, int C, int NT, int S, int U = split_unroll(NF), class Sink>
__device__ __forceinline__ void sp_all(float2 *s0, float2 *s1, const float2 *tw, Sink sink)
{
    using Fin = typename SplitTiles<NF, S>::Result;
    const float2 *fin = sp_stages<NF, INV, C, NT, S, U>(s0, s1, tw);
    __syncthreads();
    constexpr int RL = LastStage<NF, S>::R, NSL = LastStage<NF, S>::NS, TOT = NSL * C, IT = (TOT + NT - 1) / NT;
#pragma unroll
    for (int it = 0; it < IT; it++) {
        const int idx = (int)threadIdx.x + it * NT;
        if ((TOT % NT) != 0 && idx >= TOT) break;
        const int c = idx % C, j = idx / C;
#pragma unroll
        for (int r = 0; r < RL; r++) sink(it, r, c, j + r * NSL, fin[(j + r * NSL) * C + Fin::at(j + r * NSL, c)]);
    }
}

} // namespace bc
