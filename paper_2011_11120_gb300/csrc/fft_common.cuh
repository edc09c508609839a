// Building blocks of the four-step register FFT kernels.  Each translation unit that includes this
// header gets its own copies (internal linkage).
#pragma once

#include "common.cuh"

namespace mdc {
namespace {

constexpr int FFT_THREADS = 256;

// ------------------------------------------------------------------ four-step kernels
// nt = N1 * N2 (N1, N2 in {8, 16, 32}).  Pass A: for each residue n2, an N1-point DFT in
// registers over t = n1 * N2 + n2, then the twiddle W_nt^(n2 k1); pass B: for each k1 an
// N2-point DFT over the N2 consecutive rows k1 * N2 + n2.  Result bin k = k1 + N1 * k2
// sits in row k1 * N2 + k2.  Four shared-memory sweeps per transform instead of
// 2 log2(nt) + 1 for radix 2.  Layout: row t of P complex sequences at t * P + (t / N2) * BP, BP
// chosen so that both passes spread a warp's 8-byte accesses over distinct bank pairs.

__host__ __device__ constexpr int brev_bits(int i, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
    return r;
}
__host__ __device__ constexpr int clog2(int n) { return n <= 1 ? 0 : 1 + clog2(n / 2); }

// Roots of unity as compile-time constants: cos and sin of 2*pi/R from the half-angle identities
// (cos(t/2) = sqrt((1 + cos t) / 2), sin(t/2) = sin t / (2 cos(t/2))) starting at t = pi/2, then
// powers by angle addition, all in double precision and rounded once to float.
struct Rot {
    double c, s;
};
constexpr double newton_sqrt(double x) {
    double r = x > 1.0 ? x : 1.0;
    for (int i = 0; i < 64; ++i) r = 0.5 * (r + x / r);
    return r;
}
constexpr Rot unit_root(int R, int m) {   // exp(+2 pi i m / R)
    Rot b{0.0, 1.0};
    if (R == 1) b = Rot{1.0, 0.0};
    if (R == 2) b = Rot{-1.0, 0.0};
    for (int r = 4; r < R; r *= 2) {
        const double c = newton_sqrt(0.5 * (1.0 + b.c));
        b = Rot{c, b.s / (2.0 * c)};
    }
    Rot w{1.0, 0.0};
    for (int i = 0; i < m; ++i) w = Rot{w.c * b.c - w.s * b.s, w.s * b.c + w.c * b.s};
    return w;
}

// exp(-2 pi i m / 32) for m < 16: every twiddle of the in-register DFTs (R <= 32) is one of
// these; as constant-bank operands they need no load.
#define MDC_ROOT32(m) float2{(float)unit_root(32, m).c, -(float)unit_root(32, m).s}
__constant__ float2 kRoot32[16] = {
    MDC_ROOT32(0),  MDC_ROOT32(1),  MDC_ROOT32(2),  MDC_ROOT32(3),  MDC_ROOT32(4),  MDC_ROOT32(5),
    MDC_ROOT32(6),  MDC_ROOT32(7),  MDC_ROOT32(8),  MDC_ROOT32(9),  MDC_ROOT32(10), MDC_ROOT32(11),
    MDC_ROOT32(12), MDC_ROOT32(13), MDC_ROOT32(14), MDC_ROOT32(15)};
#undef MDC_ROOT32

// Complex add and subtract as one packed two-lane float32 instruction (sm_100 and later);
// each lane rounds to nearest like the scalar operation.
__device__ __forceinline__ float2 padd(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 pa, pb, pr;\n\t"
        "mov.b64 pa, {%2, %3};\n\t"
        "mov.b64 pb, {%4, %5};\n\t"
        "add.rn.f32x2 pr, pa, pb;\n\t"
        "mov.b64 {%0, %1}, pr;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 psub(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 pa, pb, pr;\n\t"
        "mov.b64 pa, {%2, %3};\n\t"
        "mov.b64 pb, {%4, %5};\n\t"
        "sub.rn.f32x2 pr, pa, pb;\n\t"
        "mov.b64 {%0, %1}, pr;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// Length-R DFT (R <= 32) of a register array, forward sign exp(-2 pi i n k / R) or, with INV,
// the inverse sign (unscaled): decimation in frequency (natural order in, bit-reversed order
// out), then a compile-time permutation back to natural order.  After unrolling every index
// and twiddle choice is a constant: quarter turns are a swap, eighth turns take the
// equal-magnitude short form, the rest multiply by a table constant.
template <int R, bool INV>
__device__ __forceinline__ void reg_fft(float2 (&a)[R]) {
    static_assert(R <= 32, "register DFT length");
    constexpr int L = clog2(R);
    constexpr float h8 = (float)unit_root(8, 1).c;
#pragma unroll
    for (int st = 0; st < L; ++st) {
        const int h = R >> (st + 1);          // half span of this stage
#pragma unroll
        for (int g = 0; g < R; g += 2 * h) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const float2 u = a[g + j], v = a[g + j + h];
                a[g + j] = padd(u, v);
                float2 d = psub(u, v);
                const int m = j << st;       // twiddle exp(-+2 pi i m / R)
                if (m == 0) {
                } else if (4 * m == R) {
                    d = INV ? make_float2(-d.y, d.x) : make_float2(d.y, -d.x);
                } else if (8 * m == R) {
                    d = INV ? make_float2(h8 * (d.x - d.y), h8 * (d.x + d.y))
                            : make_float2(h8 * (d.x + d.y), h8 * (d.y - d.x));
                } else if (8 * m == 3 * R) {
                    d = INV ? make_float2(-h8 * (d.x + d.y), h8 * (d.x - d.y))
                            : make_float2(h8 * (d.y - d.x), -h8 * (d.x + d.y));
                } else {
                    const float2 w = kRoot32[m * (32 / R)];
                    d = cmul(d, INV ? cconj(w) : w);
                }
                a[g + j + h] = d;
            }
        }
    }
    float2 b[R];
#pragma unroll
    for (int i = 0; i < R; ++i) b[i] = a[brev_bits(i, L)];
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = b[i];
}

// PP: complex sequences per CTA, or 0 for the default of about 8192 complex values per tile (the
// few-column variant PP = max(1024 / NT, 2) spreads small batches over more CTAs).
template <int N1, int N2, int PP = 0> struct FourStep {
    static constexpr int NT = N1 * N2;
    static constexpr int P0 = 8192 / NT;
    static constexpr int P = PP ? PP : (P0 > 32 ? 32 : (P0 < 8 ? 8 : P0));   // complex sequences per CTA
    static constexpr int CT = 2 * P;                                  // real columns per CTA
    // Rows of P complex values, unpadded, plus BP slots after every block of N2 rows: with P < 16
    // consecutive rows (or blocks, in pass B) then fill all 16 bank pairs, and rows stay 16-byte
    // aligned for vector accesses.
    static constexpr int RS = P;
    static constexpr int BP = P < 16 ? P : 0;
    static constexpr int ZSIZE = NT * RS + N1 * BP;                  // float2 elements
    static constexpr size_t smem_full = (size_t)(NT + ZSIZE) * sizeof(float2);   // twiddles of a whole period, tile
    static_assert(ZSIZE * sizeof(float2) >= FFT_THREADS * 4 * sizeof(double), "reduction fits the tile");
    __device__ static __forceinline__ int zi(int t, int j) { return t * RS + (t / N2) * BP + j; }
};

// Second pass of the four-step transform: the length-N2 DFTs over n2 of every block k1, in
// place; ends with a barrier.
template <int N1, int N2, bool INV, int PP = 0>
__device__ __forceinline__ void four_step_pass_b(float2* z) {
    using F = FourStep<N1, N2, PP>;
    constexpr int P = F::P;
    for (int task = threadIdx.x; task < P * N1; task += FFT_THREADS) {
        const int j = task % P, k1 = task / P;
        float2 r[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) r[n2] = z[F::zi(k1 * N2 + n2, j)];
        reg_fft<N2, INV>(r);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) z[F::zi(k1 * N2 + k2, j)] = r[k2];
    }
    __syncthreads();
}

// tw: the twiddle table W_NT^m of the transform's sign (conjugated for INV) for the whole period m < NT.
template <int N1, int N2, bool INV, int PP = 0>
__device__ __forceinline__ void four_step(float2* z, const float2* tw) {
    using F = FourStep<N1, N2, PP>;
    constexpr int P = F::P;
    for (int task = threadIdx.x; task < P * N2; task += FFT_THREADS) {
        const int j = task % P, n2 = task / P;
        float2 r[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) r[n1] = z[F::zi(n1 * N2 + n2, j)];
        reg_fft<N1, INV>(r);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) {
            const float2 v = k1 == 0 ? r[0] : cmul(r[k1], tw[n2 * k1]);
            z[F::zi(k1 * N2 + n2, j)] = v;
        }
    }
    __syncthreads();
    four_step_pass_b<N1, N2, INV, PP>(z);
}

// Row holding bin (or time sample) q after four_step.
template <int N1, int N2>
__device__ __forceinline__ int out_row(int q) { return (q % N1) * N2 + q / N1; }

// Few columns: the default tile would leave most SMs idle (fewer CTAs than half the SMs); smaller
// tiles then shorten each CTA's work.  (With one or more default CTAs per SM the smaller tiles only
// add waves: measured slower at 3721 columns of 1024 samples.)
template <int N1, int N2>
constexpr int few_cols_p() { return 1024 / (N1 * N2) > 2 ? 1024 / (N1 * N2) : 2; }
inline bool few_columns(int C, int ct) { return (C + ct - 1) / ct < 148 / 2; }

// The transform alone: no window, base or previous-output terms, column sums or reversal.
inline bool irfft_plain(const IrfftArgs& a) {
    return !a.cut && !a.base && !a.colsum && !a.reverse_out && a.a_mdc.h == 1.f && !a.a_mdc.d &&
           a.a_prev.h == 0.f && !a.a_prev.d && !a.xw_w && !a.fwd_X;
}

}  // namespace

// The inverse transform of nt = N1 * N2 <= 1024 samples (fft_inv.cuh; instantiated per size).  Returns
// true if the kernel also made the forward transform of IrfftArgs::fwd_X.
template <int N1, int N2>
bool irfft4_launch(mdc_plan* p, const IrfftArgs& a, cudaStream_t s);

}  // namespace mdc
