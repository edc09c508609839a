// The inverse transform of nt = N1 * N2 <= 1024 samples with its fused epilogues (I_wmax^H and F^H of
// Eq. 3 plus the terms of IrfftArgs), one register pass per factor:
//
//   pass A  thread (j, n2) reads the bins k = n1 N2 + n2 of the column pair j straight from the spectrum
//           (and the mirrored ones, conjugated; bins outside the band are zero and not read), N1-point
//           DFT over n1, twiddle, into the shared tile;
//   pass B  thread (j, k1) reads the tile's block k1, N2-point DFT: its registers then hold the samples
//           t = k1 + N1 k2 of the pair, which go through the epilogue to memory without another trip
//           through shared memory.  With FUSE the same registers (windowed) are also the first operand
//           of the forward transform of the output: X[k], k = k2 + N2 k1', is
//             sum_t1 W_N1^(t1 k1') [ W_NT^(t1 k2) sum_t2 W_N2^(t2 k2) x[t1 + N1 t2] ],
//           whose inner DFT over t2 runs at once in registers (t1 = k1); then the twiddle, one exchange
//           through the tile and N1-point DFTs over t1 leave bin k in row k, and the two columns of each
//           pair are separated and stored.
//
// What bounds it: the latency of the loads at 2-3 CTAs per SM (ncu at nt = 1024, plain: issue 45 %, long
// scoreboard stalls first, DRAM 42 %).  Against the form that staged the spectrum and the outputs in the
// tile (zero fill, three more barriers, a third more instructions): 8281 x 128 columns of 1024 samples,
// 40 bins, plain: 1.59 -> 1.44 ms; 1681 x 256 columns of 512 samples inside LSQR: 1.13 -> 1.07 ms on
// average; 441 columns of 256 samples inside LSQR: 18.2 -> 14.5 us (with the few-column tiles).
#pragma once

#include "fft_common.cuh"

namespace mdc {
namespace {

// MODE 1 (plain): the output is the transform alone; MODE 0: the general epilogue; MODE 2: the general
// epilogue with the LSQR x/w step of IrfftArgs.  V2: columns come in aligned pairs (8-byte accesses).
template <int N1, int N2, int MODE, int PP, bool FUSE, bool V2>
__global__ void __launch_bounds__(FFT_THREADS, MODE == 1 ? 3 : 2) irfft4_kernel(IrfftArgs a) {
    constexpr bool PLAIN = MODE == 1, XW = MODE == 2;
    static_assert(!(FUSE && PLAIN), "the fused forward transform follows the general epilogue");
    using F = FourStep<N1, N2, PP>;
    constexpr int NT = F::NT, CT = F::CT, P = F::P;
    extern __shared__ __align__(16) float2 sm2[];
    float2* tw = sm2;                  // exp(+2 pi i m / NT) for the whole period
    float2* z = sm2 + NT;
    double* red = reinterpret_cast<double*>(z + F::ZSIZE);
    const int c0 = blockIdx.x * CT;
    for (int i = threadIdx.x; i < NT / 2; i += FFT_THREADS) {
        const float2 w = a.tw[i];
        tw[i] = make_float2(w.x, -w.y);
        tw[i + NT / 2] = make_float2(-w.x, w.y);
    }
    pdl_wait();                                          // the spectrum; the twiddles above are constants
    if (a.active && *a.active == 0) return;
    // every thread keeps one column pair (FFT_THREADS is a multiple of P)
    const int j = threadIdx.x % P, c = c0 + 2 * j;
    const bool has0 = c < a.C, has1 = c + 1 < a.C;
    [[maybe_unused]] const long long ny = (long long)a.nf * a.S * a.ldv;
    {
        size_t oa = 0, ob = 0;
        if (has0) {
            const int sa = c / a.nv, va = c - sa * a.nv;
            oa = (size_t)sa * a.ldv + a.voff + va;
            if (has1) {
                const int sb = (c + 1) / a.nv, vb = c + 1 - sb * a.nv;
                ob = (size_t)sb * a.ldv + a.voff + vb;
            }
        }
        const size_t kstride = (size_t)a.S * a.ldv;
        // both columns as one 16-byte load when they are adjacent and every row keeps the alignment
        const bool pair16 = has1 && ob == oa + 1 && ((uintptr_t)(a.Y + oa) & 15) == 0 && (kstride & 1) == 0;
        const int kend = a.k0 + a.nf;
        const float isc = a.scale, sg = a.conj_in ? -1.f : 1.f;
        constexpr int BA0 = PLAIN ? 4 : 8, BA = BA0 < N1 / 2 ? BA0 : N1 / 2;     // bins in flight per thread
        constexpr int TASKS = (P * N2 + FFT_THREADS - 1) / FFT_THREADS;
#pragma unroll 1
        for (int it = 0; it < TASKS; ++it) {
            const int n2 = (threadIdx.x + it * FFT_THREADS) / P;
            const bool mine = n2 < N2;                   // (few columns: fewer tasks than threads)
            float2 r[N1];
#pragma unroll
            for (int b = 0; b < N1; b += BA) {
                // bin kk of k = n1 N2 + n2: k itself in the lower half, NT - k (mirrored) in the upper
                const bool mir = b >= N1 / 2;
                const int kmin = mir ? (N1 - b - BA) * N2 + 1 : b * N2;       // smallest bin of the batch
                if (kmin >= kend) {                      // uniform: nothing of the band in this batch
#pragma unroll
                    for (int u = 0; u < BA; ++u) r[b + u] = make_float2(0.f, 0.f);
                    continue;
                }
                float4 q[BA];
#pragma unroll
                for (int u = 0; u < BA; ++u) {
                    const int kk = mir ? (N1 - b - u) * N2 - n2 : (b + u) * N2 + n2;
                    q[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (has0 && mine && kk >= a.k0 && kk < kend) {
                        const size_t o = (size_t)(kk - a.k0) * kstride;
                        if (pair16) {
                            q[u] = *reinterpret_cast<const float4*>(MDC_AT(a.Y, oa + o, 2, ny, a.err, 20));
                        } else {
                            const float2 A = *MDC_AT(a.Y, oa + o, 1, ny, a.err, 21);
                            q[u].x = A.x;
                            q[u].y = A.y;
                            if (has1) {
                                const float2 B = *MDC_AT(a.Y, ob + o, 1, ny, a.err, 22);
                                q[u].z = B.x;
                                q[u].w = B.y;
                            }
                        }
                    }
                }
                const float s = mir ? -sg : sg;          // sign of the imaginary parts
#pragma unroll
                for (int u = 0; u < BA; ++u) {
                    // each value scaled, then joined (a solve's Green's functions show every rounding)
                    const float si = s * isc;
                    float ay = si * q[u].y, by = si * q[u].w;
                    if ((b + u == 0 || b + u == N1 / 2) && n2 == 0) ay = by = 0.f;     // DC, Nyquist
                    r[b + u] = make_float2(__fsub_rn(isc * q[u].x, by), __fadd_rn(ay, isc * q[u].z));
                }
            }
            reg_fft<N1, true>(r);
            if (it == 0) __syncthreads();                // the twiddles, whose loads ran meanwhile
            if (mine) {
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1)
                    z[F::zi(k1 * N2 + n2, j)] = k1 == 0 ? r[0] : cmul(r[k1], tw[n2 * k1]);
            }
        }
    }
    __syncthreads();

    [[maybe_unused]] const long long nx = (long long)NT * a.C;
    auto ld2 = [&](const float* p, size_t o, [[maybe_unused]] int site) {
        if constexpr (V2) return *reinterpret_cast<const float2*>(MDC_AT(p, o, 2, nx, a.err, site));
        else return make_float2(*MDC_AT(p, o, 1, nx, a.err, site), has1 ? *MDC_AT(p, o + 1, 1, nx, a.err, site) : 0.f);
    };
    auto st2 = [&](float* p, size_t o, float2 v, [[maybe_unused]] int site) {
        if constexpr (V2) {
            *reinterpret_cast<float2*>(MDC_AT(p, o, 2, nx, a.err, site)) = v;
        } else {
            *MDC_AT(p, o, 1, nx, a.err, site) = v.x;
            if (has1) *MDC_AT(p, o + 1, 1, nx, a.err, site) = v.y;
        }
    };
    float am = 1.f, ab = 0.f, ap = 0.f, xkx = 0.f, xkw = 0.f, xia = 0.f;
    bool has_prev = false, want_ss = false;
    int cut0 = 0x7fffffff, cut1 = cut0, fcut0 = cut0, fcut1 = cut0;
    if constexpr (!PLAIN) {
        am = coef(a.a_mdc);
        ab = coef(a.a_base);
        ap = coef(a.a_prev);
        has_prev = (a.a_prev.h != 0.f) || (a.a_prev.d != nullptr);
        want_ss = a.colsum != nullptr;
        if (a.cut && has0) cut0 = *MDC_AT(a.cut, c, 1, a.C, a.err, 25);
        if (a.cut && has1) cut1 = *MDC_AT(a.cut, c + 1, 1, a.C, a.err, 25);
        if (FUSE && a.fwd_cut && has0) fcut0 = *MDC_AT(a.fwd_cut, c, 1, a.C, a.err, 26);
        if (FUSE && a.fwd_cut && has1) fcut1 = *MDC_AT(a.fwd_cut, c + 1, 1, a.C, a.err, 26);
    }
    if constexpr (XW) {
        xkx = (float)*a.xw_kx;
        xkw = (float)*a.xw_kw;
        xia = (float)*a.xw_ia;
    }
    float ss[4] = {0.f, 0.f, 0.f, 0.f};   // sums of squares, columns c, c + 1 of even and of odd k2
    for (int task = threadIdx.x; task < P * N1; task += FFT_THREADS) {
        const int k1 = task / P;
        float2 r[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) r[n2] = z[F::zi(k1 * N2 + n2, j)];
        reg_fft<N2, true>(r);
        // r[k2] is the sample t = k1 + N1 k2 of the pair
        if (has0) {
            const size_t o0 = (size_t)k1 * a.C + c, ostep = (size_t)N1 * a.C;
            if constexpr (PLAIN) {
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) st2(a.out, o0 + k2 * ostep, r[k2], 23);
            } else {
                constexpr int E0 = XW ? 4 : 8, E = E0 < N2 ? E0 : N2;       // samples in flight per thread
#pragma unroll
                for (int b = 0; b < N2; b += E) {
                    float2 bv[E], pv[E], wv[XW ? E : 1], xv[XW ? E : 1];
                    size_t oo[E];
#pragma unroll
                    for (int u = 0; u < E; ++u) {
                        const size_t o = o0 + (b + u) * ostep;
                        oo[u] = o;
                        if (a.reverse_out) {
                            const int t = k1 + N1 * (b + u);
                            oo[u] = (size_t)((NT - t) & (NT - 1)) * a.C + c;
                        }
                        bv[u] = a.base ? ld2(a.base, o, 27) : make_float2(0.f, 0.f);
                        pv[u] = has_prev ? ld2(a.out, oo[u], 28) : make_float2(0.f, 0.f);
                        if constexpr (XW) {
                            wv[u] = ld2(a.xw_w, o, 29);
                            xv[u] = ld2(a.xw_x, o, 30);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < E; ++u) {
                        const int k2 = b + u, t = k1 + N1 * k2;
                        const int tau = k2 < N2 / 2 ? t : NT - t;            // t < NT / 2 iff k2 < N2 / 2
                        const float v0 = tau >= cut0 ? 0.f : r[k2].x, v1 = tau >= cut1 ? 0.f : r[k2].y;
                        const float2 v = make_float2(am * v0 + ab * bv[u].x + ap * pv[u].x,
                                                     am * v1 + ab * bv[u].y + ap * pv[u].y);
                        if (want_ss) {
                            ss[2 * (k2 & 1)] = fmaf(v.x, v.x, ss[2 * (k2 & 1)]);
                            ss[2 * (k2 & 1) + 1] = fmaf(v.y, v.y, ss[2 * (k2 & 1) + 1]);
                        }
                        st2(a.out, oo[u], v, 31);
                        if constexpr (XW) {
                            const size_t o = o0 + k2 * ostep;
                            st2(a.xw_x, o, make_float2(fmaf(xkx, wv[u].x, xv[u].x), fmaf(xkx, wv[u].y, xv[u].y)), 32);
                            st2(a.xw_w, o, make_float2(fmaf(xkw, wv[u].x, xia * pv[u].x),
                                                       fmaf(xkw, wv[u].y, xia * pv[u].y)), 33);
                        }
                        if constexpr (FUSE)
                            r[k2] = make_float2(tau >= fcut0 ? 0.f : v.x, tau >= fcut1 ? 0.f : v.y);
                    }
                }
            }
        }
        if constexpr (FUSE) {
            // (columns past the end hold the transform of zeros)
            reg_fft<N2, false>(r);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2)
                z[F::zi(k1 * N2 + k2, j)] = k2 == 0 ? r[0] : cmul(r[k2], cconj(tw[k1 * k2]));
        }
    }
    if constexpr (PLAIN) return;
    if (want_ss) {
        red[2 * threadIdx.x] = (double)ss[0] + (double)ss[2];
        red[2 * threadIdx.x + 1] = (double)ss[1] + (double)ss[3];
    }
    if (FUSE || want_ss) __syncthreads();
    if (want_ss && threadIdx.x < CT && c0 + (int)threadIdx.x < a.C) {
        double tot = 0.0;
        for (int i = threadIdx.x >> 1; i < FFT_THREADS; i += P) tot += red[2 * i + (threadIdx.x & 1)];
        *MDC_AT(a.colsum, c0 + threadIdx.x, 1, a.C, a.err, 34) = tot;
    }
    if constexpr (FUSE) {
        for (int task = threadIdx.x; task < P * N2; task += FFT_THREADS) {
            const int k2 = task / P;
            float2 r[N1];
#pragma unroll
            for (int t1 = 0; t1 < N1; ++t1) r[t1] = z[F::zi(t1 * N2 + k2, j)];
            reg_fft<N1, false>(r);
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) z[F::zi(k1 * N2 + k2, j)] = r[k1];
        }
        __syncthreads();
        // separate the two columns of each pair (scale 1/2, optional conjugation); bin k is in row k
        constexpr int G = FFT_THREADS / CT;
        const int cl = threadIdx.x % CT, g = threadIdx.x / CT, cc = c0 + cl;
        if (cc >= a.C) return;
        const int s = cc / a.nv, v = cc - s * a.nv;
        const size_t dsto = (size_t)s * a.ldv + a.fwd_voff + v;
        const size_t kstride = (size_t)a.S * a.ldv;
        const int jj = cl >> 1;
        const bool odd = (cl & 1) != 0;
        for (int kk = g; kk < a.nf; kk += G) {
            const int k = a.k0 + kk;
            const float2 Z = z[F::zi(k, jj)];
            const float2 Zm = k == 0 ? Z : z[F::zi(NT - k, jj)];
            float2 x = odd ? make_float2(0.5f * (Z.y + Zm.y), 0.5f * (Zm.x - Z.x))
                           : make_float2(0.5f * (Z.x + Zm.x), 0.5f * (Z.y - Zm.y));
            if (a.fwd_conj) x.y = -x.y;
            *MDC_AT(a.fwd_X, dsto + (size_t)kk * kstride, 1, ny, a.err, 18) = x;
        }
    }
}

template <int N1, int N2, int MODE, int PP, bool FUSE, bool V2>
void irfft4_go(mdc_plan* p, const IrfftArgs& a, cudaStream_t s) {
    using F = FourStep<N1, N2, PP>;
    constexpr size_t smem = F::smem_full + (MODE == 1 ? 0 : (size_t)FFT_THREADS * 2 * sizeof(double));
    static SmemLimit attr;
    attr.ensure(irfft4_kernel<N1, N2, MODE, PP, FUSE, V2>, (int)smem);
    LaunchScope ls(p, s, MDC_KC_IRFFT);
    launch_pdl(irfft4_kernel<N1, N2, MODE, PP, FUSE, V2>, dim3((a.C + F::CT - 1) / F::CT), FFT_THREADS, smem, s, a);
}

template <int N1, int N2, int PP, bool V2>
void irfft4_mode(mdc_plan* p, const IrfftArgs& a, bool fuse, cudaStream_t s) {
    if (irfft_plain(a)) irfft4_go<N1, N2, 1, PP, false, V2>(p, a, s);
    else if (a.xw_w && fuse) irfft4_go<N1, N2, 2, PP, true, V2>(p, a, s);
    else if (a.xw_w) irfft4_go<N1, N2, 2, PP, false, V2>(p, a, s);
    else if (fuse) irfft4_go<N1, N2, 0, PP, true, V2>(p, a, s);
    else irfft4_go<N1, N2, 0, PP, false, V2>(p, a, s);
}

}  // namespace

template <int N1, int N2>
bool irfft4_launch(mdc_plan* p, const IrfftArgs& a, cudaStream_t s) {
    auto even = [](const void* q) { return ((uintptr_t)q & 7) == 0; };
    const bool v2 = a.C % 2 == 0 && even(a.out) && even(a.base) && even(a.xw_w) && even(a.xw_x);
    constexpr int PS = few_cols_p<N1, N2>();
    const bool few = few_columns(a.C, FourStep<N1, N2>::CT) && PS < FourStep<N1, N2>::P;
    const bool fuse = a.fwd_X && !a.reverse_out;
    if (few) {
        if (v2) irfft4_mode<N1, N2, PS, true>(p, a, fuse, s);
        else irfft4_mode<N1, N2, PS, false>(p, a, fuse, s);
    } else {
        if (v2) irfft4_mode<N1, N2, 0, true>(p, a, fuse, s);
        else irfft4_mode<N1, N2, 0, false>(p, a, fuse, s);
    }
    return fuse;
}

}  // namespace mdc
