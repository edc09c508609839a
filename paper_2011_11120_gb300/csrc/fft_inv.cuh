// The inverse transform of nt = N1 * N2 <= 1024 samples with its fused epilogues (I_wmax^H and F^H of
// Eq. 3 plus the terms of IrfftArgs), one register pass per factor:
//
//   pass A  thread (j, n2) reads the bins k = n1 N2 + n2 of the column pair j straight from the spectrum
//           (and the mirrored ones, conjugated; bins outside the band are zero and not read), N1-point
//           DFT over n1, twiddle, into the shared tile;
//   pass B  thread (j, k1) reads the tile's block k1, N2-point DFT.  Plain transforms store their samples
//           t = k1 + N1 k2 from the registers.  The others leave them in the tile, and the epilogue walks
//           its rows, VEC columns per thread.  With FUSE the windowed outputs in the tile are then
//           transformed forward: X[k], k = k2 + N2 k1', is
//             sum_t1 W_N1^(t1 k1') [ W_NT^(t1 k2) sum_t2 W_N2^(t2 k2) x[t1 + N1 t2] ]
//           (or with the N1-point DFTs first, see STD below), and the two columns of each pair are
//           separated and stored.
//
// What bounds it: the latency of the loads at 2-3 CTAs per SM.  Against the form that staged the spectrum in
// the tile too (zero fill, one more barrier): 8281 x 128 columns of 1024 samples, 40 bins, plain: 1.59 ->
// 1.44 ms; inside LSQR, on average over a solve: 441 columns of 256 samples 18.0 -> 11.1 us (with the few-column
// tiles), 1681 x 32 columns of 512 samples, 100 bins: 145 -> 142 us, 1681 x 31 (with the forward transform,
// which was a launch of its own for columns not in fours): 211 -> 168 us; 3721 / 841 x 20 columns of 1024
// samples in a deconvolution 204 -> 203 us.
#pragma once

#include "fft_common.cuh"

namespace mdc {
namespace {

// MODE 1 (plain): the output is the transform alone; MODE 0: the general epilogue; MODE 2: the general
// epilogue with the LSQR x/w step of IrfftArgs.  VEC: columns come one by one, in aligned pairs (8-byte
// accesses) or in aligned fours (also accessed by pairs; never with time reversal).
//
// Rounding.  The order of every float32 operation depends on the length and on VEC alone, not on the tile or
// the mode (joins, sums and the epilogue are written out as fused multiply-adds), so that a solve gives the same bits
// whatever launches it is made of: a Green's function g- = R f+ - f- that is a small difference of large fields
// shows each change.  Fours take the sums in other groups and another order than pairs and single columns.
//
// CTAs per SM: three, with fewer registers, where the tile allows it (not with 1024 samples and the forward
// transform's sums, 80 KB); the x/w step needs the registers.
constexpr int irfft4_ctas(int nt, int mode, bool fuse) { return mode == 2 || (fuse && nt == 1024) ? 2 : 3; }
template <int N1, int N2, int MODE, int PP, bool FUSE, int VEC>
__global__ void __launch_bounds__(FFT_THREADS, irfft4_ctas(N1 * N2, MODE, FUSE)) irfft4_kernel(IrfftArgs a) {
    constexpr bool PLAIN = MODE == 1, XW = MODE == 2;
    static_assert(!(FUSE && PLAIN), "the fused forward transform follows the general epilogue");
    using F = FourStep<N1, N2, PP>;
    constexpr int NT = F::NT, CT = F::CT, P = F::P;
    extern __shared__ __align__(16) float2 sm2[];
    float2* tw = sm2;                  // exp(+2 pi i m / NT) for the whole period
    float2* z = sm2 + NT;
    float* red = reinterpret_cast<float*>(z + F::ZSIZE);       // chains of the sums of squares
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
        constexpr int BA0 = irfft4_ctas(NT, MODE, FUSE) == 2 ? 8 : 4, BA = BA0 < N1 / 2 ? BA0 : N1 / 2;     // bins in flight per thread
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
                    const float si = s * isc;
                    float ay = si * q[u].y, by = si * q[u].w;
                    if ((b + u == 0 || b + u == N1 / 2) && n2 == 0) ay = by = 0.f;     // DC, Nyquist
                    r[b + u] = make_float2(fmaf(isc, q[u].x, -by), fmaf(isc, q[u].z, ay));
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
    if constexpr (PLAIN) {
        // Columns that are not in aligned pairs: stored from the registers, each pair is two stores of every
        // other word of a row.  From nt = 512 on they go out through the tile, a column per thread
        // (8281 x 255 columns, registers against tile: nt = 1024 4.45 and 3.89 ms, 512 1.64 and 1.52, 256 0.69 and
        // 0.72, 64 0.225 and 0.240).
        constexpr bool ROWS = VEC == 1 && NT >= 512;
        for (int task = threadIdx.x; task < P * N1; task += FFT_THREADS) {
            const int k1 = task / P;
            float2 r[N2];
#pragma unroll
            for (int n2 = 0; n2 < N2; ++n2) r[n2] = z[F::zi(k1 * N2 + n2, j)];
            reg_fft<N2, true>(r);
            if constexpr (ROWS) {
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) z[F::zi(k1 * N2 + k2, j)] = r[k2];
                continue;
            }
            if (!has0) continue;
            // r[k2] is the sample t = k1 + N1 k2 of the pair
            const size_t o0 = (size_t)k1 * a.C + c, ostep = (size_t)N1 * a.C;
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                const size_t o = o0 + k2 * ostep;
                if constexpr (VEC > 1) {
                    *reinterpret_cast<float2*>(MDC_AT(a.out, o, 2, nx, a.err, 23)) = r[k2];
                } else {
                    *MDC_AT(a.out, o, 1, nx, a.err, 23) = r[k2].x;
                    if (has1) *MDC_AT(a.out, o + 1, 1, nx, a.err, 24) = r[k2].y;
                }
            }
        }
        if constexpr (ROWS) {
            __syncthreads();
            const int cl = threadIdx.x % CT;
            if (c0 + cl < a.C) {
#pragma unroll 8
                for (int rho = threadIdx.x / CT; rho < NT; rho += FFT_THREADS / CT) {
                    const int t = (rho % N2) * N1 + rho / N2;
                    *MDC_AT(a.out, (size_t)t * a.C + c0 + cl, 1, nx, a.err, 24) =
                        reinterpret_cast<const float*>(z + F::zi(rho, 0))[cl];
                }
            }
        }
        return;
    }
    four_step_pass_b<N1, N2, true, PP>(z);

    // Row rho of the tile holds the sample t = (rho mod N2) N1 + rho / N2.  A thread takes VEC columns of
    // the rows t0, t0 + TS, ...; outputs go back into the tile where they are needed again.
    constexpr int Q = CT / VEC, TS = FFT_THREADS / Q, PER = NT / TS, B0 = VEC == 4 ? (XW ? 2 : 4) : 8, B = B0 < PER ? B0 : PER;
    // Sums of squares: the rows of one column with equal rho mod CHAINS are added up in float32 in ascending
    // order, then the chains in double.  That is what a thread of the default tile has; smaller
    // tiles keep the chains and take them from the tile.
    constexpr int CHAINS = VEC * (FFT_THREADS / FourStep<N1, N2>::CT);
    static_assert(PP != 0 || CHAINS == TS, "one chain per thread and column");
    const float am = coef(a.a_mdc), ab = coef(a.a_base), ap = coef(a.a_prev);
    const bool has_prev = (a.a_prev.h != 0.f) || (a.a_prev.d != nullptr), want_ss = a.colsum != nullptr;
    const bool keep = FUSE || (PP != 0 && want_ss);
    float xkx = 0.f, xkw = 0.f, xia = 0.f;
    if constexpr (XW) {
        xkx = (float)*a.xw_kx;
        xkw = (float)*a.xw_kw;
        xia = (float)*a.xw_ia;
    }
    struct __align__(4 * VEC) Vec { float v[VEC]; };
    auto ld = [&](const float* p, size_t o, [[maybe_unused]] int site) {
        return *reinterpret_cast<const Vec*>(MDC_AT(p, o, VEC, nx, a.err, site));
    };
    auto st = [&](float* p, size_t o, const Vec& v, [[maybe_unused]] int site) {
        *reinterpret_cast<Vec*>(MDC_AT(p, o, VEC, nx, a.err, site)) = v;
    };
    const int cl = VEC * (threadIdx.x % Q), t0 = threadIdx.x / Q, cq = c0 + cl;
    Vec ss{};
    if (cq < a.C) {
        int cut[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) cut[i] = a.cut ? *MDC_AT(a.cut, cq + i, 1, a.C, a.err, 25) : 0x7fffffff;
#pragma unroll 1
        for (int b0 = 0; b0 < PER; b0 += B) {
            Vec bv[B], pv[B], wv[XW ? B : 1], xv[XW ? B : 1];
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int rho = t0 + (b0 + u) * TS, t = (rho % N2) * N1 + rho / N2;
                const size_t o = (size_t)t * a.C + cq, oo = VEC != 4 && a.reverse_out ? (size_t)((NT - t) & (NT - 1)) * a.C + cq : o;
                bv[u] = a.base ? ld(a.base, o, 27) : Vec{};
                pv[u] = has_prev ? ld(a.out, oo, 28) : Vec{};
                if constexpr (XW) {
                    wv[u] = ld(a.xw_w, o, 29);
                    xv[u] = ld(a.xw_x, o, 30);
                }
            }
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int rho = t0 + (b0 + u) * TS, t = (rho % N2) * N1 + rho / N2, tau = t < NT / 2 ? t : NT - t;
                const size_t o = (size_t)t * a.C + cq, oo = VEC != 4 && a.reverse_out ? (size_t)((NT - t) & (NT - 1)) * a.C + cq : o;
                Vec* slot = reinterpret_cast<Vec*>(reinterpret_cast<float*>(z + F::zi(rho, 0)) + cl);
                Vec v = *slot;
#pragma unroll
                for (int i = 0; i < VEC; ++i) {
                    const float y = tau >= cut[i] ? 0.f : v.v[i];
                    v.v[i] = VEC == 4 ? fmaf(ap, pv[u].v[i], fmaf(am, y, __fmul_rn(ab, bv[u].v[i])))
                                      : fmaf(ap, pv[u].v[i], fmaf(ab, bv[u].v[i], __fmul_rn(am, y)));
                    if (PP == 0) ss.v[i] = fmaf(v.v[i], v.v[i], ss.v[i]);
                }
                st(a.out, oo, v, 31);
                if (keep) *slot = v;
                if constexpr (XW) {
                    Vec nx1, nw1;
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        nx1.v[i] = fmaf(xkx, wv[u].v[i], xv[u].v[i]);
                        nw1.v[i] = fmaf(xkw, wv[u].v[i], xia * pv[u].v[i]);
                    }
                    st(a.xw_x, o, nx1, 32);
                    st(a.xw_w, o, nw1, 33);
                }
            }
        }
    } else if (FUSE && VEC == 1 && cq == a.C && (cl & 1)) {
        // the column past an odd number of columns: its slots hold rounding errors of its partner's transform
        for (int m = 0; m < PER; ++m) reinterpret_cast<float*>(z + F::zi(t0 + m * TS, 0))[cl] = 0.f;
    }
    if (PP == 0 && want_ss) *reinterpret_cast<Vec*>(red + VEC * threadIdx.x) = ss;
    if (FUSE || want_ss) __syncthreads();
    if (PP != 0 && want_ss) {
        for (int idx = threadIdx.x; idx < P * CHAINS; idx += FFT_THREADS) {
            float2 sum = make_float2(0.f, 0.f);          // both columns of pair idx % P
#pragma unroll 16
            for (int m = 0; m < NT / CHAINS; ++m) {
                const float2 v = z[F::zi(idx / P + m * CHAINS, idx % P)];
                sum = make_float2(fmaf(v.x, v.x, sum.x), fmaf(v.y, v.y, sum.y));
            }
            reinterpret_cast<float2*>(red)[idx] = sum;
        }
        __syncthreads();
    }
    if (want_ss && threadIdx.x < CT && c0 + (int)threadIdx.x < a.C) {
        double tot = 0.0;
        for (int i = threadIdx.x; i < CT * CHAINS; i += CT) tot += (double)red[i];
        *MDC_AT(a.colsum, c0 + threadIdx.x, 1, a.C, a.err, 34) = tot;
    }
    if constexpr (FUSE) {
        const int fcut0 = a.fwd_cut && has0 ? *MDC_AT(a.fwd_cut, c, 1, a.C, a.err, 26) : 0x7fffffff;
        const int fcut1 = a.fwd_cut && has1 ? *MDC_AT(a.fwd_cut, c + 1, 1, a.C, a.err, 26) : 0x7fffffff;
        // Columns in aligned fours: the order of the head of this file, bin k in row k.  Others: N1-point
        // DFTs first, as the forward kernel does (the same operations where N1 = N2), bin k in row out_row(k).
        constexpr bool STD = N1 != N2 && VEC != 4;
        if constexpr (STD) {
            static_assert(P * N2 <= FFT_THREADS, "one task per thread");
            const int n2 = threadIdx.x / P;
            float2 r[N1];
            if (n2 < N2) {
#pragma unroll
                for (int n1 = 0; n1 < N1; ++n1) {
                    const int t = n1 * N2 + n2, tau = n1 < N1 / 2 ? t : NT - t;
                    const float2 v = z[F::zi(out_row<N1, N2>(t), j)];
                    r[n1] = make_float2(tau >= fcut0 ? 0.f : v.x, tau >= fcut1 ? 0.f : v.y);
                }
            }
            __syncthreads();                             // the tile has been read
            if (n2 < N2) {
                reg_fft<N1, false>(r);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1)
                    z[F::zi(k1 * N2 + n2, j)] = k1 == 0 ? r[0] : cmul(r[k1], cconj(tw[n2 * k1]));
            }
            __syncthreads();
            four_step_pass_b<N1, N2, false, PP>(z);
        } else {
            for (int task = threadIdx.x; task < P * N1; task += FFT_THREADS) {
                const int k1 = task / P;
                float2 r[N2];
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) {
                    const int t = k1 + N1 * k2, tau = k2 < N2 / 2 ? t : NT - t;
                    const float2 v = z[F::zi(k1 * N2 + k2, j)];
                    r[k2] = make_float2(tau >= fcut0 ? 0.f : v.x, tau >= fcut1 ? 0.f : v.y);
                }
                reg_fft<N2, false>(r);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2)
                    z[F::zi(k1 * N2 + k2, j)] = k2 == 0 ? r[0] : cmul(r[k2], cconj(tw[k1 * k2]));
            }
            __syncthreads();
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
        }
        auto row = [&](int q) { return STD ? out_row<N1, N2>(q) : q; };
        // separate the two columns of each pair (scale 1/2, optional conjugation)
        constexpr int G = FFT_THREADS / CT;
        const int cf = threadIdx.x % CT, g = threadIdx.x / CT, cc = c0 + cf;
        if (cc >= a.C) return;
        const int s = cc / a.nv, v = cc - s * a.nv;
        const size_t dsto = (size_t)s * a.ldv + a.fwd_voff + v;
        const size_t kstride = (size_t)a.S * a.ldv;
        const int jj = cf >> 1;
        const bool odd = (cf & 1) != 0;
        for (int kk = g; kk < a.nf; kk += G) {
            const int k = a.k0 + kk;
            const float2 Z = z[F::zi(row(k), jj)];
            const float2 Zm = k == 0 ? Z : z[F::zi(row(NT - k), jj)];
            float2 x = odd ? make_float2(0.5f * (Z.y + Zm.y), 0.5f * (Zm.x - Z.x))
                           : make_float2(0.5f * (Z.x + Zm.x), 0.5f * (Z.y - Zm.y));
            if (a.fwd_conj) x.y = -x.y;
            *MDC_AT(a.fwd_X, dsto + (size_t)kk * kstride, 1, ny, a.err, 18) = x;
        }
    }
}

template <int N1, int N2, int MODE, int PP, bool FUSE, int VEC>
void irfft4_go(mdc_plan* p, const IrfftArgs& a, cudaStream_t s) {
    using F = FourStep<N1, N2, PP>;
    constexpr size_t smem = F::smem_full + (MODE == 1 ? 0 : (size_t)FFT_THREADS * 4 * sizeof(float));
    static SmemLimit attr;
    attr.ensure(irfft4_kernel<N1, N2, MODE, PP, FUSE, VEC>, (int)smem);
    LaunchScope ls(p, s, MDC_KC_IRFFT);
    launch_pdl(irfft4_kernel<N1, N2, MODE, PP, FUSE, VEC>, dim3((a.C + F::CT - 1) / F::CT), FFT_THREADS, smem, s, a);
}

template <int N1, int N2, int PP>
void irfft4_mode(mdc_plan* p, const IrfftArgs& a, bool fuse, cudaStream_t s) {
    auto aligned = [&](int cols) {
        const uintptr_t m = 4 * cols - 1;
        return a.C % cols == 0 && (((uintptr_t)a.out | (uintptr_t)a.base | (uintptr_t)a.xw_w | (uintptr_t)a.xw_x) & m) == 0;
    };
    if (irfft_plain(a)) {
        if (aligned(2)) irfft4_go<N1, N2, 1, PP, false, 2>(p, a, s);
        else irfft4_go<N1, N2, 1, PP, false, 1>(p, a, s);
    } else if (aligned(4) && !a.reverse_out) {
        if (a.xw_w && fuse) irfft4_go<N1, N2, 2, PP, true, 4>(p, a, s);
        else if (a.xw_w) irfft4_go<N1, N2, 2, PP, false, 4>(p, a, s);
        else if (fuse) irfft4_go<N1, N2, 0, PP, true, 4>(p, a, s);
        else irfft4_go<N1, N2, 0, PP, false, 4>(p, a, s);
    } else {
        if (a.xw_w && fuse) irfft4_go<N1, N2, 2, PP, true, 1>(p, a, s);
        else if (a.xw_w) irfft4_go<N1, N2, 2, PP, false, 1>(p, a, s);
        else if (fuse) irfft4_go<N1, N2, 0, PP, true, 1>(p, a, s);
        else irfft4_go<N1, N2, 0, PP, false, 1>(p, a, s);
    }
}

}  // namespace

template <int N1, int N2>
bool irfft4_launch(mdc_plan* p, const IrfftArgs& a, cudaStream_t s) {
    constexpr int PS = few_cols_p<N1, N2>();
    const bool few = few_columns(a.C, FourStep<N1, N2>::CT) && PS < FourStep<N1, N2>::P;
    const bool fuse = a.fwd_X && !a.reverse_out;
    if (few) irfft4_mode<N1, N2, PS>(p, a, fuse, s);
    else irfft4_mode<N1, N2, 0>(p, a, fuse, s);
    return fuse;
}

}  // namespace mdc
