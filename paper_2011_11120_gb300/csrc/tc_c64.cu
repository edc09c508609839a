// Tensor-core (tcgen05) products for the complex64 kernel copy: K-hat and K-hat^H of Eq. 3 for more
// columns than the GEMV serves, at float32 accuracy.
//
// The complex product is the real GEMM of tc_gemm.cu on the interleaved (re, im) storage,
//   forward  D[r][n'] = sum_K' G^[r][K'] BT[n'][K'],  K' = 2s + c,  BT[2n] = (Xr, -Xi), BT[2n+1] = (Xi, Xr)
//   adjoint  D[m][n'] = sum_r G^[r][m] BT[n'][r],     m = 2s + c,   BT[2n] = Yr,        BT[2n+1] = Yi
// with every float32 factor written as three bfloat16 terms x = x0 + x1 + x2 (each the rounded
// remainder) and the six products
//   x0 y0  and  x0 y1 + x1 y0 + x1 y1 + x0 y2 + x2 y0
// (the dropped ones are below 2^-25 of |x y|).  Nothing is scaled: the sum of the terms is exact for
// magnitudes from 2^-110 (the last bit of x2 is then bfloat16's smallest subnormal, 2^-133) to 3.38e38
// (255.5 2^120, where x0 rounds to infinity); smaller values lose what lies below 2^-133, larger finite ones
// make the outputs they enter NaN or infinite, as an entry that is not finite does.
//
// Accuracy.  The tensor core's float32 accumulation truncates, by about 2^-25 of the running sum per
// MMA, which a long chain adds up (1e-6 over 48 MMAs).  So x0 y0 goes into an accumulator of its own
// that is emptied every chunk of 64 reduction elements (32 on the narrowest tile) into float32 registers
// (round to nearest), and the five small products, 2^-8 of the sum, into two others (even and odd
// halves of a step) that are emptied every 2048 elements, when the registers' sum joins the totals.
// Against 64 bits a forward pass with random data of 64 columns on 3721 x 3721 (100 on 9801 x 9801) is
// off by 2.0e-7 (1.9e-7), where the float32 GEMM it took the place of had 3.3e-7 (3.3e-7).
//
// What bounds it.  Six MMAs take 6 BN / 2 cycles per 16 reduction elements of a 128 x BN tile (384 at
// BN = 128), the kernel's bytes from HBM (8 KB per 16 elements and 128 rows) about 350 cycles with
// all 152 SMs reading: the two balance at 64 columns.  A goes through tensor memory, not shared
// memory: its float32 tile is read once by the converter warps and its three terms are then MMA
// operands that cost no shared-memory bandwidth (as shared-memory operands the six MMAs alone would
// saturate it).
#include <optional>

#include "tc_common.cuh"

namespace mdc {
namespace {

constexpr int C64_BM = 128;                 // rows per tile (TMEM lanes)
constexpr int C64_KS = 32;                  // reduction elements per step
constexpr int C64_TERMS = 3;
constexpr int C64_GROUP = 64;               // steps between drains of the small products
constexpr uint32_t C64_A_BYTES = C64_BM * C64_KS * 4;       // float32 tile of A: 16 KB
constexpr uint32_t C64_ACOLS = C64_TERMS * C64_KS / 2;      // TMEM columns of one converted A step
// warps 0..7: epilogue (two per TMEM lane quarter), 8..15: converters (two per lane quarter, taking
// alternate steps), 16 (and 20, see C64Ring::SEP): TMA, 17: MMA issue of x0 y0, 18 and 19: of the small
// products, one thread each.  An issuing thread takes about 48 cycles per MMA and 100 per barrier
// operation: one alone took 1250 cycles per step, two 1100, where the tensor cores need 774 at BN = 128
// and 560 below.
// Barriers of a step g sit in rings of C64_RING entries: ready[g % 8] (its three B terms landed and
// its A terms are in TMEM) and done[g % 8] (its MMAs completed): one wait and one commit per step and
// issuer (with a barrier per resource, and one issuer, a step took 1900 cycles whatever BN was).
constexpr int C64_RING = 8;
// Bound on the wait for each of the B producer's last copies: they land in microseconds, but their
// barrier also counts the converters, which may have given up.
constexpr unsigned long long C64_DRAIN_NS = 20000000ull;
constexpr int C64_STG_LD = 20;              // output staging row pitch (floats)

template <int BN> struct C64Ring {
    static constexpr uint32_t B_BYTES = C64_TERMS * BN * C64_KS * 2;      // three terms of one step of B
    static constexpr int NB = BN <= 32 ? 8 : (BN <= 64 ? 6 : (BN <= 96 ? 5 : 4));
    static constexpr int NAFIT = (200 * 1024 - NB * (int)B_BYTES) / (int)C64_A_BYTES;
    static constexpr int NA = NAFIT < C64_RING ? NAFIT : C64_RING;
    // SEP: a warp of its own loads B (narrow tiles, whose steps are shorter; wide tiles need the
    // registers of the twentieth warp's limit of 96 instead of 80)
    static constexpr bool SEP = BN <= 64;
    static constexpr int THREADS = (SEP ? 21 : 20) * 32;
    // TMEM: NHH buffers of x0 y0, two accumulators of small products, NW converted A steps
    static constexpr int NHH = BN > 96 ? 1 : 2;
    static constexpr int CHS = BN <= 32 ? 1 : 2;      // steps per chunk of x0 y0
    static_assert(C64_GROUP % CHS == 0, "groups of whole chunks");
    static constexpr int NW = (512 - (NHH + 2) * BN) / (int)C64_ACOLS >= 4 ? 4 : 2;
    static_assert(NB <= C64_RING && NA <= C64_RING && NW <= C64_RING / 2,
                  "a step's barrier is not reused before its waiters ran");
    static constexpr size_t smem =
        (size_t)NB * B_BYTES + (size_t)NA * C64_A_BYTES + 1024 + 512 + 8 * 32 * C64_STG_LD * 4;
    static_assert((NHH + 2) * BN + NW * (int)C64_ACOLS <= 512, "tensor memory");
    static_assert(smem <= 227 * 1024, "shared memory");
};

struct C64Args {
    int nf;             // frequencies
    int ksteps;         // reduction steps of C64_KS elements
    int nout;           // output rows: nr (forward) or ns (adjoint)
    int ncol;           // complex columns
    float2* out;
    int ldo, voff_o;
    int* err;
    unsigned long long wait_ns;
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"((unsigned long long)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// Shared-memory matrix descriptor of B: K-major, 64-byte swizzle (layout type 4), 512 bytes per group
// of eight 64-byte rows; only the low word holds the address.
constexpr uint32_t C64_DESC_HI = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return (addr >> 4) | (1u << 16); }
// D(tmem) (+)= A(tmem) * B(smem), kind::f16: D float32, A and B bfloat16, N = BN, M = 128.  The
// operands are warp-uniform values of a converged warp, so they sit in uniform registers.
template <int BN>
__device__ __forceinline__ void c64_mma(uint32_t d, uint32_t a, uint32_t b_lo, uint32_t acc) {
    constexpr uint32_t idesc =
        (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(C64_BM >> 4) << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 bd;\n\t"
        "mov.b64 bd, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], bd, %4, p;\n\t}\n" ::"r"(d),
        "r"(a), "r"(b_lo), "r"(C64_DESC_HI), "r"(idesc), "r"(acc)
        : "memory");
}

// The leading bfloat16 term of a pair, packed (first value in the low half); the pair becomes its
// remainder (exact in float32).
__device__ __forceinline__ uint32_t take_term(float& a, float& b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const uint32_t w = *reinterpret_cast<const uint32_t*>(&h);
    a -= __uint_as_float(w << 16);
    b -= __uint_as_float(w & 0xffff0000u);
    return w;
}

// Persistent CTA (one per SM) over tiles (column tile fastest, then row tile, then frequency).  Every
// mbarrier wait is bounded; a warp whose wait runs out records a code and leaves its loop, and the
// others follow when their own waits run out.
template <bool ADJ, int BN>
__global__ void __launch_bounds__(C64Ring<BN>::THREADS, 1)
    tc_c64_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, C64Args a,
                  const int* active, int n_tiles_n, int n_tiles_m, int n_tiles) {
    if (active && *active == 0) return;
    using R = C64Ring<BN>;
    constexpr int NA = R::NA, NB = R::NB, NW = R::NW, NHH = R::NHH, CHS = R::CHS;
    constexpr bool SEP = R::SEP;
    constexpr uint32_t B_BYTES = R::B_BYTES;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = su32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t abase = base + NB * B_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + NB * B_BYTES + NA * C64_A_BYTES);
    // afull[NA], ready[8], done[8], acce[2], corre, drain, tmem slot
    const uint32_t afull0 = su32(bars);
    const uint32_t ready0 = afull0 + 8 * NA, done0 = ready0 + 8 * C64_RING;
    const uint32_t acce0 = done0 + 8 * C64_RING, corre = acce0 + 16, drain0 = corre + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NA + 2 * C64_RING + 4);
    static_assert(NA + 2 * C64_RING + 5 <= 64, "barrier space");
    float* stage = reinterpret_cast<float*>(bars + 64);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t_first = (int)blockIdx.x, t_stride = (int)gridDim.x;
    const unsigned long long wl = a.wait_ns;
    const int ksteps = a.ksteps;

    if (warp == 0) tmem_alloc(su32(tmem_slot), 512);
    if (threadIdx.x == 32) {
        for (int i = 0; i < NA; ++i) mbar_init(afull0 + 8 * i, 1);
        for (int i = 0; i < C64_RING; ++i) {
            mbar_init(ready0 + 8 * i, 5);        // four converter warps and the B producer (with its bytes)
            mbar_init(done0 + 8 * i, 3);             // the three issuers' commits
        }
        for (int i = 0; i < 2; ++i) mbar_init(acce0 + 8 * i, 8);
        mbar_init(corre, 8);
        mbar_init(drain0, 3);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    constexpr uint32_t CORR = NHH * BN, ACOL = CORR + 2 * BN;      // TMEM columns
    const int per_freq = n_tiles_n * n_tiles_m;
    auto coords = [&](int t, int& k, int& m0, int& n0) {
        k = t / per_freq;
        const int rem = t - k * per_freq;
        const int mt = rem / n_tiles_n;
        m0 = mt * C64_BM;
        n0 = (rem - mt * n_tiles_n) * BN;
    };

    if (warp == 16 || warp == 20) {
        if (lane == 0) {
            // TMA: warp 16 loads A, and B as well unless warp 20 does.  A step's slots are free when the
            // MMAs of the step that used them before are done.  In the joint loop A runs NA - NB steps
            // ahead, so that one wait frees both.
            const bool do_a = warp == 16, do_b = !SEP || warp == 20;
            constexpr int AHEAD = SEP ? 0 : NA - NB;
            static_assert(AHEAD >= 0, "A ring at least as deep as B's");
            const unsigned depth = SEP && do_a ? NA : NB;
            unsigned g = 0, ga = 0;                      // steps walked, A copies issued
            int s = 0, y = 0, ta = t_first, ka = 0;      // slots; A's tile and step within it
            auto load_a = [&]() {
                if (ta >= n_tiles) return;
                int k, m0, n0;
                coords(ta, k, m0, n0);
                const uint32_t bar = afull0 + 8 * y;
                mbar_expect_tx(bar, C64_A_BYTES);
                // forward: 128 rows x 32 floats (swizzled); adjoint: 32 rows x 128 floats
                if (!ADJ) tma_load_3d(abase + y * C64_A_BYTES, &tmA, bar, ka * C64_KS, m0, k);
                else tma_load_3d(abase + y * C64_A_BYTES, &tmA, bar, m0, ka * C64_KS, k);
                ++ga;
                if (++y == NA) y = 0;
                if (++ka == ksteps) {
                    ka = 0;
                    ta += t_stride;
                }
            };
            for (int i = 0; i < AHEAD; ++i) load_a();
            bool ok = true;
            for (int tile = t_first; tile < n_tiles && ok; tile += t_stride) {
                int k, m0, n0;
                coords(tile, k, m0, n0);
                for (int kb = 0; kb < ksteps; ++kb, ++g) {
                    const unsigned f = g - depth;                // the step that used the slot before
                    if (g >= depth && !mbar_wait_idle(done0 + 8 * (f % C64_RING), (f / C64_RING) & 1, a.err, 22, wl)) {
                        ok = false;
                        break;
                    }
                    if (do_a) load_a();
                    if (do_b) {
                        const uint32_t bar = ready0 + 8 * (g % C64_RING);
                        mbar_expect_tx(bar, B_BYTES);
                        tma_load_4d(base + s * B_BYTES, &tmB, bar, kb * C64_KS, n0, k, 0);
                        if (++s == NB) s = 0;
                    }
                }
            }
            // every copy this thread issued has landed before the CTA can exit
            for (unsigned q = ga > NA ? ga - NA : 0; q < ga; ++q)
                mbar_wait_idle(afull0 + 8 * (q % NA), (q / NA) & 1, a.err, 21, TC_DRAIN_NS);
            if (do_b)
                for (unsigned q = g > NB ? g - NB : 0; q < g; ++q)
                    mbar_wait_idle(ready0 + 8 * (q % C64_RING), (q / C64_RING) & 1, a.err, 23, C64_DRAIN_NS);
        }
    } else if (warp == 17) {
        if (lane == 0) {
            // MMA issue of x0 y0
            unsigned g = 0, ci = 0;              // steps and chunks issued
            int s = 0;                           // B slot
            bool ok = true;
            for (int tile = t_first; tile < n_tiles && ok; tile += t_stride)
                for (int kb = 0; kb < ksteps; ++kb, ++g) {
                    const bool start = kb % CHS == 0;
                    if ((start && ci >= NHH &&
                         !mbar_wait_idle(acce0 + 8 * (ci % NHH), (ci / NHH - 1) & 1, a.err, 24, wl)) ||
                        !mbar_wait_idle(ready0 + 8 * (g % C64_RING), (g / C64_RING) & 1, a.err, 25, wl)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (ci % NHH) * BN, at = tmem + ACOL + (g % NW) * C64_ACOLS;
                    const uint32_t bd = desc_lo(base + s * B_BYTES);
                    c64_mma<BN>(d, at, bd, start ? 0u : 1u);
                    c64_mma<BN>(d, at + 8, bd + 2, 1u);
                    umma_commit(done0 + 8 * (g % C64_RING));
                    if (kb % CHS == CHS - 1 || kb == ksteps - 1) ++ci;
                    if (++s == NB) s = 0;
                }
            // every MMA this thread issued has completed before TMEM is freed
            umma_commit(drain0);
            mbar_wait_idle(drain0, 0, a.err, 28, TC_DRAIN_NS);
        }
    } else if (warp >= 18) {
        if (lane == 0) {
            // MMA issue of the small products of half kk of each step, into an accumulator of its own
            const int kk = warp - 18;
            const uint32_t d = tmem + CORR + kk * BN;
            unsigned g = 0, di = 0;              // steps issued, times the accumulator was started
            int s = 0;
            bool ok = true;
            constexpr uint32_t TERM = BN * 64 / 16;                     // descriptor units between B terms
            for (int tile = t_first; tile < n_tiles && ok; tile += t_stride)
                for (int kb = 0; kb < ksteps; ++kb, ++g) {
                    const bool fresh = kb % C64_GROUP == 0;
                    // a new start waits until the epilogue has emptied the accumulator
                    if ((fresh && di > 0 && !mbar_wait_idle(corre, (di - 1) & 1, a.err, 27, wl)) ||
                        !mbar_wait_idle(ready0 + 8 * (g % C64_RING), (g / C64_RING) & 1, a.err, 26, wl)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a0 = tmem + ACOL + (g % NW) * C64_ACOLS + kk * 8, a1 = a0 + 16, a2 = a0 + 32;
                    const uint32_t b0 = desc_lo(base + s * B_BYTES) + kk * 2, b1 = b0 + TERM, b2 = b1 + TERM;
                    c64_mma<BN>(d, a0, b1, fresh ? 0u : 1u);
                    c64_mma<BN>(d, a1, b0, 1u);
                    c64_mma<BN>(d, a1, b1, 1u);
                    c64_mma<BN>(d, a0, b2, 1u);
                    c64_mma<BN>(d, a2, b0, 1u);
                    umma_commit(done0 + 8 * (g % C64_RING));
                    di += fresh;
                    if (++s == NB) s = 0;
                }
            umma_commit(drain0);
            mbar_wait_idle(drain0, 0, a.err, 33, TC_DRAIN_NS);
        }
    } else if (warp >= 8) {
        // converters: lane row R of the tile, float32 -> three bfloat16 terms in tensor memory
        const int q = warp & 3, grp = (warp - 8) >> 2, row = 32 * q + lane;
        unsigned g = 0;
        int y = grp % NA;
        uint32_t ph = 0;
        bool ok = true;
        for (int tile = t_first; tile < n_tiles && ok; tile += t_stride)
            for (int kb = 0; kb < ksteps; ++kb, ++g) {
                if ((int)(g & 1) != grp) continue;
                const int w = (int)(g % NW);
                if (!warp_wait(afull0 + 8 * y, ph, a.err, 29, wl)) {
                    ok = false;
                    break;
                }
                const unsigned char* at = gbase + NB * B_BYTES + (size_t)y * C64_A_BYTES;
                float v[C64_KS];
                if (!ADJ) {
                    // 16-byte chunk c of the 128-byte row sits at chunk c ^ (row % 8)
#pragma unroll
                    for (int c = 0; c < C64_KS / 4; ++c) {
                        const float4 f = *reinterpret_cast<const float4*>(at + row * 128 + ((c ^ (row & 7)) << 4));
                        v[4 * c] = f.x;
                        v[4 * c + 1] = f.y;
                        v[4 * c + 2] = f.z;
                        v[4 * c + 3] = f.w;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < C64_KS; ++i)
                        v[i] = reinterpret_cast<const float*>(at)[i * C64_BM + row];
                }
                // the MMAs that read this TMEM buffer on its previous use are complete
                const unsigned f = g - NW;
                if (g >= NW && !warp_wait(done0 + 8 * (f % C64_RING), (f / C64_RING) & 1, a.err, 30, wl)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t dst = tmem + ((uint32_t)(32 * q) << 16) + ACOL + (uint32_t)w * C64_ACOLS;
#pragma unroll 1
                for (int t = 0; t < C64_TERMS; ++t) {
                    uint32_t h[C64_KS / 2];
#pragma unroll
                    for (int i = 0; i < C64_KS / 2; ++i) h[i] = take_term(v[2 * i], v[2 * i + 1]);
                    tmem_st16(dst + t * (C64_KS / 2), h);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(ready0 + 8 * (g % C64_RING));
                y += 2;
                if (y >= NA) {
                    y -= NA;
                    ph ^= 1;
                }
            }
    } else {
        const int q = warp & 3;                  // TMEM lane quarter
        constexpr int BH = BN / 2;               // accumulator columns of this warp
        const int cbeg = (warp >> 2) * BH;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)cbeg;
        float* stg = stage + warp * (32 * C64_STG_LD);
        const int nch = (ksteps + CHS - 1) / CHS;
        unsigned g0 = 0, ci = 0;                 // first step of the tile, chunks consumed
        bool ok = true;
        for (int tile = t_first; tile < n_tiles && ok; tile += t_stride, g0 += ksteps) {
            int k, m0, n0;
            coords(tile, k, m0, n0);
            float acc[BH];
            float4 tot[BH / 4];
            float4* totp = tot;
            asm volatile("" : "+l"(totp));       // keeps the totals out of the registers
#pragma unroll
            for (int c = 0; c < BH; ++c) acc[c] = 0.f;
            auto add = [&](uint32_t from) {
#pragma unroll
                for (int c0 = 0; c0 < BH; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld16(from + c0, v);
#pragma unroll
                    for (int j = 0; j < 16; ++j) acc[c0 + j] += __uint_as_float(v[j]);
                }
            };
            for (int ch = 0; ch < nch; ++ch, ++ci) {
                const int buf = (int)(ci % NHH);
                const unsigned e = g0 + (unsigned)min(CHS * ch + CHS - 1, ksteps - 1);       // the chunk's last step
                if (!warp_wait(done0 + 8 * (e % C64_RING), (e / C64_RING) & 1, a.err, 31, wl)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                add(tl + (uint32_t)(buf * BN));
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acce0 + 8 * buf);
                if ((ch + 1) % (C64_GROUP / CHS) == 0 || ch == nch - 1) {
                    add(tl + CORR);
                    add(tl + CORR + BN);
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(corre);
                    // the group's sum joins the totals, which sit in local memory (a visit every 64 steps)
                    const bool first = ch < C64_GROUP / CHS;
#pragma unroll
                    for (int c = 0; c < BH; c += 8) {
                        float4 t0 = make_float4(0.f, 0.f, 0.f, 0.f), t1 = t0;
                        if (!first) {
                            t0 = totp[c / 4];
                            t1 = totp[c / 4 + 1];
                        }
                        totp[c / 4] = make_float4(t0.x + acc[c], t0.y + acc[c + 1], t0.z + acc[c + 2], t0.w + acc[c + 3]);
                        totp[c / 4 + 1] =
                            make_float4(t1.x + acc[c + 4], t1.y + acc[c + 5], t1.z + acc[c + 6], t1.w + acc[c + 7]);
                        asm volatile("" ::: "memory");
                    }
#pragma unroll
                    for (int c = 0; c < BH; ++c) acc[c] = 0.f;
                }
            }
            if (!ok) break;
            // 16 accumulator columns (8 complex output columns) of the warp's 32 rows at a time, through
            // a staging tile, so that each store instruction writes 8 rows x 64 contiguous bytes
            constexpr int NROWS = ADJ ? 16 : 32;
            const int orow0 = ADJ ? (m0 + 32 * q) >> 1 : m0 + 32 * q;
#pragma unroll 1
            for (int c0 = 0; c0 < BH; c0 += 16) {
                float v[16], w[16];
#pragma unroll
                for (int i4 = 0; i4 < 4; ++i4) {
                    const float4 t = totp[c0 / 4 + i4];
                    v[4 * i4] = t.x;
                    v[4 * i4 + 1] = t.y;
                    v[4 * i4 + 2] = t.z;
                    v[4 * i4 + 3] = t.w;
                }
                if (!ADJ) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) w[j] = v[j];
                } else {
                    // rows 2s and 2s + 1 of the real product hold the two halves of output row s
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float pr = __shfl_xor_sync(0xffffffffu, v[2 * j], 1);
                        const float pi = __shfl_xor_sync(0xffffffffu, v[2 * j + 1], 1);
                        w[2 * j] = v[2 * j] + pi;
                        w[2 * j + 1] = v[2 * j + 1] - pr;
                    }
                }
                if (!ADJ || (lane & 1) == 0) {
                    float* rowp = stg + (ADJ ? lane >> 1 : lane) * C64_STG_LD;
#pragma unroll
                    for (int i4 = 0; i4 < 4; ++i4)
                        *reinterpret_cast<float4*>(rowp + 4 * i4) =
                            make_float4(w[4 * i4], w[4 * i4 + 1], w[4 * i4 + 2], w[4 * i4 + 3]);
                }
                __syncwarp();
                const int cc = lane >> 3, n = ((n0 + cbeg + c0) >> 1) + 2 * cc;
#pragma unroll
                for (int it = 0; it < NROWS / 8; ++it) {
                    const int rr = (lane & 7) + 8 * it, orow = orow0 + rr;
                    const float4 val = *reinterpret_cast<const float4*>(stg + rr * C64_STG_LD + 4 * cc);
                    if (orow < a.nout && n < a.ncol &&
                        MDC_INB(((size_t)k * a.nout + orow) * a.ldo + a.voff_o + n, n + 1 < a.ncol ? 2 : 1,
                                (long long)a.nf * a.nout * a.ldo, a.err, 140)) {
                        float2* dst = a.out + ((size_t)k * a.nout + orow) * a.ldo + a.voff_o + n;
                        if (n + 1 < a.ncol && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
                            *reinterpret_cast<float4*>(dst) = val;
                        } else {
                            dst[0] = make_float2(val.x, val.y);
                            if (n + 1 < a.ncol) dst[1] = make_float2(val.z, val.w);
                        }
                    }
                }
                __syncwarp();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------ operand preparation
// Spectra [nf][rows][ldi] (ncol columns from voff) -> three bfloat16 planes [3][nf][2 ncol][pitch] of
// BT.  A CTA stages 256 rows x 8 columns through shared memory: reads of 64 contiguous bytes per row,
// writes of one packed pair per thread along the reduction axis.
constexpr int C64_PREP_ROWS = 256, C64_PREP_COLS = 8;

template <bool ADJ>
__global__ void __launch_bounds__(256) tc_c64_prep(const float2* __restrict__ X, int ldi, int voff, int rows,
                                                   int ncol, int pitch, uint32_t* __restrict__ BT,
                                                   const int* active, int* err) {
    if (active && *active == 0) return;
    __shared__ float2 tile[C64_PREP_ROWS][C64_PREP_COLS + 1];
    const int k = blockIdx.z, s0 = blockIdx.y * C64_PREP_ROWS, n0 = blockIdx.x * C64_PREP_COLS;
    const float2* Xk = X + (size_t)k * rows * ldi + voff;
#pragma unroll
    for (int u = 0; u < C64_PREP_COLS; ++u) {
        const int idx = threadIdx.x + 256 * u;
        const int rr = idx >> 3, j = idx & 7, s = s0 + rr;
        const bool in = s < rows && n0 + j < ncol &&
                        MDC_INB((size_t)k * rows * ldi + voff + (size_t)s * ldi + n0 + j, 1,
                                (long long)gridDim.z * rows * ldi, err, 141);
        tile[rr][j] = in ? Xk[(size_t)s * ldi + n0 + j] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const size_t row2 = (size_t)pitch / 2;                       // packed pairs per row
    const size_t plane = (size_t)gridDim.z * 2 * ncol * row2;    // packed pairs per plane
    if (!ADJ) {
        // one (re, im) pair of column n per thread: (Xr, -Xi) into row 2n, (Xi, Xr) into row 2n + 1
        const int s = s0 + threadIdx.x;
        if (s >= rows) return;
#pragma unroll
        for (int j = 0; j < C64_PREP_COLS; ++j) {
            const int n = n0 + j;
            if (n >= ncol) break;
            float2 v = tile[threadIdx.x][j];
            const size_t o = ((size_t)k * 2 * ncol + 2 * n) * row2 + s;
            if (!MDC_INB(o, row2 + 1, (long long)plane, err, 142)) break;
#pragma unroll
            for (int t = 0; t < C64_TERMS; ++t) {
                const uint32_t h = take_term(v.x, v.y);          // Xr low, Xi high
                BT[t * plane + o] = h ^ 0x80000000u;
                BT[t * plane + o + row2] = (h >> 16) | (h << 16);
            }
        }
    } else {
        // rows r, r + 1 of four columns per thread: Yr pairs into row 2n, Yi pairs into row 2n + 1
        const int tt = threadIdx.x & 127, jb = (threadIdx.x >> 7) * (C64_PREP_COLS / 2);
        const int r = s0 + 2 * tt;
        if (r >= rows) return;
#pragma unroll
        for (int jj = 0; jj < C64_PREP_COLS / 2; ++jj) {
            const int n = n0 + jb + jj;
            if (n >= ncol) break;
            float2 va = tile[2 * tt][jb + jj], vb = tile[2 * tt + 1][jb + jj];
            const size_t o = ((size_t)k * 2 * ncol + 2 * n) * row2 + (r >> 1);
            if (!MDC_INB(o, row2 + 1, (long long)plane, err, 143)) break;
#pragma unroll
            for (int t = 0; t < C64_TERMS; ++t) {
                BT[t * plane + o] = take_term(va.x, vb.x);
                BT[t * plane + o + row2] = take_term(va.y, vb.y);
            }
        }
    }
}

// ------------------------------------------------------------------ host side
// Column tile for n2 = 2 ncol real columns: the smallest of 32, 64, 96, 128 that holds them, else the
// one with the least total work (a tile costs about 57 + BN in shared-memory time: its A tile and
// its B reads).
int c64_bn(int n2) {
    for (int bn : {32, 64, 96, 128})
        if (n2 <= bn) return bn;
    int best = 128;
    for (int bn : {96, 64})
        if ((n2 + bn - 1) / bn * (57 + bn) < (n2 + best - 1) / best * (57 + best)) best = bn;
    return best;
}

template <bool ADJ, int BN>
void c64_go(const CUtensorMap& mA, const CUtensorMap& mB, const C64Args& a, const int* active, int tiles_n,
            int tiles_m, cudaStream_t s) {
    static SmemLimit attr;
    attr.ensure(tc_c64_kernel<ADJ, BN>, (int)C64Ring<BN>::smem);
    const int n_tiles = tiles_n * tiles_m * a.nf, sms = sm_count();
    tc_c64_kernel<ADJ, BN><<<n_tiles < sms ? n_tiles : sms, C64Ring<BN>::THREADS, C64Ring<BN>::smem, s>>>(
        mA, mB, a, active, tiles_n, tiles_m, n_tiles);
}

int c64_pitch(const mdc_plan* p, bool adjoint) { return adjoint ? (int)round_up(p->nr, 8) : (int)(2 * p->ldg); }

}  // namespace

// Three planes of 2 ncol rows in the longer of the two directions' pitch, in 16-bit elements.
size_t tc_c64_scratch_elems(const mdc_plan* p, int ncol) {
    const size_t kf = (size_t)c64_pitch(p, false), ka = (size_t)c64_pitch(p, true);
    return (size_t)C64_TERMS * p->nf * 2 * ncol * (kf > ka ? kf : ka);
}

bool tc_c64_ready(const mdc_plan* p, int ncol) {
    return p->storage == MDC_C64 && p->tcB != nullptr && (ncol < C64_TILE_COLS ? ncol : C64_TILE_COLS) <= p->tc_cap &&
           encode_fn() != nullptr;
}

namespace {
// Columns [voff, voff + ncol) with column tiles of bn real columns.
bool c64_slab(mdc_plan* p, bool adjoint, const float2* in, int ldi, int voff_i, float2* out, int ldo, int voff_o,
              int ncol, int bn, cudaStream_t s, const int* active, bool scoped) {
    const int rows = adjoint ? p->nr : p->ns;                  // reduction rows of the spectra
    const int pitch = c64_pitch(p, adjoint);
    const uint64_t kp = 2 * (uint64_t)p->ldg;
    auto enc = encode_fn();
    if (!enc) return false;
    CUtensorMap mA, mB;
    {
        const cuuint64_t dims[3] = {kp, (cuuint64_t)p->nr, (cuuint64_t)p->nf};
        const cuuint64_t strides[2] = {kp * 4, kp * 4 * p->nr};
        const cuuint32_t boxf[3] = {C64_KS, C64_BM, 1}, boxa[3] = {C64_BM, C64_KS, 1}, es[3] = {1, 1, 1};
        if (enc(&mA, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, p->G, dims, strides, adjoint ? boxa : boxf, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, adjoint ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    {
        // the extents are the written ones: past them (reduction tail, unused tile columns) TMA reads zeros
        const cuuint64_t red = adjoint ? (cuuint64_t)rows : 2 * (cuuint64_t)rows, n2 = 2 * (cuuint64_t)ncol;
        const cuuint64_t dims[4] = {red, n2, (cuuint64_t)p->nf, C64_TERMS};
        const cuuint64_t rb = 2 * (cuuint64_t)pitch;
        const cuuint64_t strides[3] = {rb, rb * n2, rb * n2 * p->nf};
        const cuuint32_t box[4] = {C64_KS, (cuuint32_t)bn, 1, C64_TERMS}, es[4] = {1, 1, 1, 1};
        if (enc(&mB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, p->tcB, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    std::optional<LaunchScope> scope;
    if (scoped) scope.emplace(p, s, MDC_KC_TC_PREP);
    const dim3 pg((unsigned)((ncol + C64_PREP_COLS - 1) / C64_PREP_COLS),
                  (unsigned)((rows + C64_PREP_ROWS - 1) / C64_PREP_ROWS), (unsigned)p->nf);
    if (adjoint)
        tc_c64_prep<true><<<pg, 256, 0, s>>>(in, ldi, voff_i, rows, ncol, pitch, (uint32_t*)p->tcB, active, p->err_flag);
    else
        tc_c64_prep<false><<<pg, 256, 0, s>>>(in, ldi, voff_i, rows, ncol, pitch, (uint32_t*)p->tcB, active, p->err_flag);
    scope.reset();
    C64Args a{};
    a.nf = p->nf;
    a.ksteps = (int)(((adjoint ? (int64_t)rows : 2 * (int64_t)rows) + C64_KS - 1) / C64_KS);
    a.nout = adjoint ? p->ns : p->nr;
    a.ncol = ncol;
    a.out = out;
    a.ldo = ldo;
    a.voff_o = voff_o;
    a.err = p->err_flag;
    a.wait_ns = p->wait_ns;
    const int tiles_n = (2 * ncol + bn - 1) / bn;
    const int tiles_m = (int)(((adjoint ? 2 * (int64_t)p->ns : (int64_t)p->nr) + C64_BM - 1) / C64_BM);
    if (scoped) scope.emplace(p, s, adjoint ? MDC_KC_PRODUCT_ADJ : MDC_KC_PRODUCT_FWD);
#define MDC_C64_CASE(BNV)                                                                 \
    case BNV:                                                                             \
        if (adjoint) c64_go<true, BNV>(mA, mB, a, active, tiles_n, tiles_m, s);           \
        else c64_go<false, BNV>(mA, mB, a, active, tiles_n, tiles_m, s);                  \
        break;
    switch (bn) {
        MDC_C64_CASE(32)
        MDC_C64_CASE(64)
        MDC_C64_CASE(96)
        MDC_C64_CASE(128)
    }
#undef MDC_C64_CASE
    return true;
}
}  // namespace

// An operand of fewer columns than the product's takes it slab by slab, each of whole column tiles, so the
// sums are the same.
bool launch_tc_c64(mdc_plan* p, bool adjoint, const float2* in, int ldi, int voff_i, float2* out, int ldo,
                   int voff_o, int ncol, cudaStream_t s, const int* active, bool scoped) {
    const int bn = c64_bn(2 * ncol), tile = bn / 2;
    const int slab = ncol <= p->tc_cap ? ncol : p->tc_cap / tile * tile;
    for (int c = 0; c < ncol; c += slab)
        if (!c64_slab(p, adjoint, in, ldi, voff_i + c, out, ldo, voff_o + c, ncol - c < slab ? ncol - c : slab, bn, s,
                      active, scoped))
            return false;
    return true;
}

}  // namespace mdc
