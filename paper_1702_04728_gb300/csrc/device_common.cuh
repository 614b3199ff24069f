// Device code shared by the fused kernels (FP32 FFT form and tensor-core DFT
// form): packed FP32x2 complex arithmetic, small DFTs with compile-time
// twiddles, the exact 4+4-bit unpack, tensor-memory access and the two
// up-channelisation passes (Sec. 3.2) that run out of tensor memory.
#pragma once

#include "bf_internal.h"

#include <cstdint>

namespace chimebf {
namespace {

// ---------------------------------------------------------------------------
// packed FP32x2 helpers (sm_100+: FADD2 / FMUL2 / FFMA2)
// ---------------------------------------------------------------------------
struct cp {            // two complex values in SoA form
    float2 re, im;
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 bc(float v) { return make_float2(v, v); }

__device__ __forceinline__ cp cadd(cp a, cp b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ cp csub(cp a, cp b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a * (C + i S), C and S pairs (per element of the pair)
__device__ __forceinline__ cp cmulp(cp a, float2 C, float2 S) {
    return {fma2(a.im, make_float2(-S.x, -S.y), mul2(a.re, C)), fma2(a.re, S, mul2(a.im, C))};
}
__device__ __forceinline__ cp ld_cp(const float4* p) {
    const float4 v = *p;
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

__device__ __forceinline__ void dft4(cp& a0, cp& a1, cp& a2, cp& a3) {
    const cp s02 = cadd(a0, a2), d02 = csub(a0, a2), s13 = cadd(a1, a3);
    // (a1 - a3) * (-i) = (a1.im - a3.im) + i (a3.re - a1.re)
    const cp d13 = {sub2(a1.im, a3.im), sub2(a3.re, a1.re)};
    a0 = cadd(s02, s13);
    a2 = csub(s02, s13);
    a1 = cadd(d02, d13);
    a3 = csub(d02, d13);
}

// A packed multiply-add whose three operands are all registers of their own takes 3.7 cycles of a
// scheduler, one that shares a constant or uniform operand 2.3 and a packed add 2.1 (measured, 2 or
// more warps); hence compile-time twiddles where the transform allows them, and plain products
// before an add-only first stage where the twiddles differ per lane.
//
// Radix-2 butterfly with a twiddle, factored for fused multiply-adds: with
// w = c (1 + i t), (a, b) -> (a + w b, a - w b) as p = (1 + i t) b (two FMA)
// and a +- c p (four FMA), six operations instead of a complex product and two
// complex additions (eight).  kRot: the twiddle is -i w, by exchanging p's parts.
// t = Im w / c with c as rounded, so both parts of w carry one rounding; the two
// roundings of p and the sums are relative to |b|, whatever the size of t.
template <bool kRot>
__device__ __forceinline__ void bfly_p(cp& a, cp& b, float2 pre, float2 pim, float c) {
    if constexpr (kRot) {
        b = {fma2(pim, bc(-c), a.re), fma2(pre, bc(c), a.im)};
        a = {fma2(pim, bc(c), a.re), fma2(pre, bc(-c), a.im)};
    } else {
        b = {fma2(pre, bc(-c), a.re), fma2(pim, bc(-c), a.im)};
        a = {fma2(pre, bc(c), a.re), fma2(pim, bc(c), a.im)};
    }
}
template <bool kRot>
__device__ __forceinline__ void bfly_ct(cp& a, cp& b, float c, float t) {
    bfly_p<kRot>(a, b, fma2(b.im, bc(-t), b.re), fma2(b.re, bc(t), b.im), c);
}

// cos and sin of 2 pi e / 32, e = 0..8
__device__ __forceinline__ constexpr double cos32(int e) {
    constexpr double t[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                             0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                             0.19509032201612826785, 0.0};
    return t[e];
}
__device__ __forceinline__ constexpr double sin32(int e) { return cos32(8 - e); }

// The butterfly with w = exp(-2 pi i E / 32), 0 <= E < 16 (E >= 8: -i times E - 8).
template <int E>
__device__ __forceinline__ void bfly(cp& a, cp& b) {
    static_assert(E >= 0 && E < 16, "angle out of range");
    if constexpr (E == 0) {
        const cp y = cadd(a, b), z = csub(a, b);
        a = y;
        b = z;
    } else if constexpr (E == 8) {
        // w = -i: a - i b = (a.re + b.im, a.im - b.re)
        const cp y = {add2(a.re, b.im), sub2(a.im, b.re)};
        const cp z = {sub2(a.re, b.im), add2(a.im, b.re)};
        a = y;
        b = z;
    } else if constexpr ((E & 7) == 4) {
        // 45 degrees: the tangent is 1, so sums in place of two FMAs with a constant (the same bits; 0.3 % of
        // an FP32-form launch)
        bfly_p<(E >= 8)>(a, b, add2(b.re, b.im), sub2(b.im, b.re), (float)cos32(4));
    } else {
        constexpr float c = (float)cos32(E & 7), t = (float)(-sin32(E & 7) / (double)c);
        bfly_ct<(E >= 8)>(a, b, c, t);
    }
}

// forward DFT8 (2 x 4), natural order in and out; the last stage's twiddles
// W8^k fused into its butterflies
__device__ __forceinline__ void dft8(cp (&x)[8]) {
    dft4(x[0], x[2], x[4], x[6]);
    dft4(x[1], x[3], x[5], x[7]);
    bfly<0>(x[0], x[1]);
    bfly<4>(x[2], x[3]);
    bfly<8>(x[4], x[5]);
    bfly<12>(x[6], x[7]);
    // X[k] = x[2k], X[k + 4] = x[2k + 1]
    cp y[8];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        y[k1] = x[2 * k1];
        y[k1 + 4] = x[2 * k1 + 1];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = y[k];
}

// dft16 leaves X[k + 8 (l & 1) + 4 (l >> 1)] in slot 4 r + l, with (r, k) = (0, 0), (1, 2),
// (2, 1), (3, 3): put them in natural order.
__device__ __forceinline__ void dft16_order(cp (&x)[16]) {
    cp y[16];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int k = r == 1 ? 2 : r == 2 ? 1 : r;
#pragma unroll
        for (int l = 0; l < 4; ++l) y[k + 8 * (l & 1) + 4 * (l >> 1)] = x[4 * r + l];
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = y[k];
}

// One radix-4 group of dft16's second stage: inputs in slots 4 r + b, twiddle V^b with
// V = exp(-2 pi i E / 32).
template <int E>
__device__ __forceinline__ void dft16_group(cp& x0, cp& x1, cp& x2, cp& x3) {
    bfly<2 * E>(x0, x2);
    bfly<2 * E>(x1, x3);
    bfly<E>(x0, x1);                         // out 0 and 2
    bfly<E + 8>(x2, x3);                     // out 1 and 3
}

// forward DFT16 (4 x 4) of x[n] exp(-2 pi i S n / 32), natural order in and out: S = 0 is the
// plain transform; S = 1 (the odd bins of a zero-padded DFT32) carries its input twiddles
// inside the butterflies (176 operations against 148, where a separate product takes 60 more)
template <int S = 0>
__device__ __forceinline__ void dft16(cp (&x)[16]) {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        bfly<8 * S>(x[b], x[8 + b]);
        bfly<8 * S>(x[4 + b], x[12 + b]);
        bfly<4 * S>(x[b], x[4 + b]);         // k = 0, 2
        bfly<4 * S + 8>(x[8 + b], x[12 + b]);    // k = 1, 3
    }
    dft16_group<S>(x[0], x[1], x[2], x[3]);
    dft16_group<S + 4>(x[4], x[5], x[6], x[7]);
    dft16_group<S + 2>(x[8], x[9], x[10], x[11]);
    dft16_group<S + 6>(x[12], x[13], x[14], x[15]);
    dft16_order(x);
}

// ---------------------------------------------------------------------------
// 4+4-bit unpack (Table 1) of the same byte position in two words.  A nibble at bit q of a word sits
// in the mantissa of 2^23; one FFMA2 scales it back by 2^-q and removes 2^23 and the +8 offset --
// exact throughout.
// ---------------------------------------------------------------------------
// The same bits in a uniform register (every lane holds x): an operand that costs no register read.
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_or_sync(0xffffffffu, x); }
__device__ __forceinline__ float uniform(float x) { return __uint_as_float(uniform(__float_as_uint(x))); }

// The nibbles of one polarisation in a byte pair (low byte polarisation 0): masks and the
// constants of the exact rescaling.
struct PolSel {
    uint32_t mi, mr;
    float si, bi, sr, br;
};
// (called by whole warps; uniform registers for these are worth 4 % of an FP32-form launch)
__device__ __forceinline__ PolSel pol_sel(int pol) {
    const float s = pol ? 1.f / 256.f : 1.f;
    return {uniform(pol ? 0xF00u : 0xFu), uniform(pol ? 0xF000u : 0xF0u), uniform(s),
            uniform(-(8388608.f * s + 8.f)), uniform(s * 0.0625f), uniform(-(524288.f * s + 8.f))};
}
__device__ __forceinline__ float2 nibm(uint32_t g0, uint32_t g1, uint32_t m, float s, float b) {
    return fma2(make_float2(__uint_as_float((g0 & m) | 0x4B000000u), __uint_as_float((g1 & m) | 0x4B000000u)),
                bc(s), bc(b));
}

// bin rows: swizzle that makes the 128-bit shared accesses conflict-free
__device__ __forceinline__ int bsw(int L) { return L ^ ((L >> 3) & 1); }

// E-W weights of cylinders 1..3 for one beam (cylinder 0 is the phase origin, weight 1).
struct EwW {
    float2 R[3], I[3], NI[3];
};

__device__ __forceinline__ void load_ew(const float2* __restrict__ ew, int table, int j, EwW& w) {
#pragma unroll
    for (int c = 1; c < kCyl; ++c) {
        const float2 v = ew[(table * kEw + j) * kCyl + c];
        w.R[c - 1] = bc(v.x);
        w.I[c - 1] = bc(v.y);
        w.NI[c - 1] = bc(-v.y);
    }
}

// E-W weights of beam j for frame F of a segment: the per-frame table of a
// tracking request, else the channel's static table.
__device__ __forceinline__ void load_ew_frame(const Seg& sg, const float2* __restrict__ ew, int F, int j, EwW& w) {
    if (sg.ew_frames) {
        load_ew(sg.ew_frames, F, j, w);
    } else {
        load_ew(ew, sg.table, j, w);
    }
}

// Twiddles of the first up-channel pass: [b / 2][c] = (Re, Re', Im, Im') of exp(-2 pi i b c / 128) for b
// and b + 1.  In constant memory: the FP32 form reads them by a warp-uniform index and so through
// uniform registers (1.3 % of a launch); the tensor-core forms, whose up-channel warps have a scheduler's
// slots to themselves less often, from a copy in shared memory (constant reads there cost 3 %).
struct PairTw {
    float4 w[kUp / 16][8];
};
constexpr double cos128(int e) {                         // cos(2 pi e / 128)
    constexpr double t[33] = {1.0, 0.99879545620517239271, 0.99518472667219688624, 0.98917650996478097345,
                              0.98078528040323044913, 0.97003125319454399260, 0.95694033573220886494,
                              0.94154406518302077841, 0.92387953251128675613, 0.90398929312344333159,
                              0.88192126434835502971, 0.85772861000027206990, 0.83146961230254523708,
                              0.80320753148064490981, 0.77301045336273696081, 0.74095112535495909118,
                              0.70710678118654752440, 0.67155895484701840063, 0.63439328416364549822,
                              0.59569930449243334347, 0.55557023301960222474, 0.51410274419322172659,
                              0.47139673682599764856, 0.42755509343028209432, 0.38268343236508977173,
                              0.33688985339222005069, 0.29028467725446236764, 0.24298017990326388995,
                              0.19509032201612826785, 0.14673047445536175166, 0.098017140329560601994,
                              0.049067674327418014255, 0.0};
    const int k = e & (kUp - 1), h = k > 64 ? 128 - k : k;
    return h > 32 ? -t[64 - h] : t[h];
}
constexpr PairTw make_pair_tw() {
    PairTw p{};
    for (int b = 0; b < kUp / 8; b += 2)
        for (int c = 0; c < 8; ++c) {
            p.w[b / 2][c].x = (float)cos128(b * c);
            p.w[b / 2][c].y = (float)cos128((b + 1) * c);
            p.w[b / 2][c].z = (float)-cos128(b * c - 32);
            p.w[b / 2][c].w = (float)-cos128((b + 1) * c - 32);
        }
    return p;
}
__constant__ PairTw kPairTw = make_pair_tw();

// ---------------------------------------------------------------------------
// tensor-memory access (tcgen05), one warp per 32-lane quarter
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_st4(uint32_t taddr, float a, float b, float c, float d) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 :: "r"(taddr), "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(__float_as_uint(c)),
                    "r"(__float_as_uint(d))
                 : "memory");
}

// 64 consecutive columns: two fine channels c, c+1 x 16 residues b, as SoA pairs
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, cp (&y)[16]) {
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
        "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
        "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
          "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
          "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
          "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int b = 0; b < 16; ++b) {
        y[b].re = make_float2(__uint_as_float(r[2 * b]), __uint_as_float(r[32 + 2 * b]));
        y[b].im = make_float2(__uint_as_float(r[2 * b + 1]), __uint_as_float(r[32 + 2 * b + 1]));
    }
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------
// mbarriers with bounded waits
// ---------------------------------------------------------------------------
constexpr unsigned long long kWaitNs = 2000000000ull;   // default bound on every mbarrier wait (2 s)

__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
    return ok != 0;
}

// Wait for the completion of phase `parity` of an mbarrier: false once `limit`
// ns have passed without it.  The timer is read only after a first test has failed, and then once in a
// number of tests: a read costs some hundred cycles, and the waits are on the path of every hand-off.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, unsigned long long limit) {
    if (mbar_try(mbar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 16; ++i)
            if (mbar_try(mbar, parity)) return true;
        if (globaltimer() - t0 > limit) return false;
    }
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mbar) : "memory");
}

// Segment of a work item, by halving: a scan from the first segment, each read of which is a trip to the
// constant cache, costs launches of 160 two-frame channels 4 %.
__device__ __forceinline__ int seg_of(const Batch& bt, int item) {
    int lo = 0, hi = bt.n_segs;
#pragma unroll 1
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (bt.segs[mid].item_begin <= item)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// Pass units (see PassUnits): item and pass range [ps0, ps1) of unit `un`.
__device__ __forceinline__ void pass_unit(const PassUnits& u, int un, int& item, int& ps0, int& ps1) {
    constexpr int kPasses = kTds * kPol;
    if (un < u.n_full) {
        item = un;
        ps0 = 0;
        ps1 = kPasses;
    } else {
        const int v = un - u.n_full, parts = kPasses / u.g;
        item = u.n_full + v / parts;
        ps0 = (v % parts) * u.g;
        ps1 = ps0 + u.g;
    }
}

// A thread of a split item has published the sums of n passes: true for the one that completes the
// six (all of them are then visible to it).  The token holds the launch's epoch and the passes
// counted so far, so a launch that was abandoned leaves nothing to clean up, and nothing waits.
__device__ __forceinline__ bool add_passes(unsigned long long* tok, unsigned long long epoch, unsigned n) {
    asm volatile("fence.acq_rel.gpu;" ::: "memory");    // the published sums before the token
    unsigned long long seen = *(volatile unsigned long long*)tok, next;
    for (;;) {
        next = ((seen >> 3) == epoch ? seen : epoch << 3) + n;
        const unsigned long long was = atomicCAS(tok, seen, next);
        if (was == seen) break;                        // else another part's thread has counted: try again
        seen = was;
    }
    if ((next & 7u) != (unsigned)(kTds * kPol)) return false;
    asm volatile("fence.acq_rel.gpu;" ::: "memory");    // the other parts' sums after their tokens
    return true;
}

// The published sums of an item's six passes for one beam (`in`: its place in pass 0).  All loads come
// before the caller's first store, which could alias them as far as the compiler knows: with
// stores in between, the adds of a one-frame request take 8 us longer.
__device__ __forceinline__ void load_passes(const float* in, float (&v)[kTds * kPol][kSub]) {
#pragma unroll
    for (int k = 0; k < kTds * kPol; ++k)
#pragma unroll
        for (int q = 0; q < kSub; ++q) v[k][q] = __ldcg(in + (size_t)k * (kSub * kNs) + q * kNs);
}

// CTA barrier that also orders tensor-memory accesses across it.
__device__ __forceinline__ void cta_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Second up-channel pass for one thread (TMEM lane, bin half hh): 16-point DFTs
// over the residue b for fine channels q = c + 8 d, two c at a time (SoA), then
// |.|^2 into the fftshifted sub-channels (d + 8) mod 16, the two fine channels of
// a SoA pair added first.  With `dump` set, the up-channelised voltages of bin m
// are written instead (fine channel q' order).
__device__ __forceinline__ void upchan_pass2(uint32_t tlane, int hh, float (&acc)[kSub], float2* dump) {
#pragma unroll 1
    for (int cpi = 0; cpi < 4; ++cpi) {
        cp y[16];
        tmem_ld64(tlane + hh * 256 + 64 * cpi, y);
        dft16(y);
        if (dump) {
#pragma unroll
            for (int dd = 0; dd < 16; ++dd) {
                const int c0 = 2 * cpi;
                dump[(c0 + 8 * dd + kUp / 2) & (kUp - 1)] = make_float2(y[dd].re.x, y[dd].im.x);
                dump[(c0 + 1 + 8 * dd + kUp / 2) & (kUp - 1)] = make_float2(y[dd].re.y, y[dd].im.y);
            }
        } else {
#pragma unroll
            for (int dd = 0; dd < 16; ++dd) {
                const float2 p = fma2(y[dd].im, y[dd].im, mul2(y[dd].re, y[dd].re));
                acc[(dd + 8) & 15] += p.x + p.y;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the tensor-core forms' accumulator layout: lane = bin, columns [0, 128) = Re X(t),
// [128, 256) = Im X(t) of block time t = 16 a + b
// ---------------------------------------------------------------------------
// TMEM access for the split Re/Im layout: 16 two-column loads (Re at base +
// 16 a + b0, Im at base + 128 + 16 a + b0, a = 0..7) -> SoA pairs (b0, b0 + 1).
__device__ __forceinline__ void tmem_ld_p1(uint32_t base, cp (&z)[8]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%2, %3}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%4, %5}, [%34];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%6, %7}, [%35];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8, %9}, [%36];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%10, %11}, [%37];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%12, %13}, [%38];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%14, %15}, [%39];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%16, %17}, [%40];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%18, %19}, [%41];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%20, %21}, [%42];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%22, %23}, [%43];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%24, %25}, [%44];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%26, %27}, [%45];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%28, %29}, [%46];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%30, %31}, [%47];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(base), "r"(base + 16), "r"(base + 32), "r"(base + 48), "r"(base + 64), "r"(base + 80),
          "r"(base + 96), "r"(base + 112), "r"(base + 128), "r"(base + 144), "r"(base + 160), "r"(base + 176),
          "r"(base + 192), "r"(base + 208), "r"(base + 224), "r"(base + 240)
        : "memory");
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        z[a].re = make_float2(__uint_as_float(r[2 * a]), __uint_as_float(r[2 * a + 1]));
        z[a].im = make_float2(__uint_as_float(r[16 + 2 * a]), __uint_as_float(r[16 + 2 * a + 1]));
    }
}

__device__ __forceinline__ void tmem_st2(uint32_t taddr, float a, float b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};"
                 :: "r"(taddr), "r"(__float_as_uint(a)), "r"(__float_as_uint(b)) : "memory");
}

// 32 consecutive columns -> 32 floats
__device__ __forceinline__ void tmem_ld32f(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// First up-channel pass in place on the split layout (t = 16 a + b): 8-point
// DFT over a for the residue pair (b0, b0 + 1), twiddled by exp(-2 pi i b c / 128).
__device__ __forceinline__ void upchan_pass1_split(uint32_t base, const float4* tw_s) {
#pragma unroll 1
    for (int bp = 0; bp < 8; ++bp) {
        const int b0 = 2 * bp;
        cp z[8];
        tmem_ld_p1(base + b0, z);
        dft8(z);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            if (c) {
                const float4 tw = tw_s[bp * 8 + c];
                z[c] = cmulp(z[c], make_float2(tw.x, tw.y), make_float2(tw.z, tw.w));
            }
            tmem_st2(base + 16 * c + b0, z[c].re.x, z[c].re.y);
            tmem_st2(base + 128 + 16 * c + b0, z[c].im.x, z[c].im.y);
        }
    }
}

// Second pass on the split layout: Re of (c, b) at 16 c + b, Im at 128 + 16 c + b.
__device__ __forceinline__ void upchan_pass2_split(uint32_t base, float2 (&acc)[kSub], float2* dump) {
#pragma unroll 1
    for (int cpi = 0; cpi < 4; ++cpi) {
        float re[32], im[32];
        tmem_ld32f(base + 32 * cpi, re);
        tmem_ld32f(base + 128 + 32 * cpi, im);
        cp y[16];
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            y[b].re = make_float2(re[b], re[16 + b]);
            y[b].im = make_float2(im[b], im[16 + b]);
        }
        dft16(y);
        if (dump) {
#pragma unroll
            for (int dd = 0; dd < 16; ++dd) {
                const int c0 = 2 * cpi;
                dump[(c0 + 8 * dd + kUp / 2) & (kUp - 1)] = make_float2(y[dd].re.x, y[dd].im.x);
                dump[(c0 + 1 + 8 * dd + kUp / 2) & (kUp - 1)] = make_float2(y[dd].re.y, y[dd].im.y);
            }
        } else {
#pragma unroll
            for (int dd = 0; dd < 16; ++dd) {
                const float2 p = fma2(y[dd].im, y[dd].im, mul2(y[dd].re, y[dd].re));
                acc[(dd + 8) & 15] = add2(acc[(dd + 8) & 15], p);
            }
        }
    }
}

}  // namespace
}  // namespace chimebf
