// Tensor-core forms of the fan-beam path for sm_103a (arXiv 1702.04728, Sec. 3 and 3.1).
//
// The N-S stage (zero-padded FFT kept at the 256 bins of Eq. 1) is evaluated as the equivalent
// dense DFT over the clamped rows on tcgen05:
//
//   X[m][t] = sum_n exp(-2 pi i n L(m) / 512) y_j[n][t],   m < 256, n < 256,
//
// with y_j the E-W phased feed line (Sec. 3) of block time t.  With C = cos, S = sin of
// 2 pi n L(m) / 512 and y = yr + i yi this is four real products,
//
//   Re X = C yr + S yi,   Im X = C yi - S yr,
//
// so one FP16 image of C and S and one copy of yr and yi serve both parts (the minus sign is the
// instruction's operand negation).  FP16 operands, FP32 accumulation; y is split y = hi + lo (22
// bits together) and the twiddles are hi, for three terms hi + lo.  Terms: 1 = T_hi y_hi,
// 2 = + T_hi y_lo, 3 = + T_lo y_hi.
//
// A cluster of two CTAs on neighbouring SMs owns a work item (channel segment, frame F, E-W beam j)
// and its six passes (3 blocks x 2 pols), one tcgen05 pair (cta_group::2, M = 256, N = 128, K = 16)
// per step:
//   * CTA r keeps the hi twiddles of bins 128 r .. 128 r + 127 for all feeds in shared memory
//     (128 KB), reloaded only when the item's channel changes;
//   * CTA r builds yr and yi of block times 64 r .. 64 r + 63 (unpack, E-W toward beam j, FP16), its
//     half of the pair's N = 128 columns; the tensor cores of both SMs read both halves, so nothing
//     is copied between the CTAs.  The lo twiddles of the 3-term form stream through the ring;
//   * the accumulator of a pass is 128 bins x (128 Re + 128 Im) columns per CTA, half of tensor
//     memory, so passes alternate between the halves and the MMAs of pass p + 1 overlap the
//     up-channel passes (Sec. 3.2) of pass p.
//
// Per CTA: warps 0-10 build (a task is 8 times of a 32-feed chunk, 8 feeds of one time per thread; the
// warps take the tasks in turn, with the next one's raw rows prefetched into registers), warp 11 loads
// the twiddles and, in the first CTA, issues the MMAs of the pair, warps 12-15 (one per tensor-memory
// lane quarter) run the up-channel passes and detection for one bin per thread.  16 warps is what the
// register file gives at 128 a thread; with 8 builders, one per group of 8 times, the loads and the
// arithmetic of two warps leave each scheduler idle for half of its cycles (10, 25 and 22 % slower with 1, 2
// and 3 terms).  Hand-offs are mbarriers only; every wait is bounded by %globaltimer, and on expiry
// the CTA records the failure, leaves its loops (the other CTA's waits then expire too) and waits for its
// copies and MMAs under way.
//
// Bound: the issue slots and the FP32 pipe that the builders' unpack and E-W arithmetic and the one
// up-channel warp of a scheduler share (61 % and 54 % of cycles for 1 term); the tensor pipe needs 512 x
// terms cycles of a chunk (3 terms: it and the shared-memory reads of its operands).  Per 4 x
// 49152-sample request on 152 SMs: 0.88 / 1.05 / 1.36 ms for 1 / 2 / 3 terms.
#include "device_common.cuh"

#include <cuda_fp16.h>

#include <cstdint>
#include <mutex>

namespace chimebf {
namespace {

// Operands are K-major without swizzle (twiddles: bf_internal.h): 8-row x 16-byte core matrices, k-groups
// (8 feeds) *LBO and 8-row groups *SBO bytes apart.
constexpr int kTNch = kFeed / kTFeeds;            // 8 chunks per pass
constexpr int kTGroups = 8;                       // build tasks of a chunk in a CTA (8 times x 32 feeds each)
constexpr int kTBuild = 11;                       // builder warps
constexpr int kTMma = kTBuild;                    // the MMA / twiddle warp
constexpr int kTUp = 4;                           // up-channel warps
constexpr int kTThreads = 32 * (kTBuild + 1 + kTUp);
// Register split (setmaxnreg, by warpgroup): builders and the MMA warp kTRegBuild, up-channel warps
// kTRegUp (104 and 200: 4 % slower with 1 term); the launcher checks that the launch gives
// enough (with fewer, the up-channel warps' increase could never be granted).
constexpr int kTRegBuild = 112, kTRegUp = 176;

template <int TERMS>
struct TcCfg {
    static constexpr bool A_LO = TERMS == 3, B_LO = TERMS >= 2;
    // data: yr and yi (hi, then lo) of a k-group side by side, 128 bytes each, and a pad that puts the
    // eight lanes of a 128-bit store (two times, four k-groups, see the builders) in distinct bank
    // groups; for three terms there is room for half of it, a store then takes two passes
    static constexpr int B_LBO = (B_LO ? 512 : 256) + (A_LO ? 16 : 32), B_SBO = kTFeeds / 8 * B_LBO;
    static constexpr int B_STAGE = kTGroups * B_SBO;                   // 64 times
    static constexpr int STAGE = B_STAGE + (A_LO ? 2 * kTTw : 0);      // and the chunk's lo twiddles
    static constexpr int NB = TERMS == 1 ? 6 : TERMS == 2 ? 5 : 3;     // ring stages
    // arrivals on "stage full" in the first CTA: the build tasks of both CTAs (one of the first CTA's also
    // for its lo twiddles); 3 terms: the second CTA's lo twiddles
    static constexpr int FULL = 2 * kTGroups + (A_LO ? 1 : 0);
    static constexpr int BARS = 3 * NB + 7;
    static constexpr size_t SM_A = (size_t)kTNch * 2 * kTTw;           // 128 KB
    static constexpr size_t SM_RING = (size_t)NB * STAGE;
    static constexpr size_t SM_TW = sizeof(PairTw);
    static constexpr size_t SMEM = SM_A + SM_RING + SM_TW + 8 * BARS;
    static_assert(SMEM + 128 <= 227 * 1024, "dynamic and static shared memory");
};

// instruction descriptor: kind::f16, A = B = F16, D = F32, both K-major, M = 256 (the pair), N = 128;
// bit 13 negates A
constexpr uint32_t kTIdesc = (1u << 4) | ((128u >> 3) << 17) | ((256u >> 4) << 24);
constexpr uint32_t kTIdescNeg = kTIdesc | (1u << 13);

// Shared-memory matrix descriptor (no swizzle, version 1): the address field is the low bits of the low
// word, so an operand x bytes on has the low word + x / 16 (shared memory stays below 2^18 bytes).
struct Desc {
    uint32_t lo, hi;
};
__device__ __forceinline__ Desc tdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return {(saddr >> 4) | (lbo >> 4) << 16, (sbo >> 4) | 1u << 14};
}

// One MMA of the pair, issued by the lane with `leader` set; the whole warp runs the code around it, so
// that descriptors stay in uniform registers.
__device__ __forceinline__ void tmma(uint32_t leader, uint32_t dtmem, uint32_t alo, uint32_t ahi, uint32_t blo,
                                     uint32_t bhi, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
        "setp.ne.b32 p, %7, 0;\n\t"
        "setp.ne.b32 q, %0, 0;\n\t"
        "mov.b64 a, {%2, %3};\n\t"
        "mov.b64 b, {%4, %5};\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%1], a, b, %6, p;\n\t}"
        :: "r"(leader), "r"(dtmem), "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accum)
        : "memory");
}

// commit of the leader's outstanding MMAs to the same mbarrier in both CTAs
__device__ __forceinline__ void tcommit(uint32_t leader, uint32_t mbar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%1], %2;\n\t}"
        :: "r"(leader), "r"(mbar), "h"((uint16_t)3) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_id() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t n_clusters() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
    return r;
}
// address in CTA `cta` of the cluster of a local shared-memory address
__device__ __forceinline__ uint32_t cta_addr(uint32_t a, uint32_t cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrival on an mbarrier of any CTA of the cluster (shared::cluster address).  What it announces was
// written for the asynchronous proxy (fence.proxy.async) or to tensor memory (tcgen05.fence), so no
// cluster-wide release of other memory is needed; one here is a memory barrier and an L1 invalidation per
// chunk, 40 % of the time of a 1-term launch.
__device__ __forceinline__ void arrive_cluster(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(mbar) : "memory");
}
__device__ __forceinline__ void expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}
// bulk copy global -> this CTA's shared memory
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
__device__ __forceinline__ uint32_t h2(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float2 unh2(uint32_t u) { return __half22float2(*reinterpret_cast<const __half2*>(&u)); }

struct RawT {
    uint4 v[kCyl];
};
// the thread's 8 feeds x 2 pols of every cylinder at chunk kc (p: its row at feed octet 0 of chunk 0)
__device__ __forceinline__ void load_raw(const uint8_t* p, int kc, RawT& r) {
#pragma unroll
    for (int c = 0; c < kCyl; ++c)
        r.v[c] = __ldg(reinterpret_cast<const uint4*>(p + kc * (kTFeeds * kPol) + c * (kFeed * kPol)));
}

// One task: unpack 8 feeds of one time, E-W toward beam j in FP32, FP16 hi (+ lo) of yr and yi; dst is
// the task's 16-byte place in yr, yi 128 bytes on, lo 256.
template <int TERMS>
__device__ __forceinline__ void build(const RawT& raw, const PolSel& ps, const EwW& w, unsigned char* dst) {
    uint32_t vr[4], vi[4], lr[4], li[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {                        // feeds 2k, 2k + 1 as a SoA pair
        cp y;
#pragma unroll
        for (int c = 0; c < kCyl; ++c) {
            const uint32_t g = k == 0 ? raw.v[c].x : k == 1 ? raw.v[c].y : k == 2 ? raw.v[c].z : raw.v[c].w;
            const uint32_t h = g >> 16;
            const float2 xi = nibm(g, h, ps.mi, ps.si, ps.bi), xr = nibm(g, h, ps.mr, ps.sr, ps.br);
            if (c == 0) {
                y = {xr, xi};
            } else {
                y.re = fma2(xi, w.NI[c - 1], fma2(xr, w.R[c - 1], y.re));
                y.im = fma2(xr, w.I[c - 1], fma2(xi, w.R[c - 1], y.im));
            }
        }
        vr[k] = h2(y.re.x, y.re.y);
        vi[k] = h2(y.im.x, y.im.y);
        if constexpr (TERMS >= 2) {
            const float2 br = unh2(vr[k]), bi = unh2(vi[k]);
            lr[k] = h2(y.re.x - br.x, y.re.y - br.y);
            li[k] = h2(y.im.x - bi.x, y.im.y - bi.y);
        }
    }
    *reinterpret_cast<uint4*>(dst) = make_uint4(vr[0], vr[1], vr[2], vr[3]);
    *reinterpret_cast<uint4*>(dst + 128) = make_uint4(vi[0], vi[1], vi[2], vi[3]);
    if constexpr (TERMS >= 2) {
        *reinterpret_cast<uint4*>(dst + 256) = make_uint4(lr[0], lr[1], lr[2], lr[3]);
        *reinterpret_cast<uint4*>(dst + 384) = make_uint4(li[0], li[1], li[2], li[3]);
    }
}

// MODE: 0 = detect and integrate, 1 = dump up-channelised voltages, 2 = dump the N-S/E-W beams of
//       the GEMM, 3 = stall check (the MMA warps or the builders stop after bt.stall_chunks chunks, so
//       the other warps' waits run out against the launch's bound).
template <int TERMS, int MODE>
__global__ void __launch_bounds__(kTThreads, 1) fused_tc_kernel(const __grid_constant__ Batch bt) {
    using C = TcCfg<TERMS>;
    constexpr int NB = C::NB;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, passes_s;      // passes_s: passes that the first up-channel warp has read
    __shared__ uint32_t lo_last_s[NB];     // 3 terms: phase of lofull that the stage's last copy completes
    unsigned char* ring = smem + C::SM_A;
    float4* tw_s = reinterpret_cast<float4*>(ring + C::SM_RING);
    uint64_t* mbar_s = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(tw_s) + C::SM_TW);

    // the warp number in a uniform register: the roles' branches are then uniform too, without which the nested
    // ones cost the tensor-core forms 12, 15 and 17 % (1, 2 and 3 terms)
    const int tid = threadIdx.x, warp = (int)uniform((uint32_t)tid >> 5), lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const uint32_t smem0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    const uint32_t bar0 = static_cast<uint32_t>(__cvta_generic_to_shared(&mbar_s[0]));
    auto bfull = [&](int s) { return bar0 + 8u * (uint32_t)s; };               // first CTA: stage s of both CTAs
    auto bempty = [&](int s) { return bar0 + 8u * (uint32_t)(NB + s); };       // MMA commit
    auto lofull = [&](int s) { return bar0 + 8u * (uint32_t)(2 * NB + s); };   // this CTA's lo twiddles
    auto accfull = [&](int b) { return bar0 + 8u * (uint32_t)(3 * NB + b); };  // last commit of a pass
    auto tfree = [&](int b) { return bar0 + 8u * (uint32_t)(3 * NB + 2 + b); };    // first CTA: both CTAs' up-channel warps
    const uint32_t afull = bar0 + 8u * (uint32_t)(3 * NB + 4);                 // this CTA's resident twiddles
    const uint32_t aother = afull + 8u, adone = afull + 16u;

    if (warp == 0) {
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(&tmem_base_s));
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" :: "r"(dst) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        auto init = [](uint32_t b, uint32_t n) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(b), "r"(n) : "memory");
        };
        for (int i = 0; i < NB; ++i) {
            init(bfull(i), C::FULL);
            init(bempty(i), 1);
            init(lofull(i), 1);
            lo_last_s[i] = 1;              // a fresh barrier passes a wait on parity 1
        }
        for (int i = 0; i < 2; ++i) {
            init(accfull(i), 1);
            init(tfree(i), 2 * kTUp);
        }
        init(afull, 1);
        init(aother, 1);
        init(adone, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_s = passes_s = 0;
    }
    for (int i = tid; i < 64; i += kTThreads) tw_s[i] = kPairTw.w[i >> 3][i & 7];
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();                        // both CTAs' barriers exist before any remote arrival
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_s;
    const unsigned long long wlim = bt.wait_ns ? bt.wait_ns : kWaitNs;
    const int pair = (int)cluster_id(), npairs = (int)n_clusters();
    const PassUnits units = bt.units;

    static_assert((kTBuild + 1) % 4 == 0 && kTUp % 4 == 0, "the register split is by warpgroup");
    if (warp <= kTMma) {
        // one setmaxnreg for all warps of a warpgroup, as the instruction requires: builders 8-10 share the MMA
        // warp's.  (In branches that do not hold the warps' code the compiler keeps all of it to the launch's
        // count and spills.)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kTRegBuild) : "memory");
        if (warp == kTMma) {
            // ------------------------------ twiddle loads and MMAs ------------------------------
            // The whole warp runs this and the leader lane issues: in a branch of one lane every descriptor
            // would be computed in vector registers and moved over (3 % of the 1- and 2-term forms).
            const int stall_at = MODE == 3 && bt.stall_mma ? bt.stall_chunks : -1;
            if (stall_at != 0) {
                const uint32_t leader = lane == 0;
                uint32_t p_bfull = 0, p_tfree = 0, p_a = 0, p_lo = 0;
                const unsigned char* a_cur = nullptr;
                uint32_t s = 0, pass = 0;
                uint32_t a_last = 1;               // phase that the last load of resident twiddles completes
                bool ok = true, stalled = false;
                int chunks = 0;
                // a wait of the whole warp
                auto wait = [&](uint32_t bar, uint32_t parity) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, wlim)) && ok;
                };
                // A wait for all MMAs issued so far.  The second CTA's warp comes here while the first has many
                // passes to go, so the bound is on each pass.
                auto wait_mma = [&](uint32_t parity) {
                    bool done;
                    int seen;
                    do {
                        seen = *(volatile int*)&passes_s;
                        done = __all_sync(0xffffffffu, mbar_wait(adone, parity, wlim));
                    } while (!done && __any_sync(0xffffffffu, *(volatile int*)&passes_s != seen));
                    ok = done && ok;
                };
                const Desc da = tdesc(smem0, kTALbo, kTASbo), db = tdesc(smem0 + (uint32_t)C::SM_A, C::B_LBO, C::B_SBO);
                const Desc dl = tdesc(smem0 + (uint32_t)C::SM_A + C::B_STAGE, kTALbo, kTASbo);    // lo twiddles
                int seg_cursor = 0;
                for (int un = pair; un < units.n_units && ok; un += npairs) {
                    int item, ps0, ps1;
                    pass_unit(units, un, item, ps0, ps1);
                    while (seg_cursor + 1 < bt.n_segs && bt.segs[seg_cursor + 1].item_begin <= item) ++seg_cursor;
                    const unsigned char* a_img = bt.segs[seg_cursor].a_img;
                    if (a_img != a_cur) {
                        if (a_cur) {
                            // the MMAs that read the old twiddles are complete before they are replaced
                            if (rank == 0) tcommit(leader, adone);
                            wait_mma((p_a >> 1) & 1u);
                            p_a ^= 2u;
                        }
                        a_last = p_a & 1u;
                        if (leader) {
                            expect_tx(afull, (uint32_t)C::SM_A);
#pragma unroll 1
                            for (int kc = 0; kc < kTNch; ++kc)
                                bulk_g2s(smem0 + (uint32_t)(kc * 2 * kTTw), a_img + (size_t)(kc * 2 + (int)rank) * (2 * kTTw),
                                         2 * kTTw, afull);
                        }
                        __syncwarp();
                        wait(afull, p_a & 1u);
                        if (rank == 1) {
                            if (leader) arrive_cluster(cta_addr(aother, 0));
                            __syncwarp();
                        } else {
                            wait(aother, p_a & 1u);
                        }
                        p_a ^= 1u;
                        a_cur = a_img;
                    }
                    for (int ps = ps0; ps < ps1 && ok; ++ps, ++pass) {
                        if (rank == 1) {
                            if constexpr (C::A_LO) {
#pragma unroll 1
                                for (int kc = 0; kc < kTNch && ok; ++kc) {
                                    // this CTA's lo twiddles of the stage have landed
                                    wait(lofull((int)s), (p_lo >> s) & 1u);
                                    p_lo ^= 1u << s;
                                    if (ok && leader) arrive_cluster(cta_addr(bfull((int)s), 0));
                                    __syncwarp();
                                    if (++s == (uint32_t)NB) s = 0;
                                }
                                if (__any_sync(0xffffffffu, *(volatile int*)&abort_s != 0)) ok = false;
                            }
                            continue;
                        }
                        const uint32_t buf = pass & 1u;
                        if (pass >= 2) {
                            // the up-channel warps of both CTAs have read this accumulator half (pass - 2)
                            wait(tfree((int)buf), (p_tfree >> buf) & 1u);
                            p_tfree ^= 1u << buf;
                        }
                        const uint32_t re = tmem + 256u * buf, im = re + 128u;
#pragma unroll 1
                        for (int kc = 0; kc < kTNch && ok; ++kc) {
                            if constexpr (MODE == 3) {
                                if (chunks++ == stall_at) {
                                    stalled = true;
                                    ok = false;
                                    break;
                                }
                            }
                            wait(bfull((int)s), (p_bfull >> s) & 1u);
                            p_bfull ^= 1u << s;
                            if (!ok) break;
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint32_t a0 = da.lo + (uint32_t)kc * (2 * kTTw / 16), b0 = db.lo + s * (C::STAGE / 16u);
                            const uint32_t l0 = dl.lo + s * (C::STAGE / 16u);
#pragma unroll
                            for (int ks = 0; ks < kTFeeds / 16; ++ks) {
                                const uint32_t c = a0 + ks * (2 * kTALbo / 16), sn = c + kTTw / 16;
                                const uint32_t yr = b0 + ks * (2 * C::B_LBO / 16), yi = yr + 128 / 16;
                                const uint32_t more = (kc | ks) ? 1u : 0u;
                                tmma(leader, re, c, da.hi, yr, db.hi, kTIdesc, more);
                                tmma(leader, im, c, da.hi, yi, db.hi, kTIdesc, more);
                                tmma(leader, re, sn, da.hi, yi, db.hi, kTIdesc, 1u);
                                tmma(leader, im, sn, da.hi, yr, db.hi, kTIdescNeg, 1u);
                                if constexpr (C::B_LO) {
                                    const uint32_t zr = yr + 256 / 16, zi = yr + 384 / 16;
                                    tmma(leader, re, c, da.hi, zr, db.hi, kTIdesc, 1u);
                                    tmma(leader, im, c, da.hi, zi, db.hi, kTIdesc, 1u);
                                    tmma(leader, re, sn, da.hi, zi, db.hi, kTIdesc, 1u);
                                    tmma(leader, im, sn, da.hi, zr, db.hi, kTIdescNeg, 1u);
                                }
                                if constexpr (C::A_LO) {
                                    const uint32_t cl = l0 + ks * (2 * kTALbo / 16), sl = cl + kTTw / 16;
                                    tmma(leader, re, cl, da.hi, yr, db.hi, kTIdesc, 1u);
                                    tmma(leader, im, cl, da.hi, yi, db.hi, kTIdesc, 1u);
                                    tmma(leader, re, sl, da.hi, yi, db.hi, kTIdesc, 1u);
                                    tmma(leader, im, sl, da.hi, yr, db.hi, kTIdescNeg, 1u);
                                }
                            }
                            tcommit(leader, bempty((int)s));
                            if (kc == kTNch - 1) tcommit(leader, accfull((int)buf));
                            if (++s == (uint32_t)NB) s = 0;
                        }
                        if (__any_sync(0xffffffffu, *(volatile int*)&abort_s != 0)) ok = false;
                    }
                }
                // every issued MMA and load is complete before shared and tensor memory are released
                if (rank == 0) tcommit(leader, adone);
                wait_mma((p_a >> 1) & 1u);
                wait(afull, a_last);
                if (!ok && !stalled) abort_s = 1;
            }
        } else {
            // ------------------------------ builders ------------------------------
            // The warps take the CTA's tasks (unit, pass, chunk, group of 8 times) in turn.  Lane bits 0-1 take
            // the four feed octets of a chunk, bits 2-4 eight times: a quarter warp loads 64 contiguous bytes
            // of two rows (lanes on eight different lines at one offset take a pass of the L1 data banks each, 11 %
            // of the time of a 1-term launch)
            const int t = 64 * (int)rank + (lane >> 2), oct = lane & 3;
            unsigned char* dst0 = ring + oct * C::B_LBO + (lane >> 2) * 16;
            const uint32_t full0 = cta_addr(bar0, 0);                      // the first CTA's bfull(0)
            // the next task, whose rows are loaded while the current one is built
            int un = pair, ps = 0, ps1 = 0, kc = warp / kTGroups, g = warp % kTGroups, sgi = 0, F = 0, j = 0;
            bool more = un < units.n_units, new_unit = true, new_pass = true;
            auto enter_unit = [&] {
                int item;
                pass_unit(units, un, item, ps, ps1);
                while (sgi + 1 < bt.n_segs && bt.segs[sgi + 1].item_begin <= item) ++sgi;
                const int local = item - bt.segs[sgi].item_begin;
                F = local >> 2;
                j = local & 3;
            };
            // this thread's part of the rows of a block in the carried and in the new samples, and the first
            // of its rows that is new
            const uint8_t *carried = nullptr, *fresh = nullptr;
            int first_fresh = 0;
            auto enter_block = [&] {
                const Seg& sg = bt.segs[sgi];
                const long long row0 = (long long)F * kFrame + (ps >> 1) * kUp;
                const long long left = sg.carry_rows - row0;
                first_fresh = left < 0 ? 0 : left < kUp ? (int)left : kUp;
                carried = sg.carry + row0 * kInput + 16 * oct;
                fresh = sg.vin - left * kInput + 16 * oct;
            };
            auto load_task = [&](RawT& r) {
                const int row = t + 8 * g;
                load_raw((row < first_fresh ? carried : fresh) + (uint32_t)(row * kInput), kc, r);
            };
            uint32_t s = (uint32_t)(warp / kTGroups), parity = 1;             // a fresh barrier passes a wait on parity 1
            // A wait for a stage's previous use must not pass on the use before that one.  The warp's previous task
            // saw the release of the stage NB chunks before it, and commits are in order, so that use is over
            // if the warp advances by at most NB chunks at a time.
            static_assert((kTBuild + kTGroups - 1) / kTGroups <= C::NB, "a builder's step between tasks");
            bool ok = true;
            int chunks = warp / kTGroups;                               // of the task at hand, from the launch's first
            const int stall_at = MODE == 3 && !bt.stall_mma ? bt.stall_chunks : -1;
            EwW w;
            PolSel sel;
            // builds the task whose rows are in cur and loads the one after it
            auto task = [&](const RawT& cur, RawT& nxt) {
                if (new_pass) {
                    if (new_unit) load_ew_frame(bt.segs[sgi], bt.ew, F, j, w);
                    sel = pol_sel(ps & 1);
                    if (__any_sync(0xffffffffu, *(volatile int*)&abort_s != 0)) ok = false;   // the warp stops as one
                }
                const int g0 = g, kc0 = kc, sg0 = sgi;
                new_unit = new_pass = false;
                uint32_t ds = kTBuild / kTGroups;
                g += kTBuild % kTGroups;
                if (g >= kTGroups) {
                    g -= kTGroups;
                    ++ds;
                }
                kc += (int)ds;
                if (kc >= kTNch) {
                    kc -= kTNch;
                    new_pass = true;
                    if (++ps == ps1) {
                        un += npairs;
                        new_unit = true;
                        more = un < units.n_units;
                        if (more) enter_unit();
                    }
                    if (more) enter_block();
                }
                if (more) load_task(nxt);
                // the MMAs have read stage s in both CTAs
                if (!mbar_wait(bempty((int)s), parity, wlim)) ok = false;
                // the warp stops as one (a wait expired in any lane)
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    return;
                }
                if constexpr (C::A_LO) {
                    if (g0 == 0 && lane == 0) {
                        // the chunk's lo twiddles (second half of the image) into the stage
                        const uint32_t bar = lofull((int)s);
                        *(volatile uint32_t*)&lo_last_s[s] = parity ^ 1u;
                        expect_tx(bar, 2 * kTTw);
                        bulk_g2s(smem0 + (uint32_t)C::SM_A + s * (uint32_t)C::STAGE + (uint32_t)C::B_STAGE,
                                 bt.segs[sg0].a_img + 2 * C::SM_A + (size_t)(kc0 * 2 + (int)rank) * (2 * kTTw), 2 * kTTw, bar);
                    }
                }
                build<TERMS>(cur, sel, w, dst0 + s * (uint32_t)C::STAGE + g0 * C::B_SBO);
                if constexpr (C::A_LO) {
                    // in the first CTA the task that requested the chunk's lo twiddles stands for them too (a barrier more
                    // for the MMA warp to test between two chunks' MMAs costs 2 %, the second CTA's done like this 1 %)
                    if (rank == 0 && g0 == 0 && !__all_sync(0xffffffffu, mbar_wait(lofull((int)s), parity ^ 1u, wlim))) {
                        ok = false;
                        return;
                    }
                }
                // the generic-proxy stores are visible to the tensor cores
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive_cluster(full0 + 8u * s);
                s += ds;
                if constexpr (MODE == 3) chunks += (int)ds;
                if (s >= (uint32_t)C::NB) {
                    s -= (uint32_t)C::NB;
                    parity ^= 1u;
                }
            };
            // two tasks per loop body: the raw rows alternate between registers without copies
            RawT ra, rb;
            if (more) {
                enter_unit();
                enter_block();
                load_task(ra);
            }
            while (more && ok) {
                if (MODE == 3 && stall_at >= 0 && chunks >= stall_at) break;
                task(ra, rb);
                if (!more || !ok) break;
                if (MODE == 3 && stall_at >= 0 && chunks >= stall_at) break;
                task(rb, ra);
            }
            if (!ok) abort_s = 1;
        }
    } else {
        // ------------------------------ up-channel warps ------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(kTRegUp) : "memory");
        const int q4 = warp & 3;                                     // tensor-memory lane quarter
        const int ell = 32 * q4 + lane, m = 128 * (int)rank + ell;   // this thread's bin
        const uint32_t free0 = cta_addr(tfree(0), 0);
        uint32_t p_acc = 0, pass = 0;
        bool ok = true;
        int sgi = 0;
        for (int un = pair; un < units.n_units && ok; un += npairs) {
            int item, ps0, ps1;
            pass_unit(units, un, item, ps0, ps1);
            while (sgi + 1 < bt.n_segs && bt.segs[sgi + 1].item_begin <= item) ++sgi;
            const Seg& sg = bt.segs[sgi];
            const int local = item - sg.item_begin;
            const int F = local >> 2, j = local & 3;
            const bool whole = ps1 - ps0 == kTds * kPol;
            // sums of the item's passes of each polarisation
            float acc0[kSub], acc1[kSub];
#pragma unroll
            for (int q = 0; q < kSub; ++q) acc0[q] = acc1[q] = 0.f;
            for (int ps = ps0; ps < ps1 && ok; ++ps, ++pass) {
                const uint32_t buf = pass & 1u;
                const uint32_t base = tmem + (static_cast<uint32_t>(32 * q4) << 16) + 256u * buf;
                if (!mbar_wait(accfull((int)buf), (p_acc >> buf) & 1u, wlim)) ok = false;
                p_acc ^= 1u << buf;
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                float2 pw[kSub];
#pragma unroll
                for (int q = 0; q < kSub; ++q) pw[q] = make_float2(0.f, 0.f);
                float2* dump = MODE == 1 || MODE == 2
                                   ? bt.dump + ((((long long)(F * kTds + (ps >> 1)) * kPol + (ps & 1)) * kEw + j) * kNs + m) * kUp
                                   : nullptr;
                if constexpr (MODE == 2) {
                    for (int c4 = 0; c4 < 4; ++c4) {
                        float re[32], im[32];
                        tmem_ld32f(base + 32 * c4, re);
                        tmem_ld32f(base + 128 + 32 * c4, im);
                        for (int b = 0; b < 32; ++b) dump[32 * c4 + b] = make_float2(re[b], im[b]);
                    }
                } else {
                    upchan_pass1_split(base, tw_s);
                    tmem_wait_st();
                    upchan_pass2_split(base, pw, MODE == 1 ? dump : nullptr);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive_cluster(free0 + 8u * buf);
                if (tid == 32 * (kTMma + 1)) *(volatile int*)&passes_s = (int)pass + 1;
                if constexpr (MODE == 0) {
                    if (whole) {
#pragma unroll
                        for (int q = 0; q < kSub; ++q) {
                            const float v = pw[q].x + pw[q].y;
                            if (ps & 1)
                                acc1[q] += v;
                            else
                                acc0[q] += v;
                        }
                    } else {
                        // part of an item: publish the pass; the thread that completes the six adds them
                        const int slot = item - units.n_full;
                        float* o = bt.part + ((size_t)slot * (kTds * kPol) + ps) * (kSub * kNs) + m;
#pragma unroll
                        for (int q = 0; q < kSub; ++q) o[q * kNs] = pw[q].x + pw[q].y;
                        if (add_passes(bt.part_tok + (size_t)slot * kNs + m, bt.epoch, 1)) {
                            float v[kTds * kPol][kSub];
                            load_passes(bt.part + (size_t)slot * (kTds * kPol) * (kSub * kNs) + m, v);
                            float* out = sg.out + (long long)(kNs * j + m) * sg.beam_stride + F;
#pragma unroll
                            for (int q = 0; q < kSub; ++q)
                                out[(long long)q * sg.sub_stride] = ((v[0][q] + v[2][q]) + v[4][q]) + ((v[1][q] + v[3][q]) + v[5][q]);
                        }
                    }
                }
                if (__any_sync(0xffffffffu, *(volatile int*)&abort_s != 0)) ok = false;   // the warp stops as one
            }
            if constexpr (MODE == 0) {
                if (whole && ok) {
                    float* out = sg.out + (long long)(kNs * j + m) * sg.beam_stride + F;
#pragma unroll
                    for (int q = 0; q < kSub; ++q) out[(long long)q * sg.sub_stride] = acc0[q] + acc1[q];
                }
            }
        }
        if (!ok) abort_s = 1;
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (C::A_LO) {
        // no builder issues any more; copies under way when a wait ran out have to land before this memory is
        // given up (after a run that completed there are none)
        if (tid < NB) mbar_wait(lofull(tid), lo_last_s[tid], wlim);
        __syncwarp();
    }
    // both CTAs are done with each other's barriers and, in a run that completed, with the MMAs
    cluster_sync();
    if (abort_s && tid == 0 && bt.status) atomicExch(bt.status, 1);
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" :: "r"(tmem) : "memory");
    }
}

// Once per device and kernel: the register split must fit in what the kernel was launched with
// (else the up-channel warps' increase could never be granted: such a build is refused), and the
// shared-memory size is set.
template <int TERMS, int MODE>
cudaError_t launch_tc(const Batch& b, int pairs, cudaStream_t s) {
    if (b.n_items <= 0) return cudaSuccess;
    if (pairs < 1 || (b.units.g < kTds * kPol && (!b.part || !b.part_tok))) return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    static std::once_flag once[kMaxDevices];
    static cudaError_t result[kMaxDevices];
    std::call_once(once[dev], [&] {
        cudaFuncAttributes fa;
        cudaError_t r = cudaFuncGetAttributes(&fa, fused_tc_kernel<TERMS, MODE>);
        if (r == cudaSuccess && (kTBuild + 1) * kTRegBuild + kTUp * kTRegUp > kTThreads / 32 * fa.numRegs) r = cudaErrorInvalidConfiguration;
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(fused_tc_kernel<TERMS, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)TcCfg<TERMS>::SMEM);
        result[dev] = r;
    });
    if (result[dev] != cudaSuccess) return result[dev];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    cfg.blockDim = dim3(kTThreads);
    cfg.dynamicSmemBytes = TcCfg<TERMS>::SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, fused_tc_kernel<TERMS, MODE>, b);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace

cudaError_t fused_tc_launch(const Batch& b, int terms, int mode, int pairs, cudaStream_t s) {
    switch (terms * 10 + mode) {
        case 10: return launch_tc<1, 0>(b, pairs, s);
        case 11: return launch_tc<1, 1>(b, pairs, s);
        case 12: return launch_tc<1, 2>(b, pairs, s);
        case 13: return launch_tc<1, 3>(b, pairs, s);
        case 20: return launch_tc<2, 0>(b, pairs, s);
        case 21: return launch_tc<2, 1>(b, pairs, s);
        case 22: return launch_tc<2, 2>(b, pairs, s);
        case 23: return launch_tc<2, 3>(b, pairs, s);
        case 30: return launch_tc<3, 0>(b, pairs, s);
        case 31: return launch_tc<3, 1>(b, pairs, s);
        case 32: return launch_tc<3, 2>(b, pairs, s);
        case 33: return launch_tc<3, 3>(b, pairs, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace chimebf
