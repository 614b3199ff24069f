// Fused FP32 fan-beam kernel for sm_103a (arXiv 1702.04728, Sec. 3).
//
// One CTA of 12 warps per SM owns a work item = (channel segment, output
// frame F, E-W beam j) and runs six passes over it, one per (128-sample
// block, polarisation).  Arithmetic is packed FP32x2 (FFMA2 / FADD2) in
// structure-of-arrays form: every value is a pair of two time samples (or two
// fine channels) that go through identical operations.
//
//  phase A, warps 0-7 in two teams of four; a team's iteration is 16 time samples
//    * a warp takes two row pairs (four time rows, staged in shared memory by
//      cp.async) and loads them with transposing ldmatrix, so that lane (n2, row
//      pair) receives the bytes of feeds 16 n1 + n2 for all 16 n1 of every
//      cylinder, both rows and both polarisations of a feed in one word; it
//      unpacks the 4+4-bit nibbles (Table 1) exactly and forms E-W beam j
//      (Sec. 3) in registers -- applied before the N-S transform, legal because
//      both are linear and the phases do not depend on the feed;
//    * the zero-padded 512-point N-S FFT (Sec. 3.1) is 32 x 16: every lane runs
//      the DFT32 over n1 of its 16 values (two DFT16, the odd bins' twiddles at
//      compile time), one shared-memory transpose, then the twiddles
//      exp(-2 pi i n2 k / 512) and a DFT16 over n2; all 512 bins of a row pair
//      land in its row of the team's bin buffer;
//  gather + first up-channel pass, warps 8-11 (thread = N-S beams m, m + 128)
//    * bin L(m) of the clamp table (Eq. 1) is picked from the 8 rows of each
//      time residue pair, an 8-point DFT runs in registers, and the twiddled
//      result is parked in tensor memory (TMEM);
//  second up-channel pass (after the 128 samples of the block)
//    * 16-point DFTs from TMEM complete the 128-point FFT (Sec. 3.2), then
//      |.|^2 is accumulated into the 16 fftshifted sub-channels (Sec. 3).
//
// The corner turn of the paper's second kernel (time-slowest to
// time-fastest) is the gather into TMEM lanes: one (beam j, pol, block) is
// 256 beams x 128 samples x 8 B = 256 KB = all of TMEM.  Only packed input
// and float output touch global memory.
#include "device_common.cuh"

#include <cstdint>
#include <mutex>

namespace chimebf {
namespace {

constexpr int kWarps = 8;                   // phase-A (producer) warps: two teams of four
constexpr int kTeam = 4;                    // team q takes the iterations it = q mod 2, warp w of it row pairs 2w, 2w + 1
constexpr int kCons = 4;                    // gather / up-channel (consumer) warps, one per TMEM lane quarter
constexpr int kThreads = 32 * (kWarps + kCons);

// named barriers: 0 = whole CTA; FULL of bin buffer b (one team and the consumers); consumers
// only.  The release of a bin buffer (EMPTY) is an mbarrier the consumer warps arrive on, so
// producer warps wait for the consumers without waiting for each other.
constexpr int kBarFull = 1, kBarCons = 3;
constexpr int kFullThreads = 32 * (kTeam + kCons);

// Register split (setmaxnreg): the launch gives every warp kRegLaunch registers per
// thread; the producer warpgroups (warps 0-7) raise theirs to kRegProd and the
// consumer warpgroup (warps 8-11) lowers its to kRegCons, within the same total.
constexpr int kRegLaunch = 168, kRegProd = 176, kRegCons = 152;
static_assert(kWarps * kRegProd + kCons * kRegCons <= (kWarps + kCons) * kRegLaunch,
              "the register split must fit in the launch's register file share");

// shared memory (a bin is one SoA pair of 16 bytes: re0, re1, im0, im1)
constexpr int kRows = 8;                             // row pairs of a bin buffer (16 time samples)
constexpr int kBinsF4 = kRows * kBins;               // 8 row pairs x 512 bins (one of two buffers)
constexpr int kRowB = kBins * 16;                    // bytes of a row pair's bins, before that of its transpose
constexpr int kRawRow = kInput + 32;                 // raw row stride: four rows in distinct bank groups
constexpr int kRawB = 4 * kRawRow;                   // per producer warp: its two row pairs
constexpr size_t kSmemBins = 2 * (size_t)kBinsF4 * 16;   // one buffer per team
constexpr size_t kSmemRaw = (size_t)kWarps * kRawB;      // raw rows (cp.async), one iteration ahead
constexpr size_t kSmemLut = 2 * kNs * sizeof(int);   // bins and beams in gather order
constexpr size_t kSmemTwl = kLaneTwLen * sizeof(float2);           // exp(-2 pi i n2 k / 512), [8][32 k] x 2 n2
constexpr size_t kSmemPark = (size_t)kSub * kNs * sizeof(float);   // first half of the current item
constexpr size_t kSmemTotal = kSmemBins + kSmemRaw + kSmemLut + kSmemTwl + kSmemPark;

__device__ __forceinline__ uint32_t smem_sa(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 128-bit shared-memory access by 32-bit shared address.  The XOR swizzles
// below become one LOP3 with an immediate per access on top of a per-lane base.
__device__ __forceinline__ void sts_cp(uint32_t addr, cp a) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                 :: "r"(addr), "f"(a.re.x), "f"(a.re.y), "f"(a.im.x), "f"(a.im.y) : "memory");
}
__device__ __forceinline__ cp lds_cp(uint32_t addr) {
    cp a;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(a.re.x), "=f"(a.re.y), "=f"(a.im.x), "=f"(a.im.y) : "r"(addr) : "memory");
    return a;
}

// Four 8 x 8 matrices of 16-bit elements, transposed: lane i gets, from matrix m (row addresses
// in lanes 8 m .. 8 m + 7), rows 2 (i & 3) (low half) and 2 (i & 3) + 1 (high half) of column i >> 2.
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// Lane i of a producer warp stands for row pair R = i & 1 of the warp's two and for
// n2 = (i >> 2) + 8 H, H = (i >> 1) & 1, until the transpose.
//
// Address that the lane passes to ldsm4t: matrix = cylinder i >> 3, matrix row i & 7 = 2 x + e,
// x = R + 2 H: time row e of row pair R, feeds 8 H .. 8 H + 7 (+ 16 n1, 32 bytes each).  Rows of
// kRawRow bytes put the eight 16-byte matrix rows in distinct bank groups.
__device__ __forceinline__ uint32_t raw_lane(uint32_t raw, int lane) {
    const int x = (lane >> 1) & 3, e = lane & 1;
    return raw + (uint32_t)((2 * (x & 1) + e) * kRawRow + (lane >> 3) * (kFeed * kPol) + 16 * (x >> 1));
}

// Transpose slot (16 bytes) of n2 within row k of row pair R: n2 = 8 H + 4 b2 + 2 b1 + b0 goes to
// 8 b2 + ((4 (b1 ^ R) + 2 H + b0) ^ (k & 7)): the eight lanes that a 128-bit store serves at once
// (two n2, both H, both R) and the eight rows that a load serves fall in distinct bank groups.
__device__ __forceinline__ constexpr uint32_t tslot(int n2, int R) {
    return (uint32_t)(8 * ((n2 >> 2) & 1) + (4 * (((n2 >> 1) & 1) ^ R) + 2 * (n2 >> 3) + (n2 & 1)));
}

// Phase A for one warp and its two row pairs (SoA pairs of time rows):
//   raw    the lane's ldsm4t address (raw_lane)
//   twl    shared address of the lane's first entry of the [8][32] twiddle table
//   rows   the two row pairs' bins (2 x 8 KB; the transpose runs in place)
// Only warp-level synchronisation.  Hooks: `before_tb` runs before the bin rows are first written,
// `after_raw`, which requests the next raw rows, between the halves of the first transform, where half of
// the registers are free (right after the unpack, with all of them taken, 0.5 % slower; after the second
// half, too late, 4 %).
//
// Bound: the FMA pipe with the register reads of its operands, 530 packed operations per row pair
// here and 178 in the consumers: 64 % of its cycles, with 52 % of the issue slots; the two producer
// warps of a scheduler set the pace, the consumers wait for a good third of their time.  4 channels x 49152
// samples take 1.40 ms.  One row pair per warp and three warps at 128 registers, with lane-dependent twiddles
// in both transforms, are 6 % slower; the unpack straight from the transposing loads spares a store and
// two loads of the phased feeds per row pair and the odd half's divergent twiddles (4 %).
template <class AfterRaw, class BeforeTb>
__device__ __forceinline__ void phase_a(uint32_t raw, const PolSel& ps, const EwW& w, uint32_t twl,
                                        uint32_t rows, int lane, AfterRaw after_raw, BeforeTb before_tb) {
    cp y[16];
#pragma unroll
    for (int n1 = 0; n1 < 16; ++n1) {
        uint32_t g[4];
        ldsm4t(raw + 32u * n1, g);
#pragma unroll
        for (int c = 0; c < kCyl; ++c) {
            const uint32_t h = g[c] >> 16;
            const float2 xi = nibm(g[c], h, ps.mi, ps.si, ps.bi), xr = nibm(g[c], h, ps.mr, ps.sr, ps.br);
            if (c == 0) {
                y[n1] = {xr, xi};
            } else {
                y[n1].re = fma2(xi, w.NI[c - 1], fma2(xr, w.R[c - 1], y[n1].re));
                y[n1].im = fma2(xr, w.I[c - 1], fma2(xi, w.R[c - 1], y[n1].im));
            }
        }
    }
    {
        const int n2 = (lane >> 2) + 4 * (lane & 2), R = lane & 1;
        const uint32_t tw_ = rows + (uint32_t)(R * kRowB) + 16u * tslot(n2, R);
        cp v[16];
#pragma unroll
        for (int n1 = 0; n1 < 16; ++n1) v[n1] = y[n1];
        dft16<0>(v);                                     // even outputs: k = 2 k1
        // the bin rows may still be read as the previous bins
        before_tb();
#pragma unroll
        for (int k1 = 0; k1 < 16; ++k1) sts_cp((tw_ ^ (uint32_t)(16 * ((2 * k1) & 7))) + 256u * (2 * k1), v[k1]);
        after_raw();
        dft16<1>(y);                                     // odd outputs: k = 2 k1 + 1
#pragma unroll
        for (int k1 = 0; k1 < 16; ++k1)
            sts_cp((tw_ ^ (uint32_t)(16 * ((2 * k1 + 1) & 7))) + 256u * (2 * k1 + 1), y[k1]);
    }
    __syncwarp();
    // lane = k: twiddles and DFT16 over n2, bins L = 32 k2 + k; bsw(L) = 32 k2 + bsw(k).  The twiddles
    // are read here, not held through the first half, whose registers are all taken.
    float2 tw[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const cp t = lds_cp(twl + 512u * i);
        tw[2 * i] = t.re;
        tw[2 * i + 1] = t.im;
    }
#pragma unroll
    for (int R = 0; R < 2; ++R) {
        const uint32_t row = rows + (uint32_t)(R * kRowB);
        const uint32_t tr_ = row + 256u * (uint32_t)lane + 16u * (uint32_t)(lane & 7);
        cp v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int n2 = 4 * (q & 3) + (q >> 2);       // in the order dft16 consumes them
            const uint32_t sl = tslot(n2, R);
            v[n2] = lds_cp((tr_ ^ (16u * (sl & 7))) + 16u * (sl & 8));
        }
#pragma unroll
        for (int n2 = 1; n2 < 16; ++n2) v[n2] = cmulp(v[n2], bc(tw[n2].x), bc(tw[n2].y));
        dft16(v);
        // every lane has read the row before the bins are written over it
        __syncwarp();
        const uint32_t bw = row + 16u * (uint32_t)bsw(lane);
#pragma unroll
        for (int k2 = 0; k2 < 16; ++k2) sts_cp(bw + 512u * k2, v[k2]);
    }
}

// ---------------------------------------------------------------------------
// the fused kernel
// ---------------------------------------------------------------------------
__device__ __forceinline__ void bar_sync_n(int id, int n) { asm volatile("bar.sync %0, %1;" :: "r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive_n(int id, int n) { asm volatile("bar.arrive %0, %1;" :: "r"(id), "r"(n) : "memory"); }

// 16-byte asynchronous global -> shared copy (no registers), grouped per iteration
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// Warps 0-7 (producers) run phase A for their row pairs; warps 8-11 (consumers,
// one per TMEM lane quarter) gather the clamped bins, run the first up-channel
// pass into TMEM and, after each block, the second pass and the detection for
// two bins each (m and m + 128).  Each team of producers owns one bin buffer and
// every other iteration: it arrives on the named barrier FULL[b] after writing
// its buffer, the consumers arrive on the mbarrier EMPTY[b] after reading it, so
// phase A of an iteration overlaps the gather of the one before and the second
// up-channel pass.  A team's warp is at most one iteration of its buffer ahead
// of the slowest consumer, so no barrier phase ever mixes iterations.  The EMPTY
// waits are bounded; on expiry the kernel carries on (keeping every barrier
// matched) and reports through the status word.
//
// kMode: items = whole items and halves (units of 6 and 3 passes), parts = every item in parts of
// 1 or 2 passes (a launch of few items), dump = up-channelised voltages instead of detection.  An
// output is H0 + H1, H0 = (P0 + P1) + P2 and H1 = (P3 + P4) + P5 of its item's passes, in every mode.
constexpr int kItems = 0, kParts = 1, kDump = 2;
template <int kMode>
__global__ void __launch_bounds__(kThreads, 1) fused_fp32_kernel(const __grid_constant__ Batch bt) {
    extern __shared__ __align__(256) unsigned char smem[];   // the swizzles XOR address bits 4-7
    float4* bins_all = reinterpret_cast<float4*>(smem);
    unsigned char* raw_all = smem + kSmemBins;
    int* lut_s = reinterpret_cast<int*>(smem + kSmemBins + kSmemRaw);
    int* beam_s = lut_s + kNs;
    float4* twl_s = reinterpret_cast<float4*>(smem + kSmemBins + kSmemRaw + kSmemLut);
    float* park_s = reinterpret_cast<float*>(smem + kSmemBins + kSmemRaw + kSmemLut + kSmemTwl);
    __shared__ uint32_t tmem_base_s;
    __shared__ __align__(8) uint64_t empty_s[2];
    __shared__ int expired_s, table_s;                       // table_s: the table in lut_s and beam_s

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t empty0 = smem_sa(&empty_s[0]);

    if (warp == 0) {
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(&tmem_base_s));
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" :: "r"(dst) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < kLaneTwLen / 2; i += kThreads) twl_s[i] = reinterpret_cast<const float4*>(bt.twl)[i];
    if (tid == 0) {
        for (int i = 0; i < 2; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(empty0 + 8u * i), "n"(kCons) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        expired_s = 0;
        table_s = -1;
    }
    cta_sync();
    const uint32_t tmem = tmem_base_s;
    constexpr int kPasses = kTds * kPol;
    const unsigned long long wlim = bt.wait_ns ? bt.wait_ns : kWaitNs;

    const PassUnits units = bt.units;
    static_assert(kPasses == 6, "an item is two halves of three passes");

    if (warp < kWarps) {
        // ---------------------------------- producers ----------------------------------
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(kRegProd) : "memory");
        const int team = warp / kTeam, tw = warp % kTeam;
        const uint32_t raw_sa = smem_sa(raw_all) + (uint32_t)(warp * kRawB);
        const uint32_t raw_ld = raw_lane(raw_sa, lane);
        const uint32_t rows = smem_sa(bins_all + team * kBinsF4 + 2 * tw * kBins);
        const uint32_t empty = empty0 + 8u * (uint32_t)team;
        const uint32_t twl = smem_sa(twl_s) + 16u * lane;
        uint32_t g = 0;                                   // this team's iterations so far
        for (int un = blockIdx.x; un < units.n_units; un += gridDim.x) {
            int item, ps0, ps1;
            pass_unit(units, un, item, ps0, ps1);
            const int sgi = seg_of(bt, item);
            const Seg& sg = bt.segs[sgi];
            const int local = item - sg.item_begin;
            const int F = local >> 2, j = local & 3;
            // time rows 16 a + 2 it + {0, 1} of row pairs a = 2 tw, 2 tw + 1
            const long long row0 = (long long)F * kFrame + 32 * tw;
            // this lane's part of row row0 in the carried and in the new samples, and the number of rows
            // from it that are carried: a row's address is then a comparison and 32-bit arithmetic
            // (3 % of a launch against 64-bit products per row)
            const uint8_t* const carried = sg.carry + row0 * kInput + 16 * lane;
            const uint8_t* const fresh = sg.vin + (row0 - sg.carry_rows) * kInput + 16 * lane;
            const int left = row0 < sg.carry_rows ? (int)(sg.carry_rows - row0) : 0;
            // this warp's four rows of iteration (ps, it) into its raw buffer
            auto fetch = [&](int ps, int it) {
                const int r0 = (ps >> 1) * kUp + 2 * it;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = r0 + 16 * (k >> 1) + (k & 1);
                    const uint8_t* p = (r < left ? carried : fresh) + (uint32_t)(r * kInput);
                    const uint32_t d = raw_sa + (uint32_t)(k * kRawRow) + 16u * lane;
#pragma unroll
                    for (int c = 0; c < kCyl; ++c) cp16(d + c * (kFeed * kPol), p + c * (kFeed * kPol));
                }
                cp_commit();
            };
            fetch(ps0, team);
            EwW w;
            load_ew_frame(sg, bt.ew, F, j, w);
            for (int ps = ps0; ps < ps1; ++ps) {
                const PolSel sel = pol_sel(ps & 1);
#pragma unroll 1
                for (int it = team; it < 8; it += 2, ++g) {
                    cp_wait<0>();
                    __syncwarp();
                    phase_a(raw_ld, sel, w, twl, rows, lane,
                            [&] {
                                // every lane has its words: the next iteration's rows may replace them
                                __syncwarp();
                                if (it < 6)
                                    fetch(ps, it + 2);
                                else if (ps + 1 < ps1)
                                    fetch(ps + 1, team);
                            },
                            [&] {
                                // the buffer is free once the consumers gathered this team's last
                                // iteration (release number g - 1)
                                if (g >= 1 && !mbar_wait(empty, (g - 1u) & 1u, wlim)) expired_s = 1;
                            });
                    bar_arrive_n(kBarFull + team, kFullThreads);
                }
            }
        }
    } else {
        // ---------------------------------- consumers ----------------------------------
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kRegCons) : "memory");
        const int cq = warp - kWarps;                    // TMEM lane quarter
        const int ctid = tid - 32 * kWarps;
        const uint32_t tlane = tmem + (static_cast<uint32_t>(32 * cq) << 16);
        const int m0 = 32 * cq + lane;                   // consumer slots m0 (half 0) and m0 + 128 (half 1)
        uint32_t g = 0;
        for (int un = blockIdx.x; un < units.n_units; un += gridDim.x) {
            int item, ps0, ps1;
            pass_unit(units, un, item, ps0, ps1);
            const int sgi = seg_of(bt, item);
            const Seg& sg = bt.segs[sgi];
            const int local = item - sg.item_begin;
            const int F = local >> 2, j = local & 3;
            // lanes may have parted in the last unit's add_passes; barriers and tensor memory want the whole warp
            // (behind add_passes itself it costs 1 %, here nothing)
            __syncwarp();
            // the table changes with the channel only (reloading it for every item costs 0.8 %); its number
            // is in shared memory because a register more costs 1 %
            if (sg.table != *(volatile int*)&table_s) {
                bar_sync_n(kBarCons, 32 * kCons);         // the previous table's reads are done
                // consumer slot i (TMEM lane + 128 x half) takes beam order[i]
                for (int i = ctid; i < kNs; i += 32 * kCons) {
                    const int bm = bt.order[sg.table * kNs + i];
                    beam_s[i] = bm;
                    lut_s[i] = bt.lut[sg.table * kNs + bm];
                }
                if (ctid == 0) table_s = sg.table;
                bar_sync_n(kBarCons, 32 * kCons);
            }
            const bool whole = ps1 - ps0 == kPasses;
            const int Lsw0 = bsw(lut_s[m0]), Lsw1 = bsw(lut_s[m0 + 128]);
            // the slots' beams (gather order); output addresses are formed where they are used
            auto out0 = [&] { return sg.out + (long long)(kNs * j + beam_s[m0]) * sg.beam_stride + F; };
            auto out1 = [&] { return sg.out + (long long)(kNs * j + beam_s[m0 + 128]) * sg.beam_stride + F; };
            // sums of the passes of the current half item (passes 0-2 or 3-5)
            float acc0[kSub], acc1[kSub];
#pragma unroll
            for (int s2 = 0; s2 < kSub; ++s2) {
                acc0[s2] = 0.f;
                acc1[s2] = 0.f;
            }
            for (int ps = ps0; ps < ps1; ++ps) {
                const int blk = ps >> 1, pol = ps & 1;
#pragma unroll 1
                for (int it = 0; it < 8; ++it, ++g) {
                    const uint32_t b = g & 1u;
                    bar_sync_n(kBarFull + (int)b, kFullThreads);
                    const float4* bins = bins_all + b * kBinsF4;
                    // gather + 8-point DFT over a (tau = 16 a + b, b = 2 it, 2 it + 1), both bin halves
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int Lsw = hh ? Lsw1 : Lsw0;
                        cp z[8];
#pragma unroll
                        for (int a = 0; a < 8; ++a) z[a] = ld_cp(bins + a * kBins + Lsw);
                        dft8(z);
                        const int b0 = 2 * it;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            if (c) {
                                const float4 t = kPairTw.w[it][c];
                                z[c] = cmulp(z[c], make_float2(t.x, t.y), make_float2(t.z, t.w));
                            }
                            tmem_st4(tlane + hh * 256 + 2 * (16 * c + b0), z[c].re.x, z[c].im.x, z[c].re.y,
                                     z[c].im.y);
                        }
                    }
                    __syncwarp();                                   // this warp's reads of buffer b are done
                    if (lane == 0) mbar_arrive(empty0 + 8u * b);
                }
                tmem_wait_st();
                // second pass: 16-point DFT over b for fine channels q = c + 8 d (this warp's lanes only)
                const long long dbase = ((((long long)(F * kTds + blk) * kPol + pol) * kEw + j) * kNs) * kUp;
                auto pass2 = [&](int hh, float (&acc)[kSub]) {
                    float p[kSub];                            // this pass's sums
#pragma unroll
                    for (int s2 = 0; s2 < kSub; ++s2) p[s2] = 0.f;
                    upchan_pass2(tlane, hh, p, kMode == kDump ? bt.dump + dbase + (long long)beam_s[m0 + 128 * hh] * kUp : nullptr);
                    if constexpr (kMode == kParts) {
                        float* mine = bt.part + ((size_t)(item - units.n_full) * kPasses + ps) * (kSub * kNs) + m0 + 128 * hh;
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) mine[s2 * kNs] = p[s2];
                    } else {
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) acc[s2] += p[s2];
                    }
                };
                pass2(0, acc0);
                pass2(1, acc1);
                // the next pass's gathers overwrite these TMEM columns in this warp's program order
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if constexpr (kMode == kParts) {
                    // the thread that completes the item's six passes adds them (slots m0 and m0 + 128)
                    const int slot = item - units.n_full;
                    if (add_passes(bt.part_tok + (size_t)slot * kNs + m0, bt.epoch, 1)) {
                        const float* in = bt.part + (size_t)slot * kPasses * (kSub * kNs) + m0;
#pragma unroll 1
                        for (int hh = 0; hh < 2; ++hh) {
                            float* o = hh ? out1() : out0();
                            float v[kPasses][kSub];
                            load_passes(in + 128 * hh, v);
#pragma unroll
                            for (int s2 = 0; s2 < kSub; ++s2)
                                o[(long long)s2 * sg.sub_stride] =
                                    ((v[0][s2] + v[1][s2]) + v[2][s2]) + ((v[3][s2] + v[4][s2]) + v[5][s2]);
                        }
                    }
                    __syncwarp();        // as at the unit's start, for the next pass
                }
                if constexpr (kMode == kItems) {
                    if (whole && ps == kPasses / 2 - 1) {
                        // whole item: H0 (passes 0-2) parks in shared memory until H1 is done
                        // (each thread reads back only its own words)
                        float* pk = park_s;
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) {
                            pk[s2 * kNs + m0] = acc0[s2];
                            pk[s2 * kNs + m0 + 128] = acc1[s2];
                            acc0[s2] = 0.f;
                            acc1[s2] = 0.f;
                        }
                    }
                }
            }
            if constexpr (kMode == kItems) {
                if (whole) {
                    // all loads before the first store: the stores could alias them as far as
                    // the compiler knows, and would otherwise serialise the loads
                    const float* pk = park_s;
                    float h[kSub];
#pragma unroll
                    for (int s2 = 0; s2 < kSub; ++s2) h[s2] = pk[s2 * kNs + m0];
                    float* o = out0();
#pragma unroll
                    for (int s2 = 0; s2 < kSub; ++s2) o[(long long)s2 * sg.sub_stride] = h[s2] + acc0[s2];
#pragma unroll
                    for (int s2 = 0; s2 < kSub; ++s2) h[s2] = pk[s2 * kNs + m0 + 128];
                    o = out1();
#pragma unroll
                    for (int s2 = 0; s2 < kSub; ++s2) o[(long long)s2 * sg.sub_stride] = h[s2] + acc1[s2];
                } else {
                    // half unit: publish this half; the second of the two halves to finish
                    // adds them (per thread: slots m0 and m0 + 128)
                    const int slot = item - units.n_full, half = ps0 ? 1 : 0;
                    float* mine = bt.part + ((size_t)slot * 2 + half) * (kSub * kNs);
#pragma unroll
                    for (int s2 = 0; s2 < kSub; ++s2) {
                        mine[s2 * kNs + m0] = acc0[s2];
                        mine[s2 * kNs + m0 + 128] = acc1[s2];
                    }
                    if (add_passes(bt.part_tok + (size_t)slot * kNs + m0, bt.epoch, kPasses / 2)) {
                        // H0 + H1 in either order: one addition of two terms is exact-commutative
                        const float* other = bt.part + ((size_t)slot * 2 + (half ^ 1)) * (kSub * kNs);
                        float h[kSub];
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) h[s2] = __ldcg(other + s2 * kNs + m0);
                        float* o = out0();
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) o[(long long)s2 * sg.sub_stride] = acc0[s2] + h[s2];
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) h[s2] = __ldcg(other + s2 * kNs + m0 + 128);
                        o = out1();
#pragma unroll
                        for (int s2 = 0; s2 < kSub; ++s2) o[(long long)s2 * sg.sub_stride] = acc1[s2] + h[s2];
                    }
                }
            }
        }
    }

    cta_sync();
    if (expired_s && tid == 0 && bt.status) atomicExch(bt.status, 1);
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(tmem) : "memory");
    }
}

// ---------------------------------------------------------------------------
// inspection kernels sharing the device code above
// ---------------------------------------------------------------------------

// Stages 1+2 of 4 consecutive rows per CTA (one warp: two row pairs), then the clamp gather.
__global__ void __launch_bounds__(32) debug_beams_kernel(const uint8_t* __restrict__ vin, long long T,
                                                          const int16_t* __restrict__ lut,
                                                          const float2* __restrict__ ew, const float2* __restrict__ twl,
                                                          float2* __restrict__ out) {
    __shared__ __align__(256) float4 bins2[2 * kBins];    // 256-byte rows: the swizzles XOR address bits 4-7
    __shared__ __align__(256) unsigned char raw[kRawB];
    const int lane = threadIdx.x;
    const long long t0 = (long long)blockIdx.x * 4;
    const int pol = blockIdx.y & 1, j = blockIdx.y >> 1;
    __shared__ float4 twl_s[kLaneTwLen / 2];
    for (int i = lane; i < kLaneTwLen / 2; i += 32) twl_s[i] = reinterpret_cast<const float4*>(twl)[i];
    EwW w;
    load_ew(ew, 0, j, w);
    for (int k = 0; k < 4; ++k) {
        const uint4* p = reinterpret_cast<const uint4*>(vin + min(t0 + k, T - 1) * kInput);
        for (int i = lane; i < kInput / 16; i += 32) *reinterpret_cast<uint4*>(raw + k * kRawRow + 16 * i) = __ldg(p + i);
    }
    __syncwarp();
    phase_a(raw_lane(smem_sa(raw), lane), pol_sel(pol), w, smem_sa(twl_s) + 16u * lane, smem_sa(bins2), lane, [] {},
            [] {});
    __syncwarp();
    for (int i = lane; i < 4 * kNs; i += 32) {
        const int r = i >> 8, mm = i & 255;          // r: row 0..3 = slot (r >> 1), element (r & 1)
        const long long t = t0 + r;
        if (t >= T) continue;
        const float4 v = bins2[(r >> 1) * kBins + bsw(lut[mm])];
        out[((t * kPol + pol) * kEw + j) * kNs + mm] = (r & 1) ? make_float2(v.y, v.w) : make_float2(v.x, v.z);
    }
}

__global__ void debug_unpack_kernel(const uint8_t* __restrict__ in, float2* __restrict__ out, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const PolSel ps = pol_sel(0);                        // by the whole warp
    if (i >= n) return;
    const uint32_t g = in[i];                            // as a polarisation-0 byte
    const float2 re = nibm(g, g, ps.mr, ps.sr, ps.br), im = nibm(g, g, ps.mi, ps.si, ps.bi);
    out[i] = make_float2(re.x, im.x);
}


// Shared-memory opt-in, and a check that the compiled kernel was given the
// registers per thread the setmaxnreg split assumes: with fewer, the producers'
// increase could not be granted, so such a build is refused instead of launched.
// Done once per device (the outcome is kept and returned on every launch); the flags
// have internal linkage, so two copies of the library in one process keep their own.
template <int kMode>
cudaError_t prepare_fp32() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    static std::once_flag once[kMaxDevices];
    static cudaError_t result[kMaxDevices];
    std::call_once(once[dev], [&] {
        cudaFuncAttributes fa;
        cudaError_t r = cudaFuncGetAttributes(&fa, fused_fp32_kernel<kMode>);
        if (r == cudaSuccess && fa.numRegs < kRegLaunch) r = cudaErrorInvalidConfiguration;
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(fused_fp32_kernel<kMode>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemTotal);
        result[dev] = r;
    });
    return result[dev];
}

}  // namespace

namespace {
template <int kMode>
cudaError_t launch_fp32(const Batch& b, int grid, cudaStream_t s) {
    if (b.n_items <= 0) return cudaSuccess;
    if (b.units.g < kTds * kPol && (!b.part || !b.part_tok)) return cudaErrorInvalidValue;
    cudaError_t e = prepare_fp32<kMode>();
    if (e != cudaSuccess) return e;
    fused_fp32_kernel<kMode><<<grid, kThreads, kSmemTotal, s>>>(b);
    return cudaGetLastError();
}
}  // namespace

cudaError_t fused_fp32_launch(const Batch& b, int grid, cudaStream_t s) {
    return b.units.g < kTds * kPol / 2 ? launch_fp32<kParts>(b, grid, s) : launch_fp32<kItems>(b, grid, s);
}

cudaError_t fused_fp32_dump_launch(const Batch& b, int grid, cudaStream_t s) { return launch_fp32<kDump>(b, grid, s); }

int fused_fp32_max_grid(int device) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
    return sms;
}

cudaError_t debug_beams_launch(const uint8_t* vin, long long T, const int16_t* lut, const float2* ew,
                               const float2* twl, float2* out, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    dim3 grid((unsigned)((T + 3) / 4), kPol * kEw);
    debug_beams_kernel<<<grid, 32, 0, s>>>(vin, T, lut, ew, twl, out);
    return cudaGetLastError();
}

cudaError_t debug_unpack_launch(const uint8_t* in, float* out, long long n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    debug_unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(in, reinterpret_cast<float2*>(out), n);
    return cudaGetLastError();
}

}  // namespace chimebf
