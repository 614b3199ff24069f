// Internal interface between the host runtime (runtime.cpp) and the CUDA
// kernels (fused_fp32.cu).  Not part of the public C ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace chimebf {

// Geometry the kernels are built for (Sec. 1, Sec. 2, Sec. 3, Table 1).
constexpr int kCyl = 4;          // cylinders
constexpr int kFeed = 256;       // feeds per cylinder (N)
constexpr int kPol = 2;          // polarisations
constexpr int kBins = 512;       // zero-padded N-S FFT length (N P, P = 2)
constexpr int kNs = 256;         // N-S beams kept by the clamp
constexpr int kEw = 4;           // E-W beams
constexpr int kUp = 128;         // up-channelisation FFT length
constexpr int kFds = 8;          // fine channels per output sub-channel
constexpr int kTds = 3;          // 128-sample blocks per output frame
constexpr int kSub = kUp / kFds; // 16 sub-channels
constexpr int kFrame = kUp * kTds;   // 384 samples per frame
constexpr int kInput = kCyl * kFeed * kPol;   // 2048 bytes per time sample
constexpr int kBeams = kEw * kNs;    // 1024 intensity beams
constexpr int kLaneTwLen = 32 * 16;     // twiddles between the FP32 form's two N-S stages

// Segments per launch (kernel-parameter space holds the descriptors).
constexpr int kMaxSegs = 160;

// One (request, channel): a frame stream made of `carry_rows` leftover rows
// followed by the request's new rows.
struct Seg {
    const uint8_t* vin;      // row 0 of this channel's new samples [n][2048]
    const uint8_t* carry;    // leftover rows [carry_rows][2048] (may be null)
    float* out;              // &out[beam 0][sub 16*chan][frame 0] of the request
    long long beam_stride;   // elements between beams  (16 * n_chan * n_frames)
    int sub_stride;          // elements between sub-channels (n_frames)
    int carry_rows;          // 0..383
    int n_frames;            // frames of this segment
    int table;               // row of the per-frequency tables
    int item_begin;          // first work item; 4 items (E-W beams) per frame
    int pad_;
    const float2* ew_frames; // tracking E-W beams: [n_frames][4 ew][4 cyl] phases, or null (static)
    const unsigned char* a_img;  // tensor-core form: FP16 twiddle image(s) of this segment's table
};

// Work units of a launch whose items (six passes each) go to `slots` CTAs or CTA pairs in turn: whole
// items, and the items of a last round that leaves slots idle in parts of g passes, g the smallest
// from `least_g` that gives every part a slot of its own (parts in several rounds lose more between
// units, most of a pass each, than they balance: FP32 form, 108 items on 152 CTAs, 181 us in single passes
// and 121 whole; three terms, 48 items on 76 pairs, 64 and 62).  Every output adds the six passes' sums in
// one fixed order, whether or not its item was split, so the result does not depend on how a request was
// batched.
struct PassUnits {
    int n_full;     // items run whole: 0 .. n_full - 1
    int g;          // passes of a part of the others (1, 2, 3; 6: none is split)
    int n_units;    // n_full + (6 / g) x (split items)
};
inline PassUnits pass_units(int n_items, int slots, int least_g) {
    constexpr int kPasses = kTds * kPol;
    const int rem = n_items % slots;
    for (int g = least_g; rem > 0 && g <= kPasses / 2; ++g)
        if (rem * (kPasses / g) <= slots) return {n_items - rem, g, n_items - rem + rem * (kPasses / g)};
    return {n_items, kPasses, n_items};
}
// Room for the sums of split items on `grid` CTAs (as many slots, or half as many of CTA pairs): every part has a
// slot, so at most grid / 2 items are split (in halves), and they publish at most 2 grid sums of 16 x 256 floats:
// grid / 3 items in thirds all six passes each, fewer in the other cases (items in halves publish two in
// the FP32 form, and six, of grid / 4 items, in the tensor-core forms).
inline size_t part_items(int grid) { return (size_t)grid / 2; }
inline size_t part_sums(int grid) { return 2 * (size_t)grid; }

struct Batch {
    int n_segs;
    int n_items;
    const int16_t* lut;      // [n_tables][256]   clamp table, Eq. (1)
    const int16_t* order;    // [n_tables][256]   FP32 form: beam taken by consumer slot (TMEM lane + 128 x half)
    const float2* ew;        // [n_tables][4 ew][4 cyl] E-W phases
    const float2* twl;       // FP32 form: exp(-2 pi i n k / 512) at [n / 2][k][n & 1], n < 16, k < 32
    float2* dump;            // debug: up-channelised voltages instead of detection
    int* status;                 // set non-zero by a kernel whose bounded wait expired
    unsigned long long wait_ns;  // bound on each device-side wait (0: the default, 2 s)
    int stall_mma;               // stall check: the MMA warps (else the builders) stop ...
    int stall_chunks;            // ... after this many chunks of 32 feeds
    PassUnits units;             // work units of the launch
    float* part;                 // sums of split items' passes [item][6] or halves [item][2], each [16][256]
    unsigned long long* part_tok;    // [item][256] passes published (see add_passes)
    unsigned long long epoch;        // this launch's number within the plan (from 1)
    Seg segs[kMaxSegs];
};

// Launches of the CUDA code; each returns the launch status.
cudaError_t fused_fp32_launch(const Batch& b, int grid, cudaStream_t s);
cudaError_t fused_fp32_dump_launch(const Batch& b, int grid, cudaStream_t s);
cudaError_t debug_beams_launch(const uint8_t* vin, long long n_samples, const int16_t* lut,
                               const float2* ew, const float2* twl, float2* out, cudaStream_t s);
cudaError_t debug_unpack_launch(const uint8_t* in, float* out, long long n, cudaStream_t s);
int fused_fp32_max_grid(int device);   // CTAs that fit at once (1 per SM)

// Tensor-core form on `pairs` clusters of two CTAs over b.units: `terms` = 1, 2 or 3 GEMM terms; mode
// 0 = detect, 1 = dump up-channelised voltages, 2 = dump the N-S/E-W beams of the GEMM, 3 = stall check:
// the MMA warps or the builders stop (b.stall_mma, b.stall_chunks), so the other warps' waits run out and the
// kernel reports through `status`.
cudaError_t fused_tc_launch(const Batch& b, int terms, int mode, int pairs, cudaStream_t s);
// Tensor-core form: a table's twiddle image, C (part 0) and S (part 1) = cos and sin of 2 pi n L(m) / 512
// in FP16, in the order of the kernel's shared memory operand: chunks of kTFeeds feeds, the CTAs of a
// pair (128 bins each), C and S blocks of 8-row x 16-byte core matrices.  For three terms the image of
// the rest (lo) follows.
constexpr int kTFeeds = 32;                       // feeds per chunk
constexpr int kTTw = 128 * kTFeeds * 2;           // 8 KB: C or S of 128 bins for one chunk
// operand blocks: k-groups (8 feeds) kTALbo and 8-row groups kTASbo bytes apart
constexpr int kTALbo = 128, kTASbo = kTFeeds / 8 * kTALbo;
constexpr size_t tc_a_bytes(int terms) { return (size_t)kNs * 2 * kFeed * 2 * (terms == 3 ? 2 : 1); }
constexpr size_t tc_a_offset(int m, int n, int part) {
    return (((size_t)(n / kTFeeds) * 2 + m / 128) * 2 + part) * kTTw + (size_t)(m % 128 / 8) * kTASbo +
           (n % kTFeeds / 8) * kTALbo + (m % 8) * 16 + (n % 8) * 2;
}
cudaError_t skymap_launch(const float* in, int n_beams, long long per_beam, float* map, cudaStream_t s);
cudaError_t dedisperse_launch(const float* in, const int* delays, int n_sub, long long nf, long long n_out,
                              float* out, cudaStream_t s);
// Allocation-free dedispersion: the device's static delay table (address
// looked up once per device; the caller has made `device` current).
constexpr int kDdStaticMaxSub = kSub * 4096;    // 4096 channels x 16 sub-channels
constexpr int kMaxDevices = 64;
cudaError_t dedisperse_static_table(int device, int** table);
cudaError_t rescale_u8_launch(const float* in, long long rows, long long nf, uint8_t* codes, float* stats,
                              cudaStream_t s);
// FP32 FMA-pipe probe: 4 CTAs per SM (at most n_sink / 256) of 256 threads, each
// thread `iters` (rounded up to 4) x 16 FFMA2 (paired) or 32 scalar FMA; *flop = flops issued.
cudaError_t fma_probe_launch(bool paired, long long iters, float* sink, long long n_sink, int sms, double* flop,
                             cudaStream_t s);

}  // namespace chimebf
