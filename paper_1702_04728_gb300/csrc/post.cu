// Kernels that run on the fan-beam output (arXiv 1702.04728, Sec. 3, Sec. 3.3,
// Table 1): the frequency- and time-summed sky map of Fig. 3 and the 8-bit
// rescaling of the intensity listed in Table 1.
#include "bf_internal.h"

#include <algorithm>
#include <cstdint>
#include <mutex>

namespace chimebf {
namespace {

constexpr int kMapThreads = 256;

// One CTA per beam: sum of the beam's [n_sub][n_frames] block (contiguous),
// fixed-order tree reduction in FP32.
__global__ void __launch_bounds__(kMapThreads) skymap_kernel(const float* __restrict__ in, long long per_beam,
                                                             float* __restrict__ map) {
    __shared__ float red[kMapThreads / 32];
    const float* p = in + (long long)blockIdx.x * per_beam;
    float s = 0.f;
    const long long n4 = per_beam / 4;
    const bool al = ((reinterpret_cast<uintptr_t>(p) & 15) == 0);
    if (al) {
        const float4* p4 = reinterpret_cast<const float4*>(p);
        for (long long i = threadIdx.x; i < n4; i += kMapThreads) {
            const float4 v = __ldg(p4 + i);
            s += (v.x + v.y) + (v.z + v.w);
        }
        for (long long i = 4 * n4 + threadIdx.x; i < per_beam; i += kMapThreads) s += __ldg(p + i);
    } else {
        for (long long i = threadIdx.x; i < per_beam; i += kMapThreads) s += __ldg(p + i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = threadIdx.x < kMapThreads / 32 ? red[threadIdx.x] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) map[blockIdx.x] = t;
    }
}

// 8-bit codes of (beam, sub-channel) rows: mean and population standard
// deviation over the row's frames, then code = clip(floor(64 + 16 (x - mean) /
// std + 1/2), 0, 255), a constant row giving 64.  FP32: the sums run over x -
// x0 (x0 = the row's first frame), which keeps a constant row exactly constant
// (mean = x0, std = 0) and makes the rounding error of the mean scale with the
// row's spread instead of its level.  Valid for |x - mean| below ~1e18 (the
// squares stay finite).  The sums run frame by frame, so a thread's two chains of
// adds set the time of its row and rows in flight hide it: a CTA of four warps
// stages 32 rows in shared memory of just their size (10 CTAs per SM at 128
// frames), loads and reads 16 bytes at a time (rows padded to an odd number of
// 16-byte words); one warp runs the sums, a thread per row, and all four write the
// codes, a lane per four frames, straight to memory.  Rows longer than kU8Whole are
// staged in chunks, once per sweep (sum, squares, codes), since whole rows would
// leave too few CTAs.  Bound by instructions (0.55 of the issue slots), so 16 / std is
// formed once per row, the codes are rounded by an addition instead of two conversions,
// and places in shared memory advance without products: 65536 rows of 128 frames 14.3 us
// (16.6 without these; one warp per CTA, five CTAs per SM, scalar accesses: 55), eight times
// as many 77 us (94); 42 and 336 MB, 6 and 49 us of HBM.
constexpr int kU8Rows = 32;
constexpr int kU8Threads = 128;
constexpr int kU8Whole = 512;          // longest row staged whole
constexpr int kU8Chunk = 256;          // frames per chunk of longer rows

// floats between staged rows of up to n frames: a multiple of 4 whose quarter is odd
__host__ __device__ constexpr int u8_stride(int n) { return 4 * (((n + 3) / 4) | 1); }

// kVec: rows are a multiple of 4 frames and start on 16 bytes (codes: 4 bytes).  Len: numbers the frames of
// a row, 64 bits for rows beyond 2^31 frames only (for all rows they cost up to 10 %).
template <bool kVec, class Len>
__global__ void __launch_bounds__(kU8Threads) rescale_u8_kernel(const float* __restrict__ in, long long rows, Len nf,
                                                                  int chunk, uint8_t* __restrict__ codes,
                                                                  float* __restrict__ stats) {
    extern __shared__ __align__(16) float st[];
    __shared__ float2 fit_s[kU8Rows];                     // mean and 16 / std, -1 for a row without spread
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long r0 = (long long)blockIdx.x * kU8Rows;
    const int nr = (int)min((long long)kU8Rows, rows - r0);
    const int S = u8_stride(chunk);
    const float* src = in + r0 * nf;
    constexpr int V = kVec ? 4 : 1;                       // frames per access

    // n frames from f0 of the CTA's rows; whole rows are one contiguous block, walked without divisions
    auto stage = [&](Len f0, int n) {
        __syncthreads();
        if (n == nf) {
            const int per = (int)nf / V, total = nr * per, dr = kU8Threads / per, dc = kU8Threads % per;
            const int step = dr * S + V * dc, wrap = S - V * per;
            int c = tid % per, o = tid / per * S + V * c;     // o: the access's place among the staged rows
#pragma unroll 8
            for (int i = tid; i < total; i += kU8Threads) {
                if constexpr (kVec)
                    *reinterpret_cast<float4*>(st + o) = __ldg(reinterpret_cast<const float4*>(src) + i);
                else
                    st[o] = __ldg(src + i);
                o += step;
                c += dc;
                if (c >= per) {
                    c -= per;
                    o += wrap;
                }
            }
        } else {
#pragma unroll 4
            for (int r = warp; r < nr; r += kU8Threads / 32)
                for (int i = lane; i < n / V; i += 32) {
                    const float* p = src + (long long)r * nf + f0 + V * i;
                    if constexpr (kVec)
                        *reinterpret_cast<float4*>(st + r * S + 4 * i) = __ldg(reinterpret_cast<const float4*>(p));
                    else
                        st[r * S + i] = __ldg(p);
                }
        }
        __syncthreads();
    };
    // f(frame, value) over the n staged frames of row `lane` in order
    const float* row = st + lane * S;
    auto each = [&](int n, auto f) {
        if constexpr (kVec) {
#pragma unroll 8
            for (int k = 0; k < n; k += 4) {
                const float4 v = *reinterpret_cast<const float4*>(row + k);
                f(k, v.x);
                f(k + 1, v.y);
                f(k + 2, v.z);
                f(k + 3, v.w);
            }
        } else {
#pragma unroll 8
            for (int k = 0; k < n; ++k) f(k, row[k]);
        }
    };
    const bool sums = warp == 0 && lane < nr, single = chunk >= nf;
    float x0 = 0.f, s = 0.f, q = 0.f;
    for (Len f0 = 0; f0 < nf; f0 += chunk) {
        const int n = (int)min((Len)chunk, nf - f0);
        stage(f0, n);
        if (!sums) continue;
        if (f0 == 0) {
            x0 = row[0];
            each(n, [&](int k, float v) {
                if (k) s += v - x0;
            });
        } else {
            each(n, [&](int, float v) { s += v - x0; });
        }
    }
    const float mean = x0 + s / (float)nf;
    for (Len f0 = 0; f0 < nf; f0 += chunk) {
        const int n = (int)min((Len)chunk, nf - f0);
        if (!single) stage(f0, n);
        if (!sums) continue;
        each(n, [&](int, float v) {
            const float d = v - mean;
            q = fmaf(d, d, q);
        });
    }
    if (sums) {
        const float sd = sqrtf(q / (float)nf);
        fit_s[lane] = make_float2(mean, sd > 0.f ? 16.f / sd : -1.f);
        if (stats) {
            stats[2 * (r0 + lane)] = mean;
            stats[2 * (r0 + lane) + 1] = sd;
        }
    }
    __syncthreads();
    for (Len f0 = 0; f0 < nf; f0 += chunk) {
        const int n = (int)min((Len)chunk, nf - f0);
        if (!single) stage(f0, n);
        uint8_t* dst = codes + r0 * nf + f0;
        // the clamped value's floor sits in the low byte of its sum with 2^23, rounded down
        auto code = [&](float2 fit, float x) -> uint32_t {
            const float v = fit.y < 0.f ? 64.f : fminf(fmaxf(fmaf(x - fit.x, fit.y, 64.5f), 0.f), 255.f);
            return __float_as_uint(__fadd_rd(v, 8388608.f));
        };
        if (kVec || single) {
            const int per = n / V, total = nr * per, dr = kU8Threads / per, dc = kU8Threads % per;
            const int step = dr * S + V * dc, wrap = S - V * per;
            int r = tid / per, c = tid % per, o = r * S + V * c;
#pragma unroll 4
            for (int i = tid; i < total; i += kU8Threads) {
                const float2 fit = fit_s[r];
                if constexpr (kVec) {
                    const float4 v = *reinterpret_cast<const float4*>(st + o);
                    const uint32_t lo = __byte_perm(code(fit, v.x), code(fit, v.y), 0x0040);
                    const uint32_t hi = __byte_perm(code(fit, v.z), code(fit, v.w), 0x0040);
                    uint8_t* to = single ? dst + 4 * (size_t)i : dst + (size_t)r * nf + 4 * c;
                    *reinterpret_cast<uint32_t*>(to) = __byte_perm(lo, hi, 0x5410);
                } else {
                    dst[i] = (uint8_t)code(fit, st[o]);
                }
                r += dr;
                c += dc;
                o += step;
                if (c >= per) {
                    c -= per;
                    ++r;
                    o += wrap;
                }
            }
        } else {
#pragma unroll 2
            for (int r = warp; r < nr; r += kU8Threads / 32) {
                const float2 fit = fit_s[r];
                for (int i = lane; i < n; i += 32) dst[(size_t)r * nf + i] = (uint8_t)code(fit, st[r * S + i]);
            }
        }
    }
}

// Incoherent dedispersion to one DM: series[beam][t] = sum over sub-channels s
// of in[beam][s][t + d_s], t < n_out.  Threads run along t, so each sub-channel row
// is read with coalesced (unaligned) loads.  A CTA takes up to 1024 frames of a beam, kR of them per
// thread and wt apart, so that a row is read as one piece.
//
// The sub-channels are cut into `parts` runs (by their number alone), each summed in order, and the runs' sums
// are added in order, so a sample has the same bits in a series of any length.  `groups` of wt threads share
// the runs; the first one adds its own runs as they come, which keeps the sums of the longest tiles below
// 48 KB.  Eight rows at a time, their delays in two loads, keep some 100 KB in flight per SM; short
// series (kR = 1) need four CTAs for that, 32 registers a thread.
//
// Bound by HBM and, below some 200 frames, by latency.  1024 sub-channels x 1017 frames to 630: 435 us
// (6.1 TB/s), 200 frames to 194: 156, 96 to 90: 76, 64 to 58: 56, 40 to 34: 50; a contiguous share of the
// sub-channels per thread group, whose number follows the length, took 439, 155, 76, 55 and 45.  16 runs
// instead of 20: 84 us at 90 frames (five groups); 24, one more than fits in 48 KB, 2 % more at 998.
constexpr int kDdThreads = 512;
constexpr int kDdParts = 20;           // most runs of sub-channels, each of 32 or more
constexpr int kDdRows = 8;             // rows loaded at a time; a run is a multiple of them
static_assert(kSub % kDdRows == 0, "a channel's sub-channels are whole loads");

template <int kR>
__global__ void __launch_bounds__(kDdThreads, kR == 1 ? 4 : 0) dedisperse_kernel(const float* __restrict__ in,
                                                                  const int* __restrict__ delays, int n_sub, long long nf,
                                                                  long long n_out, int wt, int groups, int parts,
                                                                  float* __restrict__ out) {
    extern __shared__ float run_s[];     // [..][kR][wt]: sum of the first group's runs, then of each other run
    const int g = threadIdx.x / wt, c = threadIdx.x - g * wt;     // wt is a multiple of 32
    const long long t0 = (long long)blockIdx.x * (kR * wt) + c;
    const int beam = blockIdx.y;
    bool in_range[kR];
#pragma unroll
    for (int r = 0; r < kR; ++r) in_range[r] = t0 + r * wt < n_out;
    auto first = [&](int q) { return n_sub / kDdRows * q / parts * kDdRows; };   // first sub-channel of run q
    const int own = parts / groups;                               // runs of the first group
    int q = parts * g / groups, s = first(q);
    const int q1 = parts * (g + 1) / groups;
    const float* row = in + ((long long)beam * n_sub + s) * nf + t0;
#pragma unroll 1
    for (; q < q1; ++q) {
        const int s1 = first(q + 1);
        float acc[kR];
#pragma unroll
        for (int r = 0; r < kR; ++r) acc[r] = 0.f;
#pragma unroll 1
        for (; s < s1; s += kDdRows, row += kDdRows * nf) {
            int d[kDdRows];
#pragma unroll
            for (int k = 0; k < kDdRows; k += 4)
                *reinterpret_cast<int4*>(d + k) = __ldg(reinterpret_cast<const int4*>(delays + s + k));
            float v[kDdRows][kR];
#pragma unroll
            for (int k = 0; k < kDdRows; ++k) {
                const float* p = row + k * nf + d[k];
#pragma unroll
                for (int r = 0; r < kR; ++r) v[k][r] = in_range[r] ? __ldg(p + r * wt) : 0.f;
            }
#pragma unroll
            for (int k = 0; k < kDdRows; ++k)
#pragma unroll
                for (int r = 0; r < kR; ++r) acc[r] += v[k][r];
        }
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            float* to = run_s + (max(0, q - own + 1) * kR + r) * wt + c;
            *to = q > 0 && q < own ? *to + acc[r] : acc[r];
        }
    }
    __syncthreads();
    for (int r = g; r < kR; r += groups) {
        if (t0 + r * wt >= n_out) continue;
        float sum = run_s[r * wt + c];
        for (int k = 1; k <= parts - own; ++k) sum += run_s[(k * kR + r) * wt + c];
        out[(long long)beam * n_out + t0 + r * wt] = sum;
    }
}

// Delay table of the allocation-free dedispersion entry point: one array per
// device, shared by every plan of the process (see bf_dedisperse_static).
__device__ __align__(256) int g_dd_delays[kDdStaticMaxSub];


// FP32 FMA-pipe probe: every thread runs kProbeChains independent chains of
// packed (FFMA2) or scalar FMAs, so the pipe, not latency, sets the rate.  The
// chains converge to c / (1 - b) and stay finite; their sum is stored so that
// no FMA can be removed.
constexpr int kProbeThreads = 256;
constexpr int kProbeChains = 16;

template <bool kPair>
__global__ void __launch_bounds__(kProbeThreads) fma_probe_kernel(long long iters, float* __restrict__ sink) {
    float2 a[kProbeChains];
    const float t = 1e-3f * (float)(threadIdx.x & 31);
#pragma unroll
    for (int k = 0; k < kProbeChains; ++k) a[k] = make_float2(t + (float)k, t - (float)k);
    const float2 b = make_float2(0.9999f, 0.99991f), c = make_float2(1e-4f, 2e-4f);
#pragma unroll 1
    for (long long i = 0; i < iters; i += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int k = 0; k < kProbeChains; ++k) {
                if constexpr (kPair) {
                    a[k] = __ffma2_rn(a[k], b, c);
                } else {
                    a[k].x = __fmaf_rn(a[k].x, b.x, c.x);
                    a[k].y = __fmaf_rn(a[k].y, b.y, c.y);
                }
            }
        }
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kProbeChains; ++k) s += a[k].x + a[k].y;
    sink[(long long)blockIdx.x * kProbeThreads + threadIdx.x] = s;
}

}  // namespace

cudaError_t dedisperse_static_table(int device, int** table) {
    static std::mutex mu;
    static int* ptrs[kMaxDevices] = {};
    if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!ptrs[device]) {
        // once per device, with that device current (the caller has set it)
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_dd_delays);
        if (e != cudaSuccess) return e;
        ptrs[device] = static_cast<int*>(p);
    }
    *table = ptrs[device];
    return cudaSuccess;
}

cudaError_t dedisperse_launch(const float* in, const int* delays, int n_sub, long long nf, long long n_out,
                              float* out, cudaStream_t s) {
    if (n_out <= 0) return cudaSuccess;
    // tiles of equal width up to 1024 frames, up to 256 threads along them
    const long long tiles = (n_out + 1023) / 1024, width = (n_out + tiles - 1) / tiles;
    const int r = (int)((width + 255) / 256), wt = (int)(((width + r - 1) / r + 31) / 32 * 32);
    // groups: as many as fill the CTA, fewer where that leaves the longest share of the runs as it is
    const int parts = std::max(1, std::min(kDdParts, n_sub / 32)), most = std::min(kDdThreads / wt, parts);
    const int share = (parts + most - 1) / most, groups = (parts + share - 1) / share;
    const dim3 grid((unsigned)((n_out + r * wt - 1) / (r * wt)), kBeams);
    const size_t smem = (size_t)(parts - parts / groups + 1) * r * wt * sizeof(float);   // at most 45 KB: 11 sums of 1024 frames
    auto kernel = r == 1 ? dedisperse_kernel<1> : r == 2 ? dedisperse_kernel<2> : r == 3 ? dedisperse_kernel<3> : dedisperse_kernel<4>;
    kernel<<<grid, wt * groups, smem, s>>>(in, delays, n_sub, nf, n_out, wt, groups, parts, out);
    return cudaGetLastError();
}

cudaError_t skymap_launch(const float* in, int n_beams, long long per_beam, float* map, cudaStream_t s) {
    if (n_beams <= 0) return cudaSuccess;
    skymap_kernel<<<n_beams, kMapThreads, 0, s>>>(in, per_beam, map);
    return cudaGetLastError();
}

cudaError_t fma_probe_launch(bool paired, long long iters, float* sink, long long n_sink, int sms, double* flop,
                             cudaStream_t s) {
    const long long blocks = std::min<long long>(4LL * sms, n_sink / kProbeThreads);
    if (blocks <= 0 || iters <= 0) return cudaErrorInvalidValue;
    const long long it4 = (iters + 3) / 4 * 4;
    *flop = (double)blocks * kProbeThreads * (double)it4 * kProbeChains * 4.0;
    if (paired)
        fma_probe_kernel<true><<<(unsigned)blocks, kProbeThreads, 0, s>>>(it4, sink);
    else
        fma_probe_kernel<false><<<(unsigned)blocks, kProbeThreads, 0, s>>>(it4, sink);
    return cudaGetLastError();
}

cudaError_t rescale_u8_launch(const float* in, long long rows, long long nf, uint8_t* codes, float* stats,
                              cudaStream_t s) {
    if (rows <= 0 || nf <= 0) return cudaSuccess;
    const long long ctas = (rows + kU8Rows - 1) / kU8Rows;
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;                  // more than any memory holds
    const bool vec = (nf & 3) == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0 && (reinterpret_cast<uintptr_t>(codes) & 3) == 0;
    const int chunk = nf <= kU8Whole ? (int)nf : kU8Chunk;
    const size_t smem = (size_t)kU8Rows * u8_stride(chunk) * sizeof(float);
    // more shared memory than a launch gets by default, once per device (rows of 2^31 frames go in chunks)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    static std::once_flag once[kMaxDevices];
    static cudaError_t result[kMaxDevices];
    std::call_once(once[dev], [&] {
        const int most = (int)(kU8Rows * u8_stride(kU8Whole) * sizeof(float));
        result[dev] = cudaFuncSetAttribute(rescale_u8_kernel<true, int>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (result[dev] == cudaSuccess)
            result[dev] = cudaFuncSetAttribute(rescale_u8_kernel<false, int>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    });
    if (result[dev] != cudaSuccess) return result[dev];
    if (nf + kU8Chunk > 0x7fffffffLL) {
        auto kernel = vec ? rescale_u8_kernel<true, long long> : rescale_u8_kernel<false, long long>;
        kernel<<<(unsigned)ctas, kU8Threads, smem, s>>>(in, rows, nf, chunk, codes, stats);
    } else {
        auto kernel = vec ? rescale_u8_kernel<true, int> : rescale_u8_kernel<false, int>;
        kernel<<<(unsigned)ctas, kU8Threads, smem, s>>>(in, rows, (int)nf, chunk, codes, stats);
    }
    return cudaGetLastError();
}

}  // namespace chimebf
