// The denoiser over one padded line of pixels, for images of any width: the forward
// layers of widths 32, 64 and 128 and every backward contraction on the tensor cores,
// the forward layers of other widths on the FP32 pipe.
//
// Layout.  All slices of a layer form one line of pixels: slice b, row y, column x
// sits at q = (b (H + 1) + y) Wp + x with Wp = W + 1 (or up to 3 more), so every row
// is followed by a zero column and every slice by a zero row, which serve as the zero
// padding of both neighbours.  A 3 x 3 convolution is then nine shifts of the line,
//     out[q] = sum over ky, kx of W[ky][kx] in[q + (ky - 1) Wp + (kx - 1)],
// whatever W and H are.  Channels are stored in planes of 8 (16 bytes per pixel):
// plane c holds channels 8c .. 8c + 7 of every pixel.  That is the tensor core's
// unswizzled operand layout (8 rows x 16 bytes = one contiguous core matrix), whose
// descriptors may start at any pixel, so one staged copy of the line serves all
// nine taps (the swizzled layouts need a copy per column shift), and staging is
// plain contiguous bulk copies.
//
// The padding costs (W + 1)(H + 1) / (W H): 1.03 at 64 x 64, 1.02 at 83 x 83.
#include <cuda_bf16.h>

#include "kernels.cuh"
#include "ptx.cuh"

namespace cpi {
namespace {

constexpr int kMaxTiles = 4;                // 128-pixel tiles per unit
constexpr int kLineRound = 1024;            // the longest unit of any pass (512 on the tensor cores)
// Positions: below, units of one tile (which lines under 304 x 256 positions, two units
// per SM, take for their speed anyway) and margins of 128, not 512 positions, so that
// small images' lines fit the workspace.
constexpr uint32_t kShortLine = 1u << 15;
constexpr int kMaxStages = 4;
constexpr int kConvThreads = 320;           // warp 0 copies, warp 1 issues MMAs, warps 2..9 epilogue
constexpr int kEpiThreads = 256;
constexpr size_t kSmemMax = 227 * 1024;
constexpr int kStackThreads = 256;

// Elements of one layer's prepared weights, bf16 [tap][plane][output channel][8].
constexpr int weight_elems(int kc, int nout) { return 9 * kc * nout * 8; }
constexpr int kW0Elems = weight_elems(2, 32), kW1Elems = weight_elems(4, 32), kW3Elems = weight_elems(4, 16);
constexpr int kWFwdElems = kW0Elems + 2 * kW1Elems + kW3Elems;
constexpr int kWAllElems = kWFwdElems + 2 * kW1Elems;      // training: + the input gradients' weights of layers 1, 2

// Parameter offsets in the model blob.
constexpr int64_t kPW0 = 0, kPB0 = kPW0 + 32 * 9 * 9, kPW1 = kPB0 + 32, kPB1 = kPW1 + 32 * 32 * 9, kPW2 = kPB1 + 32,
                  kPB2 = kPW2 + 32 * 32 * 9, kPW3 = kPB2 + 32, kPB3 = kPW3 + 32 * 9;
static_assert(kPB3 + 1 == kDenoiserParams, "model blob layout");

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// Shared-memory matrix descriptor without swizzle: core matrices of 8 rows x 16
// bytes (128 contiguous bytes); lbo / sbo in bytes.  K-major: lbo = next core
// matrix along K, sbo = next 8 rows along M / N.
__device__ __forceinline__ uint64_t sdesc_plain(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1u << 46;
    return d;
}

struct Pixel {
    uint32_t b, y, x;
    bool valid;         // an image pixel (not padding)
};
__device__ __forceinline__ Pixel pixel_of(uint32_t q, const DnFlat& g) {
    const uint32_t row = q / (uint32_t)g.Wp;
    const uint32_t b = row / (uint32_t)(g.H + 1);
    Pixel p;
    p.x = q - row * (uint32_t)g.Wp;
    p.b = b;
    p.y = row - b * (uint32_t)(g.H + 1);
    p.valid = q < g.Q && p.x < (uint32_t)g.W && p.y < (uint32_t)g.H;
    return p;
}

// The buffers whose margins the stack kernel clears: up to 7 of up to 4 planes.
struct Margins {
    uint8_t* buf[7];
    int n;
};

// A gradient delta (FP32) as two bf16 terms, hi = bf16(delta) and lo = bf16(delta -
// hi) (the difference is exact), so hi + lo is delta within 2^-17 and every product
// with a bf16 value is exact in FP32.  Eight channels to one 16-byte word of each.
__device__ __forceinline__ void split8(const float* v, uint4& hi, uint4& lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * j]), h1 = __float2bfloat16_rn(v[2 * j + 1]);
        const __nv_bfloat16 l0 = __float2bfloat16_rn(v[2 * j] - __bfloat162float(h0));
        const __nv_bfloat16 l1 = __float2bfloat16_rn(v[2 * j + 1] - __bfloat162float(h1));
        h[j] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
        l[j] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}
// One position's gradient at y: three bf16 terms that add up to it (the tensor core's
// first channels) and the FP32 value.
__device__ __forceinline__ uint4 dy_record(float dy) {
    const __nv_bfloat16 t0 = __float2bfloat16_rn(dy);
    const float r1 = dy - __bfloat162float(t0);
    const __nv_bfloat16 t1 = __float2bfloat16_rn(r1);
    const __nv_bfloat16 t2 = __float2bfloat16_rn(r1 - __bfloat162float(t1));
    return make_uint4((uint32_t)__bfloat16_as_ushort(t0) | ((uint32_t)__bfloat16_as_ushort(t1) << 16),
                      (uint32_t)__bfloat16_as_ushort(t2), __float_as_uint(dy), 0u);
}
// v[j] = 0 where the activation (8 bf16 in m, never negative) is not positive
__device__ __forceinline__ void mask8(float* v, const uint4& m) {
    const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!(__uint_as_float(w[j] << 16) > 0.0f)) v[2 * j] = 0.0f;
        if (!(__uint_as_float(w[j] & 0xffff0000u) > 0.0f)) v[2 * j + 1] = 0.0f;
    }
}

// ------------------------------------------------------------------ scale, input stack, weights
// Per-block sums of squares in float64 (n_blocks partials, summed in a fixed order
// by the consumer).
__global__ void __launch_bounds__(512) dnf_sumsq_kernel(const float* __restrict__ g, int64_t n,
                                                        double* __restrict__ part) {
    dep_wait();
    dep_launch();
    __shared__ double red[512];
    double acc = 0.0;
    const int64_t step = (int64_t)gridDim.x * 512;
    int64_t i = (int64_t)blockIdx.x * 512 + threadIdx.x;
    for (; i + 3 * step < n; i += 4 * step) {   // four loads in flight
        const float v0 = g[i], v1 = g[i + step], v2 = g[i + 2 * step], v3 = g[i + 3 * step];
        acc += (double)v0 * (double)v0;
        acc += (double)v1 * (double)v1;
        acc += (double)v2 * (double)v2;
        acc += (double)v3 * (double)v3;
    }
    for (; i < n; i += step) acc += (double)g[i] * (double)g[i];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = 256; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// First blocks: the stacked input, one thread per position of the line with its
// margins: bf16(Gamma[nb(b, c)] s) for the 9 slices of the angular neighbourhood
// (zero outside the angular grid; channels 9..15 zero), zeros in the padding; and
// zeros into the front and back margins of the other buffers.  s = 1 / rms from
// the kSumBlocks partial sums, formed by every block in the same order.
// Remaining blocks: the weights of the four layers, rounded to bf16, as
// [tap][plane][output channel][8 input channels] (layer 0: 2 planes, channels 9..15
// zero; last layer: 16 output channels, all but the first zero).
__global__ void __launch_bounds__(kStackThreads) dnf_stack_kernel(
    const DnFlat g, const float* __restrict__ gamma, const double* __restrict__ part, int nparts, int64_t n, int hb,
    int wb, const float* __restrict__ model, int stack_blocks, float* __restrict__ scale_out, uint8_t* __restrict__ xin,
    const Margins mg, int w_elems, __nv_bfloat16* __restrict__ wt) {
    dep_wait();
    dep_launch();
    part = after_wait(part);
    if ((int)blockIdx.x >= stack_blocks) {
        const int i = ((int)blockIdx.x - stack_blocks) * kStackThreads + (int)threadIdx.x;
        if (i >= w_elems) return;
        if (i >= kWFwdElems) {   // input gradients of layers 1, 2: flipped taps, input and output channels swapped
            const int l = (i - kWFwdElems) / kW1Elems, r = (i - kWFwdElems) % kW1Elems;
            const int e = r & 7, ci = (r >> 3) % 32, c = (r >> 8) % 4, tap = r >> 10;
            wt[i] = __float2bfloat16_rn(model[(l == 0 ? kPW1 : kPW2) + ((int64_t)(8 * c + e) * 32 + ci) * 9 + (8 - tap)]);
            return;
        }
        int r = i, kc = 4, nout = 32, cin = 32, cout = 32;
        int64_t base = 0;
        if (r < kW0Elems) {
            kc = 2;
            cin = 9;
        } else if ((r -= kW0Elems) < kW1Elems) {
            base = kPW1;
        } else if ((r -= kW1Elems) < kW1Elems) {
            base = kPW2;
        } else {
            r -= kW1Elems;
            base = kPW3;
            nout = 16;
            cout = 1;
        }
        const int e = r & 7, co = (r >> 3) % nout, c = (r >> 3) / nout % kc, tap = (r >> 3) / (nout * kc);
        const int ci = 8 * c + e;
        wt[i] = __float2bfloat16_rn(ci < cin && co < cout ? model[base + ((int64_t)co * cin + ci) * 9 + tap] : 0.0f);
        return;
    }
    __shared__ double red[kStackThreads];
    double t = 0.0;
    for (int i = threadIdx.x; i < nparts; i += kStackThreads) t += part[i];
    red[threadIdx.x] = t;
    __syncthreads();
    for (int s = kStackThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    const double ms = red[0] / (double)n;
    const float s = ms > 0.0 ? (float)(1.0 / sqrt(ms)) : 1.0f;
    if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = s;

    const int64_t HW = (int64_t)g.H * g.W;
    for (int64_t i = (int64_t)blockIdx.x * kStackThreads + threadIdx.x; i < g.PL;
         i += (int64_t)stack_blocks * kStackThreads) {
        const int64_t qs = i - g.G;
        const Pixel p = pixel_of(qs < 0 ? 0xffffffffu : (uint32_t)qs, g);
        uint32_t pk[5] = {0u, 0u, 0u, 0u, 0u};
        if (p.valid) {
            const int br = (int)p.b / wb, bc = (int)p.b - br * wb;
            const float* src = gamma + (int64_t)p.b * HW + (int64_t)p.y * g.W + p.x;
#pragma unroll
            for (int c = 0; c < 9; ++c) {
                const int dr = c / 3 - 1, dc = c % 3 - 1;
                const bool in = br + dr >= 0 && br + dr < hb && bc + dc >= 0 && bc + dc < wb;
                const float v = in ? src[((int64_t)dr * wb + dc) * HW] * s : 0.0f;
                const uint32_t u = __bfloat16_as_ushort(__float2bfloat16_rn(v));
                pk[c / 2] |= (c & 1) ? (u << 16) : u;
            }
        }
        const int64_t plane = g.PL * 16;
        *reinterpret_cast<uint4*>(xin + i * 16) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        *reinterpret_cast<uint4*>(xin + plane + i * 16) = make_uint4(pk[4], 0u, 0u, 0u);
        if (qs < 0 || qs >= (int64_t)g.Q)
            for (int k = 0; k < mg.n; ++k)
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4*>(mg.buf[k] + c * plane + i * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
}

// ------------------------------------------------------------------ convolution
// One layer, persistent: a CTA per SM walks the units of U = 128 T consecutive
// pixels of the line.  Warp 0 (one thread) stages the weights once and then, per
// unit, the line from one row above to one row below (the three bands of U + 2
// pixels a row apart: one contiguous copy per plane, or three when a row is longer
// than a unit); warp 1 (one lane of it) issues per tile of 128 pixels 9 taps x KC / 2
// MMAs (M = 128 pixels, N = NOUT channels, K = 16) into one of two TMEM
// accumulators and frees the stage; warps 2..9 drain the other accumulator:
//   kHidden: bias, ReLU, bf16, planes (zeros in the padding);
//   kInfer (last layer): y = x[4] + sum + bias, divided by the scale, to the image;
//   kTrain (last layer): e = y - s target; the record of dy = 2 e / count (hi, lo
//     bf16 and the FP32 value) and this CTA's sums of e^2 and dy;
//   kGrad: input gradient of a hidden layer.  The 8 staged planes are the 4 hi and
//     the 4 lo planes of the gradient at its output, both multiplied by the same
//     (flipped) weights; the sums are masked by the activation > 0 and split again,
//     hi over the activation itself, and this CTA's per-channel sums kept.  kLoFirst:
//     all lo terms are summed before the hi ones, so that half of the truncated
//     additions find a small sum: against 64 bits the first layer's weight gradients
//     come to 0.9998 of the error of FP32 sums, in the order of the taps to 1.0031 (28
//     training steps of widths 24 to 128; 588 -> 594 us at 32x32 vs 30x30).  Images 64
//     wide keep the order of the taps.
// Every wait is bounded; on a time-out the CTA records it, drains its own copies
// and MMAs, frees its tensor memory and stops.
//
// What bounds it: an MMA of N = 32 is limited by reading A (128 x 16 bf16) from
// shared memory (55 cycles each), and a hidden layer moves 128 bytes per pixel
// through HBM (1024 slices of 64 x 64: 115 us, 0.50 GB at 4.3 TB/s; 175 us with the
// MMAs issued by a diverged lane).  Units of 512 pixels, so that the row before and
// after adds a quarter to what is staged; 8 epilogue warps drain two tiles at a time.
enum Mode { kHidden, kInfer, kTrain, kGrad };

struct ConvArgs {
    const uint8_t* in;            // planes 0..3 (kGrad: hi)
    const uint8_t* in_lo;         // kGrad: lo planes
    const uint8_t* wt;
    const float* bias;
    uint8_t* out;                 // kHidden: planes; kGrad: hi planes, which hold the activation; kTrain: records
    uint8_t* out_lo;              // kGrad
    const float* gamma;           // last layer: the network's input (y_out may be the same buffer)
    const float* target;          // kTrain
    const float* scale;
    float* y_out;                 // kInfer
    double* loss_part;            // kTrain: per CTA
    float* bias_part;             // kTrain: [CTA][32] (first entry used); kGrad: [CTA][32]
    float inv;                    // kTrain: 2 / count
    int stages;
    unsigned int* status;
    unsigned long long timeout_ns;
};

template <int KC, int NOUT, int MODE, bool kLoFirst>
__global__ void __launch_bounds__(kConvThreads, 1) dnf_conv_kernel(const DnFlat g, const ConvArgs a) {
    constexpr bool kLast = MODE == kInfer || MODE == kTrain;
    constexpr int KW = KC == 8 ? 4 : KC;                       // planes of the weights
    constexpr uint32_t kWBytes = (uint32_t)weight_elems(KW, NOUT) * 2;
    constexpr uint32_t kCols = 2 * kMaxTiles * NOUT;           // two accumulators
    extern __shared__ uint8_t smem_dn[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dn) + 127) & ~(uintptr_t)127);
    uint8_t* sw = sm;
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + kWBytes);
    uint64_t* empty = full + kMaxStages;
    uint64_t* tfull = empty + kMaxStages;
    uint64_t* tempty = tfull + 2;
    uint64_t* wbar = tempty + 2;
    uint64_t* drain = wbar + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint8_t* ring = sm + kWBytes + 128;
    const uint32_t plane_s = (uint32_t)g.SP * 16u;              // staged bytes per plane
    const uint32_t stage_bytes = KC * plane_s;
    const int U = g.T * 128, stages = a.stages;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    unsigned int* const status = a.status;
    const unsigned long long timeout_ns = a.timeout_ns;

    if (tid == 0) {
        for (int k = 0; k < kMaxStages; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&tfull[k], 1);
            mbar_init(&tempty[k], kEpiThreads);
        }
        mbar_init(wbar, 1);
        mbar_init(drain, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kCols);
        tmem_relinquish();
    }
    dep_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    dep_launch();      // after the allocation is held (ptx.cuh)
    const uint32_t tmem_base = *tmem_slot;

    float bsum[MODE == kGrad ? 32 : 1];                         // epilogue: sums over this thread's pixels
    double lsum = 0.0;
#pragma unroll
    for (int i = 0; i < (MODE == kGrad ? 32 : 1); ++i) bsum[i] = 0.0f;

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------ copies
            mbar_arrive_expect_tx(wbar, kWBytes);
            bulk_load(sw, a.wt, kWBytes, wbar);
            uint32_t k = 0;   // units issued
            bool ok = true;
            for (int u = blockIdx.x; u < g.n_units; u += gridDim.x, ++k) {
                const int s = (int)(k % (uint32_t)stages);
                if (!mbar_wait_bounded(&empty[s], ((k / (uint32_t)stages) & 1u) ^ 1u, abort_flag, status, timeout_ns)) {
                    ok = false;
                    break;
                }
                mbar_arrive_expect_tx(&full[s], stage_bytes);
                // first pixel needed: one row and one column before the unit
                const int64_t first = (g.G + (int64_t)u * U - g.Wp - 1) * 16;
                uint8_t* dst = ring + (size_t)s * stage_bytes;
                for (int c = 0; c < KC; ++c, dst += plane_s) {
                    const uint8_t* src = (c < 4 ? a.in + c * g.PL * 16 : a.in_lo + (c - 4) * g.PL * 16) + first;
                    if (g.Wp <= U + 2) {
                        bulk_load(dst, src, plane_s, &full[s]);
                    } else {
                        for (int ky = 0; ky < 3; ++ky)
                            bulk_load(dst + (size_t)ky * (U + 2) * 16, src + (int64_t)ky * g.Wp * 16,
                                      (uint32_t)(U + 2) * 16u, &full[s]);
                    }
                }
            }
            if (!ok || *abort_flag) {   // copies of this thread still in flight land before the CTA ends
                mbar_wait_bounded(wbar, 0, nullptr, nullptr, timeout_ns);
                for (uint32_t j = k > (uint32_t)stages ? k - stages : 0u; j < k; ++j)
                    mbar_wait_bounded(&full[j % (uint32_t)stages], (j / (uint32_t)stages) & 1u, nullptr, nullptr,
                                      timeout_ns);
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer (whole warp, one lane issues)
        constexpr uint32_t idesc = idesc_bf16(128, NOUT);
        const uint32_t on = elect_one() ? 1u : 0u;
        bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(wbar, 0, abort_flag, status, timeout_ns)), any = false;
        const uint64_t bd0 = sdesc_plain(smem_u32(sw), NOUT * 16, 128);
        int s = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        for (int u = blockIdx.x; ok && u < g.n_units; u += gridDim.x) {
            ok = mbar_wait_bounded(&tempty[acc], acc_phase ^ 1, abort_flag, status, timeout_ns) &&
                 mbar_wait_bounded(&full[s], phase, abort_flag, status, timeout_ns);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint64_t ad0 = sdesc_plain(smem_u32(ring + (size_t)s * stage_bytes), plane_s, 128);
            for (int t = 0; t < g.T; ++t) {
                const uint32_t d = tmem_base + (uint32_t)(acc * kMaxTiles + t) * NOUT;
                constexpr int kPart = kLoFirst ? KW : KC;       // planes summed tap by tap
#pragma unroll
                for (int i = 0; i < 9 * KC / kPart; ++i) {
                    const int tap = i % 9, plane = KC - kPart - i / 9 * kPart;
                    // descriptor addresses count 16-byte units: one pixel each
                    const uint64_t ad = ad0 + (uint64_t)(uint32_t)(tap / 3 * g.bstride + tap % 3 + t * 128);
#pragma unroll
                    for (int h = 0; h < kPart / 2; ++h)
                        umma_bf16(on, d, ad + (uint64_t)((uint32_t)(plane + 2 * h) * (uint32_t)g.SP),
                                       bd0 + (uint64_t)((tap * KW + 2 * h % KW) * NOUT), idesc, (i | h) ? 1u : 0u);
                }
            }
            any = true;
            umma_commit(on, &empty[s]);
            umma_commit(on, &tfull[acc]);
            if (++s == stages) {
                s = 0;
                phase ^= 1;
            }
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1;
            }
        }
        if (!ok && any) {   // the MMAs issued must finish before the tensor memory is freed
            umma_commit(on, drain);
            mbar_wait_bounded(drain, 0, nullptr, nullptr, timeout_ns);
        }
    } else {
        // ---------------------------------------------------------- epilogue
        const int quarter = warp & 3;                             // TMEM lane quarter of this warp
        const int half = (warp - 2) >> 2;                         // tiles half, half + 2, ...
        const int64_t HW = (int64_t)g.H * g.W;
        const float sc = kLast ? __ldg(after_wait(a.scale)) : 1.0f;
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int u = blockIdx.x; u < g.n_units; u += gridDim.x) {
            if (!mbar_wait_bounded(&tfull[acc], acc_phase, abort_flag, status, timeout_ns)) break;
            tc_fence_after();
            const uint32_t d0 = tmem_base + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(acc * kMaxTiles * NOUT);
#pragma unroll 1
            for (int t = half; t < g.T; t += 2) {
                const uint32_t q = (uint32_t)u * (uint32_t)U + (uint32_t)(t * 128 + 32 * quarter + lane);
                const Pixel p = pixel_of(q, g);
                const int64_t at = (g.G + (int64_t)q) * 16;
                if constexpr (kLast) {
                    uint32_t r[16];
                    tmem_ld_32x32b_x16(d0 + (uint32_t)(t * NOUT), r);
                    tmem_ld_wait();
                    float dy = 0.0f;
                    if (p.valid) {
                        const int64_t o = (int64_t)p.b * HW + (int64_t)p.y * g.W + p.x;
                        const float xcen = bf16r(a.gamma[o] * sc);
                        const float y = xcen + (__uint_as_float(r[0]) + __ldg(a.bias));
                        if constexpr (MODE == kInfer) {
                            a.y_out[o] = y / sc;
                        } else {
                            const float e = y - __ldg(a.target + o) * sc;
                            dy = e * a.inv;
                            lsum += (double)e * (double)e;
                        }
                    }
                    if constexpr (MODE == kTrain) {
                        bsum[0] += dy;
                        *reinterpret_cast<uint4*>(a.out + at) = dy_record(dy);
                    }
                } else {
                    uint32_t r[32];
                    tmem_ld_32x32b_x32(d0 + (uint32_t)(t * NOUT), r);
                    uint8_t* dst = a.out + at;
                    if constexpr (MODE == kGrad) {
                        uint4 m[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) m[c] = *reinterpret_cast<const uint4*>(dst + c * g.PL * 16);
                        tmem_ld_wait();
                        uint8_t* dst_lo = a.out_lo + at;
#pragma unroll
                        for (int c = 0; c < 4; ++c, dst += g.PL * 16, dst_lo += g.PL * 16) {
                            float v[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = p.valid ? __uint_as_float(r[8 * c + j]) : 0.0f;
                            mask8(v, m[c]);
#pragma unroll
                            for (int j = 0; j < 8; ++j) bsum[8 * c + j] += v[j];
                            uint4 hi, lo;
                            split8(v, hi, lo);
                            *reinterpret_cast<uint4*>(dst) = hi;
                            *reinterpret_cast<uint4*>(dst_lo) = lo;
                        }
                    } else {
                        tmem_ld_wait();
#pragma unroll
                        for (int c = 0; c < 4; ++c, dst += g.PL * 16) {
                            uint32_t pk[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int co = 8 * c + 2 * j;
                                const float v0 = fmaxf(__uint_as_float(r[co]) + __ldg(a.bias + co), 0.0f);
                                const float v1 = fmaxf(__uint_as_float(r[co + 1]) + __ldg(a.bias + co + 1), 0.0f);
                                pk[j] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v0)) |
                                        ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v1)) << 16);
                                if (!p.valid) pk[j] = 0u;
                            }
                            *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&tempty[acc]);
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1;
            }
        }
    }

    __syncwarp();                                               // warps 0 and 1: lane 0 joins the others
    if constexpr (MODE == kGrad || MODE == kTrain) {   // this CTA's sums: lanes in a fixed butterfly, then the warps
        __shared__ float bred[kEpiThreads / 32][MODE == kGrad ? 32 : 1];
        __shared__ double lred[kEpiThreads / 32];
        if (warp >= 2) {
#pragma unroll
            for (int i = 0; i < (MODE == kGrad ? 32 : 1); ++i) {
                float v = bsum[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) bred[warp - 2][i] = v;
            }
            if constexpr (MODE == kTrain) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
                if (lane == 0) lred[warp - 2] = lsum;
            }
        }
        __syncthreads();
        if (tid < (MODE == kGrad ? 32 : 1)) {
            float v = 0.0f;
            for (int w = 0; w < kEpiThreads / 32; ++w) v += bred[w][tid];
            a.bias_part[blockIdx.x * 32 + tid] = v;
        }
        if (MODE == kTrain && tid == 0) {
            double v = 0.0;
            for (int w = 0; w < kEpiThreads / 32; ++w) v += lred[w];
            a.loss_part[blockIdx.x] = v;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kCols);
    }
}

// ------------------------------------------------------------------ convolution on the FP32 pipe
// The forward layers of widths other than 32, 64 and 128.  The network subtracts
// nearly all of its input, so one hidden activation that rounds to the other
// bfloat16 neighbour moves an output by 0.5%: these widths keep the sums they have
// always had, one FP32 fused multiply-add after the other over (input channel, tap),
// and the kernel only has to feed the pipe.  (Tensor-core sums measured 10.9 times
// the old kernel's speed at 83 x 83 but 1.5 times its error against 64 bits.)
//
// A CTA takes U consecutive positions of the line; every plane of 8 input channels is
// staged as float [channel][position] with the bands above and below (or as three
// separate bands when a row is longer than U).  A thread sums 8 positions (two
// groups of 4, 128 apart, so that its 16-byte loads are free of bank conflicts) x 8
// output channels: channel pairs in the two lanes of packed FP32 registers, so the
// weights come as pairs and a staged value is used for 3 taps x 8 channels.  Bound
// by the FP32 pipe: 288 FMA per position and channel.
// The last layer (1 output channel): 4 positions per thread.
constexpr int kExThreads = 256;

constexpr int ex_unit(int cout) { return cout == 1 ? 1024 : 512; }

template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(kExThreads, 2) dnf_conv_exact_kernel(const DnFlat g, const ConvArgs a,
                                                                       const float* __restrict__ w) {
    dep_wait();
    dep_launch();
    const uint8_t* const planes = after_wait(a.in);
    constexpr int U = ex_unit(COUT), KC = CIN == 9 ? 2 : 4;
    constexpr int WS = COUT == 1 ? 12 : 9 * COUT;               // weights per input channel
    extern __shared__ __align__(16) float sm_ex[];
    float* sw = sm_ex;                                          // [CIN][tap][COUT]
    float* sv = sm_ex + CIN * WS;                               // [8][pitch]
    const int pitch = (g.SP + 3) & ~3;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < CIN * 9 * COUT; i += kExThreads) {
        const int co = i % COUT, tap = i / COUT % 9, ci = i / (9 * COUT);
        sw[ci * WS + tap * COUT + co] = bf16r(w[((int64_t)co * CIN + ci) * 9 + tap]);
    }
    const int pxg = COUT == 1 ? warp : warp & 1, cog = COUT == 1 ? 0 : warp >> 1;
    const int base = pxg * (COUT == 1 ? 128 : 256) + lane * 4;
    const int64_t HW = (int64_t)g.H * g.W;
    const float sc = MODE == kHidden ? 1.0f : __ldg(after_wait(a.scale));
    double lsum = 0.0;
    float bsum = 0.0f;

    for (int u = blockIdx.x; u < g.n_units; u += gridDim.x) {
        f32x2 acc[COUT == 1 ? 1 : 8][4];
        float acc1[4];
#pragma unroll
        for (int i = 0; i < (COUT == 1 ? 1 : 8); ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[i][c] = 0ull;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc1[i] = 0.0f;
        const int64_t first = g.G + (int64_t)u * U - g.Wp - 1;
#pragma unroll 1
        for (int c = 0; c < KC; ++c) {
            __syncthreads();                                    // the previous plane is consumed
            const uint8_t* src = planes + ((int64_t)c * g.PL + first) * 16;
            for (int i = tid; i < g.SP; i += kExThreads) {
                int64_t o = i;
                if (g.Wp > U) {                                 // separate bands of bstride positions
                    const int band = i < g.bstride ? 0 : (i < 2 * g.bstride ? 1 : 2);
                    o = i - band * g.bstride + (int64_t)band * g.Wp;
                }
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + o * 16));
                const uint32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    sv[(2 * j) * pitch + i] = __uint_as_float(r[j] << 16);
                    sv[(2 * j + 1) * pitch + i] = __uint_as_float(r[j] & 0xffff0000u);
                }
            }
            __syncthreads();
            const int nci = CIN - 8 * c < 8 ? CIN - 8 * c : 8;
#pragma unroll 1
            for (int ci = 0; ci < nci; ++ci) {
                const float* vb = sv + ci * pitch + base;
                const float* wr = sw + (8 * c + ci) * WS;
                if constexpr (COUT == 1) {
                    const float4 wa = *reinterpret_cast<const float4*>(wr), wb = *reinterpret_cast<const float4*>(wr + 4);
                    const float wt[9] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w, wr[8]};
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const float4 v0 = *reinterpret_cast<const float4*>(vb + ky * g.bstride);
                        const float2 v1 = *reinterpret_cast<const float2*>(vb + ky * g.bstride + 4);
                        const float v[6] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y};
#pragma unroll
                        for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                            for (int p = 0; p < 4; ++p) acc1[p] = __fmaf_rn(wt[3 * ky + kx], v[p + kx], acc1[p]);
                    }
                } else {
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        f32x2 d[2][6];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float4 v0 = *reinterpret_cast<const float4*>(vb + ky * g.bstride + 128 * h);
                            const float2 v1 = *reinterpret_cast<const float2*>(vb + ky * g.bstride + 128 * h + 4);
                            d[h][0] = pk2(v0.x, v0.x), d[h][1] = pk2(v0.y, v0.y), d[h][2] = pk2(v0.z, v0.z);
                            d[h][3] = pk2(v0.w, v0.w), d[h][4] = pk2(v1.x, v1.x), d[h][5] = pk2(v1.y, v1.y);
                        }
#pragma unroll
                        for (int kx = 0; kx < 3; ++kx) {
                            const ulonglong2* wp = reinterpret_cast<const ulonglong2*>(wr + (3 * ky + kx) * COUT + 8 * cog);
                            const ulonglong2 q0 = wp[0], q1 = wp[1];
                            const f32x2 wv[4] = {q0.x, q0.y, q1.x, q1.y};
#pragma unroll
                            for (int p = 0; p < 8; ++p)
#pragma unroll
                                for (int k = 0; k < 4; ++k) acc[p][k] = fma2(wv[k], d[p >> 2][(p & 3) + kx], acc[p][k]);
                        }
                    }
                }
            }
        }
        if constexpr (COUT == 1) {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const uint32_t q = (uint32_t)u * U + (uint32_t)(base + p);
                const Pixel px = pixel_of(q, g);
                float dy = 0.0f;
                if (px.valid) {
                    const int64_t o = (int64_t)px.b * HW + (int64_t)px.y * g.W + px.x;
                    const float y = bf16r(a.gamma[o] * sc) + (acc1[p] + __ldg(a.bias));
                    if constexpr (MODE == kInfer) {
                        a.y_out[o] = y / sc;
                    } else {
                        const float e = y - __ldg(a.target + o) * sc;
                        dy = e * a.inv;
                        lsum += (double)e * (double)e;
                    }
                }
                if constexpr (MODE == kTrain) {
                    bsum += dy;
                    *reinterpret_cast<uint4*>(a.out + (g.G + (int64_t)q) * 16) = dy_record(dy);
                }
            }
        } else {
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const uint32_t q = (uint32_t)u * U + (uint32_t)(base + (p >> 2) * 128 + (p & 3));
                const bool valid = pixel_of(q, g).valid;
                uint32_t pk[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float v0, v1;
                    unpk2(acc[p][k], v0, v1);
                    v0 = fmaxf(v0 + __ldg(a.bias + 8 * cog + 2 * k), 0.0f);
                    v1 = fmaxf(v1 + __ldg(a.bias + 8 * cog + 2 * k + 1), 0.0f);
                    pk[k] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v0)) |
                            ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v1)) << 16);
                    if (!valid) pk[k] = 0u;
                }
                *reinterpret_cast<uint4*>(a.out + ((int64_t)cog * g.PL + g.G + (int64_t)q) * 16) =
                    make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        }
    }
    if constexpr (MODE == kTrain) {
        __shared__ float bred[kExThreads / 32];
        __shared__ double lred[kExThreads / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            bsum += __shfl_xor_sync(0xffffffffu, bsum, o);
            lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        }
        if (lane == 0) bred[warp] = bsum, lred[warp] = lsum;
        __syncthreads();
        if (tid == 0) {
            float b = 0.0f;
            double l = 0.0;
            for (int k = 0; k < kExThreads / 32; ++k) b += bred[k], l += lred[k];
            a.bias_part[blockIdx.x * 32] = b;
            a.loss_part[blockIdx.x] = l;
        }
    }
}

// ------------------------------------------------------------------ gradient at the last hidden layer
// delta[ci] = (a3[ci] > 0) sum over taps of W3[ci][8 - tap] dy[q + tap], FP32; hi
// over a3 (the mask, read first by the same thread), lo beside it; per-CTA sums.
// One output channel makes this a 9-term sum per channel, not a contraction worth a
// tensor core: two pixels per thread share the weights read from shared memory.
constexpr int kTopThreads = 256;
constexpr int kTopPixels = 2 * kTopThreads;
constexpr int kTopCtas = 4 * kDnMaxCtas;
__global__ void __launch_bounds__(kTopThreads) dnf_top_grad_kernel(const DnFlat g, const uint8_t* __restrict__ rec,
                                                                   const float* __restrict__ w3, uint8_t* a3,
                                                                   uint8_t* __restrict__ lo_out,
                                                                   float* __restrict__ bias_part) {
    dep_wait();
    dep_launch();
    rec = after_wait(rec);
    __shared__ __align__(16) float sw[9][32];
    __shared__ float bred[kTopThreads / 32][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < 288; i += kTopThreads) sw[i / 32][i % 32] = bf16r(w3[(i % 32) * 9 + 8 - i / 32]);
    __syncthreads();
    float bsum[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) bsum[i] = 0.0f;
    const float* dyv = reinterpret_cast<const float*>(rec) + 2;       // the record's FP32 value
    const int64_t end = ((int64_t)g.Q + 127) / 128 * 128;
    for (int64_t q0 = (int64_t)blockIdx.x * kTopPixels; q0 < end; q0 += (int64_t)gridDim.x * kTopPixels) {
        float d[2][9];
        bool live[2], valid[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int64_t q = q0 + k * kTopThreads + tid;
            live[k] = q < end;
            valid[k] = live[k] && pixel_of((uint32_t)q, g).valid;
#pragma unroll
            for (int t = 0; t < 9; ++t) {    // neighbours before the line are 0; those behind it were written as 0
                const int64_t qn = q + (int64_t)(t / 3 - 1) * g.Wp + t % 3 - 1;
                d[k][t] = valid[k] && qn >= 0 ? __ldg(dyv + 4 * (g.G + qn)) : 0.0f;
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float v[2][8];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int j = 0; j < 8; ++j) v[k][j] = 0.0f;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const float4 w0 = *reinterpret_cast<const float4*>(&sw[t][8 * c]);
                const float4 w1 = *reinterpret_cast<const float4*>(&sw[t][8 * c + 4]);
                const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[k][j] = __fmaf_rn(w[j], d[k][t], v[k][j]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!live[k]) continue;
                const int64_t at = ((int64_t)c * g.PL + g.G + q0 + k * kTopThreads + tid) * 16;
                mask8(v[k], *reinterpret_cast<const uint4*>(a3 + at));
#pragma unroll
                for (int j = 0; j < 8; ++j) bsum[8 * c + j] += v[k][j];
                uint4 hi, lo;
                split8(v[k], hi, lo);
                *reinterpret_cast<uint4*>(a3 + at) = hi;
                *reinterpret_cast<uint4*>(lo_out + at) = lo;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        float v = bsum[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) bred[warp][i] = v;
    }
    __syncthreads();
    if (tid < 32) {
        float v = 0.0f;
        for (int w = 0; w < kTopThreads / 32; ++w) v += bred[w][tid];
        bias_part[blockIdx.x * 32 + tid] = v;
    }
}

// ------------------------------------------------------------------ weight gradients
//     dW[co][ci][ky][kx] = sum over q of delta[co][q] in[ci][q + (ky - 1) Wp + (kx - 1)]
// is a contraction over the pixels of the line (delta is 0 in the padding), and the
// planes are its operands as they stand: 8 pixels x 16 bytes are a core matrix with
// the channels contiguous (MN-major).  Per 16 pixels and ky one MMA: M = 128 rows
// (kx, ci): the layer input staged three times, a pixel apart, 8 channels per plane
// (rows past 3 KC x 8 multiply whatever lies behind and are dropped); N = NB columns:
// the hi and lo terms of delta (4 + 4 planes; the last layer: one plane of records,
// columns 0..2); TMEM columns ky NB + n.  Warp 4 (one thread) copies, warp 5 (one
// lane of it) issues, warps 0..3 add every unit's sums to FP32 registers while the next
// unit runs into the other accumulator: tensor-core sums are truncated, so an
// accumulator left to grow over all of a CTA's pixels is biased in proportion to
// their number (measured on the last layer: 7.4e-6 of the gradient at 80x80 vs 12x12
// against 4.6e-7 in FP32).  The last layer's gradients, exact but for these sums, go in
// runs of 64 pixels: over 28 training steps of widths 24 to 128 the error of the whole
// gradient against 64 bits is 0.98 of that of FP32 sums (1.02 at most), with runs of a
// unit it was 1.00 (1.07 at most, always above 1 at widths 32 and 128).
// hold: images 64 wide, whose gradients have been summed in one accumulator to the end
// since before the line, keep that over the same blocks of up to 32 rows of a slice per
// CTA, so that the gradients at that width stay what they were.  It is the less exact
// sum: 5.2e-5 of the gradient from 64 bits at 64x64 vs 32x32, drained per unit 1.0e-6
// (2020 us a step against 2094 with the other widths' order of lo and hi terms, which
// goes with it).  Only the first unit has an accumulator of its own, which makes up for
// the zero column that is summed with every row: 0.972 of the error of the sums over the
// images' own pixels (16 steps; without it 1.011).
// 1024 slices of 64 x 64, 32 -> 32: 192 us, 0.83 GB at 4.3 TB/s.  At the end the CTA
// writes rows (kx, ci) x columns (ky, n) to part[cta].  Every wait is bounded.
constexpr int kWgThreads = 192;
constexpr int kWgMaxStages = 4;
struct WgArgs {
    const uint8_t* in;          // KC planes
    const uint8_t* d_hi;        // NB = 64: 4 planes; NB = 16: the record plane
    const uint8_t* d_lo;
    float* part;
    int U, bstride, SP, stages;
    int n_blocks;               // runs of pixels that CTAs take: U of them, or (hold) rows of one slice
    bool hold;                  // one accumulator for all of a CTA's blocks
    uint32_t slack;             // bytes behind the ring that the dropped rows may touch
    unsigned int* status;
    unsigned long long timeout_ns;
};

// A CTA's way through its blocks, U pixels at a time.
constexpr int kHoldRows = 32;
struct WgWalk {
    int v;               // block
    int64_t q, left;     // first pixel, pixels of the block from there on (a multiple of 16)
    __device__ __forceinline__ void block(const DnFlat& g, const WgArgs& a, int i) {
        v = i;
        if (v >= a.n_blocks) return;
        if (a.hold) {   // the last rows of a slice may run on into its zero row
            const int rows = min(g.H, kHoldRows), per = (g.H + rows - 1) / rows;
            const int b = v / per, y0 = (v - b * per) * rows;
            q = ((int64_t)b * (g.H + 1) + y0) * g.Wp;
            left = ((int64_t)min(rows, g.H - y0) * g.Wp + 15) / 16 * 16;
        } else {        // delta and the input's margin are defined up to the next multiple of 16
            q = (int64_t)v * a.U;
            left = min((int64_t)a.U, ((int64_t)g.Q + 15) / 16 * 16 - q);
        }
    }
    __device__ __forceinline__ bool live(const WgArgs& a) const { return v < a.n_blocks; }
    __device__ __forceinline__ bool last(const WgArgs& a) const { return left <= a.U && v + (int)gridDim.x >= a.n_blocks; }
    __device__ __forceinline__ void next(const DnFlat& g, const WgArgs& a) {
        q += a.U;
        left -= a.U;
        if (left <= 0) block(g, a, v + (int)gridDim.x);
    }
};

// kRun: K steps (16 pixels) per run, 0: a unit's, or all of a CTA's (hold)
template <int KC, int NB, int kRun>
__global__ void __launch_bounds__(kWgThreads, 1) dnf_wgrad_kernel(const DnFlat g, const WgArgs a) {
    constexpr int kDPlanes = NB / 8;                       // staged delta planes (NB = 16: the second stays unused)
    constexpr uint32_t kCols = 3 * NB;
    constexpr uint32_t kTmemCols = NB == 64 ? 512 : 128;   // two accumulators
    constexpr int kRows = 3 * KC * 8, kDrainWarps = (kRows + 31) / 32;
    extern __shared__ uint8_t smem_dn[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dn) + 127) & ~(uintptr_t)127);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm);
    uint64_t* empty = full + kWgMaxStages;
    uint64_t* tfull = empty + kWgMaxStages;
    uint64_t* tempty = tfull + 2;
    uint64_t* drain = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint8_t* ring = sm + 128;
    const uint32_t dplane = (uint32_t)a.U * 16u, aplane = (uint32_t)a.SP * 16u;
    const uint32_t stage_bytes = kDPlanes * dplane + 3 * KC * aplane;
    const int stages = a.stages;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < kWgMaxStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&tfull[k], 1);
            mbar_init(&tempty[k], 32 * kDrainWarps);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 5) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    dep_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    dep_launch();      // after the allocation is held (ptx.cuh)
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 4 && lane == 0) {
        uint32_t k = 0;
        bool ok = true;
        WgWalk w;
        for (w.block(g, a, (int)blockIdx.x); w.live(a); w.next(g, a), ++k) {
            const int s = (int)(k % (uint32_t)stages);
            if (!mbar_wait_bounded(&empty[s], ((k / (uint32_t)stages) & 1u) ^ 1u, abort_flag, a.status, a.timeout_ns)) {
                ok = false;
                break;
            }
            const int64_t at = (g.G + w.q) * 16;
            uint8_t* dst = ring + (size_t)s * stage_bytes;
            mbar_arrive_expect_tx(&full[s], (NB == 64 ? 8u : 1u) * dplane + 3u * KC * aplane);
            for (int c = 0; c < (NB == 64 ? 8 : 1); ++c)
                bulk_load(dst + c * dplane, (c < 4 ? a.d_hi + c * g.PL * 16 : a.d_lo + (c - 4) * g.PL * 16) + at, dplane,
                          &full[s]);
            dst += kDPlanes * dplane;
            for (int kx = 0; kx < 3; ++kx)
                for (int c = 0; c < KC; ++c, dst += aplane) {
                    const uint8_t* src = a.in + c * g.PL * 16 + at + (int64_t)(kx - 1 - g.Wp) * 16;
                    if (g.Wp <= a.U) {
                        bulk_load(dst, src, aplane, &full[s]);
                    } else {
                        for (int ky = 0; ky < 3; ++ky)
                            bulk_load(dst + (size_t)ky * dplane, src + (int64_t)ky * g.Wp * 16, dplane, &full[s]);
                    }
                }
        }
        if (!ok || *abort_flag)
            for (uint32_t j = k > (uint32_t)stages ? k - stages : 0u; j < k; ++j)
                mbar_wait_bounded(&full[j % (uint32_t)stages], (j / (uint32_t)stages) & 1u, nullptr, nullptr, a.timeout_ns);
    } else if (warp == 5) {
        // both operands MN-major
        constexpr uint32_t idesc = idesc_bf16(128, NB) | (1u << 15) | (1u << 16);
        const uint32_t on = elect_one() ? 1u : 0u;
        bool ok = true, any = false;
        int s = 0, acc = 0, units = 0;
        uint32_t phase = 0, acc_phase = 0;
        WgWalk w;
        for (w.block(g, a, (int)blockIdx.x); w.live(a); w.next(g, a), ++units) {
            const bool first = !a.hold || units < 2, last = !a.hold || units == 0 || w.last(a);
            ok = (!first || mbar_wait_bounded(&tempty[acc], acc_phase ^ 1, abort_flag, a.status, a.timeout_ns)) &&
                 mbar_wait_bounded(&full[s], phase, abort_flag, a.status, a.timeout_ns);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const int steps = (int)min(w.left, (int64_t)a.U) / 16;
            const uint32_t base = smem_u32(ring + (size_t)s * stage_bytes);
            uint32_t d = tmem_base + (uint32_t)acc * kCols;
            uint64_t bd = sdesc_plain(base, 128, dplane);
            uint64_t ad = sdesc_plain(base + kDPlanes * dplane, 128, aplane);
            auto sum = [&](int n, bool fresh) {
                for (int k = 0; k < n; ++k, ad += 16, bd += 16) {
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky)
                        umma_bf16(on, d + (uint32_t)(ky * NB), ad + (uint64_t)(uint32_t)(ky * a.bstride), bd, idesc,
                                       fresh && k == 0 ? 0u : 1u);
                }
            };
            if constexpr (kRun == 0) {
                sum(steps, first);
            } else {
                sum(min(kRun, steps), true);
                for (int k = kRun; k < steps; k += kRun) {      // the next run: the other accumulator
                    umma_commit(on, &tfull[acc]);
                    if (++acc == 2) {
                        acc = 0;
                        acc_phase ^= 1;
                    }
                    ok = __all_sync(0xffffffffu,
                                    mbar_wait_bounded(&tempty[acc], acc_phase ^ 1, abort_flag, a.status, a.timeout_ns));
                    if (!ok) break;
                    tc_fence_after();
                    d = tmem_base + (uint32_t)acc * kCols;
                    sum(min(kRun, steps - k), true);
                }
            }
            any = true;
            if (!ok) break;
            umma_commit(on, &empty[s]);
            if (++s == stages) {
                s = 0;
                phase ^= 1;
            }
            if (!last) continue;
            umma_commit(on, &tfull[acc]);
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1;
            }
        }
        if (!ok && any) {   // the MMAs issued must finish before the tensor memory is freed
            umma_commit(on, drain);
            mbar_wait_bounded(drain, 0, nullptr, nullptr, a.timeout_ns);
        }
    } else if (warp < kDrainWarps) {
        float run[kCols];
#pragma unroll
        for (uint32_t c = 0; c < kCols; ++c) run[c] = 0.0f;
        bool ok = true;
        int acc = 0;
        uint32_t acc_phase = 0;
        int left = 0;                                       // K steps of the unit still to come
        WgWalk w;
        w.block(g, a, (int)blockIdx.x);
        bool more = a.hold && !w.last(a);                   // hold: the sums of the units after the first
        for (int v = blockIdx.x; v < a.n_blocks;) {
            if (kRun > 0 && left == 0)
                left = (int)min((int64_t)a.U, ((int64_t)g.Q + 15) / 16 * 16 - (int64_t)v * a.U) / 16;
            if (!mbar_wait_bounded(&tfull[acc], acc_phase, abort_flag, a.status, a.timeout_ns)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem_base + ((uint32_t)(32 * warp) << 16) + (uint32_t)acc * kCols;
#pragma unroll
            for (uint32_t c0 = 0; c0 < kCols; c0 += 16) {
                uint32_t r[16];
                tmem_ld_32x32b_x16(d + c0, r);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) run[c0 + j] += __uint_as_float(r[j]);
            }
            tc_fence_before();
            mbar_arrive(&tempty[acc]);
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1;
            }
            if (a.hold) {
                if (!more) break;
                more = false;
                continue;
            }
            left = kRun > 0 ? max(0, left - kRun) : 0;
            if (left == 0) v += (int)gridDim.x;
        }
        const int row = 32 * warp + lane;
        if (ok && row < kRows) {
            float4* out = reinterpret_cast<float4*>(a.part + ((size_t)blockIdx.x * kRows + row) * kCols);
#pragma unroll
            for (uint32_t c = 0; c < kCols; c += 4) out[c / 4] = make_float4(run[c], run[c + 1], run[c + 2], run[c + 3]);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// The layer's gradients from the per-CTA partials, in a fixed order.  Block (ci,
// tap) < 9 CIN: thread (group of 8, co) adds the terms' columns of its share of
// the CTAs, then the groups are added in order; the last block: the bias sums (and,
// for the last layer, the loss).
template <int CIN, int KC, int COUT>
__global__ void __launch_bounds__(256) dnf_wgrad_reduce_kernel(const float* __restrict__ part, int nparts,
                                                               const float* __restrict__ bias_part, int nbias,
                                                               const double* __restrict__ loss_part, int nloss, int64_t n,
                                                               float* __restrict__ grad, float* __restrict__ loss) {
    dep_wait();
    dep_launch();
    part = after_wait(part);
    bias_part = after_wait(bias_part);
    loss_part = after_wait(loss_part);
    constexpr int NB = COUT == 32 ? 64 : 16, kCols = 3 * NB, kRows = 3 * KC * 8;
    __shared__ float red[8][32];
    const int co = threadIdx.x & 31, grp = threadIdx.x >> 5;
    float s = 0.0f;
    if (blockIdx.x < 9 * CIN) {
        const int ci = blockIdx.x / 9, tap = blockIdx.x % 9;
        const size_t o = (size_t)((tap % 3) * KC * 8 + ci) * kCols + (tap / 3) * NB + co;
        if (co < COUT)
            for (int i = grp; i < nparts; i += 8) {
                const float* p = part + (size_t)i * kRows * kCols + o;
                s += COUT == 32 ? p[0] + p[32] : (p[0] + p[1]) + p[2];
            }
        red[grp][co] = s;
        __syncthreads();
        if (grp == 0 && co < COUT) {
            s = 0.0f;
            for (int k = 0; k < 8; ++k) s += red[k][co];
            grad[((int64_t)co * CIN + ci) * 9 + tap] = s;
        }
        return;
    }
    if (co < COUT)
        for (int i = grp; i < nbias; i += 8) s += bias_part[i * 32 + co];
    red[grp][co] = s;
    __syncthreads();
    if (grp == 0 && co < COUT) {
        s = 0.0f;
        for (int k = 0; k < 8; ++k) s += red[k][co];
        grad[(int64_t)COUT * CIN * 9 + co] = s;
    }
    if (loss != nullptr && grp == 1) {
        double t = 0.0;
        for (int i = co; i < nloss; i += 32) t += loss_part[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (co == 0) *loss = (float)(t / (double)n);
    }
}

// ------------------------------------------------------------------ host
// Short lines gain from kernels placed ahead, on long ones the gaps do not count and the
// placed CTAs cost.  Chained and plain at the tensor-core widths, us: 32x64 vs 8x9 (154
// thousand positions) 56 / 62, 64x64 vs 14x16 (946 thousand) 169 / 171, 32x32 vs 31x32
// (1.08 million) 180 / 182, 64x64 vs 20x20 (1.69 million) 253 / 248, 64x64 vs 32x32 547 /
// 517; training 182 / 209, 569 / 587, 632 / 651, 922 / 936, 2052 / 2029.  The FP32 layers of
// the other widths are launched plainly on any line; two of their CTAs fill an SM.  With
// them chained and not (the rest of the call chained): 24x31 vs 8x8 135 / 117, 30x25 vs
// 9x8 163 / 117, 47x53 vs 10x12 420 / 372, 60x87 vs 12x12 746 / 709, 83x83 vs 12x12 1020 /
// 975, the other way round 94x60 vs 8x8 429 / 441 and 43x58 vs 10x14 426 / 438; training
// 221 / 204, 251 / 207, 617 / 567, 1122 / 1071, 1511 / 1459, 643 / 654, 636 / 646.
bool in_chain(const DnFlat& g) { return g.Q < (1u << 20); }

template <typename K>
cudaError_t allow_smem(K kernel, bool (&done)[64]) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!done[dev]) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax - 2048);
        if (e != cudaSuccess) return e;
        done[dev] = true;
    }
    return cudaSuccess;
}

constexpr size_t kDynMax = kSmemMax - 2048;      // the static sums of the training kernels fit beside it

// Tiles per unit: 512 pixels (a quarter of the staged line is overlap at 64 wide),
// fewer when that would leave SMs without a second unit or two stages do not fit.
template <int KC, int NOUT>
int choose_tiles(const DnFlat& g, int sm_count, size_t* fixed) {
    *fixed = 128 + (size_t)weight_elems(KC == 8 ? 4 : KC, NOUT) * 2 + 128;
    int T = g.Q < kShortLine ? 1 : kMaxTiles;
    while (T > 1 && ((int64_t)g.Q + T * 128 - 1) / (T * 128) < 2 * (int64_t)sm_count) T /= 2;
    for (; T > 1; T /= 2) {
        const int U = T * 128;
        const size_t sp = U + 2 + 2 * (size_t)(g.Wp < U + 2 ? g.Wp : U + 2);
        if (2 * sp * 16 * KC + *fixed <= kDynMax) break;
    }
    return T;
}

template <int KC, int NOUT, int MODE, bool kLoFirst = false>
cudaError_t launch_conv(DnFlat g, ConvArgs a, int sm_count, cudaStream_t st, int* ctas = nullptr) {
    static bool attr[64] = {};
    cudaError_t e = allow_smem(dnf_conv_kernel<KC, NOUT, MODE, kLoFirst>, attr);
    if (e != cudaSuccess) return e;
    size_t fixed = 0;
    g.T = choose_tiles<KC, NOUT>(g, sm_count, &fixed);
    const int U = g.T * 128;
    g.n_units = (int)(((int64_t)g.Q + U - 1) / U);
    g.bstride = g.Wp < U + 2 ? g.Wp : U + 2;
    g.SP = U + 2 + 2 * g.bstride;
    const size_t stage = (size_t)KC * g.SP * 16;
    a.stages = (int)((kDynMax - fixed) / stage);
    if (a.stages > kMaxStages) a.stages = kMaxStages;
    if (a.stages < 2) return cudaErrorInvalidValue;
    const int grid = g.n_units < sm_count ? g.n_units : sm_count;
    if (ctas) *ctas = grid;
    return launch_kernel(in_chain(g), dnf_conv_kernel<KC, NOUT, MODE, kLoFirst>, grid, kConvThreads,
        fixed + a.stages * stage, st, g, a);
}

// The forward layer CIN -> COUT on whichever unit the width takes.
template <int CIN, int COUT, int MODE>
cudaError_t launch_forward(DnFlat g, const ConvArgs& a, const float* w, int sm_count, cudaStream_t st, int* ctas = nullptr) {
    if (g.tensor) return launch_conv<CIN == 9 ? 2 : 4, COUT == 1 ? 16 : 32, MODE>(g, a, sm_count, st, ctas);
    static bool attr[64] = {};
    cudaError_t e = allow_smem(dnf_conv_exact_kernel<CIN, COUT, MODE>, attr);
    if (e != cudaSuccess) return e;
    constexpr int U = ex_unit(COUT);
    g.n_units = (int)(((int64_t)g.Q + U - 1) / U);
    g.bstride = g.Wp <= U ? g.Wp : U + 4;
    g.SP = U + 2 + 2 * g.bstride;
    const size_t smem = sizeof(float) * ((size_t)CIN * (COUT == 1 ? 12 : 9 * COUT) + 8 * (size_t)((g.SP + 3) & ~3));
    int grid = (MODE == kTrain ? 1 : 2) * sm_count;
    if (g.n_units < grid) grid = g.n_units;
    if (ctas) *ctas = grid;
    return launch_kernel(false, dnf_conv_exact_kernel<CIN, COUT, MODE>, grid, kExThreads, smem, st, g, a, w);
}

template <int CIN, int KC, int COUT, int kRun = 0>
cudaError_t launch_wgrad(const DnFlat& g, WgArgs a, const float* bias_part, int nbias, const double* loss_part, int nloss,
                         int64_t n, float* grad, float* loss, int sm_count, cudaStream_t st) {
    constexpr int NB = COUT == 32 ? 64 : 16;
    static bool attr[64] = {};
    cudaError_t e = allow_smem(dnf_wgrad_kernel<KC, NB, kRun>, attr);
    if (e != cudaSuccess) return e;
    // pixels per unit: up to 256 (the staged halo of two rows is shared by more of
    // them), fewer when two stages do not fit or SMs would stay idle
    auto shape = [&](int U) {
        a.U = U;
        a.bstride = g.Wp < U ? g.Wp : U;
        a.SP = U + 2 * a.bstride;
        a.slack = (uint32_t)(16 - 3 * KC) * a.SP * 16;
        return (size_t)(NB / 8) * U * 16 + (size_t)3 * KC * a.SP * 16;
    };
    int U = 256;
    size_t stage = shape(U);
    while (U > 64 && (256 + a.slack + 2 * stage > kDynMax || ((int64_t)g.Q + U - 1) / U < sm_count)) stage = shape(U -= 16);
    if (256 + a.slack + 2 * stage > kDynMax) return cudaErrorInvalidValue;
    a.n_blocks = (int)(((int64_t)g.Q + U - 1) / U);
    if (a.hold) {
        const int rows = g.H < kHoldRows ? g.H : kHoldRows;
        const int len = (rows * g.Wp + 15) / 16, parts = (16 * len + U - 1) / U;     // even parts of a block
        stage = shape(U = (len + parts - 1) / parts * 16);
        a.n_blocks = (int)((int64_t)g.Q / g.Wp / (g.H + 1)) * ((g.H + rows - 1) / rows);
    }
    a.stages = (int)((kDynMax - 256 - a.slack) / stage);
    if (a.stages > kWgMaxStages) a.stages = kWgMaxStages;
    int grid = a.n_blocks < sm_count ? a.n_blocks : sm_count;
    if (grid > kDnMaxCtas) grid = kDnMaxCtas;
    e = launch_kernel(in_chain(g), dnf_wgrad_kernel<KC, NB, kRun>, grid, kWgThreads, 256 + a.stages * stage + a.slack, st, g, a);
    if (e != cudaSuccess) return e;
    return launch_kernel(in_chain(g), dnf_wgrad_reduce_kernel<CIN, KC, COUT>, 9 * CIN + 1, 256, 0, st, a.part, grid,
        bias_part, nbias, loss_part, nloss, n, grad, loss);
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

cudaError_t launch_inputs(const DnFlat& g, const float* gamma_in, const float* model, int hb, int wb, uint8_t* ws,
                          uint8_t* xin, const Margins& mg, int w_elems, int sm_count, cudaStream_t st) {
    const int64_t n = (int64_t)hb * wb * g.H * g.W;
    double* sums = reinterpret_cast<double*>(ws + g.sums);
    const cudaError_t e = launch_kernel(false, dnf_sumsq_kernel, kDnSumBlocks, 512, 0, st, gamma_in, n, sums);
    if (e != cudaSuccess) return e;
    const int64_t want = (g.PL + kStackThreads - 1) / kStackThreads;
    const int sblocks = (int)(want < 16 * (int64_t)sm_count ? want : 16 * (int64_t)sm_count);
    const int wblocks = (w_elems + kStackThreads - 1) / kStackThreads;
    return launch_kernel(in_chain(g), dnf_stack_kernel, sblocks + wblocks, kStackThreads, 0, st, g, gamma_in, sums,
        kDnSumBlocks, n, hb, wb, model, sblocks, reinterpret_cast<float*>(ws + g.scale), xin, mg, w_elems,
        reinterpret_cast<__nv_bfloat16*>(ws + g.wt));
}

}  // namespace

bool dn_flat_plan(int ha, int wa, int hb, int wb, bool training, size_t ws_bytes, DnFlat* out) {
    DnFlat g{};
    g.H = ha;
    g.W = wa;
    g.tensor = wa == 32 || wa == 64 || wa == 128;
    g.Wp = g.tensor ? wa + 1 : (wa + 4) / 4 * 4;      // the FP32 kernel reads its bands as 16-byte words
    const int64_t Q = (int64_t)hb * wb * (ha + 1) * g.Wp;
    if (Q >= ((int64_t)1 << 31) - kLineRound) return false;
    g.Q = (uint32_t)Q;
    g.G = g.Wp + 1;
    // the longest unit of any pass (short lines on the tensor cores run in units of 128)
    const int round = !g.tensor ? kLineRound : (Q < kShortLine ? 128 : kLineRound / 2);
    g.PL = g.G + (Q + round - 1) / round * round + g.Wp + 1;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = up256(o + bytes);
        return at;
    };
    g.scale = take(sizeof(float));
    g.sums = take(sizeof(double) * kDnSumBlocks);
    g.wt = take(sizeof(__nv_bfloat16) * (size_t)(training ? kWAllElems : kWFwdElems));
    if (!training) {
        g.act[0] = take((size_t)g.PL * 64);      // the input (2 planes), later layer 1's output
        g.act[1] = take((size_t)g.PL * 64);
    } else {
        g.xin = take((size_t)g.PL * 32);
        for (int l = 0; l < 3; ++l) g.act[l] = take((size_t)g.PL * 64);
        for (int l = 0; l < 2; ++l) g.lo[l] = take((size_t)g.PL * 64);
        g.rec = take((size_t)g.PL * 16);
        g.part = take(sizeof(float) * (size_t)kDnMaxCtas * 96 * 192);
        g.bpart = take(sizeof(float) * 32 * (size_t)(3 * kDnMaxCtas + kTopCtas));
    }
    *out = g;
    return o <= ws_bytes;
}

cudaError_t dn_flat_denoise(const DnFlat& g, const float* model, const float* gamma_in, float* gamma_out, int hb, int wb,
                            uint8_t* ws, int sm_count, unsigned int* status, unsigned long long timeout_ns,
                            cudaStream_t st) {
    const int64_t n = (int64_t)hb * wb * g.H * g.W;
    uint8_t* x = ws + g.act[0];
    uint8_t* c = ws + g.act[1];
    // The last layer reads the input pixel by pixel as it writes the output, and FP32
    // layers read the model: an output that overlaps them otherwise than in place goes
    // through the workspace.
    auto on = [&](const float* p, int64_t len) { return gamma_out < p + len && p < gamma_out + n; };
    const bool apart = (gamma_out == gamma_in || !on(gamma_in, n)) && !on(model, kDenoiserParams);
    float* y = apart ? gamma_out : reinterpret_cast<float*>(x);
    const uint8_t* wt = ws + g.wt;
    const Margins mg{{x, c}, 2};
    cudaError_t e = launch_inputs(g, gamma_in, model, hb, wb, ws, x, mg, kWFwdElems, sm_count, st);
    ConvArgs a{};
    a.status = status;
    a.timeout_ns = timeout_ns;
    a.in = x, a.out = c, a.wt = wt, a.bias = model + kPB0;
    if (e == cudaSuccess) e = launch_forward<9, 32, kHidden>(g, a, model + kPW0, sm_count, st);
    a.in = c, a.out = x, a.wt = wt + 2 * kW0Elems, a.bias = model + kPB1;
    if (e == cudaSuccess) e = launch_forward<32, 32, kHidden>(g, a, model + kPW1, sm_count, st);
    a.in = x, a.out = c, a.wt += 2 * kW1Elems, a.bias = model + kPB2;
    if (e == cudaSuccess) e = launch_forward<32, 32, kHidden>(g, a, model + kPW2, sm_count, st);
    a.in = c, a.out = nullptr, a.wt += 2 * kW1Elems, a.bias = model + kPB3;
    a.gamma = gamma_in, a.scale = reinterpret_cast<const float*>(ws + g.scale), a.y_out = y;
    if (e == cudaSuccess) e = launch_forward<32, 1, kInfer>(g, a, model + kPW3, sm_count, st);
    if (e == cudaSuccess && !apart)
        e = cudaMemcpyAsync(gamma_out, y, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, st);
    return e;
}

cudaError_t dn_flat_grad(const DnFlat& g, const float* model, const float* gamma_in, const float* gamma_target, int hb,
                         int wb, uint8_t* ws, float* grad, float* loss, int sm_count, unsigned int* status,
                         unsigned long long timeout_ns, cudaStream_t st) {
    const int64_t n = (int64_t)hb * wb * g.H * g.W;
    if (sm_count > kDnMaxCtas) sm_count = kDnMaxCtas;
    uint8_t* x = ws + g.xin;
    uint8_t* act[3] = {ws + g.act[0], ws + g.act[1], ws + g.act[2]};
    uint8_t* lo[2] = {ws + g.lo[0], ws + g.lo[1]};
    uint8_t* rec = ws + g.rec;
    const uint8_t* wt = ws + g.wt;
    double* sums = reinterpret_cast<double*>(ws + g.sums);
    float* bpart[4];
    const int slot[4] = {0, 1, 3, 2};             // layer 2's (kTopCtas of them) last
    for (int l = 0; l < 4; ++l) bpart[l] = reinterpret_cast<float*>(ws + g.bpart) + (size_t)slot[l] * 32 * kDnMaxCtas;
    const Margins mg{{act[0], act[1], act[2], lo[0], lo[1]}, 5};
    cudaError_t e = launch_inputs(g, gamma_in, model, hb, wb, ws, x, mg, kWAllElems, sm_count, st);
    // forward: a1, a2, a3, and the record of the gradient at y
    ConvArgs a{};
    a.status = status;
    a.timeout_ns = timeout_ns;
    a.in = x, a.out = act[0], a.wt = wt, a.bias = model + kPB0;
    if (e == cudaSuccess) e = launch_forward<9, 32, kHidden>(g, a, model + kPW0, sm_count, st);
    a.in = act[0], a.out = act[1], a.wt = wt + 2 * kW0Elems, a.bias = model + kPB1;
    if (e == cudaSuccess) e = launch_forward<32, 32, kHidden>(g, a, model + kPW1, sm_count, st);
    a.in = act[1], a.out = act[2], a.wt += 2 * kW1Elems, a.bias = model + kPB2;
    if (e == cudaSuccess) e = launch_forward<32, 32, kHidden>(g, a, model + kPW2, sm_count, st);
    a.in = act[2], a.out = rec, a.wt += 2 * kW1Elems, a.bias = model + kPB3;
    a.gamma = gamma_in, a.target = gamma_target, a.scale = reinterpret_cast<const float*>(ws + g.scale);
    a.loss_part = sums, a.bias_part = bpart[3], a.inv = 2.0f / (float)n;
    int top = 0, nb[3] = {};
    if (e == cudaSuccess) e = launch_forward<32, 1, kTrain>(g, a, model + kPW3, sm_count, st, &top);
    // backward.  The gradient at hidden layer l's output (masked) takes the place of
    // its activation (hi) once the weight gradient that reads the activation is done.
    WgArgs w{};
    w.hold = g.W == 64;
    w.part = reinterpret_cast<float*>(ws + g.part);
    w.status = status;
    w.timeout_ns = timeout_ns;
    w.in = act[2], w.d_hi = rec;
    if (e == cudaSuccess)
        e = w.hold ? launch_wgrad<32, 4, 1>(g, w, bpart[3], top, sums, top, n, grad + kPW3, loss, sm_count, st)
                   : launch_wgrad<32, 4, 1, 4>(g, w, bpart[3], top, sums, top, n, grad + kPW3, loss, sm_count, st);
    if (e == cudaSuccess) {
        const int64_t blocks = ((int64_t)g.Q + kTopPixels - 1) / kTopPixels;
        nb[2] = (int)(blocks < kTopCtas ? blocks : kTopCtas);
        e = launch_kernel(in_chain(g), dnf_top_grad_kernel, nb[2], kTopThreads, 0, st, g, rec, model + kPW3, act[2],
            lo[0], bpart[2]);
    }
    const uint8_t* wtb = wt + 2 * kWFwdElems;
    for (int l = 2; l >= 1; --l) {
        w.in = act[l - 1], w.d_hi = act[l], w.d_lo = lo[l & 1];
        if (e == cudaSuccess)
            e = launch_wgrad<32, 4, 32>(g, w, bpart[l], nb[l], nullptr, 0, n, grad + (l == 2 ? kPW2 : kPW1), nullptr,
                sm_count, st);
        ConvArgs b{};
        b.status = status;
        b.timeout_ns = timeout_ns;
        b.in = act[l], b.in_lo = lo[l & 1], b.wt = wtb + (size_t)(l - 1) * 2 * kW1Elems;
        b.out = act[l - 1], b.out_lo = lo[(l - 1) & 1], b.bias_part = bpart[l - 1];
        if (e == cudaSuccess)
            e = w.hold ? launch_conv<8, 32, kGrad>(g, b, sm_count, st, &nb[l - 1])
                       : launch_conv<8, 32, kGrad, true>(g, b, sm_count, st, &nb[l - 1]);
    }
    w.in = x, w.d_hi = act[0], w.d_lo = lo[0];
    if (e == cudaSuccess)
        e = launch_wgrad<9, 2, 32>(g, w, bpart[0], nb[0], nullptr, 0, n, grad + kPW0, nullptr, sm_count, st);
    return e;
}

}  // namespace cpi
