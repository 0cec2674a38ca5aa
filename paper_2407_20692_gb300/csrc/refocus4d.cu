// 4-D multilinear refocusing (Section 4.1: the prototype interpolates Gamma in
// all four coordinates, the interpolation points depending on the plane).
// Plane p has four coefficients (alpha, beta, gamma, delta).  For output pixel
// x (centred spatial coordinates) and angular pixel j (centred), Gamma is
// sampled at
//     u_a = alpha x + beta (j in spatial pixels)      (spatial point)
//     u_b = gamma (x in angular pixels) + delta j     (angular point)
// by multilinear interpolation over the 16 neighbouring grid points (taps
// outside either grid count as 0), and the samples are summed over j.
// gamma = 0, delta = 1 is the 2-D refocusing of refocus.cu.
//
// The sample point separates into a column part (x_c, j_c) -> (xa, xb) and a
// row part (x_r, j_r) -> (ya, yb).  Stage 1 contracts the columns: for every
// pair of rows (ya, yb), Gamma restricted to them is a W_b x W_a matrix
// G[xb][xa] (one 2-D box of Gamma's slice-major layout), and
//     C[p][ya][yb][x_c] = sum_{j_c} sum_{xa, xb taps} w w G[xb][xa],
// one CTA per (ya, yb) for every plane of the chunk, the box staged in shared
// memory with a 2-pixel zero border (or read from global memory when it does
// not fit), Kahan-compensated over j_c and stored as a float pair (sum and
// compensation).  Stage 2 contracts the rows (a 1/W_b share of the work) in
// double-float FP32 arithmetic, exact up to one final rounding:
//     out[p][x_r][x_c] = sum_{j_r} sum_{ya, yb taps} w w C[p][ya][yb][x_c].
// Coordinates are 32.32 fixed point, A(x) + B(j), each rounded once from FP64;
// fractions rounded to 24 bits (exact weights).
//
// This file is compiled without FMA contraction (Kahan steps).
#include "kernels.cuh"
#include "ptx.cuh"

namespace cpi {
namespace {

constexpr int kPad = 2;              // zero border of the staged box
constexpr int kR4Threads = 256;

constexpr long long kXBias = 128ll + ((long long)kPad << 32);

__device__ __forceinline__ long long r4_fix(double v) { return __double2ll_rn(v * 4294967296.0); }

struct R4Frac {
    int i;
    float f;
};
__device__ __forceinline__ R4Frac r4_split(long long u) {
    const long long u24 = (u + 128) >> 8;
    return {(int)(u24 >> 24), (float)(int)(u24 & 0xFFFFFF) * 0x1p-24f};
}

__device__ __forceinline__ void r4_kahan(float& acc, float& cmp, float v) {
    const float y = v - cmp;
    const float t = acc + y;
    cmp = (t - acc) - y;
    acc = t;
}

// Per-plane coordinate tables (fixed point), chunk planes p0 .. p0 + np - 1:
//   x axis: TAx[p][c] = alpha (c - cxa) + cxa,        TBx[p][j] = beta sx (j - cxb)
//           TAbx[p][c] = gamma (c - cxa) / sx + cxb,  TBbx[p][j] = delta (j - cxb)
//           (TAx and TAbx with the 24-bit rounding bias and the box's border added)
//   y axis: the same with rows (ha, hb, sy).
__global__ void r4_tables_kernel(const Plane4Block co, int np, int ha, int wa, int hb, int wb,
                                 long long* __restrict__ t, int64_t stride) {
    dep_wait();
    dep_launch();
    const int p = blockIdx.x;
    if (p >= np) return;
    const double al = co.c[p][0], be = co.c[p][1], ga = co.c[p][2], de = co.c[p][3];
    const double cxa = 0.5 * (wa - 1), cya = 0.5 * (ha - 1), cxb = 0.5 * (wb - 1), cyb = 0.5 * (hb - 1);
    const double sx = (double)wa / (double)wb, sy = (double)ha / (double)hb;
    long long* TAx = t + 0 * stride + (int64_t)p * wa;
    long long* TAbx = t + 1 * stride + (int64_t)p * wa;
    long long* TBx = t + 2 * stride + (int64_t)p * wb;
    long long* TBbx = t + 3 * stride + (int64_t)p * wb;
    long long* TAy = t + 4 * stride + (int64_t)p * ha;
    long long* TAby = t + 5 * stride + (int64_t)p * ha;
    long long* TBy = t + 6 * stride + (int64_t)p * hb;
    long long* TBby = t + 7 * stride + (int64_t)p * hb;
    for (int c = threadIdx.x; c < wa; c += blockDim.x) {
        TAx[c] = r4_fix(al * (c - cxa) + cxa) + kXBias;
        TAbx[c] = r4_fix(ga * (c - cxa) / sx + cxb) + kXBias;
    }
    for (int j = threadIdx.x; j < wb; j += blockDim.x) {
        TBx[j] = r4_fix(be * sx * (j - cxb));
        TBbx[j] = r4_fix(de * (j - cxb));
    }
    for (int r = threadIdx.x; r < ha; r += blockDim.x) {
        TAy[r] = r4_fix(al * (r - cya) + cya);
        TAby[r] = r4_fix(ga * (r - cya) / sy + cyb);
    }
    for (int j = threadIdx.x; j < hb; j += blockDim.x) {
        TBy[j] = r4_fix(be * sy * (j - cyb));
        TBby[j] = r4_fix(de * (j - cyb));
    }
}

// Stage 1: CTA (yb, ya0 .. ya0 + K - 1): the boxes of those K row pairs, interleaved
// in shared memory as [xb][xa][K rows]; every plane of the chunk, G planes at a time;
// thread w of a pass takes plane p0 + w / wa and column x_c = w % wa (so narrow images
// still give every thread work).  The taps of (plane, x_c, j_c) do not depend on the
// row pair: each is formed once and one 4, 8 or 16-byte load fetches it for all K
// rows, whose sums run in packed FP32 lanes.  About 26 instructions form the taps, 4
// load, and 10 K / 2 sum, so K = 4 wherever the box fits, else 2 (128 x 128), else 1.
// The pitch of the box's rows is one entry short of (or past) a whole number of bank
// cycles: with alpha > 1 the lanes of a load spread over more than one cycle of banks,
// and where gamma has the sign of alpha - 1 they also step to the next row as they
// spread, so a row that starts one entry early brings them back (the other sign: one
// entry late).  Counted over 41 planes at 128 x 128, K = 2: 10.9 wavefronts per 4
// loads against 15.7 with rows on the same bank; 8 is the least.  sB holds
// the G planes' angular-column tables.  Bound by the issue of the taps and by the
// shared-memory reads (4 K bytes x 4 taps a thread).
template <int K>
struct BoxOf;
template <>
struct BoxOf<1> {
    typedef float T;
    static __device__ __forceinline__ void set(T& b, const float* v) { b = v[0]; }
};
template <>
struct BoxOf<2> {
    typedef f32x2 T;
    static __device__ __forceinline__ void set(T& b, const float* v) { b = pk2(v[0], v[1]); }
};
template <>
struct BoxOf<4> {
    typedef ulonglong2 T;
    static __device__ __forceinline__ void set(T& b, const float* v) { b = make_ulonglong2(pk2(v[0], v[1]), pk2(v[2], v[3])); }
};

__device__ __forceinline__ void r4_kahan2(f32x2& acc, f32x2& cmp, f32x2 v) {
    const f32x2 y = sub2(v, cmp);
    const f32x2 t = add2(acc, y);
    cmp = sub2(sub2(t, acc), y);
    acc = t;
}
// one bilinear sample of both lanes, Kahan-added
__device__ __forceinline__ void r4_sample2(f32x2& acc, f32x2& cmp, f32x2 fa, f32x2 ga, f32x2 fb, f32x2 gb, f32x2 v00,
                                           f32x2 v01, f32x2 v10, f32x2 v11) {
    const f32x2 top = fma2(fa, v01, mul2(ga, v00));
    const f32x2 bot = fma2(fa, v11, mul2(ga, v10));
    r4_kahan2(acc, cmp, fma2(fb, bot, mul2(gb, top)));
}

constexpr int kColThreads = 1024;      // at most; 512 where two or three CTAs fit an SM
template <int K, int kCtas>
__global__ void __launch_bounds__(kCtas == 3 ? 512 : kColThreads, kCtas == 3 ? 3 : 1) r4_cols_kernel(const float* __restrict__ g, int np, int G, int ha,
                                                                 int wa, int hb, int wb, int WP,
                                                                 const long long* __restrict__ t, int64_t stride,
                                                                 float* __restrict__ c_hi, float* __restrict__ c_lo) {
    typedef typename BoxOf<K>::T Box;
    constexpr int NP = K > 1 ? K / 2 : 1;                  // packed sums per thread
    extern __shared__ __align__(16) float sm[];
    const int yb = blockIdx.x, ya0 = blockIdx.y * K, nt = blockDim.x;
    const int nb = min(K, ha - ya0);                       // rows of this CTA
    const int64_t ma = (int64_t)ha * wa;
    const int HP = wb + 2 * kPad;                          // padded box: HP rows (xb) x WP columns (xa)
    longlong2* sB = reinterpret_cast<longlong2*>(sm);      // [G][wb]: (TBx, TBbx) of the pass's planes
    Box* box = reinterpret_cast<Box*>(sB + (size_t)G * wb);
    for (int i = threadIdx.x; i < HP * WP; i += nt) {
        const int r = i / WP, xb = r - kPad, xa = i - r * WP - kPad;
        float v[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
            v[k] = (k < nb && xb >= 0 && xb < wb && xa >= 0 && xa < wa)
                       ? __ldg(g + (int64_t)(yb * wb + xb) * ma + (int64_t)(ya0 + k) * wa + xa)
                       : 0.0f;
        BoxOf<K>::set(box[i], v);
    }
    dep_launch();
    dep_wait();   // Gamma was complete before the tables' kernel began
    t = after_wait(t);
    for (int p0 = 0; p0 < np; p0 += G) {
        const int gp = min(G, np - p0);
        __syncthreads();   // boxes ready / previous pass's tables consumed
        for (int i = threadIdx.x; i < gp * wb; i += nt) {
            const int k = i / wb, j = i - k * wb;
            sB[i] = make_longlong2(t[2 * stride + (int64_t)(p0 + k) * wb + j], t[3 * stride + (int64_t)(p0 + k) * wb + j]);
        }
        __syncthreads();
        for (int w = threadIdx.x; w < gp * wa; w += nt) {
            const int kp = w / wa, xc = w - kp * wa, p = p0 + kp;
            const longlong2* B = sB + kp * wb;
            const long long ax = t[0 * stride + (int64_t)p * wa + xc];
            const long long abx = t[1 * stride + (int64_t)p * wa + xc];
            f32x2 acc[NP], cmp[NP];
            float acc1 = 0.0f, cmp1 = 0.0f;
#pragma unroll
            for (int k = 0; k < NP; ++k) acc[k] = cmp[k] = 0ull;
#pragma unroll (K == 1 ? 4 : 2)
            for (int jc = 0; jc < wb; ++jc) {
                const longlong2 b = B[jc];
                const long long ua = ax + b.x, ub = abx + b.y;
                const int xa = min(max((int)(ua >> 32), 0), wa + kPad);
                const int xb = min(max((int)(ub >> 32), 0), wb + kPad);
                const float fa = (float)((uint32_t)ua >> 8) * 0x1p-24f, ga = 1.0f - fa;
                const float fb = (float)((uint32_t)ub >> 8) * 0x1p-24f, gb = 1.0f - fb;
                const Box* q = box + xb * WP + xa;
                if constexpr (K == 1) {
                    const float top = __fmaf_rn(fa, q[1], ga * q[0]);
                    const float bot = __fmaf_rn(fa, q[WP + 1], ga * q[WP]);
                    r4_kahan(acc1, cmp1, __fmaf_rn(fb, bot, gb * top));
                } else {
                    const f32x2 fa2 = pk2(fa, fa), ga2 = pk2(ga, ga), fb2 = pk2(fb, fb), gb2 = pk2(gb, gb);
                    if constexpr (K == 2) {
                        r4_sample2(acc[0], cmp[0], fa2, ga2, fb2, gb2, q[0], q[1], q[WP], q[WP + 1]);
                    } else {
                        const ulonglong2 v00 = q[0], v01 = q[1], v10 = q[WP], v11 = q[WP + 1];
                        r4_sample2(acc[0], cmp[0], fa2, ga2, fb2, gb2, v00.x, v01.x, v10.x, v11.x);
                        r4_sample2(acc[1], cmp[1], fa2, ga2, fb2, gb2, v00.y, v01.y, v10.y, v11.y);
                    }
                }
            }
            int64_t o = (((int64_t)p * ha + ya0) * hb + yb) * wa + xc;
            if constexpr (K == 1) {
                c_hi[o] = acc1;
                c_lo[o] = -cmp1;
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k, o += (int64_t)hb * wa) {
                    float s[2], e[2];
                    unpk2(acc[k / 2], s[0], s[1]);
                    unpk2(cmp[k / 2], e[0], e[1]);
                    if (k < nb) {
                        c_hi[o] = s[k & 1];
                        c_lo[o] = -e[k & 1];
                    }
                }
            }
        }
    }
}

// The same for a box too large for shared memory (256 x 256): one row pair per CTA,
// taps read from global memory.
constexpr int kColThreadsG = 512;
__global__ void __launch_bounds__(kColThreadsG) r4_cols_global_kernel(const float* __restrict__ g, int np, int G, int ha,
                                                                      int wa, int hb, int wb,
                                                                      const long long* __restrict__ t, int64_t stride,
                                                                      float* __restrict__ c_hi, float* __restrict__ c_lo) {
    extern __shared__ __align__(16) float sm[];
    const int yb = blockIdx.x, ya = blockIdx.y;
    const int64_t ma = (int64_t)ha * wa;
    longlong2* sB = reinterpret_cast<longlong2*>(sm);
    const float* gbase = g + ((int64_t)yb * wb) * ma + (int64_t)ya * wa;
    dep_wait();
    dep_launch();
    t = after_wait(t);
    for (int p0 = 0; p0 < np; p0 += G) {
        const int gp = min(G, np - p0);
        __syncthreads();
        for (int i = threadIdx.x; i < gp * wb; i += kColThreadsG) {
            const int k = i / wb, j = i - k * wb;
            sB[i] = make_longlong2(t[2 * stride + (int64_t)(p0 + k) * wb + j], t[3 * stride + (int64_t)(p0 + k) * wb + j]);
        }
        __syncthreads();
        for (int w = threadIdx.x; w < gp * wa; w += kColThreadsG) {
            const int kp = w / wa, xc = w - kp * wa, p = p0 + kp;
            const longlong2* B = sB + kp * wb;
            const long long ax = t[0 * stride + (int64_t)p * wa + xc];
            const long long abx = t[1 * stride + (int64_t)p * wa + xc];
            float acc = 0.0f, cmp = 0.0f;
            for (int jc = 0; jc < wb; ++jc) {
                const longlong2 b = B[jc];
                const long long ua = ax + b.x, ub = abx + b.y;
                const float fa = (float)((uint32_t)ua >> 8) * 0x1p-24f, ga = 1.0f - fa;
                const float fb = (float)((uint32_t)ub >> 8) * 0x1p-24f, gb = 1.0f - fb;
                float s[2][2];
#pragma unroll
                for (int db = 0; db < 2; ++db)
#pragma unroll
                    for (int da = 0; da < 2; ++da) {
                        const int xa = (int)(ua >> 32) - kPad + da, xb = (int)(ub >> 32) - kPad + db;
                        s[db][da] = (xa >= 0 && xa < wa && xb >= 0 && xb < wb) ? __ldg(gbase + (int64_t)xb * ma + xa) : 0.0f;
                    }
                const float top = __fmaf_rn(fa, s[0][1], ga * s[0][0]);
                const float bot = __fmaf_rn(fa, s[1][1], ga * s[1][0]);
                r4_kahan(acc, cmp, __fmaf_rn(fb, bot, gb * top));
            }
            const int64_t o = (((int64_t)p * ha + ya) * hb + yb) * wa + xc;
            c_hi[o] = acc;
            c_lo[o] = -cmp;
        }
    }
}

// (sh, sl) += wa * wb * (ch + cl) with error-free FP32 transformations: the
// weight product and the leading product are split exactly with fused
// multiply-adds (TwoProduct), the leading term is added by TwoSum; the
// remaining second-order terms go to sl.  The sum is exact up to O(u^2) per
// term; one rounding (sh + sl) ends it.
__device__ __forceinline__ void r4_df_add(float& sh, float& sl, float wa, float wb, float ch, float cl) {
    const float pw = wa * wb;
    const float ew = __fmaf_rn(wa, wb, -pw);
    const float th = pw * ch;
    float te = __fmaf_rn(pw, ch, -th);
    te = __fmaf_rn(pw, cl, __fmaf_rn(ew, ch, te));
    const float s = sh + th;
    const float bb = s - sh;
    const float err = (sh - (s - bb)) + (th - bb);
    sl = sl + (err + te);
    sh = s;
}

// Stage 2: CTA (block of G output rows, plane); thread w takes row
// blockIdx.x * G + w / wa and column w % wa.  Double-float sums (r4_df_add).
__global__ void __launch_bounds__(kR4Threads) r4_rows_kernel(const float* __restrict__ c_hi,
                                                             const float* __restrict__ c_lo, int G, int ha, int wa,
                                                             int hb, const long long* __restrict__ t, int64_t stride,
                                                             float* __restrict__ out) {
    const int p = blockIdx.y;
    dep_wait();
    dep_launch();
    t = after_wait(t);
    c_hi = after_wait(c_hi);
    c_lo = after_wait(c_lo);
    for (int w = threadIdx.x; w < G * wa; w += kR4Threads) {
        const int k = w / wa, xc = w - k * wa, xr = blockIdx.x * G + k;
        if (xr >= ha) continue;
        const long long ay = t[4 * stride + (int64_t)p * ha + xr];
        const long long aby = t[5 * stride + (int64_t)p * ha + xr];
        float sh = 0.0f, sl = 0.0f;
        for (int jr = 0; jr < hb; ++jr) {
            const R4Frac fa = r4_split(ay + t[6 * stride + (int64_t)p * hb + jr]);
            const R4Frac fb = r4_split(aby + t[7 * stride + (int64_t)p * hb + jr]);
#pragma unroll
            for (int db = 0; db < 2; ++db) {
                const int yb = fb.i + db;
                if (yb < 0 || yb >= hb) continue;
                const float wbw = db ? fb.f : 1.0f - fb.f;
#pragma unroll
                for (int da = 0; da < 2; ++da) {
                    const int ya = fa.i + da;
                    if (ya < 0 || ya >= ha) continue;
                    const float waw = da ? fa.f : 1.0f - fa.f;
                    const int64_t o = (((int64_t)p * ha + ya) * hb + yb) * wa + xc;
                    r4_df_add(sh, sl, waw, wbw, c_hi[o], c_lo[o]);
                }
            }
        }
        out[((int64_t)p * ha + xr) * wa + xc] = sh + sl;
    }
}

}  // namespace

Refocus4dLayout refocus4d_layout(int ha, int wa, int hb, int wb, int n_planes) {
    Refocus4dLayout L{};
    const int64_t per_plane = (int64_t)ha * hb * wa;          // C entries per plane
    int chunk = n_planes < kRefocus4dChunk ? n_planes : kRefocus4dChunk;
    while (chunk > 1 && (int64_t)chunk * per_plane * 8 > ((int64_t)4 << 30)) chunk /= 2;
    L.chunk = chunk;
    int m = ha;
    if (wa > m) m = wa;
    if (hb > m) m = hb;
    if (wb > m) m = wb;
    L.stride = (int64_t)chunk * m;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = (o + bytes + 255) / 256 * 256;
        return at;
    };
    L.tables = take(sizeof(long long) * 8 * (size_t)L.stride);
    L.c_hi = take(sizeof(float) * (size_t)(chunk * per_plane));
    L.c_lo = take(sizeof(float) * (size_t)(chunk * per_plane));
    L.bytes = o;
    return L;
}

namespace {
constexpr size_t kR4SmemCap = 224 * 1024;
constexpr size_t kR4TableCap = 16 * 1024;

// planes per pass of the column stage, evenly over the passes
int r4_col_group(int threads, int wa, int wb, int np) {
    int G = threads / wa;
    while (G > 1 && (size_t)G * wb * sizeof(longlong2) > kR4TableCap) --G;
    if (G < 1) G = 1;
    if (G > np) G = np;
    const int passes = (np + G - 1) / G;
    return (np + passes - 1) / passes;
}

struct ColPlan {
    int K, WP, threads, G;
    size_t smem;
};
// Rows per CTA (4, 2, 1): as many as fit, while the grid keeps ~4 CTAs per SM of a
// 152-SM GPU.  K = 0: not even one row's box fits.
// skew: the sign of alpha - 1 against gamma over the planes (see r4_cols_kernel).
ColPlan r4_col_plan(int ha, int wa, int hb, int wb, int np, double skew) {
    for (int K : {4, 2, 1}) {
        if (K > 1 && (int64_t)hb * ((ha + K - 1) / K) < 4 * 152) continue;
        const int bank = 32 / K, tight = wa + 2 * kPad;
        const int want = skew >= 0.0 ? bank - 1 : 1;
        for (int WP : {tight + (want - tight % bank + bank) % bank, tight}) {
            const size_t box = (size_t)(wb + 2 * kPad) * WP * K * sizeof(float);
            for (int threads : {512, 1024}) {
                const int G = r4_col_group(threads, wa, wb, np);
                const size_t smem = (size_t)G * wb * sizeof(longlong2) + box;
                if (smem <= (threads == 512 ? kR4SmemCap / 2 : kR4SmemCap)) return {K, WP, threads, G, smem};
            }
        }
    }
    return {};
}

template <int K, int kCtas>
cudaError_t launch_cols_t(const ColPlan& c, const float* g, int np, int ha, int wa, int hb, int wb, const long long* t,
                        int64_t stride, float* c_hi, float* c_lo, cudaStream_t st) {
    static bool attr[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr[dev]) {
        if ((e = cudaFuncSetAttribute(r4_cols_kernel<K, kCtas>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kR4SmemCap)) !=
            cudaSuccess)
            return e;
        attr[dev] = true;
    }
    const dim3 grid((unsigned)hb, (unsigned)((ha + K - 1) / K));
    return launch_kernel(true, r4_cols_kernel<K, kCtas>, grid, c.threads, c.smem, st, g, np, c.G, ha, wa, hb, wb, c.WP, t, stride,
                         c_hi, c_lo);
}

// The kernel compiled for two CTAs of 512 threads on an SM (56 to 64 registers) or for
// three (40).  Three pay where the grid is more than four and a half CTAs per SM and most
// of a CTA's threads have work: 46x26 vs 97x12 with 90 planes 462 -> 356 us, 32x30 vs
// 92x18, 68: 366 -> 304, 44x27 vs 41x41, 82: 353 -> 295 (with a 4-byte box per row and
// about 40 registers they took 359, 315 and 286).  On smaller grids the narrower register
// set costs: 17x63 vs 24x31, 42 (408 CTAs): 93 -> 110.
template <int K>
cudaError_t launch_cols(const ColPlan& c, const float* g, int np, int ha, int wa, int hb, int wb, const long long* t,
                        int64_t stride, float* c_hi, float* c_lo, cudaStream_t st) {
    const int64_t ctas = (int64_t)hb * ((ha + K - 1) / K);
    if (c.threads == 512 && c.smem <= kR4SmemCap / 3 && ctas > 700 && c.G * wa >= 360)
        return launch_cols_t<K, 3>(c, g, np, ha, wa, hb, wb, t, stride, c_hi, c_lo, st);
    return launch_cols_t<K, 1>(c, g, np, ha, wa, hb, wb, t, stride, c_hi, c_lo, st);
}
}  // namespace

cudaError_t launch_refocus4d_chunk(const float* gamma_f32, int ha, int wa, int hb, int wb, const Plane4Block& coef,
                                   int np, uint8_t* ws, const Refocus4dLayout& L, float* out, cudaStream_t st) {
    long long* t = reinterpret_cast<long long*>(ws + L.tables);
    float* c_hi = reinterpret_cast<float*>(ws + L.c_hi);
    float* c_lo = reinterpret_cast<float*>(ws + L.c_lo);
    cudaError_t e = launch_kernel(false, r4_tables_kernel, np, 128, 0, st, coef, np, ha, wa, hb, wb, t, L.stride);
    if (e != cudaSuccess) return e;
    double skew = 0.0;
    for (int p = 0; p < np; ++p) skew += (coef.c[p][0] - 1.0) * coef.c[p][2];
    const ColPlan c = r4_col_plan(ha, wa, hb, wb, np, skew);
    if (c.K == 4) e = launch_cols<4>(c, gamma_f32, np, ha, wa, hb, wb, t, L.stride, c_hi, c_lo, st);
    else if (c.K == 2) e = launch_cols<2>(c, gamma_f32, np, ha, wa, hb, wb, t, L.stride, c_hi, c_lo, st);
    else if (c.K == 1) e = launch_cols<1>(c, gamma_f32, np, ha, wa, hb, wb, t, L.stride, c_hi, c_lo, st);
    else {
        const int G = r4_col_group(kColThreadsG, wa, wb, np);
        static bool attr[64] = {};
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        if (!attr[dev]) {   // angular rows of more than 3072 pixels: a table above 48 KiB
            if ((e = cudaFuncSetAttribute(r4_cols_global_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)) !=
                cudaSuccess)
                return e;
            attr[dev] = true;
        }
        e = launch_kernel(true, r4_cols_global_kernel, dim3((unsigned)hb, (unsigned)ha), kColThreadsG,
                          sizeof(longlong2) * (size_t)G * wb, st, gamma_f32, np, G, ha, wa, hb, wb, t, L.stride, c_hi, c_lo);
    }
    if (e != cudaSuccess) return e;
    const int Gr = wa < kR4Threads ? kR4Threads / wa : 1;
    return launch_kernel(true, r4_rows_kernel, dim3((unsigned)((ha + Gr - 1) / Gr), (unsigned)np), kR4Threads, 0, st,
        c_hi, c_lo, Gr, ha, wa, hb, t, L.stride, out);
}

}  // namespace cpi
