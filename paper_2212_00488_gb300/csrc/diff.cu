// Differentiable form of the left-base cost and aggregation (FP32): a soft
// argmin over the aggregated cost, and its backward as the adjoint of the
// cross aggregation over the same frozen supports.
//
//   g          = (77 R + 150 G + 29 B) / 256 on [0, 1]       (float grey)
//   census codes and arms: frozen (not differentiated), computed by the
//              integer path from the pair's uint8 images
//   C(x,y,d)   = w_AD (1 - exp(-|gL(x,y) - gR(x-d,y)| / l_AD))
//              + w_MC (1 - exp(-MC / l_MC))                    (Eqs. 3-5)
//              = P(theta) when x < d
//   CA(x,y,d)  = Eqs. 7-8 over the frozen arms, divided by the support size
//   dhat       = sum_d d softmax_d(-CA / tau)
//
// The volume is never stored: forward and backward walk the disparities in
// chunks of kDC, keeping per chunk the x-aggregated slab and, in backward,
// the slab's gradients, as two planes [y][x] of four disparities each. Every
// pair of the batch has its own buffers, and the per-chunk kernels take all
// pairs in one launch.
//
// Sums over arms are direct (at most 2 wx + 1 and 2 wy + 1 terms, in ascending
// order), which keeps FP32 aggregates within about 6e-6 of their exact value. The
// order is part of the result: sums over blocks of four cells are no less exact
// and a third faster, but move every aggregate's last place, and the parameter
// gradients, where almost all of a pixel's terms cancel, then miss their 64-bit
// values by up to four times as much on some inputs (and by less on others).
// Along x a thread sums the windows of four neighbouring pixels side by side:
// it reads each cell of their joint span once and adds it to the windows that
// hold it, two disparities per instruction. The adjoint of each sum is a banded
// difference array walked in a fixed order by one thread, so no float atomics
// are used and results are deterministic.
//
// 4 pairs of 718 x 496, D 73, forward and backward (arms at their caps in a third
// of the planes): 9.1 ms with one window per thread over planes [kDC][y][x] and
// separate kernels for the horizontal adjoint and the cost gradient, 4.7 ms
// now. Bound by issue slots in the cost and the adjoints, by L1 in the vertical sums.
#include "internal.cuh"

namespace stereo {

constexpr int kDiffNT = 256;   // threads of the per-pixel kernels

namespace {

constexpr int kDC = 8;   // disparities per chunk
// pixel tiles of the kernels that sum along y
constexpr int kTileX = 32, kTileY = 8;
__constant__ float kGreyW[3] = {77.f / 256.f, 150.f / 256.f, 29.f / 256.f};

__global__ void diff_grey_kernel(const float *__restrict__ rgb_l, const float *__restrict__ rgb_r,
                                 float *__restrict__ g_l, float *__restrict__ g_r, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const size_t b = blockIdx.z;                  // pair
    rgb_l += b * n * 3;
    rgb_r += b * n * 3;
    g_l += b * n;
    g_r += b * n;
    const float *rgb = blockIdx.y ? rgb_r : rgb_l;
    float g = __fmul_rn(kGreyW[0], rgb[3 * i]);
    g = __fadd_rn(g, __fmul_rn(kGreyW[1], rgb[3 * i + 1]));
    g = __fadd_rn(g, __fmul_rn(kGreyW[2], rgb[3 * i + 2]));
    (blockIdx.y ? g_r : g_l)[i] = g;
}

// Support size n(x,y) = sum over the vertical span of each row's x window, as the
// difference of two prefixes: a block takes 32 columns and kNSRows rows and
// keeps the prefixes of those rows and the kMaxWy above and below in shared
// memory. (A loop over the span: 35 us at 4 x 718 x 496; this way 8.)
constexpr int kNSRows = 66, kNSAll = kNSRows + 2 * kMaxWy;   // 128 rows: 8 groups of 16
static_assert(kNSAll == 128, "eight threads of sixteen rows per column");
__global__ void __launch_bounds__(kDiffNT) diff_nsupport_kernel(const uint32_t *__restrict__ arm, int X, int Y,
                                                                float *__restrict__ ns)
{
    __shared__ int pre[kNSAll + 1][32];               // pre[i]: widths of rows y0 - kMaxWy .. + i - 1
    __shared__ int tot[8][32];
    const int c = threadIdx.x % 32, q = threadIdx.x / 32;
    const int x = blockIdx.x * 32 + c, y0 = blockIdx.y * kNSRows;
    const size_t b = blockIdx.z;                      // pair
    arm += b * X * Y;
    ns += b * X * Y;
    int w[16], s = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int y = y0 - kMaxWy + 16 * q + i;
        w[i] = 0;
        if (x < X && y >= 0 && y < Y) {
            const uint32_t a = __ldg(arm + (size_t)y * X + x);
            w[i] = (int)(a & 0xFF) + (int)((a >> 8) & 0xFF) + 1;
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) s += w[i];
    tot[q][c] = s;
    __syncthreads();
    s = 0;
    for (int i = 0; i < q; ++i) s += tot[i][c];
    if (q == 0) pre[0][c] = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) pre[16 * q + i + 1][c] = s += w[i];
    __syncthreads();
    for (int r = q; r < kNSRows && y0 + r < Y && x < X; r += 8) {
        const size_t i = (size_t)(y0 + r) * X + x;
        const uint32_t a = __ldg(arm + i);
        const int p = r + kMaxWy;
        ns[i] = (float)(pre[p + (int)(a >> 24) + 1][c] - pre[p - (int)((a >> 16) & 0xFF)][c]);
    }
}

struct Theta {
    float wad, wmc, lad, lmc;
};

__device__ __forceinline__ Theta load_theta(const float *t) { return Theta{t[0], t[1], t[2], t[3]}; }

// Sums of the chunk's disparities, two to a register pair.
struct Sum8 {
    unsigned long long v[kDC / 2];
};
__device__ __forceinline__ void add8(Sum8 &s, const ulonglong2 a, const ulonglong2 b)
{
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s.v[0]) : "l"(a.x));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s.v[1]) : "l"(a.y));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s.v[2]) : "l"(b.x));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s.v[3]) : "l"(b.y));
}
// Bits lo .. hi of a word, as far as it has them: which of the next 32 cells lie in
// a window. A bit test per cell and window is half the work of two compares.
__device__ __forceinline__ uint32_t span_mask(int lo, int hi)
{
    if (hi < 0 || lo > 31) return 0u;
    return (~0u << max(lo, 0)) & (~0u >> (31 - min(hi, 31)));
}
__device__ __forceinline__ void unpack8(const Sum8 &s, float (&o)[kDC])
{
#pragma unroll
    for (int j = 0; j < kDC / 2; ++j) {
        o[2 * j] = __uint_as_float((uint32_t)s.v[j]);
        o[2 * j + 1] = __uint_as_float((uint32_t)(s.v[j] >> 32));
    }
}

// Cost and x window sums. A block takes SEG columns of a row quad: the costs of
// the chunk's disparities for those columns and a wx halo go to shared memory
// (two planes of four disparities per row), then a thread owns CPT = SEG / 64
// neighbouring pixels of one row and sums their windows. 256 columns cost the
// least halo; 64 columns give a small image four times the blocks
// (63 us a chunk at 4 x 718 x 496, 68 with 64 columns; 10 us at 2 x 205 x 123, 14
// with 256).
template <int CPT>
__host__ __device__ __forceinline__ int cxpad(int i)
{
    // CPT = 4: a cell skipped every four keeps the lanes' 16-byte loads in distinct banks
    return CPT == 4 ? i + (i >> 2) : i;
}
template <int SEG>
__host__ __device__ __forceinline__ int costx_pitch(int X, int wx)
{
    return cxpad<SEG / 64>(X < SEG + 2 * wx ? X : SEG + 2 * wx) + 1;
}
template <int SEG>
size_t costx_smem(int X, int wx)
{
    return (size_t)8 * costx_pitch<SEG>(X, wx) * sizeof(float4);
}

template <int SEG>
__global__ void __launch_bounds__(kDiffNT) diff_costx_kernel(
    const float *__restrict__ gL, const float *__restrict__ gR, const uint32_t *__restrict__ pixL,
    const uint32_t *__restrict__ pixR, const uint32_t *__restrict__ arm, const float *__restrict__ theta, int X, int Y,
    int D, int d0, int wx, float4 *__restrict__ hs)
{
    extern __shared__ float4 cell[];                  // [4 rows][2][P]
    __shared__ float mc[8];
    constexpr int CPT = SEG / 64;
    static_assert(4 * SEG == CPT * kDiffNT, "the windows of four rows, CPT per thread");
    pdl_trigger();
    const int x0 = blockIdx.x * SEG, y0 = blockIdx.y * 4;
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    const int P = costx_pitch<SEG>(X, wx);
    pdl_wait();
    gL += b * n;
    gR += b * n;
    pixL += b * n;
    pixR += b * n;
    arm += b * n;
    hs += b * 2 * n;
    const Theta th = load_theta(theta);
    const float Pc = th.wad * (1.f - expf(-1.f / th.lad)) + th.wmc * (1.f - expf(-6.f / th.lmc));
    const int kn = min(kDC, D - d0);
    // the census term takes seven values: one exp per Hamming distance
    if (threadIdx.x < 7) mc[threadIdx.x] = th.wmc * (1.f - expf(-(float)threadIdx.x / th.lmc));
    const float inv_lad = 1.f / th.lad;
    const int xs = max(x0 - wx, 0), xe = min(x0 + SEG + wx, X);   // staged columns
    const int nc = xe - xs, nr = min(4, Y - y0);
    __syncthreads();
    for (int i = threadIdx.x; i < nc * nr; i += kDiffNT) {
        const int r = i / nc, x = xs + i - r * nc;
        const size_t row = (size_t)(y0 + r) * X;
        const float gl = gL[row + x];
        const uint32_t pl = pixL[row + x];
        float c[kDC];
        // the chunk's disparities unrolled, so their loads and exps overlap
#pragma unroll
        for (int k = 0; k < kDC; ++k) {
            const int d = d0 + k;
            c[k] = k < kn ? Pc : 0.f;
            if (k < kn && x >= d) {
                const float a = fabsf(gl - gR[row + x - d]);
                const int h = __popc((pl ^ pixR[row + x - d]) & 0x3F00u);
                c[k] = th.wad * (1.f - expf(-a * inv_lad)) + mc[h];
            }
        }
        float4 *o = cell + 2 * r * P + cxpad<CPT>(x - xs);
        o[0] = make_float4(c[0], c[1], c[2], c[3]);
        o[P] = make_float4(c[4], c[5], c[6], c[7]);
    }
    __syncthreads();
    const int r = threadIdx.x / 64, xb = x0 + threadIdx.x % 64 * CPT;
    Sum8 s[CPT] = {};
    if (r < nr && xb < X) {
        int lo[CPT], len[CPT], t0 = X, t1 = 0;
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int x = min(xb + j, X - 1);
            const uint32_t am = arm[(size_t)(y0 + r) * X + x];
            lo[j] = x - (int)(am & 0xFF) - xs;
            len[j] = (int)(am & 0xFF) + (int)((am >> 8) & 0xFF);
            t0 = min(t0, lo[j]);
            t1 = max(t1, lo[j] + len[j]);
        }
        const ulonglong2 *c = reinterpret_cast<const ulonglong2 *>(cell + 2 * r * P);
        for (int tb = t0; tb <= t1; tb += 32) {
            uint32_t m[CPT];
#pragma unroll
            for (int j = 0; j < CPT; ++j) m[j] = span_mask(lo[j] - tb, lo[j] + len[j] - tb);
            for (int t = tb; t <= min(tb + 31, t1); t += 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int ti = cxpad<CPT>(min(t + i, t1));
                    const ulonglong2 u = c[ti], v = c[P + ti];
#pragma unroll
                    for (int j = 0; j < CPT; ++j)
                        if (m[j] & (1u << i)) add8(s[j], u, v);
                }
#pragma unroll
                for (int j = 0; j < CPT; ++j) m[j] >>= 4;
            }
        }
    }
    if constexpr (CPT == 1) {
        if (r < nr && xb < X) {
            ulonglong2 *o = reinterpret_cast<ulonglong2 *>(hs) + (size_t)(y0 + r) * X + xb;
            o[0] = make_ulonglong2(s[0].v[0], s[0].v[1]);
            o[n] = make_ulonglong2(s[0].v[2], s[0].v[3]);
        }
    } else {
        // through shared memory, so that the stores are coalesced
        __syncthreads();
        if (r < nr && xb < X) {
            ulonglong2 *c = reinterpret_cast<ulonglong2 *>(cell + 2 * r * P);
#pragma unroll
            for (int j = 0; j < CPT; ++j)
                if (xb + j < X) {
                    c[cxpad<CPT>(xb + j - x0)] = make_ulonglong2(s[j].v[0], s[j].v[1]);
                    c[P + cxpad<CPT>(xb + j - x0)] = make_ulonglong2(s[j].v[2], s[j].v[3]);
                }
        }
        __syncthreads();
        const int x = x0 + threadIdx.x;
        static_assert(SEG == kDiffNT, "one column per thread");
        if (x < X)
            for (int j = 0; j < 2 * nr; ++j)
                hs[(j & 1) * n + (size_t)(y0 + (j >> 1)) * X + x] = cell[j * P + cxpad<CPT>(x - x0)];
    }
}

// Vertical sums of Eq. 8 for the chunk's disparities: the rows of the warp's joint
// span, each read once and coalesced, eight at a time, added where the pixel's
// own span holds them (a loop over each pixel's span: 197-276 us a chunk with the
// softmax at 4 x 718 x 496, 75-78 now; four rows per thread 84-91). Called by whole
// warps of 32 columns; sums in ascending y.
__device__ __forceinline__ void vsum(const float4 *__restrict__ hs, size_t n, int x, int lo, int hi, int X, Sum8 &s)
{
    constexpr int R = 8;
    const int t0 = __reduce_min_sync(0xffffffffu, lo), t1 = __reduce_max_sync(0xffffffffu, hi);
    const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(hs) + x;
    s = Sum8{};
    for (int tb = t0; tb <= t1; tb += 32) {
        uint32_t m = span_mask(lo - tb, hi - tb);
        for (int t = tb; t <= min(tb + 31, t1); t += R) {
            ulonglong2 u[R], v[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const ulonglong2 *r = p + (size_t)min(t + i, t1) * X;
                u[i] = __ldg(r);
                v[i] = __ldg(r + n);
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (m & (1u << i)) add8(s, u[i], v[i]);
            m >>= R;
        }
    }
}

// The vertical sums of a pixel, windows of one row (wy 0: kTall false) without
// vsum(), which reads eight rows at a time: at 2 x 65 x 232, D 83, W_y 0 the forward
// took 160 us with it, 141 without. (A branch for such spans inside vsum() made the
// compiler give up the eight loads in flight, 20 % on every other window.)
template <bool kTall>
__device__ __forceinline__ void vwindow(const float4 *__restrict__ hs, size_t n, int x, int y, uint32_t am, int X, Sum8 &s)
{
    if constexpr (kTall) {
        vsum(hs, n, x, y - (int)((am >> 16) & 0xFF), y + (int)(am >> 24), X, s);
    } else {
        const ulonglong2 *r = reinterpret_cast<const ulonglong2 *>(hs) + (size_t)y * X + x;
        s = Sum8{};
        add8(s, __ldg(r), __ldg(r + n));
    }
}

// Forward: aggregated cost along y per pixel and an online softmax over d.
// state = (max z, sum exp(z - max), sum d exp(z - max)) per pixel.
template <bool kTall>
__global__ void __launch_bounds__(kDiffNT) diff_vagg_softmax_kernel(
    const float4 *__restrict__ hs, const uint32_t *__restrict__ arm, const float *__restrict__ ns, int X, int Y, int D,
    int d0, float inv_tau, float *__restrict__ state, int first, int last, float *__restrict__ dhat,
    float *__restrict__ stats)
{
    pdl_trigger();
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    hs += b * 2 * n;
    ns += b * n;
    state += b * 3 * n;
    dhat += b * n;
    stats += b * 2 * n;
    // 2-D tiles of kTileX x kTileY pixels: the warps of a block walk the
    // same rows, so their vertical windows meet in L1
    const int x = blockIdx.x * kTileX + (int)(threadIdx.x % kTileX), xc = min(x, X - 1);
    const int y = blockIdx.y * kTileY + (int)(threadIdx.x / kTileX);
    pdl_wait();
    if (y >= Y) return;                               // whole warps
    const uint32_t am = arm[b * n + (size_t)y * X + xc];
    Sum8 sum;
    vwindow<kTall>(hs, n, xc, y, am, X, sum);
    if (x >= X) return;
    const size_t i = (size_t)y * X + x;
    const float inv_n = 1.f / ns[i];
    float m = first ? -INFINITY : state[3 * i], s = first ? 0.f : state[3 * i + 1],
          sd = first ? 0.f : state[3 * i + 2];
    float ca[kDC];
    unpack8(sum, ca);
#pragma unroll
    for (int k = 0; k < kDC; ++k) {
        if (d0 + k >= D) break;
        const float z = -(ca[k] * inv_n) * inv_tau;
        const float d = (float)(d0 + k);
        if (z > m) {
            const float f = expf(m - z);
            s = s * f + 1.f;
            sd = sd * f + d;
            m = z;
        } else {
            const float e = expf(z - m);
            s += e;
            sd += d * e;
        }
    }
    if (last) {
        dhat[i] = sd / s;
        stats[2 * i] = m;
        stats[2 * i + 1] = s;
    } else {
        state[3 * i] = m;
        state[3 * i + 1] = s;
        state[3 * i + 2] = sd;
    }
}

// Backward 1: d dhat / d CA = p_d (d - dhat) (-1/tau) / n, times the
// incoming gradient, for the chunk (the aggregated slab is recomputed).
template <bool kTall>
__global__ void __launch_bounds__(kDiffNT) diff_gca_kernel(
    const float4 *__restrict__ hs, const uint32_t *__restrict__ arm, const float *__restrict__ ns, int X, int Y, int D,
    int d0, float inv_tau, const float *__restrict__ dhat, const float *__restrict__ stats,
    const float *__restrict__ go, float4 *__restrict__ g0)
{
    pdl_trigger();
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    hs += b * 2 * n;
    ns += b * n;
    dhat += b * n;
    stats += b * 2 * n;
    go += b * n;
    g0 += b * 2 * n;
    // 2-D tiles of kTileX x kTileY pixels: the warps of a block walk the
    // same rows, so their vertical windows meet in L1
    const int x = blockIdx.x * kTileX + (int)(threadIdx.x % kTileX), xc = min(x, X - 1);
    const int y = blockIdx.y * kTileY + (int)(threadIdx.x / kTileX);
    pdl_wait();
    if (y >= Y) return;                               // whole warps
    const uint32_t am = arm[b * n + (size_t)y * X + xc];
    Sum8 sum;
    vwindow<kTall>(hs, n, xc, y, am, X, sum);
    if (x >= X) return;
    const size_t i = (size_t)y * X + x;
    const float inv_n = 1.f / ns[i];
    const float m = stats[2 * i], s = stats[2 * i + 1], e = dhat[i], gi = go[i];
    float v[kDC];
    unpack8(sum, v);
#pragma unroll
    for (int k = 0; k < kDC; ++k) {
        float r = 0.f;
        if (d0 + k < D) {
            const float z = -(v[k] * inv_n) * inv_tau;
            const float p = expf(z - m) / s;
            r = gi * p * ((float)(d0 + k) - e) * (-inv_tau) * inv_n;
        }
        v[k] = r;
    }
    g0[i] = make_float4(v[0], v[1], v[2], v[3]);
    g0[n + i] = make_float4(v[4], v[5], v[6], v[7]);
}

// Backward 2: adjoint of the vertical sum. G1(x, y') collects the anchors
// (x, y) whose span [y - up, y + down] contains y'. As a difference array: a
// thread owns one column and one disparity of the chunk over a band of kVB
// rows; every anchor whose span reaches the band adds its value at the band
// row where the span enters and subtracts it one row past where the span
// ends (anchors in ascending y), and a running sum down the band gives G1.
// Each thread works alone in a fixed order: deterministic, no atomics, and
// about 2 (kVB + 2 wy) / kVB operations per output instead of 2 wy + 1. Eight rows
// are requested at a time: one by one between the shared stores, a row cost a
// thread 390 ns of latency (76 us a chunk at 4 x 718 x 496, 37 us at 2 x 205 x 123; now
// 47 and 11). Longer bands with a ring would read fewer rows twice (128
// rows: 46 us), but an addition's rounding error then stays in the running sum
// for the whole band, and the parameter gradients, sums of everything, lost a
// digit.
constexpr int kVB = 32, kVTNT = 128;              // 16 columns x kDC disparities
__global__ void __launch_bounds__(kVTNT) diff_vT_kernel(const float *__restrict__ g0, const uint32_t *__restrict__ arm,
                                                        int X, int Y, int wy, float *__restrict__ g1)
{
    __shared__ float delta[kVB + 1][kVTNT];
    pdl_trigger();
    const int t = threadIdx.x, k = t % kDC;
    const int x = blockIdx.x * (kVTNT / kDC) + t / kDC, y0 = blockIdx.y * kVB;
#pragma unroll
    for (int i = 0; i <= kVB; ++i) delta[i][t] = 0.f;
    pdl_wait();
    if (x >= X) return;
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    arm += b * n + x;
    const size_t at = (b * 2 + k / 4) * n * 4 + 4 * x + k % 4;   // plane k / 4, its word k % 4
    const float *gp = g0 + at;
    float *out = g1 + at;
    const int ye = min(y0 + kVB, Y);              // band rows [y0, ye)
    const int ya = max(y0 - wy, 0), yb = min(ye - 1 + wy, Y - 1);
    constexpr int R = 8;
    uint32_t am[R];
    float v[R];
    auto load = [&](int y) {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const size_t i = (size_t)min(y + j, yb) * X;
            am[j] = __ldg(arm + i);
            v[j] = __ldg(gp + i * 4);
        }
    };
    load(ya);
    for (int y = ya; y <= yb; y += R) {
        uint32_t ca[R];
        float cv[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            ca[j] = am[j];
            cv[j] = v[j];
        }
        load(y + R);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int lo = y + j - (int)((ca[j] >> 16) & 0xFF), hi = y + j + (int)(ca[j] >> 24);
            if (y + j <= yb && hi >= y0 && lo < ye) {
                delta[max(lo, y0) - y0][t] += cv[j];
                if (hi + 1 < ye) delta[hi + 1 - y0][t] -= cv[j];
            }
        }
    }
    float s = 0.f;
#pragma unroll 8
    for (int i = 0; i < ye - y0; ++i) {
        s += delta[i][t];
        out[(size_t)(y0 + i) * X * 4] = s;
    }
}

// Backward 3 and 4 in one: the adjoint of the horizontal sum, then through the
// cost. A block takes kHRows rows of a segment of up to kHSeg - kDC + 1 columns of
// one pair.
//  * G2(x', y) collects the pixels (x, y) whose own window [x - left, x + right]
//    contains x'. A thread owns two disparities (one arm word serves both) and a
//    band of kHB columns of the segment and its next kDC - 1 columns: each pixel
//    whose window reaches the band adds its value where the window enters and
//    subtracts it one column past where it ends (pixels in ascending x, eight
//    requested at a time), and a running sum gives the band. G2 stays where the
//    difference arrays were, in shared memory: nothing else is kept there, so
//    that six blocks fit an SM.
//  * A cell (x, y, d) passes v = G2 dC/dgL to its left pixel and -v to the right
//    pixel x - d: v takes the place of G2, and the block takes the right pixels
//    whose cells of this chunk all lie in its columns. The four parameters get
//    one partial per block, summed later in a fixed order.
// (Two kernels, G2 through memory: 76 + 63 us a chunk at 4 x 718 x 496; 116 now.)
constexpr int kHSeg = 512, kHB = 32, kHNT = 128, kHRows = 2;
static_assert(kHRows * kHSeg / kHB * kDC / 2 == kHNT, "one (row, band, disparity pair) per thread");
// [kHB + 1][kHPitch] pairs: entry i of thread t at i kHPitch + t. The odd pitch
// also keeps the columns of a band in distinct banks.
constexpr int kHPitch = kHNT + 1;
constexpr int kHSmem = (kHB + 1) * kHPitch * (int)sizeof(float2);
__host__ __device__ __forceinline__ int hgrad_segments(int X) { return (X + kHSeg - kDC) / (kHSeg - kDC + 1); }
// Rows of a block, a multiple of kHRows, and blocks of a pair and chunk. Each has one
// partial of 16 bytes: images of a few columns with many chunks take more rows a
// block, so that the partials stay below about 50 bytes a pixel.
int hgrad_rows(int X, int nchunks) { return kHRows * std::max(1, nchunks * hgrad_segments(X) / (4 * X)); }
int hgrad_blocks(int X, int Y, int nchunks)
{
    const int rows = hgrad_rows(X, nchunks);
    return hgrad_segments(X) * ((Y + rows - 1) / rows);
}

// s += v with the rounding error carried along in c (Kahan). A sum that overflows
// stays infinite: its error, inf - inf at the next term, would make it NaN.
__device__ __forceinline__ void kahan(float &s, float &c, float v)
{
    const float y = __fsub_rn(v, c), t = __fadd_rn(s, y), e = __fsub_rn(__fsub_rn(t, s), y);
    c = fabsf(e) < INFINITY ? e : 0.f;
    s = t;
}
__global__ void __launch_bounds__(kHNT) diff_hgrad_kernel(
    const float *__restrict__ g1, const uint32_t *__restrict__ arm, const float *__restrict__ gL,
    const float *__restrict__ gR, const uint32_t *__restrict__ pixL, const uint32_t *__restrict__ pixR,
    const float *__restrict__ theta, int X, int Y, int D, int d0, int wx, int rows, int first,
    float *__restrict__ acc_l, float *__restrict__ acc_r, float *__restrict__ part, size_t part_pair)
{
    __shared__ float2 dl[(kHB + 1) * kHPitch];
    __shared__ float eh_t[8];
    __shared__ float sh[4][kHNT / 32];
    static_assert(kHSmem + 256 <= 48 * 1024, "static shared memory");
    pdl_trigger();
    const int nseg = hgrad_segments(X), seg = (X + nseg - 1) / nseg;
    const int s0 = blockIdx.x * seg, s1 = min(s0 + seg, X);   // the segment's left pixels
    const int s2 = min(s1 + kDC - 1, X);                      // the columns whose cells it needs
    const size_t b = blockIdx.z, n = (size_t)X * Y;           // pair
    pdl_wait();
    g1 += b * kDC * n;
    arm += b * n;
    gL += b * n;
    gR += b * n;
    pixL += b * n;
    pixR += b * n;
    acc_l += b * n;
    acc_r += b * n;
    const Theta th = load_theta(theta);
    const float inv_lad = 1.f / th.lad, inv_lmc = 1.f / th.lmc;
    const float kad = th.wad * inv_lad;                 // w_AD / l_AD
    const float dad = th.wad * inv_lad * inv_lad;       // w_AD / l_AD^2
    const float dmc = th.wmc * inv_lmc * inv_lmc;       // w_MC / l_MC^2
    // exp(-h / l_MC) for the seven Hamming distances
    if (threadIdx.x < 7) eh_t[threadIdx.x] = expf(-(float)threadIdx.x * inv_lmc);
    const float ea1 = expf(-inv_lad);
    const int kn = min(kDC, D - d0);
    float t0 = 0.f, t1 = 0.f, t2 = 0.f, t3 = 0.f, e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;
    // (once for kHRows; without the loop the kernel gets other code, 80 registers for
    // 92, and a step at 4 x 718 x 496 takes 4.77 ms, not 4.61)
    const int y_end = min(((int)blockIdx.y + 1) * rows, Y);
    for (int y = blockIdx.y * rows; y < y_end; y += kHRows) {
        const int nr = min(kHRows, y_end - y);
        __syncthreads();                                      // the previous rows are done with shared memory
        constexpr int per_row = kHNT / kHRows;
        {
            const int j = threadIdx.x / per_row, k = threadIdx.x % (kDC / 2);
            const int bx0 = s0 + kHB * (int)(threadIdx.x % per_row / (kDC / 2));
            const int be = min(bx0 + kHB, s2);                // band columns [bx0, be)
            float2 *d = dl + threadIdx.x;
            if (j < nr && bx0 < be) {
                const size_t r = (size_t)(y + j) * X;
                const float2 *gp = reinterpret_cast<const float2 *>(g1) + 2 * ((k / 2) * n + r) + k % 2;
                const uint32_t *ap = arm + r;
#pragma unroll
                for (int i = 0; i <= kHB; ++i) d[i * kHPitch] = make_float2(0.f, 0.f);
                const int xa = max(bx0 - wx, 0), xb = min(be - 1 + wx, X - 1);
                constexpr int R = 8;
                uint32_t am[R];
                float2 v[R];
                auto load = [&](int x) {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int xi = min(x + i, xb);
                        am[i] = __ldg(ap + xi);
                        v[i] = __ldg(gp + 2 * xi);
                    }
                };
                load(xa);
                for (int x = xa; x <= xb; x += R) {
                    uint32_t ca[R];
                    float2 cv[R];
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        ca[i] = am[i];
                        cv[i] = v[i];
                    }
                    load(x + R);
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int lo = x + i - (int)(ca[i] & 0xFF), hi = x + i + (int)((ca[i] >> 8) & 0xFF);
                        if (x + i <= xb && hi >= bx0 && lo < be) {
                            float2 &p = d[(max(lo, bx0) - bx0) * kHPitch];
                            p = make_float2(p.x + cv[i].x, p.y + cv[i].y);
                            if (hi + 1 < be) {
                                float2 &q = d[(hi + 1 - bx0) * kHPitch];
                                q = make_float2(q.x - cv[i].x, q.y - cv[i].y);
                            }
                        }
                    }
                }
                float2 s = make_float2(0.f, 0.f);
#pragma unroll 8
                for (int i = 0; i < kHB; ++i) {
                    const float2 u = d[i * kHPitch];
                    s = make_float2(s.x + u.x, s.y + u.y);
                    d[i * kHPitch] = s;
                }
            }
        }
        __syncthreads();
        // pairs of column c (from s0) of row j: entries c % kHB of four threads
        auto at = [&](int j, int c) { return dl + (c % kHB) * kHPitch + j * per_row + c / kHB * (kDC / 2); };
        for (int i = threadIdx.x; i < nr * (s2 - s0); i += kHNT) {
            const int j = i >= s2 - s0, x = s0 + i - j * (s2 - s0);
            const size_t r = (size_t)(y + j) * X;
            const float gl = gL[r + x];
            const uint32_t pl = pixL[r + x];
            float2 *gj = at(j, x - s0);
            float g[kDC];
#pragma unroll
            for (int k = 0; k < kDC / 2; ++k) {
                g[2 * k] = gj[k].x;
                g[2 * k + 1] = gj[k].y;
            }
            const bool own = x < s1;
            float al = 0.f, u0 = 0.f, u1 = 0.f, u2 = 0.f, u3 = 0.f;
            // the chunk's disparities unrolled, so their loads and exps overlap
#pragma unroll
            for (int k = 0; k < kDC; ++k) {
                const int d = d0 + k;
                float v = 0.f;
                if (k < kn) {
                    float ea = ea1, a = 1.f;                  // the terms of P (|a| = 1, h = 6)
                    int h = 6;
                    if (x >= d) {
                        const float diff = gl - gR[r + x - d];
                        a = fabsf(diff);
                        h = __popc((pl ^ pixR[r + x - d]) & 0x3F00u);
                        ea = expf(-a * inv_lad);
                        const float sgn = diff > 0.f ? 1.f : (diff < 0.f ? -1.f : 0.f);
                        v = g[k] * kad * ea * sgn;
                    }
                    const float eh = eh_t[h];
                    u0 += g[k] * (1.f - ea);
                    u1 += g[k] * (1.f - eh);
                    u2 += g[k] * (-ea * a * dad);
                    u3 += g[k] * (-eh * (float)h * dmc);
                    al += v;
                }
                g[k] = v;
            }
#pragma unroll
            for (int k = 0; k < kDC / 2; ++k) gj[k] = make_float2(g[2 * k], g[2 * k + 1]);
            if (own) {
                acc_l[r + x] = first ? al : acc_l[r + x] + al;
                kahan(t0, e0, u0);
                kahan(t1, e1, u1);
                kahan(t2, e2, u2);
                kahan(t3, e3, u3);
            }
        }
        __syncthreads();
        // right pixel x is the match of the left pixels x + d0 .. x + d0 + kn - 1
        const int ra = max(s0 - d0, 0), nright = max(s1 - d0 - ra, 0);
        for (int i = threadIdx.x; i < nr * nright; i += kHNT) {
            const int j = i >= nright, x = ra + i - j * nright;
            const size_t r = (size_t)(y + j) * X;
            float ar = 0.f;
#pragma unroll
            for (int k = 0; k < kDC; ++k)
                if (x + d0 + k < s2) {
                    const float2 v = at(j, x + d0 + k - s0)[k / 2];
                    ar -= k % 2 ? v.y : v.x;
                }
            acc_r[r + x] = first ? ar : acc_r[r + x] + ar;
        }
    }
    // block partials of the parameter gradients
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t0 += __shfl_down_sync(0xffffffffu, t0, o);
        t1 += __shfl_down_sync(0xffffffffu, t1, o);
        t2 += __shfl_down_sync(0xffffffffu, t2, o);
        t3 += __shfl_down_sync(0xffffffffu, t3, o);
    }
    if (lane == 0) {
        sh[0][w] = t0;
        sh[1][w] = t1;
        sh[2][w] = t2;
        sh[3][w] = t3;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        float s = 0.f;
        for (int k = 0; k < kHNT / 32; ++k) s += sh[threadIdx.x][k];
        part[b * part_pair + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + threadIdx.x] = s;
    }
}

__global__ void diff_finish_kernel(const float *__restrict__ acc_l, const float *__restrict__ acc_r, int n,
                                   float *__restrict__ grad_l, float *__restrict__ grad_r)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const size_t b = blockIdx.y;                  // pair
    acc_l += b * n;
    acc_r += b * n;
    grad_l += b * n * 3;
    grad_r += b * n * 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        grad_l[3 * i + c] = acc_l[i] * kGreyW[c];
        grad_r[3 * i + c] = acc_r[i] * kGreyW[c];
    }
}

// Sum of all block partials in a fixed order (double accumulation), in two
// levels so that the FP64 adds spread over the GPU. Level 1: block j sums the
// contiguous segment j of the partials (thread t takes its elements t, t +
// kRedNT, ... in turn, then a fixed pairwise tree adds the threads' sums).
// Level 2: one block adds the kRedBlocks segment sums by the same fixed tree.
// Neither order depends on scheduling.
constexpr int kRedNT = 256;
constexpr int kRedBlocks = 128;

__device__ __forceinline__ void tree_sum4(double (*sh)[kRedNT], double s0, double s1, double s2, double s3)
{
    const int t = threadIdx.x;
    sh[0][t] = s0;
    sh[1][t] = s1;
    sh[2][t] = s2;
    sh[3][t] = s3;
    __syncthreads();
    for (int o = kRedNT / 2; o > 0; o >>= 1) {
        if (t < o)
#pragma unroll
            for (int c = 0; c < 4; ++c) sh[c][t] += sh[c][t + o];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kRedNT) diff_theta_segments_kernel(const float *__restrict__ part, int nparts,
                                                                     double *__restrict__ seg)
{
    __shared__ double sh[4][kRedNT];
    const int t = threadIdx.x, len = (nparts + kRedBlocks - 1) / kRedBlocks;
    const int k0 = min(nparts, (int)blockIdx.x * len), k1 = min(nparts, k0 + len);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int k = k0 + t; k < k1; k += kRedNT) {
        const float4 v = *reinterpret_cast<const float4 *>(part + (size_t)k * 4);
        s0 += (double)v.x;
        s1 += (double)v.y;
        s2 += (double)v.z;
        s3 += (double)v.w;
    }
    tree_sum4(sh, s0, s1, s2, s3);
    if (t < 4) seg[blockIdx.x * 4 + t] = sh[t][0];
}

__global__ void __launch_bounds__(kRedNT) diff_theta_reduce_kernel(const double *__restrict__ seg,
                                                                   float *__restrict__ grad)
{
    static_assert(kRedBlocks <= kRedNT, "one segment sum per thread");
    __shared__ double sh[4][kRedNT];
    const int t = threadIdx.x;
    const bool h = t < kRedBlocks;
    tree_sum4(sh, h ? seg[t * 4] : 0.0, h ? seg[t * 4 + 1] : 0.0, h ? seg[t * 4 + 2] : 0.0, h ? seg[t * 4 + 3] : 0.0);
    if (t < 4) grad[t] = (float)sh[t][0];
}

}  // namespace

// Workspace of a batch: per-pair planes [B][...] of each kind, then the
// parameter-gradient partials [B][chunk][block][4]. With base == nullptr
// only the size is computed.
struct DiffWs {
    float *gl, *gr;
    uint8_t *ql, *qr;
    uint32_t *pixl, *pixr, *arml;
    float *ns, *state, *accl, *accr, *s0, *s1, *s2, *part;
    double *seg;
};

size_t diff_layout(char *base, int X, int Y, int B, int D, DiffWs *w)
{
    const size_t n = (size_t)X * Y, nb = (size_t)B;
    const size_t nchunks = (D + kDC - 1) / kDC;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base ? base + off : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    DiffWs t;
    t.gl = (float *)take(nb * n * 4);                        // float grey
    t.gr = (float *)take(nb * n * 4);
    t.ql = (uint8_t *)take(nb * n);                          // integer grey of the uint8 images
    t.qr = (uint8_t *)take(nb * n);
    t.pixl = (uint32_t *)take(nb * n * 4);                   // pixel words, arm words of the left images
    t.pixr = (uint32_t *)take(nb * n * 4);
    t.arml = (uint32_t *)take(nb * n * 4);
    t.ns = (float *)take(nb * n * 4);                        // support size
    t.state = (float *)take(nb * n * 4 * 3);                 // online softmax state
    t.accl = (float *)take(nb * n * 4);                      // intensity-gradient accumulators
    t.accr = (float *)take(nb * n * 4);
    t.s0 = (float *)take(nb * kDC * n * 4);                  // slabs: x sums, their gradient, its vertical adjoint
    t.s1 = (float *)take(nb * kDC * n * 4);
    t.s2 = (float *)take(nb * kDC * n * 4);
    t.part = (float *)take(nb * nchunks * hgrad_blocks(X, Y, (int)nchunks) * 16);   // parameter-gradient partials
    t.seg = (double *)take(kRedBlocks * 4 * sizeof(double)); // their segment sums
    if (w) *w = t;
    return off;
}

size_t diff_workspace_bytes(int X, int Y, int B, int D)
{
    return diff_layout(nullptr, X, Y, B, D, nullptr);
}

cudaError_t diff_setup()
{
    cudaError_t e = cudaFuncSetAttribute(diff_costx_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)costx_smem<256>(4096, kMaxWx));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(diff_costx_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)costx_smem<64>(4096, kMaxWx));
    return e;
}

cudaError_t diff_run(const DiffArgs &a, cudaStream_t s)
{
    const int X = a.W, Y = a.H, n = X * Y, B = a.B;
    DiffWs w;
    diff_layout((char *)a.ws, X, Y, B, a.D, &w);
    const int nblk = (n + kDiffNT - 1) / kDiffNT;
    const int nchunks = (a.D + kDC - 1) / kDC;
    const int nseg = hgrad_segments(X), rows = hgrad_rows(X, nchunks), yblocks = (Y + rows - 1) / rows;
    const size_t part_chunk = (size_t)hgrad_blocks(X, Y, nchunks) * 4, part_pair = part_chunk * nchunks;
    const float inv_tau = 1.f / a.tau;
    const dim3 tiles((X + kTileX - 1) / kTileX, (Y + kTileY - 1) / kTileY, B);
    static_assert(kTileX == 32 && kTileX * kTileY == kDiffNT, "one thread per pixel of a tile, a warp per row");
    cudaError_t e = cudaSuccess;
    // frozen supports of every pair (integer path), support sizes, float grey
    diff_grey_kernel<<<dim3(nblk, 2, B), kDiffNT, 0, s>>>(a.left, a.right, w.gl, w.gr, n);
    // (the arms of the left images only: nothing here uses the right base)
    if ((e = launch_grey(a.left_u8, a.right_u8, w.ql, w.qr, X, Y * B, s)) != cudaSuccess) return e;
    for (int b0 = 0; b0 < B; b0 += kMaxSupImages / 2) {
        SupImage im[kMaxSupImages];
        const int nb = min(B - b0, kMaxSupImages / 2);
        for (int k = 0; k < nb; ++k) {
            const size_t o = (size_t)(b0 + k) * n;
            im[2 * k] = SupImage{w.ql + o, w.pixl + o, w.arml + o, nullptr, nullptr, X, Y, 0};
            im[2 * k + 1] = SupImage{w.qr + o, w.pixr + o, nullptr, nullptr, nullptr, X, Y, 0};
        }
        if ((e = launch_support(im, 2 * nb, a.wx, a.wy, a.tc, a.err, s)) != cudaSuccess) return e;
    }
    diff_nsupport_kernel<<<dim3((X + 31) / 32, (Y + kNSRows - 1) / kNSRows, B), kDiffNT, 0, s>>>(w.arml, X, Y, w.ns);
    float4 *hs = (float4 *)w.s0;                      // x sums
    const dim3 vgrid((X + kVTNT / kDC - 1) / (kVTNT / kDC), (Y + kVB - 1) / kVB, B);
    // narrow segments where wide ones would not give every SM two blocks
    const bool narrow = (long)((X + 255) / 256) * ((Y + 3) / 4) * B < 304;
    const int seg = narrow ? 64 : 256;
    const dim3 cgrid((X + seg - 1) / seg, (Y + 3) / 4, B);
    for (int c = 0; c < nchunks && e == cudaSuccess; ++c) {
        const int d0 = c * kDC;
        e = launch_dependent(narrow ? diff_costx_kernel<64> : diff_costx_kernel<256>, cgrid, dim3(kDiffNT),
                             narrow ? costx_smem<64>(X, a.wx) : costx_smem<256>(X, a.wx), s, w.gl, w.gr, w.pixl,
                             w.pixr, w.arml, a.theta, X, Y, a.D, d0, a.wx, hs);
        if (e != cudaSuccess) break;
        if (!a.backward) {
            e = launch_dependent(a.wy ? diff_vagg_softmax_kernel<true> : diff_vagg_softmax_kernel<false>, tiles,
                                 dim3(kDiffNT), 0, s, hs, w.arml, w.ns, X, Y, a.D, d0, inv_tau, w.state, c == 0,
                                 c == nchunks - 1, a.dhat, a.stats);
            continue;
        }
        if ((e = launch_dependent(a.wy ? diff_gca_kernel<true> : diff_gca_kernel<false>, tiles, dim3(kDiffNT), 0, s, hs,
                                  w.arml, w.ns, X, Y, a.D, d0, inv_tau, a.dhat, a.stats, a.grad_dhat,
                                  (float4 *)w.s1)) != cudaSuccess ||
            (e = launch_dependent(diff_vT_kernel, vgrid, dim3(kVTNT), 0, s, w.s1, w.arml, X, Y, a.wy, w.s2)) !=
                cudaSuccess)
            break;
        e = launch_dependent(diff_hgrad_kernel, dim3(nseg, yblocks, B), dim3(kHNT), 0, s, w.s2,
                             w.arml, w.gl, w.gr, w.pixl, w.pixr, a.theta, X, Y, a.D, d0, a.wx, rows, c == 0, w.accl,
                             w.accr, w.part + c * part_chunk, part_pair);
    }
    if (e != cudaSuccess) return e;
    if (a.backward) {
        diff_finish_kernel<<<dim3(nblk, B), kDiffNT, 0, s>>>(w.accl, w.accr, n, a.grad_left, a.grad_right);
        diff_theta_segments_kernel<<<kRedBlocks, kRedNT, 0, s>>>(w.part, (int)(part_pair / 4 * B), w.seg);
        diff_theta_reduce_kernel<<<1, kRedNT, 0, s>>>(w.seg, a.grad_theta);
    }
    return cudaGetLastError();
}

}  // namespace stereo
