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
// the slab's gradients, all as [y][x][kDC] so that a pixel's disparities are two
// 16-byte accesses. Every pair of the batch has its own buffers, and the
// per-chunk kernels take all pairs in one launch.
//
// Sums over arms run over whole blocks of four cells where the window holds
// them and single cells at its ends (step4), at most 3 + 10 + 3 terms along x
// and 3 + 15 + 3 along y for the default caps: every term is a sum of cells of
// the window itself, so an aggregate keeps the accuracy of a direct sum and a
// NaN stays in the windows that hold it. The adjoint of each sum is a banded
// difference array walked in a fixed order by one thread, so no float atomics
// are used and results are deterministic.
//
// 4 pairs of 718 x 496, D 73, forward and backward (arms at their caps in a third
// of the planes): 9.1 ms with direct sums over planes [kDC][y][x] and separate
// kernels for the horizontal adjoint and the cost gradient, 4.2 ms now. Bound by
// the L1 traffic of the vertical sums and the dependent chains of the adjoints.
#include "internal.cuh"

namespace stereo {

constexpr int kDiffNT = 256;   // threads of the per-pixel kernels

namespace {

constexpr int kDC = 8;   // disparities per chunk
// pixel tiles of the kernels that sum along y (blocks of kTileX * kTileY = 256 threads)
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

// Support size n(x,y) = sum over the vertical span of each row's x window.
__global__ void diff_nsupport_kernel(const uint32_t *__restrict__ arm, int X, int Y, float *__restrict__ ns)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= X * Y) return;
    const size_t b = blockIdx.y;                  // pair
    arm += b * X * Y;
    ns += b * X * Y;
    const int y = i / X, x = i - y * X;
    const uint32_t a = arm[i];
    const int up = (a >> 16) & 0xFF, down = a >> 24;
    int s = 0;
    for (int t = -up; t <= down; ++t) {
        const uint32_t b = arm[(size_t)(y + t) * X + x];
        s += (int)(b & 0xFF) + (int)((b >> 8) & 0xFF) + 1;
    }
    ns[i] = (float)s;
}

struct Theta {
    float wad, wmc, lad, lmc;
};

__device__ __forceinline__ Theta load_theta(const float *t) { return Theta{t[0], t[1], t[2], t[3]}; }

__device__ __forceinline__ void add4(float (&s)[kDC], int j, const float4 v)
{
    s[j] += v.x;
    s[j + 1] += v.y;
    s[j + 2] += v.z;
    s[j + 3] += v.w;
}

// The next term of a window sum over [t, hi]: a whole aligned block of four cells
// if the window holds it, else cell t.
__device__ __forceinline__ bool step4(int t, int hi) { return (t & 3) == 0 && t + 3 <= hi; }

// Cost and x window sums. A block takes kCXSeg columns of a row quad: the costs
// of the chunk's disparities for those columns and a wx halo go to shared memory
// (two float4 planes per row), with the sums of aligned column quads beside
// them; then a thread owns one column and sums its own windows. It also writes
// the sum of its four rows, the blocks of the vertical sums.
constexpr int kCXSeg = 256;
static_assert(kCXSeg == kDiffNT, "one column per thread");

__host__ __device__ __forceinline__ int costx_pitch(int X, int wx)
{
    return ((X < kCXSeg + 2 * wx + 4 ? X : kCXSeg + 2 * wx + 4) + 3) / 4 * 4;
}
size_t diff_costx_smem(int X, int wx) { return (size_t)costx_pitch(X, wx) * 5 / 4 * 4 * 2 * sizeof(float4); }

__global__ void __launch_bounds__(kDiffNT) diff_costx_kernel(
    const float *__restrict__ gL, const float *__restrict__ gR, const uint32_t *__restrict__ pixL,
    const uint32_t *__restrict__ pixR, const uint32_t *__restrict__ arm, const float *__restrict__ theta, int X, int Y,
    int D, int d0, int wx, float4 *__restrict__ hs, float4 *__restrict__ bs)
{
    extern __shared__ float4 csm[];
    __shared__ float mc[8];
    pdl_trigger();
    const int x0 = blockIdx.x * kCXSeg, y0 = blockIdx.y * 4;
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    const int P = costx_pitch(X, wx);
    float4 *cell = csm, *quad = csm + 8 * P;          // [4 rows][2][P], [4 rows][2][P / 4]
    pdl_wait();
    gL += b * n;
    gR += b * n;
    pixL += b * n;
    pixR += b * n;
    arm += b * n;
    hs += b * 2 * n;
    bs += b * 2 * X * (size_t)((Y + 3) / 4);
    const Theta th = load_theta(theta);
    const float Pc = th.wad * (1.f - expf(-1.f / th.lad)) + th.wmc * (1.f - expf(-6.f / th.lmc));
    const int kn = min(kDC, D - d0);
    // the census term takes seven values: one exp per Hamming distance
    if (threadIdx.x < 7) mc[threadIdx.x] = th.wmc * (1.f - expf(-(float)threadIdx.x / th.lmc));
    const float inv_lad = 1.f / th.lad;
    const int xs = max(x0 - wx, 0) & ~3, xe = min(x0 + kCXSeg + wx, X);   // staged columns
    __syncthreads();
    for (int r = 0; r < 4 && y0 + r < Y; ++r) {
        const size_t row = (size_t)(y0 + r) * X;
        for (int x = xs + (int)threadIdx.x; x < xe; x += kDiffNT) {
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
            cell[(2 * r) * P + x - xs] = make_float4(c[0], c[1], c[2], c[3]);
            cell[(2 * r + 1) * P + x - xs] = make_float4(c[4], c[5], c[6], c[7]);
        }
    }
    __syncthreads();
    const int nq = (xe - xs) / 4;                     // whole quads
    for (int i = threadIdx.x; i < 8 * nq; i += kDiffNT) {
        const int j = i / nq, q = i - j * nq;
        if (y0 + j / 2 >= Y) break;
        const float4 *c = cell + j * P + 4 * q;
        const float4 u = c[0], v = c[1], w = c[2], z = c[3];
        quad[j * (P / 4) + q] = make_float4(u.x + v.x + w.x + z.x, u.y + v.y + w.y + z.y, u.z + v.z + w.z + z.z,
                                            u.w + v.w + w.w + z.w);
    }
    __syncthreads();
    const int x = x0 + threadIdx.x;
    if (x >= X) return;
    float sum[kDC];
#pragma unroll
    for (int k = 0; k < kDC; ++k) sum[k] = 0.f;
    for (int r = 0; r < 4 && y0 + r < Y; ++r) {
        const size_t i = (size_t)(y0 + r) * X + x;
        const uint32_t am = arm[i];
        const int hi = x + (int)((am >> 8) & 0xFF) - xs;
        const float4 *c0 = cell + 2 * r * P, *q0 = quad + 2 * r * (P / 4);
        float s[kDC];
#pragma unroll
        for (int k = 0; k < kDC; ++k) s[k] = 0.f;
        for (int t = x - (int)(am & 0xFF) - xs; t <= hi;) {
            const bool four = step4(t, hi);
            const float4 *p = four ? q0 + (t >> 2) : c0 + t;
            add4(s, 0, p[0]);
            add4(s, 4, p[four ? P / 4 : P]);
            t += four ? 4 : 1;
        }
        hs[2 * i] = make_float4(s[0], s[1], s[2], s[3]);
        hs[2 * i + 1] = make_float4(s[4], s[5], s[6], s[7]);
#pragma unroll
        for (int k = 0; k < kDC; ++k) sum[k] += s[k];
    }
    float4 *o = bs + 2 * ((size_t)(y0 / 4) * X + x);
    o[0] = make_float4(sum[0], sum[1], sum[2], sum[3]);
    o[1] = make_float4(sum[4], sum[5], sum[6], sum[7]);
}

// Vertical sums of Eq. 8 for the chunk's disparities at once, over the anchor's
// span [y - up, y + down]: row sums at its ends, the sums of whole row quads
// between.
__device__ __forceinline__ void vsum_chunk(const float4 *__restrict__ hs, const float4 *__restrict__ bs,
                                           const uint32_t am, int x, int y, int X, float (&out)[kDC])
{
#pragma unroll
    for (int k = 0; k < kDC; ++k) out[k] = 0.f;
    const int hi = y + (int)(am >> 24);
    hs += 2 * x;
    bs += 2 * x;
    for (int t = y - (int)((am >> 16) & 0xFF); t <= hi;) {
        const bool four = step4(t, hi);
        const float4 *p = (four ? bs : hs) + (size_t)(four ? t >> 2 : t) * (2 * X);
        add4(out, 0, p[0]);
        add4(out, 4, p[1]);
        t += four ? 4 : 1;
    }
}

// Forward: aggregated cost along y per pixel and an online softmax over d.
// state = (max z, sum exp(z - max), sum d exp(z - max)) per pixel.
__global__ void diff_vagg_softmax_kernel(const float4 *__restrict__ hs, const float4 *__restrict__ bs,
                                         const uint32_t *__restrict__ arm, const float *__restrict__ ns, int X, int Y,
                                         int D, int d0, float inv_tau, float *__restrict__ state, int first, int last,
                                         float *__restrict__ dhat, float *__restrict__ stats)
{
    pdl_trigger();
    // 2-D tiles of kTileX x kTileY pixels: the warps of a block walk the
    // same anchor rows, so their vertical windows meet in L1
    const int x = blockIdx.x * kTileX + (int)(threadIdx.x % kTileX);
    const int y = blockIdx.y * kTileY + (int)(threadIdx.x / kTileX);
    pdl_wait();
    if (x >= X || y >= Y) return;
    const int i = y * X + x;
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    hs += b * 2 * n;
    bs += b * 2 * X * (size_t)((Y + 3) / 4);
    arm += b * n;
    ns += b * n;
    state += b * 3 * n;
    dhat += b * n;
    stats += b * 2 * n;
    const uint32_t am = arm[i];
    const float inv_n = 1.f / ns[i];
    float m = first ? -INFINITY : state[3 * i], s = first ? 0.f : state[3 * i + 1],
          sd = first ? 0.f : state[3 * i + 2];
    float ca[kDC];
    vsum_chunk(hs, bs, am, x, y, X, ca);
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
__global__ void diff_gca_kernel(const float4 *__restrict__ hs, const float4 *__restrict__ bs,
                                const uint32_t *__restrict__ arm, const float *__restrict__ ns, int X, int Y, int D,
                                int d0, float inv_tau, const float *__restrict__ dhat, const float *__restrict__ stats,
                                const float *__restrict__ go, float4 *__restrict__ g0)
{
    pdl_trigger();
    const int x = blockIdx.x * kTileX + (int)(threadIdx.x % kTileX);
    const int y = blockIdx.y * kTileY + (int)(threadIdx.x / kTileX);
    pdl_wait();
    if (x >= X || y >= Y) return;
    const int i = y * X + x;
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    hs += b * 2 * n;
    bs += b * 2 * X * (size_t)((Y + 3) / 4);
    arm += b * n;
    ns += b * n;
    dhat += b * n;
    stats += b * 2 * n;
    go += b * n;
    g0 += b * 2 * n;
    const uint32_t am = arm[i];
    const float inv_n = 1.f / ns[i];
    const float m = stats[2 * i], s = stats[2 * i + 1], e = dhat[i], gi = go[i];
    float ca[kDC], v[kDC];
    vsum_chunk(hs, bs, am, x, y, X, ca);
#pragma unroll
    for (int k = 0; k < kDC; ++k) {
        v[k] = 0.f;
        if (d0 + k < D) {
            const float z = -(ca[k] * inv_n) * inv_tau;
            const float p = expf(z - m) / s;
            v[k] = gi * p * ((float)(d0 + k) - e) * (-inv_tau) * inv_n;
        }
    }
    g0[2 * (size_t)i] = make_float4(v[0], v[1], v[2], v[3]);
    g0[2 * (size_t)i + 1] = make_float4(v[4], v[5], v[6], v[7]);
}

// Backward 2: adjoint of the vertical sum. G1(x, y') collects the anchors
// (x, y) whose span [y - up, y + down] contains y'. As a difference array: a
// thread owns one column and one disparity of the chunk over a band of kVB
// rows; every anchor whose span reaches the band adds its value at the band
// row where the span enters and subtracts it one row past where the span
// ends (anchors in ascending y), and a running sum down the band gives G1.
// Each thread works alone in a fixed order: deterministic, no atomics, and
// about 2 (kVB + 2 wy) / kVB operations per output instead of 2 wy + 1.
constexpr int kVB = 32;
static_assert(kDiffNT == 32 * kDC, "a block is 32 columns x the chunk's disparities");
__global__ void __launch_bounds__(kDiffNT) diff_vT_kernel(const float *__restrict__ g0,
                                                          const uint32_t *__restrict__ arm, int X, int Y, int wy,
                                                          float *__restrict__ g1)
{
    __shared__ float delta[kDiffNT][kVB + 1];     // odd pitch: the lanes of a warp hit distinct banks
    pdl_trigger();
    const int k = threadIdx.x % kDC, xi = threadIdx.x / kDC;   // 32 columns x kDC disparities
    const int x = blockIdx.x * 32 + xi, y0 = blockIdx.y * kVB;
    pdl_wait();
    if (x >= X) return;
    const size_t b = blockIdx.z, n = (size_t)X * Y;   // pair
    arm += b * n + x;
    const float *gp = g0 + (b * n + x) * kDC + k;
    float *out = g1 + (b * n + x) * kDC + k;
    float *dl = delta[threadIdx.x];
    const int ye = min(y0 + kVB, Y);              // band rows [y0, ye)
#pragma unroll
    for (int i = 0; i <= kVB; ++i) dl[i] = 0.f;
    const int ya = max(y0 - wy, 0), yb = min(ye - 1 + wy, Y - 1);
#pragma unroll 8
    for (int y = ya; y <= yb; ++y) {
        const uint32_t am = __ldg(arm + (size_t)y * X);
        const float v = __ldg(gp + (size_t)y * X * kDC);   // rows [ya, yb] are in the image: loaded ahead of the test
        const int lo = y - (int)((am >> 16) & 0xFF), hi = y + (int)(am >> 24);
        if (hi >= y0 && lo < ye) {
            dl[max(lo, y0) - y0] += v;
            if (hi + 1 < ye) dl[hi + 1 - y0] -= v;
        }
    }
    float s = 0.f;
    for (int i = 0; i < ye - y0; ++i) {
        s += dl[i];
        out[(size_t)(y0 + i) * X * kDC] = s;
    }
}

// Backward 3 and 4 in one: the adjoint of the horizontal sum, then through the
// cost. A block takes one row segment of up to kHSeg - kDC + 1 columns of one
// pair.
//  * G2(x', y) collects the pixels (x, y) whose own window [x - left, x + right]
//    contains x'. The chunk's G1 values and the arm words of the segment, its
//    next kDC - 1 columns and a wx halo are staged in shared memory; a thread
//    owns one disparity and a band of kHB columns: each pixel whose window
//    reaches the band adds its value where the window enters and subtracts it
//    one column past where it ends (pixels in ascending x), and a running sum
//    gives the band. The staged columns skip one every 16, so that the bands of
//    a warp read distinct banks.
//  * A cell (x, y, d) passes v = G2 dC/dgL to its left pixel and -v to the right
//    pixel x - d: v goes through shared memory, and the block takes the right
//    pixels whose cells of this chunk all lie in its columns. The four
//    parameters get one partial per block, summed later in a fixed order.
constexpr int kHSeg = 512, kHB = 16;
static_assert(kHSeg / kHB * kDC == kDiffNT, "one (band, disparity) per thread");
__host__ __device__ __forceinline__ int hpad(int i) { return i + (i >> 4); }
__host__ __device__ __forceinline__ int hgrad_segments(int X) { return (X + kHSeg - kDC) / (kHSeg - kDC + 1); }

size_t diff_hgrad_smem(int wx)
{
    const int span = hpad(kHSeg + 2 * wx) + 1;
    return (size_t)span * kDC * 4 + (size_t)span * 4 + (size_t)kDiffNT * (kHB + 1) * 4;
}
static_assert(kDiffNT * (kHB + 1) >= kDC * kHSeg, "the difference arrays' space takes the cells' values");

__global__ void __launch_bounds__(kDiffNT) diff_hgrad_kernel(
    const float *__restrict__ g1, const uint32_t *__restrict__ arm, const float *__restrict__ gL,
    const float *__restrict__ gR, const uint32_t *__restrict__ pixL, const uint32_t *__restrict__ pixR,
    const float *__restrict__ theta, int X, int Y, int D, int d0, int wx, int rows, int first,
    float *__restrict__ acc_l, float *__restrict__ acc_r, float *__restrict__ part, size_t part_pair)
{
    extern __shared__ __align__(16) float hsm[];
    __shared__ float eh_t[8];
    __shared__ float sh[4][kDiffNT / 32];
    pdl_trigger();
    const int span = hpad(kHSeg + 2 * wx) + 1;
    float *gs = hsm;                                          // [span][kDC] staged G1, then G2
    uint32_t *as = reinterpret_cast<uint32_t *>(hsm + span * kDC);   // [span] arm words
    float *delta = hsm + span * (kDC + 1);                    // [kDiffNT][kHB + 1], then v [kDC][kHSeg]
    const int nseg = hgrad_segments(X), seg = (X + nseg - 1) / nseg;
    const int s0 = blockIdx.x * seg, s1 = min(s0 + seg, X);   // the segment's left pixels
    const int s2 = min(s1 + kDC - 1, X);                      // the columns whose cells it needs
    const int xs = s0 - wx;                                   // column of staged index 0
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
    float t0 = 0.f, t1 = 0.f, t2 = 0.f, t3 = 0.f;
    for (int y = blockIdx.y * rows; y < min(((int)blockIdx.y + 1) * rows, Y); ++y) {
        const size_t r = (size_t)y * X;
        __syncthreads();                                      // the previous row is done with shared memory
        const int sa = max(xs, 0), sb = min(s2 + wx, X);
        for (int i = threadIdx.x; i < (sb - sa) * 2; i += kDiffNT) {
            const int x = sa + (i >> 1);
            reinterpret_cast<float4 *>(gs)[hpad(x - xs) * 2 + (i & 1)] =
                __ldg(reinterpret_cast<const float4 *>(g1) + (r + x) * 2 + (i & 1));
        }
        for (int x = sa + (int)threadIdx.x; x < sb; x += kDiffNT) as[hpad(x - xs)] = __ldg(arm + r + x);
        __syncthreads();
        {
            const int k = threadIdx.x % kDC, bx0 = s0 + kHB * (int)(threadIdx.x / kDC);
            const int be = min(bx0 + kHB, s2);                // band columns [bx0, be)
            float *dl = delta + threadIdx.x * (kHB + 1);
            float acc[kHB];
            const bool work = bx0 < be;
            if (work) {
#pragma unroll
                for (int i = 0; i <= kHB; ++i) dl[i] = 0.f;
                const int xa = max(bx0 - wx, 0), xb = min(be - 1 + wx, X - 1);
#pragma unroll 4
                for (int x = xa; x <= xb; ++x) {
                    const uint32_t am = as[hpad(x - xs)];
                    const float v = gs[hpad(x - xs) * kDC + k];
                    const int lo = x - (int)(am & 0xFF), hi = x + (int)((am >> 8) & 0xFF);
                    if (hi >= bx0 && lo < be) {
                        dl[max(lo, bx0) - bx0] += v;
                        if (hi + 1 < be) dl[hi + 1 - bx0] -= v;
                    }
                }
                float s = 0.f;
#pragma unroll
                for (int i = 0; i < kHB; ++i) {
                    s += dl[i];
                    acc[i] = s;
                }
            }
            __syncthreads();                                  // every thread is done with the staged values
            if (work)
#pragma unroll
                for (int i = 0; i < kHB; ++i)
                    if (bx0 + i < be) gs[hpad(bx0 + i - xs) * kDC + k] = acc[i];
        }
        __syncthreads();
        for (int x = s0 + (int)threadIdx.x; x < s2; x += kDiffNT) {
            const float gl = gL[r + x];
            const uint32_t pl = pixL[r + x];
            const float4 ga = *reinterpret_cast<const float4 *>(gs + hpad(x - xs) * kDC);
            const float4 gb = *reinterpret_cast<const float4 *>(gs + hpad(x - xs) * kDC + 4);
            const float g[kDC] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
            const bool own = x < s1;
            float al = 0.f;
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
                    if (own) {
                        const float eh = eh_t[h];
                        t0 += g[k] * (1.f - ea);
                        t1 += g[k] * (1.f - eh);
                        t2 += g[k] * (-ea * a * dad);
                        t3 += g[k] * (-eh * (float)h * dmc);
                        al += v;
                    }
                }
                delta[k * kHSeg + x - s0] = v;
            }
            if (own) acc_l[r + x] = first ? al : acc_l[r + x] + al;
        }
        __syncthreads();
        // right pixel x is the match of the left pixels x + d0 .. x + d0 + kn - 1
        for (int x = max(s0 - d0, 0) + (int)threadIdx.x; x < s1 - d0; x += kDiffNT) {
            float ar = 0.f;
#pragma unroll
            for (int k = 0; k < kDC; ++k)
                if (x + d0 + k < s2) ar -= delta[k * kHSeg + x + d0 + k - s0];
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
        for (int k = 0; k < kDiffNT / 32; ++k) s += sh[threadIdx.x][k];
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
    uint32_t *pixl, *pixr, *arml, *armr, *armcl, *armcr, *keyl, *keyr;
    float *ns, *state, *accl, *accr, *s0, *s1, *s2, *s3, *part;
    double *seg;
};

size_t diff_layout(char *base, int X, int Y, int wy, int B, int D, DiffWs *w)
{
    const size_t n = (size_t)X * Y, nb = (size_t)B;
    const size_t nblk = (n + kDiffNT - 1) / kDiffNT;
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
    t.pixl = (uint32_t *)take(nb * n * 4);                   // pixel and arm words
    t.pixr = (uint32_t *)take(nb * n * 4);
    t.arml = (uint32_t *)take(nb * n * 4);
    t.armr = (uint32_t *)take(nb * n * 4);
    t.armcl = (uint32_t *)take(nb * armc_words(X, Y, wy) * 4);
    t.armcr = (uint32_t *)take(nb * armc_words(X, Y, wy) * 4);
    t.keyl = (uint32_t *)take(nb * n * 4);                   // keys (written by the support pass)
    t.keyr = (uint32_t *)take(nb * n * 4);
    t.ns = (float *)take(nb * n * 4);                        // support size
    t.state = (float *)take(nb * n * 4 * 3);                 // online softmax state
    t.accl = (float *)take(nb * n * 4);                      // intensity-gradient accumulators
    t.accr = (float *)take(nb * n * 4);
    t.s0 = (float *)take(nb * kDC * n * 4);                  // slabs
    t.s1 = (float *)take(nb * kDC * n * 4);
    t.s2 = (float *)take(nb * kDC * n * 4);
    t.s3 = (float *)take(nb * kDC * n * 4);
    t.part = (float *)take(nb * nchunks * nblk * 16);        // parameter-gradient partials
    t.seg = (double *)take(kRedBlocks * 4 * sizeof(double)); // their segment sums
    if (w) *w = t;
    return off;
}

size_t diff_workspace_bytes(int X, int Y, int wy, int B, int D)
{
    return diff_layout(nullptr, X, Y, wy, B, D, nullptr);
}

cudaError_t diff_setup()
{
    cudaError_t e = cudaFuncSetAttribute(diff_costx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)diff_costx_smem(4096, kMaxWx));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(diff_hgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)diff_hgrad_smem(kMaxWx));
}

cudaError_t diff_run(const DiffArgs &a, cudaStream_t s)
{
    const int X = a.W, Y = a.H, n = X * Y, B = a.B;
    DiffWs w;
    diff_layout((char *)a.ws, X, Y, a.wy, B, a.D, &w);
    const int nblk = (n + kDiffNT - 1) / kDiffNT;
    const int nchunks = (a.D + kDC - 1) / kDC;
    // parameter-gradient partials, one per block of the cost gradient: they
    // take the planes [armr, ns) that this form leaves unused, with more rows
    // to a block where a narrow image's would not hold them
    const size_t room = (size_t)((char *)w.ns - (char *)w.armr);
    const int nseg = hgrad_segments(X);
    int rows = 1;
    while ((size_t)B * nchunks * nseg * ((Y + rows - 1) / rows) * 16 > room) ++rows;
    const int yblocks = (Y + rows - 1) / rows;
    float *part = (float *)w.armr;
    const size_t part_chunk = (size_t)nseg * yblocks * 4, part_pair = part_chunk * nchunks;
    const float inv_tau = 1.f / a.tau;
    const dim3 tiles((X + kTileX - 1) / kTileX, (Y + kTileY - 1) / kTileY, B);
    static_assert(kTileX * kTileY == kDiffNT, "one thread per pixel of a tile");
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
    diff_nsupport_kernel<<<dim3(nblk, B), kDiffNT, 0, s>>>(w.arml, X, Y, w.ns);
    float4 *hs = (float4 *)w.s0, *bs = (float4 *)w.s3;   // x sums, their row-quad sums
    const dim3 cgrid((X + kCXSeg - 1) / kCXSeg, (Y + 3) / 4, B);
    for (int c = 0; c < nchunks && e == cudaSuccess; ++c) {
        const int d0 = c * kDC;
        e = launch_dependent(diff_costx_kernel, cgrid, dim3(kDiffNT), diff_costx_smem(X, a.wx), s, w.gl, w.gr, w.pixl,
                             w.pixr, w.arml, a.theta, X, Y, a.D, d0, a.wx, hs, bs);
        if (e != cudaSuccess) break;
        if (!a.backward) {
            e = launch_dependent(diff_vagg_softmax_kernel, tiles, dim3(kDiffNT), 0, s, hs, bs, w.arml, w.ns, X, Y, a.D,
                                 d0, inv_tau, w.state, c == 0, c == nchunks - 1, a.dhat, a.stats);
            continue;
        }
        if ((e = launch_dependent(diff_gca_kernel, tiles, dim3(kDiffNT), 0, s, hs, bs, w.arml, w.ns, X, Y, a.D, d0,
                                  inv_tau, a.dhat, a.stats, a.grad_dhat, (float4 *)w.s1)) != cudaSuccess ||
            (e = launch_dependent(diff_vT_kernel, dim3((X + 31) / 32, (Y + kVB - 1) / kVB, B), dim3(kDiffNT), 0, s,
                                  w.s1, w.arml, X, Y, a.wy, w.s2)) != cudaSuccess)
            break;
        e = launch_dependent(diff_hgrad_kernel, dim3(nseg, yblocks, B), dim3(kDiffNT), diff_hgrad_smem(a.wx), s, w.s2,
                             w.arml, w.gl, w.gr, w.pixl, w.pixr, a.theta, X, Y, a.D, d0, a.wx, rows, c == 0, w.accl,
                             w.accr, part + c * part_chunk, part_pair);
    }
    if (e != cudaSuccess) return e;
    if (a.backward) {
        diff_finish_kernel<<<dim3(nblk, B), kDiffNT, 0, s>>>(w.accl, w.accr, n, a.grad_left, a.grad_right);
        diff_theta_segments_kernel<<<kRedBlocks, kRedNT, 0, s>>>(part, (int)(part_pair / 4 * B), w.seg);
        diff_theta_reduce_kernel<<<1, kRedNT, 0, s>>>(w.seg, a.grad_theta);
    }
    return cudaGetLastError();
}

}  // namespace stereo
