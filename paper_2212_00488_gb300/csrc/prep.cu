// Preprocessing kernels: grey conversion (Sec. III step 1), 2x mean-pool
// downscale (Sec. III-A, Eq. 2), and the per-pixel support data of the fused
// kernel: mini-census code (Sec. III-B) and the four cross arms (Sec. III-C).
// These are short passes over a few MB: each pixel is read from HBM once,
// the grey + downscale pass keeps its neighbourhoods in registers and the
// support pass stages them in shared memory.
#include "internal.cuh"

#include <type_traits>

namespace stereo {
namespace {

__device__ __forceinline__ uint32_t luma(uint32_t r, uint32_t g, uint32_t b)
{
    // Step 1 gives no formula: BT.601 weights in 8-bit fixed point, rounded.
    return (77u * r + 150u * g + 29u * b + 128u) >> 8;
}

// The weights of luma() as the bytes of one word (r in byte 0).
constexpr uint32_t kLumaW = 77u | (150u << 8) | (29u << 16);

// luma() of the four pixels in three aligned words (w0 = r0 g0 b0 r1, w1 =
// g1 b1 r2 g2, w2 = b2 r3 g3 b3), packed one grey byte per pixel: each
// weighted sum is a four-byte dot product of the pixel's (r, g, b, -) bytes
// with (77, 150, 29, 0), and its byte 1 is the grey value (sum >> 8).
__device__ __forceinline__ uint32_t luma4(uint32_t w0, uint32_t w1, uint32_t w2)
{
    const uint32_t l0 = __dp4a(w0, kLumaW, 128u);
    const uint32_t l1 = __dp4a(__funnelshift_r(w0, w1, 24), kLumaW, 128u);
    const uint32_t l2 = __dp4a(__funnelshift_r(w1, w2, 16), kLumaW, 128u);
    const uint32_t l3 = __dp4a(w2, kLumaW << 8, 128u);
    return __byte_perm(__byte_perm(l0, l1, 0x5151), __byte_perm(l2, l3, 0x5151), 0x5410);
}

// RGB (HWC) -> grey for both images (blockIdx.y selects the image). Each
// thread converts four consecutive pixels; with a 4-byte aligned source those
// twelve bytes are three aligned 32-bit loads.
template <bool kAligned>
__global__ void grey_kernel(const uint8_t *__restrict__ rgb_l, const uint8_t *__restrict__ rgb_r,
                            uint8_t *__restrict__ g_l, uint8_t *__restrict__ g_r, long n)
{
    const uint8_t *rgb = blockIdx.y ? rgb_r : rgb_l;
    uint8_t *g = blockIdx.y ? g_r : g_l;
    long p = 4 * ((long)blockIdx.x * blockDim.x + threadIdx.x);
    if (p >= n) return;
    if (kAligned && p + 4 <= n) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(rgb + 3 * p);
        *reinterpret_cast<uint32_t *>(g + p) = luma4(__ldg(w), __ldg(w + 1), __ldg(w + 2));
    } else {
        for (long q = p; q < p + 4 && q < n; ++q)
            g[q] = (uint8_t)luma(rgb[3 * q], rgb[3 * q + 1], rgb[3 * q + 2]);
    }
}

// Grey conversion and Eq. 2 downscale in one pass (the downscaling path): with K =
// 2, m = 1 the mean of the 3x3 window centred on (2x, 2y), coordinates clamped to
// the image, rounded half up: (sum + 4) / 9. Thread (band, c) of one image owns
// full-res columns 4c .. 4c + 3 and makes the means of output columns 2c, 2c + 1, rows
// 4 band .. 4 band + 3. It converts rows 8 band - 1 .. 8 band + 7 of its columns (row
// coordinates clamped), each from three words, all requested before the first is
// used; the grey of pixel 4c - 1 comes from its left neighbour (a shuffle; lane 0
// loads it itself). A window's last column 2x + 1 always lies in the image. Grey
// values stay in registers; the left image's full-res grey of rows 8 band .. 8
// band + 7 is written for the scale-up. Bands cover ceil(H / 2) rows so that the
// last row of an odd H gets its grey.
//
// kAligned: W a multiple of 4 and word-aligned rows. Else a row's words are funnel
// shifts of the aligned words that hold its pixels, the last group of a row may
// be partial, and stores go by halfwords or bytes (1482 x 994: 10.3 us as two
// kernels, 8.8 as one with a branch a row, 5.8 now). The frames of a batch share a launch of each kind.
constexpr int kGDT = 128;                  // threads per CTA
constexpr int kGDB = 4;                    // output rows per thread
constexpr int kGDR = 2 * kGDB + 1;         // full-res rows per thread

template <int N>
struct GreyArgs {
    int n;
    int start[N + 1];                      // first CTA of each image (two per frame)
    GreyJob job[N / 2];
};

template <bool kAligned, int N>
__global__ void __launch_bounds__(kGDT) grey_down_kernel(const __grid_constant__ GreyArgs<N> A)
{
    pdl_trigger();
    int im = 0;
    while (im + 1 < A.n && (int)blockIdx.x >= A.start[im + 1]) ++im;
    const GreyJob &J = A.job[im >> 1];
    const bool right = im & 1;
    const int W = J.W, H = J.H, X = W / 2, Y = H / 2;
    const int ncol = (W + 3) / 4, nthr = ncol * (((H + 1) / 2 + kGDB - 1) / kGDB);
    const int t0 = ((int)blockIdx.x - A.start[im]) * kGDT + threadIdx.x;
    // threads past the end take the last thread's pixels for the shuffles
    // and store nothing
    const bool live = t0 < nthr;
    const int t = live ? t0 : nthr - 1;
    const int band = t / ncol, c = t - band * ncol;   // left neighbour (band, c - 1) is thread t - 1
    const int lane = threadIdx.x & 31;
    const uint8_t *rgb = right ? J.rgb_r : J.rgb_l;
    uint8_t *s = right ? J.s_r : J.s_l, *gf = J.gf_l;
    const int nc = min(4, W - 4 * c);                 // columns of the group
    const uint8_t *end = rgb + (size_t)W * H * 3;
    pdl_wait();   // launched early behind the previous frame's last kernel, which still reads gf and s
    uint32_t w[kGDR][3], wh[kGDR];
#pragma unroll
    for (int r = 0; r < kGDR; ++r) {
        const int fy = min(max(8 * band - 1 + r, 0), H - 1);
        const uint8_t *p = rgb + ((size_t)fy * W + 4 * c) * 3;
        if (kAligned) {
            const uint32_t *q = reinterpret_cast<const uint32_t *>(p);
#pragma unroll
            for (int i = 0; i < 3; ++i) w[r][i] = __ldg(q + i);
            wh[r] = lane == 0 && c > 0 ? __ldg(q - 1) : 0u;
        } else {
            // Sixteen aligned bytes hold the group's twelve; a partial group takes
            // bytes of the next row along, which no result of the image uses.
            const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3) * 8;
            const uint32_t *q = reinterpret_cast<const uint32_t *>(p - sh / 8);
            uint32_t a[4] = {0, 0, 0, 0}, h = 0;
            if (reinterpret_cast<const uint8_t *>(q + 4) <= end) {
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = __ldg(q + i);
                if (lane == 0 && c > 0) h = __ldg(q - 1);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) w[r][i] = __funnelshift_r(a[i], a[i + 1], sh);
            wh[r] = __funnelshift_r(h, a[0], sh);
        }
    }
    if (!kAligned && 8 * band + kGDR - 2 >= H - 3) {
        // groups whose sixteen bytes would end past the image (in its last three
        // rows): byte loads, once for a row that is taken more than once
#pragma unroll 1
        for (int f = max(H - 3, 0); f < H; ++f) {
            const uint8_t *p = rgb + ((size_t)f * W + 4 * c) * 3;
            if (p - (reinterpret_cast<uintptr_t>(p) & 3) + 16 <= end) continue;
            uint32_t v[3] = {0, 0, 0}, h = 0;
#pragma unroll
            for (int j = 0; j < 12; ++j)
                if (j < 3 * nc) v[j >> 2] |= (uint32_t)__ldg(p + j) << (8 * (j & 3));
            if (c > 0) h = (uint32_t)__ldg(p - 3) << 8 | (uint32_t)__ldg(p - 2) << 16 | (uint32_t)__ldg(p - 1) << 24;
#pragma unroll
            for (int k = 0; k < kGDR; ++k)
                if (min(max(8 * band - 1 + k, 0), H - 1) == f) w[k][0] = v[0], w[k][1] = v[1], w[k][2] = v[2], wh[k] = h;
        }
    }
    // horizontal 3-sums of row r at full-res columns 4c and 4c + 2
    uint32_t hs[kGDR][2];
#pragma unroll
    for (int r = 0; r < kGDR; ++r) {
        // the word before this thread's first: pixel 4c - 1 in bytes 1..3
        const uint32_t prev = __shfl_up_sync(0xffffffffu, w[r][2], 1);
        const uint32_t hw = lane == 0 ? wh[r] : prev;
        const uint32_t g = luma4(w[r][0], w[r][1], w[r][2]);
        // pixel 4c - 1, or pixel 0 (clamped) for the first column group
        const uint32_t gh = c > 0 ? __dp4a(hw, kLumaW << 8, 128u) >> 8 : (g & 0xFFu);
        hs[r][0] = __dp4a(g, 0x00000101u, gh);
        hs[r][1] = __dp4a(g, 0x01010100u, 0u);
        const int fy = 8 * band - 1 + r;
        if (live && !right && r > 0 && fy < H) {
            uint8_t *o = gf + (size_t)fy * W + 4 * c;
            if (kAligned) {
                *reinterpret_cast<uint32_t *>(o) = g;
            } else if (W % 2 == 0) {                   // (the grey planes start on 256 bytes)
                *reinterpret_cast<uint16_t *>(o) = (uint16_t)g;
                if (nc == 4) *reinterpret_cast<uint16_t *>(o + 2) = (uint16_t)(g >> 16);
            } else {
                for (int i = 0; i < nc; ++i) o[i] = (uint8_t)(g >> (8 * i));
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int i = 0; i < kGDB; ++i) {
        const int y = kGDB * band + i;
        if (y >= Y) break;
        const uint32_t m0 = (hs[2 * i][0] + hs[2 * i + 1][0] + hs[2 * i + 2][0] + 4u) / 9u;
        const uint32_t m1 = (hs[2 * i][1] + hs[2 * i + 1][1] + hs[2 * i + 2][1] + 4u) / 9u;
        uint8_t *o = s + (size_t)y * X + 2 * c;
        if (kAligned || (X % 2 == 0 && 2 * c + 1 < X)) {
            // X even: output pixel 2c starts a 2-byte aligned pair
            *reinterpret_cast<uint16_t *>(o) = (uint16_t)(m0 | m1 << 8);
        } else {
            if (2 * c < X) o[0] = (uint8_t)m0;
            if (2 * c + 1 < X) o[1] = (uint8_t)m1;
        }
    }
}

// Support data: mini-census code and the four cross arms of every pixel.
//
// A CTA takes kSX x SY pixels of one image, with a warp per row. Each warp
// follows one direction (left, right, up, down) for one row quad, a
// lane holding four adjacent pixels as the bytes of one word. A step moves all
// four to the next pixel of the arm: the shifted word is a funnel shift of two
// staged words (left, right) or the word of the next row (up, down), |I - c|
// is one four-byte absolute difference and the test against tc a borrow-free
// byte compare, so a step costs six instructions for four pixels whatever the
// arms' lengths. The four rows of a quad go through a step together, which
// hides the latency of each, and a warp stops when none of its 512 arms goes
// on (tested every four steps) or can: the staged pixels beyond the image repeat its
// border, so an arm that reaches it would never end there by itself. Bound by the ALU pipe. At 718 x 496 (two
// images) 34.5 us with one thread following each arm eight pixels at a time
// and a queue for the arms that go on, 16.5 us now (cold L2, both).
constexpr int kSX = 128;                     // columns of a CTA
constexpr uint32_t kHi = 0x80808080u;

// Words staged beyond each side of a row: a scan of wx steps reads that far,
// the census reads two pixels.
__host__ __device__ constexpr int sup_hw(int wx) { return wx > 4 ? (wx + 3) / 4 : 1; }
__host__ __device__ constexpr int sup_row_words(int wx) { return kSX / 4 + 2 * sup_hw(wx); }
// Shared memory: staged rows [SY + 2][row words], staged columns [SY + 2 wy]
// [kSX / 4], results [5][SY][kSX / 4] (four arms, census), all in words.
template <int SY>
__host__ __device__ constexpr int sup_smem(int wx, int wy)
{
    return 4 * ((SY + 2) * sup_row_words(wx) + (SY + 2 * wy) * (kSX / 4) + 5 * SY * (kSX / 4));
}
static_assert(sup_smem<16>(kMaxWx, kMaxWy) <= 48 * 1024, "fits the default shared memory of a CTA");

// Four pixels x .. x + 3 of row `row` (columns clamped to the image; x is a
// multiple of 4). The pixels come from the aligned words that hold them: a word
// that starts in the image ends inside its allocation (planes start on 256-byte
// boundaries of a larger one, or their size is a whole number of words). No
// branch, so that several loads are in flight: a quad over the right edge is
// the last whole one, its bytes moved down and its last byte repeated.
template <bool kNarrow>
__device__ __forceinline__ uint32_t load_quad(const uint8_t *row, int x, int X)
{
    if (kNarrow) {                                         // fewer than four columns
        uint32_t v = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) v |= (uint32_t)__ldg(row + min(max(x + i, 0), X - 1)) << (8 * i);
        return v;
    }
    const int xc = min(max(x, 0), X - 4);
    const uintptr_t a = reinterpret_cast<uintptr_t>(row + xc);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~(uintptr_t)3);
    const uint32_t sh = (uint32_t)(a & 3) * 8;
    const uint32_t q = __funnelshift_r(__ldg(w), __ldg(w + (sh != 0)), sh);
    return __byte_perm(q, 0u, x < 0 ? 0u : 0x33333210u >> (4 * min(x - xc, 4)));
}

// Stages the rows of the horizontal scans and the columns of the vertical ones,
// the loads of one pass (a 21 x 31 window takes one) before its first store.
template <bool kNarrow, int SY>
__device__ __forceinline__ void stage(const SupImage &I, uint32_t *rows, uint32_t *cols, int x0, int y0, int hw, int wy)
{
    constexpr int P = kSX / 4, NT = 32 * SY;
    constexpr int B = (SY + 2 * kMaxWy + SY - 1) / SY;        // column words of a thread, all at once
    const int X = I.X, Y = I.Y, RW = P + 2 * hw, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i0 = threadIdx.x; i0 < (SY + 2) * RW; i0 += 2 * NT) {
        uint32_t v[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = min(i0 + k * NT, (SY + 2) * RW - 1), r = i / RW;
            v[k] = load_quad<kNarrow>(I.g + (size_t)min(max(y0 - 1 + r, 0), Y - 1) * X, x0 + 4 * (i - r * RW - hw), X);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (i0 + k * NT < (SY + 2) * RW) rows[i0 + k * NT] = v[k];
    }
    if (!I.arm) return;
    for (int r = warp; r < SY + 2 * wy; r += B * SY) {
        uint32_t v[B];
#pragma unroll
        for (int k = 0; k < B; ++k)
            v[k] = load_quad<kNarrow>(I.g + (size_t)min(max(y0 - wy + r + k * SY, 0), Y - 1) * X, x0 + 4 * lane, X);
#pragma unroll
        for (int k = 0; k < B; ++k)
            if (r + k * SY < SY + 2 * wy) cols[(r + k * SY) * P + lane] = v[k];
    }
}

// Byte compare of a scan step: bit 7 of each byte of the result is set when
// |w - c| >= tc. `bm` holds tc (tc < 128) or tc - 128 in every byte; |0x80
// keeps the subtraction inside its byte. The other bits are garbage.
template <bool kBig>
__device__ __forceinline__ uint32_t differs(uint32_t w, uint32_t c, uint32_t bm)
{
    const uint32_t ad = __vabsdiffu4(w, c);
    const uint32_t t = (ad | kHi) - bm;
    return kBig ? (ad & t) : (ad | t);
}

template <bool kBig>
__device__ __forceinline__ void arm_step(uint32_t w, uint32_t c, uint32_t bm, uint32_t &dead, uint32_t &n)
{
    dead |= differs<kBig>(w, c, bm);
    n += (~dead & kHi) >> 7;
}

// Horizontal arms of a lane's four pixels in four rows: `row` is the lane's
// word of the first row, `pitch` the row pitch; kDir -1 left, +1 right. No pixel of
// the lane has more than `room` pixels of the image in that direction.
template <bool kBig, int kDir>
__device__ __forceinline__ void scan_x(const uint32_t *row, int pitch, int cap, int room, uint32_t bm, uint32_t (&n)[4])
{
    uint32_t c[4], cur[4], dead[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c[j] = cur[j] = row[j * pitch];
        dead[j] = n[j] = 0;
    }
    for (int t = 0; t < cap; t += 4) {
        row += kDir;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t nx = row[j * pitch];
#pragma unroll
            for (int s = 1; s <= 4; ++s) {
                const uint32_t w = s == 4      ? nx
                                   : kDir < 0 ? __funnelshift_l(nx, cur[j], 8 * s)
                                              : __funnelshift_r(cur[j], nx, 8 * s);
                if (t + s <= cap) arm_step<kBig>(w, c[j], bm, dead[j], n[j]);
            }
            cur[j] = nx;
        }
        if (__all_sync(0xffffffffu, (dead[0] & dead[1] & dead[2] & dead[3] & kHi) == kHi || t + 4 >= room)) break;
    }
}

// Vertical arms: `col` is the lane's word of the first row in the staged
// columns; kDir -1 up, +1 down. The four rows slide over the column, one new
// word per step.
template <bool kBig, int kDir>
__device__ __forceinline__ void scan_y(const uint32_t *col, int cap, uint32_t bm, uint32_t (&n)[4])
{
    constexpr int P = kSX / 4;
    uint32_t c[4], w[4], dead[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c[j] = w[j] = col[j * P];                 // at step t row j sees the word of row j + kDir t
        dead[j] = n[j] = 0;
    }
    const uint32_t *edge = col + (kDir < 0 ? 0 : 3 * P);
    for (int t = 0; t < cap; t += 4) {
#pragma unroll
        for (int s = 1; s <= 4; ++s) {
            if (t + s <= cap) {
                edge += kDir * P;
                // the slot of the row that left the window takes the new word
                w[kDir < 0 ? (8 - s) & 3 : (s - 1) & 3] = *edge;
#pragma unroll
                for (int j = 0; j < 4; ++j) arm_step<kBig>(w[(j + kDir * s + 8) & 3], c[j], bm, dead[j], n[j]);
            }
        }
        if (__all_sync(0xffffffffu, (dead[0] & dead[1] & dead[2] & dead[3] & kHi) == kHi)) break;
    }
}

template <int N>
struct SupArgs {
    int n, wx, wy, tc;
    uint32_t *err;
    int start[N + 1];                        // first CTA of each image
    SupImage im[N];
};

template <int N, bool kBig, int SY, int kPerSM>
__global__ void __launch_bounds__(32 * SY, kPerSM) support_kernel(const __grid_constant__ SupArgs<N> A)
{
    extern __shared__ __align__(16) uint32_t sup[];
    pdl_trigger();
    int im = 0;
    while (im + 1 < A.n && (int)blockIdx.x >= A.start[im + 1]) ++im;
    const SupImage I = A.im[im];
    const int X = I.X, Y = I.Y, wx = A.wx, wy = A.wy;
    const int tile = blockIdx.x - A.start[im], tyi = tile / I.nx;
    const int x0 = (tile - tyi * I.nx) * kSX, y0 = tyi * SY;
    const int hw = sup_hw(wx), RW = kSX / 4 + 2 * hw;
    constexpr int P = kSX / 4;
    uint32_t *rows = sup;                                  // [SY + 2][RW], from row y0 - 1, word -hw
    uint32_t *cols = rows + (SY + 2) * RW;                 // [SY + 2 wy][P], from row y0 - wy
    uint32_t *res = cols + (SY + 2 * wy) * P;              // [5][SY][P]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();                                            // the grey image of the previous kernel
    if ((blockIdx.x | threadIdx.x) == 0) *A.err = 0u;

    if (X >= 4)
        stage<false, SY>(I, rows, cols, x0, y0, hw, wy);
    else
        stage<true, SY>(I, rows, cols, x0, y0, hw, wy);
    __syncthreads();

    if (I.arm) {
        const int dir = warp / (SY / 4), q = warp % (SY / 4);
        const uint32_t bm = (uint32_t)(A.tc - (kBig ? 128 : 0)) * 0x01010101u;
        uint32_t n[4];
        const uint32_t *rw = rows + (1 + 4 * q) * RW + hw + lane, *cl = cols + (wy + 4 * q) * P + lane;
        if (dir == 0)
            scan_x<kBig, -1>(rw, RW, wx, x0 + 4 * lane < X ? x0 + 4 * lane + 3 : 0, bm, n);
        else if (dir == 1)
            scan_x<kBig, 1>(rw, RW, wx, X - 1 - (x0 + 4 * lane), bm, n);
        else if (dir == 2)
            scan_y<kBig, -1>(cl, min(wy, y0 + 4 * q + 3), bm, n);
        else
            scan_y<kBig, 1>(cl, min(wy, Y - 1 - (y0 + 4 * q)), bm, n);
#pragma unroll
        for (int j = 0; j < 4; ++j) res[(dir * SY + 4 * q + j) * P + lane] = n[j];
    }
    {
        // census of row `warp` (Fig. 3 is missing: six neighbours in rows y-1..y+1,
        // mirror-symmetric in x; bit k set when neighbour k is strictly darker)
        const uint32_t *r0 = rows + warp * RW + hw + lane, *r1 = r0 + RW, *r2 = r1 + RW;
        const uint32_t c = r1[0], cl = c & ~kHi;
        const uint32_t nb[6] = {__funnelshift_l(r0[-1], r0[0], 8), __funnelshift_r(r0[0], r0[1], 8),
                                __funnelshift_l(r1[-1], c, 16),    __funnelshift_r(c, r1[1], 16),
                                __funnelshift_l(r2[-1], r2[0], 8), __funnelshift_r(r2[0], r2[1], 8)};
        uint32_t code = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const uint32_t t = (nb[k] | kHi) - cl;         // bit 7: the low seven bits are not darker
            code |= (((~nb[k] & c) | (~(nb[k] ^ c) & ~t)) & kHi) >> (7 - k);
        }
        res[(4 * SY + warp) * P + lane] = code;
    }
    __syncthreads();

    // outputs: a thread takes one column of a row quad, so every store is coalesced
    const int ox = threadIdx.x % kSX, q = threadIdx.x / kSX, x = x0 + ox;
    if (x >= X) return;
    const uint8_t *rb = reinterpret_cast<const uint8_t *>(res) + 4 * q * kSX + ox;
    const uint8_t *gb = reinterpret_cast<const uint8_t *>(rows + (1 + 4 * q) * RW + hw) + ox;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int y = y0 + 4 * q + j;
        if (y >= Y) break;
        const size_t i = (size_t)y * X + x;
        I.pix[i] = (uint32_t)gb[4 * j * RW] | (uint32_t)rb[(4 * SY + j) * kSX] << 8;
        if (I.key) I.key[i] = 0xFFFFFFFFu;         // WTA key preset: the fused kernel takes atomic minima
        if (!I.arm) continue;
        // the scans run over clamped pixels: arms end at the image border
        const int l = min((int)rb[j * kSX], x), r = min((int)rb[(SY + j) * kSX], X - 1 - x);
        const int u = min((int)rb[(2 * SY + j) * kSX], y), d = min((int)rb[(3 * SY + j) * kSX], Y - 1 - y);
        I.arm[i] = pack_arm(l, r, u, d);
        if (!I.armc) continue;
        uint16_t *ac = reinterpret_cast<uint16_t *>(I.armc);
        ac[2 * armc_index(y, x, X)] = (uint16_t)(l | r << 8);
        // the fused kernel takes output row y in row y + wy; it reads the rows
        // before and after those too, and does nothing with them
        ac[2 * armc_index(y + wy, x, X) + 1] = (uint16_t)armc_slots(y, u, d);
        if (y < wy) ac[2 * armc_index(y, x, X) + 1] = 0;
        if (y == Y - 1) {
            for (int i = Y; i < wy; ++i) ac[2 * armc_index(i, x, X) + 1] = 0;
            for (int i = Y + wy; i & 3; ++i) ac[2 * armc_index(i, x, X) + 1] = 0;
        }
    }
}

__global__ void unpack_kernel(const uint32_t *__restrict__ pix, const uint32_t *__restrict__ arm,
                              uint8_t *grey, uint8_t *census, uint32_t *arms, long n)
{
    long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t p = pix[i];
    if (grey) grey[i] = (uint8_t)(p & 0xFF);
    if (census) census[i] = (uint8_t)((p >> 8) & 0x3F);
    if (arms) arms[i] = arm[i];
}

}  // namespace

cudaError_t launch_grey(const uint8_t *rgb_l, const uint8_t *rgb_r, uint8_t *g_l, uint8_t *g_r,
                        int W, int H, cudaStream_t s)
{
    long n = (long)W * H;
    long quads = (n + 3) / 4;
    dim3 grid((unsigned)((quads + 255) / 256), 2);
    bool aligned = ((reinterpret_cast<uintptr_t>(rgb_l) | reinterpret_cast<uintptr_t>(rgb_r)) & 3) == 0;
    if (aligned)
        grey_kernel<true><<<grid, 256, 0, s>>>(rgb_l, rgb_r, g_l, g_r, n);
    else
        grey_kernel<false><<<grid, 256, 0, s>>>(rgb_l, rgb_r, g_l, g_r, n);
    return cudaGetLastError();
}

namespace {

template <bool kAligned, int N>
cudaError_t grey_down_run(const GreyJob *jobs, int n, cudaStream_t s)
{
    GreyArgs<N> A;
    A.n = 2 * n;
    A.start[0] = 0;
    for (int i = 0; i < n; ++i) {
        A.job[i] = jobs[i];
        const int W = jobs[i].W, H = jobs[i].H;
        const int blocks = ((W + 3) / 4 * (((H + 1) / 2 + kGDB - 1) / kGDB) + kGDT - 1) / kGDT;
        A.start[2 * i + 1] = A.start[2 * i] + blocks;
        A.start[2 * i + 2] = A.start[2 * i + 1] + blocks;
    }
    return launch_dependent(grey_down_kernel<kAligned, N>, dim3(A.start[2 * n]), dim3(kGDT), 0, s, A);
}

}  // namespace

cudaError_t launch_grey_down(const GreyJob *jobs, int n, cudaStream_t s, int *launches)
{
    if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
    GreyJob kind[2][kMaxBatch];
    int m[2] = {0, 0};
    for (int i = 0; i < n; ++i) {
        const GreyJob &j = jobs[i];
        if (j.W < 2 || j.H < 2) return cudaErrorInvalidValue;
        const uintptr_t a = reinterpret_cast<uintptr_t>(j.rgb_l) | reinterpret_cast<uintptr_t>(j.rgb_r);
        const int k = j.W % 4 == 0 && (a & 3) == 0;
        kind[k][m[k]++] = j;
    }
    cudaError_t e = cudaSuccess;
    if (m[1]) {
        ++*launches;
        e = m[1] == 1 ? grey_down_run<true, 2>(kind[1], 1, s) : grey_down_run<true, 2 * kMaxBatch>(kind[1], m[1], s);
    }
    if (m[0] && e == cudaSuccess) {
        ++*launches;
        e = m[0] == 1 ? grey_down_run<false, 2>(kind[0], 1, s) : grey_down_run<false, 2 * kMaxBatch>(kind[0], m[0], s);
    }
    return e;
}

namespace {

template <int N>
cudaError_t support_run(const SupImage *im, int n, int wx, int wy, int tc, uint32_t *err, cudaStream_t s)
{
    SupArgs<N> A;
    const auto lay = [&](int sy) {                        // CTAs of sy rows
        A.start[0] = 0;
        for (int i = 0; i < n; ++i) A.start[i + 1] = A.start[i] + A.im[i].nx * ((im[i].Y + sy - 1) / sy);
        return A.start[n];
    };
    A.n = n;
    A.wx = wx;
    A.wy = wy;
    A.tc = tc;
    A.err = err;
    for (int i = 0; i < n; ++i) {
        A.im[i] = im[i];
        A.im[i].nx = (im[i].X + kSX - 1) / kSX;
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const auto go = [&](auto rows, auto kernel, auto big) {
        constexpr int SY = decltype(rows)::value;
        return launch_dependent(tc < 128 ? kernel : big, dim3(A.start[n]), dim3(32 * SY), sup_smem<SY>(wx, wy), s, A);
    };
    using std::integral_constant;
    // Frames whose CTAs of eight rows all get an SM of their own: an SM then issues
    // half the scan steps (W_x 21, flat blocks: 64 x 48 6.3 -> 5.1 us, 381 x 195 9.6 ->
    // 6.9; W_x 141: 114 x 44 17.0 -> 14.6 us). The halo of two such CTAs costs more than that
    // where an SM has several (718 x 496: 21.5 against 16.9 us).
    if (lay(8) <= sms)
        return go(integral_constant<int, 8>{}, support_kernel<N, false, 8, 2>, support_kernel<N, true, 8, 2>);
    // Images whose CTAs all run at once with two on an SM take the form with 64
    // registers, which has more scan steps' loads in flight; more CTAs take
    // three on an SM (40 registers). Flat blocks, W_x 21, 64 against 40 registers, launches in a
    // row: 512 x 384 (192 CTAs) 12.0 and 14.4 us, 640 x 400 (250) 11.7 and 16.1; past two on an SM
    // 718 x 496 (372) 16.7 and 16.6, 960 x 540 (544) 21.0 and 20.6, 1920 x 1080 (2040) 67.5 and 65.2.
    if (lay(16) <= 2 * sms)
        return go(integral_constant<int, 16>{}, support_kernel<N, false, 16, 2>, support_kernel<N, true, 16, 2>);
    return go(integral_constant<int, 16>{}, support_kernel<N, false, 16, 3>, support_kernel<N, true, 16, 3>);
}

}  // namespace

cudaError_t launch_support(const SupImage *im, int n, int wx, int wy, int tc, uint32_t *err, cudaStream_t s)
{
    if (n < 1 || n > kMaxSupImages || wx > kMaxWx || wy > kMaxWy) return cudaErrorInvalidValue;
    // the kernel's argument holds every image: two for a frame, more for a batch
    return n <= 2 ? support_run<2>(im, n, wx, wy, tc, err, s)
                  : support_run<kMaxSupImages>(im, n, wx, wy, tc, err, s);
}

cudaError_t launch_unpack_planes(const uint32_t *pix, const uint32_t *arm, uint8_t *grey,
                                 uint8_t *census, uint32_t *arms, int X, int Y, cudaStream_t s)
{
    long n = (long)X * Y;
    unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pix, arm, grey, census, arms, n);
    return cudaGetLastError();
}

}  // namespace stereo
