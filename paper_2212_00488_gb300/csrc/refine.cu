// Post-processing kernel: GCP cross-check (Eq. 10, Step 6), 3x3 median of
// D^L, bilateral-estimation fill (Eq. 11, Step 7) and on the downscaling path the
// 2x scale-up (Step 8), for up to kMaxBatch frames in one launch.
#include "internal.cuh"

namespace stereo {
namespace {

constexpr int kRefNT = 512;
constexpr int kMaxRefineX = 4096;   // processed width limit
constexpr int kRefLoad = 2;         // columns per thread in one round of loads

__device__ __forceinline__ int med3(int a, int b, int c)
{
    return max(min(a, b), min(max(a, b), c));
}

// Median of nine values: the classic exchange network on three sorted rows.
__device__ __forceinline__ int median9(int v0, int v1, int v2, int v3, int v4, int v5, int v6, int v7, int v8)
{
    // sort each triple
    int a0 = min(min(v0, v1), v2), a2 = max(max(v0, v1), v2), a1 = v0 + v1 + v2 - a0 - a2;
    int b0 = min(min(v3, v4), v5), b2 = max(max(v3, v4), v5), b1 = v3 + v4 + v5 - b0 - b2;
    int c0 = min(min(v6, v7), v8), c2 = max(max(v6, v7), v8), c1 = v6 + v7 + v8 - c0 - c2;
    // the median is the median of (max of mins, median of medians, min of maxes)
    int lo = max(max(a0, b0), c0);
    int mi = med3(a1, b1, c1);
    int hi = min(min(a2, b2), c2);
    return med3(lo, mi, hi);
}

// Step 7 at a pixel x that is not a GCP, from the nearest GCPs li < x (hl:
// there is one) and ri > x (hr) of its row, the row's medians dm and
// brightness gr.
__device__ __forceinline__ float fill_value(int x, int li, int ri, bool hl, bool hr, const uint8_t *dm,
                                            const uint8_t *gr, int T, int fill_mode)
{
    if (hl && hr) {
        const int i = x - li, j = ri - x;
        const int a = dm[li], b = dm[ri];
        if (fill_mode == 1) return (float)(i < j ? a : b);      // the closer GCP (Fig. 5a)
        if (fill_mode == 2) return (float)min(a, b);            // the smaller disparity (Fig. 5b)
        // linear fill between the two GCPs (Step 7); exact numerator
        if (abs(a - b) <= T) return __fdiv_rn(__int2float_rn(a * j + b * i), __int2float_rn(i + j));
        const int ga = abs((int)gr[li] - (int)gr[x]);
        const int gb = abs((int)gr[ri] - (int)gr[x]);
        return (float)(ga < gb ? a : b);
    }
    if (hl) return (float)dm[li];
    if (hr) return (float)dm[ri];
    return 0.0f;
}

// Step 8 along x, full-resolution units: the odd column 2x + 1 between the
// low-res pixels x (value a, brightness ga) and x + 1 (b, gb) takes a + b
// when they differ by at most T, else twice the side whose low-res
// brightness is strictly closer to the full-res pixel's (gfull), else b.
__device__ __forceinline__ float odd_value(float a, float b, int ga, int gb, int gfull, int T)
{
    if (fabsf(__fsub_rn(a, b)) <= (float)T) return __fadd_rn(a, b);
    return __fmul_rn(2.0f, abs(ga - gfull) < abs(gb - gfull) ? a : b);
}

// The nearest set bit of a row mask strictly before x, -1 if none, and strictly
// after it, `none` if none. Matched pixels lie close together, so the word of x or
// its neighbour nearly always has one.
__device__ __forceinline__ int bit_before(const uint32_t *mask, int x)
{
    int w = x >> 5;
    uint32_t m = mask[w] & ((1u << (x & 31)) - 1u);
    while (m == 0u && w > 0) m = mask[--w];
    return m ? 32 * w + 31 - __clz(m) : -1;
}
__device__ __forceinline__ int bit_after(const uint32_t *mask, int nw, int x, int none)
{
    int w = x >> 5;
    uint32_t m = mask[w] & ~((2u << (x & 31)) - 1u);
    while (m == 0u && w + 1 < nw) m = mask[++w];
    return m ? 32 * w + __ffs(m) - 1 : none;
}

// kUp (the downscaling path): CTA k of a frame takes low-res rows by = 2k and
// by + 1 (those below Y) and full-res rows 2 by .. 2 by + 3. It cross-checks,
// takes the medians of and fills low-res rows r_j = min(rb + j, Y - 1), j = 0, 1, 2
// (rb = min(by, Y - 1)); row r_2 only gives the vertical mean of full-res row
// 2 by + 3 and is filled again by the next CTA. The filled rows stay in shared
// memory for Step 8:
//  * along x: even full-res columns 2x take 2 D(x), odd ones odd_value();
//  * along y: full-res row 2y takes low-res row y, row 2y + 1 the mean of
//    rows y and y + 1 (row y at the last row).
// Else: rows by and by + 1, which end at the fill.
//
// Every row the CTA reads is requested in one round of loads. The GCPs of a row
// are a bit mask (one ballot per 32 columns), so a pixel finds the nearest ones on
// either side from a word or two, without a scan over the row or a pass per
// direction. A CTA's chain of phases bounds it, so it has 512 threads (256: 14.2 us,
// 768: 9.0 but 11.6 instead of 10.2 at 960 x 540): 718 x 496 and the scale-up 11.1 us with
// scans and per-pixel indices, 9.3 us now; 1920 x 1080 42 and 31 us. The maps, medians and
// filled rows of rows by and by + 1 are written for the debug and map outputs.
template <int N>
struct RefineArgs {
    int n, T, fill_mode;
    int start[N + 1];                                  // first CTA of each frame
    RefineJob job[N];
};

template <bool kUp> constexpr int kRefRows = kUp ? 3 : 2;

template <bool kUp, int N>
__global__ void __launch_bounds__(kRefNT) refine_kernel(const __grid_constant__ RefineArgs<N> A)
{
    constexpr int NR = kRefRows<kUp>;
    extern __shared__ __align__(16) uint8_t sm[];
    pdl_trigger();
    int f = 0;
    while (f + 1 < A.n && (int)blockIdx.x >= A.start[f + 1]) ++f;
    const RefineJob &J = A.job[f];
    const int X = J.X, Y = J.Y, W = J.W, H = J.H, T = A.T, fill_mode = A.fill_mode;
    const int t = threadIdx.x, lane = t & 31;
    const int by = 2 * ((int)blockIdx.x - A.start[f]);
    const int rb = min(by, Y - 1), nw = (X + 31) / 32;
    uint32_t *gcp = reinterpret_cast<uint32_t *>(sm);                 // [NR][nw] GCP bits
    float *dp = reinterpret_cast<float *>(gcp + NR * nw);             // [NR][X] filled rows
    uint8_t *dl5 = reinterpret_cast<uint8_t *>(dp + NR * X);          // [NR + 2][X] D^L rows clamp(rb - 1 + i)
    uint8_t *dr3 = dl5 + (NR + 2) * X, *gr3 = dr3 + NR * X, *dm3 = gr3 + NR * X;
    uint8_t *gfo3 = dm3 + NR * X;                                     // [3][X] full-res grey at (2 r_j, 2x + 1)
    pdl_wait();                                        // the keys of the fused kernel

    for (int xb = 0; xb < X; xb += kRefLoad * kRefNT) {
        uint32_t v[NR + 2 + 3 * NR][kRefLoad];
#pragma unroll
        for (int c = 0; c < kRefLoad; ++c) {
            const int x = xb + t + c * kRefNT;
            if (x < X) {
#pragma unroll
                for (int i = 0; i < NR + 2; ++i)
                    v[i][c] = __ldg(J.key_l + (size_t)min(max(rb - 1 + i, 0), Y - 1) * X + x);
#pragma unroll
                for (int j = 0; j < NR; ++j) {
                    const int r = min(rb + j, Y - 1);
                    v[NR + 2 + j][c] = __ldg(J.key_r + (size_t)r * X + x);
                    v[2 * NR + 2 + j][c] = __ldg(J.gs + (size_t)r * X + x);
                    if (kUp) v[3 * NR + 2 + j][c] = __ldg(J.gf + (size_t)(2 * r) * W + 2 * x + 1);   // 2x + 1 < 2X <= W
                }
            }
        }
#pragma unroll
        for (int c = 0; c < kRefLoad; ++c) {
            const int x = xb + t + c * kRefNT;
            if (x < X) {
#pragma unroll
                for (int i = 0; i < NR + 2; ++i) dl5[i * X + x] = (uint8_t)(v[i][c] & 0xFF);
#pragma unroll
                for (int j = 0; j < NR; ++j) {
                    dr3[j * X + x] = (uint8_t)(v[NR + 2 + j][c] & 0xFF);
                    gr3[j * X + x] = (uint8_t)v[2 * NR + 2 + j][c];
                    if (kUp) gfo3[j * X + x] = (uint8_t)v[3 * NR + 2 + j][c];
                }
            }
        }
    }
    __syncthreads();

    // Eq. 10 and the 3x3 median of D^L
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int cj = min(rb + j, Y - 1) - rb + 1;   // row r_j of D^L is dl5 row cj; its neighbours cj -+ 1
        const uint8_t *du = dl5 + (cj - 1) * X, *dc = dl5 + cj * X, *dd = dl5 + (cj + 1) * X;
        const uint8_t *drc = dr3 + j * X;
        const bool emit = j < 2 && by + j < Y;
        const size_t ro = (size_t)(by + j) * X;
        for (int xb = 0; xb < X; xb += kRefNT) {      // whole warps, for the ballots
            const int x = xb + t;
            bool isg = false;
            if (x < X) {
                const int k = dc[x];
                isg = x - k >= 0 && drc[x - k] == k;
                const int xm = max(x - 1, 0), xp = min(x + 1, X - 1);
                const int m = median9(du[xm], du[x], du[xp], dc[xm], dc[x], dc[xp], dd[xm], dd[x], dd[xp]);
                dm3[j * X + x] = (uint8_t)m;
                if (emit) {
                    if (J.dl) J.dl[ro + x] = (uint8_t)k;
                    if (J.dr) J.dr[ro + x] = drc[x];
                    if (J.gcp) J.gcp[ro + x] = isg;
                    if (J.dm) J.dm[ro + x] = (uint8_t)m;
                }
            }
            const uint32_t bits = __ballot_sync(0xffffffffu, isg);
            if (lane == 0 && x < X) gcp[j * nw + (x >> 5)] = bits;
        }
    }
    __syncthreads();

    // Step 7: GCPs keep their median, the others are filled from the nearest ones
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const uint32_t *g = gcp + j * nw;
        const uint8_t *dm = dm3 + j * X, *gr = gr3 + j * X;
        const bool emit = j < 2 && by + j < Y;
        for (int x = t; x < X; x += kRefNT) {
            float v;
            if ((g[x >> 5] >> (x & 31)) & 1u) {
                v = (float)dm[x];
            } else {
                const int li = bit_before(g, x), ri = bit_after(g, nw, x, X);
                v = fill_value(x, li, ri, li >= 0, ri < X, dm, gr, T, fill_mode);
            }
            if (kUp) dp[j * X + x] = v;
            if (emit && J.dplus) J.dplus[(size_t)(by + j) * X + x] = v;
        }
    }
    if (!kUp) return;
    __syncthreads();

    // Step 8: low-res column bx makes full-res columns 2 bx, 2 bx + 1 of rows 2 by .. 2 by + 3
    const int nbx = (W + 1) / 2;
    for (int bx = t; bx < nbx; bx += kRefNT) {
        const int xo = 2 * bx;
        const bool odd = xo + 1 < W;
        const bool pair = odd && bx + 1 < X;          // odd column between two low-res pixels
        const int xc = min(bx, X - 1);
        float e[NR], o[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const float a = dp[k * X + xc];
            e[k] = __fmul_rn(2.0f, a);
            o[k] = pair ? odd_value(a, dp[k * X + bx + 1], gr3[k * X + bx], gr3[k * X + bx + 1], gfo3[k * X + bx], T)
                        : e[k];
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int yo = 2 * (by + k);
            if (yo >= H) break;
            const float e0 = e[k], o0 = o[k];
            float e1 = e0, o1 = o0;
            if (by + k + 1 < Y) {
                e1 = __fmul_rn(0.5f, __fadd_rn(e0, e[k + 1]));
                o1 = __fmul_rn(0.5f, __fadd_rn(o0, o[k + 1]));
            }
            float *r0 = J.out + (size_t)yo * W + xo;
            if (J.pairs) {                              // W even, out 8-byte aligned: aligned pairs
                *reinterpret_cast<float2 *>(r0) = make_float2(e0, o0);
                if (yo + 1 < H) *reinterpret_cast<float2 *>(r0 + W) = make_float2(e1, o1);
            } else {
                r0[0] = e0;
                if (odd) r0[1] = o0;
                if (yo + 1 < H) {
                    r0[W] = e1;
                    if (odd) r0[W + 1] = o1;
                }
            }
        }
    }
}

template <bool kUp>
size_t refine_smem(int X)
{
    constexpr int NR = kRefRows<kUp>;
    return (size_t)NR * ((X + 31) / 32) * 4 + (size_t)X * (NR * 4 + NR + 2 + 3 * NR + (kUp ? NR : 0));
}

template <bool kUp, int N>
cudaError_t refine_run(const RefineJob *jobs, int n, int T, int fill_mode, cudaStream_t s)
{
    RefineArgs<N> A;
    A.n = n;
    A.T = T;
    A.fill_mode = fill_mode;
    A.start[0] = 0;
    size_t smem = 0;
    for (int i = 0; i < n; ++i) {
        RefineJob &j = A.job[i] = jobs[i];
        if (j.X < 1 || j.Y < 1 || j.X > kMaxRefineX || (kUp && (2 * j.X > j.W || 2 * j.Y > j.H)))
            return cudaErrorInvalidValue;
        j.pairs = j.W % 2 == 0 && (reinterpret_cast<uintptr_t>(j.out) & 7) == 0;
        A.start[i + 1] = A.start[i] + (kUp ? ((j.H + 1) / 2 + 1) / 2 : (j.Y + 1) / 2);
        smem = std::max(smem, refine_smem<kUp>(j.X));
    }
    return launch_dependent(refine_kernel<kUp, N>, dim3(A.start[n]), dim3(kRefNT), smem, s, A);
}

}  // namespace

cudaError_t refine_setup()
{
    cudaError_t e = cudaSuccess;
    auto one = [&](auto kernel, size_t smem) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
    one(refine_kernel<true, 1>, refine_smem<true>(kMaxRefineX));
    one(refine_kernel<false, 1>, refine_smem<false>(kMaxRefineX));
    one(refine_kernel<true, kMaxBatch>, refine_smem<true>(kMaxRefineX));
    one(refine_kernel<false, kMaxBatch>, refine_smem<false>(kMaxRefineX));
    return e;
}

cudaError_t launch_refine(const RefineJob *jobs, int n, bool up, int T, int fill_mode, cudaStream_t s)
{
    if (n < 1 || n > kMaxBatch || fill_mode < 0 || fill_mode > 2) return cudaErrorInvalidValue;
    if (n == 1)
        return up ? refine_run<true, 1>(jobs, n, T, fill_mode, s) : refine_run<false, 1>(jobs, n, T, fill_mode, s);
    return up ? refine_run<true, kMaxBatch>(jobs, n, T, fill_mode, s)
              : refine_run<false, kMaxBatch>(jobs, n, T, fill_mode, s);
}

}  // namespace stereo
