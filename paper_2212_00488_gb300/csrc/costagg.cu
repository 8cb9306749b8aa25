// Fused matching cost + cross-based aggregation + winner-take-all for both
// base images: Eqs. 3-9 of the paper (Sec. III-B, III-C) in one kernel.
//
// The paper (Steps 3 and 5 of Sec. IV) writes the x-aggregated volume CA_x to
// global memory and reads it back for the y pass. Here nothing of the volume
// leaves the SM: each CTA sweeps its tile top to bottom and keeps, per
// (column, disparity, base), a ring of 64 running vertical prefix sums in
// shared memory.
//
// Tile: one CTA owns a strip of XS columns for each base and a slab of DS
// disparities [d0, d0+DS).
//  * Left base columns:  x in [x0, x0+XS).
//  * Right base columns: x in [x0-d0+sft, x0-d0+sft+XS). Shearing the right
//    strip by d0 makes both bases read one row of left-base costs: by Eq. 6,
//    C^R(x, y, d) = C^L(x+d, y, d), and for d in the slab the right windows
//    land inside [x0+sft-wx, x0+sft+XS+DS-1+wx), next to the left windows. The
//    shift back by sft uses up the spare entries of the prefix rows, so that at
//    718 columns 96 of them give every slab 8 strips, 152 CTAs in all.
//  * Output rows: all of them in the tiles that fill whole waves of the GPU, a band
//    in the rest. The sweep starts wy rows above the band and ends wy below.
//
// What bounds it: the instructions of the few warps an SM has room for beside
// the ring (issue slots 55 % used, shared-memory pipe 83 %). 718 x 496 x 73:
// 68.6 us, from 80.8 us with 100 columns, 7 + 12 warps and halfword loads for
// the right base. The steps: packed prefixes in plain 32-bit adds with one
// 8-byte load per window end for both bases (one path for all warps), the ring
// slots of both window ends from the support pass, and 96 columns, which is six
// consumer warps with every lane in use, leave room for twelve row slots in two
// planes, and let the producers be spread over the schedulers by their work.
//
// Warp roles (the row buffers between them form a ring of RS slots; rows
// 4k..4k+3 share one full and one empty mbarrier):
//  * Producer warp p (NPW of them) fills rows y = p, p + NPW, ...: for each
//    disparity d = d0 + q of the slab, the exclusive row prefix
//      S_q[i] = sum_{j<i} C^L(x0 - wx + j, y, d)                  (Eq. 7)
//    with C^L = P when the pixel or its match x - d is outside the image.
//    Each lane sums KE consecutive costs (one table lookup each: the AD and
//    census terms of Eqs. 3-5 combined), a warp scan adds the lanes' totals.
//    Two disparities share a prefix word when every horizontal window sum is
//    below 2^16 (checked on the host), else each has its own (modulo 2^32).
//  * Consumer thread (base, column) holds the slab's DS = 4 disparities and
//    takes four rows per step:
//      CA_x = S_q[hi] - S_q[lo] over the pixel's own left/right arms  (Eq. 7)
//      V(y+1) = V(y) + CA_x  -> ring slot y mod 64
//      CA(yo) = V(yo + down + 1) - V(yo - up), yo = y - wy          (Eq. 8)
//      key = min over d of (CA << 8 | d)                             (Eq. 9)
//    The minimum over slabs is one atomicMin per pixel and base. The packed
//    key keeps the smallest d among equal costs, the tie rule of Step 5.
// Vertical sums are modular uint32 and kept multiplied by 256 (V << 8): a
// difference of two ring entries is then CA << 8 exactly, because every
// window sum is below 2^24 (checked on the host), and a key is one add of d.
// A column's arm words of four rows arrive in one 16-byte load (armc_index).
//
// Every wait on an mbarrier is bounded: after a.wait_limit polls the thread
// sets a.err and returns, so a broken hand-off ends the kernel with an error
// status instead of hanging the GPU.
#include "internal.cuh"

#include <type_traits>

namespace stereo {
namespace {

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
                 : "memory");
}

// One poll of the phase with the given parity. A thread whose phase is not
// complete is suspended until the phase completes or at most kSuspendNs have
// passed, so waiting warps leave the issue slots to the warps doing the work.
constexpr uint32_t kSuspendNs = 1000;

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of `bar` with the given parity to complete,
// warp-uniform: the warp goes on only if every lane saw the phase complete.
// After `limit` polls (each suspends at most kSuspendNs) the error word is set
// and false is returned to every lane.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, uint32_t limit, uint32_t *err)
{
    bool ok = false;
    for (uint32_t it = 0; !ok && it < limit; ++it) ok = mbar_try_wait(bar, parity);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && (threadIdx.x & 31) == 0) atomicOr(err, 1u);
    return ok;
}

// Combined cost table: entry (h, ad) = AD(ad) + MC(h) at h * kLutPitch + ad
// (16-bit entries; Hamming distances 0..6). A row pitch of 136 words moves
// the rows of successive h by 8 banks, so lanes with small ad and small h
// read distinct banks.
constexpr int kLutRows = 7;
constexpr int kLutPitch = 272;

// Warp ids of the producers. A warp runs on scheduler id mod 4 for good, and a
// consumer warp has about 1.6 times the instructions per row quad of one of
// eight producers, so the producers go one by one to the scheduler with the
// least work; ids in between stay idle. Byte w % 8 of word[w / 8]: the
// producer that warp w is, 255 for none (the consumers are warps 0 .. ncw - 1).
struct Roles {
    uint64_t word[4] = {~0ull, ~0ull, ~0ull, ~0ull};
    int warps = 0;
};
constexpr Roles producer_roles(int ncw, int npw)
{
    int load[4] = {}, next[4] = {};
    for (int w = 0; w < ncw; ++w) load[w % 4] += 13 * npw;
    for (int q = 0; q < 4; ++q)
        for (next[q] = q; next[q] < ncw; next[q] += 4) {
        }
    Roles r;
    for (int p = 0; p < npw; ++p) {
        int b = 0;
        for (int q = 1; q < 4; ++q)
            if (load[q] < load[b] || (load[q] == load[b] && next[q] < next[b])) b = q;
        r.word[next[b] / 8] ^= (uint64_t)(255 ^ p) << (8 * (next[b] % 8));
        if (next[b] >= r.warps) r.warps = next[b] + 1;
        load[b] += 64;
        next[b] += 4;
    }
    return r;
}
template <int XS_, int DS_, int KE_, int RS_, bool S16_, int DPT_, int NPW_, int WX_, int NS_,
          bool SPLIT_ = false>
struct Tile {
    static constexpr int XS = XS_;            // columns per base
    static constexpr int DS = DS_;            // disparities per CTA
    static constexpr int KE = KE_;            // prefix entries per producer lane (odd)
    static constexpr int RS = RS_;            // row slots between producers and consumers
    static constexpr bool S16 = S16_;         // pairs of disparities share a prefix word (window sums < 2^16)
    static constexpr int WX = WX_;            // largest wx the tile takes
    static constexpr bool SPLIT = SPLIT_;     // 16-bit form with a window's two sides below 2^16 each, not their sum
    static constexpr int NS = NS_;            // time of a row step in ns with every SM busy (estimate())
    static constexpr int DPT = DPT_;          // disparities per consumer thread
    static constexpr int G = DS / DPT;        // consumer threads per column (adjacent lanes)
    static constexpr int LPX = 32 / G;        // columns per consumer warp
    static constexpr int NCT = 2 * XS * G;    // consumer threads with a column
    static constexpr int NCTP = (NCT + 31) / 32 * 32;   // consumer threads, whole warps
    static constexpr int NPW = NPW_;          // producer warps; warp p fills rows y = p (mod NPW)
    static constexpr Roles ROLES = producer_roles(NCTP / 32, NPW);
    static constexpr int NT = 32 * ROLES.warps;
    static constexpr int NE = 32 * KE;        // S[0..NE]
    // S row pitch in entries: the G groups of a consumer warp read rows that
    // start LPX words apart modulo the 32 banks (with one group any pitch does)
    static constexpr int SWP = NE + (G == 1 ? 4 : LPX);
    static constexpr int NB = RS / 4;         // row quads share a full and an empty barrier
    static constexpr int B_BAR = 2 * NB * 8;
    static constexpr int B_RING = kRing * NCT * DPT * 4;
    // 16-bit form: a row slot holds two planes of SWP entries of two words, one
    // for each base (a word per pair of disparities). 32-bit form: one plane
    // per disparity, SWP words each. Same bytes.
    static constexpr int B_SX = RS * DS * SWP * 4;
    static constexpr int B_LUT = kLutRows * kLutPitch * 2;
    static constexpr int BYTES = B_BAR + B_RING + B_SX + B_LUT;
    static_assert(DS % DPT == 0 && 32 % G == 0, "the threads of a column sit in adjacent lanes of one warp");
    static_assert(DPT == 4, "ring entries are 16 bytes");
    static_assert(!S16 || (DS == 4 && G == 1), "an entry holds the slab's four disparities");
    static_assert(XS + DS - 1 + 2 * WX <= NE, "the prefix rows cover the strip and its halo");
    static_assert(KE % 2 == 1, "odd KE keeps the producer lanes' strided stores in distinct banks");
    static_assert(NT <= 1024, "");
    static_assert(RS == NPW, "producer warp p owns row slot p");
    static_assert(RS % 4 == 0, "slots are handed over in row quads");
    static_assert(BYTES <= 232448, "tile exceeds shared memory");
};

template <int N> struct VecOf;
template <> struct VecOf<4> { using type = uint4; };

template <int N>
__device__ __forceinline__ uint32_t &vget(typename VecOf<N>::type &v, int k);
template <>
__device__ __forceinline__ uint32_t &vget<4>(uint4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

__device__ __forceinline__ void mbar_inval(uint64_t *bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// How far the right strip of a slab is moved back towards the left strip: as
// far as the spare entries of the prefix rows cover the gap. It saves high
// slabs their last strip.
template <class T>
__host__ __device__ __forceinline__ int right_shift(const CostAggArgs &a, int d0)
{
    const int spare = T::NE - (T::XS + T::DS - 1 + 2 * a.wx);
    return d0 < spare ? d0 : spare;
}

// First disparity of slab s: the last slab ends at D, over the one before it
// where D is not a multiple of DS (equal keys, so the minimum is the same).
template <class T>
__host__ __device__ __forceinline__ int slab_d0(const CostAggArgs &a, int s)
{
    const int last = a.D > T::DS ? a.D - T::DS : 0;
    return s * T::DS < last ? s * T::DS : last;
}

// One tile (x-strip from x0, disparity slab from d0, output rows [ya, yb)) of one frame; ya is a multiple of 4.
// The sweep starts at a row quad at most wy rows above and ends wy rows below. `reuse`
// is set when this CTA already ran a tile: its barriers are invalidated before
// they are initialised again and the cost table is already in place.
template <class T>
__device__ __forceinline__ void costagg_tile(const CostAggArgs &a, const int x0, const int d0, const int ya,
                                             const int yb, unsigned char *smem, const bool reuse)
{
    using Vec = typename VecOf<T::DPT>::type;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);
    uint64_t *empty = full + T::NB;
    Vec *ring = reinterpret_cast<Vec *>(smem + T::B_BAR);                     // [64][NCT]
    uint32_t *sx = reinterpret_cast<uint32_t *>(smem + T::B_BAR + T::B_RING);   // [RS][DS][SWP] (32-bit)
    uint2 *sxp = reinterpret_cast<uint2 *>(sx);                                 // [RS][2 bases][SWP] (16-bit)
    uint16_t *lut = reinterpret_cast<uint16_t *>(smem + T::B_BAR + T::B_RING + T::B_SX);  // [7][kLutPitch]

    const int t = threadIdx.x, lane = t & 31;
    const int X = a.X, D = a.D, wx = a.wx, wy = a.wy;
    const int y0 = max(ya - wy, 0) & ~3;          // input rows [y0, Y)
    const int Y = min(a.Y, yb + wy);
    const uint32_t limit = a.wait_limit;
    const int sft = right_shift<T>(a, d0);        // right base columns start at x0 - d0 + sft

    // combined cost table: AD(|grey difference|) + MC(Hamming)
    if (!reuse)
        for (int i = t; i < kLutRows * kLutPitch; i += T::NT) {
            const int h = i / kLutPitch, ad = i - h * kLutPitch;
            lut[i] = ad < 256 ? (uint16_t)(a.lut_ad[ad] + a.lut_mc[h]) : (uint16_t)0;
        }
    if (t == 0) {
        for (int s = 0; s < T::NB; ++s) {
            if (reuse) {
                mbar_inval(&full[s]);
                mbar_inval(&empty[s]);
            }
            mbar_init(&full[s], 128);               // the four producing warps of a row quad
            mbar_init(&empty[s], T::NCTP);          // every consumer thread
        }
    }
    if (!reuse) pdl_wait();                       // the support words and keys of the previous kernel
    __syncthreads();

    if (t >= T::NCTP) {
        // ======================= producers: warp pw fills rows pw, pw + NPW, ... in slot pw
        constexpr uint64_t r0 = T::ROLES.word[0], r1 = T::ROLES.word[1], r2 = T::ROLES.word[2], r3 = T::ROLES.word[3];
        const int pw = (int)((t < 256 ? r0 : t < 512 ? r1 : t < 768 ? r2 : r3) >> (t >> 5 & 7) * 8) & 255;
        if (pw == 255) return;
        const uint32_t P = a.P;
        const int xb = x0 - wx + lane * T::KE;      // x of this lane's first entry
        // per-lane constants: clamped load offsets and, per (entry, disparity),
        // whether the pixel and its match lie in the image
        int offl[T::KE], offr[T::KE + T::DS - 1];
        using Mask = typename std::conditional<(T::KE * T::DS > 32), uint64_t, uint32_t>::type;
        Mask inimg = 0;
#pragma unroll
        for (int k = 0; k < T::KE; ++k) offl[k] = min(max(xb + k, 0), X - 1);
#pragma unroll
        for (int k = 0; k < T::KE + T::DS - 1; ++k) offr[k] = min(max(xb + k - d0 - (T::DS - 1), 0), X - 1);
#pragma unroll
        for (int k = 0; k < T::KE; ++k)
#pragma unroll
            for (int q = 0; q < T::DS; ++q)
                if (xb + k >= d0 + q && xb + k < X) inimg |= (Mask)1 << (k * T::DS + q);
        const bool all_in = __all_sync(0xffffffffu, inimg == (Mask)(~(Mask)0 >> (8 * sizeof(Mask) - T::KE * T::DS)));
        // pixels of one row: the lane's KE entries and their KE + DS - 1 matches
        uint32_t pv0[T::KE], qv0[T::KE + T::DS - 1];
        auto load = [&](int y, uint32_t (&pv)[T::KE], uint32_t (&qv)[T::KE + T::DS - 1]) {
            if (y >= Y) return;
            const uint32_t *pl = a.pix_l + (size_t)y * X;
            const uint32_t *pr = a.pix_r + (size_t)y * X;
            if (all_in) {
                // every entry and match lies in the image: one base per row,
                // the entries at fixed offsets from it
                const uint32_t *bl = pl + xb, *br = pr + (xb - d0 - (T::DS - 1));
#pragma unroll
                for (int k = 0; k < T::KE; ++k) pv[k] = __ldg(bl + k);
#pragma unroll
                for (int k = 0; k < T::KE + T::DS - 1; ++k) qv[k] = __ldg(br + k);
            } else {
#pragma unroll
                for (int k = 0; k < T::KE; ++k) pv[k] = __ldg(pl + offl[k]);
#pragma unroll
                for (int k = 0; k < T::KE + T::DS - 1; ++k) qv[k] = __ldg(pr + offr[k]);
            }
        };
        // The next row's pixels are loaded into the same registers as soon
        // as this row's costs are formed, and the wait for a free slot comes
        // after the scan, so load latency and hand-off overlap the work.
        load(y0 + pw, pv0, qv0);
        // matching cost of entry k at disparity d0 + q (its match is qv index
        // k + DS-1 - q): one table lookup for the AD and census terms, or P
        // outside the image (only warps that touch a border test it)
        auto cost = [&](auto border, int k, int q) -> uint32_t {
            constexpr bool kBorder = decltype(border)::value;
            const uint32_t pk = pv0[k], qk = qv0[k + T::DS - 1 - q];
            const uint32_t ad = __vabsdiffu4(pk, qk) & 0xFFu;     // |grey difference| from the low bytes
            uint32_t v = lut[__popc((pk ^ qk) & 0x3F00u) * kLutPitch + ad];
            if (kBorder) v = (inimg >> (k * T::DS + q)) & 1u ? v : P;
            return v;
        };
        uint32_t ph = 1;                            // parity of the empty phase to wait for
        const int s = pw;                           // this warp's row slot
        for (int y = y0 + pw; y < Y; y += T::NPW, ph ^= 1u) {
            if constexpr (T::S16) {
                // The costs of disparities 2j and 2j+1 travel as the halves of
                // one word, and so do their prefixes, in plain 32-bit adds: a
                // prefix word is S_2j + 2^16 S_2j+1 modulo 2^32, carries and
                // all, so a difference of two is the pair of window sums
                // whenever both lie below 2^16 (checked on the host).
                uint32_t c2[2][T::KE], run2[2] = {0u, 0u};
                auto form = [&](auto border) {
#pragma unroll
                    for (int k = 0; k < T::KE; ++k)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            c2[j][k] = __byte_perm(cost(border, k, 2 * j), cost(border, k, 2 * j + 1), 0x5410);
                            run2[j] += c2[j][k];
                        }
                };
                if (all_in)
                    form(std::false_type{});
                else
                    form(std::true_type{});
                load(y + T::NPW, pv0, qv0);
                uint32_t incl2[2] = {run2[0], run2[1]};
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t u = __shfl_up_sync(0xffffffffu, incl2[j], o);
                        if (lane >= o) incl2[j] += u;
                    }
                }
                // Right base: disparity d0 + k is needed at position x + k. The
                // pair's second disparity one position on is the same word plus
                // one cost of that disparity (r2), and entry i of the right
                // base's plane holds pair 0 two positions back beside pair 1.
                uint32_t n2[2] = {incl2[0] - run2[0], incl2[1] - run2[1]};   // prefix before the lane's first entry
                uint32_t r0[T::KE], r1[T::KE];
                uint2 e[T::KE];
#pragma unroll
                for (int k = 0; k < T::KE; ++k) {
                    r0[k] = n2[0] + (c2[0][k] & 0xFFFF0000u);
                    r1[k] = n2[1] + (c2[1][k] & 0xFFFF0000u);
                    n2[0] += c2[0][k];
                    n2[1] += c2[1][k];
                    e[k] = make_uint2(n2[0], n2[1]);
                }
                const uint32_t q2 = __shfl_up_sync(0xffffffffu, r0[T::KE - 2], 1);
                const uint32_t q1 = __shfl_up_sync(0xffffffffu, r0[T::KE - 1], 1);
                if (y >= y0 + T::RS && !mbar_wait_warp(&empty[s >> 2], ph, limit, a.err)) return;
                // lanes write entries KE apart (KE odd): no bank conflicts
                uint2 *row = sxp + s * (2 * T::SWP);
#pragma unroll
                for (int k = 0; k < T::KE; ++k) row[1 + lane * T::KE + k] = e[k];
                if (lane == 0) row[0] = make_uint2(0u, 0u);
                row += T::SWP;
#pragma unroll
                for (int k = 0; k < T::KE; ++k)
                    row[lane * T::KE + k] = make_uint2(k == 0 ? q2 : k == 1 ? q1 : r0[k >= 2 ? k - 2 : 0], r1[k]);
            } else {
                uint32_t c[T::DS][T::KE];
                uint32_t run[T::DS];
                auto form = [&](auto border) {
#pragma unroll
                    for (int q = 0; q < T::DS; ++q) run[q] = 0;
#pragma unroll
                    for (int k = 0; k < T::KE; ++k)
#pragma unroll
                        for (int q = 0; q < T::DS; ++q) {
                            run[q] += cost(border, k, q);
                            c[q][k] = run[q];
                        }
                };
                if (all_in)
                    form(std::false_type{});
                else
                    form(std::true_type{});
                load(y + T::NPW, pv0, qv0);
                uint32_t incl[T::DS];
#pragma unroll
                for (int q = 0; q < T::DS; ++q) incl[q] = run[q];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                    for (int q = 0; q < T::DS; ++q) {
                        const uint32_t u = __shfl_up_sync(0xffffffffu, incl[q], o);
                        if (lane >= o) incl[q] += u;
                    }
                }
                if (y >= y0 + T::RS && !mbar_wait_warp(&empty[s >> 2], ph, limit, a.err)) return;
#pragma unroll
                for (int q = 0; q < T::DS; ++q) {
                    const uint32_t excl = incl[q] - run[q];
                    uint32_t *row = sx + (s * T::DS + q) * T::SWP;
#pragma unroll
                    for (int k = 0; k < T::KE; ++k) row[1 + lane * T::KE + k] = excl + c[q][k];
                    if (lane == 0) row[0] = 0;
                }
            }
            mbar_arrive(&full[s >> 2]);
            if (y + 1 == Y)                               // the quad's rows that do not exist
                for (int k = y & 3; k < 3; ++k) mbar_arrive(&full[s >> 2]);
        }
        return;
    }

    // =========================== consumers: thread (base, column, DPT disparities)
    // thread t: group g = t mod G, column index t / G over both bases (a warp
    // may hold columns of both bases; the G threads of a column never straddle
    // warps since G divides 32)
    const int g = t & (T::G - 1);                 // disparity group of this thread
    const int ci = t / T::G;
    // threads past the last column only keep the hand-off going
    const bool active = T::NCT == T::NCTP || t < T::NCT;
    const int b = ci >= T::XS;
    const int x = active ? ci - b * T::XS : T::XS - 1;
    const int col = b ? x0 - d0 + sft + x : x0 + x;
    const bool valid = active && col >= 0 && col < X;
    const int colc = min(max(col, 0), X - 1);
    const int dg = d0 + g * T::DPT;               // first disparity of the group
    uint32_t *key = (b ? a.key_r : a.key_l) + colc;
    // combined arm words, four rows per 16-byte quad (armc_index): row r holds
    // the left/right arms of row r (low half) and the ring slots of the
    // vertical window of row r - wy (high half)
    const uint4 *armq = reinterpret_cast<const uint4 *>(b ? a.armc_r : a.armc_l) + colc;
    // ring entries of this thread (an idle thread reads the last column's
    // entries and never writes)
    Vec *myring = ring + (active ? t : T::NCT - 1);
    // prefix word of slot 0 at this pixel's own column (32-bit form: of the group's first disparity)
    const uint32_t *srow0 = sx + (g * T::DPT) * T::SWP + x + wx + (b ? g * T::DPT + sft : 0);
    // entry of slot 0 at this pixel's own column (16-bit form; the right base's plane is two entries on)
    const uint2 *prow0 = sxp + x + wx + (b ? T::SWP + 2 + sft : 0);
    const int rows = yb + wy;                     // row steps: inputs y0..Y-1, outputs lag by wy
    const int nquad = (rows + 3) >> 2;            // arm-word quads

    if (active) {
        Vec z;
#pragma unroll
        for (int k = 0; k < T::DPT; ++k) vget<T::DPT>(z, k) = 0;
        myring[((y0 - 1) & (kRing - 1)) * T::NCT] = z;   // V(y0) = 0 (V(r) sits in slot (r - 1) mod 64)
    }
    uint32_t V[T::DPT];
#pragma unroll
    for (int k = 0; k < T::DPT; ++k) V[k] = 0;

    // x-window sums of one input row for this thread's disparities, times 256
    // (modulo 2^32). 16-bit form: one 8-byte load per end of the window, and a
    // byte permutation takes a half and places it at bits 8..23.
    auto hsum = [&](int slot, uint32_t am, uint32_t (&cax)[T::DPT]) {
        const int hi = ((am >> 8) & 0xFF) + 1, lo = am & 0xFF;
        if constexpr (T::S16) {
            const uint2 *w = prow0 + slot * (2 * T::SWP);
            const uint2 h = w[hi], l = w[-lo];
            auto place = [&](uint32_t w0, uint32_t w1, int k) {
                return __byte_perm(k < 2 ? w0 : w1, 0u, k % 2 ? 0x4324 : 0x4104);
            };
            if constexpr (T::SPLIT) {
                // the window in two, at the pixel's own column
                const uint2 m = w[0];
                const uint32_t a0 = h.x - m.x, a1 = h.y - m.y, b0 = m.x - l.x, b1 = m.y - l.y;
#pragma unroll
                for (int k = 0; k < 4; ++k) cax[k] = place(a0, a1, k) + place(b0, b1, k);
            } else {
                const uint32_t w0 = h.x - l.x, w1 = h.y - l.y;
#pragma unroll
                for (int k = 0; k < 4; ++k) cax[k] = place(w0, w1, k);
            }
        } else {
            const uint32_t *r0 = srow0 + slot * (T::DS * T::SWP);
#pragma unroll
            for (int k = 0; k < T::DPT; ++k) {
                const uint32_t *rk = r0 + k * (T::SWP + (b ? 1 : 0));
                cax[k] = (rk[hi] - rk[-lo]) << 8;
            }
        }
    };
    // V(y + 1) into ring slot y mod 64; the four rows of a step (y a
    // multiple of 4) land in consecutive slots of one step base
    auto push = [&](Vec *step_base, int j, const uint32_t (&cax)[T::DPT]) {
        Vec w;
#pragma unroll
        for (int k = 0; k < T::DPT; ++k) {
            V[k] += cax[k];
            vget<T::DPT>(w, k) = V[k];
        }
        if (active) step_base[j * T::NCT] = w;
    };
    // Four rows per step, one wait per step. While all four rows are inputs
    // the step has no branch but the wait, so the loads and arithmetic of
    // the rows interleave; idle threads and rows without an output do the
    // same work and drop it. Arm words are fetched a step ahead. Slabs that
    // lie wholly below D run without the per-disparity range test.
    auto sweep = [&](auto part) {
        constexpr bool kPart = decltype(part)::value;
        // packed WTA key of output row yo over this thread's disparities
        auto vkey = [&](uint32_t am) -> uint32_t {
            // the support pass has the slots of both ends of the window (armc_slots)
            Vec vl = myring[((am >> 16) & 0xFF) * T::NCT];              // V(yo - up)
            Vec vh = myring[(am >> 24) * T::NCT];                       // V(yo + down + 1)
            uint32_t best = 0xFFFFFFFFu;
#pragma unroll
            for (int k = 0; k < T::DPT; ++k) {
                // (V(hi) - V(lo)) << 8 is CA << 8 exactly: the key (CA << 8 | d) is one add
                const uint32_t kk = vget<T::DPT>(vh, k) - vget<T::DPT>(vl, k) + (uint32_t)(dg + k);
                best = (!kPart || dg + k < D) ? min(best, kk) : best;
            }
            return best;
        };
        constexpr int R = 4;                      // rows per step: one arm-word quad
        uint4 am = __ldg(armq + (y0 >> 2) * X);
        auto atomics = [&](auto inputs, int y, uint32_t (&kk)[R]) {
            constexpr bool kInputs = decltype(inputs)::value;   // rows y .. y+3 all exist
            // the G threads of a column (adjacent lanes) combine their
            // disparity groups' minima; one atomic per column and row
            if constexpr (T::G > 1) {
#pragma unroll
                for (int j = 0; j < R; ++j)
#pragma unroll
                    for (int o = 1; o < T::G; o <<= 1) kk[j] = min(kk[j], __shfl_xor_sync(0xffffffffu, kk[j], o));
            }
            if (g == 0 && valid) {
#pragma unroll
                for (int j = 0; j < R; ++j)
                    if (y + j - wy >= ya && (kInputs || y + j < rows)) atomicMin(key + (y + j - wy) * X, kk[j]);
            }
        };
        int y = y0;
        int ys = 0;                               // slot of row y (rows y + j take ys + j)
        uint32_t ph = 0;                          // parity of the full phase of those slots
        auto next_slots = [&]() {
            ys += R;
            if (ys == T::RS) {
                ys = 0;
                ph ^= 1u;
            }
        };
        // steps whose four rows are all inputs: no branch but the wait
        for (; y + R - 1 < Y; y += R) {
            const uint4 an = __ldg(armq + min((y >> 2) + 1, nquad - 1) * X);
            uint32_t c[R][T::DPT], kk[R];
            Vec *const sb = myring + (y & (kRing - 1)) * T::NCT;
            if (!mbar_wait_warp(&full[ys >> 2], ph, limit, a.err)) return;
#pragma unroll
            for (int j = 0; j < R; ++j) hsum(ys + j, vget<4>(am, j), c[j]);
            mbar_arrive(&empty[ys >> 2]);
            if (y + R - 1 - wy < ya) {                    // no output yet: only the prefixes
#pragma unroll
                for (int j = 0; j < R; ++j) push(sb, j, c[j]);
                am = an;
                next_slots();
                continue;
            }
#pragma unroll
            // output row r - wy reads V down to slot r - 2wy, which shares
            // its ring slot with r + 2 when wy = 31, so each row's key is
            // taken before the next row is pushed
            for (int j = 0; j < R; ++j) {
                push(sb, j, c[j]);
                kk[j] = vkey(vget<4>(am, j));
            }
            atomics(std::true_type{}, y, kk);
            am = an;
            next_slots();
        }
        // the last input rows and the output rows that lag them
        for (; y < rows; y += R) {
            const uint4 an = __ldg(armq + min((y >> 2) + 1, nquad - 1) * X);
            uint32_t c[R][T::DPT], kk[R];
            Vec *const sb = myring + (y & (kRing - 1)) * T::NCT;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const int r = y + j;
                if (r < Y) {
                    if (j == 0 && !mbar_wait_warp(&full[ys >> 2], ph, limit, a.err))
                        return;
                    hsum(ys + j, vget<4>(am, j), c[j]);
                    if (j == R - 1 || r + 1 == Y) mbar_arrive(&empty[ys >> 2]);
                    push(sb, j, c[j]);
                }
                kk[j] = vkey(vget<4>(am, j));
            }
            atomics(std::false_type{}, y, kk);
            am = an;
            next_slots();
        }
    };
    if (d0 + T::DS <= D)
        sweep(std::false_type{});
    else
        sweep(std::true_type{});
}

// Tiles of a frame, slab by slab. A slab needs strips x0 = 0, XS, ... until both
// bases are covered: the left base reads columns [x0, x0 + XS), the right base
// [x0 - d0 + sft, x0 - d0 + sft + XS), so low slabs need fewer than high ones.
template <class T>
__host__ __device__ __forceinline__ int slab_strips(const CostAggArgs &a, int slab)
{
    const int d0 = slab_d0<T>(a, slab);
    return (a.X + d0 - right_shift<T>(a, d0) + T::XS - 1) / T::XS;
}

// CTA t of a frame: the first a.head tiles (strip, slab) of a.tiles are swept from
// the first row to the last, the others in row bands of a.band rows: all of them
// in the first band, then in the next. (The count comes with the arguments: with
// every CTA adding it up over the slabs, 3283 x 16 x 104, W_x 61, took 69.8 us for 65.6.)
template <class T>
__device__ __forceinline__ void run_tile(const CostAggArgs &a, int t, unsigned char *smem, bool reuse)
{
    int ya = 0, yb = a.Y;
    if (t >= a.head) {
        const int rest = a.tiles - a.head, band = (t - a.head) / rest;
        t -= band * rest;
        ya = band * a.band;
        yb = min(ya + a.band, a.Y);
    }
    int s = 0;
    for (int n = slab_strips<T>(a, 0); t >= n; n = slab_strips<T>(a, s)) {
        t -= n;
        ++s;
    }
    costagg_tile<T>(a, t * T::XS, slab_d0<T>(a, s), ya, yb, smem, reuse);
}

template <class T>
__global__ void __launch_bounds__(T::NT, 1) costagg_wta_kernel(const CostAggArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_trigger();
    run_tile<T>(a, blockIdx.x, smem, false);
}

// Persistent form for a batch of frames: one CTA per SM takes tiles (job,
// strip, slab) from a global counter until none is left. Jobs come largest
// first, so the long sweeps start early and the short ones fill the tail.
template <class T>
__global__ void __launch_bounds__(T::NT, 1) costagg_batch_kernel(const __grid_constant__ BatchArgs b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_tile;
    pdl_trigger();
    bool reuse = false;
    for (;;) {
        if (threadIdx.x == 0) {
            // stop taking tiles once a bounded wait has given up anywhere
            const bool failed = *(volatile uint32_t *)b.job[0].err != 0u;
            s_tile = failed ? b.total_tiles : (int)atomicAdd(b.counter, 1u);
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile >= b.total_tiles) return;
        int j = 0;
        while (j + 1 < b.njobs && tile >= b.tile_start[j + 1]) ++j;
        run_tile<T>(b.job[j], tile - b.tile_start[j], smem, reuse);
        reuse = true;
        __syncthreads();
    }
}

// Tile shapes (XS x DS, KE, RS, 16-bit prefixes, DPT, producer warps, largest
// wx, ns per row step). The times are what fits the frames of a sweep that keep
// every SM busy, relative to tile 0: at 718 x 496 x 73 alone tile 4 takes 93, in
// frames of several waves 106, where it was picked at a loss of up to 17 % (sweep of
// 83 frames: picks 1.2 % from the best tile on average before, 0.6 % now; 210 pairs
// of 320 to 3840 columns: 1 % less time on average, up to 12 % less and 4 % more).
// One CTA per SM; the ring of 64 prefix rows per (column, disparity, base)
// dominates shared memory. Every shape gives the same keys.
using T0 = Tile<96, 4, 5, 12, true, 4, 12, 26, 121>;  // window sums < 2^16; at 718 columns 8 strips for every slab
using T1 = Tile<96, 4, 7, 8, true, 4, 8, 58, 158>;    // window sums < 2^16
using T2 = Tile<104, 4, 5, 4, false, 4, 4, 26, 200>;  // 32-bit prefixes
using T3 = Tile<104, 4, 7, 4, false, 4, 4, 58, 236>;  // 32-bit prefixes
using T4 = Tile<64, 4, 5, 16, true, 4, 16, 46, 106>; // narrow frames, window sums < 2^16
using T5 = Tile<100, 4, 5, 8, true, 4, 8, 28, 141>;   // window sums < 2^16
// slabs of 8 disparities: two threads per column, 32-bit prefixes (the
// batch autotuner's deeper slab)
using T6 = Tile<48, 8, 5, 4, false, 4, 4, 52, 259>;
// wide horizontal windows (Table I: W_x up to 141 per side), wx <= 174,
// 32-bit prefixes; 64 columns leave room for 8 producer warps and row slots
using T7 = Tile<64, 4, 13, 8, false, 4, 8, 174, 205>;
// wx up to 66 (Table I's W_x = 61) with 32-bit prefixes: 7 prefix entries
// per producer lane leave room for 8 producer warps and row slots
using T8 = Tile<88, 4, 7, 8, false, 4, 8, 66, 170>;

// Tiles 3 and 8 where the sums of a window's two sides stay below 2^16 though
// their total need not (W_x 41 and 61 at cost scale 512): packed prefixes after
// all, with one more load per window. Faster than four 32-bit prefixes a row
// (1436 x 992, W_x 41: 134 -> 94 us, W_x 61: 160 -> 140 us).
using T3S = Tile<96, 4, 7, 8, true, 4, 8, 58, 160, true>;
using T8S = Tile<88, 4, 7, 12, true, 4, 12, 66, 148, true>;
bool split_fits(const CostAggArgs &a)
{
    return (uint64_t)std::max(a.wx + 1, T3S::KE) * a.P < 65536u;
}

template <class T> struct Tag { using type = T; };

// Calls f(Tag<T>) for the tile shape with the given id, in its split form where
// `split`; false for an unknown id.
template <class F>
bool with_tile(int id, bool split, F &&f)
{
    if (split && id == 3) { f(Tag<T3S>{}); return true; }
    if (split && id == 8) { f(Tag<T8S>{}); return true; }
    switch (id) {
    case 0: f(Tag<T0>{}); return true;
    case 1: f(Tag<T1>{}); return true;
    case 2: f(Tag<T2>{}); return true;
    case 3: f(Tag<T3>{}); return true;
    case 4: f(Tag<T4>{}); return true;
    case 5: f(Tag<T5>{}); return true;
    case 6: f(Tag<T6>{}); return true;
    case 7: f(Tag<T7>{}); return true;
    case 8: f(Tag<T8>{}); return true;
    default: return false;
    }
}
static_assert(kNumTiles == 9, "tile ids 0..8");

template <class T>
bool fits(const CostAggArgs &a)
{
    if (a.wx > T::WX) return false;
    // 16-bit prefixes need every horizontal window sum, and every producer
    // lane's sum of KE costs, below 2^16
    return !T::S16 || (uint64_t)max(T::SPLIT ? a.wx + 1 : 2 * a.wx + 1, T::KE) * a.P < 65536u;
}


template <class T>
cudaError_t setup_one()
{
    cudaError_t e = cudaSuccess;
    if ((e = cudaFuncSetAttribute(costagg_wta_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, T::BYTES)) !=
        cudaSuccess)
        return e;
    return cudaFuncSetAttribute(costagg_batch_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, T::BYTES);
}

// Tiles of a frame: the strips of all slabs (slab_strips). Neighbouring slabs
// mostly have the same number of strips, so they are counted in runs of equal ones.
template <class T>
int tiles_of(const CostAggArgs &a)
{
    const int last = (a.D - 1) / T::DS;                       // the last slab, on its own: it may overlap
    int n = slab_strips<T>(a, last);
    for (int s = 0; s < last;) {
        const int strips = slab_strips<T>(a, s);
        // the columns to cover grow by the disparities past right_shift's spare entries
        const int spare = T::NE - (T::XS + T::DS - 1 + 2 * a.wx);
        const int end = std::min(last, (strips * T::XS - a.X + spare) / T::DS + 1);   // first slab with more
        n += strips * (end - s);
        s = end;
    }
    return n;
}

// Row steps of one tile when a frame of Y rows is cut into bands of `band` rows
// (a multiple of 4): the band, the wy rows its windows reach above and below
// it, and about 40 rows' worth of start-up (table, first rows, launch).
int band_steps(const CostAggArgs &a, int band)
{
    return (band >= a.Y ? a.Y + a.wy : std::min(a.Y, band + a.wy) + a.wy) + 40;
}

int band_rows(const CostAggArgs &a, int nb) { return ((a.Y + nb - 1) / nb + 3) / 4 * 4; }

constexpr int kMaxBands = 8;

// The ways a frame's tiles can be cut into bands; they do not depend on the tile
// shape, so the pick works them out once.
struct Cuts {
    int n = 0;
    int rows[kMaxBands], bands[kMaxBands], steps[kMaxBands];
    int whole;                                                // row steps of a tile in one piece
    explicit Cuts(const CostAggArgs &a) : whole(band_steps(a, a.Y))
    {
        for (int nb = 1; nb <= kMaxBands; ++nb) {
            const int r = band_rows(a, nb);
            if (n && r == rows[n - 1]) continue;
            rows[n] = r;
            bands[n] = (a.Y + r - 1) / r;
            steps[n++] = band_steps(a, r);
        }
    }
};

template <class T>
cudaError_t launch_batch_one(BatchArgs &b, int nsm, cudaStream_t s)
{
    for (int j = 0; j < b.njobs; ++j) {
        if (!fits<T>(b.job[j])) return cudaErrorInvalidValue;
        b.job[j].tiles = tiles_of<T>(b.job[j]);
    }
    // bands where the frames' tiles leave SMs idle: few tiles go in rounds over
    // the SMs, many even out and leave about half a long tile at the end
    double best = 0;
    int nb = 1;
    for (int n = 1; n <= kMaxBands; ++n) {
        double sum = 0, last = 0;
        long tiles = 0;
        for (int j = 0; j < b.njobs; ++j) {
            const CostAggArgs &a = b.job[j];
            const int rows = band_rows(a, n), steps = band_steps(a, rows);
            const long nt = (long)a.tiles * ((a.Y + rows - 1) / rows);
            tiles += nt;
            sum += (double)nt * steps;
            last = std::max(last, (double)steps);
        }
        const double rounds = (double)((tiles + nsm - 1) / nsm);
        const double t = std::max(last, rounds < 4 ? rounds * sum / tiles : sum / nsm + 0.5 * last);
        if (n == 1 || t < best) {
            best = t;
            nb = n;
        }
    }
    b.total_tiles = 0;
    for (int j = 0; j < b.njobs; ++j) {
        CostAggArgs &a = b.job[j];
        a.band = band_rows(a, nb);
        a.head = 0;
        b.tile_start[j] = b.total_tiles;
        b.total_tiles += a.tiles * ((a.Y + a.band - 1) / a.band);
    }
    b.tile_start[b.njobs] = b.total_tiles;
    cudaError_t e = cudaMemsetAsync(b.counter, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const int grid = b.total_tiles < nsm ? b.total_tiles : nsm;
    costagg_batch_kernel<T><<<grid, T::NT, T::BYTES, s>>>(b);
    return cudaGetLastError();
}

// Time of a frame in ns with this tile in its best cut, waves of CTAs times their
// row steps times the tile's measured time per step; sets the tile count and the cut. A small
// frame's tiles leave SMs idle: all of them go in bands (360 x 248 x 36: 38.1 us
// in one band, 56 CTAs of 152 SMs, 17.8 us cut). A larger frame's last wave does:
// whole waves of tiles stay in one piece, without the wy rows a band sweeps above
// and below its own, and the rest go in bands (1436 x 992, W_x 61, 171 tiles:
// all in two bands 140 us, 152 whole and 19 in bands 106; 3840 x 2160, 4.4
// waves: 707 and 644 us).
template <class T>
int64_t estimate(CostAggArgs &a, const Cuts &cuts, int nsm)
{
    a.tiles = tiles_of<T>(a);
    const int waves = a.tiles / nsm;
    int64_t best = -1;
    for (int k = 0; k <= waves; k += std::max(waves, 1)) {    // none or all full waves whole
        const int rest = a.tiles - k * nsm;
        for (int i = 0; i < cuts.n; ++i) {
            const int rounds = (rest * cuts.bands[i] + nsm - 1) / nsm;
            const int64_t t = ((int64_t)k * cuts.whole + (int64_t)rounds * cuts.steps[i]) * T::NS;
            if (best < 0 || t < best) {
                best = t;
                a.head = k * nsm;
                a.band = cuts.rows[i];
            }
        }
    }
    return best;
}

template <class T>
cudaError_t launch_one(const CostAggArgs &a, cudaStream_t s)
{
    const int ctas = a.head + (a.tiles - a.head) * ((a.Y + a.band - 1) / a.band);
    return launch_dependent(costagg_wta_kernel<T>, dim3(ctas), dim3(T::NT), T::BYTES, s, a);
}

}  // namespace

cudaError_t costagg_setup()
{
    cudaError_t e = cudaSuccess;
    for (int id = 0; id < kNumTiles && e == cudaSuccess; ++id)
        for (bool split : {false, true})
            if (e == cudaSuccess) with_tile(id, split, [&](auto tag) { e = setup_one<typename decltype(tag)::type>(); });
    return e;
}

namespace {

// The tile of a frame (a.tile, or the one with the least time), with its cut set; -1: none fits.
int pick(CostAggArgs &a, int nsm)
{
    const Cuts cuts(a);
    const bool split = split_fits(a);
    int best = -1;
    int64_t bt = 0;
    CostAggArgs c = a;
    for (int id = std::max(a.tile, 0); id < (a.tile >= 0 ? a.tile + 1 : kNumTiles); ++id)
        with_tile(id, split, [&](auto tag) {
            using T = typename decltype(tag)::type;
            if (!fits<T>(c)) return;
            const int64_t t = estimate<T>(c, cuts, nsm);
            if (best < 0 || t < bt) {
                best = id;
                bt = t;
                a.tiles = c.tiles;
                a.head = c.head;
                a.band = c.band;
            }
        });
    return best;
}

}  // namespace

int costagg_pick(const CostAggArgs &a, int nsm)
{
    CostAggArgs c = a;
    c.tile = -1;
    return pick(c, nsm);
}

bool costagg_fits(const CostAggArgs &a, int tile)
{
    bool ok = false;
    with_tile(tile, split_fits(a), [&](auto tag) { ok = fits<typename decltype(tag)::type>(a); });
    return ok;
}

cudaError_t launch_costagg_batch(BatchArgs &b, int tile, int nsm, cudaStream_t s)
{
    if (b.njobs < 1 || b.njobs > kMaxBatch) return cudaErrorInvalidValue;
    cudaError_t e = cudaErrorInvalidValue;
    with_tile(tile, split_fits(b.job[0]),
              [&](auto tag) { e = launch_batch_one<typename decltype(tag)::type>(b, nsm, s); });
    return e;
}

cudaError_t launch_costagg(const CostAggArgs &a, cudaStream_t s)
{
    if (a.wy > kMaxWy || a.wy < 0 || a.wx < 0 || a.wx > kMaxWx) return cudaErrorInvalidValue;
    CostAggArgs c = a;
    const int tile = pick(c, a.num_sms);
    cudaError_t e = cudaErrorInvalidValue;
    with_tile(tile, split_fits(a), [&](auto tag) { e = launch_one<typename decltype(tag)::type>(c, s); });
    return e;
}

}  // namespace stereo
