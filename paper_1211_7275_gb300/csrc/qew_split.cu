// qew_split.cu -- the fused FP32-split kernel of the qEW relaxation: elastic force + pinning
// force + Euler update + cell renormalisation + disorder regeneration, K Euler steps per HBM
// round trip (temporal blocking), with the checkpoint partial sums fused after the last step.
//
// Method: Eq. 1 of arXiv:1211.7275 with eta = c = 1, discretised in x with periodic boundary
// conditions and integrated by explicit Euler (Sec. III.B); pinning force interpolated from
// random values at integer (i, n) (Sec. III.B and the cases of Sec. IV.C); observables of
// Eqs. 3-5 (Sec. II).
//
// State of a site: integer cell n and FP32 offset d in [0, 1) (u = n + d), held in registers,
// plus its disorder cache, held in shared memory.
//   random field           the nodes of the cell, (R(n) + f, R(n+1) + f): the drive f is folded in, so
//                          F_p + f is one subtraction and one FMA
//   linear-spline random   the forces F_p = G - G(+1) of two neighbouring cells, of which the site is in
//   bond (Case 3)          one, and the node beyond them in the direction of the drive (above for f >= 0).  79% of the moves at the threshold go back
//                          where the site came from (it chatters across a jump of its force): they flip
//                          one bit of a lane mask and draw nothing (0.05 instead of 0.17 draws per
//                          site-update; 736-site tiles late in a relaxation 4.7e11 -> 9.3e11 su/s)
//   cubic random bond      the coefficients A, B, C of F_p + f = A + d (B + d C) over the cell (from the
//                          spline nodes V(n-1 .. n+2)) and the nodes V(n), V(n+1), V(n+2) that a move up
//                          reuses
//
// Work decomposition: one warp owns one tile of 32 * S sites of a chain, S consecutive sites
// per lane.  A tile advanced K steps needs K extra sites on each side (the stencil's light
// cone): the window is [start - pad, start - pad + 32 S) with pad = K rounded up to 4, and the owned
// sites [start, start + w_own); the outermost sites of the window go stale one
// per step from each edge and are never stored.  Windows wrap around periodic chains (any
// number of times for chains shorter than a tile).  Halo exchange inside a step is three warp
// shuffles and there is no block-wide barrier.
//
// What bounds it, and the shape of a step.  The kernel is bound by instruction issue and by the
// latency of a step's serial parts at 12 to 16 warps per SM, not by memory.  So
//   - the update loop works on register pairs with packed FP32 instructions (half the issue slots; the
//     FP32 pipe itself is as busy as with scalar ones, 61% at 992-site tiles) and reads both sites'
//     cache values with one 16-byte load;
//   - renormalisation is branch-free (n += floor(d), d -= floor(d)), with the floor by two packed
//     additions: as a conversion it took the conversion pipe 7.6 clocks per site;
//   - a funnel shift per site collects what moved how far (MoveCodes), so that moves by one cell need
//     no copy of the cells for the consumers; a rare path takes moves by more;
//   - requests are queued by ballots, without a prefix sum, and the Philox values evaluated 32 lanes at
//     a time, straight into the shared-memory cache of the requesting sites;
//   - what is the same in all lanes is kept in uniform registers (see uniform()).
// 16 x 2^20 random-field chains at the threshold, 992-site tiles, K = 32: 0.94 -> 0.59 warp-instructions
// per site-update, 75% -> 67% issue, 560 -> 400 us per launch (1.03e12 -> 1.33e12 su/s).
#include <algorithm>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "qew_internal.h"
#include "qew_tma.cuh"

namespace qew {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// Chain-local index of window position x (window start wstart, |wstart| <= K).  A window wraps
// at most once around a chain at least as long as the window; shorter chains take the modulo.
// The wrap is taken in 64 bits: past the end of a chain of up to 2^31 - 1 sites, g itself may
// not fit in an int32.
__device__ __forceinline__ int32_t site_index(int64_t wstart, int x, bool contiguous, int32_t L)
{
    const int64_t g = wstart + x;
    if (contiguous)
        return static_cast<int32_t>(g);
    if (g >= -static_cast<int64_t>(L) && g < 2 * static_cast<int64_t>(L))
        return static_cast<int32_t>(g < 0 ? g + L : (g >= L ? g - L : g));
    return wrap_site(g, L);
}

// Bytes of disorder cache per site in HBM, beside the third node.
template <int KIND>
struct CacheBytes {
    static constexpr int hbm = pair_kind(KIND) ? 8 : quad_kind(KIND) ? 20 : 0;
};

// ---- two sites at a time ----
// A lane's S = 2H + 1 consecutive sites are two runs of H sites and one last site.  Site j of the
// first run and site j of the second (lane sites j and H + j) share a 64-bit register pair, and
// their elastic force, Euler update and cell move are packed FP32 operations (two sites per issue
// slot, each rounded as the scalar operation).  The right neighbours of pair j are pair j + 1, so
// no operand has to be re-paired inside a run.
using pair_t = unsigned long long;

__device__ __forceinline__ pair_t pk(float lo, float hi)
{
    pair_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo(pair_t p)
{
    return __uint_as_float(static_cast<unsigned>(p));
}
__device__ __forceinline__ float hi(pair_t p)
{
    return __uint_as_float(static_cast<unsigned>(p >> 32));
}
__device__ __forceinline__ pair_t add2(pair_t a, pair_t b)
{
    pair_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair_t sub2(pair_t a, pair_t b)
{
    pair_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// floor of both halves, |x| < 2^22: adding 1.5 * 2^23 rounded down leaves the floor in a float whose
// last place is 1.
__device__ __forceinline__ pair_t floor2(pair_t x)
{
    const pair_t big = pk(12582912.0f, 12582912.0f);
    pair_t r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(big));
    return sub2(r, big);
}
__device__ __forceinline__ pair_t fma2(pair_t a, pair_t b, pair_t c)
{
    pair_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// ---- shared memory of one warp tile ----
//   slot    4 B per site, linear: offsets and then cells arrive and leave through it; in between it
//           holds the cell that each site's cache belongs to
//   loop    what the update loop reads, a row of 32 float4 per pair (row t is pair H - 1 - t, row H
//           the last site): one conflict-free 16-byte load per pair and step.  (first, second) value
//           of both sites: RF (R(n) + f, R(n+1) + f); linear-spline random bond the force F_p of
//           two neighbouring cells; cubic kinds the coefficients (A, B), and C in rows of float2
//   nodes   what only a cell move reads, linear: the node beyond the two cells (linear-spline random
//           bond), V(n), V(n+1) and V(n+2) (cubic kinds)
//   queue   kQueue requests of 2 B
// RF takes 12 B per site and so 16 warps per SM at 992-site tiles, the register limit.
template <int KIND, int S>
struct Tile {
    static constexpr int H = S / 2;
    static constexpr int TW = 32 * S;
    static constexpr bool has_pair = pair_kind(KIND);
    static constexpr bool has_quad = quad_kind(KIND);
    static constexpr bool has_cache = has_pair || has_quad;
    // Cells wait in registers while the offsets come through the slot, instead of following them by a
    // second copy.  The cubic kinds' 480-site tiles have the registers for it: a launch of 16 steps is 1%
    // shorter on 512 x 2^16 sites, and 4% on a few tiles; the random field lost 2%, Case 3 0.5%.
    static constexpr bool early_cells = has_quad;
    static constexpr int slot = 0;
    static constexpr int loop = 4 * TW;
    static constexpr int loopc = loop + (has_cache ? 512 * (H + 1) : 0);
    static constexpr int top = loopc + (has_quad ? 256 * (H + 1) : 0);     // one float per site
    static constexpr int nodes = top + (has_quad || KIND == kRBGLinear ? 4 * TW : 0);   // one float2 per site
    static constexpr int queue = nodes + (has_quad ? 8 * TW : 0);
    static constexpr int kQueue = 256;
    // whether a single cell against the drive is an ordinary move (else it takes the rare path of far
    // moves): a fifth of the linear-spline random bond's moves, a few in 10^4 of the other kinds'
    static constexpr bool kDown = KIND == kRBGLinear || KIND == kRBGCubic;
    // KIND none stages offsets and cells side by side, having no cache to make room for, and so does the
    // random field up to 736-site tiles, where the room does not cost a warp: one wait instead of two at
    // each end of a launch.  A launch of one step on 2^20 sites, 736-site tiles: 27 -> 22 us.  (Case 3 so
    // only at 224-site tiles, 32768 sites 4.9 -> 4.6 ms per 5000 steps; wider ones lost 2% to 4%.)
    static constexpr bool side_by_side = !has_cache || (KIND == kRF && S <= 23) || (KIND == kRBGLinear && S <= 7);
    static constexpr int slot2 = !has_cache ? 4 * TW : side_by_side ? queue + 2 * kQueue : slot;
    static constexpr int bytes = !has_cache ? 8 * TW : queue + 2 * kQueue + (side_by_side ? 4 * TW : 0);
};

// Per-lane mask of the sites that moved in a step.  Bit t is pair H - 1 - t's second site, bit D + t
// its first site, bit D + H the last site; D (a multiple of 3) leaves room for H bits, and a mask of
// more than 32 sites takes 64 bits.
template <int S>
struct Moves {
    static constexpr int H = S / 2;
    static constexpr bool wide = S > 32;
    static constexpr int D = wide ? 32 : 3 * ((H + 2) / 3);
    using mask = typename std::conditional<wide, unsigned long long, unsigned>::type;
    static constexpr mask last = mask(1) << (D + H);
    static __host__ __device__ constexpr mask first(int p) { return mask(1) << (D + H - 1 - p); }
    static __host__ __device__ constexpr mask second(int p) { return mask(1) << (H - 1 - p); }
};

__device__ __forceinline__ int mask_popc(unsigned m) { return __popc(m); }
__device__ __forceinline__ int mask_popc(unsigned long long m) { return __popcll(m); }

// m without bit b; 0 stays 0 (b is -1 then: the shift clamps).
__device__ __forceinline__ unsigned mask_drop(unsigned m, int b)
{
    unsigned one;
    asm("shl.b32 %0, 1, %1;" : "=r"(one) : "r"(b));
    return m & ~one;
}
__device__ __forceinline__ unsigned long long mask_drop(unsigned long long m, int b)
{
    unsigned long long one;
    asm("shl.b64 %0, 1, %1;" : "=l"(one) : "r"(b));
    return m & ~one;
}

// Collects the move codes of a step.  The top three bits of floor(d) as a float say how far a site
// moved: 0b000 (or 0b100, -0) not at all, 0b001 one cell up, 0b101 one cell down, and a set middle
// bit two cells or more (or not a number).  One funnel shift per site appends them to a word; the
// codes of a run go round three words, so that code k of word w, shifted, lands on the run's bit.
template <int S>
struct MoveCodes {
    static constexpr int H = S / 2;
    static constexpr unsigned kOnes = 0x09249249u;
    unsigned a[3] = {0u, 0u, 0u};   // first run
    unsigned b[3] = {0u, 0u, 0u};   // second run
    unsigned last = 0u;

    __device__ __forceinline__ void put(int p, float first, float second)
    {
        a[p % 3] = __funnelshift_l(__float_as_uint(first), a[p % 3], 3);
        b[p % 3] = __funnelshift_l(__float_as_uint(second), b[p % 3], 3);
    }
    __device__ __forceinline__ void put_last(float fl) { last = __float_as_uint(fl); }

    // moved: sites that changed cell; down: of those, by one cell downwards (when nothing is far);
    // far: some site of the lane moved two cells or more, or, unless DOWN, moved against the drive
    // (downwards, with NEG upwards)
    template <bool DOWN, bool NEG>
    __device__ __forceinline__ void masks(typename Moves<S>::mask& moved, typename Moves<S>::mask& down, bool& far) const
    {
        using mask = typename Moves<S>::mask;
        constexpr unsigned kFar = (DOWN || NEG) ? kOnes << 1 : (kOnes << 1) | (kOnes << 2);
        auto against = [](unsigned c) -> unsigned { return (!DOWN && NEG) ? c & ~(c >> 2) & kOnes : 0u; };
        unsigned mv[2] = {0u, 0u}, dn[2] = {0u, 0u};
        unsigned any = last & ((DOWN || NEG) ? 0x40000000u : 0xC0000000u);
        if (!DOWN && NEG)
            any |= static_cast<unsigned>(static_cast<int>(last) > 0);
#pragma unroll
        for (int w = 0; w < 3; ++w) {
            const int n = (H - w + 2) / 3;       // codes in word w
            if (n <= 0)
                continue;
            const int sh = H - 1 - w - 3 * (n - 1);
            if constexpr (Moves<S>::wide) {
                const unsigned c[2] = {b[w], a[w]};
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    any |= (c[r] & kFar) | against(c[r]);
                    mv[r] |= ((c[r] | (c[r] >> 1)) & kOnes) << sh;
                    if (DOWN)
                        dn[r] |= ((c[r] >> 2) & kOnes) << sh;
                }
            } else {
                const unsigned c = (a[w] << Moves<S>::D) + b[w];
                any |= (c & kFar) | against(c);
                mv[0] += ((c | (c >> 1)) & kOnes) << sh;
                if (DOWN)
                    dn[0] += ((c >> 2) & kOnes) << sh;
            }
        }
        moved = mv[0];
        down = dn[0];
        if constexpr (Moves<S>::wide) {
            moved |= static_cast<mask>(mv[1]) << 32;
            down |= static_cast<mask>(dn[1]) << 32;
        }
        if (last & 0x7FFFFFFFu) {
            moved |= Moves<S>::last;
            if (DOWN && (last & 0x80000000u))
                down |= Moves<S>::last;
        }
        far = any != 0;
    }
    // The sites that moved two cells or more.
    __device__ __forceinline__ typename Moves<S>::mask far_ones() const
    {
        unsigned m[2] = {0u, 0u};
#pragma unroll
        for (int w = 0; w < 3; ++w) {
            const int n = (H - w + 2) / 3;
            if (n <= 0)
                continue;
            const int sh = H - 1 - w - 3 * (n - 1);
            if constexpr (Moves<S>::wide) {
                m[0] |= ((b[w] >> 1) & kOnes) << sh;
                m[1] |= ((a[w] >> 1) & kOnes) << sh;
            } else {
                m[0] += ((((a[w] << Moves<S>::D) + b[w]) >> 1) & kOnes) << sh;
            }
        }
        typename Moves<S>::mask r = m[0];
        if constexpr (Moves<S>::wide)
            r |= static_cast<typename Moves<S>::mask>(m[1]) << 32;
        return (last & 0x40000000u) ? r | Moves<S>::last : r;
    }
};

// F_p + f of a lane's pair (row t = H - 1 - p) and of its last site, at offsets d, from shared memory.
template <int KIND, int S>
struct Force {
    const float4* rows;     // loop rows, at this lane
    const float2* rows_c;
    pair_t f2;

    // upper: linear-spline random bond, whether the sites are in the upper of their two cells
    __device__ __forceinline__ pair_t pair(int p, pair_t d, typename Moves<S>::mask upper) const
    {
        const int t = S / 2 - 1 - p;
        if constexpr (KIND == kRF) {
            const float4 q = rows[32 * t];
            const pair_t q0 = pk(q.x, q.y), q1 = pk(q.z, q.w);
            return fma2(d, sub2(q1, q0), q0);
        } else if constexpr (KIND == kRBGLinear) {
            const float4 q = rows[32 * t];
            return add2(pk((upper & Moves<S>::first(p)) ? q.z : q.x, (upper & Moves<S>::second(p)) ? q.w : q.y), f2);
        } else if constexpr (quad_kind(KIND)) {
            const float4 q = rows[32 * t];
            const float2 c = rows_c[32 * t];
            return fma2(d, fma2(d, pk(c.x, c.y), pk(q.z, q.w)), pk(q.x, q.y));
        } else {
            return f2;
        }
    }
    __device__ __forceinline__ float last(float d, typename Moves<S>::mask upper) const
    {
        if constexpr (KIND == kRF) {
            const float4 q = rows[32 * (S / 2)];
            return fmaf(d, q.z - q.x, q.x);
        } else if constexpr (KIND == kRBGLinear) {
            const float4 q = rows[32 * (S / 2)];
            return ((upper & Moves<S>::last) ? q.z : q.x) + lo(f2);
        } else if constexpr (quad_kind(KIND)) {
            const float4 q = rows[32 * (S / 2)];
            return fmaf(d, fmaf(d, rows_c[32 * (S / 2)].x, q.z), q.x);
        } else {
            return lo(f2);
        }
    }
};

// Position of the highest set bit (m != 0).
__device__ __forceinline__ int mask_top(unsigned m) { return 31 - __clz(m); }
__device__ __forceinline__ int mask_top(unsigned long long m) { return 63 - __clzll(static_cast<long long>(m)); }

// Registers per thread allowed to the kernel, the fastest measured of 96 .. 184 on each shape.  Both
// ways cost: at 992-site random-field tiles 120 (and the same 16 warps per SM) instead of 128 lost 2%,
// 104 with a shorter queue and 18 warps also 2%, 160 (12 warps) 9%; Case 3 at 736-site tiles gains 4%
// from 144 over 112, at 480-site tiles 2% from 104 over 112.
template <int KIND, int S>
struct MaxRegs {
    static constexpr int value = quad_kind(KIND) ? (S <= 8 ? 80 : 128) :
                                 KIND == kRBGLinear ? (S <= 8 ? 64 : S <= 16 ? 104 : S <= 23 ? 144 : S <= 31 ? 168 : 184) :
                                                      (S <= 8 ? 64 : S <= 16 ? 112 : S <= 31 ? 128 : 160);
};

// The cell of window position x at this point of the K loop, in every lane.
template <int KIND, int S>
__device__ __forceinline__ int32_t cell_at(int32_t* s_cell, int x, int lane, int32_t N0, const pair_t (&c)[S / 2], float cT,
                                           typename Moves<S>::mask upper)
{
    constexpr int H = S / 2;
    if constexpr (KIND == kRBGLinear) {
        const int src = x / S, j = x - src * S;
        const int b = (j == 2 * H) ? Moves<S>::D + H : (j < H) ? Moves<S>::D + H - 1 - j : 2 * H - 1 - j;
        return s_cell[x] + static_cast<int32_t>(__shfl_sync(kFull, upper, src) >> b & 1u);
    }
    if constexpr (KIND == kNone) {   // nothing else keeps the slot up to date
#pragma unroll
        for (int p = 0; p < H; ++p) {
            s_cell[lane * S + p] = N0 + __float2int_rn(lo(c[p]));
            s_cell[lane * S + H + p] = N0 + __float2int_rn(hi(c[p]));
        }
        s_cell[lane * S + 2 * H] = N0 + __float2int_rn(cT);
        __syncwarp();
    }
    return s_cell[x];
}

// Partial sums of F_p, u - r and (u - r)^2 over the owned sites at this point of the K loop, r the
// reference cell `ref`: FP32 sums over runs of S sites, FP32 warp reduction, then one FP64 shift to
// the chain's reference in lane 0.  The runs start `len` sites before the tile, where `len` is the
// number of steps since the last observation, or since the last whole K steps after it: the sums
// then do not depend on how steps and observations are spread over launches.  Each lane adds up
// other sites than its own, so the values go through the slot.
template <int KIND, int S>
__device__ __forceinline__ void observe_tile(const SplitLaunch& a, float f, int tile, int chain, int obs, int32_t ref,
                                             int owned, int pad, int32_t N0, int lane, const pair_t (&c)[S / 2],
                                             const pair_t (&d)[S / 2], float cT, float dT, typename Moves<S>::mask upper,
                                             int32_t* s_cell, float* s_off, const float* s_loop, const float* s_loopc)
{
    using T = Tile<KIND, S>;
    using M = Moves<S>;
    constexpr int H = S / 2;
    const float dref = static_cast<float>(ref - N0);   // exact
    const int first = lane * S - a.obs_len[obs];       // this lane's run, from the first owned site
    float* slot = T::has_cache ? reinterpret_cast<float*>(s_cell) : s_off;
    float sF = 0.0f, sy = 0.0f, syy = 0.0f;
    int cnt = 0;
    // The run's loads have to be ahead of its serial sums.  4 x 2^25 random-field sites, 36 observations
    // over 1024 steps: 16.2 ms with four ahead and two 4-byte loads per cached value, 9.1 so.
    constexpr int kRun = KIND == kRF ? S : 8;
    if constexpr (T::has_cache) {
#pragma unroll
        for (int p = 0; p <= H; ++p) {
            // both sites of a pair from one row (the last site's row has one)
            const int row = (p < H) ? H - 1 - p : H;
            const int j0 = (p < H) ? p : 2 * H;
            const float4 q = reinterpret_cast<const float4*>(s_loop)[32 * row + lane];
            const float d0 = (p < H) ? lo(d[p < H ? p : 0]) : dT, d1 = hi(d[p < H ? p : 0]);
            float F0, F1;
            if constexpr (KIND == kRF) {
                F0 = fmaf(d0, q.z - q.x, q.x) - f;
                F1 = fmaf(d1, q.w - q.y, q.y) - f;
            } else if constexpr (KIND == kRBGLinear) {
                F0 = (upper & ((p < H) ? M::first(p) : M::last)) ? q.z : q.x;
                F1 = (upper & M::second(p < H ? p : 0)) ? q.w : q.y;
            } else {
                const float2 C = reinterpret_cast<const float2*>(s_loopc)[32 * row + lane];
                F0 = fmaf(d0, fmaf(d0, C.x, q.z), q.x) - f;
                F1 = fmaf(d1, fmaf(d1, C.y, q.w), q.y) - f;
            }
            slot[lane * S + j0] = F0;
            if (p < H)
                slot[lane * S + H + p] = F1;
        }
        __syncwarp();
#pragma unroll kRun
        for (int j = 0; j < S; ++j) {
            const int o = first + j;
            if (o >= 0 && o < owned)
                sF += slot[pad + o];
        }
        __syncwarp();
    }
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const int p = (j < H) ? j : (j < 2 * H) ? j - H : 0;
        const float dj = (j < H) ? lo(d[p]) : (j < 2 * H) ? hi(d[p]) : dT;
        const float cj = (j < H) ? lo(c[p]) : (j < 2 * H) ? hi(c[p]) : cT;
        slot[lane * S + j] = (cj - dref) + dj;   // u - ref
    }
    __syncwarp();
#pragma unroll kRun
    for (int j = 0; j < S; ++j) {
        const int o = first + j;
        if (o >= 0 && o < owned) {
            const float y = slot[pad + o];
            sy += y;
            syy = fmaf(y, y, syy);
            ++cnt;
        }
    }
    if constexpr (T::has_cache) {
        // the slot's cells again
        __syncwarp();
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const int p = (j < H) ? j : (j < 2 * H) ? j - H : 0;
            int32_t n = N0 + __float2int_rn((j < H) ? lo(c[p]) : (j < 2 * H) ? hi(c[p]) : cT);
            if (KIND == kRBGLinear && (upper & ((j < H) ? M::first(p) : (j < 2 * H) ? M::second(p) : M::last)))
                n -= 1;
            s_cell[lane * S + j] = n;
        }
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sF += __shfl_down_sync(kFull, sF, o);
        sy += __shfl_down_sync(kFull, sy, o);
        syy += __shfl_down_sync(kFull, syy, o);
        cnt += __shfl_down_sync(kFull, cnt, o);
    }
    if (lane == 0) {
        const double c_ref = a.shift[chain];
        const double rel = static_cast<double>(ref) - c_ref;
        const double dsy = sy;
        double* dst = a.partial + (static_cast<size_t>(obs) * a.partial_stride + a.tile_base + tile) * 4;
        dst[0] = sF;
        dst[1] = dsy + cnt * rel;
        dst[2] = static_cast<double>(syy) + rel * (2.0 * dsy + cnt * rel);
        dst[3] = c_ref;
    }
}

// A value that is the same in every lane, in a uniform register: the warp reduction returns it there,
// and what is computed from it (addresses, the disorder's counter words, branches) follows.  Per-lane
// registers are what the kernel is short of; the warp index alone gained 0.5% (random field) to 4%
// (uniform random bond).
__device__ __forceinline__ unsigned uniform(unsigned v)
{
    return __reduce_max_sync(kFull, v);
}

// OBS: whether the launch observes at all.  The observation code in the step loop takes registers
// from it, so that launches without any (nearly all of a long relaxation's) have a kernel of their own.
// NEG: chains of a negative drive, whose ordinary moves go downwards (signed_kind).  As one kernel for both signs, by a
// branch or by selecting at the moves, the random field lost 3% to 12%; without the distinction 16 x 2^20
// sites at -f_c, -3 f_c took, ms per 512 steps (random field, uniform cubic, Case 3; at f_c, 3 f_c):
// 10.8 27.2 (8.2 18.5), 16.0 39.9 (10.7 21.0), 18.0 74.6 (12.2 39.3); with it 8.4 18.9,
// 12.3 26.7, 12.1 37.6.
template <int KIND, int S, bool OBS, bool NEG>
__global__ void __maxnreg__((MaxRegs<KIND, S>::value)) split_step_kernel(SplitLaunch a)
{
    using T = Tile<KIND, S>;
    using M = Moves<S>;
    using mask = typename M::mask;
    constexpr int H = T::H;
    constexpr int TW = T::TW;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t s_bar[8];

    const int lane = threadIdx.x & 31;
    const int warp = static_cast<int>(uniform(threadIdx.x >> 5));
    const int tile = blockIdx.x * (blockDim.x >> 5) + warp;
    if (tile >= a.n_tiles)
        return;  // whole warp; the kernel uses no block-wide barrier

    unsigned char* wsm = smem_raw + static_cast<size_t>(warp) * T::bytes;
    int32_t* s_cell = reinterpret_cast<int32_t*>(wsm + T::slot);
    float* s_off = reinterpret_cast<float*>(wsm + T::slot2);
    float* s_loop = reinterpret_cast<float*>(wsm + T::loop);     // loop rows as floats
    float* s_loopc = reinterpret_cast<float*>(wsm + T::loopc);
    float* s_top = reinterpret_cast<float*>(wsm + T::top);
    float2* s_nodes = reinterpret_cast<float2*>(wsm + T::nodes);
    uint16_t* s_q = reinterpret_cast<uint16_t*>(wsm + T::queue);

    const int K = a.K;
    const int pad = a.pad;   // first owned window position
    const WarpTile wt = a.tiles[tile];
    const int32_t L = static_cast<int32_t>(uniform(wt.L));
    const int32_t start = static_cast<int32_t>(uniform(wt.start));
    const int owned = min(a.w_own, L - start);
    const int64_t wstart = static_cast<int64_t>(start) - pad;
    const bool contiguous = (wstart >= 0) && (wstart + TW <= L);
    const float f = __uint_as_float(uniform(__float_as_uint(wt.f)));
    const uint32_t s = uniform(wt.s);
    const int32_t period = static_cast<int32_t>(uniform(wt.period));
    const int64_t chain0 = wt.p - wt.start;   // state index of the chain's first site

    // ---- stage the window in this warp's shared-memory slice ----
    // Contiguous, 16-byte aligned windows arrive by TMA bulk copies (one per array, completion
    // on the warp's mbarrier); windows that wrap around the chain or start unaligned use
    // coalesced read-only loads.  Offsets come first, with the cache, and then the cells through
    // the same slot, where they stay.
    const int64_t p0 = wt.p - pad;
    const bool has_top = T::has_quad || (KIND == kRBGLinear && a.in.q3 != nullptr);   // see SplitState
    const bool tma_in = contiguous && (p0 & 3) == 0;
    uint64_t* bar = &s_bar[warp];
    if (tma_in) {
        if (lane == 0) {
            mbar_init(bar, 1);
            fence_mbar_init();
            mbar_arrive_expect_tx(bar, TW * (4 + CacheBytes<KIND>::hbm + (T::side_by_side ? 4 : 0) + (has_top ? 4 : 0)));
            tma_load_1d(s_off, a.in.off + p0, TW * 4, bar);
            if constexpr (T::side_by_side)
                tma_load_1d(s_cell, a.in.cell + p0, TW * 4, bar);
            if constexpr (T::has_pair)
                tma_load_1d(s_loop, a.in.rf + p0, TW * 8, bar);
            if constexpr (T::has_quad) {
                tma_load_1d(s_nodes, a.in.qn + p0, TW * 8, bar);
                tma_load_1d(s_loop, a.in.qab + p0, TW * 8, bar);
                tma_load_1d(s_loopc, a.in.qc + p0, TW * 4, bar);
            }
            if (has_top)
                tma_load_1d(s_top, a.in.q3 + p0, TW * 4, bar);
        }
        __syncwarp();   // no lane polls the barrier before it is initialised
    }
    int32_t cells[T::early_cells ? S : 1];
    if constexpr (T::early_cells) {
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const int x = 32 * j + lane;
            cells[j] = __ldg(a.in.cell + (contiguous ? p0 + x : chain0 + site_index(wstart, x, false, L)));
        }
    }
    if (tma_in) {
        const bool landed = __all_sync(kFull, mbar_wait(bar, 0));   // warp-uniform outcome
        if (!landed) {
            // the copy did not land: flag it, give the copies one more bounded wait, drop the tile
            if (lane == 0)
                atomicExch(a.error, 1);
            mbar_wait(bar, 0);
            return;
        }
    } else {
        for (int x = lane; x < TW; x += 32) {
            const int64_t p = chain0 + site_index(wstart, x, contiguous, L);
            s_off[x] = __ldg(a.in.off + p);
            if constexpr (T::side_by_side)
                s_cell[x] = __ldg(a.in.cell + p);
            if constexpr (T::has_pair)
                reinterpret_cast<float2*>(s_loop)[x] = __ldg(a.in.rf + p);
            if constexpr (T::has_quad) {
                s_nodes[x] = __ldg(a.in.qn + p);
                reinterpret_cast<float2*>(s_loop)[x] = __ldg(a.in.qab + p);
                s_loopc[x] = __ldg(a.in.qc + p);
            }
            if (has_top)
                s_top[x] = __ldg(a.in.q3 + p);
        }
        __syncwarp();
    }

    // Offsets, two sites to a register pair.  Of a linear-spline random-bond site the sign bit says
    // that it is in the upper of its two cached cells (offsets themselves are never negative).
    pair_t c[H], d[H];
    float cT, dT;
    mask upper = 0;
#pragma unroll
    for (int p = 0; p < H; ++p) {
        float d0 = s_off[lane * S + p], d1 = s_off[lane * S + H + p];
        if constexpr (KIND == kRBGLinear) {
            if (__float_as_int(d0) < 0)
                upper |= M::first(p);
            if (__float_as_int(d1) < 0)
                upper |= M::second(p);
            d0 = fabsf(d0);
            d1 = fabsf(d1);
        }
        d[p] = pk(d0, d1);
    }
    dT = s_off[lane * S + 2 * H];
    if constexpr (KIND == kRBGLinear) {
        if (__float_as_int(dT) < 0)
            upper |= M::last;
        dT = fabsf(dT);
    }
    // The cache, from the linear order of memory to the rows of the update loop.
    if constexpr (T::has_cache) {
        float2 q[S];
        float qc[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
            q[j] = reinterpret_cast<float2*>(s_loop)[lane * S + j];
            if constexpr (T::has_quad)
                qc[j] = s_loopc[lane * S + j];
        }
        __syncwarp();   // every lane has read: the rows may overwrite the linear order
#pragma unroll
        for (int p = 0; p <= H; ++p) {
            const int row = (p < H) ? H - 1 - p : H;
            const int j0 = (p < H) ? p : 2 * H, j1 = (p < H) ? H + p : 2 * H;
            reinterpret_cast<float4*>(s_loop)[32 * row + lane] = make_float4(q[j0].x, q[j1].x, q[j0].y, q[j1].y);
            if constexpr (T::has_quad)
                reinterpret_cast<float2*>(s_loopc)[32 * row + lane] = make_float2(qc[j0], qc[j1]);
        }
        // the offsets are in registers: the cells may overwrite the slot
        if constexpr (T::early_cells) {
            __syncwarp();
#pragma unroll
            for (int j = 0; j < S; ++j)
                s_cell[32 * j + lane] = cells[j];
            __syncwarp();
        } else if constexpr (!T::side_by_side) {
            fence_proxy_async_shared();
            __syncwarp();
            if (tma_in) {
                if (lane == 0) {
                    mbar_arrive_expect_tx(bar, TW * 4);
                    tma_load_1d(s_cell, a.in.cell + p0, TW * 4, bar);
                }
                const bool landed = __all_sync(kFull, mbar_wait(bar, 1));
                if (!landed) {
                    if (lane == 0)
                        atomicExch(a.error, 1);
                    mbar_wait(bar, 1);
                    return;
                }
            } else {
                for (int x = lane; x < TW; x += 32)
                    s_cell[x] = __ldg(a.in.cell + chain0 + site_index(wstart, x, contiguous, L));
                __syncwarp();
            }
        }
    }
    // Cells are carried as exact small floats relative to the warp's reference cell N0 (window
    // position 0): a neighbour difference is then (c' - c) + (d' - d), three FP32 operations.
    // Neighbouring displacements differ by less than 2^12, so a tile's cells stay far below 2^24.
    const int32_t N0 = static_cast<int32_t>(uniform(s_cell[0]));
#pragma unroll
    for (int p = 0; p < H; ++p)
        c[p] = pk(static_cast<float>(s_cell[lane * S + p] - N0), static_cast<float>(s_cell[lane * S + H + p] - N0));
    cT = static_cast<float>(s_cell[lane * S + 2 * H] - N0);
    __syncwarp();   // N0 is read by every lane before any cell changes
    if constexpr (KIND == kRBGLinear) {
        // from here on the slot holds the lower of each site's two cached cells
#pragma unroll
        for (int p = 0; p < H; ++p) {
            if (upper & M::first(p))
                s_cell[lane * S + p] -= 1;
            if (upper & M::second(p))
                s_cell[lane * S + H + p] -= 1;
        }
        if (upper & M::last)
            s_cell[lane * S + 2 * H] -= 1;
        __syncwarp();
        if (!has_top) {
#pragma unroll 1
            for (int x = lane; x < TW; x += 32)
                s_top[x] = pair_node_f32<KIND>(a.keys, s, site_index(wstart, x, contiguous, L),
                                               wrap_node(s_cell[x] + (NEG ? 0 : 2), period), f);
            __syncwarp();
        }
    }

    Force<KIND, S> force;
    force.rows = reinterpret_cast<const float4*>(s_loop) + lane;
    force.rows_c = reinterpret_cast<const float2*>(s_loopc) + lane;
    force.f2 = pk(f, f);
    const pair_t dt2 = pk(a.dt, a.dt);

    // ---- K Euler steps: state in registers, cache in shared memory ----
    unsigned n_cross = 0;
    const unsigned lanes_below = (1u << lane) - 1u;
    // observations inside the launch: the next one, the reference cell of its sums, and the step
    // before which the next thing has to be done about it
    int obs = 0, obs_ref = 0, obs_step = OBS ? a.obs_at[0] - a.obs_len[0] : -1;
    bool obs_marked = false;
#pragma unroll 1
    for (int k = 0;; ++k) {
        while (OBS && k == obs_step) {
            if (!obs_marked) {
                // the sums are relative to the cell, at this step, of the site `len` before the tile
                obs_ref = cell_at<KIND, S>(s_cell, pad - a.obs_len[obs], lane, N0, c, cT, upper);
                __syncwarp();   // read by every lane before the slot is written again
                obs_marked = true;
            } else {
                observe_tile<KIND, S>(a, f, tile, wt.chain, obs, obs_ref, owned, pad, N0, lane, c, d, cT, dT, upper, s_cell,
                                      s_off, s_loop, s_loopc);
                obs_marked = false;
                ++obs;
            }
            obs_step = (obs < a.n_obs) ? a.obs_at[obs] - (obs_marked ? 0 : a.obs_len[obs]) : -1;
        }
        if (k == K)
            break;
        // Window positions 0 and TW - 1 take themselves as their outer neighbour: they go stale
        // either way, and a zero slope there keeps the stale edge from drifting off and making
        // spurious cell moves (each of which would draw disorder values).
        const float cr = __shfl_down_sync(kFull, lo(c[0]), 1);
        const float dr = __shfl_down_sync(kFull, lo(d[0]), 1);
        const float DpT = (lane == 31) ? 0.0f : (cr - cT) + (dr - dT);   // the lane's last site to its right
        const float Dl0 = __shfl_up_sync(kFull, DpT, 1);
        const float Dl = (lane == 0) ? 0.0f : Dl0;                       // to the lane's first site
        // the last pair's right neighbours: the second run's first site, and the last site
        const pair_t DpL = add2(sub2(pk(hi(c[0]), cT), c[H - 1]), sub2(pk(hi(d[0]), dT), d[H - 1]));
        pair_t Dm = pk(Dl, lo(DpL));   // u_j - u_{j-1}
        MoveCodes<S> codes;
#pragma unroll
        for (int p = 0; p < H; ++p) {
            const pair_t Dp = (p + 1 < H) ? add2(sub2(c[p + 1 < H ? p + 1 : p], c[p]), sub2(d[p + 1 < H ? p + 1 : p], d[p])) : DpL;
            const pair_t g = force.pair(p, d[p], upper);   // F_p + f
            const pair_t dn = fma2(dt2, add2(sub2(Dp, Dm), g), d[p]);
            Dm = Dp;
            // Branch-free renormalisation.  d - floor(d) is exact; a tiny negative d can round up
            // to exactly 1, which is a valid representation (the interpolated force is continuous).
            const pair_t fl = floor2(dn);
            c[p] = add2(c[p], fl);
            d[p] = sub2(dn, fl);
            codes.put(p, lo(fl), hi(fl));
        }
        {
            const float g = force.last(dT, upper);
            const float dn = fmaf(a.dt, (DpT - hi(DpL)) + g, dT);
            const float fl = floorf(dn);
            cT += fl;
            dT = dn - fl;
            codes.put_last(fl);
        }
        mask moved = 0, down = 0;
        bool lane_far = false;
        if (T::has_cache || a.crossings)
            codes.template masks<T::kDown, NEG>(moved, down, lane_far);
        if (a.crossings)
            n_cross += __reduce_add_sync(kFull, static_cast<unsigned>(mask_popc(moved)));
        if constexpr (T::has_cache) {
            const bool far = __any_sync(kFull, lane_far);
            mask req = moved;   // requests: sites whose cache has to change
            if constexpr (KIND == kRBGLinear) {
                if (far) {
                    // Some site moved two cells or more.  Each lane redraws those of its own, the new cell
                    // being the lower (NEG: upper) of the two in the cache, and the others take the queue.
                    // 16 x 2^20 sites driven at 8 f_c, where most steps of a tile have a far move, ms per 512
                    // steps: 147 with all moved sites redrawn, 117 with the far ones in the queue among
                    // the others, 110 so.
                    const mask m = codes.far_ones();
                    const int32_t base = NEG ? N0 - 1 : N0;
#pragma unroll
                    for (int p = 0; p < H; ++p) {
                        if (m & M::first(p))
                            s_cell[lane * S + p] = base + __float2int_rn(lo(c[p]));
                        if (m & M::second(p))
                            s_cell[lane * S + H + p] = base + __float2int_rn(hi(c[p]));
                    }
                    if (m & M::last)
                        s_cell[lane * S + 2 * H] = base + __float2int_rn(cT);
                    moved &= ~m;
                    upper = NEG ? (upper | m) : (upper & ~m);
                    for (mask left = m; left != 0;) {
                        const int b = mask_top(left);
                        left = mask_drop(left, b);
                        const bool first = b >= M::D;
                        const int t = first ? b - M::D : b;
                        const int x = lane * S + (H - 1 - t) + (first ? 0 : H) + (t == H ? S : 0);
                        float* row = s_loop + 4 * (32 * t + lane) + (first ? 0 : 1);
                        const int32_t i = contiguous ? static_cast<int32_t>(wstart) + x : site_index(wstart, x, contiguous, L);
                        const int32_t lower = s_cell[x];
                        float g = 0.0f, prev = 0.0f;
#pragma unroll 1
                        for (int r = 0; r < 3; ++r) {
                            const float v = pair_node_f32<KIND>(a.keys, s, i, wrap_node(lower + (NEG ? 2 - r : r), period), f);
                            row[NEG ? 2 : 0] = g;
                            g = NEG ? v - prev : prev - v;
                            prev = v;
                        }
                        row[NEG ? 0 : 2] = g;
                        s_top[x] = prev;
                    }
                }
                down &= moved;
                const mask up = moved & ~down;
                req = (up & upper) | (down & ~upper);
                upper = (upper | up) & ~down;
            } else if (far) {
                // the lanes leave their new cells in the slot, and every site that moved redraws all of
                // its nodes
#pragma unroll
                for (int p = 0; p < H; ++p) {
                    s_cell[lane * S + p] = N0 + __float2int_rn(lo(c[p]));
                    s_cell[lane * S + H + p] = N0 + __float2int_rn(hi(c[p]));
                }
                s_cell[lane * S + 2 * H] = N0 + __float2int_rn(cT);
            }
            // Queue the requests, one per lane and pass: a lane's slot is its rank in the ballot of the
            // lanes that still have one (no prefix sum; three or four passes empty the masks)
            unsigned have = __ballot_sync(kFull, req != 0);
            if (have) {
                do {
                    int n_here = 0;
                    do {
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const int b = mask_top(req);
                            unsigned e = (lane << 7) + b;
                            if (T::kDown)
                                e += static_cast<unsigned>(down >> (b & (M::wide ? 63 : 31)) & 1u) << 6;
                            const int q = n_here + __popc(have & lanes_below);
                            if (req != 0)
                                s_q[q] = static_cast<uint16_t>(e);
                            req = mask_drop(req, b);
                            n_here += __popc(have);
                            have = __ballot_sync(kFull, req != 0);
                        }
                    } while (have && n_here <= T::kQueue - 64);
                    __syncwarp();
                    for (int base = 0; base < n_here; base += 32) {
                        if (base + lane < n_here) {
                            const int e = s_q[base + lane];
                            const int b = e & 63, src = e >> 7;
                            const bool first = b >= M::D;
                            const int t = first ? b - M::D : b;            // row of the pair
                            const int x = src * S + (H - 1 - t) + (first ? 0 : H) + (t == H ? S : 0);
                            float* row = s_loop + 4 * (32 * t + src) + (first ? 0 : 1);
                            const int step = KIND != kRBGLinear && far ? 0 : (T::kDown ? (e & 64) != 0 : NEG) ? -1 : 1;
                            const int32_t i = contiguous ? static_cast<int32_t>(wstart) + x
                                                         : site_index(wstart, x, contiguous, L);
                            const int32_t slot = s_cell[x];
                            if constexpr (KIND == kRF) {
                                // a move keeps the node between the two cells and draws the one beyond
                                // the new cell; a far move draws both
                                constexpr int beyond = NEG ? 0 : 1;
                                const int32_t nn = slot + step;
                                const float old = row[2 * beyond];
                                const float v = pair_node_f32<KIND>(a.keys, s, i, wrap_node(nn + beyond, period), f);
                                row[2 - 2 * beyond] = far ? pair_node_f32<KIND>(a.keys, s, i, wrap_node(nn + 1 - beyond, period), f) : old;
                                row[2 * beyond] = v;
                                if (!far)
                                    s_cell[x] = nn;
                            } else if constexpr (KIND == kRBGLinear) {
                                // The pair of cells moves on by one, in the direction of the drive with one
                                // new node beyond it, against it with its three nodes drawn anew, in the
                                // drive's order.  (The first draw inside the loop as well: 2% slower at f_c,
                                // 5% at 3 f_c.)
                                constexpr int behind = NEG ? 2 : 0, front = NEG ? 0 : 2;   // F_p of the two cells, in that order
                                const bool ahead = NEG ? step < 0 : step > 0;
                                const int32_t lower = slot + step;
                                const int32_t n0 = lower + (ahead != NEG ? 2 : 0);
                                float v = pair_node_f32<KIND>(a.keys, s, i, wrap_node(n0, period), f);
                                float gb = row[front], prev = s_top[x];
                                float gf = NEG ? v - prev : prev - v;   // F_p of the cell between the two nodes
                                prev = v;
                                if (!ahead) {
#pragma unroll 1
                                    for (int r = 1; r < 3; ++r) {
                                        v = pair_node_f32<KIND>(a.keys, s, i, wrap_node(n0 + (NEG ? -r : r), period), f);
                                        gb = gf;
                                        gf = NEG ? v - prev : prev - v;
                                        prev = v;
                                    }
                                }
                                row[behind] = gb;
                                row[front] = gf;
                                s_top[x] = prev;
                                s_cell[x] = lower;
                            } else {
                                // The spline over the new cell n needs V(n-1 .. n+2).  The cache holds
                                // V, V(+1), V(+2) of the old cell: an up move draws V(n+2), a down move
                                // V(n-1) and V(n) (V(n-1) is not kept), a far move all four.
                                const int32_t nn = slot + step;
                                if (!far)
                                    s_cell[x] = nn;
                                const bool up = step > 0;
                                const float2 o = s_nodes[x];
                                float n0 = o.x, n1 = o.y, n2 = s_top[x];
                                float n3 = quad_node_f32<KIND>(a.keys, s, i, wrap_node(up ? nn + 2 : nn - 1, period));
                                if (!up) {
                                    const float v = n3;
                                    n3 = n1;
                                    n2 = n0;
                                    n0 = v;
#pragma unroll 1
                                    for (int r = 0; r < (far ? 3 : 1); ++r) {
                                        const float w = quad_node_f32<KIND>(a.keys, s, i, wrap_node(nn + r, period));
                                        if (r == 0)
                                            n1 = w;
                                        else if (r == 1)
                                            n2 = w;
                                        else
                                            n3 = w;
                                    }
                                }
                                s_nodes[x] = make_float2(n1, n2);
                                s_top[x] = n3;
                                float A, B, C;
                                rb_coefficients(n0, n1, n2, n3, f, A, B, C);
                                row[0] = A;
                                row[2] = B;
                                s_loopc[2 * (32 * t + src) + (first ? 0 : 1)] = C;
                            }
                        }
                        __syncwarp();
                    }
                } while (have);
            }
        }
    }

    if (a.crossings) {
        if (lane == 0 && n_cross)
            atomicAdd(a.crossings, static_cast<unsigned long long>(n_cross));
    }
    if (K == 0)
        return;


    // ---- write the owned sites back: registers -> shared -> global ----
    __syncwarp();
    const int64_t out0 = wt.p;
    const bool tma_out = ((pad & 3) == 0) && ((out0 & 3) == 0) && ((owned & 3) == 0);
    if constexpr (!T::has_cache || KIND == kRBGLinear) {
        // (the other kinds' slots already hold the cells)
#pragma unroll
        for (int p = 0; p < H; ++p) {
            s_cell[lane * S + p] = N0 + __float2int_rn(lo(c[p]));
            s_cell[lane * S + H + p] = N0 + __float2int_rn(hi(c[p]));
        }
        s_cell[lane * S + 2 * H] = N0 + __float2int_rn(cT);
    }
    // offsets, into the slot: side by side at once, else once the cells have left it
    auto put_offsets = [&]() {
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const int p = (j < H) ? j : (j < 2 * H) ? j - H : 0;
            float dj = (j < H) ? lo(d[p]) : (j < 2 * H) ? hi(d[p]) : dT;
            if constexpr (KIND == kRBGLinear) {
                if (upper & ((j < H) ? M::first(p) : (j < 2 * H) ? M::second(p) : M::last))
                    dj = -dj;
            }
            s_off[lane * S + j] = dj;
        }
    };
    if constexpr (T::side_by_side)
        put_offsets();
    if constexpr (T::has_cache) {
        // the cache back to linear order
        float2 q[S];
        float qc[S];
#pragma unroll
        for (int p = 0; p <= H; ++p) {
            const int row = (p < H) ? H - 1 - p : H;
            const int j0 = (p < H) ? p : 2 * H;
            const float4 r = reinterpret_cast<const float4*>(s_loop)[32 * row + lane];
            q[j0] = make_float2(r.x, r.z);
            if (p < H)
                q[H + (p < H ? p : 0)] = make_float2(r.y, r.w);
            if constexpr (T::has_quad) {
                const float2 r2 = reinterpret_cast<const float2*>(s_loopc)[32 * row + lane];
                qc[j0] = r2.x;
                if (p < H)
                    qc[H + (p < H ? p : 0)] = r2.y;
            }
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < S; ++j) {
            reinterpret_cast<float2*>(s_loop)[lane * S + j] = q[j];
            if constexpr (T::has_quad)
                s_loopc[lane * S + j] = qc[j];
        }
        if (tma_out) {
            fence_proxy_async_shared();   // generic-proxy writes above -> visible to the bulk copy
            __syncwarp();
            if (lane == 0) {
                const uint32_t cnt = static_cast<uint32_t>(owned);
                tma_store_1d(a.out.cell + out0, s_cell + pad, cnt * 4);
                if constexpr (T::side_by_side)
                    tma_store_1d(a.out.off + out0, s_off + pad, cnt * 4);
                if constexpr (T::has_pair)
                    tma_store_1d(a.out.rf + out0, reinterpret_cast<float2*>(s_loop) + pad, cnt * 8);
                if constexpr (T::has_quad) {
                    tma_store_1d(a.out.qn + out0, s_nodes + pad, cnt * 8);
                    tma_store_1d(a.out.qab + out0, reinterpret_cast<float2*>(s_loop) + pad, cnt * 8);
                    tma_store_1d(a.out.qc + out0, s_loopc + pad, cnt * 4);
                }
                if (has_top)
                    tma_store_1d(a.out.q3 + out0, s_top + pad, cnt * 4);
                tma_store_commit();
                tma_store_wait_read_all();   // the slot may be overwritten
            }
            __syncwarp();
        } else {
            __syncwarp();
            for (int o = lane; o < owned; o += 32) {
                const int x = o + pad;
                const int64_t p = out0 + o;
                a.out.cell[p] = s_cell[x];
                if constexpr (T::side_by_side)
                    a.out.off[p] = s_off[x];
                if constexpr (T::has_pair)
                    a.out.rf[p] = reinterpret_cast<float2*>(s_loop)[x];
                if constexpr (T::has_quad) {
                    a.out.qn[p] = s_nodes[x];
                    a.out.qab[p] = reinterpret_cast<float2*>(s_loop)[x];
                    a.out.qc[p] = s_loopc[x];
                }
                if (has_top)
                    a.out.q3[p] = s_top[x];
            }
            __syncwarp();
        }
    }
    if constexpr (T::has_cache && T::side_by_side)
        return;
    if constexpr (!T::side_by_side)
        put_offsets();
    if (tma_out) {
        fence_proxy_async_shared();
        __syncwarp();
        if (lane == 0) {
            tma_store_1d(a.out.off + out0, s_off + pad, static_cast<uint32_t>(owned) * 4);
            if constexpr (!T::has_cache)
                tma_store_1d(a.out.cell + out0, s_cell + pad, static_cast<uint32_t>(owned) * 4);
            tma_store_commit();
            // shared memory must outlive the reads (the writes end with the kernel)
            tma_store_wait_read_all();
        }
    } else {
        __syncwarp();
        for (int o = lane; o < owned; o += 32) {
            a.out.off[out0 + o] = s_off[o + pad];
            if constexpr (!T::has_cache)
                a.out.cell[out0 + o] = s_cell[o + pad];
        }
    }
}

template <int KIND, int S, bool OBS, bool NEG>
cudaError_t launch_split_as(int tiles_per_cta, const SplitLaunch& a, cudaStream_t st)
{
    const size_t smem = static_cast<size_t>(tiles_per_cta) * Tile<KIND, S>::bytes;
    auto kern = split_step_kernel<KIND, S, OBS, NEG>;
    // raise the dynamic shared-memory limit of this kernel on this device to the largest shape in
    // use; under a lock, so that two threads raising it at once cannot leave the smaller value
    static std::mutex s_mu;
    static int s_limit[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    {
        std::lock_guard<std::mutex> g(s_mu);
        const bool tracked = dev >= 0 && dev < 64;
        if (!tracked || static_cast<int>(smem) > s_limit[dev]) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
            if (e != cudaSuccess)
                return e;
            if (tracked)
                s_limit[dev] = static_cast<int>(smem);
        }
    }
    const int grid = (a.n_tiles + tiles_per_cta - 1) / tiles_per_cta;
    if (grid == 0)
        return cudaSuccess;
    kern<<<grid, 32 * tiles_per_cta, smem, st>>>(a);
    return cudaGetLastError();
}

template <int KIND, int S>
cudaError_t launch_split(int tiles_per_cta, const SplitLaunch& a, cudaStream_t st)
{
    if constexpr (signed_kind(KIND))
        if (a.neg)
            return a.n_obs > 0 ? launch_split_as<KIND, S, true, true>(tiles_per_cta, a, st) :
                                 launch_split_as<KIND, S, false, true>(tiles_per_cta, a, st);
    return a.n_obs > 0 ? launch_split_as<KIND, S, true, false>(tiles_per_cta, a, st) :
                         launch_split_as<KIND, S, false, false>(tiles_per_cta, a, st);
}

__global__ void split_tiles_kernel(const ChainDesc* chains, int cls, int32_t w_own, const int32_t* first, WarpTile* tiles)
{
    const int32_t c = blockIdx.x;
    const ChainDesc ch = chains[c];
    if (chain_class(ch.kind, ch.neg) != cls)
        return;
    WarpTile* mine = tiles + first[c];
    for (int64_t k = threadIdx.x; k * w_own < ch.L; k += blockDim.x) {
        const int32_t start = static_cast<int32_t>(k * w_own);
        mine[k] = WarpTile{ch.offset + start, start, ch.L, c, ch.s, ch.f32, ch.period};
    }
}

// ---------------------------------------------------------------------------------------
// Initialisation (flat start or a given FP64 state) and conversion back to FP64.
// Block tiles of w_tile sites, one thread per site.
// ---------------------------------------------------------------------------------------
__global__ void split_init_kernel(const ChainDesc* chains, const TileDesc* tiles, int32_t w_tile, SplitState st,
                                  PhiloxKeys keys, const double* u_in)
{
    const TileDesc td = tiles[blockIdx.x];
    const ChainDesc ch = chains[td.chain];
    for (int x = threadIdx.x; x < w_tile; x += blockDim.x) {
        const int32_t i = td.start + x;
        if (i >= ch.L)
            break;
        const int64_t p = ch.offset + i;
        int32_t n = 0;
        float d = 0.0f;
        if (u_in) {
            const double u = u_in[ch.dense + i];
            const double fl = floor(u);
            n = static_cast<int32_t>(fl);
            d = static_cast<float>(u - fl);
            if (d >= 1.0f) {
                d = 0.0f;
                n += 1;
            }
        }
        st.cell[p] = n;
        st.off[p] = d;
        const int32_t M = ch.period;
        const int32_t m0 = wrap_node(n - 1, M), m1 = wrap_node(n, M), m2 = wrap_node(n + 1, M), m3 = wrap_node(n + 2, M);
        if (ch.kind == kRF)
            st.rf[p] = make_float2(pair_node_f32<kRF>(keys, ch.s, i, m1, ch.f32), pair_node_f32<kRF>(keys, ch.s, i, m2, ch.f32));
        else if (ch.kind == kRBGLinear)
        {
            // the site's cell and the next one in the direction of the drive; the sign of the offset says
            // that the site is in the upper one
            const bool neg = ch.neg;
            const float g1 = rbg_f32(keys, ch.s, i, m1), g2 = rbg_f32(keys, ch.s, i, m2);
            const float g3 = rbg_f32(keys, ch.s, i, neg ? m0 : m3);
            st.rf[p] = neg ? make_float2(g3 - g1, g1 - g2) : make_float2(g1 - g2, g2 - g3);
            if (st.q3)
                st.q3[p] = g3;
            st.off[p] = neg ? -d : d;
        }
        else if (ch.kind == kRB || ch.kind == kRBGCubic) {
            const bool uni = ch.kind == kRB;
            const float p0 = uni ? rb_f32(keys, ch.s, i, m0) : rbg_f32(keys, ch.s, i, m0);
            const float p1 = uni ? rb_f32(keys, ch.s, i, m1) : rbg_f32(keys, ch.s, i, m1);
            const float p2 = uni ? rb_f32(keys, ch.s, i, m2) : rbg_f32(keys, ch.s, i, m2);
            const float p3 = uni ? rb_f32(keys, ch.s, i, m3) : rbg_f32(keys, ch.s, i, m3);
            float A, B, C;
            rb_coefficients(p0, p1, p2, p3, ch.f32, A, B, C);
            st.qn[p] = make_float2(p1, p2);
            st.q3[p] = p3;
            st.qab[p] = make_float2(A, B);
            st.qc[p] = C;
        }
    }
}

__global__ void split_to_f64_kernel(const ChainDesc* chains, const TileDesc* tiles, int32_t w_tile, SplitState st,
                                    double* u_out, int32_t* cells_out)
{
    const TileDesc td = tiles[blockIdx.x];
    const ChainDesc ch = chains[td.chain];
    for (int x = threadIdx.x; x < w_tile; x += blockDim.x) {
        const int32_t i = td.start + x;
        if (i >= ch.L)
            break;
        const int64_t p = ch.offset + i;
        if (u_out)
            u_out[ch.dense + i] = static_cast<double>(st.cell[p]) + static_cast<double>(fabsf(st.off[p]));
        if (cells_out)
            cells_out[ch.dense + i] = st.cell[p];
    }
}

}  // namespace

bool split_supported(int kind, int S)
{
    if (quad_kind(kind))
        return S == 7 || S == 15;
    if (kind == kNone)
        return S == 7 || S == 15 || S == 23 || S == 31;
    return S == 7 || S == 15 || S == 23 || S == 31 || S == 39;
}

template <int KIND>
constexpr int tile_bytes(int S)
{
    switch (S) {
    case 7: return Tile<KIND, 7>::bytes;
    case 15: return Tile<KIND, 15>::bytes;
    case 23: return Tile<KIND, 23>::bytes;
    case 31: return Tile<KIND, 31>::bytes;
    default: return Tile<KIND, 39>::bytes;
    }
}

size_t split_smem_bytes(int kind, int S, int tiles_per_cta)
{
    const int b = kind == kRF ? tile_bytes<kRF>(S) : kind == kRBGLinear ? tile_bytes<kRBGLinear>(S) :
                  kind == kNone ? tile_bytes<kNone>(S) : tile_bytes<kRB>(S);
    return static_cast<size_t>(tiles_per_cta) * b;
}

template <int KIND>
constexpr int max_regs(int S)
{
    switch (S) {
    case 7: return MaxRegs<KIND, 7>::value;
    case 15: return MaxRegs<KIND, 15>::value;
    case 23: return MaxRegs<KIND, 23>::value;
    case 31: return MaxRegs<KIND, 31>::value;
    default: return MaxRegs<KIND, 39>::value;
    }
}

int split_warps_per_sm(int kind, int S)
{
    const int regs = kind == kRBGLinear ? max_regs<kRBGLinear>(S) : quad_kind(kind) ? max_regs<kRB>(S) : max_regs<kRF>(S);
    return std::min(65536 / (32 * regs), static_cast<int>(227 * 1024 / split_smem_bytes(kind, S, 1)));
}

cudaError_t split_step(int kind, int S, int tiles_per_cta, const SplitLaunch& a, cudaStream_t st)
{
    if (kind == kRF) {
        switch (S) {
        case 7: return launch_split<kRF, 7>(tiles_per_cta, a, st);
        case 15: return launch_split<kRF, 15>(tiles_per_cta, a, st);
        case 23: return launch_split<kRF, 23>(tiles_per_cta, a, st);
        case 31: return launch_split<kRF, 31>(tiles_per_cta, a, st);
        case 39: return launch_split<kRF, 39>(tiles_per_cta, a, st);
        }
    } else if (kind == kRBGLinear) {
        switch (S) {
        case 7: return launch_split<kRBGLinear, 7>(tiles_per_cta, a, st);
        case 15: return launch_split<kRBGLinear, 15>(tiles_per_cta, a, st);
        case 23: return launch_split<kRBGLinear, 23>(tiles_per_cta, a, st);
        case 31: return launch_split<kRBGLinear, 31>(tiles_per_cta, a, st);
        case 39: return launch_split<kRBGLinear, 39>(tiles_per_cta, a, st);
        }
    } else if (kind == kRB) {
        switch (S) {
        case 7: return launch_split<kRB, 7>(tiles_per_cta, a, st);
        case 15: return launch_split<kRB, 15>(tiles_per_cta, a, st);
        }
    } else if (kind == kRBGCubic) {
        switch (S) {
        case 7: return launch_split<kRBGCubic, 7>(tiles_per_cta, a, st);
        case 15: return launch_split<kRBGCubic, 15>(tiles_per_cta, a, st);
        }
    } else if (kind == kNone) {
        switch (S) {
        case 7: return launch_split<kNone, 7>(tiles_per_cta, a, st);
        case 15: return launch_split<kNone, 15>(tiles_per_cta, a, st);
        case 23: return launch_split<kNone, 23>(tiles_per_cta, a, st);
        case 31: return launch_split<kNone, 31>(tiles_per_cta, a, st);
        }
    }
    return cudaErrorInvalidValue;
}

cudaError_t split_tiles(const ChainDesc* chains, int32_t n_chains, int cls, int32_t w_own, const int32_t* first,
                        WarpTile* tiles, cudaStream_t stream)
{
    split_tiles_kernel<<<n_chains, 256, 0, stream>>>(chains, cls, w_own, first, tiles);
    return cudaGetLastError();
}

cudaError_t split_init(const ChainDesc* chains, int32_t, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile,
                       SplitState st, uint64_t seed, int, const double* u_in, cudaStream_t stream)
{
    if (n_tiles == 0)
        return cudaSuccess;
    split_init_kernel<<<n_tiles, 256, 0, stream>>>(chains, tiles, w_tile, st, philox_key_schedule(seed), u_in);
    return cudaGetLastError();
}

cudaError_t split_to_f64(const ChainDesc* chains, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile,
                         SplitState st, double* u_out, int32_t* cells_out, cudaStream_t stream)
{
    if (n_tiles == 0)
        return cudaSuccess;
    split_to_f64_kernel<<<n_tiles, 256, 0, stream>>>(chains, tiles, w_tile, st, u_out, cells_out);
    return cudaGetLastError();
}

}  // namespace qew
