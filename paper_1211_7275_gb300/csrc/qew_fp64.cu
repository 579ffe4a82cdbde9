// qew_fp64.cu -- the plain FP64 path of the qEW relaxation: FP64 state in HBM (ping-pong), a tile of sites
// per block advanced by several Euler steps in shared memory, and each site's disorder values cached for
// the cell they were drawn for (regenerated when the site changes cell).
//
// Method: Eq. 1 of arXiv:1211.7275 with eta = c = 1, periodic in x, explicit Euler with all
// forces from the old state (Sec. III.B); pinning force by linear interpolation of R (RF), as
// minus the derivative of the Catmull-Rom spline through V or G (cubic random bond, Cases 1-2),
// or as G(n) - G(n+1) (linear-spline random bond, Case 3) (Sec. III.B, Sec. IV.C); observables
// of Eqs. 3-5.  Every FP64 operation is an explicit round-to-nearest intrinsic so that no
// multiply-add is contracted: the rounding sequence is the textbook one, operation by operation,
// (1 - d) R(n) + d R(n+1) for the force and u + dt ((lap + f) + F) for the update, with
// lap = (u_{i+1} + u_{i-1}) - 2 u_i.
#include "qew_internal.h"

namespace qew {
namespace {

// One disorder node in FP64: R (RF), V (uniform random bond) or G (Gaussian random bond).
// (n is the cell-relative node index; `period` > 0 makes the disorder periodic in u)
template <int KIND>
__device__ __forceinline__ double node_f64(uint64_t seed, uint32_t s, int32_t i, int32_t n, int32_t period)
{
    n = wrap_node(n, period);
    if constexpr (KIND == kRF)
        return rf_f64(seed, s, i, n);
    else if constexpr (KIND == kRB)
        return rb_f64(seed, s, i, n);
    else
        return rbg_f64(seed, s, i, n);
}

// ---- the step kernel ----
// A block advances a tile of w_own sites by K steps on the window of w_own + 2 (K - 1) sites whose
// values the last owned one depends on (plus one neighbour on each side): one site per thread and
// round, displacements in shared memory (double-buffered), what the update reads in registers.
//
// What bounds it: the FP64 unit takes one warp instruction in 16 clocks per SM, and the next
// instruction of the same warp waits 65.  A step itself is 11 FP64 operations (RF); a disorder value
// (log, sqrt, cospi) is some 80.  So
//   - a cell is left when u - floor is outside [0, 1), an integer test of its high word: no floor and
//     no conversion for the sites that stay;
//   - the sites of the block that did change cell are queued and their values drawn by as few warps as
//     hold them.  Drawn where they occur, a warp with one crossing among its 32 sites spent the time
//     of 32 (16 x 2^20 RF sites over the first 64 steps: 2.03 ms per step then, 0.65 now);
//   - a small batch is spread over many SMs in small tiles and advanced K steps per launch.
// Loop values of a site: RF R(n), R(n+1); linear spline F; cubic ca, 2 b, 3 c of the force.
// Cached nodes of a site in cell n: V(n + lo) .. V(n + lo + n_nodes - 1), the force's.  With look-ahead
// there are n_look of them, from V(n + lo - used): the one that a move in the direction of the drive will
// need (neg: a negative drive's, downwards), and for the linear spline, whose sites move up and down
// across a node, both; the force's start at `used`.
template <int KIND>
struct F64Site {
    static constexpr int n_nodes = pair_kind(KIND) ? 2 : quad_kind(KIND) ? 4 : 0;
    static constexpr int lo = quad_kind(KIND) ? -1 : 0;
    static constexpr int n_look = KIND == kRBGLinear ? 4 : n_nodes > 0 ? n_nodes + 1 : 0;
    static __host__ __device__ constexpr int used(bool neg) { return KIND == kRBGLinear || (neg && n_nodes > 0) ? 1 : 0; }
    static constexpr int n_loop = KIND == kRF ? 2 : KIND == kRBGLinear ? 1 : quad_kind(KIND) ? 3 : 0;
};
// A node that has not been drawn.
constexpr int kNoNode = 0x7FF80000;   // high word (a quiet NaN)
__device__ __forceinline__ bool no_node(double v) { return __double2hiint(v) == kNoNode; }

// The loop values of a cell from its nodes, in the rounding sequence of the force's definition.
template <int KIND>
__device__ __forceinline__ void loop_values(const double* p, double* v)
{
    if constexpr (KIND == kRF) {
        v[0] = p[0];
        v[1] = p[1];
    } else if constexpr (KIND == kRBGLinear) {
        v[0] = __dsub_rn(p[0], p[1]);   // minus the slope of the linear spline through G
    } else if constexpr (quad_kind(KIND)) {
        // -1/2 [(p2 - p0) + 2 b d + 3 c d^2], b = 2p0 - 5p1 + 4p2 - p3, c = -p0 + 3p1 - 3p2 + p3
        v[0] = __dsub_rn(p[2], p[0]);
        v[1] = __dmul_rn(2.0, __dsub_rn(__dadd_rn(__dsub_rn(__dmul_rn(2.0, p[0]), __dmul_rn(5.0, p[1])), __dmul_rn(4.0, p[2])), p[3]));
        v[2] = __dmul_rn(3.0, __dadd_rn(__dsub_rn(__dsub_rn(__dmul_rn(3.0, p[1]), p[0]), __dmul_rn(3.0, p[2])), p[3]));
    }
}

template <int KIND>
__device__ __forceinline__ double force_f64(double d, const double* v)
{
    if constexpr (KIND == kRF)
        return __dadd_rn(__dmul_rn(__dsub_rn(1.0, d), v[0]), __dmul_rn(d, v[1]));
    else if constexpr (KIND == kRBGLinear)
        return v[0];
    else if constexpr (quad_kind(KIND))
        return __dmul_rn(-0.5, __dadd_rn(__dadd_rn(v[0], __dmul_rn(v[1], d)), __dmul_rn(__dmul_rn(v[2], d), d)));
    else
        return 0.0;
}

template <int KIND, int SPT>
__device__ __forceinline__ void f64_step_body(const F64Step& a, const TileDesc td, const ChainDesc& ch, double* smem)
{
    using V = F64Site<KIND>;
    constexpr int NN = V::n_nodes, NL = V::n_loop;
    const int NT = blockDim.x;
    const int tid = threadIdx.x;
    const int W = NT * SPT;          // room for active sites
    const int32_t L = ch.L;
    const int K = a.K;
    const int owned = min(a.w_own, L - td.start);
    const int active = owned + 2 * (K - 1);
    const int64_t first = static_cast<int64_t>(td.start) - (K - 1);   // site of window position 0

    double* s_u = smem;                                     // [2][W + 2]: positions -1 .. W
    double* s_p = s_u + 2 * (W + 2);                        // nodes [NN][W]
    int32_t* s_cell = reinterpret_cast<int32_t*>(s_p + static_cast<size_t>(a.n_nodes) * W);   // cell of the nodes
    uint16_t* s_q = reinterpret_cast<uint16_t*>(s_cell + W);
    __shared__ int s_count[3];
    if (tid < 3)
        s_count[tid] = 0;

    auto site_of = [&](int x) -> int32_t {
        const int64_t g = first + x;
        return (g >= 0 && g < L) ? static_cast<int32_t>(g) : wrap_site(g, L);
    };

    double u[SPT], cell[SPT], v[SPT][NL > 0 ? NL : 1];
    int32_t n0[SPT];
#pragma unroll
    for (int r = 0; r < SPT; ++r) {
        const int x = tid + r * NT;
        if (x < active) {
            const int64_t p = ch.offset + site_of(x);
            u[r] = a.u_in[p];
            if constexpr (NN > 0) {
                n0[r] = a.in.ncache[p];
                cell[r] = static_cast<double>(n0[r]);
                s_cell[x] = n0[r];
                double nodes[NN];
#pragma unroll
                for (int c = 0; c < NN; ++c) {
                    nodes[c] = a.in.c[c][p];
                    s_p[c * W + x] = nodes[c];
                }
                loop_values<KIND>(nodes, v[r]);
            }
        }
    }
    if (tid < 2) {   // the window's outer neighbours, as they are at the start
        const int x = tid == 0 ? -1 : active;
        const double un = a.u_in[ch.offset + site_of(x)];
        s_u[x + 1] = un;
        s_u[(W + 2) + x + 1] = un;
    }
    __syncthreads();   // (the request counters)

    for (int k = 0;; ++k) {
        double* now = s_u + (k & 1) * (W + 2) + 1;
        double d[SPT];
        bool moved[SPT];
#pragma unroll
        for (int r = 0; r < SPT; ++r) {
            const int x = tid + r * NT;
            moved[r] = false;
            if (x < active) {
                now[x] = u[r];
                if constexpr (NN > 0) {
                    d[r] = __dsub_rn(u[r], cell[r]);
                    moved[r] = static_cast<unsigned>(__double2hiint(d[r])) >= 0x3FF00000u;   // not in [0, 1)
                    if (moved[r])
                        s_q[atomicAdd(&s_count[k % 3], 1)] = static_cast<uint16_t>(x);
                }
            }
        }
        __syncthreads();
        if constexpr (NN > 0) {
            const int nq = s_count[k % 3];
            if (tid == 0)
                s_count[(k + 2) % 3] = 0;   // last read in step k - 1, next used in step k + 2
            if (nq > 0) {
                for (int q = tid; q < nq; q += NT) {
                    const int x = s_q[q];
                    const int32_t n = __double2int_rd(now[x]);
                    const int32_t move = n - s_cell[x];
                    if (move != 0) {   // 0: u - floor rounded up to 1
                        double p[NN];
                        const int shift = (move == 1 || move == -1) ? move : NN;
                        if (shift == 1) {
#pragma unroll
                            for (int c = 0; c + 1 < NN; ++c)
                                p[c] = s_p[(c + 1) * W + x];
                        } else if (shift == -1) {
#pragma unroll
                            for (int c = 1; c < NN; ++c)
                                p[c] = s_p[(c - 1) * W + x];
                        }
                        const int32_t i = site_of(x);
                        const int trips = (shift == NN) ? NN : 1;
#pragma unroll 1
                        for (int j = 0; j < trips; ++j) {
                            const int c = (shift == 1) ? NN - 1 : j;
                            const double w = node_f64<KIND>(a.seed, ch.s, i, n + V::lo + c, ch.period);
#pragma unroll
                            for (int cc = 0; cc < NN; ++cc)
                                if (cc == c)
                                    p[cc] = w;
                        }
#pragma unroll
                        for (int c = 0; c < NN; ++c)
                            s_p[c * W + x] = p[c];
                        s_cell[x] = n;
                    }
                }
                __syncthreads();
#pragma unroll
                for (int r = 0; r < SPT; ++r) {
                    if (moved[r]) {
                        const int x = tid + r * NT;
                        double p[NN];
#pragma unroll
                        for (int c = 0; c < NN; ++c)
                            p[c] = s_p[c * W + x];
                        loop_values<KIND>(p, v[r]);
                        cell[r] = static_cast<double>(s_cell[x]);
                        d[r] = __dsub_rn(u[r], cell[r]);
                    }
                }
            }
        }
        if (k == K)
            break;
#pragma unroll
        for (int r = 0; r < SPT; ++r) {
            const int x = tid + r * NT;
            if (x < active) {
                const double lap = __fma_rn(-2.0, u[r], __dadd_rn(now[x + 1], now[x - 1]));   // 2 u is exact
                u[r] = __dadd_rn(u[r], __dmul_rn(a.dt, __dadd_rn(__dadd_rn(lap, ch.f64), force_f64<KIND>(d[r], v[r]))));
            }
        }
    }
#pragma unroll
    for (int r = 0; r < SPT; ++r) {
        const int x = tid + r * NT;
        const int o = x - (K - 1);
        if (x < active && o >= 0 && o < owned) {
            const int64_t p = ch.offset + td.start + o;
            a.u_out[p] = u[r];
            if constexpr (NN > 0) {
                const int32_t n = s_cell[x];
                if (a.out.ncache != a.in.ncache || n != n0[r]) {
                    a.out.ncache[p] = n;
#pragma unroll
                    for (int c = 0; c < NN; ++c)
                        a.out.c[c][p] = s_p[c * W + x];
                }
            }
        }
    }
}

// Per block tile: sum F, sum (u - c), sum (u - c)^2 of the current state u_in, c the chain's
// reference shift.  (The cached cell is floor(u) between launches.)
template <int KIND>
__device__ __forceinline__ void f64_observe_body(const F64Launch& a, double (*red)[256 / 32])
{
    using V = F64Site<KIND>;
    const TileDesc td = a.tiles[blockIdx.x];
    const ChainDesc ch = a.chains[td.chain];
    const double c = a.shift[td.chain];
    const int used = a.look ? V::used(ch.f64 < 0.0) : 0;
    double tF = 0.0, t1 = 0.0, t2 = 0.0;
    for (int x = threadIdx.x; x < a.w_tile; x += blockDim.x) {
        const int32_t i = td.start + x;
        if (i >= ch.L)
            break;
        const int64_t p = ch.offset + i;
        const double u = a.u_in[p];
        if constexpr (V::n_nodes > 0) {
            double nodes[V::n_nodes], v[V::n_loop];
#pragma unroll
            for (int k = 0; k < V::n_nodes; ++k)
                nodes[k] = a.st.c[used + k][p];
            loop_values<KIND>(nodes, v);
            tF = __dadd_rn(tF, force_f64<KIND>(__dsub_rn(u, static_cast<double>(a.st.ncache[p])), v));
        }
        const double y = __dsub_rn(u, c);
        t1 = __dadd_rn(t1, y);
        t2 = __dadd_rn(t2, __dmul_rn(y, y));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        tF += __shfl_down_sync(0xffffffffu, tF, o);
        t1 += __shfl_down_sync(0xffffffffu, t1, o);
        t2 += __shfl_down_sync(0xffffffffu, t2, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][warp] = tF;
        red[1][warp] = t1;
        red[2][warp] = t2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sF = 0.0, s1 = 0.0, s2 = 0.0;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) {
            sF += red[0][w];
            s1 += red[1][w];
            s2 += red[2][w];
        }
        double* dst = a.partial + static_cast<size_t>(blockIdx.x) * 4;
        dst[0] = sF;
        dst[1] = s1;
        dst[2] = s2;
        dst[3] = c;
    }
}

template <int KIND>
__device__ __forceinline__ void init_nodes(const F64State& st, int64_t p, uint64_t seed, uint32_t s, int32_t i, int32_t n,
                                           int32_t period, int look, bool neg)
{
    using V = F64Site<KIND>;
    const int count = look ? V::n_look : V::n_nodes;
    const int lo = V::lo - (look ? V::used(neg) : 0);
#pragma unroll 1
    for (int c = 0; c < count; ++c)
        st.c[c][p] = node_f64<KIND>(seed, s, i, n + lo + c, period);
}

__global__ void f64_init_kernel(const ChainDesc* chains, const TileDesc* tiles, int32_t w_tile, F64State st,
                                uint64_t seed, const double* u_in, int look)
{
    const TileDesc td = tiles[blockIdx.x];
    const ChainDesc ch = chains[td.chain];
    for (int x = threadIdx.x; x < w_tile; x += blockDim.x) {
        const int32_t i = td.start + x;
        if (i >= ch.L)
            break;
        const int64_t p = ch.offset + i;
        const double u = u_in ? u_in[p] : 0.0;
        st.u[p] = u;
        const int32_t n = static_cast<int32_t>(floor(u));
        st.ncache[p] = n;
        const int32_t M = ch.period;
        if (ch.kind == kRF)
            init_nodes<kRF>(st, p, seed, ch.s, i, n, M, look, ch.f64 < 0.0);
        else if (ch.kind == kRBGLinear)
            init_nodes<kRBGLinear>(st, p, seed, ch.s, i, n, M, look, ch.f64 < 0.0);
        else if (ch.kind == kRB)
            init_nodes<kRB>(st, p, seed, ch.s, i, n, M, look, ch.f64 < 0.0);
        else if (ch.kind == kRBGCubic)
            init_nodes<kRBGCubic>(st, p, seed, ch.s, i, n, M, look, ch.f64 < 0.0);
    }
}

__global__ void f64_cells_kernel(const ChainDesc* chains, const TileDesc* tiles, int32_t w_tile, const double* u,
                                 int32_t* cells_out)
{
    const TileDesc td = tiles[blockIdx.x];
    const ChainDesc ch = chains[td.chain];
    for (int x = threadIdx.x; x < w_tile; x += blockDim.x) {
        const int32_t i = td.start + x;
        if (i >= ch.L)
            break;
        const int64_t p = ch.offset + i;
        cells_out[p] = static_cast<int32_t>(floor(u[p]));
    }
}

// The same for few sites (one per thread), where a draw is 5500 clocks of waiting and a step 900: each
// site holds the next node it will need, so a move up only shifts its nodes and lists the site; the
// listed sites' missing nodes are drawn together once a warp of them has gathered, or at once when a
// force needs one.  One 1024-site RF chain at f = 1, us per step: 22.7 with one launch per step on one
// SM, 3.3 in small tiles with every draw in its own step, 1.47 so, 1.38 with the draws split in two.
template <int KIND, bool NEG>
__device__ __forceinline__ void f64_look_body(const F64Step& a, const TileDesc td, const ChainDesc& ch, double* smem)
{
    using V = F64Site<KIND>;
    constexpr int NN = V::n_nodes, NX = V::n_look, NL = V::n_loop, used = V::used(NEG), lo_look = V::lo - used;
    const int NT = blockDim.x;
    // (the linear spline's sites keep listing outer nodes that they may never use: us per step at 1024,
    // 2^16 and 2^18 sites 2.84, 5.43, 19.4 gathering a quarter as for the others, 2.29, 5.12, 18.2 so)
    const int gather = KIND == kRBGLinear ? NT / 2 : max(32, NT / 4);
    const int x = threadIdx.x;
    const int32_t L = ch.L;
    const int K = a.K;
    const int owned = min(a.w_own, L - td.start);
    const int active = owned + 2 * (K - 1);
    const int64_t first = static_cast<int64_t>(td.start) - (K - 1);   // site of window position 0

    double* s_u = smem;                                     // [2][NT + 2]: positions -1 .. NT
    double* s_p = s_u + 2 * (NT + 2);                       // nodes [NX][NT]
    double* s_f = s_p + static_cast<size_t>(a.n_nodes) * NT;   // [2][NX][NT / 2]: factors being drawn
    int32_t* s_cell = reinterpret_cast<int32_t*>(s_f + static_cast<size_t>(a.n_nodes) * NT);
    uint16_t* s_q = reinterpret_cast<uint16_t*>(s_cell + NT);
    __shared__ int s_count[2];   // listed sites; the two take turns
    if (x < 2)
        s_count[x] = 0;

    auto site_of = [&](int at) -> int32_t {
        const int64_t g = first + at;
        return (g >= 0 && g < L) ? static_cast<int32_t>(g) : wrap_site(g, L);
    };
    const bool mine = x < active;
    double u = 0.0, cell = 0.0, d = 0.0, v[NL > 0 ? NL : 1];
    int32_t n = 0;
    bool missing = false;
    if (mine) {
        const int64_t p = ch.offset + site_of(x);
        u = a.u_in[p];
        if constexpr (NX > 0) {
            n = a.in.ncache[p];
            cell = static_cast<double>(n);
            s_cell[x] = n;
            double nodes[NX];
#pragma unroll
            for (int c = 0; c < NX; ++c) {
                nodes[c] = a.in.c[c][p];
                s_p[c * NT + x] = nodes[c];
                missing = missing || no_node(nodes[c]);
            }
            loop_values<KIND>(nodes + used, v);
        }
    }
    if (x < 2) {   // the window's outer neighbours, as they are at the start
        const int at = x == 0 ? -1 : active;
        const double un = a.u_in[ch.offset + site_of(at)];
        s_u[at + 1] = un;
        s_u[(NT + 2) + at + 1] = un;
    }
    __syncthreads();
    int turn = 0, slot = -1;
    if (missing) {
        slot = atomicAdd(&s_count[0], 1);
        s_q[slot] = static_cast<uint16_t>(x);
    }

    for (int k = 0;; ++k) {
        double* now = s_u + (k & 1) * (NT + 2) + 1;
        if constexpr (NX > 0) {
            bool urgent = false;
            if (mine) {
                now[x] = u;
                d = __dsub_rn(u, cell);
                const unsigned h = static_cast<unsigned>(__double2hiint(d));
                if (h >= 0x3FF00000u) {   // not in [0, 1)
                    // (1, 2) is one cell up and (-1, 0) one down, exactly; else the floor decides (u - floor
                    // may have rounded up to 1; -0 is in cell 0)
                    const bool edge = (h == 0x3FF00000u || h == 0x80000000u) && __double2loint(d) == 0;   // 1 or -0
                    int32_t move;
                    if (h < 0x40000000u && !edge)
                        move = 1;
                    else if (h >= 0x80000000u && h < 0xBFF00000u && !edge)
                        move = -1;
                    else
                        move = __double2int_rd(u) - n;
                    if (move != 0) {
                        n += move;
                        cell = static_cast<double>(n);
                        d = __dsub_rn(u, cell);
                        const double none = __hiloint2double(kNoNode, 0);
                        double nodes[NX];
#pragma unroll
                        for (int c = 0; c < NX; ++c) {
                            nodes[c] = none;
                            if (move == 1 && c + 1 < NX)
                                nodes[c] = s_p[(c + 1) * NT + x];
                            if (move == -1 && c > 0)
                                nodes[c] = s_p[(c - 1) * NT + x];
                        }
#pragma unroll
                        for (int c = 0; c < NX; ++c) {
                            s_p[c * NT + x] = nodes[c];
                            if (c >= used && c < used + NN)
                                urgent = urgent || no_node(nodes[c]);
                        }
                        s_cell[x] = n;
                        loop_values<KIND>(nodes + used, v);
                        if (slot < 0) {
                            slot = atomicAdd(&s_count[turn], 1);
                            s_q[slot] = static_cast<uint16_t>(x);
                        }
                    }
                }
            }
            if (__syncthreads_or(urgent || slot >= gather - 1)) {
                const int listed = s_count[turn];
                // A Gaussian value is a radius times an angle's cosine: for up to half as many sites as
                // threads, the first half of the threads draws the radii and the second the cosines, on
                // other warps, in 50 and 30 serial operations instead of 80.
                const int half = NT / 2;
                const bool split = KIND != kRB && listed <= half;
                const int part = split && x >= half ? 1 : 0;
                if (split) {
                    const int q = x - part * half;
                    if (q < listed) {
                        const int at = s_q[q];
                        const int32_t i = site_of(at), base = s_cell[at] + lo_look;
#pragma unroll 1
                        for (int c = 0; c < NX; ++c) {
                            if (!no_node(s_p[c * NT + at]))
                                continue;
                            const uint4 w = disorder_words(a.seed, ch.s, i, wrap_node(base + c, ch.period), KIND == kRF ? kTagRF : kTagRBG);
                            s_f[part * NX * half + c * half + q] = part ? gauss_angle_f64(w) : gauss_radius_f64(w);
                        }
                    }
                    __syncthreads();
                    if (x < listed) {
                        const int at = s_q[x];
#pragma unroll
                        for (int c = 0; c < NX; ++c)
                            if (no_node(s_p[c * NT + at]))
                                s_p[c * NT + at] = __dmul_rn(s_f[c * half + x], s_f[(NX + c) * half + x]);
                    }
                } else {
                    // In a crowded round a site that lost all of its force's nodes (a move of several cells)
                    // draws only those, and is listed again for the others: a steep line, whose sites move so
                    // in every step, would never use them (2^20 sites, 16 steps: random field 8.6 ms, Case 3
                    // 10.5, with all drawn, 7.3 and 7.7 so).
                    for (int q = x; q < listed; q += NT) {
                        const int at = s_q[q];
                        const int32_t i = site_of(at), base = s_cell[at] + lo_look;
                        const bool lost = no_node(s_p[used * NT + at]) && no_node(s_p[(used + NN - 1) * NT + at]);
#pragma unroll 1
                        for (int c = lost ? used : 0; c < (lost ? used + NN : NX); ++c)
                            if (no_node(s_p[c * NT + at]))
                                s_p[c * NT + at] = node_f64<KIND>(a.seed, ch.s, i, base + c, ch.period);
                    }
                }
                turn ^= 1;
                slot = -1;
                if (x == 0)
                    s_count[turn] = 0;   // last read a gathering ago
                __syncthreads();
                if (urgent) {
                    double nodes[NN];
#pragma unroll
                    for (int c = 0; c < NN; ++c)
                        nodes[c] = s_p[(used + c) * NT + x];
                    loop_values<KIND>(nodes, v);
                    if (!split && no_node(s_p[(NEG ? 0 : NX - 1) * NT + x])) {
                        slot = atomicAdd(&s_count[turn], 1);
                        s_q[slot] = static_cast<uint16_t>(x);
                    }
                }
            }
        } else {
            if (mine)
                now[x] = u;
            __syncthreads();
        }
        if (k == K)
            break;
        if (mine) {
            const double lap = __fma_rn(-2.0, u, __dadd_rn(now[x + 1], now[x - 1]));   // 2 u is exact
            u = __dadd_rn(u, __dmul_rn(a.dt, __dadd_rn(__dadd_rn(lap, ch.f64), force_f64<KIND>(d, v))));
        }
    }
    const int o = x - (K - 1);
    if (mine && o >= 0 && o < owned) {
        const int64_t p = ch.offset + td.start + o;
        a.u_out[p] = u;
        if constexpr (NX > 0) {
            a.out.ncache[p] = n;
#pragma unroll
            for (int c = 0; c < NX; ++c)
                a.out.c[c][p] = s_p[c * NT + x];
        }
    }
}

__global__ void __launch_bounds__(256, 1) f64_look_any(F64Step a)
{
    extern __shared__ double smem_f64[];
    const TileDesc td = a.tiles[blockIdx.x];
    const ChainDesc ch = a.chains[td.chain];
    const bool neg = ch.f64 < 0.0;
    if (ch.kind == kRF)
        neg ? f64_look_body<kRF, true>(a, td, ch, smem_f64) : f64_look_body<kRF, false>(a, td, ch, smem_f64);
    else if (ch.kind == kRB)
        neg ? f64_look_body<kRB, true>(a, td, ch, smem_f64) : f64_look_body<kRB, false>(a, td, ch, smem_f64);
    else if (ch.kind == kRBGLinear)
        f64_look_body<kRBGLinear, false>(a, td, ch, smem_f64);
    else if (ch.kind == kRBGCubic)
        neg ? f64_look_body<kRBGCubic, true>(a, td, ch, smem_f64) : f64_look_body<kRBGCubic, false>(a, td, ch, smem_f64);
    else
        f64_look_body<kNone, false>(a, td, ch, smem_f64);
}

// Tiles of mixed kinds share one launch: the kind is uniform per block (one chain).
template <int SPT>
__global__ void __launch_bounds__(256, 1) f64_step_any(F64Step a)
{
    extern __shared__ double smem_f64[];
    const TileDesc td = a.tiles[blockIdx.x];
    const ChainDesc ch = a.chains[td.chain];
    if (ch.kind == kRF)
        f64_step_body<kRF, SPT>(a, td, ch, smem_f64);
    else if (ch.kind == kRB)
        f64_step_body<kRB, SPT>(a, td, ch, smem_f64);
    else if (ch.kind == kRBGLinear)
        f64_step_body<kRBGLinear, SPT>(a, td, ch, smem_f64);
    else if (ch.kind == kRBGCubic)
        f64_step_body<kRBGCubic, SPT>(a, td, ch, smem_f64);
    else
        f64_step_body<kNone, SPT>(a, td, ch, smem_f64);
}

__global__ void __launch_bounds__(256) f64_observe_any(F64Launch a)
{
    __shared__ double red[3][256 / 32];
    const int kind = a.chains[a.tiles[blockIdx.x].chain].kind;
    if (kind == kRF)
        f64_observe_body<kRF>(a, red);
    else if (kind == kRB)
        f64_observe_body<kRB>(a, red);
    else if (kind == kRBGLinear)
        f64_observe_body<kRBGLinear>(a, red);
    else if (kind == kRBGCubic)
        f64_observe_body<kRBGCubic>(a, red);
    else
        f64_observe_body<kNone>(a, red);
}

}  // namespace

size_t f64_step_smem(const F64Shape& s, int n_nodes)
{
    const size_t W = static_cast<size_t>(s.threads) * s.sites_per_thread;
    return 8 * (2 * (W + 2) + n_nodes * W) + 4 * W + 2 * W;
}

// Shape by the number of sites, each line where the next shape measured faster (RF, us per step):
//   1024 sites    128 threads x 32 steps with look-ahead 1.47, x 16 steps 1.60, without look-ahead 4.9
//   2^16 sites    256 x 16 with look-ahead 3.0, 128 x 16 3.6, 128 x 32 5.3, without 5.1
//   2^19 sites    256 x 16 with look-ahead 21.0, without 25.7
//   2^24 sites    128 threads of 4 sites x 8 steps without look-ahead 651 (Case 3 on half of them 367, against
//                 550 with look-ahead, whose outer nodes its moves up and down keep discarding), 4 steps 669
// Few sites are latency: 65 clocks per FP64 operation whatever a block does, so small tiles on as many
// SMs as there are.  Then it is FP64 throughput, where a wide halo is work done twice.  A batch of uniform
// random-bond chains alone, whose draws are a few operations, gives up look-ahead at 3 x 2^18 sites (us per
// step with it and without, at f_c, 3 f_c and from a steep line: 2^19 sites 33.3 34.0, 39.4 35.8, 80 54; 2^20
// sites 63.2 59.0, 75.2 69.1, 151 98).  One step per launch
// updates the cached disorder in place and takes no second copy of it, for batches beyond 2^29 sites (30 GB
// with it for RF, 47 GB for the cubic kinds); at 2^27 RF sites it runs 9.1 ms per step against 5.2.
F64Shape f64_shape(int64_t n_sites, int kinds_mask)
{
    if (n_sites <= (int64_t(1) << 13))
        return F64Shape{128, 1, 32, true};
    if (n_sites <= (int64_t(1) << 15))
        return F64Shape{128, 1, 16, true};
    if (n_sites <= (int64_t(1) << 20) && (kinds_mask != 1 << kRB || n_sites < (int64_t(3) << 18)))
        return F64Shape{256, 1, 16, true};
    if (n_sites <= (int64_t(1) << 29))
        return F64Shape{128, 4, 8, false};
    return F64Shape{256, 4, 1, false};
}

template <int SPT>
static cudaError_t f64_step_as(const F64Step& a, const F64Shape& s, cudaStream_t st)
{
    const size_t smem = f64_step_smem(s, a.n_nodes);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(f64_step_any<SPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
        if (e != cudaSuccess)
            return e;
    }
    f64_step_any<SPT><<<a.n_tiles, s.threads, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t f64_step(const F64Step& a, const F64Shape& s, cudaStream_t st)
{
    if (a.n_tiles == 0)
        return cudaSuccess;
    if (!s.look)
        return f64_step_as<4>(a, s, st);
    f64_look_any<<<a.n_tiles, s.threads, f64_step_smem(s, 2 * a.n_nodes), st>>>(a);
    return cudaGetLastError();
}

cudaError_t f64_observe(const F64Launch& a, cudaStream_t st)
{
    if (a.n_tiles == 0)
        return cudaSuccess;
    f64_observe_any<<<a.n_tiles, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t f64_init(const ChainDesc* chains, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile, F64State st,
                     uint64_t seed, int look, const double* u_in, cudaStream_t stream)
{
    if (n_tiles == 0)
        return cudaSuccess;
    f64_init_kernel<<<n_tiles, 256, 0, stream>>>(chains, tiles, w_tile, st, seed, u_in, look);
    return cudaGetLastError();
}

cudaError_t f64_cells(const ChainDesc* chains, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile,
                      const double* u, int32_t* cells_out, cudaStream_t stream)
{
    if (n_tiles == 0)
        return cudaSuccess;
    f64_cells_kernel<<<n_tiles, 256, 0, stream>>>(chains, tiles, w_tile, u, cells_out);
    return cudaGetLastError();
}

}  // namespace qew
