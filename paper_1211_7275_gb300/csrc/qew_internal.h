// qew_internal.h -- declarations shared by the translation units of the qEW library (kernel
// launchers and the buffers they work on).  Not part of the public C ABI (include/qew.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include <string>

#include "qew_device.cuh"

namespace qew {

// FP32-split state: cell n (int32), in-cell offset d (float, [0,1)) and the disorder cache
// of each site.  The random field keeps (R(n) + f, R(n+1) + f) in rf.  The linear-spline random bond
// keeps F_p = G - G(+1) of two neighbouring cells in rf, the sign of d saying that the site is in the
// upper one, and in q3 the node beyond them in the direction of the drive; where memory is short q3 is
// NULL and each launch draws that node anew.  The cubic kinds keep the nodes V(n), V(n+1) in qn, V(n+2)
// in q3, and the coefficients of F_p + f = A + d (B + d C) over cell n (from V(n-1) .. V(n+2)) in qab
// (A, B) and qc (C).  A chain of kind NONE uses none of them.
struct SplitState {
    int32_t* cell;
    float* off;
    float2* rf;
    float2* qn;
    float* q3;
    float2* qab;
    float* qc;
};

// FP64 state: displacement u, and the disorder cache of the cell `ncache` it was drawn for:
// RF R(n), R(n+1) in c[0], c[1]; RB V(n-1..n+2) in c[0..3]; with look-ahead (few sites) one node more,
// and for the linear-spline random bond one less as well, not drawn yet where it is a NaN.  Between launches ncache is floor(u).
struct F64State {
    double* u;
    int32_t* ncache;
    double* c[5];
};

// Most observations that one launch of the fused kernel records.
constexpr int kMaxLaunchObs = 24;

struct SplitLaunch {
    const WarpTile* tiles;   // tiles of one class
    int32_t n_tiles;
    int32_t neg;             // the class's drives are negative
    int32_t tile_base;       // partial-sum slot of tiles[0]
    SplitState in, out;
    int32_t K;               // Euler steps in this launch (0: observe only)
    int32_t pad;             // sites of a tile's window before its first owned one (>= K)
    int32_t w_own;           // owned sites per tile
    float dt;
    uint64_t seed;
    int32_t n_obs;           // observations in this launch: per-tile partial sums of the state
    uint16_t obs_at[kMaxLaunchObs];    // after so many of its steps (increasing),
    uint16_t obs_len[kMaxLaunchObs];   // the last so many of which belong to the observation's own segment
    const double* shift;     // per-chain reference cell c of the sums
    double* partial;         // [n_obs][partial_stride][4]: sum F, sum (u - c), sum (u - c)^2, c
    int64_t partial_stride;  // tiles of all kinds
    unsigned long long* crossings;  // if not null: cell crossings are added here
    int32_t* error;          // 1: a bounded wait on a bulk copy gave up; 2: neighbouring cells 2^12 apart
    PhiloxKeys keys;         // round keys of `seed`
};

// Writes the warp tiles of the chains of one class: chain c's, w_own sites each, at tiles[first[c]].
cudaError_t split_tiles(const ChainDesc* chains, int32_t n_chains, int cls, int32_t w_own, const int32_t* first,
                        WarpTile* tiles, cudaStream_t stream);
// Sites per lane of the fused kernel for each supported tile width (tile_w = 32 * S).
bool split_supported(int kind, int sites_per_lane);
size_t split_smem_bytes(int kind, int sites_per_lane, int tiles_per_cta);
int split_warps_per_sm(int kind, int sites_per_lane);   // resident warps (tiles), by registers and shared memory
cudaError_t split_step(int kind, int sites_per_lane, int tiles_per_cta, const SplitLaunch& a, cudaStream_t st);
cudaError_t split_init(const ChainDesc* chains, int32_t n_chains, const TileDesc* tiles, int32_t n_tiles,
                       int32_t w_tile, SplitState st, uint64_t seed, int any_rb, const double* u_in,
                       cudaStream_t stream);
cudaError_t split_to_f64(const ChainDesc* chains, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile,
                         SplitState st, double* u_out, int32_t* cells_out, cudaStream_t stream);
// Sets *error to 2 if neighbouring cells of the FP32-split state differ by 2^12 or more (the range
// in which the fused kernel's cell arithmetic is exact); max_L is the longest chain.
cudaError_t split_range_guard(const ChainDesc* chains, int32_t n_chains, int64_t max_L, const int32_t* cell,
                              int32_t* error, cudaStream_t stream);

struct F64Launch {           // an observation
    const TileDesc* tiles;   // block tiles of w_tile sites
    int32_t n_tiles;
    int32_t w_tile;
    const ChainDesc* chains;
    F64State st;
    int32_t look;            // the caches hold look-ahead nodes
    const double* u_in;
    const double* shift;
    double* partial;
};

// Launch shape of the FP64 step kernel: a block of `threads` threads with `sites_per_thread` sites each
// advances up to K steps.
struct F64Shape {
    int threads, sites_per_thread, K;
    bool look;   // sites hold the nodes their next move will need (one site per thread)
    int w_own() const { return threads * sites_per_thread - 2 * (K - 1); }
};

struct F64Step {
    const TileDesc* tiles;   // tiles of w_own sites
    int32_t n_tiles;
    int32_t w_own;
    int32_t K;               // steps in this launch, up to the shape's
    int32_t n_nodes;         // nodes per site of the batch's largest cache (room in shared memory)
    const ChainDesc* chains;
    const double* u_in;
    double* u_out;
    F64State in, out;        // disorder caches (the same arrays for in place: K = 1 only)
    double dt;
    uint64_t seed;
};

F64Shape f64_shape(int64_t n_sites, int kinds_mask);
size_t f64_step_smem(const F64Shape& s, int n_nodes);
cudaError_t f64_step(const F64Step& a, const F64Shape& s, cudaStream_t st);
cudaError_t f64_observe(const F64Launch& a, cudaStream_t st);
cudaError_t f64_init(const ChainDesc* chains, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile,
                     F64State st, uint64_t seed, int look, const double* u_in, cudaStream_t stream);
cudaError_t f64_cells(const ChainDesc* chains, const TileDesc* tiles, int32_t n_tiles, int32_t w_tile,
                      const double* u, int32_t* cells_out, cudaStream_t stream);

// Second pass of n_obs observations: per chain, sum the partials of its tiles in a fixed order, record
// (sum F, S1, S2, c) into obs[index[k]][chain] and move the chain's reference c to the centre of mass at
// the last of them (rounded to an integer cell).
struct ObsList {
    int32_t n;
    int32_t index[kMaxLaunchObs];
};
cudaError_t reduce_chains(const ChainDesc* chains, int32_t n_chains, const double* partial, int64_t partial_stride,
                          double* shift, double* obs, const ObsList& list, cudaStream_t stream);

// Structure factor (Eq. 6): rows of u(x) - c0 per chain, sq_row(L) doubles apart (with sq_half(L), L of them,
// read as L/2 complex numbers; else the padded layout of an in-place real-to-complex FFT), from the split state
// (split != NULL) or the FP64 state; then, from the transforms, the mean over chains of |Z(n)|^2 / L^2 for
// n = 1 .. n_modes.
bool sq_half(int32_t L);
int64_t sq_row(int32_t L);
cudaError_t sq_rows(const ChainDesc* chains, int32_t n_chains, int32_t L, const SplitState* split, const double* u64,
                    double* rows, cudaStream_t stream);
cudaError_t sq_power(const void* Z, int32_t L, int32_t n_chains, int32_t n_modes, double* S, cudaStream_t stream);

// Message returned by qew_last_error(NULL) for calls without a handle (this thread).
void set_last_error(const std::string& msg);

// Launch one warp whose mbarrier wait cannot complete; it sets *d_error after spin_limit polls.
cudaError_t bounded_wait_selftest(int32_t* d_error, int spin_limit, cudaStream_t stream);

cudaError_t philox_words(const uint32_t* ctr, const uint32_t* key, int64_t n_blocks, uint32_t* out,
                         cudaStream_t stream);
cudaError_t disorder_values(int kind, int fp64, uint64_t seed, uint32_t s, const int64_t* i, const int64_t* n,
                            int64_t count, double* out, cudaStream_t stream);

}  // namespace qew
