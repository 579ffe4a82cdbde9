// qew_sq.cu -- the structure factor of Eq. 6 (Sec. II of arXiv:1211.7275):
//     S_q = mean over chains of |(1/L) sum_x u(x) e^{-iqx}|^2,  q = 2 pi n / L,  n = 1 .. L/2.
// The line is written as FP64 rows, transformed by cuFFT, and the mode powers are averaged over the
// chains, in a fixed order.  For even L (from 4) a row is read as L/2 complex numbers (even sites real, odd sites
// imaginary), transformed at half the length, and the two modes k and L/2 - k are separated where their
// powers are taken (sq_power_half_kernel): the transform of a real row is never written.  Odd L: a
// real-to-complex transform of rows of 2 (L/2 + 1) values.
#include "qew_internal.h"

namespace qew {
namespace {

// Row c holds u(x) - c0 for chain c, where c0 is the cell (FP32-split) or the floor (FP64) of
// site 0: the shift leaves every mode n >= 1 unchanged and keeps the values small, so the
// transform's rounding error stays at the scale of the line's width, not of its position.
__global__ void sq_rows_split_kernel(const ChainDesc* chains, int32_t n_chains, SplitState st, int32_t L, int64_t P,
                                     double* rows)
{
    for (int c = blockIdx.y; c < n_chains; c += gridDim.y) {
        const ChainDesc ch = chains[c];
        const int32_t c0 = st.cell[ch.offset];
        double* row = rows + static_cast<int64_t>(c) * P;
        for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < L;
             i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
            const int64_t p = ch.offset + i;
            row[i] = static_cast<double>(st.cell[p] - c0) + static_cast<double>(fabsf(st.off[p]));   // exact
        }
    }
}

__global__ void sq_rows_f64_kernel(const ChainDesc* chains, int32_t n_chains, const double* u, int32_t L, int64_t P,
                                   double* rows)
{
    for (int c = blockIdx.y; c < n_chains; c += gridDim.y) {
        const ChainDesc ch = chains[c];
        const double c0 = floor(u[ch.offset]);
        double* row = rows + static_cast<int64_t>(c) * P;
        for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < L;
             i += static_cast<int64_t>(gridDim.x) * blockDim.x)
            row[i] = u[ch.offset + i] - c0;
    }
}

// S[k] = scale * sum over chains c (in order) of |Z_c(k + 1)|^2, k < n_modes.  One thread per
// mode: a warp reads 32 consecutive complex values of a row, coalesced.
__global__ void sq_power_kernel(const double2* Z, int64_t Pz, int32_t n_chains, int32_t n_modes, double scale,
                                double* S)
{
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < n_modes;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double acc = 0.0;
        for (int c = 0; c < n_chains; ++c) {
            const double2 z = Z[static_cast<int64_t>(c) * Pz + k + 1];
            acc = fma(z.x, z.x, fma(z.y, z.y, acc));
        }
        S[k] = acc * scale;
    }
}

// The same from the half-length transforms Z of rows z(j) = u(2j) + i u(2j + 1), M = L/2: with
// E = (Z(k) + Z*(M-k)) / 2 and O = -i (Z(k) - Z*(M-k)) / 2 the mode is X(k) = E + e^{-2 pi i k / L} O, and
// X(M-k) is the conjugate of E - e^{-2 pi i k / L} O; X(M) = Re Z(0) - Im Z(0).  One thread per pair
// (k, M - k), all chains: the factor is computed once per pair.  Bound by FP64 arithmetic, some 20
// operations per pair and chain; 16 x 2^20: 344 us before, as cuFFT's separation pass and the power of
// its output.
__global__ void sq_power_half_kernel(const double2* Z, int64_t M, int32_t n_chains, int32_t n_modes, double scale, double* S)
{
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; 2 * k <= M;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        if (k == 0) {
            if (n_modes < M)
                continue;
            double acc = 0.0;
            for (int c = 0; c < n_chains; ++c) {
                const double2 z = Z[static_cast<int64_t>(c) * M];
                const double x = z.x - z.y;
                acc = fma(x, x, acc);
            }
            S[M - 1] = acc * scale;
            continue;
        }
        const int64_t m = M - k;
        if (k > n_modes)   // then m > n_modes as well
            continue;
        double sn, cs;
        sincospi(static_cast<double>(k) / static_cast<double>(M), &sn, &cs);   // e^{-2 pi i k / L} = cs - i sn
        double acc_k = 0.0, acc_m = 0.0;
#pragma unroll 4
        for (int c = 0; c < n_chains; ++c) {
            const double2 a = Z[static_cast<int64_t>(c) * M + k], b = Z[static_cast<int64_t>(c) * M + m];
            const double er = a.x + b.x, ei = a.y - b.y;   // 2 E
            const double pr = a.y + b.y, pi = b.x - a.x;   // 2 O
            const double wr = fma(cs, pr, sn * pi), wi = fma(cs, pi, -(sn * pr));
            const double xr = er + wr, xi = ei + wi, yr = er - wr, yi = ei - wi;
            acc_k = fma(xr, xr, fma(xi, xi, acc_k));
            acc_m = fma(yr, yr, fma(yi, yi, acc_m));
        }
        S[k - 1] = 0.25 * acc_k * scale;
        if (m != k && m <= n_modes)
            S[m - 1] = 0.25 * acc_m * scale;
    }
}

int sq_grid(int64_t n)
{
    const int64_t blocks = (n + 255) / 256;
    return static_cast<int>(blocks < 4 * 152 ? (blocks < 1 ? 1 : blocks) : 4 * 152);
}

}  // namespace

bool sq_half(int32_t L)
{
    return L % 2 == 0 && L >= 4;
}

int64_t sq_row(int32_t L)
{
    return sq_half(L) ? L : 2 * (static_cast<int64_t>(L) / 2 + 1);
}

cudaError_t sq_rows(const ChainDesc* chains, int32_t n_chains, int32_t L, const SplitState* split, const double* u64,
                    double* rows, cudaStream_t stream)
{
    const int64_t P = sq_row(L);
    const dim3 grid(sq_grid(L) / 4 + 1, n_chains < 4096 ? n_chains : 4096);
    if (split)
        sq_rows_split_kernel<<<grid, 256, 0, stream>>>(chains, n_chains, *split, L, P, rows);
    else
        sq_rows_f64_kernel<<<grid, 256, 0, stream>>>(chains, n_chains, u64, L, P, rows);
    return cudaGetLastError();
}

cudaError_t sq_power(const void* Z, int32_t L, int32_t n_chains, int32_t n_modes, double* S, cudaStream_t stream)
{
    const double scale = 1.0 / (static_cast<double>(L) * static_cast<double>(L) * n_chains);
    if (sq_half(L)) {
        const int64_t M = L / 2;
        sq_power_half_kernel<<<sq_grid(M / 2 + 1), 256, 0, stream>>>(static_cast<const double2*>(Z), M, n_chains, n_modes, scale, S);
        return cudaGetLastError();
    }
    const int64_t Pz = static_cast<int64_t>(L) / 2 + 1;
    sq_power_kernel<<<sq_grid(n_modes), 256, 0, stream>>>(static_cast<const double2*>(Z), Pz, n_chains, n_modes,
                                                          scale, S);
    return cudaGetLastError();
}

}  // namespace qew
