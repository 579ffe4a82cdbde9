// A stand-in for the CUDA runtime, the kernels' launchers and cuFFT, for tests of the library's host
// code (csrc/qew_capi.cu) without a device.  Device memory is addresses that nothing stands behind; a
// test sets how much of it there is, or which of the next allocations fails.  The launchers run nothing:
// they check that every array that their kernel reads or writes has an address, which is what decides on
// a device between a result and a memory fault, and count the launches that would have none.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include <cuda_runtime.h>
#include <cufft.h>

#include "qew_internal.h"

namespace {

std::map<uintptr_t, size_t> live;
uintptr_t next_address = uintptr_t(1) << 44;
size_t held = 0, peak = 0, capacity = ~size_t(0);
int64_t until_failure = -1;   // allocations until one fails (-1: none does)
int64_t launches = 0, bad = 0;
std::string first_bad;
int64_t off_stream = 0;       // copies and fills that other work does not wait for
int32_t last_K = 0, last_in_place = 0, last_n_obs = 0, max_n_obs = 0, last_has_q3 = 0;

void need(const void* p, const char* what)
{
    if (!p) {
        ++bad;
        if (first_bad.empty())
            first_bad = what;
    }
}

void on_stream(cudaStream_t)
{
    ++launches;
}

void split_arrays(const qew::SplitState& s, int kind, const char* what)
{
    need(s.cell, what);
    need(s.off, what);
    if (qew::pair_kind(kind))
        need(s.rf, what);
    if (qew::quad_kind(kind)) {
        need(s.qn, what);
        need(s.q3, what);
        need(s.qab, what);
        need(s.qc, what);
    }
}

}  // namespace

extern "C" {

void fake_reset()
{
    until_failure = -1;
    capacity = ~size_t(0);
    peak = held;
    launches = bad = off_stream = 0;
    max_n_obs = 0;
    first_bad.clear();
}
void fake_fail_after(int64_t allocations) { until_failure = allocations; }
void fake_capacity(size_t bytes) { capacity = bytes; }
size_t fake_held() { return held; }
size_t fake_peak() { return peak; }
int64_t fake_launches() { return launches; }
int64_t fake_bad() { return bad; }
const char* fake_first_bad() { return first_bad.c_str(); }
int64_t fake_off_stream() { return off_stream; }
int32_t fake_last_K() { return last_K; }
int32_t fake_last_in_place() { return last_in_place; }
int32_t fake_max_n_obs() { return max_n_obs; }
int32_t fake_last_has_q3() { return last_has_q3; }

cudaError_t __wrap_cudaMalloc(void** p, size_t size)
{
    *p = nullptr;
    if (until_failure >= 0 && until_failure-- == 0)
        return cudaErrorMemoryAllocation;
    if (held + size > capacity)
        return cudaErrorMemoryAllocation;
    *p = reinterpret_cast<void*>(next_address);
    live[next_address] = size;
    next_address += (size + 511) & ~size_t(511);
    held += size;
    peak = held > peak ? held : peak;
    return cudaSuccess;
}
cudaError_t __wrap_cudaFree(void* p)
{
    auto it = live.find(reinterpret_cast<uintptr_t>(p));
    if (it != live.end()) {
        held -= it->second;
        live.erase(it);
    }
    return cudaSuccess;
}
cudaError_t __wrap_cudaMallocHost(void** p, size_t size) { return (*p = std::calloc(1, size)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t __wrap_cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }

static cudaError_t copy(void* dst, const void* src, size_t size, cudaMemcpyKind kind)
{
    need(dst, "copy to");
    need(src, "copy from");
    if (kind == cudaMemcpyDeviceToHost && dst)
        std::memset(dst, 0, size);
    return cudaSuccess;
}
// (the legacy default stream does not order itself with a non-blocking one: only copies to the host,
// which the host has waited for the stream before, may go there)
cudaError_t __wrap_cudaMemcpy(void* dst, const void* src, size_t size, cudaMemcpyKind kind)
{
    off_stream += kind != cudaMemcpyDeviceToHost;
    return copy(dst, src, size, kind);
}
cudaError_t __wrap_cudaMemcpyAsync(void* dst, const void* src, size_t size, cudaMemcpyKind kind, cudaStream_t)
{
    return copy(dst, src, size, kind);
}
cudaError_t __wrap_cudaMemset(void* p, int, size_t)
{
    ++off_stream;
    need(p, "fill");
    return cudaSuccess;
}
cudaError_t __wrap_cudaMemsetAsync(void* p, int, size_t, cudaStream_t)
{
    need(p, "fill");
    return cudaSuccess;
}
cudaError_t __wrap_cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t __wrap_cudaSetDevice(int) { return cudaSuccess; }
cudaError_t __wrap_cudaGetLastError() { return cudaSuccess; }
cudaError_t __wrap_cudaPeekAtLastError() { return cudaSuccess; }
const char* __wrap_cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t __wrap_cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(8); return cudaSuccess; }
cudaError_t __wrap_cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t __wrap_cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaErrorNotSupported; }
cudaError_t __wrap_cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t __wrap_cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t __wrap_cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t __wrap_cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t __wrap_cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(8); return cudaSuccess; }
cudaError_t __wrap_cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(8); return cudaSuccess; }
cudaError_t __wrap_cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t __wrap_cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t __wrap_cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }

cufftResult cufftPlanMany(cufftHandle* plan, int, int*, int*, int, int, int*, int, int, cufftType, int) { *plan = 1; return CUFFT_SUCCESS; }
cufftResult cufftSetStream(cufftHandle, cudaStream_t) { return CUFFT_SUCCESS; }
cufftResult cufftExecZ2Z(cufftHandle, cufftDoubleComplex* in, cufftDoubleComplex* out, int) { need(in, "fft"); need(out, "fft"); return CUFFT_SUCCESS; }
cufftResult cufftExecD2Z(cufftHandle, cufftDoubleReal* in, cufftDoubleComplex* out) { need(in, "fft"); need(out, "fft"); return CUFFT_SUCCESS; }
cufftResult cufftDestroy(cufftHandle) { return CUFFT_SUCCESS; }

}  // extern "C"

namespace qew {

cudaError_t split_tiles(const ChainDesc* chains, int32_t, int, int32_t, const int32_t* first, WarpTile* tiles, cudaStream_t s)
{
    on_stream(s);
    need(chains, "split_tiles");
    need(first, "split_tiles");
    need(tiles, "split_tiles");
    return cudaSuccess;
}
bool split_supported(int kind, int S) { return S == 7 || S == 15 || (!quad_kind(kind) && (S == 23 || S == 31 || (S == 39 && kind != kNone))); }
size_t split_smem_bytes(int, int S, int tiles) { return static_cast<size_t>(tiles) * 32 * S * 28; }
int split_warps_per_sm(int, int) { return 16; }
cudaError_t split_step(int kind, int, int, const SplitLaunch& a, cudaStream_t s)
{
    on_stream(s);
    need(a.tiles, "split_step tiles");
    split_arrays(a.in, kind, "split_step in");
    if (a.K > 0)
        split_arrays(a.out, kind, "split_step out");
    if (a.n_obs > 0) {
        need(a.partial, "split_step partials");
        need(a.shift, "split_step shift");
    }
    need(a.error, "split_step error");
    last_K = a.K;
    last_n_obs = a.n_obs;
    max_n_obs = a.n_obs > max_n_obs ? a.n_obs : max_n_obs;
    last_has_q3 = a.in.q3 != nullptr;
    return cudaSuccess;
}
cudaError_t split_init(const ChainDesc* chains, int32_t, const TileDesc* tiles, int32_t, int32_t, SplitState st, uint64_t, int,
                       const double*, cudaStream_t s)
{
    on_stream(s);
    need(chains, "split_init");
    need(tiles, "split_init");
    split_arrays(st, kNone, "split_init");
    return cudaSuccess;
}
cudaError_t split_to_f64(const ChainDesc* chains, const TileDesc* tiles, int32_t, int32_t, SplitState st, double*, int32_t*, cudaStream_t s)
{
    on_stream(s);
    need(chains, "split_to_f64");
    need(tiles, "split_to_f64");
    split_arrays(st, kNone, "split_to_f64");
    return cudaSuccess;
}
cudaError_t split_range_guard(const ChainDesc* chains, int32_t, int64_t, const int32_t* cell, int32_t* error, cudaStream_t s)
{
    on_stream(s);
    need(chains, "range guard");
    need(cell, "range guard");
    need(error, "range guard");
    return cudaSuccess;
}

// (only the shapes that matter here: look-ahead, several steps, one step in place)
F64Shape f64_shape(int64_t n_sites, int)
{
    if (n_sites <= (int64_t(1) << 20))
        return F64Shape{256, 1, 16, true};
    if (n_sites <= (int64_t(1) << 29))
        return F64Shape{128, 4, 8, false};
    return F64Shape{256, 4, 1, false};
}
size_t f64_step_smem(const F64Shape&, int) { return 0; }
static void f64_arrays(const F64State& s, int n, const char* what)
{
    need(s.ncache, what);
    for (int c = 0; c < n; ++c)
        need(s.c[c], what);
}
cudaError_t f64_step(const F64Step& a, const F64Shape& s, cudaStream_t st)
{
    on_stream(st);
    need(a.tiles, "f64_step tiles");
    need(a.chains, "f64_step chains");
    need(a.u_in, "f64_step u");
    need(a.u_out, "f64_step u");
    f64_arrays(a.in, a.n_nodes, "f64_step in");
    f64_arrays(a.out, a.n_nodes, "f64_step out");
    last_K = s.K;
    last_in_place = a.in.ncache == a.out.ncache;
    return cudaSuccess;
}
cudaError_t f64_observe(const F64Launch& a, cudaStream_t st)
{
    on_stream(st);
    need(a.tiles, "f64_observe tiles");
    need(a.u_in, "f64_observe u");
    need(a.partial, "f64_observe partials");
    need(a.st.ncache, "f64_observe cache");
    return cudaSuccess;
}
cudaError_t f64_init(const ChainDesc* chains, const TileDesc* tiles, int32_t, int32_t, F64State st, uint64_t, int, const double*, cudaStream_t s)
{
    on_stream(s);
    need(chains, "f64_init");
    need(tiles, "f64_init");
    need(st.u, "f64_init");
    f64_arrays(st, 2, "f64_init");
    return cudaSuccess;
}
cudaError_t f64_cells(const ChainDesc* chains, const TileDesc* tiles, int32_t, int32_t, const double* u, int32_t* cells, cudaStream_t s)
{
    on_stream(s);
    need(chains, "f64_cells");
    need(tiles, "f64_cells");
    need(u, "f64_cells");
    need(cells, "f64_cells");
    return cudaSuccess;
}
cudaError_t reduce_chains(const ChainDesc* chains, int32_t, const double* partial, int64_t, double* shift, double* obs, const ObsList&,
                          cudaStream_t s)
{
    on_stream(s);
    need(chains, "reduce");
    need(partial, "reduce");
    need(shift, "reduce");
    need(obs, "reduce");
    return cudaSuccess;
}
bool sq_half(int32_t L) { return L % 2 == 0 && L >= 4; }
int64_t sq_row(int32_t L) { return sq_half(L) ? L : 2 * (static_cast<int64_t>(L) / 2 + 1); }
cudaError_t sq_rows(const ChainDesc* chains, int32_t, int32_t, const SplitState* split, const double* u64, double* rows, cudaStream_t s)
{
    on_stream(s);
    need(chains, "sq_rows");
    need(split ? static_cast<const void*>(split->cell) : u64, "sq_rows");
    need(rows, "sq_rows");
    return cudaSuccess;
}
cudaError_t sq_power(const void* Z, int32_t, int32_t, int32_t, double* S, cudaStream_t s)
{
    on_stream(s);
    need(Z, "sq_power");
    need(S, "sq_power");
    return cudaSuccess;
}
cudaError_t bounded_wait_selftest(int32_t*, int, cudaStream_t) { return cudaSuccess; }
cudaError_t philox_words(const uint32_t*, const uint32_t*, int64_t, uint32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t disorder_values(int, int, uint64_t, uint32_t, const int64_t*, const int64_t*, int64_t, double*, cudaStream_t) { return cudaSuccess; }

}  // namespace qew
