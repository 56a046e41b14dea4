// noalloc.cu -- pic_field_solve_noalloc: the integer Poisson solve and E = -grad phi
// of one instance, computed without allocating any memory.
//
// Some callers cannot allocate device memory: code that runs while a CUDA graph is
// being captured, latency-critical loops in which an allocation could block or
// fragment the heap, and host frameworks that own every byte of device memory
// through their own pools.  This entry point serves them.  The caller passes the
// fixed-point charge deposits and the output array; the only scratch the solve
// needs (two 128-bit sums per chunk of nodes) lives in the file-scope device array
// below, which every GPU that loads the library holds until the process exits.  The math is the same as the handle's field phase (without
// its optional density smoother: the deposits are used as given):
//   Z_j = sum_s z_s D_s[j],  R_j = sum_{1<=k<=j, k<N} Z_k,  U = sum_{1<=k<N} (N-k) Z_k,
//   E_j = lambda (N (R_{j-1} + R_j) - 2U)      (0 < j < N),
//   E_0 = lambda (-2U - 2N Z_0),  E_N = lambda (2N R_{N-1} - 2U + 2N Z_N),
//   lambda = delta / (2 N S eps0).
#include <mutex>
#include <string>

#include "common.cuh"

namespace bitpic {
namespace {

constexpr int kNoAllocMaxCells = 65536;
constexpr int kNoAllocMaxNodes = kNoAllocMaxCells + 1;
constexpr int kMaxDevices = 64;
// Nodes of a chunk, one a thread: 257 blocks at the largest size, so that a block adds up
// the chunk sums in two rounds.  Up to kNoAllocOneBlock nodes one block does it all in one
// launch.  A call waited for alone, before and after: 65,536 cells 164 -> 25 us (11 us in
// a row), 20,000 73 -> 22, 2,912 26 -> 21, 500 24 -> 17.5, 64 23 -> 16.4; the launches and
// the host's checks are what is left.
constexpr int kNoAllocChunk = 256;
constexpr int kNoAllocOneBlock = 1024;

// Scratch shared by every call on a device: per chunk of nodes the sums of Z'_j and of
// (N-j) Z'_j over its interior nodes.
static __device__ __align__(256) i128 g_scratch[2 * ((kNoAllocMaxNodes + kNoAllocChunk - 1) / kNoAllocChunk)];

// Device address of g_scratch per device, from the last lookup made with that device
// current and no capture in progress on the call's stream.
std::mutex g_mutex;
void* g_scratch_addr[kMaxDevices] = {};

struct NoAllocArgs {
    const long long* charge;  // nspecies x (N+1) deposits, species-major
    int ncells;
    int nspecies;
    int z[kMaxSpecies];
    double lambda;
    i128* scratch;            // [2c], [2c+1]: the sums of chunk c
    double* E;
};

__device__ __forceinline__ i128 incl_scan_warp(i128 v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const i128 t = shfl_up_i128(v, d);
        if (lane >= d) v += t;
    }
    return v;
}

__device__ __forceinline__ i128 sum_warp(i128 v)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += shfl_i128(v, (threadIdx.x & 31) ^ d);
    return v;
}

__device__ __forceinline__ i128 charge_at(const NoAllocArgs& a, int j)
{
    i128 z = 0;
    for (int k = 0; k < a.nspecies; ++k)
        z += (i128)a.z[k] * (i128)a.charge[(int64_t)k * (a.ncells + 1) + j];
    return z;
}

// Sum of v over the block, for every thread.  sh: 33 entries.
__device__ __forceinline__ i128 block_sum(i128 v, i128* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = sum_warp(v);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const i128 t = sum_warp(lane < nw ? sh[lane] : (i128)0);
        if (lane == 0) sh[32] = t;
    }
    __syncthreads();
    const i128 t = sh[32];
    __syncthreads();
    return t;
}

// Inclusive prefix of v over the block.
__device__ __forceinline__ i128 block_scan(i128 v, i128* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const i128 inc = incl_scan_warp(v);
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const i128 w = lane < nw ? sh[lane] : (i128)0;
        const i128 wi = incl_scan_warp(w);
        if (lane < nw) sh[lane] = wi - w;
    }
    __syncthreads();
    return sh[warp] + inc;
}

// E of node j from R_{j-1} and Z_j (the wall nodes' Z enters E alone).
__device__ __forceinline__ double field_at(const NoAllocArgs& a, int j, i128 Rprev, i128 z, i128 U)
{
    const int N = a.ncells;
    const i128 NN = (i128)N;
    i128 G;
    if (j == 0) G = -2 * U - 2 * NN * z;
    else if (j == N) G = 2 * NN * Rprev - 2 * U + 2 * NN * z;
    else G = NN * (2 * Rprev + z) - 2 * U;
    return a.lambda * i128_to_double(G);
}

// The whole solve in one block (one node a thread) where the nodes fit: one launch.
__global__ void __launch_bounds__(1024) k_solve_noalloc(const NoAllocArgs a)
{
    __shared__ i128 sh[33];
    const int N = a.ncells, j = threadIdx.x;
    const i128 z = j <= N ? charge_at(a, j) : (i128)0;
    const i128 in = (j > 0 && j < N) ? z : (i128)0;
    const i128 U = block_sum((i128)(N - j) * in, sh);
    const i128 R = block_scan(in, sh);
    if (j <= N) a.E[j] = field_at(a, j, R - in, z, U);
}

// Larger instances in chunks of kNoAllocChunk nodes, a block each: the chunks' sums, then
// every block adds up the sums of the chunks before its own and of all of them and scans
// its nodes.  (All nodes in the threads of one block, 64 consecutive ones a thread, took
// 146 us for 65,536 cells: a serial chain of uncoalesced 128-bit accesses on one SM.)
__global__ void __launch_bounds__(kNoAllocChunk) k_sums_noalloc(const NoAllocArgs a)
{
    __shared__ i128 sh[33];
    const int N = a.ncells, j = blockIdx.x * kNoAllocChunk + threadIdx.x;
    const i128 in = (j > 0 && j < N) ? charge_at(a, j) : (i128)0;
    const i128 s = block_sum(in, sh), w = block_sum((i128)(N - j) * in, sh);
    if (threadIdx.x == 0) {
        a.scratch[2 * blockIdx.x] = s;
        a.scratch[2 * blockIdx.x + 1] = w;
    }
}

__global__ void __launch_bounds__(kNoAllocChunk) k_emit_noalloc(const NoAllocArgs a)
{
    __shared__ i128 sh[33];
    const int N = a.ncells, j = blockIdx.x * kNoAllocChunk + threadIdx.x;
    const i128 z = j <= N ? charge_at(a, j) : (i128)0;
    const i128 in = (j > 0 && j < N) ? z : (i128)0;
    i128 before = 0, u = 0;
    for (int c = threadIdx.x; c < (int)gridDim.x; c += kNoAllocChunk) {
        if (c < (int)blockIdx.x) before += a.scratch[2 * c];
        u += a.scratch[2 * c + 1];
    }
    const i128 U = block_sum(u, sh), R0 = block_sum(before, sh);
    const i128 R = R0 + block_scan(in, sh);
    if (j <= N) a.E[j] = field_at(a, j, R - in, z, U);
}

// The device address of the scratch array for the current device.  Host code must not
// hand the symbol itself to a kernel.  Outside stream capture the address is looked up
// on every call (cheap; a device reset or a new context reloads the module at another
// address); during a capture the lookup could load the module inside it, so the address
// of the last lookup on this device is reused and a first call under capture fails.
int scratch_for_current_device(cudaStream_t st, void** out, std::string* why)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        *why = std::string("cudaGetDevice: ") + cudaGetErrorString(e);
        return PIC_ECUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) {
        *why = "device index out of range";
        return PIC_EINVAL;
    }
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) {
        *why = std::string("cudaStreamIsCapturing: ") + cudaGetErrorString(e);
        return PIC_ECUDA;
    }
    std::lock_guard<std::mutex> lock(g_mutex);
    if (cs == cudaStreamCaptureStatusNone) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess || !p) {
            *why = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e);
            return PIC_ECUDA;
        }
        g_scratch_addr[dev] = p;
    } else if (!g_scratch_addr[dev]) {
        *why = "the first call on a device must not be made during stream capture";
        return PIC_EINVAL;
    }
    *out = g_scratch_addr[dev];
    return PIC_OK;
}

}  // namespace

// defined with pic_last_error: the message pic_last_error(NULL) returns
void set_global_error(const std::string& msg);

}  // namespace bitpic

using namespace bitpic;

extern "C" PIC_API int pic_field_solve_noalloc(int32_t ncells, int32_t nspecies,
                                               const int64_t* charge, const int32_t* z,
                                               double delta, int64_t unit, double eps0,
                                               double* E, void* stream)
{
    set_global_error("");
    if (ncells < 1 || ncells > kNoAllocMaxCells) {
        set_global_error("pic_field_solve_noalloc: ncells must be in [1, " +
                         std::to_string(kNoAllocMaxCells) + "] (the size of its static scratch)");
        return PIC_EINVAL;
    }
    if (nspecies < 1 || nspecies > kMaxSpecies || !charge || !z || !E || unit <= 0 ||
        !(delta > 0) || !(eps0 > 0)) {
        set_global_error("pic_field_solve_noalloc: bad arguments");
        return PIC_EINVAL;
    }
    void* scratch = nullptr;
    std::string why;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int rc = scratch_for_current_device(st, &scratch, &why);
    if (rc != PIC_OK) {
        set_global_error("pic_field_solve_noalloc: " + why);
        return rc;
    }
    NoAllocArgs a;
    a.charge = reinterpret_cast<const long long*>(charge);
    a.ncells = ncells;
    a.nspecies = nspecies;
    for (int k = 0; k < kMaxSpecies; ++k) a.z[k] = k < nspecies ? z[k] : 0;
    a.lambda = delta / (2.0 * (double)ncells * (double)unit * eps0);
    a.scratch = static_cast<i128*>(scratch);
    a.E = E;
    const int nodes = ncells + 1;
    if (nodes <= kNoAllocOneBlock) {
        k_solve_noalloc<<<1, (nodes + 31) / 32 * 32, 0, st>>>(a);
    } else {
        const int blocks = (nodes + kNoAllocChunk - 1) / kNoAllocChunk;
        k_sums_noalloc<<<blocks, kNoAllocChunk, 0, st>>>(a);
        k_emit_noalloc<<<blocks, kNoAllocChunk, 0, st>>>(a);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_global_error(std::string("pic_field_solve_noalloc: ") + cudaGetErrorString(e));
        return PIC_ECUDA;
    }
    return PIC_OK;
}
