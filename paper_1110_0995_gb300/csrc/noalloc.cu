// Area and volume of closed triangle meshes without any device allocation.
//
// Some callers cannot allocate device memory: code that runs under a
// framework which owns the whole device memory pool (a cudaMalloc there fails
// or fragments the pool), code in a latency-critical loop where cudaMalloc's
// implicit synchronisation is not acceptable, and embedded callers with a
// fixed memory budget.  This file gives them a variant of the library's
// per-cell area / volume reduction whose scratch space (the per-block partial
// sums) lives in a fixed, file-scope device array instead of memory the
// library allocates.  Inputs and outputs are still the caller's buffers.
//
// The scratch array exists once per device that loads the library and stays
// there until the process exits.  Meshes of small cells do not touch it; every
// call with a larger cell shares it, and it keeps the last such call's
// contents; each call writes every partial it later reads, so nothing has to
// start at zero.  Two such calls whose kernels overlap on the GPU (different
// streams, or different host threads) race on the array.
//
// The array's device address belongs to the CUDA context that loaded the
// module.  It is looked up on a device's first call and again whenever the
// context current on that device changes (a cudaDeviceReset, or a driver
// context the caller made current), keyed by the context's unique id.
#include "lbibm.h"

#include <cuda.h>
#include <cuda_runtime.h>
#include <cooperative_groups.h>

#include <mutex>
#include <vector>

namespace cg = cooperative_groups;

namespace {

constexpr int NA_BLOCK = 256;                 // triangles per block (chunk)
constexpr int NA_MAX_PARTIALS = 65536;        // 65,536 x 16 B = 1 MiB of scratch
constexpr int NA_MAX_DEVICES = 64;

// Per-block partial sums (area, volume) of the reduction, indexed
// cell * max_chunks + chunk.  Host code must not pass this symbol to a kernel:
// on the host it is only a stand-in; its device address comes from
// cudaGetSymbolAddress below.
static __device__ __align__(256) double2 g_noalloc_partials[NA_MAX_PARTIALS];

std::mutex g_setup_mutex;
void* g_scratch_ptr[NA_MAX_DEVICES] = {};
unsigned long long g_scratch_ctx[NA_MAX_DEVICES] = {};
int g_sms[NA_MAX_DEVICES] = {};

// Unique id of the context current on the calling thread (driver entry points
// through the runtime, so the library needs no link against libcuda).
typedef CUresult (*ctx_get_current_fn)(CUcontext*);
typedef CUresult (*ctx_get_id_fn)(CUcontext, unsigned long long*);

cudaError_t current_context_id(unsigned long long* id) {
    static ctx_get_current_fn get_current = nullptr;
    static ctx_get_id_fn get_id = nullptr;
    if (!get_current || !get_id) {
        void* a = nullptr;
        void* b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa);
        if (e != cudaSuccess || qa != cudaDriverEntryPointSuccess) return e != cudaSuccess ? e : cudaErrorNotSupported;
        e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb);
        if (e != cudaSuccess || qb != cudaDriverEntryPointSuccess) return e != cudaSuccess ? e : cudaErrorNotSupported;
        get_current = (ctx_get_current_fn)a;
        get_id = (ctx_get_id_fn)b;
    }
    CUcontext c = nullptr;
    if (get_current(&c) != CUDA_SUCCESS || !c) return cudaErrorDeviceUninitialized;
    if (get_id(c, id) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    return cudaSuccess;
}

// Device address of the scratch array in the current context and the device's
// SM count, looked up (under a lock) on the first call on a device and whenever
// that device's current context has changed since the last lookup.
cudaError_t scratch_address(double2** out, int* sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NA_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    unsigned long long id = 0;
    const bool have_id = current_context_id(&id) == cudaSuccess;   // false: no context current yet
    if (!have_id || !g_scratch_ptr[dev] || g_scratch_ctx[dev] != id) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_partials);   // makes the primary context current if none is
        if (e != cudaSuccess) return e;
        e = current_context_id(&id);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        g_scratch_ptr[dev] = p;
        g_scratch_ctx[dev] = id;
    }
    *out = (double2*)g_scratch_ptr[dev];
    *sms = g_sms[dev];
    return cudaSuccess;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Cells of up to NA_CLUSTER_TRIS triangles: one launch, a cluster of one to
// eight blocks per cell, whose partial sums the first block reads from the
// others' shared memory (no scratch).  What bounds the reduction is this GPU's
// FP64 pipe (two operations per clock per SM), at few cells the latency of one
// triangle's chain, and in two launches the gap between them.  So the volume
// takes its cross product from the area's (a . (b - a) x (c - a) is the same
// determinant, and cancels less), the factors 1/2 and 1/6 are applied once per
// cell, and a cell's triangles go in equal shares of whole warps to the largest
// cluster with which all blocks are resident at once: more blocks per cell
// balance the SMs, fewer leave more triangles to each block's one reduction.
// Measured on GB300, us per call, two launches -> this: one 1,280-triangle
// cell 11.8 -> 8.2, 62 cells (87,040 triangles) 25.5 -> 16.4, 406 cells (542,720)
// 57.3 -> 53.3 (with eight blocks for each of the 406: 72.6).  Cells beyond 32
// chunks of 256 keep the two launches, which spread one cell over any number of SMs.
constexpr int NA_CLUSTER = 8;
constexpr int NA_CLUSTER_TRIS = 32 * NA_BLOCK;
constexpr int NA_RESIDENT = 6;                // blocks per SM at 40 registers a thread (24 bytes spilled)

// (area x 2, volume x 6) of triangle t, added to s and v.
__device__ __forceinline__ void triangle_terms(const double* __restrict__ xyz, const int* __restrict__ tris, int t,
                                               double& s, double& v) {
    const int ia = tris[3 * t], ib = tris[3 * t + 1], ic = tris[3 * t + 2];
    const double ax = xyz[3 * ia], ay = xyz[3 * ia + 1], az = xyz[3 * ia + 2];
    const double ux = xyz[3 * ib] - ax, uy = xyz[3 * ib + 1] - ay, uz = xyz[3 * ib + 2] - az;
    const double wx = xyz[3 * ic] - ax, wy = xyz[3 * ic + 1] - ay, wz = xyz[3 * ic + 2] - az;
    const double nx = uy * wz - uz * wy, ny = uz * wx - ux * wz, nz = ux * wy - uy * wx;
    s += sqrt(nx * nx + ny * ny + nz * nz);
    v += ax * nx + ay * ny + az * nz;
}

// Block sums of s and v: s on thread 0, v on thread 16.  The first exchange
// leaves the sums of s to a warp's lower half and those of v to its upper half,
// which halves the FP64 additions.
__device__ __forceinline__ double block_sums(double s, double v, double (*sh)[2]) {
    const bool hi = threadIdx.x & 16;
    double x = hi ? v : s;
    const double y = __shfl_xor_sync(0xffffffffu, hi ? s : v, 16);
    x += y;
    for (int o = 8; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o, 16);
    if ((threadIdx.x & 15) == 0) sh[threadIdx.x >> 5][hi] = x;
    __syncthreads();
    if (threadIdx.x == 0 || threadIdx.x == 16)
        for (int w = 1; w < NA_BLOCK / 32; ++w) x += sh[w][hi];
    return x;
}

__global__ void __launch_bounds__(NA_BLOCK, NA_RESIDENT)
    k_area_volume_cluster(const double* __restrict__ xyz, const int* __restrict__ tris, const int* __restrict__ cell_start,
                          int max_tris, double* area, double* volume) {
    __shared__ double sh[NA_BLOCK / 32][2];
    __shared__ double sum[2];
    const cg::cluster_group cl = cg::this_cluster();
    const int c = blockIdx.y, blocks = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    // (at most max_tris, from the host's copy of the offsets: a bound for device
    // offsets that disagree with it)
    const int t0 = cell_start[c], n = max(0, min(cell_start[c + 1] - t0, max_tris));
    const int share = ((n + 31) / 32 + blocks - 1) / blocks * 32;
    const int t1 = t0 + min(n, (rank + 1) * share);
    double s = 0.0, v = 0.0;
    for (int t = t0 + rank * share + threadIdx.x; t < t1; t += NA_BLOCK) triangle_terms(xyz, tris, t, s, v);
    const double x = block_sums(s, v, sh);
    if (threadIdx.x == 0) sum[0] = x;
    if (threadIdx.x == 16) sum[1] = x;
    cl.sync();
    if (rank == 0 && (threadIdx.x == 0 || threadIdx.x == 16)) {
        const int k = threadIdx.x >> 4;
        double S = x;
        for (int r = 1; r < blocks; ++r) S += cl.map_shared_rank(sum, r)[k];
        if (k == 0) area[c] = 0.5 * S;
        else volume[c] = S / 6.0;
    }
    cl.sync();   // the other blocks' shared memory stays until it has been read
}

// Pass 1: block (chunk, cell) sums area and 6 x volume of up to NA_BLOCK
// triangles of one cell in FP64 and writes one partial.
__global__ void __launch_bounds__(NA_BLOCK) k_area_volume_partials(const double* __restrict__ xyz,
                                                                  const int* __restrict__ tris,
                                                                  const int* __restrict__ cell_start,
                                                                  int max_chunks, double2* partials) {
    const int c = blockIdx.y;
    const int k = blockIdx.x;
    const int t0 = cell_start[c], t1 = cell_start[c + 1];
    const int t = t0 + k * NA_BLOCK + threadIdx.x;
    if (t0 + k * NA_BLOCK >= t1) return;   // the whole block is past this cell's triangles
    double s = 0.0, v = 0.0;
    if (t < t1) triangle_terms(xyz, tris, t, s, v);
    __shared__ double sh[NA_BLOCK / 32][2];
    const double x = block_sums(s, v, sh);
    double* out = &partials[(long long)c * max_chunks + k].x;
    if (threadIdx.x == 0) out[0] = 0.5 * x;
    if (threadIdx.x == 16) out[1] = x / 6.0;
}

// Pass 2: one warp per cell adds the cell's partials in a fixed order.  The
// chunk count comes from the device offsets and is clamped to the row stride
// the host derived from its copy, so offsets that disagree with the host copy
// give a wrong sum but never a read outside the cell's row of partials.
__global__ void k_area_volume_final(const int* __restrict__ cell_start, int n_cells, int max_chunks,
                                    const double2* partials, double* area, double* volume) {
    const int c = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= n_cells) return;
    const int nt = cell_start[c + 1] - cell_start[c];
    int nk = (nt + NA_BLOCK - 1) / NA_BLOCK;
    nk = nk < 0 ? 0 : (nk > max_chunks ? max_chunks : nk);
    double S = 0.0, V = 0.0;
    for (int k = lane; k < nk; k += 32) {
        const double2 p = partials[(long long)c * max_chunks + k];
        S += p.x;
        V += p.y;
    }
    S = warp_sum(S);
    V = warp_sum(V);
    if (lane == 0) {
        area[c] = S;
        volume[c] = V;
    }
}

}  // namespace

extern "C" lb_status ibm_area_volume_noalloc(const double* xyz, const int32_t* tris, const int32_t* cell_tri_start,
                                             const int32_t* cell_tri_start_host, int n_cells, double* area,
                                             double* volume, void* cuda_stream) {
    if (n_cells < 0 || (n_cells > 0 && (!xyz || !tris || !cell_tri_start || !cell_tri_start_host || !area || !volume)))
        return LB_ERR_ARG;
    if (n_cells == 0) return LB_OK;
    if (n_cells > 65535) return LB_ERR_ARG;                    // grid y limit
    int max_chunks = 0;
    for (int c = 0; c < n_cells; ++c) {
        const int nt = cell_tri_start_host[c + 1] - cell_tri_start_host[c];
        if (nt < 0 || cell_tri_start_host[c] < 0) return LB_ERR_ARG;
        const int nk = (nt + NA_BLOCK - 1) / NA_BLOCK;
        if (nk > max_chunks) max_chunks = nk;
    }
    if (max_chunks == 0) max_chunks = 1;
    // the scratch holds one partial per (cell, chunk of 256 triangles)
    if ((long long)n_cells * max_chunks > NA_MAX_PARTIALS) return LB_ERR_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // looked up on either path: any call before a capture prepares every later one
    double2* scratch = nullptr;
    int sms = 0;
    if (scratch_address(&scratch, &sms) != cudaSuccess) return LB_ERR_CUDA;
    int max_tris = max_chunks * NA_BLOCK;
    if (max_tris <= NA_CLUSTER_TRIS) {
        int cluster = NA_CLUSTER;
        while (cluster > 1 && (long long)cluster * n_cells > (long long)NA_RESIDENT * sms) cluster /= 2;
        const double* x = xyz;
        const int *t = tris, *c0 = cell_tri_start;
        void* args[] = {(void*)&x, (void*)&t, (void*)&c0, (void*)&max_tris, (void*)&area, (void*)&volume};
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = cluster;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cluster, n_cells);
        cfg.blockDim = dim3(NA_BLOCK);
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelExC(&cfg, (const void*)k_area_volume_cluster, args) == cudaSuccess ? LB_OK : LB_ERR_CUDA;
    }
    // each launch's own status (cudaLaunchKernel returns it; an error left over
    // from an unrelated earlier call is neither consumed nor reported here)
    const double* a_xyz = xyz;
    const int* a_tris = tris;
    const int* a_start = cell_tri_start;
    void* args1[] = {(void*)&a_xyz, (void*)&a_tris, (void*)&a_start, (void*)&max_chunks, (void*)&scratch};
    if (cudaLaunchKernel((const void*)k_area_volume_partials, dim3(max_chunks, n_cells), dim3(NA_BLOCK), args1, 0,
                         s) != cudaSuccess)
        return LB_ERR_CUDA;
    const double2* a_scr = scratch;
    void* args2[] = {(void*)&a_start, (void*)&n_cells, (void*)&max_chunks, (void*)&a_scr, (void*)&area,
                     (void*)&volume};
    if (cudaLaunchKernel((const void*)k_area_volume_final, dim3((n_cells + 7) / 8), dim3(256), args2, 0, s) !=
        cudaSuccess)
        return LB_ERR_CUDA;
    return LB_OK;
}
