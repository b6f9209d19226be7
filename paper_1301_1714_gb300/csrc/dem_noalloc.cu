// dem_sort_cells_static: the cell hash and (cell, id) counting sort for callers that
// must not allocate device memory.
//
// Who needs this: a process that has already reserved all of the GPU's memory for its
// own pool (so a cudaMalloc from this library would fail or fragment that pool), and a
// loop that forbids allocation after start-up because cudaMalloc/cudaFree can block or
// synchronise the device at unpredictable moments. Such callers pass their own input and
// output buffers; the temporary counters and slot arrays this sort needs live in one
// fixed array of device memory that the library declares at file scope (about 6 MB, held
// on every GPU that loads the library until the process exits).
//
// The static array is shared by every call: calls whose work overlaps on the GPU (two
// streams, or two host threads) race on it and give wrong results. Each call clears the
// counters it relies on before use.
#include <algorithm>
#include <cstdint>
#include <mutex>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "dem.h"
#include "dem_dev.cuh"

namespace {

constexpr uint32_t SA_MAX_N = DEM_STATIC_SORT_MAX_N;
constexpr uint32_t SA_MAX_CELLS = DEM_STATIC_SORT_MAX_CELLS;
constexpr int SA_THREADS = 256;
constexpr int SA_ITEMS = 8;
constexpr uint32_t SA_TILE = SA_THREADS * SA_ITEMS;
constexpr uint32_t SA_MAX_PART = (SA_MAX_CELLS + 1 + SA_TILE - 1) / SA_TILE;

// offsets (in 32-bit words) of the pieces of the scratch array
constexpr size_t SA_OFF_CNT = 0;                                   // SA_MAX_CELLS + 1 counts
constexpr size_t SA_OFF_RANK = ((SA_MAX_CELLS + 1 + 63) / 64) * 64;  // SA_MAX_N ranks within a cell
constexpr size_t SA_OFF_TMP = SA_OFF_RANK + SA_MAX_N;              // SA_MAX_N cell-major slots
constexpr size_t SA_OFF_PART = SA_OFF_TMP + SA_MAX_N;              // SA_MAX_PART scan partials
constexpr size_t SA_WORDS = SA_OFF_PART + SA_MAX_PART;

static __device__ __align__(256) uint32_t g_sort_scratch[SA_WORDS];

// Device address of g_sort_scratch on each device, and the grid of the sort (taken once per
// device).
std::mutex g_mu;
constexpr int SA_MAX_DEVICES = 64;
void* g_addr[SA_MAX_DEVICES] = {nullptr};
int g_resident[SA_MAX_DEVICES] = {0};   // blocks of k_sa_sort resident at once
constexpr int SA_PER_SM = 2;

__device__ __forceinline__ uint32_t sa_axis(double xa, double o, double h, float inv_h, int64_t dim) {
    bool clamped = false;
    return demgb::cell_of_axis(__dsub_rn(xa, o), h, inv_h, dim, clamped);
}

// The whole sort in one cooperative launch: as a memset and six kernels it took 67 us for
// 200,003 positions and 47 us for 2,001, most of it launches; now 56 and 34. The phases are
// separated by grid barriers (every block is resident; 1 / 2 / 4 / 8 blocks per SM took 61 /
// 56 / 62 / 69 us at 200,003):
//   0 clear the counts  1 cell key and rank within the cell  2 sums of tiles of counts
//   3 exclusive prefix (each block adds up the tile sums before its tiles: at most 513)
//   4 particles into cell-major slots  5 place of a particle in its cell = number of
//   cell-mates with a smaller id (each thread reads its whole cell, so the work grows with
//   the square of the cells' occupancy)
__global__ void __launch_bounds__(SA_THREADS) k_sa_sort(uint32_t n, const double* __restrict__ x, double ox, double oy,
                                                        double oz, double h, float inv_h, int64_t nx, int64_t ny,
                                                        int64_t nz, uint32_t m, uint32_t ntiles, uint32_t* cell_of,
                                                        uint32_t* order, uint32_t* cell_start, uint32_t* scratch) {
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    __shared__ uint32_t ws[SA_THREADS / 32], s_pre;
    uint32_t* cnt = scratch + SA_OFF_CNT;
    uint32_t* rank = scratch + SA_OFF_RANK;
    uint32_t* tmp = scratch + SA_OFF_TMP;
    uint32_t* part = scratch + SA_OFF_PART;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    const uint32_t first = blockIdx.x * SA_THREADS + tid, step = gridDim.x * SA_THREADS;
    for (uint32_t k = first; k < m; k += step) cnt[k] = 0u;
    grid.sync();
    for (uint32_t k = first; k < n; k += step) {
        const uint32_t i = sa_axis(x[3 * (size_t)k], ox, h, inv_h, nx);
        const uint32_t j = sa_axis(x[3 * (size_t)k + 1], oy, h, inv_h, ny);
        const uint32_t l = sa_axis(x[3 * (size_t)k + 2], oz, h, inv_h, nz);
        const uint32_t key = (l * (uint32_t)ny + j) * (uint32_t)nx + i;
        cell_of[k] = key;
        rank[k] = atomicAdd(&cnt[key], 1u);
    }
    grid.sync();
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        uint32_t s = 0;
        for (int i = 0; i < SA_ITEMS; ++i) {
            const uint32_t k = t * SA_TILE + i * SA_THREADS + tid;
            if (k < m) s += cnt[k];
        }
        s = __reduce_add_sync(0xffffffffu, s);
        if (lane == 0) ws[wid] = s;
        __syncthreads();
        if (tid == 0) {
            uint32_t u = 0;
            for (int w = 0; w < SA_THREADS / 32; ++w) u += ws[w];
            part[t] = u;
        }
        __syncthreads();
    }
    grid.sync();
    uint32_t seen = 0, before = 0;
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        uint32_t u = 0;
        for (uint32_t k = seen + tid; k < t; k += SA_THREADS) u += part[k];
        if (tid == 0) s_pre = 0u;
        __syncthreads();
        u = __reduce_add_sync(0xffffffffu, u);
        if (lane == 0 && u) atomicAdd(&s_pre, u);
        uint32_t v[SA_ITEMS];
        uint32_t s = 0;
        for (int i = 0; i < SA_ITEMS; ++i) {
            const uint32_t k = t * SA_TILE + tid * SA_ITEMS + i;
            v[i] = k < m ? cnt[k] : 0u;
            s += v[i];
        }
        uint32_t inc = s;
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t w = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= (uint32_t)off) inc += w;
        }
        if (lane == 31) ws[wid] = inc;
        __syncthreads();
        before += s_pre;
        seen = t;
        uint32_t run = before + (inc - s);
        for (uint32_t w = 0; w < wid; ++w) run += ws[w];
        for (int i = 0; i < SA_ITEMS; ++i) {
            const uint32_t k = t * SA_TILE + tid * SA_ITEMS + i;
            if (k < m) cell_start[k] = run;
            run += v[i];
        }
        __syncthreads();
    }
    grid.sync();
    for (uint32_t k = first; k < n; k += step) tmp[cell_start[cell_of[k]] + rank[k]] = k;
    grid.sync();
    for (uint32_t s = first; s < n; s += step) {
        const uint32_t p = tmp[s];
        const uint32_t c = cell_of[p];
        const uint32_t lo = cell_start[c], hi = cell_start[c + 1];
        uint32_t r = 0;
        for (uint32_t k = lo; k < hi; ++k) r += tmp[k] < p ? 1u : 0u;
        order[lo + r] = p;
    }
}

}  // namespace

extern "C" dem_status dem_sort_cells_static(int64_t n, const double* x, const double* origin, double cell,
                                            const int64_t* dims, uint32_t* cell_of, uint32_t* order,
                                            uint32_t* cell_start, void* cuda_stream) {
    if (n < 0 || !origin || !dims || !(cell > 0.0)) return DEM_ERR_INVALID_ARG;
    // each axis first (so that the product cannot overflow), then the product
    for (int a = 0; a < 3; ++a)
        if (dims[a] < 1 || dims[a] > (int64_t)SA_MAX_CELLS) return DEM_ERR_INVALID_ARG;
    const int64_t ncells = dims[0] * dims[1] * dims[2];
    if (n > (int64_t)SA_MAX_N || ncells > (int64_t)SA_MAX_CELLS) return DEM_ERR_INVALID_ARG;
    if (!cell_start || (n > 0 && (!x || !cell_of || !order))) return DEM_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= SA_MAX_DEVICES) {
        cudaGetLastError();
        return DEM_ERR_CUDA;
    }
    uint32_t* scratch = nullptr;
    int resident = 0;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_addr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_sort_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return DEM_ERR_CUDA;
            }
            // two blocks per SM are enough for the largest sizes and leave the barriers cheap
            int sms = 0, per = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sa_sort, SA_THREADS, 0) != cudaSuccess || per < 1) {
                cudaGetLastError();
                return DEM_ERR_CUDA;
            }
            g_resident[dev] = sms * std::min(per, SA_PER_SM);
            g_addr[dev] = p;
        }
        scratch = (uint32_t*)g_addr[dev];
        resident = g_resident[dev];
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    uint32_t nn = (uint32_t)n, m = (uint32_t)ncells + 1, nb = (m + SA_TILE - 1) / SA_TILE;
    // as many blocks as there are pieces of work for, all of them resident
    const uint32_t want = std::max(1u, std::max((std::max(nn, m / SA_ITEMS) + SA_THREADS - 1) / SA_THREADS, nb));
    uint32_t blocks = std::min(want, (uint32_t)resident);
    double ox = origin[0], oy = origin[1], oz = origin[2], h = cell;
    float inv_h = (float)(1.0 / cell);
    int64_t nx = dims[0], ny = dims[1], nz = dims[2];
    void* args[] = {&nn, &x, &ox, &oy, &oz, &h, &inv_h, &nx, &ny, &nz, &m, &nb, &cell_of, &order, &cell_start, &scratch};
    if (cudaLaunchCooperativeKernel((const void*)k_sa_sort, dim3(blocks), dim3(SA_THREADS), args, 0, st) != cudaSuccess) {
        cudaGetLastError();
        return DEM_ERR_CUDA;
    }
    return DEM_OK;
}
