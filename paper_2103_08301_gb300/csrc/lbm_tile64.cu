// The step of FP64 and of small FP32 grids, and the fields, by tiles
// (lbm_tile64.cuh): plan and launch.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <vector>

#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_kernels.cuh"
#include "lbm_tile64.cuh"

namespace lbm {

namespace {

template <typename real, int MODE, typename IX>
void *pick(bool walls, bool pres)
{
    if (walls && pres) return (void *)step_kernel_tile64<real, true, true, MODE, IX>;
    if (walls) return (void *)step_kernel_tile64<real, true, false, MODE, IX>;
    if (pres) return (void *)step_kernel_tile64<real, false, true, MODE, IX>;
    return (void *)step_kernel_tile64<real, false, false, MODE, IX>;
}
template <typename real>
void *fields_kernel(bool walls, bool pres, bool big)
{
    return big ? pick<real, MODE_FIELDS, long long>(walls, pres) : pick<real, MODE_FIELDS, int>(walls, pres);
}
template <typename real>
void *step_kernel_of(bool walls, bool pres, bool big)
{
    return big ? pick<real, MODE_STEP, long long>(walls, pres) : pick<real, MODE_STEP, int>(walls, pres);
}

}  // namespace

// Tile height: the one whose busiest SM has the least to do (a tile costs its
// rows and about 1.2 more for its halo's densities, phi and Laplacians; at
// 128 x 128 on 152 SMs that is 4, at 4096 x 512 it is 8). With walls the two rows
// next to a wall share a tile (rows % th != 1). CTAs: a tile each up to the
// resident ones (and the slots of the partials), which stride over the rest.
cudaError_t tile64_plan(int precision, int nx, int ny, bool walls, bool pres, bool big, int sms, Tile64 *p)
{
    void *fn = precision == 64 ? step_kernel_of<double>(walls, pres, big) : step_kernel_of<float>(walls, pres, false);
    const long long rows = walls ? ny - 2 : ny;
    p->sx = pres && (nx - 1) % T64_TX == 0 ? 1 : 0;
    const long long ntx = (nx + p->sx + T64_TX - 1) / T64_TX;
    double least = 0;
    p->th = 0;
    for (int th = T64_MAX; th >= 2; --th) {
        if (walls && rows % th == 1) continue;
        const long long t = ntx * ((rows + th - 1) / th);
        const double cost = (double)((t + sms - 1) / sms) * (th + 1.2);
        if (p->th == 0 || cost < 0.98 * least) { least = cost; p->th = th; }
    }
    p->ntx = (int)ntx;
    p->sy = 0;
    if (p->th == 0) {  // rows = 1 (mod 840): one row down, so the last tile holds two
        p->th = T64_MAX;
        p->sy = 1;
    }
    const long long ntiles = ntx * ((rows + p->sy + p->th - 1) / p->th);
    p->ntiles = (int)ntiles;
    int occ = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, T64_TX * p->th, 0);
    if (e != cudaSuccess) return e;
    p->ctas = (int)std::min<long long>(ntiles, std::min<long long>(MAX_CTAS, (long long)sms * std::max(1, occ)));
    p->threads = T64_TX * p->th;
    p->rot = 0;
    return cudaSuccess;
}

// Tile64::rot for a launch of `ctas`: of 0 .. 3 the one whose busiest CTA has the
// fewest tiles with a pressure column, over up to 256 rows of tiles.
void tile64_rotate(Tile64 *p, bool on, int ctas)
{
    p->rot = 0;
    if (!on || p->ntiles <= ctas) return;
    const int rows = std::min(p->ntiles / p->ntx, 256);
    int least = INT_MAX;
    std::vector<int> heavy(ctas);
    for (int rot = 0; rot < std::min(p->ntx, 4); ++rot) {
        std::fill(heavy.begin(), heavy.end(), 0);
        int most = 0;
        for (int by = 0; by < rows; ++by) {
            const int turn = by * rot % p->ntx, first = turn ? p->ntx - turn : 0;  // where column 0 went
            const int last = (first ? first : p->ntx) - 1;                          // and column ntx-1
            for (const int r : {first, last}) most = std::max(most, ++heavy[(by * p->ntx + r) % ctas]);
        }
        if (most < least) { least = most; p->rot = rot; }
    }
}

template <typename real>
cudaError_t tile64_launch(const KArgs<real> &A, bool walls, bool pres, bool big, const Tile64 &p, int ctas,
                          cudaStream_t st)
{
    T64Plan T{p.th, p.ntx, p.ntiles, p.sx, p.sy, p.rot};
    void *args[] = {(void *)&A, (void *)&T};
    return cudaLaunchKernel(step_kernel_of<real>(walls, pres, big), dim3(ctas), dim3(p.threads), args, 0, st);
}

namespace {

// cuPointerGetAttributes from the driver, looked up once through the runtime.
PFN_cuPointerGetAttributes_v7000 pointer_attributes()
{
    static const PFN_cuPointerGetAttributes_v7000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &p, 7000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<PFN_cuPointerGetAttributes_v7000>(p);
    }();
    return fn;
}

// Whether a kernel may write `bytes` at p itself: memory of device `dev`, aligned
// to its elements, all of it in one allocation. A range that leaves its allocation
// goes the way of host destinations, whose copy refuses it.
bool writable_here(const void *p, size_t bytes, size_t align, int dev)
{
    const PFN_cuPointerGetAttributes_v7000 query = pointer_attributes();
    if ((uintptr_t)p % align != 0 || !query) return false;
    unsigned type = 0, managed = 0;
    int ordinal = -1;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute at[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                 CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                 CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *data[5] = {&type, &managed, &ordinal, &start, &size};
    if (query(5, at, data, (CUdeviceptr)p) != CUDA_SUCCESS) return false;
    return type == CU_MEMORYTYPE_DEVICE && !managed && ordinal == dev && (CUdeviceptr)p >= start &&
           (CUdeviceptr)p - start <= size && bytes <= size - (size_t)((CUdeviceptr)p - start);
}
bool overlap(const void *a, size_t na, const void *b, size_t nb)
{
    return (uintptr_t)a < (uintptr_t)b + nb && (uintptr_t)b < (uintptr_t)a + na;
}

}  // namespace

template <typename real>
void fields_route(FieldsOut<real> &o, int nx, int ny, const void *busy, size_t busy_bytes)
{
    const size_t N = (size_t)nx * ny * sizeof(real), W = 2 * (size_t)nx * sizeof(real);
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    o.scratch = 0;
    for (int k = 0; k < 5; ++k) {
        const size_t bytes = k < 3 ? N : W;
        o.bytes[k] = bytes;
        bool direct = o.dst[k] && writable_here(o.dst[k], bytes, sizeof(real), dev) && !overlap(o.dst[k], bytes, busy, busy_bytes);
        for (int j = 0; direct && j < 5; ++j)
            if (j != k && o.dst[j] && overlap(o.dst[k], bytes, o.dst[j], j < 3 ? N : W)) direct = false;
        o.ptr[k] = direct ? (real *)o.dst[k] : nullptr;
        o.offset[k] = o.scratch;
        if (o.dst[k] && !direct) o.scratch += (bytes + 255) / 256 * 256;
    }
}

template <typename real>
cudaError_t fields_tiles(KArgs<real> A, const FieldsOut<real> &o, bool walls, bool pres, bool big, int sms, cudaStream_t st)
{
    if (!walls) {  // no wall loads
        for (int k = 3; k < 5; ++k)
            if (o.ptr[k]) {
                const cudaError_t e = cudaMemsetAsync(o.ptr[k], 0, o.bytes[k], st);
                if (e != cudaSuccess) return e;
            }
    }
    A.fout = nullptr;
    A.reverse = 0;
    A.o_rho = o.ptr[0]; A.o_vx = o.ptr[1]; A.o_vy = o.ptr[2]; A.o_tw = o.ptr[3]; A.o_pw = o.ptr[4];
    Tile64 p;
    cudaError_t e = tile64_plan(sizeof(real) * 8, A.nx, A.ny, walls, pres, big, sms, &p);
    if (e != cudaSuccess) return e;
    T64Plan T{p.th, p.ntx, p.ntiles, p.sx, p.sy, 0};
    void *args[] = {(void *)&A, (void *)&T};
    // no per-CTA slots: enough CTAs for every SM's threads
    const int ctas = (int)std::min<long long>(p.ntiles, (long long)sms * 8);
    return cudaLaunchKernel(fields_kernel<real>(walls, pres, big), dim3(ctas), dim3(p.threads), args, 0, st);
}

template <typename real>
cudaError_t fields_copy(const FieldsOut<real> &o, cudaStream_t st)
{
    for (int k = 0; k < 5; ++k)
        if (o.dst[k] && o.dst[k] != (void *)o.ptr[k]) {
            const cudaError_t e = cudaMemcpyAsync(o.dst[k], o.ptr[k], o.bytes[k], cudaMemcpyDefault, st);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

#define INST(real)                                                                                                     \
    template cudaError_t tile64_launch<real>(const KArgs<real> &, bool, bool, bool, const Tile64 &, int,               \
                                             cudaStream_t);                                                           \
    template void fields_route<real>(FieldsOut<real> &, int, int, const void *, size_t);                              \
    template cudaError_t fields_tiles<real>(KArgs<real>, const FieldsOut<real> &, bool, bool, bool, int, cudaStream_t); \
    template cudaError_t fields_copy<real>(const FieldsOut<real> &, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace lbm
