// The FP64 step and fields by tiles (lbm_tile64.cuh): plan and launch.
#include <cuda_runtime.h>

#include <algorithm>

#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_kernels.cuh"
#include "lbm_tile64.cuh"

namespace lbm {

namespace {

template <int MODE, typename IX>
void *pick(bool walls, bool pres)
{
    if (walls && pres) return (void *)step_kernel_tile64<true, true, MODE, IX>;
    if (walls) return (void *)step_kernel_tile64<true, false, MODE, IX>;
    if (pres) return (void *)step_kernel_tile64<false, true, MODE, IX>;
    return (void *)step_kernel_tile64<false, false, MODE, IX>;
}
void *kernel(int mode, bool walls, bool pres, bool big)
{
    if (mode == MODE_STEP) return big ? pick<MODE_STEP, long long>(walls, pres) : pick<MODE_STEP, int>(walls, pres);
    return big ? pick<MODE_FIELDS, long long>(walls, pres) : pick<MODE_FIELDS, int>(walls, pres);
}

}  // namespace

// Tile height: the one whose busiest SM has the least to do (a tile costs its
// rows and about 1.2 more for its halo's densities, phi and Laplacians; at
// 128 x 128 on 152 SMs that is 4, at 4096 x 512 it is 8). With walls the two rows
// next to a wall share a tile (rows % th != 1). CTAs: a tile each up to the
// slots of the per-CTA partials, then the resident CTAs stride over them.
cudaError_t tile64_plan(int nx, int ny, bool walls, bool pres, bool big, int sms, Tile64 *p)
{
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
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel(MODE_STEP, walls, pres, big),
                                                                  T64_TX * p->th, 0);
    if (e != cudaSuccess) return e;
    p->ctas = (int)std::min<long long>(ntiles, std::min<long long>(MAX_CTAS, (long long)sms * std::max(1, occ)));
    p->threads = T64_TX * p->th;
    return cudaSuccess;
}

cudaError_t tile64_launch(const KArgs<double> &A, int mode, bool walls, bool pres, bool big, const Tile64 &p, int ctas,
                          cudaStream_t st)
{
    T64Plan T{p.th, p.ntx, p.ntiles, p.sx, p.sy};
    void *args[] = {(void *)&A, (void *)&T};
    return cudaLaunchKernel(kernel(mode, walls, pres, big), dim3(ctas), dim3(p.threads), args, 0, st);
}

}  // namespace lbm
