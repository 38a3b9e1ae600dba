// C ABI of the GB300 EOS-multiphase lattice Boltzmann solver (see include/lbm.h).
// Host orchestration only: argument checks, thermodynamic set-up in FP64,
// device workspace, kernel launches on the context stream, diagnostics and
// checkpoints. Every step of the method runs in the kernels of lbm_kernels.cuh.
#include <cuda_runtime.h>
#include <cudaTypedefs.h>  // PFN_cuTensorMapEncodeTiled (fetched at run time; no link to the driver library)

#include <mutex>
#include <vector>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>

#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_kernels.cuh"
#include "lbm_tile.cuh"

namespace {

constexpr int STRIP = lbm::STRIP;  // widest strip (columns per CTA)
// threads per CTA of the step kernels of a precision and staging choice
inline int cta_threads(int precision, bool staged)
{
    if (precision == 64) return staged ? lbm::threads_per_cta<double, true>() : lbm::threads_per_cta<double, false>();
    return staged ? lbm::threads_per_cta<float, true>() : lbm::threads_per_cta<float, false>();
}
constexpr size_t ALIGN = 256;
constexpr uint64_t CKPT_MAGIC = 0x4C424D434B505431ull;  // "LBMCKPT1"

size_t align_up(size_t v) { return (v + ALIGN - 1) / ALIGN * ALIGN; }

// Host-side fault injection for the failure-detection tests (read at every
// lbm_init): LBM_FAULT=alloc fails lbm_init as if its last device allocation
// had failed, after the workspace was allocated, so the error path's clean-up
// runs; LBM_FAULT=param fails it as if the thermodynamics had no solution.
// CTAs whose share of the work is under this many rows per strip take the
// row-pair kernel that issues a segment's first three stage pairs together
// (measured: 4096 x 512 +8.6%, 1024 x 128 +6%; 16384 x 2048, ~358 rows per
// CTA, 0.9% slower with it)
constexpr long long EARLY_ROWS = 128;

bool fault_is(const char *kind)
{
    const char *f = std::getenv("LBM_FAULT");
    return f && std::strcmp(f, kind) == 0;
}

struct Layout {
    size_t pops;      // one population array
    size_t f0, f1, mass, J, ext, err, dout, total;
    size_t rho, side;  // in-place contexts: density plane and pressure-column side buffer
};

// inplace: one population array (f1 = f0) plus the density plane and the side
// buffer of the in-place step
Layout layout_of(int nx, int ny, int precision, bool inplace = false)
{
    Layout L{};
    const size_t sz = precision == 64 ? 8 : 4;
    L.pops = align_up((size_t)9 * lbm::pitch_of(nx) * ny * sz);
    size_t o = 0;
    L.f0 = o; o += L.pops;
    if (inplace) {
        L.f1 = L.f0;
        L.rho = o; o += align_up((size_t)lbm::pitch_of(nx) * ny * sz);
        L.side = o; o += align_up((size_t)2 * 9 * ny * sz);
    } else {
        L.f1 = o; o += L.pops;
    }
    L.mass = o; o += align_up(lbm::MAX_CTAS * sizeof(double));
    L.J = o; o += align_up(lbm::MAX_CTAS * sizeof(double));
    L.ext = o; o += align_up((size_t)lbm::MAX_CTAS * 4 * sz);
    L.err = o; o += align_up(sizeof(int));
    L.dout = o; o += align_up(8 * sizeof(double));
    L.total = o;
    return L;
}

// big: a context may take 64-bit population offsets (node indices, and the
// 9 ny plane-rows of a tensor map, stay below 2^31); otherwise 9 pitch ny < 2^31.
bool grid_ok(const lbm_grid *g, bool big = false)
{
    if (!g) return false;
    if (g->precision != 32 && g->precision != 64) return false;
    if (g->walls != 0 && g->walls != 1) return false;
    if (g->bc_x != 0 && g->bc_x != 1) return false;
    if (g->nx < (g->bc_x ? 4 : 1) || g->ny < (g->walls ? 4 : 1)) return false;
    if (big) return (long long)lbm::pitch_of(g->nx) * g->ny < (1ll << 31) && 9ll * g->ny < (1ll << 31);
    return lbm::idx32_ok(g->nx, g->ny);
}

} // namespace

struct lbm_ctx {
    lbm_grid grid{};
    lbm_eos eos{};
    lbm_drive drive{};
    double tau = 1.0, wet = 0.0;
    double T = 0, Tc = 0, rho_g = 0, rho_l = 0, p_sat = 0, rho_in = 0, rho_out = 0;
    double rho_in_l = 0, rho_out_l = 0;
    lbm::Thermo th{};  // EOS at the working temperature
    lbm_collision coll{};  // BGK unless lbm_set_collision chose MRT
    cudaStream_t stream = nullptr;
    unsigned char *ws = nullptr;
    bool own_ws = false;
    Layout L{};
    int cur = 0;          // which population array holds the current state
    // in-place streaming (lbm_init_inplace): one population array, cur = 0;
    // aa_odd: the array holds the odd-parity layout (after an odd number of
    // in-place steps since it last held the natural one)
    bool inplace = false, aa_odd = false;
    lbm::AAPlan aa{};
    // its FP32 step by row pairs in place (long segments): strip plan and maps
    struct { bool on; int W, nstrips, nctas, band; long long units; } aas{};
    CUtensorMap tmap_aa[3];  // boxes of AA_SP columns by 9, 1 and 2 planes
    int64_t step = 0;
    int W = STRIP, nstrips = 0, yf0 = 0, nyf = 0;
    int W_opt = 0;  // LBM_OPT_STRIP (0: widest)
    int pitch = 0;  // plane pitch of the population rows (>= nx)
    bool big = false;  // 9 pitch ny >= 2^31: kernels with 64-bit population offsets
    bool early = false;  // row-pair kernel issuing a segment's first three stage pairs together
    bool pdl = true;     // LBM_OPT_PDL: row-pair steps launched with programmatic serialization
    long long units = 0;
    int band = 0;  // rows per band of the work-unit order
    int nctas = 0;
    int ctas_per_sm_opt = 0;
    int reverse = 0;
    int sms = 0;
    bool allow_staged = true;  // LBM_OPT_STAGED
    bool staged = false;       // bulk-copy staged kernel selected for this grid
    bool allow_rows2 = true;   // LBM_OPT_ROWS2
    bool rows2 = false;        // row-pair FP32 step kernel selected for this grid
    bool allow_tma = true;     // LBM_OPT_TMA
    int pf = 0;                // LBM_OPT_PREFETCH (row pairs ahead, 0 = off)
    // general wall geometry (lbm_mask.cu): set when the mask adds solid nodes
    // to the wall rows, or when LBM_OPT_GENERAL forces that path
    lbm::MaskPath *mask = nullptr;
    bool mask_rows2 = false;  // its FP32 step by row pairs, over the row-pair plan
    std::vector<uint8_t> mask_host;  // the caller's mask (empty: none)
    bool force_general = false;
    bool fault_skip = false;  // LBM_OPT_FAULT_SKIP_COPY (test hook)
    // graph replay of lbm_step: graph_steps launches captured from buffer 0
    // (contexts with a stream of their own; LBM_OPT_GRAPH_STEPS)
    int graph_steps = 64;
    cudaGraphExec_t graph = nullptr;
    bool tma_ok = false;       // tmap[] encoded (FP32, pitch a multiple of 4)
    CUtensorMap tmap[2];       // 2-D views of the two population buffers for the row-pair stage
    bool tile_maps_ok = false;  // tmap_tile[] encoded
    CUtensorMap tmap_tile[2];   // the same views with the tile kernel's boxes (T_BOX x 9)
    bool allow_tile = false;    // LBM_OPT_TILE (measured slower than the row-pair kernel)
    bool t64 = false;           // FP64: the tile kernel (lbm_tile64.cu) for the step and the fields
    lbm::Tile64 t64p{};
    bool tile = false;          // the plan steps with step_kernel_tile (ntx tiles along x)
    int ntx = 0;
    // fields scratch (allocated on first host-pointer lbm_fields)
    unsigned char *fscratch = nullptr;
    size_t fscratch_bytes = 0;
    // non-blocking NaN check
    int *h_err = nullptr;
    cudaEvent_t err_ev = nullptr;
    bool err_pending = false;
    char last_error[512] = {0};
};

namespace {

lbm_status cuda_fail(lbm_ctx *c, cudaError_t e, const char *where)
{
    if (c) std::snprintf(c->last_error, sizeof c->last_error, "%s: %s", where, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
}

#define CK(call, where)                                            \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, where);   \
    } while (0)

template <typename real>
lbm::KArgs<real> make_args(const lbm_ctx *ctx)
{
    lbm::KArgs<real> A{};
    const int src = ctx->cur, dst = 1 - ctx->cur;
    A.fin = (const real *)(ctx->ws + (src ? ctx->L.f1 : ctx->L.f0));
    A.fout = (real *)(ctx->ws + (dst ? ctx->L.f1 : ctx->L.f0));
    A.plane = (long long)ctx->grid.nx * ctx->grid.ny;
    A.nx = ctx->grid.nx;
    A.ny = ctx->grid.ny;
    A.pitch = ctx->pitch;
    A.W = ctx->W;
    A.nstrips = ctx->nstrips;
    A.yf0 = ctx->yf0;
    A.nyf = ctx->nyf;
    A.units = ctx->units;
    A.band = ctx->band;
    A.nctas = ctx->nctas;
    A.reverse = ctx->reverse;
    const double k = ctx->eos.k;
    A.RT = (real)(ctx->eos.R * ctx->T);
    A.a = (real)ctx->eos.a;
    A.b4 = (real)(0.25 * ctx->eos.b);
    A.k2 = (real)(k * k);
    A.kappa = (real)ctx->eos.kappa;
    A.tau = (real)ctx->tau;
    A.inv_tau = (real)(1.0 / ctx->tau);
    A.omb = (real)(1.0 - 1.0 / ctx->tau);
    A.gx = (real)ctx->drive.gx;
    A.gy = (real)ctx->drive.gy;
    A.wet = (real)ctx->wet;
    A.rho_in_g = (real)ctx->rho_in;
    A.rho_in_l = (real)ctx->rho_in_l;
    A.rho_out_g = (real)ctx->rho_out;
    A.rho_out_l = (real)ctx->rho_out_l;
    A.ph_g = (real)ctx->rho_g;
    A.inv_dph = ctx->rho_l > ctx->rho_g ? (real)(1.0 / (ctx->rho_l - ctx->rho_g)) : real(0);
    lbm::args64(A, ctx->eos.kappa, ctx->eos.k * ctx->eos.k, ctx->eos.R * ctx->T, ctx->eos.a, ctx->tau);
    A.nu = (real)((ctx->tau - 0.5) / 3.0);
    A.eos_kind = ctx->th.kind;
    A.bpr = (real)ctx->th.b;
    A.aalpha = (real)ctx->th.aalpha;
    const lbm_collision &cl = ctx->coll;
    A.mrt = cl.kind == LBM_COLL_MRT;
    A.ushift = A.mrt ? (real)(1.0 / cl.s_j) : (real)ctx->tau;
    if (A.mrt) {
        const double s_nu = cl.s_nu > 0 ? cl.s_nu : 1.0 / ctx->tau;
        A.m_e = (real)(cl.s_e / 36.0); A.m_eps = (real)(cl.s_eps / 36.0);
        A.m_j = (real)(cl.s_j / 6.0); A.m_q = (real)(cl.s_q / 12.0); A.m_nu = (real)(s_nu / 4.0);
    }
    A.mass_part = (double *)(ctx->ws + ctx->L.mass);
    A.J_acc = (double *)(ctx->ws + ctx->L.J);
    A.ext = (real *)(ctx->ws + ctx->L.ext);
    A.err = (int *)(ctx->ws + ctx->L.err);
    return A;
}

template <typename real, bool STAGED, bool PADDED>
void *kernel_ptr(bool walls, bool pres)
{
    using namespace lbm;
    if (walls && pres) return (void *)step_kernel<real, true, true, STAGED, PADDED>;
    if (walls) return (void *)step_kernel<real, true, false, STAGED, PADDED>;
    if (pres) return (void *)step_kernel<real, false, true, STAGED, PADDED>;
    return (void *)step_kernel<real, false, false, STAGED, PADDED>;
}

template <typename real>
void *kernel_ptr(bool walls, bool pres, bool staged, bool padded)
{
    if (staged) return padded ? kernel_ptr<real, true, true>(walls, pres) : kernel_ptr<real, true, false>(walls, pres);
    return padded ? kernel_ptr<real, false, true>(walls, pres) : kernel_ptr<real, false, false>(walls, pres);
}

}  // namespace

namespace {
lbm_status aa_natural(lbm_ctx *ctx);
}  // namespace

namespace {

template <bool PADDED, int EARLY>
void *rows2_kernel_ptr(bool walls, bool pres)
{
    using namespace lbm;
    if (walls && pres) return (void *)step_kernel_rows2<true, true, PADDED, false, int, EARLY>;
    if (walls) return (void *)step_kernel_rows2<true, false, PADDED, false, int, EARLY>;
    if (pres) return (void *)step_kernel_rows2<false, true, PADDED, false, int, EARLY>;
    return (void *)step_kernel_rows2<false, false, PADDED, false, int, EARLY>;
}


void *step_kernel_ptr(const lbm_ctx *ctx)
{
    const bool padded = ctx->pitch != ctx->grid.nx;
    if (ctx->big) {
        if (ctx->rows2) return lbm_big_rows2_kernel_ptr(ctx->grid.walls, ctx->grid.bc_x, padded);
        return lbm_big_step_kernel_ptr(ctx->grid.precision, ctx->grid.walls, ctx->grid.bc_x, ctx->staged, padded);
    }
    if (ctx->rows2) {
        if (ctx->early)
            return padded ? rows2_kernel_ptr<true, 3>(ctx->grid.walls, ctx->grid.bc_x)
                          : rows2_kernel_ptr<false, 3>(ctx->grid.walls, ctx->grid.bc_x);
        return padded ? rows2_kernel_ptr<true, 1>(ctx->grid.walls, ctx->grid.bc_x)
                      : rows2_kernel_ptr<false, 1>(ctx->grid.walls, ctx->grid.bc_x);
    }
    return ctx->grid.precision == 64 ? kernel_ptr<double>(ctx->grid.walls, ctx->grid.bc_x, ctx->staged, padded)
                                     : kernel_ptr<float>(ctx->grid.walls, ctx->grid.bc_x, ctx->staged, padded);
}

size_t dyn_smem(const lbm_ctx *ctx)
{
    if (!ctx->staged) return 0;
    if (ctx->rows2) return lbm::rows2_smem_bytes();
    return ctx->grid.precision == 64 ? lbm::staged_smem_bytes<double>()
                                     : lbm::staged_smem_bytes<float>();
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    static std::mutex m;
    std::lock_guard<std::mutex> lock(m);
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    }
    return fn;
}

// The 2-D view of one FP32 population buffer that the row-pair stage reads:
// x = column (pitch wide, stride 4 pitch bytes per y), y = 9 * row + plane;
// boxes of R2_SP columns by 9 planes (one stencil row), zero fill outside.
bool encode_population_map(CUtensorMap *map, void *base, int pitch, int ny, int box_cols = lbm::R2_SP,
                           unsigned box_planes = 9)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc || pitch % 4 != 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)pitch, (cuuint64_t)9 * (cuuint64_t)ny};
    const cuuint64_t strides[1] = {(cuuint64_t)pitch * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, box_planes};
    const cuuint32_t elem[2] = {1u, 1u};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int threads_of(const lbm_ctx *ctx)
{
    if (ctx->t64) return ctx->t64p.threads;
    if (ctx->rows2) return lbm::R2_BLOCK;
    return cta_threads(ctx->grid.precision, ctx->staged);
}

// Band height of the work-unit order: about one CTA's share of rows, so that
// consecutive CTAs hold neighbouring strips of one band (at least 8 rows; the
// whole column, i.e. strip-major order, when there are fewer CTAs than
// strips). With walls no band boundary may fall between fluid rows 1|2 or
// ny-3|ny-2 (fluid offsets 1 and nyf-1).
//
// A segment costs its rows and about five more for its halo, so a last band of one
// to five rows (and more than one strip) is avoided: its CTAs would march through
// many short segments, and the step waits for them. The next height that leaves six
// or none: no higher, since far above the share a CTA's rows lie in two strips, out
// of step with their neighbours (14491 x 1739, share 268: 355 us a step; bands of 276
// and 308, 376 and 462). FP32 row pairs, us per step with the share and with the band
// chosen: 1999 x 1500, last band of 4 rows, 58.6 and 51.1 (walls: 2 rows, 79.9 and
// 57.6); 5343 x 1244, 3 rows, 143 and 98.6; 1180 x 741, 1 row, 37.4 and 21.2. Six
// rows or more do not show (4096 x 1024, 46 and 47: 10 and 35 rows, 73.1 and 72.9).
int band_rows(int nyf, int nstrips, int nctas, int walls)
{
    const long long share = ((long long)nyf * nstrips + nctas - 1) / nctas;
    int band = (int)std::min<long long>(nyf, std::max<long long>(8, share));
    auto fits = [&](int b) { return !walls || b >= nyf || (nyf - 1) % b != 0; };
    while (!fits(band)) ++band;
    const int last = nyf % band;
    if (nstrips > 1 && last > 0 && last < 6 && share >= std::max(6, 2 * last + 2))
        for (int b = band + 1; b <= band + std::max(3, band / 4) && b < nyf; ++b)
            if (fits(b) && (nyf % b == 0 || nyf % b >= 6)) { band = b; break; }
    return std::max(1, band);
}

// CTAs of the strip plan with per_sm of them resident on an SM, and its bands.
void plan_strip_ctas(lbm_ctx *ctx, int per_sm)
{
    long long n = (long long)ctx->sms * per_sm;
    n = std::min<long long>(n, std::max<long long>(1, ctx->units / 2));
    n = std::min<long long>(n, lbm::MAX_CTAS);
    ctx->nctas = (int)std::max<long long>(1, n);
    ctx->band = band_rows(ctx->nyf, ctx->nstrips, ctx->nctas, ctx->grid.walls);
}

// Strip partition and the CTA count of the step grid.
lbm_status plan_launch(lbm_ctx *ctx)
{
    const int nx = ctx->grid.nx;
    const int wmax = std::min(ctx->W_opt > 0 ? ctx->W_opt : STRIP, STRIP);
    int W = lbm::strip_width(nx, wmax, ctx->grid.bc_x);
    // bulk-copy staging needs 16-byte aligned row segments
    ctx->staged = ctx->allow_staged && (ctx->pitch % 4 == 0) && (W % 4 == 0);
    // row pairs: FP32 staged grids with strips of at most R2_W columns (a
    // multiple of 4)
    ctx->rows2 = ctx->allow_rows2 && ctx->staged && ctx->grid.precision == 32 &&
                 lbm::cols_per_thread<float, true>() == 1;
    const int W2 = ctx->rows2 ? lbm::strip_width(nx, std::min(wmax, lbm::R2_W), ctx->grid.bc_x) : 0;
    if (W2 % 4 != 0) ctx->rows2 = false;
    const bool plain = ctx->mask_host.empty() && !ctx->force_general;  // no solid nodes
    constexpr long long TILE_NODES = 4096;  // see below
    const bool t32 = ctx->rows2 && !ctx->big && !ctx->fault_skip && !ctx->allow_tile && ctx->ctas_per_sm_opt == 0 &&
                     plain && ctx->W_opt == 0 && (long long)nx * ctx->grid.ny <= TILE_NODES * ctx->sms;
    ctx->yf0 = ctx->grid.walls ? 1 : 0;
    ctx->nyf = ctx->grid.walls ? ctx->grid.ny - 2 : ctx->grid.ny;
    if (ctx->rows2 && plain && !t32 && !ctx->allow_tile && !ctx->grid.bc_x && nx % 4 != 0) {
        // Odd periodic widths that one or two strips of one row a thread (128 columns)
        // hold, but not as many of row pairs (124). Us per step, row pairs against one
        // row: 125 x 48000, 167 and 125 (walls: 184 and 132); 125 x 6400, 30 and 29 (33
        // and 30). With two strips against three it depends on the rows that a CTA
        // marches: 250 x 3200, 13 rows, 26 and 28 (27 and 33); 250 x 8000, 32 rows, 49
        // and 51 (55 and 52); 250 x 24000, 95 rows, 126 and 122 (144 and 128). From
        // three on row pairs are as fast or faster (381 x 15748: 111 and 123; 128 and 128).
        const int n1 = (nx + W - 1) / W, n2 = (nx + W2 - 1) / W2;
        const long long rows = (long long)n2 * ctx->nyf / (5 * ctx->sms);
        if (n2 > n1 && (n1 == 1 || (n1 == 2 && rows >= (ctx->grid.walls ? 24 : 64)))) ctx->rows2 = false;
    }
    if (ctx->rows2) W = W2;
    ctx->W = W;
    ctx->nstrips = (nx + W - 1) / W;
    ctx->units = (long long)ctx->nstrips * ctx->nyf;
    ctx->early = false;  // chosen once the CTA count is known
    ctx->t64 = false;    // likewise

    {
        cudaError_t e = cudaFuncSetAttribute(step_kernel_ptr(ctx), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)dyn_smem(ctx));
        if (e != cudaSuccess) return cuda_fail(ctx, e, "smem attribute");
    }
    int per_sm = ctx->ctas_per_sm_opt;
    if (per_sm <= 0) {
        int occ = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &occ, step_kernel_ptr(ctx), threads_of(ctx), dyn_smem(ctx));
        if (e != cudaSuccess) return cuda_fail(ctx, e, "occupancy");
        per_sm = std::max(1, occ);
    }
    plan_strip_ctas(ctx, per_sm);
    if (ctx->rows2 && !ctx->big && ctx->units < EARLY_ROWS * ctx->nctas) {
        ctx->early = true;
        cudaError_t e = cudaFuncSetAttribute(step_kernel_ptr(ctx), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)dyn_smem(ctx));
        if (e != cudaSuccess) return cuda_fail(ctx, e, "smem attribute");
    }
    // Tiles (lbm_tile64.cuh): FP64 always (us per step, strips against tiles, between
    // pressure columns: 1024 x 256, 123 and 91; 4096 x 512, 628 and 552; 16384 x 2048, 9490
    // and 8440; periodic: 1024 x 256, 95 and 83; 4096 x 512, 507 and 523, and from there
    // on strips are 3 to 10% faster, which this rule leaves unused), FP32
    // up to 4096 nodes per SM, where a row-pair CTA marches so few rows that the
    // densities above and below its segment cost as much as its own (us per step, row
    // pairs against tiles: 512 x 128, 7.3 and 5.3; 1024 x 256, 12.6 and 10.0; 2048 x 256,
    // 3449 nodes per SM, 17.3 and 16.1; 2048 x 290, 3907, 18.2 and 17.7; 2048 x 320, 4312,
    // 19.2 and 19.3; 4096 x 512, 13797, 47 and 57). The strip kernels remain for an
    // explicit strip width or CTA count, unstaged runs and solid nodes.
    if ((ctx->grid.precision == 64 || t32) && ctx->allow_staged && ctx->W_opt == 0) {
        cudaError_t e = lbm::tile64_plan(ctx->grid.precision, nx, ctx->grid.ny, ctx->grid.walls, ctx->grid.bc_x, ctx->big, ctx->sms, &ctx->t64p);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "occupancy");
        ctx->t64 = true;
        ctx->nctas = ctx->t64p.ctas;
        if (ctx->ctas_per_sm_opt > 0)
            ctx->nctas = (int)std::min<long long>({(long long)ctx->sms * ctx->ctas_per_sm_opt, ctx->t64p.ntiles,
                                                   lbm::MAX_CTAS});
        lbm::tile64_rotate(&ctx->t64p, ctx->grid.bc_x && ctx->grid.precision == 64, ctx->nctas);
    }
    // short segments with tensor-load staging: one CTA per 32 x 8 tile instead
    // (no tile boundary between the wall-shear rows ny-3 | ny-2, and the
    // outlet column never alone in a tile: its stencil reaches two columns back)
    ctx->tile = false;
    if (ctx->early && ctx->allow_tile && ctx->tile_maps_ok && ctx->allow_tma && !ctx->fault_skip) {
        const int nx = ctx->grid.nx;
        const long long ntx = (nx + lbm::T_TX - 1) / lbm::T_TX, nty = (ctx->nyf + lbm::T_TY - 1) / lbm::T_TY;
        bool ok = ntx * nty <= lbm::MAX_CTAS;
        if (ctx->grid.walls) ok = ok && (ctx->nyf - 1) % lbm::T_TY != 0;
        if (ctx->grid.bc_x) ok = ok && nx % lbm::T_TX != 1;
        if (ok) {
            void *fn = ctx->grid.walls ? (ctx->grid.bc_x ? (void *)lbm::step_kernel_tile<true, true>
                                                         : (void *)lbm::step_kernel_tile<true, false>)
                                       : (ctx->grid.bc_x ? (void *)lbm::step_kernel_tile<false, true>
                                                         : (void *)lbm::step_kernel_tile<false, false>);
            cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)lbm::tile_smem_bytes());
            if (e != cudaSuccess) return cuda_fail(ctx, e, "smem attribute");
            ctx->tile = true;
            ctx->ntx = (int)ntx;
            ctx->nctas = (int)(ntx * nty);
        }
    }
    return LBM_OK;
}

// src_map: tensor map of A.fin where that is not the context's current buffer
template <typename real>
cudaError_t launch(lbm_ctx *ctx, const lbm::KArgs<real> &A, const CUtensorMap *src_map = nullptr)
{
    if (ctx->t64)
        return lbm::tile64_launch<real>(A, ctx->grid.walls, ctx->grid.bc_x, ctx->big, ctx->t64p, ctx->nctas,
                                        ctx->stream);
    void *fn = step_kernel_ptr(ctx);
    if (ctx->tile) {
        // one CTA per 32 x 8 tile, every stencil row staged by a tensor load
        lbm::KArgs<real> B = A;
        fn = ctx->grid.walls ? (ctx->grid.bc_x ? (void *)lbm::step_kernel_tile<true, true>
                                               : (void *)lbm::step_kernel_tile<true, false>)
                             : (ctx->grid.bc_x ? (void *)lbm::step_kernel_tile<false, true>
                                               : (void *)lbm::step_kernel_tile<false, false>);
        int ntx = ctx->ntx;
        void *args[] = {(void *)&B, (void *)&ctx->tmap_tile[ctx->cur], (void *)&ntx};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctx->nctas);
        cfg.blockDim = dim3(lbm::T_THREADS);
        cfg.dynamicSmemBytes = lbm::tile_smem_bytes();
        cfg.stream = ctx->stream;
        cfg.attrs = at;
        cfg.numAttrs = ctx->pdl ? 1 : 0;
        return cudaLaunchKernelExC(&cfg, fn, args);
    }
    if (ctx->rows2) {
        // the row-pair kernel also takes the tensor map of its source buffer
        static const CUtensorMap unused{};
        lbm::KArgs<real> B = A;
        B.tma = ctx->tma_ok && ctx->allow_tma;
        B.pf = ctx->pf;
        if (ctx->fault_skip) {
            B.poll_limit = 4096;
            fn = (void *)lbm::step_kernel_rows2<true, true, false, true>;
        }
        const CUtensorMap *m = !B.tma ? &unused : (src_map ? src_map : &ctx->tmap[ctx->cur]);
        void *args[] = {(void *)&B, (void *)m};
        if (ctx->pdl && ctx->early && !ctx->fault_skip) {
            // programmatic dependent launch: the kernel waits for the previous
            // grid before touching memory, so its launch and set-up overlap
            // the previous step's tail (short-segment plans: config 2 +2.9%;
            // the benchmark channel measured 0.1% slower with it)
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[0].val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(ctx->nctas);
            cfg.blockDim = dim3(threads_of(ctx));
            cfg.dynamicSmemBytes = dyn_smem(ctx);
            cfg.stream = ctx->stream;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            return cudaLaunchKernelExC(&cfg, fn, args);
        }
        return cudaLaunchKernel(fn, dim3(ctx->nctas), dim3(threads_of(ctx)), args, dyn_smem(ctx),
                                ctx->stream);
    }
    void *args[] = {(void *)&A};
    return cudaLaunchKernel(fn, dim3(ctx->nctas), dim3(threads_of(ctx)), args, dyn_smem(ctx),
                            ctx->stream);
}

void drop_graph(lbm_ctx *ctx)
{
    if (ctx->graph) cudaGraphExecDestroy(ctx->graph);
    ctx->graph = nullptr;
}

template <typename real>
lbm_status do_steps(lbm_ctx *ctx, int64_t n);

// graph_steps steps starting from buffer 0, captured once and replayed (the
// captured launches hold the kernel arguments of that moment: any change of
// plan, option or collision drops the graph)
template <typename real>
lbm_status build_graph(lbm_ctx *ctx)
{
    cudaGraph_t g = nullptr;
    CK(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal), "graph capture");
    const int cur0 = ctx->cur;
    const bool odd0 = ctx->aa_odd;
    const int64_t step0 = ctx->step;
    const int keep = ctx->graph_steps;
    ctx->graph_steps = 0;  // capture single launches
    lbm_status st = do_steps<real>(ctx, keep);
    ctx->graph_steps = keep;
    cudaError_t e2 = cudaStreamEndCapture(ctx->stream, &g);
    ctx->cur = cur0;  // capture records; nothing ran
    ctx->aa_odd = odd0;
    ctx->step = step0;
    if (st != LBM_OK) { if (g) cudaGraphDestroy(g); return st; }
    if (e2 != cudaSuccess) return cuda_fail(ctx, e2, "graph end capture");
    cudaError_t e = cudaGraphInstantiate(&ctx->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) { ctx->graph = nullptr; return cuda_fail(ctx, e, "graph instantiate"); }
    return LBM_OK;
}

// the phase lbm_step's graphs start from: buffer 0, or for in-place
// contexts the natural layout
int phase_of(const lbm_ctx *ctx) { return ctx->inplace ? (ctx->aa_odd ? 1 : 0) : ctx->cur; }

template <typename real>
lbm_status one_step(lbm_ctx *ctx)
{
    lbm::KArgs<real> A = make_args<real>(ctx);
    if (ctx->inplace && ctx->aas.on) {
        lbm::KArgs<float> B = make_args<float>(ctx);
        B.W = ctx->aas.W;
        B.nstrips = ctx->aas.nstrips;
        B.units = ctx->aas.units;
        B.nctas = ctx->aas.nctas;
        B.band = ctx->aas.band;
        cudaError_t e = lbm::aa_strips_step(B, (float *)(ctx->ws + ctx->L.f0), (float *)(ctx->ws + ctx->L.rho), ctx->tmap_aa,
                                            ctx->grid.walls, ctx->aa_odd, ctx->big, ctx->sms, ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "in-place step launch");
        ctx->aa_odd = !ctx->aa_odd;
        ctx->step += 1;
        return LBM_OK;
    }
    if (ctx->inplace) {
        cudaError_t e = lbm::aa_step<real>(A, (real *)(ctx->ws + ctx->L.f0), (real *)(ctx->ws + ctx->L.rho),
                                           (real *)(ctx->ws + ctx->L.side), ctx->grid.walls, ctx->grid.bc_x,
                                           ctx->aa_odd, ctx->big, ctx->aa, ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "in-place step launch");
        ctx->aa_odd = !ctx->aa_odd;
        ctx->step += 1;
        return LBM_OK;
    }
    cudaError_t e;
    if (!ctx->mask) {
        e = launch<real>(ctx, A);
    } else if (sizeof(real) == 4 && ctx->mask_rows2) {
        lbm::KArgs<float> B = make_args<float>(ctx);
        B.tma = ctx->tma_ok && ctx->allow_tma;
        B.pf = ctx->pf;
        e = lbm::mask_rows2_launch(ctx->mask, B, &ctx->tmap[ctx->cur], ctx->early, ctx->stream);
    } else {
        e = lbm::mask_launch<real>(ctx->mask, A, lbm::MODE_STEP, ctx->stream);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "step launch");
    ctx->cur = 1 - ctx->cur;
    ctx->step += 1;
    return LBM_OK;
}

template <typename real>
lbm_status do_steps(lbm_ctx *ctx, int64_t n)
{
    // the graph starts from buffer 0: a run that starts from buffer 1 takes one
    // single launch first
    if (ctx->graph_steps > 0 && ctx->stream && phase_of(ctx) == 1 && n > ctx->graph_steps) {
        lbm_status s = one_step<real>(ctx);
        if (s != LBM_OK) return s;
        --n;
    }
    while (ctx->graph_steps > 0 && ctx->stream && n >= ctx->graph_steps && phase_of(ctx) == 0) {
        if (!ctx->graph) {
            lbm_status s = build_graph<real>(ctx);
            if (s != LBM_OK) return s;
        }
        CK(cudaGraphLaunch(ctx->graph, ctx->stream), "graph launch");
        ctx->step += ctx->graph_steps;  // an even count: the state ends in buffer 0 (natural layout) again
        n -= ctx->graph_steps;
    }
    for (int64_t s = 0; s < n; ++s) {
        lbm_status st = one_step<real>(ctx);
        if (st != LBM_OK) return st;
    }
    return LBM_OK;
}

// In-place contexts: bring the array back to the natural layout (every
// reader and writer of the state outside the step expects it); asynchronous.
lbm_status aa_natural(lbm_ctx *ctx)
{
    if (!ctx->inplace || !ctx->aa_odd) return LBM_OK;
    CK(lbm::aa_swap(ctx->grid.precision, ctx->ws + ctx->L.f0, ctx->grid.walls, ctx->grid.bc_x, ctx->big, ctx->grid.nx,
                    ctx->grid.ny, ctx->pitch, ctx->sms, ctx->stream),
       "layout swap");
    ctx->aa_odd = false;
    return LBM_OK;
}

// CTAs whose diagnostic slots hold the step's partials
int diag_ctas(const lbm_ctx *ctx)
{
    return !ctx->inplace ? ctx->nctas : (ctx->aas.on ? ctx->aas.nctas : ctx->aa.nctas);
}

template <typename real>
lbm_status do_fields(lbm_ctx *ctx, void *rho, void *ux, void *uy, void *tw, void *pw)
{
    if (lbm_status s0 = aa_natural(ctx)) return s0;
    // device destinations are written by the kernel; others (and, with a wall
    // mask, absent ones) through a scratch kept from the first call that needs it
    lbm::FieldsOut<real> o{};
    void *dst[5] = {rho, ux, uy, tw, pw};
    for (int k = 0; k < 5; ++k) o.dst[k] = dst[k];
    lbm::fields_route(o, ctx->grid.nx, ctx->grid.ny, ctx->ws, ctx->L.total);
    size_t need = o.scratch, spare = 0;
    if (ctx->mask)
        for (int k = 0; k < 5; ++k)
            if (!o.dst[k]) spare += align_up(o.bytes[k]);
    need += spare;
    if (need > ctx->fscratch_bytes) {
        if (ctx->fscratch) cudaFree(ctx->fscratch);
        ctx->fscratch = nullptr;
        ctx->fscratch_bytes = 0;
        CK(cudaMalloc((void **)&ctx->fscratch, need), "fields scratch");
        ctx->fscratch_bytes = need;
    }
    o.use(ctx->fscratch);
    lbm::KArgs<real> A = make_args<real>(ctx);
    if (ctx->mask) {
        A.fout = nullptr;
        // solid nodes read zero: one pass over the scratch outputs, one over each
        // direct one, none over those that nobody asked for
        real *p[5];
        size_t at = o.scratch;
        if (o.scratch) CK(cudaMemsetAsync(ctx->fscratch, 0, o.scratch, ctx->stream), "fields memset");
        for (int k = 0; k < 5; ++k) {
            p[k] = o.ptr[k];
            if (!p[k]) {
                p[k] = (real *)(ctx->fscratch + at);
                at += align_up(o.bytes[k]);
            } else if ((void *)p[k] == o.dst[k]) {
                CK(cudaMemsetAsync(p[k], 0, o.bytes[k], ctx->stream), "fields memset");
            }
        }
        A.o_rho = p[0]; A.o_vx = p[1]; A.o_vy = p[2]; A.o_tw = p[3]; A.o_pw = p[4];
        CK(lbm::mask_launch<real>(ctx->mask, A, lbm::MODE_FIELDS, ctx->stream), "fields launch");
    } else {
        CK(lbm::fields_tiles<real>(A, o, ctx->grid.walls, ctx->grid.bc_x, ctx->big, ctx->sms, ctx->stream), "fields launch");
    }
    CK(lbm::fields_copy(o, ctx->stream), "fields copy");
    CK(cudaStreamSynchronize(ctx->stream), "fields sync");
    return LBM_OK;
}

template <typename real>
void reset_acc(lbm_ctx *ctx)
{
    lbm::reset_acc_kernel<real><<<(lbm::MAX_CTAS + 255) / 256, 256, 0, ctx->stream>>>(
        (double *)(ctx->ws + ctx->L.mass), (double *)(ctx->ws + ctx->L.J),
        (real *)(ctx->ws + ctx->L.ext), (int *)(ctx->ws + ctx->L.err), lbm::MAX_CTAS);
}

// The library stores populations row-interleaved, f[y][i][x] with plane
// pitch P >= nx; the ABI exchanges plane-major f[i][y][x]. One strided 2D
// copy per plane converts.
cudaError_t copy_planes(const lbm_ctx *ctx, void *dst, const void *src, bool to_abi)
{
    const size_t sz = ctx->grid.precision == 64 ? 8 : 4;
    const size_t nx = ctx->grid.nx, ny = ctx->grid.ny, row = nx * sz, prow = (size_t)ctx->pitch * sz;
    for (int i = 0; i < 9; ++i) {
        cudaError_t e;
        if (to_abi)
            e = cudaMemcpy2DAsync((char *)dst + i * nx * ny * sz, row, (const char *)src + i * prow, 9 * prow,
                                  row, ny, cudaMemcpyDefault, ctx->stream);
        else
            e = cudaMemcpy2DAsync((char *)dst + i * prow, 9 * prow, (const char *)src + i * nx * ny * sz, row,
                                  row, ny, cudaMemcpyDefault, ctx->stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

struct CkptHeader {
    uint64_t magic;
    int32_t nx, ny, walls, bc_x, precision, nctas;
    int64_t step;
    int32_t cur, inplace;  // inplace: one population array (in the natural layout) follows
};

} // namespace

namespace {
// A checkpoint's per-CTA partials for a plan of n CTAs: those of a plan with
// more CTAs (m) are folded into the first n, so that the totals stay.
template <typename real>
void fold_partials(double *mass, double *J, real *ext, int n, int m)
{
    for (int c = n; c < m; ++c) {
        mass[c % n] += mass[c];
        J[c % n] += J[c];
        mass[c] = J[c] = 0.0;
        real *to = ext + 4 * (c % n), *from = ext + 4 * c;
        for (int k = 0; k < 4; ++k) {
            to[k] = k & 1 ? std::max(to[k], from[k]) : std::min(to[k], from[k]);
            from[k] = k & 1 ? -INFINITY : INFINITY;
        }
    }
}
} // namespace

bool lbm_encode_population_map(CUtensorMap *map, void *base, int pitch, int ny)
{
    return encode_population_map(map, base, pitch, ny);
}

namespace {
template <typename real>
cudaError_t step_between(lbm_ctx *ctx, const void *fin, void *fout)
{
    lbm::KArgs<real> A = make_args<real>(ctx);
    A.fin = (const real *)fin;
    A.fout = (real *)fout;
    CUtensorMap map;
    if (ctx->tma_ok && !encode_population_map(&map, const_cast<void *>(fin), ctx->pitch, ctx->grid.ny))
        return cudaErrorInvalidValue;
    return launch<real>(ctx, A, &map);
}
}  // namespace

cudaError_t lbm_ctx_step_between(lbm_ctx *ctx, const void *fin, void *fout, cudaStream_t stream)
{
    if (ctx->inplace || ctx->mask || ctx->tile) return cudaErrorNotSupported;
    const cudaStream_t own = ctx->stream;
    ctx->stream = stream;
    const cudaError_t e =
        ctx->grid.precision == 64 ? step_between<double>(ctx, fin, fout) : step_between<float>(ctx, fin, fout);
    ctx->stream = own;
    return e;
}

int *lbm_ctx_error_word(lbm_ctx *ctx) { return (int *)(ctx->ws + ctx->L.err); }

namespace {

// In-place FP32 contexts between pressure columns whose row-pair plan gives CTAs
// AA_ROWS_MIN rows or more: the step by row pairs in place. A segment's first rows
// are filled from the density plane, so short segments keep the tiles, whose cost
// does not depend on segments (us per step, tiles against strips: 8192 x 1024,
// 94 rows, 218 and 181; 8192 x 768, 70 rows, 166 and 141; 4096 x 1024, 47 rows,
// 113 and 109; 4096 x 512, 24 rows, 53 and 65). The two cross somewhere between 24
// and 47 rows; the line is kept above both, at the cost of 4% just below it.
constexpr long long AA_ROWS_MIN = 48;
lbm_status plan_inplace_strips(lbm_ctx *ctx)
{
    auto &s = ctx->aas;
    s = {};
    const lbm_grid &g = ctx->grid;
    if (g.precision != 32 || !g.bc_x || ctx->pitch % 4 != 0) return LBM_OK;
    s.W = lbm::strip_width(g.nx, lbm::AA_W, true);
    if (s.W % 4 != 0) return LBM_OK;
    s.nstrips = (g.nx + s.W - 1) / s.W;
    s.units = (long long)s.nstrips * ctx->nyf;
    int per_sm = 0;
    cudaError_t e = lbm::aa_strips_plan(g.walls, ctx->big, &per_sm);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "in-place strip plan");
    s.nctas = (int)std::max<long long>(1, std::min<long long>({(long long)ctx->sms * std::max(1, per_sm), s.units / 2,
                                                               (long long)lbm::MAX_CTAS}));
    if (s.units < AA_ROWS_MIN * s.nctas) return LBM_OK;
    s.band = band_rows(ctx->nyf, s.nstrips, s.nctas, g.walls);
    static const unsigned planes[3] = {9, 1, 2};
    for (int k = 0; k < 3; ++k)
        if (!encode_population_map(&ctx->tmap_aa[k], ctx->ws + ctx->L.f0, ctx->pitch, g.ny, lbm::AA_SP, planes[k]))
            return LBM_OK;
    s.on = true;
    return LBM_OK;
}

// Whether an FP32 step with solid nodes runs by row pairs (else the general-geometry
// kernels, four to six of them: one more with walls, one with pressure columns). Row
// pairs pay for the nodes that their strips of W columns are padded to, the others
// for launches and for passes over memory. In us per step, row pairs against the
// others. Neither walls nor pressure columns: 256 x 256, 11.4 and 10.6; 2048 x 256,
// 25.1 and 22.1; 1024 x 1024, 37.3 and 38.4; 4096 x 1024, 95 and 153; narrow: 127 x
// 5000, 38 and 26; 97 x 60000, 172 and 214. With either, narrow lattices of middle
// size alone: 97 x 6000 (walls), 30.1 and 26.7; 250 x 3000, 34.2 and 32.1; 97 x 1000,
// 13.3 and 14.9; 97 x 60000, 157 and 212; walls and columns, 130 x 4000, 31.5 and
// 27.8; 130 x 30000, 133 and 149. Constants: nodes per SM.
bool mask_pairs(const lbm_ctx *ctx)
{
    const double sms = ctx->sms, n = (double)ctx->grid.nx * ctx->grid.ny / sms,
                 padded = (double)ctx->units * ctx->W / sms;
    if (!ctx->grid.walls && !ctx->grid.bc_x) return n > 0.6 * padded + 2150;
    const bool narrow = padded > 1.25 * n, short_runs = ctx->units / 2 <= 5 * ctx->sms;  // two rows a CTA
    return !narrow || short_runs || n > 0.46 * padded + 1645;
}

// (Re)selects the general-geometry path: kept when the caller's mask adds
// solid nodes to the wall rows or LBM_OPT_GENERAL forces it; the diagnostic
// slots then follow its CTA count.
lbm_status plan_geometry(lbm_ctx *ctx)
{
    lbm::mask_free(ctx->mask);
    ctx->mask = nullptr;
    const uint8_t *m = ctx->mask_host.empty() ? nullptr : ctx->mask_host.data();
    if (ctx->big && (m || ctx->force_general)) {
        std::snprintf(ctx->last_error, sizeof ctx->last_error,
                      "the general-geometry kernels need 9 pitch ny < 2^31");
        return LBM_ERR_ARG;
    }
    lbm_status st = lbm::mask_setup(m, ctx->grid, ctx->pitch, ctx->sms, ctx->force_general, ctx->stream, &ctx->mask,
                                    ctx->last_error, sizeof ctx->last_error);
    ctx->mask_rows2 = false;
    if (st != LBM_OK || !ctx->mask) return st;
    if (ctx->rows2 && !ctx->big && mask_pairs(ctx)) {
        // the strip plan with this kernel's own residency
        ctx->tile = false;
        int per_sm = ctx->ctas_per_sm_opt;
        for (bool early : {false, true}) {
            int occ = 0;
            cudaError_t e = lbm::mask_rows2_plan(ctx->mask, early, &occ);
            if (e != cudaSuccess) return cuda_fail(ctx, e, "mask step plan");
            if (ctx->ctas_per_sm_opt <= 0) per_sm = early ? std::min(per_sm, std::max(1, occ)) : std::max(1, occ);
        }
        plan_strip_ctas(ctx, per_sm);
        ctx->early = ctx->units < EARLY_ROWS * ctx->nctas;
        ctx->mask_rows2 = true;
        return LBM_OK;
    }
    ctx->nctas = lbm::mask_blocks(ctx->mask);
    return st;
}

}  // namespace


extern "C" {

const char *lbm_status_string(lbm_status s)
{
    switch (s) {
    case LBM_OK: return "ok";
    case LBM_ERR_ARG: return "invalid argument";
    case LBM_ERR_PARAM: return "invalid physical parameter";
    case LBM_ERR_CUDA: return "CUDA error";
    case LBM_ERR_OOM: return "out of memory";
    case LBM_ERR_NAN: return "non-finite or non-positive density";
    case LBM_ERR_STATE: return "incompatible checkpoint";
    case LBM_ERR_TIMEOUT: return "a bounded wait for staged data gave up";
    }
    return "unknown status";
}

const char *lbm_last_error(const lbm_ctx *ctx) { return ctx ? ctx->last_error : ""; }

size_t lbm_workspace_bytes(const lbm_grid *grid)
{
    if (!grid_ok(grid, true)) return 0;
    return layout_of(grid->nx, grid->ny, grid->precision).total;
}

size_t lbm_workspace_bytes_inplace(const lbm_grid *grid)
{
    if (!grid_ok(grid, true)) return 0;
    return layout_of(grid->nx, grid->ny, grid->precision, true).total;
}

} // extern "C"

namespace {

lbm_status init_ctx(const lbm_grid *grid, const lbm_eos *eos, double tau, const uint8_t *wall_mask,
                    double wetting, const lbm_drive *drive, const double *rho0, void *workspace, size_t ws_bytes,
                    void *stream, bool inplace, lbm_ctx **out)
{
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    if (!grid_ok(grid, true) || !eos || !rho0) return LBM_ERR_ARG;
    if (!(tau > 0.5) || !(eos->k > 0) || !(eos->kappa >= 0) || !(eos->a > 0) || !(eos->b > 0) ||
        !(eos->R > 0) || !(eos->T_over_Tc > 0) || !std::isfinite(wetting))
        return LBM_ERR_PARAM;

    lbm_ctx *ctx = new (std::nothrow) lbm_ctx();
    if (!ctx) return LBM_ERR_OOM;
    ctx->grid = *grid;
    ctx->eos = *eos;
    if (drive) ctx->drive = *drive;
    else { ctx->drive.dp = 0; ctx->drive.p_ref = NAN; ctx->drive.gx = ctx->drive.gy = 0; }
    ctx->tau = tau;
    ctx->wet = wetting;
    ctx->stream = (cudaStream_t)stream;

    // Thermodynamics (host FP64).
    lbm::ChannelThermo ct;
    if (lbm::channel_thermo(*eos, ctx->drive, grid->bc_x, &ct) || fault_is("param")) {
        lbm_free(ctx);
        return LBM_ERR_PARAM;
    }
    ctx->th = ct.th;
    ctx->T = ct.T; ctx->Tc = ct.Tc;
    ctx->rho_g = ct.rho_g; ctx->rho_l = ct.rho_l; ctx->p_sat = ct.p_sat;
    ctx->rho_in = ct.rho_in; ctx->rho_out = ct.rho_out;
    ctx->rho_in_l = ct.rho_in_l; ctx->rho_out_l = ct.rho_out_l;

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        lbm_status s = cuda_fail(ctx, e, "device query");
        lbm_free(ctx);
        return s;
    }

    ctx->inplace = inplace;
    ctx->L = layout_of(grid->nx, grid->ny, grid->precision, inplace);
    ctx->pitch = lbm::pitch_of(grid->nx);
    ctx->big = !lbm::idx32_ok(grid->nx, grid->ny);
    if (workspace) {
        if (ws_bytes < ctx->L.total || ((uintptr_t)workspace % ALIGN) != 0) {
            lbm_free(ctx);
            return LBM_ERR_ARG;
        }
        ctx->ws = (unsigned char *)workspace;
    } else {
        e = cudaMalloc((void **)&ctx->ws, ctx->L.total);
        if (e != cudaSuccess) {
            cudaGetLastError();
            lbm_free(ctx);
            return LBM_ERR_OOM;
        }
        ctx->own_ws = true;
    }
    e = cudaMallocHost((void **)&ctx->h_err, sizeof(int));
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->err_ev, cudaEventDisableTiming);
    if (e == cudaSuccess && fault_is("alloc")) e = cudaErrorMemoryAllocation;
    if (e != cudaSuccess) {
        lbm_status s = cuda_fail(ctx, e, "host flag");
        lbm_free(ctx);
        return s;
    }
    *ctx->h_err = 0;

    // tensor maps of both buffers (the plan chooses kernels by them)
    if (grid->precision == 32)
        ctx->tma_ok = encode_population_map(&ctx->tmap[0], ctx->ws + ctx->L.f0, ctx->pitch, grid->ny) &&
                      encode_population_map(&ctx->tmap[1], ctx->ws + ctx->L.f1, ctx->pitch, grid->ny);
    if (grid->precision == 32)
        ctx->tile_maps_ok =
            encode_population_map(&ctx->tmap_tile[0], ctx->ws + ctx->L.f0, ctx->pitch, grid->ny, lbm::T_BOX) &&
            encode_population_map(&ctx->tmap_tile[1], ctx->ws + ctx->L.f1, ctx->pitch, grid->ny, lbm::T_BOX);
    if (wall_mask) ctx->mask_host.assign(wall_mask, wall_mask + (size_t)grid->nx * grid->ny);
    lbm_status st = plan_launch(ctx);
    if (st != LBM_OK) { lbm_free(ctx); return st; }
    st = plan_geometry(ctx);
    if (st != LBM_OK) { lbm_free(ctx); return st; }
    if (inplace) {
        e = lbm::aa_plan(grid->precision, ctx->big, grid->walls, grid->bc_x, grid->nx, grid->ny, ctx->sms, &ctx->aa);
        if (e != cudaSuccess) {
            lbm_status s = cuda_fail(ctx, e, "in-place plan");
            lbm_free(ctx);
            return s;
        }
    }

    if (inplace) {
        st = plan_inplace_strips(ctx);
        if (st != LBM_OK) { lbm_free(ctx); return st; }
    }

    // Initial state f = f_eq(rho0, 0) in both arrays (in-place contexts: the
    // one array, natural layout; the kernel then stores each value twice to
    // the same slot).
    const size_t N = (size_t)grid->nx * grid->ny;
    double *d_rho0 = nullptr;
    e = cudaMallocAsync((void **)&d_rho0, N * sizeof(double), ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_rho0, rho0, N * sizeof(double), cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) {
        const int blocks = (int)std::min<size_t>((N + 255) / 256, (size_t)ctx->sms * 8);
        if (grid->precision == 64) {
            lbm::init_kernel<double><<<blocks, 256, 0, ctx->stream>>>(
                d_rho0, (double *)(ctx->ws + ctx->L.f0), (double *)(ctx->ws + ctx->L.f1), grid->nx, ctx->pitch,
                grid->ny);
            reset_acc<double>(ctx);
        } else {
            lbm::init_kernel<float><<<blocks, 256, 0, ctx->stream>>>(
                d_rho0, (float *)(ctx->ws + ctx->L.f0), (float *)(ctx->ws + ctx->L.f1), grid->nx, ctx->pitch,
                grid->ny);
            reset_acc<float>(ctx);
        }
        e = cudaGetLastError();
        cudaFreeAsync(d_rho0, ctx->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) {
        lbm_status s = cuda_fail(ctx, e, "init");
        lbm_free(ctx);
        return s;
    }
    *out = ctx;
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_init(const lbm_grid *grid, const lbm_eos *eos, double tau, const uint8_t *wall_mask,
                    double wetting, const lbm_drive *drive, const double *rho0, void *workspace, size_t ws_bytes,
                    void *stream, lbm_ctx **out)
{
    return init_ctx(grid, eos, tau, wall_mask, wetting, drive, rho0, workspace, ws_bytes, stream, false, out);
}

lbm_status lbm_init_inplace(const lbm_grid *grid, const lbm_eos *eos, double tau, double wetting,
                            const lbm_drive *drive, const double *rho0, void *workspace, size_t ws_bytes,
                            void *stream, lbm_ctx **out)
{
    return init_ctx(grid, eos, tau, nullptr, wetting, drive, rho0, workspace, ws_bytes, stream, true, out);
}

lbm_status lbm_relaxed_coexistence(const lbm_eos *eos, double tau, const lbm_collision *coll, int32_t precision,
                                   int32_t ny, int64_t steps, void *stream, double *rho_g, double *rho_l,
                                   double *p_gas, double *p_liq)
{
    if (!eos || (precision != 32 && precision != 64) || ny < 16 || steps < 0) return LBM_ERR_ARG;
    lbm::Thermo th{};
    double Tc = 0, g = 0, l = 0, ps = 0;
    if (lbm::thermo_of(*eos, &th, &Tc) || lbm::maxwell(th, &g, &l, &ps)) return LBM_ERR_PARAM;
    // a liquid slab between rows ny/4 and 3ny/4 of a periodic 4 x ny box, tanh
    // profile of width 4 between the Maxwell densities
    const int nx = 4;
    std::vector<double> rho0((size_t)nx * ny);
    for (int y = 0; y < ny; ++y) {
        const double sl = 0.5 * (std::tanh(2.0 * (y - 0.25 * ny) / 4.0) - std::tanh(2.0 * (y - 0.75 * ny) / 4.0));
        for (int x = 0; x < nx; ++x) rho0[(size_t)y * nx + x] = g + (l - g) * sl;
    }
    const lbm_grid grid{nx, ny, 0, 0, precision};
    lbm_ctx *ctx = nullptr;
    lbm_status st = lbm_init(&grid, eos, tau, nullptr, 0.0, nullptr, rho0.data(), nullptr, 0, stream, &ctx);
    if (st != LBM_OK) return st;
    if (coll) st = lbm_set_collision(ctx, coll);
    if (st == LBM_OK) st = lbm_step(ctx, steps);
    std::vector<double> r64((size_t)nx * ny);
    std::vector<float> r32((size_t)nx * ny);
    if (st == LBM_OK)
        st = lbm_fields(ctx, precision == 64 ? (void *)r64.data() : (void *)r32.data(), nullptr, nullptr, nullptr,
                        nullptr);
    if (st == LBM_OK) st = lbm_step(ctx, 0);  // the bad-density flag of the last steps
    if (st == LBM_OK) {
        lbm_diag_t d;
        st = lbm_diag(ctx, &d);
        if (st == LBM_OK && d.nan_detected) st = LBM_ERR_NAN;
    }
    lbm_free(ctx);
    if (st != LBM_OK) return st;
    auto at = [&](int y) { return precision == 64 ? r64[(size_t)y * nx] : (double)r32[(size_t)y * nx]; };
    const double rg = at(0), rl = at(ny / 2), k2 = eos->k * eos->k;
    if (rho_g) *rho_g = rg;
    if (rho_l) *rho_l = rl;
    if (p_gas) *p_gas = k2 * lbm::eos_pressure(th, rg);
    if (p_liq) *p_liq = k2 * lbm::eos_pressure(th, rl);
    return LBM_OK;
}

lbm_status lbm_step(lbm_ctx *ctx, int64_t n)
{
    if (!ctx || n < 0) return LBM_ERR_ARG;
    lbm_status flag = LBM_OK;
    if (ctx->err_pending && cudaEventQuery(ctx->err_ev) == cudaSuccess) {
        ctx->err_pending = false;
        // bit 0: bad density; bit 1: a bounded stage wait gave up
        if (*ctx->h_err & 1) flag = LBM_ERR_NAN;
        else if (*ctx->h_err) flag = LBM_ERR_TIMEOUT;
    }
    if (n == 0) return flag;
    lbm_status s = ctx->grid.precision == 64 ? do_steps<double>(ctx, n) : do_steps<float>(ctx, n);
    if (s != LBM_OK) return s;
    if (!ctx->err_pending) {
        cudaError_t e = cudaMemcpyAsync(ctx->h_err, ctx->ws + ctx->L.err, sizeof(int),
                                        cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaEventRecord(ctx->err_ev, ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "error flag");
        ctx->err_pending = true;
    }
    return flag;
}

lbm_status lbm_fields(lbm_ctx *ctx, void *rho, void *ux, void *uy, void *tau_wall, void *p_wall)
{
    if (!ctx) return LBM_ERR_ARG;
    return ctx->grid.precision == 64 ? do_fields<double>(ctx, rho, ux, uy, tau_wall, p_wall)
                                     : do_fields<float>(ctx, rho, ux, uy, tau_wall, p_wall);
}

namespace {
void enqueue_diag(lbm_ctx *ctx, double *dout)
{
    if (ctx->grid.precision == 64)
        lbm::diag_kernel<double><<<1, 256, 0, ctx->stream>>>(
            (double *)(ctx->ws + ctx->L.mass), (double *)(ctx->ws + ctx->L.J),
            (double *)(ctx->ws + ctx->L.ext), (int *)(ctx->ws + ctx->L.err), diag_ctas(ctx), dout);
    else
        lbm::diag_kernel<float><<<1, 256, 0, ctx->stream>>>(
            (double *)(ctx->ws + ctx->L.mass), (double *)(ctx->ws + ctx->L.J),
            (float *)(ctx->ws + ctx->L.ext), (int *)(ctx->ws + ctx->L.err), diag_ctas(ctx), dout);
}
}  // namespace

lbm_status lbm_diag_async(lbm_ctx *ctx, double *dst)
{
    if (!ctx || !dst || ((uintptr_t)dst % 8) != 0) return LBM_ERR_ARG;
    double *dout = (double *)(ctx->ws + ctx->L.dout);
    enqueue_diag(ctx, dout);
    CK(cudaGetLastError(), "diag launch");
    CK(cudaMemcpyAsync(dst, dout, 7 * sizeof(double), cudaMemcpyDefault, ctx->stream), "diag copy");
    return LBM_OK;
}

lbm_status lbm_diag(lbm_ctx *ctx, lbm_diag_t *out)
{
    if (!ctx || !out) return LBM_ERR_ARG;
    double *dout = (double *)(ctx->ws + ctx->L.dout);
    enqueue_diag(ctx, dout);
    CK(cudaGetLastError(), "diag launch");
    double h[8];
    CK(cudaMemcpyAsync(h, dout, 7 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream), "diag copy");
    CK(cudaStreamSynchronize(ctx->stream), "diag sync");
    std::memset(out, 0, sizeof *out);
    out->step = ctx->step;
    out->mass = ctx->step > 0 ? h[0] : 0.0;
    out->wall_shear_sum = h[1];
    const bool any = ctx->step > 0 && ctx->grid.walls;
    out->tau_wall_min = any ? h[2] : 0.0;
    out->tau_wall_max = any ? h[3] : 0.0;
    out->p_wall_min = any ? h[4] : 0.0;
    out->p_wall_max = any ? h[5] : 0.0;
    out->nan_detected = ((int)h[6] & 1) != 0;  // bit 1 (a stage wait gave up) is lbm_step's LBM_ERR_TIMEOUT
    out->T = ctx->T; out->Tc = ctx->Tc;
    out->rho_g = ctx->rho_g; out->rho_l = ctx->rho_l; out->p_sat = ctx->p_sat;
    out->rho_in = ctx->rho_in; out->rho_out = ctx->rho_out;
    out->rho_in_l = ctx->rho_in_l; out->rho_out_l = ctx->rho_out_l;
    return LBM_OK;
}

lbm_status lbm_reset_diag(lbm_ctx *ctx)
{
    if (!ctx) return LBM_ERR_ARG;
    double *mass = (double *)(ctx->ws + ctx->L.mass), *J = (double *)(ctx->ws + ctx->L.J);
    if (ctx->grid.precision == 64)
        lbm::reset_acc_kernel<double><<<(lbm::MAX_CTAS + 255) / 256, 256, 0, ctx->stream>>>(
            mass, J, (double *)(ctx->ws + ctx->L.ext), nullptr, lbm::MAX_CTAS);
    else
        lbm::reset_acc_kernel<float><<<(lbm::MAX_CTAS + 255) / 256, 256, 0, ctx->stream>>>(
            mass, J, (float *)(ctx->ws + ctx->L.ext), nullptr, lbm::MAX_CTAS);
    CK(cudaGetLastError(), "reset diag");
    return LBM_OK;
}

lbm_status lbm_populations(lbm_ctx *ctx, void *dst)
{
    if (!ctx || !dst) return LBM_ERR_ARG;
    if (lbm_status s = aa_natural(ctx)) return s;
    CK(copy_planes(ctx, dst, ctx->ws + (ctx->cur ? ctx->L.f1 : ctx->L.f0), true), "populations copy");
    CK(cudaStreamSynchronize(ctx->stream), "populations sync");
    return LBM_OK;
}

lbm_status lbm_load_populations(lbm_ctx *ctx, const void *src)
{
    if (!ctx || !src) return LBM_ERR_ARG;
    // both arrays, so never-written slots (solid rows, unreached boundary
    // slots) agree with the loaded state
    CK(copy_planes(ctx, ctx->ws + ctx->L.f0, src, false), "load copy");
    if (!ctx->inplace) CK(copy_planes(ctx, ctx->ws + ctx->L.f1, src, false), "load copy");
    ctx->aa_odd = false;
    CK(cudaStreamSynchronize(ctx->stream), "load sync");
    return LBM_OK;
}

size_t lbm_checkpoint_bytes(const lbm_ctx *ctx)
{
    if (!ctx) return 0;
    const size_t sz = ctx->grid.precision == 64 ? 8 : 4;
    return sizeof(CkptHeader) + (ctx->inplace ? 1 : 2) * ctx->L.pops + (size_t)lbm::MAX_CTAS * (16 + 4 * sz) +
           sizeof(int);
}

lbm_status lbm_checkpoint(lbm_ctx *ctx, void *host_buf, size_t bytes)
{
    if (!ctx || !host_buf || bytes < lbm_checkpoint_bytes(ctx)) return LBM_ERR_ARG;
    const size_t sz = ctx->grid.precision == 64 ? 8 : 4;
    if (lbm_status s = aa_natural(ctx)) return s;
    const int narr = ctx->inplace ? 1 : 2;
    CkptHeader h{CKPT_MAGIC, ctx->grid.nx, ctx->grid.ny, ctx->grid.walls, ctx->grid.bc_x,
                 ctx->grid.precision, diag_ctas(ctx), ctx->step, ctx->cur, ctx->inplace ? 1 : 0};
    unsigned char *p = (unsigned char *)host_buf;
    std::memcpy(p, &h, sizeof h);
    p += sizeof h;
    // both population arrays: slots no population reaches keep older values
    // (in-place contexts: the one array, in the natural layout)
    CK(cudaMemcpyAsync(p, ctx->ws + ctx->L.f0, narr * ctx->L.pops, cudaMemcpyDeviceToHost, ctx->stream), "ckpt");
    p += narr * ctx->L.pops;
    CK(cudaMemcpyAsync(p, ctx->ws + ctx->L.mass, lbm::MAX_CTAS * 8, cudaMemcpyDeviceToHost, ctx->stream), "ckpt");
    p += lbm::MAX_CTAS * 8;
    CK(cudaMemcpyAsync(p, ctx->ws + ctx->L.J, lbm::MAX_CTAS * 8, cudaMemcpyDeviceToHost, ctx->stream), "ckpt");
    p += lbm::MAX_CTAS * 8;
    CK(cudaMemcpyAsync(p, ctx->ws + ctx->L.ext, lbm::MAX_CTAS * 4 * sz, cudaMemcpyDeviceToHost, ctx->stream), "ckpt");
    p += lbm::MAX_CTAS * 4 * sz;
    CK(cudaMemcpyAsync(p, ctx->ws + ctx->L.err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream), "ckpt");
    CK(cudaStreamSynchronize(ctx->stream), "ckpt sync");
    return LBM_OK;
}

lbm_status lbm_restore(lbm_ctx *ctx, const void *host_buf, size_t bytes)
{
    if (!ctx || !host_buf || bytes < lbm_checkpoint_bytes(ctx)) return LBM_ERR_ARG;
    CkptHeader h;
    std::memcpy(&h, host_buf, sizeof h);
    if (h.magic != CKPT_MAGIC || h.nx != ctx->grid.nx || h.ny != ctx->grid.ny || h.walls != ctx->grid.walls ||
        h.bc_x != ctx->grid.bc_x || h.precision != ctx->grid.precision || (h.inplace != 0) != ctx->inplace)
        return LBM_ERR_STATE;
    const size_t sz = ctx->grid.precision == 64 ? 8 : 4;
    const int narr = ctx->inplace ? 1 : 2;
    const unsigned char *p = (const unsigned char *)host_buf + sizeof h;
    const size_t nparts = (size_t)lbm::MAX_CTAS * (16 + 4 * sz);
    const int own = diag_ctas(ctx), theirs = std::min<int>(h.nctas, lbm::MAX_CTAS);
    std::unique_ptr<unsigned char[]> part;  // folded partials, where the file's plan had more CTAs
    const unsigned char *mass = p + narr * ctx->L.pops;
    if (theirs > own) {
        part.reset(new (std::nothrow) unsigned char[nparts]);
        if (!part) return LBM_ERR_OOM;
        std::memcpy(part.get(), mass, nparts);
        mass = part.get();
        unsigned char *J = part.get() + lbm::MAX_CTAS * 8, *ext = J + lbm::MAX_CTAS * 8;
        if (ctx->grid.precision == 64) fold_partials((double *)part.get(), (double *)J, (double *)ext, own, theirs);
        else fold_partials((double *)part.get(), (double *)J, (float *)ext, own, theirs);
    }
    const unsigned char *J = mass + lbm::MAX_CTAS * 8, *ext = J + lbm::MAX_CTAS * 8;
    CK(cudaMemcpyAsync(ctx->ws + ctx->L.f0, p, narr * ctx->L.pops, cudaMemcpyHostToDevice, ctx->stream), "restore");
    p += narr * ctx->L.pops + nparts;
    CK(cudaMemcpyAsync(ctx->ws + ctx->L.mass, mass, lbm::MAX_CTAS * 8, cudaMemcpyHostToDevice, ctx->stream), "restore");
    CK(cudaMemcpyAsync(ctx->ws + ctx->L.J, J, lbm::MAX_CTAS * 8, cudaMemcpyHostToDevice, ctx->stream), "restore");
    CK(cudaMemcpyAsync(ctx->ws + ctx->L.ext, ext, lbm::MAX_CTAS * 4 * sz, cudaMemcpyHostToDevice, ctx->stream), "restore");
    CK(cudaMemcpyAsync(ctx->ws + ctx->L.err, p, sizeof(int), cudaMemcpyHostToDevice, ctx->stream), "restore");
    CK(cudaStreamSynchronize(ctx->stream), "restore sync");
    ctx->step = h.step;
    ctx->cur = h.cur;
    ctx->aa_odd = false;
    ctx->err_pending = false;
    ctx->nctas = std::max(ctx->nctas, 1);
    return LBM_OK;
}

lbm_status lbm_set_collision(lbm_ctx *ctx, const lbm_collision *c)
{
    if (!ctx) return LBM_ERR_ARG;
    drop_graph(ctx);
    if (!c) { ctx->coll = lbm_collision{}; return LBM_OK; }
    if (c->kind == LBM_COLL_BGK) { ctx->coll = *c; return LBM_OK; }
    if (c->kind != LBM_COLL_MRT) return LBM_ERR_ARG;
    for (double r : {c->s_e, c->s_eps, c->s_j, c->s_q})
        if (!(r > 0.0 && r < 2.0)) return LBM_ERR_ARG;
    if (!(c->s_nu <= 0.0 || c->s_nu < 2.0) || std::isnan(c->s_nu)) return LBM_ERR_ARG;
    ctx->coll = *c;
    return LBM_OK;
}

lbm_status lbm_set_option(lbm_ctx *ctx, lbm_option opt, int64_t value)
{
    if (!ctx) return LBM_ERR_ARG;
    drop_graph(ctx);  // the captured launches hold the old arguments
    switch (opt) {
    case LBM_OPT_CTAS_PER_SM:
        if (value < 0 || value > 32) return LBM_ERR_ARG;
        ctx->ctas_per_sm_opt = (int)value;
        break;
    case LBM_OPT_REVERSE:
        ctx->reverse = value != 0;
        return LBM_OK;
    case LBM_OPT_STRIP:
        if (value < 2 || value > STRIP) return LBM_ERR_ARG;
        ctx->W_opt = (int)value;
        break;
    case LBM_OPT_STAGED:
        ctx->allow_staged = value != 0;
        break;
    case LBM_OPT_ROWS2:
        ctx->allow_rows2 = value != 0;
        break;
    case LBM_OPT_TMA:
        ctx->allow_tma = value != 0;
        break;  // re-plan: the tile kernel needs tensor loads
    case LBM_OPT_PREFETCH:
        if (value < 0 || value > 4) return LBM_ERR_ARG;
        ctx->pf = (int)value;
        return LBM_OK;
    case LBM_OPT_GENERAL:
        if (value != 0 && (ctx->big || ctx->inplace)) return LBM_ERR_ARG;  // 32-bit offsets, two arrays only
        ctx->force_general = value != 0;
        break;
    case LBM_OPT_PDL:
        ctx->pdl = value != 0;
        drop_graph(ctx);
        return LBM_OK;
    case LBM_OPT_GRAPH_STEPS:
        if (value < 0 || (value & 1) || value > 1 << 20) return LBM_ERR_ARG;
        ctx->graph_steps = (int)value;
        drop_graph(ctx);
        return LBM_OK;
    case LBM_OPT_FAULT_SKIP_COPY:
        // the test build exists for walls, pressure columns and unpadded rows
        if (value != 0) {
            if (!(ctx->rows2 && !ctx->inplace && !ctx->mask && !ctx->big && ctx->grid.walls && ctx->grid.bc_x &&
                  ctx->pitch == ctx->grid.nx))
                return LBM_ERR_ARG;
            cudaError_t e = cudaFuncSetAttribute((void *)lbm::step_kernel_rows2<true, true, false, true>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)lbm::rows2_smem_bytes());
            if (e != cudaSuccess) return cuda_fail(ctx, e, "smem attribute");
        }
        ctx->fault_skip = value != 0;
        break;  // re-plan: the test build is a row-pair kernel
    case LBM_OPT_TILE:
        ctx->allow_tile = value != 0;
        break;
    default:
        return LBM_ERR_ARG;
    }
    // Re-plan; per-CTA accumulators are folded into the new partition only
    // through their totals, so reset them to keep the reduction exact.
    const int old = ctx->nctas;
    const bool was_general = ctx->mask != nullptr;
    lbm_status s = plan_launch(ctx);
    if (s == LBM_OK) s = plan_geometry(ctx);
    if (s == LBM_OK && (old != ctx->nctas || was_general != (ctx->mask != nullptr))) {
        if (ctx->grid.precision == 64) reset_acc<double>(ctx); else reset_acc<float>(ctx);
    }
    return s;
}

lbm_status lbm_launch_info(const lbm_ctx *ctx, int64_t *ctas, int64_t *threads, int64_t *units,
                           int64_t *staged)
{
    if (!ctx) return LBM_ERR_ARG;
    if (ctx->inplace && ctx->aas.on) {
        if (ctas) *ctas = ctx->aas.nctas;
        if (threads) *threads = lbm::R2_BLOCK;
        if (units) *units = ctx->aas.units;
        if (staged) *staged = 1;
        return LBM_OK;
    }
    if (ctx->inplace) {
        // CTAs striding over the 32 x 8 tiles (FP32: two rows per thread)
        if (ctas) *ctas = ctx->aa.nctas;
        if (threads) *threads = ctx->aa.threads;
        if (units) *units = (int64_t)ctx->aa.ntx * ctx->aa.nty;
        if (staged) *staged = 0;
        return LBM_OK;
    }
    if (ctx->mask) {
        // the general-geometry kernels, a node per thread, also where FP32 steps by row pairs
        if (ctas) *ctas = lbm::mask_blocks(ctx->mask);
        if (threads) *threads = 256;
        if (units) *units = (int64_t)ctx->grid.nx * ctx->grid.ny;
        if (staged) *staged = 0;
        return LBM_OK;
    }
    if (ctas) *ctas = ctx->nctas;
    if (threads) *threads = threads_of(ctx);
    if (units) *units = ctx->t64 ? ctx->t64p.ntiles : (ctx->tile ? ctx->nctas : ctx->units);
    if (staged) *staged = ctx->staged ? 1 : 0;
    return LBM_OK;
}

void lbm_free(lbm_ctx *ctx)
{
    if (!ctx) return;
    if (ctx->stream || ctx->ws) cudaStreamSynchronize(ctx->stream);
    if (ctx->own_ws && ctx->ws) cudaFree(ctx->ws);
    lbm::mask_free(ctx->mask);
    drop_graph(ctx);
    if (ctx->fscratch) cudaFree(ctx->fscratch);
    if (ctx->h_err) cudaFreeHost(ctx->h_err);
    if (ctx->err_ev) cudaEventDestroy(ctx->err_ev);
    delete ctx;
}

} // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free single step.
//
// Some callers cannot allocate device memory at the point where they step the
// lattice: code running inside another framework's memory pool (a raw
// allocation would bypass the pool's accounting and limits), or an embedded
// host that sizes every device buffer up front. This entry point performs one
// step between two caller-owned population buffers and keeps the only scratch
// it needs - the per-CTA diagnostic partials and the error word - in a fixed
// device array that the library declares at file scope. Nothing is allocated
// per call.
// ---------------------------------------------------------------------------

namespace {

constexpr int NOALLOC_MAX_CTAS = 4096;

// Per-CTA partials of one step: mass, wall-shear sum, four extrema (stored as
// double so both precisions fit) and the bad-density flag.
struct NoallocScratch {
    double mass[NOALLOC_MAX_CTAS];
    double J[NOALLOC_MAX_CTAS];
    double ext[4 * NOALLOC_MAX_CTAS];
    int err;
};

constexpr int NOALLOC_MAX_DEVICES = 64;
NoallocScratch *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};
std::mutex g_noalloc_mutex;

} // namespace

// The scratch itself. In host code this name is only a stand-in for the
// device object; its device address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

namespace {

// Device address of the scratch on the current device, resolved on the first
// call made with that device current.
cudaError_t noalloc_scratch(NoallocScratch **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<NoallocScratch *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

template <typename real>
lbm_status noalloc_launch(lbm_ctx *c, NoallocScratch *sc, const void *f_in, void *f_out, double *diag_out,
                          int32_t *err_out)
{
    real *ext = reinterpret_cast<real *>(sc->ext);
    lbm::reset_acc_kernel<real><<<(c->nctas + 255) / 256, 256, 0, c->stream>>>(sc->mass, sc->J, ext, &sc->err,
                                                                                 c->nctas);
    lbm::KArgs<real> A = make_args<real>(c);
    A.fin = static_cast<const real *>(f_in);
    A.fout = static_cast<real *>(f_out);
    A.mass_part = sc->mass;
    A.J_acc = sc->J;
    A.ext = ext;
    A.err = &sc->err;
    cudaError_t e = launch<real>(c, A);
    if (e != cudaSuccess) return cuda_fail(nullptr, e, "noalloc step");
    if (diag_out)
        lbm::diag_kernel<real><<<1, 256, 0, c->stream>>>(sc->mass, sc->J, ext, &sc->err, c->nctas, diag_out);
    e = cudaGetLastError();
    if (e == cudaSuccess && err_out)
        e = cudaMemcpyAsync(err_out, &sc->err, sizeof(int32_t), cudaMemcpyDeviceToDevice, c->stream);
    return e == cudaSuccess ? LBM_OK : cuda_fail(nullptr, e, "noalloc launch");
}

} // namespace

extern "C" lbm_status lbm_step_noalloc(const lbm_grid *grid, const lbm_eos *eos, double tau,
                                       double wetting, const lbm_drive *drive, const void *f_in,
                                       void *f_out, int64_t ctas, double *diag_out, int32_t *err_out,
                                       void *stream)
{
    if (!grid_ok(grid) || !eos || !f_in || !f_out || f_in == f_out) return LBM_ERR_ARG;
    if (ctas < 0 || ctas > NOALLOC_MAX_CTAS) return LBM_ERR_ARG;
    // buffers must hold whole values of the grid precision; the staged kernels
    // also need 16-byte aligned rows (checked below)
    const uintptr_t esz = grid->precision == 64 ? 8 : 4;
    if (((uintptr_t)f_in | (uintptr_t)f_out) % esz != 0) return LBM_ERR_ARG;
    if (((uintptr_t)diag_out) % 8 != 0 || ((uintptr_t)err_out) % 4 != 0) return LBM_ERR_ARG;
    if (!(tau > 0.5) || !(eos->k > 0) || !(eos->kappa >= 0) || !(eos->a > 0) || !(eos->b > 0) ||
        !(eos->R > 0) || !(eos->T_over_Tc > 0) || !std::isfinite(wetting))
        return LBM_ERR_PARAM;

    NoallocScratch *sc = nullptr;
    cudaError_t e = noalloc_scratch(&sc);
    if (e != cudaSuccess) return LBM_ERR_CUDA;

    // Launch plan and physics on the host stack only (no workspace).
    lbm_ctx c;
    c.grid = *grid;
    c.pitch = grid->nx;  // caller buffers: rows of 9 nx values
    c.eos = *eos;
    if (drive) c.drive = *drive;
    else { c.drive.dp = 0; c.drive.p_ref = NAN; c.drive.gx = c.drive.gy = 0; }
    c.tau = tau;
    c.wet = wetting;
    c.stream = static_cast<cudaStream_t>(stream);
    // The staged kernels copy population rows with bulk asynchronous copies,
    // which need 16-byte aligned addresses: a caller buffer that does not start
    // on a 16-byte boundary (a view with an element offset) takes the register-
    // prefetch kernel, which gives identical results.
    if (((uintptr_t)f_in | (uintptr_t)f_out) % 16 != 0) c.allow_staged = false;
    lbm::ChannelThermo ct;
    if (lbm::channel_thermo(*eos, c.drive, grid->bc_x, &ct)) return LBM_ERR_PARAM;
    c.th = ct.th;
    c.T = ct.T; c.Tc = ct.Tc;
    c.rho_g = ct.rho_g; c.rho_l = ct.rho_l; c.p_sat = ct.p_sat;
    c.rho_in = ct.rho_in; c.rho_out = ct.rho_out;
    c.rho_in_l = ct.rho_in_l; c.rho_out_l = ct.rho_out_l;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    if (plan_launch(&c) != LBM_OK) return LBM_ERR_CUDA;
    if (ctas > 0) c.nctas = (int)std::min<long long>(ctas, c.t64 ? c.t64p.ntiles : std::max<long long>(1, c.units / 2));
    c.nctas = std::min(c.nctas, NOALLOC_MAX_CTAS);
    if (c.t64) lbm::tile64_rotate(&c.t64p, c.grid.bc_x && c.grid.precision == 64, c.nctas);
    c.band = band_rows(c.nyf, c.nstrips, c.nctas, c.grid.walls);
    return grid->precision == 64 ? noalloc_launch<double>(&c, sc, f_in, f_out, diag_out, err_out)
                                 : noalloc_launch<float>(&c, sc, f_in, f_out, diag_out, err_out);
}
