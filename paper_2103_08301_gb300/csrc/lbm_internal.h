// Declarations shared by the host translation units of the solver library.
#pragma once

#ifdef __CUDACC__
#include <cuda.h>  // CUtensorMap
#endif

#include <cstdint>

#include "lbm.h"

namespace lbm {

// Equation-of-state parameters at absolute temperature T: Carnahan-Starling
// (kind 0) or Peng-Robinson (kind 1, Eq. 2.18, with aalpha = a alpha(T)).
struct Thermo {
    double a, b, R, T;
    int kind = 0;
    double aalpha = 0.0;
};

double eos_pressure(const Thermo &t, double rho);
double eos_dpressure(const Thermo &t, double rho);
// Critical point (PR: alpha(Tc) = 1).
void eos_critical(int kind, double a, double b, double R, double *Tc, double *rhoc);
// Standard PR temperature function alpha(T) for acentric factor omega.
double pr_alpha(double omega, double T_over_Tc);
// Maxwell coexistence below Tc; returns nonzero at or above Tc.
int maxwell(const Thermo &t, double *rho_g, double *rho_l, double *p_sat);
// Density on the gas (liquid) branch whose EOS pressure is p. A pressure
// beyond the branch's end gives the spinodal density and sets *saturated.
// Nonzero if p <= 0 (gas) or if there is no liquid branch (T >= Tc).
int gas_density(const Thermo &t, double p, double *rho, bool *saturated = nullptr);
int liquid_density(const Thermo &t, double p, double *rho, bool *saturated = nullptr);
// Thermodynamic state of an lbm_eos: T, Tc and the Thermo; nonzero on bad parameters.
int thermo_of(const lbm_eos &e, Thermo *t, double *Tc);

// Thermodynamics of one channel: Maxwell coexistence (rho_g = rho_l = 0 above
// Tc: no phase blending) and, with pressure columns, the column densities on
// both branches at the mesh pressures p_ref +- dp/2 (p_ref NaN: k^2 p_sat).
// sat[0..3] flag a column density held at a spinodal (gas_in, liq_in,
// gas_out, liq_out). Returns nonzero if the parameters admit no columns.
struct ChannelThermo {
    Thermo th{};
    double T = 0, Tc = 0, rho_g = 0, rho_l = 0, p_sat = 0;
    double rho_in = 0, rho_out = 0, rho_in_l = 0, rho_out_l = 0;
    bool sat[4] = {false, false, false, false};
};
int channel_thermo(const lbm_eos &e, const lbm_drive &d, bool bc_x, ChannelThermo *out);
double node_noise(uint64_t seed, uint64_t node, double amp);

// Row pitch of a population plane: nx rounded up to 4 columns, so that every
// row segment of the bulk-copy staged kernel is 16-byte aligned.
inline int pitch_of(int nx) { return (nx + 3) & ~3; }

// Whether 32-bit population offsets address the grid: 9 pitch ny < 2^31
// (about 238 million nodes). Larger single-channel grids take the kernels
// with 64-bit offsets; the batch, the wall-mask path, the allocation-free
// entry and the adjoint keep the 32-bit bound.
inline bool idx32_ok(int nx, int ny) { return 9ll * pitch_of(nx) * ny < (1ll << 31); }

// Strip width for an nx-column channel: the widest up to w_max, except that
// the outlet column must not open a strip (its stencil reaches two columns
// back); widths that keep 16-byte alignment (multiples of 4) are preferred.
inline int strip_width(int nx, int w_max, bool bc_x)
{
    int W = w_max;
    if (!(bc_x && nx > W && nx % W == 1)) return W;
    for (int w = (W - 1) & ~3; w >= 4; w -= 4)
        if (nx % w != 1) return w;
    for (int w = W - 1; w >= 2; --w)
        if (nx % w != 1) return w;
    return W;
}

} // namespace lbm

#ifdef __CUDACC__
// 2-D tensor map of one FP32 population array (pitch wide, 9 * ny plane-rows)
// in the form the row-pair stage loads it (lbm_api.cu); false if the driver
// entry point is unavailable or the layout does not qualify.
bool lbm_encode_population_map(CUtensorMap *map, void *base, int pitch, int ny);
// One step of a context between two states outside it, each in the context's
// own layout (rows of nine planes, plane pitch pitch_of(nx), 9 * pitch * ny
// values, 256-byte aligned), on `stream`; slots that no population
// reaches keep their contents in `fout`. The context's own state and step
// counter are untouched; bad densities are flagged in its error word (device),
// lbm_ctx_error_word. Two-array contexts without a wall mask. lbm_api.cu.
cudaError_t lbm_ctx_step_between(lbm_ctx *ctx, const void *fin, void *fout, cudaStream_t stream);
int *lbm_ctx_error_word(lbm_ctx *ctx);

namespace lbm {
template <typename real>
struct KArgs;
// The general-geometry step on a lattice with a solid mask (lbm_mask.cu).
// mask_setup validates the mask, builds the ghost table and allocates the
// path's device tables; *out stays NULL (LBM_OK) when the mask adds no solid
// node to the wall rows, unless `force`. mask_launch runs one step (mode
// MODE_STEP) or the fields (MODE_FIELDS) of A.fin on `stream`.
struct MaskPath;
lbm_status mask_setup(const uint8_t *mask, const lbm_grid &g, int pitch, int sms, bool force, cudaStream_t stream,
                      MaskPath **out, char *err, size_t errlen);
void mask_free(MaskPath *m);
int mask_blocks(const MaskPath *m);  // CTAs of the collide kernel (diagnostic slots)
template <typename real>
cudaError_t mask_launch(const MaskPath *m, const KArgs<real> &A, int mode, cudaStream_t stream);
// The FP32 step by row pairs over the caller's plan (A.nctas CTAs, strips of
// A.W; map: tensor map of A.fin), and its resident CTAs per SM.
cudaError_t mask_rows2_plan(const MaskPath *m, bool early, int *ctas_per_sm);
cudaError_t mask_rows2_launch(const MaskPath *m, const KArgs<float> &A, const CUtensorMap *map, bool early,
                              cudaStream_t stream);

// In-place streaming (the AA pattern) of a single context (lbm_inplace.cu):
// one population array F, a density plane rho (pitch * ny) and a side buffer
// (2 * ny * 9) for the pressure columns. aa_plan sizes the tile grid and the
// CTA counts; aa_step runs one step of F (even: natural layout in, odd-parity
// layout out; odd: the reverse); aa_swap turns an odd-parity F back into the
// natural layout in place.
struct AAPlan {
    int ntx, nty, sx, sy;  // tile grid of the step and its shifts
    int nctas;             // CTAs of the step (its diagnostic slots)
    int threads;           // threads per CTA of the step
    int dens_blocks;       // CTAs of the density pass
};
cudaError_t aa_plan(int precision, bool big, bool walls, bool pres, int nx, int ny, int sms, AAPlan *p);
template <typename real>
cudaError_t aa_step(const KArgs<real> &A, real *F, real *rho, real *side, bool walls, bool pres, bool odd, bool big,
                    const AAPlan &p, cudaStream_t st);
// The FP32 step by row pairs in place, for channels between pressure columns:
// A holds the strip plan (strips of at most AA_W columns, A.nctas CTAs), maps the
// tensor maps of F with boxes of AA_SP columns by 9, 1 and 2 planes. aa_strips_plan
// gives the resident CTAs per SM.
cudaError_t aa_strips_plan(bool walls, bool big, int *ctas_per_sm);
cudaError_t aa_strips_step(const KArgs<float> &A, float *F, float *rho, const CUtensorMap *maps, bool walls, bool odd,
                           bool big, int sms, cudaStream_t st);
cudaError_t aa_swap(int precision, void *F, bool walls, bool pres, bool big, int nx, int ny, int P, int sms,
                    cudaStream_t st);
}  // namespace lbm
#endif

// The step kernels with 64-bit population offsets (lbm_big.cu), and the FP32
// row-pair step likewise, for grids whose 9 pitch ny slots reach 2^31.
void *lbm_big_step_kernel_ptr(int precision, bool walls, bool pres, bool staged, bool padded);
void *lbm_big_rows2_kernel_ptr(bool walls, bool pres, bool padded);

#ifdef __CUDACC__
namespace lbm {
// The FP64 step and fields by tiles (lbm_tile64.cu): tile height, grid and CTA
// count for a lattice, and one launch over `ctas` CTAs (diagnostic slots).
struct Tile64 {
    int th, ntx, ntiles, sx, sy, ctas, threads, rot;
};
cudaError_t tile64_plan(int precision, int nx, int ny, bool walls, bool pres, bool big, int sms, Tile64 *p);
void tile64_rotate(Tile64 *p, bool on, int ctas);  // the order of the tiles for that many CTAs
template <typename real>
cudaError_t tile64_launch(const KArgs<real> &A, bool walls, bool pres, bool big, const Tile64 &p, int ctas,
                          cudaStream_t st);

// Destinations of the macroscopic fields rho, ux, uy (nx ny values), tau_w, p_w
// (2 nx), any of them NULL. fields_route decides which a kernel writes itself
// (memory of this device, in one allocation, that overlaps neither another output
// nor the `busy` range, the state): ptr = dst; the others need `scratch` bytes, output
// k at offset[k], which the caller points ptr[k] to. fields_tiles computes the
// outputs with a ptr; fields_copy brings the scratch ones to their destinations.
template <typename real>
struct FieldsOut {
    void *dst[5];
    real *ptr[5];
    size_t bytes[5], offset[5], scratch;
    void use(unsigned char *mem)
    {
        for (int k = 0; k < 5; ++k)
            if (dst[k] && !ptr[k]) ptr[k] = (real *)(mem + offset[k]);
    }
};
template <typename real>
void fields_route(FieldsOut<real> &o, int nx, int ny, const void *busy, size_t busy_bytes);
template <typename real>
cudaError_t fields_tiles(KArgs<real> A, const FieldsOut<real> &o, bool walls, bool pres, bool big, int sms, cudaStream_t st);
template <typename real>
cudaError_t fields_copy(const FieldsOut<real> &o, cudaStream_t st);
}  // namespace lbm
#endif
