// bz_internal.h -- internal declarations shared by the host set-up code, the
// C ABI and the CUDA kernels of the spectral collision library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/bzcoll.h"

namespace bz {

constexpr int kMaxDim = 3;
constexpr int kTile = 32;          // cells per tile in the Fourier scratch layout

// Set the thread-local message and return `code`.
int fail(int code, const std::string &msg);
int cuda_fail(cudaError_t e, const char *what);

// Device memory the library holds beyond one call (grid, kernel and mesh
// tables, the autotuner's batch, cached graph scratch, the error word).  Every
// such block goes through dev_malloc / dev_free, which count the live blocks;
// alloc_fault_due() consumes one step of the host-side failure countdown that
// bz_inject_alloc_failure arms (true: fail this allocation without calling
// CUDA).  The per-call pool scratch draws on the same countdown.
cudaError_t dev_malloc(void **p, size_t bytes);
template <typename X> cudaError_t dev_malloc(X **p, size_t bytes) {
    return dev_malloc(reinterpret_cast<void **>(p), bytes);
}
void dev_free(void *p);
bool alloc_fault_due();

// Let `kernel` launch with `bytes` of dynamic shared memory on the current
// device: the attribute call, made only when the kernel needs more than it has
// been allowed so far (it costs about half a microsecond of every launch).
cudaError_t allow_dynamic_smem(const void *kernel, size_t bytes);

// Device error word (one per device context), latched by kernels.
enum DeviceError : int { kDevOk = 0, kDevNonFinite = 1, kDevTimeout = 2 };

// Kernel-facing view of a grid.
struct GridView {
    int dim, N, h, M;
    int64_t nv;        // N^d
    int64_t nm;        // M^d (full mode set)
    int64_t nhalf;     // (h+1) M^(d-1): modes with k_1 >= 0
    double L, dv, s;
};

}  // namespace bz

struct bz_grid {
    bz::GridView v;
    int device;
    // 1-D DFT factors E[k+h][j] = (-1)^k exp(-2 pi i (k j mod N)/N), k in K_h.
    double2 *d_E64;
    float2 *d_E32;
    // conservation: inverse Gram matrix of the invariants (1, v, |v|^2) on the grid
    double cinv[25];
};

constexpr int kModesumVariants = 10;   // register-blocked FP32 mode-sum kernel variants
constexpr int kMaxSplit = 8;          // most CTAs that share a tile's tasks

// Task tables of one layout, for a tile on S = 1 .. kMaxSplit CTAs, in one block.
struct TaskTables {
    int *block;
    int off[kMaxSplit];      // ints before the table of S CTAs, at S - 1
    float bal[kMaxSplit];    // its most loaded warp's load
    float work;              // load of all tasks
};

struct bz_modes {
    const bz_grid *g;
    double gamma, b0;
    int nq;
    // radial table F(a2, b2) = B-hat for |l+m|^2 = a2 <= d h^2, |l-m|^2 = b2 <= d (2h)^2
    int arows, bcols;
    double *h_F;        // host copy (FP64)
    double *d_F64;
    float *d_F32;
    // symmetric weight streams and task tables of the FP32 2-D kernel, one per
    // variant (k_modesum32.cu); d_W32 / w32_rowmax alias the variant
    // in use (null if the generic kernel serves this grid)
    float *var_W[kModesumVariants];
    TaskTables var_task[kModesumVariants];
    int var_rowmax[kModesumVariants];
    int variant;          // index of the selected variant
    int variant_fixed;    // 1: chosen by BZ_MODESUM_VARIANT (no last-wave split)
    float *small_W;       // weight stream and task tables of the small-launch variant (two outputs per thread)
    TaskTables small_task;
    int small_rowmax;
    void *w64;            // FP64 weight stream and task table, null if unused
    TaskTables task64;
    int rowmax64;
    int variant64;        // layout of the FP64 tables (entry of the variant list), -1 if none
    float *wx2;           // FP32X2 weight stream: the FP64 stream's layout and task table, each
                          // step's weights as FP32 (hi, lo) parts; null if unused
    int modesum_variant;  // variant id reported to callers (index + 1; 0: no choice of variants, N > 48)
    float *d_W32;
    int w32_rowmax;       // largest staged weight row (floats)
    int64_t pairs_sym;   // unordered pairs per cell (algorithmic unit)
    int tile_dft;        // 1: the tile FFT kernels of k_dft32.cu serve this grid in FP32
    int tile_dft64;      // ... and in FP64 (also the FP32X2 form's forward transform)
    double scale;        // s^(d + gamma)
    double penalty;      // c of the Boltzmann model's penalty rate nu = c rho (IMEX stages)
    // fast spectral (Carleman) form, k_fast.cu: method 1 replaces the mode sum
    // of eq. CF1 by nconv + 1 FFT convolutions with the direction factors
    // [(nconv + 1)][M][M] complex: (c_p alpha_p + i alpha'_p)(k), then
    // (1 + i Lambda)(k).  For even ndirs, direction p + ndirs/2 is direction p
    // with alpha and alpha' exchanged (same gain product), so nconv = ndirs/2
    // and c_p = 2; for odd ndirs nconv = ndirs and c_p = 1.
    int method;          // 0: eq. KM / eq. CF1 direct sum; 1: fast form
    int ndirs;
    int nconv;
    double *h_fast;      // host FP64 copy (interleaved re, im)
    double2 *d_fast64;
    float2 *d_fast32;
};

namespace bz {
// Finite-volume mesh of the transport step (fv_mesh.cpp, k_transport.cu):
// polygonal cells with at most kFvMaxFaces faces, per-cell tables in
// [cell][slot] layout, FP64 and FP32 copies of the real-valued ones.
constexpr int kFvMaxFaces = 8;
constexpr int kFvCentral = 5;       // central stencil: the cell and its 5 nearest cells (2 x 3 cells)
constexpr int kFvCentral3 = 11;     // degree 2: the cell and its 11 nearest cells (2 x 6 cells)
constexpr int kFvCoef3 = 5;         // degree 2: coefficients of xi, eta, xi^2, xi eta, eta^2
constexpr int kFvRegular = 0x100;     // flag in ncen: a full stencil that starts with the neighbours of all the
                                      // cell's faces in order, and a sector at every vertex

// Tables of the transport step, one row per position p of the processing order
// (cell order[p]).  Order 2 reconstructs a gradient (B = 2 coefficients from
// K = kFvCentral stencil cells), order 3 the 5 coefficients of the zero-mean
// scaled Taylor basis phi = (xi, eta, xi^2 - mu20, xi eta - mu11, eta^2 -
// mu02), xi = (x - x_b)/h, from K = kFvCentral3 cells.  The FP64 tables have
// factors folded in that save FP64 operations: order 2 is scaled to xi, eta
// too, Rc is divided by lambda_0 where the cell has sectors, and in cells
// flagged kFvRegular the rows of Rc give p_0, the sectors' share taken off.
template <typename T> struct FvTables {
    const T *Rs;            // [p][face][4]  sector inverses (row-major 2 x 2)
    const T *quad;          // [p][4]  FP32: (mu20, mu11, mu02, h^2); FP64: the degree-2 smoothness form's
                            //         coefficients (4 mu20 + 4, mu20 + mu02 + 1, 4 mu02 + 4, 4 mu11)
    const T *fn;            // [p][face][2]  |e| n_e outward
    const T *fs;            // [p][face][2]  the same, exactly opposite on the two sides of a face (fn may differ by
                            //               rounding across a period): which side is upwind
    const T *phi;           // [p][face][B]  means of the basis over the face
    const T *phig;          // [p][face][2][B]  order 3: the basis at the face's two Gauss points
    const T *Rc;            // [p][B][K]  least-squares rows
    const T *inv_area;      // [p]
};
// A thin cell (perimeter times largest radius over area above this; 4 for an
// equilateral triangle) cancels its face fluxes to L by that much.
constexpr double kFvThin = 50.0;
constexpr int kFvThinFlag = 0x10;     // in meta: a thin cell
constexpr int kFvSplitFlag = 0x20;    // in meta: a cell with a split face
constexpr int kFvSplit = 1 << 30;     // in d_two: a face whose two sides' normals are not exactly opposite (the two
                                      // copies of a face across a period)
}  // namespace bz

struct bz_mesh {
    int device;
    int order;              // 1: piecewise constant, 2: CWENO of degree 1, 3: CWENO of degree 2
    int64_t n_cells, n_faces_interior, n_faces_boundary;
    int64_t n_rows;         // faces as d_fid numbers them
    int max_faces;
    // index tables by position of the processing order (cells sorted along a
    // Morton curve of their barycentres), values are cell indices
    int *d_order;           // [p] cell
    int *d_meta;            // [p] faces | kFvThinFlag | kFvSplitFlag | not-owner bits << 8 | boundary bits << 16 | two-sided
                            // bits << 24 (bit q: face q); the owner of a face is its first cell in the
                            // processing order; a two-sided face bounds a thin cell
    int *d_nb;              // [p][face] neighbour, -1 boundary
    int *d_fid;             // [p][face] face index, numbered in the processing order of the owners
    int *d_two;             // [p][face] index of a two-sided face, | kFvSplit
    int64_t n_two;
    int *d_ncen;            // [p] central stencil size (<= K), | kFvRegular (any polygon): the stencil starts with
                            // the face neighbours in face order, sector s on faces s, s + 1
    int *d_cen;             // [p][K]
    int *d_nsec;            // [p] sectors
    int *d_sec;             // [p][face][2] sector cells
    // triangle meshes of order 2: per position p three int4 {i, ncen, 0, qbits}, {cen[0..3]},
    // {cen[4], nb[0..2]} with i = order[p] and qbits holding, in 2 bits per face, the index of the
    // same face in the neighbour; one level of loads gives a block all its indices
    int4 *d_tripos;
    // walls with full accommodation (fv_mesh_set_walls): per position and face
    // the wall index (-1: none), per wall the face's slot p * kFvMaxFaces + q
    // and (theta_w, u_w1, u_w2) in FP64 and FP32
    int *d_wall;
    int64_t *d_wallslot;
    double *d_wall64;
    float *d_wall32;
    int64_t n_walls;
    // host copies for the wall look-up: counter-clockwise vertex lists (CSR),
    // the neighbour of every face and the position of every cell
    int64_t *h_ptr, *h_vtx;
    int *h_nb, *h_pos;
    void *d_real64;         // one block holding the FvTables<double> arrays
    void *d_real32;         // one block holding the FvTables<float> arrays
    bz::FvTables<double> t64;
    bz::FvTables<float> t32;
};

namespace bz {

// ---- kernels (k_dft.cu) ---------------------------------------------------
// Forward DFT of f [n][N^d] into the tiled half spectrum fhat
// [ceil(n/32)][nhalf][32] complex.  hi/lo split output when lo != nullptr.
cudaError_t launch_dft_forward_f64(const GridView &g, const double2 *E, const double *f,
                                   double2 *fhat, int64_t n, cudaStream_t st);
cudaError_t launch_dft_forward_f32(const GridView &g, const float2 *E, const float *f,
                                   float2 *fhat, int64_t n, cudaStream_t st);
// FP64 transform of FP32 input (the FP32X2 form's forward DFT).
cudaError_t launch_dft_forward_f64_f32in(const GridView &g, const double2 *E, const float *f,
                                         double2 *fhat, int64_t n, cudaStream_t st);

// Inverse Gram matrix of the collision invariants, passed by value to kernels.
struct Cinv {
    double v[25];
};

// Epilogue options of the inverse DFT.
struct InvEpilogue {
    int conserve;             // apply the conservation projection
    int check;                // unused here (input check is done on f)
    const void *P;            // if non-null: write G = Q - P instead of Q
};
cudaError_t launch_dft_inverse_f64(const GridView &g, const double2 *E, const double2 *Qhat,
                                   double *Q, int64_t n, double scale, const double *cinv,
                                   const InvEpilogue &ep, cudaStream_t st);
cudaError_t launch_dft_inverse_f32(const GridView &g, const float2 *E, const float2 *Qhat,
                                   float *Q, int64_t n, double scale, const double *cinv,
                                   const InvEpilogue &ep, cudaStream_t st);

// ---- tile FFT kernels (k_dft32.cu), FP32 and FP64: 2-D, N in {16, 24, 32, 48}; 3-D, N = 16; FP32: 2-D, N = 64 ----
bool dft32_tile_supported(const GridView &g, bool fp64);
int dft32_setup();   // twiddles on the current device
cudaError_t launch_dft32_forward_tile(const GridView &g, const float *f, float2 *fhat, int64_t n, cudaStream_t st);
cudaError_t launch_dft32_inverse_tile(const GridView &g, const float2 *Qhat, float *Q, int64_t n, double scale,
                                      const double *cinv, const InvEpilogue &ep, cudaStream_t st, bool pdl = false);
cudaError_t launch_dft64_forward_tile(const GridView &g, const double *f, double2 *fhat, int64_t n,
                                      cudaStream_t st);
cudaError_t launch_dft64_forward_tile_f32in(const GridView &g, const float *f, double2 *fhat, int64_t n,
                                            cudaStream_t st);
cudaError_t launch_dft64_inverse_tile(const GridView &g, const double2 *Qhat, double *Q, int64_t n, double scale,
                                      const double *cinv, const InvEpilogue &ep, cudaStream_t st);

// ---- register-blocked FP32 2-D mode sum (k_modesum32.cu) --------------------
constexpr int kMaxGroup = 16;      // instances per grouped launch
struct Mode32Item {
    const void *fhat;     // float2 or double2 spectra, tiled layout
    void *Qhat;
    const void *W;        // weight stream of the kernel's scalar type
    const int *tasks;     // task table for WARPS x split warps
    int h, M, nhalf, wrow_max;
    int64_t n;
    int split;            // CTAs that share a tile's tasks
};
struct Mode32Group {
    int nitems;
    int64_t tile_start[kMaxGroup + 1];   // prefix sums of CTAs (tiles of 8 to 32 cells, times the split)
    Mode32Item item[kMaxGroup];
};
bool modesum32_available(const bz_modes *m);
cudaError_t launch_modesum32(const bz_modes *m, const float2 *fhat, float2 *Qhat, int64_t n, cudaStream_t st,
                             bool pdl = false);
// Cells one SM holds at a time in the handle's FP32 mode-sum kernel (CTAs per
// SM x cells per CTA; 32 where the register-blocked kernels do not serve it).
int modesum32_wave_cells_per_sm(const bz_modes *m);
// Whether the handle's FP32 mode sum splits the tiles of a partial wave over
// several CTAs (32-cell variants chosen by timing).
bool modesum32_tail_splits(const bz_modes *m);
// Whether batches of at most half a wave run on a one-CTA-per-SM sibling of
// the handle's variant (bit-identical results).
bool modesum32_small_batches_fast(const bz_modes *m);
bool modesum64_available(const bz_modes *m);
cudaError_t launch_modesum64(const bz_modes *m, const double2 *fhat, double2 *Qhat, int64_t n, cudaStream_t st);
// FP32X2 (double-float) mode sum on the FP64 tables: FP64 spectra in, Q-hat
// rounded to FP32 out (k_modesum32.cu).
bool modesum_x2_available(const bz_modes *m);
cudaError_t launch_modesum_x2(const bz_modes *m, const double2 *fhat, float2 *Qhat, int64_t n, cudaStream_t st);
cudaError_t launch_modesum32_group(const bz_modes *const *ms, const float2 *const *fhat, float2 *const *Qhat,
                                   const int64_t *n, int count, cudaStream_t st);

// ---- fast spectral form (k_fast.cu), 2-D, N in {8, 16, 24, 32, 48} --------
bool fast_supported(const GridView &g);
int fast_pad_length(int N);        // P of the zero-padded convolution grid
int fast_cells_per_cta(int N);
int fast_setup();                  // twiddles of k_fast.cu on the current device
cudaError_t launch_fast_f32(const bz_modes *m, const float2 *fhat, float2 *Qhat, int64_t n, cudaStream_t st);
cudaError_t launch_fast_f64(const bz_modes *m, const double2 *fhat, double2 *Qhat, int64_t n, cudaStream_t st);

// ---- kernels (k_modesum.cu) -----------------------------------------------
cudaError_t launch_modesum_generic_f64(const GridView &g, const double *F, int bcols,
                                       const double2 *fhat, double2 *Qhat, int64_t n,
                                       cudaStream_t st);
cudaError_t launch_modesum_generic_f32(const GridView &g, const float *F, int bcols,
                                       const float2 *fhat, float2 *Qhat, int64_t n,
                                       cudaStream_t st);

// ---- kernels (k_imex.cu) --------------------------------------------------
struct StageCoef {
    int stage;                 // 0-based l
    int nprev;                 // l
    double at[5], a[5];        // At[l][m], A[l][m] for m < l
    double all;                // A[l][l]
    double dt, eps;
    double nuf;                // penalty rate nu = nuf * rho
    double coef;               // dt A_ll nuf / eps: c = coef * rho
    int store_F;               // 0: F_l equals f^n exactly (stage 0 of a step) and is not written
    int store_P;               // 0: no later stage reads P_l
    int use_G;                 // 0: every G is zero (a whole step of the BGK model) and none is read
};
cudaError_t launch_imex_stage_f64(const GridView &g, const StageCoef &c, const double *fn,
                                  double *F, const double *G, double *P, const double *Lres,
                                  int64_t stride, int64_t n, cudaStream_t st);
cudaError_t launch_imex_stage_f32(const GridView &g, const StageCoef &c, const float *fn,
                                  float *F, const float *G, float *P, const float *Lres,
                                  int64_t stride, int64_t n, cudaStream_t st);
cudaError_t launch_check_input_f64(const double *f, int64_t count, int *err, cudaStream_t st);
cudaError_t launch_check_input_f32(const float *f, int64_t count, int *err, cudaStream_t st);
cudaError_t launch_fill_zero(void *p, int64_t bytes, cudaStream_t st);

// ---- transport residual (k_transport.cu) ----------------------------------
// Order 1: L from f in one pass.  Orders 2 and 3: the reconstruction pass
// writes the upwind mean over every face (FP64: the flux), FX [face][nv], each
// velocity by the cell it leaves; then L [cell][nv] = the sum of v.n times a
// cell's face rows over |P_i|.  FP32, order 2 on triangles without walls (N divisible by 4,
// 16-byte aligned rows: fv_value_mode): the reconstruction writes each cell's
// values at its three faces, FV [cell][3][nv], and the flux pass reads those
// of the cell and its neighbours.  Scratch: fv_scratch_rows() rows of nv.
bool fv_value_mode(const bz_mesh *mesh, const GridView &g, const void *f, const void *L);
cudaError_t fv_values_setup();      // once per mesh: lets the value passes take their shared memory
int64_t fv_scratch_rows(const bz_mesh *mesh, bool f32, bool step);
// Whether an IMEX step takes every face as two-sided: FP32, degree 2, thin cells.
// A step can be unstable in thin cells (their CFL limit is far below the
// others'), and growth by many orders of magnitude within a step shows the
// rounding of every cell around them: there the sums stay term by term those
// of the two-sided Rusanov form.
bool fv_two_sided(const bz_mesh *mesh, bool f32);
cudaError_t launch_fv_faces_two_f32(const bz_mesh *mesh, const GridView &g, const float *f, float *FX, cudaStream_t st);
cudaError_t launch_fv_sum_two_f32(const bz_mesh *mesh, const GridView &g, const float *FX, float *L, cudaStream_t st);
cudaError_t launch_fv_values_f32(const bz_mesh *mesh, const GridView &g, const float *f, float *FV, cudaStream_t st);
cudaError_t launch_fv_flux_values_f32(const bz_mesh *mesh, const GridView &g, const float *FV, float *L,
                                      cudaStream_t st);
// walls need one CTA to hold all velocities of a cell
bool fv_walls_supported(const bz_mesh *mesh, const GridView &g);
cudaError_t launch_fv_first_f64(const bz_mesh *mesh, const GridView &g, const double *f, double *L, cudaStream_t st);
cudaError_t launch_fv_first_f32(const bz_mesh *mesh, const GridView &g, const float *f, float *L, cudaStream_t st);
cudaError_t launch_fv_faces_f64(const bz_mesh *mesh, const GridView &g, const double *f, double *FX, cudaStream_t st);
cudaError_t launch_fv_faces_f32(const bz_mesh *mesh, const GridView &g, const float *f, float *FX, cudaStream_t st);
cudaError_t launch_fv_sum_f64(const bz_mesh *mesh, const GridView &g, const double *FX, double *L, cudaStream_t st);
cudaError_t launch_fv_sum_f32(const bz_mesh *mesh, const GridView &g, const float *FX, float *L, cudaStream_t st);

// Device error word of the current device (allocated on first use; api.cu).
int *device_error_word();

// One collision evaluation (forward DFT, mode sum, inverse DFT; the launches of
// collide_batch) with the Fourier scratch at `scratch`, which must hold
// collide_scratch_size() bytes; requests no device memory (api.cu).
size_t collide_scratch_size(const bz_modes *m, int precision, int64_t n);
int collide_on_scratch(const bz_modes *m, int precision, int flags, const void *f, void *Q, int64_t n,
                       void *scratch, cudaStream_t st);

}  // namespace bz
