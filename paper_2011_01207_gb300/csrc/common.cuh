// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <cufft.h>
#include <cuda_bf16.h>
#include <cstdint>
#include <string>

#include "../../include/amoebapol.h"
#include "rules.h"

#define AP_WARP 32
#define AP_BLOCK_ATOMS 32          // atoms per block, paper Sec. 2.3: B_size = 32
#define AP_CAND_SELF (1 << 30)     // a candidate that is an atom of the block itself

// physical constants (readings: the paper gives none)
#define AP_COULOMB 332.063713       // kcal A / (mol e^2)
#define AP_DEBYE 4.80321            // Debye per e*A
#define AP_SQRT_PI 1.7724538509055159
#define AP_SHORT_RANGE 4.0          // A, radius of the learned guess's neighbourhood feature

// 32-byte aligned 4-vector of doubles (the CUDA 13 double4 is deprecated)
struct __align__(32) dvec4 { double x, y, z, w; };

template <class T> struct V4;
template <> struct V4<float> { typedef float4 type; };
template <> struct V4<double> { typedef dvec4 type; };

template <class T> struct FftTypes;
template <> struct FftTypes<float> { typedef cufftComplex cplx; };
template <> struct FftTypes<double> { typedef cufftDoubleComplex cplx; };

// device-side solver state (one per context)
struct PcgState {
    double rz;         // r . z of the current iterate
    double pq;         // accumulator: p . A p
    double rz_new;     // accumulator: r . z after the update
    double zz;         // accumulator: |alpha r|^2 after the update
    double gamma;      // step length of the current iteration
    double beta;       // conjugation coefficient for the next direction
    double eps;        // convergence measure (Debye)
    double eps0;       // measure for the initial guess
    double tol;        // threshold (Debye)
    int iter;          // iterations done
    int max_iter;
    int done;          // 1 when converged or out of iterations
    int status;        // AP_OK / AP_NOT_CONVERGED
    unsigned int blocks_done;   // last-block-done counter of the q = A p kernel
    unsigned int blocks_done2;  // last-block-done counter of the update kernel
    int nonfinite;     // set when a reduction produced NaN/Inf
    int guard;         // iterations started by the graph loop (hard bound on the WHILE node)
};

// 64-bit fixed point (two's complement in unsigned long long so that atomicAdd applies):
// fields, forces and torque terms with 34 fractional bits, the energy with 30 (paper Sec. 2.4)
#define AP_FX_BITS 34
#define AP_FX_EBITS 30
__host__ __device__ __forceinline__ long long ap_to_fx(double v) { return llrint(v * 17179869184.0); }   // 2^34
__device__ __forceinline__ long long ap_to_fx(float v) { return llrintf(v * 17179869184.0f); }
__host__ __device__ __forceinline__ double ap_from_fx(long long a) { return (double)a * (1.0 / 17179869184.0); }
// value k of an accumulator array that holds FP64 numbers or (fixed != 0) fixed-point integers
__device__ __forceinline__ double acc_value(const double *acc, size_t k, int fixed) {
    return fixed ? ap_from_fx(reinterpret_cast<const long long *>(acc)[k]) : acc[k];
}

// one block pair (I, J) in block I's list: J, its exclusion-mask slot or -1, and the origin of block J
// relative to block I's, periodic image included (c_J - c_I + L k), as hi + lo float pairs
struct __align__(16) TileRec {
    int J, excl;
    float hx, hy, hz, lx, ly, lz;
};

struct ap_ctx {
    ap_params prm;
    int prec = AP_MIXED;      // arithmetic: AP_MIXED (FP32 pairs/PME) or AP_FP64
    int fixed = 0;            // 1: 64-bit fixed-point accumulation (AP_FIXED)
    int n = 0, n_pad = 0, n_blocks = 0;
    cudaStream_t s0 = nullptr;          // caller's stream
    cudaStream_t s1 = nullptr;          // internal stream (reciprocal branch)
    cudaStream_t s2 = nullptr, s3 = nullptr;   // capture of the solve loop's body (main, reciprocal)
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    std::string err;
    int sm_count = 0;
    int one_stream = 0;                 // a batch of several replicas is being captured: every replica's
                                        // kernels in one chain (ap_batch_capture)

    // neighbour blocks
    int *perm = nullptr;      // [n_pad] slot -> atom (-1 for padding)
    int *iperm = nullptr;     // [n] atom -> slot
    float4 *bcenter = nullptr;   // [n_blocks] block centre (x,y,z) at the last build
    TileRec *tiles = nullptr;    // [cap_tiles] block pairs (I, J), both orders, sorted by I then J
    unsigned *excl_mask = nullptr;  // [cap_excl] words, 32 per slot: word j-lane, bit i-lane
    int n_tiles = 0, cap_tiles = 0, n_excl_tiles = 0, cap_excl = 0;
    int *tile_off = nullptr;     // [n_blocks+1] first tile of each block
    int image_dims = 0;          // bit d: the box is too short along d for one image per tile
    // pair lists of the configuration (lists.cu, walked as in pair_walk.cuh)
    int list_mult = 1;           // images an atom can appear in beside one block (2 per short dimension)
    void *boxes = nullptr;       // T4 [n_blocks][2] centres and half extents at the present positions
    int4 *ncand = nullptr;       // [n_blocks] candidate atoms in the block's four segments
    int *cand_j = nullptr;       // [cap][32] candidate's slot | AP_CAND_SELF
    void *cand_pos = nullptr;    // T4 [cap][32] candidate's position beside the block, Thole factor
    unsigned *list = nullptr;    // the lists' entries, two per word (while they are made also the candidates'
                                 // masks: rules.h)
    uint2 *list_meta = nullptr;  // [chunk][16] where each target pair's list lies
    double *e1s = nullptr;       // [3][n_pad] short-range first-order induced field (feature)
    long cap_lists = 0;          // tiles x images the candidate and list arrays hold
    int lists_valid = 0;
    // scratch for the build
    int *cell_count = nullptr; int cap_cells = 0;
    int *tmp_int = nullptr; int cap_tmp = 0;
    float4 *bhalf = nullptr;     // [n_blocks] half extents of the blocks at the last build
    int *nb_info = nullptr;      // [8] a build's results read back together (neighbour.cu)

    // configuration (sorted slots; element type T = float or double). Positions are stored
    // relative to the origin of the slot's block (its centre at the list build, bcenter):
    // small numbers, so FP32 keeps ~1e-6 A at any box size; pair kernels see differences
    // only, and the chunk positions are formed relative to block I's origin in FP64.
    void *posq = nullptr;     // T4: x, y, z (relative to the block origin), q
    void *posw = nullptr;     // T4: x, y, z again, alpha^-1/2 (Thole); padding far outside
    int4 *stb = nullptr;      // [n_pad] smooth-PME stencil origin floor(K x / L) mod K per dimension
    void *stw = nullptr;      // T4 [n_pad] its fractional part K x / L - floor(K x / L), from FP64
    void *dipd = nullptr;     // T4: dx, dy, dz, alpha^-1/2 (Thole)
    void *quad0 = nullptr;    // T4: Qxx, Qxy, Qxz, Qyy
    void *quad1 = nullptr;    // T4: Qyz, Qzz, alpha, q
    double *alpha = nullptr;  // [n_pad]
    double *E = nullptr;      // [3][n_pad] permanent field (SoA)
    double *acc = nullptr;    // [3][n_pad] real-space accumulator
    void *rec = nullptr;      // T [3][n_pad] reciprocal field from the gather
    double *rot = nullptr;    // [n_pad][9] frame matrices (columns x,y,z)
    double *mpl = nullptr;    // [n_pad][10] local multipoles (sorted), for torques
    int *frame_s = nullptr;   // [n_pad][3] frames in slot indices (type, z-slot, x-slot)
    double *fvec = nullptr;   // [n_pad][6] minimum-image vectors to the z- and x-atoms
    int config_valid = 0;

    // PCG
    double *mu = nullptr, *r = nullptr, *qv = nullptr;   // [3][n_pad]
    double *dg = nullptr;     // [n_pad] diagonal of A: 1/alpha - self coefficient (0 for padding)
    // mixed and fixed-point modes: the PCG vectors in FP32, one float4 (x, y, z, unused) per slot
    float4 *mu_f = nullptr, *r_f = nullptr, *q_f = nullptr;   // [n_pad] each
    float2 *dga_f = nullptr;  // [n_pad] (1/alpha - self coefficient, alpha), 0 for padding
    int *hist_count = nullptr;   // device: steps held by a batch step's trajectory history
    void *p = nullptr;        // T4 [n_pad] search direction
    PcgState *st = nullptr;   // device
    double *red_part = nullptr;   // [3 * ceil(n_pad/256)] per-block partial sums of the PCG dots
    PcgState *st_host = nullptr;  // pinned mirror

    // PME
    int K[3] = {0, 0, 0};
    size_t ngrid = 0, ncgrid = 0;
    void *grid = nullptr;     // T [Kz][Ky][Kx]
    void *cgrid = nullptr;    // complex [Kz][Ky][Kx/2+1]
    void *green = nullptr;    // T [Kz][Ky][Kx/2+1]  B(m) C(m)
    void *grid2 = nullptr;    // second real grid (potential of the permanent multipoles, kept for forces)
    long long *grid_fx = nullptr;   // AP_FIXED: the spread's fixed-point grid (kept cleared)
    cufftHandle plan_r2c = 0, plan_c2r = 0;
    float2 *fft_tw = nullptr;     // the library's own transforms (fft.cu): roots of the three sizes
    float *fft_green = nullptr;   // and B C in their order; NULL where cuFFT is used

    // forces
    double *frc = nullptr;    // [3][n_pad] force accumulator (sorted)
    double *gdip = nullptr;   // [3][n_pad] dU/d(global dipole)
    double *gquad = nullptr;  // [6][n_pad] dU/d(global quadrupole)
    double *red = nullptr;    // small reduction scratch
    double *mu_s = nullptr;   // [3][n_pad] dipoles given to the force call (sorted)
    double *gbuf = nullptr;   // [30][n_pad] PME potential derivatives for the forces
    void *cgrid_v = nullptr;  // complex [Kz][Ky][Kx/2+1]: transform of the permanent potential (virial)
    double *vir_active = nullptr;   // virial accumulator of the force call in progress (or NULL)
    float *mlp_feat = nullptr;   // [n_pad][16] learned-guess features (slot order)
    float *mlp_y = nullptr;      // [n_pad][3] network outputs (slot order)

    // launch shapes chosen by ap_autotune (0 = default)
    int tune_mv_per_sm = 0;   // matvec CTAs per SM (0: as many as fit, the resident grid)
    int tune_pme_threads = 128;
    // Jacobi/DIIS solver (allocated by its first call)
    void *diis_st = nullptr;         // device state: window matrix, coefficients, convergence
    void *diis_st_host = nullptr;    // pinned mirror
    double *diis_y = nullptr;        // [depth][3][n_pad] ring of Jacobi updates y_k
    double *diis_e = nullptr;        // [depth][3][n_pad] ring of their errors e_k
    double *diis_part = nullptr;     // [AP_DIIS_MAX_DEPTH][blocks] partial dots
    int diis_cap = 0;                // window length the rings hold
    int last_solver = 0;             // the last solve: 0 PCG, 1 Jacobi/DIIS, 2 the two-set PCG
    void *dp = nullptr;              // buffers of the two-dipole-set path (allocated on first use)
    cudaGraphExec_t diis_exec = nullptr;
    // graph of the solve loop
    cudaGraphExec_t solve_exec = nullptr;
    int graph_ok = 0;         // 1 when the conditional-while graph is usable
    int graph_tried = 0;
};

// error helpers -------------------------------------------------------------------------
int ap_fail(ap_ctx *c, int code, const std::string &msg);
#define AP_CUDA(call)                                                                    \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess)                                                           \
            return ap_fail(ctx, AP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)
#define AP_CUFFT(call)                                                                   \
    do {                                                                                 \
        cufftResult r_ = (call);                                                         \
        if (r_ != CUFFT_SUCCESS)                                                         \
            return ap_fail(ctx, AP_ERR_CUDA, std::string(#call) + ": cufft error " + std::to_string((int)r_)); \
    } while (0)

// the stream of the reciprocal branch beside `main`, whose usual partner is `aux`
inline cudaStream_t aux_stream(const ap_ctx *ctx, cudaStream_t main, cudaStream_t aux) { return ctx->one_stream ? main : aux; }

// launch helpers --------------------------------------------------------------------------
static inline int ap_grid_for(long n, int threads) { return (int)((n + threads - 1) / threads); }

// entry points implemented in the translation units ------------------------------------
int nb_build(ap_ctx *ctx, const double *d_xyz, const int *d_off, const int *d_atoms, int n_excl);
int cfg_load(ap_ctx *ctx, const double *d_xyz, const double *d_mpole, const int *d_frame,
             const double *d_alpha);
int lists_launch(ap_ctx *ctx, cudaStream_t s);   // pair lists of the loaded configuration
int lists_alloc(ap_ctx *ctx);
// when a context is made: the shared-memory limits of the kernels it launches (allow_smem in pair_walk.cuh)
int lists_init(ap_ctx *ctx);
int real_init(ap_ctx *ctx);
int forces_init(ap_ctx *ctx);
int md_init(ap_ctx *ctx);
int real_field_launch(ap_ctx *ctx, cudaStream_t s);
int real_matvec_launch(ap_ctx *ctx, const void *p, cudaStream_t s);
int real_matvec_resident_per_sm(ap_ctx *ctx);
int short_matvec_launch(ap_ctx *ctx, const void *p, double *out, cudaStream_t s);
int pme_init(ap_ctx *ctx);
bool fft_supported(const ap_ctx *ctx);
int fft_init(ap_ctx *ctx, const float *green);
int fft_roundtrip_own(ap_ctx *ctx, const float *in, float2 *c, float *out, cudaStream_t s);
int fft_there_own(ap_ctx *ctx, const float *in, float2 *c, cudaStream_t s);
int fft_back_own(ap_ctx *ctx, float2 *c, float *out, cudaStream_t s);
int2 fft_factors(const ap_ctx *ctx, int d);
int pme_multipole_field(ap_ctx *ctx, cudaStream_t s);              // permanent: grid2 keeps phi_M
// T_rec p -> rec; grid_cleared: the caller has zeroed the context's grid (no clearing here)
int pme_dipole_field(ap_ctx *ctx, const void *p, cudaStream_t s, bool grid_cleared = false);
int dipole_operator_into(ap_ctx *ctx, cudaStream_t main, cudaStream_t aux);   // T p, both branches
// a set of PME work grids and (where the transforms are cuFFT's) plans; the context owns one, others allow concurrent passes
struct PmeBufs {
    void *grid = nullptr, *cgrid = nullptr;
    long long *grid_fx = nullptr;
    cufftHandle r2c = 0, c2r = 0;
};
int pme_bufs_create(ap_ctx *ctx, PmeBufs *b);
void pme_bufs_destroy(PmeBufs *b);
// T_rec p -> rec_out, on the given grids (NULL: the context's own)
int pme_dipole_field_into(ap_ctx *ctx, const void *p, void *rec_out, const PmeBufs *bufs, cudaStream_t s);
int real_matvec2_launch(ap_ctx *ctx, const void *p0, const void *p1, double *acc0, double *acc1,
                        cudaStream_t s);   // T_real on two dipole sets
int field_finish(ap_ctx *ctx, double *d_field_out);
int pcg_solve(ap_ctx *ctx, const double *d_guess, double tol, int max_iter, double *d_mu,
              ap_solve_info *info);
// energy, forces and (d_virial non-NULL) the virial [9] at caller-order dipoles d_mu
int forces_run(ap_ctx *ctx, const double *d_mu, double *d_energy, double *d_forces, double *d_virial);
// the same with extra terms before the frame chain rule; vir: a virial accumulator (virial_acc) or NULL
int forces_run_ex(ap_ctx *ctx, const double *d_mu, double *d_energy, double *d_forces,
                  int (*extra)(ap_ctx *, cudaStream_t), double *vir);
// forces of -(f/2) mu.T mu alone (mz: zeroed multipoles); vir as above
int mutual_forces_run(ap_ctx *ctx, const double *d_mu, void *const *mz, double *gd, double *gq,
                      double *d_forces, double *vir);
double *virial_acc(ap_ctx *ctx, int which);   // nine device slots: 0 a force call, 1 the mutual pass
int virial_out(ap_ctx *ctx, const double *a, const double *b, double *d_virial);   // a - b -> FP64 [9]
// smooth-PME potential derivatives for the forces; with vir non-NULL also the structure-factor
// share of the virial (permanent-induced and induced-induced, or induced-induced alone for _mu)
int pme_forces_derivs(ap_ctx *ctx, const void *mu4, double *gbuf, cudaStream_t s, double *vir);
int pme_forces_derivs_mu(ap_ctx *ctx, const void *mu4, double *gbuf, cudaStream_t s, double *vir);
int diis_solve(ap_ctx *ctx, const double *d_guess, double tol, int max_iter, int depth, double *d_mu,
               ap_solve_info *info);
void diis_release(ap_ctx *ctx);
int diis_info(ap_ctx *ctx, ap_solve_info *info);   // state of the last DIIS solve; synchronizes
int dp_set_pairs(ap_ctx *ctx, int n_pairs, const int *d_pairs, const double *d_scales);
int dp_fields(ap_ctx *ctx, double *d_field_d, double *d_field_p);
int dp_solve(ap_ctx *ctx, const double *gd, const double *gp, double tol, int max_iter, double *d_mu_d,
             double *d_mu_p, ap_solve_info *info);
int dp_forces(ap_ctx *ctx, const double *d_mu_d, const double *d_mu_p, double *d_energy, double *d_forces,
              double *d_virial);
int dp_info(ap_ctx *ctx, ap_solve_info *info);
int dp_matvec2_launch(ap_ctx *ctx, cudaStream_t s);
void dp_release(ap_ctx *ctx);
void diis_forget_graph(ap_ctx *ctx);
void dp_forget_graph(ap_ctx *ctx);   // drop the captured two-set solve loop (launch shapes changed)
