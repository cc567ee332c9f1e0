// kernels.h -- host-side launchers of the libfld CUDA kernels.
#pragma once
#include <cuda_runtime.h>
#include "common.cuh"
#include "df.cuh"
#include "fld.h"

namespace fld {

// Physical constants of one step, precomputed on the host.  theta is the
// time discretisation of the theta-method: the operator A carries theta
// times the face weights and loss rates, the right-hand side the full ones.
struct PhysDev {
    double dt, c, Dmax, Rmin, sigma, adot;
    double h[3];        // cell widths
    double dt_h2[3];    // theta dt / h^2 (face weights of A per unit D)
    double wmax[3];     // theta dt D_max / h^2, the weight of a capped face
    double dtcs;        // dt c sigma (right-hand side and photon balance)
    double one_dta;     // 1 + theta dt adot/a (mass term of A)
    double dta;         // dt adot/a
    double mdtcs;       // theta dt c sigma (mass term of A)
    double theta, inv_theta;
    double ebc[6];      // E_b of the Dirichlet faces: x lo, x hi, y lo, ...
    int dmask;          // bit s set: side s (2 axis + upper) is Dirichlet
    float wmax32[3];    // FP32 copy of wmax
    float sigmaL32;     // sigma L_unit
    float twoL_h32[3];  // 2 L_unit / h
    float thr32;        // screen threshold on 9 (kappa_f L)^2 + (R L)^2
    int limiter;        // 0 paper, 1 Levermore-Pomraning
    // double-float constants of the mixed-precision kernels (k_mixed.cu)
    df sigh[3];         // sigma h: optical depth of a cell per unit n_HI
    df cw[3];           // theta dt c / h: a face weight is cw K S / sqrt(X)
    df rminh[3];        // R_min h
    df wmaxd[3];        // wmax (hi = wmax32)
    df one_dta_d, mdtcs_d;   // mass term m = one_dta + mdtcs n_HI
    df dtcs_d, dta_d;        // loss rate dt (c sigma n_HI + adot/a)
    df dtm_d;                // dt = dtm 2^dt_exp, dtm in [1, 2)
    df ith_d;                // 1 / theta
    int dt_exp;
    int df_limiter;     // the df limiter's constants lie in the FP32 range
};

// Operator of one level: mass term m, lower-face weights, inverse diagonal.
template <class T>
struct Op {
    T *m, *wx, *wy, *wz, *invd;
};

// Weights of the Dirichlet faces of a level (theta-scaled, on the diagonal
// of A), packed by side in the order x lo, x hi, y lo, y hi, z lo, z hi; the
// face of cell (i,j,k) on an x side has index j + ny k, on a y side
// i + nx k, on a z side i + nx j.  w == nullptr: no Dirichlet face.
struct Bnd {
    double* w;
    int mask;           // Dirichlet sides, bit 2 axis + upper
};

__host__ __device__ inline long long bnd_side_size(const Dims& d, int s) {
    const int a = s >> 1;
    return a == 0 ? (long long)d.ny * d.nz : (a == 1 ? (long long)d.nx * d.nz : (long long)d.nx * d.ny);
}
__host__ __device__ inline long long bnd_offset(const Dims& d, int s) {
    long long o = 0;
    for (int q = 0; q < s; q++) o += bnd_side_size(d, q);
    return o;
}

// Cell (i, j, k) of face f (within side sd) of level d.
__device__ __forceinline__ void bnd_cell(const Dims& d, int sd, long long f, int& i, int& j, int& k) {
    const int a = sd >> 1, hi = sd & 1;
    const unsigned nu = a == 0 ? d.ny : d.nx;
    const int v = (int)((unsigned)f / nu), u = (int)((unsigned)f - (unsigned)v * nu);
    if (a == 0) { i = hi ? d.nx - 1 : 0; j = u; k = v; }
    else if (a == 1) { i = u; j = hi ? d.ny - 1 : 0; k = v; }
    else { i = u; j = v; k = hi ? d.nz - 1 : 0; }
}

// Per-block lists of the faces the FP32 screen could not settle, finished
// by a compacted FP64 pass.  entries == nullptr disables the lists.
struct FaceList {
    unsigned* entries;   // block b owns entries[b * cap, (b + 1) * cap)
    unsigned* counts;    // entries used per block
    int cap;
};

// ---- assembly (k_assemble.cu)
// The assembly kernels walk the planes in nzb z-blocks of kch planes each
// (grid sh); a launch covers the z-blocks [zb0, zb0 + nzb) (nzb < 0: all),
// so the assembly of a grid can follow its planes as they arrive.  The
// face lists belong to the blocks of this decomposition.
struct AsmShape {
    ColShape sh;
    int kch, nzb;
};
AsmShape asm_shape(const Dims& d);
// Pass 1: opacity, face limiter and weights (FP64, plus FP32 copies of the
// weights and mass term when op32.m != nullptr); flags invalid inputs.
// Reads E and n_HI of planes zb0 * kch - 1 .. (zb0 + nzb) * kch - 1.
void launch_assemble_faces(const Dims& d, const PhysDev& p, const double* E, const double* nHI,
                           const double* eta, Op<double> op, Op<float> op32, double* sc,
                           FaceList fl, cudaStream_t s, int zb0 = 0, int nzb = -1);
// FP64 limiter for the listed faces of those z-blocks (one block per list
// segment).
void launch_assemble_fix(const Dims& d, const PhysDev& p, const double* E, const double* nHI,
                         Op<double> op, Op<float> op32, FaceList fl, cudaStream_t s, int zb0 = 0,
                         int nzb = -1);
// Size of the face lists for a level: blocks of the faces launch and
// entries per block (0 when lists are not used).
void face_list_shape(const Dims& d, int limiter, long long* blocks, int* cap);
// Pass 2: right-hand side b, inverse diagonals (FP64 if op.invd, FP32 if
// op32.invd), the FP64 diagonal if diag64, ||b||^2 into slot0 and max |b|
// into slot1.  Cells on a Dirichlet face (p.dmask) also get the face's
// limiter weight: stored in bnd, added to m (FP64 and FP32) and its flux
// to b.  Needs the weights of the planes one past its z-blocks (upper
// z faces) and E of the planes on either side.
void launch_assemble_rhs(const Dims& d, const PhysDev& p, const double* E, const double* nHI,
                         const double* eta, Op<double> op, Op<float> op32, double* b, double* diag64,
                         Bnd bnd, const RedArgs& ra, cudaStream_t s, int zb0 = 0, int nzb = -1);
// The limiter weights of the Dirichlet faces of the cells in planes [k0, k1)
// into bnd.w, all sides in one launch; launch_assemble_rhs and
// launch_asm_rhs_mx read them.  (In the right-hand side's sweep, where the
// face cells are one or two lanes of a warp, the FP64 limiter cost 50 of its
// 87 us at 128 x 64 x 64; this launch takes 8.)
void launch_bnd_weights(const Dims& d, const PhysDev& p, const double* E, const double* nHI, Bnd bnd, int k0, int k1,
                        cudaStream_t s);
// Photons through the Dirichlet faces over the step (before the finalisation
// overwrites E): per side s the sum of w_b (inv_theta (E - E_b) + dE) into slot
// S_OUT0 + s and the sum of its absolute values into S_OUTABS0 + s, all sides
// in one launch (reduction ra with op R_STORE2; it uses the six counters and
// partials after ra's).
void launch_bnd_outflow(const Dims& d, const PhysDev& p, Bnd bnd, const double* E, const double* dE,
                        const RedArgs& ra, cudaStream_t st);
// Blocks per side of such a launch, and side sd's share of the reduction.
constexpr int BND_MAX_BLOCKS = 1024;
inline int bnd_blocks(const Dims& d) {
    long long m = 0;
    for (int s = 0; s < 6; s += 2) m = bnd_side_size(d, s) > m ? bnd_side_size(d, s) : m;
    const int b = red_blocks(m);
    return b < BND_MAX_BLOCKS ? b : BND_MAX_BLOCKS;
}
__device__ __forceinline__ RedArgs bnd_red(RedArgs ra, int sd) {
    ra.partials += sd * BND_MAX_BLOCKS;
    ra.counter += 1 + sd;
    ra.slot0 = S_OUT0 + sd;
    ra.slot1 = S_OUTABS0 + sd;
    return ra;
}

// ---- mixed-precision step on the FP32 pipe in double-float arithmetic
// (k_mixed.cu).  The fine operator is (A, L): the FP32 operator of the
// V-cycles and the low parts of m and the weights.
// Pass 1: m and the face weights (df), input validation into sc[S_BAD], the
// maxima of E, n_HI and eta into sc[S_EMAX], sc[S_NMAX], sc[S_ETAMAX] (the
// caller zeroes them with the other slots before the assembly).
// Faces the FP32 screen does not settle go to the per-block lists fl (when
// fl.entries is set), finished by launch_asm_fix_mx.
void launch_asm_faces_mx(const Dims& d, const PhysDev& p, const double* E, const double* nHI, const double* eta,
                         Op<float> A, Op<float> L, double* sc, FaceList fl, cudaStream_t s, int zb0 = 0,
                         int nzb = -1);
// The df limiter for the listed faces of those z-blocks.
void launch_asm_fix_mx(const Dims& d, const PhysDev& p, const double* E, const double* nHI, Op<float> A,
                       Op<float> L, FaceList fl, cudaStream_t s, int zb0 = 0, int nzb = -1);
// Pass 2: b (FP64), ||b||^2 and max |b| (reduction ra, R_STORE_SUM_MAX), the
// FP32 inverse diagonal A.invd, Dirichlet face weights into bnd and m; scg:
// the slots of pass 1's maxima.  Needs pass 1 of its z-blocks and the one
// above.
// Bf: where its pointers are set, also the bfloat16 copies (nearest) of the
// FP32 weights wx, wy, wz and of the FP32 inverse diagonal.
void launch_asm_rhs_mx(const Dims& d, const PhysDev& p, const double* E, const double* nHI, const double* eta,
                       Op<float> A, Op<float> L, double* b, Bnd bnd, const RedArgs& ra, const double* scg,
                       cudaStream_t s, int zb0 = 0, int nzb = -1, Op<unsigned short> Bf = {});
// r32 = b 2^-ks (nearest float); ||r32||^2, max |r32| (R_IRRES).
void launch_ir_scale_b(long long n, const double* b, int ks, float* r32, const RedArgs& ra, cudaStream_t s);
// The refinement unknown x (dE) of the mixed solver is a df pair per cell
// (float2), scaled by 2^-K with K the step's scale exponent (from the
// maxima in scg, the context's slots).
// x += 2^ks x32 (assign: x = 2^ks x32); p_last (optional): x32 still lacks
// the last CG iteration's update, x32 + sc[S_ALPHA] p_last in FP32 is used
void launch_ir_update_mx(long long n, void* x, const float* x32, const double* sc, bool assign, int ks,
                         const float* p_last, const double* scg, int dt_exp, cudaStream_t s);
// r = b - m x - sum_f w_f (x - x_nbr) in df; ||r32||^2, max |r32| of r32 =
// r 2^-ks (nearest float) (R_IRRES), r32 itself only with write.
void launch_ir_residual(const Dims& d, Op<float> A, Op<float> L, const double* b, const void* x, int ks,
                        float* r32, bool write, const RedArgs& ra, const double* scg, int dt_exp, cudaStream_t s);
ColShape ir_residual_shape(const Dims& d);
// E_out = max(E + dE, 0) and the photon-balance sums as launch_finalize,
// summed in df relative to the scales of the maxima in scg; dE the df x.
void launch_finalize_mx(long long n, const PhysDev& p, const double* E, const void* dE, const double* nHI,
                        const double* eta, double* E_out, const RedArgs& ra, const double* scg, cudaStream_t s);
// launch_bnd_outflow with dE the df x
void launch_bnd_outflow_mx(const Dims& d, const PhysDev& p, Bnd bnd, const double* E, const void* dE,
                           const RedArgs& ra, const double* scg, cudaStream_t st);
// the df x as FP64 values (fld_solve's output)
void launch_dE_to_f64(long long n, const void* x, double* out, const double* scg, int dt_exp, cudaStream_t s);
// out = h + l in FP64 (inspection hooks)
void launch_df_to_f64(long long n, const float* h, const float* l, double* out, cudaStream_t s);
// y = A x with the df operator, in FP64 (test hook)
void launch_apply_mx(const Dims& d, Op<float> A, Op<float> L, const double* x, double* y, cudaStream_t s);

// ---- multigrid (k_mg.cu), T = float or double
// With Dirichlet faces (FB, CB) also the coarse face weights (sum of the 4
// fine ones / 16); the coarse mass term, the mean of the children's full m,
// gives back the difference: m_c -= w_c.
template <class T>
void launch_coarsen(const Dims& f, const Dims& c, Op<T> F, Op<T> C, Bnd FB, Bnd CB, cudaStream_t s);
template <class T>
void launch_invd(const Dims& d, Op<T> A, const Op<T>& src, cudaStream_t s);
template <class T>
void launch_smooth_zero(const Dims& d, Op<T> A, const T* r, T* z, cudaStream_t s);
template <class T>
void launch_rb_colour(const Dims& d, Op<T> A, const T* r, T* z, int colour, cudaStream_t s);
template <class T>
void launch_jacobi(const Dims& d, Op<T> A, const T* r, const T* z, T* out, double omega,
                   bool zero_guess, cudaStream_t s);
template <class T>
void launch_residual(const Dims& d, Op<T> A, const T* r, const T* z, T* res, cudaStream_t s);
template <class T>
void launch_restrict(const Dims& f, const Dims& c, const T* rf, T* rc, cudaStream_t s);
template <class T>
void launch_prolong_add(const Dims& f, const Dims& c, const T* ec, T* zf, cudaStream_t s);
// ---- FP64 sweeps, a red/black pair of cells per thread (k_pair.cu); need an
// even x extent.  res: the residual at the red cells after a sweep from zero,
// n / 2 values, cell l at l >> 1.
bool pair_ok(const Dims& d);
void launch_zero_pair(const Dims& d, Op<double> A, const double* r, double* z, cudaStream_t s);
void launch_residual_pair(const Dims& d, Op<double> A, const double* z, double* res, cudaStream_t s);
// launch_restrict_pair also serves the FP32 cycle up to this many coarse cells:
// a cell per thread there keeps the GPU full where four cells per thread
// (launch_restrict4) leave it idle, and costs more instructions per cell.
// A step of 64^3 (coarse 32^3) takes 951 us instead of 976, of 128x64x64 1244
// instead of 1286; with the coarse 64^3 of 128^3 as well, one of 128^3 with
// four groups 4434 instead of 4340, and of 512^3 57.2 ms instead of 53.9.
constexpr long long RESTRICT_PAIR_CELLS = 131072;
template <class T>
void launch_restrict_pair(const Dims& f, const Dims& c, const T* res, T* rc, cudaStream_t s);
// z += P ec at the cells of colour col
void launch_correct_pair(const Dims& f, const Dims& c, const double* ec, double* z, int col, cudaStream_t s);
// one colour of a sweep, with <r, z> of the result when dot is given
void launch_colour_pair(const Dims& d, Op<double> A, const double* r, double* z, int col, const RedArgs* dot,
                        cudaStream_t s);
void launch_pq_pair(const Dims& d, Op<double> A, const double* z, const double* p_in, double* p_out, double* q,
                    const RedArgs& ra, cudaStream_t s);

// ---- coarsest grid (k_coarse.cu): the explicit inverse in ainv (n x n words
// of 8 bytes: FP64 for T = double, a float pair high + low for T = float;
// fp32: of FP32 accuracy up to 160 cells, else FP64 accuracy).  dense: n x n
// FP64 words of scratch; flag: one word of scratch; a non-positive pivot
// sets sc[S_BAD] = 2.
template <class T>
void launch_coarse_setup(const Dims& d, Op<T> A, double* dense, double* ainv, double* sc, unsigned* flag, bool fp32,
                         cudaStream_t s);
template <class T>
void launch_coarse_apply(int n, const double* ainv, const T* r, T* z, cudaStream_t s);

// ---- Krylov and refinement (k_cg.cu)
template <class T>
void launch_dot(long long n, const T* a, const T* b, const RedArgs& ra, cudaStream_t s);
template <class T>
void launch_cg_p_matvec(const Dims& d, Op<T> A, const T* z, const T* p_in, T* p_out, T* q,
                        const RedArgs& ra, cudaStream_t s);
template <class T>
void launch_cg_update(long long n, T* x, T* r, const T* p, const T* q, const RedArgs& ra,
                      cudaStream_t s);
template <class T>
void launch_apply(const Dims& d, Op<T> A, const T* x, T* y, cudaStream_t s);
// element-wise precision conversions (test hooks)
void launch_f64_to_f32(long long n, const double* a, float* b, cudaStream_t s);
void launch_f32_to_f64(long long n, const float* a, double* b, cudaStream_t s);
// Device-side CG convergence test: sc[S_KITER] += 1 and the conditional h
// set to continue while sc[S_RR] > sc[S_THRESH], S_KITER < S_MAXIT and no
// non-finite reduction (one thread).
// Slots of a reduction done in chunks (at most 8).
struct SlotList {
    int n;
    int s[8];
};
// sc[slot] = the chunks' slot summed in chunk order, for each listed slot,
// and the non-finite flag of any chunk.
void launch_combine_sums(const double* chunk_sc, int nch, double* sc, const SlotList& sl, cudaStream_t s);
// Reductions done in nch chunks, each into its own block of NUM_SLOTS
// slots: sc[s_sum] = the chunks' s_sum summed in chunk order, sc[s_max] =
// their s_max maximised, and the non-finite flag of any chunk.
void launch_combine_chunks(const double* chunk_sc, int nch, double* sc, int s_sum, int s_max, cudaStream_t s);
void launch_cg_check(cudaGraphConditionalHandle h, double* sc, cudaStream_t s,
                     const cudaGraphConditionalHandle* h2 = nullptr);
// The launch shape of launch_residual64 (callers that size reduction
// scratch for it check its block count).
ColShape residual64_shape(const Dims& d);
// r64 = b - A x (FP64); ||r64||^2 -> slot0, max|r64| -> slot1.  diag (may
// be null) is the stored FP64 diagonal.
void launch_residual64(const Dims& d, Op<double> A, const double* diag, const double* b, const double* x,
                       double* r, const RedArgs& ra, cudaStream_t s);
// E_out = max(E + dE, 0); sums for the photon balance into S_BAL (dE),
// S_EMIT (eta), S_ABSORB (n_HI E^theta), S_ESUM (E^theta), the floor's
// energy into S_FLOOR, sum dE^2 into S_DE2, sum E_out^2 into S_EN2
// (reduction R_STORE7_FIN).
void launch_finalize(long long n, const PhysDev& p, const double* E, const double* dE,
                     const double* nHI, const double* eta, double* E_out, const RedArgs& ra,
                     cudaStream_t s);
void launch_opacity_update(long long n, const double* E, const double* nH, const double* nHI,
                           double* out, double dt, double c, double sigma, double hnu,
                           double alpha_B, cudaStream_t s);

// ---- persistent coarse tail of the V-cycle (k_tail.cu): levels L[0] (the
// first level at or below the size threshold) to L[nlev - 1] (the coarsest)
// in one launch of one cluster of `cluster` CTAs.  L[0].r is the input,
// L[0].z the output; the other r, z, t are the levels' work vectors.
constexpr int TAIL_MAX_LEVELS = 12;
// levels of at most this many cells run in one CTA in shared memory
constexpr long long TAIL_SOLO_CELLS = 4096;
constexpr long long TAIL_SOLO_CELLS64 = 512;   // FP64
// the largest level of an FP64 tail: at 32^3 the 16 SMs of a cluster take 40 us
// for a level whose six launches over the whole GPU take 27
constexpr int TAIL_CELLS64 = 4096;
constexpr size_t TAIL_SMEM_MAX = 208 * 1024;
template <class T>
struct TailLevel {
    Dims d;
    Op<T> A;
    T *r, *z, *t;
    int o_r, o_z, o_t, o_c, o_i;   // shared-memory offsets of a solo level's r, z,
                                   // red residual, coefficients, pair table
};
template <class T>
struct TailArgs {
    int nlev, pre, post;
    int paper_order;  // post-sweeps red then black (else black then red)
    // filled by plan_tail:
    int small_from;   // first level run by one CTA in shared memory
    int slab;         // level run as halo slabs of the cluster's CTAs (-1: none)
    int slab_axis;
    int big_coarse;   // the coarsest grid is applied by the whole cluster
    int coef_smem;    // solo coefficients in shared memory
    int solve;        // layout of a whole inner solve by one CTA
    int o_slab_r, o_slab_z, o_slab_t, o_slab_i, o_p, o_ainv;
    int smem_bytes;
    const double* ainv;   // coarsest inverse (see launch_coarse_setup)
    TailLevel<T> L[TAIL_MAX_LEVELS];
};
// Chooses how the levels run and the shared-memory layout for a cluster of
// that many CTAs; false if it does not fit.
template <class T>
bool plan_tail(TailArgs<T>& a, int cluster, bool solve);
template <class T>
cudaError_t launch_vtail(const TailArgs<T>& a, int cluster, cudaStream_t s);
// the cluster size to launch the tail with (16 or 8 CTAs), 0 if no cluster
// of the tail kernel can be resident on this device
template <class T>
int vtail_cluster();

// ---- persistent inner solves over a work list (k_tail.cu, mixed
// precision): each cluster takes requests by ticket and runs a request's
// whole FP32 MG-PCG solve (V-cycles over all its levels and the CG vector
// operations) to ||r||^2 <= sc[S_THRESH] or sc[S_MAXIT] iterations.
struct PsReq {
    TailArgs<float> v;   // all levels; L[0].r is the CG residual (in: the
                         // right-hand side, x = 0), L[0].z the preconditioned one
    float *x, *p, *q;    // fine-level CG vectors
    double* sc;          // the request's scalar slots: S_THRESH, S_MAXIT in;
                         // S_KITER, S_RR, S_RHO.., S_NONFINITE out
    int cta;             // 1: solved by one CTA with every level in its
                         // shared memory (plan_tail with solve), else by a cluster
    int pad_;
};
constexpr int PS_MAX_BATCH = 256;
constexpr int PS_CLUSTER = 8;
// the most dynamic shared memory of a persistent launch
constexpr size_t PS_SMEM_MAX = 208 * 1024;
struct PsBatch {
    int n;          // requests: [0, ncl) by clusters, [ncl, n) by single CTAs
    int ncl;
    unsigned* ticket;                 // two counters, set to 0 by launch_psolve
    const PsReq* req[PS_MAX_BATCH];   // device descriptors, in work-list order
};
struct PsShape {
    int cluster;    // CTAs per cluster
    int clusters;   // clusters resident at once
};
PsShape psolve_shape();
// one launch: min(n, resident clusters) clusters drain the work list; smem
// is the largest smem_bytes of the batch's plans
cudaError_t launch_psolve(const PsBatch& b, size_t smem, cudaStream_t s);

// Sets the calling thread's fld_last_error message (fld_api.cu).
void record_error(const char* msg);
// The per-face boundary conditions of g are consistent (fld_create's rule);
// otherwise false with the reason in msg (fld_api.cu).
bool bc_valid(const fld_grid* g, char* msg, size_t len);

// Launch shape of a four-cells-per-thread sweep: threads per block (a
// power of two up to 256, x lanes first) and the total blocks aimed at (the
// z-chunk length follows).  Chosen per level and kernel by fld_autotune.
struct Tune {
    int threads = 256;
    int target = 152 * 8;
    int pf = 1;             // L2 prefetch distance in planes (0: none; FP32 sweeps)
};

// Lanes along x of a sweep's blocks, whose threads tile h: 16 or 8 where 32 (16)
// would leave more than a tenth of them past the row's end (24 or 40 threads
// in 32s leave 25 and 37 %; a row of 8 lanes of 16 bytes is still one line).
// Only for launches that fill the GPU: below, the idle lanes cost nothing and
// the extra row ends do.  Per launch at 320^3 (rows of 40 threads, p/q 80), 32
// lanes -> this rule: smoothing 145 -> 123 us, residual 77 -> 67, black sweep
// 106 -> 96, red 139 -> 120, correction 58 -> 42, restriction 66 -> 46, p/q 233
// -> 220.
constexpr long long ROW_LANES_MIN = 1 << 18;
inline int row_lanes(const Dims& h) {
    int lanes = 32;
    if ((long long)h.nx * h.ny * h.nz < ROW_LANES_MIN) return lanes;
    for (int b : {16, 8}) {
        const int now = (h.nx + lanes - 1) / lanes * lanes, less = (h.nx + b - 1) / b * b;
        if (10 * less < 9 * now) lanes = b;
    }
    return lanes;
}

// Launch shape of a sweep whose threads tile h (x extent in threads).  The
// default record stands for the library's own choice: z-chunks 14 planes long
// where that leaves at least five blocks per SM (the last wave of two or three
// per SM then costs little, and a chunk's first plane, which reads three
// planes, is a small share), else 8, else 4 planes where 1.5 blocks per SM
// remain, else one.  A fixed 152 x 8 blocks gave two and a half waves and
// chunks of 52 to 128 planes at 512^3 and one or two planes at 128^3.
// Measured per launch, fixed -> this rule: p/q 1024 -> 824 us, smoothing 447 ->
// 411, residual 247 -> 215, black sweep 407 -> 340, red sweep 401 -> 369 at
// 512^3; p/q 29 -> 25, smoothing 18.0 -> 15.6, red 20.9 -> 16.3 at 128^3
// (longer chunks there: p/q 28 at 7 planes; shorter at 512^3: red 386 at 7,
// smoothing 423).
inline ColShape sweep_shape(const Dims& h, const Tune& tn) {
    const Tune def;
    const int lanes = row_lanes(h);
    if (tn.threads != def.threads || tn.target != def.target) return col_shape(h, tn.threads, tn.target, lanes);
    const ColShape one = col_shape(h, def.threads, 1, lanes);
    const long long xy = (long long)one.grid.x * one.grid.y;
    long long blocks = xy * h.nz;
    for (int kch : {14, 8, 4}) {
        const long long b = xy * ((h.nz + kch - 1) / kch);
        if (b >= (kch > 4 ? 152 * 5 : 152 * 3 / 2)) {
            blocks = b;
            break;
        }
    }
    if (blocks > RED_MAX_BLOCKS) blocks = RED_MAX_BLOCKS;
    return col_shape(h, def.threads, (int)blocks, lanes);
}
constexpr int TUNE_FIELDS = 3;      // entries of one tuning-table record
constexpr int TUNE_PF_MAX = 8;

// ---- FP32 four-cells-per-thread sweeps (k_fine4.cu); need nx % 4 == 0
bool fine4_ok(const Dims& d);
// x (optional): also x += alpha_prev p_in, the previous iteration's update
// of x (see launch_cg_update4 with x null)
void launch_cg_p_matvec4(const Dims& d, Op<float> A, const float* z, const float* p_in, float* p_out,
                         float* q, const RedArgs& ra, cudaStream_t s, const Tune& tn = Tune{},
                         float* x = nullptr);
// after_zero_sweep: z comes from one red/black sweep from z = 0 (black
// last), so the residual is sum_f w_f z_nbr at red cells and 0 at black
// ones; red_compressed (with after_zero_sweep, where red_compress_ok):
// stored red-compressed, res[l >> 1] for red cell l
void launch_residual4(const Dims& d, Op<float> A, const float* r, const float* z, float* res,
                      cudaStream_t s, const Tune& tn = Tune{}, bool after_zero_sweep = false,
                      bool red_compressed = false);
bool red_compress_ok(const Dims& f);
void launch_smooth_zero4(const Dims& d, Op<float> A, const float* r, float* z, cudaStream_t s,
                         const Tune& tn = Tune{});
void launch_rb_colour4(const Dims& d, Op<float> A, const float* r, float* z, int colour,
                       cudaStream_t s, const Tune& tn = Tune{});
// The same sweeps with the smoothing operator's coefficients (wx, wy, wz,
// invd; m unused) stored as bfloat16 (the upper 16 bits of the FP32
// values, rounded to nearest); the residual only in its zero-guess form.
void launch_smooth_zero4(const Dims& d, Op<unsigned short> A, const float* r, float* z, cudaStream_t s,
                         const Tune& tn = Tune{});
void launch_rb_colour4(const Dims& d, Op<unsigned short> A, const float* r, float* z, int colour,
                       cudaStream_t s, const Tune& tn = Tune{});
void launch_rb_colour4_dot(const Dims& d, Op<unsigned short> A, const float* r, float* z, int colour,
                           const RedArgs& ra, cudaStream_t s, const Tune& tn = Tune{});
void launch_residual4(const Dims& d, Op<unsigned short> A, const float* z, float* res, cudaStream_t s,
                      const Tune& tn, bool red_compressed);
// ---- red/black compressed sweeps (k_fine8.cu): bfloat16 coefficients, one
// sweep down and one up; need nx % 8 == 0.  zr, zb, res: n / 2 values, cell l
// of the colour at l >> 1.
bool fine8_ok(const Dims& d);
// zr, zb: one red/black sweep from zero
void launch_zero8(const Dims& d, Op<unsigned short> A, const float* r, float* zr, float* zb, cudaStream_t s,
                  const Tune& tn);
// res: its residual at the red cells (launch_restrict4's compressed form)
void launch_residual8(const Dims& d, Op<unsigned short> A, const float* zb, float* res, cudaStream_t s,
                      const Tune& tn);
// zr += P ec at the red cells
void launch_correct8(const Dims& f, const Dims& c, const float* ec, float* zr, cudaStream_t s, const Tune& tn);
// zb from zr; then z (natural order) from zb, with <r, z> when dot is given
void launch_black8(const Dims& d, Op<unsigned short> A, const float* r, const float* zr, float* zb, cudaStream_t s,
                   const Tune& tn);
void launch_red8(const Dims& d, Op<unsigned short> A, const float* r, const float* zb, float* z, const RedArgs* dot,
                 cudaStream_t s, const Tune& tn);
// B.wx, wy, wz, invd = the bfloat16 values nearest to A's (n a multiple of 4).
void launch_op_to_bf16(long long n, Op<float> A, Op<unsigned short> B, cudaStream_t s);
void launch_dot4(long long n, const float* a, const float* b, const RedArgs& ra, cudaStream_t s);
// one colour of a sweep followed by <r, z> of the result (reduction ra)
void launch_rb_colour4_dot(const Dims& d, Op<float> A, const float* r, float* z, int colour,
                           const RedArgs& ra, cudaStream_t s, const Tune& tn = Tune{});
// red_compressed: rf is a red-compressed residual (k_residual4 after a
// zero-guess sweep), cell l red ? rf[l >> 1] : 0
void launch_restrict4(const Dims& f, const Dims& c, const float* rf, float* rc, cudaStream_t s,
                      const Tune& tn = Tune{}, bool red_compressed = false);
// Fused post-smoothing sweep (black then red), out of place zi -> zo, with
// <r, zo> into *dot when dot is given; post4_ok tells if a level qualifies.
bool post4_ok(const Dims& d);
void launch_post_smooth4(const Dims& d, Op<float> A, const float* r, const float* zi, float* zo,
                         const RedArgs* dot, cudaStream_t s, const Tune& tn = Tune{});
// zo = z + P ec (out of place)
void launch_prolong_to4(const Dims& f, const Dims& c, const float* ec, const float* z, float* zo,
                        cudaStream_t s);
void launch_prolong_add4(const Dims& f, const Dims& c, const float* ec, float* zf, cudaStream_t s,
                         const Tune& tn = Tune{});
// x null: r -= alpha q only, the update of x deferred to the next
// launch_cg_p_matvec4 (and the last one to launch_ir_update)
void launch_cg_update4(long long n, float* x, float* r, const float* p, const float* q,
                       const RedArgs& ra, cudaStream_t s);

}  // namespace fld
