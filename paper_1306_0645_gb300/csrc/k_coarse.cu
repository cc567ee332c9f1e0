// k_coarse.cu -- the coarsest grid of the V-cycle: its explicit inverse,
// formed once per assembly, and z = A^-1 r.
//
// The inverse comes from Gauss-Jordan elimination without pivoting (stable
// for the symmetric positive definite operator) in FP32:
//  - up to 160 cells one CTA holds the matrix in registers, PT x PT entries
//    per thread.  A step publishes the pivot row and column in shared memory
//    (two buffers, so one barrier per step) and updates every entry.  What
//    bounds it is the serial chain of n steps (barrier, reciprocal, two
//    shared-memory reads), 0.3 to 0.5 us each: 24 us at 64 cells, 64 at 128.
//    Steps of 32 rows as below take 22 and 56 us, which a step of a 16^3
//    or 128x64x64 grid does not show.
//  - larger grids take elimination steps of 32 rows, one launch per step over
//    64 x 64 tiles of the whole matrix (two copies, read and written in
//    turn).  Every CTA inverts the 32 x 32 pivot block itself, in the registers
//    of one warp while the others load the tile, which costs less than another
//    launch: a step of 693 cells takes 10.4 us, 13.5 with the inversion by the
//    whole CTA and a barrier per row.
// The mixed solver uses that FP32 inverse up to 160 cells.  The FP64 solver,
// and the mixed one above 160 cells, refine it to FP64 column by column,
// x += X32 (e - A x) with the residual in FP64 through the 7-point operator
// (7 products per entry, where FP64 elimination needs n).  FP64 runs at 1/64
// of the FP32 rate here, so one FP64 elimination of a 64-cell grid costs more
// than the FP32 one and its refinement together.  A column whose residual
// does not reach rounding level (an operator too ill-conditioned for an FP32
// inverse to contract the error) raises a flag, and an FP64 elimination
// launched behind it, which otherwise returns at once, replaces the result.
#include "kernels.h"

namespace fld {

namespace {

constexpr int GJ_ONE_MAX = 160;    // cells inverted by one CTA in registers
constexpr int GJ64_MAX = 128;      // the same in FP64 (fallback)
constexpr int GB = 32;             // rows per step of the blocked elimination
constexpr int GT = 64;             // its tile

// Adds row c of the operator's dense matrix to row (zeroed before): diagonal
// m + sum of the face weights, -w_f at the neighbours (summed where a
// periodic axis of 1 or 2 cells makes neighbours coincide).
template <class T, class M>
__device__ __forceinline__ void dense_row(const Dims& d, const Op<T>& A, int c, M* row) {
    int i, j, k;
    cell_ijk(c, d, i, j, k);
    const int sy = d.nx, sz = d.nx * d.ny;
    double diag = (double)A.m[c];
    auto add = [&](T wt, int nb) {
        diag += (double)wt;
        if (nb == c) diag -= (double)wt;
        else row[nb] = row[nb] - (M)wt;
    };
    if (i > 0) add(A.wx[c], c - 1); else if (d.px) add(A.wx[c], c + d.nx - 1);
    if (i < d.nx - 1) add(A.wx[c + 1], c + 1); else if (d.px) add(A.wx[c - (d.nx - 1)], c - (d.nx - 1));
    if (j > 0) add(A.wy[c], c - sy); else if (d.py) add(A.wy[c], c + (d.ny - 1) * sy);
    if (j < d.ny - 1) add(A.wy[c + sy], c + sy); else if (d.py) add(A.wy[c - (d.ny - 1) * sy], c - (d.ny - 1) * sy);
    if (k > 0) add(A.wz[c], c - sz); else if (d.pz) add(A.wz[c], c + (d.nz - 1) * sz);
    if (k < d.nz - 1) add(A.wz[c + sz], c + sz); else if (d.pz) add(A.wz[c - (d.nz - 1) * sz], c - (d.nz - 1) * sz);
    row[c] = (M)diag;
}

// Entry i of the coarsest inverse as its solver reads it: FP64, or a float
// pair high + low (FP32 solver).
template <class T>
__device__ __forceinline__ void put_inv(double* X, long long i, double v) {
    if constexpr (sizeof(T) == 4) {
        const float h = (float)v;
        reinterpret_cast<float2*>(X)[i] = make_float2(h, (float)(v - (double)h));
    } else {
        X[i] = v;
    }
}
// FP32 scratch copy of the inverse
template <class T>
__device__ __forceinline__ void put_inv(float* X, long long i, double v) { X[i] = (float)v; }

// In-place inverse of the n x n matrix held by S x S threads, entry
// (ty + S q, tx + S b) in a[q][b]; buf: 4 S PT values of shared memory.
// Step k: p = M[k][k]; M'[k][k] = 1/p, M'[k][j] = M[k][j]/p,
// M'[i][k] = -M[i][k]/p, M'[i][j] = M[i][j] - M[i][k] (M[k][j]/p).  Returns
// false where a pivot was not positive (taken as 1).
template <int S, int PT, class T>
__device__ __forceinline__ bool gj_invert(T (&a)[PT][PT], int n, T* buf, int tx, int ty) {
    constexpr int N = S * PT;
    bool ok = true;
#pragma unroll
    for (int ka = 0; ka < PT; ka++) {
        for (int kk = 0; kk < S; kk++) {
            const int k = ka * S + kk;
            if (k >= n) break;
            T* row = buf + (k & 1) * 2 * N;
            T* col = row + N;
            if (ty == kk) {
#pragma unroll
                for (int b = 0; b < PT; b++) row[tx + S * b] = a[ka][b];
            }
            if (tx == kk) {
#pragma unroll
                for (int q = 0; q < PT; q++) col[ty + S * q] = a[q][ka];
            }
            __syncthreads();
            T p = row[k];
            if (!(p > T(0))) {
                ok = false;
                p = T(1);
            }
            const T ip = T(1) / p;
            T rv[PT], cv[PT];
#pragma unroll
            for (int b = 0; b < PT; b++) rv[b] = row[tx + S * b] * ip;
#pragma unroll
            for (int q = 0; q < PT; q++) cv[q] = col[ty + S * q];
#pragma unroll
            for (int q = 0; q < PT; q++)
#pragma unroll
                for (int b = 0; b < PT; b++) a[q][b] = a[q][b] - cv[q] * rv[b];
            if (ty == kk) {
#pragma unroll
                for (int b = 0; b < PT; b++) a[ka][b] = rv[b];
            }
            if (tx == kk) {
#pragma unroll
                for (int q = 0; q < PT; q++) a[q][ka] = -cv[q] * ip;
            }
            if (tx == kk && ty == kk) a[ka][ka] = ip;
        }
    }
    return ok;
}

// The inverse of the coarsest operator (n <= S PT cells) by one CTA in
// precision R, to X (ld n) as O.  flag != null: raised on a non-positive
// pivot (the refinement's fallback); else sc[S_BAD] = 2.  only_if != null:
// return unless it is raised.
template <class T, class R, class O, int S, int PT>
__global__ void __launch_bounds__(S* S) k_gj_inverse(Dims d, Op<T> A, O* __restrict__ X, double* sc, unsigned* flag,
                                                      const unsigned* only_if) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (only_if && *only_if == 0u) return;
    R* M = reinterpret_cast<R*>(smem_raw);
    __shared__ R buf[4 * S * PT];
    const int n = (int)d.n;
    const int tx = threadIdx.x % S, ty = threadIdx.x / S;
    if (flag && threadIdx.x == 0) *flag = 0u;
    for (int q = threadIdx.x; q < n * n; q += S * S) M[q] = R(0);
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += S * S) dense_row(d, A, c, M + c * n);
    __syncthreads();
    R a[PT][PT];
#pragma unroll
    for (int q = 0; q < PT; q++)
#pragma unroll
        for (int b = 0; b < PT; b++) {
            const int i = ty + S * q, j = tx + S * b;
            a[q][b] = i < n && j < n ? M[i * n + j] : R(0);
        }
    const bool ok = gj_invert<S, PT>(a, n, buf, tx, ty);
#pragma unroll
    for (int q = 0; q < PT; q++)
#pragma unroll
        for (int b = 0; b < PT; b++) {
            const int i = ty + S * q, j = tx + S * b;
            if (i < n && j < n) put_inv<T>(X, (long long)i * n + j, (double)a[q][b]);
        }
    if (!ok && threadIdx.x == 0) {
        if (flag) *flag = 1u;
        else sc[S_BAD] = 2.0;
    }
}

// ---- blocked elimination, n > GJ_ONE_MAX

// In-place inverse of a symmetric positive definite 32 x 32 matrix held by a
// warp, row i of column `lane` in a[i], without pivoting: M'[k][j] = M[k][j] / p,
// M'[i][j] = M[i][j] - f_i M'[k][j] with f_i = M[i][k], and 1 / p, -f_i / p in
// column k.  Each step takes its pivot row from a[0] and shifts the rows by
// one, so the loop stays rolled (32 steps leave them in place).  By symmetry
// f_i is the pivot row's entry in column i (negated for i < k), so every lane
// publishes one value and reads all 32 as eight vectors; with one shuffle per
// f_i a step of the elimination of 693 cells took 11.6 us instead of 10.4.  The
// next pivot row is published before the other rows are updated.  Returns false where a pivot was not positive (taken as
// 1).
__device__ __forceinline__ bool warp_invert(float (&a)[GB], float (&buf)[2][GB], int lane) {
    bool ok = true;
    buf[0][lane] = a[0];
#pragma unroll 1
    for (int k = 0; k < GB; k++) {
        __syncwarp();
        float f[GB];
#pragma unroll
        for (int q = 0; q < GB / 4; q++)
            *reinterpret_cast<float4*>(f + 4 * q) = *reinterpret_cast<const float4*>(buf[k & 1] + 4 * q);
        float p = f[0];
        if (!(p > 0.0f)) {
            ok = false;
            p = 1.0f;
        }
        const float ip = 1.0f / p;
        const bool own = lane == k;
        const float rv = own ? ip : a[0] * ip;
        a[0] = fmaf(-f[1], rv, own ? 0.0f : a[1]);
        buf[(k + 1) & 1][(lane - k - 1) & 31] = lane < k + 1 ? -a[0] : a[0];
#pragma unroll
        for (int i = 2; i < GB; i++) a[i - 1] = fmaf(-f[i], rv, own ? 0.0f : a[i]);
        a[GB - 1] = rv;
    }
    return ok;
}

// The dense matrix in FP32 (a warp per row); clears the flag.
template <class T>
__global__ void __launch_bounds__(256) k_dense32(Dims d, Op<T> A, float* __restrict__ M, unsigned* flag) {
    const int n = (int)d.n;
    const int lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0) *flag = 0u;
    for (int c = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < n; c += (int)(gridDim.x * blockDim.x) >> 5) {
        float* row = M + (long long)c * n;
        for (int q = lane; q < n; q += 32) row[q] = 0.0f;
        __syncwarp();
        if (lane == 0) dense_row(d, A, c, row);
    }
}

// One elimination step with the pivot block of rows [kb, kb + 32) (the rows
// past n as identity): with P the pivot block and t = P^-1 M[kb, :] (the
// block's own columns P^-1), M'[kb, :] = t and M'[i, j] = M[i, j] -
// M[i, kb] t[:, j] for the other rows, M[i, j] taken as 0 in the block's own
// columns.  A CTA owns a 64 x 64 tile; a thread 4 x 4 entries of it.
__global__ void __launch_bounds__(256) k_gj_block(int n, int kb, const float* __restrict__ M, float* __restrict__ N,
                                                  unsigned* flag) {
    __shared__ float P[GB][GB + 1];
    __shared__ float C[GT][GB + 1];     // M[i, kb]
    __shared__ float Rw[GB][GT + 1];    // M[kb, j], then t
    __shared__ __align__(16) float buf[2][GB];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int i0 = blockIdx.y * GT, j0 = blockIdx.x * GT;
    float o[4][4];
#pragma unroll
    for (int q = 0; q < 4; q++)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const int i = i0 + ty + 16 * q, j = j0 + tx + 16 * b;
            const bool own = j >= kb && j < kb + GB;
            o[q][b] = i < n && j < n && !own ? M[(long long)i * n + j] : 0.0f;
        }
    if (tid < 32) {
        float a[GB];
#pragma unroll
        for (int i = 0; i < GB; i++)
            a[i] = kb + i < n && kb + tid < n ? M[(long long)(kb + i) * n + kb + tid] : (i == tid ? 1.0f : 0.0f);
        const bool ok = warp_invert(a, buf, tid);
        if (!ok && tid == 0) *flag = 1u;
#pragma unroll
        for (int i = 0; i < GB; i++) P[i][tid] = a[i];
    } else {
        for (int q = tid - 32; q < GB * GT; q += 224) {
            const int r = q / GT, j = j0 + q % GT;
            Rw[r][q % GT] = kb + r < n && j < n ? M[(long long)(kb + r) * n + j] : 0.0f;
            const int i = i0 + q / GB, cc = kb + q % GB;
            C[q / GB][q % GB] = i < n && cc < n ? M[(long long)i * n + cc] : 0.0f;
        }
    }
    __syncthreads();
    // t: rows ty + 16 q (q < 2), columns tx + 16 b (b < 4)
    float t[2][4] = {};
    for (int m = 0; m < GB; m++) {
        const float p0 = P[ty][m], p1 = P[ty + 16][m];
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const float v = Rw[m][tx + 16 * b];
            t[0][b] = fmaf(p0, v, t[0][b]);
            t[1][b] = fmaf(p1, v, t[1][b]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 4; b++) {
        const int jl = j0 + tx + 16 * b - kb;
        const bool own = jl >= 0 && jl < GB;
        Rw[ty][tx + 16 * b] = own ? P[ty][jl] : t[0][b];
        Rw[ty + 16][tx + 16 * b] = own ? P[ty + 16][jl] : t[1][b];
    }
    __syncthreads();
    for (int m = 0; m < GB; m++) {
        float v[4];
#pragma unroll
        for (int b = 0; b < 4; b++) v[b] = Rw[m][tx + 16 * b];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float cq = C[ty + 16 * q][m];
#pragma unroll
            for (int b = 0; b < 4; b++) o[q][b] = fmaf(-cq, v[b], o[q][b]);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; q++)
#pragma unroll
        for (int b = 0; b < 4; b++) {
            const int i = i0 + ty + 16 * q, j = j0 + tx + 16 * b;
            if (i < n && j < n) {
                const int il = i - kb;
                N[(long long)i * n + j] = il >= 0 && il < GB ? Rw[il][tx + 16 * b] : o[q][b];
            }
        }
}

// ---- refinement of the FP32 inverse to FP64

// (A x)_c for CB columns x[c * CB + b], and the row's diagonal.
template <class T, int CB>
__device__ __forceinline__ void apply_row(const Dims& d, const Op<T>& A, int c, const double* x, double (&y)[CB], double& dg) {
    int i, j, k;
    cell_ijk(c, d, i, j, k);
    const int sy = d.nx, sz = d.nx * d.ny;
    const double m = (double)A.m[c];
    dg = m;
    double xc[CB];
#pragma unroll
    for (int b = 0; b < CB; b++) {
        xc[b] = x[c * CB + b];
        y[b] = m * xc[b];
    }
    auto add = [&](T wt, int nb) {
        const double w = (double)wt;
        dg += w;
#pragma unroll
        for (int b = 0; b < CB; b++) y[b] += w * (xc[b] - x[nb * CB + b]);
    };
    if (i > 0) add(A.wx[c], c - 1); else if (d.px) add(A.wx[c], c + d.nx - 1);
    if (i < d.nx - 1) add(A.wx[c + 1], c + 1); else if (d.px) add(A.wx[c - (d.nx - 1)], c - (d.nx - 1));
    if (j > 0) add(A.wy[c], c - sy); else if (d.py) add(A.wy[c], c + (d.ny - 1) * sy);
    if (j < d.ny - 1) add(A.wy[c + sy], c + sy); else if (d.py) add(A.wy[c - (d.ny - 1) * sy], c - (d.ny - 1) * sy);
    if (k > 0) add(A.wz[c], c - sz); else if (d.pz) add(A.wz[c], c + (d.nz - 1) * sz);
    if (k < d.nz - 1) add(A.wz[c + sz], c + sz); else if (d.pz) add(A.wz[c - (d.nz - 1) * sz], c - (d.nz - 1) * sz);
}

// Columns [CB b, CB b + CB) of the inverse: x from X32, then x += X32^T
// (e - A x) until the largest residual entry is at the rounding level of the
// products it is formed from (2 diag |x| bounds every w_f (x - x_nbr) of a
// neighbouring row).  Columns that stop improving before that, or need more
// than REFINE_MAX corrections, raise the flag.  Bound by the L2 reads of X32
// (all of it per CTA and correction) and the FP64 residual, so the columns are
// spread evenly over the SMs, with a thread per row up to 768: 162 us at 693
// cells and 13 at 64, where four columns per CTA of 256 threads took 276 us at
// 693.
constexpr int REFINE_MAX = 8;
constexpr int REFINE_THREADS = 768;
// entries of a row of r: room for vector loads
constexpr int refine_row(int cb) { return cb == 3 ? 4 : (cb > 4 ? 8 : cb); }
template <class T, int CB>
__global__ void __launch_bounds__(REFINE_THREADS) k_coarse_refine(Dims d, Op<T> A, const float* __restrict__ X32,
                                                                  double* __restrict__ X, unsigned* flag) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int RB = refine_row(CB);
    const int n = (int)d.n, nt = blockDim.x;
    double* x = reinterpret_cast<double*>(smem_raw);     // [n][CB]
    float* r = reinterpret_cast<float*>(x + (n * CB + 1) / 2 * 2);     // [n][RB]
    __shared__ double wscale[REFINE_THREADS / 32];
    __shared__ float wmax[REFINE_THREADS / 32];
    const int c0 = blockIdx.x * CB;
    for (int q = threadIdx.x; q < n * CB; q += nt) {
        const int c = c0 + q % CB;
        x[q] = c < n ? (double)X32[(long long)(q / CB) * n + c] : 0.0;
    }
    float prev = 1e30f;
    bool good = false;
    for (int it = 0;; it++) {
        __syncthreads();
        float mx = 0.0f;
        double sc = 1.0;
        for (int c = threadIdx.x; c < n; c += nt) {
            double y[CB], dg;
            apply_row<T, CB>(d, A, c, x, y, dg);
#pragma unroll
            for (int b = 0; b < CB; b++) {
                const double e = c0 + b < n ? (c == c0 + b ? 1.0 : 0.0) - y[b] : 0.0;
                const float e32 = (float)e;
                r[c * RB + b] = e32;
                mx = fmaxf(mx, isfinite(e32) ? fabsf(e32) : 1e30f);
                sc = fmax(sc, 2.0 * dg * fabs(x[c * CB + b]));
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
        sc = warp_max(sc);
        if ((threadIdx.x & 31) == 0) {
            wmax[threadIdx.x >> 5] = mx;
            wscale[threadIdx.x >> 5] = sc;
        }
        __syncthreads();
        mx = wmax[0];
        sc = wscale[0];
        for (int q = 1; q < nt / 32; q++) {
            mx = fmaxf(mx, wmax[q]);
            sc = fmax(sc, wscale[q]);
        }
        good = (double)mx <= 4.0 * 2.220446049250313e-16 * sc;
        if (good || it >= REFINE_MAX || mx > 0.25f * prev) break;
        prev = mx;
        for (int i = threadIdx.x; i < n; i += nt) {
            float acc[CB];
#pragma unroll
            for (int b = 0; b < CB; b++) acc[b] = 0.0f;
#pragma unroll 16
            for (int q = 0; q < n; q++) {
                const float w = X32[(long long)q * n + i];
                float rr[RB];
                if constexpr (RB >= 4) {
#pragma unroll
                    for (int v = 0; v < (CB + 3) / 4; v++)
                        *reinterpret_cast<float4*>(rr + 4 * v) = *reinterpret_cast<const float4*>(r + q * RB + 4 * v);
                } else {
#pragma unroll
                    for (int b = 0; b < CB; b++) rr[b] = r[q * RB + b];
                }
#pragma unroll
                for (int b = 0; b < CB; b++) acc[b] = fmaf(w, rr[b], acc[b]);
            }
#pragma unroll
            for (int b = 0; b < CB; b++) x[i * CB + b] += (double)acc[b];
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < n * CB; q += nt) {
        const int c = c0 + q % CB;
        if (c < n) put_inv<T>(X, (long long)(q / CB) * n + c, x[q]);
    }
    if (!good && threadIdx.x == 0) *flag = 1u;
}

// ---- FP64 fallback beyond GJ64_MAX cells

// One CTA: dense matrix M, in-place Cholesky (lower triangle becomes L), then
// the explicit inverse Ainv = L^-T L^-1, one column per thread.  A
// non-positive pivot sets sc[S_BAD] = 2.  Returns unless the flag is raised.
template <class T>
__global__ void k_chol_inverse(Dims d, Op<T> A, double* M, double* Ainv, double* sc, const unsigned* only_if) {
    if (*only_if == 0u) return;
    const int n = (int)d.n;
    __shared__ int fail;
    if (threadIdx.x == 0) fail = 0;
    for (long long q = threadIdx.x; q < (long long)n * n; q += blockDim.x) M[q] = 0.0;
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += blockDim.x) dense_row(d, A, c, M + (long long)c * n);
    __syncthreads();
    for (int j = 0; j < n; j++) {
        if (threadIdx.x == 0) {
            const double piv = M[(long long)j * n + j];
            if (!(piv > 0.0)) { fail = 1; M[(long long)j * n + j] = 1.0; }
            else M[(long long)j * n + j] = sqrt(piv);
        }
        __syncthreads();
        const double ljj = M[(long long)j * n + j];
        for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) M[(long long)i * n + j] /= ljj;
        __syncthreads();
        // trailing update of the lower triangle: M[i][k] -= L[i][j] L[k][j], j < k <= i
        for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) {
            const double lij = M[(long long)i * n + j];
            for (int k = j + 1; k <= i; k++) M[(long long)i * n + k] -= lij * M[(long long)k * n + j];
        }
        __syncthreads();
    }
    if (fail && threadIdx.x == 0) sc[S_BAD] = 2.0;
    // inverse, column t: L y = e_t, then L^T x = y, written in Ainv[:, t]
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        for (int i = 0; i < t; i++) Ainv[(long long)i * n + t] = 0.0;
        for (int i = t; i < n; i++) {
            double s = (i == t) ? 1.0 : 0.0;
            for (int k = t; k < i; k++) s -= M[(long long)i * n + k] * Ainv[(long long)k * n + t];
            Ainv[(long long)i * n + t] = s / M[(long long)i * n + i];
        }
        for (int i = n - 1; i >= 0; i--) {
            double s = Ainv[(long long)i * n + t];
            for (int k = i + 1; k < n; k++) s -= M[(long long)k * n + i] * Ainv[(long long)k * n + t];
            Ainv[(long long)i * n + t] = s / M[(long long)i * n + i];
        }
        if (sizeof(T) == 4)
            for (int i = 0; i < n; i++) put_inv<T>(Ainv, (long long)i * n + t, Ainv[(long long)i * n + t]);
    }
}

// ---- z = A^-1 r: a warp per row, the row's products summed by lanes
template <class T>
__global__ void __launch_bounds__(128) k_coarse_apply(int n, const double* __restrict__ Ainv, const T* __restrict__ r,
                                                      T* __restrict__ z) {
    const int lane = threadIdx.x & 31;
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += (int)(gridDim.x * blockDim.x) >> 5) {
        const T v = coarse_row<32, T>(Ainv, n, i, lane, [&](int q) { return r[q]; });
        if (lane == 0) z[i] = v;
    }
}

// A kernel's limit of dynamic shared memory belongs to the function and is
// shared by every host thread, so each instantiation only ever sets the most
// it can need (never this call's size: another thread's smaller grid would
// lower it between this call and its launch).
template <class T, class R, class O, int S, int PT>
void gj_go(const Dims& d, Op<T> A, O* X, double* sc, unsigned* flag, const unsigned* only_if, cudaStream_t s) {
    constexpr size_t most = (size_t)S * PT * S * PT * sizeof(R);
    const size_t bytes = (size_t)d.n * (size_t)d.n * sizeof(R);
    auto kern = k_gj_inverse<T, R, O, S, PT>;
    if (bytes > 40 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    kern<<<1, S * S, bytes, s>>>(d, A, X, sc, flag, only_if);
}

// FP32 elimination by one CTA; 256 threads up to 64 cells (a barrier over 8
// warps instead of 32)
template <class T, class O>
void gj_one(const Dims& d, Op<T> A, O* X, double* sc, unsigned* flag, cudaStream_t s) {
    if (d.n <= 32) gj_go<T, float, O, 16, 2>(d, A, X, sc, flag, nullptr, s);
    else if (d.n <= 64) gj_go<T, float, O, 16, 4>(d, A, X, sc, flag, nullptr, s);
    else if (d.n <= 128) gj_go<T, float, O, 32, 4>(d, A, X, sc, flag, nullptr, s);
    else gj_go<T, float, O, 32, 5>(d, A, X, sc, flag, nullptr, s);
}

// x and r of CB columns (launch_coarse_setup chooses CB so that they fit)
constexpr size_t REFINE_SMEM = 96 * 1024;
template <class T, int CB>
void refine_go(const Dims& d, Op<T> A, const float* X32, double* X, unsigned* flag, cudaStream_t s) {
    const size_t x = ((size_t)d.n * CB + 1) / 2 * 2 * sizeof(double);
    const size_t bytes = x + (size_t)d.n * refine_row(CB) * sizeof(float);
    auto kern = k_coarse_refine<T, CB>;
    if (bytes > 40 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)REFINE_SMEM);
    const int rows = (int)(d.n + 31) / 32 * 32;
    const int threads = rows < 256 ? 256 : (rows < REFINE_THREADS ? rows : REFINE_THREADS);
    kern<<<(unsigned)((d.n + CB - 1) / CB), threads, bytes, s>>>(d, A, X32, X, flag);
}

}  // namespace

// ---------------------------------------------------------------- launchers

template <class T>
void launch_coarse_setup(const Dims& d, Op<T> A, double* dense, double* ainv, double* sc, unsigned* flag, bool fp32,
                         cudaStream_t s) {
    const int n = (int)d.n;
    if (fp32 && n <= GJ_ONE_MAX) {
        gj_one<T, double>(d, A, ainv, sc, nullptr, s);
        return;
    }
    // the FP32 inverse in the dense buffer (room for two FP32 matrices)
    float* M = reinterpret_cast<float*>(dense);
    if (n <= GJ_ONE_MAX) {
        gj_one<T, float>(d, A, M, sc, flag, s);
    } else {
        float* other = M + (size_t)n * n;
        k_dense32<T><<<(n + 7) / 8, 256, 0, s>>>(d, A, M, flag);
        const int g = (n + GT - 1) / GT;
        for (int kb = 0; kb < n; kb += GB) {
            k_gj_block<<<dim3(g, g), 256, 0, s>>>(n, kb, M, other, flag);
            float* t = M;
            M = other;
            other = t;
        }
    }
    // columns per CTA: one wave of CTAs up to 5 columns each (693 cells: 162 us
    // with 5 columns, 276 with 4 in two uneven waves of 256 threads), beyond
    // that 4 while their x and r fit 96 KB (k_coarse_refine).  Six to eight
    // columns, one wave up to 1216 cells, were not measured.
    if (n <= 152) refine_go<T, 1>(d, A, M, ainv, flag, s);
    else if (n <= 2 * 152) refine_go<T, 2>(d, A, M, ainv, flag, s);
    else if (n <= 3 * 152) refine_go<T, 3>(d, A, M, ainv, flag, s);
    else if (n <= 4 * 152) refine_go<T, 4>(d, A, M, ainv, flag, s);
    else if (n <= 5 * 152) refine_go<T, 5>(d, A, M, ainv, flag, s);
    else if (n <= 2048) refine_go<T, 4>(d, A, M, ainv, flag, s);
    else refine_go<T, 2>(d, A, M, ainv, flag, s);
    if (n <= 64) gj_go<T, double, double, 32, 2>(d, A, ainv, sc, nullptr, flag, s);
    else if (n <= GJ64_MAX) gj_go<T, double, double, 32, 4>(d, A, ainv, sc, nullptr, flag, s);
    else k_chol_inverse<T><<<1, 1024, 0, s>>>(d, A, dense, ainv, sc, flag);
}
template <class T>
void launch_coarse_apply(int n, const double* ainv, const T* r, T* z, cudaStream_t s) {
    k_coarse_apply<T><<<(n + 3) / 4, 128, 0, s>>>(n, ainv, r, z);
}

#define INST(T)                                                                                              \
    template void launch_coarse_setup<T>(const Dims&, Op<T>, double*, double*, double*, unsigned*, bool,     \
                                         cudaStream_t);                                                     \
    template void launch_coarse_apply<T>(int, const double*, const T*, T*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace fld
