// k_mg.cu -- geometric multigrid V-cycle pieces for the 7-point FLD system
// (the preconditioner of Table 1): coarse operators, red/black Gauss-Seidel
// and weighted Jacobi smoothing, residual, full-weighting restriction and
// trilinear prolongation (the dense coarsest-grid solve: k_coarse.cu).
//
// Cell-centred full coarsening; operators by rediscretisation (coarse face
// weight = sum of the 4 fine face weights across the coarse face / 16,
// coarse mass term = mean of the 8 children); prolongation trilinear with
// 1-D weights 3/4 (nearer coarse cell) and 1/4 (farther one), ghost cells
// equal to the boundary cell on zero-gradient axes and wrapped on periodic
// ones; restriction is the transpose of prolongation divided by 8.
#include "kernels.h"

namespace fld {

// Sum over the faces of cell c of w_f * u_nbr, and of w_f.
template <class T>
__device__ __forceinline__ void nbr_sums(const Dims& d, const Op<T>& A, long long c, int i, int j,
                                         int k, const T* __restrict__ u, T& swu, T& sw) {
    const long long sy = d.nx, sz = (long long)d.nx * d.ny;
    T a = T(0), s = T(0);
    {
        const T wl = A.wx[c];
        if (i > 0) { a += wl * u[c - 1]; s += wl; }
        else if (d.px) { a += wl * u[c + d.nx - 1]; s += wl; }
        if (i < d.nx - 1) { const T wu = A.wx[c + 1]; a += wu * u[c + 1]; s += wu; }
        else if (d.px) { const long long up = c - (d.nx - 1); const T wu = A.wx[up]; a += wu * u[up]; s += wu; }
    }
    {
        const T wl = A.wy[c];
        if (j > 0) { a += wl * u[c - sy]; s += wl; }
        else if (d.py) { a += wl * u[c + (long long)(d.ny - 1) * sy]; s += wl; }
        if (j < d.ny - 1) { const T wu = A.wy[c + sy]; a += wu * u[c + sy]; s += wu; }
        else if (d.py) { const long long up = c - (long long)(d.ny - 1) * sy; const T wu = A.wy[up]; a += wu * u[up]; s += wu; }
    }
    {
        const T wl = A.wz[c];
        if (k > 0) { a += wl * u[c - sz]; s += wl; }
        else if (d.pz) { a += wl * u[c + (long long)(d.nz - 1) * sz]; s += wl; }
        if (k < d.nz - 1) { const T wu = A.wz[c + sz]; a += wu * u[c + sz]; s += wu; }
        else if (d.pz) { const long long up = c - (long long)(d.nz - 1) * sz; const T wu = A.wz[up]; a += wu * u[up]; s += wu; }
    }
    swu = a;
    sw = s;
}

// Sum over the faces of cell c of w_f * u_nbr * v_nbr (smoothing from a
// zero guess needs the red neighbours' values r * invd on the fly).
template <class T>
__device__ __forceinline__ T nbr_sum_prod(const Dims& d, const Op<T>& A, long long c, int i, int j,
                                          int k, const T* __restrict__ u, const T* __restrict__ v) {
    const long long sy = d.nx, sz = (long long)d.nx * d.ny;
    T a = T(0);
    if (i > 0) a += A.wx[c] * u[c - 1] * v[c - 1];
    else if (d.px) a += A.wx[c] * u[c + d.nx - 1] * v[c + d.nx - 1];
    if (i < d.nx - 1) a += A.wx[c + 1] * u[c + 1] * v[c + 1];
    else if (d.px) { const long long up = c - (d.nx - 1); a += A.wx[up] * u[up] * v[up]; }
    if (j > 0) a += A.wy[c] * u[c - sy] * v[c - sy];
    else if (d.py) { const long long lo = c + (long long)(d.ny - 1) * sy; a += A.wy[c] * u[lo] * v[lo]; }
    if (j < d.ny - 1) a += A.wy[c + sy] * u[c + sy] * v[c + sy];
    else if (d.py) { const long long up = c - (long long)(d.ny - 1) * sy; a += A.wy[up] * u[up] * v[up]; }
    if (k > 0) a += A.wz[c] * u[c - sz] * v[c - sz];
    else if (d.pz) { const long long lo = c + (long long)(d.nz - 1) * sz; a += A.wz[c] * u[lo] * v[lo]; }
    if (k < d.nz - 1) a += A.wz[c + sz] * u[c + sz] * v[c + sz];
    else if (d.pz) { const long long up = c - (long long)(d.nz - 1) * sz; a += A.wz[up] * u[up] * v[up]; }
    return a;
}


// ------------------------------------------------------------ operators

// Rediscretised coarse operator in precision T (FP64 for the FP64 cycle;
// FP32 from the FP32 operator for the mixed solver's cycle, which alone
// reads the coarse levels there).
//
// BND: also the coarse Dirichlet face weights, the sum of the 4 fine weights
// across each coarse face / 16 as for interior faces.  The mean of the 8
// children's m holds their boundary weights / 8 = 2 w_c; the rediscretised
// mass term has w_c, so w_c is taken back off, side by side in order.  (One
// launch per side and level took 97 us of a 1.5 ms step at 128 x 64 x 64.)
template <class T, bool BND>
__global__ void k_coarsen(Dims f, Dims cd, Op<T> F, Op<T> C, Bnd FB, Bnd CB) {
    COL_BEGIN(cd)
        const int I = i, J = j, K = k;
        const long long fx = f.nx, fxy = (long long)f.nx * f.ny;
        const long long base = 2LL * I + fx * 2LL * J + fxy * 2LL * K;
        T ms = 0;
#pragma unroll
        for (int dk = 0; dk < 2; dk++)
#pragma unroll
            for (int dj = 0; dj < 2; dj++)
#pragma unroll
                for (int di = 0; di < 2; di++) ms += F.m[base + di + fx * dj + fxy * dk];
        T sx = 0, sy = 0, sz = 0;
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int b = 0; b < 2; b++) {
                sx += F.wx[base + fx * a + fxy * b];
                sy += F.wy[base + a + fxy * b];
                sz += F.wz[base + a + fx * b];
            }
        T mc = ms * (T)0.125;
        if (BND) {
            const int ijk[3] = {i, j, k}, nn[3] = {cd.nx, cd.ny, cd.nz};
#pragma unroll
            for (int sd = 0; sd < 6; sd++) {
                const int a = sd >> 1;
                if (!((CB.mask >> sd) & 1) || ijk[a] != ((sd & 1) ? nn[a] - 1 : 0)) continue;
                const long long u = a == 0 ? j : i, v = a == 2 ? j : k;
                const long long nuc = a == 0 ? cd.ny : cd.nx, nuf = 2 * nuc;
                const long long f00 = bnd_offset(f, sd) + 2 * u + nuf * 2 * v;
                const double wc =
                    ((FB.w[f00] + FB.w[f00 + 1]) + (FB.w[f00 + nuf] + FB.w[f00 + nuf + 1])) * 0.0625;
                CB.w[bnd_offset(cd, sd) + u + nuc * v] = wc;
                mc = (T)(mc - wc);
            }
        }
        C.m[c] = mc;
        C.wx[c] = sx * (T)0.0625;
        C.wy[c] = sy * (T)0.0625;
        C.wz[c] = sz * (T)0.0625;
    }
}

// Inverse diagonal of A in precision T, the diagonal summed in the
// precision S of the operator src it is formed from.
template <class T, class S>
__global__ void k_invd(Dims d, Op<T> A, Op<S> src) {
    COL_BEGIN(d)
        S swu, sw;
        // u unused: pass m as a harmless array for the weight sum only
        nbr_sums<S>(d, src, c, i, j, k, src.m, swu, sw);
        const S diag = src.m[c] + sw;
        A.invd[c] = (T)((S)1 / diag);
    }
}

// ------------------------------------------------------------- smoothers

// First red/black Gauss-Seidel sweep from z = 0: red cells get r / diag,
// black cells (r + sum_f w_f z_red_nbr) / diag with the red values formed
// on the fly.
template <class T>
__global__ void k_smooth_zero(Dims d, Op<T> A, const T* __restrict__ r, T* __restrict__ z) {
    COL_BEGIN(d)
        if (((i + j + k) & 1) == 0) {
            z[c] = r[c] * A.invd[c];
        } else {
            z[c] = A.invd[c] * (r[c] + nbr_sum_prod<T>(d, A, c, i, j, k, r, A.invd));
        }
    }
}

// One colour of a red/black Gauss-Seidel sweep; every dimension is even on
// a smoothed level, so cell (2s + ((j + k + colour) & 1), j, k) enumerates
// the colour.
template <class T>
__global__ void k_rb_colour(Dims d, Op<T> A, const T* __restrict__ r, T* z, int colour) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int kch = (d.nz + (int)gridDim.z - 1) / (int)gridDim.z;
    const int k0 = (int)blockIdx.z * kch, k1 = min(d.nz, k0 + kch);
    if (s >= (d.nx >> 1) || j >= d.ny) return;
    const long long nxy = (long long)d.nx * d.ny;
    for (int k = k0; k < k1; k++) {
        const int i = 2 * s + ((j + k + colour) & 1);
        const long long c = (long long)k * nxy + (long long)j * d.nx + i;
        T swu, sw;
        nbr_sums<T>(d, A, c, i, j, k, z, swu, sw);
        z[c] = A.invd[c] * (r[c] + swu);
    }
}

// Weighted Jacobi: out = z + omega (r - A z) / diag, or omega r / diag from
// a zero guess.
template <class T>
__global__ void k_jacobi(Dims d, Op<T> A, const T* __restrict__ r, const T* __restrict__ z,
                         T* __restrict__ out, T omega, int zero_guess) {
    COL_BEGIN(d)
        if (zero_guess) {
            out[c] = omega * A.invd[c] * r[c];
        } else {
            T swu, sw;
            nbr_sums<T>(d, A, c, i, j, k, z, swu, sw);
            const T Az = A.m[c] * z[c] + sw * z[c] - swu;
            out[c] = z[c] + omega * A.invd[c] * (r[c] - Az);
        }
    }
}

template <class T>
__global__ void k_residual(Dims d, Op<T> A, const T* __restrict__ r, const T* __restrict__ z,
                           T* __restrict__ res) {
    COL_BEGIN(d)
        T swu, sw;
        nbr_sums<T>(d, A, c, i, j, k, z, swu, sw);
        res[c] = r[c] - (A.m[c] * z[c] + sw * z[c] - swu);
    }
}

// ------------------------------------------------------------- transfers

// Fine index of tap t (0..3 = offsets -1, 0, +1, +2 from 2I) along an axis,
// with the ghost rule; weights 1/4, 3/4, 3/4, 1/4.
__device__ __forceinline__ int fine_tap(int I, int t, int nf, int periodic) {
    int f = 2 * I - 1 + t;
    if (f < 0) f = periodic ? f + nf : 0;
    if (f >= nf) f = periodic ? f - nf : nf - 1;
    return f;
}

template <class T>
__global__ void k_restrict(Dims f, Dims cd, const T* __restrict__ rf, T* __restrict__ rc) {
    const T wt[4] = {T(0.25), T(0.75), T(0.75), T(0.25)};
    COL_BEGIN(cd)
        const int I = i, J = j, K = k;
        int fi[4], fj[4], fk[4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            fi[t] = fine_tap(I, t, f.nx, f.px);
            fj[t] = fine_tap(J, t, f.ny, f.py);
            fk[t] = fine_tap(K, t, f.nz, f.pz);
        }
        T acc = T(0);
#pragma unroll
        for (int tk = 0; tk < 4; tk++) {
            T acc_j = T(0);
#pragma unroll
            for (int tj = 0; tj < 4; tj++) {
                const long long row = (long long)f.nx * (fj[tj] + (long long)f.ny * fk[tk]);
                T acc_i = T(0);
#pragma unroll
                for (int ti = 0; ti < 4; ti++) acc_i += wt[ti] * rf[row + fi[ti]];
                acc_j += wt[tj] * acc_i;
            }
            acc += wt[tk] * acc_j;
        }
        rc[c] = acc * T(0.125);
    }
}

// Coarse neighbours of fine index i: nearer (weight 3/4) and farther (1/4).
__device__ __forceinline__ void coarse_pair(int i, int nc, int periodic, int& I0, int& I1) {
    I0 = i >> 1;
    int J = (i & 1) ? I0 + 1 : I0 - 1;
    if (J < 0) J = periodic ? nc - 1 : I0;
    if (J >= nc) J = periodic ? 0 : I0;
    I1 = J;
}

template <class T>
__global__ void k_prolong_add(Dims f, Dims cd, const T* __restrict__ ec, T* __restrict__ zf) {
    COL_BEGIN(f)
        int Ix[2], Iy[2], Iz[2];
        coarse_pair(i, cd.nx, cd.px, Ix[0], Ix[1]);
        coarse_pair(j, cd.ny, cd.py, Iy[0], Iy[1]);
        coarse_pair(k, cd.nz, cd.pz, Iz[0], Iz[1]);
        const T w[2] = {T(0.75), T(0.25)};
        T acc = T(0);
#pragma unroll
        for (int b = 0; b < 2; b++) {
            T acc_j = T(0);
#pragma unroll
            for (int a = 0; a < 2; a++) {
                const long long row = (long long)cd.nx * (Iy[a] + (long long)cd.ny * Iz[b]);
                acc_j += w[a] * (w[0] * ec[row + Ix[0]] + w[1] * ec[row + Ix[1]]);
            }
            acc += w[b] * acc_j;
        }
        zf[c] += acc;
    }
}

// ---------------------------------------------------------------- launchers

static const int TPB = 256;

template <class T>
void launch_coarsen(const Dims& f, const Dims& c, Op<T> F, Op<T> C, Bnd FB, Bnd CB, cudaStream_t s) {
    ColShape sh = col_shape(c);
    if (CB.mask) k_coarsen<T, true><<<sh.grid, sh.block, 0, s>>>(f, c, F, C, FB, CB);
    else k_coarsen<T, false><<<sh.grid, sh.block, 0, s>>>(f, c, F, C, FB, CB);
}
template <class T>
void launch_invd(const Dims& d, Op<T> A, const Op<T>& src, cudaStream_t s) {
    ColShape sh = col_shape(d);
    k_invd<T, T><<<sh.grid, sh.block, 0, s>>>(d, A, src);
}
template <class T>
void launch_smooth_zero(const Dims& d, Op<T> A, const T* r, T* z, cudaStream_t s) {
    ColShape sh = col_shape(d);
    k_smooth_zero<T><<<sh.grid, sh.block, 0, s>>>(d, A, r, z);
}
template <class T>
void launch_rb_colour(const Dims& d, Op<T> A, const T* r, T* z, int colour, cudaStream_t s) {
    Dims h = d;
    h.nx = d.nx / 2;
    ColShape sh = col_shape(h);
    k_rb_colour<T><<<sh.grid, sh.block, 0, s>>>(d, A, r, z, colour);
}
template <class T>
void launch_jacobi(const Dims& d, Op<T> A, const T* r, const T* z, T* out, double omega,
                   bool zero_guess, cudaStream_t s) {
    ColShape sh = col_shape(d);
    k_jacobi<T><<<sh.grid, sh.block, 0, s>>>(d, A, r, z, out, (T)omega, zero_guess ? 1 : 0);
}
template <class T>
void launch_residual(const Dims& d, Op<T> A, const T* r, const T* z, T* res, cudaStream_t s) {
    ColShape sh = col_shape(d);
    k_residual<T><<<sh.grid, sh.block, 0, s>>>(d, A, r, z, res);
}
template <class T>
void launch_restrict(const Dims& f, const Dims& c, const T* rf, T* rc, cudaStream_t s) {
    ColShape sh = col_shape(c);
    k_restrict<T><<<sh.grid, sh.block, 0, s>>>(f, c, rf, rc);
}
template <class T>
void launch_prolong_add(const Dims& f, const Dims& c, const T* ec, T* zf, cudaStream_t s) {
    ColShape sh = col_shape(f);
    k_prolong_add<T><<<sh.grid, sh.block, 0, s>>>(f, c, ec, zf);
}
#define INST(T)                                                                                    \
    template void launch_invd<T>(const Dims&, Op<T>, const Op<T>&, cudaStream_t);                   \
    template void launch_coarsen<T>(const Dims&, const Dims&, Op<T>, Op<T>, Bnd, Bnd, cudaStream_t); \
    template void launch_smooth_zero<T>(const Dims&, Op<T>, const T*, T*, cudaStream_t);            \
    template void launch_rb_colour<T>(const Dims&, Op<T>, const T*, T*, int, cudaStream_t);         \
    template void launch_jacobi<T>(const Dims&, Op<T>, const T*, const T*, T*, double, bool,        \
                                   cudaStream_t);                                                  \
    template void launch_residual<T>(const Dims&, Op<T>, const T*, const T*, T*, cudaStream_t);     \
    template void launch_restrict<T>(const Dims&, const Dims&, const T*, T*, cudaStream_t);         \
    template void launch_prolong_add<T>(const Dims&, const Dims&, const T*, T*, cudaStream_t);
INST(float)
INST(double)

}  // namespace fld
