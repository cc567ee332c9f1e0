// k_tail.cu -- the coarse tail of the multigrid V-cycle (Table 1's
// preconditioner) as one persistent kernel: every level at or below a size
// threshold, from the first such level down to the dense coarsest grid and
// back up, runs in a single launch of one thread-block cluster.
//
// Below ~32^3 cells a level's sweeps are latency-bound: each launch costs a
// few microseconds whatever its size, and a V-cycle has about six of them per
// level.  Here the phases of those levels (pre-smoothing, residual,
// restriction, coarsest solve, prolongation, post-smoothing) are separated by
// barriers inside the kernel.  The cluster barrier is the hardware one (all
// CTAs of a cluster are co-scheduled), so no software spin is involved, and
// values that cross CTAs go through global memory and are read back with
// L1-bypassing loads (.cg).  A level runs in one of three ways (plan_tail):
//  - solo: up to 4096 cells, CTA 0 alone with everything in shared memory;
//  - slab: the level above, in halo slabs of the longest axis, without
//    exchange between the CTAs within a leg of the cycle;
//  - phase by phase over the cluster, a cluster barrier after each.
//
// The arithmetic of every phase is that of the level kernels of k_mg.cu and
// k_fine4.cu (red/black Gauss-Seidel from a zero guess, colour sweeps, the
// residual after a zero-guess sweep or r - A z, full-weighting restriction,
// trilinear prolongation, dense inverse on the coarsest grid), so the tail
// gives the V-cycle those kernels give, up to rounding.
//
// The same phases also serve k_psolve, which runs whole inner MG-PCG solves
// of small grids (every level, then the CG vector operations) for a work
// list of requests in one launch (see the section below).
//
// Registers: 1024 threads leave 64 each.  k_vtail<float> spills 8 words,
// k_vtail<double> none; k_psolve, which holds the cluster solve, both
// one-CTA solves and the whole tail, spills 131.
#include <cooperative_groups.h>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace fld {

namespace {

constexpr int TAIL_THREADS = 1024;

// Vectors written inside the kernel by other CTAs live in global memory and
// are read through L2 (.cg).
template <class T>
__device__ __forceinline__ T ldw(const T* p, int i) {
    return __ldcg(p + i);
}

// Cell offsets within a level are 32-bit: tail and persistent-solve levels
// hold fewer than 2^31 cells (the size limits of fld_params bound them).

// sum_f w_f u_nbr and sum_f w_f of cell c
template <class T>
__device__ __forceinline__ void tail_nbr_sums(const Dims& d, const Op<T>& A, int c, int i, int j, int k,
                                              const T* u, T& swu, T& sw) {
    const int sy = d.nx, sz = d.nx * d.ny;
    T a = T(0), s = T(0);
    {
        const T wl = A.wx[c];
        if (i > 0) { a += wl * ldw(u, c - 1); s += wl; }
        else if (d.px) { a += wl * ldw(u, c + d.nx - 1); s += wl; }
        if (i < d.nx - 1) { const T wu = A.wx[c + 1]; a += wu * ldw(u, c + 1); s += wu; }
        else if (d.px) { const int up = c - (d.nx - 1); const T wu = A.wx[up]; a += wu * ldw(u, up); s += wu; }
    }
    {
        const T wl = A.wy[c];
        if (j > 0) { a += wl * ldw(u, c - sy); s += wl; }
        else if (d.py) { a += wl * ldw(u, c + (d.ny - 1) * sy); s += wl; }
        if (j < d.ny - 1) { const T wu = A.wy[c + sy]; a += wu * ldw(u, c + sy); s += wu; }
        else if (d.py) { const int up = c - (d.ny - 1) * sy; const T wu = A.wy[up]; a += wu * ldw(u, up); s += wu; }
    }
    {
        const T wl = A.wz[c];
        if (k > 0) { a += wl * ldw(u, c - sz); s += wl; }
        else if (d.pz) { a += wl * ldw(u, c + (d.nz - 1) * sz); s += wl; }
        if (k < d.nz - 1) { const T wu = A.wz[c + sz]; a += wu * ldw(u, c + sz); s += wu; }
        else if (d.pz) { const int up = c - (d.nz - 1) * sz; const T wu = A.wz[up]; a += wu * ldw(u, up); s += wu; }
    }
    swu = a;
    sw = s;
}

// sum_f w_f u_nbr v_nbr (the red neighbours r * invd of a zero-guess sweep)
template <class T>
__device__ __forceinline__ T tail_nbr_sum_prod(const Dims& d, const Op<T>& A, int c, int i, int j, int k,
                                               const T* u, const T* v) {
    const int sy = d.nx, sz = d.nx * d.ny;
    T a = T(0);
    if (i > 0) a += A.wx[c] * ldw(u, c - 1) * v[c - 1];
    else if (d.px) a += A.wx[c] * ldw(u, c + d.nx - 1) * v[c + d.nx - 1];
    if (i < d.nx - 1) a += A.wx[c + 1] * ldw(u, c + 1) * v[c + 1];
    else if (d.px) { const int up = c - (d.nx - 1); a += A.wx[up] * ldw(u, up) * v[up]; }
    if (j > 0) a += A.wy[c] * ldw(u, c - sy) * v[c - sy];
    else if (d.py) { const int lo = c + (d.ny - 1) * sy; a += A.wy[c] * ldw(u, lo) * v[lo]; }
    if (j < d.ny - 1) a += A.wy[c + sy] * ldw(u, c + sy) * v[c + sy];
    else if (d.py) { const int up = c - (d.ny - 1) * sy; a += A.wy[up] * ldw(u, up) * v[up]; }
    if (k > 0) a += A.wz[c] * ldw(u, c - sz) * v[c - sz];
    else if (d.pz) { const int lo = c + (d.nz - 1) * sz; a += A.wz[c] * ldw(u, lo) * v[lo]; }
    if (k < d.nz - 1) a += A.wz[c + sz] * ldw(u, c + sz) * v[c + sz];
    else if (d.pz) { const int up = c - (d.nz - 1) * sz; a += A.wz[up] * ldw(u, up) * v[up]; }
    return a;
}

// Cell coordinates by 32-bit unsigned division.
__device__ __forceinline__ void tail_ijk(int c, const Dims& d, int& i, int& j, int& k) {
    const unsigned cu = (unsigned)c, nx = (unsigned)d.nx, nxy = (unsigned)d.nx * (unsigned)d.ny;
    const unsigned kk = cu / nxy;
    const unsigned rem = cu - kk * nxy;
    const unsigned jj = rem / nx;
    k = (int)kk;
    j = (int)jj;
    i = (int)(rem - jj * nx);
}

// A thread's strided walk c = c0, c0 + s, ... over a level's cells with the
// coordinates kept incrementally: the stride is split once into (di, dj, dk)
// in the level's mixed radix, so a step costs a few adds and compares
// instead of two divisions (i + di < 2 nx and j + dj + 1 < 2 ny, so one
// carry each suffices).
struct Walk {
    int c, s, n;
    int i, j, k, di, dj, dk, nx, ny;
    __device__ __forceinline__ Walk(const Dims& d, int c0, int stride)
        : c(c0), s(stride), n((int)d.n), nx(d.nx), ny(d.ny) {
        tail_ijk(c0 < n ? c0 : 0, d, i, j, k);
        const unsigned su = (unsigned)stride, nxu = (unsigned)d.nx, nyu = (unsigned)d.ny;
        const unsigned t = su / nxu;
        di = (int)(su - t * nxu);
        dk = (int)(t / nyu);
        dj = (int)(t - (unsigned)dk * nyu);
    }
    __device__ __forceinline__ bool more() const { return c < n; }
    __device__ __forceinline__ void next() {
        c += s;
        i += di;
        if (i >= nx) { i -= nx; j++; }
        j += dj;
        if (j >= ny) { j -= ny; k++; }
        k += dk;
    }
};

// The same walk over the cells of one colour, (i + j + k) % 2 == col, of a
// level with an even x extent: half-index h over the n / 2 cells of that
// colour, x position 2 t + ((col + j + k) & 1), so no lane of a warp idles
// on a cell of the other colour.
struct WalkC {
    int h, s, n2;
    int t, j, k, dt, dj, dk, nx2, ny, nx, col;
    __device__ __forceinline__ WalkC(const Dims& d, int colour, int h0, int stride)
        : h(h0), s(stride), n2((int)(d.n >> 1)), nx2(d.nx >> 1), ny(d.ny), nx(d.nx), col(colour) {
        const unsigned hu = (unsigned)(h0 < n2 ? h0 : 0), n2x = (unsigned)nx2, nyu = (unsigned)d.ny;
        const unsigned r = hu / n2x;
        t = (int)(hu - r * n2x);
        k = (int)(r / nyu);
        j = (int)(r - (unsigned)k * nyu);
        const unsigned su = (unsigned)stride;
        const unsigned q = su / n2x;
        dt = (int)(su - q * n2x);
        dk = (int)(q / nyu);
        dj = (int)(q - (unsigned)dk * nyu);
    }
    __device__ __forceinline__ bool more() const { return h < n2; }
    __device__ __forceinline__ int i() const { return 2 * t + ((col + j + k) & 1); }
    __device__ __forceinline__ int c() const { return i() + nx * (j + ny * k); }
    __device__ __forceinline__ void next() {
        h += s;
        t += dt;
        if (t >= nx2) { t -= nx2; j++; }
        j += dj;
        if (j >= ny) { j -= ny; k++; }
        k += dk;
    }
};

// f(c, i, j, k) for every cell of colour col in this thread's share: the
// colour walk where nx is even, else the plain walk with the other colour
// skipped.  The cells are independent, so the order does not matter.
template <class F>
__device__ __forceinline__ void for_colour(const Dims& d, int col, int tid, int nth, F f) {
    if ((d.nx & 1) == 0) {
        for (WalkC w(d, col, tid, nth); w.more(); w.next()) f(w.c(), w.i(), w.j, w.k);
    } else {
        for (Walk w(d, tid, nth); w.more(); w.next())
            if (((w.i + w.j + w.k) & 1) == col) f(w.c, w.i, w.j, w.k);
    }
}

__device__ __forceinline__ int tail_fine_tap(int I, int t, int nf, int periodic) {
    int f = 2 * I - 1 + t;
    if (f < 0) f = periodic ? f + nf : 0;
    if (f >= nf) f = periodic ? f - nf : nf - 1;
    return f;
}

__device__ __forceinline__ void tail_coarse_pair(int i, int nc, int periodic, int& I0, int& I1) {
    I0 = i >> 1;
    int J = (i & 1) ? I0 + 1 : I0 - 1;
    if (J < 0) J = periodic ? nc - 1 : I0;
    if (J >= nc) J = periodic ? 0 : I0;
    I1 = J;
}

// The global vectors of one level as a cluster phase sees them.
template <class T>
struct Vec {
    T *r, *z, *t;
};

// Phase loops: the participating threads stride over the level's cells.
#define TAIL_LOOP(c, n) for (int c = tid; c < (int)(n); c += nth)

// Down-leg phases of level L into the coarse right-hand side rc:
// smoothing from zero (and further pre-sweeps), t = r - A z, rc = R t.
template <class T, class Sync>
__device__ void tail_down(const TailLevel<T>& L, Vec<T> v, const Dims& cd, T* rc, int pre, int tid, int nth,
                          Sync sync) {
    const Dims& d = L.d;
    const Op<T>& A = L.A;
    const T* r = v.r;
    T* z = v.z;
    if (pre >= 1) {
        // red cells r / diag, black cells from the red ones' r / diag (the
        // two colours independent, so in one phase)
        for_colour(d, 0, tid, nth, [&](int c, int, int, int) { z[c] = ldw(r, c) * A.invd[c]; });
        for_colour(d, 1, tid, nth, [&](int c, int i, int j, int k) {
            z[c] = A.invd[c] * (ldw(r, c) + tail_nbr_sum_prod<T>(d, A, c, i, j, k, r, A.invd));
        });
        sync();
        for (int it = 1; it < pre; it++)
            for (int colour = 0; colour < 2; colour++) {
                for_colour(d, colour, tid, nth, [&](int c, int i, int j, int k) {
                    T swu, sw;
                    tail_nbr_sums<T>(d, A, c, i, j, k, z, swu, sw);
                    z[c] = A.invd[c] * (ldw(r, c) + swu);
                });
                sync();
            }
    } else {
        TAIL_LOOP(c, d.n) z[c] = T(0);
        sync();
    }
    for (Walk w(d, tid, nth); w.more(); w.next()) {
        const int c = w.c;
        T swu, sw;
        tail_nbr_sums<T>(d, A, c, w.i, w.j, w.k, z, swu, sw);
        const T zc = ldw((const T*)z, c);
        v.t[c] = ldw(r, c) - (A.m[c] * zc + sw * zc - swu);
    }
    sync();
    const T wt[4] = {T(0.25), T(0.75), T(0.75), T(0.25)};
    for (Walk w(cd, tid, nth); w.more(); w.next()) {
        int fi[4], fj[4], fk[4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            fi[t] = tail_fine_tap(w.i, t, d.nx, d.px);
            fj[t] = tail_fine_tap(w.j, t, d.ny, d.py);
            fk[t] = tail_fine_tap(w.k, t, d.nz, d.pz);
        }
        T acc = T(0);
#pragma unroll
        for (int tk = 0; tk < 4; tk++) {
            T acc_j = T(0);
#pragma unroll
            for (int tj = 0; tj < 4; tj++) {
                const int row = d.nx * (fj[tj] + d.ny * fk[tk]);
                T acc_i = T(0);
#pragma unroll
                for (int ti = 0; ti < 4; ti++) acc_i += wt[ti] * ldw((const T*)v.t, row + fi[ti]);
                acc_j += wt[tj] * acc_i;
            }
            acc += wt[tk] * acc_j;
        }
        rc[w.c] = acc * T(0.125);
    }
    sync();
}

// Up-leg phases of level L: z += P zc, then the post-sweeps.
template <class T, class Sync>
__device__ void tail_up(const TailLevel<T>& L, Vec<T> v, const Dims& cd, const T* zc, int post, int first, int tid,
                        int nth, Sync sync) {
    const Dims& d = L.d;
    const Op<T>& A = L.A;
    T* z = v.z;
    const T w2[2] = {T(0.75), T(0.25)};
    for (Walk w(d, tid, nth); w.more(); w.next()) {
        const int c = w.c;
        int Ix[2], Iy[2], Iz[2];
        tail_coarse_pair(w.i, cd.nx, cd.px, Ix[0], Ix[1]);
        tail_coarse_pair(w.j, cd.ny, cd.py, Iy[0], Iy[1]);
        tail_coarse_pair(w.k, cd.nz, cd.pz, Iz[0], Iz[1]);
        T acc = T(0);
#pragma unroll
        for (int b = 0; b < 2; b++) {
            T acc_j = T(0);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int row = cd.nx * (Iy[q] + cd.ny * Iz[b]);
                acc_j += w2[q] * (w2[0] * ldw(zc, row + Ix[0]) + w2[1] * ldw(zc, row + Ix[1]));
            }
            acc += w2[b] * acc_j;
        }
        z[c] = ldw((const T*)z, c) + acc;
    }
    sync();
    // first: the colour the post-sweep starts with (1 black: symmetric cycle)
    for (int it = 0; it < post; it++)
        for (int q = 0; q < 2; q++) {
            const int colour = q == 0 ? first : 1 - first;
            for_colour(d, colour, tid, nth, [&](int c, int i, int j, int k) {
                T swu, sw;
                tail_nbr_sums<T>(d, A, c, i, j, k, z, swu, sw);
                z[c] = A.invd[c] * (ldw((const T*)v.r, c) + swu);
            });
            sync();
        }
}

// ---------------------------------------------------------------------------
// Small levels in one CTA ("solo"): every vector in shared memory, and for
// FP32 the coefficients too (copied asynchronously before they are needed), a
// block barrier between phases.  A thread owns pairs of cells (2h, 2h + 1)
// along x, one red and one black; a table per level holds what the phases need
// of a pair's position (face flags, parities, coarse cell), so no phase
// divides.  A phase takes about 1.8 us at 16^3 and 0.5 us at 8^3: one SM's
// instruction issue and fetch bound it (a 16^3 cycle is 84,600 warp
// instructions, issued in a third of the cycles; the largest stall is for the
// next instruction), not the barriers.
//
// z starts as r * invd at red cells (whoever produces r writes it), so the
// first red/black sweep from zero is one black phase; the residual after it is
// zero at black cells and sum_f w_f z_nbr at red ones; the restriction reads
// only the red residuals (two per fine row); and since a colour's sweep never
// reads that colour's old values, the correction is added only to the colour
// that the first post-sweep does not replace.

extern __shared__ __align__(16) unsigned char tail_smem[];

template <class U>
__device__ __forceinline__ U* sm(int off) {
    return reinterpret_cast<U*>(tail_smem + off);
}

// A pair's table entry: coarse cell, face flags of the pair, parities of j, k.
constexpr unsigned PI_XL = 1u << 16, PI_XU = 1u << 17, PI_YL = 1u << 18, PI_YU = 1u << 19, PI_ZL = 1u << 20,
                   PI_ZU = 1u << 21, PI_YO = 1u << 22, PI_ZO = 1u << 23;

// which cell of the pair has colour col
__device__ __forceinline__ int pair_odd(unsigned info, int col) {
    return (int)(((info >> 22) ^ (info >> 23)) & 1u) ^ col;
}

// coefficient q (0 invd, 1..3 wx, wy, wz, 4 m) of cell i
template <bool CS, class T>
__device__ __forceinline__ T coef(const TailLevel<T>& L, int q, int i) {
    if constexpr (CS) return sm<T>(L.o_c)[q * (int)L.d.n + i];
    else return __ldg((q == 0 ? L.A.invd : q == 1 ? L.A.wx : q == 2 ? L.A.wy : q == 3 ? L.A.wz : L.A.m) + i);
}

// sum_f w_f u_nbr of cell c (sw: also sum_f w_f).  A missing neighbour (zero
// gradient) reads the cell itself with weight 0.
template <bool CS, bool SW, class T>
__device__ __forceinline__ T solo_sum(const TailLevel<T>& L, const T* u, int c, unsigned info, int odd, T* sw) {
    const int nx = L.d.nx, nxy = L.d.nx * L.d.ny;
    T a = T(0), s = T(0);
    auto face = [&](int q, bool lo, bool up, int periodic, int stride, int wrap) {
        const int om = lo ? (periodic ? wrap : 0) : -stride;
        const T wl = coef<CS>(L, q, c);
        a += wl * u[c + om];
        const int op = up ? (periodic ? -wrap : 0) : stride;
        T wu = coef<CS>(L, q, c + op);
        if (up && !periodic) wu = T(0);
        a += wu * u[c + op];
        if (SW) s += wl + wu;
    };
    face(1, (info & PI_XL) && !odd, (info & PI_XU) && odd, L.d.px, 1, nx - 1);
    face(2, (info & PI_YL) != 0, (info & PI_YU) != 0, L.d.py, nx, nxy - nx);
    face(3, (info & PI_ZL) != 0, (info & PI_ZU) != 0, L.d.pz, nxy, (int)L.d.n - nxy);
    if (SW) *sw = s;
    return a;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(__cvta_generic_to_global(src)) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Starts the copies of the solo levels' coefficients (CS) and of the coarsest
// inverse, and fills the pair tables; cp_async_wait and a barrier complete it.
template <bool CS, class T>
__device__ void solo_prefetch(const TailArgs<T>& a, int tid, int nth) {
    for (int l = a.small_from; l < a.nlev - 1; l++) {
        const TailLevel<T>& L = a.L[l];
        const int n = (int)L.d.n;
        if (CS) {
            const T* src[5] = {L.A.invd, L.A.wx, L.A.wy, L.A.wz, L.A.m};
            const int nq = l == 0 && a.solve ? 5 : 4;
            const int per = 16 / (int)sizeof(T);    // n is a multiple of 8
#pragma unroll
            for (int q = 0; q < 5; q++)
                if (q < nq)
                    for (int i = per * tid; i < n; i += per * nth) cp_async16(sm<T>(L.o_c) + q * n + i, src[q] + i);
        }
        const Dims& cd = a.L[l + 1].d;
        const int nx2 = L.d.nx >> 1, ny = L.d.ny, nz = L.d.nz;
        unsigned* tab = sm<unsigned>(L.o_i);
        for (int h = tid; h < n >> 1; h += nth) {
            const unsigned r = (unsigned)h / (unsigned)nx2;
            const int t = h - (int)r * nx2;
            const int k = (int)(r / (unsigned)ny), j = (int)r - k * ny;
            tab[h] = (unsigned)(t + cd.nx * ((j >> 1) + cd.ny * (k >> 1))) | (t == 0 ? PI_XL : 0) |
                     (t == nx2 - 1 ? PI_XU : 0) | (j == 0 ? PI_YL : 0) | (j == ny - 1 ? PI_YU : 0) |
                     (k == 0 ? PI_ZL : 0) | (k == nz - 1 ? PI_ZU : 0) | ((j & 1) ? PI_YO : 0) | ((k & 1) ? PI_ZO : 0);
        }
    }
    if (a.o_ainv >= 0) {
        const int nc = (int)a.L[a.nlev - 1].d.n;
        const double* src = a.ainv;
        // nc^2 words of 8 bytes: pairs of them, the odd last one alone
        for (int i = 2 * tid; i + 1 < nc * nc; i += 2 * nth) cp_async16(sm<double>(a.o_ainv) + i, src + i);
        if (tid == 0 && (nc * nc) % 2) sm<double>(a.o_ainv)[nc * nc - 1] = src[nc * nc - 1];
    }
}

template <bool CS, class T>
__device__ __forceinline__ void solo_colour(const TailLevel<T>& L, int col, int tid, int nth) {
    T* z = sm<T>(L.o_z);
    const T* r = sm<T>(L.o_r);
    const unsigned* tab = sm<unsigned>(L.o_i);
    for (int h = tid; h < (int)(L.d.n >> 1); h += nth) {
        const unsigned info = tab[h];
        const int odd = pair_odd(info, col), c = 2 * h + odd;
        z[c] = coef<CS>(L, 0, c) * (r[c] + solo_sum<CS, false, T>(L, z, c, info, odd, nullptr));
    }
}

// Restriction of fine level F's residual to coarse cell (I, J, K), fine tap
// plane tk: red: the red residuals t (pairs), else the full array t.
template <class T>
__device__ __forceinline__ T restrict_plane(const Dims& d, const T* t, bool red, int I, int J, int K, int tk) {
    const T wt[4] = {T(0.25), T(0.75), T(0.75), T(0.25)};
    const int nx2 = d.nx >> 1;
    const int fz = tail_fine_tap(K, tk, d.nz, d.pz);
    T acc = T(0);
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const int fy = tail_fine_tap(J, q, d.ny, d.py);
        const int row = fy + d.ny * fz;
        T v;
        if (red) {
            // red cells of the row: even x (2I, 2I + 2) or odd x (2I - 1,
            // 2I + 1); a tap folded onto a red boundary cell adds to its weight
            const bool o = ((fy + fz) & 1) != 0;
            int s = o ? I - 1 : I + 1;
            const bool out = s < 0 || s >= nx2;
            if (out) s = s < 0 ? nx2 - 1 : 0;
            const T far = out && !d.px ? T(0) : t[row * nx2 + s];
            const bool folded = !d.px && (o ? I == nx2 - 1 : I == 0);
            v = (folded ? T(1) : T(0.75)) * t[row * nx2 + I] + T(0.25) * far;
        } else {
            v = T(0);
#pragma unroll
            for (int p = 0; p < 4; p++) v += wt[p] * t[row * d.nx + tail_fine_tap(I, p, d.nx, d.px)];
        }
        acc += wt[q] * v;
    }
    return acc;
}

// Down-leg of solo level l: pre-sweeps, residual, r (and r * invd into z) of
// level l + 1.
template <bool CS, class T>
__device__ void solo_down(const TailArgs<T>& a, int l, int tid, int nth) {
    const TailLevel<T>& L = a.L[l];
    const TailLevel<T>& C = a.L[l + 1];
    const int n = (int)L.d.n;
    T* z = sm<T>(L.o_z);
    const T* r = sm<T>(L.o_r);
    const unsigned* tab = sm<unsigned>(L.o_i);
    const bool red = a.pre >= 1;
    if (red) {
        solo_colour<CS, T>(L, 1, tid, nth);
        __syncthreads();
        for (int it = 1; it < a.pre; it++)
            for (int col = 0; col < 2; col++) {
                solo_colour<CS, T>(L, col, tid, nth);
                __syncthreads();
            }
        T* t = sm<T>(L.o_t);
        for (int h = tid; h < n >> 1; h += nth) {
            const unsigned info = tab[h];
            const int odd = pair_odd(info, 0), c = 2 * h + odd;
            T v = solo_sum<CS, false, T>(L, z, c, info, odd, nullptr);
            // further sweeps leave r - A z with the diagonal's z at red cells
            if (a.pre > 1) v = (r[c] + v) - z[c] / coef<CS>(L, 0, c);
            t[h] = v;
        }
    } else {
        for (int c = tid; c < n; c += nth) z[c] = T(0);
    }
    __syncthreads();
    const int nc = (int)C.d.n;
    const T* t = red ? sm<T>(L.o_t) : r;
    T* rc = sm<T>(C.o_r);
    T* zc = sm<T>(C.o_z);
    // four lanes per coarse cell, one fine plane each
    for (int it = tid; it < ((4 * nc + 31) & ~31); it += nth) {
        const int c = min(it >> 2, nc - 1), tk = it & 3;
        int I, J, K;
        tail_ijk(c, C.d, I, J, K);
        T v = restrict_plane<T>(L.d, t, red, I, J, K, tk);
        v *= tk == 0 || tk == 3 ? T(0.25) : T(0.75);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (tk == 0 && it < 4 * nc) {
            v *= T(0.125);
            rc[c] = v;
            if (l + 1 < a.nlev - 1) zc[c] = v * coef<CS>(C, 0, c);
        }
    }
    __syncthreads();
}

// Interpolated coarse correction at the cell of pair info (odd: which).
template <class T>
__device__ __forceinline__ T solo_interp(const Dims& cd, const T* zc, unsigned info, int odd) {
    const int nx = cd.nx, nxy = cd.nx * cd.ny;
    const int c = (int)(info & 0xffffu);
    auto off = [&](bool up, bool lo_end, bool up_end, int periodic, int stride, int wrap) {
        if (up) return up_end ? (periodic ? -wrap : 0) : stride;
        return lo_end ? (periodic ? wrap : 0) : -stride;
    };
    const int ox = off(odd != 0, (info & PI_XL) != 0, (info & PI_XU) != 0, cd.px, 1, nx - 1);
    const int oy = off((info & PI_YO) != 0, (info & PI_YL) != 0, (info & PI_YU) != 0, cd.py, nx, nxy - nx);
    const int oz = off((info & PI_ZO) != 0, (info & PI_ZL) != 0, (info & PI_ZU) != 0, cd.pz, nxy, (int)cd.n - nxy);
    auto row = [&](int b) { return T(0.75) * zc[b] + T(0.25) * zc[b + ox]; };
    auto plane = [&](int b) { return T(0.75) * row(b) + T(0.25) * row(b + oy); };
    return T(0.75) * plane(c) + T(0.25) * plane(c + oz);
}

// Up-leg of solo level l: the correction, then the post-sweeps.
template <bool CS, class T>
__device__ void solo_up(const TailArgs<T>& a, int l, int tid, int nth) {
    const TailLevel<T>& L = a.L[l];
    T* z = sm<T>(L.o_z);
    const T* zc = sm<T>(a.L[l + 1].o_z);
    const unsigned* tab = sm<unsigned>(L.o_i);
    const int first = a.paper_order ? 0 : 1;
    for (int h = tid; h < (int)(L.d.n >> 1); h += nth) {
        const unsigned info = tab[h];
        const int odd = pair_odd(info, 1 - first);
        z[2 * h + odd] += solo_interp<T>(a.L[l + 1].d, zc, info, odd);
        if (a.post == 0) z[2 * h + 1 - odd] += solo_interp<T>(a.L[l + 1].d, zc, info, 1 - odd);
    }
    __syncthreads();
    for (int it = 0; it < a.post; it++)
        for (int q = 0; q < 2; q++) {
            solo_colour<CS, T>(L, q == 0 ? first : 1 - first, tid, nth);
            __syncthreads();
        }
}

// z = A^-1 r on the coarsest grid by one CTA, in shared memory.  Lanes per
// row: 16 in FP32 (64 rows fill 1024 threads), 4 in FP64, where the shuffle
// sum's additions cost as much as the products (a warp's FP64 instruction
// takes 16 cycles of the SM's FP64 pipe).
template <class T>
__device__ void solo_coarsest(const TailArgs<T>& a, int tid, int nth) {
    const TailLevel<T>& L = a.L[a.nlev - 1];
    const int n = (int)L.d.n;
    const T* r = sm<T>(L.o_r);
    T* z = sm<T>(L.o_z);
    constexpr int G = sizeof(T) == 4 ? 16 : 4;
    auto rd = [&](int q) { return r[q]; };
    for (int it = tid; it < ((G * n + 31) & ~31); it += nth) {
        const int row = min(it / G, n - 1);
        const T v = a.o_ainv >= 0 ? coarse_row<G, T>(sm<double>(a.o_ainv), n, row, it % G, rd)
                                  : coarse_row<G, T>(a.ainv, n, row, it % G, rd);
        if (it % G == 0 && it < G * n) z[row] = v;
    }
    __syncthreads();
}

// The same by the whole cluster, r and z in global memory (a warp per row);
// ends with a cluster barrier.
template <class T>
__device__ void cluster_coarsest(const TailArgs<T>& a, cg::cluster_group& cl) {
    const TailLevel<T>& L = a.L[a.nlev - 1];
    const int n = (int)L.d.n;
    auto rd = [&](int q) { return __ldcg(L.r + q); };
    const int warp = ((int)cl.block_rank() * TAIL_THREADS + (int)threadIdx.x) >> 5;
    for (int row = warp; row < n; row += TAIL_THREADS / 32 * (int)cl.num_blocks()) {
        const T v = coarse_row<32, T>(a.ainv, n, row, threadIdx.x & 31, rd);
        if ((threadIdx.x & 31) == 0) L.z[row] = v;
    }
    cl.sync();
}

// ---------------------------------------------------------------------------
// A level of up to about 32^3 cells over the cluster ("slab"): CTA b owns q
// coarse planes of the longest axis (f) and the 2q fine planes they cover.  It
// keeps r and z of those and of three planes on either side in its shared
// memory and forms the halo's values itself, so the down-leg (black sweep,
// residual, restriction) and the up-leg (correction, black, red) need no
// exchange between CTAs: two cluster barriers per level instead of six, each
// of which cost 2 to 3 us with its round trips through L2.  The extra cells
// (at q = 1: 6, 4, 6, 4, 2 planes in the five phases against 2 each) are
// cheap beside that.  Coefficients are read through L1, several cells' loads
// issued together.
template <class T>
struct Slab {
    int U2, U, V, P2, P, nF, K0, K1;     // pairs per row, cells per row, rows, pairs and cells per plane, planes
    int su, sv, sf;                      // global strides
    int pu, pv, pf;
    const T *wu, *wv, *wf, *invd;
    int Cu, Cv, Cf;                      // coarse extents
    int cu, cv, cf;                      // coarse global strides
    int base;                            // virtual plane of slot 0
    int o_r, o_z, o_t, o_i;
};

template <class T>
__device__ __forceinline__ Slab<T> slab_of(const TailArgs<T>& a, cg::cluster_group& cl) {
    const TailLevel<T>& L = a.L[a.slab];
    const Dims& d = L.d;
    const Dims& c = a.L[a.slab + 1].d;
    Slab<T> s;
    // axes: f the slab axis, u and v the other two in order
    const bool fx = a.slab_axis == 0, fz = a.slab_axis == 2;
    s.U = fx ? d.ny : d.nx; s.V = fz ? d.ny : d.nz; s.nF = fx ? d.nx : (fz ? d.nz : d.ny);
    s.U2 = s.U >> 1; s.P2 = s.U2 * s.V; s.P = 2 * s.P2;
    s.su = fx ? d.nx : 1; s.sv = fz ? d.nx : d.nx * d.ny; s.sf = fx ? 1 : (fz ? d.nx * d.ny : d.nx);
    s.pu = fx ? d.py : d.px; s.pv = fz ? d.py : d.pz; s.pf = fx ? d.px : (fz ? d.pz : d.py);
    s.wu = fx ? L.A.wy : L.A.wx; s.wv = fz ? L.A.wy : L.A.wz; s.wf = fx ? L.A.wx : (fz ? L.A.wz : L.A.wy);
    s.invd = L.A.invd;
    s.Cu = fx ? c.ny : c.nx; s.Cv = fz ? c.ny : c.nz; s.Cf = fx ? c.nx : (fz ? c.nz : c.ny);
    s.cu = fx ? c.nx : 1; s.cv = fz ? c.nx : c.nx * c.ny; s.cf = fx ? 1 : (fz ? c.nx * c.ny : c.nx);
    const int q = (s.Cf + (int)cl.num_blocks() - 1) / (int)cl.num_blocks();
    s.K0 = min(s.Cf, (int)cl.block_rank() * q);
    s.K1 = min(s.Cf, s.K0 + q);
    s.base = 2 * s.K0 - 3;
    s.o_r = a.o_slab_r; s.o_z = a.o_slab_z; s.o_t = a.o_slab_t; s.o_i = a.o_slab_i;
    return s;
}

// Actual plane of virtual plane f, or -1 if there is none.
template <class T>
__device__ __forceinline__ int slab_plane(const Slab<T>& s, int f) {
    if (f >= 0 && f < s.nF) return f;
    if (!s.pf) return -1;
    f %= s.nF;
    return f < 0 ? f + s.nF : f;
}

// f(plane, pair) over np planes from virtual plane f0, B items in flight:
// load(q, plane, pair, ok) for each of a batch, then use(q) for each.
template <int B, class T, class L, class U>
__device__ __forceinline__ void slab_loop(const Slab<T>& s, int f0, int np, L load, U use) {
    const int tot = np * s.P2;
    const int dp = TAIL_THREADS / s.P2, dh = TAIL_THREADS - dp * s.P2;
    int pl = (int)threadIdx.x / s.P2, hp = (int)threadIdx.x - pl * s.P2;
    for (int it = threadIdx.x; it < tot; it += B * TAIL_THREADS) {
#pragma unroll
        for (int q = 0; q < B; q++) {
            load(q, f0 + pl, hp, it + q * TAIL_THREADS < tot);
            hp += dh;
            pl += dp;
            if (hp >= s.P2) { hp -= s.P2; pl++; }
        }
#pragma unroll
        for (int q = 0; q < B; q++) use(q);
    }
}

constexpr unsigned SI_UL = 1u << 20, SI_UU = 1u << 21, SI_VL = 1u << 22, SI_VU = 1u << 23;

// pair table of a plane: u / 2, v, row-end flags
template <class T>
__device__ void slab_table(const Slab<T>& s) {
    unsigned* tab = sm<unsigned>(s.o_i);
    for (int h = threadIdx.x; h < s.P2; h += TAIL_THREADS) {
        const int v = h / s.U2, u2 = h - v * s.U2;
        tab[h] = (unsigned)u2 | ((unsigned)v << 10) | (u2 == 0 ? SI_UL : 0) | (u2 == s.U2 - 1 ? SI_UU : 0) |
                 (v == 0 ? SI_VL : 0) | (v == s.V - 1 ? SI_VU : 0);
    }
}

// One cell's six weights (and invd) and which of its faces end the level.
template <class T>
struct SlabCell {
    T w[6], id;
    int c;               // index in the slab's vectors, -1: nothing to do
    unsigned end;        // bit 2 axis + upper (u, v, f)
};

// The cell of colour col of pair hp in virtual plane f.
template <bool INVD, class T>
__device__ __forceinline__ void slab_cell(const Slab<T>& s, int f, int hp, int col, bool ok, SlabCell<T>& x) {
    const int fa = ok ? slab_plane(s, f) : -1;
    x.c = -1;
    if (fa < 0) return;
    const unsigned info = sm<unsigned>(s.o_i)[hp];
    const int u2 = (int)(info & 1023u), v = (int)((info >> 10) & 1023u);
    const int odd = ((v + fa) & 1) ^ col;
    const int g = (2 * u2 + odd) * s.su + v * s.sv + fa * s.sf;
    x.c = (f - s.base) * s.P + 2 * hp + odd;
    const bool uu = (info & SI_UU) && odd, vu = (info & SI_VU) != 0, fu = fa == s.nF - 1;
    x.end = ((info & SI_UL) && !odd ? 1u : 0u) | (uu ? 2u : 0u) | ((info & SI_VL) ? 4u : 0u) | (vu ? 8u : 0u) |
            (fa == 0 ? 16u : 0u) | (fu ? 32u : 0u);
    auto upper = [&](const T* w, bool end, int periodic, int stride, int wrap) {
        const T v = __ldg(w + g + (end ? (periodic ? -wrap : 0) : stride));
        return end && !periodic ? T(0) : v;
    };
    x.w[0] = __ldg(s.wu + g);
    x.w[1] = upper(s.wu, uu, s.pu, s.su, (s.U - 1) * s.su);
    x.w[2] = __ldg(s.wv + g);
    x.w[3] = upper(s.wv, vu, s.pv, s.sv, (s.V - 1) * s.sv);
    x.w[4] = __ldg(s.wf + g);
    x.w[5] = upper(s.wf, fu, s.pf, s.sf, (s.nF - 1) * s.sf);
    if (INVD) x.id = __ldg(s.invd + g);
}

// sum_f w_f z_nbr; a missing neighbour reads the cell itself with weight 0
// (neighbours along f by slot, also across a periodic end).
template <class T>
__device__ __forceinline__ T slab_sum(const Slab<T>& s, const SlabCell<T>& x, const T* z) {
    const T* zc = z + x.c;
    const int wu = s.pu ? s.U - 1 : 0, wv = s.pv ? (s.V - 1) * s.U : 0;
    T v = x.w[0] * zc[(x.end & 1u) ? wu : -1];
    v += x.w[1] * zc[(x.end & 2u) ? -wu : 1];
    v += x.w[2] * zc[(x.end & 4u) ? wv : -s.U];
    v += x.w[3] * zc[(x.end & 8u) ? -wv : s.U];
    v += x.w[4] * zc[(x.end & 16u) && !s.pf ? 0 : -s.P];
    v += x.w[5] * zc[(x.end & 32u) && !s.pf ? 0 : s.P];
    return v;
}

template <class T>
struct SlabBatch {
    // cells whose loads a thread issues together: 3 (at 32^3 a phase has 3, 2
    // or 1 per thread); in FP64 the FP64 pipe bounds the phases, not the loads
    static constexpr int B = sizeof(T) == 4 ? 3 : 1;
};

// z of colour col on np planes from f0.
template <class T>
__device__ __forceinline__ void slab_colour(const Slab<T>& s, int col, int f0, int np) {
    constexpr int B = SlabBatch<T>::B;
    T* z = sm<T>(s.o_z);
    const T* r = sm<T>(s.o_r);
    SlabCell<T> x[B];
    slab_loop<B>(
        s, f0, np, [&](int q, int f, int hp, bool ok) { slab_cell<true>(s, f, hp, col, ok, x[q]); },
        [&](int q) {
            if (x[q].c >= 0) z[x[q].c] = x[q].id * (r[x[q].c] + slab_sum(s, x[q], z));
        });
}

// r from global memory, the pre-sweep, the residual, and the owned planes of
// the next level's r to global memory (the caller's cluster barrier follows).
template <class T>
__device__ void slab_down(const TailArgs<T>& a, const Slab<T>& s) {
    if (s.K0 >= s.K1) return;
    constexpr int B = SlabBatch<T>::B;
    const TailLevel<T>& L = a.L[a.slab];
    T* rs = sm<T>(s.o_r);
    T* z = sm<T>(s.o_z);
    T* t = sm<T>(s.o_t);
    const unsigned* tab = sm<unsigned>(s.o_i);
    const int f0 = 2 * s.K0, nf = 2 * (s.K1 - s.K0);
    {
        T rv[2 * B], iv[2 * B];
        int at[B];
        slab_loop<B>(
            s, f0 - 3, nf + 6,
            [&](int q, int f, int hp, bool ok) {
                const int fa = ok ? slab_plane(s, f) : -1;
                at[q] = -1;
                if (fa < 0) return;
                const unsigned info = tab[hp];
                const int g = 2 * (int)(info & 1023u) * s.su + (int)((info >> 10) & 1023u) * s.sv + fa * s.sf;
                at[q] = (f - s.base) * s.P + 2 * hp;
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    rv[2 * q + e] = __ldcg(L.r + g + e * s.su);
                    iv[2 * q + e] = __ldg(s.invd + g + e * s.su);
                }
            },
            [&](int q) {
                if (at[q] < 0) return;
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    rs[at[q] + e] = rv[2 * q + e];
                    z[at[q] + e] = rv[2 * q + e] * iv[2 * q + e];
                }
            });
    }
    __syncthreads();
    slab_colour(s, 1, f0 - 2, nf + 4);
    __syncthreads();
    {
        SlabCell<T> x[B];
        int at[B];
        slab_loop<B>(
            s, f0 - 1, nf + 2,
            [&](int q, int f, int hp, bool ok) {
                slab_cell<false>(s, f, hp, 0, ok, x[q]);
                at[q] = (f - (f0 - 1)) * s.P2 + hp;
            },
            [&](int q) {
                if (x[q].c >= 0) t[at[q]] = slab_sum(s, x[q], z);
            });
    }
    __syncthreads();
    // four lanes per coarse cell, one fine plane each (see restrict_plane)
    const T wt[4] = {T(0.25), T(0.75), T(0.75), T(0.25)};
    const int Pc = s.Cu * s.Cv, nc = (s.K1 - s.K0) * Pc;
    T* rc = a.L[a.slab + 1].r;
    for (int it = threadIdx.x; it < ((4 * nc + 31) & ~31); it += TAIL_THREADS) {
        const int c = min(it >> 2, nc - 1), tk = it & 3;
        const int dk = c / Pc, rem = c - dk * Pc, J = rem / s.Cu, I = rem - J * s.Cu, K = s.K0 + dk;
        int f = 2 * K - 1 + tk;
        if (!s.pf) f = min(max(f, 0), s.nF - 1);
        const T* tp = t + (f - (f0 - 1)) * s.P2;
        T v = T(0);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int fv = tail_fine_tap(J, q, s.V, s.pv);
            const bool o = ((fv + f) & 1) != 0;
            int e = o ? I - 1 : I + 1;
            const bool out = e < 0 || e >= s.U2;
            if (out) e = e < 0 ? s.U2 - 1 : 0;
            const T far = out && !s.pu ? T(0) : tp[fv * s.U2 + e];
            const bool folded = !s.pu && (o ? I == s.U2 - 1 : I == 0);
            v += wt[q] * ((folded ? T(1) : T(0.75)) * tp[fv * s.U2 + I] + T(0.25) * far);
        }
        v *= wt[tk];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (tk == 0 && it < 4 * nc) rc[I * s.cu + J * s.cv + K * s.cf] = v * T(0.125);
    }
}

// The correction from the next level's z (global memory), the post-sweep, and
// the owned planes of z to global memory.
template <class T>
__device__ void slab_up(const TailArgs<T>& a, const Slab<T>& s) {
    if (s.K0 >= s.K1) return;
    const TailLevel<T>& L = a.L[a.slab];
    const T* rs = sm<T>(s.o_r);
    T* z = sm<T>(s.o_z);
    T* zc = sm<T>(s.o_t);       // coarse planes K0 - 2 .. K1 + 1, rows of Cu
    const unsigned* tab = sm<unsigned>(s.o_i);
    const int f0 = 2 * s.K0, nf = 2 * (s.K1 - s.K0);
    const int Pc = s.Cu * s.Cv, ncp = (s.K1 - s.K0) + 4;
    const T* zg = a.L[a.slab + 1].z;
    for (int it = threadIdx.x; it < ncp * Pc; it += TAIL_THREADS) {
        const int dk = it / Pc, rem = it - dk * Pc, J = rem / s.Cu, I = rem - J * s.Cu;
        int K = s.K0 - 2 + dk;
        if (K < 0 || K >= s.Cf) {
            if (!s.pf) continue;
            K %= s.Cf;
            if (K < 0) K += s.Cf;
        }
        zc[it] = __ldcg(zg + I * s.cu + J * s.cv + K * s.cf);
    }
    __syncthreads();
    // red z = r * invd + correction (black ones are replaced by the sweep)
    slab_loop<1>(
        s, f0 - 2, nf + 4,
        [&](int, int f, int hp, bool ok) {
            const int fa = ok ? slab_plane(s, f) : -1;
            if (fa < 0) return;
            const unsigned info = tab[hp];
            const int u2 = (int)(info & 1023u), v = (int)((info >> 10) & 1023u);
            const int odd = (v + fa) & 1;
            const int at = (f - s.base) * s.P + 2 * hp + odd;
            const T id = __ldg(s.invd + (2 * u2 + odd) * s.su + v * s.sv + fa * s.sf);
            int I1 = odd ? u2 + 1 : u2 - 1;
            if (I1 < 0) I1 = s.pu ? s.Cu - 1 : u2;
            if (I1 >= s.Cu) I1 = s.pu ? 0 : u2;
            const int J0 = v >> 1;
            int J1 = (v & 1) ? J0 + 1 : J0 - 1;
            if (J1 < 0) J1 = s.pv ? s.Cv - 1 : J0;
            if (J1 >= s.Cv) J1 = s.pv ? 0 : J0;
            const int Kv = f >> 1;
            int K1 = (f & 1) ? Kv + 1 : Kv - 1;
            if (!s.pf && (K1 < 0 || K1 >= s.Cf)) K1 = Kv;
            const T* pa = zc + (Kv - (s.K0 - 2)) * Pc;
            const T* pb = zc + (K1 - (s.K0 - 2)) * Pc;
            auto row = [&](const T* b) { return T(0.75) * b[u2] + T(0.25) * b[I1]; };
            const T e0 = T(0.75) * row(pa + J0 * s.Cu) + T(0.25) * row(pa + J1 * s.Cu);
            const T e1 = T(0.75) * row(pb + J0 * s.Cu) + T(0.25) * row(pb + J1 * s.Cu);
            z[at] = rs[at] * id + (T(0.75) * e0 + T(0.25) * e1);
        },
        [](int) {});
    __syncthreads();
    slab_colour(s, 1, f0 - 1, nf + 2);
    __syncthreads();
    slab_colour(s, 0, f0, nf);
    __syncthreads();
    slab_loop<1>(
        s, f0, nf,
        [&](int, int f, int hp, bool ok) {
            if (!ok) return;
            const unsigned info = tab[hp];
            const int g = 2 * (int)(info & 1023u) * s.su + (int)((info >> 10) & 1023u) * s.sv + f * s.sf;
            const int at = (f - s.base) * s.P + 2 * hp;
            L.z[g] = z[at];
            L.z[g + s.su] = z[at + 1];
        },
        [](int) {});
}

// What a CTA can do before the tail's input is ready.
template <class T>
__device__ __forceinline__ void tail_prologue(const TailArgs<T>& a, cg::cluster_group& cl) {
    if (cl.block_rank() == 0) {
        if (sizeof(T) == 4 && a.coef_smem) solo_prefetch<true, T>(a, threadIdx.x, TAIL_THREADS);
        else solo_prefetch<false, T>(a, threadIdx.x, TAIL_THREADS);
    }
    if (a.slab >= 0) slab_table(slab_of(a, cl));
}

// The solo levels, r of the first from and its z to global memory.
template <bool CS, class T>
__device__ void solo_levels(const TailArgs<T>& a, cg::cluster_group& cl) {
    const int tid = threadIdx.x, nth = TAIL_THREADS;
    const int ls = a.small_from, nl = a.nlev;
    const TailLevel<T>& F = a.L[ls];
    const TailLevel<T>& Z = a.L[nl - 1];
    if (!(a.big_coarse && ls == nl - 1)) {
        for (int c = tid; c < (int)F.d.n; c += nth) {
            const T v = __ldcg(F.r + c);
            sm<T>(F.o_r)[c] = v;
            if (ls < nl - 1) sm<T>(F.o_z)[c] = v * __ldg(F.A.invd + c);
        }
        cp_async_wait();
        __syncthreads();
    }
    for (int l = ls; l < nl - 1; l++) solo_down<CS, T>(a, l, tid, nth);
    if (a.big_coarse) {
        const int n = (int)Z.d.n;
        if (ls < nl - 1)
            for (int c = tid; c < n; c += nth) Z.r[c] = sm<T>(Z.o_r)[c];
        cl.sync();
        cluster_coarsest<T>(a, cl);
        if (ls == nl - 1) return;
        for (int c = tid; c < n; c += nth) sm<T>(Z.o_z)[c] = __ldcg(Z.z + c);
        __syncthreads();
    } else {
        solo_coarsest<T>(a, tid, nth);
    }
    for (int l = nl - 2; l >= ls; l--) solo_up<CS, T>(a, l, tid, nth);
    for (int c = tid; c < (int)F.d.n; c += nth) F.z[c] = sm<T>(F.o_z)[c];
}

// One V-cycle from the tail's first level down and back up, run by every
// thread of the calling cluster after tail_prologue.  end_sync: a last cluster
// barrier, so that L[0].z is visible to the whole cluster on return.
template <class T>
__device__ __forceinline__ void tail_cycle(const TailArgs<T>& a, cg::cluster_group& cl, bool end_sync) {
    const int gthreads = TAIL_THREADS * (int)cl.num_blocks();
    const int gtid = (int)cl.block_rank() * TAIL_THREADS + (int)threadIdx.x;
    const int nl = a.nlev, ls = a.small_from;
    const int lg = a.slab >= 0 ? a.slab : ls;      // levels 0 .. lg - 1 phase by phase over the cluster
    auto csync = [&]() { cl.sync(); };
    for (int l = 0; l < lg; l++) {
        const TailLevel<T>& L = a.L[l];
        tail_down<T>(L, Vec<T>{L.r, L.z, L.t}, a.L[l + 1].d, a.L[l + 1].r, a.pre, gtid, gthreads, csync);
    }
    if (a.slab >= 0) {
        __syncthreads();
        slab_down<T>(a, slab_of(a, cl));
        cl.sync();
    }
    if (cl.block_rank() == 0) {
        if (sizeof(T) == 4 && a.coef_smem) solo_levels<true, T>(a, cl);
        else solo_levels<false, T>(a, cl);
    } else if (a.big_coarse) {
        cl.sync();
        cluster_coarsest<T>(a, cl);
    }
    if (lg > 0 || a.slab >= 0 || end_sync) cl.sync();
    if (a.slab >= 0) {
        slab_up<T>(a, slab_of(a, cl));
        if (lg > 0 || end_sync) cl.sync();
    }
    for (int l = lg - 1; l >= 0; l--) {
        const TailLevel<T>& L = a.L[l];
        tail_up<T>(L, Vec<T>{L.r, L.z, L.t}, a.L[l + 1].d, a.L[l + 1].z, a.post, a.paper_order ? 0 : 1, gtid,
                   gthreads, csync);
    }
    (void)nl;
}

template <class T>
__global__ void __launch_bounds__(TAIL_THREADS) k_vtail(const __grid_constant__ TailArgs<T> a) {
    cg::cluster_group cl = cg::this_cluster();
    tail_prologue<T>(a, cl);
    tail_cycle<T>(a, cl, false);
}

// ---------------------------------------------------------------------------
// Persistent inner solves over a work list (mixed precision).
//
// Each cluster takes a ticket, solves that request's FP32 system A x = r by
// MG-preconditioned CG (Table 1's solver: the V-cycle over all of the
// request's levels, then the CG vector operations) to its threshold or
// iteration cap, and takes the next ticket; the requests may have any grid
// sizes.  Phases are separated by the hardware cluster barrier and the dot
// products are summed in a fixed order (per thread in its cell order with
// error-free FP32 products, per CTA by warps, then the CTAs' partials in
// rank order, read by every CTA from distributed shared memory), so every
// CTA computes the same scalars and a request's result depends only on the
// cluster shape, never on the other requests or on which cluster took it.

// Sum of v over the cluster, the same in every thread of every CTA.  part:
// a __shared__ slot of this CTA, not written again before the next cluster
// barrier that follows this call.
__device__ __forceinline__ double ps_cluster_sum(double v, double* part, cg::cluster_group& cl) {
    __shared__ double wsum[TAIL_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    if (lane == 0) wsum[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double t = wsum[lane];
        t = warp_sum(t);
        if (lane == 0) *part = t;
    }
    cl.sync();
    double tot = 0.0;
    const unsigned nb = cl.num_blocks();
    for (unsigned b = 0; b < nb; b++) tot += *cl.map_shared_rank(part, b);
    return tot;
}

// The inner solve of one request: r holds the scaled residual, x = 0.
__device__ void ps_solve(const PsReq& R, cg::cluster_group& cl, double* part) {
    const TailArgs<float>& a = R.v;
    const Dims& d = a.L[0].d;
    const Op<float>& A = a.L[0].A;
    float* r = a.L[0].r;
    float* z = a.L[0].z;
    float* p = R.p;
    float* q = R.q;
    float* x = R.x;
    const int nth = TAIL_THREADS * (int)cl.num_blocks();
    const int tid = (int)cl.block_rank() * TAIL_THREADS + (int)threadIdx.x;
    const int n = (int)d.n;
    const double thresh = __ldcg(R.sc + S_THRESH);
    const int maxit = (int)__ldcg(R.sc + S_MAXIT);
    double rho = 0.0, rho_old = 0.0, beta = 0.0, pq = 0.0, alpha = 0.0, rr = __ldcg(R.sc + S_RR);
    int k = 0, slot = 0;
    bool bad = false;
    tail_prologue<float>(a, cl);
    while (k < maxit) {
        tail_cycle<float>(a, cl, true);   // z = M r
        DotAcc<float> arz;
        for (int c = tid; c < n; c += nth) arz.add(__ldcg(r + c), __ldcg(z + c));
        rho = ps_cluster_sum(arz.value(), part + slot, cl);
        slot = (slot + 1) & 3;
        beta = k == 0 ? 0.0 : rho / rho_old;
        rho_old = rho;
        const float bf = (float)beta;
        if (k == 0)
            for (int c = tid; c < n; c += nth) p[c] = __ldcg(z + c);
        else
            for (int c = tid; c < n; c += nth) p[c] = fmaf(bf, __ldcg(p + c), __ldcg(z + c));
        cl.sync();
        // q = A p and <p, q>
        DotAcc<float> apq;
        for (Walk w(d, tid, nth); w.more(); w.next()) {
            const int c = w.c;
            float swu, sw;
            tail_nbr_sums<float>(d, A, c, w.i, w.j, w.k, p, swu, sw);
            const float pc = __ldcg(p + c);
            const float qc = A.m[c] * pc + sw * pc - swu;
            q[c] = qc;
            apq.add(pc, qc);
        }
        pq = ps_cluster_sum(apq.value(), part + slot, cl);
        slot = (slot + 1) & 3;
        alpha = rho / pq;
        const float af = (float)alpha;
        // x += alpha p, r -= alpha q, ||r||^2
        DotAcc<float> arr;
        for (int c = tid; c < n; c += nth) {
            // x starts at 0 (the caller's x32 is not cleared)
            x[c] = k == 0 ? af * __ldcg(p + c) : fmaf(af, __ldcg(p + c), __ldcg(x + c));
            const float rn = fmaf(-af, __ldcg(q + c), __ldcg(r + c));
            r[c] = rn;
            arr.add(rn, rn);
        }
        rr = ps_cluster_sum(arr.value(), part + slot, cl);
        slot = (slot + 1) & 3;
        k++;
        if (!isfinite(rho) || !isfinite(alpha) || !isfinite(rr)) {
            bad = true;
            break;
        }
        if (rr <= thresh) break;
    }
    if (cl.block_rank() == 0 && threadIdx.x == 0) {
        double* sc = R.sc;
        sc[S_RHO] = rho;
        sc[S_RHO_OLD] = rho_old;
        sc[S_BETA] = beta;
        sc[S_PQ] = pq;
        sc[S_ALPHA] = alpha;
        sc[S_RR] = rr;
        sc[S_KITER] = (double)k;
        sc[S_FIRST] = 0.0;
        if (bad) sc[S_NONFINITE] = 1.0;
    }
}

// Sum of a per-thread compensated pair over the CTA: warps by shuffles on the
// FP32 pipe (five FP64 additions per warp would cost 80 cycles of the SM's FP64
// pipe each, times 32 warps), then warp 0 the warps' partials; thread 0 passes
// the sum to use(), which may write shared memory that every thread reads after
// the call.  A third component keeps FP64's accuracy (1.2e-16 to 3.0e-16 rms of
// a sum of 2048 to 8192 products; 1.3e-16 to 3.1e-16 with FP64 additions,
// 1.4e-15 to 2.1e-15 with the pairs alone).
template <class U>
__device__ __forceinline__ void ps_block_sum(DotAcc<float> v, U use) {
    __shared__ DotSum part[TAIL_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    DotSum s{v.hi, v.lo, 0.0f};
    auto reduce = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float uh = __shfl_xor_sync(0xffffffffu, s.hi, o);
            const float ul = __shfl_xor_sync(0xffffffffu, s.lo, o);
            const float uc = __shfl_xor_sync(0xffffffffu, s.c, o);
            s.merge(uh, ul, uc);
        }
    };
    reduce();
    if (lane == 0) part[warp] = s;
    __syncthreads();
    if (warp == 0) {
        s = part[lane];
        reduce();
        if (lane == 0) use(s.value());
    }
    __syncthreads();
}

// The inner solve of a small request by one CTA: a V-cycle of solo levels from
// the fine one down, p and r in shared memory, x and q of a thread's own pairs
// of cells in registers.  FP64 scalars are formed by one thread.
constexpr int PS_PAIRS = 4;      // pairs per thread: fine grids up to 8192 cells
template <bool CS>
__device__ void ps_solve_cta(const PsReq& R) {
    __shared__ float s_beta, s_alpha;
    __shared__ int s_stop;
    __shared__ double s_rho, s_pq, s_rr;
    const TailArgs<float>& a = R.v;
    const int nl = a.nlev, tid = threadIdx.x, nth = TAIL_THREADS;
    const TailLevel<float>& L = a.L[0];
    const int n2 = (int)(L.d.n >> 1);
    float* r = sm<float>(L.o_r);
    float* z = sm<float>(L.o_z);
    float* p = sm<float>(a.o_p);
    const unsigned* tab = sm<unsigned>(L.o_i);
    solo_prefetch<CS, float>(a, tid, nth);
    float2 x[PS_PAIRS], q[PS_PAIRS];
#pragma unroll
    for (int e = 0; e < PS_PAIRS; e++) {
        const int h = tid + e * nth;
        x[e] = make_float2(0.f, 0.f);
        if (h < n2) {
            const float2 v = __ldcg(reinterpret_cast<const float2*>(L.r) + h);
            const float2 iv = __ldg(reinterpret_cast<const float2*>(L.A.invd) + h);
            reinterpret_cast<float2*>(r)[h] = v;
            reinterpret_cast<float2*>(z)[h] = make_float2(v.x * iv.x, v.y * iv.y);
        }
    }
    const double thresh = __ldcg(R.sc + S_THRESH);
    const int maxit = (int)__ldcg(R.sc + S_MAXIT);
    if (tid == 0) {
        s_rho = s_pq = 0.0;
        s_beta = s_alpha = 0.0f;
        s_rr = __ldcg(R.sc + S_RR);
    }
    double rho_old = 0.0;        // thread 0's
    bool bad = false;
    int k = 0;
    cp_async_wait();
    __syncthreads();
    while (k < maxit) {
        for (int l = 0; l < nl - 1; l++) solo_down<CS, float>(a, l, tid, nth);
        solo_coarsest<float>(a, tid, nth);
        for (int l = nl - 2; l >= 0; l--) solo_up<CS, float>(a, l, tid, nth);
        DotAcc<float> acc;
#pragma unroll
        for (int e = 0; e < PS_PAIRS; e++) {
            const int h = tid + e * nth;
            if (h < n2) {
                const float2 rv = reinterpret_cast<const float2*>(r)[h], zv = reinterpret_cast<const float2*>(z)[h];
                acc.add(rv.x, zv.x);
                acc.add(rv.y, zv.y);
            }
        }
        ps_block_sum(acc, [&](double rho) {
            s_beta = k == 0 ? 0.0f : (float)(rho / rho_old);
            rho_old = rho;
            s_rho = rho;
        });
        const float bf = s_beta;
#pragma unroll
        for (int e = 0; e < PS_PAIRS; e++) {
            const int h = tid + e * nth;
            if (h < n2) {
                float2 pv = reinterpret_cast<const float2*>(z)[h];
                if (k > 0) {
                    const float2 po = reinterpret_cast<const float2*>(p)[h];
                    pv = make_float2(fmaf(bf, po.x, pv.x), fmaf(bf, po.y, pv.y));
                }
                reinterpret_cast<float2*>(p)[h] = pv;
            }
        }
        __syncthreads();
        acc = DotAcc<float>();
#pragma unroll
        for (int e = 0; e < PS_PAIRS; e++) {
            const int h = tid + e * nth;
            if (h < n2) {
                const unsigned info = tab[h];
                float qv[2];
#pragma unroll
                for (int odd = 0; odd < 2; odd++) {
                    const int c = 2 * h + odd;
                    float sw;
                    const float swu = solo_sum<CS, true, float>(L, p, c, info, odd, &sw);
                    const float pc = p[c];
                    qv[odd] = coef<CS>(L, 4, c) * pc + sw * pc - swu;
                    acc.add(pc, qv[odd]);
                }
                q[e] = make_float2(qv[0], qv[1]);
            }
        }
        ps_block_sum(acc, [&](double pq) {
            const double alpha = s_rho / pq;
            s_pq = pq;
            s_alpha = (float)alpha;
            s_stop = isfinite(s_rho) && isfinite(alpha) ? 0 : 2;
        });
        const float af = s_alpha;
        acc = DotAcc<float>();
#pragma unroll
        for (int e = 0; e < PS_PAIRS; e++) {
            const int h = tid + e * nth;
            if (h < n2) {
                const float2 pv = reinterpret_cast<const float2*>(p)[h];
                float2 rv = reinterpret_cast<const float2*>(r)[h];
                x[e] = make_float2(fmaf(af, pv.x, x[e].x), fmaf(af, pv.y, x[e].y));
                rv = make_float2(fmaf(-af, q[e].x, rv.x), fmaf(-af, q[e].y, rv.y));
                reinterpret_cast<float2*>(r)[h] = rv;
                reinterpret_cast<float2*>(z)[h] =
                    make_float2(rv.x * coef<CS>(L, 0, 2 * h), rv.y * coef<CS>(L, 0, 2 * h + 1));
                acc.add(rv.x, rv.x);
                acc.add(rv.y, rv.y);
            }
        }
        ps_block_sum(acc, [&](double rr) {
            s_rr = rr;
            if (!isfinite(rr)) s_stop = 2;
            else if (s_stop == 0 && rr <= thresh) s_stop = 1;
        });
        k++;
        if (s_stop) {
            bad = s_stop == 2;
            break;
        }
    }
#pragma unroll
    for (int e = 0; e < PS_PAIRS; e++) {
        const int h = tid + e * nth;
        if (h < n2) reinterpret_cast<float2*>(R.x)[h] = x[e];
    }
    if (tid == 0) {
        double* sc = R.sc;
        sc[S_RHO] = s_rho;
        sc[S_RHO_OLD] = rho_old;
        sc[S_BETA] = (double)s_beta;
        sc[S_PQ] = s_pq;
        sc[S_ALPHA] = s_rho / s_pq;
        sc[S_RR] = s_rr;
        sc[S_KITER] = (double)k;
        sc[S_FIRST] = 0.0;
        if (bad) sc[S_NONFINITE] = 1.0;
    }
}

__global__ void __launch_bounds__(TAIL_THREADS) k_psolve(const __grid_constant__ PsBatch b) {
    __shared__ __align__(16) PsReq R;
    __shared__ double part[4];
    __shared__ int item;
    cg::cluster_group cl = cg::this_cluster();
    for (;;) {
        if (cl.block_rank() == 0 && threadIdx.x == 0) item = (int)atomicAdd(b.ticket, 1u);
        cl.sync();
        const int it = *cl.map_shared_rank(&item, 0);
        // every CTA has read the ticket before CTA 0 may draw the next one
        // or exit (its shared memory must outlive the remote reads)
        cl.sync();
        if (it >= b.ncl) break;
        const unsigned* src = reinterpret_cast<const unsigned*>(b.req[it]);
        unsigned* dst = reinterpret_cast<unsigned*>(&R);
        for (int w = threadIdx.x; w < (int)(sizeof(PsReq) / 4); w += TAIL_THREADS) dst[w] = __ldcg(src + w);
        __syncthreads();
        ps_solve(R, cl, part);
        // the last reduction's remote reads are done before the next request
        cl.sync();
    }
    // then the small requests, each CTA on its own (no remote accesses
    // follow, so the CTAs may finish independently)
    for (;;) {
        if (threadIdx.x == 0) item = b.ncl + (int)atomicAdd(b.ticket + 1, 1u);
        __syncthreads();
        const int it = item;
        __syncthreads();
        if (it >= b.n) break;
        const unsigned* src = reinterpret_cast<const unsigned*>(b.req[it]);
        unsigned* dst = reinterpret_cast<unsigned*>(&R);
        for (int w = threadIdx.x; w < (int)(sizeof(PsReq) / 4); w += TAIL_THREADS) dst[w] = __ldcg(src + w);
        __syncthreads();
        if (R.v.coef_smem) ps_solve_cta<true>(R);
        else ps_solve_cta<false>(R);
        __syncthreads();
    }
}

}  // namespace

namespace {

cudaLaunchConfig_t tail_config(int cluster, cudaStream_t s, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster, 1, 1);
    cfg.blockDim = dim3(TAIL_THREADS, 1, 1);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

// Chooses how each level of the tail runs and lays out the shared memory.
// Solo: from the first level of at most TAIL_SOLO_CELLS cells that fits
// (4096: a 16^3 level's operator takes 64 KB); in FP64 512, since one SM's two
// FP64 lanes take 50 us for a 16^3 level, halo slabs on eight SMs 15.
// The level above it as a slab where Table 1's cycle (one sweep down, one up)
// runs and its planes fit.  Any other level phase by phase over the cluster.
// Coefficients move to shared memory in FP32 where they fit.  A coarsest grid
// of more than 256 (FP64: 160) cells is applied by the whole cluster: n^2
// products then cost more on one SM than two more cluster barriers.
// solve: the layout of a whole inner solve by one CTA (every level solo).
template <class T>
bool plan_tail(TailArgs<T>& a, int cluster, bool solve) {
    const int nl = a.nlev;
    const TailLevel<T>& Z = a.L[nl - 1];
    a.solve = solve ? 1 : 0;
    a.big_coarse = !solve && cluster > 1 && Z.d.n > (sizeof(T) == 4 ? 256 : 160) ? 1 : 0;
    const size_t limit = solve ? PS_SMEM_MAX : TAIL_SMEM_MAX;
    auto fits = [&](int ls, int slab, bool cs) {
        size_t off = 0;
        auto take = [&](size_t bytes) {
            const size_t o = off;
            off += (bytes + 15) & ~(size_t)15;
            return (int)o;
        };
        size_t region = 0;
        int P2 = 0;
        if (slab >= 0) {
            const Dims& d = a.L[slab].d;
            const int n[3] = {d.nx, d.ny, d.nz};
            const int f = n[2] >= n[0] && n[2] >= n[1] ? 2 : (n[1] >= n[0] ? 1 : 0);
            const int U = n[f == 0 ? 1 : 0], V = n[f == 2 ? 1 : 2];
            const size_t P = (size_t)U * V, q = (n[f] / 2 + cluster - 1) / cluster;
            if (P > 8192 || U > 2046 || V > 1023) return false;
            P2 = (int)(P / 2);
            a.slab_axis = f;
            a.o_slab_r = take((2 * q + 6) * P * sizeof(T));
            // z and the red residual share their room with the solo vectors
            // (CTA 0 is never in both)
            a.o_slab_z = (int)off;
            region = (2 * q + 6) * P * sizeof(T);
            a.o_slab_t = (int)(off + region);
            region += (q + 1) * P * sizeof(T);
        }
        const size_t base = off;
        for (int l = ls; l < nl; l++) {
            const size_t n = (size_t)a.L[l].d.n;
            a.L[l].o_r = take(n * sizeof(T));
            a.L[l].o_z = take(n * sizeof(T));
            if (l < nl - 1) a.L[l].o_t = take(n / 2 * sizeof(T));
        }
        if (off < base + region) off = (base + region + 15) & ~(size_t)15;
        for (int l = ls; l < nl - 1; l++) {
            const size_t n = (size_t)a.L[l].d.n;
            if (cs) a.L[l].o_c = take((solve && l == 0 ? 5 : 4) * n * sizeof(T));
            a.L[l].o_i = take(n / 2 * sizeof(unsigned));
        }
        if (solve) a.o_p = take((size_t)a.L[0].d.n * sizeof(T));
        a.o_ainv = -1;
        if (Z.d.n <= 64) a.o_ainv = take((size_t)Z.d.n * (size_t)Z.d.n * sizeof(double));
        if (slab >= 0) a.o_slab_i = take((size_t)P2 * sizeof(unsigned));
        a.small_from = ls;
        a.slab = slab;
        a.coef_smem = cs ? 1 : 0;
        a.smem_bytes = (int)off;
        return off <= limit;
    };
    const bool one = a.pre == 1 && a.post == 1 && !a.paper_order;
    const long long most = solve ? 2LL * PS_PAIRS * TAIL_THREADS : sizeof(T) == 8 ? TAIL_SOLO_CELLS64 : TAIL_SOLO_CELLS;
    for (int ls = 0; ls < nl && (!solve || ls == 0); ls++) {
        if (ls < nl - 1 && a.L[ls].d.n > most) continue;
        for (int slab = ls > 0 && one && !solve ? ls - 1 : -1; slab >= -1; slab = slab >= 0 ? -1 : -2)
            for (int cs = sizeof(T) == 4 ? 1 : 0; cs >= 0; cs--)
                if (fits(ls, slab, cs != 0)) return true;
    }
    return false;
}

template <class T>
cudaError_t launch_vtail(const TailArgs<T>& a, int cluster, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    // every level solo: one CTA
    const bool solo = a.small_from == 0 && a.slab < 0 && !a.big_coarse;
    cudaLaunchConfig_t cfg = tail_config(solo ? 1 : cluster, s, attr);
    cfg.dynamicSmemBytes = a.smem_bytes;
    return cudaLaunchKernelEx(&cfg, k_vtail<T>, a);
}

// The largest cluster (16 CTAs, a non-portable size, else the portable 8)
// of which at least one can be resident; 0 if none.
template <class T>
int vtail_cluster() {
    if (cudaFuncSetAttribute(k_vtail<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        cudaGetLastError();
    if (cudaFuncSetAttribute(k_vtail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAIL_SMEM_MAX) !=
        cudaSuccess)
        cudaGetLastError();
    for (int cluster : {16, 8}) {
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = tail_config(cluster, nullptr, attr);
        cfg.dynamicSmemBytes = TAIL_SMEM_MAX;
        int n = 0;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, k_vtail<T>, &cfg);
        if (e != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (n > 0) return cluster;
    }
    return 0;
}

// Cluster size of the persistent solves (fixed per device, so a request's
// arithmetic never depends on the launch that carries it) and how many such
// clusters can be resident at once; {0, 0} if none fits.
PsShape psolve_shape() {
    static thread_local int dev = -1;
    static thread_local PsShape shape{0, 0};
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) {
        cudaGetLastError();
        return PsShape{0, 0};
    }
    if (d == dev) return shape;
    dev = d;
    shape = PsShape{0, 0};
    if (cudaFuncSetAttribute(k_psolve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS_SMEM_MAX) !=
        cudaSuccess)
        cudaGetLastError();
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tail_config(PS_CLUSTER, nullptr, attr);
    cfg.dynamicSmemBytes = PS_SMEM_MAX;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_psolve, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    if (n > 0) shape = PsShape{PS_CLUSTER, n};
    return shape;
}

cudaError_t launch_psolve(const PsBatch& b, size_t smem, cudaStream_t s) {
    const PsShape sh = psolve_shape();
    if (sh.cluster == 0) return cudaErrorNotSupported;
    if (b.n < 1) return cudaSuccess;
    // enough clusters for the cluster requests and for one CTA per small one
    const int ncta = b.n - b.ncl;
    int clusters = b.ncl > (ncta + sh.cluster - 1) / sh.cluster ? b.ncl : (ncta + sh.cluster - 1) / sh.cluster;
    if (clusters > sh.clusters) clusters = sh.clusters;
    cudaError_t e = cudaMemsetAsync(b.ticket, 0, 2 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tail_config(sh.cluster, s, attr);
    cfg.gridDim = dim3(sh.cluster * clusters, 1, 1);
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, k_psolve, b);
}

template bool plan_tail<float>(TailArgs<float>&, int, bool);
template bool plan_tail<double>(TailArgs<double>&, int, bool);
template cudaError_t launch_vtail<float>(const TailArgs<float>&, int, cudaStream_t);
template cudaError_t launch_vtail<double>(const TailArgs<double>&, int, cudaStream_t);
template int vtail_cluster<float>();
template int vtail_cluster<double>();

}  // namespace fld
