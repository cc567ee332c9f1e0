// k_pair.cu -- the FP64 solver's sweeps, a pair of cells (2s, 2s + 1) along x
// per thread, one red and one black.
//
// GB300 has two FP64 lanes per SM and clock, so these kernels are bound by FP64
// instructions first (1.05 M pairs at 128^3: 1.8 us per FP64 instruction and
// pair), then by L2 and DRAM.  The scalar kernels of k_mg.cu and k_cg.cu issue
// an instruction for a whole warp where a colour needs half its lanes, form a
// red neighbour's r / diag again for each of its six black neighbours, r - A z
// at black cells where it vanishes, the correction at the black cells that the
// next sweep replaces, and p = z + beta p seven times per cell.  Here every
// lane works, values along the z walk stay in registers, those along x come
// from the adjacent lane, and after one sweep from zero the residual is
// sum_f w_f z_nbr at red cells (stored by pair), the restriction reads the red
// values alone, and the correction goes to the colour that is kept.
//
// FP64 instructions per pair, before -> here (and us per launch at 128^3):
// first sweep 30 -> 11 (68 -> 44), residual 32 -> 6 (82 -> 22), colour sweep 16
// -> 8 (39 -> 31), correction 30 -> 9 (68 -> 25), p/q 46 -> 35 (114 -> 84);
// restriction per coarse cell 84 -> 33 (50 -> 21).
#include "walk4.cuh"

namespace fld {

namespace {

struct WalkP {
    int s, j, k0, k1;
    bool valid;
    long long nxy;
    int c, ym, yp;            // first cell of the pair, and of the pairs of rows j -+ 1, within a plane
    int xl, xr;               // first cell of the pairs beside it (wrapped; its own where there is none)
    bool has_xr, has_yp, load_l, load_r;
};

__device__ __forceinline__ WalkP walkp_of(const Dims& d) {
    WalkP w;
    const int nx2 = d.nx >> 1;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    w.valid = s < nx2 && j < d.ny;
    w.s = min(s, nx2 - 1);
    w.j = min(j, d.ny - 1);
    const int kch = (d.nz + (int)gridDim.z - 1) / (int)gridDim.z;
    w.k0 = (int)blockIdx.z * kch;
    w.k1 = min(d.nz, w.k0 + kch);
    w.nxy = (long long)d.nx * d.ny;
    const int row = w.j * d.nx;
    w.c = row + 2 * w.s;
    w.ym = w.j > 0 ? w.c - d.nx : (d.py ? w.c + (d.ny - 1) * d.nx : w.c);
    w.has_yp = w.j < d.ny - 1 || d.py;
    w.yp = w.j < d.ny - 1 ? w.c + d.nx : (d.py ? w.c - (d.ny - 1) * d.nx : w.c);
    const bool first = w.s == 0, last = w.s == nx2 - 1;
    w.xl = first ? (d.px ? row + d.nx - 2 : w.c) : w.c - 2;
    w.xr = last ? (d.px ? row : w.c) : w.c + 2;
    w.has_xr = !last || d.px;
    w.load_l = threadIdx.x == 0 || first;
    w.load_r = threadIdx.x == blockDim.x - 1 || last;
    return w;
}

__device__ __forceinline__ double2 ld2(const double* __restrict__ p, long long i) {
    return *reinterpret_cast<const double2*>(p + i);
}
__device__ __forceinline__ double sel(double2 v, int o) { return o ? v.y : v.x; }

// The six face weights of the pair's cell at position o.
struct FacesP {
    double xl, xu, yl, yu, zl, zu;
};
__device__ __forceinline__ FacesP facesp(const Op<double>& A, const WalkP& w, long long p, double2 wzc, double2 wzu,
                                         bool has_zu, int o) {
    FacesP f;
    const double2 wx = ld2(A.wx, p + w.c);
    // executed by every lane: rows of both parities may share a warp
    const double nx = __shfl_down_sync(FULL, wx.x, 1);
    f.xl = sel(wx, o);
    f.xu = o ? (w.has_xr ? (w.load_r ? A.wx[p + w.xr] : nx) : 0.0) : wx.y;
    f.yl = sel(ld2(A.wy, p + w.c), o);
    f.yu = w.has_yp ? sel(ld2(A.wy, p + w.yp), o) : 0.0;
    f.zl = sel(wzc, o);
    f.zu = has_zu ? sel(wzu, o) : 0.0;
    return f;
}

// x neighbours of the cell at position o: v the other cell of the pair, u the
// value of the other colour's cell beyond (this lane's own at l: that of the
// pairs beside it is theirs)
__device__ __forceinline__ double farp(double own, int o) {
    const double l = __shfl_up_sync(FULL, own, 1);
    const double r = __shfl_down_sync(FULL, own, 1);
    return o ? r : l;
}

}  // namespace

// z of one red/black sweep from zero (natural order).
__global__ void __launch_bounds__(256) k_zero_pair(Dims d, Op<double> A, const double* __restrict__ r,
                                                   double* __restrict__ z) {
    const WalkP w = walkp_of(d);
    if (w.k0 >= w.k1) return;
    auto U = [&](long long i, int o) { return r[i + o] * A.invd[i + o]; };
    long long p = (long long)w.k0 * w.nxy;
    int o = 1 - ((w.j + w.k0) & 1);            // position of the black cell
    double ud = U(p + w.c + zdn(d, w.k0, w.nxy), o);
    double2 rc = ld2(r, p + w.c), ic = ld2(A.invd, p + w.c), wzc = ld2(A.wz, p + w.c);
    for (int k = w.k0; k < w.k1; k++) {
        const long long up = zup(d, k, w.nxy);
        const bool has_zu = k < d.nz - 1 || d.pz;
        const double2 rn = ld2(r, p + w.c + up), in = ld2(A.invd, p + w.c + up), wzu = ld2(A.wz, p + w.c + up);
        const FacesP f = facesp(A, w, p, wzc, wzu, has_zu, o);
        const double uc = sel(rc, 1 - o) * sel(ic, 1 - o);       // the pair's red value
        const double uu = sel(rn, o) * sel(in, o);               // red in plane k + 1
        const double um = U(p + w.ym, o), up_ = U(p + w.yp, o);
        double far = farp(uc, o);
        if (o ? w.load_r : w.load_l) far = U(p + (o ? w.xr : w.xl), 1 - o);
        double a = f.xl * (o ? uc : far);
        a = fma(f.xu, o ? far : uc, a);
        a = fma(f.yl, um, a);
        a = fma(f.yu, up_, a);
        a = fma(f.zl, ud, a);
        a = fma(f.zu, uu, a);
        const double b = sel(ic, o) * (sel(rc, o) + a);
        if (w.valid) *reinterpret_cast<double2*>(z + p + w.c) = o ? make_double2(uc, b) : make_double2(b, uc);
        ud = uc;
        rc = rn;
        ic = in;
        wzc = wzu;
        p += w.nxy;
        o ^= 1;
    }
}

// At the cells of colour col, from the other colour's z: RES: res[pair] =
// sum_f w_f z_nbr; else z = invd (r + sum_f w_f z_nbr) in place, with DOT also
// <r, z> (the last sweep of the cycle).
template <bool RES, bool DOT>
__global__ void __launch_bounds__(256) k_sweep_pair(Dims d, Op<double> A, const double* __restrict__ r, double* z,
                                                    double* __restrict__ res, int col, RedArgs ra) {
    const WalkP w = walkp_of(d);
    DotAcc<double> da;
    if (w.k0 < w.k1) {
        long long p = (long long)w.k0 * w.nxy;
        int o = ((w.j + w.k0) & 1) ^ col;
        const double* zr = z;
        // the other colour's values of the pair's plane and the planes beside
        // it: position 1 - o in this plane, o in the others
        double ud = zr[p + w.c + zdn(d, w.k0, w.nxy) + o];
        double uc = zr[p + w.c + 1 - o];
        double2 wzc = ld2(A.wz, p + w.c);
        for (int k = w.k0; k < w.k1; k++) {
            const long long up = zup(d, k, w.nxy);
            const bool has_zu = k < d.nz - 1 || d.pz;
            const double uu = zr[p + w.c + up + o];
            const double2 wzu = ld2(A.wz, p + w.c + up);
            const FacesP f = facesp(A, w, p, wzc, wzu, has_zu, o);
            const double um = zr[p + w.ym + o], up_ = zr[p + w.yp + o];
            double far = farp(uc, o);
            if (o ? w.load_r : w.load_l) far = zr[p + (o ? w.xr : w.xl) + 1 - o];
            double a = f.xl * (o ? uc : far);
            a = fma(f.xu, o ? far : uc, a);
            a = fma(f.yl, um, a);
            a = fma(f.yu, up_, a);
            a = fma(f.zl, ud, a);
            a = fma(f.zu, uu, a);
            if (RES) {
                if (w.valid) res[(p + w.c) >> 1] = a;
            } else {
                const double2 rc = ld2(r, p + w.c);
                const double v = A.invd[p + w.c + o] * (sel(rc, o) + a);
                if (w.valid) {
                    z[p + w.c + o] = v;
                    if (DOT) {
                        da.add(sel(rc, o), v);
                        da.add(sel(rc, 1 - o), uc);
                    }
                }
            }
            ud = uc;
            uc = uu;
            wzc = wzu;
            p += w.nxy;
            o ^= 1;
        }
    }
    if (DOT) {
        double acc[1] = {da.value()};
        const bool mx[1] = {false};
        grid_reduce<1>(acc, mx, ra);
    }
}

// Full weighting of a residual given at the red cells by pair (see
// k_restrict): per fine row the red taps are 2I, 2I + 2 (even red) or 2I - 1,
// 2I + 1, with weights 3/4 and 1/4; a tap folded onto a red boundary cell adds
// to its weight.  One coarse cell per thread: 32 independent loads, all but a
// few of them L1 hits.
template <class T>
__global__ void __launch_bounds__(256) k_restrict_pair(Dims f, Dims cd, const T* __restrict__ t,
                                                       T* __restrict__ rc) {
    COL_BEGIN(cd)
        const int nx2 = f.nx >> 1;
        auto tap = [](int I, int q, int n, int per) {
            int v = 2 * I - 1 + q;
            if (v < 0) v = per ? v + n : 0;
            if (v >= n) v = per ? v - n : n - 1;
            return v;
        };
        // the pairs beside I, and whether a boundary folds onto I's red cell
        const bool lo = i == 0, hi = i == nx2 - 1;
        const int im = lo ? nx2 - 1 : i - 1, ip = hi ? 0 : i + 1;
        int fj[4], fk[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            fj[q] = tap(j, q, f.ny, f.py);
            fk[q] = tap(k, q, f.nz, f.pz);
        }
        T acc = T(0);
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const T* plane = t + (long long)fk[a] * f.ny * nx2;
#pragma unroll
            for (int b = 0; b < 4; b++) {
                const T wt = T((a == 0 || a == 3 ? 0.25 : 0.75) * (b == 0 || b == 3 ? 0.25 : 0.75) * 0.125);
                const T* row = plane + fj[b] * nx2;
                const bool o = ((fj[b] + fk[a]) & 1) != 0;
                const bool end = !f.px && (o ? lo : hi), fold = !f.px && (o ? hi : lo);
                acc = fma(fold ? wt : T(0.75) * wt, row[i], acc);
                acc = fma(end ? T(0) : T(0.25) * wt, row[o ? im : ip], acc);
            }
        }
        rc[c] = acc;
    }
}

// zf += P ec at the cells of colour col (see k_prolong_add).
__global__ void __launch_bounds__(256) k_correct_pair(Dims f, Dims cd, const double* __restrict__ ec, double* zf,
                                                      int col) {
    Dims h = f;
    h.nx = f.nx >> 1;
    h.n = f.n >> 1;
    auto other = [](int I, int up, int n, int per) {
        int v = up ? I + 1 : I - 1;
        if (v < 0) v = per ? n - 1 : I;
        if (v >= n) v = per ? 0 : I;
        return v;
    };
    COL_BEGIN(h)
        const int o = ((j + k) & 1) ^ col;
        const int i1 = other(i, o, cd.nx, cd.px);
        const int j0 = j >> 1, j1 = other(j0, j & 1, cd.ny, cd.py);
        const int k0 = k >> 1, k1 = other(k0, k & 1, cd.nz, cd.pz);
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const double wt = ((q & 1) ? 0.25 : 0.75) * ((q & 2) ? 0.25 : 0.75);
            const long long row = ((long long)((q & 2) ? k1 : k0) * cd.ny + ((q & 1) ? j1 : j0)) * cd.nx;
            acc = fma(0.75 * wt, ec[row + i], acc);
            acc = fma(0.25 * wt, ec[row + i1], acc);
        }
        zf[2 * c + o] += acc;
    }
}

// p_out = z + beta p_in;  q = A p_out;  <p_out, q> (see k_cg_p_matvec).
__global__ void __launch_bounds__(256) k_pq_pair(Dims d, Op<double> A, const double* __restrict__ z,
                                                 const double* __restrict__ p_in, double* __restrict__ p_out,
                                                 double* __restrict__ q, RedArgs ra) {
    const double beta = ra.sc[S_BETA];
    const WalkP w = walkp_of(d);
    DotAcc<double> da;
    if (w.k0 < w.k1) {
        auto P = [&](long long i) {
            const double2 a = ld2(z, i), b = ld2(p_in, i);
            return make_double2(fma(beta, b.x, a.x), fma(beta, b.y, a.y));
        };
        auto P1 = [&](long long i) { return fma(beta, p_in[i], z[i]); };
        long long p = (long long)w.k0 * w.nxy;
        double2 pc = P(p + w.c), pd = P(p + w.c + zdn(d, w.k0, w.nxy)), wzc = ld2(A.wz, p + w.c);
        for (int k = w.k0; k < w.k1; k++) {
            const long long up = zup(d, k, w.nxy);
            const bool has_zu = k < d.nz - 1 || d.pz;
            const double2 pu = P(p + w.c + up);
            double2 wzu = ld2(A.wz, p + w.c + up);
            const double2 wx = ld2(A.wx, p + w.c), wy = ld2(A.wy, p + w.c), m = ld2(A.m, p + w.c);
            double2 wyu = ld2(A.wy, p + w.yp);
            if (!w.has_yp) wyu = make_double2(0.0, 0.0);
            const double2 wu = has_zu ? wzu : make_double2(0.0, 0.0);
            const double2 ym = P(p + w.ym), yp = P(p + w.yp);
            double L = __shfl_up_sync(FULL, pc.y, 1), R = __shfl_down_sync(FULL, pc.x, 1);
            double wr = __shfl_down_sync(FULL, wx.x, 1);
            if (w.load_l) L = P1(p + w.xl + 1);
            if (w.load_r) {
                R = P1(p + w.xr);
                wr = w.has_xr ? A.wx[p + w.xr] : 0.0;
            }
            double2 qv;
            qv.x = m.x * pc.x;
            qv.y = m.y * pc.y;
            const double dx = pc.x - pc.y;
            qv.x = fma(wx.x, pc.x - L, qv.x);
            qv.x = fma(wx.y, dx, qv.x);
            qv.y = fma(-wx.y, dx, qv.y);
            qv.y = fma(wr, pc.y - R, qv.y);
            qv.x = fma(wy.x, pc.x - ym.x, qv.x);
            qv.y = fma(wy.y, pc.y - ym.y, qv.y);
            qv.x = fma(wyu.x, pc.x - yp.x, qv.x);
            qv.y = fma(wyu.y, pc.y - yp.y, qv.y);
            qv.x = fma(wzc.x, pc.x - pd.x, qv.x);
            qv.y = fma(wzc.y, pc.y - pd.y, qv.y);
            qv.x = fma(wu.x, pc.x - pu.x, qv.x);
            qv.y = fma(wu.y, pc.y - pu.y, qv.y);
            if (w.valid) {
                *reinterpret_cast<double2*>(p_out + p + w.c) = pc;
                *reinterpret_cast<double2*>(q + p + w.c) = qv;
                da.add(pc.x, qv.x);
                da.add(pc.y, qv.y);
            }
            pd = pc;
            pc = pu;
            wzc = wzu;
            p += w.nxy;
        }
    }
    double acc[1] = {da.value()};
    const bool mx[1] = {false};
    grid_reduce<1>(acc, mx, ra);
}

// ---------------------------------------------------------------- launchers

// Blocks of 256 threads; planes per chunk: 4 (a chunk's first plane reads
// three planes), fewer while a level has fewer than two blocks per SM.
static ColShape shape_pair(const Dims& d) {
    Dims h = d;
    h.nx = d.nx >> 1;
    const int lanes = row_lanes(h);
    const ColShape one = col_shape(h, 256, 1, lanes);
    const long long xy = (long long)one.grid.x * one.grid.y;
    long long blocks = xy * ((d.nz + 3) / 4);
    if (blocks < 152 * 2) blocks = xy * d.nz < 152 * 2 ? xy * d.nz : 152 * 2;
    if (blocks > RED_MAX_BLOCKS) blocks = RED_MAX_BLOCKS;
    return col_shape(h, 256, (int)blocks, lanes);
}

bool pair_ok(const Dims& d) { return d.nx % 2 == 0; }

void launch_zero_pair(const Dims& d, Op<double> A, const double* r, double* z, cudaStream_t s) {
    const ColShape sh = shape_pair(d);
    k_zero_pair<<<sh.grid, sh.block, 0, s>>>(d, A, r, z);
}
void launch_residual_pair(const Dims& d, Op<double> A, const double* z, double* res, cudaStream_t s) {
    const ColShape sh = shape_pair(d);
    k_sweep_pair<true, false><<<sh.grid, sh.block, 0, s>>>(d, A, nullptr, const_cast<double*>(z), res, 0, RedArgs{});
}
template <class T>
void launch_restrict_pair(const Dims& f, const Dims& c, const T* res, T* rc, cudaStream_t s) {
    const ColShape sh = col_shape(c, 128, 152 * 16);
    k_restrict_pair<T><<<sh.grid, sh.block, 0, s>>>(f, c, res, rc);
}
template void launch_restrict_pair<float>(const Dims&, const Dims&, const float*, float*, cudaStream_t);
template void launch_restrict_pair<double>(const Dims&, const Dims&, const double*, double*, cudaStream_t);
void launch_correct_pair(const Dims& f, const Dims& c, const double* ec, double* z, int col, cudaStream_t s) {
    Dims h = f;
    h.nx = f.nx >> 1;
    const ColShape sh = col_shape(h);
    k_correct_pair<<<sh.grid, sh.block, 0, s>>>(f, c, ec, z, col);
}
void launch_colour_pair(const Dims& d, Op<double> A, const double* r, double* z, int col, const RedArgs* dot,
                        cudaStream_t s) {
    const ColShape sh = shape_pair(d);
    if (dot) k_sweep_pair<false, true><<<sh.grid, sh.block, 0, s>>>(d, A, r, z, nullptr, col, *dot);
    else k_sweep_pair<false, false><<<sh.grid, sh.block, 0, s>>>(d, A, r, z, nullptr, col, RedArgs{});
}
void launch_pq_pair(const Dims& d, Op<double> A, const double* z, const double* p_in, double* p_out, double* q,
                    const RedArgs& ra, cudaStream_t s) {
    const ColShape sh = shape_pair(d);
    k_pq_pair<<<sh.grid, sh.block, 0, s>>>(d, A, z, p_in, p_out, q, ra);
}

}  // namespace fld
