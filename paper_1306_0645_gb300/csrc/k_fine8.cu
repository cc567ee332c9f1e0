// k_fine8.cu -- the V-cycle's sweeps with one colour at a time in memory
// ("red/black compressed"): FP32 vectors, bfloat16 coefficients, one sweep
// down and one up, levels whose x extent is a multiple of 8.
//
// Each pair of cells (2m, 2m + 1) along x holds one red and one black cell,
// so the red (black) values of a level are n / 2 floats, cell l at l >> 1.  A
// thread owns eight cells of a row, four of each colour: one float4 per
// compressed array.  Of a cell's six neighbours, all of the other colour, the
// four in y and z have the same pair index, so they are whole aligned float4
// of the other colour's array; the two in x are the thread's own float4 and
// one value of the adjacent lane.
//
// What a cycle then moves on a level, per cell: the first sweep reads r and
// the coefficients and writes both colours compressed (16 bytes); the residual
// reads the black values and the weights (10); the correction is added to the
// red values alone, since the black sweep replaces the black ones (4.5); the
// black sweep reads red, r and the coefficients and writes black (16); the red
// sweep reads black, r and the coefficients and writes z in natural order
// (18).  With z in natural order throughout (k_fine4.cu) it was 16, 12, 8.5,
// 18 and 18, with half of every loaded neighbour vector unused and twice the
// load instructions per cell; those sweeps ran at 0.60 to 0.71 of the copy
// rate, bound by load latency and issue, not by bytes.
//
// Registers: at their launch bounds (three or four blocks per SM) the first
// sweep takes 80 and spills 22 words, the residual and the black sweep 64 and
// spill 12 and 13, the red sweep 80 and spills one with <r, z>; other bounds
// were not measured.  At 320^3 (512^3) the first sweep runs at 0.63 (0.79) of
// the copy rate, the black sweep at 0.80 (0.94).
//
// Every value is formed by the operations of k_fine4.cu in the same order, so
// the cycle is theirs up to which products the compiler contracts.
#include "walk4.cuh"

namespace fld {

namespace {

struct Walk8 {
    int i8, j, k0, k1, nx8;
    bool valid;
    long long nxy;
};

__device__ __forceinline__ Walk8 walk8_of(const Dims& d) {
    Walk8 w;
    w.nx8 = d.nx >> 3;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    w.valid = i < w.nx8 && j < d.ny;
    w.i8 = min(i, w.nx8 - 1);
    w.j = min(j, d.ny - 1);
    const int kch = (d.nz + (int)gridDim.z - 1) / (int)gridDim.z;
    w.k0 = (int)blockIdx.z * kch;
    w.k1 = min(d.nz, w.k0 + kch);
    w.nxy = (long long)d.nx * d.ny;
    return w;
}

// What does not change along the walk: in-plane offsets of the thread's cells
// and of the rows beside it, and which x neighbours the adjacent lane holds.
struct Row8 {
    int c, ym, yp;       // first cell, and the same cell of rows j -+ 1, within a plane
    int xl, xr;          // pair index, within a plane, of the far black/red values at the row's ends
    int xw;              // first cell of the next vector (for its lower face weight)
    bool has_xr, has_yp, load_l, load_r;
};

__device__ __forceinline__ Row8 row8_of(const Dims& d, const Walk8& w) {
    Row8 g;
    const int row = w.j * d.nx;      // a plane holds at most 2^22 cells
    const int i0 = 8 * w.i8;
    g.c = row + i0;
    g.ym = w.j > 0 ? g.c - d.nx : (d.py ? g.c + (d.ny - 1) * d.nx : g.c);
    g.has_yp = w.j < d.ny - 1 || d.py;
    g.yp = w.j < d.ny - 1 ? g.c + d.nx : (d.py ? g.c - (d.ny - 1) * d.nx : g.c);
    const bool first = i0 == 0, last = i0 + 8 >= d.nx;
    g.xl = (first ? (d.px ? row + d.nx - 2 : g.c) : g.c - 2) >> 1;
    g.xr = (last ? (d.px ? row : g.c + 6) : g.c + 8) >> 1;
    g.xw = last ? row : g.c + 8;
    g.has_xr = !last || d.px;
    g.load_l = threadIdx.x == 0 || first;
    g.load_r = threadIdx.x == blockDim.x - 1 || last;
    return g;
}

__device__ __forceinline__ uint4 ldc8(const unsigned short* __restrict__ p, long long i) {
    return __ldg(reinterpret_cast<const uint4*>(p + i));
}
// FP32 value of the even (o = 0) or odd cell's bfloat16 in a pair's word;
// sel = pick(o)
__device__ __forceinline__ unsigned pick(int o) { return o ? 0x3244u : 0x1044u; }
__device__ __forceinline__ float half_of(unsigned word, unsigned sel) {
    return __uint_as_float(__byte_perm(word, 0u, sel));
}
__device__ __forceinline__ float4 halves(uint4 v, unsigned sel) {
    return make_float4(half_of(v.x, sel), half_of(v.y, sel), half_of(v.z, sel), half_of(v.w, sel));
}
// the even or odd cells of eight FP32 values
__device__ __forceinline__ float4 evens(float4 a, float4 b, int o) {
    return o ? make_float4(a.y, a.w, b.y, b.w) : make_float4(a.x, a.z, b.x, b.z);
}

// The six face weights of the four cells at parity o: the lower ones their
// own, the upper ones the next cell's along x, row j + 1's and plane k + 1's.
struct Faces8 {
    float4 xl, xu, yl, yu, zl, zu;
};
__device__ __forceinline__ Faces8 faces8(const unsigned short* __restrict__ wx, const Row8& g, long long plane,
                                         uint4 wxc, uint4 wyc, uint4 wyp, uint4 wzc, uint4 wzu, bool has_zu, int o) {
    Faces8 f;
    const unsigned s = pick(o);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    f.xl = halves(wxc, s);
    // rows of both parities share a warp where a row is shorter than it: every
    // lane takes part in the shuffle
    const unsigned nx = __shfl_down_sync(FULL, wxc.x, 1);
    if (o) {
        float last = 0.0f;
        if (g.has_xr) last = g.load_r ? __uint_as_float((unsigned)wx[plane + g.xw] << 16) : half_of(nx, pick(0));
        f.xu = make_float4(half_of(wxc.y, pick(0)), half_of(wxc.z, pick(0)), half_of(wxc.w, pick(0)), last);
    } else {
        f.xu = halves(wxc, pick(1));
    }
    f.yl = halves(wyc, s);
    f.yu = g.has_yp ? halves(wyp, s) : zero;
    f.zl = halves(wzc, s);
    f.zu = has_zu ? halves(wzu, s) : zero;
    return f;
}

// lower and upper x neighbours of the four cells at parity o, v the other
// colour's values of the same pairs and far the one beyond them
struct XNbr8 {
    float4 lo, up;
};
__device__ __forceinline__ XNbr8 xnbr8(float4 v, float far, int o) {
    XNbr8 x;
    if (o) {
        x.lo = v;
        x.up = make_float4(v.y, v.z, v.w, far);
    } else {
        x.lo = make_float4(far, v.x, v.y, v.z);
        x.up = v;
    }
    return x;
}
// (uniform in a row; the shuffles are executed by every lane of the warp)
__device__ __forceinline__ float far8(float4 v, int o) {
    const float l = __shfl_up_sync(FULL, v.w, 1);
    const float r = __shfl_down_sync(FULL, v.x, 1);
    return o ? r : l;
}

__device__ __forceinline__ void st4s(float* p, long long i, float4 v) { *reinterpret_cast<float4*>(p + i) = v; }

}  // namespace

// ---------------------------------------------------------- first sweep

// z of one red/black sweep from zero: red r * invd, black
// invd (r + sum_f w_f z_red), both compressed.  A plane's red values are the
// z neighbours of the next plane's black cells, so each is formed once along
// the walk; the rows beside the thread's are formed again from r and invd,
// which the neighbouring threads stream.
__global__ void __launch_bounds__(256, 3) k_zero8(Dims d, Op<unsigned short> A, const float* __restrict__ r,
                                                  float* __restrict__ zr, float* __restrict__ zb, int pf) {
    const Walk8 w = walk8_of(d);
    if (w.k0 >= w.k1) return;
    const Row8 g = row8_of(d, w);
    const unsigned short* __restrict__ invd = A.invd;
    // r * invd at the cells of parity o of the vector at i
    auto U = [&](long long i, int o) {
        const float4 v = evens(ld4(r, i), ld4(r, i + 4), o), q = halves(ldc8(invd, i), pick(o));
        return make_float4(v.x * q.x, v.y * q.y, v.z * q.z, v.w * q.w);
    };
    long long p = (long long)w.k0 * w.nxy;
    int o = 1 - ((w.j + w.k0) & 1);      // parity of the black cells of this row and plane
    // in plane k -+ 1 the cells at parity o are red
    float4 ud = U(p + g.c + zdn(d, w.k0, w.nxy), o);
    float4 ra = ld4(r, p + g.c), rb = ld4(r, p + g.c + 4);
    uint4 iv = ldc8(invd, p + g.c);
    uint4 wzc = ldc8(A.wz, p + g.c);
    for (int k = w.k0; k < w.k1; k++) {
        const long long ahead = p + g.c + (long long)pf * w.nxy;
        if (pf_here(k, pf, w.k1)) {
            pf2(A.wx, ahead);
            pf2(A.wy, ahead);
        }
        if (pf_above(k, pf, w.k1, d.nz)) {
            pf2(r, ahead + w.nxy);
            pf2(invd, ahead + w.nxy);
            pf2(A.wz, ahead + w.nxy);
        }
        const long long up = zup(d, k, w.nxy);
        const bool has_zu = k < d.nz - 1 || d.pz;
        const float4 na = ld4(r, p + g.c + up), nb = ld4(r, p + g.c + up + 4);
        const uint4 ni = ldc8(invd, p + g.c + up);
        const uint4 wzu = ldc8(A.wz, p + g.c + up);
        const Faces8 f = faces8(A.wx, g, p, ldc8(A.wx, p + g.c), ldc8(A.wy, p + g.c), ldc8(A.wy, p + g.yp), wzc, wzu,
                                has_zu, o);
        // red values of this row (parity 1 - o), of rows j -+ 1 and of plane k + 1 (parity o)
        float4 rv = evens(ra, rb, 1 - o), q = halves(iv, pick(1 - o));
        const float4 uc = make_float4(rv.x * q.x, rv.y * q.y, rv.z * q.z, rv.w * q.w);
        const float4 ym = U(p + g.ym, o), yp = U(p + g.yp, o);
        rv = evens(na, nb, o);
        q = halves(ni, pick(o));
        const float4 uu = make_float4(rv.x * q.x, rv.y * q.y, rv.z * q.z, rv.w * q.w);
        float far = far8(uc, o);
        if (o ? g.load_r : g.load_l) {
            const long long pair = (p >> 1) + (o ? g.xr : g.xl);
            const long long c = 2 * pair + 1 - o;
            far = r[c] * __uint_as_float((unsigned)invd[c] << 16);
        }
        const XNbr8 x = xnbr8(uc, far, o);
        const float4 rc = evens(ra, rb, o), iq = halves(iv, pick(o));
        float4 b;
#define B1(X)                                                                                              \
        b.X = iq.X * (rc.X + f.xl.X * x.lo.X + f.xu.X * x.up.X + f.yl.X * ym.X + f.yu.X * yp.X + f.zl.X * ud.X + \
                      f.zu.X * uu.X);
        B1(x) B1(y) B1(z) B1(w)
#undef B1
        if (w.valid) {
            st4s(zr, (p + g.c) >> 1, uc);
            st4s(zb, (p + g.c) >> 1, b);
        }
        ud = uc;
        ra = na;
        rb = nb;
        iv = ni;
        wzc = wzu;
        p += w.nxy;
        o ^= 1;
    }
}

// ------------------------------------------- sweeps from the other colour

// u: the other colour's values (compressed).  At the cells of colour col:
//  S_RES    out = sum_f w_f u                    (compressed; the residual at
//           red cells after a zero-guess sweep, see k_residual4)
//  S_SWEEP  out = invd (r + sum_f w_f u)         (compressed)
//  S_FINAL  the same, z written in natural order with u at the other cells;
//           with DOT also <r, z>
enum Sweep8 { S_RES, S_SWEEP, S_FINAL };
template <int MODE, bool DOT>
__global__ void __launch_bounds__(256, MODE == S_FINAL ? 3 : 4)
    k_sweep8(Dims d, Op<unsigned short> A, const float* __restrict__ r, const float* __restrict__ u,
             float* __restrict__ out, int col, RedArgs ra, int pf) {
    const Walk8 w = walk8_of(d);
    DotAcc<float> da;
    if (w.k0 < w.k1) {
        const Row8 g = row8_of(d, w);
        long long p = (long long)w.k0 * w.nxy;
        int o = ((w.j + w.k0) & 1) ^ col;
        float4 uc = ld4(u, (p + g.c) >> 1);
        float4 ud = ld4(u, (p + g.c + zdn(d, w.k0, w.nxy)) >> 1);
        uint4 wzc = ldc8(A.wz, p + g.c);
        for (int k = w.k0; k < w.k1; k++) {
            const long long ahead = p + g.c + (long long)pf * w.nxy;
            if (pf_here(k, pf, w.k1)) {
                if (MODE != S_RES) {
                    pf2(r, ahead);
                    pf2(A.invd, ahead);
                }
                pf2(A.wx, ahead);
                pf2(A.wy, ahead);
            }
            if (pf_above(k, pf, w.k1, d.nz)) {
                pf2(u, (ahead + w.nxy) >> 1);
                pf2(A.wz, ahead + w.nxy);
            }
            const long long up = zup(d, k, w.nxy);
            const bool has_zu = k < d.nz - 1 || d.pz;
            const float4 uu = ld4(u, (p + g.c + up) >> 1);
            const uint4 wzu = ldc8(A.wz, p + g.c + up);
            const Faces8 f = faces8(A.wx, g, p, ldc8(A.wx, p + g.c), ldc8(A.wy, p + g.c), ldc8(A.wy, p + g.yp), wzc,
                                    wzu, has_zu, o);
            const float4 ym = ld4(u, (p + g.ym) >> 1), yp = ld4(u, (p + g.yp) >> 1);
            float far = far8(uc, o);
            if (o ? g.load_r : g.load_l) far = u[(p >> 1) + (o ? g.xr : g.xl)];
            const XNbr8 x = xnbr8(uc, far, o);
            float4 b;
            if (MODE == S_RES) {
#define R1(X)                                                                                                     \
                b.X = f.xl.X * x.lo.X + f.xu.X * x.up.X + f.yl.X * ym.X + f.yu.X * yp.X + f.zl.X * ud.X + f.zu.X * uu.X;
                R1(x) R1(y) R1(z) R1(w)
#undef R1
                if (w.valid) st4s(out, (p + g.c) >> 1, b);
            } else {
                const float4 r0 = ld4(r, p + g.c), r1 = ld4(r, p + g.c + 4);
                const float4 rc = evens(r0, r1, o), iq = halves(ldc8(A.invd, p + g.c), pick(o));
#define C1(X)                                                                                                      \
                b.X = iq.X * (rc.X + f.xl.X * x.lo.X + f.xu.X * x.up.X + f.yl.X * ym.X + f.yu.X * yp.X +           \
                              f.zl.X * ud.X + f.zu.X * uu.X);
                C1(x) C1(y) C1(z) C1(w)
#undef C1
                if (w.valid) {
                    if (MODE == S_SWEEP) {
                        st4s(out, (p + g.c) >> 1, b);
                    } else {
                        const float4 z0 = o ? make_float4(uc.x, b.x, uc.y, b.y) : make_float4(b.x, uc.x, b.y, uc.y);
                        const float4 z1 = o ? make_float4(uc.z, b.z, uc.w, b.w) : make_float4(b.z, uc.z, b.w, uc.w);
                        st4s(out, p + g.c, z0);
                        st4s(out, p + g.c + 4, z1);
                        if (DOT) {
                            da.add(r0.x, z0.x);
                            da.add(r0.y, z0.y);
                            da.add(r0.z, z0.z);
                            da.add(r0.w, z0.w);
                            da.add(r1.x, z1.x);
                            da.add(r1.y, z1.y);
                            da.add(r1.z, z1.z);
                            da.add(r1.w, z1.w);
                        }
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

// ------------------------------------------------------------- correction

// zr += P ec at the red cells (see k_prolong_add4): the thread's eight fine
// cells interpolate from coarse cells 4 i8 - 1 .. 4 i8 + 4 of rows J0 = j / 2
// and its neighbour towards j, and of planes K = k / 2 and its neighbour
// towards k; the raw rows of the window K - 1, K, K + 1 stay in registers.
__global__ void __launch_bounds__(256, 3) k_correct8(Dims f, Dims cd, const float* __restrict__ ec,
                                                     float* __restrict__ zr, int pf) {
    const Walk8 w = walk8_of(f);
    if (w.k0 >= w.k1) return;
    auto wrap = [](int v, int n, int periodic) {
        return v < 0 ? (periodic ? v + n : 0) : v >= n ? (periodic ? v - n : n - 1) : v;
    };
    const int I = 4 * w.i8;
    const int xm = wrap(I - 1, cd.nx, cd.px), xp = wrap(I + 4, cd.nx, cd.px);
    const bool load_l = threadIdx.x == 0 || I == 0;
    const bool load_r = threadIdx.x == blockDim.x - 1 || I + 4 >= cd.nx;
    const int J0 = w.j >> 1;
    const int J1 = wrap((w.j & 1) ? J0 + 1 : J0 - 1, cd.ny, cd.py);
    const long long cxy = (long long)cd.nx * cd.ny;
    struct Raw {
        float4 v;
        float l, r;
    };
    auto row = [&](int K, int J) {
        const long long b = (long long)K * cxy + (long long)J * cd.nx;
        Raw q;
        q.v = ld4(ec, b + I);
        q.l = __shfl_up_sync(FULL, q.v.w, 1);
        q.r = __shfl_down_sync(FULL, q.v.x, 1);
        if (load_l) q.l = ec[b + xm];
        if (load_r) q.r = ec[b + xp];
        return q;
    };
    // x step at the fine cells of parity o: 3/4 of coarse cell I + i, 1/4 of
    // the one below (o = 0) or above it
    auto xs = [](const Raw& q, int o) {
        const float4 v = q.v;
        const float4 n = o ? make_float4(v.y, v.z, v.w, q.r) : make_float4(q.l, v.x, v.y, v.z);
        return make_float4(fmaf(0.75f, v.x, 0.25f * n.x), fmaf(0.75f, v.y, 0.25f * n.y),
                           fmaf(0.75f, v.z, 0.25f * n.z), fmaf(0.75f, v.w, 0.25f * n.w));
    };
    int K = w.k0 >> 1;
    Raw am = row(wrap(K - 1, cd.nz, cd.pz), J0), bm = row(wrap(K - 1, cd.nz, cd.pz), J1);
    Raw a0 = row(K, J0), b0 = row(K, J1);
    Raw ap = row(wrap(K + 1, cd.nz, cd.pz), J0), bp = row(wrap(K + 1, cd.nz, cd.pz), J1);
    const float w0 = 0.75f * 0.75f, w1 = 0.25f * 0.75f, w2 = 0.75f * 0.25f, w3 = 0.25f * 0.25f;
    for (int k = w.k0; k < w.k1; k++) {
        if (k > w.k0 && (k & 1) == 0) {
            K = k >> 1;
            am = a0;
            bm = b0;
            a0 = ap;
            b0 = bp;
            ap = row(wrap(K + 1, cd.nz, cd.pz), J0);
            bp = row(wrap(K + 1, cd.nz, cd.pz), J1);
        }
        const long long h = ((long long)k * w.nxy + (long long)w.j * f.nx + 8 * w.i8) >> 1;
        if (pf_here(k, pf, w.k1)) pf2(zr, h + (((long long)pf * w.nxy) >> 1));
        const int o = (w.j + k) & 1;      // parity of the red cells
        const bool odd = (k & 1) != 0;
        const float4 A0 = xs(a0, o), B0 = xs(b0, o);
        const float4 A1 = xs(odd ? ap : am, o), B1 = xs(odd ? bp : bm, o);
        if (w.valid) {
            float4 z = ld4(zr, h);
#define P1(X) z.X = __fadd_rn(z.X, fmaf(w3, B1.X, fmaf(w2, A1.X, fmaf(w1, B0.X, w0 * A0.X))));
            P1(x) P1(y) P1(z) P1(w)
#undef P1
            st4s(zr, h, z);
        }
    }
}

// ---------------------------------------------------------------- launchers

// Levels the compressed sweeps take: eight cells per thread, and at least two
// threads per row.
bool fine8_ok(const Dims& d) { return d.nx % 8 == 0 && d.nx >= 16; }

static ColShape shape8(const Dims& d, const Tune& tn) {
    Dims h = d;
    h.nx = d.nx / 8;
    return sweep_shape(h, tn);
}

void launch_zero8(const Dims& d, Op<unsigned short> A, const float* r, float* zr, float* zb, cudaStream_t s,
                  const Tune& tn) {
    const ColShape sh = shape8(d, tn);
    k_zero8<<<sh.grid, sh.block, 0, s>>>(d, A, r, zr, zb, tn.pf);
}
void launch_residual8(const Dims& d, Op<unsigned short> A, const float* zb, float* res, cudaStream_t s,
                      const Tune& tn) {
    const ColShape sh = shape8(d, tn);
    k_sweep8<S_RES, false><<<sh.grid, sh.block, 0, s>>>(d, A, nullptr, zb, res, 0, RedArgs{}, tn.pf);
}
void launch_correct8(const Dims& f, const Dims& c, const float* ec, float* zr, cudaStream_t s, const Tune& tn) {
    const ColShape sh = shape8(f, tn);
    k_correct8<<<sh.grid, sh.block, 0, s>>>(f, c, ec, zr, tn.pf);
}
void launch_black8(const Dims& d, Op<unsigned short> A, const float* r, const float* zr, float* zb, cudaStream_t s,
                   const Tune& tn) {
    const ColShape sh = shape8(d, tn);
    k_sweep8<S_SWEEP, false><<<sh.grid, sh.block, 0, s>>>(d, A, r, zr, zb, 1, RedArgs{}, tn.pf);
}
void launch_red8(const Dims& d, Op<unsigned short> A, const float* r, const float* zb, float* z, const RedArgs* dot,
                 cudaStream_t s, const Tune& tn) {
    const ColShape sh = shape8(d, tn);
    if (dot) k_sweep8<S_FINAL, true><<<sh.grid, sh.block, 0, s>>>(d, A, r, zb, z, 0, *dot, tn.pf);
    else k_sweep8<S_FINAL, false><<<sh.grid, sh.block, 0, s>>>(d, A, r, zb, z, 0, RedArgs{}, tn.pf);
}

}  // namespace fld
