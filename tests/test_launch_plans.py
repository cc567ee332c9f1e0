"""Launch shapes, limits, prefetch ranges and sums of the library's sources on
the host: a small program with the library's own inline functions is compiled
and run here (no GPU)."""
import os
import subprocess

import pytest

from paper_1306_0645_gb300 import build

# Every plane a walk names (own plane, and one above it) must lie in the grid.
PREFETCH = r"""
for (int nz = 1; nz <= 70; nz++)
    for (int gz = 1; gz <= nz; gz++) {
        const int kch = (nz + gz - 1) / gz;
        for (int pf = 0; pf <= fld::TUNE_PF_MAX; pf++)
            for (int b = 0; b < gz; b++) {
                const int k0 = b * kch, k1 = nz < k0 + kch ? nz : k0 + kch;
                for (int k = k0; k < k1; k++) {
                    int top = -1;
                    if (fld::pf_here(k, pf, k1)) top = k + pf;
                    if (fld::pf_above(k, pf, k1, nz)) top = k + pf + 1;
                    if (top >= nz) return fail("plane", nz, gz, pf, k);
                    if (pf == 0 && top >= 0) return fail("prefetch off", nz, gz, pf, k);
                    // and every plane but the first pf + 1 of a chunk is named
                    if (pf > 0 && k + pf + 1 < k1 && top != k + pf + 1) return fail("missed", nz, gz, pf, k);
                }
            }
    }
"""

# Blocks of a stencil sweep: whole warps whatever the extents, the plane
# covered, no more blocks than the reductions hold partial sums for.
SHAPES = r"""
const int ny_[] = {1, 2, 3, 4, 5, 7, 8, 12, 16, 33, 96, 1000};
for (int nx = 1; nx <= 140; nx++)
    for (int ny : ny_)
        for (int nz : {1, 2, 3, 8, 30, 200})
            for (int threads : {32, 64, 128, 256})
                for (int lanes : {8, 16, 32}) {
                    fld::Dims d;
                    d.nx = nx; d.ny = ny; d.nz = nz; d.px = d.py = d.pz = 0;
                    d.n = (long long)nx * ny * nz;
                    const fld::ColShape s = fld::col_shape(d, threads, 152 * 8, lanes);
                    const int n = s.block.x * s.block.y * s.block.z;
                    if (n % 32 || n > threads) return fail("block", nx, ny, threads, n);
                    if ((int)(s.block.x * s.grid.x) < nx || (int)(s.block.y * s.grid.y) < ny)
                        return fail("plane", nx, ny, threads, lanes);
                    if ((long long)s.grid.x * s.grid.y * s.grid.z > fld::RED_MAX_BLOCKS || (int)s.grid.z > nz)
                        return fail("blocks", nx, ny, nz, threads);
                }
"""


# The shared-memory limits that the coarsest grid's launchers set, recorded in
# place of the runtime call (the launches themselves find no device).
RECORD = r"""
#include <map>
#include <cuda_runtime.h>
static std::map<const void*, int> g_limit;
static int g_lowered = 0;
template <class F>
static cudaError_t record_limit(F* f, cudaFuncAttribute, int bytes) {
    auto it = g_limit.emplace((const void*)f, bytes).first;
    if (it->second != bytes) g_lowered = 1;
    return cudaSuccess;
}
#define cudaFuncSetAttribute record_limit
#include "k_coarse.cu"
"""
LIMITS = r"""
for (int n : {64, 102, 125, 128, 130, 150, 160, 161, 300, 609, 693, 702, 760, 761, 854, 1024, 2048, 2049, 4096}) {
    fld::Dims d;
    d.nx = n; d.ny = d.nz = 1; d.px = d.py = d.pz = 0; d.n = n;
    for (bool fp32 : {false, true}) {
        fld::launch_coarse_setup<float>(d, fld::Op<float>{}, nullptr, nullptr, nullptr, nullptr, fp32, nullptr);
        if (g_lowered) return fail("limit depends on the call", n, fp32, 0, 0);
    }
    fld::launch_coarse_setup<double>(d, fld::Op<double>{}, nullptr, nullptr, nullptr, nullptr, false, nullptr);
    if (g_lowered) return fail("limit depends on the call", n, 2, 0, 0);
}
if (g_limit.empty()) return fail("no limit recorded", 0, 0, 0, 0);
"""

# The sum of 1024 threads' compensated pairs in the order of the one-CTA solve's
# block sum: exact up to the two roundings of value(), as FP64 additions are
# to a few (long double has 64 bits and more).
SUMS = r"""
unsigned long long x = 88172645463325252ull;
auto uniform = [&]() {
    x ^= x << 13; x ^= x >> 7; x ^= x << 17;
    return (double)(x >> 11) * (1.0 / 9007199254740992.0);
};
for (int trial = 0; trial < 400; trial++) {
    fld::DotSum v[1024];
    long double exact = 0.0L;
    for (auto& t : v) {
        const float hi = (float)(uniform() * uniform() * uniform());
        const float lo = (float)((uniform() - 0.5) * hi * 5.9e-8);
        t = fld::DotSum{hi, lo, 0.0f};
        exact += (long double)hi + (long double)lo;
    }
    for (int o = 1; o < 1024; o <<= 1)
        for (int q = 0; q < 1024; q += 2 * o) v[q].merge(v[q + o].hi, v[q + o].lo, v[q + o].c);
    const long double err = (long double)v[0].value() - exact;
    if ((err < 0 ? -err : err) > 2.3e-16L * exact) return fail("block sum", trial, (int)(err / exact * 1e18L), 0, 0);
}
"""

# Every tail that fld_create accepts (a coarsest grid of at most 4096 cells) has
# a plan within its shared memory; a coarsest grid beyond that has none and is
# reported, not launched.
TAILS = r"""
auto plan = [&](auto zero, const int (&c)[3], int nlev, int cluster, int sweeps, bool solve, int* bytes) {
    fld::TailArgs<decltype(zero)> a{};
    a.nlev = nlev;
    a.pre = sweeps < 2 ? 1 : sweeps - 2;
    a.post = sweeps < 2 ? 1 : 2;
    a.paper_order = sweeps == 1;
    for (int l = 0; l < nlev; l++) {
        fld::Dims& d = a.L[l].d;
        const int f = 1 << (nlev - 1 - l);
        d.nx = c[0] * f; d.ny = c[1] * f; d.nz = c[2] * f;
        d.n = (long long)d.nx * d.ny * d.nz;
    }
    const bool ok = fld::plan_tail(a, cluster, solve);
    *bytes = a.smem_bytes;
    return ok;
};
const int e[] = {1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 45, 64, 100, 128, 255, 512, 1000, 1024, 4096};
int bytes = 0;
for (int x : e)
    for (int y : e)
        for (int z : e) {
            const int c[3] = {x, y, z};
            if ((long long)x * y * z > 4096) continue;
            for (int nlev = 2; nlev <= 5 && ((long long)x * y * z << 3 * (nlev - 1)) <= (1 << 24); nlev++)
                for (int cluster : {8, 16})
                    for (int sweeps = 0; sweeps < 4; sweeps++) {
                        if (!plan(0.0f, c, nlev, cluster, sweeps, false, &bytes) || bytes > (int)fld::TAIL_SMEM_MAX)
                            return fail("FP32 tail", x, y, z, nlev);
                        if (!plan(0.0, c, nlev, cluster, sweeps, false, &bytes) || bytes > (int)fld::TAIL_SMEM_MAX)
                            return fail("FP64 tail", x, y, z, nlev);
                        if (plan(0.0f, c, nlev, cluster, sweeps, true, &bytes) && bytes > (int)fld::PS_SMEM_MAX)
                            return fail("one-CTA solve", x, y, z, nlev);
                    }
        }
const int big[3] = {32, 32, 32};
if (plan(0.0, big, 2, 16, 0, false, &bytes)) return fail("a coarsest grid that does not fit", 32, 32, 32, bytes);
"""


def run_host(tmp_path, body, head='#include "walk4.cuh"\n'):
    """Compiles body into a program with the library's code and runs it."""
    src = tmp_path / "plan.cu"
    src.write_text("#include <cstdio>\n" + head +
                   "static int fail(const char* what, int a, int b, int c, int d) {\n"
                   '    printf("%s: %d %d %d %d\\n", what, a, b, c, d);\n    return 1;\n}\n'
                   "int main() {\n" + body + "    return 0;\n}\n")
    exe = str(tmp_path / "plan")
    cmd = [build.nvcc()] + build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.INCLUDE, "-I",
                                         build.CSRC, str(src), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, r.stdout


def test_prefetched_planes_lie_in_the_grid(tmp_path):
    run_host(tmp_path, PREFETCH)


def test_sweep_blocks_are_whole_warps(tmp_path):
    run_host(tmp_path, SHAPES)


def test_shared_memory_limits_do_not_depend_on_the_call(tmp_path):
    # the limit belongs to the function, so a smaller one set by one thread
    # would refuse another thread's launch
    run_host(tmp_path, LIMITS, RECORD)


def test_block_sum_of_pairs_keeps_fp64_accuracy(tmp_path):
    run_host(tmp_path, SUMS)


def test_every_accepted_tail_has_a_plan(tmp_path):
    run_host(tmp_path, TAILS, '#include "k_tail.cu"\n')
