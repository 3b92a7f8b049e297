"""FP64 draws, coefficients and pairs of csrc/ compiled for the host: the
same source as the kernels' (host_cuda/cuda_runtime.h stands in for CUDA), so
that rare values can be fed to it without a GPU."""
import ctypes
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SHIM = r"""
#include <thread>
#include <vector>
#include "mlkd_warp_pair.cuh"
using namespace mlkd;
// -ln u, nu and chi of the uniforms n1, n2, n3 (2^-B units), and the unit
// coefficients of a phase of length s with that nu
template <int B> static void draw1(const uint64_t *n, double s, double *out)
{
    const DrawFixed d = draw_fixed<B>(n[0], n[1], n[2], 1);
    const Background<double>::Unit u = Background<double>::kd_unit<true>(fx::pos_of(s), d.nu * d.nu);
    out[0] = d.nu_(), out[1] = d.chi_(), out[2] = fx::to_double(d.E), out[3] = u.D, out[4] = u.om, out[5] = u.beta;
}
extern "C" void draws(int B, const uint64_t *n, const double *s, int64_t count, double *out)
{
    init_draw_tables<double>();
    for (int64_t i = 0; i < count; ++i)
        B == 53 ? draw1<53>(n + 3 * i, s[i], out + 6 * i) : draw1<24>(n + 3 * i, s[i], out + 6 * i);
}
// the unit coefficients of phases of length s with normal variates nu
extern "C" void units(const double *s, const double *nu, int64_t count, double *out)
{
    for (int64_t i = 0; i < count; ++i) {
        const fx::Pos p = fx::pos_of(nu[i]);
        const Background<double>::Unit u = Background<double>::kd_unit<true>(fx::pos_of(s[i]), p * p);
        out[4 * i] = u.D, out[4 * i + 1] = u.om, out[4 * i + 2] = u.beta, out[4 * i + 3] = u.hs;
    }
}
// a, d, h(s) and om of kd_coeffs (the heterogeneous pairs) for R = sigma = 1, mu = 0
extern "C" void het_units(const double *s, const double *nu, int64_t count, double *out)
{
    Background<double> bg;
    bg.R = bg.invR = bg.sigma = 1.0, bg.mu = 0.0, bg.two_c2 = 2.0;
    for (int64_t i = 0; i < count; ++i) bg.kd_coeffs(s[i], nu[i], out[4 * i], out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
}

struct Least {
    double least = 1.0;
    void coarse(double, double E, double) { least = E < least ? E : least; }
};
struct Problem {
    double R, mu, sigma, dt;
    int32_t n, M, level;
    uint32_t request;
    uint64_t seed;
};
static LevelCtx<double> level_ctx(const Problem &p, PhiloxKeys &keys)
{
    LevelCtx<double> L;
    L.bg.R = p.R, L.bg.invR = 1.0 / p.R, L.bg.mu = p.mu, L.bg.sigma = p.sigma;
    L.bg.dt = p.dt, L.bg.Rdt = p.R * p.dt, L.bg.inv_Rdt = 1.0 / (p.R * p.dt);
    L.bg.c = p.sigma / p.R, L.bg.c_lo = std::fma(-L.bg.c, p.R, p.sigma) / p.R;
    L.n = p.n, L.M = p.M, L.init = 0, L.word2 = (uint32_t)p.level << 24, L.request = p.request;
    L.divM.init(p.M);
    for (int r = 0; r < 10; ++r) {
        keys.k0[r] = (uint32_t)p.seed + (uint32_t)r * 0x9E3779B9u;
        keys.k1[r] = (uint32_t)(p.seed >> 32) + (uint32_t)r * 0xBB67AE85u;
    }
    return L;
}
// positions at T and events of coupled pairs from the origin, and the
// smallest coarse optical length E~ met
template <int RECIPE>
static double run(const Problem &p, uint64_t first, int64_t count, double *xf, double *xc, int32_t *kf, int32_t *kc)
{
    PhiloxKeys keys;
    const LevelCtx<double> L = level_ctx(p, keys);
    Least tr;
    init_draw_tables<double>();
    for (int64_t i = 0; i < count; ++i) {
        PairState<double> st;
        bool done = pair_start<double, 1, RECIPE>(st, first + (uint64_t)i, L, keys, true);
        while (!done) done = pair_event<double, 1, RECIPE, Least>(st, L, keys, true, &tr);
        pair_drift<double, 1>(st, L, true);
        xf[i] = st.xf, xc[i] = st.xc, kf[i] = (int32_t)st.k, kc[i] = (int32_t)st.evc;
    }
    return tr.least;
}
extern "C" double pairs(int u24, const Problem *p, uint64_t first, int64_t count, double *xf, double *xc, int32_t *kf,
                        int32_t *kc)
{
    return u24 ? run<1>(*p, first, count, xf, xc, kf, kc) : run<0>(*p, first, count, xf, xc, kf, kc);
}
// the same pairs, each by a warp; a pair that takes more than `most` steps is
// left there with kf = -1
template <int RECIPE>
static void run_warps(const Problem &p, uint64_t first, int64_t count, int most, double *xf, double *xc, int32_t *kf, int32_t *kc)
{
    PhiloxKeys keys;
    const LevelCtx<double> L = level_ctx(p, keys);
    init_draw_tables<double>();
    pthread_barrier_init(&host_warp, nullptr, 32);
    std::vector<std::thread> lanes;
    for (int lane = 0; lane < 32; ++lane)
        lanes.emplace_back([&, lane] {
            host_lane = lane;
            for (int64_t i = 0; i < count; ++i) {
                PairState<double> st;
                bool done = pair_start<double, 1, RECIPE>(st, first + (uint64_t)i, L, keys, true);
                int steps = 0;
                while (!done && steps < most) {
                    done = warp_pair_step<double, RECIPE>(st, L, keys, true, lane);
                    ++steps;
                }
                pair_drift<double, 1>(st, L, true);
                if (lane == 0) xf[i] = st.xf, xc[i] = st.xc, kf[i] = done ? (int32_t)st.k : -1, kc[i] = (int32_t)st.evc;
            }
        });
    for (auto &t : lanes) t.join();
    pthread_barrier_destroy(&host_warp);
}
extern "C" void warp_pairs(int u24, const Problem *p, uint64_t first, int64_t count, int most, double *xf, double *xc,
                           int32_t *kf, int32_t *kc)
{
    if (u24) run_warps<1>(*p, first, count, most, xf, xc, kf, kc);
    else run_warps<0>(*p, first, count, most, xf, xc, kf, kc);
}
"""


class Problem(ctypes.Structure):
    _fields_ = [("R", ctypes.c_double), ("mu", ctypes.c_double), ("sigma", ctypes.c_double), ("dt", ctypes.c_double),
                ("n", ctypes.c_int32), ("M", ctypes.c_int32), ("level", ctypes.c_int32), ("request", ctypes.c_uint32),
                ("seed", ctypes.c_uint64)]


def build(folder):
    src, so = os.path.join(folder, "shim.cpp"), os.path.join(folder, "shim.so")
    with open(src, "w") as fh:
        fh.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fwrapv", "-pthread", "-shared", "-fPIC", "-I", os.path.join(HERE, "host_cuda"),
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2004_04071_gb300", "csrc"), src,
                    "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.draws.restype = lib.warp_pairs.restype = lib.units.restype = lib.het_units.restype = None
    lib.pairs.restype = ctypes.c_double
    return lib


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def draws(lib, B, n, s):
    """(nu, chi, E, D, om, beta) of the uniforms n[:, 3] 2^-B and phases of length s."""
    n = np.ascontiguousarray(n, np.uint64)
    s = np.ascontiguousarray(np.broadcast_to(np.asarray(s, np.float64), len(n)))
    out = np.zeros((len(n), 6))
    lib.draws(B, ptr(n), ptr(s), ctypes.c_int64(len(n)), ptr(out))
    return out.T


def units(lib, s, nu, het=False):
    """(D, om, beta, h) of kd_unit, or (a, d, h, om) of kd_coeffs."""
    out = np.zeros((len(s), 4))
    (lib.het_units if het else lib.units)(ptr(s), ptr(nu), ctypes.c_int64(len(s)), ptr(out))
    return out.T


def problem(d, level):
    return Problem(1.0 / (d["eps"] * d["eps"]), 0.0, 1.0 / d["eps"], d["dt0"] / d["M"] ** level,
                   int(round(d["T"] / d["dt0"])) * d["M"] ** level, d["M"], level, 0, d["seed"])


def pairs(lib, d, level, first, count, u24=False, warp=0):
    """xf, xc, kf, kc of coupled pairs of the free-space problem d, and the
    smallest E~; warp: one pair per warp, that many steps at most."""
    xf, xc = np.zeros(count), np.zeros(count)
    kf, kc = np.zeros(count, np.int32), np.zeros(count, np.int32)
    at = (ctypes.byref(problem(d, level)), ctypes.c_uint64(first), ctypes.c_int64(count))
    if warp:
        lib.warp_pairs(int(u24), *at, warp, ptr(xf), ptr(xc), ptr(kf), ptr(kc))
        return xf, xc, kf, kc, None
    least = lib.pairs(int(u24), *at, ptr(xf), ptr(xc), ptr(kf), ptr(kc))
    return xf, xc, kf, kc, least


# (eps, pair, 24-bit stream) of level 6 of BOUNDARY: E / (R dt) of one of the
# pair's first events is below a whole number by less than FP64 resolves
BOUNDARY = dict(T=1.0, dt0=0.5, M=2, L=6, seed=59, qoi=0, init=0)
AT_BOUNDARY = [(float.fromhex(e), pair, u24) for e, pair, u24 in (
    ("0x1.5ab3fced1e871p-4", 1, False), ("0x1.ea4fec05af416p-4", 1, False), ("0x1.0608ee7b3f7a3p-3", 5, False),
    ("0x1.c784eeb88ed90p-4", 7, False), ("0x1.5f18e07268fccp-4", 9, False), ("0x1.e40e71800ea5ap-4", 2, True),
    ("0x1.cd1257f72e48cp-4", 4, True), ("0x1.b79b2aeed81c9p-4", 10, True), ("0x1.cc76e56447539p-4", 17, True))]

# (eps, pair, 24-bit stream) of level 2 of FLIGHTS: a fine flight ends at a
# coarse step's end, and E is below that many times R dt by an ulp
FLIGHTS = dict(T=1.0, dt0=0.5, M=8, L=2, seed=59, qoi=0, init=0)
AT_COARSE_END = [(float.fromhex(e), pair, u24) for e, pair, u24 in (
    ("0x1.7c9c195fd5b89p-3", 4, False), ("0x1.66eea40163041p-3", 6, False), ("0x1.89c447c373d0fp-3", 8, False),
    ("0x1.8c8140f251fe6p-3", 15, False), ("0x1.47dc91b20357bp-3", 26, False), ("0x1.3a6d4cc372c57p-3", 2, True),
    ("0x1.5a7f45cc71943p-3", 4, True), ("0x1.16666c0a0a363p-3", 7, True), ("0x1.4bce96d5cd39dp-2", 29, True))]
