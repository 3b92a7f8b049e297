"""Writes mlkd_fixed_tables.h: the constants of the 64-bit fixed-point
functions of mlkd_fixed.h.

Every polynomial is evaluated in the form c0 - x (c1 - x (c2 - ...)) with all
c >= 0: its terms alternate.  The leading coefficients are 64-bit fractions;
from a term below 2^-29 on, the rest of the sum is a 32-bit fraction scaled by
2^shift.  Coefficients interpolate at the Chebyshev nodes of the range, in
50-digit arithmetic, with the degree chosen so that the largest error is below
2^-62 (log and sine/cosine use the plain Taylor terms).

    python paper_2004_04071_gb300/csrc/gen_fixed.py > mlkd_fixed_tables.h
"""
import mpmath as mp

mp.mp.dps = 50
TWO64 = mp.mpf(2) ** 64


def chebyshev_interpolant(f, hi, deg):
    """Monomial coefficients (lowest first) of the interpolant of f at the Chebyshev nodes of [0, hi]."""
    nodes = [hi * (1 + mp.cos(mp.pi * (k + mp.mpf(1) / 2) / (deg + 1))) / 2 for k in range(deg + 1)]
    V = mp.matrix([[x ** j for j in range(deg + 1)] for x in nodes])
    c = mp.lu_solve(V, mp.matrix([f(x) for x in nodes]))
    return [c[j] for j in range(deg + 1)]


def series(coef, n0, terms=70):
    return lambda s: mp.fsum(coef(n) * s ** (n - n0) for n in range(n0, n0 + terms))


def near_minimax(f, hi):
    for deg in range(6, 26):
        c = chebyshev_interpolant(f, hi, deg)
        err = max(abs(mp.polyval(list(reversed(c)), hi * i / 400) - f(hi * mp.mpf(i) / 400)) for i in range(401))
        if err < mp.mpf(2) ** -62:
            break
    assert all((-1) ** j * c[j] > 0 for j in range(deg + 1)), "terms do not alternate"
    return [abs(v) for v in c]


def emit(name, polys, what):
    """polys: (magnitudes of the alternating coefficients, lowest first; largest x) of
    polynomials that are evaluated together."""
    cut = max(next(j for j in range(len(c)) if c[j] * hi ** j < mp.mpf(2) ** -29) for c, hi in polys)
    print("// %s" % what)
    rows, tails = [], []
    for c, _ in polys:
        sh = int(mp.floor(-mp.log(c[cut], 2)))
        rows.append(["0x%016xull" % int(mp.nint(min(v * TWO64, TWO64 - 1))) for v in c[:cut]])
        t = [int(mp.nint(v * mp.mpf(2) ** (32 + sh))) for v in c[cut:]]
        while t[-1] == 0:
            t.pop()
        tails.append((sh, t))
    n = max(len(t) for _, t in tails)
    print("struct %s {" % name)
    print("    static constexpr int kLead = %d, kTail = %d;" % (cut, n))
    for i, (sh, t) in enumerate(tails):
        print("    static constexpr int kShift%d = %d;" % (i, sh))
        print("    static constexpr uint32_t tail%d[kTail] = {%s};" % (i, ", ".join("0x%08xu" % v for v in t + [0] * (n - len(t)))))
    print("};")
    print("MLKD_CONSTANT uint64_t k%s[%d][%d] = {" % (name, cut, len(polys)))
    print(",\n".join("    {" + ", ".join(r[j] for r in rows) + "}" for j in range(cut)) + "};")


def main():
    print("// Constants of mlkd_fixed.h, written by gen_fixed.py beside this file.")
    print("// MLKD_CONSTANT is defined there: constant memory on the device.")
    print("#pragma once\n#include <cstdint>\nnamespace mlkd {\nnamespace fx {")
    one = mp.mpf(1)
    H = series(lambda n: mp.mpf((-1) ** n) / mp.factorial(n), 2)
    F = series(lambda n: mp.mpf((-1) ** n * (2 - n)) / mp.factorial(n), 3)
    emit("PolyHF", [(near_minimax(lambda s: 2 * H(s), one), one), (near_minimax(F, one), one)],
         "2 h(s)/s^2, h(s) = exp(-s) + s - 1, and f(s)/s^3, f(s) = 2(exp(-s) - 1) + s(exp(-s) + 1), 0 <= s <= 1")
    hmax = mp.mpf("0.368")
    emit("PolyW", [(near_minimax(lambda h: mp.sqrt(2 * H(h)), hmax), hmax)],
         "sqrt(2 (exp(-h) + h - 1))/h, 0 <= h <= exp(-1)")
    # 2^-f = 1 - f P(f)
    P = lambda f: (1 - mp.mpf(2) ** -f) / f if f else mp.log(2)
    emit("PolyE", [(near_minimax(P, one), one)], "(1 - 2^-f)/f, 0 <= f <= 1")
    # sin z = z (1 - z2 S(z2)), cos z = 1 - z2 C(z2), z2 = z^2 <= (pi/4)^2
    z2 = (mp.pi / 4) ** 2
    emit("PolySC", [([1 / mp.factorial(2 * k + 3) for k in range(9)], z2), ([1 / mp.factorial(2 * k + 2) for k in range(10)], z2)],
         "(1 - sin(z)/z)/z^2 and (1 - cos(z))/z^2 in z^2, |z| <= pi/4")
    print("constexpr uint64_t kLn2_64 = 0x%016xull;   // ln 2 in 2^-64" % int(mp.nint(mp.log(2) * TWO64)))
    print("constexpr uint64_t kLn2_58 = 0x%016xull;   // ln 2 in 2^-58" % int(mp.nint(mp.log(2) * mp.mpf(2) ** 58)))
    print("constexpr uint64_t kLog2e_63 = 0x%016xull; // log2 e in 2^-63" % int(mp.nint(mp.mpf(2) ** 63 / mp.log(2))))
    print("constexpr uint64_t kTwoPi_61 = 0x%016xull; // 2 pi in 2^-61" % int(mp.nint(2 * mp.pi * mp.mpf(2) ** 61)))
    print("constexpr uint64_t kInvTwoPi_64 = 0x%016xull; // 1/(2 pi) in 2^-64" % int(mp.nint(TWO64 / (2 * mp.pi))))
    # log: reciprocals of the upper ends of 128 intervals of [1/2, 1), and their logarithms
    C = [(1 << 23) // (129 + j) for j in range(128)]
    print("// floor(2^15 256/(129 + j)) and ln of that fraction, in 2^-64")
    print("#define MLKD_LOG_RECIPROCALS \\")
    print(", \\\n".join("    " + ", ".join("%du" % v for v in C[i:i + 12]) for i in range(0, 128, 12)))
    print("#define MLKD_LOG_TABLE \\")
    T = [int(mp.nint(mp.log(mp.mpf(v) / 2 ** 15) * TWO64)) for v in C]
    print(", \\\n".join("    " + ", ".join("0x%016xull" % v for v in T[i:i + 4]) for i in range(0, 128, 4)))
    print("}  // namespace fx\n}  // namespace mlkd")


if __name__ == "__main__":
    main()
