"""Writes k_tanh64_table.cuh, the table of dcp_tanh64 (run by hand after a
change; tests/test_tanh64_host.py checks the table's values).

Row i covers one interval of |x|: a node a and the Taylor coefficients
c0 .. c6 of tanh at a.  Intervals (k_tanh64.cuh computes the index from the
exponent and leading mantissa bits): row 0 below 2^-9 (a = 0), then 16
intervals per binade up to 2^-3, 64 up to 1 and 128 up to 20.

The node is not the midpoint but a double near it (within 1/32 of the
interval; anywhere in it from 16 on, where c7 h^7 is tiny) where tanh is within 2^-12 ulp of a double (Gal's accurate tables,
Gal and Bachelis, ACM TOMS 17(1), 1991), so c0 adds almost nothing to the
rounding of the final operation.  The coefficients are computed in 200-bit
arithmetic and rounded once.
"""
import os
import random

import mpmath

mpmath.mp.prec = 200

LO, A_END, B_END, END = -9, -3, 0, 20.0  # binades 2^-9.., 2^-3.., 1.., |x| < 20


def intervals():
    out = []
    for e in range(LO, A_END):
        out += [(2.0 ** e * (1 + k / 16), 2.0 ** e / 16) for k in range(16)]
    for e in range(A_END, B_END):
        out += [(2.0 ** e * (1 + k / 64), 2.0 ** e / 64) for k in range(64)]
    e = 0
    while 2.0 ** e < END:
        out += [(2.0 ** e * (1 + k / 128), 2.0 ** e / 128) for k in range(128)
                if 2.0 ** e * (1 + k / 128) < END]
        e += 1
    return out


def taylor(a):
    """tanh's Taylor coefficients at a: t' = 1 - t^2."""
    c = [mpmath.tanh(a)]
    for n in range(6):
        # (n + 1) c_{n+1} = [n = 0] - sum_k c_k c_{n-k}
        s = sum(c[k] * c[n - k] for k in range(n + 1))
        c.append(((1 if n == 0 else 0) - s) / (n + 1))
    return c


def node(lo, width, rng):
    best, err = None, None
    for _ in range(40000):
        # (from 16 on tanh is so flat that the whole interval is searched)
        a = lo + width * (0.5 + rng.uniform(-1, 1) / (32 if lo < 16 else 2))
        t = mpmath.tanh(mpmath.mpf(a))
        d = float(t)
        u = mpmath.mpf(2) ** (mpmath.frexp(mpmath.mpf(d))[1] - 53)
        e = abs((t - d) / u)
        if err is None or e < err:
            best, err = a, e
        if err < mpmath.mpf(2) ** -12:
            break
    return best


def rows():
    rng = random.Random(7)
    out = [[0.0] + [float(v) for v in taylor(mpmath.mpf(0))]]
    mpmath.mp.prec = 120
    for lo, w in intervals():
        a = node(lo, w, rng)
        mpmath.mp.prec = 200
        out.append([a] + [float(v) for v in taylor(mpmath.mpf(a))])
        mpmath.mp.prec = 120
    mpmath.mp.prec = 200
    return out


if __name__ == "__main__":
    r = rows()
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "k_tanh64_table.cuh")
    with open(path, "w") as f:
        f.write("// k_tanh64_table.cuh -- written by gen_tanh64_table.py: rows (a, c0 .. c6) of\n"
                "// dcp_tanh64's table.\n")
        f.write("#define DCP_TANH_ROWS %d\n" % len(r))
        f.write("__device__ __align__(64) const double dcp_tanh_tab[DCP_TANH_ROWS][8] = {\n")
        for x in r:
            f.write("{" + ",".join(v.hex() for v in x) + "},\n")
        f.write("};\n")
