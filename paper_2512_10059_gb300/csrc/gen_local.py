"""Generate ``boys_local_tables.h`` (at build time, into the build directory):
local expansions, in integers, of the anchor F_k that starts the downward
recurrence at order k:

* region A, x < x_0: r_{A,k}(x) = P(x)/Q(x) with the printed Appendix D coefficients;
* region B, x_0 <= x < x_1: what the upward recurrence makes of F_0 = r_B(x) at
  order k, F_{l+1} = ((2l+1) F_l - e^{-x}) / (2x); the downward recurrence from it
  gives back the same F_l down to r_B(x), and does so without cancellation;
* region C: F_k = (sqrt(pi)/2) (2k-1)!!/2^k x^{-k-1/2}.

In A and B x is cut into intervals of 1/16, in C the mantissa M of x = M 4^h, M in
[1, 4), into 256 intervals per factor of two (512 above order 12, where the power
is steep).  On an interval the variable is t in [0, 1), the distance from the
right edge over the width: F_k falls with x and its derivatives alternate in
sign, so every coefficient of the expansion about the right edge is positive and
the device sums need no signs.  The polynomial of degree 7 interpolates the
anchor, evaluated in 320-bit fixed point, at the eight Chebyshev nodes of the
interval (relative difference below 2^-61), so the tables are another way of
evaluating the same approximants.  Entries 0..190 are region A's, 191..464 region
B's (whose first interval is the one that holds x_0), then come those of M in
[2, 4) and of M in [1, 2).

An entry is 64 bytes: b_0..b_4 in units of 2^-u of F_k, where the largest value on
the interval lies in [2^62, 2^63); b_5..b_7 in 2^5 of those units (32 bits
each); w and two exponents.  In A and B w = e^{-(j+1)/16} 2^v in [2^63, 2^64), so that
e^{-x} 2^(v-1) = w e / 2^64 with e = 2^63 e^{t/16}, and the exponents are
n = v - 1 - u + 6 (low 16 bits) and 1079 - v (high 16 bits, signed).  In C, where
e^{-x} counts as 0, w = 0 and the exponents are 1084 - u (for h = 0) and 0.

A second table (``boys_grid_table.h``, for the pairwise kernel) holds F_m at the
multiples of 1/16 up to 64 to the last bit of a double, m = 0..40.

Usage:  python gen_local.py > boys_local_tables.h; python gen_local.py grid > boys_grid_table.h
"""
import importlib.util
import os

HERE = os.path.dirname(os.path.abspath(__file__))
STEP = 16            # intervals per unit of x
FIRST_B, LAST = 190, 463  # the intervals that hold x_0 and x_1
W = 320              # fixed-point bits of the generator


def _rationals():
    spec = importlib.util.spec_from_file_location("gen_coeffs_fixed", os.path.join(HERE, "gen_coeffs_fixed.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    rb_p, rb_q, ra_p, ra_q, _, _ = mod.tables()
    return rb_p, rb_q, ra_p, ra_q


def _scaled(c):
    n, d = float(c).as_integer_ratio()
    return (n << W) // d


def _horner(c, x):
    v = c[-1]
    for a in reversed(c[:-1]):
        v = ((v * x) >> W) + a
    return v


def nodes(n):
    """Chebyshev nodes of [0, 1], rounded to 30 bits (any nodes near them do)."""
    import math
    return [int((0.5 - 0.5 * math.cos(math.pi * (2 * i + 1) / (2 * n))) * (1 << 30)) << (W - 30) for i in range(n)]


def interpolant(values, at):
    """Monomial coefficients (scaled by 2^W) of the polynomial through (at, values)."""
    n, dd = len(at), list(values)
    for lev in range(1, n):
        for i in range(n - 1, lev - 1, -1):
            dd[i] = ((dd[i] - dd[i - 1]) << W) // (at[i] - at[i - lev])
    c = [0] * n
    for i in range(n - 1, -1, -1):  # Newton form to monomials
        nxt = [0] + c[:n - 1]
        for d in range(n):
            nxt[d] -= (c[d] * at[i]) >> W
        nxt[0] += dd[i]
        c = nxt
    return c


def rounded(v, bits):
    """v 2^-W in units of 2^-bits, to nearest."""
    sh = W - bits
    return (v + (1 << (sh - 1))) >> sh


def exp_series(t):
    """e^{t}, t and the result scaled by 2^W, 0 <= t < 1."""
    s = term = 1 << W
    i = 0
    while term:
        i += 1
        term = ((term * t) >> W) // i
        s += term
    return s


def exp_neg_edges(count):
    """e^{-j/16}, j = 0..count-1, scaled by 2^W."""
    inv = (1 << (2 * W)) // exp_series((1 << W) // STEP)
    out = [1 << W]
    for _ in range(count - 1):
        out.append((out[-1] * inv) >> W)
    return out


def exp_coeffs():
    """Degree-7 interpolant of e^{t/16} on [0, 1]: e_0..e_4 in Q63, e_5..e_7 in Q58."""
    at = nodes(8)
    c = interpolant([exp_series(t // STEP) for t in at], at)
    return [rounded(v, 63) for v in c[:5]] + [rounded(v, 58) for v in c[5:]]


def log2_intervals(k):
    """Intervals per factor of two of region C's mantissa, as a power of two."""
    return 8 if k <= 12 else 9


def entry(coeffs, top, edge=None):
    """One table entry from the expansion, its largest value and e^{-x} at its right edge."""
    u = 63 + W - top.bit_length()
    row = [rounded(v, u) for v in coeffs[:5]] + [rounded(v, u - 5) for v in coeffs[5:]]
    assert all(b >= 0 for b in row) and max(row[5:]) < 1 << 32
    if edge is None:
        return (*row, 1084 - u, 0, 0)
    v = 64 + W - edge.bit_length()
    w = rounded(edge, v)
    n = v - 1 - u + 6
    assert w < 1 << 64 and 0 <= n < 64
    return (*row, n, 1079 - v, w)


def half_pi_root():
    """sqrt(pi) / 2, scaled by 2^W (Machin's formula)."""
    import math
    pi, guard = 0, 32
    for mul, d in ((16, 5), (-4, 239)):
        t, i, sign = (1 << (W + guard)) // d, 1, 1
        while t:
            pi += sign * mul * (t // i)
            t //= d * d
            i, sign = i + 2, -sign
    return math.isqrt((pi >> guard) << W) // 2


def table_c():
    """Region C's entries, [33][2 * 2^log2_intervals(k)]."""
    import math
    at, one, root = nodes(8), 1 << W, half_pi_root()
    out = [[] for _ in range(33)]
    for bits, orders in ((8, range(0, 13)), (9, range(13, 33))):
        n = 1 << bits
        for octave in (1, 0):
            for j in range(n):
                # the nodes and the left edge, as M scaled by 2^W
                xs = [((one + ((j + 1) * one - t) // n) << octave) for t in at] + [(one + j * one // n) << octave]
                f = [(root << W) // math.isqrt(x << W) for x in xs]
                inv = [(one << W) // x for x in xs]
                for k in range(33):
                    if k in orders:
                        out[k].append(entry(interpolant(f[:8], at), f[8]))
                    f = [(v * i * (2 * k + 1)) >> (W + 1) for v, i in zip(f, inv)]
    return out


def table():
    """[33][] entries (b_0..b_7, two exponents, w), in the units of the module docstring."""
    rb_p, rb_q, ra_p, ra_q = _rationals()
    at, edges = nodes(8), exp_neg_edges(LAST + 2)
    out = []
    for k in range(33):
        p, q = [_scaled(c) for c in ra_p[k]], [_scaled(c) for c in ra_q[k]]

        def r(x):
            return (_horner(p, x) << W) // _horner(q, x)

        out.append([entry(interpolant([r((((j + 1) << W) - t) // STEP) for t in at], at), r((j << W) // STEP), edges[j + 1])
                    for j in range(FIRST_B + 1)])
    p, q = [_scaled(c) for c in rb_p], [_scaled(c) for c in rb_q]
    grow = [exp_series(t // STEP) for t in at]

    def upward(x, e):
        f = [(_horner(p, x) << W) // _horner(q, x)]
        for l in range(32):
            f.append((((2 * l + 1) * f[l] - e) << W) // (2 * x))
        return f

    for j in range(FIRST_B, LAST + 1):
        at_nodes = [upward((((j + 1) << W) - t) // STEP, (edges[j + 1] * g) >> W) for t, g in zip(at, grow)]
        left = upward((j << W) // STEP, edges[j])
        for k in range(33):
            out[k].append(entry(interpolant([f[k] for f in at_nodes], at), left[k], edges[j + 1]))
    return [ab + c for ab, c in zip(out, table_c())]


GRID, GRID_ORDERS = 1024, 41


def grid():
    """F_m(j/16), m = 0..40, j = 1..1024, [m][j-1], scaled by 2^W, from the definition:
    e^{-x} sum_i (2x)^i / ((2m+1)(2m+3)...(2m+2i+1)) at the highest order, downward below."""
    edges, out = exp_neg_edges(GRID + 1), [[] for _ in range(GRID_ORDERS)]
    for j in range(1, GRID + 1):
        x2, m = (2 * j << W) // STEP, GRID_ORDERS - 1
        term = total = (1 << W) // (2 * m + 1)
        i = 0
        while term:
            i += 1
            term = ((term * x2) >> W) // (2 * m + 2 * i + 1)
            total += term
        f = (total * edges[j]) >> W
        out[m].append(f)
        for m in range(GRID_ORDERS - 2, -1, -1):
            f = (((f * x2) >> W) + edges[j]) // (2 * m + 1)
            out[m].append(f)
    return out


def emit_grid():
    """``boys_grid_table.h``: the grid's values as correctly rounded doubles."""
    out = ["// F_m(j/16) as doubles; generated by gen_local.py when the library is built.", "#pragma once",
           f"#define BOYS_GRID {GRID}", f"#define BOYS_GRID_ORDERS {GRID_ORDERS}",
           "static __device__ const double g_grid_f[BOYS_GRID_ORDERS][BOYS_GRID] = {"]
    out += ["{" + ",".join((v / (1 << W)).hex() for v in row) + "}," for row in grid()]
    return "\n".join(out + ["};"]) + "\n"


def emit():
    rows = table()
    out = ["// Local expansions of the anchors; generated by gen_local.py when the library is built.", "#pragma once",
           f"#define BOYS_LOCAL_FIRST_C {FIRST_B + 1 + LAST - FIRST_B + 1}"]
    for k, row in enumerate(rows):
        out.append(f"static __device__ const unsigned long long g_local_{k}[{len(row)}][8] __attribute__((aligned(64))) = {{")
        out += ["{" + ",".join("0x%X" % v for v in
                               (*r[:5], r[5] | r[6] << 32, r[7] | r[8] << 32 | (r[9] & 0xFFFF) << 48, r[10])) + "}," for r in row]
        out.append("};")
    out += [f"#define BOYS_LOCAL_EXP_C{i} 0x{v:X}ULL" for i, v in enumerate(exp_coeffs())]
    return "\n".join(out) + "\n"


if __name__ == "__main__":
    import sys
    sys.stdout.write(emit_grid() if "grid" in sys.argv else emit())
