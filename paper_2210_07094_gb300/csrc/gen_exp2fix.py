"""Writes exp2fix_table.inc: the table and the polynomial of the fixed-point
2^x of exp2fix.cuh, evaluated with 60 digits: 256 entries 2^(j/256) as 64-bit
fractions (1.0 = 2^63, rounded to nearest), and a_1..a_4 with
2^(g/256) = 1 + g (a_1 + g (a_2 + g (a_3 + g a_4))) for g in [0, 1),
interpolated at the Chebyshev points of [0, 1] (error below 2^-56.5), scaled by
2^72, 2^82, 2^60 and 2^60; then log2(e)/2 as a 64-bit fraction.  Run from this
directory: python gen_exp2fix.py"""
from decimal import Decimal, getcontext

getcontext().prec = 60
LN2 = Decimal(2).ln()
PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494")


def cos(x):
    s = t = Decimal(1)
    k = 0
    while abs(t) > Decimal(10) ** -58:
        k += 2
        t = -t * x * x / (k * (k - 1))
        s += t
    return s


def nearest(v):
    return int(v.to_integral_value())


def table():
    return [nearest((Decimal(j) / 256 * LN2).exp() * 2 ** 63) for j in range(256)]


def polynomial():
    """Newton's interpolation of (2^(g/256) - 1)/g, expanded to powers of g."""
    xs = [(1 + cos(PI * (2 * i + 1) / 8)) / 2 for i in range(4)]
    d = [((x / 256 * LN2).exp() - 1) / x for x in xs]
    for k in range(1, 4):
        for i in range(3, k - 1, -1):
            d[i] = (d[i] - d[i - 1]) / (xs[i] - xs[i - k])
    a = [Decimal(0)] * 4
    for k in range(3, -1, -1):  # a <- a (g - x_k) + d_k
        a = [(a[i - 1] if i else Decimal(0)) - xs[k] * a[i] for i in range(4)]
        a[0] += d[k]
    return a


def main():
    a = polynomial()
    scaled = [nearest(a[0] * 2 ** 72), nearest(a[1] * 2 ** 82), nearest(a[2] * 2 ** 60), nearest(a[3] * 2 ** 60)]
    out = ["// generated by gen_exp2fix.py"]
    for name, v in zip(("EXP2FIX_A1", "EXP2FIX_A2", "EXP2FIX_A3", "EXP2FIX_A4"), scaled):
        out.append(f"constexpr uint64_t {name} = 0x{v:x}ull;")
    out.append(f"constexpr uint64_t EXP2FIX_LOG2E_HALF = 0x{nearest(1 / LN2 / 2 * 2 ** 64):x}ull;")
    out.append("static __device__ const uint64_t g_exp2fix_tab[256] = {")
    t = table()
    for j in range(0, 256, 4):
        out.append("    " + " ".join(f"0x{v:016x}ull," for v in t[j:j + 4]))
    out.append("};")
    with open("exp2fix_table.inc", "w") as f:
        f.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
