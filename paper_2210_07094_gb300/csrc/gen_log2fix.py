"""Writes log2fix_table.inc: the table and the polynomial of the fixed-point
logarithm of log2fix.cuh, evaluated with 60 digits.  For each of 256 intervals
[1 + j/256, 1 + (j+1)/256): r_j = ceil(2^31 / (1 + j/256)) and -log2(r_j / 2^31)
as a fraction of 2^60; b_1..b_5 with log2(1 + g/256) = g (b_1 - g (b_2 - g (b_3 - g
(b_4 - g b_5)))) for g in [0, 1), interpolated at the Chebyshev points of [0, 1]
(error below 2^-58), scaled by 2^71, 2^80, 2^57, 2^65 and 2^65.  Run from this
directory: python gen_log2fix.py"""
from decimal import Decimal

from gen_exp2fix import LN2, PI, cos, nearest


def table():
    out = []
    for j in range(256):
        r = -(-(1 << 31) * 256 // (256 + j))
        out.append((r, nearest(-(Decimal(r) / 2 ** 31).ln() / LN2 * 2 ** 60)))
    return out


def polynomial(n=5):
    """Newton's interpolation of log2(1 + g/256)/g, expanded to powers of g,
    the signs of the odd powers taken out."""
    xs = [(1 + cos(PI * (2 * i + 1) / (2 * n))) / 2 for i in range(n)]
    d = [(1 + x / 256).ln() / LN2 / x for x in xs]
    for k in range(1, n):
        for i in range(n - 1, k - 1, -1):
            d[i] = (d[i] - d[i - 1]) / (xs[i] - xs[i - k])
    a = [Decimal(0)] * n
    for k in range(n - 1, -1, -1):
        a = [(a[i - 1] if i else Decimal(0)) - xs[k] * a[i] for i in range(n)]
        a[0] += d[k]
    return [v if i % 2 == 0 else -v for i, v in enumerate(a)]


def main():
    out = ["// generated by gen_log2fix.py"]
    for i, (b, s) in enumerate(zip(polynomial(), (71, 80, 57, 65, 65))):
        out.append(f"constexpr uint64_t LOG2FIX_B{i + 1} = 0x{nearest(b * Decimal(2) ** s):x}ull;")
    out.append("struct __align__(16) Log2FixEntry {\n  uint64_t l;\n  uint32_t r, pad;\n};")
    out.append("static __device__ const Log2FixEntry g_log2fix_tab[256] = {")
    for r, l in table():
        out.append(f"    {{0x{l:x}ull, 0x{r:x}u, 0u}},")
    out.append("};")
    with open("log2fix_table.inc", "w") as f:
        f.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
