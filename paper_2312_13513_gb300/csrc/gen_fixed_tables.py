"""Writes fixed_tables.h: the constants of the fixed-point exponential and logarithm (fixed.cuh).

* 2^(j / 256) for j = 0 .. 255 as 64-bit mantissas (value times 2^62, rounded to nearest);
* for j = 0 .. 127 a 16-bit reciprocal c_j of the midpoint of [1 + j / 128, 1 + (j + 1) / 128)
  (value times 2^16), and -log2(c_j) times 2^60, rounded to nearest;
* the Taylor coefficients of 2^x and of log2(1 + x) at the scales fixed.cuh states.

Everything is computed in 60-digit decimal arithmetic, so the header is reproducible bit for bit
on any host.  Run:  python gen_fixed_tables.py > fixed_tables.h
"""
from decimal import ROUND_HALF_EVEN, Decimal, getcontext

getcontext().prec = 60


def nearest(v: Decimal) -> int:
    return int(v.to_integral_value(rounding=ROUND_HALF_EVEN))


def rows(vals, per=4):
    out = []
    for i in range(0, len(vals), per):
        out.append("    " + ", ".join(vals[i:i + per]) + ("," if i + per < len(vals) else "") + " \\")
    return out


def main() -> None:
    ln2 = Decimal(2).ln()
    u64 = lambda n: f"0x{n:016x}ull"
    out = ["// Generated by gen_fixed_tables.py; do not edit.",
           "#pragma once",
           "// 2^(j / 256) times 2^62, j = 0 .. 255",
           "#define CHEM_FX_EXP2_VALUES \\"]
    out += rows([u64(nearest((ln2 * j / 256).exp() * 2 ** 62)) for j in range(256)])
    c = [nearest(Decimal(2 ** 16) / (1 + (Decimal(j) + Decimal("0.5")) / 128)) for j in range(128)]
    out += ["", "// reciprocals c_j times 2^16 and their logarithms -log2(c_j) times 2^60, j = 0 .. 127",
            "#define CHEM_FX_RCP_VALUES \\"]
    out += rows([f"0x{v:05x}u" for v in c], 8)
    out += ["", "#define CHEM_FX_LOG2_VALUES \\"]
    out += rows([u64(nearest(-(Decimal(v) / 2 ** 16).ln() / ln2 * 2 ** 60)) for v in c])
    out += ["", "namespace chem {", "namespace fx {",
            "// 2^x = 1 + sum a_k x^k, a_k = ln(2)^k / k!, with x = u 2^-8, u in [0, 1):",
            "// a_1, a_2 2^-8k scaled by 2^72 and 2^80, a_3 .. a_5 by 2^60"]
    a = [None]
    f = Decimal(1)
    for k in range(1, 6):
        f = f * ln2 / k
        a.append(f / Decimal(2) ** (8 * k))
    out.append(f"constexpr unsigned long long kE1 = {u64(nearest(a[1] * 2 ** 72))};")
    out.append(f"constexpr unsigned long long kE2 = {u64(nearest(a[2] * 2 ** 80))};")
    for k in (3, 4, 5):
        out.append(f"constexpr unsigned int kE{k} = 0x{nearest(a[k] * 2 ** 60):08x}u;")
    out += ["// log2(1 + r) = sum b_k rho^k, r = rho 2^-8: b_k = (-1)^(k+1) 2^-8k / (k ln 2), times 2^70"]
    for k in range(1, 8):
        b = (-1) ** (k + 1) / (Decimal(k) * ln2) / Decimal(2) ** (8 * k)
        out.append(f"constexpr long long kL{k} = {nearest(b * 2 ** 70)}ll;")
    out.append("// log2(e) times 2^63 and ln 2 as a double")
    out.append(f"constexpr unsigned long long kLog2e = {u64(nearest(2 ** 63 / ln2))};")
    out.append(f"constexpr double kLn2 = {float(ln2).hex()};")
    out += ["}  // namespace fx", "}  // namespace chem"]
    print("\n".join(out))


if __name__ == "__main__":
    main()
