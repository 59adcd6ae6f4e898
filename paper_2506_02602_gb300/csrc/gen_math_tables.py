"""Generate math_tables.cuh: the constants of the table-driven fp64 exp and log.

exp (Tang 1989, "Table-driven implementation of the exponential function in IEEE
floating-point arithmetic"): x = (128 m + j) ln2/128 + r, exp(x) = 2^m 2^(j/128) e^r with
|r| <= ln2/256; the table holds 2^(j/128), j = 0..127, each correctly rounded.

exp2 in fixed point (exp2_q52): 2^(j/2^10) and 2^(j/2^20) - 1, j = 0..1023, rounded to 64-bit
integers in units of 2^-63 and 2^-64.

log2 in fixed point (log2_q58): c_j = 2^15 / (1 + (j + 1/2) / 256), j = 0..255, rounded to
integers, and -log2(c_j 2^-15) of the rounded c_j in units of 2^-58.

log (Tang 1990, "Table-driven implementation of the logarithm function"): x = 2^e f,
f in [1, 2), c_j = RN(1 / (1 + j/64)) with j the nearest 64th of f - 1, r = f c_j - 1
(one FMA), log x = e ln2 + L_j + log1p(r) with L_j = -ln(c_j) correctly rounded for the
stored double c_j.  For inputs in [0.5, 1) (e = -1) a second table holds -ln(2 c_j), so
the result near 1 keeps full relative accuracy.

Double-float log (ff.cuh): the same reduction with c_j rounded to fp32, -ln(c_j) of the stored
c_j as a pair of fp32 numbers, and ln2 as a 16-bit number plus a pair.

Every value is computed with 60-digit decimal arithmetic and rounded once to double.
Run:  python gen_math_tables.py > math_tables.cuh
"""
from decimal import Decimal, getcontext
from struct import pack, unpack

getcontext().prec = 60
LN2 = Decimal(2).ln()


def hexd(x: Decimal) -> str:
    return float(x).hex()


def f32(x) -> float:
    return unpack("f", pack("f", float(x)))[0]


def pair(x: Decimal):
    h = f32(x)
    return h, f32(x - Decimal(h))


def main():
    out = ["// math_tables.cuh -- generated by gen_math_tables.py; do not edit.",
           "// Constants of the table-driven fp64 exp / log (Tang 1989, 1990).",
           "#pragma once", "", "namespace chem {", ""]
    out.append("// 2^(j/128), j = 0..127")
    out.append("__device__ const double k_exp2_128[128] = {")
    for j in range(128):
        out.append(f"    {hexd((Decimal(j) / 128 * LN2).exp())},")
    out.append("};")
    out.append("// 2^(j/2^10) in units of 2^-63 plus half a unit of a 53-bit mantissa, j = 0..1023")
    out.append("__device__ const unsigned long long k_exp2_hi[1024] = {")
    for j in range(1024):
        v = int(((Decimal(j) / 1024 * LN2).exp() * 2**63).to_integral_value()) + 1024
        out.append(f"    {v:#018x}ull,")
    out.append("};")
    out.append("// 2^(j/2^20) - 1 in units of 2^-64, j = 0..1023")
    out.append("__device__ const unsigned long long k_exp2_lo[1024] = {")
    for j in range(1024):
        v = int((((Decimal(j) / 2**20 * LN2).exp() - 1) * 2**64).to_integral_value())
        out.append(f"    {v:#016x}ull,")
    out.append("};")
    cq = [int((2**15 / (1 + (j + Decimal(1) / 2) / 256)).to_integral_value()) for j in range(256)]
    out.append("// c_j = RN(2^15 / (1 + (j + 1/2) / 256)), j = 0..255")
    out.append("__device__ const unsigned short k_log2_c[256] = {")
    for j in range(0, 256, 8):
        out.append("    " + " ".join(f"{c}," for c in cq[j:j + 8]))
    out.append("};")
    out.append("// -log2(c_j 2^-15) in units of 2^-58")
    out.append("__device__ const long long k_log2_q58[256] = {")
    for c in cq:
        v = int((-(Decimal(c) / 2**15).ln() / LN2 * 2**58).to_integral_value())
        out.append(f"    {v}ll,")
    out.append("};")
    inv = [float(1 / (1 + Decimal(j) / 64)) for j in range(65)]
    out.append("// c_j = RN(1 / (1 + j/64)), j = 0..64")
    out.append("__device__ const double k_log_inv[65] = {")
    for c in inv:
        out.append(f"    {c.hex()},")
    out.append("};")
    out.append("// L_j = -ln(c_j) for the stored c_j")
    out.append("__device__ const double k_log_tab[65] = {")
    for c in inv:
        out.append(f"    {hexd(-Decimal(c).ln())},")
    out.append("};")
    out.append("// -ln(2 c_j): the same table for inputs in [0.5, 1), where e ln2 and L_j would cancel")
    out.append("__device__ const double k_log_tab_m1[65] = {")
    for c in inv:
        out.append(f"    {hexd(-(2 * Decimal(c)).ln())},")
    out.append("};")
    out.append("// {c_j = RN32(1 / (1 + j/64)), -ln(c_j) as a pair, 0}, j = 0..64")
    out.append("__device__ const float k_ln_ff[65][4] = {")
    for j in range(65):
        c = f32(1 / (1 + Decimal(j) / 64))
        h, lo = pair(-Decimal(c).ln())
        out.append(f"    {{{c.hex()}f, {h.hex()}f, {lo.hex()}f, 0.0f}},")
    out.append("};")
    ln2 = float(LN2)
    ln2a = 0.693145751953125
    ln2b, ln2c = pair(LN2 - Decimal(ln2a))
    out += [
        f"constexpr double kLn2Hi = {ln2.hex()};",
        f"constexpr double kLn2Lo = {hexd(LN2 - Decimal(ln2))};",
        f"constexpr double kInvLn2x128 = {hexd(128 / LN2)};",
        f"constexpr double kLn2d128Hi = {float(LN2 / 128).hex()};",
        f"constexpr double kLn2d128Lo = {hexd(LN2 / 128 - Decimal(float(LN2 / 128)))};",
        f"constexpr double kLog2E = {hexd(1 / LN2)}, kLog2_10 = {hexd(Decimal(10).ln() / LN2)};",
        f"constexpr unsigned kLn2Q64Hi = {int(LN2 * 2**64) >> 32:#x}u, kLn2Q64Lo = {int(LN2 * 2**64) & 0xffffffff:#x}u;",
        f"constexpr long long kLog2E_q62 = {int((1 / LN2 * 2**62).to_integral_value()):#x}ll;",
        f"constexpr unsigned long long kLog2E_q127Hi = {int(1 / LN2 * 2**127) >> 64:#x}ull, "
        f"kLog2E_q127Lo = {int(1 / LN2 * 2**127) & (2**64 - 1):#x}ull;",
        f"constexpr long long kLog2EThird_q64 = {int((1 / LN2 / 3 * 2**64).to_integral_value()):#x}ll;",
        f"constexpr float kLn2A = {ln2a.hex()}f, kLn2B = {ln2b.hex()}f, kLn2C = {ln2c.hex()}f;",
        f"constexpr double kLn10 = {hexd(Decimal(10).ln())};",
        f"constexpr double kInvLn10 = {hexd(1 / Decimal(10).ln())};",
        "", "}  // namespace chem", ""]
    print("\n".join(out))


if __name__ == "__main__":
    main()
