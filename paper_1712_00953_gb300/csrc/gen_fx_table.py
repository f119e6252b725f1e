"""Generate fx_table.h: the integer tables and constants of fx.cuh.

RK_FX_EXP2_VALUES[j] = 2^(j/256) scaled by 2^63, j = 0..255 (the table of Tang,
"Table-driven implementation of the exponential function in IEEE
floating-point arithmetic", ACM TOMS 15(2), 1989, held as 64-bit integers);
RK_FX_INV_C_VALUES[j] = 2^64 / (1 + (j + 1/2)/128), j = 0..127, and
RK_FX_LOG2_C_VALUES[j] = -log2 of that rounded value over 2^64, scaled by 2^59
(the tables of Tang's logarithm, ACM TOMS 16(4), 1990); ln 2 scaled by 2^64,
log2 e by 2^63 and log2(1e-6) by 2^52.  Values are
computed with 60-digit decimal arithmetic and rounded once.

    python paper_1712_00953_gb300/csrc/gen_fx_table.py > paper_1712_00953_gb300/csrc/fx_table.h
"""

from decimal import ROUND_HALF_EVEN, Decimal, getcontext

N = 256


def main():
    getcontext().prec = 60
    ln2 = Decimal(2).ln()

    def r(x):
        return int(x.to_integral_value(rounding=ROUND_HALF_EVEN))

    lines = ["// Generated by gen_fx_table.py: RK_FX_EXP2_VALUES[j] = 2^(j/256) 2^63 rounded.",
             "#pragma once", f"#define RK_FX_EXP2_N {N}", "#define RK_FX_EXP2_VALUES \\"]
    for j in range(N):
        v = r((ln2 * j / N).exp() * Decimal(2) ** 63)
        lines.append(f"    0x{v:016x}ull" + (", \\" if j + 1 < N else ""))
    inv_c = [r(Decimal(2) ** 64 / (1 + (Decimal(j) + Decimal(1) / 2) / 128)) for j in range(128)]
    log_c = [r(-(Decimal(v) / Decimal(2) ** 64).ln() / ln2 * Decimal(2) ** 59) for v in inv_c]
    for name, vals in (("INV_C", inv_c), ("LOG2_C", log_c)):
        lines.append(f"#define RK_FX_{name}_VALUES \\")
        lines += [f"    0x{v:016x}ull" + (", \\" if j < 127 else "") for j, v in enumerate(vals)]
    lines.append(f"#define RK_FX_LN2 0x{r(ln2 * Decimal(2) ** 64):016x}ull")
    lines.append(f"#define RK_FX_LN2_HI 0x{r(ln2 * Decimal(2) ** 64) >> 32:08x}u")
    lines.append(f"#define RK_FX_LN2_LO 0x{r(ln2 * Decimal(2) ** 64) & 0xFFFFFFFF:08x}u")
    lines.append(f"#define RK_FX_LOG2E 0x{r(Decimal(2) ** 63 / ln2):016x}ull")
    lines.append(f"#define RK_FX_LOG2_1EM6 ({r(Decimal(10).ln() * -6 / ln2 * Decimal(2) ** 52)}ll)")
    print("\n".join(lines))


if __name__ == "__main__":
    main()
