"""Writes fx_table.inc: the constants of the integer-pipe exponential
(mag_fx.cuh), computed from their definitions with 60-digit decimal arithmetic:

  FX_LOG2E_HI, _LO  floor(2^127 log2 e), as two 64-bit words
  FX_LN2            round(2^72 ln2 / 256)
  T[j]              round(2^63 2^(-j/256)), j = 0..255

Run: python gen_fx_table.py > fx_table.inc
"""
from decimal import ROUND_FLOOR, ROUND_HALF_EVEN, Decimal as D, getcontext

getcontext().prec = 60
LN2 = D(2).ln()


def main():
    log2e = int((D(2) ** 127 / LN2).to_integral_value(ROUND_FLOOR))
    print("// Generated by gen_fx_table.py.")
    print("#define FX_LOG2E_HI 0x%016Xull" % (log2e >> 64))
    print("#define FX_LOG2E_LO 0x%016Xull" % (log2e & (2**64 - 1)))
    print("#define FX_LN2 0x%016Xull" % int((LN2 / 256 * D(2) ** 72).to_integral_value(ROUND_HALF_EVEN)))
    print("#define FX_TABLE_SIZE 256")
    print("#define FX_TABLE_ENTRIES \\")
    rows = []
    for j in range(0, 256, 4):
        v = [int((D(2) ** 63 * (-(LN2 * j) / 256).exp()).to_integral_value(ROUND_HALF_EVEN)) for j in range(j, j + 4)]
        rows.append("  " + ", ".join("0x%016Xull" % x for x in v))
    print(", \\\n".join(rows))


main()
