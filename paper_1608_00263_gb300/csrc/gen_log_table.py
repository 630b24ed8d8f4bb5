"""Writes qs_log_table.inc: the table of the complex128 statistics' logarithm
(stat_terms_f64 in qs_stats.cu), pairs (c_i, -ln c_i) with c_i the FP32 value nearest
1 / (1 + (i + 1/2) / SIZE).

The logarithms are formed in 40 decimal digits and rounded once.  The build
writes the file into its object directory (build.py).
"""
import decimal
import struct

BITS = 11
SIZE = 1 << BITS


def reciprocal(i):
    return struct.unpack("f", struct.pack("f", 1.0 / (1.0 + (i + 0.5) / SIZE)))[0]


def entries():
    with decimal.localcontext() as ctx:
        ctx.prec = 40
        return [(c, float(-decimal.Decimal(c).ln())) for c in map(reciprocal, range(SIZE))]


def emit():
    out = ["// generated by gen_log_table.py",
           "constexpr int kLogBits = %d;" % BITS,
           "__device__ const double2 kLogTable[1 << kLogBits] = {"]
    out += ["    {%s, %s}," % (c.hex(), v.hex()) for c, v in entries()]
    return "\n".join(out + ["};", ""])
