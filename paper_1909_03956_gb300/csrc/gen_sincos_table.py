"""Write the tables of exp(i 2 pi k / 1024), k = 0 .. 1023, evaluated with
mpmath at 50 digits:

    sincos_table.inc      {cos, sin}, each correctly rounded to float64
    sincos_table_df.inc   {cos high, cos low, sin high, sin low}: the float32
                          nearest to each value and that nearest to the rest

The float64 and double-float predictors evaluate exp(i 2 pi t) by table-driven
argument reduction (the classic table-lookup method, e.g. P. T. P. Tang,
ACM TOMS 15(2), 1989): t = k/1024 + f with |f| <= 1/2048, then
exp(i 2 pi t) = exp(i 2 pi k/1024) * exp(i 2 pi f), the second factor from
short Taylor series. This script only produces the table entries.

    python paper_1909_03956_gb300/csrc/gen_sincos_table.py
"""
import os

import mpmath
import numpy as np

mpmath.mp.dps = 50
HERE = os.path.dirname(os.path.abspath(__file__))


def _f32_pair(x):
    h = np.float32(float(x))               # two roundings: the low part takes up what the first leaves
    return h, np.float32(float(x - mpmath.mpf(float(h))))


def _write(name, head, rows):
    with open(os.path.join(HERE, name), "w") as f:
        f.write("// Generated by gen_sincos_table.py: %s,\n// k = 0 .. 1023.\n{\n" % head)
        f.writelines("    {%s},\n" % ", ".join(r) for r in rows)
        f.write("}\n")


def main():
    val = [(mpmath.cospi(mpmath.mpf(k) / 512), mpmath.sinpi(mpmath.mpf(k) / 512)) for k in range(1024)]
    _write("sincos_table.inc", "{cos, sin}(2 pi k / 1024), correctly rounded to float64",
           [[repr(float(c)), repr(float(s))] for c, s in val])
    _write("sincos_table_df.inc", "{cos, sin}(2 pi k / 1024) as pairs of float32",
           [["%.9gf" % float(x) if "." in "%.9g" % float(x) or "e" in "%.9g" % float(x) else "%.9g.0f" % float(x)
             for v in cs for x in _f32_pair(v)] for cs in val])


if __name__ == "__main__":
    main()
