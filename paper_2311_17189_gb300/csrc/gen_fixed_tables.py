"""Writes the fixed-point tables of the kernels' exponential and cos/sin, which stand in
csrc/tami_devmath.cuh (kExpTab, kTrigTab), from 60-digit values:

  kExpTab[j]  = round((1 - 2^(-j/1024)) 2^64), j = 0..1023
  kTrigTab[j] = (round(cos(j pi/512) 2^61), round(sin(j pi/512) 2^61)), j = 0..256

    python gen_fixed_tables.py          # prints both tables as they stand there
"""
import mpmath as mp

mp.mp.dps = 60


def rounded(v):
    return int(mp.nint(v))


def block(name, vals, shape):
    lines = []
    for i in range(0, len(vals), 4):
        lines.append("  " + ", ".join("0x%016xull" % v for v in vals[i:i + 4]))
    return "__device__ const __align__(16) unsigned long long %s[%s] = {\n%s};" % (name, shape, ",\n".join(lines))


def exp_table():
    return [rounded((1 - mp.power(2, -mp.mpf(j) / 1024)) * mp.power(2, 64)) for j in range(1024)]


def trig_table():
    out = []
    for j in range(257):
        a = j * mp.pi / 512
        out += [rounded(mp.cos(a) * mp.power(2, 61)), rounded(mp.sin(a) * mp.power(2, 61))]
    return out


if __name__ == "__main__":
    print("// Fixed-point tables of the exponential and of cos/sin (tami_devmath.cuh), written by")
    print("// gen_fixed_tables.py from 60-digit values.")
    print(block("kExpTab", exp_table(), "1024"))
    print(block("kTrigTab", trig_table(), "514"))
