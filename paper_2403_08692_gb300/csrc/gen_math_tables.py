"""Writes math_tables.inc, the tables of the FP64 exponential and sine/cosine
in math_fp64.cuh: 2^(k/64) for k = 0 .. 63, and the sine and cosine of
2 pi k / 64 for k = 0 .. 64, each as the nearest double and the nearest double
to what it leaves; ln 2 / 64 split so that n times its high part is exact for
|n| < 2^17.  Values come from Python's decimal module at 60 digits (sine and
cosine from their Taylor series, pi from Machin's formula).

Run: python gen_math_tables.py > math_tables.inc
"""
from decimal import Decimal, getcontext, ROUND_HALF_EVEN

getcontext().prec = 60
STEPS = 64


def two(v):
    hi = float(v)  # float() of a Decimal rounds correctly
    return hi.hex(), float(v - Decimal(hi)).hex()


def atan_inv(n):
    """arctan(1/n) by its series."""
    x, total, k, sign = Decimal(1) / n, Decimal(0), 1, 1
    power = x
    while power > Decimal(10) ** -58:
        total += sign * power / k
        power /= n * n
        k += 2
        sign = -sign
    return total


def sin_cos(x):
    s, c, term, k = Decimal(0), Decimal(0), Decimal(1), 0
    while abs(term) > Decimal(10) ** -58 or k < 4:
        if k % 2:
            s += term if k % 4 == 1 else -term
        else:
            c += term if k % 4 == 0 else -term
        k += 1
        term = term * x / k
    return s, c


def circle(k, pi):
    """Sine and cosine of 2 pi k / STEPS, exact on the axes."""
    quarter, rest = divmod(k, STEPS // 4)
    s, c = sin_cos(2 * pi * rest / STEPS) if rest else (Decimal(0), Decimal(1))
    for _ in range(quarter):
        s, c = c, -s
    return s, c


def main():
    pi = 4 * (4 * atan_inv(5) - atan_inv(239))
    step = Decimal(2).ln() / STEPS
    grid = Decimal(2) ** -42  # 36 significant bits
    hi = (step / grid).to_integral_value(rounding=ROUND_HALF_EVEN) * grid
    print("// Generated by gen_math_tables.py; do not edit.")
    print(f"#define GAPS_EXP_STEP_INV {float(STEPS / Decimal(2).ln()).hex()}")
    print(f"#define GAPS_EXP_STEP_HI {float(hi).hex()}")
    print(f"#define GAPS_EXP_STEP_LO {float(step - hi).hex()}")
    print(f"#define GAPS_TWO_PI {float(2 * pi).hex()}")
    print("// {2^(k/64), remainder}, k = 0 .. 63")
    print("#define GAPS_EXP_TABLE \\")
    print(", \\\n".join("  {%s, %s}" % two((Decimal(2).ln() * k / STEPS).exp()) for k in range(STEPS)))
    print("// {sin, cos, remainder of sin, of cos} of 2 pi k / 64, k = 0 .. 64")
    print("#define GAPS_CIRCLE_TABLE \\")
    rows = []
    for k in range(STEPS + 1):
        s, c = circle(k, pi)
        (sh, sl), (ch, cl) = two(s), two(c)
        rows.append("  {%s, %s, %s, %s}" % (sh, ch, sl, cl))
    print(", \\\n".join(rows))


if __name__ == "__main__":
    main()
