"""The FP64 path's table of 2^(j/512) in two words (csrc/exp_table.cuh), recomputed
with 80 digits: the first word is the value rounded to double, the second the rest
rounded to double.  (The paths' tests see 1e-12 and would not notice a wrong second
word.)  Without a GPU."""
import os
import re
from decimal import Decimal, getcontext

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_entry():
    getcontext().prec = 80
    src = open(os.path.join(ROOT, "paper_2407_11349_gb300", "csrc", "exp_table.cuh")).read()
    pairs = re.findall(r"\{(-?0x[0-9a-f.]+p[+-]\d+), (-?0x[0-9a-f.]+p[+-]\d+)\}", src)
    assert len(pairs) == 512
    for j, words in enumerate(pairs):
        hi, lo = (float.fromhex(w) for w in words)
        v = (Decimal(j) * Decimal(2).ln() / 512).exp()
        assert hi == float(v), j  # float() rounds correctly
        assert lo == float(v - Decimal(hi)), j


def test_the_method_at_its_points():
    """exp(x) = 2^m (T0 + (T0 p + T1)) with x = k ln2 / 512 + r, the kernel's
    operations in order (products and sums rounded; a fused product where the
    kernel has one), against 80 digits: within 0.6 units in the last place."""
    from fractions import Fraction as Q
    getcontext().prec = 80
    src = open(os.path.join(ROOT, "paper_2407_11349_gb300", "csrc", "exp_table.cuh")).read()
    tab = [tuple(float.fromhex(w) for w in p) for p in re.findall(r"\{(-?0x[0-9a-f.]+p[+-]\d+), (-?0x[0-9a-f.]+p[+-]\d+)\}", src)]

    def fma(a, b, c):  # correctly rounded
        q = Q(a) * Q(b) + Q(c)
        return q.numerator / q.denominator

    worst = 0.0
    for i in range(400):
        x = -((i * 0.7548776662466927) % 1.0) * (1.0 if i % 2 else 700.0)
        k = round(Q(fma(x, float.fromhex("0x1.71547652b82fep+9"), 6755399441055744.0)) - 6755399441055744)
        r = fma(float(k), -float.fromhex("0x1.62e42fefa39efp-10"), x)
        r = fma(float(k), -float.fromhex("0x1.abc9e3b39803fp-65"), r)
        q = fma(r, 1.0 / 24.0, 1.0 / 6.0)
        q = fma(r, q, 0.5)
        p = fma(r * r, q, r)
        t = tab[k & 511]
        y = t[0] + fma(t[0], p, t[1])
        exact = (Decimal(x) - Decimal(k >> 9) * Decimal(2).ln()).exp()
        worst = max(worst, abs(float((Decimal(y) - exact) / Decimal(2) ** -52)) / (1.0 if y < 2.0 else 2.0))
    assert worst <= 0.6
