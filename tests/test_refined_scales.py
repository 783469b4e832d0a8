"""Powers of two that the refined weight solve forms by writing an exponent
field (fx_pow2f, defined for exponents -126 .. 127): every use in the source,
evaluated at the ends of the ranges that the source declares."""

import itertools
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _source():
    with open(os.path.join(ROOT, "paper_2107_03632_gb300", "csrc", "refined.cu")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_scales_are_normal_floats():
    src = _source()
    m = re.search(r"kRefMinExp = (-?\d+), kRefMaxExp = (\d+), kRefLambda = (\d+);", src)
    assert m, "no declared range of the exponents"
    lo, hi, lam = map(int, m.groups())
    # e and el are held at the lower end, e0 is rejected below it
    assert "e = max(em, kRefMinExp)" in src and "(it == 0 && em < kRefMinExp)" in src and "e > kRefMaxExp" in src
    assert "- 126, kRefMinExp)" in src and "el > e0 + kRefLambda" in src
    uses = re.findall(r"fx_pow2f\(([^()]*)\)", src)
    assert len(uses) >= 9
    for use in uses:
        assert set(re.findall(r"[a-z]\w*", use)) <= {"e", "e0", "el"}, use
        for e, e0, d in itertools.product((lo, hi), (lo, hi), (0, 1)):
            k = eval(use, {}, {"e": e, "e0": e0, "el": (e0 + lam) if d else lo})
            assert -126 <= k <= 127, (use, k)
