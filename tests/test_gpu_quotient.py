"""scalar_quotient (csrc/sellsolve.cuh), the alpha and beta of every solve,
against the IEEE quotient (numpy's division).

Bound: q1 = a y (1 + e) with the seed's error e, |e| <= 2^-22, differs from the
quotient by a relative 2^-44 + 2^-52; the correction adds y (a - m q1), whose
remainder is exact to 2^-53 of itself and whose y is off by 2^-22, so before the
last rounding the relative error is at most (2^-44 + 2^-52)(2^-22 + 2^-52) <
2^-65.  One rounding then gives the IEEE quotient or, where that one lies within
2^-12 ulp of a tie, its neighbour: at most one unit in the last place apart, and
for random operands almost always equal (two in 2^12 differ at most).  Operands
outside the guards are divided: equal bits."""
import os
import subprocess

import numpy as np
import pytest

from paper_1107_0538_gb300.build import nvcc_path

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def make(field, mantissa, sign=0):
    """Doubles from exponent fields (0..2047), mantissas (52 bits) and signs."""
    bits = (np.asarray(sign, np.uint64) << np.uint64(63)) | (np.asarray(field, np.uint64) << np.uint64(52)) | \
        np.asarray(mantissa, np.uint64)
    return bits.view(np.float64)


def guarded(a, b):
    """Whether the fast form may be taken: both exponent fields in [64, 1982], at most 900 apart."""
    ea, eb = [(v.view(np.uint64) >> np.uint64(52)).astype(np.int64) & 0x7ff for v in (a, b)]
    return (ea >= 64) & (ea <= 1982) & (eb >= 64) & (eb <= 1982) & (np.abs(ea - eb) <= 900)


def operands():
    rng = np.random.default_rng(7)
    n = 1 << 20
    mant = lambda k: rng.integers(0, 1 << 52, k, dtype=np.uint64)   # noqa: E731
    A, B = [make(rng.integers(900, 1150, n), mant(n), rng.integers(0, 2, n))], [
        make(rng.integers(900, 1150, n), mant(n), rng.integers(0, 2, n))]
    # mantissas beside 1 and 2, against each other and against random ones
    edge = np.concatenate([np.arange(64), (1 << 52) - 1 - np.arange(64), (1 << 51) + np.arange(-32, 32),
                           (1 << 29) * np.arange(8), (1 << 29) * np.arange(1, 9) - 1]).astype(np.uint64)
    ma, mb = [v.ravel() for v in np.meshgrid(np.concatenate([edge, mant(64)]), np.concatenate([edge, mant(64)]))]
    for fa, fb in ((1023, 1023), (1022, 1023), (1500, 700), (700, 1500)):
        for s in (0, 1):
            A.append(make(np.full(ma.size, fa), ma, s))
            B.append(make(np.full(ma.size, fb), mb, 1 - s))
    # the guards' limits on both sides, and what is outside: zero, subnormals, infinity, NaN
    fields = np.array([0, 1, 63, 64, 65, 963, 964, 965, 1081, 1082, 1083, 1981, 1982, 1983, 2046, 2047])
    m = np.array([0, 1, 1 << 51, (1 << 52) - 1], np.uint64)
    f, mm, s = [v.ravel() for v in np.meshgrid(fields, m, [0, 1])]
    v = make(f, mm, s)
    a, b = [w.ravel() for w in np.meshgrid(v, v)]
    return np.concatenate(A + [a]), np.concatenate(B + [b])


def test_quotient_is_within_one_unit_of_the_division(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = tmp_path / "quotient_check"
    subprocess.run([nvcc_path(), "-O3", "-std=c++17", "-gencode=arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_1107_0538_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-o", str(exe),
                    os.path.join(ROOT, "tests", "quotient_check.cu")], check=True)
    a, b = operands()
    with open(tmp_path / "in", "wb") as f:
        np.array([a.size], np.int64).tofile(f)
        a.tofile(f)
        b.tofile(f)
    subprocess.run([str(exe), str(tmp_path / "in"), str(tmp_path / "out")], check=True, timeout=120)
    q, d = np.fromfile(tmp_path / "out").reshape(2, -1)
    with np.errstate(all="ignore"):
        want = a / b
    same = (q.view(np.uint64) == want.view(np.uint64)) | (np.isnan(q) & np.isnan(want))
    fast = guarded(a, b)
    assert fast.sum() > 1 << 20 and (~fast).sum() > 1000
    assert np.array_equal(np.isnan(d), np.isnan(want)) and np.array_equal(d[~np.isnan(d)], want[~np.isnan(d)])
    assert same[~fast].all()
    ulps = np.abs(q.view(np.int64)[fast] - want.view(np.int64)[fast])
    assert ulps.max() <= 1, (a[fast][ulps.argmax()], b[fast][ulps.argmax()])
    random = slice(0, 1 << 20)
    assert np.mean(~same[random]) <= 2.0 ** -11
