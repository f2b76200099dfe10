"""The arithmetic that the FP64 stages are made of (dfloat.cuh, weno_df.cuh),
compiled for the host, against long double at the error bounds that follow from
its steps, and at the ends of its ranges."""
import os
import re

import numpy as np
import pytest

import _host_build as H

L = np.longdouble
SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), os.pardir,
                   "paper_2207_05258_gb300", "csrc", "line_df.cuh")
PAIR, DIV, RSQRT2, MUL, TO_DOUBLE, MADD, ADD, RECIP, RSQRT, TO_FLOAT = range(10)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return H.load(tmp_path_factory.mktemp("host"))


def run(lib, op, a, b=None):
    a = np.ascontiguousarray(a, float)
    b = a.copy() if b is None else np.ascontiguousarray(b, float)
    r = np.zeros(len(a))
    h, l = np.zeros(len(a), np.float32), np.zeros(len(a), np.float32)
    lib.host_arith(op, len(a), H.ptr(a), H.ptr(b), H.ptr(r), H.ptr(h), H.ptr(l))
    return r, h.astype(L) + l.astype(L)


def spread(lo, hi, n=20000, seed=1):
    g = np.random.default_rng(seed)
    return 2.0 ** g.uniform(lo, hi, n) * g.choice([-1, 1], n)


def rel(x, exact):
    return float((np.abs(x - exact) / np.abs(exact)).max())


def test_to_pair(lib):
    """24 leading bits, and the other 29 rounded to 24."""
    x = spread(-100, 40)
    assert rel(run(lib, PAIR, x)[1], x.astype(L)) <= 2.0 ** -47
    x = np.array([0.0, 2.0 ** -127, 1e-300, 5e-324])
    assert (run(lib, PAIR, np.r_[x, -x])[1] == 0).all()
    x = np.array([2.0 ** 40, 1e300, np.inf, np.nan])
    assert np.isnan(run(lib, PAIR, np.r_[x, -x])[1]).all()
    x = np.array([2.0 ** -126, np.nextafter(2.0 ** 40, 0)])
    assert (run(lib, PAIR, x)[1] != 0).all() and rel(run(lib, PAIR, x)[1], x.astype(L)) <= 2.0 ** -24


def test_to_double_and_to_float(lib):
    x = spread(-126, 127).astype(np.float32)
    assert (run(lib, TO_DOUBLE, x)[0] == x).all()
    assert (run(lib, TO_DOUBLE, np.array([0.0, 1e-40, -1e-45]))[0] == 0).all()
    x = spread(-125, 126)
    r = run(lib, TO_FLOAT, x)[0]
    assert rel(r, x) <= 2.0 ** -23 and (np.abs(r) <= np.abs(x)).all()  # truncated
    assert (run(lib, TO_FLOAT, [0.0, 1e-39, -1e-320])[0] == 0).all()
    assert np.isnan(run(lib, TO_FLOAT, [2.0 ** 127, -1e300, np.inf, np.nan])[0]).all()


def test_pair_operations(lib):
    a, b = spread(-20, 20, seed=2), spread(-20, 20, seed=3)
    A, B = run(lib, PAIR, a)[1], run(lib, PAIR, b)[1]
    # (to_pair truncates the leading word: second words up to 2^-23)
    # product: that of the second words, 2^-46, and two roundings of a sum below 2^-21.4
    assert rel(run(lib, MUL, a, b)[1], A * B) <= 2.0 ** -44
    s = run(lib, ADD, a, b)[1]
    # sum: two roundings of sums of second words
    assert (np.abs(s - (A + B)) <= 2.0 ** -46 * (np.abs(A) + np.abs(B))).all()
    s = run(lib, MADD, a, b)[1]
    assert (np.abs(s - (A * B + 1)) <= 2.0 ** -43.5 * (np.abs(A * B) + 1)).all()
    # quotient: the first one's error, below 2^-21, times the reciprocal's, 2^-22;
    # reciprocal root: 3/2 of 2^-21.5 squared
    assert rel(run(lib, DIV, a, b)[1], A / B) <= 2.0 ** -42.5
    a = np.abs(a)
    assert rel(run(lib, RSQRT2, a)[1], 1 / np.sqrt(np.abs(A))) <= 2.0 ** -42


def test_fp64_reciprocals(lib):
    """One unit in the last place, also where the FP32 seed's range ends."""
    edge = np.array([2.0 ** -100, 2.0 ** 100])
    x = np.r_[spread(-300, 300), spread(-101, -99), spread(99, 101), edge, np.nextafter(edge, 0),
              np.nextafter(edge, np.inf), 1e-307, -1e307, 2.0 ** -126, 2.0 ** 127]
    assert rel(run(lib, RECIP, x)[0].astype(L), 1 / x.astype(L)) <= 2.0 ** -52
    x = np.abs(x)
    assert rel(run(lib, RSQRT, x)[0].astype(L), 1 / np.sqrt(x.astype(L))) <= 2.0 ** -52
    with np.errstate(divide="ignore"):
        x = np.array([0.0, np.inf, -np.inf, np.nan])
        assert np.array_equal(run(lib, RECIP, x)[0], 1 / x, equal_nan=True)
    assert np.isnan(run(lib, RSQRT, [-1.0, np.nan])[0]).all()
    assert np.array_equal(run(lib, RSQRT, [0.0, np.inf])[0], [np.inf, 0.0])


def test_derivative_flux_is_p0_of_the_split_fluxes():
    """The FP64 derivative flux, with the coefficients read from the source, is
    both sides' p_0' of Sec. 2.1 taken from the split fluxes."""
    sympy = pytest.importorskip("sympy")
    with open(SRC) as f:
        body = f.read()
    body = body[body.index("double derivative_flux_fp64("):]
    body = body[:body.index("\n}")]
    F, U, h, N = (sympy.symbols("%s0:4" % c) for c in ("F", "U", "h", "N"))
    al, dx = sympy.symbols("alpha dx")
    env = {"sub": lambda x, y: x - y, "add": lambda x, y: x + y, "mul": lambda x, y: x * y,
           "madd": lambda x, y, z: x * y + z, "alpha": al, "dx": dx, "c": 0, "m": 0, "k": 1, "p": 2, "q": 3}
    for name, v in (("F", F), ("U", U), ("h", h), ("N", N)):
        env["r_" + name] = lambda c, i, v=v: v[i]
    body = re.sub(r"r\.(\w)\(", r"r_\1(", body)
    number = re.compile(r"(?<![\w.])(\d+\.\d+)")
    stmts = re.findall(r"(?:const double |, )(\w+) = (.*?)(?=, \w+ = |;)", body, re.S)
    stmts += [("out", re.search(r"return (.*?);", body, re.S).group(1))]
    for name, e in stmts:
        if name in env:  # (the points' indices)
            continue
        e = number.sub(r"sympy.nsimplify('\1')", e.replace("\n", " "))
        env[name] = eval(e, {"sympy": sympy}, env)
    f = {s: [(F[i] + s * al * U[i]) / 2 for i in range(4)] for s in (1, -1)}
    H_ = {s: [dx * (h[i] + s * al * N[i]) / 2 for i in range(4)] for s in (1, -1)}

    def dp0(a, b):
        return (a[0] - 8 * a[1] + 7 * a[2]) / 4 + (b[0] - 2 * b[1] - 5 * b[2]) / 12

    both = dp0(f[1][:3], H_[1][:3]) - dp0(f[-1][:0:-1], [-x for x in H_[-1][:0:-1]])
    assert len(stmts) >= 9 and sympy.expand(both - env["out"]) == 0
