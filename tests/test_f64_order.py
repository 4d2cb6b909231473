"""Node order, windows and scales of the FP64 contraction in digits (csrc/f64_order.cuh), compiled for the host: the order is
a permutation for any rule, and rounding the operands to 55-bit fixed point per window leaves every element, however small,
within the error that a chain of FP64 multiply-adds has."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle.wpccc_oracle as oc
import wpccc_inputs as wi
from scipy import special

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_04252_gb300", "csrc")
LD = np.longdouble
U = LD(2) ** -53


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("order") / "order")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, os.path.join(HERE, "f64_order_host.cpp"), "-o", out], check=True)

    def run(Geta, Gtau, kR, tau=()):
        lines = subprocess.run([out, str(Geta), str(Gtau), repr(float(kR))] + [repr(float(t)) for t in tau], check=True,
                               capture_output=True, text=True).stdout.split("\n")
        return int(lines[0]), np.array(lines[1].split(), dtype=int), np.array(lines[2].split(), dtype=int)
    return run


@pytest.mark.parametrize("Geta,Gtau", [(1, 1), (5, 5), (31, 1), (1, 37), (73, 7), (27, 19), (48, 48), (50, 30), (128, 48)])
@pytest.mark.parametrize("kR", [1e-3, 8.0, 47.9, 120.0, 5e3, float("inf"), float("nan")])
def test_the_order_is_a_permutation_in_whole_windows(order, Geta, Gtau, kR):
    win, nodes, s = order(Geta, Gtau, kR, [-1.0, 0.3, 1.0])
    assert win in (32, 64, 128, 512)
    assert np.array_equal(np.sort(nodes), np.arange(Geta * Gtau))
    assert np.abs(s).max() <= 145          # 2^s and 2^-s stay far inside FP64's range


def _fixed(x, win):
    """Rows in fixed point per window: integers below 2^55 times the power of two above the row's largest value."""
    y = np.zeros(x.shape, LD)
    for g in range(0, x.shape[1], win):
        blk = x[:, g:g + win]
        m = np.abs(blk).max(1)
        e = np.array([int(np.ceil(np.log2(v * LD(1.01)))) if v > 0 else 0 for v in m])
        unit = LD(2) ** (e - 55)
        y[:, g:g + win] = np.rint(blk / unit[:, None]) * unit[:, None]
    return y


@pytest.mark.parametrize("ZT,ZP,Geta,Gtau,z", [(1.0, 1.0, 48, 48, z) for z in (-2.0, 14.0, 16.0, 28.0, -36.0, 50.0, 90.0)] +
                         [(2.0, 2.0, 48, 48, 14.0), (1.0, 6.0, 128, 48, 20.0), (1.0, 1.0, 50, 30, 24.0), (1.0, 1.0, 24, 16, 40.0),
                          (1.0, 1.0, 16, 16, -40.0), (1.0, 1.0, 48, 48, 150.0)])
def test_small_elements_keep_the_accuracy_of_a_chain(order, ZT, ZP, Geta, Gtau, z):
    basis = wi.make_basis(ZT, ZP, (3, 3), (1, 1), (4, 4), 2.5, True, Geta=Geta, Gtau=Gtau)
    b, v = 1.0, 1.5
    T, P, R = basis.T, basis.P, np.hypot(b, z)
    nd = oc._nodes(basis, b, v, z)
    AT = oc._state_tables(T, T.f, nd["rT"], nd["cT"], basis.grid.r)
    AP = oc._state_tables(P, P.f, nd["rP"], nd["cP"], basis.grid.r)
    kR = min(ZT, ZP) * R
    win, nodes, sexp = order(Geta, Gtau, kR, basis.quad.tau)
    scale = (LD(2) ** np.tile(sexp, Geta))[nodes]
    worst = 0.0
    for qp, q in ((0, 0), (1, 1), (0, 1)):
        rows, cols, d = np.nonzero(T.st_m == qp)[0], np.nonzero(P.st_m == q)[0], abs(q - qp)
        W = nd["base"] * (-1j) ** d * special.jv(d, nd["x"]) / nd["rT"]
        for pot in (nd["rT"], np.full(nd["rT"].shape, -ZT)):
            a = (AT[rows] * pot)[:, nodes].astype(LD)
            for w in (W.real, W.imag):
                g = (w * AP[cols])[:, nodes].astype(LD)
                terms = np.abs(a) @ np.abs(g).T
                err = np.abs(_fixed(a * scale, win) @ _fixed(g / scale, win).T - a @ g.T)
                worst = max(worst, float((err / np.maximum(U * terms, np.finfo(LD).tiny)).max()))
    # a chain of G multiply-adds is bounded by G units of 2^-53 sum |terms|; measured on these rules it reaches 15 to 35
    assert worst <= 40.0
