"""The recursion compiled for the host (csrc/ck_fixed.cuh) over the gas constants that the library accepts, and
the proof that its fixed-point form cannot leave its range unnoticed.

Smooth: a density wave at uniform pressure and Mach 0.05.  Near gamma = 1 the sound speed is far below the
recursion's unit of velocity; in fixed point alone the density would be 1.6e-15 off at gamma 1.02.  The step has
to be right to half a last place of rho, rho c and E (2^-53).  Steep: every coefficient as large as the
state.  A large gamma magnifies (gamma - 1)(E - rho u^2 / 2) out of the format (1e-14 off at gamma 7, no digit right
at 30).  Right to a last place (2^-52) in the mean.  Either way twice what FP64 leaves is enough where that
is more (its pressure cancels for a huge gamma)."""
import os
import re
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2304_09724_gb300", "csrc")


def build(tmp_path, name, *args):
    exe = str(tmp_path / name)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wno-return-type", "-I", CSRC, os.path.join(HERE, name + ".cpp"), "-o", exe])
    return [list(map(float, line.split())) for line in subprocess.check_output([exe, *args], text=True).splitlines()]


def test_range_check_sees_every_value(tmp_path):
    """The operand checks over all of 64 bits: nothing in range refused, nothing out of range let through."""
    assert build(tmp_path, "fx_host") == [[0, 0, 0], [0, 0, 0]]


def test_recursion_over_gas_constants(tmp_path):
    rows = build(tmp_path, "ck_host")
    assert len(rows) == 12
    for gamma, *err in rows:
        for q in range(3):
            assert err[q] <= max(2.0 ** -53, 2.0 * err[3 + q]), f"gamma {gamma:g}: {err[:3]}, FP64 {err[3:6]}"
            steep, fp64 = err[6 + 2 * q:8 + 2 * q]
            assert steep <= max(2.0 ** -52, 2.0 * fp64), f"gamma {gamma:g}, steep, component {q}: {steep}, FP64 {fp64}"


def majorant(eps, gm1):
    """Largest operand of the 2D Euler recursion beyond the leading ones, when every spatial coefficient of degree s
    is at most eps^s, leading values at most 1, 1/rho0 at most 2, and all terms have one sign."""
    sub = lambda i: [(a, b, c) for a in range(i[0] + 1) for b in range(i[1] + 1) for c in range(i[2] + 1)]
    mul = lambda A, B, i: sum(A[t] * B[i[0] - t[0], i[1] - t[1], i[2] - t[2]] for t in sub(i))
    S = [{(m, n, 0): eps ** (m + n) for m in range(5) for n in range(5 - m)} for _ in range(4)]
    u, v, mu, mv, nv, p, H, uH, vH = ({} for _ in range(9))
    worst = 0.0
    for k in range(4):
        for i in ((m, n, k) for m in range(5 - k) for n in range(5 - k - m)):
            lead = sum(i) == 0
            for A, q in ((u, 1), (v, 2)):
                num = S[q][i] + sum(S[0][t] * A[i[0] - t[0], i[1] - t[1], i[2] - t[2]] for t in sub(i) if sum(t))
                A[i] = 1.0 if lead else 2.0 * num
                worst = worst if lead else max(worst, num, A[i])
            mu[i], mv[i], nv[i] = mul(S[1], u, i), mul(S[1], v, i), mul(S[2], v, i)
            e = S[3][i] + 0.5 * (mu[i] + nv[i])
            p[i] = 2.0 if lead else gm1 * e
            H[i] = 1.0 if lead else S[3][i] + p[i]
            worst = worst if lead else max(worst, e, H[i])
            uH[i], vH[i] = mul(u, H, i), mul(v, H, i)
        for m in range(4 - k):
            for n in range(4 - k - m):
                x, y = (m + 1, n, k), (m, n + 1, k)
                for q, (f, g) in enumerate(((S[1][x], S[2][y]), (mu[x] + p[x], mv[y]), (mv[x], nv[y] + p[y]), (uH[x], vH[y]))):
                    S[q][m, n, k + 1] = ((m + 1) * f + (n + 1) * g) / (k + 1)
                    worst = max(worst, S[q][m, n, k + 1]) if k < 3 else worst
    return worst


def test_any_units(tmp_path):
    """The same states in units from 2^-400 to 2^500: a time series differs by its rounding only."""
    rows = build(tmp_path, "ck_host", "units")
    assert len(rows) == 48
    for er, ev, worst in rows:
        assert worst <= 1e-13, f"density 2^{er:g}, velocity 2^{ev:g}: {worst}"


def test_growths_suffice():
    """At the last growth every operand is below 1/4, the format's range, for the largest gamma it is used for."""
    src = open(os.path.join(CSRC, "ck_fixed.cuh")).read()
    tries = int(re.search(r"kCkTries = (\d+);", src).group(1))
    gamma = float(re.search(r"gamma <= ([\d.]+);", src).group(1))
    assert majorant(2.0 ** (1 - tries), gamma - 1.0) < 0.25
