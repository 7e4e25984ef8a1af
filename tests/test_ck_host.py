"""The 1D Euler recursion compiled for the host (csrc/ck_fixed.cuh), over the gas constants that the library
accepts: a density wave at uniform pressure and Mach 0.05.  Near gamma = 1 the sound speed is far below the
recursion's unit of velocity; in fixed point alone the density would be 1.6e-15 off at gamma 1.02.  At every gamma the
step has to be right to half a last place of rho, rho c and E (2^-53), or to twice what FP64 leaves where
that is more (its pressure cancels for a huge gamma)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2304_09724_gb300", "csrc")


def test_recursion_over_gas_constants(tmp_path):
    exe = str(tmp_path / "ck_host")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wno-return-type", "-I", CSRC, os.path.join(HERE, "ck_host.cpp"), "-o", exe])
    rows = [list(map(float, line.split())) for line in subprocess.check_output([exe], text=True).splitlines()]
    assert len(rows) == 11
    for gamma, *err in rows:
        for q in range(3):
            assert err[q] <= max(2.0 ** -53, 2.0 * err[3 + q]), f"gamma {gamma:g}: {err[:3]}, FP64 {err[3:]}"
