"""The FP64 collision of the library (equilibria as products of deviations),
compiled as plain C++, against the moment cube that every other arithmetic
takes, both measured against 80-bit arithmetic from the same start.

Tolerances.  Error: the two forms round the same number of deviation-sized
terms per population, so their errors are two samples of one distribution; over
a few thousand populations they scatter by some per cent, and a factor of 1.5 is
allowed.  Totals: a step stores 27 values per node and lattice, each rounded by
at most 2^-53 of the largest deviation; the bound is that sum over the steps
with the largest deviation taken as amplitude + 0.3 T_ref U (or rho0 U)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2203_01316_gb300", "csrc")


@pytest.fixture(scope="module")
def flow(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("flow") / "collision_flow")
    subprocess.run(["g++", "-O2", "-std=c++17", "-w", "-I", os.path.join(HERE, "host"), "-I", CSRC,
                    os.path.join(HERE, "host", "collision_flow.cpp"), "-o", exe], check=True)

    def run(*args):
        out = subprocess.run([exe] + [str(a) for a in args], check=True, capture_output=True, text=True).stdout
        return [float(x) for x in out.split()]
    return run


@pytest.mark.parametrize("kind", ["trt", "cum1st"])
@pytest.mark.parametrize("dims", [(13, 11, 1), (9, 7, 5)])
@pytest.mark.parametrize("U,amp,Tref", [(0.1, 0.05, 1.0), (1e-3, 1e-2, 1.0), (1e-3, 1e-4, 0.3), (1e-6, 1e-7, 300.0)])
def test_error_is_that_of_the_moment_cube(flow, dims, U, amp, Tref, kind):
    f, h, f_cube, h_cube, mass, energy = flow(*dims, U, amp, kind, Tref, 20, 5)
    assert f <= 1.5 * f_cube and h <= 1.5 * h_cube
    largest = amp + 0.3 * U * max(1.0, Tref)
    assert abs(mass) <= 20 * 27 * 2.0 ** -53 * largest and abs(energy) <= 20 * 27 * 2.0 ** -53 * largest


@pytest.mark.parametrize("kind", ["trt", "cum1st"])
@pytest.mark.parametrize("Tref", [1.0, 300.0])
def test_rest_state_stays(flow, Tref, kind):
    assert flow(3, 4, 5, 0.0, 0.0, kind, Tref, 100, 1) == [0.0] * 6


def test_totals_hold_over_many_steps(flow):
    mass, energy = flow(8, 8, 1, 1e-3, 1e-3, "cum1st", 1.0, 2000, 3)[4:]
    bound = 2000 * 27 * 2.0 ** -53 * (1e-3 + 0.3e-3)
    assert abs(mass) <= bound and abs(energy) <= bound
