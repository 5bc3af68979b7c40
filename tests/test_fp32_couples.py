"""The kernel's order of the pair sums, mirror couples (a, b, c) + (a, b, -c)
first, in the column emulator of tests/fp32_floor (the plain slit, 1000 steps;
see test_fp32_floor.py): in FP64 it is the oracle's scheme, and in FP32, with the
kernel's collision, the couples' mean-field differences cancel along the walls
bit for bit, so the column keeps a net x-force of 1.7e-7 of the drive where pairs
summed one by one keep 2.2e-5.  Errors within the bounds that the FP32 slit has
on the GPU (u_x 1e-4, flux 2e-5, n 1e-6; measured 3.0e-5, 1.3e-5, 1.6e-7)."""
from test_fp32_floor import _errors, _run, reference  # noqa: F401


def test_couples_in_fp64_are_the_oracle(reference):  # noqa: F811
    x, inner, drive = _run("double", "dd", "couple")
    en, eux, euz, _ = _errors(x, reference)
    assert en < 1e-8 and eux < 1e-8 and euz < 1e-8
    assert abs(inner) < 1e-9 * drive


def test_couples_leave_no_net_force_along_the_walls(reference):  # noqa: F811
    x, inner, drive = _run("float", "fc", "couple")
    _, inner_one, _ = _run("float", "fc", "sym")
    en, eux, _, ef = _errors(x, reference)
    assert abs(inner) < 1e-6 * drive and abs(inner) < 0.1 * abs(inner_one)
    assert en < 1e-6 and eux < 1e-4 and ef < 2e-5
