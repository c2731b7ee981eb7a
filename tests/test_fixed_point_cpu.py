"""The fixed-point pair arithmetic of the binary64 mode against extended precision, on the host."""
import os
import subprocess


def test_pair_terms_within_their_bounds(tmp_path):
    here = os.path.dirname(os.path.abspath(__file__))
    exe = str(tmp_path / "fixed_pair_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-o", exe,
                    os.path.join(here, "fixed_pair_check.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout.split()
    used, close, wrong = (int(x) for x in out[:3])
    worst_f, worst_p, bias, worst_4, worst_heavy = (float(x) for x in out[3:])
    assert used > 100000 and close > 10000 and wrong == 0, out
    assert worst_f <= 1.0 and worst_p <= 1.0, out  # in units of the stated bounds
    assert abs(bias) < 2.0 ** -58, out  # no systematic part
    assert worst_4 <= 2.0, out  # r^2 a power of four: F within 2^-56
    # terms of 1 whose last place is 2^-53, cut off there in each component
    assert worst_heavy <= 3 ** 0.5, out
