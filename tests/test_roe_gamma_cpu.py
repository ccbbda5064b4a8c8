"""The integer-pipe Roe flux (csrc/fv_roe.h, compiled for the host) in its form for
large gamma, where H~ - c~ |u~_n| turns negative (gamma > 3) and c~^2 is a small difference of
large numbers: nearly every face is taken, and none is further from long double
than the FP64 evaluation (or 4 units: test_roe_cpu.py)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CASES = 20000


def test_large_gamma_is_taken_and_no_further_from_exact_than_fp64(tmp_path):
    exe = str(tmp_path / "roe_gamma")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-Wno-unknown-pragmas", "-o", exe,
                    os.path.join(HERE, "native", "roe_gamma.cpp")], check=True)
    p = subprocess.run([exe, str(CASES)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stdout + p.stderr
    lines = p.stdout.splitlines()
    assert len(lines) == 88
    for line in lines:
        name, dim, refused, worst, rms, worst64, rms64 = line.split()
        assert int(refused) <= 0.1 * CASES, line
        assert float(worst) <= max(4.0, float(worst64)), line
        assert float(rms) <= float(rms64), line
