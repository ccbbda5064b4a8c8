"""The integer-pipe Roe flux of the kernels (csrc/fv_roe.h), compiled for the
host and compared with the same flux in long double.

The tolerance.  Errors are measured against the magnitudes that a component
sums, in units of 2^-53 of them.  The result is rounded once (1 unit; the mass
flux twice), and every intermediate keeps 56 bits or more of those magnitudes
through at most 16 truncations of 1/8 unit: 4 units, where no difference of
nearly equal terms is taken.  Where one is (|u~_n| - c~ near a sonic point,
E - rho |u|^2 / 2 at a high Mach number) the FP64 evaluation loses digits too,
and its worst error is the bound; over a whole regime the rms error is not
above that of the FP64 evaluation."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_integer_flux_is_no_further_from_exact_than_fp64(tmp_path):
    exe = str(tmp_path / "roe_check")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-Wno-unknown-pragmas", "-o", exe,
                    os.path.join(HERE, "native", "roe_check.cpp")], check=True)
    p = subprocess.run([exe, "100000"], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stdout + p.stderr
    lines = p.stdout.splitlines()
    assert len(lines) == 11
    for line in lines[:-1]:
        name, dim, refused, worst, rms, worst64, rms64 = line.split()
        assert int(refused) == 0, line
        assert float(worst) <= max(4.0, float(worst64)), line
        assert float(rms) <= float(rms64), line
    assert lines[-1] == "refused 30 of 30"
