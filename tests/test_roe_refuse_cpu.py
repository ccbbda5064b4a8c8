"""Faces with a side of negative pressure are not for the integer-pipe Roe flux
(csrc/fv_roe.h, compiled for the host): it has to report every one of them, at
any ratio of kinetic to total energy, so that the FP64 evaluation decides what
becomes of them."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_face_of_negative_pressure_is_taken(tmp_path):
    exe = str(tmp_path / "roe_refuse")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-Wno-unknown-pragmas", "-o", exe,
                    os.path.join(HERE, "native", "roe_refuse.cpp")], check=True)
    p = subprocess.run([exe, "400000"], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stdout + p.stderr
    lines = p.stdout.splitlines()
    assert len(lines) == 8
    for line in lines:
        name, dim, found, taken = line.split()
        assert int(found) > 300000, line
        assert int(taken) == 0, line
