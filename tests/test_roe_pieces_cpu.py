"""The pieces of the integer-pipe arithmetic (csrc/fv_roe.h, compiled for the
host), each against what its comment says."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_pieces_do_what_they_say(tmp_path):
    exe = str(tmp_path / "roe_pieces")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-Wno-unknown-pragmas", "-o", exe,
                    os.path.join(HERE, "native", "roe_pieces.cpp")], check=True)
    p = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.splitlines()[-1] == "ok", p.stdout + p.stderr
