"""The arithmetic of the device headers compiled for the host: accuracy of the double precision column multipliers."""
import os
import subprocess

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")
CSRC = os.path.join(os.path.dirname(os.path.dirname(HOST)), "paper_1809_07592_gb300", "csrc")


def compiled(name, tmp_path):
    exe = str(tmp_path / name)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", HOST, "-I", CSRC, os.path.join(HOST, name + ".cpp"), "-o", exe],
                   check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout


def test_double_precision_column_multipliers(tmp_path):
    """A multiplier is at most one product of two rounded roots. In units u = 2^-53: each part of a root is off by
    at most u/2, so a root by sqrt(1/2) u; the product rounds each part by at most (|ac| + |bd|) u + |x| u <= 2 u,
    so by 2 sqrt(2) u. Together 3 sqrt(2) u, and terms of order u^2."""
    worst = max(float(v) for v in compiled("multipliers", tmp_path).split())
    assert 0 < worst <= 3 * 2 ** 0.5 * (1 + 1e-9)


def test_single_precision_stage_powers(tmp_path):
    """A power is a rounded root or one squaring (1 - 2 s^2, 2 s c) away from one. In units u = 2^-24: s and c are off by
    at most u/2, which moves the parts by at most 4 |s| u/2 and 2 (|s| + |c|) u/2, 2 u and sqrt(2) u; each is
    rounded once more, by u/2. Together hypot(2.5, 1.92) u = 3.16 u, and terms of order u^2."""
    worst = float(compiled("powers", tmp_path))
    assert 0 < worst <= (2.5 ** 2 + (2 ** 0.5 + 0.5) ** 2) ** 0.5 * (1 + 1e-6)


def test_table_angles_are_reduced_exactly(tmp_path):
    """The angle of a table root is a quotient below one half of a quarter turn, rounded once: by 2^-55 of it at most."""
    assert 0 < float(compiled("turns", tmp_path)) <= 1
