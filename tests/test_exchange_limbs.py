"""The grid exchange's sums travel as three words that CTAs add to with atomics: the
limbs of up to 511 x 8 (or 255 x 16) addends must join to the exact 128-bit sum, with
the counts and the exception marks apart.  Built for the host from the kernels' header."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_limbs_join_to_the_exact_sum(tmp_path):
    exe = str(tmp_path / "limbs")
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "exchange_limbs_driver.cpp")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
