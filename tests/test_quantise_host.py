"""Quantisation and range truncation settled in float-float (quantise_ff,
truncate_ff, compiled for the host) equal the double evaluations wherever they
settle one; they settle every point away from half-integers and nearly all rays."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_float_float_quantisation_and_truncation_equal_double(tmp_path):
    exe = str(tmp_path / "quantise_check")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-Xcompiler",
                    "-ffp-contract=off", "-x", "cu", os.path.join(HERE, "host", "quantise_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.returncode
    t = out.stdout.split()
    points, settled, random, random_settled, rays, rays_settled = (int(t[i]) for i in (1, 3, 5, 7, 9, 11))
    assert points == 2000000 and random > 1000000 and random_settled == random
    assert settled < points              # built half-integers are declined
    assert rays > 500000 and rays_settled > 0.999 * rays
