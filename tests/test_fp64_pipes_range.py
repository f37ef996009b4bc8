"""The integer-pipe binary64 operations of csrc/fp64_pipes.cuh at the ends of
their range, compiled for the host: a quotient below 2^-1022 is refused, and
nearly nothing else is."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_ends_of_the_range(tmp_path):
    exe = str(tmp_path / "pipes_range")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe,
                           os.path.join(HERE, "fp64_pipes_range_host.cpp")])
    for seed in (1, 2):
        n = 500000
        differ, normal, refused = map(int, subprocess.check_output([exe, str(n), str(seed)]).split())
        assert differ == 0
        assert normal > 3.5 * n and refused < 0.15 * n
