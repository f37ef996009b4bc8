"""The integer-pipe binary64 operations of csrc/fp64_pipes.cuh, compiled for
the host: every result equals the host's IEEE operation bit for bit, also with
the hardware approximations they start from off by their full error bounds."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_operations_equal_ieee(tmp_path):
    exe = str(tmp_path / "pipes")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe,
                           os.path.join(HERE, "fp64_pipes_host.cpp")])
    for seed in (1, 2):
        differ, refused = map(int, subprocess.check_output([exe, "2000000", str(seed)]).split())
        assert differ == 0
        assert 0 < refused < 1000000  # only operands far outside 2^-511 .. 2^512
