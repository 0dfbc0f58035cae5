"""csrc/launch.cuh on the host, with a fake of the runtime calls it makes (tests/launch_fake.cpp):
the attributes are set once, a launch that fails because they are gone is repeated once, and an error
that an earlier call left behind makes no kernel run twice (its counters would count twice)."""
import os
import subprocess

from paper_2411_14631_gb300 import abi, build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_launch_kernel(tmp_path):
    exe = str(tmp_path / "launch_fake")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I" + build.CSRC, "-I" + include, "-x", "c++",
                        os.path.join(HERE, "launch_fake.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    got = {n: tuple(int(v) for v in rest) for n, *rest in (line.split() for line in out.splitlines())}
    assert got == {"first": (abi.OK, 1, 2), "cached": (abi.OK, 1, 0),
                   "left_behind": (abi.ECUDA, 1, 0),
                   "attributes_lost": (abi.OK, 1, 2),
                   "refused": (abi.ECUDA, 0, 0), "after": (abi.OK, 1, 0)}
