"""Builds internals.cu (or internals_solver.cu) against libovl.so and loads it: host functions of the library that are tested
without an entry point."""
import ctypes
import os
import subprocess

from paper_1410_7170_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(name="internals"):
    so = build.build()
    out = os.path.join(HERE, "_build", "lib%s.so" % name)
    os.makedirs(os.path.dirname(out), exist_ok=True)
    src = os.path.join(HERE, name + ".cu")
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(so)):
        subprocess.run([build._nvcc(), *build.ARCH, "-O1", "-std=c++17", "-w", "--expt-relaxed-constexpr", "-shared",
                        "-Xcompiler", "-fPIC", src, so, "-Xlinker", "-rpath=" + os.path.dirname(so), "-o", out],
                       check=True)
    return ctypes.CDLL(out)
