"""Host programs on the library's own headers: the C++ that decides a call's route, and its device functions compiled for the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_00237_gb300", "csrc")


def build(source, folder):
    """The program's path; `source` is C++ that may include the library's headers and call its functions."""
    from paper_2205_00237_gb300 import build as B
    lib = B.build()
    src, exe = os.path.join(str(folder), "main.cu"), os.path.join(str(folder), "main")
    with open(src, "w") as f:
        f.write(source)
    r = subprocess.run([os.environ.get("NVCC", "nvcc"), *B.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                        "-Xcompiler", "-ffp-contract=off", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "tests"), src, "-o", exe,
                        lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return exe


def run(exe, lines):
    """One line of numbers in, one line of numbers out."""
    text = "\n".join(" ".join(repr(float(x)) for x in ln) for ln in lines) + "\n"
    r = subprocess.run([exe], input=text, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return [[float(x) for x in ln.split()] for ln in r.stdout.splitlines()]
