"""Test helper: a small program linked with the library's host object (csrc/host.cu), for host functions that the
C ABI does not export.  `main` gets the command line; its standard output is returned by lines."""
import os
import subprocess

from paper_2105_08806_gb300 import build as B

PROLOGUE = """
#include <cstdio>
#include <cstdlib>
#include "host.cuh"
void pg_free_batch(BatchState *) {}
"""


def host_program(folder, body):
    B.build()
    src, exe = str(folder / "prog.cu"), str(folder / "prog")
    open(src, "w").write(PROLOGUE + body)
    subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), "-o", exe, src,
                    os.path.join(B.BUILD, "host.o")], check=True, capture_output=True)

    def run(args=(), stdin=""):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True, input=stdin).stdout
        return out.splitlines()
    return run
