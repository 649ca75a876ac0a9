"""A test build of the library: some translation units compiled again with
other definitions and linked with the objects of the built library, to be
loaded by a child process in its place."""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

from paper_1710_05155_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def library(out_dir, units, defines) -> str:
    def compile_(unit):
        obj = os.path.join(str(out_dir), unit + ".o")
        subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, *("-D" + d for d in defines), "-I", build.INCLUDE,
                        "-c", os.path.join(build.CSRC, unit + ".cu"), "-o", obj], check=True)
        return obj

    build.build()
    with cf.ThreadPoolExecutor(max_workers=len(units)) as ex:
        objs = list(ex.map(compile_, units))
    for src in build.sources():
        if os.path.basename(src)[:-3] not in units:
            objs.append(os.path.join(build.OUT_DIR, os.path.basename(src) + ".o"))
    lib = os.path.join(str(out_dir), "libka_variant.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", lib, *objs, "-cudart", "static"], check=True)
    return lib


def run(lib, code, *args) -> str:
    """Run `code` in a child process whose library is `lib`; its output."""
    head = ("import sys; from paper_1710_05155_gb300 import build; "
            f"build.LIB = {lib!r}; build.up_to_date = lambda: True\n")
    r = subprocess.run([sys.executable, "-c", head + code, *map(str, args)], capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")])))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
