"""Kernels on a CPU, one CTA at a time, with a check of the order of their accesses to shared memory (cta.h, cta.cpp)."""
import ctypes
import os
import re
import subprocess

from paper_2608_03676_b200.build import CSRC, ROOT

HERE = os.path.dirname(os.path.abspath(__file__))
#: what a PTX statement stands for, by its instruction
PTX = {
    "rcp.approx.ftz.f32": "y = 1.0f / x;",
    "bar.sync 1,": "cta::bar(1, NT);",
    "bar.sync 2,": "cta::bar(2, NL);",
    "barrier.cta.red.or.pred": "r = cta::bar_or(3, NL, p);",
    "griddepcontrol": ";",
    "st.global.cs.v4.s32": "*p = v;",
    "mbarrier": "abort();",               # (bulk copies: the builds without them are the ones that run here)
    "createpolicy": "abort();",
}


def without_ptx(text):
    def one(m):
        found = [c for ptx, c in PTX.items() if ptx in m.group(0)]
        assert len(found) == 1, m.group(0)
        return found[0]
    text = re.sub(r"\basm\s*(?:volatile)?\s*\(.*?\);", one, text, flags=re.S)
    return re.sub(r"extern __shared__ (?:__align__\(\d+\) )?([\w ]+) (\w+)\[\];", r"\1* \2 = reinterpret_cast<\1*>(cta::dynamic);", text)


def load(folder, driver, sources):
    """The driver (C++, beside this file) and copies of the kernel sources that it includes, as a library."""
    for name in sources:
        with open(os.path.join(CSRC, name)) as f, open(os.path.join(folder, name), "w") as g:
            g.write(without_ptx(f.read()))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    flags = ["-std=c++17", "-O0", "-fPIC", "-w", "-ffp-contract=off", "-I", folder, "-I", HERE, "-I", os.path.join(ROOT, "include"), "-I",
             os.path.join(cuda, "include")]
    objs = []
    for name, extra in (("cta.cpp", []), (driver, ["-fsanitize=thread"])):
        objs.append(os.path.join(folder, name + ".o"))
        subprocess.run(["g++"] + flags + extra + ["-c", os.path.join(HERE, name), "-o", objs[-1]], check=True)
    lib = os.path.join(folder, "libcta.so")
    subprocess.run(["g++", "-shared", "-o", lib] + objs, check=True)
    so = ctypes.CDLL(lib)
    so.cta_first.restype = ctypes.c_char_p
    return so
