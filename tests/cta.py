"""Kernels on a CPU, one CTA at a time, with a check of the order of their accesses to shared memory (cta.h, cta.cpp)."""
import ctypes
import os
import re
import subprocess

from paper_2608_03676_b200.build import CSRC, ROOT

HERE = os.path.dirname(os.path.abspath(__file__))
#: what a PTX statement stands for, by how it begins; {0}, {1}, ... are its operands
PTX = {
    "rcp.approx.ftz.f32": "{0} = 1.0f / ({1});",
    "min.NaN.f32": "{0} = cta::least({operands});",
    "max.NaN.f32": "{0} = cta::largest({operands});",
    "mul.rn.f32x2": "{0} = cta::pack(cta::low({1}) * cta::low({2}), cta::high({1}) * cta::high({2}));",
    "add.rn.f32x2 %0, %0": "{0} = cta::pack(cta::low({0}) + cta::low({1}), cta::high({0}) + cta::high({1}));",
    "fma.rn.f32x2 %0, %1, %2, %0": "{0} = cta::pack(fmaf(cta::low({1}), cta::low({2}), cta::low({0})), fmaf(cta::high({1}), cta::high({2}), cta::high({0})));",
    "mov.b64 {": "{{ {0} = cta::low({2}); {1} = cta::high({2}); }}",
    "mov.b64 %0": "{0} = cta::pack({1}, {2});",
    "bar.sync 1,": "cta::bar(1, {0});",
    "bar.sync 2,": "cta::bar(2, {0});",
    "{ .reg .pred p, q; setp.ne.s32 p, %1, 0; barrier.cta.red.or.pred q, 3, %2": "{0} = cta::bar_or(3, {2}, {1});",
    "griddepcontrol": ";",
    "st.global.cs.v4.s32": "*({0}) = make_int4({1}, {2}, {3}, {4});",
    "st.global.u32": "*({0}) = {1};",
    "ld.shared.u32": "{0} = *static_cast<uint32_t*>(cta::shared({1}));",
    "ld.shared.v2.u32": "{{ const uint2 q = *static_cast<uint2*>(cta::shared({2})); {0} = q.x; {1} = q.y; }}",
    "st.shared.u32": "*static_cast<uint32_t*>(cta::shared({0})) = {1};",
    "red.shared.max.u32": "atomicMax(static_cast<uint32_t*>(cta::shared({0})), {1});",
    "red.shared.and.b32": "atomicAnd(static_cast<uint32_t*>(cta::shared({0})), {1});",
    "red.shared.or.b32": "atomicOr(static_cast<uint32_t*>(cta::shared({0})), {1});",
    "red.shared.add.u32": "atomicAdd(static_cast<uint32_t*>(cta::shared({0})), {1});",
    "{ .reg .pred p; setp.ne.u32 p, %2, 0; @p red.shared.max.u32": "if ({2}) atomicMax(static_cast<uint32_t*>(cta::shared({0})), {1});",
    "{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.shared.u32": "if ({2}) *static_cast<uint32_t*>(cta::shared({0})) = {1};",
    "{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.global.u32": "if ({2}) *({0}) = {1};",
    "bfind.u32": "{0} = ({1}) ? 31u - (uint32_t)__builtin_clz({1}) : ~0u;",
    # bulk copies and clusters: the builds without them are the ones that run here
    "mbarrier": "abort();", "{\\n\\t.reg .pred p;\\n\\tmbarrier": "abort();", "fence.mbarrier": "abort();", "cp.async.bulk": "abort();",
    "createpolicy": "abort();", "barrier.cluster": "abort();", "mapa": "abort();", "ld.shared::cluster": "abort();",
}


def operands(text):
    """The expressions of `"constraint"(expression)`, in order."""
    found = []
    for m in re.finditer(r'"[=+]?[a-z]"\s*\(', text):
        end, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[end], 0)
            end += 1
        found.append(text[m.end():end - 1])
    return found


def without_ptx(text):
    def one(m):
        ptx = re.match(r'\s*"([^"]*)"', m.group(1)).group(1)
        found = [c for begin, c in PTX.items() if ptx.startswith(begin)]
        assert len(found) == 1, m.group(0)
        ops = operands(m.group(1))
        return found[0].format(*ops, operands=", ".join(ops))
    text = re.sub(r"\basm\s*(?:volatile)?\s*\((.*?)\);", one, text, flags=re.S)
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
