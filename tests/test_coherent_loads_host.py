"""CPU check of the loads of kernels that may be launched before their predecessors have finished.

Such a kernel (it begins with pdl_begin) is alive while the kernel before it writes its inputs.
Non-coherent loads -- __ldg, and loads the compiler may make non-coherent through const
__restrict__ pointers -- are specified only for memory that nothing writes during the kernel's
whole life, so they are kept to the tables that no kernel writes.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2007_13394_gb300", "csrc")
TABLES = {"tw", "ksq", "winv", "kvec0", "amp", "tab"}  # copied from the host, written by no kernel


def _code(f):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())


def _functions(code):
    """(signature, body) of every __global__ or __device__ function."""
    out = []
    for m in re.finditer(r"__(?:global|device)__[^;{]*\{", code):
        depth, i = 1, m.end()
        while depth:
            depth += (code[i] == "{") - (code[i] == "}")
            i += 1
        out.append((m.group(0), code[m.end():i]))
    return out


def _early_files():
    return [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and "pdl_launch(" in _code(f)]


def test_there_are_early_kernels():
    files = _early_files()
    assert "k_sort.cu" in files and "k_fft.cu" in files and "k_power.cu" in files
    for f in files:  # every kernel of these files waits for its predecessors first
        for sig, body in _functions(_code(f)):
            if "__global__" in sig:
                assert body.lstrip().startswith("pdl_begin();"), (f, sig[:120])


def test_const_restrict_only_on_tables():
    for f in _early_files():
        for sig, _ in _functions(_code(f)):
            names = set(re.findall(r"const \w+\*\s*__restrict__\s+(\w+)", sig))
            # shared memory of the CTA, passed to its own device functions
            shared = {"run_lo", "run_pre", "th"} if "__device__" in sig else set()
            assert names <= TABLES | shared, (f, sig[:120], names - TABLES)


def test_ldg_only_on_tables():
    for f in _early_files() + ["fft_engine.cuh"]:
        for arg in re.findall(r"__ldg\(\s*([\w.]+)", _code(f)):
            assert arg.split(".")[-1] in TABLES, (f, arg)
