"""Kernels that may start before their predecessors end (launch_pdl) do not
declare what those may still be writing read-only: the state, the potential and
tables made by a kernel are taken without __restrict__ and read without __ldg,
which a compiler may move above the wait or serve from a cache that does not
see the writes.  Only tables copied by the host, in full before the launch, are."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_4090_gb300", "csrc")
HOST_TABLES = {"kr64", "K", "disp", "items"}      # the kernel table, the semigroup's K and displacements, batch fields


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.inc"))):
        out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", open(f).read())
    return out


def test_nothing_written_by_a_predecessor_is_read_only():
    src = _sources()
    text = "\n".join(src.values())
    names = set()
    for t in src.values():
        for m in re.finditer(r"launch_pdl\((.*?)st(?:ream)?,", t, re.S):
            names |= set(re.findall(r"\b(\w+_kernel\w*|split_\w+)\b", m.group(1)))
        for m in re.finditer(r"\bk = (\w+)<", t):            # hjlo_kern.inc chooses the pass kernel first
            names.add(m.group(1))
    assert {"pass_kernel", "pass_kernel_dense", "integral_table_kernel", "split_emit"} <= names
    assert "adjoint_pass_kernel" in names
    for name in sorted(names):
        sig = re.search(r"__global__ void (?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?%s\((.*?)\)\s*\{" % name, text,
                        re.S)
        assert sig, name
        for p in re.findall(r"\*\s*__restrict__\s+(\w+)", sig.group(1)):
            assert p in HOST_TABLES, (name, p)
    for f, t in src.items():
        for arg in re.findall(r"__ldg\(\s*([\w.>\-]+)", t):
            assert arg.split(".")[-1].split(">")[-1] in HOST_TABLES, (f, arg)
