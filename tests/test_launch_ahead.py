"""Kernels launched ahead of their predecessor's end (launch_after) read what it
writes, so none of their inputs may be declared read-only for the kernel's whole
life: `const __restrict__` allows non-coherent loads, which require that."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_03426_gb300", "csrc")


def _kernels():
    """(name, parameters, body) of every kernel definition."""
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", src):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            j = src.index("\n}", i)
            yield m.group(1), src[m.end():i - 1], src[i:j]


def test_kernels_launched_ahead_declare_no_read_only_inputs():
    ahead = [(name, par) for name, par, body in _kernels() if "after_previous()" in body]
    assert {"k_step_stored", "k_step_periodic", "k_step_periodic4", "k_step_fix", "k_adj_fix", "k_adj_step_periodic",
            "k_adj_step_periodic4", "k_flush_faces", "k_lerp", "k_pad_coarse64", "k_coupled_nu", "k_fused",
            "k_xfused"} <= {n for n, _ in ahead}
    bad = [(n, p) for n, p in ahead if re.search(r"const\s+\w+\s*\*\s*(const\s+)?__restrict__", p)]
    assert not bad, bad


def test_every_kernel_launched_ahead_waits():
    names = set()
    for f in glob.glob(os.path.join(CSRC, "*.cu")):
        for call in re.findall(r"(?:launch_after(?:_if)?\(|const auto k =)(.*?);", open(f).read(), flags=re.S):
            names |= set(re.findall(r"\bk_\w+", call))
    waits = {n for n, _, body in _kernels() if "after_previous()" in body}
    assert names and names <= waits, names - waits
