"""Programmatic dependent launches: a kernel that waits inside itself for the kernel before it
(pdl_wait) starts while that one still writes, so what earlier kernels of the chain write must not be
declared read-only for its lifetime (`const T *__restrict__`), and its sweep partials and inputs are
loaded past the non-coherent cache.  Read from the sources: the fault has no visible effect until a
compiler uses the qualifier."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_03683_gb300", "csrc")
# what no kernel of a chain writes: the plan's tables, the coefficients, the rows' total rates
CONSTANTS = {"tiles", "tc", "prow", "pmap", "R"}


def kernels():
    """(name, parameter list, body) of every __global__ function."""
    for fn in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, fn)).read()
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(", src):
            i = src.index(")", m.end())
            params = src[m.end():i]
            j = src.index("{", i)
            depth, k = 1, j + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[k], 0)
                k += 1
            yield m.group(1), params, src[j:k]


def test_chained_kernels_declare_only_constants_read_only():
    chained = {n: (p, b) for n, p, b in kernels() if "pdl_wait()" in b}
    assert {"k_fin_net", "k_fin_vjp_net", "k_stream_sym_unit", "k_vjp_tiles", "k_stream_c32",
            "k_stream_c32_half"} <= set(chained)
    for name, (params, body) in chained.items():
        read_only = set(re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params))
        assert read_only <= CONSTANTS, f"{name}: {sorted(read_only - CONSTANTS)} may be written while it runs"
        # the epilogues' partials and the sweeps' inputs go through L2
        for buf in ("tp", "fg", "lam"):
            if re.search(rf"const\s+[\w:]+\s*\*\s*{buf}\b", params):
                assert not re.search(rf"[^\w]{buf}\[", body), f"{name}: plain load of {buf}"
