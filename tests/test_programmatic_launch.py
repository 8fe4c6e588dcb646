"""Order of kernels that overlap by programmatic stream serialization: a grid that started early is
ordered after the one before only by griddepcontrol.wait (PTX ISA), and a later launch, or a graph node
with a full edge from the last grid alone, is ordered after the earlier ones only through that chain.
So a kernel that lets its dependents start (griddepcontrol.launch_dependents) has to wait itself,
after its last store, on every path to its end. Read from the source, without a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1307_0719_gb300", "csrc")


def _kernels(src):
    """(name, body) of every __global__ function definition."""
    for m in re.finditer(r"__global__\b[^;{]*?(\w+)\s*\((?!\s*\()[^;{]*\)\s*\{", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.group(1), src[m.end():i - 1]


def test_kernels_that_release_dependents_wait_for_their_prerequisites():
    found = 0
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        n = len(re.findall(r'asm volatile\("griddepcontrol\.launch_dependents', src))
        seen = 0
        for name, body in _kernels(src):
            if "griddepcontrol.launch_dependents" not in body:
                continue
            seen += 1
            # the wait is the last statement, and nothing returns before it
            assert re.search(r'asm volatile\("griddepcontrol\.wait;"[^;]*\);\s*$', body), (f, name)
            assert "return" not in re.sub(r"\[[&=]?\]\s*\([^)]*\)\s*\{[^}]*\}", "", body), (f, name)
        assert seen == n, (f, "launch_dependents outside a kernel body")
        if "cudaLaunchAttributeProgrammaticStreamSerialization" in src:
            assert seen, (f, "overlapped launches of a kernel that neither releases nor waits")
        found += seen
    assert found
