"""What the kernels' sources have to say for a launch that may start before the one it follows has ended."""
import os
import re

import paper_2609_35800_gb300 as hg

CSRC = os.path.join(os.path.dirname(os.path.abspath(hg.__file__)), "csrc")


def _kernels():
    """(name, body) of every __global__ function."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"__global__ void(?: __(?:launch_bounds|maxnreg)__\([^{;]*?\))?\s+(\w+)\(", text):
            start = text.index("{", m.end())
            depth, i = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield m.group(1), text[start + 1:i - 1]


def test_every_dependent_launch_waits_before_it_touches_memory():
    """A grid sees what the grids before it wrote only after its own wait (no other grid's wait or trigger stands
    in for it): every kernel waits on every path, before its first copy, load or store of global memory."""
    seen = []
    for name, body in _kernels():
        if name == "wait_probe_kernel":  # an ordinary launch
            continue
        code = re.sub(r"//[^\n]*", "", body)
        wait = re.search(r"^  grid_dependency_wait\(\);", code, re.M)  # a statement of its own, under no condition
        assert wait, name
        assert code.count("grid_dependency_wait()") == 1, name
        before = code[:wait.start()]
        assert not re.search(r"stage_rows|ldg|cp_async|bulk_g2s|tma_load|->|reinterpret_cast<const [^>]*\*>\(p\.", before), name
        assert not re.findall(r"return", before.replace("if ((int)blockIdx.x >= p.total_items) return;", "")), name
        seen.append(name)
    assert {"decode_kernel", "quantize_tiles_kernel", "dequantize_kernel", "append_kernel", "clear_kernel",
            "salient_norm_kernel", "salient_select_kernel"} == set(seen)
