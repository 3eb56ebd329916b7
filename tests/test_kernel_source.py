"""Kernels launched with programmatic serialisation run beside the launch before them: what a
launch can write must not be read through the read-only path, whose loads are for data that
does not change while the kernel runs and may be moved above the wait."""
import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2301_08068_gb300", "csrc",
                   "rmp_kernels.cu")
# written at upload only, complete before any launch that reads it
UPLOADED = ("&kReverse5", "&m.table", "top ", "box ", "brick ", "reinterpret_cast<const uint32_t*>(m.bricks)",
            "prims32 ")


def kernels(text):
    """name -> (parameters, body) of every __global__ function."""
    out = {}
    for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        out[m.group(1)] = (text[m.end():i - 1], text[i:text.index("\n}\n", i)])
    return out


def test_no_read_only_loads_beside_a_predecessor():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    found = kernels(text)
    launched = set(re.findall(r"launch_after(?:_shared)?\(\s*(\w+_kernel)", text))
    assert {"raycast_rmp_kernel", "raycast_batch_kernel", "raycast_state_kernel", "batch_prep_kernel",
            "scan_rmp_kernel", "esdf_eval_kernel"} <= launched
    for name in launched:
        params, body = found[name]
        assert body.index("wait_previous()") < body.index("launch_next()"), name
        for param in params.split(","):
            assert "__restrict__" not in param or re.search(r"\bprims(32)?$", param.strip()), (name, param)
    evaluation = text[:text.index("dense_bricks_kernel")]     # the map build kernels follow
    for arg in re.findall(r"__ldg\(([^;]*)", evaluation):
        assert arg.startswith(UPLOADED), arg
