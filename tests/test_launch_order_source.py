"""What the kernels' sources must keep to so that calls on one stream take effect in order (tetra_device.cuh, programmatic
dependent launch): read from the source, because a launch that starts too early is not an error that a run shows."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35465_b200", "csrc")


def kernels():
    """name -> (parameters, body) of every __global__ function, comments taken out."""
    found = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = open(os.path.join(CSRC, f)).read()
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(([^)]*)\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            found[m.group(1)] = (m.group(2), text[m.end():at])
    return found


KERNELS = kernels()


def test_the_kernels_are_found():
    assert {"k_pack", "k_q4_pack", "k_gemv_list", "k_gemv_batched", "k_gemv_units", "k_q4_gemv", "k_q4_list_main",
            "k_decode_packed", "k_q4_rows", "k_prepare_x"} <= set(KERNELS)


def test_a_kernel_that_writes_packed_codes_does_not_release_its_dependents():
    writers = [name for name, (params, _) in KERNELS.items()
               if any("packed" in p and "const" not in p for p in params.split(","))]
    assert set(writers) >= {"k_pack", "k_q4_pack"}
    for name in writers:
        assert "pdl_release" not in KERNELS[name][1], name


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_a_kernel_that_releases_its_dependents_waits_for_its_predecessors(name):
    body = KERNELS[name][1]
    assert "pdl_release" not in body or "pdl_wait" in body
