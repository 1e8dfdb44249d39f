"""What the kernels' sources must keep to, read from the source because a run does not show it: calls on one stream take
effect in order (tetra_device.cuh, programmatic dependent launch), and launches ask the device for its size."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35465_b200", "csrc")


def sources():
    """(file name, text without comments) of the CUDA sources."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, f)).read()
            yield f, re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def kernels():
    """name -> (parameters, body) of every __global__ function."""
    found = {}
    for _, text in sources():
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


def waits_before_it_reads_and_releases(body, workspace):
    """A kernel whose dependents read the workspace ahead of their own wait: it waits for what wrote it first of all."""
    return body.index("pdl_wait") < body.index("pdl_release") and workspace not in body[:body.index("pdl_wait")]


def test_the_kernel_ahead_of_the_planned_list_waits_before_it_reads_the_plan_or_releases():
    body = KERNELS["k_prepare_x"][1]
    assert waits_before_it_reads_and_releases(body, "ws")
    assert not waits_before_it_reads_and_releases(body.replace("pdl_wait", "X").replace("pdl_release", "pdl_wait").replace("X", "pdl_release"), "ws")
    assert not waits_before_it_reads_and_releases(body.replace("pdl_wait", "p = ws; pdl_wait"), "ws")


def test_no_launch_is_written_for_one_number_of_multiprocessors():
    for f, text in sources():
        assert not re.search(r"\b148\b", text), f


def test_clusters_stay_within_what_the_scale_tables_addresses_hold():
    """A shared-memory address of a cluster's CTA holds its rank from bit 24 on; the decoder keeps one shifted left."""
    text = "".join(t for _, t in sources())
    shift = int(re.search(r"kNormShift = (\d+);", text).group(1))
    assert re.search(r"kNormClusterMax = 1 << \(32 - 24 - kNormShift\);", text)
    assert int(re.search(r"kBatMaxCluster = (\d+);", text).group(1)) <= 1 << (32 - 24 - shift)
    users = [f for f, t in sources() if "cudaLaunchAttributeClusterDimension" in t]
    assert users == ["tetra_batched.cu"] and "static_assert(kBatMaxCluster <= kNormClusterMax" in text
