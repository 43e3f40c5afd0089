"""The bounds-checking build covers the grouping: every kernel of group.cu that
stores at a computed index checks it (read from the source, so without a GPU)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_02259_gb300", "csrc")


def _bodies(src, head):
    """{name: text} of the functions whose declaration matches `head`."""
    out = {}
    for m in re.finditer(head, src):
        i = src.index("{", m.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[j], 0)
            j += 1
        out[m.group(1)] = src[i:j]
    return out


def test_every_grouping_kernel_checks_its_indices():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "group.cu")).read())
    helpers = _bodies(src, r"__device__ __forceinline__ void (write_item|mark_neighbour)\(")
    kernels = _bodies(src, r"__global__ void __launch_bounds__\(kGroupThreads\)\s+(k_\w+)\(")
    assert set(kernels) == {"k_runs", "k_pairs", "k_rank", "k_offsets", "k_place", "k_compact"}
    for name, text in {**helpers, **kernels}.items():
        checked = "APIC_DBG_CHECK" in text or all(h + "(" in text for h in helpers)
        assert checked, name


def test_the_gather_checks_the_order_before_it_uses_it():
    src = open(os.path.join(CSRC, "kernels.cu")).read()
    text = _bodies(src, r"__global__ void (k_gather)\(")["k_gather"]
    before = text[:text.index("APIC_DBG_CHECK(g >= 0 && g < n")]
    assert "scene_of_particle" not in before and "g < 0" not in before
