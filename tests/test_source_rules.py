"""Rules that every kernel source keeps and that no run can show to be broken: what would hold only by luck, on
the code as compiled today."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_02191_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def code(path):
    """The file without comments."""
    text = open(path).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def body(text, name):
    """The body of the kernel `name`."""
    at = text.index("{", re.search(r"\b%s\s*\([^;]*?\)\s*(?=\{)" % name, text).start())
    depth = 0
    for k in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[at:k + 1]
    raise AssertionError(name)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_read_only_loads(path):
    # kernels are set up while the one before them still writes (launch_next): nothing of a call's data is
    # read-only for their lifetime, and an invariant load may be moved to before the wait
    text = code(path)
    text = re.sub(r"T load_settled\(const T\* p\) \{[^}]*\}", "", text)
    assert not re.search(r"\b__ldg\s*\(|\.nc\b|__restrict__", text)
    # loads in assembly stay behind the wait only as volatile ones
    assert not re.search(r'asm\s*\(\s*"ld\.global', text)


def test_settled_loads_follow_a_settled_kernel():
    # the one kernel with read-only loads: what it reads with them was written before its predecessors, which
    # let it take its place only after their own wait
    text = {os.path.basename(p): code(p) for p in SOURCES}
    used = {n: len(re.findall(r"\bload_settled\(", t)) for n, t in text.items()}
    apply = body(text["robe_strips.cu"], "strip_apply_kernel")
    assert {n for n, k in used.items() if k} == {"robe_device.cuh", "robe_strips.cu"} and used["robe_device.cuh"] == 1
    assert used["robe_strips.cu"] == len(re.findall(r"\bload_settled\(", apply))
    assert set(re.findall(r"\bload_settled\(\(?(\w+(?:\.\w+)?)", apply)) <= {"a.K", "a.V", "a.grad_out"}
    prepare = text["robe_strips.cu"][text["robe_strips.cu"].index("void launch_strips_prepare"):]
    launched = re.findall(r"launch_next\((\w+)", prepare[:prepare.index("void launch_strips(")])
    assert launched
    for name in launched:
        assert re.match(r"\{\s*follow_settled\(\);", body(text["robe_strips.cu"], name)), name


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_warp_calls_name_lanes_that_are_sure_to_arrive(path):
    # the lanes active at one call need not be those at the next: a mask read from the hardware is no promise
    assert "__activemask" not in code(path)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_every_gradient_read_is_checked_in_the_index_check_build(path):
    # a read of grad_out stands behind a check that names it, at most four lines further up
    lines = code(path).splitlines()
    for n, line in enumerate(lines):
        if re.search(r"(__ldcs|__ldca|load_settled)\((rows? \+|grad \+|ge\)|a\.grad_out)", line):
            assert re.search("ROBE_CHK_GRAD|ROBE_DBG_GRAD_POS", " ".join(lines[max(0, n - 4):n + 1])), (n + 1, line)


def test_index_check_run_picks_every_test_of_a_kernel_path():
    # a test of the parity file runs on the index-check build too, unless it is one of those named here: workloads at full
    # size (run against it by hand), and what launches no kernel of its own
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    pick = re.search(r"pick = \((.*?)\)\n", open(os.path.join(root, "tests", "test_gpu_debug_build.py")).read(), re.S).group(1)
    words = re.sub(r'["\s]+', " ", pick).replace(" or ", "|").strip().split("|") + ["two_calls", "fused_sgd"]
    tests = re.findall(r"^def (test_\w+)\(", open(os.path.join(root, "tests", "test_gpu_parity.py")).read(), re.M)
    left = {t for t in tests if not any(w.strip() in t for w in words)}
    assert {t for t in left if not re.search(r"full_size|full_batch|whole_array|reduced_batch|cfg5|cfg2|errors|refuse|validate|empty|share_one_array|"
                                             r"bf16|huge_ids|max_array|many_tables_and_large", t)} == set()
