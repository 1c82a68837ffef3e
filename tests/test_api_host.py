"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, and rejects bad arguments before touching the device."""
import ctypes as C
import os
import re

import numpy as np
import pytest

import paper_2108_02191_b200 as robe
from oracle import robe_oracle as orc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "robe.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(robe_[a-z_0-9]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    names = declared_functions()
    assert len(names) >= 11
    lib = C.CDLL(robe.LIB_PATH)
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(robe.EXPORTS) == names
    for n in names:
        assert callable(getattr(robe, n)), f"binding lacks {n}"


def test_binding_has_no_fallback_import():
    src = open(os.path.join(ROOT, "paper_2108_02191_b200", "binding.py")).read()
    assert "oracle" not in src
    for f in os.listdir(os.path.join(ROOT, "paper_2108_02191_b200", "csrc")):
        assert "oracle" not in open(os.path.join(ROOT, "paper_2108_02191_b200", "csrc", f)).read()


@pytest.mark.parametrize("args", [
    (0, 1, 1, 1), (10, 0, 4, 1), (10, 4, 0, 1), (10, 4, 4, 0), (10, 6, 4, 1), (10, 12, 4, 1), (3, 2, 4, 1),
    (2**32, 4, 16, 1), (2**32 - 15, 4, 16, 1), (10**6, 4, 40000, 1),
])
def test_create_rejects_bad_shapes(args):
    with pytest.raises(robe.RobeError) as ei:
        robe.robe_create(*args, 1)
    assert ei.value.status == robe.ROBE_ERR_INVALID_ARG


def test_create_accepts_limits_and_constants_match_oracle():
    for M, Z, d, T in [(1, 1, 1, 1), (2**32 - 16, 4, 16, 26), (4096, 4, 16, 4), (100, 100, 100, 3)]:
        for seed in (0, 0x0B0F, 2**64 - 1):
            h = robe.robe_create(M, Z, d, T, seed)
            k = robe.robe_get_hash_constants(h)
            assert k == [int(v) for v in orc.hash_constants(seed)]
            robe.robe_destroy(h)


def test_options_and_errors_without_device():
    h = robe.robe_create(4096, 4, 16, 4, 7)
    for key, val in [(robe.ROBE_OPT_SIGN, 2), (robe.ROBE_OPT_BWD_MODE, 5), (99, 0),
                     (robe.ROBE_OPT_VALIDATE, -1), (robe.ROBE_OPT_FWD_KERNEL, 5), (robe.ROBE_OPT_BWD_KERNEL, 7),
                     (robe.ROBE_OPT_INDEX_TYPE, 2), (robe.ROBE_OPT_BAG_LAYOUT, 2)]:
        with pytest.raises(robe.RobeError):
            robe.robe_set_option(h, key, val)
    robe.robe_set_option(h, robe.ROBE_OPT_SIGN, 1)
    robe.robe_set_option(h, robe.ROBE_OPT_SIGN, 0)
    robe.robe_set_option(h, robe.ROBE_OPT_INDEX_TYPE, robe.ROBE_I32)
    robe.robe_set_option(h, robe.ROBE_OPT_INDEX_TYPE, robe.ROBE_I64)
    robe.robe_set_option(h, robe.ROBE_OPT_BAG_LAYOUT, robe.ROBE_BAGS_TABLE_MAJOR)
    robe.robe_set_option(h, robe.ROBE_OPT_BAG_LAYOUT, robe.ROBE_BAGS_SAMPLE_MAJOR)
    lib = robe.binding.raw()
    # forward before attach: no array (dummy non-null pointers are never dereferenced)
    dummy = C.c_void_p(0x1000)
    assert lib.robe_forward(h, dummy, None, 2, 8, dummy, None) == robe.ROBE_ERR_NO_ARRAY
    # null pointers and inconsistent sizes
    assert lib.robe_forward(h, None, None, 2, 8, dummy, None) == robe.ROBE_ERR_INVALID_ARG
    assert lib.robe_forward(h, dummy, None, 2, 7, dummy, None) == robe.ROBE_ERR_INVALID_ARG
    assert lib.robe_forward(h, dummy, None, -1, 8, dummy, None) == robe.ROBE_ERR_INVALID_ARG
    assert lib.robe_forward(None, dummy, None, 2, 8, dummy, None) == robe.ROBE_ERR_INVALID_ARG
    assert lib.robe_backward(h, None, dummy, None, 2, 8, dummy, 0.0, None, 0, None) == robe.ROBE_ERR_INVALID_ARG
    # fused SGD needs the array
    assert lib.robe_backward(h, dummy, dummy, None, 2, 8, None, 0.1, None, 0, None) == robe.ROBE_ERR_NO_ARRAY
    # misaligned array pointer
    assert lib.robe_attach_array(h, C.c_void_p(0x1004), robe.ROBE_F32) == robe.ROBE_ERR_INVALID_ARG
    assert lib.robe_attach_array(h, dummy, 7) == robe.ROBE_ERR_INVALID_ARG
    # deterministic mode: workspace is required and sized by the library
    robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, robe.ROBE_BWD_DETERMINISTIC)
    need = robe.robe_backward_workspace_bytes(h, 2, 8)
    assert need >= 4 * 4 * 8 * 4 and need % 256 == 0
    assert lib.robe_backward(h, dummy, dummy, None, 2, 8, dummy, 0.0, None, 0, None) == robe.ROBE_ERR_WORKSPACE
    assert lib.robe_backward(h, dummy, dummy, None, 2, 8, dummy, 0.0, dummy, need // 2, None) == robe.ROBE_ERR_WORKSPACE
    robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, robe.ROBE_BWD_ATOMIC)
    assert robe.robe_backward_workspace_bytes(h, 2, 8) == 0
    assert robe.robe_status_string(robe.ROBE_ERR_WORKSPACE).startswith("workspace")
    assert robe.robe_status_string(0) == "ok"
    robe.robe_destroy(h)


def test_workspace_grows_with_blocks():
    h = robe.robe_create(25_000_000, 1, 128, 26, 1)
    robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, robe.ROBE_BWD_DETERMINISTIC)
    a = robe.robe_backward_workspace_bytes(h, 1024, 1024 * 26)
    b = robe.robe_backward_workspace_bytes(h, 2048, 2048 * 26)
    assert b > a >= 16 * 1024 * 26 * 128
    robe.robe_destroy(h)


def test_workspace_asks_for_no_more_than_it_used_to():
    # callers hold workspaces of a size, and the static call has a limit: blocks (four words each), ids (one
    # word), hand-over records and the counters; bounds of strips may not come on top of that
    up = lambda v: -(-v // 256) * 256
    asked = {}
    for M, d, Z in [(300_000_000, 128, 128), (250_000_000, 64, 16), (2_400_000, 32, 32), (2_600_000, 128, 127),
                    (540_000, 16, 8), (1_200_000, 128, 128), (4096, 16, 4), (129, 128, 128), (25_000_000, 100, 100),
                    (5_400_000, 128, 128), (5_800_000, 128, 128)]:
        h = robe.robe_create(M, Z, d, 1, 1)
        robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, robe.ROBE_BWD_DETERMINISTIC)
        for nnz in [1, 100, 9375, M // (2 * d) + 1, M // (2 * d) + 500, M // d, 1_300_000]:
            nb = nnz * -(-d // Z)
            was = (4 * up(4 * nb) + up(4 * nnz) + 4 * 256 * 592 + 4 * 256 + 256
                   + up(400 * min(max(nb // 128, 64), 1 << 20)))
            asked[M, nnz] = robe.robe_backward_workspace_bytes(h, nnz, nnz)
            assert asked[M, nnz] <= was, (M, d, Z, nnz)
        # and a workspace sized for the largest call is enough for every smaller one
        sizes = [robe.robe_backward_workspace_bytes(h, n, n) for n in range(1, 60_000, 7)]
        assert all(a <= b for a, b in zip(sizes, sizes[1:])), (M, d, Z)
        robe.robe_destroy(h)
    # 1.3 M rows of one block that touch 300 M slots densely: within the static call's limit
    assert asked[300_000_000, 1_300_000] <= robe.ROBE_STATIC_SCRATCH_BYTES


def test_workspace_holds_the_strips_bounds_and_nothing_more():
    # the bounds of strips go by the array's length alone, whatever the number of blocks; a longer array's go to
    # buffers that are there anyway
    for M, strips in [(540_000, 8438), (1_200_000, 18_750), (5_400_000, 21_094), (5_800_000, 0), (25_000_000, 0)]:
        room = 256 + 2 * -(-4 * (strips + 1) // 256) * 256 if strips else 0
        for nnz in [M // 32 + 1, M // 4, 2 * M]:  # touched densely: blocks of 16 on half of the slots or more
            figures = []
            for m in (M, 1 << 31):
                h = robe.robe_create(m, 16, 16, 1, 1)
                robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, robe.ROBE_BWD_DETERMINISTIC)
                figures.append(robe.robe_backward_workspace_bytes(h, nnz, nnz))
                robe.robe_destroy(h)
            assert figures[0] - figures[1] == room, (M, nnz, figures)


def test_sort_based_variants_refuse_sizes_beyond_their_32_bit_numbering():
    # block numbers, bag numbers and gradient positions are 32-bit in the binned / deterministic /
    # Adam paths: larger calls are refused before anything is launched (dummy pointers are never read)
    lib = robe.binding.raw()
    dummy = C.c_void_p(0x1000)
    h = robe.robe_create(1 << 20, 4, 16, 1, 3)        # C = 4 blocks per id
    assert lib.robe_attach_array(h, dummy, robe.ROBE_F32) == robe.ROBE_OK
    big = 1 << 30                                     # 2^30 ids -> 2^32 blocks
    for mode in (robe.ROBE_BWD_DETERMINISTIC, robe.ROBE_BWD_BINNED):
        robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, mode)
        assert lib.robe_backward(h, dummy, dummy, None, big, big, dummy, 0.0, dummy, 1 << 40, None) \
            == robe.ROBE_ERR_UNSUPPORTED
    assert lib.robe_backward_adam(h, dummy, dummy, None, big, big, dummy, dummy, 0.1, 0.9, 0.999, 1e-8, 1,
                                  dummy, 1 << 40, None) == robe.ROBE_ERR_UNSUPPORTED
    assert lib.robe_backward_deterministic_static(h, dummy, dummy, None, big, big, dummy, 0.0, None) \
        == robe.ROBE_ERR_UNSUPPORTED
    # atomic mode has no such limit on the host side, but still wants consistent sizes
    robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, robe.ROBE_BWD_ATOMIC)
    assert lib.robe_backward(h, dummy, dummy, None, big, big - 1, dummy, 0.0, None, 0, None) \
        == robe.ROBE_ERR_INVALID_ARG
    robe.robe_destroy(h)


def test_header_is_plain_c_and_cpp(tmp_path):
    # the boundary is a C ABI: the header must compile as C11 and as C++ with nothing but itself
    import subprocess
    inc = os.path.join(ROOT, "include")
    for comp, std, ext in (("gcc", "-std=c11", "c"), ("g++", "-std=c++11", "cpp")):
        src = tmp_path / f"use_robe.{ext}"
        src.write_text('#include "robe.h"\nint main(void) { robe_handle_t h = 0; return robe_destroy(h) == ROBE_OK; }\n')
        r = subprocess.run([comp, std, "-Wall", "-Wextra", "-Werror", "-pedantic", "-fsyntax-only", "-I", inc, str(src)],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr


C_PROGRAM = r"""
#include <stdio.h>
#include <string.h>
#include "robe.h"
int main(void) {
    robe_handle_t h = 0;
    uint64_t k[9];
    if (robe_create(&h, 4096, 4, 16, 4, 7) != ROBE_OK) return 1;
    if (robe_get_hash_constants(h, k) != ROBE_OK || k[0] != ((1ull << 61) - 1)) return 2;
    if (robe_set_option(h, ROBE_OPT_SIGN, 1) != ROBE_OK) return 3;
    if (robe_forward(h, (const void*)0x1000, 0, 2, 8, (float*)0x1000, 0) != ROBE_ERR_NO_ARRAY) return 4;
    if (robe_create(&h, 10, 12, 4, 1, 7) != ROBE_ERR_INVALID_ARG) return 5;  /* Z > d, not a multiple */
    if (strcmp(robe_status_string(ROBE_ERR_WORKSPACE), "workspace missing, misaligned or too small") != 0) return 6;
    printf("%llu\n", (unsigned long long)k[1]);
    return 0;
}
"""


def test_c_program_links_and_calls_the_library(tmp_path):
    # a C caller, not ctypes: compile against include/robe.h, link librobe.so, run the host-only calls
    import subprocess
    src = tmp_path / "caller.c"
    src.write_text(C_PROGRAM)
    exe = tmp_path / "caller"
    lib_dir = os.path.dirname(robe.LIB_PATH)
    r = subprocess.run(["gcc", "-std=c11", "-Wall", "-Werror", "-I", os.path.join(ROOT, "include"), str(src), "-o",
                        str(exe), "-L", lib_dir, "-l:" + os.path.basename(robe.LIB_PATH), "-Wl,-rpath," + lib_dir],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr)
    assert int(r.stdout.strip()) == int(orc.hash_constants(7)[1])  # A_h as the oracle draws it


FAKE_TENSORS = r"""
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
import paper_2108_02191_b200 as robe
h = robe.robe_create(4096, 4, 16, 4, 7)
with FakeTensorMode():  # CUDA tensors without memory, as tracing and shape propagation hand them over
    ids = torch.empty(8, dtype=torch.int64, device="cuda")
    out = torch.empty(2, 4, 16, device="cuda")
for call in (lambda: robe.robe_forward(h, ids, None, 2, out),
             lambda: robe.robe_backward(h, out, ids, None, 2, out),
             lambda: robe.robe_apply_sgd(h, out, 0.1)):
    try:
        call()
    except Exception as e:
        print("raised", type(e).__name__)
"""


def test_tensors_without_memory_raise_and_do_not_end_the_process():
    import subprocess
    import sys
    r = subprocess.run([sys.executable, "-c", FAKE_TENSORS], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
    assert r.stdout.count("raised") == 3, r.stdout + r.stderr[-2000:]


def test_only_a_handle_is_taken_for_one():
    # eight bytes of anything else (an array that holds the address, a plain integer of that size) are refused
    from types import SimpleNamespace
    h = robe.robe_create(4096, 4, 16, 4, 7)
    stream = SimpleNamespace(cuda_stream=0)
    with pytest.raises(robe.RobeError) as ei:  # the handle itself: the library says what is missing
        robe.robe_apply_sgd(h, None, 0.1, True, stream)
    assert ei.value.status == robe.ROBE_ERR_INVALID_ARG
    for other in (np.array([h.value], dtype=np.uint64), C.c_uint64(h.value), bytearray(C.string_at(C.addressof(h), 8))):
        with pytest.raises(C.ArgumentError):
            robe.robe_apply_sgd(other, None, 0.1, True, stream)
    robe.robe_destroy(h)
