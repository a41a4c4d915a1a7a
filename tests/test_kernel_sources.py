"""Rules of the kernels launched as programmatic dependents that no run can be
trusted to show (a breach would hang now and then, or read stale memory), held
to the sources themselves."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_00539_gb300", "csrc")


def _body(text, at):
    """The block that opens at or after `at`."""
    start = text.index("{", at)
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i]
    raise ValueError("unbalanced braces")


def _kernels():
    """(name, parameters, body) of every kernel, comments taken out."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(\w+)\s*\(", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[end], 0)
                end += 1
            out.append((m.group(1), text[m.end():end], _body(text, end)))
    return out


KERNELS = _kernels()
TRIGGER = re.compile(r"pdl_wait\(\)|pdl_trigger\(\)|griddepcontrol\.launch_dependents")


def test_kernels_found():
    names = {n for n, _, _ in KERNELS}
    assert {"fwd_pair_kernel", "fwd_kernel", "dq_kernel", "dkdv_kernel", "dq_gemm_kernel", "decode_tc_kernel"} <= names


@pytest.mark.parametrize("name", [n for n, _, b in KERNELS if "tmem_alloc" in b])
def test_trigger_follows_the_allocation(name):
    """A kernel that holds tensor memory lets its successor start only after
    the block-wide barrier behind its own allocation: the successor may allocate
    before it waits, and each would wait for the other."""
    body = next(b for n, _, b in KERNELS if n == name)
    allocated = body.index("__syncthreads()", body.index("tmem_alloc"))
    for m in TRIGGER.finditer(body):
        # a block that leaves before the allocation needs none
        leaves = re.match(r"[^{}]*\breturn;", body[m.end():])
        assert m.start() > allocated or leaves, name


@pytest.mark.parametrize("name", [n for n, _, b in KERNELS if "pdl_" in b])
def test_nothing_counts_as_constant(name):
    """Loads of a dependent kernel that the compiler may take for constant may
    be moved before its wait: no __restrict__ parameters, no __ldg."""
    params, body = next((p, b) for n, p, b in KERNELS if n == name)
    assert "__restrict__" not in params and "__ldg" not in body


def test_page_table_and_offsets_are_plain_loads():
    for name, function in (("ism_internal.cuh", "paged_row"), ("ism_rope.cu", "seq_of")):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        at = text.index(function + "(")
        assert "__restrict__" not in text[at:text.index(")", at)] and "__ldg" not in _body(text, at)


def test_early_reads_go_to_l2():
    """What is read before the kernel's own wait comes from L2: the lengths and
    the page table of the decode, O and dO of the dependent Delta."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "ism_decode_tc.cu")).read())
    assert re.findall(r"[^\n]*\bcache_len\b[^\n]*", text) == [
        "__device__ __forceinline__ int32_t cached(const DecodeArgs& a, int b) { return ld_gpu(a.cache_len + b); }"]
    assert "ld_gpu(page_entry(" in text and "paged_row(" not in text
    body = next(b for n, _, b in KERNELS if n == "delta_kernel")
    loads = re.findall(r"=([^;]*(?:\bO\b|\bdO\b)[^;]*);", body)
    assert len(loads) == 2 and all("__ldcg" in x for x in loads)


def test_split_forward_triggers_behind_its_last_barrier():
    """The merge behind a split forward starts when every warp is done: the
    first thread of a block to trigger does so for the block."""
    body = next(b for n, _, b in KERNELS if n == "fwd_pair_kernel")
    assert body.rindex("pdl_trigger()") > body.rindex("__syncthreads()")


def test_metadata_is_read_as_it_was_written():
    """The metadata kernels read tiles and bounds that they wrote themselves:
    nothing of theirs counts as constant."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "ism_meta.cu")).read())
    assert "__restrict__" not in text and "__ldg" not in text
