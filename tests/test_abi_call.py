"""The struct forms of the entry points (ism_call_*): the packed structs match
the header's layout, every form reaches the entry point it names (seen by that
entry point's own refusals), and the sizes are those of the direct queries.
Host checks only: nothing is launched."""
import ctypes as C
import os
import re
import subprocess
import sysconfig

import numpy as np
import pytest
import torch

from paper_2408_00539_gb300 import ism

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    return ism.load(build_if_missing=True)


def _segs():
    return ism.Segments.from_numpy([0, 300, 430], [0, 2, 3], [100, 300, 130], [0, 1, 0], device="cpu")


def _head(form=0, hq=4, hkv=2, d=128, dtype=0, scale=0.1, descales=(1.0, 1.0, 1.0)):
    return (*_segs().fields(), hq, hkv, d, dtype, form, scale, *descales)


def test_struct_sizes(tmp_path, lib):
    src = tmp_path / "s.c"
    src.write_text('#include "ism.h"\n#include <stdio.h>\nint main(void) { printf("%zu %zu", sizeof(ism_pass_call_t), '
                   'sizeof(ism_append_call_t)); return 0; }\n')
    exe = str(tmp_path / "s")
    cc = (sysconfig.get_config_var("CC") or "gcc").split()[0]
    try:
        subprocess.run([cc, "-I" + os.path.join(ROOT, "include"), str(src), "-o", exe], check=True)
    except FileNotFoundError:
        pytest.skip("no C compiler")
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert [int(x) for x in re.findall(r"\d+", out)] == [ism._PASS.size, ism._APPEND.size]


@pytest.mark.parametrize("hq,hkv,d,dtype", [(4, 2, 128, 0), (3, 1, 64, 0), (2, 2, 64, 1), (4, 4, 128, 2)])
def test_sizes(lib, hq, hkv, d, dtype):
    segs = _segs()
    s, sh = segs.struct(), ism._Shape(hq, hkv, d, dtype, 0.1)
    head = (*segs.fields(), hq, hkv, d, dtype, 0, 0.1, 0.0, 0.0, 0.0)
    n = C.c_size_t()
    assert lib.ism_attn_fwd_workspace_size(C.byref(s), C.byref(sh), C.byref(n)) == 0
    assert ism._pass_sizes(head, False) == n.value
    if dtype == 2:
        with pytest.raises(ism.IsmError):
            ism._pass_sizes(head, True)
        return
    want = []
    for f in (lib.ism_attn_bwd_workspace_size, lib.ism_attn_bwd_workspace_size_min):
        assert f(C.byref(s), C.byref(sh), C.byref(n)) == 0
        want.append(n.value)
    assert ism._pass_sizes(head, True) == tuple(want)


@pytest.mark.skipif(torch.cuda.is_available(), reason="made-up addresses: only where no GPU is visible")
def test_forms_reach_their_entry_points(lib):
    def fwd(rope=(0, 0, 0), plan=(0, 0, 0), **head):
        code = lib.ism_call_fwd(ism._PASS.pack(*_head(**head), *rope, *plan, *(0,) * 14))
        return code, lib.ism_last_error().decode()

    assert fwd(dtype=2) == (2, "e4m3 inputs only in ism_attn_fwd_e4m3")
    assert fwd(form=1)[0] == 1 and "needs shape->dtype ISM_E4M3" in fwd(form=1)[1]
    assert "descales" in fwd(form=1, dtype=2, descales=(0.0, 1.0, 1.0))[1]
    assert "rope tables" in fwd(form=2)[1]
    assert "256-byte aligned" in fwd(plan=(8, 0, 0))[1]
    assert "softmax_scale" in fwd(scale=1e-60)[1]  # zero as a float
    assert "must be non-NULL" in fwd()[1]
    assert lib.ism_call_bwd(ism._PASS.pack(*_head(), 0, 0, 0, 0, 0, 0, *(0,) * 14)) == 1
    assert lib.ism_call_fwd(None) == 1 and lib.ism_call_bwd(None) == 1 and lib.ism_call_append(None) == 1

    def append(form, dtype=0, page=0, scale=0.1):
        call = ism._APPEND.pack(4, 2, 128, dtype, form, scale, 1.0, 1.0, 1.0, 0, 0, 0, 2, 8, 1, 4, page, 1, 0, 0, 0, 0,
                                0, 0, 0, 64, 0, 0, 0, 0, 0, 0, 0, 0, 0)
        return lib.ism_call_append(call), lib.ism_last_error().decode()

    assert append(0)[0] == 1 and "caches" in append(0)[1]
    assert append(0, dtype=2)[0] == 2
    assert "needs ISM_E4M3" in append(1)[1]
    assert "page_size 100" in append(4, page=100)[1]
    assert "prefill_append_rope needs ISM_BF16" in append(2, dtype=1)[1]
    assert "paged_rope needs ISM_BF16" in append(6, dtype=1)[1]


@pytest.mark.parametrize("x", [[3, 5], (3, 5), np.array([3, 5], np.int64), [3.0, 5.0], [np.int32(3), 5]])
def test_host_array(x):
    addr, n, owner = ism._host_array(x, np.int32, "i")
    assert n == 2 and list((C.c_int32 * 2).from_address(addr)) == [3, 5]
