"""The C-ABI library loads without a GPU and exports every symbol include/avsg.h declares."""
import ctypes
import os
import re

import paper_2609_37538_b200 as avsg

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "avsg.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(avsg_[a-z_]+)\s*\(", text)))


def test_header_and_binding_agree():
    assert _declared() == sorted(avsg.EXPORTS)


def test_library_exports_every_declared_symbol():
    lib = avsg.load_library()
    for name in _declared():
        assert hasattr(lib, name), name


def test_struct_layouts_match_the_header():
    assert ctypes.sizeof(avsg.AvsgConfig) == 56
    assert ctypes.sizeof(avsg.AvsgStepArgs) == 120
    assert ctypes.sizeof(avsg.AvsgStats) == 104
    assert ctypes.sizeof(avsg.AvsgNoAllocArgs) == 120


def test_error_strings_and_argument_errors_need_no_gpu():
    lib = avsg.load_library()
    for code in (0, -1, -2, -3, -4, -5, -6):
        assert lib.avsg_strerror(code)
    assert lib.avsg_strerror(-99) == b"unknown error"
    h = ctypes.c_void_p()
    assert lib.avsg_create(None, ctypes.byref(h)) == avsg.EINVAL
    bad = avsg.AvsgConfig(1, 1000, 656, 16, 1, 16, 0, 0)            # slots not a power of two
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EINVAL
    bad = avsg.AvsgConfig(1, 1024, 650, 16, 1, 16, 0, 0)            # row bytes not a multiple of 16
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EINVAL
    bad = avsg.AvsgConfig(1, 1024, 656, 600, 2, 16, 0, 0)           # Eq. 7: 2 * 600 > 1024
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.ECAPACITY
    bad = avsg.AvsgConfig(1, 65536, 656, 2048, 2, 16, 0, 0)         # more slots than a cluster holds
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EUNSUPPORTED
    bad = avsg.AvsgConfig(1, 1024, 656, 16, 1, 16, 0, 0, 0, 0, 0, 0, 0, 3)       # cluster size not a power of two
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EINVAL
    bad = avsg.AvsgConfig(1, 1024, 656, 16, 1, 200, 0, 0)
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EINVAL
    assert lib.avsg_step(None, None, None) == avsg.EINVAL
    assert lib.avsg_destroy(None) == avsg.EINVAL
    bad = avsg.AvsgConfig(1, 1024, 656, 16, 1, 16, 6, 0)            # transfer mode beyond the last one
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EINVAL
    bad = avsg.AvsgConfig(1, 1024, 656, 16, 1, 16, 0, 0, avsg.INDEX_DIRECT, 0)   # direct index without max_context
    assert lib.avsg_create(ctypes.byref(bad), ctypes.byref(h)) == avsg.EINVAL
    st = avsg.AvsgStats()
    for call in (lambda: lib.avsg_stats(None, ctypes.byref(st)), lambda: lib.avsg_table_stats(None, 0, ctypes.byref(st)),
                 lambda: lib.avsg_sync_status(None, None), lambda: lib.avsg_clear_status(None),
                 lambda: lib.avsg_probe_wait_limit(None, None), lambda: lib.avsg_set_transfer_mode(None, 0),
                 lambda: lib.avsg_set_timing(None, 1), lambda: lib.avsg_set_transfer_geometry(None, 148, 256),
                 lambda: lib.avsg_save_state(None, None), lambda: lib.avsg_restore_state(None, None),
                 lambda: lib.avsg_reset(None, None, 0), lambda: lib.avsg_step_host(None, None, None)):
        assert call() == avsg.EINVAL
    p = ctypes.c_void_p()
    assert lib.avsg_host_kv_alloc(0, 0, ctypes.byref(p), None) == avsg.EINVAL          # no bytes
    assert lib.avsg_host_kv_alloc(4096, 2, ctypes.byref(p), None) == avsg.EINVAL       # unknown flag
    assert lib.avsg_host_kv_alloc(4096, 0, None, None) == avsg.EINVAL                  # nowhere to put the address
    assert lib.avsg_host_kv_alloc(1 << 60, 0, ctypes.byref(p), None) == avsg.EINVAL    # beyond any address space
    assert lib.avsg_host_kv_free(None) == avsg.EINVAL
    assert lib.avsg_host_kv_free(ctypes.c_void_p(4096)) == avsg.EINVAL                 # not from the allocator


def test_product_sources_do_not_touch_the_oracle():
    pkg = os.path.join(ROOT, "paper_2609_37538_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                text = open(os.path.join(dirpath, f)).read()
                assert "oracle" not in text.lower().replace("no cpu fallback", ""), f


def test_host_buffers_are_used_in_place_only_where_all_of_them_is_mapped(tmp_path):
    import subprocess
    from paper_2609_37538_b200 import build
    exe = str(tmp_path / "mapped_range")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Wextra", "-I", "/usr/local/cuda/include", "-I", build.CSRC, "-o", exe,
                           os.path.join(ROOT, "tests", "abi", "mapped_range.cpp")])
    run = subprocess.run([exe], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout


def test_lengths_are_taken_from_any_iterable():
    """Lists, arrays and one-shot iterators of integers, of other numbers and of values that wrap give the same lengths."""
    import types
    import numpy as np
    from paper_2609_37538_b200.binding import PreparedCall, _c_array
    got = []
    lib = types.SimpleNamespace(avsg_step=lambda h, ref, stream: got.append(list(call._vlen)) or 0)
    call = PreparedCall(types.SimpleNamespace(_lib=lib, _h=None), [0, 1, 2], [16, 16, 16], 1, 1)
    want = [5, -1, 7]
    kinds = [want, tuple(want), np.array(want), np.array(want, np.float64), [5.0, -1, 7.9], [5, 2**32 - 1, 7]]
    for values in kinds + [iter(k) for k in kinds] + [(v for v in k) for k in kinds]:
        call.run(16, values, 16, stream=0)
        assert got[-1] == want
    for values in kinds + [iter(k) for k in kinds]:
        owner, at = _c_array("i", values, 3)
        assert list((ctypes.c_int32 * 3).from_address(at)) == want
    assert _c_array("I", None, 3) == (None, None)


def test_native_calls_take_what_the_binding_takes():
    """The extension module fills the argument blocks as ctypes would, and hands the rest to the binding's conversions."""
    import types
    import numpy as np
    import pytest
    import torch
    from paper_2609_37538_b200 import binding as b
    seen = []

    def note(ctx, args, stream, which):
        a = b.AvsgStepArgs.from_address(args)
        seen.append((which, ctx, stream, {k: getattr(a, k) for k, _ in a._fields_}, list(call._vlen)))
        return 0 if a.slots != 99 else avsg.ECAPACITY
    fn = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    step, host = fn(lambda *a: note(*a, "step")), fn(lambda *a: note(*a, "host"))
    cell = ctypes.c_uint64(77)
    ctx = types.SimpleNamespace(_cell=cell, _lib=types.SimpleNamespace(avsg_step=step, avsg_step_host=host))
    call = b.PreparedCall(ctx, [0, 1, 2], [16, 32, 48], 2, 5, kv_rows=[7, 8, 9])
    t, n = torch.zeros(4, dtype=torch.int32), np.zeros(4, np.int32)
    call.run(t, [1, 2, -3], n, 2**64 + 5, None, 6)
    which, h, st, a, vlen = seen[-1]
    assert (which, h, st, vlen) == ("step", 77, 6, [1, 2, -3]) and (a["n"], a["n_tokens"], a["topk"]) == (3, 2, 5)
    assert (a["indices"], a["slots"], a["hit"], a["miss_count"]) == (t.data_ptr(), n.ctypes.data, 5, None)
    assert (a["stage_one_done"], a["stage_one_done_value"], a["arriving"], a["verified_len_dev"]) == (None, 0, None, None)
    call.run(8, t, 8, True, 0, types.SimpleNamespace(cuda_stream=11), True, (t, -1), n)
    which, h, st, a, vlen = seen[-1]
    assert (which, st, a["verified_len_dev"], a["hit"], a["miss_count"]) == ("host", 11, t.data_ptr(), 1, None)
    assert (a["stage_one_done"], a["stage_one_done_value"], a["arriving"]) == (t.data_ptr(), 2**64 - 1, n.ctypes.data)
    want = [5, -1, 7]
    kinds = [want, tuple(want), np.array(want), np.array(want, np.float64), [5.0, -1, 7.9], [5, 2**32 - 1, 7], [np.int32(5), -1, True + 6]]
    for values in kinds + [iter(k) for k in kinds]:
        call.run(16, values, 16, stream=0)
        assert seen[-1][4] == want and seen[-1][3]["verified_len_dev"] is None and seen[-1][2] is None
    for bad in (dict(indices="x"), dict(slots=1.5), dict(hit=[]), dict(verified_len=[1, "a", 2]), dict(verified_len=[1, 2]),
                dict(verified_len=3), dict(stage_one_done=(None, 1)), dict(stage_one_done=5)):
        with pytest.raises((TypeError, ValueError)):
            call.run(**{**dict(indices=8, verified_len=want, slots=8, stream=0), **bad})
    with pytest.raises(avsg.AvsgError) as e:
        call.run(8, want, 99, stream=0)
    assert e.value.code == avsg.ECAPACITY
    cell.value = 0                                       # a closed context
    call.run(8, want, 8, stream=0)
    assert seen[-1][1] is None

    got = []

    def take(args, stream):
        a = b.AvsgNoAllocArgs.from_address(args)
        arrays = [None if not at else list((k * a.n).from_address(at)) for at, k in ((a.kv_base, ctypes.c_uint64), (a.row_stride, ctypes.c_uint64),
                                                                                     (a.verified_len, ctypes.c_int32), (a.kv_rows, ctypes.c_uint32))]
        got.append(({k: getattr(a, k) for k, _ in a._fields_}, arrays, stream))
        return avsg.EINVAL if a.max_lifetime == 7 else 0
    keep = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p)(take)
    before, b._noalloc_fn = b._noalloc_fn, b._address_of(keep)
    try:
        for n_tab in (3, 40):                            # (40: more than one call may have)
            tok, life, rows = torch.zeros((n_tab, 64), dtype=torch.int32), torch.zeros((n_tab, 64), dtype=torch.int8), torch.zeros((n_tab, 64, 48), dtype=torch.uint8)
            ids = torch.zeros((n_tab, 2, 5), dtype=torch.int32)
            lens, kv = list(range(n_tab)), [16 * i for i in range(n_tab)]
            for kvs, ls, strides, rws in ((kv, lens, None, None), (tuple(kv), np.array(lens), [48] * n_tab, iter(lens)),
                                          (iter(kv), [float(v) for v in lens], tuple([2**64 + 48] * n_tab), [2**32 + v for v in lens])):
                avsg.step_noalloc(tok, life, rows, ids, kvs, ls, max_lifetime=4, slots=ids, stream=9, row_stride=strides, kv_rows=rws)
                a, arrays, st = got[-1]
                assert (a["n"], a["n_tokens"], a["topk"], a["buffer_slots"], a["row_bytes"], a["max_lifetime"], st) == (n_tab, 2, 5, 64, 48, 4, 9)
                assert (a["tok"], a["life"], a["buffer"], a["indices"], a["slots"]) == (tok.data_ptr(), life.data_ptr(), rows.data_ptr(), ids.data_ptr(), ids.data_ptr())
                assert a["hit"] is None and a["miss_count"] is None and a["status"] is None
                assert arrays == [kv, [48] * n_tab if strides else None, lens, lens if rws is not None else None]
        some = dict(max_lifetime=4, slots=ids, stream=0)
        avsg.step_noalloc(tok, life, rows, ids, [t] * n_tab, lens, hit=n, miss_count=5, status=t, **some)
        assert got[-1][1][0] == [t.data_ptr()] * n_tab and (got[-1][0]["hit"], got[-1][0]["miss_count"]) == (n.ctypes.data, 5)
        with pytest.raises(avsg.AvsgError):
            avsg.step_noalloc(tok, life, rows, ids, kv, lens, max_lifetime=7, slots=ids, stream=0)
        with pytest.raises(ValueError):
            avsg.step_noalloc(tok[0], life, rows, ids, kv, lens, **some)
        with pytest.raises(TypeError):
            avsg.step_noalloc(tok, life, rows, ids, ["a"] * n_tab, lens, **some)
        with pytest.raises(IndexError):
            avsg.step_noalloc(tok, life, rows, ids, kv + [0], lens, **some)
    finally:
        b._noalloc_fn = before


def test_calls_without_the_extension_module(monkeypatch):
    """Another Python than the module was built for: the same calls by ctypes, which take and refuse the same."""
    from paper_2609_37538_b200 import binding as b
    monkeypatch.setattr(b, "_calls", False)
    monkeypatch.setattr(b, "_current_stream_fn", None)
    test_native_calls_take_what_the_binding_takes()
    test_lengths_are_taken_from_any_iterable()


def test_the_library_builds_without_the_extension_module(monkeypatch, tmp_path):
    """No C++ compiler for the module, or no Python.h: the library is there all the same."""
    import pytest
    from paper_2609_37538_b200 import build
    monkeypatch.setattr(build, "CALLS", str(tmp_path / "_python_calls.so"))
    for compiler in ("/nonexistent/g++", "false"):
        monkeypatch.setenv("CXX", compiler)
        with pytest.warns(UserWarning, match="extension module"):
            assert build.build_library() == build.LIB and os.path.exists(build.LIB)
