"""The C-ABI library loads and exports every symbol include/tpq.h declares; the
context-free entry points agree with the oracle's closed forms.  No GPU needed."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2411_07942_b200 import build, binding

    build.build()
    return binding.lib()


def _declared():
    text = open(os.path.join(ROOT, "include", "tpq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(tpq_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported_and_bound(lib):
    from paper_2411_07942_b200 import binding

    names = _declared()
    assert len(names) >= 20
    for n in names:
        assert hasattr(lib, n), f"{n} is declared in tpq.h but not exported"
        assert n in binding.SIGNATURES, f"{n} has no ctypes signature"
    assert sorted(binding.SIGNATURES) == names


def test_status_strings_and_version(lib):
    assert lib.tpq_status_string(0) == b"ok"
    seen = {lib.tpq_status_string(i) for i in range(8)}
    assert len(seen) == 8
    assert b"sm_100a" in lib.tpq_version()


@pytest.mark.parametrize("T,E,k", [(1, 8, 0), (3, 65, 1), (16, 256, 4), (2048, 5120, 80), (64, 4608, 72),
                                   (8192, 8192, 128), (7, 253, 9), (5, 33, 33)])
def test_payload_bytes_closed_form(lib, corc, T, E, k):
    assert lib.tpq_payload_bytes_for(T, E, k) == corc.payload_bytes(T, E, k)


def test_payload_bytes_degenerate(lib):
    assert lib.tpq_payload_bytes_for(0, 8, 0) == 0
    assert lib.tpq_payload_bytes_for(4, 8, 9) == 0
    assert lib.tpq_payload_bytes(None, 16) == 0


def test_null_context_is_rejected_not_crashed(lib):
    assert lib.tpq_destroy(None) == 0
    assert lib.tpq_quantize_pack(None, 0, None, 1, 8, None, 0, None) == 1
    assert lib.tpq_dequant_reduce(None, None, 0, 1, None, 0, 8, None) == 1
    assert lib.tpq_calibrate_ranges(None, 0, None, 1, 1, 8, None) == 1
    assert lib.tpq_select_features(None, -1, None, None) == 1
    assert lib.tpq_last_error(None) == b""
    assert lib.tpq_num_selected(None) == -1


def test_create_validates_before_touching_cuda(lib):
    import ctypes

    h = ctypes.c_void_p()
    for args in [(0, 8, 4, 0.01), (2, 0, 4, 0.01), (2, 8, 9, 0.01), (2, 8, 1, 0.01), (2, 8, 4, -0.5), (2, 8, 4, 1.5), (65, 8, 4, 0.01)]:
        assert lib.tpq_create(ctypes.byref(h), *args) == 1
        assert not h.value
    assert lib.tpq_create(None, 2, 8, 4, 0.01) == 1


def test_product_never_imports_the_oracle():
    """The product path shares nothing with the oracle: no file of the package names it."""
    pkg = os.path.join(ROOT, "paper_2411_07942_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".h", ".cuh")):
                src = open(os.path.join(dirpath, f)).read()
                assert "import oracle" not in src and "from oracle" not in src and "tpqo_" not in src, f


def test_pointer_arrays_are_checked_like_the_c_signature(lib):
    """What stands for a host array of addresses: sequences of addresses, None or c_void_p, and arrays of c_void_p.  Arrays
    of other elements (a 32-bit one is half as long as the library reads), numbers that are no plain integers (a
    one-element tensor has an __index__) and single addresses are refused."""
    import ctypes

    import numpy as np
    import torch

    from paper_2411_07942_b200 import binding

    def read(obj, n):
        return list((ctypes.c_uint64 * n).from_buffer_copy(bytes(obj)))

    assert read(binding._ptrs([4096, 2 ** 47]), 2) == [4096, 2 ** 47]
    assert read(binding._ptrs((1, None, ctypes.c_void_p(7))), 3) == [1, 0, 7]
    assert read(binding._ptrs((ctypes.c_void_p * 2)(5, 6)), 2) == [5, 6]
    assert read(binding._ptrs([-1]), 1) == [2 ** 64 - 1]
    for bad in ((ctypes.c_uint32 * 2)(1, 2), (ctypes.c_uint64 * 2)(1, 2), (ctypes.c_float * 2)()):
        with pytest.raises(ctypes.ArgumentError):
            binding._ptrs(bad)
    for bad in ([torch.tensor(4096)], [np.int64(4096)], [4096.0], ["x"]):
        with pytest.raises(TypeError):
            binding._ptrs(bad)
    ok = (ctypes.c_void_p * 2)()
    for name, args in (("tpq_quantize_pack_batch", (0, 2, None, 1, 8, None, 0, None)), ("tpq_dequant_reduce", (None, 2, 1, None, 0, 8, None)),
                       ("tpq_quantize_pack_push", (0, None, 1, 8, None, None, 2, 0, 1, None))):
        fn, types = getattr(lib, name), binding.SIGNATURES[name][1]
        for j, kind in enumerate(types):
            if kind is not ctypes.POINTER(ctypes.c_void_p):
                continue
            with_ok = [None, *args]
            with_ok[j] = ok
            assert fn(*with_ok) == binding.TPQ_ERR_INVALID_ARG          # (no context)
            for bad in (4096, b"12345678", (ctypes.c_uint32 * 2)()):
                wrong = [None, *args]
                wrong[j] = bad
                with pytest.raises(ctypes.ArgumentError):
                    fn(*wrong)


def test_extension_calls_pass_on_what_ctypes_would(lib):
    """Every call of the extension module, bound to recorders: plain arguments arrive as the C signature types them (64-bit
    addresses, 32-bit tags, sizes, None for an optional pointer); any other form is left to ctypes without a call."""
    import ctypes

    from paper_2411_07942_b200 import binding

    seen, keep, addresses = [], [], []
    for name in binding._CALLS:
        res, types = binding.SIGNATURES[name]
        plain = [ctypes.c_void_p if isinstance(a, type) and issubclass(a, ctypes._Pointer) else a for a in types]

        def record(*args, _name=name):
            lists = {i: n for i, a in enumerate(binding.SIGNATURES[_name][1]) if a is ctypes.POINTER(ctypes.c_void_p) for n in [2]}
            seen.append((_name, [[(ctypes.c_uint64 * n).from_address(x)[j] for j in range(n)] if (n := lists.get(i)) else x
                                 for i, x in enumerate(args)]))
            return 7

        fn = ctypes.CFUNCTYPE(res, *plain)(record)
        keep.append(fn)
        addresses.append(ctypes.cast(fn, ctypes.c_void_p).value)
    c, ctx, big, st = binding._calls, 2 ** 47 + 8, 2 ** 64 - 16, 2 ** 63 + 64
    calls = [  # function, arguments, what the library's entry point receives
        (c.calibrate_ranges, (ctx, 1, big, 3, 4, 8, st), "tpq_calibrate_ranges", [ctx, 1, big, 3, 4, 8, st]),
        (c.quantize_pack, (ctx, -1, big, 2 ** 40, 8, 32, 2 ** 63, 0), "tpq_quantize_pack", [ctx, -1, big, 2 ** 40, 8, 32, 2 ** 63, None]),
        (c.quantize_pack_batch, (ctx, 5, [16, big], -3, 8, (48, 64), 9, st), "tpq_quantize_pack_batch", [ctx, 5, 2, [16, big], -3, 8, [48, 64], 9, st]),
        (c.dequant_reduce, (ctx, [16, big], 4, 48, 1, 8, None, st), "tpq_dequant_reduce", [ctx, [16, big], 2, 4, 48, 1, 8, st]),
        (c.dequant_reduce, (ctx, (16, big), 4, 48, 0, 8, 80, st), "tpq_dequant_reduce_bias", [ctx, [16, big], 2, 4, 48, 0, 8, 80, st]),
        (c.dequant_reduce_arrivals, (ctx, [16, big], 4, 48, 1, 8, None, 96, 2 ** 32 - 1, 2 ** 64 - 1, st), "tpq_dequant_reduce_arrivals",
         [ctx, [16, big], 2, 4, 48, 1, 8, None, 96, 2 ** 32 - 1, 2 ** 64 - 1, st]),
        (c.quantize_pack_push, (ctx, 0, 32, 4, 8, [16, big], [20, 24], 2 ** 63, 2 ** 32 - 1, st), "tpq_quantize_pack_push",
         [ctx, 0, 32, 4, 8, [16, big], [20, 24], 2, 2 ** 63, 2 ** 32 - 1, st]),
        (c.linear_quantize_pack, (ctx, 2, 32, 48, 4, 8, 64, 9, None, st), "tpq_linear_quantize_pack", [ctx, 2, 32, 48, 4, 8, 64, 9, None, st]),
        (c.linear_quantize_pack, (ctx, 2, 32, 48, 4, 8, 64, 9, 80, st), "tpq_linear_quantize_pack", [ctx, 2, 32, 48, 4, 8, 64, 9, 80, st]),
    ]
    try:
        c.bind(addresses)
        for fn, args, name, want in calls:
            assert fn(*args) == 7
            assert seen.pop() == (name, want)
            for i, a in enumerate(args):
                if isinstance(a, (list, tuple)):
                    others = [list(a[:1]) + [None], [1.0, 2], [True, 2], [-1, 2], [2 ** 64, 2], (ctypes.c_void_p * 2)(1, 2), 4096, [1] * 65, "12"]
                    if fn in (c.quantize_pack_batch, c.quantize_pack_push):
                        others.append(list(a) + [1])   # (not as long as the other list)
                else:
                    others = [True, 1.0, "1", ctypes.c_void_p(1), 2 ** 64, [1]] + ([] if i in (6, 8) else [None])
                for other in others:
                    assert fn(*args[:i], other, *args[i + 1:]) is None, (name, i, other)
            assert fn(*args[:-1]) is None and fn(*args, 0) is None
        assert not seen
        t = binding.Tpq.__new__(binding.Tpq)   # a closed context: refused by the library, as through ctypes
        t._h, t._p, t.N, t.E = ctypes.c_void_p(), None, 2, 8
    finally:
        c.bind([ctypes.cast(getattr(lib, n), ctypes.c_void_p).value for n in binding._CALLS])
    for call in (lambda: t.quantize_pack_batch(0, [16, 16], 1, [16, 16], 9), lambda: t.dequant_reduce([16, 16], 1, 16), lambda: t.quantize_pack(0, 16, 1, 16, 9)):
        with pytest.raises(binding.TpqError) as e:
            call()
        assert e.value.status == binding.TPQ_ERR_INVALID_ARG
    with pytest.raises(AssertionError):
        t.quantize_pack_batch(0, [16, 16], 1, [16], 9)


@pytest.mark.parametrize("cc", ["no-such-compiler", "false", "sh -c 'exit 1'"])
def test_library_is_built_without_a_compiler_for_the_extension(lib, monkeypatch, tmp_path, cc):
    """The C library needs neither a C compiler nor the Python headers: build() brings it about and warns; an extension module
    that is out of date does not stay behind."""
    from paper_2411_07942_b200 import build

    order = []
    monkeypatch.setattr(build, "build_lib", lambda force=False, verbose=False: order.append("lib"), raising=False)
    compile_calls = build.build_calls
    monkeypatch.setattr(build, "build_calls", lambda force=False: (order.append("calls"), compile_calls(force)))
    monkeypatch.setenv("CC", cc)
    monkeypatch.setattr(build, "CALLS", tmp_path / build.CALLS.name)
    build.CALLS.write_bytes(b"built from another source")
    os.utime(build.CALLS, (0, 0))
    with pytest.warns(RuntimeWarning, match="calls.c"):
        assert build.build() == build.LIB
    assert order == ["lib", "calls"] and not build.CALLS.exists()


def test_library_loads_without_the_extension_module(lib):
    """Where the extension module is not there, a warning says so and every call goes through ctypes."""
    import subprocess
    import sys

    code = """
import sys, warnings
sys.modules["paper_2411_07942_b200._calls"] = None   # (an import of it fails)
from paper_2411_07942_b200 import binding
with warnings.catch_warnings(record=True) as w:
    warnings.simplefilter("always")
    binding.lib()
assert [x.category for x in w] == [RuntimeWarning] and "_calls" in str(w[0].message)
import ctypes
t = binding.Tpq.__new__(binding.Tpq)   # a closed context: what the library itself answers
t._h, t._p, t.N, t.E = ctypes.c_void_p(), None, 2, 8
calls = [lambda: t.calibrate_ranges(0, 16, 1, 1), lambda: t.quantize_pack(0, 16, 1, 16, 9),
         lambda: t.quantize_pack_batch(0, [16, 16], 1, [16, 16], 9), lambda: t.dequant_reduce([16, 16], 1, 16),
         lambda: t.dequant_reduce([16, 16], 1, 16, bias_ptr=16), lambda: t.dequant_reduce([16, 16], 1, 16, arrived_ptr=16, epoch=1),
         lambda: t.quantize_pack_push(0, 16, 1, [16], [16], 9, 1), lambda: t.linear_quantize_pack(0, 16, 16, 1, 8, 16, 9)]
for call in calls:
    try:
        call()
    except binding.TpqError as e:
        assert e.status == binding.TPQ_ERR_INVALID_ARG
    else:
        raise AssertionError("no error")
"""
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr


def test_extension_module_is_of_this_interpreter(lib, monkeypatch, tmp_path):
    """Its file name carries the interpreter's tag, that file is the one loaded, and one without a tag does not stay."""
    import sysconfig

    from paper_2411_07942_b200 import binding, build

    assert build.CALLS.name == "_calls" + sysconfig.get_config_var("EXT_SUFFIX") != "_calls.so"
    assert os.path.samefile(binding._calls.__file__, build.CALLS)
    monkeypatch.setattr(build, "CALLS", tmp_path / build.CALLS.name)
    (tmp_path / "_calls.so").write_bytes(b"built for another interpreter")
    build.build_calls()
    assert sorted(os.listdir(tmp_path)) == [build.CALLS.name]
