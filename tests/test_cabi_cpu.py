"""Host-side checks of the C-ABI library that need no GPU."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2605_03110_b200 import build as ada_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    return ctypes.CDLL(ada_build.build())


def declared_functions():
    src = open(os.path.join(ROOT, "include", "ada.h")).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(ada_[a-z_0-9]+)\s*\(", src)))


def test_every_declared_symbol_is_exported(lib):
    names = declared_functions()
    assert {"ada_create", "ada_normalize", "ada_select_full", "ada_cascade_step",
            "ada_gram_op_count", "ada_device_status"} <= set(names)
    for n in names:
        assert hasattr(lib, n), n


def test_binding_lists_the_same_symbols():
    from paper_2605_03110_b200 import binding
    assert sorted(binding.SYMBOLS) == declared_functions()


def test_op_count_on_host(lib, golden):
    f = lib.ada_gram_op_count
    f.argtypes = [ctypes.c_int, ctypes.c_int64, ctypes.c_int64, ctypes.c_int64]
    f.restype = ctypes.c_uint64
    assert f(0, 512, 4096, 0) == 512 * 512 * 4096
    assert f(1, 512, 4096, 240) == 512 * 240 * 4096
    assert f(1, 8192, 4096, 8192) == f(0, 8192, 4096, 0)       # r = T costs the full Gram
    assert f(1, 16, 8, 17) == 0 and f(0, -1, 8, 0) == 0
    assert f(0, 16384, 4096, 0) == 16384 ** 2 * 4096           # no 32-bit overflow
    for kind, *row in golden("table7_and_cost_model.txt"):     # Table 7: L * T^2 with d = 1
        if kind == "indep":
            _, L, T, printed = row
            assert abs(int(L) * f(0, int(T), 1, 0) / 1e6 - float(printed)) < 0.006


def test_status_strings(lib):
    f = lib.ada_status_string
    f.restype = ctypes.c_char_p
    f.argtypes = [ctypes.c_int]
    assert f(0) == b"ADA_OK" and f(7) == b"ADA_ERR_TIMEOUT" and f(8) == b"ADA_ERR_BAD_TAU"
    assert len({f(i) for i in range(8)}) == 8


def test_create_rejects_bad_arguments_before_touching_a_device(lib):
    h = ctypes.c_void_p()
    f = lib.ada_create
    f.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_int] + [ctypes.c_int64] * 3 + [ctypes.c_int]
    assert f(ctypes.byref(h), 0, 0, 128, 64, 0) == 1            # ADA_ERR_INVALID_ARG
    assert f(ctypes.byref(h), 0, 1, 128, 64, 5) == 1
    assert f(None, 0, 1, 128, 64, 0) == 1
    # the per-sequence list counts live in 21-bit fields: longer sequences are refused
    assert f(ctypes.byref(h), 0, 1, (1 << 21), 64, 1) == 1
    assert f(ctypes.byref(h), 0, 1 << 12, 1 << 20, 64, 1) == 1   # maxB * maxT above 2^30
    assert h.value is None


def _calls():
    """Every native call with CPU tensors and no context: argument lists by name, with the places of
    required and of optional tensors."""
    import torch
    t = torch.zeros(64)
    lists = [t] * 8 + [None] * 2
    return {
        "select_full": ([None, t, 1, 8, 8, 8, 0, 0.3, t, t, None, 0], (1, 8, 9), (10,)),
        "select_full_heads": ([None, t, 8, 1, 8, 8, 0, 0.3, t, t, None, 0], (1, 8, 9), (10,)),
        "cascade_step": ([None, t, 1, 8, 8, 8, 0, 0.3] + lists + [0, 0], (1,) + tuple(range(8, 16)), (16, 17)),
        "cascade_step_heads": ([None, t, 8, 1, 8, 8, 0, 0.3] + lists + [0, 0], (1,) + tuple(range(8, 16)), (16, 17)),
        "cascade_step_adaptive": ([None, t, 1, 8, 8, 8, 0, t, None] + lists + [None, 0, 0],
                                  (1, 7) + tuple(range(9, 17)), (17, 18, 19)),
        "nearest_rep": ([None, t, 1, 8, 8, 8, 0, t, t, t, None, 0], (1, 7, 8, 9), (10,)),
        "attention_reps": ([None, t, t, t, 8, 1, 16, 16, 1, t, t, None, t, 16, 0, 0], (1, 2, 3, 9, 10, 12), (11,)),
    }


@pytest.mark.parametrize("name", sorted(_calls()))
def test_native_calls_take_tensors_where_tensors_belong(name):
    """A number or None in the place of a tensor raises instead of becoming a device address."""
    from paper_2605_03110_b200 import binding
    binding.lib()
    call = getattr(binding._fast, name)
    args, required, optional = _calls()[name]
    assert call(*args) == 1                                     # ADA_ERR_INVALID_ARG: no context
    for i in required + optional:
        for wrong in (4096, 1.5, "x") + ((None,) if i in required else ()):
            with pytest.raises(AttributeError):
                call(*args[:i], wrong, *args[i + 1:])
        assert call(*args[:i], args[1], *args[i + 1:]) == 1
    with pytest.raises(TypeError):
        call(*args[:-1])
    if name in ("select_full", "cascade_step"):
        assert call(*args[:7], "0.3", *args[8:]) == 1           # what float() takes
        for wrong, error in ((None, TypeError), ("x", ValueError)):
            with pytest.raises(error):
                call(*args[:7], wrong, *args[8:])


def test_policy_has_to_be_a_policy():
    from types import SimpleNamespace

    import torch

    from paper_2605_03110_b200 import binding
    binding.lib()
    state = SimpleNamespace(dtype=torch.float64, is_cuda=True, numel=lambda: 1, data_ptr=lambda: 0)
    X, i = torch.zeros(8, 8), torch.zeros(8, dtype=torch.int32)
    args = (SimpleNamespace(addr=None), X, state)
    stream = SimpleNamespace(cuda_stream=0)
    with pytest.raises(ctypes.ArgumentError):
        binding.ada_cascade_step_adaptive(*args, ctypes.c_double(0.1), i, i, stream=stream)
    for policy in (None, binding.TauPolicy(0.2, 0.1, 0.25, 0.35)):
        with pytest.raises(binding.AdaError):
            binding.ada_cascade_step_adaptive(*args, policy, i, i, stream=stream)


def test_native_module_carries_the_interpreter_abi(monkeypatch):
    """Another interpreter neither loads this one's module nor takes the build for complete; a module that
    is not there is explained."""
    import importlib.machinery
    import sys

    from paper_2605_03110_b200 import binding
    ada_build.build()
    assert os.path.basename(ada_build.PYCALL) == "_pycall" + importlib.machinery.EXTENSION_SUFFIXES[0]
    assert not ada_build.is_stale()
    monkeypatch.setattr(ada_build, "PYCALL", ada_build.PYCALL.replace("_pycall.", "_pycall.other-"))
    assert ada_build.is_stale()
    import paper_2605_03110_b200
    monkeypatch.delattr(paper_2605_03110_b200, "_pycall", raising=False)
    monkeypatch.setitem(sys.modules, "paper_2605_03110_b200._pycall", None)
    monkeypatch.setattr(binding, "_lib", None)
    with pytest.raises(RuntimeError, match="paper_2605_03110_b200.build"):
        binding.lib()


def _run_host_code(tmp_path, body):
    """Compiles `body` as main() beside the library's host-side launch rules and runs it."""
    src = tmp_path / "rules.cc"
    src.write_text('#include "launch_policy.h"\n#undef NDEBUG\n#include <assert.h>\nint main() {' + body + "return 0; }")
    exe = str(tmp_path / "rules")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", ada_build.CSRC, "-o", exe, str(src)], check=True)
    subprocess.run([exe], check=True)


def test_one_stream_launches_without_the_attribute(tmp_path):
    _run_host_code(tmp_path, """
        ada::SoleStream w;
        assert(!w.holds(7));
        assert(w.begin(7)); w.end();                  // the first stream takes the place ...
        assert(w.holds(7) && !w.holds(8));
        assert(!w.begin(8));                          // ... and every other one is refused
        assert(w.begin(7)); w.end();
        const unsigned long long seen = w.mark();
        w.idle(false, 8, seen);                       // another stream idle: nothing is known about 7
        assert(w.holds(7) && !w.begin(8));
        assert(w.begin(7)); w.end();                  // a launch after the mark
        w.idle(false, 7, seen);
        assert(w.holds(7) && !w.begin(8));
        w.idle(false, 7, w.mark());                   // its own stream idle, nothing launched since
        assert(!w.holds(7) && w.begin(8)); w.end();
        assert(!w.begin(7));
        w.idle(true, 0, w.mark());                    // the whole device idle
        assert(w.begin(7));                           // not handed to the driver yet:
        const unsigned long long pending = w.mark();
        w.end();
        w.idle(true, 0, pending);                     // the synchronisation did not wait for it
        assert(w.holds(7) && !w.begin(8));
        w.idle(true, 0, w.mark());
        assert(!w.holds(7));
    """)


def test_limit_of_the_waits_inside_a_launch(tmp_path):
    """Two seconds, but for the launch that may be placed piece by piece beside other streams' kernels."""
    _run_host_code(tmp_path, """
        auto seconds = [](bool alone) { return ada::wait_limit_units(alone) * 1048576e-9; };
        assert(seconds(false) > 1.99 && seconds(false) < 2.01);
        assert(seconds(true) > 19.9 && seconds(true) < 20.1);
    """)


@pytest.mark.parametrize("unit,ask", [("short_step.cu", "ada::step_short_ctas(&ctx, 32, 2048, 128)"),
                                      ("gram_tc2.cu", "ada::gram_tc2_hb_rows(&ctx, 1, 4096)")])
def test_a_kernel_that_cannot_be_configured_leaves_no_error_behind(tmp_path, unit, ask):
    """Where the runtime refuses a kernel's shared memory, these two report it by their result; the launchers
    that ask for the last error afterwards must not find this one.  (The refusal is played by a stand-in.)"""
    src = tmp_path / "unit.cu"
    src.write_text(f"""
        #include <cuda_runtime.h>
        #include <stdio.h>
        static cudaError_t pending = cudaSuccess;
        template <class F> static cudaError_t refuse(F, cudaFuncAttribute, int) {{ return pending = cudaErrorInvalidValue; }}
        static cudaError_t take_last() {{ const cudaError_t e = pending; pending = cudaSuccess; return e; }}
        #define cudaFuncSetAttribute refuse
        #define cudaGetLastError take_last
        #include "{unit}"
        namespace ada {{
        void prof_begin(ada_ctx*, int, cudaStream_t) {{}}
        void prof_end(ada_ctx*, cudaStream_t) {{}}
        bool coop_begin(ada_ctx*, cudaStream_t) {{ return false; }}
        void coop_end(ada_ctx*, bool) {{}}
        }}
        static ada_ctx ctx;
        int main() {{
            ctx.sm_count = 148;
            if ({ask} != 0) return puts("configured"), 1;
            if (pending != cudaSuccess) return puts("an error is left behind"), 2;
            return 0;
        }}""")
    exe = str(tmp_path / "unit")
    if not os.path.exists(ada_build.NVCC):
        pytest.skip("needs nvcc")
    subprocess.run([ada_build.NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", ada_build.CSRC, "-o", exe, str(src)],
                   check=True, capture_output=True)
    assert subprocess.run([exe], capture_output=True, text=True).stdout == ""
