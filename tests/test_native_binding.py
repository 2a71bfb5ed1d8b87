"""The native side of the binding (csrc/py_call.cpp) against a stand-in for the library, on the CPU: what a call does to
the interpreter around it.  The stand-in's entry points have the library's names and return what the test asks for."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STUB = """
#include <chrono>
#include <thread>
extern "C" {
volatile int gdn_stub_go = 0;
// 0 as soon as another thread has set the flag, 4 if none has within two seconds
static int wait_for_flag() {
    for (int i = 0; i < 2000 && !gdn_stub_go; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    return gdn_stub_go ? 0 : 4;
}
#define ENTRY(name) int name(...) { return wait_for_flag(); }
ENTRY(gdn_chunk_prefill) ENTRY(gdn_chunk_prefill_f32) ENTRY(gdn_chunk_prefill_bf16_simt) ENTRY(gdn_chunk_prefill_noalloc)
ENTRY(gdn_chunk_prefill_raw) ENTRY(gdn_chunk_prefill_gated) ENTRY(gdn_decode_step) ENTRY(gdn_attn_causal_prefill)
}
"""

# CUDA tensors without memory: they pass the checks, and the stand-in reads none of their (null) pointers.
PRELUDE = """
import ctypes, importlib.machinery, importlib.util, sys, threading, time
import torch
spec = importlib.util.spec_from_file_location("_call", sys.argv[1] + "/_call.so",
                                              loader=importlib.machinery.ExtensionFileLoader("_call", sys.argv[1] + "/_call.so"))
native = importlib.util.module_from_spec(spec)
spec.loader.exec_module(native)
stub = ctypes.CDLL(sys.argv[1] + "/libgdn.so")
go = ctypes.c_int.in_dll(stub, "gdn_stub_go")

class Cuda(torch.Tensor):
    @staticmethod
    def __new__(cls, *shape, dtype=torch.bfloat16):
        return torch.Tensor._make_wrapper_subclass(cls, shape, dtype=dtype, device="cuda")
    @classmethod
    def __torch_dispatch__(cls, func, types, args=(), kwargs=None):
        raise RuntimeError("no memory behind this tensor")

def f32(*shape):
    return Cuda(*shape, dtype=torch.float32)

B, T, H, D = 2, 70, 3, 128
def prefill_args(io=torch.bfloat16):
    x = lambda: Cuda(B, T, H, D, dtype=io)
    return [x(), x(), x(), f32(B, T, H), f32(B, T, H), f32(B, H, D, D), x(), f32(B, H, D, D), None, 64, 0]
def calls():
    p = prefill_args()
    for name in ("gdn_chunk_prefill", "gdn_chunk_prefill_bf16_simt", "gdn_chunk_prefill_noalloc"):
        yield name, p
    yield "gdn_chunk_prefill_f32", prefill_args(torch.float32)
    yield "gdn_chunk_prefill_raw", p[:5] + [0.05, 1e-6] + p[5:]
    yield "gdn_chunk_prefill_gated", p[:6] + [Cuda(B, T, H, D), f32(D), 1e-6] + p[6:]
    row = lambda: Cuda(B, H, D)
    yield "gdn_decode_step", [row(), row(), row(), f32(B, H), f32(B, H), f32(B, H, D, D), row(), 0]
    yield "gdn_attn_causal_prefill", [Cuda(B, T, H, D), Cuda(B, T, 1, D), Cuda(B, T, 1, D), Cuda(B, T, H, D), None, 0.1, 0]
"""


@pytest.fixture(scope="module")
def stand_in(tmp_path_factory):
    """A folder with the built extension module and the stand-in it finds next to itself."""
    from paper_2607_14568_b200 import build
    build.build()
    where = tmp_path_factory.mktemp("native")
    shutil.copy(build.CALL, where / "_call.so")
    (where / "stub.cpp").write_text(STUB)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-pthread", str(where / "stub.cpp"), "-o", str(where / "libgdn.so")],
                   check=True)
    return str(where)


def _run(stand_in, body):
    res = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(body), stand_in], cwd=ROOT, capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0, f"exit {res.returncode}\n{res.stdout}\n{res.stderr[-3000:]}"


def test_other_threads_run_during_a_call(stand_in):
    """A call may block (a full launch queue, or a queue behind a host callback written in Python): the interpreter lock is
    released meanwhile, so that another Python thread can go on and do what the call waits for."""
    _run(stand_in, """
        for name, args in calls():
            go.value = 0
            def later():
                time.sleep(0.02)
                go.value = 1
            t = threading.Thread(target=later)
            t.start()
            rc = getattr(native, name)(*args)
            t.join()
            assert rc == 0, f"{name}: no other thread ran while the entry point was waiting (status {rc})"
    """)


def test_a_tensor_that_cannot_give_its_address_raises(stand_in):
    """Inside a vmap a tensor has no address of its own and torch throws a C++ exception when it is asked for one: that has to
    come out as a Python exception (it ended the process when it left the C function)."""
    _run(stand_in, """
        go.value = 1
        for name, args in calls():
            def mapped(x):
                return getattr(native, name)(x, *args[1:])
            batch = Cuda(5, *args[0].shape, dtype=args[0].dtype)
            try:
                torch.func.vmap(mapped)(batch)
            except RuntimeError as e:
                assert "data pointer" in str(e), f"{name}: {e}"
            else:
                raise AssertionError(f"{name}: no exception")
    """)
