"""The host's record of what stands in front of a call in its stream (csrc/call_order.h), compiled and driven on the CPU: a
commit may read its inputs early only behind a verify of its own context on its own stream, with nobody's call in between."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NONE, VERIFY, COMMIT, COMMIT_VERIFY, OTHER = range(5)
SHIM = """
#include "call_order.h"
using lumo::CallOrder;
extern "C" {
void* make() { return new CallOrder(); }
int begin(void* c, int dev, const void* st) { return static_cast<CallOrder*>(c)->begin(dev, st); }
void done(void* c, int kind) { static_cast<CallOrder*>(c)->done(static_cast<CallOrder::Kind>(kind)); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2609_23900_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    so = ctypes.CDLL(str(d / "shim.so"))
    so.make.restype = ctypes.c_void_p
    so.begin.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    so.done.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return so


def call(lib, ctx, kind, stream=1, dev=0, ok=True):
    before = lib.begin(ctx, dev, stream)
    if ok:
        lib.done(ctx, kind)
    return before


def test_a_contexts_own_calls_on_one_stream_are_known(lib):
    a = lib.make()
    assert call(lib, a, VERIFY) == NONE
    assert call(lib, a, COMMIT) == VERIFY
    assert call(lib, a, COMMIT_VERIFY) == COMMIT
    assert call(lib, a, OTHER) == COMMIT_VERIFY
    assert call(lib, a, VERIFY) == OTHER


@pytest.mark.parametrize("kind", [VERIFY, COMMIT, COMMIT_VERIFY, OTHER])
def test_a_call_of_another_context_in_between_is_not(lib, kind):
    a, b = lib.make(), lib.make()
    call(lib, a, VERIFY)
    call(lib, b, kind)                        # accept, path_from_node, commit of another context ...
    assert call(lib, a, COMMIT) == NONE
    call(lib, a, VERIFY)
    call(lib, b, kind, ok=False)              # ... even one that failed half way
    assert call(lib, a, COMMIT) == NONE
    call(lib, a, VERIFY)
    assert call(lib, a, COMMIT) == VERIFY


def test_another_stream_a_failed_call_and_another_device(lib):
    a, b = lib.make(), lib.make()
    call(lib, a, VERIFY, stream=1)
    assert call(lib, a, COMMIT, stream=2) == NONE
    call(lib, a, VERIFY, ok=False)
    assert call(lib, a, COMMIT) == NONE
    call(lib, a, VERIFY, dev=0)
    call(lib, b, OTHER, dev=1)
    assert call(lib, a, COMMIT, dev=0) == VERIFY
