"""The convolution's split of a sequence into CTAs and warps (csrc/conv_split.h), on the CPU: every entry and channel covered,
within the kernel's limits, and no warps for runs that do not exist where they would keep other CTAs waiting for a place."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = """
#include "conv_split.h"
extern "C" void split(int C, int Ns, int run, int seqs, int sms, int* out) {
  const lumo::ConvSplit s = lumo::conv_split(C, Ns, run, seqs, sms);
  out[0] = s.runs; out[1] = s.groups; out[2] = s.log_groups; out[3] = s.slabs; out[4] = lumo::kConvWarps; out[5] = lumo::kConvMaxEntries;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2609_23900_b200", "csrc"),
                           str(d / "shim.cpp"), "-o", str(d / "shim.so")])
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("seqs", [1, 9, 10, 64])
@pytest.mark.parametrize("run", [4, 8, 16])
def test_every_size(lib, run, seqs):
    out, sms = (ctypes.c_int * 6)(), 148
    for Ns in range(1, 1025):
        for C in (192, 1024, 4096, 8192):
            lib.split(C, Ns, run, seqs, sms, out)
            runs, groups, log_groups, slabs, warps, most = out
            need = -(-Ns // run)
            parts = -(-Ns // (runs * run))                 # CTAs along a sequence, as the launch counts them
            assert groups == 1 << log_groups and 1 <= runs * groups <= warps and runs * run <= most
            assert slabs * groups * 128 >= C > (slabs - 1) * groups * 128
            assert parts * runs >= need and parts == -(-need // warps)      # as few CTAs as hold the runs
            even = -(-need // parts)
            if parts > 1 and parts * slabs * seqs > 4 * sms and even <= 6:
                assert runs == even                        # several waves: no idle warps where five CTAs or more then fit an SM
            else:
                assert runs == min(need, warps)
