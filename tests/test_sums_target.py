"""Where lbpc_sums_async lets its reduction write the caller's memory: the rule by itself, on what the runtime says of
an address (a host program built from csrc/lbpc_sums_target.h)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <stdio.h>
#include "lbpc_sums_target.h"
using namespace lbpc;
static char* const A = (char*)0x7f0000001000;  // an address; nothing reads it
static AddressInfo at(cudaMemoryType type, int device, long long off, unsigned long long access = 3, long long shift = 0) {
  AddressInfo a{};
  a.at.type = type;
  a.at.device = device;
  a.at.devicePointer = type == cudaMemoryTypeUnregistered ? nullptr : A + off + shift;
  a.access = access;
  return a;
}
static void say(const char* name, bool on_device, AddressInfo f, AddressInfo l, long long off = 0) {
  double* p = sums_target((double*)(A + off), on_device, 0, f, l);
  printf("%s %lld\n", name, p ? (long long)((char*)p - A) : -1);
}
int main() {
  const auto D = cudaMemoryTypeDevice, H = cudaMemoryTypeHost, M = cudaMemoryTypeManaged, U = cudaMemoryTypeUnregistered;
  say("device_1", true, at(D, 0, 0), at(D, 0, 15));
  say("device_0", false, at(D, 0, 0), at(D, 0, 15));
  say("pinned_0", false, at(H, 0, 0), at(H, 0, 15));
  say("pinned_0_mapped_elsewhere", false, at(H, 0, 0, 3, 4096), at(H, 0, 15, 3, 4096));
  say("pinned_1", true, at(H, 0, 0), at(H, 0, 15));
  say("other_device_1", true, at(D, 1, 0), at(D, 1, 15));
  say("managed_1", true, at(M, 0, 0), at(M, 0, 15));
  say("managed_0", false, at(M, 0, 0), at(M, 0, 15));
  say("pageable_0", false, at(U, 0, 0, 0), at(U, 0, 15, 0));
  say("pinned_ends_within", false, at(H, 0, 0), at(U, 0, 15, 0));
  say("pinned_mapped_apart", false, at(H, 0, 0), at(H, 0, 15, 3, 64));
  say("read_only_1", true, at(D, 0, 0, 1), at(D, 0, 15, 1));
  say("read_only_tail_0", false, at(H, 0, 0), at(H, 0, 15, 1));
  say("misaligned", true, at(D, 0, 4), at(D, 0, 19), 4);
  return 0;
}
"""
DIRECT = {"device_1": 0, "pinned_0": 0, "pinned_0_mapped_elsewhere": 4096}


def test_only_agreeing_writable_memory_is_written_directly(tmp_path):
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not gxx or not os.path.exists(nvcc):
        pytest.skip("needs g++ and the CUDA headers")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1709_04400_gb300", "csrc"), "-I", cuda, "-o", str(exe),
                    str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    got = dict(line.split() for line in out.splitlines())
    assert len(got) == 14
    for name, value in got.items():
        assert int(value) == DIRECT.get(name, -1), name
