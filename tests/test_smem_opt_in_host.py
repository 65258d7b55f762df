"""The shared-memory opt-in against a fake runtime with two devices, whose limits
are kept per function and device (no GPU needed): it reaches every device, not
only the first one of the process, never lowers a limit, and reports what it
cannot give."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1710_09421_gb300", "csrc")

FAKE = """
#pragma once
#include <stddef.h>
#include <map>
#include <utility>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
enum cudaDeviceAttr { cudaDevAttrMaxSharedMemoryPerBlockOptin = 97 };
struct cudaFuncAttributes { size_t sharedSizeBytes; int maxDynamicSharedSizeBytes; };
constexpr int OPTIN = 227 * 1024, STATIC = 640, DEFAULT = 48 * 1024 - STATIC;
inline int g_dev = 0;
inline std::map<std::pair<int, const void *>, int> g_limit;
inline int limit(const void *f) { auto i = g_limit.find({g_dev, f}); return i == g_limit.end() ? DEFAULT : i->second; }
inline cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
inline cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = OPTIN; return cudaSuccess; }
inline cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *f)
{ a->sharedSizeBytes = STATIC; a->maxDynamicSharedSizeBytes = limit(f); return cudaSuccess; }
inline cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v)
{ if (v < 0 || v + STATIC > OPTIN) return cudaErrorInvalidValue; g_limit[{g_dev, f}] = v; return cudaSuccess; }
"""

WRAP = """
#include "ekl_smem.h"
extern "C" {
void set_device(int d) { g_dev = d; }
int opt_in(long f, long bytes) { return (int)ekl::smem_opt_in((const void *)f, (size_t)bytes); }
int allowed(long f) { return limit((const void *)f); }
int most() { return OPTIN - STATIC; }
}
"""


@pytest.fixture(scope="module")
def rt(tmp_path_factory):
    d = tmp_path_factory.mktemp("smem")
    (d / "cuda_runtime.h").write_text(FAKE)
    (d / "wrap.cpp").write_text(WRAP)
    so = d / "libsmem.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", CSRC, str(d / "wrap.cpp"), "-o",
                    str(so)], check=True)
    return ctypes.CDLL(str(so))


def test_every_device_gets_it_and_no_call_lowers_it(rt):
    big, small = 200 * 1024, 57 * 1024
    for dev in (0, 1):
        rt.set_device(dev)
        assert rt.opt_in(16, big) == 0 and rt.allowed(16) >= big
    for dev in (0, 1, 0):
        rt.set_device(dev)
        assert rt.opt_in(16, small) == 0 and rt.allowed(16) >= big
    assert rt.opt_in(32, small) == 0 and rt.allowed(32) >= small  # another function has its own limit


def test_edges(rt):
    rt.set_device(0)
    assert rt.opt_in(48, 1024) == 0  # below the default: nothing to do
    assert rt.opt_in(56, 48 * 1024) == 0 and rt.allowed(56) >= 48 * 1024  # above it with the static part
    assert rt.opt_in(64, rt.most()) == 0 and rt.allowed(64) >= rt.most()
    assert rt.opt_in(80, rt.most() + 1) != 0
