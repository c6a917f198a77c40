"""Which kernel the library's host code launches, and how, seen through a CUDA runtime that runs
nothing (fake_cudart.c, linked with the library's own objects): no GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

from tests.conftest import ROOT

import paper_2605_08755_gb300 as laq
from paper_2605_08755_gb300 import _lib, build

FAKE = ctypes.c_void_p(0x10000)   # never dereferenced
SMS = 152


def cuda_include():
    nvcc = os.path.realpath(build._nvcc())
    return os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")


@pytest.fixture(scope="module")
def F(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp("fake")
    objs = [os.path.join(build.BUILD_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    obj, so = str(d / "fake.o"), str(d / "liblaq_fake.so")
    subprocess.run([shutil.which("gcc"), "-O1", "-fPIC", "-I", cuda_include(), "-c",
                    os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", obj], check=True)
    subprocess.run([shutil.which("g++"), "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so, obj]
                   + objs, check=True)
    L = ctypes.CDLL(so)
    real = _lib.lib()
    for name in ("laq_gemm_wxg128", "laq_gemm_wxg128_config", "laq_gemm_wxg128_prologue",
                 "laq_gemm_chain", "laq_pass_run"):
        getattr(L, name).argtypes = getattr(real, name).argtypes
    L.fake_last_kernel.restype = ctypes.c_char_p
    return L


def launched(F):
    """(kernel, grid x, grid y, warps, cluster, dynamic shared memory) of the last launch."""
    out = (ctypes.c_longlong * 6)()
    F.fake_last_shape(out)
    name = F.fake_last_kernel().decode()
    kind = "batch" if "gemm_batch_kernel" in name else "general" if "gemm_kernel" in name else name
    return kind, out[0], out[1], out[3] // 32, out[4], out[5]


def gemm(F, cfg, M, K, N, bits):
    assert F.laq_gemm_wxg128_config(FAKE, M, K, N, FAKE, FAKE, FAKE, bits, FAKE, ctypes.byref(cfg),
                                    None) == 0
    return launched(F)


@pytest.mark.parametrize("M,K,N,bits", [(16, 4096, 24576, 3), (8, 2560, 6144, 4), (5, 512, 48, 3),
                                        (1, 2560, 151936, 3)])
def test_an_edited_plan_is_what_runs(F, M, K, N, bits):
    plan = lambda: laq.laq_gemm_plan(M, K, N, bits, SMS)
    c = plan()
    _, slots, cluster = c.batch
    assert gemm(F, c, M, K, N, bits)[:3] == ("batch", -(-(N // 16) // (c.batch[0] * slots)), cluster)
    c.pdl = 1   # not part of the shape
    assert gemm(F, c, M, K, N, bits)[0] == "batch"
    for edit in (dict(tiles_per_cta=3 - min(c.tiles_per_cta, 2), warps=c.warps * 2 % 16 or 8),
                 dict(tiles_per_cta=1, warps=5), dict(cluster=c.cluster % 8 * 2 or 1),
                 dict(stages=c.stages + 1 if c.stages < 4 else 3)):
        c = plan()
        for field, value in edit.items():
            setattr(c, field, value)
        kind, gx, gy, warps, _, _ = gemm(F, c, M, K, N, bits)
        assert (kind, gx, gy, warps) == ("general", -(-(N // 16) // c.tiles_per_cta), c.cluster,
                                         c.warps), edit


@pytest.mark.parametrize("M", [1, 4, 8, 16])
def test_a_plan_survives_its_dictionary(F, M):
    for K, N in ((2560, 6144), (4096, 24576), (2560, 151936)):
        c = laq.laq_gemm_plan(M, K, N, 3, SMS)
        again = laq.GemmConfig.make(**c.as_dict())
        assert bytes(again) == bytes(c)
        assert gemm(F, again, M, K, N, 3) == gemm(F, c, M, K, N, 3)


def entries(M, dims):
    arr = (_lib.Gemv * len(dims))()
    for i, (K, N) in enumerate(dims):
        arr[i] = _lib.Gemv(FAKE, FAKE, FAKE, FAKE, FAKE, M, K, N, 3, 1)
    return arr


@pytest.mark.parametrize("what", ["general", "batch", "norm", "chain", "pass"])
def test_every_device_is_granted_shared_memory(F, what):
    """Function attributes hold for one device: the second GPU of a process asks for its own."""
    ws = ctypes.c_void_p(0x200000)
    dims = [(4096, 4096), (4096, 2560)]

    def run():
        if what == "chain":
            return F.laq_gemm_chain(entries(1, dims), 2, ws, 1 << 20, None)
        if what == "pass":
            plan, _ = _lib.pass_plan(entries(1, dims), 2, SMS)
            return F.laq_pass_run(plan, ctypes.c_void_p(0x100000), ws, 1 << 20, None)
        M = 1 if what == "general" else 16
        cfg = laq.laq_gemm_plan(M, 4096, 24576, 3, SMS)
        assert (cfg.batch is None) == (what == "general")
        if what == "norm":
            pro = _lib.GemmPrologue(_lib.PROLOGUE_RMSNORM, 1e-6, None, None, FAKE)
            return F.laq_gemm_wxg128_prologue(FAKE, M, 4096, 24576, FAKE, FAKE, FAKE, 3, FAKE,
                                              ctypes.byref(pro), ctypes.byref(cfg), None)
        return F.laq_gemm_wxg128_config(FAKE, M, 4096, 24576, FAKE, FAKE, FAKE, 3, FAKE,
                                        ctypes.byref(cfg), None)
    try:
        for device in (0, 1, 0):
            F.fake_set_device(device)
            n = F.fake_launches()
            assert (run(), F.fake_launches() - n) == (0, 1), device
            assert launched(F)[5] > 48 * 1024
    finally:
        F.fake_set_device(0)


def test_attention_copies_stay_inside_the_step(tmp_path):
    """Every address a copy of a step is given, also one of no bytes past the row's last token, lies
    in rows that exist: in a cache filled to its last row the next one is past the allocation."""
    src = tmp_path / "offsets.cpp"
    src.write_text("""
#include <cuda_runtime.h>
#include <stdint.h>
#include <cstdio>
#include "laq_internal.cuh"
int main() {
    for (int left = 1; left <= 16; ++left) {
        bool seen[16 * 16] = {};
        for (int lane = 0; lane < 32; ++lane)
            for (int u = 0; u < 8; ++u) {
                const int o = laq::attn_copy_offset(lane, u, left);
                if (o < 0 || o % 8 || o + 8 > left * 128) return 1;
                if (2 * u + lane / 16 < left) seen[o / 8] = true;
            }
        for (int j = 0; j < left * 16; ++j)
            if (!seen[j]) return 2;
    }
    return 0;
}
""")
    exe = str(tmp_path / "offsets")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-I", cuda_include(), "-I", build.CSRC, "-o",
                    exe, str(src)], check=True)
    assert subprocess.run([exe]).returncode == 0
