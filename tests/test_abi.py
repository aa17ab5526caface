"""Host-side checks that need no GPU: the library builds, loads and exports what the header declares."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2606_12243_b200 import build
    path = build.build()
    return ctypes.CDLL(path)


def _declared():
    text = open(os.path.join(ROOT, "include", "viasd.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(viasd_[a-z_0-9]+)\s*\(", text)))


def test_header_symbols_are_exported(lib):
    names = _declared()
    assert {"viasd_init_model", "viasd_verify_step", "viasd_slim_forward", "viasd_full_forward",
            "viasd_tier_accept", "viasd_kv_commit"} <= set(names)
    for n in names:
        assert hasattr(lib, n), n


def test_binding_lists_every_export():
    from paper_2606_12243_b200 import binding
    assert sorted(binding.EXPORTS) == _declared()


def test_host_only_calls(lib):
    from paper_2606_12243_b200 import binding as vb
    assert vb.lib().viasd_strerror(0) == b"ok"
    assert vb.lib().viasd_strerror(vb.VIASD_EINVAL) == b"invalid argument"
    cfg = vb.make_config(32, 4096, 32, 32, 128, 11008, 32000, "bf16", 1, 1033, 9)
    n = vb.workspace_bytes(cfg, 16)
    assert 1 << 20 < n < 1 << 30
    bad = vb.make_config(32, 4096, 32, 5, 128, 11008, 32000, "bf16", 1, 1033, 9)   # heads % kv_heads != 0
    assert vb.workspace_bytes(bad, 16) == 0
    assert vb.workspace_bytes(vb.make_config(32, 4096, 32, 32, 128, 11008, 32000, "bf16", 1, 1033, 65), 16) == 0


def test_struct_layouts_match_header():
    """Sizes the C compiler gives the public structs equal the ctypes mirrors."""
    import subprocess, tempfile, textwrap
    from paper_2606_12243_b200 import binding as vb
    src = textwrap.dedent('''
        #include <stdio.h>
        #include "viasd.h"
        int main(void) {
            printf("%zu %zu %zu %zu %zu %zu %zu\\n", sizeof(viasd_config), sizeof(viasd_weights), sizeof(viasd_cache),
                   sizeof(viasd_draft), sizeof(viasd_params), sizeof(viasd_result), sizeof(viasd_stats));
            return 0;
        }''')
    with tempfile.TemporaryDirectory() as d:
        c = os.path.join(d, "t.c")
        open(c, "w").write(src)
        exe = os.path.join(d, "t")
        subprocess.check_call(["gcc", "-I", os.path.join(ROOT, "include"), c, "-o", exe])
        sizes = [int(x) for x in subprocess.check_output([exe]).split()]
    mirrors = [vb.Config, vb.Weights, vb.Cache, vb.Draft, vb.Params, vb.Result, vb.Stats]
    assert sizes == [ctypes.sizeof(m) for m in mirrors]


def test_gemm_of_more_than_128_rows_takes_nothing_per_row(lib, tmp_path):
    """The one-CTA GEMM takes up to 256 rows of a plain product; what keeps something per row (norm factors, rotary positions), or
    a second plane, ends at 128 and is refused above (before anything of the launch is looked at)."""
    import subprocess
    src = tmp_path / "t.cpp"
    src.write_text("""
        #include <cuda_runtime.h>
        #include "gemm_tc.cuh"
        extern "C" int call(int (*f)(const TcLaunch &, cudaStream_t), int rows, int nt, int has_lo, int epi, int norm) {
            static float x[1];
            TcLaunch L;
            memset(&L, 0, sizeof(L));
            L.rows = rows; L.nt = nt; L.has_lo = has_lo; L.epi = epi; L.ssq_in = norm ? x : nullptr; L.n_seg = 1; L.sm_count = 148;
            return f(L, nullptr);                              // (no columns: a launch that is taken is empty)
        }""")
    so = tmp_path / "t.so"
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I/usr/local/cuda/include",
                           "-I", os.path.join(ROOT, "paper_2606_12243_b200", "csrc"), str(src), "-o", str(so)])
    call = ctypes.CDLL(str(so)).call
    launch = ctypes.cast(lib["_Z14launch_gemm_tcRK8TcLaunchP11CUstream_st"], ctypes.c_void_p)
    store, add, swiglu, add_norm, qkv_rope = range(5)
    got = lambda *a: call(launch, *a)
    for rows, nt in ((1, 16), (128, 128)):
        assert [got(rows, nt, lo, epi, norm) for lo in (0, 1) for epi in range(5) for norm in (0, 1)] == [0] * 20
    assert got(129, 144, 0, store, 0) == got(256, 256, 0, store, 0) == 0
    for rows, nt in ((129, 144), (256, 256)):
        assert [got(rows, nt, 0, epi, 0) for epi in (add, swiglu, add_norm, qkv_rope)] == [-1] * 4
        assert got(rows, nt, 1, store, 0) == got(rows, nt, 0, store, 1) == -1
    assert got(257, 272, 0, store, 0) == got(17, 16, 0, store, 0) == got(0, 16, 0, store, 0) == -1


def test_no_launch_overtakes_the_first_ones_attributes(tmp_path):
    """Two threads launch a kernel for the first time: the second one's launch may not go out before the kernel's shared-memory limit has
    been raised; a failure is not remembered as done."""
    import subprocess
    from paper_2606_12243_b200 import build as B
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text("""
        #include "common.cuh"
        #include <chrono>
        #include <thread>
        static std::atomic<bool> done[64], ready(false);
        int main() {
            if (once_on_device(done, 3, [] { return (int)VIASD_ECUDA; }) != VIASD_ECUDA) return 1;
            auto set = [] { std::this_thread::sleep_for(std::chrono::milliseconds(300)); ready = true; return (int)VIASD_OK; };
            std::thread first([&] { once_on_device(done, 3, set); });
            std::this_thread::sleep_for(std::chrono::milliseconds(100));
            if (once_on_device(done, 3, set) != VIASD_OK || !ready) return 2;
            first.join();
            int again = 0;
            once_on_device(done, 3, [&] { ++again; return (int)VIASD_OK; });        // done there,
            once_on_device(done, 4, [&] { ++again; return (int)VIASD_OK; });        // not on another device,
            once_on_device(done, 64, [&] { ++again; return (int)VIASD_OK; });       // and always where there is no place
            return again == 2 ? 0 : 3;
        }""")
    subprocess.check_call([B.NVCC, *B.FLAGS, "-I", B.CSRC, str(src), "-o", str(exe), "-lpthread"])
    assert subprocess.call([str(exe)]) == 0
