"""What the library keeps between calls: kernel attributes, set once in every CUDA context, however many threads make the first call."""
import subprocess
import sys
import textwrap

import pytest

from paper_2609_36938_b200 import build


def test_a_first_call_from_many_threads_runs_once_and_is_waited_for(tmp_path):
    src = tmp_path / "once.cu"
    src.write_text(textwrap.dedent("""
        #include <chrono>
        #include <thread>
        #include <vector>
        #include "janus_common.cuh"
        uint64_t janus::current_context_id() { return 0; }
        int main() {
            janus::once_per_context once;
            std::atomic<int> runs{0}, early{0};
            int value[3] = {0, 0, 0};                       // plain memory: visible to whoever has returned from run_in
            std::vector<std::thread> threads;
            for (int i = 0; i < 24; ++i)
                threads.emplace_back([&, i] {
                    const int c = i % 3;
                    once.run_in(100 + c, [&] {
                        std::this_thread::sleep_for(std::chrono::milliseconds(20));
                        ++runs;
                        value[c] = 1;
                        return cudaSuccess;
                    });
                    if (value[c] != 1) ++early;
                });
            for (auto& t : threads) t.join();
            for (int i = 0; i < 2; ++i) once.run_in(0, [&] { ++runs; return cudaSuccess; });        // no context yet: nothing to remember
            for (int i = 0; i < 2; ++i) once.run_in(7, [&] { ++runs; return i == 0 ? cudaErrorUnknown : cudaSuccess; });      // a failure is not remembered
            once.run_in(7, [&] { ++runs; return cudaSuccess; });
            return runs == 7 && early == 0 ? 0 : 1;
        }
    """))
    exe = tmp_path / "once"
    subprocess.check_call([build._nvcc(), "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0


@pytest.mark.gpu
def test_calls_work_in_every_context_of_a_device():
    """The C library in a process with two contexts on one device, without torch: each needs the kernels' attributes."""
    build.build()
    script = textwrap.dedent("""
        import ctypes, struct, sys
        cu, lib = ctypes.CDLL("libcuda.so.1"), ctypes.CDLL(sys.argv[1])
        def ck(r):
            assert r == 0, r
        ck(cu.cuInit(0))
        dev, primary, second = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_void_p()
        ck(cu.cuDeviceGet(ctypes.byref(dev), 0))
        ck(cu.cuDevicePrimaryCtxRetain(ctypes.byref(primary), dev))
        ck(cu.cuCtxCreate_v2(ctypes.byref(second), 0, dev))
        lib.janus_topk.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 4 + [ctypes.c_size_t] + [ctypes.c_void_p] * 2
        lib.janus_indexer_topk_static.argtypes = [ctypes.c_void_p, ctypes.c_int64] * 2 + [ctypes.c_void_p] * 2 + [ctypes.c_int64] + [ctypes.c_void_p] * 3 + [
            ctypes.c_int] * 3 + [ctypes.c_int64] * 2 + [ctypes.c_int] * 3 + [ctypes.c_void_p] * 5
        n, k = 10000, 5
        scores = struct.pack(f"{n}f", *[float((i * 7919) % n) for i in range(n)])
        for ctx in (primary, second, primary):
            ck(cu.cuCtxSetCurrent(ctx))
            src, idx = ctypes.c_void_p(), ctypes.c_void_p()
            ck(cu.cuMemAlloc_v2(ctypes.byref(src), ctypes.c_size_t(4 * n)))
            ck(cu.cuMemAlloc_v2(ctypes.byref(idx), ctypes.c_size_t(4 * k)))
            ck(cu.cuMemcpyHtoD_v2(src, scores, ctypes.c_size_t(4 * n)))
            ck(lib.janus_topk(src, n, 1, n, 0, 0, k, idx, None, None, None, 0, None, None))
            ck(cu.cuCtxSynchronize())
            got = (ctypes.c_int * k)()
            ck(cu.cuMemcpyDtoH_v2(got, idx, ctypes.c_size_t(4 * k)))
            assert sorted((i * 7919) % n for i in got) == list(range(n - k, n)), list(got)
            # one key of 64 that looks at the query, on the library's own scratch: every context has an array of its own
            ops, row = ctypes.c_void_p(), [0x3f80] * 64
            ck(cu.cuMemAlloc_v2(ctypes.byref(ops), ctypes.c_size_t(1 << 16)))
            ck(cu.cuMemsetD8_v2(ops, 0, ctypes.c_size_t(1 << 16)))
            q, w, keys = ops.value, ops.value + 4096, ops.value + 8192
            ck(cu.cuMemcpyHtoD_v2(ctypes.c_uint64(q), struct.pack("256H", *(row * 4)), ctypes.c_size_t(512)))
            ck(cu.cuMemcpyHtoD_v2(ctypes.c_uint64(w), struct.pack("4f", 1, 1, 1, 1), ctypes.c_size_t(16)))
            ck(cu.cuMemcpyHtoD_v2(ctypes.c_uint64(keys + 128 * 37), struct.pack("64H", *row), ctypes.c_size_t(128)))
            ck(lib.janus_indexer_topk_static(q, 256, keys, 64, w, None, 0, None, None, None, 1, 4, 64, 64, 0, 0, 0, 1, idx, None, None, None, None))
            ck(cu.cuCtxSynchronize())
            ck(cu.cuMemcpyDtoH_v2(got, idx, ctypes.c_size_t(4)))
            assert got[0] == 37, got[0]
    """)
    subprocess.run([sys.executable, "-c", script, build.LIB_PATH], check=True, timeout=120)


def test_page_demand_plan_keeps_to_the_clusters_of_the_device(tmp_path):
    """The rule that sizes page demand launches: no cluster above what the device takes, a slice of one chunk where marking needs it."""
    src = tmp_path / "plan.cpp"
    src.write_text(textwrap.dedent("""
        #include "page_demand_plan.h"
        using namespace janus;
        int main() {
            const int64_t idx[] = {0, 1, 8192, 8193, 131072, 131073, 1 << 26};
            for (int largest = 8; largest <= 16; largest += 8)
                for (int64_t n_idx : idx)
                    for (int64_t w = 1; w < (int64_t(1) << 26); w += 1 + w / 7) {
                        const PdPlan p = page_demand_plan(n_idx, static_cast<int>(w), largest);
                        if (p.cluster > largest || p.cluster < 4 || p.clusters < 1 || p.clusters > PD_MAX_CLUSTERS) return 1;
                        if (p.one_launch && (p.clusters != 1 || w > p.cluster * PD_THREADS || n_idx > PD_ONE_LAUNCH_INDICES)) return 2;
                        if (!p.one_launch && p.clusters < PD_MAX_CLUSTERS && w > int64_t(p.cluster) * p.clusters * PD_THREADS) return 3;
                    }
            return 0;
        }
    """))
    exe = tmp_path / "plan"
    subprocess.check_call(["g++", "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0


def test_topk_clusters_split_the_rows_they_are_launched_for(tmp_path):
    """The rules that share rows out: cluster sizes that the device's kernels take, no cluster for rows that it would leave to its first CTA, and
    rows of a length that only the device knows are split under the same sizes as the others."""
    src = tmp_path / "plan.cpp"
    src.write_text(textwrap.dedent("""
        #include "topk_plan.h"
        using namespace janus;
        int main() {
            for (int64_t rows = 1; rows <= 200; ++rows) {
                const int unknown = topk_cluster_size(rows, -1.);
                if (unknown != 1 && unknown != 2 && unknown != 4 && unknown != 8) return 1;
                if (topk_split_from(unknown) <= 8192) return 2;
                for (double n = 0; n < 300e3; n += 500) {
                    const int c = topk_cluster_size(rows, n);
                    if (c != 1 && c != 2 && c != 4 && c != 8) return 3;
                    if (c > 1 && n < topk_split_from(c)) return 4;
                    if (c > 1 && unknown == 1) return 5;
                }
            }
            // on both sides of the lines in rows: what measured faster there
            const struct { int rows; double n; int cluster; } at[] = {{8, 40e3, 8}, {9, 40e3, 2}, {9, 50e3, 4}, {14, 50e3, 4}, {15, 50e3, 2}, {30, 40e3, 2},
                                                                      {31, 40e3, 1}, {36, 40e3, 1}, {33, 112e3, 8}, {34, 112e3, 2}, {74, 64e3, 2}, {75, 64e3, 1}};
            for (const auto& a : at)
                if (topk_cluster_size(a.rows, a.n) != a.cluster) return 6;
            return 0;
        }
    """))
    exe = tmp_path / "plan"
    subprocess.check_call(["g++", "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0
