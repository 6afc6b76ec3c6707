"""The table of what has been done per kernel and device (csrc/once.cuh), compiled for the host: more kernels on two devices than the
library has, several threads, failures, keys beyond the table and devices beyond the mask."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_15014_b200", "csrc")

PROGRAM = r"""
#include "once.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\\n", __LINE__, #x); return 1; } } while (0)
static char kernels[16 * 2000];
int main() {
    static nm::OncePerDevice once;
    static std::atomic<int> calls[2][400];
    std::vector<std::thread> threads;
    for (int t = 0; t < 4; ++t)
        threads.emplace_back([] {
            for (int round = 0; round < 50; ++round)
                for (int k = 0; k < 400; ++k)
                    for (int dev = 0; dev < 2; ++dev) once.run(kernels + 16 * k, dev, [&] { ++calls[dev][k]; return 0; });
        });
    for (auto& t : threads) t.join();
    for (int dev = 0; dev < 2; ++dev)
        for (int k = 0; k < 400; ++k) CHECK(calls[dev][k] == 1);
    int n = 0;
    for (int i = 0; i < 3; ++i) CHECK(once.run(kernels + 16 * 400, 5, [&] { ++n; return 7; }) == 7);  // a failure is tried again
    CHECK(n == 3 && once.run(kernels + 16 * 400, 5, [&] { ++n; return 0; }) == 0 && once.run(kernels + 16 * 400, 5, [&] { ++n; return 1; }) == 0 && n == 4);
    n = 0;
    for (int i = 0; i < 2; ++i) once.run(kernels, 64, [&] { ++n; return 0; });
    for (int i = 0; i < 2; ++i) once.run(kernels, -1, [&] { ++n; return 0; });
    CHECK(n == 4);
    n = 0;
    for (int round = 0; round < 2; ++round)
        for (int k = 0; k < 2000; ++k) once.run(kernels + 16 * k, 9, [&] { ++n; return 0; });
    CHECK(n == 2000 + 2000 - 1024);  // what the table does not hold is done every time
    puts("ok");
}
"""


def test_once_per_kernel_and_device(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-O1", "-pthread", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


def test_every_launch_path_goes_through_the_table():
    """The projections and the linear layers set the attribute nowhere by themselves."""
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh")) and name not in ("api.cu", "probe.cu"):
            assert "cudaFuncSetAttribute(" not in open(os.path.join(CSRC, name)).read().replace("cudaFuncSetAttribute(max", ""), name
