"""What the library remembers about kernels it has set up is kept per device and may be asked from several threads: the
class is plain C++, compiled and run here with a counter in the place of the CUDA calls."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "vgc_once.cuh"
static vgc::OncePerDevice once;
static std::atomic<int> runs[3][80];
static int call(int device, int kernel, int result = 0)
{
    return once(&runs[0][kernel], device, [&] { if (result == 0) ++runs[device < 0 ? 2 : device][kernel]; return result; });
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main()
{
    CHECK(call(0, 7, 5) == 5 && call(0, 7) == 0 && runs[0][7] == 1);      // a failure is not remembered
    CHECK(call(0, 7, 5) == 0 && runs[0][7] == 1);                         // a success is
    CHECK(call(1, 7) == 0 && runs[1][7] == 1);                            // ... for its own device only
    CHECK(call(-1, 7) == 0 && call(-1, 7) == 0 && runs[2][7] == 2);       // no such device: every time
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([t] { for (int i = 0; i < 4000; ++i) call(i & 1, 10 + (i + t) % 40); });
    for (auto &t : threads) t.join();
    for (int k = 10; k < 50; ++k)
        for (int d = 0; d < 2; ++d) {
            const int before = runs[d][k];
            CHECK(before >= 1 && before <= 8);                            // calls that met may both have run it
            CHECK(call(d, k) == 0 && runs[d][k] == before);               // from then on none does
        }
    for (int k = 0; k < 80; ++k) CHECK(call(0, k) == 0 && runs[0][k] >= 1);   // more than there is room for
    return 0;
}
"""


def test_kernels_are_set_up_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-pthread", "-I",
                    os.path.join(ROOT, "paper_1802_06058_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert done.returncode == 0, done.stdout
