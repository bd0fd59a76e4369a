"""What the stepping kernels need set up on a device (dynamic shared-memory
limits) is set up on each device, not once per process: the bookkeeping, with
device numbers in the place of devices."""
import os
import re
import subprocess

from paper_1904_06881_gb300 import build as B

SOURCE = r"""
#include <cassert>
#include <thread>
#include <vector>
#include "tlb_internal.h"
int main()
{
    static std::atomic<int> known[64];
    int asked[70] = {};
    auto get = [&](int dev, int answer) {
        return tlb::once_per_device(known, dev, [&] { ++asked[dev]; return answer; });
    };
    for (int round = 0; round < 3; ++round)
        for (int dev = 0; dev < 64; ++dev) assert(get(dev, 100 + dev) == 100 + dev);
    for (int dev = 0; dev < 64; ++dev) assert(asked[dev] == 1);
    assert(get(69, 7) == 7 && get(69, 8) == 8);                // beyond the array: asked each time
    static std::atomic<int> fresh[64];
    int n = 0;
    auto flaky = [&] { return n++ == 0 ? 0 : 5; };             // a failure is asked again
    assert(tlb::once_per_device(fresh, 3, flaky) == 0 && tlb::once_per_device(fresh, 3, flaky) == 5);
    assert(tlb::once_per_device(fresh, 3, flaky) == 5 && n == 2);
    static std::atomic<int> shared[64];
    std::vector<std::thread> th;
    std::atomic<int> wrong{0};
    for (int k = 0; k < 8; ++k)
        th.emplace_back([&, k] {
            for (int dev = 0; dev < 64; ++dev)
                if (tlb::once_per_device(shared, (dev + 8 * k) % 64, [&] { return 1 + (dev + 8 * k) % 64; }) !=
                    1 + (dev + 8 * k) % 64)
                    ++wrong;
        });
    for (auto &t : th) t.join();
    assert(wrong == 0);
    return 0;
}
"""


def test_each_device_is_asked_once(tmp_path):
    src, exe = str(tmp_path / "once.cu"), str(tmp_path / "once")
    with open(src, "w") as fh:
        fh.write(SOURCE)
    subprocess.check_call([B._nvcc()] + B.ARCH + ["-O1", "-std=c++17", "-diag-suppress", "177", "-I", B.CSRC, "-I",
                                                  os.path.join(B.ROOT, "include"), "-o", exe, src])
    subprocess.check_call([exe])


def test_attributes_are_set_per_device():
    """cudaFuncSetAttribute holds on the current device: nowhere behind a per-process flag."""
    for name in os.listdir(B.CSRC):
        with open(os.path.join(B.CSRC, name)) as fh:
            text = fh.read()
        for m in re.finditer("cudaFuncSetAttribute", text):
            assert "once_per_device" in text[max(0, m.start() - 900):m.start()], name
