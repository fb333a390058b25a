"""A kernel's dynamic shared-memory limit under several host threads: kernels whose size differs from plan to plan (slabs, halo tiles, first layers) raise
the limit on first use, and a thread that asked for less must not leave it below what another was promised."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# The runtime's two calls are stand-ins: the first to set the limit is held up until the other thread's call has returned (or waits for this one).
HARNESS = r"""
#include "boda_internal.h"
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <thread>

static std::atomic<int> attribute{0}, calls{0}, finished{0};
static int device = 0;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes)
{
    if (calls++ == 0)
        for (int i = 0; i < 500 && finished == 0; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    attribute = bytes;
    return cudaSuccess;
}
int main(int argc, char** argv)
{
    device = std::atoi(argv[3]);
    boda::DeviceSmemLimit limit;
    const void* kernel = nullptr;
    auto first_call = [&](int bytes) { if (limit.ensure(kernel, (size_t)bytes) != cudaSuccess) std::abort(); ++finished; };
    std::thread a([&] { first_call(std::atoi(argv[1])); });
    while (calls == 0) std::this_thread::yield();
    std::thread b([&] { first_call(std::atoi(argv[2])); });
    a.join();
    b.join();
    first_call(std::atoi(argv[1]));                     // a later call of the smaller plan
    std::printf("%d\n", (int)attribute);
}
"""


@pytest.mark.parametrize("first,second", [(100000, 200000), (200000, 100000)])
@pytest.mark.parametrize("device", [0, 63, 64])
def test_two_first_calls_leave_the_larger_limit(tmp_path, first, second, device):
    src, exe = tmp_path / "limit.cpp", tmp_path / "limit"
    src.write_text(HARNESS)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1606_00094_b200", "csrc"),
                    "-isystem", os.path.join(cuda, "include"), "-o", str(exe), str(src)], check=True)
    res = subprocess.run([str(exe), str(first), str(second), str(device)], capture_output=True, text=True, timeout=60, check=True)
    assert int(res.stdout) == max(first, second)


THREADS = r"""
import threading
import torch
from paper_1606_00094_b200 import binding as B

def layer(shape, tile):
    N, C, H, W, K, R, S, stride, pad, relu = shape
    g = torch.Generator(device="cuda"); g.manual_seed(1)
    x, w = (torch.randint(-3, 4, n, generator=g, device="cuda").float() for n in ((N, C, H, W), (K, C, R, S)))
    want = torch.nn.functional.conv2d(x.double(), w.double(), padding=pad).float()
    return B.ConvPlan(shape, variant=2, tile_id=tile), x, w, want

# two plans of one kernel each time, the first with less shared memory
pairs = [[layer((2, 40, 12, 12, 32, 3, 3, 1, 1, 0), t) for t in (35, 46)],                                                    # slabs of 32 and 256 channels
         [layer((2, 40, 12, h, 64, 3, 3, 1, 1, 0), 5) for h in (12, 100)]]                                                     # halo slabs of few and many rows
B._load_calls()
torch.cuda.synchronize()
for pair in pairs:
    gate, got = threading.Barrier(2), [None, None]
    def run(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            gate.wait()
            got[i] = [pair[i][0](pair[i][1], pair[i][2]) for _ in range(3)]
        stream.synchronize()
    threads = [threading.Thread(target=run, args=(i,)) for i in (0, 1)]
    for t in threads: t.start()
    for t in threads: t.join()
    for i in (0, 1):
        assert got[i] is not None and all(torch.equal(y, pair[i][3]) for y in got[i]), pair[i][0].describe()
assert B.boda_query_status() == 0
print("ok")
"""


@pytest.mark.gpu
def test_first_calls_of_two_sizes_in_two_threads():
    res = subprocess.run([sys.executable, "-c", THREADS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.strip().endswith("ok"), res.stdout + res.stderr
