"""Several host threads, each with a context of its own, may make their first call at the same time: what the library looks up
once per process must not be seen half made.  The two functions are taken from the source and run against stand-ins for the
CUDA calls, which answer slowly."""
import os
import re
import shutil
import subprocess

import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_00130_b200", "csrc", "tc_common.cuh")

STAND_INS = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
typedef void (*EncodeTiledFn)(int);
enum cudaError_t { cudaSuccess = 0 };
enum cudaDriverEntryPointQueryResult { cudaDriverEntryPointSuccess = 0 };
enum { cudaEnableDefault = 0 };
enum cudaDeviceAttr { cudaDevAttrMultiProcessorCount = 16 };
static void encode(int) {}
static void slow() { std::this_thread::sleep_for(std::chrono::milliseconds(300)); }
static cudaError_t cudaGetDriverEntryPoint(const char*, void** p, int, cudaDriverEntryPointQueryResult* q) {
  slow(); *p = reinterpret_cast<void*>(&encode); *q = cudaDriverEntryPointSuccess; return cudaSuccess;
}
static cudaError_t cudaGetLastError() { return cudaSuccess; }
static cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
static cudaError_t cudaDeviceGetAttribute(int* n, cudaDeviceAttr, int) { slow(); *n = 123; return cudaSuccess; }
"""
MAIN = r"""
int main() {
  std::atomic<int> bad{0};
  std::vector<std::thread> ts;
  for (int i = 0; i < 8; ++i)
    ts.emplace_back([&, i] {
      std::this_thread::sleep_for(std::chrono::milliseconds(20 * i));
      if (encode_fn() != &encode) ++bad;
      if (num_sms() != 123) ++bad;
    });
  for (auto& t : ts) t.join();
  std::printf("%d", bad.load());
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_first_calls_from_several_threads(tmp_path):
    text = open(HEADER).read()
    parts = [re.search(r"^%s\(\) \{.*?^\}" % f, text, re.S | re.M).group(0) for f in ("EncodeTiledFn encode_fn", "int num_sms")]
    src = tmp_path / "t.cpp"
    src.write_text(STAND_INS + "\n".join(parts) + MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-o", str(tmp_path / "t"), str(src)], check=True)
    assert subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=60).stdout == "0"
