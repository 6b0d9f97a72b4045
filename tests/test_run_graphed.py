"""Work that fails while its graph is being captured: the capture is closed, its
launches are not counted, and the next call captures anew.  The library's own
run_graphed is compiled here against a fake of the CUDA calls it makes, with a
body that throws the way a failed launch does; no GPU is involved.
"""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <string>
typedef int cudaError_t;
typedef void* cudaStream_t;
typedef void* cudaGraph_t;
typedef void* cudaGraphExec_t;
constexpr int cudaSuccess = 0, cudaStreamCaptureModeThreadLocal = 1;
struct CudaError { cudaError_t err; std::string where; };
#define CK(x) do { cudaError_t e_ = (x); if (e_) throw CudaError{e_, #x}; } while (0)
std::atomic<int64_t> g_kernel_launches{0};
struct ncl_kkt_s { bool capturing = false; int prof_on = 0; cudaStream_t cap_stream = nullptr; };
int depth = 0, graphs = 0, replays = 0;
bool broken = false;   // an open capture that saw an error
static cudaError_t cudaStreamBeginCapture(cudaStream_t, int) { return depth++ ? 401 : 0; }
static cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  depth--;
  *g = broken ? nullptr : &graphs;
  graphs += !broken;
  const int e = broken ? 901 : 0;
  broken = false;
  return e;
}
static cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, int) { *x = &replays; return 0; }
static cudaError_t cudaGraphDestroy(cudaGraph_t) { graphs--; return 0; }
static cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { replays++; return 0; }
static cudaError_t cudaGetLastError() { return 0; }
"""

MAIN = r"""
int main() {
  ncl_kkt_s h;
  cudaGraphExec_t exec = nullptr;
  int64_t nodes = 0;
  int calls = 0, fail_at = 1, n = 0, thrown = 0, direct = 0;
  auto body = [&](cudaStream_t) {
    if (!h.capturing) direct++;
    for (int k = 0; k < 5; k++) {
      g_kernel_launches.fetch_add(1);
      if (n == fail_at && k == 2) { broken = true; throw CudaError{701, "launch"}; }
    }
  };
  for (n = 0; n < 4; n++) {
    try {
      run_graphed(&h, &exec, &nodes, &calls, true, nullptr, body);
    } catch (const CudaError& e) {
      thrown += e.err == 701;
    }
    if (depth || h.capturing) return 10 + n;
  }
  // direct, failed capture, capture and replay, replay
  std::printf("%d %d %d %d %d %d\n", thrown, direct, replays, graphs, (int)nodes, (int)g_kernel_launches.load());
  return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="no C++ compiler")
def test_capture_is_closed_when_its_work_throws(tmp_path):
    with open(os.path.join(ROOT, "paper_2510_05885_gb300", "csrc", "api.cu")) as f:
        src = f.read()
    code = re.search(r"((?:struct Capture \{.*?)?template <typename F>\nvoid run_graphed.*?\n\}\n)", src, re.S).group(1)
    cpp = tmp_path / "t.cpp"
    cpp.write_text(FAKE + code + MAIN)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O1", str(cpp), "-o", exe], check=True)
    run = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0
    assert run.stdout.split() == ["1", "1", "2", "0", "5", "15"]
