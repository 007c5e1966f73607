"""A call that runs part of its work on a second stream joins it on its error paths too
(csrc/side_chain.h), with stand-ins for the CUDA calls that write down their order."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_10863_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include <cstdio>
#include <string>
#include "side_chain.h"
static std::string calls;
static int fail_record = 0;
extern "C" {
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t s) {
  calls += s == (cudaStream_t)2 ? " record-side" : " record-main";
  return fail_record ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) {
  calls += s == (cudaStream_t)1 ? " main-waits" : " side-waits";
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { calls += " sync-side"; return cudaSuccess; }
}
int main() {
  auto run = [](cudaError_t e) {
    calls.clear();
    const cudaError_t r = run_with_side((cudaStream_t)1, (cudaStream_t)2, (cudaEvent_t)3,
                                        [&] { calls += " body"; return e; });
    std::printf("%d%s\n", (int)(r == e), calls.c_str());
  };
  run(cudaSuccess);
  run(cudaErrorInvalidConfiguration);
  fail_record = 1;
  run(cudaErrorInvalidConfiguration);
}
"""


@pytest.mark.skipif(not shutil.which("g++") or not os.path.isdir(os.path.join(CUDA, "include")),
                    reason="needs g++ and the CUDA headers")
def test_errors_join_the_side_stream(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-I" + os.path.join(CUDA, "include"), str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")[:3]
    assert out == ["1 body", "1 body record-side main-waits", "1 body record-side sync-side"]


def test_the_triangle_product_uses_it():
    """The only product with a second stream starts its chains through run_with_side."""
    text = open(os.path.join(CSRC, "kernels.cu")).read()
    body = text[text.index("static cudaError_t matvec_tri_cached("):]
    assert "run_with_side(" in body[:body.index("\n}\n")]
