"""Scopes that keep streams in step when an error passes through
(csrc/stream_scope.cuh, compiled here against stand-ins of the CUDA calls)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2404_09452_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
pytestmark = pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")), reason="needs the CUDA headers")

PRELUDE = r"""
#include <cstdio>
#include "stream_scope.cuh"
static long id(const void *p) { return (long)p; }
extern "C" const char *cudaGetErrorString(cudaError_t) { return "failed"; }
extern "C" cudaError_t cudaStreamSynchronize(cudaStream_t s) { std::printf("sync %ld\n", id(s)); return cudaSuccess; }
extern "C" cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { std::printf("record %ld on %ld\n", id(e), id(s)); return cudaSuccess; }
extern "C" cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { std::printf("%ld waits for %ld\n", id(s), id(e)); return cudaSuccess; }
struct Buffer { ~Buffer() { std::printf("release\n"); } };
using namespace dfjk;
"""


def _run(tmp_path, main):
    (tmp_path / "t.cpp").write_text(PRELUDE + main)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", CUDA, "-o", exe, str(tmp_path / "t.cpp")], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()


@pytest.mark.parametrize("stream", [0, 7])  # 0: the legacy default stream
@pytest.mark.parametrize("throws", [0, 1])
def test_drain_before_release(tmp_path, stream, throws):
    out = _run(tmp_path, "int main() { try { Buffer b; StreamDrain d{(cudaStream_t)%d}; if (%d) throw 1; } catch (int) {} }"
               % (stream, throws))
    assert out == ["sync %d" % stream, "release"]


SIDE = r"""
int main() {
  const cudaStream_t st = (cudaStream_t)%d, side = (cudaStream_t)2;
  try {
    SideScope s(st, side, (cudaEvent_t)11, (cudaEvent_t)12);
    s.fork();
    if (%d) throw 1;
    s.join();
  } catch (int) {}
}
"""


@pytest.mark.parametrize("throws", [0, 1])
def test_side_stream_is_joined(tmp_path, throws):
    out = _run(tmp_path, SIDE % (1, throws))
    assert out == ["record 11 on 1", "2 waits for 11", "record 12 on 2", "1 waits for 12"]


def test_one_stream_needs_no_events(tmp_path):
    assert _run(tmp_path, SIDE % (2, 1)) == []


def test_builds_fork_through_the_scope():
    text = open(os.path.join(CSRC, "dfjk_api.cu")).read()
    build = text[text.index("void build_one("):text.index("// Buffers of the density build")]
    assert "side.fork()" in build and "cudaStreamWaitEvent" not in build
