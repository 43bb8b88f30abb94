"""Host logic around a packed handle's streams and buffers (gs_api.cu and gs_pool.cu), compiled with
g++ against a small stand-in for the CUDA runtime: which launches may overlap the one before them,
what the driver is asked on each call, and when idle device buffers go back to the device.
No GPU is needed: streams are plain numbers and device memory is a byte count.
"""
import os
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
CSRC = ROOT / "paper_2609_33977_gb300" / "csrc"
CUDA_INCLUDE = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"

FAKES = r"""
#include "gs_common.cuh"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <new>
#include <string>

static std::map<void*, size_t> g_live;          // device allocations
static size_t g_used = 0, g_capacity = size_t(1) << 34;
static int g_asked = 0;                          // capture queries
static cudaStreamCaptureStatus g_capture = cudaStreamCaptureStatusNone;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_used + n > g_capacity) return cudaErrorMemoryAllocation;
  *p = std::malloc(1);
  g_live[*p] = n;
  g_used += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  g_used -= g_live.at(p);
  g_live.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = g_capacity - g_used; *t = size_t(1) << 34; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long* id) { *id = (unsigned long long)(uintptr_t)s + 7; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) { ++g_asked; *st = g_capture; return cudaSuccess; }
}

void gs::decode_release(gs_packed*) {}   // no scratch of other streams here

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)
static cudaStream_t stream(int i) { return reinterpret_cast<cudaStream_t>((uintptr_t)(i * 64)); }   // 0: the legacy stream
// a handle as gs_pack leaves it
static gs_packed* packed(cudaStream_t s) {
  gs_packed* p = new gs_packed();
  gs::handle_on_stream(p, s);
  p->fresh = 1;
  return p;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx or not (CUDA_INCLUDE / "cuda_runtime.h").exists():
        pytest.skip("g++ or the CUDA headers are not available")
    d = tmp_path_factory.mktemp("use")

    def build_and_run(name, body):
        src = d / f"{name}.cpp"
        src.write_text(FAKES + "int main() {\n" + body + "\nreturn 0;\n}\n")
        exe = d / name
        # what the tested calls never reach (kernels, the rest of the CUDA runtime) stays unresolved
        r = subprocess.run([gxx, "-std=c++17", "-O1", "-x", "c++", str(CSRC / "gs_api.cu"), str(CSRC / "gs_pool.cu"),
                            str(src), "-x", "none", f"-I{CSRC}", f"-I{ROOT / 'include'}", f"-I{CUDA_INCLUDE}", "-no-pie",
                            "-pthread", "-Wl,--unresolved-symbols=ignore-all", "-o", str(exe)],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stdout + r.stderr
    return build_and_run


@pytest.mark.parametrize("s", [0, 1])
def test_no_launch_overlaps_packing_until_an_ordinary_one_is_queued(run, s):
    """Any number of threads may ask before the first launch is in the stream, and a launch that
    fails or is captured does not follow packing: each of them still gets an ordinary launch."""
    run(f"overlap{s}", f"""
      gs_packed* p = packed(stream({s}));
      CHECK(!gs::may_overlap(p, stream({s})));
      CHECK(!gs::may_overlap(p, stream({s})));      // a second thread, before the first one's launch is queued
      g_capture = cudaStreamCaptureStatusActive;
      gs::launch_queued(p, stream({s}));            // captured, not run (the legacy stream cannot be)
      g_capture = cudaStreamCaptureStatusNone;
      CHECK({s} == 0 || !gs::may_overlap(p, stream({s})));
      gs::launch_queued(p, stream(3));              // on another stream
      CHECK({s} == 0 || !gs::may_overlap(p, stream({s})));
      CHECK(gs::may_overlap(p, stream(3)));         // ordered behind packing by an event
      gs::launch_queued(p, stream({s}));
      CHECK(gs::may_overlap(p, stream({s})));
      gs_packed* q = packed(cudaStreamPerThread);   // one address, a stream in every thread
      gs::launch_queued(q, cudaStreamPerThread);
      CHECK(!gs::may_overlap(q, cudaStreamPerThread));
      gs_packed* r = packed(stream(0));             // the legacy stream's other name
      CHECK(!gs::may_overlap(r, cudaStreamLegacy));
      gs::launch_queued(r, cudaStreamLegacy);
      CHECK(gs::may_overlap(r, stream(0)));
    """)


def test_any_allocation_that_finds_the_device_full_releases_idle_buffers(run):
    """The split scratch of a second stream (lib_malloc) as well as a handle's own buffers."""
    run("full", """
      g_capacity = 100 << 20;
      gs_packed* p = packed(stream(1));
      void *a = nullptr, *b = nullptr;
      CHECK(gs::handle_malloc(p, &a, 60 << 20) == GS_OK);
      gs_free(p);
      CHECK(g_used == (60 << 20));                          // kept, idle
      CHECK(gs::lib_malloc(&b, 90 << 20) == GS_OK && b);    // fits only once it is gone
      CHECK(g_used == (90 << 20));
      CHECK(gs::lib_malloc(&a, 90 << 20) == GS_ERR_OOM && !a);
      cudaFree(b);
      p = packed(stream(1));
      CHECK(gs::handle_malloc(p, &a, 60 << 20) == GS_OK);
      gs_free(p);
      gs_packed* q = packed(stream(2));
      CHECK(gs::handle_malloc(q, &a, 90 << 20) == GS_OK);
      gs_free(q);
    """)


def test_idle_buffers_age_in_packs_and_releases(run):
    """A program that goes on packing without releasing gives unused buffers back too."""
    run("age", """
      gs_packed* p = packed(stream(1));
      void* a = nullptr;
      CHECK(gs::handle_malloc(p, &a, 1 << 20) == GS_OK);
      gs_free(p);
      CHECK(g_live.size() == 1);
      gs_packed* q = packed(stream(2));                 // other stream: does not take it
      CHECK(gs::handle_malloc(q, &a, 512) == GS_OK);
      CHECK(g_live.size() == 2);
      for (int i = 0; i < 1000; ++i) {
        gs_packed* r = packed(stream(2));
        for (int k = 0; k < 9; ++k) CHECK(gs::handle_malloc(r, &a, 512) == GS_OK);   // never released
      }
      CHECK(g_live.size() == 1 + 9000);
    """)


def test_trim_gives_every_idle_buffer_back_and_keeps_those_in_use(run):
    run("trim", """
      void* a = nullptr;
      gs_packed* keep = packed(stream(1));
      CHECK(gs::handle_malloc(keep, &a, 4096) == GS_OK);
      for (int s = 0; s < 3; ++s) {
        gs_packed* p = packed(stream(s));
        for (int k = 0; k < 5; ++k) CHECK(gs::handle_malloc(p, &a, (size_t)1 << (10 + k)) == GS_OK);
        gs_free(p);
      }
      CHECK(g_live.size() == 16);
      gs_trim();
      CHECK(g_live.size() == 1 && g_used == 4096);
      gs_free(keep);
      gs_trim();
      CHECK(g_live.empty());
    """)


def test_capture_is_asked_about_only_where_it_can_be(run):
    """The legacy stream cannot be captured: a call there asks the driver nothing.  Elsewhere a call
    asks once, and a handle captured or used on another stream loses its claim to the pool."""
    run("capture", """
      gs_packed* p[3] = {packed(stream(0)), packed(stream(0)), packed(stream(0))};
      g_capture = cudaStreamCaptureStatusActive;   // were it asked
      for (int i = 0; i < 4; ++i) gs::handles_used(p, 3, stream(0));
      gs::launch_queued(p[0], stream(0));
      gs::handles_used(p, 1, stream(0));
      CHECK(g_asked == 0 && !p[0]->shared && !p[2]->shared && gs::may_overlap(p[0], stream(0)));
      g_capture = cudaStreamCaptureStatusNone;
      gs::handles_used(p, 1, stream(1));
      CHECK(g_asked == 0 && p[0]->shared && !p[1]->shared);
      gs_packed* q[3] = {packed(stream(1)), packed(stream(1)), packed(stream(2))};
      gs::handles_used(q, 2, stream(1));
      CHECK(g_asked == 1 && !q[0]->shared && !q[1]->shared);
      g_capture = cudaStreamCaptureStatusActive;
      gs::handles_used(q, 3, stream(1));
      CHECK(g_asked == 2 && q[0]->shared && q[1]->shared && q[2]->shared);
      gs::handles_used(q, 3, stream(1));
      CHECK(g_asked == 2);
    """)
