"""Error paths of the wide-plane factorisation (csrc/factor.cu) on the host.

The compiled object is linked with stand-ins for the CUDA runtime and for the panel kernels'
launchers, which record what is called and fail on request; nothing needs a GPU.  Whatever
fails, the call reports it, every buffer that it took goes back to the allocator, none before
the work on both of its streams has been waited for, and the handle keeps no pointer to one.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1909_01467_gb300", "csrc")

RUNTIME = r"""
#include <cuda_runtime_api.h>
#include <set>
extern std::set<void*> busy;
cudaError_t step(const char* name, cudaStream_t on = nullptr);
static cudaStream_t const kMain = (cudaStream_t)0x10, kAux = (cudaStream_t)0x20;
extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = kAux; return step("stream"); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { busy.erase(s); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)0x30; return step("event"); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return step("record"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) {
  const cudaError_t e = step("wait");
  if (e == cudaSuccess && s == kMain) busy.erase(kAux);   // its work is now waited for through s
  return e;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { static void* p; return &p; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return step("kernel", kMain); }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
}
"""

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include <string>
#include <vector>
#include "internal.h"
static std::string fail_call;                 // name of the call that fails
static int fail_at = 0;                       // on which of its calls
std::set<void*> busy;                         // streams with work that nobody waited for
static std::set<void*> taken;                 // buffers
static bool early = false;
cudaError_t step(const char* name, cudaStream_t on = nullptr) {
  if (fail_call == name && --fail_at == 0) return cudaErrorUnknown;
  if (on) busy.insert(on);
  return cudaSuccess;
}
// ---- launchers of the panel kernels, storage and allocator --------------------------------
namespace lsw {
TileStore tile_store(const Ctx&) { return {0, 1}; }
void split_tile_bytes(const Ctx&, int, size_t& a, size_t& b) { a = b = 64; }
int gj_panel_width_tc() { return 128; }
cudaError_t prepare_gj_panel_tc() { return step("prepare"); }
cudaError_t launch_gj_panel_inverse(Ctx&, int, int, cudaStream_t s) { return step("inverse", s); }
cudaError_t launch_split_panel(Ctx&, int, int, const SplitJobs&, void*, void*, long long, long long,
                               int, cudaStream_t s) { return step("split", s); }
cudaError_t launch_gj_panel_product_tma(Ctx&, int, int, int, int, int, int, const void*,
                                        const void*, long long, long long, int, cudaStream_t s) {
  return step("product", s);
}
cudaError_t launch_factor(Ctx& c);
void* Allocator::get(size_t) const {
  if (step("alloc") != cudaSuccess) return nullptr;
  void* p = malloc(1);
  taken.insert(p);
  return p;
}
void Allocator::put(void* p) const {
  if (!p) return;
  early = early || !busy.empty();
  if (!taken.erase(p)) early = true;
}
}  // namespace lsw
int main(int argc, char** argv) {
  using namespace lsw;
  fail_call = argv[1];
  fail_at = atoi(argv[2]);
  Ctx c;
  c.p.precision = strcmp(argv[3], "C64") ? LSWEEP_C128 : LSWEEP_C64;
  c.dim = 3;
  c.half_rows = atoi(argv[4]) != 0;
  c.stream = (cudaStream_t)0x10;
  c.bmax = 576;
  c.bpmax = 578;
  c.Lmax = 3;
  c.d_fac = (void*)0x1000;
  SubGeom g{};
  g.b = 576;
  g.bp = 578;
  g.L = 3;
  g.bs = half_stride(576);
  c.subs.push_back(g);
  const cudaError_t e = launch_factor(c);
  printf("%d taken %zu early %d kept %d\n", (int)e != 0, taken.size(), (int)early,
         (int)(c.f_fac != nullptr || c.f_subs != nullptr));
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    from paper_1909_01467_gb300 import build
    obj = os.path.join(build.OUT_DIR, "obj", "factor.o")
    if not os.path.exists(obj):
        build.build()
    d = tmp_path_factory.mktemp("factor")
    (d / "h.cu").write_text(HARNESS)
    (d / "rt.cpp").write_text(RUNTIME)
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run([build._nvcc(), "-std=c++17", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"),
                    "-c", str(d / "h.cu"), "-o", str(d / "h.o")], check=True)
    subprocess.run(["g++", "-I" + include, str(d / "rt.cpp"), str(d / "h.o"), obj, "-o", str(d / "h")], check=True)
    return lambda *a: subprocess.run([str(d / "h"), *map(str, a)], check=True, capture_output=True,
                                     text=True).stdout.strip()


@pytest.mark.parametrize("precision,half", [("C64", 1), ("C64", 0), ("C128", 0)])
def test_success_gives_everything_back(harness, precision, half):
    assert harness("none", 0, precision, half) == "0 taken 0 early 0 kept 0"


# panels of 128: five per plane.  The calls of one panel step in order: two splits and a product on
# either side, record, wait, the next panel's inverse on the second stream, record, product, ...
@pytest.mark.parametrize("call,nth", [
    ("prepare", 1), ("alloc", 1), ("alloc", 2), ("alloc", 3), ("stream", 1), ("event", 1),
    ("event", 2), ("inverse", 1), ("inverse", 2), ("inverse", 7), ("split", 1), ("split", 4),
    ("product", 1), ("product", 2), ("product", 3), ("product", 4), ("product", 9), ("record", 1),
    ("record", 2), ("wait", 1), ("wait", 2)])
@pytest.mark.parametrize("half", [1, 0])
def test_failure_gives_everything_back(harness, call, nth, half):
    if call == "alloc" and nth == 3 and not half:
        pytest.skip("two buffers without half rows")
    assert harness(call, nth, "C64", half) == "1 taken 0 early 0 kept 0"
