"""lsa_layer_group_host's own bookkeeping, without a GPU: lsa_api.cu (host code only) is compiled with a fake CUDA runtime whose n-th
event creation fails.  The call says so, and the next one does not use events that were never made."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = "/usr/local/cuda/include"

HARNESS = r"""
#include "lsa_api.cu"
#include <cstdlib>
static int creations, fail_at, null_events;
static char handles[4096];
extern "C" {
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)&handles[0]; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  if (++creations == fail_at) return cudaErrorMemoryAllocation;
  *e = (cudaEvent_t)&handles[creations];
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { null_events += e == nullptr; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t e, unsigned) { null_events += e == nullptr; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
const char* cudaGetErrorName(cudaError_t) { return "error"; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
}
namespace lsa {
bool index_shape_supported(int, int) { return true; }
bool attn_shape_supported(int, int, int) { return true; }
bool paged_scores_tc_supported(const IndexArgs&) { return false; }
bool fine_paged_tc_supported(const IndexArgs&) { return false; }
bool index8_supported(const IndexArgs&) { return true; }
bool attn_tc_supported(const AttnArgs&) { return false; }
cudaError_t launch_index8(const IndexArgs&, cudaStream_t, int64_t*) { return cudaSuccess; }
cudaError_t launch_attn(const AttnArgs&, cudaStream_t, int64_t*) { return cudaSuccess; }
}
int main(int argc, char** argv) {
  lsa_params p{};
  p.struct_size = sizeof(p); p.n_heads_idx = 8; p.d_idx = 64; p.page = 64; p.sub_block = 8; p.keep_pages = 8; p.k_sparse = 16; p.k_sink = 4;
  p.k_swa = 32; p.n_heads = 16; p.d_qk = 128; p.d_v = 128; p.sm_scale = 1.f; p.n_layers = 2; p.hi_enable = 1; p.kv_page = 64;
  alignas(256) static unsigned char ws[1 << 20], stage0[1 << 20], stage1[1 << 20], any[4096];
  lsa_ctx* c = nullptr;
  if (lsa_create(&c, 0, nullptr, ws, sizeof(ws)) != LSA_OK) return 10;
  const void* in[2] = {any, any};
  void* out[2] = {any, any};
  void* stage[2] = {stage0, stage1};
  auto call = [&](int64_t n_query, const void* const* kv) {
    return lsa_layer_group_host(c, &p, any, (const float*)any, any, nullptr, any, 0, n_query, 200, in, kv, kv, 128, 128, out, 16, stage, sizeof(stage0));
  };
  if (call(0, nullptr) != LSA_OK) return 11;        // no queries: nothing is looked at
  if (call(3, nullptr) != LSA_ERR_ARG) return 12;
  fail_at = creations + std::atoi(argv[1]);
  if (call(100, in) != LSA_ERR_CUDA) return 13;
  if (call(100, in) != LSA_OK) return 14;
  if (null_events != 0) return 15;
  return lsa_destroy(c) == LSA_OK ? 0 : 16;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INCLUDE):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("host_group")
    src = d / "harness.cpp"
    src.write_text(HARNESS)
    exe = d / "harness"
    # launchers that the test never reaches stay undefined
    subprocess.run(["g++", "-std=c++17", "-O1", "-x", "c++", str(src), "-I", os.path.join(ROOT, "paper_2608_01662_b200", "csrc"), "-I", CUDA_INCLUDE,
                    "-o", str(exe), "-Wl,--unresolved-symbols=ignore-all", "-no-pie"], check=True)
    return str(exe)


@pytest.mark.parametrize("nth", [1, 4, 7, 12, 18])
def test_events_that_could_not_be_made(harness, nth):
    assert subprocess.run([harness, str(nth)], timeout=60).returncode == 0
