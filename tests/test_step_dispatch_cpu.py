"""mclbm_step's choice of kernels when a launch is refused, on the host: the entry points of
csrc/mclbm_abi.cu linked with a fake of the CUDA runtime and of the launchers, whose cluster and grid
launches return a given error."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1511_04552_gb300", "csrc")

FAKE = r"""
#include <cstdio>
#include <cstdlib>
#include "mclbm_internal.h"
namespace {
cudaError_t grid_error, cluster_error;
bool with_grid;
int grids, clusters, captured, graph_steps, singles;
bool capturing;
cudaStream_t asked;
}
namespace mcl {
StepConfig choose_step_config(int, int, int) { return StepConfig{}; }
cudaError_t prepare_cluster(StepConfig* c, const Layout&, bool, bool, cudaStream_t st) {
  asked = st;
  c->cl_ctas = 16;
  c->cl_run = with_grid ? 400 : 64;
  c->cl_threads = 128;
  return cudaSuccess;
}
cudaError_t prepare_resident(StepConfig* c, const Layout&, bool, bool) {
  c->re_gx = c->re_gy = 4;
  c->re_ctas = with_grid ? 16 : 0;
  return cudaSuccess;
}
cudaError_t launch_cluster(const StepArgs&, const StepConfig&, int, uint32_t, uint32_t*, cudaStream_t) {
  ++clusters;
  return cluster_error;
}
cudaError_t launch_resident(const StepArgs&, const StepConfig&, int, void*, uint32_t*, cudaStream_t) {
  ++grids;
  return grid_error;
}
cudaError_t launch_step(const StepArgs&, const StepConfig&, const CUtensorMap*, cudaStream_t) {
  ++(capturing ? captured : singles);
  return cudaSuccess;
}
cudaError_t launch_epoch_advance(uint32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_init(void*, const Layout&, const StepConsts&, const float*, int, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_residual(const void*, const Layout&, const StepConsts&, float*, bool, double*, double*,
                            cudaStream_t) {
  return cudaSuccess;
}
// not reached with the step kernel that choose_step_config gives here
cudaError_t prepare_step(StepConfig*, const Layout&) { return cudaErrorUnknown; }
cudaError_t make_state_tensor_map(CUtensorMap*, void*, const Layout&, int, int) {
  return cudaErrorUnknown;
}
cudaError_t make_two_step_tensor_map(CUtensorMap*, void*, const Layout&) { return cudaErrorUnknown; }
cudaError_t prepare_two_f32(StepConfig*, const Layout&) { return cudaErrorUnknown; }
cudaError_t launch_two_f32(const StepArgs&, const StepConfig&, const CUtensorMap*, cudaStream_t) {
  return cudaErrorUnknown;
}
int step_tile_width(const StepConfig&) { return 32; }
}  // namespace mcl
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorName(cudaError_t) { return "error"; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  a->type = cudaMemoryTypeDevice;
  a->device = 0;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  capturing = true;
  captured = 0;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  *g = nullptr;
  return cudaSuccess;
}
// a graph is the number of its steps
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>((size_t)captured);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  graph_steps += (int)(size_t)e;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
int main(int, char** v) {
  with_grid = std::atoi(v[1]) != 0;
  grid_error = (cudaError_t)std::atoi(v[2]);
  cluster_error = (cudaError_t)std::atoi(v[3]);
  mclbm_t* h = nullptr;
  if (mclbm_create(32, 32, 1e3, 6.2, 0.01, 20e-9, nullptr, &h)) return 1;
  const size_t bytes = mclbm_buffer_bytes(h);
  void* buf = std::aligned_alloc(256, (bytes + 255) / 256 * 256);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(0x1234);
  if (mclbm_bind(h, buf, bytes, st) || mclbm_init(h, 0, nullptr)) return 2;
  const int first = mclbm_step(h, 37), second = mclbm_step(h, 37);
  std::printf("%d %d %d %d %d %d %d\n", first, second, (int)mclbm_steps_done(h), grids, clusters,
              graph_steps + singles, asked == st);
  return 0;
}
"""

COOPERATIVE, CLUSTER, CONFIGURATION, RESOURCES, FAULT = 720, 912, 9, 701, 719
ECUDA = -4


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or
                                                            "/usr/local/cuda/bin/nvcc")))
    d = tmp_path_factory.mktemp("dispatch")
    (d / "fake.cpp").write_text(FAKE)
    exe = str(d / "dispatch")
    # what the scenarios do not reach is left out, so that the fake need not have it
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffunction-sections", "-fdata-sections", "-x", "c++", os.path.join(CSRC, "mclbm_abi.cu"),
                    os.path.join(CSRC, "mclbm_model.cpp"), str(d / "fake.cpp"),
                    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", os.path.join(cuda, "include"), "-ldl", "-o", exe,
                    "-Wl,--gc-sections"], check=True)

    def go(grid, grid_error, cluster_error):
        env = {k: v for k, v in os.environ.items() if not k.startswith("MCLBM_")}
        out = subprocess.run([exe, str(int(grid)), str(grid_error), str(cluster_error)], env=env,
                             capture_output=True, text=True, check=True).stdout
        return tuple(int(x) for x in out.split())
    return go


def test_resident_kernels_take_the_calls(run):
    # return codes, steps done; launches of the grid, of the cluster; steps one by one; bound stream asked
    assert run(False, 0, 0) == (0, 0, 74, 0, 2, 0, 1)
    assert run(True, 0, 0) == (0, 0, 74, 2, 0, 2, 1)  # the odd last steps


@pytest.mark.parametrize("error", [CLUSTER, CONFIGURATION, RESOURCES])
def test_refused_cluster_goes_on_step_by_step(run, error):
    """The first call's launch is refused and its steps go one by one, as do all later ones."""
    assert run(False, 0, error) == (0, 0, 74, 0, 1, 74, 1)


def test_refused_grid_and_cluster_go_on_step_by_step(run):
    assert run(True, COOPERATIVE, 0) == (0, 0, 74, 1, 2, 0, 1)
    assert run(True, COOPERATIVE, CLUSTER) == (0, 0, 74, 1, 1, 74, 1)


def test_other_errors_are_reported(run):
    for grid, errors in ((False, (0, FAULT)), (True, (FAULT, 0))):
        first, second, steps = run(grid, *errors)[:3]
        assert first == second == ECUDA and steps == 0
