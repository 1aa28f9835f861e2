"""The launch graph's argument updates (rvh_graph.cu), on the host against
stand-ins for the CUDA runtime's graph calls: every launch runs with its own
call's arguments, batches without counters that repeat update no node, and a
batch with counters is neither compared with the one before nor copied for it."""
import os
import shutil
import subprocess

import pytest

from paper_2012_12618_gb300 import build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>
#include "rvh_graph.cu"

using namespace rvh;

namespace rvh {
bool fused_ext(const FusedArgs& a) { return a.f[0].line_model != 0; }
const void* fused_kernel_fn(int dim, bool ext) { return (const void*)(size_t)(16 + 2 * dim + ext); }
const void* worklist_kernel_fn() { return (const void*)8; }
int fused_threads() { return 256; }
}  // namespace rvh

static int n_updates, n_exec, live, n_graphs;
struct Node { FusedArgs a; unsigned grid; };
struct Graph { std::map<int, Node> nodes; };
static Graph* last_launched;
static Node node(const cudaKernelNodeParams* p) { return Node{*(const FusedArgs*)p->kernelParams[0], p->gridDim.x}; }

extern "C" {
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = (cudaGraph_t) new Graph(); ++n_graphs; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (Graph*)g; --n_graphs; return cudaSuccess; }
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* n, cudaGraph_t g, const cudaGraphNode_t*, size_t,
                                   const cudaKernelNodeParams* p) {
  Graph* G = (Graph*)g;
  const int id = (int)G->nodes.size() + 1;
  G->nodes[id] = node(p);
  *n = (cudaGraphNode_t)(size_t)id;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
  *x = (cudaGraphExec_t) new Graph(*(Graph*)g);
  ++n_exec;
  ++live;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete (Graph*)x; --live; return cudaSuccess; }
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t x, cudaGraphNode_t n, const cudaKernelNodeParams* p) {
  ((Graph*)x)->nodes[(int)(size_t)n] = node(p);
  ++n_updates;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) { last_launched = (Graph*)x; return cudaSuccess; }
}

static int bad;
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); ++bad; } } while (0)

// a frame (its buffers' address) counted in copy slot of the counters (-1: without counters)
static FusedArgs make(size_t frame, int slot) {
  FusedArgs a;
  memset((void*)&a, 0, sizeof(a));
  a.f[0].az = (const float*)frame;
  if (slot < 0) return a;
  a.stats = (unsigned long long*)(size_t)(4096 + 128 * slot);
  a.stats_next = (unsigned long long*)(size_t)(4096 + 128 * (slot ^ 1));
  return a;
}

static void run(LaunchGraph& g, const FusedArgs& a, int grid, bool with_work) {
  CHECK(g.launch(a, 2, grid, 100, with_work, nullptr) == cudaSuccess);
  CHECK(last_launched->nodes.size() == (with_work ? 2u : 1u));
  for (auto& kv : last_launched->nodes) CHECK(memcmp(&kv.second.a, &a, sizeof(a)) == 0);
  CHECK(last_launched->nodes[with_work ? 2 : 1].grid == (unsigned)grid);  // the fused kernel's
}

int main() {
  for (int with_work = 0; with_work < 2; ++with_work) {
    LaunchGraph g;
    // a repeated batch without counters: no update
    for (int k = 0; k < 5; ++k) run(g, make(64, -1), 10, with_work);
    CHECK(n_updates == 0 && g.builds == 1 && g.replays == 4);
    // one frame again and again with its counters, neither compared nor copied
    for (int k = 0; k < 6; ++k) run(g, make(64, k & 1), 10, with_work);
    CHECK(n_updates == 6 * (1 + with_work) && !g.have_last && g.last.stats == nullptr);
    // the arguments of before the counters, now outdated in the graph
    run(g, make(64, -1), 10, with_work);
    // other frames and grids
    for (int k = 0; k < 12; ++k) run(g, make(64 + 64 * (k % 3), k % 2 - 1), 10 + k % 4, with_work);
    CHECK(g.builds == 1 && g.replays == 23);
    n_updates = 0;
    // the other kernel instantiation: another graph
    FusedArgs e = make(64, 0);
    e.f[0].line_model = 1;
    run(g, e, 7, with_work);
    CHECK(g.builds == 2 && n_graphs == 1);
  }
  CHECK(live == 0 && n_graphs == 0);
  return bad ? 1 : 0;
}
"""


def test_argument_updates(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    src, exe = tmp_path / "graph.cpp", str(tmp_path / "graph")
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-I" + inc, "-I" + build.CSRC, "-I" + build.INCLUDE, str(src),
                    "-o", exe], check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
