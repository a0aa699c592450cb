"""The dependencies of captured product slices (csrc/capture_edges.h).  A slice reads its slopes before it
waits for the slice ahead of it, so only the edge from that slice may be programmatic; the one from its
sensor's launch, joined through an event, has to be full.  A graph of the step's shape is captured with
the same functions and asked for its edges (it is never launched)."""
import os
import subprocess

import pytest

from paper_1608_00386_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "capture_edges.h"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { printf("%s: %s\n", #x, cudaGetErrorString(e_)); exit(1); } } while (0)
template <int I> __global__ void k() {}
static std::map<const void*, const char*> names;
template <int I> void launch(const char* name, cudaStream_t s, bool programmatic) {
    names[(const void*)k<I>] = name;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = cfg.blockDim = dim3(1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = programmatic ? 1 : 0;
    CK(cudaLaunchKernelEx(&cfg, k<I>));
}
int main() {
    cudaStream_t s0, s1, s3;
    for (cudaStream_t* s : {&s0, &s1, &s3}) CK(cudaStreamCreateWithFlags(s, cudaStreamNonBlocking));
    cudaEvent_t ev[8];
    for (cudaEvent_t& e : ev) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    auto after = [&](cudaStream_t a, cudaStream_t b, int i) {   // b waits for a
        CK(cudaEventRecord(ev[i], a));
        CK(cudaStreamWaitEvent(b, ev[i], 0));
    };
    CK(cudaStreamBeginCapture(s0, cudaStreamCaptureModeThreadLocal));
    launch<0>("surfaces", s0, false);
    after(s0, s1, 0);
    after(s0, s3, 1);
    launch<1>("low_order", s1, false);
    launch<2>("sensing_a", s0, true);
    after(s1, s3, 2);
    cudaGraphNode_t slice = nullptr;
    CK(mcao::overlap_captured(s3, slice));   // no slice before: nothing changes
    launch<3>("slice_low", s3, false);
    CK(mcao::captured_kernel(s3, &slice));
    after(s0, s3, 3);
    CK(mcao::overlap_captured(s3, slice));
    launch<4>("slice_a", s3, false);
    CK(mcao::captured_kernel(s3, &slice));
    launch<5>("sensing_b", s0, false);
    after(s0, s3, 4);
    CK(mcao::overlap_captured(s3, slice));
    launch<6>("slice_b", s3, false);
    launch<7>("reduction", s3, true);
    after(s1, s0, 5);
    after(s3, s0, 6);
    cudaGraph_t g;
    CK(cudaStreamEndCapture(s0, &g));
    size_t n = 0;
    CK(cudaGraphGetEdges(g, nullptr, nullptr, nullptr, &n));
    std::vector<cudaGraphNode_t> from(n), to(n);
    std::vector<cudaGraphEdgeData> data(n);
    CK(cudaGraphGetEdges(g, from.data(), to.data(), data.data(), &n));
    auto name = [&](cudaGraphNode_t v) {
        cudaGraphNodeType t;
        CK(cudaGraphNodeGetType(v, &t));
        if (t != cudaGraphNodeTypeKernel) return "other";
        cudaKernelNodeParams p{};
        CK(cudaGraphKernelNodeGetParams(v, &p));
        return names.count(p.func) ? names[p.func] : "unknown";
    };
    for (size_t i = 0; i < n; ++i)
        printf("%s %s %s\n", name(from[i]), name(to[i]), data[i].type == cudaGraphDependencyTypeProgrammatic ? "programmatic" : "full");
    return 0;
}
"""


def test_a_slice_overlaps_the_slice_before_alone(tmp_path):
    src, exe = tmp_path / "edges.cu", str(tmp_path / "edges")
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", os.path.join(build.HERE, "csrc"), str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
    edges = sorted(tuple(line.split()) for line in out.stdout.splitlines())
    assert edges == sorted([
        ("surfaces", "low_order", "full"),
        ("surfaces", "slice_low", "full"),
        ("surfaces", "sensing_a", "programmatic"),
        ("low_order", "slice_low", "full"),
        ("slice_low", "slice_a", "programmatic"),
        ("sensing_a", "slice_a", "full"),
        ("sensing_a", "sensing_b", "full"),
        ("slice_a", "slice_b", "programmatic"),
        ("sensing_b", "slice_b", "full"),
        ("slice_b", "reduction", "programmatic"),
    ]), edges
