"""What a quantize call makes of a launch that fails (csrc/abs_launch.h), against a fake of the runtime's calls: only a grid that does not fit sends the call to the two
kernels, and every other error is the call's."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include "abs_launch.h"
#include <cstdio>
#include <cstdlib>

static cudaError_t launch_error, query_error, last_error = cudaSuccess;
static int room, launches, queries, attributes;
static unsigned cluster_blocks;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void*, void**) {
    ++launches;
    attributes = (int)cfg->numAttrs;
    cluster_blocks = attributes == 2 && cfg->attrs[1].id == cudaLaunchAttributeClusterDimension ? cfg->attrs[1].val.clusterDim.x : 0;
    return last_error = launch_error;
}
extern "C" cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
    ++queries;
    *n = room;
    return query_error;
}
extern "C" cudaError_t cudaGetLastError() { const cudaError_t e = last_error; last_error = cudaSuccess; return e; }
extern "C" cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }

static void kernel(int) {}
int main(int, char** v) {
    const Together together = (Together)atoi(v[1]);
    const int grid = atoi(v[2]);
    launch_error = (cudaError_t)atoi(v[3]);
    query_error = (cudaError_t)atoi(v[4]);
    room = atoi(v[5]);
    const abs_status_t rc = quantize_launched(launch_any(together, kernel, grid, 256, nullptr, 1), nullptr);
    printf("%d %d %d %d %u %d\n", (int)rc, launches, queries, attributes, cluster_blocks, (int)last_error);
}
'''
APART, COOPERATIVE, CLUSTER = 0, 1, 2
OK, INVALID, OUT_OF_RESOURCES, TOO_LARGE, BAD_CLUSTER, NO_IMAGE, CAPTURE = 0, 1, 701, 720, 912, 209, 901
NOT_RESIDENT, ERR_CUDA = -1, 6


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch")
    (d / "main.cpp").write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2603_28765_b200", "csrc"), "-isystem", os.path.join(cuda, "include"),
                    "-o", str(d / "main"), str(d / "main.cpp")], check=True)
    return str(d / "main")


@pytest.mark.parametrize("together,grid,launch,query,room,status", [
    (CLUSTER, 8, OK, OK, 142, 0),
    (CLUSTER, 8, OUT_OF_RESOURCES, OK, 142, NOT_RESIDENT),
    (CLUSTER, 8, BAD_CLUSTER, OK, 0, NOT_RESIDENT),         # the runtime says that there is no room
    (CLUSTER, 8, INVALID, OK, 0, NOT_RESIDENT),
    (CLUSTER, 8, BAD_CLUSTER, OK, 142, ERR_CUDA),           # a wrong attribute
    (CLUSTER, 8, INVALID, OK, 142, ERR_CUDA),
    (CLUSTER, 8, NO_IMAGE, NO_IMAGE, 0, ERR_CUDA),          # no code for the device: the question fails like the launch
    (CLUSTER, 8, CAPTURE, OK, 142, ERR_CUDA),
    (CLUSTER, 8, TOO_LARGE, OK, 142, NOT_RESIDENT),
    (COOPERATIVE, 80, OK, OK, 0, 0),
    (COOPERATIVE, 80, TOO_LARGE, OK, 0, NOT_RESIDENT),
    (COOPERATIVE, 80, OUT_OF_RESOURCES, OK, 0, ERR_CUDA),
    (APART, 80, OUT_OF_RESOURCES, OK, 0, ERR_CUDA),
    (COOPERATIVE, 1, OK, OK, 0, 0),
])
def test_only_a_grid_without_room_takes_the_two_kernels(program, together, grid, launch, query, room, status):
    out = subprocess.run([program, *map(str, (together, grid, launch, query, room))], check=True, capture_output=True, text=True).stdout
    rc, launches, queries, attributes, cluster_blocks, left = map(int, out.split())
    assert (rc, launches) == (status, 1)
    assert queries <= (together == CLUSTER and launch != OK)
    assert attributes == (2 if together != APART and grid > 1 else 1) and cluster_blocks == (grid if together == CLUSTER else 0)
    assert left == (launch if status == ERR_CUDA else 0)    # a refusal that is answered is not left for the caller's own error checks
