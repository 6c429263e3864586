"""The pinned staging of the batched training launch (qsim_staging.h) against a stand-in of the CUDA
calls it makes: buffers are kept per device, and never handed out while a copy may read
them (runs without a GPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "qsim_staging.h"
#include <cstdio>
#include <cstdlib>
static int device, allocs, frees, record_fails, sync_fails;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return record_fails ? cudaErrorInvalidValue : cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return sync_fails ? cudaErrorInvalidValue : cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { ++allocs; *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void*) { ++frees; return cudaSuccess; }
}
int main() {
    for (int i = 0; i < 10; ++i) {  // a thread that alternates between two devices
        device = i & 1;
        qsim::Staging* s = qsim::staging_slot();
        if (!s || !s->take(1000)) return 1;
        s->used(nullptr);
    }
    if (allocs != 4 || frees != 0) return 2;
    device = 2;
    qsim::Staging* s = qsim::staging_slot();
    record_fails = sync_fails = 1;  // nothing tells when the copy is done
    void* p = s->take(1000);
    s->used(nullptr);
    s->take(1000);
    s->used(nullptr);
    void* q = s->take(1000);  // the first slot's turn again
    if (q == p) return 3;
    device = 99;
    return qsim::staging_slot() ? 4 : 0;
}
"""


def test_staging_slots(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2311_13081_gb300", "csrc"),
                    "-I", os.path.join(cuda, "include"), str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
