// common.cu -- error reporting, launch counts and kernel marks.
#include <stdio.h>

#include "common.cuh"

namespace gb3 {

// set by the C-ABI layer to record the message of the last CUDA failure
thread_local char g_cuda_msg[256];

int cuda_fail(cudaError_t e, const char* what, const char* file, int line) {
    snprintf(g_cuda_msg, sizeof g_cuda_msg, "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
    if (e == cudaErrorMemoryAllocation) return FMM_E_OOM;
    return FMM_E_CUDA;
}

// SM count per device, queried on first use (0 = not yet known)
static int g_sm_count[64] = {0};
int sm_count() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 148;  // a query that fails only sizes grid-stride loops
    }
    int n = __atomic_load_n(&g_sm_count[dev], __ATOMIC_RELAXED);
    if (n <= 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            return 148;
        }
        __atomic_store_n(&g_sm_count[dev], n, __ATOMIC_RELAXED);
    }
    return n;
}

thread_local long long g_launches = 0;
void note_launch() { ++g_launches; }
long long launches_so_far() { return g_launches; }

thread_local cudaEvent_t* g_marks = nullptr;
thread_local int g_marks_hit = 0;
void kernel_marks(cudaEvent_t* ev) {
    g_marks = ev;
    g_marks_hit = 0;
}
void mark_begin(cudaStream_t s) {
    if (g_marks && cudaEventRecord(g_marks[0], s) == cudaSuccess) g_marks_hit |= 1;
}
void mark_end(cudaStream_t s) {
    if (g_marks && cudaEventRecord(g_marks[1], s) == cudaSuccess) g_marks_hit |= 2;
}
bool marks_recorded() { return g_marks_hit == 3; }

}  // namespace gb3
