// The library's host code (m1_api.cu) on a stand-in of the CUDA runtime that keeps
// "device" memory on the host and runs no kernel: what a step answers when the launch of
// the coarse levels is refused while a cycle is recorded.  Arguments: precision (0, 1)
// and how many of the first launches are refused; prints the status of three steps, how many
// graphs were made and how many of these launches were taken.  (tests/test_refused_launch.py builds and runs it.)
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "m1_api.cu"

static cudaError_t g_last = cudaSuccess;
static int g_refuse = 0, g_graphs = 0, g_taken = 0;

#ifndef __CUDA_ARCH__
extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)&g_last; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)&g_graphs; return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long)
{
    *x = (cudaGraphExec_t)&g_graphs;
    ++g_graphs;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)&g_last; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)&g_last; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}
#endif

namespace m1 {
#define NOOP(name, ...) template <typename R> void name(__VA_ARGS__) {}
NOOP(launch_sweep, const Level<R>*, WorkList, Ctl*, bool, int, int, cudaStream_t, bool, bool, double*, bool, int)
NOOP(launch_apply, const Level<R>*, WorkList, Ctl*, int, int, double*, int, cudaStream_t, bool)
NOOP(launch_norm_state, const Level<R>*, WorkList, const Ctl*, double*, cudaStream_t)
NOOP(launch_restrict, const Level<R>*, const Level<R>*, WorkList, Ctl*, int, cudaStream_t, bool)
NOOP(launch_restrict_sig, const Level<R>*, const Level<R>*, WorkList, cudaStream_t)
NOOP(launch_prolong, const Level<R>*, const Level<R>*, WorkList, Ctl*, int, int, cudaStream_t, bool)
NOOP(launch_make_rhs, const Level<R>*, WorkList, const Ctl*, int, cudaStream_t)
NOOP(launch_finalize, Ctl*, const Level<R>*, int, const double*, const double*, int, int, BatchCtl*, cudaStream_t, const int*)
NOOP(launch_pack_state, const double*, const double*, const double*, const double*, double, Cell4<R>*, int, cudaStream_t)
NOOP(launch_pack_sig, const double*, const double*, Sig2<R>*, int, cudaStream_t)
NOOP(launch_check_state, const Cell4<R>*, const Sig2<R>*, int, double, unsigned int*, cudaStream_t)
void launch_coef64(const Level<double>*, WorkList, cudaStream_t) {}
void launch_fas_aw32(const Level<float>*, WorkList, Ctl*, cudaStream_t) {}
void launch_defect(const Level<double>*, const Level<float>*, WorkList, Ctl*, double*, cudaStream_t, bool) {}
void launch_defect_dw(const Level<double>*, const Level<float>*, const DwLevel*, WorkList, Ctl*, double*, cudaStream_t, bool) {}
void launch_dw_split(const Level<double>*, const DwLevel*, WorkList, cudaStream_t) {}
void launch_accumulate(const Level<double>*, const Level<float>*, WorkList, Ctl*, int, cudaStream_t, const DwLevel*) {}
int strip_rows(int, int, int) { return 1; }
int strip_ring(int, int) { return 0; }
size_t tail_smem(int, int, int, int) { return 0; }
size_t tail32_smem(int, int, int, int) { return 0; }
cudaError_t tail_prepare() { return cudaSuccess; }
cudaError_t tail32_prepare() { return cudaSuccess; }
static cudaError_t tail_answer()
{
    if (g_refuse <= 0) return ++g_taken, cudaSuccess;
    --g_refuse;
    return g_last = cudaErrorInvalidConfiguration;
}
cudaError_t launch_tail(const Level<double>*, int, int, WorkList, Ctl*, const unsigned char*, const int2*,
                        size_t, int, cudaStream_t)
{
    return tail_answer();
}
cudaError_t launch_tail32(const Level<float>*, int, int, WorkList, Ctl*, const unsigned char*, const int2*,
                          unsigned, size_t, int, cudaStream_t)
{
    return tail_answer();
}
}  // namespace m1

int main(int argc, char** argv)
{
    if (argc < 3) return 2;
    g_refuse = std::atoi(argv[2]);
    m1_grid_desc d = {};
    d.dim = 2; d.nx = d.ny = 16; d.lx = d.ly = 1.0; d.lmax = 3; d.c = d.a_r = d.c_v = 1.0;
    d.precision = std::atoi(argv[1]);
    m1_grid_t g = nullptr;
    if (m1_create_grid(&d, nullptr, &g) != M1_OK) return 3;
    std::vector<double> one(256, 1.0), zero(256, 0.0);
    if (m1_set_state(g, one.data(), zero.data(), zero.data(), one.data(), one.data(), one.data(), 0) != M1_OK)
        return 4;
    m1_solve_params p;
    m1_default_params(&p);
    p.max_cycles = 3;
    for (int k = 0; k < 3; ++k) std::printf("%d ", (int)m1_implicit_step(g, 1.0, &p, nullptr));
    std::printf("%d %d\n", g_graphs, g_taken);
    return 0;
}
