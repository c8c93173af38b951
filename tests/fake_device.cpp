// Test-only: a stand-in for the CUDA runtime and the kernels, so that the host runtime (api.cpp) runs on the CPU.
// Device memory is host memory and copies happen at once.  The kernels do nothing, except that launch_finish moves
// every system on by a step (each solve ends after its max_iter steps) and the control words are gathered.
//
// Counted: copies whose source lies on the caller's stack and that no synchronisation has followed when a kernel
// is launched (the runtime may still read such a source), calls by name, and live device bytes.
#include <cuda_runtime.h>
#include <pthread.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include "symbolic.h"

using namespace asm2;

namespace {

std::mutex mu;
std::map<void*, size_t> live;
std::map<std::string, long long> calls;
size_t live_bytes = 0, h2d_bytes = 0;
int sms = 152, stack_copies = 0, late_stack_copies = 0;

void count(const char* name) {
    std::lock_guard<std::mutex> lk(mu);
    calls[name]++;
}
void kernel(const char* name) {
    count(name);
    late_stack_copies += stack_copies;
    stack_copies = 0;
}
bool on_stack(const void* p) {
    pthread_attr_t a;
    void* base = nullptr;
    size_t size = 0;
    pthread_getattr_np(pthread_self(), &a);
    pthread_attr_getstack(&a, &base, &size);
    pthread_attr_destroy(&a);
    return p >= base && p < static_cast<char*>(base) + size;
}

}  // namespace

extern "C" {

void fk_reset(int n_sms) {
    sms = n_sms;
    calls.clear();
    h2d_bytes = 0;
    stack_copies = late_stack_copies = 0;
}
long long fk_calls(const char* name) { return calls[name]; }
long long fk_live_bytes() { return (long long)live_bytes; }
long long fk_h2d_bytes() { return (long long)h2d_bytes; }
int fk_late_stack_copies() { return late_stack_copies; }

int asm_residual_noalloc(void*, const double*, const double*, double*, double*) { return 6; }

cudaError_t cudaMalloc(void** p, size_t n) {
    std::lock_guard<std::mutex> lk(mu);
    *p = std::calloc(1, n);
    live[*p] = n;
    live_bytes += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> lk(mu);
    live_bytes -= live[p];
    live.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return *p = std::calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    count("cudaMemcpyAsync");
    if (kind == cudaMemcpyHostToDevice) {
        h2d_bytes += n;
        if (on_stack(s)) stack_copies++;
    }
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return stack_copies = 0, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return stack_copies = 0, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)std::malloc(1), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free((void*)e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* a, size_t* b) { return *a = *b = (size_t)1 << 38, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 233472;
    return cudaSuccess;
}
}

namespace asm2 {

size_t apply_ring_bytes(int slots, int chunk) { return (size_t)slots * chunk + 128; }
size_t apply_smem_bytes(int nf, int nc, int prec, bool lump32) { return y_layout(nf, nc, prec, lump32).total; }
size_t apply_lump_bytes(int nf, int nc, bool mirror) { return y_layout(nf, nc, 0, false).fine * (mirror ? 2 : 1); }
ApplyConfig apply_local_vectors(int nsub, int all, int, int slots, int chunk, int sm_smem, int n_sms, int force, int) {
    const int fit = all > 0 ? std::min(2, sm_smem / (all + (int)apply_ring_bytes(slots, chunk) + 1024)) : 0;
    if (force == 0 && fit >= 1 && nsub <= fit * n_sms) return {Y_SMEM, all, slots, chunk};
    return {Y_DEVICE, 0, 2, chunk};
}
int ortho_coop_grid(int, int, int) { return 0; }
int noalloc_prepare(int) { return 0; }

void launch_finish(const SysTab* tab, const VecItem* items, int n, cudaStream_t) {
    kernel("finish");
    for (int i = 0; i < n; i++) {
        int* c = tab[items[i].sys].ctl;
        if (items[i].chunk != 0 || c[C_PHASE] == PH_DONE) continue;
        if (c[C_PHASE] == PH_INIT)
            c[C_PHASE] = PH_ARNOLDI;
        else if (++c[C_ITERS] >= c[C_MAXIT])
            c[C_PHASE] = PH_DONE, c[C_STATUS] = 0;
    }
}
void launch_gather_ctl(const SysTab* tab, int n, int* out, cudaStream_t) {
    kernel("gather_ctl");
    for (int k = 0; k < n; k++) std::memcpy(out + k * C_NCTL, tab[k].ctl, sizeof(int) * C_NCTL);
}
void launch_mgs(const SysTab*, const VecItem*, int, int, cudaStream_t) { kernel("mgs"); }
void launch_init(const SysTab*, const VecItem*, int, cudaStream_t) { kernel("init"); }
void launch_pack(const long long*, const int*, long long, int, unsigned char*, const double*, cudaStream_t) { kernel("pack"); }
void launch_pack_lanes(const long long*, const int*, long long, int, unsigned char*, const double*, cudaStream_t) {
    kernel("pack_lanes");
}
void launch_place(const PkPiece* p, int n, const void* src, void* dst, cudaStream_t) {
    kernel("place");
    for (int i = 0; i < n; i++)
        std::memcpy(static_cast<char*>(dst) + 16LL * p[i].dst, static_cast<const char*>(src) + 16LL * p[i].src, 16LL * p[i].n);
}
void launch_post(const SysTab*, const VecItem*, int, cudaStream_t) { kernel("post"); }
void launch_prep(const SysTab*, const VecItem*, int, cudaStream_t) { kernel("prep"); }
void launch_spmv(const SysTab*, const RowItem*, int, cudaStream_t) { kernel("spmv"); }
void launch_apply(const SysTab*, const SubDesc*, int, int, bool, ApplyConfig cfg, cudaStream_t) {
    kernel(cfg.ymode == Y_PACKET ? "apply_lanes" : "apply_rows");
}
void launch_boxsum(const SysTab*, const BoxItem*, int, int, cudaStream_t) { kernel("boxsum"); }
void launch_coarse(const int*, const int*, const double*, double*, int, cudaStream_t) { kernel("coarse"); }
void launch_factor(const FactDesc*, int, int, FactErr*, const int*, cudaStream_t) { kernel("factor"); }
void launch_assemble(const int*, const int*, const int*, const double*, const double*, double*, long long, cudaStream_t,
                     const int*, int) {
    kernel("assemble");
}
void launch_ell_fill(const double*, const int*, int, int, double*, int, cudaStream_t) { kernel("ell_fill"); }
void launch_restrict(const SysTab*, const SubDesc*, const int2*, int, int, bool, cudaStream_t) { kernel("restrict"); }
void launch_coarse_apply(const SysTab*, const RowItem*, int, const BoxItem*, int, const RowItem*, int, const VecItem*, int,
                         bool, cudaStream_t) {}

}  // namespace asm2
