// The library's host code of a single-key call on a stand-in for the CUDA
// runtime (test infrastructure only): device memory is host memory, no kernel
// runs, and what the calls pass to the runtime is looked at.  Built together
// with tdes_api.cu and tdes_small.cu; the launchers of the other kernels are
// stubs here.
//
// Usage: tdes_fake_runtime <case>; 0: as it should be, 1: not so (says why).
//   free      tdes_key_free clears the schedule's round keys before it frees them
//   launch    ... as does a key schedule whose kernel cannot be launched
//   sync      ... or whose stream reports an error
//   params    a per-lane-table call hands the runtime the schedule's own round
//             keys as the kernel's parameters (no copy is left on a stack)
//   copies    a key schedule copies nothing back from the device
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "../../include/tdes.h"
#include "../../paper_2007_10752_gb300/csrc/tdes_internal.h"
#include "../../paper_2007_10752_gb300/csrc/tdes_keysched.cuh"

static const uint8_t kSub[2][48][48] = TDES_SUBKEY_INIT;
static void* g_schedule = nullptr;  // the last tdes_ks allocated, and the state of its
static int g_cleared = -1;          // round keys when it was freed: 1 all zero, 0 not
static cudaError_t g_launch = cudaSuccess, g_sync = cudaSuccess;
static int g_copies_back = 0;
static const void* g_param0 = nullptr;  // the first parameter of the last kernel launched

// ------------------------------------------------------------- allocation
void* operator new(size_t n, const std::nothrow_t&) noexcept {
    void* p = malloc(n);
    if (p) memset(p, 0xA5, n);
    if (n == sizeof(tdes_ks)) g_schedule = p;
    return p;
}
static void check_freed(void* p) {
    if (p == nullptr || p != g_schedule) return;
    g_cleared = 1;
    const uint8_t* b = static_cast<const uint8_t*>(p) + offsetof(tdes_ks, host_chunk);
    for (size_t i = 0; i < sizeof(tdes_ks::host_chunk); ++i)
        if (b[i]) g_cleared = 0;
}
void operator delete(void* p) noexcept { check_freed(p); free(p); }
void operator delete(void* p, size_t) noexcept { check_freed(p); free(p); }

// ---------------------------------------------------------------- runtime
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*,
                            dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void** args, size_t, cudaStream_t) {
    g_param0 = args[0];
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void** args, size_t, cudaStream_t) {
    g_param0 = args[0];
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void** args) {
    g_param0 = args[0];
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind kind, cudaStream_t) {
    g_copies_back += kind == cudaMemcpyDeviceToHost;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    memset(a, 0, sizeof *a);
    a->type = cudaMemoryTypeDevice;
    a->devicePointer = const_cast<void*>(p);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return g_sync; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
}

// ------------------------------------------------ the other files' launchers
namespace tdes {
cudaError_t launch_keysched(const Keys24& keys, int, uint32_t*, uint32_t*, uint8_t* enc, uint8_t* dec,
                            cudaStream_t) {
    for (int i = 0; i < 2 * TDES_SUBKEY_WORDS; ++i) {  // as the kernel does
        const int dir = i / TDES_SUBKEY_WORDS, c = i % TDES_SUBKEY_WORDS;
        (dir ? dec : enc)[c] = tdes_subkey_chunk(keys.b, &kSub[dir][c / 8][6 * (c % 8)]);
    }
    return g_launch;
}
cudaError_t launch_ecb(const uint32_t*, const uint8_t*, int, const void*, void*, uint64_t, bool,
                       Geometry, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_ctr(const uint32_t*, const uint8_t*, int, uint32_t, uint32_t, const void*, void*,
                       uint64_t, bool, Geometry, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_cbc_halo(const void*, uint64_t*, uint64_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_cbc_dec(const uint32_t*, const uint8_t*, int, uint64_t, const void*, void*, uint64_t,
                           const uint64_t*, bool, Geometry, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_cbc_enc(const uint8_t*, int, uint64_t, const void*, void*, uint64_t,
                           cudaStream_t) { return cudaSuccess; }
int wide_ctas_per_sm(int) { return 2; }
int sbox_gate_count() { return 0; }
}  // namespace tdes

// ------------------------------------------------------------------ cases
static int no(const char* why) {
    fprintf(stderr, "%s\n", why);
    return 1;
}

int main(int argc, char** argv) {
    if (argc < 2) return 2;
    uint8_t k[3][8];
    for (int i = 0; i < 24; ++i) k[i / 8][i % 8] = (uint8_t)(37 * i + 11);
    const bool bad_launch = !strcmp(argv[1], "launch"), bad_sync = !strcmp(argv[1], "sync");
    if (bad_launch) g_launch = cudaErrorUnknown;
    if (bad_sync) g_sync = cudaErrorUnknown;
    tdes_ks_t* ks = nullptr;
    const int rc = tdes_key_schedule(k[0], k[1], k[2], &ks);
    if (bad_launch || bad_sync) {
        if (rc != TDES_ECUDA || ks != nullptr) return no("the error was not reported");
        return g_cleared == 1 ? 0 : no("round keys left in freed memory");
    }
    if (rc != TDES_OK) return no("key schedule");
    uint8_t want[2][TDES_SUBKEY_WORDS];
    for (int dir = 0; dir < 2; ++dir)
        for (int c = 0; c < TDES_SUBKEY_WORDS; ++c)
            want[dir][c] = tdes_subkey_chunk(&k[0][0], &kSub[dir][c / 8][6 * (c % 8)]);
    if (memcmp(ks->host_chunk, want, sizeof want)) return no("the host's round keys are wrong");
    if (!strcmp(argv[1], "copies") && g_copies_back) return no("copied from the device");
    if (!strcmp(argv[1], "params")) {
        const size_t n = 8 * 40000;
        void* buf = aligned_alloc(16, n);
        for (int dir = 0; dir < 2; ++dir) {
            g_param0 = nullptr;
            if ((dir ? tdes_ecb_decrypt : tdes_ecb_encrypt)(ks, buf, buf, n, nullptr) != TDES_OK)
                return no("call");
            if (g_param0 != ks->host_chunk[dir]) return no("the round keys were copied for the launch");
        }
    }
    tdes_key_free(ks);
    return g_cleared == 1 ? 0 : no("round keys left in freed memory");
}
