// tdes_internal.h -- launchers shared by the C ABI (tdes_api.cu) and the
// kernels (tdes_kernels.cu).  Not part of the public interface.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

// The library's key-schedule object (opaque tdes_ks_t in include/tdes.h).
struct tdes_ks {
    int device;
    int stages;             // DES passes per block: 3 (EDE3) or 1 (single DES)
    void* mem;              // one cudaMalloc holding everything below
    uint32_t* tab[2];       // bitsliced round-constant tables: [0] encrypt, [1] decrypt
    uint8_t* chunk[2];      // scalar-path round-key groups: [0] encrypt, [1] decrypt
    uint8_t host_chunk[2][384];  // host copies of the groups (kernel parameters); wipe() before freeing
};

namespace tdes {

// Records the message tdes_last_error() returns on this host thread.
void set_last_error(const char* msg);

// Clears key material.  The compiler may drop a plain memset of memory that is
// freed or left next; it has to keep this one.
inline void wipe(void* p, size_t n) {
    memset(p, 0, n);
    asm volatile("" : : "r"(p) : "memory");
}

// True if the GPU can address `p` with the same pointer: device or managed
// memory, or page-locked host memory mapped into the device address space
// (what cudaHostAlloc gives on a unified-address system).  Pageable host
// memory is refused: a kernel access to it could fault.  Sets *host (where
// given) for host memory and leaves it alone otherwise.
bool gpu_addressable(const void* p, bool* host = nullptr);
// True for page-locked host memory (whether or not it is mapped).
bool host_memory(const void* p);

// Launches a kernel; overlap: it may start while the kernel before it on the
// stream still runs (programmatic dependent launch), if that one allows it
// (launch_dependents).  A single-key call's kernel stages its tables, then waits
// for the one before to complete (wait_for_primary) before it reads or writes
// any data, so back-to-back calls overlap one's start with the other's end: 4
// blocks 6.1 -> 4.4 us a call, 9 MB ECB 28.7 -> 25.8, 40 MB CTR 96.3 -> 92.4,
// 200 MB CBC decryption 481 -> 477.
template <class Kernel, class... Args>
inline cudaError_t launch_kernel(Kernel* kernel, unsigned grid, unsigned threads, size_t smem,
                                 cudaStream_t s, bool overlap, Args... args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = threads;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess) cudaGetLastError();  // reported by the caller, not left for the next check
    return e;
}

#ifdef __CUDACC__
// Programmatic dependent launch: lets the next kernel of the stream start once
// every CTA of this grid has said so or has ended; and waits for the grid
// before this one to complete (at once after an ordinary launch).
__device__ __forceinline__ void launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_primary() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

constexpr int kTileBlocks = 1024;  // blocks per warp tile: 32 lanes x 32 blocks
constexpr int kWideWarps = 8;      // warps per CTA for large inputs
// A call of so many tiles (512 MiB, 1.2 ms) neither starts beside the kernel before
// nor lets the next start beside it: the next one's CTAs, waiting, take every place
// that its own leave.  Beside a row of 1 GiB calls, a small call on another stream
// waited for a whole kernel each time (2.4 ms, the first 3.3); so it waits until the
// kernel's first CTAs end (after 1.3 ms), and from then on 0.05 to 0.1 ms.  The row
// takes 3 to 9 us a call longer (ECB 2441 -> 2445).
constexpr uint32_t kOverlapTiles = 1u << 16;
constexpr int kTableWords = 3328;  // words of one bitsliced round-constant table
constexpr int kChunkBytes = 384;   // 48 rounds x 8 six-bit round-key groups

struct Keys24 {
    uint8_t b[24];
};

// Launch geometry for `ntiles` warp tiles on the current device.
struct Geometry {
    int grid;
    int threads;
    int sms;
    bool overlap;  // launch_kernel
};

// The blocks of a call that run one per thread after the kernel's tiles: n of
// them, right after the tiles' blocks; keys is the call's scalar round-key
// groups on the device.
struct Tail {
    const uint32_t* keys;
    uint32_t n;
};
Geometry geometry_for(uint64_t ntiles, int kernel_id, int device);

enum KernelId { kEcb = 0, kCtr = 1, kCbcDec = 2, kNumKernels = 3 };

// `stages` (1 or 3) selects the single-DES or the EDE3 kernels; the tables
// passed must have been built for the same number of stages.  chunks: the
// scalar round-key groups of the same key and direction, on the device.
cudaError_t launch_keysched(const Keys24& keys, int stages, uint32_t* tab_enc, uint32_t* tab_dec,
                            uint8_t* chunk_enc, uint8_t* chunk_dec, cudaStream_t s);
cudaError_t launch_ecb(const uint32_t* tab, const uint8_t* chunks, int stages, const void* in,
                       void* out, uint64_t nblocks, bool vec16, Geometry g, cudaStream_t s);
cudaError_t launch_ctr(const uint32_t* tab_enc, const uint8_t* chunks, int stages, uint32_t nonce,
                       uint32_t ctr0, const void* in, void* out, uint64_t nblocks, bool vec16,
                       Geometry g, cudaStream_t s);
cudaError_t launch_cbc_halo(const void* in, uint64_t* halo, uint64_t nblocks, cudaStream_t s);
cudaError_t launch_cbc_dec(const uint32_t* tab_dec, const uint8_t* chunks, int stages, uint64_t iv,
                           const void* in, void* out, uint64_t nblocks, const uint64_t* halo,
                           bool vec16, Geometry g, cudaStream_t s);
cudaError_t launch_cbc_enc(const uint8_t* chunk_enc, int stages, uint64_t iv, const void* in,
                           void* out, uint64_t nblocks, cudaStream_t s);

// One block per thread (tdes_small.cu), for calls too small to fill the GPU
// with bitsliced tiles.  keys: the call's scalar round-key groups of the
// wanted direction, on the device and on the host; iv: the CBC IV, or nonce << 32 | ctr0 for CTR.
constexpr int kSmallThreads = 128;  // per CTA: spreads a small call over many SMs
enum SmallMode { kSmallEcb = 0, kSmallCtr = 1, kSmallCbcDec = 2 };
struct SmallKeys {
    const uint8_t* dev;
    const uint8_t* host;
};
inline SmallKeys small_keys(const tdes_ks* ks, int dir) {
    return {ks->chunk[dir], ks->host_chunk[dir]};
}
cudaError_t launch_small(SmallKeys keys, int stages, int mode, uint64_t iv, const void* in,
                         void* out, uint64_t nblocks, int threads, cudaStream_t s);

// Occupancy (CTAs per SM) of a bitsliced kernel at kWideWarps warps per CTA.
int wide_ctas_per_sm(int kernel_id);
int sbox_gate_count();

}  // namespace tdes
