// tdes_small.cu -- single-key calls too small to fill the GPU with bitsliced
// tiles: one 64-bit block per thread, in two kernels: tdes_small_kernel (one
// copy of the tables per CTA) and, from 28673 blocks, tdes_lanes_kernel (one
// copy per lane, no bank conflicts).
//
// A bitsliced tile is 1024 blocks and costs each lane about 12 k logic
// operations (48 rounds over 64 bit-planes), so a call of a few tiles takes
// one tile's latency however few blocks it holds.  Here each thread runs its
// own block through the scalar round (tdes_block_scalar_swap: the expansion
// windows as two rotates, eight S-box/permutation table lookups, IP and FP as
// bit swaps), a chain of 48 dependent rounds (16 for single DES).
// The table and the call's round-key words are staged in shared memory once
// per CTA: 2.4 KB, where nibble tables for IP and FP made it 6.4 KB (a call of
// 64 blocks 4.04 -> 3.52 us, of 24576 6.14 -> 5.48 us, device time).
#include <cuda_runtime.h>

#include <atomic>

#include "tdes_internal.h"
#include "tdes_keysched.cuh"
#include "tdes_lanes.cuh"
#include "tdes_scalar.cuh"

namespace tdes {

__device__ const __align__(16) uint32_t kSmallSP[8][64] = TDES_SP_INIT;

struct SmallTables {
    uint32_t sp[8 * 64];
    uint32_t keys[TDES_SUBKEY_WORDS / 4];
};

__device__ __forceinline__ uint64_t small_load_be(const uint8_t* p, uint64_t i) {
    return bswap64(reinterpret_cast<const uint64_t*>(p)[i]);
}

// mode: kSmallEcb (chunks of the direction wanted), kSmallCtr (block i is
// E(nonce || ctr0 + i) XOR in_i; iv = nonce << 32 | ctr0), kSmallCbcDec
// (D(in_i) XOR in_{i-1}, in_{-1} = iv).  In place is safe for ECB and CTR
// (each thread reads and writes only its own block); for CBC decryption the
// host uses this kernel in place only with a single CTA, whose threads all
// read before any writes.
// SPREAD: only the first kSmallThreads threads of a CTA take a block (launch_small).
template <int ROUNDS, bool SPREAD>
__global__ void __launch_bounds__(1024)
tdes_small_kernel(const uint8_t* __restrict__ chunks, int mode, uint64_t iv, const uint8_t* in,
                  uint8_t* out, uint64_t nblocks) {
    __shared__ __align__(16) SmallTables st;
    launch_dependents();
    for (int i = threadIdx.x; i < 8 * 64 / 4; i += blockDim.x)
        reinterpret_cast<uint4*>(st.sp)[i] = __ldg(reinterpret_cast<const uint4*>(&kSmallSP[0][0]) + i);
    for (int i = threadIdx.x; i < TDES_SUBKEY_WORDS / 4; i += blockDim.x)
        st.keys[i] = __ldg(reinterpret_cast<const uint32_t*>(chunks) + i);
    wait_for_primary();
    uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (SPREAD)
        b = threadIdx.x < kSmallThreads ? (uint64_t)blockIdx.x * kSmallThreads + threadIdx.x : nblocks;
    uint64_t x = 0, prev = 0;
    if (b < nblocks) {
        if (mode == kSmallCtr) {
            x = (iv & 0xFFFFFFFF00000000ull) | (uint32_t)((uint32_t)iv + (uint32_t)b);
            prev = small_load_be(in, b);
        } else {
            x = small_load_be(in, b);
            if (mode == kSmallCbcDec) prev = b ? small_load_be(in, b - 1) : iv;
        }
    }
    __syncthreads();  // tables staged; every read of this CTA precedes its writes
    if (b < nblocks) {
        uint64_t y = tdes_block_scalar_swap<ROUNDS>(x, st.sp, st.keys);
        if (mode != kSmallEcb) y ^= prev;
        reinterpret_cast<uint64_t*>(out)[b] = bswap64(y);
    }
}

// ---- one block per thread, a copy of the tables per lane (tdes_lanes.cuh) ----
constexpr uint64_t kLanesMinBlocks = 28672;
// Calls of so few CTAs of tdes_small_kernel may start beside the kernel before
// (launch_kernel).  Where that one fills the GPU they find their places as its
// first CTAs end, and all 16 together on one SM took 13 us instead of 3.5.  Two or more
// therefore get 512 threads, of which those past the CTA's blocks only help to stage
// the table, so that an SM has room for two to four: 1100 tiles after 2048 blocks,
// again and again, 55 -> 31.9 us (both waiting for the call before: 39.3; with 256
// threads 36.5).  Shared memory asked for instead did the same, but a CTA of 48 KB
// waits for an idle SM, beside a 1 GiB call for that call's end.
constexpr uint64_t kOverlapCtas = 16;
constexpr int kOverlapThreads = 512;

template <int ROUNDS>
__global__ void __launch_bounds__(512, 3)
tdes_lanes_kernel(const __grid_constant__ LaneKeys keys, int mode, uint64_t iv, const uint8_t* in,
                  uint8_t* out, uint32_t nblocks) {
    extern __shared__ __align__(16) uint8_t lane_tab[];
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane4 = (threadIdx.x & 31u) * 4u;
    uint64_t x = 0, prev = 0;
    if (b < nblocks) {
        if (mode == kSmallCtr) {
            x = (iv & 0xFFFFFFFF00000000ull) | (uint32_t)((uint32_t)iv + b);
            prev = small_load_be(in, b);
        } else {
            x = small_load_be(in, b);
            if (mode == kSmallCbcDec) prev = b ? small_load_be(in, b - 1) : iv;
        }
    }
    lane_tables(lane_tab, &kSmallSP[0][0]);  // while the data is on its way
    __syncthreads();
    if (b >= nblocks) return;
    uint64_t y = lane_block<ROUNDS>(x, keys.w, lane4, lane_tab);
    if (mode != kSmallEcb) y ^= prev;
    reinterpret_cast<uint64_t*>(out)[b] = bswap64(y);
}

// Whether a call takes tdes_lanes_kernel.  Below kLanesMinBlocks the few warps
// an SM has do not fill its shared memory's cycles and writing 64 KB of tables
// costs more than the conflicts (16384 blocks: 6.8 us against 4.3 us of
// tdes_small_kernel; 24576: 6.2 against 5.5; 32768: 5.1 against over 6).  CBC
// decryption only out of place: its CTAs write while others still read.
static bool use_lanes(int mode, const void* in, const void* out, uint64_t nblocks) {
    return nblocks > kLanesMinBlocks && nblocks <= (1ull << 30) &&
           (mode != kSmallCbcDec || in != out);
}

template <int ROUNDS>
static cudaError_t lanes_launch(const uint8_t* host_chunks, int mode, uint64_t iv, const void* in,
                                void* out, uint32_t nblocks, cudaStream_t s) {
    static std::atomic<uint64_t> ready{0};  // devices whose shared-memory limit is raised
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(ready.load() >> dev & 1u)) {
        e = cudaFuncSetAttribute(tdes_lanes_kernel<ROUNDS>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kLaneTableBytes);
        if (e != cudaSuccess) return e;
        if (dev < 64) ready.fetch_or(1ull << dev);
    }
    // CTAs of one size, as few per SM (1 to 3) as hold the call in 512 threads
    // each: every SM gets the same share, and fewer copies of the tables to write.
    const uint32_t per_sm = nblocks <= (uint32_t)sms * 512u ? 1u : nblocks <= (uint32_t)sms * 1024u ? 2u : 3u;
    const uint32_t ctas = (uint32_t)sms * per_sm;
    uint32_t threads = ((nblocks + ctas - 1) / ctas + 31u) / 32u * 32u;
    threads = threads > 512u ? 512u : threads;
    // The round keys go to the runtime from where the schedule holds them: an
    // argument by value would leave copies on the stack.
    static_assert(sizeof(LaneKeys) == sizeof(tdes_ks::host_chunk[0]), "the schedule's round keys");
    const uint8_t* src = static_cast<const uint8_t*>(in);
    uint8_t* dst = static_cast<uint8_t*>(out);
    void* args[] = {const_cast<uint8_t*>(host_chunks), &mode, &iv, &src, &dst, &nblocks};
    // Not started beside the kernel before: the free places it would take are
    // spread unevenly over the SMs (two calls of 1 MiB 20.5 -> 21.7 us).
    e = cudaLaunchKernel((const void*)tdes_lanes_kernel<ROUNDS>, (nblocks + threads - 1) / threads, threads,
                         args, kLaneTableBytes, s);
    if (e != cudaSuccess) cudaGetLastError();  // as launch_kernel
    return e;
}

cudaError_t launch_small(SmallKeys keys, int stages, int mode, uint64_t iv, const void* in,
                         void* out, uint64_t nblocks, int threads, cudaStream_t s) {
    if (use_lanes(mode, in, out, nblocks))
        return stages == 1
                   ? lanes_launch<16>(keys.host, mode, iv, in, out, (uint32_t)nblocks, s)
                   : lanes_launch<48>(keys.host, mode, iv, in, out, (uint32_t)nblocks, s);
    const uint64_t grid = (nblocks + threads - 1) / threads;
    auto launch = [&](auto kernel, unsigned cta) {
        return launch_kernel(kernel, (unsigned)grid, cta, 0, s, grid <= kOverlapCtas, keys.dev, mode, iv,
                             static_cast<const uint8_t*>(in), static_cast<uint8_t*>(out), nblocks);
    };
    if (threads == kSmallThreads && grid > 1 && grid <= kOverlapCtas)
        return launch(stages == 1 ? tdes_small_kernel<16, true> : tdes_small_kernel<48, true>,
                      kOverlapThreads);
    return launch(stages == 1 ? tdes_small_kernel<16, false> : tdes_small_kernel<48, false>,
                  (unsigned)threads);
}

}  // namespace tdes
