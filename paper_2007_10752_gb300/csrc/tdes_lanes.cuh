// tdes_lanes.cuh -- one block per thread with a copy of the S-box tables per
// lane: the scalar rounds of tdes_scalar.cuh ("Bit-level Parallelization of
// 3DES Encryption on GPU", Sec. III-B) without shared-memory bank conflicts.
//
// In tdes_small_kernel the 32 lanes of a warp look up random words of one
// 64-word table, 3.5 bank conflicts a lookup on average, and a 1 MiB call
// spends its 15 us on them: 27 warps an SM x 384 lookups x 3.5 cycles.  Here
// shared memory holds one copy of the S-box/permutation words per lane
// (64 KB), so a lookup takes one cycle; the word of S-box pair q (0..3),
// parity h and input x for lane l is at
//     q * 16384 + x * 256 + h * 128 + l * 4.
// The masked bytes of rotr(R, 27) (h = 0) and rotr(R, 23) (h = 1) are the
// inputs of the pairs, so one byte permute of (window word, lane offset) is a
// lookup's whole address (q and h sit in the load's immediate), and a round is
// 16 logic operations and 8 loads: two rotates, two XOR-and-masks with the key
// words (kernel parameters), eight permutes, four XORs.  IP and FP are bit
// swaps instead of table lookups.  Device time of one call, before and after
// (CUDA graph): 32768 blocks 6.2 -> 5.1 us, 65536 9.8 -> 6.2 us, 131072 15.0 -> 9.0 us, 196608
// 22.0 -> 12.7 us.
#pragma once
#include "tdes_internal.h"
#include "tdes_scalar.cuh"

namespace tdes {

constexpr int kLaneTableBytes = 4 * 64 * 256;

constexpr uint32_t kPairSbox = 0x35712460u;  // nibble 4h + q: the S-box of pair q, parity h
static_assert(TDES_SUBKEY_WORDS == 384, "48 rounds of 8 key bytes");

struct LaneKeys {  // 48 rounds x (ke, ko), by value
    uint32_t w[TDES_SUBKEY_WORDS / 4];
};

// Fills the tables: sp is the 8 x 64 words of TDES_SP_INIT.  Row i / 8 of the
// 16-byte stores is a (q, x, h); eight stores fill its 32 lanes' copies.
__device__ __forceinline__ void lane_tables(uint8_t* __restrict__ tab,
                                            const uint32_t* __restrict__ sp) {
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < 512 * 8; i += blockDim.x) {
        const uint32_t row = i >> 3, q = row >> 7, v = (row >> 1) & 63u, h = row & 1u;
        const uint32_t word = sp[((kPairSbox >> (16 * h + 4 * q)) & 7u) * 64 + v];
        reinterpret_cast<uint4*>(tab)[i] = make_uint4(word, word, word, word);
    }
}

__device__ __forceinline__ uint32_t lane_f(uint32_t R, uint32_t ke, uint32_t ko, uint32_t lane4,
                                           const uint8_t* __restrict__ tab) {
    const uint32_t m = 0x3F3F3F3Fu;
    const uint32_t we = (__funnelshift_r(R, R, 27) ^ ke) & m;
    const uint32_t wo = (__funnelshift_r(R, R, 23) ^ ko) & m;
    auto at = [&](uint32_t w, int q, int h) {
        // byte q of w above lane4's byte 0; bytes 2 and 3 zero
        const uint32_t off = __byte_perm(w, lane4, 0x5504 | (q << 4));
        return *reinterpret_cast<const uint32_t*>(tab + off + q * 16384 + h * 128);
    };
    const uint32_t a = at(we, 0, 0) ^ at(wo, 0, 1) ^ at(we, 1, 0);
    const uint32_t b = at(wo, 1, 1) ^ at(we, 2, 0) ^ at(wo, 2, 1);
    const uint32_t c = at(we, 3, 0) ^ at(wo, 3, 1);
    return a ^ b ^ c;
}

// One block (a 64-bit value with bit 1 at position 63) through ROUNDS rounds:
// keys holds the rounds' (ke, ko) words, lane4 the lane's offset 4 * lane.
template <int ROUNDS, class Keys>
__device__ __forceinline__ uint64_t lane_block(uint64_t x, const Keys& keys, uint32_t lane4,
                                               const uint8_t* __restrict__ tab) {
    uint32_t L = (uint32_t)(x >> 32), R = (uint32_t)x;
    swap_ip(L, R);
#pragma unroll
    for (int r = 0; r < ROUNDS; r += 2) {
        L ^= lane_f(R, keys[2 * r], keys[2 * r + 1], lane4, tab);
        R ^= lane_f(L, keys[2 * r + 2], keys[2 * r + 3], lane4, tab);
        if ((r & 15) == 14) {  // end of a DES pass: R16 || L16 continues as the next L0 || R0
            const uint32_t u = L;
            L = R;
            R = u;
        }
    }
    swap_fp(L, R);
    return ((uint64_t)L << 32) | R;
}

}  // namespace tdes
