// tdes_scalar.cuh -- one-block-at-a-time 3DES paths: the scalar round (one
// block per thread; small calls, small batch messages, short CBC chains) and
// the warp-cooperative round (one serial CBC-encryption chain per warp).
//
// Both compute the same EDE3 block as the bitsliced core of
// tdes_bitslice.cuh ("Bit-level Parallelization of 3DES Encryption on GPU",
// Sec. III-B), one 64-bit block at a time, with the expansion windows read
// out of rotated halves and the S-boxes and permutation as lookups.  ROUNDS
// is 48 (EDE3) or 16 (single DES, on the first 16 rounds' key words).
#pragma once
#include "tdes_bitslice.cuh"
#include "generated/tdes_generated_scalar.cuh"

// ---------------------------------------------------------------- scalar path
// One block at a time (serial CBC encryption).  A block is a 64-bit value
// with bit 1 at position 63 (big-endian bytes); a half has bit 1 at 31.

TDES_HD uint32_t rotr32(uint32_t x, int n) { return (x >> n) | (x << ((32 - n) & 31)); }

TDES_HD uint64_t permute64(uint64_t v, const uint8_t* __restrict__ src) {
    uint64_t r = 0;
    for (int j = 0; j < 64; ++j) r |= ((v >> (63 - src[j])) & 1ull) << (63 - j);
    return r;
}

// One Feistel round of the scalar path.  The expansion windows of S-boxes
// 1, 7, 5, 3 are the four bytes of rotr(R, 27) and those of S-boxes 2, 8, 6, 4
// the four bytes of rotr(R, 23) (six bits each, first bit most significant),
// so two rotates and two XORs with the round's key words ke/ko form all eight
// S-box inputs; sp[64g + x] is S-box g followed by the permutation.  Each
// six-bit index is extracted already scaled by 4 (a byte offset into sp).
TDES_HD uint32_t sp_at(const uint32_t* __restrict__ sp, int g, uint32_t byte_off) {
    return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(sp + 64 * g) +
                                               byte_off);
}

TDES_HD uint32_t tdes_f_scalar(uint32_t R, uint32_t ke, uint32_t ko,
                               const uint32_t* __restrict__ sp) {
    const uint32_t we = rotr32(R, 27) ^ ke;
    const uint32_t wo = rotr32(R, 23) ^ ko;
    const uint32_t a = sp_at(sp, 0, (we << 2) & 0xFCu) ^ sp_at(sp, 6, (we >> 6) & 0xFCu) ^
                       sp_at(sp, 4, (we >> 14) & 0xFCu);
    const uint32_t b = sp_at(sp, 2, (we >> 22) & 0xFCu) ^ sp_at(sp, 1, (wo << 2) & 0xFCu) ^
                       sp_at(sp, 7, (wo >> 6) & 0xFCu);
    const uint32_t c = sp_at(sp, 5, (wo >> 14) & 0xFCu) ^ sp_at(sp, 3, (wo >> 22) & 0xFCu);
    return a ^ b ^ c;
}

// sp: 8 x 64 S-box/permutation words; keys: 48 rounds x (ke, ko) words (the
// round-key groups in the byte order of the expansion windows); ip/fp: the
// permutations as 0-based source bits.
TDES_HD uint64_t tdes_block_scalar(uint64_t v, const uint32_t* __restrict__ sp,
                                   const uint32_t* __restrict__ keys,
                                   const uint8_t* __restrict__ ip, const uint8_t* __restrict__ fp) {
    v = permute64(v, ip);
    uint32_t L = (uint32_t)(v >> 32), R = (uint32_t)v;
    for (int r = 0; r < 48; ++r) {
        const uint32_t t = L ^ tdes_f_scalar(R, keys[2 * r], keys[2 * r + 1], sp);
        L = R;
        R = t;
        if ((r & 15) == 15) {  // end of a DES pass: undo the last swap (R16 || L16)
            const uint32_t u = L;
            L = R;
            R = u;
        }
    }
    return permute64(((uint64_t)L << 32) | R, fp);
}

// Permutation of a 64-bit block by 16 nibble tables (tab[n][v]: the output
// bits contributed by value v in input nibble n); 16 independent lookups.
TDES_HD uint64_t permute64_nib(uint64_t v, const uint64_t* __restrict__ tab) {
    uint64_t r = 0;
#pragma unroll
    for (int n = 0; n < 16; ++n) r |= tab[16 * n + (uint32_t)((v >> (60 - 4 * n)) & 15u)];
    return r;
}

// The same EDE3 block as tdes_block_scalar with the permutations by nibble
// tables (ipn/fpn: 16 x 16 words each) instead of bit loops: a form of the host
// check alone, which no kernel takes (they take tdes_block_scalar_swap).  The 16
// rounds of a DES pass are unrolled by two so that the halves alternate in place,
// and each round's key words are loaded one round ahead, off the chain of
// dependent operations that sets the latency of a block.
template <int ROUNDS = 48>
TDES_HD uint64_t tdes_block_scalar_nib(uint64_t v, const uint32_t* __restrict__ sp,
                                       const uint32_t* __restrict__ keys,
                                       const uint64_t* __restrict__ ipn,
                                       const uint64_t* __restrict__ fpn) {
    constexpr int rounds = ROUNDS;
    v = permute64_nib(v, ipn);
    uint32_t L = (uint32_t)(v >> 32), R = (uint32_t)v;
    uint32_t ke = keys[0], ko = keys[1];
#pragma unroll
    for (int r = 0; r < rounds; r += 2) {
        const uint32_t ke1 = keys[2 * r + 2], ko1 = keys[2 * r + 3];
        L ^= tdes_f_scalar(R, ke, ko, sp);
        const int rn = r + 2 < rounds ? r + 2 : r;  // the last prefetch rereads the last pair
        ke = keys[2 * rn];
        ko = keys[2 * rn + 1];
        R ^= tdes_f_scalar(L, ke1, ko1, sp);
        if ((r & 15) == 14) {  // end of a DES pass: R16 || L16 continues as the next L0 || R0
            const uint32_t u = L;
            L = R;
            R = u;
        }
    }
    return permute64_nib(((uint64_t)L << 32) | R, fpn);
}

// IP and FP as swaps of bit groups between the halves: IP is a transpose of
// the block's 8x8 bit matrix followed by a row reordering, and each of its
// five steps exchanges one index bit (the masked exchanges of Warren, "Hacker's
// Delight", Sec. 7-3).
TDES_HD void bit_swap(uint32_t& a, uint32_t& b, int n, uint32_t m) {
    const uint32_t t = ((a >> n) ^ b) & m;
    b ^= t;
    a ^= t << n;
}
TDES_HD void swap_ip(uint32_t& l, uint32_t& r) {
    bit_swap(l, r, 4, 0x0F0F0F0Fu);
    bit_swap(l, r, 16, 0x0000FFFFu);
    bit_swap(r, l, 2, 0x33333333u);
    bit_swap(r, l, 8, 0x00FF00FFu);
    bit_swap(l, r, 1, 0x55555555u);
}
TDES_HD void swap_fp(uint32_t& l, uint32_t& r) {
    bit_swap(l, r, 1, 0x55555555u);
    bit_swap(r, l, 8, 0x00FF00FFu);
    bit_swap(r, l, 2, 0x33333333u);
    bit_swap(l, r, 16, 0x0000FFFFu);
    bit_swap(l, r, 4, 0x0F0F0F0Fu);
}

// tdes_block_scalar_nib with the permutations as bit swaps: no tables to stage
// and no lookups for them.
template <int ROUNDS = 48>
TDES_HD uint64_t tdes_block_scalar_swap(uint64_t v, const uint32_t* __restrict__ sp,
                                        const uint32_t* __restrict__ keys) {
    uint32_t L = (uint32_t)(v >> 32), R = (uint32_t)v;
    swap_ip(L, R);
    uint32_t ke = keys[0], ko = keys[1];
#pragma unroll
    for (int r = 0; r < ROUNDS; r += 2) {
        const uint32_t ke1 = keys[2 * r + 2], ko1 = keys[2 * r + 3];
        L ^= tdes_f_scalar(R, ke, ko, sp);
        const int rn = r + 2 < ROUNDS ? r + 2 : r;  // the last prefetch rereads the last pair
        ke = keys[2 * rn];
        ko = keys[2 * rn + 1];
        R ^= tdes_f_scalar(L, ke1, ko1, sp);
        if ((r & 15) == 14) {  // end of a DES pass: R16 || L16 continues as the next L0 || R0
            const uint32_t u = L;
            L = R;
            R = u;
        }
    }
    swap_fp(L, R);
    return ((uint64_t)L << 32) | R;
}

TDES_HD uint64_t bswap64(uint64_t x) {
    x = ((x & 0x00FF00FF00FF00FFull) << 8) | ((x >> 8) & 0x00FF00FF00FF00FFull);
    x = ((x & 0x0000FFFF0000FFFFull) << 16) | ((x >> 16) & 0x0000FFFF0000FFFFull);
    return (x << 32) | (x >> 32);
}

#ifdef __CUDACC__
// One serial CBC-encryption chain per warp: lane l computes half bit
// i = 32 - l of the round function, i.e. one output bit of one S-box
// (TDES_LANE_SBOX_INIT), and one ballot gathers the 32 bits.  The chain is
// bound by the latency of its dependent operations, so everything else is
// kept off that path:
// - the round key is folded into the lane's 64-entry truth table, one table
//   per round and lane (12 KB of shared memory per chain, chain_tables), loaded
//   a round ahead;
// - the lane's bit of L, known a round ahead, complements the table, so the
//   ballot is the new R;
// - the table's half is chosen by one bit of R while the other five rotate into
//   a one-hot mask, and what is balloted is whether (half AND mask) is zero:
//   R -> {bit test, select} || {rotate, shift} -> AND test -> ballot;
// - FP of one block and IP of the next cancel on the chain (IP(P ^ FP(S)) =
//   IP(P) ^ S): IP of the next block's plaintext and FP of the output before run
//   beside a block's rounds (chain_walk), in the gaps between their steps.
// One block takes 0.730 us (2048-block call; 0.900 with IP and FP on the chain and
// the key XORed into the rotated R; 0.777 with IP before a block's rounds and FP
// after them, which only one warp is there to hide), 31 clocks a round; single DES
// 0.299 us (0.336; 0.343).
struct ChainLane {
    uint32_t mlo, mhi, rot, keypos;
};

// Writes the tables of rounds first, first + step, ... of the chain: entry x of
// a round's table is the lane's output bit for S-box input x ^ key group.
// keys: the chain's round-key groups (the scalar layout), in shared or global
// memory.
template <int ROUNDS>
__device__ __forceinline__ void chain_tables(uint2* __restrict__ tab, const ChainLane& c,
                                             const uint8_t* __restrict__ keys, uint32_t lane,
                                             uint32_t first, uint32_t step) {
    for (uint32_t r = first; r < ROUNDS; r += step) {
        const uint32_t k = keys[8 * r + c.keypos];
        uint32_t lo = (k & 32u) ? c.mhi : c.mlo, hi = (k & 32u) ? c.mlo : c.mhi;
        // XOR of input bit j exchanges neighbouring groups of 2^j entries
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const uint32_t m = j == 0   ? 0x55555555u
                               : j == 1 ? 0x33333333u
                               : j == 2 ? 0x0F0F0F0Fu
                               : j == 3 ? 0x00FF00FFu
                                        : 0x0000FFFFu;
            const int s = 1 << j;
            if (k >> j & 1u) {
                lo = ((lo >> s) & m) | ((lo & m) << s);
                hi = ((hi >> s) & m) | ((hi & m) << s);
            }
        }
        tab[32 * r + lane] = make_uint2(lo, hi);
    }
}

// The ROUNDS rounds on halves (L, R) in the warp's registers (the same in
// every lane); tab: the chain's tables.
template <int ROUNDS>
__device__ __forceinline__ void chain_rounds(uint32_t& L, uint32_t& R, uint32_t rot, uint32_t lane,
                                             const uint2* __restrict__ tab) {
    const uint32_t b5 = 1u << ((rot + 5u) & 31u);
    uint32_t Lm = 0u - ((L >> lane) & 1u);
    uint2 t = tab[lane];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const uint2 tn = tab[32 * (r + 1 < ROUNDS ? r + 1 : r) + lane];
        const uint32_t half = (R & b5) ? t.y ^ Lm : t.x ^ Lm;
        const uint32_t hot = __funnelshift_l(0u, 1u, __funnelshift_r(R, R, rot));
        Lm = 0u - ((R >> lane) & 1u);
        const uint32_t n = __ballot_sync(0xFFFFFFFFu, (half & hot) != 0u);
        L = R;
        R = n;
        if ((r & 15) == 15) {  // end of a DES pass: R16 || L16 continues as L0 || R0
            const uint32_t u = L;
            L = R;
            R = u;
            Lm = 0u - ((L >> lane) & 1u);
        }
        t = tn;
    }
}

// A whole chain: out_i = E(in_i XOR out_{i-1}), out_{-1} = iv, blocks as
// big-endian bytes.
template <int ROUNDS>
__device__ __forceinline__ void chain_walk(const uint8_t* in, uint8_t* out, uint64_t nblocks,
                                           uint64_t iv, uint32_t rot, uint32_t lane,
                                           const uint2* __restrict__ tab) {
    const uint64_t* p = reinterpret_cast<const uint64_t*>(in);
    uint64_t* q = reinterpret_cast<uint64_t*>(out);
    uint32_t sl = (uint32_t)(iv >> 32), sr = (uint32_t)iv;  // IP of the previous output
    swap_ip(sl, sr);
    uint64_t x = bswap64(p[0]);
    uint32_t pl = (uint32_t)(x >> 32), pr = (uint32_t)x;  // IP of the block's plaintext
    swap_ip(pl, pr);
    uint64_t next = nblocks > 1 ? p[1] : 0;
    for (uint64_t i = 0; i < nblocks; ++i) {
        uint32_t L = pl ^ sl, R = pr ^ sr;
        // beside the rounds: the plaintext of the next block and the output before
        x = bswap64(next);
        pl = (uint32_t)(x >> 32);
        pr = (uint32_t)x;
        swap_ip(pl, pr);
        if (i + 2 < nblocks) next = p[i + 2];
        swap_fp(sl, sr);
        if (i > 0 && lane == 0) q[i - 1] = bswap64(((uint64_t)sl << 32) | sr);
        chain_rounds<ROUNDS>(L, R, rot, lane, tab);
        sl = L;
        sr = R;
    }
    swap_fp(sl, sr);
    if (lane == 0) q[nblocks - 1] = bswap64(((uint64_t)sl << 32) | sr);
}
#endif
