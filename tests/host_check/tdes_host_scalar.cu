// Host-side run of the scalar forms the kernels take (test infrastructure
// only): the block rounds with IP and FP as bit swaps, and the counter
// bit-planes of the CTR tiles.
//
// Usage: tdes_host_scalar <sw_enc|sw_dec|s1_enc|s1_dec> <48 hex K1||K2||K3>
//   reads whole 8-byte blocks on stdin, writes the results on stdout;
//   s1_*: 16 rounds on the key words of (K1, K1, K1), as for single DES.
// Usage: tdes_host_scalar planes <nonce> <c> <lane>
//   writes the 64 bit-planes of the lane's 32 counter blocks (32 words of the
//   blocks' first halves, then 32 of the second).
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../../paper_2007_10752_gb300/csrc/tdes_keysched.cuh"
#include "../../paper_2007_10752_gb300/csrc/tdes_scalar.cuh"

static const uint8_t kSub[2][48][48] = TDES_SUBKEY_INIT;
static const uint32_t kSP[8][64] = TDES_SP_INIT;

int main(int argc, char** argv) {
    if (argc == 5 && !strcmp(argv[1], "planes")) {
        uint32_t A[2][32];
        counter_planes((uint32_t)strtoull(argv[2], nullptr, 0), (uint32_t)strtoull(argv[3], nullptr, 0),
                       (uint32_t)strtoull(argv[4], nullptr, 0), A[0], A[1]);
        fwrite(A, sizeof A, 1, stdout);
        return 0;
    }
    if (argc != 3 || strlen(argv[2]) != 48) return 2;
    uint8_t keys[24];
    for (int i = 0; i < 24; ++i) {
        char h[3] = {argv[2][2 * i], argv[2][2 * i + 1], 0};
        keys[i] = (uint8_t)strtoul(h, nullptr, 16);
    }
    const bool dec = strstr(argv[1], "dec") != nullptr, one = strncmp(argv[1], "s1", 2) == 0;
    if (one)
        for (int i = 8; i < 24; ++i) keys[i] = keys[i - 8];
    alignas(16) uint8_t chunks[TDES_SUBKEY_WORDS];
    for (int r = 0; r < 48; ++r)
        for (int g = 0; g < 8; ++g) chunks[8 * r + g] = tdes_subkey_chunk(keys, &kSub[dec][r][6 * g]);
    const uint32_t* kw = reinterpret_cast<const uint32_t*>(chunks);
    uint64_t v;
    while (fread(&v, 8, 1, stdin) == 1) {
        v = bswap64(v);
        v = one ? tdes_block_scalar_swap<16>(v, &kSP[0][0], kw) : tdes_block_scalar_swap<48>(v, &kSP[0][0], kw);
        v = bswap64(v);
        fwrite(&v, 8, 1, stdout);
    }
    return 0;
}
