// GENERATED by paper_2007_10752_gb300/gen/emit_cuda.py -- do not edit.
// Round of the bitsliced path for tables with a different key per bit
// position (from the S-box circuits in gen/sbox_lop3.json).
#pragma once
#include <cstdint>

// Needs TDES_HD and lop3<LUT>(a, b, c) from tdes_bitslice.cuh.

// The same round for tables whose masks differ from bit to bit (one key
// per bit position: tiles of small messages under many keys).  The
// multiply-add form of a masked XOR holds only for all-0 or all-1 masks,
// so the doubled expansion inputs take a plain XOR; the multipliers are
// not read.
TDES_HD void tdes_round_mixed(uint32_t (&T)[32], const uint32_t (&S)[32],
                              const uint32_t* __restrict__ k) {
    {  // S-box 1
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 4);
    const uint32_t x0 = S[31] ^ kd.x;  // second copy
    const uint32_t x1 = S[0] ^ kd.y;
    const uint32_t x2 = S[1];
    const uint32_t x3 = S[2];
    const uint32_t x4 = S[3];
    const uint32_t x5 = S[4];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 0);
    const uint32_t s0_0 = lop3<0x17>(x5, x4, x2);
    const uint32_t s0_1 = lop3<0x1d>(s0_0, x3, x2);
    const uint32_t s0_2 = lop3<0x6b>(x3, s0_1, x1);
    const uint32_t s0_3 = lop3<0x69>(x5, s0_2, x4);
    const uint32_t s0_4 = lop3<0x97>(s0_3, x2, x1);
    const uint32_t s0_5 = lop3<0x4f>(s0_1, x5, x3);
    const uint32_t s0_6 = lop3<0x5e>(s0_3, x5, x4);
    const uint32_t s0_7 = lop3<0xd1>(s0_4, s0_5, s0_6);
    const uint32_t s0_8 = lop3<0xe4>(s0_7, s0_3, x0);
    T[8] = lop3<0x96>(T[8], s0_8, kc.x);
    const uint32_t s0_9 = lop3<0x59>(x5, x3, x0);
    const uint32_t s0_10 = lop3<0x56>(s0_8, s0_9, s0_1);
    const uint32_t s0_11 = lop3<0x61>(x5, x3, x0);
    const uint32_t s0_12 = lop3<0x34>(s0_10, s0_7, s0_11);
    const uint32_t s0_13 = lop3<0x58>(s0_3, x5, x3);
    const uint32_t s0_14 = lop3<0x6d>(s0_2, s0_13, s0_4);
    const uint32_t s0_15 = lop3<0x53>(s0_10, s0_2, x3);
    const uint32_t s0_16 = lop3<0x79>(s0_15, s0_12, x4);
    const uint32_t s0_17 = lop3<0x78>(s0_14, s0_16, x0);
    T[22] = lop3<0x96>(T[22], s0_17, kc.z);
    const uint32_t s0_18 = lop3<0xdc>(s0_17, s0_11, x3);
    const uint32_t s0_19 = lop3<0xd6>(s0_18, s0_3, x2);
    const uint32_t s0_20 = lop3<0xe4>(s0_12, s0_19, x1);
    T[16] = lop3<0x96>(T[16], s0_20, kc.y);
    const uint32_t s0_21 = lop3<0xf9>(s0_10, s0_6, x1);
    const uint32_t s0_22 = lop3<0xe1>(s0_21, s0_16, x5);
    const uint32_t s0_23 = lop3<0x5b>(s0_22, s0_1, x2);
    const uint32_t s0_24 = lop3<0x96>(s0_23, x1, x0);
    T[30] = lop3<0x96>(T[30], s0_24, kc.w);
    }
    {  // S-box 2
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 12);
    const uint32_t x0 = S[3] ^ kd.x;  // second copy
    const uint32_t x1 = S[4] ^ kd.y;
    const uint32_t x2 = S[5];
    const uint32_t x3 = S[6];
    const uint32_t x4 = S[7];
    const uint32_t x5 = S[8];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 8);
    const uint32_t s1_0 = lop3<0x38>(x5, x2, x1);
    const uint32_t s1_1 = lop3<0x78>(x4, x3, x1);
    const uint32_t s1_2 = lop3<0x96>(s1_1, s1_0, x3);
    const uint32_t s1_3 = lop3<0x84>(x3, s1_1, x5);
    const uint32_t s1_4 = lop3<0x05>(s1_3, x3, x1);
    const uint32_t s1_5 = lop3<0x4a>(x5, s1_4, x0);
    const uint32_t s1_6 = lop3<0xad>(s1_5, s1_4, s1_1);
    const uint32_t s1_7 = lop3<0xd0>(s1_5, x5, x1);
    const uint32_t s1_8 = lop3<0xc5>(s1_7, x2, x4);
    const uint32_t s1_9 = lop3<0x46>(s1_8, s1_0, x0);
    const uint32_t s1_10 = lop3<0x2d>(s1_6, s1_9, x2);
    T[12] = lop3<0x69>(T[12], s1_10, kc.x);
    const uint32_t s1_11 = lop3<0xe9>(s1_10, s1_5, x0);
    const uint32_t s1_12 = lop3<0x31>(s1_10, s1_4, s1_8);
    const uint32_t s1_13 = lop3<0x04>(s1_12, s1_11, x4);
    const uint32_t s1_14 = lop3<0x96>(s1_5, s1_13, s1_2);
    T[17] = lop3<0x96>(T[17], s1_14, kc.w);
    const uint32_t s1_15 = lop3<0x67>(s1_12, s1_3, s1_0);
    const uint32_t s1_16 = lop3<0xac>(s1_15, s1_6, s1_2);
    const uint32_t s1_17 = lop3<0x69>(s1_16, x1, x0);
    T[27] = lop3<0x96>(T[27], s1_17, kc.y);
    const uint32_t s1_18 = lop3<0x92>(s1_16, x5, x1);
    const uint32_t s1_19 = lop3<0xf9>(s1_18, s1_14, s1_5);
    const uint32_t s1_20 = lop3<0x96>(s1_19, s1_11, s1_8);
    T[1] = lop3<0x69>(T[1], s1_20, kc.z);
    }
    {  // S-box 3
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 20);
    const uint32_t x0 = S[7] ^ kd.x;  // second copy
    const uint32_t x1 = S[8] ^ kd.y;
    const uint32_t x2 = S[9];
    const uint32_t x3 = S[10];
    const uint32_t x4 = S[11];
    const uint32_t x5 = S[12];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 16);
    const uint32_t s2_0 = lop3<0x3c>(x5, x3, x1);
    const uint32_t s2_1 = lop3<0x86>(x5, x4, x2);
    const uint32_t s2_2 = lop3<0xb1>(s2_1, s2_0, x4);
    const uint32_t s2_3 = lop3<0x69>(x1, s2_2, x0);
    const uint32_t s2_4 = lop3<0xde>(s2_1, s2_0, x1);
    const uint32_t s2_5 = lop3<0xbe>(s2_4, x1, x0);
    const uint32_t s2_6 = lop3<0x62>(s2_5, s2_3, x2);
    const uint32_t s2_7 = lop3<0x87>(s2_6, s2_4, x3);
    T[15] = lop3<0x69>(T[15], s2_7, kc.y);
    const uint32_t s2_8 = lop3<0xf4>(s2_7, x5, x3);
    const uint32_t s2_9 = lop3<0x37>(s2_8, s2_3, x0);
    const uint32_t s2_10 = lop3<0x46>(s2_9, s2_6, x4);
    const uint32_t s2_11 = lop3<0x72>(s2_10, s2_1, x5);
    const uint32_t s2_12 = lop3<0x5e>(s2_11, s2_3, x3);
    const uint32_t s2_13 = lop3<0xb6>(s2_8, x4, x1);
    const uint32_t s2_14 = lop3<0xb5>(s2_11, s2_8, x0);
    const uint32_t s2_15 = lop3<0x36>(s2_14, x1, s2_1);
    const uint32_t s2_16 = lop3<0xd6>(s2_15, x0, x2);
    const uint32_t s2_17 = lop3<0x69>(s2_16, x4, s2_0);
    T[23] = lop3<0x69>(T[23], s2_17, kc.x);
    const uint32_t s2_18 = lop3<0x25>(s2_17, s2_10, s2_9);
    const uint32_t s2_19 = lop3<0x87>(s2_18, s2_12, x1);
    T[29] = lop3<0x96>(T[29], s2_19, kc.z);
    const uint32_t s2_20 = lop3<0xb3>(s2_19, s2_13, x5);
    const uint32_t s2_21 = lop3<0xc6>(s2_20, s2_3, x0);
    T[5] = lop3<0x96>(T[5], s2_21, kc.w);
    }
    {  // S-box 4
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 28);
    const uint32_t x0 = S[11] ^ kd.x;  // second copy
    const uint32_t x1 = S[12] ^ kd.y;
    const uint32_t x2 = S[13];
    const uint32_t x3 = S[14];
    const uint32_t x4 = S[15];
    const uint32_t x5 = S[16];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 24);
    const uint32_t s3_0 = lop3<0x78>(x3, x2, x0);
    const uint32_t s3_1 = lop3<0x87>(x4, x2, x1);
    const uint32_t s3_2 = lop3<0x7c>(s3_1, x1, x0);
    const uint32_t s3_3 = lop3<0x65>(s3_2, s3_0, x2);
    const uint32_t s3_4 = lop3<0x96>(s3_3, s3_1, x0);
    const uint32_t s3_5 = lop3<0x59>(s3_4, s3_1, x1);
    const uint32_t s3_6 = lop3<0xd2>(s3_0, s3_5, s3_2);
    const uint32_t s3_7 = lop3<0x84>(s3_6, s3_5, x0);
    const uint32_t s3_8 = lop3<0x34>(s3_6, s3_4, x0);
    const uint32_t s3_9 = lop3<0x1c>(s3_8, s3_4, x4);
    const uint32_t s3_10 = lop3<0x1e>(s3_3, s3_8, s3_7);
    const uint32_t s3_11 = lop3<0x1b>(s3_10, s3_4, x5);
    T[0] = lop3<0x69>(T[0], s3_11, kc.w);
    const uint32_t s3_12 = lop3<0x8d>(s3_10, s3_4, x5);
    T[9] = lop3<0x69>(T[9], s3_12, kc.z);
    const uint32_t s3_13 = lop3<0x96>(s3_10, s3_9, x3);
    const uint32_t s3_14 = lop3<0x27>(s3_13, s3_6, x5);
    T[25] = lop3<0x96>(T[25], s3_14, kc.x);
    const uint32_t s3_15 = lop3<0xb1>(s3_13, s3_6, x5);
    T[19] = lop3<0x96>(T[19], s3_15, kc.y);
    }
    {  // S-box 5
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 36);
    const uint32_t x0 = S[15] ^ kd.x;  // second copy
    const uint32_t x1 = S[16] ^ kd.y;
    const uint32_t x2 = S[17];
    const uint32_t x3 = S[18];
    const uint32_t x4 = S[19];
    const uint32_t x5 = S[20];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 32);
    const uint32_t s4_0 = lop3<0x82>(x4, x2, x0);
    const uint32_t s4_1 = lop3<0x49>(x5, x3, x2);
    const uint32_t s4_2 = lop3<0xc2>(x4, s4_0, s4_1);
    const uint32_t s4_3 = lop3<0x29>(x2, s4_2, x3);
    const uint32_t s4_4 = lop3<0xc9>(s4_2, x5, x0);
    const uint32_t s4_5 = lop3<0x61>(s4_4, x4, x3);
    const uint32_t s4_6 = lop3<0x16>(s4_2, x5, x2);
    const uint32_t s4_7 = lop3<0x32>(s4_6, s4_3, x4);
    const uint32_t s4_8 = lop3<0x9e>(s4_4, s4_3, s4_1);
    const uint32_t s4_9 = lop3<0x8a>(s4_8, x3, x1);
    const uint32_t s4_10 = lop3<0xa8>(s4_8, s4_0, x4);
    const uint32_t s4_11 = lop3<0xec>(s4_10, s4_5, s4_1);
    const uint32_t s4_12 = lop3<0xd2>(s4_11, s4_7, x1);
    T[2] = lop3<0x69>(T[2], s4_12, kc.w);
    const uint32_t s4_13 = lop3<0x64>(s4_9, s4_11, s4_7);
    const uint32_t s4_14 = lop3<0xb6>(s4_13, x4, x0);
    const uint32_t s4_15 = lop3<0x7c>(s4_13, s4_8, s4_3);
    const uint32_t s4_16 = lop3<0x95>(s4_9, s4_15, s4_6);
    const uint32_t s4_17 = lop3<0xa5>(s4_9, s4_2, s4_1);
    const uint32_t s4_18 = lop3<0x96>(s4_17, s4_10, x0);
    T[13] = lop3<0x96>(T[13], s4_18, kc.y);
    const uint32_t s4_19 = lop3<0x96>(s4_16, s4_14, x1);
    T[7] = lop3<0x96>(T[7], s4_19, kc.x);
    const uint32_t s4_20 = lop3<0x69>(s4_19, s4_13, s4_18);
    const uint32_t s4_21 = lop3<0xc6>(s4_14, s4_20, s4_12);
    T[24] = lop3<0x69>(T[24], s4_21, kc.z);
    }
    {  // S-box 6
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 44);
    const uint32_t x0 = S[19] ^ kd.x;  // second copy
    const uint32_t x1 = S[20] ^ kd.y;
    const uint32_t x2 = S[21];
    const uint32_t x3 = S[22];
    const uint32_t x4 = S[23];
    const uint32_t x5 = S[24];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 40);
    const uint32_t s5_0 = lop3<0xc6>(x1, x3, x2);
    const uint32_t s5_1 = lop3<0x2d>(x5, x4, x2);
    const uint32_t s5_2 = lop3<0xa2>(s5_1, x5, x3);
    const uint32_t s5_3 = lop3<0x96>(x0, s5_0, x4);
    const uint32_t s5_4 = lop3<0x3e>(s5_1, x2, x1);
    const uint32_t s5_5 = lop3<0x86>(s5_0, x5, x1);
    const uint32_t s5_6 = lop3<0x59>(s5_4, x0, s5_3);
    const uint32_t s5_7 = lop3<0x4a>(s5_3, x4, x2);
    const uint32_t s5_8 = lop3<0x61>(x0, s5_7, x2);
    const uint32_t s5_9 = lop3<0x38>(s5_8, s5_0, x1);
    const uint32_t s5_10 = lop3<0x36>(s5_9, x1, x5);
    const uint32_t s5_11 = lop3<0x96>(s5_9, s5_10, s5_7);
    T[3] = lop3<0x69>(T[3], s5_11, kc.x);
    const uint32_t s5_12 = lop3<0xcb>(s5_2, s5_11, x4);
    const uint32_t s5_13 = lop3<0x3d>(s5_9, s5_5, s5_3);
    const uint32_t s5_14 = lop3<0x9c>(x3, s5_6, s5_12);
    T[18] = lop3<0x69>(T[18], s5_14, kc.w);
    const uint32_t s5_15 = lop3<0x7c>(s5_10, s5_7, x1);
    const uint32_t s5_16 = lop3<0x73>(s5_4, s5_15, x0);
    const uint32_t s5_17 = lop3<0x35>(s5_16, s5_13, s5_3);
    T[28] = lop3<0x69>(T[28], s5_17, kc.y);
    const uint32_t s5_18 = lop3<0x87>(s5_17, s5_2, s5_16);
    const uint32_t s5_19 = lop3<0xc9>(s5_14, s5_18, s5_11);
    const uint32_t s5_20 = lop3<0x1e>(s5_15, s5_13, s5_8);
    const uint32_t s5_21 = lop3<0x36>(s5_20, s5_19, x1);
    T[10] = lop3<0x69>(T[10], s5_21, kc.z);
    }
    {  // S-box 7
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 52);
    const uint32_t x0 = S[23] ^ kd.x;  // second copy
    const uint32_t x1 = S[24] ^ kd.y;
    const uint32_t x2 = S[25];
    const uint32_t x3 = S[26];
    const uint32_t x4 = S[27];
    const uint32_t x5 = S[28];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 48);
    const uint32_t s6_0 = lop3<0x69>(x5, x2, x0);
    const uint32_t s6_1 = lop3<0x93>(x5, x3, x1);
    const uint32_t s6_2 = lop3<0x5e>(s6_1, x4, x1);
    const uint32_t s6_3 = lop3<0x81>(s6_1, x3, x0);
    const uint32_t s6_4 = lop3<0x26>(s6_3, s6_2, x2);
    const uint32_t s6_5 = lop3<0x52>(x4, s6_4, x3);
    const uint32_t s6_6 = lop3<0xe1>(s6_5, s6_4, x1);
    const uint32_t s6_7 = lop3<0xea>(s6_6, x5, x0);
    const uint32_t s6_8 = lop3<0x69>(s6_7, s6_4, x4);
    const uint32_t s6_9 = lop3<0x69>(s6_6, x1, x5);
    const uint32_t s6_10 = lop3<0x36>(s6_6, s6_3, x3);
    const uint32_t s6_11 = lop3<0x69>(s6_10, s6_9, x2);
    const uint32_t s6_12 = lop3<0xb8>(s6_0, s6_11, s6_1);
    const uint32_t s6_13 = lop3<0x69>(s6_12, x1, x4);
    T[11] = lop3<0x69>(T[11], s6_13, kc.y);
    const uint32_t s6_14 = lop3<0x0d>(s6_13, s6_6, x5);
    const uint32_t s6_15 = lop3<0x02>(s6_13, s6_8, x5);
    const uint32_t s6_16 = lop3<0x39>(s6_15, s6_9, x0);
    T[6] = lop3<0x96>(T[6], s6_16, kc.w);
    const uint32_t s6_17 = lop3<0x7d>(s6_14, s6_3, x0);
    const uint32_t s6_18 = lop3<0xca>(s6_17, s6_8, s6_11);
    T[21] = lop3<0x96>(T[21], s6_18, kc.z);
    const uint32_t s6_19 = lop3<0xe1>(s6_13, s6_11, s6_3);
    const uint32_t s6_20 = lop3<0xf8>(s6_17, x4, x2);
    const uint32_t s6_21 = lop3<0x67>(s6_1, s6_20, s6_19);
    T[31] = lop3<0x96>(T[31], s6_21, kc.x);
    }
    {  // S-box 8
    const uint4 kd = *reinterpret_cast<const uint4*>(k + 60);
    const uint32_t x0 = S[27] ^ kd.x;  // second copy
    const uint32_t x1 = S[28] ^ kd.y;
    const uint32_t x2 = S[29];
    const uint32_t x3 = S[30];
    const uint32_t x4 = S[31];
    const uint32_t x5 = S[0];
    const uint4 kc = *reinterpret_cast<const uint4*>(k + 56);
    const uint32_t s7_0 = lop3<0x91>(x1, x4, x2);
    const uint32_t s7_1 = lop3<0xe5>(s7_0, x5, x3);
    const uint32_t s7_2 = lop3<0x9a>(x1, s7_1, x4);
    const uint32_t s7_3 = lop3<0x61>(x1, x4, x3);
    const uint32_t s7_4 = lop3<0x4d>(s7_3, s7_0, x3);
    const uint32_t s7_5 = lop3<0x8a>(s7_4, x4, x0);
    const uint32_t s7_6 = lop3<0x69>(s7_5, s7_3, x2);
    const uint32_t s7_7 = lop3<0x94>(s7_2, s7_6, x5);
    const uint32_t s7_8 = lop3<0x6a>(x0, s7_7, s7_4);
    const uint32_t s7_9 = lop3<0xb3>(s7_8, s7_6, x5);
    const uint32_t s7_10 = lop3<0xb2>(s7_9, s7_2, s7_4);
    const uint32_t s7_11 = lop3<0x3e>(s7_10, x1, x5);
    const uint32_t s7_12 = lop3<0x69>(x0, s7_8, s7_2);
    T[14] = lop3<0x96>(T[14], s7_12, kc.z);
    const uint32_t s7_13 = lop3<0x39>(s7_11, s7_6, s7_5);
    const uint32_t s7_14 = lop3<0x69>(s7_13, s7_8, x5);
    T[26] = lop3<0x96>(T[26], s7_14, kc.y);
    const uint32_t s7_15 = lop3<0xa6>(s7_14, s7_5, x1);
    const uint32_t s7_16 = lop3<0x69>(s7_15, s7_10, x0);
    const uint32_t s7_17 = lop3<0x74>(s7_16, x5, s7_6);
    T[4] = lop3<0x69>(T[4], s7_17, kc.x);
    const uint32_t s7_18 = lop3<0xe4>(s7_16, s7_6, x5);
    T[20] = lop3<0x69>(T[20], s7_18, kc.w);
    }
}

