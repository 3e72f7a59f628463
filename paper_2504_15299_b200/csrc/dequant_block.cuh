// Dequantization of a row of a packed block in blocks of 32 codes (16 registers of half pairs), shared by the grouped GEMM kernels.
#pragma once
#include "tc_common.cuh"

// Sixteen registers (32 codes, block b of a row) of a stored segment of SW bits per code: SW words.
template <int GS, int SW>
__device__ __forceinline__ void load_block(uint32_t row, int b, uint32_t (&w)[SW]) {
    constexpr int CS = GS * SW / 8 < 16 ? GS * SW / 8 : 16;
    const int ob = 4 * SW * b;
    const uint32_t addr = row + (uint32_t)((ob / CS) * D2MOE_TILE_ROWS * CS + ob % CS);
    if constexpr (SW == 8) {
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(addr));
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "r"(addr + D2MOE_TILE_ROWS * CS));
    } else if constexpr (SW == 4) {
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(addr));
    } else if constexpr (SW == 2) {
        asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(addr));
    } else {
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[0]) : "r"(addr));
    }
}

// One field of every code of a block (the bits of `field`, repeated in both halves of the mask) as half pairs: v = field * mult + addend
template <int SW>
__device__ __forceinline__ void fma_block(const uint32_t (&w)[SW], uint32_t field, const uint32_t (&mult)[8 / SW], uint32_t c, uint32_t (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        constexpr int PER = 16 / SW;                            // registers per word
        const int e = i % PER;
        const uint32_t src = (e & 1) ? w[i / PER] >> 8 : w[i / PER];      // pair e of the word: bytes (0,2) or (1,3), bit SW*(e/2)
        v[i] = hfma2_bits(src & (field << ((e >> 1) * SW)), mult[e >> 1], c);
    }
}
template <int SW>
__device__ __forceinline__ void fma_block_more(const uint32_t (&w)[SW], uint32_t field, const uint32_t (&mult)[8 / SW], uint32_t (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        constexpr int PER = 16 / SW;
        const int e = i % PER;
        const uint32_t src = (e & 1) ? w[i / PER] >> 8 : w[i / PER];
        v[i] = hfma2_bits(src & (field << ((e >> 1) * SW)), mult[e >> 1], v[i]);
    }
}
// multipliers of the fields at bit positions 0, SW, 2 SW, ... of a byte lane, from that of position 0
template <int SW>
__device__ __forceinline__ void field_mults(float m0, uint32_t (&mult)[8 / SW]) {
    mult[0] = as_u32(h2dup(m0));
    const uint32_t step = (uint32_t)(15 - SW) * 0x04000400u;            // 2^-SW, exact
#pragma unroll
    for (int q = 1; q < 8 / SW; ++q) mult[q] = hmul2_bits(mult[q - 1], step);
}
