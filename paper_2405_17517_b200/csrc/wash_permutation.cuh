// The permutation pi_i of a selected coordinate: Fisher-Yates over the models, position
// k = N-1 .. 1 swapped with j = floor(word * (k+1) / 2^32), the words taken in order from the
// coordinate's Philox blocks (block b = words 4b .. 4b+3).  Three carriers of the same
// permutation: nibbles of a 32-bit register (N <= 8), nibbles of a 64-bit register (N <= 16),
// bytes in shared memory (any N; drawn by a lane, or for up to 32 coordinates by a warp).
#pragma once
#include "wash_device.cuh"

namespace wash {

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// pi(n) in nibble n of the result, N <= 8: every shift is a 32-bit one
__device__ __forceinline__ uint32_t draw_permutation_packed32(int n_models, uint32_t i, uint32_t tensor, uint32_t step_lo,
                                                              uint32_t step_hi8, const PhiloxKeys &keys)
{
    uint32_t perm = 0x76543210u;
    Philox4 w{0, 0, 0, 0};
    for (int k = n_models - 1, m = 0; k >= 1; --k, ++m) {
        if ((m & 3) == 0) w = philox4x32_10(i, tensor, step_lo, step_hi8 | (1u + (static_cast<uint32_t>(m) >> 2)), keys);
        const uint32_t r = w.x;
        w.x = w.y; w.y = w.z; w.z = w.w;
        const uint32_t sk = 4u * k, sj = 4u * __umulhi(r, static_cast<uint32_t>(k + 1));
        const uint32_t diff = ((perm >> sk) ^ (perm >> sj)) & 15u;   // swap nibbles k and j
        perm ^= (diff << sk) | (diff << sj);
    }
    return perm;
}

// pi(n) in nibble n of the result, N <= 16
__device__ __forceinline__ uint64_t draw_permutation_packed(int n_models, uint32_t i, uint32_t tensor, uint32_t step_lo,
                                                            uint32_t step_hi8, const PhiloxKeys &keys)
{
    if (n_models <= 8) return 0xFEDCBA9800000000ull | draw_permutation_packed32(n_models, i, tensor, step_lo, step_hi8, keys);
    uint64_t perm = 0xFEDCBA9876543210ull;
    Philox4 w{0, 0, 0, 0};
    for (int k = n_models - 1, m = 0; k >= 1; --k, ++m) {
        if ((m & 3) == 0) w = philox4x32_10(i, tensor, step_lo, step_hi8 | (1u + (static_cast<uint32_t>(m) >> 2)), keys);
        const uint32_t r = w.x;
        w.x = w.y; w.y = w.z; w.z = w.w;
        const uint32_t sk = 4u * k, sj = 4u * __umulhi(r, static_cast<uint32_t>(k + 1));
        const uint64_t diff = ((perm >> sk) ^ (perm >> sj)) & 15ull;   // swap nibbles k and j
        perm ^= (diff << sk) | (diff << sj);
    }
    return perm;
}

// Words (4 bytes) from one lane's permutation to the next in the layout of draw_permutations_by_warp:
// odd, so that lanes that read the same place of theirs fall into different banks.
__host__ __device__ constexpr uint32_t wide_pitch(int n_models) { return (static_cast<uint32_t>(n_models + 3) / 4u) | 1u; }

// The permutations of `count` <= 32 coordinates (lane l < count holds the l-th one's coord and tensor),
// 16 < N <= 64, by a whole warp; pi_l(n) is byte n of s_perm + l * wide_pitch(N) words.  The Philox blocks
// of all coordinates are dealt to the lanes, each leaving its four swap partners where the permutation
// will be, so that no lane draws eight blocks in a row; then lane l takes the partners of coordinate l
// into registers and runs the chain of swaps.  (A lane's 64 bytes would fit its registers, but the
// places they are swapped at are data.)
__device__ __forceinline__ void draw_permutations_by_warp(uint32_t *s_perm, int n_models, uint32_t count, uint32_t coord,
                                                          uint32_t tensor, uint32_t step_lo, uint32_t step_hi8, const PhiloxKeys &keys)
{
    constexpr uint32_t kMaxBlocks = (kMaxN + 2) / 4;
    const uint32_t lane = threadIdx.x & 31u, pitch = wide_pitch(n_models), blocks = static_cast<uint32_t>(n_models + 2) / 4u;
    const uint32_t inverse = ((1u << 20) + blocks - 1u) / blocks;   // i / blocks = i * inverse >> 20 for i < 544
    for (uint32_t first = 0; first < count * blocks; first += 32) {
        const uint32_t i = first + lane, l = min((i * inverse) >> 20, count - 1u), b = i - l * blocks;
        const uint32_t its_coord = __shfl_sync(0xFFFFFFFFu, coord, l), its_tensor = __shfl_sync(0xFFFFFFFFu, tensor, l);
        if (i < count * blocks) {
            const Philox4 w = philox4x32_10(its_coord, its_tensor, step_lo, step_hi8 | (1u + b), keys);
            const uint32_t k = static_cast<uint32_t>(n_models) - 1u - 4u * b;   // the block's words swap positions k, k-1, k-2, k-3 (those >= 1)
            s_perm[l * pitch + b] = __umulhi(w.x, k + 1u) | (__umulhi(w.y, k) << 8) | (__umulhi(w.z, k - 1u) << 16) | (__umulhi(w.w, k - 2u) << 24);
        }
        __syncwarp();
    }
    if (lane < count) {
        uint32_t *mine = s_perm + lane * pitch;
        uint32_t partners[kMaxBlocks];
#pragma unroll
        for (uint32_t b = 0; b < kMaxBlocks; ++b) partners[b] = b < blocks ? mine[b] : 0u;
#pragma unroll
        for (uint32_t q = 0; q < kMaxN / 4; ++q)
            if (4u * q < static_cast<uint32_t>(n_models)) mine[q] = 0x03020100u + q * 0x04040404u;
        uint8_t *perm = reinterpret_cast<uint8_t *>(mine);
        int k = n_models - 1;
#pragma unroll
        for (uint32_t b = 0; b < kMaxBlocks; ++b) {
            if (b >= blocks) break;
#pragma unroll
            for (int q = 0; q < 4; ++q, --k) {
                if (k < 1) break;
                const uint32_t j = (partners[b] >> (8 * q)) & 255u;
                const uint8_t pk = perm[k], pj = perm[j];
                perm[k] = pj;
                perm[j] = pk;
            }
        }
    }
    __syncwarp();
}

// pi(n) in s_perm[n * stride], any N
static __device__ __noinline__ void draw_permutation_u8(uint8_t *s_perm, int stride, int n_models, uint32_t i,
                                                        uint32_t tensor, uint32_t step_lo, uint32_t step_hi8,
                                                        const PhiloxKeys &keys)
{
    for (int n = 0; n < n_models; ++n) s_perm[n * stride] = static_cast<uint8_t>(n);
    Philox4 w{0, 0, 0, 0};
    for (int k = n_models - 1, m = 0; k >= 1; --k, ++m) {
        if ((m & 3) == 0) w = philox4x32_10(i, tensor, step_lo, step_hi8 | (1u + (static_cast<uint32_t>(m) >> 2)), keys);
        const uint32_t r = w.x;
        w.x = w.y; w.y = w.z; w.z = w.w;
        const uint32_t j = __umulhi(r, static_cast<uint32_t>(k + 1));
        const uint8_t pk = s_perm[k * stride], pj = s_perm[j * stride];
        s_perm[k * stride] = pj;
        s_perm[j * stride] = pk;
    }
}

}  // namespace wash
