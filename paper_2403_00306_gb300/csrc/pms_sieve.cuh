// pms_sieve.cuh -- the sieve form's word of a window (pms_sieve.cu), written by
// the packing kernel and read by the sieve kernel. Not part of the public ABI.
#pragma once

#include "pms_internal.h"

namespace pms {

constexpr int kSvSuf = 3;   // letters inside a word of marks

// The word index of a middle with planes (hi, lo): hi << kMid | (lo ^ F(hi)),
// F linear over exclusive-or with these columns. With 32-bit words the low
// five index bits are the bank: the columns put the 3 kMid single-letter
// changes and 0 into different banks.
template <int kMid>
__host__ __device__ constexpr uint32_t sv_column(int p)
{
    if (kMid == 5)
        return p == 0 ? 6u : p == 1 ? 12u : p == 2 ? 24u : p == 3 ? 17u : 3u;
    if (kMid == 4)
        return p == 0 ? 0u : p == 1 ? 5u : p == 2 ? 9u : 6u;
    return p == 2 ? 3u : 0u;
}

template <int kMid>
__host__ __device__ constexpr uint32_t sv_fold(uint32_t hi)
{
    uint32_t f = 0;
    for (int p = 0; p < kMid; ++p)
        f ^= ((hi >> p) & 1u) ? sv_column<kMid>(p) : 0u;
    return f;
}

template <int kMid>
__host__ __device__ constexpr uint32_t sv_index(uint32_t hi, uint32_t lo)
{
    return (hi << kMid) | (lo ^ sv_fold<kMid>(hi));
}

// Letters of the prefix part of a sieve word: this many for each plane.
template <int kMid>
__host__ __device__ constexpr int sv_pre()
{
    return (32 - 6 - 2 * kMid) / 2;        // 8, 9, 10 letters for kMid = 5, 4, 3
}

// A window as one word: last three letters (hi plane << 3 | lo plane) in bits
// 0..5, the index of the middle letters above them, then the lo and the hi
// plane of the prefix letters. Needs l - kMid - 3 <= sv_pre<kMid>().
template <int kMid>
__host__ __device__ __forceinline__ uint32_t sieve_word(uint32_t h, uint32_t lo, int l)
{
    constexpr int kPre = sv_pre<kMid>();
    constexpr uint32_t kMask = (1u << kMid) - 1u;
    const int A = l - kMid - kSvSuf;
    const uint32_t suf = (((h >> (A + kMid)) & 7u) << 3) | ((lo >> (A + kMid)) & 7u);
    const uint32_t mid = sv_index<kMid>((h >> A) & kMask, (lo >> A) & kMask);
    const uint32_t pre_l = lo & ((1u << A) - 1u), pre_h = h & ((1u << A) - 1u);
    return suf | (mid << 6) | (pre_l << (6 + 2 * kMid)) | (pre_h << (6 + 2 * kMid + kPre));
}

}  // namespace pms
