// pms_sieve.cuh -- the sieve form's word of a window (pms_sieve.cu), written by
// the packing kernel and read by the sieve kernel. Not part of the public ABI.
#pragma once

#include "pms_internal.h"

namespace pms {

constexpr int kSvSuf = 3;   // letters inside a word of marks

// The word index of a middle with planes (hi, lo): hi << kMid | (lo ^ F(hi)),
// F linear over exclusive-or with these columns (with six letters, lo's bit 5
// is folded into the bits below it too). With 32-bit words the low five index
// bits are the bank: the columns put the 3 kMid single-letter changes and 0
// into different banks.
template <int kMid>
__host__ __device__ constexpr uint32_t sv_column(int p)
{
    if (kMid >= 5)
        return p == 0 ? 6u : p == 1 ? 12u : p == 2 ? 24u : p == 3 ? 17u : p == 4 ? 3u : 10u;
    if (kMid == 4)
        return p == 0 ? 0u : p == 1 ? 5u : p == 2 ? 9u : 6u;
    return p == 2 ? 3u : 0u;
}

template <int kMid>
__host__ __device__ constexpr uint32_t sv_fold(uint32_t hi, uint32_t lo)
{
    uint32_t f = kMid == 6 && (lo & 32u) ? 5u : 0u;
    for (int p = 0; p < kMid; ++p)
        f ^= ((hi >> p) & 1u) ? sv_column<kMid>(p) : 0u;
    return f;
}

template <int kMid>
__host__ __device__ constexpr uint32_t sv_index(uint32_t hi, uint32_t lo)
{
    return (hi << kMid) | (lo ^ sv_fold<kMid>(hi, lo));
}

// lo of an index (the fold changes the low five bits only and does not read them)
template <int kMid>
__host__ __device__ constexpr uint32_t sv_lo(uint32_t index)
{
    const uint32_t low = index & ((1u << kMid) - 1u);
    return low ^ sv_fold<kMid>(index >> kMid, low);
}

constexpr int kSvPre = 16;   // prefix letters a window's word has room for

// A window for the sieve: x = its last three letters (hi plane << 3 | lo plane)
// in bits 0..5 and the index of the middle letters above them, y = the lo plane
// of its prefix letters and, from bit 16, their hi plane. Needs
// 0 <= l - kMid - 3 <= kSvPre.
template <int kMid>
__host__ __device__ __forceinline__ uint2 sieve_word(uint32_t h, uint32_t lo, int l)
{
    constexpr uint32_t kMask = (1u << kMid) - 1u;
    const int A = l - kMid - kSvSuf;
    const uint32_t suf = (((h >> (A + kMid)) & 7u) << 3) | ((lo >> (A + kMid)) & 7u);
    const uint32_t mid = sv_index<kMid>((h >> A) & kMask, (lo >> A) & kMask);
    uint2 w;
    w.x = suf | (mid << 6);
    w.y = (lo & ((1u << A) - 1u)) | ((h & ((1u << A) - 1u)) << 16);
    return w;
}

}  // namespace pms
