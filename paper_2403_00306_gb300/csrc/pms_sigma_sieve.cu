// pms_sigma_sieve.cu -- general alphabets, q = n, d <= 4: the letters of a tree
// node found by a sieve (sm_103a).
//
// As in pms_sigma.cu a seed is a window x of s_1, its rows are the windows w of
// the other sequences with d_H(x, w) <= 2d, and a node is a set P of k <= d
// changed positions; its candidates are the k-tuples of letters other than x's
// there. A row has slack s = d - popc(D_w ^ P) changes left on P (D_w: its
// mismatches with x), and allows exactly the tuples that differ from its own
// letters on at most s of the positions of P where it differs from x (where it
// agrees with x every candidate mismatches it, which popc(D_w ^ P) counts). The
// depth-first search of pms_sigma.cu tries letter after letter and rescans the
// rows each time. Here the tuples are a bit map in shared memory: a word per
// choice of up to two letters, a bit per letter at the last position; at k = 4
// the first letter is fixed and its choices are taken one after another. The
// rows of a sequence mark the tuples they allow, and the marks of the sequences
// are intersected, smallest sequence first, until few tuples are left; those
// are looked up in the remaining sequences' rows. Most rows that pass have no
// slack and allow one tuple: one atomic OR by one lane. A row with slack marks
// the subcubes in which s letters are free, a warp at a time.
//
// A warp works on a node alone; nothing waits for another warp while a seed's
// nodes last. What a row needs (slack, letters, where it differs) fits in one
// word, listed once per node for the first sequences.
//
// What bounds it: instruction issue. Protein (9,4), n = 20, m = 600 (one GB300):
// 1.4 M blocks of a node and a first letter, three sequences each before fewer
// than one chance tuple of 6859 is left; 54.1 ms in the depth-first form
// (latency of its row lists: 4.2e9 comparisons at 0.016 of the POPC rate),
// 7.0 ms with a CTA per node (barriers, and waits for the warp with the rows
// that have slack), 2.6 ms with a warp per node. (9,3): 240 -> 106 us;
// (11,4): 706 -> 385 us; 16 letters, (9,4): 105.8 -> 3.3 ms.
#include <algorithm>

#include "pms_internal.h"

namespace pms {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kSsThreads = 256;
constexpr int kSsWarps = kSsThreads / 32;
// Lanes that still hold tuples, at or below which they are looked up instead of
// marking the next sequence: a lookup reads a sequence's rows once per tuple.
constexpr int kSsLookupLanes = 1;
// Sequences whose rows are listed per node, and the room for their entries.
constexpr int kSsListSeqs = 4, kSsListCap = 384;

__device__ uint32_t g_ss_binom[33][5];   // C(a, k), k <= 4

// One seed as the node search reads it.
struct SsSeed {
    const unsigned long long *L;     // row e: letter at position p in bits b p .. b p + b - 1
    const uint32_t *D;               // row e: mismatch mask against x; null: in L from bit b l on
    const int *off;                  // rows of sequence i: [off[i], off[i + 1])
    const int *order;                // the other sequences, fewest rows first
    int seqs;                        // how many
    int l, d, b, sigma;
    unsigned long long x;            // the seed's letters
};

__device__ __forceinline__ uint32_t ss_mask(const SsSeed &S, int e)
{
    return S.D ? S.D[e] : (uint32_t)(S.L[e] >> (S.b * S.l));
}

struct SsCount {
    unsigned int nodes, pruned, leaves, reduce, verify;
};

__device__ __forceinline__ int ss_letter(unsigned long long w, int b, int p)
{
    return (int)(w >> (b * p)) & ((1 << b) - 1);
}

// Positions at which two packed strings differ: a field's bits ORed onto its lowest.
__device__ __forceinline__ int ss_distance(unsigned long long a, unsigned long long c, int b, unsigned long long ones)
{
    const unsigned long long x = a ^ c;
    unsigned long long y = x;
    for (int s = 1; s < b; ++s)
        y |= x >> s;
    return __popcll(y & ones);
}

// Stores the string c as raw key number `slot`, if there is room for it.
__device__ __forceinline__ void ss_store(unsigned long long *raw, unsigned long long raw_cap, unsigned long long slot,
                                         unsigned long long c, int l, int b)
{
    if (slot < raw_cap) {
        unsigned long long key = 0;
        for (int q = 0; q < l; ++q)
            key = (key << b) | (unsigned long long)ss_letter(c, b, q);
        raw[3 * slot] = 0;
        raw[3 * slot + 1] = 0;
        raw[3 * slot + 2] = key;
    }
}

// Appends the string c to the raw keys (one lane).
__device__ __forceinline__ void ss_put(const SigmaParams &p, unsigned long long c, int l, int b)
{
    ss_store(p.raw, p.raw_cap, atomicAdd(p.raw_count, 1ull), c, l, b);
}

// Is there a row of sequence i within the node bound? Warp-uniform.
__device__ __forceinline__ bool ss_row_passes(const SsSeed &S, int i, uint32_t P, int lane, SsCount &ct)
{
    for (int e0 = S.off[i]; e0 < S.off[i + 1]; e0 += 32) {
        const int e = e0 + lane;
        bool hit = false;
        if (e < S.off[i + 1]) {
            ct.reduce++;
            hit = __popc(ss_mask(S, e) ^ P) <= S.d;
        }
        if (__any_sync(kFull, hit))
            return true;
    }
    return false;
}

// What row e means at node P (positions pos): bits 0..4, 5..9, ... its letters
// there, bits 20..23 where it differs from x, bits 24.. its slack; kSsNoRow for
// a row beyond the bound.
constexpr uint32_t kSsNoRow = kFull;
__device__ __forceinline__ uint32_t ss_entry(const SsSeed &S, int e, uint32_t P, int k, const int (&pos)[4])
{
    const uint32_t De = ss_mask(S, e);
    const int s = S.d - __popc(De ^ P);
    if (s < 0)
        return kSsNoRow;
    const unsigned long long w = S.L[e];
    uint32_t v = (uint32_t)s << 24;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (j < k)
            v |= ((uint32_t)ss_letter(w, S.b, pos[j]) << (5 * j)) | (((De >> pos[j]) & 1u) << (20 + j));
    return v;
}

// The tuples of a block that 32 rows allow (entry v of each lane), marked in map.
// kPre: the first letter is `a`, and the word letters are the second and third;
// otherwise they are the first k - 1.
template <bool kPre>
__device__ __forceinline__ void ss_mark(uint32_t v, int a, int k, int sigma, uint32_t all, uint32_t *map, int lane)
{
    int s = v == kSsNoRow ? -1 : (int)(v >> 24);
    uint32_t fr = (v >> 20) & 15u, let = v & 0xfffffu;
    if (kPre) {
        s -= ((fr & 1u) && (int)(let & 31u) != a) ? 1 : 0;
        fr >>= 1;
        let >>= 5;
    }
    const int J = kPre ? 2 : k - 1;                 // word letters
    const int l0 = (int)(let & 31u), l1 = (int)((let >> 5) & 31u);
    const int at = J == 2 ? l0 * sigma + l1 : J == 1 ? l0 : 0;
    const uint32_t last = 1u << ((let >> (5 * J)) & 31u);
    const uint32_t words = (1u << J) - 1u;
    const bool bit_free = (fr >> J) & 1u;           // the row differs from x at the last position
    if (s == 0 && (fr & words) == words)
        atomicOr(map + at, bit_free ? last : all);
    uint32_t todo = __ballot_sync(kFull, s > 0 || (s == 0 && (fr & words) != words));
    const uint32_t mine = ((uint32_t)max(s, 0) << 24) | (fr << 20) | let;
    while (todo) {
        const uint32_t u = __shfl_sync(kFull, mine, __ffs(todo) - 1);
        todo &= todo - 1u;
        const int us = (int)(u >> 24), r0 = (int)(u & 31u), r1 = (int)((u >> 5) & 31u);
        const uint32_t g = (u >> 20) & words;       // word letters that count
        const bool gb = (u >> (20 + J)) & 1u;
        const int fw = __popc(g);
        // us word letters off: only the row's last letter, unless a change is left for it
        const uint32_t mb = (us > fw || !gb) ? all : 1u << ((u >> (5 * J)) & 31u);
        if (us >= fw) {   // every word
            const int size = J == 2 ? sigma * sigma : J == 1 ? sigma : 1;
            for (int q = lane; q < size; q += 32)
                atomicOr(map + q, mb);
            if (us > fw || mb == all || fw == 0)
                continue;
        }
        // us of the word letters off (fewer than fw), then us - 1 off: every last letter
        if (J == 2 && g == 3u && us >= 1) {
            const uint32_t m = us == 2 ? all : mb;
            if (lane < sigma) {
                atomicOr(map + r0 * sigma + lane, m);
                atomicOr(map + lane * sigma + r1, m);
            }
            if (us == 1 && lane == 0)
                atomicOr(map + r0 * sigma + r1, all);
        } else if (J == 2 && fw == 1) {
            // one word letter counts, the other is free: us = 0 its row or column; us = 1 (= fw) that with every last letter
            if (lane < sigma)
                atomicOr(map + (g == 1u ? r0 * sigma + lane : lane * sigma + r1), us == 0 ? mb : all);
        } else if (J == 1 && lane == 0) {
            atomicOr(map + r0, us == 0 ? mb : all);   // us = 1 = fw: its own word whole
        }
    }
}

// Puts the letters of map word `word` of a block into c, at all positions of the node but the
// last (positions pos, 8 bits each); false if one of them is x's own: the word is not the node's.
template <bool kPre>
__device__ __forceinline__ bool ss_word(unsigned long long x, int b, int sigma, int word, int a, int k, uint32_t pos,
                                        unsigned long long &c)
{
    bool ok = true;
    c = x;
    for (int j = k - 2; j >= 0; --j) {
        int letter = a;
        if (!kPre || j > 0) {
            letter = word % sigma;
            word /= sigma;
        }
        const int at = (int)(pos >> (8 * j)) & 31;
        ok = ok && letter != ss_letter(x, b, at);
        c = (c & ~(((1ull << b) - 1ull) << (b * at))) | ((unsigned long long)letter << (b * at));
    }
    return ok;
}

// Every string left in the map of a block is a motif: a lane stores those of its own words.
// Returns how many there are. Out of line: the blocks of most nodes end empty. One string at
// a time by the whole warp, (9,3), 20 letters, n = 2, m = 600 took 1830 us (now 640).
template <int kQuads, bool kPre>
__device__ __noinline__ unsigned int ss_store_all(unsigned long long *raw, unsigned long long *raw_count,
                                                  unsigned long long raw_cap, unsigned long long x, int l, int b,
                                                  int sigma, int a, int k, uint32_t pos, const uint32_t *map, int lane)
{
    unsigned long long c;
    unsigned int mine = 0;
    for (int q = 0; q < 4 * kQuads; ++q) {
        const int word = 4 * (32 * (q >> 2) + lane) + (q & 3);
        if (map[word] != 0u && ss_word<kPre>(x, b, sigma, word, a, k, pos, c))
            mine += __popc(map[word]);
    }
    unsigned int upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(kFull, upto, o);
        upto += lane >= o ? y : 0u;
    }
    const unsigned int found = __shfl_sync(kFull, upto, 31);
    unsigned long long slot = 0;
    if (lane == 0 && found != 0u)
        slot = atomicAdd(raw_count, (unsigned long long)found);
    slot = __shfl_sync(kFull, slot, 0) + upto - mine;
    const int sh = b * ((int)(pos >> (8 * (k - 1))) & 31);
    for (int q = 0; mine != 0u && q < 4 * kQuads; ++q) {
        const int word = 4 * (32 * (q >> 2) + lane) + (q & 3);
        uint32_t v = map[word];
        if (v == 0u || !ss_word<kPre>(x, b, sigma, word, a, k, pos, c))
            continue;
        c &= ~(((1ull << b) - 1ull) << sh);
        for (; v != 0u; v &= v - 1u)
            ss_store(raw, raw_cap, slot++, c | ((unsigned long long)(__ffs(v) - 1) << sh), l, b);
    }
    __syncwarp();
    return found;
}

// The block of node P whose first letter is `a` (kPre), or the whole node.
template <int kQuads, bool kPre>
__device__ __forceinline__ void ss_block(const SigmaParams &p, const SsSeed &S, uint32_t P, int k, const int (&pos)[4],
                                         int a, const uint32_t *list, const int (&from)[kSsListSeqs + 1], int listed,
                                         uint32_t *map, int lane, SsCount &ct)
{
    const int b = S.b, sigma = S.sigma;
    const uint32_t all = sigma == 32 ? kFull : (1u << sigma) - 1u;
    const uint32_t first = all & ~(1u << ss_letter(S.x, b, pos[k - 1]));
    // the lane's words, four at a time: (32 j + lane) 4 + 0..3; those beyond the
    // node's are never marked
    uint4 *map4 = reinterpret_cast<uint4 *>(map) + lane;
    uint4 cur[kQuads];
#pragma unroll
    for (int j = 0; j < kQuads; ++j)
        cur[j] = make_uint4(first, first, first, first);
    uint32_t left = 0;
    int si = 0;
    while (si < S.seqs) {
        if (si < listed) {
            for (int e0 = from[si]; e0 < from[si + 1]; e0 += 32)
                ss_mark<kPre>(e0 + lane < from[si + 1] ? list[e0 + lane] : kSsNoRow, a, k, sigma, all, map, lane);
        } else {
            const int i = S.order[si], e1 = S.off[i + 1];
            for (int e0 = S.off[i]; e0 < e1; e0 += 32) {
                uint32_t v = kSsNoRow;
                if (e0 + lane < e1) {
                    ct.reduce++;
                    v = ss_entry(S, e0 + lane, P, k, pos);
                }
                ss_mark<kPre>(v, a, k, sigma, all, map, lane);
            }
        }
        __syncwarp();
        left = 0;
#pragma unroll
        for (int j = 0; j < kQuads; ++j) {
            const uint4 m = map4[32 * j];
            map4[32 * j] = make_uint4(0u, 0u, 0u, 0u);
            cur[j] = make_uint4(cur[j].x & m.x, cur[j].y & m.y, cur[j].z & m.z, cur[j].w & m.w);
            left |= cur[j].x | cur[j].y | cur[j].z | cur[j].w;
        }
        __syncwarp();
        const int lanes = __popc(__ballot_sync(kFull, left != 0u));
        ++si;
        if (lanes == 0)
            return;
        if (lanes <= kSsLookupLanes)
            break;
    }
    uint32_t who = __ballot_sync(kFull, left != 0u);
    if (!who)
        return;
    // what is left, lane by lane
    unsigned long long ones = 0;
    for (int q = 0; q < S.l; ++q)
        ones |= 1ull << (b * q);
#pragma unroll
    for (int j = 0; j < kQuads; ++j)
        map4[32 * j] = cur[j];
    __syncwarp();
    if (si == S.seqs) {
        const uint32_t at = (uint32_t)(pos[0] | (pos[1] << 8) | (pos[2] << 16) | (pos[3] << 24));
        const unsigned int found = ss_store_all<kQuads, kPre>(p.raw, p.raw_count, p.raw_cap, S.x, S.l, b, sigma, a, k, at,
                                                              map, lane);
        if (lane == 0)
            ct.leaves += found;
        who = 0u;
    }
    while (who) {
        const int holder = __ffs(who) - 1;
        who &= who - 1u;
        // lane k takes the holder's k-th word
        uint32_t v = lane < 4 * kQuads ? map[4 * (32 * (lane >> 2) + holder) + (lane & 3)] : 0u;
        uint32_t have = __ballot_sync(kFull, v != 0u);
        while (have) {
            const int src = __ffs(have) - 1;
            const uint32_t vs = __shfl_sync(kFull, v, src);
            if (lane == src)
                v &= v - 1u;
            have = __ballot_sync(kFull, v != 0u);
            // the string: x with the tuple's letters on P
            unsigned long long c = S.x;
            bool ok = true;
            int rest = 4 * (32 * (src >> 2) + holder) + (src & 3);
            for (int j = k - 1; j >= 0; --j) {
                int x = __ffs(vs) - 1;
                if (kPre && j == 0) {
                    x = a;
                } else if (j < k - 1) {
                    x = rest % sigma;
                    rest /= sigma;
                }
                ok = ok && x != ss_letter(S.x, b, pos[j]);   // a word of one of x's own letters is not the node's
                c = (c & ~(((1ull << b) - 1ull) << (b * pos[j]))) | ((unsigned long long)x << (b * pos[j]));
            }
            if (!ok)
                continue;
            if (lane == 0)
                ct.leaves++;
            for (int sj = si; ok && sj < S.seqs; ++sj) {
                const int i = S.order[sj];
                bool found = false;
                for (int e0 = S.off[i]; !found && e0 < S.off[i + 1]; e0 += 32) {
                    const int e = e0 + lane;
                    bool hit = false;
                    if (e < S.off[i + 1]) {
                        ct.verify++;
                        hit = ss_distance(S.L[e], c, b, ones) <= S.d;
                    }
                    found = __any_sync(kFull, hit);
                }
                ok = found;
            }
            if (ok && lane == 0)
                ss_put(p, c, S.l, b);
        }
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kQuads; ++j)
        map4[32 * j] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
}

// The node P by a warp; map: its words, clear on entry and on return; list:
// room for kSsListCap entries.
template <int kQuads>
__device__ __forceinline__ void ss_node(const SigmaParams &p, const SsSeed &S, uint32_t P, uint32_t *map, uint32_t *list,
                                        int lane, SsCount &ct)
{
    const int k = __popc(P);
    if (lane == 0)
        ct.nodes++;
    for (int si = 0; si < S.seqs; ++si)
        if (!ss_row_passes(S, S.order[si], P, lane, ct)) {
            if (lane == 0)
                ct.pruned++;
            return;
        }
    if (k == 0) {   // the seed itself; the bound was its exact distance
        if (lane == 0) {
            ct.leaves++;
            ss_put(p, S.x, S.l, S.b);
        }
        return;
    }
    int pos[4] = {0, 0, 0, 0};
    {
        uint32_t M = P;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < k) {
                pos[j] = __ffs(M) - 1;
                M &= M - 1u;
            }
    }
    // a node whose letters are taken in turn lists its rows for the first sequences
    int from[kSsListSeqs + 1] = {0, 0, 0, 0, 0};
    int listed = 0;
    if (k < 4) {
        ss_block<kQuads, false>(p, S, P, k, pos, 0, list, from, 0, map, lane, ct);
        return;
    }
    bool room = true;
#pragma unroll
    for (int si = 0; si < kSsListSeqs; ++si) {
        int n = from[si];
        if (si < S.seqs && room) {
            const int i = S.order[si], e1 = S.off[i + 1];
            for (int e0 = S.off[i]; e0 < e1; e0 += 32) {
                uint32_t v = kSsNoRow;
                if (e0 + lane < e1) {
                    ct.reduce++;
                    v = ss_entry(S, e0 + lane, P, k, pos);
                }
                const uint32_t bal = __ballot_sync(kFull, v != kSsNoRow);
                const int at = n + __popc(bal & ((1u << lane) - 1u));
                if (v != kSsNoRow && at < kSsListCap)
                    list[at] = v;
                n += __popc(bal);
            }
            room = n <= kSsListCap;
            if (room)
                listed = si + 1;
        }
        from[si + 1] = room ? n : from[si];
    }
    __syncwarp();
    const int xa = ss_letter(S.x, S.b, pos[0]);
    for (int a = 0; a < S.sigma; ++a)
        if (a != xa)
            ss_block<kQuads, true>(p, S, P, k, pos, a, list, from, listed, map, lane, ct);
}

// The r-th position subset by size, then colexicographically (as sg_unrank).
__device__ __forceinline__ uint32_t ss_unrank(int r, int l)
{
    int k = 0;
    while (r >= (int)g_ss_binom[l][k])
        r -= (int)g_ss_binom[l][k++];
    uint32_t P = 0;
    int c = l - 1;
    for (int j = k; j >= 1; --j) {
        while ((int)g_ss_binom[c][j] > r)
            --c;
        P |= 1u << c;
        r -= (int)g_ss_binom[c][j];
        --c;
    }
    return P;
}

// Persistent CTAs take items (seed, part); a part is every parts-th node of the
// seed. Rows: a pass over every window sets a mask bit for those within 2d (kept
// in shared memory where it has room) and counts them per sequence, a second
// stores their masks and letters, in shared memory where they fit.
//
// kSplit: several warps share the windows of a sequence, in groups of 128. With few
// sequences a seed's rows would otherwise wait for one warp each: (9,1), 20 letters,
// n = 2, m = 8000, whole solves, 760 us without and 235 us with it. A kernel of its
// own, as the shares' bookkeeping costs the others 2 % ((9,4), n = 20, 2.55 and 2.60 ms).
template <int kQuads, int kMinBlocks, bool kSplit>
__global__ void __launch_bounds__(kSsThreads, kMinBlocks) sigma_sieve_kernel(SigmaParams p, SigmaSieve q)
{
    extern __shared__ __align__(16) unsigned char ss_raw[];
    __shared__ int s_cnt[kNMax], s_off[kNMax + 1], s_order[kNMax], s_part[kNMax];
    __shared__ int s_item, s_next, s_skip;
    __shared__ unsigned long long s_ct[kSgCntNum];
    // the warps' maps, their lists (the masks of a seed's rows while these are collected), the rows
    uint32_t *map = reinterpret_cast<uint32_t *>(ss_raw);
    uint32_t *lists = map + q.map_words, *s_mask = lists;
    unsigned long long *smem_L = reinterpret_cast<unsigned long long *>(lists + kSsWarps * kSsListCap);
    uint32_t *smem_D = reinterpret_cast<uint32_t *>(smem_L + p.smem_rows);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c = tid; c < kSgCntNum; c += kSsThreads)
        s_ct[c] = 0;
    for (int w = tid; w < q.map_words; w += kSsThreads)
        map[w] = 0u;
    const int NWm = (p.W + 31) / 32;
    const bool masks = p.n * NWm <= kSsMaskWords;
    const size_t NW = (size_t)p.n * p.W;
    // warps that share a sequence, and the first group of 32 windows of the u-th of them
    auto shares = [&] { return kSplit ? q.shares : 1; };
    auto first_of = [&](int u) { return kSplit ? min(4 * (u * ((NWm + 3) / 4) / q.shares), NWm) : u * NWm; };
    if (tid == 0)
        s_cnt[0] = 0;
    for (;;) {
        if (tid == 0)
            s_item = (int)atomicAdd(p.head, 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= p.nseeds * q.parts)
            break;
        const int seed = item / q.parts, part = item - seed * q.parts;
        uint32_t x[kSigMaxPlanes];
#pragma unroll
        for (int g = 0; g < kSigMaxPlanes; ++g)
            x[g] = g < p.b ? p.planes[(size_t)g * NW + seed] : 0u;   // a window of s_1
        auto differs = [&](int i, int w) {
            const uint32_t *at = p.planes + (i * p.W + w);   // n W < 2^22
            uint32_t mm = 0;
#pragma unroll
            for (int g = 0; g < kSigMaxPlanes; ++g)
                if (g < p.b)
                    mm |= x[g] ^ __ldg(at + g * NW);
            return mm;
        };
        for (int t = warp; t < (p.n - 1) * shares(); t += kSsWarps) {
            const int i = 1 + t / shares(), part_of = t % shares();
            const int c1 = first_of(part_of + 1);
            int cnt = 0;
            for (int c0 = first_of(part_of); c0 < c1; c0 += 4) {
                // four groups of 32 windows, their loads in flight together
                uint32_t mm[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    mm[u] = differs(i, min(32 * (c0 + u) + lane, p.W - 1));
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t bal = __ballot_sync(kFull, 32 * (c0 + u) + lane < p.W && __popc(mm[u]) <= 2 * p.d);
                    if (masks && lane == 0 && c0 + u < NWm)
                        s_mask[i * NWm + c0 + u] = bal;
                    cnt += __popc(bal);
                }
            }
            if (lane == 0)
                (shares() > 1 ? s_part[t] : s_cnt[i]) = cnt;
        }
        __syncthreads();
        if (shares() > 1) {
            if (tid >= 1 && tid < p.n) {
                int cnt = 0;
                for (int u = 0; u < shares(); ++u)
                    cnt += s_part[(tid - 1) * shares() + u];
                s_cnt[tid] = cnt;
            }
            __syncthreads();
        }
        if (tid == 0) {
            int o = 0, empty = 0;
            for (int i = 0; i < p.n; ++i) {
                s_off[i] = o;
                o += s_cnt[i];
                empty += i != 0 && s_cnt[i] == 0;
            }
            s_off[p.n] = o;
            s_skip = empty > 0;
            s_next = part;
            if (part == 0) {
                s_ct[kSgSeeds] += 1;
                s_ct[kSgSeedsInfeasible] += empty > 0;
                s_ct[kSgCmpRows] += (unsigned long long)(p.n - 1) * p.W;
            }
        }
        if (tid >= 1 && tid < p.n) {
            int rank = 0;
            for (int j = 1; j < p.n; ++j)
                rank += s_cnt[j] < s_cnt[tid] || (s_cnt[j] == s_cnt[tid] && j < tid);
            s_order[rank] = tid;
        }
        __syncthreads();
        if (!s_skip) {
            SsSeed S;
            const bool joint = (p.b + 1) * p.l <= 64;   // a row's mask above its letters
            uint32_t *D = joint ? nullptr : smem_D;
            unsigned long long *L = smem_L;
            if (s_off[p.n] > p.smem_rows) {
                uint32_t *base = p.scratch + (size_t)blockIdx.x * (1 + p.b) * p.scratch_rows;
                L = reinterpret_cast<unsigned long long *>(base);   // scratch_rows is even
                D = joint ? nullptr : base + 2 * (size_t)p.scratch_rows;
            }
            for (int t = warp; t < (p.n - 1) * shares(); t += kSsWarps) {
                const int i = 1 + t / shares(), part_of = t % shares();
                const int c1 = first_of(part_of + 1);
                int e = s_off[i];
                for (int u = 0; u < part_of; ++u)
                    e += s_part[t - part_of + u];
#pragma unroll 2
                for (int c = first_of(part_of); c < c1; ++c) {
                    const int w = 32 * c + lane;
                    uint32_t bal;
                    if (masks)
                        bal = s_mask[i * NWm + c];
                    else
                        bal = __ballot_sync(kFull, w < p.W && __popc(differs(i, min(w, p.W - 1))) <= 2 * p.d);
                    if ((bal >> lane) & 1u) {
                        const int at = e + __popc(bal & ((1u << lane) - 1u));
                        const uint32_t mm = differs(i, w);
                        const unsigned long long let = __ldg(q.letters + (size_t)i * p.W + w);
                        L[at] = joint ? let | ((unsigned long long)mm << (p.b * p.l)) : let;
                        if (!joint)
                            D[at] = mm;
                    }
                    e += __popc(bal);
                }
            }
            __syncthreads();
            S.D = D;
            S.L = L;
            S.off = s_off;
            S.order = s_order;
            S.seqs = p.n - 1;
            S.l = p.l;
            S.d = p.d;
            S.b = p.b;
            S.sigma = p.sigma;
            S.x = __ldg(q.letters + seed);
            SsCount ct{};
            for (;;) {
                int r = 0;
                if (lane == 0)
                    r = atomicAdd(&s_next, q.parts);
                r = __shfl_sync(kFull, r, 0);
                if (r >= (int)p.nodes)
                    break;
                ss_node<kQuads>(p, S, ss_unrank(r, p.l), map + warp * q.warp_words, lists + warp * kSsListCap, lane, ct);
            }
            unsigned int red = ct.reduce, ver = ct.verify;
            red = __reduce_add_sync(kFull, red);
            ver = __reduce_add_sync(kFull, ver);
            if (lane == 0) {
                atomicAdd(&s_ct[kSgNodes], (unsigned long long)ct.nodes);
                atomicAdd(&s_ct[kSgNodesPruned], (unsigned long long)ct.pruned);
                atomicAdd(&s_ct[kSgChecks], (unsigned long long)ct.leaves);
                atomicAdd(&s_ct[kSgLeaves], (unsigned long long)ct.leaves);
                atomicAdd(&s_ct[kSgCmpReduce], (unsigned long long)red);
                atomicAdd(&s_ct[kSgCmpVerify], (unsigned long long)ver);
            }
        }
        __syncthreads();   // rows, offsets and s_item are rewritten for the next item
    }
    __syncthreads();
    if (tid < kSgCntNum)
        atomicAdd(&p.counters[tid], s_ct[tid]);
}

using SsKernel = void (*)(SigmaParams, SigmaSieve);

// 16 words a lane hold up to 22 letters (484 words); 32 letters need 32.
SsKernel ss_kernel(const SigmaSieve &q)
{
    if (q.shares > 1)
        return q.warp_words <= 512 ? sigma_sieve_kernel<4, 3, true> : sigma_sieve_kernel<8, 2, true>;
    return q.warp_words <= 512 ? sigma_sieve_kernel<4, 3, false> : sigma_sieve_kernel<8, 2, false>;
}

}  // namespace

bool sigma_sieve_plan(int n, int l, int d, int b, int sigma, SigmaSieve *q)
{
    if (n < 2 || d > 4 || b < 2 || b * l > 64)
        return false;
    q->warp_words = sigma * sigma <= 512 ? 512 : 1024;
    q->map_words = kSsWarps * q->warp_words;
    q->row_bytes = (b + 1) * l <= 64 ? 8 : 12;
    q->shares = std::max(1, kSsWarps / (n - 1));
    return true;
}

size_t sigma_sieve_smem(const SigmaSieve &q, int rows)
{
    return 4 * ((size_t)q.map_words + kSsWarps * kSsListCap) + (size_t)q.row_bytes * rows;
}

cudaError_t sigma_sieve_init()
{
    uint32_t binom[33][5] = {};
    for (int a = 0; a <= 32; ++a)
        for (int k = 0; k <= 4; ++k)
            binom[a][k] = k == 0 ? 1u : a == 0 ? 0u : binom[a - 1][k - 1] + binom[a - 1][k];
    cudaError_t e = cudaMemcpyToSymbol(g_ss_binom, binom, sizeof binom);
    for (const SsKernel f : {(SsKernel)sigma_sieve_kernel<4, 3, false>, (SsKernel)sigma_sieve_kernel<8, 2, false>,
                             (SsKernel)sigma_sieve_kernel<4, 3, true>, (SsKernel)sigma_sieve_kernel<8, 2, true>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute((const void *)f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSsSmemMax);
    return e;
}

cudaError_t sigma_sieve_occupancy(const SigmaSieve &q, int rows, int *blocks_per_sm)
{
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, ss_kernel(q), kSsThreads,
                                                         sigma_sieve_smem(q, rows));
}

cudaError_t launch_sigma_sieve(const SigmaParams &p, const SigmaSieve &q, int blocks, cudaStream_t st)
{
    ss_kernel(q)<<<blocks, kSsThreads, sigma_sieve_smem(q, p.smem_rows), st>>>(p, q);
    return cudaGetLastError();
}

}  // namespace pms
