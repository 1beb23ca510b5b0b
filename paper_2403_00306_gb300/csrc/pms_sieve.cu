// pms_sieve.cu -- the sieve form of the DNA search (sm_103a).
//
// The tree search (pms_kernels.cu) decides one candidate set per seed and
// pays where windows within d of a candidate are common: few tree nodes fail,
// and most leaves are verified one by one. The sieve turns the question round.
// The 4^l strings are a bit map; a window w of sequence i marks its ball
// B(w, d); the motifs are the strings that every sequence marks (Definitions
// 3-5 with q = n), or that at least q sequences mark (the quorum form). Its
// cost depends on n, W and |B(l, d)| only, not on how many strings survive.
//
// The map is cut into blocks that live in shared memory and registers. A
// string is split into a prefix of A letters, kMid middle letters and three
// last letters. A block is one prefix; its words are the 4^kMid middles; the
// 64 bits of a word are the last three letters. A window at prefix distance t
// has r = d - t changes left in the block, so it touches exactly the words of
// the ball B(mid(w), r) around its own middle, and in the word at middle
// distance t2 the bits of the ball of radius r - t2 around its own last three
// letters (a 64-bit table entry). On the outermost shell, t2 = r, that is a
// single bit. Balls of 2-bit letters are invariant under exclusive-or, so a
// word's index is the window's index XOR an entry of one table of changes,
// the same for every window.
//
// A warp (or a team of warps) owns a block: 4^kMid words of marks in shared
// memory, and the strings still alive (or the hit counters of the quorum form)
// in registers, a fixed share per thread. Marks are shared-memory atomic ORs
// without a result: nothing waits for them, so windows need no order, and one
// takes as long for 32 random banks as for 32 different ones (2.8 to 3.7
// cycles a warp operation on GB300, against 3.8 and 6.2 for a load-or-store).
// A window with two or more changes left is worked on by the whole warp, a lane
// per word (the changes of a group of 32 lie in different banks: the index is a
// linear permutation of the middle's planes chosen for that, and exclusive-or
// with a window's index keeps banks distinct). Windows with one change left
// touch 16 words: they are listed, and 32 of them worked on at once, a lane each.
//
// What bounds it: instruction issue and the marks. One GB300, n = 20:
// (13,4) m = 1000 (20 sequences x 988 windows x 1024 blocks, 20.7 words marked
// per window and block) 316 us, 190 M warp instructions, 16.8 M mark operations,
// 2.3 instructions a cycle; 64 registers and 25 warps per SM. The same search in
// the tree form takes 7409 us. Load-or-stores in place of the atomics, a warp
// per block: 587 us, 325 M instructions.
#include "pms_sieve.cuh"

#include <algorithm>
#include <cstring>

namespace pms {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kSvWarps = 8;
constexpr int kSvThreads = kSvWarps * 32;
constexpr int kSvMaxShell = 5;             // changed middle letters, at most kMid
// Lanes that still hold strings, at or below which a block looks its strings up
// in the remaining sequences instead of marking them.
constexpr int kSvLookupLanes = 2;

// Index change of one changed letter: number e = 1 + 3 p + v changes position
// p by v + 1 (exclusive-or of the 2-bit code); e = 0 is no change.
template <int kMid>
__host__ __device__ constexpr uint32_t sv_single(int e)
{
    return e == 0 ? 0u
                  : sv_index<kMid>((uint32_t)((((e - 1) % 3 + 1) >> 1) & 1) << ((e - 1) / 3),
                                   (uint32_t)(((e - 1) % 3 + 1) & 1) << ((e - 1) / 3));
}

// Changes of t >= 2 middle letters, in groups of 32 with different banks where
// that is possible; the last group repeats changes in its unused places.
constexpr int kSvGroupsMax = 40;
struct SvTable {
    uint16_t change[kSvGroupsMax * 32];    // byte offsets of word indexes
    int first[kSvMaxShell + 2];            // first group of the shell of t changes; [t + 1] is its end
};

__device__ SvTable g_sv_table[3];          // kMid = 3, 4, 5
// bits of the ball of radius v around last letters s, one half of the 64: [v][s][half]
__device__ uint32_t g_sv_ball[4][64][2];

// groups of the shell of two changes: the table entries a lane keeps in registers
template <int kMid>
__host__ __device__ constexpr int sv_groups2()
{
    return kMid == 5 ? 3 : kMid == 4 ? 2 : 1;
}

// Shared memory of a CTA besides its teams' marks.
struct SvSmem {
    uint32_t ball[4 * 64 * 2];             // g_sv_ball
    uint16_t change[kSvGroupsMax * 32];
    uint32_t list[kSvWarps][64];           // windows with one change left, until 32 are there
    int first[kSvMaxShell + 2];
    long long item[kSvWarps];              // per team
    int alive[kSvWarps][3];                // per team: lanes that hold strings alive after sequence i, at i % 3
};

template <int kMid>
struct SvMarks {
    static constexpr int kWords = 1 << (2 * kMid);
    static constexpr uint32_t kHalf = 4 * kWords;      // bytes of the marks of one half of the words
    static constexpr uint32_t kBytes = 2 * kHalf;
};

__device__ __forceinline__ void red_or(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// The distance of two strings as sieve words (see sieve_word), prefix included.
template <int kMid>
__device__ __forceinline__ int sv_distance(uint32_t a, uint32_t b)
{
    constexpr uint32_t kMask = (1u << kMid) - 1u;
    const uint32_t x = a ^ b;
    const uint32_t hi = (x >> (6 + kMid)) & kMask;
    const uint32_t lo = ((x >> 6) & kMask) ^ sv_fold<kMid>(hi);
    const uint32_t mid = hi | lo, suf = (x | (x >> 3)) & 7u;
    const uint32_t pre = kMid == 5   ? ((x >> 24) | (x >> 16)) & 0xffu
                         : kMid == 4 ? ((x >> 23) | (x >> 14)) & 0x1ffu
                                     : ((x >> 22) | (x >> 12)) & 0x3ffu;
    return __popc((pre << 16) | (mid << 8) | suf);
}

// The windows of one sequence mark the block's words; the team's warps take
// 32 windows in turn. marks: shared address, aligned to kBytes, so that a word
// address is an exclusive-or away from another.
template <int kMid, int kShare>
__device__ __forceinline__ void sv_mark(const uint32_t *__restrict__ win, int W, int d, uint32_t block, uint32_t marks,
                                        uint32_t *list, const SvSmem &sm, uint32_t slot0,
                                        const uint32_t (&d2)[sv_groups2<kMid>()], int g, int lane)
{
    using M = SvMarks<kMid>;
    constexpr int kPre = sv_pre<kMid>();
    constexpr uint32_t kCode = (1u << (6 + 2 * kMid)) - 1u;
    constexpr uint32_t kPreMask = ((1u << kPre) - 1u) << (6 + 2 * kMid);
    constexpr uint32_t kWordMask = (4u << (2 * kMid)) - 4u;
    constexpr int kStep = 32 * kShare;
    const bool edge = (lane & 15) < 1 + 3 * kMid;
    const uint32_t *ball2 = sm.ball + (2 - ((lane & 15) != 0)) * 128 + (lane >> 4);
    const uint32_t lt = (1u << lane) - 1u;
    int n1 = 0;
    int w0 = 32 * g;
    uint32_t next = w0 + lane < W ? __ldg(win + w0 + lane) : 0u;
    for (; w0 < W; w0 += kStep) {
        const uint32_t x = next ^ block;
        const bool in = w0 + lane < W;
        if (w0 + kStep + lane < W)
            next = __ldg(win + w0 + kStep + lane);
        const int r = in ? d - __popc((x | (x >> kPre)) & kPreMask) : -1;
        const uint32_t code = x & kCode;
        // the window's own word: byte address in the half that holds its last three letters
        const uint32_t own = marks ^ ((code >> 6) << 2) ^ ((code & 32u) ? M::kHalf : 0u);
        if (r == 0)
            red_or(own, 1u << (code & 31u));
        const uint32_t one = __ballot_sync(kFull, r == 1);
        if (r == 1)
            list[n1 + __popc(one & lt)] = code;
        n1 += __popc(one);
        uint32_t wide = __ballot_sync(kFull, r >= 2);
        const uint32_t packed = ((code >> 4) & kWordMask) | ((code & 63u) << 16) | ((uint32_t)r << 24);
        while (wide) {
            const int src = __ffs(wide) - 1;
            wide &= wide - 1u;
            const uint32_t v = __shfl_sync(kFull, packed, src);
            const uint32_t wa = marks ^ (v & kWordMask);   // the word in the lower half's marks
            const uint32_t suf = (v >> 16) & 63u;
            const uint32_t wh = wa ^ ((v & (32u << 16)) ? M::kHalf : 0u);
            const uint32_t bit = 1u << (suf & 31u);
            if ((v >> 24) == 2u) {
                // no change and one change: half a warp per half of the words
                // (slot0: the lane's change and half; ball2: its table column)
                if (edge)
                    red_or(wa ^ slot0, ball2[2 * suf]);
#pragma unroll
                for (int t = 0; t < sv_groups2<kMid>(); ++t)
                    red_or(wh ^ d2[t], bit);
            } else {
                const int rr = (int)(v >> 24);
                const uint32_t *ball = sm.ball + 2 * suf;
                if (edge)
                    red_or(wa ^ slot0, ball[min(rr - ((lane & 15) != 0), 3) * 128 + (lane >> 4)]);
                const int tmax = min(rr, kMid);
                const uint16_t *ch = sm.change + lane;
                for (int t = 2; t <= tmax; ++t) {
                    const int q1 = sm.first[t + 1];
                    if (t == rr) {
#pragma unroll 3
                        for (int q = sm.first[t]; q < q1; ++q)
                            red_or(wh ^ ch[q * 32], bit);
                    } else {
                        const int rad = min(rr - t, 3);
                        const uint32_t b0 = ball[rad * 128], b1 = ball[rad * 128 + 1];
#pragma unroll 3
                        for (int q = sm.first[t]; q < q1; ++q) {
                            const uint32_t wc = wa ^ ch[q * 32];
                            red_or(wc, b0);
                            red_or(wc ^ M::kHalf, b1);
                        }
                    }
                }
            }
        }
        // windows with one change left, a lane each once 32 (or the last) are listed
        const bool last = w0 + kStep >= W;
        while (n1 >= 32 || (last && n1 > 0)) {
            __syncwarp();
            const uint32_t v = list[lane], up = list[32 + lane];
            if (lane < n1) {
                const uint32_t suf = v & 63u;
                const uint32_t wa = marks ^ ((v & ~63u) >> 4);
                red_or(wa, sm.ball[128 + 2 * suf]);
                red_or(wa ^ M::kHalf, sm.ball[128 + 2 * suf + 1]);
                const uint32_t wh = wa ^ ((suf & 32u) ? M::kHalf : 0u);
                const uint32_t bit = 1u << (suf & 31u);
#pragma unroll
                for (int e = 1; e <= 3 * kMid; ++e)
                    red_or(wh ^ (sv_single<kMid>(e) << 2), bit);
            }
            __syncwarp();
            list[lane] = up;
            n1 = max(0, n1 - 32);
            __syncwarp();
        }
    }
}

// Does a window of the sequence lie within d of the string c? Warp-uniform.
template <int kMid>
__device__ __forceinline__ bool sv_occurs(const uint32_t *__restrict__ win, int W, int d, uint32_t c, int lane)
{
    for (int w0 = 0; w0 < W; w0 += 32) {
        const int w = w0 + lane;
        const bool hit = w < W && sv_distance<kMid>(__ldg(win + w), c) <= d;
        if (__any_sync(kFull, hit))
            return true;
    }
    return false;
}

// Up to 32 strings, one per lane (`has`): those that occur in the sequences
// first..n-1 too are appended to the raw codes, once per window of the seed
// sequences within d, as the tree form finds them.
template <int kMid>
__device__ __noinline__ void sv_emit(const InstDev *__restrict__ inst, uint64_t *raw, uint32_t *raw_count, uint32_t *flags,
                                     const uint32_t *__restrict__ win, bool has, uint32_t c, int first, int lane)
{
    const int n = inst->n, W = inst->W, d = inst->d, l = inst->l;
    uint32_t todo = __ballot_sync(kFull, has);
    int copies = 0;
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const uint32_t cc = __shfl_sync(kFull, c, src);
        bool ok = true;
        for (int i = first; ok && i < n; ++i)
            ok = sv_occurs<kMid>(win + (size_t)i * W, W, d, cc, lane);
        if (!ok)
            continue;
        int k = 0;
        const int nw = inst->nseed * W;   // the windows of s_1..s_{n-q+1} are contiguous
        for (int w = lane; w < nw; w += 32)
            k += sv_distance<kMid>(__ldg(win + w), cc) <= d;
        k = __reduce_add_sync(kFull, k);
        if (lane == src)
            copies = k;
    }
    int incl = copies;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o)
            incl += y;
    }
    const int all = __shfl_sync(kFull, incl, 31);
    if (all == 0)
        return;
    uint32_t base = 0;
    if (lane == 0)
        base = atomicAdd(raw_count, (uint32_t)all);
    base = __shfl_sync(kFull, base, 0) + (uint32_t)(incl - copies);
    if (copies > 0) {
        constexpr uint32_t kMask = (1u << kMid) - 1u;
        constexpr int kPre = sv_pre<kMid>();
        const int A = l - kMid - kSvSuf;
        const uint32_t mh = (c >> (6 + kMid)) & kMask, ml = ((c >> 6) & kMask) ^ sv_fold<kMid>(mh);
        const uint32_t pre_l = (c >> (6 + 2 * kMid)) & ((1u << kPre) - 1u), pre_h = c >> (6 + 2 * kMid + kPre);
        const uint32_t h = pre_h | (mh << A) | (((c >> 3) & 7u) << (A + kMid));
        const uint32_t lo = pre_l | (ml << A) | ((c & 7u) << (A + kMid));
        uint64_t key = 0;
        for (int k = 0; k < l; ++k)
            key = (key << 2) | (uint64_t)((((h >> k) & 1u) << 1) | ((lo >> k) & 1u));
        for (int k = 0; k < copies; ++k) {
            const uint32_t pos = base + (uint32_t)k;
            if (pos < inst->raw_cap)
                raw[inst->raw_off + pos] = key;
            else
                atomicOr(flags, kFlagOverflow);
        }
    }
}

// The string of bit `bit` of mark word `at` ([half][word]) of a block.
template <int kMid>
__device__ __forceinline__ uint32_t sv_string(uint32_t block, int at, int bit)
{
    constexpr int kWords = SvMarks<kMid>::kWords;
    return block | ((uint32_t)(at & (kWords - 1)) << 6) | ((uint32_t)(at / kWords) << 5) | (uint32_t)bit;
}

// Bits of piece k whose counter exceeds v: the planes compared with v, low plane first.
template <int kPlanes, int kPieces>
__device__ __forceinline__ uint32_t sv_above(const uint32_t (&cnt)[kPlanes][kPieces], int k, int v)
{
    uint32_t gt = 0u;
#pragma unroll
    for (int s = 0; s < kPlanes; ++s)
        gt = ((v >> s) & 1) ? gt & cnt[s][k] : gt | cnt[s][k];
    return gt;
}

template <int kShare>
__device__ __forceinline__ void team_sync(int team)
{
    if (kShare == 1)
        __syncwarp();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(kShare * 32) : "memory");
}

// Copies the tables to shared memory (the caller synchronises) and places the
// CTA's mark buffers, aligned to their size, before them.
template <int kMid>
__device__ __forceinline__ SvSmem &sv_setup(unsigned char *raw, int buffers, unsigned char *&marks_ptr, uint32_t &marks0)
{
    using M = SvMarks<kMid>;
    const uint32_t raw0 = (uint32_t)__cvta_generic_to_shared(raw);
    marks0 = (raw0 + M::kBytes - 1) & ~(M::kBytes - 1);
    marks_ptr = raw + (marks0 - raw0);
    SvSmem &sm = *reinterpret_cast<SvSmem *>(marks_ptr + buffers * M::kBytes);
    const SvTable &tab = g_sv_table[kMid - 3];
    for (int i = threadIdx.x; i < kSvGroupsMax * 32; i += kSvThreads)
        sm.change[i] = tab.change[i];
    for (int i = threadIdx.x; i < 4 * 64 * 2; i += kSvThreads)
        sm.ball[i] = (&g_sv_ball[0][0][0])[i];
    if (threadIdx.x < kSvMaxShell + 2)
        sm.first[threadIdx.x] = tab.first[threadIdx.x];
    return sm;
}

// A lane's change of at most one letter (half a warp per half of the words) and of two.
template <int kMid>
__device__ __forceinline__ void sv_lane_changes(const SvSmem &sm, int lane, uint32_t &slot0,
                                                uint32_t (&d2)[sv_groups2<kMid>()])
{
    slot0 = 0;
#pragma unroll
    for (int e = 0; e <= 3 * kMid; ++e)
        slot0 = (lane & 15) == e ? sv_single<kMid>(e) << 2 : slot0;
    slot0 ^= lane >= 16 ? SvMarks<kMid>::kHalf : 0u;
#pragma unroll
    for (int t = 0; t < sv_groups2<kMid>(); ++t)
        d2[t] = sm.change[(sm.first[2] + t) * 32 + lane];
}

// Item it of a launch: its instance and block.
template <int kMid>
struct SvBlock {
    int I;
    InstDev in;
    uint32_t block;        // the block's prefix, as in a window's word
    const uint32_t *win;   // the instance's window words
    __device__ __forceinline__ SvBlock(const SieveParams &p, long long it)
    {
        constexpr int kPre = sv_pre<kMid>();
        int lo = 0, hi = p.nseg - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (p.seg[mid].work_lo <= it)
                lo = mid;
            else
                hi = mid - 1;
        }
        I = p.seg[lo].inst;
        in = p.inst[I];
        const uint32_t b = (uint32_t)(it - p.seg[lo].work_lo);   // the prefix letters' planes, hi above lo
        const int A = in.l - kMid - kSvSuf;
        block = ((b & ((1u << A) - 1u)) << (6 + 2 * kMid)) | ((b >> A) << (6 + 2 * kMid + kPre));
        win = reinterpret_cast<const uint32_t *>(p.planes + in.plane_off);
    }
};

// Buffers of marks in a CTA: one per team of one warp, else two.
template <int kShare>
__host__ __device__ constexpr int sv_buffers()
{
    return kShare == 1 ? kSvWarps : 2 * kSvWarps / kShare;
}

// Items are blocks; a team of kShare warps of a CTA takes one at a time and
// its warps split the windows of every sequence. kPlanes = 0: q = n, a thread
// keeps its share of the strings alive in registers, and a block ends once
// none is alive or the last few have been looked up window by window.
// kPlanes > 0: the quorum form, kPlanes bit-sliced hit counters (kShare = 1).
template <int kMid, int kPlanes, int kShare, int kMinBlocks>
__global__ void __launch_bounds__(kSvThreads, kMinBlocks) sieve_kernel(SieveParams p)
{
    extern __shared__ __align__(16) unsigned char sv_raw[];
    using M = SvMarks<kMid>;
    constexpr int kPieces = 2 * M::kWords / (32 * kShare);   // mark words of a thread
    constexpr int kVec = kPieces % 4 == 0 ? 4 : 1;           // of them in one access
    constexpr int kPre = sv_pre<kMid>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int team = warp / kShare, g = warp % kShare;
    unsigned char *marks_ptr;
    uint32_t marks0;
    SvSmem &sm = sv_setup<kMid>(sv_raw, sv_buffers<kShare>(), marks_ptr, marks0);
    if (threadIdx.x < 3 * kSvWarps)
        (&sm.alive[0][0])[threadIdx.x] = 0;
    // a team of several warps marks sequence i in buffer i % 2, so that one
    // barrier a sequence is enough
    constexpr int kBuf = kShare > 1 ? 2 : 1;
    const uint32_t marks = marks0 + team * kBuf * M::kBytes;
    uint32_t *mw = reinterpret_cast<uint32_t *>(marks_ptr + team * kBuf * M::kBytes);
    // piece k of this thread: mark word sv_at(k)
    const int tid = g * 32 + lane;
    auto at_of = [&](int k) { return (k / kVec) * (32 * kShare * kVec) + tid * kVec + k % kVec; };
#pragma unroll
    for (int k = 0; k < kPieces * kBuf; ++k)
        mw[at_of(k)] = 0u;
    __syncthreads();
    uint32_t slot0, d2[sv_groups2<kMid>()];
    sv_lane_changes<kMid>(sm, lane, slot0, d2);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the packed windows are complete and visible
    for (;;) {
        long long it = 0;
        if (g == 0) {
            if (lane == 0)
                it = (long long)atomicAdd(p.head, 1ull);
            it = __shfl_sync(kFull, it, 0);
        }
        if (kShare > 1) {
            if (g == 0 && lane == 0)
                sm.item[team] = it;
            team_sync<kShare>(team);
            it = sm.item[team];
            team_sync<kShare>(team);
        }
        if (it >= p.total)
            break;
        SvBlock<kMid> blk(p, it);
        const InstDev &in = blk.in;
        const uint32_t block = blk.block;
        const uint32_t *win = blk.win;
        // what is left of the block's strings goes back to its marks
        uint32_t left = 0;   // != 0: this thread holds some
        int i = 0;
        if constexpr (kPlanes == 0) {
            uint32_t cur[kPieces];
#pragma unroll
            for (int k = 0; k < kPieces; ++k)
                cur[k] = kFull;
            while (i < in.n) {
                const uint32_t buf = kShare > 1 ? (uint32_t)(i & 1) : 0u;
                uint32_t *mb = mw + buf * (2 * M::kWords);
                sv_mark<kMid, kShare>(win + (size_t)i * in.W, in.W, in.d, block, marks + buf * M::kBytes, sm.list[warp],
                                      sm, slot0, d2, g, lane);
                team_sync<kShare>(team);
                int lanes = 32 * kShare;
                if (kShare > 1 && i > 0) {   // after the sequence before
                    lanes = *(volatile int *)&sm.alive[team][(i - 1) % 3];
                    if (g == 0 && lane == 0)
                        *(volatile int *)&sm.alive[team][(i + 1) % 3] = 0;
                }
                left = 0;
#pragma unroll
                for (int k = 0; k < kPieces; k += kVec) {
                    if constexpr (kVec == 4) {
                        uint4 *m4 = reinterpret_cast<uint4 *>(mb + at_of(k));
                        const uint4 m = *m4;
                        *m4 = make_uint4(0u, 0u, 0u, 0u);
                        cur[k] &= m.x;
                        cur[k + 1] &= m.y;
                        cur[k + 2] &= m.z;
                        cur[k + 3] &= m.w;
                        left |= cur[k] | cur[k + 1] | cur[k + 2] | cur[k + 3];
                    } else {
                        cur[k] &= mb[at_of(k)];
                        mb[at_of(k)] = 0u;
                        left |= cur[k];
                    }
                }
                const int mine = __popc(__ballot_sync(kFull, left != 0u));
                if (kShare > 1) {
                    if (lane == 0)
                        atomicAdd(&sm.alive[team][i % 3], mine);
                } else {
                    __syncwarp();
                    lanes = mine;
                }
                ++i;
                if (lanes <= kSvLookupLanes)
                    break;
            }
            if (kShare > 1) {   // the counters are zero again before the next block
                team_sync<kShare>(team);
                if (g == 0 && lane < 3)
                    sm.alive[team][lane] = 0;
            }
            if (__any_sync(kFull, left != 0u)) {
#pragma unroll
                for (int k = 0; k < kPieces; ++k)
                    mw[at_of(k)] = cur[k];
            }
        } else {
            uint32_t cnt[kPlanes > 0 ? kPlanes : 1][kPieces];
#pragma unroll
            for (int s = 0; s < kPlanes; ++s)
#pragma unroll
                for (int k = 0; k < kPieces; ++k)
                    cnt[s][k] = 0u;
            while (i < in.n) {
                sv_mark<kMid, 1>(win + (size_t)i * in.W, in.W, in.d, block, marks, sm.list[warp], sm, slot0, d2, 0, lane);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < kPieces; ++k) {
                    uint32_t m = mw[at_of(k)];
                    mw[at_of(k)] = 0u;
#pragma unroll
                    for (int s = 0; s < kPlanes; ++s) {
                        const uint32_t c = cnt[s][k];
                        cnt[s][k] = c ^ m;
                        m &= c;
                    }
                }
                __syncwarp();
                ++i;
                // a string needs q - (n - i) hits by now; the block ends once none has them
                const int need1 = in.q - (in.n - i) - 1;
                if (need1 < 0)
                    continue;
                left = 0;
#pragma unroll
                for (int k = 0; k < kPieces; ++k)
                    left |= sv_above<kPlanes, kPieces>(cnt, k, need1);
                if (!__any_sync(kFull, left != 0u))
                    break;
            }
            if (__any_sync(kFull, left != 0u)) {
#pragma unroll
                for (int k = 0; k < kPieces; ++k)
                    mw[at_of(k)] = sv_above<kPlanes, kPieces>(cnt, k, in.q - 1);
            }
        }
        // the strings of a warp's threads, the pieces of one thread at a time
        uint32_t holders = __ballot_sync(kFull, left != 0u);
        if (holders) {
            __syncwarp();
            while (holders) {
                const int who = __ffs(holders) - 1;
                holders &= holders - 1u;
                for (int k0 = 0; k0 < kPieces; k0 += 32) {
                    const int k = k0 + lane;
                    const int at = ((k / kVec) * (32 * kShare) + g * 32 + who) * kVec + k % kVec;
                    uint32_t v = k < kPieces ? mw[at] : 0u;
                    while (__any_sync(kFull, v != 0u)) {
                        const bool has = v != 0u;
                        const int bit = has ? __ffs(v) - 1 : 0;
                        v &= v - 1u;
                        sv_emit<kMid>(p.inst + blk.I, p.raw, p.raw_count + blk.I, p.flags + blk.I, win, has,
                                      sv_string<kMid>(block, at, bit), i, lane);
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kPieces; ++k)
                mw[at_of(k)] = 0u;
            __syncwarp();
        }
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

// The form for few blocks, q = n: a CTA per block, whose warps take the
// sequences i = warp, warp + kSvWarps, ... with marks of their own, so that
// they meet only once, to intersect what they are left with.
template <int kMid, int kMinBlocks>
__global__ void __launch_bounds__(kSvThreads, kMinBlocks) sieve_split_kernel(SieveParams p)
{
    extern __shared__ __align__(16) unsigned char sv_raw[];
    using M = SvMarks<kMid>;
    constexpr int kPieces = 2 * M::kWords / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *marks_ptr;
    uint32_t marks0;
    SvSmem &sm = sv_setup<kMid>(sv_raw, kSvWarps, marks_ptr, marks0);
    const uint32_t marks = marks0 + warp * M::kBytes;
    uint32_t *all = reinterpret_cast<uint32_t *>(marks_ptr);
    uint32_t *mw = all + warp * (2 * M::kWords);
    int *dead = &sm.alive[0][0];
#pragma unroll
    for (int k = 0; k < kPieces; ++k)
        mw[k * 32 + lane] = 0u;
    __syncthreads();
    uint32_t slot0, d2[sv_groups2<kMid>()];
    sv_lane_changes<kMid>(sm, lane, slot0, d2);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the packed windows are complete and visible
    for (long long it = blockIdx.x; it < p.total; it += gridDim.x) {
        if (threadIdx.x == 0)
            *dead = 0;
        __syncthreads();
        SvBlock<kMid> blk(p, it);
        const InstDev &in = blk.in;
        uint32_t cur[kPieces];
#pragma unroll
        for (int k = 0; k < kPieces; ++k)
            cur[k] = kFull;
        for (int i = warp; i < in.n && !*(volatile int *)dead; i += kSvWarps) {
            sv_mark<kMid, 1>(blk.win + (size_t)i * in.W, in.W, in.d, blk.block, marks, sm.list[warp], sm, slot0, d2, 0,
                             lane);
            __syncwarp();
            uint32_t left = 0;
#pragma unroll
            for (int k = 0; k < kPieces; ++k) {
                cur[k] &= mw[k * 32 + lane];
                mw[k * 32 + lane] = 0u;
                left |= cur[k];
            }
            __syncwarp();
            if (!__any_sync(kFull, left != 0u) && lane == 0)
                *(volatile int *)dead = 1;
        }
#pragma unroll
        for (int k = 0; k < kPieces; ++k)
            mw[k * 32 + lane] = cur[k];
        __syncthreads();
        if (!*(volatile int *)dead) {
            // mark word at: warp at / 32 % kSvWarps
            for (int at = warp * 32 + lane; at < 2 * M::kWords; at += kSvThreads) {
                uint32_t v = kFull;
#pragma unroll
                for (int t = 0; t < kSvWarps; ++t)
                    v &= all[t * (2 * M::kWords) + at];
                while (__any_sync(kFull, v != 0u)) {
                    const bool has = v != 0u;
                    const int bit = has ? __ffs(v) - 1 : 0;
                    v &= v - 1u;
                    sv_emit<kMid>(p.inst + blk.I, p.raw, p.raw_count + blk.I, p.flags + blk.I, blk.win, has,
                                  sv_string<kMid>(blk.block, at, bit), in.n, lane);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPieces; ++k)
            mw[k * 32 + lane] = 0u;
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

template <int kMid>
void fill_table(SvTable &t)
{
    std::memset(&t, 0, sizeof t);
    int group = 0;
    t.first[0] = t.first[1] = 0;
    for (int shell = 2; shell <= kSvMaxShell; ++shell) {
        t.first[shell] = group;
        if (shell <= kMid) {
            // every change of `shell` middle letters, by bank
            uint16_t bank[32][256];
            int nb[32] = {}, total = 0;
            for (uint32_t hi = 0; hi < (1u << kMid); ++hi)
                for (uint32_t lo = 0; lo < (1u << kMid); ++lo) {
                    int c = 0;
                    for (int p = 0; p < kMid; ++p)
                        c += (((hi | lo) >> p) & 1u) ? 1 : 0;
                    if (c != shell)
                        continue;
                    const uint32_t x = sv_index<kMid>(hi, lo);
                    bank[x & 31u][nb[x & 31u]++] = (uint16_t)x;
                    ++total;
                }
            // groups of 32, the fullest banks first, a bank again only when all are used
            const int groups = (total + 31) / 32;
            for (int q = 0; q < groups; ++q) {
                int used = 0;
                const int room = std::min(32, total - 32 * q);
                while (used < room) {
                    bool taken[32] = {};
                    for (; used < room; ++used) {
                        int best = -1;
                        for (int k = 0; k < 32; ++k)
                            if (!taken[k] && nb[k] > 0 && (best < 0 || nb[k] > nb[best]))
                                best = k;
                        if (best < 0)
                            break;
                        taken[best] = true;
                        t.change[(group + q) * 32 + used] = (uint16_t)(bank[best][--nb[best]] << 2);
                    }
                }
                for (; used < 32; ++used)   // OR is idempotent: a place may repeat another
                    t.change[(group + q) * 32 + used] = t.change[(group + q) * 32 + used - room];
            }
            group += groups;
        }
        t.first[shell + 1] = group;
    }
}

cudaError_t launch_kernel(void (*kernel)(SieveParams), const SieveParams &p, long long blocks, size_t smem, cudaStream_t st)
{
    const cudaError_t e =
        cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = dependent_launch(attr, (int)blocks, kSvThreads, smem, st);
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <int kMid, int kPlanes, int kShare, int kMinBlocks>
cudaError_t launch(const SieveParams &p, int sms, cudaStream_t st)
{
    const size_t smem = (sv_buffers<kShare>() + 1) * (size_t)SvMarks<kMid>::kBytes + sizeof(SvSmem);
    const long long teams = kSvWarps / kShare;
    return launch_kernel(sieve_kernel<kMid, kPlanes, kShare, kMinBlocks>, p,
                         std::min<long long>((long long)sms * kMinBlocks, (p.total + teams - 1) / teams), smem, st);
}

template <int kMid, int kMinBlocks>
cudaError_t launch_split(const SieveParams &p, int sms, cudaStream_t st)
{
    const size_t smem = (kSvWarps + 1) * (size_t)SvMarks<kMid>::kBytes + sizeof(SvSmem);
    return launch_kernel(sieve_split_kernel<kMid, kMinBlocks>, p,
                         std::min<long long>((long long)sms * kMinBlocks, p.total), smem, st);
}

}  // namespace

cudaError_t sieve_init_tables()
{
    static SvTable t[3];
    fill_table<3>(t[0]);
    fill_table<4>(t[1]);
    fill_table<5>(t[2]);
    uint32_t ball[4][64][2] = {};
    for (int v = 0; v < 4; ++v)
        for (int s = 0; s < 64; ++s)
            for (int u = 0; u < 64; ++u) {
                const int x = s ^ u, diff = (x | (x >> 3)) & 7;
                if ((diff & 1) + ((diff >> 1) & 1) + (diff >> 2) <= v)
                    ball[v][s][u >> 5] |= 1u << (u & 31);
            }
    const cudaError_t e = cudaMemcpyToSymbol(g_sv_table, t, sizeof t);
    if (e != cudaSuccess)
        return e;
    return cudaMemcpyToSymbol(g_sv_ball, ball, sizeof ball);
}

cudaError_t launch_sieve(const SieveParams &p, int mid, int planes, int share, int sms, cudaStream_t st)
{
    if (planes > 0)
        return mid == 4 ? launch<4, 5, 1, 2>(p, sms, st) : launch<3, 7, 1, 3>(p, sms, st);
    if (mid == 5)
        return share == 1 ? launch<5, 0, 1, 2>(p, sms, st) : launch<5, 0, 8, 4>(p, sms, st);
    if (mid == 4)
        return share == 1 ? launch<4, 0, 1, 4>(p, sms, st) : launch_split<4, 5>(p, sms, st);
    return share == 1 ? launch<3, 0, 1, 5>(p, sms, st) : launch_split<3, 5>(p, sms, st);
}

}  // namespace pms
