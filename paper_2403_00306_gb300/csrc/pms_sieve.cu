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
// The map is cut into blocks (of 2^12 to 2^18 strings) that live in shared memory and registers. A
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
// What bounds it. Where windows mark many words of a block: instruction issue
// and the marks; (13,4), n = 20, m = 1000 (20 sequences x 988 windows x 1024
// blocks, 20.7 words marked per window and block) 316 us, 190 M warp
// instructions, 17 M mark operations, 2.3 instructions a cycle. The tree form
// takes 7409 us there; load-or-stores in place of the atomics, a warp per
// block, took 587 us and 325 M instructions. Where they mark few: the 50 or so
// instructions that sort 32 windows by the changes they have left; larger
// blocks pay them less often. (17,5), n = 20, m = 1200: 5 middle letters and a
// warp per block 5429 us, 6 letters and a CTA per block 4326 us (now 4102; the tree
// 7747 us); (15,4) 449 and 392 us (668 us). With six letters 32 KB of marks
// serve a CTA of eight warps, and what is lost is their wait for the slowest
// (5.8 of 14 cycles per instruction), so few windows favour the warp per block.
#include "pms_sieve.cuh"

#include <algorithm>
#include <cstring>

namespace pms {

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kSvWarps = 8;
constexpr int kSvThreads = kSvWarps * 32;
constexpr int kSvMaxShell = 6;             // changed middle letters, at most kMid
// Threads that still hold strings, at or below which a block looks its strings up
// in the remaining sequences instead of marking them. A CTA that shares six
// letters waits for the warp with the most strings. Solves, us, at 0, 2, 6 and 12:
// (17,5), n = 20, m = 1200 4303, 4102, 4214 and 4627 (4326 before the look-ups had
// four loads in flight); five letters at 2, 12 and
// 24: (13,4), n = 20, m = 600 162, 150 and 152; a warp per block, 256 mixed
// instances, 2 and 5: 24.4 and 24.0 ms.
template <int kMid, int kShare>
constexpr int kSvLookupLanes = kMid == 6 ? 2 : kShare == 1 ? 5 : 12;

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
constexpr int kSvGroupsMax = 132;
template <int kMid>
__host__ __device__ constexpr int sv_groups()
{
    return kMid == 6 ? 129 : kMid == 5 ? 33 : kMid == 4 ? 10 : 2;
}
struct SvTable {
    uint16_t change[kSvGroupsMax * 32];    // byte offsets of word indexes
    int first[kSvMaxShell + 2];            // first group of the shell of t changes; [t + 1] is its end
};

__device__ SvTable g_sv_table[4];          // kMid = 3, 4, 5, 6
// bits of the ball of radius v around last letters s, one half of the 64: [v][s][half]
__device__ uint32_t g_sv_ball[4][64][2];

// changes of t of kMid letters
template <int kMid>
__host__ __device__ constexpr int sv_shell(int t)
{
    int c = 1;
    for (int i = 0; i < t; ++i)
        c = c * 3 * (kMid - i) / (i + 1);
    return c;
}

// groups of the shell of two changes: the table entries a lane keeps in registers
template <int kMid>
__host__ __device__ constexpr int sv_groups2()
{
    return kMid == 6 ? 5 : kMid == 5 ? 3 : kMid == 4 ? 2 : 1;
}

// Shared memory of a CTA besides its marks, which it precedes: the marks are
// aligned to one half of a buffer.
template <int kMid, int kWarps = kSvWarps>
struct SvSmem {
    uint32_t ball[4 * 64 * 2];             // g_sv_ball
    uint16_t change[sv_groups<kMid>() * 32];
    uint32_t list[kWarps][64];             // windows with one change left, until 32 are there
    int first[kSvMaxShell + 2];
    long long item;                        // of the CTA, when its warps share a block
    int alive[3];                          // lanes that hold strings alive after sequence i, at i % 3
};

template <int kMid>
struct SvMarks {
    static constexpr int kWords = 1 << (2 * kMid);
    static constexpr uint32_t kHalf = 4 * kWords;      // bytes of the marks of one half of the words
    static constexpr uint32_t kBytes = 2 * kHalf;
};

// Marks: an atomic OR on shared memory without a result. No memory clobber: the
// barriers around a sequence's marks order them against the plain accesses.
__device__ __forceinline__ void red_or(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(addr), "r"(v));
}
__device__ __forceinline__ void red_or_if(bool on, uint32_t addr, uint32_t v)
{
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p red.shared.or.b32 [%1], %2; }" ::"r"((uint32_t)on), "r"(addr),
                 "r"(v));
}

// What a pass over windows does with the words of their balls: mark them, or
// count the strings that are marked already.
struct SvMark {
    static constexpr bool kCount = false;
    __device__ __forceinline__ void operator()(uint32_t addr, uint32_t bits, bool = true) { red_or(addr, bits); }
    __device__ __forceinline__ void if_(bool on, uint32_t addr, uint32_t bits) { red_or_if(on, addr, bits); }
};
struct SvCount {
    static constexpr bool kCount = true;
    unsigned long long found = 0;
    // once: not a lane that repeats another's change
    __device__ __forceinline__ void operator()(uint32_t addr, uint32_t bits, bool once = true)
    {
        uint32_t v;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
        found += once ? (uint32_t)__popc(v & bits) : 0u;
    }
    __device__ __forceinline__ void if_(bool on, uint32_t addr, uint32_t bits)
    {
        if (on)
            (*this)(addr, bits);
    }
};

// The distance of two strings as sieve words (see sieve_word), prefix included.
template <int kMid>
__device__ __forceinline__ int sv_distance(uint2 a, uint2 b)
{
    const uint32_t x = a.x ^ b.x, y = a.y ^ b.y;
    const uint32_t mid = (x >> (6 + kMid)) | sv_lo<kMid>(x >> 6), suf = (x | (x >> 3)) & 7u;
    return __popc(((y | (y >> 16)) & 0xffffu) | (mid << 16) | (suf << 22));
}

// What a lane changes in the words of a window, as offsets from the window's
// own word: at most one letter (with up to 16 such changes, half a warp for
// each half of the words) and two letters. The lanes left over repeat a change.
template <int kMid>
struct SvLane {
    static constexpr bool kBoth = 1 + 3 * kMid <= 16;
    uint32_t single;                    // and, with kBoth, the half
    uint32_t pair[sv_groups2<kMid>()];
    int t;                              // letters `single` changes
    int half;                           // the half of the words `single` works on first
    template <class Smem>
    __device__ __forceinline__ SvLane(const Smem &sm, int lane)
    {
        const int e0 = kBoth ? (lane & 15) : lane < 1 + 3 * kMid ? lane : lane - 16;
        half = kBoth ? lane >> 4 : 0;
        single = 0;
#pragma unroll
        for (int e = 1; e <= 3 * kMid; ++e)
            single = e0 == e ? sv_single<kMid>(e) << 2 : single;
        t = e0 >= 1 && e0 <= 3 * kMid ? 1 : 0;
        single += (uint32_t)half * SvMarks<kMid>::kHalf;
#pragma unroll
        for (int k = 0; k < sv_groups2<kMid>(); ++k)
            pair[k] = sm.change[(sm.first[2] + k) * 32 + lane];
    }
};

// The windows of one sequence mark the block's words (or count the strings
// marked there, see SvCount); kShare warps take 32 windows in turn. marks: shared address, aligned to kHalf, so that within a
// half a word address is an exclusive-or away from another. prefix: the
// block's, as in a window's word.
template <int kMid, int kShare, class Op, class Smem>
__device__ __forceinline__ void sv_pass(Op &op, const uint2 *__restrict__ win, int W, int d, uint32_t prefix,
                                        uint32_t marks, uint32_t *list, const Smem &sm, const SvLane<kMid> &my, int g,
                                        int lane)
{
    using M = SvMarks<kMid>;
    constexpr int kStep = 32 * kShare;
    constexpr bool kBoth = SvLane<kMid>::kBoth;
    const uint32_t lt = (1u << lane) - 1u;
    const bool once1 = (kBoth ? lane & 15 : lane) <= 3 * kMid;   // `single` is no other lane's
    const uint32_t single0 = marks + my.single;
    const uint32_t *ball2 = sm.ball + (2 - my.t) * 128 + my.half;   // radius 2 or 1 of the last letters
    int n1 = 0;
    int w0 = 32 * g;
    uint2 next = w0 + lane < W ? __ldg(win + w0 + lane) : make_uint2(0u, 0u);
    for (; w0 < W; w0 += kStep) {
        const uint32_t y = next.y ^ prefix, code = next.x;
        const bool in = w0 + lane < W;
        if (w0 + kStep + lane < W)
            next = __ldg(win + w0 + kStep + lane);
        const int r = in ? d - __popc((y | (y >> 16)) & 0xffffu) : -1;
        // word offset in a half's marks; the last three letters choose half and bit
        const uint32_t off = (code >> 6) << 2;
        op.if_(r == 0, (marks + (code & 32u) * (M::kHalf / 32u)) ^ off, 1u << (code & 31u));
        const uint32_t one = __ballot_sync(kFull, r == 1);
        if (r == 1)
            list[n1 + __popc(one & lt)] = code;
        n1 += __popc(one);
        uint32_t two = __ballot_sync(kFull, r == 2);
        const uint32_t packed = off | (code << 16);   // bits 16..21: the last letters; above them what is not used
        while (two) {
            const uint32_t v = __shfl_sync(kFull, packed, __ffs(two) - 1);
            two &= two - 1u;
            const uint32_t o = v & 0xffffu, suf = (v >> 16) & 63u;
            op(single0 ^ o, ball2[2 * suf], once1);
            if (!kBoth)
                op((single0 + M::kHalf) ^ o, ball2[2 * suf + 1], once1);
            const uint32_t wh = (marks + (suf >> 5) * M::kHalf) ^ o, bit = 1u << (suf & 31u);
#pragma unroll
            for (int t = 0; t < sv_groups2<kMid>(); ++t)
                op(wh ^ my.pair[t], bit, 32 * t + lane < sv_shell<kMid>(2));
        }
        uint32_t more = __ballot_sync(kFull, r > 2);
        while (more) {
            const int src = __ffs(more) - 1;
            more &= more - 1u;
            const uint32_t v = __shfl_sync(kFull, packed, src);
            const int rr = __shfl_sync(kFull, r, src);
            const uint32_t o = v & 0xffffu, suf = (v >> 16) & 63u;
            const uint32_t *ball = sm.ball + 2 * suf;
            op(single0 ^ o, ball[min(rr - my.t, 3) * 128 + my.half], once1);
            if (!kBoth)
                op((single0 + M::kHalf) ^ o, ball[min(rr - my.t, 3) * 128 + 1], once1);
            const int tmax = min(rr, kMid);
            const uint16_t *ch = sm.change + lane;
            for (int t = 2; t <= tmax; ++t) {
                const int q1 = sm.first[t + 1];
                // groups of the shell without repeated changes
                const int whole = Op::kCount ? sm.first[t] + ((sv_shell<kMid>(t) - lane + 31) >> 5) : q1;
                if (t == rr) {
                    const uint32_t wh = (marks + (suf >> 5) * M::kHalf) ^ o, bit = 1u << (suf & 31u);
#pragma unroll 4
                    for (int q = sm.first[t]; q < q1; ++q)
                        op(wh ^ ch[q * 32], bit, q < whole);
                } else {
                    const uint32_t wa = marks ^ o;
                    const int rad = min(rr - t, 3);
                    const uint32_t b0 = ball[rad * 128], b1 = ball[rad * 128 + 1];
#pragma unroll 4
                    for (int q = sm.first[t]; q < q1; ++q) {
                        const uint32_t wc = wa ^ ch[q * 32];
                        op(wc, b0, q < whole);
                        op(wc + M::kHalf, b1, q < whole);
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
                const uint32_t suf = v & 63u, o = (v >> 6) << 2;
                op(marks ^ o, sm.ball[128 + 2 * suf]);
                op((marks + M::kHalf) ^ o, sm.ball[128 + 2 * suf + 1]);
                const uint32_t wh = (marks + (suf >> 5) * M::kHalf) ^ o, bit = 1u << (suf & 31u);
#pragma unroll
                for (int e = 1; e <= 3 * kMid; ++e)
                    op(wh ^ (sv_single<kMid>(e) << 2), bit);
            }
            __syncwarp();
            list[lane] = up;
            n1 = max(0, n1 - 32);
            __syncwarp();
        }
    }
}

template <int kMid, int kShare, class Smem>
__device__ __forceinline__ void sv_mark(const uint2 *__restrict__ win, int W, int d, uint32_t prefix, uint32_t marks,
                                        uint32_t *list, const Smem &sm, const SvLane<kMid> &my, int g, int lane)
{
    SvMark op;
    sv_pass<kMid, kShare>(op, win, W, d, prefix, marks, list, sm, my, g, lane);
}

// Strings of a block from which their windows in the seed sequences are counted
// by a pass over those windows, as marking does, instead of string by string: a
// string's own look at the windows costs about 8 instructions per 32 of them, the
// pass 60 to 300 whatever the number of strings. Whole solves, us, without and
// with it: (9,2), n = 20, m = 1200 105 and 63; (11,3), n = 20, m = 1200 147 and
// 82; 256 mixed instances, some of 600 k motifs, 34.6 and 25.1 ms.
constexpr int kSvCountFrom = 32;

// Where an instance's motifs go.
struct SvOut {
    uint64_t *raw;
    uint32_t *raw_count, *key_count, *buckets, *flags;
};

// Adds to an instance's raw count (one lane). The count has 32 bits, and dense
// answers over long sequences exceed them: the flag says so from then on.
__device__ __forceinline__ void sv_raw_add(SvOut out, unsigned long long v)
{
    const uint32_t add = (uint32_t)min(v, 0xffffffffull);
    const uint32_t was = atomicAdd(out.raw_count, add);
    if (add != v || was + add < was)
        atomicOr(out.flags, kFlagRawBeyond);
}

// Adds the windows of win[0..W) within d of each string marked in the block,
// summed over the strings, to the raw count; kShare warps take part.
template <int kMid, int kShare, class Smem>
__device__ __noinline__ void sv_count(const uint2 *__restrict__ win, int W, int d, uint32_t prefix, uint32_t marks,
                                      uint32_t *list, const Smem &sm, SvOut out, int g, int lane)
{
    SvCount op;
    const SvLane<kMid> my(sm, lane);
    sv_pass<kMid, kShare>(op, win, W, d, prefix, marks, list, sm, my, g, lane);
    unsigned long long all = op.found;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        all += __shfl_xor_sync(kFull, all, o);
    if (lane == 0 && all != 0ull)
        sv_raw_add(out, all);
}

// Does a window of the sequence lie within d of the string c? Warp-uniform.
template <int kMid>
__device__ __forceinline__ bool sv_occurs(const uint2 *__restrict__ win, int W, int d, uint2 c, int lane)
{
    for (int w0 = 0; w0 < W; w0 += 128) {   // four loads in flight
        bool hit = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int w = min(w0 + 32 * k + lane, W - 1);   // the last window again
            hit |= sv_distance<kMid>(__ldg(win + w), c) <= d;
        }
        if (__any_sync(kFull, hit))
            return true;
    }
    return false;
}

// Up to 32 strings, one per lane (`has`): those that occur in the sequences
// first..n-1 too are appended to the keys. The raw count grows by the windows of
// the seed sequences within d of them, as often as the tree form finds them
// (unless these are counted already).
template <int kMid>
__device__ __noinline__ void sv_emit(const InstDev *__restrict__ inst, SvOut out, const uint2 *__restrict__ win,
                                     bool has, uint2 c, int first, bool counted, int lane)
{
    const int n = inst->n, W = inst->W, d = inst->d, l = inst->l;
    uint32_t todo = __ballot_sync(kFull, has);
    int copies = 0;
    if (counted && first >= n) {
        copies = has ? 1 : 0;
        todo = 0u;
    }
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const uint2 cc = make_uint2(__shfl_sync(kFull, c.x, src), __shfl_sync(kFull, c.y, src));
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
    const uint32_t found = __ballot_sync(kFull, copies > 0);
    if (found == 0u)
        return;
    const int all = __reduce_add_sync(kFull, copies);
    uint32_t base = 0;
    if (lane == 0) {
        if (!counted)
            sv_raw_add(out, (unsigned long long)all);
        base = atomicAdd(out.key_count, (uint32_t)__popc(found));
    }
    base = __shfl_sync(kFull, base, 0) + (uint32_t)__popc(found & ((1u << lane) - 1u));
    if (copies > 0 && base < inst->raw_cap) {   // beyond it the raw count tells
        const int A = l - kMid - kSvSuf;
        const uint32_t mid = c.x >> 6;
        const uint32_t h = (c.y >> 16) | ((mid >> kMid) << A) | (((c.x >> 3) & 7u) << (A + kMid));
        const uint32_t lo = (c.y & 0xffffu) | (sv_lo<kMid>(mid) << A) | ((c.x & 7u) << (A + kMid));
        uint64_t key = 0;
        for (int k = 0; k < l; ++k)
            key = (key << 2) | (uint64_t)((((h >> k) & 1u) << 1) | ((lo >> k) & 1u));
        out.raw[inst->raw_off + base] = key;
        if (inst->buckets >= 0)
            atomicAdd(out.buckets + inst->buckets + bucket_of(key, l), 1u);
    }
}

__device__ __forceinline__ SvOut out_of(const SieveParams &p, int I)
{
    return SvOut{p.raw, p.raw_count + I, p.key_count + I, p.buckets, p.flags + I};
}

// The string of bit `bit` of mark word `at` ([half][word]) of a block.
template <int kMid>
__device__ __forceinline__ uint2 sv_string(uint32_t prefix, int at, int bit)
{
    constexpr int kWords = SvMarks<kMid>::kWords;
    return make_uint2(((uint32_t)(at & (kWords - 1)) << 6) | ((uint32_t)(at / kWords) << 5) | (uint32_t)bit, prefix);
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
__device__ __forceinline__ void share_sync()
{
    if (kShare == 1)
        __syncwarp();
    else
        __syncthreads();
}

// Shared memory: the tables, then the buffers of marks at the next multiple of
// kHalf of the shared address space, in which dynamic shared memory starts
// after what the system reserves (`reserved`: 1 KB).
template <int kMid, int kWarps = kSvWarps>
__host__ __device__ constexpr uint32_t sv_marks_at(uint32_t reserved)
{
    using M = SvMarks<kMid>;
    return (reserved + (uint32_t)sizeof(SvSmem<kMid, kWarps>) + M::kHalf - 1) / M::kHalf * M::kHalf;
}
template <int kMid, int kWarps = kSvWarps>
size_t sv_smem_bytes(int reserved, int buffers)
{
    return sv_marks_at<kMid, kWarps>((uint32_t)reserved) - reserved + (size_t)buffers * SvMarks<kMid>::kBytes;
}

// Copies the tables to shared memory and clears the marks; returns the shared
// address of the first buffer.
template <int kMid, int kWarps = kSvWarps>
__device__ __forceinline__ uint32_t sv_setup(unsigned char *raw, int buffers)
{
    using M = SvMarks<kMid>;
    SvSmem<kMid, kWarps> &sm = *reinterpret_cast<SvSmem<kMid, kWarps> *>(raw);
    const uint32_t raw0 = (uint32_t)__cvta_generic_to_shared(raw);
    const uint32_t marks0 = sv_marks_at<kMid, kWarps>(raw0);
    const SvTable &tab = g_sv_table[kMid - 3];
    for (int i = threadIdx.x; i < sv_groups<kMid>() * 32; i += 32 * kWarps)
        sm.change[i] = tab.change[i];
    for (int i = threadIdx.x; i < 4 * 64 * 2; i += 32 * kWarps)
        sm.ball[i] = (&g_sv_ball[0][0][0])[i];
    if (threadIdx.x < kSvMaxShell + 2)
        sm.first[threadIdx.x] = tab.first[threadIdx.x];
    if (threadIdx.x < 3)
        sm.alive[threadIdx.x] = 0;
    uint4 *m4 = reinterpret_cast<uint4 *>(raw + (marks0 - raw0));
    for (int i = threadIdx.x; i < buffers * (int)(M::kBytes / 16); i += 32 * kWarps)
        m4[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    return marks0;
}

// Item it of a launch: its instance and block.
struct SvBlock {
    int I;
    InstDev in;
    uint32_t prefix;     // the block's, as in a window's word
    const uint2 *win;    // the instance's windows
    __device__ __forceinline__ SvBlock(const SieveParams &p, long long it, int mid_letters)
    {
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
        // the prefix letters' planes, hi above lo
        const uint32_t b = (uint32_t)(it - p.seg[lo].work_lo + p.seg[lo].block_lo);
        const int A = in.l - mid_letters - kSvSuf;
        prefix = (b & ((1u << A) - 1u)) | ((b >> A) << 16);
        win = p.planes + in.plane_off;
    }
};

// Buffers of marks in a CTA: one per warp that works alone. A CTA that shares
// a block marks sequence i in buffer i % 2, so that one barrier a sequence is
// enough, where two buffers leave room for as many CTAs.
template <int kMid, int kPlanes, int kShare>
__host__ __device__ constexpr int sv_buffers()
{
    return kShare == 1 ? kSvWarps : (kPlanes == 0 && kMid <= 5 ? 2 : 1);
}

// Items are blocks; kShare warps take one at a time (1, or all of the CTA) and
// split the windows of every sequence. kPlanes = 0: q = n, a thread keeps its
// share of the strings alive in registers, and a block ends once none is alive
// or the last few have been looked up window by window. kPlanes > 0: the quorum
// form, kPlanes bit-sliced hit counters.
template <int kMid, int kPlanes, int kShare, int kMinBlocks>
__global__ void __launch_bounds__(kSvThreads, kMinBlocks) sieve_kernel(SieveParams p)
{
    extern __shared__ __align__(16) unsigned char sv_raw[];
    using M = SvMarks<kMid>;
    static_assert(kShare == 1 || kShare == kSvWarps, "a warp or the CTA works on a block");
    constexpr int kPieces = 2 * M::kWords / (32 * kShare);   // mark words of a thread
    constexpr int kVec = kPieces % 4 == 0 ? 4 : 1;           // of them in one access
    constexpr int kAll = sv_buffers<kMid, kPlanes, kShare>();
    constexpr int kBuf = kShare == 1 ? 1 : kAll;             // buffers a block uses
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = kShare == 1 ? 0 : warp, own = kShare == 1 ? warp : 0;
    SvSmem<kMid> &sm = *reinterpret_cast<SvSmem<kMid> *>(sv_raw);
    const uint32_t marks0 = sv_setup<kMid>(sv_raw, kAll);
    const uint32_t marks = marks0 + own * M::kBytes;
    uint32_t *mw =
        reinterpret_cast<uint32_t *>(sv_raw + (marks - (uint32_t)__cvta_generic_to_shared(sv_raw)));
    // piece k of this thread
    const int tid = g * 32 + lane;
    auto at_of = [&](int k) { return (k / kVec) * (32 * kShare * kVec) + tid * kVec + k % kVec; };
    const SvLane<kMid> my(sm, lane);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the packed windows are complete and visible
    for (;;) {
        long long it = 0;
        if (g == 0) {
            if (lane == 0)
                it = (long long)atomicAdd(p.head, 1ull);
            it = __shfl_sync(kFull, it, 0);
        }
        if (kShare > 1) {
            __syncthreads();   // the last item has been read, the counters of its block too
            if (threadIdx.x == 0)
                sm.item = it;
            if (threadIdx.x < 3)
                sm.alive[threadIdx.x] = 0;
            __syncthreads();
            it = sm.item;
        }
        if (it >= p.total)
            break;
        SvBlock blk(p, it, kMid);
        const InstDev &in = blk.in;
        // what is left of the block's strings goes back to its marks
        uint32_t left = 0;   // != 0: this thread holds some
        int i = 0, holding = 0;   // holding: threads that do, of the block
        if constexpr (kPlanes == 0) {
            uint32_t cur[kPieces];
#pragma unroll
            for (int k = 0; k < kPieces; ++k)
                cur[k] = kFull;
            while (i < in.n) {
                const uint32_t buf = kBuf > 1 ? (uint32_t)(i & 1) : 0u;
                uint32_t *mb = mw + buf * (2 * M::kWords);
                sv_mark<kMid, kShare>(blk.win + (size_t)i * in.W, in.W, in.d, blk.prefix, marks + buf * M::kBytes,
                                      sm.list[warp], sm, my, g, lane);
                share_sync<kShare>();
                int lanes = 32 * kShare;
                if (kBuf > 1 && i > 0) {   // after the sequence before
                    lanes = *(volatile int *)&sm.alive[(i - 1) % 3];
                    if (threadIdx.x == 0)
                        *(volatile int *)&sm.alive[(i + 1) % 3] = 0;
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
                if (kShare == 1) {
                    __syncwarp();
                    lanes = mine;
                } else if (lane == 0) {
                    atomicAdd(&sm.alive[i % 3], mine);
                }
                if (kShare > 1 && kBuf == 1) {
                    // everybody has added, and the marks are clear; the slot read
                    // here is cleared two sequences later at the earliest
                    __syncthreads();
                    lanes = *(volatile int *)&sm.alive[i % 3];
                    if (threadIdx.x == 0)
                        *(volatile int *)&sm.alive[(i + 1) % 3] = 0;
                }
                ++i;
                holding = lanes;
                if (lanes <= kSvLookupLanes<kMid, kShare>)
                    break;
            }
            if (kBuf > 1)
                __syncthreads();   // a buffer's marks are all taken before strings are put into it
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
                sv_mark<kMid, kShare>(blk.win + (size_t)i * in.W, in.W, in.d, blk.prefix, marks, sm.list[warp], sm, my, g, lane);
                share_sync<kShare>();
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
                ++i;
                // a string needs q - (n - i) hits by now; the block ends once none has them
                const int need1 = in.q - (in.n - i) - 1;
                left = 0;
                if (need1 >= 0) {
#pragma unroll
                    for (int k = 0; k < kPieces; ++k)
                        left |= sv_above<kPlanes, kPieces>(cnt, k, need1);
                }
                if (kShare == 1) {
                    __syncwarp();
                    if (!__any_sync(kFull, need1 < 0 || left != 0u))
                        break;
                } else if (!__syncthreads_or(need1 < 0 || left != 0u)) {
                    break;
                }
            }
            holding = kShare == 1 ? __popc(__ballot_sync(kFull, left != 0u)) : __syncthreads_count(left != 0u);
            if (__any_sync(kFull, left != 0u)) {
#pragma unroll
                for (int k = 0; k < kPieces; ++k)
                    mw[at_of(k)] = sv_above<kPlanes, kPieces>(cnt, k, in.q - 1);
            }
        }
        const bool counted = i == in.n && holding >= kSvCountFrom / 2;
        if (counted) {   // the windows of s_1..s_{n-q+1} are contiguous
            share_sync<kShare>();
            sv_count<kMid, kShare>(blk.win, in.nseed * in.W, in.d, blk.prefix, marks, sm.list[warp], sm,
                                   out_of(p, blk.I), g, lane);
            share_sync<kShare>();
        }
        // the strings of a warp's threads: of many threads, a string of each at a time; of few,
        // the pieces of one thread at a time
        uint32_t holders = __ballot_sync(kFull, left != 0u);
        if (holders) {
            __syncwarp();
            const bool many = __popc(holders) > kPieces / 4;
            while (holders) {
                const int who = many ? lane : __ffs(holders) - 1;
                holders = many ? 0u : holders & (holders - 1u);
                for (int k0 = 0; k0 < kPieces; k0 += many ? 1 : 32) {
                    const int k = many ? k0 : k0 + lane;
                    const int at = ((k / kVec) * (32 * kShare) + g * 32 + who) * kVec + k % kVec;
                    uint32_t v = k < kPieces ? mw[at] : 0u;
                    while (__any_sync(kFull, v != 0u)) {
                        const bool has = v != 0u;
                        const int bit = has ? __ffs(v) - 1 : 0;
                        v &= v - 1u;
                        sv_emit<kMid>(p.inst + blk.I, out_of(p, blk.I), blk.win, has,
                                      sv_string<kMid>(blk.prefix, at, bit), i, counted, lane);
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
// sequences i = warp, warp + kSplitWarps, ... with marks of their own, so that
// they meet only once, to intersect what they are left with. Twenty warps: what
// a solve waits for is one warp's sequences, and most instances have about
// twenty (whole solves, 8 warps and 20: (9,2), n = 20, m = 600, 32.1 and 20.5 us;
// (11,3), n = 17, m = 733, from host memory, 87 and 67 us).
constexpr int kSplitWarps = 20;
template <int kMid, int kMinBlocks>
__global__ void __launch_bounds__(32 * kSplitWarps, kMinBlocks) sieve_split_kernel(SieveParams p)
{
    extern __shared__ __align__(16) unsigned char sv_raw[];
    using M = SvMarks<kMid>;
    constexpr int kPieces = 2 * M::kWords / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SvSmem<kMid, kSplitWarps> &sm = *reinterpret_cast<SvSmem<kMid, kSplitWarps> *>(sv_raw);
    const uint32_t marks0 = sv_setup<kMid, kSplitWarps>(sv_raw, kSplitWarps);
    const uint32_t marks = marks0 + warp * M::kBytes;
    uint32_t *all = reinterpret_cast<uint32_t *>(sv_raw + (marks0 - (uint32_t)__cvta_generic_to_shared(sv_raw)));
    uint32_t *mw = all + warp * (2 * M::kWords);
    int *dead = &sm.alive[0];
    const SvLane<kMid> my(sm, lane);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the packed windows are complete and visible
    for (long long it = blockIdx.x; it < p.total; it += gridDim.x) {
        if (threadIdx.x == 0)
            sm.alive[0] = sm.alive[1] = 0;
        __syncthreads();
        SvBlock blk(p, it, kMid);
        const InstDev &in = blk.in;
        uint32_t cur[kPieces];
#pragma unroll
        for (int k = 0; k < kPieces; ++k)
            cur[k] = kFull;
        for (int i = warp; i < in.n; i += kSplitWarps) {
            // another warp may set the flag at any time: the lanes decide together, as the marks need them all
            if (__any_sync(kFull, *(volatile int *)dead))
                break;
            sv_mark<kMid, 1>(blk.win + (size_t)i * in.W, in.W, in.d, blk.prefix, marks, sm.list[warp], sm, my, 0,
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
            // mark word at: warp at / 32 % kSplitWarps
            int strings = 0;
            for (int at = warp * 32 + lane; at < 2 * M::kWords; at += 32 * kSplitWarps) {
                uint32_t v = kFull;
#pragma unroll
                for (int t = 0; t < kSplitWarps; ++t)
                    v &= all[t * (2 * M::kWords) + at];
                all[at] = v;
                strings += __popc(v);
            }
            strings = __reduce_add_sync(kFull, strings);
            if (lane == 0 && strings > 0)
                atomicAdd(&sm.alive[1], strings);
            __syncthreads();
            const bool counted = *(volatile int *)&sm.alive[1] >= kSvCountFrom;
            if (counted) {
                sv_count<kMid, kSplitWarps>(blk.win, in.nseed * in.W, in.d, blk.prefix, marks0, sm.list[warp], sm,
                                            out_of(p, blk.I), warp, lane);
            }
            for (int at = warp * 32 + lane; at < 2 * M::kWords; at += 32 * kSplitWarps) {
                uint32_t v = all[at];
                while (__any_sync(kFull, v != 0u)) {
                    const bool has = v != 0u;
                    const int bit = has ? __ffs(v) - 1 : 0;
                    v &= v - 1u;
                    sv_emit<kMid>(p.inst + blk.I, out_of(p, blk.I), blk.win, has,
                                  sv_string<kMid>(blk.prefix, at, bit), in.n, counted, lane);
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
            uint16_t bank[32][128];
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

cudaError_t launch_kernel(void (*kernel)(SieveParams), const SieveParams &p, long long blocks, size_t smem,
                          cudaStream_t st, int threads = kSvThreads)
{
    const cudaError_t e =
        cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = dependent_launch(attr, (int)blocks, threads, smem, st);
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <int kMid, int kPlanes, int kShare, int kMinBlocks>
cudaError_t launch(const SieveParams &p, int sms, int per_sm, int reserved, cudaStream_t st)
{
    const long long teams = kSvWarps / kShare;
    return launch_kernel(sieve_kernel<kMid, kPlanes, kShare, kMinBlocks>, p,
                         std::min<long long>((long long)sms * std::min(kMinBlocks, per_sm), (p.total + teams - 1) / teams),
                         sv_smem_bytes<kMid>(reserved, sv_buffers<kMid, kPlanes, kShare>()), st);
}

template <int kMid, int kMinBlocks>
cudaError_t launch_split(const SieveParams &p, int sms, int per_sm, int reserved, cudaStream_t st)
{
    return launch_kernel(sieve_split_kernel<kMid, kMinBlocks>, p,
                         std::min<long long>((long long)sms * std::min(kMinBlocks, per_sm), p.total),
                         sv_smem_bytes<kMid, kSplitWarps>(reserved, kSplitWarps), st, 32 * kSplitWarps);
}

// The tables as they are uploaded. Made once, by whichever thread creates the first
// context, and only read after that: contexts may be created by several threads at a
// time, and an upload beside another context's running kernel writes the same bytes.
struct SvTables {
    SvTable t[4];
    uint32_t ball[4][64][2] = {};
    SvTables()
    {
        fill_table<3>(t[0]);
        fill_table<4>(t[1]);
        fill_table<5>(t[2]);
        fill_table<6>(t[3]);
        for (int v = 0; v < 4; ++v)
            for (int s = 0; s < 64; ++s)
                for (int u = 0; u < 64; ++u) {
                    const int x = s ^ u, diff = (x | (x >> 3)) & 7;
                    if ((diff & 1) + ((diff >> 1) & 1) + (diff >> 2) <= v)
                        ball[v][s][u >> 5] |= 1u << (u & 31);
                }
    }
};

}  // namespace

cudaError_t sieve_init_tables()
{
    static const SvTables tables;
    const cudaError_t e = cudaMemcpyToSymbol(g_sv_table, tables.t, sizeof tables.t);
    if (e != cudaSuccess)
        return e;
    return cudaMemcpyToSymbol(g_sv_ball, tables.ball, sizeof tables.ball);
}

cudaError_t launch_sieve(const SieveParams &p, int mid, int planes, int share, int sms, int per_sm, cudaStream_t st)
{
    int dev = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess)
        return e;
    if (per_sm <= 0)
        per_sm = 1 << 16;
    if (planes > 0)
        return mid == 5   ? launch<5, 5, 8, 3>(p, sms, per_sm, reserved, st)
               : mid == 4 ? launch<4, 5, 1, 2>(p, sms, per_sm, reserved, st)
                          : launch<3, 7, 1, 3>(p, sms, per_sm, reserved, st);
    if (mid == 6)
        return launch<6, 0, 8, 4>(p, sms, per_sm, reserved, st);
    if (mid == 5)
        return share == 1 ? launch<5, 0, 1, 2>(p, sms, per_sm, reserved, st) : launch<5, 0, 8, 4>(p, sms, per_sm, reserved, st);
    if (mid == 4)
        return share == 1 ? launch<4, 0, 1, 4>(p, sms, per_sm, reserved, st) : launch_split<4, 2>(p, sms, per_sm, reserved, st);
    return share == 1 ? launch<3, 0, 1, 5>(p, sms, per_sm, reserved, st) : launch_split<3, 2>(p, sms, per_sm, reserved, st);
}

}  // namespace pms
