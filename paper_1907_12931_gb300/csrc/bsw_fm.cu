// bsw_fm.cu - FM-index and super-maximal exact matches (Section IV).
//
// The text is T = ref + revcomp(ref) (Section IV-A: the SMEM search works on
// the reference with its reverse complement), followed by a terminator $
// smaller than every base.  One FM-index of T serves both directions: since
// revcomp(T) = T, a pattern P and revcomp(P) occur equally often, and the
// pair of their suffix-array intervals (the bi-interval [k, l, s] of
// Algorithms 2-3) can be extended by one base on either side.
//
// O (Algorithm 1) is kept in buckets of eta = 32 BWT positions: entry t holds,
// for each base, its first row plus its count in BWT[0, 32t), and the low and
// the high bits of the bucket's 32 BWT bases as one 32-bit word each: 32 bytes,
// one DRAM sector per lookup (the paper's CPU layout uses 64-byte entries with a
// byte per base for AVX2 compares; bit planes and population counts serve the
// GPU).  One lookup gives a base's row and the occurrences of the larger ones;
// the $ row is stored as base 0 and subtracted.
//
// SMEMs of a read X (Li 2012; Algorithm 4): from a position x, extend X[x]
// forward base by base, keeping the match each time its number of occurrences
// is about to shrink (one per distinct count, longest match last); then extend
// those matches backward one base at a time, longest first.  A match that can
// no longer be extended while no longer one survives at that base is an SMEM.
// The next x is the end of the longest match from x; every SMEM holds exactly
// one of the visited x.  No search starts at an N or at a base that T does not
// hold: no match contains either.
//
// The starts x depend on the forward searches alone, so the search is cut in
// two kernels whose lanes do the same work at the same time: k_smem_scan takes
// a read per lane, one base per step, and notes the starts; k_smem_store takes a
// start per lane and does its forward and backward pass.  Where the budget does
// not hold the starts of all reads at once they run in rounds.  A read with more than
// kListCap matches in one list is finished by a launch with lists in global
// memory (k_smem_global), where a lane does a whole read.  One pass keeps up to
// W.keep records per read in a scratch buffer; after a prefix sum of the
// counts a gather sorts them into place, and the rare reads with more are searched
// again, writing in place.
#include <cuda_runtime.h>
#include <climits>
#include <cstdint>
#include <vector>

#include "bsw.h"
#include "bsw_launch.h"

namespace bsw {

// ------------------------------------------------------------------ host build

// Index of one text (codes 0..3, length n) from its suffix array sa[0..n].
void fm_from_sa(const uint8_t *text, int64_t n, const int32_t *sa, FmHost &out)
{
    const int64_t N = n + 1;
    out.n = N;
    out.occ.assign((size_t)(N / 32 + 1), FmEntry{{0, 0, 0, 0}, 0, 0, {0, 0}});
    uint32_t cnt[4] = {0, 0, 0, 0};
    out.primary = -1;
    for (int64_t i = 0; i < N; ++i) {
        if ((i & 31) == 0) {
            FmEntry &e = out.occ[(size_t)(i >> 5)];
            for (int c = 0; c < 4; ++c) e.cnt[c] = cnt[c];
        }
        int b;
        if (sa[i] == 0) {
            out.primary = i;                              // the $ row: stored as 0, not counted
            b = 0;
        } else {
            b = text[sa[i] - 1];
            ++cnt[b];
        }
        FmEntry &e = out.occ[(size_t)(i >> 5)];
        e.lo |= (uint32_t)(b & 1) << (i & 31);
        e.hi |= (uint32_t)(b >> 1) << (i & 31);
    }
    if ((N & 31) == 0) {
        FmEntry &e = out.occ[(size_t)(N >> 5)];
        for (int c = 0; c < 4; ++c) e.cnt[c] = cnt[c];
    }
    out.C[0] = 1;                                         // the terminator sorts first
    for (int c = 0; c < 4; ++c) out.C[c + 1] = out.C[c] + cnt[c];
    for (FmEntry &e : out.occ)                            // the first row of each base, so that a lookup gives rows
        for (int c = 0; c < 4; ++c) e.cnt[c] += (uint32_t)out.C[c];
}

// --------------------------------------------------------------------- device

namespace {

// A bucket of O in registers, by one 256-bit load: the lanes of a warp look up
// rows all over the table, so a load costs a pass of the L1 per lane, and a
// bucket read as 128 and 64 bits two.
struct Bucket {
    uint32_t cnt[4], lo, hi, pad[2];
};
__device__ __forceinline__ Bucket load_bucket(const FmEntry *e)
{
    Bucket v;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v.cnt[0]), "=r"(v.cnt[1]), "=r"(v.cnt[2]), "=r"(v.cnt[3]), "=r"(v.lo), "=r"(v.hi), "=r"(v.pad[0]), "=r"(v.pad[1])
        : "l"(e));
    return v;
}

// What a lookup of O at row i gives for base b (Algorithm 1): row = C[b] + the
// occurrences of b in BWT[0, i), and above = those of the bases larger than b
// plus a constant (only differences of it are used).
struct Occ {
    uint32_t row, above;
};
__device__ __forceinline__ Occ occ_in(const FmDev &F, const Bucket &v, uint32_t i, uint32_t b)
{
    const uint32_t y = i & 31u;
    const uint32_t m = (1u << y) - 1u;                                       // bases j < y
    const uint32_t x = v.lo ^ (0u - (b & 1u)), z = v.hi ^ (0u - (b >> 1));   // both bits zero where base j is b
    Occ o;
    o.row = (b < 2 ? (b == 0 ? v.cnt[0] : v.cnt[1]) : (b == 2 ? v.cnt[2] : v.cnt[3])) + (uint32_t)__popc(~(x | z) & m);
    if (b == 0 && F.primary - (i - y) < y) --o.row;                          // the $ row, stored as base 0
    // larger than 0: either bit set; than 1: the high one; than 2: both
    const uint32_t g = b == 0 ? (v.lo | v.hi) : b == 1 ? v.hi : b == 2 ? (v.lo & v.hi) : 0u;
    const uint32_t zw = v.cnt[2] + v.cnt[3];
    o.above = (b == 0 ? v.cnt[1] + zw : b == 1 ? zw : b == 2 ? v.cnt[3] : 0u) + (uint32_t)__popc(g & m);
    return o;
}

// The extension of the rows [a, a + s) by base b (Algorithm 2): the rows of bP
// are [row, row + size); above = the occurrences among the s rows' preceding
// bases of those larger than b.  Both ends of a small interval usually lie in
// one bucket, which is then read once.
struct Ext {
    uint32_t row, size, above;
};
__device__ __forceinline__ Ext extend(const FmDev &F, uint32_t a, uint32_t s, uint32_t b)
{
    const uint32_t e = a + s;
    const Bucket v0 = load_bucket(F.occ + (a >> 5));
    Bucket v1 = v0;
    if ((e >> 5) != (a >> 5)) v1 = load_bucket(F.occ + (e >> 5));
    const Occ o0 = occ_in(F, v0, a, b), o1 = occ_in(F, v1, e, b);
    return Ext{o0.row, o1.row - o0.row, o1.above - o0.above};
}

// C[c], the first row of base c (c = 4: past the last).
__device__ __forceinline__ uint32_t first_row(const FmDev &F, int c)
{
    return c < 2 ? (c == 0 ? F.C[0] : F.C[1]) : c == 2 ? F.C[2] : c == 3 ? F.C[3] : F.C[4];
}

// The bases a search can start at, bit c for base c: those the text holds (no N).
__device__ __forceinline__ uint32_t text_bases(const FmDev &F)
{
    uint32_t m = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) m |= (uint32_t)(F.C[c + 1] != F.C[c]) << c;
    return m;
}

// A read of the batch: its packed bases (a read starts on a byte) and its base
// offset, which addresses the N bitmap.
struct ReadRef {
    const uint8_t *q;
    int64_t off;
    __device__ __forceinline__ ReadRef() : q(nullptr), off(0) {}
    __device__ __forceinline__ ReadRef(const SmemIn &R, int64_t o) : q(R.reads + (o >> 2)), off(o) {}
    // Base pos: 0..3, or 4 for an N.
    __device__ __forceinline__ int base(const SmemIn &R, int pos) const
    {
        if (R.reads_n && ((__ldg(R.reads_n + ((off + pos) >> 3)) >> ((off + pos) & 7)) & 1)) return 4;
        return (__ldg(q + (pos >> 2)) >> (2 * (pos & 3))) & 3;
    }
};

// All SMEMs of at least min_len bases of the reads t < t_end taken from the
// counter W.ctr->next (read ids[t]).  Store mode: count[r], and the first W.keep
// matches at scratch[r * W.keep], in the order they are found
// (k_smem_gather sorts them); a read with more is finished by a write-mode
// launch.  Write mode: the records at out[first[r]], in increasing start order.
// A lane's list holds any read of the batch.
//
// The lane is a small state machine so that every pass of the main loop makes
// exactly one extension on every lane that has work (the memory lookups of
// Algorithm 1 dominate; lanes of a warp run in step instead of each following
// its own loop nest).  States between extensions:
//   kRead  take the next read;     kCall  start the search from x;
//   kBack  forward pass over, start the backward pass;
//   kEnd   the search from x is over;
//   kFwd   pending: extend the match forward by X[i];
//   kBwd   pending: extend the list's p-th longest match backward by X[j].
//
// An extension of P by base b on the left (Algorithm 2) maps its rows [k, k +
// s) to [C[b] + O(b, k), C[b] + O(b, k + s)).  A forward extension by c
// (Algorithm 3) is the same step on revcomp(P)'s rows [l, l + s) with b = 3 -
// c, and P's rows move up by as many as revcomp(P) has occurrences preceded by
// the terminator or by a base larger than b (they sort before); a backward one
// needs no more than the rows, as no forward extension follows.
template <bool WRITE>
__device__ void smem_lanes(const SmemIn &R, const FmDev &F, int min_len, int64_t t_end, const int32_t *ids,
                           BiIv *list, const SmemWork &W)
{
    enum { kRead, kCall, kBack, kEnd, kFwd, kBwd };
    const uint32_t held = text_bases(F);
    int state = kRead;
    int r = 0, n = 0, call0 = 0;
    int64_t o = 0;
    int L = 0, x = 0, i = 0, j = 0, p = 0, m = 0, mc = 0, top = 0, next = 0, last = 0;
    uint32_t vk = 0, vl = 0, vs = 0, ls = 0;                            // the forward match; the last survivor's size
    ReadRef read;
    auto base_at = [&](int pos) { return read.base(R, pos); };
    auto emit = [&](int start, int end, uint32_t k, uint32_t s) {
        if (end - start < min_len) return;
        if (WRITE) W.out[o + n] = bsw_smem_t{(int32_t)r, start, end - start, 0, (int64_t)k, (int64_t)s};
        else if (n < W.keep) W.scratch[o + n] = make_uint4((uint32_t)start, (uint32_t)(end - start), k, s);
        ++n;
    };
    for (;;) {
        // settle: run the bookkeeping up to the next extension
        while (state < kFwd) {
            if (state == kRead) {
                const int64_t t = atomicAdd(&W.ctr->next, 1u);
                if (t >= t_end) return;
                r = ids[t];
                L = R.read_len[r];
                read = ReadRef(R, R.read_off[r]);
                o = WRITE ? W.first[r] : (int64_t)r * W.keep;
                n = 0;
                x = 0;
                state = kCall;
            } else if (state == kCall) {
                if (x >= L) {
                    if (!WRITE) W.count[r] = n;
                    state = kRead;
                    continue;
                }
                const int c0 = base_at(x);
                if (!((held >> c0) & 1u)) {
                    ++x;
                    continue;
                }
                vk = first_row(F, c0);
                vl = first_row(F, 3 - c0);
                vs = first_row(F, c0 + 1) - vk;
                m = 0;
                i = x + 1;
                if (i < L) {
                    state = kFwd;
                } else {
                    list[m++] = BiIv{vk, vs, L};
                    state = kBack;
                }
            } else if (state == kBack) {
                // the list is in order of increasing length: the p-th longest
                // is entry top - p, and survivors go back from the top down
                top = m - 1;
                next = list[top].e;
                call0 = n;
                last = INT_MAX;
                j = x - 1;
                p = 0;
                mc = 0;
                if (j >= 0) {
                    state = kBwd;
                } else {                                                // at the read start: the longest is an SMEM
                    emit(0, next, list[top].k, list[top].s);
                    state = kEnd;
                }
            } else {                                                    // kEnd
                // this search emitted starts in decreasing order
                if (WRITE)
                    for (int64_t a = o + call0, b = o + n - 1; a < b; ++a, --b) {
                        const bsw_smem_t u = W.out[a];
                        W.out[a] = W.out[b];
                        W.out[b] = u;
                    }
                x = next;
                state = kCall;
            }
        }

        // one extension, the same code on every lane
        const bool fwd = state == kFwd;
        uint32_t a = vl, s = vs;
        if (!fwd) {
            a = list[top - p].k;
            s = list[top - p].s;
        }
        const int cb = base_at(fwd ? i : j);
        const uint32_t b = (uint32_t)(fwd ? 3 - (cb & 3) : cb & 3);
        const Ext u = extend(F, a, s, b);
        const uint32_t s2 = cb > 3 ? 0u : u.size;                       // an N extends nothing

        if (fwd) {
            if (s2 != vs) {                                             // X[x..i) is the longest with its count
                list[m++] = BiIv{vk, vs, i};
                if (s2 == 0) {
                    state = kBack;
                    continue;
                }
            }
            vk += u.above + (F.primary - a < s ? 1u : 0u);
            vl = u.row;
            vs = s2;
            if (++i == L) {                                             // the match reaches the read end
                list[m++] = BiIv{vk, vs, L};
                state = kBack;
            }
        } else {
            if (s2 == 0) {
                if (mc == 0 && j + 1 < last) {                          // no longer match survives: an SMEM
                    last = j + 1;
                    emit(last, list[top - p].e, a, s);
                }
            } else if (mc == 0 || s2 != ls) {
                list[top - mc] = BiIv{u.row, s2, list[top - p].e};
                ls = s2;
                ++mc;
            }
            if (++p == m) {
                if (mc == 0) {
                    state = kEnd;
                } else {
                    m = mc;
                    mc = 0;
                    p = 0;
                    if (--j < 0) {                                      // at the read start
                        emit(0, list[top].e, list[top].k, list[top].s);
                        state = kEnd;
                    }
                }
            }
        }
    }
}

// Store mode: counts and scratch records by atomics, as several lanes may work
// on one read.  A read whose list does not fit is marked with kSmemOvf, which no
// count reaches, and listed once.
constexpr unsigned long long kSmemOvf = 1ull << 40;

__device__ __forceinline__ void emit_match(const SmemWork &W, int min_len, int r, int start, int end, uint32_t k, uint32_t s)
{
    if (end - start < min_len) return;
    const unsigned long long n = atomicAdd(reinterpret_cast<unsigned long long *>(W.count + r), 1ull);
    if (n < W.keep) W.scratch[(int64_t)r * W.keep + n] = make_uint4((uint32_t)start, (uint32_t)(end - start), k, s);
}

__device__ __forceinline__ void overflow_read(const SmemWork &W, int r)
{
    if (atomicAdd(reinterpret_cast<unsigned long long *>(W.count + r), kSmemOvf) < kSmemOvf)
        W.ovf_list[atomicAdd(&W.totals->overflows, 1u)] = r;
}

// The starts of the searches of reads [r0, r0 + nr): a warp takes 32 of them, a
// lane one, a base per step.  The longest match from the read's start is an SMEM;
// the other starts go to the group's part of W.starts (start | lane << 16), which
// has the reads' own room: one long read among short ones takes no other group's.
__global__ void __launch_bounds__(kSmemThreads) k_smem_scan(SmemIn R, FmDev F, int min_len, SmemWork W, int64_t r0, int64_t nr)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (g * 32 >= nr) return;
    const int r = (int)(r0 + g * 32 + lane);
    const bool mine = g * 32 + lane < nr;
    const int L = mine ? R.read_len[r] : 0;
    ReadRef read;
    if (mine) read = ReadRef(R, R.read_off[r]);
    const unsigned room = __reduce_add_sync(kAll, mine ? (unsigned)smem_room(L) : 0u);
    unsigned long long part = 0;
    if (lane == 0) part = atomicAdd(&W.ctr->used, (unsigned long long)room);
    part = __shfl_sync(kAll, part, 0);
    uint32_t *starts = W.starts + part;
    const uint32_t held = text_bases(F);
    uint32_t quad = 0;
    int i = 0, x = -1, n = 0;                // the next base; the search's start (-1: none); starts noted
    uint32_t vk = 0, vl = 0, vs = 0;         // the match X[x..i), its rows and those of its reverse complement
    while (__any_sync(kAll, i < L)) {
        if ((i & 3) == 0 && i < L) quad = __ldg(read.q + (i >> 2));       // four bases; their N bits come one by one
        const int c = i >= L ? 4 : R.reads_n ? read.base(R, i) : (int)((quad >> (2 * (i & 3))) & 3u);
        const uint32_t b = 3u - (uint32_t)(c & 3);
        const Ext u = extend(F, vl, vs, b);
        const uint32_t s2 = c < 4 ? u.size : 0u;
        const bool ends = i < L && x >= 0 && s2 == 0;
        if (ends && x == 0) emit_match(W, min_len, r, 0, i, vk, vs);
        const bool starts_here = i < L && (x < 0 || ends) && ((held >> c) & 1u);
        if (starts_here) {
            vk = first_row(F, c);
            vl = first_row(F, 3 - c);
            vs = first_row(F, c + 1) - vk;
        } else {
            vk += u.above + (F.primary - vl < vs ? 1u : 0u);
            vl = u.row;
            vs = s2;
        }
        const unsigned st = __ballot_sync(kAll, starts_here && i > 0);
        if (starts_here && i > 0) {
            const int at = n + __popc(st & below);
            if (at < (int)room) starts[at] = (uint32_t)i | ((uint32_t)lane << 16);
            else overflow_read(W, r);
        }
        n += __popc(st);
        if (starts_here) x = i;
        else if (ends) x = -1;
        if (i < L && ++i == L) {
            if (x == 0) emit_match(W, min_len, r, 0, L, vk, vs);
            vl = vs = 0;                                                  // done: look up row 0
        }
    }
    if (lane == 0) W.group[g] = SmemGroup{(int64_t)part, min(n, (int)room), 0};
}

// The searches from the noted starts: a warp works through the starts of
// groups of 32 reads, its lanes taking the next one as they finish.  A lane's
// matches lie in shared memory, 10 bytes each: rows and end (the rows of
// revcomp(P), which the forward search needs, play no part once it is over).
// A pass of the main loop makes one extension on every lane, forward or
// backward; a forward one is a backward one of revcomp(P), see smem_lanes.
// Bound by the lookups (random 32-byte reads, mostly L2 hits).  200 k reads of
// 151 bp against a 32 Mbp text: k_smem_scan 0.28 ms and this kernel 1.10 ms, with
// 25 and 18 of 32 lanes active; one kernel with a lane per read, lists of 16-byte
// entries and two loads per bucket took 1.84 ms at 15 lanes.  24 matches a lane
// and 7 blocks an SM run as fast as 28 and 6, 1% faster than 20 and 8.
__global__ void __launch_bounds__(kSmemThreads) k_smem_store(SmemIn R, FmDev F, int min_len, SmemWork W, int64_t r0, int64_t ng)
{
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ uint2 ks[kListCap * kSmemThreads];
    __shared__ uint16_t ends[kListCap * kSmemThreads];
    const int lane = threadIdx.x & 31, me = threadIdx.x;
    const unsigned below = (1u << lane) - 1u;
    int64_t rg = 0;                          // the first read of the warp's group, its starts and the next of them
    const uint32_t *starts = W.starts;
    int nq = 0, head = 0;
    bool left = true;                        // groups are left
    int r = -1, L = 0, x = 0, i = 0, j = 0;  // the lane's read (-1: none), the search's start; the next base either way
    ReadRef read;
    bool fwd = true;
    int c = 4, cpos = -1;                    // the base last read, and its position
    int m = 0, p = 0, mc = 0, top = 0, last = 0;
    uint32_t vk = 0, vl = 0, vs = 0, ls = 0; // the forward match; the last survivor's count
    for (;;) {
        if (head == nq && left) {
            uint32_t t = 0;
            if (lane == 0) t = atomicAdd(&W.ctr->next, 1u);
            const int64_t g = (int64_t)__shfl_sync(kAll, t, 0);
            left = g < ng;
            nq = head = 0;
            if (left) {
                const SmemGroup G = W.group[g];
                rg = r0 + g * 32;
                starts = W.starts + G.at;
                nq = G.n;
            }
        }
        const unsigned want = __ballot_sync(kAll, r < 0);
        if (want && head < nq) {
            const int t = head + __popc(want & below);
            if (r < 0 && t < nq) {
                const uint32_t st = starts[t];
                r = (int)(rg + (st >> 16));
                x = (int)(st & 0xffffu);
                read = ReadRef(R, R.read_off[r]);
                L = R.read_len[r];
                c = read.base(R, x);                                     // a base of the text
                cpos = x;
                vk = first_row(F, c);
                vl = first_row(F, 3 - c);
                vs = first_row(F, c + 1) - vk;
                i = x + 1;
                m = 0;
                fwd = true;
            }
            head = min(head + __popc(want), nq);
        }
        if (__ballot_sync(kAll, r >= 0) == 0) {
            if (!left && head == nq) return;
        } else if (r >= 0) {
            const int pos = fwd ? i : j;
            if (pos != cpos) {
                c = pos < L ? read.base(R, pos) : 4;                     // the read's end stops a search as an N does
                cpos = pos;
            }
            uint32_t a = vl, s = vs;
            if (!fwd) {
                const uint2 q = ks[(top - p) * kSmemThreads + me];
                a = q.x;
                s = q.y;
            }
            const uint32_t b = (uint32_t)(fwd ? 3 - (c & 3) : c & 3);
            const Ext u = extend(F, a, s, b);
            const uint32_t s2 = c < 4 ? u.size : 0u;
            if (fwd) {
                if (s2 != vs || i == L) {                                // X[x..i) is the longest with its count
                    if (m < kListCap) {
                        ks[m * kSmemThreads + me] = make_uint2(vk, vs);
                        ends[m * kSmemThreads + me] = (uint16_t)i;
                        ++m;
                        if (s2 == 0) {                                   // the forward pass is over
                            fwd = false;
                            top = m - 1;
                            p = mc = 0;
                            j = x - 1;
                            last = INT_MAX;
                        }
                    } else {
                        overflow_read(W, r);
                        r = -1;
                    }
                }
                vk += u.above + (F.primary - a < s ? 1u : 0u);
                vl = u.row;
                vs = s2;
                ++i;
            } else {
                // longest first: the list is in order of increasing length, the
                // p-th longest is entry top - p, and survivors go back from the
                // top down
                if (s2 == 0) {
                    if (mc == 0 && j + 1 < last) {                       // no longer match survives: an SMEM
                        last = j + 1;
                        emit_match(W, min_len, r, last, ends[(top - p) * kSmemThreads + me], a, s);
                    }
                } else if (mc == 0 || s2 != ls) {
                    ks[(top - mc) * kSmemThreads + me] = make_uint2(u.row, s2);
                    ends[(top - mc) * kSmemThreads + me] = ends[(top - p) * kSmemThreads + me];
                    ls = s2;
                    ++mc;
                }
                if (++p == m) {
                    m = mc;
                    p = mc = 0;
                    if (m == 0) {
                        r = -1;
                    } else if (--j < 0) {                                // at the read start
                        const uint2 v = ks[top * kSmemThreads + me];
                        emit_match(W, min_len, r, 0, ends[top * kSmemThreads + me], v.x, v.y);
                        r = -1;
                    }
                }
            }
        }
    }
}

// The reads ids[0..n_ids) with lists in global memory, cap entries per lane
// (enough for any read of the batch).
template <bool WRITE>
__global__ void __launch_bounds__(256) k_smem_global(SmemIn R, FmDev F, int min_len, SmemWork W, const int32_t *ids,
                                                     int64_t n_ids, BiIv *lists, int cap)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n_ids) return;                     // at most n_ids lanes take reads: list slots g < n_ids
    smem_lanes<WRITE>(R, F, min_len, n_ids, ids, lists + g * cap, W);
}

// first[r] = the records before read r, first[n] = their number: sums of tiles of
// kFirstTile reads, then each tile's prefix.  The reads with more records than
// were kept are listed on the way.
constexpr int kFirstThreads = 256, kFirstPer = 8, kFirstTile = kFirstThreads * kFirstPer;

__device__ __forceinline__ int64_t block_sum(int64_t v)
{
    __shared__ int64_t w[kFirstThreads / 32];
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = v;
    __syncthreads();
    int64_t t = 0;
    for (int k = 0; k < kFirstThreads / 32; ++k) t += w[k];
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(kFirstThreads) k_smem_sums(int64_t n_reads, SmemWork W)
{
    int64_t v = 0;
    for (int u = 0; u < kFirstPer; ++u) {
        const int64_t r = (int64_t)blockIdx.x * kFirstTile + u * kFirstThreads + threadIdx.x;
        const int64_t c = r < n_reads ? W.count[r] : 0;
        if (c > W.keep) W.many[atomicAdd(&W.totals->many, 1u)] = (int32_t)r;
        v += c;
    }
    v = block_sum(v);
    if (threadIdx.x == 0) W.tile_sum[blockIdx.x] = v;
}

__global__ void __launch_bounds__(kFirstThreads) k_smem_first(int64_t n_reads, SmemWork W)
{
    __shared__ int64_t warp_sum[kFirstThreads / 32];
    int64_t before = 0;
    for (int64_t b = threadIdx.x; b < blockIdx.x; b += kFirstThreads) before += W.tile_sum[b];
    before = block_sum(before);
    const int64_t r0 = (int64_t)blockIdx.x * kFirstTile + (int64_t)threadIdx.x * kFirstPer;
    int64_t c[kFirstPer], sum = 0;
#pragma unroll
    for (int u = 0; u < kFirstPer; ++u) {
        c[u] = r0 + u < n_reads ? W.count[r0 + u] : 0;
        sum += c[u];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t x = sum;
    for (int d = 1; d < 32; d <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) warp_sum[wid] = x;
    __syncthreads();
    int64_t at = before + x - sum;
    for (int k = 0; k < wid; ++k) at += warp_sum[k];
#pragma unroll
    for (int u = 0; u < kFirstPer; ++u) {
        if (r0 + u < n_reads) W.first[r0 + u] = at;
        at += c[u];
        if (r0 + u == n_reads - 1) {
            W.first[n_reads] = at;
            W.totals->records = at;
        }
    }
}

// Records of the reads with at most W.keep from the scratch to out[first[r]],
// sorted by start (a read's SMEMs have distinct starts).
__global__ void __launch_bounds__(256) k_smem_gather(int64_t n_reads, SmemWork W)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_reads; r += stride) {
        const int c = (int)W.count[r];
        if (c > W.keep) continue;
        const uint4 *v = W.scratch + r * W.keep;
        for (int k = 0; k < c; ++k) {
            const uint4 u = v[k];
            int rank = 0;
            for (int q = 0; q < c; ++q) rank += v[q].x < u.x;
            W.out[W.first[r] + rank] = bsw_smem_t{(int32_t)r, (int32_t)u.x, (int32_t)u.y, 0, (int64_t)u.z, (int64_t)u.w};
        }
    }
}

int grid_for(int64_t n, int per_block, int sms, int per_sm)
{
    const int64_t b = (n + per_block - 1) / per_block;
    return (int)(b < (int64_t)sms * per_sm ? (b > 0 ? b : 1) : (int64_t)sms * per_sm);
}

}  // namespace

int64_t smem_tiles(int64_t n_reads) { return (n_reads + kFirstTile - 1) / kFirstTile; }

cudaError_t launch_smem_clear(int64_t n_reads, const SmemWork &W, cudaStream_t st)
{
    const cudaError_t e = cudaMemsetAsync(W.count, 0, sizeof(int64_t) * (size_t)n_reads, st);
    return e != cudaSuccess ? e : cudaMemsetAsync(W.totals, 0, sizeof(SmemTotals), st);
}

cudaError_t launch_smem_store(const SmemIn &R, const FmDev &F, int min_len, const SmemWork &W, int64_t r0, int64_t nr,
                              cudaStream_t st, int sms)
{
    const cudaError_t e = cudaMemsetAsync(W.ctr, 0, sizeof(SmemCounters), st);
    if (e != cudaSuccess) return e;
    const int64_t ng = (nr + 31) / 32;
    constexpr int warps = kSmemThreads / 32;
    k_smem_scan<<<(unsigned)((ng + warps - 1) / warps), kSmemThreads, 0, st>>>(R, F, min_len, W, r0, nr);
    k_smem_store<<<grid_for(ng, warps, sms, kSmemBlocksPerSm), kSmemThreads, 0, st>>>(R, F, min_len, W, r0, ng);
    return cudaGetLastError();
}

cudaError_t launch_smem_global(bool write, const SmemIn &R, const FmDev &F, int min_len, const SmemWork &W,
                               const int32_t *ids, int64_t n_ids, BiIv *lists, int cap, cudaStream_t st, int sms)
{
    if (n_ids <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(W.ctr, 0, sizeof(SmemCounters), st);
    if (e != cudaSuccess) return e;
    const int blocks = grid_for(n_ids, 256, sms, 8);
    if (write) k_smem_global<true><<<blocks, 256, 0, st>>>(R, F, min_len, W, ids, n_ids, lists, cap);
    else k_smem_global<false><<<blocks, 256, 0, st>>>(R, F, min_len, W, ids, n_ids, lists, cap);
    return cudaGetLastError();
}

cudaError_t launch_smem_first(int64_t n_reads, const SmemWork &W, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(&W.totals->many, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    const unsigned tiles = (unsigned)smem_tiles(n_reads);
    k_smem_sums<<<tiles, kFirstThreads, 0, st>>>(n_reads, W);
    k_smem_first<<<tiles, kFirstThreads, 0, st>>>(n_reads, W);
    return cudaGetLastError();
}

cudaError_t launch_smem_gather(int64_t n_reads, const SmemWork &W, cudaStream_t st, int sms)
{
    if (n_reads <= 0) return cudaSuccess;
    k_smem_gather<<<grid_for(n_reads, 256, sms, 8), 256, 0, st>>>(n_reads, W);
    return cudaGetLastError();
}

}  // namespace bsw
