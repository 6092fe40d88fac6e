// bsw_short.cu - short queries of small batches: one pair per warp, the row in
// registers.
//
// The per-thread kernels give a pair to a lane, so a batch lasts at least as
// long as one lane takes for its longest pair, 100 to 300 us however few pairs
// there are.  Here lane L of a warp holds columns C*L .. C*L + C - 1 of the row
// (H and E of Section V-A's one row) in registers, C = 4, 5, 6 or 8 for queries up
// to 128, 160, 192 or 256 bases, and a row costs one pass: the cells of Eq. 2, F as a
// max-plus prefix over the lanes (F(i,j) = max(0, max_{k<j} (M_k - o - e -
// (j-1-k)e)), Eq. 3's affine gaps), the row maximum and its column as one warp
// reduction, and the band adjustment (rule c) from two ballots.
//
// What bounds it: with few pairs the latency of a row (about 600 cycles: the
// five shuffles of the prefix and the reductions, one after the other), with
// many the instructions of a row.  97 pairs of 151 bp reads take 97 us where the
// per-thread kernels take 196, 8000 pairs of 250 bp reads 297 against 555.  64
// registers (8 blocks of 4 warps) run 4000 such pairs in 656 us instead of 290,
// 8 columns a lane for every query above 128 bases 473; blocks of 2 warps spread
// the pairs over the SMs more evenly (4000 pairs with N: 293 us against 373).
#include <cuda_runtime.h>
#include <cstdint>

#include "bsw_device.cuh"
#include "bsw_launch.h"

namespace bsw {

namespace {

constexpr int kShortThreads = 64;

// Extend the pair of record R with the whole warp.  Slot j of the row holds
// H(i-1, j-1) and E(i, j); slot n (the row end once the band reaches the query
// end) is not kept: it is never a diagonal, and whether it is zero is hl > 0.
// Columns outside [lo, hi) keep their slots, which a band that grows past an
// earlier row's end reads again.  Scores stay below 2^22 (row key H * 512 +
// column).
template <int C, bool NM>
__device__ unsigned long long short_pair(const Batch &B, const Params &P, const PairRec &R, bsw_result_t *out)
{
    const int lane = threadIdx.x & 31, j0 = lane * C;
    const int n = R.n, m = R.m, h0 = R.h0;
    const int wb = clip_band(P, n, R.w);
    const int a = P.a, mb = -P.b, e_del = P.e_del, e_ins = P.e_ins;
    const int oe_del = P.o_del + e_del, oe_ins = P.o_ins + e_ins, ce = C * e_ins;
    // the lane's query codes and N bits
    uint32_t q = 0, qn = 0;
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const int64_t pos = R.q_off + j0 + k;
        if (j0 + k < n) {
            q |= (((uint32_t)__ldg(B.q + (pos >> 2)) >> (2 * (pos & 3))) & 3u) << (2 * k);
            if (NM && B.q_n) qn |= (((uint32_t)__ldg(B.q_n + (pos >> 3)) >> (pos & 7)) & 1u) << k;
        }
    }
    int Hs[C], Es[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const int j = j0 + k;
        Hs[k] = j >= n ? 0 : j == 0 ? h0 : max(0, h0 - P.o_ins - j * e_ins);
        Es[k] = 0;
    }
    int lo = 0, hi = n;
    int best = h0, bi = -1, bj = -1, gbest = -1, gi = -1, moff = 0;
    unsigned long long ncell = 0;
    uint32_t tw = 0;                     // the lane's byte of 128 target rows: four bases, N bits in 8-11
    for (int i = 0; i < m; ++i) {
        if ((i & 127) == 0) {
            const int r = i + 4 * lane;
            tw = 0;
            if (r < m) {
                tw = __ldg(B.t + ((R.t_off + r) >> 2));
                if (NM && B.t_n) {
                    const int64_t pos = R.t_off + r;
                    tw |= (((uint32_t)__ldg(B.t_n + (pos >> 3)) >> (pos & 7)) & 15u) << 8;
                }
            }
        }
        const uint32_t tq = __shfl_sync(kFull, tw, (i >> 2) & 31);
        const uint32_t x = q ^ (((tq >> (2 * (i & 3))) & 3u) * 0x5555u);      // field k is zero where base j0 + k is t_i
        const bool tn = NM && ((tq >> (8 + (i & 3))) & 1u);
        lo = max(lo, i - wb);
        hi = min(min(hi, i + wb + 1), n);
        const int hl0 = lo == 0 ? max(0, h0 - oe_del - i * e_del) : 0;         // H(i, lo-1), Eq. 3 first column
        // the lane's columns in the band, and slot hi (the row end) if it is one of its
        const uint32_t upto = (1u << min(max(hi - j0, 0), C)) - 1u;
        const uint32_t in = upto & ~((1u << min(max(lo - j0, 0), C)) - 1u);
        const uint32_t end = hi < n && hi >= j0 && hi < j0 + C ? 1u << (hi - j0) : 0u;
        int M[C], E[C], Fl[C];
        int floc = 0;
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const int d = (in >> k) & 1u ? Hs[k] : 0;
            E[k] = (in >> k) & 1u ? Es[k] : 0;
            int sc = (x & (3u << (2 * k))) ? mb : a;
            if (NM && (tn || ((qn >> k) & 1u))) sc = -1;
            M[k] = __viaddmin_s32(d, sc, d << 8);                             // match <= 127: at most 0 for d = 0
            Fl[k] = floc;
            floc = __viaddmax_s32_relu(floc, -e_ins, M[k] - oe_ins);
        }
        int v = floc + (lane + 1) * ce;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) v = max(v, __shfl_up_sync(kFull, v, s));
        int vex = __shfl_up_sync(kFull, v, 1);
        if (lane == 0) vex = 0;
        const int g = max(0, vex) - lane * ce;                                 // F entering the lane's first column
        int h[C], key = 0;
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const int f = __viaddmax_s32(g, -k * e_ins, Fl[k]);
            h[k] = (in >> k) & 1u ? __vimax3_s32(M[k], E[k], f) : 0;
            key = max(key, h[k] * 512 + j0 + k);
        }
        const int kw = (int)__reduce_max_sync(kFull, (unsigned)key);
        int hin = __shfl_up_sync(kFull, h[C - 1], 1);
        if (lane == 0) hin = hl0;
        uint32_t bits = 0;                                                     // the lane's non-zero slots in [lo, hi]
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const int left = k ? h[k ? k - 1 : 0] : hin;
            const int e2 = (in >> k) & 1u ? __viaddmax_s32_relu(E[k], -e_del, M[k] - oe_del) : 0;
            if (((in | end) >> k) & 1u) {
                Hs[k] = left;
                Es[k] = e2;
                if (left | e2) bits |= 1u << k;
            }
        }
        const int rm = kw >> 9, rj = kw & 511;
        if (hi > lo) ncell += (unsigned)(hi - lo);
        int hl = hl0;
        if (max(lo, hi) == n) {
            if (hi > lo) {
                int hv = h[0];
#pragma unroll
                for (int k = 1; k < C; ++k)
                    if ((n - 1) % C == k) hv = h[k];
                hl = __shfl_sync(kFull, hv, (n - 1) / C);
            }
            if (hl >= gbest) gi = i;
            gbest = max(gbest, hl);
        }
        if (rm == 0) break;
        if (rm > best) {
            best = rm; bi = i; bj = rj;
            moff = max(moff, abs(rj - i));
        } else if (P.zdrop > 0) {
            const int di = i - bi, dj = rj - bj;
            const int drop = di > dj ? best - rm - (di - dj) * e_del : best - rm - (dj - di) * e_ins;
            if (drop > P.zdrop) break;
        }
        // rule c: the first non-zero slot of [lo, hi), the last of [lo, hi] plus 2
        const int fc = bits ? j0 + __ffs(bits) - 1 : n, lc = bits ? j0 + 31 - __clz(bits) : -1;
        lo = min((int)__reduce_min_sync(kFull, (unsigned)fc), hi);
        const int lr = (int)__reduce_max_sync(kFull, (unsigned)(lc + 1)) - 1;
        const int last = hi == n && hl > 0 ? n /* its slot */ : max(lr, lo - 1);
        hi = min(last + 2, n);
    }
    if (lane == 0) store_result(out, best, bj + 1, bi + 1, gi + 1, gbest, moff);
    return ncell;
}

// The pairs of classes [c0, c1), which lie one after the other in the sorted
// order, longest queries first; a warp takes the next pair as it finishes one.
template <bool NM>
__global__ void __launch_bounds__(kShortThreads) k_short(Batch B, Params P, Work W, int c0, int c1)
{
    const int lane = threadIdx.x & 31;
    const int start = W.cls_start[c0];
    int count = 0;
    for (int c = c0; c < c1; ++c) count += W.cls_count[c];
    unsigned long long cells = 0;
    for (;;) {
        int g = 0;
        if (lane == 0) g = (int)atomicAdd(&W.cls_next[c0], 1u);
        g = __shfl_sync(kFull, g, 0);
        if (g >= count) break;
        const PairRec R = W.rec[start + g];
        bsw_result_t *out = &B.out[W.order[start + g]];
        cells += R.n <= 128   ? short_pair<4, NM>(B, P, R, out)
                 : R.n <= 160 ? short_pair<5, NM>(B, P, R, out)
                 : R.n <= 192 ? short_pair<6, NM>(B, P, R, out)
                              : short_pair<8, NM>(B, P, R, out);
    }
    if (lane == 0 && cells) atomicAdd(W.cells, cells);
}

}  // namespace

cudaError_t launch_short(const Batch &B, const Params &P, const Work &W, int c0, int c1, cudaStream_t st, int sms)
{
    constexpr int warps = kShortThreads / 32;
    const int64_t want = (B.n + warps - 1) / warps, most = (int64_t)sms * 16;
    const int blocks = (int)(want < most ? want : most);
    if (B.q_n || B.t_n) k_short<true><<<blocks, kShortThreads, 0, st>>>(B, P, W, c0, c1);
    else k_short<false><<<blocks, kShortThreads, 0, st>>>(B, P, W, c0, c1);
    return cudaGetLastError();
}

}  // namespace bsw
