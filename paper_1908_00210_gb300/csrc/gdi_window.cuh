// gdi_window.cuh -- window building blocks of libgdi.so, shared by the grid-scale kernels
// (gdi_grid.cu) and the CTA-resident counting kernel (gdi_kernels.cu).
//
// A window is W consecutive ranks of one colour class.  Inside it the +1 group, in order of flip
// threshold gamma ascending (then position), and the -1 group, by gamma descending, each see the
// exact running G (reading R2 of Algorithm 3).  The k-th member of the +1 group flips iff
// a_k = gamma_(k) + 2k <= G (-1: gamma_(k) - 2k >= G), so all that matters of a group is how many
// members have their threshold on either side of a value: windows are counted, not sorted.  Stage
// maps summarise a window on the lattice x = G - c = -64 .. 62 around a reference G c.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gdi_device.cuh"

namespace gdi {
namespace win {

constexpr int NT = 64;                  // lattice points of a stage map
constexpr int WBINS = 256;              // words a window's distances are counted in
constexpr int BIN_L = 190;              // distance -BIN_L is bin 0 (everything below too) in 256 bins
constexpr unsigned long long STEP_MASK = (1ull << (NT - 1)) - 1ull;

struct StageMap {
    unsigned long long mask;            // bit j: the step from lattice point j to j + 1 rises
    int32_t ylo;                        // output index of lattice point 0
    int32_t pad;
};

// counts of all bins before this lane's PER, by one warp
template <int PER>
__device__ __forceinline__ uint32_t bins_before(const uint32_t (&v)[PER])
{
    const int lane = threadIdx.x & 31;
    uint32_t tot = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) tot += v[i];
    uint32_t run = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, run, o);
        if (lane >= o) run += y;
    }
    run -= tot;
    return run;
}

// The two stage maps of a window from its histogram, by one warp: lane l holds the counts of the PER
// bins d = PER l - L ... (v[i]: +1 group low 16 bits, -1 group high 16; run: the counts of the bins
// before).  The members of a group in
// flip order are the bins in d order, so a bin with h members of which C come before it in the group
// holds a_k = d + 2C, d + 2C + 2, ...: h consecutive lattice intervals, one run of mask bits.
// out[0] = +1 group (flips iff a_k <= x), out[1] = -1 group (flips iff a_k <= -x).
template <int PER>
__device__ __forceinline__ void stage_maps_of(const uint32_t (&v)[PER], uint32_t run, int L, StageMap *out)
{
    const int lane = threadIdx.x & 31;
    unsigned long long kp = 0, km = 0;
    int32_t cle = 0, cge = 0;
    {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int32_t d = lane * PER + i - L;
            const int32_t hp = (int32_t)(v[i] & 0xFFFFu), hm = (int32_t)(v[i] >> 16);
            if (hp) {
                // a in (x_j, x_j + 2] clears step j; a <= -NT (j < 0) counts into ylo
                const int32_t j0 = (d + 2 * (int32_t)(run & 0xFFFFu) + NT - 1) >> 1;
                const int32_t lo = max(j0, 0), cnt = hp - (lo - j0);
                cle += hp - max(cnt, 0);
                if (cnt > 0 && lo < NT) kp |= (cnt >= NT ? ~0ull : (1ull << cnt) - 1ull) << lo;
            }
            if (hm) {
                // b = -a in [x_j, x_j + 2) clears step j; b >= -NT (j >= 0) counts into ylo
                const int32_t jt = (NT - (d + 2 * (int32_t)(run >> 16))) >> 1;
                const int32_t lo = max(jt - hm + 1, 0), cnt = jt - lo + 1;
                cge += max(cnt, 0);
                if (cnt > 0 && lo < NT) km |= (cnt >= NT ? ~0ull : (1ull << cnt) - 1ull) << lo;
            }
            run += v[i];
        }
    }
    const uint32_t kp0 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)kp);
    const uint32_t kp1 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(kp >> 32));
    const uint32_t km0 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)km);
    const uint32_t km1 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(km >> 32));
    const uint32_t cc = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)cle | ((uint32_t)cge << 16));
    if (lane == 0) {
        out[0].mask = ~(((unsigned long long)kp1 << 32) | kp0) & STEP_MASK;
        out[0].ylo = -(int32_t)(cc & 0xFFFFu);
        out[1].mask = ~(((unsigned long long)km1 << 32) | km0) & STEP_MASK;
        out[1].ylo = (int32_t)(cc >> 16);
    }
}

// The two stage maps of one window (positions [ws, ws + wlen), wlen <= 32 * S) for replica r, by one
// warp.  Nothing is sorted: the lattice sees thresholds only through the histogram of their distance d
// from c (d in the group's flip direction), so one shared atomic per member and one scan of the bins
// replace a sorting network of 36 stages.
//   * d > NT never flips on the lattice and is left out (+1: a_k >= d > 62; -1: a_k > 64).
//   * No member below -62 (the common case): 128 bins, four per lane.  Otherwise 256 bins from -190
//     on, the first taking everything below: with at most 64 members there, each has a_k <= -64 and
//     flips at every lattice point whatever its distance; with more, at least 64 flip at every lattice
//     point and the window leaves the lattice from each, which is also what the counts then say.
// bins: WBINS words of this warp's own, 16-byte aligned.
template <int S>
__device__ __forceinline__ void window_maps(const int32_t *gam_r, const uint8_t *s0, int ws, int wlen, int r,
                                            int32_t c, uint32_t *bins, StageMap *out)
{
    const int lane = threadIdx.x & 31;
    int32_t dv[S];
    uint32_t ng = 0;                      // bit s: member s is in the -1 group
    bool wide = false;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const int pos = s * 32 + lane;
        dv[s] = NT + 1;
        if (pos < wlen) {
            const int32_t g = gam_r[ws + pos];
            const uint32_t neg = (s0[ws + pos] >> r) & 1u;
            dv[s] = neg ? c - g : g - c;
            ng |= neg << s;
            wide |= dv[s] < -62;
        }
    }
    const bool w = __any_sync(0xFFFFFFFFu, wide);
    uint4 *b4 = reinterpret_cast<uint4 *>(bins);
    b4[lane] = make_uint4(0u, 0u, 0u, 0u);
    if (w) b4[lane + 32] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    const int L = w ? BIN_L : 62;
#pragma unroll
    for (int s = 0; s < S; ++s)
        if (dv[s] <= NT) atomicAdd(&bins[max(dv[s] + L, 0)], (ng >> s) & 1u ? 0x10000u : 1u);
    __syncwarp();
    if (!w) {
        const uint4 q = b4[lane];
        const uint32_t v[4] = {q.x, q.y, q.z, q.w};
        stage_maps_of<4>(v, bins_before<4>(v), 62, out);
    } else {
        const uint4 q = b4[2 * lane], p = b4[2 * lane + 1];
        const uint32_t v[8] = {q.x, q.y, q.z, q.w, p.x, p.y, p.z, p.w};
        stage_maps_of<8>(v, bins_before<8>(v), BIN_L, out);
    }
    __syncwarp();
}

// The same for windows of any size (up to 32,767: counts share words), members read from shared memory:
// positions [p0, p1) of a window counted into its WBINS bins (zeroed) by one warp; several warps may
// count parts of one window.  bins_to_maps then reads the maps off them.
__device__ __forceinline__ void count_members(const int32_t *gam_r, const uint8_t *s0, int p0, int p1, int r, int32_t c,
                                              uint32_t *bins)
{
    for (int i = p0 + (int)(threadIdx.x & 31); i < p1; i += 32) {
        const int32_t g = gam_r[i];
        const bool neg = (s0[i] >> r) & 1u;
        const int32_t d = neg ? c - g : g - c;
        if (d <= NT) atomicAdd(&bins[max(d + BIN_L, 0)], neg ? 0x10000u : 1u);
    }
}

__device__ __forceinline__ void bins_to_maps(const uint32_t *bins, StageMap *out)
{
    const uint4 *b4 = reinterpret_cast<const uint4 *>(bins);
    const int lane = threadIdx.x & 31;
    const uint4 q = b4[2 * lane], p = b4[2 * lane + 1];
    const uint32_t v[8] = {q.x, q.y, q.z, q.w, p.x, p.y, p.z, p.w};
    stage_maps_of<8>(v, bins_before<8>(v), BIN_L, out);
}

static __device__ __forceinline__ int stage_apply(const StageMap &m, int t)
{
    if (t < 0) return -1;
    const int y = m.ylo + __popcll(m.mask & ((1ull << t) - 1ull));
    return (y >= 0 && y < NT) ? y : -1;
}

// a window's 32 * PER bins (distance -L first) to inclusive prefix counts in place, by one warp; its stage
// maps too (out != null)
template <int PER>
__device__ __forceinline__ void bins_to_prefix(uint32_t *bins, int L, StageMap *out)
{
    uint4 *b4 = reinterpret_cast<uint4 *>(bins);
    const int lane = threadIdx.x & 31;
    uint32_t v[PER], c[PER];
#pragma unroll
    for (int i = 0; i < PER / 4; ++i) {
        const uint4 q = b4[PER / 4 * lane + i];
        v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
    }
    const uint32_t run = bins_before<PER>(v);
    c[0] = run + v[0];
#pragma unroll
    for (int i = 1; i < PER; ++i) c[i] = c[i - 1] + v[i];
#pragma unroll
    for (int i = 0; i < PER / 4; ++i)
        b4[PER / 4 * lane + i] = make_uint4(c[4 * i], c[4 * i + 1], c[4 * i + 2], c[4 * i + 3]);
    if (out) stage_maps_of<PER>(v, run, L, out);
    __syncwarp();
}

// prefix counts of one window: bin i holds the members with distance <= i - L; full: none lies below -L
struct WindowCounts {
    const uint32_t *pre;                // null: none kept
    int32_t c;                          // reference G of the distances
    int L;
    bool full;
};

// A group's flips off a window's prefix counts (shift sh: 0 = +1 group, 16 = -1 group), by one warp.
// z = the entering G's distance from the bins' reference on the group's flipping side, so that a member
// with distance d has margin e = z - d and #{e >= y} = C(z - y).  K: known, or -1 and found.  Members with
// e > y flip, and of those with e == y the first `left`.  False when the bins do not reach that far.
__device__ __forceinline__ bool binned_flips(const WindowCounts &wc, int sh, int32_t z, int32_t &K, int32_t &y, int32_t &left)
{
    if (z > NT) return false;
    const int lane = threadIdx.x & 31;
    const int i0 = z + wc.L;
    auto at = [&](int i) { return i < 0 ? 0 : (int32_t)((wc.pre[i] >> sh) & 0xFFFFu); };
    if (K < 0) {
        for (int k0 = 0; K < 0; k0 += 32) {
            const int i = i0 - 2 * (k0 + lane);
            const unsigned hit = __ballot_sync(0xFFFFFFFFu, (i >= 0 || wc.full) && at(i) <= k0 + lane);
            if (hit) K = k0 + __ffs(hit) - 1;
            else if (i0 - 2 * (k0 + 32) < 0) return false;
        }
    }
    y = INT32_MAX;
    left = 0;
    if (K == 0) return true;
    const int i = i0 - 2 * K;
    if (i < 0 && !wc.full) return false;
    const int32_t n0 = at(i), n1 = at(i + 1), n2 = at(i + 2);
    int32_t ties = 0;
    y = 2 * K - 1;
    if (n0 != K) {
        if (n1 >= K) {
            left = K - n0;
            ties = n1 - n0;
        } else {
            y = 2 * K - 2;
            left = K - n1;
            ties = n2 - n1;
        }
        if (left == ties) { --y; left = 0; }
    }
    return true;
}

// Replay of one window (positions [ws, we)) of replica r from the exact entering G g, by one warp: both
// groups in order; emit(wbits) takes the flips, bit l of wbits[s] for position ws + 32 s + l.  With e = the distance of a member's threshold
// on the flipping side of G, the members flip in e order and the k-th (from 0) flips iff e >= 2k, so with
// N(y) = #{e >= y} the number of flips is K = max{k : N(2k - 2) >= k}, and as N(2K) <= K <= N(2K - 2)
// the last of them has e >= 2K, = 2K - 1 or = 2K - 2: three counts give the threshold, and equal
// members flip in position order.  K1, K2: the flips of the first and second group when the stage
// maps gave them (the window was entered on the lattice), else -1: searched, four-way, three counts
// to a reduction.  wc: the window's prefix counts, which answer all of this in a few reads where
// they reach.  Returns G after the window.
template <int SL, class Emit>
__device__ __forceinline__ int32_t replay_window(const int32_t *gr, const uint8_t *s0, int r, int ws, int we,
                                                 int32_t g, bool plus_first, int K1, int K2, const WindowCounts &wc,
                                                 const Emit &emit)
{
    static_assert(32 * SL < 1024, "three counts share a word");
    const int lane = threadIdx.x & 31;
    // members of the window in registers (slot s = positions ws + 32 s + lane)
    int32_t gv[SL];
    uint32_t ng = 0, vd = 0;            // bit s: member is -1 / exists
#pragma unroll
    for (int s = 0; s < SL; ++s) {
        const int i = ws + 32 * s + lane;
        gv[s] = 0;
        if (i < we) {
            gv[s] = gr[i];
            vd |= 1u << s;
            ng |= ((uint32_t)(s0[i] >> r) & 1u) << s;
        }
    }
    // both groups off the counts: one pass over the members, each against its group's cut
    if (wc.pre) {
        int32_t Ka = K1, Kb = K2, ya, yb, la, lb;
        const int32_t xa = plus_first ? g - wc.c : wc.c - g;             // on the first group's side
        if (binned_flips(wc, plus_first ? 0 : 16, xa, Ka, ya, la)) {
            const int32_t xb = 2 * Ka - xa;                              // on the second's, after it
            if (binned_flips(wc, plus_first ? 16 : 0, xb, Kb, yb, lb)) {
                // members at distance d < c* flip, and of those at c* the first l*
                const int32_t ca = Ka ? xa - ya : INT32_MIN, cb = Kb ? xb - yb : INT32_MIN;
                const int32_t cp = plus_first ? ca : cb, cm = plus_first ? cb : ca;
                int32_t lp = plus_first ? la : lb, lm = plus_first ? lb : la;
                uint32_t wbits[SL];
                const unsigned before = (1u << lane) - 1u;
#pragma unroll
                for (int s = 0; s < SL; ++s) {
                    const bool neg = (ng >> s) & 1u, in = (vd >> s) & 1u;
                    const int32_t d = neg ? wc.c - gv[s] : gv[s] - wc.c, cut = neg ? cm : cp;
                    bool f = in && d < cut;
                    if (lp | lm) {
                        const bool tie = in && d == cut;
                        const unsigned tn = __ballot_sync(0xFFFFFFFFu, tie && neg), tp = __ballot_sync(0xFFFFFFFFu, tie && !neg);
                        f |= tie && __popc((neg ? tn : tp) & before) < (neg ? lm : lp);
                        lp = max(lp - __popc(tp), 0);
                        lm = max(lm - __popc(tn), 0);
                    }
                    wbits[s] = __ballot_sync(0xFFFFFFFFu, f);
                }
                emit(wbits);
                return g + (plus_first ? 2 * (Kb - Ka) : 2 * (Ka - Kb));
            }
        }
    }
    uint32_t wbits[SL];
#pragma unroll
    for (int s = 0; s < SL; ++s) wbits[s] = 0;
#pragma unroll 1
    for (int ph = 0; ph < 2; ++ph) {
        const bool plus = plus_first == (ph == 0);
        const uint32_t mem = vd & (plus ? ~ng : ng);
        int32_t e[SL];
#pragma unroll
        for (int s = 0; s < SL; ++s) e[s] = (mem >> s) & 1u ? (plus ? g - gv[s] : gv[s] - g) : -1;
        // #{e >= y0}, #{e >= y1}, #{e >= y2} in bits 0, 10 and 20
        auto count3 = [&](int32_t y0, int32_t y1, int32_t y2) {
            uint32_t n = 0;
#pragma unroll
            for (int s = 0; s < SL; ++s)
                n += (e[s] >= y0 ? 1u : 0u) + (e[s] >= y1 ? 1u << 10 : 0u) + (e[s] >= y2 ? 1u << 20 : 0u);
            return __reduce_add_sync(0xFFFFFFFFu, n);
        };
        int32_t K = ph == 0 ? K1 : K2, y, left;
        if (K < 0) {
            int32_t n0 = 0;
#pragma unroll
            for (int s = 0; s < SL; ++s) n0 += e[s] >= 0 ? 1 : 0;
            n0 = __reduce_add_sync(0xFFFFFFFFu, n0);
            int32_t lo = min(n0, 1), hi = n0;
            while (lo < hi) {
                const int32_t sp = hi - lo;
                const int32_t m1 = lo + ((sp + 3) >> 2), m2 = lo + ((2 * sp + 3) >> 2), m3 = lo + ((3 * sp + 3) >> 2);
                const uint32_t n = count3(2 * m1 - 2, 2 * m2 - 2, 2 * m3 - 2);
                if ((int32_t)(n >> 20) >= m3) lo = m3;
                else if ((int32_t)((n >> 10) & 1023u) >= m2) { lo = m2; hi = m3 - 1; }
                else if ((int32_t)(n & 1023u) >= m1) { lo = m1; hi = m2 - 1; }
                else hi = m1 - 1;
            }
            K = lo;
        }
        y = 2 * K - 1;
        left = 0;
        if (K > 0) {
            const uint32_t n = count3(2 * K, 2 * K - 1, 2 * K - 2);
            const int32_t n0 = n & 1023u, n1 = (n >> 10) & 1023u, n2 = n >> 20;
            if (n0 != K) {
                if (n1 < K) --y;
                left = n1 >= K ? K - n0 : K - n1;
                if (left == (n1 >= K ? n1 - n0 : n2 - n1)) { --y; left = 0; }
            }
        }
        if (K == 0) continue;
        if (left == 0) {
#pragma unroll
            for (int s = 0; s < SL; ++s) wbits[s] |= __ballot_sync(0xFFFFFFFFu, e[s] > y);
        } else {
#pragma unroll
            for (int s = 0; s < SL; ++s) {
                const unsigned tm = __ballot_sync(0xFFFFFFFFu, e[s] == y);
                const int32_t idx = __popc(tm & ((1u << lane) - 1u));
                wbits[s] |= __ballot_sync(0xFFFFFFFFu, e[s] > y || (e[s] == y && idx < left));
                left -= __popc(tm);
            }
        }
        g = plus ? g - 2 * K : g + 2 * K;
    }
    emit(wbits);
    return g;
}

// the flips of a window (positions [ws, we)) into a flip bitmap.  With W a multiple of 32 every window
// owns whole words; otherwise windows share words and OR their bits in atomically, so windows may be
// replayed concurrently.
template <int SL>
__device__ __forceinline__ void flips_to_bitmap(const uint32_t (&wbits)[SL], int ws, int we, uint32_t *fb, int W)
{
    const int lane = threadIdx.x & 31;
    if ((W & 31) == 0) {
#pragma unroll
        for (int s = 0; s < SL; ++s)
            if (lane == s && ws + 32 * s < we) fb[(ws >> 5) + s] = wbits[s];
    } else if (lane == 0) {
        const int sh = ws & 31;
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            if (!wbits[s]) continue;
            const int q = (ws >> 5) + s;
            atomicOr(&fb[q], wbits[s] << sh);
            if (sh) atomicOr(&fb[q + 1], wbits[s] >> (32 - sh));
        }
    }
}

// The same for windows of any size, members read from shared memory in each pass; emit(i0, bits) takes the
// flips of positions i0 .. i0 + 31 (once per group).
template <class Emit>
__device__ __noinline__ int32_t replay_large(const int32_t *gr, const uint8_t *s0, int r, int ws, int we, int32_t g,
                                             bool plus_first, int K1, int K2, const WindowCounts &wc, const Emit &emit)
{
    const int lane = threadIdx.x & 31;
    for (int ph = 0; ph < 2; ++ph) {
        const bool plus = plus_first == (ph == 0);
        auto margin = [&](int i) {
            const bool neg = (s0[i] >> r) & 1u;
            return plus == neg ? -1 : (plus ? g - gr[i] : gr[i] - g);
        };
        auto count = [&](int32_t y) {
            int32_t n = 0;
            for (int i = ws + lane; i < we; i += 32) n += margin(i) >= y ? 1 : 0;
            return (int32_t)__reduce_add_sync(0xFFFFFFFFu, n);
        };
        int32_t K = ph == 0 ? K1 : K2, y, left;
        if (!wc.pre || !binned_flips(wc, plus ? 0 : 16, plus ? g - wc.c : wc.c - g, K, y, left)) {
            if (K < 0) {
                int32_t hi = count(0), lo = min(hi, 1);
                while (lo < hi) {
                    const int32_t mid = (lo + hi + 1) >> 1;
                    if (count(2 * mid - 2) >= mid) lo = mid; else hi = mid - 1;
                }
                K = lo;
            }
            y = 2 * K - 1;
            left = 0;
            if (K > 0) {
                const int32_t n0 = count(2 * K), n1 = count(2 * K - 1);
                if (n0 != K && n1 < K) --y;
                left = n0 == K ? 0 : (n1 >= K ? K - n0 : K - n1);
            }
        }
        if (K == 0) continue;
        for (int i0 = ws; i0 < we; i0 += 32) {
            const int32_t e = i0 + lane < we ? margin(i0 + lane) : INT32_MIN;
            const unsigned tm = __ballot_sync(0xFFFFFFFFu, e == y);
            const int32_t idx = __popc(tm & ((1u << lane) - 1u));
            const unsigned bits = __ballot_sync(0xFFFFFFFFu, e > y || (e == y && idx < left));
            left -= min(left, __popc(tm));
            if (bits) emit(i0, bits);
        }
        g = plus ? g - 2 * K : g + 2 * K;
    }
    return g;
}

// flips of both groups of a window entered at lattice index t (-1: off the lattice), in order: -1 from
// where its stage maps leave the lattice
__device__ __forceinline__ void mapped_flips(bool plus_first, int t, const StageMap *maps, int &K1, int &K2)
{
    K1 = K2 = -1;
    const int u = stage_apply(maps[plus_first ? 0 : 1], t);
    if (u >= 0) {
        K1 = plus_first ? t - u : u - t;
        const int v = stage_apply(maps[plus_first ? 1 : 0], u);
        if (v >= 0) K2 = plus_first ? v - u : u - v;
    }
}

// replay_window for a window entered at lattice index t with its stage maps
template <int SL, class Emit>
__device__ __forceinline__ int32_t replay_mapped(const int32_t *gr, const uint8_t *s0, int r, int ws, int we, int32_t g,
                                                 bool plus_first, int t, const StageMap *maps,
                                                 const WindowCounts &wc, const Emit &emit)
{
    int K1, K2;
    mapped_flips(plus_first, t, maps, K1, K2);
    return replay_window<SL>(gr, s0, r, ws, we, g, plus_first, K1, K2, wc, emit);
}

}  // namespace win
}  // namespace gdi
