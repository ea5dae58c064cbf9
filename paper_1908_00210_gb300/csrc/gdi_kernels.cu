// gdi_kernels.cu -- sm_103a kernels of libgdi.so: the GDI annealing sweep (Algorithm 3 of
// Cook, Jin, Tan, arXiv:1908.00210), its initial state, the exact-balance repair and the cut.
//
// CTA-resident path: one thread block anneals one (instance, replica) at a time with the whole
// spin vector in shared memory (int8 per vertex); the rank-space CSR streams from L2/HBM.  The
// block loops over its work items (persistent), sweeps, colour classes and windows without
// leaving the kernel, so an anneal of M sweeps is one launch.
//
// Work items are taken from a size-sorted queue (an atomic counter over the largest-first order),
// so long instances start first and short ones fill the tail.
//
// Per window (a chunk of W consecutive ranks of one colour class):
//   1. thresholds: for every spin, the local field h_i = sum_j w_ij s_j over its CSR row (Eq. 2),
//      a Philox4x32-10 draw u_i, the largest energy change E*(u_i) that the draw accepts (binary
//      search of the table row), and from it the flip threshold in G:
//        s_i = +1 flips iff G >= gamma_i = ceil((B h_i + 4A - E*) / 4A)
//        s_i = -1 flips iff G <= gamma_i = floor((E* + B h_i - 4A) / 4A)
//      (dE = B s_i h_i + 4A (1 - s_i G), Eq. 4-6 with G counting the other spins).
//   2. the +1 group and the -1 group of the window each see the exact running G in threshold
//      order (Algorithm 3's atomically updated G, serialised): with e_i = G - gamma_i (+1 group) or
//      gamma_i - G (-1 group), the k-th spin in e-descending order flips iff e_(k) >= 2k, ties by rank.
//      The number of flips K and the last margin come from counts of e, not from a sort.
//   3. G changes by -2K (+1 group) or +2K (-1 group): one shared-memory update per group, the
//      block-level analogue of the paper's atomicAdd on G.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "gdi_device.cuh"
#include "gdi_internal.h"
#include "gdi_window.cuh"

namespace {

using namespace gdi;
using namespace gdi::win;

// ---------------------------------------------------------------------------------------------
struct Smem {
    int8_t *sig;        // [max_n] spins of the current item, rank order
    int8_t *flag;       // [max_n] repair decisions (during the sweeps: bins)
    uint32_t *row;      // [1 or 2][row_stride] table rows
    int32_t *red32;     // [BS/32 + 2]
    int64_t *red64;     // [BS/32 + 2]
    int32_t *G;         // running magnetisation of the item
};

// h_i = sum_j w_ij s_j over the CSR row of local rank r (Eq. 2)
__device__ __forceinline__ int32_t local_field(const GdiDevProblem &P, int64_t base, int32_t r,
                                               const int8_t *sig)
{
    const int64_t e0 = P.row_ptr[base + r], e1 = P.row_ptr[base + r + 1];
    int32_t h = 0;
    for (int64_t e = e0; e < e1; ++e) {
        const uint32_t c = __ldg(P.col + e);
        const int32_t s = sig[c & 0x7FFFFFFFu];
        h += (c >> 31) ? -s : s;
    }
    return h;
}

// Algorithm 2 (the paper's standard annealer, GDI_FLAG_STANDARD): every spin of the window forms
// the balance term from the complete graph of Eq. 5, i.e. sums all n spins itself (an O(n) read per
// spin, which is what the decoupled G of Algorithm 3 removes), on the state at the window start,
// and flips iff its draw accepts dE = B s h + 4A (1 - s G) -- the same test as "G >= gamma" with
// the threshold gamma of step 1.  All decisions are taken before any spin of the window changes.
// The sums are read 16 spins at a time (every lane of a warp reads the same 16 bytes) into four
// independent dot-product chains.
template <int BS>
__device__ void standard_window(const Smem &S, const int32_t *gam, const int8_t *s0, int32_t wlo, int32_t Wn, int32_t n)
{
    int32_t dG = 0;
    const uint4 *sv = reinterpret_cast<const uint4 *>(S.sig);    // 16-byte aligned by the layout
    const int32_t nv = n >> 4;
    for (int32_t p = threadIdx.x; p < Wn; p += BS) {
        int32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;     // sum of all spins, read by this spin
#pragma unroll 4
        for (int32_t k = 0; k < nv; ++k) {
            const uint4 v = sv[k];
            a0 = __dp4a((int)v.x, 0x01010101, a0);
            a1 = __dp4a((int)v.y, 0x01010101, a1);
            a2 = __dp4a((int)v.z, 0x01010101, a2);
            a3 = __dp4a((int)v.w, 0x01010101, a3);
        }
        for (int32_t j = 16 * nv; j < n; ++j) a0 += S.sig[j];
        const int32_t G = (a0 + a1) + (a2 + a3);
        const int sg = s0[p];
        const bool flip = sg > 0 ? G >= gam[p] : G <= gam[p];
        S.flag[wlo + p] = flip ? 1 : 0;
        dG += flip ? -2 * sg : 0;
    }
    dG = block_sum<BS, int32_t>(dG, S.red32);
    for (int32_t p = threadIdx.x; p < Wn; p += BS)
        if (S.flag[wlo + p]) S.sig[wlo + p] = (int8_t)(-s0[p]);
    if (threadIdx.x == 0) *S.G += dG;
}

// #majority spins with repair key (s_i h_i) <= x, and with key == x (when eq != null)
template <int BS>
__device__ int32_t repair_count(const GdiDevProblem &P, int64_t base, int32_t n, const Smem &S,
                                int maj, int64_t x, bool strict)
{
    int32_t c = 0;
    for (int32_t r = threadIdx.x; r < n; r += BS) {
        if (S.sig[r] != maj) continue;
        const int64_t key = (int64_t)maj * local_field(P, base, r, S.sig);
        c += strict ? (key < x) : (key <= x);
    }
    return block_sum<BS, int32_t>(c, S.red32);
}

// Exact-balance repair: flip the k majority spins with the smallest (s_i h_i, rank) keys.
template <int BS>
__device__ void repair(const GdiDevProblem &P, int64_t base, int32_t n, const Smem &S)
{
    __syncthreads();
    const int32_t G = *S.G;
    const int32_t target = n & 1;
    const int32_t aG = G < 0 ? -G : G;
    if (aG <= target) return;
    const int32_t k = (aG - target) / 2;
    const int maj = G > 0 ? 1 : -1;
    // kappa = smallest key value with count(key <= kappa) >= k ; keys lie in [-deg, deg]
    int64_t lo = -(int64_t)P.max_degree - 1, hi = (int64_t)P.max_degree + 1;
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (repair_count<BS>(P, base, n, S, maj, mid, false) >= k) hi = mid; else lo = mid + 1;
    }
    const int64_t kappa = lo;
    const int32_t less = repair_count<BS>(P, base, n, S, maj, kappa, true);
    const int32_t t = k - less;
    const int32_t chunk = (n + BS - 1) / BS;
    const int32_t p0 = threadIdx.x * chunk, p1 = min(p0 + chunk, n);
    // keys of my chunk are recomputed below before any spin of the item changes: compute flags first
    int32_t ties = 0;
    for (int32_t r = p0; r < p1; ++r) {
        if (S.sig[r] != maj) continue;
        ties += ((int64_t)maj * local_field(P, base, r, S.sig) == kappa);
    }
    int32_t total;
    int32_t idx = block_excl_scan<BS>(ties, S.red32, &total);
    // decide every flip before writing any spin (keys are defined on the pre-repair state)
    for (int32_t r = p0; r < p1; ++r) {
        int8_t f = 0;
        if (S.sig[r] == maj) {
            const int64_t key = (int64_t)maj * local_field(P, base, r, S.sig);
            bool flip = key < kappa;
            if (key == kappa) flip = (idx++ < t);
            f = flip ? 1 : 0;
        }
        S.flag[r] = f;
    }
    __syncthreads();
    for (int32_t r = threadIdx.x; r < n; r += BS)
        if (S.flag[r]) S.sig[r] = (int8_t)(-maj);
    __syncthreads();
    if (threadIdx.x == 0) *S.G = G - 2 * maj * k;
    __syncthreads();
}

// One pass over the item's rows, a team of lanes per row: the item's cut (the sum of the weights whose
// ends differ, / 2).  mode 1: also counts the repair keys s_i h_i of the majority spins in hist[key + D];
// mode 2: instead marks each majority spin's flag, 1 for a key below kappa and 2 for one equal to it.
template <int BS>
__device__ int64_t item_fields(const GdiDevProblem &P, int64_t base, int32_t n, int32_t mean_deg, const Smem &S, int mode,
                               int maj, int32_t *hist, int32_t kappa)
{
    const int tl = mean_deg >= 16 ? 3 : (mean_deg >= 8 ? 2 : (mean_deg >= 4 ? 1 : 0));
    const int T = 1 << tl, sub = threadIdx.x & (T - 1);
    int64_t c = 0;
    for (int32_t k0 = 0; k0 < n; k0 += BS >> tl) {
        const int32_t i = k0 + ((int32_t)threadIdx.x >> tl);
        int32_t diff = 0, deg = 0;                      // weights of the differing neighbours, of all
        int8_t si = 0;
        if (i < n) {
            si = S.sig[i];
            const int64_t e0 = P.row_ptr[base + i], e1 = P.row_ptr[base + i + 1];
            if (P.col16) {
                for (int64_t e = e0 + sub; e < e1; e += T) {
                    const uint32_t cc = __ldg(P.col16 + e);
                    const int32_t w = (cc >> 15) ? -1 : 1;
                    deg += w;
                    diff += S.sig[cc & 0x7FFFu] != si ? w : 0;
                }
            } else {
                for (int64_t e = e0 + sub; e < e1; e += T) {
                    const uint32_t cc = __ldg(P.col + e);
                    const int32_t w = (cc >> 31) ? -1 : 1;
                    deg += w;
                    diff += S.sig[cc & 0x7FFFFFFFu] != si ? w : 0;
                }
            }
        }
        c += diff;
        if (mode) {
            int32_t key = deg - 2 * diff;                // s_i h_i
            for (int o = T >> 1; o >= 1; o >>= 1) key += __shfl_xor_sync(0xFFFFFFFFu, key, o);
            if (i < n && sub == 0) {
                if (mode == 1) {
                    if (si == maj) atomicAdd(&hist[key + P.max_degree], 1);
                } else {
                    S.flag[i] = si != maj ? 0 : (key < kappa ? 1 : (key == kappa ? 2 : 0));
                }
            }
        }
    }
    return block_sum<BS, int64_t>(c, S.red64) / 2;
}

// Results of an annealed item: cut and G before and after the exact-balance repair (the k majority spins
// with the smallest (s_i h_i, rank) keys flip).  The keys are counted in scratch while the cut is taken,
// so the repair costs two more passes over the rows; where 2 max_degree + 1 bins do not fit the scratch,
// the key bound is searched instead, a pass per step.  Ends with a block barrier.
template <int BS>
__device__ void finish_item(const GdiDevProblem &P, const GdiDevRun &R, int64_t base, int32_t n, int32_t mean_deg,
                            const Smem &S, int32_t *scratch, int scratch_words, int32_t item, bool write)
{
    __shared__ int32_t sel[2];
    __syncthreads();
    const int32_t raw_G = *S.G;
    const int32_t target = n & 1, aG = raw_G < 0 ? -raw_G : raw_G;
    const bool fix = !(R.flags & GDI_DEV_NO_REPAIR) && aG > target;
    const int32_t nb = 2 * P.max_degree + 1;
    const bool counted = fix && nb <= scratch_words;
    const int maj = raw_G > 0 ? 1 : -1;
    if (counted) {
        for (int32_t b = threadIdx.x; b < nb; b += BS) scratch[b] = 0;
        __syncthreads();
    }
    const int64_t raw_cut = item_fields<BS>(P, base, n, mean_deg, S, counted ? 1 : 0, maj, scratch, 0);
    int64_t fin_cut = raw_cut;
    if (counted) {
        const int32_t k = (aG - target) / 2;
        __syncthreads();
        if (threadIdx.x < 32) {
            // kappa = the smallest key with k keys at or below it; t = how many keys equal to it flip
            const int lane = threadIdx.x;
            int32_t before = 0;
            for (int32_t b0 = 0; b0 < nb; b0 += 32) {
                int32_t x = b0 + lane < nb ? scratch[b0 + lane] : 0;
                const int32_t own = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
                    if (lane >= o) x += y;
                }
                const unsigned m = __ballot_sync(0xFFFFFFFFu, before + x >= k);
                if (m) {
                    const int f = __ffs(m) - 1;
                    if (lane == f) {
                        sel[0] = b0 + f - P.max_degree;
                        sel[1] = k - (before + x - own);
                    }
                    break;
                }
                before += __shfl_sync(0xFFFFFFFFu, x, 31);
            }
        }
        __syncthreads();
        const int32_t kappa = sel[0], t = sel[1];
        item_fields<BS>(P, base, n, mean_deg, S, 2, maj, nullptr, kappa);
        __syncthreads();
        // equal keys flip in rank order: contiguous chunks keep it
        const int32_t chunk = (n + BS - 1) / BS;
        const int32_t p0 = min((int32_t)threadIdx.x * chunk, n), p1 = min(p0 + chunk, n);
        int32_t ties = 0;
        for (int32_t r = p0; r < p1; ++r) ties += S.flag[r] == 2;
        int32_t total;
        int32_t idx = block_excl_scan<BS>(ties, S.red32, &total);
        for (int32_t r = p0; r < p1; ++r) {
            const int f = S.flag[r];
            if (f == 1 || (f == 2 && idx++ < t)) S.sig[r] = (int8_t)-maj;
        }
        if (threadIdx.x == 0) *S.G = raw_G - 2 * maj * k;
        __syncthreads();
        fin_cut = item_fields<BS>(P, base, n, mean_deg, S, 0, 0, nullptr, 0);
    } else if (fix) {
        repair<BS>(P, base, n, S);
        fin_cut = item_fields<BS>(P, base, n, mean_deg, S, 0, 0, nullptr, 0);
    }
    __syncthreads();
    if (threadIdx.x == 0 && write) {
        R.raw_G[item] = raw_G;
        R.raw_cut[item] = raw_cut;
        R.final_G[item] = *S.G;
        R.final_cut[item] = fin_cut;
    }
    __syncthreads();
}

__host__ __device__ inline size_t align16c(size_t x) { return (x + 15) & ~(size_t)15; }

// what a launch keeps in shared memory beyond the necessary (GdiDevRun::cta_opts)
constexpr int CTA_OPT_ROWS2 = 1;    // the next sweep's table row beside the current one
constexpr int CTA_OPT_ES = 2;       // whole-block windows: the next window's E* (else drawn in place)
constexpr int CTA_OPT_BINS = 4;     // whole-block windows: 512 bins of margins (else 16)
// GdiDevRun::cta_stage: columns the staging buffer holds (rows beyond are read from global memory);
// cta_rofs: row offsets beside it.  Where a block's rows of all classes fit both, they are staged once per
// item, else the next class's (window's) while the current one is decided.

// lanes per rank of a field sum: the layout whose longest chain of dependent reads is shortest
// (rounds x (row / T + about 4 reads' worth of reduction and threshold latency per round))
template <int BS>
__device__ __forceinline__ int team_log2(int32_t nown, int32_t mean_deg)
{
    int best = 0x7FFFFFFF, tl = 0;
    for (int l = 0; l <= 5; ++l) {
        const int32_t rounds = ((nown << l) + BS - 1) / BS;
        const int32_t chain = rounds * (((mean_deg + (1 << l) - 1) >> l) + 4);
        if (chain < best) { best = chain; tl = l; }
    }
    return tl;
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// E* of ranks [r0, r1) of an item at sweep sw (table row `row` of length rlen) into es[r - org], by threads
// t of nth: one Philox call per aligned quad of ranks
__device__ __forceinline__ void draw_estar(const GdiDevRun &R, int32_t r0, int32_t r1, int32_t org, int32_t q, int32_t rep,
                                           int32_t sw, const uint32_t *row, int32_t rlen, float Tsw, int32_t *es, int t,
                                           int nth)
{
    if (r1 <= r0) return;
    for (int32_t qd = (r0 >> 2) + t; qd <= ((r1 - 1) >> 2); qd += nth) {
        uint4 u4 = philox4x32_10(make_uint4((uint32_t)qd, (uint32_t)sw, (uint32_t)q, (uint32_t)rep), R.key0, R.key1);
        // (rolled: a class is short, so straight-line code is fetched more often than it is reused)
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
            const int32_t r = 4 * qd + j;
            if (r >= r0 && r < r1) es[r - org] = estar_of(row, rlen, R.mode, u4.x, Tsw);
            u4.x = u4.y;
            u4.y = u4.z;
            u4.z = u4.w;
        }
    }
}

// Columns from entry al on (a 16-byte boundary; whole pieces, the column array is padded), `pieces` of
// them, and the offsets from al of nrows rows (bounds rp) into shared memory, by threads t of nth.  The
// caller waits (cp_async_wait_all) before its block barrier.
__device__ __forceinline__ void stage_rows(const GdiDevProblem &P, const int64_t *rp, int32_t nrows, int64_t al, int32_t pieces,
                                           int32_t *rofs, uint16_t *cbuf, int t, int nth)
{
    for (int32_t k = t; k < pieces; k += nth) cp_async16(cbuf + 8 * k, P.col16 + al + 8 * (int64_t)k);
    for (int32_t i = t; i <= nrows; i += nth) rofs[i] = (int32_t)(rp[i] - al);
}

// Both preparations of a class (window) by warps w of nw: the first few draw (about 250 instructions a
// quad), the others stage, so that neither waits for the other's latency
template <class Draw, class Stage>
__device__ __forceinline__ void split_ahead(int32_t nranks, int w, int nw, const Draw &draw, const Stage &stage, bool both)
{
    const int lane = threadIdx.x & 31;
    if (!both) {
        draw(w * 32 + lane, nw * 32);
        return;
    }
    const int quads = (nranks + 3) / 4 + 1;
    const int dw = min((quads + 31) / 32, max(1, 3 * nw / 4));
    if (w < dw) draw(w * 32 + lane, dw * 32);
    if (dw == nw) stage(w * 32 + lane, nw * 32);
    else if (w >= dw) stage((w - dw) * 32 + lane, (nw - dw) * 32);
}

// Flip thresholds of ranks [lo, lo + nr) of an item from the shared spins and E* (es[i], i counted from lo),
// a team of 2^tl lanes per rank; put(i, sign, threshold) by each team's first lane.  rofs != null: row i
// is entries rofs[i] ... from gcol on, the first `lim` of them staged in shared memory.  Teams are
// aligned lane groups of one warp; every lane takes part in every round's shuffles (the round count is the
// block's).  A row of more than `longrow` entries per lane is summed by the whole warp: a power-law
// graph's class holds hubs of hundreds of entries, which one team would keep the block waiting for.
template <int BS, class Put>
__device__ __forceinline__ void team_thresholds(const GdiDevProblem &P, const int8_t *sig, int64_t base, int32_t lo, int32_t nr,
                                                int tl, int32_t longrow, const int32_t *rofs, const uint16_t *cbuf,
                                                int32_t lim, const uint16_t *gcol, const int32_t *es, int a_shift,
                                                const Put &put)
{
    const int T = 1 << tl, sub = threadIdx.x & (T - 1), lane = threadIdx.x & 31;
    const int32_t limit = longrow << tl;
    const bool has_long = P.max_degree > limit;
    // spin of an entry, signed by its weight
    auto spin16 = [&](uint32_t cc) {
        const int32_t sv = sig[cc & 0x7FFFu];
        return (cc >> 15) ? -sv : sv;
    };
    auto spin32 = [&](uint32_t cc) {
        const int32_t sv = sig[cc & 0x7FFFFFFFu];
        return (cc >> 31) ? -sv : sv;
    };
    for (int32_t k0 = 0; k0 < nr; k0 += BS >> tl) {
        const int32_t i = k0 + ((int32_t)threadIdx.x >> tl);
        int32_t h = 0;
        int64_t g0 = 0;                 // rows read from the whole CSR: entries g0 + [e0, e1)
        int32_t e0 = 0, e1 = 0;
        if (i < nr) {
            if (rofs) {
                e0 = rofs[i];
                e1 = rofs[i + 1];
            } else {
                g0 = P.row_ptr[base + lo + i];
                e1 = (int32_t)(P.row_ptr[base + lo + i + 1] - g0);
            }
        }
        // entries first, first + step, ... of a row
        auto sum = [&](int64_t g, int32_t first, int32_t end, int32_t step) {
            int32_t x = 0;
            if (rofs) {
                if (end <= lim) {
#pragma unroll 4
                    for (int32_t e = first; e < end; e += step) x += spin16(cbuf[e]);
                } else {
#pragma unroll 4
                    for (int32_t e = first; e < end; e += step) x += spin16(__ldg(gcol + e));
                }
            } else if (P.col16) {
                for (int32_t e = first; e < end; e += step) x += spin16(__ldg(P.col16 + g + e));
            } else {
#pragma unroll 4
                for (int32_t e = first; e < end; e += step) x += spin32(__ldg(P.col + g + e));
            }
            return x;
        };
        const bool lng = e1 - e0 > limit;
        if (!lng) h = sum(g0, e0 + sub, e1, T);
        for (int o = T >> 1; o >= 1; o >>= 1) h += __shfl_xor_sync(0xFFFFFFFFu, h, o);
        if (has_long) {
            unsigned m = __ballot_sync(0xFFFFFFFFu, lng && sub == 0);
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const int64_t g = __shfl_sync(0xFFFFFFFFu, g0, src);
                const int32_t b = __shfl_sync(0xFFFFFFFFu, e0, src), e = __shfl_sync(0xFFFFFFFFu, e1, src);
                const int32_t x = __reduce_add_sync(0xFFFFFFFFu, sum(g, b + lane, e, 32));
                if (lane == src) h = x;
            }
        }
        if (i < nr && sub == 0) {
            const int sg = sig[lo + i];
            const int32_t e = es[i];
            put(i, sg, a_shift >= 0 ? gamma_of_shift(sg, h, e, P.A, P.B, a_shift) : gamma_of(sg, h, e, P.A, P.B));
        }
    }
}

// ---------------------------------------------------------------------------------------------
// CTA-resident kernel for windows that one warp does not hold: whole colour classes (W = 0), W > 256,
// instances whose class buffers do not fit the counting kernel, and Algorithm 2.  Windows are taken one
// after another from the exact running G.  Per window: every thread counts its thresholds' margins e
// (the distance on the flipping side of the window-start G) into shared bins as it makes them; one warp
// reads both groups' flips off the bins -- members flip in e order, the k-th iff e >= 2k, so the first
// k with N(2k) <= k is the number of flips K, and the last one has e >= 2K, = 2K - 1 or = 2K - 2; the
// second group sees the same margins shifted by the first group's 2K -- and then every thread decides its
// ranks, equal margins by position.  Three block barriers per window, four where a tie is cut; a
// counting pass and a scan per group with its own barriers took about 26.  Draws and rows of the next
// window are prepared by the other warps while one reads the bins, as in the counting kernel.  Measured:
// ER 2000, 8 replicas, whole-class windows, 200 sweeps 23.7 -> 7.3 ms; Algorithm 2 on a 71 x 71 torus, 100 sweeps
// 15.6 -> 8.4 ms (what bounds that are the shared reads of the n-spin sums, 16 bytes each).
struct CtaBlockLayout {
    size_t red64, red32, G, row, sig, flag, gam, es, s0, rofs, cbuf, total;
    int row_stride, nb;
};

__host__ __device__ inline CtaBlockLayout cta_block_layout(const GdiDevProblem &P, int32_t max_row, int BS, int opts,
                                                           int32_t stage)
{
    CtaBlockLayout L;
    const size_t mw = (size_t)P.max_window + 8;
    size_t o = 0;
    L.red64 = o; o = align16c(o + sizeof(int64_t) * (BS / 32 + 2));
    L.red32 = o; o = align16c(o + sizeof(int32_t) * (BS / 32 + 2));
    L.G = o; o = align16c(o + 16);
    L.row_stride = (max_row + 3) & ~3;
    L.row = o; o = align16c(o + sizeof(uint32_t) * (size_t)L.row_stride * ((opts & CTA_OPT_ROWS2) ? 2 : 1));
    L.sig = o; o = align16c(o + (size_t)P.max_n);
    // the repair flags and, during the sweeps, the bins (nb first group, 2 nb second) and the tie counts
    // of 32 ranks each share their bytes
    L.nb = (opts & CTA_OPT_BINS) ? 512 : 16;
    const size_t bins = 4 * (3 * (size_t)L.nb + mw / 32 + 1), fl = (size_t)P.max_n;
    L.flag = o; o = align16c(o + (fl > bins ? fl : bins));
    L.gam = o; o = align16c(o + 4 * (size_t)P.max_window);
    L.es = o; o = align16c(o + ((opts & CTA_OPT_ES) ? 4 * (size_t)P.max_window : 0));
    L.s0 = o; o = align16c(o + (size_t)P.max_window);
    L.rofs = o; o = align16c(o + (stage ? 4 * mw : 0));
    L.cbuf = o; o = align16c(o + 2 * (size_t)stage);
    L.total = o;
    return L;
}

// one group's flips off its bins h[m] (members with margin m < lim), of which n0 members have margin >= 0,
// by one warp: K, and (y, left) such that the members with e > y flip and of those with e == y the first
// `left` in position order.  False when K lies beyond the bins.
__device__ __forceinline__ bool group_flips(const int32_t *h, int lim, int32_t n0, int32_t &K, int32_t &y, int32_t &left)
{
    const int lane = threadIdx.x & 31;
    int32_t above = n0;                                  // members with margin >= m0
    for (int m0 = 0; m0 < lim; m0 += 32) {
        const int m = m0 + lane;
        const int32_t own = m < lim ? h[m] : 0;
        int32_t x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t v = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += v;
        }
        const int32_t N = above - (x - own);             // members with margin >= m
        const unsigned hit = __ballot_sync(0xFFFFFFFFu, !(lane & 1) && m < lim && N <= (m >> 1));
        if (hit) {
            const int f = __ffs(hit) - 1;
            K = (m0 + f) >> 1;
            y = INT32_MAX;
            left = 0;
            if (K == 0) return true;
            const int32_t n2 = __shfl_sync(0xFFFFFFFFu, N, f), h1 = h[2 * K - 1], h2 = h[2 * K - 2];
            int32_t ties = 0;
            if (n2 == K) {
                y = 2 * K - 1;
            } else if (n2 + h1 >= K) {
                y = 2 * K - 1;
                left = K - n2;
                ties = h1;
            } else {
                y = 2 * K - 2;
                left = K - n2 - h1;
                ties = h2;
            }
            if (left && left == ties) { --y; left = 0; }
            return true;
        }
        above -= __shfl_sync(0xFFFFFFFFu, x, 31);
    }
    return false;
}

// count of members of group grp (signs s0) with margin >= x relative to g, block-wide
template <int BS>
__device__ int32_t count_ge(const int32_t *gam, const int8_t *s0, int32_t Wn, int grp, int32_t g, int64_t x, int32_t *red)
{
    int32_t c = 0;
    for (int32_t p = threadIdx.x; p < Wn; p += BS) {
        if (s0[p] != grp) continue;
        const int64_t d = grp > 0 ? (int64_t)g - gam[p] : (int64_t)gam[p] - g;
        c += (d >= x);
    }
    return block_sum<BS, int32_t>(c, red);
}

template <int BS>
__global__ void __launch_bounds__(BS, 1024 / BS) gdi_cta_block_kernel(GdiDevProblem P, GdiDevRun R)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem S = {};
    const bool rows2 = (R.cta_opts & CTA_OPT_ROWS2) != 0, staged = R.cta_stage > 0;
    const bool pre = (R.cta_opts & CTA_OPT_ES) != 0;
    const CtaBlockLayout L = cta_block_layout(P, R.max_row, BS, R.cta_opts, R.cta_stage);
    S.red64 = reinterpret_cast<int64_t *>(smem_raw + L.red64);
    S.red32 = reinterpret_cast<int32_t *>(smem_raw + L.red32);
    S.G = reinterpret_cast<int32_t *>(smem_raw + L.G);
    S.row = reinterpret_cast<uint32_t *>(smem_raw + L.row);
    S.sig = reinterpret_cast<int8_t *>(smem_raw + L.sig);
    S.flag = reinterpret_cast<int8_t *>(smem_raw + L.flag);
    const int NB = L.nb;
    int32_t *h1 = reinterpret_cast<int32_t *>(smem_raw + L.flag);      // [NB] first group, margin 0 ...
    int32_t *h2 = h1 + NB;                                             // [2 NB] second group, margin -NB ...
    int32_t *tcnt = h2 + 2 * NB;                                       // [windows' ranks / 32] ties
    int32_t *gam = reinterpret_cast<int32_t *>(smem_raw + L.gam);
    int32_t *es = pre ? reinterpret_cast<int32_t *>(smem_raw + L.es) : gam;   // in place: E*, then gamma
    int8_t *s0 = reinterpret_cast<int8_t *>(smem_raw + L.s0);
    int32_t *rofs = reinterpret_cast<int32_t *>(smem_raw + L.rofs);
    uint16_t *cbuf = reinterpret_cast<uint16_t *>(smem_raw + L.cbuf);
    {
        // the launch must have given the whole layout (the host sizes it with the same function)
        uint32_t dyn;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
        if ((size_t)dyn < L.total) {
            if (threadIdx.x == 0 && blockIdx.x == 0) atomicCAS(R.err, 0, GDI_DEVERR_INPUT);
            return;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool standard = (R.flags & GDI_DEV_STANDARD) != 0;
    const int a_shift = (P.A > 0 && (P.A & (P.A - 1)) == 0) ? 2 + __ffs(P.A) - 1 : -1;   // log2(4A)
    const int32_t items = P.num_instances * P.replicas;
    __shared__ int32_t next_item;
    __shared__ int32_t nge[2];                          // members with margin >= 0, by group
    struct Decision { int32_t y[2], left[2], slow; };
    __shared__ Decision dec;
    while (true) {
        // persistent blocks take (instance, replica) items from a queue sorted by size, largest
        // first; items are independent, so the assignment does not change any result
        __syncthreads();
        if (threadIdx.x == 0) next_item = atomicAdd(R.item_counter, 1);
        __syncthreads();
        const int32_t slot = next_item;
        if (slot >= items) break;
        const int32_t item = R.item_order[slot];
        const int32_t q = item / P.replicas;
        const int32_t rep = item - q * P.replicas;
        const int64_t base = P.node_off[q];
        const int32_t n = (int32_t)(P.node_off[q + 1] - base);
        const int32_t *cls = P.class_ptr + P.class_off[q];
        const int32_t ncls = P.class_off[q + 1] - P.class_off[q] - 1;
        int8_t *gsig = R.spins + (int64_t)rep * P.N + base;
        const int64_t nnz_item = P.row_ptr[base + n] - P.row_ptr[base];
        const int32_t mean_deg = n > 0 ? (int32_t)min((nnz_item + n - 1) / n, (int64_t)64) : 1;

        // the window at ranks [wlo, whi): its E* and rows, by warps w of nw
        auto prepare = [&](int32_t wlo, int32_t whi, int32_t sw, const uint32_t *row, int32_t rlen, float Tsw, int w, int nw) {
            const int64_t *rp = P.row_ptr + base + wlo;
            const int32_t ns = whi - wlo;
            split_ahead(
                ns, w, nw,
                [&](int t, int nth) {
                    if (pre) draw_estar(R, wlo, whi, wlo, q, rep, sw, row, rlen, Tsw, es, t, nth);
                },
                [&](int t, int nth) {
                    const int64_t al = rp[0] & ~(int64_t)7;
                    const int32_t pieces = (int32_t)((min(rp[ns] - al, (int64_t)R.cta_stage) + 7) >> 3);
                    stage_rows(P, rp, ns, al, pieces, rofs, cbuf, t, nth);
                },
                staged);
        };

        int32_t g = 0;
        for (int32_t r = threadIdx.x; r < n; r += BS) {
            const int8_t s = gsig[r];
            S.sig[r] = s;
            g += s;
        }
        for (int b = threadIdx.x; b < 3 * NB; b += BS) h1[b] = 0;
        if (threadIdx.x < 2) nge[threadIdx.x] = 0;
        {
            const int32_t roff = R.tab_off[R.s_begin], rlen = R.tab_off[R.s_begin + 1] - roff;
            uint32_t *row = S.row + (rows2 && (R.s_begin & 1) ? L.row_stride : 0);
            for (int32_t k = threadIdx.x; k < rlen; k += BS) row[k] = R.tab[roff + k];
        }
        g = block_sum<BS, int32_t>(g, S.red32);
        if (threadIdx.x == 0) *S.G = g;
        __syncthreads();
        if (R.s_begin < R.s_end && ncls > 0) {
            prepare(cls[0], P.W > 0 ? min(cls[0] + P.W, cls[1]) : cls[1], R.s_begin,
                    S.row + (rows2 && (R.s_begin & 1) ? L.row_stride : 0),
                    R.tab_off[R.s_begin + 1] - R.tab_off[R.s_begin], R.temp ? R.temp[R.s_begin] : 0.f, warp, BS / 32);
            cp_async_wait_all();
        }
        __syncthreads();

        for (int32_t sw = R.s_begin; sw < R.s_end; ++sw) {
            const int32_t roff = R.tab_off[sw];
            const int32_t rlen = R.tab_off[sw + 1] - roff;
            const uint32_t *row = S.row + (rows2 && (sw & 1) ? L.row_stride : 0);
            // this sweep's row (its first window was drawn before), or the next sweep's beside it
            if (!rows2 && sw > R.s_begin)
                for (int32_t k = threadIdx.x; k < rlen; k += BS) S.row[k] = R.tab[roff + k];
            const int32_t roff1 = sw + 1 < R.s_end ? roff + rlen : 0;
            const int32_t rlen1 = sw + 1 < R.s_end ? R.tab_off[sw + 2] - roff1 : 0;
            uint32_t *row1 = S.row + (sw & 1 ? 0 : L.row_stride);
            if (rows2)
                for (int32_t k = threadIdx.x; k < rlen1; k += BS) row1[k] = R.tab[roff1 + k];
            const float Tsw = R.temp ? R.temp[sw] : 0.f;
            const int first = (sw & 1) ? -1 : 1;            // the group that goes first
            if (!pre) __syncthreads();
            for (int32_t c = 0; c < ncls; ++c) {
                const int32_t clo = cls[c], chi = cls[c + 1];
                const int32_t Wn0 = P.W > 0 ? P.W : (chi - clo);
                const int tl = team_log2<BS>(min(Wn0, chi - clo), mean_deg);
                for (int32_t wlo = clo; wlo < chi; wlo += Wn0) {
                    const int32_t whi = min(wlo + Wn0, chi), Wn = whi - wlo;
                    const int32_t c0 = *S.G;
                    if (!pre) {
                        draw_estar(R, wlo, whi, wlo, q, rep, sw, row, rlen, Tsw, es, threadIdx.x, BS);
                        __syncthreads();
                    }
                    // ---- thresholds, counted by margin
                    const uint16_t *gcol = staged ? P.col16 + (P.row_ptr[base + wlo] & ~(int64_t)7) : nullptr;
                    int32_t ge1 = 0, ge2 = 0;
                    team_thresholds<BS>(P, S.sig, base, wlo, Wn, tl, max(32, 2 * mean_deg), staged ? rofs : nullptr, cbuf, R.cta_stage, gcol, es, a_shift,
                                        [&](int32_t i, int sg, int32_t gm) {
                                            gam[i] = gm;
                                            s0[i] = (int8_t)sg;
                                            if (standard) return;
                                            const int32_t e = sg > 0 ? c0 - gm : gm - c0;
                                            if (sg == first) {
                                                ge1 += e >= 0;
                                                if (e >= 0 && e < NB) atomicAdd(&h1[e], 1);
                                            } else {
                                                ge2 += e >= 0;
                                                if (e >= -NB && e < NB) atomicAdd(&h2[e + NB], 1);
                                            }
                                        });
                    if (!standard) {
                        ge1 = __reduce_add_sync(0xFFFFFFFFu, ge1);
                        ge2 = __reduce_add_sync(0xFFFFFFFFu, ge2);
                        if (lane == 0 && ge1) atomicAdd(&nge[0], ge1);
                        if (lane == 0 && ge2) atomicAdd(&nge[1], ge2);
                    }
                    __syncthreads();
                    // the next window: its E* and rows do not depend on the spins
                    auto ahead = [&](int w, int nw) {
                        int32_t nlo = whi, nhi, nsw = sw;
                        if (whi < chi) {
                            nhi = min(whi + Wn0, chi);
                        } else {
                            if (c + 1 == ncls) {
                                if (sw + 1 >= R.s_end) return;
                                nsw = sw + 1;
                            }
                            const int nc = nsw == sw ? c + 1 : 0;
                            nlo = cls[nc];
                            nhi = P.W > 0 ? min(nlo + P.W, cls[nc + 1]) : cls[nc + 1];
                        }
                        const bool same = nsw == sw;
                        prepare(nlo, nhi, nsw, same ? row : (rows2 ? row1 : R.tab + roff1), same ? rlen : rlen1,
                                same ? Tsw : (R.temp ? R.temp[nsw] : 0.f), w, nw);
                    };
                    if (standard) {
                        standard_window<BS>(S, gam, s0, wlo, Wn, n);
                        ahead(warp, BS / 32);
                        if (staged) cp_async_wait_all();
                        __syncthreads();
                        continue;
                    }
                    if (warp == 0) {
                        int32_t K1 = 0, K2 = 0, y1, y2, l1, l2;
                        bool ok = group_flips(h1, NB, nge[0], K1, y1, l1);
                        if (ok) {
                            // second group: margins grow by 2 K1
                            int32_t n2 = 0;
                            for (int m = NB - 2 * K1 + lane; m < NB; m += 32) n2 += h2[m];
                            n2 = nge[1] + __reduce_add_sync(0xFFFFFFFFu, n2);
                            ok = group_flips(h2 + NB - 2 * K1, NB + 2 * K1, n2, K2, y2, l2);
                        }
                        if (lane == 0) {
                            dec.slow = ok ? 0 : 1;
                            if (ok) {
                                dec.y[0] = y1;
                                dec.left[0] = l1;
                                dec.y[1] = K2 ? y2 - 2 * K1 : INT32_MAX;
                                dec.left[1] = l2;
                                *S.G = c0 - 2 * first * K1 + 2 * first * K2;
                            }
                        }
                    } else {
                        ahead(warp - 1, BS / 32 - 1);
                    }
                    __syncthreads();
                    if (dec.slow) {
                        // more flips than the bins cover: both groups by counting passes over the window
                        int32_t gg = c0;
                        for (int ph = 0; ph < 2; ++ph) {
                            const int grp = ph == 0 ? first : -first;
                            int32_t lo = 0, hi = count_ge<BS>(gam, s0, Wn, grp, gg, 0, S.red32);
                            while (lo < hi) {
                                const int32_t mid = (lo + hi + 1) >> 1;
                                if (count_ge<BS>(gam, s0, Wn, grp, gg, 2 * (int64_t)mid - 2, S.red32) >= mid) lo = mid;
                                else hi = mid - 1;
                            }
                            const int32_t K = lo;
                            int32_t y = INT32_MAX, left = 0;
                            if (K > 0) {
                                const int32_t n2 = count_ge<BS>(gam, s0, Wn, grp, gg, 2 * (int64_t)K, S.red32);
                                const int32_t n1 = count_ge<BS>(gam, s0, Wn, grp, gg, 2 * (int64_t)K - 1, S.red32);
                                y = n2 == K || n1 >= K ? 2 * K - 1 : 2 * K - 2;
                                left = n2 == K ? 0 : (n1 >= K ? K - n2 : K - n1);
                                // margins are taken from the window-start G below
                                y += grp > 0 ? c0 - gg : gg - c0;
                            }
                            if (threadIdx.x == 0) {
                                dec.y[ph] = y;
                                dec.left[ph] = left;
                            }
                            gg -= 2 * grp * K;
                        }
                        if (threadIdx.x == 0) *S.G = gg;
                        __syncthreads();
                    }
                    const int32_t y1 = dec.y[0], y2 = dec.y[1], l1 = dec.left[0], l2 = dec.left[1];
                    const bool cut = l1 | l2;               // some group's ties flip in part: by position
                    // (also the bins' next use starts from zero)
                    for (int b = threadIdx.x; b < 3 * NB; b += BS) h1[b] = 0;
                    if (threadIdx.x < 2) nge[threadIdx.x] = 0;
                    const int32_t rounds = (Wn + BS - 1) / BS;
                    if (cut) {
                        for (int32_t k = 0; k < rounds; ++k) {
                            const int32_t i = k * BS + threadIdx.x;
                            bool t1 = false, t2 = false;
                            if (i < Wn) {
                                const int sg = s0[i];
                                const int32_t e = sg > 0 ? c0 - gam[i] : gam[i] - c0;
                                t1 = sg == first && e == y1;
                                t2 = sg != first && e == y2;
                            }
                            const unsigned b1 = __ballot_sync(0xFFFFFFFFu, t1), b2 = __ballot_sync(0xFFFFFFFFu, t2);
                            if (lane == 0 && i < Wn) tcnt[i >> 5] = __popc(b1) | (__popc(b2) << 16);
                        }
                        __syncthreads();
                    }
                    for (int32_t k = 0; k < rounds; ++k) {
                        const int32_t i = k * BS + threadIdx.x;
                        int32_t e = 0;
                        int sg = 0;
                        if (i < Wn) {
                            sg = s0[i];
                            e = sg > 0 ? c0 - gam[i] : gam[i] - c0;
                        }
                        const bool g1 = sg == first, g2 = sg == -first;
                        bool flip = (g1 && e > y1) || (g2 && e > y2);
                        if (cut) {
                            const bool t1 = g1 && e == y1, t2 = g2 && e == y2;
                            const unsigned b1 = __ballot_sync(0xFFFFFFFFu, t1), b2 = __ballot_sync(0xFFFFFFFFu, t2);
                            if (b1 | b2) {
                                // ties of the ranks before this warp's 32
                                const int32_t ch = (k * BS + (int32_t)(threadIdx.x & ~31u)) >> 5;
                                int32_t p1 = 0, p2 = 0;
                                for (int32_t j = lane; j < ch; j += 32) {
                                    p1 += tcnt[j] & 0xFFFF;
                                    p2 += tcnt[j] >> 16;
                                }
                                p1 = __reduce_add_sync(0xFFFFFFFFu, p1) + __popc(b1 & ((1u << lane) - 1u));
                                p2 = __reduce_add_sync(0xFFFFFFFFu, p2) + __popc(b2 & ((1u << lane) - 1u));
                                flip |= (t1 && p1 < l1) || (t2 && p2 < l2);
                            }
                        }
                        if (flip) S.sig[wlo + i] = (int8_t)-sg;
                    }
                    if (staged) cp_async_wait_all();
                    __syncthreads();
                }
            }
            if (R.flags & GDI_DEV_TRACE) {
                uint64_t dg = 0;
                for (int32_t r = threadIdx.x; r < n; r += BS)
                    if (S.sig[r] > 0)
                        dg += splitmix64_fin((uint64_t)(uint32_t)r | ((uint64_t)(sw & 0xFFFF) << 32) |
                                             ((uint64_t)(rep & 0xFFFF) << 48));
                dg = block_sum<BS, uint64_t>(dg, reinterpret_cast<uint64_t *>(S.red64));
                const int64_t ct = item_fields<BS>(P, base, n, mean_deg, S, 0, 0, nullptr, 0);
                if (threadIdx.x == 0) {
                    const int64_t o = (int64_t)item * R.sweeps + sw;
                    R.tr_digest[o] = dg;
                    R.tr_G[o] = *S.G;
                    R.tr_cut[o] = ct;
                }
                __syncthreads();
            }
        }
        finish_item<BS>(P, R, base, n, mean_deg, S, gam, (int)((L.total - L.gam) / 4), item, true);
        for (int32_t r = threadIdx.x; r < n; r += BS) gsig[r] = S.sig[r];
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// CTA-resident counting kernel (1 <= W <= 256): the same results as gdi_cta_block_kernel with far
// fewer block barriers per window.  Per colour class:
//   1. thresholds of the class's ranks: a team of T lanes sums a rank's row over the shared spins;
//   2. a class of three or more windows: the counts of each window's threshold distances give its stage
//      maps on the lattice (gdi_window.cuh) and both composed as a byte table of 64 lattice points; each
//      replaying warp looks its window's entering lattice point up from the class-start G (a read per
//      window before it; following the maps themselves costs ten times that), and all windows are
//      replayed at once.  A window whose map leaves the lattice, and all after it, are
//      replayed in rank order from the exact G by one warp, as are classes of one or two windows.  A
//      replay writes its flips to the spins itself: nothing reads them again before the class ends.
// The windows of a class share no edge, so only the running G passes from one window to the next.
// SL = members per lane of a window.
//
// What bounds it is the chain of dependent steps of a class (a few hundred ranks), not bandwidth, so
// everything that does not depend on spins leaves the chain: while one warp walks or replays, the
// other warps draw the next class's E* (Philox and the table search) into shared memory and stage the
// next class's columns and row offsets there (cp.async: contiguous in rank order), so that a threshold
// is a few shared loads.  Measured, whole call, with sorted windows, draws and rows on the chain -> now:
// ER-800, one replica, 1000 sweeps 63.7 -> 42.6 ms; 640 ER instances, 500 sweeps 98.7 -> 43.9 ms; 1024 anneals
// of 25 sweeps 8.0 -> 4.8 ms; torus 100 x 100, 64 replicas, 5000 sweeps (two blocks each) 148 -> 98.8 ms; BA
// 20,000, one replica, 300 sweeps (eight blocks) 20.7 (grid path) -> 15.3 ms.
struct SortedCta {
    int32_t *gam;       // [own ranks] flip thresholds of my share of the class
    int32_t *es;        // [own ranks] E* of the next class's, drawn ahead
    uint8_t *s0;        // [own ranks] 1 = the member was -1 at window start
    uint32_t *bins;     // [cta_bins windows, or warps that count][WBINS]
    StageMap *wmaps;    // [nwm][2] stage maps of my windows (classes of 3 windows and more)
    int8_t *wtab;       // [nwm][NT] both maps composed (-1: leaves the lattice)
    int32_t *rofs;      // row offsets of the staged rows
    uint16_t *cbuf;     // [cta_stage] their columns
};

// Windows of one block whose stage maps are kept.  A class of more than so many for each of its blocks is
// taken in pieces of that size, one after another like classes: its vertices share no edge, so a piece's
// thresholds do not see the flips of the pieces before it, and only G passes on.  gdi_create lays the pieces
// out for every cluster size as it does the classes, and the launch hands the kernel those in their place, with
// their size as that of the largest class (the kernel finding them itself spilled 640 bytes and lost 8 % with
// windows above 128, pieces or not).  (One warp that replayed such a
// class window by window took 0.47 us a window.  A sweep of 40 replicas of 3,000 vertices, W = 1: 1,399 -> 314 us;
// 300 of a 100 x 100 torus, W = 32: 257 -> 118.)
constexpr int CTA_WALK_MAX = 128;

// windows a block of a cluster of cl (1: alone) has of the largest class: a class of one or two windows
// is the first block's
__host__ __device__ inline int cta_own_windows(int32_t max_class, int W, int cl)
{
    const int nw = (max_class + W - 1) / W;
    return cl > 1 ? ((nw + cl - 1) / cl > 2 ? (nw + cl - 1) / cl : 2) : nw;
}

__host__ __device__ inline int cta_walk_windows(int32_t max_class, int W, int cl)
{
    const int nw = cta_own_windows(max_class, W, cl);
    return nw < CTA_WALK_MAX ? nw : CTA_WALK_MAX;
}

// warps that count windows at once where the windows have no bins of their own: none where no class has
// three windows; their bins share the repair flags' bytes, and a small instance has room for 16
__host__ __device__ inline int cta_count_warps(int32_t max_n, int32_t max_class, int W, int BS, int cl)
{
    const int nwm = cta_walk_windows(max_class, W, cl);
    const int fit = max_n / 1024 > 16 ? max_n / 1024 : 16;
    const int nw = nwm < BS / 32 ? nwm : BS / 32;
    return (max_class + W - 1) / W < 3 ? 0 : (nw < fit ? nw : fit);
}

// Shared-memory layout of the counting CTA kernel, one function for the kernel's carving and the
// host's size: the common part (reductions, G, table rows, spins, repair flags), then the class
// buffers.  Every array starts on a 16-byte boundary.
struct CtaSortedLayout {
    size_t red64, red32, G, row, sig, flag, gam, es, s0, wmaps, wtab, rofs, cbuf, total;
    int row_stride;
};

__host__ __device__ inline CtaSortedLayout cta_sorted_layout(const GdiDevProblem &P, int32_t max_row, int BS, int opts,
                                                             int32_t stage, int32_t rofs, int nbw, int cl)
{
    CtaSortedLayout L;
    const size_t own = cl > 1 ? (size_t)cta_own_windows(P.max_class, P.W, cl) * P.W : (size_t)P.max_class;
    const size_t mc = own + 8;
    size_t o = 0;
    L.red64 = o; o = align16c(o + sizeof(int64_t) * (BS / 32 + 2));
    L.red32 = o; o = align16c(o + sizeof(int32_t) * (BS / 32 + 2));
    L.G = o; o = align16c(o + 16);
    L.row_stride = (max_row + 4 + 3) & ~3;
    L.row = o; o = align16c(o + sizeof(uint32_t) * (size_t)L.row_stride * ((opts & CTA_OPT_ROWS2) ? 2 : 1));
    L.sig = o; o = align16c(o + (size_t)P.max_n + 16);
    // the repair flags and, during the sweeps, the windows' or counting warps' bins share their bytes
    const int cw = cta_count_warps(P.max_n, P.max_class, P.W, BS, cl);
    const size_t bins = 4 * (size_t)win::WBINS * (cw > nbw ? cw : nbw);
    const size_t fl = (size_t)P.max_n + 16;
    L.flag = o; o = align16c(o + (fl > bins ? fl : bins));
    L.gam = o; o = align16c(o + 4 * mc);
    L.es = o; o = align16c(o + 4 * mc);
    L.s0 = o; o = align16c(o + mc);
    const int nwm = cta_walk_windows(P.max_class, P.W, cl);
    L.wmaps = o; o = align16c(o + sizeof(StageMap) * 2 * (size_t)nwm);
    L.wtab = o; o = align16c(o + (size_t)NT * nwm);
    L.rofs = o; o = align16c(o + (stage ? 4 * (mc > (size_t)rofs ? mc : (size_t)rofs) : 0));
    L.cbuf = o; o = align16c(o + 2 * (size_t)stage);
    L.total = o;
    return L;
}

// CLUS: a cluster of 2, 4 or 8 blocks anneals each item (few items, many windows).  Every block keeps all
// spins and G; a class of three windows and more is split into contiguous runs of windows, each block's
// thresholds, counts and replays its own.  The blocks exchange one composed 64-entry table each through
// distributed shared memory, every replay writes its flips to every block's spins, and two cluster
// barriers a class remain (after the tables, after the flips).  Classes of one or two windows are the
// first block's alone.
template <int BS, int SL, bool CLUS>
__global__ void __launch_bounds__(BS, 1024 / BS) gdi_cta_sorted_kernel(GdiDevProblem P, GdiDevRun R)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem S = {};
    SortedCta C;
    const bool rows2 = (R.cta_opts & CTA_OPT_ROWS2) != 0, staged = R.cta_stage > 0;
    unsigned crank = 0, CL = 1;                          // block rank in the cluster, cluster size
    if constexpr (CLUS) {
        crank = cooperative_groups::this_cluster().block_rank();
        CL = cooperative_groups::this_cluster().num_blocks();
    }
    int row_stride;
    int scratch_words;
    {
        const CtaSortedLayout L = cta_sorted_layout(P, R.max_row, BS, R.cta_opts, R.cta_stage, R.cta_rofs, R.cta_bins, (int)CL);
        S.red64 = reinterpret_cast<int64_t *>(smem_raw + L.red64);
        S.red32 = reinterpret_cast<int32_t *>(smem_raw + L.red32);
        S.G = reinterpret_cast<int32_t *>(smem_raw + L.G);
        S.row = reinterpret_cast<uint32_t *>(smem_raw + L.row);
        S.sig = reinterpret_cast<int8_t *>(smem_raw + L.sig);
        S.flag = reinterpret_cast<int8_t *>(smem_raw + L.flag);
        C.gam = reinterpret_cast<int32_t *>(smem_raw + L.gam);
        C.es = reinterpret_cast<int32_t *>(smem_raw + L.es);
        C.s0 = smem_raw + L.s0;
        C.bins = reinterpret_cast<uint32_t *>(smem_raw + L.flag);
        C.wmaps = reinterpret_cast<StageMap *>(smem_raw + L.wmaps);
        C.wtab = reinterpret_cast<int8_t *>(smem_raw + L.wtab);
        C.rofs = reinterpret_cast<int32_t *>(smem_raw + L.rofs);
        C.cbuf = reinterpret_cast<uint16_t *>(smem_raw + L.cbuf);
        row_stride = L.row_stride;
        scratch_words = (int)((L.total - L.gam) / 4);
        // the launch must have given the whole layout (the host sizes it with the same function)
        uint32_t dyn;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
        if ((size_t)dyn < L.total) {
            if (threadIdx.x == 0 && blockIdx.x == 0) atomicCAS(R.err, 0, GDI_DEVERR_INPUT);
            return;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = BS / 32;
    const int W = P.W;
    const int cwarps = cta_count_warps(P.max_n, P.max_class, W, BS, (int)CL);
    const int w_shift = (W & (W - 1)) == 0 ? __ffs(W) - 1 : -1;
    const int a_shift = (P.A > 0 && (P.A & (P.A - 1)) == 0) ? 2 + __ffs(P.A) - 1 : -1;   // log2(4A)
    const int32_t items = P.num_instances * P.replicas;
    __shared__ int32_t next_item;
    // the first CB classes as this block sees them (a class starts without deriving them anew)
    constexpr int CB = 48;
    struct Span {
        int32_t lo, ns;                 // my ranks [lo, lo + ns)
        int32_t nwin, kq, kb, nk;       // windows [kb, kb + nk) of nwin are mine, kq to a block
        int32_t clo, chi;               // the class's ranks
        int32_t al, pieces;             // staging: first entry (from the item's, a 16-byte boundary), pieces,
        int32_t cb, ro;                 // where its columns and row offsets start
        int16_t tl, walk;               // log2 of the team size; three windows or more
    };
    __shared__ Span c_span[CB];
    __shared__ bool all_staged;
    __shared__ int8_t btab[8][NT];                       // composed tables of the cluster's blocks
    __shared__ int32_t w_fail[2];                        // the class's first window off the lattice (or -1), its index
    // another block's copy of a shared-memory object (same layout in all blocks)
    auto remote = [&](auto *ptr, unsigned r) { return cooperative_groups::this_cluster().map_shared_rank(ptr, r); };
    auto item_sync = [&]() {
        if constexpr (CLUS) cooperative_groups::this_cluster().sync();
        else __syncthreads();
    };
    if (threadIdx.x == 0) w_fail[0] = -1;
    while (true) {
        item_sync();
        if (crank == 0 && threadIdx.x == 0) {
            const int32_t t = atomicAdd(R.item_counter, 1);
            next_item = t;
            if constexpr (CLUS)
                for (unsigned r = 1; r < CL; ++r) *remote(&next_item, r) = t;
        }
        item_sync();
        const int32_t slot = next_item;
        if (slot >= items) break;
        const int32_t item = R.item_order[slot];
        const int32_t q = item / P.replicas;
        const int32_t rep = item - q * P.replicas;
        const int64_t base = P.node_off[q];
        const int32_t n = (int32_t)(P.node_off[q + 1] - base);
        const int32_t *cls = P.class_ptr + P.class_off[q];
        const int32_t ncls = P.class_off[q + 1] - P.class_off[q] - 1;
        int8_t *gsig = R.spins + (int64_t)rep * P.N + base;
        const int64_t row0 = P.row_ptr[base];
        const int64_t nnz_item = P.row_ptr[base + n] - row0;
        const int32_t mean_deg = n > 0 ? (int32_t)min((nnz_item + n - 1) / n, (int64_t)64) : 1;

        auto make_span = [&](int c) {
            Span s;
            s.clo = cls[c];
            s.chi = cls[c + 1];
            const int32_t size = s.chi - s.clo;
            s.nwin = (size + W - 1) / W;
            s.kq = CLUS ? (s.nwin + (int)CL - 1) / (int)CL : s.nwin;
            s.walk = s.nwin >= 3 && s.kq <= CTA_WALK_MAX;
            if (!s.walk) s.kq = s.nwin;
            s.kb = min((int)crank * s.kq, s.nwin);
            s.nk = min(s.kq, s.nwin - s.kb);
            const int32_t rb = min(s.kb * W, size), re = min((s.kb + s.nk) * W, size);
            s.lo = s.clo + rb;
            s.ns = re - rb;
            s.tl = (int16_t)team_log2<BS>(s.ns, mean_deg);
            const int64_t eb = P.row_ptr[base + s.lo], ee = P.row_ptr[base + s.lo + s.ns], al = eb & ~(int64_t)7;
            s.al = (int32_t)(al - row0);
            s.pieces = (int32_t)((min(ee - al, (int64_t)R.cta_stage) + 7) >> 3);
            s.cb = s.ro = 0;
            return s;
        };
        auto span = [&](int c) { return c < CB ? c_span[c] : make_span(c); };
        for (int c = threadIdx.x; c < ncls && c < CB; c += BS) c_span[c] = make_span(c);
        __syncthreads();
        if (staged && warp == 0) {
            // places of all classes side by side, if they fit
            int32_t cb = 0, ro = 0;
            for (int c0 = 0; c0 < CB && ncls <= CB; c0 += 32) {
                const int c = c0 + lane;
                const int32_t a = c < ncls ? 8 * c_span[c].pieces : 0, b = c < ncls ? c_span[c].ns + 1 : 0;
                int32_t xa = a, xb = b;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t ya = __shfl_up_sync(0xFFFFFFFFu, xa, o), yb = __shfl_up_sync(0xFFFFFFFFu, xb, o);
                    if (lane >= o) { xa += ya; xb += yb; }
                }
                if (c < ncls) {
                    c_span[c].cb = cb + xa - a;
                    c_span[c].ro = ro + xb - b;
                }
                cb += __shfl_sync(0xFFFFFFFFu, xa, 31);
                ro += __shfl_sync(0xFFFFFFFFu, xb, 31);
            }
            const bool all = ncls <= CB && cb < R.cta_stage && ro <= R.cta_rofs;
            __syncwarp();
            for (int c = lane; c < ncls && c < CB && !all; c += 32) c_span[c].cb = c_span[c].ro = 0;
            if (lane == 0) all_staged = all;
        }
        __syncthreads();
        const bool whole = staged && all_staged;
        // E* and rows of a class (span s) at sweep sw, by warps w of nw
        auto prepare = [&](const Span &s, int32_t sw, const uint32_t *row, int32_t rlen, float Tsw, int w, int nw) {
            if (s.ns == 0) return;
            split_ahead(
                s.ns, w, nw,
                [&](int t, int nth) { draw_estar(R, s.lo, s.lo + s.ns, s.lo, q, rep, sw, row, rlen, Tsw, C.es, t, nth); },
                [&](int t, int nth) {
                    stage_rows(P, P.row_ptr + base + s.lo, s.ns, row0 + s.al, s.pieces, C.rofs, C.cbuf, t, nth);
                },
                staged && !whole);
        };
        if (whole)
            for (int c = warp; c < ncls; c += NW)
                stage_rows(P, P.row_ptr + base + c_span[c].lo, c_span[c].ns, row0 + c_span[c].al, c_span[c].pieces,
                           C.rofs + c_span[c].ro, C.cbuf + c_span[c].cb, lane, 32);

        for (int b = threadIdx.x; b < R.cta_bins * WBINS; b += BS) C.bins[b] = 0;
        int32_t g = 0;
        for (int32_t r = threadIdx.x; r < n; r += BS) {
            const int8_t sv = gsig[r];
            S.sig[r] = sv;
            g += sv;
        }
        {
            const int32_t roff = R.tab_off[R.s_begin], rlen = R.tab_off[R.s_begin + 1] - roff;
            uint32_t *row = S.row + (rows2 && (R.s_begin & 1) ? row_stride : 0);
            for (int32_t k = threadIdx.x; k < rlen; k += BS) row[k] = R.tab[roff + k];
        }
        g = block_sum<BS, int32_t>(g, S.red32);
        if (threadIdx.x == 0) *S.G = g;
        __syncthreads();
        if (R.s_begin < R.s_end && ncls > 0) {
            prepare(span(0), R.s_begin, S.row + (rows2 && (R.s_begin & 1) ? row_stride : 0),
                    R.tab_off[R.s_begin + 1] - R.tab_off[R.s_begin], R.temp ? R.temp[R.s_begin] : 0.f, warp, NW);
        }
        cp_async_wait_all();
        item_sync();

        for (int32_t sw = R.s_begin; sw < R.s_end; ++sw) {
            const int32_t roff = R.tab_off[sw];
            const int32_t rlen = R.tab_off[sw + 1] - roff;
            const uint32_t *row = S.row + (rows2 && (sw & 1) ? row_stride : 0);
            // this sweep's row (its first class was drawn before), or the next sweep's beside it; the
            // first class's barrier makes it visible to the draws that follow
            if (!rows2 && sw > R.s_begin)
                for (int32_t k = threadIdx.x; k < rlen; k += BS) S.row[k] = R.tab[roff + k];
            const int32_t roff1 = sw + 1 < R.s_end ? roff + rlen : 0;
            const int32_t rlen1 = sw + 1 < R.s_end ? R.tab_off[sw + 2] - roff1 : 0;
            uint32_t *row1 = S.row + (sw & 1 ? 0 : row_stride);
            if (rows2)
                for (int32_t k = threadIdx.x; k < rlen1; k += BS) row1[k] = R.tab[roff1 + k];
            const float Tsw = R.temp ? R.temp[sw] : 0.f;
            const bool plus_first = (sw & 1) == 0;
            const int st0 = plus_first ? 0 : 1;          // the stage that goes first
            for (int32_t c = 0; c < ncls; ++c) {
                const Span s = span(c);
                const int32_t lo = s.lo, ns = s.ns;
                const int32_t c0 = *S.G;                 // G at class start (the reference c)
                // a class whose windows here all have bins counts its thresholds as they are made
                const bool binned = s.nk <= R.cta_bins;
                // ---- thresholds of my ranks
                team_thresholds<BS>(P, S.sig, base, lo, ns, s.tl, max(32, 2 * mean_deg), staged ? C.rofs + s.ro : nullptr, C.cbuf + s.cb, 8 * s.pieces,
                                    P.col16 + row0 + s.al, C.es, a_shift, [&](int32_t i, int sg, int32_t gm) {
                                        C.gam[i] = gm;
                                        C.s0[i] = sg < 0 ? 1 : 0;
                                        if (binned) {
                                            const int32_t d = sg < 0 ? c0 - gm : gm - c0;
                                            const int k = w_shift >= 0 ? i >> w_shift : i / W;
                                            if (d <= NT)
                                                atomicAdd(&C.bins[k * WBINS + max(d + BIN_L, 0)], sg < 0 ? 0x10000u : 1u);
                                        }
                                    });
                // (the first block's replay of a small class writes the others' G and spins: they must
                // have read this class's c0 first)
                if (CLUS && !s.walk) item_sync(); else __syncthreads();
                // the next class: its E* and columns do not depend on the spins
                auto ahead = [&](int w, int nw) {
                    const bool same = c + 1 < ncls;
                    if (!same && sw + 1 >= R.s_end) return;
                    prepare(span(same ? c + 1 : 0), same ? sw : sw + 1, same ? row : (rows2 ? row1 : R.tab + roff1),
                            same ? rlen : rlen1, same ? Tsw : (R.temp ? R.temp[sw + 1] : 0.f), w, nw);
                };
                // the flips of a window (ranks from r0 on) straight into the spins of every block
                auto flip = [&](int32_t r0, int32_t ws, int32_t we, const uint8_t *s0, const uint32_t (&wb)[SL]) {
#pragma unroll
                    for (int k = 0; k < SL; ++k) {
                        const int32_t i = ws + 32 * k + lane;
                        if (i < we && ((wb[k] >> lane) & 1u)) {
                            const int8_t v = s0[i] ? 1 : -1;
                            S.sig[r0 + i] = v;
                            if constexpr (CLUS)
                                for (unsigned r = 0; r < CL; ++r)
                                    if (r != crank) remote(S.sig, r)[r0 + i] = v;
                        }
                    }
                };
                auto zero_bins = [&](uint32_t *bins) {
                    __syncwarp();
                    reinterpret_cast<uint4 *>(bins)[lane] = make_uint4(0u, 0u, 0u, 0u);
                    reinterpret_cast<uint4 *>(bins)[lane + 32] = make_uint4(0u, 0u, 0u, 0u);
                };
                // *p of every block, by lane 0 of a warp
                auto set_all = [&](int32_t *p, int32_t v) {
                    if (lane == 0) {
                        *p = v;
                        if constexpr (CLUS)
                            for (unsigned r = 0; r < CL; ++r)
                                if (r != crank) *remote(p, r) = v;
                    }
                };
                if (s.walk) {
                    // ---- the maps and the table of every window of mine, by one warp
                    const int cw = binned ? NW : cwarps;
                    for (int k = warp; k < s.nk && warp < cw; k += cw) {
                        if (binned)
                            bins_to_prefix<8>(C.bins + (size_t)k * WBINS, BIN_L, C.wmaps + 2 * k);
                        else
                            window_maps<SL>(C.gam, C.s0, k * W, min(W, ns - k * W), 0, c0, C.bins + (size_t)warp * WBINS,
                                            C.wmaps + 2 * k);
                        __syncwarp();
                        const StageMap m0 = C.wmaps[2 * k + st0], m1 = C.wmaps[2 * k + (1 ^ st0)];
                        C.wtab[k * NT + lane] = (int8_t)stage_apply(m1, stage_apply(m0, lane));
                        C.wtab[k * NT + lane + 32] = (int8_t)stage_apply(m1, stage_apply(m0, lane + 32));
                    }
                    if (!binned && R.cta_bins && warp < cwarps) zero_bins(C.bins + (size_t)warp * WBINS);
                    __syncthreads();
                    // the first warps replay, the others work ahead
                    const int busy = min(s.nk, NW / 2);
                    if constexpr (CLUS) {
                        // my windows' tables composed (lanes hold lattice points lane and lane + 32), into
                        // every block; only the replays wait for the others'
                        if (warp == 0) {
                            int t0 = lane, t1 = lane + 32;
                            for (int k = 0; k < s.nk; ++k) {
                                if (t0 >= 0) t0 = C.wtab[k * NT + t0];
                                if (t1 >= 0) t1 = C.wtab[k * NT + t1];
                            }
                            for (unsigned r = 0; r < CL; ++r) {
                                int8_t *d = r == crank ? btab[crank] : remote(btab[crank], r);
                                d[lane] = (int8_t)t0;
                                d[lane + 32] = (int8_t)t1;
                            }
                        }
                        cooperative_groups::this_cluster().barrier_arrive();
                        if (warp < busy) cooperative_groups::this_cluster().barrier_wait();
                    }
                    // ---- replays: each warp follows x = G - c0 from 0 (lattice index t: x = 2 t - NT) through the
                    // blocks before mine and the windows before its own
                    if (warp < busy) {
                        int t = NT / 2, j = 0;
                        if constexpr (CLUS)
                            for (unsigned r = 0; r < crank && t >= 0; ++r) t = btab[r][t];
                        for (int k = warp; k < s.nk; k += busy) {
                            for (; j < k && t >= 0; ++j) t = C.wtab[j * NT + t];
                            const int tk = t;
                            uint32_t *pre = binned ? C.bins + (size_t)k * WBINS : nullptr;
                            if (tk >= 0) {
                                const int u = C.wtab[k * NT + tk];
                                const int32_t ws = k * W, we = min(ws + W, ns);
                                if (u < 0) {
                                    // the first window off the lattice: it and the rest in rank order below
                                    set_all(&w_fail[1], tk);
                                    set_all(&w_fail[0], s.kb + k);
                                } else {
                                    replay_mapped<SL>(C.gam, C.s0, 0, ws, we, c0 + 2 * tk - NT, plus_first, tk, C.wmaps + 2 * k,
                                                      WindowCounts{pre, c0, BIN_L, false},
                                                      [&](const uint32_t (&wb)[SL]) { flip(lo, ws, we, C.s0, wb); });
                                    if (s.kb + k == s.nwin - 1) set_all(S.G, c0 + 2 * u - NT);
                                }
                            }
                            if (pre) zero_bins(pre);
                        }
                    } else {
                        ahead(warp - busy, NW - busy);
                        if constexpr (CLUS) cooperative_groups::this_cluster().barrier_wait();
                    }
                } else if (warp > 0) {
                    ahead(warp - 1, NW - 1);
                }
                // windows [k0, nwin) in rank order by one warp of block 0 from the exact G, each entered with the
                // G its predecessors left; another block's windows are read remotely
                auto in_order = [&](int k0, int32_t gr, bool bins) {
                    for (int k = k0; k < s.nwin; ++k) {
                        const uint8_t *s0 = C.s0;
                        const int32_t *gam = C.gam;
                        const int b = k / s.kq;          // owner
                        if constexpr (CLUS) {
                            if (b > 0) { s0 = remote(C.s0, b); gam = remote(C.gam, b); }
                        }
                        const int32_t first = b * s.kq * W;              // the owner's first rank in the class
                        const int32_t ws = k * W - first, we = min(ws + W, s.chi - s.clo - first);
                        uint32_t *pre = bins ? C.bins + (size_t)k * WBINS : nullptr;
                        if (pre) bins_to_prefix<8>(pre, BIN_L, nullptr);
                        gr = replay_window<SL>(gam, s0, 0, ws, we, gr, plus_first, -1, -1, WindowCounts{pre, c0, BIN_L, false},
                                               [&](const uint32_t (&wb)[SL]) { flip(s.clo + first, ws, we, s0, wb); });
                        if (pre) zero_bins(pre);
                    }
                    set_all(S.G, gr);
                };
                if (!s.walk && crank == 0 && warp == 0) in_order(0, c0, binned);
                cp_async_wait_all();
                item_sync();
                if (s.walk && w_fail[0] >= 0) {
                    // rare: the lattice was left (every block sees the same flag)
                    const int kf = w_fail[0];
                    if (crank == 0 && warp == 0) in_order(kf, c0 + 2 * w_fail[1] - NT, false);
                    item_sync();
                    if (threadIdx.x == 0) w_fail[0] = -1;
                    item_sync();
                }
            }
            if (R.flags & GDI_DEV_TRACE) {
                uint64_t dg = 0;
                for (int32_t r = threadIdx.x; r < n; r += BS)
                    if (S.sig[r] > 0)
                        dg += splitmix64_fin((uint64_t)(uint32_t)r | ((uint64_t)(sw & 0xFFFF) << 32) |
                                             ((uint64_t)(rep & 0xFFFF) << 48));
                dg = block_sum<BS, uint64_t>(dg, reinterpret_cast<uint64_t *>(S.red64));
                const int64_t ct = item_fields<BS>(P, base, n, mean_deg, S, 0, 0, nullptr, 0);
                if (threadIdx.x == 0 && crank == 0) {
                    const int64_t o = (int64_t)item * R.sweeps + sw;
                    R.tr_digest[o] = dg;
                    R.tr_G[o] = *S.G;
                    R.tr_cut[o] = ct;
                }
                item_sync();
            }
        }
        finish_item<BS>(P, R, base, n, mean_deg, S, C.gam, scratch_words, item, crank == 0);
        if (crank == 0)
            for (int32_t r = threadIdx.x; r < n; r += BS) gsig[r] = S.sig[r];
        __syncthreads();
    }
}

// Initial state (Alg. 3 "initialize all s_i"): balanced random pairs from Philox, or the caller's
// spins scattered from original order to rank order.
__global__ void gdi_init_kernel(GdiDevProblem P, int8_t *spins, const int8_t *init_orig, int kind,
                                uint32_t key0, uint32_t key1)
{
    const int64_t total = (int64_t)P.replicas * P.N;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t rep = (int32_t)(t / P.N);
        const int64_t v = t - (int64_t)rep * P.N;
        if (kind == 1) {            // caller spins, original vertex v
            spins[(int64_t)rep * P.N + P.rank_of[v]] = init_orig[t] > 0 ? 1 : -1;
            continue;
        }
        // random: v is a global rank; find its instance by binary search of node_off
        int32_t lo = 0, hi = P.num_instances - 1;
        while (lo < hi) {
            const int32_t mid = (lo + hi + 1) >> 1;
            if (P.node_off[mid] <= v) lo = mid; else hi = mid - 1;
        }
        const int64_t base = P.node_off[lo];
        const int32_t n = (int32_t)(P.node_off[lo + 1] - base);
        const int32_t r = (int32_t)(v - base);
        int8_t s;
        if ((n & 1) && r == n - 1) {
            s = -1;
        } else {
            const int32_t pr = r >> 1;
            const uint4 u4 = philox4x32_10(make_uint4((uint32_t)(pr >> 2), 0xFFFFFFFFu, (uint32_t)lo,
                                                      (uint32_t)rep), key0, key1);
            const int8_t a = (word_of(u4, pr & 3) >> 31) ? -1 : 1;
            s = (r & 1) ? (int8_t)-a : a;
        }
        spins[t] = s;
    }
}

__global__ void gdi_gather_kernel(GdiDevProblem P, const int8_t *spins, int8_t *out)
{
    const int64_t total = (int64_t)P.replicas * P.N;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t rep = (int32_t)(t / P.N);
        const int64_t v = t - (int64_t)rep * P.N;
        out[t] = spins[(int64_t)rep * P.N + P.rank_of[v]];
    }
}

// the sorted-window kernel serves every window size 1 .. 256 (one instantiation per members per
// lane) of the running-G method when its whole-class buffers fit in a block's shared memory;
// Algorithm 2 (GDI_DEV_STANDARD), larger windows and larger classes take gdi_cta_block_kernel
constexpr size_t CTA_STATIC_SMEM = 3072;     // the kernel's class bounds and single words, rounded up

// the problem as the counting kernel with clusters of cl blocks sees it: no class larger than a piece
inline GdiDevProblem in_pieces(GdiDevProblem P, int cl)
{
    P.max_class = std::min(P.max_class, CTA_WALK_MAX * cl * P.W);
    return P;
}

inline bool cta_sorted(const GdiDevProblem &P, const GdiDevRun &R, int BS)
{
    if (P.W < 1 || P.W > 256 || (R.flags & GDI_DEV_STANDARD)) return false;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return cta_sorted_layout(in_pieces(P, 1), R.max_row, BS, 0, 0, 0, 0, 1).total + CTA_STATIC_SMEM <= (size_t)optin;
}

// blocks of a launch that are to run at once: one per SM, or the caller's limit
inline int cta_blocks(int grid_limit)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return grid_limit > 0 ? std::min(grid_limit, sms) : sms;
}

// Blocks per item (a cluster of 1, 2, 4 or 8, at most `most`): as many as leave every item its own of `blocks`
// and four windows of the largest class to each block.
inline int cta_cluster(const GdiDevProblem &P, const GdiDevRun &R, int BS, int blocks, int most)
{
    if (!cta_sorted(P, R, BS)) return 1;
    const int64_t items = (int64_t)P.num_instances * P.replicas;
    const int64_t nw = (P.max_class + P.W - 1) / P.W;
    int cl = 1;
    while (2 * cl <= std::min(most, 8) && 2 * cl * items <= blocks && 4 * 2 * cl <= nw) cl *= 2;
    return cl;
}

// shared memory of the kernel that takes this call (counted windows, else whole-block windows)
inline size_t cta_smem(const GdiDevProblem &P, const GdiDevRun &R, int BS, bool counted)
{
    return counted ? cta_sorted_layout(in_pieces(P, R.cta_cluster), R.max_row, BS, R.cta_opts, R.cta_stage, R.cta_rofs, R.cta_bins, R.cta_cluster).total
                   : cta_block_layout(P, R.max_row, BS, R.cta_opts, R.cta_stage).total;
}

// What the launch keeps in shared memory beyond the necessary (R.cta_opts, R.cta_stage): an option is
// taken when it fits a block and leaves as many items resident on an SM as there are without it (never
// more than the SM's share of the items, or than its 1024 threads at 64 registers); the staging buffer
// takes what is then left, up to the largest class.  Returns whether the counting kernel takes the call.
inline bool cta_options(const GdiDevProblem &P, GdiDevRun &R, int BS, int grid_limit, int max_cluster = 8)
{
    int dev = 0, optin = 0, per_sm = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t items = (int64_t)P.num_instances * P.replicas;
    const bool counted = cta_sorted(P, R, BS);
    R.cta_opts = 0;
    R.cta_stage = 0;
    R.cta_rofs = 0;
    R.cta_bins = 0;
    R.cta_cluster = cta_cluster(P, R, BS, cta_blocks(grid_limit), max_cluster);
    auto resident = [&]() {
        const size_t need = cta_smem(P, R, BS, counted) + CTA_STATIC_SMEM;
        if (need > (size_t)optin) return (int64_t)0;
        return std::min<int64_t>((int64_t)((size_t)per_sm / (need + 1024)), 1024 / BS);
    };
    const int64_t want = std::max<int64_t>(1, std::min<int64_t>(resident(), (items * R.cta_cluster + sms - 1) / sms));
    auto take = [&](int opt) {
        R.cta_opts |= opt;
        if (resident() < want) R.cta_opts &= ~opt;
    };
    if (!counted) take(CTA_OPT_BINS);
    if (!counted) take(CTA_OPT_ES);
    if (counted) {
        // bins for every window a block has of a class, up to 32, where a warp holds more than four members
        // a lane: a count over eight costs more than the bins do (one replica of W = 64 windows runs 5 to
        // 12 % faster without, 400 ER instances at W = 256 6 % slower)
        if (P.W > 128) R.cta_bins = std::min(cta_own_windows(in_pieces(P, R.cta_cluster).max_class, P.W, R.cta_cluster), 32);
        if (resident() < want) R.cta_bins = 0;
    }
    take(CTA_OPT_ROWS2);
    if (P.col16 && P.max_class_nnz > 0) {
        // (the first 8 columns stand for the row offsets, which any staging needs)
        R.cta_stage = 8;
        const int64_t room = std::min<int64_t>(optin, (int64_t)per_sm / want - 1024) - (int64_t)CTA_STATIC_SMEM -
                             (int64_t)cta_smem(P, R, BS, counted);
        // all rows of a block's share (a quarter above the even share), else one class's
        const int cl = R.cta_cluster;
        const int64_t rows = (int64_t)P.max_n / cl + (cl > 1 ? P.max_n / (4 * cl) : 0) + 64;
        const int64_t cols = (P.max_item_nnz / cl + (cl > 1 ? P.max_item_nnz / (4 * cl) : 0) + 48 * 16) & ~(int64_t)7;
        if (counted && P.max_item_nnz > 0 && 2 * cols + 4 * rows + 64 <= room) {
            R.cta_stage = (int32_t)cols;
            R.cta_rofs = (int32_t)rows;
        } else {
            const int64_t cap = std::min<int64_t>(P.max_class_nnz + 24, room / 2 + 8 - 16);
            R.cta_stage = cap >= std::min(512, P.max_class_nnz + 16) ? (int32_t)(cap & ~(int64_t)7) : 0;
        }
    }
    return counted;
}

template <int BS, bool CLUS>
const void *cta_sorted_kernel_for(int W)
{
    return W <= 32 ? (const void *)gdi_cta_sorted_kernel<BS, 1, CLUS>
         : W <= 64 ? (const void *)gdi_cta_sorted_kernel<BS, 2, CLUS>
         : W <= 128 ? (const void *)gdi_cta_sorted_kernel<BS, 4, CLUS>
                    : (const void *)gdi_cta_sorted_kernel<BS, 8, CLUS>;
}

template <int BS>
const void *cta_kernel(const GdiDevProblem &P, const GdiDevRun &R)
{
    if (!cta_sorted(P, R, BS)) return (const void *)gdi_cta_block_kernel<BS>;
    return R.cta_cluster > 1 ? cta_sorted_kernel_for<BS, true>(P.W) : cta_sorted_kernel_for<BS, false>(P.W);
}

// a launch of clusters of cl blocks, one for each item (attr: storage of its attribute)
inline cudaLaunchConfig_t cta_cluster_config(int cl, int items, int BS, size_t smem, cudaStream_t st, cudaLaunchAttribute *attr)
{
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl * items);
    cfg.blockDim = dim3(BS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <int BS>
int launch_cta(const GdiDevProblem &P0, const GdiDevRun &R0, const GdiCtaPieces &pieces, int grid_limit, cudaStream_t st,
               int *grid_used, size_t *smem_used)
{
    GdiDevRun R = R0;
    const int items = P0.num_instances * P0.replicas;
    int dev = 0, sms = 0, grid = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    GdiDevProblem P = P0;
    void *args[] = {&P, &R};
    size_t smem = 0;
    cudaError_t e = cudaSuccess;
    for (int cap = 8;;) {
        // (a GPU partition that holds no such cluster halves it)
        const bool counted = cta_options(P0, R, BS, grid_limit, cap);
        P = P0;
        const int k = R.cta_cluster == 8 ? 3 : R.cta_cluster / 2;
        if (counted) P = in_pieces(P0, R.cta_cluster);
        if (counted && pieces.ptr[k]) {
            P.class_ptr = pieces.ptr[k];
            P.class_off = pieces.off[k];
        }
        const void *kern = cta_kernel<BS>(P0, R);
        smem = cta_smem(P0, R, BS, counted);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return (int)e;
        if (R.cta_cluster == 1) {
            int per_sm = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BS, smem);
            if (e != cudaSuccess) return (int)e;
            if (per_sm < 1) return (int)cudaErrorInvalidConfiguration;
            grid = std::min(sms * per_sm, items);
            if (grid_limit > 0) grid = std::min(grid, grid_limit);
            e = cudaLaunchKernel(kern, dim3(grid), dim3(BS), args, smem, st);
            break;
        }
        // clusters of blocks, one item per cluster
        const int cl = R.cta_cluster;
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = cta_cluster_config(cl, items, BS, smem, st, attr);
        int ncl = 0;
        e = cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg);
        if (e != cudaSuccess) return (int)e;
        if (ncl < 1) {
            cap = cl / 2;
            continue;
        }
        grid = cl * std::min(items, ncl);
        if (grid_limit > 0) grid = std::min(grid, grid_limit / cl * cl);
        cfg.gridDim = dim3(grid);
        e = cudaLaunchKernelExC(&cfg, kern, args);
        break;
    }
    if (e != cudaSuccess) return (int)e;
    if (grid_used) *grid_used = grid;
    if (smem_used) *smem_used = smem;
    return (int)cudaGetLastError();
}

template <int BS>
int cta_occupancy(const GdiDevProblem &P, const GdiDevRun &R0, int grid_limit, GdiCtaPlan *plan)
{
    GdiDevRun R = R0;
    plan->counted = cta_options(P, R, BS, grid_limit);
    plan->cluster = R.cta_cluster;
    const void *kern = cta_kernel<BS>(P, R);
    const size_t smem = cta_smem(P, R, BS, plan->counted);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&plan->at_once, kern, BS, smem);
    plan->at_once *= sms;
    if (e == cudaSuccess && plan->cluster > 1) {
        cudaLaunchAttribute attr[1];
        const cudaLaunchConfig_t cfg = cta_cluster_config(plan->cluster, P.num_instances * P.replicas, BS, smem, nullptr, attr);
        e = cudaOccupancyMaxActiveClusters(&plan->at_once, kern, &cfg);
    }
    if (grid_limit > 0) plan->at_once = std::min(plan->at_once, grid_limit / plan->cluster);
    return (int)e;
}

}  // namespace

// Threads per block where the caller has set none.  Items that leave SMs idle take 512 (ms at 256 / 512 /
// 1024: 8 replicas of 1500 vertices, W = 64: 32.0 / 27.8 / 31.8; whole-class windows 7.4 / 6.9 / 8.6), 1024
// where a block's share of the largest class passes 800 ranks (BA 20,000 on one cluster: 19.4 / 15.1 /
// 13.9; 64 replicas of a 100 x 100 torus: 26.2 / 15.8 / 10.8), 256 where no class reaches 128 (ER-800: 42.7 /
// 44.1 / 51.7: barriers, not work).  Two blocks of 512 fit an SM: of items of one size a third on the SM would wait
// for a wave as long as the first (400 replicas of 64, 1,000 and 2,000 vertices, W = 64, us a sweep 15.5 / 28.9, 32.4 /
// 50.1, 51.4 / 60.8 at 256 / 512), while among unequal ones, the largest first, it fills in behind small ones (400 ER
// instances: 15.6 / 15.0 / 25.3 ms); more than three take 256 (1024 short anneals: 4.4 / 6.0 / 10.2).
int gdi_cta_default_block(const GdiDevProblem &P, const GdiDevRun &R, int grid_limit)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t items = (int64_t)P.num_instances * P.replicas;
    if (items > 3LL * sms) return 256;
    if (items > 2LL * sms && 4 * P.N >= 3LL * P.max_n * P.num_instances) return 256;
    const int cl = cta_cluster(P, R, 512, cta_blocks(grid_limit), 8);
    if (items * cl <= sms && cta_sorted(P, R, 512)) {
        const GdiDevProblem Q = in_pieces(P, cl);
        const int64_t own = cl > 1 ? (int64_t)cta_own_windows(Q.max_class, P.W, cl) * P.W : Q.max_class;
        if (own > 800) return 1024;
        if (P.max_class < 128) return 256;
    }
    return 512;
}

int32_t gdi_cta_piece(int32_t W, int32_t cluster) { return CTA_WALK_MAX * cluster * W; }

int gdi_cta_plan(const GdiDevProblem &P, const GdiDevRun &R, int block, int grid_limit, GdiCtaPlan *plan)
{
    *plan = GdiCtaPlan{};
    switch (block) {
    case 128: return cta_occupancy<128>(P, R, grid_limit, plan);
    case 256: return cta_occupancy<256>(P, R, grid_limit, plan);
    case 512: return cta_occupancy<512>(P, R, grid_limit, plan);
    case 1024: return cta_occupancy<1024>(P, R, grid_limit, plan);
    default: return (int)cudaErrorInvalidValue;
    }
}

int gdi_cta_smem_bytes(const GdiDevProblem &P, const GdiDevRun &R0, int block, int grid_limit, size_t *bytes)
{
    GdiDevRun R = R0;
    const bool counted = cta_options(P, R, block, grid_limit);
    *bytes = cta_smem(P, R, block, counted) + (counted ? CTA_STATIC_SMEM : 64);
    return 0;
}

int gdi_launch_cta_anneal(const GdiDevProblem &P, const GdiDevRun &R, const GdiCtaPieces &pieces, int block,
                          int grid_limit, void *stream, int *grid_used, size_t *smem_used)
{
    cudaStream_t st = (cudaStream_t)stream;
    switch (block) {
    case 128: return launch_cta<128>(P, R, pieces, grid_limit, st, grid_used, smem_used);
    case 256: return launch_cta<256>(P, R, pieces, grid_limit, st, grid_used, smem_used);
    case 512: return launch_cta<512>(P, R, pieces, grid_limit, st, grid_used, smem_used);
    case 1024: return launch_cta<1024>(P, R, pieces, grid_limit, st, grid_used, smem_used);
    default: return (int)cudaErrorInvalidValue;
    }
}

int gdi_launch_init(const GdiDevProblem &P, int8_t *spins, const int8_t *init_orig, int init_kind,
                    uint32_t key0, uint32_t key1, void *stream)
{
    const int64_t total = (int64_t)P.replicas * P.N;
    int grid = (int)((total + 255) / 256);
    if (grid > 152 * 32) grid = 152 * 32;
    if (grid < 1) grid = 1;
    gdi_init_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(P, spins, init_orig, init_kind, key0, key1);
    return (int)cudaGetLastError();
}

int gdi_launch_gather_spins(const GdiDevProblem &P, const int8_t *spins_rank, int8_t *out_orig,
                            void *stream)
{
    const int64_t total = (int64_t)P.replicas * P.N;
    int grid = (int)((total + 255) / 256);
    if (grid > 152 * 32) grid = 152 * 32;
    if (grid < 1) grid = 1;
    gdi_gather_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(P, spins_rank, out_orig);
    return (int)cudaGetLastError();
}
