// Scratch consolidation (Sec. 2.1, 2.4, 2.5): seed selection, cosine assignment of the
// remaining scratch rows to seeds, group masses and merge weights.
#include <type_traits>

#include "select.cuh"

namespace cask {

namespace {

constexpr int kTile = 64;
constexpr int kThreads = 256;

// ---- 1. seeds: the m greatest scratch rows; ordered list of their rows -------------------
__global__ void __launch_bounds__(kSelThreads) seeds_kernel(const UnitDesc* __restrict__ desc,
                                                            const float* __restrict__ s,
                                                            const int32_t* __restrict__ plan,
                                                            uint8_t* __restrict__ kind,
                                                            int32_t* __restrict__ seed_of,
                                                            float* __restrict__ weight,
                                                            float* __restrict__ sim, int32_t* __restrict__ grp,
                                                            int32_t* __restrict__ seed_rows,
                                                            unsigned long long* __restrict__ mass_fx,
                                                            int32_t* __restrict__ njoin, int max_m) {
    __shared__ SelectSmem sm;
    const int u = blockIdx.x;
    const UnitDesc& ud = desc[u];
    const int T = ud.T, P = ud.P;
    const int64_t o = ud.tok_off;
    int r = max(0, min(plan[u * 8 + CASK_PLAN_R], T - P));
    int m = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
    // a row left as MERGED/SEED by an earlier call on the same arrays is scratch again
    for (int i = threadIdx.x; i < T; i += blockDim.x) {
        uint8_t kd = kind[o + i];
        if (kd == CASK_KIND_SEED || kd == CASK_KIND_MERGED) kind[o + i] = CASK_KIND_DROPPED;
        seed_of[o + i] = -1;
        weight[o + i] = 0.f;
        grp[o + i] = -1;
        if (sim) sim[o + i] = -2.f;
    }
    for (int j = threadIdx.x; j <= max_m; j += blockDim.x) mass_fx[(size_t)u * (max_m + 1) + j] = 0ull;
    if (threadIdx.x == 0) njoin[u] = 0;
    __syncthreads();
    if (m <= 0) return;
    block_topk_mark(s + o, kind + o, P, T - r, m, CASK_KIND_SEED, sm);
    // ordered list of the seed rows
    block_ordered_rows(kind + o, P, T - r, CASK_KIND_SEED, sm, [&](unsigned idx, int i) {
        if (idx < (unsigned)m) {
            seed_rows[ud.seed_base + idx] = i;
            seed_of[o + i] = i;
            grp[o + i] = (int)idx;
        }
    });
}

// ---- 1 for longer units on the event path: prefix eviction, core and seed selection in one CTA per unit ----
// The same result as prefix_evict_kernel, select_core_kernel and seeds_kernel in turn, in three sweeps over the unit's scores:
//   1. smallest and greatest key of the prefix and of the scratch range;
//   2. one histogram per range over the keys' own span (2,048 bins of equal width in the order-preserving image, i.e. about
//      logarithmic in the score): the bins that hold the ranks pkeep, c and c + m follow from one scan each.  Fixed top
//      digits put most scores of a cache into a few bins, whose shared-memory atomics then queue;
//   3. every row's kind is written once: rows in bins above a boundary bin are decided, the few rows inside one (some tens)
//      are listed, ranked exactly (key descending, row ascending) by counting, and marked.
// A boundary bin with more rows than a list holds (thousands of equal scores) sends the range through the radix selection.
// Without LISTS sweep 3 also gives every row the slot and the weight of a dropped one; the compaction overwrites those of the
// rows that stay.  Group numbers need no initial value: only rows that joined a group are asked for it.
// Bound by latency, and with units of tens of thousands of rows by the instructions one SM issues: some ten a row and sweep.  288
// units of 33,280 rows 64 us (115 with three radix sweeps), 512 of 4,700 to 32,700 rows 83 (160), 112 of 8,448 15 (25), 112 of
// 13,312 with a 12,288-row prefix 19 (36), eight of 33,280 27 (50).
// LISTS (want_slot_lists): the defaults of the dropped rows are written already.  Sweep 3 then compares keys with the boundary
// bins' own keys, looks only at the few rows above them, and sets a bit per kept row and one per seed in shared memory; those,
// counted and scanned, give the slots in order, which the compaction takes over.  (The sweeps by range pay for long units only:
// 112 units of 8,448 rows are 2 us slower with them.)  The first three of the figures above become 48, 72 and 17; eight of
// 33,280 23, with the slots.
constexpr int kBins = 2048;
constexpr int kListMax = 1024;

struct DecideSmem {
    union {
        struct { unsigned hist[2][kBins]; } h;                       // sweep 2
        struct {
            unsigned long long cand[3][kListMax];                    // sweep 3: boundary rows of pkeep, c, c + m
            int seeds[kListMax];
        } l;
        SelectSmem plain[2];                                         // radix selection
    };
    unsigned red[4][kSelThreads / 32];
    unsigned warp_cnt[kSelThreads / 32];
    unsigned n_cand[3], n_seeds;
    int bin[3];
    unsigned krem[3], neq[3];
};

// The boundary bins of up to two ranks (descending, 1-based; 0: none) in a histogram.  Fills bin / krem / neq [first..].
__device__ __forceinline__ void boundary_bins(DecideSmem& sm, const unsigned* hist, const unsigned (&rank)[2], int n_ranks, int first) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    static_assert(kBins == 2 * kSelThreads, "two bins per thread");
    const int b0 = kBins - 1 - 2 * tid;                  // this thread's bins, descending: b0, b0 - 1
    const unsigned c0 = hist[b0], c1 = hist[b0 - 1];
    unsigned incl = c0 + c1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    __syncthreads();
    if (lane == 31) sm.warp_cnt[w] = incl;
    __syncthreads();
    unsigned wv = sm.warp_cnt[lane], wincl = wv;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, wincl, off);
        if (lane >= off) wincl += v;
    }
    const unsigned before = __shfl_sync(0xffffffffu, wincl - wv, w) + incl - c0 - c1;
    for (int r = 0; r < n_ranks; ++r) {
        const unsigned k = rank[r];
        if (k > before && k <= before + c0) { sm.bin[first + r] = b0; sm.krem[first + r] = k - before; sm.neq[first + r] = c0; }
        else if (k > before + c0 && k <= before + c0 + c1) {
            sm.bin[first + r] = b0 - 1; sm.krem[first + r] = k - before - c0; sm.neq[first + r] = c1;
        }
    }
}

// Where the slots go (LISTS).
struct SlotLists {
    int words, Bmax, max_B;              // words: of 32 rows, of the longest unit
    int32_t *n_kept, *n_seed, *seed_slot, *slot_src;
    uint8_t* slot_kind;
};

// f(key) of every score in [lo, hi), one CTA, U loads in flight a thread.
template <int U, typename F>
__device__ __forceinline__ void sweep_keys(const float* __restrict__ su, int lo, int hi, F f) {
    int i = lo + (int)threadIdx.x;
    for (; i + (U - 1) * kSelThreads < hi; i += U * kSelThreads) {
        float x[U];
#pragma unroll
        for (int q = 0; q < U; ++q) x[q] = su[i + q * kSelThreads];
#pragma unroll
        for (int q = 0; q < U; ++q) f(order_key(x[q]));
    }
    float x[U];
#pragma unroll
    for (int q = 0; q < U; ++q) x[q] = su[min(i + q * kSelThreads, hi - 1)];
#pragma unroll
    for (int q = 0; q < U; ++q)
        if (i + q * kSelThreads < hi) f(order_key(x[q]));
}

template <int PER_SM, bool LISTS>       // CTAs per SM: one when every unit has an SM of its own (twice the registers, twice the rows in flight)
__global__ void __launch_bounds__(kSelThreads, PER_SM) decide_long_kernel(
    const UnitDesc* __restrict__ desc, const float* __restrict__ s, int32_t* __restrict__ plan,
    uint8_t* __restrict__ kind, int32_t* __restrict__ seed_of, float* __restrict__ sim,
    int32_t* __restrict__ grp, int32_t* __restrict__ seed_rows, unsigned long long* __restrict__ mass_fx,
    int32_t* __restrict__ njoin, int32_t* __restrict__ unit_status, int max_m, int32_t* __restrict__ assign,
    float* __restrict__ weight, SlotLists sl) {
    __shared__ DecideSmem sm;
    extern __shared__ unsigned row_bits[];               // LISTS: [2][sl.words] kept rows, seeds
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int kU = 8 / PER_SM;                       // rows a thread has in flight
    pdl_wait();
    const int u = blockIdx.x;
    const UnitDesc& ud = desc[u];
    const int T = ud.T, P = ud.P;
    const int64_t o = ud.tok_off;
    const float* su = s + o;
    uint8_t* kd_u = kind + o;
    const int pkeep = ud.plan[CASK_PLAN_PKEEP], c = max(0, ud.plan[CASK_PLAN_C]), m = max(0, ud.plan[CASK_PLAN_M]);
    const int r = max(0, min(ud.plan[CASK_PLAN_R], T - P)), hi = T - r, span = hi - P;
    if (tid < 8) plan[u * 8 + tid] = ud.plan[tid];
    for (int j = tid; j <= max_m; j += kSelThreads) mass_fx[(size_t)u * (max_m + 1) + j] = 0ull;
    if (tid == 0) { njoin[u] = 0; unit_status[u] = 0; }
    // which ranks have a boundary inside their range (a selection of nothing or of everything has none)
    const bool sel_p = P > pkeep && pkeep > 0;
    const bool sel_a = c > 0 && c < span, sel_b = m > 0 && c + m < span;
    // ---- sweep 1: key spans
    unsigned mn[2] = {0xffffffffu, 0xffffffffu}, mx[2] = {0u, 0u};
    const int first = sel_p ? 0 : P, last = sel_a || sel_b ? hi : P;      // rows whose scores are looked at
    if constexpr (LISTS) {
        if (sel_p) sweep_keys<kU>(su, 0, P, [&](unsigned k) { mn[0] = min(mn[0], k); mx[0] = max(mx[0], k); });
        if (sel_a || sel_b) sweep_keys<kU>(su, P, hi, [&](unsigned k) { mn[1] = min(mn[1], k); mx[1] = max(mx[1], k); });
        for (int x = tid; x < 2 * sl.words; x += kSelThreads) row_bits[x] = 0u;
    } else {
        for (int i0 = first + tid; i0 < last; i0 += kU * kSelThreads) {
            float x[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q) x[q] = su[min(i0 + q * kSelThreads, last - 1)];
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const unsigned k = order_key(x[q]);
                const int g = min(i0 + q * kSelThreads, last - 1) >= P;
                if (g) { mn[1] = min(mn[1], k); mx[1] = max(mx[1], k); }
                else { mn[0] = min(mn[0], k); mx[0] = max(mx[0], k); }
            }
        }
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        mn[g] = __reduce_min_sync(0xffffffffu, mn[g]);
        mx[g] = __reduce_max_sync(0xffffffffu, mx[g]);
        if (lane == 0) { sm.red[2 * g][w] = mn[g]; sm.red[2 * g + 1][w] = mx[g]; }
    }
    for (int b = tid; b < 2 * kBins; b += kSelThreads) sm.h.hist[0][b] = 0;
    if (tid < 3) sm.n_cand[tid] = 0;
    if (tid == 0) sm.n_seeds = 0;
    __syncthreads();
    unsigned base[2];
    int shift[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        base[g] = __reduce_min_sync(0xffffffffu, sm.red[2 * g][lane]);
        const unsigned top = __reduce_max_sync(0xffffffffu, sm.red[2 * g + 1][lane]);
        const unsigned width = top > base[g] ? top - base[g] : 0u;
        shift[g] = max(0, 32 - __clz((int)width) - 11);      // (top - base) >> shift < 2,048
    }
    // ---- sweep 2: histograms
    if constexpr (LISTS) {
        if (sel_p) sweep_keys<kU>(su, 0, P, [&](unsigned k) { atomicAdd(&sm.h.hist[0][(k - base[0]) >> shift[0]], 1u); });
        if (sel_a || sel_b) sweep_keys<kU>(su, P, hi, [&](unsigned k) { atomicAdd(&sm.h.hist[1][(k - base[1]) >> shift[1]], 1u); });
    } else {
        for (int i0 = first + tid; i0 < last; i0 += kU * kSelThreads) {
            float x[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q) x[q] = su[min(i0 + q * kSelThreads, last - 1)];
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const int i = i0 + q * kSelThreads, g = i >= P;
                if (i < last) atomicAdd(&sm.h.hist[g][(order_key(x[q]) - (g ? base[1] : base[0])) >> (g ? shift[1] : shift[0])], 1u);
            }
        }
    }
    __syncthreads();
    {
        const unsigned rp[2] = {(unsigned)pkeep, 0u}, rs[2] = {(unsigned)c, (unsigned)(c + m)};
        if (sel_p) boundary_bins(sm, sm.h.hist[0], rp, 1, 0);
        if (sel_a || sel_b) boundary_bins(sm, sm.h.hist[1], rs, 2, 1);
    }
    __syncthreads();
    // Boundary bins; a selection of everything cuts below bin 0, one of nothing above the last bin.
    const int bp = sel_p ? sm.bin[0] : (P <= pkeep ? -1 : kBins);
    const int ba = sel_a ? sm.bin[1] : (c > 0 ? -1 : kBins);
    const int bb = sel_b ? sm.bin[2] : (m > 0 ? -1 : ba);
    const unsigned kp = sm.krem[0], ka = sm.krem[1], kb = sm.krem[2];
    const bool over_p = sel_p && sm.neq[0] > kListMax;
    const bool over_s = (sel_a && sm.neq[1] > kListMax) || (sel_b && sm.neq[2] > kListMax) || m > kListMax;
    __syncthreads();                                     // the lists take the histograms' place
    auto mark = [&](int i, uint8_t kd) {
        kd_u[i] = kd;
        if (LISTS) {
            atomicOr(&row_bits[i >> 5], 1u << (i & 31));
            if (kd == CASK_KIND_SEED) atomicOr(&row_bits[sl.words + (i >> 5)], 1u << (i & 31));
        } else if (kd == CASK_KIND_SEED) {
            sm.l.seeds[min(atomicAdd(&sm.n_seeds, 1u), (unsigned)kListMax - 1)] = i;
        }
    };
    // ---- sweep 3: kinds
    if constexpr (LISTS) {
        // As keys: above c* a row is decided, above l* it is listed (0: all, ~0: none; a score's key is never 0).
        auto top_of = [&](int g, int b) {                        // greatest key of bin b
            const unsigned long long v = (unsigned long long)base[g] + ((unsigned long long)(b + 1) << shift[g]);
            return v == 0ull ? 0u : (unsigned)min(v - 1ull, 0xffffffffull);
        };
        const unsigned cp = sel_p ? top_of(0, bp) : P <= pkeep ? 0u : ~0u, lp = sel_p && !over_p ? top_of(0, bp - 1) : cp;
        const unsigned ca = over_s ? ~0u : sel_a ? top_of(1, ba) : c > 0 ? 0u : ~0u, la = sel_a && !over_s ? top_of(1, ba - 1) : ca;
        const unsigned cb = over_s ? ~0u : sel_b ? top_of(1, bb) : m > 0 ? 0u : ~0u, lb = sel_b && !over_s ? top_of(1, bb - 1) : cb;
        const unsigned low_s = min(la, lb);
        for (int i0 = tid; i0 < T; i0 += kU * kSelThreads) {
            float x[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q) x[q] = su[min(i0 + q * kSelThreads, T - 1)];
            unsigned some = 0;                               // rows to look at: most rows of a long unit are dropped
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const int i = i0 + q * kSelThreads;
                if (i < T && (i >= hi || order_key(x[q]) > (i < P ? lp : low_s))) some |= 1u << q;
            }
            for (; some; some &= some - 1) {
                const int at = __ffs(some) - 1, i = i0 + at * kSelThreads;
                float xi = x[0];                             // (out of the registers: a second load is another latency a row, 300 units of 9,000 34.9 us for 33.1)
#pragma unroll
                for (int q = 1; q < kU; ++q) xi = at == q ? x[q] : xi;
                const unsigned key = order_key(xi);
                uint8_t kd = CASK_KIND_DROPPED;
                int list = -1;
                if (i >= hi) kd = CASK_KIND_RECENT;
                else if (i < P) {
                    if (key > cp) kd = CASK_KIND_PREFIX;
                    else list = 0;
                } else if (key > ca) kd = CASK_KIND_CORE;
                else if (key > la) list = 1;
                else if (key > cb) kd = CASK_KIND_SEED;
                else list = 2;
                if (list >= 0) sm.l.cand[list][atomicAdd(&sm.n_cand[list], 1u)] = ((unsigned long long)key << 32) | (0xFFFFFFFFu - (unsigned)i);
                else mark(i, kd);
            }
        }
    } else {
        for (int i0 = tid; i0 < T; i0 += kU * kSelThreads) {
            float x[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q) x[q] = su[min(i0 + q * kSelThreads, T - 1)];
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const int i = i0 + q * kSelThreads;
                if (i >= T) break;
                const unsigned key = order_key(x[q]);
                const unsigned long long pair = ((unsigned long long)key << 32) | (0xFFFFFFFFu - (unsigned)i);
                uint8_t kd = CASK_KIND_DROPPED;
                if (i < P) {
                    const int b = sel_p ? (int)((key - base[0]) >> shift[0]) : 0;
                    if (b > bp) kd = CASK_KIND_PREFIX;
                    else if (sel_p && b == bp && !over_p) sm.l.cand[0][atomicAdd(&sm.n_cand[0], 1u)] = pair;
                } else if (i >= hi) {
                    kd = CASK_KIND_RECENT;
                } else if (!over_s) {
                    const int b = sel_a || sel_b ? (int)((key - base[1]) >> shift[1]) : 0;
                    if (b > ba) kd = CASK_KIND_CORE;
                    else if (sel_a && b == ba) sm.l.cand[1][atomicAdd(&sm.n_cand[1], 1u)] = pair;
                    else if (m > 0 && b > bb) kd = CASK_KIND_SEED;
                    else if (sel_b && b == bb) sm.l.cand[2][atomicAdd(&sm.n_cand[2], 1u)] = pair;
                    if (kd == CASK_KIND_SEED) sm.l.seeds[min(atomicAdd(&sm.n_seeds, 1u), (unsigned)kListMax - 1)] = i;
                }
                kd_u[i] = kd;
                seed_of[o + i] = -1;
                assign[o + i] = -1;
                weight[o + i] = 0.f;
                if (sim) sim[o + i] = -2.f;
            }
        }
    }
    __syncthreads();
    // ---- boundary rows by exact rank
    for (int x = 0; x < 3; ++x) {
        const int n = (int)sm.n_cand[x];
        for (int t = tid; t < n; t += kSelThreads) {
            const unsigned long long me = sm.l.cand[x][t];
            unsigned ahead = 0;
            for (int y = 0; y < n; ++y) ahead += sm.l.cand[x][y] > me;
            const int i = (int)(0xFFFFFFFFu - (unsigned)me);
            uint8_t kd = CASK_KIND_DROPPED;
            if (x == 0) kd = ahead < kp ? CASK_KIND_PREFIX : CASK_KIND_DROPPED;
            else if (x == 1) {
                // the rest of the bin of rank c: seeds, up to rank c + m when that lies in the same bin
                if (ahead < ka) kd = CASK_KIND_CORE;
                else if (m > 0 && (bb < ba || ahead < kb)) kd = CASK_KIND_SEED;
            } else if (ahead < kb) {
                kd = CASK_KIND_SEED;
            }
            if (kd != CASK_KIND_DROPPED) mark(i, kd);
        }
    }
    __syncthreads();
    if (LISTS && !over_p && !over_s) {
        // ---- slots: kept rows in ascending order, the seeds numbered among themselves
        const int words = (T + 31) >> 5, per = (words + kSelThreads - 1) / kSelThreads, w0 = tid * per;
        unsigned n = 0;                                  // kept rows, seeds << 16 of this thread's words
        for (int x = w0; x < min(w0 + per, words); ++x)
            n += (unsigned)__popc(row_bits[x]) | ((unsigned)__popc(row_bits[sl.words + x]) << 16);
        unsigned incl = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        if (lane == 31) sm.warp_cnt[w] = incl;
        __syncthreads();
        unsigned wincl = sm.warp_cnt[lane];
        const unsigned wv = wincl;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, wincl, off);
            if (lane >= off) wincl += v;
        }
        if (tid == kSelThreads - 1) {
            sl.n_kept[u] = min((int)(wincl & 0xFFFFu), sl.Bmax);
            sl.n_seed[u] = min((int)(wincl >> 16), m);
        }
        unsigned run = __shfl_sync(0xffffffffu, wincl - wv, w) + incl - n;
        auto emit = [&](int i, int t, int j, bool seed) {
            if (t < sl.Bmax) {
                sl.slot_src[(size_t)u * sl.Bmax + t] = i;
                sl.slot_kind[(size_t)u * sl.Bmax + t] =
                    i < P ? CASK_KIND_PREFIX : i >= hi ? CASK_KIND_RECENT : seed ? CASK_KIND_SEED : CASK_KIND_CORE;
            }
            if (seed && j < m) {
                seed_rows[ud.seed_base + j] = i;
                seed_of[o + i] = i;
                grp[o + i] = j;
                sl.seed_slot[(size_t)u * sl.max_B + j] = min(t, sl.Bmax - 1);
            }
        };
        for (int x = 0; x < per; ++x) {
            // a word with few rows is its thread's; the full ones (kept prefix, recent rows) the warp takes one by one, a lane a row
            unsigned keep = w0 + x < words ? row_bits[w0 + x] : 0u;
            const unsigned seeds = w0 + x < words ? row_bits[sl.words + w0 + x] : 0u, all = keep;
            const bool dense = __popc(keep) > 6;
            for (unsigned todo = __ballot_sync(0xffffffffu, dense); todo; todo &= todo - 1) {
                const int from = __ffs(todo) - 1;
                const unsigned kw = __shfl_sync(0xffffffffu, all, from), sw = __shfl_sync(0xffffffffu, seeds, from);
                const unsigned at = __shfl_sync(0xffffffffu, run, from), below = (1u << lane) - 1u;
                if ((kw >> lane) & 1u)
                    emit(32 * ((32 * w + from) * per + x) + lane, (int)(at & 0xFFFFu) + __popc(kw & below), (int)(at >> 16) + __popc(sw & below),
                         (sw >> lane) & 1u);
            }
            for (unsigned at = run; !dense && keep; keep &= keep - 1) {
                const int b = __ffs(keep) - 1;
                const bool seed = (seeds >> b) & 1u;
                emit(32 * (w0 + x) + b, (int)(at & 0xFFFFu), (int)(at >> 16), seed);
                at += 1u + ((unsigned)seed << 16);
            }
            __syncwarp();
            run += (unsigned)__popc(all) | ((unsigned)__popc(seeds) << 16);
        }
        return;
    }
    if (LISTS && tid == 0) sl.n_kept[u] = -1;         // the compaction finds the slots itself
    if (LISTS && !over_s && m > 0) {
        // (the prefix goes through the radix selection)  seeds in any order, sorted below
        for (int x = tid; x < (T + 31) >> 5; x += kSelThreads)
            for (unsigned b = row_bits[sl.words + x]; b; b &= b - 1)
                sm.l.seeds[min(atomicAdd(&sm.n_seeds, 1u), (unsigned)kListMax - 1)] = 32 * x + __ffs(b) - 1;
        __syncthreads();
    }
    if (!over_s && m > 0) {
        // the seeds in ascending row order: every seed counts the lower ones
        const int ns = min(min((int)sm.n_seeds, m), kListMax);
        for (int t = tid; t < ns; t += kSelThreads) {
            const int i = sm.l.seeds[t];
            int at = 0;
            for (int y = 0; y < ns; ++y) at += sm.l.seeds[y] < i;
            seed_rows[ud.seed_base + at] = i;
            seed_of[o + i] = i;
            grp[o + i] = at;
        }
    }
    if (!over_p && !over_s) return;
    // ---- thousands of equal scores at a boundary (or more seeds than a list holds): radix selection
    __syncthreads();
    if (over_p) {
        for (int i = tid; i < P; i += kSelThreads) kd_u[i] = CASK_KIND_DROPPED;
        __syncthreads();
        block_topk_mark(su, kd_u, 0, P, pkeep, CASK_KIND_PREFIX, sm.plain[0]);
        __syncthreads();
    }
    if (!over_s) return;
    block_topk2_mark<true>(su, kd_u, P, hi, c, CASK_KIND_CORE, m, CASK_KIND_SEED, sm.plain[0], sm.plain[1]);
    if (m <= 0) return;
    block_ordered_rows(kd_u, P, hi, CASK_KIND_SEED, sm.plain[0], [&](unsigned idx, int i) {
        if (idx < (unsigned)m) {
            seed_rows[ud.seed_base + idx] = i;
            seed_of[o + i] = i;
            grp[o + i] = (int)idx;
        }
    });
}

// ---- seed keys: gathered in the layout the assignment kernel wants, with their norms ---------------------------------------
template <typename T>
struct SeedTable {
    const T* K;
    T* seed_k;
    float* seed_norm;
    int layout;                      // SeedLayout
    int64_t part_rows;
};

template <typename T> struct alignas(4 * sizeof(T)) Four { T x[4]; };

// Four neighbouring channels from c on of seed row `at`.
template <typename T>
__device__ __forceinline__ void store_seed(const SeedTable<T>& t, const Shape& sh, int64_t at, int c, const Four<T>& x, const float (&wc)[4]) {
    const int d = sh.d;
    if (t.layout == SEED_PAIR) {
        Four<T> hi, lo;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float wf = wc[k] * Elem<T>::ld(&x.x[k]);
            Elem<T>::st(&hi.x[k], wf);
            Elem<T>::st(&lo.x[k], wf - Elem<T>::ld(&hi.x[k]));
        }
        T* dst = t.seed_k + at * 2 * d + c;
        *reinterpret_cast<Four<T>*>(dst) = hi;
        *reinterpret_cast<Four<T>*>(dst + d) = lo;
    } else if (t.layout == SEED_SPLIT) {
        Four<__nv_bfloat16> p[3];
#pragma unroll
        for (int k = 0; k < 4; ++k) split3(Elem<T>::ld(&x.x[k]), p[0].x[k], p[1].x[k], p[2].x[k]);
        __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(t.seed_k) + at * d + c;
#pragma unroll
        for (int k = 0; k < 3; ++k) *reinterpret_cast<Four<__nv_bfloat16>*>(dst + k * t.part_rows * d) = p[k];
    } else {
        *reinterpret_cast<Four<T>*>(t.seed_k + at * d + c) = x;
    }
}

// The unit's seeds j = j0, j0 + step, ... below m, one warp a row and R rows in flight: offsets first, loads after, with no branch
// between the loads (a branch per row makes every row wait for the one before).  A lane holds four neighbouring channels, so
// d <= 128 is one round.  off_of(j): element offset of seed j's key.
// The norm is the sum over the lanes l of the chains f_l^2 + f_(l+32)^2 + ..., so the row goes through `pass`, the warp's own 128
// elements of shared memory, to be read that way round.  That order of additions is kept because two seeds whose cosines with a row
// agree to 1e-7 are told apart by it.  (3,072 units of 640 rows: 80 us; the chains handed from lane to lane by shuffles 93, the
// row's channels read a second time from memory 95, sums over a lane's four neighbouring channels, in another order, 68.)
template <int R, typename T, typename OffOf>
__device__ __forceinline__ void gather_seeds(const SeedTable<T>& t, const Shape& sh, int64_t base, int j0, int step, int m, T* pass, OffOf off_of) {
    const int lane = threadIdx.x & 31, d = sh.d;
    for (; j0 < m; j0 += R * step) {
        int64_t off[R];
#pragma unroll
        for (int q = 0; q < R; ++q) off[q] = off_of(min(j0 + q * step, m - 1));
        float n2[R];
#pragma unroll
        for (int q = 0; q < R; ++q) n2[q] = 0.f;
        for (int c0 = 0; c0 < d; c0 += 128) {
            const int c = c0 + 4 * lane;
            Four<T> x[R];
            float wc[4] = {1.f, 1.f, 1.f, 1.f}, wl[4] = {1.f, 1.f, 1.f, 1.f};        // weights of channels c + k, c0 + lane + 32 k
            if (c < d) {
#pragma unroll
                for (int q = 0; q < R; ++q) x[q] = *reinterpret_cast<const Four<T>*>(t.K + off[q] + c);
            }
            if (sh.chan_w) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (c < d) wc[k] = sh.chan_w[c + k];
                    if (c0 + lane + 32 * k < d) wl[k] = sh.chan_w[c0 + lane + 32 * k];
                }
            }
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (c < d) {
                    if (j0 + q * step < m) store_seed(t, sh, base + j0 + q * step, c, x[q], wc);
                    reinterpret_cast<Four<T>*>(pass)[lane] = x[q];
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float f = c0 + lane + 32 * k < d ? Elem<T>::ld(&pass[lane + 32 * k]) : 0.f;
                    n2[q] = fmaf(wl[k] * f, f, n2[q]);
                }
                __syncwarp();
            }
        }
#pragma unroll
        for (int q = 0; q < R; ++q) {
            float n = n2[q];
#pragma unroll
            for (int sft = 16; sft >= 1; sft >>= 1) n += __shfl_xor_sync(0xffffffffu, n, sft);
            if (lane == 0 && j0 + q * step < m) t.seed_norm[base + j0 + q * step] = sqrtf(n);
        }
    }
}

// ---- 2. gather of the seed keys: a launch of its own, but for short units ----------------------------------------------------------
// One warp a seed.  Bound by latency (seed list, page table, key), so the SM is kept full of warps, each with one row; two or
// four rows a warp are no faster.  512 paged units of some 130 seeds each 21 us (25 with the registers unbounded and two-byte
// loads), 112 contiguous ones of 128 seeds 10.7.
constexpr int kGatherWarps = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kGatherWarps, 8) seed_gather_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, SeedTable<T> tab, const int32_t* __restrict__ plan, const float* __restrict__ s,
    const int32_t* __restrict__ seed_rows, unsigned long long* __restrict__ mass_fx, int max_m, float eps) {
    pdl_wait();
    const int u = blockIdx.y, j = blockIdx.x * kGatherWarps + (threadIdx.x >> 5);
    const UnitDesc& ud = desc[u];
    const int m = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
    if (j >= m) return;
    const int row = CASK_IDX(seed_rows[ud.seed_base + j], ud.T, sh.err);
    __shared__ alignas(16) T pass[kGatherWarps][128];
    gather_seeds<1>(tab, sh, ud.seed_base, j, 1, j + 1, pass[threadIdx.x >> 5], [&](int) { return row_elem_off(sh, ud, ud.k_off, row); });
    if ((threadIdx.x & 31) == 0) mass_fx[(size_t)u * (max_m + 1) + j] = mass_to_fx(row_mass(sh, s, eps, ud.tok_off + row));
}

// ---- 1+2 for units of at most kSmallSpan rows: prefix eviction, core selection, seed selection and the seed gather in one CTA
// per unit (the event path; the staged calls keep their own kernels and give the same result).  Keys and kinds live in shared
// memory; the boundary ranks come out of one histogram per range over the keys' own span, and rows inside a boundary bin are
// ranked by counting, as in decide_long_kernel.  (Ranking every row by counting is quadratic: two units of 1,024 rows took
// 34 us, now 12.)  Bound by latency, and with thousands of units by the seeds' scattered rows: half the time goes to the gather,
// so the block table is read at the start and four rows a warp are in flight.
// Threads a unit (THREADS, PER_SM): every step but the gather is a chain of short latencies, and the gather takes m / (4 * warps) rounds of
// one more, so a unit that has an SM to itself gets as many threads as it has use for: 1,024, or 512 where it has no more rows.
// With several units an SM the chains of one hide behind those of the others: 512 up to three units an SM, then 256.
// Event in us with 256, 512 and 1,024: 8 units of 640 rows 50.5, 44.5, 44.5; 4 of 1,000 (m = 128) 61.8, 52.6, 50.6; 100 of 1,000 118, 108, 106;
// 148 of 330 55.3, 54.1, 55.1; 200 of 640 115, 109, 113; 288 of 640 146, 137, 141; 440 of 640 191, 188; 600 of 1,000 410, 412; 1,200
// of 640 462, 461; 3,072 of 640 1,136, 1,155.  256 threads four an SM, which spill nothing: kernel of those 3,072 78.9 to 70.5 us, where five
// an SM (48 registers) spilled 96 bytes a thread; 512 three an SM (40 registers) 90.6.
constexpr int kSmallBins = 1024;
template <typename T, int THREADS, int PER_SM>
__global__ void __launch_bounds__(THREADS, PER_SM) decide_small_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, SeedTable<T> tab, const float* __restrict__ s, int32_t* __restrict__ plan,
    uint8_t* __restrict__ kind, int32_t* __restrict__ seed_of, float* __restrict__ sim, int32_t* __restrict__ grp,
    int32_t* __restrict__ seed_rows, unsigned long long* __restrict__ mass_fx, int32_t* __restrict__ njoin,
    int32_t* __restrict__ unit_status, int max_m, float eps) {
    constexpr int kPer = kSmallSpan / THREADS, kWarps = THREADS / 32, kPerBin = kSmallBins / THREADS;
    static_assert(kSmallSpan == kSmallBins && kPer >= 1 && kWarps <= 32, "rows and bins go to the threads alike");
    __shared__ alignas(16) unsigned keys[kSmallSpan];
    __shared__ uint8_t kd[kSmallSpan];
    __shared__ int32_t pages[kSmallSpan];                // the unit's block table: looked up before it is needed
    __shared__ union {
        unsigned hist[2][kSmallBins];
        struct { int16_t cand[3][kSmallSpan]; int16_t seeds[kSmallSpan]; } l;
    } sm;
    __shared__ unsigned red[4][kWarps], wsum[2][kWarps], n_cand[3], n_seeds;
    __shared__ int bin[3];
    __shared__ unsigned krem[3];
    pdl_wait();
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const UnitDesc& ud = desc[u];
    const int T_ = ud.T, P = ud.P;
    const int64_t o = ud.tok_off;
    const int pkeep = ud.plan[CASK_PLAN_PKEEP], c = max(0, ud.plan[CASK_PLAN_C]), m = max(0, ud.plan[CASK_PLAN_M]);
    const int r = max(0, min(ud.plan[CASK_PLAN_R], T_ - P)), hi = T_ - r, span = hi - P;
    mass_fx += (size_t)u * (max_m + 1);
    if (tid < 8) plan[u * 8 + tid] = ud.plan[tid];
    // which ranks have a boundary inside their range (a selection of nothing or of everything has none)
    const bool sel_p = P > pkeep && pkeep > 0, sel_a = c > 0 && c < span, sel_b = m > 0 && c + m < span;
    unsigned key[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) key[q] = tid + q * THREADS < T_ ? order_key(s[o + tid + q * THREADS]) : 0u;
    if (sh.page_size > 0)
        for (int x = tid; x * sh.page_size < T_; x += THREADS) pages[x] = sh.bt[ud.bt0 + x];
    // ---- key spans of the prefix (0) and the scratch range (1)
    unsigned mn[2] = {0xffffffffu, 0xffffffffu}, mx[2] = {0u, 0u};
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int i = tid + q * THREADS;
        keys[i] = key[q];
        if (i < P) { mn[0] = min(mn[0], key[q]); mx[0] = max(mx[0], key[q]); }
        else if (i < hi) { mn[1] = min(mn[1], key[q]); mx[1] = max(mx[1], key[q]); }
        sm.hist[0][i] = 0u;
        sm.hist[1][i] = 0u;
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        mn[g] = __reduce_min_sync(0xffffffffu, mn[g]);
        mx[g] = __reduce_max_sync(0xffffffffu, mx[g]);
        if (lane == 0) { red[2 * g][w] = mn[g]; red[2 * g + 1][w] = mx[g]; }
    }
    if (tid < 3) n_cand[tid] = 0;
    if (tid == 0) { n_seeds = 0; njoin[u] = 0; unit_status[u] = 0; mass_fx[max_m] = 0ull; }
    __syncthreads();
    unsigned base[2];
    int shift[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        base[g] = __reduce_min_sync(0xffffffffu, red[2 * g][lane & (kWarps - 1)]);
        const unsigned top = __reduce_max_sync(0xffffffffu, red[2 * g + 1][lane & (kWarps - 1)]);
        const unsigned width = top > base[g] ? top - base[g] : 0u;
        shift[g] = max(0, 32 - __clz((int)width) - 10);      // (top - base) >> shift < 1,024
    }
    auto bin_of = [&](int q, int g) { return (int)((key[q] - base[g]) >> shift[g]); };
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int i = tid + q * THREADS;
        if (i < P ? sel_p : (i < hi && (sel_a || sel_b))) atomicAdd(&sm.hist[i >= P][i < P ? bin_of(q, 0) : bin_of(q, 1)], 1u);
    }
    __syncthreads();
    // ---- bins that hold the ranks pkeep, c and c + m: each thread has kPerBin bins of either histogram, in descending order
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        unsigned h[kPerBin], tot = 0;
#pragma unroll
        for (int x = 0; x < kPerBin; ++x) { h[x] = sm.hist[g][kSmallBins - 1 - kPerBin * tid - x]; tot += h[x]; }
        unsigned incl = tot;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        if (lane == 31) wsum[g][w] = incl;
        __syncthreads();
        unsigned before = incl - tot + __reduce_add_sync(0xffffffffu, lane < w ? wsum[g][lane] : 0u);
        const unsigned rank[2] = {(unsigned)(g == 0 ? (sel_p ? pkeep : 0) : (sel_a ? c : 0)), (unsigned)(g == 1 && sel_b ? c + m : 0)};
#pragma unroll
        for (int x = 0; x < kPerBin; ++x) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (rank[k] > before && rank[k] <= before + h[x]) {
                    bin[g + k] = kSmallBins - 1 - kPerBin * tid - x;
                    krem[g + k] = rank[k] - before;
                }
            before += h[x];
        }
    }
    __syncthreads();
    // a selection of everything cuts below bin 0, one of nothing above the last bin
    const int bp = sel_p ? bin[0] : (P <= pkeep ? -1 : kSmallBins);
    const int ba = sel_a ? bin[1] : (c > 0 ? -1 : kSmallBins);
    const int bb = sel_b ? bin[2] : (m > 0 ? -1 : ba);
    const unsigned kp = krem[0], ka = krem[1], kb = krem[2];
    // ---- kinds; rows inside a boundary bin are listed (the lists take the histograms' place)
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int i = tid + q * THREADS;
        uint8_t k = CASK_KIND_DROPPED;
        int list = -1;
        if (i < P) {
            const int b = sel_p ? bin_of(q, 0) : 0;
            if (b > bp) k = CASK_KIND_PREFIX;
            else if (sel_p && b == bp) list = 0;
        } else if (i >= hi) {
            k = CASK_KIND_RECENT;
        } else {
            const int b = sel_a || sel_b ? bin_of(q, 1) : 0;
            if (b > ba) k = CASK_KIND_CORE;
            else if (sel_a && b == ba) list = 1;
            else if (m > 0 && b > bb) k = CASK_KIND_SEED;
            else if (sel_b && b == bb) list = 2;
        }
        if (i < T_) {
            kd[i] = k;
            if (list >= 0) sm.l.cand[list][atomicAdd(&n_cand[list], 1u)] = (int16_t)i;
        }
    }
    __syncthreads();
    for (int x = 0; x < 3; ++x) {
        const int n = (int)n_cand[x];
        for (int t = tid; t < n; t += THREADS) {
            const int i = sm.l.cand[x][t];
            const unsigned me = keys[i];
            unsigned ahead = 0;
            for (int y = 0; y < n; ++y) {
                const int j = sm.l.cand[x][y];
                ahead += keys[j] > me || (keys[j] == me && j < i);
            }
            if (x == 0) { if (ahead < kp) kd[i] = CASK_KIND_PREFIX; }
            else if (x == 1) {
                // the rest of the bin of rank c: seeds, up to rank c + m when that lies in the same bin
                if (ahead < ka) kd[i] = CASK_KIND_CORE;
                else if (m > 0 && (bb < ba || ahead < kb)) kd[i] = CASK_KIND_SEED;
            } else if (ahead < kb) {
                kd[i] = CASK_KIND_SEED;
            }
        }
    }
    __syncthreads();
    // ---- outputs; the seeds in ascending row order (a warp's rows are contiguous: one ballot a step, one sum over warps)
    const int i0 = w * (kSmallSpan / kWarps);
    unsigned ballots[kPer], mine = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int i = i0 + 32 * q + lane;
        ballots[q] = __ballot_sync(0xffffffffu, i < T_ && kd[i] == CASK_KIND_SEED);
        mine += __popc(ballots[q]);
    }
    if (lane == 0) wsum[0][w] = mine;
    __syncthreads();
    const unsigned of_warp = lane < kWarps ? wsum[0][lane] : 0u;
    const unsigned all = __reduce_add_sync(0xffffffffu, of_warp);
    unsigned rank = __reduce_add_sync(0xffffffffu, lane < w ? of_warp : 0u);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int i = i0 + 32 * q + lane;
        if (i < T_) {
            const bool seed = (ballots[q] >> lane) & 1u;
            const int at = (int)(rank + __popc(ballots[q] & ((1u << lane) - 1u)));
            kind[o + i] = kd[i];
            seed_of[o + i] = seed ? i : -1;
            if (sim) sim[o + i] = -2.f;
            if (seed) {
                sm.l.seeds[at] = (int16_t)i;
                seed_rows[ud.seed_base + at] = i;
                grp[o + i] = at;
            }
        }
        rank += __popc(ballots[q]);
    }
    __syncthreads();
    const int ns = min((int)all, m);
    for (int j = tid; j < ns; j += THREADS) mass_fx[j] = mass_to_fx(row_mass(sh, s, eps, o + sm.l.seeds[j]));
    constexpr size_t kPass = kWarps * 128 * sizeof(T);       // for the gather: the keys are no longer needed, but may be too small a place
    __shared__ alignas(16) uint8_t more[kPass > sizeof(keys) ? kPass : 16];
    T* pass = reinterpret_cast<T*>(kPass > sizeof(keys) ? more : reinterpret_cast<uint8_t*>(keys)) + 128 * w;
    gather_seeds<4>(tab, sh, ud.seed_base, w, kWarps, ns, pass, [&](int j) {
        const int i = sm.l.seeds[j];
        if (sh.page_size == 0) return ud.k_off + (int64_t)i * sh.row_stride;
        const int x = i / sh.page_size;
        return page_row(sh, pages[x], i - x * sh.page_size) * sh.row_stride;
    });
}

// ---- 3. assignment: cosine of every scratch row against every seed, argmax, threshold -----
template <typename T>
__global__ void __launch_bounds__(kThreads) assign_simt_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const T* __restrict__ K, const float* __restrict__ s,
    const int32_t* __restrict__ plan, const int32_t* __restrict__ seed_rows, const T* __restrict__ seed_k,
    const float* __restrict__ seed_norm, uint8_t* __restrict__ kind, int32_t* __restrict__ seed_of,
    float* __restrict__ sim, int32_t* __restrict__ grp, unsigned long long* __restrict__ mass_fx,
    int32_t* __restrict__ njoin, int max_m, float tau, float eps) {
    extern __shared__ float smem[];
    const int u = blockIdx.y;
    const UnitDesc& ud = desc[u];
    const int T_ = ud.T, P = ud.P;
    const int r = max(0, min(plan[u * 8 + CASK_PLAN_R], T_ - P));
    const int m = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
    const int lo = P + blockIdx.x * kTile, hi = T_ - r;
    if (m <= 0 || lo >= hi) return;
    const int d = sh.d, pitch = d + 1;
    float* St = smem;
    float* Rt = smem + kTile * pitch;
    float* rnorm = Rt + kTile * pitch;     // [64] norms of the stationary rows
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    const int nrows = min(kTile, hi - lo);

    // stationary tile: 64 candidate rows
    {
        const int vec_per_row = d / 8;
        for (int idx = threadIdx.x; idx < kTile * vec_per_row; idx += kThreads) {
            int rr = idx / vec_per_row, c8 = (idx % vec_per_row) * 8;
#pragma unroll
            for (int t = 0; t < 8; ++t)
                St[rr * pitch + c8 + t] =
                    (rr < nrows) ? Elem<T>::ld(K + row_elem_off(sh, ud, ud.k_off, lo + rr) + c8 + t) : 0.f;
        }
    }
    __syncthreads();
    {
        // 4 threads per row, fixed combination order
        int rr = threadIdx.x / 4, part = threadIdx.x % 4;
        float n2 = 0.f;
        for (int c = part; c < d; c += 4) n2 = fmaf((sh.chan_w ? sh.chan_w[c] : 1.f) * St[rr * pitch + c], St[rr * pitch + c], n2);
        n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
        n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
        if (part == 0) rnorm[rr] = sqrtf(n2);
    }
    float best[4];
    int best_u[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) { best[a] = -INFINITY; best_u[a] = -1; }

    for (int u0 = 0; u0 < m; u0 += kTile) {
        __syncthreads();
        const int vec_per_row = d / 8;
        const int nseed = min(kTile, m - u0);
        for (int idx = threadIdx.x; idx < kTile * vec_per_row; idx += kThreads) {
            int rr = idx / vec_per_row, c8 = (idx % vec_per_row) * 8;
#pragma unroll
            for (int t = 0; t < 8; ++t)
                Rt[rr * pitch + c8 + t] =
                    (rr < nseed) ? (sh.chan_w ? sh.chan_w[c8 + t] : 1.f) *
                                       Elem<T>::ld(seed_k + (size_t)(ud.seed_base + u0 + rr) * d + c8 + t)
                                 : 0.f;
        }
        __syncthreads();
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
#pragma unroll 4
        for (int c = 0; c < d; ++c) {
            float sa[4], rb[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) sa[a] = St[(ty + 16 * a) * pitch + c];
#pragma unroll
            for (int b = 0; b < 4; ++b) rb[b] = Rt[(tx + 16 * b) * pitch + c];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(sa[a], rb[b], acc[a][b]);
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int su = u0 + tx + 16 * b;
            if (su >= m) continue;
            float nu = seed_norm[ud.seed_base + su];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                float nj = rnorm[ty + 16 * a];
                float sm_ = (nj > 0.f && nu > 0.f) ? acc[a][b] / (nj * nu) : 0.f;
                if (sm_ > best[a]) { best[a] = sm_; best_u[a] = su; }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) {
            float ob = __shfl_xor_sync(0xffffffffu, best[a], off);
            int ou = __shfl_xor_sync(0xffffffffu, best_u[a], off);
            if (ou >= 0 && (ob > best[a] || (ob == best[a] && ou < best_u[a]) || best_u[a] < 0)) {
                best[a] = ob;
                best_u[a] = ou;
            }
        }
        int rr = ty + 16 * a;
        int i = lo + rr;
        if (tx == 0 && rr < nrows && kind[ud.tok_off + i] == CASK_KIND_DROPPED) {
            if (sim) sim[ud.tok_off + i] = best[a];
            unsigned long long fx = mass_to_fx(row_mass(sh, s, eps, ud.tok_off + i));
            if (best_u[a] >= 0 && best[a] >= tau) {
                kind[ud.tok_off + i] = CASK_KIND_MERGED;
                seed_of[ud.tok_off + i] = seed_rows[ud.seed_base + CASK_IDX(best_u[a], m, sh.err)];
                grp[ud.tok_off + i] = best_u[a];
                atomicAdd(&mass_fx[(size_t)u * (max_m + 1) + best_u[a]], fx);
                atomicAdd(&njoin[u], 1);
            } else {
                atomicAdd(&mass_fx[(size_t)u * (max_m + 1) + max_m], fx);
            }
        }
    }
}

// ---- 3b. assignment under the un-squared per-band distance of Sec. 2.5 -----------------------------------------
// d_kappa(k_j, k_u) = sum_f w_f ||k_jf - k_uf||_2 over the rotary bands (pairs of channels), used as the similarity
// 1 - d_kappa / (D_j + D_u), D_x = sum_f w_f ||k_xf||_2.  One square root per (row, seed, band), so the special-
// function pipe bounds it; same tiling as assign_simt_kernel (64 rows x 64 seeds per step, 4 x 4 per thread).
__device__ __forceinline__ float sqrt_fast(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <typename T>
__global__ void __launch_bounds__(kThreads) assign_band_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const T* __restrict__ K, const float* __restrict__ s,
    const int32_t* __restrict__ plan, const int32_t* __restrict__ seed_rows, const T* __restrict__ seed_k,
    uint8_t* __restrict__ kind, int32_t* __restrict__ seed_of, float* __restrict__ sim, int32_t* __restrict__ grp,
    unsigned long long* __restrict__ mass_fx, int32_t* __restrict__ njoin, int max_m, float tau, float eps) {
    extern __shared__ float2 smem2[];
    const int u = blockIdx.y;
    const UnitDesc& ud = desc[u];
    const int T_ = ud.T, P = ud.P;
    const int r = max(0, min(plan[u * 8 + CASK_PLAN_R], T_ - P));
    const int m = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
    const int lo = P + blockIdx.x * kTile, hi = T_ - r;
    if (m <= 0 || lo >= hi) return;
    const int d = sh.d, nb = d / 2, pitch = nb + 1;      // a row is nb bands of (x, y); odd pitch: no bank conflicts
    float2* St = smem2;                                   // [64][pitch] stationary rows
    float2* Rt = St + kTile * pitch;                      // [64][pitch] seeds of the current step
    float* rlen = reinterpret_cast<float*>(Rt + kTile * pitch);   // [64] D of the stationary rows
    float* slen = rlen + kTile;                           // [64] D of the seeds of the current step
    float* bw = slen + kTile;                             // [d/2] band weights
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    const int nrows = min(kTile, hi - lo);
    const int second = sh.band_layout == 0 ? nb : 1, step = sh.band_layout == 0 ? 1 : 2;   // band f: channels (f*step, f*step + second)
    for (int f = threadIdx.x; f < nb; f += kThreads) bw[f] = sh.band_w[f];
    // rows of a tile into band order
    auto stage = [&](float2* dst, const T* base, int64_t row_off, bool valid, int rr, int f) {
        float2 v = make_float2(0.f, 0.f);
        if (valid) {
            v.x = Elem<T>::ld(base + row_off + f * step);
            v.y = Elem<T>::ld(base + row_off + f * step + second);
        }
        dst[rr * pitch + f] = v;
    };
    for (int idx = threadIdx.x; idx < kTile * nb; idx += kThreads) {
        const int rr = idx / nb, f = idx % nb;
        stage(St, K, rr < nrows ? row_elem_off(sh, ud, ud.k_off, lo + rr) : 0, rr < nrows, rr, f);
    }
    __syncthreads();
    // D of a row: four threads per row, a quarter of the bands each, fixed combination order
    auto band_len = [&](const float2* row, int part) {
        float D = 0.f;
        for (int f = part; f < nb; f += 4) {
            const float2 v = row[f];
            D = fmaf(bw[f], sqrt_fast(fmaf(v.x, v.x, v.y * v.y)), D);
        }
        D += __shfl_xor_sync(0xffffffffu, D, 1);
        D += __shfl_xor_sync(0xffffffffu, D, 2);
        return D;
    };
    {
        const int rr = threadIdx.x / 4, part = threadIdx.x % 4;
        const float D = band_len(St + rr * pitch, part);
        if (part == 0) rlen[rr] = D;
    }
    float best[4];
    int best_u[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) { best[a] = -INFINITY; best_u[a] = -1; }

    for (int u0 = 0; u0 < m; u0 += kTile) {
        __syncthreads();
        const int nseed = min(kTile, m - u0);
        for (int idx = threadIdx.x; idx < kTile * nb; idx += kThreads) {
            const int rr = idx / nb, f = idx % nb;
            stage(Rt, seed_k, (int64_t)(ud.seed_base + u0 + rr) * d, rr < nseed, rr, f);
        }
        __syncthreads();
        {
            const int rr = threadIdx.x / 4, part = threadIdx.x % 4;
            const float D = band_len(Rt + rr * pitch, part);
            if (part == 0) slen[rr] = D;
        }
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
#pragma unroll 2
        for (int f = 0; f < nb; ++f) {
            const float w = bw[f];
            float2 sv[4], rv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) sv[a] = St[(ty + 16 * a) * pitch + f];
#pragma unroll
            for (int b = 0; b < 4; ++b) rv[b] = Rt[(tx + 16 * b) * pitch + f];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const float dx = sv[a].x - rv[b].x, dy = sv[a].y - rv[b].y;
                    acc[a][b] = fmaf(w, sqrt_fast(fmaf(dx, dx, dy * dy)), acc[a][b]);
                }
        }
        __syncthreads();        // slen is complete
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int su = u0 + tx + 16 * b;
            if (su >= m) continue;
            const float Du = slen[tx + 16 * b];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float Dj = rlen[ty + 16 * a];
                float sm_ = (Dj > 0.f && Du > 0.f) ? 1.f - acc[a][b] / (Dj + Du) : 0.f;
                if (sm_ > best[a]) { best[a] = sm_; best_u[a] = su; }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) {
            float ob = __shfl_xor_sync(0xffffffffu, best[a], off);
            int ou = __shfl_xor_sync(0xffffffffu, best_u[a], off);
            if (ou >= 0 && (ob > best[a] || (ob == best[a] && ou < best_u[a]) || best_u[a] < 0)) {
                best[a] = ob;
                best_u[a] = ou;
            }
        }
        int rr = ty + 16 * a;
        int i = lo + rr;
        if (tx == 0 && rr < nrows && kind[ud.tok_off + i] == CASK_KIND_DROPPED) {
            if (sim) sim[ud.tok_off + i] = best[a];
            unsigned long long fx = mass_to_fx(row_mass(sh, s, eps, ud.tok_off + i));
            if (best_u[a] >= 0 && best[a] >= tau) {
                kind[ud.tok_off + i] = CASK_KIND_MERGED;
                seed_of[ud.tok_off + i] = seed_rows[ud.seed_base + CASK_IDX(best_u[a], m, sh.err)];
                grp[ud.tok_off + i] = best_u[a];
                atomicAdd(&mass_fx[(size_t)u * (max_m + 1) + best_u[a]], fx);
                atomicAdd(&njoin[u], 1);
            } else {
                atomicAdd(&mass_fx[(size_t)u * (max_m + 1) + max_m], fx);
            }
        }
    }
}

// ---- 4. merge weights w_i = a_i / m_G, lost mass, status ---------------------------------
constexpr int kWeightRows = 4;     // rows per thread
__global__ void weights_kernel(const UnitDesc* __restrict__ desc, Shape sh, const float* __restrict__ s,
                               const int32_t* __restrict__ plan, const int32_t* __restrict__ grp,
                               const unsigned long long* __restrict__ mass_fx,
                               const int32_t* __restrict__ njoin, float* __restrict__ weight,
                               int32_t* __restrict__ unit_status, float* __restrict__ lost_mass, int max_m,
                               float eps, const int32_t* __restrict__ err) {
    const int u = blockIdx.y;
    const UnitDesc& ud = desc[u];
    const unsigned long long* mf = mass_fx + (size_t)u * (max_m + 1);
    const int T = ud.T;
    const int64_t o = ud.tok_off;
    // four rows per thread, a block apart (most rows belong to no group and only read their group index; a CTA
    // per 256 rows spent its time being launched)
    const int i0 = blockIdx.x * (kWeightRows * (int)blockDim.x) + threadIdx.x;
    int gidx[kWeightRows];
#pragma unroll
    for (int j = 0; j < kWeightRows; ++j) {
        const int i = i0 + j * (int)blockDim.x;
        gidx[j] = i < T ? grp[o + i] : -1;
    }
#pragma unroll
    for (int j = 0; j < kWeightRows; ++j) {
        const int i = i0 + j * (int)blockDim.x;
        if (gidx[j] >= 0 && gidx[j] < max_m) weight[o + i] = row_mass(sh, s, eps, o + i) / fx_to_mass(mf[gidx[j]]);
    }
    if (i0 == 0) {
        int fl = plan[u * 8 + CASK_PLAN_FLAGS];
        if ((fl & CASK_ST_DECODE_CONSOLIDATED) && njoin[u] == 0) fl |= CASK_ST_MERGE_INACTIVE;
        unit_status[u] = fl | *err;     // device-side flags of this call (bounded wait gave up, bad page id)
        lost_mass[u] = fx_to_mass(mf[max_m]);
    }
}

template <typename T>
cudaError_t run(const Launch& L, const cask_params& prm, const float* s, const int32_t* plan, uint8_t* kind,
                int32_t* seed_of, float* weight, float* sim, int32_t* unit_status, float* lost_mass,
                Workspace& ws, const cask_outputs* out) {
    const bool fused = out != nullptr;
    int32_t* assign = fused ? out->assign : nullptr;
    const Shape& sh = L.sh;
    const int max_m = L.max_m;
    const bool use_tc = !L.force_simt && L.tmap_encode && assign_tc_supported(L) && !sh.band_w;
    const int layout = !use_tc ? SEED_PLAIN : sh.dtype == CASK_DTYPE_FP32 ? SEED_SPLIT : sh.chan_w ? SEED_PAIR : SEED_PLAIN;
    int64_t part_rows = 256;             // rows from one part of the seed keys to the next (SEED_SPLIT)
    for (int u = 0; u < sh.n_units; ++u) part_rows += L.hdesc[u].plan[CASK_PLAN_M];
    const bool small_units = L.max_T <= kSmallUnitRows;
    cudaError_t e = cudaSuccess;
    const SeedTable<T> tab{(const T*)L.k, (T*)ws.seed_k, ws.seed_norm, layout, part_rows};
    ws.slot_lists = false;
    if (fused && !small_units) {
        ws.slot_lists = ws.filled && (use_tc || max_m == 0);
        const int words = ws.slot_lists ? (L.max_T + 31) >> 5 : 0;
        const SlotLists sl{words, out->Bmax, ws.max_B, ws.n_mem, ws.n_seed, ws.seed_slot, out->slot_src, out->slot_kind};
        const auto kern = ws.slot_lists ? (sh.n_units <= L.sms ? decide_long_kernel<1, true> : decide_long_kernel<2, true>)
                                        : (sh.n_units <= L.sms ? decide_long_kernel<1, false> : decide_long_kernel<2, false>);
        Timed t(L, KID_SEEDS);
        e = launch_dependent(L.stream, kern, sh.n_units, kSelThreads, 8 * words, L.desc, s, const_cast<int32_t*>(plan), kind,
                             seed_of, sim, ws.grp, ws.seed_rows, ws.mass_fx, ws.njoin, unit_status, max_m, assign, weight, sl);
    } else if (fused) {
        Timed t(L, KID_SEEDS);
        size_t fixed = 0;
        const int way = sh.n_units <= L.sms && L.max_T > 512 ? 2 : sh.n_units <= 3 * L.sms ? 1 : 0;      // see decide_small_kernel
        const auto kern = way == 0 ? decide_small_kernel<T, 256, 4> : way == 1 ? decide_small_kernel<T, 512, 2> : decide_small_kernel<T, 1024, 1>;
        e = allow_smem(L, kSmemBitConsolidate + 3 * (sizeof(T) == 4) + way, kern, kMaxSpread, &fixed);
        if (e == cudaSuccess)
            e = launch_dependent(L.stream, kern, sh.n_units, 256 << way, spread_smem(L, sh.n_units, fixed, 0), L.desc, sh,
                                 tab, s, const_cast<int32_t*>(plan), kind, seed_of, sim, ws.grp, ws.seed_rows, ws.mass_fx, ws.njoin,
                                 unit_status, max_m, prm.eps);
    } else {
        Timed t(L, KID_SEEDS);
        seeds_kernel<<<sh.n_units, select_threads(L.max_T), 0, L.stream>>>(L.desc, s, plan, kind, seed_of, weight, sim,
                                                               ws.grp, ws.seed_rows, ws.mass_fx, ws.njoin, max_m);
    }
    if (e != cudaSuccess) return e;
    if (max_m > 0) {
        if (!(fused && small_units)) {
            Timed t(L, KID_SEED_GATHER);
            e = launch_dependent(L.stream, seed_gather_kernel<T>, dim3((max_m + kGatherWarps - 1) / kGatherWarps, sh.n_units), 32 * kGatherWarps, 0, L.desc, sh, tab, plan, s,
                                 ws.seed_rows, ws.mass_fx, max_m, prm.eps);
            if (e != cudaSuccess) return e;
        }
        if (use_tc) {
            e = launch_assign_tc(L, prm, s, plan, kind, seed_of, sim, ws, L.tmap_encode);
            if (e != cudaSuccess) return e;
        } else if (sh.band_w) {
            const size_t smem = (size_t)2 * kTile * (sh.d / 2 + 1) * sizeof(float2) + ((size_t)2 * kTile + sh.d / 2) * sizeof(float);
            e = cudaFuncSetAttribute(assign_band_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem);
            if (e != cudaSuccess) return e;
            Timed t(L, KID_ASSIGN);
            assign_band_kernel<T><<<dim3((L.max_T + kTile - 1) / kTile, sh.n_units), kThreads, smem, L.stream>>>(
                L.desc, sh, (const T*)L.k, s, plan, ws.seed_rows, (const T*)ws.seed_k, kind, seed_of, sim, ws.grp,
                ws.mass_fx, ws.njoin, max_m, prm.tau, prm.eps);
        } else {
        const size_t smem = ((size_t)2 * kTile * (sh.d + 1) + kTile) * sizeof(float);
        e = cudaFuncSetAttribute(assign_simt_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        const int max_nd = L.max_T;   // upper bound on decode rows of any unit
        Timed t(L, KID_ASSIGN);
        assign_simt_kernel<T><<<dim3((max_nd + kTile - 1) / kTile, sh.n_units), kThreads, smem, L.stream>>>(
            L.desc, sh, (const T*)L.k, s, plan, ws.seed_rows, (const T*)ws.seed_k, ws.seed_norm, kind, seed_of,
            sim, ws.grp, ws.mass_fx, ws.njoin, max_m, prm.tau, prm.eps);
        }
    }
    if (!fused) {      // the event path leaves the weights, the status words and the lost mass to the compaction's scan
        Timed t(L, KID_WEIGHTS);
        weights_kernel<<<dim3((L.max_T + 256 * kWeightRows - 1) / (256 * kWeightRows), sh.n_units), 256, 0, L.stream>>>(
            L.desc, sh, s, plan, ws.grp, ws.mass_fx, ws.njoin, weight, unit_status, lost_mass, max_m, prm.eps, ws.err);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_consolidate(const Launch& L, const cask_params& prm, const float* s, const int32_t* plan,
                               uint8_t* kind, int32_t* seed_of, float* weight, float* sim,
                               int32_t* unit_status, float* lost_mass, Workspace& ws, const cask_outputs* out) {
    if (L.sh.dtype == CASK_DTYPE_BF16)
        return run<__nv_bfloat16>(L, prm, s, plan, kind, seed_of, weight, sim, unit_status, lost_mass, ws, out);
    return run<float>(L, prm, s, plan, kind, seed_of, weight, sim, unit_status, lost_mass, ws, out);
}

}  // namespace cask
