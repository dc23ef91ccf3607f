// Windowed attention-mass scoring on the 5th-generation tensor cores (head_dim <= 128, 32 window-query rows or more).
//
// Both passes contract window queries Q_w [<=512 rows, d] with 128-key tiles of K:
//   pass N (normaliser): D[query, key]  -> per query row a reference r and sum of 2^(y - r)
//   pass S (score mass): D[key, query]  -> per key  sum_r roww_r * 2^(y_kr - rowm_r)
// so that the reduction always runs along the TMEM columns a single thread owns.  The two
// passes use the same shared-memory operand tiles (K-major, 128-byte swizzle, written by
// TMA); only the role of the operands (A <-> B) differs.
//
// One persistent CTA per SM, 20 warps:
//   warp 0      TMA producer (one lane): Q once per segment, K tiles through a ring of 2 to 4 stages
//   warps 1-2   one lane each issues tcgen05.mma and the commits: warp 1 for the even accumulator
//               slots, warp 2 for the odd ones (pass S with four blocks: slots 0-1 and 2-3), so that one keeps the
//               tensor pipe fed while the other waits for a slot to be released (warp 1 also owns the TMEM allocation)
//   warps 4-19  epilogue: tcgen05.ld of the fp32 accumulators + the exponentials
// The 512 TMEM columns are four accumulator slots of 128 columns (one 128-row block of
// queries each).  The epilogue warps form two groups of eight (two per TMEM lane quadrant, 64
// columns each); group g drains slots g and g+2 in turn, so while it works on one of its
// slots the tensor pipe refills the other and neither side waits for the other.
//
// Slots by row count (template parameter NB, 128-row query blocks a tile is contracted with): with up to 512 rows (NB = 4)
// the four slots are the four blocks of one key tile; with up to 256 (NB = 2) they are two blocks of two consecutive
// tiles, with up to 128 (NB = 1) one block of four tiles.  Such a group of 4 / NB tiles is a "step" below: whatever the row
// count, a step fills all four slots, so both groups always have a slot to refill while they drain the other (with one
// tile a step, 256 rows left half of the TMEM unused and every group waited for its own contraction).  More than 512
// rows are cut into row groups of at most 512: the tile sequence holds every unit once per row group, the normaliser pass
// needs nothing else, and the score pass leaves one partial score per row group, added in order by score_fold.  A head_dim
// below 128 is padded with zeros by TMA (columns past the tensor's inner extent are filled), which costs tensor work only.
//
// fp32 caches (SPLIT): every fp32 number is the exact sum of three bf16 parts h + m + l (8 bits of the significand each), made
// once per event by split_rows (split.cu), and a product of two numbers is taken as the six part products lh, mh, mm, hl, hm,
// hh; the three left out are below 2^-26 of the product, a quarter of what one fp32 rounding loses.  The small ones go into the
// accumulator first, so that only the last eight additions round at full magnitude.  A tile and a query block are six 16 KB
// regions each (part, 64-channel half) and a region is refilled as soon as its last product is done.  The contraction then
// takes 48 instructions a tile, 4,100 clk at the 85 clk one takes alone, and bounds the pass, with the refill of the h
// regions behind it (16 units of 8,448 rows, 448 query rows, d = 128: 93 us a pass = 6,100 clk a tile; the SIMT kernels took
// 812 and 660; with the issuer's loop left rolled 112).  Against the same scores in 64 bits: 4.3e-7 of their norm off and 1.6e-6 in
// the worst row, where the SIMT kernels were 6.4e-7 and 4.0e-6 off.
// Measured against the SIMT kernels that served these shapes before (both passes, event on 8 units of 33,280 rows with 1,024
// query rows and given normalisers: 2.64 to 0.09 ms; 128 units of 4,608 rows, 256 query rows, head_dim 64: 1.61 to 0.11 ms).
//
// The exponentials are the bottleneck (16 ex2 per clock per SM against 65,536 per tile), so a
// fixed share of the columns is evaluated on the FMA pipe instead: round-to-nearest split
// 2^t = 2^n * 2^f, |f| <= 1/2, degree-5 minimax polynomial for 2^f (relative error 2.4e-7,
// the same order as ex2.approx).
//
// Work is split by tiles, not by units: CTA b owns the contiguous tile range
// [total*b/grid, total*(b+1)/grid) of the unit-major tile sequence and walks it segment by
// segment (a segment = its tiles inside one unit).  Pass N leaves one partial per segment
// row and column half at index 2*(unit + CTA) + half; make_row_table folds them.  Every mbarrier wait is
// bounded; when one gives up the CTA raises an error flag, drains and frees its TMEM.
#include <cmath>
#include <type_traits>

#include "tc_common.cuh"

namespace cask {

namespace {

using namespace tc;

constexpr int kTileKeys = 128;
constexpr int kMaxD = 128;
constexpr int kSlots = 4;                 // accumulator slots of 128 TMEM columns
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 4 * kSlots;
constexpr int kThreadsTc = (kEpiWarp0 + kEpiWarps) * 32;
constexpr int kIssuers = 2;               // two slots each: an epilogue group's, or (pass S, NB = 4) two neighbours
constexpr uint32_t kQBlockBytes = 128 * 128;           // one 128-row query block inside a region
constexpr uint32_t kKRegionBytes = 128 * 128;          // 128 keys x 64 bf16
constexpr uint32_t kKStageBytes = 2 * kKRegionBytes;
constexpr int kMaxSms = 1024;                          // upper bound used when sizing the partial tables

// Pairs of columns (of the 8 in a 16-column chunk of the streamed path) whose exponential runs on the FMA pipe.
// (Score pass: the last pair of a chunk.)
constexpr uint32_t kPolyPairs16N = 0x80u;

// What follows from the number of query blocks a tile is contracted with.
template <int NB, bool SPLIT = false>
struct Cfg {
    static_assert(NB == 1 || NB == 2 || NB == 4, "a step fills the four slots");
    static_assert(!SPLIT || NB == 1, "three parts of one query block fill the shared memory");
    static constexpr int kTps = kSlots / NB;                    // key tiles a step covers
    static constexpr int kStages = SPLIT ? 6 : NB == 4 ? 2 : NB == 2 ? 3 : 4;   // SPLIT: regions of one tile
    static constexpr uint32_t kKBytes = kStages * (SPLIT ? kKRegionBytes : kKStageBytes);
    static constexpr uint32_t kQRegionBytes = (NB == 1 ? 128 : 256) * 128;   // 256 (128) rows x 64 bf16
    static constexpr uint32_t kQBytes = (SPLIT ? 6 : NB == 4 ? 4 : 2) * kQRegionBytes;   // row halves x K blocks (x parts)
    static constexpr int kParts = NB == 1 ? 4 : 2;              // pass N: partials per row (column half; NB = 1: and group)
    static constexpr int kRed = NB == 4 ? 4 : 8;                // pass S: partial key sums per step and lane
    static constexpr int kRedPerTile = NB == 1 ? 2 : 4;
    // steps the partial key sums of pass S are kept; the two groups stay within two steps of one another (SPLIT: one, the
    // ring holds one tile)
    static constexpr uint32_t kRedDepth = SPLIT ? 4 : 8;
    static constexpr int kLag = NB == 4 ? 2 : 1;                // pass S: steps between a tile and the fold of its sums
};

template <int STAGES>
struct __align__(8) Barriers {
    uint64_t q_full[kSlots], q_empty[kSlots];   // one pair per 128-row block of the window queries
    uint64_t k_full[STAGES], k_empty[STAGES];
    uint64_t d_full[kSlots], d_empty[kSlots];
    uint64_t rw_full[3], rw_empty[3];   // pass S: a row table is written / the segment that used it is done
    uint64_t red_full[8];   // pass S: every warp's partial key sums of a step are in shared memory
    uint64_t mma_drain[2];  // give-up path only: an issuer's contractions in flight have completed
};

template <int NB, bool SPLIT>
struct TcSmemTail {
    Barriers<Cfg<NB, SPLIT>::kStages> bar;
    long long clk0;
    uint64_t ns0;
    uint32_t tmem_base;
    int abort;
    alignas(16) float rc[3][512];  // pass S: log2(roww) - rowm per query row, one buffer per segment in turn
    float red[Cfg<NB, SPLIT>::kRedDepth][Cfg<NB>::kRed][128];   // pass S: partial key sums per (tile of the step, group, column half)
};

template <int NB, bool SPLIT>
constexpr size_t smem_bytes() { return 1024 + Cfg<NB, SPLIT>::kQBytes + Cfg<NB, SPLIT>::kKBytes + sizeof(TcSmemTail<NB, SPLIT>); }
static_assert(smem_bytes<1, false>() <= 227 * 1024 && smem_bytes<2, false>() <= 227 * 1024 &&
              smem_bytes<4, false>() <= 227 * 1024 && smem_bytes<1, true>() <= 227 * 1024, "shared memory budget");

// The query rows of a launch: `rows` = g*W per unit, cut into `groups` row groups of `per` rows (the last may have fewer).
struct RowGroups {
    int rows, per, groups;
    __host__ __device__ int count(int rg) const { return (rg + 1) * per <= rows ? per : rows - rg * per; }
};

// 2^t for a pair of t in [-125, 125] on the FMA pipe (packed arithmetic).
__device__ __forceinline__ uint64_t ex2_poly2(uint64_t t2) {
    const uint64_t magic = pack2(12582912.f, 12582912.f);
    const uint64_t fl = add2(t2, magic);
    const uint64_t f = sub2(t2, sub2(fl, magic));
    uint64_t p = pack2(1.327644451521337e-3f, 1.327644451521337e-3f);
    p = fma2(p, f, pack2(9.67553723603487e-3f, 9.67553723603487e-3f));
    p = fma2(p, f, pack2(5.550713464617729e-2f, 5.550713464617729e-2f));
    p = fma2(p, f, pack2(2.4022120237350464e-1f, 2.4022120237350464e-1f));
    p = fma2(p, f, pack2(6.931469440460205e-1f, 6.931469440460205e-1f));
    p = fma2(p, f, pack2(1.0000001192092896f, 1.0000001192092896f));
    float p0, p1, n0, n1;
    unpack2(p, p0, p1);
    unpack2(fl, n0, n1);
    return pack2(__int_as_float(__float_as_int(p0) + (__float_as_int(n0) << 23)),
                 __int_as_float(__float_as_int(p1) + (__float_as_int(n1) << 23)));
}

// 16 bytes of the row table by a shared-space load: through a generic pointer the same read goes the way of
// global loads and comes back later (the score pass is 2.5 % faster this way).
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
    float4 r;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(a));
    return r;
}

// Sum of the n <= 4 partial key sums of one key (one per epilogue group and column half, 128 floats apart), added in
// that order; the four reads are independent shared-space loads, so the fold costs one latency and not four.
__device__ __forceinline__ float fold_partials(const float* p, int n) {
    const uint32_t a = smem_u32(p);
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[k]) : "r"(a + 512u * (uint32_t)min(k, n - 1)));
    float acc = v[0];
#pragma unroll
    for (int k = 1; k < 4; ++k)
        if (k < n) acc += v[k];
    return acc;
}

// ---- the masked form of a tile: bit x of `vis` = this thread's row sees column x of the block -------------------------------------
// One small rolled body for every tile that is not streamed (the causal diagonal, the ends of a unit, ragged columns): written out
// per block and per case it is 11 KB of instructions that each of sixteen warps fetches once a segment, and a causal tile
// took longer than a full one; leaving out blocks nobody sees in that form made it slower still, by the second case's code.
// The order of the additions is that of 32-column blocks (four sums over every fourth column, added up per block; the normaliser's
// block moves its reference to its own greatest column first and adds column by column).  It is kept because rows whose scores
// agree to 1e-7 at a selection boundary are told apart by it.  (3,072 units of 640 rows, one tile of five causal: 339 and 337 us
// a pass; with the sums of 16-column chunks, in another order, 316 and 318.)
__device__ __forceinline__ unsigned low_bits(int n) { return n >= 32 ? ~0u : n <= 0 ? 0u : (1u << n) - 1u; }

// Pass S: adds sum_r 2^(y_r*scale2 + nc[r]) over the visible rows (columns) r of a 32-column block to the packed partial sums.
__device__ __forceinline__ void mass_block(const float (&v)[32], uint32_t nc32, unsigned vis, float scale2, uint64_t& a01) {
    const uint64_t s2 = pack2(scale2, scale2);
    float b[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const float4 c4 = lds_f4(nc32 + 16u * x);
        float t0, t1, t2, t3;
        unpack2(fma2(pack2(v[4 * x], v[4 * x + 1]), s2, pack2(c4.x, c4.y)), t0, t1);
        unpack2(fma2(pack2(v[4 * x + 2], v[4 * x + 3]), s2, pack2(c4.z, c4.w)), t2, t3);
        if (vis & (1u << (4 * x))) b[0] += ex2(t0);
        if (vis & (2u << (4 * x))) b[1] += ex2(t1);
        if (vis & (4u << (4 * x))) b[2] += ex2(t2);
        if (vis & (8u << (4 * x))) b[3] += ex2(t3);
    }
    a01 = add2(a01, pack2((b[0] + b[1]) + (b[2] + b[3]), 0.f));
}

// Pass N: folds the visible columns of a 32-column block into the running (reference, sum of 2^(y*scale2 - reference)).
__device__ __forceinline__ void norm_block(const float (&v)[32], unsigned vis, float scale2, float& mref, float& lr) {
    float cm = kNegBig;
#pragma unroll
    for (int x = 0; x < 32; ++x)
        if (vis & (1u << x)) cm = fmaxf(cm, v[x]);
    cm *= scale2;
    if (vis && cm > mref) {
        lr *= ex2(mref - cm);
        mref = cm;
    }
#pragma unroll
    for (int x = 0; x < 32; ++x)
        if (vis & (1u << x)) lr += ex2(fmaf(v[x], scale2, -mref));
}

// Walks this CTA's contiguous range of key tiles, segment by segment (a segment: tiles of one row group of one unit).  The
// tile sequence is unit-major and holds a unit's tiles once per row group.  The next unit's descriptor fields are fetched
// a unit ahead, so a change of segment costs no memory round trip.
template <bool GROUPED>       // false: one row group
struct TileWalk {
    const UnitDesc* desc;
    int t, t_end, u, n_units, rg_, groups_;
    int tile0, T;
    int nx_tile0, nx_T;
    __device__ void init(const UnitDesc* d, int units, int total_tiles, int n_groups) {
        desc = d;
        n_units = units;
        groups_ = n_groups;
        t = (int)(((long long)total_tiles * blockIdx.x) / gridDim.x);
        t_end = (int)(((long long)total_tiles * (blockIdx.x + 1)) / gridDim.x);
        u = warp_find_unit(n_units, t, [&](int v) { return d[v].tile0 * groups(); });
        T = desc[u].T;
        rg_ = GROUPED ? (t - desc[u].tile0 * groups()) / n_tiles() : 0;
        tile0 = desc[u].tile0 * groups() + rg() * n_tiles();
        prefetch();
    }
    __device__ void prefetch() {
        const int v = min(u + 1, n_units - 1);
        nx_tile0 = desc[v].tile0 * groups();
        nx_T = desc[v].T;
    }
    __device__ int n_tiles() const { return (T + kTileKeys - 1) / kTileKeys; }
    __device__ int groups() const { return GROUPED ? groups_ : 1; }
    __device__ int rg() const { return GROUPED ? rg_ : 0; }        // row group of the current segment
    __device__ bool valid() const { return t < t_end; }
    __device__ int key_begin() const { return (t - tile0) * kTileKeys; }
    __device__ int seg_tiles() const { return min(t_end, tile0 + n_tiles()) - t; }
    __device__ void next_segment() {
        t += seg_tiles();
        if (t < t_end) {
            if (rg() + 1 < groups()) {
                ++rg_;
                tile0 += n_tiles();
            } else {
                rg_ = 0;
                ++u;
                tile0 = nx_tile0;
                T = nx_T;
                prefetch();
            }
        }
    }
};

// CTA that owns tile x when `total` tiles are split over `grid` CTAs as in TileWalk::init: the last b with total * b / grid <= x, that
// is with b * total < (x + 1) * grid.  (32-bit division when it fits: a 64-bit one is a sequence of a hundred instructions.)
__device__ __forceinline__ int owner_cta(int x, int total, int grid) {
    const unsigned long long n = (unsigned long long)(x + 1) * grid - 1;
    return n < (1ull << 32) ? (int)((uint32_t)n / (uint32_t)total) : (int)(n / (uint32_t)total);
}

// First normaliser partial of a row and their number, for a unit's (and row group's) tiles [tile0, tile0 + n_tiles).
__device__ __forceinline__ void partial_range(int tile0, int T, int nb, int total_tiles, int grid, int& lo, int& cnt) {
    const int parts = nb == 1 ? 4 : 2, n_tiles = (T + kTileKeys - 1) / kTileKeys;
    lo = parts * owner_cta(tile0, total_tiles, grid);
    cnt = parts * owner_cta(tile0 + n_tiles - 1, total_tiles, grid) + parts - lo;
}

// Pass S: the defaults of a segment's rows (RowDefaults), by one warp.
__device__ __noinline__ void fill_rows(const RowDefaults& f, int64_t first, int n, int lane) {
    for (int i = lane; i < n; i += 32) {
        const int64_t o = first + i;
        f.kind[o] = CASK_KIND_DROPPED;
        f.seed_of[o] = -1;
        f.assign[o] = -1;
        f.weight[o] = 0.f;
        if (f.sim) f.sim[o] = -2.f;
    }
}

// The row table of a segment of the score pass: for every query row of its unit and row group the one constant that turns a
// logit into its share of the score, roww * 2^(y - rowm) = 2^(y + rc), rc = log2(roww) - rowm.  rowm is the greatest reference of
// the row's (reference, sum) partials (one per CTA of the normaliser pass that had tiles of the unit, and column half; NB = 1:
// and group), roww = 1/(rows * sum 2^(y - rowm)), the sums added in the order of the partials.  With caller-supplied natural-log
// normalisers: rowm = lse*log2(e), roww = 1/rows.  `n` threads share the rows; `first` hands the normalisers out.  part_step: floats
// from a partial of a row to the next (rgs.per).
//
// The score pass makes its own tables when most CTAs have one segment or two (units x row groups up to the CTAs): the epilogue's
// threads the first one, the warp that has nothing else to do the later ones, ahead of time.  That saves a launch with the
// latencies in it (two fp32 units 86 to 72 us, 16 287 to 274, eight bf16 ones 63 to 60).  With more units a CTA walks many short
// segments and one warp does not keep up (3,072 units of five tiles: pass 344 to 467 us): there score_row_tables makes them
// all beforehand.
template <int kU>                            // partials in flight per row
__device__ __forceinline__ void make_row_table(int u, int rg, int lo, int cnt, bool first, const RowGroups& rgs, int nb,
                                               const float* __restrict__ part_m, const float* __restrict__ part_l,
                                               const float* __restrict__ lse_in, float* __restrict__ lse_out, float* __restrict__ rc,
                                               int limit, int idx, int n, int part_step) {
    const int rows = rgs.count(rg), parts = nb == 1 ? 4 : 2;
    const size_t ou = (size_t)u * rgs.rows + rg * rgs.per;
    const float inv_rows = 1.f / (float)rgs.rows;
    if (lse_in) {
        for (int r = idx; r < limit; r += n) {
            if (r >= rows) { rc[r] = -1.0e30f; continue; }
            const float lse = lse_in[ou + r];
            rc[r] = log2f(inv_rows) - __fmul_rn(lse, kLog2e);      // (rounded twice, as a stored rowm is)
            if (lse_out && first) lse_out[ou + r] = lse;
        }
        return;
    }
    const size_t p0 = ((size_t)parts * (u * rgs.groups + rg) + lo) * part_step;
#pragma unroll 1
    for (int r = idx; r < limit; r += n) {
        if (r >= rows) { rc[r] = -1.0e30f; continue; }
        const float *pm = part_m + p0 + r, *pl = part_l + p0 + r;
        float vm[kU], vl[kU], m = kNegBig, l = 0.f;
        auto load = [&](int b, bool sums) {
#pragma unroll
            for (int x = 0; x < kU; ++x) {
                const int at = min(b + x, cnt - 1) * part_step;
                vm[x] = pm[at];
                if (sums) vl[x] = pl[at];
            }
        };
        for (int b = 0; b < cnt; b += kU) {
            load(b, cnt <= kU);
#pragma unroll
            for (int x = 0; x < kU; ++x) m = fmaxf(m, vm[x]);
        }
        for (int b = 0; b < cnt; b += kU) {
            if (cnt > kU) load(b, true);
#pragma unroll
            for (int x = 0; x < kU; ++x)
                if (b + x < cnt) l += vl[x] * exp2f(vm[x] - m);
        }
        rc[r] = log2f(inv_rows / l) - m;
        if (lse_out && first) lse_out[ou + r] = (m + log2f(l)) * kLn2;
    }
}

// in the score pass: a call of its own (see produce_paged_call), the eight partials of units that a few CTAs shared in one go
__device__ __noinline__ void row_table(int u, int rg, int T, int tile0, bool first, const RowGroups& rgs, int nb, int total_tiles,
                                       int grid, const float* __restrict__ part_m, const float* __restrict__ part_l,
                                       const float* __restrict__ lse_in, float* __restrict__ lse_out, float* __restrict__ rc, int idx,
                                       int n, int part_step) {
    int lo = 0, cnt = 1;
    if (!lse_in) partial_range(tile0, T, nb, total_tiles, grid, lo, cnt);
    make_row_table<8>(u, rg, lo, cnt, first, rgs, nb, part_m, part_l, lse_in, lse_out, rc, 512, idx, n, part_step);
}

__device__ __forceinline__ void copy_table(const float* __restrict__ tables, int u, int rg, const RowGroups& rgs, float* rc, int idx, int n) {
    const int rows = rgs.count(rg);
    const float* src = tables + (size_t)u * rgs.rows + rg * rgs.per;
#pragma unroll 4
    for (int r = idx; r < 512; r += n) rc[r] = r < rows ? src[r] : -1.0e30f;
}

constexpr int kRowThreads = 512;
__global__ void __launch_bounds__(kRowThreads) score_row_tables(const UnitDesc* __restrict__ desc, RowGroups rgs, int nb, int total_tiles,
                                                                int grid, const float* __restrict__ part_m,
                                                                const float* __restrict__ part_l, float* __restrict__ tables,
                                                                float* __restrict__ lse_out) {
    pdl_wait();
    const int u = blockIdx.x / rgs.groups, rg = blockIdx.x - u * rgs.groups;
    const UnitDesc& ud = desc[u];
    __shared__ int range[2];                     // some divisions: one thread finds it for the block
    if (threadIdx.x == 0) {
        const int n_tiles = (ud.T + kTileKeys - 1) / kTileKeys;
        partial_range(ud.tile0 * rgs.groups + rg * n_tiles, ud.T, nb, total_tiles, grid, range[0], range[1]);
    }
    __syncthreads();
    make_row_table<4>(u, rg, range[0], range[1], true, rgs, nb, part_m, part_l, nullptr, lse_out,
                      tables + (size_t)u * rgs.rows + rg * rgs.per, rgs.count(rg), threadIdx.x, kRowThreads, rgs.per);
}

// Rows by which query block b is turned inside its 128 TMEM lanes in the normaliser pass: lane l holds row (l + turn) mod 128 of
// the block.  In a tile on the causal diagonal the early window positions see few keys and the late ones many; a lane quadrant is
// a sub-partition with its own special-function unit, and with every block laid out alike (128 window positions a block)
// the last quadrant would evaluate 88 % of a full tile's exponentials there and the first one 13 %.
template <int PASS, int NB>
__device__ __forceinline__ constexpr int block_turn(int b) { return PASS == 0 ? (128 / NB) * b % 128 : 0; }

template <int PASS, int NB>
__device__ __forceinline__ void load_query_block(const CUtensorMap* tmQ, uint64_t* bar, uint8_t* q_smem, int b, int n_kb, int row0, int u) {
    constexpr uint32_t region = Cfg<NB>::kQRegionBytes;
    uint8_t* dst = q_smem + (b >> 1) * 2 * region + (b & 1) * kQBlockBytes;
    for (int kb = 0; kb < n_kb; ++kb)
        for (int x = 0; x < 4; ++x)
            tma_load_3d(dst + kb * region + x * 4096, tmQ, bar, kb * 64, row0 + ((32 * x + block_turn<PASS, NB>(b)) & 127), u);
}

// The TMA producer of a paged cache (one warp).  A lane owns a page piece of a tile and issues its boxes.  The block table is read for as many
// tiles of a segment at once as the lanes have pieces, and one such batch ahead of its use: nothing touches a page number, not even to
// check it, before its own tiles are issued, so the table's latency hides behind the batch before.  (One lane going through the pieces took
// 5,600 clk a tile with pages of 16 rows; lanes that looked up and checked their pages a tile ahead waited for them every tile, 2,800 clk, more
// than the tiles of 256 query rows and fewer take: 216 units of 6,600 rows, 64 query rows, pages of 16, passes 119 + 118 to 94 + 97 us (76 + 70 with
// contiguous rows), event 388 to 340; with 256 query rows 466 to 410, head_dim 64 369 to 345; 512 rows even.)  The waits, and the order of copies, are those of the contiguous
// producer in score_tc_kernel.
template <int PASS, int NB, bool PLAIN>
__device__ __forceinline__ void produce_paged(const CUtensorMap* tmK, const CUtensorMap* tmQ, const Shape& sh, TileWalk<!PLAIN> wk,
                                              int per, int block_rows, int sub_rows, int n_kb, uint8_t* q_smem, uint8_t* k_smem,
                                              TcSmemTail<NB, false>* tail) {
    using C = Cfg<NB, false>;
    constexpr int kStages = C::kStages;
    auto& bar = tail->bar;
    volatile int* abort_flag = &tail->abort;
    const int lane = threadIdx.x & 31, n_blk = (per + block_rows - 1) / block_rows;
    const int piece_shift = 31 - __clz(sub_rows), tile_shift = 7 - piece_shift;      // rows of a piece, pieces of a tile
    const int my_tile = lane >> tile_shift, my_piece = lane & ((1 << tile_shift) - 1);
    uint32_t kit = 0, seg = 0;
    bool ok = true;
    TileWalk<!PLAIN> pf = wk;
    int pf_t = 0, bt0 = -1;
    struct Batch { int n, page, in_page; };
    auto next_batch = [&]() {
        Batch b{0, 0, 0};
        if (!pf.valid()) return b;
        const int left = pf.seg_tiles() - pf_t, row = pf.key_begin() + (pf_t + my_tile) * kTileKeys + my_piece * sub_rows;
        if (bt0 < 0) bt0 = pf.desc[pf.u].bt0;
        b.n = min(left, 32 >> tile_shift);
        if (my_tile < b.n && row < pf.T) {
            const int pg = row / sh.page_size;
            b.page = sh.bt[bt0 + pg];
            b.in_page = row - pg * sh.page_size;
        }
        pf_t += b.n;
        if (b.n == left) { pf.next_segment(); pf_t = 0; bt0 = -1; }
        return b;
    };
    Batch cur = next_batch(), nxt = next_batch();
    int at = 0;                                  // tile of the batch
    for (; wk.valid() && ok; wk.next_segment(), ++seg) {
        const int key_begin = wk.key_begin(), nt = wk.seg_tiles();
        for (int t = 0; t < nt && ok; ++t, ++kit) {
            const int st = kit % kStages;
            ok = mbar_wait<true>(&bar.k_empty[st], ((kit / kStages) & 1u) ^ 1u, abort_flag);
            if (!ok) break;
            uint8_t* dst = k_smem + st * kKStageBytes + my_piece * sub_rows * 128;
            // pieces past the end of the unit are not read (their accumulator rows / columns are masked by the epilogue)
            const int n_sub = min(kTileKeys >> piece_shift, (wk.T - key_begin - t * kTileKeys + sub_rows - 1) >> piece_shift);
            if (lane == 0) mbar_expect_tx(&bar.k_full[st], (uint32_t)(n_sub << piece_shift) * (128u * n_kb));
            __syncwarp();
            if (my_tile == at && my_piece < n_sub) {
                const int prow = (int)page_row(sh, cur.page, cur.in_page);
                tma_load_2d(dst, tmK, &bar.k_full[st], 0, prow);
                if (n_kb == 2) tma_load_2d(dst + kKRegionBytes, tmK, &bar.k_full[st], 64, prow);
            }
            if (++at == cur.n) {
                cur = nxt;
                nxt = next_batch();
                at = 0;
            }
            for (int j = 0; t == 0 && j < NB && ok; ++j) {
                ok = mbar_wait<true>(&bar.q_empty[j], (seg & 1u) ^ 1u, abort_flag);
                if (!ok || lane != 0) continue;
                if (j >= n_blk) { mbar_arrive(&bar.q_full[j]); continue; }
                mbar_expect_tx(&bar.q_full[j], n_kb * kQBlockBytes);
                load_query_block<PASS, NB>(tmQ, &bar.q_full[j], q_smem, j, n_kb, wk.rg() * per + j * block_rows, wk.u);
            }
        }
    }
    if (!ok && lane == 0) {
        // copies already issued may still be landing: give each armed stage a bounded wait
        for (uint32_t j = (kit >= (uint32_t)kStages ? kit - kStages : 0); j < kit; ++j)
            for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.k_full[j % kStages], (j / kStages) & 1u); ++it) {}
        for (int j = 0; j < NB; ++j)
            for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.q_full[j], seg & 1u); ++it) {}
    }
}

// The same as a call of its own, for the score pass: inlined there, its registers make the epilogue spill (contiguous caches of 448
// query rows 133 to 139 us).  The normaliser pass has room for it, and is 1 % slower with a call in it.
template <int PASS, int NB, bool PLAIN>
__device__ __noinline__ void produce_paged_call(const CUtensorMap* tmK, const CUtensorMap* tmQ, const Shape& sh, TileWalk<!PLAIN> wk,
                                                int per, int block_rows, int sub_rows, int n_kb, uint8_t* q_smem, uint8_t* k_smem,
                                                TcSmemTail<NB, false>* tail) {
    produce_paged<PASS, NB, PLAIN>(tmK, tmQ, sh, wk, per, block_rows, sub_rows, n_kb, q_smem, k_smem, tail);
}

// PASS 0: normaliser, 1: score mass; NB: 128-row query blocks per key tile; PLAIN: head_dim 113..128 and one row group, so
// that the compiler knows the numbers of 64-channel halves, contraction steps and row groups.  (The general form of the
// code costs those shapes 1 to 3 %: branches between the issuer's instructions, registers spilled in the epilogue.)
// SPLIT: fp32 caches; PLAIN is then about the head_dim only.
template <int PASS, int NB, bool PLAIN, bool SPLIT>
__global__ void __launch_bounds__(kThreadsTc, 1)
score_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ,
                const UnitDesc* __restrict__ desc, Shape sh, RowGroups rgs, float scale2, int total_tiles, int sub_rows,
                float* __restrict__ part_m, float* __restrict__ part_l, const float* __restrict__ lse_in,
                float* __restrict__ lse_out, const float* __restrict__ tables, float* __restrict__ s, int64_t s_group_stride,
                const __grid_constant__ RowDefaults fill, int ahead, const float* __restrict__ scratch, int32_t* __restrict__ err) {
    using C = Cfg<NB, SPLIT>;
    constexpr int kStages = C::kStages, kTps = C::kTps;
    constexpr int kRows = 128;                               // query rows per slot
    constexpr uint32_t kQRegionBytes = C::kQRegionBytes;
    constexpr bool kPairs = PASS == 1 && NB == 4;            // a contraction fills two neighbouring slots
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* q_smem = smem;
    uint8_t* k_smem = smem + C::kQBytes;
    using Tail = TcSmemTail<NB, SPLIT>;
    Tail* tail = reinterpret_cast<Tail*>(k_smem + C::kKBytes);
    auto& bar = tail->bar;
    volatile int* abort_flag = &tail->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_kb = PLAIN || sh.d > 64 ? 2 : 1;            // 64-channel halves of a row that hold data
    const int n_ks = PLAIN ? 8 : (sh.d + 15) >> 4;          // contraction steps of 16 channels
    auto rows_in = [&](int rg) { return PLAIN && !SPLIT ? rgs.rows : rgs.count(rg); };      // query rows of a row group

    if (threadIdx.x == 0) {
        for (int i = 0; i < kSlots; ++i) { mbar_init(&bar.q_full[i], 1); mbar_init(&bar.q_empty[i], NB == 1 ? kIssuers : 1); }
        for (int i = 0; i < kStages; ++i) { mbar_init(&bar.k_full[i], 1); mbar_init(&bar.k_empty[i], kIssuers); }
        for (int i = 0; i < kSlots; ++i) { mbar_init(&bar.d_full[i], 1); mbar_init(&bar.d_empty[i], 8); }
        // (the first table is written by the epilogue's threads, one arrival a warp; the later ones by one warp)
        for (int i = 0; i < 3; ++i) { mbar_init(&bar.rw_full[i], i == 0 ? kEpiWarps : 1); mbar_init(&bar.rw_empty[i], kEpiWarps); }
        for (int i = 0; i < 8; ++i) mbar_init(&bar.red_full[i], kEpiWarps);
        mbar_init(&bar.mma_drain[0], 1);
        mbar_init(&bar.mma_drain[1], 1);
        tail->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tail->tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tail->tmem_base;
    // Pass S started under pass N (`ahead`): keys and queries are fetched and contracted at once, and only what needs the
    // normalisers waits for the end of pass N.  What is read before that (descriptors, block table, keys, queries, the parts of fp32 rows)
    // was complete, in the memory that all SMs see, when pass N came back from its wait, and pass S is not let go before all of that
    // pass's CTAs have come back: pdl_wait() waits first and releases afterwards.  With score_row_tables between the two, pass N itself is
    // over.  Nothing changes it while pass S runs.  (The fence drops what this SM's L1 may hold of an earlier call's; reading past the
    // L1 instead costs eight units of 640 rows 0.3 us of 49.6.)
    if (PASS == 0 && ahead) asm volatile("griddepcontrol.wait;" ::: "memory");        // (`ahead` there: the next kernel starts when this one has ended)
    else if (PASS == 0 || !ahead) pdl_wait();
    else __threadfence();

    TileWalk<!PLAIN || SPLIT> wk;
    wk.init(desc, sh.n_units, total_tiles, rgs.groups);
    // CTA 0 reports the SM clock it ran at (cycles over wall time), so that a pass can be held against the
    // exponential roof at the clock the power limit left it, not only at the nominal one.  (The start values wait in
    // shared memory: in registers they would cost every warp four.)
    if (blockIdx.x == 0 && threadIdx.x == 0) { tail->clk0 = clock64(); tail->ns0 = global_ns(); }

    // Pass S: are the normalisers of the walk's unit spread over more than four CTAs (few long units)?  Then a row has many partials,
    // and one warp takes 30 to 45 us for a table that all of the epilogue's threads make in a few; such a unit is a CTA's first
    // segment or its second one, and the epilogue makes both tables before it starts.  (NB = 1: 128 rows are little for a warp
    // too.)  Event of 8 units of 8,448 rows 124 to 87 us, 12 of them with 448 query rows 122 to 98, 8 of 33,280 205 to 171.
    auto spread_unit = [&](const TileWalk<!PLAIN || SPLIT>& x) {
        return PASS == 1 && NB > 1 && !tables && !lse_in && x.valid() && (long long)x.n_tiles() * gridDim.x > 4ll * total_tiles;
    };
    if (warp == 0) {
        // ================= TMA producer =================
        bool paged = false;
        if constexpr (!SPLIT) {
            paged = sh.page_size > 0;
            if (paged && PASS == 1) produce_paged_call<PASS, NB, PLAIN>(&tmK, &tmQ, sh, wk, rgs.per, kRows, sub_rows, n_kb, q_smem, k_smem, tail);
            else if (paged) produce_paged<PASS, NB, PLAIN>(&tmK, &tmQ, sh, wk, rgs.per, kRows, sub_rows, n_kb, q_smem, k_smem, tail);
        }
        if (!paged && lane == 0) {
            uint32_t kit = 0, seg = 0;
            bool ok = true;
            for (; wk.valid() && ok; wk.next_segment(), ++seg) {
                const UnitDesc& ud = desc[wk.u];
                const int krow0 = SPLIT ? (int)ud.tok_off : (int)(ud.k_off / sh.row_stride);
                const int key_begin = wk.key_begin();
                const int nt = wk.seg_tiles();
                if constexpr (SPLIT) {
                    // parts in the order of their use, l, m, h; part p of the keys starts p * sub_rows rows down the table
                    for (int t = 0; t < nt && ok; ++t, ++kit) {
                        for (int r = 0; r < 6 && ok; ++r) {
                            if ((r & 1) >= n_kb) continue;
                            ok = mbar_wait<true>(&bar.k_empty[r], (kit & 1u) ^ 1u, abort_flag);
                            if (!ok) break;
                            mbar_expect_tx(&bar.k_full[r], kKRegionBytes);
                            tma_load_2d(k_smem + r * kKRegionBytes, &tmK, &bar.k_full[r], 64 * (r & 1),
                                        (2 - (r >> 1)) * sub_rows + krow0 + key_begin + t * kTileKeys);
                        }
                        if (t == 0 && ok) {
                            ok = mbar_wait<true>(&bar.q_empty[0], (seg & 1u) ^ 1u, abort_flag);
                            if (!ok) break;
                            mbar_expect_tx(&bar.q_full[0], 3 * n_kb * kQBlockBytes);
                            for (int r = 0; r < 6; ++r)
                                for (int x = 0; x < 4 && (r & 1) < n_kb; ++x)
                                    tma_load_3d(q_smem + r * kQRegionBytes + x * 4096, &tmQ, &bar.q_full[0], 64 * (r & 1),
                                                wk.rg() * rgs.per + 32 * x, (2 - (r >> 1)) * sh.n_units + wk.u);
                        }
                    }
                    continue;
                }
                const int n_blk = (rgs.per + kRows - 1) / kRows;
                for (int t = 0; t < nt && ok; ++t, ++kit) {
                    const int st = kit % kStages;
                    ok = mbar_wait<true>(&bar.k_empty[st], ((kit / kStages) & 1u) ^ 1u, abort_flag);
                    if (!ok) break;
                    uint8_t* dst = k_smem + st * kKStageBytes;
                    const int key0 = key_begin + t * kTileKeys;
                    mbar_expect_tx(&bar.k_full[st], n_kb * kKRegionBytes);
                    tma_load_2d(dst, &tmK, &bar.k_full[st], 0, krow0 + key0);
                    if (n_kb == 2) tma_load_2d(dst + kKRegionBytes, &tmK, &bar.k_full[st], 64, krow0 + key0);
                    if (t == 0) {
                        // The segment's query blocks, each as soon as the previous segment's last contraction
                        // with that block has completed: block 0 is back in shared memory while the tensor pipe
                        // still works on the later blocks of the previous unit.  (The first key tile of the
                        // segment went out before, so it does not wait behind them.)  Every block of the NB is
                        // armed in every segment, so that a barrier's phase is the segment's number; a block that
                        // no row group fills (NB = 4, up to 384 rows) is neither loaded nor contracted.
                        for (int j = 0; j < NB && ok; ++j) {
                            ok = mbar_wait<true>(&bar.q_empty[j], (seg & 1u) ^ 1u, abort_flag);
                            if (!ok) break;
                            if (j >= n_blk) { mbar_arrive(&bar.q_full[j]); continue; }
                            mbar_expect_tx(&bar.q_full[j], n_kb * kQBlockBytes);
                            load_query_block<PASS, NB>(&tmQ, &bar.q_full[j], q_smem, j, n_kb, wk.rg() * rgs.per + j * kRows, wk.u);
                        }
                    }
                }
            }
            if (!ok && SPLIT) {
                // copies already issued may still be landing: give each region, and the query block, a bounded wait
                for (int r = 0; r < 6; ++r)
                    for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.k_full[r], kit & 1u); ++it) {}
                for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.q_full[0], seg & 1u); ++it) {}
            } else if (!ok) {
                // copies already issued may still be landing: give each armed stage a bounded wait
                for (uint32_t j = (kit >= (uint32_t)kStages ? kit - kStages : 0); j < kit; ++j)
                    for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.k_full[j % kStages], (j / kStages) & 1u); ++it) {}
                for (int j = 0; j < NB; ++j)
                    for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.q_full[j], seg & 1u); ++it) {}
            }
        }
    } else if (warp <= kIssuers) {
        // ================= MMA issuers =================
        if (lane == 0) {
            const int j0 = warp - 1;               // this issuer's slots: j0, j0 + 2
            uint32_t kit = 0, seg = 0;
            uint32_t use[2] = {0, 0};              // contractions issued into each of them
            bool ok = true;
            // Low descriptor words of the two operand bases; every tile of both operands is reached by
            // adding a compile-time constant (the address field counts 16-byte units and cannot carry).
            const uint32_t q_lo = umma_desc_lo(smem_u32(q_smem)), k_lo = umma_desc_lo(smem_u32(k_smem));
            for (; wk.valid() && ok; wk.next_segment(), ++seg) {
                const int nt = wk.seg_tiles();
                if constexpr (SPLIT) {
                    for (int t = 0; t < nt && ok; ++t, ++kit) {
                        if (t == 0) ok = mbar_wait<true>(&bar.q_full[0], seg & 1u, abort_flag);
                        const int j = t & 3, p = j >> 1;              // the tile's slot
                        const bool mine = (j & 1) == j0;
                        if (ok && mine) {
                            ok = mbar_wait<true>(&bar.d_empty[j], (use[p] & 1u) ^ 1u, abort_flag);
                            ++use[p];
                        }
                        if (!ok) break;
                        // key parts l, m, h (regions 0-1, 2-3, 4-5); query parts in the same places
#pragma unroll
                        for (int kp = 0; kp < 3; ++kp) {
                            for (int kb = 0; kb < n_kb && ok; ++kb) ok = mbar_wait<true>(&bar.k_full[2 * kp + kb], kit & 1u, abort_flag);
                            if (!ok) break;
                            if (mine) {
                                tc_fence_after();
                                const uint32_t idesc = umma_idesc(128);
#pragma unroll
                                for (int qi = 0; qi < 3; ++qi) {
                                    // l: with h; m: with h, m; h: with l, m, h
                                    if (kp == 0 && qi != 2) continue;
                                    if (kp == 1 && qi == 0) continue;
                                    const int qp = kp == 1 ? 3 - qi : qi;
#pragma unroll
                                    for (int kk = 0; kk < 8; ++kk) {
                                        if (kk >= n_ks) break;
                                        const uint32_t at = (uint32_t)((kk >> 2) * kKRegionBytes + (kk & 3) * 32) >> 4;
                                        const uint32_t dk = k_lo + ((2 * kp * kKRegionBytes) >> 4) + at;
                                        const uint32_t dq = q_lo + ((2 * qp * kQRegionBytes) >> 4) + at;
                                        const uint32_t a = PASS == 1 ? dk : dq, b = PASS == 1 ? dq : dk;
                                        if (kp == 0 && kk == 0) tc_mma_lo<false>(tmem_base + 128 * j, a, b, idesc);
                                        else tc_mma_lo<true>(tmem_base + 128 * j, a, b, idesc);
                                    }
                                }
                            }
                            for (int kb = 0; kb < n_kb; ++kb) {
                                if (mine) tc_commit(&bar.k_empty[2 * kp + kb]);
                                else mbar_arrive(&bar.k_empty[2 * kp + kb]);
                            }
                        }
                        if (!ok) break;
                        if (mine) tc_commit(&bar.d_full[j]);
                        if (t == nt - 1) tc_commit(&bar.q_empty[0]);
                    }
                    continue;
                }
                // Pass S with four query blocks: blocks 2i and 2i + 1 lie behind one another in shared memory and their slots in TMEM, so
                // one instruction contracts the tile with both (N = 256; issuer i).  It reads the tile's operand once instead of twice:
                // 2,048 clk a tile where the 128-column form takes 2,280 (a loop of nothing but these instructions on one tile).  Score
                // pass: 3,072 units of 640 rows 340 to 315 us, 112 of 8,448 139 to 133, 288 of 33,280 1,493 to 1,479.
                if constexpr (kPairs) {
                    const int i0 = 2 * j0;                            // first of the issuer's two blocks
                    // the rows of 64-row halves in use (row_plan takes four blocks from 257 rows a group up: both issuers have some)
                    const int cols = min(256, (rgs.per - kRows * i0 + 63) & ~63);
                    const bool two = cols > kRows;
                    const uint32_t idesc = umma_idesc(cols), qblk_lo = q_lo + ((j0 * 2 * kQRegionBytes) >> 4);
                    for (int t = 0; t < nt && ok; ++t, ++kit) {
                        const int st = kit % kStages;
                        ok = mbar_wait<true>(&bar.k_full[st], (kit / kStages) & 1u, abort_flag);
                        if (!ok) break;
                        if (t == 0) {
                            ok = mbar_wait<true>(&bar.q_full[i0], seg & 1u, abort_flag);
                            if (ok) ok = mbar_wait<true>(&bar.q_full[i0 + 1], seg & 1u, abort_flag);
                            if (!ok) break;
                        }
                        ok = mbar_wait<true>(&bar.d_empty[i0], (use[0] & 1u) ^ 1u, abort_flag);
                        if (ok && two) ok = mbar_wait<true>(&bar.d_empty[i0 + 1], (use[0] & 1u) ^ 1u, abort_flag);
                        if (!ok) break;
                        ++use[0];
                        tc_fence_after();
                        const uint32_t kst_lo = k_lo + st * (kKStageBytes >> 4);
                        tc_mma_lo<false>(tmem_base + 128 * i0, kst_lo, qblk_lo, idesc);
#pragma unroll
                        for (int kk = 1; kk < 8; ++kk) {
                            const int kb = kk >> 2, ks = kk & 3;
                            if (kk >= n_ks) break;
                            tc_mma_lo<true>(tmem_base + 128 * i0, kst_lo + ((kb * kKRegionBytes + ks * 32) >> 4),
                                            qblk_lo + ((kb * kQRegionBytes + ks * 32) >> 4), idesc);
                        }
                        tc_commit(&bar.d_full[i0]);
                        if (two) tc_commit(&bar.d_full[i0 + 1]);
                        tc_commit(&bar.k_empty[st]);
                        if (t == nt - 1) {
                            // last use of the segment's query blocks
                            tc_commit(&bar.q_empty[i0]);
                            tc_commit(&bar.q_empty[i0 + 1]);
                        }
                    }
                    continue;
                }
                // A parity wait is only sound for a waiter that has met every phase before: each issuer waits for every
                // key tile and every query block of its own, whether it has a contraction with them or not.
                for (int t = 0; t < nt && ok; ++t, ++kit) {
                    const int st = kit % kStages;
                    ok = mbar_wait<true>(&bar.k_full[st], (kit / kStages) & 1u, abort_flag);
                    if (!ok) break;
                    const uint32_t kst_lo = k_lo + st * (kKStageBytes >> 4);
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        const int j = j0 + 2 * p, b = j % NB;
                        if (!ok) break;
                        if (t == 0 && (NB == 4 || p == 0)) {          // the segment's query block b has landed
                            ok = mbar_wait<true>(&bar.q_full[b], seg & 1u, abort_flag);
                            if (!ok) break;
                        }
                        if (NB < 4 && t % kTps != j / NB) continue;    // slot j belongs to another tile of the step
                        if (kRows * b >= rgs.per) {                   // no rows in this block
                            if (NB == 4 && t == nt - 1) mbar_arrive(&bar.q_empty[b]);
                            continue;
                        }
                        ok = mbar_wait<true>(&bar.d_empty[j], (use[p] & 1u) ^ 1u, abort_flag);
                        if (!ok) break;
                        ++use[p];
                        tc_fence_after();
                        const uint32_t qblk_lo = q_lo + (((b >> 1) * 2 * kQRegionBytes + (b & 1) * (128 * 128)) >> 4);
                        // (a row past the group's own is one of the next group or a zero, and has no weight; pass S reads no
                        // more than the first half of a block with 64 rows or fewer)
                        const uint32_t idesc = umma_idesc(PASS == 1 && rgs.per - kRows * b <= 64 ? 64 : 128);
                        if (PASS == 1) tc_mma_lo<false>(tmem_base + 128 * j, kst_lo, qblk_lo, idesc);
                        else tc_mma_lo<false>(tmem_base + 128 * j, qblk_lo, kst_lo, idesc);
#pragma unroll
                        for (int kk = 1; kk < 8; ++kk) {
                            const int kb = kk >> 2, ks = kk & 3;
                            if (kk >= n_ks) break;
                            const uint32_t dq = qblk_lo + ((kb * kQRegionBytes + ks * 32) >> 4);
                            const uint32_t dk = kst_lo + ((kb * kKRegionBytes + ks * 32) >> 4);
                            if (PASS == 1) tc_mma_lo<true>(tmem_base + 128 * j, dk, dq, idesc);
                            else tc_mma_lo<true>(tmem_base + 128 * j, dq, dk, idesc);
                        }
                        tc_commit(&bar.d_full[j]);
                        if (NB == 4 && t == nt - 1) tc_commit(&bar.q_empty[b]);      // last use of query block b in this segment
                    }
                    tc_commit(&bar.k_empty[st]);
                    if (NB < 4 && t == nt - 1) tc_commit(&bar.q_empty[j0 % NB]);
                }
            }
            if (!ok) {
                // contractions already issued may still be running: the TMEM they write is freed below, so give them
                // a bounded wait (a commit completes when everything this thread issued before it has)
                tc_commit(&bar.mma_drain[j0]);
                for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.mma_drain[j0], 0u); ++it) {}
            }
        }
    } else if (warp == 3) {
        // ================= pass S: row tables of the later segments, up to two segments ahead; row defaults =================
        if (PASS == 1 && ahead) pdl_wait();
        if (PASS == 1 && wk.valid()) {
            bool ok = true;
            auto fill_segment = [&](const TileWalk<!PLAIN || SPLIT>& f) {
                if (!fill.kind || f.rg() > 0) return;
                fill_rows(fill, desc[f.u].tok_off + f.key_begin(), min(f.seg_tiles() * kTileKeys, f.T - f.key_begin()), lane);
            };
            TileWalk<!PLAIN || SPLIT> before = wk;
            wk.next_segment();
            for (uint32_t seg = 1; wk.valid() && ok; wk.next_segment(), ++seg) {
                const uint32_t buf = seg % 3u;
                ok = mbar_wait<true>(&bar.rw_empty[buf], ((seg / 3u) & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                if (seg > 1 || !spread_unit(wk)) {
                    if (tables) copy_table(tables, wk.u, wk.rg(), rgs, tail->rc[buf], lane, 32);
                    else
                        row_table(wk.u, wk.rg(), wk.T, wk.tile0, wk.t == wk.tile0, rgs, NB, total_tiles, gridDim.x, part_m, part_l, lse_in,
                                  lse_out, tail->rc[buf], lane, 32, rgs.per);
                    __syncwarp();
                    // table 0's barrier counts the epilogue's warps: stand in for them
                    if (lane < (buf == 0 ? kEpiWarps : 1)) mbar_arrive(&bar.rw_full[buf]);
                }
                fill_segment(before);
                before = wk;
            }
            if (ok) fill_segment(before);
        }
    } else if (warp >= kEpiWarp0) {
        // ================= epilogue =================
        const int ew = warp - kEpiWarp0;
        const int qd = ew & 3;                   // TMEM lane quadrant (== warp % 4)
        const int ch = (ew >> 2) & 1;            // which 64 columns of a slot
        const int g = ew >> 3;                   // group: drains slots g and g + 2 in turn
        const int etid = ew * 32 + lane;
        const uint32_t taddr = tmem_base + ((uint32_t)(32 * qd) << 16) + 64 * ch;
        constexpr int kStates = NB == 4 ? 2 : 1;
        const int j0 = g, j1 = g + 2;            // this group's slots
        const int b0 = j0 % NB, b1 = j1 % NB;    // the query blocks in them
        const int to0 = j0 / NB, to1 = j1 / NB;  // the tiles of a step they hold
        uint32_t sit = 0, seg = 0;               // steps and segments so far
        uint32_t use[2] = {0, 0};                // uses so far of the two slots (NB = 4: a slot in use is used in every step)
        auto uses = [&](int p) { return NB == 4 ? sit : use[p]; };
        bool ok = true;
        // pass S: where the folded key sums of the last steps go (-1: nowhere); the fold runs kLag steps late.  One tile of
        // a step per folding warp: NB = 4 the warps ew < 4, NB = 2 those with ch = 0, NB = 1 all.
        const bool folds = NB == 4 ? ew < 4 : NB == 2 ? ch == 0 : true;
        const int fold_to = NB == 4 ? 0 : NB == 2 ? g : 2 * ch + g;
        int32_t pend_off[C::kLag];              // the oldest last
#pragma unroll
        for (int i = 0; i < C::kLag; ++i) pend_off[i] = -1;
        // pass N: running reference / sum of the query rows this thread works on
        float mm[kStates], l_run[kStates];
#pragma unroll
        for (int i = 0; i < kStates; ++i) { mm[i] = kNegBig; l_run[i] = 0.f; }

        if (PASS == 1 && ahead) {
            // The code of the row tables once through on nothing while pass N still runs: fetching its instructions is most of what
            // the first table costs (one partial address for all, out of `scratch`, into the room of the key sums).  A unit of one tile
            // (the 1): one round over the partials, whatever the segment's own unit has.  The rounds of a unit that many CTAs share go on
            // when pass N, short there, is long over: event of four units of 9,000 rows 79.4 us with them, 72.5 without.  (ahead > 1: pass N
            // leaves SMs free.  Else this CTA began when pass N's had left its SM, and there is little to wait for: those four units 71.2
            // to 69.7, with head_dim 64 74.0 to 72.2, eight of 9,000 82.1 to 81.0; 112 of 8,448 even.)
            if (!tables && wk.valid() && ahead > 1)
                row_table(wk.u, 0, 1, wk.tile0, false, rgs, NB, total_tiles, gridDim.x, scratch, scratch, nullptr, nullptr,
                          &tail->red[0][0][0], etid, 32 * kEpiWarps, 0);
            pdl_wait();
        }
        if (PASS == 1 && wk.valid()) {
            if (tables) copy_table(tables, wk.u, wk.rg(), rgs, tail->rc[0], etid, 32 * kEpiWarps);
            else
                row_table(wk.u, wk.rg(), wk.T, wk.tile0, wk.t == wk.tile0, rgs, NB, total_tiles, gridDim.x, part_m, part_l, lse_in, lse_out,
                          tail->rc[0], etid, 32 * kEpiWarps, rgs.per);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar.rw_full[0]);
            TileWalk<!PLAIN || SPLIT> nx = wk;
            nx.next_segment();
            if (spread_unit(nx)) {                       // the second table as well: see there
                row_table(nx.u, nx.rg(), nx.T, nx.tile0, nx.t == nx.tile0, rgs, NB, total_tiles, gridDim.x, part_m, part_l, lse_in, lse_out,
                          tail->rc[1], etid, 32 * kEpiWarps, rgs.per);
                asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
                if (etid == 0) mbar_arrive(&bar.rw_full[1]);
            }
        }
        for (; wk.valid() && ok; wk.next_segment(), ++seg) {
            const int T = wk.T;
            const int rows_g = rows_in(wk.rg()), rg0 = wk.rg() * rgs.per;
            // pass S: place of the first score of the segment's unit and row group (score_tc_supported: it fits 32 bits)
            const int32_t s_off = (int32_t)(wk.rg() * s_group_stride + desc[wk.u].tok_off);
            const int last_all = sh.causal ? T - sh.W : T - 1;     // last key every query sees
            const float* rc = tail->rc[seg % 3u];
            if (PASS == 1) {
                ok = mbar_wait<true>(&bar.rw_full[seg % 3u], (seg / 3u) & 1u, abort_flag);
                if (!ok) break;
            } else {
#pragma unroll
                for (int i = 0; i < kStates; ++i) { mm[i] = kNegBig; l_run[i] = 0.f; }
            }
            const int key_begin = wk.key_begin();
            const int nt = wk.seg_tiles();
            // The columns of its two slots this warp reads: half of each.  (Pass S: a ragged last block has fewer; a
            // half-filled 64 goes the streamed way whole, its spare columns hold other rows or zeros, without weight.)
            const int cend0 = PASS == 1 ? min(64, rgs.per - 128 * b0 - 64 * ch) : 64;
            const int cend1 = PASS == 1 ? min(64, rgs.per - 128 * b1 - 64 * ch) : 64;
            const bool full_cols = NB == 4 || (128 * b0 < rgs.per && (PASS == 0 || cend0 > 32));
            // NB = 4: does this warp read the group's second slot?  Up to 384 rows leave the fourth slot unused, up to 448 its second
            // half, and pass S then evaluates no exponential of it.  (448 rows spread over the four slots, 112 in each, keep the
            // two groups equally busy, 112 units of 13,312 rows 194 against 197 us, but add a key's terms in another order.)
            const bool slot1 = NB < 4 || 128 * b1 < rgs.per, second = slot1 && (NB < 4 || cend1 > 0);
            const int row0 = 128 * b0 + ((32 * qd + block_turn<PASS, NB>(b0)) & 127) + lane;   // pass N, in the row group
            const int row1 = 128 * b1 + ((32 * qd + block_turn<PASS, NB>(b1)) & 127) + lane;
            const int lastvis0 = (row0 < rows_g) ? (sh.causal ? T - sh.W + ((rg0 + row0) % sh.W) : T - 1) : -1;
            const int lastvis1 = (row1 < rows_g) ? (sh.causal ? T - sh.W + ((rg0 + row1) % sh.W) : T - 1) : -1;
            if (PASS == 0 && full_cols && to0 < nt && key_begin + (to0 + 1) * kTileKeys - 1 <= last_all) {
                // The rows have no reference at the start of a segment, and a streamed tile without one is redone
                // whole.  Once per segment, before its first step: wait for the step's slots (the waits inside
                // the loop then pass at once), read the first chunk of each and take its maximum as the reference.
                float w[16];
#pragma unroll
                for (int p = 0; p < kStates; ++p) {
                    const int j = p ? j1 : j0;
                    if (p == 1 && !second) break;
                    ok = mbar_wait<true>(&bar.d_full[j], uses(p) & 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    tc_ld16(taddr + 128 * j, w);
                    tc_wait_ld_regs(w);
                    float cm = w[0];
#pragma unroll
                    for (int x = 1; x < 16; ++x) cm = fmaxf(cm, w[x]);
                    mm[p] = cm * scale2;
                }
                if (!ok) break;
            }
            for (int t0 = 0; t0 < nt && ok; t0 += kTps, ++sit) {
                const int key0 = key_begin + t0 * kTileKeys;           // first key of the step
                // every tile of the step is there and every query sees all of it
                const bool fast = t0 + kTps <= nt && key0 + kTps * kTileKeys - 1 <= last_all;
                // pass S: packed pairs of partial key sums; NB = 4: of the step's one tile, else one set per slot
                uint64_t a01[3 - kStates], a23[3 - kStates];
#pragma unroll
                for (int i = 0; i < 3 - kStates; ++i) { a01[i] = 0ull; a23[i] = 0ull; }
                if (fast && full_cols) {
                    // Streamed form of the common step: eight chunks of 16 columns.  The arguments of a chunk's
                    // exponentials are formed first; that frees the accumulator registers, so the next chunk's
                    // TMEM load (or the slot's release) is issued before the exponentials and its latency hides
                    // behind them.
                    const uint64_t s2 = pack2(scale2, scale2);
                    float v[16];
                    float lbs[4] = {0.f, 0.f, 0.f, 0.f};      // pass N: the sums of a slot's four chunks
                    ok = mbar_wait<true>(&bar.d_full[j0], uses(0) & 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    tc_ld16(taddr + 128 * j0, v);
                    tc_wait_ld_regs(v);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const int p = c >> 2, j = p ? j1 : j0, col = 16 * (c & 3);
                        const int ps = NB == 4 ? p : 0;          // pass N: the row state of the slot
                        const int pa = NB == 4 ? 0 : p;          // pass S: the key sums of the slot
                        uint64_t t2[8];
                        if (PASS == 1) {
                            const uint32_t nc32 = smem_u32(&rc[kRows * (p ? b1 : b0) + 64 * ch + col]);
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                const float4 c4 = lds_f4(nc32 + 16u * x);
                                t2[2 * x] = fma2(pack2(v[4 * x], v[4 * x + 1]), s2, pack2(c4.x, c4.y));
                                t2[2 * x + 1] = fma2(pack2(v[4 * x + 2], v[4 * x + 3]), s2, pack2(c4.z, c4.w));
                            }
                        } else {
                            const uint64_t nm2 = pack2(-mm[ps], -mm[ps]);
#pragma unroll
                            for (int x = 0; x < 8; ++x) t2[x] = fma2(pack2(v[2 * x], v[2 * x + 1]), s2, nm2);
                        }
                        if (PASS == 1 && (c == 3 || c == 7)) {           // the slot's last columns are in registers
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&bar.d_empty[j]);
                        }
                        if (c == 3 && second) {
                            ok = mbar_wait<true>(&bar.d_full[j1], uses(1) & 1u, abort_flag);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        if (c < 7 && (c != 3 || second)) tc_ld16(taddr + 128 * (((c + 1) >> 2) ? j1 : j0) + 16 * ((c + 1) & 3), v);
                        if (PASS == 1) {
#pragma unroll
                            for (int x = 0; x < 8; ++x) {
                                float t0_, t1_;
                                unpack2(t2[x], t0_, t1_);
                                const uint64_t e2 = x == 7
                                                        ? ex2_poly2(pack2(fmaxf(t0_, -125.f), fmaxf(t1_, -125.f)))
                                                        : pack2(ex2(t0_), ex2(t1_));
                                if (x & 1) a23[pa] = add2(a23[pa], e2); else a01[pa] = add2(a01[pa], e2);
                            }
                        } else {
                            uint64_t b01 = 0ull, b23 = 0ull;
#pragma unroll
                            for (int x = 0; x < 8; ++x) {
                                float t0_, t1_;
                                unpack2(t2[x], t0_, t1_);
                                const uint64_t e2 = ((kPolyPairs16N >> x) & 1u)
                                                        ? ex2_poly2(pack2(fminf(fmaxf(t0_, -125.f), 125.f), fminf(fmaxf(t1_, -125.f), 125.f)))
                                                        : pack2(ex2(t0_), ex2(t1_));
                                if (x & 1) b23 = add2(b23, e2); else b01 = add2(b01, e2);
                            }
                            float s0, s1;
                            unpack2(add2(b01, b23), s0, s1);
                            lbs[c & 3] = s0 + s1;
                            if (c == 3 || c == 7) {
                                // The four chunk sums of the slot are checked together, once, before the slot is
                                // released: a check per chunk drains the warp's exponentials eight times a step.
                                const bool redo = !(lbs[0] <= 65536.f) || !(lbs[1] <= 65536.f) || !(lbs[2] <= 65536.f) ||
                                                  !(lbs[3] <= 65536.f);
                                if (__any_sync(0xffffffffu, redo)) {
                                    // Some row of the warp has a column that exceeds its reference by more than 16
                                    // (or its reference is still unset).  The whole warp reads the slot's 64 columns
                                    // again (the loads are warp-wide; the slot is still held); the rows concerned
                                    // move their reference to the maximum of the 64 and redo the four sums.
                                    float w[16];
                                    float cm = kNegBig;
#pragma unroll
                                    for (int k = 0; k < 4; ++k) {
                                        tc_ld16(taddr + 128 * j + 16 * k, w);
                                        tc_wait_ld_regs(w);
#pragma unroll
                                        for (int x = 0; x < 16; ++x) cm = fmaxf(cm, w[x]);
                                    }
                                    cm *= scale2;
                                    if (redo && cm > mm[ps]) {
                                        l_run[ps] *= ex2(mm[ps] - cm);
                                        mm[ps] = cm;
                                    }
#pragma unroll
                                    for (int k = 0; k < 4; ++k) {
                                        tc_ld16(taddr + 128 * j + 16 * k, w);
                                        tc_wait_ld_regs(w);
                                        if (redo) {
                                            float lb = 0.f;
#pragma unroll
                                            for (int x = 0; x < 16; ++x) lb += ex2(fmaf(w[x], scale2, -mm[ps]));
                                            lbs[k] = lb;
                                        }
                                    }
                                    __syncwarp();
                                }
#pragma unroll
                                for (int k = 0; k < 4; ++k) l_run[ps] += lbs[k];
                                // the slot is no longer needed
                                tc_fence_before();
                                __syncwarp();
                                if (lane == 0) mbar_arrive(&bar.d_empty[j]);
                            }
                        }
                        if (c == 3 && !second) break;
                        if (c < 7) tc_wait_ld_regs(v);
                    }
                    if (!ok) break;
                    if (PASS == 1 && NB == 4 && slot1 && !second) {       // the slot is the other column half's alone
                        ok = mbar_wait<true>(&bar.d_full[j1], uses(1) & 1u, abort_flag);
                        if (!ok) break;
                        if (lane == 0) mbar_arrive(&bar.d_empty[j1]);
                    }
                    ++use[0];
                    ++use[1];
                } else {
#pragma unroll 1
                    for (int p = 0; p < 2; ++p) {
                        const int j = p ? j1 : j0;
                        if (kRows * (p ? b1 : b0) >= rgs.per || t0 + (p ? to1 : to0) >= nt) break;     // slot j is not used
                        ok = mbar_wait<true>(&bar.d_full[j], (NB == 4 ? sit : p ? use[1] : use[0]) & 1u, abort_flag);
                        if (!ok) break;
                        if (p) ++use[1]; else ++use[0];
                        tc_fence_after();
                        const int ktile = key0 + (NB == 4 ? 0 : (p ? to1 : to0)) * kTileKeys;     // first key of the slot's tile
                        const bool tfast = ktile + kTileKeys - 1 <= last_all;
                        const int cend = p ? cend1 : cend0;
                        const int jmin = ktile + 32 * qd + lane - (T - sh.W);     // pass S: first window position that sees the thread's key
                        const int nvis = (p ? lastvis1 : lastvis0) - (ktile + 64 * ch) + 1;   // pass N: columns of this warp the row sees
                        float mref = NB == 4 && p ? mm[kStates - 1] : mm[0], lr = NB == 4 && p ? l_run[kStates - 1] : l_run[0];
                        uint64_t s01 = NB == 4 ? a01[0] : 0ull;
#pragma unroll 1
                        for (int cc = 0; cc < cend; cc += 32) {           // (cend is a multiple of 32)
                            const int r0 = kRows * (p ? b1 : b0) + 64 * ch + cc;              // pass S: first query row of the block
                            unsigned vis = ~0u;
                            if (PASS == 0) {
                                vis = low_bits(nvis - cc);
                            } else if (!tfast && sh.causal) {
                                // window position of the first column, and columns up to the next head's first
                                int pos = (rg0 + r0) % sh.W;
                                if ((sh.W & 15) == 0) {                   // each half of the block lies inside one head
                                    const int pos1 = pos + 16 == sh.W ? 0 : pos + 16;
                                    vis = (~low_bits(jmin - pos) & 0xFFFFu) | (~low_bits(jmin - pos1) << 16);
                                } else {
                                    vis = 0u;
                                    for (int x = 0; x < 32; ++x) {
                                        vis |= (pos >= jmin ? 1u : 0u) << x;
                                        if (++pos == sh.W) pos = 0;
                                    }
                                }
                            }
                            if (!__any_sync(0xffffffffu, vis)) continue;                      // nothing in the warp sees the block
                            float v[32];
                            tc_ld32(taddr + 128 * j + cc, v);
                            tc_wait_ld_regs(v);
                            if (PASS == 1) mass_block(v, smem_u32(&rc[r0]), vis, scale2, s01);
                            else norm_block(v, vis, scale2, mref, lr);
                        }
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bar.d_empty[j]);
                        if (PASS == 1) {
                            if (NB == 4 || p == 0) a01[0] = s01;
                            else a01[2 - kStates] = s01;
                        } else if (NB == 4 && p) {
                            mm[kStates - 1] = mref; l_run[kStates - 1] = lr;
                        } else {
                            mm[0] = mref; l_run[0] = lr;
                        }
                    }
                    if (!ok) break;
                }
                if (PASS == 1 && ok) {
#pragma unroll
                    for (int i = 0; i < 3 - kStates; ++i) {
                        float x0, x1, x2, x3;
                        unpack2(a01[i], x0, x1);
                        unpack2(a23[i], x2, x3);
                        // the tile the sums belong to and this warp's place among its partials
                        const int tile = NB == 4 ? 0 : (i ? to1 : to0);
                        tail->red[sit % C::kRedDepth][tile * C::kRedPerTile + (NB == 1 ? ch : ew >> 2)][32 * qd + lane] = (x0 + x1) + (x2 + x3);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.red_full[sit % C::kRedDepth]);
                    if (folds) {
                        // Fold the sums of kLag steps ago: every warp finished that step long ago.  The key ring keeps the
                        // two groups within two steps of one another, so the buffer read here cannot be the one being
                        // rewritten.
                        const int32_t off = pend_off[C::kLag - 1];
                        if (sit >= (uint32_t)C::kLag) {
                            const uint32_t pk = sit - C::kLag;
                            ok = mbar_wait<true>(&bar.red_full[pk % C::kRedDepth], (pk / C::kRedDepth) & 1u, abort_flag);
                            if (!ok) break;
                            const float acc = fold_partials(&tail->red[pk % C::kRedDepth][fold_to * C::kRedPerTile][32 * qd + lane], C::kRedPerTile);
                            if (off >= 0) s[off] = acc;
                        }
                        const int my_key = key0 + fold_to * kTileKeys + 32 * qd + lane;
                        if (C::kLag == 2) pend_off[C::kLag - 1] = pend_off[0];
                        pend_off[0] = (t0 + fold_to < nt && my_key < T) ? s_off + my_key : -1;
                    }
                }
            }
            if (PASS == 1 && ok) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar.rw_empty[seg % 3u]);
            }
            if (PASS == 0 && ok) {
#pragma unroll
                for (int i = 0; i < kStates; ++i) {
                    const int my_row = i ? row1 : row0;
                    if (my_row < rows_g) {
                        const size_t o = ((size_t)(wk.u * rgs.groups + wk.rg() + blockIdx.x) * C::kParts + (NB == 1 ? 2 * g : 0) + ch) *
                                             rgs.per + my_row;
                        part_m[o] = mm[i];
                        part_l[o] = l_run[i];
                    }
                }
            }
        }
        if (PASS == 1 && folds && ok) {
            // the last steps of this CTA
            for (uint32_t pk = (sit >= (uint32_t)C::kLag ? sit - C::kLag : 0); pk < sit; ++pk) {
                if (!mbar_wait<true>(&bar.red_full[pk % C::kRedDepth], (pk / C::kRedDepth) & 1u, abort_flag)) break;
                const float acc = fold_partials(&tail->red[pk % C::kRedDepth][fold_to * C::kRedPerTile][32 * qd + lane], C::kRedPerTile);
                const int32_t off = pend_off[pk + 1 == sit ? 0 : C::kLag - 1];
                if (off >= 0) s[off] = acc;
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && tail->abort) atomicOr(err, CASK_ST_TIMEOUT);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint64_t ns = global_ns() - tail->ns0;
        const long long clk = clock64() - tail->clk0;
        err[2 + PASS] = ns > 0 ? (int32_t)((double)clk * 1.0e6 / (double)ns) : 0;      // kHz
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// More than one row group: the score of a key is the sum of its row groups' partial scores, in order.
constexpr int kFoldThreads = 256, kFoldKeys = 4;
__global__ void __launch_bounds__(kFoldThreads) score_fold(const UnitDesc* __restrict__ desc, int groups, int64_t group_stride,
                                                           const float* __restrict__ part, float* __restrict__ s) {
    pdl_wait();
    const UnitDesc& ud = desc[blockIdx.y];
    const int T = ud.T;
    const int64_t o = ud.tok_off;
    const int i0 = blockIdx.x * (kFoldThreads * kFoldKeys) + threadIdx.x;
    float acc[kFoldKeys];
#pragma unroll
    for (int x = 0; x < kFoldKeys; ++x) acc[x] = 0.f;
    for (int g = 0; g < groups; ++g)
#pragma unroll
        for (int x = 0; x < kFoldKeys; ++x) {
            const int i = i0 + x * kFoldThreads;
            if (i < T) acc[x] += part[g * group_stride + o + i];
        }
#pragma unroll
    for (int x = 0; x < kFoldKeys; ++x) {
        const int i = i0 + x * kFoldThreads;
        if (i < T) s[o + i] = acc[x];
    }
}

// How the query rows of a unit are served: row groups and query blocks per tile.  A tile costs NB * 1024 clk of the
// exponential pipe, and at least some 1,600 clk of the key stream (32 KB): the cheapest division wins, the one with the
// fewest groups among equals.
struct RowPlan {
    RowGroups rg;
    int nb;
};
constexpr int kMaxRowGroups = 8;
RowPlan row_plan(int rows, int dtype) {
    if (dtype == CASK_DTYPE_FP32) {       // three parts: one block a tile
        const int groups = (rows + 127) / 128;
        const int per = ((rows + groups - 1) / groups + 31) & ~31;
        return RowPlan{RowGroups{rows, per, (rows + per - 1) / per}, 1};
    }
    const int nbs[3] = {4, 2, 1}, cost[3] = {4096, 2048, 1600};
    RowPlan best{};
    int best_cost = 0;
    for (int i = 0; i < 3; ++i) {
        const int groups = (rows + 128 * nbs[i] - 1) / (128 * nbs[i]);
        if (best.nb && groups * cost[i] >= best_cost) continue;
        best_cost = groups * cost[i];
        const int per = ((rows + groups - 1) / groups + 31) & ~31;
        best.nb = nbs[i];
        best.rg = RowGroups{rows, per, (rows + per - 1) / per};
    }
    return best;
}

// The shapes these kernels take (the addresses of a batch are checked in score_tc_supported).
bool shape_fits(int dtype, int d, int rows) {
    return d <= kMaxD && rows >= 32 && row_plan(rows, dtype).rg.groups <= kMaxRowGroups;
}

}  // namespace

// Workspace of the tensor-core path: floats per normaliser-partial table, and partial scores per cache row.
ScoreTcSizes score_tc_sizes(int dtype, int d, int rows, int n_units) {
    if (!shape_fits(dtype, d, rows)) return ScoreTcSizes{0, 0};
    const RowPlan pl = row_plan(rows, dtype);
    const size_t parts = pl.nb == 1 ? Cfg<1>::kParts : Cfg<4>::kParts;
    return ScoreTcSizes{parts * ((size_t)n_units * pl.rg.groups + kMaxSms) * pl.rg.per,
                        pl.rg.groups > 1 ? (size_t)pl.rg.groups : 0};
}

constexpr int kGivenLong = 24;        // tiles a CTA
bool given_score_long(int dtype, int d, int rows, int total_tiles, int sms) {
    return shape_fits(dtype, d, rows) && (int64_t)total_tiles * row_plan(rows, dtype).rg.groups >= (int64_t)kGivenLong * (sms > 0 ? sms : 128);
}

// Rows per TMA box of the key stream: a whole 128-key tile for a contiguous cache, one page piece for
// a paged one (0: the page size does not tile 128 rows).
static int key_box_rows(const Shape& sh) {
    if (sh.page_size == 0) return kTileKeys;
    if (sh.page_size % kTileKeys == 0) return kTileKeys;
    if (sh.page_size >= 8 && kTileKeys % sh.page_size == 0) return sh.page_size;
    return 0;
}

bool score_tc_supported(const Launch& L) {
    const Shape& sh = L.sh;
    if (!shape_fits(sh.dtype, sh.d, sh.rows)) return false;
    const int64_t groups = row_plan(sh.rows, sh.dtype).rg.groups;
    if (L.total_tiles * groups >= (int64_t)1 << 31 || L.sum_T * groups >= (int64_t)1 << 31) return false;
    if (sh.dtype == CASK_DTYPE_FP32) return 3 * L.sum_T < (int64_t)1 << 31;      // the split table is dense
    if (sh.page_size) return key_box_rows(sh) != 0 && sh.n_pages * sh.page_size < ((int64_t)1 << 31);
    int64_t max_row = 0;
    for (int u = 0; u < sh.n_units; ++u) {
        const UnitDesc& d = L.hdesc[u];
        if (d.k_off % sh.row_stride != 0) return false;
        max_row = std::max<int64_t>(max_row, d.k_off / sh.row_stride + d.T);
    }
    return max_row < (int64_t)1 << 31;
}

namespace {
template <int NB, bool PLAIN, bool SPLIT>
cudaError_t launch_passes(const Launch& L, const RowGroups& rg, const CUtensorMap& tmK, const CUtensorMap& tmQ, int sub_rows,
                          const float* lse_in, float* s, float* lse_out, Workspace& ws) {
    const Shape& sh = L.sh;
    const int total = L.total_tiles * rg.groups;
    const int grid = std::max(1, std::min(std::min(L.sms > 0 ? L.sms : 128, kMaxSms), total));
    constexpr size_t smem = smem_bytes<NB, SPLIT>();
    const float scale2 = kLog2e * (float)(1.0 / std::sqrt((double)sh.d));      // logits in log2 units
    const auto norm = score_tc_kernel<0, NB, PLAIN, SPLIT>, mass = score_tc_kernel<1, NB, PLAIN, SPLIT>;
    // Whether a pass may start while the kernel before it still runs (launch_dependent).  Its warps then take the slots that kernel's
    // leave, and where those are not the first ones of the SM the CTA runs up to 8 % slower, tile for tile, from the first to the
    // last: with the score pass of 288 units of 33,280 rows, a third of the CTAs (pass 1,260 to 1,360 us).
    // With given normalisers the score pass gains nothing but the launch: 7 to 23 tiles a CTA 0.4 to 2 % better beside the descriptor
    // kernel (units of 8,448 rows, 512 query rows).  Longer passes (given_score_long) are launched the same way, but that kernel does not
    // release them, so that they start when it and the last CTAs of the call before are gone, without the 4 us of an ordinary launch:
    // eight units of 33,280 rows 159.9 to 157.2 us (168 beside those CTAs), 288 of 2,000 201.8 to 198.2, 112 of 4,608 121.6 to 119.1.
    // fp32: the kernel before is split_rows_kernel, which releases the pass however long.  With an ordinary launch and so (event): 16 units
    // of 8,448 rows (512 query rows) 197 and 190 us, 12 with 1,024 rows 218 and 212; 24 of them, or 40 with 512 rows, within the 3 % that the
    // runs differ by.  Not released by that kernel: the same.
    // Behind the normaliser pass it has its first keys, queries and contractions done and its code fetched by the end of that pass
    // (`ahead`): events of 8 units of 640 rows 54.0 to 49.9 us (0.3 tiles a CTA), two fp32 ones of 1,024 52.1 to 50.0, 128 of 4,608 at
    // head_dim 64 (31 tiles) 182 to 176; 24 to 60 tiles 0.5 to 2.5 % (100 units of 11,366 rows 485.7 to 479.4), 90 to 200 up to 1.5, 250 and
    // 300 even, 400 and 600 up to 1 % worse (400 units of 28,416 rows 4,259 and 4,305).
    // Normaliser pass, which finds few CTAs in its way: early is better by 0.4 to 1.5 % up to 28 tiles, from 112 to 506 the two are
    // within the 1 % that the runs differ by (506: 3,603 and 3,574, 3,549 and 3,510).
    const int bit = kSmemBitScore + 2 * (NB >> 1) + 6 * PLAIN + 12 * SPLIT;
    cudaError_t e = lse_in ? cudaSuccess : allow_smem(L, bit, norm, smem);
    if (e == cudaSuccess) e = allow_smem(L, bit + 1, mass, smem);
    const bool own_tables = !lse_in && sh.n_units * rg.groups > grid;       // the row tables by a kernel of their own
    if (e == cudaSuccess && !lse_in) {
        Timed t(L, KID_SCORE_NORM);
        e = launch_kernel(total < 256 * grid, L.stream, norm, grid, kThreadsTc, smem, tmK, tmQ, L.desc, sh, rg, scale2, total, sub_rows, ws.part_m,
                             ws.part_l, nullptr, nullptr, nullptr, nullptr, 0, RowDefaults{}, own_tables, nullptr, ws.err);
    }
    if (e == cudaSuccess && own_tables) {
        Timed t(L, KID_ROW_COMBINE);
        // A row a thread (the rows rolled: the code runs once): with four rows a thread, 128 threads, 288 units of 640 rows 134.9 to 133.4 us,
        // 300 of 4,000 548 to 542.  Launched dependent, but the normaliser pass does not release it, so that its CTAs hold no slots of
        // that pass or of the next and it need not wait for an ordinary launch: 296 units of 640 143.6 to 142.4, 600 270 to 267.7.
        e = launch_dependent(L.stream, score_row_tables, sh.n_units * rg.groups, kRowThreads, 0, L.desc, rg, NB, total, grid, ws.part_m,
                             ws.part_l, ws.rowm, lse_out);
    }
    if (e == cudaSuccess) {
        Timed t(L, KID_SCORE_MASS);
        const bool early = lse_in || total < 256 * grid;
        e = launch_kernel(early, L.stream, mass, grid, kThreadsTc, smem, tmK, tmQ, L.desc, sh, rg, scale2, total, sub_rows, ws.part_m,
                             ws.part_l, lse_in, lse_out, own_tables ? ws.rowm : nullptr, rg.groups > 1 ? ws.s_part : s, rg.groups > 1 ? L.sum_T : 0, L.fill,
                             early && !lse_in ? (grid < L.sms ? 2 : 1) : 0, ws.roww, ws.err);
        ws.filled = L.fill.kind != nullptr;
        if (e == cudaSuccess && rg.groups > 1) {
            const int per = kFoldThreads * kFoldKeys;
            e = launch_dependent(L.stream, score_fold, dim3((L.max_T + per - 1) / per, sh.n_units), kFoldThreads, 0, L.desc,
                                 rg.groups, L.sum_T, ws.s_part, s);
            ++*L.launches;
        }
    }
    return e;
}
}  // namespace

cudaError_t launch_score_tc(const Launch& L, const float* lse_in, float* s, float* lse_out, Workspace& ws,
                            void* tmap_encode_fn) {
    const Shape& sh = L.sh;
    EncodeTiledFn encode = (EncodeTiledFn)tmap_encode_fn;
    const bool split = sh.dtype == CASK_DTYPE_FP32;
    if (split) {
        cudaError_t e = launch_split_rows(L, ws, true);
        if (e != cudaSuccess) return e;
    }
    int64_t k_rows = split ? 3 * L.sum_T : sh.page_size ? sh.n_pages * sh.page_size : 0;
    for (int u = 0; u < sh.n_units && !sh.page_size && !split; ++u)
        k_rows = std::max<int64_t>(k_rows, L.hdesc[u].k_off / sh.row_stride + L.hdesc[u].T);
    const int sub_rows = split ? (int)L.sum_T : key_box_rows(sh);      // split: rows from one part to the next
    const RowPlan pl = row_plan(sh.rows, sh.dtype);
    CUtensorMap tmK, tmQ;
    if (!encode_rows_bf16(tmap_encode_fn, &tmK, split ? ws.k_split : L.k, (uint64_t)k_rows, sh.d,
                          (uint64_t)(split ? sh.d : sh.row_stride) * 2, split ? kTileKeys : sub_rows))
        return cudaErrorInvalidValue;
    {
        cuuint64_t dims[3] = {(cuuint64_t)sh.d, (cuuint64_t)sh.rows, (cuuint64_t)sh.n_units * (split ? 3 : 1)};
        cuuint64_t strides[2] = {(cuuint64_t)sh.d * 2, (cuuint64_t)sh.rows * sh.d * 2};
        cuuint32_t box[3] = {64, 32, 1};
        cuuint32_t estr[3] = {1, 1, 1};
        if (encode(&tmQ, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, split ? ws.q_split : const_cast<void*>(L.q), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    if (split)
        return sh.d > 112 ? launch_passes<1, true, true>(L, pl.rg, tmK, tmQ, sub_rows, lse_in, s, lse_out, ws)
                          : launch_passes<1, false, true>(L, pl.rg, tmK, tmQ, sub_rows, lse_in, s, lse_out, ws);
    auto go_nb = [&](auto plain) {
        constexpr bool kPlain = decltype(plain)::value;
        if (pl.nb == 2) return launch_passes<2, kPlain, false>(L, pl.rg, tmK, tmQ, sub_rows, lse_in, s, lse_out, ws);
        if (pl.nb == 1) return launch_passes<1, kPlain, false>(L, pl.rg, tmK, tmQ, sub_rows, lse_in, s, lse_out, ws);
        return launch_passes<4, kPlain, false>(L, pl.rg, tmK, tmQ, sub_rows, lse_in, s, lse_out, ws);
    };
    return sh.d > 112 && pl.rg.groups == 1 ? go_nb(std::true_type{}) : go_nb(std::false_type{});
}

}  // namespace cask
