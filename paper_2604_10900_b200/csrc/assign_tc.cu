// Assignment of scratch rows to seeds on the tensor cores (Sec. 2.5: cosine as the base merge
// geometry): D[row, seed] = <k_row, k_seed> for 128-row tiles of the decode region against the
// unit's gathered seed keys, then per row the argmax of the cosine and the threshold tau.  Any head_dim up to 128:
// TMA fills the channels past a shorter row with zeros (128 units of 4,608 rows at head_dim 64: 430 to 35 us against the
// SIMT kernel that served them before).
//
// The contraction is small (2*128*m*128 flop per tile) next to the 32 KB of K it consumes, so the
// kernel is bound by the K stream: a 4-stage TMA ring feeds one persistent CTA per SM.
// What kept it from the stream's rate, 288 units of 33,280 rows with 64 and 96 seeds (508 and 586 us, 4.8 and 4.2 TB/s): one issuer took 1,730 clk a
// tile, 850 of them blocked on the tensor pipe and the rest in two barrier probes one after the other, where two overlap them (452, 588); each group
// walked through the other groups' tiles and added up the lost mass with ten shuffles a tile instead of a unit (410, 541); the seed of the
// greatest cosine was looked for in every chunk (409, 477); waiting warps read the abort flag after every probe (382, 454: 6.4 and 5.4 TB/s).
//   warp 0      TMA producer: seed matrix once per unit, K tiles through the ring
//   warps 1-2   tcgen05.mma issue, even and odd tiles (warp 1 also owns the TMEM allocation)
//   warps 4-19  epilogue in groups of four warps (one per TMEM lane quadrant); group e takes the
//               tiles e, e+G, e+2G, ... of the CTA and owns one accumulator buffer, so up to G
//               tiles are in flight and the global-memory round trips of a tile (row kind, score,
//               the fixed-point mass atomics) overlap with the next tiles
// With m <= 128 seeds in every unit the TMEM holds four buffers of 128 columns, one per group.  With more
// seeds it holds two buffers of 256 columns and two groups share each: one takes the first seed columns and
// finishes the row, the other takes the rest and hands its best seed over through shared memory.
//
// More than 256 seeds (MANY): their columns are taken in chunks of at most 128, a launch each, with four buffers.  A row's greatest and second
// greatest value and the former's seed go from launch to launch through the workspace; the launch with a unit's last chunk finishes its
// rows.  Rows that the sums of the tensor cores cannot tell (see kCloseSeeds) are listed, and assign_close_kernel decides them by the sums of
// assign_simt_kernel, which served these shapes before: a row goes where that kernel sends it.  Chunks of 128 and four buffers, not of
// 256 and two: a pass of the former takes half of one of the latter (0.44 and 0.87 ms for 9.6 M rows).  Event (512 query rows) of 16 units of
// 15,276 rows (380 seeds) 1,248 to 250 us, 104 of 27,043 (270) 10,980 to 1,337, 240 of 3,000 (576) 4,829 to 748, 4 of 9,000 (860) 517 to
// 195, 8 of 1,024 (434) 141 to 75, one of 3,000 (1,386) 303 to 166.
//
// fp32 caches (SPLIT): the contraction takes the bf16 parts of the rows and the seeds (split.cu) in six products as the scoring
// passes do (score_tc.cu), one tile of six 16 KB regions at a time, m <= 128; the row norms come from the split.  What that sum
// cannot tell, which of two seeds within 8e-6 of one another a row is closer to, or on which side of tau it lies, is decided by the
// plain fp32 cosines of assign_simt_kernel (see kClose): a row goes where that kernel sends it.  (16 units of 8,448 rows, m = 96:
// 236 us on the SIMT kernel, 48 here, 33 without the plain cosines.)
#include "tc_common.cuh"

namespace cask {

namespace {

using namespace tc;

constexpr int kTileRows = 128;
constexpr int kStages = 4;
constexpr int kEpiWarp0 = 4;
constexpr int kMaxGroups = 4;
constexpr int kThreadsA = (kEpiWarp0 + 4 * kMaxGroups) * 32;
// A parity wait is only sound for a waiter that has seen the phase before the one it waits for complete: a phase
// further behind has the same parity as the one awaited and the wait would pass at once.  Tile t uses key stage
// t % kStages and belongs to epilogue group t % n_bufs (n_bufs = 4 or 2), so with kStages a multiple of n_bufs a group
// meets every phase of the stages it reads, in order.  Any other ring depth lets a fast group reach a stage whose
// previous tile (another group's) has not landed yet, pass the wait and release the stage early.
static_assert(kStages % kMaxGroups == 0, "key ring depth must be a multiple of the epilogue group count");
constexpr uint32_t kSeedRegionBytes = 256 * 128;       // 256 seeds x 64 bf16
constexpr uint32_t kSeedBytes = 2 * kSeedRegionBytes;
constexpr uint32_t kKRegionBytes = 128 * 128;
constexpr uint32_t kKStageBytes = 2 * kKRegionBytes;

constexpr int kRegions = 6;                // SPLIT: (part l, m, h) x (64-channel half) of a tile
struct __align__(8) ABarriers {
    uint64_t b_full[2], b_empty[2];   // seed matrix buffers (two when every unit has at most 128 columns)
    uint64_t k_full[kRegions], k_empty[kRegions];   // the ring's stages, or the regions of one tile
    uint64_t d_full[kMaxGroups], d_empty[kMaxGroups];
    uint64_t inv_ready[kMaxGroups];   // a group's table of inverse seed norms is written
    uint64_t x_full[2];      // shared buffers: the second group's best seed of a tile is in shared memory
    uint64_t mma_drain[2];   // give-up path only: an issuer's contractions in flight have completed
};

struct ASmemTail {
    ABarriers bar;
    uint32_t tmem_base;
    int abort;
    alignas(16) float inv_nu[kMaxGroups][2][256];   // 1/|k_seed| (0 for a zero seed): every epilogue group keeps its
                                        // own copy, double-buffered over the units it has tiles in
    int seed_row[kMaxGroups][2][256];   // cache row of every seed of the unit, buffered the same way
    alignas(16) float w[128]; // channel weights of the similarity (1 when none are given)
    float x_val[2][2][128];   // shared buffers: best dot product / seed norm and its seed,
    int x_idx[2][2][128];     //   per buffer, per use parity, per tile row
};

constexpr size_t kSmemBytesA = 1024 + kSeedBytes + kStages * kKStageBytes + sizeof(ASmemTail);
static_assert(2 * kRegions * kKRegionBytes <= kSeedBytes + kStages * kKStageBytes, "SPLIT: seeds and one tile, six regions each");

// MANY: the seeds of a launch, and what goes from one to the next.
struct Chunk {
    int c0, width;                   // seeds [c0, c0 + width) of every unit
    float2* best;                    // [sumT] greatest and second greatest dot product / seed norm of a row so far
    int32_t* best_u;                 // [sumT] the former's seed
    int32_t *close, *n_close;        // [sumT], [1] rows left to assign_close_kernel
};

constexpr uint8_t kKindClose = 0x80;     // MANY: kind of a listed row until assign_close_kernel has decided it

// Walks this CTA's contiguous range of scratch tiles, unit by unit.
struct TileWalk {
    const UnitDesc* desc;
    int g, g_end, u, n_units;
    int c0;                          // units of no more seeds are passed over
    __device__ void init(const UnitDesc* d, int n_units_, int total, int first_seed) {
        desc = d;
        n_units = n_units_;
        c0 = first_seed;
        g = (int)(((long long)total * blockIdx.x) / gridDim.x);
        g_end = (int)(((long long)total * (blockIdx.x + 1)) / gridDim.x);
        u = warp_find_unit(n_units, g, [&](int v) { return d[v].atile0; });
        skip_empty();
    }
    __device__ void skip_empty() {
        for (;;) {
            while (u < n_units - 1 && g >= desc[u].atile0 + desc[u].n_atiles) ++u;
            if (c0 == 0 || g >= g_end || desc[u].plan[CASK_PLAN_M] > c0) return;
            g = min(g_end, desc[u].atile0 + desc[u].n_atiles);
        }
    }
    __device__ bool valid() const { return g < g_end; }
    __device__ int tile_in_unit() const { return g - desc[u].atile0; }
    // tiles of the current unit that belong to this CTA from g on
    __device__ int run() const { return min(g_end, desc[u].atile0 + desc[u].n_atiles) - g; }
    __device__ void advance(int n) {
        g += n;
        if (g < g_end) { ++u; skip_empty(); }
    }
};

// 16 bytes of shared memory by a shared-space load (through a generic pointer the read takes the path of global loads).
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 r;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a));
    return r;
}

// Squared (channel-weighted) norm of one staged key row as a packed pair of partial sums.  The row's sixteen
// 16-byte pieces are read in a lane-dependent order (no bank conflicts); a bf16 is the upper half of an fp32, so
// two integer operations unpack a pair.  The 128-byte swizzle stores logical piece p of row r at position
// p ^ (r & 7), which matters only for finding the piece's channel weights.  Four running sums, one per 32-bit
// word of a piece, keep the dependent chain of packed multiply-adds at sixteen links instead of sixty-four.
template <bool WEIGHTED, bool FULL>
__device__ __forceinline__ uint64_t row_norm2(const uint8_t* base, int lane, int row, const float* w, int n_kb) {
    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
    const uint32_t b32 = smem_u32(base);
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {
        if (!FULL && kb >= n_kb) break;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int pos = (c + lane) & 7;
            const uint4 raw = lds128(b32 + kb * kKRegionBytes + (pos << 4));
            const uint32_t wv[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint64_t f2 = pack2(__uint_as_float(wv[x] << 16), __uint_as_float(wv[x] & 0xFFFF0000u));
                if (WEIGHTED) {
                    const float2 w2 = *reinterpret_cast<const float2*>(&w[kb * 64 + ((pos ^ (row & 7)) << 3) + 2 * x]);
                    acc[x] = fma2(fma2(f2, pack2(w2.x, w2.y), 0ull), f2, acc[x]);
                } else {
                    acc[x] = fma2(f2, f2, acc[x]);
                }
            }
        }
    }
    return add2(add2(acc[0], acc[1]), add2(acc[2], acc[3]));
}

// Best seed among the accumulator columns [c_lo, c_hi) of this thread's row: the greatest dot * 1/|k_seed|, the
// first seed among equals.  PAIR = 1: a seed owns two adjacent columns (the hi and lo parts of its weighted key)
// whose sum is its dot product.  Sixteen columns at a time, the next sixteen on their way meanwhile.  A chunk costs a multiply (packed in
// pairs) and a maximum per seed; the position of the maximum is looked for only in a chunk that beats everything before it: first its half
// of the chunk, then its place there, so that the chain of selections is half as long.  SECOND: the second greatest value as well.
template <int PAIR>
__device__ __forceinline__ void chunk_products(const float (&v)[16], uint32_t inv32, int cc, int c_hi, float (&p)[2][PAIR ? 4 : 8]) {
    constexpr int kHalf = PAIR ? 4 : 8;          // seeds per half chunk
    const int u0 = PAIR ? cc >> 1 : cc, u_hi = PAIR ? c_hi >> 1 : c_hi;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int x = 0; x < kHalf; x += 4) {
            const int at = h * kHalf + x;        // (inverse norms 16 bytes at a time, shared-space)
            const uint4 q = lds128(inv32 + (uint32_t)(u0 + at) * 4u);
            const uint64_t n01 = pack2(__uint_as_float(q.x), __uint_as_float(q.y)), n23 = pack2(__uint_as_float(q.z), __uint_as_float(q.w));
            if (PAIR) {
                unpack2(mul2(pack2(v[2 * at] + v[2 * at + 1], v[2 * at + 2] + v[2 * at + 3]), n01), p[h][x], p[h][x + 1]);
                unpack2(mul2(pack2(v[2 * at + 4] + v[2 * at + 5], v[2 * at + 6] + v[2 * at + 7]), n23), p[h][x + 2], p[h][x + 3]);
            } else {
                unpack2(mul2(pack2(v[at], v[at + 1]), n01), p[h][x], p[h][x + 1]);
                unpack2(mul2(pack2(v[at + 2], v[at + 3]), n23), p[h][x + 2], p[h][x + 3]);
            }
        }
    if (cc + 16 > c_hi) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int x = 0; x < kHalf; ++x)
                if (u0 + h * kHalf + x >= u_hi) p[h][x] = -INFINITY;
    }
}

template <int PAIR, bool SECOND>
__device__ __forceinline__ void best_of_chunk(const float (&v)[16], uint32_t inv32, int cc, int c_hi, float& best, int& best_u, float& second) {
    constexpr int kHalf = PAIR ? 4 : 8;
    const int u0 = PAIR ? cc >> 1 : cc;
    float p[2][kHalf];
    chunk_products<PAIR>(v, inv32, cc, c_hi, p);
    float m0 = -INFINITY, m1 = -INFINITY, b2 = -INFINITY;
#pragma unroll
    for (int x = 0; x < kHalf; ++x) {
        if (SECOND) b2 = fmaxf(b2, fmaxf(fminf(m0, p[0][x]), fminf(m1, p[1][x])));
        m0 = fmaxf(m0, p[0][x]);
        m1 = fmaxf(m1, p[1][x]);
    }
    const float bm = fmaxf(m0, m1);
    if (SECOND) second = fmaxf(fmaxf(second, b2), fmaxf(fminf(m0, m1), fminf(best, bm)));
    if (bm > best) {
        best = bm;
        const bool low = m0 == bm;
        int at = kHalf - 1;
#pragma unroll
        for (int x = kHalf - 2; x >= 0; --x) {
            float w;
            asm("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\tselp.f32 %0, %1, %2, q;\n\t}" : "=f"(w) : "f"(p[0][x]), "f"(p[1][x]), "r"((int)low));
            if (w == bm) at = x;
        }
        best_u = u0 + at + (low ? 0 : kHalf);
    }
}

template <int PAIR, bool SECOND = false>
__device__ __forceinline__ void best_seed(uint32_t taddr, const float* inv, int c_lo, int c_hi, float& best, int& best_u, float& second) {
    const uint32_t inv32 = smem_u32(inv);
    const int last = max(c_lo, (c_hi - 1) & ~15);      // (every load is unconditional: past the last chunk it is that one again)
    float a[16], b[16];
    tc_ld16(taddr + c_lo, a);
#pragma unroll 1
    for (int cc = c_lo; cc < c_hi; cc += 32) {
        tc_wait_ld_regs(a);
        tc_ld16(taddr + min(cc + 16, last), b);
        best_of_chunk<PAIR, SECOND>(a, inv32, cc, c_hi, best, best_u, second);
        tc_wait_ld_regs(b);
        tc_ld16(taddr + min(cc + 32, last), a);
        if (cc + 16 < c_hi) best_of_chunk<PAIR, SECOND>(b, inv32, cc + 16, c_hi, best, best_u, second);
    }
    tc_wait_ld_regs(a);
}

// The value alone, and the chunk it is in; the seed of the rows that join (`ask`) afterwards.  Few rows do (tau is 0.9), and a search in
// every chunk is two fifths of the instructions a tile takes.
__device__ __forceinline__ void best_value(uint32_t taddr, const float* inv, int c_hi, float& best, int& best_chunk) {
    const uint32_t inv32 = smem_u32(inv);
    const int last = max(0, (c_hi - 1) & ~15);
    auto look = [&](const float (&v)[16], int cc) __attribute__((always_inline)) {
        float p[2][8];
        chunk_products<0>(v, inv32, cc, c_hi, p);
        float m0 = p[0][0], m1 = p[1][0];
#pragma unroll
        for (int x = 1; x < 7; x += 2) {
            m0 = fmaxf(fmaxf(m0, p[0][x]), p[0][x + 1]);
            m1 = fmaxf(fmaxf(m1, p[1][x]), p[1][x + 1]);
        }
        m0 = fmaxf(fmaxf(m0, m1), fmaxf(p[0][7], p[1][7]));
        if (m0 > best) { best = m0; best_chunk = cc; }
    };
    float a[16], b[16];
    tc_ld16(taddr, a);
#pragma unroll 1
    for (int cc = 0; cc < c_hi; cc += 32) {
        tc_wait_ld_regs(a);
        tc_ld16(taddr + min(cc + 16, last), b);
        look(a, cc);
        tc_wait_ld_regs(b);
        tc_ld16(taddr + min(cc + 32, last), a);
        if (cc + 16 < c_hi) look(b, cc + 16);
    }
    tc_wait_ld_regs(a);
}
__device__ __forceinline__ int find_seed(uint32_t taddr, const float* inv, int c_hi, bool ask, float best, int best_chunk) {
    const uint32_t inv32 = smem_u32(inv);
    int best_u = -1;
    unsigned todo = __ballot_sync(0xffffffffu, ask);
    while (todo) {                               // chunk by chunk, for all rows that have theirs there
        const int cc = __shfl_sync(0xffffffffu, best_chunk, __ffs(todo) - 1);
        float v[16], p[2][8];
        tc_ld16(taddr + cc, v);
        tc_wait_ld_regs(v);
        chunk_products<0>(v, inv32, cc, c_hi, p);
        int at = 15;
#pragma unroll
        for (int x = 14; x >= 0; --x)
            if (p[x >> 3][x & 7] == best) at = x;
        const bool here = ask && best_chunk == cc;
        if (here) best_u = cc + at;
        todo &= ~__ballot_sync(0xffffffffu, here);
    }
    return best_u;
}

// fp32 rows whose best cosine is within kClose of another seed's or of tau are decided by the sums assign_simt_kernel takes, one
// multiply-add after the other in the order of the channels.  A margin, not a bound: the two kernels' cosines differ by up to 1.2e-6 (768,000
// of them), so two seeds 7.6e-6 apart come out in the same order either way unless the keys are made for it (see kCloseSeeds).  Without
// this, one event of 16 units of 8,448 rows in eight sent a row to another seed.
constexpr float kClose = 1.f / 131072.f;
// bf16 rows, MANY.  The plain sum of 128 products rounds 127 times by at most 2^-24 of the norms' product: 7.6e-6.  The tensor cores' sum lacks
// at most 4.8e-6: a product is cut at 2^-25 of the greatest magnitude of its step (keys of one great channel and 120 equal small ones show it,
// product by product), a step's sum at 2^-23.  Between the kernels two cosines may so move by 2.5e-5 against one another and one
// by 1.25e-5 against tau, where the row's norm adds 1e-6.  The greatest difference of one cosine over twelve kinds of keys, 168,000 rows each
// (normal, channels of 8 and 800 times the rest, log-normal, all positive, near one another), is 3.3e-6, but keys can be made of which a margin of
// 7.6e-6 sends a row elsewhere.
constexpr float kCloseSeeds = 3.5f / 131072.f, kCloseTau = 2.f / 131072.f;

// Of the seeds marked in `close` the one of greatest plain cosine, the first among equals; its cosine in sm.  Four seeds at a time.  The
// loops stay rolled: the code runs once or twice a CTA, and fetching its instructions takes longer than they do.
__device__ __noinline__ int plain_best(const float* __restrict__ K, const Shape& sh, const UnitDesc& ud, int row, const int* srow,
                                       const float* __restrict__ seed_norm, const uint32_t (&close)[4], float& sm) {
    const int d4 = sh.d / 4;
    const float4* rp = reinterpret_cast<const float4*>(K + row_elem_off(sh, ud, ud.k_off, row));
    sm = -INFINITY;
    int best_u = -1, w = 0;
    for (uint32_t left = close[0];;) {
        int c[4], n = 0;
        float nu[4];
        const float4* sp[4];
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            while (!left && w < 3) left = close[++w];
            if (left) {
                c[k] = 32 * w + __ffs(left) - 1;
                left &= left - 1;
                n = k + 1;
            }
            const int at = c[min(k, max(n - 1, 0))];
            if (n) {
                sp[k] = reinterpret_cast<const float4*>(K + row_elem_off(sh, ud, ud.k_off, CASK_IDX(srow[at], ud.T, sh.err)));
                nu[k] = seed_norm[at];
            }
        }
        if (n == 0) return best_u;
        const float4 *s0 = sp[0], *s1 = sp[1], *s2 = sp[2], *s3 = sp[3];
        // the rows into L1 first, a load a line and all of them in flight
#pragma unroll 1
        for (int x = 0; x < d4; x += 8) {
            float t;
            asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(t) : "l"(rp + x));
            asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(t) : "l"(s0 + x));
            asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(t) : "l"(s1 + x));
            asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(t) : "l"(s2 + x));
            asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(t) : "l"(s3 + x));
        }
        float a[4] = {0.f, 0.f, 0.f, 0.f}, m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
        for (int x = 0; x < d4; ++x) {
            const float4 r = rp[x], v[4] = {s0[x], s1[x], s2[x], s3[x]};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                a[k] = fmaf(r.w, v[k].w, fmaf(r.z, v[k].z, fmaf(r.y, v[k].y, fmaf(r.x, v[k].x, a[k]))));
            m[0] = fmaf(r.x, r.x, m[0]);
            m[1] = fmaf(r.y, r.y, m[1]);
            m[2] = fmaf(r.z, r.z, m[2]);
            m[3] = fmaf(r.w, r.w, m[3]);
        }
        const float nj = sqrtf((m[0] + m[1]) + (m[2] + m[3]));
#pragma unroll 1
        for (int k = 0; k < n; ++k) {
            const float x = nj > 0.f && nu[k] > 0.f ? a[0] / (nj * nu[k]) : 0.f;
            if (x > sm) { sm = x; best_u = c[k]; }
            a[0] = a[1]; a[1] = a[2]; a[2] = a[3];
        }
    }
}

// The TMA producer of a paged cache (one warp).  The block table is read for several tiles of a unit at once, a lane per page piece,
// and one such batch ahead of its use: nothing touches a page number, not even to check it, before its own tiles are issued, so
// the table's latency hides behind the batch before.  The units' descriptors come the same way, 32 units at a time.
// (Looked up and checked tile by tile, the page numbers and the descriptors were waited for: 1,600 clk a tile with pages of
// 64 rows, where the tile's copies and its epilogue need some 1,900 between them.  512 units of 4,700 to 33,000 rows in pages of 64
// 616 -> 525 us, 3,072 units of 640 rows in pages of 16 105 -> 76; as a call of its own 530 and 85.)
__device__ __forceinline__ void produce_paged(const CUtensorMap* tmK, const CUtensorMap* tmSeed, const UnitDesc* __restrict__ desc,
                                              const Shape& sh, int g, int g_end, int u, int c0, int sub_rows, int wpair, int n_kb, bool dual,
                                              uint8_t* b_smem, uint8_t* k_smem, ASmemTail* tail) {
    ABarriers& bar = tail->bar;
    volatile int* abort_flag = &tail->abort;
    const int lane = threadIdx.x & 31;
    const int piece_shift = 31 - __clz(sub_rows), tile_shift = 7 - piece_shift;      // rows of a piece, pieces of a tile
    static_assert(kTileRows == 128, "");
    const int pieces = 1 << tile_shift, my_tile = lane >> tile_shift, my_piece = lane & (pieces - 1);
    const uint32_t seed_region = dual ? 128u * 128u : kSeedRegionBytes;
    // descriptors of the units first_u + lane
    int first_u = u - 32, c_at0 = 0, c_nat = 0, c_bt0 = 0, c_P = 0, c_T = 0, c_seed = 0, c_m = 0;
    auto cache_units = [&]() {
        if (u - first_u < 32) return;
        first_u = u;
        const UnitDesc& d = desc[min(u + lane, sh.n_units - 1)];
        c_at0 = d.atile0; c_nat = d.n_atiles; c_bt0 = d.bt0; c_P = d.P; c_T = d.T; c_seed = d.seed_base + c0; c_m = d.plan[CASK_PLAN_M];
    };
    struct Batch { int n, row0, T, seed; bool fresh; int page, in_page; };
    int last_u = -1;
    auto next_batch = [&]() {
        Batch b{0, 0, 0, 0, false, 0, 0};
        if (g >= g_end) return b;
        cache_units();
        int at0 = __shfl_sync(0xffffffffu, c_at0, u - first_u), nat = __shfl_sync(0xffffffffu, c_nat, u - first_u);
        for (;;) {
            while (u < sh.n_units - 1 && g >= at0 + nat) {
                ++u;
                cache_units();
                at0 = __shfl_sync(0xffffffffu, c_at0, u - first_u);
                nat = __shfl_sync(0xffffffffu, c_nat, u - first_u);
            }
            if (c0 == 0 || __shfl_sync(0xffffffffu, c_m, u - first_u) > c0) break;
            g = min(g_end, at0 + nat);
            if (g >= g_end) return b;
        }
        const int P = __shfl_sync(0xffffffffu, c_P, u - first_u), bt0 = __shfl_sync(0xffffffffu, c_bt0, u - first_u);
        b.T = __shfl_sync(0xffffffffu, c_T, u - first_u);
        b.seed = __shfl_sync(0xffffffffu, c_seed, u - first_u);
        b.n = min(min(g_end, at0 + nat) - g, 32 >> tile_shift);
        b.row0 = (P & ~(sub_rows - 1)) + (g - at0) * kTileRows;
        b.fresh = u != last_u;
        last_u = u;
        const int row = b.row0 + my_tile * kTileRows + my_piece * sub_rows, pg = row / sh.page_size;
        if (my_tile < b.n && row < b.T) {
            b.page = sh.bt[bt0 + pg];
            b.in_page = row - pg * sh.page_size;
        }
        g += b.n;
        return b;
    };
    uint32_t kit = 0, ucount = 0;
    bool ok = true;
    Batch cur = next_batch();
    while (cur.n > 0 && ok) {
        const Batch nxt = next_batch();
        if (cur.fresh) {
            const uint32_t sb = dual ? (ucount & 1u) : 0u, suse = dual ? (ucount >> 1) : ucount;
            ok = mbar_wait<true>(&bar.b_empty[sb], (suse & 1u) ^ 1u, abort_flag);
            if (!ok) break;
            if (lane == 0) {
                mbar_expect_tx(&bar.b_full[sb], n_kb * seed_region);
                uint8_t* bdst = b_smem + sb * 2 * seed_region;
                tma_load_2d(bdst, tmSeed, &bar.b_full[sb], 0, cur.seed << wpair);
                if (n_kb == 2) tma_load_2d(bdst + seed_region, tmSeed, &bar.b_full[sb], 64, cur.seed << wpair);
            }
            ++ucount;
        }
        for (int t = 0; t < cur.n && ok; ++t, ++kit) {
            const int st = kit % kStages;
            ok = mbar_wait<true>(&bar.k_empty[st], ((kit / kStages) & 1u) ^ 1u, abort_flag);
            if (!ok) break;
            uint8_t* dst = k_smem + st * kKStageBytes + my_piece * sub_rows * 128;
            const int n_sub = min(pieces, (cur.T - cur.row0 - t * kTileRows + sub_rows - 1) >> piece_shift);
            if (lane == 0) mbar_expect_tx(&bar.k_full[st], (uint32_t)(n_sub << piece_shift) * (128u * n_kb));
            __syncwarp();
            if (my_tile == t && my_piece < n_sub) {
                const int prow = (int)page_row(sh, cur.page, cur.in_page);
                tma_load_2d(dst, tmK, &bar.k_full[st], 0, prow);
                if (n_kb == 2) tma_load_2d(dst + kKRegionBytes, tmK, &bar.k_full[st], 64, prow);
            }
        }
        cur = nxt;
    }
    if (!ok)
        for (uint32_t j = (kit >= (uint32_t)kStages ? kit - kStages : 0); j < kit; ++j)
            for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.k_full[j % kStages], (j / kStages) & 1u); ++it) {}
}

// FULL: head_dim 113..128 (the compiler then knows the numbers of channel halves and contraction steps)
template <bool FULL, bool SPLIT, bool MANY>
__global__ void __launch_bounds__(kThreadsA, 1)
assign_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmSeed,
                 const UnitDesc* __restrict__ desc, Shape sh, int total_tiles, int n_bufs, int sub_rows, int wpair,
                 int seed_part_rows, const float* __restrict__ K, const float* __restrict__ k_norm,
                 const float* __restrict__ s, const int32_t* __restrict__ plan,
                 const int32_t* __restrict__ seed_rows, const float* __restrict__ seed_norm,
                 uint8_t* __restrict__ kind, int32_t* __restrict__ seed_of, float* __restrict__ sim,
                 int32_t* __restrict__ grp, unsigned long long* __restrict__ mass_fx,
                 int32_t* __restrict__ njoin, int32_t* __restrict__ mem_row, int32_t* __restrict__ mem_seed, int max_m, float tau,
                 float eps, int32_t* __restrict__ err, const Chunk chunk) {
    const int c0 = MANY ? chunk.c0 : 0;                  // first seed of the launch
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* b_smem = smem;
    uint8_t* k_smem = smem + (SPLIT ? kRegions * kKRegionBytes : kSeedBytes);
    ASmemTail* tail = reinterpret_cast<ASmemTail*>(smem + kSeedBytes + kStages * kKStageBytes);
    ABarriers& bar = tail->bar;
    volatile int* abort_flag = &tail->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_kb = FULL || sh.d > 64 ? 2 : 1;          // 64-channel halves of a row that hold data
    const int n_ks = FULL ? 8 : (sh.d + 15) >> 4;        // contraction steps of 16 channels
    const int buf_cols = 512 / n_bufs;                   // TMEM columns per accumulator buffer
    const int split = kMaxGroups / n_bufs;               // groups sharing one buffer (1 or 2)
    // At most 128 accumulator columns in every unit: the seed matrix is loaded as 128 rows and the shared-memory
    // area holds two of them, so the next unit's seeds arrive while the tensor pipe still works on this unit's.
    const bool dual = n_bufs == kMaxGroups;
    // n_bufs is 2 or 4: positions among the buffers by mask and shift (a remainder by a run-time value is a division
    // sequence, and the epilogue warps take one per tile, their own or not)
    const uint32_t buf_mask = (uint32_t)n_bufs - 1u, buf_shift = n_bufs == 4 ? 2u : 1u;
    const uint32_t seed_region = dual ? 128u * 128u : kSeedRegionBytes;      // one 64-channel half of a seed buffer

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(&bar.b_full[i], 1); mbar_init(&bar.b_empty[i], SPLIT || !dual ? 1 : 2); }
        for (int i = 0; i < kRegions; ++i) { mbar_init(&bar.k_full[i], 1); mbar_init(&bar.k_empty[i], SPLIT ? 1 : 1 + 4); }
        for (int i = 0; i < kMaxGroups; ++i) { mbar_init(&bar.d_full[i], 1); mbar_init(&bar.d_empty[i], 4 * split); }
        for (int i = 0; i < kMaxGroups; ++i) mbar_init(&bar.inv_ready[i], 128);
        mbar_init(&bar.x_full[0], 4);
        mbar_init(&bar.x_full[1], 4);
        mbar_init(&bar.mma_drain[0], 1);
        mbar_init(&bar.mma_drain[1], 1);
        tail->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 128) tail->w[threadIdx.x] = sh.chan_w && (int)threadIdx.x < sh.d ? sh.chan_w[threadIdx.x] : 1.f;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tail->tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tail->tmem_base;
    pdl_wait();

    TileWalk wk;
    wk.init(desc, sh.n_units, total_tiles, c0);

    if (warp == 0) {
        // ================= TMA producer =================
        if (!SPLIT && sh.page_size) {
            produce_paged(&tmK, &tmSeed, desc, sh, wk.g, wk.g_end, wk.u, c0, sub_rows, wpair, n_kb, dual, b_smem, k_smem, tail);
        } else if (lane == 0) {
            uint32_t kit = 0, ucount = 0;
            bool ok = true;
            while (wk.valid() && ok) {
                const UnitDesc& ud = desc[wk.u];
                if constexpr (SPLIT) {
                    const int nt = wk.run();
                    const int krow0 = (int)ud.tok_off + ud.P + wk.tile_in_unit() * kTileRows;
                    for (int t = 0; t < nt && ok; ++t, ++kit) {
                        // parts in the order of their use, l, m, h; part p of the keys starts p * sub_rows rows down the table
                        for (int r = 0; r < kRegions && ok; ++r) {
                            if ((r & 1) >= n_kb) continue;
                            ok = mbar_wait<true>(&bar.k_empty[r], (kit & 1u) ^ 1u, abort_flag);
                            if (!ok) break;
                            mbar_expect_tx(&bar.k_full[r], kKRegionBytes);
                            tma_load_2d(k_smem + r * kKRegionBytes, &tmK, &bar.k_full[r], 64 * (r & 1),
                                        (2 - (r >> 1)) * sub_rows + krow0 + t * kTileRows);
                        }
                        if (t == 0 && ok) {
                            ok = mbar_wait<true>(&bar.b_empty[0], (ucount & 1u) ^ 1u, abort_flag);
                            if (!ok) break;
                            mbar_expect_tx(&bar.b_full[0], 3 * n_kb * kKRegionBytes);
                            for (int r = 0; r < kRegions; ++r)
                                if ((r & 1) < n_kb)
                                    tma_load_2d(b_smem + r * kKRegionBytes, &tmSeed, &bar.b_full[0], 64 * (r & 1),
                                                (2 - (r >> 1)) * seed_part_rows + ud.seed_base);
                        }
                    }
                    ++ucount;
                    wk.advance(nt);
                    continue;
                }
                const uint32_t sb = dual ? (ucount & 1u) : 0u, suse = dual ? (ucount >> 1) : ucount;
                ok = mbar_wait<true>(&bar.b_empty[sb], (suse & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                mbar_expect_tx(&bar.b_full[sb], n_kb * seed_region);
                uint8_t* bdst = b_smem + sb * 2 * seed_region;
                tma_load_2d(bdst, &tmSeed, &bar.b_full[sb], 0, (ud.seed_base + c0) << wpair);
                if (n_kb == 2) tma_load_2d(bdst + seed_region, &tmSeed, &bar.b_full[sb], 64, (ud.seed_base + c0) << wpair);
                ++ucount;
                const int krow0 = (int)(ud.k_off / sh.row_stride) + ud.P + wk.tile_in_unit() * kTileRows;
                const int nt = wk.run();
                for (int t = 0; t < nt && ok; ++t, ++kit) {
                    const int st = kit % kStages;
                    ok = mbar_wait<true>(&bar.k_empty[st], ((kit / kStages) & 1u) ^ 1u, abort_flag);
                    if (!ok) break;
                    uint8_t* dst = k_smem + st * kKStageBytes;
                    mbar_expect_tx(&bar.k_full[st], n_kb * kKRegionBytes);
                    tma_load_2d(dst, &tmK, &bar.k_full[st], 0, krow0 + t * kTileRows);
                    if (n_kb == 2) tma_load_2d(dst + kKRegionBytes, &tmK, &bar.k_full[st], 64, krow0 + t * kTileRows);
                }
                wk.advance(nt);
            }
            if (!ok && SPLIT) {
                for (int r = 0; r < kRegions; ++r)
                    for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.k_full[r], kit & 1u); ++it) {}
                for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.b_full[0], ucount & 1u); ++it) {}
            } else if (!ok) {
                for (uint32_t j = (kit >= (uint32_t)kStages ? kit - kStages : 0); j < kit; ++j)
                    for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.k_full[j % kStages], (j / kStages) & 1u); ++it) {}
            }
        }
    } else if (warp == 1 || (!SPLIT && dual && warp == 2)) {        // (with two buffers a second issuer's contractions only delay the first one's)
        // ================= MMA issuers: even and odd tiles =================
        if (lane == 0) {
            uint32_t kit = 0, ucount = 0;
            bool ok = true;
            const uint32_t b_lo = umma_desc_lo(smem_u32(b_smem)), k_lo = umma_desc_lo(smem_u32(k_smem));
            while (wk.valid() && ok) {
                const UnitDesc& ud = desc[wk.u];
                const int m_all = max(0, min(plan[wk.u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
                const int m = MANY ? min(m_all - c0, chunk.width) : m_all;
                const uint32_t idesc = umma_idesc(max(16, ((m << wpair) + 15) & ~15));
                if constexpr (SPLIT) {
                    ok = mbar_wait<true>(&bar.b_full[0], ucount & 1u, abort_flag);
                    if (!ok) break;
                    ++ucount;
                    const int nt = wk.run();
                    for (int t = 0; t < nt && ok; ++t, ++kit) {
                        const uint32_t buf = kit & buf_mask, use = kit >> buf_shift;
                        ok = mbar_wait<true>(&bar.d_empty[buf], (use & 1u) ^ 1u, abort_flag);
#pragma unroll
                        for (int kp = 0; kp < 3; ++kp) {
                            for (int kb = 0; kb < n_kb && ok; ++kb) ok = mbar_wait<true>(&bar.k_full[2 * kp + kb], kit & 1u, abort_flag);
                            if (!ok) break;
                            tc_fence_after();
#pragma unroll
                            for (int qi = 0; qi < 3; ++qi) {
                                // row part l: with seed part h; m: with h, m; h: with l, m, h
                                if (kp == 0 && qi != 2) continue;
                                if (kp == 1 && qi == 0) continue;
                                const int qp = kp == 1 ? 3 - qi : qi;
#pragma unroll
                                for (int kk = 0; kk < 8; ++kk) {
                                    if (kk >= n_ks) break;
                                    const uint32_t at = (uint32_t)((kk >> 2) * kKRegionBytes + (kk & 3) * 32) >> 4;
                                    const uint32_t dk = k_lo + ((2 * kp * kKRegionBytes) >> 4) + at;
                                    const uint32_t ds = b_lo + ((2 * qp * kKRegionBytes) >> 4) + at;
                                    if (kp == 0 && kk == 0) tc_mma_lo<false>(tmem_base + buf * buf_cols, dk, ds, idesc);
                                    else tc_mma_lo<true>(tmem_base + buf * buf_cols, dk, ds, idesc);
                                }
                            }
                            for (int kb = 0; kb < n_kb; ++kb) tc_commit(&bar.k_empty[2 * kp + kb]);
                        }
                        if (!ok) break;
                        tc_commit(&bar.d_full[buf]);
                    }
                    wk.advance(nt);
                    if (ok) tc_commit(&bar.b_empty[0]);
                    continue;
                }
                const uint32_t sb = dual ? (ucount & 1u) : 0u, suse = dual ? (ucount >> 1) : ucount;
                ok = mbar_wait<true>(&bar.b_full[sb], suse & 1u, abort_flag);
                if (!ok) break;
                ++ucount;
                const uint32_t bu_lo = b_lo + ((sb * 2 * seed_region) >> 4), half_lo = seed_region >> 4;
                const int nt = wk.run();
                for (int t = 0; t < nt && ok; ++t, ++kit) {
                    if (dual && (kit & 1u) != (uint32_t)warp - 1u) continue;
                    const int st = kit % kStages;
                    const uint32_t buf = kit & buf_mask, use = kit >> buf_shift;
                    ok = mbar_wait<true>(&bar.k_full[st], (kit / kStages) & 1u, abort_flag);
                    if (!ok) break;
                    ok = mbar_wait<true>(&bar.d_empty[buf], (use & 1u) ^ 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t kst_lo = k_lo + st * (kKStageBytes >> 4);
                    const uint32_t d_addr = tmem_base + buf * buf_cols;
                    tc_mma_lo<false>(d_addr, kst_lo, bu_lo, idesc);
#pragma unroll
                    for (int kk = 1; kk < 8; ++kk) {
                        const int kb = kk >> 2, ks = kk & 3;
                        if (kk >= n_ks) break;
                        tc_mma_lo<true>(d_addr, kst_lo + ((kb * kKRegionBytes + ks * 32) >> 4),
                                        bu_lo + kb * half_lo + ((ks * 32) >> 4), idesc);
                    }
                    tc_commit(&bar.d_full[buf]);
                    tc_commit(&bar.k_empty[st]);
                }
                wk.advance(nt);
                if (ok) tc_commit(&bar.b_empty[sb]);
            }
            if (!ok) {
                // contractions already issued may still be running: the TMEM they write is freed below, so give them
                // a bounded wait (a commit completes when everything this thread issued before it has)
                tc_commit(&bar.mma_drain[warp - 1]);
                for (uint32_t it = 0; it < 4096 && !mbar_try(&bar.mma_drain[warp - 1], 0u); ++it) {}
            }
        }
    } else if (warp >= kEpiWarp0) {
        // ================= epilogue =================
        const int ew = warp - kEpiWarp0;
        const int qd = ew & 3;                               // TMEM lane quadrant (== warp % 4)
        const uint32_t eg = (uint32_t)(ew >> 2) & buf_mask;   // buffer: tiles eg, eg + n_bufs, ...
        const int half = (ew >> 2) >> buf_shift;                 // 0: finishes the row; 1: the later seed columns only
        const uint32_t taddr = tmem_base + ((uint32_t)(32 * qd) << 16) + eg * buf_cols;
        const int my_row = 32 * qd + lane;                   // row of the tile this thread owns
        uint32_t kit = 0, ucount = 0;
        bool ok = true;
        while (wk.valid() && ok) {
            const UnitDesc& ud = desc[wk.u];
            const int u = wk.u;
            const int T = ud.T, P = ud.P;
            const int64_t tok_off = ud.tok_off;
            const int seed_base = ud.seed_base + c0;
            const int r = max(0, min(plan[u * 8 + CASK_PLAN_R], T - P));
            const int m_all = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
            const int m = MANY ? max(0, min(m_all - c0, chunk.width)) : m_all;
            // MANY: is this the launch that finishes the unit's rows?
            const bool last = !MANY || (m_all <= c0 + chunk.width && (m > 0 || c0 == 0));
            const int hi = T - r;
            const int a0 = P - (!SPLIT && sh.page_size ? P % sub_rows : 0);
            // shared buffers: the finishing group also computes the row norm, so it takes fewer seed columns
            const int mc = m << wpair;               // accumulator columns in use
            const int c_split = split == 2 ? min(mc, 32 * max(1, (((mc + 31) >> 5) - 2) / 2)) : mc;
            unsigned long long* mass_u = mass_fx + (size_t)u * (max_m + 1);
            const int tile0 = wk.tile_in_unit();
            const int nt = wk.run();
            // Does this group take a tile of the unit?  Only then it needs the table of inverse seed norms; it
            // builds its own copy (two values per thread) and meets on its own barrier, so the groups never
            // wait for one another between units.
            const int first = (int)((eg + (uint32_t)n_bufs - (kit & buf_mask)) & buf_mask);
            if (first >= nt) {
                kit += nt;
                wk.advance(nt);
                continue;
            }
            float* inv = tail->inv_nu[ew >> 2][ucount & 1u];
            int* srow = tail->seed_row[ew >> 2][ucount & 1u];
            {
                const int gt = (ew & 3) * 32 + lane;           // thread of the group
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c = gt + 128 * h;
                    const float nu = (c < m) ? seed_norm[seed_base + c] : 0.f;
                    inv[c] = nu > 0.f ? 1.f / nu : 0.f;
                    srow[c] = (c < m) ? seed_rows[seed_base + c] : 0;
                }
                mbar_arrive(&bar.inv_ready[ew >> 2]);
                ok = mbar_wait<true>(&bar.inv_ready[ew >> 2], ucount & 1u, abort_flag);
                if (!ok) break;
            }
            ++ucount;
            uint8_t kd_n = (uint8_t)CASK_KIND_RECENT;
            float s_n = 0.f, mi_n = 0.f, nj_n = 0.f;
            bool pre = false;
            unsigned long long lost = 0ull;                  // masses of the thread's rows that join no group, and rows of the warp that do
            int n_joined = 0;
            for (int t = first; t < nt && ok; t += n_bufs) {
                const uint32_t tile = kit + (uint32_t)t;
                const int st = tile % kStages;
                const uint32_t use = tile >> buf_shift;
                if (half == 1) {
                    // second group of a shared buffer: best seed among the columns [c_split, m)
                    ok = mbar_wait<true>(&bar.d_full[eg], use & 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    float best = -INFINITY, second = 0.f;
                    int best_u = -1;
                    if (wpair) best_seed<1>(taddr, inv, c_split, mc, best, best_u, second);
                    else best_seed<0>(taddr, inv, c_split, mc, best, best_u, second);
                    tc_fence_before();
                    tail->x_val[eg][use & 1u][my_row] = best;
                    tail->x_idx[eg][use & 1u][my_row] = best_u;
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&bar.d_empty[eg]);
                        mbar_arrive(&bar.x_full[eg]);
                    }
                    continue;
                }
                // The row's kind and score are used after the contraction.  They were requested during this
                // group's previous tile of the unit (a load issued here would still be waited for before the
                // norm: the cache is saturated by the key stream and a miss costs well over a thousand cycles);
                // only a group's first tile of a unit loads them directly.
                const int i = a0 + (tile0 + t) * kTileRows + my_row;
                const bool in_range = i >= P && i < hi;
                uint8_t kd = (uint8_t)CASK_KIND_RECENT;
                float s_c = 0.f, mi_c = 0.f, nj_c = 0.f;
                if (pre) {
                    kd = kd_n; s_c = s_n; mi_c = mi_n;
                    if (SPLIT) nj_c = nj_n;
                } else if (in_range && last) {
                    kd = kind[tok_off + i];
                    s_c = s[tok_off + i];
                    if (sh.mass_in) mi_c = sh.mass_in[tok_off + i];
                    if (SPLIT) nj_c = k_norm[tok_off + i];
                }
                // the same fields of this group's next tile of the unit, in flight during this tile (a row's kind
                // is read and written by the thread that owns the row only, so reading it early sees the same byte)
                pre = last && t + n_bufs < nt;
                float2 carried = make_float2(-INFINITY, -INFINITY);
                int carried_u = -1;
                if (MANY && c0 > 0 && in_range) {
                    carried = chunk.best[tok_off + i];
                    carried_u = chunk.best_u[tok_off + i];
                    // (a launch that gave up a wait has written nothing here: what the workspace held before it is no seed)
                    if ((unsigned)carried_u >= (unsigned)c0) {
                        carried = make_float2(-INFINITY, -INFINITY);
                        carried_u = -1;
                    }
                }
                kd_n = (uint8_t)CASK_KIND_RECENT; s_n = 0.f; mi_n = 0.f;
                if (pre) {
                    const int in_ = i + n_bufs * kTileRows;
                    if (in_ >= P && in_ < hi) {
                        kd_n = kind[tok_off + in_];
                        s_n = s[tok_off + in_];
                        if (sh.mass_in) mi_n = sh.mass_in[tok_off + in_];
                        if (SPLIT) nj_n = k_norm[tok_off + in_];
                    }
                }
                // squared norm of this thread's row, read from the staged tile (any order of the
                // sixteen 16-byte pieces of the row gives the same set of elements)
                uint64_t n2p = 0ull;
                if (!SPLIT) {
                    ok = mbar_wait<true>(&bar.k_full[st], (tile / kStages) & 1u, abort_flag);
                    if (!ok) break;
                }
                if (!SPLIT && last) {
                    const uint8_t* base = k_smem + st * kKStageBytes + my_row * 128;
                    if (!sh.chan_w) n2p = row_norm2<false, FULL>(base, lane, my_row, tail->w, n_kb);
                    else n2p = row_norm2<true, FULL>(base, lane, my_row, tail->w, n_kb);
                }
                float n2, n2b;
                unpack2(n2p, n2, n2b);
                n2 += n2b;
                __syncwarp();
                if (!SPLIT && lane == 0) mbar_arrive(&bar.k_empty[st]);
                ok = mbar_wait<true>(&bar.d_full[eg], use & 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
                float best = -INFINITY, second = -INFINITY;
                int best_u = -1;
                // Few rows join where tau is high: their seeds are looked for afterwards.  Where most join, that is a second way through all chunks:
                // kernel of 112 units of 8,448 rows of which all join 73 us, searched in every chunk 67; 240 of 2,256 43.5 and 41.5.  How many join
                // depends on the cache as well, but every way to go by that costs more where few do than it gives back: 288 units of 33,280 rows
                // with 96 and 64 seeds 424 and 392 us by tau alone, by the joiners of the warp's tile before 442 and 414 (the flag in a register, in
                // shared memory 462 and 417), by those of the unit so far 455 and 408.
                const bool late = !SPLIT && !MANY && dual && !wpair && tau >= 0.5f;
                int best_chunk = 0;
                if (late) best_value(taddr, inv, mc, best, best_chunk);
                else if (!SPLIT && wpair) best_seed<1>(taddr, inv, 0, c_split, best, best_u, second);
                else best_seed<0, SPLIT || MANY>(taddr, inv, 0, c_split, best, best_u, second);
                if (MANY) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.d_empty[eg]);
                    if (best_u >= 0) best_u += c0;
                    second = fmaxf(fmaxf(second, carried.y), fminf(best, carried.x));
                    if (!(best > carried.x)) { best = carried.x; best_u = carried_u; }       // (the first seed among equals)
                    if (!last) {
                        if (in_range && m > 0) {
                            chunk.best[tok_off + i] = make_float2(best, second);
                            chunk.best_u[tok_off + i] = best_u;
                        }
                        continue;
                    }
                }
                if (MANY && n2 == 0.f && m_all > 0) { best = 0.f; best_u = 0; }        // a row of zeros: cosine 0 with every seed, nothing to tell apart
                bool cand = in_range && (late ? best > -INFINITY : best_u >= 0) && kd == CASK_KIND_DROPPED;
                if (MANY) {
                    // (a row that certainly stays below tau goes to no seed, whichever is the nearest)
                    const float nj = sqrtf(n2), at_tau = tau * nj, by = kCloseTau * nj;
                    const bool unsure = in_range && m_all > 0 && n2 != 0.f && kd == CASK_KIND_DROPPED &&
                                        !(best_u >= 0 && (best < at_tau - by || (best > at_tau + by && second < best - kCloseSeeds * nj)));
                    const unsigned ub = __ballot_sync(0xffffffffu, unsure);
                    if (ub) {
                        int at = 0;
                        if (lane == 0) at = atomicAdd(chunk.n_close, __popc(ub));
                        at = __shfl_sync(0xffffffffu, at, 0) + __popc(ub & ((1u << lane) - 1u));
                        if (unsure) {
                            chunk.close[at] = (int)(tok_off + i);
                            kind[tok_off + i] = kKindClose;
                        }
                    }
                    cand = cand && !unsure;
                }
                uint32_t close[4] = {0u, 0u, 0u, 0u};            // SPLIT: the plain cosines decide between these seeds
                const float least = best - kClose * nj_c;
                const bool plain = SPLIT && cand && nj_c > 0.f && (second >= least || fabsf(best - tau * nj_c) <= kClose * nj_c);
                if (SPLIT && __any_sync(0xffffffffu, plain)) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        if (32 * b >= m) break;
                        float v[32];
                        tc_ld32(taddr + 32 * b, v);
                        tc_wait_ld_regs(v);
#pragma unroll
                        for (int x = 0; x < 32; x += 4) {
                            const uint4 q = lds128(smem_u32(inv) + (uint32_t)(32 * b + x) * 4u);
                            if (v[x] * __uint_as_float(q.x) >= least) close[b] |= 1u << x;
                            if (v[x + 1] * __uint_as_float(q.y) >= least) close[b] |= 2u << x;
                            if (v[x + 2] * __uint_as_float(q.z) >= least) close[b] |= 4u << x;
                            if (v[x + 3] * __uint_as_float(q.w) >= least) close[b] |= 8u << x;
                        }
                        if (m < 32 * b + 32) close[b] &= (1u << (m - 32 * b)) - 1u;
                    }
                }
                float sm_ = 0.f;
                if (late) {
                    const float nj = sqrtf(n2);
                    sm_ = cand && nj > 0.f ? best / nj : 0.f;
                    best_u = find_seed(taddr, inv, mc, cand && sm_ >= tau, best, best_chunk);
                }
                if (!MANY) tc_fence_before();
                if (!MANY && split == 2) {
                    // The other group's candidate has the larger seed indices, so it wins only when strictly
                    // better: the same outcome as one scan over all columns.  The buffer is released after this
                    // read, so the other group cannot start the buffer's next use (and overwrite its hand-over
                    // slot or run a barrier phase ahead) before it.
                    ok = mbar_wait<true>(&bar.x_full[eg], use & 1u, abort_flag);
                    if (!ok) break;
                    const float ov = tail->x_val[eg][use & 1u][my_row];
                    if (ov > best) {
                        best = ov;
                        best_u = tail->x_idx[eg][use & 1u][my_row];
                    }
                }
                if (!MANY) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar.d_empty[eg]);
                }

                if (cand) {
                    const float nj = SPLIT ? nj_c : sqrtf(n2);              // best = <k_row, k_seed> / |k_seed| (0 for a zero seed)
                    if (!late) sm_ = nj > 0.f ? best / nj : 0.f;
                    if (SPLIT && plain) best_u = plain_best(K, sh, ud, i, srow, seed_norm + seed_base, close, sm_);
                    if (sim) sim[tok_off + i] = sm_;
                }
                const bool joined = cand && sm_ >= tau;
                float sc = 0.f;                                   // a_i = score + eps (+ the mass it carries)
                if (in_range) { const float a = s_c + eps; sc = sh.mass_in ? a + mi_c : a; }
                const unsigned long long fx = cand ? mass_to_fx(sc) : 0ull;
                if (joined) {
                    const int bu = CASK_IDX(best_u, m_all, err);
                    kind[tok_off + i] = CASK_KIND_MERGED;
                    seed_of[tok_off + i] = MANY ? seed_rows[ud.seed_base + bu] : srow[bu];
                    grp[tok_off + i] = bu;
                    atomicAdd(&mass_u[bu], fx);
                }
                // Joiner count and lost mass go out once per warp and unit: the fixed-point sums are exact, so
                // the grouping of the additions does not show in the result.
                const unsigned jb = __ballot_sync(0xffffffffu, joined);
                if (jb && mem_row) {                              // (few: the compaction takes them from this list)
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&njoin[u], __popc(jb));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(jb & ((1u << lane) - 1u));
                    if (joined && at < T) {
                        mem_row[tok_off + at] = i;
                        mem_seed[tok_off + at] = best_u;
                    }
                }
                n_joined += __popc(jb);
                if (!joined) lost += fx;
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) lost += __shfl_xor_sync(0xffffffffu, lost, off);
            if (lane == 0) {
                if (n_joined && !mem_row) atomicAdd(&njoin[u], n_joined);
                if (lost) atomicAdd(&mass_u[max_m], lost);
            }
            kit += nt;
            wk.advance(nt);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && tail->abort) atomicOr(err, CASK_ST_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// MANY: the rows whose cosines with two seeds, or with one and tau, lie within what the sums of the tensor cores may be off.  A CTA a row, a
// thread every 256th seed; the additions are those of assign_simt_kernel.  Bound by latency: list, unit, row and seeds in series, and half of
// the time goes to the fetch of code that runs once, so a seed's row is read 64 bytes at a time (128, twice the code: event of 240
// units of 3,000 rows with 1,071 of them listed 847 us, so 835; 4 of 9,000, 51 listed, 233 and 227; 8 of 1,024, two listed, 78.9
// and 78.2).  16 units of 15,276 rows, 380 seeds: 44 us with a warp a row, 15 so.
// Caches whose rows repeat list many of them where tau lets them join: a copy of a seed is as near to a row as the seed.  A seed's row then is read
// once for eight (kCloseRows) rows of a unit, which stand side by side in the list, and if more than a quarter of all rows are listed
// they are taken tile by tile, four rows by four seeds a thread and 16 bytes of each from shared memory at a time, in parts of at most 80 channels.
// Kernels of the assignment in us, element by element in parts of 64 and so, in brackets the SIMT kernel that these shapes had before: 104 units of
// 27,000 rows drawn from 64 keys (tau -1, 270 seeds) 12,850 and 10,640 (12,020), 240 of 3,000 (0.3, 750) 5,630 and 5,160 (5,790), four of
// 9,000 615 and 529 (539), 104 of 7,000 at head_dim 72 2,100 and 1,745 (1,776), at 96 2,630 and 2,210 (2,270).  The line: with a third to a half of
// the rows listed, eight at a time and by tiles, 104 of 7,000 at head_dim 72 2,310 and 1,790; with a sixth 104 of 27,000 7,910 and 10,560.  Rows of
// zeros, whose cosine is 0 without a sum, are not listed: half of the rows 17.1 to 0.68 ms.
constexpr int kCloseThreads = 256, kCloseRows = 8, kClosePitch = 132;      // (pitch: 16-byte pieces, and no conflicts where four threads take a row)
struct CloseSmem {
    alignas(16) float row[kCloseRows][kClosePitch];
    float norm[kCloseRows];
    float best[kCloseRows][kCloseThreads / 32];
    int best_u[kCloseRows][kCloseThreads / 32];
};
constexpr int kCloseTile = 64, kClosePart = 80;      // rows and seeds of a tile; channels of it in shared memory at a time
struct CloseTile {
    float row[kCloseTile][kClosePart + 4], seed[kCloseTile][kClosePart + 4], norm[kCloseTile];      // (16-byte pieces without conflicts)
};

// The greatest of `width` lanes, the first seed among equals.
__device__ __forceinline__ void close_fold(float& b, int& bu, int width) {
    for (int off = width / 2; off >= 1; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, b, off);
        const int ou = __shfl_xor_sync(0xffffffffu, bu, off);
        if (ou >= 0 && (ob > b || (ob == b && ou < bu) || bu < 0)) { b = ob; bu = ou; }
    }
}
// Greatest cosine (the first seed among equals) of the R rows in shared memory, to best[.][0] and best_u[.][0].
template <int R>
__device__ __forceinline__ void close_best(CloseSmem& sm, const __nv_bfloat16* __restrict__ seed_k, const float* __restrict__ seed_norm, int seed_base, int m, int d) {
    const int tid = threadIdx.x, lane = tid & 31;
    if (R > 1) {
        if (tid < 4 * R) {
            float n2 = 0.f;
            for (int c = tid & 3; c < d; c += 4) n2 = fmaf(sm.row[tid >> 2][c], sm.row[tid >> 2][c], n2);
            n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
            n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
            if ((tid & 3) == 0) sm.norm[tid >> 2] = sqrtf(n2);
        }
        __syncthreads();
    }
    float best[R];
    int best_u[R];
#pragma unroll
    for (int r = 0; r < R; ++r) { best[r] = -INFINITY; best_u[r] = -1; }
    for (int j = tid; j < m; j += kCloseThreads) {
        const uint4* seed = reinterpret_cast<const uint4*>(seed_k + (size_t)(seed_base + j) * d);
        const float nu = seed_norm[seed_base + j];
        float acc[R], n2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0.f;
#pragma unroll(R == 1 ? 4 : 2)
        for (int c = 0; c < d / 8; ++c) {
            const uint4 v = seed[c];
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 r0 = *reinterpret_cast<const float4*>(&sm.row[r][8 * c]), r1 = *reinterpret_cast<const float4*>(&sm.row[r][8 * c + 4]);
                const float x[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
                for (int y = 0; y < 8; ++y) {
                    if (R == 1) n2[y & 3] = fmaf(x[y], x[y], n2[y & 3]);
                    acc[r] = fmaf(x[y], __uint_as_float(y & 1 ? w[y >> 1] & 0xFFFF0000u : w[y >> 1] << 16), acc[r]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float nj = R == 1 ? sqrtf((n2[0] + n2[1]) + (n2[2] + n2[3])) : sm.norm[r];
            const float v = nj > 0.f && nu > 0.f ? acc[r] / (nj * nu) : 0.f;
            if (v > best[r]) { best[r] = v; best_u[r] = j; }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        close_fold(best[r], best_u[r], 32);
        if (lane == 0) { sm.best[r][tid >> 5] = best[r]; sm.best_u[r][tid >> 5] = best_u[r]; }
    }
    __syncthreads();
    if (tid >= 32) return;
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
        float b = sm.best[r][lane & (kCloseThreads / 32 - 1)];
        int bu = sm.best_u[r][lane & (kCloseThreads / 32 - 1)];
        close_fold(b, bu, kCloseThreads / 32);
        if (lane == 0) { sm.best[r][0] = b; sm.best_u[r][0] = bu; }
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kCloseThreads, 4) assign_close_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const __nv_bfloat16* __restrict__ K, const float* __restrict__ s, const int32_t* __restrict__ plan,
    const int32_t* __restrict__ seed_rows, const __nv_bfloat16* __restrict__ seed_k, const float* __restrict__ seed_norm, uint8_t* __restrict__ kind,
    int32_t* __restrict__ seed_of, float* __restrict__ sim, int32_t* __restrict__ grp, unsigned long long* __restrict__ mass_fx,
    int32_t* __restrict__ njoin, int32_t* __restrict__ mem_row, int32_t* __restrict__ mem_seed, int max_m, float tau, float eps,
    const int32_t* __restrict__ close, const int32_t* __restrict__ n_close, int total_tiles, int sub_rows) {
    __shared__ union { CloseSmem list; CloseTile tile; } both;
    CloseSmem& sm = both.list;
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, n = *n_close, d = sh.d;
    auto finish = [&](const UnitDesc& ud, int u, int m, int i, float best, int best_u) {
        const int64_t at = ud.tok_off + i;
        if (sim) sim[at] = best;
        const unsigned long long fx = mass_to_fx(row_mass(sh, s, eps, at));
        const bool joined = best_u >= 0 && best >= tau;
        atomicAdd(&mass_fx[(size_t)u * (max_m + 1) + (joined ? best_u : max_m)], fx);
        kind[at] = joined ? CASK_KIND_MERGED : CASK_KIND_DROPPED;
        if (!joined) return;
        seed_of[at] = seed_rows[ud.seed_base + CASK_IDX(best_u, m, sh.err)];
        grp[at] = best_u;
        const int p = atomicAdd(&njoin[u], 1);
        if (mem_row && p < ud.T) {
            mem_row[ud.tok_off + p] = i;
            mem_seed[ud.tok_off + p] = best_u;
        }
    };
    if (n > total_tiles * (kTileRows / 4)) {
        // more than a quarter of all rows: tile by tile, as assign_simt_kernel goes
        CloseTile& sm = both.tile;
        const int ty = tid / 16, tx = tid % 16, n_parts = (d + kClosePart - 1) / kClosePart, part = (d / 8 + n_parts - 1) / n_parts * 8;
        for (int w = blockIdx.x; w < total_tiles * (kTileRows / kCloseTile); w += gridDim.x) {
            const int g = w / (kTileRows / kCloseTile);
            const int u = warp_find_unit(sh.n_units, g, [&](int v) { return desc[v].atile0; });
            const UnitDesc& ud = desc[u];
            const int P = ud.P, m = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M])), hi = ud.T - max(0, min(plan[u * 8 + CASK_PLAN_R], ud.T - P));
            const int lo = P - (sh.page_size ? P % sub_rows : 0) + (g - ud.atile0) * kTileRows + w % (kTileRows / kCloseTile) * kCloseTile;
            auto listed = [&](int r) { return lo + r >= P && lo + r < hi && kind[ud.tok_off + lo + r] == kKindClose; };
            if (!__syncthreads_or(tid < kCloseTile && listed(tid))) continue;
            auto clamped = [&](int r) { return row_elem_off(sh, ud, ud.k_off, max(0, min(lo + r, ud.T - 1))); };
            {
                const __nv_bfloat16* k = K + clamped(tid / 4);
                float n2 = 0.f;
                for (int c = tid & 3; c < d; c += 4) n2 = fmaf(__bfloat162float(k[c]), __bfloat162float(k[c]), n2);
                n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
                n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
                if ((tid & 3) == 0) sm.norm[tid / 4] = sqrtf(n2);
            }
            float best[4];
            int best_u[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) { best[a] = -INFINITY; best_u[a] = -1; }
            for (int u0 = 0; u0 < m; u0 += kCloseTile) {
                float acc[4][4] = {};
                for (int c0 = 0; c0 < d; c0 += part) {
                    const int vecs = min(part, d - c0) / 8;
                    __syncthreads();
                    for (int e = tid; e < 2 * kCloseTile * vecs; e += kCloseThreads) {
                        const int r = e / vecs % kCloseTile, c = e % vecs * 8;
                        const bool of_row = e < kCloseTile * vecs;
                        const uint4 v = *reinterpret_cast<const uint4*>((of_row ? K + clamped(r) : seed_k + (size_t)(ud.seed_base + min(u0 + r, m - 1)) * d) + c0 + c);
                        float4* to = reinterpret_cast<float4*>((of_row ? sm.row[r] : sm.seed[r]) + c);
                        to[0] = make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
                        to[1] = make_float4(__uint_as_float(v.z << 16), __uint_as_float(v.z & 0xFFFF0000u), __uint_as_float(v.w << 16), __uint_as_float(v.w & 0xFFFF0000u));
                    }
                    __syncthreads();
#pragma unroll 1
                    for (int c = 0; c < 8 * vecs; c += 4) {
                        float4 x[4];
#pragma unroll
                        for (int a = 0; a < 4; ++a) x[a] = *reinterpret_cast<const float4*>(&sm.row[ty + 16 * a][c]);
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const float4 y = *reinterpret_cast<const float4*>(&sm.seed[tx + 16 * b][c]);
#pragma unroll
                            for (int a = 0; a < 4; ++a) acc[a][b] = fmaf(x[a].w, y.w, fmaf(x[a].z, y.z, fmaf(x[a].y, y.y, fmaf(x[a].x, y.x, acc[a][b]))));
                        }
                    }
                }
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int j = u0 + tx + 16 * b;
                    if (j >= m) continue;
                    const float nu = seed_norm[ud.seed_base + j];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const float nj = sm.norm[ty + 16 * a];
                        const float v = nj > 0.f && nu > 0.f ? acc[a][b] / (nj * nu) : 0.f;
                        if (v > best[a]) { best[a] = v; best_u[a] = j; }
                    }
                }
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                close_fold(best[a], best_u[a], 16);
                if (tx == 0 && listed(ty + 16 * a)) finish(ud, u, m, lo + ty + 16 * a, best[a], best_u[a]);
            }
            __syncthreads();
        }
        return;
    }
    const int step = n > kCloseRows * (int)gridDim.x ? kCloseRows : 1;
    int run = 0;
    for (int x0 = blockIdx.x * step, x = x0; x0 < n; x += run) {
        const int end = min(n, x0 + step);
        if (x >= end) {
            x0 += gridDim.x * step;
            x = x0;
            run = 0;
            continue;
        }
        // the rows of the first one's unit
        const UnitDesc& last_unit = desc[sh.n_units - 1];
        const int listed = CASK_IDX(close[min(x + (lane & (kCloseRows - 1)), end - 1)], (int)last_unit.tok_off + last_unit.T, sh.err);
        const int u = warp_find_unit(sh.n_units, __shfl_sync(0xffffffffu, listed, 0), [&](int v) { return (int)desc[v].tok_off; });
        const UnitDesc& ud = desc[u];
        const int tok_off = (int)ud.tok_off, T = ud.T, m = max(0, min(plan[u * 8 + CASK_PLAN_M], ud.plan[CASK_PLAN_M]));
        // (one at least, so that the loop goes on whatever the list holds)
        run = max(1, __ffs(~__ballot_sync(0xffffffffu, lane < kCloseRows && x + lane < end && listed >= tok_off && listed < tok_off + T)) - 1);
        __syncthreads();
        for (int e = tid; e < (run > 1 ? kCloseRows : 1) * 128; e += kCloseThreads) {
            const int r = e >> 7, c = e & 127;
            if (c < d) sm.row[r][c] = r < run ? __bfloat162float(K[row_elem_off(sh, ud, ud.k_off, CASK_IDX(close[x + r] - tok_off, T, sh.err)) + c]) : 0.f;
        }
        __syncthreads();
        if (run > 1) close_best<kCloseRows>(sm, seed_k, seed_norm, ud.seed_base, m, d);
        else close_best<1>(sm, seed_k, seed_norm, ud.seed_base, m, d);
        if (tid < run) finish(ud, u, m, CASK_IDX(close[x + tid] - tok_off, T, sh.err), sm.best[tid][0], sm.best_u[tid][0]);
    }
}

}  // namespace

// Rows per TMA box of the key stream (see the scoring kernel): 128, one page piece, or 0 if unsupported.
int assign_tc_box_rows(const Shape& sh) {
    if (sh.page_size == 0) return kTileRows;
    if (sh.page_size % kTileRows == 0) return kTileRows;
    if (sh.page_size >= 8 && kTileRows % sh.page_size == 0) return sh.page_size;
    return 0;
}

bool assign_many(int dtype, bool weighted, int max_m, int64_t sum_T) {
    return dtype == CASK_DTYPE_BF16 && !weighted && max_m > 256 && sum_T < (int64_t)1 << 31;
}

bool assign_tc_supported(const Launch& L) {
    const Shape& sh = L.sh;
    const int cols = L.max_m << (sh.chan_w ? 1 : 0);      // a weighted seed takes two accumulator columns
    if (sh.d > 128 || (cols > 256 && !assign_many(sh.dtype, sh.chan_w != nullptr, L.max_m, L.sum_T)) || L.max_m < 1 || L.total_atiles < 1) return false;
    if (sh.dtype == CASK_DTYPE_FP32) return !sh.chan_w && L.max_m <= 128 && 3 * L.sum_T < (int64_t)1 << 31;
    if (sh.page_size) return assign_tc_box_rows(sh) != 0 && sh.n_pages * sh.page_size < ((int64_t)1 << 31);
    int64_t max_row = 0;
    for (int u = 0; u < sh.n_units; ++u) {
        const UnitDesc& d = L.hdesc[u];
        if (d.k_off % sh.row_stride != 0) return false;
        max_row = std::max<int64_t>(max_row, d.k_off / sh.row_stride + d.T);
    }
    return max_row < (int64_t)1 << 31;
}

cudaError_t launch_assign_tc(const Launch& L, const cask_params& prm, const float* s, const int32_t* plan,
                             uint8_t* kind, int32_t* seed_of, float* sim, Workspace& ws, void* tmap_encode_fn) {
    const Shape& sh = L.sh;
    const bool split = sh.dtype == CASK_DTYPE_FP32;
    if (split) {
        cudaError_t e = launch_split_rows(L, ws, false);
        if (e != cudaSuccess) return e;
    }
    int64_t k_rows = split ? 3 * L.sum_T : sh.page_size ? sh.n_pages * sh.page_size : 0, sum_m = 0;
    for (int u = 0; u < sh.n_units; ++u) {
        if (!sh.page_size && !split) k_rows = std::max<int64_t>(k_rows, L.hdesc[u].k_off / sh.row_stride + L.hdesc[u].T);
        sum_m += L.hdesc[u].plan[CASK_PLAN_M];
    }
    const int sub_rows = split ? (int)L.sum_T : assign_tc_box_rows(sh);      // split: rows from one part to the next
    CUtensorMap tmK, tmSeed;
    if (!encode_rows_bf16(tmap_encode_fn, &tmK, split ? ws.k_split : L.k, (uint64_t)k_rows, sh.d,
                          (uint64_t)(split ? sh.d : sh.row_stride) * 2, split ? kTileRows : sub_rows))
        return cudaErrorInvalidValue;
    // the seed table has 256 spare rows behind the last seed, so a full box never leaves the allocation
    const int wpair = sh.chan_w ? 1 : 0;
    const bool many = (L.max_m << wpair) > 256;
    const int n_bufs = many || (L.max_m << wpair) <= 128 ? 4 : 2;      // accumulator buffers; four: seed boxes of 128 rows
    if (!encode_rows_bf16(tmap_encode_fn, &tmSeed, ws.seed_k, split ? 3 * ((uint64_t)sum_m + 256) : ((uint64_t)sum_m << wpair) + 256, sh.d, (uint64_t)sh.d * 2, n_bufs == 4 ? 128 : 256))
        return cudaErrorInvalidValue;
    const int grid = std::max(1, std::min(L.sms > 0 ? L.sms : 128, L.total_atiles));
    const bool full = sh.d > 112;
    auto kern = many ? (full ? assign_tc_kernel<true, false, true> : assign_tc_kernel<false, false, true>)
                : split ? (full ? assign_tc_kernel<true, true, false> : assign_tc_kernel<false, true, false>)
                        : (full ? assign_tc_kernel<true, false, false> : assign_tc_kernel<false, false, false>);
    cudaError_t e = allow_smem(L, many ? kSmemBitAssignMany + full : kSmemBitAssign + full + 2 * split, kern, kSmemBytesA);
    if (e != cudaSuccess) return e;
    // chunks of equal width, a multiple of the contraction's 16 columns
    const int n_chunks = many ? (L.max_m + 127) / 128 : 1;
    Chunk chunk{0, many ? ((L.max_m + n_chunks - 1) / n_chunks + 15) / 16 * 16 : 0, (float2*)ws.row_best, ws.row_best_u, ws.close, ws.err + 4};
    for (int k = 0; k < n_chunks; ++k, chunk.c0 += chunk.width) {
        Timed t(L, KID_ASSIGN);
        e = launch_dependent(L.stream, kern, grid, kThreadsA, kSmemBytesA, tmK, tmSeed, L.desc, sh, L.total_atiles, n_bufs, sub_rows,
                             wpair, (int)sum_m + 256, split ? (const float*)L.k : nullptr, ws.k_norm, s, plan, ws.seed_rows, ws.seed_norm, kind, seed_of, sim, ws.grp,
                             ws.mass_fx, ws.njoin, ws.slot_lists ? ws.mem_row : nullptr, ws.mem_slot, L.max_m, prm.tau, prm.eps, ws.err, chunk);
        if (e != cudaSuccess) return e;
    }
    if (!many) return e;
    // four CTAs an SM, which the shared memory that they ask for spreads over all of them (see spread_smem)
    const int close_grid = 4 * (L.sms > 0 ? L.sms : 128);
    size_t fixed = 0;
    e = allow_smem(L, kSmemBitAssignMany + 2, assign_close_kernel, kMaxSpread, &fixed);
    if (e != cudaSuccess) return e;
    Timed t(L, KID_ASSIGN);
    return launch_dependent(L.stream, assign_close_kernel, close_grid, kCloseThreads, spread_smem(L, close_grid, fixed, 0), L.desc, sh, (const __nv_bfloat16*)L.k, s, plan,
                            ws.seed_rows, (const __nv_bfloat16*)ws.seed_k, ws.seed_norm, kind, seed_of, sim, ws.grp, ws.mass_fx, ws.njoin,
                            ws.slot_lists ? ws.mem_row : nullptr, ws.mem_slot, L.max_m, prm.tau, prm.eps, ws.close, ws.err + 4, L.total_atiles, sub_rows);
}

}  // namespace cask
