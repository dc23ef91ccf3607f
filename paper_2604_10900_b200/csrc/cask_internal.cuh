// Internal declarations shared by the kernels and the C-ABI layer of libcask.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/cask.h"

namespace cask {

// Per-unit descriptor, built on the host for every call and uploaded to the
// head of the workspace.  Offsets are in elements of the cache dtype.
struct UnitDesc {
    int64_t k_off;
    int64_t v_off;
    int64_t q_off;
    int64_t tok_off;
    int32_t T, P, B, reserve;
    int32_t plan[8];
    int32_t chunk0;     // first score-partial chunk of this unit
    int32_t n_chunks;   // key chunks of this unit in the normaliser pass
    int32_t seed_base;  // first entry of this unit in the seed tables
    int32_t atile0;     // first 128-row scratch tile of this unit in the assignment pass
    int32_t n_atiles;   // scratch tiles of this unit: ceil((T - r - P)/128) when m > 0, else 0
    int32_t tile0;      // first 128-key tile of this unit in the unit-major tile sequence of the scoring passes
    int32_t bt0;        // paged cache: first entry of this unit in the block table
    int32_t pad;
};

struct Shape {
    int n_units, d, g, W, rows;   // rows = g*W
    int dtype;
    int64_t row_stride;
    int causal;
    // paged cache (page_size > 0): row i of a unit lives in physical page bt[bt0 + i / page_size]
    int page_size;
    int64_t n_pages;
    const int32_t* bt;   // device
    int32_t* err;        // device flag word (CASK_ST_TIMEOUT, CASK_ST_BOUNDS)
    const float* mass_in;   // device, optional [sumT]: group mass a row already carries
    const float* chan_w;    // device, optional [d]: channel weights of the merge similarity
    const float* band_w;    // device, optional [d/2]: band weights of the un-squared per-band distance (Sec. 2.5)
    int band_layout;        // 0: band f = channels (f, f + d/2); 1: channels (2f, 2f + 1)
    // host-resident caches: only the value rows the compaction reads are on the device, packed unit after unit
    // in ascending row order; v_pos[tok_off + i] is the position of row i inside its unit's run, v_base[u] the
    // first packed row of unit u (both NULL when V is the full cache)
    const int32_t* v_pos;
    const int64_t* v_base;
};

// Kernel ids for the optional per-kernel event timing.
enum KernelId {
    KID_SCORE_NORM = 0, KID_ROW_COMBINE, KID_SCORE_MASS, KID_PREFIX_EVICT, KID_SELECT_CORE, KID_SEEDS,
    KID_SEED_GATHER, KID_ASSIGN, KID_WEIGHTS, KID_SLOT_SCAN, KID_GATHER_MERGE, KID_DIAGNOSTICS, KID_SPLIT, KID_COUNT
};

// Records a CUDA event pair around every launch while switched on (defined in api.cu).
struct Profiler {
    bool on = false;
    void begin(int id, cudaStream_t st);
    void end(cudaStream_t st);
    void* impl = nullptr;
};

// Everything a launch needs, resolved by the API layer.
// Per-row outputs of an event that hold the same for every row that is not kept (kind == nullptr: nobody asks).  The tensor-core
// score pass writes them, a warp it has to spare in every CTA, under the exponentials; the selection kernel, with one CTA a unit,
// then writes the kept rows only.
struct RowDefaults {
    uint8_t* kind;       // CASK_KIND_DROPPED
    int32_t* seed_of;    // -1
    int32_t* assign;     // -1
    float* weight;       // 0
    float* sim;          // -2 (may be NULL)
};

struct Launch {
    cudaStream_t stream;
    Shape sh;
    const UnitDesc* desc;     // device
    const UnitDesc* hdesc;    // host copy (for grid sizing)
    const void* k;
    const void* v;
    const void* q;
    int max_T, max_m, max_chunks, total_chunks, total_atiles, max_P, max_B, total_tiles;
    int64_t sum_T;
    int64_t* launches;        // counter to bump
    Profiler* prof;
    void* tmap_encode;        // cuTensorMapEncodeTiled or nullptr
    int force_simt;
    int sms;                  // multiprocessors of the context's device (0: not known)
    RowDefaults fill;         // what the scoring call may write beside the scores
    struct SmemKept* smem;    // what this context has found out about its kernels' shared memory (NULL: nothing is kept)
};

// Kernels that a context has given their dynamic shared memory already, by their bits, and the static shared memory that the
// compiler gave each of them.
struct SmemKept {
    uint64_t allowed = 0;
    int fixed[64] = {};
};

// Lets a kernel use `bytes` of dynamic shared memory: once per context and kernel (`bit`, below 64, names the kernel).  *fixed: its
// static shared memory.
template <typename K>
inline cudaError_t allow_smem(const Launch& L, int bit, K kern, size_t bytes, size_t* fixed = nullptr) {
    if (L.smem && (L.smem->allowed >> bit) & 1) {
        if (fixed) *fixed = (size_t)L.smem->fixed[bit];
        return cudaSuccess;
    }
    cudaFuncAttributes attr{};
    cudaError_t e = cudaFuncGetAttributes(&attr, kern);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    if (fixed) *fixed = attr.sharedSizeBytes;
    if (L.smem) {
        L.smem->allowed |= (uint64_t)1 << bit;
        L.smem->fixed[bit] = (int)attr.sharedSizeBytes;
    }
    return cudaSuccess;
}
constexpr int kSmemBitScore = 0, kSmemBitAssign = 28, kSmemBitConsolidate = 32, kSmemBitCopy = 40, kSmemBitAssignMany = 60;   // first bit of each file's kernels

// Dynamic shared memory with which no more CTAs of a kernel share an SM than the grid needs (`need` bytes if that is more).
// CTAs that start while the kernel before them leaves go to the SMs that are free first, as many as fit: 288 CTAs of which
// three fit an SM ran on 97 of the 148.  (288 units of 640 rows, selection kernel: event 175 to 169 us; eight units of 33,280
// rows, compaction: 183 to 178.  Not for kernels beside the scoring passes: the row combine, padded so, cost an event of
// 3.6 ms 0.1 ms.)  `fixed`: the kernel's static shared memory, as allow_smem gives it.
constexpr size_t kMaxSpread = 116 << 10;             // the most that spreading asks for (one CTA per SM)
constexpr size_t kReserved = 1024;                   // what the system takes of the shared memory of every CTA
inline size_t spread_smem(const Launch& L, int64_t grid, size_t fixed, size_t need) {
    const int64_t per_sm = (grid + L.sms - 1) / std::max(L.sms, 1);
    if (L.sms < 1 || per_sm > 7) return need;
    constexpr size_t kSm = 228 << 10;
    const size_t least = kSm / (size_t)(per_sm + 1) + 256;           // per CTA: one more than per_sm does not fit
    return std::max(need, least > fixed + kReserved ? (least - fixed - kReserved + 127) / 128 * 128 : 0);
}

// Kernels of a call follow one another by programmatic dependent launch: a kernel launched with launch_dependent() may start
// while the one before it still runs, sets itself up (barriers, TMEM, descriptors of the operands) and calls pdl_wait() before
// it touches anything that kernel wrote.  pdl_wait() returns when every kernel before has completed, and only then lets the
// next one start, so that at most two kernels of a call are on the device.  (The order of the two is relied upon: the score pass, started
// under the normaliser pass, reads what was complete when that pass came back from its wait without waiting itself.)  Together with the descriptors' upload by a kernel
// (upload.cu): events on 8 units of 640 rows 85.5 to 73.1 us, 128 units of 4,608 rows at head_dim 64 230 to 219, 16 fp32 units
// of 8,448 rows 331 to 307, events of milliseconds unchanged.
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool early, cudaStream_t stream, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_dependent(cudaStream_t stream, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, A... args) {
    return launch_kernel(true, stream, kern, grid, block, smem, args...);
}

// Scope guard around one kernel launch: counts it and, in profiling mode, times it.
struct Timed {
    const Launch& L;
    Timed(const Launch& l, int id) : L(l) {
        ++*L.launches;
        if (L.prof && L.prof->on) L.prof->begin(id, L.stream);
    }
    ~Timed() {
        if (L.prof && L.prof->on) L.prof->end(L.stream);
    }
};

constexpr int kChunkKeys = 2048;    // keys per normaliser-pass chunk
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kNegBig = -1.0e30f;   // finite stand-in for -inf in running maxima

// ---- workspace carving ------------------------------------------------------
struct Workspace {
    UnitDesc* desc;
    float* s;            // [sumT]   scores when the caller keeps none
    float* rowm;         // [units*rows] row offset in log2 units
    float* roww;         // [units*rows] row weight 1/(rows * sum)
    float* part_m;       // [total_chunks*rows], or what score_tc_sizes says where that is more
    float* part_l;       // the same
    float* s_part;       // [row groups, sumT] partial scores (tensor-core scoring with more than 512 query rows)
    int32_t* seed_rows;  // [sum m]     seed cache rows, ascending per unit
    float* seed_norm;    // [sum m]
    void* seed_k;        // [sum m_pad, d] gathered seed keys (cache dtype, or three bf16 parts of sum m + 256 rows each)
    void* k_split;       // fp32 caches on the tensor cores: [3, sumT, d] bf16 parts of the keys
    void* q_split;       //   [3, units*rows, d] bf16 parts of the queries
    float* k_norm;       //   [sumT] norms of the key rows
    bool split_ready;    // this call has filled k_split and k_norm
    int32_t* grp;        // [sumT] seed slot (0..m) of a joined row, -1
    unsigned long long* mass_fx;  // [units*(max_m+1)] fixed-point group masses (+ lost mass)
    int32_t* njoin;      // [units]
    float* row_best;     // assignment to more than 256 seeds (assign_many): [sumT, 2] greatest and second greatest value of a row so far,
    int32_t* row_best_u; //   [sumT] the former's seed,
    int32_t* close;      //   [sumT] rows that the plain cosines decide
    int32_t* mem_row;    // [sumT] rows of kind 4/5 in ascending order; slot lists: the rows that joined (njoin), in any order
    int32_t* mem_slot;   // [sumT] slot each of them feeds; slot lists: the number of their seed
    int32_t* n_mem;      // [units]; slot lists: kept rows, -1: this unit has no lists
    int32_t* seed_slot;  // [units*max_B] slots of kind SEED, any order; slot lists: in the order of the seeds
    int32_t* n_seed;     // [units]
    bool filled;         // the scoring call has written Launch::fill
    bool slot_lists;     // the selection of this call has listed the slots, and the assignment kernel lists the rows that join
    int32_t max_B;
    int32_t* err;        // [8] flags (0, 1), clocks of the scoring passes (2, 3), entries of `close` (4)
    float* stats_a;      // [units, d] query-statistics scorer: head-pooled mu * kappa per band (re, im)
    size_t bytes;
};

// ---- kernels (defined in the .cu files) --------------------------------------
// Descriptors into the workspace, flag words cleared (upload.cu).  release: the kernel that follows may start beside this one (all but a
// long score pass with given normalisers, see launch_passes).
// *reads_staging: the kernel still reads `staged` (page-locked).
cudaError_t upload_descriptors(cudaStream_t stream, const UnitDesc* staged, int n, UnitDesc* dst, int32_t* err, bool release, bool* reads_staging);
cudaError_t launch_score_simt(const Launch& L, const float* lse_in, float* s, float* lse_out,
                              Workspace& ws);
cudaError_t launch_row_combine(const Launch& L, const float* lse_in, float* lse_out, Workspace& ws);
cudaError_t launch_prefix_evict(const Launch& L, const float* s, uint8_t* kind, int32_t* plan);
cudaError_t launch_select_core(const Launch& L, const float* s, const int32_t* plan, uint8_t* kind);
cudaError_t launch_consolidate(const Launch& L, const cask_params& prm, const float* s,
                               const int32_t* plan, uint8_t* kind, int32_t* seed_of, float* weight,
                               float* sim, int32_t* unit_status, float* lost_mass, Workspace& ws,
                               const cask_outputs* out = nullptr);
// out != nullptr ("fused", the event path only): `plan` and `kind` are still unwritten; one kernel per unit then does the prefix eviction
// and the core and seed selection, and for units of at most kSmallUnitRows rows the seed gather as well.
constexpr int kSmallUnitRows = 1024;
// Longer units' rows get assign = -1 and weight = 0 there.
// Long units of which little is kept: the selection kernel lists the slots and the assignment kernel the rows that join, so that the
// compaction need not look at every row again, and the score pass writes what the dropped rows get (RowDefaults).  That moves
// work from the compaction's many CTAs to the one a unit has in the selection, so it pays only where the kept rows are few against
// the rows: event of eight units of 33,280 rows (1,024 kept) 172.8 to 163.1 us, selection and compaction of 288 of them (512)
// 134 to 103 us, of 512 of 4,700 to 33,000 (512) 218 to 182.  At 16 rows a slot it is even (112 of 8,448, 512 kept: 52 and 50);
// with nine (4,608, 512 kept) the event is 3 % slower, with six and a half (13,312, 2,048 kept) 2 %.
constexpr int kMaxListRows = 61440;                      // two bits a row in the selection's shared memory, 48 KB in all
inline bool want_slot_lists(const Launch& L) {
    return L.max_T > kSmallUnitRows && L.max_T <= kMaxListRows && L.max_T >= 16 * std::max(L.max_B, 1);
}
// ev != nullptr (the event path, after a fused launch_consolidate): the compaction also writes the merge weights, the status words
// and the lost mass, which the fused consolidation left out, and ORs late device flags into the status words.
struct EventFusion {
    const int32_t* plan;
    int32_t* unit_status;
    float* lost_mass;
};
cudaError_t launch_compact(const Launch& L, const cask_params& prm, const float* s, const uint8_t* kind,
                           const int32_t* seed_of, float* weight, const cask_outputs& out, Workspace& ws,
                           const EventFusion* ev = nullptr);
// Host-resident caches: rank of every row among the rows of its unit whose values the compaction reads
// (kind != 0), the number of such rows per unit and the exclusive prefix of those numbers.
cudaError_t launch_value_ranks(const Launch& L, const uint8_t* kind, int32_t* v_pos, int32_t* n_need, int64_t* v_base);
// Page-locked values: a kernel reads the rows with v_pos >= 0 from host memory and packs them behind one another.
cudaError_t launch_value_gather(const Launch& L, const void* v_host, void* v_packed, const int32_t* v_pos,
                                const int64_t* v_base);
// Paged cache: copies the compacted rows into the unit's own pages (slot t -> logical row t).
cudaError_t launch_writeback(const Launch& L, const cask_outputs& out, void* k_pool, void* v_pool);
// rho_core / rho_rep and the within-group dispersion of Sec. 2.6 per unit (any of the pointers may be NULL).
cudaError_t launch_diagnostics(const Launch& L, const cask_params& prm, const float* s, const uint8_t* kind,
                               const cask_outputs& out);

// Tensor-core assignment of scratch rows to seeds (cosine Gram + argmax), same outputs as the SIMT kernel.
bool assign_many(int dtype, bool weighted, int max_m, int64_t sum_T);      // seeds in chunks (they need row_best and the like)
bool assign_tc_supported(const Launch& L);      // fp32 caches: through their bf16 parts
int assign_tc_box_rows(const Shape& sh);   // rows per TMA box of the key stream, 0 if the page size does not fit
cudaError_t launch_assign_tc(const Launch& L, const cask_params& prm, const float* s, const int32_t* plan,
                             uint8_t* kind, int32_t* seed_of, float* sim, Workspace& ws, void* tmap_encode_fn);

// Query-statistics scorer (App. B): horizon kernel and horizon-averaged mean score, one pass over the keys.
cudaError_t launch_score_stats(const Launch& L, const cask_query_stats& qs, float* s, Workspace& ws);

// fp32 rows as three bf16 parts (split.cu): bytes the parts take, and the kernel (keys unless this call has split them before).
struct SplitSizes {
    size_t k_bytes, q_bytes, norm_bytes;
};
SplitSizes split_sizes(int dtype, int d, int64_t sum_T, int64_t q_rows);
cudaError_t launch_split_rows(const Launch& L, Workspace& ws, bool queries);

// Tensor-core scoring (tcgen05 + TMA); returns cudaErrorNotSupported when the shape does not fit.
bool score_tc_supported(const Launch& L);
// Does the score pass of a batch with given normalisers have so many tiles a CTA that it should find the SMs empty (see launch_passes)?
bool given_score_long(int dtype, int d, int rows, int total_tiles, int sms);
struct ScoreTcSizes {
    size_t part_floats;      // floats per normaliser-partial table
    size_t s_parts;          // partial scores per cache row (0: the score pass writes the scores themselves)
};
ScoreTcSizes score_tc_sizes(int dtype, int d, int rows, int n_units);
cudaError_t launch_score_tc(const Launch& L, const float* lse_in, float* s, float* lse_out,
                            Workspace& ws, void* tmap_encode_fn);

// Last unit u in [0, n) with key(u) <= t (key ascends, key(0) <= t): 32 probes a round, so a few cache latencies whatever n
// is.  All lanes of the warp call it.
template <typename F>
__device__ __forceinline__ int warp_find_unit(int n, int t, F key) {
    const int lane = threadIdx.x & 31;
    int lo = 0, len = n;
    while (len > 1) {
        const int step = (len + 31) / 32, at = lo + lane * step;
        const unsigned hit = __ballot_sync(0xffffffffu, at < lo + len && key(at) <= t);
        const int k = hit ? 31 - __clz(hit) : 0;
        len = min(step, len - k * step);
        lo += k * step;
    }
    return lo;
}

// ---- small device helpers ------------------------------------------------------
// Physical row (in units of rows of the K/V arrays) of logical row i of a unit in a paged cache.  A
// page id outside the pool raises CASK_ST_BOUNDS and is replaced by page 0, so nothing is read out
// of bounds.
__device__ __forceinline__ int64_t page_row(const Shape& sh, int32_t pg, int in_page) {
    if ((uint64_t)(int64_t)pg >= (uint64_t)sh.n_pages) {
        atomicOr(sh.err, CASK_ST_BOUNDS);
        pg = 0;
    }
    return (int64_t)pg * sh.page_size + in_page;
}
__device__ __forceinline__ int64_t paged_row(const Shape& sh, int bt0, int i) {
    return page_row(sh, sh.bt[bt0 + i / sh.page_size], i % sh.page_size);
}
__device__ __forceinline__ int64_t paged_row(const Shape& sh, const UnitDesc& ud, int i) { return paged_row(sh, ud.bt0, i); }
// Merge weight a_i of the row at per-row index idx (Sec. 2.4): score + eps, plus the mass it already carries.
__device__ __forceinline__ float row_mass(const Shape& sh, const float* __restrict__ s, float eps, int64_t idx) {
    const float a = s[idx] + eps;
    return sh.mass_in ? a + sh.mass_in[idx] : a;
}
// Element offset of logical row i of a unit in the K (unit_off = k_off) or V (v_off) array.
__device__ __forceinline__ int64_t row_elem_off(const Shape& sh, const UnitDesc& ud, int64_t unit_off, int i) {
    if (sh.page_size == 0) return unit_off + (int64_t)i * sh.row_stride;
    return paged_row(sh, ud, i) * sh.row_stride;
}
// Element offset of the value row i of unit u.
__device__ __forceinline__ int64_t v_elem_off(const Shape& sh, const UnitDesc& ud, int u, int i) {
    if (sh.v_pos) return (sh.v_base[u] + sh.v_pos[ud.tok_off + i]) * (int64_t)sh.d;
    return row_elem_off(sh, ud, ud.v_off, i);
}

// Self-checking build (-DCASK_BOUNDS, libcask_bounds.so): every index the kernels take from an array that they or an
// earlier kernel wrote (seed rows, member rows, slots, seed numbers) is checked against its range before it addresses
// memory.  A bad one raises CASK_ST_BOUNDS in the call's flag word and is replaced by 0, so nothing is read or written
// out of bounds and nothing traps.  The ordinary build compiles the checks out.
#ifdef CASK_BOUNDS
__device__ __forceinline__ int checked_index(int i, int n, int32_t* err) {
    if ((unsigned)i >= (unsigned)n) {
        atomicOr(err, CASK_ST_BOUNDS);
        return 0;
    }
    return i;
}
#define CASK_IDX(i, n, err) ::cask::checked_index((i), (n), (err))
#else
#define CASK_IDX(i, n, err) (i)
#endif

template <typename T> struct Elem;
template <> struct Elem<float> {
    static __device__ __forceinline__ float ld(const float* p) { return *p; }
    static __device__ __forceinline__ void st(float* p, float x) { *p = x; }
};
template <> struct Elem<__nv_bfloat16> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }
};

// x = h + m + l, exactly (see split.cu).  A finite x that rounds to infinity (above bf16's greatest number) is rounded towards zero.
__device__ __forceinline__ void split3(float x, __nv_bfloat16& h, __nv_bfloat16& m, __nv_bfloat16& l) {
    h = __float2bfloat16_rn(x);
    if (__hisinf(h)) h = __float2bfloat16_rz(x);
    const float r = x - __bfloat162float(h);
    m = __float2bfloat16_rn(r);
    l = __float2bfloat16_rn(r - __bfloat162float(m));
}

// How the gathered seed keys are laid out: as they are, with the channel weights as hi/lo rows of the cache dtype, or as
// three bf16 parts that are part_rows rows apart.
enum SeedLayout { SEED_PLAIN = 0, SEED_PAIR = 1, SEED_SPLIT = 3 };

// order-preserving map float -> uint32 (greater float <=> greater key)
__device__ __forceinline__ uint32_t order_key(float x) {
    uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// fixed-point image of a mass a in [0, 2^20): 2^43 steps per unit
constexpr double kMassScale = 8796093022208.0;   // 2^43
__device__ __forceinline__ unsigned long long mass_to_fx(float a) {
    return (unsigned long long)__float2ll_rn(a * (float)kMassScale);      // (a power of two: the product is exact in fp32 too)
}
__device__ __forceinline__ float fx_to_mass(unsigned long long f) {
    return (float)((double)f / kMassScale);
}

}  // namespace cask
