// Compaction to the budget (Sec. 2.3: |R| <= B) with the weighted K/V merge of Sec. 2.4:
//   slot order = ascending anchor row; kinds 1..3 and lone seeds are byte copies;
//   a seed with joiners holds sum_i w_i k_i, sum_i w_i v_i (members in ascending row order).
#include <type_traits>

#include "tc_common.cuh"

namespace cask {

namespace {

// On the event path the scan also does what weights_kernel does in the staged consolidation call (merge weights
// w_i = a_i / m_G of the rows of kind 4/5, the unit's status word and lost mass): same formulas, same bits, one
// launch fewer.  s == nullptr: not fused, the weights are already there.
struct FusedWeights {
    const float* s;
    const int32_t* grp;
    const unsigned long long* mass_fx;
    const int32_t* njoin;
    const int32_t* plan;
    int32_t* unit_status;
    float* lost_mass;
    const int32_t* err;
    Shape sh;
    int max_m;
    float eps;
};

constexpr int kScanThreads = 1024;
constexpr int kScanMaxIters = 63;      // rows per unit below 64,512: the one-scan path of slot_scan_kernel

// ==== scan, copy and merge as kernels of their own: units above kLongMaxRows rows and budgets above kLongMaxSlots ================
// ---- 1. per-unit ordered scan: slots, index map, member list -------------------------------
__global__ void __launch_bounds__(kScanThreads) slot_scan_kernel(
    const UnitDesc* __restrict__ desc, const uint8_t* __restrict__ kind, const int32_t* __restrict__ seed_of,
    float* __restrict__ weight, int Bmax, int32_t* __restrict__ n_out, int32_t* __restrict__ slot_src,
    uint8_t* __restrict__ slot_kind, float* __restrict__ slot_mass, int32_t* __restrict__ assign,
    int32_t* __restrict__ mem_row, int32_t* __restrict__ mem_slot, int32_t* __restrict__ n_mem,
    int32_t* __restrict__ seed_slot, int32_t* __restrict__ n_seed, int max_B, FusedWeights fw,
    int32_t* __restrict__ err) {
    __shared__ unsigned wk[kScanThreads / 32], wm[kScanThreads / 32];
    __shared__ unsigned cell[kScanMaxIters * (kScanThreads / 32)];
    __shared__ int seeds_listed;
    if (threadIdx.x == 0) seeds_listed = 0;
    pdl_wait();
    const int u = blockIdx.x;
    const UnitDesc& ud = desc[u];
    const int T = ud.T;
    const int64_t o = ud.tok_off;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned base_k = 0, base_m = 0;
    const int iters = (T + (int)blockDim.x - 1) / (int)blockDim.x;
    if (iters <= kScanMaxIters) {
        // Two coalesced sweeps around one scan: per (iteration, warp) cell the number of kept rows and of group
        // members, an exclusive scan over the cells in row order, then every row finds its slot from its cell's
        // base and the lower lanes of its warp.
        // (both sweeps read four rows' kinds a round, so that the loads are in flight together)
        const int cells = iters * nw;
        for (int it0 = 0; it0 < iters; it0 += 4) {
            uint8_t kd4[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = (it0 + q) * blockDim.x + threadIdx.x;
                kd4[q] = (it0 + q < iters && i < T) ? kind[o + i] : (uint8_t)0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (it0 + q >= iters) break;          // uniform over the block
                const uint8_t kd = kd4[q];
                const bool keep = kd >= CASK_KIND_PREFIX && kd <= CASK_KIND_SEED;
                const bool mem = kd == CASK_KIND_SEED || kd == CASK_KIND_MERGED;
                const unsigned bk = __ballot_sync(0xffffffffu, keep), bm = __ballot_sync(0xffffffffu, mem);
                if (lane == 0) cell[(it0 + q) * nw + w] = (unsigned)__popc(bk) | ((unsigned)__popc(bm) << 16);
            }
        }
        __syncthreads();
        // exclusive scan of the packed (kept, member) counts; a cell holds at most 32 of each and a unit fewer
        // than 65,536 kept rows and members in this path, so the halves never carry into each other
        {
            const int per = (cells + (int)blockDim.x - 1) / (int)blockDim.x;
            const int c0 = threadIdx.x * per, c1 = min(cells, c0 + per);
            unsigned sum = 0;
            for (int c = c0; c < c1; ++c) sum += cell[c];
            // block exclusive scan of `sum`
            unsigned incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                unsigned v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            if (lane == 31) wk[w] = incl;
            __syncthreads();
            unsigned wbase = 0;
            for (int x = 0; x < w; ++x) wbase += wk[x];
            unsigned run = wbase + incl - sum;
            unsigned total = 0;
            for (int x = 0; x < nw; ++x) total += wk[x];
            __syncthreads();
            for (int c = c0; c < c1; ++c) {
                const unsigned v = cell[c];
                cell[c] = run;
                run += v;
            }
            base_k = total & 0xFFFFu;
            base_m = total >> 16;
        }
        __syncthreads();
        for (int it0 = 0; it0 < iters; it0 += 4) {
            uint8_t kd4[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = (it0 + q) * blockDim.x + threadIdx.x;
                kd4[q] = (it0 + q < iters && i < T) ? kind[o + i] : (uint8_t)0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int it = it0 + q;
                if (it >= iters) break;                   // uniform over the block
                const int i = it * blockDim.x + threadIdx.x;
                const uint8_t kd = kd4[q];
                const bool keep = kd >= CASK_KIND_PREFIX && kd <= CASK_KIND_SEED;
                const bool mem = kd == CASK_KIND_SEED || kd == CASK_KIND_MERGED;
                const unsigned bk = __ballot_sync(0xffffffffu, keep), bm = __ballot_sync(0xffffffffu, mem);
                const unsigned cb = cell[it * nw + w];
                const unsigned below = (1u << lane) - 1u;
                if (i < T) {
                    int slot = -1;
                    if (keep) {
                        slot = (int)((cb & 0xFFFFu) + __popc(bk & below));
                        if (slot < Bmax) {
                            slot_src[(size_t)u * Bmax + slot] = i;
                            slot_kind[(size_t)u * Bmax + slot] = kd;
                        } else {
                            slot = -1;        // more kept rows than slots: cannot happen for a valid plan
                        }
                    }
                    assign[o + i] = slot;
                    if (mem) mem_row[o + (cb >> 16) + __popc(bm & below)] = i;
                    if (kd >= CASK_KIND_PREFIX && kd <= CASK_KIND_CORE) weight[o + i] = 1.f;
                    if (kd == CASK_KIND_DROPPED) weight[o + i] = 0.f;
                    if (fw.s && mem) {
                        const int gi = fw.grp[o + i];
                        if (gi >= 0 && gi < fw.max_m)
                            weight[o + i] = row_mass(fw.sh, fw.s, fw.eps, o + i) /
                                            fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + gi]);
                    }
                }
            }
        }
    } else {
    for (int i0 = 0; i0 < T; i0 += blockDim.x) {
            const int i = i0 + threadIdx.x;
            const uint8_t kd = (i < T) ? kind[o + i] : (uint8_t)0;
            const bool keep = kd >= CASK_KIND_PREFIX && kd <= CASK_KIND_SEED;
            const bool mem = kd == CASK_KIND_SEED || kd == CASK_KIND_MERGED;
            const unsigned bk = __ballot_sync(0xffffffffu, keep), bm = __ballot_sync(0xffffffffu, mem);
            __syncthreads();
            if (lane == 0) { wk[w] = __popc(bk); wm[w] = __popc(bm); }
            __syncthreads();
            unsigned pk = 0, pm = 0, ak = 0, am = 0;
            for (int x = 0; x < nw; ++x) {
                if (x < w) { pk += wk[x]; pm += wm[x]; }
                ak += wk[x];
                am += wm[x];
            }
            const unsigned below = (1u << lane) - 1u;
            if (i < T) {
                int slot = -1;
                if (keep) {
                    slot = (int)(base_k + pk + __popc(bk & below));
                    if (slot < Bmax) {
                        slot_src[(size_t)u * Bmax + slot] = i;
                        slot_kind[(size_t)u * Bmax + slot] = kd;
                    } else {
                        slot = -1;        // more kept rows than slots: cannot happen for a valid plan
                    }
                }
                assign[o + i] = slot;
                if (mem) mem_row[o + base_m + pm + __popc(bm & below)] = i;
                if (kd >= CASK_KIND_PREFIX && kd <= CASK_KIND_CORE) weight[o + i] = 1.f;
                if (kd == CASK_KIND_DROPPED) weight[o + i] = 0.f;
                if (fw.s && mem) {
                    const int gi = fw.grp[o + i];
                    if (gi >= 0 && gi < fw.max_m)
                        weight[o + i] = row_mass(fw.sh, fw.s, fw.eps, o + i) /
                                        fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + gi]);
                }
            }
            base_k += ak;
            base_m += am;
        }
    }
    const int nk = min((int)base_k, Bmax), nm = (int)base_m;
    if (threadIdx.x == 0) { n_out[u] = nk; n_mem[u] = nm; }
    if (fw.s && threadIdx.x == 0) {
        int fl = fw.plan[u * 8 + CASK_PLAN_FLAGS];
        if ((fl & CASK_ST_DECODE_CONSOLIDATED) && fw.njoin[u] == 0) fl |= CASK_ST_MERGE_INACTIVE;
        fw.unit_status[u] = fl | *fw.err;     // device-side flags of this call so far
        fw.lost_mass[u] = fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + fw.max_m]);
    }
    for (int t = nk + threadIdx.x; t < Bmax; t += blockDim.x) {
        slot_src[(size_t)u * Bmax + t] = -1;
        slot_kind[(size_t)u * Bmax + t] = 0;
        slot_mass[(size_t)u * Bmax + t] = 0.f;
    }
    __syncthreads();
    // the slots that hold a representative, for the merge kernel (any order)
    for (int t = threadIdx.x; t < nk; t += blockDim.x)
        if (slot_kind[(size_t)u * Bmax + t] == CASK_KIND_SEED) {
            const int at = atomicAdd(&seeds_listed, 1);
            if (at < max_B) seed_slot[(size_t)u * max_B + at] = t;
        }
    __syncthreads();
    if (threadIdx.x == 0) n_seed[u] = min(seeds_listed, max_B);
    // members point at their seed's slot
    for (int e = threadIdx.x; e < nm; e += blockDim.x) {
        const int i = CASK_IDX(mem_row[o + e], T, err);
        int slot = -1;
        if (kind[o + i] == CASK_KIND_SEED) {
            slot = assign[o + i];
        } else {
            const int sd = seed_of[o + i];
            if (sd >= 0 && sd < T && kind[o + sd] == CASK_KIND_SEED) slot = assign[o + sd];
            assign[o + i] = slot;
        }
        mem_slot[o + e] = slot;
    }
}

// ---- 2. byte copy of every slot's anchor row by bulk async copies through shared memory ----
// A warp owns batches of up to 32 consecutive slots of one unit.  Every lane starts the bulk copy of its slot's K
// and V row (row bytes each, any source row) into the warp's staging buffer; when the batch has landed (mbarrier,
// byte count) one lane writes it out with two bulk stores, because consecutive slots are contiguous in k_out and
// v_out.  Two staging buffers per warp, so the loads of a batch run under the stores of the one before.  No
// registers hold data, which leaves enough copies in flight to load HBM with units of a few hundred rows.
constexpr int kCopyWarps = 6;
constexpr int kCopyStageBytes = 16384;       // per warp and stage: K half + V half

struct CopyCtl {
    uint64_t bar[kCopyWarps][2];
    int abort;
};

template <typename T>
__global__ void __launch_bounds__(kCopyWarps * 32) slot_copy_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const T* __restrict__ K, const T* __restrict__ V,
    const float* __restrict__ s, float eps, int Bmax, int slots, const int32_t* __restrict__ n_out,
    const int32_t* __restrict__ slot_src, T* __restrict__ k_out, T* __restrict__ v_out,
    float* __restrict__ slot_mass) {
    using namespace tc;
    extern __shared__ __align__(128) uint8_t copy_smem[];
    __shared__ CopyCtl ctl;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t row_bytes = (uint32_t)(sh.d * sizeof(T));
    const int sb = min(32, (int)(kCopyStageBytes / 2 / row_bytes));     // slots per batch
    if (threadIdx.x == 0) {
        for (int i = 0; i < kCopyWarps; ++i) { mbar_init(&ctl.bar[i][0], 1); mbar_init(&ctl.bar[i][1], 1); }
        ctl.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();
    volatile int* abort_flag = &ctl.abort;
    uint8_t* my = copy_smem + (size_t)w * 2 * kCopyStageBytes;
    const int bpu = (slots + sb - 1) / sb;                               // batches per unit
    const int64_t total = (int64_t)sh.n_units * bpu;
    uint32_t it = 0;
    bool ok = true;
    for (int64_t bi = (int64_t)blockIdx.x * kCopyWarps + w; bi < total && ok; bi += (int64_t)gridDim.x * kCopyWarps) {
        const int u = (int)(bi / bpu), t0 = (int)(bi - (int64_t)u * bpu) * sb;
        const int nv = min(sb, n_out[u] - t0);
        if (nv <= 0) continue;
        const UnitDesc& ud = desc[u];
        const uint32_t st = it & 1u;
        uint8_t* kbuf = my + st * kCopyStageBytes;
        uint8_t* vbuf = kbuf + kCopyStageBytes / 2;
        // the stores that read this buffer two batches ago must have read it
        if (lane == 0) {
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            mbar_expect_tx(&ctl.bar[w][st], (uint32_t)nv * 2u * row_bytes);
        }
        __syncwarp();
        if (lane < nv) {
            const int src = CASK_IDX(slot_src[(size_t)u * Bmax + t0 + lane], ud.T, sh.err);
            const T* kr = K + row_elem_off(sh, ud, ud.k_off, src);
            const T* vr = V + v_elem_off(sh, ud, u, src);
            const uint32_t bar = smem_u32(&ctl.bar[w][st]);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(kbuf + lane * row_bytes)), "l"(kr), "r"(row_bytes), "r"(bar) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(vbuf + lane * row_bytes)), "l"(vr), "r"(row_bytes), "r"(bar) : "memory");
            slot_mass[(size_t)u * Bmax + t0 + lane] = row_mass(sh, s, eps, ud.tok_off + src);
        }
        ok = mbar_wait(&ctl.bar[w][st], (it >> 1) & 1u, abort_flag);
        if (!ok) break;
        if (lane == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            const size_t dst = ((size_t)u * Bmax + t0) * sh.d;
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(k_out + dst), "r"(smem_u32(kbuf)), "r"((uint32_t)nv * row_bytes) : "memory");
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(v_out + dst), "r"(smem_u32(vbuf)), "r"((uint32_t)nv * row_bytes) : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        ++it;
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // (the kernel's end waits for the writes)
    if (!ok && lane == 0) {
        // a copy that was started may still be landing: give the two barriers a bounded chance to complete
        for (uint32_t k = 0; k < 4096 && !mbar_try(&ctl.bar[w][it & 1u], (it >> 1) & 1u); ++k) {}
        atomicOr(sh.err, CASK_ST_TIMEOUT);
    }
}

// ---- 3. one warp per representative with joiners: ordered weighted merge over its copy -----
// CH > 0: head_dim == 32 * CH, every lane owns CH contiguous channels and reads them with one vector load per row;
// CH == 0: any head_dim up to 256, channels lane, lane + 32, ...  The sums per channel are the same either way.
template <typename T, int CH>
__global__ void __launch_bounds__(256) slot_merge_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const T* __restrict__ K, const T* __restrict__ V,
    const float* __restrict__ s, const float* __restrict__ weight, float eps, int Bmax,
    const int32_t* __restrict__ seed_slot, const int32_t* __restrict__ n_seed, int max_B,
    const int32_t* __restrict__ mem_row, const int32_t* __restrict__ mem_slot,
    const int32_t* __restrict__ n_mem, T* __restrict__ k_out, T* __restrict__ v_out,
    float* __restrict__ slot_mass, int32_t* __restrict__ unit_status) {
    pdl_wait();
    const int u = blockIdx.y;
    const UnitDesc& ud = desc[u];
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    // Last kernel of an event: flags raised on the device since the status words were written (a bulk copy of the
    // compaction that gave up) join them.  A page id outside the pool was already met by the scoring pass.
    if (unit_status && blockIdx.x == 0 && threadIdx.x == 0 && *sh.err) unit_status[u] |= *sh.err;
    if (j >= n_seed[u]) return;
    const int t = CASK_IDX(seed_slot[(size_t)u * max_B + j], Bmax, sh.err);
    const int d = sh.d;
    const int64_t o = ud.tok_off;
    constexpr int kMaxPerLane = 8;      // d <= 256
    float ak[kMaxPerLane], av[kMaxPerLane];
#pragma unroll
    for (int x = 0; x < kMaxPerLane; ++x) { ak[x] = 0.f; av[x] = 0.f; }
    int count = 0;
    float msum = 0.f;
    const int nm = n_mem[u];
    // A representative nobody joined keeps the byte copy of its row: count the list entries of this slot first (the
    // list is shared by the unit's warps and stays in cache) and leave before any row is requested.
    {
        int total = 0;
        for (int e0 = 0; e0 < nm; e0 += 32) {
            const int e = e0 + lane;
            total += __popc(__ballot_sync(0xffffffffu, e < nm && mem_slot[o + e] == t));
        }
        if (total <= 1) return;
    }
    // The member list of the unit is walked 128 entries at a time (the eight index loads of a round are independent)
    // and the round's own members are listed in shared memory in ascending order; their rows are then read four at a
    // time, so the latency of a row is paid once per four members and not once per member, and added in list order.
    constexpr int kWalk = 4;
    __shared__ int32_t hits[8][32 * kWalk];
    int32_t* my_hits = hits[threadIdx.x >> 5];
    const unsigned below = (1u << lane) - 1u;
    for (int e0 = 0; e0 < nm; e0 += 32 * kWalk) {
        int row[kWalk];
        bool hit[kWalk];
#pragma unroll
        for (int q = 0; q < kWalk; ++q) {
            const int e = e0 + 32 * q + lane;
            row[q] = (e < nm) ? mem_row[o + e] : -1;
            hit[q] = (e < nm) && mem_slot[o + e] == t;
        }
        int n_hits = 0;
#pragma unroll
        for (int q = 0; q < kWalk; ++q) {
            const unsigned bal = __ballot_sync(0xffffffffu, hit[q]);
            if (hit[q]) my_hits[n_hits + __popc(bal & below)] = row[q];
            n_hits += __popc(bal);
        }
        __syncwarp();
        constexpr int kRows = 4;           // member rows in flight per warp
        for (int h0 = 0; h0 < n_hits; h0 += kRows) {
            if (CH > 0) {
                struct alignas((CH > 0 ? CH : 1) * sizeof(T)) Vec { T x[CH > 0 ? CH : 1]; };
                Vec kv[kRows], vv[kRows];
                float wi[kRows], ai[kRows];
                // Offsets first, loads after, uses last, with no branch in between: a branch inside the loop over the
                // rows (paged or not, carried mass or not) makes every row wait for the one before it.
                int64_t io[kRows], ko[kRows], vo[kRows];
#pragma unroll
                for (int q = 0; q < kRows; ++q)
                    io[q] = o + CASK_IDX(my_hits[min(h0 + q, n_hits - 1)], ud.T, sh.err);
                if (sh.page_size == 0 && !sh.v_pos) {
#pragma unroll
                    for (int q = 0; q < kRows; ++q) {
                        ko[q] = ud.k_off + (io[q] - o) * sh.row_stride;
                        vo[q] = ud.v_off + (io[q] - o) * sh.row_stride;
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < kRows; ++q) {
                        ko[q] = row_elem_off(sh, ud, ud.k_off, (int)(io[q] - o));
                        vo[q] = v_elem_off(sh, ud, u, (int)(io[q] - o));
                    }
                }
#pragma unroll
                for (int q = 0; q < kRows; ++q) {
                    wi[q] = weight[io[q]];
                    ai[q] = s[io[q]];
                    kv[q] = reinterpret_cast<const Vec*>(K + ko[q])[lane];
                    vv[q] = reinterpret_cast<const Vec*>(V + vo[q])[lane];
                }
                if (sh.mass_in) {
                    float mi[kRows];
#pragma unroll
                    for (int q = 0; q < kRows; ++q) mi[q] = sh.mass_in[io[q]];
#pragma unroll
                    for (int q = 0; q < kRows; ++q) ai[q] = (ai[q] + eps) + mi[q];      // row_mass()
                } else {
#pragma unroll
                    for (int q = 0; q < kRows; ++q) ai[q] += eps;
                }
#pragma unroll
                for (int q = 0; q < kRows; ++q) {
                    if (h0 + q >= n_hits) break;
                    msum += ai[q];
                    ++count;
#pragma unroll
                    for (int x = 0; x < CH; ++x) {
                        ak[x] = fmaf(wi[q], Elem<T>::ld(&kv[q].x[x]), ak[x]);
                        av[x] = fmaf(wi[q], Elem<T>::ld(&vv[q].x[x]), av[x]);
                    }
                }
            } else {
                for (int q = 0; q < kRows && h0 + q < n_hits; ++q) {
                    const int i = CASK_IDX(my_hits[h0 + q], ud.T, sh.err);
                    const float wq = weight[o + i];
                    msum += row_mass(sh, s, eps, o + i);
                    ++count;
                    const T* kr = K + row_elem_off(sh, ud, ud.k_off, i);
                    const T* vr = V + v_elem_off(sh, ud, u, i);
#pragma unroll
                    for (int x = 0; x < kMaxPerLane; ++x) {
                        const int c = lane + 32 * x;
                        if (c < d) {
                            ak[x] = fmaf(wq, Elem<T>::ld(kr + c), ak[x]);
                            av[x] = fmaf(wq, Elem<T>::ld(vr + c), av[x]);
                        }
                    }
                }
            }
        }
        __syncwarp();
    }
    if (count > 1) {       // a lone seed keeps its byte copy
        T* ko = k_out + ((size_t)u * Bmax + t) * d;
        T* vo = v_out + ((size_t)u * Bmax + t) * d;
#pragma unroll
        for (int x = 0; x < kMaxPerLane; ++x) {
            const int c = CH > 0 ? lane * CH + x : lane + 32 * x;
            if ((CH > 0 && x < CH) || (CH == 0 && c < d)) {
                Elem<T>::st(ko + c, ak[x]);
                Elem<T>::st(vo + c, av[x]);
            }
        }
        if (lane == 0) slot_mass[(size_t)u * Bmax + t] = msum;
    }
}

// ---- slots in batches: copied rows and merged ones (shared by the two one-kernel compactions below) ---------------------
constexpr int kFusedWarps = 8;
// Bytes per warp and stage (K half + V half): three CTAs per SM in both kernels, with the slot tables of 2,048-row budgets
// beside the staging in the longer units' one.
constexpr int kSmallStage = 4096, kLongStage = 3072;
constexpr int staging_bytes(int stage) { return kFusedWarps * 2 * stage; }

template <typename T>
struct RowSource {
    const T *K, *V;
    const float *s, *weight;
    float eps;
    const FusedWeights& fw;
    const UnitDesc& ud;
    const Shape& sh;
    int u;
};

template <int N> struct alignas(4 * N) Words { uint32_t w[N]; };
// Channel x of them (whole words, so that a row can be left out without its registers going to memory).
template <typename T, int N>
__device__ __forceinline__ float channel(const Words<N>& p, int x) {
    if (sizeof(T) == 4) return __uint_as_float(p.w[x < N ? x : 0]);
    const uint32_t w = p.w[(x >> 1) < N ? x >> 1 : 0];
    return __uint_as_float(x & 1 ? w & 0xFFFF0000u : w << 16);
}

// Two kinds of work, handed out to the warps of a unit's CTAs one after the other:
//   * the slots that others joined, `per_item` of them at a time: their members' rows are added up (ascending row order, fp32, rounded
//     once) and written out.  A lane looks one member up (page, score, carried mass, group mass) and the rows are loaded kRows at
//     a time whatever slots they feed: eight where a lane's piece of a row is one word, else four (eight of two words spill, and cost eight
//     units of 33,280 rows 2 us).  Where the rows lie and what they count goes through shared memory: by shuffles, six a row, a member took
//     0.24 us of a group's time, now 0.15 (128 units of 4,608 rows at head_dim 64, kernel alone 31.2 to 27.5; 8 of 9,000 29.1 to 24.1; 240 of
//     1,024 whose other rows all join 69.4 to 64.6).  But by shuffles for the other head dims (CH == 0), whose loads follow each row's place:
//     100 units of 5,000 rows at head_dim 96, kernel alone 55.6 to 68.7 through shared memory, 361 to 462 where all other rows join;
//     8 at 80 27.1 to 29.3.  They come first: a group is a chain of memory latencies, three and one more per
//     kRows members.
//   * batches of consecutive slots: bulk copies of the rows of the other ones into the warp's staging buffer, then bulk stores, two
//     for a batch without merged slots, because consecutive slots are contiguous in the output; two buffers, so the copies of a
//     batch run under the stores of the one before.
// With the groups of a batch of slots added up by the warp that copies the batch, a few warps had most of the members of a unit, since the
// slots with members lie together, and the kernel waited for them.  Kernel alone, with them and now: 128 units of 4,608 rows at head_dim
// 64 35.8 and 31.2 us, 112 of 13,312 71.9 and 65.8, 112 of 9,000 32.8 and 27.6, 3,072 of 640 300 and 290, 8 of 640 17.2 and 14.9.
// per_item (kernel alone, us): one where a unit has several CTAs, so that no warp has several groups to add up while others have none: 8
// units of 3,000 rows 17.1, with four 21.3; 112 of 1,900 31.3, 36.9.  Else four, which share their latencies: 240 units of 1,024
// of which all others join 62.0, with one 72.1; 3,072 of 640 338, 362 (eight: 337).
// Units of more than kListCap members have no list of the slots with members, and all slots are looked through: eight consecutive ones
// at a time, 240 units of 9,000 rows (2,048 kept) of which all others join 559, with one 703; of 3,000 (1,536) 211, 296.  But one where
// groups have more than four members on average, 112 of 9,000 (512) 313, with four 381, with eight 530; or more than two and there are
// fewer than four items of eight a warp: 112 of 1,900 (512) 92, with eight 99; 40 of them 60, 76.
//   row_of(slot) -> cache row; first(slot) -> place in the list of the slot's first member (first(nk): the end).
//   member(place) -> cache row; busy(i), i < n_busy -> slots, all those with two members or more among them.
// CH > 0: head_dim == 32 * CH, a lane owns CH contiguous channels; CH == 0: any head_dim up to 256, channels lane, lane + 32, ...
template <typename T, int CH, int STAGE, typename RowOf, typename First, typename Member, typename Busy>
__device__ __forceinline__ void copy_batches(const RowSource<T>& in, int nk, int parts, int part, uint8_t* staging,
                                             uint64_t (*bars)[2], int* next_item, int* abort_word, T* __restrict__ k_out,
                                             T* __restrict__ v_out, float* __restrict__ slot_mass, int Bmax,
                                             int32_t* __restrict__ err, int per_item, int n_busy, RowOf row_of, First first, Member member,
                                             Busy busy) {
    using namespace tc;
    constexpr int kPer = CH > 0 ? CH : 8;
    constexpr int kRows = CH > 0 && CH * sizeof(T) <= 4 ? 8 : 4;           // member rows in flight
    struct alignas((CH > 0 ? CH : 1) * sizeof(T)) Vec { T x[CH > 0 ? CH : 1]; };
    using Piece = Words<(CH > 0 ? CH * sizeof(T) / 4 : 1)>;      // a lane's channels of a row
    const Shape& sh = in.sh;
    const UnitDesc& ud = in.ud;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, u = in.u, d = sh.d;
    const int64_t o = ud.tok_off;
    const uint32_t row_bytes = CH > 0 ? (uint32_t)(32 * CH * sizeof(T)) : (uint32_t)(d * sizeof(T));
    const int sb = min(32, (int)(STAGE / 2 / row_bytes));                  // slots per batch
    volatile int* abort_flag = abort_word;
    uint8_t* my = staging + w * 2 * STAGE;
    // (a warp's merged slots come before its batches of rows to copy: the staging area is free until then)
    int64_t* at_k = reinterpret_cast<int64_t*>(my);
    int64_t* at_v = at_k + 32;
    float2* counts = reinterpret_cast<float2*>(at_v + 32);
    static_assert(2 * STAGE >= 24 * 32, "one member a lane");
    const int nb = (nk + sb - 1) / sb, n_items = (n_busy + per_item - 1) / per_item;
    uint32_t it = 0;
    bool ok = true;
    while (ok) {
        int b = 0;
        if (lane == 0) b = atomicAdd(next_item, 1);
        b = __shfl_sync(0xffffffffu, b, 0) * parts + part;
        if (b >= n_items + nb) break;
        if (b < n_items) {
            // ---- merged slots, a lane a slot
            const bool mine = lane < per_item && b * per_item + lane < n_busy;
            const int t = mine ? busy(b * per_item + lane) : 0;
            const int f = mine ? first(t) : 0, members = mine ? first(t + 1) - f : 0;
            const bool merged = members > 1;
            if (!__any_sync(0xffffffffu, merged)) continue;
            float mg_t = 0.f;                      // group mass of slot t (event path: the weights are formed here)
            if (in.fw.s && merged) {
                const int gi = min(max(CASK_IDX(in.fw.grp[o + row_of(t)], max(in.fw.max_m, 1), err), 0), in.fw.max_m);
                mg_t = fx_to_mass(in.fw.mass_fx[(size_t)u * (in.fw.max_m + 1) + gi]);
            }
            float ak[kPer], av[kPer], msum;
            auto clear = [&] {
                msum = 0.f;
#pragma unroll
                for (int x = 0; x < kPer; ++x) { ak[x] = 0.f; av[x] = 0.f; }
            };
            auto finish = [&](int sl) {
                T* kw = k_out + ((size_t)u * Bmax + sl) * d;
                T* vw = v_out + ((size_t)u * Bmax + sl) * d;
                if (CH > 0) {
                    Vec k1, v1;
#pragma unroll
                    for (int x = 0; x < (CH > 0 ? CH : 1); ++x) {
                        Elem<T>::st(&k1.x[x], ak[x]);
                        Elem<T>::st(&v1.x[x], av[x]);
                    }
                    reinterpret_cast<Vec*>(kw)[lane] = k1;
                    reinterpret_cast<Vec*>(vw)[lane] = v1;
                } else {
#pragma unroll
                    for (int x = 0; x < kPer; ++x)
                        if (lane + 32 * x < d) {
                            Elem<T>::st(kw + lane + 32 * x, ak[x]);
                            Elem<T>::st(vw + lane + 32 * x, av[x]);
                        }
                }
                if (lane == 0) slot_mass[(size_t)u * Bmax + sl] = msum;
            };
            clear();
            const int count = merged ? members : 0;
            int before = count;                // members of the item's slots below this one
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, before, off);
                if (lane >= off) before += x;
            }
            const int total = __shfl_sync(0xffffffffu, before, 31);
            before -= count;
            for (int e0 = 0; e0 < total; e0 += 32) {
                const int n = min(32, total - e0), e = e0 + min(lane, n - 1);
                int sl = 0;                    // slot of member e: the last one with at most e members below it
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1) {
                    const int x = __shfl_sync(0xffffffffu, before, sl + step);
                    if (x <= e) sl += step;
                }
                const int in_group = e - __shfl_sync(0xffffffffu, before, sl);
                const int row = CASK_IDX(member(__shfl_sync(0xffffffffu, f, sl) + in_group), ud.T, err);
                const unsigned ends = __ballot_sync(0xffffffffu, in_group + 1 == __shfl_sync(0xffffffffu, members, sl));
                const int64_t ko = row_elem_off(sh, ud, ud.k_off, row), vo = v_elem_off(sh, ud, u, row);
                const float ae = row_mass(sh, in.s, in.eps, o + row);
                const float mg = __shfl_sync(0xffffffffu, mg_t, sl);
                const float we = in.fw.s ? ae / mg : in.weight[o + row];
                if (CH > 0) {
                    __syncwarp();
                    at_k[lane] = ko;
                    at_v[lane] = vo;
                    counts[lane] = make_float2(we, ae);
                    __syncwarp();
                }
                for (int c0 = 0; c0 < n; c0 += kRows) {
                    Piece kr[kRows], vr[kRows];
                    if (CH > 0) {
#pragma unroll
                        for (int q = 0; q < kRows; ++q) {
                            kr[q] = vr[q] = Piece{};
                            if (c0 + q < n) {
                                kr[q] = reinterpret_cast<const Piece*>(in.K + at_k[c0 + q])[lane];
                                vr[q] = reinterpret_cast<const Piece*>(in.V + at_v[c0 + q])[lane];
                            }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < kRows; ++q) {
                        if (c0 + q >= n) break;
                        const float wi = CH > 0 ? counts[c0 + q].x : __shfl_sync(0xffffffffu, we, c0 + q);
                        msum += CH > 0 ? counts[c0 + q].y : __shfl_sync(0xffffffffu, ae, c0 + q);
                        const int64_t kq = CH > 0 ? 0 : __shfl_sync(0xffffffffu, ko, c0 + q);
                        const int64_t vq = CH > 0 ? 0 : __shfl_sync(0xffffffffu, vo, c0 + q);
#pragma unroll
                        for (int x = 0; x < kPer; ++x) {
                            if (CH > 0) {
                                ak[x] = fmaf(wi, channel<T>(kr[q], x), ak[x]);
                                av[x] = fmaf(wi, channel<T>(vr[q], x), av[x]);
                            } else if (lane + 32 * x < d) {
                                ak[x] = fmaf(wi, Elem<T>::ld(in.K + kq + lane + 32 * x), ak[x]);
                                av[x] = fmaf(wi, Elem<T>::ld(in.V + vq + lane + 32 * x), av[x]);
                            }
                        }
                        if ((ends >> (c0 + q)) & 1u) {
                            finish(__shfl_sync(0xffffffffu, t, __shfl_sync(0xffffffffu, sl, c0 + q)));
                            clear();
                        }
                    }
                }
            }
            continue;
        }
        // ---- rows to copy
        const int t0 = (b - n_items) * sb;
        const int nv = min(sb, nk - t0);
        const uint32_t st = it & 1u;
        uint8_t* kbuf = my + st * STAGE;
        uint8_t* vbuf = kbuf + STAGE / 2;
        const int t = t0 + lane;
        const bool copied = lane < nv && first(t + 1) - first(t) < 2;
        const int n_copied = __popc(__ballot_sync(0xffffffffu, copied));
        // the stores that read this buffer two batches ago must have read it (every lane has groups of its own)
        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        if (CH > 0 && it == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // (the members' places are written over)
        if (lane == 0) mbar_expect_tx(&bars[w][st], (uint32_t)n_copied * 2u * row_bytes);
        __syncwarp();
        if (copied) {
            const int row = CASK_IDX(row_of(t), ud.T, err);
            const T* kr = in.K + row_elem_off(sh, ud, ud.k_off, row);
            const T* vr = in.V + v_elem_off(sh, ud, u, row);
            const uint32_t bar = smem_u32(&bars[w][st]);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(kbuf + lane * row_bytes)), "l"(kr), "r"(row_bytes), "r"(bar) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(vbuf + lane * row_bytes)), "l"(vr), "r"(row_bytes), "r"(bar) : "memory");
            slot_mass[(size_t)u * Bmax + t] = row_mass(sh, in.s, in.eps, o + row);
        }
        ok = mbar_wait(&bars[w][st], (it >> 1) & 1u, abort_flag);
        __syncwarp();
        if (!ok) break;
        // a batch without merged slots in two pieces, else slot by slot
        const bool whole = n_copied == nv;
        if (whole ? lane == 0 : copied) {
            const size_t dst = ((size_t)u * Bmax + t) * d;
            const uint32_t from = lane * row_bytes, bytes = whole ? (uint32_t)nv * row_bytes : row_bytes;
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(k_out + dst), "r"(smem_u32(kbuf) + from), "r"(bytes) : "memory");
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(v_out + dst), "r"(smem_u32(vbuf) + from), "r"(bytes) : "memory");
        }
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        ++it;
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok && lane == 0) {
        // a copy that was started may still be landing: give the barrier a bounded chance to complete
        for (uint32_t k = 0; k < 4096 && !mbar_try(&bars[w][it & 1u], (it >> 1) & 1u); ++k) {}
        atomicOr(err, CASK_ST_TIMEOUT);
    }
}

// Last kernel of an event: what a CTA raised joins all status words, by the CTA itself, once per flag (err[1] holds those that
// went out; it is cleared with the flags at the start of the call).  The words are only ever ORed into from the selection kernel
// on, which clears them, so no CTA has to know how far the others are: a fence before the last CTA looked took 5 to
// 7 us at the end of every event (eight units of 640 rows 55.5 to 54.8 us, eight of 33,280 162 to 160, 288 of 640 150 to 146).
__device__ __forceinline__ void late_flags(const FusedWeights& fw, int n_units, int32_t* __restrict__ err) {
    if (!fw.s) return;
    __syncthreads();                               // the CTA's own flags are raised
    if (threadIdx.x >= 32) return;
    const int flags = *(volatile int32_t*)err;
    if (!flags) return;
    int mine = threadIdx.x == 0 ? flags & ~atomicOr(&err[1], flags) : 0;
    mine = __shfl_sync(0xffffffffu, mine, 0);
    if (mine)
        for (int x = threadIdx.x; x < n_units; x += 32) atomicOr(&fw.unit_status[x], mine);
}

// Status word and lost mass of a unit (event path).
__device__ __forceinline__ void write_status(const FusedWeights& fw, int u) {
    int fl = fw.plan[u * 8 + CASK_PLAN_FLAGS];
    if ((fl & CASK_ST_DECODE_CONSOLIDATED) && fw.njoin[u] == 0) fl |= CASK_ST_MERGE_INACTIVE;
    atomicOr(&fw.unit_status[u], fl | *(volatile int32_t*)fw.err);     // device-side flags of this call so far
    fw.lost_mass[u] = fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + fw.max_m]);
}

// ---- units of at most kSmallRows rows: scan, copy and merge in one kernel -----------------------------------------------
// `parts` CTAs per unit, each with the unit's whole scan in shared memory (a thousand rows: cheaper than a kernel that hands
// it over) and every parts-th item of work (copy_batches).  Bound by HBM and, with few units, by latency; three CTAs of
// 74 KB per SM keep about 140 KB in flight.
// 3,072 paged units of 640 rows (512 kept, bf16, d = 128): 301 us = 5.3 TB/s of rows in and out, where the scan, copy and merge
// kernels took 29 + 420; 288 such units 35 us (80 before), 8 units 15 (33 before, each with its launch).
constexpr int kSmallRows = 1024;

template <typename T, int CH>       // CH: see copy_batches
__global__ void __launch_bounds__(kFusedWarps * 32, 3) compact_small_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const T* __restrict__ K, const T* __restrict__ V,
    const uint8_t* __restrict__ kind, const int32_t* __restrict__ seed_of, const float* __restrict__ s, float* __restrict__ weight,
    float eps, int Bmax, int parts, int32_t* __restrict__ n_out, int32_t* __restrict__ slot_src, uint8_t* __restrict__ slot_kind,
    float* __restrict__ slot_mass, int32_t* __restrict__ assign, T* __restrict__ k_out, T* __restrict__ v_out, FusedWeights fw,
    int32_t* __restrict__ err) {
    using namespace tc;
    constexpr int kThreads = kFusedWarps * 32, kIters = kSmallRows / kThreads;
    static_assert(kIters * kFusedWarps == 32, "one cell per lane");
    extern __shared__ __align__(128) uint8_t copy_smem[];
    __shared__ uint64_t bars[kFusedWarps][2];
    __shared__ int abort_, next_item, n_busy;
    __shared__ unsigned cell[32], totals, wsum[kFusedWarps];
    __shared__ int16_t src[kSmallRows], list[kSmallRows];      // row of a slot; members slot by slot
    __shared__ int16_t busy[kSmallRows / 2];                   // slots with two members or more
    __shared__ int start[kSmallRows + 1];                      // first of a slot's members
    // tables of the scan, in the staging area until the copies begin
    int16_t* slot_of = reinterpret_cast<int16_t*>(copy_smem);  // slot a row feeds
    int16_t* m_row = slot_of + kSmallRows;
    int16_t* m_slot = m_row + kSmallRows;
    uint8_t* kd_s = reinterpret_cast<uint8_t*>(m_slot + kSmallRows);
    static_assert(7 * kSmallRows <= staging_bytes(kSmallStage), "the tables fit the staging area");
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int u = blockIdx.x / parts, part = blockIdx.x - u * parts;
    if (tid == 0) {
        for (int i = 0; i < kFusedWarps; ++i) { mbar_init(&bars[i][0], 1); mbar_init(&bars[i][1], 1); }
        abort_ = 0;
        next_item = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int t = tid; t <= kSmallRows; t += kThreads) start[t] = 0;
    pdl_wait();
    const UnitDesc& ud = desc[u];
    const int T_ = ud.T;
    const int64_t o = ud.tok_off;
    const unsigned below = (1u << lane) - 1u;
    // ---- slots and members in row order: one ballot per (256 rows, warp) cell, one scan over the cells
    uint8_t kd[kIters];
    int sd[kIters];
#pragma unroll
    for (int q = 0; q < kIters; ++q) kd[q] = q * kThreads + tid < T_ ? kind[o + q * kThreads + tid] : (uint8_t)0;
#pragma unroll
    for (int q = 0; q < kIters; ++q) sd[q] = kd[q] == CASK_KIND_MERGED ? seed_of[o + q * kThreads + tid] : -1;
#pragma unroll
    for (int q = 0; q < kIters; ++q) {
        const bool keep = kd[q] >= CASK_KIND_PREFIX && kd[q] <= CASK_KIND_SEED;
        const bool mem = kd[q] == CASK_KIND_SEED || kd[q] == CASK_KIND_MERGED;
        const unsigned bk = __ballot_sync(0xffffffffu, keep), bm = __ballot_sync(0xffffffffu, mem);
        if (lane == 0) cell[q * kFusedWarps + w] = (unsigned)__popc(bk) | ((unsigned)__popc(bm) << 16);
        kd_s[q * kThreads + tid] = kd[q];
    }
    __syncthreads();
    if (w == 0) {
        const unsigned v = cell[lane];
        unsigned incl = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned x = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += x;
        }
        cell[lane] = incl - v;
        if (lane == 31) totals = incl;
    }
    __syncthreads();
    const int nk = min((int)(totals & 0xFFFFu), Bmax), nm = (int)(totals >> 16);
#pragma unroll
    for (int q = 0; q < kIters; ++q) {
        const int i = q * kThreads + tid;
        const bool keep = kd[q] >= CASK_KIND_PREFIX && kd[q] <= CASK_KIND_SEED;
        const bool mem = kd[q] == CASK_KIND_SEED || kd[q] == CASK_KIND_MERGED;
        const unsigned bk = __ballot_sync(0xffffffffu, keep), bm = __ballot_sync(0xffffffffu, mem);
        const unsigned cb = cell[q * kFusedWarps + w];
        int slot = keep ? (int)((cb & 0xFFFFu) + __popc(bk & below)) : -1;
        if (slot >= Bmax) slot = -1;             // more kept rows than slots: cannot happen for a valid plan
        slot_of[i] = (int16_t)slot;
        if (slot >= 0) src[slot] = (int16_t)i;
        if (mem) m_row[(cb >> 16) + __popc(bm & below)] = (int16_t)i;
    }
    __syncthreads();
    // ---- every row's slot (a merged row's is its seed's) and weight
#pragma unroll
    for (int q = 0; q < kIters; ++q) {
        const int i = q * kThreads + tid;
        if (i >= T_) break;
        if (kd[q] == CASK_KIND_MERGED && sd[q] >= 0 && sd[q] < T_ && kd_s[sd[q]] == CASK_KIND_SEED) slot_of[i] = slot_of[sd[q]];
        if (q % parts != part) continue;
        assign[o + i] = slot_of[i];
        if (kd[q] >= CASK_KIND_PREFIX && kd[q] <= CASK_KIND_CORE) weight[o + i] = 1.f;
        if (kd[q] == CASK_KIND_DROPPED) weight[o + i] = 0.f;
        if (fw.s && (kd[q] == CASK_KIND_SEED || kd[q] == CASK_KIND_MERGED)) {
            const int gi = fw.grp[o + i];
            if (gi >= 0 && gi < fw.max_m)
                weight[o + i] = row_mass(sh, s, eps, o + i) / fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + gi]);
        }
    }
    if (part == 0) {
        if (tid == 0) {
            n_out[u] = nk;
            if (fw.s) write_status(fw, u);
        }
        for (int t = tid; t < Bmax; t += kThreads) {
            slot_src[(size_t)u * Bmax + t] = t < nk ? src[t] : -1;
            slot_kind[(size_t)u * Bmax + t] = t < nk ? kd_s[src[t]] : (uint8_t)0;
            if (t >= nk) slot_mass[(size_t)u * Bmax + t] = 0.f;
        }
    }
    __syncthreads();
    // ---- members by slot: counts, their exclusive scan, stable placement (a member counts the earlier ones of its slot)
    for (int e = tid; e < nm; e += kThreads) {
        const int t = slot_of[m_row[e]];
        m_slot[e] = (int16_t)t;
        if (t >= 0) atomicAdd(&start[t], 1);
    }
    __syncthreads();
    {
        int c[kIters], sum = 0;                     // members, slots with two or more << 16 (in slot order: every CTA of the unit the same)
#pragma unroll
        for (int q = 0; q < kIters; ++q) { c[q] = start[kIters * tid + q]; sum += c[q] + ((c[q] > 1) << 16); }
        int incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += x;
        }
        if (lane == 31) wsum[w] = (unsigned)incl;
        __syncthreads();
        int run = incl - sum;
        for (int x = 0; x < w; ++x) run += (int)wsum[x];
#pragma unroll
        for (int q = 0; q < kIters; ++q) {
            start[kIters * tid + q] = run & 0xFFFF;
            if (c[q] > 1) busy[run >> 16] = (int16_t)(kIters * tid + q);
            run += c[q] + ((c[q] > 1) << 16);
        }
        if (tid == kThreads - 1) { start[kSmallRows] = run & 0xFFFF; n_busy = run >> 16; }
    }
    __syncthreads();
    for (int e = tid; e < nm; e += kThreads) {
        const int t = m_slot[e];
        if (t < 0) continue;
        int before = 0;
        for (int x = 0; x < e; ++x) before += m_slot[x] == t;
        list[start[t] + before] = m_row[e];
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // bulk copies write over the tables from here on
    __syncthreads();
    // ---- batches of slots
    const RowSource<T> in{K, V, s, weight, eps, fw, ud, sh, u};
    copy_batches<T, CH, kSmallStage>(
        in, nk, parts, part, copy_smem, bars, &next_item, &abort_, k_out, v_out, slot_mass, Bmax, err, parts > 1 ? 1 : 4, n_busy,
        [&](int t) { return (int)src[t]; }, [&](int t) { return start[t]; }, [&](int e) { return (int)list[e]; },
        [&](int i) { return (int)busy[i]; });
    late_flags(fw, sh.n_units, err);
}

// ---- longer units: the same in one kernel, with lists instead of per-row tables ------------------------------------------
// `parts` CTAs per unit.  Each reads all of the unit's kinds, 16 rows a load, twice: once to count kept rows and group members
// per (pass, warp) cell, and after one scan of the cells to list them, which yields the slots in order.  (Few rows of a long
// unit are kept: everything after the counting is work on some hundreds of entries.  What a dropped row gets in the per-row
// outputs, the selection kernel has written.)  Up to kListCap members sit in shared memory, placed slot by slot in row order by
// counting the earlier ones of a slot.  More (thousands of merged rows) are listed in the workspace and placed there by one warp, 32
// at a time, while the others look up the slots of the next kListCap.  (Event of 32 units of 8,448 rows of which all others join:
// 375 us; with every representative's warp walking the whole list 1,374, with a scan, a copy and a merge kernel 342.)
// 8 units of 33,280 rows (1,024 kept) 33 us, where the scan, copy and merge kernels took 29 + 21 and two more launches; 16 fp32
// units of 8,448 27 (21 + 20), 112 bf16 ones 35 (21 + 35), 288 of 33,280 63 (57 + 65), 112 of 13,312 with 2,048 kept 69 (19 + 74,
// of which the copies run at the rate of HBM).
// LISTS (want_slot_lists): slots, seeds and joined rows are listed already and the kinds are not read.  Eight units of 33,280 rows 33 to
// 26 us, 288 of them 62 to 52, 512 of 4,700 to 33,000 120 to 106, 112 of 8,448 35 to 31.5.
constexpr int kListCap = 1024;
constexpr int kLongThreads = kFusedWarps * 32;
constexpr int kMaxCells = 512;                      // (pass, warp) cells: 64 passes of 4,096 rows
constexpr int kLongMaxRows = 64 * 16 * kLongThreads - 16;
constexpr int kLongMaxSlots = 12288;                // 8 bytes of shared memory per slot
inline size_t long_smem(int slots) { return staging_bytes(kLongStage) + (size_t)slots * 8 + 16; }

// Bit b of the result: byte b of w (a row's kind, 0..5) is kept (1..4) / a group member (4, 5).
__device__ __forceinline__ unsigned nibble(unsigned bits) { return ((bits & 0x01010101u) * 0x10204080u) >> 28; }
__device__ __forceinline__ unsigned keep_bits(unsigned w) {
    return nibble((w | (w >> 1) | (w >> 2)) & ~((w >> 2) & w));
}
__device__ __forceinline__ unsigned member_bits(unsigned w) { return nibble(w >> 2); }

// What the selection and the assignment kernel have listed (LISTS; n_kept = -1: this unit has no lists after all).
struct GivenLists {
    const int32_t *n_kept, *n_seed, *seed_slot, *seed_rows;
    int max_B;
};

template <typename T, int CH, bool LISTS>
__global__ void __launch_bounds__(kLongThreads, 3) compact_long_kernel(
    const UnitDesc* __restrict__ desc, Shape sh, const T* __restrict__ K, const T* __restrict__ V,
    const uint8_t* __restrict__ kind, const int32_t* __restrict__ seed_of, const float* __restrict__ s, float* __restrict__ weight,
    float eps, int Bmax, int slots, int parts, int32_t* __restrict__ n_out, int32_t* __restrict__ slot_src,
    uint8_t* __restrict__ slot_kind, float* __restrict__ slot_mass, int32_t* __restrict__ assign, int32_t* __restrict__ mem_row,
    int32_t* __restrict__ mem_slot, GivenLists given, T* __restrict__ k_out, T* __restrict__ v_out, FusedWeights fw,
    int32_t* __restrict__ err) {
    using namespace tc;
    extern __shared__ __align__(128) uint8_t copy_smem[];
    __shared__ uint64_t bars[kFusedWarps][2];
    __shared__ int abort_, next_item, n_busy;
    __shared__ unsigned totals, wsum[kFusedWarps];
    __shared__ int list[kListCap];                                         // members slot by slot
    __shared__ uint16_t busy[kListCap / 2];                                // slots with two members or more
    int* src = reinterpret_cast<int*>(copy_smem + staging_bytes(kLongStage));   // [slots] 2 * row + (1: a seed) of a slot, ascending
    int* start = src + slots + 1;                                          // [slots + 1] first of a slot's members (start[-1]: 0)
    // in the staging area until the copies begin: row and slot of the members; kept rows and members before every cell
    int* m_row = reinterpret_cast<int*>(copy_smem);
    int* m_slot = m_row + kListCap;
    unsigned* cell = reinterpret_cast<unsigned*>(m_slot + kListCap);
    unsigned* cell_m = cell + kMaxCells;
    unsigned* mask = cell_m + kMaxCells;                                   // of 16 rows: kept, members << 16
    constexpr int kMasks = staging_bytes(kLongStage) / 4 - 2 * kListCap - 2 * kMaxCells;
    static_assert(kMasks >= 8192, "the lists fit the staging area, with the masks of 131,072 rows");
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int u = blockIdx.x / parts, part = blockIdx.x - u * parts;
    if (tid == 0) {
        for (int i = 0; i < kFusedWarps; ++i) { mbar_init(&bars[i][0], 1); mbar_init(&bars[i][1], 1); }
        abort_ = 0;
        next_item = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int t = tid; t <= slots + 1; t += kLongThreads) start[t - 1] = 0;
    __syncthreads();                                         // (with given lists the counting begins at once)
    pdl_wait();
    const UnitDesc& ud = desc[u];
    const int T_ = ud.T;
    const int64_t o = ud.tok_off;
    const uint8_t* ku = kind + o;
    int nk = LISTS ? given.n_kept[u] : -1, nm = 0;
    int n_joined = 0;                                        // given lists: members that are not seeds, the first ones
    bool in_smem = true, given_lists = false;
    auto slot_of = [&](int i) {                              // slot whose anchor is row i, a seed; else -1
        int lo = 0, hi = nk - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((src[mid] >> 1) <= i) lo = mid; else hi = mid - 1;
        }
        return nk > 0 && src[lo] == 2 * i + 1 ? lo : -1;
    };
    if (LISTS && nk >= 0) {
        nm = given.n_seed[u] + fw.njoin[u];
        if (nm > kListCap) nk = -1;                          // (thousands of members: listed in the workspace below, in row order)
    }
    if (LISTS && nk >= 0) {
        // ---- the selection has listed the slots and the seeds, the assignment the rows that joined
        nk = min(nk, min(Bmax, slots));
        const int m = given.n_seed[u];
        n_joined = nm - m;
        given_lists = true;
        const int32_t* seed_slot = given.seed_slot + (size_t)u * given.max_B;
        for (int e = tid; e < nm; e += kLongThreads) {
            const bool joined = e < n_joined;
            const int i = CASK_IDX(joined ? mem_row[o + e] : given.seed_rows[ud.seed_base + e - n_joined], T_, err);
            const int gi = CASK_IDX(joined ? mem_slot[o + e] : e - n_joined, max(m, 1), err);
            const int t = CASK_IDX(seed_slot[gi], max(nk, 1), err);
            m_row[e] = i;
            m_slot[e] = t;
            atomicAdd(&start[t], 1);
            if (e % parts == part) {
                weight[o + i] = row_mass(sh, s, eps, o + i) / fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + gi]);
                if (joined) assign[o + i] = t;
            }
        }
        for (int t = tid; t < nk; t += kLongThreads) {
            const int i = CASK_IDX(slot_src[(size_t)u * Bmax + t], T_, err);
            const bool seed = slot_kind[(size_t)u * Bmax + t] == CASK_KIND_SEED;
            src[t] = 2 * i + (int)seed;
            if (t % parts == part) {
                assign[o + i] = t;
                if (!seed) weight[o + i] = 1.f;
            }
        }
    } else {
        // ---- kinds, 16 rows a thread: rows 16 j - mis .. 16 j - mis + 15, so that a load is aligned; the words at the two ends
        // are put together byte by byte
        const int mis = (int)((uintptr_t)ku & 15u);
        const int words = (T_ + mis + 15) >> 4, passes = (words + kLongThreads - 1) / kLongThreads;
        auto load16 = [&](int j) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            const int r0 = 16 * j - mis;
            if (r0 >= 0 && r0 + 16 <= T_) return *reinterpret_cast<const uint4*>(ku + r0);
            if (r0 < T_) {
                unsigned x[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int b = 0; b < 16; ++b)
                    if (r0 + b >= 0 && r0 + b < T_) x[b >> 2] |= (unsigned)ku[r0 + b] << (8 * (b & 3));
                v = make_uint4(x[0], x[1], x[2], x[3]);
            }
            return v;
        };
        auto masks16 = [&](const uint4& v) {
            return keep_bits(v.x) | (keep_bits(v.y) << 4) | (keep_bits(v.z) << 8) | (keep_bits(v.w) << 12) |
                   ((member_bits(v.x) | (member_bits(v.y) << 4) | (member_bits(v.z) << 8) | (member_bits(v.w) << 12)) << 16);
        };
        for (int p0 = 0; p0 < passes; p0 += 4) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = load16((p0 + q) * kLongThreads + tid);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (p0 + q >= passes) break;
                const unsigned km = masks16(v[q]);
                const int j = (p0 + q) * kLongThreads + tid;
                if (j < kMasks) mask[j] = km;
                const unsigned n = __reduce_add_sync(0xffffffffu, (unsigned)__popc(km & 0xFFFFu) | ((unsigned)__popc(km >> 16) << 16));
                if (lane == 0) cell[(p0 + q) * kFusedWarps + w] = n;
            }
        }
        __syncthreads();
        // Exclusive scan over the cells.  A cell counts at most 512 of each; kept rows and members are counted in 16 bits each here
        // and carried in 32 further on, so the two running sums are scanned one after the other.
        if (w < 2) {
            const int cells = passes * kFusedWarps, per = (cells + 31) / 32, c0 = min(cells, lane * per), c1 = min(cells, c0 + per);
            unsigned sum = 0;
            for (int c = c0; c < c1; ++c) sum += w == 0 ? cell[c] & 0xFFFFu : cell[c] >> 16;
            unsigned incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned x = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += x;
            }
            unsigned run = incl - sum;
            if (lane == 31) (w == 0 ? totals : wsum[0]) = incl;
            if (w == 1)
                for (int c = c0; c < c1; ++c) { cell_m[c] = run; run += cell[c] >> 16; }
            __syncwarp();
            asm volatile("bar.sync 1, 64;" ::: "memory");        // warp 1 has read the counts
            if (w == 0)
                for (int c = c0; c < c1; ++c) { const unsigned n = cell[c] & 0xFFFFu; cell[c] = run; run += n; }
        }
        __syncthreads();
        nk = min((int)totals, min(Bmax, slots));
        nm = (int)wsum[0];
        in_smem = nm <= kListCap;
        // ---- the lists
        const int per_part = (T_ + parts - 1) / parts, f0 = min(T_, part * per_part), f1 = min(T_, f0 + per_part);
        for (int pass = 0; pass < passes; ++pass) {
            const int j = pass * kLongThreads + tid;
            const unsigned km = j < kMasks ? mask[j] : masks16(load16(j)), kb = km & 0xFFFFu, mb = km >> 16;
            if (!__any_sync(0xffffffffu, km)) continue;
            const unsigned n = (unsigned)__popc(kb) | ((unsigned)__popc(mb) << 16);
            unsigned incl = n;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned x = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += x;
            }
            int slot = (int)(cell[pass * kFusedWarps + w] + ((incl - n) & 0xFFFFu));
            int e = (int)(cell_m[pass * kFusedWarps + w] + ((incl - n) >> 16));
            const int r0 = 16 * j - mis;
            // A seed is a member of its own slot.  (Members are few and take a loop; kept rows come in runs of hundreds, the
            // prefix and the recent rows, and take sixteen predicated stores: a loop over their bits costs 200 clk a row.)
            for (unsigned bits = mb; bits; bits &= bits - 1) {
                const int b = __ffs(bits) - 1;
                const int own = (kb >> b) & 1u ? slot + __popc(kb & ((1u << b) - 1u)) : -2;
                if (in_smem) { m_row[e] = r0 + b; m_slot[e] = own < nk ? own : -1; }
                else mem_row[o + e] = r0 + b;         // (the unit's other CTAs write the same)
                ++e;
            }
            if (kb) {
                const bool fits = slot + 16 <= nk;
#pragma unroll
                for (int b = 0; b < 16; ++b) {
                    if ((kb >> b) & 1u) {
                        if (fits || slot < nk) src[slot] = 2 * (r0 + b) + (int)((mb >> b) & 1u);
                        ++slot;
                    }
                }
            }
        }
        // A staged call: what a dropped row gets, over this part's share of the rows (on the event path the selection wrote it).
        if (!fw.s)
            for (int i = f0 + tid; i < f1; i += kLongThreads) {
                const uint8_t kd = ku[i];
                if (kd == CASK_KIND_DROPPED) weight[o + i] = 0.f;
                if (kd == CASK_KIND_DROPPED || kd == CASK_KIND_MERGED) assign[o + i] = -1;
            }
        __syncthreads();
        // ---- slot of every kept and merged row, their weights, the slot tables
        // (With thousands of members the loop is a chain of memory latencies: four a thread then, the loads of each kind together.  A few
        // hundred are one round either way, and take 2 to 8 us longer with the loads of three more.)
        auto settle_members = [&](auto u_) {
            constexpr int kU = decltype(u_)::value;
            for (int e0 = tid; e0 < nm; e0 += kU * kLongThreads) {
                int row[kU], sd[kU], gi[kU], t[kU];
                float am[kU];
                uint8_t kd[kU];
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    const int e = min(e0 + q * kLongThreads, nm - 1);
                    row[q] = in_smem ? m_row[e] : CASK_IDX(mem_row[o + e], T_, err);
                    t[q] = in_smem ? m_slot[e] : -3;
                }
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    const bool mine = row[q] >= f0 && row[q] < f1;
                    sd[q] = seed_of[o + row[q]];                     // (a seed points at itself)
                    gi[q] = fw.s && mine ? fw.grp[o + row[q]] : -1;
                    kd[q] = in_smem ? (uint8_t)CASK_KIND_MERGED : ku[row[q]];
                }
#pragma unroll
                for (int q = 0; q < kU; ++q) am[q] = gi[q] >= 0 ? row_mass(sh, s, eps, o + row[q]) : 0.f;
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    if (e0 + q * kLongThreads >= nm) break;
                    const int i = row[q];
                    if (t[q] == -3 && kd[q] == CASK_KIND_SEED) t[q] = slot_of(i);
                    else if (t[q] < -1) {
                        t[q] = slot_of(sd[q]);
                        if (i >= f0 && i < f1) assign[o + i] = t[q];
                    }
                    if (in_smem) m_slot[e0 + q * kLongThreads] = t[q];
                    if (t[q] >= 0) atomicAdd(&start[t[q]], 1);
                    if (gi[q] >= 0 && gi[q] < fw.max_m) weight[o + i] = am[q] / fx_to_mass(fw.mass_fx[(size_t)u * (fw.max_m + 1) + gi[q]]);
                }
            }
        };
        if (in_smem) settle_members(std::integral_constant<int, 1>{});
        else settle_members(std::integral_constant<int, 4>{});
        for (int t = tid; t < nk; t += kLongThreads) {
            const int i = src[t] >> 1;
            if (i < f0 || i >= f1) continue;
            const uint8_t kd = ku[i];
            assign[o + i] = t;
            if (kd != CASK_KIND_SEED) weight[o + i] = 1.f;
            slot_src[(size_t)u * Bmax + t] = i;
            slot_kind[(size_t)u * Bmax + t] = kd;
        }
    }
    if (part == 0) {
        if (tid == 0) {
            n_out[u] = nk;
            if (fw.s) write_status(fw, u);
        }
        for (int t = nk + tid; t < Bmax; t += kLongThreads) {
            slot_src[(size_t)u * Bmax + t] = -1;
            slot_kind[(size_t)u * Bmax + t] = 0;
            slot_mass[(size_t)u * Bmax + t] = 0.f;
        }
    }
    __syncthreads();
    // ---- counts -> first places, then every member's place: the first one of its slot, plus the earlier members of the slot
    {
        const int per = (nk + kLongThreads - 1) / kLongThreads, t0 = min(nk, tid * per), t1 = min(nk, t0 + per);
        // (members in shared memory, at most kListCap: the slots with two or more are counted along in the upper half, in slot order, so
        // that every CTA of the unit numbers them the same way)
        auto step = [&](int n) { return n + (in_smem && n > 1 ? 1 << 16 : 0); };
        const int low = in_smem ? 0xFFFF : -1;
        int sum = 0;
        for (int t = t0; t < t1; ++t) sum += step(start[t]);
        int incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += x;
        }
        if (lane == 31) wsum[w] = (unsigned)incl;
        __syncthreads();
        int run = incl - sum;
        for (int x = 0; x < w; ++x) run += (int)wsum[x];
        for (int t = t0; t < t1; ++t) {
            const int n = start[t];
            start[t] = run & low;
            if (n > 1 && in_smem) busy[run >> 16] = (uint16_t)t;
            run += step(n);
        }
        if (tid == kLongThreads - 1) { start[nk] = run & low; n_busy = in_smem ? run >> 16 : nk; }        // the last thread ends on the total
    }
    __syncthreads();
    if (in_smem)
        for (int e = tid; e < nm; e += kLongThreads) {
            const int t = m_slot[e];
            if (t < 0) continue;
            int before = 0, x = 0;
            if (LISTS && given_lists) {
                const int row = m_row[e];
                before = e < n_joined && (src[t] >> 1) < row;          // the slot's seed
                for (; x < n_joined; ++x) before += m_slot[x] == t && m_row[x] < row;
            } else {
#pragma unroll 4
                for (; x + 4 <= e; x += 4) {
                    const int4 v = *reinterpret_cast<const int4*>(m_slot + x);
                    before += (v.x == t) + (v.y == t) + (v.z == t) + (v.w == t);
                }
                for (; x < e; ++x) before += m_slot[x] == t;
            }
            list[start[t] + before] = m_row[e];
        }
    else {
        // The members in row order, kListCap at a time: their slots by all warps but the first, which places the kListCap before them.
        // start[t] moves along and ends up as the end of slot t's members.  (The unit's other CTAs write the same.)
        auto chunk = [&](int b) { return m_row + 2 * kListCap * b; };       // rows, slots
        auto look_up = [&](int e0, int* rows, int first, int step) {
            constexpr int kU = 5;                                   // (224 threads: one round)
            const int n = min(kListCap, nm - e0);
            for (int x0 = first; x0 < n; x0 += kU * step) {
                int row[kU], sd[kU];
                uint8_t kd[kU];
#pragma unroll
                for (int q = 0; q < kU; ++q) row[q] = CASK_IDX(mem_row[o + e0 + min(x0 + q * step, n - 1)], T_, err);
#pragma unroll
                for (int q = 0; q < kU; ++q) { kd[q] = ku[row[q]]; sd[q] = seed_of[o + row[q]]; }
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    const int x = x0 + q * step;
                    if (x >= n) break;
                    rows[x] = row[q];
                    rows[kListCap + x] = slot_of(kd[q] == CASK_KIND_SEED ? row[q] : sd[q]);
                }
            }
        };
        look_up(0, chunk(0), tid, kLongThreads);
        __syncthreads();
        for (int e0 = 0, b = 0; e0 < nm; e0 += kListCap, b ^= 1) {
            if (w > 0) {
                look_up(e0 + kListCap, chunk(b ^ 1), tid - 32, kLongThreads - 32);
            } else {
                const int* rows = chunk(b);
                const int n = min(kListCap, nm - e0);
                for (int x0 = 0; x0 < n; x0 += 32) {
                    const int x = x0 + lane, t = x < n ? rows[kListCap + x] : -1;
                    const unsigned same = __match_any_sync(0xffffffffu, t);
                    const int at = t >= 0 ? start[t] + __popc(same & ((1u << lane) - 1u)) : 0;
                    __syncwarp();
                    if (t >= 0) {
                        mem_slot[o + at] = rows[x];
                        if (lane == 31 - __clz(same)) start[t] = at + 1;
                    }
                    __syncwarp();
                }
            }
            __syncthreads();
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // bulk copies write over the list from here on
    __syncthreads();
    // ---- batches of slots
    const RowSource<T> in{K, V, s, weight, eps, fw, ud, sh, u};
    const int at = in_smem ? 0 : -1;                         // (placed in the workspace: start[t] is the end of slot t's members)
    const int* members = in_smem ? list : mem_slot + o;
    int one = nm > 4 * nk || (nm > 2 * nk && nk < 256 * parts);
    // (Opaque: with the counts in view the compiler makes other code of the whole kernel, 25 % slower at head_dim 64.)
    asm volatile("" : "+r"(one));
    const int per_item = in_smem ? (parts > 1 ? 1 : 4) : (one ? 1 : 8);
    copy_batches<T, CH, kLongStage>(
        in, nk, parts, part, copy_smem, bars, &next_item, &abort_, k_out, v_out, slot_mass, Bmax, err, per_item,
        n_busy, [&](int t) { return src[t] >> 1; }, [&](int t) { return start[t + at]; },
        [&](int e) { return members[e]; }, [&](int i) { return in_smem ? (int)busy[i] : i; });
    late_flags(fw, sh.n_units, err);
}

// ---- host-resident caches: which value rows the compaction will read, and where they sit once packed ----
__global__ void __launch_bounds__(kScanThreads) value_rank_kernel(const UnitDesc* __restrict__ desc,
                                                                  const uint8_t* __restrict__ kind,
                                                                  int32_t* __restrict__ v_pos,
                                                                  int32_t* __restrict__ n_need) {
    __shared__ unsigned wsum[kScanThreads / 32];
    const int u = blockIdx.x;
    const UnitDesc& ud = desc[u];
    const int T = ud.T;
    const int64_t o = ud.tok_off;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int chunk = (T + (int)blockDim.x - 1) / (int)blockDim.x;
    const int b = threadIdx.x * chunk, e = min(T, b + chunk);
    unsigned cnt = 0;
    for (int i = b; i < e; ++i) cnt += (kind[o + i] != CASK_KIND_DROPPED);
    unsigned incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        unsigned v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    unsigned base = 0, total = 0;
    for (int x = 0; x < nw; ++x) {
        if (x < w) base += wsum[x];
        total += wsum[x];
    }
    unsigned rank = base + incl - cnt;
    for (int i = b; i < e; ++i) {
        const bool need = kind[o + i] != CASK_KIND_DROPPED;
        v_pos[o + i] = need ? (int)rank : -1;
        rank += need;
    }
    if (threadIdx.x == 0) n_need[u] = (int)total;
}

// v_base[u] = value rows needed by the units before u: one CTA, every thread a contiguous run of units.
__global__ void __launch_bounds__(1024) value_base_kernel(int n_units, const int32_t* __restrict__ n_need,
                                                          int64_t* __restrict__ v_base) {
    __shared__ int64_t wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per = (n_units + (int)blockDim.x - 1) / (int)blockDim.x;
    const int u0 = min(n_units, (int)threadIdx.x * per), u1 = min(n_units, u0 + per);
    int64_t sum = 0;
    for (int u = u0; u < u1; ++u) sum += n_need[u];
    int64_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    int64_t run = incl - sum;
    for (int x = 0; x < w; ++x) run += wsum[x];
    for (int u = u0; u < u1; ++u) {
        v_base[u] = run;
        run += n_need[u];
    }
}

// Page-locked values: every warp fetches the needed ones of 32 rows over the bus.  A row is a few 16-byte loads side by
// side; eight rows' loads are in flight per warp, so that the bus sees a hundred kilobytes requested at any time.
constexpr int kFetchLoads = 8;
__global__ void __launch_bounds__(256) value_gather_kernel(const UnitDesc* __restrict__ desc, int row_vecs, const uint4* __restrict__ v_host,
                                                           uint4* __restrict__ v_packed, const int32_t* __restrict__ v_pos,
                                                           const int64_t* __restrict__ v_base) {
    __shared__ int2 list[8][32];         // (row, place) of the warp's needed rows
    const int u = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const UnitDesc& ud = desc[u];
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int pos = i < ud.T ? v_pos[ud.tok_off + i] : -1;
    const unsigned need = __ballot_sync(0xffffffffu, pos >= 0);
    if (pos >= 0) list[w][__popc(need & ((1u << lane) - 1u))] = make_int2(i, pos);
    __syncwarp();
    const int n = __popc(need) * row_vecs;
    const uint4* src = v_host + ud.tok_off * row_vecs;
    uint4* dst = v_packed + v_base[u] * row_vecs;
    for (int x0 = lane; x0 < n; x0 += 32 * kFetchLoads) {
        uint4 v[kFetchLoads];
        int to[kFetchLoads];
#pragma unroll
        for (int q = 0; q < kFetchLoads; ++q) {
            const int x = min(x0 + 32 * q, n - 1), r = x / row_vecs, c = x - r * row_vecs;
            const int2 e = list[w][r];
            to[q] = e.y * row_vecs + c;
            v[q] = __ldcs(src + (int64_t)e.x * row_vecs + c);
        }
#pragma unroll
        for (int q = 0; q < kFetchLoads; ++q)
            if (x0 + 32 * q < n) dst[to[q]] = v[q];
    }
}

// ---- 4. paged cache: the compacted rows go back into the unit's own pages, slot t at logical row t ----
template <typename T>
__global__ void __launch_bounds__(256) writeback_kernel(const UnitDesc* __restrict__ desc, Shape sh, int Bmax,
                                                        const int32_t* __restrict__ n_out, const T* __restrict__ k_out,
                                                        const T* __restrict__ v_out, T* __restrict__ k_pool,
                                                        T* __restrict__ v_pool) {
    const int u = blockIdx.y;
    const UnitDesc& ud = desc[u];
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= n_out[u] || t >= ud.T) return;
    const int d = sh.d, nvec = d * (int)sizeof(T) / 16;
    const int64_t dst = paged_row(sh, ud, t) * sh.row_stride;
    const T* ks = k_out + ((size_t)u * Bmax + t) * d;
    const T* vs = v_out + ((size_t)u * Bmax + t) * d;
    for (int x = lane; x < 2 * nvec; x += 32) {
        const bool isv = x >= nvec;
        const int c = isv ? x - nvec : x;
        reinterpret_cast<uint4*>((isv ? v_pool : k_pool) + dst)[c] = reinterpret_cast<const uint4*>(isv ? vs : ks)[c];
    }
}

template <typename T>
cudaError_t run(const Launch& L, const cask_params& prm, const float* s, const uint8_t* kind,
                const int32_t* seed_of, float* weight, const cask_outputs& out, Workspace& ws, const EventFusion* ev) {
    const Shape& sh = L.sh;
    FusedWeights fw{};
    if (ev) fw = FusedWeights{s, ws.grp, ws.mass_fx, ws.njoin, ev->plan, ev->unit_status, ev->lost_mass, ws.err, sh, L.max_m, prm.eps};
    int32_t* const status = ev ? ev->unit_status : nullptr;
    if (L.max_T <= kSmallRows) {
        auto kern = sh.d == 128 ? compact_small_kernel<T, 4> : sh.d == 64 ? compact_small_kernel<T, 2> : compact_small_kernel<T, 0>;
        constexpr int smem = staging_bytes(kSmallStage);
        static_assert(smem <= kMaxSpread, "");
        size_t fixed = 0;
        cudaError_t e = allow_smem(L, kSmemBitCopy + 2 + 3 * (sizeof(T) == 4) + (sh.d == 128 ? 0 : sh.d == 64 ? 1 : 2), kern, kMaxSpread, &fixed);
        if (e != cudaSuccess) return e;
        // as many CTAs per unit as fit the device at once, so that a few units' rows move at more than a few SMs' rate
        const int parts = std::max(1, std::min(8, 3 * (L.sms > 0 ? L.sms : 128) / std::max(sh.n_units, 1)));
        Timed t(L, KID_GATHER_MERGE);
        return launch_dependent(L.stream, kern, sh.n_units * parts, kFusedWarps * 32,
                                spread_smem(L, (int64_t)sh.n_units * parts, fixed, smem), L.desc, sh, (const T*)L.k,
                                (const T*)L.v, kind, seed_of, s, weight, prm.eps, out.Bmax, parts, out.n_out, out.slot_src,
                                out.slot_kind, out.slot_mass, out.assign, (T*)out.k_out, (T*)out.v_out, fw, ws.err);
    }
    const int table = std::min(out.Bmax, std::max(L.max_B, 1));
    if (L.max_T <= kLongMaxRows && table <= kLongMaxSlots) {
        const bool lists = ev && ws.slot_lists;
        auto kern = lists ? (sh.d == 128 ? compact_long_kernel<T, 4, true> : sh.d == 64 ? compact_long_kernel<T, 2, true> : compact_long_kernel<T, 0, true>)
                          : (sh.d == 128 ? compact_long_kernel<T, 4, false> : sh.d == 64 ? compact_long_kernel<T, 2, false> : compact_long_kernel<T, 0, false>);
        const int bit = kSmemBitCopy + 8 + 6 * lists + 3 * (sizeof(T) == 4) + (sh.d == 128 ? 0 : sh.d == 64 ? 1 : 2);
        size_t fixed = 0;
        cudaError_t e = allow_smem(L, bit, kern, std::max(kMaxSpread, long_smem(kLongMaxSlots)), &fixed);
        if (e != cudaSuccess) return e;
        const GivenLists given{ws.n_mem, ws.n_seed, ws.seed_slot, ws.seed_rows, ws.max_B};
        const int per_sm = std::max(1, std::min(3, (int)((227 << 10) / (long_smem(table) + fixed + kReserved))));
        const int parts = std::max(1, std::min(16, per_sm * (L.sms > 0 ? L.sms : 128) / std::max(sh.n_units, 1)));
        Timed t(L, KID_GATHER_MERGE);
        return launch_dependent(L.stream, kern, sh.n_units * parts, kLongThreads,
                                spread_smem(L, (int64_t)sh.n_units * parts, fixed, long_smem(table)), L.desc, sh, (const T*)L.k,
                                (const T*)L.v, kind, seed_of, s, weight, prm.eps, out.Bmax, table, parts, out.n_out, out.slot_src,
                                out.slot_kind, out.slot_mass, out.assign, ws.mem_row, ws.mem_slot, given, (T*)out.k_out,
                                (T*)out.v_out, fw, ws.err);
    }
    cudaError_t e;
    {
        Timed t(L, KID_SLOT_SCAN);
        e = launch_dependent(L.stream, slot_scan_kernel, sh.n_units, kScanThreads, 0, L.desc, kind, seed_of,
                             weight, out.Bmax, out.n_out, out.slot_src, out.slot_kind, out.slot_mass, out.assign, ws.mem_row,
                             ws.mem_slot, ws.n_mem, ws.seed_slot, ws.n_seed, ws.max_B, fw, ws.err);
        if (e != cudaSuccess) return e;
    }
    const int slots = min(out.Bmax, max(L.max_B, 1));
    {
        // the merge kernel overwrites slots the copy kernel wrote: same stream, in order
        Timed t(L, KID_GATHER_MERGE);
        const int sb = std::min(32, (int)(kCopyStageBytes / 2 / (sh.d * sizeof(T))));
        const int64_t batches = (int64_t)sh.n_units * ((slots + sb - 1) / sb);
        const int copy_smem_bytes = kCopyWarps * 2 * kCopyStageBytes;
        e = allow_smem(L, kSmemBitCopy + (sizeof(T) == 4), slot_copy_kernel<T>, copy_smem_bytes);
        if (e != cudaSuccess) return e;
        const int copy_grid = (int)std::min<int64_t>((batches + kCopyWarps - 1) / kCopyWarps, L.sms > 0 ? L.sms : 128);   // one CTA per SM
        e = launch_dependent(L.stream, slot_copy_kernel<T>, std::max(copy_grid, 1), kCopyWarps * 32, copy_smem_bytes, L.desc, sh,
                             (const T*)L.k, (const T*)L.v, s, prm.eps, out.Bmax, slots, out.n_out, out.slot_src, (T*)out.k_out,
                             (T*)out.v_out, out.slot_mass);
        if (e != cudaSuccess) return e;
        auto merge = [&](auto kern, dim3 grid) {
            return launch_dependent(L.stream, kern, grid, 256, 0, L.desc, sh, (const T*)L.k, (const T*)L.v, s, weight, prm.eps,
                                    out.Bmax, ws.seed_slot, ws.n_seed, ws.max_B, ws.mem_row, ws.mem_slot, ws.n_mem, (T*)out.k_out,
                                    (T*)out.v_out, out.slot_mass, status);
        };
        // one warp per representative: on the event path no unit has more than max_m of them (the plan's count);
        // a staged call may be handed any kinds, so there the slot count bounds them
        const int reps = ev ? std::max(L.max_m, 1) : std::min(slots, ws.max_B);
        e = merge(sh.d == 128 ? slot_merge_kernel<T, 4> : sh.d == 64 ? slot_merge_kernel<T, 2> : slot_merge_kernel<T, 0>,
                  dim3((reps + 7) / 8, sh.n_units));
        ++*L.launches;
    }
    return e;
}

}  // namespace

cudaError_t launch_value_ranks(const Launch& L, const uint8_t* kind, int32_t* v_pos, int32_t* n_need, int64_t* v_base) {
    Timed t(L, KID_SLOT_SCAN);
    value_rank_kernel<<<L.sh.n_units, kScanThreads, 0, L.stream>>>(L.desc, kind, v_pos, n_need);
    value_base_kernel<<<1, 1024, 0, L.stream>>>(L.sh.n_units, n_need, v_base);
    ++*L.launches;
    return cudaGetLastError();
}

cudaError_t launch_value_gather(const Launch& L, const void* v_host, void* v_packed, const int32_t* v_pos,
                                const int64_t* v_base) {
    const int row_vecs = L.sh.d * (L.sh.dtype == CASK_DTYPE_BF16 ? 2 : 4) / 16;
    Timed t(L, KID_GATHER_MERGE);
    value_gather_kernel<<<dim3((L.max_T + 255) / 256, L.sh.n_units), 256, 0, L.stream>>>(
        L.desc, row_vecs, (const uint4*)v_host, (uint4*)v_packed, v_pos, v_base);
    return cudaGetLastError();
}

cudaError_t launch_writeback(const Launch& L, const cask_outputs& out, void* k_pool, void* v_pool) {
    const Shape& sh = L.sh;
    const int slots = min(out.Bmax, max(L.max_B, 1));
    const dim3 grid((slots + 7) / 8, sh.n_units);
    Timed t(L, KID_GATHER_MERGE);
    if (sh.dtype == CASK_DTYPE_BF16)
        writeback_kernel<__nv_bfloat16><<<grid, 256, 0, L.stream>>>(L.desc, sh, out.Bmax, out.n_out,
                                                                   (const __nv_bfloat16*)out.k_out, (const __nv_bfloat16*)out.v_out,
                                                                   (__nv_bfloat16*)k_pool, (__nv_bfloat16*)v_pool);
    else
        writeback_kernel<float><<<grid, 256, 0, L.stream>>>(L.desc, sh, out.Bmax, out.n_out, (const float*)out.k_out,
                                                            (const float*)out.v_out, (float*)k_pool, (float*)v_pool);
    return cudaGetLastError();
}

cudaError_t launch_compact(const Launch& L, const cask_params& prm, const float* s, const uint8_t* kind,
                           const int32_t* seed_of, float* weight, const cask_outputs& out, Workspace& ws,
                           const EventFusion* ev) {
    if (L.sh.dtype == CASK_DTYPE_BF16) return run<__nv_bfloat16>(L, prm, s, kind, seed_of, weight, out, ws, ev);
    return run<float>(L, prm, s, kind, seed_of, weight, out, ws, ev);
}

}  // namespace cask
