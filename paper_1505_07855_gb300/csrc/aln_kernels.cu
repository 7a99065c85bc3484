// Search kernels and their launcher.
//
// Both forms answer most reads from seeds (aln_seed.cuh) and search the trees of the
// others.  Plain form: one launch per batch, in which a warp looks up the seeds of its
// reads and then searches one tree a lane.  Persistent form: the seed search, a wider
// one, the D scan of the reads left, and one launch of (SMs x resident blocks) in which
// a lane pulls its next read from a device queue counter, so a few long reads do not
// hold a whole warp's worth of short ones; then the heavy phase.
//
// Stack bound: the match child is pushed below the alternatives, so entries on
// the stack have non-decreasing difference counts from bottom to top and a
// node is only expanded when it is on top; expanding a node with d differences
// adds one entry with d and at most 9 with d+1 (4 mismatches when the read base
// is N, 1 insertion, 4 deletions), and only when no entry with d+1 is on the
// stack.  Hence at most 1 + 9*B entries for budget B; the capacity is chosen
// from z so the overflow flag cannot be raised.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <string>

#include "aln_flat.cuh"
#include "aln_search.cuh"
#include "aln_seed.cuh"

namespace aln {

#ifdef ALN_STATS
// Instrumented build only: event counters of the persistent kernel.
//  0 loop iterations (lane)   1 fetch iterations (lane)   2 Occ fetches
//  3 table fetches            4 warp-level fetch issues    5 lanes at those issues
//  6 reads finished           7 control rounds             8 stack pops
//  9 warp trips                10 live lanes at those trips
// 11 cycles in control         12 cycles in fetch + apply   13 cycles in the hand-over
//    (11-13 measured by lane 0 of each warp between warp re-formations)
__device__ unsigned long long g_stats[16];
#define STAT_ADD(i, v) atomicAdd(&g_stats[i], static_cast<unsigned long long>(v))
#endif

// Whether a search of these limits can be answered from seeds: the derived
// arrays are there, a transcript has one gap at most, and the caller has set no
// bound on the tree search's work (its reports are that search's).
bool seed_supported(const DIndex &X, const SearchParams &p) {
    return X.lo && min(p.max_gapo, p.z) <= 1u && !p.bounded;
}

// One thread per read, the tree search.
template <int STACK_CAP>
__device__ __forceinline__ void plain_tree(const DIndex &X, const ReadBatch &rb, const SearchParams &p, uint32_t r,
                                           uint32_t *sb, uint32_t *sn, aln_read_result *res, aln_hit *hits) {
    const uint32_t m = rb.len[r];
    const uint32_t z = rb.z ? rb.z[r] : p.z;
    const ReadView rv{sb, sn};
    if (m <= ALN_MAX_READ_LEN && m > 0) load_read(rb, rb.offset[r], m, sb, sn);
    Search<STACK_CAP> S;
    S.run(X, rv, m, z, p, res + r, hits + static_cast<uint64_t>(r) * p.hit_cap);
}

template <int STACK_CAP>
__global__ void __launch_bounds__(kThreads) aln_plain_kernel(DIndex X, ReadBatch rb, uint32_t n_reads, SearchParams p,
                                                             aln_read_result *res, aln_hit *hits) {
    __shared__ uint32_t s_bases[kReadWords * kThreads];
    __shared__ uint32_t s_nmask[kMaskWords * kThreads];
    const uint32_t r = blockIdx.x * kThreads + threadIdx.x;
    if (r >= n_reads) return;
    plain_tree<STACK_CAP>(X, rb, p, r, s_bases + threadIdx.x, s_nmask + threadIdx.x, res, hits);
}

// The same after a seed search: a warp answers what it can of its reads (at most 32),
// kPlainLanes lanes a read, and then searches the trees of the others, a lane each,
// on its own, so that some warps search trees while others look up seeds.  It takes
// as many reads as fill the device once, up to 32: a batch of nothing but repeats
// then has as many trees in flight, and as full warps, as without the seed search.
// 400 000 reads of 60 bases out of 30 000 copies take 70.6 ms and 100 000 23.1, where
// blocks of 32 reads whose first threads searched the rest took 112 and 34 and the
// tree search alone takes 66.6 and 24.0; 100 000 reads of 100 bases on 100 Mbp, next
// to none of them left, 0.455 ms (0.475, and 52).  Resident blocks an SM: 5 / 6 / 7 /
// 8 take 76.5 / 70.6 / 69.2 / 70.2 and 27.8 / 23.1 / 25.9 / 27.7 ms for the copies,
// 0.571 / 0.455 / 0.452 / 0.434 for the others.  (With the gapped stage in line as it
// is now, 71.2, 22.4 and 0.415 ms with 6.)
#ifndef ALN_PLAIN_BLOCKS
#define ALN_PLAIN_BLOCKS 6
#endif
constexpr int kPlainLanes = 16, kPlainBlocks = ALN_PLAIN_BLOCKS;
constexpr uint32_t kPlainStep = 32 / kPlainLanes;  // reads a warp takes at once
constexpr uint32_t kPlainTargets = 32, kPlainPlaces = 2048;

template <int STACK_CAP>
__global__ void __launch_bounds__(kThreads, kPlainBlocks) aln_plain_seed_kernel(
    const __grid_constant__ DIndex X, const __grid_constant__ ReadBatch rb, uint32_t n_reads, uint32_t warp_reads,
    const __grid_constant__ SearchParams p, aln_read_result *res, aln_hit *hits) {
    __shared__ SeedRead<kPlainTargets> s_read[kThreads / kPlainLanes];
    __shared__ uint32_t s_bases[kReadWords * kThreads], s_nmask[kMaskWords * kThreads], s_rest[kThreads];
    const uint32_t group = threadIdx.x / kPlainLanes, lane = threadIdx.x & 31u, col = threadIdx.x & ~31u;
    const uint64_t first = (static_cast<uint64_t>(blockIdx.x) * (kThreads / 32) + threadIdx.x / 32) * warp_reads;
    uint32_t left = 0;  // reads in the warp's part of s_rest
    for (uint32_t t = 0; t < warp_reads && first + t < n_reads; t += kPlainStep) {
        const uint64_t r = first + t + group % kPlainStep;
        const bool active = t + group % kPlainStep < warp_reads && r < n_reads;
        const SeedAnswer got = seed_search<kPlainLanes, kPlainTargets, false>(
            X, rb, p, s_read[group], static_cast<uint32_t>(r), active, kPlainPlaces, res, hits);
        const bool rest = active && got != kSeedDone && threadIdx.x % kPlainLanes == 0;
        const unsigned all = __ballot_sync(0xFFFFFFFFu, rest);
        if (rest) s_rest[col + left + __popc(all & ((1u << lane) - 1u))] = static_cast<uint32_t>(r);
        left += __popc(all);
    }
    __syncwarp();
    if (lane < left)
        plain_tree<STACK_CAP>(X, rb, p, s_rest[threadIdx.x], s_bases + threadIdx.x, s_nmask + threadIdx.x, res, hits);
}

#ifndef ALN_PERSISTENT_MIN_BLOCKS
#define ALN_PERSISTENT_MIN_BLOCKS 6  // 6 resident blocks per SM (80 registers, 8 shared stack entries) measured best
#endif

template <int STACK_CAP, int SMEM, bool SCORE>
__global__ void __launch_bounds__(kThreads, ALN_PERSISTENT_MIN_BLOCKS) aln_persistent_kernel(DIndex X, ReadBatch rb, uint32_t n_reads,
                                                                  SearchParams p, aln_read_result *res,
                                                                  aln_hit *hits, uint32_t *queue,
                                                                  const uint32_t *order, const uint2 *dbp,
                                                                  const uint32_t *left) {
    cudaGridDependencySynchronize();
    // after a seed search that left no read, the queue starts at its end
    if (__all_sync(0xFFFFFFFFu, *reinterpret_cast<volatile uint32_t *>(queue) >= n_reads)) return;
    __shared__ uint32_t s_bases[kReadWords * kThreads];
    __shared__ uint32_t s_nmask[kMaskWords * kThreads];
    __shared__ uint4 s_stack[SMEM * kThreads];
    uint32_t *sb = s_bases + threadIdx.x, *sn = s_nmask + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u, warp_col = threadIdx.x & ~31u;
    uint4 stk[STACK_CAP - SMEM], cand[kCandCap];
    FlatLane<STACK_CAP, SMEM, SCORE> L;
    L.sstk = s_stack + threadIdx.x;
    L.stk = stk;
    L.cand = cand;
    L.has_next = false;
    // The reads that a seed search has left are few and heavy: they go to all warps
    // of the grid, and a warp's other lanes help from the start.  (Taken up 32 a warp,
    // 1284 of 50 000 reads of 60 bases out of 3000 copies 5 % apart took the first 41
    // warps 353 ms, where the tree search of all of them takes 46; now 19.  Where three
    // quarters of the lanes would have a read, all take one: 100 000 reads of one letter
    // 4.2 ms, 4.7 shared out.)
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * (kThreads / 32);
    const bool takes = !left || *left >= 24 * warps || lane * warps < *left;
    L.phase = takes ? PH_IDLE : PH_FREE;
    L.r = 0xFFFFFFFFu;
    L.sp = 0;
    L.base = 0;
    L.K = X.kmer_k;
    L.role = ROLE_OWN;
    L.owner = lane;
    L.outstanding = 0;
    L.heavy_seen = false;
    L.nc = 0;
    L.flags = 0;
    L.own_rv = ReadView{sb, sn};
    L.rv = L.own_rv;
#ifdef ALN_STATS
    unsigned long long st_it = 0, st_f = 0, st_occ = 0, st_tab = 0, st_wi = 0, st_wl = 0, st_wa = 0, st_wal = 0;
    unsigned long long st_cc = 0, st_cf = 0, st_ce = 0;
#endif
    // All 32 lanes of the warp stay in the loop until every lane is free and the
    // queue is empty; each trip is: control, one converged fetch, the hand-over.
    // The trip count is warp-uniform; at p.loop_limit trips the warp stops and
    // flags what it has not finished (stop_at_limit).
    bool at_limit = false;
    for (unsigned long long it = 0;; it++) {
        if (it >= p.loop_limit) {
            at_limit = true;
            break;
        }
        FetchReq fr;
#ifdef ALN_STATS
        const unsigned long long k0 = clock64();
#endif
        L.control(X, rb, n_reads, p, res, hits, queue, order, dbp, sb, sn, fr);
        __syncwarp();
#ifdef ALN_STATS
        const unsigned long long k1 = clock64();
#endif
#ifdef ALN_STATS
        st_it++;
        {
            const unsigned busy = __ballot_sync(0xFFFFFFFFu, L.phase != PH_FREE);
            if (lane == 0) {
                st_wa++;
                st_wal += __popc(busy);
            }
        }
#endif
        if (fr.kind != F_NONE) {
#ifdef ALN_STATS
            const unsigned am = __activemask();
            st_f++;
            st_occ += fr.kind == F_OCC;
            st_tab += fr.kind == F_TABLE;
            if (lane == __ffs(am) - 1) {
                st_wi++;
                st_wl += __popc(am);
            }
#endif
            uint32_t lo4[4], hi4[4];
            fetch4(X, fr, lo4, hi4);
            L.apply(X, lo4, hi4);
        }
#ifdef ALN_STATS
        __syncwarp();
        const unsigned long long k2 = clock64();
#endif
        L.exchange(lane, s_bases, s_nmask, warp_col, p.help_after);
#ifdef ALN_STATS
        if (lane == 0) {
            st_cc += k1 - k0;
            st_cf += k2 - k1;
            st_ce += clock64() - k2;
        }
#endif
        if (!__any_sync(0xFFFFFFFFu, L.phase != PH_FREE)) break;
    }
    if (at_limit) L.stop_at_limit(lane, n_reads, p, res, queue, order);
#ifdef ALN_STATS
    STAT_ADD(0, st_it); STAT_ADD(1, st_f); STAT_ADD(2, st_occ); STAT_ADD(3, st_tab);
    STAT_ADD(4, st_wi); STAT_ADD(5, st_wl); STAT_ADD(6, L.st_reads); STAT_ADD(7, L.st_rounds);
    STAT_ADD(8, L.st_pops); STAT_ADD(9, st_wa); STAT_ADD(10, st_wal);
    STAT_ADD(11, st_cc); STAT_ADD(12, st_cf); STAT_ADD(13, st_ce);
#endif
}

// ---------------------------------------------------------------- heavy phase
//
// Reads whose owner lane passed heavy_after expansions were handed over by the
// persistent search (kFlagDemoted) and are searched here by every lane of the
// GPU, one deepening pass per launch: a pass's subtrees are tasks in a ring in
// global memory; a lane takes a task, searches it depth first (sharing it with
// the idle lanes of its warp exactly as the persistent search does), gives its
// bottom stack entries back to the ring while the ring runs low, and merges the
// candidates it found into the read's hash table (least witness per interval by
// atomicMin).  After each pass one block per read applies the iterative
// deepening rule to the table and either writes the result or starts the next
// pass.  The hit set, witnesses and counts are those of the other forms.

__device__ __forceinline__ unsigned long long global_ns() {  // the GPU's nanosecond timer
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t vload(const uint32_t *p) { return *reinterpret_cast<const volatile uint32_t *>(p); }

// Task t is published once its slot is written: ready[t % cap] = t + 1.
__device__ __forceinline__ void heavy_push(const HeavyCtx &H, const uint4 &node, uint32_t hid, uint32_t s) {
    atomicAdd(&H.hdr->outstanding, 1u);
    const uint32_t t = atomicAdd(&H.hdr->tail, 1u);
    HeavyTask task;
    task.node = node;
    task.hid = hid;
    task.s = s;
    task.pad0 = task.pad1 = 0;
    H.pool[t % kHeavyPool] = task;
    __threadfence();
    atomicExch(&H.ready[t % kHeavyPool], t + 1u);
}

__device__ __forceinline__ unsigned long long mix_id(unsigned long long x) {
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdULL;
    x ^= x >> 33;
    return x;
}

// Insert candidate (lo, hi) of strand s with witness key; returns false if the
// read's table for that strand is full.
__device__ bool heavy_insert(const HeavyCtx &H, uint32_t hid, uint32_t s, uint32_t lo, uint32_t hi, uint32_t key,
                             uint32_t score) {
    HeavySlot *T = H.slots + (static_cast<uint64_t>(hid) * 2 + s) * kHeavySlots;
    const unsigned long long id = (static_cast<unsigned long long>(lo) << 32) | hi;
    uint32_t j = static_cast<uint32_t>(mix_id(id)) & (kHeavySlots - 1);
    const unsigned long long wkey = (static_cast<unsigned long long>(score) << 32) | key;
    // Many lanes insert the same few intervals of a repeat-rich read: a plain
    // read first skips the atomics that would change nothing.  Safe with a stale
    // value: a slot's id only goes from 0 to its final value, and its key only
    // decreases, so a stale read can only cause an atomic, never skip one that
    // was needed.
    for (uint32_t probe = 0; probe < kHeavySlots; probe++, j = (j + 1) & (kHeavySlots - 1)) {
        unsigned long long cur = __ldcg(&T[j].id);
        if (cur == 0ull) {
            cur = atomicCAS(&T[j].id, 0ull, id);
            if (cur == 0ull) {
                atomicMin(&T[j].wkey, wkey);
                atomicAdd(&H.reads[hid].distinct[s], 1u);
                return true;
            }
        }
        if (cur == id) {
            if (__ldcg(&T[j].wkey) > wkey) atomicMin(&T[j].wkey, wkey);
            return true;
        }
    }
    return false;
}

// One block per handed-over read: cleared tables and the root of each strand
// the lower bound admits as a task, for the deepening pass the read was in when
// it was handed over (R->B, written by its lane).  Each pass starts from the
// root with no candidates, so the passes before it need not be searched again.
__device__ void heavy_start_one(const HeavyCtx &H, uint32_t hid, const uint2 *dbp, uint32_t n_text) {
    HeavySlot *T = H.slots + static_cast<uint64_t>(hid) * 2 * kHeavySlots;
    for (uint32_t j = threadIdx.x; j < 2 * kHeavySlots; j += blockDim.x) {
        T[j].id = 0ull;
        T[j].wkey = ~0ull;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        HeavyRead *R = H.reads + hid;
        const uint2 a = dbp[2ull * R->r], b = dbp[2ull * R->r + 1];
        const uint32_t d0 = d_at(a.x, a.y, 0), d1 = d_at(b.x, b.y, 0);
        R->state = 0;
        R->flags = 0;
        R->distinct[0] = R->distinct[1] = 0;
        const uint4 root = make_uint4(0, n_text + 1, pack_info(0, 0, 0, 0, 0, 0, OP_M), 0);
        if (d0 <= R->B) heavy_push(H, root, hid, 0);
        if (d1 <= R->B) heavy_push(H, root, hid, 1);
    }
}

// Blocks of the start and decide kernels per SM: a call without heavy reads, the
// usual one, only pays for launching them (1.3 us with 1 or 2 blocks an SM, 1.4 with
// 4, 2.1 with one a possible read, 2048); clearing the tables of 2048 heavy reads
// takes 41 / 25 / 20 / 15 us, writing their results 110 us with 2, 90 with 4.
constexpr uint32_t kHeavyBlocksPerSm = 2;

__global__ void aln_heavy_start_kernel(SearchParams p, const uint2 *dbp, uint32_t n_text) {
    cudaGridDependencySynchronize();
    const uint32_t n = min(p.heavy.hdr->n_heavy, kHeavyReads);
    for (uint32_t hid = blockIdx.x; hid < n; hid += gridDim.x) {
        heavy_start_one(p.heavy, hid, dbp, n_text);
        __syncthreads();
    }
}

template <int STACK_CAP, bool SCORE>
__device__ __forceinline__ void heavy_pass(const DIndex &X, const ReadBatch &rb, const SearchParams &p,
                                           const uint2 *dbp) {
    constexpr int SMEM = kSmemStackDefault;
    __shared__ uint32_t s_bases[kReadWords * kThreads];
    __shared__ uint32_t s_nmask[kMaskWords * kThreads];
    __shared__ uint4 s_stack[SMEM * kThreads];
    const HeavyCtx H = p.heavy;
    uint32_t *sb = s_bases + threadIdx.x, *sn = s_nmask + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u, warp_col = threadIdx.x & ~31u;
    const unsigned FULL = 0xFFFFFFFFu;
    uint4 stk[STACK_CAP - SMEM], cand[kCandCap];
    FlatLane<STACK_CAP, SMEM, SCORE> L;
    L.sstk = s_stack + threadIdx.x;
    L.stk = stk;
    L.cand = cand;
    L.has_next = false;
    L.phase = PH_IDLE;
    L.r = 0;
    L.sp = 0;
    L.base = 0;
    L.K = X.kmer_k;
    L.role = ROLE_OWN;
    L.owner = lane;
    L.outstanding = 0;
    L.heavy_seen = false;
    L.nc = 0;
    L.flags = 0;
    L.own_rv = ReadView{sb, sn};
    L.rv = L.own_rv;
    uint32_t hid = 0;
    const uint32_t n_heavy = min(vload(&H.hdr->n_heavy), kHeavyReads);
    if (n_heavy == 0) return;
    // Ring entries kept available: one per warp of the grid, so that owners
    // split their subtrees only while lanes wait for work (a mark of two per
    // lane cut them into tasks of about 128 expansions and ran longer).  The
    // ring then holds at most low_water + 32 per warp, within its capacity
    // (the launch bounds the grid).
    const uint32_t low_water = gridDim.x * (kThreads / 32u);
    // consecutive trips with no lane of the warp at work, and since when (warp-uniform)
    uint32_t idle_trips = 0;
    unsigned long long idle_since = 0;
    bool idle_expired = false;
    uint32_t trips = 0, busy = 0;  // this lane's trips, and those it spent on a task
    for (unsigned long long it = 0;; it++) {
        if (it >= p.loop_limit || idle_expired) {  // guard: unfinished tasks mark their reads, the warp stops
            if (lane == 0 && p.status) atomicOr(p.status, ALN_STATUS_LOOP_LIMIT);
            if (L.role == ROLE_OWN && L.phase != PH_IDLE && L.phase != PH_FREE)
                atomicOr(&H.reads[hid].flags, ALN_FLAG_LOOP_LIMIT);
            break;
        }
        FetchReq fr;
        fr.kind = F_NONE;
        trips++;
        busy += (L.phase != PH_IDLE && L.phase != PH_FREE) ? 1u : 0u;
        // control: advance the lane's task until it needs four extensions
        for (int round = 0; round < 32; round++) {
            if (L.phase == PH_FREE || L.phase == PH_RETURN || L.phase == PH_IDLE) break;
            if (L.phase == PH_WAIT) {
                if (L.outstanding) break;
                L.phase = PH_DFS;
            }
            if (!L.has_next && L.sp == L.base) {
                L.sp = L.base = 0;
                if (L.role == ROLE_HELP) {
                    L.phase = PH_RETURN;
                    L.ret_i = 0;
                    break;
                }
                if (L.outstanding) {
                    L.phase = PH_WAIT;
                    break;
                }
                // task done: its candidates into the read's table, then the next task
                uint32_t f = L.flags & ALN_FLAG_INCOMPLETE;
                for (uint32_t j = 0; j < L.nc; j++) {
                    const uint4 c = L.cand[j];
                    if (!heavy_insert(H, hid, c.z >> 31, c.x, c.y, c.z, c.w)) f |= ALN_FLAG_CAND_OVERFLOW;
                }
                if (f) atomicOr(&H.reads[hid].flags, f);
                atomicAdd(&H.hdr->expansions, static_cast<unsigned long long>(L.work));
                atomicSub(&H.hdr->outstanding, 1u);
                L.phase = PH_IDLE;
                break;
            }
            if (++L.work > p.work_limit) {
                L.flags |= ALN_FLAG_WORK_LIMIT;
                L.sp = L.base;
                L.has_next = false;
                continue;
            }
            if (L.expand_top(p, fr)) break;
        }
        __syncwarp();
        if (fr.kind != F_NONE) {
            uint32_t lo4[4], hi4[4];
            fetch4(X, fr, lo4, hi4);
            L.apply(X, lo4, hi4);
        }
        // the ring runs low: lanes give their bottom stack entries back to it (its
        // level read by one lane, the tickets taken once per warp); helpers too,
        // or the subtrees a warp's idle lanes take from its owners could never
        // reach other warps (L.r holds the read's list entry either way)
        const bool can_push = L.phase == PH_DFS && (L.sp - L.base >= 2 || (L.sp - L.base >= 1 && L.has_next));
        const unsigned pushers = __ballot_sync(FULL, can_push);
        if (pushers) {
            const uint32_t src = __ffs(pushers) - 1;
            uint32_t t0 = 0xFFFFFFFFu;
            if (lane == src && vload(&H.hdr->tail) - vload(&H.hdr->head) < low_water) {
                atomicAdd(&H.hdr->outstanding, static_cast<uint32_t>(__popc(pushers)));  // before publishing
                t0 = atomicAdd(&H.hdr->tail, static_cast<uint32_t>(__popc(pushers)));
            }
            t0 = __shfl_sync(FULL, t0, src);
            if (t0 != 0xFFFFFFFFu && can_push) {
                const uint32_t t = t0 + __popc(pushers & ((1u << lane) - 1u));
                const uint4 e = L.stk_get(L.base);
                L.base++;
                HeavyTask task;
                task.node = e;
                task.hid = L.r;
                task.s = L.s;
                task.pad0 = task.pad1 = 0;
                H.pool[t % kHeavyPool] = task;
                __threadfence();
                atomicExch(&H.ready[t % kHeavyPool], t + 1u);
            }
        }
        // a helper merges its candidates into the read's table itself: the
        // hand-back through the owner moves one per trip, and a subtree of a
        // repeat-rich read can hold hundreds
        if (L.phase == PH_RETURN && L.ret_i < L.nc) {
            uint32_t f = 0;
            for (uint32_t j = L.ret_i; j < L.nc; j++) {
                const uint4 c = L.cand[j];
                if (!heavy_insert(H, L.r, c.z >> 31, c.x, c.y, c.z, c.w)) f |= ALN_FLAG_CAND_OVERFLOW;
            }
            if (f) atomicOr(&H.reads[L.r].flags, f);
            L.ret_i = L.nc;
        }
        L.exchange(lane, s_bases, s_nmask, warp_col, 0u);
        // idle lanes take tasks from the ring, one claim per warp
        const unsigned idle = __ballot_sync(FULL, L.phase == PH_IDLE);
        if (idle) {
            const uint32_t leader = __ffs(idle) - 1;
            uint32_t first = 0, got = 0;
            if (lane == leader) {
                const uint32_t want = __popc(idle);
                uint32_t h = vload(&H.hdr->head);
                for (int tries = 0; tries < 64; tries++) {
                    const uint32_t t = vload(&H.hdr->tail);
                    const int avail = static_cast<int>(t - h);
                    if (avail <= 0) break;
                    const uint32_t g = min(want, static_cast<uint32_t>(avail));
                    const uint32_t old = atomicCAS(&H.hdr->head, h, h + g);
                    if (old == h) {
                        first = h;
                        got = g;
                        break;
                    }
                    h = old;
                }
            }
            first = __shfl_sync(FULL, first, leader);
            got = __shfl_sync(FULL, got, leader);
            const uint32_t rank = __popc(idle & ((1u << lane) - 1u));
            if (L.phase == PH_IDLE) {
                if (rank < got) {
                    const uint32_t t = first + rank;
                    uint32_t spins = 0;
                    while (vload(&H.ready[t % kHeavyPool]) != t + 1u && spins < (1u << 22)) spins++;
                    if (spins >= (1u << 22)) {  // a published task that never appeared: give up
                        if (p.status) atomicOr(p.status, ALN_STATUS_LOOP_LIMIT);
                        L.phase = PH_FREE;
                    } else {
                        __threadfence();  // the task's slot was written before its ready word
                        const HeavyTask *slot = H.pool + (t % kHeavyPool);
                        HeavyTask task;
                        task.node = __ldcg(&slot->node);
                        task.hid = __ldcg(&slot->hid);
                        task.s = __ldcg(&slot->s);
                        hid = task.hid;
                        const HeavyRead R = H.reads[hid];
                        L.r = hid;  // the list entry (a helper gets it with the subtree)
                        L.m = R.m;
                        L.z = R.z;
                        L.B = R.B;
                        L.s = task.s;
                        load_read(rb, rb.offset[R.r], R.m, sb, sn);
                        const uint2 bp = dbp[2ull * R.r + task.s];
                        if (task.s) {
                            L.bpb0 = bp.x;
                            L.bpb1 = bp.y;
                        } else {
                            L.bpa0 = bp.x;
                            L.bpa1 = bp.y;
                        }
                        L.rv = L.own_rv;
                        L.role = ROLE_OWN;
                        L.next = task.node;
                        L.has_next = true;
                        L.sp = L.base = 0;
                        L.nc = 0;
                        L.work = 0;
                        L.flags = 0;
                        L.outstanding = 0;
                        L.phase = PH_DFS;
                    }
                } else if (got == 0 && vload(&H.hdr->outstanding) == 0) {
                    L.phase = PH_FREE;  // the pass is over
                }
            }
            if (__ballot_sync(FULL, L.phase != PH_IDLE && L.phase != PH_FREE) == 0) {
                // back off (0.25 to 16 us) so that idle warps leave the ring's
                // counters to the lanes that publish and take tasks; 4 s without
                // work ends the warp (a task that never came)
                const unsigned long long now = global_ns();
                if (idle_trips == 0) idle_since = now;
                idle_expired = __shfl_sync(FULL, now - idle_since > 4000000000ull ? 1u : 0u, 0) != 0;
                __nanosleep(256u << min(idle_trips, 6u));
                idle_trips++;
            } else {
                idle_trips = 0;
            }
        } else {
            idle_trips = 0;
        }
        if (__ballot_sync(FULL, L.phase != PH_FREE) == 0) break;
    }
    const uint32_t wt = __reduce_add_sync(FULL, trips), wb = __reduce_add_sync(FULL, busy);
    if (lane == 0) {
        atomicAdd(&H.hdr->lane_trips, static_cast<unsigned long long>(wt));
        atomicAdd(&H.hdr->busy_trips, static_cast<unsigned long long>(wb));
    }
}

template <int STACK_CAP, bool SCORE>
__global__ void __launch_bounds__(kThreads, ALN_PERSISTENT_MIN_BLOCKS) aln_heavy_pass_kernel(DIndex X, ReadBatch rb,
                                                                                           SearchParams p,
                                                                                           const uint2 *dbp) {
    cudaGridDependencySynchronize();
    heavy_pass<STACK_CAP, SCORE>(X, rb, p, dbp);
}

// Result of a handed-over read from its tables, by the threads of a block: hits of
// value v (diffs, at most fin, or in the score-ordered mode the score) listed in the
// order (v, strand, k, l), counted in the strata of the least value and the one after
// it.  A thread places a hit by the number of listed hits before it, so a read of
// n listed hits takes n / 128 rounds over them.  (One thread, searching the 2048
// slots for each hit in turn, took 8.9 ms for 2048 reads, a block each, and 11.4 ms
// on 152 blocks; this takes 0.11 ms on 304.)
__device__ void heavy_write(const SearchParams &p, const HeavySlot *T, const HeavyRead *R, uint32_t fin,
                            aln_read_result *res, aln_hit *hits) {
    constexpr uint32_t kSlots = 2 * kHeavySlots;
    const bool score = p.strata == ALN_STRATA_SCORE;
    __shared__ uint32_t s_1, s_2, s_best, s_kept;     // least value, the next one, fewest diffs at the least, hits listed
    __shared__ unsigned long long s_c0, s_c1;         // widths at the two values
    __shared__ uint16_t s_slot[kSlots];               // the listed hits' slots
    auto value = [&](unsigned long long wkey) {
        return score ? static_cast<uint32_t>(wkey >> 32) : (static_cast<uint32_t>(wkey) >> 28) & 7u;
    };
    if (threadIdx.x == 0) {
        s_1 = s_2 = 0xFFFFFFFFu;
        s_best = 255;
        s_kept = 0;
        s_c0 = s_c1 = 0;
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < kSlots; j += blockDim.x)
        if (T[j].id && (score || value(T[j].wkey) <= fin)) atomicMin(&s_1, value(T[j].wkey));
    __syncthreads();
    if (score) {
        for (uint32_t j = threadIdx.x; j < kSlots; j += blockDim.x)
            if (T[j].id && value(T[j].wkey) > s_1) atomicMin(&s_2, value(T[j].wkey));
    } else if (threadIdx.x == 0 && s_1 < fin) {
        s_2 = s_1 + 1;
    }
    __syncthreads();
    const uint32_t v1 = s_1, v2 = s_2;
    for (uint32_t j = threadIdx.x; j < kSlots; j += blockDim.x) {
        if (!T[j].id) continue;
        const uint32_t v = value(T[j].wkey);
        const unsigned long long w = (T[j].id & 0xFFFFFFFFull) - (T[j].id >> 32);
        if (v == v1) {
            atomicAdd(&s_c0, w);
            atomicMin(&s_best, (static_cast<uint32_t>(T[j].wkey) >> 28) & 7u);
        } else if (v == v2) {
            atomicAdd(&s_c1, w);
        }
    }
    __syncthreads();
    const bool many = score && p.max_best && s_c0 > p.max_best;
    for (uint32_t j = threadIdx.x; j < kSlots; j += blockDim.x) {
        if (!T[j].id) continue;
        const uint32_t v = value(T[j].wkey);
        if (score ? v == v1 || (!many && v == v2) : v <= fin) s_slot[atomicAdd(&s_kept, 1u)] = static_cast<uint16_t>(j);
    }
    __syncthreads();
    const uint32_t kept = s_kept, nout = min(kept, p.hit_cap);
    for (uint32_t i = threadIdx.x; i < kept; i += blockDim.x) {
        const HeavySlot e = T[s_slot[i]];
        const uint32_t key = static_cast<uint32_t>(e.wkey), o = (value(e.wkey) << 1) | (key >> 31);
        uint32_t before = 0;
        for (uint32_t j = 0; j < kept && before < nout; j++) {
            const HeavySlot f = T[s_slot[j]];
            const uint32_t fo = (value(f.wkey) << 1) | (static_cast<uint32_t>(f.wkey) >> 31);
            before += fo < o || (fo == o && f.id < e.id) ? 1u : 0u;
        }
        if (before < nout)
            put_hit(hits + static_cast<uint64_t>(R->r) * p.hit_cap + before, static_cast<uint32_t>(e.id >> 32),
                    static_cast<uint32_t>(e.id) - 1u, key);
    }
    if (threadIdx.x == 0) {
        const bool any = kept > 0;
        aln_read_result out;
        out.c0 = static_cast<uint32_t>(min(any ? s_c0 : 0ull, 0xFFFFFFFFull));
        out.c1 = static_cast<uint32_t>(min(any ? s_c1 : 0ull, 0xFFFFFFFFull));
        out.d_best = static_cast<uint8_t>(any ? s_best : 255u);
        out.best_score = static_cast<uint8_t>(score ? (any ? min(v1, 254u) : 255u) : 0u);
        out.n_hits = static_cast<uint8_t>(nout);
        out.flags = static_cast<uint8_t>((R->flags & 0xFFu) | (many ? ALN_FLAG_MANY_BEST : 0u) |
                                         (kept > p.hit_cap ? ALN_FLAG_HIT_OVERFLOW : 0u));
        res[R->r] = out;
    }
}

// One block per handed-over read after a pass: the iterative deepening rule on
// its table; the result, or the next pass's budget, cleared tables and roots.
__device__ void heavy_decide_one(const SearchParams &p, uint32_t hid, const uint2 *dbp, uint32_t n_text,
                                 aln_read_result *res, aln_hit *hits, int last) {
    const HeavyCtx H = p.heavy;
    HeavyRead *R = H.reads + hid;
    if (R->state != 0) return;
    HeavySlot *T = H.slots + static_cast<uint64_t>(hid) * 2 * kHeavySlots;
    __shared__ uint32_t s_dmin, s_n;
    __shared__ uint32_t s_next;  // 0 finish, else the next pass budget
    __shared__ uint32_t s_final;
    if (threadIdx.x == 0) {
        s_dmin = 255;
        s_n = 0;
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < 2 * kHeavySlots; j += blockDim.x)
        if (T[j].id) {
            atomicMin(&s_dmin, (static_cast<uint32_t>(T[j].wkey) >> 28) & 7u);
            atomicAdd(&s_n, 1u);
        }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t z = R->z, B = R->B;
        uint32_t next = 0, fin = 0;
        if (s_n > static_cast<uint32_t>(kCandCap)) R->flags |= ALN_FLAG_CAND_OVERFLOW;
        if ((R->flags & ALN_FLAG_INCOMPLETE) || p.strata != ALN_STRATA_BEST1) {
            fin = z;
        } else if (s_n == 0) {
            if (B < z) next = min(z, B + 2);
            fin = 0;
        } else {
            const uint32_t F = min(z, s_dmin + 1);
            if (F <= B) fin = F;
            else next = F;
        }
        if (next && last) {  // cannot happen within kHeavyPasses passes; leave no read without a result
            R->flags |= ALN_FLAG_LOOP_LIMIT;
            next = 0;
            fin = B;
        }
        s_next = next;
        s_final = fin;
    }
    __syncthreads();
    if (s_next) {  // next pass: clear the tables, then the roots
        for (uint32_t j = threadIdx.x; j < 2 * kHeavySlots; j += blockDim.x) {
            T[j].id = 0ull;
            T[j].wkey = ~0ull;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            R->B = s_next;
            R->distinct[0] = R->distinct[1] = 0;
            const uint2 a = dbp[2ull * R->r], b = dbp[2ull * R->r + 1];
            const uint4 root = make_uint4(0, n_text + 1, pack_info(0, 0, 0, 0, 0, 0, OP_M), 0);
            if (d_at(a.x, a.y, 0) <= s_next) heavy_push(H, root, hid, 0);
            if (d_at(b.x, b.y, 0) <= s_next) heavy_push(H, root, hid, 1);
        }
        return;
    }
    heavy_write(p, T, R, s_final, res, hits);
    if (threadIdx.x == 0) R->state = 1;
}

__global__ void aln_heavy_decide_kernel(SearchParams p, const uint2 *dbp, uint32_t n_text, aln_read_result *res,
                                        aln_hit *hits, int last) {
    cudaGridDependencySynchronize();
    const uint32_t n = min(p.heavy.hdr->n_heavy, kHeavyReads);
    for (uint32_t hid = blockIdx.x; hid < n; hid += gridDim.x) {
        heavy_decide_one(p, hid, dbp, n_text, res, hits, last);
        __syncthreads();
    }
}

// The whole phase in one cooperative launch, a grid barrier where the kernels
// above follow each other: for a call of at most kHeavyReads reads, whose time is
// that of its launches when, as usual, no read is heavy (64 reads take 29 us so, 47
// with the eleven kernels).
template <int STACK_CAP, bool SCORE>
__global__ void __launch_bounds__(kThreads, ALN_PERSISTENT_MIN_BLOCKS) aln_heavy_all_kernel(
    DIndex X, ReadBatch rb, SearchParams p, const uint2 *dbp, aln_read_result *res, aln_hit *hits) {
    const uint32_t n = min(p.heavy.hdr->n_heavy, kHeavyReads);  // no kernel of the phase changes it
    if (n == 0) return;
    const cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    for (uint32_t hid = blockIdx.x; hid < n; hid += gridDim.x) {
        heavy_start_one(p.heavy, hid, dbp, X.t[0].n);
        __syncthreads();
    }
    for (uint32_t pass = 0; pass < kHeavyPasses; pass++) {
        grid.sync();
        heavy_pass<STACK_CAP, SCORE>(X, rb, p, dbp);
        grid.sync();
        for (uint32_t hid = blockIdx.x; hid < n; hid += gridDim.x) {
            heavy_decide_one(p, hid, dbp, X.t[0].n, res, hits, pass + 1 == kHeavyPasses ? 1 : 0);
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------- end of the heavy phase

#ifdef ALN_STATS
cudaError_t debug_stats(unsigned long long *out, int reset) {
    cudaError_t e = cudaMemcpyFromSymbol(out, g_stats, sizeof(g_stats));
    if (e == cudaSuccess && reset) {
        unsigned long long z[16] = {};
        e = cudaMemcpyToSymbol(g_stats, z, sizeof(z));
    }
    return e;
}
#endif

// D-array pre-pass.  Thread t runs the greedy D scan of strand t & 1 of read
// t >> 1 on that strand's other index (strand 0 on X, strand 1 on X reversed)
// and stores its breakpoints; reads the search would flag before any scan get
// zeros.  The persistent search then starts from these instead of scanning.
__device__ __forceinline__ void dscan_one(const DIndex &X, const ReadBatch &rb, const SearchParams &p, uint32_t r,
                                          uint32_t s, uint32_t *sb, uint32_t *sn, uint2 *dbp) {
    const uint32_t m = rb.len[r];
    const uint32_t z = rb.z ? rb.z[r] : p.z;
    uint2 out = make_uint2(0u, 0u);
    if (m >= 1 && m <= ALN_MAX_READ_LEN && z <= ALN_MAX_Z && z <= p.z) {
        load_read(rb, rb.offset[r], m, sb, sn);
        const ReadView rv{sb, sn};
        d_scan(X.t[s], rv, m, s, min(z + 1, 8u), out.x, out.y);
    }
    dbp[2ull * r + s] = out;
}

__global__ void __launch_bounds__(kThreads) aln_dscan_kernel(DIndex X, ReadBatch rb, uint32_t n, SearchParams p,
                                                             uint2 *dbp) {
    __shared__ uint32_t s_bases[kReadWords * kThreads];
    __shared__ uint32_t s_nmask[kMaskWords * kThreads];
    const uint64_t t = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x;
    if (t >= 2ull * n) return;
    dscan_one(X, rb, p, static_cast<uint32_t>(t >> 1), static_cast<uint32_t>(t & 1u), s_bases + threadIdx.x,
              s_nmask + threadIdx.x, dbp);
}

// ---------------------------------------------------------------- seed search
//
// aln_seed_kernel answers the reads whose parts lead to few places (see
// aln_seed.cuh), G lanes a read; aln_seed_wide_kernel takes the reads it leaves for more lanes,
// a warp each with room for kCandCap targets; aln_dscan_list_kernel scans the D
// arrays of what is left then, which the persistent search and the heavy phase
// search as before: the rest fills the visit order from its end, and the queue
// starts where it begins.  The lists and their counts stay on the device.

struct SeedCounts {          // in the scratch's first words, cleared before the call's kernels
    uint32_t wide, taken;    // reads left by the first kernel; those the second has taken up
    uint32_t rest;           // reads left for the tree search
};

// Room for targets and places to look at, first for a read's 8 or 16 lanes: past
// that the other reads of the warp wait for it, so it goes to a warp of its own
// (300 000 mates on 3.1 Gbp: 6.96 / 5.91 / 5.36 ms with 1024 / 256 / 64 places).
// There, kCandCap targets are what the tree search keeps.
constexpr uint32_t kSeedTargets = 32;
#ifndef ALN_SEED_PLACES
#define ALN_SEED_PLACES 64
#endif
constexpr uint32_t kSeedPlaces = ALN_SEED_PLACES;

// Resident blocks per SM: 4 / 5 / 6 take 3.39 / 3.11 / 3.00 ms for 1 M reads of 100
// bases on 100 Mbp and 5.85 / 5.48 / 5.36 ms for 300 000 mates on 3.1 Gbp (latency; 6
// spills in the gapped path); the wide kernel is the same with 4 and 5.
#ifndef ALN_SEED_MIN_BLOCKS
#define ALN_SEED_MIN_BLOCKS 6
#endif
#ifndef ALN_WIDE_MIN_BLOCKS
#define ALN_WIDE_MIN_BLOCKS 5
#endif

template <int G, bool SCORE>
__global__ void __launch_bounds__(kThreads, ALN_SEED_MIN_BLOCKS) aln_seed_kernel(const __grid_constant__ DIndex X, ReadBatch rb, uint32_t n, const __grid_constant__ SearchParams p,
                                                            aln_read_result *res, aln_hit *hits, SeedCounts *counts,
                                                            uint32_t *wide, uint32_t *order_end) {
    __shared__ SeedRead<kSeedTargets> s_read[kThreads / G];
    if (blockIdx.x == 0) {  // what the later kernels report and count in
        if (p.status && threadIdx.x == 0) *p.status = 0;
        if (p.heavy.hdr && threadIdx.x < sizeof(HeavyHdr) / 4)
            reinterpret_cast<uint32_t *>(p.heavy.hdr)[threadIdx.x] = 0;
    }
    const uint64_t r = (static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x) / G;
    const bool active = r < n;
    const SeedAnswer got = seed_search<G, kSeedTargets, SCORE>(X, rb, p, s_read[threadIdx.x / G],
                                                               static_cast<uint32_t>(r), active, kSeedPlaces, res, hits);
    if (active && got != kSeedDone && (threadIdx.x & (G - 1)) == 0) {
        if (got == kSeedTree) *(order_end - 1 - atomicAdd(&counts->rest, 1u)) = static_cast<uint32_t>(r);
        else wide[atomicAdd(&counts->wide, 1u)] = static_cast<uint32_t>(r);
    }
}

template <bool SCORE>
__global__ void __launch_bounds__(kThreads, ALN_WIDE_MIN_BLOCKS) aln_seed_wide_kernel(const __grid_constant__ DIndex X, ReadBatch rb, const __grid_constant__ SearchParams p,
                                                                 aln_read_result *res, aln_hit *hits,
                                                                 SeedCounts *counts, const uint32_t *wide,
                                                                 uint32_t *order_end) {
    __shared__ SeedRead<kCandCap> s_read[kThreads / 32];
    cudaGridDependencySynchronize();
    const uint32_t lane = threadIdx.x & 31u, n = counts->wide;
    for (;;) {
        uint32_t i = 0;
        if (lane == 0) i = atomicAdd(&counts->taken, 1u);
        i = __shfl_sync(0xFFFFFFFFu, i, 0);
        if (i >= n) break;
        const uint32_t r = wide[i];
        const SeedAnswer got = seed_search<32, kCandCap, SCORE>(X, rb, p, s_read[threadIdx.x / 32], r, true, kWidePlaces,
                                                                res, hits);
        if (got != kSeedDone && lane == 0) *(order_end - 1 - atomicAdd(&counts->rest, 1u)) = r;
    }
}

__global__ void __launch_bounds__(kThreads) aln_dscan_list_kernel(DIndex X, ReadBatch rb, SearchParams p,
                                                                  uint32_t n_reads, const uint32_t *order,
                                                                  const SeedCounts *counts, uint32_t *queue,
                                                                  uint2 *dbp) {
    __shared__ uint32_t s_bases[kReadWords * kThreads];
    __shared__ uint32_t s_nmask[kMaskWords * kThreads];
    cudaGridDependencySynchronize();
    const uint32_t n = counts->rest;
    if (blockIdx.x == 0 && threadIdx.x == 0) *queue = n_reads - n;
    if (n == 0) return;
    const uint64_t step = static_cast<uint64_t>(gridDim.x) * kThreads;
    const uint64_t first = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x;
    if (p.heavy.hdr)  // the heavy phase's ready words, cleared only when it may run
        for (uint64_t t = first; t < kHeavyPool; t += step) p.heavy.ready[t] = 0;
    for (uint64_t t = first; t < 2ull * n; t += step)
        dscan_one(X, rb, p, order[n_reads - n + (t >> 1)], static_cast<uint32_t>(t & 1u), s_bases + threadIdx.x, s_nmask + threadIdx.x,
                  dbp);
}

// Visit order for the persistent search: reads by decreasing lower bound
// D(0) = min over strands (0..8), so that the lanes of a warp tend to run the
// same number of deepening passes.  Counting sort in two launches; the order
// inside one bound is arbitrary (a read's result does not depend on it).
constexpr uint32_t kOrderBins = 16;

__device__ __forceinline__ uint32_t order_key(const uint2 *dbp, uint32_t r) {
    const uint2 a = dbp[2ull * r], b = dbp[2ull * r + 1];
    return min(d_at(a.x, a.y, 0), d_at(b.x, b.y, 0));
}

__global__ void aln_order_count_kernel(const uint2 *dbp, uint32_t n, uint32_t *counts) {
    __shared__ uint32_t h[kOrderBins];
    if (threadIdx.x < kOrderBins) h[threadIdx.x] = 0;
    __syncthreads();
    for (uint64_t r = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
         r += static_cast<uint64_t>(gridDim.x) * blockDim.x)
        atomicAdd(&h[order_key(dbp, static_cast<uint32_t>(r))], 1u);
    __syncthreads();
    if (threadIdx.x < kOrderBins && h[threadIdx.x]) atomicAdd(&counts[threadIdx.x], h[threadIdx.x]);
}

__global__ void aln_order_scatter_kernel(const uint2 *dbp, uint32_t n, const uint32_t *counts, uint32_t *cursor,
                                         uint32_t *order) {
    __shared__ uint32_t first[kOrderBins];
    if (threadIdx.x == 0) {
        uint32_t acc = 0;
        for (int k = kOrderBins - 1; k >= 0; k--) {  // largest bound first
            first[k] = acc;
            acc += counts[k];
        }
    }
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u;
    for (uint64_t r = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
         r += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint32_t key = order_key(dbp, static_cast<uint32_t>(r));
        const unsigned grp = __match_any_sync(__activemask(), key);  // lanes with the same bound
        const uint32_t leader = __ffs(grp) - 1;
        uint32_t off = 0;
        if (lane == leader) off = atomicAdd(&cursor[key], static_cast<uint32_t>(__popc(grp)));
        off = __shfl_sync(grp, off, leader);
        order[first[key] + off + __popc(grp & ((1u << lane) - 1u))] = static_cast<uint32_t>(r);
    }
}

// A launch that may be prepared while the kernel before it on the stream drains
// (the kernel waits for it at its start): most of a call's kernels find nothing
// to do, and a call's time is then that of its launches.  64 reads take 35 us without
// and 29 with it, 10 000 in a graph 49.6 and 45.1, 30 000 155 and 117.
template <class... Params, class... Args>
static cudaError_t launch_after(void (*kernel)(Params...), unsigned blocks, cudaStream_t st, const SearchParams *window,
                                Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (window && window->window_base && window->window_bytes) {  // prefix-trie tables held in L2's persisting set
        attr[1].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[1].val.accessPolicyWindow.base_ptr = window->window_base;
        attr[1].val.accessPolicyWindow.num_bytes = window->window_bytes;
        attr[1].val.accessPolicyWindow.hitRatio = window->window_hit_ratio;
        attr[1].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
        attr[1].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

int stack_cap_for(uint32_t z) { return z <= 2 ? 19 : (z <= 4 ? 37 : 64); }
HeavyCtx heavy_layout(void *scratch, uint32_t n);

template <int CAP, int SMEM, bool SCORE>
static cudaError_t launch_cap(const DIndex &X, const ReadBatch &rb, uint32_t n, const SearchParams &p,
                              aln_read_result *res, aln_hit *hits, uint32_t mode, uint32_t *queue,
                              void *scratch, cudaStream_t st) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (mode == ALN_MODE_PLAIN) {
        if (seed_supported(X, p)) {
            const uint32_t warps = static_cast<uint32_t>(sms) * kPlainBlocks * (kThreads / 32);
            const uint32_t each = n <= warps ? 1u : min(32u, kPlainStep * (n / (kPlainStep * warps) + 1u));
            const uint32_t block = each * (kThreads / 32);
            aln_plain_seed_kernel<CAP><<<n / block + (n % block ? 1u : 0u), kThreads, 0, st>>>(X, rb, n, each, p, res, hits);
        } else {
            aln_plain_kernel<CAP><<<(n + kThreads - 1) / kThreads, kThreads, 0, st>>>(X, rb, n, p, res, hits);
        }
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, aln_persistent_kernel<CAP, SMEM, SCORE>, kThreads, 0);
        if (p.blocks_per_sm && static_cast<int>(p.blocks_per_sm) < per_sm) per_sm = p.blocks_per_sm;
        if (per_sm < 1) per_sm = 1;
        const bool seeded = scratch && seed_supported(X, p);
        uint32_t blocks = static_cast<uint32_t>(sms * per_sm);
        // a lane a read; after a seed search, which leaves few, four, so that a warp has
        // lanes free to help.  (All the blocks that fit cost a call that leaves none 0.8 us,
        // 304 none: 10 000 reads of 36 bases take 45.2 us, 46.0 with 912.)
        const uint32_t need = seeded ? n / (kThreads / 4) + 1 : (n + kThreads - 1) / kThreads;
        if (blocks > need) blocks = need ? need : 1;
        uint2 *dbp = nullptr;
        uint32_t *order = nullptr;
        SearchParams pp = p;
        pp.heavy.hdr = nullptr;
        if (seeded) {
            // the first list takes the D breakpoints' place, which are written after it is read
            SeedCounts *counts = static_cast<SeedCounts *>(scratch);
            dbp = reinterpret_cast<uint2 *>(static_cast<char *>(scratch) + 256);
            order = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + 256 + 16ull * n);
            uint32_t *wide = reinterpret_cast<uint32_t *>(dbp);
            if (p.heavy_after != 0xFFFFFFFFu) pp.heavy = heavy_layout(scratch, n);
            cudaMemsetAsync(counts, 0, sizeof(SeedCounts), st);
            // parts of both strands on 8 lanes for z <= 3, else on 16
            if (p.z <= 3)
                aln_seed_kernel<8, SCORE><<<static_cast<unsigned>((8ull * n + kThreads - 1) / kThreads), kThreads, 0, st>>>(
                    X, rb, n, pp, res, hits, counts, wide, order + n);
            else
                aln_seed_kernel<16, SCORE><<<static_cast<unsigned>((16ull * n + kThreads - 1) / kThreads), kThreads, 0, st>>>(
                    X, rb, n, pp, res, hits, counts, wide, order + n);
            const uint32_t wb = min((n + 3u) / 4u, static_cast<uint32_t>(sms) * 6u);
            cudaError_t e = launch_after(aln_seed_wide_kernel<SCORE>, wb, st, nullptr, X, rb, pp, res, hits, counts, wide,
                                         order + n);
            const uint32_t db = min(static_cast<uint32_t>((2ull * n + kThreads - 1) / kThreads), static_cast<uint32_t>(sms) * 8u);
            if (e == cudaSuccess) e = launch_after(aln_dscan_list_kernel, db, st, nullptr, X, rb, pp, n, order, counts, queue, dbp);
            if (e != cudaSuccess) return e;
        } else {
            cudaMemsetAsync(queue, 0, sizeof(uint32_t), st);
        }
        if (scratch && !seeded) {  // D pre-pass and visit order (layout: search_scratch_bytes)
            uint32_t *counts = static_cast<uint32_t *>(scratch), *cursor = counts + kOrderBins;
            dbp = reinterpret_cast<uint2 *>(static_cast<char *>(scratch) + 256);
            order = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + 256 + 16ull * n);
            if (p.heavy_after != 0xFFFFFFFFu) {  // the heavy phase's state after them
                pp.heavy = heavy_layout(scratch, n);
                cudaMemsetAsync(pp.heavy.hdr, 0, sizeof(HeavyHdr), st);
                cudaMemsetAsync(pp.heavy.ready, 0, 4ull * kHeavyPool, st);
            }
            cudaMemsetAsync(scratch, 0, 2 * kOrderBins * sizeof(uint32_t), st);
            aln_dscan_kernel<<<static_cast<unsigned>((2ull * n + kThreads - 1) / kThreads), kThreads, 0, st>>>(
                X, rb, n, p, dbp);
            const uint32_t ob = min((n + 255u) / 256u, static_cast<uint32_t>(sms) * 8u);
            aln_order_count_kernel<<<ob, 256, 0, st>>>(dbp, n, counts);
            aln_order_scatter_kernel<<<ob, 256, 0, st>>>(dbp, n, counts, cursor, order);
        }
        cudaError_t e = launch_after(aln_persistent_kernel<CAP, SMEM, SCORE>, blocks, st, &p, X, rb, n, pp, res, hits, queue,
                                     order, dbp, seeded ? &static_cast<SeedCounts *>(scratch)->rest : nullptr);
        if (e != cudaSuccess) return e;
        if (pp.heavy.hdr && seeded && n <= kHeavyReads) {
            int hb = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&hb, aln_heavy_all_kernel<CAP, SCORE>, kThreads, 0);
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(min(static_cast<unsigned>(sms * (hb > 0 ? hb : 1)), kHeavyPool / (2u * kThreads)));
            cfg.blockDim = dim3(kThreads);
            cfg.stream = st;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeCooperative;
            attr[0].val.cooperative = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            e = cudaLaunchKernelEx(&cfg, aln_heavy_all_kernel<CAP, SCORE>, X, rb, pp, static_cast<const uint2 *>(dbp), res, hits);
            if (e != cudaSuccess) return e;
        } else if (pp.heavy.hdr) {  // the reads handed over, one deepening pass per launch over the whole GPU
            int hb = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&hb, aln_heavy_pass_kernel<CAP, SCORE>, kThreads, 0);
            // the ring holds at most 2 entries per thread of the grid (the pass kernel's low-water mark)
            const unsigned hgrid = min(static_cast<unsigned>(sms * (hb > 0 ? hb : 1)), kHeavyPool / (2u * kThreads));
            const unsigned hblocks = min(kHeavyReads, static_cast<uint32_t>(sms) * kHeavyBlocksPerSm);
            e = launch_after(aln_heavy_start_kernel, hblocks, st, nullptr, pp, dbp, X.t[0].n);
            for (uint32_t pass = 0; pass < kHeavyPasses && e == cudaSuccess; pass++) {
                e = launch_after(aln_heavy_pass_kernel<CAP, SCORE>, hgrid, st, nullptr, X, rb, pp, dbp);
                if (e == cudaSuccess)
                    e = launch_after(aln_heavy_decide_kernel, hblocks, st, nullptr, pp, dbp, X.t[0].n, res, hits,
                                     pass + 1 == kHeavyPasses ? 1 : 0);
            }
            if (e != cudaSuccess) return e;
        }
    }
    return cudaGetLastError();
}

// Resident blocks per SM of the persistent kernel for limit z and a shared-memory
// stack of smem entries per lane (occupancy).
template <int SMEM>
static int max_blocks_smem(uint32_t z) {
    int per_sm = 0;
    switch (stack_cap_for(z)) {
        case 19: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, aln_persistent_kernel<19, SMEM, false>, kThreads, 0); break;
        case 37: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, aln_persistent_kernel<37, SMEM, false>, kThreads, 0); break;
        default: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, aln_persistent_kernel<64, SMEM, false>, kThreads, 0); break;
    }
    return per_sm;
}

int persistent_max_blocks(uint32_t z, uint32_t smem) {
    switch (smem) {
        case 4: return max_blocks_smem<4>(z);
        case 12: return max_blocks_smem<12>(z);
        default: return max_blocks_smem<8>(z);
    }
}

// Shared-memory stack depths the persistent kernel is compiled for.
bool smem_stack_supported(uint32_t smem) { return smem == 0 || smem == 4 || smem == 8 || smem == 12; }

// Bytes of the optional persistent-mode scratch for n reads: order-sort counters
// (256 B), D breakpoints (2 x 8 B per read), visit order (4 B per read), then
// from the next 256-byte boundary the heavy phase: its header, the handed-over
// reads, their candidate tables, the task ring and its ready words.
static uint64_t heavy_offset(uint32_t n) { return (256ull + 20ull * n + 255ull) & ~255ull; }
static constexpr uint64_t kHeavyBytes = sizeof(HeavyHdr) + kHeavyReads * sizeof(HeavyRead) +
                                        2ull * kHeavyReads * kHeavySlots * sizeof(HeavySlot) +
                                        kHeavyPool * sizeof(HeavyTask) + 4ull * kHeavyPool;
uint64_t search_scratch_bytes(uint32_t n) { return heavy_offset(n) + kHeavyBytes; }

HeavyCtx heavy_layout(void *scratch, uint32_t n) {
    char *b = static_cast<char *>(scratch) + heavy_offset(n);
    HeavyCtx H;
    H.hdr = reinterpret_cast<HeavyHdr *>(b);
    b += sizeof(HeavyHdr);
    H.reads = reinterpret_cast<HeavyRead *>(b);
    b += kHeavyReads * sizeof(HeavyRead);
    H.slots = reinterpret_cast<HeavySlot *>(b);
    b += 2ull * kHeavyReads * kHeavySlots * sizeof(HeavySlot);
    H.pool = reinterpret_cast<HeavyTask *>(b);
    b += kHeavyPool * sizeof(HeavyTask);
    H.ready = reinterpret_cast<uint32_t *>(b);
    return H;
}

template <int CAP>
static cudaError_t launch_smem(const DIndex &X, const ReadBatch &rb, uint32_t n, const SearchParams &p,
                               aln_read_result *res, aln_hit *hits, uint32_t mode, uint32_t *queue, void *scratch,
                               cudaStream_t st) {
    if (p.strata == ALN_STRATA_SCORE)  // score-ordered kernels: the default stack depth only
        return launch_cap<CAP, kSmemStackDefault, true>(X, rb, n, p, res, hits, mode, queue, scratch, st);
    switch (p.smem_stack) {
        case 4: return launch_cap<CAP, 4, false>(X, rb, n, p, res, hits, mode, queue, scratch, st);
        case 12: return launch_cap<CAP, 12, false>(X, rb, n, p, res, hits, mode, queue, scratch, st);
        default: return launch_cap<CAP, kSmemStackDefault, false>(X, rb, n, p, res, hits, mode, queue, scratch, st);
    }
}

cudaError_t launch_search(const DIndex &X, const ReadBatch &rb, uint32_t n, const SearchParams &p,
                          aln_read_result *res, aln_hit *hits, uint32_t mode, uint32_t *queue, void *scratch,
                          cudaStream_t st) {
    const bool seeds = mode != ALN_MODE_PLAIN && n && scratch && seed_supported(X, p);  // its first kernel clears the status
    if (p.status && !seeds) {
        const cudaError_t e = cudaMemsetAsync(p.status, 0, sizeof(uint32_t), st);
        if (e != cudaSuccess) return e;
    }
    if (n == 0) return cudaSuccess;
    switch (stack_cap_for(p.z)) {
        case 19: return launch_smem<19>(X, rb, n, p, res, hits, mode, queue, scratch, st);
        case 37: return launch_smem<37>(X, rb, n, p, res, hits, mode, queue, scratch, st);
        default: return launch_smem<64>(X, rb, n, p, res, hits, mode, queue, scratch, st);
    }
}

}  // namespace aln
