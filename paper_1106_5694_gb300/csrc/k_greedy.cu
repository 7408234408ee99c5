// k_greedy.cu -- greedy starting assignment (Section 3.1, read as the global
// greedy: repeatedly take the largest remaining benefit, ties to the lowest
// agent, then the lowest job).
//
// Parallel form: deferred acceptance (below), from bounds on the best benefit
// of each agent in each tile of jobs.  Fallback (a refused launch, or the
// DGS_GREEDY_ROUNDS=1 knob): locally-dominant rounds.  Under the strict total
// order on pairs (benefit desc, agent asc, job asc), every free agent finds
// its best free job and every free job its best free agent; mutually-best
// pairs are matched.  The globally largest remaining pair is always mutually
// best and the matched pairs are disjoint, so the rounds produce exactly the
// sequential global-greedy assignment.
//
// Pass 1 reads a once in 64x64 tiles and, in the same pass, writes the
// transposed copy at, checks |a| < 2^29 and computes what the greedy start
// that follows needs: each agent's best benefit in every tile of jobs.
#include <algorithm>
#include <cstdlib>

#include "dgs_internal.cuh"

namespace dgs {
namespace {

constexpr int kT = 64;  // tile edge

// Pass 1 over 64 x 64 tiles, 256 threads.  A tile's rows go to shared memory in
// 16-byte chunks, chunk c of row r at place c ^ (r / 4 mod 16): a row's chunks
// fill all banks, and so do the chunks c of eight rows 4l that the transposing
// read takes together.  Each thread then reads the 4 x 4 block of rows 4l ..
// and columns 4c .., writes its columns as 16 bytes of four rows of at, and
// (kBounds) raises the tile's maxima of its rows.  Rows and columns past n read
// as 0, which changes no range and leaves bounds valid.  What bounds it: HBM
// (read a, write at); with one element per shared-memory instruction and the
// row maxima by shuffles it was 465 instructions a warp and tile, 55% of the
// issue slots (n = 10000, under ncu: 147 us, now 128, 92% of the measured
// copy rate).
//
// a_src: the caller's matrix with row pitch n when w.a is the workspace's
// pitched copy still to be filled; this pass reads a_src (a warp per row, 32
// consecutive columns per load, from any 4-byte boundary) and writes the copy
// as it goes.  Null: w.a is read.
template <bool kBounds>
__device__ __forceinline__ void greedy_pass1_body(const Workspace& w, int32_t tiles_x, int32_t tiles_total,
                                                  int32_t bid, int32_t nblk, const int32_t* a_src = nullptr) {
    __shared__ __align__(16) int32_t s[kT * kT];
    __shared__ uint32_t s_top[kT];
    const int32_t n = w.n;
    const int t = threadIdx.x, lane16 = t & 15, row0 = t >> 4;
    auto chunk = [&](int r, int c) -> int4* { return reinterpret_cast<int4*>(s) + r * 16 + (c ^ ((r >> 2) & 15)); };
    if (kBounds && t < kT) s_top[t] = 0u;
    int32_t lo = 0, hi = 0;
    for (int32_t tile = bid; tile < tiles_total; tile += nblk) {
        const int32_t I0 = (tile / tiles_x) * kT;
        const int32_t J0 = (tile % tiles_x) * kT;
        if (a_src == nullptr) {
            int4 x[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int32_t i = I0 + row0 + 16 * p, j = J0 + lane16 * 4;
                x[p] = i < n && j < w.lda ? *reinterpret_cast<const int4*>(w.a + (size_t)i * w.lda + j)
                                          : make_int4(0, 0, 0, 0);
            }
#pragma unroll
            for (int p = 0; p < 4; ++p) *chunk(row0 + 16 * p, lane16) = x[p];
        } else {
            const int lane = t & 31;
            int32_t x[8][2];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int32_t i = I0 + (t >> 5) + 8 * q;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int32_t j = J0 + lane + 32 * h;
                    x[q][h] = i < n && j < n ? a_src[(size_t)i * n + j] : 0;
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = (t >> 5) + 8 * q, c = lane + 32 * h;
                    reinterpret_cast<int32_t*>(chunk(r, c >> 2))[c & 3] = x[q][h];
                }
        }
        __syncthreads();
        if (a_src != nullptr) {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int32_t r = row0 + 16 * p, i = I0 + r, j = J0 + lane16 * 4;
                if (i < n && j < w.lda)
                    *reinterpret_cast<int4*>(const_cast<int32_t*>(w.a) + (size_t)i * w.lda + j) = *chunk(r, lane16);
            }
        }
        // rows 4 lane16 .., columns 4 row0 ..
        int4 b[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) b[e] = *chunk(lane16 * 4 + e, row0);
        const int32_t j = J0 + row0 * 4;
        int32_t* at = w.at + (size_t)j * w.ldt + I0 + lane16 * 4;
        if (j < n) *reinterpret_cast<int4*>(at) = make_int4(b[0].x, b[1].x, b[2].x, b[3].x);
        if (j + 1 < n) *reinterpret_cast<int4*>(at + w.ldt) = make_int4(b[0].y, b[1].y, b[2].y, b[3].y);
        if (j + 2 < n) *reinterpret_cast<int4*>(at + 2 * (size_t)w.ldt) = make_int4(b[0].z, b[1].z, b[2].z, b[3].z);
        if (j + 3 < n) *reinterpret_cast<int4*>(at + 3 * (size_t)w.ldt) = make_int4(b[0].w, b[1].w, b[2].w, b[3].w);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int32_t top = max(max(b[e].x, b[e].y), max(b[e].z, b[e].w));
            lo = min(lo, min(min(b[e].x, b[e].y), min(b[e].z, b[e].w)));
            hi = max(hi, top);
            if (kBounds) atomicMax(&s_top[lane16 * 4 + e], (uint32_t)(top + kBenefitLimit));
        }
        __syncthreads();
        if (kBounds && t < kT) {  // (the next tile's maxima come after its first barrier)
            if (I0 + t < n) {
                uint32_t* bound = w.g_bound + (size_t)(I0 + t) * w.bound_tiles + (J0 >> w.bound_shift);
                if (w.bound_shift == kBoundShift) *bound = s_top[t];
                else atomicMax(bound, s_top[t]);
            }
            s_top[t] = 0u;
        }
    }
    report_range(w, lo, hi);
}

// tiles tile0 .. tiles_total - 1 (row-major: a band of whole tile rows)
template <bool kBounds>
__global__ void __launch_bounds__(256) greedy_pass1_kernel(Workspace w, int32_t tiles_x, int32_t tiles_total,
                                                           int32_t tile0, const int32_t* a_src) {
    greedy_pass1_body<kBounds>(w, tiles_x, tiles_total, tile0 + blockIdx.x, gridDim.x, a_src);
}

// Rounds: every owner's best partner in its row of mat (a for agents, at for
// jobs), a warp per row.
__global__ void __launch_bounds__(256) greedy_best_kernel(Workspace w, const int32_t* mat, int32_t ld,
                                                          unsigned long long* keys) {
    const int lane = threadIdx.x & 31;
    for (int32_t o = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); o < w.n; o += gridDim.x * (blockDim.x / 32)) {
        unsigned long long best = 0;
        for (int32_t c = lane; c < w.n; c += 32) best = umax64(best, pack_benefit(mat[(size_t)o * ld + c], (uint32_t)c));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) best = umax64(best, __shfl_xor_sync(0xffffffffu, best, off));
        if (lane == 0) keys[o] = best;
    }
}

// Match every mutually-best (agent, job) pair.
__device__ __forceinline__ void greedy_match_body(const Workspace& w, int32_t bid, int32_t nblk) {
    DeviceState* st = w.st;
    if (st->status != kRunning || st->greedy_remaining == 0) return;
    for (int32_t i = bid * blockDim.x + threadIdx.x; i < w.n; i += nblk * blockDim.x) {
        if (!w.free_a[i]) continue;
        const int32_t j = key_index(w.g_row[i]);
        if (j < 0 || j >= w.n) {  // every free agent has a free best job
            st->error = kErrInternal;
            st->status = kError;
            continue;
        }
        if (key_index(w.g_col[j]) == i) {
            w.tau[i] = j;
            w.sigma[j] = i;
            w.free_a[i] = 0;
            w.free_j[j] = 0;
            atomicSub(&st->greedy_remaining, 1);
            st->greedy_matched = 1;
        }
    }
}

__global__ void greedy_match_kernel(Workspace w) { greedy_match_body(w, blockIdx.x, gridDim.x); }

// Rescan: for each free "owner" whose best partner was taken, find the best
// free partner in its row of mat (a for agents over jobs, at for jobs over
// agents).  One CTA per owner; 16-byte loads, several in flight per thread.
__global__ void __launch_bounds__(256) greedy_rescan_kernel(Workspace w, const int32_t* mat, int32_t ld,
                                                            unsigned long long* keys, const uint8_t* owner_free,
                                                            const uint8_t* partner_free, int32_t count_round) {
    DeviceState* st = w.st;
    if (count_round && blockIdx.x == 0 && threadIdx.x == 0 && st->greedy_matched) {
        st->greedy_rounds += 1;  // the match kernel before this one matched pairs
        st->greedy_matched = 0;
    }
    if (st->status != kRunning || st->greedy_remaining == 0) return;
    __shared__ unsigned long long red[8];
    const int32_t n = w.n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int32_t o = blockIdx.x; o < n; o += gridDim.x) {
        if (!owner_free[o]) continue;
        const int32_t b = key_index(keys[o]);
        if (b >= 0 && b < n && partner_free[b]) continue;  // best partner still free
        const int32_t* row = mat + (size_t)o * ld;
        if (tid == 0) atomicAdd((unsigned long long*)&st->greedy_rescans, 1ull);
        unsigned long long best = 0;
#pragma unroll 4
        for (int32_t c = tid * 4; c < n; c += 1024) {
            const int4 v = *reinterpret_cast<const int4*>(row + c);
            const uint32_t fr = *reinterpret_cast<const uint32_t*>(partner_free + c);
            const int32_t vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (c + e < n && ((fr >> (8 * e)) & 0xffu)) best = umax64(best, pack_benefit(vals[e], (uint32_t)(c + e)));
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) best = umax64(best, __shfl_xor_sync(0xffffffffu, best, off));
        if (lane == 0) red[warp] = best;
        __syncthreads();
        if (tid == 0) {
            unsigned long long m = 0;
            for (int q = 0; q < 8; ++q) m = umax64(m, red[q]);
            keys[o] = m;
        }
        __syncthreads();
    }
}

// Deferred acceptance (Gale and Shapley 1962, agents proposing).  Every
// agent ranks the jobs by (benefit desc, job asc) and every job ranks the
// agents by (benefit desc, agent asc); both rankings are induced by the one
// strict total order on pairs (benefit desc, agent asc, job asc), so the
// stable matching is unique and equals the global greedy assignment: the
// greedy matching is stable, and in any other perfect matching the first
// pair, in that order, where the two differ is a greedy pair, which blocks
// the other matching.  Deferred acceptance in any order of proposals reaches
// it.
//
// Form: g_col[j] holds the key (biased benefit, ~agent) of the job's holder
// and only grows (64-bit atomicMax).  Agent i beats the holder of job j iff
// its own key (a[i][j] biased, ~i) is larger.  A free agent proposes to its
// best job among those whose holder it beats; a proposal that raises the key
// displaces the holder, who proposes next.  A failed proposal looks again.
//
// Bounds: g_bound[i][t] is an upper bound on the biased benefit of agent i's
// best job in tile t among those whose holder it beats (0: none).  Pass 1
// sets it to the tile's maximum.  Holders' keys only grow, so the jobs an
// agent beats only become fewer, and the maximum that a look at the tile
// finds (with holders' keys that may be stale, that is lower) stays a bound
// for good: it is written back, and any value ever stored is valid, so the
// bounds need no ordering between the threads that follow one agent over
// time.  A proposal takes the tiles in the order of their bounds (ties: the
// lower tile, which has the lower jobs) and reads their benefits and holders'
// keys until no other tile's bound can beat the best job found (a larger
// value, or the same value in a lower tile).
//
// Padded rectangular instances (dgs_solve_rect): the dummy agents' rows (or
// the dummy jobs' columns) are all zero, so they tie everywhere and queue up:
// each dummy fails at every job that a lower dummy takes, one round trip after
// the other (1500 agents, 2001 jobs: 1.0 of 1.8 ms).  There the real agents
// first propose to real jobs of benefit >= 0 only, and wait when none takes
// them; then one CTA places the dummies (greedy_rect_fill_kernel); then the
// agents that still wait propose to any job.  Pairs of benefit 0 come in the
// order of their agents, then jobs, real ones before dummies, so that is the
// order of the one total order.
//
// What bounds it: round trips to memory, one chain of displacements after the
// other (bounds, tiles, atomic), and the instructions of the looks; not bytes.
// A look of a warp reads its four best bounds' tiles at once (3 KB).  An agent
// displaced late has to look at most of its tiles (the good jobs are taken), so
// a chain is followed by a group of four warps, each with its share of the
// tiles: a proposal then takes about 1.5 microseconds when one look is enough
// and 5 when all are needed.  Measured (single solve, greedy start after pass
// 1), against reading an agent's whole row and every holder's key per proposal
// with the four best jobs kept for later proposals: peer-shaped n = 10000 0.48
// -> 0.24 ms, n = 4096 0.167 -> 0.117, uniform n = 20000 0.47 -> 0.17.  One
// warp per chain 0.30 ms at n = 10000, two 0.26, eight 0.50; eight tiles per
// look 0.29 (fewer CTAs fit); prefetching an agent's remaining tiles into L2:
// no change.  A batched launch has chains enough to fill the chip, so there
// one warp follows a chain (1024 peer-shaped instances, n in [64, 4096]: 22.4
// -> 4.7 ms).
//
// A group's first agent is its number in the grid, the next ones come from a
// counter; it follows the chain of displacements that starts with each: the
// agent it displaced proposes next, until a proposal lands on a job nobody
// held.  Every free agent is thus in exactly one group's hands, no group waits
// for another, and the launch ends when every chain has ended.
constexpr int kDaThreads = 256;
constexpr int kDaPerSm = 4;
constexpr int kDaGroup = 4;  // warps that follow one chain
constexpr int kDaPicks = 4;  // 64-job tiles that one look of a warp reads
constexpr int32_t kDaTies = 64;       // proposals of one walk over tied jobs (da_walk_ties)
constexpr int32_t kDaTieWait = 64;    // displacements until the next walk, after one that found nothing;
constexpr int32_t kDaTieFailed = 4;   // a failed proposal counts as so many
constexpr int kDaWarps = kDaThreads / 32;
constexpr uint64_t kDaTimeoutNs = 16000000000ull;  // bound on one warp's work (internal error beyond)

// 64-bit atomic max with acquire-release order at GPU scope.
__device__ __forceinline__ unsigned long long atomic_max_acq_rel(unsigned long long* p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.acq_rel.gpu.global.max.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}

__device__ __forceinline__ unsigned long long pack_key(uint32_t hi, uint32_t lo) {
    return ((unsigned long long)hi << 32) | lo;
}

// What a proposal reads of an instance: the jobs 0 .. n - 1, those with a
// (biased) benefit of at least `floor`.
struct DaView {
    const int32_t* a;
    unsigned long long* keys;
    uint32_t* bounds;
    int32_t n, lda, tiles, pitch, shift;  // tiles with such jobs, bounds per agent
    uint32_t floor;
};
__device__ __forceinline__ DaView da_view(const Workspace& w, int32_t jobs, uint32_t floor) {
    return DaView{w.a,           w.g_col,       w.g_bound, jobs, w.lda, bound_tiles(jobs, w.bound_shift),
                  w.bound_tiles, w.bound_shift, floor};
}

// Barrier of a group of kGroup warps (named barriers 1.., one per group).
template <int kGroup>
__device__ __forceinline__ void group_bar(int grp) {
    if (kGroup == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(kGroup * 32) : "memory");
}

// What the warps of a group exchange: the best job found and the best bound
// not looked at yet, as (value, ~job) and (value, ~tile), by turns in two
// buffers; the outcome of the proposal.
template <int kGroup>
struct DaShared {
    unsigned long long best[2][kGroup], left[2][kGroup];
    int32_t out;
};

// The value of this lane's best job of the four in x among those whose holder
// (keys h0, h1) agent i beats; 0 when there is none.  Jobs from column c on, of
// which those below n exist.
__device__ __forceinline__ uint32_t da_best4(const int4& x, const ulonglong2& h0, const ulonglong2& h1, int32_t c,
                                             int32_t n, uint32_t me_lo) {
    const uint32_t b0 = (uint32_t)(x.x + kBenefitLimit), b1 = (uint32_t)(x.y + kBenefitLimit);
    const uint32_t b2 = (uint32_t)(x.z + kBenefitLimit), b3 = (uint32_t)(x.w + kBenefitLimit);
    uint32_t r = pack_key(b0, me_lo) > h0.x ? b0 : 0u;
    if (pack_key(b1, me_lo) > h0.y && c + 1 < n) r = max(r, b1);
    if (pack_key(b2, me_lo) > h1.x && c + 2 < n) r = max(r, b2);
    if (pack_key(b3, me_lo) > h1.y && c + 3 < n) r = max(r, b3);
    return r;
}
// The lowest of those jobs whose value is r.
__device__ __forceinline__ int32_t da_column4(const int4& x, const ulonglong2& h0, const ulonglong2& h1, int32_t c,
                                              uint32_t r, uint32_t me_lo) {
    if ((uint32_t)(x.x + kBenefitLimit) == r && pack_key(r, me_lo) > h0.x) return c;
    if ((uint32_t)(x.y + kBenefitLimit) == r && pack_key(r, me_lo) > h0.y) return c + 1;
    if ((uint32_t)(x.z + kBenefitLimit) == r && pack_key(r, me_lo) > h1.x) return c + 2;
    return c + 3;
}

// One look of a warp at tiles of 64 jobs (see da_propose): the kDaPicks best
// bounds, at most one of each lane, half a warp per tile.  mv, mt: this
// lane's largest bound left and its tile; bv, bt: value and tile of the best
// job known.  Returns the best job found, (value, ~job), 0 when none; `mine`:
// this lane's tile was one of them and `found` is its new bound.
__device__ __forceinline__ unsigned long long da_look64(const DaView& d, const int32_t* row, uint32_t me_lo, uint32_t mv,
                                                        int32_t mt, uint32_t bv, int32_t bt, bool& mine,
                                                        uint32_t& found) {
    constexpr uint32_t kAll = 0xffffffffu;
    constexpr int32_t kNone = 0x7fffffff;
    const int lane = threadIdx.x & 31, half = lane >> 4;
    int32_t tile[kDaPicks / 2];
    uint32_t left = (mv > bv || (mv == bv && mt < bt)) ? mv : 0u;
    int turn = -1;
#pragma unroll
    for (int k = 0; k < kDaPicks; ++k) {
        const uint32_t v = __reduce_max_sync(kAll, left);
        const int32_t t = (int32_t)__reduce_min_sync(kAll, left == v && v != 0u ? (uint32_t)mt : (uint32_t)kNone);
        if (mt == t && v != 0u) {
            left = 0u;
            turn = k;
        }
        if ((k & 1) == 0) tile[k / 2] = t;
        else tile[k / 2] = half ? t : tile[k / 2];
    }
    int4 x[kDaPicks / 2];
    ulonglong2 h0[kDaPicks / 2], h1[kDaPicks / 2];
    int32_t c[kDaPicks / 2];
#pragma unroll
    for (int q = 0; q < kDaPicks / 2; ++q) {
        c[q] = tile[q] == kNone ? d.n : tile[q] * kT + (lane & 15) * 4;
        if (c[q] < d.n) {
            x[q] = __ldg(reinterpret_cast<const int4*>(row + c[q]));
            h0[q] = __ldcg(reinterpret_cast<const ulonglong2*>(d.keys + c[q]));
            h1[q] = __ldcg(reinterpret_cast<const ulonglong2*>(d.keys + c[q] + 2));
        }
    }
    uint32_t lv[kDaPicks / 2], top = 0u;
#pragma unroll
    for (int q = 0; q < kDaPicks / 2; ++q) {
        lv[q] = c[q] < d.n ? da_best4(x[q], h0[q], h1[q], c[q], d.n, me_lo) : 0u;
        top = max(top, lv[q]);
    }
    const uint32_t r = __reduce_max_sync(kAll, top);
    uint32_t lc = (uint32_t)kNone;
    if (top == r && r != 0u) {  // (few lanes)
#pragma unroll
        for (int q = 0; q < kDaPicks / 2; ++q)
            if (lv[q] == r) lc = min(lc, (uint32_t)da_column4(x[q], h0[q], h1[q], c[q], r, me_lo));
    }
    const uint32_t rc = __reduce_min_sync(kAll, lc);
    // each tile's maximum, to the lane whose tile it is
#pragma unroll
    for (int q = 0; q < kDaPicks / 2; ++q) {
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) lv[q] = max(lv[q], __shfl_xor_sync(kAll, lv[q], off));
        const uint32_t m = __shfl_sync(kAll, lv[q], (turn & 1) * 16);
        if ((turn >> 1) == q) found = m;
    }
    mine = turn >= 0;
    return r >= d.floor ? ((unsigned long long)r << 32) | ~rc : 0ull;
}

// The same at wider tiles (2^shift jobs, shift > kBoundShift; instances of a
// batch): one tile, the warp's best bound.
__device__ __forceinline__ unsigned long long da_look_wide(const DaView& d, const int32_t* row, uint32_t me_lo,
                                                           uint32_t mv, int32_t mt, uint32_t bv, int32_t bt, bool& mine,
                                                           uint32_t& found) {
    constexpr uint32_t kAll = 0xffffffffu;
    constexpr int32_t kNone = 0x7fffffff;
    const int lane = threadIdx.x & 31;
    const uint32_t left = (mv > bv || (mv == bv && mt < bt)) ? mv : 0u;
    const uint32_t v = __reduce_max_sync(kAll, left);
    mine = false;
    if (v == 0u) return 0ull;
    const int32_t t = (int32_t)__reduce_min_sync(kAll, left == v ? (uint32_t)mt : (uint32_t)kNone);
    const int32_t end = min(d.n, (t + 1) << d.shift);
    uint32_t top = 0u, lc = (uint32_t)kNone;
#pragma unroll 2
    for (int32_t c = (t << d.shift) + lane * 4; c < end; c += 128) {
        const int4 x = __ldg(reinterpret_cast<const int4*>(row + c));
        const ulonglong2 h0 = __ldcg(reinterpret_cast<const ulonglong2*>(d.keys + c));
        const ulonglong2 h1 = __ldcg(reinterpret_cast<const ulonglong2*>(d.keys + c + 2));
        const uint32_t b = da_best4(x, h0, h1, c, d.n, me_lo);
        if (b > top) {
            top = b;
            lc = (uint32_t)da_column4(x, h0, h1, c, b, me_lo);
        }
    }
    const uint32_t r = __reduce_max_sync(kAll, top);
    const uint32_t rc = __reduce_min_sync(kAll, top == r ? lc : (uint32_t)kNone);
    mine = mt == t;
    found = r;
    return r >= d.floor ? ((unsigned long long)r << 32) | ~rc : 0ull;
}

// Tied values.  A proposal to job c has just displaced that job's holder
// (`old`, below the proposer's key `mine`) or failed against it: the turn is the
// displaced agent's, or the proposer's again.  c was the best job of whose turn
// it is, at some benefit v, so it has lost every job that it ranks above c, and
// now c.  Its next job of benefit v after c is therefore its best one, once
// every job between has been looked at.  The walk does just that: 128 jobs from
// c's group of 64 on (one load of the row and two of the keys per lane), the
// proposal, and on with whose turn it then is, until a job was free, none of
// the 128 will do, or kDaTies proposals are made (so that the caller's bound on
// time is looked at).
//
// It is tried after every displacement and failure for as long as walks find
// something, and again kDaTieWait displacements after one that did not (earlier
// when proposals fail).  Without it every turn was a look of the whole group, and
// where many agents want the same jobs for few different values that is one look
// per agent and job: constant n = 4096 23 ms, now 11.2, n = 20000 89 -> 35; values
// in [0, 2) n = 4096 7.3 -> 3.1; in [0, 4) 3.2 -> 1.36, n = 20000 13 -> 4.8.  Without
// ties it costs at most 1 us (peer-shaped n = 4096 117.6 -> 118.3 us, 10000 263.7
// -> 264.4): a walk that finds nothing takes as long, and tried after every
// failure it cost 2 to 3.  It does not help identical agents whose jobs differ in
// value: there every turn is still a look.
struct DaWalk {
    int32_t out;   // as da_propose returns it (-3: agent i's turn)
    int32_t tied;  // its next `tied`
};
__device__ __noinline__ DaWalk da_walk_ties(const int32_t* a, unsigned long long* keys, int32_t n, int32_t lda,
                                            int32_t i, int32_t c, unsigned long long mine, unsigned long long old) {
    constexpr uint32_t kAll = 0xffffffffu, kNone = 0x7fffffffu;
    const int lane = threadIdx.x & 31;
    int32_t who = i;
    for (int32_t q = 0; old != 0ull; ++q) {
        if (old < mine) {  // displaced: its turn
            who = key_index(old);
            mine = old;
        }
        uint32_t next = kNone;
        const int32_t c4 = (c & ~(kT - 1)) + lane * 4;
        if (q < kDaTies && c4 < n && c4 + 3 > c) {
            const int32_t v = (int32_t)(mine >> 32) - kBenefitLimit;
            const int4 x = __ldg(reinterpret_cast<const int4*>(a + (size_t)who * lda + c4));
            const ulonglong2 h0 = __ldcg(reinterpret_cast<const ulonglong2*>(keys + c4));
            const ulonglong2 h1 = __ldcg(reinterpret_cast<const ulonglong2*>(keys + c4 + 2));
            if (x.w == v && mine > h1.y && c4 + 3 < n) next = (uint32_t)c4 + 3u;
            if (x.z == v && mine > h1.x && c4 + 2 < n && c4 + 2 > c) next = (uint32_t)c4 + 2u;
            if (x.y == v && mine > h0.y && c4 + 1 < n && c4 + 1 > c) next = (uint32_t)c4 + 1u;
            if (x.x == v && mine > h0.x && c4 > c) next = (uint32_t)c4;
        }
        next = __reduce_min_sync(kAll, next);
        if (next == kNone) return DaWalk{who == i ? -3 : who, q > 0 ? 0 : -kDaTieWait};
        c = (int32_t)next;
        if (lane == 0) old = atomic_max_acq_rel(keys + c, mine);
        old = __shfl_sync(kAll, old, 0);
    }
    return DaWalk{-1, 0};
}

// One proposal of agent i (and its retries after failed ones) by a group of
// kGroup warps.  Tile t belongs to lane (t / kGroup) % 32 of warp t % kGroup.
// s_b: the group's copy of the agent's bounds (each thread reads and writes
// only its own tiles' entries).  tied (the group's first warp's): below 0 the
// displacements to come until a walk over tied jobs is tried.  Returns the agent
// whose turn is next (it was displaced), -1 when the job was free, -4 when no job
// of benefit d.floor takes the agent (that is an error when every job counts,
// d.floor = 1), -2 on an error.
template <int kGroup>
__device__ __forceinline__ int32_t da_propose(const DaView& d, int32_t i, uint32_t* s_b, DaShared<kGroup>& sh, int grp,
                                              int gw, int32_t& looks, int32_t& tied) {
    constexpr uint32_t kAll = 0xffffffffu;
    constexpr int32_t kNone = 0x7fffffff;
    const int lane = threadIdx.x & 31;
    const int32_t t_first = lane * kGroup + gw;
    const uint32_t me_lo = ~(uint32_t)i;
    uint32_t* bounds = d.bounds + (size_t)i * d.pitch;
    const int32_t* row = d.a + (size_t)i * d.lda;
    int turn = 0;
    for (int32_t attempt = 0; attempt <= 2 * d.n + 2; ++attempt) {
        uint32_t mv = 0u;    // this lane's largest bound not looked at yet
        int32_t mt = kNone;  // and its (lowest) tile
        for (int32_t t = t_first; t < d.tiles; t += 32 * kGroup) {
            uint32_t b = __ldcg(bounds + t);
            if (b < d.floor) b = 0u;
            s_b[t] = b;
            if (b > mv) {
                mv = b;
                mt = t;
            }
        }
        uint32_t bv = 0u;  // the best job found by the group: value, column
        int32_t bc = kNone;
        for (;;) {
            bool mine;
            uint32_t found = 0u;
            const int32_t bt = bv == 0u ? kNone : bc >> d.shift;
            unsigned long long best = d.shift == kBoundShift
                                          ? da_look64(d, row, me_lo, mv, mt, bv, bt, mine, found)
                                          : da_look_wide(d, row, me_lo, mv, mt, bv, bt, mine, found);
            looks += __popc(__ballot_sync(kAll, mine));
            // the bounds found, for good; not looked at again in this attempt
            if (mine) {
                if (found != mv) __stcg(bounds + mt, found);
                s_b[mt] = 0u;
                mv = 0u;
                mt = kNone;
                for (int32_t t = t_first; t < d.tiles; t += 32 * kGroup) {
                    const uint32_t b = s_b[t];
                    if (b > mv) {
                        mv = b;
                        mt = t;
                    }
                }
            }
            // (value, ~job) and (value, ~tile): larger is better
            const uint32_t l = __reduce_max_sync(kAll, mv);
            const uint32_t lt = __reduce_min_sync(kAll, mv == l ? (uint32_t)mt : (uint32_t)kNone);
            unsigned long long more = ((unsigned long long)l << 32) | ~lt;
            if (kGroup > 1) {
                if (lane == 0) {
                    sh.best[turn][gw] = best;
                    sh.left[turn][gw] = more;
                }
                group_bar<kGroup>(grp);
#pragma unroll
                for (int k = 0; k < kGroup; ++k) {
                    best = umax64(best, sh.best[turn][k]);
                    more = umax64(more, sh.left[turn][k]);
                }
                turn ^= 1;
            }
            if ((uint32_t)(best >> 32) > bv || ((uint32_t)(best >> 32) == bv && (int32_t)(~(uint32_t)best) < bc)) {
                bv = (uint32_t)(best >> 32);
                bc = (int32_t)(~(uint32_t)best);
            }
            const uint32_t v = (uint32_t)(more >> 32);
            if (v == 0u || bv > v || (bv == v && (bc >> d.shift) < (int32_t)(~(uint32_t)more))) break;
        }
        // some job always accepts a free agent, and every failed proposal
        // rules a job out, so an agent needs at most 2 n + 2 attempts
        if (bv == 0u) return d.floor > 1u ? -4 : -2;
        if (bc >= d.n) return -2;
        int32_t out = -2;
        if (gw == 0) {
            const unsigned long long mine = ((unsigned long long)bv << 32) | me_lo;
            unsigned long long old = 0ull;
            if (lane == 0) old = atomic_max_acq_rel(d.keys + bc, mine);
            old = __shfl_sync(kAll, old, 0);
            out = old < mine ? (old == 0ull ? -1 : key_index(old)) : -3;  // -3: taken meanwhile, look again
            if (out != -1 && (tied += out == -3 ? kDaTieFailed : 1) >= 0) {
                const DaWalk r = da_walk_ties(d.a, d.keys, d.n, d.lda, i, bc, mine, old);
                out = r.out;
                tied = r.tied;
            }
        }
        if (kGroup > 1) {
            if (gw == 0 && lane == 0) sh.out = out;
            group_bar<kGroup>(grp);
            out = sh.out;
            group_bar<kGroup>(grp);
        }
        if (out != -3) return out;
    }
    return -2;
}

// The agents of one launch: 0 .. count - 1, or (list not null) the st->da_wait
// entries of list; the jobs 0 .. jobs - 1 of biased benefit >= floor; waits:
// marks the agents that no such job takes.
struct DaPhase {
    const int32_t* list;
    int32_t count, jobs;
    uint32_t floor;
    uint8_t* waits;
};

template <int kGroup>
__global__ void __launch_bounds__(kDaThreads, kDaPerSm) greedy_da_kernel(Workspace w, DaPhase ph) {
    extern __shared__ __align__(16) uint32_t s_bounds[];
    constexpr int kGroups = kDaWarps / kGroup;
    __shared__ DaShared<kGroup> s_sh[kGroups];
    DeviceState* st = w.st;
    __shared__ int32_t s_status, s_next[kGroups];
    if (threadIdx.x == 0) s_status = *(volatile int32_t*)&st->status;
    __syncthreads();
    if (s_status != kRunning) return;
    const DaView d = da_view(w, ph.jobs, ph.floor);
    const int32_t count = ph.list ? st->da_wait : ph.count;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = warp / kGroup, gw = warp % kGroup;
    const bool leader = gw == 0 && lane == 0;
    uint32_t* s_b = s_bounds + (size_t)grp * d.tiles;
    const int32_t groups = (int32_t)gridDim.x * kGroups;
    int32_t looks = 0, longest = 0, tied = -kDaTieWait;
    const uint64_t t_start = globaltimer_ns();
    // (neighbouring agents on different SMs)
    int32_t next = grp * (int32_t)gridDim.x + (int32_t)blockIdx.x;
    while (next < count) {
        int32_t a = ph.list ? ph.list[next] : next, r, steps = 1;
        // the chain of displacements that starts with agent a
        while ((r = da_propose<kGroup>(d, a, s_b, s_sh[grp], grp, gw, looks, tied)) >= 0) {
            a = r;
            ++steps;
            if ((steps & 63) == 0) {  // bounded in time
                if (leader) s_next[grp] = globaltimer_ns() - t_start > kDaTimeoutNs;
                group_bar<kGroup>(grp);
                const bool late = s_next[grp] != 0;
                group_bar<kGroup>(grp);
                if (late) {
                    r = -3;
                    break;
                }
            }
        }
        longest = max(longest, steps);
        if (r == -4) {
            if (leader) ph.waits[a] = 1;
        } else if (r < -1) {
            if (leader) {
                st->error = r == -3 ? kErrWaitTimeout : kErrInternal;
                st->status = kError;
            }
            break;
        }
        if (leader) s_next[grp] = groups + atomicAdd(&st->da_next, 1);
        group_bar<kGroup>(grp);
        next = s_next[grp];
        group_bar<kGroup>(grp);
    }
    if (lane == 0 && looks) {
        atomicAdd((unsigned long long*)&st->greedy_rescans, (unsigned long long)looks);
        atomicMax(&st->greedy_rounds, longest);  // turns along the longest chain (a walk over ties is one)
    }
    if (leader && w.phase_ns) {  // diagnostics (DGS_PHASE_TIMERS=1)
        const uint64_t t = globaltimer_ns() - t_start;
        atomicMax(w.phase_ns + kPtDaLastNs, (unsigned long long)t);
        atomicAdd(w.phase_ns + kPtDaSumNs, (unsigned long long)t);
        atomicMax(w.phase_ns + kPtDaChain, (unsigned long long)longest);
        atomicMax(w.phase_ns + kPtDaGroupScans, (unsigned long long)looks);
    }
}

// Loop condition of the locally-dominant rounds run as a device-side loop
// (three kernels and this one per iteration): go on while agents are
// unmatched; more than n + 8 rounds is an internal error.
__global__ void greedy_loop_cond_kernel(Workspace w, unsigned long long cond) {
    DeviceState* st = w.st;
    const int32_t it = ++st->loop_iterations;
    st->loop_launches += 4;
    if (st->status == kRunning && st->greedy_remaining > 0 && it > w.n + 8) {
        st->error = kErrInternal;
        st->status = kError;
    }
    cudaGraphSetConditional(cond, (st->status == kRunning && st->greedy_remaining > 0) ? 1u : 0u);
}

// Between the two proposal phases of a padded instance with real_n agents and
// real_m jobs (one of them n): the free jobs go to the dummy agents, both in
// ascending order; or the dummy jobs to the waiting agents.  The agents that
// still wait are listed.  One CTA.
__global__ void __launch_bounds__(1024) greedy_rect_fill_kernel(Workspace w, int32_t real_n, int32_t real_m,
                                                               const uint8_t* waits, int32_t* list) {
    DeviceState* st = w.st;
    if (st->status != kRunning) return;
    __shared__ int32_t s_sums[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t n = w.n;
    constexpr unsigned long long kZero = (unsigned long long)kBenefitLimit << 32;  // a benefit of 0, biased
    // (marked entries of 0 .. n - 1, in order: take(index, rank))
    auto each_marked = [&](auto&& marked, auto&& take) -> int32_t {
        int32_t before = 0;
        for (int32_t c0 = 0; c0 < n; c0 += 1024) {
            const int32_t x = c0 + tid;
            const bool m = x < n && marked(x);
            const uint32_t b = __ballot_sync(0xffffffffu, m);
            if (lane == 0) s_sums[warp] = __popc(b);
            __syncthreads();
            const uint32_t sums = (uint32_t)s_sums[lane];
            const int32_t at = before + (int32_t)__reduce_add_sync(0xffffffffu, lane < warp ? sums : 0u) +
                               __popc(b & ((1u << lane) - 1u));
            before += (int32_t)__reduce_add_sync(0xffffffffu, sums);
            if (m) take(x, at);
            __syncthreads();
        }
        return before;
    };
    int32_t left;
    if (real_n < n) {
        const int32_t extra = n - real_n;
        each_marked([&](int32_t j) { return w.g_col[j] == 0ull; },
                    [&](int32_t j, int32_t r) {
                        if (r < extra) w.g_col[j] = kZero | (unsigned long long)(~(uint32_t)(real_n + r));
                    });
        left = each_marked([&](int32_t i) { return waits[i] != 0; }, [&](int32_t i, int32_t r) { list[r] = i; });
    } else {
        const int32_t extra = n - real_m;
        const int32_t all = each_marked([&](int32_t i) { return waits[i] != 0; },
                                        [&](int32_t i, int32_t r) {
                                            if (r < extra)
                                                w.g_col[real_m + r] = kZero | (unsigned long long)(~(uint32_t)i);
                                            else list[r - extra] = i;
                                        });
        left = all > extra ? all - extra : 0;
    }
    if (tid == 0) {
        st->da_wait = left;
        st->da_next = 0;
    }
}

// The start from the jobs' holders: both maps, D (the holder's key has the
// benefit) and f.
__global__ void __launch_bounds__(256) greedy_da_start_kernel(Workspace w) {
    DeviceState* st = w.st;
    // (uniform for the CTA, whose sum comes at the end: another CTA may report a
    // job without a holder meanwhile)
    if (__syncthreads_or(st->status != kRunning)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->greedy_remaining = 0;
    long long f = 0;
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < w.n; j += gridDim.x * blockDim.x) {
        const unsigned long long key = w.g_col[j];
        const int32_t i = key_index(key);
        if (i < 0 || i >= w.n) {
            st->error = kErrInternal;
            st->status = kError;
            continue;
        }
        const int32_t d = (int32_t)(key >> 32) - kBenefitLimit;
        w.sigma[j] = i;
        w.tau[i] = j;
        w.diag[j] = d;
        f += d;
    }
    add_objective(st, f);
}

// |a| < 2^29 check alone (for calls that neither run pass 1 nor a checking
// evaluation).  The pitched rows are read as one array (padding columns are 0,
// which changes nothing), four 16-byte loads in flight per thread: HBM-bound
// (n = 10000, 400 MB: 115 us with one load in flight and a column test per
// element, now 62).
__global__ void __launch_bounds__(256) range_check_kernel(Workspace w) {
    const int4* a = reinterpret_cast<const int4*>(w.a);
    const size_t total = (size_t)w.n * (size_t)(w.lda / 4), stride = (size_t)gridDim.x * blockDim.x;
    int32_t lo = 0, hi = 0;
    constexpr int kAhead = 4;
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += kAhead * stride) {
        int4 v[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) v[k] = q + k * stride < total ? a[q + k * stride] : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            lo = min(lo, min(min(v[k].x, v[k].y), min(v[k].z, v[k].w)));
            hi = max(hi, max(max(v[k].x, v[k].y), max(v[k].z, v[k].w)));
        }
    }
    report_range(w, lo, hi);
}

// The same, filling the pitched copy w.a from the caller's rows of n int32.
__global__ void __launch_bounds__(256) repitch_check_kernel(Workspace w, const int32_t* a_src) {
    const int lane = threadIdx.x & 31;
    int32_t lo = 0, hi = 0;
    for (int32_t i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); i < w.n; i += gridDim.x * (blockDim.x / 32)) {
        const int32_t* src = a_src + (size_t)i * w.n;
        int32_t* dst = const_cast<int32_t*>(w.a) + (size_t)i * w.lda;
        constexpr int kAhead = 8;
        for (int32_t j = lane; j < w.lda; j += 32 * kAhead) {
            int32_t x[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k) x[k] = j + 32 * k < w.n ? src[j + 32 * k] : 0;
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                if (j + 32 * k < w.lda) dst[j + 32 * k] = x[k];
                lo = min(lo, x[k]);
                hi = max(hi, x[k]);
            }
        }
    }
    report_range(w, lo, hi);
}

// Batched: pass 1 of the queued instances, items of about four tiles of one
// instance.  The CTAs take neighbouring items at the same time, so that what
// is read and written together lies together: with a contiguous range of items
// per CTA, in as many instances as there are CTAs, 1024 instances of n in
// [64, 4096] took 5.7 ms, now 4.2 (88% of the measured copy rate over the
// matrix, its transpose and the re-pitched copies).  Items of two or eight
// tiles: 4.4 ms.
__global__ void __launch_bounds__(256) greedy_pass1_batched_kernel(BatchQueues q) {
    const int32_t total = q.q0[q.cap];
    for (int32_t item = blockIdx.x; item < total; item += gridDim.x) {
        const int32_t k = find_slot(q.q0, q.cap, item);
        const int32_t bid = item - q.q0[k], nblk = q.q0[k + 1] - q.q0[k];
        const Instance& in = q.inst[k];
        const Workspace w = in.w;
        const int32_t tx = (w.n + kT - 1) / kT, tiles = tx * tx;
        greedy_pass1_body<true>(w, tx, tiles, bid, nblk, in.a_src);
    }
}

// Deferred acceptance of every instance in kStageGreedy in one launch: the
// agents of all those instances form one index space (prefix offsets q0 of
// the kScanGreedyDA scan, which also zeroes q1[0], the shared counter); a
// warp takes its first agents of that space by its number, later ones from
// the counter, and follows each one's chain of displacements inside its
// instance, exactly as greedy_da_kernel does for a single solve.
__global__ void __launch_bounds__(kDaThreads, kDaPerSm) greedy_da_batched_kernel(BatchQueues q) {
    __shared__ uint32_t s_bounds[kDaWarps][kInstanceBoundTiles];
    __shared__ DaShared<1> s_sh[kDaWarps];
    const int32_t total = q.q0[q.cap];
    if (total <= 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* s_b = s_bounds[warp];
    const int32_t warps = (int32_t)gridDim.x * kDaWarps;
    int32_t looks = 0, longest = 0, tied = -kDaTieWait, k_last = -1, first = 0, end = 0;
    DaView d{};
    auto flush = [&] {  // looks and chains are counted per instance
        if (k_last >= 0 && lane == 0 && looks) {
            DeviceState* st = q.inst[k_last].w.st;
            atomicAdd((unsigned long long*)&st->greedy_rescans, (unsigned long long)looks);
            atomicMax(&st->greedy_rounds, longest);
        }
        looks = longest = 0;
    };
    const int32_t per = total >= 4 * warps ? 4 : 1;  // agents taken at a time (one look-up of their instance)
    int32_t chunk = warp * (int32_t)gridDim.x + (int32_t)blockIdx.x;
    while ((int64_t)chunk * per < total) {
        const int32_t g_end = min(total, (chunk + 1) * per);
        for (int32_t g = chunk * per; g < g_end; ++g) {
            if (g < first || g >= end) {  // another instance
                flush();
                k_last = find_slot(q.q0, q.cap, g);
                first = q.q0[k_last];
                end = q.q0[k_last + 1];
                d = da_view(q.inst[k_last].w, q.inst[k_last].w.n, 1u);
            }
            int32_t a = g - first, r, steps = 1;
            while ((r = da_propose<1>(d, a, s_b, s_sh[warp], warp, 0, looks, tied)) >= 0) {
                a = r;
                ++steps;
            }
            longest = max(longest, steps);
            if (r == -2 && lane == 0) {
                DeviceState* st = q.inst[k_last].w.st;
                st->error = kErrInternal;
                st->status = kError;
            }
        }
        if (lane == 0) chunk = warps + atomicAdd(q.q1, 1);
        chunk = __shfl_sync(0xffffffffu, chunk, 0);
    }
    flush();
}

// The assignment of every instance in kStageGreedy from its jobs' holders
// (D and f follow in the start kernel).
__global__ void greedy_da_finish_batched_kernel(BatchTable t) {
    for_each_entry(t, kStageGreedy, [&](const Instance& in, int32_t bid, int32_t nblk) {
        const Workspace& w = in.w;
        DeviceState* st = w.st;
        // every queued agent of the instance was placed by the launch before
        // (the instance's blocks must not test greedy_remaining, which block
        // 0 clears here for the advance kernel)
        if (st->status != kRunning) return;
        if (bid == 0 && threadIdx.x == 0) st->greedy_remaining = 0;
        for (int32_t j = bid * blockDim.x + threadIdx.x; j < w.n; j += nblk * blockDim.x) {
            const int32_t i = key_index(w.g_col[j]);
            if (i < 0 || i >= w.n) {
                st->error = kErrInternal;
                st->status = kError;
                continue;
            }
            w.sigma[j] = i;
            w.tau[i] = j;
        }
    });
}

}  // namespace

cudaError_t launch_range_check(const Workspace& w, const int32_t* a_src, cudaStream_t s) {
    if (a_src != nullptr) repitch_check_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(w, a_src);
    else range_check_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(w);
    return cudaGetLastError();
}

// Pass 1 over the rows of tile rows [row_tile0, row_tile1) (64 rows each):
// the bands of a matrix that arrives in pieces can be processed as they land.
cudaError_t launch_greedy_pass1_rows(const Workspace& w, bool bounds, int32_t row_tile0, int32_t row_tile1,
                                     const int32_t* a_src, cudaStream_t s) {
    const int32_t tx = (w.n + kT - 1) / kT;
    const int32_t t0 = row_tile0 * tx, t1 = (row_tile1 < tx ? row_tile1 : tx) * tx;
    const int32_t count = t1 - t0;
    if (count <= 0) return cudaSuccess;
    const int32_t grid = count < dgs::device_sms() * 8 ? count : dgs::device_sms() * 8;
    if (bounds) greedy_pass1_kernel<true><<<grid, 256, 0, s>>>(w, tx, t1, t0, a_src);
    else greedy_pass1_kernel<false><<<grid, 256, 0, s>>>(w, tx, t1, t0, a_src);
    return cudaGetLastError();
}

cudaError_t launch_greedy_pass1_bounds(const Workspace& w, int32_t row_tile0, int32_t row_tile1, const int32_t* a_src,
                                       cudaStream_t s) {
    return launch_greedy_pass1_rows(w, true, row_tile0, row_tile1, a_src, s);
}
cudaError_t launch_greedy_pass1(const Workspace& w, const int32_t* a_src, cudaStream_t s) {
    return launch_greedy_pass1_rows(w, false, 0, (w.n + kT - 1) / kT, a_src, s);
}

cudaError_t launch_greedy_loop_cond(const Workspace& w, unsigned long long handle, cudaStream_t s) {
    greedy_loop_cond_kernel<<<1, 1, 0, s>>>(w, handle);
    return cudaGetLastError();
}

cudaError_t launch_greedy_best(const Workspace& w, cudaStream_t s) {
    const int32_t grid = dgs::device_sms() * 8;
    greedy_best_kernel<<<grid, 256, 0, s>>>(w, w.a, w.lda, w.g_row);
    greedy_best_kernel<<<grid, 256, 0, s>>>(w, w.at, w.ldt, w.g_col);
    return cudaGetLastError();
}

cudaError_t launch_greedy_round(const Workspace& w, cudaStream_t s) {
    const int32_t nb = (w.n + 255) / 256;
    greedy_match_kernel<<<nb < dgs::device_sms() * 4 ? nb : dgs::device_sms() * 4, 256, 0, s>>>(w);
    const int32_t g = w.n < dgs::device_sms() * 8 ? w.n : dgs::device_sms() * 8;  // one owner per CTA at a time
    greedy_rescan_kernel<<<g, 256, 0, s>>>(w, w.a, w.lda, w.g_row, w.free_a, w.free_j, 1);
    greedy_rescan_kernel<<<g, 256, 0, s>>>(w, w.at, w.ldt, w.g_col, w.free_j, w.free_a, 0);
    return cudaGetLastError();
}

// Pass 1 of the instances queued by the kScanPass1 scan (blocks over the
// 64x64 tiles of a).
cudaError_t launch_b_pass1(const BatchQueues& q, cudaStream_t s) {
    greedy_pass1_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(q);
    return cudaGetLastError();
}

// CTAs of a deferred acceptance launch with `smem` bytes of bounds per CTA: as
// many per SM as fit, so that all are resident.
int32_t da_grid(size_t smem) {
    int32_t per_sm = kDaPerSm;
    while (per_sm > 1 && per_sm * (smem + 2048) > 227 * 1024) --per_sm;
    return dgs::device_sms() * per_sm;
}

// The greedy start of every instance in kStageGreedy (deferred acceptance:
// queue the agents, one launch, then the assignments; the advance kernel
// moves the instances on once greedy_remaining is 0).
cudaError_t launch_b_greedy(const BatchTable& rows, const BatchQueues& q, cudaStream_t s) {
    cudaError_t e = launch_b_scan(q, kScanGreedyDA, s);
    if (e != cudaSuccess) return e;
    greedy_da_batched_kernel<<<da_grid(0), kDaThreads, 0, s>>>(q);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    greedy_da_finish_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(rows);
    return cudaGetLastError();
}



// DGS_GREEDY_ROUNDS=1: the locally-dominant rounds instead of deferred
// acceptance (tests; the same assignment).  Read at every call.
int32_t greedy_rounds_env() {
    const char* e = std::getenv("DGS_GREEDY_ROUNDS");
    return (e && std::atoi(e) == 1) ? 1 : 0;
}

// Chains that are followed at the same time: all of them up to n = 512, then
// at least 512 and half of the agents, at most what fits.  Where agents want the
// same jobs every chain in flight runs into the others (constant matrices, n =
// 1021 1.94 ms, 2.45 with a chain per agent; n = 1532 3.9, 4.8; n = 2100 6.4, 7.1;
// a third of the agents 1.95, 3.1, 5.1); elsewhere more chains gain little
// (peer-shaped n = 1021 66.2 us, 66.9; n = 1532 76.1, 75.1; n = 2100 92.3, 91.5; a
// third 66.5, 77.6, 93.6, and uniform values in [0, 1e6), n = 1532, 38.4, 37.6 and
// 40.5).
int32_t da_chains(int32_t n) { return std::min(n, std::max(512, (n + 1) / 2)); }

cudaError_t launch_greedy_da(const Workspace& w, int32_t real_n, int32_t real_m, cudaStream_t s) {
    if (greedy_rounds_env() || w.g_bound == nullptr) return cudaErrorNotSupported;
    constexpr int kGroups = kDaWarps / kDaGroup;
    const size_t smem = sizeof(uint32_t) * kGroups * (size_t)w.bound_tiles;
    cudaError_t e = ensure_smem_limit<greedy_da_kernel<kDaGroup>>(smem);
    if (e != cudaSuccess) return e;
    const int32_t grid = std::min(da_grid(smem), (da_chains(w.n) + kGroups - 1) / kGroups);
    if (real_n == w.n && real_m == w.n) {
        greedy_da_kernel<kDaGroup><<<grid, kDaThreads, smem, s>>>(w, DaPhase{nullptr, w.n, w.n, 1u, nullptr});
    } else {
        greedy_da_kernel<kDaGroup>
            <<<grid, kDaThreads, smem, s>>>(w, DaPhase{nullptr, real_n, real_m, (uint32_t)kBenefitLimit, w.free_a});
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        greedy_rect_fill_kernel<<<1, 1024, 0, s>>>(w, real_n, real_m, w.free_a, w.rescan_list);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        greedy_da_kernel<kDaGroup>
            <<<grid, kDaThreads, smem, s>>>(w, DaPhase{w.rescan_list, 0, real_m, 1u, nullptr});
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int32_t nb = (w.n + 255) / 256;
    greedy_da_start_kernel<<<nb < dgs::device_sms() * 4 ? nb : dgs::device_sms() * 4, 256, 0, s>>>(w);
    return cudaGetLastError();
}

}  // namespace dgs
