// k_control.cu -- the switching loop of Algorithm 3 (Section 5) on the GPU.
//
// Slots.  Agent slot i (priority t = i) holds agent i's candidate (gain,
// job j_i); job slot j (priority t = n + j) holds job j's candidate (gain,
// agent i_j).  A slot with gain > 0 proposes the 2-exchange of the agent
// pair {i, sigma(j_i)} or {sigma(j), i_j} (partners looked up in the current
// sigma); such slots are the edges of the conflict check.
//
// One sweep = CC (Algorithm 4) + parallel switch + re-evaluation:
//   * CC claims agent pairs in priority order.  Its result (the priority
//     greedy matching of the edges) is computed exactly, chunk by chunk of
//     the priority order: edges touching an agent claimed by an earlier chunk
//     are rejected at once; the chunk's other edges run deterministic
//     reservations among themselves (each writes its priority into both
//     agents with atomicMin; an edge holding both agents is accepted and
//     claims them; edges touching a claimed agent are rejected; repeat).
//     Rejected edges form the set C (reading R3).  An accepted edge has no
//     earlier accepted neighbour and every rejected edge has one, which is
//     exactly the sequential outcome.
//   * Accepted exchanges are agent-disjoint, so each commits independently
//     when its gain under the current sigma is > 0.
//   * Slots not in C are re-evaluated (reading R4) by reading the row-best
//     keys key_a / key_j, which the update kernels keep equal to a fresh
//     evaluation of every row under the current sigma.
//
// The controller is one CTA that keeps running sweeps while they commit
// nothing (sigma, hence every row best, is then unchanged and re-evaluation
// is a read of the keys).  A sweep that commits exchanges stops it: the
// update kernels re-evaluate the affected rows on the whole GPU, then the
// controller is launched again and refreshes every slot not in C.
#include <algorithm>
#include <cstdlib>

#include "../../include/dgs.h"
#include "dgs_internal.cuh"

namespace dgs {
namespace {

constexpr int kCtlThreads = 1024;

// Slot edge word: agent u (bits 0..16), agent v (17..33), applies (34): its
// exchange raises f under the current sigma, revives (35): the slot's row has
// a positive gain under the current sigma, so that re-evaluating the slot
// gives it a candidate again, place (36..40): the slot's place among the 32 of
// its chunk.  The edges of a chunk (32 consecutive slots) are stored from its
// first entry on, in slot order, with their number beside them.  Edge positions
// follow slot priority, so a position is a priority.
constexpr unsigned long long kApplies = 1ull << 34;
constexpr unsigned long long kRevives = 1ull << 35;
constexpr int kPlaceShift = 36;
__device__ __forceinline__ unsigned long long edge_word(int32_t u, int32_t v) {
    return (unsigned long long)(uint32_t)u | ((unsigned long long)(uint32_t)v << 17);
}
__device__ __forceinline__ int32_t edge_u(unsigned long long e) { return (int32_t)(e & 0x1FFFFu); }
__device__ __forceinline__ int32_t edge_v(unsigned long long e) { return (int32_t)((e >> 17) & 0x1FFFFu); }

__device__ __forceinline__ int32_t exchange_gain(const Workspace& w, int32_t u, int32_t v) {
    if (u == v) return 0;
    const int32_t ju = w.tau[u], jv = w.tau[v];
    return w.a[(size_t)u * w.lda + jv] + w.a[(size_t)v * w.lda + ju] - w.diag[ju] - w.diag[jv];
}

// Block-wide exclusive scan of one int per thread (1024 threads).
// (kT threads, at most 1024; warp_sums holds 33 entries)
template <int kT = 1024>
__device__ __forceinline__ int32_t block_scan(int32_t x, int32_t* warp_sums, int32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t incl = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int32_t o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int32_t v = lane < kT / 32 ? warp_sums[lane] : 0;
        int32_t wi = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t o = __shfl_up_sync(0xffffffffu, wi, off);
            if (lane >= off) wi += o;
        }
        warp_sums[lane] = wi - v;
        if (lane == 31) warp_sums[32] = wi;
    }
    __syncthreads();
    const int32_t r = warp_sums[warp] + incl - x;
    *total = warp_sums[32];
    __syncthreads();
    return r;
}

// Controller scratch placement.  Mode 2: reservations, 32-bit edges, the head
// of the accepted list, claims and edge states in shared memory; mode 1: the
// same, but the list's edges only when there are at most `edges` of them, else
// in global memory; mode 0: everything in global memory.  (The slot of each
// edge position is read only at a commit and when an edge comes back, and is
// in global memory.)
constexpr size_t kCtlStaticSmem = 2048;  // bound on the controller's static shared memory (checked at ControllerShared)
constexpr size_t kCtlSmemLimit = 227 * 1024 - kCtlStaticSmem;
constexpr int32_t kListCap = 2048;  // accepted (or coloured) positions listed in shared memory
constexpr int32_t kCand = 128;      // candidates listed at a time by a colouring window

struct CtlLayout {
    int32_t edges, list_cap;                                    // entries
    size_t edges_at, list, claimed, estate, bytes;              // byte offsets (res is first), total
};

__host__ __device__ __forceinline__ CtlLayout controller_layout(int32_t n, int32_t mode) {
    CtlLayout l{};
    l.edges_at = 4 * (size_t)n;
    l.list_cap = 2 * n < kListCap ? 2 * n : kListCap;
    const size_t rest = 3 * (size_t)n;  // claims (n) and edge states (2n)
    if (mode == 2) {
        l.edges = 2 * n;
    } else {
        const size_t used = l.edges_at + 2 * (size_t)l.list_cap + rest;
        const size_t room = used < kCtlSmemLimit ? (kCtlSmemLimit - used) / 4 : 0;
        l.edges = room < (size_t)n ? (int32_t)room : n;
    }
    l.list = l.edges_at + 4 * (size_t)l.edges;
    l.claimed = l.list + 2 * (size_t)l.list_cap;
    l.estate = l.claimed + (size_t)n;
    l.bytes = l.estate + 2 * (size_t)n;
    return l;
}

// Controller scratch.  res: per agent, the reservation key of the current DR
// round; claimed: per agent, the stamp of the sweep that claimed it; estate:
// per edge position (alive / applies / fresh bits); E: per edge position, the
// two agents of its exchange.  The list of accepted positions is two-tier:
// the first `cap` entries in shared memory (16-bit positions), the rest in
// global memory.
struct CtlScratch {
    uint32_t* res;
    uint8_t* claimed;
    uint8_t* estate;
    void* edges;
    int32_t* acc_g;  // accepted positions beyond the shared-memory part
};

// Edge states: alive, applicable, and whether the slot's re-evaluation gives
// a candidate (all fixed while no exchange commits, but for edges that are
// re-evaluated); the accepted edges of a committing sweep are marked kAccBit.
// A colouring window keeps colour + 1 (1..31) in the upper five bits.
enum : uint8_t { kAlive = 1, kAppl = 2, kRevive = 4, kAccBit = 8 };
constexpr int kColourShift = 3;

struct TwoTier {
    uint16_t* s;
    int32_t cap;
    int32_t* g;
    __device__ __forceinline__ void put(int32_t i, int32_t v) const {
        if (i < cap) s[i] = (uint16_t)v;
        else g[i - cap] = v;
    }
    __device__ __forceinline__ int32_t get(int32_t i) const { return i < cap ? (int32_t)s[i] : g[i - cap]; }
};

// Reservation key of edge position p in DR round r: each round's keys are
// smaller than every earlier round's, so reservations never need clearing
// (the array is reset once per key period).
constexpr uint32_t kPosBits = 18, kRoundSpanMax = 1u << 14;
__device__ __forceinline__ uint32_t round_base(uint32_t r, uint32_t span) {
    return (span - 1u - (r & (span - 1u))) << kPosBits;
}

template <typename EdgeT>
struct Codec;
template <>
struct Codec<uint32_t> {  // n <= 65535
    static __device__ __forceinline__ uint32_t make(int32_t u, int32_t v) { return (uint32_t)u | ((uint32_t)v << 16); }
    static __device__ __forceinline__ int32_t u(uint32_t e) { return (int32_t)(e & 0xFFFFu); }
    static __device__ __forceinline__ int32_t v(uint32_t e) { return (int32_t)(e >> 16); }
};
template <>
struct Codec<unsigned long long> {
    static __device__ __forceinline__ unsigned long long make(int32_t u, int32_t v) {
        return (unsigned long long)(uint32_t)u | ((unsigned long long)(uint32_t)v << 32);
    }
    static __device__ __forceinline__ int32_t u(unsigned long long e) { return (int32_t)(uint32_t)e; }
    static __device__ __forceinline__ int32_t v(unsigned long long e) { return (int32_t)(e >> 32); }
};


// An accepted slot of a quiet sweep is re-evaluated from its row's key, which
// stays current for as long as no exchange commits.  A slot whose row has no
// positive gain dies: its candidate arrays are left as they are, since a slot
// that is not in C at the next commit is refreshed from the keys there.  A
// slot that comes back records its candidate (it may be in C at the next
// commit); returns its edge.  (Reading the row's key, target and partner here,
// for the few slots that come back, costs less than having every slot's
// re-evaluation prepared before each controller launch.)
template <typename EdgeT>
__device__ __forceinline__ EdgeT revive_slot(const Workspace& w, int32_t t) {
    const int32_t n = w.n;
    if (t < n) {
        const unsigned long long key = w.key_a[w.tau[t]];
        const int32_t j = key_index(key);
        w.ag_gain[t] = key_gain(key);
        w.ag_job[t] = j;
        return Codec<EdgeT>::make(t, w.sigma[j]);
    }
    const unsigned long long key = w.key_j[t - n];
    w.jb_gain[t - n] = key_gain(key);
    w.jb_agent[t - n] = key_index(key);
    return Codec<EdgeT>::make(w.sigma[t - n], key_index(key));
}

// Colouring window.  In a sweep in which no accepted exchange applies (a quiet
// sweep) sigma does not change, so every accepted edge is stale and is only
// re-evaluated: it dies or comes back, applicable, at its position.  Round k
// of a run of such sweeps accepts the greedy set of the edges left after the
// rounds before it, so a stale edge is accepted exactly in the round that
// first-fit edge colouring in position order gives it (the smallest colour
// that no earlier stale edge sharing one of its agents has), and an
// applicable edge in the first round from its birth on that no earlier stale
// edge sharing an agent holds; the first such round ends the run with an
// event.  A window colours the stale edges with colours below a bound `cap`
// (at most kColourCap): cap falls to the first round in which an applicable
// edge is accepted, and to the round after the one in which an edge that
// comes back is accepted (it takes part from then on).  The cap rounds left
// are applied at once, as that many quiet sweeps.
//
// What bounds it: a quiet sweep of a long run accepts a handful of edges
// (2 to 6 of several thousand) and most of the list hangs on a few agents
// (those left with a poor job), a chain in which every colour depends on the
// one before, so latency.  The whole CTA lists, in position order, the next
// kCand edges that still have a free colour below cap, and for every 32 of
// them which earlier ones share an agent; one warp walks them 32 at a time.
// Each round, every edge without a pending earlier neighbour takes its lowest
// free colour, and where some agent has many of the 32, the pending edges at
// the first pending edge's busier agent get its free colours in order, all at
// once, up to the first whose other agent holds one of these colours or has a
// pending earlier edge elsewhere.  The list is short, so that the next one
// leaves out what closed since (128 listed; 64 and 32 were 2 to 6% slower on
// peer-shaped and distance instances, 512 on uniform ones).  Measured, the
// whole solve, against reservations over the whole list eight colours at a
// time: uniform [0, 1e6) n = 10000 12.0 -> 3.1 ms, n = 20000 31.0 -> 7.0 ms,
// distances n = 2048 from a random start 8.4 -> 6.3 ms.  (Cycles in windows,
// uniform n = 10000: one edge per step over 32-position chunks in place 5.0M,
// rounds over the edges without a pending earlier neighbour alone 5.7M, since
// nearly every round had one, this form 3.1M.)
//
// res (as colour masks): per agent, the colours held there (all zero on entry
// and on return).  Only with the scratch in shared memory; Eg: the edges, in
// shared memory when Eg == null.  Returns the number F of quiet sweeps run;
// s.hist holds each round's accepted count, and *event_next says that an
// applicable edge is accepted in the sweep after them.
constexpr int32_t kColourCap = 31;
// Coloured edges after which the bound is halved (31, 15, 7, 3, 1, then the
// window is given up), so that the list of coloured edges never outgrows its
// shared-memory part: that many edges per round are work for reservations.
constexpr int32_t kColourBudget = kListCap / 5 - 32;
// A window follows a quiet sweep that accepted at most this many edges: a
// sweep by reservations costs 7k cycles and more, the walk about 250 per edge
// (less where many share an agent), so both meet at 30 to 100.
constexpr int32_t kColourMaxAccepted = 64;

struct WindowShared {
    uint32_t cap, event_below;  // bounds as bit masks (event_below: ~0 without an event)
    int32_t cursor, next, coloured, rounds;
    int32_t hist[32], nth[32];
    uint32_t conf[kCand], word[kCand];  // the listed edges: agents in 15 bits each, applicable (15), comes back (31)
    uint16_t pos[kCand];
};

// Everything that the controller keeps in static shared memory.
struct ControllerShared {
    WindowShared win;
    unsigned long long pt[kPtCount];  // diagnostics
    unsigned long long gain, deadline;
    long long swaps, f;
    int32_t warp_sums[33];
    int32_t L, live, stop, acc, app, y, sweeps, event, max_sweeps, trace_cap, events;
    int32_t window;  // the next sweeps may run as a colouring window
    uint32_t round, stamp;
};
constexpr size_t kSmallLoopShared = 2 * sizeof(int32_t);  // small_loop_kernel's own
// (the dynamic part begins at the next multiple of 128)
static_assert((sizeof(ControllerShared) + kSmallLoopShared + 127) / 128 * 128 <= kCtlStaticSmem,
              "the launches ask for all shared memory but kCtlStaticSmem");

template <int kT>
__device__ __forceinline__ int32_t colour_window(const Workspace& w, const CtlLayout& lay, uint32_t* Eg, int32_t L,
                                                 int32_t limit, WindowShared& s, int32_t* warp_sums, int32_t& s_live,
                                                 bool* event_next, unsigned long long* s_pt) {
    using C = Codec<uint32_t>;
    constexpr int kWarps = kT / 32;
    constexpr uint32_t kAgent = 0x7FFFu, kApplBit = 1u << 15, kBackBit = 1u << 31;
    constexpr int kSpan = 4;  // positions per thread and step of the listing
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint32_t* const mask = reinterpret_cast<uint32_t*>(smem_raw);
    uint32_t* const Es = reinterpret_cast<uint32_t*>(smem_raw + lay.edges_at);
    uint16_t* const list = reinterpret_cast<uint16_t*>(smem_raw + lay.list);
    uint8_t* const estate = smem_raw + lay.estate;
    auto edge_at = [&](int32_t p) -> uint32_t { return Eg == nullptr ? Es[p] : Eg[p]; };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s.cap = (1u << min(limit, kColourCap)) - 1u;
        s.event_below = ~0u;
        s.cursor = 0;
        s.coloured = 0;
    }
    if (tid < 32) s.hist[tid] = 0;
    __syncthreads();
    for (;;) {
        // the next kCand positions that have a free colour below cap, in order
        const uint32_t cap0 = s.cap;
        int32_t base = s.cursor, count = 0;
        for (; base < L && count < kCand; base += kSpan * kT) {
            uint32_t word[kSpan], b[kSpan];
            int32_t mine = 0;
#pragma unroll
            for (int k = 0; k < kSpan; ++k) {
                const int32_t p = base + (warp * kSpan + k) * 32 + lane;
                const uint8_t es = p < L ? estate[p] : (uint8_t)0;
                const uint32_t e = (es & kAlive) ? edge_at(p) : 0u;
                const bool open = (es & kAlive) && (~(mask[C::u(e)] | mask[C::v(e)]) & cap0) != 0u;
                word[k] = e | ((es & kAppl) ? kApplBit : 0u) | ((es & kRevive) ? kBackBit : 0u);
                b[k] = __ballot_sync(0xffffffffu, open);
                mine += __popc(b[k]);
            }
            if (lane == 0) warp_sums[warp] = mine;
            __syncthreads();
            const uint32_t c = lane < kWarps ? (uint32_t)warp_sums[lane] : 0u;
            int32_t at = count + (int32_t)__reduce_add_sync(0xffffffffu, lane < warp ? c : 0u);
            count += (int32_t)__reduce_add_sync(0xffffffffu, c);
#pragma unroll
            for (int k = 0; k < kSpan; ++k) {
                const int32_t q = at + __popc(b[k] & ((1u << lane) - 1u));
                if (((b[k] >> lane) & 1u) && q < kCand) {
                    const int32_t p = base + (warp * kSpan + k) * 32 + lane;
                    s.word[q] = word[k];
                    s.pos[q] = (uint16_t)p;
                    if (q == kCand - 1) s.next = p + 1;
                }
                at += __popc(b[k]);
            }
            __syncthreads();
        }
        for (int32_t k = warp; k * 32 < min(count, kCand); k += kWarps) {
            const int32_t q = k * 32 + lane;
            const uint32_t word = q < count ? s.word[q] : 0u;
            const uint32_t u = word & kAgent, v = (word >> 16) & kAgent;
            uint32_t conf = 0u;
#pragma unroll
            for (int j = 0; j < 31; ++j) {
                const uint32_t wj = __shfl_sync(0xffffffffu, word, j);
                const uint32_t uj = wj & kAgent, vj = (wj >> 16) & kAgent;
                if (uj == u || vj == u || uj == v || vj == v) conf |= 1u << j;
            }
            s.conf[q] = conf & ((1u << lane) - 1u);
        }
        __syncthreads();
        if (warp == 0) {
            uint32_t cap = cap0, below = s.event_below;
            int32_t m = s.coloured, budget = kColourBudget;
            while (m >= budget) budget += kColourBudget;
            const uint32_t before = (1u << lane) - 1u;
            for (int32_t b0 = 0; b0 < min(count, kCand) && cap != 0u; b0 += 32) {
                const int32_t q = b0 + lane;
                const bool valid = q < count;
                const uint32_t word = valid ? s.word[q] : 0u;
                const uint32_t u = word & kAgent, v = (word >> 16) & kAgent;
                const bool appl = (word & kApplBit) != 0u;
                const uint32_t conf = s.conf[q];
                const bool busy = __any_sync(0xffffffffu, __popc(conf) >= 4);  // some agent has many of the 32
                uint32_t mu = mask[u], mv = mask[v], mine = 0u;
                uint32_t open = valid ? ~(mu | mv) & cap : 0u;
                uint32_t pend = __ballot_sync(0xffffffffu, open != 0u);
                while (pend) {
                    const bool ready = open != 0u && (pend & conf) == 0u;
                    uint32_t low = ready ? open & (0u - open) : 0u;
                    uint32_t x = u, h = v, at_h = 0u;
                    if (busy) {
                        // the first pending edge's agent with more pending edges
                        const int i = __ffs(pend) - 1;
                        const uint32_t wi = __shfl_sync(0xffffffffu, word, i);
                        const uint32_t ui = wi & kAgent, vi = (wi >> 16) & kAgent;
                        const uint32_t hu = __ballot_sync(0xffffffffu, open && (u == ui || v == ui));
                        const uint32_t hv = __ballot_sync(0xffffffffu, open && (u == vi || v == vi));
                        const bool pick_u = __popc(hu) >= __popc(hv);
                        const uint32_t hub = pick_u ? ui : vi;
                        at_h = pick_u ? hu : hv;
                        const uint32_t free = ~mask[hub] & cap;
                        if ((free >> lane) & 1u) s.nth[__popc(free & before)] = lane;
                        if ((at_h >> lane) & 1u) {
                            h = hub;
                            x = u == hub ? v : u;
                        }
                        const uint32_t mx = u == hub ? mv : mu;  // (of the edges at the hub: their other agent's colours)
                        const uint32_t badm = __ballot_sync(
                            0xffffffffu, ((at_h >> lane) & 1u) && ((mx & free) != 0u || (conf & pend & ~at_h) != 0u));
                        // (the first edge bad: by itself, from both its agents' colours)
                        const uint32_t take = at_h & ((badm & (0u - badm)) - 1u);
                        __syncwarp();
                        if ((take >> lane) & 1u) {
                            const int32_t r = __popc(take & before);
                            low = r < __popc(free) ? 1u << s.nth[r] : 0u;
                        }
                    }
                    uint32_t bound = ~0u;
                    if (low != 0u && appl) {
                        bound = low - 1u;
                        below = min(below, bound);
                    } else if (low != 0u && (word & kBackBit)) {
                        bound = (low << 1) - 1u;
                    }
                    cap &= __reduce_and_sync(0xffffffffu, bound);
                    const bool taken = !appl && (low & cap) != 0u;
                    if (taken) {
                        mine = low;
                        atomicOr(&mask[x], low);
                    }
                    if (busy) {  // the hub's edges raise its mask once
                        const bool in = (at_h >> lane) & 1u;
                        const uint32_t add = __reduce_or_sync(0xffffffffu, taken && in ? low : 0u);
                        if (taken && !in) atomicOr(&mask[h], low);
                        if (lane == __ffs(at_h) - 1) atomicOr(&mask[h], add);
                    } else if (taken) {
                        atomicOr(&mask[h], low);
                    }
                    __syncwarp();
                    mu = mask[u];
                    mv = mask[v];
                    open = valid && mine == 0u ? ~(mu | mv) & cap : 0u;
                    pend = __ballot_sync(0xffffffffu, open != 0u);
                }
                const uint32_t cm = __ballot_sync(0xffffffffu, mine != 0u);
                if (mine != 0u) {
                    const int32_t c = __ffs(mine) - 1, p = s.pos[q];
                    atomicAdd(&s.hist[c], 1);
                    estate[p] = (uint8_t)(kAlive | ((word & kBackBit) ? kRevive : 0) | ((c + 1) << kColourShift));
                    list[m + __popc(cm & before)] = (uint16_t)p;
                }
                m += __popc(cm);
                if (m >= budget) {  // more edges per round than this form is for
                    budget += kColourBudget;
                    cap &= cap >> ((__popc(cap) + 1) / 2);
                }
            }
            below = __reduce_min_sync(0xffffffffu, below);
            if (lane == 0) {
                s.cap = cap;
                s.cursor = count >= kCand ? s.next : L;
                s.coloured = m;
                s.event_below = below;
                if (s_pt) s_pt[kPtCtlColourWalks] += 1;
            }
        }
        __syncthreads();
        if (s.cap == 0u || s.cursor >= L) break;
    }
    if (warp == 0) {
        // a round with live edges accepts at least one (and an edge of colour
        // c has neighbours of every colour below c): the run ends before the
        // first empty round
        const int32_t bound = __popc(s.cap);
        const uint32_t full = __ballot_sync(0xffffffffu, lane < bound && s.hist[lane] > 0);
        if (lane == 0) s.rounds = __popc(full);
    }
    __syncthreads();
    const int32_t F = s.rounds, m = s.coloured;
    int32_t died = 0;
    for (int32_t q = tid; q < m; q += kT) {
        const int32_t p = list[q];
        const uint8_t es = estate[p];
        const uint32_t e = edge_at(p);
        mask[C::u(e)] = 0u;
        mask[C::v(e)] = 0u;
        uint8_t now = es & (uint8_t)((1 << kColourShift) - 1);
        if ((es >> kColourShift) <= F) {  // accepted in one of the F rounds: re-evaluated
            if (es & kRevive) {
                const uint32_t back = revive_slot<uint32_t>(w, w.ctl_slot[p]);
                if (Eg == nullptr) Es[p] = back;
                else Eg[p] = back;
                now = kAlive | kAppl;
            } else {
                now = 0;
                ++died;
            }
        }
        estate[p] = now;
    }
    if (died) atomicSub(&s_live, died);
    if (s_pt && tid == 0) s_pt[kPtCtlColourEdges] += m;
    *event_next = s.event_below == s.cap && __popc(s.cap) == F;
    __syncthreads();
    return F;
}

// Switching loop (see the file comment).
// span: reservation-key period (power of two <= kRoundSpanMax); stamp_wrap:
// claim-stamp period (<= 255).  Both are shortened only by a test knob.
// colour_pass: runs of quiet sweeps go through colouring windows (only with
// the scratch in shared memory); 0 turns them off.
template <typename EdgeT, int kT = kCtlThreads>
__device__ __forceinline__ void controller_body(const Workspace& w, int32_t smem_mode, const CtlScratch& g,
                                                uint32_t span, uint32_t stamp_wrap, int32_t compact_min,
                                                int32_t colour_pass) {
    using C = Codec<EdgeT>;
    DeviceState* st = w.st;
    if (st->status != kRunning) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ ControllerShared sh;
    int32_t(&warp_sums)[33] = sh.warp_sums;
    int32_t &s_L = sh.L, &s_live = sh.live, &s_stop = sh.stop, &s_acc = sh.acc, &s_app = sh.app, &s_y = sh.y;
    int32_t &s_sweeps = sh.sweeps, &s_event = sh.event, &s_max_sweeps = sh.max_sweeps, &s_trace_cap = sh.trace_cap;
    int32_t &s_events = sh.events, &s_window = sh.window;
    WindowShared& s_win = sh.win;
    uint32_t &s_round = sh.round, &s_stamp = sh.stamp;
    unsigned long long &s_gain = sh.gain, &s_deadline = sh.deadline;
    long long &s_swaps = sh.swaps, &s_f = sh.f;

    const int32_t n = w.n;
    const int tid = threadIdx.x;
    uint32_t* res = g.res;
    uint8_t* claimed = g.claimed;
    uint8_t* estate = g.estate;
    EdgeT* E = static_cast<EdgeT*>(g.edges);
    uint16_t* lists_s = nullptr;
    int32_t list_cap = 0, es_cap = 0;
    EdgeT* Es = nullptr;
    if (smem_mode >= 1) {
        const CtlLayout lay = controller_layout(n, smem_mode);
        list_cap = lay.list_cap;
        es_cap = sizeof(EdgeT) == 4 ? lay.edges : 0;
        res = reinterpret_cast<uint32_t*>(smem_raw);
        Es = reinterpret_cast<EdgeT*>(smem_raw + lay.edges_at);
        lists_s = reinterpret_cast<uint16_t*>(smem_raw + lay.list);
        claimed = smem_raw + lay.claimed;
        estate = smem_raw + lay.estate;
        if (smem_mode == 2) E = Es;
    }
    // Mode 1: the edges of a launch whose list is at most es_cap long, or is
    // compacted to that length, are in shared memory, longer lists' in global.
    TwoTier accl{lists_s, list_cap, g.acc_g};
    unsigned long long* pt = (tid == 0) ? w.phase_ns : nullptr;
    long long tp = clock64();
    // diagnostics (DGS_PHASE_TIMERS=1): thread 0 sums into shared memory and
    // adds the sums to global memory once per launch, so that the counters
    // add no global round trips to the loops they time
    unsigned long long(&s_pt)[kPtCount] = sh.pt;
    if (pt)
        for (int k = 0; k < kPtCount; ++k) s_pt[k] = 0ull;
#define DGS_PT(slot, v) \
    if (pt) s_pt[slot] += (unsigned long long)(v);
#define DGS_CT(slot)                     \
    if (pt) {                            \
        const long long now = clock64(); \
        s_pt[slot] += (unsigned long long)(now - tp); \
        tp = now;                        \
    }

    // ---------------------------------------------------------------- entry
    // The slot refresh and the per-slot edge data were prepared by the grid
    // (prepare_edges_kernel); here the edges are listed in priority order.
    {
        // Warp wp lists the chunks of its own range (ranges ascend with wp): it
        // sums their edge counts, and with the 32 warps' sums each warp knows
        // where its edges go, so positions follow slot order (the priority
        // order).  (The loads first, then the clearing, which waits for
        // nothing.)
        constexpr int kWarps = kT / 32;
        const int32_t lane = tid & 31, wp = tid >> 5;
        const int32_t nchunks = (2 * n + 31) >> 5;
        const int32_t per = (nchunks + kWarps - 1) / kWarps;
        const int32_t c_lo = min(nchunks, wp * per), c_hi = min(nchunks, c_lo + per);
        uint32_t cnt = 0;
        for (int32_t c = c_lo + lane; c < c_hi; c += 32) cnt += (uint32_t)w.sl_chunk[c];
        if (tid == 0) {
            s_swaps = st->swaps;
            s_events = st->events;
            s_sweeps = st->sweeps;
            s_max_sweeps = st->max_sweeps;
            s_deadline = st->deadline_ns;
            s_trace_cap = st->trace_capacity;
            s_f = st->f;
            st->need_update = 0;
            st->y_count = 0;
            s_round = 0;
            s_stamp = 0;
            s_window = 0;
        }
        // (in words of 16 and 4 bytes: what lies past the last one's end is
        // padding, or edges and states that are written only later)
        for (int32_t i = tid; i < (n + 3) / 4; i += kT) {
            reinterpret_cast<uint4*>(res)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
            reinterpret_cast<uint32_t*>(claimed)[i] = 0u;
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) warp_sums[wp] = (int32_t)cnt;
        __syncthreads();
        const uint32_t sums = lane < kWarps ? (uint32_t)warp_sums[lane] : 0u;
        const int32_t total = (int32_t)__reduce_add_sync(0xffffffffu, sums);
        int32_t pos0 = (int32_t)__reduce_add_sync(0xffffffffu, lane < wp ? sums : 0u);
        if (es_cap > 0 && total <= es_cap) E = Es;  // the whole list fits in shared memory
        auto list_edge = [&](int32_t pos, int32_t c, unsigned long long e) {
            w.ctl_slot[pos] = c * 32 + (int32_t)((e >> kPlaceShift) & 31u);
            E[pos] = C::make(edge_u(e), edge_v(e));
            estate[pos] = kAlive | ((e & kApplies) ? kAppl : 0) | ((e & kRevives) ? kRevive : 0);
        };
        for (int32_t cb = c_lo; cb < c_hi; cb += 32) {
            const int32_t mine = cb + lane < c_hi ? w.sl_chunk[cb + lane] : 0;
            int32_t incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t o = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += o;
            }
            const int32_t excl = incl - mine, edges = __shfl_sync(0xffffffffu, incl, 31);
            // the edges of these 32 chunks, one per lane and step wherever they
            // are (a search in the prefix sums finds the chunk), kAhead steps'
            // loads in flight
            constexpr int kAhead = 4;
            for (int32_t q0 = 0; q0 < edges; q0 += 32 * kAhead) {
                int32_t c[kAhead];
                unsigned long long e[kAhead];
#pragma unroll
                for (int k = 0; k < kAhead; ++k) {
                    const int32_t q = q0 + 32 * k + lane;
                    c[k] = 0;
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(0xffffffffu, excl, c[k] + step) <= q) c[k] += step;
                    const int32_t at = q - __shfl_sync(0xffffffffu, excl, c[k]);
                    c[k] += cb;
                    e[k] = q < edges ? w.sl_edge[(size_t)c[k] * 32 + at] : 0ull;
                }
#pragma unroll
                for (int k = 0; k < kAhead; ++k) {
                    const int32_t q = q0 + 32 * k + lane;
                    if (q < edges) list_edge(pos0 + q, c[k], e[k]);
                }
            }
            pos0 += edges;
        }
        if (tid == 0) s_L = s_live = total;
        __syncthreads();
    }
    DGS_CT(kPtCtlEntry)

    // ------------------------------------------------------------- sweeps
    // Quiet sweeps turn at least one stale slot into a fresh one each, so one
    // launch runs at most 2n + 1 of them; more means an internal error.
    int32_t L = s_L;
    bool masks = false;  // res holds the agents' colour masks, all zero (else reservation keys)
    for (int32_t quiet = 0;; ++quiet) {
        if (tid == 0) {
            // loop condition of Algorithm 3 (some slot has delta > 0), sweep
            // cap and deadline; decided by one thread so that all agree
            int32_t stop = 0;
            if (s_live == 0) {
                st->status = kDone;
                stop = 1;
            } else if ((s_max_sweeps > 0 && s_sweeps >= s_max_sweeps) ||
                       (s_deadline != 0 && globaltimer_ns() > s_deadline)) {
                st->status = kTimeout;
                stop = 1;
            } else if (quiet > 2 * n + 1) {
                st->error = kErrInternal;
                st->status = kError;
                stop = 1;
            }
            s_stop = stop;
            s_acc = 0; s_app = 0; s_y = 0; s_gain = 0ull; s_event = 0;
            s_stamp = s_stamp + 1u;
        }
        __syncthreads();
        DGS_CT(kPtCtlTop)
        if (s_stop) break;
        DGS_PT(kPtCtlSweeps, 1)
        DGS_PT(kPtCtlLiveSum, s_live)
        DGS_PT(kPtCtlListSum, L)
        // An edge that dies in a quiet sweep never lives again in this launch.
        // Once fewer than half of the L listed positions are live, compact the
        // list in place, keeping the priority order (positions are
        // priorities, and deterministic reservations depend only on their
        // order), so that later sweeps scan live edges only; the reservation
        // keys restart with the new positions.
        if (s_live * 2 < L && L >= compact_min) {
            // (mode 1: into shared memory when the live edges fit there)
            EdgeT* const Ed = s_live <= es_cap ? Es : E;
            const bool bounded = es_cap > 0 && Ed == Es;
            int32_t base = 0;
            for (int32_t c0 = 0; c0 < L; c0 += kT) {
                const int32_t p = c0 + tid;
                const uint8_t es = p < L ? estate[p] : (uint8_t)0;
                const bool alive = (es & kAlive) != 0;
                const EdgeT e = alive ? E[p] : (EdgeT)0;
                const int32_t slot = alive ? w.ctl_slot[p] : 0;
                int32_t total;
                const int32_t pos = base + block_scan<kT>(alive ? 1 : 0, warp_sums, &total);  // every read is done
                if (alive) {
                    if (!bounded || pos < es_cap) Ed[pos] = e;
                    estate[pos] = es;
                    w.ctl_slot[pos] = slot;
                }
                base += total;
            }
            if (!masks)
                for (int32_t i = tid; i < n; i += kT) res[i] = 0xFFFFFFFFu;
            __syncthreads();
            if (tid == 0) {
                s_L = base;
                s_round = 0u;
                if (bounded && base > es_cap) {  // the live count disagreed with the list
                    st->error = kErrInternal;
                    st->status = kError;
                    s_stop = 1;
                }
            }
            __syncthreads();
            if (s_stop) break;
            L = s_L;
            E = Ed;
        }
        // Colouring window (see colour_window): F >= 1 quiet sweeps at once,
        // or none when an applicable edge is accepted in this very sweep (or
        // the window was given up); then this sweep goes on as usual.
        // (shared-memory modes hold n <= 32767: 32-bit edges)
        if (sizeof(EdgeT) == 4 && colour_pass && smem_mode >= 1 && s_window) {
            if (!masks) {
                for (int32_t i = tid; i < n; i += kT) res[i] = 0u;
                masks = true;
                __syncthreads();
            }
            const int32_t left = s_max_sweeps > 0 ? s_max_sweeps - s_sweeps : kColourCap;
            bool event_next;
            const int32_t F =
                colour_window<kT>(w, controller_layout(n, smem_mode), E == Es ? nullptr : reinterpret_cast<uint32_t*>(E),
                                  L, left, s_win, warp_sums, s_live, &event_next, pt ? s_pt : nullptr);
            if (tid < F) {
                const int32_t sw = s_sweeps + tid;
                if (sw < s_trace_cap) {
                    if (st->trace_accepted) st->trace_accepted[sw] = s_win.hist[tid];
                    if (st->trace_applied) st->trace_applied[sw] = 0;
                    if (st->trace_objective) st->trace_objective[sw] = s_f;
                }
            }
            __syncthreads();
            if (tid == 0) {
                s_sweeps = s_sweeps + F;
                s_window = (F > 0 && !event_next) ? 1 : 0;
                DGS_PT(kPtCtlColourPasses, 1)
                DGS_PT(kPtCtlColourRounds, F)
            }
            __syncthreads();
            DGS_CT(kPtCtlColour)
            if (F > 0) continue;
        }
        if (s_stamp >= stamp_wrap) {  // claim stamps wrap: clear them once
            for (int32_t i = tid; i < n; i += kT) claimed[i] = 0;
            __syncthreads();
            if (tid == 0) s_stamp = 1;
            __syncthreads();
        }
        if (masks || ((s_round & (span - 1u)) == 0u && s_round != 0u)) {  // no keys yet, or they wrap
            for (int32_t i = tid; i < n; i += kT) res[i] = 0xFFFFFFFFu;
            masks = false;
            __syncthreads();
        }
        const uint8_t stamp = (uint8_t)s_stamp;
        // CC (Algorithm 4): the accepted set is the greedy one in priority
        // order (a slot is accepted when neither agent of its exchange was
        // claimed by an earlier accepted slot).  The list is taken in chunks
        // of one edge per thread, in order: an edge touching an agent claimed
        // by an earlier chunk is rejected at once; the chunk's other edges
        // are decided among themselves by deterministic reservations (each
        // round, the remaining candidates reserve both agents with a key that
        // orders them by position; an edge holding both reservations is
        // accepted and claims its agents; an edge touching a newly claimed
        // agent is rejected; the first remaining candidate always wins, so
        // every round accepts at least one edge).  Claims of a chunk reach
        // the next through a barrier, so the result is the greedy one.
        {
            int32_t ev = 0;
            // edges per thread and chunk (a chunk is kPer * kT
            // positions); four per thread crossed fewer barriers but was
            // slower (uniform n = 10000: 22.2 ms against 18.8 ms), so one
            constexpr int kPer = 1;
            for (int32_t c0 = 0; c0 < L; c0 += kPer * kT) {
                int32_t p[kPer], u[kPer], v[kPer];
                uint8_t es[kPer];
                bool cand[kPer];
                bool any = false;
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    p[k] = c0 + k * kT + tid;
                    es[k] = p[k] < L ? estate[p[k]] : (uint8_t)0;
                    u[k] = 0;
                    v[k] = 0;
                    cand[k] = false;
                    if (es[k] & kAlive) {
                        const EdgeT e = E[p[k]];
                        u[k] = C::u(e);
                        v[k] = C::v(e);
                        cand[k] = claimed[u[k]] != stamp && claimed[v[k]] != stamp;
                    }
                    any |= cand[k];
                }
                for (int32_t r = 0; __syncthreads_or(any); ++r) {
                    if (r > kPer * kT) {  // every round accepts the first candidate
                        if (tid == 0) {
                            st->error = kErrInternal;
                            st->status = kError;
                            s_stop = 1;
                        }
#pragma unroll
                        for (int k = 0; k < kPer; ++k) cand[k] = false;
                        any = false;
                        continue;
                    }
                    if ((s_round & (span - 1u)) == 0u && s_round != 0u) {  // reservation keys wrap
                        for (int32_t i = tid; i < n; i += kT) res[i] = 0xFFFFFFFFu;
                        __syncthreads();
                    }
                    const uint32_t base = round_base(s_round, span);
#pragma unroll
                    for (int k = 0; k < kPer; ++k) {
                        if (!cand[k]) continue;
                        // (lanes of a warp that reserve the same agent were
                        // first made to agree on their smallest key with
                        // __match_any_sync / __reduce_min_sync: 3.7 times
                        // slower on uniform n = 10000, so every candidate
                        // issues its own atomics)
                        const uint32_t key = base | (uint32_t)p[k];
                        if (key < res[u[k]]) atomicMin(&res[u[k]], key);
                        if (key < res[v[k]]) atomicMin(&res[v[k]], key);
                    }
                    __syncthreads();
#pragma unroll
                    for (int k = 0; k < kPer; ++k) {
                        const uint32_t key = base | (uint32_t)p[k];
                        if (cand[k] && res[u[k]] == key && res[v[k]] == key) {
                            claimed[u[k]] = stamp;
                            claimed[v[k]] = stamp;
                            const int32_t idx = atomicAdd(&s_acc, 1);
                            accl.put(idx, p[k]);
                            ev |= (es[k] & kAppl) ? 1 : 0;
                            cand[k] = false;
                        }
                    }
                    __syncthreads();  // this round's claims are visible
                    any = false;
#pragma unroll
                    for (int k = 0; k < kPer; ++k) {
                        if (cand[k] && (claimed[u[k]] == stamp || claimed[v[k]] == stamp)) cand[k] = false;  // rejected
                        any |= cand[k];
                    }
                    if (tid == 0) s_round = s_round + 1u;
                }
            }
            if (ev) s_event = 1;
            __syncthreads();
        }
        DGS_CT(kPtCtlPass1)
        if (s_stop) break;  // an internal error of the conflict check
        const int32_t nacc = s_acc;
        if (s_event) {
            // parallel switch: accepted exchanges are agent-disjoint; those
            // that raise f under the current sigma commit.  C (every live slot
            // that was not accepted) keeps its candidates (reading R4); its
            // marks are cleared where they are read (prepare_edges_body).
            // (The sums go through the warp first: 64-bit atomics of every
            // thread on one shared word are retry loops.)
            for (int32_t q = tid; q < nacc; q += kT) estate[accl.get(q)] |= kAccBit;
            __syncthreads();
            const int32_t slot0 = tid < L ? w.ctl_slot[tid] : 0;  // in flight during the commits
            const int lane = tid & 31;
            for (int32_t q0 = tid - lane; q0 < nacc; q0 += kT) {
                const int32_t q = q0 + lane;
                const int32_t p = q < nacc ? accl.get(q) : 0;
                const bool commits = q < nacc && (estate[p] & kAppl);
                const uint32_t cm = __ballot_sync(0xffffffffu, commits);
                if (cm == 0u) continue;
                int32_t qy = 0;
                if (lane == 0) {
                    qy = atomicAdd(&s_y, 2 * __popc(cm));
                    atomicAdd(&s_app, __popc(cm));
                }
                qy = __shfl_sync(0xffffffffu, qy, 0) + 2 * __popc(cm & ((1u << lane) - 1u));
                long long gain = 0;
                if (commits) {
                    const EdgeT e = E[p];
                    const int32_t u = C::u(e), v = C::v(e);
                    const int32_t ju = w.tau[u], jv = w.tau[v];
                    const int32_t x1 = w.a[(size_t)u * w.lda + jv];
                    const int32_t x2 = w.a[(size_t)v * w.lda + ju];
                    gain = (long long)x1 + x2 - w.diag[ju] - w.diag[jv];
                    w.tau[u] = jv;
                    w.tau[v] = ju;
                    w.sigma[jv] = u;
                    w.sigma[ju] = v;
                    w.diag[jv] = x1;
                    w.diag[ju] = x2;
                    w.y_list[qy] = ju;
                    w.y_list[qy + 1] = jv;
                    w.in_y[ju] = 1;
                    w.in_y[jv] = 1;
                    w.moved[u] = 1;
                    w.moved[v] = 1;
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) gain += __shfl_xor_sync(0xffffffffu, gain, off);
                if (lane == 0) atomicAdd(&s_gain, (unsigned long long)gain);
            }
            for (int32_t p = tid; p < L; p += kT) {
                const uint8_t es = estate[p];
                if (!(es & kAlive) || (es & kAccBit)) continue;
                const int32_t t = p == tid ? slot0 : w.ctl_slot[p];
                if (t < n) w.in_ca[t] = 1;
                else w.in_cj[t - n] = 1;
            }
            __syncthreads();  // the sums are complete
            if (tid == 0) {
                const int32_t sw = s_sweeps;
                s_f += (long long)s_gain;
                s_swaps += s_app;
                if (sw < s_trace_cap) {
                    if (st->trace_accepted) st->trace_accepted[sw] = nacc;
                    if (st->trace_applied) st->trace_applied[sw] = s_app;
                    if (st->trace_objective) st->trace_objective[sw] = s_f;
                }
                s_sweeps = sw + 1;
                s_events += 1;
                st->y_count = s_y;
                st->rescan_count = 0;
                st->need_update = 1;
                st->phase = kPhaseRefreshAll;
            }
            DGS_CT(kPtCtlEvent)
            break;
        }
        // quiet sweep: sigma unchanged, so the keys are current.  Accepted
        // slots are re-evaluated (their precomputed outcome); the others stay
        // in C with their candidates for the next sweep.
        int32_t died = 0;
        for (int32_t q = tid; q < nacc; q += kT) {
            const int32_t p = accl.get(q);
            if (estate[p] & kRevive) {
                E[p] = revive_slot<EdgeT>(w, w.ctl_slot[p]);
                estate[p] = kAlive | kAppl;
            } else {
                estate[p] = 0;
                ++died;
            }
        }
        if (died) atomicSub(&s_live, died);
        if (tid == 0) s_window = nacc <= kColourMaxAccepted ? 1 : 0;
        DGS_PT(kPtCtlAccSum, nacc)
        if (tid == 0 && s_sweeps < s_trace_cap) {
            const int32_t sw = s_sweeps;
            if (st->trace_accepted) st->trace_accepted[sw] = nacc;
            if (st->trace_applied) st->trace_applied[sw] = 0;
            if (st->trace_objective) st->trace_objective[sw] = s_f;
        }
        if (tid == 0) s_sweeps = s_sweeps + 1;
        __syncthreads();
        DGS_CT(kPtCtlPost)
    }
#undef DGS_CT
#undef DGS_PT
    if (pt)
        for (int k = 0; k < kPtCount; ++k)
            if (s_pt[k]) atomicAdd(pt + k, s_pt[k]);
    if (tid == 0) {
        st->sweeps = s_sweeps;
        st->edge_count = s_live;
        st->f = s_f;
        st->swaps = s_swaps;
        st->events = s_events;
    }
    __syncthreads();  // shared memory is reused by the caller's next call
}

// counted: the launch is the last kernel of an iteration of the device-side
// switching loop (a conditional WHILE graph node, five kernels per iteration).
// The loop is bounded: more than 16 n + 4096 iterations is an internal error.
// cond != 0: it also sets the loop condition from the loop state.
template <typename EdgeT>
__global__ void __launch_bounds__(kCtlThreads, 1) controller_kernel(Workspace w, int32_t smem_mode, CtlScratch g,
                                                                   uint32_t span, uint32_t stamp_wrap,
                                                                   int32_t compact_min, int32_t colour_pass,
                                                                   int32_t counted, unsigned long long cond) {
    controller_body<EdgeT>(w, smem_mode, g, span, stamp_wrap, compact_min, colour_pass);
    if (counted && threadIdx.x == 0) {
        DeviceState* st = w.st;
        const int32_t it = ++st->loop_iterations;
        st->loop_launches += 5;
        if (st->status == kRunning && it > 16 * w.n + 4096) {
            st->error = kErrInternal;
            st->status = kError;
        }
        if (cond != 0) cudaGraphSetConditional(cond, st->status == kRunning ? 1u : 0u);
    }
}

// Before each controller launch: clear the marks of the last event, re-
// evaluate every slot not in C from the current row keys (reading R4), and
// for every slot with a candidate (delta > 0) record its edge (the agents of
// its exchange under the current sigma, whether that exchange raises f now,
// and whether the slot's re-evaluation would give it a candidate).  One
// thread per slot.
__device__ __forceinline__ void prepare_edges_body(const Workspace& w, int32_t bid, int32_t nblk) {
    DeviceState* st = w.st;
    if (st->status != kRunning) return;
    const int32_t n = w.n;
    const int32_t stride = nblk * blockDim.x;
    const int32_t yc = st->y_count;
    const bool reeval_all = st->reeval_all != 0;
    for (int32_t t = bid * blockDim.x + threadIdx.x; t < yc; t += stride) {
        const int32_t j = w.y_list[t];
        w.in_y[j] = 0;
        w.moved[w.sigma[j]] = 0;
    }
    // (whole warps: 32 consecutive slots form one chunk)
    const int32_t lane = (int32_t)(threadIdx.x & 31u);
    for (int32_t t0 = bid * blockDim.x + threadIdx.x - lane; t0 < 2 * n; t0 += stride) {
        const int32_t t = t0 + lane;
        unsigned long long key = 0ull;
        int32_t gain = 0, target = -1;
        bool in_c;
        if (t < n) {
            key = w.key_a[w.tau[t]];
            in_c = w.in_ca[t];
            if (in_c) w.in_ca[t] = 0;  // the next commit marks its own
            in_c = in_c && !reeval_all;
            if (!in_c) {
                w.ag_gain[t] = key ? key_gain(key) : 0;
                w.ag_job[t] = key ? key_index(key) : -1;
            }
            gain = in_c ? w.ag_gain[t] : (key ? key_gain(key) : 0);
            target = in_c ? w.ag_job[t] : (key ? key_index(key) : -1);
        } else if (t < 2 * n) {
            const int32_t j = t - n;
            key = w.key_j[j];
            in_c = w.in_cj[j];
            if (in_c) w.in_cj[j] = 0;
            in_c = in_c && !reeval_all;
            if (!in_c) {
                w.jb_gain[j] = key ? key_gain(key) : 0;
                w.jb_agent[j] = key ? key_index(key) : -1;
            }
            gain = in_c ? w.jb_gain[j] : (key ? key_gain(key) : 0);
            target = in_c ? w.jb_agent[j] : (key ? key_index(key) : -1);
        }
        const uint32_t bm = __ballot_sync(0xffffffffu, gain > 0);
        if (gain > 0) {
            const int32_t u = (t < n) ? t : w.sigma[t - n];
            const int32_t v = (t < n) ? w.sigma[target] : target;
            const unsigned long long e =
                edge_word(u, v) | (exchange_gain(w, u, v) > 0 ? kApplies : 0ull) | (key ? kRevives : 0ull);
            w.sl_edge[t0 + __popc(bm & ((1u << lane) - 1u))] = e | ((unsigned long long)lane << kPlaceShift);
        }
        if (lane == 0) w.sl_chunk[t0 >> 5] = __popc(bm);
    }
}

__global__ void prepare_edges_kernel(Workspace w) { prepare_edges_body(w, blockIdx.x, gridDim.x); }

// Rows whose best is no longer known: rows of changed jobs, and rows whose
// best partner column changed holder.  Their keys are cleared and listed.
__device__ __forceinline__ void mark_rescan_body(const Workspace& w, int32_t bid, int32_t nblk) {
    DeviceState* st = w.st;
    if (st->status != kRunning || !st->need_update) return;
    for (int32_t j = bid * blockDim.x + threadIdx.x; j < w.n; j += nblk * blockDim.x) {
        bool need = w.in_y[j];
        const unsigned long long ka = w.key_a[j];
        const unsigned long long kj = w.key_j[j];
        if (!need && ka) need = w.in_y[key_index(ka)];
        if (!need && kj) need = w.moved[key_index(kj)];
        if (need) {
            w.key_a[j] = 0;
            w.key_j[j] = 0;
            w.rescan_list[atomicAdd(&st->rescan_count, 1)] = j;
        }
    }
}

__global__ void mark_rescan_kernel(Workspace w) { mark_rescan_body(w, blockIdx.x, gridDim.x); }

// Row j of G recomputed in full by the CTA from row sigma(j) of a (read
// directly) and row j of at (`atrow`: global memory, or its copy staged in
// shared memory), gathered through sigma; its two keys are raised to the row's
// best.  With `scatter` and j a changed job, the row also pushes G[k][j] =
// G[j][k] into every other row k (the only entries of row k that changed),
// through the same atomic keys.  red_a / red_j: 16 entries each.  Ends with
// a CTA barrier (red_* and the staged row may be reused).
__device__ __forceinline__ void row_task_compute(const Workspace& w, int32_t j, const int32_t* atrow, bool scatter_ok,
                                                 unsigned long long* red_a, unsigned long long* red_j) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t n = w.n;
    const int32_t n4 = (n + 3) / 4;
    const int32_t sjj = w.sigma[j];
    const int32_t dj = w.diag[j];
    const bool scatter = scatter_ok && w.in_y[j];
    const int32_t* arow = w.a + (size_t)sjj * w.lda;
    int32_t bg = 0, bc = -1, bs = 0x7fffffff;
#pragma unroll 2
    for (int32_t q = tid; q < n4; q += blockDim.x) {
        const int32_t k0 = 4 * q;
        const int4 x4 = *reinterpret_cast<const int4*>(arow + k0);
        const int4 s4 = *reinterpret_cast<const int4*>(w.sigma + k0);
        const int4 d4 = *reinterpret_cast<const int4*>(w.diag + k0);
        const int32_t xs[4] = {x4.x, x4.y, x4.z, x4.w};
        const int32_t ss[4] = {s4.x, s4.y, s4.z, s4.w};
        const int32_t ds[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int32_t k = k0 + e;
            if (k >= n) break;
            const int32_t sk = ss[e];
            const int32_t g = xs[e] + atrow[sk] - dj - ds[e];
            const bool gt = g > bg, eq = g == bg;
            bs = gt ? sk : (eq ? min(bs, sk) : bs);
            bc = gt ? k : bc;
            bg = max(bg, g);
            if (scatter && g > 0 && k != j && g >= key_gain(w.key_a[k])) {
                atomicMax(&w.key_a[k], pack_gain(g, (uint32_t)j));
                atomicMax(&w.key_j[k], pack_gain(g, (uint32_t)sjj));
            }
        }
    }
    unsigned long long ka = bg > 0 ? pack_gain(bg, (uint32_t)bc) : 0ull;
    unsigned long long kj = bg > 0 ? pack_gain(bg, (uint32_t)bs) : 0ull;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ka = umax64(ka, __shfl_xor_sync(0xffffffffu, ka, off));
        kj = umax64(kj, __shfl_xor_sync(0xffffffffu, kj, off));
    }
    if (lane == 0) { red_a[warp] = ka; red_j[warp] = kj; }
    __syncthreads();
    if (tid == 0) {
        unsigned long long ma = 0, mj = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { ma = umax64(ma, red_a[q]); mj = umax64(mj, red_j[q]); }
        if (ma) {
            atomicMax(&w.key_a[j], ma);
            atomicMax(&w.key_j[j], mj);
        }
    }
    __syncthreads();
}

// Full re-evaluation of one listed row (row tasks): row j of at staged in
// shared memory by one TMA bulk copy when kStage.  Returns false (CTA-uniform)
// if the staged copy did not arrive within the wait limit.
template <bool kStage>
__device__ __forceinline__ bool row_task_row(const Workspace& w, int32_t j, int32_t* atrow_s, uint64_t* bar,
                                             uint32_t& phase, unsigned long long* red_a,
                                             unsigned long long* red_j) {
    const int32_t* atrow = w.at + (size_t)j * w.ldt;
    if (kStage) {
        if (threadIdx.x == 0) {
            const uint32_t bytes = 16u * (uint32_t)((w.n + 3) / 4);
            mbar_arrive_expect_tx(bar, bytes);
            bulk_g2s(atrow_s, atrow, bytes, bar);
            // the row of a meanwhile into L2
            bulk_prefetch_l2(w.a + (size_t)w.sigma[j] * w.lda, bytes);
        }
        const bool ok = mbar_wait_bounded(bar, phase);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) mbar_wait_bounded(bar, phase);  // the copy may still land: wait once more
            return false;
        }
        phase ^= 1u;
        atrow = atrow_s;
    }
    row_task_compute(w, j, atrow, true, red_a, red_j);
    return true;
}

template <bool kStage>
__device__ __forceinline__ void row_tasks_body(const Workspace& w, int32_t bid, int32_t nblk) {
    DeviceState* st = w.st;
    if (st->status != kRunning || !st->need_update) return;
    const int32_t count = st->rescan_count;
    const int32_t n = w.n;
    if (use_full_update(count, n, st->update_policy)) return;
    if (bid == 0 && threadIdx.x == 0) {
        st->row_updates += 1;
        st->rows_recomputed += count;
    }
    extern __shared__ __align__(128) unsigned char smem_raw[];
    int32_t* atrow_s = reinterpret_cast<int32_t*>(smem_raw);
    __shared__ unsigned long long red_a[16], red_j[16];
    __shared__ __align__(8) uint64_t bar;
    if (kStage && threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    for (int32_t t = bid; t < count; t += nblk) {
        if (!row_task_row<kStage>(w, w.rescan_list[t], atrow_s, &bar, phase, red_a, red_j)) {
            if (threadIdx.x == 0) { st->error = kErrWaitTimeout; st->status = kError; }
            return;
        }
    }
}

template <bool kStage>
__global__ void __launch_bounds__(512) row_tasks_kernel(Workspace w) {
    row_tasks_body<kStage>(w, blockIdx.x, gridDim.x);
}

// Row j of G re-evaluated in full by one warp (the row task of the
// single-CTA switching loop and of batches): the same gains, tie-breaks and
// scatter into the other rows' keys as row_task_compute, four columns per lane
// and step (each lane sees its columns in ascending order, so its first
// maximum is its lowest column, and the packed keys combine across lanes).
__device__ __forceinline__ void row_task_warp(const Workspace& w, int32_t j) {
    const int lane = threadIdx.x & 31;
    const int32_t n = w.n;
    const int32_t sjj = w.sigma[j];
    const int32_t dj = w.diag[j];
    const bool scatter = w.in_y[j];
    const int32_t* arow = w.a + (size_t)sjj * w.lda;
    const int32_t* atrow = w.at + (size_t)j * w.ldt;
    int32_t bg = 0, bc = -1, bs = 0x7fffffff;
#pragma unroll 2
    for (int32_t k0 = lane * 4; k0 < n; k0 += 128) {
        const int4 x4 = *reinterpret_cast<const int4*>(arow + k0);
        const int4 s4 = *reinterpret_cast<const int4*>(w.sigma + k0);
        const int4 d4 = *reinterpret_cast<const int4*>(w.diag + k0);
        const int32_t xs[4] = {x4.x, x4.y, x4.z, x4.w};
        const int32_t ss[4] = {s4.x, s4.y, s4.z, s4.w};
        const int32_t ds[4] = {d4.x, d4.y, d4.z, d4.w};
        int32_t ys[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) ys[e] = k0 + e < n ? atrow[ss[e]] : 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int32_t k = k0 + e;
            if (k >= n) break;
            const int32_t g = xs[e] + ys[e] - dj - ds[e];
            const bool gt = g > bg, eq = g == bg;
            bs = gt ? ss[e] : (eq ? min(bs, ss[e]) : bs);
            bc = gt ? k : bc;
            bg = max(bg, g);
            if (scatter && g > 0 && k != j && g >= key_gain(w.key_a[k])) {
                atomicMax(&w.key_a[k], pack_gain(g, (uint32_t)j));
                atomicMax(&w.key_j[k], pack_gain(g, (uint32_t)sjj));
            }
        }
    }
    unsigned long long ka = bg > 0 ? pack_gain(bg, (uint32_t)bc) : 0ull;
    unsigned long long kj = bg > 0 ? pack_gain(bg, (uint32_t)bs) : 0ull;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ka = umax64(ka, __shfl_xor_sync(0xffffffffu, ka, off));
        kj = umax64(kj, __shfl_xor_sync(0xffffffffu, kj, off));
    }
    if (lane == 0 && ka) {
        atomicMax(&w.key_a[j], ka);
        atomicMax(&w.key_j[j], kj);
    }
}

// The whole switching loop of Algorithm 3 in one CTA, for small n (the
// per-launch cost of the five kernels of an iteration would dominate): per
// iteration the rows marked by the last committing sweep are re-evaluated
// (row tasks, one warp per row; identical keys to a full evaluation, see the
// update kernels), the slots refreshed, then the controller's sweeps; until
// the loop state stops running.  Bounded like the graph loop.
template <typename EdgeT, int kT>
__global__ void __launch_bounds__(kT, 1) small_loop_kernel(Workspace w, int32_t smem_mode, CtlScratch g,
                                                                   uint32_t span, uint32_t stamp_wrap,
                                                                   int32_t compact_min, int32_t colour_pass) {
    __shared__ int32_t s_go, s_count;
    static_assert(sizeof(s_go) + sizeof(s_count) == kSmallLoopShared, "");
    DeviceState* st = w.st;
    const int32_t n = w.n;
    const int tid = threadIdx.x, warp = tid >> 5;
    for (;;) {
        mark_rescan_body(w, 0, 1);
        __syncthreads();
        if (tid == 0) {
            const bool rows = st->status == kRunning && st->need_update;
            s_count = rows ? st->rescan_count : 0;
            if (rows) {
                st->row_updates += 1;
                st->rows_recomputed += s_count;
            }
        }
        __syncthreads();
        for (int32_t t = warp; t < s_count; t += kT / 32) row_task_warp(w, w.rescan_list[t]);
        __syncthreads();
        prepare_edges_body(w, 0, 1);
        __syncthreads();
        controller_body<EdgeT, kT>(w, smem_mode, g, span, stamp_wrap, compact_min, colour_pass);
        if (tid == 0) {
            const int32_t it = ++st->loop_iterations;
            if (st->status == kRunning && it > 16 * n + 4096) {
                st->error = kErrInternal;
                st->status = kError;
            }
            s_go = st->status == kRunning;
        }
        __syncthreads();
        if (!s_go) break;
    }
}

// The row-owner form of the full difference evaluation (Algorithm 2 for every
// slot, the A-transpose variant): CTA b owns rows j = b, b + nblk, ... of G and
// recomputes each from row sigma(j) of a and row j of the maintained at, with
// the next row of at already in flight to the second shared-memory stage
// (TMA bulk copies) while the current row is evaluated.  It touches 8n^2 bytes
// per evaluation (the tile-pair kernel reads each benefit once, 4n^2) but needs
// only one key update per row.  Keys are raised with atomicMax, so the result
// is the tile-pair kernel's: the same maxima with the same tie-breaks.
template <bool kStage>
__global__ void __launch_bounds__(512) row_owner_evaluation_kernel(Workspace w, int32_t conditional) {
    DeviceState* st = w.st;
    if (st->status != kRunning) return;
    if (conditional && !(st->need_update && use_full_update(st->rescan_count, w.n, st->update_policy))) return;
    if (conditional && blockIdx.x == 0 && threadIdx.x == 0) st->full_evals += 1;
    if (!conditional && blockIdx.x == 0 && threadIdx.x == 0 && st->sweeps == 0) st->f_initial = st->f;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ unsigned long long red_a[16], red_j[16];
    __shared__ __align__(8) uint64_t bar[2];
    const int32_t n = w.n;
    const uint32_t bytes = 16u * (uint32_t)((n + 3) / 4);
    int32_t* const stage0 = reinterpret_cast<int32_t*>(smem_raw);  // stage b at stage0 + b * ldt
    if (kStage && threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    int32_t j = blockIdx.x;
    if (kStage && threadIdx.x == 0 && j < n) {
        mbar_arrive_expect_tx(&bar[0], bytes);
        bulk_g2s(stage0, w.at + (size_t)j * w.ldt, bytes, &bar[0]);
    }
    uint32_t phase = 0;  // bit b: parity of stage b's next completion
    for (int32_t it = 0; j < n; ++it, j += gridDim.x) {
        const int b = it & 1;
        const int32_t* atrow = w.at + (size_t)j * w.ldt;
        if (kStage) {
            // the other stage was last read by the previous row, which ended
            // with a CTA barrier: it is free for the next row's copy
            const int32_t jn = j + (int32_t)gridDim.x;
            if (threadIdx.x == 0 && jn < n) {
                mbar_arrive_expect_tx(&bar[b ^ 1], bytes);
                bulk_g2s(stage0 + (b ^ 1) * w.ldt, w.at + (size_t)jn * w.ldt, bytes, &bar[b ^ 1]);
            }
            const uint32_t pb = (phase >> b) & 1u;
            const bool ok = mbar_wait_bounded(&bar[b], pb);
            phase ^= 1u << b;
            if (__syncthreads_or(!ok)) {
                if (threadIdx.x == 0) {
                    st->error = kErrWaitTimeout;
                    st->status = kError;
                    // this row's copy and the next one may still be in flight
                    // into this CTA's shared memory: wait for them (bounded)
                    // before leaving
                    mbar_wait_bounded(&bar[b], pb);
                    if (jn < n) mbar_wait_bounded(&bar[b ^ 1], (phase >> (b ^ 1)) & 1u);
                }
                return;
            }
            atrow = stage0 + b * w.ldt;
        }
        row_task_compute(w, j, atrow, false, red_a, red_j);
    }
}

// tau given (greedy result, identity or the caller's permutation): build
// sigma, D and f; validate a caller's permutation.
__device__ __forceinline__ void start_from_tau_body(const Workspace& w, const int32_t* user_tau, int32_t mode,
                                                    uint8_t* seen, int32_t bid, int32_t nblk) {
    DeviceState* st = w.st;
    // (uniform for the CTA: another CTA may report a bad start meanwhile)
    if (__syncthreads_or(st->status != kRunning)) return;
    long long f = 0;
    for (int32_t i = bid * blockDim.x + threadIdx.x; i < w.n; i += nblk * blockDim.x) {
        int32_t j;
        if (mode == 2) j = i;                 // identity
        else if (mode == 3) j = user_tau[i];  // caller's permutation
        else j = w.tau[i];                    // greedy result
        if (j < 0 || j >= w.n || atomicExch(reinterpret_cast<unsigned int*>(seen) + j, 1u) != 0u) {
            st->error = kErrUserInit;
            st->status = kError;
            continue;
        }
        w.tau[i] = j;
        w.sigma[j] = i;
        const int32_t d = w.a[(size_t)i * w.lda + j];
        w.diag[j] = d;
        f += d;
    }
    add_objective(st, f);
}

__global__ void start_from_tau_kernel(Workspace w, const int32_t* user_tau, int32_t mode, uint8_t* seen) {
    start_from_tau_body(w, user_tau, mode, seen, blockIdx.x, gridDim.x);
}

__global__ void finish_kernel(Workspace w, int32_t* sigma_out) {
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.n; i += gridDim.x * blockDim.x)
        sigma_out[i] = w.tau[i];
}

// The dgs_status code of a finished loop state (the device side of
// map_device_status).
__device__ __forceinline__ int32_t device_status_code(const DeviceState* st) {
    if (st->status == kTimeout) return DGS_TIMEOUT;
    if (st->status != kError) return DGS_OK;
    if (st->error == kErrRange) return DGS_ERR_RANGE;
    if (st->error == kErrUserInit) return DGS_ERR_INVALID;
    return DGS_ERR_INTERNAL;
}

// Outputs that the device can write (device memory, or pinned host memory)
// are written here: a copy of the loop state and a host callback that fills
// pageable ones cost 70 to 90 us at the end of a solve.
__global__ void finish_outputs_kernel(Workspace w, int32_t* sigma_out, int64_t* objective, int32_t* status,
                                      dgs_stats* stats, int64_t launches, int32_t sequential) {
    const DeviceState* st = w.st;
    const bool failed = st->status == kError;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.n; i += gridDim.x * blockDim.x)
        sigma_out[i] = failed ? -1 : w.tau[i];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (objective) *objective = st->f;
        if (status) *status = device_status_code(st);
        if (stats) {
            dgs_stats s{};
            s.sweeps = st->sweeps;
            s.events = st->events;
            s.swaps_applied = st->swaps;
            s.greedy_rounds = st->greedy_rounds;
            s.full_evaluations = sequential ? 0 : st->full_evals + 1;
            s.row_updates = sequential ? 0 : st->row_updates;
            s.rows_recomputed = sequential ? 0 : st->rows_recomputed;
            s.initial_objective = st->f_initial;
            s.kernel_launches = launches + st->loop_launches;
            s.greedy_rescans = st->greedy_rescans;
            s.status = device_status_code(st);
            *stats = s;
        }
    }
}

// ------------------------------------------------------- batched launches
// Initialise the fresh instances of the table: clear their small arrays and
// write the loop state (stage kStageNew).  Entries walk 16-byte chunks.
__global__ void init_batched_kernel(BatchTable t, int32_t update_policy) {
    const int32_t count = *t.count;
    for (int32_t g = blockIdx.x; g < count; g += gridDim.x) {
        const BatchEntry e = t.e[g];
        const Instance& in = t.inst[e.inst];
        if (!in.fresh) continue;
        const Workspace& w = in.w;
        const size_t chunks = in.zero_bytes / 16;
        const size_t stride = (size_t)e.nblk * blockDim.x;
        for (size_t q = (size_t)e.bid * blockDim.x + threadIdx.x; q < chunks; q += stride)
            *reinterpret_cast<uint4*>(in.zero_begin + 16 * q) = make_uint4(0u, 0u, 0u, 0u);
        // (a caller's matrix that needs re-pitching, n % 4 != 0 or misaligned, is
        // copied into the workspace by pass 1, which reads it anyway)
        if (e.bid == 0 && threadIdx.x == 0) {
            DeviceState h{};
            h.status = kRunning;
            h.phase = kPhaseRefreshAll;
            h.max_sweeps = in.max_sweeps;
            h.greedy_remaining = w.n;
            h.update_policy = update_policy;
            h.stage = kStageNew;
            h.init_mode = in.init_mode;
            h.reeval_all = in.reeval_all;
            if (in.deadline_us > 0) h.deadline_ns = globaltimer_ns() + (uint64_t)in.deadline_us * 1000ull;
            *w.st = h;
        }
    }
}

__global__ void start_batched_kernel(BatchTable t) {
    for_each_entry(t, kStageStart, [&](const Instance& in, int32_t bid, int32_t nblk) {
        start_from_tau_body(in.w, in.user_tau, in.w.st->init_mode, in.seen, bid, nblk);
    });
}

__global__ void mark_rescan_batched_kernel(BatchTable t) {
    for_each_entry(t, kStageSwitch, [&](const Instance& in, int32_t bid, int32_t nblk) {
        mark_rescan_body(in.w, bid, nblk);
    });
}

// The rows queued by the kScanSwitch scan (q1: their weights), every CTA an
// equal share of the weight; a row by the whole CTA, the at row staged by TMA;
// one mbarrier for the CTA's whole sequence of rows.  What bounds a row is
// latency (staging, loads, reduction: 4 to 5 microseconds), and below that the
// 8 n bytes, so CTAs are small and many per SM where their rows are short
// (launch_b_row_tasks).  The gather through sigma has to come from shared
// memory: from L1 it takes a cycle per column (1024 peer-shaped instances, n in
// [64, 4096], 562k rows: 4.1 ms with a warp per row, 3.7 now; 8.2 ms with
// 512 threads per row and equal numbers of rows per CTA).
template <int kT>
__global__ void __launch_bounds__(kT) row_tasks_batched_kernel(BatchQueues q) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    int32_t* atrow_s = reinterpret_cast<int32_t*>(smem_raw);
    __shared__ unsigned long long red_a[16], red_j[16];
    __shared__ __align__(8) uint64_t bar;
    __shared__ Workspace w;
    if (q.q1[q.cap] <= 0) return;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    bool dead = false;
    for_each_range(q.inst, q.q1, q.cap, blockIdx.x, gridDim.x, [&](const Instance& in, int32_t lo, int32_t hi) {
        if (dead) return;
        __syncthreads();  // the copy is no longer read
        if (threadIdx.x == 0) w = in.w;
        __syncthreads();
        const int32_t weight = row_weight(w.n, q.cap);  // the rows that begin in [lo, hi)
        for (int32_t r = (lo + weight - 1) / weight; r * weight < hi; ++r) {
            if (!row_task_row<true>(w, w.rescan_list[r], atrow_s, &bar, phase, red_a, red_j)) {
                if (threadIdx.x == 0) { w.st->error = kErrWaitTimeout; w.st->status = kError; }
                dead = true;  // the buffer may still be written: no further copies into it
                return;
            }
        }
    });
}

// Per-slot work counts of one phase as exclusive prefix offsets (q0, q1; cap
// + 1 entries each), with the counters a single solve updates at the same
// point.  One CTA of 1024 threads.
//   kScanPass1:  q0 = pass-1 blocks of instances in kStageNew
//   kScanGreedyDA: q0 = agents of the instances in kStageGreedy (every q1
//                entry is 0: q1[0] is the deferred acceptance's shared counter)
//   kScanStart:  q0 = evaluation tiles of instances in kStageStart
//   kScanSwitch: q0 = evaluation tiles of the updates that re-evaluate every
//                row, q1 = weight of the rows of the updates that use row tasks
__global__ void __launch_bounds__(1024) scan_batched_kernel(BatchQueues q, int32_t phase) {
    __shared__ int32_t warp_sums[33];
    int32_t carry0 = 0, carry1 = 0;
    for (int32_t c0 = 0; c0 < q.cap; c0 += 1024) {
        const int32_t k = c0 + (int32_t)threadIdx.x;
        int32_t x0 = 0, x1 = 0;
        if (k < q.cap) {
            const Instance& in = q.inst[k];
            DeviceState* st = in.w.st;
            const int32_t n = in.w.n;
            if (st != nullptr && n > 0) {
                const int32_t stage = st->stage;
                const bool running = st->status == kRunning;
                if (phase == kScanPass1) {
                    if (stage == kStageNew) x0 = batch_blocks_pass1(n);
                } else if (phase == kScanGreedyDA) {
                    if (stage == kStageGreedy && running && st->greedy_remaining > 0) x0 = n;
                } else if (phase == kScanStart) {
                    if (stage == kStageStart && running) x0 = eval_tiles(n);
                } else if (phase == kScanSwitch) {
                    if (stage == kStageSwitch && running && st->need_update) {
                        const int32_t count = st->rescan_count;
                        if (use_full_update(count, n, st->update_policy)) {
                            x0 = eval_tiles(n);
                            st->full_evals += 1;
                        } else {
                            x1 = count * row_weight(n, q.cap);
                            st->row_updates += 1;
                            st->rows_recomputed += count;
                        }
                    }
                }
            }
        }
        int32_t t0, t1;
        const int32_t p0 = block_scan(x0, warp_sums, &t0);
        const int32_t p1 = block_scan(x1, warp_sums, &t1);
        if (k < q.cap) {
            q.q0[k] = carry0 + p0;
            q.q1[k] = carry1 + p1;
        }
        carry0 += t0;
        carry1 += t1;
    }
    if (threadIdx.x == 0) {
        q.q0[q.cap] = carry0;
        q.q1[q.cap] = carry1;
    }
}

__global__ void prepare_edges_batched_kernel(BatchTable t) {
    for_each_entry(t, kStageSwitch, [&](const Instance& in, int32_t bid, int32_t nblk) {
        prepare_edges_body(in.w, bid, nblk);
    });
}

__global__ void __launch_bounds__(kCtlThreads, 1) controller_batched_kernel(BatchTable t, uint32_t span,
                                                                           uint32_t stamp_wrap, int32_t compact_min,
                                                                           int32_t colour_pass) {
    for_each_entry(t, kStageSwitch, [&](const Instance& in, int32_t, int32_t) {
        const CtlScratch c{in.ctl.res, in.ctl.claimed, in.ctl.estate, in.ctl.edges, in.ctl.acc};
        controller_body<uint32_t>(in.w, in.ctl_mode, c, span, stamp_wrap, compact_min, colour_pass);
    });
}

// The switching loop of an instance has ended: write its assignment.
__global__ void finish_batched_kernel(BatchTable t) {
    for_each_entry(t, kStageSwitch, [&](const Instance& in, int32_t bid, int32_t nblk) {
        const DeviceState* st = in.w.st;
        if (st->status != kDone && st->status != kTimeout) return;
        for (int32_t i = bid * blockDim.x + threadIdx.x; i < in.w.n; i += nblk * blockDim.x)
            in.sigma_out[i] = in.w.tau[i];
    });
}

// Stage transitions of the instances in from_stage (one thread each).
__global__ void advance_batched_kernel(BatchTable t, int32_t from_stage) {
    const int32_t count = *t.count;
    for (int32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < count; g += gridDim.x * blockDim.x) {
        const Instance& in = t.inst[t.e[g].inst];
        DeviceState* st = in.w.st;
        if (st->stage != from_stage) continue;
        const bool running = st->status == kRunning;
        int32_t next = from_stage;
        if (from_stage == kStageNew) {
            next = !running ? kStageDone : (st->init_mode == 0 ? kStageGreedy : kStageStart);
        } else if (from_stage == kStageGreedy) {
            next = !running ? kStageDone : (st->greedy_remaining == 0 ? kStageStart : kStageGreedy);
        } else if (from_stage == kStageStart) {
            st->f_initial = st->f;
            next = running ? kStageSwitch : kStageDone;
        } else if (from_stage == kStageSwitch) {
            next = running ? kStageSwitch : kStageDone;
        }
        st->stage = next;
    }
}

}  // namespace

int32_t controller_smem_mode(int32_t n) {
    int32_t mode = 0;
    if (n <= 32767 && controller_layout(n, 2).bytes <= kCtlSmemLimit) mode = 2;
    else if (n <= 32767 && controller_layout(n, 1).bytes <= kCtlSmemLimit) mode = 1;
    return min(mode, env_controller_mode_cap());
}

size_t controller_smem_bytes(int32_t n) {
    const int32_t mode = controller_smem_mode(n);
    return mode == 0 ? 0 : controller_layout(n, mode).bytes;
}

// DGS_SMALL_LOOP_N: the largest n whose switching loop runs in one CTA
// (small_loop_kernel); 0 turns it off (read on every call).  Only with the
// default update policy (the test knob that forces an update path keeps the
// grid kernels).
int32_t small_loop_max_n() {
    const char* e = std::getenv("DGS_SMALL_LOOP_N");
    return e ? std::atoi(e) : 768;  // measured: faster up to n = 512, slower from n = 1024
}

bool use_small_loop(const Workspace& w) {
    return w.n <= small_loop_max_n() && controller_smem_mode(w.n) == 2 && env_update_policy() == 0 &&
           w.row_owner_eval == 0;
}

template <int kT>
static cudaError_t launch_small_loop_t(const Workspace& w, const CtlGlobal& gs, cudaStream_t s) {
    const int32_t mode = controller_smem_mode(w.n);
    const size_t smem = controller_smem_bytes(w.n);
    CtlScratch c{gs.res, gs.claimed, gs.estate, gs.edges, gs.acc};
    if (smem + kCtlStaticSmem > 48 * 1024) {
        cudaError_t e = ensure_smem_limit<small_loop_kernel<uint32_t, kT>>(smem);
        if (e != cudaSuccess) return e;
    }
    const bool short_wrap = env_short_wraps() != 0;
    small_loop_kernel<uint32_t, kT><<<1, kT, smem, s>>>(w, mode, c, short_wrap ? 4u : kRoundSpanMax,
                                                         short_wrap ? 5u : 250u, env_compact_min(),
                                                         env_colour_pass());
    return cudaGetLastError();
}

// DGS_SMALL_LOOP_THREADS (256, 512 or 1024; read on every launch): the CTA
// width of the single-CTA loop.  Measured at n = 256 (uniform [0, 1000), 52
// sweeps): 0.32 / 0.29 / 0.30 ms; peer-shaped: 0.150 / 0.144 / 0.143 ms.
int32_t small_loop_threads() {
    const char* e = std::getenv("DGS_SMALL_LOOP_THREADS");
    const int32_t x = e ? std::atoi(e) : 512;
    return (x == 256 || x == 1024) ? x : 512;
}

cudaError_t launch_small_loop(const Workspace& w, const CtlGlobal& gs, cudaStream_t s) {
    switch (small_loop_threads()) {
        case 1024: return launch_small_loop_t<1024>(w, gs, s);
        case 512: return launch_small_loop_t<512>(w, gs, s);
        default: return launch_small_loop_t<256>(w, gs, s);
    }
}

cudaError_t launch_controller_impl(const Workspace& w, const CtlGlobal& gs, cudaStream_t s, bool counted,
                                   unsigned long long handle) {
    const int32_t mode = controller_smem_mode(w.n);
    const size_t smem = controller_smem_bytes(w.n);
    CtlScratch c{gs.res, gs.claimed, gs.estate, gs.edges, gs.acc};
    const bool narrow = w.n <= 65535;
    if (smem + kCtlStaticSmem > 48 * 1024) {
        cudaError_t e = narrow ? ensure_smem_limit<controller_kernel<uint32_t>>(smem)
                               : ensure_smem_limit<controller_kernel<unsigned long long>>(smem);
        if (e != cudaSuccess) return e;
    }
    const bool short_wrap = env_short_wraps() != 0;
    const uint32_t span = short_wrap ? 4u : kRoundSpanMax;
    const uint32_t stamp_wrap = short_wrap ? 5u : 250u;
    const int32_t cmin = env_compact_min();
    const int32_t cp = env_colour_pass();
    if (narrow)
        controller_kernel<uint32_t><<<1, kCtlThreads, smem, s>>>(w, mode, c, span, stamp_wrap, cmin, cp, counted, handle);
    else
        controller_kernel<unsigned long long><<<1, kCtlThreads, smem, s>>>(w, mode, c, span, stamp_wrap, cmin, cp,
                                                                          counted, handle);
    return cudaGetLastError();
}

cudaError_t launch_prepare_edges(const Workspace& w, cudaStream_t s) {
    int grid = (2 * w.n + 255) / 256;
    if (grid > dgs::device_sms() * 8) grid = dgs::device_sms() * 8;
    prepare_edges_kernel<<<grid, 256, 0, s>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_mark_rescan(const Workspace& w, cudaStream_t s) {
    int grid = (w.n + 255) / 256;
    if (grid > dgs::device_sms() * 4) grid = dgs::device_sms() * 4;
    mark_rescan_kernel<<<grid, 256, 0, s>>>(w);
    return cudaGetLastError();
}

constexpr int32_t kRowStageMaxN = 54 * 1024;

cudaError_t launch_row_tasks(const Workspace& w, cudaStream_t s) {
    int grid = dgs::device_sms() * 2;
    if (w.n <= kRowStageMaxN) {
        const size_t smem = 4 * (size_t)w.ldt;
        // as many CTAs as fit (four of 512 threads per SM): the few hundred
        // rows of an update then go in one wave
        const int fit = (int)((227 * 1024) / (smem + 2048));
        grid = dgs::device_sms() * (fit > 4 ? 4 : fit < 1 ? 1 : fit);
        // (at every size: what a kernel has without, 48 KB, includes its static part)
        cudaError_t e = ensure_smem_limit<row_tasks_kernel<true>>(smem);
        if (e != cudaSuccess) return e;
        row_tasks_kernel<true><<<grid, 512, smem, s>>>(w);
    } else {
        row_tasks_kernel<false><<<grid, 512, 0, s>>>(w);
    }
    return cudaGetLastError();
}

// Two stages of one row of at each: up to 27 * 1024 columns (216 KB).
constexpr int32_t kRowOwnerStageMaxN = 27 * 1024;

cudaError_t launch_row_owner_evaluation(const Workspace& w, int32_t conditional, cudaStream_t s) {
    if (w.n <= kRowOwnerStageMaxN) {
        const size_t smem = 2 * 4 * (size_t)w.ldt;
        cudaError_t e = ensure_smem_limit<row_owner_evaluation_kernel<true>>(smem);
        if (e != cudaSuccess) return e;
        const int per_sm = smem <= 110 * 1024 ? 2 : 1;
        row_owner_evaluation_kernel<true><<<dgs::device_sms() * per_sm, 512, smem, s>>>(w, conditional);
    } else {
        row_owner_evaluation_kernel<false><<<dgs::device_sms() * 2, 512, 0, s>>>(w, conditional);
    }
    return cudaGetLastError();
}

cudaError_t launch_start_from_tau(const Workspace& w, const int32_t* user_tau, int32_t mode, uint8_t* seen,
                                  cudaStream_t s) {
    int grid = (w.n + 255) / 256;
    if (grid > dgs::device_sms() * 4) grid = dgs::device_sms() * 4;
    start_from_tau_kernel<<<grid, 256, 0, s>>>(w, user_tau, mode, seen);
    return cudaGetLastError();
}

// ---------------------------------------------------- batched launchers
// rows: entries over the agents/slots of each instance (256 threads per
// block); one: one entry per instance.

cudaError_t launch_b_init(const BatchTable& rows, cudaStream_t s) {
    init_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(rows, env_update_policy());
    return cudaGetLastError();
}

cudaError_t launch_b_start(const BatchTable& rows, cudaStream_t s) {
    start_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(rows);
    return cudaGetLastError();
}

cudaError_t launch_b_mark_rescan(const BatchTable& rows, cudaStream_t s) {
    mark_rescan_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(rows);
    return cudaGetLastError();
}

// max_n: no queued instance is larger.  128 threads per row up to n = 4096 (a
// row is then at most 16 KB, 13 CTAs per SM), else 512.
template <int kT>
static cudaError_t launch_b_row_tasks_t(const BatchQueues& q, size_t smem, cudaStream_t s) {
    cudaError_t e = ensure_smem_limit<row_tasks_batched_kernel<kT>>(smem);
    if (e != cudaSuccess) return e;
    const int by_smem = (int)((227 * 1024) / (smem + 2048)), by_threads = 2048 / kT;
    const int per_sm = std::max(1, std::min({by_smem, by_threads, 13}));
    row_tasks_batched_kernel<kT><<<dgs::device_sms() * per_sm, kT, smem, s>>>(q);
    return cudaGetLastError();
}

cudaError_t launch_b_row_tasks(const BatchQueues& q, int32_t max_n, cudaStream_t s) {
    const size_t smem = 4 * (size_t)((max_n + 63) / 64 * 64);
    return max_n <= 4096 ? launch_b_row_tasks_t<128>(q, smem, s) : launch_b_row_tasks_t<512>(q, smem, s);
}

cudaError_t launch_b_scan(const BatchQueues& q, int32_t phase, cudaStream_t s) {
    scan_batched_kernel<<<1, 1024, 0, s>>>(q, phase);
    return cudaGetLastError();
}

cudaError_t launch_b_prepare_edges(const BatchTable& rows, cudaStream_t s) {
    prepare_edges_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(rows);
    return cudaGetLastError();
}

// Instances of a batched launch have n <= 32767 (16-bit edge positions and
// 32-bit edge words); each CTA lays out its shared memory for its own n.
cudaError_t launch_b_controller(const BatchTable& one, cudaStream_t s) {
    const size_t smem = kCtlSmemLimit;
    cudaError_t e = ensure_smem_limit<controller_batched_kernel>(smem);
    if (e != cudaSuccess) return e;
    const bool short_wrap = env_short_wraps() != 0;
    controller_batched_kernel<<<dgs::device_sms(), kCtlThreads, smem, s>>>(one, short_wrap ? 4u : kRoundSpanMax,
                                                            short_wrap ? 5u : 250u, env_compact_min(),
                                                            env_colour_pass());
    return cudaGetLastError();
}

cudaError_t launch_b_finish(const BatchTable& rows, cudaStream_t s) {
    finish_batched_kernel<<<dgs::device_sms() * 8, 256, 0, s>>>(rows);
    return cudaGetLastError();
}

cudaError_t launch_b_advance(const BatchTable& one, int32_t from_stage, cudaStream_t s) {
    advance_batched_kernel<<<8, 256, 0, s>>>(one, from_stage);
    return cudaGetLastError();
}

cudaError_t launch_finish_outputs(const Workspace& w, int32_t* sigma_out, int64_t* objective, int32_t* status,
                                  dgs_stats* stats, int64_t launches, int32_t sequential, cudaStream_t s) {
    int grid = (w.n + 255) / 256;
    if (grid > dgs::device_sms() * 4) grid = dgs::device_sms() * 4;
    finish_outputs_kernel<<<grid, 256, 0, s>>>(w, sigma_out, objective, status, stats, launches, sequential);
    return cudaGetLastError();
}

cudaError_t launch_finish(const Workspace& w, int32_t* sigma_out, cudaStream_t s) {
    int grid = (w.n + 255) / 256;
    if (grid > dgs::device_sms() * 4) grid = dgs::device_sms() * 4;
    finish_kernel<<<grid, 256, 0, s>>>(w, sigma_out);
    return cudaGetLastError();
}

}  // namespace dgs
