// map_run.cuh -- a whole MAP run (Section 2 of the paper) in one persistent cooperative launch.
//
// k_run runs every outer iteration of a run whose iterations start from the accepting vertices
// (the frontier start): round 1 pushes u + 1 from each accepting vertex u to its readers, round
// r + 1 pushes from the vertices changed in round r, until a round changes nothing; then the
// self-map test and the elimination, and the next iteration.  One grid barrier per round, one per
// self-map test; no launch and no host step in between.
//
// Per-vertex state W, all zero between iterations:
//   asynchronous  one word (value << 32 | ~round): an atomicMax with a larger value wins, and the
//                 old word tells in the same round trip whether the vertex rose, whether it had
//                 risen in this round already (then it is listed) and whether it had no value.
//                 On equal values the older round has the larger low half and stays.
//   synchronous   two words, written in even and odd rounds, (round << 33 | rose << 32 | value):
//                 the words of the other parity are frozen during a round, so every value read is
//                 the one of the round before (the exact Jacobi step).  The first push of a round to
//                 a vertex puts the round's stamp on its word, whether the value rose or not, so
//                 one atomicMax also finds the rows of the frontier (their lengths are the
//                 canonical relaxation count) and the vertices to list, each exactly once.
// So a push costs one random sector (asynchronous: one atomic; synchronous: a 16-byte load and, if
// it can change anything, one atomic on the same sector), and nothing is cleared between rounds.
//
// Compaction.  A vertex that has a value in outer iteration k + 1 had one in iteration k (the
// accepting set only shrinks), and every reader of such a vertex, or of a vertex still accepting, had
// one too.  So after an iteration in which few vertices had a value, the run goes on in the
// graph those vertices and the accepting ones induce, renumbered: the readers with their new
// numbers, and per vertex one 16-byte record (reader range, own offer, original id).  Random
// accesses over the full arrays are bound by address translation (measured: 42 G/s over 2 GB against
// 128 G atomics/s and 300 G loads/s over a packed array), and the compact arrays stay in L2.
//
// Floods.  When a list holds a large share of the whole graph's vertices (one value sweeping a giant
// component), its random accesses cost more than reading everything in order: from there on the iteration
// runs in scan mode (Run::scan_round), with 4-byte state arrays, pushes that nothing waits for and all vertices
// read in order every round, in pieces that go round the blocks.  Asynchronous, a vertex's value is read again when it
// is pushed (acyclic graphs of 4 M vertices, degree 4 / 8 / 16, ms for six iterations, without 17.6 / 29.5 / 47.2, with 11.7 /
// 18.7 / 28.0; dense start 16.7 / 18.4 / 22.1: from degree 10 or so such floods would be better off with that, but others of
// the same size and degree are not -- random 1.3 against 2.5 ms, layered 1.9 against 7.4).
//
// What it measured, ms per run (dense start in a CUDA graph -> here, k_own and k_tail included): layered 2^26
// asynchronous 16.7 -> 2.5, 2^24 synchronous 7.9 -> 1.7, 10^6 asynchronous 3.0 -> 0.81, a random graph of 16,384
// vertices synchronous 0.52 -> 0.16.
#pragma once
#include "map_kernels.cuh"

namespace mapk {

constexpr int RT = 512; // threads per block
#ifndef MAPGPU_RUN_BLOCKS
#define MAPGPU_RUN_BLOCKS 2 // resident blocks per SM the register budget is sized for
#endif
#ifndef MAPGPU_RUN_P
#define MAPGPU_RUN_P 1 // pushes per thread and step, all in flight together
#endif
constexpr int RUN_P = MAPGPU_RUN_P;
// a list of at least 1/16 of the whole graph (and RUN_SCAN_MIN entries) goes to scan mode, and back to lists below
// 1/64.  Layered graphs with a planted cycle, ms per synchronous / asynchronous run, lists only -> with scans:
// 2 M vertices 1.22 / 0.71 -> 0.57 / 0.41, 5 M 10.0 / 3.2 -> 3.2 / 1.6, 64-graph batch 6.4 / 5.1 -> 5.6 / 5.3 (shares
// 32 and 128: 5 M 3.2 / 2.4; 8 and 32: 14 M async 3.2 instead of 2.85)
constexpr uint32_t RUN_SCAN_SHARE = 16, RUN_LIST_SHARE = 64;
constexpr uint32_t RUN_SCAN_MIN = 8192;
constexpr uint32_t RUN_CAP = 8 * RT; // entries a block stages per round and list
constexpr uint32_t RUN_HIST = 512;  // outer iterations whose rounds come back with the result

struct alignas(128) Line64 {
    unsigned long long v;
};

// what a run reports; written at its end by one thread into page-locked host memory (or the device copy)
struct RunRes {
    uint32_t verdict, witness, outer, status;
    uint32_t nacc, gave_up;
    unsigned long long inner_total, relax, frontier_rows, ph_rounds, ph_check;
    uint32_t hist[RUN_HIST];
};

// zeroed before every run
struct RunCtl {
    Line64 bar[3];    // grid barriers by sequence number mod 3: arrivals << 48 | summed payload
    Cnt32 lcnt[3];    // |list| by the run's round number mod 3
    Cnt32 tcnt[2];    // |touched| by outer iteration mod 2
    Cnt32 acnt;       // accepting vertices listed
    Cnt32 xcnt, ecnt; // compaction: accepting vertices without a value, reader entries
    Cnt32 witness;    // NONE - the smallest self-mapped vertex (0: none)
    Line64 relax, frows;
    uint32_t gave_up;
    Line64 obar[3];   // k_own's grid barriers
    Cnt32 ocnt[2];    // k_own: vertices with a value, by outer iteration mod 2
    // what k_run leaves to k_own (hand = 1), and either to k_tail (2): the compact graph and where the run stands
    uint32_t hand, next, V, set, outer, nacc;
    unsigned long long inner_total, ph_rounds, ph_check, t0;
};

struct RunArgs {
    uint32_t n, words;
    const uint32_t *rowptr, *rrowptr, *rcol, *acc0;
    uint32_t *acc;
    unsigned long long *W;       // 2n words, zero
    uint32_t *la, *lb, *alist;   // n entries each: two lists, the accepting vertices
    uint32_t *touched, *tval;    // n entries each: vertices with a value in this iteration, and that value
    uint32_t *rank;              // n entries: original id -> 1 + number in the compact graph
    uint32_t *pool;              // 3n words: two sets of compact arrays
    RunCtl *ctl;
    RunRes *res;
    uint32_t *hist;              // rounds of every outer iteration (hist_cap entries)
    uint32_t hist_cap;
    uint32_t *out;               // map vector (MAP_NONE encoding), n entries; NULL: not wanted
    uint64_t m;
    uint32_t nacc0, max_outer, max_inner, lc_passes;
    uint32_t count_round1;       // asynchronous relaxations: the pushes of round 1 (else m per iteration)
    uint64_t timeout_ns;
    const uint32_t *prep;        // not NULL: (error, accepting vertices, entries) that k_prepare found
    uint32_t tail_cap, own_cap;  // compact graphs of at most this many vertices are left to k_tail / k_own (0: none)
    uint32_t tail_m;             // ... and of at most this many entries to k_tail where k_own could go on
    // batched runs
    const uint32_t *comp;
    CompState *cs;
    uint32_t *chist;
    uint32_t ncomp;
};

struct RunSmem {
    uint32_t o[RT], b[RT], incl[RT], scan[RT / 32];
    uint32_t list[RUN_CAP], touch[RUN_CAP];
    uint32_t ln, tn, lbase, tbase;
    unsigned long long word;
    uint32_t ok, ebase;
    unsigned long long part[RT / 32];
};

__device__ __forceinline__ uint32_t run_block_scan(uint32_t x, uint32_t *s)
{
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    x = warp_inclusive_scan(x);
    if (lane == 31) s[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t t = lane < RT / 32 ? s[lane] : 0;
#pragma unroll
        for (int off = 1; off < RT / 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, t, off);
            if (lane >= (unsigned)off) t += y;
        }
        if (lane < RT / 32) s[lane] = t;
    }
    __syncthreads();
    return warp ? x + s[warp - 1] : x;
}

// payload of a barrier: a count (bits 0-31), blocks that found a self-mapped vertex (32-46), a stop request (47)
constexpr unsigned long long RUN_STOP = 1ull << 47, RUN_FOUND = 1ull << 32, RUN_COUNT = RUN_FOUND - 1;

// Bounded grid-wide barrier; every block adds `payload` (thread 0's) and *total gets the sum, so the
// counts the next step needs come with the release instead of by another read.  One release
// reduction to arrive, acquire loads to wait: 1.3 us with 304 blocks, against 2.6 us for a returning
// atomic, a reset and a generation word with 912.  Returns false if the wait gave up.
template <class Smem>
__device__ __forceinline__ bool run_barrier(RunCtl *c, Line64 *bar, Smem &sh, uint32_t &seq, unsigned long long payload,
                                            unsigned long long &total)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t slot = seq % 3;
        // (the next barrier's word was last read before the barrier before this one)
        if (blockIdx.x == 0) *(volatile unsigned long long *)&bar[(seq + 1) % 3].v = 0;
        unsigned long long *w = &bar[slot].v, x = 0;
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(w), "l"((1ull << 48) | payload) : "memory");
        uint32_t ok = 1;
        for (uint32_t it = 0;; ++it) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(w) : "memory");
            if ((x >> 48) == gridDim.x) break;
            if (it > BAR_SPIN_LIMIT) {
                ok = 0;
                *(volatile uint32_t *)&c->gave_up = 1;
                break;
            }
        }
        sh.word = x & ((1ull << 48) - 1);
        sh.ok = ok;
    }
    __syncthreads();
    total = sh.word;
    ++seq;
    return sh.ok != 0;
}

// append w (where flag) to the staged list s_buf (count *s_cnt); what does not fit goes to g directly
__device__ __forceinline__ void stage_emit(bool flag, uint32_t w, uint32_t *s_buf, uint32_t *s_cnt, uint32_t *g, uint32_t *gcnt)
{
    const unsigned mask = __ballot_sync(0xFFFFFFFFu, flag);
    if (!mask) return;
    const unsigned lane = lane_id(), leader = __ffs(mask) - 1;
    uint32_t pos = 0;
    if (lane == leader) pos = atomicAdd(s_cnt, (uint32_t)__popc(mask));
    pos = __shfl_sync(0xFFFFFFFFu, pos, leader) + __popc(mask & ((1u << lane) - 1u));
    const bool over = flag && pos >= RUN_CAP;
    if (flag && !over) s_buf[pos] = w;
    if (__any_sync(0xFFFFFFFFu, over)) {
        const unsigned om = __ballot_sync(0xFFFFFFFFu, over);
        uint32_t at = 0;
        const unsigned ol = __ffs(om) - 1;
        if (lane == ol) at = atomicAdd(gcnt, (uint32_t)__popc(om));
        at = __shfl_sync(0xFFFFFFFFu, at, ol) + __popc(om & ((1u << lane) - 1u));
        if (over) g[at] = w;
    }
}

// entries [beg, end) in chunks of RT per block: get(i, o, b, len) gives an entry's offer and reader
// range, begin(total) runs once per chunk, and the (offer, reader position) pairs are spread
// evenly over the block's threads, RUN_P per thread and step: act(live, o, pos) for RUN_P pairs
template <class Get, class Begin, class Act>
__device__ __forceinline__ void expand(RunSmem &sh, uint64_t beg, uint64_t end, Get get, Begin begin, Act act)
{
    for (uint64_t c0 = beg; c0 < end; c0 += RT) {
        const uint64_t i = c0 + threadIdx.x;
        uint32_t o = 0, b = 0, len = 0;
        if (i < end) get(i, o, b, len);
        const uint32_t incl = run_block_scan(len, sh.scan);
        sh.o[threadIdx.x] = o;
        sh.b[threadIdx.x] = b - (incl - len); // reader position of pair p: b[owner] + p (32-bit wrap intended)
        sh.incl[threadIdx.x] = incl;
        __syncthreads();
        const uint32_t total = sh.incl[RT - 1];
        begin(i < end, i, incl - len, len, total);
        for (uint64_t p0 = 0; p0 < total; p0 += RT * RUN_P) {
            bool live[RUN_P];
            uint32_t off[RUN_P], pos[RUN_P], pair[RUN_P];
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) {
                const uint64_t p = p0 + j * RT + threadIdx.x;
                live[j] = p < total;
                off[j] = pos[j] = 0;
                pair[j] = (uint32_t)p;
                if (live[j]) {
                    uint32_t lo = 0, hi = RT - 1; // the owner: first entry with incl > p
#pragma unroll
                    for (int st = 1; st < RT; st *= 2) {
                        const uint32_t mid = (lo + hi) >> 1;
                        if (sh.incl[mid] > (uint32_t)p) hi = mid;
                        else lo = min(mid + 1, hi);
                    }
                    off[j] = sh.o[lo];
                    pos[j] = sh.b[lo] + (uint32_t)p;
                }
            }
            act(live, off, pos, pair);
        }
        __syncthreads(); // before the shared arrays are refilled
    }
}

// the space a run works in: the whole graph, or the compact graph of a later iteration
struct Space {
    uint32_t V, na;          // vertices, accepting vertices listed
    const uint4 *meta;       // compact: (first reader, end, own offer, original id); NULL: the whole graph
    const uint32_t *rc;      // readers
    const uint32_t *row;     // compact: row lengths (NULL: from rowptr)
    const uint32_t *comp;    // batched: graph of each vertex
};

// compact arrays, set h (0 or 1) in the pool of 3n words
__device__ __forceinline__ uint32_t pool_cap(uint32_t n) { return (n / 8) & ~3u; }
__device__ __forceinline__ uint32_t *pool_set(const RunArgs &a, uint32_t h) { return a.pool + (uint64_t)h * ((a.n + a.n / 2) & ~3u); }

template <bool SYNC, bool BATCH> struct Run {
    static constexpr uint32_t S = (SYNC || BATCH) ? 2 : 1; // state words per vertex

    const RunArgs &a;
    RunSmem &sh;
    Space sp;
    uint32_t seq = 0, lseq = 0; // barriers and rounds of the whole run so far
    unsigned long long relax = 0, frows = 0;

    __device__ Run(const RunArgs &a_, RunSmem &s_) : a(a_), sh(s_) {}

    __device__ __forceinline__ uint32_t id_of(uint32_t v) const { return sp.meta ? __ldcg(&sp.meta[v].w) : v; }
    __device__ __forceinline__ bool accepting(uint32_t v) const
    {
        return sp.meta ? __ldcg(&sp.meta[v].z) != 0 : ((__ldcg(a.acc + (v >> 5)) >> (v & 31u)) & 1u) != 0;
    }

    __device__ __forceinline__ uint32_t readers(uint32_t v) const
    {
        if (!sp.meta) return __ldg(a.rrowptr + v + 1) - __ldg(a.rrowptr + v);
        const uint4 q = __ldcg(sp.meta + v);
        return q.y - q.x;
    }

    // one push of offer o to reader w in round r: raised first in this round, with no value
    // before, and (where counted) first reached in this round
    struct Pushed {
        bool listed, fresh, row;
    };
    __device__ __forceinline__ void push(const bool (&live)[RUN_P], const uint32_t (&o)[RUN_P], const uint32_t (&w)[RUN_P],
                                         uint32_t r, Pushed (&out)[RUN_P])
    {
        if constexpr (SYNC) {
            ulonglong2 rec[RUN_P];
#pragma unroll
            for (int j = 0; j < RUN_P; ++j)
                rec[j] = live[j] ? __ldcg(reinterpret_cast<const ulonglong2 *>(a.W) + w[j]) : make_ulonglong2(0, 0);
            unsigned long long neww[RUN_P], old[RUN_P];
            bool todo[RUN_P];
            uint32_t base[RUN_P];
            const unsigned long long stamp = (unsigned long long)r << 33;
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) {
                const unsigned long long cur = (r & 1) ? rec[j].y : rec[j].x, prev = (r & 1) ? rec[j].x : rec[j].y;
                const uint32_t cv = (uint32_t)cur;
                if ((cur >> 33) != r) { // not reached in this round yet: the value so far is the larger word's
                    base[j] = max(cv, (uint32_t)prev);
                    neww[j] = stamp | ((unsigned long long)(o[j] > base[j]) << 32) | max(o[j], base[j]);
                    todo[j] = live[j];
                } else { // reached: the word holds the value so far (not raised) or the best offer (raised)
                    base[j] = cv;
                    neww[j] = stamp | (1ull << 32) | o[j];
                    todo[j] = live[j] && o[j] > cv;
                }
            }
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) old[j] = todo[j] ? atomicMax(a.W + 2ull * w[j] + (r & 1), neww[j]) : 0ull;
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) {
                const bool mine = (old[j] >> 33) == r; // this round's already
                out[j].row = todo[j] && !mine;
                out[j].listed = todo[j] && ((neww[j] >> 32) & 1u) && !(mine && ((old[j] >> 32) & 1u));
                out[j].fresh = out[j].listed && base[j] == 0;
            }
        } else {
            unsigned long long old[RUN_P];
            uint32_t seen[RUN_P];
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) {
                seen[j] = r;
                if (BATCH && live[j]) seen[j] = atomicExch(reinterpret_cast<uint32_t *>(a.W + 2ull * w[j] + 1), r);
                old[j] = live[j] ? atomicMax(a.W + (uint64_t)S * w[j], ((unsigned long long)o[j] << 32) | (uint32_t)~r)
                                 : ~0ull;
            }
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) {
                const bool rose = live[j] && (uint32_t)(old[j] >> 32) < o[j];
                out[j].row = live[j] && seen[j] != r;
                out[j].listed = rose && (uint32_t)old[j] != (uint32_t)~r;
                out[j].fresh = rose && (old[j] >> 32) == 0;
            }
        }
    }

    // the value a vertex listed in round r - 1 offers in round r (live, asynchronous)
    __device__ __forceinline__ uint32_t value_of(uint32_t u, uint32_t r) const
    {
        if constexpr (SYNC) return (uint32_t)__ldcg(a.W + 2ull * u + ((r - 1) & 1));
        else return (uint32_t)(__ldcg(a.W + (uint64_t)S * u) >> 32);
    }

    __device__ __forceinline__ void entry(uint32_t u, uint32_t r, bool with_value, uint32_t &o, uint32_t &b, uint32_t &len)
    {
        const uint32_t val = with_value ? value_of(u, r) : 0u;
        uint32_t e;
        if (sp.meta) {
            const uint4 q = __ldcg(sp.meta + u);
            b = q.x;
            e = q.y;
            o = max(val, q.z);
        } else {
            b = __ldg(a.rrowptr + u);
            e = __ldg(a.rrowptr + u + 1);
            o = max(val, ((__ldcg(a.acc + (u >> 5)) >> (u & 31u)) & 1u) ? u + 1 : 0u);
        }
        // round 1: an eliminated vertex offers nothing, nor does one of a finished graph
        bool idle = o == 0;
        if (BATCH && !with_value) idle = idle || !*(volatile uint32_t *)&a.cs[__ldcg(sp.comp + u)].active;
        len = idle ? 0u : e - b;
    }

    // a frontier row: its length to the relaxation count (batched: of its graph g too); the whole warp calls it
    __device__ __forceinline__ void count_row(bool row, uint32_t len, uint32_t g)
    {
        if (row) {
            relax += len;
            ++frows;
        }
        if constexpr (BATCH) {
            const uint32_t c = row ? g : NONE, l = row ? len : 0u;
            const unsigned same = __match_any_sync(0xFFFFFFFFu, c);
            const unsigned lo = __reduce_add_sync(same, l & 0xFFFFu);
            const unsigned hi = __reduce_add_sync(same, l >> 16);
            const unsigned long long sum = (unsigned long long)lo + ((unsigned long long)hi << 16);
            if (c != NONE && lane_id() == (unsigned)(__ffs(same) - 1) && sum)
                atomicAdd((unsigned long long *)&a.cs[c].relax, sum);
        }
    }
    __device__ __forceinline__ void add_row(bool row, uint32_t w)
    {
        uint32_t len = 0, g = NONE;
        if (row) {
            len = sp.row ? __ldcg(sp.row + w) : __ldg(a.rowptr + w + 1) - __ldg(a.rowptr + w);
            if (BATCH) g = __ldcg(sp.comp + w);
        }
        count_row(row, len, g);
    }

    // one round over `list` (nl entries); returns false if a wait gave up
    __device__ __forceinline__ bool round(const uint32_t *list, uint32_t nl, uint32_t *next, uint32_t r, uint32_t outer,
                                          bool timing, unsigned long long &total)
    {
        RunCtl *c = a.ctl;
        // (list counters rotate by the run's round number: the one after this was last used two rounds ago)
        ++lseq;
        uint32_t *lcnt = &c->lcnt[lseq % 3].v, *tcnt = &c->tcnt[outer & 1].v;
        if (threadIdx.x == 0) {
            sh.ln = sh.tn = 0;
            if (blockIdx.x == 0) *(volatile uint32_t *)&c->lcnt[(lseq + 1) % 3].v = 0;
        }
        __syncthreads();
        const uint64_t per = ((uint64_t)nl + gridDim.x - 1) / gridDim.x;
        const uint64_t beg = min((uint64_t)nl, blockIdx.x * per), end = min((uint64_t)nl, beg + per);
        bool local = false;
        auto get = [&](uint64_t i, uint32_t &o, uint32_t &b, uint32_t &len) {
            entry(local ? sh.list[i] : __ldcg(list + i), r, local || r > 1, o, b, len);
        };
        auto begin = [&](bool, uint64_t, uint32_t, uint32_t, uint32_t tot) {
            if (!SYNC && !BATCH && threadIdx.x == 0 && (r > 1 || local || a.count_round1)) relax += tot;
        };
        auto act = [&](const bool (&live)[RUN_P], const uint32_t (&o)[RUN_P], const uint32_t (&pos)[RUN_P],
                       const uint32_t (&)[RUN_P]) {
            uint32_t w[RUN_P];
            Pushed done[RUN_P];
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) w[j] = live[j] ? __ldcg(sp.rc + pos[j]) : 0u; // (compact: written in this launch)
            push(live, o, w, r, done);
#pragma unroll
            for (int j = 0; j < RUN_P; ++j) {
                if ((SYNC || BATCH) && r > 1) add_row(done[j].row, w[j]);
                if (BATCH && done[j].listed) changed(w[j], r);
                stage_emit(done[j].listed, w[j], sh.list, &sh.ln, next, lcnt);
                stage_emit(done[j].fresh, w[j], sh.touch, &sh.tn, a.touched, tcnt);
            }
        };
        expand(sh, beg, end, get, begin, act);
        if (!SYNC && !BATCH) {
            // the block pushes the live values of the vertices it listed itself once more (lc_passes
            // times), so that values travel several edges per barrier; they stay listed
            uint32_t q = 0;
            local = true;
            for (uint32_t pass = 0; pass < a.lc_passes; ++pass) {
                const uint32_t e = min(sh.ln, RUN_CAP); // final: a block barrier ended the last chunk
                __syncthreads();                        // (read by every thread before it grows)
                if (e == q) break;
                expand(sh, q, e, get, begin, act);
                q = e;
            }
        }
        __syncthreads();
        const uint32_t ln = sh.ln, kept = min(ln, RUN_CAP), tkept = min(sh.tn, RUN_CAP);
        if (threadIdx.x == 0 && kept) sh.lbase = atomicAdd(lcnt, kept);
        if (threadIdx.x == 32 && tkept) sh.tbase = atomicAdd(tcnt, tkept);
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < kept; i += RT) next[sh.lbase + i] = sh.list[i];
        for (uint32_t i = threadIdx.x; i < tkept; i += RT) a.touched[sh.tbase + i] = sh.touch[i];
        return run_barrier(c, c->bar, sh, seq, (unsigned long long)ln + (timing ? RUN_STOP : 0ull), total);
    }

    // ---- scan mode (whole graph): three arrays of n words in the pool.
    //   synchronous   A / B = the inboxes of even / odd rounds, val = the values (as in k_tail)
    //   asynchronous  val = the values, A = the value pushed last; batched, B / tval = the last odd / even round a row was
    //                 reached in (the round before is read while this round's pushes come in)
    __device__ __forceinline__ uint32_t *scan_val() const { return a.pool; }
    __device__ __forceinline__ uint32_t *scan_a() const { return a.pool + a.n; }
    __device__ __forceinline__ uint32_t *scan_b() const { return a.pool + 2ull * a.n; }
    __device__ __forceinline__ uint32_t *scan_reach(uint32_t r) const { return (r & 1) ? scan_b() : a.tval; }

    // from lists to scans after round r: the state words into the arrays and back to zero; a vertex of round r's
    // list looks as if its value had just come in
    __device__ __forceinline__ bool enter_scan(uint32_t r, unsigned long long &total)
    {
        const uint64_t nthreads = (uint64_t)gridDim.x * RT;
        for (uint64_t v = (uint64_t)blockIdx.x * RT + threadIdx.x; v < a.n; v += nthreads) {
            uint32_t x, in;
            if constexpr (SYNC) {
                ulonglong2 *p = reinterpret_cast<ulonglong2 *>(a.W) + v;
                const ulonglong2 q = __ldcg(p);
                if (q.x | q.y) *p = make_ulonglong2(0, 0);
                const unsigned long long cur = (r & 1) ? q.y : q.x;
                x = max((uint32_t)q.x, (uint32_t)q.y);
                in = (cur >> 33) == r && ((cur >> 32) & 1u) ? x : 0u;
                scan_val()[v] = in ? 0u : x;
                ((r & 1) ? scan_b() : scan_a())[v] = in;
                ((r & 1) ? scan_a() : scan_b())[v] = 0;
            } else {
                const unsigned long long q = __ldcg(a.W + (uint64_t)S * v);
                if (q) a.W[(uint64_t)S * v] = 0;
                if (BATCH && q) a.W[2ull * v + 1] = 0;
                x = (uint32_t)(q >> 32);
                scan_val()[v] = x;
                scan_a()[v] = (uint32_t)q == (uint32_t)~r ? 0u : x;
                if (BATCH) scan_reach(0)[v] = scan_reach(1)[v] = 0;
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) *(volatile uint32_t *)&a.ctl->ocnt[0].v = 0;
        return run_barrier(a.ctl, a.ctl->bar, sh, seq, 0, total);
    }

    // round r: what came in in round r - 1 is taken (first: from the list of round r - 1, whose rows are counted
    // already) and, unless past the limit, pushed on; total = the vertices that changed in round r - 1
    __device__ __forceinline__ bool scan_round(uint32_t r, bool first, bool pushes, bool timing, unsigned long long &total)
    {
        constexpr uint32_t U = 4, CHUNK = RT * U; // words in flight per thread
        uint32_t *const val = scan_val(), *const in = (r & 1) ? scan_a() : scan_b(), *const to = SYNC ? ((r & 1) ? scan_b() : scan_a()) : val;
        // pieces of RT vertices go round the blocks: a wave through consecutive vertices (layers) is everybody's
        const uint64_t step = (uint64_t)gridDim.x * RT, v0 = (uint64_t)blockIdx.x * RT, v1 = a.n;
        uint32_t hits = 0;
        __syncthreads();
        if (threadIdx.x == 0) sh.ln = 0;
        __syncthreads();
        for (uint64_t c0 = v0; c0 < v1; c0 += step * U) { // (block-uniform)
            // three steps with U loads in flight each: what came in; for the warps' words with something in
            // them what the vertex holds, its row and graph; the rest
            uint32_t y[U], z[U], len[U], g[U];
            bool row[U];
#pragma unroll
            for (uint32_t k = 0; k < U; ++k) {
                const uint64_t v = c0 + k * step + threadIdx.x;
                y[k] = v < v1 ? __ldcg((SYNC ? in : val) + v) : 0u;
                if (!SYNC) z[k] = v < v1 ? __ldcg(scan_a() + v) : 0u;
                row[k] = !SYNC && BATCH && v < v1 && __ldcg(scan_reach(r - 1) + v) == r - 1;
            }
            uint32_t some = 0; // (warp-uniform) bit k: something in the warp's word k
#pragma unroll
            for (uint32_t k = 0; k < U; ++k) {
                const uint32_t v = (uint32_t)(c0 + k * step + threadIdx.x);
                if (SYNC) row[k] = y[k] != 0;
                len[k] = 0;
                g[k] = NONE;
                if (!__any_sync(0xFFFFFFFFu, row[k] || (!SYNC && y[k] > z[k]))) continue;
                some |= 1u << k;
                if (c0 + k * step + threadIdx.x >= v1) continue;
                if (SYNC) z[k] = __ldcg(val + v);
                if (SYNC || BATCH) len[k] = __ldg(a.rowptr + v + 1) - __ldg(a.rowptr + v);
                if (BATCH) g[k] = __ldcg(sp.comp + v);
            }
#pragma unroll
            for (uint32_t k = 0; k < U; ++k) {
                if (!((some >> k) & 1u)) continue;
                const uint32_t v = (uint32_t)(c0 + k * step + threadIdx.x);
                if (SYNC && c0 + k * step + threadIdx.x < v1) in[v] = 0; // (whole lines)
                const bool hit = y[k] != 0 && y[k] > z[k];
                if (hit) (SYNC ? val : scan_a())[v] = y[k];
                if ((SYNC || BATCH) && !first && r > 2) count_row(row[k], len[k], g[k]); // frontier rows of round r - 1
                if (BATCH && hit) changed_graph(g[k], r - 1);
                const unsigned m = __ballot_sync(0xFFFFFFFFu, hit);
                if (!m) continue;
                uint32_t at = 0;
                if (lane_id() == 0) at = atomicAdd(&sh.ln, (uint32_t)__popc(m));
                at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(m & ((1u << lane_id()) - 1u));
                if (hit) {
                    sh.list[at] = v;
                    sh.touch[at] = y[k];
                }
            }
            __syncthreads();
            const uint32_t nq = sh.ln; // (the hits of several chunks are pushed together)
            __syncthreads();           // (read by every warp before the next chunk's hits are added: all take one branch)
            if (nq + CHUNK <= RUN_CAP && c0 + step * U < v1) continue;
            hits += nq;
            if (pushes)
                expand(
                    sh, 0, nq,
                    [&](uint64_t i, uint32_t &o, uint32_t &b, uint32_t &len) {
                        const uint32_t u = sh.list[i];
                        b = __ldg(a.rrowptr + u);
                        len = __ldg(a.rrowptr + u + 1) - b;
                        uint32_t x = sh.touch[i];
                        if (!SYNC) scan_a()[u] = x = __ldcg(val + u); // (raised since, perhaps: not pushed twice)
                        o = max(x, ((__ldcg(a.acc + (u >> 5)) >> (u & 31u)) & 1u) ? u + 1 : 0u);
                    },
                    [&](bool, uint64_t, uint32_t, uint32_t, uint32_t tot) {
                        if (!SYNC && !BATCH && threadIdx.x == 0) relax += tot;
                    },
                    [&](const bool (&live)[RUN_P], const uint32_t (&o)[RUN_P], const uint32_t (&pos)[RUN_P], const uint32_t (&)[RUN_P]) {
#pragma unroll
                        for (int j = 0; j < RUN_P; ++j) {
                            if (!live[j]) continue;
                            const uint32_t w = __ldcg(sp.rc + pos[j]);
                            atomicMax(to + w, o[j]);
                            if (!SYNC && BATCH) atomicMax(scan_reach(r) + w, r);
                        }
                    });
            __syncthreads();
            if (threadIdx.x == 0) sh.ln = 0;
            __syncthreads();
        }
        return run_barrier(a.ctl, a.ctl->bar, sh, seq, (unsigned long long)hits + (timing ? RUN_STOP : 0ull), total);
    }

    // from scans back to lists after round r, in the place of the scan that would take what round r pushed: the
    // values into the state words, the vertices that changed in round r to `list`, those with a value to the
    // touched list; total = the length of `list`
    __device__ __forceinline__ bool leave_scan(uint32_t r, uint32_t outer, uint32_t *list, unsigned long long &total)
    {
        constexpr uint32_t U = 4, CHUNK = RT * U;
        RunCtl *c = a.ctl;
        ++lseq;
        uint32_t *const lcnt = &c->lcnt[lseq % 3].v, *const tcnt = &c->tcnt[outer & 1].v;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *(volatile uint32_t *)&c->lcnt[(lseq + 1) % 3].v = 0;
            *(volatile uint32_t *)tcnt = 0; // (the touched list is made anew)
        }
        if (!run_barrier(c, c->bar, sh, seq, 0, total)) return false;
        uint32_t *const val = scan_val(), *const in = (r & 1) ? scan_b() : scan_a();
        uint32_t listed = 0;
        for (uint64_t c0 = (uint64_t)blockIdx.x * CHUNK; c0 < a.n; c0 += (uint64_t)gridDim.x * CHUNK) { // (block-uniform)
            uint32_t x[U], got = 0; // per vertex: its value; got: bits 0-3 = changed in round r
            uint32_t nt = 0, nl = 0;
#pragma unroll
            for (uint32_t k = 0; k < U; ++k) {
                const uint64_t v = c0 + k * RT + threadIdx.x;
                x[k] = v < a.n ? __ldcg(val + v) : 0u;
                bool row = false, ch = false;
                if constexpr (SYNC) {
                    const uint32_t y = v < a.n ? __ldcg(in + v) : 0u;
                    row = y != 0;
                    ch = y > x[k];
                    x[k] = max(x[k], y);
                } else if (v < a.n) {
                    ch = x[k] > __ldcg(scan_a() + v);
                    row = BATCH && __ldcg(scan_reach(r) + v) == r;
                }
                if ((SYNC || BATCH) && r > 1 && __any_sync(0xFFFFFFFFu, row)) add_row(row, (uint32_t)v);
                if (ch) {
                    got |= 1u << k;
                    ++nl;
                    if (BATCH) changed((uint32_t)v, r);
                }
                if (x[k]) {
                    ++nt;
                    if constexpr (SYNC) {
                        const unsigned long long w = ch ? (unsigned long long)r << 33 | 1ull << 32 | x[k] : x[k];
                        reinterpret_cast<ulonglong2 *>(a.W)[v] = (r & 1) ? make_ulonglong2(0, w) : make_ulonglong2(w, 0);
                    } else {
                        a.W[(uint64_t)S * v] = (unsigned long long)x[k] << 32 | (uint32_t)~(ch ? r : 0u);
                        if (BATCH) a.W[2ull * v + 1] = row ? r : 0u;
                    }
                }
            }
            const uint32_t both = run_block_scan(nt << 16 | nl, sh.scan); // (at most 2,048 each)
            if (threadIdx.x == RT - 1) {
                sh.tbase = atomicAdd(tcnt, both >> 16);
                sh.lbase = atomicAdd(lcnt, both & 0xFFFFu);
                listed += both & 0xFFFFu;
            }
            __syncthreads();
            uint32_t ta = sh.tbase + (both >> 16) - nt, la = sh.lbase + (both & 0xFFFFu) - nl;
#pragma unroll
            for (uint32_t k = 0; k < U; ++k) {
                const uint32_t v = (uint32_t)c0 + k * RT + threadIdx.x;
                if (x[k]) a.touched[ta++] = v;
                if ((got >> k) & 1u) list[la++] = v;
            }
            __syncthreads(); // (the bases are read)
        }
        if (threadIdx.x == RT - 1) sh.ln = listed;
        __syncthreads();
        return run_barrier(c, c->bar, sh, seq, sh.ln, total);
    }

    // batched: vertex v's graph changed in round r
    __device__ __forceinline__ void changed(uint32_t v, uint32_t r) { changed_graph(__ldcg(sp.comp + v), r); }
    __device__ __forceinline__ void changed_graph(uint32_t g, uint32_t r)
    {
        CompState &s = a.cs[g];
        if (*(volatile uint32_t *)&s.last_change < r) atomicMax(&s.last_change, r);
    }
};

// per-graph end of an outer iteration in a batched run: does graph S go on?
__device__ __forceinline__ bool comp_goes_on(const volatile CompState &S, uint32_t status, uint32_t max_outer, uint32_t &left,
                                             bool &limit)
{
    limit = false;
    left = S.nacc;
    if (status != ST_OK || S.witness != NONE || S.touched == 0) return false;
    left = S.nacc - S.elim;
    if (left == 0) return false;
    limit = (max_outer && S.outer >= max_outer) || S.outer > S.nacc0;
    return !limit;
}

// one block (every thread of it): the end of an outer iteration for every graph of a batch; the number that
// go on.  s: a shared word.
__device__ __forceinline__ uint32_t end_graphs(const RunArgs &a, uint32_t status, uint32_t *s)
{
    unsigned on = 0;
    for (uint32_t g = threadIdx.x; g < a.ncomp; g += blockDim.x) {
        volatile CompState &S = a.cs[g];
        if (!S.active) continue;
        const uint32_t it = S.outer, rounds = S.last_change + 1;
        if (it - 1 < CH_CAP) a.chist[(size_t)g * CH_CAP + it - 1] = rounds;
        S.inner_total = S.inner_total + rounds;
        S.relax = S.relax + S.m; // round 1 covers every row
        uint32_t left;
        bool limit;
        const bool more = comp_goes_on(S, status, a.max_outer, left, limit);
        if (status != ST_OK) S.status = status;
        else if (limit) S.status = ST_LIMIT;
        if (status == ST_OK && S.witness != NONE) S.verdict = 1;
        else S.nacc = left;
        if (more) {
            S.outer = it + 1;
            S.witness = NONE;
            S.elim = S.touched = S.last_change = 0;
            ++on;
        } else {
            S.active = 0;
        }
    }
    on = __reduce_add_sync(0xFFFFFFFFu, on);
    __syncthreads();
    if (threadIdx.x == 0) *s = 0;
    __syncthreads();
    if (lane_id() == 0 && on) atomicAdd(s, on);
    __syncthreads();
    return *s;
}

template <bool SYNC, bool BATCH>
__global__ void __launch_bounds__(RT, MAPGPU_RUN_BLOCKS) k_run(const __grid_constant__ RunArgs a)
{
    __shared__ RunSmem sh;
    Run<SYNC, BATCH> run(a, sh);
    RunCtl *c = a.ctl;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    const uint64_t tid = (uint64_t)blockIdx.x * RT + threadIdx.x, nthreads = (uint64_t)gridDim.x * RT;
    const uint32_t n = a.n;
    const uint64_t t0 = global_ns();
    uint64_t mark = t0, ph_rounds = 0, ph_check = 0;
    auto phase = [&](uint64_t &acc) {
        const uint64_t now = global_ns();
        if ((int64_t)(now - mark) > 0) {
            acc += now - mark;
            mark = now;
        }
    };
    auto late = [&] { return lead && (int64_t)(global_ns() - t0) > (int64_t)a.timeout_ns; };
    uint32_t *la = a.la, *lb = a.lb, *alist = a.alist;
    unsigned long long total = 0;
    bool alive = true; // no wait has given up

    // the accepting set of the run, the list of its vertices, and an empty map vector
    for (uint64_t base = tid - threadIdx.x; base < a.words; base += nthreads) { // (block-uniform)
        const uint64_t i = base + threadIdx.x;
        uint32_t x = i < a.words ? __ldg(a.acc0 + i) : 0u;
        if (i < a.words) a.acc[i] = x;
        const uint32_t incl = run_block_scan(__popc(x), sh.scan);
        if (threadIdx.x == RT - 1) sh.lbase = incl ? atomicAdd(&c->acnt.v, incl) : 0u;
        __syncthreads();
        uint32_t at = sh.lbase + incl - __popc(x);
        for (; x; x &= x - 1) alist[at++] = (uint32_t)i * 32u + __ffs(x) - 1;
        __syncthreads();
    }
    if (!a.out) {
        // (no map asked for)
    } else if (((uintptr_t)a.out & 15u) == 0) {
        uint4 *o4 = reinterpret_cast<uint4 *>(a.out);
        for (uint64_t i = tid; i < n / 4; i += nthreads) o4[i] = make_uint4(NONE, NONE, NONE, NONE);
        for (uint64_t i = (uint64_t)(n / 4) * 4 + tid; i < n; i += nthreads) a.out[i] = NONE;
    } else {
        for (uint64_t i = tid; i < n; i += nthreads) a.out[i] = NONE;
    }
    alive = run_barrier(c, c->bar, sh, run.seq, 0, total);

    Space &sp = run.sp;
    sp.V = n;
    sp.na = a.nacc0;
    sp.meta = nullptr;
    sp.rc = a.rcol;
    sp.row = nullptr;
    sp.comp = a.comp;
    uint32_t outer = 0, status = ST_OK, verdict = 0, witness = NONE, nacc = a.nacc0, set = 1;
    unsigned long long inner_total = 0;
    bool go = a.nacc0 != 0, compactable = true, hand = false;
    while (go && alive) {
        ++outer;
        if (lead && (SYNC || !a.count_round1)) run.relax += a.m; // round 1 covers every row
        // ---- rounds to the fix-point
        const uint32_t *list = alist;
        uint32_t nl = sp.na, r = 0;
        bool scan = false; // scan mode; then `first`: the state has just been brought into its arrays
        for (bool first = false;;) {
            if (!scan) {
                ++r;
                alive = run.round(list, nl, (r & 1) ? la : lb, r, outer, (r & 3u) == 0 && late(), total);
                if (!alive) break;
                if (!SYNC && !BATCH && r > 1) run.frows += lead ? nl : 0u; // the vertices that pushed
                nl = (uint32_t)(total & RUN_COUNT);
                list = (r & 1) ? la : lb;
                if (total & RUN_STOP) status = ST_TIMEOUT;
                else if (nl && r + 1 > a.max_inner) status = ST_LIMIT;
                if (!nl || status != ST_OK) break;
                if (!sp.meta && nl >= max(n / RUN_SCAN_SHARE, RUN_SCAN_MIN)) {
                    scan = first = true;
                    if (!(alive = run.enter_scan(r, total))) break;
                }
            } else { // (one scan takes what round r pushed and pushes round r + 1)
                const bool pushes = r + 1 <= a.max_inner;
                if (!(alive = run.scan_round(r + 1, first, pushes, (r & 3u) == 0 && late(), total))) break;
                first = false;
                nl = (uint32_t)(total & RUN_COUNT); // changed in round r
                if (!SYNC && !BATCH && lead && pushes) run.frows += nl;
                if (total & RUN_STOP) status = ST_TIMEOUT;
                else if (nl && !pushes) status = ST_LIMIT;
                if (nl && pushes) ++r;
                if (!nl || status != ST_OK) break;
                if (nl < n / RUN_LIST_SHARE) {
                    uint32_t *const next = (r & 1) ? la : lb;
                    if (!(alive = run.leave_scan(r, outer, next, total))) break;
                    scan = false;
                    nl = (uint32_t)(total & RUN_COUNT);
                    list = next;
                    if (nl && r + 1 > a.max_inner) status = ST_LIMIT;
                    if (!nl || status != ST_OK) break;
                }
            }
        }
        if (!alive) break;
        inner_total += r;
        if (lead) {
            if (outer - 1 < a.hist_cap) a.hist[outer - 1] = r;
            if (outer - 1 < RUN_HIST) a.res->hist[outer - 1] = r;
            phase(ph_rounds);
        }
        // ---- self-map test and elimination over the vertices with a value; their state back to zero
        uint32_t T = *(volatile uint32_t *)&c->tcnt[outer & 1].v;
        const uint32_t bound = scan ? n : T;
        uint32_t have = 0;
        if (lead) *(volatile uint32_t *)&c->tcnt[(outer + 1) & 1].v = 0;
        uint32_t elim = 0, wit = NONE, settled = 0;
        for (uint64_t base = tid - lane_id(); base < bound; base += nthreads) { // (warp-uniform)
            const uint64_t i = base + lane_id();
            uint32_t g = NONE, removed = 0, val = 0;
            if (i < bound) {
                const uint32_t v = scan ? (uint32_t)i : __ldcg(a.touched + i);
                // (exchanges, not stores: scattered 8-byte stores ran at 14 G/s here, atomics at over 100)
                uint32_t x;
                if (scan) {
                    x = __ldcg(run.scan_val() + v);
                    have += x != 0;
                } else if constexpr (SYNC) {
                    x = max((uint32_t)atomicExch(a.W + 2ull * v, 0ull), (uint32_t)atomicExch(a.W + 2ull * v + 1, 0ull));
                } else {
                    x = (uint32_t)(atomicExch(a.W + (uint64_t)run.S * v, 0ull) >> 32);
                    if (BATCH) atomicExch(a.W + 2ull * v + 1, 0ull);
                }
                if (!scan) a.tval[i] = x;
                if (BATCH && x) g = __ldcg(sp.comp + v);
                if (status == ST_OK) val = x;
                if (val && x - 1 == run.id_of(v)) {
                    wit = min(wit, x - 1);
                    if (BATCH) atomicMin(&a.cs[g].witness, x - 1);
                }
            }
            // u = val - 1 is removed.  Many vertices share a few map values: one lane per value and warp, and
            // none for the value this thread settled last
            const unsigned same_val = __match_any_sync(0xFFFFFFFFu, val);
            if (val && val != settled && lane_id() == (unsigned)(__ffs(same_val) - 1)) {
                const uint32_t u = val - 1, bit = 1u << (u & 31u);
                if ((__ldcg(a.acc + (u >> 5)) & bit) && (atomicAnd(a.acc + (u >> 5), ~bit) & bit)) { // this thread removed u
                    ++elim;
                    removed = 1;
                    if (sp.meta) const_cast<uint4 *>(sp.meta)[__ldcg(a.rank + u) - 1].z = 0; // it offers nothing any more
                }
            }
            settled = val;
            if constexpr (BATCH) { // per graph: vertices with a value and removals, one atomic per graph in the warp
                const unsigned same = __match_any_sync(0xFFFFFFFFu, g);
                const unsigned ne = __reduce_add_sync(same, removed);
                if (g != NONE && lane_id() == (unsigned)(__ffs(same) - 1)) {
                    atomicAdd(&a.cs[g].touched, (unsigned)__popc(same));
                    if (ne) atomicAdd(&a.cs[g].elim, ne);
                }
            }
        }
        { // block sums
            elim = __reduce_add_sync(0xFFFFFFFFu, elim);
            wit = __reduce_min_sync(0xFFFFFFFFu, wit);
            __syncthreads();
            if (threadIdx.x == 0) sh.ln = 0, sh.tn = NONE;
            __syncthreads();
            if (lane_id() == 0) {
                if (elim) atomicAdd(&sh.ln, elim);
                if (wit != NONE) atomicMin(&sh.tn, wit);
            }
            __syncthreads();
            elim = sh.ln;
            wit = sh.tn;
            if (threadIdx.x == 0 && wit != NONE) atomicMax(&c->witness.v, NONE - wit);
            have = __reduce_add_sync(0xFFFFFFFFu, have);
            if (have && lane_id() == 0) atomicAdd(&c->ocnt[0].v, have);
        }
        alive = run_barrier(c, c->bar, sh, run.seq,
                            (unsigned long long)elim + (wit != NONE ? RUN_FOUND : 0ull) + (late() ? RUN_STOP : 0ull), total);
        if (!alive) break;
        if (scan) T = *(volatile uint32_t *)&c->ocnt[0].v;
        if (lead) phase(ph_check);
        if constexpr (!BATCH) {
            if (status != ST_OK) go = false; // a limit inside the rounds
            else if (total & (RUN_STOP - RUN_FOUND)) {
                verdict = 1;
                witness = NONE - *(volatile uint32_t *)&c->witness.v;
                go = false;
            } else if (T == 0) {
                go = false; // nothing reaches a remaining accepting vertex
            } else {
                nacc -= (uint32_t)(total & RUN_COUNT);
                if (nacc == 0) go = false;
                else if ((a.max_outer && outer >= a.max_outer) || outer > a.nacc0) {
                    status = ST_LIMIT;
                    go = false;
                } else if (total & RUN_STOP) {
                    status = ST_TIMEOUT;
                    go = false;
                }
            }
            if (!go && a.out) // the last iteration's map
                for (uint64_t i = tid; i < bound; i += nthreads) {
                    if (scan) a.out[i] = __ldcg(run.scan_val() + i) - 1u; // (no value: MAP_NONE)
                    else a.out[run.id_of(__ldcg(a.touched + i))] = __ldcg(a.tval + i) - 1u;
                }
        } else {
            if (status == ST_OK && (total & RUN_STOP)) status = ST_TIMEOUT;
            uint32_t left;
            bool limit;
            // the maps of the graphs that end here
            for (uint64_t i = tid; a.out && i < bound; i += nthreads) {
                const uint32_t v = scan ? (uint32_t)i : __ldcg(a.touched + i), x = scan ? __ldcg(run.scan_val() + i) : __ldcg(a.tval + i);
                if (!x) continue;
                const uint32_t g = __ldcg(sp.comp + v);
                if (!comp_goes_on(a.cs[g], status, a.max_outer, left, limit))
                    a.out[run.id_of(v)] = x - 1u - *(volatile uint32_t *)&a.cs[g].off;
            }
            nacc -= (uint32_t)(total & RUN_COUNT);
            alive = run_barrier(c, c->bar, sh, run.seq, 0, total);
            if (!alive) break;
            const uint32_t on = blockIdx.x == 0 ? end_graphs(a, status, &sh.ln) : 0u;
            alive = run_barrier(c, c->bar, sh, run.seq, on, total);
            if (!alive) break;
            go = (total & RUN_COUNT) != 0;
        }
        // ---- compaction: go on in the graph of the vertices that had a value and the accepting ones
        const uint32_t cap = pool_cap(n);
        if (go && compactable && !scan && (uint64_t)T + nacc <= min(sp.V / (sp.meta ? 4u : 8u), cap)) {
            for (uint64_t i = tid; i < T; i += nthreads) a.rank[run.id_of(__ldcg(a.touched + i))] = (uint32_t)i + 1;
            if (lead) *(volatile uint32_t *)&c->acnt.v = 0;
            if (!(alive = run_barrier(c, c->bar, sh, run.seq, 0, total))) break;
            uint32_t *anew = la; // (no round is in flight)
            for (uint64_t i = tid; i < sp.na; i += nthreads) { // (one that no row holds offers nothing to anyone)
                const uint32_t v = __ldcg(alist + i);
                if (run.readers(v) == 0) continue;
                if (!run.accepting(v) || (BATCH && !*(volatile uint32_t *)&a.cs[__ldcg(sp.comp + v)].active)) continue;
                const uint32_t u = run.id_of(v);
                uint32_t k = __ldcg(a.rank + u);
                if (!(k >= 1 && k <= T && __ldcg(a.touched + k - 1) == v)) { // it has no value: after those that have
                    k = T + agg_inc(&c->xcnt.v) + 1;
                    a.touched[k - 1] = v;
                    a.rank[u] = k;
                }
                anew[agg_inc(&c->acnt.v)] = k - 1;
            }
            if (!(alive = run_barrier(c, c->bar, sh, run.seq, 0, total))) break;
            const uint32_t V2 = T + *(volatile uint32_t *)&c->xcnt.v, na2 = *(volatile uint32_t *)&c->acnt.v;
            uint32_t *const ps = pool_set(a, set ^ 1);
            uint4 *const meta2 = reinterpret_cast<uint4 *>(ps);
            uint32_t *const row2 = ps + 4ull * cap, *const comp2 = row2 + cap, *const rc2 = comp2 + cap;
            const uint64_t ecap = (uint64_t)n * 3 / 4 - 8;
            bool over = false;
            const uint64_t per = ((uint64_t)V2 + gridDim.x - 1) / gridDim.x;
            const uint64_t beg = min((uint64_t)V2, blockIdx.x * per), end = min((uint64_t)V2, beg + per);
            uint32_t first = 0; // this chunk's first entry in rc2
            expand(
                sh, beg, end,
                [&](uint64_t i, uint32_t &, uint32_t &b, uint32_t &len) {
                    const uint32_t v = __ldcg(a.touched + i);
                    if (sp.meta) {
                        const uint4 q = __ldcg(sp.meta + v);
                        b = q.x;
                        len = q.y - q.x;
                    } else {
                        b = __ldg(a.rrowptr + v);
                        len = __ldg(a.rrowptr + v + 1) - b;
                    }
                },
                [&](bool in, uint64_t i, uint32_t excl, uint32_t len, uint32_t tot) {
                    if (threadIdx.x == 0) sh.ebase = tot ? atomicAdd(&c->ecnt.v, tot) : 0u;
                    __syncthreads();
                    first = sh.ebase;
                    if ((uint64_t)first + tot > ecap) over = true;
                    if (in) {
                        const uint32_t v = __ldcg(a.touched + i), u = run.id_of(v);
                        // (batched: a graph that has ended keeps its values, and offers nothing any more)
                        const bool offers = run.accepting(v) && !(BATCH && !*(volatile uint32_t *)&a.cs[__ldcg(sp.comp + v)].active);
                        meta2[i] = make_uint4(first + excl, first + excl + len, offers ? u + 1 : 0u, u);
                        if (SYNC || BATCH)
                            row2[i] = sp.row ? __ldcg(sp.row + v) : __ldg(a.rowptr + v + 1) - __ldg(a.rowptr + v);
                        if (BATCH) comp2[i] = __ldcg(sp.comp + v);
                    }
                },
                [&](const bool (&live)[RUN_P], const uint32_t (&)[RUN_P], const uint32_t (&pos)[RUN_P],
                    const uint32_t (&pair)[RUN_P]) {
                    if (over) return;
#pragma unroll
                    for (int j = 0; j < RUN_P; ++j)
                        if (live[j]) rc2[first + pair[j]] = __ldcg(a.rank + run.id_of(__ldcg(sp.rc + pos[j]))) - 1;
                });
            if (!(alive = run_barrier(c, c->bar, sh, run.seq, over ? 1 : 0, total))) break;
            if (lead) {
                // (who goes on, if the compact graph is left to a kernel below)
                c->next = V2 <= a.tail_cap && (*(volatile uint32_t *)&c->ecnt.v <= a.tail_m || V2 > a.own_cap) ? 2u : 1u;
                *(volatile uint32_t *)&c->xcnt.v = *(volatile uint32_t *)&c->ecnt.v = 0;
            }
            if (total & RUN_COUNT) { // too many readers for the pool: stay in the whole graph
                compactable = false;
            } else {
                sp.V = V2;
                sp.na = na2;
                sp.meta = meta2;
                sp.rc = rc2;
                sp.row = row2;
                sp.comp = comp2;
                set ^= 1;
                uint32_t *const t = alist;
                alist = la;
                la = t;
                if (V2 <= max(a.tail_cap, a.own_cap)) { // small enough for one of the kernels below
                    hand = true;
                    break;
                }
            }
        }
    }
    // ---- the result
    for (unsigned long long *p : {&run.relax, &run.frows}) {
        const unsigned long long s = warp_sum64(*p);
        __syncthreads();
        if (lane_id() == 0) sh.part[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long t = 0;
            for (int w = 0; w < RT / 32; ++w) t += sh.part[w];
            if (t) atomicAdd(p == &run.relax ? &c->relax.v : &c->frows.v, t);
        }
    }
    if (hand) {
        if (lead) {
            c->V = sp.V;
            c->set = set;
            c->outer = outer;
            c->nacc = nacc;
            c->inner_total = inner_total;
            c->ph_rounds = ph_rounds;
            c->ph_check = ph_check;
            c->t0 = t0;
            c->ocnt[0].v = c->ocnt[1].v = 0; // (scan mode has counted there; k_own starts from zero)
            c->hand = c->next;
        }
        return;
    }
    if (alive) alive = run_barrier(c, c->bar, sh, run.seq, 0, total);
    if (lead) {
        RunRes *R = a.res;
        R->verdict = verdict;
        R->witness = witness;
        R->outer = outer;
        R->status = alive ? status : ST_TIMEOUT;
        R->gave_up = alive ? 0u : 1u;
        R->nacc = nacc;
        R->inner_total = inner_total;
        R->relax = *(volatile unsigned long long *)&c->relax.v;
        R->frontier_rows = *(volatile unsigned long long *)&c->frows.v;
        R->ph_rounds = ph_rounds;
        R->ph_check = ph_check;
    }
}

// ---------------------------------------------------------- counterexample --
//
// k_lasso: the shortest paths from[q] -> to[q] along rows (at least one edge), q = 0 and 1 (from NONE: none
// asked for), by breadth-first search with parent pointers, all levels in one cooperative launch.  A level
// is a handful of dependent accesses; stepped from the host, each cost a launch, two pageable copies and a wait
// besides (10^6 vertices, two searches of about ten levels: 1.0 ms, here 0.1 ms).  The path is left backwards
// in path[q] (its first 256 vertices in res->hist[256 q ..] too) and its length in res->verdict and
// res->witness (0: not reachable).
struct LassoArgs {
    uint32_t n;
    const uint32_t *rowptr, *colidx;
    uint32_t from[2], to[2];
    uint32_t *parent[2], *path[2], *qa, *qb; // n entries each (path[1]: n + 1)
    RunCtl *ctl;
    RunRes *res;
};

__global__ void __launch_bounds__(RT, MAPGPU_RUN_BLOCKS) k_lasso(const __grid_constant__ LassoArgs a)
{
    __shared__ RunSmem sh;
    RunCtl *c = a.ctl;
    const uint64_t tid = (uint64_t)blockIdx.x * RT + threadIdx.x, nthreads = (uint64_t)gridDim.x * RT;
    uint32_t seq = 0, lseq = 0;
    unsigned long long total = 0;
    for (int q = 0; q < 2; ++q)
        if (a.from[q] != NONE)
            for (uint64_t i = tid; i < a.n; i += nthreads) // (a source that is not the target is reached from the start)
                a.parent[q][i] = i == a.from[q] && a.from[q] != a.to[q] ? a.from[q] : NONE;
    bool alive = run_barrier(c, c->bar, sh, seq, 0, total), found[2] = {false, false};
    for (int q = 0; q < 2 && alive; ++q) {
        if (a.from[q] == NONE) continue;
        uint32_t *const parent = a.parent[q];
        uint32_t nl = 1;
        for (uint32_t level = 0; nl && !found[q] && alive; ++level) {
            ++lseq;
            const uint32_t *const in = (lseq & 1) ? a.qa : a.qb;
            uint32_t *const out = (lseq & 1) ? a.qb : a.qa;
            uint32_t *const cnt = &c->lcnt[lseq % 3].v;
            __syncthreads(); // (the staged list of the last level is read)
            if (threadIdx.x == 0) {
                sh.ln = sh.tn = 0;
                if (blockIdx.x == 0) *(volatile uint32_t *)&c->lcnt[(lseq + 1) % 3].v = 0;
            }
            __syncthreads();
            const uint64_t per = ((uint64_t)nl + gridDim.x - 1) / gridDim.x;
            const uint64_t beg = min((uint64_t)nl, blockIdx.x * per), end = min((uint64_t)nl, beg + per);
            expand(
                sh, beg, end,
                [&](uint64_t i, uint32_t &o, uint32_t &b, uint32_t &len) {
                    o = level ? __ldcg(in + i) : a.from[q];
                    b = __ldg(a.rowptr + o);
                    len = __ldg(a.rowptr + o + 1) - b;
                },
                [](bool, uint64_t, uint32_t, uint32_t, uint32_t) {},
                [&](const bool (&live)[RUN_P], const uint32_t (&u)[RUN_P], const uint32_t (&pos)[RUN_P], const uint32_t (&)[RUN_P]) {
#pragma unroll
                    for (int j = 0; j < RUN_P; ++j) {
                        bool fresh = false;
                        uint32_t v = 0;
                        if (live[j]) {
                            v = __ldg(a.colidx + pos[j]) & 0x7FFFFFFFu; // bit 31 is the accepting flag
                            fresh = __ldcg(parent + v) == NONE && atomicCAS(parent + v, NONE, u[j]) == NONE;
                            if (fresh && v == a.to[q]) sh.tn = 1;
                        }
                        stage_emit(fresh, v, sh.list, &sh.ln, out, cnt);
                    }
                });
            __syncthreads();
            const uint32_t ln = sh.ln, kept = min(ln, RUN_CAP);
            if (threadIdx.x == 0 && kept) sh.lbase = atomicAdd(cnt, kept);
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < kept; i += RT) out[sh.lbase + i] = sh.list[i];
            alive = run_barrier(c, c->bar, sh, seq, (unsigned long long)ln + (sh.tn ? RUN_FOUND : 0ull), total);
            nl = (uint32_t)(total & RUN_COUNT);
            found[q] = (total >> 32) != 0;
        }
    }
    // walked back by one thread each
    const uint32_t q = blockIdx.x;
    if (threadIdx.x == 0 && q < 2) {
        uint32_t k = 0;
        if (alive && a.from[q] != NONE && found[q]) {
            uint32_t v = a.to[q];
            do { // (a parent chain visits distinct vertices, the target twice when it is the source)
                if (k) v = __ldcg(a.parent[q] + v);
                a.path[q][k] = v;
                if (k < RUN_HIST / 2) a.res->hist[q * (RUN_HIST / 2) + k] = v;
                ++k;
            } while ((k == 1 || v != a.from[q]) && k <= a.n);
        }
        if (q == 0) a.res->verdict = k;
        else a.res->witness = k;
        if (q == 0) a.res->gave_up = alive ? 0u : 1u;
    }
}

// ------------------------------------------------------------ small graphs --
//
// k_tail: the same run in one thread-block cluster with the vertices' state in shared memory, for a
// whole graph of at most TAIL_N vertices per block, or for the compact graph that k_run leaves.
// A round over a few thousand vertices is a chain of latencies: through L2 and the grid barrier it
// takes 6-7 us, here 1 us or less -- a push is one 32-bit maximum into the owner's shared memory
// (nothing waits for it), and the cluster barrier takes 0.3 us.  There are no lists: vertex v belongs
// to block v mod C, and every round its owner looks whether it changed, which costs a few
// shared-memory reads per thread.
//   asynchronous  pushes raise the vertex's value itself; it changed if it is above the value it
//                 pushed last;
//   synchronous   pushes of round r go to the vertex's inbox of r's parity; in round r + 1 the owner
//                 takes what came in (the vertex was in round r's frontier: its row length to the
//                 relaxation count) and, if that is above the value, raises it and pushes.
constexpr int TT = 1024;             // threads per block
constexpr uint32_t TAIL_N = 8704;    // vertices per block: 26 bytes of shared memory each
constexpr uint32_t TAIL_C = 16;      // blocks at most
constexpr size_t TAIL_SMEM = (size_t)TAIL_N * 26;
// graphs up to here run in the cluster, larger ones over the grid (k_own).  Layered graphs, synchronous, us per
// run with k_tail / k_own: 16,000 vertices 166 / 205, 30,000 262 / 235, 60,000 317 / 238, 130,000 470 / 263
constexpr uint32_t TAIL_BEST = 16384;
// ... and of at most this many entries: sixteen SMs take some 15 G pushes/s, the chip 133 G.  us per run with k_tail / k_own:
// acyclic graphs (20 iterations, synchronous), 16,384 vertices with 147,456 entries 10,104 / 3,501, with 1 M 56,453 / 8,910,
// with 4 M 221,713 / 27,697 (dense start 0.18 s); random ones of 16,384 with 262,144 178 / 106, with 4 M 1,168 / 196 (1,340), 4,000
// with 1 M 786 / 135.  Where few vertices change a round is a chain of latencies and k_tail stays ahead: layered 16,000
// with 250,531 entries 373 / 422, asynchronous 301 / 354
constexpr uint32_t TAIL_BEST_M = 262144;
// asynchronous, a vertex per thread: looks at the vertex per round, so that values that came in meanwhile go on
// before the barrier (10^6 layered, us per run with 1 / 2 / 4 / 6 / 8 looks: 900 / 844 / 777 / 764 / 751; 4,000 random
// 80 / - / 71 / 77 / 77; 16,000 layered 163 / - / 148 / 154 / 164)
constexpr int TAIL_PASSES = 4;
constexpr uint32_t TAIL_LONG = 16;   // reader lists longer than this are walked by a whole warp

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of this block's shared word `local` in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_max(uint32_t addr, uint32_t x)
{
    asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
}
__device__ __forceinline__ void cluster_or(uint32_t addr, uint32_t x)
{
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t addr, unsigned long long x)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(x) : "memory");
}
__device__ __forceinline__ uint32_t shared_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

template <bool SYNC>
__global__ void __launch_bounds__(TT, 1) k_tail(const __grid_constant__ RunArgs a, uint32_t whole)
{
    extern __shared__ uint32_t s_mem[];
    __shared__ unsigned long long s_word[2][TAIL_C], s_part[TT / 32], s_sum;
    __shared__ uint32_t s_min[TT / 32], s_n, s_late;
    RunCtl *c = a.ctl;
    if (!whole && *(volatile uint32_t *)&c->hand != 2) return; // the run is finished (every block returns)
    if (a.prep && a.prep[0]) return;                        // k_prepare refused the graph
    const uint32_t nacc0 = a.prep ? a.prep[1] : a.nacc0;
    const uint64_t m = a.prep ? a.prep[2] : a.m;
    const uint32_t C = gridDim.x, rank = cluster_rank(), cshift = __ffs(C) - 1, cmask = C - 1;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const uint32_t V = whole ? a.n : *(volatile uint32_t *)&c->V;
    const uint32_t mine = V > rank ? (V - rank + C - 1) >> cshift : 0u; // vertices rank, rank + C, ...
    // asynchronous: x0 / x1 = the values, by outer iteration mod 2, x2 = the value pushed last
    // synchronous: x0 / x1 = the inboxes, by round mod 2, x2 = the value
    uint32_t *const x0 = s_mem, *const x1 = x0 + TAIL_N, *const x2 = x1 + TAIL_N, *const own = x2 + TAIL_N,
                    *const beg = own + TAIL_N, *const end = beg + TAIL_N;
    uint16_t *const queue = reinterpret_cast<uint16_t *>(end + TAIL_N);
    const uint32_t set = whole ? 0u : *(volatile uint32_t *)&c->set, cap = pool_cap(a.n);
    uint32_t *const ps = pool_set(a, set);
    const uint4 *meta = reinterpret_cast<const uint4 *>(ps);
    const uint32_t *row = ps + 4ull * cap, *rc = whole ? a.rcol : ps + 6ull * cap;
    for (uint32_t i = tid; i < mine; i += TT) {
        const uint32_t v = i << cshift | rank;
        x0[i] = x1[i] = x2[i] = 0;
        if (whole) {
            own[i] = ((__ldg(a.acc0 + (v >> 5)) >> (v & 31u)) & 1u) ? v + 1 : 0u;
            beg[i] = __ldg(a.rrowptr + v);
            end[i] = __ldg(a.rrowptr + v + 1);
        } else {
            const uint4 q = __ldg(meta + v);
            beg[i] = q.x;
            end[i] = q.y;
            own[i] = q.z;
        }
    }
    const uint64_t t0 = whole ? global_ns() : *(volatile unsigned long long *)&c->t0;
    const bool lead = rank == 0 && tid == 0;
    uint64_t mark = global_ns(), ph_rounds = 0, ph_check = 0;
    auto phase = [&](uint64_t &acc) {
        const uint64_t now = global_ns();
        if ((int64_t)(now - mark) > 0) {
            acc += now - mark;
            mark = now;
        }
    };
    uint32_t outer = whole ? 0u : *(volatile uint32_t *)&c->outer, nacc = whole ? nacc0 : *(volatile uint32_t *)&c->nacc;
    uint32_t status = ST_OK, verdict = 0, witness = NONE, seq = 0;
    unsigned long long relax = 0, frows = 0, inner_total = 0;
    // every block's word (the same in its threads 0 .. C - 1) to every block, then the cluster barrier; the
    // calling lane q < C gets block q's word.  The words alternate between two buffers: one is rewritten only
    // after the barrier that follows the reads of its last contents.
    auto exchange = [&](unsigned long long w) {
        const uint32_t k = seq++ & 1u;
        if (tid < C) cluster_store(cluster_addr(shared_addr(&s_word[k][rank]), tid), w);
        cluster_barrier();
        return lane < C ? s_word[k][lane] : 0ull;
    };
    auto exchange0 = [&](unsigned long long w) { // (w: thread 0's)
        if (tid == 0) s_sum = w;
        __syncthreads();
        return exchange(s_sum);
    };
    if (tid == 0) s_late = 0;
    cluster_barrier(); // every block's state is in place
    bool go = nacc != 0;
    while (go) {
        ++outer;
        uint32_t *const val = SYNC ? x2 : (outer & 1) ? x1 : x0;
        if (lead && (SYNC || !a.count_round1)) relax += m; // round 1 covers every row
        uint32_t r = 0;
        for (;;) {
            ++r;
            uint32_t *const inbox = (r & 1) ? x0 : x1; // what came in round r - 1 (synchronous)
            const uint32_t to = shared_addr(SYNC ? ((r & 1) ? x1 : x0) : val);
            const bool pushes = r <= a.max_inner; // (past the limit the last round's values are only taken)
            bool any = false;
            // did vertex i change in round r - 1 (start: is it accepting)?  o: what it offers then
            bool start = r == 1;
            auto changed = [&](uint32_t i, uint32_t &o) {
                if (start) {
                    o = own[i];
                    return o != 0;
                }
                if (SYNC) {
                    const uint32_t y = inbox[i];
                    if (!y) return false;
                    inbox[i] = 0;
                    if (r > 2) { // a frontier row of round r - 1
                        const uint32_t v = i << cshift | rank;
                        relax += whole ? __ldg(a.rowptr + v + 1) - __ldg(a.rowptr + v) : __ldg(row + v);
                        ++frows;
                    }
                    o = max(y, own[i]);
                    if (y <= val[i]) return false;
                    val[i] = y;
                    return true;
                }
                const uint32_t x = *(volatile uint32_t *)(val + i);
                if (x <= x2[i]) return false;
                x2[i] = x;
                o = max(x, own[i]);
                return true;
            };
            // offer o to the readers at rc[b, e); a long list is walked by the whole warp (all lanes call it)
            auto send = [&](uint32_t o, uint32_t b, uint32_t e) {
                if (!SYNC) {
                    if (r > 1 || a.count_round1) relax += e - b;
                    if (r > 1) frows += e != b;
                }
                for (unsigned m = __ballot_sync(0xFFFFFFFFu, e - b > TAIL_LONG); m; m &= m - 1) {
                    const int src = __ffs(m) - 1;
                    const uint32_t ob = __shfl_sync(0xFFFFFFFFu, o, src), bb = __shfl_sync(0xFFFFFFFFu, b, src),
                                   ee = __shfl_sync(0xFFFFFFFFu, e, src);
#pragma unroll 4
                    for (uint32_t j = lane; j < ee - bb; j += 32) {
                        const uint32_t w = __ldg(rc + bb + j);
                        cluster_max(cluster_addr(to + 4 * (w >> cshift), w & cmask), ob);
                    }
                    if ((int)lane == src) b = e;
                }
                for (uint32_t j = 0; j < e - b; j += 4) { // up to four readers in flight
                    uint32_t w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[k] = j + k < e - b ? __ldg(rc + b + j + k) : NONE;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (w[k] != NONE) cluster_max(cluster_addr(to + 4 * (w[k] >> cshift), w[k] & cmask), o);
                }
            };
            if (mine <= TT) { // a vertex per thread
                for (int pass = 0; pass < (SYNC ? 1 : TAIL_PASSES); ++pass) {
                    uint32_t o = 0, b = 0, e = 0;
                    if (tid < mine && changed(tid, o)) {
                        any = true;
                        b = beg[tid];
                        e = pushes ? end[tid] : b;
                    }
                    send(o, b, e);
                    start = false;
                }
            } else { // several: the changed ones are queued first, so that their lists are read side by side
                if (tid == 0) s_n = 0;
                __syncthreads();
                for (uint32_t i0 = 0; i0 < mine; i0 += TT) { // (block-uniform)
                    const uint32_t i = i0 + tid;
                    uint32_t o = 0;
                    const bool hit = i < mine && changed(i, o);
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, hit);
                    uint32_t at = 0;
                    if (m && lane == 0) at = atomicAdd(&s_n, (uint32_t)__popc(m));
                    at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(m & ((1u << lane) - 1u));
                    if (hit) queue[at] = (uint16_t)i;
                }
                __syncthreads();
                const uint32_t nq = s_n;
                any = nq != 0;
                for (uint32_t q0 = 0; pushes && q0 < nq; q0 += TT) { // (block-uniform)
                    const uint32_t q = q0 + tid;
                    uint32_t o = 0, b = 0, e = 0;
                    if (q < nq) {
                        const uint32_t i = queue[q];
                        // (synchronous: the value just taken; asynchronous: the live one)
                        o = start ? own[i] : max(*(volatile uint32_t *)(val + i), own[i]);
                        b = beg[i];
                        e = end[i];
                    }
                    send(o, b, e);
                }
            }
            if (lead && (r & 7u) == 0 && (int64_t)(global_ns() - t0) > (int64_t)a.timeout_ns) any = s_late = 1;
            any = __syncthreads_or(any);
            const unsigned long long word = exchange((any ? 1ull : 0ull) | (s_late ? 2ull : 0ull));
            const bool more = __any_sync(0xFFFFFFFFu, word & 1u), late = __any_sync(0xFFFFFFFFu, word & 2u);
            if (r == 1) continue; // (the limit and the end of the rounds: once round 1's values are taken)
            if (late) status = ST_TIMEOUT;
            else if (more && !pushes) status = ST_LIMIT;
            if (!more) break;
            if (status != ST_OK) break;
        }
        const uint32_t rounds = status == ST_TIMEOUT ? r : r - 1;
        inner_total += rounds;
        if (lead) {
            if (outer - 1 < a.hist_cap) a.hist[outer - 1] = rounds;
            if (outer - 1 < RUN_HIST) a.res->hist[outer - 1] = rounds;
            phase(ph_rounds);
        }
        if (status != ST_OK) break;
        // ---- self-map test; the map values are marked at their owners (bit 31 of the own offer)
        uint32_t wit = NONE, have = 0, settled = 0;
        for (uint32_t i0 = 0; i0 < mine; i0 += TT) {
            const uint32_t i = i0 + tid;
            const uint32_t x = i < mine ? val[i] : 0u;
            if (x) {
                have = 1;
                const uint32_t v = i << cshift | rank;
                if (x - 1 == (whole ? v : __ldg(&meta[v].w))) wit = min(wit, x - 1);
            }
            const unsigned same = __match_any_sync(0xFFFFFFFFu, x); // (many vertices share a few values)
            if (x && x != settled && lane == (unsigned)(__ffs(same) - 1)) {
                const uint32_t u = whole ? x - 1 : __ldg(a.rank + x - 1) - 1;
                cluster_or(cluster_addr(shared_addr(own) + 4 * (u >> cshift), u & cmask), 0x80000000u);
            }
            settled = x;
        }
        have = __syncthreads_or(have);
        wit = __reduce_min_sync(0xFFFFFFFFu, wit);
        if (lane == 0) s_min[warp] = wit;
        __syncthreads();
        if (tid == 0)
            for (int w = 0; w < TT / 32; ++w) wit = min(wit, s_min[w]);
        const unsigned long long seen = exchange0((unsigned long long)(NONE - wit) << 32 | have);
        have = __any_sync(0xFFFFFFFFu, seen & 1u);
        witness = NONE - __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(seen >> 32));
        if (witness != NONE) verdict = 1;
        if (verdict || !have) { // a cycle, or nothing reaches a remaining accepting vertex
            if (lead) phase(ph_check);
            break;
        }
        // ---- elimination
        uint32_t elim = 0;
        for (uint32_t i = tid; i < mine; i += TT)
            if (own[i] >> 31) {
                elim += (own[i] & 0x7FFFFFFFu) != 0;
                own[i] = 0;
            }
        elim = __reduce_add_sync(0xFFFFFFFFu, elim);
        if (lane == 0) s_min[warp] = elim;
        __syncthreads();
        if (tid == 0) {
            elim = 0;
            for (int w = 0; w < TT / 32; ++w) elim += s_min[w];
        }
        const bool late = lead && (int64_t)(global_ns() - t0) > (int64_t)a.timeout_ns;
        const unsigned long long gone = exchange0((unsigned long long)elim | (late ? 1ull << 32 : 0ull));
        nacc -= __reduce_add_sync(0xFFFFFFFFu, (uint32_t)gone);
        if (nacc == 0) go = false;
        else if ((a.max_outer && outer >= a.max_outer) || outer > nacc0) {
            status = ST_LIMIT;
            go = false;
        } else if (__any_sync(0xFFFFFFFFu, (gone >> 32) != 0)) {
            status = ST_TIMEOUT;
            go = false;
        }
        if (lead) phase(ph_check);
        if (go) // values back to none (asynchronous: the next iteration's pushes go to the other array)
            for (uint32_t i = tid; i < mine; i += TT) {
                val[i] = 0;
                if (!SYNC) x2[i] = 0;
            }
    }
    // ---- the map of the last iteration and the result
    if (a.out) {
        uint32_t *const val = SYNC ? x2 : (outer & 1) ? x1 : x0;
        for (uint32_t i = tid; i < mine; i += TT) {
            const uint32_t v = i << cshift | rank, x = val[i];
            if (whole) a.out[v] = x - 1u; // (no value: MAP_NONE)
            else if (x) a.out[__ldg(&meta[v].w)] = x - 1u;
        }
    }
    unsigned long long sums[2];
    for (int q = 0; q < 2; ++q) {
        const unsigned long long s = warp_sum64(q ? frows : relax);
        __syncthreads();
        if (lane == 0) s_part[warp] = s;
        __syncthreads();
        unsigned long long t = 0;
        if (tid == 0)
            for (int w = 0; w < TT / 32; ++w) t += s_part[w];
        sums[q] = warp_sum64(exchange0(t));
    }
    if (lead) {
        RunRes *R = a.res;
        R->verdict = verdict;
        R->witness = witness;
        R->outer = outer;
        R->status = status;
        R->gave_up = 0;
        R->nacc = nacc;
        if (!whole) { // and what k_run had counted
            inner_total += c->inner_total;
            sums[0] += c->relax.v;
            sums[1] += c->frows.v;
            ph_rounds += c->ph_rounds;
            ph_check += c->ph_check;
        }
        R->inner_total = inner_total;
        R->relax = sums[0];
        R->frontier_rows = sums[1];
        R->ph_rounds = ph_rounds;
        R->ph_check = ph_check;
    }
    cluster_barrier(); // no block leaves while another may still write into its shared memory
}

// -------------------------------------------------------- medium graphs --
//
// k_own: the same run over the grid for a whole graph, or the compact graph k_run leaves, of at most OWN_N
// vertices per SM.  Block b owns every gridDim.x-th piece of 32 vertices and keeps their reader ranges, own offers
// and last values in shared memory, and their reader lists too where they fit.  A push is a maximum
// on the reader's word in global memory that nothing waits for; every round the owner reads its share's
// words (coalesced) and pushes for those that changed.  So a round is one coalesced read, the reader ids,
// and the barrier, where k_run's lists take seven dependent accesses (list, state, reader range, reader,
// returning atomic, list position, barrier) and 1.3 us more.  Reading the whole share costs V * 4 bytes a round
// from L2, about 1 us at the largest size.  Rounds over few vertices are bound by that chain (2.3 to 3 us); floods
// by the reductions: an interleaved product of 1.6 M vertices, synchronous, sends 131 M of them in 0.99 ms, 133 G/s,
// the rate at which L2 takes scattered ones.  (Reading the word first, to leave out what raises nothing, took 1.7 ms:
// the loads wait for the reductions on their lines.)  That run took 4.4 ms with the dense start.
//   asynchronous  in[0] / in[1] = the values, by outer iteration mod 2; last = the value pushed last
//   synchronous   in[0] / in[1] = the inboxes, by round mod 2 (as in k_tail); last = the value
constexpr uint32_t OWN_N = 12288;              // vertices per block: 18 bytes of shared memory each
constexpr uint32_t OWN_SMEM = 224 * 1024;      // the rest holds reader lists
constexpr int OWN_U = 4;                       // words read ahead per thread
// asynchronous: looks at the share per round after the first, while it changes (a look is one coalesced read, the
// barrier two dependent accesses through L2 and the wait for the slowest block).  us per run with 0 / 1 / 2 / 3 / 5:
// layered 4 M 1260 / 1174 / 1150 / 1177 / 1185, 2^24 1557 / 1437 / 1387 / 1381 / 1374, 2^26 2641 / 2464 / 2440 / 2444 /
// 2434, random 300,000 395 / 368 / 362 / 366 / 380, interleaved product 6x7 255 / 221 / 204 / 199 / 193
constexpr uint32_t OWN_PASSES = 2;
// asynchronous, more vertices than this to push from: the value is read again just before, since a flood has raised many
// meanwhile, and the older value would be pushed along all of its readers for nothing.  us per run (six iterations of
// the first four) without / with: acyclic graphs of 10^6 vertices and degree 4 3,440 / 2,000, degree 16 10,760 / 3,650
// (dense start 4,900 and 7,580), 1.8 M and degree 8 10,280 / 3,680 (8,430), 500,000 and degree 64 12,500 / 4,600 (14,170);
// interleaved product 7x7 880 / 505, random 10^6 of degree 16 463 / 300.  With few vertices the read is one more access
// in a chain: layered 4 M 1,167 / 1,240 where every value is read again; limit 256 / 512 / 1,024: layered 2^24 1,422 / 1,404 /
// 1,405, acyclic 100,000 of degree 16 1,258 / 1,355 / 1,390, 300,000 of degree 4 1,128 / 1,135 / 1,144
constexpr uint32_t OWN_LIVE = 512;
constexpr uint32_t OWN_HUB = 2048;             // reader lists longer than this are walked by the whole block

struct OwnSmem {
    unsigned long long word;
    uint32_t ok, n, hubs, ebase, xbase;
    uint32_t scan[TT / 32], scan2[TT / 32], mins[TT / 32], sums[TT / 32];
    uint32_t hub[32];
    unsigned long long part[TT / 32];
};

// exclusive prefix of x over the block (TT threads), *total its sum
__device__ __forceinline__ uint32_t own_scan(uint32_t x, uint32_t *s, uint32_t &total)
{
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t incl = warp_inclusive_scan(x);
    __syncthreads(); // (s is free)
    if (lane == 31) s[warp] = incl;
    __syncthreads();
    if (warp == 0) s[lane] = warp_inclusive_scan(s[lane]);
    __syncthreads();
    total = s[TT / 32 - 1];
    return incl - x + (warp ? s[warp - 1] : 0u);
}

// PREP: behind k_prepare, which found the accepting vertices and the entries (a form of its own: asked for at run time it
// took the interleaved product 1.2 % more)
template <bool SYNC, bool BATCH, bool PREP>
__global__ void __launch_bounds__(TT, 1) k_own(const __grid_constant__ RunArgs a, uint32_t whole)
{
    extern __shared__ uint32_t s_mem[];
    __shared__ OwnSmem sh;
    RunCtl *c = a.ctl;
    if (!whole && *(volatile uint32_t *)&c->hand != 1) return; // finished, or left to k_tail (every block returns)
    if (PREP && a.prep[0]) return;                             // k_prepare refused the graph
    const auto nacc0 = [&] { return PREP ? __ldg(a.prep + 1) : a.nacc0; };
    const auto entries_all = [&] { return PREP ? (uint64_t)__ldg(a.prep + 2) : a.m; };
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const bool lead = blockIdx.x == 0 && tid == 0;
    const uint32_t n = a.n, V = whole ? n : *(volatile uint32_t *)&c->V;
    // pieces of 32 vertices go round the blocks (a wave through consecutive vertices is everybody's): the block's
    // vertex i is vertex vid(i)
    const uint32_t pieces = (V + 31) / 32, nb = gridDim.x, full = (pieces + nb - 1) / nb * 32;
    const auto vid = [&](uint32_t i) { return ((i >> 5) * nb + blockIdx.x) * 32 + (i & 31u); };
    const uint32_t my_pieces = pieces > blockIdx.x ? (pieces - blockIdx.x + nb - 1) / nb : 0u;
    const uint32_t mine = my_pieces == 0 ? 0u : my_pieces * 32 - ((pieces - 1) % nb == blockIdx.x ? pieces * 32 - V : 0u);
    const uint32_t stride = full;
    uint32_t *const last = s_mem, *const own = last + stride, *const beg = own + stride, *const end = beg + stride;
    uint16_t *const queue = reinterpret_cast<uint16_t *>(end + stride);
    uint32_t *const s_rc = end + stride + stride / 2;
    const uint32_t rc_room = OWN_SMEM / 4 - (4 * stride + stride / 2);
    uint32_t set = whole ? 1u : *(volatile uint32_t *)&c->set;
    const uint32_t cap = pool_cap(n);
    uint32_t *const ps = pool_set(a, set);
    const uint4 *meta = reinterpret_cast<const uint4 *>(ps);
    const uint32_t *row = ps + 4ull * cap, *rc = whole ? a.rcol : ps + 6ull * cap;
    uint32_t *const in0 = reinterpret_cast<uint32_t *>(a.W), *const in1 = in0 + n;
    // batched, asynchronous: the last even and the last odd round each row was reached in (its graph's relaxation count;
    // the round before is read while this round's pushes come in)
    constexpr bool REACH = BATCH && !SYNC;
    uint32_t *const reach0 = in1 + n, *const reach1 = reach0 + n;
    const uint32_t *const comp = whole ? a.comp : row + cap; // batched: graph of each vertex
    const uint64_t t0 = whole ? global_ns() : *(volatile unsigned long long *)&c->t0;
    uint64_t mark = global_ns(), ph_rounds = 0, ph_check = 0;
    auto phase = [&](uint64_t &acc) {
        const uint64_t now = global_ns();
        if ((int64_t)(now - mark) > 0) {
            acc += now - mark;
            mark = now;
        }
    };
    auto late = [&] { return lead && (int64_t)(global_ns() - t0) > (int64_t)a.timeout_ns; };

    // ---- the share's readers, offers and (where they fit) reader lists
    uint32_t entries = 0; // reader entries of the share so far
    bool cached = true;
    for (uint32_t i0 = 0; i0 < mine; i0 += TT) { // (block-uniform)
        const uint32_t i = i0 + tid;
        uint32_t b = 0, e = 0;
        if (i < mine) {
            const uint32_t v = vid(i);
            uint32_t o;
            if (whole) {
                b = __ldg(a.rrowptr + v);
                e = __ldg(a.rrowptr + v + 1);
                o = ((__ldg(a.acc0 + (v >> 5)) >> (v & 31u)) & 1u) ? v + 1 : 0u;
            } else {
                const uint4 q = __ldg(meta + v);
                b = q.x;
                e = q.y;
                o = q.z;
            }
            last[i] = 0;
            own[i] = o;
            beg[i] = b;
            end[i] = e;
        }
        uint32_t total;
        const uint32_t at = entries + own_scan(e - b, sh.scan, total);
        cached = cached && total <= rc_room - min(rc_room, entries) && entries <= rc_room;
        entries += total; // (a wrapped sum: not cached any more)
        if (cached) { // (a list that no thread copies alone in reasonable time: the warp does)
            for (unsigned m = __ballot_sync(0xFFFFFFFFu, e - b > TAIL_LONG); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const uint32_t bb = __shfl_sync(0xFFFFFFFFu, b, src), ll = __shfl_sync(0xFFFFFFFFu, e - b, src),
                               aa = __shfl_sync(0xFFFFFFFFu, at, src);
                for (uint32_t j = lane; j < ll; j += 32) s_rc[aa + j] = __ldg(rc + bb + j);
            }
            if (e - b <= TAIL_LONG)
                for (uint32_t j = 0; j < e - b; ++j) s_rc[at + j] = __ldg(rc + b + j);
        }
    }
    __syncthreads();
    if (cached) { // ranges into the copy
        uint32_t done = 0;
        for (uint32_t i0 = 0; i0 < mine; i0 += TT) {
            const uint32_t i = i0 + tid, len = i < mine ? end[i] - beg[i] : 0u;
            uint32_t total;
            const uint32_t at = done + own_scan(len, sh.scan, total);
            done += total;
            if (i < mine) {
                beg[i] = at;
                end[i] = at + len;
            }
        }
    }
    if (whole) { // the run's accepting set, and an empty map
        const uint64_t gid = (uint64_t)blockIdx.x * TT + tid, threads = (uint64_t)gridDim.x * TT;
        for (uint64_t i = gid; i < a.words; i += threads) a.acc[i] = __ldg(a.acc0 + i);
        if (BATCH && a.out) // (graphs end in different iterations)
            for (uint64_t i = gid; i < n; i += threads) a.out[i] = NONE;
    }
    __syncthreads();

    uint32_t outer = whole ? 0u : *(volatile uint32_t *)&c->outer, nacc = whole ? nacc0() : *(volatile uint32_t *)&c->nacc;
    uint32_t status = ST_OK, verdict = 0, witness = NONE, seq = 0, gate = a.tail_cap / 2;
    unsigned long long relax = 0, frows = 0, inner_total = 0, total = 0;
    bool go = nacc != 0, alive = true, hand = false;
    // a frontier row of n entries: to the relaxation count (batched: of its graph g); the whole warp calls it
    const auto count_row = [&](bool is, uint32_t len, uint32_t g) {
        if (is) {
            relax += len;
            ++frows;
        }
        if constexpr (BATCH) {
            const uint32_t k = is ? g : NONE, l = is ? len : 0u;
            const unsigned same = __match_any_sync(0xFFFFFFFFu, k);
            const unsigned lo = __reduce_add_sync(same, l & 0xFFFFu), hi = __reduce_add_sync(same, l >> 16);
            const unsigned long long sum = (unsigned long long)lo + ((unsigned long long)hi << 16);
            if (k != NONE && lane == (unsigned)(__ffs(same) - 1) && sum)
                atomicAdd((unsigned long long *)&a.cs[k].relax, sum);
        }
    };
    const auto reader = [&](uint32_t j) { return cached ? s_rc[j] : __ldg(rc + j); };
    while (go) {
        ++outer;
        uint32_t *const val = (outer & 1) ? in1 : in0; // (asynchronous)
        if (lead && (SYNC || !a.count_round1)) relax += entries_all(); // round 1 covers every row
        uint32_t r = 0;
        for (;;) {
            ++r;
            uint32_t *const inbox = (r & 1) ? in0 : in1; // what came in round r - 1 (synchronous)
            uint32_t *const to = SYNC ? ((r & 1) ? in1 : in0) : val;
            const auto push = [&](uint32_t w, uint32_t o) {
                atomicMax(to + w, o);
                if (REACH) atomicMax(((r & 1) ? reach1 : reach0) + w, r);
            };
            const bool pushes = r <= a.max_inner; // (past the limit the last round's values are only taken)
            uint32_t hits = 0;
            for (uint32_t pass = 0;; ++pass) { // (asynchronous: the share once more, a few times while it changes)
                if (tid == 0) sh.n = sh.hubs = 0;
                __syncthreads();
                const bool start = r == 1 && pass == 0;
                const uint32_t *const words = SYNC ? inbox : val;
                for (uint32_t i0 = 0; i0 < mine; i0 += TT * OWN_U) { // (block-uniform) OWN_U words in flight per thread
                    uint32_t y[OWN_U], f[OWN_U];
#pragma unroll
                    for (int k = 0; k < OWN_U; ++k) {
                        const uint32_t i = i0 + k * TT + tid;
                        y[k] = i >= mine ? 0u : start ? own[i] : __ldcg(words + vid(i));
                        if (REACH) f[k] = i >= mine || pass || r <= 2 ? 0u : __ldcg(((r & 1) ? reach0 : reach1) + vid(i));
                    }
#pragma unroll
                    for (int k = 0; k < OWN_U; ++k) {
                        const uint32_t i = i0 + k * TT + tid;
                        if (i0 + k * TT >= mine) break; // (block-uniform)
                        const unsigned some = __ballot_sync(0xFFFFFFFFu, y[k] != 0);
                        if (!some) continue; // (warp-uniform: nothing here)
                        bool hit = y[k] != 0;
                        if (!start) {
                            const uint32_t v = vid(i), g = BATCH && hit ? __ldg(comp + v) : NONE;
                            if (SYNC && i < mine) inbox[v] = 0; // (whole lines)
                            if ((SYNC || REACH) && r > 2) { // frontier rows of round r - 1
                                const bool is = SYNC ? hit : f[k] == r - 1;
                                uint32_t len = 0;
                                if (is) len = whole ? __ldg(a.rowptr + v + 1) - __ldg(a.rowptr + v) : __ldg(row + v);
                                count_row(is, len, g);
                            }
                            hit = hit && y[k] > last[i];
                            if (hit) last[i] = y[k];
                            if constexpr (BATCH) { // the graphs that changed in round r - 1
                                const unsigned same = __match_any_sync(0xFFFFFFFFu, hit ? g : NONE);
                                if (hit && lane == (unsigned)(__ffs(same) - 1) && *(volatile uint32_t *)&a.cs[g].last_change < r - 1)
                                    atomicMax(&a.cs[g].last_change, r - 1);
                            }
                        }
                        const unsigned m = __ballot_sync(0xFFFFFFFFu, hit);
                        if (!m) continue;
                        uint32_t at = 0;
                        if (lane == 0) at = atomicAdd(&sh.n, (uint32_t)__popc(m));
                        at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(m & ((1u << lane) - 1u));
                        if (hit) queue[at] = (uint16_t)i;
                    }
                }
                __syncthreads();
                const uint32_t nq = sh.n;
                hits += nq;
                if (!nq || !pushes) break;
                for (uint32_t q0 = 0; q0 < nq; q0 += TT) { // (block-uniform)
                    const uint32_t q = q0 + tid;
                    uint32_t o = 0, b = 0, e = 0;
                    if (q < nq) {
                        const uint32_t i = queue[q];
                        if (!SYNC && !start && nq > OWN_LIVE) last[i] = max(last[i], __ldcg(val + vid(i)));
                        o = start ? own[i] : max(last[i], own[i]);
                        b = beg[i];
                        e = end[i];
                        if (!SYNC && !BATCH) {
                            if (r > 1 || pass || a.count_round1) relax += e - b;
                            if (r > 1) ++frows;
                        }
                        if (e - b > OWN_HUB) { // the whole block's, below (the first 32 of a pass)
                            const uint32_t h = atomicAdd(&sh.hubs, 1u);
                            if (h < 32) {
                                sh.hub[h] = i;
                                b = e;
                            }
                        }
                    }
                    for (unsigned m = __ballot_sync(0xFFFFFFFFu, e - b > TAIL_LONG); m; m &= m - 1) {
                        const int src = __ffs(m) - 1;
                        const uint32_t ob = __shfl_sync(0xFFFFFFFFu, o, src), bb = __shfl_sync(0xFFFFFFFFu, b, src),
                                       ll = __shfl_sync(0xFFFFFFFFu, e - b, src);
#pragma unroll 4
                        for (uint32_t j = lane; j < ll; j += 32) push(reader(bb + j), ob);
                        if ((int)lane == src) b = e;
                    }
                    for (uint32_t j = 0; j < e - b; j += 4) { // up to four readers in flight
                        uint32_t w[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) w[k] = j + k < e - b ? reader(b + j + k) : NONE;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (w[k] != NONE) push(w[k], o);
                    }
                }
                __syncthreads();
                for (uint32_t h = 0; h < min(sh.hubs, 32u); ++h) {
                    const uint32_t i = sh.hub[h], b = beg[i], ll = end[i] - b;
                    const uint32_t o = start ? own[i] : max(last[i], own[i]);
#pragma unroll 4
                    for (uint32_t j = tid; j < ll; j += TT) push(reader(b + j), o);
                }
                __syncthreads(); // (the queue and the hubs are read)
                if (SYNC || BATCH || pass >= max(a.lc_passes, OWN_PASSES)) break;
            }
            alive = run_barrier(c, c->obar, sh, seq, (unsigned long long)hits + ((r & 3u) == 0 && late() ? RUN_STOP : 0ull), total);
            if (!alive) break;
            if (r == 1) continue; // (the limit and the end of the rounds: once round 1's values are taken)
            if (total & RUN_STOP) status = ST_TIMEOUT;
            else if ((total & RUN_COUNT) && !pushes) status = ST_LIMIT;
            if (!(total & RUN_COUNT) || status != ST_OK) break;
        }
        if (!alive) break;
        const uint32_t rounds = status == ST_TIMEOUT ? r : r - 1;
        inner_total += rounds;
        if (lead) {
            if (outer - 1 < a.hist_cap) a.hist[outer - 1] = rounds;
            if (outer - 1 < RUN_HIST) a.res->hist[outer - 1] = rounds;
            phase(ph_rounds);
        }
        if (!BATCH && status != ST_OK) break;
        // ---- self-map test and elimination (last[] holds the values)
        uint32_t wit = NONE, elim = 0, have = 0, settled = 0;
        for (uint32_t i0 = 0; i0 < mine; i0 += TT) {
            const uint32_t i = i0 + tid, x = i < mine ? last[i] : 0u;
            const uint32_t g = BATCH && x ? __ldg(comp + vid(i)) : NONE;
            uint32_t removed = 0;
            if (x) {
                ++have;
                if (status == ST_OK && x - 1 == (whole ? vid(i) : __ldg(&meta[vid(i)].w))) {
                    wit = min(wit, x - 1);
                    if (BATCH) atomicMin(&a.cs[g].witness, x - 1);
                }
            }
            const unsigned same = __match_any_sync(0xFFFFFFFFu, x); // (many vertices share a few values)
            if (x && x != settled && status == ST_OK && lane == (unsigned)(__ffs(same) - 1)) {
                const uint32_t u = x - 1, bit = 1u << (u & 31u);
                if ((__ldcg(a.acc + (u >> 5)) & bit) && (atomicAnd(a.acc + (u >> 5), ~bit) & bit)) removed = 1;
            }
            elim += removed;
            settled = x;
            if constexpr (BATCH) { // per graph: vertices with a value and removals, one atomic per graph in the warp
                const unsigned like = __match_any_sync(0xFFFFFFFFu, g);
                const unsigned ne = __reduce_add_sync(like, removed);
                if (g != NONE && lane == (unsigned)(__ffs(like) - 1)) {
                    atomicAdd(&a.cs[g].touched, (unsigned)__popc(like));
                    if (ne) atomicAdd(&a.cs[g].elim, ne);
                }
            }
        }
        wit = __reduce_min_sync(0xFFFFFFFFu, wit);
        elim = __reduce_add_sync(0xFFFFFFFFu, elim);
        have = __reduce_add_sync(0xFFFFFFFFu, have);
        if (lane == 0) {
            sh.mins[warp] = wit;
            sh.sums[warp] = elim;
            sh.scan[warp] = have;
        }
        __syncthreads();
        if (tid < 32) {
            wit = __reduce_min_sync(0xFFFFFFFFu, sh.mins[tid]);
            elim = __reduce_add_sync(0xFFFFFFFFu, sh.sums[tid]);
            have = __reduce_add_sync(0xFFFFFFFFu, sh.scan[tid]);
        }
        if (tid == 0) {
            if (wit != NONE) atomicMax(&c->witness.v, NONE - wit);
            if (have) atomicAdd(&c->ocnt[outer & 1].v, have);
            if (lead) *(volatile uint32_t *)&c->ocnt[(outer + 1) & 1].v = 0;
        }
        alive = run_barrier(c, c->obar, sh, seq,
                            (unsigned long long)elim + (wit != NONE ? RUN_FOUND : 0ull) + (late() ? RUN_STOP : 0ull), total);
        if (!alive) break;
        const uint32_t T = *(volatile uint32_t *)&c->ocnt[outer & 1].v;
        if (lead) phase(ph_check);
        if constexpr (BATCH) {
            if (status == ST_OK && (total & RUN_STOP)) status = ST_TIMEOUT;
            uint32_t left;
            bool limit;
            for (uint32_t i = tid; a.out && i < mine; i += TT) { // the maps of the graphs that end here
                const uint32_t x = last[i], v = vid(i);
                if (!x) continue;
                const uint32_t g = __ldg(comp + v);
                if (!comp_goes_on(a.cs[g], status, a.max_outer, left, limit))
                    a.out[whole ? v : __ldg(&meta[v].w)] = x - 1u - *(volatile uint32_t *)&a.cs[g].off;
            }
            if (!(alive = run_barrier(c, c->obar, sh, seq, 0, total))) break;
            const uint32_t on = blockIdx.x == 0 ? end_graphs(a, status, sh.sums) : 0u;
            if (!(alive = run_barrier(c, c->obar, sh, seq, on, total))) break;
            if (!(total & RUN_COUNT)) go = false;
        } else if (total & (RUN_STOP - RUN_FOUND)) {
            verdict = 1;
            witness = NONE - *(volatile uint32_t *)&c->witness.v;
            go = false;
        } else if (T == 0) {
            go = false; // nothing reaches a remaining accepting vertex
        } else {
            nacc -= (uint32_t)(total & RUN_COUNT);
            if (nacc == 0) go = false;
            else if ((a.max_outer && outer >= a.max_outer) || outer > nacc0()) {
                status = ST_LIMIT;
                go = false;
            } else if (total & RUN_STOP) {
                status = ST_TIMEOUT;
                go = false;
            }
        }
        if (!go) break;
        // ---- the next iteration: eliminated vertices offer nothing, values back to none
        const bool pack = !BATCH && T <= gate;
        const uint32_t lim = min(a.tail_cap, cap);
        const uint64_t ecap = min((uint64_t)n * 3 / 4 - 8, (uint64_t)a.tail_m);
        uint32_t *const ps2 = pool_set(a, set ^ 1);
        uint4 *const meta2 = reinterpret_cast<uint4 *>(ps2);
        uint32_t *const row2 = ps2 + 4ull * cap, *const rc2 = ps2 + 6ull * cap;
        bool over = false;
        for (uint32_t i0 = 0; i0 < mine; i0 += TT) { // (block-uniform)
            const uint32_t i = i0 + tid;
            uint32_t x = 0, o = 0, len = 0;
            if (i < mine) {
                x = last[i];
                o = own[i];
                if (o && (!((__ldcg(a.acc + ((o - 1) >> 5)) >> ((o - 1) & 31u)) & 1u) ||
                          (BATCH && !*(volatile uint32_t *)&a.cs[__ldg(comp + vid(i))].active)))
                    own[i] = o = 0;
                len = end[i] - beg[i];
                if (!SYNC && x) val[vid(i)] = 0; // (the next iteration's pushes go to the other array)
                if (REACH && x) reach0[vid(i)] = reach1[vid(i)] = 0;
                last[i] = 0;
            }
            if (!pack) continue;
            // compaction into the graph of the vertices that had a value and the accepting ones, as in k_run
            const bool member = x != 0 || (o != 0 && len != 0);
            uint32_t nm, ne;
            const uint32_t at = own_scan(member ? 1u : 0u, sh.scan, nm), ea = own_scan(member ? len : 0u, sh.scan2, ne);
            if (tid == 0) {
                sh.xbase = nm ? atomicAdd(&c->xcnt.v, nm) : 0u;
                sh.ebase = ne ? atomicAdd(&c->ecnt.v, ne) : 0u;
            }
            __syncthreads();
            const uint32_t xb = sh.xbase, eb = sh.ebase;
            if ((uint64_t)xb + nm > lim || (uint64_t)eb + ne > ecap) over = true;
            if (member && !over) {
                const uint32_t v = vid(i), id = whole ? v : __ldg(&meta[v].w), k = xb + at;
                meta2[k] = make_uint4(eb + ea, eb + ea + len, o, id);
                if (SYNC) row2[k] = whole ? __ldg(a.rowptr + v + 1) - __ldg(a.rowptr + v) : __ldg(row + v);
                a.rank[id] = k + 1;
                last[i] = k + 1; // (for the reader lists below)
            }
            __syncthreads(); // (the bases are read)
        }
        if (!pack) continue;
        alive = run_barrier(c, c->obar, sh, seq, over ? 1u : 0u, total);
        if (!alive) break;
        const uint32_t V2 = *(volatile uint32_t *)&c->xcnt.v;
        const bool fits = (total & RUN_COUNT) == 0;
        for (uint32_t i0 = 0; i0 < mine; i0 += TT) {
            const uint32_t i = i0 + tid, k = i < mine ? last[i] : 0u;
            uint32_t b = 0, e = 0, at = 0;
            if (fits && k) {
                b = beg[i];
                e = end[i];
                at = meta2[k - 1].x;
            }
            if (i < mine) last[i] = 0;
            auto number = [&](uint32_t w) { return __ldcg(a.rank + (whole ? w : __ldg(&meta[w].w))) - 1; };
            for (unsigned m = __ballot_sync(0xFFFFFFFFu, e - b > TAIL_LONG); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const uint32_t bb = __shfl_sync(0xFFFFFFFFu, b, src), ll = __shfl_sync(0xFFFFFFFFu, e - b, src),
                               aa = __shfl_sync(0xFFFFFFFFu, at, src);
                for (uint32_t j = lane; j < ll; j += 32) rc2[aa + j] = number(reader(bb + j));
                if ((int)lane == src) b = e;
            }
            for (uint32_t j = 0; j < e - b; ++j) rc2[at + j] = number(reader(b + j));
        }
        if (fits) {
            if (lead) {
                c->V = V2;
                c->set = set ^ 1;
            }
            hand = true;
            break;
        }
        // too many vertices or readers: try again once half as many have a value
        gate = min(gate, T) / 2;
        alive = run_barrier(c, c->obar, sh, seq, 0, total); // (every block has read the counts)
        if (!alive) break;
        if (lead) *(volatile uint32_t *)&c->xcnt.v = *(volatile uint32_t *)&c->ecnt.v = 0;
    }
    // ---- the map of the last iteration; the state back to zero
    if (alive && !hand) {
        uint32_t *const val = (outer & 1) ? in1 : in0;
        for (uint32_t i = tid; i < mine; i += TT) {
            uint32_t x = last[i];
            if (SYNC) {
                if (status != ST_OK) in0[vid(i)] = in1[vid(i)] = 0; // (at the fix-point the inboxes are empty)
            } else {
                if (status != ST_OK) x = max(x, __ldcg(val + vid(i)));
                if (x) val[vid(i)] = 0;
                if (REACH && x) reach0[vid(i)] = reach1[vid(i)] = 0;
            }
            if (!BATCH && a.out) {
                if (whole) a.out[vid(i)] = x - 1u; // (no value: MAP_NONE)
                else if (x) a.out[__ldg(&meta[vid(i)].w)] = x - 1u;
            }
        }
    } else if (hand && whole && a.out) { // k_tail writes the values of the last iteration over this
        for (uint32_t i = tid; i < mine; i += TT) a.out[vid(i)] = NONE;
    }
    for (int q = 0; q < 2; ++q) {
        const unsigned long long s = warp_sum64(q ? frows : relax);
        __syncthreads();
        if (lane == 0) sh.part[warp] = s;
        __syncthreads();
        if (tid == 0) {
            unsigned long long t = 0;
            for (int w = 0; w < TT / 32; ++w) t += sh.part[w];
            if (t) atomicAdd(q ? &c->frows.v : &c->relax.v, t);
        }
    }
    if (alive) alive = run_barrier(c, c->obar, sh, seq, 0, total);
    if (!lead) return;
    if (!whole) { // and what k_run had counted
        inner_total += c->inner_total;
        ph_rounds += c->ph_rounds;
        ph_check += c->ph_check;
    }
    if (hand && alive) { // (after a wait that gave up the reader lists may be unwritten: nothing is left to k_tail)
        c->outer = outer;
        c->nacc = nacc;
        c->inner_total = inner_total;
        c->ph_rounds = ph_rounds;
        c->ph_check = ph_check;
        c->t0 = t0;
        c->hand = 2;
        return;
    }
    RunRes *R = a.res;
    R->verdict = verdict;
    R->witness = witness;
    R->outer = outer;
    R->status = alive ? status : ST_TIMEOUT;
    R->gave_up = alive ? 0u : 1u;
    R->nacc = nacc;
    R->inner_total = inner_total;
    R->relax = *(volatile unsigned long long *)&c->relax.v;
    R->frontier_rows = *(volatile unsigned long long *)&c->frows.v;
    R->ph_rounds = ph_rounds;
    R->ph_check = ph_check;
    if (!whole) c->hand = 0;
}

// Set-up of a small graph in one cluster (before k_tail): bounds and validity of the CSR, the accepting set
// and its size, and the readers (reverse CSR).  Entry i holding u goes to slot start(u) + the count its
// increment of u's in-degree returned; the row of an entry is found by binary search, so that a row of any
// length is spread over all threads.  Replaces eight launches, five memsets and two stream waits: at 1,000
// vertices they were most of map_run_static's 490 us (107 now).
// (rowptr and colidx by plain loads: in place, they are written here too.)
// prep: (0 = good, 1 = rowptr[0] != 0, 2 = more than max_m entries, 3 = invalid), accepting vertices, entries,
// rowptr[0], whether some row holds two entries or more, entries that hold an accepting vertex; rank: m words;
// cnt: n + 1 words, becomes rrowptr.  FULL (map_create): also the handle's copies of rowptr and colidx (with the
// accepting flag in bit 31; they may be the inputs themselves) and the reader entries' positions; there max_m is
// the number of entries, which the host has read already, and the inputs may lie across the link: each word of them
// is read once.
struct PrepareOut {
    uint32_t *rowptr, *colidx, *rpos;
};
template <bool FULL>
__global__ void __launch_bounds__(TT, 1)
    k_prepare(uint32_t n, const uint32_t *rowptr, const uint32_t *colidx, const uint32_t *acc_in, uint32_t max_m,
              uint32_t *acc0, uint32_t *cnt, uint32_t *rcol, uint32_t *rank, uint32_t *prep, PrepareOut out)
{
    __shared__ uint32_t s_warp[TT / 32], s_part[TAIL_C], s_bad, s_acc, s_ent;
    const uint32_t C = gridDim.x, me = cluster_rank(), tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const uint32_t gid = me * TT + tid, threads = C * TT;
    const uint32_t r0 = FULL ? 0u : rowptr[0], m = FULL ? max_m : rowptr[n];
    if (r0 != 0 || m > max_m) { // (every block)
        if (gid == 0) {
            prep[0] = r0 != 0 ? 1u : 2u;
            prep[1] = 0;
            prep[2] = m;
            prep[3] = r0;
        }
        return;
    }
    if (tid == 0) s_bad = s_acc = s_ent = 0;
    cluster_barrier();
    uint32_t bad = 0, na = 0, ne = 0; // (bad: bit 0 invalid, bit 1 a row of two entries or more)
    for (uint32_t i = gid; i <= n; i += threads) cnt[i] = 0;
    for (uint32_t i0 = gid - lane; i0 <= n; i0 += threads) { // (a lane's row end comes from the next lane)
        const uint32_t i = i0 + lane, b = i <= n ? rowptr[i] : 0u;
        uint32_t e = __shfl_down_sync(0xFFFFFFFFu, b, 1);
        if (lane == 31 && i < n) e = rowptr[i + 1];
        if (i < n) bad |= (b > e ? 1u : 0u) | (e - b > 1u ? 2u : 0u);
        if (FULL && i <= n) out.rowptr[i] = b; // (in place, the same word)
    }
    const uint32_t words = (n + 31) / 32;
    for (uint32_t i = gid; i < words; i += threads) {
        uint32_t x = __ldg(acc_in + i);
        if (i == words - 1 && (n & 31u)) x &= (1u << (n & 31u)) - 1u;
        acc0[i] = x;
        na += __popc(x);
    }
    cluster_barrier(); // the counts are zero
    // (U entries in flight per thread, here and in the scatter: map_create of 32,768 vertices with 131,072 entries
    // took 86 us with one, 76 with four)
    constexpr int U = 4;
    for (uint32_t i0 = gid; i0 < m; i0 += U * threads) {
        uint32_t u[U], at[U], flag[U];
#pragma unroll
        for (int j = 0; j < U; ++j) u[j] = i0 + j * threads < m ? colidx[i0 + j * threads] : 0u;
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const bool in = i0 + j * threads < m && u[j] < n;
            at[j] = in ? atomicAdd(cnt + u[j] + 1, 1u) : 0u;
            flag[j] = FULL && in ? (__ldg(acc_in + (u[j] >> 5)) >> (u[j] & 31u)) & 1u : 0u;
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const uint32_t i = i0 + j * threads;
            if (i >= m) break;
            bad |= u[j] >= n ? 1u : 0u;
            rank[i] = at[j];
            ne += flag[j];
            if (FULL) out.colidx[i] = u[j] | flag[j] << 31;
        }
    }
    // an invalid input to every block, the counts to block 0
    const auto add = [&](uint32_t *to, uint32_t x) {
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(cluster_addr(shared_addr(to), 0)), "r"(x)
                     : "memory");
    };
    bad = __reduce_or_sync(0xFFFFFFFFu, bad);
    na = __reduce_add_sync(0xFFFFFFFFu, na);
    ne = __reduce_add_sync(0xFFFFFFFFu, ne);
    if (lane == 0) {
        for (uint32_t q = 0; q < ((bad & 1u) ? C : bad ? 1u : 0u); ++q) cluster_or(cluster_addr(shared_addr(&s_bad), q), bad);
        if (na) add(&s_acc, na);
        if (ne) add(&s_ent, ne);
    }
    cluster_barrier(); // the counts are complete
    // inclusive scan of cnt[0 .. n]: a contiguous share per block
    const uint32_t len = n + 1, share = (len + C - 1) / C, b = min(len, me * share), e = min(len, b + share);
    uint32_t sum = 0;
    for (uint32_t i = b + tid; i < e; i += TT) sum += __ldcg(cnt + i);
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) s_warp[warp] = sum;
    __syncthreads();
    if (tid < 32) {
        const uint32_t t = __reduce_add_sync(0xFFFFFFFFu, s_warp[tid]);
        if (tid < C)
            asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(shared_addr(&s_part[me]), tid)),
                         "r"(t)
                         : "memory");
    }
    cluster_barrier();
    uint32_t run = 0;
    for (uint32_t q = 0; q < me; ++q) run += s_part[q];
    for (uint32_t i0 = b; i0 < e; i0 += TT) { // (block-uniform)
        const uint32_t i = i0 + tid;
        uint32_t x = warp_inclusive_scan(i < e ? __ldcg(cnt + i) : 0u);
        __syncthreads(); // s_warp is free
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        if (warp == 0) {
            const uint32_t w = s_warp[lane], incl = warp_inclusive_scan(w);
            s_warp[lane] = incl;
        }
        __syncthreads();
        if (warp) x += s_warp[warp - 1];
        if (i < e) cnt[i] = run + x;
        run += s_warp[TT / 32 - 1];
    }
    if (gid == 0) {
        prep[0] = (s_bad & 1u) ? 3u : 0u;
        prep[1] = s_acc;
        prep[2] = m;
        prep[3] = 0;
        prep[4] = s_bad >> 1;
        prep[5] = s_ent;
    }
    cluster_barrier(); // the starts are in place
    if (s_bad & 1u) return; // (the same in every block; nobody's shared memory is read from here on)
    const uint32_t *const rows = FULL ? out.rowptr : rowptr, *const cols = FULL ? out.colidx : colidx;
    for (uint32_t i0 = gid; i0 < m; i0 += U * threads) {
        uint32_t slot[U], lo[U], left = n; // rows[lo] <= i < rows[lo + left]
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const uint32_t i = min(i0 + j * threads, m - 1);
            slot[j] = __ldcg(cnt + (cols[i] & 0x7FFFFFFFu)) + rank[i];
            lo[j] = 0;
        }
        while (left > 1) { // (the same steps for all: where left is odd, its larger half stays)
            const uint32_t half = left >> 1;
#pragma unroll
            for (int j = 0; j < U; ++j) lo[j] += rows[lo[j] + half] <= min(i0 + j * threads, m - 1) ? half : 0u;
            left -= half;
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const uint32_t i = i0 + j * threads;
            if (i >= m) break;
            rcol[slot[j]] = lo[j];
            if (FULL) out.rpos[slot[j]] = i;
        }
    }
}

} // namespace mapk
