// rcm_engine_state.cuh -- what the device-side engines share: constants, the arguments of one ordering
// (EngineArgs) and the shared memory of one engine CTA (EngineSmem).
#pragma once

#include "rcm_internal.cuh"

namespace rcm {

constexpr int kEllNb = 7;       // neighbours stored in a vertex's 32-byte row; slot 7 = degree
constexpr int kCache = 2048;    // frontier ids cached in shared memory per buffer
constexpr int kTinyMax = 32;    // components of at most this many vertices are ordered by one thread
constexpr int kWarpLevel = 32;  // narrow levels of at most this many vertices run on warp 0 alone
// A level of a few hundred vertices that holds a hub is far more work than one CTA does quickly,
// and a labelled first sweep over hubs costs more than a levels-only one: graphs with a vertex of
// more than kHubDegree neighbours take a lower frontier switch and levels-only first sweeps by
// default (24 -> 11.3 ms a call on a 1M-vertex power-law graph with hubs of 7,000 entries). Where their rows
// hold one entry in kHubShare or more, the whole-grid levels also spread long rows over a CTA's warps
// (Engine::hub_round: 6.7 ms); a few dense rows in a grid do not pay for its barriers in every round (a 192^3
// grid with one row of 600 entries 5.02 ms without, 5.66 with).
constexpr int kHubDegree = 512;
constexpr int kHubShare = 1024;
// Patterns this sparse may fall into parts: 2-nearest-neighbour meshes and their spanning trees have
// 2.7 neighbours a row, 3-nearest ones 3.7, grids 4 and 6. The probe sweep from the first start vertex runs
// one part while everything else waits (1.2M-point mesh in 20 strips 9.6 ms with it, 8.0 without); the
// component table costs a pass of union-find, 0.3 ms per million vertices. Trees, cubic and other sparse random
// graphs are as sparse, but connected and low, and the table is lost on them. So the probe runs, and gives
// up for the table where level kProbeLevels is still narrow and 3/4 of the vertices are not reached yet
// (0.05 ms of the strips' 8.0; a 50,000-vertex cubic graph, which finishes it, 0.24 ms, and 0.43 with the table).
constexpr int kPartsDegree = 32;
constexpr int kProbeLevels = 32;
// Levels of up to this many vertices are one CTA's work: a 50,000-vertex path 72 ms on 256 threads, 84 on
// CTA 0 of the grid; a 260^2 grid with its edges halved 5.6 and 5.1.
constexpr int kThinLevel = 8;
// Of a component table the grid keeps what holds 3/4 of the vertices left, from this size on (below it one
// CTA is the faster, as for whole graphs): a cubic graph of 200,000 vertices 0.28 ms on the grid, 14.8 on one
// CTA, a random tree 1.0 and 26, the giant component of a sparse random graph 1.1 and 39.
constexpr int kGridMin = 4609;
constexpr int kHubNarrow = 128;
constexpr unsigned long long kClaimNone = ~0ull;

struct EngineArgs {
    int n;                       // vertices of this graph
    int v0;                      // global id of its first vertex (rows hold global ids)
    const int* rowptr;           // global rows (overflow neighbours of rows with degree > 7)
    const int4* ell;             // 2 x int4 per vertex: 7 sorted neighbours (its own id where absent) + degree
    const int* adj;              // full sorted rows, valid for rows with degree > 7
    const int* deg;              // global
    unsigned long long* claim;   // global, 64-bit keys (kClaimNone = not reached)
    int* vis;                    // global sweep stamps
    int* qa;                     // this graph's queue / staging buffer (n ints)
    int* qb;                     // this graph's queue / staging buffer (n ints)
    int* boff;                   // this graph's per-frontier offsets (n ints)
    int* perm;                   // this graph's output segment (n ints); global ids while running
    Ctl* ctl;                    // grid control block (whole-grid executor only)
    int* status;                 // where device-detected error bits are ORed
    int* diag;                   // optional (may be null): first failed guard's site and value
    int narrow_thr;
    int fused;
    int cc_first;                // persistent grid: build the component table before the first sweep (-1: where
                                 // the rows average fewer than kPartsDegree / 10 neighbours and the probe gives up)
    int hubs;                    // whole grid: rows of more than kHubDegree neighbours hold one entry in kHubShare
                                 // or more (set on the device)
    int hub_auto;                // default launch of the persistent grid: a graph with a vertex of more
                                 // than kHubDegree neighbours takes the frontier switch kHubNarrow and
                                 // levels-only first sweeps (decided on the device from ctl->maxdeg)
    int obits;                   // low bits of a key holding the in-level order
    int profile;                 // accumulate per-phase time (CTA 0, thread 0)
    int probe;                   // whole grid: a level at which a sweep that is still narrow gives up (0 = none; set
                                 // on the device)
    long long limit_ns;
    // concurrent components (whole-grid executor only)
    int* cc_parent;              // n ints
    int* cc_size;                // n ints (indexed by root)
    unsigned long long* cc_key;  // n keys (indexed by root)
    int* cc_roots;               // cc_cap ints
    unsigned long long* cc_gkey; // next_pow2(cc_cap) keys (sort scratch beyond shared memory)
    int* cc_gidx;                // next_pow2(cc_cap) ints
    int4* cc_tab;                // cc_cap entries: (start vertex, first label, size, root)
    int cc_cap;                  // most components ordered concurrently (else one by one)
    int cc_big;                  // components at least this large run on the whole grid
    // bottom-up expansion (whole-grid executor only; fkey == null: top-down only)
    unsigned long long* fkey;    // n words: a labelled frontier vertex's key, published for bottom-up claims
    int expand_mode;             // 2 = bottom-up on every grid level, 1 = top-down, else per level by frontier size
    int bu_divisor;              // per level: bottom-up once the frontier holds n / bu_divisor vertices
    // asynchronous levels-only sweeps (whole-grid executor only; adist == null: level by level)
    unsigned long long* adist;   // n words: (~sweep stamp) << 32 | breadth-first distance
    unsigned long long* aq;      // work queue of aq_cap (distance << 32 | vertex) items
    AsyncCtl* actl;
    unsigned aq_cap;
    // middle tier (whole-grid executor launched in clusters of mid_k CTAs; 0 = off): labelled
    // levels of narrow_thr <= size < mid_thr run on cluster 0 alone, exchanging through
    // distributed shared memory, while the other CTAs wait at the next grid barrier
    int mid_k;
    int mid_thr;
    // narrow labelled levels of the whole-grid executor with their state in CTA 0's shared memory
    // (rcm_local.cuh); local_hi = 0: in global memory
    int local_hi;                // a run ends at a level of this many vertices (narrow_thr starts one)
    int local_slots, local_entries;
    unsigned* gvis;              // bitmap of n vertices: what the grid's levels visited, for the next run
};

enum { kPhExpand = 0, kPhClaim, kPhOwn, kPhLabels, kPhExchange, kPhRedist, kPhWaitNarrow, kPhOther };

// The shared-memory state of a CTA engine's local sweeps; cap = 0: none (sweeps run in global memory).
struct LocalState {
    int cap;             // vertices of the largest graph the bitmap and the packed words hold
    int idbits;          // bits of a packed word that hold a vertex or a frontier position
    int slots;           // hash slots, a power of two (direct claims: one per vertex, no keys)
    unsigned* vis;       // cap / 32 words, 16-byte aligned
    unsigned* hkey;      // (generation << idbits) | vertex; generation 0 = never used
    unsigned* hval;      // ((gmax - generation) << idbits) | smallest frontier position
    unsigned gen;        // generation of the last labelled level
    unsigned seq;        // labelled sweeps so far (tags the global claims)
    unsigned* list;      // the warps' lists of unvisited neighbours, qcap entries each
    int qcap;
    int wc[32];          // per-warp child counts
    int rest;            // vertices of the level at which the last sweep went on in global memory (0 = it did not)
};

// Shared memory of one engine CTA.
struct EngineSmem {
    EngineArgs args;
    long long st[8];             // statistics (rcm_stats order), updated by thread 0
    long long prof[8];           // per-phase ns (profile), updated by thread 0 of CTA 0
    unsigned long long prof_t;   // timestamp of the last phase boundary
    int scan[64];
    int acc_cnt;                 // CTA count accumulator feeding the exchange
    unsigned long long wkey[32]; // per-warp min keys of the last accumulate()
    int ex[4];                   // exchange results: total, pre, maxcnt
    int exc[2][4];               // the counts-only exchange's, by epoch parity (and bad)
    unsigned long long ex_key;
    int bc[8];
    unsigned long long bck;
    int tail;
    int ntail[3];                // narrow levels-only loop: new-vertex counters, by level mod 3
    struct {                     // state after a run of warp-0 levels, read by the whole CTA
        int F, d, lstart, cb, lastF, bad, qb;
        long long reached;
        unsigned long long lk;
    } wr;
    struct {                     // an out-of-line sweep of the grid: the engine's counters, and its results
        unsigned epoch, cepoch;
        int sweep_id, scan_par, ecc, size, prev_start;
        bool async_ok;
        unsigned char fused;     // args.fused after a probe
        unsigned long long key;
        long long reached;
    } sw;
    int aflag;                   // async sweep: stop flag relayed to the CTA's warps
    // middle tier: this CTA's part of each cluster exchange, read by the cluster's CTAs through
    // distributed shared memory; double-buffered by epoch parity
    unsigned long long xc_flag[2];  // (epoch << 32) | count, released at cluster scope
    unsigned long long xc_key[2];   // min (degree, id) key of the CTA's slice
    LocalState loc;
    int* hub;                    // one int per thread: a round's values by element (Engine::hub_round)
    int cache[2][kCache];
};

enum { kStComponents = 0, kStSweeps, kStTraversals, kStLevels, kStMaxEcc, kStIsolated, kStNarrow, kStGrid };

}  // namespace rcm
