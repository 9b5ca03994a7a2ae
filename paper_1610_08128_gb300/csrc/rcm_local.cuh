// rcm_local.cuh -- one CTA's sweeps over one graph with the traversal state in shared memory.
//
// A CTA engine's level is a chain of dependent steps, and with the state in global memory most of
// them are L2 round trips: the frontier's rows, the claims' atomics, the claims read back. Here only
// the rows come from global memory; everything a level writes and reads back stays on the SM:
//
//   visited   one bit per vertex of the graph (vis), cleared per sweep.
//   claims    labelled levels: the unvisited neighbours of the level, each with the smallest
//             frontier position that reaches it. They are the next level's vertices, a few hundred at
//             most on meshes, so they sit in an open-addressing hash table keyed by vertex. Keys and
//             values carry a generation number (one per level), so entries of earlier levels read as
//             empty and nothing is cleared between levels.
//   lists     per warp, the unvisited neighbours of its part of the level in (position, row) order, so
//             that claiming, testing and writing run 32 of them at a time.
//   frontier  the shared cache of EngineSmem (two buffers), beyond kCache in perm or the queue.
//
// What bounds a level is the length of one warp's instruction chain (about 6 cycles an instruction
// with the few warps of one graph, against 30 for shared memory and 300 for a row from L2), so the
// steps are kept few and wide:
//   - a warp with at most 4 frontier vertices gives each 8 lanes: lane k reads word k of the 32-byte row
//     (7 neighbours, then the degree) and has one neighbour to look at and to keep in registers; a
//     ballot over the owned neighbours lists the children in (parent, row) order, i.e. (parent label,
//     degree, id);
//   - a warp with more gives each vertex one lane and packs the unvisited neighbours into its list.
// Warps take consecutive runs of the frontier; one scan over the warps' counts ranks the level. A
// labelled level is three CTA barriers (claims done; counts; children written), a levels-only one a
// single barrier: the visited bit's atomicOr tells whether a neighbour is new.
//
// Against the sweeps with their state in global memory, GB300: the 64x64 grid (254 levels, one CTA,
// rows in shared memory too) 0.387 -> 0.129 ms; 10,000 graphs of 100 to 50,000 vertices 25.7 -> 13.7 ms;
// 500 of them 5.4 -> 2.7 ms; twenty components of 60,000 vertices each 16.3 -> 8.3 ms.
//
// At a level with more new vertices than the lists or the table take, a CTA engine's sweep goes on in global
// memory (run_wide_rest): its vertices are marked there, and the levels that follow are likely as wide. With
// every such level tried here first and then claimed through the graph's global claim words (wide_level,
// which looks the rows up three times and reads long ones one after another), 500 random graphs of up to
// 50,000 vertices and degree 8 took 18.1 ms instead of 6.1, 2,000 power-law ones of up to 20,000 vertices 33
// instead of 13, a served one of 500,000 vertices 227 instead of 79. The grid's runs end before their levels
// get that wide, and with direct claims only the lists can be too small: there wide_level takes the level.
#pragma once

#include "rcm_engine_state.cuh"

namespace rcm {

constexpr int kLocalPasses = 4;    // passes of a wide level looked at together
constexpr int kLocalProbes = 64;   // table probes before a level is taken to be too wide for it
// A list entry: (vertex, later its table slot) << kLocalPosBits | frontier position.
constexpr int kLocalPosBits = 11;
constexpr unsigned kLocalPos = (1u << kLocalPosBits) - 1u;
static_assert(kCache <= 1 << kLocalPosBits, "positions of a level held in the shared cache");
constexpr int kLocalMax = 1 << (32 - kLocalPosBits);  // vertices of the largest graph
constexpr int kLocalOverflow = 1 << 24;  // a warp's child count that says its level did not fit

// Words of the bitmap of n vertices, in whole 16-byte groups. Bits follow the global ids (vertex w: bit
// w mod 32 of word w / 32 - v0 / 32), so the first word may start in the middle.
__host__ __device__ inline int local_vis_words(long long n) { return (int)((n + 31 + 127) / 128 * 4); }
__host__ __device__ inline int local_id_bits(long long n) {
    int b = 1;
    while ((1LL << b) < n) ++b;
    return b;
}
// Shared-memory bytes of the state with a hash table of `slots` and lists of `entries` together.
__host__ __device__ inline size_t local_bytes(long long n, int slots, int entries) {
    return (size_t)local_vis_words(n) * 4 + (size_t)slots * 8 + (size_t)entries * 4;
}

// Sets up the state for graphs of at most cap vertices: vis (16-byte aligned, local_vis_words(cap)
// words), the claim words hval (one per slot), the table's keys hkey and the lists (`entries` in all).
// One thread calls; the caller synchronises before the first sweep.
__device__ __forceinline__ void local_init(LocalState* l, int cap, int slots, int entries, unsigned* vis,
                                           unsigned* hval, unsigned* hkey, unsigned* list) {
    l->list = list;
    l->qcap = entries / ((int)blockDim.x >> 5);
    l->cap = cap;
    l->idbits = local_id_bits(cap);
    l->slots = slots;
    l->vis = vis;
    l->hkey = hkey;
    l->hval = hval;
    l->gen = ~0u;  // the first level clears the claim words
    l->seq = 0;
}

// Shared-memory accesses by 32-bit shared address: through the generic pointers that an out-of-line
// function gets, every access would first find out where it points, and an atomic would branch on it.
__device__ __forceinline__ unsigned s_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned s_ld(unsigned p) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ int4 s_ld4(unsigned p) {
    int4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ void s_st(unsigned p, unsigned v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned s_or(unsigned p, unsigned v) {
    unsigned old;
    asm volatile("atom.shared.or.b32 %0, [%1], %2;" : "=r"(old) : "r"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ unsigned s_add(unsigned p, unsigned v) {
    unsigned old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ unsigned s_cas(unsigned p, unsigned c, unsigned v) {
    unsigned old;
    asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(old) : "r"(p), "r"(c), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void s_red_min(unsigned p, unsigned v) {
    asm volatile("red.shared.min.u32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void s_red_or(unsigned p, unsigned v) {
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}

// Shared stores and atomics where a word is not zero / above a limit, predicated instead of branched around.
__device__ __forceinline__ void s_st_nz(unsigned on, unsigned p, unsigned v) {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q st.shared.u32 [%0], %1;}" ::"r"(p), "r"(v), "r"(on) : "memory");
}
__device__ __forceinline__ void s_red_min_nz(unsigned on, unsigned p, unsigned v) {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q red.shared.min.u32 [%0], %1;}" ::"r"(p), "r"(v), "r"(on) : "memory");
}
// atom.cas where x > limit, else c.
__device__ __forceinline__ unsigned s_cas_above(unsigned x, unsigned limit, unsigned p, unsigned c, unsigned v) {
    unsigned old;
    asm volatile("{.reg .pred q; setp.gt.u32 q, %4, %5; mov.u32 %0, %2; @q atom.shared.cas.b32 %0, [%1], %2, %3;}"
                 : "=&r"(old) : "r"(p), "r"(c), "r"(v), "r"(x), "r"(limit) : "memory");
    return old;
}

// The same with everything in one block of local_bytes(cap, slots, entries) bytes, 16-byte aligned.
__device__ __forceinline__ void local_init(LocalState* l, int cap, int slots, int entries, unsigned* mem) {
    unsigned* hval = mem + local_vis_words(cap);
    unsigned* hkey = hval + slots;
    local_init(l, cap, slots, entries, mem, hval, hkey, hkey + slots);
}

// A labelled level too wide for the shared tables (Local::wide_level), out of line: it runs rarely and
// would cost every other level registers.
template <bool kDirect>
__device__ __noinline__ int local_wide_level(const EngineArgs* a, EngineSmem* sm, int F, int lstart, int cb,
                                             unsigned gen, unsigned seq);

// kDirect: one claim word per vertex instead of the table, and the rows in shared memory too (graphs
// small enough for that); otherwise the hash table, and rows read through L1.
template <bool kDirect>
struct Local {
    const EngineArgs* a;       // in shared memory: what a level rarely needs is read from there
    EngineSmem* sm;
    const int* rows;           // word k of vertex u's padded row: rows[8 * u + k] (global rows)
    int* perm_end;             // label L is written to perm_end[-L]
    // shared addresses: bitmap, table, this warp's list, rows (direct)
    unsigned vis, hkey, hval, list, srows;
    int qcap, n, v0, slots, shift, idbits;
    unsigned gen, seq;
    unsigned word0, value0;    // the generation's part of a key and of a claim
    int lane, wid;
    int g, k;                  // this lane's vertex group and row word
    unsigned below;            // lanes before this one

    __device__ Local(const EngineArgs* args, EngineSmem* s) {
        a = args;
        sm = s;
        rows = (const int*)a->ell;
        n = a->n;
        v0 = a->v0;
        perm_end = a->perm + (n - 1);
        const LocalState& l = s->loc;
        lane = threadIdx.x & 31;
        wid = threadIdx.x >> 5;
        g = lane >> 3;
        k = lane & 7;
        below = (1u << lane) - 1u;
        vis = s_addr(l.vis) - 4u * ((unsigned)v0 >> 5);
        hkey = s_addr(l.hkey);
        hval = s_addr(l.hval);
        srows = kDirect ? s_addr(rows) : 0u;
        qcap = l.qcap;
        list = s_addr(l.list + wid * qcap);
        slots = l.slots;
        idbits = l.idbits;
        shift = __clz(slots) + 1;  // top log2(slots) bits of the hash
        gen = l.gen;
        seq = l.seq;
    }

    __device__ int warps() const { return (int)(blockDim.x >> 5); }

    __device__ void save() const {
        if (threadIdx.x == 0) {
            sm->loc.gen = gen;
            sm->loc.seq = seq;
        }
    }

    __device__ int row_word(int u) const {
        if constexpr (kDirect) return (int)s_ld(srows + 32u * (unsigned)(u - v0) + 4u * (unsigned)k);
        else return __ldg(rows + 8 * (size_t)u + k);
    }
    __device__ void prefetch(int w) const {
        if constexpr (!kDirect) asm volatile("prefetch.global.L1 [%0];" ::"l"(rows + 8 * (size_t)w));
    }
    // The word of vertex w's bit, shifted so that the bit is the lowest.
    __device__ unsigned visited_word(int w) const {
        return __funnelshift_r(s_ld(vis + 4u * ((unsigned)w >> 5)), 0u, (unsigned)w);
    }
    __device__ bool visited(int w) const { return visited_word(w) & 1u; }

    // Vertices [j0, j1) of a level of F are this warp's: whole groups of 4, consecutive over the warps.
    __device__ void share(int F, int& j0, int& j1) const {
        const int lg = 33 - __clz(warps());  // log2 of the vertices all warps take per pass
        const int per = (F + (1 << lg) - 1) >> lg << 2;
        j0 = min(F, wid * per);
        j1 = min(F, j0 + per);
    }

    // A new generation; when the numbers run out, the table is cleared first.
    __device__ void next_generation() {
        const unsigned gmax = (1u << (32 - idbits)) - 1u;
        if (gen >= gmax) {
            __syncthreads();
            for (int i = threadIdx.x; i < slots; i += blockDim.x) {
                if constexpr (!kDirect) s_st(hkey + 4 * i, 0u);
                s_st(hval + 4 * i, ~0u);
            }
            __syncthreads();
            gen = 0;
        }
        set_generation(gen + 1u);
    }
    __device__ void set_generation(unsigned x) {
        gen = x;
        word0 = gen << idbits;
        value0 = ((1u << (32 - idbits)) - 1u - gen) << idbits;
    }

    __device__ unsigned value(int j) const { return value0 | (unsigned)j; }
    __device__ unsigned long long global_key(int j) const {
        return ((unsigned long long)(0x7fffffffu - seq) << 32) | (unsigned)j;
    }

    // Lowers the claim of unvisited vertex v0 + i to frontier position j in the table. Returns its slot,
    // -1 when the table is too full. s: the first slot to look at.
    __device__ int claim_slot(unsigned i, int j, unsigned s) const {
        const unsigned word = word0 | i;
        for (int t = 0; t < kLocalProbes; ++t) {
            unsigned cur = s_ld(hkey + 4 * s);
            if ((cur >> idbits) != gen) {  // empty: an entry of an earlier generation
                const unsigned old = s_cas(hkey + 4 * s, cur, word);
                if (old == cur) prefetch(v0 + (int)i);  // a vertex of the next level
                cur = old == cur ? word : old;
            }
            if (cur == word) {
                s_red_min(hval + 4 * s, value(j));
                return (int)s;
            }
            s = next_slot(s, i);
        }
        return -1;
    }
    // The probe after slot s: vertices that share a slot part ways.
    __device__ unsigned next_slot(unsigned s, unsigned i) const { return (s + (i << 1) + 1u) & (unsigned)(slots - 1); }

    // Rows hold only vertices of this graph (the validation pass saw to it), and absent neighbours are
    // the vertex itself, which is always visited: nothing below checks a neighbour's range.

    // The row words of this lane for P passes of 4 vertices from position j (word 7: the degree).
    template <int P, class At>
    __device__ void load(At at, int j, int j1, int (&x)[P]) const {
        int u[P];
#pragma unroll
        for (int p = 0; p < P; ++p) u[p] = j + 4 * p < j1 ? at(j + 4 * p) : -1;
#pragma unroll
        for (int p = 0; p < P; ++p) x[p] = u[p] >= 0 ? row_word(u[p]) : -1;
    }

    // Frontier position j of a labelled level (label lstart + j).
    __device__ int labelled_at(int j, unsigned cache, int lstart) const {
        return j < kCache ? (int)s_ld(cache + 4 * j) : ldcg(perm_end - (lstart + j));
    }

    // fn(j, w) for the entries beyond the padded row of every long-row vertex (lanes lm) of one pass whose
    // first position is j: its position and, on each lane, one entry (-1 past the row's end). By the
    // whole warp, 32 entries at a time, the loads of 128 issued together.
    template <class At, class Fn>
    __device__ void long_rows(At at, int j, int x, unsigned lm, Fn fn) const {
        for (unsigned m = lm; m; m &= m - 1) {
            const int src = __ffs(m) - 1, jj = j + (src >> 3);
            const int dg = __shfl_sync(0xffffffffu, x, src);
            const int* row = a->adj + __ldg(a->rowptr + at(jj));
            for (int e0 = kEllNb; e0 < dg; e0 += 128) {
                int w[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) w[r] = e0 + 32 * r + lane < dg ? __ldg(row + e0 + 32 * r + lane) : -1;
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (e0 + 32 * r < dg) fn(jj, w[r]);
            }
        }
    }

    // List entry at shared address p, where `on` is not zero: vertex w with frontier position j,
    // jbase = j - (v0 << kLocalPosBits).
    __device__ void put(unsigned on, unsigned p, int w, unsigned jbase) const {
        s_st_nz(on, p, ((unsigned)w << kLocalPosBits) + jbase);
        if constexpr (kDirect) s_red_min_nz(on, hval + 4 * (unsigned)(w - v0), value0 | (jbase & kLocalPos));
    }
    __device__ unsigned list_base(int j) const { return (unsigned)j - ((unsigned)v0 << kLocalPosBits); }

    // The padded row of vertex u.
    __device__ void row(int u, int (&r)[8]) const {
        int4 x, y;
        if constexpr (kDirect) {
            const unsigned p = srows + 32u * (unsigned)(u - v0);
            x = s_ld4(p);
            y = s_ld4(p + 16);
        } else {
            const int4* p = (const int4*)rows + 2 * (size_t)u;
            x = __ldg(p);
            y = __ldg(p + 1);
        }
        r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
        r[4] = y.x; r[5] = y.y; r[6] = y.z; r[7] = y.w;
    }

    // Exclusive prefix over the warp of c in [0, 7], by its three bits; total: the sum.
    __device__ int prefix7(int c, int& total) const {
        const unsigned b0 = __ballot_sync(0xffffffffu, c & 1), b1 = __ballot_sync(0xffffffffu, c & 2),
                       b2 = __ballot_sync(0xffffffffu, c & 4);
        total = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
        return __popc(b0 & below) + 2 * __popc(b1 & below) + 4 * __popc(b2 & below);
    }

    // Appends the unvisited neighbours of up to 32 vertices from position jb, one per lane, to this
    // warp's list in (position, row) order; count goes past qcap without writing.
    __device__ void collect(unsigned cache, int jb, int j1, int& count) {
        const int j = jb + lane;
        const unsigned on = j < j1 ? 1u : 0u;
        int r[8];
        row((int)s_ld(cache + 4 * min(j, j1 - 1)), r);
        unsigned open[kEllNb];
        int c = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) open[q] = ~visited_word(r[q]) & on;
#pragma unroll
        for (int q = 4; q < kEllNb; ++q) open[q] = 0;
        const bool wide = __any_sync(0xffffffffu, r[7] > 4);  // the row's second half is in use
        if (wide) {
#pragma unroll
            for (int q = 4; q < kEllNb; ++q) open[q] = ~visited_word(r[q]) & on;
        }
#pragma unroll
        for (int q = 0; q < kEllNb; ++q) c += (int)open[q];
        const unsigned lm = wide ? __ballot_sync(0xffffffffu, on && r[7] > kEllNb) : 0u;
        int total, at;
        if (!lm) {
            at = prefix7(c, total);
        } else {
            // rows with more than 7 entries: the rest is counted by the whole warp first
            long_list(cache, jb, r[7], lm, [&](int src, int, bool o) {
                const int m = __popc(__ballot_sync(0xffffffffu, o));
                if (lane == src) c += m;
            });
            const int incl = warp_incl_scan(c);
            total = __shfl_sync(0xffffffffu, incl, 31);
            at = incl - c;
        }
        unsigned p = list + 4u * (unsigned)(count + at);
        count += total;
        if (count > qcap) return;  // the caller sees the overflow
        const unsigned jbase = list_base(j);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            put(open[q], p, r[q], jbase);
            p += 4u * open[q];
        }
        if (wide) {
#pragma unroll
            for (int q = 4; q < kEllNb; ++q) {
                put(open[q], p, r[q], jbase);
                p += 4u * open[q];
            }
        }
        if (lm) {
            long_list(cache, jb, r[7], lm, [&](int src, int w, bool o) {
                const unsigned m = __ballot_sync(0xffffffffu, o);
                const unsigned base = __shfl_sync(0xffffffffu, p, src);
                put(o ? 1u : 0u, base + 4u * (unsigned)__popc(m & below), w, list_base(jb + src));
                if (lane == src) p += 4u * (unsigned)__popc(m);
            });
        }
    }

    // fn(src, w, open) for the entries beyond the padded rows of the lanes lm (vertex jb + src, degree
    // dg on its lane), 32 at a time by the whole warp: the entry and whether it is an unvisited vertex.
    template <class Fn>
    __device__ void long_list(unsigned cache, int jb, int dg, unsigned lm, Fn fn) const {
        for (unsigned m = lm; m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const int d = __shfl_sync(0xffffffffu, dg, src);
            const int* rw = a->adj + __ldg(a->rowptr + (int)s_ld(cache + 4 * (jb + src)));
            for (int e0 = kEllNb; e0 < d; e0 += 128) {
                int w[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) w[t] = e0 + 32 * t + lane < d ? __ldg(rw + e0 + 32 * t + lane) : -1;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    if (e0 + 32 * t >= d) break;
                    fn(src, w[t], w[t] >= 0 && !visited(max(w[t], v0)));
                }
            }
        }
    }

    // Entries [b, b + 32) of this warp's list (of c) claim their vertices in the table, and keep the slot.
    // The first probe is straight-line; what it does not settle goes on in a loop. False where the table
    // is too full.
    __device__ bool claim_list(int b, int c) const {
        const unsigned ids = (1u << idbits) - 1u;
        const unsigned on = b + lane < c ? 1u : 0u;
        const unsigned e = s_ld(list + 4 * min(b + lane, c - 1));
        const unsigned i = e >> kLocalPosBits;
        unsigned s = (i * 0x9E3779B1u) >> shift;
        const unsigned cur = s_ld(hkey + 4 * s);
        // x: the slot's word without the generation's part, above ids where it is of an earlier generation
        // (empty); lanes past the end see no empty slot
        const unsigned x = on ? cur ^ word0 : 0u;
        const unsigned old = s_cas_above(x, ids, hkey + 4 * s, cur, word0 | i) ^ word0;
        const bool made = x > ids && old == x;
        if (made) prefetch(v0 + (int)i);  // a vertex of the next level
        const unsigned hit = made || old == i ? on : 0u;
        s_red_min_nz(hit, hval + 4 * s, value0 | (e & kLocalPos));
        bool ok = true;
        if (hit != on) {
            const int t = claim_slot(i, (int)(e & kLocalPos), next_slot(s, i));
            ok = t >= 0;
            s = ok ? (unsigned)t : 0u;  // (any slot: the level is run again)
        }
        s_st_nz(on, list + 4 * (b + lane), s << kLocalPosBits | (e & kLocalPos));
        return ok;
    }

    // Which of the entries [b, b + 32) hold a child of their position, as a ballot, and what this lane's
    // names (its slot of the table, direct claims: its vertex).
    __device__ unsigned owned_list(int b, int c, unsigned& at) const {
        const unsigned e = s_ld(list + 4 * min(b + lane, c - 1));
        at = e >> kLocalPosBits;
        const unsigned v = s_ld(hval + 4 * at);
        return __ballot_sync(0xffffffffu, b + lane < c && v == (value0 | (e & kLocalPos)));
    }

    // The rank of this warp's first child among the level's, from the warps' counts; kids: their sum.
    __device__ int rank_warps(int count, int& kids) {
        const unsigned counts = s_addr(sm->loc.wc);
        if (lane == 0) s_st(counts + 4 * wid, (unsigned)count);
        __syncthreads();
        const int c = lane < warps() ? (int)s_ld(counts + 4 * lane) : 0;
        kids = __reduce_add_sync(0xffffffffu, c);
        return __reduce_add_sync(0xffffffffu, lane < wid ? c : 0);
    }

    // Child r of the level at labels lab0..: vertex w.
    __device__ void emit(int w, int r, int lab0, unsigned next) {
        if (r < kCache) s_st(next + 4 * r, (unsigned)w);
        perm_end[-(lab0 + r)] = w;
        s_red_or(vis + 4u * ((unsigned)w >> 5), 1u << ((unsigned)w & 31u));
    }

    // One labelled level of F vertices at labels [lstart, lstart + F), positions below kCache in `cache`:
    // the next level goes to `next` and to perm. Returns its size, or -1 when the lists or the table
    // were too small (nothing changed). Every thread calls; `bad` is set where a label left the graph.
    __device__ int labelled_level(int F, int lstart, unsigned cache, unsigned next, bool& bad) {
        if (F > kCache) return -1;
        int jb, j1;
        share(F, jb, j1);
        // A warp with one pass of padded rows needs no list: each lane keeps its neighbour.
        bool held = j1 - jb <= 4;
        bool open = false, fits = true;
        int x = 0;
        unsigned s0 = 0;
        int c = 0;
        if (held && jb < j1) {
            x = row_word((int)s_ld(cache + 4 * min(jb + g, j1 - 1)));
            const bool on = jb + g < j1;
            held = !__any_sync(0xffffffffu, k == 7 && x > kEllNb);
            const unsigned seen = visited_word(k < kEllNb ? x : v0);
            open = on && k < kEllNb && held && !(seen & 1u);
            if (open) {
                const unsigned i = (unsigned)(x - v0);
                if constexpr (kDirect) {
                    s_red_min(hval + 4 * i, value(jb + g));
                    s0 = i;
                } else {
                    const int s = claim_slot(i, jb + g, (i * 0x9E3779B1u) >> shift);
                    fits = s >= 0;
                    s0 = fits ? (unsigned)s : 0u;
                }
            }
        }
        const int jh = jb + g;
        if (!held) {
            for (; jb < j1; jb += 32) collect(cache, jb, j1, c);
            fits &= c <= qcap;
            if (c > qcap) c = 0;
            __syncwarp();
            if constexpr (!kDirect) {
                for (int b = 0; b < c; b += 32) fits &= claim_list(b, c);
            }
        }
        fits = __all_sync(0xffffffffu, fits);
        __syncthreads();
        // a vertex's children are the neighbours whose smallest claim is its position
        unsigned own = 0, id = 0;
        int count = 0;
        if (held) {
            own = __ballot_sync(0xffffffffu, open && s_ld(hval + 4 * s0) == value(jh));
            count = __popc(own);
        } else {
            for (int b = 0; b < c; b += 32) {
                own = owned_list(b, c, id);
                count += __popc(own);
            }
        }
        int kids;
        int rank = rank_warps(fits ? count : kLocalOverflow, kids);
        const int lab0 = lstart + F;
        if (kids >= kLocalOverflow) return -1;
        if (lab0 + kids > n) {  // never on a valid pattern
            bad = true;
            return 0;
        }
        if (held) {
            if ((own >> lane) & 1u) emit(x, rank + __popc(own & below), lab0, next);
        } else {
            for (int b = 0; b < c; b += 32) {
                if (c > 32) own = owned_list(b, c, id);
                if ((own >> lane) & 1u) {
                    const unsigned i = kDirect ? id : s_ld(hkey + 4 * id) & ((1u << idbits) - 1u);
                    emit(v0 + (int)i, rank + __popc(own & below), lab0, next);
                }
                rank += __popc(own);
            }
        }
        __syncthreads();
        return kids;
    }

    // The same level with its claims in the graph's global claim words (direct claims: in the same
    // words): no bound on its size, every step looks the rows up again.
    // Returns -1 where its labels would leave the graph (never on a valid pattern).
    __device__ int wide_level(int F, int lstart, unsigned cache, unsigned next) {
        int j0, j1;
        share(F, j0, j1);
        auto at = [&](int j) { return labelled_at(j, cache, lstart); };
        constexpr int P = kLocalPasses;
        // no vertex: below v0 (this lane has no neighbour)
        auto open = [&](int w) { return w >= v0 && !visited(w); };
        auto lower = [&](int w, int j) {
            if constexpr (kDirect) s_red_min(hval + 4 * (unsigned)(w - v0), value(j));
            else atomicMin(a->claim + w, global_key(j));
        };
        auto mine = [&](int w, int j) {
            if constexpr (kDirect) return open(w) && s_ld(hval + 4 * (unsigned)(w - v0)) == value(j);
            else return open(w) && __ldcg(a->claim + w) == global_key(j);
        };
        auto neighbour = [&](int y) { return k < kEllNb ? y : -1; };
        int x[P];
        for (int jb = j0; jb < j1; jb += 4 * P) {
            load(at, jb + g, j1, x);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (open(neighbour(x[p]))) lower(x[p], jb + g + 4 * p);
                long_rows(at, jb + 4 * p, x[p], __ballot_sync(0xffffffffu, k == 7 && x[p] > kEllNb), [&](int j, int w) {
                    if (open(w)) lower(w, j);
                });
            }
        }
        __syncthreads();
        unsigned own[P];
        auto owned = [&](int jb) {
            load(at, jb + g, j1, x);
            bool o[P];
#pragma unroll
            for (int p = 0; p < P; ++p) o[p] = mine(neighbour(x[p]), jb + g + 4 * p);
#pragma unroll
            for (int p = 0; p < P; ++p) own[p] = __ballot_sync(0xffffffffu, o[p]);
        };
        int count = 0;
        for (int jb = j0; jb < j1; jb += 4 * P) {
            owned(jb);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                count += __popc(own[p]);
                long_rows(at, jb + 4 * p, x[p], __ballot_sync(0xffffffffu, k == 7 && x[p] > kEllNb), [&](int j, int w) {
                    count += __popc(__ballot_sync(0xffffffffu, mine(w, j)));
                });
            }
        }
        int kids;
        int rank = rank_warps(count, kids);
        const int lab0 = lstart + F;
        if (lab0 + kids > n) return -1;
        auto put = [&](unsigned m, int w) {
            if ((m >> lane) & 1u) emit(w, rank + __popc(m & below), lab0, next);
            rank += __popc(m);
        };
        for (int jb = j0; jb < j1; jb += 4 * P) {
            owned(jb);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const unsigned lm = __ballot_sync(0xffffffffu, k == 7 && x[p] > kEllNb);
                for (int v = 0; v < 4; ++v) {
                    const unsigned of = lm ? 0xffu << (8 * v) : 0xffffffffu;
                    put(own[p] & of, x[p]);
                    if (!lm) break;
                    long_rows(at, jb + 4 * p, x[p], lm & of, [&](int j, int w) {
                        put(__ballot_sync(0xffffffffu, mine(w, j)), w);
                    });
                }
            }
        }
        __syncthreads();
        return kids;
    }

    // One levels-only level of F vertices: positions below kCache in `cache`, the others in the queue
    // `cur`; the new vertices go to `next` / `nxt` in any order, counted in *tail. No barrier inside.
    __device__ void levels_level(int F, unsigned cache, const int* cur, unsigned next, int* nxt, unsigned tail) {
        int jb, j1;
        share(F, jb, j1);
        auto at = [&](int j) { return j < kCache ? (int)s_ld(cache + 4 * j) : ldcg(cur + j); };
        auto put = [&](unsigned m, int w, int r) {
            if ((m >> lane) & 1u) {
                r += __popc(m & below);
                prefetch(w);
                if (r < kCache) s_st(next + 4 * r, (unsigned)w); else nxt[r] = w;
            }
        };
        // `count` new vertices of this warp: the first one's position
        auto reserve = [&](int count) {
            int r = 0;
            if (lane == 0 && count) r = (int)s_add(tail, (unsigned)count);
            return __shfl_sync(0xffffffffu, r, 0);
        };
        // 1 where vertex w was not visited; it is now
        auto reach = [&](int w) {
            const unsigned bit = 1u << ((unsigned)w & 31u);
            return s_or(vis + 4u * ((unsigned)w >> 5), bit) & bit ? 0u : 1u;
        };
        auto rest = [&](int u, int d) {  // the entries of a long row beyond the padded ones, by the warp
            const int* rw = a->adj + __ldg(a->rowptr + u);
            for (int e = kEllNb; e < d; e += 32) {
                const int w = e + lane < d ? __ldg(rw + e + lane) : -1;
                const unsigned f = __ballot_sync(0xffffffffu, w >= 0 && reach(w));
                put(f, w, reserve(__popc(f)));
            }
        };
        if (j1 - jb <= 4) {
            // one pass, eight lanes per vertex
            if (jb >= j1) return;
            const bool on = jb + g < j1;
            const int u = at(min(jb + g, j1 - 1));
            const int x = row_word(u);
            const unsigned m = __ballot_sync(0xffffffffu, on && k < kEllNb && reach(x));
            put(m, x, reserve(__popc(m)));
            for (unsigned lm = __ballot_sync(0xffffffffu, on && k == 7 && x > kEllNb); lm; lm &= lm - 1)
                rest(__shfl_sync(0xffffffffu, u, __ffs(lm) - 1), __shfl_sync(0xffffffffu, x, __ffs(lm) - 1));
            return;
        }
        for (; jb < j1; jb += 32) {
            // one vertex per lane
            const bool on = jb + lane < j1;
            const int u = at(min(jb + lane, j1 - 1));
            int r[8];
            row(u, r);
            unsigned fresh[kEllNb];
#pragma unroll
            for (int q = 0; q < kEllNb; ++q) fresh[q] = 0;
            const bool wide = __any_sync(0xffffffffu, r[7] > 4);  // the row's second half is in use
            if (on) {
#pragma unroll
                for (int q = 0; q < 4; ++q) fresh[q] = reach(r[q]);
                if (wide) {
#pragma unroll
                    for (int q = 4; q < kEllNb; ++q) fresh[q] = reach(r[q]);
                }
            }
            int c = 0, total;
#pragma unroll
            for (int q = 0; q < kEllNb; ++q) c += (int)fresh[q];
            int pos = prefix7(c, total);
            pos += reserve(total);
#pragma unroll
            for (int q = 0; q < kEllNb; ++q)
                if (fresh[q]) {
                    prefetch(r[q]);
                    if (pos < kCache) s_st(next + 4 * pos, (unsigned)r[q]); else nxt[pos] = r[q];
                    ++pos;
                }
            if (!wide) continue;
            for (unsigned lm = __ballot_sync(0xffffffffu, on && r[7] > kEllNb); lm; lm &= lm - 1)
                rest(__shfl_sync(0xffffffffu, u, __ffs(lm) - 1), __shfl_sync(0xffffffffu, r[7], __ffs(lm) - 1));
        }
    }

    // Visited bits cleared, the root's set; the caller's next barrier orders them.
    __device__ void start(int root) {
        uint4* v = (uint4*)sm->loc.vis;
        for (int i = threadIdx.x; i < local_vis_words(n) / 4; i += blockDim.x) v[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (threadIdx.x == 0) {
            sm->loc.vis[((unsigned)root >> 5) - ((unsigned)v0 >> 5)] |= 1u << ((unsigned)root & 31u);
            sm->cache[0][0] = root;
        }
    }

    // Min (degree, id) key of a level of F vertices, for every thread.
    template <class At>
    __device__ unsigned long long level_key(int F, At at) const {
        unsigned long long m = kKeyMax;
        for (int j = threadIdx.x; j < F; j += blockDim.x) {
            const int u = at(j);
            const int dg = kDirect ? (int)s_ld(srows + 32u * (unsigned)(u - v0) + 28u) : __ldg(rows + 8 * (size_t)u + 7);
            m = min(m, pack_key(dg, u));
        }
        return block_min_u64(m, sm->wkey);
    }

    // Levels-only sweep from root: eccentricity, last level's min (degree, id) key and size.
    __device__ void sweep_levels(int root, int& ecc, unsigned long long& last_key,
                                 long long& reached) {
        start(root);
        if (threadIdx.x == 0) sm->ntail[0] = 0;
        __syncthreads();
        int* cur = a->qa;
        int* nxt = a->qb;
        int F = 1, cb = 0, p = 0;
        const unsigned c0 = s_addr(sm->cache[0]), tails = s_addr(sm->ntail);
        ecc = 0;
        reached = 1;
        while (true) {
            // one barrier per level: the counter of the level after next is cleared while this one
            // runs (its last readers finished before the previous barrier)
            const int pn = p == 2 ? 0 : p + 1;
            if (threadIdx.x == 0) s_st(tails + 4 * pn, 0u);
            levels_level(F, c0 + 4 * kCache * cb, cur, c0 + 4 * kCache * (cb ^ 1), nxt, tails + 4 * p);
            __syncthreads();
            const int cnt = (int)s_ld(tails + 4 * p);
            if (cnt == 0) break;
            int* t = cur; cur = nxt; nxt = t;
            cb ^= 1;
            p = pn;
            F = cnt;
            reached += cnt;
            ++ecc;
        }
        last_key = level_key(F, [&](int j) { return j < kCache ? sm->cache[cb][j] : ldcg(cur + j); });
    }

    // Labelled levels from level d of F vertices at labels lstart.., held in cache buffer cb, until one is
    // the last (returns true: F and lstart are its) or the next has at least `hi` vertices or is level
    // `stop` (returns false: they are the next one's). `bad` is set where a label left the graph. Levels too
    // wide for the lists or the table claim in global memory; with kLeave the first of them ends the loop
    // instead (`wide`; F and lstart are its, nothing of it done).
    template <bool kLeave>
    __device__ bool labelled_levels(int& F, int& lstart, int& cb, int& d, int hi, int stop, bool& bad, bool& wide) {
        const unsigned c0 = s_addr(sm->cache[0]);
        int left = stop - d;  // counted down in place of a level number
        while (true) {
            next_generation();
            int kids = labelled_level(F, lstart, c0 + 4 * kCache * cb, c0 + 4 * kCache * (cb ^ 1), bad);
            if (kLeave && kids < 0) {
                wide = true;
                d = stop - left;
                return false;
            }
            if (kids < 0) {
                __syncthreads();  // every thread has read the counts
                kids = local_wide_level<kDirect>(a, sm, F, lstart, cb, gen, seq);
                bad |= kids < 0;
            }
            if (kids <= 0) {
                d = stop - left;
                return true;
            }
            lstart += F;
            F = kids;
            cb ^= 1;
            if (--left == 0 || F >= hi) {
                d = stop - left;
                return false;
            }
        }
    }

    // Min key of a labelled level at labels lstart.., held in cache buffer cb.
    __device__ unsigned long long labelled_key(int F, int lstart, int cb) const {
        const unsigned cache = s_addr(sm->cache[cb]);
        return level_key(F, [&](int j) { return labelled_at(j, cache, lstart); });
    }

    // Labelled sweep from root with labels from nv: eccentricity, last level's min key, size. Returns
    // false when a label left the graph. rest > 0: it ended before level ecc, of `rest` vertices (the last
    // of the size numbered), which is too wide (never with direct claims).
    __device__ bool sweep_labelled(int root, int nv, int& ecc, unsigned long long& last_key, int& size, int& rest) {
        start(root);
        if (threadIdx.x == 0) perm_end[-nv] = root;
        __syncthreads();
        ++seq;
        int F = 1, cb = 0, lstart = nv;
        bool bad = false, wide = false;
        ecc = 0;
        labelled_levels<!kDirect>(F, lstart, cb, ecc, kIntMax, kIntMax, bad, wide);
        if (!wide) last_key = labelled_key(F, lstart, cb);
        size = lstart + F - nv;
        rest = wide ? F : 0;
        return !__syncthreads_or(bad);
    }

    // A run of narrow levels on CTA 0 of the grid: level d, F (below kCache) vertices at labels lstart..
    // in perm. first: the sweep starts here, nothing else is visited; otherwise gvis holds what the grid's
    // levels visited since the last run. Runs until the sweep ends, a level has `hi` vertices or, where
    // a->probe is set and not yet passed, that level is next.
    __device__ void run(bool first, int d, int lstart, int F, int hi) {
        const int words = local_vis_words(n) / 4;
        uint4* v = (uint4*)sm->loc.vis;
        uint4* gv = (uint4*)a->gvis;
        for (int i = threadIdx.x; i < words; i += blockDim.x) {
            uint4 x = make_uint4(0u, 0u, 0u, 0u);
            if (first) {
                gv[i] = x;
            } else {
                const uint4 y = __ldcg(gv + i);
                x = v[i];
                x = make_uint4(x.x | y.x, x.y | y.y, x.z | y.z, x.w | y.w);
            }
            v[i] = x;
        }
        for (int j = threadIdx.x; j < F; j += blockDim.x) sm->cache[0][j] = ldcg(perm_end - (lstart + j));
        __syncthreads();
        if (first && threadIdx.x == 0) {
            const unsigned w = (unsigned)sm->cache[0][0];
            sm->loc.vis[w >> 5] |= 1u << (w & 31u);
        }
        __syncthreads();
        ++seq;
        const int d0 = d;
        int cb = 0;
        bool bad = false, wide = false;
        const bool end = labelled_levels<false>(F, lstart, cb, d, hi, a->probe > d ? a->probe : kIntMax, bad, wide);
        const unsigned long long key = end ? labelled_key(F, lstart, cb) : kKeyMax;
        bad = __syncthreads_or(bad);
        save();
        if (threadIdx.x == 0) {
            sm->wr.F = end ? 0 : F;
            sm->wr.lastF = end ? F : 0;
            sm->wr.d = d;
            sm->wr.lstart = lstart;
            sm->wr.lk = key;
            sm->wr.reached = d - d0 + (end ? 1 : 0);
            sm->wr.bad = bad ? 1 : 0;
        }
        __syncthreads();
    }
};

template <bool kDirect>
__device__ __noinline__ int local_wide_level(const EngineArgs* a, EngineSmem* sm, int F, int lstart, int cb,
                                             unsigned gen, unsigned seq) {
    Local<kDirect> l(a, sm);
    l.set_generation(gen);
    l.seq = seq;
    return l.wide_level(F, lstart, s_addr(sm->cache[cb]), s_addr(sm->cache[cb ^ 1]));
}

// The sweeps out of line, one register allocation of their own; results in sm->wr, what a labelled one left
// in sm->loc.rest. labelled 0: levels-only.
template <bool kDirect>
__device__ __noinline__ void local_sweep(const EngineArgs* a, EngineSmem* sm, int labelled, int root, int nv) {
    Local<kDirect> l(a, sm);
    int ecc = 0, size = 0, rest = 0;
    unsigned long long key = kKeyMax;
    long long reached = 0;
    bool ok = true;
    if (labelled) {
        ok = l.sweep_labelled(root, nv, ecc, key, size, rest);
        reached = size;
    } else {
        l.sweep_levels(root, ecc, key, reached);
    }
    l.save();
    if (threadIdx.x == 0) {
        sm->wr.d = ecc;
        sm->wr.lk = key;
        sm->wr.reached = reached;
        sm->wr.bad = ok ? 0 : 1;
        sm->loc.rest = rest;
    }
    __syncthreads();
}

// Local::run out of line; results in sm->wr (reached: levels run).
template <bool kDirect>
__device__ __noinline__ void local_run(const EngineArgs* a, EngineSmem* sm, int first, int d, int lstart, int F,
                                       int hi) {
    Local<kDirect> l(a, sm);
    l.run(first != 0, d, lstart, F, hi);
}

}  // namespace rcm
