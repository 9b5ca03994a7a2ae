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
// Levels with more new vertices than the lists or the table take claim through the graph's global
// claim words instead (wide_level), level by level, with the same result.
#pragma once

#include "rcm_engine_state.cuh"

namespace rcm {

constexpr int kLocalPasses = 4;    // passes of a wide level looked at together
constexpr int kLocalBatch = 2;     // list batches of 32 looked at together
constexpr int kLocalProbes = 64;   // table probes before a level is taken to be too wide for it
// A list entry: (vertex, later its table slot) << kLocalPosBits | frontier position.
constexpr int kLocalPosBits = 11;
constexpr unsigned kLocalPos = (1u << kLocalPosBits) - 1u;
static_assert(kCache <= 1 << kLocalPosBits, "positions of a level held in the shared cache");
constexpr int kLocalMax = 1 << (32 - kLocalPosBits);  // vertices of the largest graph
constexpr int kLocalOverflow = 1 << 24;  // a warp's child count that says its level did not fit

// Words of the bitmap of n vertices, in whole 16-byte groups.
__host__ __device__ inline int local_vis_words(long long n) { return (int)((n + 127) / 128 * 4); }
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

// The same under a predicate, with no branch around it.
__device__ __forceinline__ unsigned s_or_if(bool on, unsigned p, unsigned v, unsigned otherwise) {
    unsigned old;
    asm volatile("{.reg .pred q; setp.ne.u32 q, %3, 0; mov.u32 %0, %4; @q atom.shared.or.b32 %0, [%1], %2;}"
                 : "=&r"(old) : "r"(p), "r"(v), "r"((unsigned)on), "r"(otherwise) : "memory");
    return old;
}
__device__ __forceinline__ void s_st_if(bool on, unsigned p, unsigned v) {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q st.shared.u32 [%0], %1;}"
                 ::"r"(p), "r"(v), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ unsigned s_cas_if(bool on, unsigned p, unsigned c, unsigned v) {
    unsigned old;
    asm volatile("{.reg .pred q; setp.ne.u32 q, %4, 0; mov.u32 %0, %2; @q atom.shared.cas.b32 %0, [%1], %2, %3;}"
                 : "=&r"(old) : "r"(p), "r"(c), "r"(v), "r"((unsigned)on) : "memory");
    return old;
}
__device__ __forceinline__ void s_red_min_if(bool on, unsigned p, unsigned v) {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q red.shared.min.u32 [%0], %1;}"
                 ::"r"(p), "r"(v), "r"((unsigned)on) : "memory");
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
        vis = s_addr(l.vis);
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
    __device__ bool visited(unsigned i) const { return (s_ld(vis + 4u * (i >> 5)) >> (i & 31)) & 1u; }

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
            s = (s + 1) & (unsigned)(slots - 1);
        }
        return -1;
    }

    // This lane's neighbour as a local id, out of range where it holds none (absent, or the degree).
    __device__ unsigned neighbour(int x) const { return k < kEllNb ? (unsigned)(x - v0) : ~0u; }

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

    // Entry r of this warp's list: vertex and position.
    __device__ void put(bool on, int r, unsigned i, int j) const {
        s_st_if(on, list + 4 * r, i << kLocalPosBits | (unsigned)j);
        if constexpr (kDirect) s_red_min_if(on, hval + 4 * i, value(j));
    }

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
        const bool on = j < j1;
        int r[8];
        row((int)s_ld(cache + 4 * min(j, j1 - 1)), r);
        unsigned mask = 0;
#pragma unroll
        for (int q = 0; q < kEllNb; ++q) {
            const unsigned i = (unsigned)(r[q] - v0);
            const bool ok = i < (unsigned)n;
            mask |= (ok && !visited(ok ? i : 0u) ? 1u : 0u) << q;
        }
        if (!on) mask = 0;
        const unsigned lm = __ballot_sync(0xffffffffu, on && r[7] > kEllNb);
        int c = __popc(mask), total, at;
        if (!lm) {
            at = count + prefix7(c, total);
        } else {
            // rows with more than 7 entries: the rest is counted by the whole warp first
            long_list(cache, jb, r[7], lm, [&](int src, unsigned, bool open) {
                const int m = __popc(__ballot_sync(0xffffffffu, open));
                if (lane == src) c += m;
            });
            const int incl = warp_incl_scan(c);
            total = __shfl_sync(0xffffffffu, incl, 31);
            at = count + incl - c;
        }
        count += total;
        if (count > qcap) return;  // the caller sees the overflow
#pragma unroll
        for (int q = 0; q < kEllNb; ++q) {
            const bool open = (mask >> q) & 1u;
            put(open, at, (unsigned)(r[q] - v0), j);
            at += open ? 1 : 0;
        }
        if (lm) {
            long_list(cache, jb, r[7], lm, [&](int src, unsigned i, bool open) {
                const unsigned m = __ballot_sync(0xffffffffu, open);
                const int base = __shfl_sync(0xffffffffu, at, src);
                put(open, base + __popc(m & below), i, jb + src);
                if (lane == src) at += __popc(m);
            });
        }
    }

    // fn(src, i, open) for the entries beyond the padded rows of the lanes lm (vertex jb + src, degree
    // dg on its lane), 32 at a time by the whole warp: the entry as a local id and whether it is an
    // unvisited vertex.
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
                    const unsigned i = (unsigned)(w[t] - v0);
                    const bool ok = w[t] >= 0 && i < (unsigned)n;
                    fn(src, i, ok && !visited(ok ? i : 0u));
                }
            }
        }
    }

    // Entries [b, b + 32 Q) of this warp's list (of c) claim their vertices in the table, and keep the slot.
    // The first probes run side by side; what they do not settle goes on one by one. False where the
    // table is too full.
    template <int Q>
    __device__ bool claim_list(int b, int c) const {
        unsigned e[Q], s[Q], cur[Q];
        bool on[Q], left = false, ok = true;
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            on[p] = b + 32 * p + lane < c;
            e[p] = s_ld(list + 4 * min(b + 32 * p + lane, c - 1));
        }
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            s[p] = ((e[p] >> kLocalPosBits) * 0x9E3779B1u) >> shift;
            cur[p] = s_ld(hkey + 4 * s[p]);
        }
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            const unsigned i = e[p] >> kLocalPosBits, word = word0 | i;
            const bool empty = on[p] && (cur[p] >> idbits) != gen;  // an entry of an earlier generation
            const unsigned old = s_cas_if(empty, hkey + 4 * s[p], cur[p], word);
            if (empty && old == cur[p]) prefetch(v0 + (int)i);  // a vertex of the next level
            const bool hit = on[p] && ((empty && old == cur[p]) || old == word);
            s_red_min_if(hit, hval + 4 * s[p], value((int)(e[p] & kLocalPos)));
            on[p] = on[p] && !hit;
            left |= on[p];
        }
        if (left) {
#pragma unroll
            for (int p = 0; p < Q; ++p) {
                if (!on[p]) continue;
                const int t = claim_slot(e[p] >> kLocalPosBits, (int)(e[p] & kLocalPos), (s[p] + 1) & (unsigned)(slots - 1));
                ok &= t >= 0;
                s[p] = t >= 0 ? (unsigned)t : 0u;  // (any slot: the level is run again)
            }
        }
#pragma unroll
        for (int p = 0; p < Q; ++p)
            s_st_if(b + 32 * p + lane < c, list + 4 * (b + 32 * p + lane), s[p] << kLocalPosBits | (e[p] & kLocalPos));
        return ok;
    }

    // Which of the entries [b, b + 32 Q) hold a child of their position, as ballots, and their vertices
    // or slots; returns the number of children.
    template <int Q>
    __device__ int owned_list(int b, int c, unsigned (&own)[Q], unsigned (&at)[Q]) const {
        unsigned e[Q], v[Q];
#pragma unroll
        for (int p = 0; p < Q; ++p) e[p] = s_ld(list + 4 * min(b + 32 * p + lane, c - 1));
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            at[p] = e[p] >> kLocalPosBits;
            v[p] = s_ld(hval + 4 * at[p]);
        }
        int count = 0;
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            own[p] = __ballot_sync(0xffffffffu, b + 32 * p + lane < c && v[p] == value((int)(e[p] & kLocalPos)));
            count += __popc(own[p]);
        }
        return count;
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

    // Child r of the level at labels lab0..: vertex v0 + i.
    __device__ void emit(unsigned i, int r, int lab0, unsigned next) {
        const int w = v0 + (int)i;
        if (r < kCache) s_st(next + 4 * r, (unsigned)w);
        perm_end[-(lab0 + r)] = w;
        s_red_or(vis + 4 * (i >> 5), 1u << (i & 31));
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
        unsigned i0 = 0, s0 = 0;
        int c = 0;
        if (held && jb < j1) {
            const int x = row_word((int)s_ld(cache + 4 * min(jb + g, j1 - 1)));
            const bool on = jb + g < j1;
            i0 = (unsigned)(x - v0);
            const bool ok = on && k < kEllNb && i0 < (unsigned)n;
            open = ok && !visited(ok ? i0 : 0u);
            held = !__any_sync(0xffffffffu, on && k == 7 && x > kEllNb);
            if (held) {
                if constexpr (kDirect) {
                    s_red_min_if(open, hval + 4 * i0, value(jb + g));
                    s0 = i0;
                } else if (open) {
                    const int s = claim_slot(i0, jb + g, (i0 * 0x9E3779B1u) >> shift);
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
                for (int b = 0; b < c; b += 32 * kLocalBatch) fits &= claim_list<kLocalBatch>(b, c);
            }
        }
        fits = __all_sync(0xffffffffu, fits);
        __syncthreads();
        // a vertex's children are the neighbours whose smallest claim is its position; the first
        // batches' stay in registers
        unsigned own[kLocalBatch], id[kLocalBatch];
        int count = 0;
        if (held) {
            own[0] = __ballot_sync(0xffffffffu, open && s_ld(hval + 4 * s0) == value(jh));
            count = __popc(own[0]);
        } else {
            for (int b = 0; b < c; b += 32 * kLocalBatch) count += owned_list<kLocalBatch>(b, c, own, id);
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
            if ((own[0] >> lane) & 1u) emit(i0, rank + __popc(own[0] & below), lab0, next);
        } else {
            for (int b = 0; b < c; b += 32 * kLocalBatch) {
                if (c > 32 * kLocalBatch) owned_list<kLocalBatch>(b, c, own, id);
#pragma unroll
                for (int p = 0; p < kLocalBatch; ++p) {
                    if ((own[p] >> lane) & 1u) {
                        const unsigned i = kDirect ? id[p] : s_ld(hkey + 4 * id[p]) & ((1u << idbits) - 1u);
                        emit(i, rank + __popc(own[p] & below), lab0, next);
                    }
                    rank += __popc(own[p]);
                }
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
        auto open = [&](unsigned i) { return i < (unsigned)n && !visited(i); };
        auto lower = [&](unsigned i, int j) {
            if constexpr (kDirect) s_red_min(hval + 4 * i, value(j));
            else atomicMin(a->claim + v0 + i, global_key(j));
        };
        auto mine = [&](unsigned i, int j) {
            if constexpr (kDirect) return open(i) && s_ld(hval + 4 * i) == value(j);
            else return open(i) && __ldcg(a->claim + v0 + i) == global_key(j);
        };
        int x[P];
        for (int jb = j0; jb < j1; jb += 4 * P) {
            load(at, jb + g, j1, x);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const unsigned i = neighbour(x[p]);
                if (open(i)) lower(i, jb + g + 4 * p);
                long_rows(at, jb + 4 * p, x[p], __ballot_sync(0xffffffffu, k == 7 && x[p] > kEllNb), [&](int j, int w) {
                    if (w >= 0 && open((unsigned)(w - v0))) lower((unsigned)(w - v0), j);
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
                    count += __popc(__ballot_sync(0xffffffffu, w >= 0 && mine((unsigned)(w - v0), j)));
                });
            }
        }
        int kids;
        int rank = rank_warps(count, kids);
        const int lab0 = lstart + F;
        if (lab0 + kids > n) return -1;
        auto put = [&](unsigned m, unsigned i) {
            if ((m >> lane) & 1u) emit(i, rank + __popc(m & below), lab0, next);
            rank += __popc(m);
        };
        for (int jb = j0; jb < j1; jb += 4 * P) {
            owned(jb);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const unsigned lm = __ballot_sync(0xffffffffu, k == 7 && x[p] > kEllNb);
                for (int v = 0; v < 4; ++v) {
                    const unsigned of = lm ? 0xffu << (8 * v) : 0xffffffffu;
                    put(own[p] & of, neighbour(x[p]));
                    if (!lm) break;
                    long_rows(at, jb + 4 * p, x[p], lm & of, [&](int j, int w) {
                        const unsigned i = (unsigned)(w - v0);
                        put(__ballot_sync(0xffffffffu, w >= 0 && mine(i, j)), i);
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
        auto reach = [&](unsigned i) {
            const bool ok = i < (unsigned)n;
            return !((s_or_if(ok, vis + 4 * (i >> 5), 1u << (i & 31), ~0u) >> (i & 31)) & 1u);
        };
        if (j1 - jb <= 4) {
            // one pass, eight lanes per vertex
            if (jb >= j1) return;
            const bool on = jb + g < j1;
            const int x = row_word(at(min(jb + g, j1 - 1)));
            const unsigned m = __ballot_sync(0xffffffffu, reach(on && k < kEllNb ? (unsigned)(x - v0) : ~0u));
            put(m, x, reserve(__popc(m)));
            const unsigned lm = __ballot_sync(0xffffffffu, on && k == 7 && x > kEllNb);
            if (lm)
                long_rows(at, jb, x, lm, [&](int, int w) {
                    const unsigned f = __ballot_sync(0xffffffffu, reach(w >= 0 ? (unsigned)(w - v0) : ~0u));
                    put(f, w, reserve(__popc(f)));
                });
            return;
        }
        for (; jb < j1; jb += 32) {
            // one vertex per lane
            const bool on = jb + lane < j1;
            const int u = at(min(jb + lane, j1 - 1));
            int r[8];
            row(u, r);
            unsigned mask = 0;
#pragma unroll
            for (int q = 0; q < kEllNb; ++q) mask |= (reach(on ? (unsigned)(r[q] - v0) : ~0u) ? 1u : 0u) << q;
            int total;
            int pos = prefix7(__popc(mask), total);
            pos += reserve(total);
#pragma unroll
            for (int q = 0; q < kEllNb; ++q)
                if ((mask >> q) & 1u) {
                    prefetch(r[q]);
                    if (pos < kCache) s_st(next + 4 * pos, (unsigned)r[q]); else nxt[pos] = r[q];
                    ++pos;
                }
            for (unsigned lm = __ballot_sync(0xffffffffu, on && r[7] > kEllNb); lm; lm &= lm - 1) {
                const int src = __ffs(lm) - 1;
                const int d = __shfl_sync(0xffffffffu, r[7], src);
                const int* rw = a->adj + __ldg(a->rowptr + __shfl_sync(0xffffffffu, u, src));
                for (int e = kEllNb; e < d; e += 32) {
                    const int w = e + lane < d ? __ldg(rw + e + lane) : -1;
                    const unsigned f = __ballot_sync(0xffffffffu, reach(w >= 0 ? (unsigned)(w - v0) : ~0u));
                    put(f, w, reserve(__popc(f)));
                }
            }
        }
    }

    // Visited bits cleared, the root's set; the caller's next barrier orders them.
    __device__ void start(int root) {
        uint4* v = (uint4*)sm->loc.vis;
        for (int i = threadIdx.x; i < (n + 127) / 128; i += blockDim.x) v[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned i = (unsigned)(root - v0);
            sm->loc.vis[i >> 5] |= 1u << (i & 31);
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

    // Labelled sweep from root with labels from nv: eccentricity, last level's min key, size. Returns
    // false when a label left the graph.
    __device__ bool sweep_labelled(int root, int nv, int& ecc, unsigned long long& last_key, int& size) {
        start(root);
        if (threadIdx.x == 0) perm_end[-nv] = root;
        __syncthreads();
        ++seq;
        int F = 1, cb = 0, lstart = nv;
        const unsigned c0 = s_addr(sm->cache[0]);
        bool bad = false;
        ecc = 0;
        while (true) {
            next_generation();
            int kids = labelled_level(F, lstart, c0 + 4 * kCache * cb, c0 + 4 * kCache * (cb ^ 1), bad);
            if (kids < 0) {
                __syncthreads();  // every thread has read the counts
                kids = local_wide_level<kDirect>(a, sm, F, lstart, cb, gen, seq);
                if (kids < 0) {
                    bad = true;
                    break;
                }
            }
            if (kids == 0) break;
            lstart += F;
            F = kids;
            cb ^= 1;
            ++ecc;
        }
        last_key = level_key(F, [&](int j) { return labelled_at(j, c0 + 4 * kCache * cb, lstart); });
        size = lstart + F - nv;
        return !__syncthreads_or(bad);
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

// The sweeps out of line, one register allocation of their own; results in sm->wr. sweep 0: levels-only.
template <bool kDirect>
__device__ __noinline__ void local_sweep(const EngineArgs* a, EngineSmem* sm, int labelled, int root, int nv) {
    Local<kDirect> l(a, sm);
    int ecc = 0, size = 0;
    unsigned long long key = kKeyMax;
    long long reached = 0;
    bool ok = true;
    if (labelled) {
        ok = l.sweep_labelled(root, nv, ecc, key, size);
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
    }
    __syncthreads();
}

}  // namespace rcm
