// rcm_prep.cu -- per-graph preprocessing kernels and the bandwidth/profile kernels.
//
//  * k_degree_validate: D[v] = number of off-diagonal entries of row v (the degree vector D that
//    Alg. 3 and Alg. 4 take as input) plus the structural checks of the pattern.
//  * k_sort_rows_small / k_sort_rows_big: every row with the diagonal dropped and the neighbours in
//    increasing (degree, id), stored as a padded 32-byte row per vertex (7 neighbours + degree) and,
//    for rows of degree > 7, as a full sorted copy. (by_degree = 0: stored order instead, for the
//    sort-free variant.) Sorting each adjacency row once replaces the
//    per-level SortPerm of Sec. IV-B: when a frontier vertex scans its sorted row, the children it
//    owns come out already in (degree, id) order, so the new level is ordered by (parent label,
//    degree, id) by a prefix sum over parents alone.
//  * k_bw_scatter / k_bw_rows: bandwidth and profile of P A P^T (Sec. II-A).
#include "rcm_engine_state.cuh"
#include "rcm_prep.cuh"

namespace rcm {

constexpr int kDegLong = 64;  // longer rows are counted by the whole warp

__global__ void k_degree_validate(int n, int nnz, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                                  int* __restrict__ deg, unsigned char* __restrict__ deg8,
                                  unsigned long long* __restrict__ claim, int* __restrict__ vis, int* __restrict__ bigrows, Ctl* ctl, int small_max,
                                  unsigned long long* __restrict__ adist, unsigned long long* __restrict__ fkey,
                                  const long long* __restrict__ goff, int G) {
    __shared__ int s_max;
    __shared__ unsigned long long s_sum;
    if (threadIdx.x == 0) {
        s_max = 0;
        s_sum = 0;
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0 && (rowptr[0] != 0 || rowptr[n] != nnz || nnz < 0))
        atomicOr(&ctl->status, kErrBadCsr);
    const int stride = gridDim.x * blockDim.x;
    if (goff) {  // a batch: goff must be non-decreasing from 0 to n
        if (blockIdx.x == 0 && threadIdx.x == 0 && (goff[0] != 0 || goff[G] != n)) atomicOr(&ctl->status, kErrBadCsr);
        for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += stride)
            if (goff[g + 1] < goff[g]) atomicOr(&ctl->status, kErrBadCsr);
    }
    // A CTA takes consecutive rows, a warp 32 at a time. In a batch, every entry of a row must stay inside
    // its graph's block [goff[g], goff[g+1]): the warp finds the graph of its first row once (binary
    // search), steps forward from there, and every lane steps on to its own. (Searched for every 32 rows,
    // 14 dependent loads each, the 80M rows of 10,000 graphs took 1.09 ms here, so 0.65.)
    const int lane = threadIdx.x & 31;
    int local_max = 0;
    unsigned local_sum = 0;  // at most the CTA's entries
    const long long per = ((long long)n + gridDim.x - 1) / gridDim.x;
    const int r0 = (int)min(per * blockIdx.x, (long long)n), r1 = (int)min(per * (blockIdx.x + 1), (long long)n);
    int first = -1;  // graph of the warp's last 32 rows
    for (int v0 = r0 + (int)(threadIdx.x & ~31u); v0 < r1; v0 += blockDim.x) {
        const int v = v0 + lane;
        int lo = 0, hi = n;
        if (goff) {
            if (first < 0) {
                int l = 0, h = G - 1;
                while (l < h) {
                    const int mid = (l + h + 1) >> 1;
                    if (goff[mid] <= v0) l = mid; else h = mid - 1;
                }
                first = l;
            }
            while (first + 1 < G && goff[first + 1] <= v0) ++first;
            if (v < r1) {
                int g = first;
                while (g + 1 < G && goff[g + 1] <= v) ++g;
                lo = (int)max(goff[g], 0LL);
                hi = (int)min(goff[g + 1], (long long)n);
            }
        }
        int a = 0, b = 0, d = 0;
        bool bad = false;
        if (v < r1) {
            a = rowptr[v];
            b = rowptr[v + 1];
            if (a < 0 || b < a || b > nnz) {
                atomicOr(&ctl->status, kErrBadCsr);
                a = b = 0;
            }
        }
        // rows of more than kDegLong entries by the warp, one after another
        for (unsigned m = __ballot_sync(0xffffffffu, b - a > kDegLong); m; m &= m - 1) {
            const int src = __ffs(m) - 1, row = v0 + src;
            const int ra = __shfl_sync(0xffffffffu, a, src), rb = __shfl_sync(0xffffffffu, b, src);
            const int rlo = __shfl_sync(0xffffffffu, lo, src), rhi = __shfl_sync(0xffffffffu, hi, src);
            int c = 0;
            const int* entries = colidx + ra;  // (counted from the row's start: offsets near 2^31 do not wrap)
            for (unsigned k = lane; k < (unsigned)(rb - ra); k += 32) {
                const int w = __ldg(entries + k);
                bad |= w < rlo || w >= rhi;
                c += w != row ? 1 : 0;
            }
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == src) d = c;
        }
        if (v >= r1) {
            if (bad) atomicOr(&ctl->status, kErrBadCsr);
            continue;
        }
        {
            // the others by their thread, 8 entries at a time, all loaded before the first is looked at
            const int len = b - a;
            const int* entries = colidx + a;
            for (int k = 0; k < len && len <= kDegLong; k += 8) {
                int w[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) w[t] = k + t < len ? __ldg(entries + k + t) : v;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    bad |= w[t] < lo || w[t] >= hi;
                    d += w[t] != v ? 1 : 0;
                }
            }
            if (bad) atomicOr(&ctl->status, kErrBadCsr);
            if (b - a > small_max) bigrows[atomicAdd(&ctl->nbig, 1)] = v;
        }
        deg[v] = d;
        deg8[v] = (unsigned char)min(d, kDeg8Many);
        claim[v] = ~0ull;
        vis[v] = 0;
        if (adist) adist[v] = ~0ull;
        if (fkey) fkey[v] = 0;
        local_max = max(local_max, d);
        if (d > kHubDegree) atomicAdd(&ctl->hubsum, (unsigned long long)d);
        local_sum += (unsigned)d;
    }
    __syncwarp();
    local_max = __reduce_max_sync(0xffffffffu, local_max);
    local_sum = __reduce_add_sync(0xffffffffu, local_sum);
    if (lane == 0) {
        atomicMax(&s_max, local_max);
        atomicAdd(&s_sum, (unsigned long long)local_sum);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&ctl->maxdeg, s_max);
        atomicAdd(&ctl->degsum, s_sum);
    }
}

// Rows of at most kSmallRowMax stored entries: one thread per row (sort_small_row). Bound by the gathers of
// the neighbours' degrees. A CTA takes consecutive rows, so in a batch the bytes it gathers are one graph's
// at a time and stay in L1; with 4-byte degrees and rows dealt out in turn every gather was an L2 sector
// (10,000 graphs, 80M rows: 1.88 -> 1.12 ms, with the one-word keys of sort_row8).
__global__ void k_sort_rows_small(int n, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                                  const int* __restrict__ deg, const unsigned char* __restrict__ deg8,
                                  int* __restrict__ adj, int4* __restrict__ ell, const Ctl* ctl, int small_max,
                                  int by_degree) {
    if (ctl->status & kErrBadCsr) return;
    const long long per = ((long long)n + gridDim.x - 1) / gridDim.x;
    const int lo = (int)min(per * blockIdx.x, (long long)n), hi = (int)min(per * (blockIdx.x + 1), (long long)n);
    for (int v = lo + (int)threadIdx.x; v < hi; v += blockDim.x)
        if (rowptr[v + 1] - rowptr[v] <= small_max) sort_small_row(v, rowptr, colidx, deg, deg8, adj, ell, by_degree);
}

// Sorted row of v from keys[0, m) already sorted: the full row into adj (from offset a) and the
// padded row (first 7 + degree); one thread writes the padded row.
__device__ __forceinline__ void write_sorted_row(int v, int a, int m, const unsigned long long* keys, int* adj,
                                                 int4* ell, int t, int nt) {
    for (int i = t; i < m; i += nt) adj[a + i] = (int)(unsigned)(keys[i] & 0xffffffffu);
    if (t == 0) {
        int r[8];
        for (int i = 0; i < 7; ++i) r[i] = i < m ? (int)(unsigned)(keys[i] & 0xffffffffu) : v;
        r[7] = m;
        store_ell(ell, v, r);
    }
}

// Rows longer than the per-thread sorter (listed in bigrows), by size:
//   at most kWarpRowMax entries: one warp per row, bitonic sort in the warp's slice of shared memory
//     (the rows of scale-free graphs are mostly a few dozen entries long);
//   at most kBigRowSmem keys: one CTA per row, bitonic sort in shared memory;
//   longer: CTA 0 alone, in global scratch (scratch holds next_pow2(maxdeg) keys).
// Launched with kBigRowThreads threads and kBigRowSmem keys of dynamic shared memory.
__global__ void k_sort_rows_big(int n, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                                const int* __restrict__ deg, int* __restrict__ adj, int4* __restrict__ ell,
                                const int* __restrict__ bigrows, const Ctl* ctl,
                                unsigned long long* __restrict__ scratch, int by_degree) {
    extern __shared__ unsigned long long s_keys[];
    __shared__ int s_m;
    if (ctl->status & kErrBadCsr) return;
    const int nbig = ctl->nbig;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // one warp per row; the keys are gathered in stored order (a warp compaction skips the diagonal)
    unsigned long long* ws = s_keys + (size_t)wid * kWarpRowMax;
    for (int r = blockIdx.x * nw + wid; r < nbig; r += gridDim.x * nw) {
        const int v = bigrows[r];
        const int a = rowptr[v], b = rowptr[v + 1];
        if (b - a > kWarpRowMax) continue;
        int m = 0;
        for (int k0 = 0; k0 < b - a; k0 += 32) {
            const int k = k0 + lane;
            const int w = k < b - a ? colidx[a + k] : v;
            const bool keep = w != v;
            const unsigned bal = __ballot_sync(0xffffffffu, keep);
            if (keep) ws[m + __popc(bal & ((1u << lane) - 1u))] = row_key(deg, w, k, by_degree);
            m += __popc(bal);
        }
        int P = 1;
        while (P < m) P <<= 1;
        for (int i = m + lane; i < P; i += 32) ws[i] = kKeyMax;
        __syncwarp();
        bitonic_sort_warp(ws, P);
        write_sorted_row(v, a, m, ws, adj, ell, lane, 32);
        __syncwarp();
    }
    __syncthreads();
    // one CTA per row
    for (int r = blockIdx.x; r < nbig; r += gridDim.x) {
        const int v = bigrows[r];
        const int a = rowptr[v], b = rowptr[v + 1];
        if (b - a <= kWarpRowMax) continue;
        const int m = deg[v];
        int P = 1;
        while (P < m) P <<= 1;
        if (P > kBigRowSmem) continue;
        if (threadIdx.x == 0) s_m = 0;
        __syncthreads();
        for (unsigned k = threadIdx.x; k < (unsigned)(b - a); k += blockDim.x) {
            const int w = colidx[a + k];
            if (w != v) s_keys[atomicAdd(&s_m, 1)] = row_key(deg, w, (int)k, by_degree);
        }
        __syncthreads();
        for (int i = m + threadIdx.x; i < P; i += blockDim.x) s_keys[i] = kKeyMax;
        __syncthreads();
        bitonic_sort_cta(s_keys, P);
        write_sorted_row(v, a, m, s_keys, adj, ell, threadIdx.x, blockDim.x);
        __syncthreads();
    }
    // rows beyond shared memory, by CTA 0 in global scratch: its threads scan the list together
    // (one entry each per round), then sort the rows found one after another
    if (blockIdx.x != 0) return;
    for (int r0 = 0; r0 < nbig; r0 += blockDim.x) {
        const int r = r0 + (int)threadIdx.x;
        const bool huge = r < nbig && deg[bigrows[r]] > kBigRowSmem;
        const int cnt = __syncthreads_count(huge);
        if (cnt == 0) continue;
        if (threadIdx.x == 0) s_m = kIntMax;
        __syncthreads();
        if (huge) atomicMin(&s_m, r);
        __syncthreads();
        // sort the first huge row of this round, then rescan from just after it
        const int rr = s_m;
        __syncthreads();
        r0 = rr + 1 - (int)blockDim.x;
        const int v = bigrows[rr];
        const int m = deg[v];
        int P = 1;
        while (P < m) P <<= 1;
        const int a = rowptr[v], b = rowptr[v + 1];
        if (threadIdx.x == 0) s_m = 0;
        __syncthreads();
        for (unsigned k = threadIdx.x; k < (unsigned)(b - a); k += blockDim.x) {
            const int w = colidx[a + k];
            if (w != v) scratch[atomicAdd(&s_m, 1)] = row_key(deg, w, (int)k, by_degree);
        }
        __syncthreads();
        for (int i = m + threadIdx.x; i < P; i += blockDim.x) scratch[i] = kKeyMax;
        __syncthreads();
        bitonic_sort_cta(scratch, P);
        write_sorted_row(v, a, m, scratch, adj, ell, threadIdx.x, blockDim.x);
        __syncthreads();
    }
}

// ---- bandwidth / profile (Sec. II-A) ----

// Position of every vertex. pos starts at -1 everywhere: perm is a permutation exactly if all its n
// entries are in range and k_bw_rows then finds no vertex without a position, so plain stores will do
// where atomic exchanges looked for duplicates.
__global__ void k_bw_scatter(int n, const int* __restrict__ perm, int* __restrict__ pos, int* __restrict__ err) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int v = perm[i];
        if ((unsigned)v >= (unsigned)n) atomicOr(err, 1);
        else pos[v] = i;
    }
}

// Max and sum of beta = position of row v - least position in row v (both orders of the rows give them, so
// the rows are taken as stored: rowptr and colidx stream, and only the entries' positions are gathered, 8
// at a time per thread; rows longer than kBwLong by the whole warp). Bound by those gathers, one sector of
// L2 per entry. The whole call on the 192^3 grid: 447 us with the rows in the order of the permutation
// (every array gathered: 320 us of it) and a synchronisation between the kernels, 242 us so.
constexpr int kBwLong = 64;
__global__ void k_bw_rows(int n, const int* __restrict__ rowptr, const int* __restrict__ colidx,
                          const int* __restrict__ pos, int* __restrict__ err,
                          unsigned long long* __restrict__ out /* [0] max beta, [1] sum beta */) {
    __shared__ unsigned long long s_max, s_sum;
    if (threadIdx.x == 0) { s_max = 0; s_sum = 0; }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    int lmax = 0;
    unsigned long long lsum = 0;
    for (int v0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); v0 < n; v0 += gridDim.x * blockDim.x) {
        const int v = v0 + lane;
        int i = 0, f = 0, a = 0, b = 0;
        if (v < n) {
            i = f = pos[v];
            if (i < 0) atomicOr(err, 1);
            a = rowptr[v];
            b = rowptr[v + 1];
        }
        const int len = b - a;
        const int* entries = colidx + a;  // (counted from the row's start: offsets near 2^31 do not wrap)
        if (len <= kBwLong) {
            for (int k = 0; k < len; k += 8) {
                int w[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) w[t] = k + t < len ? entries[k + t] : v;
#pragma unroll
                for (int t = 0; t < 8; ++t) w[t] = __ldg(pos + w[t]);
#pragma unroll
                for (int t = 0; t < 8; ++t) f = min(f, w[t]);
            }
        }
        for (unsigned m = __ballot_sync(0xffffffffu, len > kBwLong); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            const int ra = __shfl_sync(0xffffffffu, a, src), rb = __shfl_sync(0xffffffffu, b, src);
            int least = kIntMax;
            const int* row = colidx + ra;
            for (unsigned k = lane; k < (unsigned)(rb - ra); k += 32) least = min(least, __ldg(pos + row[k]));
            least = __reduce_min_sync(0xffffffffu, least);
            if (lane == src) f = min(f, least);
        }
        lmax = max(lmax, i - f);
        lsum += (unsigned long long)(i - f);
    }
    lmax = __reduce_max_sync(0xffffffffu, lmax);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) {
        atomicMax(&s_max, (unsigned long long)lmax);
        atomicAdd(&s_sum, lsum);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&out[0], s_max);
        atomicAdd(&out[1], s_sum);
    }
}

}  // namespace rcm
