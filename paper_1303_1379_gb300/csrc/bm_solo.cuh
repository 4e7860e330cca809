// Small graphs on one thread-block cluster (sm_103a): the cheap matching and the
// whole search of the default mode (APFB, GPUBFS-WR, one endpoint per root; arXiv
// 1303.1379, Section 3, Algorithms 1, 3, 4) in one launch each, with the matching,
// the forest and the queue in the cluster's shared memory.
//
// What bounds a small graph is the round trip of a BFS level, not the edges: on
// the whole grid a level costs 5.6 us (a grid barrier, and queue entry -> row
// range -> rows -> matches -> claim -> append, each a trip to L2).  Here a level
// is one cluster barrier and everything it reads is shared memory, nearly all of
// it the block's own.  Ids take 16 bits.
//
// Layout, per block of a cluster of C (owner of id i: block (i / 32) mod C):
//  * rm: the rows' matches, a full copy in every block (a level reads one per
//    edge; they change only in Alternate, which writes all copies);
//  * vis: one bit per column in a tree.  The owner's bits decide (an atomic OR
//    there claims a column); the other bits are hints that save asking again,
//    refreshed from the owners when a phase takes columns back;
//  * srv: one bit per root that took an endpoint, a full copy in every block
//    (the owner's decides, its winner sets all);
//  * rcl: one bit per free row claimed as a path's end, at its owner;
//  * cm, pr, rows: a column's match, its parent and root, and its rows, at its
//    owner, which also expands it.  There is no queue: a claim sets the column's
//    bit in a second map at its owner, which lists its columns from that map after
//    the level's barrier, so no append waits for a position, and levels are spread
//    over the blocks by column id.
// A word's rows that do not fit the block's memory are read from the graph itself.
// One block (C = 1) for the smallest graphs, whose levels are too narrow for more, of
// 512 threads (1,000 rows: 25 us a search, with 1,024 threads 38 us: half as many warps
// meet at each barrier); a cluster spreads the wide levels' instructions and holds larger
// graphs.  What a level costs then is a warp's chain of instructions (about 2,500
// cycles for 64 edges a warp; a narrow level's columns go to all warps), and with
// C = 16 the barrier with its release (2,000 cycles).
// 10,000 rows, 45 k entries, cheap matching + search: 374 us on the grid, 223 us
// here (search 305 -> 182 us, 36 levels); 100 rows: 137 -> 66 us.  Queues with
// remote appends in place of the second map took 240 us for the same search, four
// edges of a thread in flight instead of two 198 us (160 us, kernel alone).
//
// The search is the persistent kernel's (k_match): levels expanded by warps
// (warp_expand_sb's edge ownership), trees carried from phase to phase, phases
// cut once they are narrow.
#pragma once
#include "bm_device.cuh"

namespace bms1 {

using bmd::Ctl;
using bmd::FULL;
using bmd::L0;
using bmd::Params;

typedef unsigned short u16;
constexpr int SOLO_T = 1024;           // threads of a cluster's block
constexpr int SOLO_T1 = 512;           // threads of a single block
constexpr int SOLO_FREE = 0xffff;      // "unmatched" in 16 bits
constexpr int SOLO_MAX = 0xfffe;       // rows and columns with a 16-bit id
constexpr int SOLO_SMEM = 216 * 1024;  // dynamic shared memory of a block
constexpr int PART = 128;              // a listed column's rows are expanded in parts of this many
constexpr int SOLO_U = 2;              // edges of a thread in flight
constexpr int TIMED_OUT = -(1 << 30);  // added to a level's columns: the launch's time is up
constexpr int SOLO_PASS = 2;           // status: the search is left to the grid
constexpr int ROW_GLOBAL = 1 << 30;    // marks row positions in the graph's own row_idx

struct SoloArgs {
    const int32_t* rm_src;  // the matching to start from (the installed one, or the caller's)
    const int32_t* cm_src;
    int32_t* rm_out;        // caller's copies of the result (nullable)
    int32_t* cm_out;
    Ctl* h_ctl;             // the host's copy of the control block (pinned)
    int32_t check_src;      // check that rm_src / cm_src are in range and inverse to each other
    int32_t check_err;      // p.ctl holds the outcome of input checks queued before
    int32_t pre;            // the first phase was run as a cheap matching, from the empty matching
    int32_t max_roots;      // from more roots than this nothing is done, and the status is SOLO_PASS
};

// Where a block keeps what, in bytes from its dynamic shared memory's start.
struct Layout {
    unsigned own_cw;  // words of 32 columns that a block owns
    unsigned beg, deg, pr, vis, fresh, srv, rcl, cm, list, rm, rows, rows_cap, bytes;
    __host__ __device__ Layout(int nr, int nc, long long nnz, int C) {
        const unsigned cw = ((unsigned)nc + 31) / 32, rw = ((unsigned)nr + 31) / 32;
        own_cw = (cw + C - 1) / C;
        const unsigned own = 32 * own_cw;
        beg = 0;
        deg = beg + 4 * own;
        pr = deg + 4 * own;
        vis = pr + 4 * own;
        fresh = vis + 4 * cw;
        srv = fresh + 8 * own_cw;
        rcl = srv + 4 * cw;
        cm = rcl + 4 * ((rw + C - 1) / C);
        list = (cm + 2 * own + 3) & ~3u;
        rm = list + 4 * (own + (unsigned)(nnz / PART));
        rows = (rm + 2 * (unsigned)nr + 15) & ~15u;
        // room for an even share of the rows and a quarter more, as far as the block's memory goes
        const long long want = C == 1 ? nnz : nnz / C + nnz / (4 * C) + 1024;
        const long long room = rows < (unsigned)SOLO_SMEM ? ((unsigned)SOLO_SMEM - rows) / 2 : 0;
        rows_cap = (unsigned)(want < room ? want : room);
        bytes = rows + 2 * rows_cap;
    }
};

// What the blocks tell one another at a cluster barrier: each adds its part to
// every block's copy.  Three rotate: step s uses slot s % 3 and clears slot
// (s + 2) % 3 after its barrier (last read before it, next added to after the next).
struct __align__(16) Pub {
    int cnt;   // columns claimed (first step of a phase: kept; first of all: roots)
    int eps;   // endpoints claimed (first step: unmatched columns)
    int flag;  // error code
    int pad;
};

struct SoloStats {
    long long levels, eps, ins, roots;
    int levels_max, last_eps, first_ep, last_ep;
};

struct SoloShared {
    SoloStats st;
    Pub pub[3];
    Pub mine;   // this block's part of the current step
    int nl[2];  // entries of the block's list, by step parity
    int used, flag;
    int base[SOLO_T];          // per warp: its columns' first row position minus their start
    unsigned ent[SOLO_T];      // per warp: (column << 16 | root)
    unsigned long long sum[4];
};

// ---- shared memory of the cluster's blocks, by 32-bit address
__device__ __forceinline__ unsigned saddr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
template <int C>
__device__ __forceinline__ unsigned at(unsigned a, int rank) {  // the same place in block `rank`
    if (C == 1) return a;
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ unsigned dld32(unsigned a) {
    unsigned v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int dld16(unsigned a) {
    u16 v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void dst32(unsigned a, unsigned v) {
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dst16(unsigned a, int v) {
    asm volatile("st.relaxed.cluster.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"((u16)v) : "memory");
}
__device__ __forceinline__ unsigned dor(unsigned a, unsigned v) {
    unsigned o;
    asm volatile("atom.relaxed.cluster.shared::cluster.or.b32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ void dred_or(unsigned a, unsigned v) {
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dred_and(unsigned a, unsigned v) {
    asm volatile("red.relaxed.cluster.shared::cluster.and.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dred_add(unsigned a, int v) {
    asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dred_min(unsigned a, int v) {
    asm volatile("red.relaxed.cluster.shared::cluster.min.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int dcas(unsigned a, int want, int v) {
    int o;
    asm volatile("atom.relaxed.cluster.shared::cluster.cas.b32 %0, [%1], %2, %3;" : "=r"(o) : "r"(a), "r"(want), "r"(v) : "memory");
    return o;
}
template <int C>
__device__ __forceinline__ int my_rank() {
    if (C == 1) return 0;
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
// Every thread of the cluster; orders all shared-memory accesses before it ahead of those after it.
template <int C>
__device__ __forceinline__ void cluster_sync() {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
template <int C>
__device__ __forceinline__ int owner(int i) {
    return C == 1 ? 0 : (i >> 5) & (C - 1);
}
template <int C>
__device__ __forceinline__ int slot_of(int i) {  // place in the owner's arrays
    return C == 1 ? i : (int)(((unsigned)i >> 5) / C * 32 + (i & 31));
}

__device__ __forceinline__ void block_add(unsigned long long* dst, unsigned v) {
    const unsigned long long s = __reduce_add_sync(FULL, v & 0xffffu) +
                                 ((unsigned long long)__reduce_add_sync(FULL, v >> 16) << 16);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(dst, s);
}

template <int C, int T>
__global__ void __launch_bounds__(T, 1) k_solo(Params p, SoloArgs a, long long nnz) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ SoloShared sm;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, wb = t & ~31;
    const int rank = my_rank<C>();
    const int nr = p.nr, nc = p.nc, words = (nc + 31) >> 5;
    const Layout lay(nr, nc, nnz, C);
    int* const col_beg = (int*)(dyn + lay.beg);        // own columns: first row position, number of rows
    int* const col_deg = (int*)(dyn + lay.deg);
    unsigned* const pr = (unsigned*)(dyn + lay.pr);    // own columns in a tree: (parent or, of a served root, its
                                                       // endpoint row) << 16 | root
    unsigned* const vis = (unsigned*)(dyn + lay.vis);
    unsigned* const fresh = (unsigned*)(dyn + lay.fresh);  // own words: columns claimed during a step, by step parity
    unsigned* const srv = (unsigned*)(dyn + lay.srv);
    unsigned* const rcl = (unsigned*)(dyn + lay.rcl);
    u16* const cm = (u16*)(dyn + lay.cm);
    unsigned* const list = (unsigned*)(dyn + lay.list);  // own columns to expand: part << 16 | column's slot
    u16* const rm = (u16*)(dyn + lay.rm);
    u16* const rows = (u16*)(dyn + lay.rows);
    const unsigned s_vis = saddr(vis), s_srv = saddr(srv), s_rcl = saddr(rcl), s_cm = saddr(cm), s_pr = saddr(pr),
                   s_rm = saddr(rm), s_fresh = saddr(fresh), s_pub = saddr(&sm.pub[0]);
    const unsigned long long t_start = bmd::globaltimer();
    const unsigned long long deadline = t_start + (unsigned long long)p.total_ns;
    if (t < 3) sm.pub[t] = Pub{0, 0, 0, 0};
    if (t < 4) sm.sum[t] = 0;
    if (t == 0) {
        sm.st = SoloStats{};
        sm.mine = Pub{0, 0, 0, 0};
        sm.nl[0] = sm.nl[1] = sm.used = sm.flag = 0;
        if (a.check_err) sm.flag = p.ctl->err;
        else if (rank == 0) p.ctl->err = 0;
    }
    for (int w = t; w < words; w += T) vis[w] = srv[w] = 0u;
    for (int w = t; w < 2 * (int)lay.own_cw; w += T) fresh[w] = 0u;
    for (int w = t; w < (int)((lay.cm - lay.rcl) >> 2); w += T) rcl[w] = 0u;
    cluster_sync<C>();  // every block has started and cleared its shared memory
    const int input_err = sm.flag;
    const bool leader = rank == 0 && t == 0;  // keeps the statistics, in shared memory
    unsigned cols = 0, edges = 0, em = 0, alt = 0;
    // ---- the matching and the own columns' rows to shared memory; unmatched columns with rows are the first roots
    if (input_err == 0) {
        bool bad = false;
        for (int r = t; r < nr; r += T) {
            int c = __ldg(&a.rm_src[r]);
            if (a.check_src && owner<C>(r) == rank && c != -1 && (c < 0 || c >= nc || __ldg(&a.cm_src[c]) != r)) {
                bad = true;
                c = -1;
            }
            if (c >= 0 && (c >= nc || !bmd::idx_ok(p, c, nc))) c = -1;
            rm[r] = (u16)(c < 0 ? SOLO_FREE : c);
        }
        int nf = 0, nroot = 0;
        for (int ow = warp; ow < (int)lay.own_cw; ow += T / 32) {
            const int w = ow * C + rank, c = w * 32 + lane, sl = ow * 32 + lane;
            int b = 0, d = 0, r = 0;
            if (c < nc) {
                b = __ldg(&p.col_ptr[c]);
                d = __ldg(&p.col_ptr[c + 1]) - b;
                r = __ldg(&a.cm_src[c]);
                if (a.check_src && r != -1 && (r < 0 || r >= nr || __ldg(&a.rm_src[r]) != c)) { bad = true; r = -1; }
                if (r >= 0 && !bmd::idx_ok(p, r, nr)) r = -1;
            }
            const bool root = r < 0 && d > 0;
            nf += r < 0;
            nroot += root;
            cm[sl] = (u16)(r < 0 ? SOLO_FREE : r);
            pr[sl] = (unsigned)c << 16 | (unsigned)c;
            const unsigned m = __ballot_sync(FULL, root);
            int incl = d;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const int v = __shfl_up_sync(FULL, incl, s);
                if (lane >= s) incl += v;
            }
            const int total = __shfl_sync(FULL, incl, 31), first = __shfl_sync(FULL, b, 0);
            int at0 = 0;
            if (lane == 0) {
                if (w < words) vis[w] = fresh[ow] = m;
                at0 = ROW_GLOBAL;
                if (*(volatile int*)&sm.used + total <= (int)lay.rows_cap) at0 = atomicAdd(&sm.used, total);
                if (at0 + total > (int)lay.rows_cap) at0 = ROW_GLOBAL;  // (others were faster)
            }
            at0 = __shfl_sync(FULL, at0, 0);
            col_beg[sl] = at0 == ROW_GLOBAL ? b + ROW_GLOBAL : at0 + incl - d;
            col_deg[sl] = d;
            if (at0 != ROW_GLOBAL)
                for (int j = lane; j < total; j += 32) {
                    const int rr = __ldg(&p.row_idx[first + j]);
                    rows[at0 + j] = (u16)(bmd::idx_ok(p, rr, nr) ? rr : 0);
                }
        }
        if (bad) sm.mine.flag = -9 /*BM_ERR_INVALID_MATCHING*/;
        nf = __reduce_add_sync(FULL, nf);
        nroot = __reduce_add_sync(FULL, nroot);
        if (lane == 0 && nf) atomicAdd(&sm.mine.eps, nf);
        if (lane == 0 && nroot) atomicAdd(&sm.mine.cnt, nroot);
    } else if (t == 0) {
        sm.mine.flag = input_err;
    }
    // Ends a step: the totals of the cluster, and (when the search goes on) the own columns claimed during it
    // in the list.  first: the owners' tree marks are copied to this block's hints.
    int step = 0, sum_cnt = 0, sum_eps = 0, flag = 0, nl = 0;
    auto end_step = [&](bool first) {
        const int s = step % 3, par = step & 1;
        ++step;
        __syncthreads();
        if (C > 1) {
            if (warp == 0) {
                const Pub v = sm.mine;
                const unsigned b = at<C>(s_pub + s * (unsigned)sizeof(Pub), lane & (C - 1));
                if (lane < C) {
                    if (v.cnt) dred_add(b, v.cnt);
                    if (v.eps) dred_add(b + 4, v.eps);
                    if (v.flag) dred_min(b + 8, v.flag);
                }
            }
            cluster_sync<C>();
            sum_cnt = sm.pub[s].cnt;
            sum_eps = sm.pub[s].eps;
            flag = sm.pub[s].flag;
        } else {
            sum_cnt = sm.mine.cnt;
            sum_eps = sm.mine.eps;
            flag = sm.mine.flag;
            __syncthreads();  // read before it is cleared
        }
        // a warp takes four own words at a time, a lane a column of each; a column of more than PART rows is
        // listed once for each part
        for (int ow0 = 4 * warp; ow0 < (int)lay.own_cw; ow0 += 4 * (T / 32)) {  // warp-uniform
            unsigned f[4];
            int n = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                f[i] = ow0 + i < (int)lay.own_cw ? fresh[par * (int)lay.own_cw + ow0 + i] : 0u;
                n += __popc(f[i]);
            }
            if (n == 0) continue;
            int pos = 0;
            if (lane == 0) pos = atomicAdd(&sm.nl[par], n);
            pos = __shfl_sync(FULL, pos, 0);  // (every lane has read the words)
            if (lane < 4 && ow0 + lane < (int)lay.own_cw) fresh[par * (int)lay.own_cw + ow0 + lane] = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (f[i] >> lane & 1u) {
                    const int sl = (ow0 + i) * 32 + lane, d = col_deg[sl];
                    list[pos + __popc(f[i] & ((1u << lane) - 1))] = (unsigned)sl;
                    if (d > PART) {
                        const int more = (d - 1) / PART, at1 = atomicAdd(&sm.nl[par], more);
#pragma unroll 1
                        for (int k = 1; k <= more; ++k) list[at1 + k - 1] = (unsigned)k << 16 | (unsigned)sl;
                    }
                }
                pos += __popc(f[i]);
            }
        }
        if (C > 1 && first)
            for (int w = t; w < words; w += T)
                if ((w & (C - 1)) != rank) vis[w] = dld32(at<C>(s_vis + 4u * w, w & (C - 1)));
        if (t == 0) {
            sm.pub[(s + 2) % 3] = Pub{0, 0, 0, 0};
            sm.mine = Pub{0, 0, 0, 0};
            sm.nl[par ^ 1] = 0;
        }
        __syncthreads();
        nl = sm.nl[par];
    };
    end_step(true);
    int n_roots = sum_cnt, n_free = sum_eps, n_front = sum_cnt;
    int initial = nc - n_free;
    int status = flag == 0 && n_roots > a.max_roots ? SOLO_PASS : flag, phases = 0, no_roots = 0;
    if (a.pre && initial > 0) {
        phases = 1;
        if (leader) {
            sm.st.levels = sm.st.levels_max = 1;
            sm.st.eps = initial;
            sm.st.roots = initial + n_roots;
            if (p.profile && p.profile_cap > 0) {
                p.profile[0] = p.profile[2] = p.profile[3] = 1;
                p.profile[1] = initial;
            }
            alt = (unsigned)initial;
        }
        initial = 0;
    }
    bool carry = p.phase_limit_is_error != 0;  // (as k_match: not under a caller's phase limit)
    int wins = 0;

    // Visits SOLO_U x 32 edges: lane's rows r (own < 0: none) of columns ent >> 16 of root ent & 0xffff.  The
    // claims of all SOLO_U are in flight together: each is a round trip to another block.
    auto visit = [&](const int (&own)[SOLO_U], const unsigned (&ent)[SOLO_U], const int (&r)[SOLO_U]) {
        int m[SOLO_U];
        unsigned got[SOLO_U];
        bool ask[SOLO_U], any_free = false;
#pragma unroll
        for (int u = 0; u < SOLO_U; ++u) {
            m[u] = own[u] >= 0 ? ((volatile u16*)rm)[r[u]] : -1;
            if (m[u] >= 0 && m[u] != SOLO_FREE && !bmd::idx_ok(p, m[u], nc)) m[u] = -1;  // checked build only
        }
#pragma unroll
        for (int u = 0; u < SOLO_U; ++u) {
            const bool matched = m[u] >= 0 && m[u] != SOLO_FREE;
            em += matched;
            any_free |= m[u] == SOLO_FREE;
            ask[u] = matched && !bmd::sb_test(vis, m[u]);
        }
#pragma unroll
        for (int u = 0; u < SOLO_U; ++u) {
            const unsigned w = (unsigned)m[u] >> 5, bit = 1u << (m[u] & 31);
            got[u] = ~0u;
            if (ask[u]) got[u] = C == 1 ? atomicOr(&vis[w], bit) : dor(at<C>(s_vis + 4 * w, (int)(w & (C - 1))), bit);
        }
#pragma unroll
        for (int u = 0; u < SOLO_U; ++u) {
            if (!ask[u]) continue;
            const unsigned w = (unsigned)m[u] >> 5, bit = 1u << (m[u] & 31);
            const int o = (int)(w & (C - 1));
            if (C > 1 && o != rank) atomicOr(&vis[w], bit);
            if (got[u] & bit) continue;
            ++wins;
            const unsigned fw = (unsigned)(step & 1) * lay.own_cw + w / C;
            if (C == 1) {
                pr[m[u]] = ent[u];
                atomicOr(&fresh[fw], bit);
            } else {
                dst32(at<C>(s_pr + 4u * slot_of<C>(m[u]), o), ent[u]);
                dred_or(at<C>(s_fresh + 4u * fw, o), bit);
            }
        }
        if (!__any_sync(FULL, any_free)) return;
        // unmatched rows: a path of the column's root ends here
#pragma unroll
        for (int u = 0; u < SOLO_U; ++u) {
            ask[u] = m[u] == SOLO_FREE && !bmd::sb_test(srv, (int)(ent[u] & 0xffffu));
            const unsigned rbit = 1u << (r[u] & 31);
            got[u] = ~0u;
            if (ask[u]) got[u] = dor(at<C>(s_rcl + 4u * (((unsigned)r[u] >> 5) / C), owner<C>(r[u])), rbit) & rbit;
        }
#pragma unroll
        for (int u = 0; u < SOLO_U; ++u) {
            if (got[u] != 0u) continue;  // not asked, or the row is claimed
            const int rt = (int)(ent[u] & 0xffffu), o = owner<C>(rt);
            const unsigned sbit = 1u << (rt & 31), sw = 4u * ((unsigned)rt >> 5);
            if (!(dor(at<C>(s_srv + sw, o), sbit) & sbit)) {
#pragma unroll 1
                for (int k = 0; k < C; ++k)
                    if (k != o) dred_or(at<C>(s_srv + sw, k), sbit);
                // the root keeps the row as its parent and the column that reached it as its match
                dst32(at<C>(s_pr + 4u * slot_of<C>(rt), o), (unsigned)r[u] << 16 | (unsigned)rt);
                dst16(at<C>(s_cm + 2u * slot_of<C>(rt), o), (int)(ent[u] >> 16));
                atomicAdd(&sm.mine.eps, 1);
            } else {  // root served meanwhile: give the row back
                dred_and(at<C>(s_rcl + 4u * (((unsigned)r[u] >> 5) / C), owner<C>(r[u])), ~(1u << (r[u] & 31)));
            }
        }
    };

#ifdef BM_CHECKED
    // Between phases, as step_check_matching: this block's copy of the rows' matches against the columns', wherever
    // they are, and its own columns' against the copy.  The next phase's levels write a served root's match.
    int checks = 0;
    auto check_matching = [&]() {
        bool bad = false;
        for (int r = t; r < nr; r += T) {
            const int c = rm[r];
            if (c != SOLO_FREE && (c >= nc || dld16(at<C>(s_cm + 2u * slot_of<C>(c), owner<C>(c))) != r)) bad = true;
        }
        for (int ow = warp; ow < (int)lay.own_cw; ow += T / 32) {
            const int c = (ow * C + rank) * 32 + lane, r = cm[ow * 32 + lane];
            if (c < nc && r != SOLO_FREE && (r >= nr || rm[r] != c)) bad = true;
        }
        if (bad && p.chk) atomicCAS(p.chk, 0, -11 /*BM_ERR_CHECK*/);
        ++checks;
        __syncthreads();
        cluster_sync<C>();
    };
#endif

    while (status == 0) {
        if (n_roots == 0) { no_roots = 1; break; }
        if (phases >= p.max_phases) {
            status = p.phase_limit_is_error ? -4 /*BM_ERR_ITER_LIMIT*/ : 1 /*BM_INCOMPLETE*/;
            break;
        }
        ++phases;
        // ---- BFS levels
        int tail = n_front, level = 0, eps = 0;
        for (;;) {
            // a narrow level's columns are dealt to all warps: a warp's time is its chain of instructions
            int width = 32;
            while (width > 1 && nl <= width / 2 * (T / 32)) width >>= 1;
            for (int g = warp * width; g < nl; g += width * (T / 32)) {  // warp-uniform
                int beg = 0, deg = 0;
                unsigned e = 0;
                if (lane < width && g + lane < nl) {
                    const int sl = (int)(list[g + lane] & 0xffffu), off = (int)(list[g + lane] >> 16) * PART;
                    if (bmd::idx_ok(p, sl, 32 * lay.own_cw) && bmd::idx_ok(p, pr[sl] & 0xffffu, nc)) {
                        e = (unsigned)((((sl >> 5) * C + rank) << 5) | (sl & 31)) << 16 | (pr[sl] & 0xffffu);
                        beg = col_beg[sl] + off;
                        deg = min(col_deg[sl] - off, PART);
                        if (bmd::sb_test(srv, (int)(e & 0xffffu))) deg = 0;  // Algorithm 4: root already served
                        else if (off == 0) ++cols;
                    }
                }
                int incl = deg;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int v = __shfl_up_sync(FULL, incl, d);
                    if (lane >= d) incl += v;
                }
                const int total = __shfl_sync(FULL, incl, 31), start = incl - deg;
                const int rk = __popc(__ballot_sync(FULL, deg > 0) & ((1u << lane) - 1));
                __syncwarp();  // the previous group's reads of the slots are done
                if (deg > 0) {
                    sm.base[wb + rk] = beg - start;
                    sm.ent[wb + rk] = e;
                }
                __syncwarp();
                if (lane == 0) edges += (unsigned)total;
                int before = 0;  // columns with edges that start before the current 32 edges
                for (int j0 = 0; j0 < total; j0 += 32 * SOLO_U) {
                    int own[SOLO_U], r[SOLO_U];
                    unsigned ent[SOLO_U];
#pragma unroll
                    for (int u = 0; u < SOLO_U; ++u) {
                        const int J0 = j0 + 32 * u;  // warp-uniform
                        own[u] = -1;
                        r[u] = 0;
                        ent[u] = 0u;
                        if (J0 >= total) continue;
                        const unsigned starts = __reduce_or_sync(
                            FULL, (deg > 0 && start >= J0 && start < J0 + 32) ? 1u << (start - J0) : 0u);
                        if (J0 + lane < total) {
                            own[u] = wb + before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
                            const int i = sm.base[own[u]] + J0 + lane;
                            r[u] = i < ROW_GLOBAL ? (int)rows[i] : __ldg(&p.row_idx[i - ROW_GLOBAL]);
                            ent[u] = sm.ent[own[u]];
                            if (!bmd::idx_ok(p, r[u], nr)) { own[u] = -1; r[u] = 0; }
                        }
                        before += __popc(starts);
                    }
                    visit(own, ent, r);
                }
            }
            wins = __reduce_add_sync(FULL, wins);
            if (lane == 0 && wins) atomicAdd(&sm.mine.cnt, wins);
            wins = 0;
            // the launch's limit, after a phase (below) and within it at every 16th level: a long path's are thousands.
            // It ends the phase in the columns' count, which every block looks at anyway (a flag of its own, read at
            // each level, cost a search 2%), and the warp that tests it is the last to get columns.
            if (rank == 0 && t == T - 1 && (level & 15) == 15 && bmd::globaltimer() > deadline) atomicAdd(&sm.mine.cnt, TIMED_OUT);
            end_step(false);
            ++level;
            eps += sum_eps;
            if (leader) {
                sm.st.ins += sum_cnt;
                if (sum_eps > 0) {
                    if (sm.st.first_ep == 0) sm.st.first_ep = level;
                    sm.st.last_ep = level;
                }
            }
            tail += sum_cnt;
            if (sum_cnt <= 0) break;  // no vertex inserted, or out of time
            if (carry && eps > 0 && phases <= bmd::CUT_PHASES && level >= bmd::CUT_MIN && level <= bmd::CUT_MAX &&
                sum_cnt * bmd::CUT_RATIO <= tail)
                break;
        }
        if (sum_cnt < 0) {
            status = -5 /*BM_ERR_TIMEOUT*/;
            break;
        }
        if (leader) {
            SoloStats& g = sm.st;
            g.levels += level;
            if (level > g.levels_max) g.levels_max = level;
            g.eps += eps;
            g.roots += n_roots;
            g.last_eps = eps;
            if (p.profile && phases <= p.profile_cap) {
                int32_t* prof = p.profile + 4 * (phases - 1);
                prof[0] = level; prof[1] = eps; prof[2] = g.first_ep; prof[3] = g.last_ep;
            }
            g.first_ep = g.last_ep = 0;
        }
        if (eps == 0) break;  // no augmenting path: the matching is maximum (Berge)
        if (phases >= bmd::CARRY_PHASES) carry = false;
        int kept = 0;
        for (int ow = warp; ow < (int)lay.own_cw; ow += T / 32) {
            const int w = ow * C + rank, sl = ow * 32 + lane, me = w * 32 + lane;
            if (w >= words) continue;  // warp-uniform
            const unsigned v = vis[w], in_tree = v >> lane & 1u;
            const int rt = (int)(pr[sl] & 0xffffu);
            // ---- Alternate: from a served root's endpoint back to the root (disjoint trees)
            if (srv[w] >> lane & 1u) {
                int r = (int)(pr[sl] >> 16), c = cm[sl];
                for (int steps = 0;; ++steps) {
                    if (steps > tail || c >= nc || r >= nr) { sm.mine.flag = -4 /*BM_ERR_ITER_LIMIT*/; break; }
                    const unsigned mc = at<C>(s_cm + 2u * slot_of<C>(c), owner<C>(c));
                    const int r2 = dld16(mc);
                    const int c2 = (int)(dld32(at<C>(s_pr + 4u * slot_of<C>(c), owner<C>(c))) >> 16);
                    dst16(mc, r);
#pragma unroll 4
                    for (int k = 0; k < C; ++k) dst16(at<C>(s_rm + 2u * r, k), c);
                    ++alt;
                    if (c == me) break;
                    r = r2;
                    c = c2;
                }
            }
            __syncwarp();
            // ---- kept trees (or only the roots left) stay; the others' columns are free to claim
            const unsigned keep = __ballot_sync(FULL, in_tree && !bmd::sb_test(srv, rt) && (carry || me == rt));
            if (lane == 0) {
                vis[w] = keep;
                fresh[(step & 1) * (int)lay.own_cw + ow] = keep;
            }
            kept += __popc(keep);
        }
        if (lane == 0 && kept) atomicAdd(&sm.mine.cnt, kept);
        __syncthreads();
        for (int w = t; w < words; w += T) srv[w] = 0u;
        for (int w = t; w < (int)((lay.cm - lay.rcl) >> 2); w += T) rcl[w] = 0u;
        if (leader && bmd::globaltimer() > deadline) sm.mine.flag = -5 /*BM_ERR_TIMEOUT*/;
        end_step(true);
#ifdef BM_CHECKED
        check_matching();
#endif
        n_front = sum_cnt;
        status = flag;
        n_roots -= eps;
        n_free -= eps;
    }
    // ---- results: every block its own words
    if (status >= 0 && status != SOLO_PASS) {
        for (int w = rank + C * warp; w < (nr + 31) >> 5; w += C * (T / 32)) {
            const int r = w * 32 + lane;
            if (r < nr) {
                const int c = rm[r] == SOLO_FREE ? -1 : rm[r];
                p.rmatch[r] = c;
                if (a.rm_out) a.rm_out[r] = c;
            }
        }
        for (int w = rank + C * warp; w < words; w += C * (T / 32)) {
            const int c = w * 32 + lane;
            if (c < nc) {
                const int v = cm[slot_of<C>(c)], r = v == SOLO_FREE ? -1 : v;
                p.cmatch[c] = r;
                if (a.cm_out) a.cm_out[c] = r;
            }
        }
    }
    block_add(&sm.sum[0], cols);
    block_add(&sm.sum[1], edges);
    block_add(&sm.sum[2], em);
    block_add(&sm.sum[3], alt);
    cluster_sync<C>();
    if (rank == 0 && t < 4) {  // the other blocks' counters
        unsigned long long v = 0;
        for (int k = 0; k < C; ++k) {
            const unsigned s = at<C>(saddr(&sm.sum[t]), k);
            v += (unsigned long long)dld32(s) | (unsigned long long)dld32(s + 4) << 32;
        }
        __syncwarp(0xfu);
        sm.sum[t] = v;
        __syncwarp(0xfu);
        if (t == 0) {
            Ctl c{};
            const int chk = bmd::ld_volatile(&p.ctl->err);  // range-checked build, or the input checks
            c.err = status < 0 ? status : 0;
            if (c.err == 0) c.err = chk;
            c.status = c.err ? c.err : status;
            c.card = nc - n_free;
            c.initial_card = initial;
            c.phases = phases + no_roots;
            c.searches = phases;
            c.n_endpoints_last = sm.st.last_eps;
            c.levels = sm.st.levels;
            c.max_levels = sm.st.levels_max;
            c.cols_expanded = (long long)sm.sum[0];
            c.edges_scanned = (long long)sm.sum[1];
            c.edges_matched = (long long)sm.sum[2];
            c.alt_steps = (long long)sm.sum[3];
            c.endpoints = sm.st.eps;
            c.inserted = sm.st.ins;
            c.roots = sm.st.roots;
            c.kernel_ns = (long long)(bmd::globaltimer() - t_start);
#ifdef BM_CHECKED
            c.checks = checks;
#endif
            *p.ctl = c;
            *a.h_ctl = c;
        }
    }
    cluster_sync<C>();  // no block leaves while another reads its shared memory
}

// The cheap matching of a small graph in one launch (launch_greedy's rules): the
// rows' states in their owners' shared memory, the columns by degree, columns of
// more than GREEDY_LIGHT rows a warp each from the block's list.  Adds to the
// installed matching; |M| goes to the control block and the host's copy.
template <int C, int T>
__global__ void __launch_bounds__(T, 1) k_solo_greedy(Params p, const int32_t* __restrict__ rdeg, Ctl* h_ctl, int check_err,
                                                     int crowded) {
    using namespace bmd;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ int s_card, s_long;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nr = p.nr, nc = p.nc;
    const int rank = my_rank<C>();
    int32_t* const state = (int32_t*)dyn;                          // own rows
    const unsigned s_state = saddr(state);
    const int own_tiles = (((nc + 31) >> 5) + C - 1) / C;
    int32_t* const longs = (int32_t*)p.queue + rank * own_tiles * 32;  // (the queue holds 2 nc words)
    // an invalid CSR is not read (the same in every block: nothing writes the word then)
    const int err = check_err ? ld_volatile(&p.ctl->err) : 0;
    if (err != 0) return;
#ifdef BM_CHECKED
    if (!check_err && rank == 0 && t == 0) p.ctl->err = 0;
#endif
    if (t == 0) s_card = s_long = 0;
    __syncthreads();
    int n = 0;
    for (int w = rank + C * warp; w < (nr + 31) >> 5; w += C * (T / 32)) {
        const int r = w * 32 + lane;
        if (r >= nr) continue;
        const bool is_free = p.rmatch[r] == -1;
        state[slot_of<C>(r)] = is_free ? rdeg[r] : GREEDY_TAKEN;
        n += !is_free;
    }
    cluster_sync<C>();
    // a block's columns: every C-th tile of 32, in a scattered order
    const int bits = own_tiles > 1 ? 32 - __clz(own_tiles - 1) : 0;  // 2^bits >= own_tiles
    auto state_at = [&](int r) { return at<C>(s_state + 4u * slot_of<C>(r), owner<C>(r)); };
    auto state_of = [&](int r) { return idx_ok(p, r, nr) ? (int)dld32(state_at(r)) : GREEDY_TAKEN; };
    auto take = [&](int r, int seen) { return dcas(state_at(r), seen, GREEDY_TAKEN) == seen; };
    const int limit[4] = {0, 2, 8, GREEDY_LIGHT};
    const bool any = crowded && nc > 2LL * nr;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        for (unsigned k0 = warp; k0 < (1u << bits); k0 += T / 32) {
            const int own = (int)scatter_bits(k0, bits);
            if (own >= own_tiles) continue;
            const int c = scatter_lane((unsigned)(own * C + rank), lane);
            if (c >= nc) continue;
            const int beg = __ldg(&p.col_ptr[c]), deg = __ldg(&p.col_ptr[c + 1]) - beg;
            if (k == 0 && deg > GREEDY_LIGHT) longs[atomicAdd(&s_long, 1)] = c;
            if (deg <= limit[k] || deg > limit[k + 1] || p.cmatch[c] != -1) continue;
            const int rot = (int)__umulhi(hash32((unsigned)c), (unsigned)deg);
            const int r = greedy_thread<4>(p.row_idx + beg, deg, rot, c, any, state_of, take);
            if (r >= 0) {
                p.rmatch[r] = c;
                p.cmatch[c] = r;
                ++n;
            }
        }
        cluster_sync<C>();
    }
    for (int k = warp; k < s_long; k += T / 32) {  // warp-uniform
        const int c = longs[k];
        if (p.cmatch[c] != -1) continue;
        const int beg = __ldg(&p.col_ptr[c]), deg = __ldg(&p.col_ptr[c + 1]) - beg;
        const int r = greedy_warp(p.row_idx + beg, deg, c, hash32((unsigned)c), crowded != 0, state_of, take);
        if (r >= 0 && lane == 0) {
            p.rmatch[r] = c;
            p.cmatch[c] = r;
            ++n;
        }
    }
    n = __reduce_add_sync(FULL, n);
    if (lane == 0 && n) dred_add(at<C>(saddr(&s_card), 0), n);
    cluster_sync<C>();
    if (rank == 0 && t == 0) {
        Ctl c{};
        c.card = s_card;
#ifdef BM_CHECKED
        c.err = ld_volatile(&p.ctl->err);
#endif
        *p.ctl = c;
        *h_ctl = c;
    }
}

}  // namespace bms1
