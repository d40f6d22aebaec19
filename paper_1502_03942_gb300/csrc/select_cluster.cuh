// select_cluster.cuh — selection by a cluster of thread blocks that exchange
// through distributed shared memory: the pivots of the first level (k_plan) and
// the exact finish (k_finish) of topk_select.
//
// Both select elements of given ranks by narrowing a window of composites: a
// histogram of the window's elements over equal bins, counted by every block in
// its own shared memory; one cluster barrier; every block sums all blocks'
// bins, finds the bin that holds the rank and takes it as the next window,
// until the bin holds few enough elements to be gathered and ranked by
// counting.  Each step costs one cluster barrier, whatever the number of
// elements, and needs no trip to global memory.
//
// What bounds them is latency (a few thousand elements per block): eight blocks
// of 1024 threads hold the 16384 draws of a sample at two per thread, and the
// finisher's candidates at up to sixteen, where one block walked 16 draws per
// thread in every pass over the sample.
#pragma once

#include "select_block.cuh"

namespace topk {

constexpr int CL_BLOCKS = 8;      // blocks per cluster (the portable limit)
constexpr int CL_NT = 1024;       // threads per block
constexpr u32 CL_BITS = 10;
constexpr u32 CL_BINS = 1u << CL_BITS; // one bin per thread in the scan
constexpr int CL_STEPS = 12;      // a window of 96 bits shrinks to one composite in ten steps
constexpr u32 CL_GATHER = 128;    // elements ranked by counting
static_assert(CL_BINS == CL_NT, "one bin per thread");

// ------------------------------------------------- cluster primitives

__device__ __forceinline__ u32 cl_rank() {
    u32 r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Barrier among all threads of the cluster; shared-memory accesses before it,
// local or remote, are visible after it.
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The same barrier in two halves.
__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// The barrier of the `nct` blocks that work on a selection: a cluster's, or one
// block alone.
__device__ __forceinline__ void cl_sync(u32 nct) {
    if (nct == 1) __syncthreads();
    else cl_sync();
}
// Address of block `rank`'s copy of the shared variable at `p`.
__device__ __forceinline__ u32 cl_map(const void* p, u32 rank) {
    u32 r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ u32 cl_ld(u32 addr) {
    u32 v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cl_st(u32 addr, u32 v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_st(u32 addr, u64 v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cl_st(u32 addr, u128 v) {
    cl_st(addr, (u64)v);
    cl_st(addr + 8, (u64)(v >> 64));
}
__device__ __forceinline__ u32 cl_atomic_add(u32 addr, u32 v) {
    u32 old;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}

// ------------------------------------------------------ window narrowing

// Shared memory of the narrowing (NTGT ranks at once), in every block.
template <int KW, int NTGT> struct ClSel {
    typedef typename Comp<KW>::t ct;
    u32 hist[2][NTGT][CL_BINS]; // by step parity
    u32 range[CL_STEPS * NTGT + 1][2]; // smallest and largest leading word over all blocks, by use
    ct gath[NTGT][CL_GATHER];
    ct res[NTGT];
    u32 wsum[CL_NT / 32];
    u32 bin[NTGT], below[NTGT], cnt[NTGT];
    u32 total;                  // elements in the first window
    u32 ng[NTGT];               // the first block's: elements gathered
};

// Clears what a selection starts from (before a block barrier).
template <int KW, int NTGT> __device__ __forceinline__ void cl_clear(ClSel<KW, NTGT>& s) {
    for (u32 i = threadIdx.x; i < 2 * NTGT * CL_BINS; i += CL_NT) (&s.hist[0][0][0])[i] = 0;
    if (threadIdx.x < NTGT) s.ng[threadIdx.x] = 0;
    if (threadIdx.x < 2 * (CL_STEPS * NTGT + 1)) (&s.range[0][0])[threadIdx.x] = threadIdx.x & 1u ? 0u : 0xFFFFFFFFu;
}

// The smallest and largest word over all threads of the blocks (all ones and
// zero where no thread has one), through range[use]; each use once.  Ends with a
// barrier of the blocks; cl_clear and another before.
template <int KW, int NTGT>
__device__ __forceinline__ void cl_range(ClSel<KW, NTGT>& s, u32 nct, int use, u32& mn, u32& mx) {
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    const u32 lane = lane_id(), r = lane >> 1;
    if (r < nct) { // lanes 2r and 2r + 1 tell block r
        if (lane & 1u) asm volatile("red.shared::cluster.max.u32 [%0], %1;" ::"r"(cl_map(&s.range[use][1], r)), "r"(mx) : "memory");
        else asm volatile("red.shared::cluster.min.u32 [%0], %1;" ::"r"(cl_map(&s.range[use][0], r)), "r"(mn) : "memory");
    }
    cl_sync(nct);
    mn = s.range[use][0];
    mx = s.range[use][1];
}
// The leading word of a composite, and the window of the words mn..mx.
template <int KW> __device__ __forceinline__ u32 lead_word(typename Comp<KW>::t c) { return (u32)(c >> KW); }
template <int KW>
__device__ __forceinline__ void lead_window(u32 mn, u32 mx, typename Comp<KW>::t& lo, typename Comp<KW>::t& hi) {
    typedef typename Comp<KW>::t ct;
    lo = (ct)mn << KW;
    hi = ((ct)mx << KW) | (((ct)1 << KW) - 1);
}

// The elements of 0-based ranks rk[t] (duplicates counted) among all blocks'
// elements inside the windows [wlo[t], whi[t]] that hold them.  each(f) calls
// f(c) for this thread's elements (the same ones every time).  `total`
// receives the number of elements in the first window.  When TO_ALL every
// block gets the result, else the cluster's first block alone; that block's
// `res` holds it.  Precondition: cl_clear, then a barrier.  False when the
// ranks do not lie in the windows (the counts passed in were wrong).
template <int KW, int NTGT, bool TO_ALL, class Each>
__device__ bool cl_select(ClSel<KW, NTGT>& s, u32 nct, Each each, typename Comp<KW>::t (&wlo)[NTGT],
                          typename Comp<KW>::t (&whi)[NTGT], u32 (&rk)[NTGT], u32& total) {
    typedef typename Comp<KW>::t ct;
    const u32 tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    u32 cnt[NTGT];
    total = 0;
    int step = 0;
    while (true) {
        u32 sh[NTGT];
        bool split = false; // the two windows differ: two histograms
#pragma unroll
        for (int t = 0; t < NTGT; ++t) {
            const int bl = bit_length_fast((ct)(whi[t] - wlo[t]));
            sh[t] = bl > (int)CL_BITS ? (u32)(bl - CL_BITS) : 0u;
            if (t > 0) split = wlo[t] != wlo[0] || whi[t] != whi[0];
        }
        u32(*h)[CL_BINS] = s.hist[step & 1];
        each([&](ct c) {
            if (c >= wlo[0] && c <= whi[0]) atomicAdd(&h[0][(u32)((ct)(c - wlo[0]) >> sh[0])], 1u);
            if (NTGT > 1 && split && c >= wlo[NTGT - 1] && c <= whi[NTGT - 1])
                atomicAdd(&h[NTGT - 1][(u32)((ct)(c - wlo[NTGT - 1]) >> sh[NTGT - 1])], 1u);
        });
        if (tid < NTGT) s.cnt[tid] = 0;
        cl_sync(nct);
        // every block sums the bins of all (thread b: bin b) and finds the ranks'
#pragma unroll
        for (int t = 0; t < NTGT; ++t) {
            u32 hv = 0, incl = 0;
            if (t == 0 || split) {
                u32 part[CL_BLOCKS]; // all loads in flight
#pragma unroll
                for (u32 r = 0; r < CL_BLOCKS; ++r) part[r] = r < nct ? cl_ld(cl_map(&h[t][tid], r)) : 0u;
#pragma unroll
                for (u32 r = 0; r < CL_BLOCKS; ++r) hv += part[r];
                incl = hv;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= (u32)o) incl += y;
                }
                if (lane == 31) s.wsum[warp] = incl;
                __syncthreads();
                u32 base = lane < warp ? s.wsum[lane] : 0u;
                base = __reduce_add_sync(0xffffffffu, base);
                incl += base;
            }
            const u32 excl = incl - hv;
            auto mark = [&](int q) {
                if (hv && rk[q] >= excl && rk[q] < incl) {
                    s.bin[q] = tid;
                    s.below[q] = excl;
                    s.cnt[q] = hv;
                }
            };
            if (t == 0) {
                mark(0);
                if (NTGT > 1 && !split) mark(NTGT - 1);
                if (tid == CL_NT - 1) s.total = incl;
            } else if (split) {
                mark(t);
            }
            __syncthreads();
        }
        if (step == 0) total = s.total;
        bool small = true;
#pragma unroll
        for (int t = 0; t < NTGT; ++t) {
            cnt[t] = s.cnt[t];
            if (cnt[t] == 0) return false; // the same in every block: all read the same counts
            const ct nlo = (ct)(wlo[t] + ((ct)s.bin[t] << sh[t]));
            const ct top = (ct)(nlo + (((ct)1 << sh[t]) - 1));
            whi[t] = (top > whi[t] || top < nlo) ? whi[t] : top;
            wlo[t] = nlo;
            rk[t] -= s.below[t];
            small = small && (cnt[t] <= CL_GATHER || wlo[t] == whi[t]);
        }
        ++step;
        if (small) break;
        if (step >= CL_STEPS) return false;
        // many elements in one bin (ties, or clusters): their own range, so that
        // the next step's bins are not spent on values that none of them has
#pragma unroll
        for (int t = 0; t < NTGT; ++t) {
            if (cnt[t] <= CL_GATHER || (t > 0 && wlo[t] == wlo[0])) continue;
            const ct lo = wlo[t], hi = whi[t];
            const int bl = bit_length_fast((ct)(hi - lo));
            const u32 s2 = bl > 32 ? (u32)(bl - 32) : 0u;
            u32 mn = 0xFFFFFFFFu, mx = 0;
            each([&](ct c) {
                if (c >= lo && c <= hi) {
                    const u32 w = (u32)((ct)(c - lo) >> s2);
                    mn = min(mn, w);
                    mx = max(mx, w);
                }
            });
            cl_range(s, nct, 1 + (step - 1) * NTGT + t, mn, mx);
            const ct nlo = (ct)(lo + ((ct)mn << s2)), nhi = (ct)(lo + ((ct)mx << s2) + (((ct)1 << s2) - 1));
            if (NTGT > 1 && t == 0 && wlo[NTGT - 1] == lo) {
                wlo[NTGT - 1] = nlo;
                whi[NTGT - 1] = nhi < hi ? nhi : hi;
            }
            wlo[t] = nlo;
            whi[t] = nhi < hi ? nhi : hi;
        }
        // the other parity's bins were read before this step's cluster barrier
        for (u32 i = tid; i < NTGT * CL_BINS; i += CL_NT) (&s.hist[step & 1][0][0])[i] = 0;
        __syncthreads();
    }
    // gather the bins' elements and rank them by counting
    const bool split = NTGT > 1 && (wlo[NTGT - 1] != wlo[0] || whi[NTGT - 1] != whi[0]);
    each([&](ct c) {
#pragma unroll
        for (int t = 0; t < NTGT; ++t) {
            if ((t > 0 && !split) || c < wlo[t] || c > whi[t] || wlo[t] == whi[t]) continue;
            const u32 slot = cl_atomic_add(cl_map(&s.ng[t], 0), 1u);
            if (slot < CL_GATHER) {
                if (TO_ALL) {
#pragma unroll
                    for (u32 r = 0; r < CL_BLOCKS; ++r)
                        if (r < nct) cl_st(cl_map(&s.gath[t][slot], r), c);
                } else {
                    cl_st(cl_map(&s.gath[t][slot], 0), c);
                }
            }
        }
    });
    cl_sync(nct);
    if (!TO_ALL && cl_rank() != 0) return true;
    // each target has CL_NT / NTGT threads, PARTS of them to an element: each
    // compares with its part of the others
    constexpr u32 PARTS = CL_NT / NTGT / CL_GATHER;
    const u32 t = tid / (CL_NT / NTGT), e = tid % (CL_NT / NTGT) / PARTS, q = tid % PARTS;
    constexpr int L = NTGT - 1;
    const ct my_lo = t ? wlo[L] : wlo[0];
    const u32 my_rk = t ? rk[L] : rk[0];
    const bool same = my_lo == (t ? whi[L] : whi[0]); // copies of one composite
    const ct* g = s.gath[split ? t : 0];
    const u32 n = same ? 0u : t ? cnt[L] : cnt[0];
    const ct v = e < n ? g[e] : (ct)0;
    u32 p = 0;
    for (u32 j = q; j < n; j += PARTS) {
        const ct o = g[j];
        p += (u32)(o < v || (o == v && j < e));
    }
#pragma unroll
    for (u32 o = 1; o < PARTS; o <<= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    if (e < n && q == 0 && p == my_rk) s.res[t] = v;
    if (same && e == 0 && q == 0) s.res[t] = my_lo;
    __syncthreads();
    return true;
}
static_assert(CL_NT / 2 >= (int)CL_GATHER, "at least one thread per gathered element of either rank");

// ----------------------------------------------------- pickPivots, level 1

// The candidates of the first level are also counted over HB_BINS equal bins
// of the bracket [pl, pr] while the pass emits them (BinHist,
// select_core.cuh), on composites whose position takes only as many bits as n
// needs.  Where the bracket is open below (above), the bins start somewhat below
// the sample's smallest (above its largest) element, because the ends of the key
// domain lie far from the data; elements outside count into the end bins.
template <int KW>
__device__ __forceinline__ typename Comp<KW>::t packed_comp(typename Comp<KW>::t c, u32 bn) {
    typedef Comp<KW> C;
    const u32 top = bn >= 32 ? 0xFFFFFFFFu : (1u << bn) - 1u;
    const u32 x = C::idx(c) < top ? C::idx(c) : top;
    return ((typename C::t)C::key(c) << bn) | x;
}
template <int KW>
__device__ __forceinline__ typename Comp<KW>::t unpacked_comp(typename Comp<KW>::t c, u32 bn) {
    typedef Comp<KW> C;
    const u32 top = bn >= 32 ? 0xFFFFFFFFu : (1u << bn) - 1u;
    return C::make((typename C::key_t)(c >> bn), (u32)c & top);
}

template <int KW> struct PlanSmem {
    ClSel<KW, 2> sel;
};

// Pivots of the first level (one cluster): every draw of the sample stays in
// the register of the thread that drew it.  Draw j falls in partition j mod p
// at a position uniform in it (Philox4x32-10 of counter 4 floor(j / 4), word
// j mod 4); the sample elements of ranks k|S|/n -/+ Delta are selected over the
// cluster.  Also clears the bins of the pass that follows.
//
// `first` = 0: pivots among the candidates that the passes so far have left, when
// they are more than the finish holds; returns at once otherwise, and where the window
// was narrowed on its source (every draw has to count).
//
// 12 us on 2^28 f32 keys, 16 where most of the sample ties with the pivots; a
// sampling kernel and a one-block pivot kernel that pass the sample through global
// memory take 17 and 30.
template <int DT> __global__ void __launch_bounds__(CL_NT) k_plan(SelArgs a, int first) {
    typedef Key<DT> K;
    constexpr int KW = K::KW;
    typedef Comp<KW> C;
    typedef typename C::t ct;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto& sel = reinterpret_cast<PlanSmem<KW>*>(smem_raw)->sel;
    // The barrier before the first remote access, in two halves: it also has to
    // cover the clearing, since a block that cleared late would wipe out what
    // another has already reduced into it.
    cl_clear(sel);
    cl_arrive();
    grid_dep_wait();
    grid_dep_release();
    constexpr u32 DPT = Lim<KW>::ELEMS / (CL_BLOCKS * CL_NT); // draws per thread
    static_assert(DPT >= 1 && DPT <= 4 && 4 % DPT == 0, "a thread's draws lie in one Philox block");
    const u32 gid = cl_rank() * CL_NT + threadIdx.x;
    const SelState* g = a.st;
    if (!first && (g->phase != PH_RUN || g->src == SRC_INPUT || g->m_win != g->m_src ||
                   g->m_src <= (u64)CL_BLOCKS * Lim<KW>::ELEMS))
        return;
    const u32 m = first ? (u32)a.n : (u32)g->m_src, draws = a.sample;
    const u64 k = first ? a.k : g->k_rem;
    const u32 level = first ? 0u : g->level, src_id = first ? (u32)SRC_INPUT : g->src;
    // (independent of the draws, whose loads it covers)
    long long jl, jr;
    pivot_ranks(draws, m, k, a.z, (a.flags & TOPK_FLAG_RAW_DELTA) != 0, jl, jr);
    const long long top = (long long)draws - 1;
    const u32 r1 = (u32)(jr < 0 ? 0 : jr > top ? top : jr);
    const u32 r0 = jl < 0 ? r1 : (u32)(jl > top ? top : jl); // (an unused lower rank follows the upper one)
    if (first && a.bins)
        for (u32 i = gid; i < HB_BINS; i += CL_BLOCKS * CL_NT) a.bins->h[i] = 0;
    ct c[DPT];
    const InputSrc<DT> src = InputSrc<DT>::make(a.keys, m);
    const CandSrc<KW> csrc{static_cast<const typename K::key_t*>(a.cand_key[src_id == SRC_CAND1 ? 1 : 0]),
                           a.cand_idx[src_id == SRC_CAND1 ? 1 : 0], m};
    {
        const u32 p = a.parts < m ? a.parts : m;
        const u32 len = m / p, rem = m - len * p;
        const u32 j0 = gid * DPT;
        const Philox4 r = philox4x32_10(j0 & ~3u, level, 0x53414D50u, 0, (u32)a.seed, (u32)(a.seed >> 32));
#pragma unroll
        for (u32 q = 0; q < DPT; ++q) {
            const u32 j = j0 + q;
            const u32 part = j % p;
            const u32 plo = part * len + (part < rem ? part : rem);
            const u32 psz = len + (part < rem ? 1 : 0);
            const u32 w = (j0 & 3u) + q;
            const u32 rv = w == 0 ? r.v[0] : w == 1 ? r.v[1] : w == 2 ? r.v[2] : r.v[3];
            const u32 pos = plo + (u32)(((u64)rv * psz) >> 32);
            typename K::key_t kq = 0;
            u32 x = 0;
            if (j < draws) {
                if (first) src.at(pos, kq, x);
                else csrc.at(pos, kq, x);
            }
            c[q] = C::make(kq, x);
        }
    }
    const u32 mine = gid * DPT < draws ? min(DPT, draws - gid * DPT) : 0u;
    u32 mn = 0xFFFFFFFFu, mx = 0;
#pragma unroll
    for (u32 q = 0; q < DPT; ++q) {
        if (q < mine) {
            mn = min(mn, lead_word<KW>(c[q]));
            mx = max(mx, lead_word<KW>(c[q]));
        }
    }
    cl_wait();
    ct wlo[2], whi[2], cmin, cmax;
    cl_range(sel, CL_BLOCKS, 0, mn, mx);
    lead_window<KW>(mn, mx, cmin, cmax);
    wlo[0] = wlo[1] = cmin;
    whi[0] = whi[1] = cmax;
    u32 rk[2] = {r0, r1}, total;
    const bool ok = cl_select<KW, 2, false>(sel, CL_BLOCKS, [&](auto f) {
#pragma unroll
        for (u32 q = 0; q < DPT; ++q)
            if (q < mine) f(c[q]);
    }, wlo, whi, rk, total);
    if (!ok) cl_sync(); // (the same in every block) no block leaves while others read its bins
    if (gid != 0) return;
    if (!first) { // arms the next pass over the candidates
        SelState* w = a.st;
        if (!ok) return; // (left to the finish)
        w->pl = jl >= 0 ? (u128)sel.res[0] : w->lo;
        w->pr = jr <= top ? (u128)sel.res[1] : w->hi;
        w->dst = src_id == SRC_CAND0 ? SRC_CAND1 : SRC_CAND0;
        w->cnt_a = 0;
        w->cnt_b = 0;
        w->dense = jl >= 0 && (jl + 1) * 16 > (long long)draws ? 1u : 0u;
        w->level = level + 1;
        w->levels_grid++;
        w->pending = 1;
        return;
    }
    SelState s = initial_state<DT>(a);
    const ct hi = C::from128(s.hi);
    const ct pl = jl >= 0 ? sel.res[0] : (ct)0, pr = jr <= top ? sel.res[1] : hi;
    s.pl = (u128)pl;
    s.pr = (u128)pr;
    s.pending = 1;
    s.level = 1;
    s.levels_grid = 1;
    s.sample_kept = draws;
    // many a-elements expected: the pass compacts whole tiles (an aligned
    // input's pass was chosen by the host, by the same rule)
    s.dense = a.first_dense >= 0 ? (u32)a.first_dense : (jl >= 0 && (jl + 1) * 16 > (long long)draws) ? 1u : 0u;
    ct b0 = packed_comp<KW>(jl >= 0 ? pl : cmin, a.idx_bits);
    ct b1 = packed_comp<KW>(jr <= top ? pr : cmax, a.idx_bits);
    if (jl < 0 || jr > top) {
        // about n / |S| elements lie beyond the sample's ends: the bins reach
        // four more brackets out, as far as the keys go
        const ct w = (ct)(b1 - b0) < (packed_comp<KW>(hi, a.idx_bits) >> 3) ? (ct)(b1 - b0) * 4 : (ct)0;
        if (jl < 0) b0 = b0 > w ? (ct)(b0 - w) : (ct)0;
        if (jr > top) b1 = packed_comp<KW>(hi, a.idx_bits) - b1 > w ? (ct)(b1 + w) : packed_comp<KW>(hi, a.idx_bits);
    }
    const int bl = bit_length_fast((ct)(b1 - b0));
    if (a.bins) {
        a.bins->base = (u128)b0;
        a.bins->shift = bl > (int)HB_BITS ? (u32)(bl - HB_BITS) : 0u;
    }
    if (!ok) {
        s.status = ST_EINTERNAL;
        s.phase = PH_ERROR;
        latch(a.err, ST_EINTERNAL);
    }
    *a.st = s;
}

// ------------------------------------------------------------- the finish

// What is left of a source that one block of the cluster finishes alone: 8 us up
// to this size, where all of them take 12 for the same elements (their barriers
// and remote accesses).
constexpr u32 FIN_SOLO = 4096;

template <int KW> struct FinSmem {
    typedef typename Comp<KW>::t ct;
    ct list[Lim<KW>::ELEMS]; // the block's share of the undecided elements
    ClSel<KW, 1> sel;
    u32 kept, over, nout;
};

// The exact finish (one cluster): the undecided elements (those of the source
// inside the window) are dealt out to the blocks and kept in shared memory,
// the one of rank k_rem is selected over the cluster, and every element not
// above it is written.  Where they do not fit (the levels before it failed twice,
// or their candidates cluster on few values) the source is streamed instead:
// twice a step, to count and for the bin's own range, then to gather and to
// write, about twenty times at most and usually five, at 40 us for 4e6 elements
// each.  `first`: the call's only kernel, the source is the input.
//
// 11.4 us for 12345 keys and 9 to 13 us at the end of a selection from 2^25 or more
// keys; one block that holds 16384 elements and samples again above that takes 13.0
// and 11 to 20.
template <int DT> __global__ void __launch_bounds__(CL_NT) k_finish(SelArgs a, int first) {
    grid_dep_wait();
    grid_dep_release();
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef typename K::key_t key_t;
    constexpr int KW = K::KW;
    typedef Comp<KW> C;
    typedef typename C::t ct;
    constexpr u32 CAP = Lim<KW>::ELEMS;
    constexpr u32 OWN = CAP / CL_NT; // list elements of one thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto& sm = *reinterpret_cast<FinSmem<KW>*>(smem_raw);
    const u32 tid = threadIdx.x, rank = cl_rank();
    SelState* g = a.st;
    const struct {
        u128 lo, hi;
        u64 m_src, m_win, k_rem, out_base;
        u32 src;
    } s = {first ? (u128)0 : g->lo, first ? key_domain_max<DT>() : g->hi,
           first ? a.n : g->m_src, first ? a.n : g->m_win, first ? a.k : g->k_rem, first ? 0 : g->out_base,
           first ? (u32)SRC_INPUT : g->src};
    if (!first && g->phase != PH_RUN) return; // finished, or an error
    const ct lo = C::from128(s.lo), hi = C::from128(s.hi);
    const u64 m = s.m_src;
    // a short source is one block's: the barriers of a cluster cost more
    const u32 nct = m <= FIN_SOLO ? 1u : (u32)CL_BLOCKS;
    if (rank >= nct) return;
    const u32 k_rem = (u32)s.k_rem;
    const InputSrc<DT> isrc = InputSrc<DT>::make(a.keys, m);
    const CandSrc<KW> csrc{static_cast<const key_t*>(a.cand_key[s.src == SRC_CAND1 ? 1 : 0]),
                           a.cand_idx[s.src == SRC_CAND1 ? 1 : 0], m};
    cl_clear(sm.sel);
    if (tid == 0) {
        sm.kept = 0;
        sm.over = 0;
        sm.nout = 0;
    }
    // (blocks of one cluster may start apart: no remote access before all have)
    cl_sync(nct);
    constexpr int U = 8; // loads in flight per thread
    const u64 stride = (u64)nct * CL_NT;
    auto load = [&](u64 base, ct (&cv)[U]) -> u32 {
        u32 keep = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u64 i = base + (u64)u * stride + (u64)rank * CL_NT + tid;
            key_t kv = 0;
            u32 x = 0;
            if (i < m) {
                if (s.src == SRC_INPUT) isrc.at(i, kv, x);
                else csrc.at(i, kv, x);
            }
            cv[u] = C::make(kv, x);
            keep |= (u32)(i < m && cv[u] >= lo && cv[u] <= hi) << u;
        }
        return keep;
    };
    const bool try_list = s.m_win <= (u64)nct * CAP;
    u32 mn = 0xFFFFFFFFu, mx = 0;
    if (try_list) {
        for (u64 base = 0; base < m; base += stride * U) {
            ct cv[U];
            const u32 keep = load(base, cv);
            u32 slot = warp_reserve((u32)__popc(keep), &sm.kept);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if ((keep >> u) & 1u) {
                    mn = min(mn, lead_word<KW>(cv[u]));
                    mx = max(mx, lead_word<KW>(cv[u]));
                    if (slot < CAP) sm.list[slot] = cv[u];
                    ++slot;
                }
            }
        }
        __syncthreads();
        if (tid < nct && sm.kept > CAP) cl_st(cl_map(&sm.over, tid), 1u); // told to every block
    }
    // a window open at an end of the key domain says nothing about where the
    // elements lie: take their own range
    ct wlo[1] = {lo}, whi[1] = {hi};
    if (try_list && (lo == (ct)0 || hi == C::from128(key_domain_max<DT>()))) {
        ct l, u;
        cl_range(sm.sel, nct, 0, mn, mx);
        lead_window<KW>(mn, mx, l, u);
        wlo[0] = l > lo ? l : lo;
        whi[0] = u < hi ? u : hi;
    } else {
        cl_sync(nct);
    }
    const bool listed = try_list && !sm.over;
    if (!listed) {
        wlo[0] = lo;
        whi[0] = hi;
    }
    const u32 kept = sm.kept < CAP ? sm.kept : CAP;
    u32 rk[1] = {k_rem - 1}, total;
    bool ok = s.k_rem >= 1 && s.k_rem <= s.m_win;
    ok = ok && cl_select<KW, 1, true>(sm.sel, nct, [&](auto f) {
        if (listed) {
#pragma unroll 4
            for (u32 i = tid; i < kept; i += CL_NT) f(sm.list[i]);
        } else {
            for (u64 base = 0; base < m; base += stride * U) {
                ct cv[U];
                const u32 keep = load(base, cv);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if ((keep >> u) & 1u) f(cv[u]);
            }
        }
    }, wlo, whi, rk, total);
    ok = ok && total == s.m_win;
    const ct kth = sm.sel.res[0];
    raw_t* out_keys = static_cast<raw_t*>(a.out_keys) + s.out_base;
    u32* out_idx = a.out_idx + s.out_base;
    const u32 counter = cl_map(&sm.nout, 0);
    // room for a warp's selected elements, counted in the first block
    auto reserve = [&](u32 cnt) -> u32 {
        u32 incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane_id() >= (u32)o) incl += y;
        }
        u32 base = 0;
        if (lane_id() == 31 && incl) base = cl_atomic_add(counter, incl);
        return __shfl_sync(0xffffffffu, base, 31) + incl - cnt;
    };
    auto put = [&](u32 slot, ct c) {
        if (slot < k_rem) {
            out_keys[slot] = K::inv((key_t)C::key(c));
            out_idx[slot] = C::idx(c);
        }
    };
    if (ok && !a.kth_only) {
        if (listed) {
            u32 selm = 0;
#pragma unroll
            for (u32 u = 0; u < OWN; ++u) {
                const u32 i = u * CL_NT + tid;
                selm |= (u32)(i < kept && sm.list[i] <= kth) << u;
            }
            u32 slot = reserve((u32)__popc(selm));
            while (selm) {
                const u32 u = (u32)(__ffs(selm) - 1);
                selm &= selm - 1;
                put(slot++, sm.list[u * CL_NT + tid]);
            }
        } else {
            for (u64 base = 0; base < m; base += stride * U) {
                ct cv[U];
                u32 selm = load(base, cv);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (cv[u] > kth) selm &= ~(1u << u);
                u32 slot = reserve((u32)__popc(selm));
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if ((selm >> u) & 1u) put(slot++, cv[u]);
            }
        }
    }
    cl_sync(nct); // every reservation is in (and no block leaves while others reach into it)
    if (rank != 0 || tid != 0) return;
    if (first) init_state<DT>(g, a);
    if (!ok || (!a.kth_only && sm.nout != k_rem)) {
        g->status = ST_EINTERNAL;
        g->phase = PH_ERROR;
        latch(a.err, ST_EINTERNAL);
        return;
    }
    static_cast<raw_t*>(a.kth_key)[0] = K::inv((key_t)C::key(kth));
    a.kth_idx[0] = C::idx(kth);
    g->out_base = s.out_base + s.k_rem;
    g->phase = PH_DONE;
}

} // namespace topk
