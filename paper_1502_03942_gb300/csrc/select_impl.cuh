// select_impl.cuh — topk_select: selection of the k smallest of n unsorted keys
// (paper, Section 2, Algorithm "select"; Section 4.1, Theorem "selectFR").
//
// Launch sequence of one call (all on the caller's stream, no host round trip):
//   k_plan   (1 cluster) sample of the input; pivots = its elements of ranks
//                        k|S|/n -/+ Delta
//   first pass  (grid)   one read of the input: a -> output, b -> candidate
//                        buffer, the candidates also counted over equal bins;
//                        the last block takes the branch and, when more
//                        candidates are left than the finish holds, arms a
//                        second pass between the ends of rank k's bin
//   k_pass   (grid)      that second pass, over the candidates (usually a few
//                        thousand are left); returns at once when not armed
//   k_plan, k_pass       once more, when many candidates are expected: a level by
//                        sampling for candidates that the bins did not part
//   k_finish (1 cluster) selection of rank k among what is left, the rest of
//                        the output and the rank-k pair
// Inputs of at most T keys take one launch: k_small (1 block) up to SMALL_MAX keys,
// k_finish above.
// k_pass also plans for itself and reads the input again after a first level that
// failed (plan_here).  The bins give the second level exact counts for nothing and
// narrow by a factor of about 1000; a new sample narrows by 30 and takes 17 us.
// k = 1 (the base case of Algorithm "select", a global minimum) and k = n
// (everything selected) take one reduction kernel instead.
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>

#include "internal.h"
#include "select_cluster.cuh"

namespace topk {

// ------------------------------------------------------------- kernels

// Read-after-atomics: the pass counters as the last block of the pass sees them.
__device__ __forceinline__ u64 atomic_read(u64* p) {
    return atomicAdd(reinterpret_cast<unsigned long long*>(p), 0ull);
}

// What the finish's list holds: what is left undecided above this is planned and
// passed over once more.
template <int KW> constexpr u64 FIN_LIST = (u64)CL_BLOCKS * Lim<KW>::ELEMS;

// The branch of Algorithm "select", taken by the last block of a pass once
// every block's counts are in (block-done counter; nobody waits), and, after a
// first level that leaves more candidates than the finish takes at once, the pivots
// of a second pass: the ends of the bin that holds rank k (exact counts, so that
// pass cannot miss).  The bins also serve when there were more candidates than the
// buffer holds; the pass then reads the input again.  A bin that holds most of
// them (and more than the finish's list) is no bracket: ties, or clusters far
// apart.  The second pass then plans for itself (plan_here), above an eighth of
// them, or, where a level by sampling stands behind it, leaves them to that, above
// nine sixteenths: half of 2^24 f32 keys within 1e-6 of 1, the others about 1e20,
// k = 0.49 n, take 139 us, 233 with the bins alone.
// `planned`: the state of a pass that did so.  All NT threads call, after the
// block's own atomics.
struct EpilogueSmem {
    u32 last, arm, wsum[32];
};
template <int KW, int NT, class Sync, bool BINS>
__device__ __forceinline__ void pass_epilogue(const SelArgs& a, EpilogueSmem& es, const SelState* planned = nullptr) {
    typedef typename Comp<KW>::t ct;
    Sync::sync();
    if (threadIdx.x == 0) {
        __threadfence();
        es.last = atomicAdd(a.pass_done, 1u) == gridDim.x - 1;
    }
    Sync::sync();
    if (!es.last) return;
    SelState* g = a.st;
    if (threadIdx.x == 0) {
        __threadfence();
        g->cnt_a = atomic_read(&g->cnt_a);
        g->cnt_b = atomic_read(&g->cnt_b);
        if (planned) {
            g->pl = planned->pl;
            g->pr = planned->pr;
            g->dst = planned->dst;
            g->level = planned->level;
            g->levels_grid = planned->levels_grid;
            g->pending = 1;
        }
        decide(*g);
        *a.pass_done = 0;
        g->cnt_a = 0; // for a pass that plans for itself
        g->cnt_b = 0;
        es.arm = a.bins && g->m_win > a.list_max && g->phase == PH_RUN && (g->src != SRC_INPUT || g->overflows != 0);
    }
    if constexpr (BINS) {
        Sync::sync();
        if (!es.arm) return;
        constexpr u32 PER = HB_BINS / NT; // consecutive bins per thread
        static_assert(HB_BINS % NT == 0, "bins per thread");
        const u32 lane = lane_id(), warp = threadIdx.x >> 5;
        u32 h[PER], t = 0;
#pragma unroll
        for (u32 q = 0; q < PER; ++q) {
            h[q] = __ldcg(a.bins->h + threadIdx.x * PER + q);
            t += h[q];
        }
        u32 incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (u32)o) incl += y;
        }
        if (lane == 31) es.wsum[warp] = incl;
        Sync::sync();
        for (u32 w = 0; w < warp; ++w) incl += es.wsum[w];
        const u32 r = (u32)(*(volatile u64*)&g->k_rem - 1), nb = (u32) * (volatile u64*)&g->m_win;
        const u32 part = a.plan_follows ? nb / 16 * 9 : nb / 8;
        const u32 most = part > (u32)FIN_LIST<KW> ? part : (u32)FIN_LIST<KW>;
        u32 run = incl - t;
#pragma unroll
        for (u32 q = 0; q < PER; ++q) {
            if (h[q] && r >= run && r < run + h[q] && h[q] < nb && h[q] <= most && h[q] <= a.cap_b) { // one thread at most
                const u32 b = threadIdx.x * PER + q;
                const u32 sh = a.bins->shift;
                const ct base = Comp<KW>::from128(a.bins->base), lo = Comp<KW>::from128(g->lo), hi = Comp<KW>::from128(g->hi);
                // the end bins also hold what lies beyond them
                const ct l = unpacked_comp<KW>((ct)(base + ((ct)b << sh)), a.idx_bits);
                const ct u = unpacked_comp<KW>((ct)(base + (((ct)b + 1) << sh) - 1), a.idx_bits);
                g->pl = (u128)(b == 0 || l < lo ? lo : l);
                g->pr = (u128)(b == HB_BINS - 1 || u > hi || u < l ? hi : u);
                g->dst = g->src == SRC_CAND0 ? SRC_CAND1 : SRC_CAND0;
                // (the input also holds what lies below the window)
                g->dense = run + (g->src == SRC_INPUT ? g->out_base : 0) > g->m_src / 16 ? 1u : 0u;
                g->level += 1;
                g->levels_grid += 1;
                g->pending = 1;
            }
            run += h[q];
        }
    }
}

// ---- partition + reduction + branch (whole grid)

template <int DT>
__device__ __forceinline__ Sink<DT> make_sink(const SelArgs& a, const SelState& s) {
    typedef typename Key<DT>::raw_t raw_t;
    typedef typename Key<DT>::key_t key_t;
    Sink<DT> sink;
    sink.out_keys = static_cast<raw_t*>(a.out_keys);
    sink.out_idx = a.out_idx;
    sink.out_base = s.out_base;
    sink.cap_a = a.kth_only ? 0 : s.k_rem;
    sink.ck = static_cast<key_t*>(a.cand_key[s.dst - 1]);
    sink.ci = a.cand_idx[s.dst - 1];
    sink.cap_b = a.cap_b;
    sink.cnt_a = &a.st->cnt_a;
    sink.cnt_b = &a.st->cnt_b;
    return sink;
}

// The bins of the first level's candidates in a block's shared memory.
template <int DT>
__device__ __forceinline__ BinHist<Key<DT>::KW> make_bins(const SelArgs& a, u32* h) {
    if (!a.bins) return BinHist<Key<DT>::KW>{nullptr, 0, 0, 0};
    return BinHist<Key<DT>::KW>{h, Comp<Key<DT>::KW>::from128(a.bins->base), a.bins->shift, a.idx_bits};
}
// Adds a block's bins to the grid's (NT threads, after a barrier).
template <int NT> __device__ __forceinline__ void add_bins(const SelArgs& a, const u32* h) {
    if (!a.bins) return;
    for (u32 i = threadIdx.x; i < HB_BINS; i += NT)
        if (h[i]) atomicAdd(a.bins->h + i, h[i]);
}

// Register-path pass (the second level; a first level on misaligned input).
template <int NT, int DT, class Src, class Bins>
__device__ __forceinline__ void pass_any(const Src& src, bool dense, typename Comp<Src::KW>::t lo,
                                         typename Comp<Src::KW>::t pl, typename Comp<Src::KW>::t pr,
                                         const Sink<DT>& sink, PassSmem<NT>& ps, WarpQ<Src::KW>& q, const Bins& bins) {
    typedef typename Comp<Src::KW>::t ct;
    if (!dense) pass_tiles_sparse<NT, DT>(src, blockIdx.x, gridDim.x, lo, pl, pr, sink, q, bins);
    else if (lo != (ct)0) pass_tiles<NT, true, true, DT>(src, blockIdx.x, gridDim.x, lo, pl, pr, sink, ps, bins);
    else pass_tiles<NT, true, false, DT>(src, blockIdx.x, gridDim.x, lo, pl, pr, sink, ps, bins);
}

// First level on misaligned input.  Streams best with four blocks on an SM: the bins'
// place and width stay in shared memory, read where an element is counted, which
// leaves the 64 registers that takes.  2^28 f32 keys at k = n / 3: 808 us a call, 1039
// with three blocks and the bins in registers.
template <int KW> struct SmemBins {
    static constexpr bool COUNTS = true, KTH = true;
    u32 h[HB_BINS];
    BinHist<KW> b;
    __device__ __forceinline__ void add(typename Comp<KW>::key_t k, u32 x) const { b.add(k, x); }
};
template <int DT> __global__ void __launch_bounds__(PASS_NT, Key<DT>::KW == 32 ? 4 : 2) k_pass_first(SelArgs a) {
    constexpr int KW = Key<DT>::KW;
    typedef Comp<KW> C;
    __shared__ PassSmem<PASS_NT> ps;
    __shared__ WarpQ<KW> wq[PASS_NT / 32];
    __shared__ __align__(16) unsigned char bins_raw[sizeof(SmemBins<KW>)];
    auto& bins = *reinterpret_cast<SmemBins<KW>*>(bins_raw);
    __shared__ EpilogueSmem es;
    for (u32 i = threadIdx.x; i < HB_BINS; i += PASS_NT) bins.h[i] = 0;
    grid_dep_wait();
    const SelState s = *a.st;
    if (s.phase != PH_RUN || !s.pending || s.src != SRC_INPUT) return;
    if (threadIdx.x == 0) bins.b = make_bins<DT>(a, bins.h);
    __syncthreads();
    pass_any<PASS_NT, DT>(InputSrc<DT>::make(a.keys, s.m_src), s.dense != 0, C::from128(s.lo), C::from128(s.pl),
                          C::from128(s.pr), make_sink<DT>(a, s), ps, wq[threadIdx.x >> 5], bins);
    grid_dep_release();
    __syncthreads();
    add_bins<PASS_NT>(a, bins.h);
    pass_epilogue<KW, PASS_NT, SyncBlock, true>(a, es);
}

// The pivots of a pass that none has armed, by every block for itself: all draw
// the same sample and select the same two of its elements, so no block waits for
// another and no launch is spent on what seldom happens: a bracket that missed
// rank k, candidates that did not fit their buffer, or bins that resolved nothing.
// A window that the finish's list (and the buffer) holds is collected as it is.  Otherwise the
// margin is four standard deviations; where that bracket would not fit the
// candidate buffer (rank k near an end of a large window) it is drawn from again,
// up to N * 16 draws of which only those inside it are kept, and its margin
// narrowed until it is expected to fit.  Sets pl, pr, dst, dense, level of `s`
// (shared); false: no use (the finish takes the source as it is).
template <int KW> struct HereSmem {
    static constexpr u32 N = KW == 32 ? 2048 : 1024;
    typename Comp<KW>::t samp[N];
    HistSelSmem<KW> hs;
    u32 kept, fits;
    long long jl, jr;
};
template <int DT> __device__ __forceinline__ CandSrc<Key<DT>::KW> cand_src(const SelArgs& a, const SelState& s) {
    const u32 c = s.src == SRC_CAND1 ? 1 : 0;
    return CandSrc<Key<DT>::KW>{static_cast<const typename Key<DT>::key_t*>(a.cand_key[c]), a.cand_idx[c], s.m_src};
}
// Draws from the source of `s`: those inside [lo, hi] are counted, and the first
// `room` kept in sm.samp.
template <int DT>
__device__ __noinline__ u32 here_sample(const SelArgs& a, const SelState& s, typename Comp<Key<DT>::KW>::t lo,
                                        typename Comp<Key<DT>::KW>::t hi, u32 draws, u32 salt, u32 room,
                                        HereSmem<Key<DT>::KW>& sm) {
    if (s.src == SRC_INPUT)
        block_sample(InputSrc<DT>::make(a.keys, s.m_src), lo, hi, draws, a.parts, a.seed, s.level, salt, sm.samp, room, &sm.kept);
    else block_sample(cand_src<DT>(a, s), lo, hi, draws, a.parts, a.seed, s.level, salt, sm.samp, room, &sm.kept);
    const u32 n = sm.kept;
    __syncthreads();
    return n;
}
template <int DT>
__device__ __noinline__ bool plan_here(const SelArgs& a, SelState& s, HereSmem<Key<DT>::KW>& sm) {
    constexpr int KW = Key<DT>::KW;
    constexpr u32 N = HereSmem<KW>::N, WANT = N / 4 * 3;
    typedef Comp<KW> C;
    typedef typename C::t ct;
    const ct lo = C::from128(s.lo), hi = C::from128(s.hi);
    ct pl = lo, pr = hi;
    double below = 0.0; // elements of the window expected below pl
    if (s.m_win > FIN_LIST<KW> || s.m_win > a.cap_b) {
        u32 in = 0, under = 0, over = 0; // draws inside [pl, pr], and in the window on either side of it
        u32 draws = 0;
        for (u32 stage = 0; stage < 2; ++stage) {
            // as many draws as leave about WANT inside the bracket
            const u32 all = in + under + over;
            const double inside = (stage ? (double)(sm.jr - sm.jl + 2) / (double)all : 1.0) * (double)s.m_win / (double)s.m_src;
            const double want = (double)WANT / (inside > 0.0 ? inside : 1.0);
            const u32 most = N * (stage ? 16 : 8), d = want < (double)most ? (u32)want : most;
            __syncthreads();
            if (d <= draws) break;
            draws = d;
            in = here_sample<DT>(a, s, pl, pr, d, 0x48455245u + stage, N, sm);
            if (in > N) return false; // (the blocks would keep different draws; 13 standard deviations off)
            if (in == 0) break; // (nothing learnt)
            if (stage) {
                under = pl > lo ? here_sample<DT>(a, s, lo, (ct)(pl - 1), d, 0x48455245u + stage, 0, sm) : 0;
                over = pr < hi ? here_sample<DT>(a, s, (ct)(pr + 1), hi, d, 0x48455245u + stage, 0, sm) : 0;
            }
            if (threadIdx.x == 0) {
                const u32 n = in + under + over;
                long long l, r;
                float z = 4.0f;
                do {
                    pivot_ranks(n, s.m_win, s.k_rem, z, false, l, r);
                    l = l < -1 ? -1 : l;
                    r = r < n ? r : n;
                    z *= 0.5f;
                    sm.fits = (double)(r - l + 1) * (double)s.m_win <= 0.75 * (double)n * (double)a.cap_b;
                } while (stage && !sm.fits && z > 0.25f);
                sm.jl = l;
                sm.jr = r;
            }
            __syncthreads();
            const u32 fits = sm.fits;
            const long long jl = sm.jl - under, jr = sm.jr - under, top = (long long)in - 1;
            const u32 r1 = (u32)(jr < 0 ? 0 : jr > top ? top : jr), r0 = jl < 0 ? r1 : (u32)(jl > top ? top : jl);
            ct x0, x1;
            block_select_two<KW, PASS_NT>(sm.samp, in, pl, pr, r0, r1, sm.hs, x0, x1);
            below = sm.jl < 0 ? 0.0 : (double)(sm.jl + 1) * (double)s.m_win / (double)(in + under + over);
            if (jl >= 0) pl = x0;
            if (jr <= top) pr = x1;
            if (fits) break;
        }
    }
    if (pl == lo && pr == hi && s.m_win > a.cap_b) return false;
    // (the input also holds what lies below the window)
    if (s.src == SRC_INPUT) below += (double)s.out_base;
    const u32 dense = below * 16.0 > (double)s.m_src ? 1u : 0u;
    __syncthreads(); // `s` has been read, and the planning's memory is free again
    if (threadIdx.x == 0) {
        s.pl = (u128)pl;
        s.pr = (u128)pr;
        s.dense = dense;
        s.dst = s.src == SRC_CAND0 ? SRC_CAND1 : SRC_CAND0;
        s.level += 1;
        s.levels_grid += 1;
    }
    __syncthreads();
    return true;
}

// The second level where it is not simply the armed pass over the candidates (out
// of line: its registers would weigh on that one).
template <int DT>
__device__ __noinline__ void pass_again(const SelArgs& a, bool armed, HereSmem<Key<DT>::KW>& here,
                                        WarpQ<Key<DT>::KW>* wq, PassSmem<PASS_NT>& ps, EpilogueSmem& es) {
    typedef Comp<Key<DT>::KW> C;
    __shared__ SelState s;
    if (threadIdx.x == 0) s = *a.st;
    __syncthreads();
    if (!armed && !plan_here<DT>(a, s, here)) return;
    const typename C::t lo = C::from128(s.lo), pl = C::from128(s.pl), pr = C::from128(s.pr);
    const Sink<DT> sink = make_sink<DT>(a, s);
    WarpQ<Key<DT>::KW>& q = wq[threadIdx.x >> 5];
    if (s.src == SRC_INPUT)
        pass_any<PASS_NT, DT>(InputSrc<DT>::make(a.keys, s.m_src), s.dense != 0, lo, pl, pr, sink, ps, q, NoBinsKth{});
    else pass_any<PASS_NT, DT>(cand_src<DT>(a, s), s.dense != 0, lo, pl, pr, sink, ps, q, NoBinsKth{});
    pass_epilogue<Key<DT>::KW, PASS_NT, SyncBlock, false>(a, es, armed ? nullptr : &s);
}

// Second level: over the candidates of the first, or over the input again, when the
// first's last block armed it or more is left than the finish holds.
template <int DT> __global__ void __launch_bounds__(PASS_NT, Key<DT>::KW == 32 ? 3 : 2) k_pass(SelArgs a) {
    typedef Key<DT> K;
    constexpr int KW = K::KW;
    typedef Comp<KW> C;
    union Smem {
        WarpQ<KW> wq[PASS_NT / 32];
        HereSmem<KW> here;
        __device__ Smem() {}
    };
    __shared__ PassSmem<PASS_NT> ps;
    __shared__ __align__(16) unsigned char smem_raw[sizeof(Smem)];
    static_assert(sizeof(Smem) == sizeof(WarpQ<KW>) * (PASS_NT / 32), "planning takes no more than the pass");
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    __shared__ EpilogueSmem es;
    grid_dep_wait();
    grid_dep_release();
    const SelState s = *a.st;
    if (s.phase != PH_RUN) return;
    if (!s.pending && (s.m_src <= FIN_LIST<KW> || (a.plan_follows && s.src != SRC_INPUT))) return;
    if (!s.pending || s.src == SRC_INPUT) {
        pass_again<DT>(a, s.pending != 0, sm.here, sm.wq, ps, es);
        return;
    }
    pass_any<PASS_NT, DT>(cand_src<DT>(a, s), s.dense != 0, C::from128(s.lo), C::from128(s.pl), C::from128(s.pr),
                          make_sink<DT>(a, s), ps, sm.wq[threadIdx.x >> 5], NoBinsKth{});
    pass_epilogue<KW, PASS_NT, SyncBlock, false>(a, es);
}

// First level, 16-byte-aligned input: a producer warp streams full tiles
// into a ring of shared-memory stages with bulk (TMA) copies while 8 consumer
// warps classify and compact, so HBM reads never wait for the compute.  Every
// wait is bounded; a timeout latches TOPK_ETIMEOUT and the block winds down
// without hanging.
constexpr int TMA_CONS = 256;
constexpr int TMA_NT = TMA_CONS + 32;
constexpr u64 WAIT_LIMIT_NS = 200ull * 1000 * 1000;

// Ring geometry.  A sparse pass has 2 blocks per SM, with room for a whole
// tile's hits in every warp's buffer; a counting pass, which has more to do for
// every key, 3 blocks with smaller rings and buffers (median of 2^28 f32 keys 275
// us against 282 with the sparse pass's geometry; k = 1024 of them 199 against
// 194).  A dense pass holds two stages per block (one counted, one being written
// out), with 3 blocks (24 consumer warps) per SM, 2 for 64-bit keys.
enum : int { PM_SPARSE = 0, PM_DENSE = 1, PM_COUNT = 2 }; // what a first-level pass does with a (few; many; counted)
template <int DT, int MODE = PM_SPARSE> struct TmaCfg {
    static constexpr bool DENSE = MODE == PM_DENSE;
    static constexpr u32 W = sizeof(typename Key<DT>::raw_t);
    static constexpr u32 TILE = TMA_CONS * 16; // elements per stage
    static constexpr u32 BYTES = TILE * W;     // 8, 16 or 32 KiB
    static constexpr u32 STAGES = MODE == PM_COUNT ? (W == 2 ? 6 : 3) : (W == 2 ? 8 : W == 4 ? 4 : 3);
    static constexpr u32 WB_CAP = W == 8 || MODE == PM_COUNT ? 256 : 512; // entries of a warp's buffer
    static constexpr u32 SMEM = STAGES * BYTES;
    static constexpr int MIN_BLOCKS = MODE == PM_SPARSE ? 1 : W == 8 ? (DENSE ? 2 : 1) : 3;
};

// Raw key bits of this thread's 16 slots from a stage (slot q at vector
// q / EPV of the thread, element q % EPV).
template <int DT>
__device__ __forceinline__ void load_raw_stage(const unsigned char* stage, typename Key<DT>::raw_t (&rr)[16]) {
    uint4 v[InputSrc<DT>::NV];
    const uint4* sp = reinterpret_cast<const uint4*>(stage);
#pragma unroll
    for (int j = 0; j < InputSrc<DT>::NV; ++j) v[j] = sp[j * TMA_CONS + threadIdx.x];
    InputSrc<DT>::unpack_raw(v, rr);
}

// A warp's buffer of elements on their way out of a first-level pass, packed:
// a tile's hits take consecutive slots (one shared-memory atomic per lane that has
// any), so a flush writes whole rows of 32.  One flush in about 30 tiles waits
// for its reservation, which the other warps and the ring cover.  Entries keep
// the raw key bits; the rows of a flush turn them into images.  (Per-lane queues,
// whose rows are as long as the fullest lane's, and which classified every entry
// again, took 0.33 ms for the counting pass on 2^28 f32 keys at k = n / 2, packed
// 0.235 ms, and 0.18 ms with the masks built off the integer pipe.)
template <int KW, u32 N> struct WarpBuf {
    static constexpr u32 CAP = N;
    typename Comp<KW>::key_t k[CAP]; // raw key bits
    u32 i[CAP];
    u32 n;
};

// Writes a warp's `cnt` entries (all at most pr): those below pl to the output,
// unless the buffer holds b elements only (ONLY_B), the rest to the
// candidates and their bins.
template <int DT, bool ONLY_B, class WB>
__device__ __forceinline__ void wb_flush(WB& w, u32 cnt, typename Comp<Key<DT>::KW>::t pl,
                                         const Sink<DT>& sink, const BinHist<Key<DT>::KW>& bins) {
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef Comp<Key<DT>::KW> C;
    const u32 lane = lane_id(), below = lanemask_lt();
    __syncwarp();
    u32 ca = 0;
    if constexpr (!ONLY_B) {
        for (u32 j = lane; j < cnt; j += 32) ca += (u32)(C::make(K::fwd((raw_t)w.k[j]), w.i[j]) < pl);
        ca = __reduce_add_sync(0xffffffffu, ca);
    }
    u64 ra = 0, rb = 0;
    if (lane == 0) {
        if (!ONLY_B && ca) ra = atomicAdd((unsigned long long*)sink.cnt_a, (unsigned long long)ca);
        if (cnt > ca) rb = atomicAdd((unsigned long long*)sink.cnt_b, (unsigned long long)(cnt - ca));
        w.n = 0;
    }
    if constexpr (!ONLY_B) ra = __shfl_sync(0xffffffffu, (unsigned long long)ra, 0);
    rb = __shfl_sync(0xffffffffu, (unsigned long long)rb, 0);
    for (u32 j0 = 0; j0 < cnt; j0 += 32) {
        const u32 j = j0 + lane;
        const bool in = j < cnt;
        const typename C::key_t kv = in ? K::fwd((raw_t)w.k[j]) : (typename C::key_t)0;
        const u32 iv = in ? w.i[j] : 0u;
        if constexpr (ONLY_B) {
            if (in) {
                sink.put_b(rb + j, kv, iv);
                bins.add(kv, iv);
            }
        } else {
            const bool isa = in && C::make(kv, iv) < pl;
            const u32 bala = __ballot_sync(0xffffffffu, isa), balb = __ballot_sync(0xffffffffu, in && !isa);
            if (isa) sink.put_a(ra + __popc(bala & below), kv, iv); // (writes nothing where cap_a = 0)
            else if (in) {
                sink.put_b(rb + __popc(balb & below), kv, iv);
                bins.add(kv, iv);
            }
            ra += __popc(bala);
            rb += __popc(balb);
        }
    }
    __syncwarp();
}

// Appends the slots of `hit`: slot q's key bits are raw_at(off) and its position
// is first + off, off = off_of(q) (q and off differ by lane).  `cnt` is the number
// of entries, the same in every lane.  All 32 lanes call.
template <int DT, bool ONLY_B, class WB, class OffOf, class RawAt>
__device__ __forceinline__ void wb_append(WB& w, u32& cnt, u32 hit, u32 first, OffOf off_of,
                                          RawAt raw_at, typename Comp<Key<DT>::KW>::t pl, const Sink<DT>& sink,
                                          const BinHist<Key<DT>::KW>& bins) {
    constexpr u32 CAP = WB::CAP;
    const u32 total = __reduce_add_sync(0xffffffffu, (u32)__popc(hit));
    if (total == 0) return;
    auto add = [&](u32 m, u32 n) {
        if (cnt + n > CAP) {
            wb_flush<DT, ONLY_B>(w, cnt, pl, sink, bins);
            cnt = 0;
        }
        if (m) {
            u32 slot = atomicAdd(&w.n, (u32)__popc(m));
            do {
                const u32 off = off_of((u32)(__ffs(m) - 1));
                m &= m - 1;
                w.k[slot] = raw_at(off);
                w.i[slot] = first + off;
                ++slot;
            } while (m);
        }
        cnt += n;
    };
    if (total <= CAP) {
        add(hit, total);
    } else { // nearly the whole tile: as many slots at a time as always fit
        constexpr u32 S = CAP / 32;
#pragma unroll 1
        for (u32 h = 0; h < 16; h += S) {
            const u32 m = (hit >> h) & ((1u << S) - 1u);
            add(m << h, __reduce_add_sync(0xffffffffu, (u32)__popc(m)));
        }
    }
}

// First level with few elements to write (sparse: a and b both; counting: b, a
// being counted in registers and never written, for a call that wants the
// rank-k pair alone).  A tile that holds neither pivot's position is tested
// with one comparison of raw key bits per element and pivot (tile bounds), the
// rare other tile on the pair; the few hits go through the warp's buffer.  No
// block barrier.  On 2^28 f32 keys at k = n / 2 the counting pass takes 0.18
// ms, against 0.47 ms for the pass that writes a.
template <int DT, bool COUNT>
__device__ void tma_consume_few(const SelArgs& a, const SelState& s, const unsigned char* stages, uint64_t* full,
                                uint64_t* empty, u64 my_n, u32* dead,
                                WarpBuf<Key<DT>::KW, TmaCfg<DT, COUNT ? PM_COUNT : PM_SPARSE>::WB_CAP>& wb,
                                const BinHist<Key<DT>::KW>& bins) {
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef typename K::key_t key_t;
    typedef Comp<K::KW> C;
    typedef typename C::t ct;
    typedef TmaCfg<DT, COUNT ? PM_COUNT : PM_SPARSE> Cfg;
    constexpr u32 EPV = InputSrc<DT>::EPV;
    const Sink<DT> sink = make_sink<DT>(a, s);
    const ct pl = C::from128(s.pl), pr = C::from128(s.pr);
    const u32 lane = lane_id();
    const InputSrc<DT> isrc = InputSrc<DT>::make(a.keys, s.m_src); // head = 0: input is 16-byte aligned
    if (lane == 0) wb.n = 0;
    __syncwarp();
    const TileBounds<DT> tbd = TileBounds<DT>::make(pl, pr);
    u32 na = 0; // (a lane sees fewer than 2^32 keys)
    const u32 one = hidden_one();
    u32 cnt = 0, stg = 0, parity = 0;
    for (u64 i = 0; i < my_n; ++i) {
        bool ok = !*(volatile u32*)dead;
        if (ok && !mbar_wait_bounded(&full[stg], parity, WAIT_LIMIT_NS)) {
            ok = false;
            *(volatile u32*)dead = 1;
            if (lane == 0) latch(a.err, ST_ETIMEOUT);
        }
        ok = __all_sync(0xffffffffu, ok);
        // positions in 32 bits (inputs hold fewer than 2^32 keys): slot q of
        // this thread is ib + (q / EPV) * TMA_CONS * EPV + q % EPV
        const u32 tb = (u32)((blockIdx.x + i * gridDim.x) * (u64)Cfg::TILE);
        const u32 ib = tb + threadIdx.x * EPV;
        auto pos = [&](int q) -> u32 { return ib + (u32)(q / (int)EPV) * (TMA_CONS * EPV) + (u32)(q % (int)EPV); };
        u32 hit = 0;
        if (ok) {
            raw_t rr[16];
            load_raw_stage<DT>(stages + (size_t)stg * Cfg::BYTES, rr);
            RawBound<DT> ba, bb;
            bool any_a, any_l;
            const bool away = tbd.get(tb, tb + Cfg::TILE - 1, ba, bb, any_a, any_l);
            if (COUNT ? away && any_a && any_l : away) {
                if constexpr (COUNT) tile_count_dispatch<DT>(rr, ba, bb, one, na, hit);
                else hit = tile_le_dispatch<DT>(rr, bb, any_l);
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const ct c = C::make(K::fwd(rr[q]), pos(q));
                    const bool in_a = COUNT && c < pl;
                    na += (u32)in_a;
                    hit |= (u32)(!in_a && c <= pr) << q;
                }
            }
        }
        // the hits' keys come from the stage, which is released after them
        const unsigned char* mine = stages + (size_t)stg * Cfg::BYTES + threadIdx.x * 16u;
        wb_append<DT, COUNT>(wb, cnt, hit, ib, [](u32 q) { return (q / EPV) * (TMA_CONS * EPV) + q % EPV; },
                             [&](u32 off) { return *reinterpret_cast<const raw_t*>(mine + off * sizeof(raw_t)); }, pl,
                             sink, bins);
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&empty[stg]); // the stage may be refilled
        if (++stg == Cfg::STAGES) {
            stg = 0;
            parity ^= 1u;
        }
    }
    // the ragged last tile, read directly by the block that owns it
    const u64 nfull = s.m_src / Cfg::TILE;
    if (s.m_src % Cfg::TILE != 0 && nfull % gridDim.x == blockIdx.x) {
        key_t kk[16];
        u32 ii[16];
        const u64 tb = nfull * (u64)Cfg::TILE;
        const u32 valid = isrc.template load16<TMA_CONS>(tb, kk, ii);
        auto pos = [&](int q) -> u32 { return isrc.template idx_of<TMA_CONS>(tb, q); };
        u32 ma = 0, le = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const ct c = C::make(kk[q], pos(q));
            if (COUNT) ma |= (u32)(c < pl) << q;
            le |= (u32)(c <= pr) << q;
        }
        ma &= valid;
        na += (u32)__popc(ma);
        wb_append<DT, COUNT>(wb, cnt, le & valid & ~ma, (u32)tb + threadIdx.x * EPV,
                             [](u32 q) { return (q / EPV) * (TMA_CONS * EPV) + q % EPV; },
                             [&](u32 off) { return static_cast<const raw_t*>(a.keys)[tb + threadIdx.x * EPV + off]; }, pl,
                             sink, bins);
    }
    if (cnt) wb_flush<DT, COUNT>(wb, cnt, pl, sink, bins);
    if constexpr (COUNT) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) na += __shfl_xor_sync(0xffffffffu, na, o); // (of fewer than 2^32 in all)
        if (lane == 0 && na) atomicAdd((unsigned long long*)sink.cnt_a, (unsigned long long)na);
    }
}

// Dense first level (many elements in a; the window starts at the smallest
// pair).  Output room is reserved per tile with one atomic per class, but
// the reservation of tile i is issued right after the block's one barrier
// of iteration i and published before the barrier of iteration i+1, so its
// latency overlaps the work of a whole tile; tile i-1 is written after that
// barrier, re-read from its shared-memory stage, which is held until then.
// Two threads take turns issuing the atomics.
//
// A tile that contains neither pivot's position is classified with two
// comparisons of raw key bits per element (tile_bounds): ties with a pivot's
// key are decided for the whole tile by which side of the pivot's position
// it lies on.  a-elements leave by per-slot warp ballots: one store
// instruction per slot writes the warp's selected keys (and one their
// positions) to consecutive addresses, the run pointers advancing by the
// slot's count.  b-elements are few; each lane writes its own at an offset
// from one warp scan.
struct DenseSmem {
    u32 wa[2][TMA_CONS / 32], wb[2][TMA_CONS / 32]; // per-warp counts, by tile parity
    u64 oa[2][TMA_CONS / 32], ob[2][TMA_CONS / 32]; // per-warp offsets inside the tile
    u64 ba[2], bb[2];                               // tile bases in the output / candidates
};

template <int DT>
__device__ void tma_consume_dense(const SelArgs& a, const SelState& s, const unsigned char* stages, uint64_t* full,
                                  uint64_t* empty, u64 my_n, u32* dead, DenseSmem& ds, PassSmem<TMA_CONS>& ps,
                                  const BinHist<Key<DT>::KW>& bins) {
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef typename K::key_t key_t;
    typedef Comp<K::KW> C;
    typedef typename C::t ct;
    typedef TmaCfg<DT, PM_DENSE> Cfg;
    typedef SyncNamed<1, TMA_CONS> Sync;
    constexpr int EPV = InputSrc<DT>::EPV;
    constexpr u32 STRIDE = TMA_CONS * EPV; // index distance between a thread's vectors
    const Sink<DT> sink = make_sink<DT>(a, s);
    const ct pl = C::from128(s.pl), pr = C::from128(s.pr);
    const u32 warp = threadIdx.x >> 5, lane = lane_id(), below = lanemask_lt();
    const InputSrc<DT> isrc = InputSrc<DT>::make(a.keys, s.m_src); // head = 0
    const key_t plk = (key_t)C::key(pl), prk = (key_t)C::key(pr);
    const u32 plx = C::idx(pl), prx = C::idx(pr);
    u32 ma_prev = 0, mb_prev = 0, stg_prev = 0, ib_prev = 0;
    bool ok_prev = false;
    u64 my_ra = 0, my_rb = 0;   // pending reservation of the issuing thread
    u32 ring = 0, ring_par = 0; // stage and phase parity of tile i
    for (u64 i = 0; i <= my_n; ++i) {
        const bool cur = i < my_n, have_prev = i > 0;
        const u32 par = (u32)(i & 1), ppar = par ^ 1u;
        u32 ma = 0, mb = 0, stg = 0, ib = 0;
        bool ok = false;
        if (cur) {
            stg = ring;
            const u32 fpar = ring_par;
            if (++ring == Cfg::STAGES) {
                ring = 0;
                ring_par ^= 1u;
            }
            ok = !*(volatile u32*)dead;
            if (ok && !mbar_wait_bounded(&full[stg], fpar, WAIT_LIMIT_NS)) {
                ok = false;
                *(volatile u32*)dead = 1;
                if (lane == 0) latch(a.err, ST_ETIMEOUT);
            }
            ok = __all_sync(0xffffffffu, ok);
            // position of slot q = ib + (q / EPV) * STRIDE + q % EPV (32-bit: positions < 2^32)
            const u32 tb = (u32)((blockIdx.x + i * gridDim.x) * (u64)Cfg::TILE);
            ib = tb + threadIdx.x * EPV;
            if (ok) {
                const u32 te = tb + Cfg::TILE - 1;
                u32 le = 0;
                if (!((plx >= tb && plx <= te) || (prx >= tb && prx <= te))) {
                    // the tile holds neither pivot's position: ties with a
                    // pivot's key are decided by the side it lies on
                    raw_t rr[16];
                    load_raw_stage<DT>(stages + (size_t)stg * Cfg::BYTES, rr);
                    const bool ta = te < plx, tl = te <= prx;
                    const RawBound<DT> ba = RawBound<DT>::le((key_t)(plk - (ta ? 0 : 1)));
                    const RawBound<DT> bb = RawBound<DT>::le((key_t)(prk - (tl ? 0 : 1)));
                    tile_masks_dispatch<DT>(rr, ba, bb, ta || plk != 0, tl || prk != 0, ma, le);
                } else {
                    key_t kk[16];
                    InputSrc<DT>::template load16_smem<TMA_CONS>(
                        reinterpret_cast<const uint4*>(stages + (size_t)stg * Cfg::BYTES), kk);
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const ct c = C::make(kk[q], ib + (u32)((q / EPV) * STRIDE + q % EPV));
                        ma |= (u32)(c < pl) << q;
                        le |= (u32)(c <= pr) << q;
                    }
                }
                mb = le & ~ma;
            }
            const u32 wa = __reduce_add_sync(0xffffffffu, (u32)__popc(ma));
            const u32 wb = __reduce_add_sync(0xffffffffu, (u32)__popc(mb));
            if (lane == 0) {
                ds.wa[par][warp] = wa;
                ds.wb[par][warp] = wb;
            }
        }
        // the issuer of tile i-1 publishes its reservation before the barrier
        const u32 issuer_cur = par ? 32u : 0u, issuer_prev = ppar ? 32u : 0u;
        if (have_prev && threadIdx.x == issuer_prev) {
            ds.ba[ppar] = my_ra;
            ds.bb[ppar] = my_rb;
        }
        Sync::sync(); // counts of tile i, base of tile i-1 in; writes of tile i-2 done
        if (cur && threadIdx.x == issuer_cur) {
            u64 ta = 0, tb2 = 0;
            for (int w = 0; w < TMA_CONS / 32; ++w) {
                ds.oa[par][w] = ta;
                ds.ob[par][w] = tb2;
                ta += ds.wa[par][w];
                tb2 += ds.wb[par][w];
            }
            my_ra = 0;
            my_rb = 0;
            if (ta) my_ra = atomicAdd((unsigned long long*)sink.cnt_a, (unsigned long long)ta);
            if (tb2) my_rb = atomicAdd((unsigned long long*)sink.cnt_b, (unsigned long long)tb2);
        }
        if (have_prev && ok_prev) {
            // this thread's element of slot q sits at a constant offset from `mine`
            const unsigned char* mine = stages + (size_t)stg_prev * Cfg::BYTES + threadIdx.x * 16u;
            auto elem = [&](u32 q) -> raw_t {
                return *reinterpret_cast<const raw_t*>(mine + (q / EPV) * (TMA_CONS * 16u) + (q % EPV) * sizeof(raw_t));
            };
            if (__any_sync(0xffffffffu, ma_prev)) {
                const u64 xa = ds.ba[ppar] + ds.oa[ppar][warp];
                if (xa + ds.wa[ppar][warp] <= sink.cap_a) { // the usual case: no per-element bound
                    raw_t* okp = sink.out_keys + sink.out_base + xa;
                    u32* oip = sink.out_idx + sink.out_base + xa;
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const bool bit = (ma_prev >> q) & 1u;
                        const u32 bal = __ballot_sync(0xffffffffu, bit);
                        // operands computed on every lane so that the stores
                        // are predicated rather than branched around; the run
                        // pointers advance by the slot's count
                        const u32 r = (u32)__popc(bal & below);
                        const raw_t key = elem(q);
                        const u32 idx = ib_prev + (u32)((q / EPV) * STRIDE + q % EPV);
                        if (bit) {
                            okp[r] = key;
                            oip[r] = idx;
                        }
                        const u32 c = (u32)__popc(bal);
                        okp += c;
                        oip += c;
                    }
                } else {
                    u64 ra = xa;
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const bool bit = (ma_prev >> q) & 1u;
                        const u32 bal = __ballot_sync(0xffffffffu, bit);
                        if (bit)
                            sink.put_a_raw(ra + __popc(bal & below), elem(q),
                                           ib_prev + (u32)((q / EPV) * STRIDE + q % EPV));
                        ra += (u32)__popc(bal);
                    }
                }
            }
            if (__any_sync(0xffffffffu, mb_prev)) { // b is sparse: each lane writes its own
                const u32 cnt = (u32)__popc(mb_prev);
                u32 incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= (u32)o) incl += y;
                }
                u64 xb = ds.bb[ppar] + ds.ob[ppar][warp] + (incl - cnt);
                u32 m = mb_prev;
                while (m) {
                    const u32 q = (u32)(__ffs(m) - 1);
                    m &= m - 1;
                    const key_t kb = K::fwd(elem(q));
                    const u32 ibq = ib_prev + (q / EPV) * STRIDE + q % EPV;
                    sink.put_b(xb++, kb, ibq);
                    bins.add(kb, ibq);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[stg_prev]); // stage may be refilled
        }
        ma_prev = ma;
        mb_prev = mb;
        stg_prev = stg;
        ib_prev = ib;
        ok_prev = ok;
    }
    // the ragged last tile, read directly by the block that owns it
    const u64 nfull = s.m_src / Cfg::TILE;
    if (s.m_src % Cfg::TILE != 0 && nfull % gridDim.x == blockIdx.x) {
        key_t kk[16];
        u32 ii[16];
        const u64 tb = nfull * (u64)Cfg::TILE;
        const u32 valid = isrc.template load16<TMA_CONS>(tb, kk, ii);
        auto pos = [&](int q) -> u32 { return isrc.template idx_of<TMA_CONS>(tb, q); };
        classify_emit<TMA_CONS, true, false, Sync>(kk, pos, valid, (ct)0, pl, pr, sink, ps, bins);
    }
}

template <int DT, int MODE>
__global__ void __launch_bounds__(TMA_NT, (TmaCfg<DT, MODE>::MIN_BLOCKS)) k_pass_tma(SelArgs a) {
    typedef TmaCfg<DT, MODE> Cfg;
    constexpr bool DENSE = MODE == PM_DENSE;
    typedef typename Key<DT>::raw_t raw_t;
    constexpr int KW = Key<DT>::KW;
    extern __shared__ __align__(128) unsigned char stages[];
    __shared__ __align__(8) uint64_t full[Cfg::STAGES];
    __shared__ __align__(8) uint64_t empty[Cfg::STAGES];
    __shared__ PassSmem<TMA_CONS> ps;
    __shared__ __align__(16) unsigned char wb_raw[DENSE ? 16 : sizeof(WarpBuf<KW, Cfg::WB_CAP>) * (TMA_CONS / 32)];
    __shared__ DenseSmem ds;
    __shared__ u32 hist[HB_BINS];
    __shared__ EpilogueSmem es;
    __shared__ u32 dead;
    for (u32 i = threadIdx.x; i < HB_BINS; i += TMA_NT) hist[i] = 0;
    grid_dep_wait();
    const SelState s = *a.st;
    if (s.phase != PH_RUN || !s.pending || s.src != SRC_INPUT || (s.dense != 0) != (MODE != PM_SPARSE)) {
        grid_dep_release(); // nothing to do (an earlier failure, or the other mode): the next launch proceeds
        return;
    }
    // the tile thresholds of the dense variant assume a window starting at the
    // smallest pair, which holds on first levels (the only ones this kernel runs)
    if (MODE != PM_SPARSE && Comp<KW>::from128(s.lo) != (typename Comp<KW>::t)0) {
        if (threadIdx.x == 0) latch(a.err, ST_EINTERNAL);
        return;
    }
    if (threadIdx.x == 0) {
        for (u32 i = 0; i < Cfg::STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], TMA_CONS / 32);
        }
        dead = 0;
        mbar_fence_init();
    }
    __syncthreads();
    const u64 nfull = s.m_src / Cfg::TILE;
    const u64 my_n = nfull > blockIdx.x ? (nfull - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    if (threadIdx.x >= TMA_CONS) { // producer warp: one lane issues the copies
        if (threadIdx.x == TMA_CONS) {
            const raw_t* keys = static_cast<const raw_t*>(a.keys);
            u32 stg = 0, epar = 1; // the first pass over the ring waits for nothing
            for (u64 i = 0; i < my_n; ++i) {
                if (i >= Cfg::STAGES) {
                    const u32 parity = epar;
                    if (*(volatile u32*)&dead || !mbar_wait_bounded(&empty[stg], parity, WAIT_LIMIT_NS)) {
                        *(volatile u32*)&dead = 1;
                        latch(a.err, ST_ETIMEOUT);
                        break;
                    }
                }
                const u64 t = blockIdx.x + i * gridDim.x;
                mbar_arrive_expect_tx(&full[stg], Cfg::BYTES);
                bulk_g2s(stages + (size_t)stg * Cfg::BYTES, keys + t * Cfg::TILE, Cfg::BYTES, &full[stg]);
                if (++stg == Cfg::STAGES) {
                    stg = 0;
                    epar ^= 1u;
                }
            }
        }
        return;
    }
    const BinHist<KW> bins = make_bins<DT>(a, hist);
    auto* wb = reinterpret_cast<WarpBuf<KW, Cfg::WB_CAP>*>(wb_raw) + (DENSE ? 0 : threadIdx.x >> 5);
    if constexpr (!DENSE) tma_consume_few<DT, MODE == PM_COUNT>(a, s, stages, full, empty, my_n, &dead, *wb, bins);
    else tma_consume_dense<DT>(a, s, stages, full, empty, my_n, &dead, ds, ps, bins);
    grid_dep_release(); // this block's stream has ended: the next kernel may start taking its place
    SyncNamed<1, TMA_CONS>::sync();
    add_bins<TMA_CONS>(a, hist);
    pass_epilogue<KW, TMA_CONS, SyncNamed<1, TMA_CONS>, true>(a, es);
}

// A short input whole, in one block: its keys into shared memory, rank k by a
// histogram over the key domain, the elements up to it written.  The cluster of
// k_finish is slower on so few (its barriers and its range step): 100 keys 5.4 us
// here, 6.3 by its first block alone; 8192 normal f32 keys 10.5 here, 12.6 by all
// eight, which pay from about 12000 keys on.
constexpr u32 SMALL_MAX = 8192;
template <int DT> using SmallSmem = BlockSmem<Key<DT>::KW, BLK_NT, SMALL_MAX>;
template <int DT> __global__ void __launch_bounds__(BLK_NT) k_small(SelArgs a) {
    grid_dep_wait();
    grid_dep_release();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (threadIdx.x == 0) init_state<DT>(a.st, a);
    __syncthreads();
    block_finish<DT, true>(a, *reinterpret_cast<SmallSmem<DT>*>(smem_raw));
}

// k = 1: the minimum pair (base case of Algorithm "select");
// k = n: every pair, plus the maximum as the rank-n pair.
template <int KW> __device__ __forceinline__ typename Comp<KW>::t shfl_xor_ct(typename Comp<KW>::t v, int o);
template <> __device__ __forceinline__ u64 shfl_xor_ct<32>(u64 v, int o) {
    return __shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
}
template <> __device__ __forceinline__ u128 shfl_xor_ct<64>(u128 v, int o) {
    const u64 lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)(u64)v, o);
    const u64 hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(u64)(v >> 64), o);
    return ((u128)hi << 64) | lo;
}

template <int KW>
__device__ typename Comp<KW>::t block_extreme(typename Comp<KW>::t v, bool want_max, typename Comp<KW>::t* red) {
    typedef typename Comp<KW>::t ct;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const ct w = shfl_xor_ct<KW>(v, o);
        v = want_max ? (w > v ? w : v) : (w < v ? w : v);
    }
    const u32 warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane_id() == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        ct b = red[0];
        for (u32 w = 1; w < nw; ++w) b = want_max ? (red[w] > b ? red[w] : b) : (red[w] < b ? red[w] : b);
        red[0] = b;
    }
    __syncthreads();
    const ct out = red[0];
    __syncthreads();
    return out;
}

// MAX: k = n; COPY: it copies every pair out (not for the rank-k pair alone).
template <int DT, bool MAX, bool COPY>
__global__ void __launch_bounds__(EXT_NT) k_extreme(SelArgs a, u32* counter, void* partials_v) {
    // (64-bit keys that are copied: the switch at run time, known to be set, keeps the
    // compiler from tying the loads to the stores; 2^17 u64 keys 6.4 us, 7.5 without)
    const bool want_max = COPY && Key<DT>::KW == 64 ? a.k == a.n : MAX, copy = COPY && want_max;
    grid_dep_wait();
    grid_dep_release();
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    constexpr int KW = K::KW;
    typedef Comp<KW> C;
    typedef typename C::t ct;
    __shared__ ct red[EXT_NT / 32];
    __shared__ u32 is_last;
    ct* partials = static_cast<ct*>(partials_v);
    const InputSrc<DT> src = InputSrc<DT>::make(a.keys, a.n);
    raw_t* ok_out = static_cast<raw_t*>(a.out_keys);
    ct best = want_max ? (ct)0 : C::max_value();
    constexpr u64 TILE = (u64)EXT_NT * 16;
    const u64 ntiles = (src.extent() + TILE - 1) / TILE; // (an input that starts inside 16 bytes reaches further)
    for (u64 t = blockIdx.x; t < ntiles; t += gridDim.x) {
        typename K::key_t kk[16];
        u32 ii[16];
        const u32 valid = src.template load16<EXT_NT>(t * TILE, kk, ii);
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            if (!((valid >> s) & 1u)) continue;
            const ct c = C::make(kk[s], ii[s]);
            best = want_max ? (c > best ? c : best) : (c < best ? c : best);
            if (copy) {
                ok_out[ii[s]] = K::inv(kk[s]);
                a.out_idx[ii[s]] = ii[s];
            }
        }
    }
    best = block_extreme<KW>(best, want_max, red);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = best;
        __threadfence();
        const u32 prev = atomicAdd(counter, 1u);
        is_last = prev == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    ct v = want_max ? (ct)0 : C::max_value();
    for (u32 i = threadIdx.x; i < gridDim.x; i += blockDim.x) {
        const volatile ct* p = partials;
        const ct w = p[i];
        v = want_max ? (w > v ? w : v) : (w < v ? w : v);
    }
    v = block_extreme<KW>(v, want_max, red);
    if (threadIdx.x == 0) {
        static_cast<raw_t*>(a.kth_key)[0] = K::inv((typename K::key_t)C::key(v));
        a.kth_idx[0] = C::idx(v);
        if (!want_max && !a.kth_only) {
            ok_out[0] = K::inv((typename K::key_t)C::key(v));
            a.out_idx[0] = C::idx(v);
        }
        SelState* g = a.st;
        init_state<DT>(g, a);
        g->phase = PH_DONE;
        g->out_base = a.k;
        atomicExch(counter, 0u);
    }
}

// ----------------------------------------------------------- host side

struct Tuning {
    u32 sample, parts, T;
    float z;
    u32 flags;
    u64 seed;
};

template <int KW> static Tuning make_tuning(const topk_params* prm, int sms) {
    constexpr u32 ELEMS = Lim<KW>::ELEMS;
    topk_params p{};
    if (prm) p = *prm;
    Tuning tu;
    tu.sample = p.sample_size ? std::min<u32>(std::max<u32>(p.sample_size, 64), ELEMS) : ELEMS;
    tu.parts = p.partitions ? p.partitions : (u32)sms;
    tu.T = p.finish_threshold ? std::min<u32>(std::max<u32>(p.finish_threshold, 64), ELEMS) : ELEMS;
    tu.z = p.delta_factor > 0.f ? p.delta_factor : 4.0f;
    tu.flags = p.flags;
    tu.seed = p.seed ? p.seed : 0x243F6A8885A308D3ull;
    return tu;
}

static SelArgs make_args(const void* keys, u64 n, u64 k, void* out_keys, u32* out_idx, void* kth_key,
                         u32* kth_idx, const Tuning& tu) {
    SelArgs a{};
    a.keys = keys;
    a.n = n;
    a.k = k;
    a.out_keys = out_keys;
    a.out_idx = out_idx;
    a.kth_key = kth_key;
    a.kth_idx = kth_idx;
    a.seed = tu.seed;
    a.parts = tu.parts;
    a.sample = tu.sample;
    a.z = tu.z;
    a.flags = tu.flags;
    a.aligned = (reinterpret_cast<uintptr_t>(keys) & 15u) == 0;
    a.idx_bits = 1; // enough for n - 1
    while (a.idx_bits < 32 && (n - 1) >> a.idx_bits) ++a.idx_bits;
    a.first_dense = -1; // decided on the device unless the host fixes it
    a.kth_only = out_keys == nullptr;
    return a;
}

// Host copy of the device pivot-rank rule, for sizing buffers.
static double est_bracket(u64 m, u64 k_rem, u32 s, float z) {
    const double kept = (double)std::min<u64>(s, m);
    const double mu_le = kept * (double)k_rem / (double)m;
    const double mu_lt = kept * (double)(k_rem - 1) / (double)m;
    const double v = std::max(0.0, mu_le * (1.0 - mu_le / kept));
    const double d = z * std::sqrt(v) + z * z / 3.0 + 1.0;
    const double jl = std::max(-1.0, std::floor(mu_le - d) - 1.0);
    const double jr = std::min(kept, std::ceil(mu_lt + d));
    return std::min((double)m, (jr - jl + 1.0) * (double)m / kept);
}

// Kernel attributes, set once per device.
template <int DT> static topk_status set_smem_attrs() {
    static std::atomic<uint64_t> done_mask{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return TOPK_ECUDA;
    const uint64_t bit = 1ull << (dev & 63);
    if (done_mask.load() & bit) return TOPK_OK;
    if (cudaFuncSetAttribute(k_pass_tma<DT, PM_SPARSE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)TmaCfg<DT, PM_SPARSE>::SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_pass_tma<DT, PM_DENSE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)TmaCfg<DT, PM_DENSE>::SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_pass_tma<DT, PM_COUNT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)TmaCfg<DT, PM_COUNT>::SMEM) != cudaSuccess)
        return TOPK_ECUDA;
    if (cudaFuncSetAttribute(k_plan<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(PlanSmem<Key<DT>::KW>)) != cudaSuccess ||
        cudaFuncSetAttribute(k_finish<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(FinSmem<Key<DT>::KW>)) != cudaSuccess ||
        cudaFuncSetAttribute(k_small<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem<DT>)) !=
            cudaSuccess)
        return TOPK_ECUDA;
    done_mask.fetch_or(bit);
    return TOPK_OK;
}

// Resident blocks per SM of each pass variant: the grid is one full wave.
template <int DT, int MODE> static int tma_grid(int sms) {
    static int occ = 0;
    if (occ == 0) {
        int o = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_pass_tma<DT, MODE>, TMA_NT,
                                                          TmaCfg<DT, MODE>::SMEM) != cudaSuccess)
            o = 1;
        occ = std::max(1, o);
    }
    return sms * occ;
}

template <int DT> static int pass_grid(int sms, bool first) {
    static int occ_first = 0, occ_rest = 0;
    if (occ_first == 0) {
        int o1 = 0, o2 = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o1, k_pass_first<DT>, PASS_NT, 0) != cudaSuccess) o1 = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o2, k_pass<DT>, PASS_NT, 0) != cudaSuccess) o2 = 1;
        occ_rest = std::max(1, o2);
        occ_first = std::max(1, o1);
    }
    return sms * (first ? occ_first : occ_rest);
}

// Pass mode of the first level: dense when more than 1/16 of the sample is
// expected below the lower pivot.  The first level's sample is `s` draws, all
// inside its window, so its pivot ranks are known before the launch; the
// mode only steers the pass (both modes give the same result).
static bool first_level_dense(u64 n, u64 k, u32 s, float z, bool raw) {
    const double mu = (double)s * (double)k / (double)n;
    const double d = raw ? z : z * std::sqrt(std::max(0.0, mu * (1.0 - mu / s))) + z * z / 3.0 + 1.0;
    const double jl = std::floor(mu - d) - 1.0;
    return jl >= 0.0 && jl + 1.0 > (double)s / 16.0;
}

// Candidate capacity for a first level over n keys: twice the expected
// bracket, at least the finisher's range.
static u64 candidate_capacity(u64 n, u64 k, const Tuning& tu) {
    u64 cap = (u64)(2.0 * est_bracket(n, k, tu.sample, tu.z)) + 4ull * tu.T;
    if (tu.flags & TOPK_FLAG_TINY_CAND) cap = tu.T;
    cap = std::max<u64>(cap, tu.T);
    cap = std::min<u64>(cap, std::max<u64>(n, tu.T));
    return (cap + 4095) & ~(u64)4095;
}

// Enqueues one selection whose state, error word and buffers `a` already
// points to.  k = 1 and k = n need `counter` (zero) and `partials`
// (EXT grid composites).  `ctx` (may be null) receives the measurement hooks.
template <int DT>
static topk_status enqueue_select(topk_ctx* ctx, SelArgs a, const Tuning& tu, int sms, u32* counter,
                                  void* partials, cudaStream_t st) {
    constexpr int KW = Key<DT>::KW;
    const u64 n = a.n, k = a.k;
    if (k == 1 || k == n) {
        if (ctx) profile_pass_begin(ctx, st);
        const auto kern = !(k == n && n > 1) ? k_extreme<DT, false, false>
                          : a.kth_only       ? k_extreme<DT, true, false>
                                             : k_extreme<DT, true, true>;
        const cudaError_t e = launch_dep(kern, sms * EXT_BLOCKS_PER_SM, EXT_NT, 0, st, 1, a, counter, partials);
        if (e != cudaSuccess) return cuda_status(e);
        if (ctx) {
            profile_pass_end(ctx, st);
            count_launch(ctx);
        }
        return cuda_status(cudaGetLastError());
    }
    topk_status rs = set_smem_attrs<DT>();
    if (rs != TOPK_OK) return rs;
    // the first level's pass mode, fixed here so that one variant is launched
    const bool bulk = a.aligned && !(tu.flags & TOPK_FLAG_NO_BULK_COPY);
    a.first_dense =
        bulk ? (first_level_dense(n, k, tu.sample, tu.z, (tu.flags & TOPK_FLAG_RAW_DELTA) != 0) ? 1 : 0) : -1;
    auto first_pass = [&]() -> cudaError_t {
        if (!bulk) return launch_dep(k_pass_first<DT>, pass_grid<DT>(sms, true), PASS_NT, 0, st, 1, a);
        if (a.first_dense && a.kth_only)
            return launch_dep(k_pass_tma<DT, PM_COUNT>, tma_grid<DT, PM_COUNT>(sms), TMA_NT,
                              TmaCfg<DT, PM_COUNT>::SMEM, st, 1, a);
        if (a.first_dense)
            return launch_dep(k_pass_tma<DT, PM_DENSE>, tma_grid<DT, PM_DENSE>(sms), TMA_NT,
                              TmaCfg<DT, PM_DENSE>::SMEM, st, 1, a);
        return launch_dep(k_pass_tma<DT, PM_SPARSE>, tma_grid<DT, PM_SPARSE>(sms), TMA_NT,
                          TmaCfg<DT, PM_SPARSE>::SMEM, st, 1, a);
    };
    const bool one = n <= tu.T;
    // Candidates on a few distant values (ties of integer-valued floats, say) fall
    // into a few bins, and what the second pass then leaves would be streamed by
    // the finish's eight blocks, at about 40 us for 4e6 of them and every step: from
    // 2^20 expected candidates on, one more level by sampling stands ready
    // (1.3 us for each of its two kernels when it is not needed; 2^28 f32 Zipf keys at
    // k = n / 2 take 578 us with it and 733 without).
    const bool resample = !one && est_bracket(n, k, tu.sample, tu.z) >= 1048576.0;
    cudaError_t e = cudaSuccess;
    if (!one) {
        // (the finish holds CL_BLOCKS times as many, but a second pass over more
        // than these takes less time)
        a.list_max = Lim<KW>::ELEMS;
        // the bins are kept where they are likely to be needed
        if (1.2 * est_bracket(n, k, tu.sample, tu.z) <= (double)a.list_max && !(tu.flags & TOPK_FLAG_RAW_DELTA))
            a.bins = nullptr;
        a.plan_follows = resample;
        e = launch_dep(k_plan<DT>, CL_BLOCKS, CL_NT, sizeof(PlanSmem<KW>), st, CL_BLOCKS, a, 1);
        if (e != cudaSuccess) return cuda_status(e);
        if (ctx) profile_pass_begin(ctx, st);
        e = first_pass();
        if (e != cudaSuccess) return cuda_status(e);
        if (ctx) profile_pass_end(ctx, st);
        e = launch_dep(k_pass<DT>, pass_grid<DT>(sms, false), PASS_NT, 0, st, 1, a);
        a.plan_follows = 0;
        if (e == cudaSuccess && resample) {
            e = launch_dep(k_plan<DT>, CL_BLOCKS, CL_NT, sizeof(PlanSmem<KW>), st, CL_BLOCKS, a, 0);
            if (e == cudaSuccess) e = launch_dep(k_pass<DT>, pass_grid<DT>(sms, false), PASS_NT, 0, st, 1, a);
        }
        if (e != cudaSuccess) return cuda_status(e);
    }
    if (one && n <= SMALL_MAX) e = launch_dep(k_small<DT>, 1, BLK_NT, sizeof(SmallSmem<DT>), st, 1, a);
    else e = launch_dep(k_finish<DT>, CL_BLOCKS, CL_NT, sizeof(FinSmem<KW>), st, CL_BLOCKS, a, one ? 1 : 0);
    if (e != cudaSuccess) return cuda_status(e);
    if (ctx) count_launch(ctx, one ? 1 : resample ? 6 : 4);
    return cuda_status(cudaGetLastError());
}

// Scratch regions of one selection: reduction partials, the candidates' bins and the
// two candidate buffers (keys, then positions) of `cap` pairs each.
struct SelectCarve {
    size_t part, bins, k0, k1, i0, i1;
};
template <int KW> static Carve select_carve(u64 cap, int sms, SelectCarve& sc) {
    const size_t kbytes = KW / 8;
    Carve cv;
    sc.part = cv.take(sizeof(typename Comp<KW>::t) * (size_t)sms * EXT_BLOCKS_PER_SM);
    sc.bins = cv.take(sizeof(LevelBins));
    sc.k0 = cv.take(cap * kbytes);
    sc.k1 = cv.take(cap * kbytes);
    sc.i0 = cv.take(cap * 4);
    sc.i1 = cv.take(cap * 4);
    return cv;
}

template <int DT>
topk_status run_select(topk_ctx* ctx, const void* keys, u64 n, u64 k, void* out_keys, u32* out_idx,
                              void* kth_key, u32* kth_idx, const topk_params* prm, cudaStream_t st) {
    constexpr int KW = Key<DT>::KW;
    const Tuning tu = make_tuning<KW>(prm, ctx->sms);
    SelArgs a = make_args(keys, n, k, out_keys, out_idx, kth_key, kth_idx, tu);
    a.st = static_cast<SelState*>(ctx->d_state);
    a.err = ctx->d_err;
    ctx->last_kind = LAST_SELECT;

    const u64 cap = (k == 1 || k == n) ? 0 : candidate_capacity(n, k, tu);
    a.cap_b = cap;
    SelectCarve sc;
    const Carve cv = select_carve<KW>(cap, ctx->sms, sc);
    const size_t off_part = sc.part, off_bins = sc.bins, off_k0 = sc.k0, off_k1 = sc.k1, off_i0 = sc.i0,
                 off_i1 = sc.i1;
    topk_status rs = ensure_scratch(ctx, cv.off);
    if (rs != TOPK_OK) return rs;
    char* base = static_cast<char*>(ctx->scratch.base);
    a.bins = reinterpret_cast<LevelBins*>(base + off_bins);
    a.pass_done = ctx->d_counter + 2;
    a.cand_key[0] = base + off_k0;
    a.cand_key[1] = base + off_k1;
    a.cand_idx[0] = reinterpret_cast<u32*>(base + off_i0);
    a.cand_idx[1] = reinterpret_cast<u32*>(base + off_i1);
    return enqueue_select<DT>(ctx, a, tu, ctx->sms, ctx->d_counter, base + off_part, st);
}

// ------------------------------------------ entry point without allocation
// topk_select_noalloc runs the same kernels as topk_select, with every piece
// of scratch (state, error word, block-done counters, reduction partials, bins
// and the two candidate buffers) in one file-scope device array instead of a
// context's cudaMalloc'd block.  The array lives in every GPU that loads the
// library until the process exits.  Host code must not pass the array's name
// to a kernel (in host code it is only a stand-in for the symbol); its device
// address is looked up once per device with cudaGetSymbolAddress.

constexpr u64 NOALLOC_MAX_N = 1ull << 22;  // largest n accepted (4 Mi keys)
// Candidate pairs per buffer.  The context path sizes its buffers as
// candidate_capacity(n, k): twice the expected first bracket plus 4 T, which
// is largest at k = n/2 and, for n = 2^22 with the default tuning, is about
// 3.4e5 pairs for 32-bit keys (s = 16384) and 4.2e5 for 64-bit keys
// (s = 8192).  2^19 covers both, so no accepted call overflows more often
// than the same call through a context; the set-up checks this relation.
constexpr u64 NOALLOC_CAP = 1ull << 19;
constexpr size_t NA_OFF_STATE = 0;         // SelState
constexpr size_t NA_OFF_WORDS = 4096;      // [0] error, [1] reduction done, [2] pass done
constexpr size_t NA_OFF_PART = 8192;       // per-block composites of the k = 1 / k = n reduction
constexpr size_t NA_PART_BYTES = 64 * 1024;
constexpr size_t NA_OFF_BINS = NA_OFF_PART + NA_PART_BYTES; // bins of the first level's candidates
constexpr size_t NA_OFF_CAND = NA_OFF_BINS + ((sizeof(LevelBins) + 255) & ~(size_t)255);
constexpr size_t NA_BYTES = NA_OFF_CAND + 2 * NOALLOC_CAP * (8 + 4); // about 12.2 MiB

// Kernel attributes and the launch-geometry queries of every key type, so
// that no later call on this device makes them (they are made once per
// process and key type otherwise, on the first call with 1 < k < n).
template <int DT> topk_status noalloc_prepare_dt(int sms) {
    topk_status rs = set_smem_attrs<DT>();
    if (rs != TOPK_OK) return rs;
    (void)tma_grid<DT, PM_SPARSE>(sms);
    (void)tma_grid<DT, PM_DENSE>(sms);
    (void)pass_grid<DT>(sms, true);
    return cudaGetLastError() == cudaSuccess ? TOPK_OK : TOPK_ECUDA;
}

template <int DT>
topk_status run_select_noalloc(char* base, int sms, const void* keys, u64 n, u64 k, void* out_keys,
                                      u32* out_idx, void* kth_key, u32* kth_idx, u32* d_status,
                                      cudaStream_t st) {
    constexpr int KW = Key<DT>::KW;
    static_assert(sizeof(SelState) <= NA_OFF_WORDS, "state region too small");
    if ((size_t)sms * EXT_BLOCKS_PER_SM * sizeof(typename Comp<KW>::t) > NA_PART_BYTES) return TOPK_EINVAL;
    const Tuning tu = make_tuning<KW>(nullptr, sms);
    SelArgs a = make_args(keys, n, k, out_keys, out_idx, kth_key, kth_idx, tu);
    u32* words = reinterpret_cast<u32*>(base + NA_OFF_WORDS);
    a.st = reinterpret_cast<SelState*>(base + NA_OFF_STATE);
    a.err = d_status ? d_status : words;
    a.cap_b = NOALLOC_CAP;
    char* cand = base + NA_OFF_CAND;
    a.cand_key[0] = cand;
    a.cand_key[1] = cand + NOALLOC_CAP * 8;
    a.cand_idx[0] = reinterpret_cast<u32*>(cand + 2 * NOALLOC_CAP * 8);
    a.cand_idx[1] = reinterpret_cast<u32*>(cand + 2 * NOALLOC_CAP * 8 + NOALLOC_CAP * 4);
    a.bins = reinterpret_cast<LevelBins*>(base + NA_OFF_BINS);
    a.pass_done = words + 2;
    // the error word and the block-done counters must start at zero (a call that failed may have left them set)
    if (cudaMemsetAsync(words, 0, 4 * sizeof(u32), st) != cudaSuccess) return TOPK_ECUDA;
    if (d_status && cudaMemsetAsync(d_status, 0, sizeof(u32), st) != cudaSuccess) return TOPK_ECUDA;
    return enqueue_select<DT>(nullptr, a, tu, sms, words + 1, base + NA_OFF_PART, st);
}

// Explicit instantiation (one translation unit per key type) and the
// matching declarations for the translation unit of the C entry points.
#define TOPK_SELECT_TEMPLATES(PREFIX, DT)                                                                  \
    PREFIX template topk_status run_select<DT>(topk_ctx*, const void*, u64, u64, void*, u32*, void*, u32*,    \
                                               const topk_params*, cudaStream_t);                            \
    PREFIX template topk_status run_select<DT_DESC + DT>(topk_ctx*, const void*, u64, u64, void*, u32*, void*, \
                                                         u32*, const topk_params*, cudaStream_t);            \
    PREFIX template topk_status run_select_noalloc<DT>(char*, int, const void*, u64, u64, void*, u32*, void*,  \
                                                       u32*, u32*, cudaStream_t);                            \
    PREFIX template topk_status noalloc_prepare_dt<DT>(int);

} // namespace topk
