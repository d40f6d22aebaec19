// batched.cu — topk_select_batched: many independent selections (rows of
// uneven length, each with its own k) in one persistent launch.
//
// The paper has no batched form; each row is the selection of Section 2
// (Algorithm "select").  A row whose k is small (k_rows) is selected by one
// thread block in one read: a sample gives an upper pivot, the row is streamed
// and its elements up to the pivot gathered in shared memory, and the element of
// rank k among them ends the row.  Every other row takes the general path: up to
// the split length it is selected whole by one block, by levels of sample,
// pivots, a partitioning pass into the block's candidate buffer, the branch, and
// the exact finish among at most T candidates (k_batched, select_block.cuh); a
// longer ("wide") row takes its first level as topk_select does, over the whole
// GPU: one block samples the row and picks its pivots (k_wide_plan), one
// grid-wide pass streams the tiles of all wide rows and classifies each against
// its own row's pivots, the last block to finish a row taking the branch
// (k_wide_pass), and the persistent kernel then finishes the wide rows from
// their candidates while it selects the short rows whole.  Rows are handed out
// longest first from a device work queue, so the blocks that finish early take
// the short rows at the end.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>

#include "internal.h"
#include "select_block.cuh"

namespace topk {

constexpr u64 BATCH_CAP = 1ull << 16; // candidate pairs per buffer per block
constexpr u32 BATCH_SAMPLE = 2048;    // draws per level (rows are short)
constexpr u32 WIDE_NONE = 0xFFFFFFFFu;  // split length that makes no row wide
constexpr u32 WIDE_SPLIT = 1u << 15;    // default split length
constexpr u32 WIDE_SAMPLE = 2048;       // draws of a wide row's first level
constexpr u32 WIDE_TILE = PASS_NT * 16; // keys per tile of the wide pass
constexpr u64 WIDE_POOL_PAIRS = 1ull << 23; // candidate pairs of all wide rows together

// Block variants: NT threads, a sample / finish buffer of CAP composites
// (T <= CAP), at least MINB resident blocks per SM.  1024 threads are capped
// at 64 registers (some spill in the level code); 512 and 256 threads get
// 128 and hold half and a quarter of the composites, so smaller blocks run
// more rows at once per SM.
template <int KW, int NT> struct BatchVariant;
template <int KW> struct BatchVariant<KW, 1024> {
    static constexpr u32 CAP = Lim<KW>::ELEMS;
    static constexpr int MINB = 1;
};
template <int KW> struct BatchVariant<KW, 512> {
    static constexpr u32 CAP = Lim<KW>::ELEMS / 2;
    static constexpr int MINB = 1;
};
template <int KW> struct BatchVariant<KW, 256> {
    static constexpr u32 CAP = Lim<KW>::ELEMS / 4;
    static constexpr int MINB = 2;
};
template <int KW, int NT> using BatchSmem = BlockSmem<KW, NT, BatchVariant<KW, NT>::CAP>;

struct BatchArgs {
    const void* keys;
    const u64* row_off; // rows + 1
    const u32* row_k;   // rows
    u32 rows;
    void* out_keys;
    u32* out_idx;
    const u64* out_off; // rows + 1
    void* kth_keys;
    u32* kth_idx;
    // Rows given by pointers instead (used by the serving loop; when set, the
    // arrays above are ignored): row i has keys row_keys[i][0..row_n[i]),
    // outputs row_out_keys[i] / row_out_idx[i] (row_k[i] entries) and
    // row_kth_key[i] / row_kth_idx[i] (one entry).
    const void* const* row_keys;
    const u64* row_n;
    void* const* row_out_keys;
    u32* const* row_out_idx;
    void* const* row_kth_key;
    u32* const* row_kth_idx;
    u32* order;         // rows: row ids, longest first
    u32* mine;          // rows: those that k_rows takes, when it does not take them all
    u32* rest;          // rows left to the general path by k_rows (null: all rows)
    u32* nrest;         // their number (zero between calls)
    u32 sms;
    u32* rows_done;     // blocks of k_rows that are done (zero between kernels)
    u32 ordered;        // k_rows takes the rows in `order` from the queue, else row i in block i
    u32* queue;         // next index into order (zero from order_rows on)
    SelState* states;   // one per block
    char* cand;         // per block: key'[2][CAP], idx[2][CAP]
    u64 seed;
    u32 parts, sample, finish_T;
    float z;
    u32 flags;
    u32* err;
    // wide rows (row arrays only; WIDE_NONE: none)
    u32 key_bytes;      // width of a key
    u32 split;          // rows longer than this are wide
    u32* wide;          // rows: ids of the wide rows, longest first
    u32* words;         // [0] wide rows, [1] planning queue, [2] rows in order, [3] rows that k_rows takes
    u64* tile_pre;      // rows + 1: tiles of the wide rows before the j-th
    u32* done;          // rows: tiles of the row classified by the wide pass
    SelState* rstate;   // rows: state of each wide row
    u64* rcand;         // rows: the row's candidate buffer in the pool (pairs), ~0 = none
    char* pool;         // key'[pool_pairs], then idx[pool_pairs]
    u64 pool_pairs;
    u64* pool_next;     // pairs of the pool handed out
};

__device__ __forceinline__ bool is_wide(const BatchArgs& b, u64 len) {
    return b.split != WIDE_NONE && b.row_keys == nullptr && len > (u64)b.split;
}

// Tiles of the wide pass over a row: tile coordinates start at the 16-byte
// boundary at or below the row's first key (InputSrc), so the first tile
// holds `head` slots before it.
__device__ __forceinline__ u64 wide_tiles(const void* keys, u64 len, u32 key_bytes) {
    const u64 head = (u64)((reinterpret_cast<uintptr_t>(keys) & 15u) / (uintptr_t)key_bytes);
    return (len + head + WIDE_TILE - 1) / WIDE_TILE;
}

// Exclusive scan of one value per thread over a block of NT threads; *total
// receives the sum.  `ws` holds NT / 32 words.
template <int NT> __device__ __forceinline__ u32 block_excl_scan(u32 v, u32* ws, u32* total) {
    const u32 lane = lane_id(), warp = threadIdx.x >> 5;
    u32 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (u32)o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const u32 x = lane < NT / 32 ? ws[lane] : 0u;
        u32 wi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= (u32)o) wi += y;
        }
        if (lane < NT / 32) ws[lane] = wi - x;
        if (lane == 31) *total = wi;
    }
    __syncthreads();
    const u32 r = ws[warp] + incl - v;
    __syncthreads();
    return r;
}

__device__ __forceinline__ u64 row_len(const BatchArgs& b, u32 i) {
    return b.row_keys ? b.row_n[i] : b.row_off[i + 1] - b.row_off[i];
}

// Orders `rows` rows (src, or all of them) by floor(log2(length)), longest first
// (one block), and, for the general path (`lists`), lists the wide ones.
template <int NT>
__device__ void order_rows(const BatchArgs& b, const u32* src, u32 rows, bool lists) {
    __shared__ u32 hist[66], start[66];
    for (u32 i = threadIdx.x; i < 66; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    constexpr int U = 4; // rows whose loads are in flight together
    for (u32 i0 = threadIdx.x; i0 < rows; i0 += U * blockDim.x) {
        u32 cls[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u32 i = i0 + u * blockDim.x;
            const u64 len = i < rows ? row_len(b, src ? src[i] : i) : 0;
            cls[u] = i >= rows ? 66u : len ? 64 - __clzll((long long)len) : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (cls[u] < 66) atomicAdd(&hist[cls[u]], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        u32 run = 0;
        for (int k = 65; k >= 0; --k) {
            start[k] = run;
            run += hist[k];
        }
        b.words[2] = rows;
        *b.queue = 0;
    }
    __syncthreads();
    for (u32 i0 = threadIdx.x; i0 < rows; i0 += U * blockDim.x) {
        u32 cls[U], row[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u32 i = i0 + u * blockDim.x;
            row[u] = i < rows ? (src ? src[i] : i) : 0;
            const u64 len = i < rows ? row_len(b, row[u]) : 0;
            cls[u] = i >= rows ? 66u : len ? 64 - __clzll((long long)len) : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (cls[u] < 66) b.order[atomicAdd(&start[cls[u]], 1u)] = row[u];
    }
    if (!lists || b.split == WIDE_NONE || b.row_keys != nullptr) return;
    // the wide rows in queue order, with the prefix of their tile counts
    __syncthreads();
    __shared__ u32 ws[32], tot;
    __shared__ u64 carry_rows, carry_tiles;
    if (threadIdx.x == 0) {
        carry_rows = 0;
        carry_tiles = 0;
        *b.pool_next = 0;
        b.words[1] = 0;
    }
    __syncthreads();
    const unsigned char* base = static_cast<const unsigned char*>(b.keys);
    for (u32 c0 = 0; c0 < rows; c0 += NT) {
        const u32 i = c0 + threadIdx.x;
        u32 row = 0, flag = 0, tiles = 0;
        if (i < rows) {
            row = b.order[i];
            const u64 len = b.row_off[row + 1] - b.row_off[row];
            if (is_wide(b, len)) {
                flag = 1;
                tiles = (u32)wide_tiles(base + b.row_off[row] * (u64)b.key_bytes, len, b.key_bytes);
            }
        }
        const u32 rpos = block_excl_scan<NT>(flag, ws, &tot);
        const u32 nr = tot;
        const u32 tpos = block_excl_scan<NT>(tiles, ws, &tot);
        const u32 nt = tot;
        if (flag) {
            const u64 j = carry_rows + rpos;
            b.wide[j] = row;
            b.tile_pre[j] = carry_tiles + tpos;
            b.done[row] = 0;
            b.rcand[row] = ~0ull;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            carry_rows += nr;
            carry_tiles += nt;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        b.words[0] = (u32)carry_rows;
        b.tile_pre[carry_rows] = carry_tiles;
    }
}

constexpr int ROWS_NT = 256;
constexpr u32 ROWS_DRAW = 128;  // keys per draw of the sample
constexpr u64 ROWS_MAX = 1ull << 19; // longest row: beyond, one block's read takes longer than the general path
template <int KW> struct RowsCfg {
    static constexpr u32 CAP = KW == 32 ? 4096 : 2048; // elements of the list (32 KB)
    static constexpr u32 KMAX = CAP / 2;               // largest k: cutting back frees half the list
    // resident blocks: 64-bit keys spill 300 bytes of the 80 registers that three
    // leave (4096 rows of 2^U(10, 18) u64 keys 542 us with three, 395 with two)
    static constexpr int PER_SM = KW == 32 ? 3 : 2;
};

// Which rows k_rows (below) takes: one block reads such a row whole, at about 8.5
// keys per ns, while the general path spreads a long row over the whole GPU for
// about 42 us (its launches and barriers) and, in all, some 1e6 keys a us.  So a long
// row pays only in a batch that keeps the GPU busy with the others: the longest may
// exceed 7/8 of 2^17 keys by 1/128 of the batch's, and by 2^18 where the general
// path would also have to run blocks of its own for rows just below the split
// length, or for more rows than two waves of them.  When a row is longer than that,
// or its k too large, the general path runs in any case; then rows up to 1/256 of
// the keys that k_rows could take are still worth it (they save the general path
// more than they take), and rows up to the split length where that takes all its
// one-block work away or they are many.
// us by k_rows / by the general path, f32, k = 100: 1 row of 2^17 43 / 41, of 2^19
// 82 / 43; 64 rows of 2^18 59 / 66, of 2^19 101 / 88; 128 rows of 2^19 106 / 112; 64 rows
// of 2^U(10, 18) 53 / 73; 4000 rows of 2000 keys and 4 of 2^18 107 / 387.
struct RowsPlan {
    enum : u32 { LEFT = 1, MID = 2, MID_LEFT = 4 }; // rows left whatever the limit; rows of 2^13 keys to the split length
    u32 longest, shortest, nshort, flags;
    u64 keys;
};
// The longest row that k_rows takes (0: it takes none).  All NT threads call.
template <int KW, int NT> __device__ u32 rows_limit(const BatchArgs& b, RowsPlan& p) {
    if (b.row_keys || b.split == WIDE_NONE) return (u32)ROWS_MAX; // (no row is spread over the GPU)
    if (threadIdx.x == 0) p = RowsPlan{0u, 0xFFFFFFFFu, 0u, 0u, 0ull};
    __syncthreads();
    u32 mx = 0, mn = 0xFFFFFFFFu, ns = 0, fl = 0;
    u64 sum = 0;
    constexpr int U = 4; // rows whose loads are in flight together
    for (u32 i0 = threadIdx.x; i0 < b.rows; i0 += U * NT) {
        u64 len[U], rank[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const u32 i = i0 + u * NT < b.rows ? i0 + u * NT : i0;
            len[u] = row_len(b, i);
            rank[u] = b.row_k[i];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * NT >= b.rows) continue;
            const u64 n = len[u], k = rank[u];
            if (k == 0 || k > n || n > 0xFFFFFFFFull) {
                mn = 0; // (reported by whoever takes it)
                continue;
            }
            const bool mid = n > 8192 && n <= b.split;
            if (n > RowsCfg<KW>::CAP && k > RowsCfg<KW>::KMAX) {
                fl |= mid ? RowsPlan::LEFT | RowsPlan::MID_LEFT : RowsPlan::LEFT;
                continue;
            }
            fl |= (mid ? RowsPlan::MID : 0u) | (n > ROWS_MAX ? RowsPlan::LEFT : 0u);
            ns += (u32)(n <= b.split);
            sum += n <= ROWS_MAX ? n : 0;
            mx = max(mx, (u32)n);
            mn = min(mn, (u32)n);
        }
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    mn = __reduce_min_sync(0xffffffffu, mn);
    ns = __reduce_add_sync(0xffffffffu, ns);
    fl = __reduce_or_sync(0xffffffffu, fl);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, (unsigned long long)sum, o);
    if (lane_id() == 0) {
        atomicMax(&p.longest, mx);
        atomicMin(&p.shortest, mn);
        atomicAdd(&p.nshort, ns);
        atomicOr(&p.flags, fl);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.keys), (unsigned long long)sum);
    }
    __syncthreads();
    const u64 total = b.row_off[b.rows] - b.row_off[0];
    const bool many = p.nshort > 2 * b.sms;
    u64 limit = ROWS_MAX;
    if ((p.flags & RowsPlan::LEFT) || p.longest > (7ull << 14) + total / 128 + ((p.flags & RowsPlan::MID) || many ? 1ull << 18 : 0ull)) {
        limit = p.keys / 256 < ROWS_MAX ? p.keys / 256 : ROWS_MAX;
        if (limit < b.split) limit = many || (p.flags & (RowsPlan::MID | RowsPlan::MID_LEFT)) == RowsPlan::MID ? b.split : 0u;
    }
    return p.shortest <= limit ? (u32)limit : 0u;
}
template <int KW> __device__ __forceinline__ bool rows_takes(u64 n, u64 k, u32 limit) {
    return n <= limit && (n <= RowsCfg<KW>::CAP || k <= RowsCfg<KW>::KMAX);
}

// Rows in order for the general path, or, with k_rows (b.rest), the rows that it
// takes; the others go to its list of those it leaves.
template <int KW> __global__ void __launch_bounds__(1024) k_batch_order(BatchArgs b) {
    grid_dep_wait();
    grid_dep_release();
    if (!b.rest) {
        order_rows<1024>(b, nullptr, b.rows, true);
        return;
    }
    __shared__ RowsPlan plan;
    __shared__ u32 nmine, nrest;
    const u32 limit = rows_limit<KW, 1024>(b, plan);
    if (limit == 0) {
        if (threadIdx.x == 0) b.words[3] = 0;
        order_rows<1024>(b, nullptr, b.rows, true);
        return;
    }
    if (!b.row_keys && b.split != WIDE_NONE && !(plan.flags & RowsPlan::LEFT) && plan.longest <= limit) { // all of them
        if (threadIdx.x == 0) b.words[3] = b.rows;
        order_rows<1024>(b, nullptr, b.rows, false);
        return;
    }
    if (threadIdx.x == 0) nmine = nrest = 0;
    __syncthreads();
    for (u32 i = threadIdx.x; i < b.rows; i += 1024) {
        const u64 n = row_len(b, i), k = b.row_k[i];
        if (k == 0 || k > n || n > 0xFFFFFFFFull || rows_takes<KW>(n, k, limit)) b.mine[atomicAdd(&nmine, 1u)] = i;
        else b.rest[atomicAdd(&nrest, 1u)] = i;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        b.words[3] = nmine;
        *b.nrest = nrest;
    }
    order_rows<1024>(b, b.mine, nmine, false);
}

// Arguments of row `row` (keys at r0, n keys, rank k) for the selection
// code of select_block.cuh; state and candidate buffers set by the caller.
template <int DT>
__device__ __forceinline__ SelArgs row_args(const BatchArgs& b, u32 row, u64 r0, u64 n, u64 k) {
    typedef typename Key<DT>::raw_t raw_t;
    SelArgs a{};
    a.keys = static_cast<const raw_t*>(b.keys) + r0;
    a.out_keys = static_cast<raw_t*>(b.out_keys) + b.out_off[row];
    a.out_idx = b.out_idx + b.out_off[row];
    a.kth_key = static_cast<raw_t*>(b.kth_keys) + row;
    a.kth_idx = b.kth_idx + row;
    a.n = n;
    a.k = k;
    a.seed = b.seed ^ ((u64)row * 0x9E3779B97F4A7C15ull);
    a.parts = b.parts;
    a.sample = b.sample;
    a.finish_T = b.finish_T;
    a.z = b.z;
    a.flags = b.flags;
    a.aligned = 0;
    a.err = b.err;
    return a;
}

template <int KW> __device__ __forceinline__ typename Comp<KW>::key_t* pool_keys(const BatchArgs& b, u64 off) {
    return reinterpret_cast<typename Comp<KW>::key_t*>(b.pool) + off;
}
template <int KW> __device__ __forceinline__ u32* pool_idx(const BatchArgs& b, u64 off) {
    return reinterpret_cast<u32*>(b.pool + ((b.pool_pairs * sizeof(typename Comp<KW>::key_t) + 255) & ~(u64)255)) +
           off;
}

// ---------------------------------------------------- rows in one read
// Rows of small k (k_rows; which, see rows_limit), one block per row, rows longest
// first from a queue.
// A row of at most CAP keys is gathered whole; a longer one is sampled (about
// one key in 128), the sample element of rank k|S|/n + Delta is the bound, and
// the row is streamed once, every element up to the bound going to a list in
// shared memory; the element of rank k is selected in the list and the elements
// up to it are written.  A list that fills up is cut back to its k smallest,
// which tightens the bound; a row whose list ends with fewer than k elements
// (a bound that was too low) goes to the general path, as do rows of larger k.
//
// One read of the keys and no candidate buffers in memory.  Bound by the latency
// of the sampling and the selections, which the SM's other blocks cover with
// their reads: three blocks of 256 threads to an SM (80 registers) took 308 us
// for a program's pass over 4096 rows of 2^U(10, 18) f32 keys, four (64
// registers, spilled) 344, two 360, two of 512 threads 376.  By levels, whose wide
// rows went through memory three times and whose blocks waited on barriers, the
// same pass took 912 us (68 us of each are the program's own).
template <int KW> struct RowsSmem {
    typename Comp<KW>::t list[RowsCfg<KW>::CAP];
    HistSelSmem<KW> hs;
    u32 n, full_at, full, row, out;
    u32 last; // the block is the kernel's last (a word of its own: `row` may still be read)
    u32 lead[2][ROWS_NT / 32];
    RowsPlan plan;
    long long rank;
};

// Rank `r` among list[0..count), whatever their range.
template <int KW>
__device__ __noinline__ typename Comp<KW>::t rows_select(RowsSmem<KW>& sm, u32 count, u32 r) {
    typedef typename Comp<KW>::t ct;
    u32 mn = 0xFFFFFFFFu, mx = 0;
    for (u32 i = threadIdx.x; i < count; i += ROWS_NT) {
        const u32 w = (u32)(sm.list[i] >> KW);
        mn = min(mn, w);
        mx = max(mx, w);
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane_id() == 0) {
        sm.lead[0][threadIdx.x >> 5] = mn;
        sm.lead[1][threadIdx.x >> 5] = mx;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < ROWS_NT / 32; ++w) {
        mn = min(mn, sm.lead[0][w]);
        mx = max(mx, sm.lead[1][w]);
    }
    return block_select_hist<KW, ROWS_NT>(sm.list, count, (ct)mn << KW, ((ct)mx << KW) | (((ct)1 << KW) - 1), r, sm.hs);
}

// Keeps list[0..have)'s elements up to `thr` and opens the list again.
template <int KW> __device__ __noinline__ void rows_cut(RowsSmem<KW>& sm, u32 have, typename Comp<KW>::t thr) {
    typedef typename Comp<KW>::t ct;
    constexpr u32 OWN = RowsCfg<KW>::CAP / ROWS_NT;
    ct keep[OWN];
    u32 km = 0;
#pragma unroll
    for (u32 u = 0; u < OWN; ++u) {
        const u32 i = u * ROWS_NT + threadIdx.x;
        keep[u] = i < have ? sm.list[i] : ~(ct)0;
        km |= (u32)(i < have && keep[u] <= thr) << u;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        sm.n = 0;
        sm.full = 0;
        sm.full_at = 0xFFFFFFFFu;
    }
    __syncthreads();
    u32 slot = warp_reserve((u32)__popc(km), &sm.n);
#pragma unroll
    for (u32 u = 0; u < OWN; ++u)
        if ((km >> u) & 1u) sm.list[slot++] = keep[u];
    __syncthreads();
}

template <int DT> __global__ void __launch_bounds__(ROWS_NT, RowsCfg<Key<DT>::KW>::PER_SM) k_rows(BatchArgs b) {
    grid_dep_wait();
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef typename K::key_t key_t;
    constexpr int KW = K::KW;
    typedef Comp<KW> C;
    typedef typename C::t ct;
    constexpr u32 CAP = RowsCfg<KW>::CAP;
    constexpr int EPV = InputSrc<DT>::EPV, NV = InputSrc<DT>::NV;
    constexpr u32 SUB = 512; // keys of a warp's step: 16 per lane
    constexpr u32 WARPS = ROWS_NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto& sm = *reinterpret_cast<RowsSmem<KW>*>(smem_raw);
    const u32 tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const bool by_ptr = b.row_keys != nullptr;
    const u32 queued = b.ordered ? b.words[3] : 0u;
    auto next_row = [&]() -> u32 {
        if (!b.ordered) return 0xFFFFFFFFu;
        const u32 idx = atomicAdd(b.queue, 1u);
        return idx < queued ? b.order[idx] : 0xFFFFFFFFu;
    };
    u32 limit = (u32)ROWS_MAX; // (rows in order were chosen)
    if (b.ordered) {
        if (queued == 0) return;
    } else {
        limit = rows_limit<KW, ROWS_NT>(b, sm.plan);
        if (limit == 0) { // none: one block orders them all for the general path
            if (blockIdx.x == 0) order_rows<ROWS_NT>(b, nullptr, b.rows, true);
            return;
        }
    }
    u32 ahead = !b.ordered ? blockIdx.x : tid == 0 ? next_row() : 0u; // (no more blocks than rows)
    while (true) {
        if (tid == 0) {
            sm.row = ahead;
            sm.n = 0;
            sm.out = 0;
            sm.full = 0;
            sm.full_at = 0xFFFFFFFFu;
        }
        __syncthreads();
        const u32 row = sm.row;
        if (row == 0xFFFFFFFFu) break;
        if (tid == 0) ahead = next_row(); // (needed a whole row later)
        const u64 r0 = by_ptr ? 0 : b.row_off[row];
        const u64 n64 = by_ptr ? b.row_n[row] : b.row_off[row + 1] - r0;
        const u64 k64 = b.row_k[row];
        if (k64 == 0 || k64 > n64 || n64 > 0xFFFFFFFFull) {
            if (tid == 0) latch(b.err, ST_EINVAL);
            __syncthreads(); // sm.row is read by all
            continue;
        }
        const bool whole = n64 <= CAP;
        if (!rows_takes<KW>(n64, k64, limit)) {
            if (tid == 0) b.rest[atomicAdd(b.nrest, 1u)] = row;
            __syncthreads();
            continue;
        }
        const u32 n = (u32)n64, k = (u32)k64;
        const raw_t* keys = by_ptr ? static_cast<const raw_t*>(b.row_keys[row]) : static_cast<const raw_t*>(b.keys) + r0;
        ct thr = C::from128(key_domain_max<DT>()); // elements above it are passed over
        if (!whole) {
            // the bound, off a sample of about n / 128 draws, one in each of as many equal parts
            const u32 draws = min(max((n / ROWS_DRAW + 3u) & ~3u, 512u), CAP / 2);
            for (u32 j0 = tid * 4; j0 < draws; j0 += ROWS_NT * 4) {
                const Philox4 r = philox4x32_10(j0, row, 0x524F5753u, 0, (u32)b.seed, (u32)(b.seed >> 32));
                raw_t x[4];
                u32 pos[4];
#pragma unroll
                for (u32 q = 0; q < 4; ++q) {
                    const u32 lo = (u32)((u64)(j0 + q) * n / draws), hi = (u32)((u64)(j0 + q + 1) * n / draws);
                    pos[q] = lo + __umulhi(r.v[q], hi - lo);
                    x[q] = keys[pos[q]];
                }
#pragma unroll
                for (u32 q = 0; q < 4; ++q) sm.list[j0 + q] = C::make(K::fwd(x[q]), pos[q]);
            }
            if (tid == 0) {
                long long jl, jr;
                pivot_ranks(draws, n, k, b.z, false, jl, jr);
                sm.rank = jr;
            }
            __syncthreads();
            const long long jr = sm.rank;
            if (jr < (long long)draws) thr = rows_select<KW>(sm, draws, (u32)jr);
            __syncthreads(); // the list is free again
        }
        // the stream: steps of 512 keys, warp by warp, on 16-byte boundaries
        const u32 head = (u32)((reinterpret_cast<uintptr_t>(keys) & 15u) / sizeof(raw_t));
        const uint4* vec = reinterpret_cast<const uint4*>(reinterpret_cast<uintptr_t>(keys) & ~(uintptr_t)15);
        const u32 ext = n + head, subs = (ext + SUB - 1) / SUB;
        u32 t = warp;
        auto inside = [&](u32 s) { return s < subs && s * SUB >= head && (s + 1) * SUB <= ext; };
        auto load = [&](u32 s, uint4(&v)[NV]) {
            if (inside(s)) {
#pragma unroll
                for (int j = 0; j < NV; ++j) v[j] = __ldcs(vec + (size_t)s * (SUB / EPV) + j * 32 + lane);
            }
        };
        while (true) {
            const key_t tk = (key_t)C::key(thr);
            const u32 tx = C::idx(thr);
            // ties with the bound's key count up to its position
            const RawBound<DT> upto = RawBound<DT>::le(tk), under = RawBound<DT>::le((key_t)(tk - 1));
            uint4 v[NV];
            load(t, v);
            while (t < subs) {
                uint4 w[NV];
                load(t + WARPS, w);
                const u32 e0 = t * SUB; // slot q is element e0 + ((q / EPV) * 32 + lane) * EPV + q % EPV
                auto pos = [&](int q) -> u32 { return e0 + (u32)((q / EPV) * 32 + lane) * EPV + (u32)(q % EPV) - head; };
                raw_t rr[16];
                u32 hit = 0;
                if (inside(t)) {
                    InputSrc<DT>::unpack_raw(v, rr);
                    const u32 p0 = e0 - head;
                    if (p0 + (SUB - 1) <= tx) hit = tile_le_dispatch<DT>(rr, upto, true);
                    else if (p0 > tx) hit = tile_le_dispatch<DT>(rr, under, tk != 0);
                    else {
#pragma unroll
                        for (int q = 0; q < 16; ++q) hit |= (u32)(C::make(K::fwd(rr[q]), pos(q)) <= thr) << q;
                    }
                } else { // the row's first or last step
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const u32 e = e0 + (u32)((q / EPV) * 32 + lane) * EPV + (u32)(q % EPV);
                        rr[q] = 0;
                        if (e >= head && e < ext) {
                            rr[q] = reinterpret_cast<const raw_t*>(vec)[e];
                            hit |= (u32)(C::make(K::fwd(rr[q]), e - head) <= thr) << q;
                        }
                    }
                }
                if (__any_sync(0xffffffffu, hit)) {
                    const u32 total = __reduce_add_sync(0xffffffffu, (u32)__popc(hit));
                    u32 at = 0;
                    if (lane == 0) at = atomicAdd(&sm.n, total);
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (at + total > CAP) { // full: every later reservation fails too, so nothing lies beyond `at`
                        if (lane == 0) {
                            atomicMin(&sm.full_at, at);
                            *(volatile u32*)&sm.full = 1;
                        }
                        break;
                    }
                    // one hit of every lane that has any at a time (few: one or two turns)
                    const u32 below = lanemask_lt();
                    u32 bal = __ballot_sync(0xffffffffu, hit);
                    do {
                        if (hit) {
                            const u32 q = (u32)(__ffs(hit) - 1);
                            hit &= hit - 1;
                            sm.list[at + (u32)__popc(bal & below)] = C::make(K::fwd(pick16(rr, q)), pos((int)q));
                        }
                        at += (u32)__popc(bal);
                        bal = __ballot_sync(0xffffffffu, hit);
                    } while (bal);
                }
                t += WARPS;
                if (__any_sync(0xffffffffu, *(volatile u32*)&sm.full)) break;
#pragma unroll
                for (int j = 0; j < NV; ++j) v[j] = w[j];
            }
            __syncthreads();
            if (!sm.full) break;
            // cut the list back to its k smallest and go on below the k-th
            const u32 have = min(sm.n, sm.full_at);
            if (have < k) break; // (k <= CAP / 2 and a step adds at most 512: cannot be)
            thr = rows_select<KW>(sm, have, k - 1);
            rows_cut<KW>(sm, have, thr);
        }
        const u32 count = min(sm.n, sm.full_at);
        if (count < k) { // the bound was too low
            if (tid == 0) b.rest[atomicAdd(b.nrest, 1u)] = row;
            __syncthreads();
            continue;
        }
        const ct kth = count == k && k == 1 ? sm.list[0] : rows_select<KW>(sm, count, k - 1);
        raw_t* ok = by_ptr ? static_cast<raw_t*>(b.row_out_keys[row]) : static_cast<raw_t*>(b.out_keys) + b.out_off[row];
        u32* oi = by_ptr ? b.row_out_idx[row] : b.out_idx + b.out_off[row];
        for (u32 base = 0; base < count; base += ROWS_NT * 8) {
            u32 selm = 0;
#pragma unroll
            for (u32 u = 0; u < 8; ++u) {
                const u32 i = base + u * ROWS_NT + tid;
                selm |= (u32)(i < count && sm.list[i] <= kth) << u;
            }
            u32 slot = warp_reserve((u32)__popc(selm), &sm.out);
            while (selm) {
                const u32 u = (u32)(__ffs(selm) - 1);
                selm &= selm - 1;
                const ct c = sm.list[base + u * ROWS_NT + tid];
                if (slot < k) {
                    ok[slot] = K::inv((key_t)C::key(c));
                    oi[slot] = C::idx(c);
                }
                ++slot;
            }
        }
        if (tid == 0) {
            *(by_ptr ? static_cast<raw_t*>(b.row_kth_key[row]) : static_cast<raw_t*>(b.kth_keys) + row) =
                K::inv((key_t)C::key(kth));
            *(by_ptr ? b.row_kth_idx[row] : b.kth_idx + row) = C::idx(kth);
        }
        __syncthreads(); // the row's shared words are done with
    }
    // the last block orders the rows left to the general path
    if (tid == 0) {
        __threadfence();
        sm.last = atomicAdd(b.rows_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!sm.last) return;
    __threadfence();
    const u32 left = *(volatile u32*)b.nrest;
    __syncthreads();
    order_rows<ROWS_NT>(b, b.rest, left, true);
    if (tid == 0) {
        *b.rows_done = 0;
        *b.nrest = 0;
    }
}

// First level of the wide rows, part 1 (one block of 256 threads per row,
// persistent over a queue, several blocks per SM): the row's sample and pivots (plan_level, with
// the larger sample of a first level), then a candidate buffer from the
// pool: twice the bracket the pivots' sample ranks predict plus a margin, at
// most BATCH_CAP pairs.  A row the pool cannot serve is left whole to the
// persistent kernel.
constexpr int WIDE_PLAN_NT = 256;

template <int DT> __global__ void __launch_bounds__(WIDE_PLAN_NT) k_wide_plan(BatchArgs b) {
    grid_dep_wait();
    constexpr int KW = Key<DT>::KW;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto& sm = *reinterpret_cast<BatchSmem<KW, WIDE_PLAN_NT>*>(smem_raw);
    __shared__ u32 s_row;
    const u32 nwide = b.words[0];
    while (true) {
        if (threadIdx.x == 0) {
            const u32 j = atomicAdd(&b.words[1], 1u);
            s_row = j < nwide ? b.wide[j] : 0xFFFFFFFFu;
        }
        __syncthreads();
        const u32 row = s_row;
        __syncthreads();
        if (row == 0xFFFFFFFFu) break;
        const u64 r0 = b.row_off[row], n = b.row_off[row + 1] - r0, k = b.row_k[row];
        if (k == 0 || k > n || n > 0xFFFFFFFFull) continue; // reported by the persistent kernel
        SelArgs a = row_args<DT>(b, row, r0, n, k);
        SelState* g = b.rstate + row;
        a.st = g;
        a.sample = WIDE_SAMPLE < BatchSmem<KW, WIDE_PLAN_NT>::ELEMS ? WIDE_SAMPLE : BatchSmem<KW, WIDE_PLAN_NT>::ELEMS;
        a.cap_b = 0;
        if (threadIdx.x == 0) init_state<DT>(g, a);
        __syncthreads();
        plan_level<DT>(a, sm, true);
        if (threadIdx.x == 0) {
            double est = (double)n;
            const long long top = (long long)sm.kept - 1;
            if (sm.kept > 0) {
                const long long l = sm.jl < 0 ? 0 : sm.jl, r = sm.jr > top ? top : sm.jr;
                est = (double)(r - l + 1) / (double)sm.kept * (double)n;
            }
            u64 cap = (u64)(2.0 * est) + 2048;
            cap = cap < n ? cap : n;
            cap = cap < BATCH_CAP ? cap : BATCH_CAP;
            cap = (cap + 255) & ~(u64)255;
            const u64 off = atomicAdd(reinterpret_cast<unsigned long long*>(b.pool_next), (unsigned long long)cap);
            if (off + cap <= b.pool_pairs) {
                g->cap_b = cap;
                b.rcand[row] = off;
            }
        }
        __syncthreads();
    }
}

__device__ __forceinline__ u64 atomic_read_u64(u64* p) {
    return atomicAdd(reinterpret_cast<unsigned long long*>(p), 0ull);
}

// First level of the wide rows, part 2: the tiles of all wide rows, in
// order, split into one contiguous run per block.  Every element is
// classified against its own row's pivots (the window is the whole row:
// a below pl, b from pl to pr); a- and b-elements leave with one reservation
// per warp and class on the row's counters.  Each warp adds its part of the
// tiles it classified of a row to the row's done count when it leaves the
// row (no block barrier); the warp that completes a row takes the branch of
// Algorithm "select" for it.
template <int DT> struct WideRow {
    typedef Comp<Key<DT>::KW> C;
    u32 row;
    u64 t0, t1;      // the row's tiles [t0, t1)
    bool live;       // the row has a candidate buffer
    typename C::t pl, pr;
    TileBounds<DT> tbd; // bounds on raw key bits for tiles away from the pivots' positions
    SelState* g;
    InputSrc<DT> src;
    Sink<DT> sink;
};

template <int DT> __device__ __forceinline__ void wide_row_open(const BatchArgs& b, u32 j, WideRow<DT>& w) {
    typedef Key<DT> K;
    typedef Comp<K::KW> C;
    w.row = b.wide[j];
    w.t0 = b.tile_pre[j];
    w.t1 = b.tile_pre[j + 1];
    const u64 off = b.rcand[w.row];
    w.live = off != ~0ull;
    if (!w.live) return;
    w.g = b.rstate + w.row;
    w.pl = C::from128(w.g->pl);
    w.pr = C::from128(w.g->pr);
    w.tbd = TileBounds<DT>::make(w.pl, w.pr);
    const u64 r0 = b.row_off[w.row];
    w.src = InputSrc<DT>::make(static_cast<const typename K::raw_t*>(b.keys) + r0, b.row_off[w.row + 1] - r0);
    w.sink.out_keys = static_cast<typename K::raw_t*>(b.out_keys) + b.out_off[w.row];
    w.sink.out_idx = b.out_idx + b.out_off[w.row];
    w.sink.out_base = 0;
    w.sink.cap_a = w.g->k_rem;
    w.sink.ck = pool_keys<K::KW>(b, off);
    w.sink.ci = pool_idx<K::KW>(b, off);
    w.sink.cap_b = w.g->cap_b;
    w.sink.cnt_a = &w.g->cnt_a;
    w.sink.cnt_b = &w.g->cnt_b;
}

// A warp leaves row w after classifying its part of `n` of the row's tiles
// (one lane; every tile is classified by `parts` warps): the warp that
// completes the row's count takes the branch.
template <int DT>
__device__ __forceinline__ void wide_row_close(const BatchArgs& b, const WideRow<DT>& w, u32 n, u32 parts) {
    if (!w.live || n == 0) return;
    __threadfence();
    const u32 prev = atomicAdd(&b.done[w.row], n);
    if ((u64)prev + n == (w.t1 - w.t0) * parts) { // all of the row's tiles: the branch
        __threadfence();
        w.g->cnt_a = atomic_read_u64(&w.g->cnt_a);
        w.g->cnt_b = atomic_read_u64(&w.g->cnt_b);
        decide(*w.g);
    }
}

// The wide pass streams with the bulk-copy engine: one producer warp copies
// the block's tiles, in order, into a ring of shared-memory stages and
// records each tile's wide row and extent; eight consumer warps classify.  A
// tile is copied from the 16-byte boundary at or below its first slot up to
// the last 16-byte boundary inside its row (so no copy reads past the row);
// the few keys after that boundary are read directly.
constexpr int WIDE_CONS = 256;               // consumer threads
constexpr int WIDE_NT = WIDE_CONS + 32;      // plus the producer warp
constexpr u64 WIDE_WAIT_NS = 200ull * 1000 * 1000;
static_assert(WIDE_CONS * 16 == (int)WIDE_TILE, "a tile is 16 keys per consumer thread");

template <int DT> struct WideCfg {
    static constexpr u32 W = sizeof(typename Key<DT>::raw_t);
    static constexpr u32 BYTES = WIDE_TILE * W;
    static constexpr u32 STAGES = W == 2 ? 8 : W == 4 ? 5 : 3;
    static constexpr u32 SMEM = STAGES * BYTES;
};

struct WideMeta {
    u32 j;      // index into the wide rows
    u32 bytes;  // bytes copied into the stage
    u64 tb;     // tile coordinate of the stage's first slot
};

template <int DT> __global__ void __launch_bounds__(WIDE_NT, 2) k_wide_pass(BatchArgs b) {
    grid_dep_wait();
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef typename K::key_t key_t;
    constexpr int KW = K::KW;
    typedef Comp<KW> C;
    typedef typename C::t ct;
    typedef WideCfg<DT> Cfg;
    constexpr int EPV = InputSrc<DT>::EPV;
    extern __shared__ __align__(128) unsigned char stages[];
    __shared__ __align__(8) uint64_t full[Cfg::STAGES];
    __shared__ __align__(8) uint64_t empty[Cfg::STAGES];
    __shared__ WideMeta meta[Cfg::STAGES];
    __shared__ WarpQ<KW> wqs[WIDE_CONS / 32];
    __shared__ u32 dead;
    const u32 nwide = b.words[0];
    if (nwide == 0) return;
    const u64 total = b.tile_pre[nwide];
    const u64 per = (total + gridDim.x - 1) / gridDim.x;
    const u64 t0 = (u64)blockIdx.x * per;
    const u64 t1 = t0 + per < total ? t0 + per : total;
    if (t0 >= t1) return;
    if (threadIdx.x == 0) {
        for (u32 i = 0; i < Cfg::STAGES; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], WIDE_CONS / 32);
        }
        dead = 0;
        mbar_fence_init();
    }
    __syncthreads();
    // the wide row holding tile t0: tile_pre[j] <= t0 < tile_pre[j + 1]
    u32 lo = 0, hi = nwide;
    while (hi - lo > 1) {
        const u32 mid = (lo + hi) >> 1;
        if (b.tile_pre[mid] <= t0) lo = mid;
        else hi = mid;
    }
    const unsigned char* kbase = static_cast<const unsigned char*>(b.keys);
    if (threadIdx.x >= WIDE_CONS) { // producer warp: one lane issues the copies
        if (threadIdx.x == WIDE_CONS) {
            u32 j = lo, stg = 0, epar = 1; // the first pass over the ring waits for nothing
            for (u64 t = t0; t < t1; ++t) {
                while (b.tile_pre[j + 1] <= t) ++j;
                if (t - t0 >= Cfg::STAGES) {
                    if (*(volatile u32*)&dead || !mbar_wait_bounded(&empty[stg], epar, WIDE_WAIT_NS)) {
                        *(volatile u32*)&dead = 1;
                        latch(b.err, ST_ETIMEOUT);
                        break;
                    }
                }
                const u32 row = b.wide[j];
                const u64 tb = (t - b.tile_pre[j]) * (u64)WIDE_TILE;
                const unsigned char* first = kbase + b.row_off[row] * Cfg::W;
                const unsigned char* abase = reinterpret_cast<const unsigned char*>(
                    reinterpret_cast<uintptr_t>(first) & ~(uintptr_t)15);
                const unsigned char* src = abase + tb * Cfg::W;
                const unsigned char* row_end = kbase + b.row_off[row + 1] * Cfg::W;
                const uintptr_t lim = reinterpret_cast<uintptr_t>(row_end) & ~(uintptr_t)15;
                u32 bytes = 0;
                if (reinterpret_cast<uintptr_t>(src) < lim) {
                    const uintptr_t avail = lim - reinterpret_cast<uintptr_t>(src);
                    bytes = avail < Cfg::BYTES ? (u32)avail : Cfg::BYTES;
                }
                meta[stg].j = j;
                meta[stg].bytes = bytes;
                meta[stg].tb = tb;
                mbar_arrive_expect_tx(&full[stg], bytes);
                if (bytes) bulk_g2s(stages + (size_t)stg * Cfg::BYTES, src, bytes, &full[stg]);
                if (++stg == Cfg::STAGES) {
                    stg = 0;
                    epar ^= 1u;
                }
            }
        }
        return;
    }
    // consumers: the hits (pair <= pr) go to the warp's per-lane queue,
    // classified and reserved in batches (select_core.cuh), drained when the
    // warp leaves the row
    const u32 lane = lane_id();
    WarpQ<KW>& wq = wqs[threadIdx.x >> 5];
    LQState qs = LQState::make();
    const ct lo0 = 0;
    WideRow<DT> w;
    w.row = 0xFFFFFFFFu;
    w.live = false;
    u32 j_cur = 0xFFFFFFFFu, ndone = 0;
    for (u64 t = t0; t < t1; ++t) {
        const u32 i = (u32)(t - t0);
        const u32 stg = i % Cfg::STAGES;
        const u32 par = (i / Cfg::STAGES) & 1u;
        bool ok = !*(volatile u32*)&dead;
        if (ok && !mbar_wait_bounded(&full[stg], par, WIDE_WAIT_NS)) {
            ok = false;
            *(volatile u32*)&dead = 1;
            if (lane == 0) latch(b.err, ST_ETIMEOUT);
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) continue; // timed out: latched; the remaining waits return at once
        const WideMeta m = meta[stg];
        if (m.j != j_cur) { // a new row: this warp leaves the previous one
            if (w.live) lq_drain<DT>(wq, qs, w.sink, lo0, w.pl, w.pr);
            __syncwarp();
            if (lane == 0 && j_cur != 0xFFFFFFFFu) wide_row_close<DT>(b, w, ndone, WIDE_CONS / 32);
            ndone = 0;
            j_cur = m.j;
            wide_row_open<DT>(b, j_cur, w);
        }
        if (w.live) {
            // slot q of this thread: tile element tb + (q / EPV) * 256 * EPV + tid * EPV + q % EPV
            const unsigned char* mine = stages + (size_t)stg * Cfg::BYTES + threadIdx.x * 16u;
            const u64 ext = w.src.extent();
            // row position of the tile's slot 0 (32 bits: rows are shorter than 2^32)
            const u32 pbase = (u32)(m.tb - w.src.head);
            auto pos = [&](int q) -> u32 {
                return pbase + (u32)((q / EPV) * WIDE_CONS * EPV) + threadIdx.x * EPV + (u32)(q % EPV);
            };
            key_t kk[16];
            u32 hit = 0;
            if (m.tb >= w.src.head && m.tb + WIDE_TILE <= ext && m.bytes == Cfg::BYTES) {
                // a tile inside the row, wholly in the stage
                raw_t rr[16];
                {
                    uint4 v[InputSrc<DT>::NV];
#pragma unroll
                    for (int jj = 0; jj < InputSrc<DT>::NV; ++jj)
                        v[jj] = *reinterpret_cast<const uint4*>(mine + jj * (WIDE_CONS * 16u));
                    InputSrc<DT>::unpack_raw(v, rr);
                }
                RawBound<DT> ba, bb;
                bool any_a, any_l;
                if (w.tbd.get(pbase, pbase + WIDE_TILE - 1, ba, bb, any_a, any_l)) {
                    hit = tile_le_dispatch<DT>(rr, bb, any_l);
                } else {
#pragma unroll
                    for (int q = 0; q < 16; ++q) hit |= (u32)(C::make(K::fwd(rr[q]), pos(q)) <= w.pr) << q;
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) kk[q] = K::fwd(rr[q]);
            } else {
                // the row's first or last tile: slots outside the row, keys past the stage
                const u32 in_stage = m.bytes / Cfg::W; // slots held by the stage
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const u32 so = (u32)((q / EPV) * WIDE_CONS * EPV) + threadIdx.x * EPV + (u32)(q % EPV);
                    const u64 e = m.tb + so;
                    kk[q] = 0;
                    if (e >= w.src.head && e < ext) {
                        raw_t r;
                        if (so < in_stage)
                            r = *reinterpret_cast<const raw_t*>(mine + (q / EPV) * (WIDE_CONS * 16u) +
                                                                (q % EPV) * sizeof(raw_t));
                        else r = w.src.keys[e]; // past the last 16-byte boundary of the row
                        kk[q] = K::fwd(r);
                        hit |= (u32)(C::make(kk[q], pos(q)) <= w.pr) << q;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[stg]); // keys are in registers
            lq_append<DT>(hit, pos, [&](u32 sq) { return pick16(kk, sq); }, lo0, w.pl, w.pr, w.sink, wq, qs);
            ++ndone;
        } else {
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[stg]);
        }
    }
    if (w.live) lq_drain<DT>(wq, qs, w.sink, lo0, w.pl, w.pr);
    __syncwarp();
    if (lane == 0 && j_cur != 0xFFFFFFFFu) wide_row_close<DT>(b, w, ndone, WIDE_CONS / 32);
}

template <int DT, int NT>
__global__ void __launch_bounds__(NT, (BatchVariant<Key<DT>::KW, NT>::MINB)) k_batched(BatchArgs b) {
    grid_dep_wait();
    typedef Key<DT> K;
    typedef typename K::raw_t raw_t;
    typedef typename K::key_t key_t;
    constexpr int KW = K::KW;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto& sm = *reinterpret_cast<BatchSmem<KW, NT>*>(smem_raw);
    __shared__ u32 s_row, s_rows;
    SelState* g = b.states + blockIdx.x;
    char* cand = b.cand + (size_t)blockIdx.x * 2 * BATCH_CAP * (sizeof(key_t) + 4);
    if (threadIdx.x == 0) s_rows = b.words[2];
    while (true) {
        if (threadIdx.x == 0) {
            const u32 idx = atomicAdd(b.queue, 1u);
            s_row = idx < s_rows ? b.order[idx] : 0xFFFFFFFFu;
        }
        __syncthreads();
        const u32 row = s_row;
        __syncthreads();
        if (row == 0xFFFFFFFFu) break;
        const bool by_ptr = b.row_keys != nullptr;
        const u64 r0 = by_ptr ? 0 : b.row_off[row];
        const u64 n = by_ptr ? b.row_n[row] : b.row_off[row + 1] - r0;
        const u64 k = b.row_k[row];
        if (k == 0 || k > n || n > 0xFFFFFFFFull) {
            if (threadIdx.x == 0) latch(b.err, ST_EINVAL);
            continue;
        }
        if (!by_ptr && is_wide(b, n) && b.rcand[row] != ~0ull) {
            // a wide row whose first level ran over the grid: finish it from
            // its candidates (further levels alternate between the row's
            // buffer and this block's second buffer)
            SelArgs a = row_args<DT>(b, row, r0, n, k);
            SelState* gw = b.rstate + row;
            const u64 off = b.rcand[row];
            a.cand_key[0] = pool_keys<KW>(b, off);
            a.cand_idx[0] = pool_idx<KW>(b, off);
            a.cand_key[1] = cand + BATCH_CAP * sizeof(key_t);
            a.cand_idx[1] = reinterpret_cast<u32*>(cand + 2 * BATCH_CAP * sizeof(key_t) + BATCH_CAP * 4);
            a.st = gw;
            a.cap_b = gw->cap_b;
            block_levels_and_finish<DT>(a, sm);
            __syncthreads();
            continue;
        }
        SelArgs a{};
        if (by_ptr) {
            a.keys = b.row_keys[row];
            a.out_keys = b.row_out_keys[row];
            a.out_idx = b.row_out_idx[row];
            a.kth_key = b.row_kth_key[row];
            a.kth_idx = b.row_kth_idx[row];
        } else {
            a.keys = static_cast<const raw_t*>(b.keys) + r0;
            a.out_keys = static_cast<raw_t*>(b.out_keys) + b.out_off[row];
            a.out_idx = b.out_idx + b.out_off[row];
            a.kth_key = static_cast<raw_t*>(b.kth_keys) + row;
            a.kth_idx = b.kth_idx + row;
        }
        a.n = n;
        a.k = k;
        a.cand_key[0] = cand;
        a.cand_key[1] = cand + BATCH_CAP * sizeof(key_t);
        a.cand_idx[0] = reinterpret_cast<u32*>(cand + 2 * BATCH_CAP * sizeof(key_t));
        a.cand_idx[1] = reinterpret_cast<u32*>(cand + 2 * BATCH_CAP * sizeof(key_t) + BATCH_CAP * 4);
        a.st = g;
        a.cap_b = BATCH_CAP;
        a.seed = b.seed ^ ((u64)row * 0x9E3779B97F4A7C15ull);
        a.parts = b.parts;
        a.sample = b.sample;
        a.finish_T = b.finish_T;
        a.z = b.z;
        a.flags = b.flags;
        a.aligned = 0;
        a.err = b.err;
        if (threadIdx.x == 0) {
            init_state<DT>(g, a);
            g->phase = PH_FINISH;
        }
        __syncthreads();
        block_levels_and_finish<DT>(a, sm);
        __syncthreads();
    }
}

// Resident blocks per SM of one variant (once per device and variant).
template <int DT, int NT> static int batched_blocks_per_sm(int device, topk_status& rs) {
    constexpr int KW = Key<DT>::KW;
    static std::atomic<int> occ[64];
    int& o0 = *reinterpret_cast<int*>(&occ[device & 63]);
    int o = occ[device & 63].load();
    rs = TOPK_OK;
    if (o == 0) {
        if (cudaFuncSetAttribute(k_batched<DT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(BatchSmem<KW, NT>)) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_batched<DT, NT>, NT, sizeof(BatchSmem<KW, NT>)) !=
                cudaSuccess) {
            rs = TOPK_ECUDA;
            return 0;
        }
        o = std::max(1, o);
        occ[device & 63].store(o);
    }
    (void)o0;
    return o;
}

// Resident blocks per SM of the wide pass, and the planning kernel's
// shared-memory attribute (once per device and key type).
template <int DT> static topk_status wide_setup(int device, int& pass_per_sm, int& plan_per_sm) {
    constexpr int KW = Key<DT>::KW;
    static std::atomic<int> occ[64];
    int o = occ[device & 63].load();
    if (o == 0) {
        int op = 0;
        if (cudaFuncSetAttribute(k_wide_plan<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(BatchSmem<KW, WIDE_PLAN_NT>)) != cudaSuccess ||
            cudaFuncSetAttribute(k_wide_pass<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)WideCfg<DT>::SMEM) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_wide_pass<DT>, WIDE_NT, WideCfg<DT>::SMEM) !=
                cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&op, k_wide_plan<DT>, WIDE_PLAN_NT,
                                                          sizeof(BatchSmem<KW, WIDE_PLAN_NT>)) != cudaSuccess)
            return TOPK_ECUDA;
        o = std::max(1, o) | (std::max(1, op) << 16);
        occ[device & 63].store(o);
    }
    pass_per_sm = o & 0xFFFF;
    plan_per_sm = o >> 16;
    return TOPK_OK;
}

template <int DT, int NT>
static topk_status launch_batched(topk_ctx* ctx, BatchArgs b, cudaStream_t st) {
    constexpr int KW = Key<DT>::KW;
    topk_status rs;
    const int per_sm = batched_blocks_per_sm<DT, NT>(ctx->device, rs);
    if (rs != TOPK_OK) return rs;
    int pass_per_sm = 1, plan_per_sm = 1;
    if (b.split != WIDE_NONE && (rs = wide_setup<DT>(ctx->device, pass_per_sm, plan_per_sm)) != TOPK_OK) return rs;
    // rows that all start at once need no order
    b.ordered = b.rows > (u32)ctx->sms * RowsCfg<KW>::PER_SM;
    const bool order = b.ordered || !b.rest;
    cudaError_t e = order ? launch_dep(k_batch_order<KW>, 1, 1024, 0, st, 1, b) : cudaSuccess;
    if (e == cudaSuccess && b.rest) {
        static std::atomic<uint64_t> attr{0};
        const uint64_t bit = 1ull << (ctx->device & 63);
        if (!(attr.load() & bit)) {
            if (cudaFuncSetAttribute(k_rows<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(RowsSmem<KW>)) != cudaSuccess)
                return TOPK_ECUDA;
            attr.fetch_or(bit);
        }
        const int grid = (int)std::min<u64>(b.rows, (u64)ctx->sms * RowsCfg<KW>::PER_SM);
        e = launch_dep(k_rows<DT>, grid, ROWS_NT, sizeof(RowsSmem<KW>), st, 1, b);
    }
    if (e == cudaSuccess && b.split != WIDE_NONE) {
        e = launch_dep(k_wide_plan<DT>, ctx->sms * plan_per_sm, WIDE_PLAN_NT, sizeof(BatchSmem<KW, WIDE_PLAN_NT>), st, 1,
                       b);
        if (e == cudaSuccess)
            e = launch_dep(k_wide_pass<DT>, ctx->sms * pass_per_sm, WIDE_NT, WideCfg<DT>::SMEM, st, 1, b);
    }
    if (e == cudaSuccess) e = launch_dep(k_batched<DT, NT>, ctx->sms * per_sm, NT, sizeof(BatchSmem<KW, NT>), st, 1, b);
    if (e != cudaSuccess) return cuda_status(e);
    count_launch(ctx, (order ? 1 : 0) + (b.rest ? 1 : 0) + (b.split != WIDE_NONE ? 3 : 1));
    return cuda_status(cudaGetLastError());
}

// Largest resident grid over the variants: the number of per-block states
// and candidate buffers the scratch must hold.
template <int DT> static int batched_max_grid(topk_ctx* ctx, topk_status& rs) {
    int m = 0;
    for (int v : {batched_blocks_per_sm<DT, 1024>(ctx->device, rs), batched_blocks_per_sm<DT, 512>(ctx->device, rs),
                  batched_blocks_per_sm<DT, 256>(ctx->device, rs)})
        m = std::max(m, v);
    return ctx->sms * m;
}

// Scratch regions of one batched launch over `rows` rows with `grid` blocks
// (and, with wide rows, the per-row arrays and the candidate pool).
struct BatchCarve {
    size_t order, mine, rest, words, states, cand;
    size_t wide, tile_pre, done, rstate, rcand, pool_next, pool;
};
template <int DT> static Carve batch_carve(u32 rows, int grid, bool wide, BatchCarve& bc) {
    typedef typename Key<DT>::key_t key_t;
    Carve cv;
    bc.order = cv.take(4ull * rows);
    bc.mine = cv.take(4ull * rows);
    bc.rest = cv.take(4ull * rows);
    bc.words = cv.take(256);
    bc.states = cv.take(sizeof(SelState) * (size_t)grid);
    bc.cand = cv.take((size_t)grid * 2 * BATCH_CAP * (sizeof(key_t) + 4));
    if (wide) {
        bc.wide = cv.take(4ull * rows);
        bc.tile_pre = cv.take(8ull * (rows + 1));
        bc.done = cv.take(4ull * rows);
        bc.rstate = cv.take(sizeof(SelState) * (size_t)rows);
        bc.rcand = cv.take(8ull * rows);
        bc.pool_next = cv.take(256);
        bc.pool = cv.take(((WIDE_POOL_PAIRS * sizeof(key_t) + 255) & ~(size_t)255) + WIDE_POOL_PAIRS * 4);
    }
    return cv;
}

template <int DT>
static topk_status run_batched(topk_ctx* ctx, BatchArgs b, int threads, bool by_rows, cudaStream_t st) {
    typedef typename Key<DT>::key_t key_t;
    constexpr int KW = Key<DT>::KW;
    topk_status rs = TOPK_OK;
    const int grid = batched_max_grid<DT>(ctx, rs);
    if (rs != TOPK_OK) return rs;
    const u32 cap = threads == 256 ? BatchVariant<KW, 256>::CAP
                                   : threads == 512 ? BatchVariant<KW, 512>::CAP : BatchVariant<KW, 1024>::CAP;
    b.finish_T = std::min(b.finish_T, cap);
    b.sample = std::min(b.sample, cap);
    b.key_bytes = (u32)sizeof(typename Key<DT>::raw_t);
    if (b.row_keys != nullptr) b.split = WIDE_NONE;
    if (b.split != WIDE_NONE) b.split = std::max(b.split, b.finish_T); // a wide row has more than T keys
    const bool wide = b.split != WIDE_NONE;
    BatchCarve bc;
    const Carve cv = batch_carve<DT>(b.rows, grid, wide, bc);
    rs = ensure_scratch(ctx, cv.off);
    if (rs != TOPK_OK) return rs;
    char* base = static_cast<char*>(ctx->scratch.base);
    b.order = reinterpret_cast<u32*>(base + bc.order);
    b.words = reinterpret_cast<u32*>(base + bc.words);
    b.queue = ctx->d_counter + 4;
    b.nrest = ctx->d_counter + 5;
    b.rows_done = ctx->d_counter + 6;
    b.sms = (u32)ctx->sms;
    b.mine = reinterpret_cast<u32*>(base + bc.mine);
    b.rest = by_rows ? reinterpret_cast<u32*>(base + bc.rest) : nullptr;
    b.states = reinterpret_cast<SelState*>(base + bc.states);
    b.cand = base + bc.cand;
    if (wide) {
        b.wide = reinterpret_cast<u32*>(base + bc.wide);
        b.tile_pre = reinterpret_cast<u64*>(base + bc.tile_pre);
        b.done = reinterpret_cast<u32*>(base + bc.done);
        b.rstate = reinterpret_cast<SelState*>(base + bc.rstate);
        b.rcand = reinterpret_cast<u64*>(base + bc.rcand);
        b.pool_next = reinterpret_cast<u64*>(base + bc.pool_next);
        b.pool = base + bc.pool;
        b.pool_pairs = WIDE_POOL_PAIRS;
    }
    if (threads == 256) return launch_batched<DT, 256>(ctx, b, st);
    if (threads == 512) return launch_batched<DT, 512>(ctx, b, st);
    return launch_batched<DT, 1024>(ctx, b, st);
}

// `by_rows`: rows of small k in one read (k_rows) before the general path.
static topk_status run_batched_dt(topk_ctx* ctx, topk_dtype dtype, const BatchArgs& b, int threads, bool by_rows,
                                  cudaStream_t st) {
    switch (dtype) {
    case TOPK_U32: return run_batched<DT_U32>(ctx, b, threads, by_rows, st);
    case TOPK_I32: return run_batched<DT_I32>(ctx, b, threads, by_rows, st);
    case TOPK_F32: return run_batched<DT_F32>(ctx, b, threads, by_rows, st);
    case TOPK_BF16: return run_batched<DT_BF16>(ctx, b, threads, by_rows, st);
    case TOPK_U64: return run_batched<DT_U64>(ctx, b, threads, by_rows, st);
    default: return TOPK_EINVAL;
    }
}

// Rows given by device pointer arrays (serving).  `ptrs` is one device
// block laid out as: row_keys[rows], row_out_keys[rows], row_out_idx[rows],
// row_kth_key[rows], row_kth_idx[rows] (pointers), row_n[rows], row_k[rows].
topk_status batched_by_pointers(topk_ctx* ctx, topk_dtype dtype, u32 rows, const void* ptrs, cudaStream_t st) {
    const char* p = static_cast<const char*>(ptrs);
    BatchArgs b{};
    b.rows = rows;
    b.row_keys = reinterpret_cast<const void* const*>(p);
    b.row_out_keys = reinterpret_cast<void* const*>(p + 8ull * rows);
    b.row_out_idx = reinterpret_cast<u32* const*>(p + 16ull * rows);
    b.row_kth_key = reinterpret_cast<void* const*>(p + 24ull * rows);
    b.row_kth_idx = reinterpret_cast<u32* const*>(p + 32ull * rows);
    b.row_n = reinterpret_cast<const u64*>(p + 40ull * rows);
    b.row_k = reinterpret_cast<const u32*>(p + 48ull * rows);
    b.split = WIDE_NONE; // rows are short (at most BATCH_ROW_MAX keys)
    b.seed = 0xA4093822299F31D0ull;
    b.parts = 16;
    b.z = 4.0f;
    b.flags = 0;
    b.err = ctx->d_err;
    ctx->last_kind = LAST_BATCHED;
    // the context's tuned setting for this dtype and row count, else the
    // setting the tuner picks for batches of short rows
    int threads = 256;
    b.sample = 1024;
    b.finish_T = dtype == TOPK_U64 ? Lim<64>::ELEMS : Lim<32>::ELEMS;
    auto it = ctx->tuned.find({(int)dtype, rows ? 63 - __builtin_clzll((u64)rows) : 0});
    if (it != ctx->tuned.end()) {
        threads = (int)it->second.block_threads;
        b.sample = it->second.sample_size;
        b.finish_T = it->second.finish_threshold;
    }
    return run_batched_dt(ctx, dtype, b, threads, true, st);
}

static int log2_floor(u64 v) { return v ? 63 - __builtin_clzll(v) : 0; }

template <int DT> static topk_status batched_reserve_dt(topk_ctx* ctx, uint32_t rows) {
    topk_status rs = TOPK_OK;
    const int grid = batched_max_grid<DT>(ctx, rs);
    if (rs != TOPK_OK) return rs;
    BatchCarve bc;
    return ensure_scratch(ctx, batch_carve<DT>(rows, grid, false, bc).off);
}

topk_status batched_reserve(topk_ctx* ctx, topk_dtype dtype, uint32_t rows) {
    if (cudaSetDevice(ctx->device) != cudaSuccess) return TOPK_ECUDA;
    switch (dtype) {
    case TOPK_U32: return batched_reserve_dt<DT_U32>(ctx, rows);
    case TOPK_I32: return batched_reserve_dt<DT_I32>(ctx, rows);
    case TOPK_F32: return batched_reserve_dt<DT_F32>(ctx, rows);
    case TOPK_BF16: return batched_reserve_dt<DT_BF16>(ctx, rows);
    case TOPK_U64: return batched_reserve_dt<DT_U64>(ctx, rows);
    default: return TOPK_EINVAL;
    }
}

// Arguments of one topk_select_batched call (after validation) with the
// settings of `p`; `threads` receives the block size.
static BatchArgs batch_args(topk_ctx* ctx, const void* d_keys, const uint64_t* d_row_off, const uint32_t* d_row_k,
                            uint32_t rows, topk_dtype dtype, void* d_out_keys, uint32_t* d_out_idx,
                            const uint64_t* d_out_off, void* d_kth_keys, uint32_t* d_kth_idx, const topk_params& p,
                            int& threads) {
    BatchArgs b{};
    b.keys = d_keys;
    b.row_off = d_row_off;
    b.row_k = d_row_k;
    b.rows = rows;
    b.out_keys = d_out_keys;
    b.out_idx = d_out_idx;
    b.out_off = d_out_off;
    b.kth_keys = d_kth_keys;
    b.kth_idx = d_kth_idx;
    b.seed = p.seed ? p.seed : 0xA4093822299F31D0ull;
    b.parts = p.partitions ? p.partitions : 16;
    const u32 elems = dtype == TOPK_U64 ? Lim<64>::ELEMS : Lim<32>::ELEMS;
    b.sample = p.sample_size ? std::min<u32>(std::max<u32>(p.sample_size, 64), elems) : BATCH_SAMPLE;
    b.finish_T = p.finish_threshold ? std::min<u32>(std::max<u32>(p.finish_threshold, 64), elems) : elems;
    b.z = p.delta_factor > 0.f ? p.delta_factor : 4.0f;
    b.flags = p.flags;
    b.err = ctx->d_err;
    b.split = p.split_rows ? p.split_rows : WIDE_SPLIT;
    threads = p.block_threads == 256 || p.block_threads == 512 ? (int)p.block_threads : 1024;
    return b;
}

static bool batch_ptrs_ok(topk_ctx* ctx, const void* d_keys, const uint64_t* d_row_off, const uint32_t* d_row_k,
                          uint32_t rows, topk_dtype dtype, void* d_out_keys, uint32_t* d_out_idx,
                          const uint64_t* d_out_off, void* d_kth_keys, uint32_t* d_kth_idx) {
    if (!ctx || !d_keys || !d_row_off || !d_row_k || !d_out_keys || !d_out_idx || !d_out_off || !d_kth_keys ||
        !d_kth_idx || rows == 0)
        return false;
    const int w = dtype_bytes(dtype);
    if (w == 0) return false;
    return reinterpret_cast<uintptr_t>(d_keys) % (uintptr_t)w == 0 &&
           reinterpret_cast<uintptr_t>(d_out_keys) % (uintptr_t)w == 0;
}

} // namespace topk

using namespace topk;

extern "C" topk_status topk_select_batched(topk_ctx* ctx, const void* d_keys, const uint64_t* d_row_off,
                                           const uint32_t* d_row_k, uint32_t rows, topk_dtype dtype,
                                           void* d_out_keys, uint32_t* d_out_idx, const uint64_t* d_out_off,
                                           void* d_kth_keys, uint32_t* d_kth_idx, const topk_params* params,
                                           void* stream) {
    if (!batch_ptrs_ok(ctx, d_keys, d_row_off, d_row_k, rows, dtype, d_out_keys, d_out_idx, d_out_off, d_kth_keys,
                       d_kth_idx))
        return TOPK_EINVAL;
    if (params && (params->flags & TOPK_FLAG_LARGEST)) return TOPK_EINVAL; // k smallest only
    if (cudaSetDevice(ctx->device) != cudaSuccess) return TOPK_ECUDA;
    topk_params p{};
    if (params) p = *params;
    // settings given by the caller are the general path's
    const bool general = p.block_threads || p.sample_size || p.finish_threshold || p.split_rows ||
                         (p.flags & (TOPK_FLAG_RAW_DELTA | TOPK_FLAG_TINY_CAND));
    if (p.block_threads == 0 && p.sample_size == 0 && p.finish_threshold == 0 && p.split_rows == 0) {
        auto it = ctx->tuned.find({(int)dtype, log2_floor(rows)});
        if (it != ctx->tuned.end()) {
            p.block_threads = it->second.block_threads;
            p.sample_size = it->second.sample_size;
            p.finish_threshold = it->second.finish_threshold;
            p.split_rows = it->second.split_rows;
        }
    }
    int threads = 1024;
    const BatchArgs b = batch_args(ctx, d_keys, d_row_off, d_row_k, rows, dtype, d_out_keys, d_out_idx, d_out_off,
                                   d_kth_keys, d_kth_idx, p, threads);
    ctx->last_kind = LAST_BATCHED;
    return run_batched_dt(ctx, dtype, b, threads, !general, static_cast<cudaStream_t>(stream));
}

extern "C" topk_status topk_tune_batched(topk_ctx* ctx, const void* d_keys, const uint64_t* d_row_off,
                                         const uint32_t* d_row_k, uint32_t rows, topk_dtype dtype, void* d_out_keys,
                                         uint32_t* d_out_idx, const uint64_t* d_out_off, void* d_kth_keys,
                                         uint32_t* d_kth_idx, const topk_params* base, topk_params* best,
                                         void* stream) {
    if (!batch_ptrs_ok(ctx, d_keys, d_row_off, d_row_k, rows, dtype, d_out_keys, d_out_idx, d_out_off, d_kth_keys,
                       d_kth_idx))
        return TOPK_EINVAL;
    if (base && (base->flags & TOPK_FLAG_LARGEST)) return TOPK_EINVAL;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return TOPK_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    topk_params b0{};
    if (base) b0 = *base;
    const u32 full = dtype == TOPK_U64 ? Lim<64>::ELEMS : Lim<32>::ELEMS;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return TOPK_ECUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return TOPK_ECUDA;
    }
    // (every row by the general path, whose settings these are: a call that gives
    // them runs all its rows there, and rows left by k_rows run there too)
    topk_status rs = TOPK_OK;
    topk_params choice = b0;
    float best_ms = 0.f;
    bool have = false;
    for (u32 threads : {256u, 512u, 1024u}) {
        const u32 cap = threads == 1024 ? full : threads == 512 ? full / 2 : full / 4;
        for (u32 sample : {512u, 1024u, 2048u, 4096u}) {
            for (u32 T : {cap, cap / 2}) {
                topk_params p = b0;
                p.block_threads = threads;
                p.sample_size = std::min(sample, cap);
                p.finish_threshold = T;
                int nt = 1024;
                const BatchArgs b = batch_args(ctx, d_keys, d_row_off, d_row_k, rows, dtype, d_out_keys, d_out_idx,
                                               d_out_off, d_kth_keys, d_kth_idx, p, nt);
                float ms = 0.f;
                for (int rep = 0; rep < 4 && rs == TOPK_OK; ++rep) { // one warm-up, best of three
                    if (cudaEventRecord(e0, st) != cudaSuccess) rs = TOPK_ECUDA;
                    if (rs == TOPK_OK) rs = run_batched_dt(ctx, dtype, b, nt, false, st);
                    if (rs == TOPK_OK && cudaEventRecord(e1, st) != cudaSuccess) rs = TOPK_ECUDA;
                    if (rs == TOPK_OK && cudaEventSynchronize(e1) != cudaSuccess) rs = TOPK_ECUDA;
                    float t = 0.f;
                    if (rs == TOPK_OK && cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) rs = TOPK_ECUDA;
                    if (rs == TOPK_OK && rep > 0) ms = rep == 1 ? t : std::min(ms, t);
                }
                if (rs == TOPK_OK) rs = topk_status_sync(ctx, stream);
                if (rs != TOPK_OK) break;
                if (!have || ms < best_ms) {
                    best_ms = ms;
                    choice = p;
                    have = true;
                }
            }
            if (rs != TOPK_OK) break;
        }
        if (rs != TOPK_OK) break;
    }
    // then the split length of wide rows, with the chosen block settings
    if (rs == TOPK_OK) {
        const topk_params blockwise = choice;
        for (u32 split : {1u << 13, 1u << 15, 1u << 17, WIDE_NONE}) {
            topk_params p = blockwise;
            p.split_rows = split;
            int nt = 1024;
            const BatchArgs b = batch_args(ctx, d_keys, d_row_off, d_row_k, rows, dtype, d_out_keys, d_out_idx,
                                           d_out_off, d_kth_keys, d_kth_idx, p, nt);
            float ms = 0.f;
            for (int rep = 0; rep < 4 && rs == TOPK_OK; ++rep) {
                if (cudaEventRecord(e0, st) != cudaSuccess) rs = TOPK_ECUDA;
                if (rs == TOPK_OK) rs = run_batched_dt(ctx, dtype, b, nt, false, st);
                if (rs == TOPK_OK && cudaEventRecord(e1, st) != cudaSuccess) rs = TOPK_ECUDA;
                if (rs == TOPK_OK && cudaEventSynchronize(e1) != cudaSuccess) rs = TOPK_ECUDA;
                float t = 0.f;
                if (rs == TOPK_OK && cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) rs = TOPK_ECUDA;
                if (rs == TOPK_OK && rep > 0) ms = rep == 1 ? t : std::min(ms, t);
            }
            if (rs == TOPK_OK) rs = topk_status_sync(ctx, stream);
            if (rs != TOPK_OK) break;
            if (ms < best_ms) {
                best_ms = ms;
                choice = p;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rs != TOPK_OK) return rs;
    ctx->tuned[{(int)dtype, log2_floor(rows)}] = choice;
    if (best) *best = choice;
    // leave the outputs as the chosen setting computes them
    int nt = 1024;
    const BatchArgs b = batch_args(ctx, d_keys, d_row_off, d_row_k, rows, dtype, d_out_keys, d_out_idx, d_out_off,
                                   d_kth_keys, d_kth_idx, choice, nt);
    ctx->last_kind = LAST_BATCHED;
    rs = run_batched_dt(ctx, dtype, b, nt, false, st);
    return rs == TOPK_OK ? topk_status_sync(ctx, stream) : rs;
}

extern "C" topk_status topk_tuning_save(topk_ctx* ctx, const char* path) {
    if (!ctx || !path) return TOPK_EINVAL;
    FILE* f = std::fopen(path, "w");
    if (!f) return TOPK_ECUDA;
    bool ok = std::fprintf(f, "topk-tuning 2\n") > 0;
    for (const auto& e : ctx->tuned)
        ok = ok && std::fprintf(f, "%s\t%d\t%d\t%u\t%u\t%u\t%u\n", ctx->device_name.c_str(), e.first.first,
                                e.first.second, e.second.block_threads, e.second.sample_size,
                                e.second.finish_threshold, e.second.split_rows) > 0;
    ok = (std::fclose(f) == 0) && ok;
    return ok ? TOPK_OK : TOPK_ECUDA;
}

extern "C" topk_status topk_tuning_load(topk_ctx* ctx, const char* path) {
    if (!ctx || !path) return TOPK_EINVAL;
    FILE* f = std::fopen(path, "r");
    if (!f) return TOPK_EINVAL;
    char line[512];
    topk_status rs = TOPK_OK;
    // version 1 files have no split column (split chosen automatically)
    int version = 0;
    if (!std::fgets(line, sizeof line, f) || std::sscanf(line, "topk-tuning %d", &version) != 1 ||
        (version != 1 && version != 2))
        rs = TOPK_EINVAL;
    std::map<std::pair<int, int>, topk_params> add;
    while (rs == TOPK_OK && std::fgets(line, sizeof line, f)) {
        char* tab = std::strchr(line, '\t');
        if (!tab) {
            rs = TOPK_EINVAL;
            break;
        }
        const std::string name(line, (size_t)(tab - line));
        int dt = 0, bucket = 0;
        unsigned th = 0, sample = 0, T = 0, split = 0;
        const int want = version == 2 ? 6 : 5;
        if (std::sscanf(tab + 1, "%d\t%d\t%u\t%u\t%u\t%u", &dt, &bucket, &th, &sample, &T, &split) != want ||
            dt < 0 || dt > 4 || (th != 256 && th != 512 && th != 1024)) {
            rs = TOPK_EINVAL;
            break;
        }
        if (name != ctx->device_name) continue;
        topk_params p{};
        p.block_threads = th;
        p.sample_size = sample;
        p.finish_threshold = T;
        p.split_rows = split;
        add[{dt, bucket}] = p;
    }
    std::fclose(f);
    if (rs == TOPK_OK)
        for (const auto& e : add) ctx->tuned[e.first] = e.second;
    return rs;
}
