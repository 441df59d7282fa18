// attention_tc.cu -- tree-masked attention on the 5th-generation tensor cores
// (K1, head_dim 64 or 128: one kernel template, kD).
//
// Tree decoding (Sec. 3.2) with the ancestor-bitset mask (Sec. 2.3): the
// flattened (layer, kv head, row block) x key-tile space is split evenly over
// a persistent grid, with the contractions on tcgen05.  A CTA that covers a
// whole unit writes its output; a unit split
// between CTAs leaves one (O, m, l) partial per CTA, and a second small kernel
// (k1_merge_split, one warp per query row) combines them by log-sum-exp after
// the first one has finished (in a verification step, beside the acceptance
// kernel at the end of the step: nothing in the step reads the attention
// output).  A call of its own on a small problem (one layer of a model) gives
// each unit to a cluster of CTAs instead, which combine their (O, m, l) through
// shared memory at the end: no partials in memory and no second kernel.  With
// the rotary embedding such a call also rotates the tree keys (in shared memory
// and in the cache) and the queries itself, where one CTA alone reads a unit's
// tree tiles.
//
//   S   = Q K^T   tcgen05.mma kind::f16, M = 128 query rows, N = 128 keys,
//                 K = kD = head_dim; Q (bf16) is the TMEM A operand, the K
//                 tile a 128-byte-swizzled K-major shared-memory operand; S
//                 accumulates in TMEM.
//   O  += P V     M = 128 rows, N = kD, K = 128 keys; P (bf16)
//                 is the TMEM A operand, the V tile an MN-major shared-memory
//                 operand; O accumulates in TMEM.
//
// One CTA per SM, 12 warps in three warpgroups:
//   warps 0, 3   TMA producers: 128-key K tiles (warp 0) and V tiles (warp 3),
//                kD / 64 boxes of 64 x 128 each, through separate rings: QK^T
//                releases a K slot, P V a V slot, so the next K tiles never
//                wait for a P V.
//   warp 1       TMEM allocation (512 columns) and the QK^T-issuing thread;
//                S is double-buffered, so the softmax of tile i overlaps
//                QK^T of tile i+1.
//   warp 2       the P V-issuing thread (O += P V of tile i as soon as P is
//                written; it releases the tile's stage).
//   warps 4-7    softmax, one thread per query row (TMEM lane): row max, exp2
//                with a lazily rescaled reference maximum (O and l are rescaled
//                only when the maximum grows by more than 2^8), P written back
//                to TMEM.
//   warps 8-11   staging and epilogue: the next unit's query rows go to the
//                second Q buffer while the current unit streams, and a finished
//                unit's O is read out, normalised and written (or left as a
//                partial for the merge) while the softmax goes on with the next.
// What bounds it is the K/V stream from HBM (7.2 TB/s in the long-context
// step), at a unit's ends the latency of staging and epilogue, and in short
// launches the fetch of cold instructions.  With the softmax warps doing the
// staging and the epilogue themselves (8 warps, one Q buffer) a unit boundary
// stalled the stream for about 5 us, 6.7 times per CTA in a 32-layer step.
// The softmax walks a score row in rolled 32-column steps, twice (maximum,
// then weights): a masked tile's extra code, unrolled over the whole row, ran
// once per unit from cold instruction memory and took 2 to 3 us.  Measured,
// before and now: the 32-layer step at 1063 keys and 40 nodes (rotary
// embedding, typical acceptance) 182 -> 159 us; at 16448 keys, where the stream
// takes all of the time, no change (1229 / 1227 us on one device, 1237 / 1244 on
// another); 16 single-layer calls at 1526 keys with their head 549 -> 491 us.
// TMEM columns: S0 [0,128), S1 [128,256) with P0 / P1 aliased onto their first
// halves, O [256,256+kD), Q0 [384,384+kD/2), Q1 behind it.  Both QK^T and P V take their A operand
// from TMEM, so each MMA reads only the 128 x 16 B operand from shared memory.
// Query row r of a block sits in TMEM lane 32*(r%4) + r/4 so that the rows
// are spread over the four lane quadrants (all four SM sub-partitions share
// the softmax).
#include <string.h>

#include "kernels.cuh"

namespace tv {

namespace {

constexpr int kBN = 128;           // keys per tile
// K and V ring depths.  More requests in flight make the long-context step
// slower: 1287 us with 3 + 3 stages, against 1226 with 2 + 2 or 2 + 3 and 1222
// with 3 + 2 or 4 + 2; the 32-layer step at 1063 keys takes 158-159 us with any.
constexpr int kKStages = 3;
constexpr int kVStages = 2;
constexpr int kMaxStages = kKStages > kVStages ? kKStages : kVStages;
constexpr int kAtom = 128 * 128;   // one 64-column swizzle atom of a 128-row tile (16 KB)
constexpr int kTcThreads = 384;    // 3 warpgroups: loads and MMA issue, softmax, staging and epilogue
// bytes of a K or V tile (128 keys x head_dim: kD / 64 atoms)
constexpr int tile_bytes(int d)
{
    return d / 64 * kAtom;
}
// bytes of the K and V rings
constexpr int attn_ring_bytes(int d)
{
    return (kKStages + kVStages) * tile_bytes(d);
}
// floats per partial slot: O[128][kD], m[128], l[128]
constexpr int slot_floats(int d)
{
    return 128 * d + 256;
}
// TMEM columns.  P_b (bf16 pairs) overwrites the first half of S_b once the
// softmax has read S_b into registers; Q (bf16 pairs) is the A operand of QK^T.
constexpr uint32_t kColS0 = 0, kColS1 = 128, kColP0 = 0, kColP1 = 128, kColO = 256, kColQ = 384;
constexpr float kRescaleLog2 = 8.f;  // rescale O only when the row max grows by more than 2^8
constexpr int kMaxCluster = 8;          // CTAs that may share a unit (the portable cluster size)
constexpr int kSmCols = 32;          // columns of S a softmax thread holds at a time (64: the same time, twice the code)
constexpr int kWholeUnitMaxTiles = 6;  // see attn_tc_plan

// One sequence of a (possibly batched) launch: its own KV cache (tensor maps),
// prefix length, tree, queries and outputs.  Its tiles occupy
// [tile_base, tile_base + n_units * T) of the flattened tile space.
struct TcSeq {
    long long tile_base;
    const __nv_bfloat16 *q;  // [n_layers][nstride][Hq][head_dim]
    __nv_bfloat16 *out;      // same layout
    const TreeDesc *tree;
    int L, N, rows, row_blocks, T;  // row_blocks: 128-row blocks in the unit index (1 when row_split is 2)
    int row_split;           // 2: the CTAs 2c and 2c + 1 take the two row blocks of the same units
    int nstride;             // nodes per layer in q / out (N, or the largest tree of a scheduled loop)
};

struct TcCommon {
    int n_seq, Hq, Hkv, group, layer_begin;
    long long total;
    int P;
    float scale_log2;
    float *part;
    int *status;
    // scheduled mode (sched != null): the tree and the prefix length come from
    // device memory (sched[0] = rung into rung_tree, sched[1] = L) and every
    // CTA derives the work split itself; seq[0] carries q, out and nstride
    const int32_t *sched;
    int32_t *sched_copy;  // the attention writes sched[0..1] here; the split merge's sched is this copy
    const TreeDesc *rung_tree[8];
    int n_rungs, n_layers, L_cap;
    int max_rows;  // rows the split merge's grid covers: of the largest row block, or of both (row_split)
    int d;         // head_dim: the kernels' kD (host side: picks the instantiation)
    int cluster;   // > 0: a cluster of that many CTAs shares each unit (one sequence; see attn_tc_clusters)
    // rotary embedding (null: the queries are already rotated): per sequence a
    // table of (cos, sin) at position L + depth for every pair of head elements
    const float2 *rope_tab;
};

// The launch's parameters for up to kSeqs sequences.  A launch of one sequence
// passes 0.5 KB of them rather than 5.4: every launch copies its parameters to
// the device.
template <int kSeqs>
struct TcParamsOf : TcCommon {
    CUtensorMap tmap[2 * kSeqs];  // K, V of each sequence: (head_dim, L + N, Hkv, layers), box (64, 128, 1, 1)
    TcSeq seq[kSeqs];
};
using TcParams = TcParamsOf<kMaxSeqPerLaunch>;
template <bool kBatched>
using TcKernelParams = TcParamsOf<kBatched ? kMaxSeqPerLaunch : 1>;

// A cluster launch's parameters.  rope: the kernel itself rotates the tree keys
// (in the cache too) and the queries, at L + depth(node).
struct TcClusterParams : TcParamsOf<1> {
    int rope;
    long long k_layer_stride, k_head_stride;  // of the K cache, elements
    __nv_bfloat16 *k;
    double inv_freq[kRopeMaxHalf];
};
template <bool kBatched, bool kCluster>
struct TcKernelArg {
    using type = TcKernelParams<kBatched>;
};
template <>
struct TcKernelArg<false, true> {
    using type = TcClusterParams;
};

// Two row blocks per kv head (grouped queries, 129 to 256 rows) and more than a
// wave of tiles: neighbouring CTAs walk the same key tiles side by side, one
// row block each, so that the second reading of a tile comes from L2.  As units
// of their own the two blocks are read a whole unit apart: at 32 layers, 32 q /
// 8 kv heads, 64 nodes at 8192 keys that streams K and V from HBM twice, and
// the step took 485 us, now 427.
__host__ __device__ inline bool split_rows(int row_blocks, long long total, int n_ctas)
{
    return row_blocks == 2 && total >= n_ctas && n_ctas >= 2;
}

// Scheduled mode: the sequence of this step from the device state.  An
// out-of-range rung or a prefix that does not fit the cache gives no work
// (the acceptance kernel reports it).
__device__ void sched_plan(const TcCommon &p, const TcSeq &first, TcSeq *sq, long long *total)
{
    *sq = first;
    sq->tile_base = 0;
    const int rung = p.sched[0], L = p.sched[1];
    const bool ok = rung >= 0 && rung < p.n_rungs && L >= 0;
    const TreeDesc *tr = p.rung_tree[ok ? rung : 0];
    const int N = tr->n;
    sq->tree = tr;
    sq->L = ok ? L : 0;
    sq->N = N;
    sq->rows = N * p.group;
    sq->row_blocks = (sq->rows + 127) / 128;
    sq->T = (sq->L + N + kBN - 1) / kBN;
    sq->row_split = split_rows(sq->row_blocks, (long long)p.n_layers * p.Hkv * sq->row_blocks * sq->T, p.P) ? 2 : 1;
    sq->row_blocks /= sq->row_split;
    *total = (ok && L + N <= p.L_cap) ? (long long)p.n_layers * p.Hkv * sq->row_blocks * sq->T : 0;
}

// Sequence holding flattened tile t, searching forward from `b` (tiles are
// visited in increasing order by every role).  kBatched = false: sequence 0.
template <bool kBatched>
__device__ __forceinline__ int seq_at(const TcKernelParams<kBatched> &p, long long t, int b)
{
    if constexpr (!kBatched) {
        return 0;
    } else {
        while (b + 1 < p.n_seq && t >= p.seq[b + 1].tile_base)
            ++b;
        return b;
    }
}

// Ranges the tile space is split over: one per CTA, or per pair of CTAs with
// the same tiles and a row block each (row_split = 2).  The host plans at most one CTA per
// tile; scheduled mode plans on the device with a grid of one CTA per SM, and
// a step with fewer tiles than that splits them over its first `total` CTAs
// only (the others get nothing), so that no CTA range inside the split is
// empty: the split merge combines the partials of consecutive CTAs.
__device__ __forceinline__ int tc_split_ctas(const TcCommon &p, long long total, int row_split)
{
    const int n = p.P / row_split;
    return (p.sched && total < n) ? (int)(total > 0 ? total : 1) : n;
}

// First flattened tile of CTA c's range (the ranges split the tile space
// evenly).  The quotients take 32-bit divisions whenever the operands fit.
__device__ __forceinline__ long long tc_seg_begin(long long total, int P, int c)
{
    const unsigned long long x = (unsigned long long)c * (unsigned long long)total;
    return x <= 0xffffffffull ? (long long)((uint32_t)x / (uint32_t)P) : (long long)(x / (unsigned long long)P);
}

// The CTA whose range holds tile t.
__device__ __forceinline__ int tc_cta_of(long long total, int P, long long t)
{
    if (total <= 0)
        return 0;
    const unsigned long long x = (unsigned long long)(t + 1) * (unsigned long long)P - 1ull;
    return x <= 0xffffffffull && (unsigned long long)total <= 0xffffffffull ? (int)((uint32_t)x / (uint32_t)total)
                                                                           : (int)(x / (unsigned long long)total);
}

// MN-major (N contiguous) 128-byte-swizzled operand: lbo = stride between
// 64-element column atoms, sbo = stride between groups of 8 K rows.
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return smem_desc_sw128(addr, lbo, sbo);
}

}  // namespace

// Allowed-key bits of 32 consecutive keys whose first has tree index tj0
// (key position minus the prefix length): bit c is set when key tj0 + c is a
// prefix key (tree index < 0) or an ancestor of the row's node (bit tj0 + c of
// its ancestor set anc, whose bits lie below the tree's node count).
__device__ __forceinline__ uint32_t tile_allow(int tj0, uint64_t anc)
{
    if (tj0 <= -32)
        return 0xffffffffu;
    if (tj0 >= 64)
        return 0u;
    if (tj0 >= 0)
        return (uint32_t)(anc >> tj0);
    const int pre = -tj0;  // 1 .. 31 prefix keys, then the tree from bit pre
    return ((1u << pre) - 1u) | (uint32_t)(anc << pre);
}

// Position of a CTA's next segment: the run of key tiles of one unit that the
// CTA covers.
struct SegPos {
    int b, u;   // sequence, unit within it
    int j0, n;  // first key tile of the unit, and how many
};

template <bool kBatched>
__device__ __forceinline__ SegPos seg_at(const TcKernelParams<kBatched> &p, const TcSeq *seqs, long long t, long long t1, int b)
{
    SegPos g;
    g.b = seq_at<kBatched>(p, t, b);
    const TcSeq &sq = seqs[g.b];
    const long long tl = t - sq.tile_base;
    g.u = (unsigned long long)tl <= 0xffffffffull ? (int)((uint32_t)tl / (uint32_t)sq.T) : (int)(tl / sq.T);
    g.j0 = (int)(tl - (long long)g.u * sq.T);
    const long long left = t1 - t;
    g.n = left < sq.T - g.j0 ? (int)left : sq.T - g.j0;
    return g;
}

// What the softmax warps need of a segment, written by the staging warps with
// the segment's queries (double-buffered like them).
struct SegInfo {
    int n, key0, L;            // key tiles, first key position, prefix length
    uint64_t anc[128];         // ancestor set of each row's node
    float m[128], l[128];      // written back by the softmax: reference maximum (log2 units) and sum of each row
};

// kCluster: the p.cluster CTAs of a cluster share one unit's key tiles, leave
// their (O, m, l) in shared memory and combine them there (log-sum-exp, in rank
// order), every CTA a share of the rows: no partials in global memory and no
// second kernel.  For problems small enough that all their clusters run at
// once (attn_tc_clusters).  Latency bounds these calls: of the 12 us of one
// layer of 32 heads at 1526 keys 3.5 go to the first keys and queries, 1.05 to
// each of three tiles, 3 to the combination and its two cluster barriers
// (the first is arrived at before TMEM is freed: 0.5 us less).  So everything that
// needs none of the caller's memory (the first unit's indices, the rotary table,
// the fetch of the roles' instructions) runs before the wait for the previous
// kernel: 0.4 to 0.7 us less per call.  With the rotary kernel
// before it and its table in memory a layer took 17.2 us in a 16-layer pass,
// rotating here 14.5.
template <int kD, bool kBatched, bool kCluster>
__global__ void __launch_bounds__(kTcThreads, 1) k1_tree_attention_tc(const __grid_constant__ typename TcKernelArg<kBatched, kCluster>::type p)
{
    static_assert(kD == 64 || kD == 128, "head_dim 64 or 128");
    constexpr int kTile = tile_bytes(kD);
    constexpr int kSlot = slot_floats(kD);
    constexpr int kClusterLd = kD + 4;  // row stride of O in shared memory (floats): conflict-free row writes
    static_assert(!(kCluster && kBatched), "clusters: one sequence");
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t k_full[kMaxStages], k_empty[kMaxStages], v_full[kMaxStages], v_empty[kMaxStages];
    __shared__ __align__(8) uint64_t s_full[2], p_full[2], pv_done[2];
    __shared__ __align__(8) uint64_t q_full[2], ml_full[2], o_free[2], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ TcSeq s_seq;
    __shared__ long long s_total;
    __shared__ SegInfo s_info[2];
    // kCluster with rope, for the unit's first and second tile that hold tree keys:
    // the K tile has landed; its tree keys are rotated.  Used once each.
    __shared__ __align__(8) uint64_t kt_full[2], kr_full[2];

    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sK = smem;                                // K ring: kKStages tiles
    uint8_t *sV = smem + (size_t)kKStages * kTile;     // V ring: kVStages tiles

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&k_full[s], 1);
            mbar_init(&k_empty[s], 1);
            mbar_init(&v_full[s], 1);
            mbar_init(&v_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&s_full[b], 1);
            mbar_init(&p_full[b], 4);
            mbar_init(&pv_done[b], 1);
            mbar_init(&q_full[b], 4);
            mbar_init(&ml_full[b], 4);
            mbar_init(&o_free[b], 4);
        }
        mbar_init(&drain_bar, 2);  // one commit from each MMA issuer
        if constexpr (kCluster) {
            for (int b = 0; b < 2; ++b) {
                mbar_init(&kt_full[b], 1);
                mbar_init(&kr_full[b], 4);
            }
        }
        abort_flag = 0;
        fence_mbar_init();
        for (int b = 0; b < (kBatched ? p.n_seq : 1); ++b) {
            prefetch_tmap(&p.tmap[2 * b]);
            prefetch_tmap(&p.tmap[2 * b + 1]);
        }
    }
    if (warp == 1) {
        tmem_alloc(&tmem_slot, 512);
        tmem_relinquish();
    }
    // (cos, sin) of every pair at L + depth, and the nodes' depths: they depend on
    // the topology and L only
    float2 *s_rope = reinterpret_cast<float2 *>(smem + attn_ring_bytes(kD));
    int8_t *s_dep = reinterpret_cast<int8_t *>(s_rope + kMaxNodes * (kD / 2));
    if constexpr (kCluster) {
        if (p.rope) {
            const TreeDesc *tree = p.seq[0].tree;
            if (threadIdx.x < kMaxNodes)
                s_dep[threadIdx.x] = tree->depth[threadIdx.x];
            const int n = (min(tree->max_depth, kMaxNodes - 1) + 1) * (kD / 2);
            for (int i = threadIdx.x; i < n; i += kTcThreads) {
                constexpr double kTwoPi = 6.283185307179586476925286766559;
                const double a = (double)(p.seq[0].L + i / (kD / 2)) * p.inv_freq[i % (kD / 2)];
                const double red = a - kTwoPi * rint(a * (1.0 / kTwoPi));
                float2 cn;
                sincosf((float)red, &cn.y, &cn.x);
                s_rope[i] = cn;
            }
        }
    }
    // Launched as a programmatic dependent, the kernel waits for the stream's
    // previous work (the previous step's compaction writes the cache) before it
    // reads or writes any of the caller's memory: each role just before its first
    // such access (wait_previous), so that its set-up, its first unit's indices and
    // the fetch of its instructions overlap what runs before.  From then on the
    // step's LM head may be launched: it fills the SMs that attention CTAs leave
    // free or release.
    auto wait_previous = [] {
        pdl_wait();
        pdl_trigger();
    };
    const TcSeq *seqs = p.seq;
    long long total = p.total;
    if (p.sched) {
        wait_previous();  // the state is an earlier kernel's
        if (threadIdx.x == 0)
            sched_plan(p, p.seq[0], &s_seq, &s_total);
        if (threadIdx.x == 32 && c == 0) {
            p.sched_copy[0] = p.sched[0];
            p.sched_copy[1] = p.sched[1];
        }
        __syncthreads();
        seqs = &s_seq;
        total = s_total;
    }
    long long t0, t1;
    if constexpr (kCluster) {
        // every rank has a tile: the host takes no more CTAs than tiles
        const int T = seqs[0].T, rank = c % p.cluster;
        const long long first = (long long)(c / p.cluster) * T;
        t0 = first + (long long)T * rank / p.cluster;
        t1 = first + (long long)T * (rank + 1) / p.cluster;
    } else {
        const int rs = kBatched ? 1 : seqs[0].row_split;
        const int P = tc_split_ctas(p, total, rs), r = c / rs;
        t0 = r < P ? tc_seg_begin(total, P, r) : total;
        t1 = r < P ? tc_seg_begin(total, P, r + 1) : total;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp < 4) {
        if (lane != 0) {
            // one thread of each warp of this warpgroup works
            wait_previous();
        } else if (warp == 0 || warp == 3) {
            // -------------------------------------------------------- TMA producers
            // warp 0 streams the K tiles, warp 3 the V tiles, each through its own
            // ring: QK^T releases a K slot, P V a V slot.
            const bool is_v = (warp == 3);
            uint64_t *full = is_v ? v_full : k_full;
            uint64_t *empty = is_v ? v_empty : k_empty;
            const int S = is_v ? kVStages : kKStages;
            uint8_t *ring = is_v ? sV : sK;
            long long issued = 0;
            int s = 0, sb = 0, tree_issued = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (long long t = t0; ok && t < t1;) {
                const SegPos g = seg_at<kBatched>(p, seqs, t, t1, sb);
                sb = g.b;
                const TcSeq &sq = seqs[sb];
                const int head = (g.u / sq.row_blocks) % p.Hkv;
                const int layer = p.layer_begin + g.u / (sq.row_blocks * p.Hkv);
                const CUtensorMap *m = &p.tmap[2 * sb + (is_v ? 1 : 0)];
                if (t == t0)
                    wait_previous();
                for (int j = 0; j < g.n; ++j) {
                    if (!mbar_wait_bounded(&empty[s], ph ^ 1u, &abort_flag, p.status)) {
                        ok = false;
                        break;
                    }
                    uint8_t *dst = ring + (size_t)s * kTile;
                    uint64_t *landed = &full[s];
                    if constexpr (kCluster) {
                        // a K tile with tree keys to rotate lands on a barrier of its own, which
                        // the rotating warps wait for; QK^T then waits for them
                        const int tree_tile = g.j0 + j - p.seq[0].L / kBN;
                        if (p.rope && !is_v && tree_tile >= 0) {
                            mbar_arrive(&full[s]);
                            landed = &kt_full[tree_tile & 1];
                            tree_issued |= 1 << (tree_tile & 1);
                        }
                    }
                    mbar_arrive_expect_tx(landed, kTile);
#pragma unroll
                    for (int a = 0; a < kD / 64; ++a)
                        tma_load_4d(dst + a * kAtom, m, landed, 64 * a, (g.j0 + j) * kBN, head, layer);
                    ++issued;
                    if (++s == S) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                t += g.n;
            }
            if (!ok) {
                for (long long it = (issued > S ? issued - S : 0); it < issued; ++it)
                    mbar_wait_drain(&full[it % S], (uint32_t)(it / S) & 1u);
                for (int b = 0; b < 2; ++b)
                    if (kCluster && ((tree_issued >> b) & 1))
                        mbar_wait_drain(&kt_full[b], 0);
            }
        } else if (warp == 1) {
            // -------------------------------------------------------- QK^T issuer
            wait_previous();
            const uint32_t idesc_s = idesc_bf16_f32(128, kBN);
            long long it = 0;
            int s = 0, sb = 0, sg = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (long long t = t0; ok && t < t1; ++sg) {
                const SegPos g = seg_at<kBatched>(p, seqs, t, t1, sb);
                sb = g.b;
                const uint32_t q_col = tmem + kColQ + (sg & 1) * (kD / 2);
                for (int j = 0; j < g.n; ++j, ++it) {
                    const int b = (int)(it & 1);
                    // K landed; P V(it - 2) has read P_b, which shares S_b's columns and was
                    // written after the softmax had read S_b; at a segment's first tile, its Q
                    // is staged
                    if (!mbar_wait_bounded(&k_full[s], ph, &abort_flag, p.status) ||
                        (it >= 2 &&
                         !mbar_wait_bounded(&pv_done[b], (uint32_t)((it - 2) >> 1) & 1u, &abort_flag, p.status)) ||
                        (j == 0 && !mbar_wait_bounded(&q_full[sg & 1], (uint32_t)(sg >> 1) & 1u, &abort_flag, p.status))) {
                        ok = false;
                        break;
                    }
                    if constexpr (kCluster) {
                        const int tree_tile = g.j0 + j - p.seq[0].L / kBN;  // 0 or 1: the tile holds tree keys
                        if (p.rope && tree_tile >= 0 &&
                            !mbar_wait_bounded(&kr_full[tree_tile & 1], 0, &abort_flag, p.status)) {
                            ok = false;
                            break;
                        }
                    }
                    tc_fence_after();
                    const uint32_t k_base = smem_u32(sK + (size_t)s * kTile);
                    const uint32_t s_col = tmem + (b ? kColS1 : kColS0);
#pragma unroll
                    for (int kk = 0; kk < kD / 16; ++kk) {
                        const uint32_t off = (uint32_t)(kk >> 2) * kAtom + (uint32_t)(kk & 3) * 32;
                        const uint64_t bdesc = smem_desc_sw128(k_base + off, 0, 1024);
                        tc_mma_f16_ts(s_col, q_col + kk * 8, bdesc, idesc_s, kk > 0 ? 1u : 0u);
                    }
                    tc_commit(&s_full[b]);
                    tc_commit(&k_empty[s]);
                    if (++s == kKStages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                t += g.n;
            }
            // arrives when every MMA issued above has retired (waited for before TMEM is released)
            tc_commit(&drain_bar);
        } else {
            // -------------------------------------------------------- P V issuer (warp 2)
            // A second issuing thread: each tcgen05.mma holds its issuer for about
            // 100 cycles at these shapes, so P V(i) issued here runs alongside
            // QK^T(i + 1) instead of queueing behind it, and the stage is released
            // that much sooner.
            wait_previous();
            const uint32_t idesc_pv = idesc_bf16_f32(128, kD, false, true);
            long long it = 0;
            int s = 0, sb = 0, sg = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (long long t = t0; ok && t < t1; ++sg) {
                const SegPos g = seg_at<kBatched>(p, seqs, t, t1, sb);
                sb = g.b;
                for (int j = 0; j < g.n; ++j, ++it) {
                    const int b = (int)(it & 1);
                    // P written; at a segment's first tile, the previous segment's O has been read
                    if (!mbar_wait_bounded(&p_full[b], (uint32_t)(it >> 1) & 1u, &abort_flag, p.status) ||
                        (j == 0 && sg > 0 &&
                         !mbar_wait_bounded(&o_free[(sg - 1) & 1], (uint32_t)((sg - 1) >> 1) & 1u, &abort_flag,
                                            p.status)) ||
                        !mbar_wait_bounded(&v_full[s], ph, &abort_flag, p.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t v_base = smem_u32(sV + (size_t)s * kTile);
                    const uint32_t p_col = tmem + (b ? kColP1 : kColP0);
#pragma unroll
                    for (int ks = 0; ks < kBN / 16; ++ks) {
                        const uint64_t bdesc = smem_desc_sw128_mn(v_base + ks * 2048, kAtom, 1024);
                        tc_mma_f16_ts(tmem + kColO, p_col + ks * 8, bdesc, idesc_pv, (j == 0 && ks == 0) ? 0u : 1u);
                    }
                    tc_commit(&v_empty[s]);
                    tc_commit(&pv_done[b]);
                    if (++s == kVStages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                t += g.n;
            }
            tc_commit(&drain_bar);
        }
    } else if (warp < 8) {
        // ------------------------------------------------------------ softmax (warps 4-7)
        const int q4 = warp & 3;  // TMEM lane quadrant of this warp
        const uint32_t lane_addr = tmem + ((uint32_t)(32 * q4) << 16);
        const int rloc = 4 * lane + q4;  // query row of this thread within the block
        wait_previous();
        long long it = 0;
        bool aborted = false;
        int sg = 0;
        for (long long t = t0; t < t1 && !aborted; ++sg) {
            SegInfo &si = s_info[sg & 1];
            if (!mbar_wait_bounded(&q_full[sg & 1], (uint32_t)(sg >> 1) & 1u, &abort_flag, p.status))
                break;
            const int n = si.n, L = si.L;
            int key0 = si.key0;
            const uint64_t anc = si.anc[rloc];
            t += n;
            float m_ref = -INFINITY, l = 0.f;
            for (int j = 0; j < n; ++j, ++it, key0 += kBN) {
                const int b = (int)(it & 1);
                if (!mbar_wait_bounded(&s_full[b], (uint32_t)(it >> 1) & 1u, &abort_flag, p.status)) {
                    aborted = true;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = lane_addr + (b ? kColS1 : kColS0);
                const bool masked = key0 + kBN > L;

                // pass 1: the row maximum over the allowed keys, kSmCols columns at a time
                float mx = -INFINITY;
#pragma unroll 1
                for (int c0 = 0; c0 < kBN; c0 += kSmCols) {
                    uint32_t r[kSmCols];
#pragma unroll
                    for (int x = 0; x < kSmCols; x += 32)
                        tmem_ld_32x32b_x32(sa + c0 + x, r + x);
                    tmem_ld_wait();
                    if (masked) {
                        // allowed: prefix keys (tree index < 0) and the ancestors in the tree, 32
                        // columns per word; the others' scores become -inf in place
#pragma unroll
                        for (int x0 = 0; x0 < kSmCols; x0 += 32) {
                            const uint32_t allow = tile_allow(key0 + c0 + x0 - L, anc);
                            if (__all_sync(0xffffffffu, allow == 0xffffffffu))
                                continue;
#pragma unroll
                            for (int x = 0; x < 32; ++x)
                                r[x0 + x] = (allow >> x) & 1u ? r[x0 + x] : 0xff800000u;
                            tmem_st_32x32b_x32(sa + c0 + x0, r + x0);
                            tmem_st_wait();
                        }
                    }
#pragma unroll
                    for (int x = 0; x < kSmCols; ++x)
                        mx = fmaxf(mx, __uint_as_float(r[x]));
                }
                mx *= p.scale_log2;  // row max in log2 units (scale > 0)

                // lazily rescaled reference maximum
                float alpha = 1.f;
                bool rescale = false;
                if (j == 0) {
                    m_ref = mx;
                } else if (mx > m_ref + kRescaleLog2) {
                    alpha = (m_ref == -INFINITY) ? 0.f : ex2_approx(m_ref - mx);
                    m_ref = mx;
                    rescale = true;
                }
                if (__any_sync(0xffffffffu, rescale)) {
                    // O holds the previous tiles' P V: wait for the last one, then scale in place
                    const long long jp = it - 1;
                    if (!mbar_wait_bounded(&pv_done[jp & 1], (uint32_t)(jp >> 1) & 1u, &abort_flag, p.status)) {
                        aborted = true;
                        break;
                    }
                    tc_fence_after();
                    l *= alpha;
#pragma unroll 1
                    for (int c0 = 0; c0 < kD; c0 += 32) {
                        uint32_t o[32];
                        tmem_ld_32x32b_x32(lane_addr + kColO + c0, o);
                        tmem_ld_wait();
#pragma unroll
                        for (int x = 0; x < 32; ++x)
                            o[x] = __float_as_uint(__uint_as_float(o[x]) * alpha);
                        tmem_st_32x32b_x32(lane_addr + kColO + c0, o);
                    }
                    tmem_st_wait();
                }

                // pass 2: P = 2^(s * scale - m_ref) as bf16 pairs into TMEM (masked entries are
                // -inf and give 0), row sum into l.  P_b's columns are S_b's: QK^T wrote S_b
                // after O += P V of tile it - 2 had read P_b.
                const float mu = (m_ref == -INFINITY) ? 0.f : m_ref;
                const uint32_t pa = lane_addr + (b ? kColP1 : kColP0);
                float rs = 0.f;
#pragma unroll 1
                for (int c0 = 0; c0 < kBN; c0 += kSmCols) {
                    uint32_t r[kSmCols];
#pragma unroll
                    for (int x = 0; x < kSmCols; x += 32)
                        tmem_ld_32x32b_x32(sa + c0 + x, r + x);
                    tmem_ld_wait();
#pragma unroll
                    for (int x0 = 0; x0 < kSmCols; x0 += 32) {
                        uint32_t pk[16];
#pragma unroll
                        for (int x = 0; x < 16; ++x) {
                            const float p0 = ex2_approx(fmaf(__uint_as_float(r[x0 + 2 * x]), p.scale_log2, -mu));
                            const float p1 = ex2_approx(fmaf(__uint_as_float(r[x0 + 2 * x + 1]), p.scale_log2, -mu));
                            rs += p0 + p1;
                            pk[x] = pack_bf16x2(p0, p1);
                        }
                        tmem_st_32x32b_x16(pa + (c0 + x0) / 2, pk);
                    }
                }
                l += rs;
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&p_full[b]);
            }
            if (aborted)
                break;
            // the segment's (m, l) for its epilogue; the buffer was read by segment sg - 2's
            if (sg >= 2 && !mbar_wait_bounded(&o_free[sg & 1], (uint32_t)((sg >> 1) - 1) & 1u, &abort_flag, p.status))
                break;
            si.m[rloc] = m_ref;
            si.l[rloc] = l;
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&ml_full[sg & 1]);
        }
    } else {
        // ------------------------------------------------------------ staging and epilogue (warps 8-11)
        // One segment ahead of the softmax: the next segment's query rows go to
        // the other Q buffer while the current one streams, and a finished
        // segment's O is read out and written while the softmax goes on with the
        // next, so a unit boundary does not stall the K/V stream.
        const int q4 = warp & 3;
        const uint32_t lane_addr = tmem + ((uint32_t)(32 * q4) << 16);
        const int rloc = 4 * lane + q4;

        struct Seg {
            int n, j0, T;
            bool first;  // the CTA's first segment
            bool valid;  // this thread's row exists
            int b, dep, L;
            uint64_t anc;
            const __nv_bfloat16 *q;  // this thread's query and output rows
            __nv_bfloat16 *out;
        };
        int sb = 0;
        auto describe = [&](long long t) {
            const SegPos sp = seg_at<kBatched>(p, seqs, t, t1, sb);
            sb = sp.b;
            const TcSeq &sq = seqs[sb];
            Seg g;
            g.n = sp.n;
            g.j0 = sp.j0;
            g.T = sq.T;
            g.first = t == t0;
            g.b = sb;
            g.L = sq.L;
            const int rb = sp.u % sq.row_blocks + (kBatched || kCluster ? 0 : c % sq.row_split);
            const int head = (sp.u / sq.row_blocks) % p.Hkv;
            const int layer_rel = sp.u / (sq.row_blocks * p.Hkv);
            g.valid = rloc < min(128, sq.rows - rb * 128);
            const int grow = rb * 128 + rloc;
            const int node = g.valid ? grow / p.group : 0;
            const int qh = head * p.group + grow % p.group;
            // the row's query / output rows and tree entries
            if (g.valid)
                g.valid = in_bounds(layer_rel < p.n_layers && node < sq.N && node < sq.nstride && node < kMaxNodes &&
                                        qh < p.Hq,
                                    p.status);
            g.anc = g.valid ? sq.tree->anc[node] : 0ull;
            g.dep = g.valid ? sq.tree->depth[node] : 0;
            const size_t row = (((size_t)layer_rel * sq.nstride + node) * p.Hq + qh) * kD;
            g.q = sq.q + row;
            g.out = sq.out + row;
            return g;
        };
        // The segment's info and its Q rows, each row in its thread's TMEM lane as
        // kD / 2 columns of bf16 pairs (the A operand of QK^T); zeros for padding rows
        auto stage = [&](const Seg &g, int sg) {
            SegInfo &si = s_info[sg & 1];
            const uint32_t col = lane_addr + kColQ + (sg & 1) * (kD / 2);
            const uint4 *src = reinterpret_cast<const uint4 *>(g.q);
            bool rotate = p.rope_tab != nullptr;
            const float2 *tab = p.rope_tab + (size_t)g.b * kRopeTableEntries + (size_t)g.dep * kRopeMaxHalf;
            if constexpr (kCluster) {
                if (p.rope) {
                    rotate = true;
                    tab = s_rope + g.dep * (kD / 2);
                }
            }
            if (!rotate) {
                // the whole row (2 kD bytes) in flight at once, then kD / 32 TMEM stores
                uint4 qv[kD / 8];
#pragma unroll
                for (int i = 0; i < kD / 8; ++i)
                    qv[i] = g.valid ? src[i] : make_uint4(0, 0, 0, 0);
#pragma unroll
                for (int qc = 0; qc < kD / 32; ++qc) {
                    uint32_t w[16];
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
                        const uint4 v = qv[qc * 4 + ch];
                        w[4 * ch] = v.x;
                        w[4 * ch + 1] = v.y;
                        w[4 * ch + 2] = v.z;
                        w[4 * ch + 3] = v.w;
                    }
                    tmem_st_32x32b_x16(col + qc * 16, w);
                }
            } else {
                // pre-rotary query: element i pairs with i + kD / 2, rotated at position
                // L + depth(node) with the sequence's (cos, sin) table
                constexpr int kHalf = kD / 64;  // 32-element chunks per half row
#pragma unroll 1
                for (int qc = 0; qc < kHalf; ++qc) {
                    uint32_t wl[16], wh[16];
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
                        const uint4 lo = g.valid ? src[qc * 4 + ch] : make_uint4(0, 0, 0, 0);
                        const uint4 hi = g.valid ? src[(qc + kHalf) * 4 + ch] : make_uint4(0, 0, 0, 0);
                        const uint32_t lw[4] = {lo.x, lo.y, lo.z, lo.w}, hw[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int i0 = 32 * qc + 8 * ch + 2 * e;
                            const float2 c0 = tab[i0], c1 = tab[i0 + 1];
                            const float a0 = __uint_as_float(lw[e] << 16), a1 = __uint_as_float(lw[e] & 0xffff0000u);
                            const float b0 = __uint_as_float(hw[e] << 16), b1 = __uint_as_float(hw[e] & 0xffff0000u);
                            wl[4 * ch + e] = pack_bf16x2(a0 * c0.x - b0 * c0.y, a1 * c1.x - b1 * c1.y);
                            wh[4 * ch + e] = pack_bf16x2(b0 * c0.x + a0 * c0.y, b1 * c1.x + a1 * c1.y);
                        }
                    }
                    tmem_st_32x32b_x16(col + qc * 16, wl);
                    tmem_st_32x32b_x16(col + (qc + kHalf) * 16, wh);
                }
            }
            si.anc[rloc] = g.anc;
            // every warp writes the same words, so that each softmax warp's wait covers them
            if (lane == 0) {
                si.n = g.n;
                si.key0 = g.j0 * kBN;
                si.L = g.L;
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&q_full[sg & 1]);
        };
        // Rotates the tree keys of the CTA's it-th tile (key tile j of its unit) in
        // shared memory and writes them to the cache: no other CTA reads that tile
        // (the launch has one row block per kv head).
        auto rotate_keys = [&](int it, int j, int head, int layer) {
            if constexpr (kCluster) {
                if (!mbar_wait_bounded(&kt_full[(j - p.seq[0].L / kBN) & 1], 0, &abort_flag, p.status))
                    return false;
                uint8_t *tile = sK + (size_t)(it % kKStages) * kTile;
                const int L = p.seq[0].L, first = max(L, j * kBN), last = min(L + p.seq[0].N, (j + 1) * kBN);
                constexpr int kCh = kD / 16;  // 8-pair pieces of a row
                __nv_bfloat16 *kc = p.k + (size_t)layer * p.k_layer_stride + (size_t)head * p.k_head_stride;
                for (int x = (int)threadIdx.x - 256; x < (last - first) * kCh; x += 128) {
                    const int slot = first + x / kCh, ch = x % kCh, row = slot - j * kBN;
                    // elements [8 ch, 8 ch + 8) and their partners kD / 2 on
                    const int hi_ch = ch + kD / 16;
                    uint4 *lo = reinterpret_cast<uint4 *>(tile + (ch >> 3) * kAtom + row * 128 + (((ch & 7) ^ (row & 7)) << 4));
                    uint4 *hi = reinterpret_cast<uint4 *>(tile + (hi_ch >> 3) * kAtom + row * 128 +
                                                          (((hi_ch & 7) ^ (row & 7)) << 4));
                    uint4 a = *lo, b = *hi;
                    __nv_bfloat16 *xa = reinterpret_cast<__nv_bfloat16 *>(&a), *xb = reinterpret_cast<__nv_bfloat16 *>(&b);
                    const float2 *cs = s_rope + s_dep[slot - L] * (kD / 2) + 8 * ch;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float2 c0 = cs[e];
                        const float x1 = __bfloat162float(xa[e]), x2 = __bfloat162float(xb[e]);
                        xa[e] = __float2bfloat16_rn(x1 * c0.x - x2 * c0.y);
                        xb[e] = __float2bfloat16_rn(x2 * c0.x + x1 * c0.y);
                    }
                    *lo = a;
                    *hi = b;
                    if (in_bounds((long long)(slot + 1) * kD <= p.k_head_stride && slot - L < kMaxNodes, p.status)) {
                        uint4 *dst = reinterpret_cast<uint4 *>(kc + (size_t)slot * kD);
                        dst[ch] = a;
                        dst[hi_ch] = b;
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&kr_full[(j - L / kBN) & 1]);
            }
            return true;
        };
        long long t = t0;
        if (t < t1) {
            Seg cur = describe(t);
            wait_previous();
            stage(cur, 0);
            if constexpr (kCluster) {
                if (p.rope) {
                    const int u = c / p.cluster, head = u % p.Hkv, layer = p.layer_begin + u / p.Hkv;
                    const int from = max(0, cur.L / kBN - cur.j0);  // the first tile that holds a tree key
                    for (int it = from; it < cur.n; ++it)
                        if (!rotate_keys(it, cur.j0 + it, head, layer))
                            break;
                }
            }
            t += cur.n;
            Seg nxt{};
            bool has_next = t < t1;
            if (has_next) {
                nxt = describe(t);
                stage(nxt, 1);
                t += nxt.n;
            }
            long long it = 0;
            for (int sg = 0;; ++sg) {
                it += cur.n;
                // the segment after the next: its query rows are asked for in L2 now, staged below
                Seg fut{};
                const bool has_fut = t < t1;
                if (has_fut) {
                    fut = describe(t);
                    t += fut.n;
                    if (fut.valid) {
#pragma unroll
                        for (int off = 0; off < 2 * kD; off += 128)
                            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char *>(fut.q) + off));
                    }
                }
                const long long last = it - 1;
                if (!mbar_wait_bounded(&ml_full[sg & 1], (uint32_t)(sg >> 1) & 1u, &abort_flag, p.status))
                    break;
                const float m_ref = s_info[sg & 1].m[rloc], l = s_info[sg & 1].l[rloc];
                if (!mbar_wait_bounded(&pv_done[last & 1], (uint32_t)(last >> 1) & 1u, &abort_flag, p.status))
                    break;
                tc_fence_after();
                const bool whole = cur.n == cur.T;
                const bool write = cur.valid && (whole || in_bounds(c < p.P && rloc < 128, p.status));
                const float inv = 1.f / l;
                uint4 *dst = reinterpret_cast<uint4 *>(cur.out);
                // a partial (O, m, l) goes to the CTA's slot; k1_merge_split finishes the unit
                float *slot = p.part + ((size_t)c * 2 + (cur.first ? 0 : 1)) * kSlot;
                float4 *pdst = reinterpret_cast<float4 *>(slot + rloc * kD);
                if constexpr (kCluster)  // the rings are drained: every tile has been consumed (a cluster's part)
                    pdst = reinterpret_cast<float4 *>(smem + (size_t)rloc * kClusterLd * 4);
#pragma unroll
                for (int c0 = 0; c0 < kD; c0 += 64) {
                    uint32_t r[64];
                    tmem_ld_32x32b_x32(lane_addr + kColO + c0, r);
                    tmem_ld_32x32b_x32(lane_addr + kColO + c0 + 32, r + 32);
                    tmem_ld_wait();
                    if (c0 + 64 == kD) {
                        // the whole row is read: the next segment's P V may overwrite O
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0)
                            mbar_arrive(&o_free[sg & 1]);
                    }
                    if (!write)
                        continue;
                    if (whole) {
#pragma unroll
                        for (int ch = 0; ch < 8; ++ch) {
                            uint4 v;
                            v.x = pack_bf16x2(__uint_as_float(r[8 * ch + 0]) * inv, __uint_as_float(r[8 * ch + 1]) * inv);
                            v.y = pack_bf16x2(__uint_as_float(r[8 * ch + 2]) * inv, __uint_as_float(r[8 * ch + 3]) * inv);
                            v.z = pack_bf16x2(__uint_as_float(r[8 * ch + 4]) * inv, __uint_as_float(r[8 * ch + 5]) * inv);
                            v.w = pack_bf16x2(__uint_as_float(r[8 * ch + 6]) * inv, __uint_as_float(r[8 * ch + 7]) * inv);
                            dst[c0 / 8 + ch] = v;
                        }
                    } else {
#pragma unroll
                        for (int x = 0; x < 16; ++x)
                            pdst[c0 / 4 + x] = make_float4(__uint_as_float(r[4 * x]), __uint_as_float(r[4 * x + 1]),
                                                           __uint_as_float(r[4 * x + 2]), __uint_as_float(r[4 * x + 3]));
                    }
                }
                if (!kCluster && !whole && write) {
                    slot[128 * kD + rloc] = m_ref;
                    slot[128 * kD + 128 + rloc] = l;
                }
                if (!has_next)
                    break;
                // every QK^T of the finished segment has been consumed: its Q buffer is free
                if (has_fut)
                    stage(fut, sg + 2);
                cur = nxt;
                nxt = fut;
                has_next = has_fut;
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    wait_previous();  // also where a role had nothing to do: the grid completes after the stream's previous work
    tc_fence_before();
    __syncwarp();
    if constexpr (kCluster)
        cluster_arrive();  // this warp's part of (O, m, l) is in shared memory
    __syncthreads();
    if (warp == 1) {
        if (lane == 0)
            mbar_wait_drain(&drain_bar, 0);
        __syncwarp();
        tmem_dealloc(tmem, 512);
    }
    if constexpr (kCluster) {
        cluster_wait();  // every CTA's (O, m, l) is in its shared memory
        if (p.cluster == 1)
            return;  // whole units: written
        const TcSeq &sq = seqs[0];
        const int n_cta = p.cluster, rank = c % n_cta, u = c / n_cta;
        const int rb = u % sq.row_blocks;
        const int head = (u / sq.row_blocks) % p.Hkv;
        const int layer_rel = u / (sq.row_blocks * p.Hkv);
        const int rows_here = abort_flag ? 0 : min(128, sq.rows - rb * 128);
        // This CTA's rows are rank, rank + n_cta, ..: kVec lanes per row, four columns
        // each, the first n_cta of them also one rank's maximum and sum; all of a
        // row's loads are in flight together.
        const int n_rows = (rows_here - rank + n_cta - 1) / n_cta;
        constexpr int kVec = kD / 4;
        const int sub = lane % kVec, base_lane = lane - sub;
        const uint32_t o_base = smem_u32(smem), m_base = smem_u32(s_info[0].m), l_base = smem_u32(s_info[0].l);
        for (int x0 = warp * 32; x0 < n_rows * kVec; x0 += kTcThreads) {
            const int i = (x0 + lane) / kVec, r = i * n_cta + rank;
            const int n = i < n_rows ? n_cta : 0;  // at head_dim 64 a warp's second row may not exist
            const uint32_t o_addr = o_base + (uint32_t)(r * kClusterLd + 4 * sub) * 4;
            float4 v[kMaxCluster];
#pragma unroll
            for (int k = 0; k < kMaxCluster; ++k)
                if (k < n)
                    v[k] = ld_cluster_f32x4(cluster_addr(o_addr, k));
            const float m = sub < n ? ld_cluster_f32(cluster_addr(m_base + 4 * r, sub)) : -INFINITY;
            const float l = sub < n ? ld_cluster_f32(cluster_addr(l_base + 4 * r, sub)) : 0.f;
            float M = m;
#pragma unroll
            for (int k = kMaxCluster / 2; k >= 1; k >>= 1)
                M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, k));
            const float w = m == -INFINITY ? 0.f : ex2_approx(m - M);  // right in the first kMaxCluster lanes
            float lsum = w * l;
#pragma unroll
            for (int k = kMaxCluster / 2; k >= 1; k >>= 1)
                lsum += __shfl_xor_sync(0xffffffffu, lsum, k);
            const float inv = 1.f / __shfl_sync(0xffffffffu, lsum, base_lane);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < kMaxCluster; ++k) {
                const float wk = __shfl_sync(0xffffffffu, w, base_lane + k);
                if (k < n)
                    acc.x += wk * v[k].x, acc.y += wk * v[k].y, acc.z += wk * v[k].z, acc.w += wk * v[k].w;
            }
            const int grow = rb * 128 + r;
            const int node = grow / p.group;
            const int qh = head * p.group + grow % p.group;
            if (n > 0 && in_bounds(layer_rel < p.n_layers && node < sq.nstride && qh < p.Hq, p.status))
                *reinterpret_cast<uint2 *>(sq.out + (((size_t)layer_rel * sq.nstride + node) * p.Hq + qh) * kD +
                                           4 * sub) =
                    make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
        }
        cluster_barrier();  // no CTA leaves while another reads its shared memory
    }
}

// Log-sum-exp merge of the partials of every unit split between CTAs.  A unit
// is split exactly when a CTA range starts inside it, so the grid runs over
// the CTA boundaries c = 1 .. P-1 (x) and groups of 8 query rows (y); the
// first boundary inside a unit handles it.  One warp per query row, each lane
// kD / 32 of the kD output columns.  Latency bounds it: the first block's
// maxima, sums and four rows are loaded together (one round trip for the usual
// unit, split between two or three CTAs), then four slots' rows at a time (2
// heads x 128 at 12000 keys, 38 slots a unit: 25.9 us a call with the maxima
// loaded first, 22.8 now); two CTAs of 256 threads per SM, so that nothing spills.
//
// kAfterStep: launched as a programmatic dependent of a verification step's
// acceptance kernel.  The attention it merges has completed by then (the
// acceptance kernel proceeds only once the LM head has, and the LM head
// completes only after the attention), so it does not wait at entry and runs
// beside the acceptance kernel; at exit it waits for the acceptance kernel,
// so that the stream's next kernel also runs after the compaction.
// Otherwise it waits at entry for the stream's previous kernel.
struct PdlWaitOnExit {
    __device__ ~PdlWaitOnExit() { pdl_wait(); }
};

// kD / 32 consecutive floats of a partial row (one lane's columns)
template <int kCpl>
struct ColVec;
template <>
struct ColVec<4> {
    float v[4];
    __device__ __forceinline__ void load(const float *src)
    {
        const float4 x = __ldcg(reinterpret_cast<const float4 *>(src));
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    }
};
template <>
struct ColVec<2> {
    float v[2];
    __device__ __forceinline__ void load(const float *src)
    {
        const float2 x = __ldcg(reinterpret_cast<const float2 *>(src));
        v[0] = x.x, v[1] = x.y;
    }
};

template <int kD, bool kBatched, bool kAfterStep>
__global__ void __launch_bounds__(256, 2) k1_merge_split(const __grid_constant__ TcKernelParams<kBatched> p)
{
    constexpr int kSlot = slot_floats(kD);
    constexpr int kCpl = kD / 32;  // output columns per lane
    if constexpr (!kAfterStep)
        pdl_wait();
    pdl_trigger();
    PdlWaitOnExit pdl_exit;
    __shared__ TcSeq s_seq;
    __shared__ long long s_total;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const TcSeq *seqs = p.seq;
    long long total = p.total;
    if (p.sched) {
        if (threadIdx.x == 0)
            sched_plan(p, p.seq[0], &s_seq, &s_total);
        __syncthreads();
        seqs = &s_seq;
        total = s_total;
    }
    const int rs = kBatched ? 1 : seqs[0].row_split;
    const int P = tc_split_ctas(p, total, rs);
    const int cb = blockIdx.x + 1;  // CTA range starting at tile t_c
    if (cb >= P)
        return;
    const long long tc = tc_seg_begin(total, P, cb);
    int b = 0;
    if constexpr (kBatched) {
        while (b + 1 < p.n_seq && tc >= seqs[b + 1].tile_base)
            ++b;
    }
    const TcSeq &sq = seqs[b];
    const int u = (int)((tc - sq.tile_base) / sq.T);
    const long long u_first = sq.tile_base + (long long)u * sq.T, u_last = u_first + sq.T;
    if (tc == u_first)
        return;  // the boundary is a unit boundary
    const int c_lo = tc_cta_of(total, P, u_first), c_hi = tc_cta_of(total, P, u_last - 1);
    if (cb != c_lo + 1)
        return;  // an earlier boundary inside this unit handles it
    const int nseg = c_hi - c_lo + 1;
    const int head = (u / sq.row_blocks) % p.Hkv;
    const int layer_rel = u / (sq.row_blocks * p.Hkv);
    const int r_all = blockIdx.y * 8 + warp;  // row of the unit: of both row blocks when split between two CTAs
    const int half = rs == 2 ? r_all / 128 : 0;
    const int r = r_all - 128 * half, rb = u % sq.row_blocks + half;
    if (r >= min(128, sq.rows - rb * 128))
        return;
    {
        const int grow = rb * 128 + r;
        if (!in_bounds(c_lo >= 0 && c_hi < P && layer_rel < p.n_layers && grow / p.group < sq.nstride &&
                           head * p.group + grow % p.group < p.Hq,
                       p.status))
            return;
    }
    // Lane j of each 32-slot block owns slot c_lo + j0 + j: its row pointer,
    // maximum and sum.  The first block's four first rows are loaded with them (a
    // unit is mostly split between two or three CTAs): one round trip to memory.
    constexpr int kEarly = 4;
    auto slot_of = [&](int k) {
        const int cc = c_lo + k;
        return p.part + ((size_t)(cc * rs + half) * 2 + (tc_seg_begin(total, P, cc) >= u_first ? 0 : 1)) * kSlot;
    };
    const float *sl = lane < nseg ? slot_of(lane) : p.part;
    float ms = lane < nseg ? __ldcg(sl + 128 * kD + r) : -INFINITY;
    float ls = lane < nseg ? __ldcg(sl + 128 * kD + 128 + r) : 0.f;
    unsigned long long row_ptr = reinterpret_cast<unsigned long long>(sl + r * kD);
    ColVec<kCpl> early[kEarly];
#pragma unroll
    for (int k = 0; k < kEarly; ++k) {
        // lane's column block of slot k
        const unsigned long long base = __shfl_sync(0xffffffffu, row_ptr, k) + 4ull * kCpl * lane;
        if (k < nseg)
            early[k].load(reinterpret_cast<const float *>(base));
    }
    float M = ms;
    for (int j0 = 32; j0 < nseg; j0 += 32)
        if (j0 + lane < nseg)
            M = fmaxf(M, __ldcg(slot_of(j0 + lane) + 128 * kD + r));
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1)
        M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, m));
    float lsum = 0.f;
    float acc[kCpl] = {};
    for (int j0 = 0; j0 < nseg; j0 += 32) {
        if (j0 > 0) {
            const bool have = j0 + lane < nseg;
            sl = have ? slot_of(j0 + lane) : p.part;
            ms = have ? __ldcg(sl + 128 * kD + r) : -INFINITY;
            ls = have ? __ldcg(sl + 128 * kD + 128 + r) : 0.f;
            row_ptr = reinterpret_cast<unsigned long long>(sl + r * kD);
        }
        const float w = (ms == -INFINITY) ? 0.f : ex2_approx(ms - M);
        lsum += w * ls;
        const int cnt = min(32, nseg - j0);
        for (int j1 = 0; j1 < cnt; j1 += 4) {
            ColVec<kCpl> v[4];
            float wk[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int src = (j1 + k) & 31;
                const unsigned long long base = __shfl_sync(0xffffffffu, row_ptr, src) + 4ull * kCpl * lane;
                wk[k] = __shfl_sync(0xffffffffu, w, src);
                if (j0 == 0 && j1 == 0)
                    v[k] = early[k];
                else if (j1 + k < cnt)
                    v[k].load(reinterpret_cast<const float *>(base));
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (j1 + k < cnt)
#pragma unroll
                    for (int x = 0; x < kCpl; ++x)
                        acc[x] += wk[k] * v[k].v[x];
        }
    }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1)
        lsum += __shfl_xor_sync(0xffffffffu, lsum, m);
    const float inv = 1.f / lsum;
    const int grow = rb * 128 + r;
    const int node = grow / p.group;
    const int qh = head * p.group + grow % p.group;
    __nv_bfloat16 *orow = sq.out + (((size_t)layer_rel * sq.nstride + node) * p.Hq + qh) * kD;
    if constexpr (kCpl == 4)
        reinterpret_cast<uint2 *>(orow)[lane] =
            make_uint2(pack_bf16x2(acc[0] * inv, acc[1] * inv), pack_bf16x2(acc[2] * inv, acc[3] * inv));
    else
        reinterpret_cast<uint32_t *>(orow)[lane] = pack_bf16x2(acc[0] * inv, acc[1] * inv);
}

// ----------------------------------------------------------------------------
// host side

// The parameters of a launch of one sequence.
static TcKernelParams<false> one_seq(const TcParams &p)
{
    TcKernelParams<false> q;
    static_cast<TcCommon &>(q) = p;
    q.tmap[0] = p.tmap[0];
    q.tmap[1] = p.tmap[1];
    q.seq[0] = p.seq[0];
    return q;
}

// The split-unit merge of an attention launch with parameters p, for head_dim
// kD.
template <int kD, bool kBatched, bool kAfterStep>
static cudaError_t merge_launch_d(const TcKernelParams<kBatched> &p, cudaStream_t stream, bool pdl)
{
    // scheduled mode chooses row_split on the device: the grid covers both choices
    const dim3 grid((p.sched ? p.P : p.P / p.seq[0].row_split) - 1, (p.max_rows + 7) / 8);
    return launch_kernel(k1_merge_split<kD, kBatched, kAfterStep>, grid, dim3(256), 0, stream, pdl, p);
}

// Whether a CTA range of the launch starts inside a unit (the split merge then
// has work).  Scheduled mode plans on the device: assumed so.
static bool any_split(const TcParams &p)
{
    if (p.P <= 1 || p.cluster > 0)
        return false;
    if (p.sched)
        return true;
    int b = 0;
    const int n = p.P / p.seq[0].row_split;
    for (int c = 1; c < n; ++c) {
        const long long t = (long long)((unsigned long long)c * (unsigned long long)p.total / (unsigned long long)n);
        while (b + 1 < p.n_seq && t >= p.seq[b + 1].tile_base)
            ++b;
        if ((t - p.seq[b].tile_base) % p.seq[b].T != 0)
            return true;
    }
    return false;
}

// The split-unit merge right behind the attention, when the launch split a unit
// (nothing to do otherwise).
static cudaError_t merge_launch(const TcParams &p, bool batched, cudaStream_t stream, bool pdl)
{
    if (!any_split(p))
        return cudaSuccess;
    if (batched)
        return p.d == 64 ? merge_launch_d<64, true, false>(p, stream, pdl)
                         : merge_launch_d<128, true, false>(p, stream, pdl);
    const TcKernelParams<false> one = one_seq(p);
    return p.d == 64 ? merge_launch_d<64, false, false>(one, stream, pdl)
                     : merge_launch_d<128, false, false>(one, stream, pdl);
}

// The attention kernel for p.d, one CTA per SM (each holds 512 TMEM columns).
static size_t attn_smem(int d, bool cluster)
{
    // a cluster launch has room for the rotary table and the depths behind the rings
    return (size_t)attn_ring_bytes(d) + 1024 + (cluster ? (size_t)kMaxNodes * (d / 2) * sizeof(float2) + kMaxNodes : 0);
}

template <int kD, bool kBatched, bool kCluster>
static cudaError_t attn_kernel_launch_d(const TcParams &p, cudaStream_t stream, bool pdl, const tb_kv *kv = nullptr)
{
    cudaError_t e;
    if ((e = allow_max_smem((const void *)k1_tree_attention_tc<kD, kBatched, kCluster>)) != cudaSuccess)
        return e;
    const size_t smem = attn_smem(kD, kCluster);
    if constexpr (kBatched) {
        return launch_kernel(k1_tree_attention_tc<kD, true, false>, dim3(p.P), dim3(kTcThreads), smem, stream, pdl, p);
    } else if constexpr (kCluster) {
        TcClusterParams q;
        static_cast<TcParamsOf<1> &>(q) = one_seq(p);
        q.rope = kv->rope_theta != 0.f && !p.rope_tab;
        if (q.rope) {
            q.k = static_cast<__nv_bfloat16 *>(kv->k);
            q.k_layer_stride = kv->layer_stride;
            q.k_head_stride = kv->head_stride;
            rope_inv_freq((double)kv->rope_theta, kv->head_dim, q.inv_freq);
        }
        return launch_kernel_cluster(k1_tree_attention_tc<kD, false, true>, dim3(p.P), dim3(kTcThreads), smem, stream,
                                     pdl, p.cluster, q);
    } else {
        return launch_kernel(k1_tree_attention_tc<kD, false, false>, dim3(p.P), dim3(kTcThreads), smem, stream, pdl,
                             one_seq(p));
    }
}

static cudaError_t attn_kernel_launch(const TcParams &p, bool batched, cudaStream_t stream, bool pdl,
                                      const tb_kv *kv = nullptr)
{
    if (p.cluster > 0)
        return p.d == 64 ? attn_kernel_launch_d<64, false, true>(p, stream, pdl, kv)
                         : attn_kernel_launch_d<128, false, true>(p, stream, pdl, kv);
    if (p.d == 64)
        return batched ? attn_kernel_launch_d<64, true, false>(p, stream, pdl)
                       : attn_kernel_launch_d<64, false, false>(p, stream, pdl);
    return batched ? attn_kernel_launch_d<128, true, false>(p, stream, pdl)
                   : attn_kernel_launch_d<128, false, false>(p, stream, pdl);
}

// Clusters of `size` CTAs of the attention kernel that can be resident at once
// on the current device (0 if none).
template <int kD>
static int attn_max_clusters(int size)
{
    static PerDevice<kMaxCluster + 1> clusters;
    return clusters.get(size, [size] {
        return ask_max_clusters((const void *)k1_tree_attention_tc<kD, false, true>, size, kTcThreads,
                                attn_smem(kD, true));
    });
}

// The attention launch's parameters, kept for a split-unit merge enqueued later.
static void stash_merge(const TcParams &p, AttnMerge *m)
{
    TcKernelParams<false> q = one_seq(p);
    static_assert(sizeof q <= sizeof(m->params), "AttnMerge holds the attention launch's parameters");
    q.sched = p.sched ? p.sched_copy : nullptr;
    memcpy(m->params, &q, sizeof q);
    m->pending = any_split(p);
}

bool attn_tc_supported(int d)
{
    return d == 64 || d == 128;
}

AttnPlan attn_tc_plan(int L, int N, int Hq, int Hkv, int n_layers, int n_sm)
{
    AttnPlan pl{};
    pl.group = Hq / Hkv;
    pl.rows = N * pl.group;
    pl.row_blocks = (pl.rows + 127) / 128;
    pl.T = (L + N + kBN - 1) / kBN;
    pl.n_units = n_layers * Hkv * pl.row_blocks;
    pl.total = (long long)pl.n_units * pl.T;
    long long P = n_sm;
    if (P > pl.total)
        P = pl.total;
    // A problem of one wave whose units are a few tiles long runs a whole unit
    // per CTA: a split would save those tiles' serial steps (about 1 us each on
    // one SM) but add the split merge's launch and round trips (measured on
    // GB300: whole units faster up to 5 tiles, even at 6-7).
    if (pl.total <= n_sm && pl.T <= kWholeUnitMaxTiles)
        P = pl.n_units;
    pl.row_split = 1;
    if (split_rows(pl.row_blocks, pl.total, n_sm)) {
        pl.row_split = 2;
        P &= ~1ll;
    }
    pl.P = (int)P;
    return pl;
}

// CTAs per unit of a stand-alone attention call of one sequence (1: no
// clusters): as many as fit the SMs with every unit's cluster resident at once;
// units of a few tiles run whole (32 q / 8 kv heads x 128, 64 nodes at 100 and
// 400 keys: 8.5 and 10.4 us whole, 10.9 and 11.1 in clusters).
// The clusters save the partials' round trip through memory and the merge
// launch, but leave SMs idle when the units do not divide them.  At head_dim
// 128 three quarters of the SMs still saturate HBM, and the clusters win at
// any length.  Otherwise they win while the longest CTA has at most about
// `size` tiles more than an even split over all SMs would give it.  Measured on
// GB300, one layer, clusters / even split: 32 kv heads x 128, 26 nodes at 700,
// 1500, 24000 keys 11.0 / 13.8, 12.7 / 16.0, 64.1 / 67.9 us; 8 heads x 128 at
// 12000 and 24000 keys 20.9 / 21.6 and 33.1 / 29.2; 64 heads x 64 at 3000 and
// 6000 keys 20.7 / 21.9 and 32.6 / 32.2.
static int attn_tc_clusters(const AttnPlan &pl, int d, int n_sm)
{
    if (pl.total <= n_sm && (pl.T <= 2 || (pl.T <= 4 && pl.rows > 64)))
        return 1;
    int size = n_sm / pl.n_units;
    size = size < kMaxCluster ? size : kMaxCluster;
    size = size < pl.T ? size : pl.T;
    for (; size > 1; --size)
        if (pl.n_units <= (d == 64 ? attn_max_clusters<64>(size) : attn_max_clusters<128>(size)))
            break;
    if (size <= 1)
        return 1;
    if (d == 128 && 4 * pl.n_units * size >= 3 * n_sm)
        return size;
    const long long longest = (pl.T + size - 1) / size, even = pl.total / n_sm;
    return longest - even <= size ? size : 1;
}

// The launch of a stand-alone call of one sequence: its cluster size (0: the
// ordinary kernel), and whether it applies the rotary embedding itself, which
// saves the rotary kernel.  It does where exactly one CTA reads a tree tile of a
// unit (one row block per kv head): units shared by clusters, and units run
// whole (then on the cluster kernel with one CTA per unit).
static int alone_cluster(const AttnPlan &pl, int d, int n_sm, bool rope, bool *fused)
{
    const int size = attn_tc_clusters(pl, d, n_sm);
    const bool whole = pl.P == pl.n_units && pl.row_split == 1;
    *fused = rope && pl.row_blocks == 1 && (size > 1 || whole);
    return size > 1 ? size : *fused ? 1 : 0;
}

bool attn_tc_fuses_rope(const tb_kv *kv, int N, int Hq, int n_layers, int n_sm)
{
    bool fused;
    alone_cluster(attn_tc_plan(kv->L, N, Hq, kv->n_kv_heads, n_layers, n_sm), kv->head_dim, n_sm,
                  kv->rope_theta != 0.f, &fused);
    return fused;
}

bool attn_tc_clustered(const tb_kv *kv, int N, int Hq, int n_layers, int n_sm)
{
    bool fused;
    return alone_cluster(attn_tc_plan(kv->L, N, Hq, kv->n_kv_heads, n_layers, n_sm), kv->head_dim, n_sm,
                         kv->rope_theta != 0.f, &fused) > 0;
}

size_t attn_tc_slot_floats(int d)
{
    return (size_t)slot_floats(d);
}

int attn_tc_units(const AttnSeq *seqs, int n_seq, int Hq, int Hkv, int n_layers)
{
    int units = 0;
    for (int b = 0; b < n_seq; ++b)
        units += attn_tc_plan(seqs[b].kv->L, seqs[b].N, Hq, Hkv, n_layers, 1).n_units;
    return units;
}

cudaError_t attn_tc_launch_batch(const AttnSeq *seqs, int n_seq, int layer_begin, int n_layers, int Hq, float *part,
                                 int *status, int n_sm, cudaStream_t stream, const char **err,
                                 const float2 *rope_tab, AttnMerge *merge_later, bool alone)
{
    if (n_seq < 1 || n_seq > kMaxSeqPerLaunch || (n_seq > 1 && merge_later)) {
        *err = "too many sequences for one attention launch";
        return cudaErrorInvalidValue;
    }
    TcParams p{};
    long long tiles = 0;
    int max_rows = 0;
    const int Hkv = seqs[0].kv->n_kv_heads;
    const int d = seqs[0].kv->head_dim;
    if (!attn_tc_supported(d)) {
        *err = "head_dim 64 or 128";
        return cudaErrorInvalidValue;
    }
    for (int b = 0; b < n_seq; ++b) {
        const tb_kv *kv = seqs[b].kv;
        if (kv->head_dim != d || kv->n_kv_heads != Hkv) {
            *err = "the sequences of one attention launch share head_dim and kv heads";
            return cudaErrorInvalidValue;
        }
        const AttnPlan pl = attn_tc_plan(kv->L, seqs[b].N, Hq, Hkv, n_layers, n_sm);
        if (!make_tmap_kv(&p.tmap[2 * b], kv->k, d, kv->L + seqs[b].N, kv->n_kv_heads, kv->n_layers,
                          kv->head_stride, kv->layer_stride, kBN, err) ||
            !make_tmap_kv(&p.tmap[2 * b + 1], kv->v, d, kv->L + seqs[b].N, kv->n_kv_heads, kv->n_layers,
                          kv->head_stride, kv->layer_stride, kBN, err))
            return cudaErrorInvalidValue;
        TcSeq &sq = p.seq[b];
        sq.tile_base = tiles;
        sq.q = static_cast<const __nv_bfloat16 *>(seqs[b].q);
        sq.out = static_cast<__nv_bfloat16 *>(seqs[b].out);
        sq.tree = seqs[b].tree;
        sq.L = kv->L;
        sq.N = seqs[b].N;
        sq.rows = pl.rows;
        sq.row_blocks = pl.row_blocks;
        sq.T = pl.T;
        sq.nstride = seqs[b].N;
        sq.row_split = 1;
        tiles += pl.total;
        max_rows = pl.rows < 128 ? (pl.rows > max_rows ? pl.rows : max_rows) : 128;
    }
    p.n_seq = n_seq;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.group = Hq / Hkv;
    p.layer_begin = layer_begin;
    p.n_layers = n_layers;
    p.total = tiles;
    // a batch splits its tiles evenly (units of different lengths)
    p.P = (int)(tiles < n_sm ? tiles : n_sm);
    p.cluster = 0;
    if (n_seq == 1) {
        // one sequence: its plan (whole units for a short one-wave problem), or in a call of its
        // own (and a step that runs it like one) clusters that share the units of a small problem
        const AttnPlan pl = attn_tc_plan(seqs[0].kv->L, seqs[0].N, Hq, Hkv, n_layers, n_sm);
        p.P = pl.P;
        bool fused = false;
        if (alone)
            p.cluster = alone_cluster(pl, d, n_sm, seqs[0].kv->rope_theta != 0.f, &fused);
        if (p.cluster > 0) {
            p.P = pl.n_units * p.cluster;
        } else if (pl.row_split == 2) {
            p.seq[0].row_split = 2;
            p.seq[0].row_blocks = 1;
            p.total = tiles / 2;
            max_rows = pl.rows;
        }
    }
    p.d = d;
    p.scale_log2 = 1.4426950408889634f / sqrtf((float)d);
    p.part = part;
    p.status = status;
    p.rope_tab = rope_tab;
    p.max_rows = max_rows;
    const bool batched = n_seq > 1;
    cudaError_t e;
    // In a forked step the grid starts when the stream's previous work is done,
    // so that all its CTAs start together (its work split is static) and before
    // the LM head's; in a chain (merge_later) it is launched as a programmatic
    // dependent.  A call of its own is launched as a programmatic
    // dependent too, and so is its merge: only the set-up overlaps what runs
    // before, each kernel waiting for the one it follows.
    const bool pdl = alone || merge_later;
    if ((e = attn_kernel_launch(p, batched, stream, pdl, seqs[0].kv)) != cudaSuccess)
        return e;
    if (merge_later) {
        stash_merge(p, merge_later);
        return cudaSuccess;
    }
    // In a step, a plain dependent of the attention: launched as a programmatic
    // one, its CTAs would take the SMs that attention CTAs release and hold them until
    // the whole grid is done, away from an LM head beside it on another stream
    // (measured on GB300: the ragged batch's step 20 us longer).
    return merge_launch(p, batched, stream, alone);
}

cudaError_t attn_tc_launch_sched(const AttnSched &sc, int Hq, float *part, int *status, int n_sm,
                                 cudaStream_t stream, const char **err, AttnMerge *merge_later)
{
    if (sc.n_rungs < 1 || sc.n_rungs > 8) {
        *err = "scheduled attention: 1..8 rungs";
        return cudaErrorInvalidValue;
    }
    const tb_kv *kv = sc.kv;
    const int d = kv->head_dim;
    if (!attn_tc_supported(d)) {
        *err = "head_dim 64 or 128";
        return cudaErrorInvalidValue;
    }
    TcParams p{};
    // the cache's whole capacity: keys past L + N are masked by the kernel
    if (!make_tmap_kv(&p.tmap[0], kv->k, d, kv->L_cap, kv->n_kv_heads, kv->n_layers, kv->head_stride,
                      kv->layer_stride, kBN, err) ||
        !make_tmap_kv(&p.tmap[1], kv->v, d, kv->L_cap, kv->n_kv_heads, kv->n_layers, kv->head_stride,
                      kv->layer_stride, kBN, err))
        return cudaErrorInvalidValue;
    TcSeq &sq = p.seq[0];
    sq.q = static_cast<const __nv_bfloat16 *>(sc.q);
    sq.out = static_cast<__nv_bfloat16 *>(sc.out);
    sq.tree = sc.rung_tree[0];
    sq.nstride = sc.N_max;
    sq.T = 1;
    sq.row_blocks = 1;
    sq.row_split = 1;
    p.n_seq = 1;
    p.Hq = Hq;
    p.Hkv = kv->n_kv_heads;
    p.group = Hq / kv->n_kv_heads;
    p.layer_begin = 0;
    p.n_layers = kv->n_layers;
    p.L_cap = kv->L_cap;
    p.P = n_sm;
    p.d = d;
    p.scale_log2 = 1.4426950408889634f / sqrtf((float)d);
    p.part = part;
    p.status = status;
    p.sched = sc.sched;
    p.sched_copy = sc.sched_copy;
    p.rope_tab = sc.rope_tab;
    p.n_rungs = sc.n_rungs;
    for (int r = 0; r < sc.n_rungs; ++r)
        p.rung_tree[r] = sc.rung_tree[r];
    p.max_rows = sc.N_max * p.group;
    cudaError_t e;
    if ((e = attn_kernel_launch(p, false, stream, merge_later != nullptr)) != cudaSuccess)
        return e;
    if (merge_later) {
        stash_merge(p, merge_later);
        return cudaSuccess;
    }
    p.sched = p.sched_copy;
    return merge_launch(p, false, stream, false);
}

cudaError_t attn_tc_launch(const tb_kv *kv, const TreeDesc *d_tree, int N, int layer_begin, int n_layers,
                           const void *q, int Hq, void *out, float *part, int *status, int n_sm,
                           cudaStream_t stream, const char **err, const float2 *rope_tab, AttnMerge *merge_later,
                           bool alone)
{
    AttnSeq one{kv, d_tree, N, q, out};
    return attn_tc_launch_batch(&one, 1, layer_begin, n_layers, Hq, part, status, n_sm, stream, err, rope_tab,
                                merge_later, alone);
}

cudaError_t attn_merge_launch(const AttnMerge &m, cudaStream_t stream)
{
    if (!m.pending)
        return cudaSuccess;
    TcKernelParams<false> p;
    memcpy(&p, m.params, sizeof p);
    return p.d == 64 ? merge_launch_d<64, false, true>(p, stream, true)
                     : merge_launch_d<128, false, true>(p, stream, true);
}

TB_BOUNDS_COUNTER(bounds_violations_attention_tc)

}  // namespace tv
