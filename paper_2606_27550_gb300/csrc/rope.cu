// rope.cu -- rotary position embedding at the tree's position offsets.
//
// The TopologyBank stores each tree's position offsets (Sec. 1, 2.3): node i
// of a step sits at position L + depth(i).  With the base model's rotary
// embedding (Llama convention: theta_i = base^(-2i/d), element i paired with
// element i + d/2) the step's queries and tree keys are rotated at those
// positions; the prefix keys were rotated when they entered the cache.
//
//   k0_rope_tree_k  one launch: a CTA per (tree node, 64 or 128 (layer, kv
//                   head) rows of it).  64 threads form the (cos, sin) of
//                   (L + depth) * theta_i for the node's depth: the angle is
//                   formed and reduced to [-pi, pi] in double (positions reach
//                   10^4-10^5 rad), sin and cos are taken in float.  That part
//                   depends on the topology and L only and runs before the wait
//                   for the stream's previous kernel (the launch is a
//                   programmatic dependent of it).  Then every thread loads its
//                   8 pairs of two rows (16 bytes from each half: the
//                   long-context step's 1024 CTAs are about one wave), rotates
//                   them and writes them back to the bf16 cache in place.  The
//                   first node of each depth (canonical order: depths do not
//                   decrease with the id) also writes its table row to the
//                   workspace for the query rotation.  head_dim 64 or 128
//                   (template kD: kD / 16 threads per row).  What bounds it is
//                   launch and load latency (16.8 MB at 32 layers).
// The queries are rotated inside the attention kernel as they are staged
// into tensor memory (attention_tc.cu), with the same table.
#include <cuda_bf16.h>
#include <string.h>

#include "kernels.cuh"

namespace tv {

constexpr int kRopeThreads = 256;      // kD / 16 threads per row of kD elements
constexpr int kRopeRowsPerThread = 2;  // two rows a CTA-width apart: four 16-byte loads in flight

constexpr int rope_rows_per_cta(int d)
{
    return kRopeThreads / (d / 16) * kRopeRowsPerThread;
}

template <int kD>
__global__ void __launch_bounds__(kRopeThreads) k0_rope_tree_k(const __grid_constant__ RopeParams p, int n_rows)
{
    static_assert(kD == 64 || kD == 128, "head_dim 64 or 128");
    constexpr int kTpr = kD / 16;  // threads per row, 8 pairs each
    constexpr int kRowsPerCta = rope_rows_per_cta(kD);
    __shared__ float2 cs[kRopeMaxHalf];
    const RopeSeq &sq = p.seq[blockIdx.z];
    const TreeDesc *tree = sq.tree;
    int L = sq.L;
    if (p.sched) {
        pdl_wait();
        const int rung = p.sched[0], Ls = p.sched[1];
        if (rung < 0 || rung >= p.n_rungs || Ls < 0 || Ls + p.rung_tree[rung]->n > p.L_cap)
            return;  // no work this step (the acceptance kernel reports it)
        tree = p.rung_tree[rung];
        L = Ls;
    }
    const int j = blockIdx.x;
    constexpr int kHalf = kD / 2;  // pairs of a row
    const bool here = j < tree->n;
    const int dep = here ? tree->depth[j] : 0;
    // The angles depend on the topology and L only: they are formed before the
    // wait for the stream's previous work.
    float2 cn = make_float2(1.f, 0.f);
    if (here && threadIdx.x < kHalf) {
        constexpr double kTwoPi = 6.283185307179586476925286766559;
        const double a = (double)(L + dep) * p.inv_freq[threadIdx.x];
        const double red = a - kTwoPi * rint(a * (1.0 / kTwoPi));
        sincosf((float)red, &cn.y, &cn.x);
        cs[threadIdx.x] = cn;
    }
    pdl_wait();
    pdl_trigger();  // the attention may be launched: it waits for this grid to complete
    if (!here)
        return;
    const int ch = (threadIdx.x % kTpr) * 8;
    __nv_bfloat16 *row[kRopeRowsPerThread];
    uint4 lo[kRopeRowsPerThread], hi[kRopeRowsPerThread];  // elements [ch, ch + 8) and [kHalf + ch, kHalf + ch + 8)
#pragma unroll
    for (int k = 0; k < kRopeRowsPerThread; ++k) {
        const int r = blockIdx.y * kRowsPerCta + k * (kRopeThreads / kTpr) + (int)(threadIdx.x / kTpr);
        row[k] = nullptr;
        lo[k] = hi[k] = make_uint4(0, 0, 0, 0);
        if (r < n_rows && in_bounds((long long)(L + j + 1) * (2 * kHalf) <= sq.head_stride && dep < kMaxNodes, nullptr)) {
            const int head = r % p.Hkv, layer = p.layer_begin + r / p.Hkv;
            row[k] = sq.k + (size_t)layer * sq.layer_stride + (size_t)head * sq.head_stride +
                     (size_t)(L + j) * (2 * kHalf);
            lo[k] = *reinterpret_cast<const uint4 *>(row[k] + ch);
            hi[k] = *reinterpret_cast<const uint4 *>(row[k] + kHalf + ch);
        }
    }
    if (threadIdx.x < kHalf && blockIdx.y == 0 && (j == 0 || tree->depth[j - 1] != dep))
        p.table[(size_t)blockIdx.z * kRopeTableEntries + dep * kRopeMaxHalf + threadIdx.x] = cn;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRopeRowsPerThread; ++k) {
        if (!row[k])
            continue;
        __nv_bfloat16 *x = reinterpret_cast<__nv_bfloat16 *>(&lo[k]), *y = reinterpret_cast<__nv_bfloat16 *>(&hi[k]);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float2 c = cs[ch + e];
            const float x1 = __bfloat162float(x[e]), x2 = __bfloat162float(y[e]);
            x[e] = __float2bfloat16_rn(x1 * c.x - x2 * c.y);
            y[e] = __float2bfloat16_rn(x2 * c.x + x1 * c.y);
        }
        *reinterpret_cast<uint4 *>(row[k] + ch) = lo[k];
        *reinterpret_cast<uint4 *>(row[k] + kHalf + ch) = hi[k];
    }
}

void rope_inv_freq(double theta, int d, double *inv_freq)
{
    // the table of the thread's last (theta, d): a model's never change
    static thread_local double last_theta = 0.0, last[kRopeMaxHalf];
    static thread_local int last_d = 0;
    if (theta != last_theta || d != last_d) {
        for (int i = 0; i < d / 2; ++i)
            last[i] = pow(theta, -2.0 * i / d);
        last_theta = theta;
        last_d = d;
    }
    memcpy(inv_freq, last, sizeof(double) * (d / 2));
}

cudaError_t rope_launch(const RopeParams &p, int n_seq, int max_nodes, int n_layers, cudaStream_t stream)
{
    if (n_seq < 1 || n_seq > TB_MAX_BATCH || (p.d != 64 && p.d != 128) || max_nodes < 1 || max_nodes > kMaxNodes)
        return cudaErrorInvalidValue;
    const int n_rows = n_layers * p.Hkv;
    const int per_cta = rope_rows_per_cta(p.d);
    const dim3 grid(max_nodes, (n_rows + per_cta - 1) / per_cta, n_seq);
    if (p.d == 64)
        return launch_kernel(k0_rope_tree_k<64>, grid, dim3(kRopeThreads), 0, stream, true, p, n_rows);
    return launch_kernel(k0_rope_tree_k<128>, grid, dim3(kRopeThreads), 0, stream, true, p, n_rows);
}

TB_BOUNDS_COUNTER(bounds_violations_rope)

}  // namespace tv
