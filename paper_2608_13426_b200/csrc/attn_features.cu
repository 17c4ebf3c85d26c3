// Feature scores and kept features of attention heads (paper Sec. 3.3: per query head the columns of Q of largest 2-norm).
//
// A cluster of eight blocks owns a head, each an eighth of its query rows: every thread sums the squares of eight adjacent columns
// over its rows (eight 16-byte loads in flight; fp32 chains of 16 exact squares, then fp64), the blocks' sums meet through
// distributed shared memory in rank order, and the first block ranks all features by comparing all pairs (at most 256 keys).
// Bound by HBM for long prompts and else by the chain of latencies, which is why nothing passes through global memory: the general
// score pass publishes partial sums, hands them to the last block of a column range and the energies to the last block of a head.
// Kernel by events: 2 heads x 600 x 128 14.4 -> 10.1 us, 8 x 1172 x 128 18.6 -> 11.5 (attn_features_eligible has whole calls).
#include "common.cuh"
#include "select.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

using namespace ptx;

constexpr int kFeatBlocks = 8;     // blocks of a cluster
constexpr int kFeatThreads = 256;
constexpr int kFeatMaxDh = kFeatThreads;

struct FeatArgs {
    const __nv_bfloat16 *q;
    int64_t q_sh, q_sr, Lq;   // element strides: head, row
    int Dh, kd;
    int32_t *idx;             // [heads, kd], ascending
};

__global__ void __launch_bounds__(kFeatThreads) attn_features_kernel(const FeatArgs a)
{
    __shared__ __align__(16) double s_part[kFeatThreads * 8];
    __shared__ double s_sum[kFeatMaxDh];
    __shared__ __align__(16) unsigned s_key[kFeatMaxDh];
    __shared__ unsigned s_kept[kFeatThreads / 32];
    pdl_wait();

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_rank();
    const int64_t head = blockIdx.x / kFeatBlocks;
    const int Dh = a.Dh, nv = Dh / 8, rows_par = kFeatThreads / nv, c = tid % nv, rsub = tid / nv;
    const int64_t per = (a.Lq + kFeatBlocks - 1) / kFeatBlocks, r0 = min(a.Lq, rank * per), r1 = min(a.Lq, r0 + per);
    if (rsub < rows_par) {
        double dacc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) dacc[e] = 0.0;
        const __nv_bfloat16 *col = a.q + head * a.q_sh + c * 8;
        for (int64_t r = r0 + rsub; r < r1; r += 16 * rows_par) {
            float facc[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) facc[e] = 0.f;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint4 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int64_t rr = r + (int64_t)(half * 8 + i) * rows_par;
                    v[i] = rr < r1 ? __ldg(reinterpret_cast<const uint4 *>(col + rr * a.q_sr)) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const unsigned w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const float lo = __uint_as_float(w[p] << 16), hi = __uint_as_float(w[p] & 0xffff0000u);
                        facc[2 * p] = fmaf(lo, lo, facc[2 * p]);
                        facc[2 * p + 1] = fmaf(hi, hi, facc[2 * p + 1]);
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) dacc[e] += (double)facc[e];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) s_part[rsub * Dh + c * 8 + e] = dacc[e];
    }
    __syncthreads();
    if (tid < Dh) {
        double s = 0.0;
#pragma unroll 4
        for (int y = 0; y < rows_par; ++y) s += s_part[y * Dh + tid];
        s_sum[tid] = s;
    }
    __syncthreads();
    cluster_sync_all();
    unsigned u = 0;
    if (rank == 0 && tid < Dh) {
        const uint32_t mine = smem_u32(&s_sum[tid]);
        double v[kFeatBlocks], s = 0.0;
#pragma unroll
        for (int r = 0; r < kFeatBlocks; ++r) asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[r]) : "r"(map_to_cta(mine, r)) : "memory");
#pragma unroll
        for (int r = 0; r < kFeatBlocks; ++r) s += v[r];
        u = sel::key_image((float)s);
    }
    __syncthreads();
    cluster_sync_all();   // a block's shared memory stays until its sums have been read
    if (rank != 0) return;
    s_key[tid] = u;
    __syncthreads();
    // those that fewer than kd others come before (larger, or equal with a lower index)
    unsigned before = 0;
    for (int i = 0; i < Dh; i += 4) {
        const uint4 o = *reinterpret_cast<const uint4 *>(&s_key[i]);
        before += (o.x > u || (o.x == u && i < tid)) ? 1u : 0u;
        before += (o.y > u || (o.y == u && i + 1 < tid)) ? 1u : 0u;
        before += (o.z > u || (o.z == u && i + 2 < tid)) ? 1u : 0u;
        before += (o.w > u || (o.w == u && i + 3 < tid)) ? 1u : 0u;
    }
    const bool keep = tid < Dh && before < (unsigned)a.kd;
    const unsigned kept = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) s_kept[warp] = __popc(kept);
    __syncthreads();
    if (keep) {
        unsigned at = __popc(kept & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) at += s_kept[w];
        a.idx[head * a.kd + at] = tid;
    }
}

}  // namespace

bool attn_features_eligible(int64_t heads, int64_t Lq, int64_t Dh)
{
    // Eight blocks a head, each with eight loads a thread in flight: short heads are bound by latency, which is shorter here; long ones
    // want the general pass's deeper pipeline, and many heads queue.  The lines are the crossings of whole calls on 128 keys, here
    // against the general pass, us with Q in L2 / with new inputs each time (one figure: new inputs):
    //   Dh 128,  2 heads: 2500 rows -4.5 / -4.5, 5200 -3.3 / -0.8, 8192 +2.3;  4: 2500 -2.7 / -1.7, 4600 +1.9 / +5.0
    //            8 heads: 2500 -1.0 / -0.4, 3000 +0.4 / +2.1;  16: 2048 -2.1 / -1.0, 2500 -0.7 / +0.5, 3000 -0.1 / +1.9, 4600 +1.5 / +3.6
    //           24 heads: 2048 -0.9 / -0.2, 3000 -0.4 / +0.8;  28: 3500 -1.3 / +0.2, 4096 -1.2 / +0.4, 4600 +0.2 / +1.7
    //           32 heads: 2048 -1.7 / -0.9, 3000 -1.0 / -0.1, 4096 -0.6 / 0.0 (whole call on 4096 keys: -0.8 / -1.2), 4600 +1.5 / +1.5
    //           40 heads: 2048 -1.0 / 0.0;  48: 2048 +2.6, 4096 +5.4;  64: 2048 +4.9
    //   Dh 64,   2 heads: 10000 -3.7 / -1.0;  8: 4096 -2.4 / -1.1, 7000 -1.1 / +1.3;  40: 4096 -3.3 / -3.1;  48: 4096 +1.0
    //   Dh 256,  1 head: 3000 -1.9 / -1.4;  2: 2048 -4.0 / -1.1;  4: 1000 -2.5 / -1.9, 2048 +2.2 / +4.5;  6: 750 -1.6 / -0.8, 1000 +2.4 / +3.3
    //            8 heads: 250 -3.0 / -1.8, 500 +1.1 / +0.8, 1000 +2.3 / +3.9
    if (Dh > 128) return Dh <= kFeatMaxDh && heads <= 8 && heads * Lq * Dh <= 1 << 20;
    return heads <= 40 && Lq * Dh <= (heads <= 2 ? 5120 : heads < 28 ? 2560 : 4352) * 128;
}

int launch_attn_features(const __nv_bfloat16 *q, int64_t q_sh, int64_t q_sr, int64_t heads, int64_t Lq, int64_t Dh, int64_t kd, int32_t *idx,
                         cudaStream_t stream)
{
    FeatArgs a = {q, q_sh, q_sr, Lq, (int)Dh, (int)kd, idx};
    prof_begin("attn_features_kernel", stream);
    cudaError_t e = launch_kernel(attn_features_kernel, dim3((unsigned)(heads * kFeatBlocks)), dim3(kFeatThreads), 0, stream, kFeatBlocks, a);
    if (e != cudaSuccess) return fail(RMM_ERR_CUDA, "attn_features_kernel: launch: %s", cudaGetErrorString(e));
    return check_launch("attn_features_kernel", stream);
}

}  // namespace rmm
