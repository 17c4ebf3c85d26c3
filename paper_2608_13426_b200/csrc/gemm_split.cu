// Reduced product Y = scale * A[:, I] B[I, :] of fp32 operands on the sm_100a tensor cores.
//
// Every operand is written as the sum of three bf16 numbers, a = a1 + a2 + a3 (each the rounding of what the ones before it
// leave: 24 bits and the signs, so the sum is exact up to 2^-26 of a), and the product of two of them as the six products
// a1 b1 + a1 b2 + a2 b1 + a2 b2 + a1 b3 + a3 b1; what is left out is below 2^-24 of |a b|.  Products of bf16 numbers are
// exact in the tensor cores, but their fp32 accumulators round toward zero: 1504 indices in one cost 1.5e-6 of the result
// (2-norm, normal operands).  So an accumulator takes 64 indices only, the small products first, and is then added to fp32
// registers that round to nearest.  Measured against 64 bits (2-norm) at 64, 1500 and 8192 indices, the FMA kernel (a partial sum
// per 16 indices, one slice) in brackets: normal operands 0.8e-7 1.2e-7 1.5e-7 (0.8e-7 1.9e-7 4.1e-7).  Operands of one sign show
// the rounding toward zero, a mean of -0.7e-7 to -1.2e-7 that the FMA kernel does not have: uniform 0.8e-7 1.1e-7 1.0e-7 (0.5e-7
// 1.5e-7 3.0e-7), exponential 1.0e-7 1.2e-7 1.2e-7 (0.5e-7 1.5e-7 3.0e-7), level at about 1000 indices; e^(2 z), z normal, whose
// largest products hide the others, 5.6e-7 2.9e-7 3.4e-7 (0.8e-7 2.7e-7 3.1e-7).  (A second accumulator, for the products of first
// parts alone, took 6 % off the uniform figure, nothing off the others, and 15 % more time: the loss is inside an instruction.)
// The split is exact only for ordinary magnitudes: a kept element that is not finite, or neither zero nor within 2^-50 .. 2^40,
// is flagged by the gather.  (Within, products of first parts are normal numbers, and what products of later parts lose below
// 2^-126 is less than 2^-26 of them.)  The FMA kernel behind this one, which otherwise returns at once, does the outputs that see
// a flag, or all of them where that is cheaper.  777 x 1500 kept x 1500 with one such element 128 us, 117 by the FMA kernel alone.
//
// Bound: tensor cores (six bf16 products a multiplication: 280 TFLOP/s at the burst rate, where the FMA pipes reach 46), 1.1 us per
// 64 indices of a 256 x 128 tile at that rate.  The tensor pipe is busy for 61 % of 338 us on 2048 x 4096 kept x 4096 (203 TFLOP/s,
// 1.5 us per 64 indices: the copies and the additions are not all hidden), for 32 % of 41.5 us on 777 x 1500 x 1500 (48 tiles for 74
// pairs, a quarter of them nine rows high; pieces and their meeting).  CTA pairs, since a tensor instruction reads both
// its operands from shared memory: 128 bytes a clock for a lone CTA's 128 x 128, all there is, 96 for each CTA of a pair.  Where a
// round of tiles would leave pairs idle its tiles are cut along the contraction; the pieces meet in whichever pair comes last.
// Whole calls, FMA kernel before: 777 x 3000 (half kept) x 1500 123 -> 56 us, 2048 x 8192 (half) x 4096 1486 -> 376 (on a given list),
// 500 x 700 (half) x 4000 48.6 -> 23.2.
#include <cuda.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

using namespace ptx;

constexpr int kTile = 128, kBk = 64, kPlanes = 3;
constexpr int kPlaneA = kTile * kBk * 2, kPlaneB = kTile / 2 * kBk * 2;   // a CTA holds its 128 rows of A and its half of B's 128 columns
constexpr int kStages = 3, kStageBytes = kPlanes * (kPlaneA + kPlaneB);
constexpr int kOffBars = kStages * kStageBytes, kSplitSmem = kOffBars + 128 + 1024;   // (1 KB to align the tiles)
constexpr int kSplitThreads = 384;            // warp 0 copies, warp 1 tensor cores, warps 4-11 add up (8 x 64 columns of 32 rows)

// ---- gather and split: dst[plane][r][j] of src[r, idx[j]] (columns), or dst[plane][j][c] of src[idx[j], c] (rows) ----
struct SplitSpec {
    const float *src;
    __nv_bfloat16 *dst;
    int64_t s_batch, s_row, s_col;   // element strides
    int64_t rows, cols, ld;          // of dst: rows x ld, cols of them valid
    int by_rows, vec;                // by_rows: the list picks rows; vec: four columns are one aligned load
    unsigned blocks_r, blocks_c;
};

struct SplitArgs {
    SplitSpec s[2];
    const int32_t *idx;   // [batch, k] or NULL (0 .. k - 1)
    int64_t k, K;
    int *status, *flags;  // flags[block]: 1 where an element cannot be split
};

constexpr int kGatherThreads = 256, kGatherRows = 16, kGatherCols = 256;   // a thread: four columns of four rows

__device__ __forceinline__ bool unusual(float x)
{
    const uint32_t e = __float_as_uint(x) & 0x7fffffffu, lo = 0x26800000u, hi = 0x53800000u;  // 2^-50, 2^40
    return e != 0u && e - lo > hi - lo;
}

__global__ void __launch_bounds__(kGatherThreads) split_gather_kernel(const SplitArgs a)
{
    pdl_wait();
    const unsigned per0 = a.s[0].blocks_r * a.s[0].blocks_c;
    const bool second = blockIdx.x >= per0;
    const SplitSpec &s = a.s[second ? 1 : 0];
    const unsigned blk = second ? blockIdx.x - per0 : blockIdx.x;
    const int64_t b = blockIdx.y;
    const int64_t r0 = (int64_t)(blk / s.blocks_c) * kGatherRows + threadIdx.x / 64, c0 = (int64_t)(blk % s.blocks_c) * kGatherCols + threadIdx.x % 64 * 4;
    const float *src = s.src + b * s.s_batch;
    const int32_t *idx = a.idx != nullptr ? a.idx + b * a.k : nullptr;
    auto kept = [&](int64_t j) -> int64_t {  // the kept index at position j (< k), -1 if it is out of range
        const int64_t i = idx != nullptr ? (int64_t)__ldg(idx + j) : j;
        if (i >= 0 && i < a.K) return i;
        atomicExch(a.status, (int)RMM_ERR_BOUNDS);
        return -1;
    };
    bool odd = false;
    if (c0 < s.ld) {
        int64_t at[4];   // columns of src, -1: zero
#pragma unroll
        for (int e = 0; e < 4; ++e) at[e] = c0 + e < s.cols ? (s.by_rows ? c0 + e : kept(c0 + e)) : -1;
        float v[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t r = r0 + 4 * i, row = r < s.rows ? (s.by_rows ? kept(r) : r) : -1;
            const float *p = src + (row < 0 ? 0 : row) * s.s_row;
            if (s.vec && row >= 0 && c0 + 3 < s.cols) {
                const float4 q = __ldg(reinterpret_cast<const float4 *>(p + c0));
                v[i][0] = q.x; v[i][1] = q.y; v[i][2] = q.z; v[i][3] = q.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[i][e] = row >= 0 && at[e] >= 0 ? __ldg(p + at[e] * s.s_col) : 0.f;
            }
        }
        const int64_t plane = s.rows * s.ld;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t r = r0 + 4 * i;
            if (r >= s.rows) break;
            __nv_bfloat16 *d = s.dst + b * kPlanes * plane + r * s.ld + c0;
#pragma unroll
            for (int e = 0; e < 4; ++e) odd |= unusual(v[i][e]);
#pragma unroll
            for (int pl = 0; pl < kPlanes; ++pl) {
                uint32_t w[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const __nv_bfloat162 x = __floats2bfloat162_rn(v[i][2 * h], v[i][2 * h + 1]);
                    w[h] = *reinterpret_cast<const uint32_t *>(&x);
                    v[i][2 * h] -= __uint_as_float(w[h] << 16);             // exact
                    v[i][2 * h + 1] -= __uint_as_float(w[h] & 0xffff0000u);
                }
                *reinterpret_cast<uint2 *>(d + pl * plane) = make_uint2(w[0], w[1]);   // rows of dst are whole 16-byte units
            }
        }
    }
    const int any = __syncthreads_or(odd);
    if (threadIdx.x == 0) a.flags[blockIdx.y * gridDim.x + blockIdx.x] = any;
}

struct SplitGemmArgs {
    int64_t M, N, k;
    int64_t y_sb, y_sr, y_sc;
    void *Y;
    int y_bf16, y_vec, tiles_m, tiles_n;
    int64_t tiles, cut_first, seg_kb;   // tiles from cut_first on: their k-blocks form one axis, cut into shares of seg_kb per CTA pair
    float scale;
    float4 *partials;     // [2 x CTAs][32][128]: the sums of a CTA's first and last tile where those are cut, rows of four columns
    unsigned *counters;   // [CTAs]
    SplitFlags f;
    int n_flags;          // of all batch elements
    int cost_a, cost_b;   // tiles of the FMA kernel that a flag of a block of A or B stands for
    int64_t most_lost;    // from more than these on that kernel does everything
    int *status;
    unsigned long long wait_ns;
    int withhold;
};

template <bool B_KMAJOR>
__global__ void __launch_bounds__(kSplitThreads, 1)
split_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const SplitGemmArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_last;
    __shared__ unsigned long long s_lost;
    const uint32_t rank = cluster_rank();
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
    auto full_bar = [&](int s) { return base + kOffBars + 8u * s; };
    auto empty_bar = [&](int s) { return base + kOffBars + 24u + 8u * s; };
    auto tfull_bar = [&](int i) { return base + kOffBars + 48u + 8u * i; };
    auto tempty_bar = [&](int i) { return base + kOffBars + 64u + 8u * i; };
    const uint32_t epi_bar = base + kOffBars + 96u;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + kOffBars + 80);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + kOffBars + 88);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull_bar(i), 1); mbar_init(tempty_bar(i), 16); }
        mbar_init(epi_bar, 8);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc<2>(smem_u32(const_cast<uint32_t *>(tmem_slot)), 2 * kTile);
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();

    // Elements that cannot be split: the FMA kernel behind does the outputs that see them, or everything if those are too many (the
    // verdict is the same in every CTA).
    if (tid == 0) s_lost = 0;
    __syncthreads();
    {
        unsigned long long lost = 0;
        for (int i = tid; i < a.n_flags; i += kSplitThreads)
            if (__ldg(a.f.flags + i) != 0) lost += i % a.f.per_batch < a.f.a_blocks ? a.cost_a : a.cost_b;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) lost += __shfl_xor_sync(0xffffffffu, lost, d);
        if (lane == 0 && lost > 0) atomicAdd(&s_lost, lost);
    }
    __syncthreads();
    const bool run = s_lost <= (unsigned long long)a.most_lost;
    if (blockIdx.x == 0 && tid == 0) *a.f.verdict = run ? (s_lost > 0 ? 1 : 0) : 2;

    const int num_kb = (int)((a.k + kBk - 1) / kBk);
    // The n-th piece of work of this pair: k-blocks [kb0, kb1) of a tile.  Whole tiles round robin, then the pair's share of the rest,
    // of whose tiles only the first and the last are cut.
    const int64_t unit = blockIdx.x / 2, pairs = gridDim.x / 2, full_rounds = a.cut_first / pairs;
    auto piece = [&](int64_t n, int64_t &tile, int &kb0, int &kb1) -> bool {
        if (!run) return false;
        if (n < full_rounds || a.seg_kb == 0) {
            tile = unit + n * pairs;
            kb0 = 0;
            kb1 = num_kb;
            return tile < a.tiles;
        }
        const int64_t begin = unit * a.seg_kb, end = min((a.tiles - a.cut_first) * num_kb, begin + a.seg_kb);
        const int64_t pos = n == full_rounds ? begin : (begin / num_kb + (n - full_rounds)) * num_kb;
        if (pos >= end) return false;
        tile = pos / num_kb;
        kb0 = (int)(pos - tile * num_kb);
        kb1 = (int)min((int64_t)num_kb, kb0 + (end - pos));
        tile += a.cut_first;
        return true;
    };
    auto place = [&](int64_t tile, int &b, int &tm, int &tn) {
        tn = (int)(tile % a.tiles_n);
        tm = (int)(tile / a.tiles_n % a.tiles_m);
        b = (int)(tile / a.tiles_n / a.tiles_m);
    };
    int64_t tile;
    int kb0, kb1;
    bool ok = true;
    uint32_t it = 0;   // k-blocks so far
    if (warp == 0) {
        if (lane == 0) {
            for (int64_t n = 0; ok && piece(n, tile, kb0, kb1); ++n) {
                int b, tm, tn;
                place(tile, b, tm, tn);
                const int row_a = (tm * 2 + (int)rank) * kTile, col_b = tn * kTile + (int)rank * (kTile / 2);
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const uint32_t s = it % kStages;
                    if (!mbar_wait_sleepy(empty_bar(s), (it / kStages & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                    if (a.withhold && blockIdx.x == 0 && it == 0) continue;  // (test switch) never requested
                    // both CTAs report their bytes to the leader's barrier; the leader arms it for the pair
                    const uint32_t lead_full = map_to_cta(full_bar(s), 0), dst = base + s * kStageBytes;
                    if (rank == 0) mbar_arrive_expect_tx(full_bar(s), 2 * kStageBytes);
#pragma unroll
                    for (int pl = 0; pl < kPlanes; ++pl) {
                        tma_load_3d_pair(dst + pl * kPlaneA, &map_a, kb * kBk, row_a, b * kPlanes + pl, lead_full);
                        // K-major: 64 columns of 64 indices; else 64 indices (rows) of 64 columns
                        tma_load_3d_pair(dst + kPlanes * kPlaneA + pl * kPlaneB, &map_b, B_KMAJOR ? kb * kBk : col_b, B_KMAJOR ? col_b : kb * kBk,
                                         b * kPlanes + pl, lead_full);
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((B_KMAJOR ? 0u : 1u) << 16) | ((uint32_t)(kTile >> 3) << 17) |
                                   ((uint32_t)(2 * kTile >> 4) << 24);
        const uint64_t da0 = smem_desc(base, 16, 1024);
        const uint64_t db0 = B_KMAJOR ? smem_desc(base + kPlanes * kPlaneA, 16, 1024) : smem_desc(base + kPlanes * kPlaneA, kBk * 128, 1024);
        const uint32_t a_hi = (uint32_t)(da0 >> 32), b_hi = (uint32_t)(db0 >> 32);
        constexpr uint32_t kAStep = 32 >> 4, kBStep = (B_KMAJOR ? 32 : 2048) >> 4;
        // the smallest products first: what the accumulator drops is relative to what it holds
        constexpr uint32_t pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
        // The warp stays together and one elected lane issues: descriptors then live in uniform registers.  (A lane on its own took
        // about 125 clocks an instruction, twice what the tensor cores need for it.)
        for (int64_t n = 0; rank == 0 && ok && piece(n, tile, kb0, kb1); ++n)
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const uint32_t s = it % kStages, buf = it & 1u;
            if (!mbar_wait(tempty_bar(buf), (it >> 1 & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
            if (!mbar_wait(full_bar(s), it / kStages & 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
            tc_fence_after();
            const uint32_t al = (uint32_t)da0 + s * (kStageBytes >> 4), bl = (uint32_t)db0 + s * (kStageBytes >> 4), d = tmem_base + buf * kTile;
            const int steps = (int)min((int64_t)(kBk / 16), (a.k - (int64_t)kb * kBk + 15) / 16);
            if (elect_one()) {
                if (steps == kBk / 16) {
#pragma unroll
                    for (int p = 0; p < 6; ++p)
#pragma unroll
                        for (int st = 0; st < kBk / 16; ++st)
                            umma_bf16_lohi<2>(d, al + pa[p] * (kPlaneA >> 4) + st * kAStep, a_hi, bl + pb[p] * (kPlaneB >> 4) + st * kBStep, b_hi, idesc,
                                              p + st > 0 ? 1u : 0u);
                } else {
#pragma unroll 1
                    for (int p = 0; p < 6; ++p)
#pragma unroll 1
                        for (int st = 0; st < steps; ++st)
                            umma_bf16_lohi<2>(d, al + pa[p] * (kPlaneA >> 4) + st * kAStep, a_hi, bl + pb[p] * (kPlaneB >> 4) + st * kBStep, b_hi, idesc,
                                              p + st > 0 ? 1u : 0u);
                }
                umma_commit<2>(empty_bar(s));
                umma_commit<2>(tfull_bar(buf));
            }
            __syncwarp();
        }
        __syncwarp();
    } else if (warp >= 4) {
        const int q = warp & 3, half = (warp - 4) >> 2, row = q * 32 + lane;
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + half * 64;
        uint32_t meets = 0;
        auto epilogue_meet = [&]() -> bool {   // warps 4-11; bounded like every wait
            __syncwarp();
            if (lane == 0) mbar_arrive(epi_bar);
            return mbar_wait(epi_bar, meets++ & 1u, abort_flag, a.status, a.wait_ns);
        };
        for (int64_t n = 0; ok && piece(n, tile, kb0, kb1); ++n) {
            float2 acc[32];  // this thread's row, 64 columns
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = make_float2(0.f, 0.f);
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                const uint32_t buf = it & 1u;
                if (!mbar_wait(tfull_bar(buf), it >> 1 & 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                tc_fence_after();
                uint32_t r0[32], r1[32];
                tmem_ld32_issue(t_row + buf * kTile, r0);
                tmem_ld32_issue(t_row + buf * kTile + 32, r1);
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_cta(tempty_bar(buf), 0));  // the leader's tensor-core warp waits on it
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    acc[i].x += __uint_as_float(r0[2 * i]);
                    acc[i].y += __uint_as_float(r0[2 * i + 1]);
                    acc[16 + i].x += __uint_as_float(r1[2 * i]);
                    acc[16 + i].y += __uint_as_float(r1[2 * i + 1]);
                }
            }
            if (!ok) break;
            if (kb1 - kb0 < num_kb) {
                // a cut tile: its pieces, of pairs u0 .. u1, meet in whichever comes last and are added in order
                const int64_t t = tile - a.cut_first, u0 = t * num_kb / a.seg_kb, u1 = ((t + 1) * num_kb - 1) / a.seg_kb;
                auto slot = [&](int64_t u) -> float4 * {   // only a tile's first pair can hold it as its last piece
                    return a.partials + ((2 * (2 * u + (u == u0 && u0 * a.seg_kb < t * num_kb ? 1 : 0)) + rank) * 32 + half * 16) * kTile + row;
                };
                float4 *mine = slot(unit);
#pragma unroll
                for (int c = 0; c < 16; ++c) __stcg(mine + c * kTile, make_float4(acc[2 * c].x, acc[2 * c].y, acc[2 * c + 1].x, acc[2 * c + 1].y));
                if (!epilogue_meet()) { ok = false; break; }
                if (tid == 128) {  // (fences are cumulative: one thread's stand for all that it has met)
                    __threadfence();
                    s_last = atomicInc(a.counters + 2 * u0 + rank, (unsigned)(u1 - u0)) == (unsigned)(u1 - u0);
                    __threadfence();
                }
                if (!epilogue_meet()) { ok = false; break; }
                const bool last = *const_cast<volatile int *>(&s_last) != 0;
                if (!epilogue_meet()) { ok = false; break; }   // (s_last is written again for the next cut tile)
                if (!last) continue;
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] = make_float2(0.f, 0.f);
                for (int64_t u = u0; u <= u1; ++u) {
                    const float4 *src = slot(u);
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const float4 w = __ldcg(src + c * kTile);
                        acc[2 * c].x += w.x; acc[2 * c].y += w.y; acc[2 * c + 1].x += w.z; acc[2 * c + 1].y += w.w;
                    }
                }
            }
            int b, tm, tn;
            place(tile, b, tm, tn);
            const int64_t m = ((int64_t)tm * 2 + rank) * kTile + row, n0 = (int64_t)tn * kTile + half * 64;
            if (m >= a.M) continue;
            const int64_t off = b * a.y_sb + m * a.y_sr + n0 * a.y_sc;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const float y[4] = {acc[2 * c].x * a.scale, acc[2 * c].y * a.scale, acc[2 * c + 1].x * a.scale, acc[2 * c + 1].y * a.scale};
                if (a.y_vec && n0 + 4 * c + 3 < a.N) {
                    *reinterpret_cast<float4 *>(static_cast<float *>(a.Y) + off + 4 * c) = make_float4(y[0], y[1], y[2], y[3]);
                    continue;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (n0 + 4 * c + e >= a.N) break;
                    const int64_t o = off + (4 * c + e) * a.y_sc;
                    if (a.y_bf16) static_cast<__nv_bfloat16 *>(a.Y)[o] = __float2bfloat16_rn(y[e]);
                    else static_cast<float *>(a.Y)[o] = y[e];
                }
            }
        }
    }
    __syncthreads();
    if (*abort_flag != 0) drain_copies();
    __syncthreads();
    tc_fence_before();
    cluster_sync_all();  // the peer may still be reading operands or accumulators that involve this CTA
    tc_fence_after();
    if (warp == 1) tmem_dealloc<2>(tmem_base, 2 * kTile);
}

}  // namespace

// The layout of one panel: batch x rows of A times batch x cols columns of B.
// Whole tiles round robin over the CTA pairs; a last round (or an only one) of few tiles is cut into one equal share per pair, where
// that saves more than the meeting of the pieces costs.  (Cutting everything instead took 476 us for 440 on 2048 x 4096 kept x
// 4096: pairs at different places of the contraction share no operands.)  Estimate in microseconds: 1.2 a k-block, 3 a round, 8
// for cut tiles, and 10 for the launches of the gather and of the idle FMA kernel behind.
static void panel_layout(int64_t batch, int64_t rows, int64_t cols, int64_t k, SplitPlan *p)
{
    const int64_t num_kb = ceil_div(k, kBk), pairs = sm_count() / 2, tiles = batch * ceil_div(rows, 2 * kTile) * ceil_div(cols, kTile);
    p->batch = batch; p->rows = rows; p->cols = cols;
    p->tiles = p->cut_first = tiles;
    p->seg_kb = 0;
    const int64_t rest = tiles % pairs;
    p->cost = 10.0 + (double)ceil_div(tiles, pairs) * (3.0 + 1.2 * (double)num_kb) + (double)(batch * (rows + cols) * k) * 10.0 / 5.0e6;  // the gather: four bytes read, six written
    const double saved = (1.0 - (double)rest / (double)pairs) * 1.2 * (double)num_kb - 8.0;
    if (rest > 0 && saved > 0.0) {
        p->cut_first = tiles - rest;
        p->seg_kb = ceil_div(rest * num_kb, pairs);
        if (p->seg_kb < 2) p->seg_kb = 2;
        p->cost -= saved;
    }
    p->lda = ceil_div(k, 8) * 8;
    p->ldb = p->b_kmajor ? p->lda : ceil_div(cols, 8) * 8;
    const int64_t b_rows = p->b_kmajor ? cols : k;
    p->a_blocks = ceil_div(rows, kGatherRows) * ceil_div(p->lda, kGatherCols);
    p->gather_blocks = p->a_blocks + ceil_div(b_rows, kGatherRows) * ceil_div(p->ldb, kGatherCols);
    size_t off = RMM_WS_HEADER_BYTES;
    p->off_a = off; off += align_up((size_t)batch * kPlanes * rows * p->lda * 2, 256);
    p->off_b = off; off += align_up((size_t)batch * kPlanes * b_rows * p->ldb * 2, 256);
    p->off_partials = off; off += (size_t)(2 * pairs) * 2 * kTile * kTile * 4;
    p->off_flags = off; off += align_up((size_t)(p->gather_blocks * batch + 1) * 4, 256);   // and the verdict
    p->total_bytes = off;
}

// The parts take six bytes an element of the kept operands, beside a user's own memory: products whose operands are larger than
// kSplitParts allows run in panels (of batch elements, then of rows and columns), one after the other in the same scratch.  The
// panels follow from the whole operands, not from the kept count, so that a workspace for more kept indices holds fewer.
// 8192 x 4096 kept x 8192 2888 us a call in one panel, 2830 in four; 16384 x 4096 kept x 8192 5966 and, in eight, 6150 to 6290.
constexpr double kSplitParts = 512.0 * 1024 * 1024;
bool plan_split(const rmm_mat_t *A, const rmm_mat_t *B, int64_t k, SplitPlan *p)
{
    const int64_t M = A->rows, N = B->cols, batch = A->batch;
    if (A->dtype != RMM_F32 || B->dtype != RMM_F32 || k > A->cols) return false;
    if ((double)batch * (double)M * (double)N * (double)k < 1.5e8) return false;   // 10 us of the FMA kernel
    if (M > INT32_MAX / 2 || N > INT32_MAX / 2 || A->cols > INT32_MAX / 2 || batch > 65535 / kPlanes || ceil_div(M, 64) > 65535) return false;
    int64_t nb = batch, rows = M, cols = N;
    while ((double)nb * (double)(rows + cols) * (double)A->cols * 2.0 * kPlanes > kSplitParts) {
        if (nb > 1) nb = ceil_div(nb, 2);
        else if (rows >= cols && rows > 2 * kTile) rows = ceil_div(rows, 4 * kTile) * 2 * kTile;
        else if (cols > 2 * kTile) cols = ceil_div(cols, 4 * kTile) * 2 * kTile;
        else return false;
    }
    p->b_kmajor = B->stride_col != 1 && B->stride_row == 1;
    panel_layout(nb, rows, cols, k, p);
    p->cost *= (double)(ceil_div(batch, nb) * ceil_div(M, rows) * ceil_div(N, cols));
    return true;
}

static SplitFlags split_flags(const rmm_mat_t *A, const rmm_mat_t *B, int64_t k, const SplitPlan &p, void *ws)
{
    SplitFlags f;
    f.flags = reinterpret_cast<const int *>(static_cast<char *>(ws) + p.off_flags);
    f.per_batch = (int)p.gather_blocks;
    f.verdict = const_cast<int *>(f.flags) + p.gather_blocks * A->batch;
    f.a_blocks = (int)p.a_blocks;
    f.a_cols = (int)ceil_div(p.lda, kGatherCols);
    f.b_rows = (int)ceil_div(p.b_kmajor ? B->cols : k, kGatherRows);
    f.b_cols = (int)ceil_div(p.ldb, kGatherCols);
    f.b_kmajor = p.b_kmajor;
    return f;
}

static int launch_panel(const rmm_mat_t *A, const rmm_mat_t *B, const int32_t *idx, int64_t k, float scale, const rmm_mat_t *Y, const SplitPlan &p,
                        void *ws, cudaStream_t stream)
{
    char *w = static_cast<char *>(ws);
    WsHeader *h = static_cast<WsHeader *>(ws);
    const int64_t M = A->rows, N = B->cols, batch = A->batch;
    auto al16 = [](const void *q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    __nv_bfloat16 *Ap = reinterpret_cast<__nv_bfloat16 *>(w + p.off_a), *Bp = reinterpret_cast<__nv_bfloat16 *>(w + p.off_b);
    const int64_t b_rows = p.b_kmajor ? N : k;
    SplitArgs g = {};
    auto spec = [&](SplitSpec &s, const rmm_mat_t *X, bool by_rows, int64_t sr, int64_t sc, __nv_bfloat16 *dst, int64_t rows, int64_t cols, int64_t ld) {
        s.src = static_cast<const float *>(X->ptr); s.dst = dst;
        s.s_batch = X->stride_batch; s.s_row = sr; s.s_col = sc;
        s.rows = rows; s.cols = cols; s.ld = ld; s.by_rows = by_rows;
        // four columns at once only where they lie next to each other: rows picked by the list, or no list at all
        s.vec = (by_rows || idx == nullptr) && sc == 1 && sr % 4 == 0 && (batch == 1 || s.s_batch % 4 == 0) && al16(s.src);
        s.blocks_r = (unsigned)ceil_div(rows, kGatherRows); s.blocks_c = (unsigned)ceil_div(ld, kGatherCols);
    };
    spec(g.s[0], A, false, A->stride_row, A->stride_col, Ap, M, k, p.lda);
    if (p.b_kmajor) spec(g.s[1], B, false, B->stride_col, B->stride_row, Bp, N, k, p.ldb);
    else spec(g.s[1], B, true, B->stride_row, B->stride_col, Bp, k, N, p.ldb);
    g.idx = idx; g.k = k; g.K = A->cols;
    g.status = &h->status; g.flags = reinterpret_cast<int *>(w + p.off_flags);
    prof_begin("split_gather_kernel", stream);
    cudaError_t e = launch_kernel(split_gather_kernel, dim3((unsigned)p.gather_blocks, (unsigned)batch), dim3(kGatherThreads), 0, stream, 1, g);
    if (e != cudaSuccess) return fail(RMM_ERR_CUDA, "split_gather_kernel: launch: %s", cudaGetErrorString(e));
    int rc = check_launch("split_gather_kernel", stream);
    if (rc != RMM_OK) return rc;

    CUtensorMap ma, mb;
    {
        const uint64_t dims[3] = {(uint64_t)k, (uint64_t)M, (uint64_t)(kPlanes * batch)}, st[2] = {(uint64_t)p.lda * 2, (uint64_t)(M * p.lda) * 2};
        const uint32_t box[3] = {kBk, kTile, 1};
        if ((rc = make_map(&ma, Ap, 3, dims, st, box, true)) != RMM_OK) return rc;
    }
    {
        const uint64_t dims[3] = {(uint64_t)(p.b_kmajor ? k : N), (uint64_t)b_rows, (uint64_t)(kPlanes * batch)},
                       st[2] = {(uint64_t)p.ldb * 2, (uint64_t)(b_rows * p.ldb) * 2};
        const uint32_t box[3] = {64, 64, 1};
        if ((rc = make_map(&mb, Bp, 3, dims, st, box, true)) != RMM_OK) return rc;
    }
    SplitGemmArgs a = {};
    a.M = M; a.N = N; a.k = k;
    a.Y = Y->ptr; a.y_sb = Y->stride_batch; a.y_sr = Y->stride_row; a.y_sc = Y->stride_col;
    a.y_bf16 = Y->dtype == RMM_BF16;
    a.y_vec = !a.y_bf16 && a.y_sc == 1 && a.y_sr % 4 == 0 && a.y_sb % 4 == 0 && al16(a.Y);
    a.tiles_m = (int)ceil_div(M, 2 * kTile); a.tiles_n = (int)ceil_div(N, kTile);
    a.tiles = p.tiles; a.cut_first = p.cut_first; a.seg_kb = p.seg_kb;
    const int64_t pairs = sm_count() / 2;
    a.scale = scale;
    a.partials = reinterpret_cast<float4 *>(w + p.off_partials);
    a.counters = h->counters;
    a.f = split_flags(A, B, k, p, ws);
    a.n_flags = (int)(p.gather_blocks * batch);
    // (64 x 128 tiles; a block of A has 16 rows, one of B 16 or 256 columns)
    a.cost_a = (int)ceil_div(N, 128); a.cost_b = (int)ceil_div(M, 64) * (p.b_kmajor ? 1 : 2);
    // A few tiles take the FMA kernel as long as its slowest block does, on an SM with two others: only products of several rounds of
    // its blocks gain by leaving the rest to the tensor cores, and not from half of the tiles on.  (One element of 1e-20: 2048 x
    // 4096 kept x 4096 1552 us -> 1064, 8192 x 4096 x 8192 11460 -> 4441; 777 x 1500 x 1500 would take 139 for 127.)
    double tile_us;
    const double fma_us = gemm_simt_cost(A, B, k, &tile_us);
    a.most_lost = p.cost + tile_us < fma_us ? batch * ceil_div(M, 64) * ceil_div(N, 128) / 2 : 0;
    a.status = &h->status;
    a.wait_ns = wait_limit_ns();
    a.withhold = debug_withhold() == WITHHOLD_GEMM;
    auto kern = p.b_kmajor ? split_gemm_kernel<true> : split_gemm_kernel<false>;
    static PerDeviceOnce configured;
    if ((e = configured.smem(kSplitSmem, split_gemm_kernel<true>, split_gemm_kernel<false>)) != cudaSuccess)
        return fail(RMM_ERR_CUDA, "split_gemm_kernel: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    prof_begin("split_gemm_kernel", stream);
    e = launch_kernel(kern, dim3(2 * (unsigned)(p.tiles < pairs && p.seg_kb == 0 ? p.tiles : pairs)), dim3(kSplitThreads), kSplitSmem, stream, 2, ma, mb, a);
    if (e != cudaSuccess) return fail(RMM_ERR_CUDA, "split_gemm_kernel: launch: %s", cudaGetErrorString(e));
    return check_launch("split_gemm_kernel", stream);
}

int launch_split_gemm(const rmm_mat_t *A, const rmm_mat_t *B, const int32_t *idx, int64_t k, float scale, const rmm_mat_t *Y, const SplitPlan &plan,
                      void *ws, cudaStream_t stream)
{
    const auto at = [](const rmm_mat_t *X, int64_t b, int64_t r, int64_t c) -> void * {
        const int64_t e = b * X->stride_batch + r * X->stride_row + c * X->stride_col;
        return static_cast<char *>(X->ptr) + e * (int64_t)dtype_size(X->dtype);
    };
    for (int64_t b = 0; b < A->batch; b += plan.batch)
        for (int64_t c = 0; c < B->cols; c += plan.cols)
            for (int64_t r = 0; r < A->rows; r += plan.rows) {
                const int64_t nb = A->batch - b < plan.batch ? A->batch - b : plan.batch, rows = A->rows - r < plan.rows ? A->rows - r : plan.rows,
                              cols = B->cols - c < plan.cols ? B->cols - c : plan.cols;
                SplitPlan p = plan;
                panel_layout(nb, rows, cols, k, &p);
                rmm_mat_t pa = *A, pb = *B, py = *Y;
                pa.ptr = at(A, b, r, 0); pb.ptr = at(B, b, 0, c); py.ptr = at(Y, b, r, c);
                pa.batch = pb.batch = py.batch = nb; pa.rows = py.rows = rows; pb.cols = py.cols = cols;
                const int32_t *list = idx != nullptr ? idx + b * k : nullptr;
                int rc = launch_panel(&pa, &pb, list, k, scale, &py, p, ws, stream);
                if (rc != RMM_OK) return rc;
                // elements that cannot be split: the FMA kernel does the outputs that see them (its scratch ends before the flags)
                const SplitFlags left = split_flags(&pa, &pb, k, p, ws);
                rc = launch_gemm_simt(&pa, &pb, list, k, scale, &py, ws, p.off_flags, stream, &left);
                if (rc != RMM_OK) return rc;
            }
    return RMM_OK;
}

}  // namespace rmm
