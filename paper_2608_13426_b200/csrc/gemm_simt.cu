// Reduced product Y = scale * A[:, I] B[I, :] (paper Sec. 3.2) on the plain FMA pipes.
//
// This kernel covers what the tensor-core paths do not: fp32 operands that are too small a product for gemm_split.cu, or whose
// elements cannot be split there, and bf16 operands with strides or alignments outside the TMA rules.  Any element strides
// are accepted.
//
// Bound: FMA issue.  A block of 128 threads owns a tile of 8 TM x 128 outputs and a thread TM x 8 of them, held as
// pairs of columns for the packed fp32 FMA (one instruction, two FMAs; with single FMAs the same kernel took 480 us
// where this takes 380): per contraction index a thread reads TM + 8 floats from shared memory for 8 TM FMAs, one index
// ahead.  16 indices per step; fp32 elements are gathered by cp.async into a ring of three steps, bf16 ones pass through
// registers; index lists are loaded a step before they are used.  Small blocks, so that several share an SM (vectorised fp32:
// three of 64 rows, five of 32; the registers of the other variants allow two of 64 rows, and in bf16 four of 32) and none
// of them waits at another's barrier.  fp32 accumulation with one partial sum per step of 16, so that rounding error grows
// with k/16 rather than k.  Outputs with fewer tiles than the GPU has room for cut the contraction axis (plan_simt): the
// slices of a tile meet in its last block, which adds them in order.
// fp32, kernel alone: 777 x 1500 kept x 1500 379 -> 119 us, 2048 x 4096 x 4096 5530 -> 1490 us (46 of the 65 TFLOP/s that
// a register-only FMA loop reaches on this GPU) against 64 x 64 tiles of 4 x 4 outputs a thread.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

constexpr int BN = 128, BK = 16, THREADS = 128, kHi = THREADS / 16, kRing = 3;

struct SimtArgs {
    const void *A, *B;
    void *Y;
    const int32_t *idx;
    int64_t M, N, K, k;
    int64_t a_sb, a_sr, a_sc, b_sb, b_sr, b_sc, y_sb, y_sr, y_sc;
    float scale;
    int *status;
    int splits, y_bf16, y_vec;
    int64_t k_split;      // contraction indices per slice (a multiple of BK)
    float4 *partials;     // [tile][slice][TM * 2][THREADS]
    unsigned *counters;   // one per tile
    SplitFlags left;      // BEHIND
};

template <bool BF16>
__device__ __forceinline__ float load_elem(const void *p, int64_t off)
{
    if constexpr (BF16)
        return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(p)[off]);
    else
        return __ldg(reinterpret_cast<const float *>(p) + off);
}

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src, bool live)  // zeros where not live
{
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(live ? 4 : 0) : "memory");
}

// VEC: rows of B are contiguous, 16-byte aligned fp32 and N is a multiple of 4
// BEHIND: only what the split product left over (a form of its own: with the look at the flags in every call, small fp32 products
// took 1 to 2 % longer, 40 x 2376 x 2553 39.7 -> 40.4 us)
template <int TM, bool IN_BF16, bool VEC, bool BEHIND>
__global__ void __launch_bounds__(THREADS) reduced_gemm_simt_kernel(const SimtArgs a)
{
    constexpr int BM = kHi * TM, PA = BM + 4, PB = BN + 4;  // pitches: rows stay 16-byte aligned
    __shared__ __align__(16) float sA[kRing][BK][PA];
    __shared__ __align__(16) float sB[kRing][BK][PB];
    __shared__ int s_last;
    pdl_wait();
    const int tid = threadIdx.x;
    const int64_t b = blockIdx.z / a.splits, slice = blockIdx.z % a.splits;
    const int64_t m0 = (int64_t)blockIdx.y * BM, n0 = (int64_t)blockIdx.x * BN;
    if constexpr (BEHIND) {
        const SplitFlags &f = a.left;
        const int verdict = __ldg(f.verdict);
        if (verdict == 0) return;
        if (verdict == 1) {   // (all slices of a tile find the same)
            const int *fa = f.flags + b * f.per_batch, *fb = fa + f.a_blocks;
            const int a_end = (int)min((int64_t)f.a_blocks, (m0 + BM) / 16 * f.a_cols);
            int set = 0;
            for (int i = (int)(m0 / 16) * f.a_cols + tid; i < a_end; i += THREADS) set |= __ldg(fa + i);
            if (f.b_kmajor) {
                const int b_end = (int)min((int64_t)f.b_rows, (n0 + BN) / 16) * f.b_cols;
                for (int i = (int)(n0 / 16) * f.b_cols + tid; i < b_end; i += THREADS) set |= __ldg(fb + i);
            } else {
                for (int r = tid; r < f.b_rows; r += THREADS) set |= __ldg(fb + r * f.b_cols + n0 / 256);
            }
            if (!__syncthreads_or(set)) return;
        }
    }
    const int64_t k_begin = slice * a.k_split, k_end = min(a.k, k_begin + a.k_split);
    const int hi = tid / 16, lo = tid % 16;   // compute: row group hi, column group lo
    const int32_t *idx = a.idx != nullptr ? a.idx + b * a.k : nullptr;
    const int64_t a0 = b * a.a_sb + m0 * a.a_sr, b0 = b * a.b_sb + n0 * a.b_sc;

    // the kept index at position kk + at (-1 past the end), not looked at before it is used a step later
    auto index_at = [&](int64_t kk, int at) -> int {
        if (kk + at >= k_end) return -1;
        return idx != nullptr ? __ldg(idx + kk + at) : (int)(kk + at);
    };
    auto bounded = [&](int64_t kk, int at, int j) -> bool {  // a bad index is reported and reads nothing
        if (kk + at < k_end && (j < 0 || j >= a.K)) atomicExch(a.status, (int)RMM_ERR_BOUNDS);
        return j >= 0 && j < a.K;
    };
    // loads: A by (index lo, rows hi + 16 i), neighbouring threads take neighbouring kept columns; B by (index hi, columns)
    constexpr int RB = BK / kHi;  // rows of B per thread
    float ra[BM / kHi], rb[RB][8];
    auto fetch = [&](int64_t kk, int ja, const int (&jb)[RB]) {
        const int64_t ac = (int64_t)ja * a.a_sc;
        const bool a_ok = bounded(kk, lo, ja);
#pragma unroll
        for (int i = 0; i < TM; ++i)
            ra[i] = a_ok && m0 + hi + kHi * i < a.M ? load_elem<IN_BF16>(a.A, a0 + (hi + kHi * i) * a.a_sr + ac) : 0.f;
#pragma unroll
        for (int w = 0; w < RB; ++w) {
            const int64_t br = b0 + (int64_t)jb[w] * a.b_sr;
            const bool b_ok = bounded(kk, hi + kHi * w, jb[w]);
            if constexpr (VEC) {
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int n = lo * 4 + 64 * v;
                    const float4 q = b_ok && n0 + n < a.N ? __ldg(reinterpret_cast<const float4 *>(static_cast<const float *>(a.B) + br + n))
                                                                : make_float4(0.f, 0.f, 0.f, 0.f);
                    rb[w][4 * v] = q.x; rb[w][4 * v + 1] = q.y; rb[w][4 * v + 2] = q.z; rb[w][4 * v + 3] = q.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    rb[w][i] = b_ok && n0 + lo + 16 * i < a.N ? load_elem<IN_BF16>(a.B, br + (lo + 16 * i) * a.b_sc) : 0.f;
            }
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int i = 0; i < TM; ++i) sA[buf][lo][hi + kHi * i] = ra[i];
#pragma unroll
        for (int w = 0; w < RB; ++w) {
            float *row = sB[buf][hi + kHi * w];
            if constexpr (VEC) {
#pragma unroll
                for (int v = 0; v < 2; ++v)
                    *reinterpret_cast<float4 *>(row + lo * 4 + 64 * v) = make_float4(rb[w][4 * v], rb[w][4 * v + 1], rb[w][4 * v + 2], rb[w][4 * v + 3]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) row[lo + 16 * i] = rb[w][i];
            }
        }
    };
    // fp32: the same elements straight to shared memory
    auto issue = [&](int64_t kk, int ja, const int (&jb)[RB], int buf) {
        if constexpr (!IN_BF16) {
            if (kk < k_end) {
                const bool a_ok = bounded(kk, lo, ja);
                const float *A = static_cast<const float *>(a.A), *B = static_cast<const float *>(a.B);
                const int64_t ac = a0 + (int64_t)ja * a.a_sc;
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const bool ok = a_ok && m0 + hi + kHi * i < a.M;
                    cp_async<4>(ptx::smem_u32(&sA[buf][lo][hi + kHi * i]), ok ? A + ac + (hi + kHi * i) * a.a_sr : A, ok);
                }
#pragma unroll
                for (int w = 0; w < RB; ++w) {
                    const int64_t br = b0 + (int64_t)jb[w] * a.b_sr;
                    const bool b_ok = bounded(kk, hi + kHi * w, jb[w]);
                    const uint32_t row = ptx::smem_u32(sB[buf][hi + kHi * w]);
                    if constexpr (VEC) {
#pragma unroll
                        for (int v = 0; v < 2; ++v) {
                            const int n = lo * 4 + 64 * v;
                            const bool ok = b_ok && n0 + n < a.N;
                            cp_async<16>(row + n * 4, ok ? B + br + n : B, ok);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const bool ok = b_ok && n0 + lo + 16 * i < a.N;
                            cp_async<4>(row + (lo + 16 * i) * 4, ok ? B + br + (lo + 16 * i) * a.b_sc : B, ok);
                        }
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    };
    // this thread's outputs: rows row_of(i), columns lo * 4 + 64 (p / 2) + 2 (p % 2) + {0, 1} for pair p
    auto row_of = [&](int i) { return hi * 4 + (i & 3) + kHi * 4 * (i >> 2); };

    uint64_t acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[i][p] = 0;

    int ja, jb[RB], buf = 0;
    auto indices = [&](int64_t kk) {
        ja = index_at(kk, lo);
#pragma unroll
        for (int w = 0; w < RB; ++w) jb[w] = index_at(kk, hi + kHi * w);
    };
    indices(k_begin);
    if constexpr (IN_BF16) {
        fetch(k_begin, ja, jb);
        store(0);
        indices(k_begin + BK);
    } else {
        issue(k_begin, ja, jb, 0);
        indices(k_begin + BK);
        issue(k_begin + BK, ja, jb, 1);
        indices(k_begin + 2 * BK);
    }
    for (int64_t kk = k_begin; kk < k_end; kk += BK, buf = buf + 1 < kRing ? buf + 1 : 0) {
        // after the barrier this step's tile is complete, and nobody reads the tile before it any more
        if constexpr (IN_BF16) {
            __syncthreads();
            fetch(kk + BK, ja, jb);
            indices(kk + 2 * BK);
        } else {
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
            __syncthreads();
            issue(kk + 2 * BK, ja, jb, buf + 2 < kRing ? buf + 2 : buf + 2 - kRing);
            indices(kk + 3 * BK);
        }
        uint64_t part[TM][4];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int p = 0; p < 4; ++p) part[i][p] = 0;
        float av[2][TM];
        uint64_t bv[2][4];
        auto operands = [&](int r) {  // of contraction index r, one ahead of the multiplications
#pragma unroll
            for (int v = 0; v < TM / 4; ++v) {
                const float4 q = *reinterpret_cast<const float4 *>(&sA[buf][r][hi * 4 + kHi * 4 * v]);
                av[r & 1][4 * v] = q.x; av[r & 1][4 * v + 1] = q.y; av[r & 1][4 * v + 2] = q.z; av[r & 1][4 * v + 3] = q.w;
            }
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(&sB[buf][r][lo * 4 + 64 * v]);
                bv[r & 1][2 * v] = q.x; bv[r & 1][2 * v + 1] = q.y;
            }
        };
        operands(0);
#pragma unroll
        for (int r = 0; r < BK; ++r) {
            if (r + 1 < BK) operands(r + 1);
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const uint64_t aa = ptx::pack2(av[r & 1][i], av[r & 1][i]);
#pragma unroll
                for (int p = 0; p < 4; ++p) part[i][p] = ptx::ffma2(aa, bv[r & 1][p], part[i][p]);
            }
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[i][p] = ptx::fadd2(acc[i][p], part[i][p]);
        if constexpr (IN_BF16) {
            if (kk + BK < k_end) store(buf + 1 < kRing ? buf + 1 : 0);
        }
    }

    float v[TM][8];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int p = 0; p < 4; ++p) ptx::unpack2(acc[i][p], v[i][2 * p], v[i][2 * p + 1]);
    if (a.splits > 1) {
        const int64_t tile = (b * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        float4 *mine = a.partials + tile * a.splits * (TM * 2) * THREADS + tid;
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q)
                __stcg(mine + (slice * TM * 2 + i * 2 + q) * THREADS, make_float4(v[i][4 * q], v[i][4 * q + 1], v[i][4 * q + 2], v[i][4 * q + 3]));
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicInc(a.counters + tile, (unsigned)a.splits - 1u) == (unsigned)a.splits - 1u;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int e = 0; e < 8; ++e) v[i][e] = 0.f;
        for (int s = 0; s < a.splits; ++s) {  // in slice order
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float4 w = __ldcg(mine + ((int64_t)s * TM * 2 + i * 2 + q) * THREADS);
                    v[i][4 * q] += w.x; v[i][4 * q + 1] += w.y; v[i][4 * q + 2] += w.z; v[i][4 * q + 3] += w.w;
                }
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int64_t m = m0 + row_of(i);
        if (m >= a.M) continue;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int64_t n = n0 + lo * 4 + 64 * q, off = b * a.y_sb + m * a.y_sr + n * a.y_sc;
            if (a.y_vec && n + 3 < a.N) {
                *reinterpret_cast<float4 *>(static_cast<float *>(a.Y) + off) =
                    make_float4(v[i][4 * q] * a.scale, v[i][4 * q + 1] * a.scale, v[i][4 * q + 2] * a.scale, v[i][4 * q + 3] * a.scale);
                continue;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (n + e >= a.N) break;
                if (a.y_bf16) static_cast<__nv_bfloat16 *>(a.Y)[off + e * a.y_sc] = __float2bfloat16_rn(v[i][4 * q + e] * a.scale);
                else static_cast<float *>(a.Y)[off + e * a.y_sc] = v[i][4 * q + e] * a.scale;
            }
        }
    }
}

constexpr int64_t kMaxSlices = 32, kMinSlice = 4 * BK;

int64_t simt_tiles(const rmm_mat_t *A, const rmm_mat_t *B, int tm) { return A->batch * ceil_div(A->rows, kHi * tm) * ceil_div(B->cols, BN); }
// slices that a product of k indices may be cut into when it has `tiles` tiles: no more blocks than four to an SM, one
// arrival counter per tile, at least four steps a slice
int64_t simt_slices_max(int64_t tiles, int64_t k)
{
    if (tiles > kHeaderCounters - 4) return 1;  // (the last four counters belong to the tensor-core kernel)
    int64_t s = 4 * (int64_t)sm_count() / tiles;
    if (s > kMaxSlices) s = kMaxSlices;
    if (s > ceil_div(k, kMinSlice)) s = ceil_div(k, kMinSlice);
    return s < 1 ? 1 : s;
}

struct SimtPlan {
    int tm, splits;
    int64_t k_split;
};

// Tile height and slices: the least estimated time, in microseconds.  A lone block leaves its SM's schedulers waiting (one
// warp each), so what counts is how many blocks share an SM; a step of 16 indices took about 1.2, 2.4 and 2.7 us for one,
// two and three blocks of 64 rows (three fit), 0.9, 1.9, 2.1, 2.2 and 2.3 us for one to five of 32 rows.  A round of blocks
// costs about 2 us outside its steps, slices another 1.5 for their meeting.  (777 x 1500 kept x 1500: 230 us with one
// slice, 134 with two, 119 with three, which the rule takes; 1500 x 2000 x 700: 231, 169, 120.)  The times are those of the
// vectorised fp32 variant and stand for all: with each variant's own number of blocks in their place, bf16 on 100 x 3000 x
// 1500 took 43 us for 59, but fp32 with B by columns took 634 for 435 on 2048 x 4096 x 1023 (32-row tiles), 864 for 650 on 2048 x
// 2000 x 4094.
// Slices whose partial sums take more than `room` bytes are not considered.
SimtPlan plan_simt(const rmm_mat_t *A, const rmm_mat_t *B, int64_t k, size_t room, double *estimate = nullptr)
{
    static const double step_us[2][5] = {{1.15, 2.4, 2.7}, {0.9, 1.9, 2.1, 2.2, 2.3}};
    SimtPlan best = {8, 1, ceil_div(k, BK) * BK};
    double best_cost = 1e300;
    const int64_t steps = ceil_div(k, BK), sms = sm_count();
    for (int tm = 8; tm >= 4; tm /= 2) {
        if (ceil_div(A->rows, kHi * tm) > 65535) continue;
        const int fit = tm == 8 ? 3 : 5;
        const double *t = step_us[tm == 8 ? 0 : 1];
        const int64_t tiles = simt_tiles(A, B, tm), most = simt_slices_max(tiles, k);
        for (int64_t s = 1; s <= most; ++s) {
            if (s > 1 && (size_t)(tiles * s) * kHi * tm * BN * sizeof(float) > room) break;
            const int64_t per = ceil_div(steps, s), blocks = tiles * ceil_div(steps, per), full = blocks / (sms * fit);
            const int64_t rest = ceil_div(blocks - full * sms * fit, sms);
            const double cost = (double)full * ((double)per * t[fit - 1] + 2.0) + (rest > 0 ? (double)per * t[rest - 1] + 2.0 : 0.0) + (s > 1 ? 1.5 : 0.0);
            if (cost < best_cost) {
                best_cost = cost;
                best = {tm, (int)ceil_div(steps, per), per * BK};
            }
        }
    }
    if (estimate != nullptr) *estimate = best_cost;
    return best;
}

template <int TM>
void launch_tm(const SimtArgs &a, bool in_bf16, bool vec, bool behind, dim3 grid, cudaStream_t stream)
{
    auto kern = reduced_gemm_simt_kernel<TM, true, false, false>;
    if (behind) kern = vec ? reduced_gemm_simt_kernel<TM, false, true, true> : reduced_gemm_simt_kernel<TM, false, false, true>;
    else if (!in_bf16) kern = vec ? reduced_gemm_simt_kernel<TM, false, true, false> : reduced_gemm_simt_kernel<TM, false, false, false>;
    launch_kernel(kern, grid, dim3(THREADS), 0, stream, 1, a);
}

}  // namespace

// Enough for every count of kept indices up to k (the plan for fewer may cut the axis differently).
size_t gemm_simt_workspace_bytes(const rmm_mat_t *A, const rmm_mat_t *B, int64_t k)
{
    size_t most = 0;
    for (int tm = 8; tm >= 4; tm /= 2) {
        const int64_t tiles = simt_tiles(A, B, tm), s = simt_slices_max(tiles, k);
        const size_t need = s > 1 ? (size_t)(tiles * s) * kHi * tm * BN * sizeof(float) : 0;
        if (need > most) most = need;
    }
    return RMM_WS_HEADER_BYTES + most;
}

double gemm_simt_cost(const rmm_mat_t *A, const rmm_mat_t *B, int64_t k, double *tile_us)
{
    double cost;
    const SimtPlan plan = plan_simt(A, B, k, SIZE_MAX, &cost);
    if (tile_us != nullptr) *tile_us = (double)(plan.k_split / BK) * (plan.tm == 8 ? 2.7 : 2.3);
    return cost;
}

int launch_gemm_simt(const rmm_mat_t *A, const rmm_mat_t *B, const int32_t *idx, int64_t k, float scale,
                     const rmm_mat_t *Y, void *ws, size_t ws_bytes, cudaStream_t stream, const SplitFlags *behind)
{
    const SimtPlan plan = plan_simt(A, B, k, ws_bytes - RMM_WS_HEADER_BYTES);
    SimtArgs a = {};
    if (behind != nullptr) a.left = *behind;
    a.A = A->ptr; a.B = B->ptr; a.Y = Y->ptr; a.idx = idx;
    a.M = A->rows; a.K = A->cols; a.N = B->cols; a.k = k;
    a.a_sb = A->stride_batch; a.a_sr = A->stride_row; a.a_sc = A->stride_col;
    a.b_sb = B->stride_batch; a.b_sr = B->stride_row; a.b_sc = B->stride_col;
    a.y_sb = Y->stride_batch; a.y_sr = Y->stride_row; a.y_sc = Y->stride_col;
    a.scale = scale;
    a.status = &reinterpret_cast<WsHeader *>(ws)->status;
    a.splits = plan.splits;
    a.k_split = plan.k_split;
    a.partials = reinterpret_cast<float4 *>(static_cast<char *>(ws) + RMM_WS_HEADER_BYTES);
    a.counters = reinterpret_cast<WsHeader *>(ws)->counters;
    a.y_bf16 = Y->dtype == RMM_BF16;
    auto al16 = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    a.y_vec = !a.y_bf16 && a.y_sc == 1 && a.y_sr % 4 == 0 && a.y_sb % 4 == 0 && al16(a.Y);
    const bool vec = B->dtype == RMM_F32 && a.b_sc == 1 && a.b_sr % 4 == 0 && a.b_sb % 4 == 0 && a.N % 4 == 0 && al16(a.B);
    dim3 grid((unsigned)ceil_div(a.N, BN), (unsigned)ceil_div(a.M, kHi * plan.tm), (unsigned)(A->batch * plan.splits));
    if (A->batch > 65535 || ceil_div(a.M, 64) > 65535)
        return fail(RMM_ERR_UNSUPPORTED, "reduced_gemm (FMA path): batch or M/64 exceeds 65535");
    prof_begin("reduced_gemm_simt_kernel", stream);
    if (plan.tm == 8) launch_tm<8>(a, A->dtype == RMM_BF16, vec, behind != nullptr, grid, stream);
    else launch_tm<4>(a, A->dtype == RMM_BF16, vec, behind != nullptr, grid, stream);
    return check_launch("reduced_gemm_simt_kernel", stream);
}

}  // namespace rmm
