// A whole product Y = scale * A[:, I] B[I, :] of small operands in one launch.
//
// Bound by latency: three launches (scores with selection, gather, product) leave the GPU idle between them and cost the host
// more than the kernels take.  Here every block holds all of A in shared memory, scores it and selects for itself, and
// multiplies it with its own 16 or 32 columns of B, of which it has fetched every row (kept or not) together with A: nothing
// that is read depends on the selection, so there is one memory latency in the call.  Blocks do not communicate.
// The kept columns are never packed: the A fragments of mma.sync are put together from 2-byte shared-memory reads (rows are
// padded by 16 bytes, so that the eight rows of a fragment fall into different banks), and ldmatrix takes the kept rows of B
// wherever they lie.  Positions past k point to a zero column of A and a zero row of B.
#include "common.cuh"
#include "select.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

constexpr int kSmallThreads = 512, kSmallWarps = kSmallThreads / 32;
constexpr int kSmallMinRows = 5, kSmallMaxRows = 64, kSmallMaxK = 2048;
constexpr int kSmallSmemMax = 200 * 1024;   // next to 14 KB of the selection's

struct SmallArgs {
    const __nv_bfloat16 *A, *B;
    int64_t a_sr, b_sr, y_sr;
    void *Y;
    int y_bf16, M, K, N, k;
    float scale;
    int32_t *idx;            // the selection, written by the first block, or
    const int32_t *given;    // ... the caller's list: nothing is scored
    float *retained;         // or NULL: with idx, the kept share of the energies
    int *status;
};

// Dynamic shared memory: A [M][a_pitch bytes] | B [K + 1][2 NB bytes] | column sums [splits][K] fp64 | the list
struct SmallLayout {
    int a_pitch, off_b, off_sum, off_list, total, splits;
};

__host__ __device__ inline SmallLayout small_layout(int M, int K, int NB)
{
    SmallLayout l;
    const int pairs = (K + 1) / 2, rows16 = (M + 15) / 16;
    l.a_pitch = (K * 2 + 15) / 16 * 16 + 16;
    l.splits = pairs >= kSmallThreads ? 1 : (kSmallThreads / pairs < rows16 ? kSmallThreads / pairs : rows16);
    l.off_b = M * l.a_pitch;
    l.off_sum = l.off_b + (K + 1) * NB * 2;
    l.off_list = l.off_sum + l.splits * 2 * pairs * 8;
    l.total = l.off_list + (K + 16) / 8 * 8 * 4;
    const int meet = kSmallWarps * 16 * NB * 4;   // the warps' sums, over the operands
    if (l.total < meet) l.total = meet;
    return l;
}

template <int ITEMS, int NB>
__global__ void __launch_bounds__(kSmallThreads) small_product_kernel(const SmallArgs a)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ sel::SelectSmem s_sel;
    const SmallLayout lay = small_layout(a.M, a.K, NB);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n0 = blockIdx.x * NB;
    unsigned char *s_b = s_dyn + lay.off_b;
    double *s_sum = reinterpret_cast<double *>(s_dyn + lay.off_sum);
    unsigned short *s_list = reinterpret_cast<unsigned short *>(s_dyn + lay.off_list);
    pdl_wait();

    // ---- operands: 16-byte copies, zeros past the last column
    const uint32_t sa_u = ptx::smem_u32(s_dyn), sb_u = ptx::smem_u32(s_b);
    const int a_vecs = lay.a_pitch / 16;
    for (int v = tid; v < a.M * a_vecs; v += kSmallThreads) {
        const int r = v / a_vecs, c = (v - r * a_vecs) * 8, left = a.K - c;
        ptx::cp_async_16(sa_u + v * 16, a.A + r * a.a_sr + (left > 0 ? c : 0), left >= 8 ? 16u : (left > 0 ? (uint32_t)left * 2u : 0u));
    }
    constexpr int kBVecs = NB / 8;
    for (int v = tid; v < (a.K + 1) * kBVecs; v += kSmallThreads) {
        const int r = v / kBVecs, c = n0 + (v % kBVecs) * 8;
        const bool in = r < a.K && c < a.N;   // N is a multiple of 8
        ptx::cp_async_16(sb_u + v * 16, in ? a.B + r * a.b_sr + c : a.B, in ? 16u : 0u);
    }
    ptx::cp_async_commit();
    ptx::cp_async_wait<0>();
    __syncthreads();

    if (a.given != nullptr) {
        for (int i = tid; i < a.k; i += kSmallThreads) {
            int j = __ldg(a.given + i);
            if (j < 0 || j >= a.K) {  // reported, and reads the zero column
                atomicExch(a.status, (int)RMM_ERR_BOUNDS);
                j = a.K;
            }
            s_list[i] = (unsigned short)j;
        }
    } else {
        // ---- scores: two columns a thread; the squares are exact in fp32 and added up in fp64, as in every score pass of so few rows
        const int pairs = (a.K + 1) / 2, span = (a.M + lay.splits - 1) / lay.splits;
        for (int w = tid; w < pairs * lay.splits; w += kSmallThreads) {
            const int s = w / pairs, p = w - s * pairs, r1 = min(a.M, (s + 1) * span);
            const unsigned char *col = s_dyn + p * 4;
            double e0 = 0.0, e1 = 0.0;
#pragma unroll 8
            for (int r = s * span; r < r1; ++r) {
                const uint32_t x = *reinterpret_cast<const uint32_t *>(col + r * lay.a_pitch);
                const float x0 = __uint_as_float(x << 16), x1 = __uint_as_float(x & 0xffff0000u);
                e0 += (double)(x0 * x0);
                e1 += (double)(x1 * x1);
            }
            s_sum[(s * pairs + p) * 2] = e0;
            s_sum[(s * pairs + p) * 2 + 1] = e1;
        }
        __syncthreads();

        // ---- selection, in every block; the first one writes the list out
        unsigned u[ITEMS];
        const int j0 = tid * ITEMS, nvalid = max(0, min(ITEMS, a.K - j0));
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            double e = 0.0;
            if (i < nvalid)
                for (int s = 0; s < lay.splits; ++s) e += s_sum[s * 2 * pairs + j0 + i];
            u[i] = i < nvalid ? sel::key_image((float)e) : 0u;
        }
        const sel::Threshold th = sel::block_threshold<ITEMS, kSmallThreads>(u, nvalid, a.k, s_sel);
        const unsigned before = sel::block_rank_blocked<ITEMS, kSmallThreads>(u, nvalid, th.tau, s_sel);
        unsigned gt_before = before >> 16, eq_before = before & 0xffffu;
        double sum_kept = 0.0, sum_all = 0.0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const bool gt = i < nvalid && u[i] > th.tau, eq = i < nvalid && u[i] == th.tau, keep = gt || (eq && eq_before < th.need_eq);
            if (keep) {
                const unsigned pos = gt_before + min(eq_before, th.need_eq);
                s_list[pos] = (unsigned short)(j0 + i);
                if (blockIdx.x == 0) a.idx[pos] = j0 + i;
            }
            gt_before += gt ? 1u : 0u;
            eq_before += eq ? 1u : 0u;
            if (a.retained != nullptr && i < nvalid) {
                const double f = (double)sel::key_value(u[i]);
                sum_all += f;
                if (keep) sum_kept += f;
            }
        }
        if (a.retained != nullptr && blockIdx.x == 0) {   // the whole block: sums in a fixed order
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
                sum_kept += __shfl_down_sync(0xffffffffu, sum_kept, d);
                sum_all += __shfl_down_sync(0xffffffffu, sum_all, d);
            }
            if (lane == 0) {
                s_sel.red[warp] = sum_kept;
                s_sel.red[32 + warp] = sum_all;
            }
            __syncthreads();
            if (tid == 0) {
                double kept = 0.0, all = 0.0;
                for (int w = 0; w < kSmallWarps; ++w) {
                    kept += s_sel.red[w];
                    all += s_sel.red[32 + w];
                }
                *a.retained = all > 0.0 ? (float)(kept / all) : 1.0f;
            }
        }
    }
    if (tid < 16) s_list[a.k + tid] = (unsigned short)a.K;   // the zero column / row
    __syncthreads();

    // ---- product: warp = 16 rows x a share of the kept indices x NB columns
    const int steps = (a.k + 15) / 16;
    int mt_slots = 1;
    while (mt_slots * 16 < a.M) mt_slots *= 2;
    const int mt = warp % mt_slots, ks = warp / mt_slots, shares = kSmallWarps / mt_slots, per = (steps + shares - 1) / shares;
    const int g = lane >> 2, t = lane & 3;
    float acc[NB / 8][4] = {};
    if (mt * 16 < a.M) {
        // rows past the end repeat the last one; their sums are not stored
        const unsigned char *row0 = s_dyn + min(mt * 16 + g, a.M - 1) * lay.a_pitch, *row1 = s_dyn + min(mt * 16 + g + 8, a.M - 1) * lay.a_pitch;
        for (int st = ks * per; st < min(steps, (ks + 1) * per); ++st) {
            const uint32_t l01 = *reinterpret_cast<const uint32_t *>(s_list + st * 16 + 2 * t), l89 = *reinterpret_cast<const uint32_t *>(s_list + st * 16 + 2 * t + 8);
            auto pair = [&](const unsigned char *row, uint32_t l) -> uint32_t {
                return (uint32_t)*reinterpret_cast<const unsigned short *>(row + (l & 0xffffu) * 2) |
                       ((uint32_t)*reinterpret_cast<const unsigned short *>(row + (l >> 16) * 2) << 16);
            };
            const uint32_t fa[4] = {pair(row0, l01), pair(row1, l01), pair(row0, l89), pair(row1, l89)};
            const uint32_t brow = sb_u + (uint32_t)s_list[st * 16 + (lane & 15)] * (NB * 2) + (lane >> 4) * 16;
#pragma unroll
            for (int c = 0; c < NB / 16; ++c) {
                uint32_t fb[4];
                ptx::ldmatrix_x4_trans(fb, brow + c * 32);
                ptx::mma_bf16_16816(acc[2 * c], fa, fb[0], fb[1]);
                ptx::mma_bf16_16816(acc[2 * c + 1], fa, fb[2], fb[3]);
            }
        }
    }
    __syncthreads();   // the operands have been read: their place takes the warps' sums
    float *s_acc = reinterpret_cast<float *>(s_dyn);
#pragma unroll
    for (int c = 0; c < NB / 8; ++c) {
        float *d = s_acc + (warp * 16 + g) * NB + c * 8 + 2 * t;
        *reinterpret_cast<float2 *>(d) = make_float2(acc[c][0], acc[c][1]);
        *reinterpret_cast<float2 *>(d + 8 * NB) = make_float2(acc[c][2], acc[c][3]);
    }
    __syncthreads();
    for (int o = tid; o < a.M * (NB / 2); o += kSmallThreads) {
        const int m = o / (NB / 2), c = (o % (NB / 2)) * 2;
        if (n0 + c >= a.N) continue;
        float y0 = 0.f, y1 = 0.f;
        for (int s = 0; s < shares; ++s) {   // in the order of the kept indices
            const float2 v = *reinterpret_cast<const float2 *>(s_acc + ((s * mt_slots + (m >> 4)) * 16 + (m & 15)) * NB + c);
            y0 += v.x;
            y1 += v.y;
        }
        const int64_t off = m * a.y_sr + n0 + c;
        if (a.y_bf16)
            *reinterpret_cast<__nv_bfloat162 *>(static_cast<__nv_bfloat16 *>(a.Y) + off) = __floats2bfloat162_rn(y0 * a.scale, y1 * a.scale);
        else
            *reinterpret_cast<float2 *>(static_cast<float *>(a.Y) + off) = make_float2(y0 * a.scale, y1 * a.scale);
    }
}

int small_columns(int64_t N) { return ceil_div(N, 16) <= sm_count() ? 16 : 32; }

template <int ITEMS, int NB>
int launch_small_as(const SmallArgs &a, cudaStream_t stream)
{
    auto kern = small_product_kernel<ITEMS, NB>;
    static PerDeviceOnce configured;
    if (cudaError_t e = configured.smem(kSmallSmemMax, kern)) return fail(RMM_ERR_CUDA, "small_product: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    prof_begin("small_product_kernel", stream);
    cudaError_t e = launch_kernel(kern, dim3((unsigned)ceil_div(a.N, NB)), dim3(kSmallThreads), (size_t)small_layout(a.M, a.K, NB).total, stream, 1, a);
    if (e != cudaSuccess) return fail(RMM_ERR_CUDA, "small_product: launch: %s", cudaGetErrorString(e));
    return check_launch("small_product_kernel", stream);
}

}  // namespace

// Whole calls through the binding, two launches (up to 32 rows) or three before and one now: 16 x 1024 x 2048 19.3 -> 17.2 us,
// 24 x 2048 x 512 21.6 -> 17.3, 64 x 512 x 256 22.5 -> 17.1, 64 x 1024 x 2048 22.7 -> 17.3; what is left is the host.  On a given list
// (rmm_reduced_gemm) 13.5 to 15.8 -> 9.2 to 10.2, and 22 to 25 -> 18 to 19 where the output is scored by a pass of its own (epilogue
// energies before).  Replayed from a graph, 1292 shapes: 1.0 to 3.3 times as fast on six in seven; slower where few indices of a
// wide B are kept, since all of its rows are read: at most 16 rows, 256 kept indices or fewer, 1536 columns or more (8 x 1024 (a
// quarter) x 4096 6.3 -> 7.8 us, 9.6 -> 11.8 for the whole product).  Up to four rows stay with the GEMV, whose sums round to
// nearest; one round of blocks at most, so that A is fetched once per SM.
bool small_eligible(const rmm_mat_t *A, const rmm_mat_t *B, const rmm_mat_t *Y)
{
    auto al16 = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    if (A->batch != 1 || A->dtype != RMM_BF16 || B->dtype != RMM_BF16) return false;
    if (A->rows < kSmallMinRows || A->rows > kSmallMaxRows || A->cols > kSmallMaxK || B->cols % 8 != 0 || B->cols > 32 * (int64_t)sm_count()) return false;
    if (A->stride_col != 1 || A->stride_row % 8 != 0 || !al16(A->ptr)) return false;
    if (B->stride_col != 1 || B->stride_row % 8 != 0 || !al16(B->ptr)) return false;
    if (Y->stride_col != 1 || Y->stride_row % 2 != 0 || reinterpret_cast<uintptr_t>(Y->ptr) % 8 != 0) return false;
    return small_layout((int)A->rows, (int)A->cols, small_columns(B->cols)).total <= kSmallSmemMax;
}

int launch_small_product(const rmm_mat_t *A, const rmm_mat_t *B, int64_t k, float scale, const rmm_mat_t *Y, int32_t *idx,
                         float *retained, const int32_t *given, int *status, cudaStream_t stream)
{
    SmallArgs a;
    a.A = static_cast<const __nv_bfloat16 *>(A->ptr); a.B = static_cast<const __nv_bfloat16 *>(B->ptr); a.Y = Y->ptr;
    a.a_sr = A->stride_row; a.b_sr = B->stride_row; a.y_sr = Y->stride_row;
    a.y_bf16 = Y->dtype == RMM_BF16;
    a.M = (int)A->rows; a.K = (int)A->cols; a.N = (int)B->cols; a.k = (int)k;
    a.scale = scale;
    a.idx = idx; a.retained = retained; a.given = given; a.status = status;
    const bool wide = small_columns(a.N) == 32;
    if (a.K <= 512) return wide ? launch_small_as<1, 32>(a, stream) : launch_small_as<1, 16>(a, stream);
    if (a.K <= 1024) return wide ? launch_small_as<2, 32>(a, stream) : launch_small_as<2, 16>(a, stream);
    return wide ? launch_small_as<4, 32>(a, stream) : launch_small_as<4, 16>(a, stream);
}

}  // namespace rmm
