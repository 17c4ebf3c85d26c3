// Reduced product Y = scale * A[:, I] B[I, :] of few rows (a decode step of a batch of sequences): 5 to 32 rows, B's rows
// contiguous, A[:, I] packed.
//
// Bound: HBM.  Every kept row of B is used once, k N 2 bytes, and nothing else is large; what is needed is bytes in
// flight on every SM and no SM without work.  The tcgen05 form (gemm_sm100.cu, 128 x 256 tiles, rows fetched by eight
// gather warps) moves 33-38 GB/s per SM and had 32 tiles for 148 SMs on 8192 columns.  Here, as in attn_decode.cu:
//   - a block of four warps owns 128 columns and a slice of the kept rows; two blocks share an SM; every warp streams
//     groups of 16 kept rows, with the 16 kept columns of A that meet them, through a private ring of 27 KB (16-byte
//     cp.async; row numbers are loaded four groups ahead: one group ahead the ring never filled, 44 us for 27);
//   - Y^T = B^T A^T: the columns of B are M of mma.m16n8k16 (ldmatrix.trans of the rows as they lie in memory), the rows
//     of A its N, eight at a time: no padding beyond eight rows;
//   - the four warps meet in shared memory, slices of the kept rows through fp32 partial sums that a second kernel adds
//     in order.
// Sums are fp32 throughout, as in the other forms.
// Measured against whole and cut 128 x 256 tiles of the tcgen05 form, gather of A included: 8 x 4096 (half kept) x 14336
// 24.0 us (40.5, 28.3), 24 x 8192 (a quarter kept) x 28672 36.5 (41.1, 41.2), 32 x 28672 (half) x 8192 68 (215, 68); at 48
// rows the last takes 93 (216, 70), so taller outputs stay with the tcgen05 form.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

constexpr int kSkWarps = 4, kSkBlocks = 2;   // warps per block, blocks per SM
constexpr int CW = 128;                      // columns per block

struct SkinnyArgs {
    const __nv_bfloat16 *ap, *b;
    const int32_t *idx;
    void *y;
    int64_t M, N, k, K;
    int64_t a_ld, a_sb, b_ld, b_sb, idx_stride, y_sb, y_sr;
    int y_bf16, pieces;
    int64_t per;          // groups of 16 kept rows per piece
    float scale;
    float *partials;      // pieces > 1: [batch][piece][M][N]
    int *status;
};

template <int NT>
struct SkinnyShape {
    static constexpr int kBytesB = 16 * CW * 2, kUnit = kBytesB + 8 * NT * 32;                   // 16 kept rows of B, 16 kept columns of A
    static constexpr int kUnits = 27648 / kUnit, kRing = kUnit * kUnits;                         // per warp
    static constexpr int kSmem = kSkWarps * kRing;
    static_assert(8 * NT * CW * 4 <= kRing, "the warps meet in the rings");
};

template <int NT>
__global__ void __launch_bounds__(kSkWarps * 32, kSkBlocks) gemm_skinny_kernel(const SkinnyArgs a)
{
    using S = SkinnyShape<NT>;
    constexpr int U = S::kUnits, CPR = CW / 8, RPI = 32 / CPR;  // 16-byte vectors per row; rows per warp request
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const uint32_t ring = ptx::smem_u32(smem) + warp * S::kRing;
    pdl_wait();

    const int64_t batch = blockIdx.z, n0 = (int64_t)blockIdx.x * CW;
    const int64_t groups = (a.k + 15) / 16, g0 = (int64_t)blockIdx.y * a.per, g1 = min(groups, g0 + a.per);
    const int n_sub = (int)max((int64_t)0, (g1 - g0 - warp + kSkWarps - 1) / kSkWarps);  // this warp's groups: g0 + warp + 4 n
    const int32_t *idx = a.idx + batch * a.idx_stride;
    const int c = lane % CPR;
    const bool col_ok = n0 + c * 8 < a.N;
    const __nv_bfloat16 *bcol = a.b + batch * a.b_sb + n0 + c * 8;
    auto rows_at = [&](int n) -> int {  // row numbers of this warp's groups n (lanes 0-15) and n + 1 (lanes 16-31), -1 past the end
        const int nn = n + (lane >> 4);
        const int64_t j = (g0 + warp + (int64_t)kSkWarps * nn) * 16 + (lane & 15);
        return nn < n_sub && j < a.k ? __ldg(idx + j) : -1;
    };
    int rows_a = rows_at(0), rows_b = rows_at(2), rows_c = rows_at(4);  // the pair in use, and the two after it
    auto load = [&](int n) {  // group n into ring entry n % U; always one commit group
        if (n < n_sub) {
            const int64_t j0 = (g0 + warp + (int64_t)kSkWarps * n) * 16;
            const int half = (n & 1) * 16;
            if (lane >> 4 == (n & 1) && j0 + (lane & 15) < a.k && (rows_a < 0 || rows_a >= a.K)) {
                atomicExch(a.status, (int)RMM_ERR_BOUNDS);  // a bad index is reported and contributes nothing
                rows_a = -1;
            }
            const uint32_t dst = ring + (n % U) * S::kUnit;
#pragma unroll
            for (int i = 0; i < 16 / RPI; ++i) {
                const int r = lane / CPR + i * RPI;
                const int row = __shfl_sync(0xffffffffu, rows_a, half + r);
                const bool live = row >= 0 && col_ok;
                ptx::cp_async_16(dst + r * (CW * 2) + ((c ^ (r & 7)) << 4), live ? bcol + (int64_t)row * a.b_ld : a.b, live ? 16u : 0u);
            }
            // row r of A[:, I]: two 16-byte halves of the group, swapped in every second four rows (bank conflicts); the
            // packed rows are zero from k to their pitch, a multiple of 8
#pragma unroll
            for (int i = 0; i < (NT + 1) / 2; ++i) {
                const int r = (lane >> 1) + 16 * i, q = lane & 1;
                const bool live = r < a.M && j0 + q * 8 < a.a_ld;
                if (r < 8 * NT)
                    ptx::cp_async_16(dst + S::kBytesB + r * 32 + ((q ^ ((r >> 2) & 1)) << 4),
                                     live ? a.ap + batch * a.a_sb + r * a.a_ld + j0 + q * 8 : a.ap, live ? 16u : 0u);
            }
            if (n & 1) {
                rows_a = rows_b;
                rows_b = rows_c;
                rows_c = rows_at(n + 5);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

#pragma unroll 1
    for (int n = 0; n < U - 1; ++n) load(n);
    float acc[NT][CW / 16][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int mt = 0; mt < CW / 16; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[nt][mt][e] = 0.f;
    const int v_row = ((lane >> 4) << 3) + (lane & 7);
    for (int n = 0; n < n_sub; ++n) {
        asm volatile("cp.async.wait_group %0;" ::"n"(U - 2) : "memory");
        __syncwarp();  // group n is there for every lane, and every lane is done with the entry refilled next
        load(n + U - 1);
        const uint32_t st = ring + (n % U) * S::kUnit;
        uint32_t fb[NT][2];  // lane (g, t): row 8 nt + g of A, kept positions 2 t, 2 t + 1 and 2 t + 8, 2 t + 9 of the group
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const uint32_t at = st - ptx::smem_u32(smem) + S::kBytesB + (nt * 8 + g) * 32 + t * 4;
            fb[nt][0] = *reinterpret_cast<const uint32_t *>(smem + (at + ((g >> 2) << 4)));
            fb[nt][1] = *reinterpret_cast<const uint32_t *>(smem + (at + (((g >> 2) ^ 1) << 4)));
        }
#pragma unroll
        for (int mt = 0; mt < CW / 16; ++mt) {
            uint32_t v[4];
            ptx::ldmatrix_x4_trans(v, st + v_row * (CW * 2) + (((2 * mt + ((lane >> 3) & 1)) ^ (v_row & 7)) << 4));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) ptx::mma_bf16_16816(acc[nt][mt], v, fb[nt][0], fb[nt][1]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();

    float *mine = reinterpret_cast<float *>(smem + warp * S::kRing);  // [row][CW]
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int mt = 0; mt < CW / 16; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (nt * 8 + 2 * t + (e & 1) < a.M) mine[(nt * 8 + 2 * t + (e & 1)) * CW + mt * 16 + g + (e >> 1) * 8] = acc[nt][mt][e];
    __syncthreads();
    for (int i = tid; i < (int)a.M * (CW / 4); i += kSkWarps * 32) {
        const int r = i / (CW / 4), cc = i % (CW / 4) * 4;
        const int64_t n = n0 + cc;
        if (n >= a.N) continue;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kSkWarps; ++w) {
            const float4 x = *reinterpret_cast<const float4 *>(smem + w * S::kRing + (r * CW + cc) * 4);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        if (a.pieces > 1) {
            __stcg(reinterpret_cast<float4 *>(a.partials + ((batch * a.pieces + blockIdx.y) * a.M + r) * a.N + n), s);
        } else {
            const int64_t off = batch * a.y_sb + r * a.y_sr + n;  // rows of Y start on 16 bytes, N is a multiple of 8
            if (a.y_bf16) {
                __nv_bfloat162 lo = __floats2bfloat162_rn(s.x * a.scale, s.y * a.scale), hi = __floats2bfloat162_rn(s.z * a.scale, s.w * a.scale);
                *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(a.y) + off) =
                    make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
            } else {
                *reinterpret_cast<float4 *>(static_cast<float *>(a.y) + off) = make_float4(s.x * a.scale, s.y * a.scale, s.z * a.scale, s.w * a.scale);
            }
        }
    }
}

// The pieces of the contraction added in order; a thread owns four columns of a row.
__global__ void __launch_bounds__(128) skinny_meet_kernel(const SkinnyArgs a)
{
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x, batch = blockIdx.z, quads = a.N / 4;
    if (i >= a.M * quads) return;
    const int64_t r = i / quads, n = i % quads * 4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int p = 0; p < a.pieces; ++p) {
        const float4 x = __ldcg(reinterpret_cast<const float4 *>(a.partials + ((batch * a.pieces + p) * a.M + r) * a.N + n));
        s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    const int64_t off = batch * a.y_sb + r * a.y_sr + n;
    if (a.y_bf16) {
        __nv_bfloat162 lo = __floats2bfloat162_rn(s.x * a.scale, s.y * a.scale), hi = __floats2bfloat162_rn(s.z * a.scale, s.w * a.scale);
        *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(a.y) + off) = make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
    } else {
        *reinterpret_cast<float4 *>(static_cast<float *>(a.y) + off) = make_float4(s.x * a.scale, s.y * a.scale, s.z * a.scale, s.w * a.scale);
    }
}

struct SkinnyGrid {
    int pieces;
    int64_t per;
};

// Slices of the kept rows: the least (rounds of blocks over the GPU) x (groups a warp walks, and about four more for what
// a block spends outside them) and, with more than one slice, four for their meeting; among one slice and the most that
// make one or two rounds.  No more than `fit` slices, which is what the workspace holds.
SkinnyGrid skinny_grid(int64_t batch, int64_t N, int64_t k, int64_t fit)
{
    SkinnyGrid g = {1, 1};
    const int64_t groups = ceil_div(k, 16), tiles = batch * ceil_div(N, CW), slots = (int64_t)sm_count() * kSkBlocks;
    int64_t best = INT64_MAX;
    for (int64_t rounds = 0; rounds <= 2; ++rounds) {
        int64_t s = rounds * slots / tiles;
        int64_t most = ceil_div(groups, 4 * kSkWarps);  // at least four groups a warp
        if (most > fit) most = fit > 1 ? fit : 1;
        s = s < 1 ? 1 : (s > most ? most : s);
        const int64_t per = ceil_div(groups, s), cost = ceil_div(tiles * ceil_div(groups, per), slots) * (ceil_div(per, kSkWarps) + 4) + (per < groups ? 4 : 0);
        if (cost < best) {
            best = cost;
            g.per = per;
            g.pieces = (int)ceil_div(groups, per);
        }
    }
    return g;
}

template <int NT>
int launch_shape(const SkinnyArgs &a, int64_t batch, cudaStream_t stream)
{
    using S = SkinnyShape<NT>;
    auto kern = gemm_skinny_kernel<NT>;
    static PerDeviceOnce configured;
    if (cudaError_t e = configured.smem(S::kSmem, kern)) return fail(RMM_ERR_CUDA, "gemm_skinny: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    prof_begin("gemm_skinny_kernel", stream);
    launch_kernel(kern, dim3((unsigned)ceil_div(a.N, CW), (unsigned)a.pieces, (unsigned)batch), dim3(kSkWarps * 32), S::kSmem, stream, 1, a);
    int rc = check_launch("gemm_skinny_kernel", stream);
    if (rc != RMM_OK || a.pieces == 1) return rc;
    prof_begin("skinny_meet_kernel", stream);
    launch_kernel(skinny_meet_kernel, dim3((unsigned)ceil_div(a.M * (a.N / 4), 128), 1, (unsigned)batch), dim3(128), 0, stream, 1, a);
    return check_launch("skinny_meet_kernel", stream);
}

}  // namespace

// Enough for every count of kept indices up to k.
size_t gemm_skinny_partial_bytes(int64_t batch, int64_t M, int64_t N, int64_t k)
{
    const int64_t tiles = batch * ceil_div(N, CW), slots = (int64_t)sm_count() * kSkBlocks;
    int64_t s = 2 * slots / tiles;
    const int64_t most = ceil_div(ceil_div(k, 16), 4 * kSkWarps);
    if (s > most) s = most;
    return s <= 1 ? 0 : align_up((size_t)(batch * s * M * N) * 4, 256);
}

// p.a packed rows (zero between k and the pitch), p.b the unpacked B with the list p.b_idx.
int launch_gemm_skinny(const TcProblem &p, cudaStream_t stream)
{
    const SkinnyGrid g = skinny_grid(p.batch, p.N, p.k, (int64_t)(p.partials_bytes / (size_t)(p.batch * p.M * p.N * 4)));
    SkinnyArgs a = {};
    a.ap = p.a; a.b = p.b; a.idx = p.b_idx; a.y = p.y;
    a.M = p.M; a.N = p.N; a.k = p.k; a.K = p.b_rows;
    a.a_ld = p.a_ld; a.a_sb = p.a_sb; a.b_ld = p.b_ld; a.b_sb = p.b_batches > 1 ? p.b_sb : 0; a.idx_stride = p.b_idx_stride;
    a.y_sb = p.y_sb; a.y_sr = p.y_sr; a.y_bf16 = p.y_bf16;
    a.pieces = g.pieces; a.per = g.per; a.scale = p.scale; a.partials = p.partials; a.status = p.status;
    switch ((int)ceil_div(p.M, 8)) {
    case 1: return launch_shape<1>(a, p.batch, stream);
    case 2: return launch_shape<2>(a, p.batch, stream);
    case 3: return launch_shape<3>(a, p.batch, stream);
    default: return launch_shape<4>(a, p.batch, stream);
    }
}

}  // namespace rmm
