// 8-bit operands for the reduced product (the paper's appendix on compatibility with quantisation reports accuracy with
// INT8 and leaves a fused low-bit kernel open; this is the W8A8 form of Y = A[:, I] B[I, :] with e4m3 codes):
//   activations  Aq[i, j] = e4m3(A[i, I_j] / s_i),  s_i = max_j |A[i, I_j]| / 448  (per-row, taken over the KEPT columns
//                only, so the step adapts to what survives the selection; an all-zero row gets s_i = 1)
//   weight       given as e4m3 codes with one scale for the tensor, stored [N, K] (contraction axis contiguous): the kept
//                bytes of every row are gathered
// Both gathers run as one streaming launch (gather_q8_stream_kernel); operands it does not take (rows above 110 KB, more than
// 32768 kept columns) as one block per row, the row staged in shared memory with 16-byte loads.
// Every decision that produces a code is taken in fp32 (IEEE division, round-to-nearest-even conversion, saturating).
#include <cuda_fp8.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

constexpr int kThreadsQ = 256;

template <bool QUANT>
__global__ void __launch_bounds__(kThreadsQ) gather_q8_kernel(const void *__restrict__ src, int64_t s_row, int K, const int32_t *__restrict__ idx,
                                                              int k, uint8_t *__restrict__ dst, int64_t ld_dst, float *__restrict__ row_scale,
                                                              int *status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ float s_red[kThreadsQ / 32];
    constexpr int ES = QUANT ? 2 : 1;
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row = blockIdx.x;
    {
        const uint4 *g = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(src) + row * s_row * ES);
        uint4 *s = reinterpret_cast<uint4 *>(smem);
        const int nvec = (K * ES + 15) / 16;  // the staged row may run a few bytes past K: rows are 16-byte multiples apart
        for (int v = tid; v < nvec; v += kThreadsQ) s[v] = __ldg(g + v);
    }
    __syncthreads();
    auto column = [&](int j) -> int {  // kept column of list position j, or -1
        if (j >= k) return -1;
        const int c = __ldg(idx + j);
        if (c < 0 || c >= K) {
            atomicExch(status, (int)RMM_ERR_BOUNDS);
            return -1;
        }
        return c;
    };
    float inv_step = 1.f, step = 1.f;
    if constexpr (QUANT) {
        const unsigned short *a16 = reinterpret_cast<const unsigned short *>(smem);
        float amax = 0.f;
        for (int j = tid; j < k; j += kThreadsQ) {
            const int c = column(j);
            if (c >= 0) amax = fmaxf(amax, fabsf(__uint_as_float((unsigned)a16[c] << 16)));
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
        if (lane == 0) s_red[warp] = amax;
        __syncthreads();
        amax = s_red[0];
#pragma unroll
        for (int w = 1; w < kThreadsQ / 32; ++w) amax = fmaxf(amax, s_red[w]);
        step = amax > 0.f ? __fdiv_rn(amax, 448.f) : 1.f;
        if (tid == 0) row_scale[row] = step;
        (void)inv_step;
    }
    uint32_t *drow = reinterpret_cast<uint32_t *>(dst + row * ld_dst);
    for (int j0 = 4 * tid; j0 < (int)ld_dst; j0 += 4 * kThreadsQ) {
        uint32_t w = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = column(j0 + e);
            uint32_t code = 0;
            if (c >= 0) {
                if constexpr (QUANT) {
                    const float x = __uint_as_float((unsigned)reinterpret_cast<const unsigned short *>(smem)[c] << 16);
                    code = __nv_cvt_float_to_fp8(__fdiv_rn(x, step), __NV_SATFINITE, __NV_E4M3);
                } else {
                    code = smem[c];
                }
            }
            w |= code << (8 * e);
        }
        drow[j0 >> 2] = w;
    }
}


// Both gathers of a product as one streaming kernel: a persistent block (1024 threads, one an SM, or 512 and two) owns a contiguous
// range of the rows of A and one of the rows of B, which share the index list.  Rows arrive by bulk asynchronous copies, several at a
// time (up to 8 rows of up to 4096 kept columns; the next ones land while these are worked on), so that the barriers, the
// wait and the row maxima's meeting are paid per handful of rows: with one 8 KB row at a time they were most of the time.
// 4096 x 8192 activations and 8192 x 8192 weights, half kept: 33 + 35 us in two launches of a row at a time, 54 us by one block an
// SM, 44 by two (185 MB): a block's steps follow one another (wait, read, meet, convert, write), so a second one fills what they
// leave idle.
//
// Quotients: a code is e4m3(a / s) with the quotient rounded as IEEE division rounds it.  q = a x (1 / s), both roundings
// to nearest, is within 3 units in the last place of that quotient, so it yields the same code unless it lies that close to
// a point where codes change: those sit 20 bits below the leading bit for |q| >= 2^-6 (three mantissa bits, ties), and
// everything smaller is divided.  Divisions are thus taken for a few elements in 10^4.
constexpr int kThreadsS = 1024;                  // one block an SM, or two of half as many threads
constexpr int kUnitsS = 8;                       // (rows at a time) x (groups of 4 outputs a thread of a row): k <= 8 * 4096
constexpr int kStreamMaxRowBytes = 110 * 1024;   // two such rows (and their zero pads) fit in shared memory
constexpr int kStreamStages = 3;

struct StreamQ8 {
    const unsigned char *src[2];   // A (bf16), B (codes)
    int64_t pitch[2], rows[2], per_block[2];   // bytes between rows; rows; rows per block
    uint8_t *dst[2];
    int64_t ld_dst;
    const int32_t *idx;
    float *row_scale;
    int K, k, rows_at_once[2], stages[2];
    int *status;
    unsigned long long wait_ns;
    int withhold;
};

__device__ __forceinline__ uint32_t e4m3_code2(float x0, float x1, float step, float inv)
{
    auto quotient = [&](float x) -> float {
        const float q = x * inv;
        const uint32_t bits = __float_as_uint(q);
        const bool near_tie = ((bits + 0x80008u) & 0xfffffu) < 16u;              // within 8 of the 20 bits' middle
        const bool small = (bits & 0x7fffffffu) < 0x3c800000u;                   // |q| < 2^-6
        return near_tie || small ? __fdiv_rn(x, step) : q;
    };
    return __nv_cvt_float2_to_fp8x2(make_float2(quotient(x0), quotient(x1)), __NV_SATFINITE, __NV_E4M3);
}

// One operand's rows of this block.  `stage` and `parity` run on from one operand to the next.
template <bool QUANT, int G, int T>
__device__ __forceinline__ bool stream_rows(const StreamQ8 &a, unsigned char *smem, uint64_t *full, int *abort_flag, unsigned (*s_red)[T / 32],
                                            const uint32_t (&cb)[2 * G], int &turn)
{
    using namespace ptx;
    constexpr int ES = QUANT ? 2 : 1, W = QUANT ? 0 : 1, R = kUnitsS / G;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int at_once = a.rows_at_once[W], nst = a.stages[W];
    const uint32_t pad = (uint32_t)(a.K + 15) / 16 * 16 * ES, pitch = pad + 16, copied = (uint32_t)(a.K * ES + 15) / 16 * 16;
    const int64_t lo = (int64_t)blockIdx.x * a.per_block[W], hi = min(a.rows[W], lo + a.per_block[W]);
    if (lo >= hi) return true;
    // 16 zero bytes after each staged row: where missing indices point
    for (int i = tid; i < 4 * nst * at_once; i += T) reinterpret_cast<uint32_t *>(smem + (size_t)(i >> 2) * pitch + pad)[i & 3] = 0;
    // B's rows land where A's pads and rows were: this thread's own accesses come before the copies (which are another proxy's)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    const uint32_t base = smem_u32(smem);
    // turns of this operand: turn t0 + n uses buffer n % nst; a barrier completes once per use
    uint32_t parity_of = 0;  // bit b: parity that the next wait on buffer b expects
#pragma unroll
    for (int b = 0; b < kStreamStages; ++b) parity_of |= ((uint32_t)(turn >> (8 * b)) & 1u) << b;
    auto issue = [&](int64_t r, int b) {  // the first warp: rows r .. of one turn, a copy per lane
        const int n = (int)min((int64_t)at_once, hi - r);
        if (lane == 0) mbar_arrive_expect_tx(smem_u32(&full[b]), copied * (uint32_t)n);
        __syncwarp();
        if (lane < n)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(base + (uint32_t)(b * at_once + lane) * pitch), "l"(a.src[W] + (r + lane) * a.pitch[W]), "r"(copied),
                           "r"(smem_u32(&full[b])) : "memory");
    };
    if (warp == 0)
        for (int b = 0; b < nst && lo + (int64_t)b * at_once < hi; ++b)
            if (!(a.withhold && blockIdx.x == 0 && b == 0)) issue(lo + (int64_t)b * at_once, b);  // (test switch: block 0's first rows are never requested)
    const int words = (int)(a.ld_dst / 4);
    const int rr = lane & 3, word_in_warp = 8 * rr + (lane >> 2);  // after the transpose lane 4 m + rr holds word 8 rr + m
    auto offset = [&](int sl) -> uint32_t { return ((cb[sl >> 1] >> (16 * (sl & 1))) & 0xffffu) * ES; };
    bool ok = true;
    int b = 0;
    for (int64_t r = lo; r < hi; r += at_once) {
        const int n = (int)min((int64_t)at_once, hi - r);
        const bool landed = mbar_wait(smem_u32(&full[b]), (parity_of >> b) & 1u, abort_flag, a.status, a.wait_ns);
        if (!__syncthreads_and(landed)) {
            drain_copies();
            ok = false;
            break;
        }
        parity_of ^= 1u << b;
        const unsigned char *rows = smem + (size_t)(b * at_once) * pitch;
        uint32_t val[R][QUANT ? 2 * G : G];   // this thread's inputs: bf16 pairs, or four bytes to a register
        [[maybe_unused]] unsigned top[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if (q < n) {
                const unsigned char *row = rows + (size_t)q * pitch;
                if constexpr (QUANT) {
                    float amax = 0.f;
#pragma unroll
                    for (int h = 0; h < 2 * G; ++h) {
                        const uint32_t x0 = *reinterpret_cast<const unsigned short *>(row + offset(2 * h));
                        const uint32_t x1 = *reinterpret_cast<const unsigned short *>(row + offset(2 * h + 1));
                        val[q][h] = x0 | (x1 << 16);
                        amax = fmaxf(amax, fmaxf(fabsf(__uint_as_float(x0 << 16)), fabsf(__uint_as_float(x1 << 16))));
                    }
                    top[q] = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));  // non-negative: ordered as its bits are
                    if (lane == 0) s_red[q][warp] = top[q];
                } else {
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        uint32_t word = 0;
#pragma unroll
                        for (int e = 0; e < 4; ++e) word |= (uint32_t)row[offset(4 * g + e)] << (8 * e);
                        val[q][g] = word;
                    }
                }
            }
        }
        __syncthreads();
        // every thread holds what it needs of this buffer: refill it.  (s_red is read before the next turn's barrier and
        // written after it.)
        if (warp == 0 && r + (int64_t)nst * at_once < hi) issue(r + (int64_t)nst * at_once, b);
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if (q < n) {
                float step = 1.f, inv = 1.f;
                if constexpr (QUANT) {
                    const float amax = __uint_as_float(__reduce_max_sync(0xffffffffu, s_red[q][lane % (T / 32)]));
                    step = amax > 0.f ? __fdiv_rn(amax, 448.f) : 1.f;
                    inv = __frcp_rn(step);
                    if (!(inv < INFINITY) || !(amax < INFINITY)) inv = 0.f;  // every quotient then counts as small: divided
                    if (tid == 0) a.row_scale[r + q] = step;
                }
                uint32_t *drow = reinterpret_cast<uint32_t *>(a.dst[W] + (r + q) * a.ld_dst);
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    uint32_t mine;  // codes of this thread's slots 4 g .. 4 g + 3
                    if constexpr (QUANT) {
                        const uint32_t v0 = val[q][2 * g], v1 = val[q][2 * g + 1];
                        mine = e4m3_code2(__uint_as_float(v0 << 16), __uint_as_float(v0 & 0xffff0000u), step, inv) |
                               (e4m3_code2(__uint_as_float(v1 << 16), __uint_as_float(v1 & 0xffff0000u), step, inv) << 16);
                    } else {
                        mine = val[q][g];
                    }
                    // 4 x 4 byte transpose among the four lanes of a quad: lane rr ends up with the word of slot 4 g + rr
                    uint32_t other = __shfl_xor_sync(0xffffffffu, mine, 1);
                    mine = (rr & 1) ? __byte_perm(mine, other, 0x3715) : __byte_perm(mine, other, 0x6240);
                    other = __shfl_xor_sync(0xffffffffu, mine, 2);
                    mine = (rr & 2) ? __byte_perm(mine, other, 0x3276) : __byte_perm(mine, other, 0x5410);
                    const int w = (g * (T / 32) + warp) * 32 + word_in_warp;
                    if (w < words) drow[w] = mine;
                }
            }
        }
        if (++b == nst) b = 0;
    }
    turn = 0;
#pragma unroll
    for (int s = 0; s < kStreamStages; ++s) turn |= (int)((parity_of >> s) & 1u) << (8 * s);
    return ok;
}

// Output j of a row comes from column idx[j].  A warp takes 128 consecutive outputs at a time (group g of the block's
// 32 x 128): in slot e = 0 .. 3 lane l reads the source of output 32 e + l of them, so the lanes of one instruction read
// neighbouring kept columns (output words owned whole by a thread made the lanes' reads 16 bytes apart at rho = 1/2:
// four lanes per bank).  The four bytes of an output word then sit in the four lanes of a quad and are brought together by
// two shuffle rounds; the warp's 32 words leave as one 128-byte store.  Column numbers (the zero pad: K rounded up to 16)
// stay in registers for all rows, two to a register.
template <int G, int T>
__global__ void __launch_bounds__(T, kThreadsS / T) gather_q8_stream_kernel(const __grid_constant__ StreamQ8 a)
{
    using namespace ptx;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t full[kStreamStages];
    __shared__ int abort_flag;
    __shared__ unsigned s_red[kUnitsS / G][T / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int b = 0; b < kStreamStages; ++b) mbar_init(smem_u32(&full[b]), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();
    uint32_t cb[2 * G];
#pragma unroll
    for (int sl = 0; sl < 4 * G; ++sl) {
        const int j = ((sl >> 2) * (T / 32) + warp) * 128 + 32 * (sl & 3) + lane;
        // Positions past the row's end are not written; they stand for the first output once more, whose quotient costs what
        // any other does (a zero's would be divided: 4096 x 4096 activations, 3072 kept, 4096 columns 97 us, 84 this way).
        uint32_t col = (uint32_t)(a.K + 15) / 16 * 16;
        if (j < a.k || j >= (int)a.ld_dst) {
            const int c = __ldg(a.idx + (j < a.k ? j : 0));
            if (c < 0 || c >= a.K) atomicExch(a.status, (int)RMM_ERR_BOUNDS);
            else col = (uint32_t)c;
        }
        if (sl & 1) cb[sl >> 1] |= col << 16;
        else cb[sl >> 1] = col;
    }
    int turn = 0;
    if (stream_rows<true, G, T>(a, smem, full, &abort_flag, s_red, cb, turn)) {
        __syncthreads();
        stream_rows<false, G, T>(a, smem, full, &abort_flag, s_red, cb, turn);
    }
}

}  // namespace

bool gather_q8_streams(int64_t a_rows, int64_t K, int64_t ld_dst)
{
    // Half of the block's outputs at least: below that most of its threads have nothing to do (4096 x 1024 activations, 512 kept,
    // and 1024 columns, whole product: 60 us, by rows 25; 2048 kept of 4096, 4096 columns: 71 and 69; 3072 kept: 83 and 89)
    // (few rows leave the SMs to the streaming blocks either way: 128 x 4096, 2048 kept, 4096 columns 28 and 30 us)
    return ld_dst > (a_rows <= 512 ? 1536 : 2048) && K <= 65520 && (K + 15) / 16 * 32 + 16 <= kStreamMaxRowBytes && ld_dst <= 4096 * kUnitsS;
}

int launch_gather_q8_pair(const void *A, int64_t a_rows, int64_t a_pitch, const void *B, int64_t b_rows, int64_t b_pitch, int64_t K,
                          const int32_t *idx, int64_t k, uint8_t *Aq, uint8_t *Bq, int64_t ld_dst, float *row_scale, int *status,
                          cudaStream_t stream)
{
    StreamQ8 a = {};
    a.src[0] = static_cast<const unsigned char *>(A); a.src[1] = static_cast<const unsigned char *>(B);
    a.pitch[0] = a_pitch; a.pitch[1] = b_pitch;
    a.rows[0] = a_rows; a.rows[1] = b_rows;
    a.dst[0] = Aq; a.dst[1] = Bq;
    a.ld_dst = ld_dst; a.idx = idx; a.row_scale = row_scale;
    a.K = (int)K; a.k = (int)k;
    a.status = status;
    a.wait_ns = wait_limit_ns();
    a.withhold = debug_withhold() == WITHHOLD_QUANT;
    // Two blocks an SM where three rows of A fit in half of the shared memory (by events, one block and two: 4096 x 8192 half kept with
    // 8192 columns 53.6 and 44.0 us, 16000 x 14336 a quarter with 4096 137.6 and 115.1, 2000 x 17920 four fifths with 8192 93 and 86.4,
    // 300 x 4096 three quarters with 4096 23.0 and 19.4, 500 x 5120 half with 5120 23.4 and 22.0); with two buffers instead of three
    // rows would land no sooner than they are worked on.
    const size_t row_a = (size_t)(K + 15) / 16 * 32 + 16, whole = 2 * (size_t)(kStreamMaxRowBytes + 16), halved = 108 * 1024;
    const bool two = kStreamStages * row_a <= halved && ld_dst <= kThreadsS / 2 * 4 * kUnitsS;
    const int threads = two ? kThreadsS / 2 : kThreadsS, g = (int)ceil_div(ld_dst, (int64_t)threads * 4);
    const size_t room = two ? halved : whole;
    int64_t blocks = 0;
    size_t smem = 0;
    for (int w = 0; w < 2; ++w) {
        const size_t pitch = (size_t)(K + 15) / 16 * 16 * (w == 0 ? 2 : 1) + 16;
        a.per_block[w] = ceil_div(a.rows[w], (int64_t)sm_count() * (two ? 2 : 1));
        // as many rows at a time as the registers hold, three buffers of them where they fit, no more than a block has
        int64_t n = kUnitsS / g;
        while (n > 1 && (kStreamStages * n * pitch > room || n > a.per_block[w])) n /= 2;
        a.rows_at_once[w] = (int)n;
        a.stages[w] = kStreamStages * n * pitch <= room ? kStreamStages : 2;
        if (a.stages[w] * n * pitch > smem) smem = a.stages[w] * n * pitch;
        const int64_t nb = ceil_div(a.rows[w], a.per_block[w]);
        if (nb > blocks) blocks = nb;
    }
    using Kernel = void (*)(StreamQ8);
    static const Kernel kernels[2][kUnitsS] = {
        {gather_q8_stream_kernel<1, 1024>, gather_q8_stream_kernel<2, 1024>, gather_q8_stream_kernel<3, 1024>, gather_q8_stream_kernel<4, 1024>,
         gather_q8_stream_kernel<5, 1024>, gather_q8_stream_kernel<6, 1024>, gather_q8_stream_kernel<7, 1024>, gather_q8_stream_kernel<8, 1024>},
        {gather_q8_stream_kernel<1, 512>, gather_q8_stream_kernel<2, 512>, gather_q8_stream_kernel<3, 512>, gather_q8_stream_kernel<4, 512>,
         gather_q8_stream_kernel<5, 512>, gather_q8_stream_kernel<6, 512>, gather_q8_stream_kernel<7, 512>, gather_q8_stream_kernel<8, 512>}};
    auto kern = kernels[two][g - 1];
    static PerDeviceOnce configured[2][kUnitsS];
    if (cudaError_t e = configured[two][g - 1].smem((int)room, kern))
        return fail(RMM_ERR_CUDA, "gather_q8: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    prof_begin("gather_q8_stream_kernel", stream);
    launch_kernel(kern, dim3((unsigned)blocks), dim3(threads), smem, stream, 1, a);
    return check_launch("gather_q8_stream_kernel", stream);
}

int launch_gather_q8(bool quantise, const void *src, int64_t rows, int64_t s_row, int64_t K, const int32_t *idx, int64_t k, uint8_t *dst,
                     int64_t ld_dst, float *row_scale, int *status, cudaStream_t stream)
{
    const size_t row_bytes = (size_t)K * (quantise ? 2 : 1);
    const size_t smem = align_up(row_bytes, 16);
    if (smem > 200 * 1024 || K > INT32_MAX / 4 || rows > INT32_MAX) return fail(RMM_ERR_UNSUPPORTED, "gather_q8: row too long");
    static PerDeviceOnce configured;
    if (cudaError_t e = configured.smem(200 * 1024, gather_q8_kernel<true>, gather_q8_kernel<false>))
        return fail(RMM_ERR_CUDA, "gather_q8: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    prof_begin("gather_q8_kernel", stream);
    if (quantise)
        launch_kernel(gather_q8_kernel<true>, dim3((unsigned)rows), dim3(kThreadsQ), smem, stream, 1, src, s_row, (int)K, idx, (int)k, dst, ld_dst,
                      row_scale, status);
    else
        launch_kernel(gather_q8_kernel<false>, dim3((unsigned)rows), dim3(kThreadsQ), smem, stream, 1, src, s_row, (int)K, idx, (int)k, dst, ld_dst,
                      row_scale, status);
    return check_launch("gather_q8_kernel", stream);
}

}  // namespace rmm
