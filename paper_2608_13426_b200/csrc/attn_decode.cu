// Reduced attention for decode steps (paper Sec. 3.3 with rho_t = 1 and a handful of query rows): feature selection,
// S~ = Q[:, I] K[:, I]^T / sqrt(Dh), softmax and P V in one pass over the key/value cache, plus a small combine.
//
// Bound: HBM.  K and V are each read once, 4 bytes per (key, column); the kept features of a 2-byte row touch every
// 32-byte sector of it, so there is nothing to gain from gathering and the packed copies of K per query head that the
// prefill form makes would multiply the traffic (8 sequences x 32 / 8 heads x 4096 keys x 128: 80 us of packing and
// 97 us of a kernel whose 128-row tiles hold one row; 35 us for this form, 134 MB of caches).  So the rows are read in
// place, the dropped features are zeros in Q, and everything else is arranged around bytes in flight:
//   - the keys of all (sequence, kv head) pairs form one axis of tiles that is cut into equal pieces, one per SM, so
//     no SM waits for another whatever the batch, the head count or the cache length;
//   - inside a block every warp is on its own: it owns 16 keys of a tile and a private ring of 24-48 KB filled by
//     16-byte cp.async (about 128 KB in flight per SM), and no block barrier is met until the piece ends;
//   - all query rows that share a kv head (group x Lq) sit in the N = 8 columns of mma.m16n8k16 with the keys as M:
//     S^T = K Q^T and O^T = V^T P^T.  128-row tcgen05 tiles would be padding here: at 8 rows the products take 16
//     instructions per 16 keys and stay below a third of the time the bytes need.
// Softmax weights are taken against a per-row maximum that is refreshed only when exceeded by 2^40 (see
// attn_fused.cu), rounded once to bf16; row sums, maxima and O stay fp32.  Pieces of one head meet in a fixed order.
#include <math.h>

#include "common.cuh"
#include "select.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

constexpr float kGrowLog2 = 40.f;  // log2 of the largest p taken against a stale maximum

struct DecodeArgs {
    const __nv_bfloat16 *q, *k, *v;
    __nv_bfloat16 *o;
    int64_t q_sb, q_sh, q_sr, k_sb, k_sh, k_sr, v_sb, v_sh, v_sr, o_sb, o_sh, o_sr;
    int Hkv, group, Lq, Lk, Dh, kd, causal;
    int rows, chunks;            // query rows per kv head (group x Lq), and how many row tiles they make
    int64_t jobs;                // B x Hkv x chunks
    int tiles;                   // key tiles per job
    int64_t per_block;           // tiles per block
    float scale_log2;            // log2(e) / sqrt(Dh)
    int32_t *idx_feat;           // [B, Hq, kd] or NULL
    float *part_o, *part_ml;     // partial pieces: [2 x blocks][row tile][Dh padded], [2 x blocks][row tile][2]
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool live)
{
    const int n = live ? 16 : 0;  // 0: the 16 bytes are zero-filled and src is not read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldm4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x)
{
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int DH, int NT, int WARPS>
struct DecodeShape {
    static constexpr int kRows = 8 * NT, kTileKeys = 16 * WARPS;
    static constexpr int kHalf = 16 * DH * 2, kStage = 2 * kHalf;              // 16 keys of K, then 16 keys of V
    static constexpr int kStages = 196608 / WARPS / kStage;                     // 192 KB of rings: 3 (wide heads) to 6
    static constexpr int kRing = kStages * kStage;                              // per warp
    static constexpr int kQPitch = DH + 8;
    static constexpr int kOffQ = WARPS * kRing, kOffKept = kOffQ + kRows * kQPitch * 2;
    static constexpr int kOffMl = kOffKept + kRows * (DH / 32) * 4, kSmem = kOffMl + WARPS * kRows * 8;
    static_assert(kRows * DH * 4 <= kRing, "the merge of a piece reuses the warp's ring");
};

template <int DH, int NT, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) attn_decode_kernel(const DecodeArgs a)
{
    using S = DecodeShape<DH, NT, WARPS>;
    constexpr int kRows = S::kRows, ST = S::kStages, CPR = DH / 8;  // 16-byte units per row
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const uint32_t ring = ptx::smem_u32(smem) + warp * S::kRing;
    __nv_bfloat16 *qs = reinterpret_cast<__nv_bfloat16 *>(smem + S::kOffQ);
    uint32_t *kept = reinterpret_cast<uint32_t *>(smem + S::kOffKept);   // [row][DH / 32] bit masks of the kept features
    float *ml = reinterpret_cast<float *>(smem + S::kOffMl);             // [warp][row][2]
    pdl_wait();

    const int64_t w_begin = (int64_t)blockIdx.x * a.per_block;
    const int64_t w_end = min(a.jobs * a.tiles, w_begin + a.per_block);
    bool first_piece = true;
    for (int64_t pos = w_begin; pos < w_end;) {
        const int64_t job = pos / a.tiles;
        const int ta = (int)(pos - job * a.tiles), tb = (int)min((int64_t)a.tiles, ta + (w_end - pos));
        pos += tb - ta;
        const int chunk = (int)(job % a.chunks);
        const int64_t bh = job / a.chunks, b = bh / a.Hkv, hk = bh % a.Hkv;
        const int row0 = chunk * kRows, nrows = min(kRows, a.rows - row0);
        const __nv_bfloat16 *kp = a.k + b * a.k_sb + hk * a.k_sh, *vp = a.v + b * a.v_sb + hk * a.v_sh;
        const int n_sub = tb - ta;  // this warp's 16-key steps

        auto load = [&](int n) {  // step n of this piece into ring entry n % ST; always one commit group
            if (n < n_sub) {
                const uint32_t dst = ring + (n % ST) * S::kStage;
                const int key0 = (ta + n) * S::kTileKeys + warp * 16;
                const int c = lane % CPR;
#pragma unroll
                for (int i = 0; i < 16 * CPR / 32; ++i) {
                    const int r = lane / CPR + i * (32 / CPR);
                    const bool live = key0 + r < a.Lk && c * 8 < a.Dh;
                    const int64_t key = live ? key0 + r : 0;
                    const uint32_t off = r * (DH * 2) + ((c ^ (r & 7)) << 4);
                    cp_async16(dst + off, live ? kp + key * a.k_sr + c * 8 : a.k, live);
                    cp_async16(dst + S::kHalf + off, live ? vp + key * a.v_sr + c * 8 : a.v, live);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int n = 0; n < ST - 1; ++n) load(n);

        // ---- feature sets of the heads in this row tile (one warp per head), Q with the dropped features zeroed
        for (int i = tid; i < (kRows - nrows) * S::kQPitch; i += WARPS * 32) qs[nrows * S::kQPitch + i] = __float2bfloat16(0.f);
        for (int i = tid; i < (kRows - nrows) * (DH / 32); i += WARPS * 32) kept[nrows * (DH / 32) + i] = 0u;
        const int h_first = row0 / a.Lq, h_last = (row0 + nrows - 1) / a.Lq;
        for (int h = h_first + warp; h <= h_last; h += WARPS) {
            const __nv_bfloat16 *qp = a.q + b * a.q_sb + (hk * a.group + h) * a.q_sh;
            uint32_t u[DH / 32];
#pragma unroll
            for (int i = 0; i < DH / 32; ++i) {
                const int f = i * 32 + lane;
                double e = 0.0;
                if (f < a.Dh)
                    for (int r = 0; r < a.Lq; ++r) {
                        const float x = __bfloat162float(qp[(int64_t)r * a.q_sr + f]);
                        e += (double)(x * x);  // the square of a bf16 number is exact in fp32
                    }
                u[i] = f < a.Dh ? sel::key_image((float)e) : 0u;  // 0: below every key
            }
            uint32_t tau = 0;  // largest value that at least kd keys reach: the image of the kd-th largest key
#pragma unroll 1
            for (int bit = 31; bit >= 0; --bit) {
                const uint32_t cand = tau | (1u << bit);
                int c = 0;
#pragma unroll
                for (int i = 0; i < DH / 32; ++i) c += u[i] >= cand ? 1 : 0;
                if (__reduce_add_sync(0xffffffffu, c) >= a.kd) tau = cand;
            }
            int c = 0;
#pragma unroll
            for (int i = 0; i < DH / 32; ++i) c += u[i] > tau ? 1 : 0;
            int need_eq = a.kd - __reduce_add_sync(0xffffffffu, c), at = 0;
            const int r_lo = max(row0, h * a.Lq), r_hi = min(row0 + nrows, (h + 1) * a.Lq);
            // the piece that holds a head's first row and first key writes its index list
            int32_t *out = a.idx_feat != nullptr && ta == 0 && r_lo == h * a.Lq
                               ? a.idx_feat + ((b * a.Hkv + hk) * a.group + h) * a.kd : nullptr;
#pragma unroll
            for (int i = 0; i < DH / 32; ++i) {
                const unsigned eq = __ballot_sync(0xffffffffu, u[i] == tau), lt = (1u << lane) - 1u;
                const bool keep = u[i] > tau || (u[i] == tau && __popc(eq & lt) < need_eq);
                need_eq -= min(need_eq, __popc(eq));
                const unsigned k_mask = __ballot_sync(0xffffffffu, keep);
                const int f = i * 32 + lane;
                if (out != nullptr && keep) out[at + __popc(k_mask & lt)] = f;
                at += __popc(k_mask);
                for (int r = r_lo; r < r_hi; ++r) {
                    qs[(r - row0) * S::kQPitch + f] = keep ? qp[(int64_t)(r - h * a.Lq) * a.q_sr + f] : __float2bfloat16(0.f);
                    if (lane == 0) kept[(r - row0) * (DH / 32) + i] = k_mask;
                }
            }
        }
        __syncthreads();
        uint32_t qf[NT][DH / 16][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks) {
                const __nv_bfloat16 *p = qs + (nt * 8 + g) * S::kQPitch + ks * 16 + t * 2;
                qf[nt][ks][0] = *reinterpret_cast<const uint32_t *>(p);
                qf[nt][ks][1] = *reinterpret_cast<const uint32_t *>(p + 8);
            }

        // ---- this warp's keys: thread (g, t) holds the logits of keys g and g + 8 against rows 2 t and 2 t + 1
        float o[NT][DH / 16][4], m[NT][2], l[NT][2];
        int last[NT][2];  // last visible key of the row (-1: none)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
            for (int mt = 0; mt < DH / 16; ++mt)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[nt][mt][e] = 0.f;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = row0 + nt * 8 + 2 * t + e;
                m[nt][e] = -INFINITY;
                l[nt][e] = 0.f;
                last[nt][e] = r < row0 + nrows ? (a.causal ? min(a.Lk - 1, r % a.Lq + a.Lk - a.Lq) : a.Lk - 1) : -1;
            }
        }
        const uint32_t k_lane = (lane & 15) * (DH * 2), k_x = lane & 7;            // ldmatrix rows of K
        const int v_row = ((lane >> 4) << 3) + (lane & 7);                          // and of V (transposed)
        for (int n = 0; n < n_sub; ++n) {
            asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
            __syncwarp();  // step n has landed for every lane, and every lane is done with the entry that is refilled now
            load(n + ST - 1);
            const uint32_t kst = ring + (n % ST) * S::kStage, vst = kst + S::kHalf;
            const int key0 = (ta + n) * S::kTileKeys + warp * 16;
            float s[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[nt][e] = 0.f;
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks) {
                uint32_t ka[4];
                ldm4(ka, kst + k_lane + (((2 * ks + (lane >> 4)) ^ k_x) << 4));
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma16816(s[nt], ka, qf[nt][ks][0], qf[nt][ks][1]);
            }
            bool odd = false;  // an infinity or NaN: perhaps a dropped feature's 0 x inf
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) odd |= !(fabsf(s[nt][e]) < INFINITY);
            if (__any_sync(0xffffffffu, odd)) {  // (never for finite logits) the kept features alone, one by one
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int kr = g + (e >> 1) * 8, row = nt * 8 + 2 * t + (e & 1);
                        float acc = 0.f;
                        for (int f = 0; f < DH; ++f)
                            if (kept[row * (DH / 32) + (f >> 5)] >> (f & 31) & 1u) {
                                const uint32_t at = (kst - ptx::smem_u32(smem)) + kr * (DH * 2) + ((((f >> 3) ^ (kr & 7)) << 4) | ((f & 7) * 2));
                                acc = fmaf(__bfloat162float(qs[row * S::kQPitch + f]),
                                           __bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(smem + at)), acc);
                            }
                        s[nt][e] = acc;
                    }
            }
            bool grow = false;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[nt][e] = key0 + g + (e >> 1) * 8 <= last[nt][e & 1] ? s[nt][e] * a.scale_log2 : -INFINITY;
                    grow |= s[nt][e] > m[nt][e & 1] + kGrowLog2;
                }
            if (__any_sync(0xffffffffu, grow)) {  // the rows' maxima so far, and the sums taken against the old ones scaled
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float mx = fmaxf(s[nt][e], s[nt][e + 2]);
#pragma unroll
                        for (int d = 4; d < 32; d <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
                        mx = fmaxf(mx, m[nt][e]);
                        const float alpha = m[nt][e] > -INFINITY ? ptx::ex2(m[nt][e] - mx) : 1.f;
                        m[nt][e] = mx;
                        l[nt][e] *= alpha;
#pragma unroll
                        for (int mt = 0; mt < DH / 16; ++mt) {
                            o[nt][mt][e] *= alpha;
                            o[nt][mt][e + 2] *= alpha;
                        }
                    }
            }
            uint32_t pb[NT][2];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const float n0 = m[nt][0] > -INFINITY ? -m[nt][0] : 0.f, n1 = m[nt][1] > -INFINITY ? -m[nt][1] : 0.f;
                const float p0 = ptx::ex2(s[nt][0] + n0), p1 = ptx::ex2(s[nt][1] + n1), p2 = ptx::ex2(s[nt][2] + n0), p3 = ptx::ex2(s[nt][3] + n1);
                l[nt][0] += p0 + p2;
                l[nt][1] += p1 + p3;
                __nv_bfloat162 x = __floats2bfloat162_rn(p0, p1), y = __floats2bfloat162_rn(p2, p3);
                pb[nt][0] = transpose8x8(*reinterpret_cast<uint32_t *>(&x));  // (key g, rows 2t) -> (row g, keys 2t)
                pb[nt][1] = transpose8x8(*reinterpret_cast<uint32_t *>(&y));
            }
#pragma unroll
            for (int mt = 0; mt < DH / 16; ++mt) {
                uint32_t va[4];
                ldm4_trans(va, vst + v_row * (DH * 2) + (((2 * mt + ((lane >> 3) & 1)) ^ (v_row & 7)) << 4));
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma16816(o[nt][mt], va, pb[nt][0], pb[nt][1]);
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();

        // ---- the warps of the block meet: maxima and sums, then O through the rings
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float sum = l[nt][e];
#pragma unroll
                for (int d = 4; d < 32; d <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
                if (g == 0) {
                    ml[(warp * kRows + nt * 8 + 2 * t + e) * 2] = m[nt][e];
                    ml[(warp * kRows + nt * 8 + 2 * t + e) * 2 + 1] = sum;
                }
            }
        float *mine = reinterpret_cast<float *>(smem + warp * S::kRing);  // [row][DH]
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int mt = 0; mt < DH / 16; ++mt)
#pragma unroll
                for (int e = 0; e < 4; ++e) mine[(nt * 8 + 2 * t + (e & 1)) * DH + mt * 16 + g + (e >> 1) * 8] = o[nt][mt][e];
        __syncthreads();
        const bool whole = ta == 0 && tb == a.tiles;
        const int64_t slot = 2 * (int64_t)blockIdx.x + (first_piece ? 0 : 1);
        for (int i = tid; i < nrows * DH; i += WARPS * 32) {
            const int r = i / DH, c = i % DH;
            float mx = -INFINITY;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) mx = fmaxf(mx, ml[(w * kRows + r) * 2]);
            float sum = 0.f, lsum = 0.f;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                const float mw = ml[(w * kRows + r) * 2], f = mw > -INFINITY ? ptx::ex2(mw - mx) : 0.f;
                if (mw > -INFINITY) sum += f * reinterpret_cast<const float *>(smem + w * S::kRing)[r * DH + c];
                lsum += f * ml[(w * kRows + r) * 2 + 1];
            }
            if (whole) {
                const int row = row0 + r;
                if (c < a.Dh)
                    a.o[b * a.o_sb + (hk * a.group + row / a.Lq) * a.o_sh + (int64_t)(row % a.Lq) * a.o_sr + c] =
                        __float2bfloat16_rn(lsum > 0.f ? sum * (1.f / lsum) : 0.f);
            } else {
                a.part_o[(slot * kRows + r) * DH + c] = sum;
                if (c == 0) {
                    a.part_ml[(slot * kRows + r) * 2] = mx;
                    a.part_ml[(slot * kRows + r) * 2 + 1] = lsum;
                }
            }
        }
        __syncthreads();
        first_piece = false;
    }
}

// Rows whose keys were cut into several pieces: one warp per row adds the pieces in order of their keys.
template <int DH, int NT>
__global__ void __launch_bounds__(128) attn_decode_combine_kernel(const DecodeArgs a)
{
    constexpr int kRows = 8 * NT;
    const int lane = threadIdx.x & 31;
    pdl_wait();
    const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int64_t job = w / kRows;
    if (job >= a.jobs) return;
    const int r = (int)(w % kRows), row = (int)(job % a.chunks) * kRows + r;
    if (row >= a.rows) return;
    const int64_t b0 = job * a.tiles / a.per_block, b1 = ((job + 1) * a.tiles - 1) / a.per_block;
    if (b0 == b1) return;  // written by its only block
    // a block's first piece is in its even slot; only the job's first block can hold it as a later piece
    auto slot = [&](int64_t blk) { return 2 * blk + (blk == b0 && b0 * a.per_block < job * a.tiles ? 1 : 0); };
    float mx = -INFINITY;
    for (int64_t blk = b0 + lane; blk <= b1; blk += 32) mx = fmaxf(mx, a.part_ml[(slot(blk) * kRows + r) * 2]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
    float acc[DH / 32], lsum = 0.f;
#pragma unroll
    for (int i = 0; i < DH / 32; ++i) acc[i] = 0.f;
#pragma unroll 4
    for (int64_t blk = b0; blk <= b1; ++blk) {
        const int64_t s = slot(blk) * kRows + r;
        const float mw = a.part_ml[s * 2], f = mw > -INFINITY ? ptx::ex2(mw - mx) : 0.f;
        lsum += f * a.part_ml[s * 2 + 1];
#pragma unroll
        for (int i = 0; i < DH / 32; ++i) {
            const float x = a.part_o[s * DH + i * 32 + lane];
            acc[i] += f > 0.f ? f * x : 0.f;
        }
    }
    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
    const int64_t bh = job / a.chunks, b = bh / a.Hkv, hk = bh % a.Hkv;
    __nv_bfloat16 *o = a.o + b * a.o_sb + (hk * a.group + row / a.Lq) * a.o_sh + (int64_t)(row % a.Lq) * a.o_sr;
#pragma unroll
    for (int i = 0; i < DH / 32; ++i)
        if (i * 32 + lane < a.Dh) o[i * 32 + lane] = __float2bfloat16_rn(acc[i] * inv);
}

struct DecodeGrid {
    int dh, nt, warps, chunks, tiles;
    int64_t jobs, per_block, blocks;
};

DecodeGrid decode_grid(const rmm_attn_desc_t *d)
{
    DecodeGrid g;
    const int64_t rows = d->Hq / d->Hkv * d->Lq;
    g.dh = d->Dh <= 64 ? 64 : (d->Dh <= 128 ? 128 : 256);
    g.nt = rows <= 8 ? 1 : 2;
    g.warps = g.dh == 256 ? 4 : 8;
    g.chunks = (int)ceil_div(rows, 8 * g.nt);
    g.jobs = d->B * d->Hkv * g.chunks;
    g.tiles = (int)ceil_div(d->Lk, 16 * g.warps);
    const int64_t total = g.jobs * g.tiles;
    g.per_block = ceil_div(total, sm_count());
    g.blocks = ceil_div(total, g.per_block);
    return g;
}

template <int DH, int NT, int WARPS>
int launch_shape(const DecodeArgs &a, int64_t blocks, cudaStream_t stream)
{
    using S = DecodeShape<DH, NT, WARPS>;
    auto kern = attn_decode_kernel<DH, NT, WARPS>;
    static PerDeviceOnce configured;
    if (configured.first()) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem);
        if (e != cudaSuccess) return fail(RMM_ERR_CUDA, "attn_decode: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    }
    prof_begin("attn_decode_kernel", stream);
    launch_kernel(kern, dim3((unsigned)blocks), dim3(WARPS * 32), S::kSmem, stream, 1, a);
    int rc = check_launch("attn_decode_kernel", stream);
    if (rc != RMM_OK) return rc;
    if (a.per_block % a.tiles == 0) return RMM_OK;  // every job lies in one block
    prof_begin("attn_decode_combine_kernel", stream);
    launch_kernel(attn_decode_combine_kernel<DH, NT>, dim3((unsigned)ceil_div(a.jobs * S::kRows, 4)), dim3(128), 0, stream, 1, a);
    return check_launch("attn_decode_combine_kernel", stream);
}

}  // namespace

bool decode_attn_eligible(const rmm_attn_desc_t *d)
{
    return d->rho_t >= 1.0 && d->mask == nullptr && d->Lq <= kDecodeMaxRows && d->Dh <= 256 &&
           d->B * d->Hkv * ceil_div(d->Hq / d->Hkv * d->Lq, 8) * 16 < INT32_MAX;
}

size_t decode_attn_workspace_bytes(const rmm_attn_desc_t *d)
{
    const DecodeGrid g = decode_grid(d);
    return align_up((size_t)g.blocks * 2 * 8 * g.nt * (g.dh + 2) * 4, 256);
}

int launch_decode_attn(const rmm_attn_desc_t *d, int64_t kd, const void *Q, const void *K, const void *V, void *O, int32_t *idx_feat,
                       void *scratch, cudaStream_t stream)
{
    const DecodeGrid g = decode_grid(d);
    DecodeArgs a = {};
    a.q = static_cast<const __nv_bfloat16 *>(Q); a.k = static_cast<const __nv_bfloat16 *>(K);
    a.v = static_cast<const __nv_bfloat16 *>(V); a.o = static_cast<__nv_bfloat16 *>(O);
    a.q_sb = d->q_stride[0]; a.q_sh = d->q_stride[1]; a.q_sr = d->q_stride[2];
    a.k_sb = d->k_stride[0]; a.k_sh = d->k_stride[1]; a.k_sr = d->k_stride[2];
    a.v_sb = d->v_stride[0]; a.v_sh = d->v_stride[1]; a.v_sr = d->v_stride[2];
    a.o_sb = d->o_stride[0]; a.o_sh = d->o_stride[1]; a.o_sr = d->o_stride[2];
    a.Hkv = (int)d->Hkv; a.group = (int)(d->Hq / d->Hkv); a.Lq = (int)d->Lq; a.Lk = (int)d->Lk; a.Dh = (int)d->Dh;
    a.kd = (int)kd; a.causal = d->causal;
    a.rows = a.group * a.Lq; a.chunks = g.chunks; a.jobs = g.jobs; a.tiles = g.tiles; a.per_block = g.per_block;
    a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)d->Dh));
    a.idx_feat = idx_feat;
    a.part_o = static_cast<float *>(scratch);
    a.part_ml = a.part_o + (size_t)g.blocks * 2 * 8 * g.nt * g.dh;
    if (g.dh == 64) return g.nt == 1 ? launch_shape<64, 1, 8>(a, g.blocks, stream) : launch_shape<64, 2, 8>(a, g.blocks, stream);
    if (g.dh == 128) return g.nt == 1 ? launch_shape<128, 1, 8>(a, g.blocks, stream) : launch_shape<128, 2, 8>(a, g.blocks, stream);
    return g.nt == 1 ? launch_shape<256, 1, 4>(a, g.blocks, stream) : launch_shape<256, 2, 4>(a, g.blocks, stream);
}

}  // namespace rmm
