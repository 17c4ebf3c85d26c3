// Reduced attention for decode steps (paper Sec. 3.3 with rho_t = 1 and a handful of query rows): feature selection,
// S~ = Q[:, I] K[:, I]^T / sqrt(Dh), softmax and P V in one pass over the key/value cache, plus a small combine.
//
// Bound: HBM.  K and V are read once per 16 query rows that share a kv head, 4 bytes per (key, column); the kept features of a 2-byte row touch every
// 32-byte sector of it, so there is nothing to gain from gathering and the packed copies of K per query head that the
// prefill form makes would multiply the traffic (8 sequences x 32 / 8 heads x 4096 keys x 128: 80 us of packing and
// 97 us of a kernel whose 128-row tiles hold one row; 33 us
// for this form, 134 MB of caches; 16 sequences x 8192 keys, 537 MB: 93 us, 0.89 of the copy rate).  So the rows are read in
// place, the dropped features are zeros in Q, and everything else is arranged around bytes in flight:
//   - the keys of a (sequence, kv head) pair are cut into as many equal pieces as fill the GPU (decode_grid);
//   - inside a block every warp is on its own: it owns 16 keys of a tile and a private ring of 24 KB filled by
//     16-byte cp.async (about 150 KB in flight per SM), and no block barrier is met until the piece ends;
//   - all query rows that share a kv head (group x Lq) sit in the N = 8 columns of mma.m16n8k16 with the keys as M:
//     S^T = K Q^T and O^T = V^T P^T.  128-row tcgen05 tiles would be padding here: at 8 rows the products take 16
//     instructions per 16 keys and stay below a third of the time the bytes need.
// Softmax weights are taken against a per-row maximum that is refreshed only when exceeded by 2^40 (see
// attn_fused.cu), rounded once to bf16; row sums, maxima and O stay fp32.  Pieces of one head meet in a fixed order.
#include <math.h>

#include <type_traits>

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
    int tiles, pieces, per;      // key tiles per job, pieces it is cut into, tiles per piece
    float scale_log2;            // log2(e) / sqrt(Dh)
    int32_t *idx_feat;           // [B, Hq, kd] or NULL
    float *part_o, *part_ml;     // pieces > 1: [blocks][row tile][Dh padded], [blocks][row tile][2]
    unsigned *counters;          // an arrival counter per job, where its last block adds the pieces up
};

constexpr int kDecodeWarps = 4, kDecodeBlocks = 2;  // warps per block, blocks per SM

template <int DH, int NT>
struct DecodeShape {
    static constexpr int kRows = 8 * NT, kTileKeys = 16 * kDecodeWarps;
    static constexpr int kUnit = 16 * DH * 2;                                    // 16 keys of K or of V
    static constexpr int kUnits = 196608 / kDecodeBlocks / kDecodeWarps / kUnit;  // 192 KB of rings per SM: 3 (wide heads) to 12 a warp
    static constexpr int kRing = kUnits * kUnit;                                 // per warp
    static constexpr int kQPitch = DH + 8;
    static constexpr int kOffQ = kDecodeWarps * kRing, kOffKept = kOffQ + kRows * kQPitch * 2;
    static constexpr int kOffMl = kOffKept + kRows * (DH / 32) * 4, kSmem = kOffMl + kDecodeWarps * kRows * 8;
    static_assert(kRows * DH * 4 <= kRing, "the merge of the warps reuses the rings");
};

// A job of few pieces: whichever of its blocks comes last adds them up, in order.  (A second launch takes 3 us of the host.)  Out of
// line, so that the loop over the keys keeps its registers, and short: what runs once a call is fetched from memory.  A warp takes a
// row, or one or two rows' pieces are shared out among the four.
template <int DH, int NT>
__device__ __noinline__ void decode_meet(const DecodeArgs &a, uint8_t *smem)
{
    constexpr int WARPS = kDecodeWarps, kRows = 8 * NT, V = DH <= 128 ? 1 : 2;
    float *s_inv = reinterpret_cast<float *>(smem);              // [WARPS], the flag behind it
    float4 *s_acc = reinterpret_cast<float4 *>(smem) + 2;        // [warp][32 V]
    int *s_last = reinterpret_cast<int *>(smem) + WARPS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, pieces = a.pieces;
    const int64_t job = blockIdx.x / pieces;
    const int row0 = (int)(job % a.chunks) * kRows, nrows = min(kRows, a.rows - row0);
    const int64_t bh = job / a.chunks, b = bh / a.Hkv, hk = bh % a.Hkv;
    __syncthreads();
    if (tid == 0) {  // (fences are cumulative: one thread's stand for all that the barrier has ordered before it)
        __threadfence();
        *s_last = atomicInc(a.counters + job, (unsigned)pieces - 1u) == (unsigned)pieces - 1u;
        __threadfence();
    }
    __syncthreads();
    if (*s_last == 0) return;
    const int64_t slot0 = job * pieces;
    const int parts = nrows >= 3 ? 1 : WARPS / nrows;
    float4 acc[V];
    auto put = [&](int r, float inv) {
        const int row = row0 + r;
        __nv_bfloat16 *o = a.o + b * a.o_sb + (hk * a.group + row / a.Lq) * a.o_sh + (int64_t)(row % a.Lq) * a.o_sr;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int c = (i * 32 + lane) * 4;
            if (c < a.Dh) {   // Dh and the strides are multiples of 8
                const __nv_bfloat162 lo = __floats2bfloat162_rn(acc[i].x * inv, acc[i].y * inv), hi = __floats2bfloat162_rn(acc[i].z * inv, acc[i].w * inv);
                *reinterpret_cast<uint2 *>(o + c) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
            }
        }
    };
    for (int u = warp; u < nrows * parts; u += WARPS) {
        const int r = u / parts;
        const float *pm = a.part_ml + ((slot0 + lane) * kRows + r) * 2;    // lane p looks after piece p
        const float mw = lane < pieces ? __ldcg(pm) : -INFINITY, lw = lane < pieces ? __ldcg(pm + 1) : 0.f;
        const float4 *src = reinterpret_cast<const float4 *>(a.part_o + (slot0 * kRows + r) * DH) + lane;
        float mx = mw;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
        const float f = mw > -INFINITY ? ptx::ex2(mw - mx) : 0.f;   // (a piece without a key has zeros for its sums)
        float lsum = f * lw;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, d);
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll (V == 1 ? 8 : 4)
        for (int p = u % parts; p < pieces; p += parts) {
            const float fp = __shfl_sync(0xffffffffu, f, p);
#pragma unroll
            for (int i = 0; i < V; ++i)
                if ((i * 32 + lane) * 4 < DH) {
                    const float4 x = __ldcg(src + (int64_t)p * kRows * (DH / 4) + i * 32);
                    acc[i].x += fp * x.x; acc[i].y += fp * x.y; acc[i].z += fp * x.z; acc[i].w += fp * x.w;
                }
        }
        const float inv = lsum == 0.f ? 0.f : 1.f / lsum;  // 0: the row sees no key; a NaN stays one
        if (parts == 1) {
            put(r, inv);
        } else {
#pragma unroll
            for (int i = 0; i < V; ++i) s_acc[(u * V + i) * 32 + lane] = acc[i];
            if (lane == 0) s_inv[r] = inv;
        }
    }
    if (parts == 1) return;
    __syncthreads();
    if (warp >= nrows) return;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < parts; ++s) {
            const float4 x = s_acc[((warp * parts + s) * V + i) * 32 + lane];
            acc[i].x += x.x; acc[i].y += x.y; acc[i].z += x.z; acc[i].w += x.w;
        }
    }
    put(warp, s_inv[warp]);
}

template <int DH, int NT, bool MEET>
__global__ void __launch_bounds__(kDecodeWarps * 32, kDecodeBlocks) attn_decode_kernel(const __grid_constant__ DecodeArgs a)
{
    using S = DecodeShape<DH, NT>;
    constexpr int WARPS = kDecodeWarps, kRows = S::kRows, U = S::kUnits, CPR = DH / 8;  // 16-byte vectors per row
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const uint32_t ring = ptx::smem_u32(smem) + warp * S::kRing;
    __nv_bfloat16 *qs = reinterpret_cast<__nv_bfloat16 *>(smem + S::kOffQ);
    uint32_t *kept = reinterpret_cast<uint32_t *>(smem + S::kOffKept);   // [row][DH / 32] bit masks of the kept features
    float *ml = reinterpret_cast<float *>(smem + S::kOffMl);             // [warp][row][2]
    pdl_wait();

    const int64_t job = blockIdx.x / a.pieces;
    const int ta = (int)(blockIdx.x % a.pieces) * a.per, tb = min(a.tiles, ta + a.per);
    const int chunk = (int)(job % a.chunks);
    const int64_t bh = job / a.chunks, b = bh / a.Hkv, hk = bh % a.Hkv;
    const int row0 = chunk * kRows, nrows = min(kRows, a.rows - row0);
    const __nv_bfloat16 *kp = a.k + b * a.k_sb + hk * a.k_sh, *vp = a.v + b * a.v_sb + hk * a.v_sh;
    const int n_sub = tb - ta;  // this warp's 16-key steps

    auto load = [&](int u) {  // unit u (K of step u / 2, then V of it) into ring entry u % U; always one commit group
        if (u < 2 * n_sub) {
            const uint32_t dst = ring + (u % U) * S::kUnit;
            const int key0 = (ta + (u >> 1)) * S::kTileKeys + warp * 16;
            const __nv_bfloat16 *src = u & 1 ? vp : kp;
            const int64_t pitch = u & 1 ? a.v_sr : a.k_sr;
            const int c = lane % CPR;
#pragma unroll
            for (int i = 0; i < 16 * CPR / 32; ++i) {
                const int r = lane / CPR + i * (32 / CPR);
                const bool live = key0 + r < a.Lk && c * 8 < a.Dh;
                ptx::cp_async_16(dst + r * (DH * 2) + ((c ^ (r & 7)) << 4), live ? src + (int64_t)(key0 + r) * pitch + c * 8 : a.k, live ? 16u : 0u);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto landed = [&]() {  // the oldest unit is there for every lane, and every lane is done with the entry refilled next
        asm volatile("cp.async.wait_group %0;" ::"n"(U - 2) : "memory");
        __syncwarp();
    };
#pragma unroll
    for (int u = 0; u < U - 1; ++u) load(u);

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
                    e += (double)(x * x);  // exact for magnitudes from 2^-63 to 2^64, as in every score pass
                }
            u[i] = f < a.Dh ? sel::key_image((float)e) : 0u;  // 0: below every key
        }
        uint32_t tau = 0;  // largest value that at least kd keys reach: the image of the kd-th largest key
#pragma unroll 1
        for (int bit = 30; bit >= 0; bit -= 2) {  // two bits a turn: three independent counts
            int c[3] = {0, 0, 0};
#pragma unroll
            for (int i = 0; i < DH / 32; ++i)
#pragma unroll
                for (int v = 0; v < 3; ++v) c[v] += u[i] >= (tau | ((unsigned)(v + 1) << bit)) ? 1 : 0;
            unsigned digit = 0;
#pragma unroll
            for (int v = 0; v < 3; ++v) digit += __reduce_add_sync(0xffffffffu, c[v]) >= a.kd ? 1u : 0u;
            tau |= digit << bit;
        }
        int c = 0;
#pragma unroll
        for (int i = 0; i < DH / 32; ++i) c += u[i] > tau ? 1 : 0;
        int need_eq = a.kd - __reduce_add_sync(0xffffffffu, c), at = 0;
        const int r_lo = max(row0, h * a.Lq), r_hi = min(row0 + nrows, (h + 1) * a.Lq);
        // the block that holds a head's first row and first key writes its index list
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
        landed();
        load(2 * n + U - 1);
        const uint32_t kst = ring + (2 * n % U) * S::kUnit;
        const int key0 = (ta + n) * S::kTileKeys + warp * 16;
        float s[NT][4], s2[NT][4];  // two chains of dependent products
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[nt][e] = s2[nt][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
            uint32_t ka[4];
            ptx::ldmatrix_x4(ka, kst + k_lane + (((2 * ks + (lane >> 4)) ^ k_x) << 4));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) ptx::mma_bf16_16816(ks & 1 ? s2[nt] : s[nt], ka, qf[nt][ks][0], qf[nt][ks][1]);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[nt][e] += s2[nt][e];
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
            pb[nt][0] = ptx::transpose8x8(*reinterpret_cast<uint32_t *>(&x));  // (key g, rows 2t) -> (row g, keys 2t)
            pb[nt][1] = ptx::transpose8x8(*reinterpret_cast<uint32_t *>(&y));
        }
        landed();
        load(2 * n + U);
        const uint32_t vst = ring + ((2 * n + 1) % U) * S::kUnit;
#pragma unroll
        for (int mt = 0; mt < DH / 16; ++mt) {
            uint32_t va[4];
            ptx::ldmatrix_x4_trans(va, vst + v_row * (DH * 2) + (((2 * mt + ((lane >> 3) & 1)) ^ (v_row & 7)) << 4));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) ptx::mma_bf16_16816(o[nt][mt], va, pb[nt][0], pb[nt][1]);
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
            for (int e = 0; e < 4; ++e)
                if (nt * 8 + 2 * t + (e & 1) < nrows) mine[(nt * 8 + 2 * t + (e & 1)) * DH + mt * 16 + g + (e >> 1) * 8] = o[nt][mt][e];
    __syncthreads();
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
        if (a.pieces == 1) {
            const int row = row0 + r;
            if (c < a.Dh)
                a.o[b * a.o_sb + (hk * a.group + row / a.Lq) * a.o_sh + (int64_t)(row % a.Lq) * a.o_sr + c] =
                    __float2bfloat16_rn(lsum == 0.f ? 0.f : sum * (1.f / lsum));  // (0: the row sees no key; a NaN stays one)
        } else {
            a.part_o[((int64_t)blockIdx.x * kRows + r) * DH + c] = sum;
            if (c == 0) {
                a.part_ml[((int64_t)blockIdx.x * kRows + r) * 2] = mx;
                a.part_ml[((int64_t)blockIdx.x * kRows + r) * 2 + 1] = lsum;
            }
        }
    }
    if constexpr (MEET) decode_meet<DH, NT>(a, smem);
}

// Jobs cut into pieces: a block per row; its warps take every fourth piece each, and meet in order.
constexpr int kCombineWarps = 4;
template <int DH, int NT>
__global__ void __launch_bounds__(kCombineWarps * 32) attn_decode_combine_kernel(const DecodeArgs a)
{
    constexpr int kRows = 8 * NT;
    __shared__ float s_acc[kCombineWarps][DH], s_l[kCombineWarps], s_m[kCombineWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();
    const int64_t job = blockIdx.x / kRows;
    const int r = (int)(blockIdx.x % kRows), row = (int)(job % a.chunks) * kRows + r;
    if (row >= a.rows) return;
    const int64_t slot0 = job * a.pieces;
    float mx = -INFINITY;
    for (int p = threadIdx.x; p < a.pieces; p += kCombineWarps * 32) mx = fmaxf(mx, a.part_ml[((slot0 + p) * kRows + r) * 2]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
    if (lane == 0) s_m[warp] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kCombineWarps; ++w) mx = fmaxf(mx, s_m[w]);
    float acc[DH / 32], lsum = 0.f;
#pragma unroll
    for (int i = 0; i < DH / 32; ++i) acc[i] = 0.f;
#pragma unroll 4
    for (int p = warp; p < a.pieces; p += kCombineWarps) {
        const int64_t s = (slot0 + p) * kRows + r;
        const float mw = a.part_ml[s * 2], f = mw > -INFINITY ? ptx::ex2(mw - mx) : 0.f;
        lsum += f * a.part_ml[s * 2 + 1];
#pragma unroll
        for (int i = 0; i < DH / 32; ++i) {
            const float x = a.part_o[s * DH + i * 32 + lane];
            acc[i] += mw > -INFINITY ? f * x : 0.f;
        }
    }
#pragma unroll
    for (int i = 0; i < DH / 32; ++i) s_acc[warp][i * 32 + lane] = acc[i];
    if (lane == 0) s_l[warp] = lsum;
    __syncthreads();
    lsum = 0.f;
#pragma unroll
    for (int w = 0; w < kCombineWarps; ++w) lsum += s_l[w];
    const float inv = lsum == 0.f ? 0.f : 1.f / lsum;  // 0: the row sees no key; a NaN stays one
    const int64_t bh = job / a.chunks, b = bh / a.Hkv, hk = bh % a.Hkv;
    __nv_bfloat16 *o = a.o + b * a.o_sb + (hk * a.group + row / a.Lq) * a.o_sh + (int64_t)(row % a.Lq) * a.o_sr;
    for (int c = threadIdx.x; c < a.Dh; c += kCombineWarps * 32) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < kCombineWarps; ++w) sum += s_acc[w][c];
        o[c] = __float2bfloat16_rn(sum * inv);
    }
}

struct DecodeGrid {
    int dh, nt, chunks, tiles, pieces, per;
    int64_t jobs, blocks;
};

// Pieces per job: the least (rounds of blocks over the GPU) x (steps of a block and about six more for what it spends
// outside them: feature selection, first loads, meeting of the warps).  Equal pieces of one job per block: cutting the
// joint axis of all jobs into exactly equal shares instead made blocks work on two jobs, one after the other with the
// loads drained in between (8 sequences x 8 kv heads x 4096 keys: 41 us a call against 33).
DecodeGrid decode_grid(const rmm_attn_desc_t *d)
{
    DecodeGrid g;
    const int64_t rows = d->Hq / d->Hkv * d->Lq, slots = (int64_t)sm_count() * kDecodeBlocks;
    g.dh = d->Dh <= 64 ? 64 : (d->Dh <= 128 ? 128 : 256);
    g.tiles = (int)ceil_div(d->Lk, 16 * kDecodeWarps);
    // Sixteen rows a block read the cache half as often as eight.  Where even blocks of one tile and eight rows leave the GPU
    // room, what a block spends on the feature sets of its heads is what counts, and eight rows have half of it (32 heads of
    // 256 on one kv head, one query, 512 keys: 52 us a call with sixteen, 32 with eight).
    g.nt = rows <= 8 || d->B * d->Hkv * ceil_div(rows, 8) * g.tiles <= slots ? 1 : 2;
    g.chunks = (int)ceil_div(rows, 8 * g.nt);
    g.jobs = d->B * d->Hkv * g.chunks;
    int64_t best = INT64_MAX;
    for (int64_t rounds = 0; rounds <= 2; ++rounds) {  // whole jobs, or the most pieces that make one or two rounds
        int64_t s = rounds * slots / g.jobs;
        s = s < 1 ? 1 : (s > g.tiles ? g.tiles : s);
        const int64_t per = ceil_div(g.tiles, s), cost = ceil_div(g.jobs * ceil_div(g.tiles, per), slots) * (per + 6);
        if (cost < best) {
            best = cost;
            g.per = (int)per;
            g.pieces = (int)ceil_div(g.tiles, per);
        }
    }
    g.blocks = g.jobs * g.pieces;
    return g;
}

template <int DH, int NT, bool MEET>
int launch_shape(const DecodeArgs &a, const DecodeGrid &g, cudaStream_t stream)
{
    using S = DecodeShape<DH, NT>;
    auto kern = attn_decode_kernel<DH, NT, MEET>;
    static PerDeviceOnce configured;
    if (cudaError_t e = configured.smem(S::kSmem, kern)) return fail(RMM_ERR_CUDA, "attn_decode: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    prof_begin("attn_decode_kernel", stream);
    launch_kernel(kern, dim3((unsigned)g.blocks), dim3(kDecodeWarps * 32), S::kSmem, stream, 1, a);
    int rc = check_launch("attn_decode_kernel", stream);
    if (MEET || rc != RMM_OK || g.pieces == 1) return rc;
    prof_begin("attn_decode_combine_kernel", stream);
    launch_kernel(attn_decode_combine_kernel<DH, NT>, dim3((unsigned)(g.jobs * S::kRows)), dim3(kCombineWarps * 32), 0, stream, 1, a);
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
    return g.pieces == 1 ? 0 : align_up((size_t)g.blocks * 8 * g.nt * (g.dh + 2) * 4, 256);
}

int launch_decode_attn(const rmm_attn_desc_t *d, int64_t kd, const void *Q, const void *K, const void *V, void *O, int32_t *idx_feat,
                       void *scratch, unsigned *counters, cudaStream_t stream)
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
    a.rows = a.group * a.Lq; a.chunks = g.chunks; a.tiles = g.tiles; a.pieces = g.pieces; a.per = g.per;
    a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)d->Dh));
    a.idx_feat = idx_feat;
    a.part_o = static_cast<float *>(scratch);
    a.part_ml = a.part_o + (size_t)g.blocks * 8 * g.nt * g.dh;
    // Where the last block of a job adds the pieces up (each job then has its counter; the header's last four belong to the
    // products).  Measured on 420 shapes against a launch of its own, through the binding and as a replayed graph.  Heads of up to
    // 128: the meeting takes 0.5 to 1.5 us of the GPU more than that launch, which starts early, and saves 3.5 us of the host.
    // So it is for short pieces of few rows, whose calls the host bounds (four tiles of heads of 128, eight of 64, up to four rows:
    // 17.9 -> 14.5 to 16.4 us a call, 10 to 14 -> 11 to 15 replayed); longer ones gain nothing (level or slower, 7 % replayed), eight
    // rows lose 7 to 16 %.  Heads of 256, whose second launch starts late: 2 to 13 % faster either way, but for short pieces of more
    // than four rows (6 % slower).
    const int64_t rows = a.rows < 8 * g.nt ? a.rows : 8 * g.nt;
    const bool worth = g.dh <= 128 ? rows <= kDecodeWarps && g.per * g.dh <= 512 : rows <= kDecodeWarps || g.per >= 6;
    const bool meet = g.pieces > 1 && worth && g.per <= 16 && g.pieces * ceil_div(rows, kDecodeWarps) <= 16 && g.jobs <= kHeaderCounters - 4;
    if (meet) a.counters = counters;
    auto launch = [&](auto dh, auto nt) {
        constexpr int kDh = decltype(dh)::value, kNt = decltype(nt)::value;
        return meet ? launch_shape<kDh, kNt, true>(a, g, stream) : launch_shape<kDh, kNt, false>(a, g, stream);
    };
    using std::integral_constant;
    auto launch_dh = [&](auto dh) { return g.nt == 1 ? launch(dh, integral_constant<int, 1>{}) : launch(dh, integral_constant<int, 2>{}); };
    if (g.dh == 64) return launch_dh(integral_constant<int, 64>{});
    if (g.dh == 128) return launch_dh(integral_constant<int, 128>{});
    return launch_dh(integral_constant<int, 256>{});
}

}  // namespace rmm
