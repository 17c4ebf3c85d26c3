// Fused reduced attention (paper Sec. 3.3): S~ = Q[:, I] K[:, I]^T / sqrt(Dh) on packed operands, softmax, and the
// product with V, with S~ and P never leaving the SM (S~ tiles in tensor memory, P tiles in shared memory, O
// accumulated in tensor memory).  One kernel skeleton, four modes:
//
//   FULL      rho_t = 1:  O = softmax(S~ + mask) V in one pass over the keys.
//   STATS     rho_t < 1, sweep 1:  lse_i = log2 sum_t 2^(x_it) per query row (x = S~ * log2(e) / sqrt(Dh)), nothing else.
//   ENERGY    rho_t < 1, sweep 2:  token scores a_t^2 = sum_i P_it^2 with P_it = bf16(2^(x_it - lse_i)), the attention
//             weight rounded once to bf16 as the paper scores it.  The roles are swapped (rows = keys, tiles of
//             queries stream past), so that a thread owns one key and sums over all queries in a register: no
//             cross-thread reduction and no atomics.
//   GATHERED  rho_t < 1, sweep 3:  O = P[:, T] V[T, :] on the kept keys (K[T], V[T] packed), P_it = bf16(2^(x_it -
//             lse_i)) against the full-row normaliser of sweep 1: no renormalisation (Sec. 3.3).
//
// One block owns 256 rows of one head as two groups of 128 and walks the other axis in tiles of 128; both groups
// consume the same tiles, so each crosses from L2 to the SM once per 256 rows.  Per tile and group: S~ on the tensor
// cores (kd of the Dh features; 128 columns of tensor memory, released as soon as the softmax warps hold the tile in
// registers); one thread per row takes p = 2^(x - m) in two chunks of 64 columns, rounds it once to bf16 and writes it
// to shared memory as the A operand of O += P V.  In FULL mode m is the row maximum seen so far, refreshed only when
// the new maximum exceeds it by more than kGrowLimit: then l and the O row in tensor memory are multiplied by
// 2^(m_old - m_new); the epilogue divides by l.  The row's largest p thus ends between 1 and 2^40, so that sums of P V are no
// smaller than V and stay in fp32's range for |V| up to 2^87 / Lk.  (A reference 40 above the maximum saves most of the
// rescales, 8 us of 132 on 32 heads x 4096 x 128, but hands the small end of V's range to the subnormal numbers: values of
// 1e-33 came out a few percent off, smaller ones as zero.)  The paper rounds the normalised weight P
// to bf16; in FULL mode the rounded quantity is p = P * l * 2^(m_row - m), the same weight up to a per-row fp32
// factor, so O differs by bf16 rounding noise only (nothing is decided from P when rho_t = 1); the modes that score or
// drop tokens round the normalised P itself.  The row sum takes each tile's largest weight as it was rounded: a row that one
// key dominates then gets that key's value back whatever the weight's scale.
// Warp 0 feeds TMA, warps 2-5 and 6-9 are the softmax/epilogue warps of the two groups (every scheduler has two of
// them to switch between), and one thread of warp 1 and of warp 10 issues the tcgen05.mma of group 0 and 1: a single
// issuing thread for both groups was the bottleneck.  Every wait is bounded.
#include <float.h>
#include <math.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace rmm {
namespace {

using namespace ptx;

enum { MODE_FULL = 0, MODE_STATS = 1, MODE_ENERGY = 2, MODE_GATHERED = 3 };

constexpr int FM = 128, FN = 128;     // rows per group, columns per step
constexpr int kGroups = 2;
constexpr int kFusedThreads = 64 + kGroups * 128 + 32;  // producer, MMA issuer 0, 8 softmax warps, MMA issuer 1
constexpr int kMmaWarp1 = 10;
constexpr int kKvStages = 3;
constexpr int kQChunk = 16384;        // row-side chunk: 128 rows x 64 features (128 bytes per row, 128-byte swizzle)
constexpr int kQTile = 2 * kQChunk;   // up to 128 kept features
constexpr int kKvChunk = 16384;       // column-side chunk: 128 keys x 64 features (or 128 keys x 64 columns of V)
constexpr int kKvTile = 2 * kKvChunk; // ring entry: a K tile (up to 128 kept features) or a V tile (up to 128 columns)
constexpr int kPChunk = 16384;        // P chunk: 128 rows x 64 keys (128 bytes per row, 128-byte swizzle)
constexpr int kPTile = 2 * kPChunk;   // P tile: 128 rows x 128 keys
constexpr int kOffQ = 0, kOffKv = kGroups * kQTile, kOffP = kOffKv + kKvStages * kKvTile, kOffBar = kOffP + kGroups * kPTile;
constexpr int kFusedSmem = kOffBar + 512;
constexpr int kTmemCols = 512;        // per group: S~ (128 columns); then O (128 columns per group)
constexpr uint32_t kTmemO = kGroups * FN;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kGrowLimit = 40.f;    // log2 of the largest p taken against a stale maximum

// Debug aid (-DRMM_ATTN_STAMPS): clocks spent per phase by the MMA issuer of group 0 and by one softmax warp of
// block 0, summed over the launch and read back with rmm_debug_attn_stamps().
#ifdef RMM_ATTN_STAMPS
__device__ unsigned long long g_astamps[16];
#define ASTAMP_DECL(cond) long long acc_[8] = {0, 0, 0, 0, 0, 0, 0, 0}, last_ = clock64(); const bool stamp_on = (cond)
#define ASTAMP(i) do { long long t_ = clock64(); acc_[i] += t_ - last_; last_ = t_; } while (0)
#define ASTAMP_FLUSH(off) do { if (stamp_on) for (int k_ = 0; k_ < 8; ++k_) atomicAdd(&g_astamps[(off) + k_], (unsigned long long)acc_[k_]); } while (0)
#else
#define ASTAMP_DECL(cond)
#define ASTAMP(i)
#define ASTAMP_FLUSH(off)
#endif

// "Rows" are what a thread owns (queries; keys in ENERGY mode), "columns" what streams past in tiles.
struct FusedArgs {
    int64_t heads, Lr, Lc;       // rows and columns per head (GATHERED: Lc = kept keys)
    int64_t diag;                // Lk - Lq of the unpacked problem: query i sees key t iff t <= i + diag (causal)
    int kd, Dh, causal;
    int groups;                  // groups of 128 rows a block owns: 2, or 1 where that keeps more SMs busy (see block_groups)
    int64_t v_off, v_div;        // V batch entry of head h = (h + v_off) / v_div
    __nv_bfloat16 *O;
    int64_t o_sh, o_sr;          // element strides of O: head, row
    float *lse;                  // [heads, lse_ld] negated log2-domain normalisers: written by STATS, read by ENERGY / GATHERED
    int64_t lse_ld;              // multiple of 64, >= Lq
    float *energy;               // ENERGY: [heads, Lr] squared token scores
    const int32_t *tok;          // GATHERED: [heads, Lc] kept key positions, ascending
    float scale_log2;            // (1 / sqrt(Dh)) * log2(e)
    MaskView mask;               // MASK: the caller's additive mask
    const uint8_t *tile_kind;    // MASK: what the mask does to a 128 x 128 tile: [plane][row block][tile], see mask_tiles_kernel
    int64_t kind_rb, kind_ld;    // row blocks per plane (even), bytes per row block (a multiple of 8)
    int *status;
    unsigned long long wait_ns;  // bound of every device-side wait
    int withhold;                // test switch: block 0 never requests its first key tile
};

// What the additive mask does to each tile of 128 queries x 128 keys, once per mask plane (the heads that share a plane
// share the answer): hides it all (the tile is skipped like one beyond the causal diagonal), leaves it alone (the
// ordinary softmax step), or has to be added.  Padding, causal, block and window masks are nearly all of the first
// two kinds, and the additions were what bound the masked kernel: each thread reads its own row of the mask, 32 rows a
// load.  2 sequences x 16 heads x 2048 x 128, padded: 2 x 244 us with every tile added, 52 us in one launch with this
// pass (6 us) in front; a mask whose every value is added: 254 -> 136 us a call on 16 heads x 2048.
// Bound by reading the mask once; a warp stops reading a tile once it knows that its values have to be added.
// Only -inf hides a key.  A tile of the lowest finite values (masks are written with them too) is skipped all the same where
// each of its rows sees some ordinary key, next to which such values weigh exactly nothing; a row that sees no other keep
// them (its weights are then equal, whatever the logits: fp32 sums).
enum { TILE_HIDDEN = 0, TILE_CLEAR = 1, TILE_ADD = 2 };
constexpr int kMaskThreads = 128;
constexpr float kMaskLow = -2e38f, kMaskOrdinary = -1e38f;  // 1e38 apart: e^-1e38 = 0 for any sum of logits below that

struct MaskTileArgs {
    MaskView mask;
    int64_t Lq, Lk, diag;
    int causal, vec;   // vec: rows are 16-byte aligned
    uint8_t *kind;
    int64_t kind_rb, kind_ld;
    int behind_heads;  // pack_heads_kernel is the launch before
};

__global__ void __launch_bounds__(kMaskThreads) mask_tiles_kernel(const MaskTileArgs a)
{
    __shared__ int s_seen[kMaskThreads / 32];
    static_assert(kMaskThreads == FM, "a thread per row of the tile");
    // pack_heads_kernel started this one after everything before itself was complete, the mask included, and nothing here reads what
    // it writes: the two run side by side, and this one waits before it ends, so that the next kernel finds both complete (2 x 16
    // heads x 2048, padded: 81 -> 76.5 us a call).
    if (a.behind_heads) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    else pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned rb = blockIdx.x / (unsigned)a.kind_ld, tile = blockIdx.x % (unsigned)a.kind_ld;
    const int64_t t0 = (int64_t)tile * FN, r0 = (int64_t)rb * FM, plane = blockIdx.z;
    const float *m = a.mask.p + (plane / a.mask.plane_heads) * a.mask.sb + (plane % a.mask.plane_heads) * a.mask.sh;
    const int64_t rows = a.mask.sr == 0 ? 1 : min((int64_t)FM, a.Lq - r0);   // one row stands for all of them
    const bool beyond = t0 >= a.Lk || r0 >= a.Lq || (a.causal && t0 > min(a.Lq, r0 + FM) - 1 + a.diag);
    bool some = false, live = false, low = false;  // some value is not zero; is not low; is low but does not hide
    auto look = [&](float v) {
        some |= !(v == 0.f);
        live |= !(v <= kMaskLow);
        low |= v <= kMaskLow && v > -INFINITY;
    };
    for (int64_t rr = warp * 8; rr < rows && !beyond; rr += kMaskThreads / 32 * 8) {
        float4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // rows and columns past the end repeat the tile's first value
            const float *row = m + (r0 + (rr + i < rows ? rr + i : 0)) * a.mask.sr + t0;
            const int64_t c = t0 + lane * 4;
            if (a.vec && c + 3 < a.Lk) {
                v[i] = __ldg(reinterpret_cast<const float4 *>(row) + lane);
            } else {
                v[i].x = __ldg(row + (c < a.Lk ? lane * 4 : 0));
                v[i].y = __ldg(row + (c + 1 < a.Lk ? lane * 4 + 1 : 0));
                v[i].z = __ldg(row + (c + 2 < a.Lk ? lane * 4 + 2 : 0));
                v[i].w = __ldg(row + (c + 3 < a.Lk ? lane * 4 + 3 : 0));
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            look(v[i].x);
            look(v[i].y);
            look(v[i].z);
            look(v[i].w);
        }
        if (__any_sync(0xffffffffu, some) && __any_sync(0xffffffffu, live)) break;
    }
    const bool w_some = __any_sync(0xffffffffu, some), w_live = __any_sync(0xffffffffu, live), w_low = __any_sync(0xffffffffu, low);
    if (lane == 0) s_seen[warp] = (w_some ? 1 : 0) | (w_live ? 2 : 0) | (w_low ? 4 : 0);
    __syncthreads();
    int seen = 0;
#pragma unroll
    for (int w = 0; w < kMaskThreads / 32; ++w) seen |= s_seen[w];
    int kind = seen & 2 ? (seen & 1 ? TILE_ADD : TILE_CLEAR) : TILE_HIDDEN;
    if ((seen & 6) == 4) {  // (block-uniform) low values only: does every row see an ordinary key?
        // a row per thread looks at four keys: the first, the last that it sees and two between; what that leaves open is
        // read row by row, until a row has no such key
        const int64_t r = r0 + threadIdx.x, visible = a.causal ? min(a.Lk, r + a.diag + 1) : a.Lk;
        const float *row = m + r * a.mask.sr;
        bool open = r < a.Lq && visible > 0;
        if (open) {
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = __ldg(row + (visible - 1) * i / 3);
            open = !(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])) >= kMaskOrdinary);
        }
        bool lone = false;
        for (unsigned left = __ballot_sync(0xffffffffu, open); left != 0 && !lone; left &= left - 1) {
            const int src = __ffs(left) - 1;
            const int64_t rr = r0 + warp * 32 + src, vis = a.causal ? min(a.Lk, rr + a.diag + 1) : a.Lk;
            const float *p = m + rr * a.mask.sr;
            bool ordinary = false;
            for (int64_t c = 0; c < vis && !ordinary; c += 256) {
                float top = -INFINITY;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (c + 32 * i + lane < vis) top = fmaxf(top, __ldg(p + c + 32 * i + lane));
                ordinary = __any_sync(0xffffffffu, top >= kMaskOrdinary);
            }
            lone = !ordinary;
        }
        if (__syncthreads_or(lone)) kind = TILE_ADD;
    }
    if (threadIdx.x == 0) a.kind[(plane * a.kind_rb + rb) * a.kind_ld + tile] = (uint8_t)kind;
    if (a.behind_heads) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// O_TILES: O leaves by tile stores (GATHERED, where a tensor map describes O: no negative strides).  Both forms in one
// kernel, chosen at run time, cost it 3 % (32 heads x 3001 x 128 73.7 -> 75.8 us).
template <int MODE, bool MASK, bool O_TILES>
__global__ void __launch_bounds__(kFusedThreads, 1)
fused_attn_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                  const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, FusedArgs a)
{
    constexpr bool kHasV = MODE == MODE_FULL || MODE == MODE_GATHERED;  // P tiles, P V products and an O accumulator
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    uint8_t *base_ptr = smem_raw;
    if (base & 1023u) {  // the swizzled tiles need a 1024-byte aligned window; nothing has been allocated yet
        if (threadIdx.x == 0) atomicExch(a.status, (int)RMM_ERR_CUDA);
        return;
    }
    const uint32_t bar0 = base + kOffBar;
    // barriers: q_full, q_empty; per group s_full[2], s_empty[2], p_full, p_empty, o_full, o_empty; kv_full[], kv_empty[]
    const uint32_t q_full = bar0, q_empty = bar0 + 8;
    auto s_full = [&](int g, int i) { return bar0 + 64u * (g + 1) + 8u * i; };
    auto s_empty = [&](int g, int i) { return bar0 + 64u * (g + 1) + 16u + 8u * i; };
    auto p_full = [&](int g) { return bar0 + 64u * (g + 1) + 32u; };
    auto p_empty = [&](int g) { return bar0 + 64u * (g + 1) + 40u; };
    auto o_full = [&](int g) { return bar0 + 64u * (g + 1) + 48u; };
    auto o_empty = [&](int g) { return bar0 + 64u * (g + 1) + 56u; };
    auto kv_full = [&](int s) { return bar0 + 256u + 8u * s; };
    auto kv_empty = [&](int s) { return bar0 + 256u + 8u * (kKvStages + s); };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + kOffBar + 16);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + kOffBar + 24);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_q) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
        if constexpr (kHasV) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
            if constexpr (O_TILES) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_o) : "memory");
        }
    }
    if (threadIdx.x == 0) {
        mbar_init(q_full, 1);
        mbar_init(q_empty, kGroups);
        for (int s = 0; s < kKvStages; ++s) { mbar_init(kv_full(s), 1); mbar_init(kv_empty(s), kGroups); }
        for (int g = 0; g < kGroups; ++g) {
            for (int i = 0; i < 2; ++i) { mbar_init(s_full(g, i), 1); mbar_init(s_empty(g, i), 4); }
            mbar_init(p_full(g), 4);
            mbar_init(p_empty(g), 1);
            mbar_init(o_full(g), 1);
            mbar_init(o_empty(g), 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc<1>(smem_u32(const_cast<uint32_t *>(tmem_slot)), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();

    const int kq = (a.kd + 63) / 64, nv = (a.Dh + 63) / 64;       // 64-column chunks of Q/K and of V
    const int rows_blk = a.groups * FM, blocks_r = (int)((a.Lr + rows_blk - 1) / rows_blk);
    const int64_t items = a.heads * blocks_r;
    // kept keys (GATHERED) with position <= limit (the same for the whole warp): T is ascending.  The lanes look at 32 places at a
    // time: every item starts with four such searches one after the other, and a memory latency per halving was a fifth of the kernel.
    auto kept_upto = [&](const int32_t *T, int64_t limit) -> int64_t {
        int64_t lo = 0, hi = a.Lc;
        while (lo < hi) {
            const int64_t step = (hi - lo + 31) / 32, at = lo + (lane + 1) * step - 1;  // the last place of the lane's part
            const int whole = __popc(__ballot_sync(0xffffffffu, at < hi && (int64_t)__ldg(T + at) <= limit));
            lo += whole * step;
            hi = min(hi, lo + step - 1);
        }
        return lo;
    };
    // the same for limit + lane
    auto kept_upto_rows = [&](const int32_t *T, int64_t limit) -> int64_t {
        const int64_t first = kept_upto(T, limit);
        const int64_t ahead = first + lane < a.Lc ? (int64_t)__ldg(T + first + lane) - limit : 32;   // at least 1; 31 of them at most matter
        const unsigned marks = __reduce_or_sync(0xffffffffu, ahead < 32 ? 1u << ahead : 0u);
        return first + __popc(marks & (0xffffffffu >> (31 - lane)));
    };
    // Column tiles [jb, je) that the 128 rows starting at r0 need (empty: jb = je = 0).
    auto tile_range = [&](int64_t head, int64_t r0, int *jb, int *je) {
        *jb = 0;
        *je = 0;
        if (r0 >= a.Lr) return;
        if constexpr (MODE == MODE_ENERGY) {
            // row = key t, visible to the queries i >= t - diag: the group's first row reaches furthest back
            const int64_t first = a.causal ? max((int64_t)0, r0 - a.diag) : 0;
            if (first >= a.Lc) return;
            *jb = (int)(first / FN);
            *je = (int)((a.Lc + FN - 1) / FN);
        } else if constexpr (MODE == MODE_GATHERED) {
            const int64_t n = a.causal ? kept_upto(a.tok + head * a.Lc, min(a.Lr - 1, r0 + FM - 1) + a.diag) : a.Lc;
            *je = (int)((n + FN - 1) / FN);
        } else {
            const int64_t last = a.causal ? min(a.Lc - 1, r0 + FM - 1 + a.diag) : a.Lc - 1;
            *je = last < 0 ? 0 : (int)(last / FN) + 1;
        }
    };
    // Tiles the block walks: the union over its groups (a group's range is a prefix or a suffix of it).
    auto block_range = [&](int64_t head, int64_t r0, int *jb, int *je) {
        int b0, e0, b1, e1;
        tile_range(head, r0, &b0, &e0);
        if (a.groups == 1) { *jb = b0; *je = e0; return; }
        tile_range(head, r0 + FM, &b1, &e1);
        if (e0 <= b0) { *jb = b1; *je = e1; }
        else if (e1 <= b1) { *jb = b0; *je = e0; }
        else { *jb = min(b0, b1); *je = max(e0, e1); }
    };
    // MASK: the tiles that are not hidden from the rows of one group, or of both (tiles past a group's causal range are hidden
    // in its list).  Eight tiles' kinds are held at a time, so a step costs a load only every eight tiles.
    struct Tiles {
        const uint8_t *k0, *k1;     // kinds of the group, and of the other one or NULL
        int at;                     // tiles 8 at .. 8 at + 7 are in `w`
        unsigned long long w;
        __device__ __forceinline__ int next(int j, int je)  // the first tile from j on, before je, that is not hidden, else je
        {
            if constexpr (MASK) {
                for (; j < je; j = (j | 7) + 1) {
                    if ((j >> 3) != at) {
                        at = j >> 3;
                        w = __ldg(reinterpret_cast<const unsigned long long *>(k0) + at);
                        if (k1 != nullptr) w |= __ldg(reinterpret_cast<const unsigned long long *>(k1) + at);
                    }
                    const unsigned long long u = w >> (8 * (j & 7));
                    if (u != 0) return min(j + ((__ffsll((long long)u) - 1) >> 3), je);
                }
                return je;
            } else {
                return j;
            }
        }
        __device__ __forceinline__ bool add(int j) const { return ((w >> (8 * (j & 7))) & 0xffu) == TILE_ADD; }  // j = the last next()
    };
    auto tiles_of = [&](int64_t head, int64_t row, bool both) -> Tiles {
        Tiles t = {nullptr, nullptr, -1, 0ull};
        if constexpr (MASK) {
            const int64_t plane = (head / a.mask.seq_heads) * a.mask.plane_step + (head % a.mask.seq_heads) % a.mask.plane_heads;
            t.k0 = a.tile_kind + (plane * a.kind_rb + row / FM) * a.kind_ld;
            if (both) t.k1 = t.k0 + a.kind_ld;
        }
        return t;
    };
    // The n-th item of this block: heaviest row blocks first (the last ones when causal; in ENERGY mode, where early
    // keys are seen by most queries, the first ones), and the direction alternates from round to round, so that the
    // block that drew the heaviest item of one round draws the lightest of the next.
    auto item_of = [&](int64_t n, int64_t *head, int64_t *r0) -> bool {
        const int64_t b = (n & 1) ? (int64_t)gridDim.x - 1 - blockIdx.x : blockIdx.x;
        const int64_t item = n * gridDim.x + b;
        if (item >= items) return false;
        *head = item % a.heads;
        const int64_t rb = item / a.heads;
        *r0 = (MODE == MODE_ENERGY ? rb : blocks_r - 1 - rb) * rows_blk;
        return true;
    };
    const int64_t rounds = (items + gridDim.x - 1) / gridDim.x;

    if (warp == 0) {
        // ------------------------------------------------------------------ producer: Q, then K_0, K_1, V_0, K_2, V_1, ...
        uint32_t ks = 0, kph = 0, n_item = 0;
        bool ok = true, first_load = true;
        auto load_kv = [&](const CUtensorMap *map, int chunks, int64_t row, int z) -> bool {
            if (!mbar_wait_sleepy(kv_empty(ks), kph ^ 1u, abort_flag, a.status, a.wait_ns)) return false;
            const uint32_t dst = base + kOffKv + ks * kKvTile;
            if (a.withhold && blockIdx.x == 0 && first_load) {
                first_load = false;  // (test switch) this tile is never requested: its barrier stays incomplete
            } else {
                mbar_arrive_expect_tx(kv_full(ks), (uint32_t)chunks * kKvChunk);
                for (int c = 0; c < chunks; ++c) tma_load_3d(dst + c * kKvChunk, map, c * 64, (int)row, z, kv_full(ks));
            }
            if (++ks == kKvStages) { ks = 0; kph ^= 1u; }
            return true;
        };
        for (int64_t n = 0; n < rounds && ok; ++n) {
            int64_t head, r0;
            if (!item_of(n, &head, &r0)) continue;
            int jb, je;
            block_range(head, r0, &jb, &je);
            Tiles tiles = tiles_of(head, r0, a.groups == 2);
            jb = tiles.next(jb, je);
            if (je <= jb) continue;
            if (lane == 0) {
                const int vb = (int)((head + a.v_off) / a.v_div);
                ok = mbar_wait_sleepy(q_empty, (n_item & 1u) ^ 1u, abort_flag, a.status, a.wait_ns);
                if (ok) {
                    mbar_arrive_expect_tx(q_full, (uint32_t)(a.groups * kq) * kQChunk);
                    for (int g = 0; g < a.groups; ++g)
                        for (int c = 0; c < kq; ++c)
                            tma_load_3d(base + kOffQ + g * kQTile + c * kQChunk, &map_q, c * 64, (int)(r0 + g * FM), (int)head, q_full);
                    ok = load_kv(&map_k, kq, (int64_t)jb * FN, (int)head);
                }
                for (int j = jb, nj; j < je && ok; j = nj) {
                    nj = tiles.next(j + 1, je);
                    if (nj < je) ok = load_kv(&map_k, kq, (int64_t)nj * FN, (int)head);
                    if constexpr (kHasV) {
                        if (ok) ok = load_kv(&map_v, nv, (int64_t)j * FN, vb);
                    }
                }
            }
            ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
            ++n_item;  // counts the items that reach the tensor cores (those with at least one tile)
        }
        __syncwarp();
    } else if (warp == 1 || warp == kMmaWarp1) {
        // ------------------------------------------------------------------ MMA issuer of group g (one thread)
        // Both issuers walk the same ring entries; each uses the tiles its group needs and releases every entry (a
        // commit arrives once this thread's earlier MMAs are done, at once if there are none).
        const int g = warp == 1 ? 0 : 1;
        const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(FN >> 3) << 17) | ((uint32_t)(FM >> 4) << 24);
        const uint32_t idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)((nv * 64) >> 3) << 17) |
                                 ((uint32_t)(FM >> 4) << 24);
        const uint64_t dq0 = smem_desc(base + kOffQ + g * kQTile, 16, 1024), dk0 = smem_desc(base + kOffKv, 16, 1024);
        const uint64_t dp0 = smem_desc(base + kOffP + g * kPTile, 16, 1024), dv0 = smem_desc(base + kOffKv, kKvChunk, 1024);
        const uint32_t q_hi = (uint32_t)(dq0 >> 32), k_hi = (uint32_t)(dk0 >> 32), p_hi = (uint32_t)(dp0 >> 32), v_hi = (uint32_t)(dv0 >> 32);
        const uint32_t q_lo = (uint32_t)dq0, k_lo = (uint32_t)dk0, p_lo = (uint32_t)dp0, v_lo = (uint32_t)dv0;
        const int steps_s = (a.kd + 15) / 16;
        const uint32_t t_s = tmem_base + g * FN, t_o = tmem_base + kTmemO + g * 128;
        uint32_t ks = 0, kph = 0, n_item = 0, s_it = 0, p_it = 0, o_it = 0;
        bool ok = true;
        int gb = 0, ge = 0;  // this group's tile range in the current item
        int gn = 0;          // MASK: the first tile from the current one on that this group needs
        ASTAMP_DECL(blockIdx.x == 0 && lane == 0 && g == 0);
        auto step_s = [&](int j) -> bool {  // S~ of tile j (if this group needs it); consumes one ring entry
            ASTAMP(7);
            if (!mbar_wait(kv_full(ks), kph, abort_flag, a.status, a.wait_ns)) return false;
            ASTAMP(0);
            if (MASK ? j == gn && gn < ge : (j >= gb && j < ge)) {
                // S~ is single-buffered: the softmax warps release it as soon as they hold the tile in registers
                if (!mbar_wait(s_empty(g, 0), (s_it & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) return false;
                ASTAMP(1);
                tc_fence_after();
                uint32_t ql = q_lo, kl = k_lo + ks * (kKvTile >> 4), acc = 0;
                if (elect_one()) {
                    for (int left = steps_s; left > 0; left -= 4, ql += kQChunk >> 4, kl += kKvChunk >> 4) {  // 64-feature chunks
                        const int ns = left < 4 ? left : 4;
                        for (int st = 0; st < ns; ++st, acc = 1u)  // 16 features = 32 bytes per step
                            umma_bf16_lohi<1>(t_s, ql + 2 * st, q_hi, kl + 2 * st, k_hi, idesc_s, acc);
                    }
                    umma_commit<1>(s_full(g, 0));
                }
                ++s_it;
            }
            if (elect_one()) umma_commit<1>(kv_empty(ks));
            __syncwarp();
            if (++ks == kKvStages) { ks = 0; kph ^= 1u; }
            ASTAMP(2);
            return true;
        };
        for (int64_t n = 0; n < rounds && ok; ++n) {
            int64_t head, r0;
            if (!item_of(n, &head, &r0)) continue;
            int jb, je;
            block_range(head, r0, &jb, &je);
            Tiles tiles = tiles_of(head, r0, a.groups == 2), own = tiles_of(head, r0 + g * FM, false);
            jb = tiles.next(jb, je);
            if (je <= jb) continue;
            if (g < a.groups) tile_range(head, r0 + g * FM, &gb, &ge);
            else gb = ge = 0;   // nothing of the item is this group's: it only hands the ring entries back
            gn = gb = own.next(gb, ge);
            if (!mbar_wait(q_full, n_item & 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
            ok = step_s(jb);
            for (int j = jb, nj; j < je && ok; j = nj) {
                nj = tiles.next(j + 1, je);
                const bool use = MASK ? j == gn && gn < ge : (j >= gb && j < ge);  // this group needs the tile
                if (MASK && use) gn = own.next(j + 1, ge);
                const bool last_use = MASK ? gn >= ge : j == ge - 1;
                if (nj < je) ok = step_s(nj);                              // S~ of the next tile runs ahead of this P V
                if (!ok) break;
                if constexpr (kHasV) {
                    ASTAMP(7);
                    if (!mbar_wait(kv_full(ks), kph, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                    ASTAMP(3);
                    if (use) {
                        if (j == gb && !mbar_wait(o_empty(g), (o_it & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                        ASTAMP(4);
                        if (!mbar_wait(p_full(g), p_it & 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                        ASTAMP(5);
                        tc_fence_after();
                        const uint32_t vl = v_lo + ks * (kKvTile >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int st = 0; st < FN / 16; ++st)  // P: K-major, 64-key chunks, 32 bytes per step; V: MN-major (rows = keys), 16 keys = 2048 bytes
                                umma_bf16_lohi<1>(t_o, p_lo + (st >> 2) * (kPChunk >> 4) + (st & 3) * 2, p_hi, vl + st * (2048 >> 4), v_hi, idesc_o,
                                                  (j != gb || st != 0) ? 1u : 0u);
                            umma_commit<1>(p_empty(g));   // "P V of this tile is complete": P may be rewritten, O may be rescaled
                            if (last_use) umma_commit<1>(o_full(g));
                        }
                        ++p_it;
                        if (last_use) ++o_it;
                    }
                    if (elect_one()) umma_commit<1>(kv_empty(ks));
                    __syncwarp();
                    if (++ks == kKvStages) { ks = 0; kph ^= 1u; }
                    ASTAMP(6);
                }
            }
            if (ok && elect_one()) umma_commit<1>(q_empty);
            __syncwarp();
            ++n_item;
        }
        ASTAMP_FLUSH(0);
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ softmax and epilogue (one row per thread)
        // A step is 128 columns, taken as two chunks of 64 so that a thread never holds more than 64 logits.
        const int g = (warp - 2) >> 2, q = warp & 3, r = q * 32 + lane;
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t t_s = t_lane + g * FN, t_o = t_lane + kTmemO + g * 128;
        float c2 = a.scale_log2;        // (1 for tiles that hold x already)
        uint64_t c22 = pack2(c2, c2);
        uint8_t *prow = base_ptr + kOffP + g * kPTile + r * 128;  // row r of each 64-key chunk: 128 bytes, 16-byte units swizzled
        uint32_t s_it = 0, p_it = 0, o_it = 0;
        bool ok = true;
        ASTAMP_DECL(blockIdx.x == 0 && warp == 2 && lane == 0);
        for (int64_t n = 0; n < rounds && ok; ++n) {
            int64_t head, r0;
            if (!item_of(n, &head, &r0)) continue;
            r0 += g * FM;
            if (g >= a.groups || r0 >= a.Lr) continue; // this group has no rows in the block, or none in the last block
            int jb, je;
            tile_range(head, r0, &jb, &je);
            Tiles tiles = tiles_of(head, r0, false);
            jb = tiles.next(jb, je);
            const int i = (int)r0 + r;                 // this thread's row (rows, columns and their sums stay below 2^31)
            __nv_bfloat16 *orow = a.O + head * a.o_sh + (int64_t)i * a.o_sr;
            if (je <= jb) {  // nothing visible for any row of this group
                if constexpr (kHasV) {
                    if (i < a.Lr)
                        for (int c = 0; c < a.Dh; c += 8) *reinterpret_cast<uint4 *>(orow + c) = make_uint4(0, 0, 0, 0);
                } else if constexpr (MODE == MODE_STATS) {
                    if (i < a.lse_ld) a.lse[head * a.lse_ld + i] = -INFINITY;  // 2^(x - inf) = 0 for every later use
                } else {
                    if (i < a.Lr) a.energy[head * a.Lr + i] = 0.f;
                }
                continue;
            }
            // columns this row sees: [first_col, last_col]
            int first_col = 0, last_col = (int)a.Lc - 1;
            if (a.causal) {
                if constexpr (MODE == MODE_ENERGY) first_col = max(0, i - (int)a.diag);
                else if constexpr (MODE == MODE_GATHERED) last_col = (int)kept_upto_rows(a.tok + head * a.Lc, r0 + q * 32 + a.diag) - 1;
                else last_col = min((int)a.Lc - 1, i + (int)a.diag);
            }
            float m = -INFINITY, l = 0.f;  // FULL / STATS: the maximum that p is taken against (log2 domain), the row sum
            float neg_lse = 0.f;           // GATHERED: this row's negated normaliser
            if constexpr (MODE == MODE_GATHERED) neg_lse = i < a.lse_ld ? a.lse[head * a.lse_ld + i] : -INFINITY;

            // 64 logits of the current tile (columns c_off .. c_off + 63) into registers; hidden columns become -inf on
            // boundary tiles (the diagonal and the ragged end)
            auto load_chunk = [&](int j, int c_off, uint32_t (&v0)[32], uint32_t (&v1)[32]) {
                tmem_ld32_issue(t_s + c_off, v0);
                tmem_ld32_issue(t_s + c_off + 32, v1);
                tmem_ld_wait();
                const int c0 = j * FN + c_off, hi = max(-1, min(63, last_col - c0)), lo = MODE == MODE_ENERGY ? max(0, min(64, first_col - c0)) : 0;
                if (!__all_sync(0xffffffffu, hi >= 63 && lo <= 0)) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        if (e > hi || e < lo) v0[e] = 0xff800000u;
                        if (e + 32 > hi || e + 32 < lo) v1[e] = 0xff800000u;
                    }
                }
            };
            // MASK: the caller's additive mask (-inf hides a key) added to this warp's rows of the S~ tile where they lie, 16
            // columns at a time, so that the steps below hold no mask values in registers; rows past the end and columns
            // past the last key read nothing.  The tile then holds x = scaled logit + M in the log2 domain, rounded: equal
            // sums give equal x, however large M is, so that x - max is what it would be in exact arithmetic (the product
            // with the scale taken inside the subtraction leaves 2^-24 of x, which an M of -1e30 turns into infinities).
            // A low finite M stays finite.
            [[maybe_unused]] auto add_mask_tile = [&](int j) {
                const int64_t c0 = (int64_t)j * FN;
                const float *mrow = a.mask.p + (head / a.mask.seq_heads) * a.mask.sb + (head % a.mask.seq_heads) * a.mask.sh + (int64_t)i * a.mask.sr + c0;
#pragma unroll 1
                for (int c = 0; c < FN; c += 16) {
                    float m4[16];
                    if (i < a.Lr && a.mask.vec && c0 + c + 15 < a.Lc) {
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const float4 q = __ldg(reinterpret_cast<const float4 *>(mrow + c) + v);
                            m4[4 * v] = q.x; m4[4 * v + 1] = q.y; m4[4 * v + 2] = q.z; m4[4 * v + 3] = q.w;
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) m4[e] = i < a.Lr && c0 + c + e < a.Lc ? __ldg(mrow + c + e) : 0.f;
                    }
                    uint32_t s16[16];
                    tmem_ld16_issue(t_s + c, s16);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float t = m4[e] * kLog2e;
                        if (m4[e] >= -FLT_MAX) t = fmaxf(t, -FLT_MAX);
                        s16[e] = __float_as_uint(fmaf(__uint_as_float(s16[e]), a.scale_log2, t));
                    }
                    tmem_st16_issue(t_s + c, s16);
                }
                tmem_st_wait();
            };
            auto release_s = [&]() {  // this warp holds what it needs of the S~ tile
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(s_empty(g, 0));
            };
            auto max_chunk = [&](const uint32_t (&v0)[32], const uint32_t (&v1)[32]) -> float {
                float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    mx0 = fmax3(mx0, __uint_as_float(v0[e]), __uint_as_float(v0[e + 1]));
                    mx1 = fmax3(mx1, __uint_as_float(v0[e + 2]), __uint_as_float(v0[e + 3]));
                    mx2 = fmax3(mx2, __uint_as_float(v1[e]), __uint_as_float(v1[e + 1]));
                    mx3 = fmax3(mx3, __uint_as_float(v1[e + 2]), __uint_as_float(v1[e + 3]));
                }
                return fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
            };
            // p = 2^(x - m) for 64 logits: row sum (unless GATHERED) and, with V, the bf16 values packed into w
            auto emit_chunk = [&](const uint32_t (&v0)[32], const uint32_t (&v1)[32], float neg_m, uint32_t (&w)[kHasV ? 32 : 1]) {
                const uint64_t nm2 = pack2(neg_m, neg_m);
                uint64_t sum_a = 0, sum_b = 0;
                auto half = [&](const uint32_t (&v)[32], int c) {
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        float x0, x1;
                        unpack2(ffma2(pack2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), c22, nm2), x0, x1);
                        // Every fourth pair on the FMA pipe, where no row maximum of the whole tile is taken: 32 heads x 3001 x 128 (2401
                        // keys) 82.4 -> 76.2 us, 16 x 8000 (half the features) 176.5 -> 166.4 for the normalisers.  The one-pass form
                        // gains as many clocks (5 %) and loses them to the clock rate (power); the energies are level.
                        float p0, p1;
                        if (MODE != MODE_FULL && (e & 6) == 6) ex2_fma(x0, x1, p0, p1);
                        else { p0 = ex2(x0); p1 = ex2(x1); }
                        if constexpr (MODE != MODE_GATHERED) (e & 2 ? sum_b : sum_a) = fadd2(e & 2 ? sum_b : sum_a, pack2(p0, p1));
                        if constexpr (kHasV) {
                            __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
                            w[(c + e) >> 1] = *reinterpret_cast<uint32_t *>(&h);
                        }
                    }
                };
                half(v0, 0);
                half(v1, 32);
                if constexpr (MODE != MODE_GATHERED) {
                    float s0, s1;
                    unpack2(fadd2(sum_a, sum_b), s0, s1);
                    l += s0 + s1;
                }
            };
            auto store_chunk = [&](int chunk, const uint32_t (&w)[kHasV ? 32 : 1]) {
                if constexpr (kHasV) {
#pragma unroll
                    for (int u = 0; u < 8; ++u)  // 16-byte units of 8 keys
                        *reinterpret_cast<uint4 *>(prow + chunk * kPChunk + ((u ^ (r & 7)) << 4)) =
                            make_uint4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
                }
            };
            // the O rows of the item before have left the P tile
            [[maybe_unused]] auto o_stored = [&]() {
                if (lane == 0) bulk_wait_read<0>();
                __syncwarp();
            };
            // m and l follow a new chunk maximum (log2 domain); returns the factor the sums taken so far have to be scaled by
            auto follow_max = [&](float mc, bool *any_grow) -> float {
                const bool grow = mc > m + kGrowLimit;
                *any_grow = __any_sync(0xffffffffu, grow);
                const float alpha = (grow && m > -INFINITY) ? ex2(m - mc) : 1.f;
                l *= alpha;
                if (grow) m = mc;
                return alpha;
            };

            for (int j = jb, nj; j < je; j = nj, ++s_it) {
                [[maybe_unused]] const bool add_mask = MASK && tiles.add(j);
                nj = tiles.next(j + 1, je);
                if constexpr (MODE == MODE_ENERGY) {
                    // the 128 normalisers of the next tile (512 bytes, the same for every thread) are pulled into L1
                    // one step ahead; the first tile's are fetched cold
                    const int64_t nxt = (int64_t)(j + 1) * FN + lane * 32;
                    if (lane < 4 && j + 1 < je && nxt < a.lse_ld)
                        asm volatile("prefetch.global.L1 [%0];" ::"l"(a.lse + head * a.lse_ld + nxt));
                }
                ASTAMP(7);
                if (!mbar_wait(s_full(g, 0), s_it & 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                ASTAMP(0);
                tc_fence_after();
                if constexpr (MASK) {
                    if (add_mask) add_mask_tile(j);
                    c2 = add_mask ? 1.f : a.scale_log2;
                    c22 = pack2(c2, c2);
                }
                uint32_t v0[32], v1[32];

                if constexpr (MODE == MODE_ENERGY) {
                    // p = bf16(2^(x - lse_i)); this key's score accumulates p^2 over the tile's 128 queries, queries of even
                    // and of odd number apart (the two halves of the packed fp32 operations: 3.5 instructions a logit where
                    // single ones took 4.5; 148 against 154 us on 8 heads x 8000)
                    uint64_t acc = 0;
                    for (int c_off = 0; c_off < FN; c_off += 64) {
                        ulonglong2 cl[16];  // the negated normalisers of these 64 queries (the same for every thread), in pairs
                        const ulonglong2 *lp = reinterpret_cast<const ulonglong2 *>(a.lse + head * a.lse_ld + (int64_t)j * FN + c_off);
#pragma unroll
                        for (int u = 0; u < 16; ++u) cl[u] = (int64_t)j * FN + c_off + 4 * u < a.lse_ld ? __ldg(lp + u) : make_ulonglong2(0, 0);
                        load_chunk(j, c_off, v0, v1);
                        if (c_off == 64) release_s();
                        auto fold = [&](const uint32_t (&v)[32], int c) {
#pragma unroll
                            for (int e = 0; e < 32; e += 2) {
                                const ulonglong2 ls = cl[(c + e) >> 2];
                                float x0, x1;
                                unpack2(ffma2(pack2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), c22, e & 2 ? ls.y : ls.x), x0, x1);
                                const __nv_bfloat162 h = __floats2bfloat162_rn(ex2(x0), ex2(x1));
                                const uint32_t hw = *reinterpret_cast<const uint32_t *>(&h);
                                const uint64_t p2 = pack2(__uint_as_float(hw << 16), __uint_as_float(hw & 0xffff0000u));
                                acc = ffma2(p2, p2, acc);
                            }
                        };
                        fold(v0, 0);
                        fold(v1, 32);
                    }
                    float acc0, acc1;
                    unpack2(acc, acc0, acc1);
                    l += acc0 + acc1;
                    continue;
                }

                if constexpr (MODE == MODE_STATS) {
                    // no P and no O: the two chunks are folded one after the other, each against its own maximum
                    for (int c_off = 0; c_off < FN; c_off += 64) {
                        load_chunk(j, c_off, v0, v1);
                        if (c_off == 64) release_s();
                        bool any_grow;
                        follow_max(max_chunk(v0, v1) * c2, &any_grow);
                        uint32_t w[1];
                        emit_chunk(v0, v1, m > -INFINITY ? -m : 0.f, w);
                    }
                    continue;
                }

                uint32_t w[kHasV ? 32 : 1];
                if constexpr (MODE == MODE_GATHERED) {
                    const float neg_m = neg_lse;   // -inf (row sees nothing): p = 0
                    load_chunk(j, 0, v0, v1);
                    emit_chunk(v0, v1, neg_m, w);
                    if (!mbar_wait(p_empty(g), (p_it & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                    if (O_TILES && j == jb) o_stored();
                    store_chunk(0, w);
                    load_chunk(j, 64, v0, v1);
                    release_s();
                    emit_chunk(v0, v1, neg_m, w);
                    store_chunk(1, w);
                } else {
                    // FULL: the maximum of all 128 logits decides about a rescale before any p is taken; the second
                    // chunk is still in registers then, the first is read from tensor memory once more
                    load_chunk(j, 0, v0, v1);
                    const float mx_a = max_chunk(v0, v1);
                    load_chunk(j, 64, v0, v1);
                    const float mx = fmaxf(mx_a, max_chunk(v0, v1));
                    bool any_grow;
                    const float alpha = follow_max(mx * c2, &any_grow);
                    if (any_grow && j > jb) {  // rows of O already hold sums taken against the old maximum
                        if (!mbar_wait(p_empty(g), (p_it & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                        tc_fence_after();
                        for (int c = 0; c < nv * 64; c += 16) {
                            uint32_t o[16];
                            tmem_ld16_issue(t_o + c, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                            tmem_st16_issue(t_o + c, o);
                        }
                        tmem_st_wait();
                    }
                    const float neg_m = m > -INFINITY ? -m : 0.f;
                    const float top = ex2(fmaf(mx, c2, neg_m));  // the tile's largest weight, as the chunks below get it
                    l += __bfloat162float(__float2bfloat16_rn(top)) - top;
                    ASTAMP(2);
                    emit_chunk(v0, v1, neg_m, w);
                    ASTAMP(3);
                    // (a repeated wait on a completed phase returns at once: the rescale above may have waited already)
                    if (!mbar_wait(p_empty(g), (p_it & 1u) ^ 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                    ASTAMP(4);
                    store_chunk(1, w);
                    load_chunk(j, 0, v0, v1);
                    release_s();
                    emit_chunk(v0, v1, neg_m, w);
                    store_chunk(0, w);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> visible to the tensor cores
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full(g));
                ++p_it;
                ASTAMP(5);
            }
            if (!ok) break;
            if constexpr (MODE == MODE_STATS) {
                if (i < a.lse_ld) a.lse[head * a.lse_ld + i] = l > 0.f ? -(m + log2f(l)) : -INFINITY;
            } else if constexpr (MODE == MODE_ENERGY) {
                if (i < a.Lr) a.energy[head * a.Lr + i] = l;
            } else {
                // ---- epilogue: O row (/ l) -> bf16 -> global
                if (!mbar_wait(o_full(g), o_it & 1u, abort_flag, a.status, a.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const float inv_l = MODE == MODE_GATHERED ? 1.f : (l > 0.f ? 1.f / l : 0.f);
                if constexpr (O_TILES) {
                    // The P tile is free (the last P V is complete): the warp's 32 rows go through it, laid out as P is, and leave by a
                    // tile store, which clips rows and columns past the end: 32 heads x 3001 x 128 (2401 keys) 86.4 -> 82.4 us.  The
                    // one-pass form, where the maps' set-up and the stores' tail weigh more, keeps direct stores (2 heads x 8192: 90.0
                    // us a call, 91.7 by tiles; 32 x 4096 level).
#pragma unroll 1
                    for (int c = 0; c < nv * 64; c += 32) {
                        uint32_t v[32];
                        tmem_ld32_issue(t_o + c, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            uint32_t ww[4];
#pragma unroll
                            for (int pp = 0; pp < 4; ++pp) {
                                __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[8 * u + 2 * pp]) * inv_l,
                                                                         __uint_as_float(v[8 * u + 2 * pp + 1]) * inv_l);
                                ww[pp] = *reinterpret_cast<uint32_t *>(&h);
                            }
                            *reinterpret_cast<uint4 *>(prow + (c >> 6) * kPChunk + (((((c >> 3) & 7) + u) ^ (r & 7)) << 4)) = make_uint4(ww[0], ww[1], ww[2], ww[3]);
                        }
                    }
                    fence_proxy_async();
                } else {
                    for (int c = 0; c < nv * 64; c += 32) {
                        uint32_t v[32];
                        tmem_ld32_issue(t_o + c, v);
                        tmem_ld_wait();
                        if (i < a.Lr) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (c + 8 * u >= a.Dh) break;
                                uint32_t ww[4];
#pragma unroll
                                for (int pp = 0; pp < 4; ++pp) {
                                    __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[8 * u + 2 * pp]) * inv_l,
                                                                             __uint_as_float(v[8 * u + 2 * pp + 1]) * inv_l);
                                    ww[pp] = *reinterpret_cast<uint32_t *>(&h);
                                }
                                *reinterpret_cast<uint4 *>(orow + c + 8 * u) = make_uint4(ww[0], ww[1], ww[2], ww[3]);
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(o_empty(g));
                    if (O_TILES && r0 + q * 32 < a.Lr) {
                        for (int c = 0; c < nv; ++c)
                            tma_store_3d(&map_o, base + kOffP + g * kPTile + c * kPChunk + q * 4096, c * 64, (int)r0 + q * 32, (int)head);
                        bulk_commit();
                    }
                }
                ++o_it;
            }
            ASTAMP(6);
        }
        if constexpr (O_TILES) {
            if (lane == 0) bulk_wait_read<0>();  // shared memory stays until the stores have read it
            __syncwarp();
        }
        ASTAMP_FLUSH(8);
    }

    __syncthreads();
    if (*abort_flag) {
        unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    tc_fence_after();
    if (warp == 1) tmem_dealloc<1>(tmem_base, kTmemCols);
}

// Groups of 128 rows per block.  Two share every K and V tile and hide each other's waits (3400 clocks a step of 256 x 128), but
// where blocks of 128 rows do not outnumber the SMs there is nothing to share an SM with: one group alone takes 2330 a step of
// 128 x 128 (either a tenth more where logits as spread as those of outlier features make it rescale), and a row block's keys are the serial chain that the launch waits for.  Kernels of 2, 8 and 16 heads x 4096, 2048 and
// 1100 x 128, causal, by two and by one: 67.5 and 51.2, 41.0 and 32.7, 26.7 and 24.6 us; the sweeps of the token reduction likewise
// (8 x 2048: 29.4 / 41.3 / 24.6 and 22.8 / 33.2 / 20.5).
// In up to two rounds a causal block's short rows follow another's long ones (item_of), so one group still wins where the longest
// sum of a pair is not much longer than the longest item: 8 x 4096 71.6 and 57.3, 16 x 2048 41.8 and 37.0, 4 x 8192 124.9 and 92.2,
// the normalisers and energies of 8 x 4096 50.1 / 74.1 and 38.9 / 55.8; 32 x 1000, items of eight tiles at most, level; 64 x 500
// 18.5 and 22.5; without a mask 8 x 4096 takes 73.8 by two and 104.4 by one.  The clocks are those of the one-pass kernel; both
// sweeps keep about their ratio, and over 20 shapes of 64 and 128 columns the rule's choice was never more than 2 us behind.  Where
// the number of tiles is not the rows', only the first rule holds: kept keys (8 x 4096 36.9 and 43.0, 5 x 4096 36.9 and 28.7), and an
// additive mask, of which nothing is known here (8 x 4096 padded, causal 71.7 and 63.5, otherwise 73.8 and 104.5).
template <int MODE, bool MASK>
int block_groups(const FusedArgs &a, int64_t sms)
{
    const int64_t blocks = ceil_div(a.Lr, FM), items = a.heads * blocks;
    if (items <= sms) return 1;
    if (MASK || MODE == MODE_GATHERED || !a.causal || items > 2 * sms) return 2;
    auto tiles = [&](int64_t rank) -> int64_t {  // of the item of this rank in the order of item_of
        const int64_t r0 = (MODE == MODE_ENERGY ? rank / a.heads : blocks - 1 - rank / a.heads) * FM;
        if (MODE == MODE_ENERGY) {
            const int64_t first = r0 > a.diag ? r0 - a.diag : 0;
            return first >= a.Lc ? 0 : ceil_div(a.Lc, FN) - first / FN;
        }
        const int64_t last = a.Lc - 1 < r0 + FM - 1 + a.diag ? a.Lc - 1 : r0 + FM - 1 + a.diag;
        return last < 0 ? 0 : last / FN + 1;
    };
    constexpr double kItem = 7000.0;  // set-up and epilogue
    double one = kItem + 2330.0 * (double)tiles(0);
    for (int64_t pair : {2 * sms - items, sms - 1}) {  // an SM's second item: the ranks of a pair add up to 2 sms - 1
        const double both = 2.0 * kItem + 2330.0 * (double)(tiles(pair) + tiles(2 * sms - 1 - pair));
        if (both > one) one = both;
    }
    return one < 0.95 * (kItem + 3400.0 * (double)tiles(0)) ? 1 : 2;
}

template <int MODE, bool MASK = false, bool O_TILES = false>
int launch_mode(const CUtensorMap &mq, const CUtensorMap &mk, const CUtensorMap &mv, const CUtensorMap &mo, const FusedArgs &a, const char *name,
                cudaStream_t stream)
{
    auto kern = fused_attn_kernel<MODE, MASK, O_TILES>;
    static PerDeviceOnce configured;
    if (cudaError_t e = configured.smem(kFusedSmem, kern)) return fail(RMM_ERR_CUDA, "fused_attn: cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    FusedArgs args = a;
    args.groups = block_groups<MODE, MASK>(a, sms);
    const int64_t items = a.heads * ceil_div(a.Lr, args.groups * FM);
    prof_begin(name, stream);
    cudaError_t e = launch_kernel(kern, dim3((unsigned)(items < sms ? items : sms)), dim3(kFusedThreads), kFusedSmem, stream, 1,
                                  mq, mk, mv, mo, args);
    if (e != cudaSuccess) return fail(RMM_ERR_CUDA, "%s: launch: %s", name, cudaGetErrorString(e));
    return check_launch(name, stream);
}

// 3-D map over a packed [heads, rows, ld] bf16 tensor with `cols` valid columns and a box of 64 columns x box_rows rows.
int packed_map(CUtensorMap *m, const __nv_bfloat16 *p, int64_t cols, int64_t rows, int64_t heads, int64_t ld, uint32_t box_rows)
{
    uint64_t dims[3] = {(uint64_t)cols, (uint64_t)rows, (uint64_t)heads};
    uint64_t st[2] = {(uint64_t)ld * 2, (uint64_t)rows * ld * 2};
    const uint32_t box[3] = {64, box_rows, 1};
    return make_map(m, const_cast<__nv_bfloat16 *>(p), 3, dims, st, box, true);
}

}  // namespace

#ifdef RMM_ATTN_STAMPS
extern "C" void rmm_debug_attn_stamps(unsigned long long *out)
{
    cudaDeviceSynchronize();
    cudaMemcpyFromSymbol(out, g_astamps, sizeof(g_astamps));
    unsigned long long z[16] = {};
    cudaMemcpyToSymbol(g_astamps, z, sizeof(z));
}
#endif

bool fused_attn_eligible(const rmm_attn_desc_t *d, int64_t kd)
{
    // heads of up to 256 columns run as two passes over 128 columns of V and O each (S~ and the weights are taken again)
    return d->Dh % 8 == 0 && d->Dh <= 256 && kd <= 128 && d->Lq <= INT32_MAX && d->Lk <= INT32_MAX;
}

size_t mask_tiles_bytes(const MaskView &m, int64_t seqs, int64_t Lq, int64_t Lk)
{
    const int64_t planes = (m.plane_step > 0 ? seqs : 1) * m.plane_heads;
    return (size_t)planes * (2 * ceil_div(Lq, kGroups * FM)) * (ceil_div(Lk, FN * 8) * 8);
}

// FULL (lse NULL, tok NULL): O = softmax(Qp Kp^T / sqrt(Dh) + mask) V; `mask` (or NULL) is the caller's additive fp32 mask on
// top of the causal one, and tile_kind room for mask_tiles_bytes().
// GATHERED (lse and tok given): Kp and V hold the kept keys only (Lk = their count, tok their positions); O = P V with
// P = bf16(2^(x + lse)) (lse negated), no renormalisation.  `diag` = Lk - Lq of the unpacked problem.
// Qp [heads, Lq, ldd], Kp [heads, Lk, ldd] packed; V [v_batches, Lk, Dh] with row pitch v_ld and batch pitch v_sb.
int launch_fused_attn(const __nv_bfloat16 *Qp, const __nv_bfloat16 *Kp, int64_t ldd, int64_t kd, const __nv_bfloat16 *V,
                      int64_t v_ld, int64_t v_sb, int64_t v_batches, int64_t v_off, int64_t v_div, __nv_bfloat16 *O,
                      int64_t o_sh, int64_t o_sr, int64_t heads, int64_t Lq, int64_t Lk, int64_t Dh, int causal, int64_t diag,
                      const float *lse, int64_t lse_ld, const int32_t *tok, const MaskView *mask, uint8_t *tile_kind, bool behind_heads,
                      int *status, cudaStream_t stream)
{
    CUtensorMap mq, mk, mv, mo;
    int rc;
    const int64_t kind_rb = 2 * ceil_div(Lq, kGroups * FM), kind_ld = ceil_div(Lk, FN * 8) * 8;
    if (mask != nullptr) {
        const int64_t planes = (mask->plane_step > 0 ? heads / mask->seq_heads : 1) * mask->plane_heads;
        if (kind_ld * kind_rb > INT32_MAX || planes > 65535) return fail(RMM_ERR_UNSUPPORTED, "fused_attn: mask too large");
        MaskTileArgs t = {*mask, Lq, Lk, diag, causal, mask->vec, tile_kind, kind_rb, kind_ld, behind_heads ? 1 : 0};
        prof_begin("mask_tiles_kernel", stream);
        launch_kernel(mask_tiles_kernel, dim3((unsigned)(kind_ld * kind_rb), 1, (unsigned)planes), dim3(kMaskThreads), 0, stream, 1, t);
        if ((rc = check_launch("mask_tiles_kernel", stream)) != RMM_OK) return rc;
    }
    if ((rc = packed_map(&mq, Qp, kd, Lq, heads, ldd, FM)) != RMM_OK) return rc;
    if ((rc = packed_map(&mk, Kp, kd, Lk, heads, ldd, FN)) != RMM_OK) return rc;
    // The O accumulators of a block hold 128 columns per query group: a wider head (up to 256 columns) is produced in
    // two passes, each over its own 128 columns of V and of O; the softmax scale keeps the full head dimension.
    for (int64_t c0 = 0; c0 < Dh; c0 += 128) {
        const int64_t dh = Dh - c0 < 128 ? Dh - c0 : 128;
        {
            uint64_t dims[3] = {(uint64_t)dh, (uint64_t)Lk, (uint64_t)v_batches};
            uint64_t st[2] = {(uint64_t)v_ld * 2, v_batches > 1 ? (uint64_t)v_sb * 2 : (uint64_t)v_ld * 2 * (uint64_t)Lk};
            const uint32_t box[3] = {64, FN, 1};
            if ((rc = make_map(&mv, const_cast<__nv_bfloat16 *>(V + c0), 3, dims, st, box, true)) != RMM_OK) return rc;
        }
        const bool o_tiles = tok != nullptr && o_sh >= 0 && o_sr >= 0;
        if (!o_tiles) {
            mo = mq;  // (O leaves without a tensor map)
        } else {
            uint64_t dims[3] = {(uint64_t)dh, (uint64_t)Lq, (uint64_t)heads};
            uint64_t st[2] = {(uint64_t)o_sr * 2, heads > 1 ? (uint64_t)o_sh * 2 : (uint64_t)o_sr * 2 * (uint64_t)Lq};
            const uint32_t box[3] = {64, 32, 1};  // a warp's rows of a 64-column chunk
            if ((rc = make_map(&mo, O + c0, 3, dims, st, box, true)) != RMM_OK) return rc;
        }
        FusedArgs a = {};
        a.heads = heads; a.Lr = Lq; a.Lc = Lk; a.diag = diag;
        a.kd = (int)kd; a.Dh = (int)dh; a.causal = causal;
        a.v_off = v_off; a.v_div = v_div > 0 ? v_div : 1;
        a.O = O + c0; a.o_sh = o_sh; a.o_sr = o_sr;
        a.lse = const_cast<float *>(lse); a.lse_ld = lse_ld; a.tok = tok;
        a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)Dh));
        a.status = status;
        a.wait_ns = wait_limit_ns();
        a.withhold = debug_withhold() == WITHHOLD_ATTN;
        if (o_tiles) {
            rc = launch_mode<MODE_GATHERED, false, true>(mq, mk, mv, mo, a, "fused_attn_gathered_kernel", stream);
        } else if (tok != nullptr) {
            rc = launch_mode<MODE_GATHERED>(mq, mk, mv, mo, a, "fused_attn_gathered_kernel", stream);
        } else if (mask != nullptr) {
            a.mask = *mask; a.tile_kind = tile_kind; a.kind_rb = kind_rb; a.kind_ld = kind_ld;
            rc = launch_mode<MODE_FULL, true>(mq, mk, mv, mo, a, "fused_attn_masked_kernel", stream);
        } else {
            rc = launch_mode<MODE_FULL>(mq, mk, mv, mo, a, "fused_attn_kernel", stream);
        }
        if (rc != RMM_OK) return rc;
    }
    return RMM_OK;
}

// Sweeps 1 and 2 of the token reduction on packed Qp [heads, Lq, ldd], Kp [heads, Lk, ldd]:
//   lse [heads, lse_ld] (lse_ld a multiple of 64, >= Lq): negated log2-domain row normalisers of softmax(S~ + mask);
//   energy [heads, Lk]: squared token scores sum_i bf16(P_it)^2.
int launch_fused_attn_scores(const __nv_bfloat16 *Qp, const __nv_bfloat16 *Kp, int64_t ldd, int64_t kd, int64_t heads,
                             int64_t Lq, int64_t Lk, int64_t Dh, int causal, float *lse, int64_t lse_ld, float *energy,
                             int *status, cudaStream_t stream)
{
    CUtensorMap mq, mk;
    int rc;
    FusedArgs a = {};
    a.heads = heads; a.diag = Lk - Lq;
    a.kd = (int)kd; a.Dh = (int)Dh; a.causal = causal;
    a.v_div = 1;
    a.lse = lse; a.lse_ld = lse_ld; a.energy = energy;
    a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)Dh));
    a.status = status;
    a.wait_ns = wait_limit_ns();
    a.withhold = debug_withhold() == WITHHOLD_ATTN;
    // sweep 1: rows = queries
    if ((rc = packed_map(&mq, Qp, kd, Lq, heads, ldd, FM)) != RMM_OK) return rc;
    if ((rc = packed_map(&mk, Kp, kd, Lk, heads, ldd, FN)) != RMM_OK) return rc;
    a.Lr = Lq; a.Lc = Lk;
    if ((rc = launch_mode<MODE_STATS>(mq, mk, mk, mk, a, "fused_attn_stats_kernel", stream)) != RMM_OK) return rc;
    // sweep 2: rows = keys, tiles of queries stream past
    if ((rc = packed_map(&mq, Kp, kd, Lk, heads, ldd, FM)) != RMM_OK) return rc;
    if ((rc = packed_map(&mk, Qp, kd, Lq, heads, ldd, FN)) != RMM_OK) return rc;
    a.Lr = Lk; a.Lc = Lq;
    return launch_mode<MODE_ENERGY>(mq, mk, mk, mk, a, "fused_attn_energy_kernel", stream);
}

}  // namespace rmm
