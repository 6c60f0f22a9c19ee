// Tensor-core kernels (tcgen05 + TMEM + TMA) for the gradients at fp32 accuracy with bf16 storage: head dimension 64 (two
// heads at a time, as the forward's kPair), or 128 with feature-map weights given in fp32.
//
// Every value that the operator computes stays an fp32 value: where it becomes an operand of a tensor-core product it is
// written as the sum of three bf16 numbers (x = hi + mid + lo leaves at most 2^-26 |x|), and the product is made of one
// MMA pass per part.  The other operand of each product is a tile of the caller's bf16 tensors, exact as it is, so three
// passes give the whole product:
//     U = X W (weights exact in bf16: one pass, fp32 weights: three)     T = dO S^T, V dS^T (images of S, dS)
//     S, dS (transposed: V^T phi, dO^T phi/den)                          dW = X^T du
// dv = phi dS and dx = du W^T have two computed operands and are rounded to bf16 when they are stored: hi hi + hi mid +
// mid hi, 2^-17 before a rounding of 2^-9.
//
// The tensor core truncates when it adds to an fp32 accumulator (measured: 4e-8 of the accumulator's value per addition,
// 1e-4 after 4700 of them), so nothing is accumulated in it over tiles: a tile's contribution is formed with its small
// parts first (dS: with hi and the lower parts in accumulators of their own) and then added, with rounding, to a master copy
// that also lives in tensor memory.
//
// One CTA per SM walks its contiguous run of 128-token tiles (a unit = one head of 128 or a pair of heads
// of 64 features).  Warps 0-7 do the element-wise work, warp 8 issues the copies and the products.  Shared memory (224 KB of
// tiles) holds ONE tile of each input, the three images and a pool in which the parts of phi / den and of du take turns,
// so a tile is a serial chain of stages that meet at barriers; the element-wise work of a stage runs while the products of the
// one before are made (du while dS, the master copies' additions while dW and dx).
//
// Thread (token, half): d = 128: the 32 logits [32 half, +32) and their features in both softmaxes; pair: head `half` of the
// pair with its 32 logits and 64 features.  du is then local to a thread, and for d = 128 the two threads of a token exchange
// sums only (through the pool), for a pair nothing.
//
// What bounds it: the chain of a tile's stages (14 / 12 us a tile in the query-side / key-side gradient kernel, 7 us in
// kside_split_tc), not the tensor pipe, memory (0.3 of the copy bandwidth) or any one pipe.  Measured, forward + backward:
// B=1 H=12 n=14040 d=128 fp32 weights 367 us (4.94 ms on the CUDA cores at first, 1.28 ms with register-tiled FMAs);
// B=1 H=30 n=17776 d=64 473 us (4.05 ms, 1.21 ms).  dW against 64 bits there: 6.2e-7 and 4.6e-7 (9.1e-7, 1.1e-6).
#pragma once
#include "sm100_backward.cuh"

namespace linattn {
namespace tc {

// 8 element-wise warps, the issuer, and three warps that only complete its group of four: registers are allotted by groups of
// four warps, and setmaxnreg gives the element-wise ones 216 of them (the split of sm100_backward.cuh; with nine warps the
// launch would be held to 168 for all).
constexpr int kSpThreads = kBwdThreads;
constexpr int kSpActive = 288;    // threads that meet: warps 0-8

struct SpSmem {   // gradient kernels
    static constexpr uint32_t kX = 0;                          // Q or K tile (key side: dk is staged here)
    static constexpr uint32_t kY = kX + kTileBytes;            // dO or V tile; then W's mid part, the staging of dq or dv, phi's hi part (key side)
    static constexpr uint32_t kImg = kY + kTileBytes;          // S or dS [f][c], hi, mid, lo
    static constexpr uint32_t kPool = kImg + 3 * kTileBytes;   // 48 KB: W's mid and lo parts | sums exchanged | phi/den of 64 tokens x 3 | du x 3
    static constexpr uint32_t kW = kPool + 3 * kWBytes;        // W^T [64][128], hi part
    static constexpr uint32_t kMisc = kW + kWBytes;
};
struct SpSmemState {   // S, z
    static constexpr uint32_t kX = 0;
    static constexpr uint32_t kY = kX + kTileBytes;
    static constexpr uint32_t kPhi = kY + kTileBytes;          // phi x 3
    static constexpr uint32_t kW = kPhi + 3 * kTileBytes;      // W^T x 3 (its first 4 KB beyond hi: sums exchanged when there is one part only)
    static constexpr uint32_t kXch = kW + 3 * kWBytes;
    static constexpr uint32_t kMisc = kXch + 4096;
};
struct SpMisc {
    static constexpr uint32_t kVec = 0;       // 128 floats: z or dz of the unit
    static constexpr uint32_t kBars = 512;    // mbarriers, TMEM slot, abort word
    static constexpr uint32_t kBytes = 512 + 8 * 12 + 16;
};
constexpr uint32_t kSpSmem = SpSmem::kMisc + SpMisc::kBytes;
constexpr uint32_t kSpSmemState = SpSmemState::kMisc + SpMisc::kBytes;
static_assert(kSpSmem <= 232448 && kSpSmemState <= 232448, "a CTA has 227 KB of shared memory");

// mbarriers: copies X, Y, the unit's images and weights, W's lower parts in the pool, W's mid part in the Y tile; products:
// logits, T, first half of dS, dS (or S, or dv), dW and dx.  Each completes once per tile (SP_SEG once per unit).
enum : int { SP_X = 0, SP_Y = 1, SP_SEG = 2, SP_WP = 3, SP_WY = 4, SP_U = 5, SP_T = 6, SP_A = 7, SP_D = 8, SP_F = 9, SP_NBARS = 10 };

struct SpArgs {
    float* rec;             // [slots][kE]: per (CTA, unit) sums of S or dS as [f][c], then z or dz; slot = cta + unit
    float* rec_w;           // [slots][kWRec]: per (CTA, unit) sums of dW as [j][c]
    const float* vec;       // [units][128]: z (query side) or dz (key side)
    uint32_t* err;
    const __nv_bfloat16* mix_a;   // Eq. 8, as in BwdArgs
    float* part_dr;
    float lin_scale;
    long long str_token, str_head, str_batch;
    int n, H, heads, tiles_per_unit;
    long long total_tiles;
    int w_parts;            // bf16 parts of the weights: 1 or 3
    uint32_t wait_limit_us;
    int test_unmet;         // tests of the time-out path only: the first tile's logits are not announced
};

struct SpCta {
    uint8_t* smem;
    uint32_t sb, bar0, tmem;
    float* vec;
    WaitCtx wc;
    __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * (uint32_t)i; }
    __device__ __forceinline__ bool wait(int i, uint32_t parity, uint32_t code) const
    {
        const bool ok = warp_wait(bar(i), parity & 1u, wc, code);
        tcgen05_fence_after();
        return ok;
    }
};

__device__ __forceinline__ SpCta sp_setup(uint8_t* raw, uint32_t misc_off, uint32_t* err, uint32_t limit_us)
{
    pdl_trigger();
    SpCta c;
    c.smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    c.sb = smem_u32(c.smem);
    c.vec = reinterpret_cast<float*>(c.smem + misc_off + SpMisc::kVec);
    uint64_t* bars = reinterpret_cast<uint64_t*>(c.smem + misc_off + SpMisc::kBars);
    c.bar0 = smem_u32(bars);
    uint32_t* slot = reinterpret_cast<uint32_t*>(&bars[SP_NBARS]);
    c.wc.err = err;
    c.wc.abort_smem = smem_u32(slot + 1);
    c.wc.limit_us = limit_us;
    if (threadIdx.x == 0) {
        slot[1] = 0u;
        for (int i = 0; i < SP_NBARS; ++i) mbar_init(c.bar(i), 1);
        fence_mbar_init();
    }
    if ((threadIdx.x >> 5) == 1) {
        tmem_alloc(smem_u32(slot), 512);
        tmem_relinquish();
    }
    pdl_wait();
    fence_proxy_async_smem();
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    c.tmem = *slot;
    return c;
}
__device__ __forceinline__ void sp_teardown(const SpCta& c)
{
    tcgen05_fence_before();
    __syncthreads();
    if ((threadIdx.x >> 5) == 1) tmem_dealloc(c.tmem, 512);
}
// Warps 0-8: what they wrote is visible to the tensor core and to TMA, their tensor-memory reads are done, and they
// agree on the verdict of their waits (the same in every thread, so nobody is left behind at a later barrier).
__device__ __forceinline__ bool sp_meet(bool ok)
{
    fence_proxy_async_smem();
    tcgen05_fence_before();
    const bool all = named_barrier_and(1, kSpActive, ok);
    tcgen05_fence_after();
    return all;
}
__device__ __forceinline__ void sp_sync() { named_barrier_sync(2, 256); }   // the element-wise warps
// After a wait that gave up: copies in flight get a short while to land before the CTA gives its memory back.
__device__ __forceinline__ void sp_settle(const SpCta& c, uint32_t par, uint32_t seg_par)
{
    constexpr uint64_t ns = 20000;
    mbar_wait(c.bar(SP_SEG), seg_par & 1u, ns);
    for (int b : {SP_X, SP_Y, SP_WP, SP_WY}) mbar_wait(c.bar(b), par & 1u, ns);
    for (int b : {SP_X, SP_Y, SP_WP}) mbar_wait(c.bar(b), (par + 1u) & 1u, ns);
}

// ---- products (one thread) ---------------------------------------------------------------------------------------------
// D = X W over the weights' parts, lowest first.
__device__ __forceinline__ void sp_logits(uint32_t d, uint32_t x, uint32_t w, uint32_t acc)
{
    constexpr uint32_t id = make_idesc_bf16(kTile, kM, 0, 0);
    mma_chain(d, desc_at(kmajor_desc(), x), desc_at(kmajor_desc(), w), 32, 32, id, 4, acc);
    mma_chain(d, desc_at(kmajor_desc(), x + kHalfTileBytes), desc_at(kmajor_desc(), w + kWBytes / 2), 32, 32, id, 4, 1u);
}
// D[t][f] += sum_c Y[t][c] img[f][c] (both K-major)
__device__ __forceinline__ void sp_t(uint32_t d, uint32_t y, uint32_t img, uint32_t acc)
{
    constexpr uint32_t id = make_idesc_bf16(kTile, kD, 0, 0);
    mma_chain(d, desc_at(kmajor_desc(), y), desc_at(kmajor_desc(), img), 32, 32, id, 4, acc);
    mma_chain(d, desc_at(kmajor_desc(), y + kHalfTileBytes), desc_at(kmajor_desc(), img + kHalfTileBytes), 32, 32, id, 4, 1u);
}
// D[t][c] += sum_f P[t][f] img[f][c] (P K-major, the image read with its rows as K)
__device__ __forceinline__ void sp_dv(uint32_t d, uint32_t p, uint32_t img, uint32_t acc)
{
    constexpr uint32_t id = make_idesc_bf16(kTile, kD, 0, 1);
    mma_chain(d, desc_at(kmajor_desc(), p), desc_at(mn_desc(kHalfTileBytes), img), 32, 2048, id, 4, acc);
    mma_chain(d, desc_at(kmajor_desc(), p + kHalfTileBytes), desc_at(mn_desc(kHalfTileBytes), img + 4 * 2048), 32, 2048, id, 4, 1u);
}
// D[c][f] += sum over `steps` * 16 tokens of Y[t][c] P[t][f]; pblk: bytes between P's two 64-feature blocks
template <int kSteps> __device__ __forceinline__ void sp_outer(uint32_t d, uint32_t y, uint32_t p, uint32_t pblk, uint32_t acc)
{
    constexpr uint32_t id = make_idesc_bf16(kD, kD, 1, 1);
    mma_chain(d, desc_at(mn_desc(kHalfTileBytes), y), desc_at(mn_desc(pblk), p), 2048, 2048, id, kSteps, acc);
}
// D[t][c] += sum_j du[t][j] W^T[j][c]
__device__ __forceinline__ void sp_dx(uint32_t d, uint32_t du, uint32_t w, uint32_t acc)
{
    constexpr uint32_t id = make_idesc_bf16(kTile, kD, 0, 1);
    mma_chain(d, desc_at(kmajor_desc(), du), desc_at(mn_desc(kWBytes / 2), w), 32, 2048, id, kM / 16, acc);
}
// D[c][j] += sum_t x[t][c] du[t][j]
__device__ __forceinline__ void sp_dw(uint32_t d, uint32_t x, uint32_t du, uint32_t acc)
{
    constexpr uint32_t id = make_idesc_bf16(kD, kM, 1, 1);
    mma_chain(d, desc_at(mn_desc(kHalfTileBytes), x), desc_at(mn_desc(kHalfTileBytes), du), 2048, 2048, id, kTile / 16, acc);
}

// ---- element-wise pieces -----------------------------------------------------------------------------------------------
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Eight consecutive values as kParts chunks of 16 bytes, one per part (hi, mid, lo), `stride` bytes apart.
template <int kParts> __device__ __forceinline__ void sp_store8(uint8_t* dst, uint32_t stride, const float* x)
{
    float r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = x[i];
#pragma unroll
    for (int s = 0; s < kParts; ++s) {
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[q] = pack_bf16(r[2 * q], r[2 * q + 1]);
            r[2 * q] -= bf_lo(w[q]);
            r[2 * q + 1] -= bf_hi(w[q]);
        }
        *reinterpret_cast<uint4*>(dst + s * stride) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Where a thread's features sit: column (= feature index of the unit) of its 32 softmax(+u) values and of its softmax(-u) ones.
template <int kPair> struct SpCols {
    static __device__ __forceinline__ int pos(int half) { return kPair ? 64 * half : 32 * half; }
    static __device__ __forceinline__ int neg(int half) { return kPair ? 64 * half + 32 : 64 + 32 * half; }
};

// exp(+-u - max) of a thread's 32 logits: e[0..31] softmax(+u), e[32..63] softmax(-u), not normalised; sums of each.  d = 128:
// the maxima run over all 64 logits of the token (both of its threads read them all).
template <int kPair>
__device__ __forceinline__ void sp_exps(uint32_t t_u, int half, float (&e)[64], float& sp, float& sn)
{
    uint32_t r[32];
    tmem_ld_x32(t_u + 32 * half, r);
    float mx, mn;
    if (kPair) {
        tmem_wait_ld();
        mx = mn = __uint_as_float(r[0]);
    } else {
        uint32_t o[32];
        tmem_ld_x32(t_u + 32 * (half ^ 1), o);
        tmem_wait_ld();
        mx = mn = __uint_as_float(o[0]);
#pragma unroll
        for (int j = 1; j < 32; ++j) {
            mx = fmaxf(mx, __uint_as_float(o[j]));
            mn = fminf(mn, __uint_as_float(o[j]));
        }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        mx = fmaxf(mx, __uint_as_float(r[j]));
        mn = fminf(mn, __uint_as_float(r[j]));
    }
    sp = 0.f;
    sn = 0.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float u = __uint_as_float(r[j]);
        e[j] = expf(u - mx);
        e[32 + j] = expf(mn - u);
        sp += e[j];
        sn += e[32 + j];
    }
}

// sum_j e_j * vec[col + j] over a thread's 32 features of one softmax
__device__ __forceinline__ float sp_dot_vec(const float* e, const float* vec)
{
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(vec + j);
        s0 = fmaf(e[j], v.x, s0);
        s1 = fmaf(e[j + 1], v.y, s1);
        s0 = fmaf(e[j + 2], v.z, s0);
        s1 = fmaf(e[j + 3], v.w, s1);
    }
    return s0 + s1;
}
__device__ __forceinline__ float sp_dot(const float* a, const float* b)
{
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        s0 = fmaf(a[j], b[j], s0);
        s1 = fmaf(a[j + 1], b[j + 1], s1);
    }
    return s0 + s1;
}

// d = 128: four sums of a token are completed by its two threads (buffer [half][128] float4); pair: they are complete.
template <int kPair> __device__ __forceinline__ float4 sp_exchange(float4* xch, int half, int row, float4 mine)
{
    if (kPair) return mine;
    xch[half * 128 + row] = mine;
    sp_sync();
    const float4 o = xch[(half ^ 1) * 128 + row];
    // the same order of addition in both threads
    return half ? make_float4(o.x + mine.x, o.y + mine.y, o.z + mine.z, o.w + mine.w)
                : make_float4(mine.x + o.x, mine.y + o.y, mine.z + o.z, mine.w + o.w);
}

// Sum over the warp's 32 tokens of 64 values per thread, f(i) the i-th: afterwards lane l holds values 2l and 2l + 1 (in the
// order of i).  A halving tree: 62 shuffles, fp32 throughout.
template <class F> __device__ __forceinline__ void sp_warp_sum64(F f, float& s0, float& s1)
{
    const int lane = threadIdx.x & 31;
    float v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const float a = f(i), b = f(i + 32);
        const bool up = lane & 16;
        v[i] = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
    }
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 2 * o; ++i) {
            const float a = v[i], b = v[i + 2 * o];
            v[i] = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, o);
        }
    }
    s0 = v[0];
    s1 = v[1];
}

// master += a (+ b): 64 columns of this thread's lane (32 when kCols = 32); `first`: master = a (+ b).
template <int kCols, bool kTwo>
__device__ __forceinline__ void sp_drain(uint32_t master, uint32_t a, uint32_t b, bool first)
{
#pragma unroll
    for (int c = 0; c < kCols; c += 32) {
        uint32_t x[32], m[32];
        tmem_ld_x32(a + c, x);
        if (kTwo) {
            tmem_ld_x32(b + c, m);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; ++j) x[j] = __float_as_uint(__uint_as_float(x[j]) + __uint_as_float(m[j]));
        }
        if (!first) {
            tmem_ld_x32(master + c, m);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; ++j) x[j] = __float_as_uint(__uint_as_float(x[j]) + __uint_as_float(m[j]));
        }
        tmem_wait_ld();
        tmem_st_x32(master + c, x);
    }
    tmem_wait_st();
}
// 64 columns of this thread's lane -> record columns: rec[(col + j) * 128 + lane row] (consecutive lanes, consecutive words)
template <int kCols> __device__ __forceinline__ void sp_store_master(float* rec, uint32_t master, int row)
{
#pragma unroll
    for (int c = 0; c < kCols; c += 32) {
        uint32_t x[32];
        tmem_ld_x32(master + c, x);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; ++j) rec[(size_t)(c + j) * kD + row] = __uint_as_float(x[j]);
    }
}
// The thread's feature sums over the CTA's tokens (lane l of every warp: its features 2l, 2l + 1) -> out[128], the four
// token quarters in order.  Barrier inside; scratch: 512 floats.
template <int kPair>
__device__ __forceinline__ void sp_store_vec(float* scratch, float* out, int warp, int lane, float s0, float s1)
{
    const int half = warp >> 2, i = 2 * lane;
    const int col = i < 32 ? SpCols<kPair>::pos(half) + i : SpCols<kPair>::neg(half) + i - 32;
    scratch[(warp & 3) * kD + col] = s0;
    scratch[(warp & 3) * kD + col + 1] = s1;
    sp_sync();
    const int t = warp * 32 + lane;
    if (t < kD) out[t] = ((scratch[t] + scratch[kD + t]) + scratch[2 * kD + t]) + scratch[3 * kD + t];
}

// A 64-column block row of fp32 values from tensor memory -> bf16 tile row (staging of a TMA store)
__device__ __forceinline__ void sp_stage(uint32_t taddr, uint8_t* blk, int row)
{
    float x[kM];
    load64(taddr, x);
    store_row_bf16(blk, row, x);
}

// ---- S, z of the keys ---------------------------------------------------------------------------------------------------
template <int kLayout, int kPair>
__global__ void __launch_bounds__(kSpThreads, 1)
kside_split_tc(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW0,
               const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2, const SpArgs a)
{
    extern __shared__ uint8_t sp_smem[];
    using L = SpSmemState;
    using Bk = Blocks<kLayout, kPair>;
    if (!bwd_smem_fits(sp_smem, kSpSmemState, a.err)) return;
    const SpCta c = sp_setup(sp_smem, L::kMisc, a.err, a.wait_limit_us);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t t_u = c.tmem, t_s = c.tmem + 128, t_ms = c.tmem + 256;
    const CUtensorMap* tmW[3] = {&tmW0, &tmW1, &tmW2};
    TileWalk w;
    w.init(a.total_tiles, a.tiles_per_unit);
    bool ok = true;
    if (warp >= 8) {
        setmaxnreg_dec<kBwdRegsIssuer>();
        if (warp == 8) {
        const bool one = lane == 0;
        auto load = [&](const CUtensorMap& tm, uint32_t off, int bar, const TileWalk& t) {
            mbar_arrive_expect_tx(c.bar(bar), kTileBytes);
            for (int b = 0; b < 2; ++b) Bk::load(c.sb + off + b * kHalfTileBytes, &tm, c.bar(bar), b, t.lt * kTile, t.g, a.H);
        };
        auto load_w = [&](const TileWalk& t) {
            mbar_arrive_expect_tx(c.bar(SP_SEG), a.w_parts * kWBytes);
            for (int s = 0; s < a.w_parts; ++s)
                for (int b = 0; b < 2; ++b)
                    tma_load_3d(c.sb + L::kW + s * kWBytes + b * (kWBytes / 2), tmW[s], c.bar(SP_SEG), 64 * b, 0, Bk::weights(t.g, a.H));
        };
        if (one && !w.done()) {
            load_w(w);
            load(tmK, L::kX, SP_X, w);
            load(tmV, L::kY, SP_Y, w);
        }
        for (; !w.done(); w.next()) {
            const uint32_t par = w.i;
            TileWalk nx = w;
            nx.next();
            if (w.first()) ok &= c.wait(SP_SEG, w.seg, kErrSeg);
            ok &= c.wait(SP_X, par, kErrMmaLoad);
            if (one) {
                for (int s = a.w_parts - 1; s >= 0; --s) sp_logits(t_u, c.sb + L::kX, c.sb + L::kW + s * kWBytes, s == a.w_parts - 1 ? 0u : 1u);
                if (!(a.test_unmet && w.i == 0)) mma_commit(c.bar(SP_U));
            }
            __syncwarp();
            ok &= c.wait(SP_U, par, kErrMmaU);
            if (one && !nx.done()) {   // K's tile has been read; W changes with the unit
                load(tmK, L::kX, SP_X, nx);
                if (nx.first()) load_w(nx);
            }
            ok &= c.wait(SP_Y, par, kErrMmaLoad);
            if (!sp_meet(ok)) break;   // phi is written
            if (one) {
                for (int s = 2; s >= 0; --s) sp_outer<8>(t_s, c.sb + L::kY, c.sb + L::kPhi + s * kTileBytes, kHalfTileBytes, s == 2 ? 0u : 1u);
                mma_commit(c.bar(SP_D));
            }
            __syncwarp();
            ok &= c.wait(SP_D, par, kErrMmaAcc);
            if (one && !nx.done()) load(tmV, L::kY, SP_Y, nx);
            if (!sp_meet(ok)) break;   // the tile's sums are in the master copy
        }
        if (!ok || !w.done()) sp_settle(c, w.i, w.seg);
        }
    } else {
        setmaxnreg_inc<kBwdRegsCompute>();
        const int half = warp >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t lb = (uint32_t)((warp & 3) * 32) << 16;
        float4* xch = reinterpret_cast<float4*>(c.smem + L::kXch);
        float z0 = 0.f, z1 = 0.f;
        for (; !w.done(); w.next()) {
            const uint32_t par = w.i;
            ok &= c.wait(SP_U, par, kErrSoftmaxU);
            float e[64], sp, sn;
            sp_exps<kPair>(t_u + lb, half, e, sp, sn);
            const float4 s = sp_exchange<kPair>(xch, half, row, make_float4(sp, sn, 0.f, 0.f));
            // rows past the end, and the head a last pair does not have, add nothing
            const bool valid = w.lt * kTile + row < a.n && Bk::head(w.g, half) < a.heads;
            const float ip = valid ? 1.f / s.x : 0.f, in = valid ? 1.f / s.y : 0.f;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                e[j] *= ip;
                e[32 + j] *= in;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int col = h ? SpCols<kPair>::neg(half) : SpCols<kPair>::pos(half);
                uint8_t* blk = c.smem + L::kPhi + (col >> 6) * kHalfTileBytes;
#pragma unroll
                for (int q = 0; q < 4; ++q) sp_store8<3>(blk + sw_chunk(row, ((col & 63) >> 3) + q), kTileBytes, &e[32 * h + 8 * q]);
            }
            if (!sp_meet(ok)) { ok = false; break; }
            float s0, s1;
            sp_warp_sum64([&](int i) { return e[i]; }, s0, s1);
            z0 = w.first() ? s0 : z0 + s0;
            z1 = w.first() ? s1 : z1 + s1;
            ok &= c.wait(SP_D, par, kErrDrain);
            sp_drain<64, false>(t_ms + lb + 64 * half, t_s + lb + 64 * half, 0, w.first());
            if (w.last()) {
                float* rec = a.rec + (size_t)(blockIdx.x + w.g) * kE;
                sp_store_master<64>(rec + (size_t)64 * half * kD, t_ms + lb + 64 * half, row);
                sp_store_vec<kPair>(reinterpret_cast<float*>(c.smem + L::kXch), rec + kD * kD, warp, lane, z0, z1);
            }
            if (!sp_meet(ok)) { ok = false; break; }
        }
    }
    sp_teardown(c);
}

// ---- query side: dq, and the sums of dS, dz, dW_q ------------------------------------------------------------------------
// TMEM: logits / dW | dS's lower parts = T = dq | dS's hi part | masters of dS and dW
template <int kLayout, int kPair, int kMixB>
__global__ void __launch_bounds__(kSpThreads, 1)
qside_bwd_split_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmDQ,
                   const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2,
                   const __grid_constant__ CUtensorMap tmS0, const __grid_constant__ CUtensorMap tmS1, const __grid_constant__ CUtensorMap tmS2,
                   const SpArgs a)
{
    extern __shared__ uint8_t sp_smem[];
    using L = SpSmem;
    using Bk = Blocks<kLayout, kPair>;
    if (!bwd_smem_fits(sp_smem, kSpSmem, a.err)) return;
    const SpCta c = sp_setup(sp_smem, L::kMisc, a.err, a.wait_limit_us);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t t_u = c.tmem, t_dw = c.tmem, t_t = c.tmem + 64, t_ds = c.tmem + 192, t_mds = c.tmem + 320, t_mdw = c.tmem + 448;
    constexpr uint32_t kPart = 64 * 128 * 2;   // one part of phi / den of 64 tokens in the pool: two blocks of 8 KB
    const CUtensorMap* tmS[3] = {&tmS0, &tmS1, &tmS2};
    TileWalk w;
    w.init(a.total_tiles, a.tiles_per_unit);
    bool ok = true;
    float dr_acc = 0.f;
    if (warp >= 8) {
        setmaxnreg_dec<kBwdRegsIssuer>();
        if (warp == 8) {
        const bool one = lane == 0;
        auto load = [&](const CUtensorMap& tm, uint32_t off, int bar, const TileWalk& t) {
            mbar_arrive_expect_tx(c.bar(bar), kTileBytes);
            for (int b = 0; b < 2; ++b) Bk::load(c.sb + off + b * kHalfTileBytes, &tm, c.bar(bar), b, t.lt * kTile, t.g, a.H);
        };
        auto load_w = [&](const CUtensorMap& tm, uint32_t off, int bar, const TileWalk& t) {
            for (int b = 0; b < 2; ++b) tma_load_3d(c.sb + off + b * (kWBytes / 2), &tm, c.bar(bar), 64 * b, 0, Bk::weights(t.g, a.H));
        };
        auto load_seg = [&](const TileWalk& t) {
            mbar_arrive_expect_tx(c.bar(SP_SEG), 3 * kTileBytes + kWBytes);
            load_w(tmW0, L::kW, SP_SEG, t);
            for (int s = 0; s < 3; ++s)
                for (int b = 0; b < 2; ++b) tma_load_3d(c.sb + L::kImg + s * kTileBytes + b * kHalfTileBytes, tmS[s], c.bar(SP_SEG), 64 * b, 0, t.g);
        };
        auto load_pool = [&](const TileWalk& t) {
            if (a.w_parts == 1) return;
            mbar_arrive_expect_tx(c.bar(SP_WP), 2 * kWBytes);
            load_w(tmW1, L::kPool, SP_WP, t);
            load_w(tmW2, L::kPool + kWBytes, SP_WP, t);
        };
        if (one && !w.done()) {
            load_seg(w);
            load_pool(w);
            load(tmQ, L::kX, SP_X, w);
            load(tmG, L::kY, SP_Y, w);
        }
        for (; !w.done(); w.next()) {
            const uint32_t par = w.i;
            TileWalk nx = w;
            nx.next();
            if (one && !nx.done())
                for (int b = 0; b < 2; ++b) {
                    Bk::prefetch_l2(&tmQ, b, nx.lt * kTile, nx.g, a.H);
                    Bk::prefetch_l2(&tmG, b, nx.lt * kTile, nx.g, a.H);
                }
            if (w.first()) ok &= c.wait(SP_SEG, w.seg, kErrSeg);
            ok &= c.wait(SP_X, par, kErrMmaLoad);
            if (a.w_parts == 3) ok &= c.wait(SP_WP, par, kErrMmaLoad);
            if (one) {
                for (int s = a.w_parts - 1; s >= 0; --s)
                    sp_logits(t_u, c.sb + L::kX, c.sb + (s ? L::kPool + (s - 1) * kWBytes : L::kW), s == a.w_parts - 1 ? 0u : 1u);
                if (!(a.test_unmet && w.i == 0)) mma_commit(c.bar(SP_U));
            }
            __syncwarp();
            ok &= c.wait(SP_Y, par, kErrMmaLoad);
            if (one) {
                for (int s = 2; s >= 0; --s) sp_t(t_t, c.sb + L::kY, c.sb + L::kImg + s * kTileBytes, s == 2 ? 0u : 1u);
                mma_commit(c.bar(SP_T));
            }
            __syncwarp();
            for (int hh = 0; hh < 2; ++hh) {   // dS^T += dO^T (phi / den), 64 tokens at a time
                if (!sp_meet(ok)) goto q_out;
                if (one) {
                    for (int s = 2; s >= 1; --s)
                        sp_outer<4>(t_t, c.sb + L::kY + hh * 8192, c.sb + L::kPool + s * kPart, kPart / 2, (s == 2 && hh == 0) ? 0u : 1u);
                    sp_outer<4>(t_ds, c.sb + L::kY + hh * 8192, c.sb + L::kPool, kPart / 2, hh == 0 ? 0u : 1u);
                    mma_commit(c.bar(hh ? SP_D : SP_A));
                }
                __syncwarp();
            }
            ok &= c.wait(SP_D, par, kErrMmaAcc);
            if (a.w_parts == 3) {
                if (one) {
                    mbar_arrive_expect_tx(c.bar(SP_WY), kWBytes);
                    load_w(tmW1, L::kY, SP_WY, w);
                }
                __syncwarp();
                ok &= c.wait(SP_WY, par, kErrMmaLoad);
            }
            if (!sp_meet(ok)) goto q_out;   // du is written, dS has left its accumulators
            if (one) {
                for (int s = 2; s >= 0; --s) sp_dw(t_dw, c.sb + L::kX, c.sb + L::kPool + s * kWBytes, s == 2 ? 0u : 1u);
                sp_dx(t_t, c.sb + L::kPool + kWBytes, c.sb + L::kW, 0u);
                if (a.w_parts == 3) sp_dx(t_t, c.sb + L::kPool, c.sb + L::kY, 1u);
                sp_dx(t_t, c.sb + L::kPool, c.sb + L::kW, 1u);
                mma_commit(c.bar(SP_F));
            }
            __syncwarp();
            ok &= c.wait(SP_F, par, kErrMmaAcc);
            if (one && !nx.done()) {
                load(tmQ, L::kX, SP_X, nx);
                if (nx.first()) load_seg(nx);
                load_pool(nx);
            }
            __syncwarp();
            if (!sp_meet(ok)) goto q_out;   // dq is staged in dO's tile
            if (one) {
                for (int b = 0; b < 2; ++b)
                    if (Bk::head(w.g, b) < a.heads) act_store<kLayout>(&tmDQ, c.sb + L::kY + b * kHalfTileBytes, Bk::x(b), w.lt * kTile, Bk::head(w.g, b), a.H);
                bulk_commit_group();
                bulk_wait_group_read<0>();
                if (!nx.done()) load(tmG, L::kY, SP_Y, nx);
            }
            __syncwarp();
        }
    q_out:
        if (one) bulk_wait_group<0>();
        __syncwarp();
        if (!w.done()) sp_settle(c, w.i, w.seg);
        }
    } else {
        setmaxnreg_inc<kBwdRegsCompute>();
        const int half = warp >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t lb = (uint32_t)((warp & 3) * 32) << 16;
        const int cp = SpCols<kPair>::pos(half), cn = SpCols<kPair>::neg(half);
        float4* xch = reinterpret_cast<float4*>(c.smem + L::kPool);
        float z0 = 0.f, z1 = 0.f;
        for (; !w.done(); w.next()) {
            const uint32_t par = w.i;
            if (w.first()) {
                if (tid < kD) c.vec[tid] = a.vec[(size_t)w.g * kD + tid];
                sp_sync();
            }
            ok &= c.wait(SP_U, par, kErrSoftmaxU);
            float e[64], sp, sn;
            sp_exps<kPair>(t_u + lb, half, e, sp, sn);
            const float4 m1 = make_float4(sp, sn, sp_dot_vec(e, c.vec + cp), sp_dot_vec(e + 32, c.vec + cn));
            const float4 s1 = sp_exchange<kPair>(xch, half, row, m1);
            const bool valid = w.lt * kTile + row < a.n && Bk::head(w.g, half) < a.heads;
            const float ip = 1.f / s1.x, in = 1.f / s1.y;
            const float den = s1.z * ip + s1.w * in;          // phi . z
            const float inv = valid ? 1.f / den : 0.f, sc = inv * a.lin_scale;
            ok &= c.wait(SP_T, par, kErrEpilogue);
            float x[64];
            {
                uint32_t r[32];
                tmem_ld_x32(t_t + lb + cp, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) x[j] = __uint_as_float(r[j]);
                tmem_ld_x32(t_t + lb + cn, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) x[32 + j] = __uint_as_float(r[j]);
            }
            const float4 s2 = sp_exchange<kPair>(xch + 256, half, row, make_float4(sp_dot(e, x), sp_dot(e + 32, x + 32), 0.f, 0.f));
            const float go = valid ? (s2.x * ip + s2.y * in) * inv : 0.f;   // dO . o
            // p . dphi of each softmax, dphi = sc (T - go z)
            const float dp = sc * ip * (s2.x - go * s1.z), dn = sc * in * (s2.y - go * s1.w);
            if (kMixB) {
                if (half == 0 || kPair) dr_acc -= go;
                if (valid) {
                    const int hd = Bk::head(w.g, half);
                    const __nv_bfloat16* ap = a.mix_a + (size_t)(hd / a.H) * a.str_batch + (size_t)(hd % a.H) * a.str_head +
                                              (size_t)(w.lt * kTile + row) * a.str_token + Bk::x(half);
                    const uint8_t* gblk = c.smem + L::kY + half * kHalfTileBytes;
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch) {
                        const uint4 av = __ldg(reinterpret_cast<const uint4*>(ap) + ch);
                        const uint4 gv = *reinterpret_cast<const uint4*>(gblk + sw_chunk(row, ch));
                        const uint32_t aw[4] = {av.x, av.y, av.z, av.w}, gw[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            dr_acc = fmaf(bf_lo(gw[q]), bf_lo(aw[q]), dr_acc);
                            dr_acc = fmaf(bf_hi(gw[q]), bf_hi(aw[q]), dr_acc);
                        }
                    }
                }
            }
            if (!kPair) sp_sync();   // the exchanged sums have been read: the pool takes phi / den
            const float fp = ip * sc, fn = in * sc;   // phi / den = e * fp, e * fn
            auto put_phi = [&]() {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int col = h ? cn : cp;
                    uint8_t* blk = c.smem + L::kPool + (col >> 6) * (kPart / 2);
                    const float f = h ? fn : fp;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = e[32 * h + 8 * q + i] * f;
                        sp_store8<3>(blk + sw_chunk(row & 63, ((col & 63) >> 3) + q), kPart, v);
                    }
                }
            };
            const bool firsthalf = row < 64;
            if (firsthalf) put_phi();
            if (!sp_meet(ok)) { ok = false; break; }
            // du while the first half of dS is formed
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 zp = *reinterpret_cast<const float4*>(c.vec + cp + j), zn = *reinterpret_cast<const float4*>(c.vec + cn + j);
                const float zpa[4] = {zp.x, zp.y, zp.z, zp.w}, zna[4] = {zn.x, zn.y, zn.z, zn.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float gp = sc * fmaf(-go, zpa[i], x[j + i]), gn = sc * fmaf(-go, zna[i], x[32 + j + i]);
                    x[j + i] = (e[j + i] * ip) * (gp - dp) - (e[32 + j + i] * in) * (gn - dn);
                }
            }
            if (!firsthalf) {
                ok &= c.wait(SP_A, par, kErrMmaAcc);
                put_phi();
            }
            if (!sp_meet(ok)) { ok = false; break; }
            {
                float s0, s1v;   // dz += phi^T dden
                const float tp = -go * fp, tn = -go * fn;
                sp_warp_sum64([&](int i) { return e[i] * (i < 32 ? tp : tn); }, s0, s1v);
                z0 = w.first() ? s0 : z0 + s0;
                z1 = w.first() ? s1v : z1 + s1v;
            }
            ok &= c.wait(SP_D, par, kErrMmaAcc);
#pragma unroll
            for (int q = 0; q < 4; ++q) sp_store8<3>(c.smem + L::kPool + sw_chunk(row, 4 * half + q), kWBytes, &x[8 * q]);
            sp_drain<64, true>(t_mds + lb + 64 * half, t_ds + lb + 64 * half, t_t + lb + 64 * half, w.first());
            if (!sp_meet(ok)) { ok = false; break; }
            ok &= c.wait(SP_F, par, kErrStore);
            sp_drain<32, false>(t_mdw + lb + 32 * half, t_dw + lb + 32 * half, 0, w.first());
            sp_stage(t_t + lb + 64 * half, c.smem + L::kY + half * kHalfTileBytes, row);
            if (w.last()) {
                float* rec = a.rec + (size_t)(blockIdx.x + w.g) * kE;
                sp_store_master<64>(rec + (size_t)64 * half * kD, t_mds + lb + 64 * half, row);
                sp_store_master<32>(a.rec_w + (size_t)(blockIdx.x + w.g) * kWRec + (size_t)32 * half * kD, t_mdw + lb + 32 * half, row);
                // the weights' parts of the next tile may be on their way into the pool's first 32 KB
                sp_store_vec<kPair>(reinterpret_cast<float*>(c.smem + L::kPool + 2 * kWBytes), rec + kD * kD, warp, lane, z0, z1);
            }
            if (!sp_meet(ok)) { ok = false; break; }
        }
    }
    if (kMixB) {
        // dL/dr: threads by a butterfly, warps in order (the tiles are free: every copy into shared memory has been waited for)
        __syncthreads();
        float* red = c.vec;
        float v = dr_acc;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && warp < 8) red[warp] = v;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
            for (int i = 0; i < 8; ++i) s += red[i];
            a.part_dr[blockIdx.x] = s;
        }
    }
    sp_teardown(c);
}

// ---- key side: dk, dv, and the sums of dW_k ------------------------------------------------------------------------------
// TMEM: logits / dW | T = dv | dk | master of dW
template <int kLayout, int kPair>
__global__ void __launch_bounds__(kSpThreads, 1)
kside_bwd_split_tc(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmDK,
                   const __grid_constant__ CUtensorMap tmDV, const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
                   const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmS0, const __grid_constant__ CUtensorMap tmS1,
                   const __grid_constant__ CUtensorMap tmS2, const SpArgs a)
{
    extern __shared__ uint8_t sp_smem[];
    using L = SpSmem;
    using Bk = Blocks<kLayout, kPair>;
    if (!bwd_smem_fits(sp_smem, kSpSmem, a.err)) return;
    const SpCta c = sp_setup(sp_smem, L::kMisc, a.err, a.wait_limit_us);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t t_u = c.tmem, t_dw = c.tmem, t_t = c.tmem + 64, t_dk = c.tmem + 192, t_mdw = c.tmem + 320;
    const CUtensorMap* tmS[3] = {&tmS0, &tmS1, &tmS2};
    TileWalk w;
    w.init(a.total_tiles, a.tiles_per_unit);
    bool ok = true;
    if (warp >= 8) {
        setmaxnreg_dec<kBwdRegsIssuer>();
        if (warp == 8) {
        const bool one = lane == 0;
        auto load = [&](const CUtensorMap& tm, uint32_t off, int bar, const TileWalk& t) {
            mbar_arrive_expect_tx(c.bar(bar), kTileBytes);
            for (int b = 0; b < 2; ++b) Bk::load(c.sb + off + b * kHalfTileBytes, &tm, c.bar(bar), b, t.lt * kTile, t.g, a.H);
        };
        auto load_w = [&](const CUtensorMap& tm, uint32_t off, int bar, const TileWalk& t) {
            for (int b = 0; b < 2; ++b) tma_load_3d(c.sb + off + b * (kWBytes / 2), &tm, c.bar(bar), 64 * b, 0, Bk::weights(t.g, a.H));
        };
        auto load_seg = [&](const TileWalk& t) {
            mbar_arrive_expect_tx(c.bar(SP_SEG), 3 * kTileBytes + kWBytes);
            load_w(tmW0, L::kW, SP_SEG, t);
            for (int s = 0; s < 3; ++s)
                for (int b = 0; b < 2; ++b) tma_load_3d(c.sb + L::kImg + s * kTileBytes + b * kHalfTileBytes, tmS[s], c.bar(SP_SEG), 64 * b, 0, t.g);
        };
        auto load_pool = [&](const TileWalk& t) {
            if (a.w_parts == 1) return;
            mbar_arrive_expect_tx(c.bar(SP_WP), 2 * kWBytes);
            load_w(tmW1, L::kPool, SP_WP, t);
            load_w(tmW2, L::kPool + kWBytes, SP_WP, t);
        };
        if (one && !w.done()) {
            load_seg(w);
            load_pool(w);
            load(tmK, L::kX, SP_X, w);
            load(tmV, L::kY, SP_Y, w);
        }
        for (; !w.done(); w.next()) {
            const uint32_t par = w.i;
            TileWalk nx = w;
            nx.next();
            if (one && !nx.done())
                for (int b = 0; b < 2; ++b) {
                    Bk::prefetch_l2(&tmK, b, nx.lt * kTile, nx.g, a.H);
                    Bk::prefetch_l2(&tmV, b, nx.lt * kTile, nx.g, a.H);
                }
            if (w.first()) ok &= c.wait(SP_SEG, w.seg, kErrSeg);
            ok &= c.wait(SP_X, par, kErrMmaLoad);
            if (a.w_parts == 3) ok &= c.wait(SP_WP, par, kErrMmaLoad);
            if (one) {
                for (int s = a.w_parts - 1; s >= 0; --s)
                    sp_logits(t_u, c.sb + L::kX, c.sb + (s ? L::kPool + (s - 1) * kWBytes : L::kW), s == a.w_parts - 1 ? 0u : 1u);
                if (!(a.test_unmet && w.i == 0)) mma_commit(c.bar(SP_U));
            }
            __syncwarp();
            ok &= c.wait(SP_Y, par, kErrMmaLoad);
            if (one) {
                for (int s = 2; s >= 0; --s) sp_t(t_t, c.sb + L::kY, c.sb + L::kImg + s * kTileBytes, s == 2 ? 0u : 1u);
                mma_commit(c.bar(SP_T));
            }
            __syncwarp();
            if (!sp_meet(ok)) goto k_out;   // phi is written: hi over V's tile, mid in the pool
            if (one) {
                sp_dv(t_t, c.sb + L::kPool, c.sb + L::kImg, 0u);
                sp_dv(t_t, c.sb + L::kY, c.sb + L::kImg + kTileBytes, 1u);
                sp_dv(t_t, c.sb + L::kY, c.sb + L::kImg, 1u);
                mma_commit(c.bar(SP_D));
            }
            __syncwarp();
            ok &= c.wait(SP_D, par, kErrMmaAcc);
            if (a.w_parts == 3) {
                if (one) {
                    mbar_arrive_expect_tx(c.bar(SP_WY), kWBytes);
                    load_w(tmW1, L::kY, SP_WY, w);
                }
                __syncwarp();
                ok &= c.wait(SP_WY, par, kErrMmaLoad);
            }
            if (!sp_meet(ok)) goto k_out;   // du is written
            if (one) {
                for (int s = 2; s >= 0; --s) sp_dw(t_dw, c.sb + L::kX, c.sb + L::kPool + s * kWBytes, s == 2 ? 0u : 1u);
                sp_dx(t_dk, c.sb + L::kPool + kWBytes, c.sb + L::kW, 0u);
                if (a.w_parts == 3) sp_dx(t_dk, c.sb + L::kPool, c.sb + L::kY, 1u);
                sp_dx(t_dk, c.sb + L::kPool, c.sb + L::kW, 1u);
                mma_commit(c.bar(SP_F));
            }
            __syncwarp();
            ok &= c.wait(SP_F, par, kErrMmaAcc);
            if (one && !nx.done()) {
                if (nx.first()) load_seg(nx);
                load_pool(nx);
            }
            __syncwarp();
            if (!sp_meet(ok)) goto k_out;   // dv is staged in V's tile, dk in K's
            if (one) {
                for (int b = 0; b < 2; ++b)
                    if (Bk::head(w.g, b) < a.heads) {
                        act_store<kLayout>(&tmDK, c.sb + L::kX + b * kHalfTileBytes, Bk::x(b), w.lt * kTile, Bk::head(w.g, b), a.H);
                        act_store<kLayout>(&tmDV, c.sb + L::kY + b * kHalfTileBytes, Bk::x(b), w.lt * kTile, Bk::head(w.g, b), a.H);
                    }
                bulk_commit_group();
                bulk_wait_group_read<0>();
                if (!nx.done()) {
                    load(tmK, L::kX, SP_X, nx);
                    load(tmV, L::kY, SP_Y, nx);
                }
            }
            __syncwarp();
        }
    k_out:
        if (one) bulk_wait_group<0>();
        __syncwarp();
        if (!w.done()) sp_settle(c, w.i, w.seg);
        }
    } else {
        setmaxnreg_inc<kBwdRegsCompute>();
        const int half = warp >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t lb = (uint32_t)((warp & 3) * 32) << 16;
        const int cp = SpCols<kPair>::pos(half), cn = SpCols<kPair>::neg(half);
        float4* xch = reinterpret_cast<float4*>(c.smem + L::kPool);
        for (; !w.done(); w.next()) {
            const uint32_t par = w.i;
            if (w.first()) {
                if (tid < kD) c.vec[tid] = a.vec[(size_t)w.g * kD + tid];   // dz
                sp_sync();
            }
            ok &= c.wait(SP_U, par, kErrSoftmaxU);
            float e[64], sp, sn;
            sp_exps<kPair>(t_u + lb, half, e, sp, sn);
            const float4 m1 = make_float4(sp, sn, sp_dot_vec(e, c.vec + cp), sp_dot_vec(e + 32, c.vec + cn));
            const float4 s1 = sp_exchange<kPair>(xch, half, row, m1);
            const float ip = 1.f / s1.x, in = 1.f / s1.y;
            ok &= c.wait(SP_T, par, kErrEpilogue);
            float x[64];
            {
                uint32_t r[32];
                tmem_ld_x32(t_t + lb + cp, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) x[j] = __uint_as_float(r[j]);
                tmem_ld_x32(t_t + lb + cn, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) x[32 + j] = __uint_as_float(r[j]);
            }
            const float4 s2 = sp_exchange<kPair>(xch + 256, half, row, make_float4(sp_dot(e, x), sp_dot(e + 32, x + 32), 0.f, 0.f));
            const float dp = ip * (s2.x + s1.z), dn = in * (s2.y + s1.w);   // p . dphi, dphi = T + dz
            if (!kPair) sp_sync();   // the exchanged sums have been read: the pool takes phi's mid part
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int col = h ? cn : cp;
                uint8_t* blk = c.smem + L::kY + (col >> 6) * kHalfTileBytes;
                const float f = h ? in : ip;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] = e[32 * h + 8 * q + i] * f;
                    sp_store8<2>(blk + sw_chunk(row, ((col & 63) >> 3) + q), L::kPool - L::kY, v);
                }
            }
            if (!sp_meet(ok)) { ok = false; break; }
            // du while dv is formed
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 zp = *reinterpret_cast<const float4*>(c.vec + cp + j), zn = *reinterpret_cast<const float4*>(c.vec + cn + j);
                const float zpa[4] = {zp.x, zp.y, zp.z, zp.w}, zna[4] = {zn.x, zn.y, zn.z, zn.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    x[j + i] = (e[j + i] * ip) * ((x[j + i] + zpa[i]) - dp) - (e[32 + j + i] * in) * ((x[32 + j + i] + zna[i]) - dn);
            }
            ok &= c.wait(SP_D, par, kErrMmaAcc);
#pragma unroll
            for (int q = 0; q < 4; ++q) sp_store8<3>(c.smem + L::kPool + sw_chunk(row, 4 * half + q), kWBytes, &x[8 * q]);
            if (!sp_meet(ok)) { ok = false; break; }
            ok &= c.wait(SP_F, par, kErrStore);
            sp_drain<32, false>(t_mdw + lb + 32 * half, t_dw + lb + 32 * half, 0, w.first());
            sp_stage(t_t + lb + 64 * half, c.smem + L::kY + half * kHalfTileBytes, row);
            sp_stage(t_dk + lb + 64 * half, c.smem + L::kX + half * kHalfTileBytes, row);
            if (w.last()) sp_store_master<32>(a.rec_w + (size_t)(blockIdx.x + w.g) * kWRec + (size_t)32 * half * kD, t_mdw + lb + 32 * half, row);
            if (!sp_meet(ok)) { ok = false; break; }
        }
    }
    sp_teardown(c);
}

// ---- combines ------------------------------------------------------------------------------------------------------------
// Fixed-order sum of the (CTA, unit) records of S, z or dS, dz: the three bf16 images [f][c] of the unit (pair: zero outside the
// heads' own blocks), the vector [128], and, where `state` is given, the heads' own records (S row-major [f][c], then z).
// grid = (ceil(kE / 256), units), 256 threads: 64 lanes x four slices of the list of CTAs, the slices added in order.
template <int kPair>
static __global__ void __launch_bounds__(256)
combine_split(const float* __restrict__ rec, __nv_bfloat16* __restrict__ img0, __nv_bfloat16* __restrict__ img1, __nv_bfloat16* __restrict__ img2,
              float* __restrict__ vec, float* __restrict__ state, int heads, int tiles_per_unit, long long total_tiles, long long P)
{
    pdl_trigger();
    pdl_wait();
    __shared__ float4 part_s[4][64];
    const int lane = threadIdx.x & 63, slice = threadIdx.x >> 6;
    const int e = (blockIdx.x * 64 + lane) * 4, g = blockIdx.y;
    const long long c0 = tile_owner((long long)g * tiles_per_unit, total_tiles, P);
    const long long c1 = tile_owner((long long)(g + 1) * tiles_per_unit - 1, total_tiles, P);
    const int cnt = (int)(c1 - c0) + 1, per = (cnt + 3) / 4, b = min(cnt, slice * per), eb = min(cnt, b + per);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < kE) {
        const float* src = rec + (size_t)(c0 + g) * kE + e;
#pragma unroll 4
        for (int i = b; i < eb; ++i) {
            const float4 x = *reinterpret_cast<const float4*>(src + (size_t)i * kE);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
    }
    part_s[slice][lane] = s;
    __syncthreads();
    if (slice != 0 || e >= kE) return;
#pragma unroll
    for (int q = 1; q < 4; ++q) {
        const float4 x = part_s[q][lane];
        s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    constexpr int d = kPair ? 64 : 128;
    if (e >= kD * kD) {
        const int i = e - kD * kD;
        *reinterpret_cast<float4*>(vec + (size_t)g * kD + i) = s;
        const int hd = kPair ? 2 * g + (i >> 6) : g;
        if (state && hd < heads) *reinterpret_cast<float4*>(state + (size_t)hd * (d * d + d) + d * d + (i & (d - 1))) = s;
        return;
    }
    const int f = e / kD, cc = e % kD;
    const bool own = !kPair || (f >> 6) == (cc >> 6);
    if (!own) s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (state && own) {
        const int hd = kPair ? 2 * g + (f >> 6) : g;
        if (hd < heads) *reinterpret_cast<float4*>(state + (size_t)hd * (d * d + d) + (size_t)(f & (d - 1)) * d + (cc & (d - 1))) = s;
    }
    float r[4] = {s.x, s.y, s.z, s.w};
    __nv_bfloat16* img[3] = {img0, img1, img2};
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const uint32_t w0 = pack_bf16(r[0], r[1]), w1 = pack_bf16(r[2], r[3]);
        r[0] -= bf_lo(w0); r[1] -= bf_hi(w0); r[2] -= bf_lo(w1); r[3] -= bf_hi(w1);
        *reinterpret_cast<uint2*>(img[p] + (size_t)g * kD * kD + e) = make_uint2(w0, w1);
    }
}

// dW[w][c][j]: sum over the heads that use weight matrix w (per_head: head % H == w; shared: all), ascending, and over the CTAs
// of each one's unit, ascending, of the unit's record [j'][c'] (pair: the head's own block).  grid = (ceil(d*d/2 / 256), per_head ?
// H : 1), 256 threads: 64 lanes of four consecutive c x four slices of the list, added in order.
template <int kPair>
static __global__ void __launch_bounds__(256)
combine_wgrad_split(const float* __restrict__ rec, float* __restrict__ dW, int heads, int H, int per_head, int tiles_per_unit, long long total_tiles,
                    long long P)
{
    pdl_trigger();
    pdl_wait();
    constexpr int d = kPair ? 64 : 128, m = d / 2;
    __shared__ float4 part_s[4][64];
    const int lane = threadIdx.x & 63, slice = threadIdx.x >> 6, wsel = blockIdx.y;
    const int r = (blockIdx.x * 64 + lane) * 4, j = r / d, cc = r % d;   // index in the head's part of the record
    const int step = per_head ? H : 1, first = per_head ? wsel : 0, pairs = (heads - first + step - 1) / step;
    const bool whole = pairs >= 4;   // many heads: whole heads per slice; few: each head's list in four parts
    const int per_slice = (pairs + 3) / 4;
    const int i0 = whole ? min(pairs, slice * per_slice) : 0, i1 = whole ? min(pairs, i0 + per_slice) : pairs;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = i0; i < i1; ++i) {
        const int hd = first + i * step, g = kPair ? hd >> 1 : hd, blk = kPair ? hd & 1 : 0;
        const long long c0 = tile_owner((long long)g * tiles_per_unit, total_tiles, P);
        const long long c1 = tile_owner((long long)(g + 1) * tiles_per_unit - 1, total_tiles, P);
        const int cnt = (int)(c1 - c0) + 1, per = whole ? cnt : (cnt + 3) / 4;
        const int b = whole ? 0 : min(cnt, slice * per), eb = min(cnt, b + per);
        const float* src = rec + (size_t)(c0 + g) * kWRec + (size_t)(32 * blk + j) * kD + 64 * blk + cc;
#pragma unroll 4
        for (int k = b; k < eb; ++k) {
            const float4 x = *reinterpret_cast<const float4*>(src + (size_t)k * kWRec);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
    }
    part_s[slice][lane] = s;
    __syncthreads();
    if (slice != 0) return;
#pragma unroll
    for (int q = 1; q < 4; ++q) {
        const float4 x = part_s[q][lane];
        s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    float* o = dW + (size_t)wsel * d * m + (size_t)cc * m + j;
    o[0] = s.x;
    o[m] = s.y;
    o[2 * m] = s.z;
    o[3 * m] = s.w;
}

}  // namespace tc
}  // namespace linattn
