// CUDA-core (fp32 FMA) kernels for linear attention with the Hedgehog feature map.
//
// These are the general path: fp32 and bf16 storage, d = 64 or 128, any n >= 1.  All arithmetic
// is fp32.  Three launches per forward:
//   kside_simt   : per run of token tiles and per (b,h) it touches, phi(k) (Eq. 6) and the partial
//                  sums of S = sum_j phi(k_j)^T v_j and z = sum_j phi(k_j) (Eq. 5)
//   combine_state: fixed-order sum of the partials (deterministic)
//   qside_simt   : phi(q) (Eq. 6), o_i = phi(q_i) S / (phi(q_i) . z) (Eq. 5)
//
// The bound is the fp32 FMA rate (72.9 TFLOP/s measured with packed pairs; scalar FMAs whose operands are all registers
// stop at 60: the packed form needs half the register reads), so every product is a register-tiled loop of packed FMAs
// (fma.rn.f32x2) fed by 16-byte shared-memory loads:
//   * a group of JG = d/8 lanes owns a token: its rows of x and phi are written and read by that group only, so the feature
//     map and phi(q) S need no CTA-wide barrier, and softmax rows are reduced by shuffles within the group;
//   * a thread holds TM tokens x 4 logits of the logits product, TM x 8 of phi(q) S and an 8 x 8 block of S.
// The token tiles of all (b,h) pairs form one head-major sequence of which every CTA takes a contiguous run (a multiple
// of the tile per CTA whatever n and the number of heads; a grid of splits x heads left a nearly empty second wave: 300
// CTAs for 296 places at 12 heads).
// Measured at B=1 H=12 n=32760 d=128 fp32: 0.94 ms a forward, 41 TFLOP/s, FMA pipe 59 / 64 % busy on the key / query side
// (3.47 ms with one 32-token chunk per CTA, eight threads a token and scalar FMAs: about four FMAs per shared-memory load);
// at B=1 H=2 n=1024 d=64: 22.5 us (59.3 us).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "f32x2.cuh"
#include "launch.cuh"

namespace linattn {

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void store_out(float* p, float x) { *p = x; }
__device__ __forceinline__ void store_out(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }
// four consecutive values; 16-byte (fp32) or 8-byte (bf16) aligned
__device__ __forceinline__ void store_out4(float* p, float a, float b, float c, float d) { *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d); }
__device__ __forceinline__ void store_out4(__nv_bfloat16* p, float a, float b, float c, float d)
{
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}
__device__ __forceinline__ float4 load4_f32(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4_f32(const __nv_bfloat16* p)
{
    const uint2 r = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ float part(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

template <int D> struct SimtShape {
    static constexpr int M = D / 2;
    static constexpr int PX = D + 4;       // pitch (floats) of token tiles: rows 16-byte aligned, consecutive rows 4 banks apart
    static constexpr int PW = M + 4;       // pitch of W, the same
    static constexpr int JG = M / 4;       // lanes per token: each holds 4 logits, i.e. 8 features, and 8 output columns
    static constexpr int TGW = 32 / JG;    // token groups per warp (2 at d = 128, 4 at d = 64)
    static constexpr int E = D * D + D;    // floats of a state record: S row-major [f][c], then z
};

// A CTA of NW warps works on tiles of TT tokens; a thread's TM tokens are rows tg + TG * i of the tile (tg its token group).
template <int D, int NW, int TM> struct SimtTile {
    static constexpr int kThreads = 32 * NW;
    static constexpr int TG = NW * SimtShape<D>::TGW;
    static constexpr int TT = TG * TM;
};

// Element strides of the activations [batch][head][token][feature] (feature contiguous) in memory.
struct ActStrides {
    long long token, head, batch;
    __device__ __forceinline__ size_t base(int g, int H) const { return (size_t)(g / H) * batch + (size_t)(g % H) * head; }
};

// First tile of CTA p's run when T tiles are dealt to P CTAs (head-major sequence of Tn tiles per (b,h) pair).
__host__ __device__ __forceinline__ long long run_begin(long long p, long long T, long long P) { return p * T / P; }

// acc[i][:] += sum_k a_i[k] * b[k][:]  for this thread's TM rows a_i (a + i * a_step, k contiguous) and NB groups of four
// columns (b + nb * b_step); accumulator pairs run along the columns.  SPREAD: row k of b is kept at row
// (k / M) M + (k % 4) M/4 + (k % M) / 4 with M = K/2 (the gradient kernels' order of W and of the state).
template <int K, int TM, int NB, bool SPREAD = false>
__device__ __forceinline__ void rows_times_matrix(const float* __restrict__ a, int a_step, const float* __restrict__ b, int pb,
                                                  int b_step, f32x2 (&acc)[TM][2 * NB])
{
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 av[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(a + i * a_step + k);
        const int row0 = (k / (K / 2)) * (K / 2) + (k % (K / 2)) / 4;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            ulonglong2 bv[NB];
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) bv[nb] = *reinterpret_cast<const ulonglong2*>(b + (SPREAD ? row0 + kk * (K / 8) : k + kk) * pb + nb * b_step);
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const f32x2 x = pack2(part(av[i], kk), part(av[i], kk));
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    acc[i][2 * nb] = fma2(x, bv[nb].x, acc[i][2 * nb]);
                    acc[i][2 * nb + 1] = fma2(x, bv[nb].y, acc[i][2 * nb + 1]);
                }
            }
        }
    }
}

// acc[a][:] += sum over rows t0 <= t < t1 of A[t][a] * B[t][:]  (FA consecutive columns of A, NB groups of four columns of B).
template <int FA, int NB>
__device__ __forceinline__ void rows_outer(const float* __restrict__ A, int pa, const float* __restrict__ B, int pb, int b_step,
                                           int t0, int t1, f32x2 (&acc)[FA][2 * NB])
{
#pragma unroll 4
    for (int t = t0; t < t1; ++t) {
        float4 av[FA / 4];
        ulonglong2 bv[NB];
#pragma unroll
        for (int a = 0; a < FA / 4; ++a) av[a] = *reinterpret_cast<const float4*>(A + t * pa + 4 * a);
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) bv[nb] = *reinterpret_cast<const ulonglong2*>(B + t * pb + nb * b_step);
#pragma unroll
        for (int a = 0; a < FA; ++a) {
            const f32x2 x = pack2(part(av[a / 4], a % 4), part(av[a / 4], a % 4));
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
                acc[a][2 * nb] = fma2(x, bv[nb].x, acc[a][2 * nb]);
                acc[a][2 * nb + 1] = fma2(x, bv[nb].y, acc[a][2 * nb + 1]);
            }
        }
    }
}

template <int R, int C> __device__ __forceinline__ void zero_acc(f32x2 (&acc)[R][C])
{
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) acc[r][c] = pack2(0.f, 0.f);
}

// The rows of a tile that belong to this warp's token groups: global -> shared (fp32, pitch PX); rows >= valid are zeroed.
// Only the warp itself reads them (besides CTA-wide products behind a barrier).  16-byte loads, all in flight together.
template <typename T, int D, int TG, int TM>
__device__ __forceinline__ void load_rows(const T* __restrict__ src, long long row_stride, float* __restrict__ dst, int valid)
{
    constexpr int V = 16 / (int)sizeof(T), LPR = D / V, RPI = 32 / LPR, TGW = SimtShape<D>::TGW, ROWS = TGW * TM, PX = SimtShape<D>::PX;
    constexpr int STEPS = (ROWS + RPI - 1) / RPI;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / LPR, col = (lane % LPR) * V;
    uint4 buf[STEPS];
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {
        const int r = s * RPI + sub, row = warp * TGW + r % TGW + TG * (r / TGW);
        buf[s] = make_uint4(0u, 0u, 0u, 0u);
        if (r < ROWS && row < valid) buf[s] = *reinterpret_cast<const uint4*>(src + (size_t)row * row_stride + col);
    }
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {
        const int r = s * RPI + sub, row = warp * TGW + r % TGW + TG * (r / TGW);
        if (r >= ROWS) continue;
        float* o = dst + row * PX + col;
        if constexpr (sizeof(T) == 4) {
            *reinterpret_cast<uint4*>(o) = buf[s];
        } else {
            const uint4 b = buf[s];
            *reinterpret_cast<uint4*>(o) = make_uint4(b.x << 16, b.x & 0xffff0000u, b.y << 16, b.y & 0xffff0000u);
            *reinterpret_cast<uint4*>(o + 4) = make_uint4(b.z << 16, b.z & 0xffff0000u, b.w << 16, b.w & 0xffff0000u);
        }
    }
}

template <int JG> __device__ __forceinline__ float group_sum(float x)
{
#pragma unroll
    for (int o = 1; o < JG; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// phi of this thread's tokens, TM x 8 values in registers: p[i][j] is feature 4 jg + j, p[i][4 + j] feature M + 4 jg + j of
// token tg + TG * i (jg = lane % JG).  x: the token group's first row of the tile (warp-private rows); W_s: pitch PW.
// Hedgehog: Eq. 6 with both softmaxes shifted by their maximum; relu: max(x, 0).  Rows >= valid get phi = 0 (they add
// nothing to S, z).  1 / sum is applied by multiplication, as one division per row and softmax.  SPREAD: see rows_times_matrix.
template <int D, int TG, int TM, bool SPREAD = false>
__device__ __forceinline__ void feature_map_rows(const float* __restrict__ x, const float* __restrict__ W_s, int tg, int jg,
                                                 int valid, int relu, float (&p)[TM][8])
{
    constexpr int M = SimtShape<D>::M, PX = SimtShape<D>::PX, PW = SimtShape<D>::PW, JG = SimtShape<D>::JG;
    if (relu) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 v = *reinterpret_cast<const float4*>(x + i * TG * PX + h * M + 4 * jg);
#pragma unroll
                for (int j = 0; j < 4; ++j) p[i][4 * h + j] = tg + TG * i < valid ? fmaxf(part(v, j), 0.f) : 0.f;
            }
        return;
    }
    f32x2 acc[TM][2];
    zero_acc(acc);
    rows_times_matrix<D, TM, 1, SPREAD>(x, TG * PX, W_s + 4 * jg, PW, 0, acc);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        float u[4];
        unpack2(acc[i][0], u[0], u[1]);
        unpack2(acc[i][1], u[2], u[3]);
        float umax = fmaxf(fmaxf(u[0], u[1]), fmaxf(u[2], u[3])), umin = fminf(fminf(u[0], u[1]), fminf(u[2], u[3]));
#pragma unroll
        for (int o = 1; o < JG; o <<= 1) {
            umax = fmaxf(umax, __shfl_xor_sync(0xffffffffu, umax, o));
            umin = fminf(umin, __shfl_xor_sync(0xffffffffu, umin, o));
        }
        float sp = 0.f, sn = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            p[i][j] = expf(u[j] - umax);       // softmax(+u), max-subtracted
            p[i][4 + j] = expf(umin - u[j]);   // softmax(-u): max(-u) = -min(u)
            sp += p[i][j];
            sn += p[i][4 + j];
        }
        const float keep = tg + TG * i < valid ? 1.f : 0.f;
        const float ip = keep / group_sum<JG>(sp), in = keep / group_sum<JG>(sn);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            p[i][j] *= ip;
            p[i][4 + j] *= in;
        }
    }
}

// This thread's phi (or anything laid out like it) to the token tile.
template <int D, int TG, int TM>
__device__ __forceinline__ void store_phi_rows(float* __restrict__ x, int jg, const float (&p)[TM][8])
{
    constexpr int M = SimtShape<D>::M, PX = SimtShape<D>::PX;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        *reinterpret_cast<float4*>(x + i * TG * PX + 4 * jg) = make_float4(p[i][0], p[i][1], p[i][2], p[i][3]);
        *reinterpret_cast<float4*>(x + i * TG * PX + M + 4 * jg) = make_float4(p[i][4], p[i][5], p[i][6], p[i][7]);
    }
}

// W [D][M] -> shared memory, pitch PW.
template <int D, int THREADS>
__device__ __forceinline__ void load_weights(const float* __restrict__ Wg, float* __restrict__ W_s)
{
    constexpr int M = SimtShape<D>::M, PW = SimtShape<D>::PW;
#pragma unroll 4
    for (int e = threadIdx.x; e < D * M / 4; e += THREADS)
        *reinterpret_cast<float4*>(W_s + (e / (M / 4)) * PW + (e % (M / 4)) * 4) = *reinterpret_cast<const float4*>(Wg + 4 * e);
}

// Per-thread sums of the 8 features a thread holds (p's layout) -> out[D], summed over the CTA's token groups in order.
// scratch: TG * D floats; begins and ends with the CTA's threads anywhere (the caller puts barriers around).
template <int D, int TG>
__device__ __forceinline__ void park_feature_sums(float* __restrict__ scratch, int tg, int jg, const float (&s)[8])
{
    constexpr int M = SimtShape<D>::M;
    *reinterpret_cast<float4*>(scratch + tg * D + 4 * jg) = make_float4(s[0], s[1], s[2], s[3]);
    *reinterpret_cast<float4*>(scratch + tg * D + M + 4 * jg) = make_float4(s[4], s[5], s[6], s[7]);
}
template <int D, int TG>
__device__ __forceinline__ void store_feature_sums(const float* __restrict__ scratch, float* __restrict__ out)
{
    if (threadIdx.x < D) {
        float acc = 0.f;
#pragma unroll 8
        for (int g = 0; g < TG; ++g) acc += scratch[g * D + threadIdx.x];
        out[threadIdx.x] = acc;
    }
}

// A D x D accumulator held as 8 x 8 blocks by D*D/64 threads (rows 8 fy + a, columns 4 cx + (D/2) b + ..), SUB = 64 * threads
// / D^2 copies of it (each summed over its share of every tile's rows) -> out, row-major.  d = 64: the copies are added in
// order through `scratch` (SUB * D * D floats).  Barriers: the caller's before, one inside.
template <int D, int THREADS>
__device__ __forceinline__ void store_square(float* __restrict__ out, float* __restrict__ scratch, const f32x2 (&acc)[8][4])
{
    constexpr int NS = D * D / 64, SUB = THREADS / NS;
    const int sub = threadIdx.x / NS, r = threadIdx.x % NS, fy = r / (D / 8), cx = r % (D / 8);
    float* dst = SUB == 1 ? out : scratch + sub * D * D;
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
            *reinterpret_cast<ulonglong2*>(dst + (8 * fy + a) * D + 4 * cx + (D / 2) * b) = make_ulonglong2(acc[a][2 * b], acc[a][2 * b + 1]);
    __syncthreads();
    if constexpr (SUB > 1) {
        for (int e = threadIdx.x; e < D * D / 4; e += THREADS) {
            float4 s = *reinterpret_cast<const float4*>(scratch + 4 * e);
#pragma unroll
            for (int k = 1; k < SUB; ++k) {
                const float4 t = *reinterpret_cast<const float4*>(scratch + k * D * D + 4 * e);
                s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
            }
            *reinterpret_cast<float4*>(out + 4 * e) = s;
        }
    }
}

constexpr int kSimtKWarps = 8;   // key side: 8 warps, two CTAs per SM (102 KB of shared memory each at d = 128)

// Shared-memory floats: W, then the K / phi tile and the V tile (or, at the end of a run's piece, the copies of S).
template <int D, int TM> constexpr size_t kside_simt_smem()
{
    constexpr int tiles = 2 * SimtTile<D, kSimtKWarps, TM>::TT * SimtShape<D>::PX;
    constexpr int copies = D == 64 ? 4 * D * D : 0;
    return sizeof(float) * (size_t)(D * SimtShape<D>::PW + (tiles > copies ? tiles : copies));
}

// CTA p works on its run of the T = G * Tn tiles.  The record of its piece of pair g goes to slot p + g * slot_step:
// slot_step = 1 in general (a run may touch several pairs); 0 when every run lies within one pair.
// partial: [slots][D*D + D] floats (S row-major [f][c], then z).
template <typename T, int D, int TM>
__global__ void __launch_bounds__(32 * kSimtKWarps, 2)
kside_simt(const T* __restrict__ k, const T* __restrict__ v, const float* __restrict__ Wk /*[H][D][M]*/,
           float* __restrict__ partial, int H, int n, int Tn, long long tiles, int slot_step, ActStrides st, int relu)
{
    using Sh = SimtShape<D>;
    using Ti = SimtTile<D, kSimtKWarps, TM>;
    constexpr int TG = Ti::TG, TT = Ti::TT, PX = Sh::PX, JG = Sh::JG, TH = Ti::kThreads;
    constexpr int NS = D * D / 64, SUB = TH / NS;
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) float smem[];
    float* W_s = smem;
    float* x_s = W_s + D * Sh::PW;
    float* v_s = x_s + TT * PX;

    const int tid = threadIdx.x, tg = tid / JG, jg = tid % JG;
    const int sub = tid / NS, fy = (tid % NS) / (D / 8), cx = (tid % NS) % (D / 8);
    const long long end = run_begin(blockIdx.x + 1, tiles, gridDim.x);
    long long tile = run_begin(blockIdx.x, tiles, gridDim.x);
    while (tile < end) {
        const int g = (int)(tile / Tn);
        const long long seg_end = min(end, (long long)(g + 1) * Tn);
        if (!relu) load_weights<D, TH>(Wk + (size_t)(g % H) * D * Sh::M, W_s);
        f32x2 acc[8][4];
        zero_acc(acc);
        float zacc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const T* kg = k + st.base(g, H);
        const T* vg = v + st.base(g, H);
        __syncthreads();   // W_s
        for (; tile < seg_end; ++tile) {
            const int t = (int)(tile - (long long)g * Tn) * TT, valid = min(TT, n - t);
            load_rows<T, D, TG, TM>(kg + (size_t)t * st.token, st.token, x_s, valid);
            load_rows<T, D, TG, TM>(vg + (size_t)t * st.token, st.token, v_s, valid);
            __syncwarp();
            float p[TM][8];
            feature_map_rows<D, TG, TM>(x_s + tg * PX, W_s, tg, jg, valid, relu, p);
            __syncwarp();   // the warp's x rows have been read
            store_phi_rows<D, TG, TM>(x_s + tg * PX, jg, p);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) zacc[j] += p[i][j];
            __syncthreads();
            rows_outer<8, 2>(x_s + 8 * fy, PX, v_s + 4 * cx, PX, D / 2, sub * (TT / SUB), (sub + 1) * (TT / SUB), acc);
            __syncthreads();   // phi and V consumed
        }
        float* out = partial + ((size_t)blockIdx.x + (size_t)g * slot_step) * Sh::E;
        park_feature_sums<D, TG>(W_s, tg, jg, zacc);
        store_square<D, TH>(out, x_s, acc);
        store_feature_sums<D, TG>(W_s, out + D * D);
        __syncthreads();   // W_s is written again
    }
}

// out[g][e] = sum over the CTAs p whose runs touch pair g, p ascending, of rec[p + g * slot_step][e].
// grid = (ceil(E/256), G); 64 threads cover 256 consecutive floats, four slices of the list each a contiguous part of it,
// and the slices are added in order.
static __global__ void __launch_bounds__(256)
combine_state(const float* __restrict__ rec, float* __restrict__ out, int E, int Tn, long long tiles, long long P, int slot_step)
{
    pdl_trigger();
    pdl_wait();
    __shared__ float4 part_s[4][64];
    const int lane = threadIdx.x & 63, slice = threadIdx.x >> 6;
    const int e = (blockIdx.x * 64 + lane) * 4, g = blockIdx.y;
    // CTAs that touch [g*Tn, (g+1)*Tn)
    long long p0 = (long long)g * Tn * P / tiles, p1 = ((long long)(g + 1) * Tn - 1) * P / tiles;
    while (run_begin(p0 + 1, tiles, P) <= (long long)g * Tn) ++p0;
    while (run_begin(p1 + 1, tiles, P) <= (long long)(g + 1) * Tn - 1) ++p1;
    const int cnt = (int)(p1 - p0) + 1, per = (cnt + 3) / 4;
    const int b = min(cnt, slice * per), eb = min(cnt, b + per);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < E) {
        const float* src = rec + ((size_t)p0 + (size_t)g * slot_step) * E + e;
#pragma unroll 8
        for (int i = b; i < eb; ++i) {
            const float4 x = *reinterpret_cast<const float4*>(src + (size_t)i * E);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
    }
    part_s[slice][lane] = s;
    __syncthreads();
    if (slice == 0 && e < E) {
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            const float4 x = part_s[q][lane];
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        *reinterpret_cast<float4*>(out + (size_t)g * E + e) = s;
    }
}

// Shared-memory floats: W, S, z, the q / phi rows of every warp.
template <int D, int NW, int TM> constexpr size_t qside_simt_smem()
{
    return sizeof(float) * (size_t)(D * SimtShape<D>::PW + D * D + D + SimtTile<D, NW, TM>::TT * SimtShape<D>::PX);
}

// CTA p works on its run of the T = G * Tn tiles; W, S, z of the pair stay in shared memory, and each warp goes through its
// rows of the tiles by itself (no barrier but at a change of pair).
// state: [G][D*D + D] floats (S then z).
// relu != 0: the ReLU kernel function instead of Eq. 6 (Wq is then not read).
// mix != nullptr: Eq. 8, out = mix_r * mix + (1 - mix_r) * (Eq. 5), mix = output of the softmax-attention branch
// (laid out like q, may be the same buffer as out), mix_r already clipped into [0, 1].
template <typename T, int D, int NW, int TM>
__global__ void __launch_bounds__(32 * NW, NW <= 8 ? 2 : 1)
qside_simt(const T* __restrict__ q, const float* __restrict__ Wq, const float* __restrict__ state,
           T* out, int H, int n, int Tn, long long tiles, const T* mix, float mix_r, ActStrides st, int relu)
{
    using Sh = SimtShape<D>;
    using Ti = SimtTile<D, NW, TM>;
    constexpr int TG = Ti::TG, TT = Ti::TT, PX = Sh::PX, JG = Sh::JG, TH = Ti::kThreads, M = Sh::M;
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) float smem[];
    float* W_s = smem;
    float* S_s = W_s + D * Sh::PW;
    float* z_s = S_s + D * D;
    float* x_s = z_s + D;

    const int tid = threadIdx.x, tg = tid / JG, jg = tid % JG;
    const long long end = run_begin(blockIdx.x + 1, tiles, gridDim.x);
    long long tile = run_begin(blockIdx.x, tiles, gridDim.x);
    float* x = x_s + tg * PX;
    while (tile < end) {
        const int g = (int)(tile / Tn);
        const long long seg_end = min(end, (long long)(g + 1) * Tn);
        __syncthreads();   // the pair before has been consumed
        if (!relu) load_weights<D, TH>(Wq + (size_t)(g % H) * D * M, W_s);
        const float* Sg = state + (size_t)g * Sh::E;
#pragma unroll 4
        for (int e = tid; e < Sh::E / 4; e += TH) reinterpret_cast<float4*>(S_s)[e] = reinterpret_cast<const float4*>(Sg)[e];   // z_s follows S_s
        __syncthreads();
        float zr[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            zr[j] = z_s[4 * jg + j];
            zr[4 + j] = z_s[M + 4 * jg + j];
        }
        const T* qg = q + st.base(g, H);
        const T* mg = mix ? mix + st.base(g, H) : nullptr;
        T* og = out + st.base(g, H);
        for (; tile < seg_end; ++tile) {
            const int t = (int)(tile - (long long)g * Tn) * TT, valid = min(TT, n - t);
            load_rows<T, D, TG, TM>(qg + (size_t)t * st.token, st.token, x_s, valid);
            __syncwarp();
            float p[TM][8], inv[TM];
            // tail rows see zero-filled q: their phi is finite (Eq. 6) or zero (ReLU); their outputs are never stored
            feature_map_rows<D, TG, TM>(x, W_s, tg, jg, TT, relu, p);
            __syncwarp();
            store_phi_rows<D, TG, TM>(x, jg, p);
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                float den = 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) den = fmaf(p[i][j], zr[j], den);
                inv[i] = 1.f / group_sum<JG>(den);
            }
            __syncwarp();
            f32x2 num[TM][4];
            zero_acc(num);
            rows_times_matrix<D, TM, 2>(x, TG * PX, S_s + 4 * jg, D, D / 2, num);
            __syncwarp();   // phi consumed: the next tile's rows may come in
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const int row = tg + TG * i;
                if (row >= valid) continue;
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const size_t e = (size_t)(t + row) * st.token + (D / 2) * b + 4 * jg;
                    float o[4];
                    unpack2(num[i][2 * b], o[0], o[1]);
                    unpack2(num[i][2 * b + 1], o[2], o[3]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) o[j] *= inv[i];
                    if (mg) {
                        const float4 m = load4_f32(mg + e);
#pragma unroll
                        for (int j = 0; j < 4; ++j) o[j] = fmaf(o[j], 1.f - mix_r, mix_r * part(m, j));
                    }
                    store_out4(og + e, o[0], o[1], o[2], o[3]);
                }
            }
        }
    }
}

// ---- host side: how a problem is dealt to CTAs, and the launches (shared by the context's entry points and the
// allocation-free one) ------------------------------------------------------------------------------------------------

constexpr int kSimtCtas = 296;   // key side: two CTAs per SM on 148 SMs
constexpr int kSimtQWarps = 16;  // query side: one CTA of 16 warps per SM (S, W and 128 rows: 167 KB at d = 128)

struct SimtRuns {
    int Tn = 0;             // tiles per (b,h) pair
    long long tiles = 0, P = 0;
    int slot_step = 1;
    bool small = false;     // TM = 1: a quarter of the tokens per tile
};

// The small tiles are taken when the large ones would leave places idle: a tile is then a thread's shortest serial chain
// (B=1 H=2 n=1024 d=64: 16 large tiles or 64 small ones for 296 places); with every place busy the large tile's ratio of
// FMAs to shared-memory loads wins.
template <int D> SimtRuns kside_runs(long long G, int n, int splits_per_pair)
{
    SimtRuns r;
    constexpr int big = SimtTile<D, kSimtKWarps, 4>::TT, little = SimtTile<D, kSimtKWarps, 1>::TT;
    r.Tn = (n + big - 1) / big;
    r.small = splits_per_pair > 0 ? r.Tn < splits_per_pair : G * r.Tn < kSimtCtas;
    if (r.small) r.Tn = (n + little - 1) / little;
    r.tiles = G * r.Tn;
    if (splits_per_pair > 0) {   // the same number of CTAs for every pair: no run crosses into another pair
        r.P = G * (splits_per_pair < r.Tn ? splits_per_pair : r.Tn);
        r.slot_step = 0;
    } else {
        r.P = r.tiles < kSimtCtas ? r.tiles : kSimtCtas;
    }
    return r;
}
template <int D> SimtRuns qside_runs(long long G, int n)
{
    SimtRuns r;
    constexpr int big = SimtTile<D, kSimtQWarps, 4>::TT, little = SimtTile<D, 8, 1>::TT;
    r.Tn = (n + big - 1) / big;
    r.small = G * r.Tn < kSimtCtas / 2;
    if (r.small) r.Tn = (n + little - 1) / little;
    r.tiles = G * r.Tn;
    const long long places = r.small ? kSimtCtas : kSimtCtas / 2;
    r.P = r.tiles < places ? r.tiles : places;
    return r;
}

// Once per device: the shared-memory limits of the kernels below.
template <typename T, int D> cudaError_t simt_forward_attributes()
{
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(kside_simt<T, D, 4>, a, (int)kside_simt_smem<D, 4>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kside_simt<T, D, 1>, a, (int)kside_simt_smem<D, 1>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(qside_simt<T, D, kSimtQWarps, 4>, a, (int)qside_simt_smem<D, kSimtQWarps, 4>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(qside_simt<T, D, 8, 1>, a, (int)qside_simt_smem<D, 8, 1>());
    return e;
}

template <typename T, int D>
cudaError_t launch_kside_simt(const SimtRuns& r, const T* k, const T* v, const float* Wk, float* partial, int H, int n, ActStrides st, int relu,
                              cudaStream_t stream)
{
    return launch_chained(r.small ? kside_simt<T, D, 1> : kside_simt<T, D, 4>, (unsigned)r.P, 32 * kSimtKWarps,
                          r.small ? kside_simt_smem<D, 1>() : kside_simt_smem<D, 4>(), stream, k, v, Wk, partial, H, n, r.Tn, r.tiles, r.slot_step,
                          st, relu);
}
template <int D> cudaError_t launch_combine_state(const SimtRuns& r, const float* partial, float* state, long long G, cudaStream_t stream)
{
    constexpr int E = SimtShape<D>::E;
    return launch_chained(combine_state, dim3((E + 255) / 256, (unsigned)G), 256, 0, stream, partial, state, E, r.Tn, r.tiles, r.P, r.slot_step);
}
template <typename T, int D>
cudaError_t launch_qside_simt(const SimtRuns& r, const T* q, const float* Wq, const float* state, T* out, int H, int n, const T* mix, float mix_r,
                              ActStrides st, int relu, cudaStream_t stream)
{
    return launch_chained(r.small ? qside_simt<T, D, 8, 1> : qside_simt<T, D, kSimtQWarps, 4>, (unsigned)r.P, r.small ? 256 : 32 * kSimtQWarps,
                          r.small ? qside_simt_smem<D, 8, 1>() : qside_simt_smem<D, kSimtQWarps, 4>(), stream, q, Wq, state, out, H, n, r.Tn,
                          r.tiles, mix, mix_r, st, relu);
}

// Feature-map weights: any supported storage type -> fp32 [H][D][M]; src is [H][D][M] or, when per_head == 0, a single
// [D][M] replicated to every head.  blockIdx.y = 0: W_q, 1: W_k.
template <typename T>
__global__ void convert_weights(const T* __restrict__ src_q, const T* __restrict__ src_k, float* __restrict__ dst_q, float* __restrict__ dst_k, int H,
                                int DM, int per_head)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)H * DM) return;
    (blockIdx.y ? dst_k : dst_q)[i] = to_f32((blockIdx.y ? src_k : src_q)[per_head ? i : i % DM]);
}

}  // namespace linattn
