// CUDA-core (fp32 FMA) kernels for the gradients of linear attention with the Hedgehog feature map:
// what the training objective (Eq. 14) back-propagates through each layer that uses Eq. 5 with the phi of Eq. 6.
//
// With dO the gradient that arrives at the layer's output, S = sum_j phi(k_j)^T v_j, z = sum_j phi(k_j),
// den_i = phi(q_i) . z and o_i = phi(q_i) S / den_i, the chain rule gives
//     dnum_i = dO_i / den_i                  dden_i = -(dO_i . o_i) / den_i
//     dphi(q_i) = S dnum_i + dden_i z        dS = sum_i phi(q_i)^T dnum_i       dz = sum_i dden_i phi(q_i)
//     dphi(k_j) = dS v_j + dz                dv_j = dS^T phi(k_j)
// and through phi (p+ = softmax(u), p- = softmax(-u), u = x W)
//     du = p+ (.) (dphi+ - p+ . dphi+) - p- (.) (dphi- - p- . dphi-)       dx = du W^T       dW += x^T du.
//
// Launches of one backward (S and z come from the forward's key-side kernels):
//   qside_bwd     : per run of token tiles: dq, and per (b,h) pair the run touches the sums of dS, dz, dW_q
//   combine_state : fixed-order sum of the dS, dz records (shared with the forward)
//   kside_bwd     : dk, dv and the run's sums of dW_k
//   combine_wgrad : fixed-order sums of the weight-gradient records over runs, batch and (shared map) heads
// All arithmetic is fp32; every sum has a fixed order, so the gradients are bit-reproducible.
//
// Bound, like the forward's, by the fp32 FMA rate (17 d^2 flops per token for both sides and the state), so the products are
// the forward's register-tiled loops of packed FMAs.  A token's rows (x, dO or V, phi, du) belong to the JG lanes that own
// it; only the sums over tokens (dS, dW), which every thread holds a block of in registers for a whole run (104 registers
// with dz), meet at a CTA barrier, two per tile.  One CTA of 256 threads per SM: W, S or dS and the tiles take 222 KB at d = 128.
// Products over a row of W or of the state (dO S^T, V dS^T, du W^T) take both operands 16 bytes along the summed index,
// a pair of partial sums per output; the rows 4 jg + j of one feature quad are kept JG rows apart (state_row), so that the lanes
// of a token read consecutive rows, 4 banks apart.
// The identity dO . o = (dO S^T) . phi / den replaces the product phi S of the forward (2 d^2 flops per token): dO S^T is
// needed anyway.
// Measured at B=1 H=12 n=14040 d=128 (bf16 activations, fp32 weights): forward + backward 1.28 ms (4.94 ms with 32-token
// chunks, eight threads a token and scalar FMAs); B=1 H=30 n=17776 d=64: 1.21 ms (4.05 ms).
#pragma once
#include "simt_kernels.cuh"

namespace linattn {

constexpr int kSimtBwdWarps = 8;
constexpr int kSimtBwdCtas = 148;   // one CTA per SM

// Where feature or column x of W or the state is kept in shared memory: quads (4 jg .. 4 jg + 3) are spread JG rows apart.
template <int D> __device__ __forceinline__ constexpr int state_row(int x)
{
    constexpr int M = D / 2, JG = M / 4;
    return (x / M) * M + (x % 4) * JG + (x % M) / 4;
}

// acc[i][4 h + j] += a_i . row(h M + 4 jg + j)  over K: a pair of sums (even, odd index) per output.
// b: base of the matrix + jg * pb.
template <int D, int K, int TM>
__device__ __forceinline__ void rows_dot_rows(const float* __restrict__ a, int a_step, const float* __restrict__ b, int pb, f32x2 (&acc)[TM][8])
{
    constexpr int M = D / 2, JG = M / 4;
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        ulonglong2 av[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const ulonglong2*>(a + i * a_step + k);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const ulonglong2 bv = *reinterpret_cast<const ulonglong2*>(b + ((r / 4) * M + (r % 4) * JG) * pb + k);
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                acc[i][r] = fma2(av[i].x, bv.x, acc[i][r]);
                acc[i][r] = fma2(av[i].y, bv.y, acc[i][r]);
            }
        }
    }
}
template <int TM> __device__ __forceinline__ void pair_sums(const f32x2 (&acc)[TM][8], float (&out)[TM][8])
{
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            float lo, hi;
            unpack2(acc[i][r], lo, hi);
            out[i][r] = lo + hi;
        }
}

// A D x D matrix (row-major in global memory) -> shared rows state_row(f), pitch PX; W likewise with pitch PW.
template <int D, int COLS, int PITCH, int THREADS>
__device__ __forceinline__ void load_spread(const float* __restrict__ src, float* __restrict__ dst)
{
#pragma unroll 4
    for (int e = threadIdx.x; e < D * COLS / 4; e += THREADS)
        *reinterpret_cast<float4*>(dst + state_row<D>(e / (COLS / 4)) * PITCH + (e % (COLS / 4)) * 4) = *reinterpret_cast<const float4*>(src + 4 * e);
}

// Softmax backward of Eq. 6 for this thread's tokens: du[i][j], logit 4 jg + j, from phi and dphi (layout of p).
template <int D, int TM>
__device__ __forceinline__ void du_rows(const float (&p)[TM][8], const float (&dphi)[TM][8], float (&du)[TM][4])
{
    constexpr int JG = SimtShape<D>::JG;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        float dp = 0.f, dn = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            dp = fmaf(p[i][j], dphi[i][j], dp);
            dn = fmaf(p[i][4 + j], dphi[i][4 + j], dn);
        }
        dp = group_sum<JG>(dp);
        dn = group_sum<JG>(dn);
#pragma unroll
        for (int j = 0; j < 4; ++j) du[i][j] = p[i][j] * (dphi[i][j] - dp) - p[i][4 + j] * (dphi[i][4 + j] - dn);
    }
}

// This thread's TM x 8 values (columns 4 jg + j and M + 4 jg + j) to the activations' rows of the tile.
template <typename T, int D, int TG, int TM>
__device__ __forceinline__ void store_rows(T* __restrict__ dst, long long row_stride, int tg, int jg, int valid, const float (&x)[TM][8])
{
    constexpr int M = D / 2;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int row = tg + TG * i;
        if (row >= valid) continue;
        T* o = dst + (size_t)row * row_stride + 4 * jg;
        store_out4(o, x[i][0], x[i][1], x[i][2], x[i][3]);
        store_out4(o + M, x[i][4], x[i][5], x[i][6], x[i][7]);
    }
}

// dx = du W^T of this thread's tokens; du_s: the token group's first du row, W_s in spread rows.
template <typename T, int D, int TG, int TM>
__device__ __forceinline__ void dx_rows(const float* __restrict__ du_s, const float* __restrict__ W_s, T* __restrict__ dst, long long row_stride,
                                        int tg, int jg, int valid)
{
    constexpr int M = D / 2, PW = SimtShape<D>::PW;
    f32x2 acc[TM][8];
    zero_acc(acc);
    rows_dot_rows<D, M, TM>(du_s, TG * PW, W_s + jg * PW, PW, acc);
    float dx[TM][8];
    pair_sums(acc, dx);
    store_rows<T, D, TG, TM>(dst, row_stride, tg, jg, valid, dx);
}

// The CTA's dW [c][j] held as 8 x 4 blocks (c = 8 cy + a, j = 4 jx + ..) by D*D/64 threads, SUB copies (see store_square).
template <int D, int THREADS>
__device__ __forceinline__ void store_wgrad(float* __restrict__ out, float* __restrict__ scratch, const f32x2 (&acc)[8][2])
{
    constexpr int M = D / 2, NS = D * D / 64, SUB = THREADS / NS;
    const int sub = threadIdx.x / NS, r = threadIdx.x % NS, cy = r / (M / 4), jx = r % (M / 4);
    float* dst = SUB == 1 ? out : scratch + sub * D * M;
#pragma unroll
    for (int a = 0; a < 8; ++a) *reinterpret_cast<ulonglong2*>(dst + (8 * cy + a) * M + 4 * jx) = make_ulonglong2(acc[a][0], acc[a][1]);
    __syncthreads();
    if constexpr (SUB > 1) {
        for (int e = threadIdx.x; e < D * M / 4; e += THREADS) {
            float4 s = *reinterpret_cast<const float4*>(scratch + 4 * e);
#pragma unroll
            for (int k = 1; k < SUB; ++k) {
                const float4 t = *reinterpret_cast<const float4*>(scratch + k * D * M + 4 * e);
                s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
            }
            *reinterpret_cast<float4*>(out + 4 * e) = s;
        }
    }
}

// Shared-memory floats: W, the state and its vector, then the token tiles (x, dO or V, phi on the query side, du) or, at the
// end of a run's piece, the copies of the dS (query side) or dW accumulators.
template <int D, int TM, bool QSIDE> constexpr size_t simt_bwd_smem()
{
    constexpr int TT = SimtTile<D, kSimtBwdWarps, TM>::TT;
    constexpr int tiles = TT * ((QSIDE ? 3 : 2) * SimtShape<D>::PX + SimtShape<D>::PW);
    constexpr int copies = D == 64 ? (QSIDE ? 4 * D * D : 2 * D * D) : 0;
    return sizeof(float) * (size_t)(D * SimtShape<D>::PW + D * SimtShape<D>::PX + D + (tiles > copies ? tiles : copies));
}

// CTA p works on its run of the T = G * Tn tiles; the records of its piece of pair g go to slot p + g.
//   relu      : 1 = the ReLU kernel function instead of Eq. 6 (no weights: Wq is NULL, part_w is not written)
//   mix_a, lin_scale, part_dr : Eq. 8.  The gradient that reaches the linear branch is lin_scale * dout (lin_scale = 1 - r^);
//               when mix_a (the softmax branch's output, laid out like q) is given, part_dr [gridDim.x] receives the
//               CTA's sum of dout . (a - o), the terms of dL/dr
//   state     : [G][D*D + D]  S row-major [f][c], then z   (from the forward's key side)
//   dq        : same layout and type as q
//   part_state: [slots][D*D + D]  sums of dS ([f][c]) and dz
//   part_w    : [slots][D*M]      sums of dW_q
template <typename T, int D, int TM>
__global__ void __launch_bounds__(32 * kSimtBwdWarps)
qside_bwd(const T* __restrict__ q, const T* __restrict__ dout, const float* __restrict__ Wq, const float* __restrict__ state,
          T* __restrict__ dq, float* __restrict__ part_state, float* __restrict__ part_w, int H, int n, int Tn, long long tiles, ActStrides st,
          int relu, const T* __restrict__ mix_a, float lin_scale, float* __restrict__ part_dr)
{
    using Sh = SimtShape<D>;
    using Ti = SimtTile<D, kSimtBwdWarps, TM>;
    constexpr int M = Sh::M, PX = Sh::PX, PW = Sh::PW, JG = Sh::JG, TG = Ti::TG, TT = Ti::TT, TH = Ti::kThreads;
    constexpr int NS = D * D / 64, SUB = TH / NS;
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) float smem[];
    float* W_s = smem;
    float* S_s = W_s + D * PW;
    float* z_s = S_s + D * PX;
    float* x_s = z_s + D;
    float* g_s = x_s + TT * PX;
    float* phi_s = g_s + TT * PX;
    float* du_s = phi_s + TT * PX;

    const int tid = threadIdx.x, tg = tid / JG, jg = tid % JG;
    const int sub = tid / NS, rs = tid % NS, fy = rs / (D / 8), cx = rs % (D / 8), cy = rs / JG, jx = rs % JG;
    const int r0 = sub * (TT / SUB), r1 = r0 + TT / SUB;
    float dr_acc = 0.f;   // this thread's share of sum dout . (a - o)
    const long long end = run_begin(blockIdx.x + 1, tiles, gridDim.x);
    long long tile = run_begin(blockIdx.x, tiles, gridDim.x);
    while (tile < end) {
        const int g = (int)(tile / Tn);
        const long long seg_end = min(end, (long long)(g + 1) * Tn);
        const float* Sg = state + (size_t)g * Sh::E;
        if (!relu) load_spread<D, M, PW, TH>(Wq + (size_t)(g % H) * D * M, W_s);
        load_spread<D, D, PX, TH>(Sg, S_s);
        if (tid < D) z_s[tid] = Sg[D * D + tid];
        const T* qg = q + st.base(g, H);
        const T* gg = dout + st.base(g, H);
        const T* ag = mix_a ? mix_a + st.base(g, H) : nullptr;
        T* dqg = dq + st.base(g, H);
        f32x2 dS[8][4], dw[8][2];
        zero_acc(dS);
        zero_acc(dw);
        float dz[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        __syncthreads();
        for (; tile < seg_end; ++tile) {
            const int t = (int)(tile - (long long)g * Tn) * TT, valid = min(TT, n - t);
            load_rows<T, D, TG, TM>(qg + (size_t)t * st.token, st.token, x_s, valid);
            load_rows<T, D, TG, TM>(gg + (size_t)t * st.token, st.token, g_s, valid);
            __syncwarp();
            float p[TM][8], dphi[TM][8];
            feature_map_rows<D, TG, TM, true>(x_s + tg * PX, W_s, tg, jg, valid, relu, p);   // rows past `valid` get phi = 0
            {
                f32x2 acc[TM][8];
                zero_acc(acc);
                rows_dot_rows<D, D, TM>(g_s + tg * PX, TG * PX, S_s + jg * PX, PX, acc);
                pair_sums(acc, dphi);   // dO S^T
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const int row = tg + TG * i;
                float den = 0.f, go = 0.f, zr[8];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 zv = *reinterpret_cast<const float4*>(z_s + h * M + 4 * jg);
#pragma unroll
                    for (int j = 0; j < 4; ++j) zr[4 * h + j] = part(zv, j);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    den = fmaf(p[i][j], zr[j], den);
                    go = fmaf(p[i][j], dphi[i][j], go);
                }
                den = group_sum<JG>(den);
                go = group_sum<JG>(go);
                const float inv = row < valid ? 1.f / den : 0.f;
                go = row < valid ? go * inv : 0.f;   // dO . o
                const float sc = lin_scale * inv;    // the linear branch's incoming gradient is lin_scale * dO
                if (ag && row < valid) {             // Eq. 8: dO . (a - o), each thread its own columns of dO . a
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 av = load4_f32(ag + (size_t)(t + row) * st.token + h * M + 4 * jg);
                        const float4 gv = *reinterpret_cast<const float4*>(g_s + row * PX + h * M + 4 * jg);
#pragma unroll
                        for (int j = 0; j < 4; ++j) dr_acc = fmaf(part(gv, j), part(av, j), dr_acc);
                    }
                    if (jg == 0) dr_acc -= go;
                }
                float f[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    dphi[i][j] = sc * fmaf(-go, zr[j], dphi[i][j]);   // S dnum + dden z
                    f[j] = p[i][j] * sc;                              // phi / den: dS = sum (phi / den)^T dO
                    dz[j] = fmaf(f[j], -go, dz[j]);
                }
                *reinterpret_cast<float4*>(phi_s + row * PX + 4 * jg) = make_float4(f[0], f[1], f[2], f[3]);
                *reinterpret_cast<float4*>(phi_s + row * PX + M + 4 * jg) = make_float4(f[4], f[5], f[6], f[7]);
            }
            if (relu) {   // d phi / d x = [x > 0], and phi > 0 exactly there
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) dphi[i][j] = p[i][j] > 0.f ? dphi[i][j] : 0.f;
                store_rows<T, D, TG, TM>(dqg + (size_t)t * st.token, st.token, tg, jg, valid, dphi);
            } else {
                float du[TM][4];
                du_rows<D, TM>(p, dphi, du);
#pragma unroll
                for (int i = 0; i < TM; ++i) *reinterpret_cast<float4*>(du_s + (tg + TG * i) * PW + 4 * jg) = make_float4(du[i][0], du[i][1], du[i][2], du[i][3]);
                __syncwarp();
                dx_rows<T, D, TG, TM>(du_s + tg * PW, W_s, dqg + (size_t)t * st.token, st.token, tg, jg, valid);
            }
            __syncthreads();
            rows_outer<8, 2>(phi_s + 8 * fy, PX, g_s + 4 * cx, PX, D / 2, r0, r1, dS);
            if (!relu) rows_outer<8, 1>(x_s + 8 * cy, PX, du_s + 4 * jx, PW, 0, r0, r1, dw);
            __syncthreads();
        }
        const size_t slot = (size_t)blockIdx.x + g;
        float* ps = part_state + slot * Sh::E;
        park_feature_sums<D, TG>(W_s, tg, jg, dz);
        store_square<D, TH>(ps, x_s, dS);
        store_feature_sums<D, TG>(W_s, ps + D * D);
        __syncthreads();
        if (!relu) {
            store_wgrad<D, TH>(part_w + slot * (D * M), x_s, dw);
            __syncthreads();
        }
    }
    if (part_dr) {   // fixed order: lanes by a butterfly, then the warps in order
        const float w = group_sum<32>(dr_acc);
        if ((tid & 31) == 0) x_s[tid >> 5] = w;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
            for (int i = 0; i < kSimtBwdWarps; ++i) s += x_s[i];
            part_dr[blockIdx.x] = s;
        }
    }
}

//   dstate: [G][D*D + D]  dS row-major [f][c], then dz
//   dk, dv: same layout and type as k, v
//   part_w: [slots][D*M]  sums of dW_k, slot p + g
template <typename T, int D, int TM>
__global__ void __launch_bounds__(32 * kSimtBwdWarps)
kside_bwd(const T* __restrict__ k, const T* __restrict__ v, const float* __restrict__ Wk, const float* __restrict__ dstate,
          T* __restrict__ dk, T* __restrict__ dv, float* __restrict__ part_w, int H, int n, int Tn, long long tiles, ActStrides st, int relu)
{
    using Sh = SimtShape<D>;
    using Ti = SimtTile<D, kSimtBwdWarps, TM>;
    constexpr int M = Sh::M, PX = Sh::PX, PW = Sh::PW, JG = Sh::JG, TG = Ti::TG, TT = Ti::TT, TH = Ti::kThreads;
    constexpr int NS = D * D / 64, SUB = TH / NS;
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) float smem[];
    float* W_s = smem;
    float* S_s = W_s + D * PW;
    float* z_s = S_s + D * PX;
    float* x_s = z_s + D;
    float* v_s = x_s + TT * PX;      // V, then phi(k) over it
    float* du_s = v_s + TT * PX;

    const int tid = threadIdx.x, tg = tid / JG, jg = tid % JG;
    const int sub = tid / NS, rs = tid % NS, cy = rs / JG, jx = rs % JG;
    const int r0 = sub * (TT / SUB), r1 = r0 + TT / SUB;
    const long long end = run_begin(blockIdx.x + 1, tiles, gridDim.x);
    long long tile = run_begin(blockIdx.x, tiles, gridDim.x);
    while (tile < end) {
        const int g = (int)(tile / Tn);
        const long long seg_end = min(end, (long long)(g + 1) * Tn);
        const float* Sg = dstate + (size_t)g * Sh::E;
        if (!relu) load_spread<D, M, PW, TH>(Wk + (size_t)(g % H) * D * M, W_s);
        load_spread<D, D, PX, TH>(Sg, S_s);
        if (tid < D) z_s[tid] = Sg[D * D + tid];
        const T* kg = k + st.base(g, H);
        const T* vg = v + st.base(g, H);
        T* dkg = dk + st.base(g, H);
        T* dvg = dv + st.base(g, H);
        f32x2 dw[8][2];
        zero_acc(dw);
        __syncthreads();
        for (; tile < seg_end; ++tile) {
            const int t = (int)(tile - (long long)g * Tn) * TT, valid = min(TT, n - t);
            load_rows<T, D, TG, TM>(kg + (size_t)t * st.token, st.token, x_s, valid);
            load_rows<T, D, TG, TM>(vg + (size_t)t * st.token, st.token, v_s, valid);
            __syncwarp();
            float p[TM][8], dphi[TM][8];
            feature_map_rows<D, TG, TM, true>(x_s + tg * PX, W_s, tg, jg, valid, relu, p);
            {
                f32x2 acc[TM][8];
                zero_acc(acc);
                rows_dot_rows<D, D, TM>(v_s + tg * PX, TG * PX, S_s + jg * PX, PX, acc);
                pair_sums(acc, dphi);
            }
            __syncwarp();   // the warp's V rows have been read
            store_phi_rows<D, TG, TM>(v_s + tg * PX, jg, p);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 zv = *reinterpret_cast<const float4*>(z_s + h * M + 4 * jg);
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) dphi[i][4 * h + j] += part(zv, j);
            }
            if (relu) {
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) dphi[i][j] = p[i][j] > 0.f ? dphi[i][j] : 0.f;
                store_rows<T, D, TG, TM>(dkg + (size_t)t * st.token, st.token, tg, jg, valid, dphi);
            } else {
                float du[TM][4];
                du_rows<D, TM>(p, dphi, du);
#pragma unroll
                for (int i = 0; i < TM; ++i) *reinterpret_cast<float4*>(du_s + (tg + TG * i) * PW + 4 * jg) = make_float4(du[i][0], du[i][1], du[i][2], du[i][3]);
            }
            __syncwarp();
            {
                f32x2 acc[TM][4];
                zero_acc(acc);
                rows_times_matrix<D, TM, 2, true>(v_s + tg * PX, TG * PX, S_s + 4 * jg, PX, D / 2, acc);
                float o[TM][8];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int r = 0; r < 4; ++r) unpack2(acc[i][r], o[i][2 * r], o[i][2 * r + 1]);
                store_rows<T, D, TG, TM>(dvg + (size_t)t * st.token, st.token, tg, jg, valid, o);
            }
            if (relu) {
                __syncwarp();   // phi consumed: the next tile's rows may come in
            } else {
                dx_rows<T, D, TG, TM>(du_s + tg * PW, W_s, dkg + (size_t)t * st.token, st.token, tg, jg, valid);
                __syncthreads();
                rows_outer<8, 1>(x_s + 8 * cy, PX, du_s + 4 * jx, PW, 0, r0, r1, dw);
                __syncthreads();
            }
        }
        if (!relu) store_wgrad<D, TH>(part_w + ((size_t)blockIdx.x + g) * (D * M), x_s, dw);
        __syncthreads();
    }
}

// dW[w][e] = sum over the pairs g that use weight matrix w (per_head: g % H == w; shared: all g), g ascending, and over the
// runs that touch g, ascending; eight slices of that list are summed side by side and added in order.
// grid = (DM / 256, per_head ? H : 1), 512 threads.
static __global__ void __launch_bounds__(512)
combine_wgrad(const float* __restrict__ rec, float* __restrict__ dW, int G, int H, int DM, int per_head, int Tn, long long tiles, long long P)
{
    pdl_trigger();
    pdl_wait();
    __shared__ float4 part_s[8][64];
    const int lane = threadIdx.x & 63, slice = threadIdx.x >> 6;
    const int e = (blockIdx.x * 64 + lane) * 4, w = blockIdx.y, step = per_head ? H : 1;
    const int pairs = per_head ? (G - w + H - 1) / H : G;
    // many pairs: every slice takes whole pairs; few: every slice takes its part of each pair's list
    const bool whole = pairs >= 8;
    const int per_slice = (pairs + 7) / 8;
    const int i0 = whole ? min(pairs, slice * per_slice) : 0, i1 = whole ? min(pairs, i0 + per_slice) : pairs;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = i0; i < i1; ++i) {
        const long long g = w + (long long)i * step;
        long long p0 = g * Tn * P / tiles, p1 = ((g + 1) * Tn - 1) * P / tiles;
        while (run_begin(p0 + 1, tiles, P) <= g * Tn) ++p0;
        while (run_begin(p1 + 1, tiles, P) <= (g + 1) * Tn - 1) ++p1;
        const int cnt = (int)(p1 - p0) + 1, per = whole ? cnt : (cnt + 7) / 8;
        const int b = whole ? 0 : min(cnt, slice * per), eb = min(cnt, b + per);
        const float* src = rec + (size_t)(p0 + g) * DM + e;
#pragma unroll 8
        for (int r = b; r < eb; ++r) {
            const float4 x = *reinterpret_cast<const float4*>(src + (size_t)r * DM);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
    }
    part_s[slice][lane] = s;
    __syncthreads();
    if (slice == 0) {
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            const float4 x = part_s[q][lane];
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        *reinterpret_cast<float4*>(dW + (size_t)w * DM + e) = s;
    }
}

// Eq. 8: dL/dr = sum of the partial sums of dout . (a - o), lane by lane and then over the lanes, if r lies in [0, 1] (the
// clip passes the gradient on the closed interval), else 0.  One warp.
static __global__ void __launch_bounds__(32) combine_dr(const float* __restrict__ part_dr, int count, int in_range, float* __restrict__ dr)
{
    pdl_trigger();
    pdl_wait();
    float acc = 0.f;
    for (int i = threadIdx.x; i < count; i += 32) acc += part_dr[i];
    acc = group_sum<32>(acc);
    if (threadIdx.x == 0) *dr = in_range ? acc : 0.f;
}

// The deal of the two gradient kernels (see kside_runs): small tiles while the large ones would leave SMs idle.
template <int D> SimtRuns bwd_runs(long long G, int n)
{
    SimtRuns r;
    constexpr int big = SimtTile<D, kSimtBwdWarps, 4>::TT, little = SimtTile<D, kSimtBwdWarps, 1>::TT;
    r.Tn = (n + big - 1) / big;
    r.small = G * r.Tn < kSimtBwdCtas;
    if (r.small) r.Tn = (n + little - 1) / little;
    r.tiles = G * r.Tn;
    r.P = r.tiles < kSimtBwdCtas ? r.tiles : kSimtBwdCtas;
    return r;
}

template <typename T, int D> cudaError_t simt_backward_attributes()
{
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(qside_bwd<T, D, 4>, a, (int)simt_bwd_smem<D, 4, true>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(qside_bwd<T, D, 1>, a, (int)simt_bwd_smem<D, 1, true>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kside_bwd<T, D, 4>, a, (int)simt_bwd_smem<D, 4, false>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kside_bwd<T, D, 1>, a, (int)simt_bwd_smem<D, 1, false>());
    return e;
}

// Eq. 8: the gradient that reaches the softmax branch, d_a = r^ * dout, element by element (any layout: `count` elements).
template <typename T>
static __global__ void __launch_bounds__(256) scale_copy(const T* __restrict__ src, T* __restrict__ dst, size_t count, float f)
{
    pdl_trigger();
    pdl_wait();
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < count; i += (size_t)gridDim.x * 256) store_out(&dst[i], f * to_f32(src[i]));
}

}  // namespace linattn
