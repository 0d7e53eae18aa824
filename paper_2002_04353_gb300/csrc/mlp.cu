// mlp.cu -- the learned departure-element proposal (alelb_mlp_*,
// alelb_samples, alelb_solver_set_mlp in include/alelb.h).
//
//   k_samples      training data from the solver itself: for every query
//                  (node, direction) its features and the slot of the exact
//                  element (FP64 departure point, exact walk) in the node's
//                  ring, with the barycentric coordinates there
//   k_mlp_fwd_bwd  forward and backward pass over tiles of 32 samples on the
//                  CUDA cores (FP16-rounded weights, FP32 arithmetic), each
//                  block's gradient to a row of its own
//   k_mlp_reduce   sum of those rows; Adam update of the FP32 master weights,
//                  FP16 copies
//   k_propose      inference for the work list of the exact path: 16 queries
//                  per warp through the three layers with FP16 tensor-core
//                  MMA (mma.sync m16n8k16, FP32 accumulation)
//   k_mlp_predict  the same inference on given features (tests)
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "internal.h"
#include "mlp.cuh"

using namespace alelb;

namespace {

constexpr int TS = 32;        // samples per training tile
constexpr int TRAIN_THREADS = 128;
constexpr int PRED_WARPS = 4; // warps per inference block

// ---------------------------------------------------------------------------
// training data
// ---------------------------------------------------------------------------
__global__ void k_samples(MeshDev M, MapStatic MS, MapScalars sc, MapScalarsF sf, int flags,
                          float *feat, int16_t *slot, float *bary, uint8_t *nring, int *err)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = M.N;
    if (a >= N) return;
    const double2 Xa = M.X[a];
    const FastMap F = fast_map(MS, sf, a, M.Xf[a]);
    double xX, xY, yX, yY, Vx, Vy, a11, a12, a21, a22, wx, wy;
    map_node(MS, sc, a, Xa.x, Xa.y, xX, xY, yX, yY, Vx, Vy);
    metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
    const int literal = (flags & FLAG_LITERAL_VG) != 0;
    mesh_velocity_term(a11, a12, a21, a22, ds(Vx, sc.Ux), ds(Vy, sc.Uy), literal != 0, wx, wy);
    const int r0 = M.ring_ptr[a], r1 = M.ring_ptr[a + 1];
    for (int i = 0; i < NQ; ++i) {
        const size_t q = (size_t)i * N + a;
        float f[MLP_IN];
        const int nr = mlp_features(M, F, a, i, f);
        for (int k = 0; k < MLP_IN; ++k) feat[q * MLP_IN + k] = f[k];
        nring[q] = (uint8_t)nr;
        int s = -1;
        double l0 = 0, xi = 0, eta = 0;
        double chx, chy, px, py;
        departure(a11, a12, a21, a22, wx, wy, (double)c_cx[i], (double)c_cy[i], Xa.x, Xa.y, chx, chy,
                  px, py);
        if (F.ok && !literal && !(chx == 0.0 && chy == 0.0)) {
            const Loc L = walk(M, a, Xa.x, Xa.y, px, py, err);
            if (L.e >= 0 && L.vnode < 0 && L.sx == 0 && L.sy == 0) {
                const int code = L.e | (1 << 28) | (1 << 30);
                for (int j = r0; j < r1; ++j)
                    if (M.ring[j] == code) s = j - r0;
                if (s >= 0) {
                    local_coords(M, L.e, 0, 0, px, py, xi, eta);
                    l0 = 1.0 - xi - eta;
                }
            }
        }
        slot[q] = (int16_t)s;
        bary[q * 3 + 0] = (float)l0;
        bary[q * 3 + 1] = (float)xi;
        bary[q * 3 + 2] = (float)eta;
    }
}

// ---------------------------------------------------------------------------
// training
// ---------------------------------------------------------------------------
__global__ void k_mlp_to_half(const float *w, __half *h, int n)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) h[p] = __float2half_rn(w[p]);
}

// Sample of minibatch position k: (mul * (base + k) + add) mod n, a
// permutation of 0..n-1 when gcd(mul, n) = 1.
__device__ __forceinline__ int64_t sample_index(int64_t k, int64_t n, int64_t mul, int64_t add)
{
    // n < 2^31, so mul * k + add < 2^63
    return (int64_t)(((uint64_t)mul * (uint64_t)k + (uint64_t)add) % (uint64_t)n);
}

// Forward and backward pass over tiles of 32 samples, 128 threads a block,
// each block's gradient to its own row of `part` and its loss to lpart[block]
// (summed in a fixed order by the next kernel: a training repeats bit for bit).
//
// FP32 fused multiply-adds bound it (41 kFLOP a sample).  Every matrix product
// is register-tiled with both operands read from shared memory as 16-byte
// vectors: rows are padded to 68 floats, so that the lanes of a quarter warp
// fall into different banks, and row-major tiles serve all three kinds of
// product (dots along a row forward, outer products over samples for the
// weight gradients and over outputs for the inputs' gradients).  The weight
// gradients stay in registers over a block's tiles.  An update on a minibatch
// of 8,192 (this kernel and k_mlp_reduce) takes 25 us, against 103 with one
// output per thread and iteration (32-way conflicts on the weight rows, 6,883
// atomics per 64 samples); 31 with the weights loaded one by one.
constexpr int LD = 68;  // padded row of 64 floats
constexpr int LO = 36;  // padded row of the 35 outputs
struct TrainSmem {
    float W2[MLP_H][LD], W3[LO][LD];
    float H1[TS][LD], H2[TS][LD], D2[TS][LD]; // activations; dA2; dA1 takes the place of H2
    float O[TS][LO];                          // outputs, then dO
    float X[TS][8], B[TS][4];
    float W1[MLP_H * MLP_IN], b1[MLP_H], b2[MLP_H], b3[LO];
    int SL[TS], NR[TS];
    double L[TRAIN_THREADS / 32];
};

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void fma4(float &c, float4 a, float4 b)
{
    c = fmaf(a.x, b.x, c);
    c = fmaf(a.y, b.y, c);
    c = fmaf(a.z, b.z, c);
    c = fmaf(a.w, b.w, c);
}
__device__ __forceinline__ void axpy4(float c[4], float a, float4 b)
{
    c[0] = fmaf(a, b.x, c[0]);
    c[1] = fmaf(a, b.y, c[1]);
    c[2] = fmaf(a, b.z, c[2]);
    c[3] = fmaf(a, b.w, c[3]);
}

__global__ void __launch_bounds__(TRAIN_THREADS, 3)
k_mlp_fwd_bwd(const __half *__restrict__ Wh, const float *__restrict__ feat,
              const int16_t *__restrict__ slot, const float *__restrict__ bary,
              const uint8_t *__restrict__ nring, int64_t n, int64_t base, int cnt, int64_t mul,
              int64_t add, float w_bary, float *__restrict__ part, double *__restrict__ lpart)
{
    extern __shared__ __align__(16) unsigned char raw[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(raw);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int tiles = (cnt + TS - 1) / TS;
    // a tile's samples: four threads each (the data is the caller's, so the
    // first tile is read before the previous update has finished)
    const auto load_samples = [&](int tile) {
        const int s = tid >> 2, r = tid & 3, k = tile * TS + s;
        const bool in = k < cnt;
        const int64_t q = in ? sample_index(base + k, n, mul, add) : 0;
        for (int c = r; c < MLP_IN; c += 4) S.X[s][c] = in ? feat[q * MLP_IN + c] : 0.0f;
        if (r < 3) S.B[s][r] = in ? bary[q * 3 + r] : 0.0f;
        if (r == 3) {
            S.SL[s] = in ? slot[q] : -1;
            S.NR[s] = in ? nring[q] : 0;
        }
    };
    load_samples(blockIdx.x);
    wait_prior_grid();
    { // the weights, eight FP16 values per load, all loads of a thread in flight
        static_assert(MLP_OFF_W2 % 8 == 0 && MLP_OFF_W3 % 8 == 0 && MLP_H % 8 == 0, "16-byte weight loads");
        constexpr int V2 = MLP_H * MLP_H / 8, V3 = MLP_OUT * MLP_H / 8, NV = (V2 + V3 + TRAIN_THREADS - 1) / TRAIN_THREADS;
        uint4 v[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            const int p = tid + c * TRAIN_THREADS;
            if (p < V2 + V3) v[c] = *reinterpret_cast<const uint4 *>(Wh + (p < V2 ? MLP_OFF_W2 + 8 * p : MLP_OFF_W3 + 8 * (p - V2)));
        }
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            const int p = tid + c * TRAIN_THREADS;
            if (p >= V2 + V3) continue;
            const int q = 8 * (p < V2 ? p : p - V2);
            float *d = p < V2 ? &S.W2[q / MLP_H][q % MLP_H] : &S.W3[q / MLP_H][q % MLP_H];
            const __half2 *h = reinterpret_cast<const __half2 *>(&v[c]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 f = __half22float2(h[k]);
                d[2 * k] = f.x;
                d[2 * k + 1] = f.y;
            }
        }
        if (tid < MLP_H) S.W3[MLP_OUT][tid] = 0.0f; // the padding row
    }
    for (int p = tid; p < MLP_H * MLP_IN; p += TRAIN_THREADS) S.W1[p] = __half2float(Wh[MLP_OFF_W1 + p]);
    if (tid < MLP_H) {
        S.b1[tid] = __half2float(Wh[MLP_OFF_B1 + tid]);
        S.b2[tid] = __half2float(Wh[MLP_OFF_B2 + tid]);
    } else if (tid < MLP_H + LO) {
        S.b3[tid - MLP_H] = tid - MLP_H < MLP_OUT ? __half2float(Wh[MLP_OFF_B3 + tid - MLP_H]) : 0.0f;
    }
    // the block's gradient: dW2 rows 4 ty .. and 32 + 4 ty .., columns 4 tx ..;
    // dW3 rows 4 ty .., columns 4 tx .., and rows 32 .. 34 by column; dW1 row
    // tid % 64, three columns; the biases by column
    float g2[2][4][4] = {}, g3[4][4] = {}, g3r[2] = {}, g1[3] = {}, gb1 = 0.f, gb2 = 0.f, gb3 = 0.f;
    double loss = 0.0; // of the warp's samples, in lane 0
    const float inv_cnt = 1.0f / (float)cnt;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (tile != (int)blockIdx.x) {
            __syncthreads(); // the previous tile's samples and dA1 have been read
            load_samples(tile);
        }
        __syncthreads();
        // layer 1: samples 4 ty .., units tx + 16 c
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j = tx + 16 * c;
            float w[MLP_IN];
#pragma unroll
            for (int k = 0; k < MLP_IN; ++k) w[k] = S.W1[j * MLP_IN + k];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float z = S.b1[j];
#pragma unroll
                for (int k = 0; k < MLP_IN; ++k) z = fmaf(w[k], S.X[4 * ty + r][k], z);
                S.H1[4 * ty + r][j] = tanhf(z);
            }
        }
        __syncthreads();
        { // layer 2
            float z[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) z[r][c] = S.b2[tx + 16 * c];
#pragma unroll 4
            for (int k = 0; k < MLP_H; k += 4) {
                float4 h[4], w[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) h[r] = ld4(&S.H1[4 * ty + r][k]);
#pragma unroll
                for (int c = 0; c < 4; ++c) w[c] = ld4(&S.W2[tx + 16 * c][k]);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) fma4(z[r][c], h[r], w[c]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) S.H2[4 * ty + r][tx + 16 * c] = tanhf(z[r][c]);
        }
        __syncthreads();
        { // layer 3: outputs tx, tx + 16 and (four lanes) tx + 32
            float z[4][3];
            const int j2 = tx < 4 ? tx + 32 : tx;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                z[r][0] = S.b3[tx];
                z[r][1] = S.b3[tx + 16];
                z[r][2] = S.b3[j2];
            }
#pragma unroll 4
            for (int k = 0; k < MLP_H; k += 4) {
                const float4 w0 = ld4(&S.W3[tx][k]), w1 = ld4(&S.W3[tx + 16][k]), w2 = ld4(&S.W3[j2][k]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float4 h = ld4(&S.H2[4 * ty + r][k]);
                    fma4(z[r][0], h, w0);
                    fma4(z[r][1], h, w1);
                    fma4(z[r][2], h, w2);
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                S.O[4 * ty + r][tx] = z[r][0];
                S.O[4 * ty + r][tx + 16] = z[r][1];
                if (tx < 4) S.O[4 * ty + r][tx + 32] = z[r][2];
            }
        }
        __syncthreads();
        { // loss and dO (in place): four lanes per sample, slots r + 4 c
            const int s = tid >> 2, r = tid & 3, nr = S.NR[s], sl = S.SL[s];
            float *o = S.O[s];
            float m = -INFINITY;
#pragma unroll
            for (int c = 0; c < MLP_K / 4; ++c)
                if (r + 4 * c < nr) m = fmaxf(m, o[r + 4 * c]);
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
            float Z = 0.f;
#pragma unroll
            for (int c = 0; c < MLP_K / 4; ++c)
                if (r + 4 * c < nr) Z += expf(o[r + 4 * c] - m);
            Z += __shfl_xor_sync(0xffffffffu, Z, 1);
            Z += __shfl_xor_sync(0xffffffffu, Z, 2);
            const float lz = logf(Z);
            const bool in = sl >= 0;
            const float osl = in ? o[sl] : 0.f; // read before any lane writes
            const float og = r < 3 ? o[MLP_K + r] : 0.f;
            float dv[MLP_K / 4];
#pragma unroll
            for (int c = 0; c < MLP_K / 4; ++c) {
                const int j = r + 4 * c;
                const float p = j < nr ? expf(o[j] - m - lz) : 0.f;
                dv[c] = in ? (p - (j == sl ? 1.f : 0.f)) * inv_cnt : 0.f;
            }
            __syncwarp();
#pragma unroll
            for (int c = 0; c < MLP_K / 4; ++c) o[r + 4 * c] = dv[c];
            const float gd = r < 3 ? og - S.B[s][r] : 0.f;
            o[MLP_K + r] = in && r < 3 ? w_bary * 2.0f * gd / 3.0f * inv_cnt : 0.f;
            // the tile's loss: FP32 over the warp's eight samples, FP64 from
            // there on, as a block's tiles grow with the number of samples
            float ls = in ? w_bary * (gd * gd) / 3.0f : 0.f;
            if (in && r == 0) ls += -(osl - m - lz);
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) ls += __shfl_xor_sync(0xffffffffu, ls, off);
            if ((tid & 31) == 0) loss += (double)ls;
        }
        __syncthreads();
        // dW3 (and its bias): outer products over the samples
#pragma unroll 4
        for (int s = 0; s < TS; ++s) {
            const float4 d = ld4(&S.O[s][4 * ty]), h = ld4(&S.H2[s][4 * tx]);
            axpy4(g3[0], d.x, h);
            axpy4(g3[1], d.y, h);
            axpy4(g3[2], d.z, h);
            axpy4(g3[3], d.w, h);
        }
#pragma unroll 4
        for (int s = 0; s < TS; ++s) {
            const float h = S.H2[s][tid & 63];
            g3r[0] = fmaf(S.O[s][32 + (tid >> 6)], h, g3r[0]);
            if (tid < 64) g3r[1] = fmaf(S.O[s][34], h, g3r[1]);
        }
        if (tid >= 64 && tid < 64 + MLP_OUT)
            for (int s = 0; s < TS; ++s) gb3 += S.O[s][tid - 64];
        { // dA2: samples 4 ty .., units 4 tx ..
            float z[4][4] = {};
#pragma unroll 3
            for (int j = 0; j < LO; j += 4) {
                float4 d[4], w[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) d[r] = ld4(&S.O[4 * ty + r][j]);
#pragma unroll
                for (int c = 0; c < 4; ++c) w[c] = ld4(&S.W3[j + c][4 * tx]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    axpy4(z[r], d[r].x, w[0]);
                    axpy4(z[r], d[r].y, w[1]);
                    axpy4(z[r], d[r].z, w[2]);
                    axpy4(z[r], d[r].w, w[3]);
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 h = ld4(&S.H2[4 * ty + r][4 * tx]);
                float4 v;
                v.x = z[r][0] * (1.0f - h.x * h.x);
                v.y = z[r][1] * (1.0f - h.y * h.y);
                v.z = z[r][2] * (1.0f - h.z * h.z);
                v.w = z[r][3] * (1.0f - h.w * h.w);
                *reinterpret_cast<float4 *>(&S.D2[4 * ty + r][4 * tx]) = v;
            }
        }
        __syncthreads();
        // dW2 and its bias
#pragma unroll 4
        for (int s = 0; s < TS; ++s) {
            const float4 d0 = ld4(&S.D2[s][4 * ty]), d1 = ld4(&S.D2[s][32 + 4 * ty]), h = ld4(&S.H1[s][4 * tx]);
            axpy4(g2[0][0], d0.x, h);
            axpy4(g2[0][1], d0.y, h);
            axpy4(g2[0][2], d0.z, h);
            axpy4(g2[0][3], d0.w, h);
            axpy4(g2[1][0], d1.x, h);
            axpy4(g2[1][1], d1.y, h);
            axpy4(g2[1][2], d1.z, h);
            axpy4(g2[1][3], d1.w, h);
        }
        if (tid < MLP_H)
            for (int s = 0; s < TS; ++s) gb2 += S.D2[s][tid];
        { // dA1 into H2
            float z[4][4] = {};
#pragma unroll 4
            for (int j = 0; j < MLP_H; j += 4) {
                float4 d[4], w[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) d[r] = ld4(&S.D2[4 * ty + r][j]);
#pragma unroll
                for (int c = 0; c < 4; ++c) w[c] = ld4(&S.W2[j + c][4 * tx]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    axpy4(z[r], d[r].x, w[0]);
                    axpy4(z[r], d[r].y, w[1]);
                    axpy4(z[r], d[r].z, w[2]);
                    axpy4(z[r], d[r].w, w[3]);
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 h = ld4(&S.H1[4 * ty + r][4 * tx]);
                float4 v;
                v.x = z[r][0] * (1.0f - h.x * h.x);
                v.y = z[r][1] * (1.0f - h.y * h.y);
                v.z = z[r][2] * (1.0f - h.z * h.z);
                v.w = z[r][3] * (1.0f - h.w * h.w);
                *reinterpret_cast<float4 *>(&S.H2[4 * ty + r][4 * tx]) = v;
            }
        }
        __syncthreads();
        // dW1 and its bias
#pragma unroll 4
        for (int s = 0; s < TS; ++s) {
            const float d = S.H2[s][tid & 63];
#pragma unroll
            for (int k = 0; k < 3; ++k) g1[k] = fmaf(d, S.X[s][3 * (tid >> 6) + k], g1[k]);
            if (tid < MLP_H) gb1 += d;
        }
    }
    float *P = part + (size_t)blockIdx.x * MLP_NP;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) P[MLP_OFF_W2 + (32 * h + 4 * ty + r) * MLP_H + 4 * tx + c] = g2[h][r][c];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) P[MLP_OFF_W3 + (4 * ty + r) * MLP_H + 4 * tx + c] = g3[r][c];
    P[MLP_OFF_W3 + (32 + (tid >> 6)) * MLP_H + (tid & 63)] = g3r[0];
    if (tid < 64) P[MLP_OFF_W3 + 34 * MLP_H + tid] = g3r[1];
#pragma unroll
    for (int k = 0; k < 3; ++k) P[MLP_OFF_W1 + (tid & 63) * MLP_IN + 3 * (tid >> 6) + k] = g1[k];
    if (tid < MLP_H) {
        P[MLP_OFF_B1 + tid] = gb1;
        P[MLP_OFF_B2 + tid] = gb2;
    }
    if (tid >= 64 && tid < 64 + MLP_OUT) P[MLP_OFF_B3 + tid - 64] = gb3;
    if ((tid & 31) == 0) S.L[tid >> 5] = loss;
    __syncthreads();
    if (tid == 0) {
        double l = 0.0;
        for (int w = 0; w < TRAIN_THREADS / 32; ++w) l += S.L[w];
        lpart[blockIdx.x] = l;
    }
}

// Sums the blocks' gradients and losses (rows of part and lpart) in a fixed
// order, adds the loss to *loss_sum and, with ADAM, updates the FP32 master
// weights and their FP16 copies; otherwise the gradient goes to g.  32
// parameters a block, eight threads each over every eighth row.
constexpr int RED_P = 32, RED_R = 8;
template <bool ADAM>
__global__ void __launch_bounds__(RED_P *RED_R)
k_mlp_reduce(const float *__restrict__ part, const double *__restrict__ lpart, int rows, double *loss_sum, float *w,
             float *m, float *v, float *g, __half *h, float lr, float c1, float c2)
{
    __shared__ float red[RED_R][RED_P + 1];
    wait_prior_grid();
    const int px = threadIdx.x % RED_P, r = threadIdx.x / RED_P, p = blockIdx.x * RED_P + px;
    float sum = 0.f;
    if (p < MLP_NP) {
#pragma unroll 8
        for (int b = r; b < rows; b += RED_R) sum += part[(size_t)b * MLP_NP + p];
    }
    red[r][px] = sum;
    __syncthreads();
    if (blockIdx.x == 0 && r == 1) { // one warp: the losses
        double l = 0.0;
        for (int b = px; b < rows; b += RED_P) l += lpart[b];
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if (px == 0) *loss_sum += l;
    }
    if (r != 0 || p >= MLP_NP) return;
    float gp = 0.f;
#pragma unroll
    for (int q = 0; q < RED_R; ++q) gp += red[q][px];
    if (!ADAM) {
        g[p] = gp;
        return;
    }
    const float mp = 0.9f * m[p] + 0.1f * gp;
    const float vp = 0.999f * v[p] + 0.001f * gp * gp;
    m[p] = mp;
    v[p] = vp;
    const float wp = w[p] - lr * (mp * c1) / (sqrtf(vp * c2) + 1e-8f);
    w[p] = wp;
    h[p] = __float2half_rn(wp);
}

// ---------------------------------------------------------------------------
// inference on the tensor cores
// ---------------------------------------------------------------------------
struct PredSmem {
    __half W1[MLP_H][16];  // input padded 6 -> 16
    __half W2[MLP_H][MLP_H];
    __half W3[40][MLP_H];  // outputs padded 35 -> 40
    float b1[MLP_H], b2[MLP_H], b3[40];
    __half Xs[PRED_WARPS][16][16];
    float Os[PRED_WARPS][16][40];
};

__device__ __forceinline__ void load_pred_weights(PredSmem &S, const __half *__restrict__ Wh)
{
    for (int p = threadIdx.x; p < MLP_H * 16; p += blockDim.x) {
        const int j = p / 16, k = p % 16;
        S.W1[j][k] = k < MLP_IN ? Wh[MLP_OFF_W1 + j * MLP_IN + k] : __float2half_rn(0.0f);
    }
    for (int p = threadIdx.x; p < MLP_H * MLP_H; p += blockDim.x) S.W2[p / MLP_H][p % MLP_H] = Wh[MLP_OFF_W2 + p];
    for (int p = threadIdx.x; p < 40 * MLP_H; p += blockDim.x) {
        const int j = p / MLP_H, k = p % MLP_H;
        S.W3[j][k] = j < MLP_OUT ? Wh[MLP_OFF_W3 + p] : __float2half_rn(0.0f);
    }
    for (int p = threadIdx.x; p < MLP_H; p += blockDim.x) {
        S.b1[p] = __half2float(Wh[MLP_OFF_B1 + p]);
        S.b2[p] = __half2float(Wh[MLP_OFF_B2 + p]);
    }
    for (int p = threadIdx.x; p < 40; p += blockDim.x) S.b3[p] = p < MLP_OUT ? __half2float(Wh[MLP_OFF_B3 + p]) : 0.0f;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ uint32_t lds32(const __half *p) { return *reinterpret_cast<const uint32_t *>(p); }

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The network on the 16 queries of this warp's tile: features in
// S.Xs[w] (FP16, rows 0..15), outputs to S.Os[w] (FP32).  All 32 lanes.
__device__ __forceinline__ void warp_forward(PredSmem &S, int w)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    uint32_t A[4][4];
    float c[8][4];
    {
        uint32_t a0[4] = {lds32(&S.Xs[w][g][2 * t]), lds32(&S.Xs[w][g + 8][2 * t]),
                          lds32(&S.Xs[w][g][8 + 2 * t]), lds32(&S.Xs[w][g + 8][8 + 2 * t])};
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const int col = nt * 8 + 2 * t;
            c[nt][0] = c[nt][2] = S.b1[col];
            c[nt][1] = c[nt][3] = S.b1[col + 1];
            mma16816(c[nt], a0, lds32(&S.W1[nt * 8 + g][2 * t]), lds32(&S.W1[nt * 8 + g][8 + 2 * t]));
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        A[q][0] = pack2(tanhf(c[2 * q][0]), tanhf(c[2 * q][1]));
        A[q][1] = pack2(tanhf(c[2 * q][2]), tanhf(c[2 * q][3]));
        A[q][2] = pack2(tanhf(c[2 * q + 1][0]), tanhf(c[2 * q + 1][1]));
        A[q][3] = pack2(tanhf(c[2 * q + 1][2]), tanhf(c[2 * q + 1][3]));
    }
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const int col = nt * 8 + 2 * t;
        c[nt][0] = c[nt][2] = S.b2[col];
        c[nt][1] = c[nt][3] = S.b2[col + 1];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            mma16816(c[nt], A[q], lds32(&S.W2[nt * 8 + g][16 * q + 2 * t]),
                     lds32(&S.W2[nt * 8 + g][16 * q + 8 + 2 * t]));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        A[q][0] = pack2(tanhf(c[2 * q][0]), tanhf(c[2 * q][1]));
        A[q][1] = pack2(tanhf(c[2 * q][2]), tanhf(c[2 * q][3]));
        A[q][2] = pack2(tanhf(c[2 * q + 1][0]), tanhf(c[2 * q + 1][1]));
        A[q][3] = pack2(tanhf(c[2 * q + 1][2]), tanhf(c[2 * q + 1][3]));
    }
#pragma unroll
    for (int nt = 0; nt < 5; ++nt) {
        const int col = nt * 8 + 2 * t;
        float d[4] = {S.b3[col], S.b3[col + 1], S.b3[col], S.b3[col + 1]};
#pragma unroll
        for (int q = 0; q < 4; ++q)
            mma16816(d, A[q], lds32(&S.W3[nt * 8 + g][16 * q + 2 * t]),
                     lds32(&S.W3[nt * 8 + g][16 * q + 8 + 2 * t]));
        S.Os[w][g][col] = d[0];
        S.Os[w][g][col + 1] = d[1];
        S.Os[w][g + 8][col] = d[2];
        S.Os[w][g + 8][col + 1] = d[3];
    }
}

__device__ __forceinline__ int masked_argmax(const float *o, int nr)
{
    int best = 0;
    float bv = o[0];
    for (int j = 1; j < nr && j < MLP_K; ++j)
        if (o[j] > bv) {
            bv = o[j];
            best = j;
        }
    return best;
}

// Proposals for the work list of the exact path (after k_stream_fast):
// prop[w] = ring element of the largest logit, or -1 (no usable map).
template <class T>
__global__ void __launch_bounds__(PRED_WARPS * 32)
k_propose(MeshDev M, MapStatic MS, MapScalarsF sf, StateDev<T> st, const __half *__restrict__ Wh,
          int flags, int *prop, unsigned long long *made)
{
    wait_prior_grid();
    __shared__ PredSmem S;
    load_pred_weights(S, Wh);
    __syncthreads();
    __shared__ unsigned pre[NQ + 1];
    if (threadIdx.x == 0) work_prefix(st.wcount, pre);
    __syncthreads();
    const unsigned n = pre[NQ];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned nwarps = gridDim.x * PRED_WARPS;
    unsigned count = 0;
    for (unsigned base = (blockIdx.x * PRED_WARPS + w) * 16u; base < n; base += nwarps * 16u) {
        int a = -1, nr = 0;
        const unsigned q = base + (unsigned)lane;
        if (lane < 16) {
            float f[MLP_IN] = {0, 0, 0, 0, 0, 0};
            if (q < n) {
                const int code = work_at(st.work, M.N, pre, q);
                a = code / NQ;
                const int i = code % NQ;
                const FastMap F = fast_map(MS, sf, a, M.Xf[a]);
                const int r = mlp_features(M, F, a, i, f);
                nr = (F.ok && !(flags & FLAG_LITERAL_VG)) ? r : 0;
            }
            for (int k = 0; k < 16; ++k) S.Xs[w][lane][k] = __float2half_rn(k < MLP_IN ? f[k] : 0.0f);
        }
        __syncwarp();
        warp_forward(S, w);
        __syncwarp();
        if (lane < 16 && q < n) {
            int pc = -1;
            if (nr > 0) {
                pc = M.ring[M.ring_ptr[a] + masked_argmax(S.Os[w][lane], nr)];
                ++count;
            }
            prop[q] = pc;
        }
        __syncwarp();
    }
    for (int off = 16; off > 0; off >>= 1) count += __shfl_down_sync(0xffffffffu, count, off);
    if (lane == 0 && count && made) atomicAdd(made, (unsigned long long)count);
}

// Inference on given features (tests): slot of the largest logit among the
// first nring, and optionally all 35 outputs.
__global__ void __launch_bounds__(PRED_WARPS * 32)
k_mlp_predict(const __half *__restrict__ Wh, const float *__restrict__ feat,
              const uint8_t *__restrict__ nring, int64_t n, int32_t *pslot, float *out)
{
    __shared__ PredSmem S;
    load_pred_weights(S, Wh);
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * PRED_WARPS;
    for (int64_t base = ((int64_t)blockIdx.x * PRED_WARPS + w) * 16; base < n; base += nwarps * 16) {
        const int64_t q = base + lane;
        if (lane < 16)
            for (int k = 0; k < 16; ++k)
                S.Xs[w][lane][k] = __float2half_rn(k < MLP_IN && q < n ? feat[q * MLP_IN + k] : 0.0f);
        __syncwarp();
        warp_forward(S, w);
        __syncwarp();
        if (lane < 16 && q < n) {
            const int nr = nring[q];
            pslot[q] = nr > 0 ? masked_argmax(S.Os[w][lane], nr) : -1;
            if (out)
                for (int j = 0; j < MLP_OUT; ++j) out[q * MLP_OUT + j] = S.Os[w][lane][j];
        }
        __syncwarp();
    }
}

uint64_t splitmix64(uint64_t &x)
{
    uint64_t z = (x += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

int64_t gcd64(int64_t a, int64_t b)
{
    while (b) {
        const int64_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

} // namespace

struct alelb_mlp {
    std::string err;
    float *d_w = nullptr, *d_m = nullptr, *d_v = nullptr, *d_g = nullptr;
    __half *d_h = nullptr;
    double *d_loss = nullptr;
    float *d_part = nullptr;   // [grid][MLP_NP] the training blocks' gradients
    double *d_lpart = nullptr; // [grid] their losses
    int grid = 0;              // most training blocks: two per SM
    int64_t t = 0;
    cudaStream_t stream = nullptr;
    DevBuf buf;
};

namespace {

alelb_status mfail(alelb_mlp *m, cudaError_t st, const char *what)
{
    m->err = std::string(what) + ": " + cudaGetErrorString(st);
    return st == cudaErrorMemoryAllocation ? ALELB_ERR_OOM : ALELB_ERR_CUDA;
}

cudaError_t refresh_half(alelb_mlp *m)
{
    k_mlp_to_half<<<(MLP_NP + 255) / 256, 256, 0, m->stream>>>(m->d_w, m->d_h, MLP_NP);
    return cudaGetLastError();
}

// The gradients of samples base .. base + cnt - 1 of the pass's order as block
// rows of m->d_part; returns their number in rows.
cudaError_t fwd_bwd(alelb_mlp *m, const float *feat, const int16_t *slot, const float *bary,
                    const uint8_t *nring, int64_t n, int64_t base, int cnt, int64_t mul, int64_t add,
                    float w_bary, int &rows)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t st = cudaFuncSetAttribute(k_mlp_fwd_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)sizeof(TrainSmem));
        if (st != cudaSuccess) return st;
        attr = true;
    }
    rows = std::min((cnt + TS - 1) / TS, m->grid);
    launch_pdl_smem(k_mlp_fwd_bwd, dim3(rows), dim3(TRAIN_THREADS), sizeof(TrainSmem), m->stream, (const __half *)m->d_h, feat,
               slot, bary, nring, n, base, cnt, mul, add, w_bary, m->d_part, m->d_lpart);
    return cudaGetLastError();
}

// After fwd_bwd: the Adam update (adam), or the gradient into m->d_g.
cudaError_t reduce(alelb_mlp *m, int rows, bool adam, float lr, float c1, float c2)
{
    const dim3 grid((MLP_NP + RED_P - 1) / RED_P), block(RED_P * RED_R);
    launch_pdl(adam ? k_mlp_reduce<true> : k_mlp_reduce<false>, grid, block, m->stream, (const float *)m->d_part,
               (const double *)m->d_lpart, rows, m->d_loss, m->d_w, m->d_m, m->d_v, m->d_g, m->d_h, lr, c1, c2);
    return cudaGetLastError();
}

} // namespace

namespace alelb {

// Proposals for the solver's current work list (deviation-form step).
cudaError_t mlp_propose(alelb_solver *s, const MapScalarsF &sf)
{
    alelb_mesh *m = s->mesh;
    with_state(s, [&](auto &st, auto &) {
        k_propose<<<2 * s->n_sm, PRED_WARPS * 32, 0, s->stream>>>(m->dev, m->mst, sf, st, s->mlp->d_h, s->flags,
                                                                   s->d_prop, s->d_stats + 2);
    });
    return cudaGetLastError();
}

} // namespace alelb

extern "C" alelb_status alelb_mlp_create(const float *params, uint64_t seed, alelb_mlp **out)
{
    if (!out) return ALELB_ERR_ARG;
    alelb_mlp *m = new (std::nothrow) alelb_mlp();
    if (!m) return ALELB_ERR_OOM;
    *out = m;
    std::vector<float> w(MLP_NP);
    if (params) {
        for (int p = 0; p < MLP_NP; ++p) w[p] = params[p];
    } else {
        // Glorot-uniform weights, zero biases
        uint64_t x = seed;
        const int fan[3][2] = {{MLP_IN, MLP_H}, {MLP_H, MLP_H}, {MLP_H, MLP_OUT}};
        const int offw[3] = {MLP_OFF_W1, MLP_OFF_W2, MLP_OFF_W3};
        const int offb[3] = {MLP_OFF_B1, MLP_OFF_B2, MLP_OFF_B3};
        for (int l = 0; l < 3; ++l) {
            const double lim = std::sqrt(6.0 / (fan[l][0] + fan[l][1]));
            for (int p = 0; p < fan[l][0] * fan[l][1]; ++p) {
                const double u = (double)(splitmix64(x) >> 11) * (1.0 / 9007199254740992.0);
                w[offw[l] + p] = (float)((2.0 * u - 1.0) * lim);
            }
            for (int p = 0; p < fan[l][1]; ++p) w[offb[l] + p] = 0.0f;
        }
    }
    cudaError_t st = cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking);
    m->d_w = m->buf.put(w, st);
    m->d_m = m->buf.alloc<float>(MLP_NP, st);
    m->d_v = m->buf.alloc<float>(MLP_NP, st);
    m->d_g = m->buf.alloc<float>(MLP_NP, st);
    m->d_h = m->buf.alloc<__half>(MLP_NP, st);
    m->d_loss = m->buf.alloc<double>(1, st);
    {
        int dev = 0, nsm = 0;
        m->grid = 2 * 152;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && nsm > 0)
            m->grid = 2 * nsm;
    }
    m->d_part = m->buf.alloc<float>((size_t)m->grid * MLP_NP, st);
    m->d_lpart = m->buf.alloc<double>(m->grid, st);
    if (st == cudaSuccess) st = cudaMemset(m->d_m, 0, MLP_NP * sizeof(float));
    if (st == cudaSuccess) st = cudaMemset(m->d_v, 0, MLP_NP * sizeof(float));
    if (st == cudaSuccess) st = cudaDeviceSynchronize(); // legacy-stream uploads before m->stream work
    if (st == cudaSuccess) st = refresh_half(m);
    if (st == cudaSuccess) st = cudaStreamSynchronize(m->stream);
    if (st != cudaSuccess) return mfail(m, st, "mlp_create");
    return ALELB_OK;
}

extern "C" void alelb_mlp_destroy(alelb_mlp *m)
{
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    m->buf.release();
    if (m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

extern "C" const char *alelb_mlp_last_error(alelb_mlp *m) { return m ? m->err.c_str() : "null network"; }

extern "C" alelb_status alelb_mlp_get_params(alelb_mlp *m, int32_t rounded, float *params)
{
    if (!m || !params) return ALELB_ERR_ARG;
    cudaError_t st = cudaSuccess;
    if (rounded) {
        std::vector<__half> h(MLP_NP);
        st = cudaMemcpyAsync(h.data(), m->d_h, MLP_NP * sizeof(__half), cudaMemcpyDeviceToHost, m->stream);
        if (st == cudaSuccess) st = cudaStreamSynchronize(m->stream);
        if (st == cudaSuccess)
            for (int p = 0; p < MLP_NP; ++p) params[p] = __half2float(h[p]);
    } else {
        st = cudaMemcpyAsync(params, m->d_w, MLP_NP * sizeof(float), cudaMemcpyDeviceToHost, m->stream);
        if (st == cudaSuccess) st = cudaStreamSynchronize(m->stream);
    }
    if (st != cudaSuccess) return mfail(m, st, "mlp_get_params");
    return ALELB_OK;
}

extern "C" alelb_status alelb_mlp_loss_grad(alelb_mlp *m, const float *feat, const int16_t *slot,
                                            const float *bary, const uint8_t *nring, int64_t n,
                                            float w_bary, double *loss, float *grad)
{
    if (!m || !feat || !slot || !bary || !nring || n < 1 || n > (1 << 30)) return ALELB_ERR_ARG;
    cudaError_t st = cudaMemsetAsync(m->d_loss, 0, sizeof(double), m->stream);
    int rows = 0;
    if (st == cudaSuccess) st = fwd_bwd(m, feat, slot, bary, nring, n, 0, (int)n, 1, 0, w_bary, rows);
    if (st == cudaSuccess) st = reduce(m, rows, false, 0.f, 0.f, 0.f);
    double ls = 0;
    if (st == cudaSuccess) st = cudaMemcpyAsync(&ls, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
    if (st == cudaSuccess && grad)
        st = cudaMemcpyAsync(grad, m->d_g, MLP_NP * sizeof(float), cudaMemcpyDeviceToHost, m->stream);
    if (st == cudaSuccess) st = cudaStreamSynchronize(m->stream);
    if (st != cudaSuccess) return mfail(m, st, "mlp_loss_grad");
    if (loss) *loss = ls / (double)n;
    return ALELB_OK;
}

extern "C" alelb_status alelb_mlp_train(alelb_mlp *m, const float *feat, const int16_t *slot,
                                        const float *bary, const uint8_t *nring, int64_t n,
                                        int32_t epochs, int32_t batch, float lr, float w_bary,
                                        uint64_t seed, double *epoch_loss)
{
    if (!m || !feat || !slot || !bary || !nring || n < 1 || n > 2147483647LL || epochs < 0 || batch < 1 ||
        batch > (1 << 20) || !(lr > 0.0f))
        return ALELB_ERR_ARG;
    uint64_t x = seed;
    cudaError_t st = cudaSuccess;
    for (int ep = 0; ep < epochs && st == cudaSuccess; ++ep) {
        int64_t mul = 1 + (int64_t)(splitmix64(x) % (uint64_t)n);
        while (gcd64(mul, n) != 1) mul = mul % n + 1;
        const int64_t add = (int64_t)(splitmix64(x) % (uint64_t)n);
        st = cudaMemsetAsync(m->d_loss, 0, sizeof(double), m->stream);
        for (int64_t base = 0; base < n && st == cudaSuccess; base += batch) {
            const int cnt = (int)std::min<int64_t>(batch, n - base);
            int rows = 0;
            st = fwd_bwd(m, feat, slot, bary, nring, n, base, cnt, mul, add, w_bary, rows);
            if (st != cudaSuccess) break;
            m->t += 1;
            const float c1 = (float)(1.0 / (1.0 - std::pow(0.9, (double)m->t)));
            const float c2 = (float)(1.0 / (1.0 - std::pow(0.999, (double)m->t)));
            st = reduce(m, rows, true, lr, c1, c2);
        }
        double ls = 0;
        if (st == cudaSuccess)
            st = cudaMemcpyAsync(&ls, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
        if (st == cudaSuccess) st = cudaStreamSynchronize(m->stream);
        if (epoch_loss) epoch_loss[ep] = ls / (double)n;
    }
    if (st != cudaSuccess) return mfail(m, st, "mlp_train");
    return ALELB_OK;
}

extern "C" alelb_status alelb_mlp_predict(alelb_mlp *m, const float *feat, const uint8_t *nring, int64_t n,
                                          int32_t *slot, float *out)
{
    if (!m || !feat || !nring || !slot || n < 1) return ALELB_ERR_ARG;
    const int64_t tiles = (n + 15) / 16;
    const int blocks = (int)std::min<int64_t>((tiles + PRED_WARPS - 1) / PRED_WARPS, 4096);
    k_mlp_predict<<<blocks, PRED_WARPS * 32, 0, m->stream>>>(m->d_h, feat, nring, n, slot, out);
    cudaError_t st = cudaGetLastError();
    if (st == cudaSuccess) st = cudaStreamSynchronize(m->stream);
    if (st != cudaSuccess) return mfail(m, st, "mlp_predict");
    return ALELB_OK;
}

extern "C" alelb_status alelb_samples(alelb_solver *s, double t, float *feat, int16_t *slot, float *bary,
                                      uint8_t *nring)
{
    if (!s || !s->mesh || !feat || !slot || !bary || !nring) return ALELB_ERR_ARG;
    alelb_mesh *m = s->mesh;
    if (m->etype != ALELB_ELEM_P2TRI) {
        s->err = "samples: the learned proposal serves 6-node triangle meshes";
        return ALELB_ERR_ARG;
    }
    const MapScalars sc = solver_map(s, map_scalars(m->T.mkind, m->T.mp, t));
    k_samples<<<(m->T.N + 127) / 128, 128, 0, s->stream>>>(m->dev, m->mst, sc, to_f32(sc, m->T), s->flags, feat,
                                                            slot, bary, nring, s->d_err);
    cudaError_t st = cudaGetLastError();
    if (st == cudaSuccess) st = cudaStreamSynchronize(s->stream);
    if (st != cudaSuccess) {
        s->err = cudaGetErrorString(st);
        return ALELB_ERR_CUDA;
    }
    return ALELB_OK;
}

extern "C" alelb_status alelb_solver_set_mlp(alelb_solver *s, alelb_mlp *m)
{
    if (!s) return ALELB_ERR_ARG;
    if (m && s->prec == ALELB_PREC_FP64) {
        s->err = "the learned proposal serves the deviation-form propagation only";
        return ALELB_ERR_ARG;
    }
    if (m && s->mesh->etype != ALELB_ELEM_P2TRI) {
        s->err = "the learned proposal serves 6-node triangle meshes";
        return ALELB_ERR_ARG;
    }
    if (m && !s->d_prop) {
        cudaError_t st = cudaSuccess;
        s->d_prop = s->buf.alloc<int>((size_t)9 * s->mesh->T.N, st);
        if (st != cudaSuccess) {
            s->err = cudaGetErrorString(st);
            return ALELB_ERR_OOM;
        }
    }
    // the network's weights are final once the solver's stream reaches this point
    if (m) cudaStreamSynchronize(m->stream);
    s->mlp = m;
    return ALELB_OK;
}

extern "C" alelb_status alelb_mlp_stats(alelb_solver *s, int64_t out[3])
{
    if (!s || !out) return ALELB_ERR_ARG;
    unsigned long long h[3] = {0, 0, 0};
    cudaError_t st = cudaMemcpyAsync(h, s->d_stats, sizeof(h), cudaMemcpyDeviceToHost, s->stream);
    if (st == cudaSuccess) st = cudaStreamSynchronize(s->stream);
    if (st != cudaSuccess) {
        s->err = cudaGetErrorString(st);
        return ALELB_ERR_CUDA;
    }
    out[0] = (int64_t)h[0]; // populations left to the exact path
    out[1] = (int64_t)h[2]; // proposals made
    out[2] = (int64_t)h[1]; // proposals accepted
    return ALELB_OK;
}
