// dsmc_mlp.cu -- the HoT surrogate network: input features, forward and
// backward passes with bfloat16 weights and FP32 accumulation, Adam, and the
// HoT it hands to the synthetic equations.  An extension: the paper takes
// the higher-order terms of Eq. (hot_constitutive) from DSMC moments alone.
//
// Training: see k_mlp_train.  The CTAs' gradient sums are added in a fixed
// order by a second kernel (the result does not depend on scheduling), which
// also takes the Adam step.
#include <cmath>
#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "dsmc_grad.cuh"
#include "dsmc_internal.h"

namespace dsmc {

namespace {

__host__ __device__ constexpr int nin(int k) { return k == 0 ? 12 : 64; }
__host__ __device__ constexpr int nout(int k) { return k == 3 ? 5 : 64; }

// offsets of W_k and b_k in the parameter vector
__host__ __device__ constexpr int poff_w(int k) {
  return k == 0 ? 0 : poff_w(k - 1) + nin(k - 1) * nout(k - 1) + nout(k - 1);
}
__host__ __device__ constexpr int poff_b(int k) { return poff_w(k) + nin(k) * nout(k); }
static_assert(poff_b(3) + nout(3) == MLP_NPARAM, "parameter count");

__device__ __forceinline__ float bf16_to_f(uint16_t h) { return __uint_as_float((uint32_t)h << 16); }

// Per cell: inputs (12), scales (4), normalised HoT targets (5, if hot) and
// weight (1 where mask = 1 and the cell state admits the inputs); a cell with
// mask = 0 is neither trained on nor replaced and gets zeros.
// The FP64 pipe bounds it (2 lanes per clock and SM): the divisions by the
// cell's own scales are one reciprocal each, the y gradients of a 1D case
// (zero) are not formed.  The count is added once per warp.
// 160 000 cells (1D): 236 us before, 61 us now.
__global__ void __launch_bounds__(128) k_mlp_data(const CellParams* __restrict__ cps,
                           const int32_t* __restrict__ cell_case,
                           const int32_t* __restrict__ cell0, int ncells, const double* __restrict__ F,
                           const double* __restrict__ hot, const double* __restrict__ kngll,
                           const uint8_t* __restrict__ mask, float* __restrict__ X, float* __restrict__ Y,
                           float* __restrict__ S, float* __restrict__ w, int32_t* __restrict__ count) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  bool ok = false;
  if (c < ncells) {
    float x[12], sc[4], y[5];
#pragma unroll
    for (int k = 0; k < 12; ++k) x[k] = 0.f;
#pragma unroll
    for (int k = 0; k < 5; ++k) y[k] = 0.f;
    sc[0] = sc[1] = sc[2] = 1.f;
    sc[3] = 0.f;
    if (mask[c] != 0) {
      const int cs = cell_case[c];
      const CellParams& cp = cps[cs];
      const int lc = c - cell0[cs];
      const double* f = F + (size_t)c * 18;
      const double rho = f[0], tt = f[4], tr = f[5];
      const double i3 = 1.0 / (3.0 + cp.d_r);
      const double T = (3.0 * tt + cp.d_r * tr) * i3;
      ok = rho > 0.0 && tt > 0.0 && tr > 0.0 && isfinite(T);
      if (ok) {
        const bool one = cp.dim == 1;
        // T^omega as exp(omega log T), within a few ulp of 64 bits; the inputs
        // are rounded to 32
        const double mu = cp.mu_ref * exp(cp.omega * log(T));
        const double sq = sqrt(T), iT = 1.0 / T, irho = 1.0 / rho, isq = sq * iT;
        // lambda / norm of rho; u_x, u_y; T_t, T_r
        const double lam = mu * irho * isq * 1.2533141373155003;  // sqrt(pi / 2)
        const double ln[5] = {lam * irho, lam * isq, lam * isq, lam * iT, lam * iT};
        double gx[5], gy[5];
        const Line1 line(cp, c, lc);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const int col = k < 3 ? k : k + 1;  // rho, u_x, u_y, T_t, T_r
          auto val = [&](int q) { return F[(size_t)q * 18 + col]; };
          if (one) {
            gx[k] = line.grad(val);
            gy[k] = 0.0;
          } else {
            grad2(cp, c, lc, val, &gx[k], &gy[k]);
          }
          x[2 * k] = (float)(ln[k] * gx[k]);
          x[2 * k + 1] = one ? 0.f : (float)(ln[k] * gy[k]);
        }
        x[10] = (float)kngll[c];
        x[11] = (float)(tr / tt);
        // grad T from the gradients of T_t and T_r
        const double gTx = (3.0 * gx[3] + cp.d_r * gx[4]) * i3, gTy = (3.0 * gy[3] + cp.d_r * gy[4]) * i3;
        double ex = 1.0, ey = 0.0;
        if (one) {
          if (gTx < 0.0) ex = -1.0;
        } else {
          const double gn = sqrt(gTx * gTx + gTy * gTy);
          if (gn > 0.0) {
            ex = gTx / gn;
            ey = gTy / gn;
          }
        }
        const double p = rho * T, ps = p * sq;
        sc[0] = (float)p;
        sc[1] = (float)ps;
        sc[2] = (float)ex;
        sc[3] = (float)ey;
        bool fin = true;
        if (hot) {
          const double* h = hot + (size_t)c * 12;
          const double ip = irho * iT, ips = ip * isq;
          const double yd[5] = {h[0] * ip, h[3] * ip, h[1] * ip, (h[6] * ex + h[7] * ey) * ips,
                                (h[9] * ex + h[10] * ey) * ips};
#pragma unroll
          for (int k = 0; k < 5; ++k) {
            fin = fin && isfinite(yd[k]);
            y[k] = (float)yd[k];
          }
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) fin = fin && isfinite(ln[k] * gx[k]) && (one || isfinite(ln[k] * gy[k]));
        ok = fin && isfinite(kngll[c]) && isfinite(tr / tt);
        if (!ok) {
#pragma unroll
          for (int k = 0; k < 12; ++k) x[k] = 0.f;
#pragma unroll
          for (int k = 0; k < 5; ++k) y[k] = 0.f;
          sc[0] = sc[1] = sc[2] = 1.f;
          sc[3] = 0.f;
        }
      }
    }
    float4* X4 = reinterpret_cast<float4*>(X + (size_t)c * 12);
    X4[0] = make_float4(x[0], x[1], x[2], x[3]);
    X4[1] = make_float4(x[4], x[5], x[6], x[7]);
    X4[2] = make_float4(x[8], x[9], x[10], x[11]);
    *reinterpret_cast<float4*>(S + (size_t)c * 4) = make_float4(sc[0], sc[1], sc[2], sc[3]);
#pragma unroll
    for (int k = 0; k < 5; ++k) Y[(size_t)c * 5 + k] = y[k];
    w[c] = ok ? 1.f : 0.f;
  }
  const unsigned used = __ballot_sync(0xffffffffu, ok);
  if ((threadIdx.x & 31) == 0 && used) atomicAdd(count, __popc(used));
}

// ---------------------------------------------------------------------------
// Loss and gradient (FP32 arithmetic on the bfloat16 weights).  A CTA of 256
// threads takes tiles of 32 cells.  Bound by the FP32 pipe once the operands
// come from shared memory in 16-byte loads: activations and deltas lie
// feature by feature (row of a feature: the tile's 32 cells, padded to 36
// words), so that
//  - a layer's forward and delta products are 4 x 4 register tiles (4 cells, 4
//    neurons a thread, two loads for 16 multiply-adds; 128 threads cover 32 x
//    64), the weights kept in both orientations with the columns n, n + 16, n
//    + 32, n + 48 of a thread adjacent;
//  - a 64 x 64 weight gradient is a 4 x 4 tile per thread of all 256, summed
//    over the cells four at a time, and stays in the thread's registers over
//    all tiles of the CTA: no gradient in shared memory, no atomics.
// The grid is one CTA per SM, and tiles of 32 keep the last round short: 12
// 800 cells are 400 tiles, 3 rounds on 152 SMs.  12 800 cells: 108 us with
// scalar products from shared memory and a gradient array there, 42 us.
// ---------------------------------------------------------------------------
constexpr int TR_TILE = 32;
constexpr int TR_THREADS = 256;
constexpr int TR_LD = TR_TILE + 4;
// shared memory, floats
constexpr int TR_W0T = 0;                       // [12][64], columns permuted
constexpr int TR_W1T = TR_W0T + 12 * 64;        // [in 64][out 64]
constexpr int TR_W2T = TR_W1T + 64 * 64;
constexpr int TR_W1 = TR_W2T + 64 * 64;         // [out 64][in 64]
constexpr int TR_W2 = TR_W1 + 64 * 64;
constexpr int TR_W3 = TR_W2 + 64 * 64;          // [5][64], plain
constexpr int TR_B = TR_W3 + 5 * 64;            // 3 x 64 + 8
constexpr int TR_A0 = TR_B + 200;               // [12][36]
constexpr int TR_A1 = TR_A0 + 12 * TR_LD;       // [64][36] x 3
constexpr int TR_A2 = TR_A1 + 64 * TR_LD;
constexpr int TR_A3 = TR_A2 + 64 * TR_LD;
constexpr int TR_D3 = TR_A3 + 64 * TR_LD;       // [5][36]
constexpr int TR_DA = TR_D3 + 5 * TR_LD;        // [64][36] x 2
constexpr int TR_DB = TR_DA + 64 * TR_LD;
constexpr int TR_WT = TR_DB + 64 * TR_LD;       // cell weights
constexpr int TR_FLOATS = TR_WT + TR_TILE;
inline size_t train_smem_bytes() { return sizeof(float) * (size_t)TR_FLOATS; }
static_assert(TR_A0 % 4 == 0 && TR_D3 % 4 == 0 && TR_DA % 4 == 0 && TR_W1T % 4 == 0, "16-byte rows");

// where column n of a 64-column row lies: the four columns of a thread (n & 15)
// are adjacent
__device__ __forceinline__ int perm64(int n) { return 4 * (n & 15) + (n >> 4); }

// acc[c][n] += sum_i A[i][4 tc + c] W[i][column n of thread tn], i < K
template <int K>
__device__ __forceinline__ void tile_product(const float* A, const float* W, int tc, int tn, float (*acc)[4]) {
#pragma unroll 8
  for (int i = 0; i < K; ++i) {
    const float4 a = *reinterpret_cast<const float4*>(A + i * TR_LD + 4 * tc);
    const float4 w = *reinterpret_cast<const float4*>(W + i * 64 + 4 * tn);
    const float av[4] = {a.x, a.y, a.z, a.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int n = 0; n < 4; ++n) acc[c][n] = fmaf(av[c], wv[n], acc[c][n]);
  }
}

// out[n][c] = tanh(b[n] + sum_i W[n][i] A[i][c])
template <int K>
__device__ __forceinline__ void layer_forward(const float* A, const float* Wt, const float* b, float* out) {
  if (threadIdx.x < 128) {
    const int tn = threadIdx.x & 15, tc = threadIdx.x >> 4;
    float acc[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const float bn = b[tn + 16 * n];
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c][n] = bn;
    }
    tile_product<K>(A, Wt, tc, tn, acc);
#pragma unroll
    for (int n = 0; n < 4; ++n)
      *reinterpret_cast<float4*>(out + (tn + 16 * n) * TR_LD + 4 * tc) =
          make_float4(tanhf(acc[0][n]), tanhf(acc[1][n]), tanhf(acc[2][n]), tanhf(acc[3][n]));
  }
}

// deltas of the layer below: out[i][c] = (1 - A[i][c]^2) sum_j W[j][i] D[j][c]
__device__ __forceinline__ void layer_delta(const float* D, const float* W, const float* A, float* out) {
  if (threadIdx.x < 128) {
    const int tn = threadIdx.x & 15, tc = threadIdx.x >> 4;
    float acc[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c][n] = 0.f;
    tile_product<64>(D, W, tc, tn, acc);
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int o = (tn + 16 * n) * TR_LD + 4 * tc;
      const float4 a = *reinterpret_cast<const float4*>(A + o);
      *reinterpret_cast<float4*>(out + o) =
          make_float4(acc[0][n] * (1.f - a.x * a.x), acc[1][n] * (1.f - a.y * a.y), acc[2][n] * (1.f - a.z * a.z),
                      acc[3][n] * (1.f - a.w * a.w));
    }
  }
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float s) {
  s = fmaf(a.x, b.x, s);
  s = fmaf(a.y, b.y, s);
  s = fmaf(a.z, b.z, s);
  return fmaf(a.w, b.w, s);
}

__device__ __forceinline__ float4 row4(const float* M, int row, int c) {
  return *reinterpret_cast<const float4*>(M + row * TR_LD + c);
}

// g[m][n] += sum_c D[tm + 16 m][c] A[tn + 16 n][c] of a 64 x 64 layer
__device__ __forceinline__ void weight_gradient(const float* D, const float* A, float (*g)[4]) {
  const int tn = threadIdx.x & 15, tm = threadIdx.x >> 4;
#pragma unroll 2
  for (int c = 0; c < TR_TILE; c += 4) {
    float4 d[4], a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      d[k] = row4(D, tm + 16 * k, c);
      a[k] = row4(A, tn + 16 * k, c);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n) g[m][n] = dot4(d[m], a[n], g[m][n]);
  }
}

__device__ __forceinline__ float row_sum(const float* M, int row, float s) {
#pragma unroll
  for (int c = 0; c < TR_TILE; c += 4) {
    const float4 v = row4(M, row, c);
    s += (v.x + v.y) + (v.z + v.w);
  }
  return s;
}

__global__ void __launch_bounds__(TR_THREADS) k_mlp_train(const uint16_t* __restrict__ wbf,
                                                          const float* __restrict__ X, const float* __restrict__ Y,
                                                          const float* __restrict__ wc,
                                                          const int32_t* __restrict__ count, int ncells,
                                                          float* __restrict__ partial,
                                                          double* __restrict__ part_loss) {
  extern __shared__ __align__(16) float sm[];
  __shared__ double red[TR_THREADS / 32];
  const int tid = threadIdx.x;
  // weights, widened
  for (int q = tid; q < 12 * 64; q += TR_THREADS) {
    const int j = q / 12, i = q % 12;
    sm[TR_W0T + i * 64 + perm64(j)] = bf16_to_f(wbf[poff_w(0) + q]);
  }
  for (int q = tid; q < 64 * 64; q += TR_THREADS) {
    const int j = q >> 6, i = q & 63;
    const float w1 = bf16_to_f(wbf[poff_w(1) + q]), w2 = bf16_to_f(wbf[poff_w(2) + q]);
    sm[TR_W1T + i * 64 + perm64(j)] = w1;
    sm[TR_W2T + i * 64 + perm64(j)] = w2;
    sm[TR_W1 + j * 64 + perm64(i)] = w1;
    sm[TR_W2 + j * 64 + perm64(i)] = w2;
  }
  for (int q = tid; q < 5 * 64; q += TR_THREADS) sm[TR_W3 + q] = bf16_to_f(wbf[poff_w(3) + q]);
  if (tid < 64) {
    sm[TR_B + tid] = bf16_to_f(wbf[poff_b(0) + tid]);
    sm[TR_B + 64 + tid] = bf16_to_f(wbf[poff_b(1) + tid]);
    sm[TR_B + 128 + tid] = bf16_to_f(wbf[poff_b(2) + tid]);
    if (tid < 5) sm[TR_B + 192 + tid] = bf16_to_f(wbf[poff_b(3) + tid]);
  }
  const int tn = tid & 15, tm = tid >> 4;
  float g0[4] = {0.f, 0.f, 0.f, 0.f}, g1[4][4], g2[4][4], g3[2] = {0.f, 0.f};
  float gb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int n = 0; n < 4; ++n) g1[m][n] = g2[m][n] = 0.f;
  const float inv_n = 1.f / (5.f * (float)max(*count, 1));
  double lsum = 0.0;
  __syncthreads();
  const int ntiles = (ncells + TR_TILE - 1) / TR_TILE;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int c0 = t * TR_TILE;
    for (int q = tid; q < TR_TILE * 12; q += TR_THREADS) {
      const int c = q / 12, i = q % 12;
      sm[TR_A0 + i * TR_LD + c] = (c0 + c < ncells) ? X[(size_t)c0 * 12 + q] : 0.f;
    }
    if (tid < TR_TILE) sm[TR_WT + tid] = (c0 + tid < ncells) ? wc[c0 + tid] : 0.f;
    __syncthreads();
    layer_forward<12>(sm + TR_A0, sm + TR_W0T, sm + TR_B, sm + TR_A1);
    __syncthreads();
    layer_forward<64>(sm + TR_A1, sm + TR_W1T, sm + TR_B + 64, sm + TR_A2);
    __syncthreads();
    layer_forward<64>(sm + TR_A2, sm + TR_W2T, sm + TR_B + 128, sm + TR_A3);
    __syncthreads();
    // output layer and the deltas of the mean squared error over the weighted
    // cells: a thread per (output, cell)
    if (tid < 5 * TR_TILE) {
      const int j = tid / TR_TILE, c = tid % TR_TILE;
      float z[4] = {sm[TR_B + 192 + j], 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int i = 0; i < 64; i += 4)
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = fmaf(sm[TR_W3 + j * 64 + i + k], sm[TR_A3 + (i + k) * TR_LD + c], z[k]);
      const float y = (c0 + c < ncells) ? Y[(size_t)(c0 + c) * 5 + j] : 0.f;
      const float r = ((z[0] + z[1]) + (z[2] + z[3]) - y) * sm[TR_WT + c];
      lsum += (double)r * (double)r;
      sm[TR_D3 + j * TR_LD + c] = 2.f * r * inv_n;
    }
    __syncthreads();
    // layer 3: gradient, bias, deltas of layer 2's output
    {
      const int j = tid >> 6, i = tid & 63;
#pragma unroll
      for (int c = 0; c < TR_TILE; c += 4) {
        const float4 a = row4(sm + TR_A3, i, c);
        g3[0] = dot4(row4(sm + TR_D3, j, c), a, g3[0]);
        if (tid < 64) g3[1] = dot4(row4(sm + TR_D3, 4, c), a, g3[1]);
      }
      if (tid < 5) gb[3] = row_sum(sm + TR_D3, tid, gb[3]);
      for (int q = tid; q < 64 * (TR_TILE / 4); q += TR_THREADS) {
        const int n = q >> 3, c = 4 * (q & 7);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const float w = sm[TR_W3 + k * 64 + n];
          const float4 d = row4(sm + TR_D3, k, c);
          s.x = fmaf(d.x, w, s.x);
          s.y = fmaf(d.y, w, s.y);
          s.z = fmaf(d.z, w, s.z);
          s.w = fmaf(d.w, w, s.w);
        }
        const float4 a = row4(sm + TR_A3, n, c);
        *reinterpret_cast<float4*>(sm + TR_DA + n * TR_LD + c) =
            make_float4(s.x * (1.f - a.x * a.x), s.y * (1.f - a.y * a.y), s.z * (1.f - a.z * a.z),
                        s.w * (1.f - a.w * a.w));
      }
    }
    __syncthreads();
    weight_gradient(sm + TR_DA, sm + TR_A2, g2);
    if (tid < 64) gb[2] = row_sum(sm + TR_DA, tid, gb[2]);
    layer_delta(sm + TR_DA, sm + TR_W2, sm + TR_A2, sm + TR_DB);
    __syncthreads();
    weight_gradient(sm + TR_DB, sm + TR_A1, g1);
    if (tid < 64) gb[1] = row_sum(sm + TR_DB, tid, gb[1]);
    layer_delta(sm + TR_DB, sm + TR_W1, sm + TR_A1, sm + TR_DA);
    __syncthreads();
    if (tn < 12) {
#pragma unroll
      for (int c = 0; c < TR_TILE; c += 4) {
        const float4 a = row4(sm + TR_A0, tn, c);
#pragma unroll
        for (int m = 0; m < 4; ++m) g0[m] = dot4(row4(sm + TR_DA, tm + 16 * m, c), a, g0[m]);
      }
    }
    if (tid < 64) gb[0] = row_sum(sm + TR_DA, tid, gb[0]);
    __syncthreads();
  }
  float* out = partial + (size_t)blockIdx.x * MLP_NPARAM;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (tn < 12) out[poff_w(0) + (tm + 16 * m) * 12 + tn] = g0[m];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      out[poff_w(1) + (tm + 16 * m) * 64 + tn + 16 * n] = g1[m][n];
      out[poff_w(2) + (tm + 16 * m) * 64 + tn + 16 * n] = g2[m][n];
    }
  }
  out[poff_w(3) + tid] = g3[0];
  if (tid < 64) {
    out[poff_w(3) + 256 + tid] = g3[1];
    out[poff_b(0) + tid] = gb[0];
    out[poff_b(1) + tid] = gb[1];
    out[poff_b(2) + tid] = gb[2];
    if (tid < 5) out[poff_b(3) + tid] = gb[3];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if ((tid & 31) == 0) red[tid >> 5] = lsum;
  __syncthreads();
  if (tid == 0) {
    double l = 0.0;
    for (int k = 0; k < TR_THREADS / 32; ++k) l += red[k];
    part_loss[blockIdx.x] = l;
  }
}

// The CTAs' gradient sums in a fixed order (32 parameters per CTA, eight
// threads each on every eighth sum); the loss; with ADAM the step.  A thread
// per parameter over all sums took 24 us at 12 800 cells, this 5 us.
template <bool ADAM>
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ partial,
                                                    const double* __restrict__ part_loss, int nblk,
                                                    const int32_t* __restrict__ count, float* __restrict__ grad,
                                                    double* __restrict__ scal, float* __restrict__ theta,
                                                    float* __restrict__ m, float* __restrict__ v,
                                                    uint16_t* __restrict__ wbf, float c1, float c2, float lr) {
  __shared__ float s[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int q = blockIdx.x * 32 + lane;
  float a = 0.f;
  if (q < MLP_NPARAM) {
#pragma unroll 4
    for (int b = w; b < nblk; b += 8) a += partial[(size_t)b * MLP_NPARAM + q];
  }
  s[w][lane] = a;
  __syncthreads();
  if (w == 0 && q < MLP_NPARAM) {
    float gq = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) gq += s[k][lane];
    grad[q] = gq;
    if (ADAM) {
      const float mq = 0.9f * m[q] + 0.1f * gq;
      const float vq = 0.999f * v[q] + 0.001f * gq * gq;
      m[q] = mq;
      v[q] = vq;
      const float th = theta[q] - lr * (mq / c1) / (sqrtf(vq / c2) + 1e-8f);
      theta[q] = th;
      wbf[q] = __bfloat16_as_ushort(__float2bfloat16_rn(th));
    }
  }
  if (blockIdx.x == 0 && w == 1) {
    double l = 0.0;
    for (int b = lane; b < nblk; b += 32) l += part_loss[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) scal[0] = l / (5.0 * (double)max(*count, 1));
  }
}

__global__ void k_mlp_bf16(const float* __restrict__ theta, uint16_t* __restrict__ wbf) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < MLP_NPARAM) wbf[q] = __bfloat16_as_ushort(__float2bfloat16_rn(theta[q]));
}

// ---------------------------------------------------------------------------
// Inference on the tensor cores: every layer is one product of the tile's
// activations (16 cells x K, bfloat16) with the layer's weights (K x N,
// bfloat16) accumulated in FP32 by mma.sync m16n8k16; bias and tanh in FP32,
// and the result, rounded to bfloat16, is already laid out as the next
// layer's A operand (the accumulator fragment of two adjacent 8-column tiles
// is the operand fragment of one 16-column k-slice).  A warp takes 16 cells
// at a time; the CTA's warps share the weights, staged in shared memory in
// rows padded so that the fragment loads of a warp hit 32 distinct banks.
// 160 000 cells: 48 us with 4 warps a CTA and two CTAs an SM, 42 us with 8 and
// three (the latency of a tile's chain of products bounds it).
// ---------------------------------------------------------------------------
constexpr int TC_WARPS = 8;
constexpr int TC_GRID = 3 * 152;  // largest grid: 24 warps an SM share three copies of the weights
constexpr int TC_K0 = 16;        // the 12 inputs padded to one k-slice
constexpr int TC_LD0 = 12;       // words per row of the padded layer-0 weights (8 used)
constexpr int TC_LD = 36;        // words per row of the 64-input weights (32 used)
constexpr int TC_W0 = 64 * TC_LD0, TC_W1 = 64 * TC_LD, TC_W3 = 8 * TC_LD;
constexpr int TC_WORDS = TC_W0 + 2 * TC_W1 + TC_W3;        // bfloat16 pairs
constexpr int TC_BIAS = 64 * 3 + 8;                         // FP32 biases
inline size_t tc_smem_bytes() { return sizeof(uint32_t) * (size_t)TC_WORDS + sizeof(float) * TC_BIAS; }

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // .x (low half) = lo
  return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One layer for the warp's 16 cells: a[KT][4] operand fragments (KT
// k-slices of 16 inputs) times the NT 8-column tiles of the weights W
// (rows of ld words, row n = output n), plus bias; d[NT][4] accumulators.
template <int KT, int NT>
__device__ __forceinline__ void tc_layer(const uint32_t (*a)[4], const uint32_t* W, int ld, const float* bias,
                                         float (*d)[4], int g, int t) {
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    const float b0 = bias[8 * j + 2 * t], b1 = bias[8 * j + 2 * t + 1];
    d[j][0] = b0;
    d[j][1] = b1;
    d[j][2] = b0;
    d[j][3] = b1;
    const uint32_t* wr = W + (8 * j + g) * ld;
#pragma unroll
    for (int k = 0; k < KT; ++k) mma16816(d[j], a[k], wr[8 * k + t], wr[8 * k + 4 + t]);
  }
}

// tanh of the accumulators of 2 KT tiles, packed as KT operand fragments
template <int KT>
__device__ __forceinline__ void tc_to_operand(float (*d)[4], uint32_t (*a)[4]) {
#pragma unroll
  for (int k = 0; k < KT; ++k) {
    a[k][0] = bf16x2(tanhf(d[2 * k][0]), tanhf(d[2 * k][1]));
    a[k][1] = bf16x2(tanhf(d[2 * k][2]), tanhf(d[2 * k][3]));
    a[k][2] = bf16x2(tanhf(d[2 * k + 1][0]), tanhf(d[2 * k + 1][1]));
    a[k][3] = bf16x2(tanhf(d[2 * k + 1][2]), tanhf(d[2 * k + 1][3]));
  }
}

__global__ void __launch_bounds__(TC_WARPS * 32) k_mlp_fwd_tc(const uint16_t* __restrict__ wbf,
                                                              const float* __restrict__ theta,
                                                              const float* __restrict__ X, int ncells,
                                                              float* __restrict__ out) {
  extern __shared__ __align__(16) uint32_t smw[];
  uint32_t* W0 = smw;
  uint32_t* W1 = W0 + TC_W0;
  uint32_t* W2 = W1 + TC_W1;
  uint32_t* W3 = W2 + TC_W1;
  float* bs = reinterpret_cast<float*>(W3 + TC_W3);
  // stage the bfloat16 weights as pairs along the input index (zero padded)
  auto pair = [&](int k, int n, int i) -> uint32_t {  // inputs i, i + 1 of output n of layer k
    const int ni = nin(k);
    if (n >= nout(k) || i >= ni) return 0u;
    const uint32_t lo = wbf[poff_w(k) + n * ni + i];
    const uint32_t hi = (i + 1 < ni) ? wbf[poff_w(k) + n * ni + i + 1] : 0u;
    return lo | (hi << 16);
  };
  for (int q = threadIdx.x; q < 64 * TC_LD0; q += blockDim.x) {
    const int n = q / TC_LD0, w = q % TC_LD0;
    W0[q] = (w < TC_K0 / 2) ? pair(0, n, 2 * w) : 0u;
  }
  for (int q = threadIdx.x; q < 64 * TC_LD; q += blockDim.x) {
    const int n = q / TC_LD, w = q % TC_LD;
    W1[q] = (w < 32) ? pair(1, n, 2 * w) : 0u;
    W2[q] = (w < 32) ? pair(2, n, 2 * w) : 0u;
  }
  for (int q = threadIdx.x; q < 8 * TC_LD; q += blockDim.x) {
    const int n = q / TC_LD, w = q % TC_LD;
    W3[q] = (w < 32) ? pair(3, n, 2 * w) : 0u;
  }
  for (int q = threadIdx.x; q < TC_BIAS; q += blockDim.x) {
    const int k = q / 64, j = q % 64;
    bs[q] = (k < 3) ? theta[poff_b(k) + j] : (j < 5 ? theta[poff_b(3) + j] : 0.f);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int ntiles = (ncells + 15) / 16;
  for (int tile = blockIdx.x * TC_WARPS + warp; tile < ntiles; tile += gridDim.x * TC_WARPS) {
    const int c0 = tile * 16;
    const int ca = c0 + g, cb = c0 + g + 8;
    auto xin = [&](int c, int i) { return (c < ncells && i < 12) ? X[(size_t)c * 12 + i] : 0.f; };
    uint32_t a0[1][4];
    a0[0][0] = bf16x2(xin(ca, 2 * t), xin(ca, 2 * t + 1));
    a0[0][1] = bf16x2(xin(cb, 2 * t), xin(cb, 2 * t + 1));
    a0[0][2] = bf16x2(xin(ca, 2 * t + 8), xin(ca, 2 * t + 9));
    a0[0][3] = bf16x2(xin(cb, 2 * t + 8), xin(cb, 2 * t + 9));
    float d[8][4];
    uint32_t a[4][4];
    tc_layer<1, 8>(a0, W0, TC_LD0, bs, d, g, t);
    tc_to_operand<4>(d, a);
    tc_layer<4, 8>(a, W1, TC_LD, bs + 64, d, g, t);
    tc_to_operand<4>(d, a);
    tc_layer<4, 8>(a, W2, TC_LD, bs + 128, d, g, t);
    tc_to_operand<4>(d, a);
    float o[1][4];
    tc_layer<4, 1>(a, W3, TC_LD, bs + 192, o, g, t);
    // row g: outputs 2t, 2t + 1 in o[0][0..1]; row g + 8 in o[0][2..3]
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = h ? cb : ca;
      if (c >= ncells) continue;
      if (2 * t < 5) out[(size_t)c * 5 + 2 * t] = o[0][2 * h];
      if (2 * t + 1 < 5) out[(size_t)c * 5 + 2 * t + 1] = o[0][2 * h + 1];
    }
  }
}

// The judge's statistics: every cell of the network (w = 1, finite
// outputs) adds its residual r = network - DSMC (5 normalised outputs), r^2
// and the DSMC terms Y to its group's sums, and 1 to its count (FP64):
// JACC doubles per group.  Sixteen lanes take one cell, a lane per sum, so
// that a cell's additions reach L2 as one 128-byte row (160 000 cells, 200
// groups: 46 us with 16 additions per thread, 28 us).
constexpr int JACC = 16;
__global__ void __launch_bounds__(256) k_mlp_judge_acc(int ncells, const float* __restrict__ out,
                                const float* __restrict__ Y,
                                const float* __restrict__ w, const int32_t* __restrict__ group,
                                double* __restrict__ jacc) {
  const int k = threadIdx.x & 15;
  const int stride = (gridDim.x * blockDim.x) >> 4;
  for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 4; c < ncells; c += stride) {
    if (w[c] == 0.f) continue;
    const float* o = out + (size_t)c * 5;
    const float* yc = Y + (size_t)c * 5;
    bool fin = true;
    for (int q = 0; q < 5; ++q) fin = fin && isfinite(o[q]);
    if (!fin) continue;
    double v = 1.0;  // k = 10: the count
    if (k < 10) {
      const int q = k < 5 ? k : k - 5;
      const double r = (double)o[q] - (double)yc[q];
      v = k < 5 ? r : r * r;
    } else if (k > 10) {
      v = (double)yc[k - 11];
    }
    double* a = jacc + (size_t)(group ? group[c] : c) * JACC + k;
    if (group) atomicAdd(a, v);
    else *a += v;
  }
}

// true if the group's residuals show the network's bias to be small: at
// least min_samples of them and, for every output, |mean r| + z SE(r) <=
// rel |mean Y| (an equivalence test: the bias is bounded, with z standard
// errors of confidence, by the fraction rel of the DSMC terms themselves)
__device__ __forceinline__ bool judge_pass(const double* a, double z, int min_samples, double rel) {
  const double n = a[10];
  if (n < (double)min_samples) return false;
  for (int k = 0; k < 5; ++k) {
    const double m = a[k] / n;
    const double var = fmax(a[5 + k] / n - m * m, 0.0) * n / (n - 1.0);
    if (fabs(m) + z * sqrt(var / n) > rel * fabs(a[11 + k] / n)) return false;
  }
  return true;
}

// the verdict of every group, once (a group without samples fails at once)
__global__ void k_mlp_verdict(int ngroups, const double* __restrict__ jacc, double z, int min_samples, double rel,
                              uint8_t* __restrict__ pass) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < ngroups) pass[g] = judge_pass(jacc + (size_t)g * JACC, z, min_samples, rel) ? 1 : 0;
}

// HoT for the synthetic equations and the judge sums (network against DSMC);
// hot and hot_out may be the same array (each thread reads its cell first).
// With pass (the groups' verdicts) a network cell keeps the DSMC HoT unless
// its group passes.  The three judge sums are reduced over the CTA before
// they are added (one address each: 160 000 cells took 488 us with an
// addition per cell, 16 us with one per CTA).
__global__ void __launch_bounds__(256) k_mlp_hot(int ncells, const float* __restrict__ out,
                          const float* __restrict__ Y,
                          const float* __restrict__ S, const float* __restrict__ w, const double* hot,
                          double* hot_out, double* __restrict__ scal, const int32_t* __restrict__ group,
                          const uint8_t* __restrict__ pass) {
  __shared__ double s_j[8];
  __shared__ int s_c[8], s_n[8];
  double jsum = 0.0;
  int jcnt = 0, nnet = 0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) {
    double h[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) h[k] = hot[(size_t)c * 12 + k];
    const float* o = out + (size_t)c * 5;
    bool fin = true;
    for (int k = 0; k < 5; ++k) fin = fin && isfinite(o[k]);
    if (w[c] != 0.f && fin) {
      for (int k = 0; k < 5; ++k) {
        const double r = (double)o[k] - (double)Y[(size_t)c * 5 + k];
        jsum += r * r;
      }
      jcnt += 5;
      if (!pass || pass[group ? group[c] : c]) {
        nnet += 1;
        const double p = S[(size_t)c * 4], ps = S[(size_t)c * 4 + 1];
        const double ex = S[(size_t)c * 4 + 2], ey = S[(size_t)c * 4 + 3];
        h[0] = (double)o[0] * p;
        h[3] = (double)o[1] * p;
        h[1] = (double)o[2] * p;
        const int base[2] = {6, 9};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const double along = h[base[r]] * ex + h[base[r] + 1] * ey;
          const double nw = (double)o[3 + r] * ps;
          h[base[r]] += (nw - along) * ex;
          h[base[r] + 1] += (nw - along) * ey;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) hot_out[(size_t)c * 12 + k] = h[k];
  }
  for (int o = 16; o > 0; o >>= 1) jsum += __shfl_xor_sync(0xffffffffu, jsum, o);
  jcnt = __reduce_add_sync(0xffffffffu, jcnt);
  nnet = __reduce_add_sync(0xffffffffu, nnet);
  if ((threadIdx.x & 31) == 0) {
    s_j[threadIdx.x >> 5] = jsum;
    s_c[threadIdx.x >> 5] = jcnt;
    s_n[threadIdx.x >> 5] = nnet;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) {
      jsum += s_j[k];
      jcnt += s_c[k];
      nnet += s_n[k];
    }
    if (jcnt > 0) {
      atomicAdd(scal + 2, jsum);
      atomicAdd(scal + 3, (double)jcnt);
    }
    if (nnet > 0) atomicAdd(scal + 4, (double)nnet);
  }
}

inline int blocks_for(int n, int t) { return (n + t - 1) / t; }

int launch_train(const Mlp& m, int ncells, cudaStream_t st) {
  cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)train_smem_bytes());
  const int ntiles = blocks_for(ncells, TR_TILE);
  const int grid = ntiles < MLP_GRID ? ntiles : MLP_GRID;
  k_mlp_train<<<grid, TR_THREADS, train_smem_bytes(), st>>>(m.wbf, m.X, m.Y, m.w, m.count, ncells, m.partial,
                                                            m.part_loss);
  return grid;
}

}  // namespace

void mlp_prepare(const Mlp& m, const CellParams* cp, const int32_t* cell_case, const int32_t* cell0, int ncells,
                 const double* fields, const double* hot, const double* kngll, const uint8_t* mask,
                 cudaStream_t st) {
  cudaMemsetAsync(m.count, 0, sizeof(int32_t), st);
  k_mlp_data<<<blocks_for(ncells, 128), 128, 0, st>>>(cp, cell_case, cell0, ncells, fields, hot, kngll, mask, m.X,
                                                       m.Y, m.S, m.w, m.count);
}

void mlp_grad(const Mlp& m, int ncells, cudaStream_t st) {
  const int grid = launch_train(m, ncells, st);
  k_mlp_reduce<false><<<blocks_for(MLP_NPARAM, 32), 256, 0, st>>>(m.partial, m.part_loss, grid, m.count, m.grad, m.scal,
                                                                  m.theta, m.m, m.v, m.wbf, 1.f, 1.f, 0.f);
}

void mlp_train_step(const Mlp& m, int ncells, int t, double lr, cudaStream_t st) {
  const int grid = launch_train(m, ncells, st);
  const float c1 = (float)(1.0 - pow(0.9, t)), c2 = (float)(1.0 - pow(0.999, t));
  k_mlp_reduce<true><<<blocks_for(MLP_NPARAM, 32), 256, 0, st>>>(m.partial, m.part_loss, grid, m.count, m.grad, m.scal,
                                                                 m.theta, m.m, m.v, m.wbf, c1, c2, (float)lr);
}

void mlp_to_bf16(const Mlp& m, cudaStream_t st) {
  k_mlp_bf16<<<blocks_for(MLP_NPARAM, 256), 256, 0, st>>>(m.theta, m.wbf);
}

void mlp_apply(const Mlp& m, int ncells, const double* hot, double* hot_out, cudaStream_t st,
               const int32_t* group, double z, int min_samples, double rel) {
  // inference on the tensor cores (bfloat16 weights and activations, FP32 sums)
  const int tiles = blocks_for(ncells, 16);
  const int grid = blocks_for(tiles, TC_WARPS) < TC_GRID ? blocks_for(tiles, TC_WARPS) : TC_GRID;
  k_mlp_fwd_tc<<<grid, TC_WARPS * 32, tc_smem_bytes(), st>>>(m.wbf, m.theta, m.X, ncells, m.out);
  cudaMemsetAsync(m.scal + 2, 0, 3 * sizeof(double), st);
  const int hb = blocks_for(ncells, 256) < 1024 ? blocks_for(ncells, 256) : 1024;
  if (z > 0.0) {
    const int jb = blocks_for(ncells, 16);
    k_mlp_judge_acc<<<jb < 152 * 8 ? jb : 152 * 8, 256, 0, st>>>(ncells, m.out, m.Y, m.w, group, m.jacc);
    k_mlp_verdict<<<blocks_for(ncells, 256), 256, 0, st>>>(ncells, m.jacc, z, min_samples, rel, m.pass);
  }
  k_mlp_hot<<<hb, 256, 0, st>>>(ncells, m.out, m.Y, m.S, m.w, hot, hot_out, m.scal, group, z > 0.0 ? m.pass : nullptr);
}

}  // namespace dsmc
