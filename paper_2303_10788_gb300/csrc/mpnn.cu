// Learned cut-set scorer: a message-passing network over the qubit
// interaction graph of a circuit with one candidate cut set applied, trained
// on measured evaluation + recombination times (its choices are judged by the
// greedy search's cost estimate, which remains the fallback).
//
//   h0      = relu(W_in x_v + b_in)                          (8 -> 64)
//   h_{l+1} = relu(Ws_l h_l + Wn_l (A h_l)_v + b_l)           l = 0, 1, 2
//   r_g     = mean_{v in g} h3_v
//   z_g     = relu(W_r1 [r_g, glob_g] + b_r1)                 (72 -> 64)
//   y_g     = w_r2 . z_g + b_r2                               predicted log time
//
// A is the degree-normalised adjacency (A = D^-1 Adj).  Weights are used in
// FP16 (rounded from an FP32 master copy that Adam updates); activations,
// gradients and accumulations are FP32.  Every step is a kernel below.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "abi_guard.hpp"
#include "kernels.cuh"

namespace ccs {
namespace mp {

constexpr int kIn = 8, kGlob = 8, kH = 64, kLayers = 3, kR = kH + kGlob;

// flat parameter layout
constexpr int oWin = 0, oBin = oWin + kH * kIn;
constexpr int oLayer = oBin + kH;
constexpr int kLayerSize = 2 * kH * kH + kH;   // Ws, Wn, b
constexpr int oWr1 = oLayer + kLayers * kLayerSize, oBr1 = oWr1 + kH * kR;
constexpr int oWr2 = oBr1 + kH, oBr2 = oWr2 + kH;
constexpr int kParams = oBr2 + 1;

// Tiling.  The nodes are taken in tiles of kTile rows by CTAs of 256 threads;
// a thread owns a 4 x 4 block of a 64 x 64 product, with both operands in
// shared memory as FP32 (8 LDS.128 per 64 FMA).  A batch of 64 graphs (about
// 14 k nodes) is 225 tiles, one wave of two CTAs per SM; the products are
// 0.7 GFLOP forward, so a layer is bound by FP32 issue and by launch latency,
// not by memory (the activations are 3.7 MB and stay in L2).  Loss and
// gradient of such a batch from host arrays: 9.11 ms with one thread per
// output, serial weight-gradient sums and an allocation per array, 0.29 ms so.
constexpr int kTile = 64, kLd = kH + 4;   // row stride of a node tile: rows 4 apart on other banks

// W (64 x 64, [o][k], FP16) transposed into shared FP32 [k][o]: a lane takes
// eight k of its own row o in one 16-byte load, so the stores are conflict-free.
__device__ __forceinline__ void stage_w_t(const half* __restrict__ W, float* __restrict__ dst) {
  for (int t = threadIdx.x; t < kH * (kH / 8); t += blockDim.x) {
    const int o = t % kH, k0 = (t / kH) * 8;
    const uint4 q = *reinterpret_cast<const uint4*>(W + o * kH + k0);
    const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = __half22float2(*reinterpret_cast<const half2*>(&w[j]));
      dst[(k0 + 2 * j) * kH + o] = f.x;
      dst[(k0 + 2 * j + 1) * kH + o] = f.y;
    }
  }
}

// acc[i][j] += sum_k X[4 ty + i][k] W[k][4 tx + j] over 64 k, k ascending
// (tx = thread % 16, ty = thread / 16).
__device__ __forceinline__ void mm64(const float* __restrict__ X, const float* __restrict__ W, int ldw,
                                     float (&acc)[4][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const float* xr = X + 4 * ty * kLd;
  const float* wr = W + 4 * tx;
#pragma unroll 4
  for (int k = 0; k < kH; k += 4) {
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4*>(xr + i * kLd + k);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 w = *reinterpret_cast<const float4*>(wr + (k + u) * ldw);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float xv = u == 0 ? x[i].x : u == 1 ? x[i].y : u == 2 ? x[i].z : x[i].w;
        acc[i][0] = fmaf(xv, w.x, acc[i][0]);
        acc[i][1] = fmaf(xv, w.y, acc[i][1]);
        acc[i][2] = fmaf(xv, w.z, acc[i][2]);
        acc[i][3] = fmaf(xv, w.w, acc[i][3]);
      }
    }
  }
}

// Rows [r0, r0 + kTile) of X (rows x 64) into a tile; rows past the end are zero.
__device__ __forceinline__ void load_tile(const float* __restrict__ X, int r0, int rows, float* __restrict__ dst) {
  for (int t = threadIdx.x; t < kTile * (kH / 4); t += blockDim.x) {
    const int r = t / (kH / 4), c = (t % (kH / 4)) * 4;
    const float4 v = r0 + r < rows ? *reinterpret_cast<const float4*>(X + (long long)(r0 + r) * kH + c)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(dst + r * kLd + c) = v;
  }
}

// One row of A X (CSR) at four columns, edges in order.
__device__ __forceinline__ float4 spmm4(const int* __restrict__ rowptr, const int* __restrict__ col,
                                        const float* __restrict__ val, const float* __restrict__ X, int row, int c) {
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int e = rowptr[row], e1 = rowptr[row + 1]; e < e1; ++e) {
    const float w = val[e];
    const float4 x = *reinterpret_cast<const float4*>(X + (long long)col[e] * kH + c);
    a.x = fmaf(w, x.x, a.x);
    a.y = fmaf(w, x.y, a.y);
    a.z = fmaf(w, x.z, a.z);
    a.w = fmaf(w, x.w, a.w);
  }
  return a;
}

// H0 = relu(X W_in^T + b_in): one thread per (node, output).
__global__ void __launch_bounds__(256) in_fwd(const float* __restrict__ X, const half* __restrict__ W,
                                              const half* __restrict__ b, int rows, float* __restrict__ Y) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)rows * kH) return;
  const int r = (int)(t / kH), o = (int)(t % kH);
  float acc = __half2float(b[o]);
#pragma unroll
  for (int i = 0; i < kIn; ++i) acc = fmaf(X[(long long)r * kIn + i], __half2float(W[o * kIn + i]), acc);
  Y[t] = fmaxf(acc, 0.f);
}

// One layer, one tile of nodes: AH = A H gathered into the tile (kept in
// AHout for the backward pass, if given), then
// Hout = relu(H Ws^T + AH Wn^T + b).  L points at Ws, Wn, b.
constexpr int kFwdSmem = (2 * kTile * kLd + 2 * kH * kH) * (int)sizeof(float);
__global__ void __launch_bounds__(256, 2) layer_fwd(const int* __restrict__ rowptr, const int* __restrict__ col,
                                                    const float* __restrict__ val, const float* __restrict__ H,
                                                    const half* __restrict__ L, int rows, float* __restrict__ AHout,
                                                    float* __restrict__ Hout) {
  extern __shared__ __align__(16) float sm[];
  float* Hs = sm;
  float* As = Hs + kTile * kLd;
  float* W1 = As + kTile * kLd;
  float* W2 = W1 + kH * kH;
  const int r0 = blockIdx.x * kTile;
  stage_w_t(L, W1);
  stage_w_t(L + kH * kH, W2);
  load_tile(H, r0, rows, Hs);
  for (int t = threadIdx.x; t < kTile * (kH / 4); t += blockDim.x) {
    const int r = t / (kH / 4), c = (t % (kH / 4)) * 4;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r0 + r < rows) {
      a = spmm4(rowptr, col, val, H, r0 + r, c);
      if (AHout) *reinterpret_cast<float4*>(AHout + (long long)(r0 + r) * kH + c) = a;
    }
    *reinterpret_cast<float4*>(As + r * kLd + c) = a;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float bj = __half2float(L[2 * kH * kH + 4 * tx + j]);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][j] = bj;
  }
  mm64(Hs, W1, kH, acc);
  mm64(As, W2, kH, acc);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + 4 * ty + i;
    if (r < rows)
      *reinterpret_cast<float4*>(Hout + (long long)r * kH + 4 * tx) =
          make_float4(fmaxf(acc[i][0], 0.f), fmaxf(acc[i][1], 0.f), fmaxf(acc[i][2], 0.f), fmaxf(acc[i][3], 0.f));
  }
}

// One graph per CTA: the mean of its nodes' rows (16 row groups, four columns
// a thread, the groups added in a fixed order), the head's hidden layer and
// the prediction; with a target also its share of the backward pass, which
// needs no other graph: dy = 2 (y - t) / G, dZ, and the gradient every one of
// its nodes receives, dR / n.
__global__ void __launch_bounds__(256) readout(const int* __restrict__ goff, const float* __restrict__ H,
                                               const float* __restrict__ glob, const half* __restrict__ W1,
                                               const half* __restrict__ b1, const half* __restrict__ w2,
                                               const half* __restrict__ b2, int graphs, float* __restrict__ RG,
                                               float* __restrict__ Z, float* __restrict__ y,
                                               const float* __restrict__ tgt, float* __restrict__ dZ,
                                               float* __restrict__ dnode) {
  __shared__ __align__(16) float part[16][kH];
  __shared__ float rg[kR], zs[kH], dz[kH];
  __shared__ float s_y;
  const int g = blockIdx.x, tid = threadIdx.x, a = goff[g], b = goff[g + 1];
  const int cg = (tid & 15) * 4, grp = tid >> 4;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int v = a + grp; v < b; v += 16) {
    const float4 h = *reinterpret_cast<const float4*>(H + (long long)v * kH + cg);
    s.x += h.x; s.y += h.y; s.z += h.z; s.w += h.w;
  }
  *reinterpret_cast<float4*>(&part[grp][cg]) = s;
  __syncthreads();
  if (tid < kH) {
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) acc += part[i][tid];
    rg[tid] = b > a ? acc / (float)(b - a) : 0.f;
  } else if (tid < kR) {
    rg[tid] = glob[g * kGlob + (tid - kH)];
  }
  __syncthreads();
  if (RG && tid < kR) RG[g * kR + tid] = rg[tid];
  {   // Z: four lanes per output, 18 terms each
    const int o = tid >> 2, q = tid & 3;
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kR / 4; ++i) acc = fmaf(rg[4 * i + q], __half2float(W1[o * kR + 4 * i + q]), acc);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (q == 0) {
      zs[o] = fmaxf(acc + __half2float(b1[o]), 0.f);
      if (Z) Z[g * kH + o] = zs[o];
    }
  }
  __syncthreads();
  if (tid < 32) {
    float acc = zs[tid] * __half2float(w2[tid]) + zs[tid + 32] * __half2float(w2[tid + 32]);
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (tid == 0) {
      s_y = acc + __half2float(b2[0]);
      y[g] = s_y;
    }
  }
  if (!tgt) return;
  __syncthreads();
  const float dy = 2.f * (s_y - tgt[g]) / (float)graphs;
  if (tid < kH) {
    dz[tid] = zs[tid] > 0.f ? dy * __half2float(w2[tid]) : 0.f;
    dZ[g * kH + tid] = dz[tid];
  }
  __syncthreads();
  if (tid < kH) {
    float acc = 0.f;
#pragma unroll 8
    for (int o = 0; o < kH; ++o) acc = fmaf(dz[o], __half2float(W1[o * kR + tid]), acc);
    dnode[g * kH + tid] = b > a ? acc / (float)(b - a) : 0.f;
  }
}

// --- backward -------------------------------------------------------------
// The head's parameter gradients and the loss: CTA o < 64 sums row o of dW_r1
// and db_r1 over the graphs, CTA 64 dw_r2, db_r2 and the mean squared error.
__global__ void __launch_bounds__(128) head_grad(const float* __restrict__ RG, const float* __restrict__ Z,
                                                 const float* __restrict__ dZ, const float* __restrict__ y,
                                                 const float* __restrict__ tgt, int graphs, float* __restrict__ loss,
                                                 float* __restrict__ grad) {
  const int o = blockIdx.x, t = threadIdx.x;
  float acc = 0.f;
  if (o < kH) {
    if (t > kR) return;
#pragma unroll 4
    for (int g = 0; g < graphs; ++g) {
      const float d = dZ[g * kH + o];
      acc += t < kR ? d * RG[g * kR + t] : d;
    }
    grad[t < kR ? oWr1 + o * kR + t : oBr1 + o] = acc;
    return;
  }
  if (t > kH + 1) return;
#pragma unroll 4
  for (int g = 0; g < graphs; ++g) {
    const float d = y[g] - tgt[g], dy = 2.f * d / graphs;
    acc += t < kH ? dy * Z[g * kH + t] : t == kH ? dy : d * d;
  }
  if (t <= kH) grad[oWr2 + t] = acc;      // oBr2 == oWr2 + 64
  else *loss = acc / graphs;
}

// dH of one node at four columns: the top layer's share of its graph's mean
// (dnode; the graph by binary search), or S + A^T T of the layer above.
__device__ __forceinline__ float4 node_grad4(const float* __restrict__ dnode, const int* __restrict__ goff, int graphs,
                                             const int* __restrict__ rowptr, const int* __restrict__ col,
                                             const float* __restrict__ valt, const float* __restrict__ S,
                                             const float* __restrict__ T, int row, int c) {
  if (dnode) {
    int lo = 0, hi = graphs;             // goff[lo] <= row < goff[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (goff[mid] <= row) lo = mid;
      else hi = mid;
    }
    return *reinterpret_cast<const float4*>(dnode + lo * kH + c);
  }
  float4 a = spmm4(rowptr, col, valt, T, row, c);
  const float4 s = *reinterpret_cast<const float4*>(S + (long long)row * kH + c);
  return make_float4(a.x + s.x, a.y + s.y, a.z + s.z, a.w + s.w);
}

// One layer's backward pass.  Per tile: dP = dH . (Hout > 0); this CTA's share
// of dW = dP^T [H | AH] and db (kept in registers over its tiles, written as
// one partial per CTA); and the gradients passed down, Sout = dP Ws and
// Tout = dP Wn (the next kernel applies A^T to Tout while it loads).  The
// weight gradients were a serial sum over all nodes in 4160 threads (1.1 ms a
// call at 14 k nodes); here they are 64 x 128 x 64 products per tile.
constexpr int kBwdSmem = (3 * kTile * kLd + 2 * kH * kH) * (int)sizeof(float);
__global__ void __launch_bounds__(256, 2) layer_bwd(const float* __restrict__ dnode, const int* __restrict__ goff,
                                                    int graphs, const int* __restrict__ rowptr,
                                                    const int* __restrict__ col, const float* __restrict__ valt,
                                                    const float* __restrict__ S, const float* __restrict__ T,
                                                    const float* __restrict__ Hout, const float* __restrict__ H,
                                                    const float* __restrict__ AH, const half* __restrict__ L, int rows,
                                                    float* __restrict__ Sout, float* __restrict__ Tout,
                                                    float* __restrict__ part) {
  extern __shared__ __align__(16) float sm[];
  float* Ps = sm;
  float* Hs = Ps + kTile * kLd;
  float* As = Hs + kTile * kLd;
  float* Ws = As + kTile * kLd;         // [o][i] of Ws, then of Wn
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int t = tid; t < 2 * kH * kH / 2; t += blockDim.x) {
    const float2 f = __half22float2(reinterpret_cast<const half2*>(L)[t]);
    Ws[2 * t] = f.x;
    Ws[2 * t + 1] = f.y;
  }
  float gs[4][4], gn[4][4], gb = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) gs[i][j] = gn[i][j] = 0.f;
  for (int r0 = blockIdx.x * kTile; r0 < rows; r0 += gridDim.x * kTile) {
    __syncthreads();                    // the previous tile is consumed
    load_tile(H, r0, rows, Hs);
    load_tile(AH, r0, rows, As);
    for (int t = tid; t < kTile * (kH / 4); t += blockDim.x) {
      const int r = t / (kH / 4), c = (t % (kH / 4)) * 4;
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r0 + r < rows) {
        d = node_grad4(dnode, goff, graphs, rowptr, col, valt, S, T, r0 + r, c);
        const float4 h = *reinterpret_cast<const float4*>(Hout + (long long)(r0 + r) * kH + c);
        d.x = h.x > 0.f ? d.x : 0.f;
        d.y = h.y > 0.f ? d.y : 0.f;
        d.z = h.z > 0.f ? d.z : 0.f;
        d.w = h.w > 0.f ? d.w : 0.f;
      }
      *reinterpret_cast<float4*>(Ps + r * kLd + c) = d;
    }
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < kTile; ++r) {   // outputs (o = 4 ty + i, column 4 tx + j) of both weight gradients
      const float4 p = *reinterpret_cast<const float4*>(Ps + r * kLd + 4 * ty);
      const float4 h = *reinterpret_cast<const float4*>(Hs + r * kLd + 4 * tx);
      const float4 a = *reinterpret_cast<const float4*>(As + r * kLd + 4 * tx);
      const float pv[4] = {p.x, p.y, p.z, p.w}, hv[4] = {h.x, h.y, h.z, h.w}, av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          gs[i][j] = fmaf(pv[i], hv[j], gs[i][j]);
          gn[i][j] = fmaf(pv[i], av[j], gn[i][j]);
        }
    }
    if (tid < kH)
      for (int r = 0; r < kTile; ++r) gb += Ps[r * kLd + tid];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      float acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
      mm64(Ps, Ws + w * kH * kH, kH, acc);
      float* out = w ? Tout : Sout;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + 4 * ty + i;
        if (r < rows)
          *reinterpret_cast<float4*>(out + (long long)r * kH + 4 * tx) =
              make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      }
    }
  }
  float* dst = part + (long long)blockIdx.x * kLayerSize;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int at = (4 * ty + i) * kH + 4 * tx;
    *reinterpret_cast<float4*>(dst + at) = make_float4(gs[i][0], gs[i][1], gs[i][2], gs[i][3]);
    *reinterpret_cast<float4*>(dst + kH * kH + at) = make_float4(gn[i][0], gn[i][1], gn[i][2], gn[i][3]);
  }
  if (tid < kH) dst[2 * kH * kH + tid] = gb;
}

// The input layer's gradients: dP0 per tile, then 64 x (8 + 1) outputs.
constexpr int kInParams = oLayer;       // W_in and b_in come first
__global__ void __launch_bounds__(256) in_bwd(const int* __restrict__ rowptr, const int* __restrict__ col,
                                              const float* __restrict__ valt, const float* __restrict__ S,
                                              const float* __restrict__ T, const float* __restrict__ H0,
                                              const float* __restrict__ X, int rows, float* __restrict__ part) {
  __shared__ __align__(16) float Ps[kTile * kLd];
  __shared__ float Xs[kTile * kIn];
  const int tid = threadIdx.x;
  float g0 = 0.f, g1 = 0.f, gb = 0.f;
  const int i = tid & 7, o = tid >> 3;  // outputs (o, i) and (o + 32, i)
  for (int r0 = blockIdx.x * kTile; r0 < rows; r0 += gridDim.x * kTile) {
    __syncthreads();
    for (int t = tid; t < kTile * kIn; t += blockDim.x)
      Xs[t] = r0 + t / kIn < rows ? X[(long long)r0 * kIn + t] : 0.f;
    for (int t = tid; t < kTile * (kH / 4); t += blockDim.x) {
      const int r = t / (kH / 4), c = (t % (kH / 4)) * 4;
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r0 + r < rows) {
        d = node_grad4(nullptr, nullptr, 0, rowptr, col, valt, S, T, r0 + r, c);
        const float4 h = *reinterpret_cast<const float4*>(H0 + (long long)(r0 + r) * kH + c);
        d.x = h.x > 0.f ? d.x : 0.f;
        d.y = h.y > 0.f ? d.y : 0.f;
        d.z = h.z > 0.f ? d.z : 0.f;
        d.w = h.w > 0.f ? d.w : 0.f;
      }
      *reinterpret_cast<float4*>(Ps + r * kLd + c) = d;
    }
    __syncthreads();
#pragma unroll 4
    for (int r = 0; r < kTile; ++r) {
      const float x = Xs[r * kIn + i];
      g0 = fmaf(Ps[r * kLd + o], x, g0);
      g1 = fmaf(Ps[r * kLd + o + 32], x, g1);
    }
    if (tid < kH)
      for (int r = 0; r < kTile; ++r) gb += Ps[r * kLd + tid];
  }
  float* dst = part + (long long)blockIdx.x * kInParams;
  dst[oWin + o * kIn + i] = g0;
  dst[oWin + (o + 32) * kIn + i] = g1;
  if (tid < kH) dst[oBin + tid] = gb;
}

__device__ __forceinline__ void adam_one(int i, float g, float* master, half* w16, float* m, float* v, float lr,
                                         float b1, float b2, float c1, float c2, float eps) {
  m[i] = b1 * m[i] + (1.f - b1) * g;
  v[i] = b2 * v[i] + (1.f - b2) * g * g;
  master[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
  w16[i] = __float2half_rn(master[i]);
}

struct AdamArgs {
  float *master, *m, *v;
  half* w16;
  float lr, b1, b2, c1, c2, eps;
};

// The CTAs' partial gradients summed (one parameter per lane, the partials
// over the eight warps in a fixed order) into grad, and the Adam update when
// master is set.  The head's gradients are in grad already.
__global__ void __launch_bounds__(256) grad_reduce(const float* __restrict__ part_in, const float* __restrict__ part_l,
                                                   int n_part, float* __restrict__ grad, AdamArgs A) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (p < oWr1) {
    const float* src;
    int stride;
    if (p < oLayer) { src = part_in + p; stride = kInParams; }
    else {
      const int l = (p - oLayer) / kLayerSize;
      src = part_l + (long long)l * n_part * kLayerSize + (p - oLayer - l * kLayerSize);
      stride = kLayerSize;
    }
#pragma unroll 4
    for (int i = w; i < n_part; i += 8) s += src[(long long)i * stride];
  }
  red[w][lane] = s;
  __syncthreads();
  if (w != 0 || p >= kParams) return;
  if (p < oWr1) {
    s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += red[i][lane];
    grad[p] = s;
  } else {
    s = grad[p];
  }
  if (A.master) adam_one(p, s, A.master, A.w16, A.m, A.v, A.lr, A.b1, A.b2, A.c1, A.c2, A.eps);
}

__global__ void to_half(const float* src, half* dst, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __float2half_rn(src[i]);
}

inline unsigned blocks(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace mp
}  // namespace ccs

using namespace ccs;
using namespace ccs::mp;

struct ccs_mpnn_s {
  int device = -1;           // (the context may be gone when the model is freed)
  float* master = nullptr;   // FP32 master weights
  half* w16 = nullptr;       // FP16 weights used by the forward
  float* grad = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  long long step = 0;
};

namespace {

// One graph batch on the device: its arrays, activations and scratch carved
// out of one allocation from the library's stream-ordered pool (41 cudaMalloc
// and cudaFree pairs a call took longer than the kernels), returned to the
// pool on the same stream.
struct Batch {
  int n = 0, g = 0, tiles = 0, n_part = 0;
  int *rowptr = nullptr, *col = nullptr, *goff = nullptr;
  float *val = nullptr, *valt = nullptr, *x = nullptr, *glob = nullptr, *tgt = nullptr;
  float* H[kLayers + 1] = {};
  float* AH[kLayers] = {};
  float *RG = nullptr, *Z = nullptr, *y = nullptr, *loss = nullptr, *dZ = nullptr, *dnode = nullptr;
  float *S[2] = {}, *T[2] = {}, *part_in = nullptr, *part_l = nullptr;
  char* mem = nullptr;
  cudaStream_t s = nullptr;
  ~Batch() {
    if (mem) cudaFreeAsync(mem, s);
  }
};

}  // namespace

// Host-side checks of a batch: every index the kernels follow stays in range.
static bool batch_ok(const ccs_graph_batch* b) {
  if (b->n_nodes < 0 || b->n_graphs <= 0 || !b->x || !b->rowptr || !b->graph_off || !b->glob) return false;
  if (b->rowptr[0] != 0 || b->graph_off[0] != 0 || b->graph_off[b->n_graphs] != b->n_nodes) return false;
  for (int g = 0; g < b->n_graphs; ++g)
    if (b->graph_off[g + 1] < b->graph_off[g]) return false;
  for (int v = 0; v < b->n_nodes; ++v)
    if (b->rowptr[v + 1] < b->rowptr[v]) return false;
  const int nnz = b->rowptr[b->n_nodes];
  if (nnz > 0 && (!b->col || !b->val || !b->val_t)) return false;
  for (int e = 0; e < nnz; ++e)
    if (b->col[e] < 0 || b->col[e] >= b->n_nodes) return false;
  return true;
}

// Gradient partials: one per CTA of the backward kernels, at most two CTAs per SM.
static int partials(ccs_ctx c, int tiles) { return std::max(1, std::min(tiles, 2 * c_sm_count(c))); }

// The batch's arrays in one pinned-buffer copy, the rest of the workspace
// behind them.  `target` set: buffers of the backward pass too.
static int upload_batch(ccs_ctx c, const ccs_graph_batch* b, const float* target, Batch& d) {
  if (!batch_ok(b)) return CCS_ERR_INVALID_ARG;
  d.s = c_stream(c);
  d.n = b->n_nodes;
  d.g = b->n_graphs;
  d.tiles = (d.n + kTile - 1) / kTile;
  d.n_part = partials(c, d.tiles);
  const size_t nnz = (size_t)b->rowptr[d.n], n = (size_t)d.n, g = (size_t)d.g;
  size_t total = 0, sent = 0;
  auto room = [&](size_t count) {
    const size_t at = total;
    total += (std::max<size_t>(count, 1) * 4 + 255) & ~(size_t)255;
    return at;
  };
  struct Item { const void* src; size_t bytes, off; };
  Item up[8];
  int n_up = 0;
  auto send = [&](const void* src, size_t count) {
    const size_t at = room(count);
    up[n_up++] = Item{src, count * 4, at};
    return at;
  };
  const size_t o_rowptr = send(b->rowptr, n + 1), o_col = send(b->col, nnz), o_val = send(b->val, nnz);
  const size_t o_valt = target ? send(b->val_t, nnz) : 0, o_goff = send(b->graph_off, g + 1);
  const size_t o_x = send(b->x, n * kIn), o_glob = send(b->glob, g * kGlob), o_tgt = target ? send(target, g) : 0;
  sent = total;
  size_t o_H[kLayers + 1], o_AH[kLayers] = {}, o_S[2] = {}, o_T[2] = {}, o_RG = 0, o_Z = 0, o_dZ = 0, o_dn = 0, o_pi = 0,
                                               o_pl = 0;
  for (int l = 0; l <= kLayers; ++l) o_H[l] = room(n * kH);
  const size_t o_y = room(g), o_loss = room(1);
  if (target) {
    for (int l = 0; l < kLayers; ++l) o_AH[l] = room(n * kH);
    for (int k = 0; k < 2; ++k) { o_S[k] = room(n * kH); o_T[k] = room(n * kH); }
    o_RG = room(g * kR);
    o_Z = room(g * kH);
    o_dZ = room(g * kH);
    o_dn = room(g * kH);
    o_pi = room((size_t)d.n_part * kInParams);
    o_pl = room((size_t)kLayers * d.n_part * kLayerSize);
  }
  d.mem = static_cast<char*>(pool_alloc(c, total));
  if (!d.mem) return CCS_ERR_OOM;
  char* host = stage_reserve(c, sent);
  if (!host) return CCS_ERR_OOM;
  for (int i = 0; i < n_up; ++i)
    if (up[i].bytes) std::memcpy(host + up[i].off, up[i].src, up[i].bytes);
  if (stage_send(c, d.mem, sent) != cudaSuccess) return CCS_ERR_CUDA;
  auto F = [&](size_t off) { return reinterpret_cast<float*>(d.mem + off); };
  auto I = [&](size_t off) { return reinterpret_cast<int*>(d.mem + off); };
  d.rowptr = I(o_rowptr); d.col = I(o_col); d.goff = I(o_goff);
  d.val = F(o_val); d.x = F(o_x); d.glob = F(o_glob);
  for (int l = 0; l <= kLayers; ++l) d.H[l] = F(o_H[l]);
  d.y = F(o_y); d.loss = F(o_loss);
  if (target) {
    d.valt = F(o_valt); d.tgt = F(o_tgt);
    for (int l = 0; l < kLayers; ++l) d.AH[l] = F(o_AH[l]);
    for (int k = 0; k < 2; ++k) { d.S[k] = F(o_S[k]); d.T[k] = F(o_T[k]); }
    d.RG = F(o_RG); d.Z = F(o_Z); d.dZ = F(o_dZ); d.dnode = F(o_dn); d.part_in = F(o_pi); d.part_l = F(o_pl);
  }
  return CCS_OK;
}

// Predictions, and with a target each graph's part of the backward pass.
static cudaError_t forward(ccs_mpnn net, Batch& d) {
  const half* W = net->w16;
  cudaStream_t s = d.s;
  cudaError_t e;
  if (d.n > 0) {
    if ((e = cudaFuncSetAttribute(layer_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem)) != cudaSuccess)
      return e;
    in_fwd<<<blocks((long long)d.n * kH), 256, 0, s>>>(d.x, W + oWin, W + oBin, d.n, d.H[0]); note_launch();
    for (int l = 0; l < kLayers; ++l) {
      layer_fwd<<<d.tiles, 256, kFwdSmem, s>>>(d.rowptr, d.col, d.val, d.H[l], W + oLayer + l * kLayerSize, d.n, d.AH[l],
                                               d.H[l + 1]); note_launch();
    }
  }
  readout<<<d.g, 256, 0, s>>>(d.goff, d.H[kLayers], d.glob, W + oWr1, W + oBr1, W + oWr2, W + oBr2, d.g, d.RG, d.Z,
                              d.y, d.tgt, d.dZ, d.dnode); note_launch();
  return cudaGetLastError();
}

// Gradients of every parameter into net->grad; the Adam step in the last
// launch when A.master is set.
static cudaError_t backward(ccs_mpnn net, Batch& d, const AdamArgs& A) {
  const half* W = net->w16;
  cudaStream_t s = d.s;
  cudaError_t e;
  head_grad<<<kH + 1, 128, 0, s>>>(d.RG, d.Z, d.dZ, d.y, d.tgt, d.g, d.loss, net->grad); note_launch();
  if ((e = cudaFuncSetAttribute(layer_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmem)) != cudaSuccess)
    return e;
  for (int l = kLayers - 1, k = 0; l >= 0; --l, k ^= 1) {
    const bool top = l == kLayers - 1;
    layer_bwd<<<d.n_part, 256, kBwdSmem, s>>>(top ? d.dnode : nullptr, d.goff, d.g, d.rowptr, d.col, d.valt,
                                              d.S[k ^ 1], d.T[k ^ 1], d.H[l + 1], d.H[l], d.AH[l],
                                              W + oLayer + l * kLayerSize, d.n, d.S[k], d.T[k],
                                              d.part_l + (size_t)l * d.n_part * kLayerSize); note_launch();
  }
  in_bwd<<<d.n_part, 256, 0, s>>>(d.rowptr, d.col, d.valt, d.S[(kLayers - 1) & 1], d.T[(kLayers - 1) & 1], d.H[0], d.x,
                                  d.n, d.part_in); note_launch();
  grad_reduce<<<blocks(kParams, 32), 256, 0, s>>>(d.part_in, d.part_l, d.n_part, net->grad, A); note_launch();
  return cudaGetLastError();
}

extern "C" {

int ccs_mpnn_num_params(void) { return kParams; }

int ccs_mpnn_create(ccs_ctx c, uint64_t seed, ccs_mpnn* out) {
  return abi_guard([](int code, const char*) { return code; }, [&]() -> int {
    if (!c || !out) return CCS_ERR_INVALID_ARG;
    *out = nullptr;
    auto* n = new ccs_mpnn_s();
    n->device = c_device(c);
    bool ok = cudaMalloc(&n->master, kParams * 4) == cudaSuccess && cudaMalloc(&n->w16, kParams * 2) == cudaSuccess &&
              cudaMalloc(&n->grad, kParams * 4) == cudaSuccess && cudaMalloc(&n->m, kParams * 4) == cudaSuccess &&
              cudaMalloc(&n->v, kParams * 4) == cudaSuccess;
    if (!ok) {
      ccs_mpnn_free(n);
      return CCS_ERR_OOM;
    }
    // He-style uniform init from a 64-bit LCG; biases zero
    std::vector<float> h(kParams, 0.f);
    uint64_t st = seed * 6364136223846793005ull + 1442695040888963407ull;
    auto uni = [&]() {
      st = st * 6364136223846793005ull + 1442695040888963407ull;
      return (float)((st >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
    };
    auto fill = [&](int off, int rows, int cols) {
      const float a = std::sqrt(6.f / (float)cols);
      for (int i = 0; i < rows * cols; ++i) h[off + i] = a * uni();
    };
    fill(oWin, kH, kIn);
    for (int l = 0; l < kLayers; ++l) {
      fill(oLayer + l * kLayerSize, kH, kH);
      fill(oLayer + l * kLayerSize + kH * kH, kH, kH);
    }
    fill(oWr1, kH, kR);
    fill(oWr2, 1, kH);
    if (ccs_mpnn_set_params(c, n, h.data()) != CCS_OK) {
      ccs_mpnn_free(n);
      return CCS_ERR_CUDA;
    }
    cudaMemset(n->m, 0, kParams * 4);
    cudaMemset(n->v, 0, kParams * 4);
    *out = n;
    return CCS_OK;
  });
}

void ccs_mpnn_free(ccs_mpnn n) {
  if (!n) return;
  cudaFree(n->master);
  cudaFree(n->w16);
  cudaFree(n->grad);
  cudaFree(n->m);
  cudaFree(n->v);
  pool_trim(n->device);   // the batches' workspace goes back to the driver
  delete n;
}

int ccs_mpnn_params(ccs_ctx c, ccs_mpnn n, float* out) {
  return abi_guard([](int code, const char*) { return code; }, [&]() -> int {
    if (!c || !n || !out) return CCS_ERR_INVALID_ARG;
    cudaStreamSynchronize(c_stream(c));
    return cudaMemcpy(out, n->master, kParams * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? CCS_OK : CCS_ERR_CUDA;
  });
}

int ccs_mpnn_set_params(ccs_ctx c, ccs_mpnn n, const float* in) {
  return abi_guard([](int code, const char*) { return code; }, [&]() -> int {
    if (!c || !n || !in) return CCS_ERR_INVALID_ARG;
    if (cudaMemcpy(n->master, in, kParams * 4, cudaMemcpyHostToDevice) != cudaSuccess) return CCS_ERR_CUDA;
    to_half<<<blocks(kParams), 256>>>(n->master, n->w16, kParams); note_launch();
    n->step = 0;
    return cudaDeviceSynchronize() == cudaSuccess ? CCS_OK : CCS_ERR_CUDA;
  });
}

int ccs_mpnn_forward(ccs_ctx c, ccs_mpnn n, const ccs_graph_batch* b, float* pred) {
  return abi_guard([](int code, const char*) { return code; }, [&]() -> int {
    if (!c || !n || !b || !pred || b->n_graphs <= 0) return CCS_ERR_INVALID_ARG;
    Batch d;
    int rc = upload_batch(c, b, nullptr, d);
    if (rc != CCS_OK) return rc;
    if (forward(n, d) != cudaSuccess) return CCS_ERR_CUDA;
    if (cudaMemcpyAsync(pred, d.y, d.g * 4, cudaMemcpyDeviceToHost, d.s) != cudaSuccess) return CCS_ERR_CUDA;
    return cudaStreamSynchronize(d.s) == cudaSuccess ? CCS_OK : CCS_ERR_CUDA;
  });
}

int ccs_mpnn_gradient(ccs_ctx c, ccs_mpnn n, const ccs_graph_batch* b, const float* target, float* loss,
                      float* grad) {
  return abi_guard([](int code, const char*) { return code; }, [&]() -> int {
    if (!c || !n || !b || !target || b->n_graphs <= 0) return CCS_ERR_INVALID_ARG;
    Batch d;
    int rc = upload_batch(c, b, target, d);
    if (rc != CCS_OK) return rc;
    if (forward(n, d) != cudaSuccess || backward(n, d, AdamArgs{}) != cudaSuccess) return CCS_ERR_CUDA;
    if (loss && cudaMemcpyAsync(loss, d.loss, 4, cudaMemcpyDeviceToHost, d.s) != cudaSuccess) return CCS_ERR_CUDA;
    if (grad && cudaMemcpyAsync(grad, n->grad, kParams * 4, cudaMemcpyDeviceToHost, d.s) != cudaSuccess)
      return CCS_ERR_CUDA;
    return cudaStreamSynchronize(d.s) == cudaSuccess ? CCS_OK : CCS_ERR_CUDA;
  });
}

int ccs_mpnn_train_step(ccs_ctx c, ccs_mpnn n, const ccs_graph_batch* b, const float* target, float lr,
                        float* loss) {
  return abi_guard([](int code, const char*) { return code; }, [&]() -> int {
    if (!c || !n || !b || !target || b->n_graphs <= 0) return CCS_ERR_INVALID_ARG;
    Batch d;
    int rc = upload_batch(c, b, target, d);
    if (rc != CCS_OK) return rc;
    n->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)n->step), c2 = 1.f - std::pow(b2, (float)n->step);
    const AdamArgs A{n->master, n->m, n->v, n->w16, lr, b1, b2, c1, c2, 1e-8f};
    if (forward(n, d) != cudaSuccess || backward(n, d, A) != cudaSuccess) return CCS_ERR_CUDA;
    if (loss && cudaMemcpyAsync(loss, d.loss, 4, cudaMemcpyDeviceToHost, d.s) != cudaSuccess) return CCS_ERR_CUDA;
    return cudaStreamSynchronize(d.s) == cudaSuccess ? CCS_OK : CCS_ERR_CUDA;
  });
}

}  // extern "C"

namespace ccs {
// Predict log times for a batch (used by the learned cut choice), on the
// calling context's stream.
int mpnn_predict(ccs_ctx c, ccs_mpnn n, const ccs_graph_batch* b, float* pred) {
  return ccs_mpnn_forward(c, n, b, pred);
}
}  // namespace ccs
