// Maximum-likelihood correction of fragment models (Sec. V-C: before the
// contraction the fragment data become self-consistent fragment models,
// which mitigates the sampling error of the Clifford fragments' shots).
//
// A fragment's model is its Choi form, one Hermitian operator per outcome o
// of its marginal wires on its d cut slots:
//   J_o = 2^-d sum_P T_f(o, P) (x)_j s_j(P_j),  s_j(P) = P^T at a quantum
//   input, P at a quantum output;  T_f(o, P) = Tr[(x)_j s_j(P_j) J_o].
// Physical: every J_o positive semidefinite, sum_o Tr J_o = 2^{q_in}.  The
// maximum-likelihood model under Gaussian shot noise of equal variance per
// T_f entry is the nearest physical one in Frobenius norm: all blocks'
// eigenvalues projected together onto {lambda >= 0, sum = 2^{q_in}}, each
// block rebuilt from its own eigenvectors (the eigenvalue projection of
// Smolin, Gambetta and Smith, PRL 108, 070502, 2012).
//
// GPU form, per group of fragments with the same d (d <= 6), the blocks of 16
// rows and more (d >= 4) by the register kernels further down:
//  1. ml_eig_kernel, one CTA per (fragment, outcome): the block's T_f row
//     (a star hub's operand is stored by preparation at its inputs and is
//     turned into Pauli digits first), the Choi block J_o (D = 2^d rows,
//     complex64, rows padded to D + 1 so that row and column sweeps are free
//     of bank conflicts), and a cyclic complex Jacobi eigendecomposition in
//     shared memory: D/2 disjoint rotations per round in the round-robin
//     order, D - 1 rounds per sweep, sweeps until no rotation is left above
//     2^-24 of the block's Frobenius norm (at most kMlMaxSweeps).  Each
//     rotation is a phase that makes the pair's off-diagonal entry real
//     followed by the real symmetric 2 x 2 Schur rotation (Golub & Van Loan,
//     Sec. 8.5).  The eigenvalues and eigenvectors go to a scratch array.
//  2. ml_threshold_kernel, one CTA per fragment: the threshold theta with
//     sum max(lambda - theta, 0) = 2^{q_in} over its eigenvalue list, by
//     Michelot's finite algorithm (J. Optim. Theory Appl. 50, 1986):
//     theta = (sum of the kept values - total) / (their count), keep the
//     values above theta, repeat until the kept set stops changing.
//  3. ml_rebuild_kernel, one CTA per (fragment, outcome): J'_o from the
//     eigenvectors with eigenvalues max(lambda - theta, 0), then T'_f(o, P);
//     written to T_f, and a hub's operand (by preparation at its inputs) is
//     rewritten in FP32.
#include "fsum.hpp"
#include "kernels.cuh"

namespace ccs {

namespace {

constexpr int kMlMaxSweeps = 30;

__device__ __forceinline__ int ml_find(const MlFrag* __restrict__ fr, int n, long long blk) {
  int lo = 0, hi = n;      // fr[lo].blk0 <= blk < fr[hi].blk0
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (fr[mid].blk0 <= blk) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Sum over the CTA (every thread gets the result); red holds 32 entries.
template <class T>
__device__ T block_sum(T v, T* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  T s = 0;
  for (int i = 0; i < nw; ++i) s += red[i];
  return s;
}

// Largest value over the CTA (every thread gets it); red holds 32 entries.
__device__ float block_max(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  float m = 0.f;
  for (int i = 0; i < nw; ++i) m = fmaxf(m, red[i]);
  return m;
}

// Entry [r][c] of the slot operator (x)_j s_j(P_j) for the Pauli digits of P
// where the entry is nonzero: returns the power of i (0..3) of the entry
// (its value is i^pw, a sign folded in as 2).  At slot j the entry needs
// P_j in {I, Z} when r_j == c_j and in {X, Y} otherwise; Z contributes
// (-1)^{r_j}; Y at an output contributes -i for r_j = 0 and +i for r_j = 1,
// its transpose at an input the opposite.
__device__ __forceinline__ int slot_entry_phase(int P, int r, int d, unsigned inmask) {
  int pw = 0;
  for (int j = 0; j < d; ++j) {
    const int pj = (P >> (2 * j)) & 3, rj = (r >> j) & 1;
    if (pj == 3) pw += 2 * rj;
    else if (pj == 2) pw += 1 + 2 * ((rj ^ 1) ^ (int)((inmask >> j) & 1));
  }
  return pw & 3;
}

__device__ __forceinline__ unsigned input_mask(const FragDev& F) {
  unsigned m = 0;
  for (int j = 0; j < F.n_slots; ++j)
    if ((F.slot_code[j] >> 8) == 0) m |= 1u << j;
  return m;
}

}  // namespace

// One CTA per (fragment, outcome o) of a group with d cut slots.
__global__ void __launch_bounds__(256, 3) ml_eig_kernel(DevPlan P, DevRes R, const MlFrag* __restrict__ fr,
                                                        int nfr, int d, float* __restrict__ scratch) {
  extern __shared__ __align__(16) float2 smc[];
  const int D = 1 << d, LD = D + 1, KP = 1 << (2 * d), H = D / 2;
  float2* A = smc;               // D x LD: the Choi block, then its rotations
  float2* V = A + D * LD;        // D x LD: the accumulated unitary, transposed (row k = column k of V)
  float* sT = reinterpret_cast<float*>(V);   // the block's T_f row (4^d), before V is set up
  float4* prm = reinterpret_cast<float4*>(V + D * LD);   // per pair: (c, s, t, Re w), (Im w, a_pp, a_qq, |a_pq|)
  int2* pq = reinterpret_cast<int2*>(prm + 2 * H);        // per pair: p, q
  int* blk_ij = reinterpret_cast<int*>(pq + H);           // pair blocks i <= j of a round: i | j << 16
  __shared__ float red[32];
  __shared__ int any_rot;
  const int tid = threadIdx.x, nt = blockDim.x;

  const long long blk = blockIdx.x;
  const MlFrag& mf = fr[ml_find(fr, nfr, blk)];
  const FragDev& F = P.frags[mf.frag];
  const int o = (int)(blk - mf.blk0);
  const unsigned inmask = input_mask(F);

  // 1. the block's row of T_f
  if (!mf.hub) {
    const float* src = R.T + F.T_off + ((long long)o << (2 * d));
    for (int i = tid; i < KP; i += nt) sT[i] = src[i];
  } else {   // hub operand Q^T[D][o]: preparation digit s at each input slot
    const long long Mo = 1ll << F.m;
    if (mf.i16) {
      const int16_t* q = reinterpret_cast<const int16_t*>(R.TQ + F.T_off);
      for (int i = tid; i < KP; i += nt) sT[i] = (float)q[(long long)i * Mo + o] * R.hub_scale;
    } else {
      for (int i = tid; i < KP; i += nt) sT[i] = R.TQ[F.T_off + (long long)i * Mo + o];
    }
    // T(P_j) = sum_s mu(P_j, s) Q(s): I = Q0 + Q1, X = 2 Q2 - Q0 - Q1,
    // Y = 2 Q3 - Q0 - Q1, Z = Q0 - Q1 (the prepared states |0>,|1>,|+>,|+i>)
    for (int j = 0; j < d; ++j) {
      if (!((inmask >> j) & 1)) continue;
      __syncthreads();
      const int st = 1 << (2 * j);
      for (int g = tid; g < KP / 4; g += nt) {
        const int b = ((g >> (2 * j)) << (2 * j + 2)) | (g & (st - 1));
        const float q0 = sT[b], q1 = sT[b + st], q2 = sT[b + 2 * st], q3 = sT[b + 3 * st];
        sT[b] = q0 + q1;
        sT[b + st] = 2.f * q2 - q0 - q1;
        sT[b + 2 * st] = 2.f * q3 - q0 - q1;
        sT[b + 3 * st] = q0 - q1;
      }
    }
  }
  __syncthreads();

  // 2. J_o[r][c] = 2^-d sum over the 2^d Paulis whose slot operator is
  //    nonzero at [r][c]
  const float scale = 1.f / (float)D;
  float nrm = 0.f;
  for (int e = tid; e < D * D; e += nt) {
    const int r = e >> d, c = e & (D - 1), x = r ^ c;
    float re = 0.f, im = 0.f;
    for (int t = 0; t < D; ++t) {
      int Pi = 0;
      for (int j = 0; j < d; ++j) {
        const int xj = (x >> j) & 1, tj = (t >> j) & 1;
        Pi |= (xj ? (tj ? 2 : 1) : (tj ? 3 : 0)) << (2 * j);
      }
      const float v = sT[Pi];
      switch (slot_entry_phase(Pi, r, d, inmask)) {
        case 0: re += v; break;
        case 1: im += v; break;
        case 2: re -= v; break;
        default: im -= v; break;
      }
    }
    re *= scale;
    im *= scale;
    A[r * LD + c] = make_float2(re, im);
    nrm += re * re + im * im;
  }
  nrm = block_sum(nrm, red);     // its barriers also end the reads of sT
  for (int e = tid; e < D * D; e += nt) {
    const int r = e >> d, c = e & (D - 1);
    V[r * LD + c] = make_float2(r == c ? 1.f : 0.f, 0.f);
  }
  const float tol = sqrtf(nrm) * 5.9604645e-8f;   // 2^-24 of the Frobenius norm
  for (int j = tid; j < H; j += nt)
    for (int i = 0; i <= j; ++i) blk_ij[j * (j + 1) / 2 + i] = i | (j << 16);

  // 3. cyclic Jacobi, round-robin pairs: round t pairs (D-1, t) and
  //    ((t + i) mod (D-1), (t - i) mod (D-1)) for i = 1 .. D/2 - 1.  With
  //    a_pq = |a_pq| w, the rotation U = [[c, s], [-s conj(w), c conj(w)]]
  //    on columns (p, q) zeroes a_pq and leaves a_pp - t |a_pq|,
  //    a_qq + t |a_pq| on the diagonal.  All of a round's rotations are
  //    applied at once, A <- U^H A U block by block: the 2 x 2 block of pairs
  //    (i, j), i < j, becomes U_i^H B U_j and its mirror block the conjugate
  //    transpose (so A stays exactly Hermitian); V^T's rows p, q take the
  //    column update of V <- V U.
  if (nrm > 0.f && D > 1) {
    const int nblk = H * (H + 1) / 2;
    const int lg_tpp = max(0, (31 - __clz(nt)) - (d - 1));   // threads per pair in the V^T update
    const int vi = tid >> lg_tpp, vl = tid & ((1 << lg_tpp) - 1);
    for (int sweep = 0; sweep < kMlMaxSweeps; ++sweep) {
      if (tid == 0) any_rot = 0;
      __syncthreads();
      for (int t = 0; t < D - 1; ++t) {
        if (tid < H) {
          int a, b;
          if (tid == 0) { a = D - 1; b = t; }
          else { a = (t + tid) % (D - 1); b = (t - tid + D - 1) % (D - 1); }
          const int p = min(a, b), q = max(a, b);
          const float app = A[p * LD + p].x, aqq = A[q * LD + q].x;
          const float2 apq = A[p * LD + q];
          const float mag = sqrtf(apq.x * apq.x + apq.y * apq.y);
          float c = 1.f, s = 0.f, tt = 0.f, wr = 1.f, wi = 0.f;
          if (mag > tol) {
            const float tau = (aqq - app) / (2.f * mag);
            tt = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
            c = 1.f / sqrtf(1.f + tt * tt);
            s = tt * c;
            wr = apq.x / mag;
            wi = apq.y / mag;
            if (tt != 0.f) any_rot = 1;
          }
          prm[2 * tid] = make_float4(c, s, tt, wr);
          prm[2 * tid + 1] = make_float4(wi, app, aqq, mag);
          pq[tid] = make_int2(p, q);
        }
        __syncthreads();
        // A: one 2 x 2 block per pair of pairs (i <= j)
        for (int e = tid; e < nblk; e += nt) {
          const int ij = blk_ij[e], i = ij & 0xffff, j = ij >> 16;
          const float4 pi0 = prm[2 * i], pj0 = prm[2 * j];
          const bool ri = pi0.z != 0.f, rj = pj0.z != 0.f;
          if (!ri && !rj) continue;
          const float4 pi1 = prm[2 * i + 1];
          const int2 pqi = pq[i];
          const int p = pqi.x, q = pqi.y;
          if (i == j) {
            A[p * LD + p] = make_float2(pi1.y - pi0.z * pi1.w, 0.f);
            A[q * LD + q] = make_float2(pi1.z + pi0.z * pi1.w, 0.f);
            A[p * LD + q] = make_float2(0.f, 0.f);
            A[q * LD + p] = make_float2(0.f, 0.f);
            continue;
          }
          const float4 pj1 = prm[2 * j + 1];
          const int2 pqj = pq[j];
          const int u = pqj.x, v = pqj.y;
          float2 b00 = A[p * LD + u], b01 = A[p * LD + v], b10 = A[q * LD + u], b11 = A[q * LD + v];
          if (rj) {   // B <- B U_j: columns c b0 - s conj(w) b1, s b0 + c conj(w) b1
            const float c = pj0.x, s = pj0.y, wr = pj0.w, wi = -pj1.x;
            const float2 y0 = make_float2(wr * b01.x - wi * b01.y, wr * b01.y + wi * b01.x);
            const float2 y1 = make_float2(wr * b11.x - wi * b11.y, wr * b11.y + wi * b11.x);
            const float2 n00 = make_float2(c * b00.x - s * y0.x, c * b00.y - s * y0.y);
            const float2 n01 = make_float2(s * b00.x + c * y0.x, s * b00.y + c * y0.y);
            const float2 n10 = make_float2(c * b10.x - s * y1.x, c * b10.y - s * y1.y);
            const float2 n11 = make_float2(s * b10.x + c * y1.x, s * b10.y + c * y1.y);
            b00 = n00; b01 = n01; b10 = n10; b11 = n11;
          }
          if (ri) {   // B <- U_i^H B: rows c r0 - s w r1, s r0 + c w r1
            const float c = pi0.x, s = pi0.y, wr = pi0.w, wi = pi1.x;
            const float2 y0 = make_float2(wr * b10.x - wi * b10.y, wr * b10.y + wi * b10.x);
            const float2 y1 = make_float2(wr * b11.x - wi * b11.y, wr * b11.y + wi * b11.x);
            const float2 n00 = make_float2(c * b00.x - s * y0.x, c * b00.y - s * y0.y);
            const float2 n01 = make_float2(c * b01.x - s * y1.x, c * b01.y - s * y1.y);
            const float2 n10 = make_float2(s * b00.x + c * y0.x, s * b00.y + c * y0.y);
            const float2 n11 = make_float2(s * b01.x + c * y1.x, s * b01.y + c * y1.y);
            b00 = n00; b01 = n01; b10 = n10; b11 = n11;
          }
          A[p * LD + u] = b00; A[p * LD + v] = b01; A[q * LD + u] = b10; A[q * LD + v] = b11;
          A[u * LD + p] = make_float2(b00.x, -b00.y);
          A[v * LD + p] = make_float2(b01.x, -b01.y);
          A[u * LD + q] = make_float2(b10.x, -b10.y);
          A[v * LD + q] = make_float2(b11.x, -b11.y);
        }
        // V^T rows p, q (one pair per group of threads, its rotation in registers)
        if (vi < H) {
          const float4 pr0 = prm[2 * vi];
          if (pr0.z != 0.f) {
            const int2 pqv = pq[vi];
            const int p = pqv.x, q = pqv.y;
            const float c = pr0.x, s = pr0.y, wr = pr0.w, wi = -prm[2 * vi + 1].x;
            for (int r = vl; r < D; r += (1 << lg_tpp)) {
              const float2 vp = V[p * LD + r], vq = V[q * LD + r];
              const float2 y = make_float2(wr * vq.x - wi * vq.y, wr * vq.y + wi * vq.x);
              V[p * LD + r] = make_float2(c * vp.x - s * y.x, c * vp.y - s * y.y);
              V[q * LD + r] = make_float2(s * vp.x + c * y.x, s * vp.y + c * y.y);
            }
          }
        }
        __syncthreads();
      }
      // stop once no off-diagonal entry exceeds the tolerance (the next
      // sweep would rotate nothing)
      float off = 0.f;
      for (int e2 = tid; e2 < D * D; e2 += nt) {
        const int r = e2 >> d, c = e2 & (D - 1);
        if (r != c) {
          const float2 x = A[r * LD + c];
          off = fmaxf(off, x.x * x.x + x.y * x.y);
        }
      }
      off = block_max(off, red);
      const int more = any_rot;
      __syncthreads();
      if (!more || off <= tol * tol) break;
    }
  }
  __syncthreads();

  // 4. eigenvalues (the real diagonal) and eigenvectors (the rows of V^T,
  //    stored row-major D x D complex: entry [k][r] = component r of vector k)
  float* ev = scratch + mf.ev_off + (long long)o * D;
  float2* vec = reinterpret_cast<float2*>(scratch + mf.vec_off) + (long long)o * D * D;
  for (int i = tid; i < D; i += nt) ev[i] = A[i * LD + i].x;
  for (int e = tid; e < D * D; e += nt) vec[e] = V[(e >> d) * LD + (e & (D - 1))];
}

// One CTA per fragment: theta over its eigenvalue list, which stays in
// registers up to 16 per thread.  A pass adds the kept values in three FP32
// parts (no fewer bits than FP64) and only the warps' sums in FP64: with FP64
// adds and compares per value a pass was bound by the FP64 units (16 fragments
// of 8192 values: 76 us, 33 us so; a pair of FP32 parts, of fewer bits, 25 us).
// Warps past the last value add and shuffle nothing: corrections of a few hundred
// values took 2 to 4 us more otherwise.
constexpr int kThetaThreads = 1024, kThetaRegs = 16;

__global__ void __launch_bounds__(kThetaThreads) ml_threshold_kernel(DevPlan P, const MlFrag* __restrict__ fr,
                                                                     const float* __restrict__ scratch,
                                                                     double* __restrict__ theta_out) {
  __shared__ double s_sum[32];
  __shared__ int s_cnt[32];
  __shared__ double s_theta;
  __shared__ long long s_kept;
  const MlFrag& mf = fr[blockIdx.x];
  const FragDev& F = P.frags[mf.frag];
  const long long n = (1ll << F.m) << mf.d;
  const float* ev = scratch + mf.ev_off;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool in_regs = n <= (long long)kThetaThreads * kThetaRegs;
  const float none = __int_as_float(0xff800000);     // -infinity: never kept
  float v[kThetaRegs];
#pragma unroll
  for (int i = 0; i < kThetaRegs; ++i) {
    const long long at = tid + (long long)i * kThetaThreads;
    v[i] = in_regs && at < n ? ev[at] : none;
  }
  double theta = -1e300;
  long long prev = -1;
  // the kept set only shrinks, so at most n + 1 passes; the cap bounds the
  // loop should rounding ever make it oscillate
  for (long long it = 0; it <= n + 1 && it < 4096; ++it) {
    const float cut = __double2float_rd(theta);      // v > theta exactly when v > cut, for a float v
    Sum3 s;
    int cnt = 0;
    if (in_regs) {
#pragma unroll
      for (int i = 0; i < kThetaRegs; ++i) {
        if (32 * warp + (long long)i * kThetaThreads >= n) break;      // the warp's values end here
        if (v[i] > cut) { s.add(v[i]); ++cnt; }
      }
    } else {
#pragma unroll 4
      for (long long i = tid; i < n; i += kThetaThreads) {
        const float x = ev[i];
        if (x > cut) { s.add(x); ++cnt; }
      }
    }
    if (32 * warp < n) {
      for (int o = 16; o > 0; o >>= 1) {
        Sum3 other;
        other.s = __shfl_xor_sync(0xffffffffu, s.s, o);
        other.c = __shfl_xor_sync(0xffffffffu, s.c, o);
        other.e = __shfl_xor_sync(0xffffffffu, s.e, o);
        s.add(other);
      }
      cnt = __reduce_add_sync(0xffffffffu, cnt);
    }
    if (lane == 0) {
      s_sum[warp] = s.value();
      s_cnt[warp] = cnt;
    }
    __syncthreads();
    if (warp == 0) {
      double t = s_sum[lane];
      long long k = s_cnt[lane];
      for (int o = 16; o > 0; o >>= 1) {
        t += __shfl_xor_sync(0xffffffffu, t, o);
        k += __shfl_xor_sync(0xffffffffu, k, o);
      }
      if (lane == 0) {
        s_kept = k;
        s_theta = k ? (t - mf.total) / (double)k : theta;
      }
    }
    __syncthreads();
    if (s_kept == prev || s_kept == 0) break;
    prev = s_kept;
    theta = s_theta > theta ? s_theta : theta;
  }
  if (tid == 0) theta_out[blockIdx.x] = theta;
}

// One CTA per (fragment, outcome o): the corrected block and T'_f row.
__global__ void __launch_bounds__(256) ml_rebuild_kernel(DevPlan P, DevRes R, const MlFrag* __restrict__ fr,
                                                         int nfr, int d, const float* __restrict__ scratch,
                                                         const double* __restrict__ theta) {
  extern __shared__ float2 smc[];
  const int D = 1 << d, LD = D + 1, KP = 1 << (2 * d);
  float2* V = smc;               // D x LD eigenvectors (row k = vector k)
  float2* J = V + D * LD;        // D x LD: J'
  float* lam = reinterpret_cast<float*>(J + D * LD);   // D clipped eigenvalues
  float* sT = lam + D;           // 4^d
  int* live = reinterpret_cast<int*>(sT + KP);          // indices of the nonzero eigenvalues
  __shared__ int n_live;
  const int tid = threadIdx.x, nt = blockDim.x;

  const long long blk = blockIdx.x;
  const MlFrag& mf = fr[ml_find(fr, nfr, blk)];
  const FragDev& F = P.frags[mf.frag];
  const int o = (int)(blk - mf.blk0);
  const unsigned inmask = input_mask(F);
  const float th = (float)theta[mf.index];
  const float* ev = scratch + mf.ev_off + (long long)o * D;
  const float2* vec = reinterpret_cast<const float2*>(scratch + mf.vec_off) + (long long)o * D * D;
  for (int e = tid; e < D * D; e += nt) V[(e >> d) * LD + (e & (D - 1))] = vec[e];
  for (int i = tid; i < D; i += nt) lam[i] = fmaxf(ev[i] - th, 0.f);
  __syncthreads();
  if (tid == 0) {
    int k = 0;
    for (int i = 0; i < D; ++i)
      if (lam[i] > 0.f) live[k++] = i;
    n_live = k;
  }
  __syncthreads();
  const int nl = n_live;
  // J'[r][c] = sum_k lam_k v_k[r] conj(v_k[c])
  for (int e = tid; e < D * D; e += nt) {
    const int r = e >> d, c = e & (D - 1);
    float re = 0.f, im = 0.f;
    for (int t = 0; t < nl; ++t) {
      const int k = live[t];
      const float l = lam[k];
      const float2 a = V[k * LD + r], b = V[k * LD + c];
      re += l * (a.x * b.x + a.y * b.y);
      im += l * (a.y * b.x - a.x * b.y);
    }
    J[r * LD + c] = make_float2(re, im);
  }
  __syncthreads();
  // T'(P) = Re Tr[S_P J'] = sum_r Re(S_P[r][c] J'[c][r]), c = r xor x(P)
  for (int Pi = tid; Pi < KP; Pi += nt) {
    int x = 0;
    for (int j = 0; j < d; ++j) {
      const int pj = (Pi >> (2 * j)) & 3;
      if (pj == 1 || pj == 2) x |= 1 << j;
    }
    float acc = 0.f;
    for (int r = 0; r < D; ++r) {
      const float2 v = J[(r ^ x) * LD + r];
      switch (slot_entry_phase(Pi, r, d, inmask)) {   // Re(i^pw (re + i im))
        case 0: acc += v.x; break;
        case 1: acc -= v.y; break;
        case 2: acc -= v.x; break;
        default: acc += v.y; break;
      }
    }
    sT[Pi] = acc;
  }
  __syncthreads();
  float* dst = R.T + F.T_off + ((long long)o << (2 * d));
  for (int i = tid; i < KP; i += nt) dst[i] = sT[i];
  if (!mf.hub) return;
  // the hub's operand by preparation at its inputs: Q(s) = Tr[E(rho_s) ...]
  // = (T_I + T_Z)/2, (T_I - T_Z)/2, (T_I + T_X)/2, (T_I + T_Y)/2
  for (int j = 0; j < d; ++j) {
    if (!((inmask >> j) & 1)) continue;
    __syncthreads();
    const int st = 1 << (2 * j);
    for (int g = tid; g < KP / 4; g += nt) {
      const int b = ((g >> (2 * j)) << (2 * j + 2)) | (g & (st - 1));
      const float tI = sT[b], tX = sT[b + st], tY = sT[b + 2 * st], tZ = sT[b + 3 * st];
      sT[b] = 0.5f * (tI + tZ);
      sT[b + st] = 0.5f * (tI - tZ);
      sT[b + 2 * st] = 0.5f * (tI + tX);
      sT[b + 3 * st] = 0.5f * (tI + tY);
    }
  }
  __syncthreads();
  const long long Mo = 1ll << F.m;
  for (int i = tid; i < KP; i += nt) R.TQ[F.T_off + (long long)i * Mo + o] = sT[i];
}

// --- blocks of 16 to 64 rows: one-sided Jacobi in registers ------------------
// With H = J - (tr J / D) I, the columns of G = H / |H|_F + I (positive
// definite, as H has no eigenvalue below -sqrt(1 - 1/D) |H|_F; its singular
// vectors are J's eigenvectors) are made orthogonal by plane
// rotations from the right (Hestenes 1958; Golub & Van Loan, Sec. 8.6): then
// v_k = g_k / |g_k|, the eigenvalue is its Rayleigh quotient with J, and no
// separate eigenvector matrix is rotated.  The mean is taken out so that the
// rounding of columns of length one is measured against the eigenvalues'
// spread, not against the mean of a nearly scalar block.  A worker of LW lanes keeps two
// groups of four columns in registers, two or four rows a lane as packed FP32
// pairs: a step rotates four disjoint pairs (their inner products reduced
// together), a round runs
// the 4 x 4 pairs across the two groups, and only then do the groups move one
// place round the tournament through shared memory, 2 (D / 4) - 1 rounds a
// sweep.  A two-sided Jacobi in shared memory moves the whole block and its
// eigenvectors once per round of D/2 pairs and is bound by that traffic (46%
// bank conflicts) and two barriers a round: 768 blocks of 64 x 64 took 4.30 ms
// and 1280 of 16 x 16 0.28 ms, here 0.93 and 0.050 ms (issue and the steps'
// latency: 51% of the issue slots at the four CTAs per SM the registers allow).
// D = 16 packs two blocks into a warp (they sweep until both are done).
template <int D>
struct MlShape {
  static constexpr int LG = D == 64 ? 6 : D == 32 ? 5 : 4;
  static constexpr int RH = D == 16 ? 1 : 2;          // row pairs of a lane
  static constexpr int LW = D / (2 * RH);             // lanes of a worker: 16 or 8
  static constexpr int NW = D / 8, NG = 2 * NW;       // workers, column groups
  static constexpr int TPB = LW * NW;                 // threads of one block: 128, 32 or 16
  static constexpr int BPC = D == 16 ? 2 : 1;         // blocks of one CTA
  static constexpr int NT = TPB * BPC;
  static constexpr int MINB = D == 64 ? 4 : 12;
  static __device__ __forceinline__ void sync() {
    if (NT <= 32) __syncwarp();
    else __syncthreads();
  }
};

// The rebuild's threads: a 4 x 4 block of J' each.
template <int D>
struct MlTile {
  static constexpr int TPB = (D / 4) * (D / 4), BPC = D == 16 ? 2 : 1, NT = TPB * BPC;
  static __device__ __forceinline__ void sync() {
    if (NT <= 32) __syncwarp();
    else __syncthreads();
  }
};

// Two FP32 lanes in a 64-bit register: Blackwell's packed FP32 arithmetic.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pk(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 upk(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// A column of the worker: per row pair the two real and the two imaginary parts.
template <int RH>
struct MlCol {
  f2 x[RH], y[RH];
};

// Bit j of x at bit 2 j (six bits).
__device__ __forceinline__ int spread6(int x) {
  x = (x | (x << 4)) & 0x30f;
  x = (x | (x << 2)) & 0x333;
  return (x | (x << 1)) & 0x555;
}

// The block as an array over the slots' digits: digit e_j = r_j + 2 c_j holds
// the entry's row and column bit.  Per slot, Pauli digits (I, X, Y, Z) turn
// into the 2 x 2 block (J00, J10, J01, J11) = (I + Z, X + iY, X - iY, I - Z) at
// an output, Y's sign the opposite at an input, and back.
template <int D>
__device__ __forceinline__ void pauli_to_block(float2* X, unsigned inmask, int lt) {
  using S = MlShape<D>;
  for (int j = 0; j < S::LG; ++j) {
    const float sg = (inmask >> j) & 1 ? -1.f : 1.f;
    const int st = 1 << (2 * j);
    for (int g = lt; g < D * D / 4; g += S::TPB) {
      float2* x = X + (((g >> (2 * j)) << (2 * j + 2)) | (g & (st - 1)));
      const float2 I = x[0], A = x[st], B = make_float2(sg * x[2 * st].x, sg * x[2 * st].y), Z = x[3 * st];
      x[0] = make_float2(I.x + Z.x, I.y + Z.y);
      x[st] = make_float2(A.x - B.y, A.y + B.x);
      x[2 * st] = make_float2(A.x + B.y, A.y - B.x);
      x[3 * st] = make_float2(I.x - Z.x, I.y - Z.y);
    }
    S::sync();
  }
}
template <int D>
__device__ __forceinline__ void block_to_pauli(float2* X, unsigned inmask, int lt) {
  using S = MlTile<D>;
  for (int j = 0; j < MlShape<D>::LG; ++j) {
    const float sg = (inmask >> j) & 1 ? -1.f : 1.f;
    const int st = 1 << (2 * j);
    for (int g = lt; g < D * D / 4; g += S::TPB) {
      float2* x = X + (((g >> (2 * j)) << (2 * j + 2)) | (g & (st - 1)));
      const float2 a = x[0], b = x[st], c = x[2 * st], e = x[3 * st];   // J00, J10, J01, J11
      x[0] = make_float2(a.x + e.x, a.y + e.y);
      x[st] = make_float2(b.x + c.x, b.y + c.y);
      x[2 * st] = make_float2(sg * (b.y - c.y), sg * (c.x - b.x));      // -i J10 + i J01
      x[3 * st] = make_float2(a.x - e.x, a.y - e.y);
    }
    S::sync();
  }
}

// Refined reciprocal square root (one Newton step on the hardware estimate).
__device__ __forceinline__ float rsqrt_n(float x) {
  const float y = rsqrtf(x);
  return y * fmaf(-0.5f * x * y, y, 1.5f);
}

// The four sums of 8 values over a worker's lanes that leave lane pair (top two
// lane bits) p with (v[2p], v[2p + 1]).
template <int LW>
__device__ __forceinline__ void reduce_pairs(const float (&v)[8], float& re, float& im) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & (LW - 1);
  const bool b1 = lane & (LW / 2), b2 = lane & (LW / 4);
  float u[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float keep = b1 ? v[i + 4] : v[i], give = b1 ? v[i] : v[i + 4];
    u[i] = keep + __shfl_xor_sync(FULL, give, LW / 2);
  }
  re = (b2 ? u[2] : u[0]) + __shfl_xor_sync(FULL, b2 ? u[0] : u[2], LW / 4);
  im = (b2 ? u[3] : u[1]) + __shfl_xor_sync(FULL, b2 ? u[1] : u[3], LW / 4);
#pragma unroll
  for (int o = LW / 8; o > 0; o >>= 1) {
    re += __shfl_xor_sync(FULL, re, o);
    im += __shfl_xor_sync(FULL, im, o);
  }
}

// Squared norms of the worker's eight columns, on every lane.
template <int D>
__device__ __forceinline__ void column_norms(const MlCol<MlShape<D>::RH> (&g)[8], float (&nr)[8]) {
  constexpr int LW = MlShape<D>::LW, RH = MlShape<D>::RH;
  float v[8], a, b;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    f2 s = mul2(g[i].x[0], g[i].x[0]);
    s = fma2(g[i].y[0], g[i].y[0], s);
#pragma unroll
    for (int h = 1; h < RH; ++h) s = fma2(g[i].y[h], g[i].y[h], fma2(g[i].x[h], g[i].x[h], s));
    const float2 t = upk(s);
    v[i] = t.x + t.y;
  }
  reduce_pairs<LW>(v, a, b);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int src = ((p >> 1) ? LW / 2 : 0) + ((p & 1) ? LW / 4 : 0);
    nr[2 * p] = __shfl_sync(0xffffffffu, a, src, LW);
    nr[2 * p + 1] = __shfl_sync(0xffffffffu, b, src, LW);
  }
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// One step: the four column pairs (p_i, q_i) made orthogonal.  With
// gamma = g_p^H g_q = |gamma| w and t the small root of t^2 + 2 zeta t = 1,
// zeta = (|q|^2 - |p|^2) / (2 |gamma|), c = 1 / sqrt(1 + t^2), z = t c w:
//   p <- c p - conj(z) q,  q <- z p + c q
// (t may carry the estimates' rounding, c and z must not: the rotation is
// unitary for any t).  The lanes of pair i compute its rotation.  A pair below
// 2^-23 of its norms' product is left alone; one above 2^-21 asks for another
// sweep.  (Between well separated eigenvalues a sweep from 2^-16 on ends below
// 2^-23, but inside a cluster, whose vectors turn by large angles, it gains a bit
// or two: stopped at 2^-16, a block of rank one and 63 other eigenvalues within
// 1e-5 kept off-diagonals of that size, 1.9e-5 of |J|_F in all, 4e-6 so.)
template <int D, int P0, int Q0, int P1, int Q1, int P2, int Q2, int P3, int Q3>
__device__ __forceinline__ void jacobi_step(MlCol<MlShape<D>::RH> (&g)[8], float (&nr)[8], bool& more) {
  constexpr int LW = MlShape<D>::LW, RH = MlShape<D>::RH;
  constexpr int pp[4] = {P0, P1, P2, P3}, qq[4] = {Q0, Q1, Q2, Q3};
  const unsigned FULL = 0xffffffffu;
  float v[8], re, im;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const auto &p = g[pp[i]], &q = g[qq[i]];
    f2 r2 = mul2(p.x[0], q.x[0]), a2 = mul2(p.x[0], q.y[0]), b2 = mul2(p.y[0], q.x[0]);
    r2 = fma2(p.y[0], q.y[0], r2);
#pragma unroll
    for (int h = 1; h < RH; ++h) {
      r2 = fma2(p.y[h], q.y[h], fma2(p.x[h], q.x[h], r2));
      a2 = fma2(p.x[h], q.y[h], a2);
      b2 = fma2(p.y[h], q.x[h], b2);
    }
    const float2 rr = upk(r2), aa = upk(a2), bb = upk(b2);
    v[2 * i] = rr.x + rr.y;
    v[2 * i + 1] = (aa.x - bb.x) + (aa.y - bb.y);
  }
  reduce_pairs<LW>(v, re, im);
  const int lane = threadIdx.x & (LW - 1);
  const bool b1 = lane & (LW / 2), b2 = lane & (LW / 4);
  const float al = b1 ? (b2 ? nr[P3] : nr[P2]) : (b2 ? nr[P1] : nr[P0]);
  const float be = b1 ? (b2 ? nr[Q3] : nr[Q2]) : (b2 ? nr[Q1] : nr[Q0]);
  const float g2 = fmaf(re, re, im * im), ab = al * be;
  const bool rot = g2 > 1.4210855e-14f * ab;                 // 2^-46
  more = more || g2 > 2.2737368e-13f * ab;                   // 2^-42
  if (!__any_sync(FULL, rot)) return;
  float c = 1.f, zr = 0.f, zi = 0.f, dn = 0.f;
  if (rot) {
    const float inv = rsqrt_n(g2), zeta = 0.5f * (be - al) * inv;
    const float t = copysignf(__fdividef(1.f, fabsf(zeta) + sqrt_approx(fmaf(zeta, zeta, 1.f))), zeta);
    c = rsqrt_n(fmaf(t, t, 1.f));
    const float sw = t * c * inv;
    zr = sw * re;
    zi = sw * im;
    dn = t * (g2 * inv);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int src = ((i >> 1) ? LW / 2 : 0) + ((i & 1) ? LW / 4 : 0);
    const float ci = __shfl_sync(FULL, c, src, LW), zx = __shfl_sync(FULL, zr, src, LW);
    const float zy = __shfl_sync(FULL, zi, src, LW), di = __shfl_sync(FULL, dn, src, LW);
    nr[pp[i]] -= di;
    nr[qq[i]] += di;
    const f2 c2 = pk(ci, ci), zx2 = pk(zx, zx), zy2 = pk(zy, zy), mx2 = pk(-zx, -zx), my2 = pk(-zy, -zy);
    auto &p = g[pp[i]], &q = g[qq[i]];
#pragma unroll
    for (int h = 0; h < RH; ++h) {
      const f2 px = p.x[h], py = p.y[h], qx = q.x[h], qy = q.y[h];
      p.x[h] = fma2(my2, qy, fma2(mx2, qx, mul2(c2, px)));
      p.y[h] = fma2(zy2, qx, fma2(mx2, qy, mul2(c2, py)));
      q.x[h] = fma2(my2, py, fma2(zx2, px, mul2(c2, qx)));
      q.y[h] = fma2(zy2, px, fma2(zx2, py, mul2(c2, qy)));
    }
  }
}

template <int D>
constexpr size_t ml_jacobi_smem() {   // per block: the exchange buffer and the column norms beside it
  return (size_t)MlShape<D>::BPC * (D * D * sizeof(float2) + D * sizeof(float));
}

template <int D>
__global__ void __launch_bounds__(MlShape<D>::NT, MlShape<D>::MINB)
    ml_jacobi_kernel(DevPlan P, DevRes R, const MlFrag* __restrict__ fr, int nfr, long long blocks,
                     float* __restrict__ scratch) {
  using S = MlShape<D>;
  constexpr int d = S::LG, LW = S::LW, RH = S::RH, NW = S::NW, NG = S::NG, KP = D * D;
  extern __shared__ __align__(16) float2 smc[];
  const int lt = threadIdx.x % S::TPB, wl = lt % LW, wk = lt / LW;
  const long long at = (long long)blockIdx.x * S::BPC + threadIdx.x / S::TPB;
  const bool live = at < blocks;                 // a CTA's spare blocks repeat the last one and write nothing
  const long long blk = live ? at : blocks - 1;
  char* base = reinterpret_cast<char*>(smc) + (size_t)(threadIdx.x / S::TPB) * (ml_jacobi_smem<D>() / S::BPC);
  float2* X = reinterpret_cast<float2*>(base);       // the exchange buffer; it holds the block to begin with
  float* nx = reinterpret_cast<float*>(X + KP);      // the column norms beside it
  const MlFrag& mf = fr[ml_find(fr, nfr, blk)];
  const FragDev& F = P.frags[mf.frag];
  const int o = (int)(blk - mf.blk0);
  const unsigned inmask = input_mask(F);

  // the block's row of T_f (a hub's operand is stored by preparation digit s
  // at its input slots: I = Q0 + Q1, X = 2 Q2 - Q0 - Q1, Y = 2 Q3 - Q0 - Q1,
  // Z = Q0 - Q1)
  const bool hub = mf.hub != 0;      // (barriers stay outside of it: two blocks may share a warp)
  if (!hub) {
    const float* src = R.T + F.T_off + ((long long)o << (2 * d));
    for (int i = lt; i < KP; i += S::TPB) X[i] = make_float2(src[i], 0.f);
  } else {
    const long long Mo = 1ll << F.m;
    if (mf.i16) {
      const int16_t* q = reinterpret_cast<const int16_t*>(R.TQ + F.T_off) + o;
#pragma unroll 8
      for (int i = lt; i < KP; i += S::TPB) X[i] = make_float2((float)q[(long long)i * Mo] * R.hub_scale, 0.f);
    } else {
      const float* q = R.TQ + F.T_off + o;
#pragma unroll 8
      for (int i = lt; i < KP; i += S::TPB) X[i] = make_float2(q[(long long)i * Mo], 0.f);
    }
  }
  S::sync();
  for (int j = 0; j < d; ++j) {
    if (hub && ((inmask >> j) & 1)) {
      const int st = 1 << (2 * j);
      for (int g = lt; g < KP / 4; g += S::TPB) {
        float2* x = X + (((g >> (2 * j)) << (2 * j + 2)) | (g & (st - 1)));
        const float q0 = x[0].x, q1 = x[st].x, q2 = x[2 * st].x, q3 = x[3 * st].x;
        x[0].x = q0 + q1;
        x[st].x = 2.f * q2 - q0 - q1;
        x[2 * st].x = 2.f * q3 - q0 - q1;
        x[3 * st].x = q0 - q1;
      }
    }
    S::sync();
  }
  pauli_to_block<D>(X, inmask, lt);

  float* ev = scratch + mf.ev_off + (long long)o * D;
  float2* vec = reinterpret_cast<float2*>(scratch + mf.vec_off) + (long long)o * D * D;
  // columns 4 w .. of worker w's top group, 4 (NG - 1 - w) .. of its bottom
  // one; row pair h of a lane is rows 2 (wl + h LW) and the next
  MlCol<RH> g[8];
  float nr[8];
  const float scale = 1.f / (float)D;
  float mean = 0.f;                                  // tr J / D
#pragma unroll 8
  for (int i = 0; i < D; ++i) mean += X[3 * spread6(i)].x;
  mean *= scale * scale;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int col = i < 4 ? 4 * wk + i : 4 * (NG - 1 - wk) + i - 4;
#pragma unroll
    for (int h = 0; h < RH; ++h) {
      const int r = 2 * (wl + h * LW);
      float4 x = *reinterpret_cast<const float4*>(X + (spread6(r) | (spread6(col) << 1)));
      x = make_float4(x.x * scale, x.y * scale, x.z * scale, x.w * scale);
      g[i].x[h] = pk(col == r ? x.x - mean : x.x, col == r + 1 ? x.z - mean : x.z);
      g[i].y[h] = pk(x.y, x.w);
      if (live) *reinterpret_cast<float4*>(vec + col * D + r) = x;      // J's columns, read again at the end
    }
  }
  column_norms<D>(g, nr);
  if (wl < 8) {
    float mine = nr[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) mine = wl == i ? nr[i] : mine;
    nx[8 * wk + wl] = mine;
  }
  S::sync();
  float fro = 0.f;
#pragma unroll 8
  for (int i = 0; i < D; ++i) fro += nx[i];
  // G = H / |H|_F + I: norms of order one whatever the block's scale.  A block that is
  // scalar to rounding, |H|_F <= 2^-24 |J|_F (|J|_F^2 = |H|_F^2 + D mean^2), or zero
  // has the unit vectors
  const bool scalar = fro <= 3.5527137e-15f * ((float)D * mean * mean);
  const float inv_fro = scalar ? 0.f : 1.f / sqrtf(fro);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int col = i < 4 ? 4 * wk + i : 4 * (NG - 1 - wk) + i - 4;
    const f2 s2 = pk(inv_fro, inv_fro);
#pragma unroll
    for (int h = 0; h < RH; ++h) {
      const int r = 2 * (wl + h * LW);
      g[i].x[h] = fma2(g[i].x[h], s2, pk(col == r ? 1.f : 0.f, col == r + 1 ? 1.f : 0.f));
      g[i].y[h] = mul2(g[i].y[h], s2);
    }
  }
  // the tournament: top group 0 stays, the others move one place round
  const int to_top = wk == 0 ? 0 : wk + 1 < NW ? wk + 1 : NW + wk;
  const int to_bot = wk == 0 ? 1 : NW + wk - 1;
  for (int sweep = 0; sweep < kMlMaxSweeps; ++sweep) {
    bool more = false;
    column_norms<D>(g, nr);
    for (int round = 0; round < NG - 1; ++round) {
      if (round == 0) {   // the pairs within each group, once a sweep
        jacobi_step<D, 0, 1, 2, 3, 4, 5, 6, 7>(g, nr, more);
        jacobi_step<D, 0, 2, 1, 3, 4, 6, 5, 7>(g, nr, more);
        jacobi_step<D, 0, 3, 1, 2, 4, 7, 5, 6>(g, nr, more);
      }
      jacobi_step<D, 0, 4, 1, 5, 2, 6, 3, 7>(g, nr, more);
      jacobi_step<D, 0, 5, 1, 6, 2, 7, 3, 4>(g, nr, more);
      jacobi_step<D, 0, 6, 1, 7, 2, 4, 3, 5>(g, nr, more);
      jacobi_step<D, 0, 7, 1, 4, 2, 5, 3, 6>(g, nr, more);
      // (an exchanged row pair is kept as its two real, then its two imaginary parts)
      S::sync();          // the previous round's columns are read
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < RH; ++h)
          *reinterpret_cast<ulonglong2*>(X + (4 * (i < 4 ? to_top : to_bot) + (i & 3)) * D + 2 * (wl + h * LW)) =
              make_ulonglong2(g[i].x[h], g[i].y[h]);
      if (wl == 0) *reinterpret_cast<float4*>(nx + 4 * to_top) = make_float4(nr[0], nr[1], nr[2], nr[3]);
      if (wl == 1) *reinterpret_cast<float4*>(nx + 4 * to_bot) = make_float4(nr[4], nr[5], nr[6], nr[7]);
      S::sync();
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < RH; ++h) {
          const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(
              X + (4 * (i < 4 ? wk : NW + wk) + (i & 3)) * D + 2 * (wl + h * LW));
          g[i].x[h] = x.x;
          g[i].y[h] = x.y;
        }
      const float4 n0 = *reinterpret_cast<const float4*>(nx + 4 * wk);
      const float4 n1 = *reinterpret_cast<const float4*>(nx + 4 * (NW + wk));
      nr[0] = n0.x; nr[1] = n0.y; nr[2] = n0.z; nr[3] = n0.w;
      nr[4] = n1.x; nr[5] = n1.y; nr[6] = n1.z; nr[7] = n1.w;
    }
    const bool go = S::NT <= 32 ? __any_sync(0xffffffffu, more) : __syncthreads_or(more);
    if (!go) break;
  }
  // unit eigenvectors v_k, in any order, and their eigenvalues as Rayleigh
  // quotients of the block itself: |H|_F (|g_k| - 1) would carry the rounding
  // of the rotations of columns of length one and more (three times the error)
  column_norms<D>(g, nr);
  S::sync();                      // the exchange buffer is free
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = 8 * wk + i;
    const float is = 1.f / sqrtf(nr[i]);
    const f2 s2 = pk(is, is);
#pragma unroll
    for (int h = 0; h < RH; ++h) {
      const int r = 2 * (wl + h * LW);
      if (scalar) {
        g[i].x[h] = pk(k == r ? 1.f : 0.f, k == r + 1 ? 1.f : 0.f);
        g[i].y[h] = pk(0.f, 0.f);
      } else {
        g[i].x[h] = mul2(g[i].x[h], s2);
        g[i].y[h] = mul2(g[i].y[h], s2);
      }
    }
  }
  for (int e = lt; e < KP / 2; e += S::TPB) {       // J's columns, row pairs split like the workers' columns
    const float4 x = reinterpret_cast<const float4*>(vec)[e];
    reinterpret_cast<float4*>(X)[e] = make_float4(x.x, x.z, x.y, x.w);
  }
  S::sync();
  float lam[8], la, lb;
#pragma unroll
  for (int half = 0; half < 2; ++half) {            // y_k = J v_k for four columns at a time
    MlCol<RH> y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int h = 0; h < RH; ++h) y[i].x[h] = y[i].y[h] = pk(0.f, 0.f);
#pragma unroll
    for (int hc = 0; hc < 2 * RH; ++hc)             // component c = 2 (w + (hc / 2) LW) + hc % 2 lies with lane w
#pragma unroll 1
      for (int w = 0; w < LW; ++w) {
        const int c = 2 * (w + (hc / 2) * LW) + (hc & 1);
        ulonglong2 j[RH];
#pragma unroll
        for (int h = 0; h < RH; ++h)
          j[h] = *reinterpret_cast<const ulonglong2*>(X + c * D + 2 * (wl + h * LW));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 gx = upk(g[4 * half + i].x[hc / 2]), gy = upk(g[4 * half + i].y[hc / 2]);
          const float a = __shfl_sync(0xffffffffu, (hc & 1) ? gx.y : gx.x, w, LW);
          const float b = __shfl_sync(0xffffffffu, (hc & 1) ? gy.y : gy.x, w, LW);
          const f2 vx = pk(a, a), vy = pk(b, b), my = pk(-b, -b);
#pragma unroll
          for (int h = 0; h < RH; ++h) {
            y[i].x[h] = fma2(j[h].y, my, fma2(j[h].x, vx, y[i].x[h]));
            y[i].y[h] = fma2(j[h].x, vy, fma2(j[h].y, vx, y[i].y[h]));
          }
        }
      }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const auto& v = g[4 * half + i];
      f2 s = fma2(v.y[0], y[i].y[0], mul2(v.x[0], y[i].x[0]));
#pragma unroll
      for (int h = 1; h < RH; ++h) s = fma2(v.y[h], y[i].y[h], fma2(v.x[h], y[i].x[h], s));
      const float2 t = upk(s);
      lam[4 * half + i] = t.x + t.y;
    }
  }
  reduce_pairs<LW>(lam, la, lb);
  if (!live) return;
  if ((wl & (LW / 4 - 1)) == 0) {         // the first lane of each quarter has two of the eight sums
    const int q = wl / (LW / 4);
    ev[8 * wk + 2 * q] = la;
    ev[8 * wk + 2 * q + 1] = lb;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)             // entry [k][r] = component r of vector k
#pragma unroll
    for (int h = 0; h < RH; ++h) {
      const float2 x = upk(g[i].x[h]), y = upk(g[i].y[h]);
      *reinterpret_cast<float4*>(vec + (8 * wk + i) * D + 2 * (wl + h * LW)) = make_float4(x.x, y.x, x.y, y.y);
    }
}

// The rebuilt block and T' row of those sizes: J' = sum_k (sqrt(l_k) v_k)
// (sqrt(l_k) v_k)^H over the live eigenvalues, a 4 x 4 block of J' per thread
// (4 LDS.128 per 64 FMA), then slot by slot to Pauli digits.  One entry per
// thread with two loads per term, and 2^d terms per T' entry, took 1.72 ms on
// 768 blocks of 64 x 64, 0.067 ms so.
template <int D>
constexpr size_t ml_rebuild_tile_smem() {
  return (size_t)MlTile<D>::BPC * (D * D * sizeof(float2) + 2 * D * sizeof(float));
}

template <int D>
__global__ void __launch_bounds__(MlTile<D>::NT) ml_rebuild_tile_kernel(DevPlan P, DevRes R,
                                                                         const MlFrag* __restrict__ fr, int nfr,
                                                                         long long blocks,
                                                                         const float* __restrict__ scratch,
                                                                         const double* __restrict__ theta) {
  using S = MlTile<D>;
  constexpr int d = MlShape<D>::LG, KP = D * D;
  extern __shared__ __align__(16) float2 smc[];
  const int lt = threadIdx.x % S::TPB;
  const long long at = (long long)blockIdx.x * S::BPC + threadIdx.x / S::TPB;
  const bool wr = at < blocks;
  const long long blk = wr ? at : blocks - 1;
  char* base = reinterpret_cast<char*>(smc) + (size_t)(threadIdx.x / S::TPB) * (ml_rebuild_tile_smem<D>() / S::BPC);
  float2* V = reinterpret_cast<float2*>(base);       // live rows first, scaled; then J' by slot digits
  float* lam = reinterpret_cast<float*>(V + KP);     // sqrt of the clipped eigenvalues
  int* row = reinterpret_cast<int*>(lam + D);        // rows of the live ones
  const MlFrag& mf = fr[ml_find(fr, nfr, blk)];
  const FragDev& F = P.frags[mf.frag];
  const int o = (int)(blk - mf.blk0);
  const unsigned inmask = input_mask(F);
  const float th = (float)theta[mf.index];
  const float* ev = scratch + mf.ev_off + (long long)o * D;
  const float2* vec = reinterpret_cast<const float2*>(scratch + mf.vec_off) + (long long)o * D * D;
  for (int i = lt; i < D; i += S::TPB) lam[i] = sqrtf(fmaxf(ev[i] - th, 0.f));
  S::sync();
  int nl = 0;
#pragma unroll 8
  for (int i = 0; i < D; ++i) {
    if (lam[i] > 0.f) {
      if (lt == 0) row[nl] = i;
      ++nl;
    }
  }
  S::sync();
  for (int e = lt; e < nl * (D / 2); e += S::TPB) {
    const int k = row[e / (D / 2)], r = 2 * (e % (D / 2));
    const float l = lam[k];
    const float4 x = *reinterpret_cast<const float4*>(vec + (long long)k * D + r);
    *reinterpret_cast<float4*>(V + (e / (D / 2)) * D + r) = make_float4(l * x.x, l * x.y, l * x.z, l * x.w);
  }
  S::sync();
  const int r0 = 4 * (lt % (D / 4)), c0 = 4 * (lt / (D / 4));
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  for (int k = 0; k < nl; ++k) {
    const float4 a01 = *reinterpret_cast<const float4*>(V + k * D + r0);
    const float4 a23 = *reinterpret_cast<const float4*>(V + k * D + r0 + 2);
    const float4 b01 = *reinterpret_cast<const float4*>(V + k * D + c0);
    const float4 b23 = *reinterpret_cast<const float4*>(V + k * D + c0 + 2);
    const float2 a[4] = {make_float2(a01.x, a01.y), make_float2(a01.z, a01.w), make_float2(a23.x, a23.y),
                         make_float2(a23.z, a23.w)};
    const float2 b[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w), make_float2(b23.x, b23.y),
                         make_float2(b23.z, b23.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][j].x = fmaf(a[i].y, b[j].y, fmaf(a[i].x, b[j].x, acc[i][j].x));
        acc[i][j].y = fmaf(-a[i].x, b[j].y, fmaf(a[i].y, b[j].x, acc[i][j].y));
      }
  }
  S::sync();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) V[spread6(r0 + i) | (spread6(c0 + j) << 1)] = acc[i][j];
  S::sync();
  block_to_pauli<D>(V, inmask, lt);
  if (wr) {
    float* dst = R.T + F.T_off + ((long long)o << (2 * d));
    for (int i = lt; i < KP; i += S::TPB) dst[i] = V[i].x;
  }
  // the hub's operand by preparation at its inputs: (I + Z)/2, (I - Z)/2, (I + X)/2, (I + Y)/2
  const bool hub = mf.hub != 0;
  for (int j = 0; j < d; ++j) {
    S::sync();
    if (hub && ((inmask >> j) & 1)) {
      const int st = 1 << (2 * j);
      for (int g = lt; g < KP / 4; g += S::TPB) {
        float2* x = V + (((g >> (2 * j)) << (2 * j + 2)) | (g & (st - 1)));
        const float tI = x[0].x, tX = x[st].x, tY = x[2 * st].x, tZ = x[3 * st].x;
        x[0].x = 0.5f * (tI + tZ);
        x[st].x = 0.5f * (tI - tZ);
        x[2 * st].x = 0.5f * (tI + tX);
        x[3 * st].x = 0.5f * (tI + tY);
      }
    }
  }
  S::sync();
  if (hub && wr) {
    const long long Mo = 1ll << F.m;
    float* q = R.TQ + F.T_off + o;
    for (int i = lt; i < KP; i += S::TPB) q[(long long)i * Mo] = V[i].x;
  }
}

template <int D>
static cudaError_t launch_jacobi(const DevPlan& p, const DevRes& r, const MlFrag* fr, const MlGroup& G, float* scratch,
                                 cudaStream_t s) {
  using S = MlShape<D>;
  const size_t sm = ml_jacobi_smem<D>();
  cudaError_t err = cudaFuncSetAttribute(ml_jacobi_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (err != cudaSuccess) return err;
  ml_jacobi_kernel<D><<<(unsigned)((G.blocks + S::BPC - 1) / S::BPC), S::NT, sm, s>>>(p, r, fr, G.count, G.blocks,
                                                                                    scratch);
  note_launch();
  return cudaGetLastError();
}

template <int D>
static cudaError_t launch_rebuild_tile(const DevPlan& p, const DevRes& r, const MlFrag* fr, const MlGroup& G,
                                       const float* scratch, const double* theta, cudaStream_t s) {
  using S = MlTile<D>;
  const size_t sm = ml_rebuild_tile_smem<D>();
  cudaError_t err =
      cudaFuncSetAttribute(ml_rebuild_tile_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (err != cudaSuccess) return err;
  ml_rebuild_tile_kernel<D><<<(unsigned)((G.blocks + S::BPC - 1) / S::BPC), S::NT, sm, s>>>(p, r, fr, G.count,
                                                                                          G.blocks, scratch, theta);
  note_launch();
  return cudaGetLastError();
}

size_t ml_eig_smem(int d) {
  const size_t D = 1u << d, LD = D + 1, KP = 1u << (2 * d), H = D / 2;
  const size_t v_floats = 2 * D * LD > KP ? 2 * D * LD : KP;   // V shares its space with the T_f row
  return 2 * D * LD * sizeof(float) + v_floats * sizeof(float) + 8 * (H + 1) * sizeof(float) +
         2 * (H + 1) * sizeof(int) + (H * (H + 1) / 2 + 1) * sizeof(int);
}
size_t ml_rebuild_smem(int d) {
  const size_t D = 1u << d, LD = D + 1, KP = 1u << (2 * d);
  return (4 * D * LD + D + KP + D) * sizeof(float);
}

// Eigendecompositions (theta null) or rebuilt blocks of one group.
static cudaError_t launch_ml_group(const DevPlan& p, const DevRes& r, const MlFrag* fr, const MlGroup& G, float* scratch,
                                   const double* theta, cudaStream_t s) {
  switch (G.d) {      // blocks of 16 rows and more: columns in registers
    case 4: return theta ? launch_rebuild_tile<16>(p, r, fr, G, scratch, theta, s) : launch_jacobi<16>(p, r, fr, G, scratch, s);
    case 5: return theta ? launch_rebuild_tile<32>(p, r, fr, G, scratch, theta, s) : launch_jacobi<32>(p, r, fr, G, scratch, s);
    case 6: return theta ? launch_rebuild_tile<64>(p, r, fr, G, scratch, theta, s) : launch_jacobi<64>(p, r, fr, G, scratch, s);
    default: break;
  }
  if (theta) ml_rebuild_kernel<<<(unsigned)G.blocks, 64, ml_rebuild_smem(G.d), s>>>(p, r, fr, G.count, G.d, scratch, theta);
  else ml_eig_kernel<<<(unsigned)G.blocks, 64, ml_eig_smem(G.d), s>>>(p, r, fr, G.count, G.d, scratch);
  note_launch();
  return cudaGetLastError();
}

// The groups are independent: the one with the largest blocks runs on `s`, the
// others beside it on the side stream (their launches do not fill the chip, and
// the large one ends in a partial wave), joined before the thresholds and at
// the end.
cudaError_t launch_ml_correct(const DevPlan& p, const DevRes& r, const MlFrag* d_frags, int n_frags,
                              const MlGroup* groups, int n_groups, float* scratch, double* theta, cudaStream_t s,
                              const SideStream& side) {
  cudaError_t err = cudaSuccess;
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1) {
      ml_threshold_kernel<<<n_frags, kThetaThreads, 0, s>>>(p, d_frags, scratch, theta);
      note_launch();
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    const bool fork = n_groups > 1;
    if (fork) {
      if ((err = cudaEventRecord(side.fork, s)) != cudaSuccess) return err;
      if ((err = cudaStreamWaitEvent(side.stream, side.fork, 0)) != cudaSuccess) return err;
    }
    for (int g = n_groups - 1; g >= 0 && err == cudaSuccess; --g)     // groups are in order of d
      err = launch_ml_group(p, r, d_frags + groups[g].first, groups[g], scratch, pass ? theta : nullptr,
                            g == n_groups - 1 ? s : side.stream);
    if (fork) {      // joined on a failed launch too: nothing stays in flight beside `s`
      cudaError_t e = cudaEventRecord(side.join, side.stream);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s, side.join, 0);
      if (err == cudaSuccess) err = e;
    }
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

}  // namespace ccs
