// Non-Clifford fragments (K4): complex64 statevectors of 2^n amplitudes in
// shared memory (the paper hands these fragments to an exact statevector
// simulator, Sec. V-B).  A variant is (preparations, the fragment's gates U,
// output basis changes), so an item (one preparation combination and a
// range of basis combinations) runs U once and then applies each basis
// combination's changes on the way out.  Gates arrive fused into 2x2 / 4x4
// unitaries.
//
// A fused op is applied in place, one group of four amplitudes (two for a
// one-qubit op) per thread: 4 loads, 88 FP32 operations and 4 stores, the next
// op's places and matrix prepared while this op's amplitudes are on their way;
// one amplitude per thread from one buffer to the other read every amplitude
// four times.  A fragment is a chain of such steps, bound by their latency;
// in a batch the instructions per step decide how much of the chip is taken
// from the Clifford branch beside it (64 circuits: 194 us beside it before,
// 72 us so; one 100-qubit circuit: 32 us before, 24.8 us so).  Amplitudes are stored at swz(i), so that
// the groups of a half warp fall on distinct 8-byte banks for nearly every pair
// of wires.
// Outputs per variant: the exact marginal on A_f and the Z-string values, both
// reduced in a fixed order (deterministic).
#include "kernels.cuh"

namespace ccs {

namespace {

__device__ __forceinline__ unsigned insert_zero(unsigned t, int pos) {
  return ((t >> pos) << (pos + 1)) | (t & ((1u << pos) - 1u));
}

// Storage place of amplitude i: bits 4 and 5 folded into the low four (linear
// over XOR).  Any four of the low six bits but three of the fifteen sets then
// map to all sixteen 8-byte banks.
__device__ __forceinline__ unsigned swz(unsigned i) {
  return i ^ ((0u - ((i >> 4) & 1u)) & 7u) ^ ((0u - ((i >> 5) & 1u)) & 14u);
}

// (re + i im) a, one product rounded, the other fused; sums of two and of four
// such products in a fixed order.  The rounding is spelled out because exact
// cancellations between amplitudes have to stay exact: the Z-string values that
// vanish then do.
__device__ __forceinline__ float2 cmul(float re, float im, float2 a) {
  return make_float2(__fmaf_rn(re, a.x, -__fmul_rn(im, a.y)), __fmaf_rn(re, a.y, __fmul_rn(im, a.x)));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}

// One-qubit op on wire a from src to dst (which may be the same buffer): M
// row-major, M[r][c] at m[2 (2 r + c)].
__device__ __forceinline__ void apply_1q(const float2* src, float2* dst, unsigned N, int a, const float* m) {
  const unsigned sa = swz(1u << a);
  for (unsigned t = threadIdx.x; t < (N >> 1); t += blockDim.x) {
    const unsigned p0 = swz(insert_zero(t, a)), p1 = p0 ^ sa;
    const float2 x0 = src[p0], x1 = src[p1];
    dst[p0] = cadd(cmul(m[0], m[1], x0), cmul(m[2], m[3], x1));
    dst[p1] = cadd(cmul(m[4], m[5], x0), cmul(m[6], m[7], x1));
  }
}

// Where an op's groups lie: group t's first amplitude has t's bits around zeros
// at the op's wires; sa, sb lead to its other members.
struct OpPlace {
  unsigned sa, sb;          // places of the wires' bits
  unsigned m1, m2;          // t's bits below both wires, between them (those above: the rest)
  unsigned one;             // one-qubit op: its wire + 1, else 0
  __device__ __forceinline__ unsigned group(unsigned t) const {
    return swz((t & m1) | ((t & m2) << 1) | ((t & ~(m1 | m2)) << 2));
  }
};
__device__ __forceinline__ OpPlace op_place(int a, int b) {
  OpPlace p{};
  if (b < 0) {
    p.one = (unsigned)a + 1u;
    return p;
  }
  const int lo = min(a, b), hi = max(a, b);
  p.sa = swz(1u << a);
  p.sb = swz(1u << b);
  p.m1 = (1u << lo) - 1u;
  p.m2 = ((1u << (hi - 1)) - 1u) & ~p.m1;
  return p;
}

// A row of a two-qubit op on its group of four amplitudes: local index c =
// bit_a + 2 bit_b, (re, im) of M[r][0], M[r][1] and of M[r][2], M[r][3].
__device__ __forceinline__ float2 row_2q(const float4& m01, const float4& m23, float2 x0, float2 x1, float2 x2, float2 x3) {
  return cadd(cadd(cmul(m01.x, m01.y, x0), cmul(m01.z, m01.w, x1)), cadd(cmul(m23.x, m23.y, x2), cmul(m23.z, m23.w, x3)));
}

__device__ __forceinline__ int digit_in(int v, int i) {
  for (int t = 0; t < i; ++t) v /= 4;
  return v % 4;
}
__device__ __forceinline__ int digit_out(int v, int qin, int i) {
  for (int t = 0; t < qin; ++t) v /= 4;
  for (int t = 0; t < i; ++t) v /= 3;
  return v % 3;
}

}  // namespace

// States of at most this many wires take four lanes per group (kernel times, one
// lane and four: 13 ops on 4 wires 9.9 and 8.9 us, 25 on 6 13.2 and 9.3 us, 31 on
// 7 14.7 and 9.8 us, 37 on 8 14.9 and 12.1 us); at 9 wires the two were equal.
constexpr int kSmallState = 8;
constexpr int kOpStage = 128;   // fused ops staged in shared memory at a time
constexpr int kZChunk = 256;    // Z-string masks built per pass

// LPG: lanes of a group (1, or 4 where the whole state is a warp's or two).
template <int LPG>
__global__ void __launch_bounds__(512) statevector_kernel(DevPlan P, DevRes R, int max_n) {
  extern __shared__ __align__(16) float2 sv_smem[];
  float2* psi = sv_smem;                                   // the state
  float2* wk = sv_smem + (1u << max_n);                    // a copy under basis changes
  float* pr = reinterpret_cast<float*>(sv_smem + (2u << max_n));              // probabilities
  float* mat_s = pr + (2u << max_n);                       // [op][32]
  OpPlace* pl_s = reinterpret_cast<OpPlace*>(mat_s + 32 * kOpStage);
  __shared__ int s_item;
  __shared__ unsigned s_abit[kMaxMeas];     // bit of each A wire in the amplitude index
  __shared__ unsigned s_zm[kZChunk];        // Z masks of a chunk of Z-strings
  __shared__ unsigned s_qm[kMaxCuts];       // bit of each quantum output
  __shared__ float s_part[16];              // marginal partial sums, one per warp
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  // the first item by block index, further ones from a counter
  for (int item = blockIdx.x; item < P.n_items_nc;) {
    const int2 it = P.items_nc[item];
    const FragDev& F = P.frags[it.x];
    const int n = F.n, qin = F.qin, qout = F.qout, nA = F.nA, nz = F.nz;
    const int n_prep = 1 << (2 * qin), n_basis = F.nv / n_prep;
    const int pc = it.y % n_prep, b0 = it.y / n_prep, b1 = min(n_basis, b0 + P.nc_basis_chunk);
    const unsigned N = 1u << n;
    const int op0 = P.moments[F.mom_off], op1 = P.moments[F.mom_off + F.n_moments];
    // a chunk of ops on its way to shared memory: the matrices as asynchronous
    // copies of 8 bytes (all in flight at once; plain loads in a loop: 29.9 us
    // for a 100-qubit circuit's kernel, 24.8 us so; with nothing cached the
    // stage 41.8 and 31.8 us), the wires as places
    auto stage = [&](int c0, int cnt) {
      static_assert(sizeof(NCOp) == 17 * 8, "two wires, then the matrix");
      const NCOp* src = P.nops + F.ops_off + c0;
      for (int i = tid; i < cnt * 16; i += blockDim.x) {
        const int o = i >> 4, w = 2 * (i & 15);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(mat_s + 32 * o + w)),
                     "l"(src[o].m + w)
                     : "memory");
      }
      for (int o = tid; o < cnt; o += blockDim.x) {
        const int2 ab = *reinterpret_cast<const int2*>(src + o);
        pl_s[o] = op_place(ab.x, ab.y);
      }
    };
    stage(op0, min(kOpStage, op1 - op0));      // beside the loads of the preparation and the masks
    {   // the prepared product state: amplitude i is the product of its inputs' entries
      unsigned inb = 0;
      for (int o = 0; o < qin; ++o) inb |= 1u << P.wires[F.qin_off + o];
      for (unsigned i = tid; i < N; i += blockDim.x) {
        float2 x = make_float2((i & ~inb) ? 0.f : 1.f, 0.f);
        if (!(i & ~inb))
          for (int o = 0; o < qin; ++o) {
            const float* m = P.prep_mats + 8 * digit_in(pc, o) + 4 * ((i >> P.wires[F.qin_off + o]) & 1u);
            x = cmul(m[0], m[1], x);
          }
        psi[swz(i)] = x;
      }
    }
    for (int j = tid; j < nA; j += blockDim.x) s_abit[j] = 1u << P.wires[F.A_off + j];
    for (int o = tid; o < qout; o += blockDim.x) s_qm[o] = 1u << P.wires[F.qout_off + o];
    auto z_masks = [&](int z0, int zc) {
      for (int k = tid; k < zc; k += blockDim.x) {
        unsigned zm = 0;
        for (int q = P.zoffs[F.zw_off + z0 + k]; q < P.zoffs[F.zw_off + z0 + k + 1]; ++q) zm ^= 1u << P.wires[q];
        s_zm[k] = zm;
      }
    };
    const bool z_once = nz <= kZChunk;     // one chunk: its masks before the ops, beside the other loads
    if (z_once) z_masks(0, nz);
    for (int c0 = op0; c0 < op1; c0 += kOpStage) {
      const int cnt = min(kOpStage, op1 - c0);
      if (c0 != op0) stage(c0, cnt);
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      // the next op's places and matrix are prepared while this op's amplitudes
      // are on their way
      const unsigned groups = N >> 2;
      OpPlace pl = pl_s[0], pl1 = pl_s[min(1, cnt - 1)];
      if constexpr (LPG == 4) {            // every group of the state at once (N <= the threads)
        const int r = tid & 3;
        const unsigned t = (unsigned)tid >> 2;
        auto row = [&](int o, int h) -> float4 { return *reinterpret_cast<const float4*>(mat_s + 32 * o + 8 * r + 4 * h); };
        float4 m01 = row(0, 0), m23 = row(0, 1);
        unsigned p0 = pl.group(t);
        for (int o = 0; o < cnt; ++o) {
          const OpPlace pl2 = pl_s[min(o + 2, cnt - 1)];
          const int nx = min(o + 1, cnt - 1);
          if (pl.one) {
            apply_1q(psi, psi, N, (int)pl.one - 1, mat_s + 32 * o);
          } else {
            float2 x0, x1, x2, x3;
            if (t < groups) { x0 = psi[p0]; x1 = psi[p0 ^ pl.sa]; x2 = psi[p0 ^ pl.sb]; x3 = psi[p0 ^ pl.sa ^ pl.sb]; }
            __syncwarp();                  // a group's four lanes have read it
            if (t < groups)
              psi[p0 ^ ((r & 1) ? pl.sa : 0u) ^ ((r & 2) ? pl.sb : 0u)] = row_2q(m01, m23, x0, x1, x2, x3);
          }
          m01 = row(nx, 0);
          m23 = row(nx, 1);
          p0 = pl1.group(t);
          pl = pl1;
          pl1 = pl2;
          __syncthreads();
        }
      } else {
        float4 m[8];
        auto fetch = [&](int o) {
#pragma unroll
          for (int i = 0; i < 8; ++i) m[i] = *reinterpret_cast<const float4*>(mat_s + 32 * o + 4 * i);
        };
        unsigned p0 = pl.group(tid);
        fetch(0);
        for (int o = 0; o < cnt; ++o) {
          const OpPlace pl2 = pl_s[min(o + 2, cnt - 1)];
          unsigned n0 = 0;
          if (pl.one) {
            apply_1q(psi, psi, N, (int)pl.one - 1, mat_s + 32 * o);
            n0 = pl1.group(tid);
          } else {
            unsigned t = tid;
            float2 x0, x1, x2, x3;
            if (t < groups) { x0 = psi[p0]; x1 = psi[p0 ^ pl.sa]; x2 = psi[p0 ^ pl.sb]; x3 = psi[p0 ^ pl.sa ^ pl.sb]; }
            n0 = pl1.group(tid);
            while (t < groups) {
              const float2 y0 = row_2q(m[0], m[1], x0, x1, x2, x3), y1 = row_2q(m[2], m[3], x0, x1, x2, x3);
              const float2 y2 = row_2q(m[4], m[5], x0, x1, x2, x3), y3 = row_2q(m[6], m[7], x0, x1, x2, x3);
              psi[p0] = y0;
              psi[p0 ^ pl.sa] = y1;
              psi[p0 ^ pl.sb] = y2;
              psi[p0 ^ pl.sa ^ pl.sb] = y3;
              t += blockDim.x;
              if (t >= groups) break;
              p0 = pl.group(t);
              x0 = psi[p0]; x1 = psi[p0 ^ pl.sa]; x2 = psi[p0 ^ pl.sb]; x3 = psi[p0 ^ pl.sa ^ pl.sb];
            }
          }
          if (o + 1 < cnt) fetch(o + 1);
          pl = pl1;
          pl1 = pl2;
          p0 = n0;
          __syncthreads();
        }
      }
    }
    if (op0 == op1) __syncthreads();
    // U |prep> stays in psi; each basis combination changes a copy, its last
    // output on the way to the probabilities
    unsigned amask = 0;
    for (int j = 0; j < nA; ++j) amask |= s_abit[j];
    const unsigned rest = (N - 1) & ~amask;
    const unsigned ncomp = 1u << (n - nA);
    // the completions c of an outcome: bits of c at the positions of `rest`,
    // the five low bits by lane
    unsigned dep_lane = 0, rest_hi = rest;
    for (int k = 0; k < 5 && rest_hi; ++k, rest_hi &= rest_hi - 1)
      if ((lane >> k) & 1) dep_lane |= rest_hi & (0u - rest_hi);
    const int parts = max(1, nwarps >> nA);     // warps per outcome
    for (int bc = b0; bc < b1; ++bc) {
      const int v = pc + n_prep * bc;
      const float2* cur = psi;
      for (int o = 0; o + 1 < qout; ++o) {
        apply_1q(cur, wk, N, P.wires[F.qout_off + o], P.basis_mats + 8 * digit_out(v, qin, o));
        __syncthreads();
        cur = wk;
      }
      if (qout > 0) {
        const int a = P.wires[F.qout_off + qout - 1];
        const float* m = P.basis_mats + 8 * digit_out(v, qin, qout - 1);
        const unsigned sa = swz(1u << a);
        for (unsigned t = tid; t < (N >> 1); t += blockDim.x) {
          const unsigned i0 = insert_zero(t, a), p0 = swz(i0);
          const float2 x0 = cur[p0], x1 = cur[p0 ^ sa];
          const float2 y0 = cadd(cmul(m[0], m[1], x0), cmul(m[2], m[3], x1));
          const float2 y1 = cadd(cmul(m[4], m[5], x0), cmul(m[6], m[7], x1));
          pr[i0] = __fmaf_rn(y0.x, y0.x, __fmul_rn(y0.y, y0.y));
          pr[i0 | (1u << a)] = __fmaf_rn(y1.x, y1.x, __fmul_rn(y1.y, y1.y));
        }
      } else {
        for (unsigned i = tid; i < N; i += blockDim.x) {
          const float2 x = cur[swz(i)];
          pr[i] = __fmaf_rn(x.x, x.x, __fmul_rn(x.y, x.y));
        }
      }
      __syncthreads();
      // marginal on A: `parts` warps per outcome, lanes over its completions,
      // then a fixed shuffle tree and the warps in order
      float* d = R.dist + F.dist_off + ((long long)v << nA);
      for (unsigned y0 = 0; y0 < (1u << nA); y0 += nwarps / parts) {
        const unsigned y = y0 + warp / parts;
        float acc = 0.f;
        if (y < (1u << nA)) {
          unsigned base = dep_lane;
          for (int j = 0; j < nA; ++j)
            if ((y >> j) & 1u) base |= s_abit[j];
          const unsigned part = warp % parts;
          if (lane < ncomp)
            for (unsigned c = part; 32 * c < ncomp; c += parts) {
              unsigned idx = base, cc = c;
              for (unsigned rm = rest_hi; rm && cc; rm &= rm - 1, cc >>= 1)
                if (cc & 1u) idx |= rm & (0u - rm);
              acc += pr[idx];
            }
          for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
          if (lane == 0) {
            if (parts == 1) d[y] = acc;
            else s_part[warp] = acc;
          }
        }
      }
      if (parts > 1) {
        __syncthreads();
        if (tid < (1 << nA)) {
          float acc = s_part[tid * parts];
          for (int k = 1; k < parts; ++k) acc += s_part[tid * parts + k];
          d[tid] = acc;
        }
      }
      // Z-string values <Z_S> = sum_x (-1)^{|x & S|} p(x): the Walsh-Hadamard
      // transform of the probabilities, in place, two bits per pass
      if (nz > 0) {
        __syncthreads();
        for (int h = 0; h < n; h += 2) {
          if (h + 1 < n) {
            for (unsigned t = tid; t < (N >> 2); t += blockDim.x) {
              const unsigned i0 = insert_zero(insert_zero(t, h), h + 1), s1 = 1u << h, s2 = 2u << h;
              const float x0 = pr[i0], x1 = pr[i0 | s1], x2 = pr[i0 | s2], x3 = pr[i0 | s1 | s2];
              const float u0 = x0 + x1, u1 = x0 - x1, u2 = x2 + x3, u3 = x2 - x3;
              pr[i0] = u0 + u2;
              pr[i0 | s1] = u1 + u3;
              pr[i0 | s2] = u0 - u2;
              pr[i0 | s1 | s2] = u1 - u3;
            }
          } else {
            for (unsigned t = tid; t < (N >> 1); t += blockDim.x) {
              const unsigned i0 = insert_zero(t, h), i1 = i0 | (1u << h);
              const float x0 = pr[i0], x1 = pr[i1];
              pr[i0] = x0 + x1;
              pr[i1] = x0 - x1;
            }
          }
          __syncthreads();
        }
        for (int z0 = 0; z0 < nz; z0 += kZChunk) {
          const int zc = min(kZChunk, nz - z0);
          if (!z_once) {
            z_masks(z0, zc);
            __syncthreads();
          }
          for (int ev = tid; ev < (zc << qout); ev += blockDim.x) {
            const int k = ev >> qout, u = ev & ((1 << qout) - 1);
            unsigned zm = s_zm[k];
            for (int o = 0; o < qout; ++o)
              if ((u >> o) & 1) zm ^= s_qm[o];
            R.zval[F.zval_off + ((long long)v * nz + z0 + k) * (1 << qout) + u] = pr[zm];
          }
          __syncthreads();
        }
      }
      __syncthreads();
    }
    if (tid == 0) s_item = (int)(gridDim.x + atomicAdd(&R.work[1], 1u));
    __syncthreads();
    item = s_item;
    __syncthreads();
  }
}

cudaError_t launch_statevector(const DevPlan& p, const DevRes& r, int max_n, int threads, int grid,
                               cudaStream_t s) {
  if (p.n_items_nc == 0) return cudaSuccess;

  const size_t smem = ((size_t)24 << max_n) + (size_t)kOpStage * (32 * sizeof(float) + 5 * sizeof(unsigned));
  auto kern = (1 << max_n) <= threads && max_n <= kSmallState ? statevector_kernel<4> : statevector_kernel<1>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  kern<<<grid, threads, smem, s>>>(p, r, max_n); note_launch();
  return cudaGetLastError();
}

}  // namespace ccs
