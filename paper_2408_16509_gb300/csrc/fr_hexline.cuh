// Sum-factorised hexahedron kernels, one thread per line of solution points.
//
// A line thread reads the N values of its line once and forms all N results
// (derivative and correction) and both face values from registers, with
// coefficients that are the same for every thread (constant operands).  One
// thread per solution point, the earlier form, read every line N times and
// took lane-varying coefficients from the constant bank; the FP32 kernels
// were bound by that shared-memory traffic (L1 at 82 %, DRAM at 40 %), about
// 20 000 four-byte reads an element and kernel at p = 4 against 12 000 here.
//
// Mapping: the pointwise phases take one thread per solution point
// (le, z = a + N b + N^2 c), the line phases one per (element, direction,
// line) with the five variables in a loop; the CTA's threads serve all of its
// elements.  Fields lie in shared memory with an odd row length (FxGeom), so
// the lines of all three directions are read without bank conflicts.
//
// The gradient kernel takes the solution jump u^C - u_f from the two traces
// itself (own and partner's, TraceArgs) instead of reading the array a
// separate kernel would write, and stores the viscous flux at the solution
// points (9 values) in place of the gradient (15): together 12 KB of 59 KB
// DRAM traffic an element and stage less at p = 4.
//
// Measured per launch, 48^3 p = 4 with FP64 registers (32^3 p = 3 FP32):
// common solution and gradient 155 + 621 -> 588 us (29 + 85 -> 96), volume 657 ->
// 560 us (92 -> 71; 0.9 of its DRAM traffic at the copy rate).  The
// gradient kernel issues on 65 % of the cycles and waits for the traces on
// most of the others.
#pragma once
#include "fr_hexfx.cuh"

namespace frgb {

// threads of a CTA of eb elements
template <int N>
__host__ __device__ constexpr int hexl_threads(int eb) {
  return (eb * N * N * N + 31) / 32 * 32;
}

// Shared memory per element: gradient u [5][PN], du [5][NF], traces [5][NF]
// (q form), gradient [15][PN]; volume f~ [15][PN], F^C [5][NF].
template <typename T, int N>
__host__ __device__ constexpr int hexl_grad_bytes() {
  using G = FxGeom<N>;
  return (20 * G::PN + (sizeof(T) == 4 ? 10 : 5) * G::NF) * int(sizeof(T));
}
template <typename T, int N>
__host__ __device__ constexpr int hexl_vol_bytes() {
  using G = FxGeom<N>;
  return (15 * G::PN + 5 * G::NF) * int(sizeof(T));
}

// Lines of a CTA, numbered direction by direction (for N = 4 and an even
// number of elements a warp's 32 lines then run the same way, on distinct
// banks; padding the directions to whole warps for the other N was slower).
template <int N>
struct LineTasks {
  int per, lines;  // slots and real lines of a direction
  __device__ __forceinline__ LineTasks(int eb, int nel) : per(eb * N * N), lines(nel * N * N) {}
  __device__ __forceinline__ int count() const { return 3 * per; }
  // element, direction, first slot, stride and minus-face flux point of line
  // t; false: no element there (a ragged last CTA)
  __device__ __forceinline__ bool get(int t, int* le, int* d, int* s0, int* st, int* fm) const {
    *d = (t >= per) + (t >= 2 * per);
    const int r = t - *d * per;
    *le = r / (N * N);
    fx_line<N>(*d, r - *le * N * N, s0, st, fm);
    return r < lines;
  }
};

// values at a line's two faces (Gauss-Lobatto: the line's end points)
template <typename T, int N>
__device__ __forceinline__ void hexl_faces(const HexOps<T>& op, const T v[N], T* f0, T* f1) {
  if (op.gather) {
    *f0 = v[0];
    *f1 = v[N - 1];
    return;
  }
  T x = op.lm[0] * v[0], y = op.lp[0] * v[0];
#pragma unroll
  for (int m = 1; m < N; ++m) {
    x += op.lm[m] * v[m];
    y += op.lp[m] * v[m];
  }
  *f0 = x;
  *f1 = y;
}

// NS gradients.  FP32 values: viscous normal flux q at the flux points (the
// mass component is zero and stays as allocated); FP64: the 15 gradient
// components there.  At the solution points the viscous flux [ne][9][nu]; RAW:
// the gradient [ne][15][nu] (anti-aliased flux).
// FP32: 64 registers (1024 threads per SM; 48 spill, 80 are slower).
template <typename T, typename TR, int N, int EPB, bool RAW>
__global__ void __launch_bounds__(hexl_threads<N>(EPB), sizeof(T) == 4 ? 4 : 2)
    k_hexl_grad(long long ne, int eb, const T* __restrict__ uin, const TR* __restrict__ X,
                const __grid_constant__ TraceArgs<T> ta, const T* __restrict__ smat, const T* __restrict__ rcpdjac,
                const __grid_constant__ HexOps<T> op, T* __restrict__ grad, ViscArgs<T> va,
                const __grid_constant__ BCTab<T> bc, Phys<T> ph) {
  using G = FxGeom<N>;
  constexpr int NU = G::NU, NF = G::NF, N2 = G::N2, PN = G::PN;
  constexpr bool QV = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const long long e0 = (long long)blockIdx.x * eb;
  const int nel = int(ne - e0 < eb ? ne - e0 : eb);
  const LineTasks<N> lines(eb, nel);
  T* us = reinterpret_cast<T*>(smem_raw);  // [eb][5][PN]
  T* ds = us + eb * 5 * PN;                // [eb][5][NF]
  T* gs = ds + eb * 5 * NF;                // [eb][15][PN]
  T* fs = gs + eb * 15 * PN;               // [eb][5][NF] traces (q form)
  const int le = threadIdx.x / NU, z = threadIdx.x - le * NU;
  const bool pt = le < nel;
  const long long e = e0 + le;
  const int slot = G::slot(z % N, (z / N) % N, z / N2);
  // all loads first, the partner codes before everything else: their values
  // address the partners' traces
  constexpr int NT = (NF + NU - 1) / NU;
  TraceSide<T> side[NT];
  T own[NT][5], jmp[NT][5], uv[5], S[9], rj = T(0);
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int t = threadIdx.x + i * blockDim.x;
    if (t < nel * NF) side[i].init(ta, e0 + t / NF, t % NF, NF);
  }
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int t = threadIdx.x + i * blockDim.x;
    if (t < nel * NF) side[i].load(ta, e0 + t / NF, t % NF, NF, own[i], jmp[i]);
  }
  if (pt) {
#pragma unroll
    for (int k = 0; k < 5; ++k)
      uv[k] = uin ? uin[(e * 5 + k) * NU + z] : T(X[(e * 5 + k) * NU + z]);
#pragma unroll
    for (int r = 0; r < 9; ++r) S[r] = smat[(e * 9 + r) * NU + z];
    rj = rcpdjac[e * NU + z];
#pragma unroll
    for (int k = 0; k < 5; ++k) us[(le * 5 + k) * PN + slot] = uv[k];
  }
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int t = threadIdx.x + i * blockDim.x;
    if (t < nel * NF) {
      const int l = t / NF, f = t - l * NF;
      side[i].jump(own[i], jmp[i]);
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        ds[(l * 5 + k) * NF + f] = jmp[i][k];
        if (QV) fs[(l * 5 + k) * NF + f] = own[i][k];
      }
    }
  }
  __syncthreads();
  // reference gradient along every line, with the correction of the jumps
  // (the face normal is -e_d on the minus face)
  for (int t = threadIdx.x; t < lines.count(); t += blockDim.x) {
    int l, d, s0, st, fm;
    if (!lines.get(t, &l, &d, &s0, &st, &fm)) continue;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const T* p = us + (l * 5 + k) * PN + s0;
      T v[N];
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = p[m * st];
      const T j0 = ds[(l * 5 + k) * NF + fm], j1 = ds[(l * 5 + k) * NF + fm + N2];
      T* o = gs + (l * 15 + d * 5 + k) * PN + s0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        T g = op.gr[i] * j1 - op.gl[i] * j0;
#pragma unroll
        for (int m = 0; m < N; ++m) g += op.d1[i][m] * v[m];
        o[i * st] = g;
      }
    }
  }
  __syncthreads();
  if (pt) {
#pragma unroll
    for (int r = 0; r < 9; ++r) S[r] *= rj;
    T g[3][5];
    T* p = gs + le * 15 * PN + slot;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const T g0 = p[k * PN], g1 = p[(5 + k) * PN], g2 = p[(10 + k) * PN];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        g[j][k] = S[j] * g0 + S[3 + j] * g1 + S[6 + j] * g2;
        p[(j * 5 + k) * PN] = g[j][k];
        if (RAW) grad[(e * 15 + j * 5 + k) * NU + z] = g[j][k];
      }
    }
    if (!RAW) {
      T uz[5], tq[9];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = us[(le * 5 + k) * PN + slot];
      viscous_point(uz, g, ph, tq);
#pragma unroll
      for (int r = 0; r < 9; ++r) grad[(e * 9 + r) * NU + z] = tq[r];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < lines.count(); t += blockDim.x) {
    int l, d, s0, st, fm;
    if (!lines.get(t, &l, &d, &s0, &st, &fm)) continue;
    const long long el = e0 + l;
    const T* p = gs + l * 15 * PN + s0;
    T g0[3][5], g1[3][5];
#pragma unroll
    for (int c = 0; c < 15; ++c) {
      T v[N];
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = p[c * PN + m * st];
      hexl_faces<T, N>(op, v, &g0[c / 5][c % 5], &g1[c / 5][c % 5]);
    }
    auto out = [&](int f, const T (&g)[3][5]) {
      if constexpr (QV) {
        T u[5], nv[3], q[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) u[k] = fs[(l * 5 + k) * NF + f];
#pragma unroll
        for (int j = 0; j < 3; ++j) nv[j] = va.fnv[(el * 3 + j) * NF + f];
        visc_q_pre(bc, ph, u, g, nv, int(va.fbc[el * NF + f]), q,
                   prescribed_at(va, el, f, NF));
#pragma unroll
        for (int k = 1; k < 5; ++k) va.q[(el * 5 + k) * NF + f] = q[k];
      } else {
#pragma unroll
        for (int c = 0; c < 15; ++c) va.q[(el * 15 + c) * NF + f] = g[c / 5][c % 5];
      }
    };
    out(fm, g0);
    out(fm + N2, g1);
  }
}

// CTAs of the largest tile per SM.  FP32 values: 5 (48 registers); with FP64
// registers the odd N spill at 48 (100 bytes at N = 5), so 4 there: 24^3 and 48^3
// p = 4, 95 -> 86 and 669 -> 616 us with the largest tile, 586 -> 560 with the
// best; N = 4 keeps 5 (48^3: 286, 315 with 4).
template <typename T, typename TR, int N>
__host__ __device__ constexpr int hexl_vol_ctas() {
  return sizeof(T) == 8 ? 2 : sizeof(TR) == 8 && N % 2 ? 4 : 5;
}

// Volume kernel: f~ = S F at the solution points, then per line the jump
// F^C - n~ . f~ at its two faces and its N divergence terms (in place of the
// line's f~), R = -div / J, the RK epilogue and the next stage's u_f.  visc:
// the viscous flux of k_hexl_grad; AA: f~ comes projected in tflux.
template <typename T, typename TR, int N, int EPB, bool NS, bool AA = false>
__global__ void __launch_bounds__(hexl_threads<N>(EPB), hexl_vol_ctas<T, TR, N>())
    k_hexl_vol(long long ne, int eb, const T* __restrict__ uin, const T* __restrict__ visc,
               const T* __restrict__ fc, const T* __restrict__ smat,
               const T* __restrict__ rcpdjac, const __grid_constant__ HexOps<T> op, Phys<T> ph,
               HexStage<T, TR> sa, const T* __restrict__ tflux = nullptr) {
  using G = FxGeom<N>;
  constexpr int NU = G::NU, NF = G::NF, N2 = G::N2, PN = G::PN;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const long long e0 = (long long)blockIdx.x * eb;
  const int nel = int(ne - e0 < eb ? ne - e0 : eb);
  const LineTasks<N> lines(eb, nel);
  T* ft = reinterpret_cast<T*>(smem_raw);  // [eb][15][PN]
  T* cs = ft + eb * 15 * PN;               // [eb][5][NF]
  const int le = threadIdx.x / NU, z = threadIdx.x - le * NU;
  const bool pt = le < nel;
  const long long e = e0 + le;
  const int slot = G::slot(z % N, (z / N) % N, z / N2);
  async_copy(cs, fc + e0 * 5 * NF, nel * 5 * NF * int(sizeof(T)), threadIdx.x, blockDim.x);
  T uz[5] = {T(0), T(0), T(0), T(0), T(0)};
  TR xr[5], ar[5];
  T rj = T(0);
  if (pt) {
    T* p = ft + le * 15 * PN + slot;
#pragma unroll
    for (int k = 0; k < 5; ++k)
      uz[k] = uin ? uin[(e * 5 + k) * NU + z] : T(sa.X[(e * 5 + k) * NU + z]);
    if constexpr (AA) {
#pragma unroll
      for (int c = 0; c < 15; ++c) p[c * PN] = tflux[(e * 15 + c) * NU + z];
    } else {
      T tq[9], f[12], S[9];
      if (NS) {
#pragma unroll
        for (int r = 0; r < 9; ++r) tq[r] = visc[(e * 9 + r) * NU + z];
      }
#pragma unroll
      for (int r = 0; r < 9; ++r) S[r] = smat[(e * 9 + r) * NU + z];
      flux_point<T, NS>(uz, tq, ph, f);
      constexpr int kIdx[5][3] = {{0, 1, 2}, {3, 6, 7}, {6, 4, 8}, {7, 8, 5}, {9, 10, 11}};
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < 5; ++k)
          p[(d * 5 + k) * PN] = S[d * 3] * f[kIdx[k][0]] + S[d * 3 + 1] * f[kIdx[k][1]] +
                                S[d * 3 + 2] * f[kIdx[k][2]];
    }
  }
  cp_async_wait_all();
  __syncthreads();
  if (pt) {  // the epilogue's inputs, read ahead of the line phase
    hex_stage_load(sa, e * 5 * NU + z, NU, xr, ar);
    rj = rcpdjac[e * NU + z];
  }
  for (int t = threadIdx.x; t < lines.count(); t += blockDim.x) {
    int l, d, s0, st, fm;
    if (!lines.get(t, &l, &d, &s0, &st, &fm)) continue;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      T* p = ft + (l * 15 + d * 5 + k) * PN + s0;
      T v[N], f0, f1;
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = p[m * st];
      hexl_faces<T, N>(op, v, &f0, &f1);
      const T j0 = cs[(l * 5 + k) * NF + fm] + f0, j1 = cs[(l * 5 + k) * NF + fm + N2] - f1;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        T g = op.gl[i] * j0 + op.gr[i] * j1;
#pragma unroll
        for (int m = 0; m < N; ++m) g += op.d1[i][m] * v[m];
        p[i * st] = g;
      }
    }
  }
  __syncthreads();
  if (pt) {
    T R[5], s[5];
    T* p = ft + le * 15 * PN + slot;
#pragma unroll
    for (int k = 0; k < 5; ++k)
      R[k] = -((p[k * PN] + p[(5 + k) * PN]) + p[(10 + k) * PN]) * rj;
    hex_stage_apply(sa, e * 5 * NU + z, NU, uz, R, xr, ar, s);
#pragma unroll
    for (int k = 0; k < 5; ++k) p[k * PN] = s[k];
  }
  if (sa.uf_next == nullptr) return;
  __syncthreads();
  for (int t = threadIdx.x; t < lines.count(); t += blockDim.x) {
    int l, d, s0, st, fm;
    if (!lines.get(t, &l, &d, &s0, &st, &fm)) continue;
    T* o = sa.uf_next + (e0 + l) * 5 * NF + fm;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const T* p = ft + (l * 15 + k) * PN + s0;
      T v[N], f0, f1;
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = p[m * st];
      hexl_faces<T, N>(op, v, &f0, &f1);
      o[k * NF] = f0;
      o[k * NF + N2] = f1;
    }
  }
}

}  // namespace frgb
