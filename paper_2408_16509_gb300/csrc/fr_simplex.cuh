// Register-blocked FP32 kernels for tetrahedra and prisms.
//
// A thread of the dense kernels (fr_kernels.cuh) forms one output point: five
// to seven shared-memory reads for every 15 multiply-adds bound them.  Here a
// thread forms ZB points of one element, so a row of values is read once for
// all of them and the operator entries come as vectors.
//
// A CTA takes groups of eb elements, a thread per solution point.  The phases
// (points, flux points, products) map the CTA's threads anew, each over its
// own number of tasks; shared memory holds the element's values between them:
// rows of 5 as a plane of four and a plane of one, rows of 15 as planes of
// four values, so that consecutive points lie on consecutive banks and equal
// points are broadcast.  The next group's inputs are prefetched to L2 while
// this one is worked on.
//
// Tetrahedra: dense D and LIFT, the correction per face (its reference normal
// is one vector).  Prisms (structure: fr_prism.cuh): level tasks form ZB
// triangle points of a level from the level's points and its quadrilateral
// flux points (D_xi, D_eta); line tasks form the points of a line from them
// and the line's two triangle flux points (D_zeta).  A gradient's d = 0, 1
// come from the level, d = 2 from the line; a divergence is their sum.
//
// As on hexahedra the gradient kernel stores the viscous flux at the solution
// points (9 values) in place of the gradient (15).
//
// Bound by the shared-memory pipe (66-82 % of its rate at p = 3) and the
// barriers between the phases; DRAM traffic would take a third to a half of the
// time (27-35 %).  Measured, us: common solution + gradient, volume
// with one thread per point -> here, the gradient with its jumps:
//   384000 tetrahedra p = 1    59 + 195, 181 -> 127,  86
//   196608 tetrahedra p = 2    50 + 200, 256 -> 148, 124
//   131712 tetrahedra p = 3    53 + 307, 354 -> 200, 174
//    48000 tetrahedra p = 4    32 + 256, 303 -> 160, 155
//   128000 prisms p = 1        33 + 107,  99 ->  84,  67
//    65536 prisms p = 2        32 + 131, 156 -> 101,  92
//    43904 prisms p = 3        32 + 202, 246 -> 120, 130
// (tensor cores, p = 3: tetrahedra 53 + 977, 449; prisms 32 + 410, 356).
// Prisms of order 4 keep the dense kernels: their interpolation to the
// triangle faces has more nonzeros than kPriMaxM0.
#pragma once
#include "fr_kernels.cuh"
#include "fr_hex.cuh"
#include "fr_prism.cuh"

namespace frgb {

// threads of a CTA at most: one per point of its elements (eb NU of them) in
// the point phases.  128 where points fill nine tenths of them (256 took 0-2 %
// longer at p = 3), else 256.
template <int NU>
__host__ __device__ constexpr int simplex_threads() {
  return 128 / NU * NU * 10 >= 128 * 9 ? 128 : 256;
}
constexpr int kSimplexMaxFaces = 5;

// Operators: a device image in shared-memory order and what is the same for
// every thread.  Output points come in NG groups of ZB, a group padded to GP
// entries (zeros past the points) so that vector reads are aligned.
// Tetrahedra: DT [NU][3][NG][GP], LT [NF][NG][GP].  Prisms: A [NT][2][NG][GP],
// LQ [NL][3 NL][NG][GP], LZ [2][NL][NT].  Then M0 by its nonzeros: values
// [NF][nm], and as ints columns [NF][nm] and (prisms) the quadrilateral flux
// points of a level QF [NL][3 NL] and the triangle flux points of a line
// TF [2][NT].
struct SimplexOps {
  const float* img;
  int nm;
  float nface[kSimplexMaxFaces][3];  // reference normal of each face
  float B[25];                       // prisms: D_zeta [NL][NL]
};

// rows of 5 of NP points: plane of four, plane of one
template <int NP>
__device__ __forceinline__ void ld5(const float* b, int i, float v[5]) {
  const float4 a = reinterpret_cast<const float4*>(b)[i];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b[4 * NP + i];
}
template <int NP>
__device__ __forceinline__ void st5(float* b, int i, const float v[5]) {
  reinterpret_cast<float4*>(b)[i] = make_float4(v[0], v[1], v[2], v[3]);
  b[4 * NP + i] = v[4];
}
// rows of 15: planes of four
template <int NP>
__device__ __forceinline__ void ld15(const float* b, int i, float v[15]) {
  const float4* p = reinterpret_cast<const float4*>(b);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4 a = p[c * NP + i];
    v[4 * c] = a.x; v[4 * c + 1] = a.y; v[4 * c + 2] = a.z; v[4 * c + 3] = a.w;
  }
  const float4 a = p[3 * NP + i];
  v[12] = a.x; v[13] = a.y; v[14] = a.z;
}
template <int NP>
__device__ __forceinline__ void st15(float* b, int i, const float v[15]) {
  float4* p = reinterpret_cast<float4*>(b);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    p[c * NP + i] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
  p[3 * NP + i] = make_float4(v[12], v[13], v[14], 0.f);
}
// a row's first ten (d = 0, 1) and last five values (d = 2)
template <int NP>
__device__ __forceinline__ void ld10(const float* b, int i, float v[10]) {
  const float4* p = reinterpret_cast<const float4*>(b);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float4 a = p[c * NP + i];
    v[4 * c] = a.x; v[4 * c + 1] = a.y; v[4 * c + 2] = a.z; v[4 * c + 3] = a.w;
  }
  const float2 a = *reinterpret_cast<const float2*>(p + 2 * NP + i);
  v[8] = a.x; v[9] = a.y;
}
template <int NP>
__device__ __forceinline__ void st10(float* b, int i, const float v[10]) {
  float4* p = reinterpret_cast<float4*>(b);
#pragma unroll
  for (int c = 0; c < 2; ++c)
    p[c * NP + i] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
  *reinterpret_cast<float2*>(p + 2 * NP + i) = make_float2(v[8], v[9]);
}
template <int NP>
__device__ __forceinline__ void ldz(const float* b, int i, float v[5]) {
  const float4* p = reinterpret_cast<const float4*>(b);
  const float2 a = reinterpret_cast<const float2*>(p + 2 * NP + i)[1];
  const float4 c = p[3 * NP + i];
  v[0] = a.x; v[1] = a.y; v[2] = c.x; v[3] = c.y; v[4] = c.z;
}
template <int NP>
__device__ __forceinline__ void stz(float* b, int i, const float v[5]) {
  float4* p = reinterpret_cast<float4*>(b);
  reinterpret_cast<float2*>(p + 2 * NP + i)[1] = make_float2(v[0], v[1]);
  p[3 * NP + i] = make_float4(v[2], v[3], v[4], 0.f);
}

// ZB consecutive operator entries (16-byte aligned; 8-byte for ZB = 2)
template <int ZB>
__device__ __forceinline__ void ld_ops(const float* p, float v[ZB]) {
#pragma unroll
  for (int i = 0; i + 4 <= ZB; i += 4) {
    const float4 a = *reinterpret_cast<const float4*>(p + i);
    v[i] = a.x; v[i + 1] = a.y; v[i + 2] = a.z; v[i + 3] = a.w;
  }
  constexpr int R = ZB / 4 * 4;
  if constexpr (ZB - R >= 2) {
    const float2 a = *reinterpret_cast<const float2*>(p + R);
    v[R] = a.x; v[R + 1] = a.y;
  }
  if constexpr ((ZB - R) % 2 == 1) v[ZB - 1] = p[ZB - 1];
}

// acc[k][i] += w[i] v[k]
template <int ZB>
__device__ __forceinline__ void rank1(float acc[5][ZB], const float w[ZB], const float* v) {
#pragma unroll
  for (int k = 0; k < 5; ++k)
#pragma unroll
    for (int i = 0; i < ZB; ++i) acc[k][i] += w[i] * v[k];
}

template <int NU, int NF>
struct SimplexGeom {
  static constexpr int P = pri_order(NU, NF);  // 0: tetrahedra
  static constexpr int NT = P ? (P + 1) * (P + 2) / 2 : NF / 4, NL = P + 1, NQ = 3 * NL;
  // strides of an element's arrays: multiples of 4 values, 4 modulo 32 or 8
  // so that neighbouring elements start on other banks
  static constexpr int pad(int n) { return (n + 3) / 4 * 4 + ((n + 3) / 4 * 4 % 32 == 0 ? 4 : 0); }
  static constexpr int U5 = pad(5 * NU), F5 = pad(5 * NF), U15 = pad(16 * NU);
  // output points that a product's thread blocks are taken from
  static constexpr int NO = P ? NT : NU;
  __host__ __device__ static constexpr int ng(int zb) { return (NO + zb - 1) / zb; }
  __host__ __device__ static constexpr int gp(int zb) { return zb == 2 ? 2 : (zb + 3) / 4 * 4; }
  // floats of the operators without M0, of M0's values, and ints
  __host__ __device__ static constexpr int ops(int zb) {
    const int w = ng(zb) * gp(zb);
    return ((P ? (2 * NT + NL * NQ) * w + 2 * NL * NT : (3 * NU + NF) * w) + 3) / 4 * 4;
  }
  __host__ __device__ static constexpr int m0(int nm) { return (NF * nm + 3) / 4 * 4; }
  __host__ __device__ static constexpr int ints(int nm) {
    return ((P ? NL * NQ + 2 * NT : 0) + NF * nm + 3) / 4 * 4;
  }
  __host__ __device__ static constexpr int words(int zb, int nm) {
    return ops(zb) + m0(nm) + ints(nm);
  }
  // per element: u, du, gradient; divergence (prisms: its two parts; the
  // first one then takes u of the next stage), jump, f~
  static constexpr int kGrad = U5 + F5 + U15;
  static constexpr int kVol = (P ? 2 : 1) * U5 + F5 + U15;
};

// Points a thread forms; 0: no such kernels for the type.  Two hide latency
// best: four or five need 128 registers a thread in the gradient kernel and
// halve the resident threads (36864 tetrahedra p = 3: 64 us with two, 92 with
// four; volume 57 and 65; 20480 prisms p = 3: 59 with two, 84 with five).
// Three divide the triangle points of prisms p = 1, 2.
template <int NU, int NF>
constexpr int simplex_zb() {
  if (NU == 8 || NU == 27 || NU == 64 || NU == 125) return 0;  // hexahedra
  return NU == 18 || NU == 6 ? 3 : 2;
}

template <int NU, int NF, int ZB>
struct SimplexSm {
  using G = SimplexGeom<NU, NF>;
  static constexpr int NG = G::ng(ZB), GP = G::gp(ZB);
  const float *op, *mv;
  const int *mc, *qf, *tf;
  float* elem;
  int nm;
  __device__ __forceinline__ SimplexSm(const SimplexOps& g, float* s) : nm(g.nm) {
    const int n = G::words(ZB, g.nm);
    for (int i = threadIdx.x; i < n / 4; i += blockDim.x)
      reinterpret_cast<float4*>(s)[i] = reinterpret_cast<const float4*>(g.img)[i];
    op = s;
    mv = s + G::ops(ZB);
    mc = reinterpret_cast<const int*>(mv + G::m0(g.nm));
    qf = mc + NF * g.nm;
    tf = qf + G::NL * G::NQ;
    elem = s + n;
  }
  // the interpolation of n values (a row of NUM) to flux point f; a row's
  // values past its nonzeros are zero
  template <class Ld, class Add>
  __device__ __forceinline__ void interp(int f, Ld&& ld, Add&& add) const {
    for (int j = 0; j < nm; ++j) {
      const float m = mv[f * nm + j];
      if (m == 0.f) break;
      ld(mc[f * nm + j]);
      add(m);
    }
  }
};

// the 16-byte blocks of n values at p into the L2 cache
template <typename T>
__device__ __forceinline__ void l2_prefetch(const T* p, long long n) {
  const unsigned long long a = reinterpret_cast<unsigned long long>(p) & ~15ull;
  const unsigned bytes =
      unsigned(reinterpret_cast<unsigned long long>(p + n) - a) & ~15u;
  if (bytes) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(bytes));
}

// NS gradients: corrected reference gradient D u + LIFT (n~ du), physical
// gradient, viscous flux at the solution points, q at the flux points.
template <int NU, int NF, int ZB>
__global__ void __launch_bounds__(simplex_threads<NU>(), 1024 / simplex_threads<NU>())
    k_simplex_grad(long long ne, int eb, const float* __restrict__ u,
                   const __grid_constant__ TraceArgs<float> ta, const float* __restrict__ smat,
                   const float* __restrict__ rcpdjac, const __grid_constant__ SimplexOps ops,
                   float* __restrict__ visc, ViscArgs<float> va,
                   const __grid_constant__ BCTab<float> bc, Phys<float> ph) {
  using G = SimplexGeom<NU, NF>;
  using M = SimplexSm<NU, NF, ZB>;
  constexpr int NT = G::NT;
  extern __shared__ __align__(16) float simplex_sm[];
  const M sm(ops, simplex_sm);
  const int le = threadIdx.x / NU, z = threadIdx.x - le * NU;
  float* us = sm.elem;  // [eb] rows of u, du, gradient
  float* ds = us + eb * G::U5;
  float* gs = ds + eb * G::F5;
  const long long ngroups = (ne + eb - 1) / eb;
  for (long long grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    const long long e0 = grp * eb;
    const int nel = int(ne - e0 < eb ? ne - e0 : eb);
    // the CTA's next group on its way from DRAM to L2
    if (threadIdx.x == 0 && grp + gridDim.x < ngroups) {
      const long long en = (grp + gridDim.x) * eb, n = ne - en < eb ? ne - en : eb;
      l2_prefetch(u + en * 5 * NU, n * 5 * NU);
      l2_prefetch(smat + en * 9 * NU, n * 9 * NU);
      l2_prefetch(rcpdjac + en * NU, n * NU);
      l2_prefetch(ta.partner + en * NF, n * NF);
      l2_prefetch(ta.uf + en * 5 * NF, n * 5 * NF);
      l2_prefetch(va.fnv + en * 3 * NF, n * 3 * NF);
    }
    const bool pt = le < nel;
    const long long e = e0 + le;
    if (pt) {
      float uz[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = u[(e * 5 + k) * NU + z];
      st5<NU>(us + le * G::U5, z, uz);
    }
#pragma unroll 1
    for (int t = threadIdx.x; t < nel * NF; t += blockDim.x) {
      const int l = t / NF, f = t - l * NF;
      float own[5], d[5];
      trace_jump(ta, e0 + l, f, NF, own, d);
      st5<NF>(ds + l * G::F5, f, d);
    }
    __syncthreads();
    if constexpr (G::P == 0) {
      constexpr int NG = M::NG, GP = M::GP;
      const float *DT = sm.op, *LT = sm.op + 3 * NU * NG * GP;
      for (int t = threadIdx.x; t < nel * NG; t += blockDim.x) {
        const int l = t / NG, g = t - l * NG, z0 = g * ZB;
        float acc[3][5][ZB] = {};
        const float* ue = us + l * G::U5;
#pragma unroll 2
        for (int q = 0; q < NU; ++q) {
          float v[5], w[ZB];
          ld5<NU>(ue, q, v);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            ld_ops<ZB>(DT + ((q * 3 + d) * NG + g) * GP, w);
            rank1<ZB>(acc[d], w, v);
          }
        }
        const float* de = ds + l * G::F5;
#pragma unroll 1
        for (int fa = 0; fa < 4; ++fa) {
          float s[5][ZB] = {};
#pragma unroll 2
          for (int f = fa * NT; f < (fa + 1) * NT; ++f) {
            float v[5], w[ZB];
            ld5<NF>(de, f, v);
            ld_ops<ZB>(LT + (f * NG + g) * GP, w);
            rank1<ZB>(s, w, v);
          }
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const float n = ops.nface[fa][d];  // the same on every thread
            if (n != 0.f) {
#pragma unroll
              for (int k = 0; k < 5; ++k)
#pragma unroll
                for (int i = 0; i < ZB; ++i) acc[d][k][i] += n * s[k][i];
            }
          }
        }
#pragma unroll
        for (int i = 0; i < ZB; ++i) {
          if (NU % ZB == 0 || z0 + i < NU) {
            float r[15];
#pragma unroll
            for (int c = 0; c < 15; ++c) r[c] = acc[c / 5][c % 5][i];
            st15<NU>(gs + l * G::U15, z0 + i, r);
          }
        }
      }
    } else {
      constexpr int NL = G::NL, NQ = G::NQ, NG = M::NG, GP = M::GP;
      const float *A = sm.op, *LQ = A + 2 * NT * NG * GP, *LZ = LQ + NL * NQ * NG * GP;
      const int nlev = nel * NL * NG;
      for (int t = threadIdx.x; t < nlev + nel * NT; t += blockDim.x) {
        if (t < nlev) {
          const int l = t / (NL * NG), r0 = t - l * NL * NG, lz = r0 / NG, g = r0 - lz * NG;
          float acc[2][5][ZB] = {};
          const float* ue = us + l * G::U5;
#pragma unroll 2
          for (int t2 = 0; t2 < NT; ++t2) {
            float v[5], w[ZB];
            ld5<NU>(ue, lz * NT + t2, v);
#pragma unroll
            for (int d = 0; d < 2; ++d) {
              ld_ops<ZB>(A + ((t2 * 2 + d) * NG + g) * GP, w);
              rank1<ZB>(acc[d], w, v);
            }
          }
          const float* de = ds + l * G::F5;
#pragma unroll 1
          for (int fa = 0; fa < 3; ++fa) {
            float s[5][ZB] = {};
#pragma unroll 2
            for (int j = fa * NL; j < (fa + 1) * NL; ++j) {
              float v[5], w[ZB];
              ld5<NF>(de, sm.qf[lz * NQ + j], v);
              ld_ops<ZB>(LQ + ((lz * NQ + j) * NG + g) * GP, w);
              rank1<ZB>(s, w, v);
            }
#pragma unroll
            for (int d = 0; d < 2; ++d) {
              const float n = ops.nface[2 + fa][d];
              if (n != 0.f) {
#pragma unroll
                for (int k = 0; k < 5; ++k)
#pragma unroll
                  for (int i = 0; i < ZB; ++i) acc[d][k][i] += n * s[k][i];
              }
            }
          }
#pragma unroll
          for (int i = 0; i < ZB; ++i) {
            if (NT % ZB == 0 || g * ZB + i < NT) {
              float r[10];
#pragma unroll
              for (int c = 0; c < 10; ++c) r[c] = acc[c / 5][c % 5][i];
              st10<NU>(gs + l * G::U15, lz * NT + g * ZB + i, r);
            }
          }
        } else {
          const int l = (t - nlev) / NT, tp = t - nlev - l * NT;
          float v[NL][5], b0[5], b1[5];
#pragma unroll
          for (int z = 0; z < NL; ++z) ld5<NU>(us + l * G::U5, z * NT + tp, v[z]);
          ld5<NF>(ds + l * G::F5, sm.tf[tp], b0);
          ld5<NF>(ds + l * G::F5, sm.tf[NT + tp], b1);
#pragma unroll
          for (int k = 0; k < 5; ++k) {
            b0[k] *= ops.nface[0][2];
            b1[k] *= ops.nface[1][2];
          }
#pragma unroll
          for (int z = 0; z < NL; ++z) {
            const float w0 = LZ[z * NT + tp], w1 = LZ[(NL + z) * NT + tp];
            float r[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
              r[k] = w0 * b0[k] + w1 * b1[k];
#pragma unroll
              for (int m = 0; m < NL; ++m) r[k] += ops.B[z * NL + m] * v[m][k];
            }
            stz<NU>(gs + l * G::U15, z * NT + tp, r);
          }
        }
      }
    }
    __syncthreads();
    if (pt) {
      float r[15], g[3][5], uz[5], tq[9], S[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) S[i] = smat[(e * 9 + i) * NU + z];
      const float rj = rcpdjac[e * NU + z];
      ld15<NU>(gs + le * G::U15, z, r);
      ld5<NU>(us + le * G::U5, z, uz);
#pragma unroll
      for (int i = 0; i < 9; ++i) S[i] *= rj;
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 5; ++k)
          g[j][k] = S[j] * r[k] + S[3 + j] * r[5 + k] + S[6 + j] * r[10 + k];
#pragma unroll
      for (int c = 0; c < 15; ++c) r[c] = g[c / 5][c % 5];
      st15<NU>(gs + le * G::U15, z, r);
      viscous_point(uz, g, ph, tq);
#pragma unroll
      for (int i = 0; i < 9; ++i) visc[(e * 9 + i) * NU + z] = tq[i];
    }
    __syncthreads();
#pragma unroll 1
    for (int t = threadIdx.x; t < nel * NF; t += blockDim.x) {
      const int l = t / NF, f = t - l * NF;
      float a[15] = {}, r[15];
      sm.interp(
          f, [&](int p) { ld15<NU>(gs + l * G::U15, p, r); },
          [&](float m) {
#pragma unroll
            for (int c = 0; c < 15; ++c) a[c] += m * r[c];
          });
      write_visc_q(va, bc, ph, e0 + l, f, NF, a);
    }
    // the next group's points overwrite u and du, last read before the
    // barrier above; its products write the gradient only after their own
  }
}

// Volume kernel: f~ = S F, the jump F^C - n~ . M0 f~, divergence and LIFT,
// R = -div / J, the RK epilogue, the next stage's u_f = M0 u_next.  visc: the
// viscous flux of k_simplex_grad.
template <int NU, int NF, int ZB, bool NS>
__global__ void __launch_bounds__(simplex_threads<NU>(), 768 / simplex_threads<NU>())
    k_simplex_vol(long long ne, int eb, const float* __restrict__ u,
                  const float* __restrict__ visc, const float* __restrict__ fc,
                  const float* __restrict__ smat, const float* __restrict__ rcpdjac,
                  const __grid_constant__ SimplexOps ops, Phys<float> ph,
                  HexStage<float, float> sa) {
  using G = SimplexGeom<NU, NF>;
  using M = SimplexSm<NU, NF, ZB>;
  constexpr int NT = G::NT, NTR = (NF + NU - 1) / NU;
  extern __shared__ __align__(16) float simplex_sm[];
  const M sm(ops, simplex_sm);
  const int le = threadIdx.x / NU, z = threadIdx.x - le * NU;
  float* rs = sm.elem;                            // [eb] divergence, then u_next
  float* zs = rs + eb * G::U5;                    // [eb] prisms: D_zeta's part
  float* js = zs + (G::P ? eb * G::U5 : 0);       // [eb] jump
  float* ft = js + eb * G::F5;                    // [eb] f~
  const long long ngroups = (ne + eb - 1) / eb;
  for (long long grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    const long long e0 = grp * eb;
    const int nel = int(ne - e0 < eb ? ne - e0 : eb);
    if (threadIdx.x == 0 && grp + gridDim.x < ngroups) {
      const long long en = (grp + gridDim.x) * eb, n = ne - en < eb ? ne - en : eb;
      l2_prefetch(u + en * 5 * NU, n * 5 * NU);
      if (NS) l2_prefetch(visc + en * 9 * NU, n * 9 * NU);
      l2_prefetch(smat + en * 9 * NU, n * 9 * NU);
      l2_prefetch(fc + en * 5 * NF, n * 5 * NF);
      l2_prefetch(rcpdjac + en * NU, n * NU);
      bool nx, na;
      hex_stage_needs(sa, &nx, &na);
      if (nx) l2_prefetch(sa.X + en * 5 * NU, n * 5 * NU);
      if (na) l2_prefetch(sa.A + en * 5 * NU, n * 5 * NU);
    }
    const bool pt = le < nel;
    const long long e = e0 + le;
    float uz[5], xr[5], ar[5], c[NTR][5], rj = 0.f;
#pragma unroll
    for (int i = 0; i < NTR; ++i) {
      const int t = threadIdx.x + i * blockDim.x;
      if (t < nel * NF) {
#pragma unroll
        for (int k = 0; k < 5; ++k) c[i][k] = fc[((e0 + t / NF) * 5 + k) * NF + t % NF];
      }
    }
    if (pt) {
      float tq[9], S[9], f[12], r[15];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = u[(e * 5 + k) * NU + z];
      if (NS) {
#pragma unroll
        for (int i = 0; i < 9; ++i) tq[i] = visc[(e * 9 + i) * NU + z];
      }
#pragma unroll
      for (int i = 0; i < 9; ++i) S[i] = smat[(e * 9 + i) * NU + z];
      flux_point<float, NS>(uz, tq, ph, f);
      constexpr int kIdx[5][3] = {{0, 1, 2}, {3, 6, 7}, {6, 4, 8}, {7, 8, 5}, {9, 10, 11}};
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < 5; ++k)
          r[d * 5 + k] = S[d * 3] * f[kIdx[k][0]] + S[d * 3 + 1] * f[kIdx[k][1]] +
                         S[d * 3 + 2] * f[kIdx[k][2]];
      st15<NU>(ft + le * G::U15, z, r);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NTR; ++i) {
      const int t = threadIdx.x + i * blockDim.x;
      if (t < nel * NF) {
        const int l = t / NF, f = t - l * NF;
        int fa;
        if constexpr (G::P == 0) fa = f / NT;
        else fa = f < 2 * NT ? f / NT : 2 + (f - 2 * NT) / (G::NL * G::NL);
        const float n0 = ops.nface[fa][0], n1 = ops.nface[fa][1], n2 = ops.nface[fa][2];
        float r[15];
        sm.interp(
            f, [&](int q) { ld15<NU>(ft + l * G::U15, q, r); },
            [&](float m) {
              const float w0 = m * n0, w1 = m * n1, w2 = m * n2;
#pragma unroll
              for (int k = 0; k < 5; ++k)
                c[i][k] -= w0 * r[k] + w1 * r[5 + k] + w2 * r[10 + k];
            });
        st5<NF>(js + l * G::F5, f, c[i]);
      }
    }
    if (pt) {  // the epilogue's inputs, read ahead of the products
      hex_stage_load(sa, e * 5 * NU + z, NU, xr, ar);
      rj = rcpdjac[e * NU + z];
    }
    __syncthreads();
    if constexpr (G::P == 0) {
      constexpr int NG = M::NG, GP = M::GP;
      const float *DT = sm.op, *LT = sm.op + 3 * NU * NG * GP;
      for (int t = threadIdx.x; t < nel * NG; t += blockDim.x) {
        const int l = t / NG, g = t - l * NG, z0 = g * ZB;
        float acc[5][ZB] = {};
        const float* fe = ft + l * G::U15;
#pragma unroll 2
        for (int q = 0; q < NU; ++q) {
          float r[15], w[ZB];
          ld15<NU>(fe, q, r);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            ld_ops<ZB>(DT + ((q * 3 + d) * NG + g) * GP, w);
            rank1<ZB>(acc, w, r + 5 * d);
          }
        }
        const float* je = js + l * G::F5;
#pragma unroll 4
        for (int f = 0; f < NF; ++f) {
          float v[5], w[ZB];
          ld5<NF>(je, f, v);
          ld_ops<ZB>(LT + (f * NG + g) * GP, w);
          rank1<ZB>(acc, w, v);
        }
#pragma unroll
        for (int i = 0; i < ZB; ++i) {
          if (NU % ZB == 0 || z0 + i < NU) {
            float r[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) r[k] = acc[k][i];
            st5<NU>(rs + l * G::U5, z0 + i, r);
          }
        }
      }
    } else {
      constexpr int NL = G::NL, NQ = G::NQ, NG = M::NG, GP = M::GP;
      const float *A = sm.op, *LQ = A + 2 * NT * NG * GP, *LZ = LQ + NL * NQ * NG * GP;
      const int nlev = nel * NL * NG;
      for (int t = threadIdx.x; t < nlev + nel * NT; t += blockDim.x) {
        if (t < nlev) {
          const int l = t / (NL * NG), r0 = t - l * NL * NG, lz = r0 / NG, g = r0 - lz * NG;
          float acc[5][ZB] = {};
#pragma unroll 2
          for (int t2 = 0; t2 < NT; ++t2) {
            float v[10], w[ZB];
            ld10<NU>(ft + l * G::U15, lz * NT + t2, v);
#pragma unroll
            for (int d = 0; d < 2; ++d) {
              ld_ops<ZB>(A + ((t2 * 2 + d) * NG + g) * GP, w);
              rank1<ZB>(acc, w, v + 5 * d);
            }
          }
#pragma unroll 2
          for (int j = 0; j < NQ; ++j) {
            float v[5], w[ZB];
            ld5<NF>(js + l * G::F5, sm.qf[lz * NQ + j], v);
            ld_ops<ZB>(LQ + ((lz * NQ + j) * NG + g) * GP, w);
            rank1<ZB>(acc, w, v);
          }
#pragma unroll
          for (int i = 0; i < ZB; ++i) {
            if (NT % ZB == 0 || g * ZB + i < NT) {
              float r[5];
#pragma unroll
              for (int k = 0; k < 5; ++k) r[k] = acc[k][i];
              st5<NU>(rs + l * G::U5, lz * NT + g * ZB + i, r);
            }
          }
        } else {
          const int l = (t - nlev) / NT, tp = t - nlev - l * NT;
          float v[NL][5], b0[5], b1[5];
#pragma unroll
          for (int z = 0; z < NL; ++z) ldz<NU>(ft + l * G::U15, z * NT + tp, v[z]);
          ld5<NF>(js + l * G::F5, sm.tf[tp], b0);
          ld5<NF>(js + l * G::F5, sm.tf[NT + tp], b1);
#pragma unroll
          for (int z = 0; z < NL; ++z) {
            const float w0 = LZ[z * NT + tp], w1 = LZ[(NL + z) * NT + tp];
            float r[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
              r[k] = w0 * b0[k] + w1 * b1[k];
#pragma unroll
              for (int m = 0; m < NL; ++m) r[k] += ops.B[z * NL + m] * v[m][k];
            }
            st5<NU>(zs + l * G::U5, z * NT + tp, r);
          }
        }
      }
    }
    __syncthreads();
    if (pt) {
      float R[5], s[5];
      ld5<NU>(rs + le * G::U5, z, R);
      if constexpr (G::P > 0) {
        ld5<NU>(zs + le * G::U5, z, s);
#pragma unroll
        for (int k = 0; k < 5; ++k) R[k] += s[k];
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) R[k] = -R[k] * rj;
      hex_stage_apply(sa, e * 5 * NU + z, NU, uz, R, xr, ar, s);
      st5<NU>(rs + le * G::U5, z, s);
    }
    if (sa.uf_next != nullptr) {
      __syncthreads();
      for (int t = threadIdx.x; t < nel * NF; t += blockDim.x) {
        const int l = t / NF, f = t - l * NF;
        float a[5] = {}, v[5];
        sm.interp(
            f, [&](int q) { ld5<NU>(rs + l * G::U5, q, v); },
            [&](float m) {
#pragma unroll
              for (int k = 0; k < 5; ++k) a[k] += m * v[k];
            });
#pragma unroll
        for (int k = 0; k < 5; ++k) sa.uf_next[((e0 + l) * 5 + k) * NF + f] = a[k];
      }
    }
    // the next group writes f~ (last read before the products' barrier) and
    // the jumps and divergence only after barriers of its own
  }
}

}  // namespace frgb
