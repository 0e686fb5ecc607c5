// FP64 hexahedron kernels whose line operators run on the integer pipe.
//
// GB300 issues FP64 instructions at 2 lanes per clock and SM, and 32 x 32 +
// 64-bit integer multiply-adds (IMAD.WIDE) at 64 (measured: 54.6 against 1.6
// per clock in chains of each).  FP64 gradient and volume kernels are bound by
// that FP64 pipe, most of it in products with the line operators.  Here those
// products are fixed-point sums:
//
//   - the N points of a line, and the values at its two faces, are converted
//     to fixed point relative to the largest magnitude among them,
//     q = v 2^(59 - E), |v| < 2^E, held as two signed limbs q = hi 2^30 + lo;
//   - operator entries are limbs too, scaled by a power of two that bounds the
//     row's sum of magnitudes, so no sum can overflow;
//   - a term is three multiply-adds, hi hi' into one 64-bit sum and
//     hi lo' + lo hi' into another (lo lo' is below the result's unit);
//   - the derivative and interpolation rows of the symmetric line points
//     are applied to sums and differences of mirrored points (exact in
//     integers), which halves the terms;
//   - a result has a unit of about 2^-60 of its bound |A|_inf max|v| and is
//     normalised and rounded once to FP64.
//
// The unit belongs to the line and the variable: an FP64 sum over the same
// line rounds its partial sums to 2^-53 of those magnitudes, whatever the
// other lines, directions and variables of the element hold.  (One exponent
// per element and field, and metric products in fixed point, lost as many bits as
// an element is stretched or a field varies within it.)  Metric products, the
// flux, the scaling by 1/J and the RK update stay in FP64; the divergence's
// three directions are added in units of the largest.  A line that holds an Inf
// or NaN gives NaN, which the epilogue flags.
//
// Threads: TPE = 32 ceil(N^3 / 32) per element, one per solution point in the
// pointwise phases and one per (field, line) in the line phases.  A line thread
// reads its N points once for all N results (and both face values), with
// coefficients that are the same for every thread (constant operands);
// one thread per point would read every line N times, with lane-varying
// coefficients.
//
// Measured per launch, 24^3 p = 4 (20^3 p = 3) Navier-Stokes: gradient with the
// solution jumps 850 + 43 -> 427 us (242 + 20 -> 140), volume 1108 -> 291 us
// (321 -> 94), against FP64 loops with one thread per point; one exponent per
// element and field and metric products in fixed point took 345 and 269 us
// (118, 96).  Both are bound by the FP64 pipe (82 and 83 % of its rate; integer
// pipes at 34-38 %): the metric products and the pointwise physics.  62 to 70
// registers; a fourth CTA per SM gained nothing.
#pragma once
#include "fr_hex.cuh"

namespace frgb {

struct alignas(8) FxCoef {
  int hi, lo;
};

// Line operators in limbs, for N points per line with H = (N + 1) / 2 and
// P = N / 2 mirrored pairs: rows i and N - 1 - i of the derivative are B_i + A_i
// and B_i - A_i with A_i = sum_m a[i][m] (v_m + v_{N-1-m}) (m = P: the middle
// point) and B_i = sum_m b[i][m] (v_m - v_{N-1-m}); ca (in A) and cb (in B)
// are the correction weights of the sum and the difference of the minus and
// plus faces' jumps; the face values are sum_m ie[m] (..+..) +- sum_m io[m]
// (..-..).
struct HexFxLine {
  FxCoef a[2][3], b[3][2], ca[2], cb[3];
};

struct HexFxOps {
  HexFxLine g, v;        // gradient; volume (the jump's scale folded in)
  FxCoef ie[3], io[2];
  int sg, sv, sm;        // row scales (powers of two) of g, v and ie / io
  int gather;            // 1: Gauss-Lobatto lines, the face points are the line
                         //    end points
};

// orders that have the fixed-point kernels (p = 1 keeps the FP64 lines: its
// 8 points would leave 24 of a warp's lanes idle)
template <typename T, int N>
__host__ __device__ constexpr bool use_hexfx() {
  return sizeof(T) == 8 && N >= 3;
}

template <int N>
struct FxGeom {
  static constexpr int NU = N * N * N, N2 = N * N, NF = 6 * N * N;
  static constexpr int P = N / 2, H = (N + 1) / 2;
  // strides of a field in shared memory (8-byte slots): an odd row length
  // keeps the lines of all three directions on distinct banks
  static constexpr int SY = N % 2 == 0 ? N + 1 : N, SZ = SY * N, PN = SZ * N;
  static constexpr int WPE = (NU + 31) / 32, TPE = 32 * WPE;
  __device__ static constexpr int slot(int a, int b, int c) { return a + SY * b + SZ * c; }
};

__host__ __device__ inline FxCoef fx_split(long long q) {
  FxCoef r;
  r.lo = int(uint32_t(q) << 2) >> 2;
  r.hi = int((q + (1LL << 29)) >> 30);
  return r;
}

__device__ __forceinline__ long long fx_join(FxCoef a) {
  return (long long)a.hi * (1 << 30) + a.lo;
}

// magnitude bits of v's high word: the largest of a line sets its exponent
__device__ __forceinline__ unsigned fx_mag(double v) {
  return unsigned(__double2hiint(v)) & 0x7fffffffu;
}

// Line exponents below this are taken as this (values under 2^-890 resolve
// to 2^-949): the shifts below then need no special case for zero.
constexpr int kFxMinExp = 132;

// exponent em = E + 1022 of a line whose largest magnitude has the bits mag:
// the biased exponent field, or more
__device__ __forceinline__ int fx_exp(unsigned mag) { return max(int(mag >> 20), kFxMinExp); }

// v 2^(59 - E), truncated toward zero (odd in v)
__device__ __forceinline__ FxCoef fx_limbs(double v, int em) {
  const int h = __double2hiint(v), s = h >> 31;
  const unsigned l = unsigned(__double2loint(v));
  const unsigned mh = (unsigned(h) & 0xfffffu) | 0x100000u;
  const unsigned long long m =
      ((unsigned long long)__funnelshift_l(l, mh, 6) << 32) | (l << 6);
  unsigned long long q;  // a shift by 64 or more gives 0
  asm("shr.b64 %0, %1, %2;" : "=l"(q) : "l"(m), "r"(em - ((h >> 20) & 0x7ff)));
  const FxCoef a = fx_split((long long)q);
  return FxCoef{(a.hi ^ s) - s, (a.lo ^ s) - s};
}

// Lines whose results need the general conversion: one with an Inf or NaN
// (exponent 2047), or with magnitudes outside 2^[-722, 777] that do not all
// vanish.
__device__ __forceinline__ bool fx_edge(unsigned mag) {
  return mag != 0 && (mag >> 20) - 300u > 1500u;
}

// R 2^(bx - 1023) for a line that fx_edge names
static __device__ __noinline__ double fx_to_edge(long long R, int bx, unsigned mag) {
  if (mag >= 0x7ff00000u) return __longlong_as_double(0x7ff8000000000000LL);
  return ldexp(double(R), bx - 1023);
}

// R 2^(bx - 1023) rounded to FP64, by integer instructions
__device__ __forceinline__ double fx_to(long long R, int bx) {
  const int rh = int(R >> 32), s = rh >> 31;
  const unsigned ah = unsigned(rh ^ s), al = unsigned(R) ^ unsigned(s);
  int n = __clz(int(ah));
  if (ah == 0) n = 32 + __clz(int(al));
  // the leading bit to bit 62, 53 bits kept, rounded half up: a carry into the
  // next power of two adds one to the exponent field, as it should
  unsigned long long t;
  asm("shl.b64 %0, %1, %2;" : "=l"(t) : "l"(((unsigned long long)ah << 32) | al), "r"(n - 1));
  t = (t + 0x200) >> 10;
  unsigned hw = unsigned(t >> 32) + (unsigned(bx + 62 - n) << 20);
  if ((ah | al) == 0) hw = 0;
  return __hiloint2double(int(hw | (unsigned(s) & 0x80000000u)), int(unsigned(t)));
}

// Sum of terms c v, three integer multiply-adds each, in units of
// 2^(60 - K) of c v, rounded (the half unit is the start of mm).
template <int K>
struct FxSum {
  long long hh = 0, mm = 1LL << (29 - K);
  __device__ __forceinline__ void add(FxCoef c, FxCoef v) {
    hh += (long long)c.hi * v.hi;
    mm += (long long)c.lo * v.hi;
    mm += (long long)c.hi * v.lo;
  }
  __device__ __forceinline__ long long value() const { return (hh << K) + (mm >> (30 - K)); }
};

// sums and differences of a line's mirrored points (limb by limb: exact)
template <int N>
struct FxPairs {
  static constexpr int P = N / 2, H = (N + 1) / 2;
  FxCoef e[H], o[P > 0 ? P : 1];
  __device__ __forceinline__ void set(const double (&v)[N], int em) {
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const FxCoef x = fx_limbs(v[m], em), y = fx_limbs(v[N - 1 - m], em);
      e[m] = FxCoef{x.hi + y.hi, x.lo + y.lo};
      o[m] = FxCoef{x.hi - y.hi, x.lo - y.lo};
    }
    if (N % 2) e[P] = fx_limbs(v[P], em);
  }
  // values at the two faces in units of the interpolation row
  __device__ __forceinline__ void faces(const HexFxOps& op, long long* f0, long long* f1) const {
    FxSum<0> s, d;
#pragma unroll
    for (int m = 0; m < H; ++m) s.add(op.ie[m], e[m]);
#pragma unroll
    for (int m = 0; m < P; ++m) d.add(op.io[m], o[m]);
    const long long x = s.value(), y = d.value();
    *f0 = x + y;
    *f1 = x - y;
  }
  // derivative of the line plus the correction of the jumps j0, j1 at its
  // minus and plus face (both along +direction): r[N] in units of 2^(60 - K)
  // of the row
  template <int K>
  __device__ __forceinline__ void derivative(const HexFxLine& L, FxCoef j0, FxCoef j1,
                                             long long* r) const {
    const FxCoef je{j0.hi + j1.hi, j0.lo + j1.lo}, jo{j0.hi - j1.hi, j0.lo - j1.lo};
#pragma unroll
    for (int i = 0; i < H; ++i) {
      FxSum<K> b;
#pragma unroll
      for (int m = 0; m < P; ++m) b.add(L.b[i][m], o[m]);
      b.add(L.cb[i], jo);
      const long long y = b.value();
      if (i == P) {  // the middle row has no A part
        r[i] = y;
        continue;
      }
      FxSum<K> a;
#pragma unroll
      for (int m = 0; m < H; ++m) a.add(L.a[i][m], e[m]);
      a.add(L.ca[i], je);
      const long long x = a.value();
      r[i] = y + x;
      r[N - 1 - i] = y - x;
    }
  }
};

// Barrier of one element's warps: named barrier le of the CTA (constant
// numbers, so that only EPB barriers are reserved).
template <int WPE, int EPB>
__device__ __forceinline__ void fx_sync(int le) {
  static_assert(EPB <= 4 || WPE == 1, "one named barrier per element");
  if constexpr (WPE == 1) {
    __syncwarp();
  } else if constexpr (EPB == 1) {
    __syncthreads();
  } else {
    constexpr int NT = 32 * WPE;
    if (le == 0) asm volatile("bar.sync 0, %0;" ::"n"(NT) : "memory");
    else if (le == 1) asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
    else if (EPB > 2 && le == 2) asm volatile("bar.sync 2, %0;" ::"n"(NT) : "memory");
    else if (EPB > 2) asm volatile("bar.sync 3, %0;" ::"n"(NT) : "memory");
  }
}

// the N values of a line and their largest magnitude (joined to mag)
template <int N>
__device__ __forceinline__ unsigned fx_load(const double* p, int st, double (&v)[N],
                                            unsigned mag = 0) {
#pragma unroll
  for (int m = 0; m < N; ++m) {
    v[m] = p[m * st];
    mag = max(mag, fx_mag(v[m]));
  }
  return mag;
}

// values at a line's two faces (Gauss-Lobatto: the line's end points)
template <int N>
__device__ __forceinline__ void fx_faces(const HexFxOps& op, const double* p, int st, double* f0,
                                         double* f1) {
  double v[N];
  const unsigned mag = fx_load<N>(p, st, v);
  if (op.gather) {
    *f0 = v[0];
    *f1 = v[N - 1];
    return;
  }
  const int em = fx_exp(mag), bx = em - 1022 + op.sm - 59 + 1023;
  FxPairs<N> w;
  long long r0, r1;
  w.set(v, em);
  w.faces(op, &r0, &r1);
  *f0 = fx_to(r0, bx);
  *f1 = fx_to(r1, bx);
  if (fx_edge(mag)) {
    *f0 = fx_to_edge(r0, bx, mag);
    *f1 = fx_to_edge(r1, bx, mag);
  }
}

// line l of direction d: first slot and stride in a field, and the flux
// point of its minus face (the plus face is N2 further)
template <int N>
__device__ __forceinline__ void fx_line(int d, int l, int* s0, int* st, int* fm) {
  using G = FxGeom<N>;
  const int j = l / N, i = l - j * N;
  *s0 = d == 0 ? G::SY * i + G::SZ * j : d == 1 ? i + G::SZ * j : i + G::SY * j;
  *st = d == 0 ? 1 : d == 1 ? G::SY : G::SZ;
  *fm = 2 * d * G::N2 + l;
}

// Shared memory per element: gradient u [5][PN], du [5][NF], gradient [15][PN];
// volume F^C [5][NF], f~ [15][PN] (8-byte slots), line magnitudes [15][N2].
template <int N>
__host__ __device__ constexpr int hexfx_bytes_per_elem(bool grad) {
  using G = FxGeom<N>;
  return ((grad ? 20 : 15) * G::PN * 8 + 5 * G::NF * 8 + (grad ? 0 : 15 * G::N2 * 4) + 15) / 16 *
         16;
}

// NS gradients: corrected reference gradient by lines, physical gradient by
// S / det J, its 15 components at the flux points by lines.  At the solution
// points the volume kernel needs the viscous flux alone: stored as stress and
// energy flux [ne][9][nu] (15 gradient components would also be 6 more to
// write and read).  RAW: the gradient itself [ne][15][nu], for the
// anti-aliased flux.
template <int N, int EPB, bool RAW>
__global__ void __launch_bounds__(EPB* FxGeom<N>::TPE, N == 3 ? 2 : 3)
    k_hexfx_grad(long long ne, const double* __restrict__ u,
                 const __grid_constant__ TraceArgs<double> ta, const double* __restrict__ smat,
                 const double* __restrict__ rcpdjac, const __grid_constant__ HexFxOps op,
                 Phys<double> ph, double* __restrict__ grad, double* __restrict__ gradf) {
  using G = FxGeom<N>;
  constexpr int NU = G::NU, NF = G::NF, N2 = G::N2, TPE = G::TPE, PN = G::PN;
  constexpr int NFT = (NF + TPE - 1) / TPE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int le = threadIdx.x / TPE, z = threadIdx.x - le * TPE;
  const long long e = (long long)blockIdx.x * (blockDim.x / TPE) + le;
  if (e >= ne) return;  // whole elements: their barriers are their own
  double* us = reinterpret_cast<double*>(smem_raw + le * hexfx_bytes_per_elem<N>(true));
  double* ds = us + 5 * PN;
  double* gs = ds + 5 * NF;
  const bool pt = z < NU;
  const int slot = G::slot(z % N, (z / N) % N, z / N2);
#pragma unroll
  for (int i = 0; i < NFT; ++i) {
    if (z + i * TPE < NF) {
      double own[5], dv[5];
      trace_jump(ta, e, z + i * TPE, NF, own, dv);
#pragma unroll
      for (int k = 0; k < 5; ++k) ds[k * NF + z + i * TPE] = dv[k];
    }
  }
  if (pt) {
#pragma unroll
    for (int k = 0; k < 5; ++k) us[k * PN + slot] = u[(e * 5 + k) * NU + z];
  }
  fx_sync<G::WPE, EPB>(le);
  // lines: (variable, direction, line) -> N reference-gradient values
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    const double j0 = ds[k * NF + fm], j1 = ds[k * NF + fm + N2];
    double v[N];
    const unsigned mag = fx_load<N>(us + k * PN + s0, st, v, max(fx_mag(j0), fx_mag(j1)));
    const int em = fx_exp(mag), bx = em - 1022 + op.sg - 60 + 1023;
    FxPairs<N> w;
    w.set(v, em);
    long long o[N];
    w.template derivative<1>(op.g, fx_limbs(j0, em), fx_limbs(j1, em), o);
    double* q = gs + (d * 5 + k) * PN + s0;
#pragma unroll
    for (int i = 0; i < N; ++i) q[i * st] = fx_to(o[i], bx);
    if (fx_edge(mag)) {
#pragma unroll
      for (int i = 0; i < N; ++i) q[i * st] = fx_to_edge(o[i], bx, mag);
    }
  }
  double S[9], rj = 0.0;
  if (pt) {
#pragma unroll
    for (int r = 0; r < 9; ++r) S[r] = smat[(e * 9 + r) * NU + z];
    rj = rcpdjac[e * NU + z];
  }
  fx_sync<G::WPE, EPB>(le);
  if (pt) {
#pragma unroll
    for (int r = 0; r < 9; ++r) S[r] *= rj;
    double g[3][5];
    double* p = gs + slot;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double g0 = p[k * PN], g1 = p[(5 + k) * PN], g2 = p[(10 + k) * PN];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        g[j][k] = S[j] * g0 + S[3 + j] * g1 + S[6 + j] * g2;
        p[(j * 5 + k) * PN] = g[j][k];
        if (RAW) grad[(e * 15 + j * 5 + k) * NU + z] = g[j][k];
      }
    }
    if (!RAW) {
      double uz[5], tq[9];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = us[k * PN + slot];
      viscous_point(uz, g, ph, tq);
#pragma unroll
      for (int r = 0; r < 9; ++r) grad[(e * 9 + r) * NU + z] = tq[r];
    }
  }
  fx_sync<G::WPE, EPB>(le);
  // (variable, direction, line) -> the three components of the variable's
  // gradient at the line's two faces
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    double* o = gradf + (e * 15 + k) * NF + fm;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double f0, f1;
      fx_faces<N>(op, gs + (j * 5 + k) * PN + s0, st, &f0, &f1);
      o[j * 5 * NF] = f0;
      o[j * 5 * NF + N2] = f1;
    }
  }
}

// Volume kernel: flux and f~ = S F in FP64, then per line the jump F^C - n~ . f~,
// divergence and correction in fixed point; R = -div / J and the RK epilogue
// in FP64, the next stage's u_f by lines in fixed point.  visc: the viscous
// flux of k_hexfx_grad; AA: f~ comes projected in tflux.
template <int N, int EPB, bool NS, bool AA = false>
__global__ void __launch_bounds__(EPB* FxGeom<N>::TPE, N == 3 ? 2 : 3)
    k_hexfx_vol(long long ne, const double* __restrict__ u, const double* __restrict__ visc,
                const double* __restrict__ fc, const double* __restrict__ smat,
                const double* __restrict__ rcpdjac, const __grid_constant__ HexFxOps op,
                Phys<double> ph, HexStage<double, double> sa,
                const double* __restrict__ tflux = nullptr) {
  using G = FxGeom<N>;
  constexpr int NU = G::NU, NF = G::NF, N2 = G::N2, TPE = G::TPE, PN = G::PN;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int le = threadIdx.x / TPE, z = threadIdx.x - le * TPE;
  const long long e = (long long)blockIdx.x * (blockDim.x / TPE) + le;
  if (e >= ne) return;  // whole elements: their barriers are their own
  double* cs = reinterpret_cast<double*>(smem_raw + le * hexfx_bytes_per_elem<N>(false));
  double* ft = cs + 5 * NF;  // [15][PN]: f~, then divergence terms (integers)
  unsigned* ml = reinterpret_cast<unsigned*>(ft + 15 * PN);
  const bool pt = z < NU;
  const int a = z % N, b = (z / N) % N, c = z / N2;
  const int slot = G::slot(a, b, c);
  async_copy(cs, fc + e * 5 * NF, 5 * NF * int(sizeof(double)), z, TPE);
  if (pt) {
    double* p = ft + slot;
    if constexpr (AA) {
#pragma unroll
      for (int q = 0; q < 15; ++q) p[q * PN] = tflux[(e * 15 + q) * NU + z];
    } else {
      double uz[5], tq[9], f[12], S[9];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = u[(e * 5 + k) * NU + z];
      if (NS) {
#pragma unroll
        for (int r = 0; r < 9; ++r) tq[r] = visc[(e * 9 + r) * NU + z];
      }
#pragma unroll
      for (int r = 0; r < 9; ++r) S[r] = smat[(e * 9 + r) * NU + z];
      flux_point<double, NS>(uz, tq, ph, f);
      // row of variable k: the three fluxes F[j][k]
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
  fx_sync<G::WPE, EPB>(le);
  // lines: jump F^C - n~ . f~ at the two faces (scale 2^sm above the line's,
  // |jump| <= 1.5 2^59; times -1 on the minus face), then the N divergence
  // terms, in place of the line's own f~ values
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    double* p = ft + (d * 5 + k) * PN + s0;
    const double c0 = cs[k * NF + fm], c1 = cs[k * NF + fm + N2];
    double v[N];
    const unsigned mag = fx_load<N>(p, st, v, max(fx_mag(c0), fx_mag(c1)));
    const int em = fx_exp(mag);
    FxPairs<N> w;
    w.set(v, em);
    long long f0, f1, o[N];
    w.faces(op, &f0, &f1);
    const FxCoef j0 = fx_split(-((fx_join(fx_limbs(c0, em)) >> op.sm) + f0));
    const FxCoef j1 = fx_split((fx_join(fx_limbs(c1, em)) >> op.sm) - f1);
    w.template derivative<2>(op.v, j0, j1, o);
#pragma unroll
    for (int i = 0; i < N; ++i) p[i * st] = __longlong_as_double(o[i]);
    ml[(d * 5 + k) * N2 + l] = mag;
  }
  fx_sync<G::WPE, EPB>(le);
  double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (pt) {
    double R[5], xr[5], ar[5];
    const double rj = rcpdjac[e * NU + z];
    hex_stage_load(sa, e * 5 * NU + z, NU, xr, ar);
    const int b0 = op.sv - 1022 - 61 + 1023;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      // the point's lines of the three directions, in units of the largest
      const unsigned m0 = ml[k * N2 + b + N * c], m1 = ml[(5 + k) * N2 + a + N * c],
                     m2 = ml[(10 + k) * N2 + a + N * b];
      const unsigned mag = max(m0, max(m1, m2));
      const int em = fx_exp(mag);
      const long long dv = (__double_as_longlong(ft[k * PN + slot]) >> min(em - fx_exp(m0), 63)) +
                           (__double_as_longlong(ft[(5 + k) * PN + slot]) >> min(em - fx_exp(m1), 63)) +
                           (__double_as_longlong(ft[(10 + k) * PN + slot]) >> min(em - fx_exp(m2), 63));
      R[k] = fx_to(dv, em + b0);
      if (fx_edge(mag)) R[k] = fx_to_edge(dv, em + b0, mag);
      R[k] = -R[k] * rj;
    }
    // (the point's u serves bare right-hand sides' unused next value only)
    hex_stage_apply(sa, e * 5 * NU + z, NU, s, R, xr, ar, s);
#pragma unroll
    for (int k = 0; k < 5; ++k) ft[k * PN + slot] = s[k];
  }
  if (sa.uf_next == nullptr) return;
  fx_sync<G::WPE, EPB>(le);
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    double* o = sa.uf_next + (e * 5 + k) * NF + fm;
    double f0, f1;
    fx_faces<N>(op, ft + k * PN + s0, st, &f0, &f1);
    o[0] = f0;
    o[N2] = f1;
  }
}

}  // namespace frgb
