// FP64 hexahedron kernels whose linear operators run on the integer pipe.
//
// GB300 issues FP64 instructions at 2 lanes per clock and SM, and 32 x 32 +
// 64-bit integer multiply-adds (IMAD.WIDE) at 64 (measured: 54.6 against 1.6
// per clock in chains of each).  The FP64 gradient and volume kernels were
// bound by that FP64 pipe (0.94 of its rate), most of it in products with
// the line operators and the metric.  Here those products are fixed-point
// sums:
//
//   - a field (one variable of one element) is converted to fixed point
//     relative to its largest magnitude in the element, q = v 2^(59 - E),
//     |v| < 2^E, held as two signed limbs q = hi 2^30 + lo (8 bytes, as the
//     double it replaces);
//   - operator and metric entries are limbs too, scaled by a power of two
//     that bounds the row's sum of magnitudes, so no sum can overflow;
//   - a term is three multiply-adds, hi hi' into one 64-bit sum and
//     hi lo' + lo hi' into another (lo lo' is below the result's unit);
//   - the derivative and interpolation rows of the symmetric line points
//     are applied to sums and differences of mirrored points (exact in
//     integers), which halves the terms;
//   - a result has a unit of about 2^-60 of its bound |A|_inf max|v| and is
//     normalised and rounded once to FP64.
//
// FP64 multiply-adds round every partial sum.  Over random smooth fields and
// sheared metrics the chain flux -> transformed flux -> jump -> divergence at a
// point is 4e-16, 1.1e-15 and 1.0e-15 (rms, p = 2, 3, 4, for a flux of one)
// from exact rational arithmetic with the exact operators; FP64 loops with
// FP64 operators are 1.3e-14, 4e-15 and 1.1e-13 from it.  The flux, the
// scaling by 1/J and the RK update stay in FP64.  A field that holds an Inf
// or NaN gives NaN, which the epilogue flags as before.
//
// Threads: TPE = 32 ceil(N^3 / 32) per element (whole warps, so that the
// field maxima reduce by warp), one per solution point in the pointwise
// phases and one per (field, line) in the line phases.  A line thread reads
// its N points once for all N results (and both face values), with
// coefficients that are the same for every thread (constant operands);
// one thread per point read every line N times, with lane-varying
// coefficients.
//
// Measured per launch, 24^3 p = 4 (20^3 p = 3) Navier-Stokes: gradient 850 -> 301
// us (242 -> 100; 344 with the solution jumps taken in the kernel, which
// saves the 43 us of a kernel for them), volume 1108 -> 268 us (321 -> 95).  What bounds them now:
// the ALU pipe and the FP64 pipe are each at 48-59 %, the rest is the latency
// of dependent integer instructions at 24 warps per SM (80 registers; 64
// spill, 96 leave fewer warps, both slower).
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

// a 64-bit integer as the two words of a slot
__device__ __forceinline__ FxCoef fx_pack(long long q) {
  return FxCoef{int(q >> 32), int(uint32_t(q))};
}

__device__ __forceinline__ long long fx_unpack(FxCoef a) {
  return (long long)(((unsigned long long)uint32_t(a.hi) << 32) | uint32_t(a.lo));
}

// magnitude bits of v's high word: the field maximum reduces on these
__device__ __forceinline__ unsigned fx_mag(double v) {
  return unsigned(__double2hiint(v)) & 0x7fffffffu;
}

// Field exponents below this are taken as this (values under 2^-890 resolve
// to 2^-949): the shifts below then need no special case for zero.
constexpr int kFxMinExp = 132;

// v 2^(59 - E) for the field exponent em = E + 1022 (the biased exponent
// field of the largest magnitude, or more), truncated
__device__ __forceinline__ long long fx_from(double v, int em) {
  const int h = __double2hiint(v), s = h >> 31;
  const unsigned l = unsigned(__double2loint(v));
  const unsigned mh = (unsigned(h) & 0xfffffu) | 0x100000u;
  const unsigned long long m =
      ((unsigned long long)__funnelshift_l(l, mh, 6) << 32) | (l << 6);
  unsigned long long q;  // a shift by 64 or more gives 0
  asm("shr.b64 %0, %1, %2;" : "=l"(q) : "l"(m), "r"(em - ((h >> 20) & 0x7ff)));
  // (the sign as one's complement: one unit)
  return (long long)(q ^ (((unsigned long long)unsigned(s) << 32) | unsigned(s)));
}

// Whether every result of a field with exponent em (and a metric exponent
// jx) is a normal number; a field with Inf / NaN (em = 2047) is not.
__device__ __forceinline__ bool fx_edge(int em, int jx = 1023) {
  return em < 300 || em > 1800 || jx < 700 || jx > 1400;
}

// R 2^(bx - 1023) for a field that fx_edge names
static __device__ __noinline__ double fx_to_edge(long long R, int bx, bool bad) {
  if (bad) return __longlong_as_double(0x7ff8000000000000LL);
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
  __device__ __forceinline__ void load(const FxCoef* p, int st) {
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const FxCoef x = p[m * st], y = p[(N - 1 - m) * st];
      e[m] = FxCoef{x.hi + y.hi, x.lo + y.lo};
      o[m] = FxCoef{x.hi - y.hi, x.lo - y.lo};
    }
    if (N % 2) e[P] = p[P * st];
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

// Maxima over an element of NV magnitudes per thread: warp maxima to
// ex[warp][NV], read after the caller's fx_sync by fx_field_max.
template <int NV>
__device__ __forceinline__ void fx_warp_max(const unsigned (&m)[NV], unsigned* ex, int w) {
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const unsigned r = __reduce_max_sync(0xffffffffu, m[k]);
    if ((threadIdx.x & 31) == 0) ex[w * NV + k] = r;
  }
}

template <int NV, int WPE>
__device__ __forceinline__ unsigned fx_field_max(const unsigned* ex, int k) {
  unsigned r = ex[k];
#pragma unroll
  for (int w = 1; w < WPE; ++w) r = max(r, ex[w * NV + k]);
  return r;
}

// The same into words that are zero before (an earlier barrier): lane q
// of each warp adds the warp's maximum of field q.
template <int NV>
__device__ __forceinline__ void fx_max_to(const unsigned (&m)[NV], unsigned* ex) {
  const unsigned lane = threadIdx.x & 31;
  unsigned mine = 0;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const unsigned r = __reduce_max_sync(0xffffffffu, m[k]);
    if (lane == k) mine = r;
  }
  if (lane < NV) atomicMax(ex + lane, mine);
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

// Fixed-point metric of an element: S (one exponent) and, for Navier-Stokes,
// S / det J (one exponent per physical direction, the columns of S).  ex
// [ne][4]: exponents em (as fx_from) of S and of the three columns.  One
// warp per element; built once per mesh.
template <int NU>
__global__ void k_fx_metric(long long ne, const double* __restrict__ smat,
                            const double* __restrict__ rcpdjac, FxCoef* __restrict__ sq,
                            FxCoef* __restrict__ jq, int* __restrict__ ex) {
  const int lane = threadIdx.x & 31;
  const long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (e >= ne) return;  // whole warps
  unsigned m[4] = {0, 0, 0, 0};
  for (int z = lane; z < NU; z += 32)
    for (int r = 0; r < 9; ++r) {
      const double s = smat[(e * 9 + r) * NU + z];
      m[0] = max(m[0], fx_mag(s));
      m[1 + r % 3] = max(m[1 + r % 3], fx_mag(s * rcpdjac[e * NU + z]));
    }
  for (int k = 0; k < 4; ++k) {
    m[k] = max(__reduce_max_sync(0xffffffffu, m[k]) >> 20, unsigned(kFxMinExp));
    if (lane == 0) ex[e * 4 + k] = int(m[k]);
  }
  // limbs below 2^58: one bit less than a field's, for sums of three
  for (int z = lane; z < NU; z += 32)
    for (int r = 0; r < 9; ++r) {
      const long long i = (e * 9 + r) * NU + z;
      const double s = smat[i];
      sq[i] = fx_split(fx_from(s, int(m[0]) + 1));
      if (jq) jq[i] = fx_split(fx_from(s * rcpdjac[e * NU + z], int(m[1 + r % 3]) + 1));
    }
}

// Shared memory per element (8-byte slots): gradient u [5][PN], du [5][NF],
// gradient [15][PN]; volume f~ [15][PN], F^C / jump [5][NF]; then warp maxima
// of up to 6 fields, element maxima of up to 15 and 8 exponents.
template <int N>
__host__ __device__ constexpr int hexfx_bytes_per_elem(bool grad) {
  using G = FxGeom<N>;
  const int slots = (grad ? 20 : 15) * G::PN + 5 * G::NF;
  return (slots * 8 + (G::WPE * 6 + 16 + 8) * 4 + 15) / 16 * 16;
}

// NS gradients: corrected reference gradient
// by lines, physical gradient by the fixed-point S / det J, its 15 components
// at the flux points by lines.  At the solution points the volume kernel
// needs the viscous flux alone: it is formed here, where the FP64 pipe is
// otherwise idle, and stored as stress and energy flux [ne][9][nu] (15
// gradient components would also be 6 more to write and read).  RAW: the
// gradient itself [ne][15][nu], for the anti-aliased flux.
template <int N, int EPB, bool RAW>
__global__ void __launch_bounds__(EPB* FxGeom<N>::TPE, N == 3 ? 2 : 3)
    k_hexfx_grad(long long ne, const double* __restrict__ u,
                 const __grid_constant__ TraceArgs<double> ta,
                 const FxCoef* __restrict__ jq, const int* __restrict__ jex,
                 const __grid_constant__ HexFxOps op, Phys<double> ph,
                 double* __restrict__ grad, double* __restrict__ gradf) {
  using G = FxGeom<N>;
  constexpr int NU = G::NU, NF = G::NF, N2 = G::N2, TPE = G::TPE, PN = G::PN;
  constexpr int NFT = (NF + TPE - 1) / TPE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int le = threadIdx.x / TPE, z = threadIdx.x - le * TPE, wz = z >> 5;
  const long long e = (long long)blockIdx.x * (blockDim.x / TPE) + le;
  if (e >= ne) return;  // whole elements: their barriers are their own
  FxCoef* us = reinterpret_cast<FxCoef*>(smem_raw + le * hexfx_bytes_per_elem<N>(true));
  FxCoef* ds = us + 5 * PN;
  FxCoef* gs = ds + 5 * NF;  // [15][PN]: integers by fx_pack, then limbs
  unsigned* ex = reinterpret_cast<unsigned*>(gs + 15 * PN);
  unsigned* eg = ex + 6 * G::WPE;                  // [15] gradient maxima
  int* ek = reinterpret_cast<int*>(eg + 16);       // [5] fields, [3] metric
  const bool pt = z < NU;
  const int a = z % N, b = (z / N) % N, c = z / N2;
  const int slot = G::slot(a, b, c);
  if (z < 15) eg[z] = 0;
  int em[5];
  {
    double uv[5], dv[NFT][5];
    unsigned mx[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      uv[k] = pt ? u[(e * 5 + k) * NU + z] : 0.0;
      mx[k] = fx_mag(uv[k]);
    }
#pragma unroll
    for (int i = 0; i < NFT; ++i) {
      if (z + i * TPE < NF) {
        double own[5];
        trace_jump(ta, e, z + i * TPE, NF, own, dv[i]);
#pragma unroll
        for (int k = 0; k < 5; ++k) mx[k] = max(mx[k], fx_mag(dv[i][k]));
      }
    }
    fx_warp_max<5>(mx, ex, wz);
    fx_sync<G::WPE, EPB>(le);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      em[k] = max(int(fx_field_max<5, G::WPE>(ex, k) >> 20), kFxMinExp);
      if (pt) us[k * PN + slot] = fx_split(fx_from(uv[k], em[k]));
#pragma unroll
      for (int i = 0; i < NFT; ++i)
        if (z + i * TPE < NF) ds[k * NF + z + i * TPE] = fx_split(fx_from(dv[i][k], em[k]));
    }
  }
  fx_sync<G::WPE, EPB>(le);
  // lines: (variable, direction, line) -> N reference-gradient values in
  // units of 2^(E + sg - 60)
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    FxPairs<N> v;
    v.load(us + k * PN + s0, st);
    long long o[N];
    v.template derivative<1>(op.g, ds[k * NF + fm], ds[k * NF + fm + N2], o);
#pragma unroll
    for (int i = 0; i < N; ++i) gs[(d * 5 + k) * PN + s0 + i * st] = fx_pack(o[i]);
  }
  FxCoef J[9];
  int jx[3];
  if (pt) {
#pragma unroll
    for (int r = 0; r < 9; ++r) J[r] = jq[(e * 9 + r) * NU + z];
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) jx[j] = jex[e * 4 + 1 + j];
  bool edge = false;
#pragma unroll
  for (int k = 0; k < 5; ++k) edge |= fx_edge(em[k], jx[k % 3]);
  if (z == 0) {
#pragma unroll
    for (int k = 0; k < 5; ++k) ek[k] = em[k];
#pragma unroll
    for (int j = 0; j < 3; ++j) ek[5 + j] = jx[j];
  }
  fx_sync<G::WPE, EPB>(le);
  // physical gradient g[j][k] = sum_i (S_ij / det J) gref_i, in units of
  // 2^(E + sg + E_j - 61), in place of the reference gradient of the point
  const int b0 = op.sg - 1022 - 1022 - 61 + 1023;  // + em + jx: exponent of a unit
  double g[3][5];
  unsigned mg[15];
#pragma unroll
  for (int q = 0; q < 15; ++q) mg[q] = 0;
  if (pt) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      FxCoef r[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) r[i] = fx_split(fx_unpack(gs[(i * 5 + k) * PN + slot]));
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        FxSum<3> s;
#pragma unroll
        for (int i = 0; i < 3; ++i) s.add(J[i * 3 + j], r[i]);
        const long long x = s.value();
        const int h = int(x >> 32);
        mg[j * 5 + k] = unsigned(h ^ (h >> 31));
        gs[(j * 5 + k) * PN + slot] = fx_pack(x);
        g[j][k] = fx_to(x, b0 + em[k] + jx[j]);
      }
    }
    if (edge) {
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 5; ++k)
          g[j][k] = fx_to_edge(fx_unpack(gs[(j * 5 + k) * PN + slot]), b0 + em[k] + jx[j],
                               em[k] >= 2047);
    }
  }
  fx_max_to<15>(mg, eg);
  if (pt) {
    if (RAW) {
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 5; ++k) grad[(e * 15 + j * 5 + k) * NU + z] = g[j][k];
    } else {
      double uz[5], tq[9];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = u[(e * 5 + k) * NU + z];
      viscous_point(uz, g, ph, tq);
#pragma unroll
      for (int r = 0; r < 9; ++r) grad[(e * 9 + r) * NU + z] = tq[r];
    }
  }
  fx_sync<G::WPE, EPB>(le);
  // each component shifted to the full width of its largest value, |x| < 2^(64
  // - clz): to below 2^63, then 2^59
  if (pt) {
#pragma unroll
    for (int q = 0; q < 15; ++q) {
      const int sh = __clz(int(eg[q])) - 1;
      gs[q * PN + slot] = fx_split((fx_unpack(gs[q * PN + slot]) << sh) >> 4);
    }
  }
  fx_sync<G::WPE, EPB>(le);
  // (variable, direction, line) -> the three components of the variable's
  // gradient at the line's two faces
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    const int bk = b0 + ek[k] + op.sm + 5;
    long long f[6];
    double v[6];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxPairs<N> w;
      w.load(gs + (j * 5 + k) * PN + s0, st);
      w.faces(op, f + 2 * j, f + 2 * j + 1);
    }
    int bx[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      bx[j] = bk + ek[5 + j] - __clz(int(eg[j * 5 + k]));
      v[2 * j] = fx_to(f[2 * j], bx[j]);
      v[2 * j + 1] = fx_to(f[2 * j + 1], bx[j]);
    }
    if (edge) {
#pragma unroll
      for (int i = 0; i < 6; ++i) v[i] = fx_to_edge(f[i], bx[i / 2], ek[k] >= 2047);
    }
    double* o = gradf + (e * 15 + k) * NF + fm;
#pragma unroll
    for (int i = 0; i < 6; ++i) o[(i / 2) * 5 * NF + (i % 2) * N2] = v[i];
  }
}

// Volume kernel: flux in FP64, f~ = S F, jump, divergence and
// correction in fixed point, R = -div / J and the RK epilogue in FP64, the
// next stage's u_f by lines in fixed point.  The three momentum variables
// share one field exponent (their flux tensor is symmetric).  visc: the
// viscous flux of k_hexfx_grad.
template <int N, int EPB, bool NS, bool AA = false>
__global__ void __launch_bounds__(EPB* FxGeom<N>::TPE, N == 3 ? 2 : 3)
    k_hexfx_vol(long long ne, const double* __restrict__ u, const double* __restrict__ visc,
                const double* __restrict__ fc, const FxCoef* __restrict__ sq,
                const int* __restrict__ sex, const double* __restrict__ rcpdjac,
                const __grid_constant__ HexFxOps op, Phys<double> ph,
                HexStage<double, double> sa, const double* __restrict__ tflux = nullptr) {
  using G = FxGeom<N>;
  constexpr int NU = G::NU, NF = G::NF, N2 = G::N2, TPE = G::TPE, PN = G::PN;
  constexpr int NFT = (NF + TPE - 1) / TPE;
  constexpr int kGrp[5] = {0, 1, 1, 1, 2};  // exponent group of a variable
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int le = threadIdx.x / TPE, z = threadIdx.x - le * TPE, wz = z >> 5;
  const long long e = (long long)blockIdx.x * (blockDim.x / TPE) + le;
  if (e >= ne) return;  // whole elements: their barriers are their own
  FxCoef* ft = reinterpret_cast<FxCoef*>(smem_raw + le * hexfx_bytes_per_elem<N>(false));
  FxCoef* jm = ft + 15 * PN;
  unsigned* ex = reinterpret_cast<unsigned*>(jm + 5 * NF);
  unsigned* es = ex + 6 * G::WPE;  // [5] maxima of the next stage value
  const bool pt = z < NU;
  const int a = z % N, b = (z / N) % N, c = z / N2;
  const int slot = G::slot(a, b, c);
  if (z < 5) es[z] = 0;
  // exponents of the point fluxes [0..2] and the interface fluxes [3..5] of
  // the mass, momentum and energy groups; the interface fluxes wait in their
  // slots (read back by the same thread)
  unsigned mx[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < NFT; ++i) {
    if (z + i * TPE < NF) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const double x = fc[(e * 5 + k) * NF + z + i * TPE];
        mx[3 + kGrp[k]] = max(mx[3 + kGrp[k]], fx_mag(x));
        jm[k * NF + z + i * TPE] = fx_pack(__double_as_longlong(x));
      }
    }
  }
  // point fluxes: mass and energy [3] each, momentum tensor [6]; AA: the
  // transformed flux [15]
  constexpr int NV = AA ? 15 : 12;
  double f[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) f[q] = 0.0;
  if (pt) {
    if constexpr (AA) {
#pragma unroll
      for (int q = 0; q < 15; ++q) f[q] = tflux[(e * 15 + q) * NU + z];
    } else {
      double uz[5], tq[9];
#pragma unroll
      for (int k = 0; k < 5; ++k) uz[k] = u[(e * 5 + k) * NU + z];
      if (NS) {
#pragma unroll
        for (int r = 0; r < 9; ++r) tq[r] = visc[(e * 9 + r) * NU + z];
      }
      flux_point<double, NS>(uz, tq, ph, f);
    }
  }
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int gq = AA ? kGrp[q % 5] : (q < 3 ? 0 : q < 9 ? 1 : 2);
    mx[gq] = max(mx[gq], fx_mag(f[q]));
  }
  fx_warp_max<6>(mx, ex, wz);
  FxCoef S[9];
  int se = 1023;
  if (!AA) {
    if (pt) {
#pragma unroll
      for (int r = 0; r < 9; ++r) S[r] = sq[(e * 9 + r) * NU + z];
    }
    se = sex[e * 4];
  }
  fx_sync<G::WPE, EPB>(le);
  // common exponent of f~ and F^C per group; f~ = S F is below
  // 3 2^(E_F + E_S) < 2^(E_F + E_S + 2)
  int ef[3], ev[3], sh[3];
  bool bad[3], edge = false;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    ef[q] = max(int(fx_field_max<6, G::WPE>(ex, q) >> 20), kFxMinExp);
    const int ec = int(fx_field_max<6, G::WPE>(ex, 3 + q) >> 20);
    const int eft = AA ? ef[q] : ef[q] + se - 1022 + 2;
    bad[q] = ef[q] >= 2047 || ec >= 2047;
    ev[q] = max(max(eft, ec), kFxMinExp);
    sh[q] = min(ev[q] - eft, 63);
    edge |= bad[q] || fx_edge(ev[q], se);
  }
  if (pt) {
    if constexpr (AA) {
#pragma unroll
      for (int q = 0; q < 15; ++q) ft[q * PN + slot] = fx_split(fx_from(f[q], ev[kGrp[q % 5]]));
    } else {
      FxCoef F[12];
#pragma unroll
      for (int q = 0; q < 12; ++q)
        F[q] = fx_split(fx_from(f[q], ef[q < 3 ? 0 : q < 9 ? 1 : 2]));
      // row of variable k: the three fluxes F[j][k]
      constexpr int kIdx[5][3] = {{0, 1, 2}, {3, 6, 7}, {6, 4, 8}, {7, 8, 5}, {9, 10, 11}};
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          FxSum<0> s;
#pragma unroll
          for (int j = 0; j < 3; ++j) s.add(S[d * 3 + j], F[kIdx[k][j]]);
          ft[(d * 5 + k) * PN + slot] = fx_split(s.value() >> sh[kGrp[k]]);
        }
    }
  }
#pragma unroll
  for (int i = 0; i < NFT; ++i)
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (z + i * TPE < NF) {
        FxCoef* p = jm + k * NF + z + i * TPE;
        *p = fx_split(fx_from(__longlong_as_double(fx_unpack(*p)), ev[kGrp[k]]));
      }
  fx_sync<G::WPE, EPB>(le);
  // lines: jump F^C - n~ . f~ at the two faces (scale 2^sm above the field's,
  // |jump| <= 1.5 2^59; times -1 on the minus face), then the N divergence
  // terms, in place of the line's own f~ values
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    FxCoef* p = ft + (d * 5 + k) * PN + s0;
    FxPairs<N> v;
    v.load(p, st);
    long long f0, f1, o[N];
    v.faces(op, &f0, &f1);
    const long long cm = fx_join(jm[k * NF + fm]), cp = fx_join(jm[k * NF + fm + N2]);
    const FxCoef j0 = fx_split(-((cm >> op.sm) + f0));
    const FxCoef j1 = fx_split((cp >> op.sm) - f1);
    v.template derivative<2>(op.v, j0, j1, o);
#pragma unroll
    for (int i = 0; i < N; ++i) p[i * st] = fx_pack(o[i]);
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
      const long long dv = fx_unpack(ft[k * PN + slot]) + fx_unpack(ft[(5 + k) * PN + slot]) +
                           fx_unpack(ft[(10 + k) * PN + slot]);
      const int q = kGrp[k];
      R[k] = fx_to(dv, ev[q] + b0);
      if (edge) R[k] = fx_to_edge(dv, ev[q] + b0, bad[q]);
      R[k] = -R[k] * rj;
    }
    // (the point's u serves bare right-hand sides' unused next value only)
    hex_stage_apply(sa, e * 5 * NU + z, NU, s, R, xr, ar, s);
  }
  if (sa.uf_next == nullptr) return;
  unsigned ms[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) ms[k] = fx_mag(s[k]);
  fx_max_to<5>(ms, es);
  fx_sync<G::WPE, EPB>(le);
  if (pt) {
#pragma unroll
    for (int k = 0; k < 5; ++k)
      ft[k * PN + slot] = fx_split(fx_from(s[k], max(int(es[k] >> 20), kFxMinExp)));
  }
  fx_sync<G::WPE, EPB>(le);
  for (int t = z; t < 15 * N2; t += TPE) {
    const int k = t / (3 * N2), r = t - k * 3 * N2, d = r / N2, l = r - d * N2;
    int s0, st, fm;
    fx_line<N>(d, l, &s0, &st, &fm);
    FxPairs<N> v;
    v.load(ft + k * PN + s0, st);
    long long f0, f1;
    v.faces(op, &f0, &f1);
    const int em = max(int(es[k] >> 20), kFxMinExp), bx = em - 1022 + op.sm - 59 + 1023;
    double v0 = fx_to(f0, bx), v1 = fx_to(f1, bx);
    if (fx_edge(em)) {
      v0 = fx_to_edge(f0, bx, em >= 2047);
      v1 = fx_to_edge(f1, bx, em >= 2047);
    }
    double* o = sa.uf_next + (e * 5 + k) * NF + fm;
    o[0] = v0;
    o[N2] = v1;
  }
}

}  // namespace frgb
