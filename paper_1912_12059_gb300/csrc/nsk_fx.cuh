// nsk_fx.cuh -- the FP64 operator's constant-matrix contractions in integer arithmetic.
//
// Why: an SM of this GPU issues 2 FP64 operations per clock and 58 to 64 32-bit integer
// operations (measured: DFMA 2.0, mad.wide.s32 58, shifts and logic 64 per clock and SM), and the
// two pipes run side by side. Two thirds of the FP64 instructions of a stage are multiply-adds of
// nodal values with the fixed operator matrices (derivative, surface lifting, face interpolation),
// so they move to the integer pipe as exact fixed-point sums; the pointwise physics stays in FP64.
//
// How: the values that meet in one line of a contraction (its NP nodal values and its two face
// values) are brought to one scale, the exponent E of the largest of them, as 62-bit magnitudes in
// two limbs, x = (h 2^32 + l 2^4) 2^(E - 1023 - 61) with h signed and 0 <= l < 2^28; the matrix
// entries are stored the same way at the exponent of the largest row sum. A product takes three
// 32 x 32 -> 64 bit multiply-adds (h h, h l, l h; l l is below the unit of the sum), sums are exact,
// and one normalisation per output rounds to FP64. Nodes and weights are symmetric about the centre of
// the line, so the rows i and NP - 1 - i share their products: one of the sums, one of the differences of
// the line's value pairs (exact), half the multiply-adds of the plain rows. Every bit of a value down to 2^-57 of the line's
// largest one is kept, where FP64 accumulation rounds each partial sum to 2^-53 of itself, so the
// result's error is smaller than that of the FP64 sums it replaces, and it does not depend on the
// order of the terms or on the thread that forms it.
//
// Measured (64^3 elements, N = 3, ms a stage, FP64 sums before): lifting 3.77 -> 1.43, volume 5.15 ->
// 1.73, prolongation 1.35 -> 0.56. Bound now: the lifting by integer issue (ALU pipe 68 %, issue slots
// 62 %, FP64 32 %), the volume kernel by both pipes (FP64 66 %, ALU 64 %) at 3.1 TB/s of DRAM traffic.
//
// Bounds: |h| <= 2^30, pair sums and differences in [-2^31, 2^31 - 1] and their low limbs below 2^29 in
// magnitude, row sums of |matrix h| <= 2^30, at most 4 terms a product sum: |sum h h| <= 2^61,
// |sum (h l + l h)| <= 4 2^59 + 2^59 < 2^62; a row's result is below 2^60 and three directions add up below
// 2^62.
//
// Exceptional values: an infinity or NaN in a line makes every output of the line NaN; a line of
// values below 2^-923 (zeros, subnormals) gives zeros, and so do results below 2^-1022.
#pragma once

#include "nsk_internal.h"

namespace nsk {

// the contraction goes to the integer pipe in FP64 on 2D and 3D elements with lines of 3 nodes or
// more. A line of 2 nodes has 4 multiply-adds per output, fewer FP64 issue slots than its
// conversions cost integer ones; on 1D elements one line is the whole element, and the serial chain
// of a conversion, product and normalisation is longer than 6 FP64 operations (64 elements, N = 3,
// single block: 54 us a step against 48).
template <typename R, int D, int NP>
__host__ __device__ constexpr bool fx_on() {
  return sizeof(R) == 8 && D >= 2 && NP >= 3;
}

constexpr unsigned kFxMin = 100u << 20;  // lines below 2^-923 share that exponent
constexpr int kFxNan = 1 << 16;          // added to the exponent of a line with an infinity or NaN,
                                         // subtracted from that of a line below 2^-923 (its sums are zero)

struct FxVal {
  int h, l;
};

__device__ __forceinline__ unsigned fx_mag(double x) { return (unsigned)__double2hiint(x) & 0x7FFFFFFFu; }

// x at the scale of E (the largest magnitude's high word with its low 20 bits set)
__device__ __forceinline__ FxVal fx_val(double x, unsigned E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned sh = (E - (hi & 0x7FFFFFFFu)) >> 20;
  const unsigned vh = (__funnelshift_l(lo, hi, 9) & 0x1FFFFFFFu) | 0x20000000u;
  unsigned long long v = ((unsigned long long)vh << 32) | (lo << 9);
  asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(sh));  // shifts of 64 and more give zero
  const int s = (int)hi >> 31;
  return FxVal{(int)(unsigned)(v >> 32) ^ s, (int)(((unsigned)v ^ (unsigned)s) >> 4)};
}

struct FxAcc {
  long long hh, cr;
  __device__ __forceinline__ void clear() { hh = cr = 0; }
  __device__ __forceinline__ void mac(const FxVal a, const int2 t) {
    hh += (long long)a.h * t.x;
    cr += (long long)a.h * t.y;
    cr += (long long)a.l * t.x;
  }
  __device__ __forceinline__ long long sum() const { return hh + (cr >> 28); }
};

// exponent of a sum of values at E with a table of biased exponent et
__device__ __forceinline__ int fx_exp(unsigned E, int et) {
  const int e = (int)(E >> 20);
  return e + et + (e >= 0x7FF ? kFxNan : (e <= (int)(kFxMin >> 20) ? -kFxNan : 0));
}

// the sum a of exponent e as FP64, rounded to nearest (sign flipped when NEG)
template <bool NEG>
__device__ __forceinline__ double fx_out(long long a, int e) {
  const unsigned long long s = (unsigned long long)(a >> 63);
  unsigned long long m = ((unsigned long long)a ^ s) - s;
  const int lz = __clzll((long long)m);
  m <<= lz & 63;
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // 2^52 <= r <= 2^53
  const int eb = e - 1019 - lz;                                  // biased exponent - 1 (r carries the hidden bit)
  unsigned hi = (unsigned)(r >> 32) + ((unsigned)eb << 20);
  unsigned lo = (unsigned)r;
  if (m == 0 || eb < 0) hi = lo = 0;
  if (eb >= 2046) hi = 0x7FF80000u;
  const unsigned sg = NEG ? ~(unsigned)s : (unsigned)s;
  return __hiloint2double((int)(hi | (sg & 0x80000000u)), (int)lo);
}

// a >> n for sums at different exponents (n of 64 and more leaves the sign)
__device__ __forceinline__ long long fx_shift(long long a, int n) {
  asm("shr.s64 %0, %0, %1;" : "+l"(a) : "r"(n));
  return a;
}

// Position of value i of line L in shared memory. Lines of 4 values are 32 bytes: the two 16-byte
// halves of every other group of 4 lines change places, so that the 8 lanes of a 16-byte access to
// consecutive lines fall on all 32 banks (4-way instead of 8-way without it for a warp's loads).
template <int NP>
__device__ __forceinline__ int fx_pos(int L, int i) {
  return L * NP + (NP == 4 ? (i ^ ((L >> 1) & 2)) : i);
}
template <int NP>
__device__ __forceinline__ void fx_load(const double* f, int L, double (&x)[NP]) {
  if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 2) {
      const double2 t = *reinterpret_cast<const double2*>(f + fx_pos<NP>(L, j));
      x[j] = t.x;
      x[j + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) x[j] = f[L * NP + j];
  }
}
template <int NP>
__device__ __forceinline__ void fx_store(double* f, int L, const long long (&x)[NP]) {
  if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 2)
      *reinterpret_cast<longlong2*>(f + fx_pos<NP>(L, j)) = make_longlong2(x[j], x[j + 1]);
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) f[L * NP + j] = __longlong_as_double(x[j]);
  }
}

// entries of one direction's operator (NskFx)
template <int NP>
__host__ __device__ constexpr int fx_entries() {
  return (NP / 2) * (NP + 2) + (NP % 2) * ((NP + 2) / 2);
}
// shared-memory copy of the tables (8-byte units): [D][entries] the direction operators, then [NP] l(+-1),
// and for the lifting the direction operators again, times mu
template <int D, int NP>
__host__ __device__ constexpr int fx_tab_smem() {
  return D * fx_entries<NP>() + NP;
}
template <int D, int NP>
__host__ __device__ constexpr int fx_tab_lift_smem() {
  return fx_tab_smem<D, NP>() + D * fx_entries<NP>();
}
template <int D, int NP, bool LIFT>
__device__ __forceinline__ void fx_stage_tables(const NskFx& f, int2* tb) {
  constexpr int NE = fx_entries<NP>();
  for (int x = threadIdx.x; x < D * NE; x += blockDim.x) {
    const int2 v = f.d[x / NE][x % NE];
    tb[x] = v;
    if constexpr (LIFT) {  // the 58-bit entry times mu's 63-bit mantissa, back at 58 bits
      const long long q = __mul64hi(((long long)v.x << 29) + ((long long)v.y << 1), f.mum);
      tb[fx_tab_smem<D, NP>() + x] = make_int2((int)(q >> 28), (int)(q & 0xFFFFFFF));
    }
  }
  for (int x = threadIdx.x; x < NP; x += blockDim.x) tb[D * NE + x] = f.l[x];
}

// n entries of a table, 16 bytes at a time where the row starts so aligned
template <int N, bool PAIRED>
__device__ __forceinline__ void fx_row(const int2* __restrict__ T, int2 (&t)[N]) {
  if constexpr (PAIRED && N % 2 == 0) {
#pragma unroll
    for (int j = 0; j < N; j += 2) {
      const int4 q = *reinterpret_cast<const int4*>(T + j);
      t[j] = make_int2(q.x, q.y);
      t[j + 1] = make_int2(q.z, q.w);
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) t[j] = T[j];
  }
}

// The NP sums of one line: x its nodal values, xp and xm its +1 and -1 face values, T the entries of
// the direction's operator; returns the line's E.
template <int NP>
__device__ __forceinline__ unsigned fx_line(const double (&x)[NP], const double xp, const double xm,
                                            const int2* __restrict__ T, long long (&acc)[NP]) {
  constexpr int W = NP + 2, H = W / 2, HP = NP / 2;
  unsigned m = kFxMin;
#pragma unroll
  for (int j = 0; j < NP; ++j) m = max(m, fx_mag(x[j]));
  m = max(max(m, fx_mag(xp)), fx_mag(xm));
  const unsigned E = m | 0xFFFFFu;
  FxVal sm[W - H], df[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const FxVal a = fx_val(j == 0 ? xm : x[j == 0 ? 0 : j - 1], E);
    const FxVal b = fx_val(j == 0 ? xp : x[j == 0 ? 0 : NP - j], E);
    sm[j] = FxVal{a.h + b.h, a.l + b.l};
    df[j] = FxVal{a.h - b.h, a.l - b.l};
  }
  if constexpr (W % 2) sm[H] = fx_val(x[NP / 2], E);
#pragma unroll
  for (int i = 0; i < HP; ++i) {
    int2 t[W];
    fx_row<W, W % 2 == 0>(T + i * W, t);
    FxAcc a, b;
    a.clear();
    b.clear();
#pragma unroll
    for (int j = 0; j < H; ++j) a.mac(df[j], t[j]);
#pragma unroll
    for (int j = 0; j < W - H; ++j) b.mac(sm[j], t[H + j]);
    const long long sa = a.sum(), sb = b.sum();
    acc[i] = sa + sb;
    acc[NP - 1 - i] = sa - sb;
  }
  if constexpr (NP % 2) {
    FxAcc a;
    a.clear();
#pragma unroll
    for (int j = 0; j < H; ++j) a.mac(df[j], T[HP * W + j]);
    acc[HP] = a.sum();
  }
  return E;
}

// both face values of one line as sums at the returned exponent: x its nodal values, T the entries of
// l(+-1) (biased exponent et)
template <int NP>
__device__ __forceinline__ int fx_ends_sum(const double (&x)[NP], const int2* __restrict__ T, const int et,
                                           long long& om, long long& op) {
  constexpr int H = NP / 2;
  unsigned m = kFxMin;
#pragma unroll
  for (int j = 0; j < NP; ++j) m = max(m, fx_mag(x[j]));
  const unsigned E = m | 0xFFFFFu;
  FxAcc a, b;
  a.clear();
  b.clear();
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const FxVal u = fx_val(x[j], E), v = fx_val(x[NP - 1 - j], E);
    a.mac(FxVal{u.h + v.h, u.l + v.l}, T[j]);
    b.mac(FxVal{u.h - v.h, u.l - v.l}, T[NP - H + j]);
  }
  if constexpr (NP % 2) a.mac(fx_val(x[H], E), T[H]);
  const long long sa = a.sum(), sb = b.sum();
  op = sa + sb;
  om = sa - sb;
  return fx_exp(E, et);
}
template <int NP>
__device__ __forceinline__ void fx_ends(const double (&x)[NP], const int2* __restrict__ T, const int et, double& om,
                                        double& op) {
  long long m, p;
  const int e = fx_ends_sum<NP>(x, T, et, m, p);
  om = fx_out<false>(m, e);
  op = fx_out<false>(p, e);
}
// one of them (+1 when plus)
template <int NP>
__device__ __forceinline__ double fx_end(const double (&x)[NP], const int2* __restrict__ T, const int et,
                                         const bool plus) {
  long long m, p;
  const int e = fx_ends_sum<NP>(x, T, et, m, p);
  return fx_out<false>(plus ? p : m, e);
}

}  // namespace nsk
