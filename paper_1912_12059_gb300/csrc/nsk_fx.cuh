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
// the line's value pairs (exact), half the multiply-adds of the plain rows. A value keeps its bits down to
// 2^-57 of the line's largest one, so an output's error is some 2^-58 of that value times the row's entries,
// whatever the order of the terms or the thread that forms it: below the rounding of FP64 sums (2^-53 of each
// partial sum) in every row that the largest value enters with an entry of ordinary size.
// A row that the largest value does not enter would lose bits of its own, smaller values: rows with exact
// zeros in the operator. On Gauss-Lobatto nodes the interpolation to the faces takes the end nodes as they are,
// and a face value enters its end row alone, so the nodes keep a scale of their own and the end rows have
// theirs. A node's own entry is zero with 3 nodes (the middle one) and on 4 Gauss-Lobatto nodes: a line in which
// such a node is 2^3 times as large as the others takes plain FP64 sums, brought to the fixed-point form row by
// row (fx_leaves). A line whose largest value lies outside the range in which sums neither overflow nor lose bits
// below 2^-1022 (NskFx; infinities, NaN and tiny values among them) takes FP64 sums and hands them on as they are.
//
// Measured (64^3 elements, N = 3, ms a stage, FP64 sums before): lifting 3.77 -> 1.42, volume 5.15 ->
// 1.82, prolongation 1.35 -> 0.56 (without the provisions for zero entries and for the range: 1.43, 1.73, 0.56). Bound now: the lifting by integer issue (ALU pipe 68 %, issue slots
// 67 %, FP64 33 %), the volume kernel by both pipes (FP64 63 %, ALU 62 %) at 3.0 TB/s of DRAM traffic.
//
// Bounds: |h| <= 2^30, pair sums and differences in [-2^31, 2^31 - 1] and their low limbs below 2^29 in
// magnitude, row sums of |matrix h| <= 2^30, at most 4 terms a product sum: |sum h h| <= 2^61,
// |sum (h l + l h)| <= 4 2^59 + 2^59 < 2^62; a row's result is below 2^60 and three directions add up below
// 2^62.
//
// Values below 2^-1042 count as zero.
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

constexpr unsigned kFxMin = 100u << 20;  // the least scale (2^-923): zeros have lost all their bits there
constexpr unsigned kFxGrade = 3u << 20;  // a value 2^-3 of the line's largest keeps 54 bits
constexpr int kFxZero = 1 << 16;         // subtracted from the exponent of a line of zeros
constexpr int kFxDbl = 1 << 17;          // "exponent" of a line whose sums are FP64 values

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

// exponent of a sum of a line whose largest magnitude is m, with a table of biased exponent et
__device__ __forceinline__ int fx_exp(unsigned m, int et) {
  return m == 0 ? et - kFxZero : (int)(m >> 20) + et;
}

// a >> n for sums at different exponents (n of 64 and more leaves the sign)
__device__ __forceinline__ long long fx_shift(long long a, int n) {
  asm("shr.s64 %0, %0, %1;" : "+l"(a) : "r"(n));
  return a;
}

// the sum a of exponent e as FP64, rounded to nearest (sign flipped when NEG);
// 0 <= eb < 2046 by the range of the lines, eb < 0 for a line of zeros (a negative zero is -1 unit)
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
  const unsigned sg = NEG ? ~(unsigned)s : (unsigned)s;
  return __hiloint2double((int)(hi | (sg & 0x80000000u)), (int)lo);
}

// the sum of a line that may have its sums in FP64
template <bool NEG>
__device__ __forceinline__ double fx_value(long long a, int e) {
  if (e < kFxDbl) return fx_out<NEG>(a, e);
  return NEG ? -__longlong_as_double(a) : __longlong_as_double(a);
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

// Whether a line of the block has its sums in FP64: cleared with the staging of the tables (a
// barrier before the contractions), read after the barrier behind them.
__device__ __forceinline__ int& fx_any_dbl() {
  __shared__ int any;
  return any;
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
  if (threadIdx.x == 0) fx_any_dbl() = 0;
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

// whether a line's largest magnitude m lies outside the fixed-point form's range (a line of zeros does not)
__device__ __forceinline__ bool fx_out_of_range(const NskFx& f, unsigned m) { return m - f.lo >= f.span && m != 0; }
// Whether a line takes FP64 sums, mn and mf the largest magnitudes of its nodal and face values. (5 and 6
// nodes: the FP64 operator's own entry of a node in its row, zero but for rounding, is off by more than the
// fixed-point form loses there.)
template <int NP>
__device__ __forceinline__ bool fx_leaves(const NskFx& f, const double (&x)[NP], const unsigned mn, const unsigned mf) {
  bool r = fx_out_of_range(f, max(mn, mf));
  if constexpr (NP == 3) r = r || fx_mag(x[1]) > max(max(fx_mag(x[0]), fx_mag(x[2])), f.lobatto ? 0 : mf) + kFxGrade;
  if (f.lobatto) {
    r = r || fx_out_of_range(f, mn);
    if constexpr (NP == 4) {
      const unsigned u = fx_mag(x[1]), v = fx_mag(x[2]), o = max(fx_mag(x[0]), fx_mag(x[3]));
      r = r || max(u, v) > max(o, min(u, v)) + kFxGrade;
    }
  }
  return r;
}

// Exponents of a line's sums: of its inner rows, of row 0 and of row NP - 1, and of row 2 of 4. Lines of 3 nodes and
// lines on Gauss-Lobatto nodes use all of them, others `in` alone.
struct FxExp {
  int in, lo, hi, in2;
};
// an FP64 value as a sum of its own exponent, v = a 2^(e - 2104), |a| < 2^59
__device__ __forceinline__ int fx_from(double v, long long& a) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7FF);
  a = ((b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll) << 6;
  if (b < 0) a = -a;
  if (e == 0) a = 0;
  return e == 0 ? -kFxZero : e + 1023;
}
// where a line's exponents are kept: in the places of its -1 and +1 face values (stride doubles apart)
template <int NP>
__device__ __forceinline__ void fx_keep(const NskParams& p, double* fm, const int stride, const FxExp e) {
  *fm = __hiloint2double(e.lo, e.in);
  if (NP == 3 || p.fx.lobatto) fm[stride] = __hiloint2double(e.hi, e.in2);
}
// offset (32-bit words from fm) of the exponent of row i
template <int NP>
__device__ __forceinline__ int fx_word(const NskParams& p, const int i, const int stride) {
  if (NP != 3 && !p.fx.lobatto) return 0;
  return i == 0 ? 1 : (i == NP - 1 ? 2 * stride + 1 : (NP == 4 && i == 2 ? 2 * stride : 0));
}

// One line of f in FP64 sums (see fx_leaves), stored with its exponents: FP64 values out of range, else, where a
// node's own entry is zero (3 and 4 nodes), a fixed-point sum of its own scale for each row. The kernels come
// back to such lines after all others, so that the rare case takes no registers in the loop over them.
template <int NP>
__device__ __forceinline__ void fx_plain(const NskParams& p, const int k, const bool mu, double* f, const int L,
                                         double* fm, const int stride) {
  double x[NP];
  fx_load<NP>(f, L, x);
  const double xm = *fm, xp = fm[stride];
  const NskTab<double>& t = p.td;
  unsigned mn = 0;
#pragma unroll
  for (int j = 0; j < NP; ++j) mn = max(mn, fx_mag(x[j]));
  const bool dbl = fx_out_of_range(p.fx, max(mn, max(fx_mag(xm), fx_mag(xp)))) || fx_out_of_range(p.fx, mn) || NP > 4;
  long long acc[NP];
  int er[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) s = fma(t.dk[k][i * NSK_MAXNP + j], x[j], s);
    s = fma(xm, 0.5 * t.lmk[k][i], fma(-xp, 0.5 * t.lpk[k][i], s));
    if (mu) s *= t.mu;
    er[i] = kFxDbl;
    acc[i] = __double_as_longlong(s);
    if (!dbl) er[i] = fx_from(s, acc[i]);
  }
  if (dbl) fx_any_dbl() = 1;
  fx_store<NP>(f, L, acc);
  fx_keep<NP>(p, fm, stride, FxExp{er[1], er[0], er[NP - 1], er[NP == 4 ? 2 : 1]});
}
// The NP sums of one line: x its nodal values, xp and xm its doubled +1 and -1 face values (without their part
// on Gauss-Lobatto nodes: fx_keep_line), T the entries of the direction's operator (times mu or not), m the
// magnitude of the sums' scale. False (the sums are then of no use: a branch around them would cost more than the
// rare line) for a line that takes FP64 sums.
template <int NP>
__device__ __forceinline__ bool fx_line(const NskParams& p, const double (&x)[NP], const double xp, const double xm, const int2* __restrict__ T,
                                        long long (&acc)[NP], unsigned& m) {
  constexpr int W = NP + 2, H = W / 2, HP = NP / 2;
  const unsigned mm = fx_mag(xm), mp = fx_mag(xp);
  unsigned mn = 0;
#pragma unroll
  for (int j = 0; j < NP; ++j) mn = max(mn, fx_mag(x[j]));
  const bool fits = !fx_leaves<NP>(p.fx, x, mn, max(mm, mp));
  double gm = xm, gp = xp;
  m = max(mn, max(mm, mp));
  if (p.fx.lobatto) {
    gm = gp = 0.0;
    m = mn;
  }
  const unsigned E = max(m, kFxMin) | 0xFFFFFu;
  FxVal sm[W - H], df[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const FxVal a = fx_val(j == 0 ? gm : x[j == 0 ? 0 : j - 1], E);
    const FxVal b = fx_val(j == 0 ? gp : x[j == 0 ? 0 : NP - j], E);
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
  return fits;
}
// The sums of fx_line into the place of the line, with their exponents; on Gauss-Lobatto nodes each face value first
// goes into its end row, at the larger of the two scales (its entry is 2 T[0]). From shared memory once
// more: held since fx_line, the face values would take the registers of its products.
template <int NP>
__device__ __forceinline__ void fx_keep_line(const NskParams& p, const int k, const bool mu, const int2* __restrict__ T,
                                             const long long (&acc)[NP], const unsigned m, double* f, const int L,
                                             double* fm, const int stride) {
  fx_store<NP>(f, L, acc);
  const int et = p.fx.ed[k] + (mu ? p.fx.mue : 0);
  FxExp e;
  e.in = e.lo = e.hi = e.in2 = fx_exp(m, et);
  if (p.fx.lobatto) {
    const int2 t = T[0];
    auto face = [&](const int row, const double g) {
      const unsigned M = max(m, fx_mag(g)), Ef = max(M, kFxMin) | 0xFFFFFu, E = max(m, kFxMin) | 0xFFFFFu;
      double* o = f + fx_pos<NP>(L, row);
      FxAcc c;
      c.clear();
      c.mac(fx_val(g, Ef), t);
      *o = __longlong_as_double(fx_shift(__double_as_longlong(*o), (int)((Ef - E) >> 20)) + 2 * c.sum());
      return fx_exp(M, et);
    };
    e.lo = face(0, *fm);
    e.hi = face(NP - 1, -fm[stride]);
  }
  fx_keep<NP>(p, fm, stride, e);
}

// both face values of one line: x its nodal values, T the entries of l(+-1)
template <int NP>
__device__ __forceinline__ void fx_ends(const NskParams& p, const double (&x)[NP], const int2* __restrict__ T,
                                        double& om, double& op) {
  constexpr int H = NP / 2;
  if (p.fx.lobatto) {  // the end nodes lie on the faces
    om = x[0];
    op = x[NP - 1];
    return;
  }
  unsigned m = 0;
#pragma unroll
  for (int j = 0; j < NP; ++j) m = max(m, fx_mag(x[j]));
  if (fx_out_of_range(p.fx, m)) {
    om = op = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      om = fma(p.td.lm[j], x[j], om);
      op = fma(p.td.lp[j], x[j], op);
    }
    return;
  }
  const unsigned E = max(m, kFxMin) | 0xFFFFFu;
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
  const int e = fx_exp(m, p.fx.el);
  om = fx_out<false>(sa - sb, e);
  op = fx_out<false>(sa + sb, e);
}
// one of them (+1 when plus)
template <int NP>
__device__ __forceinline__ double fx_end(const NskParams& p, const double (&x)[NP], const int2* __restrict__ T,
                                         const bool plus) {
  double om, op;
  fx_ends<NP>(p, x, T, om, op);
  return plus ? op : om;
}

}  // namespace nsk
