// Level-0 operator A0 = c M + A as symmetric element blocks, one thread per
// (element, row): the float64 operator of the outer CG, and the assembled
// smoother, residual and transfers of level 0 in the V-cycle precision.
//
// Storage. A0 is symmetric, so each coupling is kept once: per element the
// packed triangle of its diagonal block, and per interior face one face block
// that both elements read (the second one finds it in the L2: elements are
// numbered so that neighbours are near). Only the part of a coupling that a
// GLL nodal basis can make nonzero is stored. With the DoFs of either element
// in "face-first" order (the NF DoFs of the shared face, then the others),
// the block K of owner e and neighbour n (owner: the lower internal index) is
//   F[c][r] (c < NF, r < B): n's face DoF c against every DoF of e,
//   G[c][j] (c < B - NF, j < NF): n's other DoFs against e's face DoFs,
// i.e. the columns of K one after the other; n reads the same entries as the
// rows of K^T. Column strides are odd, so that both directions are free of
// bank conflicts in shared memory. 2D Q2: 135 instead of 261 stored entries
// per element, 3D Q2: 1,593 instead of 3,159, 3D Q3: 7,456 instead of 14,848.
//
// Blocks and the neighbours' DoFs (coalesced: the threads of an element read one
// neighbour's DoFs together) are copied to shared memory with cp.async and
// multiplied there: per warp through a ring of slots (k_symw, B <= 32), or per
// block of threads in two stages (k_sym, 64 DoFs: one element's blocks are 53
// (float32) or 106 KB, too much per warp).
//
// Measured on GB300 against one thread per element on the blocks of both
// directions (k_spmv / k_cheb with FaceOp), which is FP64-bound in float64 and short
// of loads in flight in float32:
//   float64 product, 64^3 Q2 hexahedra: 1,483 -> 1,010 us with x's copy (3.5 GB, 520
//     us at the copy rate; HBM, the shared-memory data path and the integer
//     multiply-adds are each about half busy: 15 warps per SM overlap them too little)
//   float64 product, 24^3 Q3 hexahedra: 1,340 -> 276 us
//   float64 smoothing step, 18^3 Q3 hexahedra: 1,475 -> 183 us (one stage: 220 us)
//
// Float64 products run on the integer pipe. GB300 issues 2 float64 FMAs per SM and clock
// against 64 32-bit integer multiply-adds (27 that add to 64 bits, as here), so a
// float64 block product is bound by the FP64 pipe, not by HBM. Here the operator is kept in
// 60-bit fixed point and x is converted to 58-bit fixed point with one exponent
// per element; the sum of the products is formed exactly in 64-bit integers (up
// to the product of the low halves, 2^-60 of the row's scale) and rounded once.
// Fixed point needs entries of one magnitude: row and column i are scaled by 2^-s_i,
// 2^{2 s_i} >= A_ii, after which an SPD operator has diagonal entries in (1/4, 1] and
// no entry above 1 in any row (the scales of x and y are powers of two, added to
// exponents: they cost nothing and round nothing). What a small entry loses is then
// 2^-59 sqrt(A_ii A_jj), 1/64 of a double's rounding of the diagonal; the set-up
// bounds the sum of these losses in every row and keeps the float64 form if one
// passes kFxLoss of the row (engine_impl.cuh, sym_scales). One exponent per element
// instead lost the ratio of its diagonal entries: worst row against 80-bit arithmetic,
// relative to (|A| |x|)_i, Q2 shell 2.4e-15 -> 1.1e-16 (float64 sums: 6e-16), Q3 cube
// 1.4e-15 -> 1.2e-16 (7e-16), 2D Q3 stiffness with a contrast of 1e-4 in the
// conductivity 2.6e-13 -> 1.6e-15, there kept in float64 (3.6e-16).
// An entry is a1 2^28 + a0 with |a0| <= 2^27, an x is x1 2^31 + x0 with |x0| <= 2^30.
// With sum_j |A_ij| <= 2^60, |A_ij| <= 2^58 (global exponent kA) and |x| <= 2^58, and
// T <= 304 entries in a row:
//   hi = sum a1 x1 <= 2^32 2^27,  m1 = sum a1 x0 <= 2^32 2^30,
//   m2 = sum a0 x1 <= T 2^27 2^27 < 2^62.3,
// so none overflows, and every a1 and x1 fits 32 bits. Vectors of wide range, NaN and
// infinities: see SymVec.
#pragma once
#include "face_op.cuh"
#include "kernels.cuh"

namespace aggmg {

// ---------------------------------------------------------------- fixed point
// bits of a row's entries in sum, of a single entry, of x; of the low halves of
// an entry and of x
constexpr int FX_A = 60, FX_AE = 58, FX_X = 58, FX_P = 28, FX_Q = 31;
constexpr int kFxNone = -100000;                    // exponent of zero
constexpr int kFxInf = 2600;                        // of a NaN or an infinity, above every other scaled one
constexpr int kFxSpan = 6;                          // see SymVec
constexpr int kFxWide = -(1 << 20);                 // added to the exponent of an element kept as doubles
constexpr int kFxRaw = 1823;                        // biased exponent of such an element's largest double
// largest loss of a fixed-point row relative to sum_j |A_ij|: 8 roundings of a double
// (a float64 sum of the row's 135 to 700 products rounds as often as it adds)
constexpr double kFxLoss = 8.0 / 9007199254740992.0;
// exponent of the unit of FxAcc::sum() for x with shared biased exponent E, less E
constexpr int kFxBias = FX_P + FX_Q - 1075 - (FX_X - 53);

// biased exponent of x 2^t
__device__ __forceinline__ int fx_exp(double x, int t) {
  const int h = __double2hiint(x), e = (h >> 20) & 0x7ff;
  if (e == 2047) return kFxInf;
  if (e == 0) return ((h << 1) | __double2loint(x)) ? 1 + t : kFxNone;
  return e + t;
}
// x in units of 2^{E - 1075 - (FX_X - 53)} rounded to an integer (at most 2^FX_X for
// E >= fx_exp(x, 0)), as halves (lo, hi)
__device__ __forceinline__ int2 fx_split(double x, int E) {
  const int h = __double2hiint(x);
  int e = (h >> 20) & 0x7ff;
  unsigned long long m = ((unsigned long long)(unsigned)(h & 0xfffff) << 32) | (unsigned)__double2loint(x);
  if (e) m |= 1ull << 52;
  else e = 1;
  const int sh = min(max(E - e, 0), 63);             // (below 0: x = 0)
  long long v = (long long)((((m << (FX_X - 52)) >> sh) + 1) >> 1);
  v = h < 0 ? -v : v;
  const int lo = ((int)v << (32 - FX_Q)) >> (32 - FX_Q);
  return make_int2(lo, (int)((v - lo) >> FX_Q));
}
// S * 2^q for an integer S
__device__ __forceinline__ double fx_scale(long long S, int q) {
  const double d = (double)S;
  if (q > -1000 && q < 1000) return d * __hiloint2double((q + 1023) << 20, 0);
  return scalbn(d, q);
}

struct FxAcc {
  long long hi = 0, m1 = 0, m2 = 0;
  __device__ __forceinline__ void fma(int2 a, int2 x) {
    hi += (long long)a.y * x.y;
    m1 += (long long)a.y * x.x;
    m2 += (long long)a.x * x.y;
  }
  using Sum = long long;
  // the sum in units of 2^{FX_P + FX_Q}
  __device__ __forceinline__ long long sum() const {
    return hi + ((m1 + (1ll << (FX_Q - 1))) >> FX_Q) + ((m2 + (1ll << (FX_P - 1))) >> FX_P);
  }
};
// S / 2^sh, rounded
__device__ __forceinline__ long long sum_shift(long long S, int sh) {
  if (sh == 0) return S;
  return sh > 62 ? 0 : (S + (1ll << (sh - 1))) >> sh;
}
__device__ __forceinline__ float sum_shift(float s, int) { return s; }
template <typename T>
struct PlAcc {
  T s = T(0);
  __device__ __forceinline__ void fma(T a, T x) { s += a * x; }
  using Sum = T;
  __device__ __forceinline__ T sum() const { return s; }
};

// Stored entry, x entry and accumulator of a value type
template <typename T> struct SymNum;
template <> struct SymNum<double> { using ST = int2; using SX = int2; using SX2 = int4; using Acc = FxAcc; };
template <> struct SymNum<float> { using ST = float; using SX = float; using SX2 = float2; using Acc = PlAcc<float>; };
__device__ __forceinline__ int2 sx_first(int4 v) { return make_int2(v.x, v.y); }
__device__ __forceinline__ int2 sx_second(int4 v) { return make_int2(v.z, v.w); }
__device__ __forceinline__ float sx_first(float2 v) { return v.x; }
__device__ __forceinline__ float sx_second(float2 v) { return v.y; }
__device__ __forceinline__ int2 sym_val(int2 v) { return v; }
__device__ __forceinline__ float sym_val(float v) { return v; }
__device__ __forceinline__ double sym_val(double v) { return v; }
__device__ __forceinline__ float sym_val(__nv_bfloat16 v) { return __bfloat162float(v); }

// ---------------------------------------------------------------- layout
constexpr int round_to(int k, int q) { return (k + q - 1) / q * q; }

template <int B> struct SymShape {
  static constexpr int D = FaceShape<B>::D, N = FaceShape<B>::N;
  static constexpr int NF = FaceIdx<D, N>::NF, NFACE = 2 * D, BO = B - NF;
  static constexpr int LDF = B | 1, LDG = NF | 1, LDP = B | 1;
  static constexpr int TRI = B * (B + 1) / 2;
  // x of one element in shared memory: face DoFs, then the others from an even offset
  static constexpr int XO = round_to(NF, 2), BX = XO + round_to(BO, 2);
};
// entries per element (diagonal), per face block, per transfer block, padded to 16 bytes
template <typename ST, int B> struct SymLay {
  using S = SymShape<B>;
  static constexpr int Q = 16 / (int)sizeof(ST);
  static constexpr int KD = round_to(S::TRI, Q);
  static constexpr int KB = round_to(S::NF * S::LDF + S::BO * S::LDG, Q);
  static constexpr int KP = round_to(B * S::LDP, Q);
};

template <typename T, int B>
struct SymView {
  using ST = typename SymNum<T>::ST;
  const ST* diag;         // [n][KD] packed triangle, entry (i, j), j <= i, at i (i + 1) / 2 + j
  const ST* face;         // [face block][KB]
  const int2* info;       // [n][2d] neighbour's internal index (-1 none), face block
  const int8_t* code;     // [n][2d] neighbour's local face
  const int16_t* sc;      // [n][B] scale exponents s_i (float64)
  int kA;                 // global exponent of the fixed-point entries (float64)
  int64_t n;
};

// smoother block inverses (packed triangles) or transfer blocks of level 0, one
// per element; float64 block inverses: fixed point as the operator's entries, with
// an exponent per element and scale exponents of their own (from their diagonals)
template <typename TS>
struct SymBlk {
  const TS* v;
  const int16_t *k, *s;   // [n], [n][B]
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_x(int2* dst, const int2* src) { cp_async8(dst, src); }
__device__ __forceinline__ void cp_async_x(float* dst, const float* src) { cp_async4(dst, src); }

// position of DoF r in the face-first order of local face f
template <int B>
__device__ __forceinline__ int face_first(int f, int r, bool& on) {
  using S = SymShape<B>;
  constexpr int N = S::N;
  const int k = f >> 1, s = f & 1;
  const int a = r % N, b = (r / N) % N, c = r / (N * N);
  const int ik = (k == 0) ? a : (k == 1 ? b : c);
  int j;
  if constexpr (S::D == 2) j = (k == 0) ? b : a;
  else j = ((k == 0) ? b : a) + N * ((k == 2) ? b : c);
  on = ik == s * (N - 1);
  return on ? j : S::NF + j + S::NF * (ik - (1 - s));
}

// acc += sum_{t < CNT} p[t stride] x[t]
template <typename T, int CNT, typename ST>
__device__ __forceinline__ void sym_dot(const ST* p, int stride, const typename SymNum<T>::SX* x,
                                        typename SymNum<T>::Acc& acc) {
  constexpr int kUnroll = (CNT <= 27) ? (CNT + 1) / 2 : 8;
#pragma unroll kUnroll
  for (int t = 0; t < CNT; t += 2) {
    const auto xx = *reinterpret_cast<const typename SymNum<T>::SX2*>(x + t);
    acc.fma(sym_val(p[t * stride]), sx_first(xx));
    if (CNT % 2 == 0 || t + 1 < CNT) acc.fma(sym_val(p[(t + 1) * stride]), sx_second(xx));
  }
}
// the same for x at any (unpaired) position
template <typename T, int CNT, typename ST>
__device__ __forceinline__ void sym_dot_any(const ST* p, int stride, const typename SymNum<T>::SX* x,
                                            typename SymNum<T>::Acc& acc) {
#pragma unroll
  for (int t = 0; t < CNT; ++t) acc.fma(sym_val(p[t * stride]), x[t]);
}
// acc += sum_c M(r, c) x[c] for a packed triangle M
template <typename T, int B, typename ST>
__device__ __forceinline__ void sym_tri(const ST* m, int r, const typename SymNum<T>::SX* x,
                                        typename SymNum<T>::Acc& acc) {
  const int row = r * (r + 1) / 2;
  constexpr int kUnroll = (B <= 27) ? (B + 1) / 2 : 8;
#pragma unroll kUnroll
  for (int c = 0; c < B; c += 2) {
    const auto xx = *reinterpret_cast<const typename SymNum<T>::SX2*>(x + c);
    acc.fma(sym_val(m[c <= r ? row + c : c * (c + 1) / 2 + r]), sx_first(xx));
    if (B % 2 == 0 || c + 1 < B)
      acc.fma(sym_val(m[c + 1 <= r ? row + c + 1 : (c + 1) * (c + 2) / 2 + r]), sx_second(xx));
  }
}

enum { SYM_SPMV = 0, SYM_CHEB = 1, SYM_RESTRICT = 2 };
// Stored entry and sum of the blocks that follow a product: block inverses (float64: fixed
// point), transfer blocks (T)
template <typename T, typename TD, int OP>
using SymExt = typename std::conditional<OP != SYM_CHEB, T,
    typename std::conditional<std::is_same<T, double>::value, int2, TD>::type>::type;
template <typename T, int OP>
using SymExtAcc = typename std::conditional<OP == SYM_CHEB, typename SymNum<T>::Acc, PlAcc<T>>::type;

// A vector as the kernels read it: T = double: fixed point, X[unit B + i] and one
// exponent per element (the largest biased exponent of its scaled x); T = float: the
// vector itself.
// One exponent per element (and one per row: the largest of the row's blocks) rounds a
// row that sees nothing but an element's small values, as a neighbour's row sees only
// its face, to 2^-57 of the large ones. So an element with a face whose largest value
// is below 2^-kFxSpan of the element's is kept as doubles (E + kFxWide; X the bits
// of x 2^{s_i} over its power of two), as is one with a NaN or an infinity, and its
// blocks are multiplied in float64 (sym_wide_row). Every row that an element takes
// part in then holds a term of 2^-kFxSpan of its largest value, and rounds to about
// 2^-50 of (|A| |x|)_i, for vectors of any range. (A unit vector over noise of 1e-12: rows
// beside the unit off by 6e-5 of (|A| |x|)_i before.) Of random vectors and CG
// directions (from stimuli and fronts) at most 0.4% of the elements were kept as
// doubles, mostly none; 4% of a first direction from a front on the thin shell. Cost on
// the 40^3 Q2 product (270 us): 1% of the elements 285 us, every one 1,590 us.
template <typename T> struct SymVec {
  const typename SymNum<T>::SX* X;
  const int* E;
};

// Shared memory of a block of k_sym. Two stages (of everything an element's step
// copies), so that one element's copies are in flight while the other one is
// multiplied: GB300 needs about 100 KB in flight per SM to reach its HBM rate. Then
// the face rows' partial sums, the groups' sums, exponents. G groups of B threads
// share an element: group 0 takes the diagonal block, the others two faces each;
// their sums are added at the end.
template <typename T, typename TD, int B, int OP, int KIND>
struct SymSmem {
  using S = SymShape<B>;
  using ST = typename SymNum<T>::ST;
  using SX = typename SymNum<T>::SX;
  using Sum = typename SymNum<T>::Acc::Sum;
  using SD = SymExt<T, TD, OP>;
  using XAcc = SymExtAcc<T, OP>;
  using L = SymLay<ST, B>;
  static constexpr bool kFx = std::is_same<T, double>::value;
  static constexpr bool kProduct = !(OP == SYM_CHEB && KIND == 0);
  static constexpr int G = kProduct ? 4 : 1;
  // with an operator product, the block inverse or P^T is read from memory, column
  // by column and a group's columns per thread, instead of shared memory, where only
  // one stage would fit: adjoint step of the 18^3 Q3 cube 21.3 -> 19.5 ms
  static constexpr bool kExtMem = kProduct && OP != SYM_SPMV;
  static constexpr int KE = kProduct ? L::KD + S::NFACE * L::KB : 0;
  static constexpr int KX = (OP == SYM_CHEB && !kProduct) ? SymLay<SD, B>::KD : 0;
  static constexpr int KXM = SymLay<SD, B>::KP, CPG = B / G;   // block entries in memory, columns per group
  static constexpr int NX = kProduct ? 1 + S::NFACE : 0;
  static constexpr int NTH = round_to(B * G, 32);
  static constexpr size_t kBlk = (size_t)KE * sizeof(ST);
  static constexpr size_t kExt = (size_t)KX * sizeof(SD);
  static constexpr size_t kXs = round_to(NX * S::BX * (int)sizeof(SX), 16);
  static constexpr size_t kEx = kFx ? round_to(NX * 4, 16) : 0;
  static constexpr size_t kStage = kBlk + kExt + kXs + kEx;
  static constexpr size_t kPart = kProduct ? round_to(S::NFACE * B * (int)sizeof(Sum), 16) : 0;
  static constexpr size_t kRed = round_to((G - 1) * B * (int)sizeof(Sum), 16);
  static constexpr size_t kTs = (OP == SYM_SPMV) ? 0 : round_to(S::BX * (int)sizeof(SX), 16);
  static constexpr size_t kRest = kPart + kRed + kTs + round_to((1 + 2 * (1 + S::NFACE)) * (int)sizeof(int), 16);
  static constexpr int kStages = (2 * kStage + kRest <= 225 * 1024) ? 2 : 1;
  static constexpr size_t bytes = kStages * kStage + kRest;
};

// y plus row r's products with those of its blocks whose element is kept as doubles
// (SymVec), in float64 over the stored entries. The integer sums that the kernels
// form of such blocks carry exponents so low that they are shifted out.
template <int B>
__device__ __forceinline__ double sym_wide_row(const SymView<double, B>& A, int64_t unit, int r, double y, const int2* X,
                                               const int* E) {
  using S = SymShape<B>;
  using L = SymLay<int2, B>;
  using FI = FaceIdx<S::D, S::N>;
  auto term = [](int2 a, int2 x) {
    return (double)(((long long)a.y << FX_P) + a.x) * __hiloint2double(x.y, x.x);
  };
  const int q = A.sc[(size_t)unit * B + r] - A.kA - kFxWide - kFxRaw;
  if (E[unit] < kFxWide / 2) {
    const int2 *m = A.diag + (size_t)unit * L::KD, *x = X + (size_t)unit * B;
    double s = 0.0;
#pragma unroll 4
    for (int c = 0; c < B; ++c) s += term(m[c <= r ? r * (r + 1) / 2 + c : c * (c + 1) / 2 + r], x[c]);
    y += scalbn(s, q + E[unit]);
  }
  for (int f = 0; f < S::NFACE; ++f) {
    const int2 nf = A.info[unit * S::NFACE + f];
    if (nf.x < 0 || E[nf.x] >= kFxWide / 2) continue;
    const int fn = A.code[unit * S::NFACE + f];
    const bool tr = nf.x < unit;                      // the block is the neighbour's: row of K^T
    bool on;
    const int pos = face_first<B>(f, r, on);
    const int2 *F = A.face + (size_t)nf.y * L::KB, *Gb = F + S::NF * S::LDF, *x = X + (size_t)nf.x * B;
    const int2* p = tr ? (on ? F + pos * S::LDF : Gb + (pos - S::NF) * S::LDG) : F + pos;
    double s = 0.0;
#pragma unroll 3
    for (int t = 0; t < S::NF; ++t) s += term(p[tr ? t : t * S::LDF], x[FI::face(fn, t)]);
    if (on) {
      p = tr ? F + pos * S::LDF + S::NF : Gb + pos;
#pragma unroll 3
      for (int t = 0; t < S::BO; ++t) s += term(p[tr ? t : t * S::LDG], x[FI::off(fn, t)]);
    }
    y += scalbn(s, q + E[nf.x]);
  }
  return y;
}
// The same as a call: k_sym is faster with it (V-cycle of the 18^3 Q3 cube 2,288 inline,
// 2,272 us), and the products of k_symw (40^3 Q2 272, 266 us); its smoothing steps are
// faster inline (V-cycle on 250^2 Q2 556 with the call, 542 us).
template <int B>
__device__ __noinline__ double sym_wide_row_call(SymView<double, B> A, int64_t unit, int r, double y, const int2* X,
                                                 const int* E) {
  return sym_wide_row<B>(A, unit, r, y, X, E);
}

// An element's vector copy (SymVec): E the largest scaled exponent of its values, mn
// the least of its faces' largest ones.
__device__ __forceinline__ bool fx_raw(int E, int mn) { return E == kFxInf || mn < E - kFxSpan; }
static __device__ __noinline__ int2 fx_double(double v, int q) {
  const double w = scalbn(v, q);
  return make_int2(__double2loint(w), __double2hiint(w));
}
__device__ __forceinline__ int2 fx_copy(double v, int t, int E, bool raw) {
  return raw ? fx_double(v, t + kFxRaw - E) : fx_split(v, E - t);
}
template <int B>
__device__ __forceinline__ bool on_face(int f, int r) {
  bool on;
  face_first<B>(f, r, on);
  return on;
}
// lanes (r) of the DoFs of each face, B <= 32
template <int B>
struct FaceLanes {
  unsigned v[6] = {};
  constexpr FaceLanes() {
    constexpr int N = SymShape<B>::N;
    for (int f = 0; f < SymShape<B>::NFACE; ++f)
      for (int r = 0; r < B; ++r) {
        const int i = f < 2 ? r % N : (f < 4 ? r / N % N : r / (N * N));
        if (i == (f & 1) * (N - 1)) v[f] |= 1u << (r & 31);
      }
  }
};

// Fixed-point copy of one value per thread, a block of threads holding whole
// elements (thread = slot B + r): X and E of SymVec.
template <int B, int U>
struct FxShared {
  int mx[U], mn[U], ex[U * B];
};
template <int B, int U>
__device__ __forceinline__ void fx_store(double v, bool active, int slot, int64_t unit, int r, const int16_t* sc, int2* X,
                                         int* E, FxShared<B, U>& sh) {
  using S = SymShape<B>;
  using FI = FaceIdx<S::D, S::N>;
  if (threadIdx.x < U) {
    sh.mx[threadIdx.x] = kFxNone;
    sh.mn[threadIdx.x] = kFxInf;
  }
  const size_t o = (size_t)unit * B + r;
  const int t = active ? sc[o] : 0;
  const int e = fx_exp(v, t);
  if (active) sh.ex[slot * B + r] = e;
  __syncthreads();
  if (active) {
    if (r < S::NFACE) {                               // face r's
      int m = kFxNone;
#pragma unroll
      for (int j = 0; j < S::NF; ++j) m = max(m, sh.ex[slot * B + FI::face(r, j)]);
      atomicMax(sh.mx + slot, m);
      atomicMin(sh.mn + slot, m);
    }
    bool inner = true;
#pragma unroll
    for (int f = 0; f < S::NFACE; ++f) inner = inner && !on_face<B>(f, r);
    if (inner) atomicMax(sh.mx + slot, e);
  }
  __syncthreads();
  if (active) {
    const int em = sh.mx[slot];
    const bool raw = fx_raw(em, sh.mn[slot]);
    X[o] = fx_copy(v, t, em, raw);
    if (r == 0) E[unit] = raw ? em + kFxWide : em;
  }
}

// One level-0 step, y = A0 x inside.
//   SYM_SPMV, KIND 0: out = y; 1: out = rhs - y; 2: out = y and per-block partials of (x, y)
//   SYM_CHEB, KIND as in k_cheb: Chebyshev step with the block inverses `ext`;
//     float64: also writes the new iterate's fixed-point copy (Xo, Eo)
//   SYM_RESTRICT: out = P^T (rhs - y) with the transposed transfer blocks `ext`
// (ext: column by column, LDP apart; KIND 0 of SYM_CHEB: packed triangles, which
// without a product leave room for two stages: 64 DoFs, 24^3, 108 -> 22 us)
// x: the vector itself (own values); xv: what the products read. The blocks of
// a launch loop over the elements, so that the elements in flight are
// neighbours and share face blocks through the L2.
// A face costs a row NF products with the neighbour's face DoFs, and its NF face
// rows BO more; those are dealt to all B threads of the element (B / NF partial
// sums per face row), which keeps every lane busy.
template <typename T, typename TD, int B, int OP, int KIND>
static __global__ void __launch_bounds__(SymSmem<T, TD, B, OP, KIND>::NTH)
    k_sym(SymView<T, B> A, SymBlk<typename SymSmem<T, TD, B, OP, KIND>::SD> ext, SymVec<T> xv,
          const T* __restrict__ rhs, const T* __restrict__ x, T* __restrict__ out, T* __restrict__ d, int2* Xo, int* Eo,
          T c1, T c2, double* partials, CGState* st) {
  using M = SymSmem<T, TD, B, OP, KIND>;
  using S = SymShape<B>;
  using ST = typename M::ST;
  using SD = typename M::SD;
  using SX = typename M::SX;
  using Sum = typename M::Sum;
  using Acc = typename SymNum<T>::Acc;
  using XAcc = typename M::XAcc;
  using XSum = typename XAcc::Sum;
  using L = typename M::L;
  constexpr bool kFxExt = M::kFx && OP == SYM_CHEB;   // the block inverses are in fixed point
  constexpr int G = M::G, NFACE = S::NFACE, BX = S::BX, NF = S::NF, BO = S::BO, N = S::N;
  constexpr bool kFx = M::kFx;
  constexpr int kShare = BO / N;                      // off-face terms of a face row per thread
  constexpr int FPG = (G == 1) ? NFACE : (NFACE + G - 2) / (G - 1);   // faces per group
  static_assert(B == 64, "two warps hold an element's rows");
  if (st && st->done) return;
  extern __shared__ __align__(16) unsigned char sym_sm[];
  Sum* spart = reinterpret_cast<Sum*>(sym_sm + M::kStages * M::kStage);
  Sum* sred = reinterpret_cast<Sum*>(sym_sm + M::kStages * M::kStage + M::kPart);
  SX* sts = reinterpret_cast<SX*>(sym_sm + M::kStages * M::kStage + M::kPart + M::kRed);
  int* smax = reinterpret_cast<int*>(sym_sm + M::kStages * M::kStage + M::kPart + M::kRed + M::kTs);

  const int tid = threadIdx.x;
  const int g = tid / B, r = tid - g * B;
  double part = 0.0;
  // the group's k-th face
  auto face_of = [&](int k) { return G == 1 ? k : g - 1 + k * (G - 1); };

  int2 info[FPG];
  int8_t code[FPG];
  auto load_info = [&](int64_t unit) {
    if constexpr (M::kProduct) {
#pragma unroll
      for (int k = 0; k < FPG; ++k) {
        info[k] = make_int2(-1, 0);
        code[k] = 0;
        if ((G == 1 || g > 0) && face_of(k) < NFACE) {
          info[k] = A.info[unit * NFACE + face_of(k)];
          code[k] = A.code[unit * NFACE + face_of(k)];
        }
      }
    }
  };
  // copies of an element into stage `sg` (its face info has been loaded)
  auto issue = [&](int64_t unit, int sg) {
    unsigned char* base = sym_sm + sg * M::kStage;
    ST* eb = reinterpret_cast<ST*>(base);
    SX* ex = reinterpret_cast<SX*>(base + M::kBlk + M::kExt);
    int* ee = reinterpret_cast<int*>(base + M::kBlk + M::kExt + M::kXs);
    if constexpr (M::KX > 0) {
      constexpr int QD = 16 / (int)sizeof(SD);
      const SD* src = ext.v + (size_t)unit * M::KX;
      SD* dst = reinterpret_cast<SD*>(base + M::kBlk);
      for (int p = r + B * g; p < M::KX / QD; p += B * G) cp_async16(dst + p * QD, src + p * QD);
    }
    if constexpr (M::kProduct) {
      if (g == 0) {
        const ST* src = A.diag + (size_t)unit * L::KD;
#pragma unroll 4
        for (int p = r; p < L::KD / L::Q; p += B) cp_async16(eb + p * L::Q, src + p * L::Q);
        cp_async_x(ex + r, xv.X + (size_t)unit * B + r);
        if (kFx && r == 0) cp_async4(ee, xv.E + unit);
      }
#pragma unroll
      for (int k = 0; k < FPG; ++k) {
        const int f = face_of(k);
        if (info[k].x < 0) {
          if (kFx && r == 0 && (G == 1 || g > 0)) ee[f + 1] = kFxNone;
          continue;
        }
        const ST* src = A.face + (size_t)info[k].y * L::KB;
        ST* dst = eb + L::KD + f * L::KB;
#pragma unroll 4
        for (int p = r; p < L::KB / L::Q; p += B) cp_async16(dst + p * L::Q, src + p * L::Q);
        bool on;
        int pos = face_first<B>(code[k], r, on);
        if (!on) pos += S::XO - NF;
        cp_async_x(ex + (f + 1) * BX + pos, xv.X + (size_t)info[k].x * B + r);
        if (kFx && r == 0) cp_async4(ee + f + 1, xv.E + info[k].x);
      }
    }
  };

  int64_t unit = blockIdx.x;
  unsigned mask = 0, next_mask = 0;                   // the group's faces with a neighbour (and its orientation)
  auto face_mask = [&](int64_t u) {
    unsigned m = 0;
    if constexpr (M::kProduct) {
#pragma unroll
      for (int k = 0; k < FPG; ++k)
        if (info[k].x >= 0) m |= (info[k].x < u ? 3u : 1u) << (2 * k);
    }
    return m;
  };
  int sg = 0;
  if (unit < A.n) {
    load_info(unit);
    issue(unit, 0);
    mask = face_mask(unit);
    if (M::kStages == 2 && unit + gridDim.x < A.n) load_info(unit + gridDim.x);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (; unit < A.n; unit += gridDim.x) {
    const bool lead = g == 0;
    const size_t o = (size_t)unit * B + r;
    const int64_t next = unit + gridDim.x;
    if constexpr (M::kStages == 2) {
      if (next < A.n) {
        issue(next, sg ^ 1);
        next_mask = face_mask(next);
        if (next + gridDim.x < A.n) load_info(next + gridDim.x);
      }
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    if (OP != SYM_SPMV && tid == 0) smax[0] = kFxNone;
    __syncthreads();
    unsigned char* base = sym_sm + sg * M::kStage;
    const ST* eb = reinterpret_cast<ST*>(base);
    const SD* sext = reinterpret_cast<SD*>(base + M::kBlk);
    const SX* ex = reinterpret_cast<SX*>(base + M::kBlk + M::kExt);
    const int* ee = reinterpret_cast<int*>(base + M::kBlk + M::kExt + M::kXs);
    T own = T(0), rh = T(0), dv = T(0);               // loaded ahead of their use
    int ti = 0, ui = 0;                               // scale exponents of the row and of its block inverse
    SD ev[M::kExtMem ? M::CPG : 1];
    if constexpr (M::kExtMem) {
      const SD* e = ext.v + (size_t)unit * M::KXM + (size_t)(g * M::CPG) * S::LDP + r;
#pragma unroll
      for (int c = 0; c < M::CPG; ++c) ev[c] = e[c * S::LDP];
    }
    if (lead) {
      if (M::kProduct && (KIND == 2 || OP == SYM_CHEB)) own = x[o];
      if (!(OP == SYM_SPMV && KIND != 1)) rh = rhs[o];
      if (OP == SYM_CHEB && KIND == 2) dv = d[o];
      if (kFx) ti = A.sc[o];
      if (kFxExt) ui = ext.s[o];
    }

    // ---- y = (A0 x)_r
    T y = T(0);
    int E = kFxNone;
    if constexpr (M::kProduct) {
      Sum sum = Sum(0);
      int lo = kFxNone;                               // largest (E) and least exponent of the blocks
      if constexpr (kFx) {
        E = lo = ee[0];
#pragma unroll
        for (int k = 1; k <= NFACE; ++k) {
          E = max(E, ee[k]);
          lo = min(lo, ee[k]);
        }
      }
      if (g == 0) {
        Acc acc;
        sym_tri<T, B>(eb, r, ex, acc);
        sum = sum_shift(acc.sum(), kFx ? E - ee[0] : 0);
      }
      Sum* pp = spart + r;
      constexpr int kFaceUnroll = (S::D == 2) ? FPG : 1;
#pragma unroll kFaceUnroll
      for (int k = 0; k < FPG; ++k) {
        if (G > 1 && g == 0) break;
        const int f = face_of(k);
        const unsigned m = mask >> (2 * k);
        if (!(m & 1)) {
          pp[f * B] = Sum(0);
          continue;
        }
        const bool tr = m & 2;                        // the block is the neighbour's: row of K^T
        bool on;
        const int pos = face_first<B>(f, r, on);
        const ST* F = eb + L::KD + f * L::KB;
        const ST* Gb = F + NF * S::LDF;
        const SX* xf = ex + (f + 1) * BX;
        const int sh = kFx ? E - ee[f + 1] : 0;
        Acc acc;
        sym_dot<T, NF>(tr ? (on ? F + pos * S::LDF : Gb + (pos - NF) * S::LDG) : F + pos, tr ? 1 : S::LDF, xf, acc);
        sum += sum_shift(acc.sum(), sh);
        // this thread's share of face row j's off-face terms
        const int j = r % NF, a0 = r / NF * kShare;
        Acc pa;
        sym_dot_any<T, kShare>(tr ? F + j * S::LDF + NF + a0 : Gb + a0 * S::LDG + j, tr ? 1 : S::LDG, xf + S::XO + a0, pa);
        pp[f * B] = sum_shift(pa.sum(), sh);
      }
      if (G > 1 && g > 0) sred[(g - 1) * B + r] = sum;
      __syncthreads();
      if (lead) {
#pragma unroll
        for (int k = 0; k < G - 1; ++k) sum += sred[k * B + r];
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
          bool on;
          const int j = face_first<B>(f, r, on);
          if (on) {
#pragma unroll
            for (int a = 0; a < N; ++a) sum += spart[f * B + a * NF + j];
          }
        }
        if constexpr (kFx) {
          y = fx_scale(sum, ti - A.kA + E + kFxBias);
          if (lo < kFxWide / 2) y = sym_wide_row_call<B>(A, unit, r, E < kFxWide / 2 ? 0.0 : y, xv.X, xv.E);
        } else {
          y = sum;
        }
      }
    }

    if constexpr (OP == SYM_SPMV) {
      if (lead) {
        out[o] = (KIND == 1) ? rh - y : y;
        if (KIND == 2) part += (double)own * (double)y;
      }
    } else {
      // ---- the element's residual t, then its block inverse or P^T
      const T t = rh - y;
      int Et = 0;
      if constexpr (kFxExt) {
        if (lead) atomicMax(smax, fx_exp(t, ui));
        __syncthreads();
        if (lead) Et = smax[0];
      }
      using TS = typename std::conditional<OP == SYM_CHEB, SX, T>::type;
      TS* ts = reinterpret_cast<TS*>(sts);
      XSum* xred = reinterpret_cast<XSum*>(sred);
      if (lead) {
        if constexpr (kFxExt) ts[r] = fx_split(t, Et - ui);
        else ts[r] = t;
      }
      __syncthreads();
      T res = T(0);
      XSum es = XSum(0);
      XAcc acc;
      if constexpr (M::kExtMem) {
#pragma unroll
        for (int c = 0; c < M::CPG; ++c) acc.fma(sym_val(ev[c]), ts[g * M::CPG + c]);
      } else {
        sym_tri<T, B>(sext, r, ts, acc);
      }
      es = acc.sum();
      if (G > 1 && g > 0) xred[(g - 1) * B + r] = es;
      if (G > 1) __syncthreads();
      if (lead) {
#pragma unroll
        for (int k = 0; k < G - 1; ++k) es += xred[k * B + r];
        T sv;
        if constexpr (kFxExt) sv = Et == kFxInf ? nan("") : fx_scale(es, ui + Et + kFxBias - ext.k[unit]);
        else sv = es;
        if constexpr (OP == SYM_RESTRICT) {
          out[o] = sv;
        } else {
          const T dn = (KIND == 2) ? c1 * dv + c2 * sv : c2 * sv;
          d[o] = dn;
          res = M::kProduct ? own + dn : dn;
          out[o] = res;
        }
      }
      if constexpr (kFx && OP == SYM_CHEB) {
        // largest exponents of the two warps that hold the rows: all values, face by face
        int* wmax = smax + 1;
        if (lead) {
          const int e = fx_exp(res, ti);
#pragma unroll
          for (int f = -1; f < NFACE; ++f) {
            const int m = __reduce_max_sync(0xffffffffu, f < 0 || on_face<B>(f, r) ? e : kFxNone);
            if ((tid & 31) == 0) wmax[(tid >> 5) * (1 + NFACE) + f + 1] = m;
          }
        }
        __syncthreads();
        if (lead) {
          int mn = kFxInf;
#pragma unroll
          for (int f = 0; f < NFACE; ++f) {
            const int m = max(wmax[f + 1], wmax[1 + NFACE + f + 1]);
            mn = min(mn, m);
          }
          const int em = max(wmax[0], wmax[1 + NFACE]);
          const bool raw = fx_raw(em, mn);
          Xo[o] = fx_copy(res, ti, em, raw);
          if (r == 0) Eo[unit] = raw ? em + kFxWide : em;
        }
      }
    }
    __syncthreads();                                  // the stage and the sums are free again
    if constexpr (M::kStages == 2) {
      sg ^= 1;
      mask = next_mask;
    } else if (next < A.n) {
      load_info(next);
      issue(next, 0);
      mask = face_mask(next);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if constexpr (OP == SYM_SPMV && KIND == 2) {
    const double s = block_sum<M::NTH>(part);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------- streaming form (B <= 32)
// One warp per 32 / B elements, one lane per row; each warp streams its blocks
// (diagonal, faces, Dinv) through a private ring of NS slots in shared memory,
// so that NS - 1 blocks are always in flight and no warp waits for another.
// Shared memory holds kBlocks x NWARP rings per SM; more slots or warps did not
// fit, fewer left HBM idle.
template <typename T, typename TD, int B, int OP, int KIND>
struct SymRing {
  using S = SymShape<B>;
  using ST = typename SymNum<T>::ST;
  using SX = typename SymNum<T>::SX;
  using Sum = typename SymNum<T>::Acc::Sum;
  using SD = SymExt<T, TD, OP>;
  using XAcc = SymExtAcc<T, OP>;
  using L = SymLay<ST, B>;
  static constexpr bool kFx = std::is_same<T, double>::value;
  static constexpr bool kProduct = !(OP == SYM_CHEB && KIND == 0);
  static constexpr int EPW = 32 / B;
  static constexpr int K0 = kProduct ? 0 : 1 + S::NFACE;                  // first block of an element
  static constexpr int K1 = 1 + S::NFACE + (OP == SYM_CHEB ? 1 : 0);      // one past the last
  static constexpr int NS = kProduct ? (B == 27 ? 4 : 5) : 2;             // at most K1 - K0 + 1
  static constexpr int KM = L::KD > L::KB ? L::KD : L::KB;                // entries of a slot and element
  static constexpr size_t kSlot = round_to(EPW * (KM * (int)sizeof(ST) + S::BX * (int)sizeof(SX)) + (kFx ? EPW * 4 : 0), 16);
  static constexpr size_t kWarp = NS * kSlot + round_to(EPW * S::BX * (int)sizeof(Sum), 16);
  static constexpr int NWARP = 5, NTH = NWARP * 32, kBlocks = (B == 27) ? 3 : 4;   // warps, blocks per SM
  static constexpr size_t bytes = NWARP * kWarp;
};

template <typename T, typename TD, int B, int OP, int KIND>
static __global__ void __launch_bounds__(SymRing<T, TD, B, OP, KIND>::NTH, SymRing<T, TD, B, OP, KIND>::kBlocks)
    k_symw(SymView<T, B> A, SymBlk<typename SymRing<T, TD, B, OP, KIND>::SD> ext, SymVec<T> xv,
           const T* __restrict__ rhs, const T* __restrict__ x, T* __restrict__ out, T* __restrict__ d, int2* Xo, int* Eo,
           T c1, T c2, double* partials, CGState* st) {
  using M = SymRing<T, TD, B, OP, KIND>;
  using S = SymShape<B>;
  using ST = typename M::ST;
  using SD = typename M::SD;
  using SX = typename M::SX;
  using Sum = typename M::Sum;
  using Acc = typename SymNum<T>::Acc;
  using XAcc = typename M::XAcc;
  using L = typename M::L;
  constexpr bool kFxExt = M::kFx && OP == SYM_CHEB;   // the block inverses are in fixed point
  constexpr int EPW = M::EPW, NFACE = S::NFACE, BX = S::BX, NF = S::NF, BO = S::BO, N = S::N, NS = M::NS;
  constexpr int K0 = M::K0, K1 = M::K1, NB = K1 - K0;
  static_assert(NS - 1 <= NB, "the first copies are one element's");
  constexpr bool kFx = M::kFx;
  constexpr int kShare = BO / N;                      // off-face terms of a face row per lane
  if (st && st->done) return;
  extern __shared__ __align__(16) unsigned char sym_sm[];
  const int lane = threadIdx.x & 31;
  const int sub = lane / B, r = lane - sub * B;
  const bool in = sub < EPW;
  unsigned char* wsm = sym_sm + (threadIdx.x >> 5) * M::kWarp;
  Sum* part = reinterpret_cast<Sum*>(wsm + NS * M::kSlot) + sub * BX;
  auto slot_blk = [&](int s) { return reinterpret_cast<ST*>(wsm + s * M::kSlot) + sub * M::KM; };
  auto slot_x = [&](int s) { return reinterpret_cast<SX*>(wsm + s * M::kSlot + EPW * M::KM * sizeof(ST)) + sub * BX; };
  auto slot_e = [&](int s) {
    return reinterpret_cast<int*>(wsm + s * M::kSlot + EPW * (M::KM * sizeof(ST) + BX * sizeof(SX))) + sub;
  };
  const int64_t ntiles = (A.n + EPW - 1) / EPW;
  const int64_t gw = ((int64_t)blockIdx.x * M::NTH + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * M::NTH) >> 5;
  // lanes 0 .. 2d-1 of an element hold the neighbour and face block of its faces
  auto load_info = [&](int64_t tile, int2& in_, int& code_) {
    in_ = make_int2(-1, 0);
    code_ = 0;
    const int64_t unit = tile * EPW + sub;
    if (M::kProduct && in && unit < A.n && r < NFACE) {
      in_ = A.info[unit * NFACE + r];
      code_ = A.code[unit * NFACE + r];
    }
  };
  auto issue = [&](int64_t tile, int k, int2 ti, int tc, int s) {
    const int64_t unit = tile * EPW + sub;
    ST* dst = slot_blk(s);
    if (k == 0) {
      if (in && unit < A.n) {
        const ST* src = A.diag + (size_t)unit * L::KD;
#pragma unroll
        for (int p = 0; p < (L::KD / L::Q + B - 1) / B; ++p)
          if (p * B + r < L::KD / L::Q) cp_async16(dst + (p * B + r) * L::Q, src + (p * B + r) * L::Q);
        cp_async_x(slot_x(s) + r, xv.X + (size_t)unit * B + r);
        if (kFx && r == 0) cp_async4(slot_e(s), xv.E + unit);
      }
    } else if (k <= NFACE) {
      const int from = in ? sub * B + k - 1 : 0;
      const int nb = __shfl_sync(0xffffffffu, ti.x, from), id = __shfl_sync(0xffffffffu, ti.y, from);
      const int fn = __shfl_sync(0xffffffffu, tc, from);
      if (in && unit < A.n && nb >= 0) {
        const ST* src = A.face + (size_t)id * L::KB;
#pragma unroll
        for (int p = 0; p < (L::KB / L::Q + B - 1) / B; ++p)
          if (p * B + r < L::KB / L::Q) cp_async16(dst + (p * B + r) * L::Q, src + (p * B + r) * L::Q);
        bool on;
        int pos = face_first<B>(fn, r, on);
        if (!on) pos += S::XO - NF;
        cp_async_x(slot_x(s) + pos, xv.X + (size_t)nb * B + r);
        if (kFx && r == 0) cp_async4(slot_e(s), xv.E + nb);
      }
    } else if constexpr (OP == SYM_CHEB) {
      if (in && unit < A.n) {
        constexpr int KX = SymLay<SD, B>::KD, QD = 16 / (int)sizeof(SD);
        const SD* src = ext.v + (size_t)unit * KX;
        SD* dd = reinterpret_cast<SD*>(dst);
#pragma unroll
        for (int p = 0; p < (KX / QD + B - 1) / B; ++p)
          if (p * B + r < KX / QD) cp_async16(dd + (p * B + r) * QD, src + (p * B + r) * QD);
      }
    }
  };

  int2 ic, in1, in2;
  int cc, cn1, cn2;
  load_info(gw, ic, cc);
  load_info(gw + nw, in1, cn1);
  int slot = 0;
#pragma unroll
  for (int j = 0; j < NS - 1; ++j) {
    if (gw < ntiles) issue(gw, K0 + j, ic, cc, j);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  double dot = 0.0;
  const unsigned emask = (B == 27) ? 0x07ffffffu : (((1u << (B & 31)) - 1u) << (in ? sub * B : 0));
  for (int64_t tile = gw; tile < ntiles; tile += nw) {
    const int64_t unit = tile * EPW + sub;
    const bool active = in && unit < A.n;
    const size_t o = (size_t)unit * B + r;
    load_info(tile + 2 * nw, in2, cn2);
    T own = T(0), rh = T(0), dv = T(0);
    int ti = 0, ui = 0;                               // scale exponents of the row and of its block inverse
    if (active) {
      if (M::kProduct && (KIND == 2 || OP == SYM_CHEB)) own = x[o];
      if (!(OP == SYM_SPMV && KIND != 1)) rh = rhs[o];
      if (OP == SYM_CHEB && KIND == 2) dv = d[o];
      if (kFx) ti = A.sc[o];
      if (kFxExt) ui = ext.s[o];
    }
    Sum sum = Sum(0);
    int E = kFxNone, lo = kFxNone;                    // largest and least exponent of the blocks
    T res = T(0);
    constexpr int kBlkUnroll = (S::D == 2) ? NB : 1;
#pragma unroll kBlkUnroll
    for (int k = K0; k < K1; ++k) {
      {
        // keep NS - 1 blocks in flight
        const int ka = k + NS - 1, sa = slot == 0 ? NS - 1 : slot - 1;
        if (ka < K1) issue(tile, ka, ic, cc, sa);
        else if (tile + nw < ntiles) issue(tile + nw, ka - NB, in1, cn1, sa);
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group %0;" ::"n"(NS - 1) : "memory");
        __syncwarp();
      }
      const ST* blk = slot_blk(slot);
      const SX* xs = slot_x(slot);
      if (k == 0) {
        if (active) {
          Acc acc;
          sym_tri<T, B>(blk, r, xs, acc);
          sum = acc.sum();
          if constexpr (kFx) E = lo = *slot_e(slot);
        }
      } else if (k <= NFACE) {
        const int f = k - 1;
        const int nb = __shfl_sync(0xffffffffu, ic.x, in ? sub * B + f : 0);
        const bool have = active && nb >= 0;
        bool on = false;
        int pos = 0;
        Sum s = Sum(0);
        if (have) {
          pos = face_first<B>(f, r, on);
          const ST* F = blk;
          const ST* Gb = F + NF * S::LDF;
          const bool tr = nb < unit;                  // the block is the neighbour's: row of K^T
          Acc acc;
          sym_dot<T, NF>(tr ? (on ? F + pos * S::LDF : Gb + (pos - NF) * S::LDG) : F + pos, tr ? 1 : S::LDF, xs, acc);
          s = acc.sum();
          // this lane's share of face row j's off-face terms
          const int j = r % NF, a0 = r / NF * kShare;
          Acc pa;
          sym_dot_any<T, kShare>(tr ? F + j * S::LDF + NF + a0 : Gb + a0 * S::LDG + j, tr ? 1 : S::LDG, xs + S::XO + a0, pa);
          part[r] = pa.sum();
        }
        __syncwarp();
        if (have) {
          if (on) {
#pragma unroll
            for (int a = 0; a < N; ++a) s += part[a * NF + pos];
          }
          if constexpr (kFx) {
            const int e = *slot_e(slot);
            lo = min(lo, e);
            if (e > E) {
              sum = sum_shift(sum, e - E) + s;
              E = e;
            } else {
              sum += sum_shift(s, E - e);
            }
          } else {
            sum += s;
          }
        }
      }
      if (k == NFACE || !M::kProduct) {
        // ---- the row's product, and what the operation makes of it
        T y = T(0);
        if (M::kProduct && active) {
          if constexpr (kFx) {
            y = fx_scale(sum, ti - A.kA + E + kFxBias);
            const double y0 = E < kFxWide / 2 ? 0.0 : y;
            if (lo < kFxWide / 2)
              y = OP == SYM_SPMV ? sym_wide_row_call<B>(A, unit, r, y0, xv.X, xv.E) : sym_wide_row<B>(A, unit, r, y0, xv.X, xv.E);
          } else {
            y = sum;
          }
        }
        if constexpr (OP == SYM_SPMV) {
          if (active) {
            out[o] = (KIND == 1) ? rh - y : y;
            if (KIND == 2) dot += (double)own * (double)y;
          }
        } else {
          res = rh - y;                               // the residual's row
        }
      }
      if constexpr (OP != SYM_SPMV) {
        if (k == K1 - 1) {
          const T t = res;
          int Et = 0;
          using TS = typename std::conditional<OP == SYM_CHEB, SX, T>::type;
          TS* ts = reinterpret_cast<TS*>(part);
          __syncwarp();
          if (active) {
            if constexpr (kFxExt) {
              Et = __reduce_max_sync(emask, fx_exp(t, ui));
              ts[r] = fx_split(t, Et - ui);
            } else {
              ts[r] = t;
            }
          }
          __syncwarp();
          if (active) {
            XAcc acc;
            if constexpr (OP == SYM_CHEB) {
              sym_tri<T, B>(reinterpret_cast<const SD*>(blk), r, ts, acc);
            } else {
              const SD* p = ext.v + (size_t)unit * SymLay<SD, B>::KP + r;
#pragma unroll
              for (int i = 0; i < B; ++i) acc.fma(__ldcs(p + i * S::LDP), ts[i]);
            }
            T sv;
            if constexpr (kFxExt) sv = Et == kFxInf ? nan("") : fx_scale(acc.sum(), ui + Et + kFxBias - ext.k[unit]);
            else sv = acc.sum();
            if constexpr (OP == SYM_RESTRICT) {
              out[o] = sv;
            } else {
              const T dn = (KIND == 2) ? c1 * dv + c2 * sv : c2 * sv;
              d[o] = dn;
              const T xn = M::kProduct ? own + dn : dn;
              out[o] = xn;
              if constexpr (kFx) {
                const int e = fx_exp(xn, ti), em = __reduce_max_sync(emask, e);
                const unsigned big = __ballot_sync(emask, e >= em - kFxSpan) >> (sub * B);
                constexpr FaceLanes<B> kLanes;
                bool raw = em == kFxInf;
#pragma unroll
                for (int f = 0; f < NFACE; ++f) raw = raw || !(big & kLanes.v[f]);
                Xo[o] = fx_copy(xn, ti, em, raw);
                if (r == 0) Eo[unit] = raw ? em + kFxWide : em;
              }
            }
          }
        }
      }
      __syncwarp();                                   // the slot is free again
      slot = slot + 1 == NS ? 0 : slot + 1;
    }
    ic = in1;
    cc = cn1;
    in1 = in2;
    cn1 = cn2;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if constexpr (OP == SYM_SPMV && KIND == 2) {
    const double s = block_sum<M::NTH>(dot);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
  }
}

// Threads of the element-wise kernels below: U whole elements per block.
template <int B> struct SymRows {
  static constexpr int U = (B <= 64) ? 128 / B : 1, NT = round_to(U * B, 32);
};

// Level-0 prolongation x_u += P_u e_{parent(u)}, one thread per (element, row):
// a row's entries of consecutive columns lie LDP apart, so the threads of an
// element read each column contiguously, straight from HBM (no reuse). HBM bound:
// 64^3 Q2 hexahedra 132 us (121 us at the copy rate), 24^3 Q3 115 -> 33 us against
// one thread per element.
template <typename T, int B>
static __global__ void __launch_bounds__(SymRows<B>::NT)
    k_sym_prolong(SymBlk<T> P, const int32_t* __restrict__ parent, const T* __restrict__ ec,
                  T* __restrict__ x, const int16_t* __restrict__ sc, int2* Xo, int* Eo, int64_t n, const CGState* st) {
  if (st && st->done) return;
  using S = SymShape<B>;
  constexpr int KP = SymLay<T, B>::KP, U = SymRows<B>::U, BX = (B + 1) / 2 * 2;
  constexpr bool kFx = std::is_same<T, double>::value;
  __shared__ T sx[U * BX];
  __shared__ FxShared<B, U> sh;
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * U + slot;
  const bool active = slot < U && unit < n;
  if (active) sx[slot * BX + r] = ec[(size_t)parent[unit] * B + r];
  __syncthreads();
  T v = T(0);
  if (active) {
    const T* p = P.v + (size_t)unit * KP + r;
    T s = T(0);
    constexpr int kUnroll = (B <= 27) ? B : 16;
#pragma unroll kUnroll
    for (int j = 0; j < B; ++j) s += __ldcs(p + j * S::LDP) * sx[slot * BX + j];
    v = x[(size_t)unit * B + r] + s;
    x[(size_t)unit * B + r] = v;
  }
  if constexpr (kFx) fx_store<B, U>(v, active, slot, unit, r, sc, Xo, Eo, sh);
}

// x's fixed-point copy
template <int B>
static __global__ void __launch_bounds__(SymRows<B>::NT)
    k_fx(const double* __restrict__ x, int64_t n, const int16_t* __restrict__ sc, int2* __restrict__ X,
         int* __restrict__ E, const CGState* st) {
  if (st && st->done) return;
  __shared__ FxShared<B, SymRows<B>::U> sh;
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  const int64_t unit = (int64_t)blockIdx.x * SymRows<B>::U + slot;
  const bool active = slot < SymRows<B>::U && unit < n;
  fx_store<B, SymRows<B>::U>(active ? x[(size_t)unit * B + r] : 0.0, active, slot, unit, r, sc, X, E, sh);
}
// p = z + beta p (INIT: p = z), as k_pupd, with p's fixed-point copy
template <typename TZ, int B, bool INIT>
static __global__ void __launch_bounds__(SymRows<B>::NT)
    k_pupd_fx(const TZ* __restrict__ z, double* __restrict__ p, int64_t n, const double* partials, int np,
              const int16_t* __restrict__ sc, int2* __restrict__ X, int* __restrict__ E, CGState* st) {
  if (st->done) return;
  __shared__ FxShared<B, SymRows<B>::U> sh;
  const double beta = cg_beta<SymRows<B>::NT, INIT>(partials, np, st);
  const int slot = threadIdx.x / B, r = threadIdx.x - slot * B;
  for (int64_t u0 = (int64_t)blockIdx.x * SymRows<B>::U; u0 < n; u0 += (int64_t)gridDim.x * SymRows<B>::U) {
    const int64_t unit = u0 + slot;
    const bool active = slot < SymRows<B>::U && unit < n;
    const size_t o = (size_t)unit * B + r;
    double v = 0.0;
    if (active) {
      v = INIT ? to_double(z[o]) : to_double(z[o]) + beta * p[o];
      p[o] = v;
    }
    fx_store<B, SymRows<B>::U>(v, active, slot, unit, r, sc, X, E, sh);
    __syncthreads();
  }
}

}  // namespace aggmg
