// Shared device helpers: complex arithmetic and CTA-cooperative dense
// linear algebra on row-major matrices in global memory.
//
// The batched element, macro-element and patch kernels run one CTA per
// small dense problem (n up to ~1100).  The routines below are blocked
// (block size NB) with shared-memory staging of the diagonal block and of
// the operand tiles of the trailing updates.  They assume blockDim.x == 256.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace dpgmg {

// ------------------------------------------------------------- scalar ops
template <class T> struct Ops;

template <> struct Ops<double> {
  using R = double;
  __device__ __forceinline__ static double zero() { return 0.0; }
  __device__ __forceinline__ static double add(double a, double b) { return a + b; }
  __device__ __forceinline__ static double sub(double a, double b) { return a - b; }
  __device__ __forceinline__ static double mul(double a, double b) { return a * b; }
  __device__ __forceinline__ static double mulc(double a, double b) { return a * b; }   // a conj(b)
  __device__ __forceinline__ static double fma(double a, double b, double c) { return ::fma(a, b, c); }
  __device__ __forceinline__ static double fmac(double a, double b, double c) { return ::fma(a, b, c); }  // a conj(b) + c
  __device__ __forceinline__ static double fnmac(double a, double b, double c) { return ::fma(-a, b, c); } // c - a conj(b)
  __device__ __forceinline__ static double fnma(double a, double b, double c) { return ::fma(-a, b, c); }  // c - a b
  __device__ __forceinline__ static double conj(double a) { return a; }
  __device__ __forceinline__ static double re(double a) { return a; }
  __device__ __forceinline__ static double scale(double a, double s) { return a * s; }
  __device__ __forceinline__ static double from_re(double r) { return r; }
};

template <> struct Ops<float> {
  using R = float;
  __device__ __forceinline__ static float zero() { return 0.f; }
  __device__ __forceinline__ static float add(float a, float b) { return a + b; }
  __device__ __forceinline__ static float sub(float a, float b) { return a - b; }
  __device__ __forceinline__ static float mul(float a, float b) { return a * b; }
  __device__ __forceinline__ static float mulc(float a, float b) { return a * b; }
  __device__ __forceinline__ static float fma(float a, float b, float c) { return fmaf(a, b, c); }
  __device__ __forceinline__ static float fmac(float a, float b, float c) { return fmaf(a, b, c); }
  __device__ __forceinline__ static float fnmac(float a, float b, float c) { return fmaf(-a, b, c); }
  __device__ __forceinline__ static float fnma(float a, float b, float c) { return fmaf(-a, b, c); }
  __device__ __forceinline__ static float conj(float a) { return a; }
  __device__ __forceinline__ static float re(float a) { return a; }
  __device__ __forceinline__ static float scale(float a, float s) { return a * s; }
  __device__ __forceinline__ static float from_re(float r) { return r; }
};

template <class V, class S> struct CplxOps {
  using R = S;
  __device__ __forceinline__ static V mk(S r, S i) { V v; v.x = r; v.y = i; return v; }
  __device__ __forceinline__ static V zero() { return mk(S(0), S(0)); }
  __device__ __forceinline__ static V add(V a, V b) { return mk(a.x + b.x, a.y + b.y); }
  __device__ __forceinline__ static V sub(V a, V b) { return mk(a.x - b.x, a.y - b.y); }
  __device__ __forceinline__ static V mul(V a, V b) { return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
  __device__ __forceinline__ static V mulc(V a, V b) { return mk(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); }
  __device__ __forceinline__ static V fma(V a, V b, V c) {
    return mk(c.x + a.x * b.x - a.y * b.y, c.y + a.x * b.y + a.y * b.x);
  }
  __device__ __forceinline__ static V fmac(V a, V b, V c) {   // a conj(b) + c
    return mk(c.x + a.x * b.x + a.y * b.y, c.y + a.y * b.x - a.x * b.y);
  }
  __device__ __forceinline__ static V fnmac(V a, V b, V c) {  // c - a conj(b)
    return mk(c.x - a.x * b.x - a.y * b.y, c.y - a.y * b.x + a.x * b.y);
  }
  __device__ __forceinline__ static V fnma(V a, V b, V c) {   // c - a b
    return mk(c.x - a.x * b.x + a.y * b.y, c.y - a.x * b.y - a.y * b.x);
  }
  __device__ __forceinline__ static V conj(V a) { return mk(a.x, -a.y); }
  __device__ __forceinline__ static S re(V a) { return a.x; }
  __device__ __forceinline__ static V scale(V a, S s) { return mk(a.x * s, a.y * s); }
  __device__ __forceinline__ static V from_re(S r) { return mk(r, S(0)); }
};
template <> struct Ops<double2> : CplxOps<double2, double> {};
template <> struct Ops<float2> : CplxOps<float2, float> {};

// Element colours of a structured grid: (ex mod 2, ey mod 2, ez mod 2).  Two
// elements of one colour share no vertex, edge or face, so an assembly pass
// over one colour has no write conflicts; the 8 passes run in colour order,
// which fixes the order of every sum (assembly is bitwise reproducible, unlike
// FP64 atomics).
__device__ __forceinline__ int elem_color(int64_t e, int n0, int n1) {
  const int64_t ex = e % n0, ey = (e / n0) % n1, ez = e / ((int64_t)n0 * n1);
  return (int)((ex & 1) | ((ey & 1) << 1) | ((ez & 1) << 2));
}

// ------------------------------------------------------- CTA dense kernels
constexpr int CTA_THREADS = 256;
constexpr int NB = 32;          // panel width
constexpr int TL = 32;          // output tile edge of the tiled updates

// The CTAs that share one dense problem.  Team<false> is one CTA (the
// default of every routine below).  Team<true> is a thread-block cluster of
// `n` CTAs on different SMs: each routine gives every output tile to one CTA
// (`rank`), the CTAs meet at cluster barriers between dependent phases, and
// global reads of the shared matrix bypass L1 (another SM may have written
// them since this SM cached the line).  Tile ownership is by absolute tile
// coordinates, so every entry is computed by the same instructions in the
// same order as with one CTA: results are bitwise those of Team<false>.
template <bool CL>
struct Team {
  int rank = 0, n = 1;
  __device__ __forceinline__ void sync() const {
    if constexpr (CL) {
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
      __syncthreads();
    }
  }
  template <class T>
  __device__ __forceinline__ T ld(const T* p) const {
    if constexpr (CL) return __ldcg(p);
    else return *p;
  }
  // owner of lower-triangle tile (I, J), J <= I: round robin over the packed index
  __device__ __forceinline__ bool own2(int I, int J) const {
    if constexpr (CL) return (((int64_t)I * (I + 1) / 2 + J) % n) == rank;
    else return true;
  }
  // owner of column tile t: zigzag (0..n-1, n-1..0, ...), which balances the
  // triangular work of the column tiles of a triangular inverse
  __device__ __forceinline__ bool own_col(int t) const {
    if constexpr (CL) {
      const int c = t / n, q = t % n;
      return ((c & 1) ? n - 1 - q : q) == rank;
    } else {
      return true;
    }
  }
  // owner of row tile t (plain copies)
  __device__ __forceinline__ bool own_row(int t) const {
    if constexpr (CL) return t % n == rank;
    else return true;
  }
};

// ------------------------------------------------- 32 x 32 x 32 tile products
// acc[q] += sum_t A[r][t] B[t][c] for the thread's outputs r = w + 8 q, c = lane
// (warp w of 8, q < 4), the inner step of every blocked routine below.  The
// operands come in registers: a[i] = A[4 w + i][lane], with AT a[i] = A[lane][4 w + i];
// b[i] = B[4 w + i][lane], with BT b[i] = B[lane][4 w + i] (rows of the transpose).
// At, Bt: TL x NB elements of shared memory each, Z: NB x NB (FP64 types only),
// all on 16-byte boundaries.  All 256 threads call it; it synchronises before it
// writes shared memory and before it reads it.
//
// FP32 types: FMA chains in increasing t, continued from acc.
//
// FP64 types: this GPU's FP64 pipe runs 1.7 FMAs per clock and SM, its integer
// pipe 59 32 x 32 -> 64-bit multiply-adds.  A row of A and a column of B are
// taken as fixed-point numbers with the exponent of their largest entry, 82
// bits each in limbs of 26, 28 and 28 bits, and the products of limbs down to
// 2^-56 of the largest (six of nine) are summed exactly in three 64-bit sums:
// |hi| <= 2^26, |mid|, |lo| <= 2^27, so the 64 products of a complex chunk stay
// below 2^62.  The sum is rounded once per chunk.
//
// Error: absolute, below 2^-74 max_t |A[r][t]| max_t |B[t][c]|, beside the
// final rounding.  An FMA chain's error is 2^-53 times the sum of |A[r][t] B[t][c]|,
// so the result is the more exact one wherever that sum exceeds 2^-21 of the
// product of the maxima.  Scaling the rows of A or the columns of B changes
// neither.  Scaling the inner index (the columns of A against the rows of B)
// does: triangular solves with L^H and products with a solution meet it, where
// the operands carry inverse scales of the unknowns.  With BAL column t of A and
// row t of B are first shifted by powers of two (on the exponents, exact) to
// equal maxima, which takes the product of the maxima to its smallest value.
//
// With two limbs (57 bits) the element matrices were as exact as with FMA
// chains, but not the recovery blocks on boxes far from a cube: 9 times the
// error on a 1/8 x 1/100 x 1/1000 element of order 2; with three 1.0 times.
// Over p = 1 to 5, elements from 1e-4 to 125 wide and 1:125 flat ones, rows
// scaled to unit diagonal, the errors against 128-bit arithmetic are 0.3 to 1.2
// times those of FMA chains in element matrices, in the mean and at the worst
// entry.  Tiles with an infinity, a NaN or an exponent at the top of the range
// take the FP64 chain.
//
// Bound: the integer pipe.  Measured (GB300; FP64 chains, two limbs, three): element
// stage of 800 elements of order 3 with distinct wavespeeds 88, 46, 60 ms, of 64
// of order 5 1,104, 163, 211 ms; patch inversion of 8^3, p = 3, complex128 57, 27,
// 31 ms.  The inner loops are unrolled by two steps: by four the kernels spill.
__device__ __forceinline__ int fx_exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ int fx_exponent(double2 v) { return max(fx_exponent(v.x), fx_exponent(v.y)); }

constexpr int FX_NONE = -100000;   // exponent of an all-zero row, column or entry

// round(v 2^(1104 - E)) for an exponent E >= v's biased one + sft (v is taken as v 2^sft): |f| < 2^82, as
// f = l.x 2^56 + l.y 2^28 + l.z (zero and denormals give 0)
__device__ __forceinline__ int3 fx_limbs(double v, int sft, int E) {
  const int e = fx_exponent(v);
  const int sh = E - e - sft - 29;   // shift right (left when negative) of the 53-bit mantissa
  const long long m = ((long long)((__double2hiint(v) & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  if (e == 0 || sh > 60) return make_int3(0, 0, 0);
  long long g;   // f's bits from 28 on
  int lo;        // and the 28 below
  if (sh <= 0) {
    g = sh <= -28 ? m << (-28 - sh) : m >> (28 + sh);
    lo = (int)((unsigned)m << -sh) & 0xfffffff;
  } else {
    const long long f = (m + (1ll << (sh - 1))) >> sh;
    g = f >> 28;
    lo = (int)f & 0xfffffff;
  }
  if (lo >= 1 << 27) {
    lo -= 1 << 28;
    ++g;
  }
  const int hi = (int)((g + (1ll << 27)) >> 28);
  const int mid = (int)(g - ((long long)hi << 28));
  return __double2hiint(v) < 0 ? make_int3(-hi, -mid, -lo) : make_int3(hi, mid, lo);
}

// 2^(k - 56) (h 2^56 + x 2^28 + y), rounded once (on the integer pipe)
__device__ __forceinline__ double fx_value(long long h, long long x, long long y, int k) {
  constexpr long long M56 = (1ll << 56) - 1;
  long long a = y + ((x & 0xfffffff) << 28);
  h += x >> 28;
  h += a >> 56;
  a &= M56;
  const bool neg = h < 0;
  if (neg) {
    h = -h - (a != 0);
    a = (1ll << 56) - a & M56;
  }
  unsigned long long t;   // leading bit at 63
  int q;                  // value = t 2^(q + k - 56)
  if (h != 0) {
    const int z = __clzll(h);
    q = 56 - z;
    t = z <= 56 ? ((unsigned long long)h << z) | ((unsigned long long)a >> q)
                : (((unsigned long long)h << 56) | (unsigned long long)a) << (z - 56);
  } else {
    if (a == 0) return 0.0;
    const int z = __clzll(a);
    q = -z;
    t = (unsigned long long)a << z;
  }
  const long long mant = (long long)(t >> 11) + ((t >> 10) & 1);   // 2^52 .. 2^53
  const int e = q + k - 56 + 63 + 1023;
  const long long sign = neg ? (long long)0x8000000000000000ull : 0;
  if (e >= 1 && e < 2046) return __longlong_as_double(sign | (((long long)(e - 1) << 52) + mant));
  return ldexp(__longlong_as_double(sign | ((1022ll << 52) + mant)), e - 1023);
}

// limbs of an entry: high and middle ones in a tile, low ones in Z
__device__ __forceinline__ void fx_store(double* p, int* z, double v, int sft, int E) {
  const int3 f = fx_limbs(v, sft, E);
  *reinterpret_cast<int2*>(p) = make_int2(f.x, f.y);
  *z = f.z;
}
__device__ __forceinline__ void fx_store(double2* p, int2* z, double2 v, int sft, int E) {
  const int3 f = fx_limbs(v.x, sft, E), g = fx_limbs(v.y, sft, E);
  *reinterpret_cast<int4*>(p) = make_int4(f.x, f.y, g.x, g.y);
  *z = make_int2(f.z, g.z);
}

// column c of row t of Bt: swizzled with BT, so that stores along t do not conflict
template <bool BT>
__device__ __forceinline__ int fx_col(int t, int c) { return t * TL + (BT ? c ^ t : c); }

// column t of row r of At: swizzled by even numbers with AT (pairs of t stay together)
template <bool AT>
__device__ __forceinline__ int fx_row(int r, int t) { return r * NB + (AT ? t ^ (r & ~1) : t); }

// Conversions between float and double by bits: the conversion instructions run
// on the FP64 pipe (1.7 lanes a clock and SM), these on the integer pipe.

// f as a double, exact
__device__ __forceinline__ double wide(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)   // normal: the exponent's bias grows by 896
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
  return a == 0 ? __hiloint2double((int)u, 0) : (double)f;
}
__device__ __forceinline__ double wide(double f) { return f; }

// v as (high, low): high is v rounded to 24 bits, low the rest rounded to 24
__device__ __forceinline__ float2 split_float(double v) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
  if ((unsigned)(e - (1023 - 70)) > 170u) {   // zero, small, large, not finite
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
  }
  const unsigned lo = (unsigned)__double2loint(v);
  const long long m = ((long long)((hi & 0xfffff) | 0x100000) << 32) | lo;
  int t = (int)((m + (1ll << 28)) >> 29);   // 2^23 .. 2^24
  int r = (int)(m - ((long long)t << 29));  // -2^28 .. 2^28
  if (hi < 0) {
    t = -t;
    r = -r;
  }
  return make_float2((float)t * __int_as_float((e - 1046 + 127) << 23), (float)r * __int_as_float((e - 1075 + 127) << 23));
}

template <class T> struct IsFp64 { static constexpr bool v = false; };
template <> struct IsFp64<double> { static constexpr bool v = true; };
template <> struct IsFp64<double2> { static constexpr bool v = true; };
template <class T> struct FxLow { typedef int V; };
template <> struct FxLow<double2> { typedef int2 V; };

template <class T, bool BT, bool AT = false, bool BAL = false>
__device__ void tile_product(const T a[4], const T b[4], T* At, T* Bt, T* Z, int kb, T acc[4]) {
  using O = Ops<T>;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // place of a[i] and b[i]
  auto pa = [&](int i) { return AT ? fx_row<AT>(lane, 4 * w + i) : fx_row<AT>(4 * w + i, lane); };
  auto pb = [&](int i) { return BT ? fx_col<BT>(lane, 4 * w + i) : fx_col<BT>(4 * w + i, lane); };
  auto plain = [&]() {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      At[pa(i)] = a[i];
      Bt[pb(i)] = b[i];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      T s = acc[q];
#pragma unroll 8
      for (int t = 0; t < kb; ++t) s = O::fma(At[fx_row<AT>(w + 8 * q, t)], Bt[fx_col<BT>(t, lane)], s);
      acc[q] = s;
    }
  };
  if constexpr (!IsFp64<T>::v) {
    __syncthreads();   // the last product's readers are done
    plain();
  } else {
    static_assert(!(BT && BAL), "balancing reads rows of B along the lanes");
    using Low = typename FxLow<T>::V;
    Low* Za = reinterpret_cast<Low*>(Z);   // low limbs, places as At and Bt
    Low* Zb = Za + TL * NB;
    __shared__ int s_ea[TL], s_eb[TL], s_pa[8][TL], s_pb[8][TL], s_pt[8][TL], s_tb[NB];
    int ea[4], eb[4], sa[4] = {0, 0, 0, 0}, sb[4] = {0, 0, 0, 0}, top = 0;   // exponents and shifts of a[i], b[i]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      ea[i] = fx_exponent(a[i]);
      eb[i] = fx_exponent(b[i]);
      top = max(top, max(ea[i], eb[i]));
      if (ea[i] == 0) ea[i] = FX_NONE;
      if (eb[i] == 0) eb[i] = FX_NONE;
    }
    if (__syncthreads_or(top >= 0x7fe)) {   // uniform over the CTA; also: the last product's readers are done
      plain();
      return;
    }
    if constexpr (BAL) {
      auto shift = [](int u, int v) { return u == FX_NONE || v == FX_NONE ? 0 : (v - u) >> 1; };
      int tb[4];   // largest exponent of row t = 4 w + i of B
#pragma unroll
      for (int i = 0; i < 4; ++i) tb[i] = __reduce_max_sync(0xffffffffu, eb[i]);
      if constexpr (AT) {
#pragma unroll
        for (int i = 0; i < 4; ++i) sa[i] = shift(__reduce_max_sync(0xffffffffu, ea[i]), tb[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) sb[i] = -sa[i];
      } else {   // column t = lane of A runs across the warps
        s_pt[w][lane] = max(max(ea[0], ea[1]), max(ea[2], ea[3]));
        if (lane == 0)
#pragma unroll
          for (int i = 0; i < 4; ++i) s_tb[4 * w + i] = tb[i];
        __syncthreads();
        int ta = s_pt[0][lane];
#pragma unroll
        for (int u = 1; u < 8; ++u) ta = max(ta, s_pt[u][lane]);
        const int s = shift(ta, s_tb[lane]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          sa[i] = s;
          sb[i] = -__shfl_sync(0xffffffffu, s, 4 * w + i);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (ea[i] != FX_NONE) ea[i] += sa[i];
        if (eb[i] != FX_NONE) eb[i] += sb[i];
      }
    }
    int ma = FX_NONE, mb = FX_NONE;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (!AT) ea[i] = __reduce_max_sync(0xffffffffu, ea[i]);   // over the row's t
      if (BT) eb[i] = __reduce_max_sync(0xffffffffu, eb[i]);
      ma = max(ma, ea[i]);
      mb = max(mb, eb[i]);
    }
    if (AT || !BT) {   // exponents of the rows or columns that run across the warps
      if (AT) s_pa[w][lane] = ma;
      if (!BT) s_pb[w][lane] = mb;
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (AT) ma = max(ma, s_pa[u][lane]);
        if (!BT) mb = max(mb, s_pb[u][lane]);
      }
      if (AT && w == 0) s_ea[lane] = ma;
      if (!BT && w == 0) s_eb[lane] = mb;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      fx_store(&At[pa(i)], &Za[pa(i)], a[i], sa[i], AT ? ma : ea[i]);
      fx_store(&Bt[pb(i)], &Zb[pb(i)], b[i], sb[i], BT ? eb[i] : mb);
      if (lane == 0) {
        if (!AT) s_ea[4 * w + i] = ea[i];
        if (BT) s_eb[4 * w + i] = eb[i];
      }
    }
    __syncthreads();
    const int ec = s_eb[lane];
    if constexpr (sizeof(T) == sizeof(double)) {
      const int2* Af = reinterpret_cast<const int2*>(At);
      const int2* Bf = reinterpret_cast<const int2*>(Bt);
      long long h[4] = {0, 0, 0, 0}, x[4] = {0, 0, 0, 0}, y[4] = {0, 0, 0, 0};
#pragma unroll 2
      for (int t = 0; t < NB; t += 2) {
        const int2 b0 = Bf[fx_col<BT>(t, lane)], b1 = Bf[fx_col<BT>(t + 1, lane)];
        const int c0 = Zb[fx_col<BT>(t, lane)], c1 = Zb[fx_col<BT>(t + 1, lane)];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int4 u = *reinterpret_cast<const int4*>(&Af[fx_row<AT>(w + 8 * q, t)]);
          const int2 v = *reinterpret_cast<const int2*>(&Za[fx_row<AT>(w + 8 * q, t)]);
          h[q] += (long long)u.x * b0.x;
          x[q] += (long long)u.x * b0.y;
          x[q] += (long long)u.y * b0.x;
          y[q] += (long long)u.x * c0;
          y[q] += (long long)u.y * b0.y;
          y[q] += (long long)v.x * b0.x;
          h[q] += (long long)u.z * b1.x;
          x[q] += (long long)u.z * b1.y;
          x[q] += (long long)u.w * b1.x;
          y[q] += (long long)u.z * c1;
          y[q] += (long long)u.w * b1.y;
          y[q] += (long long)v.y * b1.x;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += fx_value(h[q], x[q], y[q], s_ea[w + 8 * q] + ec - 2096);
    } else {
      const int4* Af = reinterpret_cast<const int4*>(At);
      const int4* Bf = reinterpret_cast<const int4*>(Bt);
      long long rh[4] = {0, 0, 0, 0}, rx[4] = {0, 0, 0, 0}, ry[4] = {0, 0, 0, 0};
      long long ih[4] = {0, 0, 0, 0}, ix[4] = {0, 0, 0, 0}, iy[4] = {0, 0, 0, 0};
#pragma unroll 2
      for (int t = 0; t < NB; ++t) {
        const int4 v = Bf[fx_col<BT>(t, lane)];   // (re hi, re mid, im hi, im mid)
        const int2 vl = Zb[fx_col<BT>(t, lane)];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int4 u = Af[fx_row<AT>(w + 8 * q, t)];
          const int2 ul = Za[fx_row<AT>(w + 8 * q, t)];
          rh[q] += (long long)u.x * v.x;
          rh[q] -= (long long)u.z * v.z;
          rx[q] += (long long)u.x * v.y;
          rx[q] += (long long)u.y * v.x;
          rx[q] -= (long long)u.z * v.w;
          rx[q] -= (long long)u.w * v.z;
          ry[q] += (long long)u.x * vl.x;
          ry[q] += (long long)u.y * v.y;
          ry[q] += (long long)ul.x * v.x;
          ry[q] -= (long long)u.z * vl.y;
          ry[q] -= (long long)u.w * v.w;
          ry[q] -= (long long)ul.y * v.z;
          ih[q] += (long long)u.x * v.z;
          ih[q] += (long long)u.z * v.x;
          ix[q] += (long long)u.x * v.w;
          ix[q] += (long long)u.y * v.z;
          ix[q] += (long long)u.z * v.y;
          ix[q] += (long long)u.w * v.x;
          iy[q] += (long long)u.x * vl.y;
          iy[q] += (long long)u.y * v.w;
          iy[q] += (long long)ul.x * v.z;
          iy[q] += (long long)u.z * vl.x;
          iy[q] += (long long)u.w * v.y;
          iy[q] += (long long)ul.y * v.x;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = s_ea[w + 8 * q] + ec - 2096;
        acc[q].x += fx_value(rh[q], rx[q], ry[q], k);
        acc[q].y += fx_value(ih[q], ix[q], iy[q], k);
      }
    }
  }
}

// In-place lower Cholesky A = L L^H of an n x n Hermitian matrix (row-major,
// leading dimension lda).  The strict upper triangle is not referenced and
// is left unchanged.  Returns 0 or k+1 if the k-th pivot is not positive.
// smem: >= NB*NB + 2*TL*NB elements of T.
template <class T, bool CL = false>
__device__ int cta_potrf(T* A, int n, int lda, T* smem, Team<CL> tm = Team<CL>()) {
  using O = Ops<T>;
  using R = typename O::R;
  T* D = smem;   // the diagonal block; the products' Z once the panel is solved
  T* Pi = smem + NB * NB;
  T* Pj = Pi + TL * NB;
  __shared__ int info;
  __shared__ R rdiag[NB];   // 1 / L[j][j] of the current diagonal block
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) info = 0;
  __syncthreads();
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    // diagonal block -> shared, unblocked factorisation.  With a cluster every
    // CTA factors its own copy; the cluster barrier keeps the owner's write-back
    // of the factored block (below) from reaching A before every CTA has read it.
    for (int e = tid; e < kb * kb; e += blockDim.x) {
      int i = e / kb, j = e % kb;
      D[i * NB + j] = tm.ld(&A[(size_t)(k0 + i) * lda + k0 + j]);
    }
    if constexpr (CL) tm.sync();
    else __syncthreads();
    for (int j = 0; j < kb; ++j) {
      if (tid == 0) {
        R d = O::re(D[j * NB + j]);
        if (!(d > R(0))) { if (info == 0) info = k0 + j + 1; d = R(1); }
        D[j * NB + j] = O::from_re(sqrt(d));
        rdiag[j] = R(1) / O::re(D[j * NB + j]);
      }
      __syncthreads();
      const R inv = rdiag[j];
      for (int i = j + 1 + tid; i < kb; i += blockDim.x) D[i * NB + j] = O::scale(D[i * NB + j], inv);
      __syncthreads();
      // rank-1 update of the remaining lower part
      int rem = kb - j - 1;
      for (int e = tid; e < rem * rem; e += blockDim.x) {
        int i = j + 1 + e / rem, c = j + 1 + e % rem;
        if (c <= i) D[i * NB + c] = O::fnmac(D[i * NB + j], D[c * NB + j], D[i * NB + c]);
      }
      __syncthreads();
    }
    if (tm.own2(k0 / TL, k0 / TL)) {
      for (int e = tid; e < kb * kb; e += blockDim.x) {
        int i = e / kb, j = e % kb;
        if (j <= i) A[(size_t)(k0 + i) * lda + k0 + j] = D[i * NB + j];
      }
    }
    // panel: rows below solve x L_kk^H = a
    const int k1 = k0 + kb;
    for (int i = k1 + tid; i < n; i += blockDim.x) {
      if (!tm.own2(i / TL, k0 / TL)) continue;
      T* row = A + (size_t)i * lda + k0;
      T x[NB];
      for (int j = 0; j < kb; ++j) {
        T v = tm.ld(&row[j]);
        for (int t = 0; t < j; ++t) v = O::fnmac(x[t], D[j * NB + t], v);
        x[j] = O::scale(v, rdiag[j]);
      }
      for (int j = 0; j < kb; ++j) row[j] = x[j];
    }
    tm.sync();
    // trailing update A[i][j] -= sum_t L[i][t] conj(L[j][t]), lower part
    const int m = n - k1;
    const int nt = (m + TL - 1) / TL;
    for (int bi = 0; bi < nt; ++bi) {
      for (int bj = 0; bj <= bi; ++bj) {
        const int i0 = k1 + bi * TL, j0 = k1 + bj * TL;
        if (!tm.own2(i0 / TL, j0 / TL)) continue;
        T a[4], b[4], acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int r = 4 * w + u;
          a[u] = (i0 + r < n && lane < kb) ? tm.ld(&A[(size_t)(i0 + r) * lda + k0 + lane]) : O::zero();
          b[u] = (j0 + r < n && lane < kb) ? O::conj(tm.ld(&A[(size_t)(j0 + r) * lda + k0 + lane])) : O::zero();
          acc[u] = O::zero();
        }
        tile_product<T, true>(a, b, Pi, Pj, D, kb, acc);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + w + 8 * q, j = j0 + lane;
          if (i < n && j <= i) {
            size_t o = (size_t)i * lda + j;
            A[o] = O::sub(tm.ld(&A[o]), acc[q]);
          }
        }
      }
    }
    tm.sync();   // the next block reads what every thread (and CTA) updated
  }
  __syncthreads();
  return info;
}

// Mixed products of a triangular-factor entry (real or complex) with a
// right-hand-side entry (complex or real of the same precision).
__device__ __forceinline__ double2 lmul(double l, double2 b) { return make_double2(l * b.x, l * b.y); }
__device__ __forceinline__ double2 lmul(double2 l, double2 b) { return Ops<double2>::mul(l, b); }
__device__ __forceinline__ float2 lmul(float l, float2 b) { return make_float2(l * b.x, l * b.y); }
__device__ __forceinline__ float2 lmul(float2 l, float2 b) { return Ops<float2>::mul(l, b); }
// a factor entry in the right-hand sides' type
template <class TB, class TLt> __device__ __forceinline__ TB as_type(TLt l) {
  if constexpr (sizeof(TB) == sizeof(TLt)) return l;
  else return Ops<TB>::mk(l, 0);
}
__device__ __forceinline__ double lmul(double l, double b) { return l * b; }
__device__ __forceinline__ float lmul(float l, float b) { return l * b; }

// Solve L X = B in place (L lower triangular n x n of type TLt, B n x nrhs
// of type TB; TLt may be the real type of TB).  smem (bytes): room for
// NB*NB + 2*NB*TL elements of TB.
template <class TLt, class TB>
__device__ void cta_trsm_lower(const TLt* L, int n, int ldl, TB* B, int nrhs, int ldb, char* smem) {
  using OL = Ops<TLt>;
  using OB = Ops<TB>;
  using RB = typename OB::R;
  TB* Z = reinterpret_cast<TB*>(smem);
  TLt* D = reinterpret_cast<TLt*>(smem);   // the diagonal block; the products' Z once it is solved
  TB* Lt = Z + NB * NB;
  TB* Xt = Lt + TL * NB;
  __shared__ RB rdiag[NB];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    for (int e = tid; e < kb * kb; e += blockDim.x) {
      int i = e / kb, j = e % kb;
      D[i * NB + j] = (j <= i) ? L[(size_t)(k0 + i) * ldl + k0 + j] : OL::zero();
    }
    if (tid < kb) rdiag[tid] = RB(1) / OL::re(L[(size_t)(k0 + tid) * ldl + k0 + tid]);
    __syncthreads();
    // diagonal solve: one thread per right-hand-side column
    for (int c = tid; c < nrhs; c += blockDim.x) {
      TB x[NB];
      for (int r = 0; r < kb; ++r) {
        TB v = B[(size_t)(k0 + r) * ldb + c];
        for (int t = 0; t < r; ++t) v = OB::sub(v, lmul(D[r * NB + t], x[t]));
        x[r] = OB::scale(v, rdiag[r]);
        B[(size_t)(k0 + r) * ldb + c] = x[r];
      }
    }
    __syncthreads();
    // update rows below: B[i][c] -= sum_t L[i][k0+t] X[k0+t][c]
    const int k1 = k0 + kb;
    for (int i0 = k1; i0 < n; i0 += TL) {
      TB a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = i0 + 4 * w + u;
        a[u] = (r < n && lane < kb) ? as_type<TB>(L[(size_t)r * ldl + k0 + lane]) : OB::zero();
      }
      for (int c0 = 0; c0 < nrhs; c0 += TL) {
        TB b[4], acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int t = 4 * w + u;
          b[u] = (t < kb && c0 + lane < nrhs) ? B[(size_t)(k0 + t) * ldb + c0 + lane] : OB::zero();
          acc[u] = OB::zero();
        }
        tile_product<TB, false>(a, b, Lt, Xt, Z, kb, acc);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + w + 8 * q, cc = c0 + lane;
          if (i < n && cc < nrhs) {
            size_t o = (size_t)i * ldb + cc;
            B[o] = OB::sub(B[o], acc[q]);
          }
        }
      }
    }
    __syncthreads();
  }
  __syncthreads();
}

// Solve L^H X = B in place (backward substitution), complex L and B of the
// same type T.  smem as cta_trsm_lower.
template <class T>
__device__ void cta_trsm_lower_h(const T* L, int n, int ldl, T* B, int nrhs, int ldb, char* smem) {
  using O = Ops<T>;
  using R = typename O::R;
  T* D = reinterpret_cast<T*>(smem);
  T* Lt = D + NB * NB;
  T* Xt = Lt + TL * NB;
  __shared__ R rdiag[NB];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nblk = (n + NB - 1) / NB;
  for (int kbI = nblk - 1; kbI >= 0; --kbI) {
    const int k0 = kbI * NB;
    const int kb = min(NB, n - k0);
    for (int e = tid; e < kb * kb; e += blockDim.x) {
      int i = e / kb, j = e % kb;
      D[i * NB + j] = (j <= i) ? L[(size_t)(k0 + i) * ldl + k0 + j] : O::zero();
    }
    if (tid < kb) rdiag[tid] = R(1) / O::re(L[(size_t)(k0 + tid) * ldl + k0 + tid]);
    __syncthreads();
    // diagonal: (L_kk^H) x = b  ->  x_r = (b_r - sum_{t>r} conj(D[t][r]) x_t) / D[r][r]
    for (int c = tid; c < nrhs; c += blockDim.x) {
      T x[NB];
      for (int r = kb - 1; r >= 0; --r) {
        T v = B[(size_t)(k0 + r) * ldb + c];
        for (int t = r + 1; t < kb; ++t) v = O::sub(v, O::mul(O::conj(D[t * NB + r]), x[t]));
        x[r] = O::scale(v, rdiag[r]);
        B[(size_t)(k0 + r) * ldb + c] = x[r];
      }
    }
    __syncthreads();
    // update rows above: B[i][c] -= sum_t conj(L[k0+t][i]) X[k0+t][c], i < k0
    for (int i0 = 0; i0 < k0; i0 += TL) {
      T a[4];   // rows of L^H: row r of the transpose of L's rows k0 + t (loaded along r, placed by BT below)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int t = 4 * w + u;
        a[u] = (t < kb && i0 + lane < k0) ? O::conj(L[(size_t)(k0 + t) * ldl + i0 + lane]) : O::zero();
      }
      for (int c0 = 0; c0 < nrhs; c0 += TL) {
        T b[4], acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int t = 4 * w + u;
          b[u] = (t < kb && c0 + lane < nrhs) ? B[(size_t)(k0 + t) * ldb + c0 + lane] : O::zero();
          acc[u] = O::zero();
        }
        tile_product<T, false, true, true>(a, b, Lt, Xt, D, kb, acc);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + w + 8 * q, cc = c0 + lane;
          if (i < k0 && cc < nrhs) {
            size_t o = (size_t)i * ldb + cc;
            B[o] = O::sub(B[o], acc[q]);
          }
        }
      }
    }
    __syncthreads();
  }
  __syncthreads();
}

// C (m x n) = beta*C + alpha * op(A) * B where op(A) = A^H (A is k x m,
// transA = true) or A (m x k).  B is k x n.  All of type T (alpha real).
// smem: NB*NB + 2*TL*NB elements of T.
template <class T>
__device__ void cta_gemm(bool transA, int m, int n, int k, typename Ops<T>::R alpha,
                         const T* A, int lda, const T* B, int ldb,
                         typename Ops<T>::R beta, T* C, int ldc, T* smem) {
  using O = Ops<T>;
  T* At = smem;
  T* Bt = smem + TL * NB;
  T* Z = Bt + TL * NB;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int PER = TL * TL / CTA_THREADS;   // outputs per thread
  for (int i0 = 0; i0 < m; i0 += TL) {
    for (int j0 = 0; j0 < n; j0 += TL) {
      T acc[PER];
      for (int q = 0; q < PER; ++q) acc[q] = O::zero();
      for (int k0 = 0; k0 < k; k0 += NB) {
        T a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int v = 4 * w + u;
          if (transA) a[u] = (i0 + lane < m && k0 + v < k) ? O::conj(A[(size_t)(k0 + v) * lda + i0 + lane]) : O::zero();
          else a[u] = (i0 + v < m && k0 + lane < k) ? A[(size_t)(i0 + v) * lda + k0 + lane] : O::zero();
          b[u] = (k0 + v < k && j0 + lane < n) ? B[(size_t)(k0 + v) * ldb + j0 + lane] : O::zero();
        }
        if (transA) tile_product<T, false, true, true>(a, b, At, Bt, Z, NB, acc);
        else tile_product<T, false, false, true>(a, b, At, Bt, Z, NB, acc);
      }
      for (int q = 0; q < PER; ++q) {
        int e = tid + q * CTA_THREADS;
        int r = e / TL, c = e % TL;
        int i = i0 + r, j = j0 + c;
        if (i < m && j < n) {
          size_t o = (size_t)i * ldc + j;
          T v = O::scale(acc[q], alpha);
          C[o] = (beta == 0) ? v : O::add(O::scale(C[o], beta), v);
        }
      }
    }
  }
  __syncthreads();
}

// X = L^-1 in place of X = I (L lower triangular, n x n).  Blocks of X above
// the diagonal stay zero and are skipped: n^3/6 multiply-adds.
// smem: as cta_trsm_lower<T, T>.
template <class T, bool CL = false>
__device__ void cta_trinv_lower(const T* L, int n, int ldl, T* X, int ldx, char* smem, Team<CL> tm = Team<CL>()) {
  using O = Ops<T>;
  using R = typename O::R;
  T* D = reinterpret_cast<T*>(smem);
  T* Lt = D + NB * NB;
  T* Xt = Lt + TL * NB;
  __shared__ R rdiag[NB];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    const int k1 = k0 + kb;
    for (int e = tid; e < kb * kb; e += blockDim.x) {
      int i = e / kb, j = e % kb;
      D[i * NB + j] = (j <= i) ? tm.ld(&L[(size_t)(k0 + i) * ldl + k0 + j]) : O::zero();
    }
    if (tid < kb) rdiag[tid] = R(1) / O::re(tm.ld(&L[(size_t)(k0 + tid) * ldl + k0 + tid]));
    __syncthreads();
    for (int c = tid; c < k1; c += blockDim.x) {
      if (!tm.own_col(c / TL)) continue;
      T x[NB];
      for (int r = 0; r < kb; ++r) {
        T v = tm.ld(&X[(size_t)(k0 + r) * ldx + c]);
        for (int t = 0; t < r; ++t) v = O::fnma(D[r * NB + t], x[t], v);
        x[r] = O::scale(v, rdiag[r]);
        X[(size_t)(k0 + r) * ldx + c] = x[r];
      }
    }
    __syncthreads();
    for (int i0 = k1; i0 < n; i0 += TL) {
      T a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = i0 + 4 * w + u;
        a[u] = (r < n && lane < kb) ? tm.ld(&L[(size_t)r * ldl + k0 + lane]) : O::zero();
      }
      for (int c0 = 0; c0 < k1; c0 += TL) {
        if (!tm.own_col(c0 / TL)) continue;
        T b[4], acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int t = 4 * w + u;
          b[u] = (t < kb && c0 + lane < k1) ? tm.ld(&X[(size_t)(k0 + t) * ldx + c0 + lane]) : O::zero();
          acc[u] = O::zero();
        }
        tile_product<T, false>(a, b, Lt, Xt, D, kb, acc);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + w + 8 * q, cc = c0 + lane;
          if (i < n && cc < k1) {
            size_t o = (size_t)i * ldx + cc;
            X[o] = O::sub(tm.ld(&X[o]), acc[q]);
          }
        }
      }
    }
    __syncthreads();
  }
  __syncthreads();
}

// M = X^H X (M n x n, X kdim x n): only the lower tiles are computed, the
// strictly upper tiles are written as their conjugate mirror (half the flops
// of a full product).  With `tri` X is lower triangular (kdim = n) and each
// tile sums only over rows k >= its first row (X[k][i] = 0 for k < i):
// n^3/6 multiply-adds.  smem: NB*NB + 2*TL*NB elements of T.
template <class T, bool CL = false>
__device__ void cta_herk_lower(const T* X, int kdim, int n, int ldx, T* M, int ldm, T* smem, bool tri,
                               Team<CL> tm = Team<CL>()) {
  using O = Ops<T>;
  T* At = smem;
  T* Bt = smem + TL * NB;
  T* Z = Bt + TL * NB;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int PER = TL * TL / CTA_THREADS;
  for (int i0 = 0; i0 < n; i0 += TL) {
    for (int j0 = 0; j0 <= i0; j0 += TL) {
      if (!tm.own2(i0 / TL, j0 / TL)) continue;
      T acc[PER];
      for (int q = 0; q < PER; ++q) acc[q] = O::zero();
      for (int k0 = tri ? i0 : 0; k0 < kdim; k0 += NB) {
        T a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int t = 4 * w + u;
          a[u] = (i0 + lane < n && k0 + t < kdim) ? O::conj(tm.ld(&X[(size_t)(k0 + t) * ldx + i0 + lane])) : O::zero();
          b[u] = (k0 + t < kdim && j0 + lane < n) ? tm.ld(&X[(size_t)(k0 + t) * ldx + j0 + lane]) : O::zero();
        }
        tile_product<T, false, true>(a, b, At, Bt, Z, NB, acc);
      }
      for (int q = 0; q < PER; ++q) {
        int e = tid + q * CTA_THREADS;
        int r = e / TL, c = e % TL;
        int i = i0 + r, j = j0 + c;
        if (i < n && j < n) {
          M[(size_t)i * ldm + j] = acc[q];
          if (j0 < i0) M[(size_t)j * ldm + i] = O::conj(acc[q]);
        }
      }
    }
  }
  __syncthreads();
}

template <class T, bool CL = false>
__device__ void cta_herk_lower_tri(const T* X, int n, int ldx, T* M, int ldm, T* smem, Team<CL> tm = Team<CL>()) {
  cta_herk_lower<T, CL>(X, n, n, ldx, M, ldm, smem, true, tm);
}

}  // namespace dpgmg
