// Operators by cells: y = sum_K R_K^T A_K R_K x with one stored matrix per cell
// class (classes.cuh), for the V-cycle residual (complex64) and the CG operator
// (fixed point on the tensor cores).  The assembled rows stream every stored
// entry from HBM once per product; here a class's matrix stays in L2 and shared
// memory for all its cells, so the arithmetic and the gathers set the time.
#pragma once
#include "classes.cuh"
#include "digits.cuh"

namespace dpgmg {

// The operator by cells: ybuf[cell][a] = (A_K R_K x)_a of every cell, then
// k_cell_sum adds the cells of each DOF.
static __global__ void __launch_bounds__(CLS_THREADS, CLS_CTAS) k_class_cell(const int32_t* __restrict__ idx,
                                                            const int32_t* __restrict__ cls, int n, int64_t stride,
                                                            const int4* __restrict__ items,
                                                            const int32_t* __restrict__ mem,
                                                            const float2* __restrict__ Wall,
                                                            const uint8_t* __restrict__ rflag,
                                                            const float2* __restrict__ x, float2* __restrict__ ybuf,
                                                            int64_t offU) {
  __shared__ ClassSmem sm;
  const int4 it = items[blockIdx.x];
  const int cnt = it.y, a0 = it.z;
  const int e = mem[it.x], c = cls[e];
  if ((int)threadIdx.x < cnt)
    sm.base[threadIdx.x] = sm.obase[threadIdx.x] = (int64_t)mem[it.x + threadIdx.x] * n;
  __syncthreads();
  const float2* W = Wall + c * stride;
  const int32_t* rep = idx + (int64_t)e * n;
#define DPG_ITEM(TX, MPT)                                                                                \
  if (rflag[c] != 0)                                                                                     \
    class_item<float2, TX, MPT, false>(sm, W, patch_ldr(n), n, n, a0, cnt, idx, x, x, n, ybuf, nullptr, rep, offU);  \
  else                                                                                                   \
    class_item<float2, TX, MPT, true>(sm, W, patch_ld(n), n, n, a0, cnt, idx, x, x, n, ybuf, nullptr, rep, offU)
  switch (it.w) {
    case CLS_64x32: DPG_ITEM(16, 4); break;
    case CLS_64x16: DPG_ITEM(16, 2); break;
    case CLS_64x8: DPG_ITEM(16, 1); break;
    case CLS_32x32: DPG_ITEM(8, 2); break;
    default: DPG_ITEM(8, 1); break;
  }
#undef DPG_ITEM
}

// ---- CG operator ----
__device__ __forceinline__ void df_add(float& sh, float& sl, float p, float q) {
  const float s = sh + p;
  const float bb = s - sh;
  const float e = (sh - (s - bb)) + (p - bb);
  sh = s;
  sl += e + q;
}
__device__ __forceinline__ void df_mul(float ah, float al, float xh, float xl, float& p, float& q) {
  p = ah * xh;
  q = fmaf(ah, xh, -p);
  q = fmaf(ah, xl, q);
  q = fmaf(al, xh, q);
}

// The same product for the CG operator: 56-bit fixed point on the tensor cores.
// A row a of a class matrix is 2^ea times integers below 2^55, the DOFs of a
// cell are 2^ex times such integers, and both are written as DG_S = 7 signed
// digits of 8 bits (-128 .. 127), which bf16 holds exactly.  Digit products of
// equal weight s + t = o share one FP32 accumulator per output: at most
// 7 DG_KC products of at most 2^14 each, an integer below 2^24, so every
// accumulator is exact (error-free splitting as in Mukunoki, Ozaki, Ogita and
// Imamura, "DGEMM using tensor cores", 2020).  Pairs with o > 6 lie below the
// operands' own rounding and are left out.  The seven accumulators are joined
// with error-free FP32 sums into high and low parts.
//
// Bound: 28 bf16 products per entry and real column on mma.sync (m16n8k16,
// 0.5 a clock and SM: 50 us on a layered 32 x 32 x 16 mesh, p = 3), where the
// double-float form took 12 FP32 instructions per real product.  Operator there
// 281 -> 154 us, on 16^3, p = 3, 88 -> 65 us, and 0.2 to 0.9 of the error against
// complex128 in norm (2.2e-15 to 3e-15 on residuals, before 3e-15 to 6e-15).  Tried:
// the next tile's digits prefetched into L1, no change; the conversions are
// half of the instructions, but twice as many only cost 4%.
//
// Error of an output: about 2^-55 of the row's largest entry times the column's
// largest per product, where the double-float form has 2^-48 of each product.  The
// matrices are dense, Hermitian and positive definite, and how far an output's own
// products stay below that product of the maxima goes with the spread of the
// diagonal, max A_kk / min A_kk.  Relative to sum_k |A_ak x_k|, entry by entry, the
// error is at most the assembled double-float rows' in the mean square (0.2 to 1.0
// times on random vectors, residuals, V-cycle outputs and solutions; 0.3 to 1.3
// times at the worst entry) up to a spread of 2^12 for p <= 4 and 2^11 for p = 5:
// cubes of 1/4 to 1/24 at omega h > 0.5 or so.  At 2^12, p = 5, it has twice the error on
// smooth solutions, at 2^25 (elements of 1/3000, or 1:100 flat ones) 30 to 70 times.
// So digits are kept up to digit_spread(n), beyond it the assembled rows.
//
// A CTA turns the DOFs of up to 32 cells (64 real columns,
// DG_KC rows) into digits once, in shared memory; a warp owns 16 outputs x 8
// cells, with the matrix's digits read from L2 in fragment order (512 bytes a
// warp and tile).
constexpr int DG_LD = DG_KC + 8;   // row length in shared memory: 240 bytes, 8 rows on distinct banks
constexpr int DG_COLS = 64;
constexpr int DG_THREADS = 256;
constexpr int DG_SMEM = DG_S * DG_COLS * DG_LD * 2;

__device__ __forceinline__ void mma_bf16(float c[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// the value of h in units of 2^(emax - 181): below 2^55 when emax is the column's exponent
__device__ __forceinline__ long long digit_fixed(float h, int emax) {
  const uint32_t u = __float_as_uint(h);
  const int e = max((int)(u >> 23) & 255, 1), sh = e - emax + 31;   // denormal parts: exponent 1, no leading bit
  const long long m = (u & 0x7fffff) | ((u & 0x7f800000u) ? 0x800000 : 0);
  if (sh < -25) return 0;
  const long long f = sh >= 0 ? m << min(sh, 31) : (m + (1ll << (-sh - 1))) >> -sh;
  return (int)u < 0 ? -f : f;
}

static __global__ void __launch_bounds__(DG_THREADS, 2) k_class_cell_dg(
    const int32_t* __restrict__ idx, const int32_t* __restrict__ cls, int n, int64_t stride,
    const int4* __restrict__ items, const int32_t* __restrict__ mem, const uint4* __restrict__ Dall,
    const float* __restrict__ rowscale, const uint8_t* __restrict__ rflag, const float2* __restrict__ xh,
    const float2* __restrict__ xl, float4* __restrict__ ybuf, int64_t offU) {
  extern __shared__ __align__(16) uint16_t Bs[];   // [DG_S][DG_COLS][DG_LD] digits of column 2 m + (0 re, 1 im)
  __shared__ float cscale[32];
  __shared__ int64_t base[32];
  const int4 it = items[blockIdx.x];   // first member, members, first 16-row tile, tiles
  const int cnt = it.y, c = cls[mem[it.x]];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid < 32) base[tid] = tid < cnt ? (int64_t)mem[it.x + tid] * n : -1;
  __syncthreads();
  const int nq = (cnt + 7) / 8, npair = nq * it.w, KT = (n + 15) / 16, MT = KT;
  const bool real = rflag[c] != 0;
  const uint4* Dc = Dall + c * stride;
  const float* rs = rowscale + (int64_t)c * MT * 16;
  const int32_t* rep = idx + (int64_t)mem[it.x] * n;
  for (int k0 = 0; k0 < n; k0 += DG_KC) {
    const int nkt = min(DG_KC / 16, KT - k0 / 16);
    if (k0 > 0) __syncthreads();   // the last chunk's readers are done
    // digits of the columns: a warp takes members w, w + 8, ..., lanes two rows each
    int g[4][2][2];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int m = w + 8 * j, k = k0 + 64 * i + 2 * lane + u;
          g[j][i][u] = (m < cnt && k < n && 64 * i + 2 * lane < DG_KC) ? __ldg(idx + base[m] + k) : -1;
        }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = w + 8 * j;
      if (m >= 8 * nq) break;   // uniform over the warp
      float2 h[2][2], l[2][2];
      uint32_t top = 0;   // bits of the largest magnitude
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int gi = g[j][i][u];
          h[i][u] = l[i][u] = make_float2(0.f, 0.f);
          if (gi >= 0) {
            h[i][u] = xh[gi];
            l[i][u] = xl[gi];
            if (real) {
              const int s = gi < offU ? -1 : 0;
              h[i][u] = mul_i(h[i][u], s);
              l[i][u] = mul_i(l[i][u], s);
            }
          }
          top = max(top, max(__float_as_uint(h[i][u].x) & 0x7fffffffu, __float_as_uint(h[i][u].y) & 0x7fffffffu));
        }
      top = __reduce_max_sync(0xffffffffu, top);
      // the column is 2^(emax - 181) times its integers; a largest value above 1 - 2^-7 of the power of two takes
      // the next one, so that the leading digit with its carry stays below 128
      const int emax = max((int)((top + 0x20000u) >> 23), 1);
      // 2^(emax - 128); infinities and NaN give NaN
      if (lane == 0)
        cscale[m] = top >= 0x7f800000u ? __uint_as_float(0x7fffffffu)
                                       : (emax > 1 ? __uint_as_float((uint32_t)(emax - 1) << 23)
                                                   : __uint_as_float(0x00400000u));
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int k = 64 * i + 2 * lane;
        if (k >= 16 * nkt) continue;
        uint32_t dr[DG_S], di[DG_S];
        digit_pairs(digit_fixed(h[i][0].x, emax) + digit_fixed(l[i][0].x, emax),
                    digit_fixed(h[i][1].x, emax) + digit_fixed(l[i][1].x, emax), dr);
        digit_pairs(digit_fixed(h[i][0].y, emax) + digit_fixed(l[i][0].y, emax),
                    digit_fixed(h[i][1].y, emax) + digit_fixed(l[i][1].y, emax), di);
#pragma unroll
        for (int s = 0; s < DG_S; ++s) {
          *reinterpret_cast<uint32_t*>(Bs + (s * DG_COLS + 2 * m) * DG_LD + k) = dr[s];
          *reinterpret_cast<uint32_t*>(Bs + (s * DG_COLS + 2 * m + 1) * DG_LD + k) = di[s];
        }
      }
    }
    __syncthreads();
    const int gr = lane >> 2, tq = lane & 3;
    for (int p = w; p < npair; p += DG_THREADS / 32) {
      const int mt = it.z + p / nq, q0 = p % nq;   // rows 16 mt .. + 15, members 8 q0 .. + 7
      float rh[2][4], rl[2][4];
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) rh[t][q] = rl[t][q] = 0.f;
      // real classes: one pass.  Complex ones: Ar (xr, xi), then Ai (-xi, xr)
      for (int half = 0; half < (real ? 1 : 2); ++half) {
        float acc[2][DG_S][4];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int s = 0; s < DG_S; ++s)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[t][s][q] = 0.f;
        // ldmatrix rows: lanes 0-7 column tile 0, k 0-7; 8-15 the same, k 8-15; 16-31 column tile 1
        const int col = 16 * q0 + ((lane >> 4) << 3) + (lane & 7);
        uint32_t saddr = (uint32_t)__cvta_generic_to_shared(Bs + (col ^ half) * DG_LD + ((lane >> 3) & 1) * 8);
        const uint32_t flip = (half && (gr & 1) == 0) ? 0x80008000u : 0u;   // column re of the second pass: -xi
        const uint4* Da = Dc + ((int64_t)(half * MT + mt) * KT + k0 / 16) * (DG_S * 32) + lane;
        for (int kt = 0; kt < nkt; ++kt, Da += DG_S * 32, saddr += 32) {
          uint4 a[DG_S];
#pragma unroll
          for (int s = 0; s < DG_S; ++s) a[s] = __ldg(Da + s * 32);
#pragma unroll
          for (int t = 0; t < DG_S; ++t) {
            uint32_t b0, b1, b2, b3;
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3)
                         : "r"(saddr + t * (DG_COLS * DG_LD * 2)));
            b0 ^= flip;
            b1 ^= flip;
            b2 ^= flip;
            b3 ^= flip;
#pragma unroll
            for (int s = 0; s + t < DG_S; ++s) {
              mma_bf16(acc[0][s + t], a[s], b0, b1);
              mma_bf16(acc[1][s + t], a[s], b2, b3);
            }
          }
        }
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float f = 1.f;
#pragma unroll
            for (int o = 0; o < DG_S; ++o, f *= 1.f / 256.f) df_add(rh[t][q], rl[t][q], acc[t][o][q] * f, 0.f);
          }
      }
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int m = 8 * q0 + 4 * t + tq;
        if (m >= cnt) continue;
        const float cs = cscale[m];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int a = 16 * mt + gr + 8 * r;
          if (a >= n) continue;
          const float sc = rs[a];
          auto scale = [&](float v) { return v * sc * cs; };
          float4 v = make_float4(scale(rh[t][2 * r]), scale(rl[t][2 * r]), scale(rh[t][2 * r + 1]),
                                 scale(rl[t][2 * r + 1]));
          if (real && rep[a] < offU) v = make_float4(-v.z, -v.w, v.x, v.y);   // output phase i, exact
          float4* o = ybuf + base[m] + a;
          if (k0 > 0) {   // this thread's sum over the earlier chunks
            const float4 y = *o;
            df_add(v.x, v.y, y.x, y.y);
            df_add(v.z, v.w, y.z, y.w);
          }
          *o = v;
        }
      }
    }
  }
}

// calls f(value) for the slots of DOF g in list order (a fixed-pitch row of
// tab, or a CSR row); indices and then values are loaded up to four at a time
template <class V, class F>
__device__ __forceinline__ void for_slots(const int32_t* __restrict__ tab, const int64_t* __restrict__ sptr,
                                          const int32_t* __restrict__ slots, int64_t offE, int64_t offF,
                                          const V* __restrict__ v, int64_t g, F&& f) {
  auto four = [&](int4 t) {
    V a, b, c, d;
    if (t.x >= 0) a = v[t.x];
    if (t.y >= 0) b = v[t.y];
    if (t.z >= 0) c = v[t.z];
    if (t.w >= 0) d = v[t.w];
    if (t.x >= 0) f(a);
    if (t.y >= 0) f(b);
    if (t.z >= 0) f(c);
    if (t.w >= 0) f(d);
  };
  if (tab) {
    const int32_t* row = tab + cell_row(g, offE, offF);
    if (g >= offF) {   // faces: the two sides
      const int2 t = *reinterpret_cast<const int2*>(row);
      four(make_int4(t.x, t.y, -1, -1));
    } else {
      four(*reinterpret_cast<const int4*>(row));
      if (g < offE) four(*reinterpret_cast<const int4*>(row + 4));
    }
  } else {
    const int64_t s1 = sptr[g + 1];
    for (int64_t s = sptr[g]; s < s1; s += 4)
      four(make_int4(slots[s], s + 1 < s1 ? slots[s + 1] : -1, s + 2 < s1 ? slots[s + 2] : -1,
                     s + 3 < s1 ? slots[s + 3] : -1));
  }
}

// y = sum of the cell products (mode 0) or b minus it (mode 1)
static __global__ void k_cell_sum(const int32_t* __restrict__ tab, const int64_t* __restrict__ sptr,
                           const int32_t* __restrict__ slots, int64_t offE, int64_t offF,
                           const float2* __restrict__ ybuf, const float2* __restrict__ b, float2* __restrict__ y,
                           int64_t n, int mode) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= n) return;
  float2 acc = make_float2(0.f, 0.f);
  for_slots(tab, sptr, slots, offE, offF, ybuf, g, [&](float2 v) { acc = Ops<float2>::add(acc, v); });
  y[g] = mode ? Ops<float2>::sub(b[g], acc) : acc;
}

// the same for the double-float cell products; the sums over a DOF's cells
// stay FP32 pairs, turned into complex128 once
static __global__ void k_cell_sum_df(const int32_t* __restrict__ tab, const int64_t* __restrict__ sptr,
                              const int32_t* __restrict__ slots, int64_t offE, int64_t offF,
                              const float4* __restrict__ ybuf, const double2* __restrict__ b, double2* __restrict__ y,
                              int64_t n, int mode) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= n) return;
  float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
  for_slots(tab, sptr, slots, offE, offF, ybuf, g, [&](float4 v) {
    df_add(rh, rl, v.x, v.y);
    df_add(ih, il, v.z, v.w);
  });
  const double re = wide(rh) + wide(rl), im = wide(ih) + wide(il);
  y[g] = mode ? make_double2(b[g].x - re, b[g].y - im) : make_double2(re, im);
}

// y = A x (mode 0) or b - A x (mode 1), x = xh + xl
inline void cell_op_apply_df(const CellOpDev& D, const float2* xh, const float2* xl, const double2* b, double2* y,
                             int mode, cudaStream_t st) {
  k_class_cell_dg<<<(unsigned)D.ndgitems, DG_THREADS, DG_SMEM, st>>>(D.idx, D.cls, D.n, D.dgstride(), D.dgitems, D.mem,
                                                                    D.dig, D.dgrow, D.rflag, xh, xl, D.ydf, D.offU);
  DPG_CHECK_LAUNCH();
  k_cell_sum_df<<<(unsigned)((D.ndof + 255) / 256), 256, 0, st>>>(D.tab, D.sptr, D.slots, D.offE, D.offF, D.ydf, b, y,
                                                                 D.ndof, mode);
  DPG_CHECK_LAUNCH();
}

inline void cell_op_apply(const CellOpDev& D, const float2* x, const float2* b, float2* y, int mode, cudaStream_t st) {
  k_class_cell<<<(unsigned)D.nitems, CLS_THREADS, 0, st>>>(D.idx, D.cls, D.n, D.stride(), D.items, D.mem, D.W, D.rflag,
                                                          x, D.ybuf, D.offU);
  DPG_CHECK_LAUNCH();
  k_cell_sum<<<(unsigned)((D.ndof + 255) / 256), 256, 0, st>>>(D.tab, D.sptr, D.slots, D.offE, D.offF, D.ybuf, b, y,
                                                              D.ndof, mode);
  DPG_CHECK_LAUNCH();
}

// ---- macro-grid transfers with shared class matrices ----
// BACK:  x_I = A_II^-1 r_I - Y x_S          (rows: I then S; outputs: I, scattered)
// !BACK: cbuf[K][a] = sum_i conj(Y[i][a]) r_i (rows: I; outputs: S)
// idx: [nK][nI + nS] DOFs, I then S.
template <bool BACK>
static __global__ void __launch_bounds__(CLS_THREADS, CLS_CTAS) k_class_macro(
    const int32_t* __restrict__ idx, const int32_t* __restrict__ cls, int nI, int nS, int64_t stride,
    const int4* __restrict__ items, const int32_t* __restrict__ mem, const float2* __restrict__ Wall,
    const uint8_t* __restrict__ rflag, const float2* r, float2* out, int64_t offU) {
  __shared__ ClassSmem sm;
  const int4 it = items[blockIdx.x];
  const int cnt = it.y, a0 = it.z;
  const int K = mem[it.x], c = cls[K];
  if ((int)threadIdx.x < cnt) {
    const int64_t m = mem[it.x + threadIdx.x];
    sm.base[threadIdx.x] = m * (nI + nS);
    sm.obase[threadIdx.x] = BACK ? m * (nI + nS) : m * nS;
  }
  __syncthreads();
  const float2* W = Wall + c * stride;
  const int n = BACK ? nI + nS : nI, nout = BACK ? nI : nS;
  const int32_t* rep = idx + (int64_t)K * (nI + nS) + (BACK ? 0 : nI);
  const int32_t* oidx = BACK ? idx : nullptr;
#define DPG_ITEM(TX, MPT)                                                                                            \
  if (rflag[c] != 0)                                                                                                 \
    class_item<float2, TX, MPT, false, BACK>(sm, W, patch_ldr(nout), n, nout, a0, cnt, idx, r, out, nI, out, oidx,   \
                                             rep, offU);                                                             \
  else                                                                                                               \
    class_item<float2, TX, MPT, true, BACK>(sm, W, patch_ld(nout), n, nout, a0, cnt, idx, r, out, nI, out, oidx, rep, \
                                            offU)
  switch (it.w) {
    case CLS_64x32: DPG_ITEM(16, 4); break;
    case CLS_64x16: DPG_ITEM(16, 2); break;
    case CLS_64x8: DPG_ITEM(16, 1); break;
    case CLS_32x32: DPG_ITEM(8, 2); break;
    default: DPG_ITEM(8, 1); break;
  }
#undef DPG_ITEM
}

// class matrices of both transfers from the first cell of every class (one CTA
// per class): as reals when every entry is real once the unit phases are taken out
static __global__ void k_macro_class(const int32_t* __restrict__ idx, const int64_t* __restrict__ rep, int nI, int nS,
                                     int64_t offU, bool pack, const float2* __restrict__ Y,
                                     const float2* __restrict__ Ai, float2* __restrict__ Wb, int64_t bstride,
                                     float2* __restrict__ Wc, int64_t cstride, uint8_t* __restrict__ rflag) {
  const int64_t c = blockIdx.x, K = rep[c];
  const int32_t* g = idx + K * (nI + nS);
  const float2 *Yk = Y + K * (int64_t)nI * nS, *Ak = Ai + K * (int64_t)nI * nI;
  const int n = nI + nS;
  auto phat = [&](int q) { return g[q] >= 0 && g[q] < offU ? 1 : 0; };
  // entry (row i of I, column q of [I, S]) of [A_II^-1, -Y]
  auto entry = [&](int i, int q) {
    if (q < nI) return Ak[i * nI + q];
    const float2 y = Yk[(int64_t)i * nS + q - nI];
    return make_float2(-y.x, -y.y);
  };
  bool cplx = !pack;
  if (pack)
    for (int t = threadIdx.x; t < nI * n; t += blockDim.x)
      if (mul_i(entry(t / n, t % n), phat(t % n) - phat(t / n)).y != 0.f) cplx = true;
  cplx = __syncthreads_or(cplx) != 0;
  float2 *B = Wb + c * bstride, *Cc = Wc + c * cstride;
  const int lb = (int)(cplx ? patch_ld(nI) : patch_ldr(nI)), lc = (int)(cplx ? patch_ld(nS) : patch_ldr(nS));
  for (int t = threadIdx.x; t < n * lb; t += blockDim.x) {   // B[k][a] = conj([A_II^-1, -Y][a][k])
    const int k = t / lb, a = t % lb;
    const float2 v = a < nI ? entry(a, k) : make_float2(0.f, 0.f);
    if (cplx) B[t] = make_float2(v.x, -v.y);
    else reinterpret_cast<float*>(B)[t] = a < nI ? mul_i(v, phat(k) - phat(a)).x : 0.f;
  }
  for (int t = threadIdx.x; t < nI * lc; t += blockDim.x) {  // C[i][a] = Y[i][a]
    const int i = t / lc, a = t % lc;
    const float2 v = a < nS ? Yk[(int64_t)i * nS + a] : make_float2(0.f, 0.f);
    if (cplx) Cc[t] = v;
    else reinterpret_cast<float*>(Cc)[t] = a < nS ? mul_i(v, phat(nI + a) - phat(i)).x : 0.f;
  }
  if (threadIdx.x == 0) rflag[c] = cplx ? 0 : 1;
}

static __global__ void k_macro_index(const int64_t* __restrict__ Ig, const int64_t* __restrict__ Sg, int nI, int nS,
                                     int64_t nK, int32_t* __restrict__ idx) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= nK * (nI + nS)) return;
  const int64_t K = q / (nI + nS);
  const int i = (int)(q % (nI + nS));
  idx[q] = (int32_t)(i < nI ? Ig[K * nI + i] : Sg[K * nS + i - nI]);
}

inline void macro_backsub(const MacroOpDev& D, const float2* r, float2* x, cudaStream_t st) {
  k_class_macro<true><<<(unsigned)D.nbitems, CLS_THREADS, 0, st>>>(D.idx, D.cls, D.nI, D.nS, D.bstride(), D.bitems,
                                                                  D.mem, D.Wb, D.rflag, r, x, D.offU);
  DPG_CHECK_LAUNCH();
}
inline void macro_condense_apply(const MacroOpDev& D, const float2* r, float2* cbuf, cudaStream_t st) {
  k_class_macro<false><<<(unsigned)D.ncitems, CLS_THREADS, 0, st>>>(D.idx, D.cls, D.nI, D.nS, D.cstride(), D.citems,
                                                                   D.mem, D.Wc, D.rflag, r, cbuf, D.offU);
  DPG_CHECK_LAUNCH();
}

}  // namespace dpgmg
