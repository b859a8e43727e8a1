// Operators by cells: y = sum_K R_K^T A_K R_K x with one stored matrix per cell
// class (classes.cuh), for the V-cycle residual (complex64) and the CG operator
// (double-float).  The assembled rows stream every stored entry from HBM once
// per product; here a class's matrix stays in L2 and shared memory for all its
// cells, so the FP32 pipe and the gathers set the time.
#pragma once
#include "classes.cuh"

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

// ---- double-float form (CG operator) ----
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

// The same product for the CG operator in double-float (solve.cu): matrices as
// FP32 high and low parts (W + Wl), x likewise, products and sums with
// error-free FP32 transformations.  12 FP32 instructions per real product, so
// the FP32 pipe bounds it; a thread owns 4 outputs x MPT members, 16 bytes of
// accumulator each.  ybuf: (re hi, re lo, im hi, im lo).
constexpr int CDF_K = 8;        // rows per stage
constexpr int CDF_STAGES = 3;
struct ClassDfSmem {
  __align__(16) unsigned char w[CDF_STAGES][2][CDF_K * 64 * sizeof(float2)];   // high, low parts
  __align__(16) float4 r[2][CDF_K][16 + 1];
  int64_t base[16];
};

template <int TX, int MPT, bool CX>
__device__ __forceinline__ void class_item_df(ClassDfSmem& sm, const float2* __restrict__ Wh,
                                              const float2* __restrict__ Wl, int64_t ld, int n, int a0, int cnt,
                                              const int32_t* __restrict__ idx, const float2* __restrict__ xh,
                                              const float2* __restrict__ xl, float4* __restrict__ out,
                                              const int32_t* __restrict__ rep_idx, int64_t offU) {
  constexpr int TM = 4 * TX, TN = (CLS_THREADS / TX) * MPT;
  constexpr int EL = CX ? 8 : 4;
  constexpr int ROW16 = TM * EL / 16;
  constexpr int NP = 2 * CDF_K * ROW16;                            // 16-byte pieces per stage, high then low
  constexpr int NW = (NP + CLS_THREADS - 1) / CLS_THREADS;
  constexpr int NG = (CDF_K * TN + CLS_THREADS - 1) / CLS_THREADS; // gathered values per thread and chunk
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int gk = tid % CDF_K, gm = tid / CDF_K;                    // gather: row, first member (then + 16)
  const char* W[2] = {reinterpret_cast<const char*>(Wh) + (int64_t)a0 * EL,
                      reinterpret_cast<const char*>(Wl) + (int64_t)a0 * EL};
  const int wcols = (int)(ld - a0);
  const int nch = (n + CDF_K - 1) / CDF_K;

  auto load_w = [&](int c) {
    if (c < nch) {
#pragma unroll
      for (int q = 0; q < NW; ++q) {
        const int p = tid + q * CLS_THREADS;
        if (NP % CLS_THREADS == 0 || p < NP) {
          const int part = p / (CDF_K * ROW16), pp = p % (CDF_K * ROW16), row = pp / ROW16, col = pp % ROW16;
          const int k = c * CDF_K + row;
          const bool in = k < n && col * (16 / EL) < wcols;
          cp_async16_zfill(sm.w[c % CDF_STAGES][part] + row * (TM * EL) + col * 16,
                           in ? W[part] + (int64_t)k * ld * EL + col * 16 : W[part], in);
        }
      }
    }
    cp_async_commit();
  };
  int gi[NG];
  float4 gv[NG];
  auto load_idx = [&](int c) {
    const int k = c * CDF_K + gk;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int m = gm + 16 * q;
      gi[q] = (k < n && m < cnt) ? __ldg(idx + sm.base[m] + k) : -1;
    }
  };
  auto load_val = [&]() {
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      float2 h = make_float2(0.f, 0.f), l = h;
      if (gi[q] >= 0) {
        h = xh[gi[q]];
        l = xl[gi[q]];
        if (!CX) {
          const int s = gi[q] < offU ? -1 : 0;
          h = mul_i(h, s);
          l = mul_i(l, s);
        }
      }
      gv[q] = make_float4(h.x, l.x, h.y, l.y);
    }
  };
  auto store_val = [&](int c) {
#pragma unroll
    for (int q = 0; q < NG; ++q)
      if (gm + 16 * q < TN) sm.r[c & 1][gk][gm + 16 * q] = gv[q];
  };
  float rh[MPT][4], rl[MPT][4], ih[MPT][4], il[MPT][4];
#pragma unroll
  for (int m = 0; m < MPT; ++m)
#pragma unroll
    for (int u = 0; u < 4; ++u) rh[m][u] = rl[m][u] = ih[m][u] = il[m][u] = 0.f;
#pragma unroll
  for (int c = 0; c < CDF_STAGES - 1; ++c) load_w(c);
  load_idx(0);
  load_val();
  store_val(0);
  load_idx(1);
  for (int c = 0; c < nch; ++c) {
    cp_async_wait<CDF_STAGES - 2>();
    __syncthreads();
    load_w(c + CDF_STAGES - 1);
    load_val();
    load_idx(c + 2);
    const unsigned char* wh = sm.w[c % CDF_STAGES][0] + tx * (4 * EL);
    const unsigned char* wl = sm.w[c % CDF_STAGES][1] + tx * (4 * EL);
    const float4* rs = &sm.r[c & 1][0][ty * MPT];
#pragma unroll 2
    for (int k = 0; k < CDF_K; ++k) {
      float4 rv[MPT];
#pragma unroll
      for (int m = 0; m < MPT; ++m) rv[m] = rs[k * (16 + 1) + m];
      float h[CX ? 8 : 4], l[CX ? 8 : 4];
#pragma unroll
      for (int q = 0; q < (CX ? 2 : 1); ++q) {
        *reinterpret_cast<float4*>(h + 4 * q) = *reinterpret_cast<const float4*>(wh + k * (TM * EL) + 16 * q);
        *reinterpret_cast<float4*>(l + 4 * q) = *reinterpret_cast<const float4*>(wl + k * (TM * EL) + 16 * q);
      }
#pragma unroll
      for (int m = 0; m < MPT; ++m)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float p, q;
          if constexpr (!CX) {
            df_mul(h[u], l[u], rv[m].x, rv[m].y, p, q);
            df_add(rh[m][u], rl[m][u], p, q);
            df_mul(h[u], l[u], rv[m].z, rv[m].w, p, q);
            df_add(ih[m][u], il[m][u], p, q);
          } else {   // conj(w) x
            df_mul(h[2 * u], l[2 * u], rv[m].x, rv[m].y, p, q);
            df_add(rh[m][u], rl[m][u], p, q);
            df_mul(h[2 * u + 1], l[2 * u + 1], rv[m].z, rv[m].w, p, q);
            df_add(rh[m][u], rl[m][u], p, q);
            df_mul(h[2 * u], l[2 * u], rv[m].z, rv[m].w, p, q);
            df_add(ih[m][u], il[m][u], p, q);
            df_mul(h[2 * u + 1], l[2 * u + 1], rv[m].x, rv[m].y, p, q);
            df_add(ih[m][u], il[m][u], -p, -q);
          }
        }
    }
    if (c + 1 < nch) store_val(c + 1);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int a = a0 + 4 * tx + u;
    if (a >= n) continue;
    const bool s = !CX && rep_idx[a] < offU;   // output phase i, exact
#pragma unroll
    for (int m = 0; m < MPT; ++m) {
      const int q = ty * MPT + m;
      if (q < cnt)
        out[sm.base[q] + a] = s ? make_float4(-ih[m][u], -il[m][u], rh[m][u], rl[m][u])
                                : make_float4(rh[m][u], rl[m][u], ih[m][u], il[m][u]);
    }
  }
}

static __global__ void __launch_bounds__(CLS_THREADS, 4) k_class_cell_df(const int32_t* __restrict__ idx,
                                                               const int32_t* __restrict__ cls, int n, int64_t stride,
                                                               const int4* __restrict__ items,
                                                               const int32_t* __restrict__ mem,
                                                               const float2* __restrict__ Wh,
                                                               const float2* __restrict__ Wl,
                                                               const uint8_t* __restrict__ rflag,
                                                               const float2* __restrict__ xh,
                                                               const float2* __restrict__ xl,
                                                               float4* __restrict__ ybuf, int64_t offU) {
  __shared__ ClassDfSmem sm;
  const int4 it = items[blockIdx.x];
  const int cnt = it.y, a0 = it.z;
  const int e = mem[it.x], c = cls[e];
  if ((int)threadIdx.x < cnt) sm.base[threadIdx.x] = (int64_t)mem[it.x + threadIdx.x] * n;
  __syncthreads();
  const float2 *H = Wh + c * stride, *L = Wl + c * stride;
  const int32_t* rep = idx + (int64_t)e * n;
#define DPG_ITEM(TX, MPT)                                                                                   \
  if (rflag[c] != 0)                                                                                        \
    class_item_df<TX, MPT, false>(sm, H, L, patch_ldr(n), n, a0, cnt, idx, xh, xl, ybuf, rep, offU);        \
  else                                                                                                      \
    class_item_df<TX, MPT, true>(sm, H, L, patch_ld(n), n, a0, cnt, idx, xh, xl, ybuf, rep, offU)
  switch (it.w) {   // items of at most 16 members
    case CLS_64x16: DPG_ITEM(16, 2); break;
    case CLS_64x8: DPG_ITEM(16, 1); break;
    default: DPG_ITEM(8, 1); break;   // CLS_32x16
  }
#undef DPG_ITEM
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
  const double re = (double)rh + (double)rl, im = (double)ih + (double)il;
  y[g] = mode ? make_double2(b[g].x - re, b[g].y - im) : make_double2(re, im);
}

// y = A x (mode 0) or b - A x (mode 1) in double-float, x = xh + xl
inline void cell_op_apply_df(const CellOpDev& D, const float2* xh, const float2* xl, const double2* b, double2* y,
                             int mode, cudaStream_t st) {
  k_class_cell_df<<<(unsigned)D.nitems16, CLS_THREADS, 0, st>>>(D.idx, D.cls, D.n, D.stride(), D.items16, D.mem, D.W,
                                                               D.Wlo, D.rflag, xh, xl, D.ydf, D.offU);
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
