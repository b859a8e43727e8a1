// Products with matrices that many blocks share.
//
// On a uniform mesh the matrix of a vertex patch depends only on the classes
// (impedance faces and wavespeed, Sec. 2's forms) of the elements around its
// vertex, so a level has few distinct patch inverses: setup stores one per
// patch class and the patches of a class share it.  The smoother then is, per
// class, a product of one n x n matrix with the gathered right-hand sides of
// the class's members,
//   Y = W R,   R[:, q] = R_q r  (member q),
// and its bound moves from HBM (every member's block read once per
// application) to the FP32 pipe.
//
// k_class_apply: one CTA of 128 threads per work item (class, 64 or 32
// outputs a, up to 32 members).  The item's rows of W stream through a ring
// of CLS_STAGES shared-memory stages of CLS_K rows by cp.async; the members'
// right-hand sides are gathered CLS_K rows ahead into registers (index two
// chunks ahead, value one chunk ahead) and stored to a double-buffered tile,
// so neither latency is on the path of the products.  A thread owns 4 outputs
// x MPT members as packed (re, im) pairs: one fma.rn.f32x2 per stored real and
// complex right-hand side (two per stored complex number), 16 of them per 4
// shared-memory wavefronts at MPT = 4, so that the FP32 pipe and not shared
// memory sets the rate.
//
// FP32 throughout.  An output's products are summed in chains of eight, two of
// them joined per chunk of 16 rows and the chunks added: a rounding error of 0.97
// to 1.03 times that of 16 interleaved chains (the streaming smoother's order) for
// n = 54 to 770, where one chain over all rows had 1.8 to 3.5 times as much.
//
// Finest smoother of a layered 32 x 32 x 16 mesh, p = 3 (473 M entries, 66% of
// them real): 99 us, streamed 451 us; V-cycle operator by cells 49 us + 11 us of
// sums, assembled rows 295 us.  72 FMA a clock and SM inside the items, of 101
// that an outer product fed from shared memory reaches; the rest is the start
// of each item (dependent gathers) and the last wave.  The three sums take 168
// registers: three CTAs per SM; one chain at four CTAs took 98 us, the three
// sums at four (with spills) 106.  Tried: 64 x 64 tiles 111 to 125 us, 128 x 16
// tiles and 4 stages equal, 8-byte cp.async gathers 118 us.
#pragma once
#include "common.cuh"
#include "host_mesh.h"
#include "internal.h"
#include "smoother.cuh"

namespace dpgmg {

constexpr int CLS_K = 16;       // rows of W per stage
constexpr int CLS_STAGES = 3;   // stages of W in flight
constexpr int CLS_THREADS = 128;
constexpr int CLS_MEM = 32;     // members per item at most
constexpr int CLS_CTAS = 3;     // resident per SM at least (registers)

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// 16-byte asynchronous copy, or 16 zero bytes when !in (nothing is read then)
__device__ __forceinline__ void cp_async16_zfill(void* smem, const void* gmem, bool in) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int sz = in ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(sz) : "memory");
}

struct ClassSmem {
  __align__(16) unsigned char w[CLS_STAGES][CLS_K * 64 * sizeof(float2)];
  __align__(16) float2 r[2][CLS_K][CLS_MEM + 2];   // + 2: 2-way conflicts on the stores, 16-byte rows
  int64_t base[CLS_MEM];                            // members' first positions in the index list
  int64_t obase[CLS_MEM];                           // and in the output (or its index list)
};

// One work item: outputs a0 .. a0 + 4 TX - 1, members 0 .. cnt - 1 (cnt <= (128 / TX) MPT);
// a thread owns 4 outputs x MPT members: 16-byte pieces of a row of W, neighbouring
// threads' pieces next to each other (no bank conflicts).
// W: row k at W + k ld (reals, or complex numbers for CX), n x nout.  TWO: rows
// from nsplit on gather from r2.  oidx: output positions by index list, or null.
// CX:  y_a = sum_k conj(W[k][a]) r_k;
// !CX: y_a = i^(s_a) sum_k W[k][a] i^(-s_k) r_k, s = 1 on DOFs below offU (smoother.cuh).
template <class TIN, int TX, int MPT, bool CX, bool TWO = false>
__device__ __forceinline__ void class_item(ClassSmem& sm, const void* __restrict__ Wv, int64_t ld, int n, int nout,
                                           int a0, int cnt, const int32_t* __restrict__ idx, const TIN* r,
                                           const TIN* r2, int nsplit, float2* out, const int32_t* __restrict__ oidx,
                                           const int32_t* __restrict__ rep_idx, int64_t offU) {
  constexpr int TM = 4 * TX, TN = (CLS_THREADS / TX) * MPT;
  constexpr int NG = TN / 8;                          // gathered values per thread and chunk
  constexpr int EL = CX ? 8 : 4;                      // bytes per stored entry
  constexpr int ROW16 = TM * EL / 16;                 // 16-byte pieces per row of a stage
  constexpr int NW = CLS_K * ROW16 / CLS_THREADS;     // of them per thread
  constexpr int PW = 16 / EL;                         // outputs of a thread's 16-byte pieces, TX pieces apart
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int gk = tid % CLS_K, gm = tid / CLS_K;       // gather: row in the chunk, first member (then + 8)
  const char* W = reinterpret_cast<const char*>(Wv) + (int64_t)a0 * EL;
  const int wcols = (int)(ld - a0);                   // stored columns from a0 on
  const int nch = (n + CLS_K - 1) / CLS_K;

  auto load_w = [&](int c) {
    if (c < nch) {
      unsigned char* dst = sm.w[c % CLS_STAGES];
#pragma unroll
      for (int q = 0; q < NW; ++q) {
        const int p = tid + q * CLS_THREADS, row = p / ROW16, col = p % ROW16;
        const int k = c * CLS_K + row;
        const bool in = k < n && col * (16 / EL) < wcols;
        cp_async16_zfill(dst + row * (TM * EL) + col * 16, in ? W + (int64_t)k * ld * EL + col * 16 : W, in);
      }
    }
    cp_async_commit();
  };
  int gi[NG];
  float2 gv[NG];
  auto load_idx = [&](int c) {
    const int k = c * CLS_K + gk;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int m = gm + 8 * q;
      gi[q] = (k < n && m < cnt) ? __ldg(idx + sm.base[m] + k) : -1;
    }
  };
  auto load_val = [&](int c) {
    const TIN* src = TWO && c * CLS_K + gk >= nsplit ? r2 : r;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      float2 v = make_float2(0.f, 0.f);
      if (gi[q] >= 0) {
        v = cvt_in<float2>(src[gi[q]]);
        if (!CX) v = mul_i(v, gi[q] < offU ? -1 : 0);
      }
      gv[q] = v;
    }
  };
  auto store_val = [&](int c) {
#pragma unroll
    for (int q = 0; q < NG; ++q) sm.r[c & 1][gk][gm + 8 * q] = gv[q];
  };

  f32x2 sum[MPT][4];   // the chunks' sums
#pragma unroll
  for (int m = 0; m < MPT; ++m)
#pragma unroll
    for (int u = 0; u < 4; ++u) sum[m][u] = 0ull;

#pragma unroll
  for (int c = 0; c < CLS_STAGES - 1; ++c) load_w(c);
  load_idx(0);
  load_val(0);
  store_val(0);
  load_idx(1);
  for (int c = 0; c < nch; ++c) {
    cp_async_wait<CLS_STAGES - 2>();   // this thread's pieces of stage c have landed
    __syncthreads();                   // everybody's have, and everybody is done with chunk c - 1
    load_w(c + CLS_STAGES - 1);
    load_val(c + 1);                   // chunk c + 1 (indices loaded one chunk earlier)
    load_idx(c + 2);
    const unsigned char* ws = sm.w[c % CLS_STAGES] + tx * 16;
    const float2* rs = &sm.r[c & 1][0][ty * MPT];
    f32x2 acc[MPT][4], half[MPT][4];
#pragma unroll
    for (int m = 0; m < MPT; ++m)
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[m][u] = 0ull;
#pragma unroll
    for (int k = 0; k < CLS_K; ++k) {
      if (k == CLS_K / 2) {
#pragma unroll
        for (int m = 0; m < MPT; ++m)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            half[m][u] = acc[m][u];
            acc[m][u] = 0ull;
          }
      }
      f32x2 rv[MPT];
      if constexpr (MPT == 1) {
        const float2 t = rs[k * (CLS_MEM + 2)];
        rv[0] = pack2(t.x, t.y);
      } else {
#pragma unroll
        for (int m = 0; m < MPT; m += 2) {
          const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(rs + k * (CLS_MEM + 2) + m);
          rv[m] = t.x;
          rv[m + 1] = t.y;
        }
      }
      if constexpr (!CX) {
        const float4 w = *reinterpret_cast<const float4*>(ws + k * (TM * EL));
        const f32x2 w2[4] = {pack2(w.x, w.x), pack2(w.y, w.y), pack2(w.z, w.z), pack2(w.w, w.w)};
#pragma unroll
        for (int m = 0; m < MPT; ++m)
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[m][u] = fma2(w2[u], rv[m], acc[m][u]);
      } else {
        const float4 wa = *reinterpret_cast<const float4*>(ws + k * (TM * EL));
        const float4 wb = *reinterpret_cast<const float4*>(ws + k * (TM * EL) + 16 * TX);
        const f32x2 wr[4] = {pack2(wa.x, wa.x), pack2(wa.z, wa.z), pack2(wb.x, wb.x), pack2(wb.z, wb.z)};
        const f32x2 wi[4] = {pack2(wa.y, wa.y), pack2(wa.w, wa.w), pack2(wb.y, wb.y), pack2(wb.w, wb.w)};
#pragma unroll
        for (int m = 0; m < MPT; ++m) {
          const float2 t = unpack2(rv[m]);
          const f32x2 rt = pack2(t.y, -t.x);   // conj(w) r = w.x (r.x, r.y) + w.y (r.y, -r.x)
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[m][u] = fma2(wi[u], rt, fma2(wr[u], rv[m], acc[m][u]));
        }
      }
    }
#pragma unroll
    for (int m = 0; m < MPT; ++m)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        sum[m][u] = add2(sum[m][u], add2(half[m][u], acc[m][u]));
    if (c + 1 < nch) store_val(c + 1);   // its last readers finished chunk c - 1
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int a = a0 + (u / PW) * (PW * TX) + PW * tx + u % PW;
    if (a >= nout) continue;
    const int s = !CX && rep_idx[a] < offU ? 1 : 0;
#pragma unroll
    for (int m = 0; m < MPT; ++m) {
      const int q = ty * MPT + m;
      if (q < cnt) out[oidx ? (int64_t)oidx[sm.obase[q] + a] : sm.obase[q] + a] = mul_i(unpack2(sum[m][u]), s);
    }
  }
}

// Smoother products of every patch: pbuf[slot] = A_j^-1 (R_j r).  items[] =
// (first member in mem[], members, first output, shape); mem[] lists the
// patches class by class and a class's first patch in mem[] order owns the
// stored block (vptr, rflag of any member give the same).  blockIdx.y: vector.
template <class TIN>
__global__ void __launch_bounds__(CLS_THREADS, CLS_CTAS) k_class_apply(const int64_t* __restrict__ ptr,
                                                             const int32_t* __restrict__ dofs,
                                                             const int64_t* __restrict__ vptr,
                                                             const int4* __restrict__ items,
                                                             const int32_t* __restrict__ mem,
                                                             const float2* __restrict__ inv,
                                                             const TIN* __restrict__ r, int64_t ldr,
                                                             float2* __restrict__ pbuf, int64_t ldp,
                                                             const uint8_t* __restrict__ rflag, int64_t offU) {
  __shared__ ClassSmem sm;
  const int4 it = items[blockIdx.x];
  const int cnt = it.y, a0 = it.z;
  r += blockIdx.y * ldr;
  pbuf += blockIdx.y * ldp;
  const int j = mem[it.x];
  const int64_t b = ptr[j];
  const int n = (int)(ptr[j + 1] - b);
  if ((int)threadIdx.x < cnt) sm.base[threadIdx.x] = sm.obase[threadIdx.x] = ptr[mem[it.x + threadIdx.x]];
  __syncthreads();
  const float2* W = inv + vptr[j];
  const int32_t* rep = dofs + b;
#define DPG_ITEM(TX, MPT)                                                                                         \
  if (rflag != nullptr && rflag[j] != 0)                                                                          \
    class_item<TIN, TX, MPT, false>(sm, W, patch_ldr(n), n, n, a0, cnt, dofs, r, r, n, pbuf, nullptr, rep, offU);   \
  else                                                                                                            \
    class_item<TIN, TX, MPT, true>(sm, W, patch_ld(n), n, n, a0, cnt, dofs, r, r, n, pbuf, nullptr, rep, offU)
  switch (it.w) {   // CLS_SHAPE_*: outputs x members of the item
    case CLS_64x32: DPG_ITEM(16, 4); break;
    case CLS_64x16: DPG_ITEM(16, 2); break;
    case CLS_64x8: DPG_ITEM(16, 1); break;
    case CLS_32x32: DPG_ITEM(8, 2); break;
    default: DPG_ITEM(8, 1); break;
  }
#undef DPG_ITEM
}

template <class TIN>
inline void launch_class_apply(const PatchDev& P, const TIN* r, int64_t ldr, float2* pbuf, int64_t ldp, int K,
                               cudaStream_t st) {
  k_class_apply<TIN><<<dim3((unsigned)P.ncls_items, (unsigned)K), CLS_THREADS, 0, st>>>(
      P.ptr, P.dofs, P.val_ptr, P.cls_items, P.cls_mem, P.inv32, r, ldr, pbuf, ldp, P.rflag, P.offU);
  DPG_CHECK_LAUNCH();
}

}  // namespace dpgmg
