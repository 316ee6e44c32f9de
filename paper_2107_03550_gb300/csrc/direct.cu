// History convolution A^X_n = sum_j w^X_{n,j} H^X_n (Sec. 3.1, Sec. 3.3 step
// (2)) as a stream through registers: the default form of the sweep.
//
// What bounds it: the bytes of the rings (16 B per slot FP32, 32 B FP64, each
// read once) and, where weights are streamed, of the weights; in FP64 the
// FP64 pipe (4 FMA per slot at about 2 per clock and SM) is nearly as long.
//
// Layout: the rings are cut into items of consecutive lags of one mode
// (DirectItem, one 64-byte record that holds every static quantity the warp
// needs).  One warp takes one item at a time, items handed out in strides of
// the whole grid, so neighbouring items (of like length) run side by side on
// different SMs and the last round is short.  A warp loads direct_rows() rows of 32
// slots into registers with independent 128-bit (FP64: 256-bit) loads, then
// forms their products; the record and the ring head of its next item are
// brought into L1 ahead.  Nothing is
// shared between warps but the weight table, so a short window costs one
// batch and one warp reduction, not a CTA barrier: with bulk copies into
// shared memory and a CTA per chunk (k_sweep) most chunks of the short
// high-mode windows left their stage a third full and paid the barrier and
// the CTA reduction each.
//
// Weights (FP32): every mode's weights come from the table, per lag: s = (j +
// 1/2) ds in units of the piece width as two floats, the nearest piece, a
// degree-4 polynomial in the offset, with the constant as two floats so that
// the weight is rounded once, as a stored one is.  Against 64 bits over all
// lags (N = 32768 to 262144, k_c L = 120 to 300, r = 0.58): rms 2.59e-8 of the
// weights' (stored 2.58e-8; with a constant of one float, whose rounding all
// lags of a piece share, 3.6e-8), largest 4.4e-8 of max|C| (3.8e-8; 7.7e-8);
// the table itself is within 4e-9 (2.6 to 3.9e-9 with dt's own rounding).
// About 39 instructions per 32 lags, 38 % of the issue slots, where streaming
// the weights costs half the ring bytes again (N = 262144: 804 against 1093
// us).  Degree 5 on pieces twice as wide (one more 128-bit table read per lag;
// the L1 data path is 70 % busy) took 830 us.
// FP64, the exact quadrature and windows past the table stream the weights.
//
// Sums: FP32 products in a lane, batches folded into a compensated sum
// (two_sum_add), one reduction tree per item, the items of one mode added in
// FP64 in a fixed order.  Results depend on the item table only, not on the
// grid.
#include <cuda_runtime.h>

#include <cstdint>

#include "device.cuh"
#include "internal.h"
#include "kernels.cuh"

namespace sbiem {

namespace {

// One CTA of 16 warps per SM (one copy of the weight table), in 88 registers a
// thread: 20,000 registers, the threads and the rest of the shared
// memory stay free for the passes that run beside the next step's sweep.  A
// second CTA would not fit, so a grid of one CTA per SM cannot pile up on the
// SMs that the pass before it left free (two 256-thread CTAs did: FP64 steps
// at N = 65536 of 850 instead of 590 us).  Filling the registers (20 warps of
// 96) made the sweep alone 2 % faster at N = 262144 and the step 12 % slower.
constexpr int kDirectThreads = 512;
constexpr int kDirectWarps = kDirectThreads / 32;
constexpr int kDirectRegs = 88;
constexpr int kBatchCarveout = 72;  // the ensemble's cluster passes need up to 74 KB a CTA
constexpr int kFinishThreads = 256;
constexpr int kFinishWarps = kFinishThreads / 32;

// Rows of 32 slots per batch, in groups whose registers are refilled together.
template <class R> __host__ __device__ constexpr int direct_rows() { return sizeof(R) == 8 ? 4 : 8; }
template <class R> __host__ __device__ constexpr int direct_group() { return sizeof(R) == 8 ? 2 : 4; }

struct Acc32 {
  float2 t, n;
};
struct Acc64 {
  double2 t, n;
};
template <class R> struct AccT;
template <> struct AccT<float> { using T = Acc32; };
template <> struct AccT<double> { using T = Acc64; };

// Ring slots are read once: they bypass L1 allocation (the table and the
// item records stay there).
__device__ __forceinline__ float4 ld_ring(const float4* p) {
  float4 v;
  asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p));
  return v;
}
__device__ __forceinline__ Slot64 ld_ring(const Slot64* p) {
  Slot64 v;
  asm("ld.global.nc.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];"
      : "=d"(v.t.x), "=d"(v.t.y), "=d"(v.n.x), "=d"(v.n.y)
      : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ld_w(const float2* p) { return __ldg(p); }
__device__ __forceinline__ double2 ld_w(const double2* p) { return __ldg(p); }

__device__ __forceinline__ void direct_fma(Acc32& a, const float4& s, const float2 w) {
  a.t = ffma2(make_float2(w.x, w.x), make_float2(s.x, s.y), a.t);
  a.n = ffma2(make_float2(w.y, w.y), make_float2(s.z, s.w), a.n);
}
__device__ __forceinline__ void direct_fma(Acc64& a, const Slot64& s, const double2 w) {
  a.t.x = fma(w.x, s.t.x, a.t.x);
  a.t.y = fma(w.x, s.t.y, a.t.y);
  a.n.x = fma(w.y, s.n.x, a.n.x);
  a.n.y = fma(w.y, s.n.y, a.n.y);
}

// (w^T, w^N) at lag jf - 1/2 from the table in shared memory (P pieces): dh
// + dl is ds over the piece width.  The lower part of the constant, its shift
// out of the top coefficient's word included, is three instructions of about
// 39: N = 262144 steps 922 -> 928 us, N = 65536 211 -> 213 us.
__device__ __forceinline__ float2 table_weight(const float4* __restrict__ tab, int P, float jf, float dh, float dl) {
  constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer
  const float g = fmaf(jf, dh, kMagic);
  const float u = fmaf(jf, dl, fmaf(jf, dh, kMagic - g));  // kMagic - g is exact, |u| about 1/2 at most
  const int q = __float_as_int(g) - __float_as_int(kMagic);
  const float4 g0 = tab[q], g1 = tab[P + q];
  const float2 g2 = reinterpret_cast<const float2*>(tab + 2 * P)[q];
  const float2 uu = make_float2(u, u);
  // g2: the top coefficient, with the lower part of the constant in its lower half
  float2 w = ffma2(g2, uu, make_float2(g1.z, g1.w));
  w = ffma2(w, uu, make_float2(g1.x, g1.y));
  w = ffma2(w, uu, make_float2(g0.z, g0.w));
  w = ffma2(w, uu, make_float2(__uint_as_float(__float_as_uint(g2.x) << 16),
                               __uint_as_float(__float_as_uint(g2.y) << 16)));
  return fadd2(w, make_float2(g0.x, g0.y));  // the one rounding of the weight's size
}

// Float4s of the table: two per piece and a float2.
__host__ __device__ constexpr int table_f4(int P) { return 2 * P + (P + 1) / 2; }

template <class R>
__device__ __forceinline__ DirectItem<R> ld_item(const DirectItem<R>* p) {
  static_assert(sizeof(DirectItem<R>) == 64, "four 16-byte loads");
  union {
    int4 q[4];
    DirectItem<R> it;
  } u;
  const int4* s = reinterpret_cast<const int4*>(p);
#pragma unroll
  for (int k = 0; k < 4; ++k) u.q[k] = __ldg(s + k);
  return u.it;
}

// Bring a line into L1 ahead of its use.
__device__ __forceinline__ void touch(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// The weight table into shared memory (40 bytes a piece), by every thread of
// the CTA; table_wait() before the first use.
__device__ __forceinline__ float4* table_smem() {
  extern __shared__ __align__(16) unsigned char direct_smem[];
  return reinterpret_cast<float4*>(direct_smem);
}
__device__ __forceinline__ void table_start(const float4* __restrict__ wtab, int P) {
  const uint32_t dst = smem_u32(table_smem());
  const int n = table_f4(P);
  for (int i = threadIdx.x; i < n; i += kDirectThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(wtab + i) : "memory");
}
__device__ __forceinline__ void table_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}

// The items of this warp; every thread of the CTA calls it (GEN: the table is
// staged here, behind the first loads).  The rows of a batch are consumed in
// two halves, and each half's registers are refilled at once with the next
// batch's rows, of the next item where this one ends: half a batch to a whole
// one is in flight throughout.  The records of the items ahead and their ring
// heads are brought into L1 one item early each.  BATCH: sums of a
// single-item mode go to its member's arrays (BT/BN when ahead), else to
// outT/outN (and o32T/o32N unless null).  Modes of several items leave their
// sums in partial.
template <class R, bool GEN, bool BATCH>
__device__ __forceinline__ void direct_items(const DirectItem<R>* __restrict__ items, int nitems, int m,
                                             double* __restrict__ partial, const DevFault<R>* __restrict__ fs,
                                             bool ahead, double2* outT, double2* outN, float2* o32T, float2* o32N,
                                             const float4* __restrict__ wtab, int P) {
  constexpr int U = direct_rows<R>(), G = direct_group<R>();
  if constexpr (GEN) table_start(wtab, P);
  const int lane = threadIdx.x & 31;
  const int W = gridDim.x * kDirectWarps;
  int k = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const bool any = k < nitems;
  Slot<R> v[U];
  W2<R> wv[GEN ? 1 : U];
  // load cursor: the ring (and weights) of the item whose rows are loaded
  // next, its head, the batch's first slot and the end
  const Slot<R>* lring = nullptr;
  const W2<R>* lw = nullptr;
  int lh = 0, lR = 0, li = 0, lend = 0;
  auto aim = [&](const DirectItem<R>& it, int head) {
    lring = static_cast<const Slot<R>*>(it.ring);
    if constexpr (!GEN) lw = it.w + m;
    lh = head;
    lR = it.Rn;
    li = it.i0;
    lend = min(it.i1, it.Rn + 1 - m);
  };
  auto rows = [&](int g) {
    if (li >= lend) return;
    int s0 = lh + li;
    if (s0 >= lR) s0 -= lR;
    if (li + 32 * U <= lend && s0 + 32 * U <= lR) {
      const Slot<R>* p = lring + s0 + lane;
#pragma unroll
      for (int u = 0; u < G; ++u) v[g * G + u] = ld_ring(p + 32 * (g * G + u));
      if constexpr (!GEN) {
        const W2<R>* pw = lw + (li + lane);
#pragma unroll
        for (int u = 0; u < G; ++u) wv[g * G + u] = ld_w(pw + 32 * (g * G + u));
      }
    } else {
      // the end of the item or the ring's wrap: slots past the end repeat the last
#pragma unroll
      for (int u = 0; u < G; ++u) {
        if (li + 32 * (g * G + u) >= lend) break;
        const int i = min(li + 32 * (g * G + u) + lane, lend - 1);
        int s = lh + i;
        if (s >= lR) s -= lR;
        v[g * G + u] = ld_ring(lring + s);
        if constexpr (!GEN) wv[g * G + u] = ld_w(lw + i);
      }
    }
  };
  // the item being summed: lags [jc, jend), its windows, step, mode
  int jc = 0, jend = 0, mt = 0, mn = 0, mode = 0, count = 0, member = 0;
  float dh = 0.f, dl = 0.f;
  auto take = [&](const DirectItem<R>& it) {
    jc = m + it.i0;
    jend = min(it.i1, it.Rn + 1 - m) + m;
    mt = it.mt;
    mn = it.mn;
    mode = it.mode;
    count = it.count;
    member = it.member;
    dh = it.dh;
    dl = it.dl;
  };
  if (any) {
    const DirectItem<R> it = ld_item(items + k);
    aim(it, *it.head);
#pragma unroll
    for (int g = 0; g < U / G; ++g) rows(g);
    take(it);
    if (k + W < nitems) touch(items[k + W].head);
    if (k + 2 * W < nitems) touch(items + k + 2 * W);
  }
  if constexpr (GEN) table_wait();
  if (!any) return;
  const float4* tab = table_smem();
  typename AccT<R>::T run{}, cmp{};
  for (;;) {
    const bool last = jend - jc <= 32 * U;
    if (!last) {
      li += 32 * U;
    } else if (k + W < nitems) {
      const DirectItem<R> nx = ld_item(items + k + W);
      aim(nx, *nx.head);
    } else {
      li = lend;
    }
    const bool whole = min(jend, min(mt, mn)) - jc >= 32 * U;
    // the lane's first lag, converted once: lags stay below 2^23, so adding the row and 1/2 is exact
    const float jl = static_cast<float>(jc + lane);
    typename AccT<R>::T acc{};
    if constexpr (sizeof(R) == 8) acc = run;
#pragma unroll
    for (int g = 0; g < U / G; ++g) {
      if (whole) {
#pragma unroll
        for (int u = g * G; u < g * G + G; ++u) {
          W2<R> w;
          if constexpr (GEN) w = table_weight(tab, P, jl + (32.0f * u + 0.5f), dh, dl);
          else w = wv[u];
          direct_fma(acc, v[u], w);
        }
      } else {
#pragma unroll
        for (int u = g * G; u < g * G + G; ++u) {
          if (32 * u + lane < jend - jc) {
            const int j = jc + 32 * u + lane;
            W2<R> w;
            if constexpr (GEN) w = table_weight(tab, P, jl + (32.0f * u + 0.5f), dh, dl);
            else w = wv[u];
            if (j >= mt) w.x = R(0);
            if (j >= mn) w.y = R(0);
            direct_fma(acc, v[u], w);
          }
        }
      }
      rows(g);
    }
    if constexpr (sizeof(R) == 8) {
      run = acc;  // an FP64 sum needs no folding
    } else {
      two_sum_add(run.t.x, cmp.t.x, acc.t.x);
      two_sum_add(run.t.y, cmp.t.y, acc.t.y);
      two_sum_add(run.n.x, cmp.n.x, acc.n.x);
      two_sum_add(run.n.y, cmp.n.y, acc.n.y);
    }
    if (!last) {
      jc += 32 * U;
      continue;
    }
    if constexpr (sizeof(R) == 4) {
      run.t.x += cmp.t.x;
      run.t.y += cmp.t.y;
      run.n.x += cmp.n.x;
      run.n.y += cmp.n.y;
    }
    const R sum = warp_reduce4<R>(run.t.x, run.t.y, run.n.x, run.n.y);
    if ((lane & 7) == 0) {
      const int c = lane >> 3;  // 0, 1: shear re, im; 2, 3: normal re, im
      const double d = static_cast<double>(sum);
      if (count > 1) {
        partial[4 * static_cast<int64_t>(k) + c] = d;
      } else {
        const int at = 2 * mode + (c & 1);
        double2* oT = outT;
        double2* oN = outN;
        float2* fT = o32T;
        float2* fN = o32N;
        if constexpr (BATCH) {
          const DevFault<R>& f = fs[member];
          oT = ahead ? f.BT : f.AT;
          oN = ahead ? f.BN : f.AN;
          fT = ahead ? nullptr : f.AT32;
          fN = ahead ? nullptr : f.AN32;
        }
        reinterpret_cast<double*>(c < 2 ? oT : oN)[at] = d;
        if (fT) reinterpret_cast<float*>(c < 2 ? fT : fN)[at] = static_cast<float>(d);
      }
    }
    k += W;
    if (k >= nitems) break;
    run = typename AccT<R>::T{};
    cmp = typename AccT<R>::T{};
    take(ld_item(items + k));
    if (k + W < nitems) touch(items[k + W].head);
    if (k + 2 * W < nitems) touch(items + k + 2 * W);
  }
}

template <class R, bool GEN>
__global__ void __maxnreg__(kDirectRegs)
    k_direct(const DirectItem<R>* __restrict__ items, int nitems, int m, double* __restrict__ partial,
             double2* outT, double2* outN, float2* o32T, float2* o32N, const float4* __restrict__ wtab, int P,
             const unsigned* status) {
  // a pass running beside this launch may set the status word: one decision per CTA
  if (__syncthreads_or(*status != 0u)) return;
  direct_items<R, GEN, false>(items, nitems, m, partial, nullptr, false, outT, outN, o32T, o32N, wtab, P);
  // only now may the finish start: its CTAs, waiting on the device from the
  // start of the sweep, held every register the passes beside it need (steps
  // at N = 262144 1007 instead of 886 us)
  pdl_trigger();
}

// Sum of one mode's items [first, first + count) by a warp: lanes stride over
// the items, FP64, fixed order; lane 8 q returns value q.
__device__ __forceinline__ double sum_items(const double* partial, int first, int count) {
  const int lane = threadIdx.x & 31;
  double4 a = make_double4(0.0, 0.0, 0.0, 0.0);
  for (int q = lane; q < count; q += 32) {
    const double2* p = reinterpret_cast<const double2*>(partial + 4 * static_cast<int64_t>(first + q));
    const double2 lo = __ldcg(p), hi = __ldcg(p + 1);  // L2: other CTAs of the same grid wrote them (persistent form)
    a.x += lo.x;
    a.y += lo.y;
    a.z += hi.x;
    a.w += hi.y;
  }
  return warp_reduce4<double>(a.x, a.y, a.z, a.w);
}

// Modes of several items (runs[t]: mode, first item, count): one warp each.
template <class R>
__global__ void __launch_bounds__(kFinishThreads)
    k_direct_finish(const DirectRun* __restrict__ runs, int nruns, const double* partial, double2* outT, double2* outN,
                    float2* o32T, float2* o32N, const unsigned* status) {
  const int t = (blockIdx.x * kFinishThreads + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const DirectRun r = t < nruns ? runs[t] : DirectRun{};
  pdl_wait();
  if (t >= nruns) return;
  // one read per warp: a pass running beside this launch may set the word
  if (__shfl_sync(0xffffffffu, lane == 0 ? *status : 0u, 0)) return;
  const double d = sum_items(partial, r.first, r.count);
  if ((lane & 7) == 0) {
    const int c = lane >> 3, at = 2 * r.mode + (c & 1);
    reinterpret_cast<double*>(c < 2 ? outT : outN)[at] = d;
    if (o32T) reinterpret_cast<float*>(c < 2 ? o32T : o32N)[at] = static_cast<float>(d);
  }
}

// The ensemble's runs r by a warp.
template <class R>
__device__ __forceinline__ void finish_run(const DevFault<R>* __restrict__ fs, const DirectRun& r,
                                           const double* partial, bool ahead) {
  const DevFault<R>& f = fs[r.member];
  const double d = sum_items(partial, r.first, r.count);
  const int lane = threadIdx.x & 31;
  if ((lane & 7) == 0) {
    const int c = lane >> 3, at = 2 * r.mode + (c & 1);
    double2* o = ahead ? (c < 2 ? f.BT : f.BN) : (c < 2 ? f.AT : f.AN);
    reinterpret_cast<double*>(o)[at] = d;
    if (!ahead && f.AT32) reinterpret_cast<float*>(c < 2 ? f.AT32 : f.AN32)[at] = static_cast<float>(d);
  }
}

template <class R, bool GEN>
__global__ void __maxnreg__(kDirectRegs)
    k_direct_b(const DevFault<R>* __restrict__ fs, const DirectItem<R>* __restrict__ items, int nitems, int m,
               double* __restrict__ partial, bool ahead, const float4* __restrict__ wtab, int P) {
  direct_items<R, GEN, true>(items, nitems, m, partial, fs, ahead, nullptr, nullptr, nullptr, nullptr, wtab, P);
}

template <class R>
__global__ void __launch_bounds__(kFinishThreads)
    k_direct_finish_b(const DevFault<R>* __restrict__ fs, const DirectRun* __restrict__ runs, int nruns,
                      const double* partial, bool ahead) {
  const int t = (blockIdx.x * kFinishThreads + threadIdx.x) >> 5;
  const DirectRun r = t < nruns ? runs[t] : DirectRun{};
  pdl_wait();
  if (t < nruns) finish_run<R>(fs, r, partial, ahead);
}

// Sweep, grid barrier, sums of the modes of several items, in one cooperative
// launch (the barrier of k_sweep_persist).
template <class R, bool GEN>
__global__ void __maxnreg__(kDirectRegs)
    k_direct_persist(const DevFault<R>* __restrict__ fs, const DirectItem<R>* __restrict__ items, int nitems, int m,
                     double* __restrict__ partial, bool ahead, const float4* __restrict__ wtab, int P,
                     const DirectRun* __restrict__ runs, int nruns, const SweepBarrier bar) {
  __shared__ unsigned s_epoch;
  if (threadIdx.x == 0) s_epoch = *reinterpret_cast<volatile unsigned*>(bar.epoch);
  direct_items<R, GEN, true>(items, nitems, m, partial, fs, ahead, nullptr, nullptr, nullptr, nullptr, wtab, P);
  if (!grid_barrier<R>(fs, bar, s_epoch)) return;
  for (int t = (blockIdx.x * kDirectThreads + threadIdx.x) >> 5; t < nruns;
       t += gridDim.x * kDirectWarps)
    finish_run<R>(fs, runs[t], partial, ahead);
}

size_t direct_smem_bytes(int P) { return static_cast<size_t>(table_f4(P)) * sizeof(float4); }

// Opt into the table's shared memory and set the carve-out.
template <class K> void configure_one(K kernel, bool table, int carveout) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa{};
  cudaFuncGetAttributes(&fa, kernel);
  if (table)
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         optin - static_cast<int>(fa.sharedSizeBytes));
  cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, carveout);
}

template <class... Args>
void launch(void (*kernel)(Args...), int grid, int threads, size_t smem, cudaStream_t st, bool early, bool coop, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  if (early) {
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
  } else if (coop) {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = early || coop ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Few items: spread over the SMs, one warp each, before a CTA gets a second
// (the sums are waited for); ahead of the next step, beside the passes, on as
// few SMs as hold them.
int grid_for(int grid, int n, bool ahead) {
  const int need = ahead ? (n + kDirectWarps - 1) / kDirectWarps : n;
  return grid < need ? grid : need;
}

}  // namespace

template <class R>
void configure_direct() {
  configure_one(k_direct<R, false>, false, kDirectCarveout);
  configure_one(k_direct_b<R, false>, false, kBatchCarveout);
  configure_one(k_direct_persist<R, false>, false, kBatchCarveout);
  if constexpr (sizeof(R) == 4) {
    configure_one(k_direct<R, true>, true, kDirectCarveout);
    configure_one(k_direct_b<R, true>, true, kBatchCarveout);
    configure_one(k_direct_persist<R, true>, true, kBatchCarveout);
  }
}

template <class R>
int direct_blocks_per_sm(bool gen, int P, bool persist) {
  int n = 0;
  auto ask = [&](auto kernel, size_t smem) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kDirectThreads, smem);
  };
  if constexpr (sizeof(R) == 4) {
    if (gen) {
      if (persist) ask(k_direct_persist<R, true>, direct_smem_bytes(P));
      else ask(k_direct<R, true>, direct_smem_bytes(P));
      return n;
    }
  }
  if (persist) ask(k_direct_persist<R, false>, 0);
  else ask(k_direct<R, false>, 0);
  return n;
}

template <class R>
void launch_direct(const DirectTable<R>& t, const DevFault<R>& f, int m, int grid, bool ahead, cudaStream_t st,
                   cudaEvent_t swept) {
  if (t.nitems == 0) {
    if (swept) cudaEventRecord(swept, st);  // no history (the quasi-dynamic limit)
    return;
  }
  double2* oT = ahead ? f.BT : f.AT;
  double2* oN = ahead ? f.BN : f.AN;
  float2* fT = ahead ? nullptr : f.AT32;
  float2* fN = ahead ? nullptr : f.AN32;
  double* part = reinterpret_cast<double*>(f.partial);
  auto go = [&](auto gen) {
    constexpr bool GEN = decltype(gen)::value;
    launch(k_direct<R, GEN>, grid_for(grid, t.nitems, ahead), kDirectThreads, GEN ? direct_smem_bytes(t.pieces) : 0, st, false,
           false, t.items, t.nitems, m, part, oT, oN, fT, fN, t.wtab, t.pieces,
           static_cast<const unsigned*>(f.status));
  };
  if constexpr (sizeof(R) == 4) {
    if (t.wtab) go(std::true_type{});
    else go(std::false_type{});
  } else {
    go(std::false_type{});
  }
  if (swept) cudaEventRecord(swept, st);
  if (t.nruns > 0)
    launch(k_direct_finish<R>, (t.nruns + kFinishWarps - 1) / kFinishWarps, kFinishThreads, 0, st, true, false, t.runs,
           t.nruns, static_cast<const double*>(part), oT, oN, fT, fN, static_cast<const unsigned*>(f.status));
}

template <class R>
void launch_direct_batch(const DirectTable<R>& t, const DevFault<R>* fs, double4* partial, int m, int grid, bool ahead,
                         bool persistent, const SweepBarrier& bar, cudaStream_t st) {
  if (t.nitems == 0) return;
  double* part = reinterpret_cast<double*>(partial);
  auto go = [&](auto gen) {
    constexpr bool GEN = decltype(gen)::value;
    const size_t sm = GEN ? direct_smem_bytes(t.pieces) : 0;
    const int g = grid_for(grid, t.nitems, ahead);
    if (persistent) {
      launch(k_direct_persist<R, GEN>, g, kDirectThreads, sm, st, false, true, fs, t.items, t.nitems, m, part, ahead, t.wtab,
             t.pieces, t.runs, t.nruns, bar);
    } else {
      launch(k_direct_b<R, GEN>, g, kDirectThreads, sm, st, false, false, fs, t.items, t.nitems, m, part, ahead, t.wtab, t.pieces);
      if (t.nruns > 0)
        launch(k_direct_finish_b<R>, (t.nruns + kFinishWarps - 1) / kFinishWarps, kFinishThreads, 0, st, true, false,
               fs, t.runs, t.nruns, static_cast<const double*>(part), ahead);
    }
  };
  if constexpr (sizeof(R) == 4) {
    if (t.wtab) go(std::true_type{});
    else go(std::false_type{});
  } else {
    go(std::false_type{});
  }
}

template void configure_direct<double>();
template void configure_direct<float>();
template int direct_blocks_per_sm<double>(bool, int, bool);
template int direct_blocks_per_sm<float>(bool, int, bool);
template void launch_direct<double>(const DirectTable<double>&, const DevFault<double>&, int, int, bool, cudaStream_t,
                                    cudaEvent_t);
template void launch_direct<float>(const DirectTable<float>&, const DevFault<float>&, int, int, bool, cudaStream_t,
                                   cudaEvent_t);
template void launch_direct_batch<double>(const DirectTable<double>&, const DevFault<double>*, double4*, int, int, bool,
                                          bool, const SweepBarrier&, cudaStream_t);
template void launch_direct_batch<float>(const DirectTable<float>&, const DevFault<float>*, double4*, int, int, bool,
                                         bool, const SweepBarrier&, cudaStream_t);

}  // namespace sbiem
