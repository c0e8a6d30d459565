// Device helpers shared by the column-line (precond.cu) and grouped-line
// (zgroup.cu) preconditioners: packed triangles, stiffness contractions,
// bulk copies with bounded waits.
#pragma once

#include "tn_internal.h"

// packed lower triangles: column c holds rows c..M-1 at zcol(M, c) + (row - c),
// M (M + 1) / 2 entries, padded to a multiple of 4 (16-byte copies)
__host__ __device__ constexpr int pad4(int v) { return ((v + 3) / 4) * 4; }
__host__ __device__ constexpr int zlp(int M) { return pad4(M * (M + 1) / 2); }
__host__ __device__ constexpr int zcol(int M, int c) { return c * M - c * (c - 1) / 2; }

// Q_ab(g, h) = sum_{alpha beta} g_alpha Y^{alpha a beta b} h_beta for a
// cubic-aligned stiffness (isotropic: c11 = l + 2m, c12 = l, c44 = m)
__device__ __forceinline__ double Qab(int a, int b, const double g[3], const double h[3], double c11,
                                      double c12, double c44) {
  if (a == b) {
    double s = c11 * g[a] * h[a];
    for (int al = 0; al < 3; ++al)
      if (al != a) s += c44 * g[al] * h[al];
    return s;
  }
  return c12 * g[a] * h[b] + c44 * g[b] * h[a];
}

// physical gradient of a basis function from its logical gradient lg
__device__ __forceinline__ void phys(const double lg[3], double ixx, double ixy, double iex, double iey,
                                     double dz, double g[3]) {
  g[0] = ixx * lg[0] + iex * lg[1];
  g[1] = ixy * lg[0] + iey * lg[1];
  g[2] = lg[2] / dz;
}

// ---- bulk (TMA) copies global -> shared, completion counted on an mbarrier
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// one lane: announce `bytes` on bar, then start the copies that deliver them
__device__ __forceinline__ void mbar_expect(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// hint: bring `bytes` at src into L2 (no completion to wait for)
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// wait for the phase with parity `par` of bar to complete; false once
// limit_ns nanoseconds have passed without it (the copy never landed).
// try_wait may suspend the thread inside the hardware until the phase
// completes, which suits the usual limits; limits under kPollNs poll with the
// non-blocking test_wait so that the limit itself is honoured.
constexpr unsigned long long kPollNs = 100000ull;
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned par, unsigned long long limit_ns) {
  const bool poll = limit_ns < kPollNs;
  unsigned long long t0 = 0;
  for (bool first = true;; first = false) {
    unsigned ok;
    if (poll)
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(smem_u32(bar)), "r"(par)
          : "memory");
    else
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(smem_u32(bar)), "r"(par)
          : "memory");
    if (ok) return true;
    if (first) t0 = global_ns();
    else if (global_ns() - t0 > limit_ns) return false;
  }
}
// after a timed-out wait: the bound given to the copies still in flight
constexpr unsigned long long kDrainNs = 2000000000ull;
__device__ __forceinline__ unsigned long long wait_limit(const TnWait *w) {
  return w ? w->limit_ns : kDefaultWaitNs;
}

// ---- programmatic dependent launch: a kernel starts while the one before it
// in the stream drains, reads only set-up data until grid_wait (which returns
// once every earlier kernel has completed), and lets the next one start as
// early as it likes
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// p once grid_wait has returned.  An earlier kernel may write *p while this
// one already runs, so *p is not read-only for the kernel's life, as a const
// __restrict__ parameter lets the compiler assume (it moved such a load above
// the wait); a pointer that the assembly returns carries no such promise.
template <typename P>
__device__ __forceinline__ P *after_wait(P *p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}

// the dynamic shared-memory opt-in of a kernel, once per device
template <typename K>
inline cudaError_t allow_smem(K kernel, size_t bytes, int &configured_device) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured_device == dev) return cudaSuccess;
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (err == cudaSuccess) configured_device = dev;
  return err;
}

// launch that may start before the kernel ahead of it in st has ended
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// 16-byte broadcast read of entries c4 .. c4 + 16/sizeof(T) - 1 of a vector
// that every lane of the warp reads at once
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  static constexpr int W = 4;
  __device__ static void load(const float *p, float *v) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
};
template <> struct Vec16<double> {
  static constexpr int W = 2;
  __device__ static void load(const double *p, double *v) {
    const double2 t = *reinterpret_cast<const double2 *>(p);
    v[0] = t.x; v[1] = t.y;
  }
};

// sum_cc A(cc) x_cc over cc < M with x read from the broadcast vector xv and
// A(cc) given by `ent` (three partial sums to shorten the dependent chain)
template <int M, typename T, typename Ent>
__device__ __forceinline__ T bcast_dot(const T *xv, Ent ent) {
  constexpr int W = Vec16<T>::W;
  T acc[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int c4 = 0; c4 < M; c4 += W) {
    T v[W];
    Vec16<T>::load(xv + c4, v);
#pragma unroll
    for (int u = 0; u < W; ++u)
      if (c4 + u < M) acc[(c4 + u) % 3] += ent(c4 + u) * v[u];
  }
  return (acc[0] + acc[1]) + acc[2];
}
