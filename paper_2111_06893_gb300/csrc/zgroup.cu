// Grouped-line block preconditioner (the default of the Krylov solves): plan
// and solve; zgfactor.cu is its set-up.  See precond.cu for the single-line
// form it extends.
#include <algorithm>
#include <cstdio>
#include <type_traits>
#include <vector>

#include "tn_device.h"
#include "tn_internal.h"
#include "tn_precond.h"
#include "tn_zgroup.h"

// device constants are per translation unit (no relocatable device code):
// this file keeps its own copy of the LGL tables
__constant__ LglTables c_lgl_zg;

cudaError_t tn_upload_lgl_zgroup(const LglTables *t) { return cudaMemcpyToSymbol(c_lgl_zg, t, sizeof(LglTables)); }

namespace {

// ---- the FP32 solve: packed slots, one launch per degree
// A group of G lines (3 G N rows per slab) is solved by a slot of G warps,
// one row per thread.  A CTA of four warps takes one pack at a time from a
// queue: one group of 4 lines, 3 + 1, 2 + 2, 2 + 1 + 1 or 1 + 1 + 1 + 1
// lines, largest packs first.  Each slot syncs with its own named barrier
// (a warp with __syncwarp) and streams its factor records through a ring of
// P stages in shared memory (bulk copies completing on one mbarrier per
// stage), so that up to P - 1 copies are in flight while one stage is used:
// small groups, whose per-slab work is short, get the deepest rings.
constexpr int kZgThreads = 128;  // four warps per CTA
constexpr int kZgMaxStages = 8;

// floats of staging per warp: two records of the largest group
// (4 lines) across the four warps of a CTA, so that six CTAs (FP32, N = 7)
// share an SM; smaller groups fit more stages in the same room
// stage buffer of a group of G lines: the larger of the forward stage
// (S_s^{-1} and the O factors of record s) and the backward stage (W_s and
// the O factors of record s + 1)
template <int N, int G>
__host__ __device__ constexpr int zp_stage() {
  return (zlp(3 * G * N) > 3 * G * N * zp_ws(G) ? zlp(3 * G * N) : 3 * G * N * zp_ws(G)) + 8 * 3 * G * N;
}
template <int N>
__host__ __device__ constexpr int zp_stage_per_warp() {
  return pad4((zp_stage<N, 4>() * 2 + 3) / 4);
}
template <int N>
constexpr size_t zp_smem() {
  return (4 * (size_t)zp_stage_per_warp<N>() + 4 * kZgThreads) * sizeof(float) + 4 * kZgMaxStages * 8;
}

// barrier of a slot of G > 1 warps starting at warp w0 of its CTA (0, or 2 of
// the second of two pairs).  Immediate barrier numbers: a number in a register
// claims all 16 of the CTA.  Slots of 3 and 4 warps start at 0: a test of w0
// at each of their barriers, two a slab, cost the batches 1 to 3 % (24 mirrors
// 212.2 -> 210.7 us, two 56.9 -> 55.4, means over memory placements).
template <int G>
__device__ __forceinline__ void slot_sync(int w0) {
  if (G == 1) __syncwarp();
  else if (G > 2 || w0 == 0) asm volatile("bar.sync 1, %0;\n" ::"n"(32 * G) : "memory");
  else asm volatile("bar.sync 2, %0;\n" ::"n"(32 * G) : "memory");
}
// true if p holds on any thread of the slot (and a sync)
template <int ID, int NT>
__device__ __forceinline__ bool named_any(bool p) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred q, o;\n setp.ne.u32 q, %1, 0;\n bar.red.or.pred o, %2, %3, q;\n selp.u32 %0, 1, 0, o;\n}\n"
      : "=r"(r)
      : "r"((unsigned)p), "n"(ID), "n"(NT)
      : "memory");
  return r != 0;
}
template <int G>
__device__ __forceinline__ bool slot_any(int w0, bool p) {
  if (G == 1) return __any_sync(0xffffffffu, p);
  return G > 2 || w0 == 0 ? named_any<1, 32 * G>(p) : named_any<2, 32 * G>(p);
}
__device__ __forceinline__ void mbar_inval(unsigned long long *bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// three warp-wide sums at once: the three butterflies interleaved level by
// level, so that their shuffles overlap instead of running one sum after
// the other (every lane gets the three sums)
__device__ __forceinline__ void warp_allsum3(float &a, float &b, float &c) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float a2 = __shfl_xor_sync(0xffffffffu, a, o);
    const float b2 = __shfl_xor_sync(0xffffffffu, b, o);
    const float c2 = __shfl_xor_sync(0xffffffffu, c, o);
    a += a2;
    b += b2;
    c += c2;
  }
}

// z = A_GG^{-1} r on group grp by the slot of G warps starting at warp w0;
// line li of the group is warp w0 + li, its rows (a, k) lanes a N + k < 3N:
//   forward   y_s = Linv_s (r_s - O_{s-1}^T w_{s-1}),  w_s = Linv_s^T y_s
//   backward  x_s = Linv_s^T (y_s - Linv_s O_s x_{s+1}) = w_s - W_s v_{s+1}
// (v: six numbers per line, x_{s+1}(b, N - 1) and X^T x_{s+1}).  The forward
// step forms w_s = S_s^{-1} b_s, b_s = r_s - O_{s-1}^T w_{s-1}, in one
// symmetric product, and r.z = sum_s |y_s|^2 = sum_s b_s . w_s.  O in its
// factored form acts line by line (it is block diagonal over the lines), so
// its products are warp shuffles and warp sums; S_s^{-1} b_s and W_s v cross
// lines, through broadcast vectors in shared memory (double-buffered by step
// parity).  Stage u < S: S_u^{-1} and the O factors of record u; stage u >= S:
// W_s of record s and the O factors of record s + 1, s = 2S - 2 - u.  Stage u
// uses ring buffer u % P and mbarrier u % P with phase parity (u / P) & 1.
// Writes the group's partial r.z (= |y|^2) and r.r.  A wait that runs
// out sets err->flag and ends the slot after bounded waits for the copies in
// flight.
template <int N, int G>
__device__ __forceinline__ void zp_slot(int grp, int w0, int mncol, int S, const float *__restrict__ r,
                                        float *__restrict__ z, const int4 *__restrict__ glines,
                                        const long long *__restrict__ gfac, const float *__restrict__ fac,
                                        float *__restrict__ stage, int cap, float *__restrict__ vecs,
                                        unsigned long long *__restrict__ bars, double *__restrict__ psum,
                                        unsigned long long lim, TnWait *__restrict__ err, double *__restrict__ part_rz,
                                        double *__restrict__ part_rr) {
  constexpr int M = 3 * N, N2 = N * N, n = N * N * N, MG = G * M, NT = 32 * G;
  constexpr int LP = zlp(MG), RS = zp_rec(MG, G), WS = zp_ws(G), RSS = zp_stage<N, G>();
  constexpr int LPX = LP + 8 * MG;  // forward stage: S_s^{-1} and the O factors of record s
  constexpr int BW = MG * WS;       // backward stage: W_s, then the O factors of record s + 1
  const int lt = threadIdx.x - 32 * w0;
  auto sync = [&]() { slot_sync<G>(w0); };
  auto any = [&](bool p) { return slot_any<G>(w0, p); };
  const int li = lt >> 5, lane = lt & 31;
  const bool act = lane < M;
  const int t = li * M + (act ? lane : 0);  // row of the group's blocks
  const int a = (act ? lane : 0) / N, k = (act ? lane : 0) - a * N;
  // broadcast vectors hold line lj's M entries at 32 lj (16-byte aligned)
  float *const vbuf = vecs + 4 * 32 * w0;  // [2 parities][vb][32 G] (room for 2 x 2 x 32 G)
  auto vb = [&](int par) { return vbuf + par * 2 * NT; };
  const int4 L4 = glines[grp];
  const int lid = li == 0 ? L4.x : (li == 1 ? L4.y : (li == 2 ? L4.z : L4.w));
  const int c = lid / N2, qn = lid - c * N2;
  // vector entry of this row in slab s: g0 + s * gs
  const size_t gs = (size_t)mncol * 3 * n, g0 = ((size_t)c * 3 + a) * n + (size_t)k * N2 + qn;
  auto gidx = [&](int s) { return g0 + (size_t)s * gs; };
  const float *base = fac + gfac[grp];
  const int total = 2 * S;
  int P = cap / RSS;
  P = P > kZgMaxStages ? kZgMaxStages : P;
  P = P > total ? total : P;
  // stage sources: forward stage u = S_u^{-1} and O factors of record u;
  // backward stage u (slab s = 2S - 2 - u < S - 1) = W_s of record s and the
  // O factors of record s + 1 (the last slab, s = S - 1, needs no stage)
  const int total_st = 2 * S - 1;
  int issued = 0, ib = 0;  // stages issued so far and the ring buffer of the next (same in every thread)
  const float *src = base;     // lane 0: the next stage's (first) source
  auto issue_next = [&]() {
    if (issued >= total_st) return;
    const int u = issued++, b = ib;
    ib = ib + 1 == P ? 0 : ib + 1;
    if (lt == 0) {
      float *dst = stage + (size_t)b * RSS;
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      if (u < S) {
        mbar_expect(bars + b, (unsigned)(LPX * sizeof(float)));
        bulk_g2s(dst, src, (unsigned)(LPX * sizeof(float)), bars + b);
        src = u + 1 < S ? src + RS : src - RS;  // then the backward stages from record S - 2 down
      } else {
        mbar_expect(bars + b, (unsigned)((BW + 8 * MG) * sizeof(float)));
        bulk_g2s(dst, src + LPX, (unsigned)(BW * sizeof(float)), bars + b);
        bulk_g2s(dst + BW, src + RS + LP, (unsigned)(8 * MG * sizeof(float)), bars + b);
        src -= RS;
      }
    }
  };
  // the slot agrees on the outcome (a barrier of the slot): a stage counts
  // as landed only if every thread saw it land.  wb / wpar: ring buffer and
  // phase parity of the stage waited for next (stage u: u % P, (u / P) & 1)
  int wb = 0;
  unsigned wpar = 0u;
  auto wait = [&]() {
    const bool ok = !any(!mbar_wait(bars + wb, wpar, lim));
    if (G == 1) __syncwarp();  // memory order across the warp, as the named barrier gives
    return ok;
  };
  auto wait_done = [&]() {  // advance to the next stage
    if (++wb == P) {
      wb = 0;
      wpar ^= 1u;
    }
  };
  if (lt == 0) {
    for (int b = 0; b < P; ++b) mbar_init(bars + b);
    mbar_init_fence();
  }
  sync();
  for (int u = 0; u + 1 < P; ++u) issue_next();
  float rz = 0.0f, rr = 0.0f;
  bool bad = false;
  int at = 0;  // the stage being waited for
  const int pl = zcol(MG, t) - t;
  // w = S^{-1} v, line block by line block, the block index a compile-time
  // constant so that every packed offset folds: row t of the symmetric
  // S^{-1} is the stored lower triangle's row t (blocks before this thread's
  // line, and its own block up to the diagonal) followed by its column t
  // (its own block below the diagonal, and the blocks after it)
  const int tl = act ? lane : 0;  // row within the line
  auto lblock = [&](const float *Ls, const float *v, auto LJ) {
    constexpr int c0 = decltype(LJ)::value * M;
    return bcast_dot<M, float>(v + 32 * decltype(LJ)::value,
                           [&](int cc) { return Ls[zcol(MG, c0 + cc) + t - c0 - cc]; });
  };
  auto ublock = [&](const float *Ls, const float *v, auto LJ) {
    constexpr int c0 = decltype(LJ)::value * M;
    return bcast_dot<M, float>(v + 32 * decltype(LJ)::value, [&](int cc) { return Ls[pl + c0 + cc]; });
  };
  auto dblock = [&](const float *Ls, const float *v, auto LJ) {
    constexpr int c0 = decltype(LJ)::value * M;
    return bcast_dot<M, float>(v + 32 * decltype(LJ)::value, [&](int cc) {
      return cc <= tl ? Ls[zcol(MG, c0 + cc) + t - c0 - cc] : Ls[pl + c0 + cc];
    });
  };
  auto symrow = [&](const float *Ls, const float *v) {
    float acc = 0.0f;
    auto part = [&](auto LJ) {
      constexpr int J = decltype(LJ)::value;
      if (J >= G) return;
      if (J < li) acc += lblock(Ls, v, LJ);
      else if (J == li) acc += dblock(Ls, v, LJ);
      else acc += ublock(Ls, v, LJ);
    };
    part(std::integral_constant<int, 0>{});
    part(std::integral_constant<int, 1>{});
    part(std::integral_constant<int, 2>{});
    part(std::integral_constant<int, 3>{});
    return acc;
  };
  // forward sweep
  float r0 = act ? r[gidx(0)] : 0.0f;
  float r1 = (act && S > 1) ? r[gidx(1)] : 0.0f;
  float w = 0.0f;
  for (int s = 0; s < S; ++s, ++at) {
    if (!wait()) { bad = true; break; }
    const float *Ls = stage + (size_t)wb * RSS, *XY = Ls + LP + 8 * t;
    wait_done();
    issue_next();  // every thread is past step s - 1: its buffer is free
    const int par = s & 1;
    const float rv = r0;
    r0 = r1;
    if (act && s + 2 < S) r1 = r[gidx(s + 2)];
    rr += rv * rv;
    float bv = rv;
    if (s > 0) {  // bv -= (O_{s-1}^T w_{s-1})_t, line by line
      const float x0 = XY[0], x1 = XY[1], x2 = XY[2];
      float s0 = act ? XY[4] * w : 0.0f, s1 = act ? XY[5] * w : 0.0f, s2 = act ? XY[6] * w : 0.0f;
      warp_allsum3(s0, s1, s2);
      float o = x0 * __shfl_sync(0xffffffffu, w, 0) + x1 * __shfl_sync(0xffffffffu, w, N) +
            x2 * __shfl_sync(0xffffffffu, w, 2 * N);
      if (k == N - 1) o += a == 0 ? s0 : (a == 1 ? s1 : s2);
      bv -= o;
    }
    if (act) vb(par)[lt] = bv;
    sync();
    w = symrow(Ls, vb(par));  // w_s = S_s^{-1} bv = Linv_s^T y_s
    if (!act) w = 0.0f;
    rz += bv * w;             // |y_s|^2
    if (act) z[gidx(s)] = w;  // read back by the backward sweep
  }
  // backward sweep: x_{S-1} = w_{S-1} (already in z), then
  // x_s = w_s - W_s v_{s+1}, v per line: x_{s+1}(b, N - 1) and X^T x_{s+1}
  if (!bad) {
    float x = w;
    float w1 = (act && S > 1) ? z[gidx(S - 2)] : 0.0f;
    float w2 = (act && S > 2) ? z[gidx(S - 3)] : 0.0f;
    for (int s = S - 2; s >= 0; --s, ++at) {
      if (!wait()) { bad = true; break; }
      const float *Ws = stage + (size_t)wb * RSS, *XY = Ws + BW + 8 * t;
      wait_done();
      issue_next();
      const int par = s & 1;
      const float wv = w1;
      w1 = w2;
      if (act && s >= 2) w2 = z[gidx(s - 2)];
      const float e0 = __shfl_sync(0xffffffffu, x, N - 1);
      const float e1 = __shfl_sync(0xffffffffu, x, 2 * N - 1);
      const float e2 = __shfl_sync(0xffffffffu, x, 3 * N - 1);
      float c0 = act ? XY[0] * x : 0.0f, c1 = act ? XY[1] * x : 0.0f, c2 = act ? XY[2] * x : 0.0f;
      warp_allsum3(c0, c1, c2);
      if (lane < 6) vb(par)[32 * li + lane] = lane < 3 ? (lane == 0 ? e0 : (lane == 1 ? e1 : e2))
                                                      : (lane == 3 ? c0 : (lane == 4 ? c1 : c2));
      sync();
      const float *Wr = Ws + t * WS;
      float acc = 0.0f;
#pragma unroll
      for (int l = 0; l < G; ++l) {
        const float *vl = vb(par) + 32 * l;
        acc += (Wr[6 * l] * vl[0] + Wr[6 * l + 1] * vl[1] + Wr[6 * l + 2] * vl[2]) +
               (Wr[6 * l + 3] * vl[3] + Wr[6 * l + 4] * vl[4] + Wr[6 * l + 5] * vl[5]);
      }
      x = act ? wv - acc : 0.0f;
      if (act) z[gidx(s)] = x;
    }
  }
  if (bad) {  // a copy never landed: bounded waits for every copy in flight, then report
    for (int u = at; u < issued; ++u) {
      mbar_wait(bars + wb, wpar, kDrainNs);
      wait_done();
    }
    if (lt == 0 && err) atomicExch(&err->flag, 1);
  }
  // the group's partial sums, in a fixed order
  double vrz = (double)rz, vrr = (double)rr;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    vrz += __shfl_xor_sync(0xffffffffu, vrz, o);
    vrr += __shfl_xor_sync(0xffffffffu, vrr, o);
  }
  if (lane == 0) {
    psum[(w0 + li) * 2] = vrz;
    psum[(w0 + li) * 2 + 1] = vrr;
  }
  sync();
  if (lt == 0) {
    double srz = 0.0, srr = 0.0;
    for (int ww = 0; ww < G; ++ww) {
      srz += psum[(w0 + ww) * 2];
      srr += psum[(w0 + ww) * 2 + 1];
    }
    if (part_rz) part_rz[grp] = srz;
    if (part_rr) part_rr[grp] = srr;
    for (int b = 0; b < P; ++b) mbar_inval(bars + b);  // every phase issued has completed
  }
}

// The beta step of a PCG iteration folded into the grouped-line solve: once
// every CTA of all the step's launches has written its groups' r.z and r.r
// partials, the last reduces them in a fixed order (group 0 .. ngroups - 1)
// and updates beta and the stopping test.
__device__ void fold_beta(const PcgFold &f) {
  __shared__ int last;
  __shared__ double red[2][kZgThreads / 32];
  __syncthreads();  // every slot of this CTA has written its partials
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(f.cnt, 1u) == (unsigned)(f.total - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double rz = 0.0, rr = 0.0;
  for (int t = threadIdx.x; t < f.nparts; t += blockDim.x) {
    rz += __ldcg(f.part + t);
    rr += __ldcg(f.part2 + t);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rz += __shfl_xor_sync(0xffffffffu, rz, o);
    rr += __shfl_xor_sync(0xffffffffu, rr, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = rz;
    red[1][threadIdx.x >> 5] = rr;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < kZgThreads / 32; ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    pcg_finish_beta(f.s, a, b);
    *f.cnt = 0u;
    __threadfence();
  }
}

// packs [pk0, pk0 + npk) of one degree; CTAs take packs from queue[0]
// (largest first); the last CTA to finish resets queue[0..1] for the next
// launch.  One mesh (ginst == nullptr) or a batch (per group: its mirror's
// mesh and first unknown).
template <int N, int B>
__global__ void __launch_bounds__(kZgThreads, B)
zgroup_packed_kernel(const DevMesh m1, const int *__restrict__ ginst, const DevMesh *__restrict__ meshes,
                     const long long *__restrict__ dof_off, const int4 *__restrict__ glines,
                     const long long *__restrict__ gfac, const int4 *__restrict__ packs, int pk0, int npk,
                     int *__restrict__ queue, const float *__restrict__ fac, const float *__restrict__ r,
                     float *__restrict__ z, double *__restrict__ part_rz, double *__restrict__ part_rr, const int *__restrict__ done,
                     TnWait *__restrict__ err, const PcgFold fold) {
  grid_wait();
  done = after_wait(done);
  r = after_wait(r);
  queue = after_wait(queue);
  if (done && *done) return;
  constexpr int SW = zp_stage_per_warp<N>();
  extern __shared__ __align__(16) unsigned char zsm[];
  float *const stage0 = reinterpret_cast<float *>(zsm);
  float *const vecs = stage0 + 4 * SW;
  unsigned long long *const bars = reinterpret_cast<unsigned long long *>(vecs + 4 * kZgThreads);
  __shared__ int s_pk;
  __shared__ double psum[8];
  const int warp = threadIdx.x >> 5;
  const unsigned long long lim = wait_limit(err);
  for (;;) {
    if (threadIdx.x == 0) s_pk = atomicAdd(queue, 1);
    __syncthreads();
    const int pk = s_pk;
    __syncthreads();
    if (pk >= npk) break;
    const int4 P4 = packs[pk0 + pk];
    const int ent[4] = {P4.x, P4.y, P4.z, P4.w};
    int w0 = 0, grp = -1, G = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int g = ent[i];
      if (g < 0 || grp >= 0) continue;
      const int4 L = glines[g];
      const int gs = 1 + (L.y >= 0) + (L.z >= 0) + (L.w >= 0);
      if (warp >= w0 && warp < w0 + gs) {
        grp = g;
        G = gs;
      } else {
        w0 += gs;
      }
    }
    if (grp >= 0) {
      int mncol = m1.ncol, mslab = m1.nslab;
      const float *rg = r;
      float *zg = z;
      if (ginst) {
        const int in = ginst[grp];
        mncol = meshes[in].ncol;
        mslab = meshes[in].nslab;
        const long long o = dof_off[in];
        rg += o;
        zg += o;
      }
      float *stg = stage0 + (size_t)w0 * SW;
      unsigned long long *sb = bars + kZgMaxStages * w0;
      const int cap = G * SW;
      switch (G) {
        case 1:
          zp_slot<N, 1>(grp, w0, mncol, mslab, rg, zg, glines, gfac, fac, stg, cap, vecs, sb, psum,
                                lim, err, part_rz, part_rr);
          break;
        case 2:
          zp_slot<N, 2>(grp, w0, mncol, mslab, rg, zg, glines, gfac, fac, stg, cap, vecs, sb, psum,
                                lim, err, part_rz, part_rr);
          break;
        case 3:
          zp_slot<N, 3>(grp, w0, mncol, mslab, rg, zg, glines, gfac, fac, stg, cap, vecs, sb, psum,
                                lim, err, part_rz, part_rr);
          break;
        default:
          zp_slot<N, 4>(grp, w0, mncol, mslab, rg, zg, glines, gfac, fac, stg, cap, vecs, sb, psum,
                                lim, err, part_rz, part_rr);
          break;
      }
    }
    __syncthreads();  // every slot of the pack is done with shared memory
  }
  grid_trigger();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(queue + 1, 1) == (int)gridDim.x - 1) {
      queue[0] = 0;
      queue[1] = 0;
      __threadfence();
    }
  }
  if (fold.s) fold_beta(fold);
}

// ---- the FP64 solve: three launches
//   zg_slab_kernel   a_s = S_s^{-1} r_s (left in z), c_s and d_s, every slab of
//                    every group on its own
//   zg_chain_kernel  the two chains g and f of every group
//   zg_final_kernel  x_s = a_s - Q_s g_{s-1} - W_s f_{s+1}, r.z and r.r, again
//                    every slab on its own
// All three are bound by the FP64 pipe (79, 65 and 88 % busy; 189 + 107 + 100 us
// at 2.0 M unknowns, p = 6), the chains also by their dependent steps.  Loading the last launch's factors by bulk copies
// through a ring, as the first does, was slower (441 against 383 us in all:
// fewer CTAs per SM).
// `chain` holds 12 g numbers per slab: c_s, then g_s; d_s, then f_s.
constexpr int kZgChunks = 4;   // stages of slabs per CTA of the first and last launch, at most
constexpr int kZgFill = 1024;  // CTAs the first launch aims at before a CTA takes more than one stage
constexpr int kZgBlock = 32;   // slabs the chain kernel holds at a time, however many there are
constexpr int kZgKWarp = 640;  // K entries a warp stages at a time (one record of the largest group: 600)

// what the kernels need of the groups; one degree's packs and slab ranges
struct ZgView {
  const int *inst;             // batch: mirror of every group (nullptr: one mesh)
  const DevMesh *meshes;
  const long long *dof_off;
  const int4 *lines;
  const long long *fac, *chain;  // first factor and chain entry of every group
  const int4 *packs;
  const int4 *ranges;            // (group, first slab, end slab, partial sum)
};

struct ZgGroup {
  int ncol, S;
  long long off;  // first unknown of the mirror
};
__device__ __forceinline__ ZgGroup zg_where(const DevMesh &m1, const ZgView &v, int grp) {
  if (!v.inst) return {m1.ncol, m1.nslab, 0};
  const int in = v.inst[grp];
  return {v.meshes[in].ncol, v.meshes[in].nslab, v.dof_off[in]};
}
__device__ __forceinline__ int zg_line(const int4 &L, int li) { return li == 0 ? L.x : (li == 1 ? L.y : (li == 2 ? L.z : L.w)); }
__device__ __forceinline__ int zg_size(const int4 &L) { return 1 + (L.y >= 0) + (L.z >= 0) + (L.w >= 0); }

// ---- the slabs
template <int N, int G>
struct ZgSlab {
  static constexpr int M = 3 * N, MG = G * M, C6 = 6 * G, SREC = zg_srec(MG, G), QREC = zg_qrec(MG, G), MGP = pad4(MG);
  // slabs per stage: rows on the CTA's threads, room of one slab of the largest group
  static constexpr int by_rows = kZgThreads / MG, by_room = zg_srec(12 * N, 4) / SREC;
  static constexpr int SL = by_rows < 1 ? 1 : (by_rows < by_room ? by_rows : by_room);
};
int zg_slabs(int N, int G) {
  const int MG = 3 * N * G, by_rows = kZgThreads / MG, by_room = zg_srec(12 * N, 4) / zg_srec(MG, G);
  return by_rows < 1 ? 1 : std::min(by_rows, by_room);
}
// two stages, the vector twice over (rows read it at t + m), the products, two rows of D
template <int N>
constexpr size_t zg_slab_smem() { return sizeof(double) * (size_t)(2 * zg_srec(12 * N, 4) + 3 * kZgThreads + 2 * N); }

// row t of S^{-1} v from the circulant diagonals; v repeated: v[MG + i] = v[i]
template <int MG>
__device__ __forceinline__ double circ_row(const double *__restrict__ A, const double *__restrict__ v, int t) {
  constexpr int H = (MG - 1) / 2;
  const double *const At = A + t, *const vt = v + t;
  double a0 = At[0] * vt[0], a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll
  for (int m = 1; m <= H; ++m) {
    const int back = t < m ? MG : 0;
    const double f = At[m * MG], b = At[m * MG - m + back];
    if (m & 1) {
      a1 += f * vt[m];
      a2 += b * vt[MG - m];
    } else {
      a3 += f * vt[m];
      a0 += b * vt[MG - m];
    }
  }
  if (MG % 2 == 0) a1 += At[(MG / 2) * MG] * vt[MG / 2];
  return (a0 + a1) + (a2 + a3);
}

template <int N, int G>
__device__ __forceinline__ void zg_slab(const DevMesh &m1, const ZgView &v, const int4 &rg,
                                        const double *__restrict__ fac, const double *r0, double *__restrict__ z0, double *__restrict__ chain,
                                        double *__restrict__ stage, unsigned long long *bars, const int *done,
                                        TnWait *__restrict__ err) {
  using Z = ZgSlab<N, G>;
  constexpr int M = Z::M, MG = Z::MG, C6 = Z::C6, SREC = Z::SREC, SL = Z::SL, LC = pad4(zg_circ(MG));
  constexpr int N2 = N * N, n = N * N2, ROOM = zg_srec(12 * N, 4);
  static_assert(SL * MG <= kZgThreads, "rows");
  double *const vb = stage + 2 * ROOM, *const av = vb + 2 * kZgThreads, *const dl = av + kZgThreads;
  const int tid = threadIdx.x, grp = rg.x, s0 = rg.y, s1 = rg.z;
  const ZgGroup q = zg_where(m1, v, grp);
  const double *const src = fac + v.fac[grp];
  auto issue = [&](int s) {  // the stage of slabs s ..: thread 0
    const int i = (s - s0) / SL, b = i & 1;
    const unsigned bytes = (unsigned)(min(SL, s1 - s) * SREC * sizeof(double));
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    mbar_expect(bars + b, bytes);
    bulk_g2s(stage + b * ROOM, src + (size_t)s * SREC, bytes, bars + b);
  };
  if (tid == 0) {  // the factors do not depend on the launch before this one
    mbar_init(bars);
    mbar_init(bars + 1);
    mbar_init_fence();
    issue(s0);
  }
  const int sl = tid / MG, t = tid - sl * MG, li = t / M, tl = t - li * M, a = tl / N, k = tl - a * N;
  const int lid = zg_line(v.lines[grp], li), col = lid / N2, qn = lid - col * N2;
  const bool row = sl < SL;
  const size_t gs = (size_t)q.ncol * 3 * n, g0 = q.off + ((size_t)col * 3 + a) * n + (size_t)k * N2 + qn;
  double *const ch = chain + v.chain[grp];
  const unsigned long long lim = wait_limit(err);
  if (tid < 2 * N) {  // D(0, k), k != 0, and D(N-1, k), k != N - 1; zero at the face node itself
    const int kk = tid < N ? tid : tid - N;
    dl[tid] = tid == 0 || tid == 2 * N - 1 ? 0.0 : c_lgl_zg.D[N][(tid < N ? 0 : (N - 1) * N) + kk];
  }
  __syncthreads();  // the barriers are initialised
  grid_wait();
  r0 = after_wait(r0);
  done = after_wait(done);
  const bool skip = done && *done;
  double rn = row && !skip && s0 + sl < s1 ? r0[g0 + (size_t)(s0 + sl) * gs] : 0.0;
  for (int s = s0; s < s1; s += SL) {
    const int i = (s - s0) / SL, b = i & 1;
    const bool on = row && s + sl < s1;
    const bool ok = mbar_wait(bars + b, (i >> 1) & 1, lim);
    if (on) vb[sl * 2 * MG + t] = vb[sl * 2 * MG + MG + t] = rn;
    // the stage has landed, the vector is complete, the other stage is free
    if (__syncthreads_or(!ok)) {  // a copy did not land in time: a bounded wait for it, then report
      mbar_wait(bars + b, (i >> 1) & 1, kDrainNs);
      if (tid == 0 && err) atomicExch(&err->flag, 1);
      return;
    }
    if (skip) return;
    if (tid == 0 && s + SL < s1) issue(s + SL);
    if (s + SL >= s1) grid_trigger();
    rn = row && s + SL + sl < s1 ? r0[g0 + (size_t)(s + SL + sl) * gs] : 0.0;
    const double *A = stage + b * ROOM;
    if (on) {
      const double w = circ_row<MG>(A + sl * SREC, vb + sl * 2 * MG, t);
      z0[g0 + (size_t)(s + sl) * gs] = w;
      av[tid] = w;
    }
    __syncthreads();
    // c_s = U_s^T a_s and d_s = V_s^T a_s: one thread per slab, line, component and side
    constexpr int NT6 = SL * 6 * G;
    static_assert(NT6 <= kZgThreads, "one task per thread");
    if (tid < NT6) {
      const int es = tid / (6 * G), ea = tid - es * (6 * G), el = ea / 6, e6 = ea - el * 6;
      const bool bottom = e6 >= 3;  // d (the top face) or c (the bottom face, k = 0)
      const int ec = bottom ? e6 - 3 : e6;
      if (s + es < s1) {
        const double *w = av + es * MG + el * M, *C = A + es * SREC + LC + 16 * el, *wc = w + ec * N;
        const double *D = dl + (bottom ? 0 : N), *X3 = C + 6 + ec;
        double e = 0.0;
#pragma unroll
        for (int kk = 0; kk < N; ++kk) e += D[kk] * wc[kk];
        double *const o = ch + (size_t)(s + es) * 2 * C6 + 6 * el + (bottom ? 0 : C6) + ec;
        if (bottom) {
          o[0] = C[ec] * e;
          o[3] = wc[0];
        } else {
          o[0] = wc[N - 1];
          o[3] = C[3 + ec] * e + ((X3[0] * w[N - 1] + X3[3] * w[2 * N - 1]) + X3[6] * w[3 * N - 1]);
        }
      }
    }
  }
}

template <int N>
__global__ void __launch_bounds__(kZgThreads, 3)
zg_slab_kernel(const DevMesh m1, const ZgView v, const double *__restrict__ fac, const double *__restrict__ r,
               double *__restrict__ z, double *__restrict__ chain, const int *__restrict__ done,
               TnWait *__restrict__ err) {
  extern __shared__ __align__(16) unsigned char zsm[];
  __shared__ __align__(8) unsigned long long bars[2];
  double *const stage = reinterpret_cast<double *>(zsm);
  const int4 rg = v.ranges[blockIdx.x];
  switch (zg_size(v.lines[rg.x])) {
#define TN_CASE(GG) case GG: zg_slab<N, GG>(m1, v, rg, fac, r, z, chain, stage, bars, done, err); break;
    TN_CASE(1) TN_CASE(2) TN_CASE(3) TN_CASE(4)
#undef TN_CASE
  }
}

// ---- the chains: a group of G lines on G warps of a CTA of four, which takes
// a pack of groups: 4, 3 + 1, 2 + 2, 2 + 1 + 1 or 1 + 1 + 1 + 1 lines.  Slabs
// go by blocks of kZgBlock, so that shared memory does not depend on their
// number.  One warp runs the chains, the others bring K.
constexpr int kZgChLine = pad4(12 * (kZgBlock + 1));  // chain entries of a block and the slab before or after it, per line
constexpr size_t zg_chain_smem() { return sizeof(double) * 4 * (size_t)(kZgChLine + kZgKWarp); }

// the group this warp works on: its first warp w0 in the CTA, its size (0: idle)
__device__ __forceinline__ int zg_slot(const ZgView &v, int &w0, int &G) {
  const int4 P4 = v.packs[blockIdx.x];
  const int ent[4] = {P4.x, P4.y, P4.z, P4.w}, warp = threadIdx.x >> 5;
  int at = 0;
  w0 = 0;
  G = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (ent[i] < 0) continue;
    const int gs = zg_size(v.lines[ent[i]]);
    if (warp >= at && warp < at + gs) {
      w0 = at;
      G = gs;
      return ent[i];
    }
    at += gs;
  }
  return -1;
}

// K records brought through registers: load issues, store lands them
template <int G>
struct KStage {
  static constexpr int KP = zg_kpart(G), KREC = zg_krec(G), SLK = G * kZgKWarp / KP;  // slabs per stage
  static constexpr int PER = (SLK * KP + 32 * G - 1) / (32 * G);
  double v[PER];
  __device__ __forceinline__ void load(const double *__restrict__ k, int cnt, int lt) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int at = i * 32 * G + lt, s = at / KP;
      v[i] = at < cnt * KP ? k[(size_t)s * KREC + (at - s * KP)] : 0.0;
    }
  }
  __device__ __forceinline__ void store(double *__restrict__ ks, int cnt, int lt) const {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int at = i * 32 * G + lt;
      if (at < cnt * KP) ks[at] = v[i];
    }
  }
};

// lanes per row of a chain step (112 -> 105 us at 2.0 M unknowns, p = 6): the six or twelve rows of small groups leave
// lanes over, and an FP64 instruction costs the same with a few lanes on
__host__ __device__ constexpr int chain_parts(int G) { return G == 1 ? 4 : (G == 2 ? 2 : 1); }
template <int G, typename KF, typename VF>
__device__ __forceinline__ double chain_dot(double a0, KF k, VF v, int part) {
  constexpr int P = chain_parts(G), C6 = 6 * G, STEPS = (C6 + P - 1) / P;
  double a1 = 0.0, a2 = 0.0;
#pragma unroll
  for (int i = 0; i < STEPS; ++i) {
    const int j = i * P + part;
    if (C6 % P != 0 && j >= C6) break;
    (i % 3 == 0 ? a0 : (i % 3 == 1 ? a1 : a2)) -= k(j) * v(j);
  }
  a0 += a1 + a2;
#pragma unroll
  for (int o = P / 2; o > 0; o >>= 1) a0 += __shfl_xor_sync(0x00ffffffu, a0, o);  // 6 x 4 or 12 x 2 lanes
  return a0;
}

template <int G>
__device__ __forceinline__ void zg_chain(int S, int w0, const double *__restrict__ fk, double *chain,
                                         double *__restrict__ sm) {
  constexpr int C6 = 6 * G, C12 = 12 * G, LD = zg_ld(G), NT = 32 * G;
  constexpr int KP = zg_kpart(G), KREC = zg_krec(G), SLK = KStage<G>::SLK;
  const int lt = threadIdx.x - 32 * w0, row = lt / chain_parts(G), part = lt % chain_parts(G);
  double *const ch = sm, *const ks = ch + G * kZgChLine;
  const int nblk = (S + kZgBlock - 1) / kZgBlock;
  KStage<G> K;
  // forward: slabs b0 .. b0 + nb - 1 at ch[(1 + i) C12], slab b0 - 1 at ch[0]
  for (int b0 = 0; b0 < S; b0 += kZgBlock) {
    const int nb = min(kZgBlock, S - b0), k0 = max(1, b0), k1 = min(b0 + nb, S - 1);  // steps k0 .. k1 - 1
    K.load(fk + (size_t)k0 * KREC, min(SLK, k1 - k0), lt);
    if (b0 > 0) {  // the last slab of the block before
      slot_sync<G>(w0);
      if (lt < C6) ch[lt] = ch[kZgBlock * C12 + lt];
      slot_sync<G>(w0);
    }
    for (int id = lt; id < nb * C12; id += NT) ch[C12 + id] = chain[(size_t)b0 * C12 + id];
    for (int s0 = k0; s0 < k1; s0 += SLK) {
      const int cnt = min(SLK, k1 - s0);
      slot_sync<G>(w0);
      K.store(ks, cnt, lt);
      if (s0 + SLK < k1) K.load(fk + (size_t)(s0 + SLK) * KREC, min(SLK, k1 - s0 - SLK), lt);
      slot_sync<G>(w0);
      if (lt < 32)
        for (int i = 0; i < cnt; ++i) {  // g_s = c_s - K_s g_{s-1}
          double *const g = ch + (s0 + i - b0) * C12;
          if (row < C6) {
            const double *Kr = ks + i * KP + row * LD;
            const double w = chain_dot<G>(part == 0 ? g[C12 + row] : 0.0, [&](int j) { return Kr[j]; },
                                        [&](int j) { return g[j]; }, part);
            if (part == 0) g[C12 + row] = w;
          }
          __syncwarp();
        }
    }
    slot_sync<G>(w0);
    // d_s - H_s g_{s-1}, in place of d_s
    for (int id = lt; id < nb * C6; id += NT) {
      const int i = id / C6, j = id - i * C6, s = b0 + i;
      if (s == 0) continue;
      const double *H = fk + (size_t)s * KREC + KP + j, *g = ch + i * C12;
      double a0 = ch[(1 + i) * C12 + C6 + j], a1 = 0.0, a2 = 0.0;
#pragma unroll
      for (int p = 0; p < C6; p += 3) {
        a0 -= H[p * C6] * g[p];
        a1 -= H[(p + 1) * C6] * g[p + 1];
        a2 -= H[(p + 2) * C6] * g[p + 2];
      }
      ch[(1 + i) * C12 + C6 + j] = a0 + (a1 + a2);
    }
    if (nblk > 1) {
      slot_sync<G>(w0);
      for (int id = lt; id < nb * C12; id += NT) chain[(size_t)b0 * C12 + id] = ch[C12 + id];
    }
  }
  grid_trigger();
  // backward: slabs b0 .. at ch[(1 + i) C12] (the last block is there), the
  // first f of the block below kept aside
  for (int blk = nblk - 1; blk >= 0; --blk) {
    const int b0 = blk * kZgBlock, nb = min(kZgBlock, S - b0);
    const int k1 = blk == nblk - 1 ? S - 2 : b0 + nb - 1, k0 = max(1, b0);  // steps k1 down to k0
    if (blk < nblk - 1) {
      slot_sync<G>(w0);
      const double f = lt < C6 ? ch[C12 + C6 + lt] : 0.0;
      slot_sync<G>(w0);
      for (int id = lt; id < nb * C12; id += NT) ch[C12 + id] = chain[(size_t)b0 * C12 + id];
      slot_sync<G>(w0);
      // f_{b0 + nb}: the block is full, so it goes to slab b0 - 1's place
      if (lt < C6) ch[C6 + lt] = f;
    }
    K.load(fk + (size_t)max(k0, k1 - SLK + 1) * KREC, min(SLK, k1 - k0 + 1), lt);
    for (int hi = k1; hi >= k0; hi -= SLK) {
      const int lo = max(k0, hi - SLK + 1);
      slot_sync<G>(w0);
      K.store(ks, hi - lo + 1, lt);
      if (lo > k0) K.load(fk + (size_t)max(k0, lo - SLK) * KREC, min(SLK, lo - k0), lt);
      slot_sync<G>(w0);
      if (lt < 32)
        for (int s = hi; s >= lo; --s) {  // f_s = e_s - K_s^T f_{s+1}
          const double *f = s + 1 == b0 + nb ? ch + C6 : ch + (s - b0 + 2) * C12 + C6;
          if (row < C6) {
            double *const o = ch + (s - b0 + 1) * C12 + C6 + row;
            const double *Kc = ks + (s - lo) * KP + row;
            const double w = chain_dot<G>(part == 0 ? *o : 0.0, [&](int j) { return Kc[j * LD]; },
                                        [&](int j) { return f[j]; }, part);
            if (part == 0) *o = w;
          }
          __syncwarp();
        }
    }
    slot_sync<G>(w0);
    for (int id = lt; id < nb * C12; id += NT) chain[(size_t)b0 * C12 + id] = ch[C12 + id];
  }
}

template <int N>
__global__ void __launch_bounds__(kZgThreads)
zg_chain_kernel(const DevMesh m1, const ZgView v, const double *__restrict__ fac, double *__restrict__ chain,
                const int *__restrict__ done) {
  extern __shared__ __align__(16) unsigned char zsm[];
  int w0, G;
  const int grp = zg_slot(v, w0, G);
  grid_wait();
  done = after_wait(done);
  chain = after_wait(chain);
  if ((done && *done) || grp < 0) return;
  double *const sm = reinterpret_cast<double *>(zsm) + (size_t)w0 * (kZgChLine + kZgKWarp);
  const int S = zg_where(m1, v, grp).S;
  const double *const f = fac + v.fac[grp];
  double *const c = chain + v.chain[grp];
  switch (G) {
#define TN_CASE(GG) case GG: zg_chain<GG>(S, w0, f + zg_koff(3 * N * GG, GG, S), c, sm); break;
    TN_CASE(1) TN_CASE(2) TN_CASE(3) TN_CASE(4)
#undef TN_CASE
  }
}

// ---- the correction of every slab, r.z and r.r
template <int N, int G>
__device__ __forceinline__ void zg_final(const DevMesh &m1, const ZgView &v, const int4 &rg,
                                         const double *__restrict__ fac, const double *r0, double *z0, const double *chain,
                                         double *__restrict__ qv, double &rz, double &rr) {
  using Z = ZgSlab<N, G>;
  constexpr int M = Z::M, MG = Z::MG, MGP = Z::MGP, C6 = Z::C6, C12 = 2 * C6, SL = Z::SL, N2 = N * N, n = N * N2;
  const int tid = threadIdx.x, grp = rg.x, s0 = rg.y, s1 = rg.z;
  const ZgGroup q = zg_where(m1, v, grp);
  const int S = q.S;
  const double *const qw = fac + v.fac[grp] + zg_qoff(MG, G, S);
  const double *const ch = chain + v.chain[grp];
  for (int id = tid; id < (s1 - s0) * C12; id += kZgThreads) {  // g_{s-1} | f_{s+1}
    const int i = id / C12, j = id - i * C12, s = s0 + i;
    qv[id] = j < C6 ? (s > 0 ? ch[(size_t)(s - 1) * C12 + j] : 0.0) : (s + 1 < S ? ch[(size_t)(s + 1) * C12 + j] : 0.0);
  }
  __syncthreads();
  const int sl = tid / MG, t = tid - sl * MG, li = t / M, tl = t - li * M, a = tl / N, k = tl - a * N;
  if (sl >= SL) return;
  const int lid = zg_line(v.lines[grp], li), col = lid / N2, qn = lid - col * N2;
  const size_t gs = (size_t)q.ncol * 3 * n, g0 = q.off + ((size_t)col * 3 + a) * n + (size_t)k * N2 + qn;
  for (int s = s0 + sl; s < s1; s += SL) {
    const size_t at = g0 + (size_t)s * gs;
    const double *w = qw + (size_t)s * Z::QREC + t, *f = qv + (s - s0) * C12;
    const double rv = r0[at];
    double a0 = z0[at], a1 = 0.0, a2 = 0.0;
#pragma unroll
    for (int j = 0; j < C12; j += 3) {
      a0 -= w[j * MGP] * f[j];
      a1 -= w[(j + 1) * MGP] * f[j + 1];
      a2 -= w[(j + 2) * MGP] * f[j + 2];
    }
    const double x = a0 + (a1 + a2);
    z0[at] = x;
    rz += rv * x;
    rr += rv * rv;
  }
}

template <int N>
__global__ void __launch_bounds__(kZgThreads, 4)
zg_final_kernel(const DevMesh m1, const ZgView v, const double *__restrict__ fac, const double *__restrict__ r,
                double *__restrict__ z, const double *__restrict__ chain, double *__restrict__ part_rz,
                double *__restrict__ part_rr, const int *__restrict__ done, const PcgFold fold) {
  constexpr int QV = 12 * kZgChunks * kZgThreads / (3 * N);  // 12 g numbers of at most kZgChunks kZgThreads / (3 g N) slabs
  __shared__ double qv[QV > 48 * kZgChunks ? QV : 48 * kZgChunks];
  const int4 rg = v.ranges[blockIdx.x];
  const int G = zg_size(v.lines[rg.x]);
  grid_wait();
  done = after_wait(done);
  r = after_wait(r);
  z = after_wait(z);
  chain = after_wait(chain);
  if (done && *done) return;
  double rz = 0.0, rr = 0.0;
  switch (G) {
#define TN_CASE(GG) case GG: zg_final<N, GG>(m1, v, rg, fac, r, z, chain, qv, rz, rr); break;
    TN_CASE(1) TN_CASE(2) TN_CASE(3) TN_CASE(4)
#undef TN_CASE
  }
  if (part_rz) {  // FP64 sums of the rows' sums: warp 0 for r.z, warp 1 for r.r
    __shared__ double ps[2][kZgThreads];
    ps[0][threadIdx.x] = rz;
    ps[1][threadIdx.x] = rr;
    __syncthreads();
    const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
    if (w < 2) {
      double x = 0.0;
#pragma unroll
      for (int i = 0; i < kZgThreads / 32; ++i) x += (double)ps[w][32 * i + ln];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      double *const dst = w == 0 ? part_rz : part_rr;
      if (ln == 0 && dst) dst[rg.w] = x;
    }
    if (fold.s) fold_beta(fold);
  }
}

template <typename... P, typename... A>
cudaError_t launch_zg(void (*kernel)(P...), int grid, size_t smem, bool dependent, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kZgThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int N>
cudaError_t launch_f64(const DevMesh &m, const ZGroupDev &gd, int k, const double *fac, const double *r, double *z,
                       double *prz, double *prr, const int *done, TnWait *zerr, cudaStream_t st, bool first,
                       const PcgFold &fold) {
  const ZgView v{gd.inst, gd.meshes, gd.dof_off, gd.lines, gd.fac64_off, gd.chain_off,
                 gd.packs + gd.pk_start[k], gd.ranges + gd.rg_start[k]};
  static int slab_device = -1, chain_device = -1;
  cudaError_t e = allow_smem(zg_slab_kernel<N>, zg_slab_smem<N>(), slab_device);
  if (e == cudaSuccess) e = allow_smem(zg_chain_kernel<N>, zg_chain_smem(), chain_device);
  if (e != cudaSuccess) return e;
  e = launch_zg(zg_slab_kernel<N>, gd.rg_n[k], zg_slab_smem<N>(), first, st, m, v, fac, r,
                            z, gd.chain, done, zerr);
  if (e != cudaSuccess) return e;
  e = launch_zg(zg_chain_kernel<N>, gd.pk_n[k], zg_chain_smem(), true, st, m, v, fac, gd.chain, done);
  if (e != cudaSuccess) return e;
  return launch_zg(zg_final_kernel<N>, gd.rg_n[k], 0, true, st, m, v, fac, r, z, (const double *)gd.chain, prz,
                   prr, done, fold);
}

// CTAs of the FP32 kernel for B CTAs per SM (registers) that an SM holds
template <int N, int B>
cudaError_t packed_per_sm(size_t sm, int *out) {
  auto kern = zgroup_packed_kernel<N, B>;
  static int per_sm[64] = {0};
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!per_sm[dev]) {
    // shared memory before L1: the CTAs per SM are limited by the staging rings
    err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (err == cudaSuccess && sm > 48 * 1024)
      err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    int b = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, kZgThreads, sm);
    if (err != cudaSuccess) return err;
    per_sm[dev] = b > 0 ? b : 1;
  }
  *out = per_sm[dev];
  return cudaSuccess;
}

template <int N, int B>
cudaError_t launch_packed(const DevMesh &m, const ZGroupDev &gd, int k, int grid, size_t sm, const float *fac,
                          const float *r, float *z, double *prz, double *prr, const int *done, TnWait *zerr,
                          cudaStream_t st, bool first, const PcgFold &fold) {
  auto kern = zgroup_packed_kernel<N, B>;
  if (first)
    return launch_pdl(kern, grid, kZgThreads, sm, st, m, gd.inst, gd.meshes, gd.dof_off, gd.lines, gd.fac_off,
                      gd.packs, gd.pk_start[k], gd.pk_n[k], gd.queue + kZgQueue * k, fac, r, z, prz, prr, done, zerr,
                      fold);
  kern<<<grid, kZgThreads, sm, st>>>(m, gd.inst, gd.meshes, gd.dof_off, gd.lines, gd.fac_off, gd.packs,
                                     gd.pk_start[k], gd.pk_n[k], gd.queue + kZgQueue * k, fac, r, z, prz, prr, done,
                                     zerr, fold);
  return cudaGetLastError();
}

// The FP32 kernel is persistent: as many CTAs as fit at once, never more than
// packs.  Four CTAs per SM run a pack fastest; seven (72 registers) take more
// packs at once, which pays from three rounds of packs where it saves a third
// of them: with four against so, us: crystalline stack, p = 5, 4 -> 2 rounds
// 442 -> 368; 12 slabs, p = 2, 576 columns, 3 -> 2 68 -> 52; p = 3, 900, 6 -> 4
// 150 -> 120; p = 4, 324, 4 -> 2 98 -> 77; p = 5, 576, 9 -> 5 254 -> 214; p = 6,
// whose shared memory holds six, 441, 9 -> 6 287 -> 260, 576, 12 -> 8 375 -> 343.
// Below that it is not worth it (p = 6, 993 packs, 2 -> 2 rounds: 116 -> 132; p
// = 5 at 81 columns, 2 -> 1: 62 -> 67), nor with kernels of several degrees
// side by side (24 mirrors: 268 -> 276).  In rounds rather than packs the rule
// turns off again where a round is left over (p = 6, 900 columns, 19 -> 13: 577
// us with four, as before).  From p = 7 shared memory holds four.
// grid_out: only compute the grid; else launch with it.
template <int N>
constexpr bool zp_more() { return 5 * (zp_smem<N>() + 1024) <= 228 * 1024; }
template <int N>
cudaError_t launch_f32(const DevMesh &m, const ZGroupDev &gd, int k, const float *fac, const float *r, float *z,
                       double *prz, double *prr, const int *done, TnWait *zerr, cudaStream_t st, bool first,
                       const PcgFold &fold, int *grid_out) {
  constexpr size_t sm = zp_smem<N>();
  int per_sm = 0;
  cudaError_t err = packed_per_sm<N, 4>(sm, &per_sm);
  if (err != cudaSuccess) return err;
  const int npk = gd.pk_n[k], sms = tn_sm_count();
  bool more = false;
  if constexpr (zp_more<N>()) {
    int seven = 0;
    err = packed_per_sm<N, 7>(sm, &seven);
    if (err != cudaSuccess) return err;
    auto rounds = [&](int per) { return (npk + per * sms - 1) / (per * sms); };
    more = gd.npk == 1 && rounds(per_sm) >= 3 && 3 * rounds(seven) <= 2 * rounds(per_sm);
    if (more) per_sm = seven;
  }
  const int grid = std::min(per_sm * sms, npk);
  if (grid_out) {
    *grid_out = grid;
    return cudaSuccess;
  }
  if constexpr (zp_more<N>())
    if (more) return launch_packed<N, 7>(m, gd, k, grid, sm, fac, r, z, prz, prr, done, zerr, st, first, fold);
  return launch_packed<N, 4>(m, gd, k, grid, sm, fac, r, z, prz, prr, done, zerr, st, first, fold);
}

cudaError_t zgroup_launch(const DevMesh &m, const ZGroupDev &gd, int k, int prec, const void *fac, const void *r,
                          void *z, double *prz, double *prr, const int *done, TnWait *zerr, cudaStream_t st, bool first,
                          const PcgFold &fold, int *grid_out) {
  if (prec == TN_F64 && grid_out) {
    *grid_out = gd.rg_n[k];
    return cudaSuccess;
  }
  switch (gd.pk_N[k]) {
#define TN_CASE(NN)                                                                                              \
  case NN:                                                                                                       \
    return prec == TN_F64 ? launch_f64<NN>(m, gd, k, (const double *)fac, (const double *)r, (double *)z, prz,   \
                                           prr, done, zerr, st, first, fold)                                     \
                          : launch_f32<NN>(m, gd, k, (const float *)fac, (const float *)r, (float *)z, prz, prr, \
                                           done, zerr, st, first, fold, grid_out);
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

// union-find over face matches of the lines (col * N^2 + j * N + i)
static int uf_find(std::vector<int> &p, int x) {
  while (p[x] != x) {
    p[x] = p[p[x]];
    x = p[x];
  }
  return x;
}

// the groups of one mesh (members ascending), or false if a node is shared
// by more than 4 columns
static bool mesh_groups(const tn::HostMesh &hm, std::vector<std::vector<int>> &out, char *msg, int msglen) {
  const int N = hm.N, N2 = N * N, nl = hm.ncol * N2;
  std::vector<int> par(nl);
  for (int x = 0; x < nl; ++x) par[x] = x;
  for (int c = 0; c < hm.ncol; ++c)
    for (int f = 0; f < 4; ++f) {
      const int nbc = hm.colnb[4 * c + f];
      if (nbc < 0) continue;
      const int d = f >> 1, end = (f & 1) ? N - 1 : 0;
      const int code = hm.colnbf[4 * c + f], f2 = code & 3, d2 = f2 >> 1, end2 = (f2 & 1) ? N - 1 : 0;
      for (int t = 0; t < N; ++t) {
        const int i = d == 0 ? end : t, j = d == 0 ? t : end;
        const int a2 = (code >> 2) ? N - 1 - t : t;
        const int i2 = d2 == 0 ? end2 : a2, j2 = d2 == 0 ? a2 : end2;
        const int ra = uf_find(par, c * N2 + j * N + i), rb = uf_find(par, nbc * N2 + j2 * N + i2);
        if (ra != rb) par[ra < rb ? rb : ra] = ra < rb ? ra : rb;
      }
    }
  std::vector<std::vector<int>> comp(nl);
  for (int x = 0; x < nl; ++x) comp[uf_find(par, x)].push_back(x);
  out.clear();
  for (int x = 0; x < nl; ++x) {
    if (comp[x].empty()) continue;
    if (comp[x].size() > 4) {
      std::snprintf(msg, msglen, "a cross-section node is shared by %d columns (line groups hold at most 4)",
                    (int)comp[x].size());
      return false;
    }
    out.push_back(comp[x]);
  }
  return true;
}

bool tn_zgroup_plan(const tn::HostMesh *const *hms, int n, ZGroupPlan *p, char *msg, int msglen) {
  std::vector<std::vector<std::vector<int>>> per(n);
  for (int i = 0; i < n; ++i)
    if (!mesh_groups(*hms[i], per[i], msg, msglen)) return false;
  *p = ZGroupPlan();
  p->inst_start.assign((size_t)n * 5, 0);
  p->inst_n.assign((size_t)n * 5, 0);
  // order: group size (largest first), degree, mirror -- one class per (size, degree)
  for (int g = 4; g >= 1; --g)
    for (int N = TN_MIN_N; N <= TN_MAX_N; ++N) {
      const int start = p->ngroups;
      for (int i = 0; i < n; ++i) {
        if (hms[i]->N != N) continue;
        p->inst_start[(size_t)i * 5 + g] = p->ngroups;
        for (const auto &mm : per[i]) {
          if ((int)mm.size() != g) continue;
          p->lines.push_back(make_int4(mm[0], g > 1 ? mm[1] : -1, g > 2 ? mm[2] : -1, g > 3 ? mm[3] : -1));
          p->inst.push_back(i);
          p->fac_off.push_back(p->nfac);
          p->nfac += (long long)hms[i]->nslab * zp_rec(g * 3 * N, g);
          p->fac64_off.push_back(p->nfac64);
          p->nfac64 += zg_entries(g * 3 * N, g, hms[i]->nslab);
          p->chain_off.push_back(p->nchain);
          p->nchain += (long long)hms[i]->nslab * 12 * g;
          p->ncompact += (long long)hms[i]->nslab * (zlp(g * 3 * N) + 8 * g * 3 * N);
          ++p->inst_n[(size_t)i * 5 + g];
          ++p->ngroups;
        }
      }
      if (p->ngroups == start) continue;
      if (p->ncls >= kZgMaxCls) {
        std::snprintf(msg, msglen, "too many line-group classes");
        return false;
      }
      p->cls_N[p->ncls] = N;
      p->cls_G[p->ncls] = g;
      p->cls_start[p->ncls] = start;
      p->cls_n[p->ncls] = p->ngroups - start;
      ++p->ncls;
    }
  // packs of groups filling the four warps of a CTA, per degree, largest
  // first: 4, 3 + 1, 2 + 2, 2 + 1 + 1, 1 + 1 + 1 + 1 lines
  for (int N = TN_MIN_N; N <= TN_MAX_N; ++N) {
    std::vector<int> by[5];
    for (int k = 0; k < p->ncls; ++k)
      if (p->cls_N[k] == N)
        for (int i = 0; i < p->cls_n[k]; ++i) by[p->cls_G[k]].push_back(p->cls_start[k] + i);
    if (by[1].empty() && by[2].empty() && by[3].empty() && by[4].empty()) continue;
    const int start = (int)p->packs.size();
    size_t i1 = 0;
    auto one = [&]() { return i1 < by[1].size() ? by[1][i1++] : -1; };
    for (int g4 : by[4]) p->packs.push_back(make_int4(g4, -1, -1, -1));
    for (int g3 : by[3]) p->packs.push_back(make_int4(g3, one(), -1, -1));
    for (size_t i = 0; i < by[2].size(); i += 2) {
      if (i + 1 < by[2].size()) {
        p->packs.push_back(make_int4(by[2][i], by[2][i + 1], -1, -1));
      } else {
        const int a = one();
        const int b = a >= 0 ? one() : -1;
        p->packs.push_back(make_int4(by[2][i], a, b, -1));
      }
    }
    while (i1 < by[1].size()) {
      const int a = one(), b = one(), c = one(), d = one();
      p->packs.push_back(make_int4(a, b, c, d));
    }
    if (p->npk >= kZgMaxDg) {
      std::snprintf(msg, msglen, "too many degrees for the grouped-line solve");
      return false;
    }
    p->pk_N[p->npk] = N;
    p->pk_start[p->npk] = start;
    p->pk_n[p->npk] = (int)p->packs.size() - start;
    // slab ranges of the first and last launch, in the order of the groups:
    // as many stages each as leave every SM its CTAs
    auto stages = [&](int k, int i) {
      const int sl = zg_slabs(N, p->cls_G[k]);
      return (hms[p->inst[i]]->nslab + sl - 1) / sl;
    };
    long long all = 0;
    for (int k = 0; k < p->ncls; ++k)
      if (p->cls_N[k] == N)
        for (int i = p->cls_start[k]; i < p->cls_start[k] + p->cls_n[k]; ++i) all += stages(k, i);
    const int per = (int)std::min<long long>(std::max<long long>(all / kZgFill, 1), kZgChunks);
    p->rg_start[p->npk] = (int)p->ranges.size();
    for (int k = 0; k < p->ncls; ++k) {
      if (p->cls_N[k] != N) continue;
      const int sl = zg_slabs(N, p->cls_G[k]) * per;
      for (int i = p->cls_start[k]; i < p->cls_start[k] + p->cls_n[k]; ++i) {
        const int S = hms[p->inst[i]]->nslab;
        for (int s = 0; s < S; s += sl)
          p->ranges.push_back(make_int4(i, s, std::min(S, s + sl), (int)p->ranges.size()));
      }
    }
    p->rg_n[p->npk] = (int)p->ranges.size() - p->rg_start[p->npk];
    ++p->npk;
  }
  return true;
}

// per degree present (one for a single mesh) one launch (FP32) or three
// (FP64): the first degree on st, the others on side streams forked from and
// joined back into st (also inside a capture)
cudaError_t tn_zgroup_solve(const DevMesh *m, const ZGroupDev &gd, int prec, const void *fac, const void *r, void *z,
                            double *part_rz, double *part_rr, const int *done, TnWait *zerr, cudaStream_t st,
                            const PcgFold *fold_in) {
  const DevMesh one = m ? *m : DevMesh{};
  cudaError_t err = cudaSuccess;
  PcgFold fold = fold_in ? *fold_in : PcgFold();
  if (fold.s) {  // the grids of the launches that fold, for the last-CTA count
    fold.total = 0;
    fold.nparts = tn_zgroup_partials(gd, prec);
    fold.part = part_rz;
    fold.part2 = part_rr;
    for (int k = 0; k < gd.npk && err == cudaSuccess; ++k) {
      int g = 0;
      err = zgroup_launch(one, gd, k, prec, fac, r, z, part_rz, part_rr, done, zerr, st, false, fold, &g);
      fold.total += g;
    }
    if (err != cudaSuccess) return err;
  }
  if (gd.npk > 1) err = cudaEventRecord(gd.fork, st);
  bool used[kZgSide] = {false};
  for (int k = 0; k < gd.npk && err == cudaSuccess; ++k) {
    cudaStream_t sk = st;
    if (k > 0) {
      const int sd = (k - 1) % kZgSide;
      sk = gd.side[sd];
      if (!used[sd]) {
        err = cudaStreamWaitEvent(sk, gd.fork, 0);
        used[sd] = true;
        if (err != cudaSuccess) break;
      }
    }
    // (a launch behind an event is not a programmatic dependent)
    err = zgroup_launch(one, gd, k, prec, fac, r, z, part_rz, part_rr, done, zerr, sk, gd.npk == 1, fold,
                        nullptr);
  }
  for (int sd = 0; sd < kZgSide && err == cudaSuccess; ++sd) {
    if (!used[sd]) continue;
    err = cudaEventRecord(gd.join[sd], gd.side[sd]);
    if (err == cudaSuccess) err = cudaStreamWaitEvent(st, gd.join[sd], 0);
  }
  return err;
}
