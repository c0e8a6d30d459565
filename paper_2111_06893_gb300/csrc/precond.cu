// Column-line and grouped-line block preconditioners for thin layers.
//
// The paper accelerates its Krylov solver with multigrid and an additive
// Schwarz smoother (Sec. 2.3).  The dominant difficulty of thin coating layers
// is the strong coupling across the layers: elements with aspect ratios up
// to ~1e4 and penalties sigma ~ 1/h_z on the layer interfaces (Eq. (penalty)).
// This preconditioner takes, for every vertical line of nodes (column col,
// cross-section node (i, j), all slabs, all N nodes along zeta, three
// components), the exact principal sub-matrix A_LL of the DG operator on that
// line and inverts it: A_LL is block tridiagonal over the slabs (3N x 3N
// blocks: D_s inside slab s, O_s coupling slab s to the slab below through
// the face terms of Eq. (numflux)).  Set-up: the blocks are formed from the
// same weak-form terms as the operator (FP64), factorised by block Cholesky
// along the line (one thread per line) and stored in FP32.  Application:
// one warp per line, the 3N unknowns of a slab on the lanes, forward and
// backward block substitution.  The grouped variant takes
// the lines through one cross-section point of neighbouring columns
// together (zgroup.cu), adding the lateral-face coupling between them.
#include <cstdio>
#include <type_traits>
#include <vector>

#include "tn_device.h"
#include "tn_internal.h"
#include "tn_precond.h"

// device constants are per translation unit (no relocatable device code):
// this file keeps its own copy of the LGL tables
__constant__ LglTables c_lgl_pc;

cudaError_t tn_upload_lgl_precond(const LglTables *t) {
  return cudaMemcpyToSymbol(c_lgl_pc, t, sizeof(LglTables));
}

namespace {

// Factor record of one line and slab s: [Linv_s | Z_s].
//  Linv_s: inverse of the lower Cholesky factor of the slab's Schur
//          complement, lower triangular, packed column by column (column c
//          holds rows c..M-1 at zcol(M, c) + (row - c)), M (M + 1) / 2 entries;
//  Z_s:    L_{s-1}^{-1} O_{s-1}, row-major with an odd row stride zld(M) so
//          that lanes reading one entry per row hit distinct banks.
// Both parts are padded to a multiple of 4 entries (16-byte cp.async chunks
// for float and double records).
__host__ __device__ constexpr int zld(int M) { return M | 1; }
__host__ __device__ constexpr int zzp(int M) { return pad4(M * zld(M)); }
__host__ __device__ constexpr int zrec(int M) { return zlp(M) + zzp(M); }

#define LD(a, b) c_lgl_pc.D[N][(a) * N + (b)]
#define LW(a) c_lgl_pc.w[N][(a)]

// D_s and O_s of every line through element e: one thread per line (i, j)
template <int N>
__global__ void zline_blocks_kernel(const DevMesh m, double *__restrict__ blk) {
  constexpr int M = 3 * N, N2 = N * N;
  const int e = blockIdx.x, t = threadIdx.x;
  if (t >= N2) return;
  const int s = e / m.ncol, c = e - s * m.ncol;
  const int i = t % N, j = t / N;
  const size_t line = (size_t)c * N2 + t;
  double *Dm = blk + ((line * m.nslab + s) * 2 + 0) * M * M;
  double *Om = blk + ((line * m.nslab + s) * 2 + 1) * M * M;
  for (int q = 0; q < M * M; ++q) { Dm[q] = 0.0; Om[q] = 0.0; }
  const double *cg = m.colgeo + (size_t)c * CG_NF * N2;
  const double *sg = m.slabgeo + (size_t)s * SG_NF * N;
  const int qq = j * N + i;
  const double ixx = cg[CG_IXX * N2 + qq], ixy = cg[CG_IXY * N2 + qq];
  const double iex = cg[CG_IEX * N2 + qq], iey = cg[CG_IEY * N2 + qq];
  const double det2 = cg[CG_DET * N2 + qq];
  double dz[N];
  for (int k = 0; k < N; ++k) dz[k] = sg[SG_DZ * N + k];
  const int L = m.slab_layer[s];
  const double c11 = m.layer_c[3 * L], c12 = m.layer_c[3 * L + 1], c44 = m.layer_c[3 * L + 2];
  const double Dii = LD(i, i), Djj = LD(j, j);

  // ---- volume: r on the z-line
  for (int kk = 0; kk < N; ++kk) {
    const double wJ = LW(i) * LW(j) * LW(kk) * det2 * dz[kk];
    for (int k = 0; k < N; ++k) {
      double lk[3] = {k == kk ? Dii : 0.0, k == kk ? Djj : 0.0, LD(kk, k)}, gk[3];
      phys(lk, ixx, ixy, iex, iey, dz[kk], gk);
      for (int k2 = 0; k2 < N; ++k2) {
        double l2[3] = {k2 == kk ? Dii : 0.0, k2 == kk ? Djj : 0.0, LD(kk, k2)}, g2[3];
        phys(l2, ixx, ixy, iex, iey, dz[kk], g2);
        for (int a = 0; a < 3; ++a)
          for (int b = 0; b < 3; ++b) Dm[(a * N + k) * M + b * N + k2] += wJ * Qab(a, b, gk, g2, c11, c12, c44);
      }
    }
  }
  // r on the xi- and eta-lines through the node (diagonal in k)
  for (int k = 0; k < N; ++k) {
    for (int r = 0; r < N; ++r) {
      if (r != i) {
        const int q2 = j * N + r;
        const double wJ = LW(r) * LW(j) * LW(k) * cg[CG_DET * N2 + q2] * dz[k];
        const double d = LD(r, i);
        const double g[3] = {cg[CG_IXX * N2 + q2] * d, cg[CG_IXY * N2 + q2] * d, 0.0};
        for (int a = 0; a < 3; ++a)
          for (int b = 0; b < 3; ++b) Dm[(a * N + k) * M + b * N + k] += wJ * Qab(a, b, g, g, c11, c12, c44);
      }
      if (r != j) {
        const int q2 = r * N + i;
        const double wJ = LW(i) * LW(r) * LW(k) * cg[CG_DET * N2 + q2] * dz[k];
        const double d = LD(r, j);
        const double g[3] = {cg[CG_IEX * N2 + q2] * d, cg[CG_IEY * N2 + q2] * d, 0.0};
        for (int a = 0; a < 3; ++a)
          for (int b = 0; b < 3; ++b) Dm[(a * N + k) * M + b * N + k] += wJ * Qab(a, b, g, g, c11, c12, c44);
      }
    }
  }

  const double sp1 = (double)((m.p + 1) * (m.p + 1)) * m.penC;
  // ---- faces of the element that contain line nodes
  for (int f = 0; f < 6; ++f) {
    const int d = f >> 1, sd = f & 1;
    const int idx = d == 0 ? i : (d == 1 ? j : -1);
    if (d < 2 && idx != (sd ? N - 1 : 0)) continue;
    // kind and neighbour
    int kind;  // 0 interior, 1 dirichlet, 2 neumann
    double h2 = 0.0, n11 = c11, n12 = c12, n44 = c44;
    if (d < 2) {
      const int nbc = m.colnb[4 * c + f];
      if (nbc >= 0) {
        kind = 0;
        const int code = m.colnbf[4 * c + f];
        const int f2 = code & 3, d2 = f2 >> 1, end2 = (f2 & 1) ? N - 1 : 0;
        const int t1 = d == 0 ? j : i;
        const int a2 = (code >> 2) ? N - 1 - t1 : t1;
        const int i2 = d2 == 0 ? end2 : a2, j2 = d2 == 0 ? a2 : end2;
        const double *g2 = m.colgeo + (size_t)nbc * CG_NF * N2;
        const double rx = g2[(d2 == 0 ? CG_IXX : CG_IEX) * N2 + j2 * N + i2];
        const double ry = g2[(d2 == 0 ? CG_IXY : CG_IEY) * N2 + j2 * N + i2];
        h2 = 2.0 / sqrt(rx * rx + ry * ry);
      } else {
        kind = m.bc_side == TN_BC_FIXED ? 1 : 2;
      }
    } else if (f == 4) {
      if (s + 1 < m.nslab) {
        kind = 0;
        h2 = 2.0 * m.slabgeo[((size_t)(s + 1) * SG_NF + SG_DZ) * N + N - 1];
        const int L2 = m.slab_layer[s + 1];
        n11 = m.layer_c[3 * L2]; n12 = m.layer_c[3 * L2 + 1]; n44 = m.layer_c[3 * L2 + 2];
      } else {
        kind = m.bc_bottom == TN_BC_FIXED ? 1 : 2;
      }
    } else {
      if (s > 0) {
        kind = 0;
        h2 = 2.0 * m.slabgeo[((size_t)(s - 1) * SG_NF + SG_DZ) * N + 0];
        const int L2 = m.slab_layer[s - 1];
        n11 = m.layer_c[3 * L2]; n12 = m.layer_c[3 * L2 + 1]; n44 = m.layer_c[3 * L2 + 2];
      } else {
        kind = 2;  // top: beam pressure (Neumann)
      }
    }
    if (kind == 2) continue;
    double n[3], mag = 1.0;
    if (d == 2) { n[0] = 0.0; n[1] = 0.0; n[2] = sd ? 1.0 : -1.0; }
    else {
      const double rx = d == 0 ? ixx : iex, ry = d == 0 ? ixy : iey;
      mag = sqrt(rx * rx + ry * ry);
      n[0] = (sd ? 1.0 : -1.0) * rx / mag; n[1] = (sd ? 1.0 : -1.0) * ry / mag; n[2] = 0.0;
    }
    const double cT = kind == 0 ? -0.5 : -1.0, cP = kind == 0 ? 1.0 : 2.0;
    const double s11 = kind == 0 ? 0.5 * (c11 + n11) : c11, s12 = kind == 0 ? 0.5 * (c12 + n12) : c12,
                 s44 = kind == 0 ? 0.5 * (c44 + n44) : c44;
    const int kend = sd ? N - 1 : 0;
    for (int k = 0; k < N; ++k) {
      if (d == 2 && k != kend) continue;  // line node on the face
      double W, h;
      if (d == 2) { W = LW(i) * LW(j) * det2; h = 2.0 * dz[k]; }
      else { W = (d == 0 ? LW(j) : LW(i)) * LW(k) * det2 * dz[k] * mag; h = 2.0 / mag; }
      // T1[(a,k),(b,k2)] = W Q_ab(n, grad psi_k2 at node k); added with its transpose
      for (int k2 = 0; k2 < N; ++k2) {
        double l2[3] = {k2 == k ? Dii : 0.0, k2 == k ? Djj : 0.0, LD(k, k2)}, g2[3];
        phys(l2, ixx, ixy, iex, iey, dz[k], g2);
        for (int a = 0; a < 3; ++a)
          for (int b = 0; b < 3; ++b) {
            const double v = cT * W * Qab(a, b, n, g2, c11, c12, c44);
            Dm[(a * N + k) * M + b * N + k2] += v;
            Dm[(b * N + k2) * M + a * N + k] += v;
          }
      }
      const double sig = sp1 / (kind == 0 ? (h < h2 ? h : h2) : h);
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) Dm[(a * N + k) * M + b * N + k] += cP * W * sig * Qab(a, b, n, n, s11, s12, s44);
    }
    // ---- coupling to the slab below (face zeta = -1, k = 0, neighbour's k = N-1)
    if (f == 4 && kind == 0) {
      const double W = LW(i) * LW(j) * det2;
      const double dz2 = m.slabgeo[((size_t)(s + 1) * SG_NF + SG_DZ) * N + N - 1];
      const double sig = sp1 / (2.0 * dz[0] < 2.0 * dz2 ? 2.0 * dz[0] : 2.0 * dz2);
      for (int k = 0; k < N; ++k)
        for (int k2 = 0; k2 < N; ++k2) {
          for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) {
              double v = 0.0;
              if (k == 0) {  // -1/2 V^T W Tr_ext: neighbour basis gradient at its node N-1
                double l2[3] = {k2 == N - 1 ? Dii : 0.0, k2 == N - 1 ? Djj : 0.0, LD(N - 1, k2)}, g2[3];
                phys(l2, ixx, ixy, iex, iey, dz2, g2);
                v += -0.5 * W * Qab(a, b, n, g2, n11, n12, n44);
              }
              if (k2 == N - 1) {  // +1/2 Tr^T W V_ext: own basis gradient at node 0
                double l1[3] = {k == 0 ? Dii : 0.0, k == 0 ? Djj : 0.0, LD(0, k)}, g1[3];
                phys(l1, ixx, ixy, iex, iey, dz[0], g1);
                v += 0.5 * W * Qab(b, a, n, g1, c11, c12, c44);
              }
              if (k == 0 && k2 == N - 1) v -= W * sig * Qab(a, b, n, n, s11, s12, s44);
              Om[(a * N + k) * M + b * N + k2] += v;
            }
        }
    }
  }
}

// block Cholesky along each line (FP64, in place), then FP32 factors:
// L_s column-major with inverted diagonal, Z_s = L_{s-1}^{-1} O_{s-1} row-major
template <int N>
__global__ void zline_factor_kernel(int nlines, int S, double *__restrict__ blk, float *__restrict__ fac,
                                    double *__restrict__ fac64, int *__restrict__ status) {
  constexpr int M = 3 * N;
  const int line = blockIdx.x * blockDim.x + threadIdx.x;
  if (line >= nlines) return;
  for (int s = 0; s < S; ++s) {
    double *Dm = blk + (((size_t)line * S + s) * 2 + 0) * M * M;
    if (s > 0) {
      const double *Lp = blk + (((size_t)line * S + s - 1) * 2 + 0) * M * M;
      double *Z = blk + (((size_t)line * S + s - 1) * 2 + 1) * M * M;  // O_{s-1} -> Z_s in place
      for (int col = 0; col < M; ++col)
        for (int r = 0; r < M; ++r) {
          double v = Z[r * M + col];
          for (int q = 0; q < r; ++q) v -= Lp[r * M + q] * Z[q * M + col];
          Z[r * M + col] = v / Lp[r * M + r];
        }
      for (int r = 0; r < M; ++r)
        for (int c2 = 0; c2 <= r; ++c2) {
          double v = 0.0;
          for (int q = 0; q < M; ++q) v += Z[q * M + r] * Z[q * M + c2];
          Dm[r * M + c2] -= v;
        }
    }
    for (int col = 0; col < M; ++col) {
      double v = Dm[col * M + col];
      for (int q = 0; q < col; ++q) v -= Dm[col * M + q] * Dm[col * M + q];
      if (!(v > 0.0)) {
        atomicExch(status, 1);
        v = 1e-300;
      }
      const double dgl = sqrt(v);
      Dm[col * M + col] = dgl;
      for (int r = col + 1; r < M; ++r) {
        double w = Dm[r * M + col];
        for (int q = 0; q < col; ++q) w -= Dm[r * M + q] * Dm[col * M + q];
        Dm[r * M + col] = w / dgl;
      }
    }
    // inverse of the lower-triangular factor (forward substitution on the
    // identity), packed by columns; Z_s with row stride zld(M)
    constexpr int LP = zlp(M), LDZ = zld(M), RS = zrec(M);
    float *Lf = fac + ((size_t)line * S + s) * RS;
    double *Ld = fac64 + ((size_t)line * S + s) * RS;
    for (int col = 0; col < M; ++col) {
      const int pc = zcol(M, col);
      for (int r = col; r < M; ++r) {
        double v;
        if (r == col) {
          v = 1.0 / Dm[r * M + r];
        } else {
          double acc = 0.0;
          for (int q = col; q < r; ++q) acc += Dm[r * M + q] * Ld[pc + (q - col)];
          v = -acc / Dm[r * M + r];
        }
        Ld[pc + (r - col)] = v;
        Lf[pc + (r - col)] = (float)v;
      }
    }
    for (int q = M * (M + 1) / 2; q < LP; ++q) { Lf[q] = 0.0f; Ld[q] = 0.0; }
    float *Zf = Lf + LP;
    double *Zd = Ld + LP;
    const double *Z = s > 0 ? blk + (((size_t)line * S + s - 1) * 2 + 1) * M * M : nullptr;
    for (int q = 0; q < zzp(M); ++q) {
      const int r = q / LDZ, col = q - r * LDZ;
      const double v = (Z && r < M && col < M) ? Z[r * M + col] : 0.0;
      Zf[q] = (float)v;
      Zd[q] = v;
    }
  }
}

// shared memory of one warp: two stages of one factor record, two
// broadcast vectors of 32 entries, two mbarriers
template <int N, typename F>
__host__ __device__ constexpr int zline_warp_bytes() {
  return 2 * zrec(3 * N) * (int)sizeof(F) + 2 * 32 * (int)sizeof(F) + 16;
}
template <int N, typename F>
constexpr size_t zline_smem() { return (size_t)4 * zline_warp_bytes<N, F>(); }

// z = A_LL^{-1} r on one line (one warp; lane l = a * N + k holds one unknown
// of a slab), with A_LL = L L^T block-bidiagonal:
//   forward   y_s = Linv_s (r_s - Z_s^T y_{s-1})      (y = L^{-1} r, kept in z)
//   backward  x_s = Linv_s^T (y_s - Z_{s+1} x_{s+1})  (x = L^{-T} y)
// Every product is a broadcast matrix-vector product.  The factor record of
// the next slab is brought into shared memory by one bulk copy while the
// current slab is worked on (two stages); this lane's r, q and y entries are
// loaded two slabs ahead into registers.  UPD: first r <- r - alpha q (the
// PCG residual update, written back).  Adds this lane's r.z (= |y|^2, since
// r.z = r^T L^-T L^-1 r) and r.r to rz, rr.  A staging wait that runs out
// sets *err and ends the line.
template <int N, typename T, typename F, bool UPD>
__device__ __forceinline__ void zline_line(const DevMesh &m, const F *__restrict__ fac, T *__restrict__ r,
                                           const T *__restrict__ q, T *__restrict__ z, T alpha, int line,
                                           int lane, unsigned char *smem, TnWait *err, T &rz, T &rr) {
  static_assert(sizeof(T) == sizeof(F), "vectors and factors share one precision");
  constexpr int M = 3 * N, N2 = N * N, n = N * N * N;
  constexpr int LP = zlp(M), LDZ = zld(M), RS = zrec(M);
  const int S = m.nslab;
  const int c = line / N2, qn = line - c * N2, i = qn % N, j = qn / N;
  const int a = lane / N, k = lane - (lane / N) * N;
  const bool act = lane < M;
  const int ll = act ? lane : 0;
  const size_t off = (size_t)k * N2 + j * N + i;
  const size_t ncol = m.ncol;
  const F *base = fac + (size_t)line * S * RS;
  F *const stg0 = reinterpret_cast<F *>(smem);
  T *const vb = reinterpret_cast<T *>(smem + 2 * RS * sizeof(F));  // b_s / y_s (broadcast)
  T *const vx = vb + 32;                                            // y_{s-1} / x_{s+1} (broadcast)
  unsigned long long *const bar =
      reinterpret_cast<unsigned long long *>(smem + 2 * RS * sizeof(F) + 64 * sizeof(F));
  unsigned ph = 0u, pend = 0u;  // bit b: phase parity / copy in flight of stage b
  auto stg = [&](int b) { return stg0 + b * RS; };
  auto gidx = [&](int s) { return ((size_t)(s * ncol + c) * 3 + (act ? a : 0)) * n + off; };
  auto issue = [&](int b, const F *src0, int cnt0, const F *src1, int cnt1) {
    if (lane == 0) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      mbar_expect(bar + b, (unsigned)((cnt0 + cnt1) * sizeof(F)));
      bulk_g2s(stg(b), src0, (unsigned)(cnt0 * sizeof(F)), bar + b);
      if (cnt1) bulk_g2s(stg(b) + LP, src1, (unsigned)(cnt1 * sizeof(F)), bar + b);
    }
    pend |= 1u << b;
  };
  const unsigned long long lim = wait_limit(err);
  // the warp agrees on the outcome; a stage counts as landed only if every
  // lane saw it land, so that the lanes keep one view of the stages
  auto wait = [&](int b) {
    const bool ok = __all_sync(0xffffffffu, mbar_wait(bar + b, (ph >> b) & 1u, lim));
    if (ok) {
      ph ^= 1u << b;
      pend &= ~(1u << b);
    }
    return ok;
  };
  auto drain = [&]() {  // after a timeout: a bounded wait for every copy still in flight
    if (pend & 1u) mbar_wait(bar, ph & 1u, kDrainNs);
    if (pend & 2u) mbar_wait(bar + 1, (ph >> 1) & 1u, kDrainNs);
    if (lane == 0 && err) atomicExch(&err->flag, 1);
  };
  if (lane == 0) {
    mbar_init(bar);
    mbar_init(bar + 1);
    mbar_init_fence();
  }
  __syncwarp();
  // forward sweep
  issue(0, base, RS, nullptr, 0);
  T r0 = act ? r[gidx(0)] : T(0), q0 = (UPD && act) ? q[gidx(0)] : T(0);
  T r1 = (act && S > 1) ? r[gidx(1)] : T(0), q1 = (UPD && act && S > 1) ? q[gidx(1)] : T(0);
  T yprev = T(0);
  if (lane == 0 && S > 1) bulk_prefetch_l2(base + RS, RS * sizeof(F));
  for (int s = 0; s < S; ++s) {
    const int b = s & 1;
    // the record two slabs ahead goes to L2 now, so that its bulk copy (issued
    // at the next step) is served from L2
    if (lane == 0 && s + 2 < S) bulk_prefetch_l2(base + (size_t)(s + 2) * RS, RS * sizeof(F));
    if (s + 1 < S) issue(b ^ 1, base + (size_t)(s + 1) * RS, RS, nullptr, 0);
    if (!wait(b)) { drain(); return; }
    const F *Li = stg(b), *Zs = stg(b) + LP;
    const size_t idx = gidx(s);
    T rv = r0;
    if (UPD) {
      rv -= alpha * q0;
      if (act) r[idx] = rv;
    }
    // entries two slabs ahead
    r0 = r1;
    q0 = q1;
    if (act && s + 2 < S) {
      r1 = r[gidx(s + 2)];
      if (UPD) q1 = q[gidx(s + 2)];
    }
    rr += rv * rv;
    T bv = rv;
    if (s > 0) bv -= bcast_dot<M, T>(vx, [&](int cc) { return (T)Zs[cc * LDZ + ll]; });  // Z_s^T y_{s-1}
    vb[lane] = act ? bv : T(0);
    __syncwarp();
    T y = bcast_dot<M, T>(vb, [&](int cc) { return cc <= ll ? (T)Li[zcol(M, cc) + ll - cc] : T(0); });
    if (!act) y = T(0);
    rz += y * y;
    if (act) z[idx] = y;
    yprev = y;
    __syncwarp();  // every lane is done with vx, vb and stage b
    vx[lane] = y;
    __syncwarp();
  }
  // backward sweep: slab s needs Linv_s and Z_{s+1}
  auto issue_bwd = [&](int s, int b) {
    issue(b, base + (size_t)s * RS, LP, base + (size_t)(s + 1) * RS + LP, s + 1 < S ? RS - LP : 0);
  };
  const int pl = zcol(M, ll) - ll;
  int bb = S & 1;  // the stage the forward sweep did not end on
  issue_bwd(S - 1, bb);
  T y0 = yprev;  // y_{S-1}
  T y1 = (act && S > 1) ? z[gidx(S - 2)] : T(0);
  T y2 = (act && S > 2) ? z[gidx(S - 3)] : T(0);
  if (lane == 0 && S > 1) bulk_prefetch_l2(base + (size_t)(S - 2) * RS, RS * sizeof(F));
  for (int s = S - 1; s >= 0; --s, bb ^= 1) {
    if (lane == 0 && s >= 2) bulk_prefetch_l2(base + (size_t)(s - 2) * RS, RS * sizeof(F));
    if (s > 0) issue_bwd(s - 1, bb ^ 1);
    if (!wait(bb)) { drain(); return; }
    const F *Li = stg(bb), *Zn = stg(bb) + LP;
    T yv = y0;
    y0 = y1;
    y1 = y2;
    if (act && s >= 3) y2 = z[gidx(s - 3)];
    if (s + 1 < S) yv -= bcast_dot<M, T>(vx, [&](int cc) { return (T)Zn[ll * LDZ + cc]; });  // Z_{s+1} x_{s+1}
    vb[lane] = act ? yv : T(0);
    __syncwarp();
    T x = bcast_dot<M, T>(vb, [&](int cc) { return cc >= ll ? (T)Li[pl + cc] : T(0); });
    if (!act) x = T(0);
    if (act) z[gidx(s)] = x;
    __syncwarp();  // every lane is done with vx, vb and stage bb
    vx[lane] = x;
    __syncwarp();
  }
}

// four lines (warps) per block; per-block partial sums of r.z and r.r
__device__ __forceinline__ void block_partial2(double rz, double rr, double *part_rz, double *part_rr) {
  __shared__ double red[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rz += __shfl_xor_sync(0xffffffffu, rz, o);
    rr += __shfl_xor_sync(0xffffffffu, rr, o);
  }
  if (lane == 0) { red[warp] = rz; red[4 + warp] = rr; }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (part_rz) part_rz[blockIdx.x] = red[0] + red[1] + red[2] + red[3];
    if (part_rr) part_rr[blockIdx.x] = red[4] + red[5] + red[6] + red[7];
  }
}

template <int N, typename T, typename F, bool UPD>
__global__ void __launch_bounds__(128)
zline_solve_kernel(const DevMesh m, const F *__restrict__ fac, T *__restrict__ r, const T *__restrict__ q,
                   T *__restrict__ z, const double *__restrict__ alpha, double *__restrict__ part_rz,
                   double *__restrict__ part_rr, const int *__restrict__ done, TnWait *__restrict__ err) {
  if (done && *done) return;
  extern __shared__ __align__(16) unsigned char zsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int line = blockIdx.x * 4 + warp;
  const T al = UPD ? (T)*alpha : T(0);
  T rz = T(0), rr = T(0);
  if (line < m.ncol * N * N)
    zline_line<N, T, F, UPD>(m, fac, r, q, z, al, line, lane, zsm + warp * zline_warp_bytes<N, F>(), err, rz,
                             rr);
  block_partial2((double)rz, (double)rr, part_rz, part_rr);
}

// a batch: warp w of block b handles line work[4 b + w] = (instance, line)
template <int N, typename T, typename F, bool UPD>
__global__ void __launch_bounds__(128)
zline_solve_batch_kernel(const DevMesh *__restrict__ meshes, const int2 *__restrict__ work, int nwork,
                         const long long *__restrict__ fac_off, const long long *__restrict__ dof_off,
                         const F *__restrict__ fac, T *__restrict__ r, const T *__restrict__ q,
                         T *__restrict__ z, const double *__restrict__ alpha, double *__restrict__ part_rz,
                         double *__restrict__ part_rr, const int *__restrict__ done, TnWait *__restrict__ err) {
  if (done && *done) return;
  extern __shared__ __align__(16) unsigned char zsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wi = blockIdx.x * 4 + warp;
  const T al = UPD ? (T)*alpha : T(0);
  T rz = T(0), rr = T(0);
  if (wi < nwork) {
    const int2 w = work[wi];
    const long long off = dof_off[w.x];
    zline_line<N, T, F, UPD>(meshes[w.x], fac + fac_off[w.x], r + off, UPD ? q + off : nullptr, z + off, al,
                             w.y, lane, zsm + warp * zline_warp_bytes<N, F>(), err, rz, rr);
  }
  block_partial2((double)rz, (double)rr, part_rz, part_rr);
}

template <int N>
cudaError_t setup_n(const DevMesh &m, double *blk, float *fac, double *fac64, int *status, cudaStream_t st) {
  zline_blocks_kernel<N><<<m.E, ((N * N + 31) / 32) * 32, 0, st>>>(m, blk);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  const int nlines = m.ncol * N * N;
  zline_factor_kernel<N><<<(nlines + 63) / 64, 64, 0, st>>>(nlines, m.nslab, blk, fac, fac64, status);
  return cudaGetLastError();
}

// opt in to more than 48 KB of dynamic shared memory (FP64, large N)
template <typename K>
cudaError_t zline_smem_optin(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int N, typename T, bool UPD>
cudaError_t solve_nt(const DevMesh &m, const void *fac, void *r, const void *q, void *z, const double *alpha,
                     double *part_rz, double *part_rr, const int *done, TnWait *zerr, cudaStream_t st) {
  const int blocks = (m.ncol * N * N + 3) / 4;
  constexpr size_t sm = zline_smem<N, T>();
  cudaError_t err = zline_smem_optin(zline_solve_kernel<N, T, T, UPD>, sm);
  if (err != cudaSuccess) return err;
  zline_solve_kernel<N, T, T, UPD><<<blocks, 128, sm, st>>>(m, (const T *)fac, (T *)r, (const T *)q, (T *)z,
                                                             alpha, part_rz, part_rr, done, zerr);
  return cudaGetLastError();
}

template <int N>
cudaError_t solve_n(const DevMesh &m, int prec, const void *fac, void *r, const void *q, void *z,
                    const double *alpha, double *part_rz, double *part_rr, const int *done, TnWait *zerr,
                    cudaStream_t st) {
  if (prec == TN_F64)
    return q ? solve_nt<N, double, true>(m, fac, r, q, z, alpha, part_rz, part_rr, done, zerr, st)
             : solve_nt<N, double, false>(m, fac, r, q, z, alpha, part_rz, part_rr, done, zerr, st);
  return q ? solve_nt<N, float, true>(m, fac, r, q, z, alpha, part_rz, part_rr, done, zerr, st)
           : solve_nt<N, float, false>(m, fac, r, q, z, alpha, part_rz, part_rr, done, zerr, st);
}

template <int N, typename T, bool UPD>
cudaError_t solve_batch_nt(const DevMesh *meshes, const int2 *work, int nwork, const long long *fac_off,
                           const long long *dof_off, const void *fac, void *r, const void *q, void *z,
                           const double *alpha, double *part_rz, double *part_rr, const int *done, TnWait *zerr,
                           cudaStream_t st) {
  constexpr size_t sm = zline_smem<N, T>();
  cudaError_t err = zline_smem_optin(zline_solve_batch_kernel<N, T, T, UPD>, sm);
  if (err != cudaSuccess) return err;
  zline_solve_batch_kernel<N, T, T, UPD><<<(nwork + 3) / 4, 128, sm, st>>>(
      meshes, work, nwork, fac_off, dof_off, (const T *)fac, (T *)r, (const T *)q, (T *)z, alpha, part_rz,
      part_rr, done, zerr);
  return cudaGetLastError();
}

template <int N>
cudaError_t solve_batch_n(int prec, const DevMesh *meshes, const int2 *work, int nwork, const long long *fac_off,
                          const long long *dof_off, const void *fac, void *r, const void *q, void *z,
                          const double *alpha, double *part_rz, double *part_rr, const int *done, TnWait *zerr,
                          cudaStream_t st) {
  if (prec == TN_F64)
    return q ? solve_batch_nt<N, double, true>(meshes, work, nwork, fac_off, dof_off, fac, r, q, z, alpha,
                                               part_rz, part_rr, done, zerr, st)
             : solve_batch_nt<N, double, false>(meshes, work, nwork, fac_off, dof_off, fac, r, q, z, alpha,
                                                part_rz, part_rr, done, zerr, st);
  return q ? solve_batch_nt<N, float, true>(meshes, work, nwork, fac_off, dof_off, fac, r, q, z, alpha, part_rz,
                                            part_rr, done, zerr, st)
           : solve_batch_nt<N, float, false>(meshes, work, nwork, fac_off, dof_off, fac, r, q, z, alpha,
                                             part_rz, part_rr, done, zerr, st);
}

}  // namespace

cudaError_t tn_zline_blocks(const DevMesh &m, double *blk, cudaStream_t st) {
  switch (m.N) {
#define TN_CASE(NN)                                                                        \
  case NN:                                                                                 \
    zline_blocks_kernel<NN><<<m.E, ((NN * NN + 31) / 32) * 32, 0, st>>>(m, blk);           \
    return cudaGetLastError();
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}

size_t tn_zline_block_bytes(const DevMesh &m) {
  const size_t M = 3 * m.N;
  return (size_t)m.ncol * m.N * m.N * m.nslab * 2 * M * M * sizeof(double);
}

size_t tn_zline_factor_entries(const DevMesh &m) {
  return (size_t)m.ncol * m.N * m.N * m.nslab * zrec(3 * m.N);
}

size_t tn_zline_factor_bytes(const DevMesh &m) { return tn_zline_factor_entries(m) * sizeof(float); }

int tn_zline_partials(const DevMesh &m) { return (m.ncol * m.N * m.N + 3) / 4; }

cudaError_t tn_zline_setup(const DevMesh &m, double *blk, float *fac, double *fac64, int *status,
                           cudaStream_t st) {
  switch (m.N) {
    case 3: return setup_n<3>(m, blk, fac, fac64, status, st);
    case 4: return setup_n<4>(m, blk, fac, fac64, status, st);
    case 5: return setup_n<5>(m, blk, fac, fac64, status, st);
    case 6: return setup_n<6>(m, blk, fac, fac64, status, st);
    case 7: return setup_n<7>(m, blk, fac, fac64, status, st);
    case 8: return setup_n<8>(m, blk, fac, fac64, status, st);
    case 9: return setup_n<9>(m, blk, fac, fac64, status, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t tn_zline_solve(const DevMesh &m, int prec, const void *fac, void *r, const void *q, void *z,
                           const double *alpha, double *part_rz, double *part_rr, const int *done, TnWait *zerr,
                           cudaStream_t st) {
  switch (m.N) {
#define TN_CASE(NN) \
    case NN: return solve_n<NN>(m, prec, fac, r, q, z, alpha, part_rz, part_rr, done, zerr, st);
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t tn_zline_solve_batch(int N, int prec, const DevMesh *meshes, const int2 *work, int nwork,
                                 const long long *fac_off, const long long *dof_off, const void *fac, void *r,
                                 const void *q, void *z, const double *alpha, double *part_rz, double *part_rr,
                                 const int *done, TnWait *zerr, cudaStream_t st) {
  if (nwork <= 0) return cudaSuccess;
  switch (N) {
#define TN_CASE(NN)                                                                                   \
    case NN:                                                                                         \
      return solve_batch_n<NN>(prec, meshes, work, nwork, fac_off, dof_off, fac, r, q, z, alpha, part_rz, \
                               part_rr, done, zerr, st);
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}
