// Set-up of the grouped-line block preconditioner: the blocks of the groups and
// their factors.
#include "tn_device.h"
#include "tn_internal.h"
#include "tn_precond.h"
#include "tn_zgroup.h"

// device constants are per translation unit (no relocatable device code):
// this file keeps its own copy of the LGL tables
__constant__ LglTables c_lgl_zf;

cudaError_t tn_upload_lgl_zgfactor(const LglTables *t) { return cudaMemcpyToSymbol(c_lgl_zf, t, sizeof(LglTables)); }

namespace {

#define LD(a, b) c_lgl_zf.D[N][(a) * N + (b)]
#define LW(a) c_lgl_zf.w[N][(a)]

// The lines through the matching nodes of two columns that share a lateral
// face are coupled by that face's interior-penalty and flux terms (Eqs.
// (numflux), (penalty)), which the single-line blocks leave out; with the
// penalty ~ C (p + 1)^2 / h these are the stiffest couplings left.  A group
// is a set of lines joined by such face matches (1 to 4 lines: a node inside
// a column face, on a column edge or at a corner where up to four columns
// meet); its block is the exact principal sub-matrix of A on all its lines,
// again block tridiagonal over the slabs, with 3 g N unknowns per slab and
// the cross-line face terms in the diagonal blocks.

// Cross-line block of element e = (s, c), lateral face f and face position t:
// rows = the line through the face node (this element), columns = the line
// through the matching node of the neighbour column (same slab):
//   -1/2 V^T W Tr_ext + 1/2 Tr^T W V_ext - V^T W Pen V_ext
// restricted to the two lines (the neighbour's traction and this element's
// test traction reduce to the zeta derivative and the diagonal xi / eta
// derivative entries on a line).  Zero where f has no neighbour.
template <int N>
__global__ void zgroup_cross_kernel(const DevMesh m, double *__restrict__ xblk) {
  constexpr int M = 3 * N, N2 = N * N;
  const int e = blockIdx.x, t = threadIdx.x % N, f = threadIdx.x / N;
  if (f >= 4) return;
  const int s = e / m.ncol, c = e - s * m.ncol;
  double *X = xblk + (((size_t)e * 4 + f) * N + t) * M * M;
  for (int q = 0; q < M * M; ++q) X[q] = 0.0;
  const int nbc = m.colnb[4 * c + f];
  if (nbc < 0) return;
  const int d = f >> 1, sd = f & 1, end = sd ? N - 1 : 0;
  const int i = d == 0 ? end : t, j = d == 0 ? t : end;
  const int code = m.colnbf[4 * c + f];
  const int f2 = code & 3, d2 = f2 >> 1, end2 = (f2 & 1) ? N - 1 : 0;
  const int a2 = (code >> 2) ? N - 1 - t : t;
  const int i2 = d2 == 0 ? end2 : a2, j2 = d2 == 0 ? a2 : end2;
  const double *cg = m.colgeo + (size_t)c * CG_NF * N2;
  const double *cg2 = m.colgeo + (size_t)nbc * CG_NF * N2;
  const int q1 = j * N + i, q2 = j2 * N + i2;
  const double ixx = cg[CG_IXX * N2 + q1], ixy = cg[CG_IXY * N2 + q1];
  const double iex = cg[CG_IEX * N2 + q1], iey = cg[CG_IEY * N2 + q1], det2 = cg[CG_DET * N2 + q1];
  const double jxx = cg2[CG_IXX * N2 + q2], jxy = cg2[CG_IXY * N2 + q2];
  const double jex = cg2[CG_IEX * N2 + q2], jey = cg2[CG_IEY * N2 + q2];
  const double *sg = m.slabgeo + (size_t)s * SG_NF * N;
  double dz[N];
  for (int k = 0; k < N; ++k) dz[k] = sg[SG_DZ * N + k];
  const int L = m.slab_layer[s];  // both sides lie in slab s: one material
  const double c11 = m.layer_c[3 * L], c12 = m.layer_c[3 * L + 1], c44 = m.layer_c[3 * L + 2];
  const double rx = d == 0 ? ixx : iex, ry = d == 0 ? ixy : iey;
  const double mag = sqrt(rx * rx + ry * ry);
  const double n[3] = {(sd ? 1.0 : -1.0) * rx / mag, (sd ? 1.0 : -1.0) * ry / mag, 0.0};
  const double sx = d2 == 0 ? jxx : jex, sy = d2 == 0 ? jxy : jey;
  const double h = 2.0 / mag, h2 = 2.0 / sqrt(sx * sx + sy * sy);
  const double sig = (double)((m.p + 1) * (m.p + 1)) * m.penC / (h < h2 ? h : h2);
  const double Dii = LD(i, i), Djj = LD(j, j), Dii2 = LD(i2, i2), Djj2 = LD(j2, j2);
  const double wt = d == 0 ? LW(j) : LW(i);
  for (int k = 0; k < N; ++k) {
    const double Wk = wt * LW(k) * det2 * dz[k] * mag;
    for (int k2 = 0; k2 < N; ++k2) {
      const double Wk2 = wt * LW(k2) * det2 * dz[k2] * mag;
      // neighbour basis (i2, j2, k2) at its node (i2, j2, k); own basis (i, j, k) at (i, j, k2)
      const double l2[3] = {k2 == k ? Dii2 : 0.0, k2 == k ? Djj2 : 0.0, LD(k, k2)};
      const double l1[3] = {k == k2 ? Dii : 0.0, k == k2 ? Djj : 0.0, LD(k2, k)};
      double g2[3], g1[3];
      phys(l2, jxx, jxy, jex, jey, dz[k], g2);
      phys(l1, ixx, ixy, iex, iey, dz[k2], g1);
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
          double v = -0.5 * Wk * Qab(a, b, n, g2, c11, c12, c44) + 0.5 * Wk2 * Qab(b, a, n, g1, c11, c12, c44);
          if (k == k2) v -= Wk * sig * Qab(a, b, n, n, c11, c12, c44);
          X[(a * N + k) * M + b * N + k2] = v;
        }
    }
  }
}

// block Cholesky along the slabs of one group, S_s the Schur complements:
//   S_s = D_s - V_s C V_s^T,  C = U_{s-1}^T W_{s-1}
// one CTA per group; then the FP32 records and the FP64 factors.  S_s is
// inverted by symmetric sweeps (Gauss-Jordan without exchanges, pivots = those
// of the Cholesky factorisation) on 4 x 4 tiles of its lower triangle kept in
// registers, one thread per tile: a sweep exchanges one column through shared
// memory and costs one barrier.  Bound by the FP64 pipe of the SM that has a
// 4-line group (20 operations per thread and sweep; 72 - 86 % busy).  Set-up
// of the factors with Cholesky columns in turn in global memory, the triangle
// inverted by columns and its product, before -> after: 2.0 M unknowns, p = 6
// 34.8 -> 19 ms; p = 4, 21 layers 10.2 -> 3.6 ms.
template <int N, int G>
struct ZgFactor {
  static constexpr int M = 3 * N, MG = G * M, C6 = 6 * G, TT = (MG + 3) / 4, TILES = TT * (TT + 1) / 2;
  static constexpr int NT = (TILES + 31) / 32 * 32;
  // doubles of shared memory: S^{-1} (before it: C V^T), (Q | W)^T, C, X, Y, two pivot columns
  static constexpr int WORDS = MG * MG + 2 * C6 * MG + C6 * C6 + 4 * MG + 2 * 4 * TT;
};

template <int N, int G>
__global__ void __launch_bounds__(ZgFactor<N, G>::NT)
zgroup_factor_kernel(const DevMesh m, const int4 *__restrict__ glines, const long long *__restrict__ gfac,
                     const long long *__restrict__ gfac64, int gbase, const double *__restrict__ blk,
                     const double *__restrict__ xblk, float *__restrict__ fac, double *__restrict__ fac64,
                     int *__restrict__ status) {
  using Z = ZgFactor<N, G>;
  constexpr int M = Z::M, MG = Z::MG, C6 = Z::C6, TT = Z::TT, NT = Z::NT, N2 = N * N, MGP = pad4(MG);
  const int grp = gbase + blockIdx.x, tid = threadIdx.x, S = m.nslab;
  extern __shared__ __align__(16) double fsm[];
  double *const Gs = fsm, *const Qs = Gs + MG * MG, *const Cm = Qs + 2 * C6 * MG, *const Xs = Cm + C6 * C6;
  double *const Ys = Xs + 3 * MG, *const colb = Ys + MG, *const Tc = Gs;
  __shared__ int lid[4], xof[4][4];
  __shared__ double piv[2];
  if (tid < 4) {
    const int4 L4 = glines[grp];
    lid[tid] = tid == 0 ? L4.x : (tid == 1 ? L4.y : (tid == 2 ? L4.z : L4.w));
  }
  __syncthreads();
  if (tid < 16) {  // which face block couples line t1 (rows) to line t2 (columns)
    const int t1 = tid >> 2, t2 = tid & 3;
    int x = -1;
    if (t1 < G && t2 < G && t1 != t2) {
      const int c1 = lid[t1] / N2, qq = lid[t1] - c1 * N2, i1 = qq % N, j1 = qq / N;
      for (int f = 0; f < 4; ++f) {
        const int nbc = m.colnb[4 * c1 + f];
        const int d = f >> 1, end = (f & 1) ? N - 1 : 0;
        if (nbc < 0 || (d == 0 ? i1 : j1) != end) continue;
        const int tp = d == 0 ? j1 : i1;
        const int code = m.colnbf[4 * c1 + f], f2 = code & 3, d2 = f2 >> 1, end2 = (f2 & 1) ? N - 1 : 0;
        const int a2 = (code >> 2) ? N - 1 - tp : tp;
        const int i2 = d2 == 0 ? end2 : a2, j2 = d2 == 0 ? a2 : end2;
        if (nbc * N2 + j2 * N + i2 == lid[t2]) x = f * N + tp;
      }
    }
    xof[t1][t2] = x;
  }
  __syncthreads();
  float *const f32 = fac + gfac[grp];
  double *const f64 = fac64 + gfac64[grp];
  constexpr int RS = zp_rec(MG, G), LP = zlp(MG), WS = zp_ws(G);
  constexpr int SR = zg_srec(MG, G), QR = zg_qrec(MG, G), KR = zg_krec(G), KP = zg_kpart(G), KS = zg_ld(G);
  constexpr int LC = pad4(zg_circ(MG));
  const long long qo = zg_qoff(MG, G, S), ko = zg_koff(MG, G, S);
  // O_s of line l (rows: slab s)
  auto Oblk = [&](int l, int s) { return blk + (((size_t)lid[l] * S + s) * 2 + 1) * M * M; };
  // column j of V_s applied: sum_p V_s[p][j] f(p), f indexed by rows of the
  // group; X[a][t] = O_{s-1}[(a, 0), t], Y[t] = O_s[t, (b, N - 1)] of t's component b
  auto dotV = [&](int j, auto f) {
    const int l = j / 6, jj = j - l * 6;
    if (jj < 3) return f(l * M + jj * N + N - 1);
    const double *X = Xs + (jj - 3) * MG + l * M;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < N - 1; ++k) acc += X[(jj - 3) * N + k] * f(l * M + (jj - 3) * N + k);
#pragma unroll
    for (int b = 0; b < 3; ++b) acc += X[b * N + N - 1] * f(l * M + b * N + N - 1);
    return acc;
  };
  // column j of U_s applied
  auto dotU = [&](int j, auto f) {
    const int l = j / 6, jj = j - l * 6;
    if (jj >= 3) return f(l * M + (jj - 3) * N);
    double acc = 0.0;
#pragma unroll
    for (int k = 1; k < N; ++k) acc += Ys[l * M + jj * N + k] * f(l * M + jj * N + k);
    return acc;
  };
  // this thread's tile: rows 4 ti .., columns 4 tj ..
  int ti = 0, tj = tid;
  while (tj > ti && ti < TT) {
    tj -= ti + 1;
    ++ti;
  }
  const bool tile = tid < Z::TILES;
  for (int s = 0; s < S; ++s) {
    for (int q = tid; q < 3 * MG; q += NT) {
      const int a = q / MG, t = q - a * MG, l = t / M, tl = t - l * M;
      Xs[q] = s > 0 ? Oblk(l, s - 1)[(a * N) * M + tl] : 0.0;
    }
    for (int t = tid; t < MG; t += NT) {
      const int l = t / M, tl = t - l * M, b = tl / N, k = tl - b * N;
      Ys[t] = s + 1 < S && k != 0 ? Oblk(l, s)[tl * M + b * N + N - 1] : 0.0;
    }
    __syncthreads();
    if (s > 0) {  // C V^T
      for (int q = tid; q < C6 * MG; q += NT) {
        const int i = q / MG, t = q - i * MG, l = t / M, tl = t - l * M, b = tl / N, k = tl - b * N;
        const double *c = Cm + i * C6 + 6 * l;
        double v = k == N - 1 ? c[b] : 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) v += c[3 + a] * Xs[a * MG + t];
        Tc[q] = v;
      }
      __syncthreads();
    }
    // the tile of S_s: line blocks, cross-line face blocks, minus V C V^T
    double A[4][4];
    if (tile) {
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int r = 4 * ti + x, cc = 4 * tj + y;
          double v = 0.0;
          if (r < MG && cc < MG) {
            const int t1 = r / M, t2 = cc / M, rr = r - t1 * M, c2 = cc - t2 * M;
            if (t1 == t2) {
              v = blk[(((size_t)lid[t1] * S + s) * 2 + 0) * M * M + rr * M + c2];
            } else if (xof[t1][t2] >= 0) {
              const size_t e = (size_t)s * m.ncol + lid[t1] / N2;
              v = xblk[(e * 4 * N + xof[t1][t2]) * M * M + rr * M + c2];
            }
            if (s > 0) {
              const double *T = Tc + 6 * t1 * MG + cc;
              double w = rr % N == N - 1 ? T[(rr / N) * MG] : 0.0;
#pragma unroll
              for (int a = 0; a < 3; ++a) w += Xs[a * MG + r] * T[(3 + a) * MG];
              v -= w;
            }
          }
          A[x][y] = v;
        }
      if (ti == tj) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = x + 1; y < 4; ++y) A[x][y] = A[y][x];
      }
    }
    // sweep row and column k: A_ij -= A_ik A_kj / A_kk, A_ik /= A_kk, A_kk =
    // -1 / A_kk.  Row and column k are cleared and -1 stands in for A_kk in
    // the column, which makes all of it the one update.
    for (int kt = 0; kt < TT; ++kt) {
#pragma unroll
      for (int kr = 0; kr < 4; ++kr) {
        const int k = 4 * kt + kr;
        if (k >= MG) break;
        double *const c = colb + (k & 1) * 4 * TT;
        if (tile && tj == kt) {
          if (ti == kt) {
            double dv = A[kr][kr];
            if (!(dv > 0.0)) {
              atomicExch(status, 1);
              dv = 1e-300;
            }
            piv[k & 1] = 1.0 / dv;
            A[kr][kr] = -1.0;
          }
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            c[4 * ti + x] = A[x][kr];
            A[x][kr] = 0.0;
            if (ti == kt) A[kr][x] = 0.0;
          }
        } else if (tile && ti == kt) {
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            c[4 * tj + y] = A[kr][y];
            A[kr][y] = 0.0;
          }
        }
        __syncthreads();
        if (tile) {
          const double p = piv[k & 1];
          double ci[4], cj[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            ci[x] = c[4 * ti + x] * p;
            cj[x] = c[4 * tj + x];
          }
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) A[x][y] -= ci[x] * cj[y];
        }
      }
    }
    if (tile) {
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int r = 4 * ti + x, cc = 4 * tj + y;
          if (r < MG && cc <= r) {
            Gs[r * MG + cc] = -A[x][y];
            Gs[cc * MG + r] = -A[x][y];
          }
        }
    }
    __syncthreads();
    float *const R = f32 + (long long)s * RS;
    for (int q = tid; q < MG * MG; q += NT) {  // S^{-1}, packed lower triangle
      const int cc = q / MG, r = q - cc * MG;
      if (r >= cc) R[zcol(MG, cc) + r - cc] = (float)Gs[q];
    }
    for (int q = MG * (MG + 1) / 2 + tid; q < LP; q += NT) R[q] = 0.0f;
    for (int q = tid; q < 8 * MG; q += NT) {  // factors of O_{s-1}
      const int t = q >> 3, j = q & 7, l = t / M, tl = t - l * M, tk = tl % N;
      double v = 0.0;
      if (s > 0 && (j & 3) < 3) {
        const double *O = Oblk(l, s - 1);
        if (j < 4) v = O[(j * N) * M + tl];                        // X[t][a] = O[(a, 0), t]
        else if (tk != 0) v = O[tl * M + (j - 4) * N + (N - 1)];  // Y[t][b] = O[t, (b, N - 1)]
      }
      R[LP + q] = (float)v;
    }
    double *Sd = f64 + (long long)s * SR;
    for (int q = tid; q < SR; q += NT) {
      double v = 0.0;
      if (q < zg_circ(MG)) {
        const int mm = q / MG, t = q - mm * MG, c = t + mm < MG ? t + mm : t + mm - MG;
        v = Gs[t * MG + c];
      } else if (q >= LC) {
        const int l = (q - LC) / 16, i = (q - LC) - l * 16;
        if (i < 3) {
          v = Ys[l * M + i * N + 1] / c_lgl_zf.D[N][1];  // Y[(b, 1)][b] / D(0, 1)
        } else if (i < 6) {
          const int a = i - 3;  // X[(a, 0)][a] / D(N-1, 0)
          v = Xs[a * MG + l * M + a * N] / c_lgl_zf.D[N][(N - 1) * N];
        } else if (i < 15) {
          const int b = (i - 6) / 3, a = (i - 6) % 3;
          v = Xs[a * MG + l * M + b * N + N - 1];
        }
      }
      Sd[q] = v;
    }
    // (Q_s | W_s)^T = (V_s | U_s)^T S_s^{-1}
    double *Qd = f64 + qo + (long long)s * QR;
    for (int q = tid; q < QR; q += NT) {
      const int j = q / MGP, t = q - j * MGP;
      double v = 0.0;
      if (t < MG) {
        auto row = [&](int p) { return Gs[p * MG + t]; };
        if (j < C6) {
          if (s > 0) v = dotV(j, row);
        } else if (s + 1 < S) {
          v = dotU(j - C6, row);
        }
        Qs[j * MG + t] = v;
      }
      Qd[q] = v;
    }
    __syncthreads();
    const double *const Ws = Qs + C6 * MG;
    for (int q = tid; q < MG * WS; q += NT) {  // W_s by rows
      const int t = q / WS, j = q - t * WS;
      R[LP + 8 * MG + q] = j < C6 ? (float)Ws[j * MG + t] : 0.0f;
    }
    // K_s = W_s^T V_s, H_s = V_s^T Q_s
    double *Kd = f64 + ko + (long long)s * KR;
    for (int q = tid; q < KR; q += NT) {
      double v = 0.0;
      if (s > 0) {
        if (q < KP) {
          const int i = q / KS, j = q - i * KS;
          if (i < C6 && j < C6) v = dotV(j, [&](int p) { return Ws[i * MG + p]; });
        } else {
          const int i = (q - KP) / C6, j = (q - KP) - i * C6;
          v = dotV(i, [&](int p) { return Qs[j * MG + p]; });
        }
      }
      Kd[q] = v;
    }
    for (int q = tid; q < C6 * C6; q += NT) {  // C = U_s^T W_s of the next slab
      const int i = q / C6, j = q - i * C6;
      Cm[q] = dotU(i, [&](int p) { return Ws[j * MG + p]; });
    }
    __syncthreads();
  }
}

template <int N, int G>
cudaError_t launch_factor(const DevMesh &m, const ZGroupPlan &p, const ZGroupDev &gd, int inst, const double *blk,
                          const double *xblk, float *fac, double *fac64, int *status, cudaStream_t st) {
  using Z = ZgFactor<N, G>;
  constexpr size_t sm = sizeof(double) * (size_t)Z::WORDS;
  if (sm > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(zgroup_factor_kernel<N, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  zgroup_factor_kernel<N, G><<<p.inst_n[(size_t)inst * 5 + G], Z::NT, sm, st>>>(
      m, gd.lines, gd.fac_off, gd.fac64_off, p.inst_start[(size_t)inst * 5 + G], blk, xblk, fac, fac64, status);
  return cudaGetLastError();
}

template <int N>
cudaError_t zgroup_setup_n(const DevMesh &m, const ZGroupPlan &p, const ZGroupDev &gd, int inst, double *blk,
                           double *xblk, float *fac, double *fac64, int *status, cudaStream_t st) {
  cudaError_t err = tn_zline_blocks(m, blk, st);
  if (err != cudaSuccess) return err;
  zgroup_cross_kernel<N><<<m.E, ((4 * N + 31) / 32) * 32, 0, st>>>(m, xblk);
  err = cudaGetLastError();
  // the four group sizes at once: the 4-line groups (few, long) on st, the
  // others on side streams forked from it
  if (err == cudaSuccess) err = cudaEventRecord(gd.fork, st);
  bool used[3] = {false, false, false};
  for (int g = 4; g >= 1 && err == cudaSuccess; --g) {
    if (!p.inst_n[(size_t)inst * 5 + g]) continue;
    cudaStream_t sg = st;
    if (g < 4) {
      sg = gd.side[g - 1];
      err = cudaStreamWaitEvent(sg, gd.fork, 0);
      used[g - 1] = true;
      if (err != cudaSuccess) break;
    }
    switch (g) {
      case 1: err = launch_factor<N, 1>(m, p, gd, inst, blk, xblk, fac, fac64, status, sg); break;
      case 2: err = launch_factor<N, 2>(m, p, gd, inst, blk, xblk, fac, fac64, status, sg); break;
      case 3: err = launch_factor<N, 3>(m, p, gd, inst, blk, xblk, fac, fac64, status, sg); break;
      default: err = launch_factor<N, 4>(m, p, gd, inst, blk, xblk, fac, fac64, status, sg);
    }
  }
  for (int k = 0; k < 3 && err == cudaSuccess; ++k) {
    if (!used[k]) continue;
    err = cudaEventRecord(gd.join[k], gd.side[k]);
    if (err == cudaSuccess) err = cudaStreamWaitEvent(st, gd.join[k], 0);
  }
  return err;
}

}  // namespace

size_t tn_zgroup_cross_bytes(const DevMesh &m) {
  const size_t M = 3 * m.N;
  return (size_t)m.E * 4 * m.N * M * M * sizeof(double);
}

cudaError_t tn_zgroup_setup(const DevMesh &m, const ZGroupPlan &p, const ZGroupDev &gd, int inst, double *blk,
                            double *xblk, float *fac, double *fac64, int *status, cudaStream_t st) {
  switch (m.N) {
#define TN_CASE(NN) \
    case NN: return zgroup_setup_n<NN>(m, p, gd, inst, blk, xblk, fac, fac64, status, st);
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}
