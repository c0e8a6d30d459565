// The DG elasticity operator y = A u (Sec. 2.2) in FP64 and FP32: the kernels
// of tn_apply_operator and of every Krylov iteration.
//
//   y = sum_m D_m^T F^m  -  sum_faces W ( 1/2 (T + T_ext) - sigma P[[u]] )
//   F^m_j = J^-1[m][a] (Y : S_eff)^{aj},  S_eff = w detJ sym(grad u) + L,
//   L = sum_faces W (-1/2) sym(n (x) [[u]])
// (weak form of Eq. (dg_residuals); the terms are named in kernels.cu.)
//
// Two launches.  apply_elem_kernel forms everything an element can know from
// its own field and its neighbours' face values, and writes the traction
// term its own stress contributes to each neighbour (1/2 W T at the face
// nodes) to a trace buffer; trace_add_kernel adds the terms the neighbours
// left.  So a neighbour's gradient is never rebuilt: an element reads 6 N^2
// face nodes of its neighbours instead of six whole elements, and every
// traction is formed once.
//
// Algebra that keeps divisions and square roots out of the kernel (FP64 ones
// cost tens of operations): with r = grad xi^d (unnormalised) at a lateral
// face node and the tangential weights wt,
//   W n = sgn wt det2 dz r,     W / min(h, h_ext) n n^T = wt det2 dz rho r r^T,
// rho a table of the column (CG_RXI, CG_RETA); on zeta faces W n =
// sgn wt det2 e_z and 1 / min(h, h_ext) a table of the slab (SG_HINV).  The
// lifted strain L is a change of the logical derivative along d at the two
// ends of a line: d_d u -> d_d u - 1/2 sgn [[u]] / w_end.
//
// Line products use the centro-antisymmetry of the LGL derivative matrix,
// D[N-1-a][N-1-b] = -D[a][b]: on the even and odd parts of a line they need
// about half the multiplications (36 instead of 49 operations at N = 7).
//
// Bound: neither HBM nor the FMA pipe.  FP32 (2.0 M unknowns, p = 6): 7.3 + 2.4 M
// warp instructions against 43.6 M of the form that rebuilt the neighbours'
// tractions; 17 + 7 us for the two launches (51 us before).  59 M unknowns, p = 8: 335 + 108 us (1420 us).
// FP64 is bound by its pipe (two FMAs per clock and SM): 8.0 M unknowns,
// p = 5: 1.10 ms (3.11 ms), about 65 FP64 operations per unknown (204).
// The second launch starts while the first drains (its reads of the mesh
// overlap): 24 instead of 31 us per FP32 apply at 2.0 M unknowns.
#include <algorithm>
#include <initializer_list>

#include "tn_device.h"
#include "tn_internal.h"

namespace {

// even-odd form of D (0) and D^T (1) per N: for a < N/2
//   em[a][b] = 1/2 (D[a][b] - D[a][N-1-b]),  b < N/2
//   ep[a][b] = 1/2 (D[a][b] + D[a][N-1-b]),  b < N/2;  ep[a][N/2] = D[a][N/2] for odd N
//   mid[b]   = D[N/2][b],                    b < N/2 (odd N)
template <typename T>
struct EoTab {
  T em[4][4], ep[4][5], mid[4];
};
template <typename T>
struct ApplyTabs {
  EoTab<T> eo[2];
  T w[TN_MAX_N];
  T whalf;  // 1 / (2 w_end)
};

__constant__ ApplyTabs<double> c_t64[TN_MAX_N + 1];
__constant__ ApplyTabs<float> c_t32[TN_MAX_N + 1];

template <typename T> __device__ __forceinline__ const ApplyTabs<T> &tabs(int N);
template <> __device__ __forceinline__ const ApplyTabs<double> &tabs<double>(int N) { return c_t64[N]; }
template <> __device__ __forceinline__ const ApplyTabs<float> &tabs<float>(int N) { return c_t32[N]; }

// This file is compiled without floating-point contraction and writes its
// fused operations out, so that the kernels below (and their occupancy
// variants) round alike and give bit-identical results.
template <typename T> __device__ __forceinline__ T fm(T a, T b, T c);
template <> __device__ __forceinline__ double fm(double a, double b, double c) { return fma(a, b, c); }
template <> __device__ __forceinline__ float fm(float a, float b, float c) { return fmaf(a, b, c); }

// out = D v (TR = 0) or D^T v (TR = 1) along one line of N nodes
template <int N, int TR, typename T>
__device__ __forceinline__ void line_eo(const T v[N], T out[N]) {
  constexpr int H = N / 2;
  const EoTab<T> &t = tabs<T>(N).eo[TR];
  T s[H], d[H];
#pragma unroll
  for (int a = 0; a < H; ++a) {
    s[a] = v[a] + v[N - 1 - a];
    d[a] = v[a] - v[N - 1 - a];
  }
  T mid = T(0);
#pragma unroll
  for (int a = 0; a < H; ++a) {
    T p = t.em[a][0] * d[0], q = t.ep[a][0] * s[0];
#pragma unroll
    for (int b = 1; b < H; ++b) {
      p = fm(t.em[a][b], d[b], p);
      q = fm(t.ep[a][b], s[b], q);
    }
    if (N & 1) q = fm(t.ep[a][H], v[H], q);
    out[a] = p + q;
    out[N - 1 - a] = p - q;
    if (N & 1) mid = a == 0 ? t.mid[0] * d[0] : fm(t.mid[a], d[a], mid);
  }
  if (N & 1) out[H] = mid;
}

template <typename T> struct Moduli { T c11, c12, c44; };
template <typename T> struct Map2 { T xx, xy, ex, ey; };  // d(xi, eta)/d(x, y)
template <typename T> struct Stress { T xx, yy, zz, xy, xz, yz; };

// stress of the symmetric part of the gradient with logical derivatives
// d0 (xi), d1 (eta) and d2 (already times dzeta/dz)
template <typename T>
__device__ __forceinline__ Stress<T> stress_of(const Map2<T> &J, const T d0[3], const T d1[3], const T d2[3],
                                               const Moduli<T> &C) {
  const T gxx = fm(J.xx, d0[0], J.ex * d1[0]), gyy = fm(J.xy, d0[1], J.ey * d1[1]), gzz = d2[2];
  const T gxy = fm(J.xx, d0[1], fm(J.ex, d1[1], fm(J.xy, d0[0], J.ey * d1[0])));
  const T gxz = fm(J.xx, d0[2], fm(J.ex, d1[2], d2[0])), gyz = fm(J.xy, d0[2], fm(J.ey, d1[2], d2[1]));
  const T tr = C.c12 * ((gxx + gyy) + gzz), df = C.c11 - C.c12;
  return {fm(df, gxx, tr), fm(df, gyy, tr), fm(df, gzz, tr), C.c44 * gxy, C.c44 * gxz, C.c44 * gyz};
}

// fluxes of a node (F0: xi, F1: eta, F2: zeta), wz = w det2, wJ = wz dz
template <typename T>
__device__ __forceinline__ void node_flux(const Map2<T> &J, const Stress<T> &s, T wz, T wJ, T F0[3], T F1[3], T F2[3]) {
  const T ax = wJ * J.xx, ay = wJ * J.xy, ex = wJ * J.ex, ey = wJ * J.ey;
  F0[0] = fm(ax, s.xx, ay * s.xy);
  F0[1] = fm(ax, s.xy, ay * s.yy);
  F0[2] = fm(ax, s.xz, ay * s.yz);
  F1[0] = fm(ex, s.xx, ey * s.xy);
  F1[1] = fm(ex, s.xy, ey * s.yy);
  F1[2] = fm(ex, s.xz, ey * s.yz);
  F2[0] = wz * s.xz;
  F2[1] = wz * s.yz;
  F2[2] = wz * s.zz;
}

// lateral face node with r = grad xi^d, wd = wt det2 dz, sw = +-hf wd, pw =
// wd C (p + 1)^2 rho: the traction term tw (hf W T) and the surface term of
// this element, penalty - tw
template <typename T>
__device__ __forceinline__ void lateral_terms(T rx, T ry, const Stress<T> &s, const Moduli<T> &C, T sw, T pw,
                                              const T jump[3], T tw[3], T surf[3]) {
  const T sx = sw * rx, sy = sw * ry;
  tw[0] = fm(sx, s.xx, sy * s.xy);
  tw[1] = fm(sx, s.xy, sy * s.yy);
  tw[2] = fm(sx, s.xz, sy * s.yz);
  const T rxx = rx * rx, ryy = ry * ry, c = (C.c12 + C.c44) * (rx * ry);
  surf[0] = fm(pw, fm(fm(C.c11, rxx, C.c44 * ryy), jump[0], c * jump[1]), -tw[0]);
  surf[1] = fm(pw, fm(c, jump[0], fm(C.c11, ryy, C.c44 * rxx) * jump[1]), -tw[1]);
  surf[2] = fm(pw, (C.c44 * (rxx + ryy)) * jump[2], -tw[2]);
}

// zeta face node: sw = +-hf w det2, pw = w det2 C (p + 1)^2 / min(h), p11 and
// p44 the moduli averaged over the face
template <typename T>
__device__ __forceinline__ void zeta_terms(const Stress<T> &s, T sw, T pw, T p11, T p44, const T jump[3], T tw[3],
                                           T surf[3]) {
  tw[0] = sw * s.xz;
  tw[1] = sw * s.yz;
  tw[2] = sw * s.zz;
  surf[0] = fm(pw * p44, jump[0], -tw[0]);
  surf[1] = fm(pw * p44, jump[1], -tw[1]);
  surf[2] = fm(pw * p11, jump[2], -tw[2]);
}

// what a CTA needs of one of its elements, staged in shared memory
template <typename T>
struct FaceI {
  const T *nbu;    // the neighbour's field at face position (0, 0); nullptr: no neighbour
  int ns1;         // neighbour node of position (t1, t2): + t1 ns1 + t2 (N^2 lateral, N zeta)
  T ju, hf;        // [[u]] = ju u - u_ext, own traction term hf T: (1, 1/2) interior, (2, 1) Dirichlet, (0, 0) Neumann
};
template <typename T>
struct ElemI {
  const T *u, *cg, *sg;
  T *y, *tr;
  Moduli<T> C;
  T p11[2], p44[2];  // averaged moduli of the zeta faces (bottom, top)
  T sp;              // C (p + 1)^2
  FaceI<T> f[6];
};

template <typename T> struct Geo;
template <> struct Geo<double> {
  static __device__ __forceinline__ const double *col(const DevMesh &m) { return m.colgeo; }
  static __device__ __forceinline__ const double *slab(const DevMesh &m) { return m.slabgeo; }
  static __device__ __forceinline__ const double *lay(const DevMesh &m) { return m.layer_c; }
};
template <> struct Geo<float> {
  static __device__ __forceinline__ const float *col(const DevMesh &m) { return m.colgeo32; }
  static __device__ __forceinline__ const float *slab(const DevMesh &m) { return m.slabgeo32; }
  static __device__ __forceinline__ const float *lay(const DevMesh &m) { return m.layer_c32; }
};

// face f of element (s, c) of mesh m, whose field starts at u
template <int N, typename T>
__device__ __forceinline__ void face_setup(const DevMesh &m, const T *u, int s, int c, int f, ElemI<T> &E) {
  constexpr int N2 = N * N, n = N * N2;
  FaceI<T> &F = E.f[f];
  bool fixed = false;
  F.nbu = nullptr;
  F.ns1 = 1;
  if (f < 4) {
    const int nbc = m.colnb[4 * c + f];
    fixed = m.bc_side == TN_BC_FIXED;
    if (nbc >= 0) {
      const int code = m.colnbf[4 * c + f], f2 = code & 3, end = (f2 & 1) ? N - 1 : 0, st = (f2 >> 1) == 0 ? N : 1;
      F.nbu = u + (size_t)(s * m.ncol + nbc) * 3 * n + end * ((f2 >> 1) == 0 ? 1 : N) + (code >> 2 ? (N - 1) * st : 0);
      F.ns1 = code >> 2 ? -st : st;
    }
  } else {
    const int s2 = f == 4 ? s + 1 : s - 1;  // the slab below / above
    const T *lay = Geo<T>::lay(m), *own = lay + 3 * m.slab_layer[s];
    T a11 = own[0], a44 = own[2];
    fixed = f == 4 && m.bc_bottom == TN_BC_FIXED;  // the top carries the beam (Neumann)
    if (s2 >= 0 && s2 < m.nslab) {
      const T *nb = lay + 3 * m.slab_layer[s2];
      a11 = T(0.5) * (a11 + nb[0]);
      a44 = T(0.5) * (a44 + nb[2]);
      F.nbu = u + (size_t)(s2 * m.ncol + c) * 3 * n + (f == 4 ? (N - 1) * N2 : 0);
    }
    E.p11[f - 4] = a11;
    E.p44[f - 4] = a44;
  }
  F.ju = F.nbu ? T(1) : (fixed ? T(2) : T(0));
  F.hf = F.nbu ? T(0.5) : (fixed ? T(1) : T(0));
}

// Many elements: N^2 threads per element (one per cross-section node), as
// many elements per CTA as fit 256 threads (N = 7: 245 busy lanes of 256).
// Smaller CTAs idle more lanes: 1 to 5 elements measured within 4 % of each
// other on the 2.0 M mirror, 5 to 20 % apart at p = 5, 8.  Few elements: 3
// N^2 threads per element (see apply_body_small), one element per CTA.
constexpr int kApplyThreads = 256;
enum { AM_PENCIL = 0, AM_SMALL = 1, AM_SMALL_BATCH = 2 };
constexpr int kSmallBatchThreads = 384;  // a batch's CTAs, whatever the degree
template <int N, int MODE>
__host__ __device__ constexpr int apply_eb() {
  return MODE == AM_PENCIL ? kApplyThreads / (N * N) : (MODE == AM_SMALL ? 1 : kSmallBatchThreads / (3 * N * N));
}
template <int N, int MODE>
__host__ __device__ constexpr int apply_threads() {
  return MODE == AM_PENCIL ? kApplyThreads : (MODE == AM_SMALL ? (3 * N * N + 31) / 32 * 32 : kSmallBatchThreads);
}
bool apply_small(int E, int sms) { return E <= 8 * sms; }
bool apply_small(int E) { return apply_small(E, tn_sm_count()); }
// shared memory of one element: the two lateral derivatives (the field is
// staged where the xi derivatives go), rows of i padded to an odd pitch, the
// zeta derivative at the lateral faces, and seven column tables
enum { SC_IXX = 0, SC_IXY, SC_IEX, SC_IEY, SC_DET, SC_RXI, SC_RETA, SC_NF };
template <int N>
__host__ __device__ constexpr int apply_elem_words() { return 6 * N * N * (N | 1) + (12 + SC_NF) * N * N; }
// (one thread per component: the three derivatives, the jumps and then
// surface terms of the six faces, and the column tables)
template <int N>
__host__ __device__ constexpr int apply_small_words() { return 9 * N * N * (N | 1) + (18 + SC_NF) * N * N; }
template <int N, typename T, int MODE>
__host__ __device__ constexpr size_t apply_smem() {
  return (size_t)apply_eb<N, MODE>() *
         (sizeof(ElemI<T>) + sizeof(T) * (MODE != AM_PENCIL ? apply_small_words<N>() : apply_elem_words<N>()));
}

// One thread per cross-section node (i, j) of an element, holding the zeta
// line through it in registers; the same thread works the xi line (k = j', j
// = i') and the eta line (k, i) of its pair (a, b) = (tid % N, tid / N), and
// face position (t1, t2) = (a, b) of all six faces -- the two ends of its
// own lines -- so that jumps and face terms stay in registers.
template <int N, typename T>
__device__ __forceinline__ T apply_body(const ElemI<T> &E, T *__restrict__ sm, int q, bool act, bool want_dot,
                                        T (&z)[3][N]) {
  constexpr int N2 = N * N, n = N * N2, NP = N | 1, PL = N * NP, CN = N * PL;
  T *const g0 = sm, *const g1 = sm + 3 * CN, *const sf = sm + 6 * CN, *const sc = sf + 12 * N2;
  const int a = q % N, b = q / N;
  const int row = b * NP + a;  // pencil (i, j) = (a, b), plus k PL
  const int lx = b * PL + a * NP, ly = b * PL + a;  // xi line (k, j) = (b, a); eta line (k, i) = (b, a), step NP
  // z: the zeta line of u, then its derivative, then the zeta flux
  T jump[6][3];   // neighbour values, then [[u]] at face position (a, b)
  if (act) {
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const T *p = E.f[f].nbu + (a * E.f[f].ns1 + b * (f < 4 ? N2 : N));
      const bool in = E.f[f].nbu != nullptr;
#pragma unroll
      for (int c = 0; c < 3; ++c) jump[f][c] = in ? p[c * n] : T(0);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < N; ++k) g0[c * CN + k * PL + row] = z[c][k];
    T tab[SC_NF];
#pragma unroll
    for (int t = 0; t < SC_NF; ++t) tab[t] = E.cg[(t < SC_RXI ? CG_IXX + t : CG_RXI + t - SC_RXI) * N2 + q];
#pragma unroll
    for (int t = 0; t < SC_NF; ++t) sc[t * N2 + q] = tab[t];
  }
  __syncthreads();
  // ---- derivative lines: zeta in registers, eta into g1
  if (act) {
    const T j4 = E.f[4].ju, j5 = E.f[5].ju, j2 = E.f[2].ju, j3 = E.f[3].ju;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      jump[4][c] = fm(j4, z[c][0], -jump[4][c]);
      jump[5][c] = fm(j5, z[c][N - 1], -jump[5][c]);
      T o[N];
      line_eo<N, 0, T>(z[c], o);
#pragma unroll
      for (int k = 0; k < N; ++k) z[c][k] = o[k];
    }
    // the zeta derivative at the lateral face nodes (position (j or i, k))
    if (a == 0 || a == N - 1) {
      T *const o = sf + (a == 0 ? 0 : 3 * N2) + b;
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < N; ++k) o[c * N2 + k * N] = z[c][k];
    }
    if (b == 0 || b == N - 1) {
      T *const o = sf + (b == 0 ? 6 * N2 : 9 * N2) + a;
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < N; ++k) o[c * N2 + k * N] = z[c][k];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T v[N], o[N];
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = g0[c * CN + ly + m * NP];
      jump[2][c] = fm(j2, v[0], -jump[2][c]);
      jump[3][c] = fm(j3, v[N - 1], -jump[3][c]);
      line_eo<N, 0, T>(v, o);
#pragma unroll
      for (int m = 0; m < N; ++m) g1[c * CN + ly + m * NP] = o[m];
    }
  }
  __syncthreads();
  // ---- xi lines, in place
  if (act) {
    const T j0 = E.f[0].ju, j1 = E.f[1].ju;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T v[N], o[N];
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = g0[c * CN + lx + m];
      jump[0][c] = fm(j0, v[0], -jump[0][c]);
      jump[1][c] = fm(j1, v[N - 1], -jump[1][c]);
      line_eo<N, 0, T>(v, o);
#pragma unroll
      for (int m = 0; m < N; ++m) g0[c * CN + lx + m] = o[m];
    }
  }
  __syncthreads();
  // ---- faces: traction and penalty at position (t1, t2) = (a, b)
  const ApplyTabs<T> &tb = tabs<T>(N);
  const T lf = tb.whalf;
  T surf[6][3], dot = T(0);
  const T *const dzs = E.sg + SG_DZ * N, *const idzs = E.sg + SG_IDZ * N;
  const Moduli<T> C = E.C;
  Map2<T> J = {T(0), T(0), T(0), T(0)};  // of the pencil's node
  T wdet = T(0);                         // w_i w_j det2 there
  if (act) {
    const T wab = tb.w[a] * tb.w[b], dzb = dzs[b], idzb = idzs[b];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const FaceI<T> &F = E.f[f];
      const int end = (f & 1) ? N - 1 : 0;
      const int qf = f < 2 ? a * N + end : end * N + a;
      const int at = b * PL + (f < 2 ? a * NP + end : end * NP + a);
      const Map2<T> K = {sc[SC_IXX * N2 + qf], sc[SC_IXY * N2 + qf], sc[SC_IEX * N2 + qf], sc[SC_IEY * N2 + qf]};
      const T wd = wab * sc[SC_DET * N2 + qf] * dzb;
      T d0[3], d1[3], d2[3], tw[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        d0[c] = g0[c * CN + at];
        d1[c] = g1[c * CN + at];
        d2[c] = idzb * sf[(f * 3 + c) * N2 + q];
      }
      const Stress<T> s = stress_of(K, d0, d1, d2, C);
      lateral_terms(f < 2 ? K.xx : K.ex, f < 2 ? K.xy : K.ey, s, C, F.hf * ((f & 1) ? wd : -wd),
                    wd * (E.sp * sc[(f < 2 ? SC_RXI : SC_RETA) * N2 + qf]), jump[f], tw, surf[f]);
      if (F.nbu) {
#pragma unroll
        for (int c = 0; c < 3; ++c) E.tr[(f * 3 + c) * N2 + q] = tw[c];
        if (want_dot) {
#pragma unroll
          for (int c = 0; c < 3; ++c) dot = fm(tw[c], E.u[c * n + b * N2 + qf] - jump[f][c], dot);
        }
      }
    }
    J = {sc[SC_IXX * N2 + q], sc[SC_IXY * N2 + q], sc[SC_IEX * N2 + q], sc[SC_IEY * N2 + q]};
    wdet = wab * sc[SC_DET * N2 + q];
#pragma unroll
    for (int f = 4; f < 6; ++f) {
      const FaceI<T> &F = E.f[f];
      const int k = f == 5 ? N - 1 : 0, at = k * PL + row;
      const T idz = idzs[k];
      T d0[3], d1[3], d2[3], tw[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        d0[c] = g0[c * CN + at];
        d1[c] = g1[c * CN + at];
        d2[c] = idz * z[c][k];
      }
      const Stress<T> s = stress_of(J, d0, d1, d2, C);
      zeta_terms(s, F.hf * (f == 5 ? wdet : -wdet), wdet * (E.sp * E.sg[SG_HINV * N + k]), E.p11[f - 4], E.p44[f - 4],
                 jump[f], tw, surf[f]);
      if (F.nbu) {
#pragma unroll
        for (int c = 0; c < 3; ++c) E.tr[(f * 3 + c) * N2 + q] = tw[c];
        if (want_dot) {
#pragma unroll
          for (int c = 0; c < 3; ++c) dot = fm(tw[c], E.u[c * n + k * N2 + q] - jump[f][c], dot);
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) z[c][k] = fm(f == 5 ? -lf : lf, jump[f][c], z[c][k]);
    }
  }
  __syncthreads();  // every traction has read the unlifted derivatives
  if (act) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T *const x = g0 + c * CN + lx, *const e = g1 + c * CN + ly;
      x[0] = fm(lf, jump[0][c], x[0]);
      x[N - 1] = fm(-lf, jump[1][c], x[N - 1]);
      e[0] = fm(lf, jump[2][c], e[0]);
      e[(N - 1) * NP] = fm(-lf, jump[3][c], e[(N - 1) * NP]);
    }
  }
  __syncthreads();
  // ---- per node: strain, stress, fluxes
  if (act) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int at = k * PL + row;
      const T idz = idzs[k], wz = wdet * tb.w[k];
      T d0[3], d1[3], d2[3], F2[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        d0[c] = g0[c * CN + at];
        d1[c] = g1[c * CN + at];
        d2[c] = idz * z[c][k];
      }
      node_flux(J, stress_of(J, d0, d1, d2, C), wz, wz * dzs[k], d0, d1, F2);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        g0[c * CN + at] = d0[c];
        g1[c * CN + at] = d1[c];
        z[c][k] = F2[c];
      }
    }
  }
  __syncthreads();
  // ---- weak-divergence lines, with the surface terms at their ends
  if (act) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T v[N], o[N];
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = g0[c * CN + lx + m];
      line_eo<N, 1, T>(v, o);
      o[0] += surf[0][c];
      o[N - 1] += surf[1][c];
#pragma unroll
      for (int m = 0; m < N; ++m) g0[c * CN + lx + m] = o[m];
#pragma unroll
      for (int m = 0; m < N; ++m) v[m] = g1[c * CN + ly + m * NP];
      line_eo<N, 1, T>(v, o);
      o[0] += surf[2][c];
      o[N - 1] += surf[3][c];
#pragma unroll
      for (int m = 0; m < N; ++m) g1[c * CN + ly + m * NP] = o[m];
      line_eo<N, 1, T>(z[c], o);
      o[0] += surf[4][c];
      o[N - 1] += surf[5][c];
#pragma unroll
      for (int k = 0; k < N; ++k) z[c][k] = o[k];
    }
  }
  __syncthreads();
  if (act) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int at = c * CN + k * PL + row;
        const T yv = z[c][k] + (g0[at] + g1[at]);
        E.y[c * n + k * N2 + q] = yv;
        if (want_dot) dot = fm(yv, E.u[c * n + k * N2 + q], dot);
      }
  }
  return dot;
}

// ---- few elements: three threads per pencil, one per component
// A mesh of up to some eight elements per SM runs as one wave whose time is
// one element's chain of phases; a third of the line work per thread shortens
// it (FP32 / FP64, us, against the pencil form: 128 elements p = 8 11.5 / 59
// against 16.1 / 76; 1024 elements p = 6 18.4 / 169 against 23.5 / 211),
// while its extra passes through shared memory (the zeta derivatives, the
// jumps) cost the larger meshes (1944 elements p = 6: 27 against 24 us).
// One thread per component c and cross-section node (a, b) of an element.
// In turn it is: the zeta line (i, j) = (a, b), the eta line (k, i) = (b, a)
// and the xi line (k, j) = (b, a) of component c; position (t1, t2) = (a, b)
// of the two faces across direction c (all components); and the nodes
// (a, b, k = c, c + 3, ..).  z: the zeta line of u.  Returns this thread's
// part of u . A u.
template <int N, typename T>
__device__ __forceinline__ T apply_body_small(const ElemI<T> &E, T *__restrict__ sm, int c, int q, bool act, bool want_dot,
                                        T (&z)[N]) {
  constexpr int N2 = N * N, n = N * N2, NP = N | 1, PL = N * NP, CN = N * PL;
  T *const g0 = sm, *const g1 = sm + 3 * CN, *const g2 = sm + 6 * CN, *const js = sm + 9 * CN, *const sc = js + 18 * N2;
  const int a = q % N, b = q / N;
  const int row = c * CN + b * NP + a;  // pencil (i, j) = (a, b) of component c, plus k PL
  const int lx = c * CN + b * PL + a * NP, ly = c * CN + b * PL + a;  // the xi line; the eta line, step NP
  T jump[6];  // neighbour values, then [[u]] of component c at face position (a, b)
  if (act) {
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const T *p = E.f[f].nbu + (c * n + a * E.f[f].ns1 + b * (f < 4 ? N2 : N));
      jump[f] = E.f[f].nbu ? *p : T(0);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) g0[row + k * PL] = z[k];
#pragma unroll
    for (int t = c; t < SC_NF; t += 3)
      sc[t * N2 + q] = E.cg[(t < SC_RXI ? CG_IXX + t : CG_RXI + t - SC_RXI) * N2 + q];
  }
  __syncthreads();
  // ---- derivative lines: zeta into g2, eta into g1
  if (act) {
    jump[4] = fm(E.f[4].ju, z[0], -jump[4]);
    jump[5] = fm(E.f[5].ju, z[N - 1], -jump[5]);
    T v[N], o[N];
    line_eo<N, 0, T>(z, o);
#pragma unroll
    for (int k = 0; k < N; ++k) g2[row + k * PL] = o[k];
#pragma unroll
    for (int m = 0; m < N; ++m) v[m] = g0[ly + m * NP];
    jump[2] = fm(E.f[2].ju, v[0], -jump[2]);
    jump[3] = fm(E.f[3].ju, v[N - 1], -jump[3]);
    line_eo<N, 0, T>(v, o);
#pragma unroll
    for (int m = 0; m < N; ++m) g1[ly + m * NP] = o[m];
  }
  __syncthreads();
  // ---- xi lines, in place
  if (act) {
    T v[N], o[N];
#pragma unroll
    for (int m = 0; m < N; ++m) v[m] = g0[lx + m];
    jump[0] = fm(E.f[0].ju, v[0], -jump[0]);
    jump[1] = fm(E.f[1].ju, v[N - 1], -jump[1]);
    line_eo<N, 0, T>(v, o);
#pragma unroll
    for (int m = 0; m < N; ++m) g0[lx + m] = o[m];
#pragma unroll
    for (int f = 0; f < 6; ++f) js[(f * 3 + c) * N2 + q] = jump[f];
  }
  __syncthreads();
  // ---- the two faces across direction c: traction and penalty at (a, b)
  const ApplyTabs<T> &tb = tabs<T>(N);
  const T lf = tb.whalf;
  T dot = T(0), jf[2][3], wab = T(0);
  const T *const dzs = E.sg + SG_DZ * N, *const idzs = E.sg + SG_IDZ * N;
  const Moduli<T> C = E.C;
  if (act) {
    wab = tb.w[a] * tb.w[b];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int f = 2 * c + e, end = e ? N - 1 : 0;
      const FaceI<T> &F = E.f[f];
      const int qf = c == 0 ? a * N + end : (c == 1 ? end * N + a : q), kf = c == 2 ? end : b;
      const int at = kf * PL + (c == 0 ? a * NP + end : (c == 1 ? end * NP + a : b * NP + a));
      const Map2<T> K = {sc[SC_IXX * N2 + qf], sc[SC_IXY * N2 + qf], sc[SC_IEX * N2 + qf], sc[SC_IEY * N2 + qf]};
      const T idz = idzs[kf], wdet = wab * sc[SC_DET * N2 + qf];
      T *const jp = js + f * 3 * N2 + q;
      T d0[3], d1[3], d2[3], tw[3], sf[3];
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        d0[l] = g0[l * CN + at];
        d1[l] = g1[l * CN + at];
        d2[l] = idz * g2[l * CN + at];
        jf[e][l] = jp[l * N2];
      }
      const Stress<T> s = stress_of(K, d0, d1, d2, C);
      if (c < 2) {
        const T wd = wdet * dzs[b];
        lateral_terms(c == 0 ? K.xx : K.ex, c == 0 ? K.xy : K.ey, s, C, F.hf * (e ? wd : -wd),
                      wd * (E.sp * sc[(c == 0 ? SC_RXI : SC_RETA) * N2 + qf]), jf[e], tw, sf);
      } else {
        zeta_terms(s, F.hf * (e ? wdet : -wdet), wdet * (E.sp * E.sg[SG_HINV * N + end]), E.p11[e], E.p44[e], jf[e], tw,
                   sf);
      }
#pragma unroll
      for (int l = 0; l < 3; ++l) jp[l * N2] = sf[l];
      if (F.nbu) {
#pragma unroll
        for (int l = 0; l < 3; ++l) E.tr[(f * 3 + l) * N2 + q] = tw[l];
        if (want_dot) {
#pragma unroll
          for (int l = 0; l < 3; ++l) dot = fm(tw[l], E.u[l * n + kf * N2 + qf] - jf[e][l], dot);
        }
      }
    }
  }
  __syncthreads();  // every traction has read the unlifted derivatives
  if (act) {
    T *const gd = c == 0 ? g0 + b * PL + a * NP : (c == 1 ? g1 + b * PL + a : g2 + b * NP + a);
    const int last = (N - 1) * (c == 0 ? 1 : (c == 1 ? NP : PL));
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      gd[l * CN] = fm(lf, jf[0][l], gd[l * CN]);
      gd[l * CN + last] = fm(-lf, jf[1][l], gd[l * CN + last]);
    }
  }
  __syncthreads();
  // ---- per node: strain, stress, fluxes
  if (act) {
    const Map2<T> J = {sc[SC_IXX * N2 + q], sc[SC_IXY * N2 + q], sc[SC_IEX * N2 + q], sc[SC_IEY * N2 + q]};
    const T wdet = wab * sc[SC_DET * N2 + q];
#pragma unroll
    for (int m = 0; m < (N + 2) / 3; ++m) {
      const int k = c + 3 * m, at = k * PL + b * NP + a;
      if (k >= N) break;
      const T idz = idzs[k], wz = wdet * tb.w[k];
      T d0[3], d1[3], d2[3], F2[3];
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        d0[l] = g0[l * CN + at];
        d1[l] = g1[l * CN + at];
        d2[l] = idz * g2[l * CN + at];
      }
      node_flux(J, stress_of(J, d0, d1, d2, C), wz, wz * dzs[k], d0, d1, F2);
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        g0[l * CN + at] = d0[l];
        g1[l * CN + at] = d1[l];
        g2[l * CN + at] = F2[l];
      }
    }
  }
  __syncthreads();
  // ---- weak-divergence lines, with the surface terms at their ends
  if (act) {
    T v[N], o[N];
    const T *const jp = js + c * N2 + q;
#pragma unroll
    for (int m = 0; m < N; ++m) v[m] = g0[lx + m];
    line_eo<N, 1, T>(v, o);
    o[0] += jp[0];
    o[N - 1] += jp[3 * N2];
#pragma unroll
    for (int m = 0; m < N; ++m) g0[lx + m] = o[m];
#pragma unroll
    for (int m = 0; m < N; ++m) v[m] = g1[ly + m * NP];
    line_eo<N, 1, T>(v, o);
    o[0] += jp[6 * N2];
    o[N - 1] += jp[9 * N2];
#pragma unroll
    for (int m = 0; m < N; ++m) g1[ly + m * NP] = o[m];
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = g2[row + k * PL];
    line_eo<N, 1, T>(v, z);
    z[0] += jp[12 * N2];
    z[N - 1] += jp[15 * N2];
  }
  __syncthreads();
  if (act) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int at = row + k * PL;
      const T yv = z[k] + (g0[at] + g1[at]);
      E.y[c * n + k * N2 + q] = yv;
      if (want_dot) dot = fm(yv, E.u[c * n + k * N2 + q], dot);
    }
  }
  return dot;
}

// The alpha step of a PCG iteration folded into the operator apply: once
// every CTA of the step has written its p . Ap partial, the last reduces
// all partials in a fixed order (0 .. nparts - 1) and sets alpha = rz / pAp
// (breakdown if pAp <= 0 or not finite).  A run that has finished skips the
// apply and marks the iteration inactive.
__device__ __forceinline__ bool fold_skip(const PcgFold &f) {
  if (!f.s || !f.s->done) return false;
  if (blockIdx.x == 0 && threadIdx.x == 0) f.s->active = 0;
  return true;
}
__device__ void fold_alpha(const PcgFold &f) {
  const double *__restrict__ part = f.part;
  __shared__ int last;
  __shared__ double red[32];
  __syncthreads();  // this CTA's partial is written
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(f.cnt, 1u) == (unsigned)(f.total - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double acc = 0.0;
  for (int t = threadIdx.x; t < f.nparts; t += blockDim.x) acc += __ldcg(part + t);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double pq = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) pq += red[w];
    tn_pcg_scalars *s = f.s;
    s->active = 1;
    s->pq = pq;
    if (!(pq > 0.0) || !isfinite(pq)) {
      s->breakdown = 1;
      s->done = 1;
      s->alpha = 0.0;
    } else {
      s->alpha = s->rz / pq;
    }
    *f.cnt = 0u;
    __threadfence();
  }
}

// FP32: variant 0 asks for three CTAs per SM (80 registers, some spilled at N
// = 9), variant 1 for two (up to 128).  Both round alike (bit-identical
// results); the autotuner times them on the mesh at hand (p = 6, 2.0 M
// unknowns: 25.3 / 26.4 us; p = 8, 59 M: 578 / 454 us).
template <typename T, int V>
__host__ __device__ constexpr int apply_min_blocks() { return sizeof(T) == 8 ? 1 : (V == 0 ? 3 : 2); }

// elements w0 .. w0 + nw - 1 of one mesh (meshes == nullptr: m1, element w)
// or of a batch (element work[w].y of mirror work[w].x)
template <int N, typename T, int MODE>
__device__ __forceinline__ void apply_cta(const DevMesh &m1, const DevMesh *__restrict__ meshes,
                                          const int2 *__restrict__ work, const long long *__restrict__ dof_off,
                                          const long long *__restrict__ tr_off, int w0, int nw,
                                          const T *__restrict__ u, T *__restrict__ y, T *__restrict__ trace,
                                          double *__restrict__ partial, const PcgFold &fold) {
  constexpr int N2 = N * N, n = N * N2, EB = apply_eb<N, MODE>(), NT = apply_threads<N, MODE>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ElemI<T> *const info = reinterpret_cast<ElemI<T> *>(smem_raw);
  const int tid = threadIdx.x;
  constexpr int PT = MODE == AM_PENCIL ? N2 : 3 * N2;  // threads per element
  const int el = tid / PT, r = tid - el * PT, cc = r / N2, q = r - cc * N2;
  const bool act = el < nw;
  const T *ue = u;
  if (act) {
    const int2 w = meshes ? work[w0 + el] : make_int2(0, w0 + el);
    ue += (meshes ? dof_off[w.x] : 0) + (size_t)(w.y * 3 + cc) * n + q;
  }
  for (int t = tid; t < nw * 6; t += NT) {
    const int e1 = t / 6, f = t - e1 * 6;
    ElemI<T> &E = info[e1];
    const int2 w = meshes ? work[w0 + e1] : make_int2(0, w0 + e1);
    const DevMesh &m = meshes ? meshes[w.x] : m1;
    const int e = w.y, s = e / m.ncol, col = e - s * m.ncol;
    const T *ui = meshes ? u + dof_off[w.x] : u;
    face_setup<N, T>(m, ui, s, col, f, E);
    if (f == 0) {
      const T *lay = Geo<T>::lay(m) + 3 * m.slab_layer[s];
      E.u = ui + (size_t)e * 3 * n;
      E.y = (meshes ? y + dof_off[w.x] : y) + (size_t)e * 3 * n;
      E.tr = (meshes ? trace + tr_off[w.x] : trace) + (size_t)e * 18 * N2;
      E.cg = Geo<T>::col(m) + (size_t)col * CG_NF * N2;
      E.sg = Geo<T>::slab(m) + (size_t)s * SG_NF * N;
      E.C = {lay[0], lay[1], lay[2]};
      E.sp = (T)(m.penC * (double)((m.p + 1) * (m.p + 1)));
    }
  }
  grid_wait();
  ue = after_wait(ue);
  if (fold_skip(fold)) return;
  const ElemI<T> &E = info[act ? el : 0];
  T dott;
  if constexpr (MODE != AM_PENCIL) {
    T z[N];
    if (act) {
#pragma unroll
      for (int k = 0; k < N; ++k) z[k] = ue[k * N2];
    }
    __syncthreads();
    dott = apply_body_small<N, T>(E, reinterpret_cast<T *>(info + EB) + (size_t)(act ? el : 0) * apply_small_words<N>(),
                                  cc, q, act, partial != nullptr, z);
  } else {
    T z[3][N];
    if (act) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < N; ++k) z[c][k] = ue[c * n + k * N2];
    }
    __syncthreads();
    T *sm = reinterpret_cast<T *>(info + EB) + (size_t)(act ? el : 0) * apply_elem_words<N>();
    dott = apply_body<N, T>(E, sm, q, act, partial != nullptr, z);
  }
  if (partial) {
    __shared__ double red[NT / 32];
    double dot = (double)dott;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if ((tid & 31) == 0) red[tid >> 5] = dot;
    __syncthreads();
    if (tid == 0) {
      double sum = 0.0;
      for (int w = 0; w < NT / 32; ++w) sum += red[w];
      partial[blockIdx.x] = sum;
    }
    if (fold.s) fold_alpha(fold);
  }
}

template <int N, typename T, int V, int MODE>
__global__ void __launch_bounds__((apply_threads<N, MODE>()), (MODE == AM_PENCIL ? apply_min_blocks<T, V>() : 1))
apply_elem_kernel(const DevMesh m1, int nwork, const T *__restrict__ u, T *__restrict__ y, T *__restrict__ trace,
                  double *__restrict__ partial, const PcgFold fold) {
  grid_trigger();
  constexpr int EB = apply_eb<N, MODE>();
  const int w0 = blockIdx.x * EB, nw = nwork - w0 < EB ? nwork - w0 : EB;
  apply_cta<N, T, MODE>(m1, nullptr, nullptr, nullptr, nullptr, w0, nw, u, y, trace, partial, fold);
}

// a batch in one launch: CTA b works on the elements ctas[b] = (N, first work
// item, count).  One launch per degree left most of the GPU idle: 24 mirrors
// of degrees 4 to 8 took five launches of 18 to 30 us each.
template <typename T, int V, int MODE>
__global__ void __launch_bounds__((apply_threads<9, MODE>()), (MODE == AM_PENCIL ? apply_min_blocks<T, V>() : 1))
apply_batch_kernel(const DevMesh *__restrict__ meshes, const int2 *__restrict__ work,
                   const long long *__restrict__ dof_off, const long long *__restrict__ tr_off,
                   const int4 *__restrict__ ctas, const T *__restrict__ u, T *__restrict__ y,
                   T *__restrict__ trace, double *__restrict__ partial, const PcgFold fold) {
  grid_trigger();
  const int4 C = ctas[blockIdx.x];
  const DevMesh none{};
  switch (C.x) {
#define TN_CASE(NN)                                                                                             case NN:                                                                                                        apply_cta<NN, T, MODE>(none, meshes, work, dof_off, tr_off, C.y, C.z, u, y, trace, partial, fold);                 break;
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
  }
}

// The second launch.  UPD = 0: y += the traction terms the neighbours wrote
// for this element's face nodes, one thread per surface node (N^3 - (N - 2)^3
// of N^3).  UPD = 1, inside a PCG iteration: r -= alpha (y + those terms) over
// all nodes, the residual update taking the incomplete product as it is
// (2.0 M unknowns, FP32: the two passes it replaces took 7.8 + 5 us).  Up to
// three faces meet at a node; their terms are added in the order xi, eta,
// zeta.  Bound by the bytes of the vectors and traces, with few elements by
// latency: they are spread over two CTAs per SM then (FP32 applies one after
// another, p = 2: 64 elements 12.4 -> 7.1 us, 512 12.5 -> 7.0, against as many
// elements per CTA as add_eb, 39).
template <int N>
__host__ __device__ constexpr int surf_nodes() { return N * N * N - (N - 2) * (N - 2) * (N - 2); }
constexpr int kAddThreads = 256;
template <int N>
__host__ __device__ constexpr int add_eb() { return kAddThreads * 4 / surf_nodes<N>(); }
int add_elems(int most, int E, int sms) { return std::min(most, std::max(1, E / (2 * sms))); }
// Whether the second launch lets the one after it start at once.  A launch that
// starts while the operator still runs takes whatever slots are left: a grid that
// would spread over the GPU piles up on a few SMs, one that fills it, or leaves
// most of it empty, gains the start.  In a PCG iteration it is the
// preconditioner's (mixed solves, early against late: 153 elements, p = 7, 58.6
// against 45.3 ms; 396, p = 5, 49.4 against 47.6; 1944, p = 6, 200 against 207;
// FP64, 8 elements, p = 3, 1.87 against 1.92), else the next apply (us an apply,
// FP64 / FP32):
//   one element per CTA: 216 elements, p = 4: 56 / 7.0 against 25 / 7.2; 343 to
//   512, p = 2, 3: 42 to 59 against 16 to 27; 8, p = 2: 14.6 against 15.6; 729,
//   p = 8 (1165 threads per SM): 252.5 / 21.2 against 253.3 / 22.1
//   pencils, FP32: 83 CTAs (p = 2, 2304 elements) 10.3 against 8.9; 140, p = 4,
//   14.2 against 11.5; 180, p = 3, 11.5 against 12.3; 280, p = 6, 19.3 against 20.2;
//   389, p = 6, 24.9 against 26.2 (not 288, p = 4: 20.7 against 19.3)
//   batches, whose CTAs work on several elements each: FP32, 2 mirrors 10.1
//   against 10.4, 6 22.7 against 24.5, 10 32.7 against 34.3, 24 52.7 against 55.3;
//   FP64, 2 52.1 against 53.6, 24 726.9 against 730.5
bool add_early(const ApplyArgs &a) {
  const int E = a.m ? a.m->E : a.elems, sms = a.sms;
  if (a.r) return !apply_small(E, sms) || E <= sms / 8;
  if (!a.m) return true;
  const int N = a.m->N;
  if (apply_small(E, sms)) return E <= sms / 8 || 3 * N * N * E > 600 * sms;
  return E / tn_apply_eb(N, false) > sms;
}

template <int N, typename T, int UPD>
__device__ __forceinline__ void trace_add_cta(const DevMesh &m1, const DevMesh *__restrict__ meshes,
                                              const int2 *__restrict__ work, const long long *__restrict__ dof_off,
                                              const long long *__restrict__ tr_off, int w0, int nw,
                                              T *__restrict__ y, const T *__restrict__ trace, T *__restrict__ r,
                                              const double *__restrict__ alpha, const int *__restrict__ done) {
  constexpr int N2 = N * N, n = N * N2, SN = UPD ? n : surf_nodes<N>(), EB = add_eb<N>(), RING = 4 * N - 4;
  __shared__ const T *tr[EB][6];  // the neighbour's trace of the matching face (nullptr: none)
  __shared__ int flip[EB][6];
  __shared__ long long eo[EB];    // first unknown of the element
  const int tid = threadIdx.x;
  for (int t = tid; t < nw * 6; t += kAddThreads) {
    const int el = t / 6, f = t - el * 6, w = w0 + el;
    const int2 wk = meshes ? work[w] : make_int2(0, w);
    const DevMesh &m = meshes ? meshes[wk.x] : m1;
    const int ncol = m.ncol, s = wk.y / ncol, c = wk.y - s * ncol;
    const T *t0 = meshes ? trace + tr_off[wk.x] : trace;
    if (f == 0) eo[el] = (meshes ? dof_off[wk.x] : 0) + (long long)wk.y * 3 * n;
    int e2 = -1, f2 = 0, fl = 0;
    if (f < 4) {
      const int nbc = m.colnb[4 * c + f], code = m.colnbf[4 * c + f];
      if (nbc >= 0) e2 = s * ncol + nbc;
      f2 = code & 3;
      fl = code >> 2;
    } else {
      const int s2 = f == 4 ? s + 1 : s - 1;
      if (s2 >= 0 && s2 < m.nslab) e2 = s2 * ncol + c;
      f2 = f == 4 ? 5 : 4;
    }
    tr[el][f] = e2 >= 0 ? t0 + ((size_t)e2 * 6 + f2) * 3 * N2 : nullptr;
    flip[el][f] = fl;
  }
  __syncthreads();
  grid_wait();
  done = after_wait(done);
  y = after_wait(y);
  r = after_wait(r);
  if (done && *done) return;
  const T al = UPD ? (T)*after_wait(alpha) : T(0);
#pragma unroll 4
  for (int id = tid; id < nw * SN; id += kAddThreads) {
    const int el = id / SN, rr0 = id - el * SN;
    int i, j, k;
    if (UPD) {
      k = rr0 / N2;
      const int q = rr0 - k * N2;
      j = q / N;
      i = q - j * N;
    } else if (rr0 < 2 * N2) {  // the two zeta faces, then the lateral ring of every k between them
      k = rr0 < N2 ? 0 : N - 1;
      const int q = rr0 < N2 ? rr0 : rr0 - N2;
      j = q / N;
      i = q - j * N;
    } else {
      const int rr = rr0 - 2 * N2, kk = rr / RING, g = rr - kk * RING;
      k = kk + 1;
      if (g < 2 * N) {
        j = g < N ? 0 : N - 1;
        i = g < N ? g : g - N;
      } else {
        j = ((g - 2 * N) >> 1) + 1;
        i = (g & 1) ? N - 1 : 0;
      }
    }
    T add[3] = {T(0), T(0), T(0)};
    auto take = [&](int f, int t1, int t2) {
      const T *t = tr[el][f];
      if (!t) return;
      t += t2 * N + (flip[el][f] ? N - 1 - t1 : t1);
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) add[cc] += t[cc * N2];
    };
    const long long at = eo[el] + (k * N + j) * N + i;
    T yv[3], rv[3];
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) yv[cc] = y[at + cc * n];
    if (UPD) {
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) rv[cc] = r[at + cc * n];
    }
    if (i == 0 || i == N - 1) take(i == 0 ? 0 : 1, j, k);
    if (j == 0 || j == N - 1) take(j == 0 ? 2 : 3, i, k);
    if (k == 0 || k == N - 1) take(k == 0 ? 4 : 5, i, j);
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
      const T full = yv[cc] + add[cc];
      if (UPD) r[at + cc * n] = fm(-al, full, rv[cc]);
      else y[at + cc * n] = full;
    }
  }
}

template <int N, typename T, int UPD>
__global__ void __launch_bounds__(kAddThreads)
trace_add_kernel(const DevMesh m1, int nwork, int eb, bool early, T *__restrict__ y, const T *__restrict__ trace,
                 T *__restrict__ r, const double *__restrict__ alpha, const int *__restrict__ done) {
  if (early) grid_trigger();
  const int w0 = blockIdx.x * eb, nw = nwork - w0 < eb ? nwork - w0 : eb;
  trace_add_cta<N, T, UPD>(m1, nullptr, nullptr, nullptr, nullptr, w0, nw, y, trace, r, alpha, done);
}

template <typename T, int UPD>
__global__ void __launch_bounds__(kAddThreads)
trace_add_batch_kernel(const DevMesh *__restrict__ meshes, const int2 *__restrict__ work,
                       const long long *__restrict__ dof_off, const long long *__restrict__ tr_off,
                       const int4 *__restrict__ ctas, bool early, T *__restrict__ y, const T *__restrict__ trace,
                       T *__restrict__ r, const double *__restrict__ alpha, const int *__restrict__ done) {
  if (early) grid_trigger();
  const int4 C = ctas[blockIdx.x];
  const DevMesh none{};
  switch (C.x) {
#define TN_CASE(NN)                                                                                               \
  case NN:                                                                                                        \
    trace_add_cta<NN, T, UPD>(none, meshes, work, dof_off, tr_off, C.y, C.z, y, trace, r, alpha, done);          \
    break;
    TN_CASE(3) TN_CASE(4) TN_CASE(5) TN_CASE(6) TN_CASE(7) TN_CASE(8) TN_CASE(9)
#undef TN_CASE
  }
}

// a batch's CTAs get the shared memory of the largest degree
template <typename T, int MODE>
constexpr size_t max_smem() {
  size_t m = 0;
  for (size_t v : {apply_smem<3, T, MODE>(), apply_smem<4, T, MODE>(), apply_smem<5, T, MODE>(), apply_smem<6, T, MODE>(),
                   apply_smem<7, T, MODE>(), apply_smem<8, T, MODE>(), apply_smem<9, T, MODE>()})
    m = v > m ? v : m;
  return m;
}

template <int N, typename T, int V, int MODE>
cudaError_t launch_elem(const ApplyArgs &a, cudaStream_t st) {
  constexpr size_t sm = apply_smem<N, T, MODE>();
  constexpr int EB = apply_eb<N, MODE>();
  static int configured_device = -1;
  cudaError_t err = allow_smem(apply_elem_kernel<N, T, V, MODE>, sm, configured_device);
  if (err != cudaSuccess) return err;
  return launch_pdl(apply_elem_kernel<N, T, V, MODE>, (a.m->E + EB - 1) / EB, apply_threads<N, MODE>(), sm, st, *a.m,
                    a.m->E, (const T *)a.u, (T *)a.y, (T *)a.trace, a.partial, a.fold ? *a.fold : PcgFold());
}

template <int N, typename T, int V>
cudaError_t launch_mesh(const ApplyArgs &a, cudaStream_t st) {
  return apply_small(a.m->E, a.sms) ? launch_elem<N, T, 0, AM_SMALL>(a, st) : launch_elem<N, T, V, AM_PENCIL>(a, st);
}

template <int N, typename T>
cudaError_t launch_second(const ApplyArgs &a, cudaStream_t st) {
  const int E = a.m->E, eb = add_elems(add_eb<N>(), E, a.sms), grid = (E + eb - 1) / eb;
  const bool early = add_early(a);
  return a.r ? launch_pdl(trace_add_kernel<N, T, 1>, grid, kAddThreads, 0, st, *a.m, E, eb, early, (T *)a.y,
                          (const T *)a.trace, (T *)a.r, a.alpha, a.done)
             : launch_pdl(trace_add_kernel<N, T, 0>, grid, kAddThreads, 0, st, *a.m, E, eb, early, (T *)a.y,
                          (const T *)a.trace, (T *)nullptr, (const double *)nullptr, a.done);
}

template <typename T>
cudaError_t launch_second_batch(const ApplyArgs &a, cudaStream_t st) {
  if (a.nadd <= 0) return cudaSuccess;
  const bool early = add_early(a);
  return a.r ? launch_pdl(trace_add_batch_kernel<T, 1>, a.nadd, kAddThreads, 0, st, a.meshes, a.work, a.dof_off,
                          a.tr_off, a.adds, early, (T *)a.y, (const T *)a.trace, (T *)a.r, a.alpha, a.done)
             : launch_pdl(trace_add_batch_kernel<T, 0>, a.nadd, kAddThreads, 0, st, a.meshes, a.work, a.dof_off,
                          a.tr_off, a.adds, early, (T *)a.y, (const T *)a.trace, (T *)nullptr, (const double *)nullptr, a.done);
}

template <typename T, int V, int MODE>
cudaError_t launch_batch(const ApplyArgs &a, cudaStream_t st) {
  constexpr size_t sm = max_smem<T, MODE>();
  static int configured_device = -1;
  cudaError_t err = allow_smem(apply_batch_kernel<T, V, MODE>, sm, configured_device);
  if (err != cudaSuccess) return err;
  if (a.ncta <= 0) return cudaSuccess;
  return launch_pdl(apply_batch_kernel<T, V, MODE>, a.ncta, apply_threads<9, MODE>(), sm, st, a.meshes, a.work, a.dof_off,
                    a.tr_off, a.ctas, (const T *)a.u, (T *)a.y, (T *)a.trace, a.partial, a.fold ? *a.fold : PcgFold());
}

#define TN_FOR_N(CASE) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9)

// ------------------------------------------------------------- energies
// Energy of an element, 1/2 sum_p w_p detJ_p S_p : Y : S_p with S = sym grad u
// (unlifted), by pencils as the operator: thread q keeps the zeta line of its
// node (i, j) in registers, lines along xi and eta go through shared memory.
// With G_ij = 2 S_ij (i != j), T = tr S, D = sum S_ii^2, O = sum G_ij^2 the
// density is c12 T^2 + (c11 - c12) D + c44 O, so three sums per element do
// (parts != 0: their split along the stiffness's eigen-modes, dilatational
// (c11 + 2 c12) / 3 T^2, tetragonal (c11 - c12) (D - T^2 / 3) and shear
// c44 O).  Bound by the FP64 pipe (84 % busy; 77 operations per node).  One
// thread per node with whole rows of D, the stress and a division by dz at
// every node kept the pipe as busy with more: 549 -> 419 us at 8.0 M unknowns,
// p = 5.
// SPLIT (few elements, one per CTA): three threads per pencil, one per
// component, and every third node of the pencil, for latency.
constexpr int kEnergyThreads = 256;
template <int N>
constexpr int energy_eb() { return kEnergyThreads / (N * N); }
template <int N, bool SPLIT>
constexpr size_t energy_smem(int eb) { return sizeof(double) * (size_t)eb * (SPLIT ? 9 : 6) * N * N * N; }

// elements w0 .. of one mesh (meshes == nullptr: m1, element w) or of a batch
// (element work[w].y of mirror work[w].x); out: 1 or 3 numbers per element
template <int N, bool SPLIT>
__global__ void __launch_bounds__(kEnergyThreads)
energy_pencil_kernel(const DevMesh m1, const DevMesh *__restrict__ meshes, const int2 *__restrict__ work,
                     const long long *__restrict__ dof_off, int nwork, int eb, const double *__restrict__ u,
                     double *__restrict__ out, int parts) {
  constexpr int N2 = N * N, n = N * N2, PT = SPLIT ? 3 * N2 : N2;  // threads per element
  constexpr int NC = SPLIT ? 1 : 3, NK = SPLIT ? (N + 2) / 3 : N;     // components and nodes per thread
  extern __shared__ __align__(16) double esm[];
  grid_trigger();
  const int tid = threadIdx.x, el = tid / PT, r = tid - el * PT, c0 = r / N2, q = r - c0 * N2, wi = blockIdx.x * eb + el;
  const bool act = el < eb && wi < nwork;
  double *const A = esm + (size_t)(act ? el : 0) * (SPLIT ? 9 : 6) * n, *const B = A + 3 * n;
  const int2 wk = act && meshes ? work[wi] : make_int2(0, act ? wi : 0);
  const DevMesh &m = meshes ? meshes[wk.x] : m1;
  const int e = wk.y, s = e / m.ncol, col = e - s * m.ncol;
  grid_wait();
  const double *const ue = after_wait(u) + (meshes ? dof_off[wk.x] : 0) + (size_t)e * 3 * n + q;
  double z[NC][N];
  if (act) {
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int k = 0; k < N; ++k) B[(c0 + c) * n + k * N2 + q] = z[c][k] = ue[(c0 + c) * n + k * N2];
  }
  __syncthreads();
  if (act) {  // xi lines: thread q has (j, k) = (q % N, q / N)
#pragma unroll
    for (int c = c0; c < c0 + NC; ++c) {
      double v[N], o[N];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = B[c * n + q * N + i];
      line_eo<N, 0>(v, o);
#pragma unroll
      for (int i = 0; i < N; ++i) A[c * n + q * N + i] = o[i];
    }
  }
  __syncthreads();
  if (act) {  // eta lines, in place: (i, k) = (q % N, q / N)
    const int at = (q / N) * N2 + q % N;
#pragma unroll
    for (int c = c0; c < c0 + NC; ++c) {
      double v[N], o[N];
#pragma unroll
      for (int j = 0; j < N; ++j) v[j] = B[c * n + at + j * N];
      line_eo<N, 0>(v, o);
#pragma unroll
      for (int j = 0; j < N; ++j) B[c * n + at + j * N] = o[j];
    }
  }
  __syncthreads();
  double sT = 0.0, sD = 0.0, sO = 0.0;
  if (act) {
#pragma unroll
    for (int c = 0; c < NC; ++c) line_eo<N, 0>(z[c], z[c]);
    if constexpr (SPLIT) {
#pragma unroll
      for (int k = 0; k < N; ++k) A[(6 + c0) * n + k * N2 + q] = z[0][k];
    }
  }
  if constexpr (SPLIT) __syncthreads();
  if (act) {
    const double *cg = m.colgeo + (size_t)col * CG_NF * N2 + q, *sg = m.slabgeo + (size_t)s * SG_NF * N;
    const double ixx = cg[CG_IXX * N2], ixy = cg[CG_IXY * N2], iex = cg[CG_IEX * N2], iey = cg[CG_IEY * N2];
#pragma unroll
    for (int kk = 0; kk < NK; ++kk) {
      const int k = SPLIT ? 3 * kk + c0 : kk;
      if (SPLIT && k >= N) break;
      const double id = sg[SG_IDZ * N + k], wz = tabs<double>(N).w[k] * sg[SG_DZ * N + k];
      const double *a = A + k * N2 + q, *b = B + k * N2 + q;
      const double a0 = a[0], a1 = a[n], a2 = a[2 * n], b0 = b[0], b1 = b[n], b2 = b[2 * n];
      const double z0 = SPLIT ? a[6 * n] : z[0][kk], z1 = SPLIT ? a[7 * n] : z[NC / 2][kk], z2 = SPLIT ? a[8 * n] : z[NC - 1][kk];
      const double gxx = fm(ixx, a0, iex * b0), gyy = fm(ixy, a1, iey * b1), gzz = id * z2;
      const double gxy = fm(ixx, a1, fm(iex, b1, fm(ixy, a0, iey * b0)));
      const double gxz = fm(id, z0, fm(ixx, a2, iex * b2)), gyz = fm(id, z1, fm(ixy, a2, iey * b2));
      const double t = (gxx + gyy) + gzz;
      sT = fm(wz, t * t, sT);
      sD = fm(wz, fm(gxx, gxx, fm(gyy, gyy, gzz * gzz)), sD);
      sO = fm(wz, fm(gxy, gxy, fm(gxz, gxz, gyz * gyz)), sO);
    }
    const double w2 = 0.5 * tabs<double>(N).w[q % N] * tabs<double>(N).w[q / N] * cg[CG_DET * N2];
    sT *= w2;
    sD *= w2;
    sO *= w2;
  }
  __syncthreads();
  // the element's sums in a fixed order: rows of N threads, then the rows
  if (act) {
    A[r] = sT;
    A[PT + r] = sD;
    A[2 * PT + r] = sO;
  }
  __syncthreads();
  constexpr int RW = PT / N;  // rows per sum
  if (act && r < 3 * RW) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) t += A[r * N + i];
    B[r] = t;
  }
  __syncthreads();
  if (act && r == 0) {
    double t[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      t[0] += B[i];
      t[1] += B[RW + i];
      t[2] += B[2 * RW + i];
    }
    const double *lay = m.layer_c + 3 * m.slab_layer[s];
    const double c11 = lay[0], c12 = lay[1], c44 = lay[2];
    if (parts) {
      out[3 * (size_t)wi] = (c11 + 2.0 * c12) / 3.0 * t[0];
      out[3 * (size_t)wi + 1] = (c11 - c12) * (t[1] - t[0] / 3.0);
      out[3 * (size_t)wi + 2] = c44 * t[2];
    } else {
      out[wi] = fm(c12, t[0], fm(c11 - c12, t[1], c44 * t[2]));
    }
  }
}

// layer blockIdx.x: the sum of its element energies, slab by slab in a fixed
// order.  A block per layer: one block for all 41 layers of a mesh took 205 us,
// more than the other 20 us of the call together.
__global__ void layer_sum_kernel(const DevMesh m, const double *__restrict__ elem, double *__restrict__ out) {
  __shared__ double red[8];
  const int L = blockIdx.x;
  grid_wait();
  elem = after_wait(elem);
  double acc = 0.0;
  for (int s = 0; s < m.nslab; ++s) {
    if (m.slab_layer[s] != L) continue;
    for (int c = threadIdx.x; c < m.ncol; c += blockDim.x) acc += elem[(size_t)s * m.ncol + c];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
    out[L] = sum;
  }
}

// few elements (below 8 per SM, as for the operator): split pencils, one
// element per CTA (64 elements, p = 3: 32 us a call, 37 with whole pencils);
// else as many per CTA as its threads hold
template <int N>
cudaError_t launch_energy(const DevMesh &m, const DevMesh *meshes, const int2 *work, int nwork,
                          const long long *dof_off, const double *u, double *out, int parts, cudaStream_t st) {
  constexpr int EB = energy_eb<N>();
  if (apply_small(nwork)) {
    static int few_device = -1;
    const cudaError_t err = allow_smem(energy_pencil_kernel<N, true>, energy_smem<N, true>(1), few_device);
    if (err != cudaSuccess) return err;
    return launch_pdl(energy_pencil_kernel<N, true>, nwork, (3 * N * N + 31) / 32 * 32, energy_smem<N, true>(1), st, m,
                      meshes, work, dof_off, nwork, 1, u, out, parts);
  }
  static int configured_device = -1;
  const cudaError_t err = allow_smem(energy_pencil_kernel<N, false>, energy_smem<N, false>(EB), configured_device);
  if (err != cudaSuccess) return err;
  return launch_pdl(energy_pencil_kernel<N, false>, (nwork + EB - 1) / EB, (EB * N * N + 31) / 32 * 32,
                    energy_smem<N, false>(EB), st, m, meshes, work, dof_off, nwork, EB, u, out, parts);
}

cudaError_t energies(int N, const DevMesh &m, const DevMesh *meshes, const int2 *work, int nwork,
                     const long long *dof_off, const double *u, double *out, int parts, cudaStream_t st) {
  if (nwork <= 0) return cudaSuccess;
  switch (N) {
#define TN_CASE(NN) case NN: return launch_energy<NN>(m, meshes, work, nwork, dof_off, u, out, parts, st);
    TN_FOR_N(TN_CASE)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
void fill_tabs(const LglTables *t, ApplyTabs<T> *out) {
  for (int N = TN_MIN_N; N <= TN_MAX_N; ++N) {
    const int H = N / 2;
    ApplyTabs<T> &o = out[N];
    for (int a = 0; a < N; ++a) o.w[a] = (T)t->w[N][a];
    o.whalf = (T)(0.5 / t->w[N][0]);
    for (int tr = 0; tr < 2; ++tr) {
      auto D = [&](int a, int b) { return tr ? t->D[N][b * N + a] : t->D[N][a * N + b]; };
      for (int a = 0; a < H; ++a) {
        for (int b = 0; b < H; ++b) {
          o.eo[tr].em[a][b] = (T)(0.5 * (D(a, b) - D(a, N - 1 - b)));
          o.eo[tr].ep[a][b] = (T)(0.5 * (D(a, b) + D(a, N - 1 - b)));
        }
        if (N & 1) {
          o.eo[tr].ep[a][H] = (T)D(a, H);
          o.eo[tr].mid[a] = (T)D(H, a);
        }
      }
    }
  }
}

}  // namespace

cudaError_t tn_upload_lgl_apply(const LglTables *t) {
  static ApplyTabs<double> t64[TN_MAX_N + 1];
  static ApplyTabs<float> t32[TN_MAX_N + 1];
  fill_tabs(t, t64);
  fill_tabs(t, t32);
  cudaError_t err = cudaMemcpyToSymbol(c_t64, t64, sizeof(t64));
  if (err != cudaSuccess) return err;
  return cudaMemcpyToSymbol(c_t32, t32, sizeof(t32));
}

// variant 1 exists for FP32 only
cudaError_t tn_launch_apply(const ApplyArgs &a, cudaStream_t st) {
  if (!a.m) {
    if (apply_small(a.elems, a.sms))
      return a.prec == TN_F64 ? launch_batch<double, 0, AM_SMALL_BATCH>(a, st) : launch_batch<float, 0, AM_SMALL_BATCH>(a, st);
    if (a.prec == TN_F64) return launch_batch<double, 0, AM_PENCIL>(a, st);
    return a.var == 1 ? launch_batch<float, 1, AM_PENCIL>(a, st) : launch_batch<float, 0, AM_PENCIL>(a, st);
  }
  switch (a.m->N) {
#define TN_CASE(NN)                                            \
  case NN:                                                     \
    if (a.prec == TN_F64) return launch_mesh<NN, double, 0>(a, st); \
    return a.var == 1 ? launch_mesh<NN, float, 1>(a, st) : launch_mesh<NN, float, 0>(a, st);
    TN_FOR_N(TN_CASE)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t tn_launch_trace_add(const ApplyArgs &a, cudaStream_t st) {
  if (!a.m) return a.prec == TN_F64 ? launch_second_batch<double>(a, st) : launch_second_batch<float>(a, st);
  switch (a.m->N) {
#define TN_CASE(NN) \
  case NN: return a.prec == TN_F64 ? launch_second<NN, double>(a, st) : launch_second<NN, float>(a, st);
    TN_FOR_N(TN_CASE)
#undef TN_CASE
    default: return cudaErrorInvalidValue;
  }
}

bool tn_apply_few(int E) { return apply_small(E); }
int tn_apply_eb(int N, bool few) { return few ? kSmallBatchThreads / (3 * N * N) : kApplyThreads / (N * N); }
int tn_apply_parts(int N, int E) { return apply_small(E) ? E : (E + tn_apply_eb(N, false) - 1) / tn_apply_eb(N, false); }

int tn_trace_add_eb(int N, int elems) {
  switch (N) {
#define TN_CASE(NN) case NN: return add_elems(add_eb<NN>(), elems, tn_sm_count());
    TN_FOR_N(TN_CASE)
#undef TN_CASE
    default: return 1;
  }
}

// time per apply (us) of both FP32 variants: 3 untimed applies, then 10
// between CUDA events on st
cudaError_t tn_tune_apply(ApplyArgs a, cudaStream_t st, float us[2]) {
  cudaEvent_t ev[2];
  cudaError_t err = cudaEventCreate(&ev[0]);
  if (err != cudaSuccess) return err;
  err = cudaEventCreate(&ev[1]);
  if (err != cudaSuccess) {
    cudaEventDestroy(ev[0]);
    return err;
  }
  a.prec = TN_F32;
  a.partial = nullptr;
  a.fold = nullptr;
  for (int v = 0; v < 2 && err == cudaSuccess; ++v) {
    a.var = v;
    for (int i = 0; i < 13 && err == cudaSuccess; ++i) {
      if (i == 3) err = cudaEventRecord(ev[0], st);
      if (err == cudaSuccess) err = tn_launch_apply(a, st);
      if (err == cudaSuccess) err = tn_launch_trace_add(a, st);
    }
    if (err == cudaSuccess) err = cudaEventRecord(ev[1], st);
    if (err == cudaSuccess) err = cudaEventSynchronize(ev[1]);
    float ms = 0.0f;
    if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, ev[0], ev[1]);
    us[v] = ms * 100.0f;  // 10 applies: ms / 10 * 1000
  }
  cudaEventDestroy(ev[0]);
  cudaEventDestroy(ev[1]);
  return err;
}

cudaError_t tn_launch_energy(const DevMesh &m, const double *u, double *elem, double *layer, cudaStream_t st) {
  const cudaError_t err = energies(m.N, m, nullptr, nullptr, m.E, nullptr, u, elem, 0, st);
  if (err != cudaSuccess) return err;
  return launch_pdl(layer_sum_kernel, m.n_layers, 256, 0, st, m, (const double *)elem, layer);
}

cudaError_t tn_launch_energy_parts(const DevMesh &m, const double *u, double *parts, cudaStream_t st) {
  return energies(m.N, m, nullptr, nullptr, m.E, nullptr, u, parts, 1, st);
}

cudaError_t tn_launch_energy_batch(int N, const DevMesh *meshes, const int2 *work, int nwork, const long long *dof_off,
                                   const double *u, double *out, cudaStream_t st) {
  return energies(N, DevMesh{}, meshes, work, nwork, dof_off, u, out, 0, st);
}
