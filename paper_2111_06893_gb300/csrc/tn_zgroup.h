// Factor layouts of the grouped-line preconditioner (zgfactor.cu writes them,
// zgroup.cu solves with them).
#pragma once

#include "tn_device.h"

// FP32 record of slab s: [S_s^{-1} packed by columns (lower triangle,
// zlp(MG)) | O_{s-1} in factored form (8 MG) | W_s], S_s = L_s L_s^T the
// slab's Schur complement of the block Cholesky (S_s^{-1} = Linv_s^T
// Linv_s).  The coupling block O_{s-1} (rows: slab s - 1,
// columns: slab s, block diagonal over the lines) is nonzero only in the
// rows of the bottom-face nodes (k = 0) and the columns of the top-face
// nodes (k2 = N - 1) of each line (Eqs. (numflux), (penalty) on the zeta
// face), so O = E_0 X^T + Y E_{N-1}^T with per row t: X[t][a] = O[(a, 0), t]
// and Y[t][b] = O[t, (b, N - 1)] (Y zero on k = 0 rows).  Row t stores
// X[t][0..2], 0, Y[t][0..2], 0.  The solve applies the coupling through
// these factors instead of storing Z_s = Linv_{s-1} O_{s-1} densely.
// The record ends with the backward sweep's coupling W_s = S_s^{-1} [Y_s | E_0]
// (MG x 6G, rows padded to zp_ws(G)), S_s = L_s L_s^T the slab's Schur
// complement and Y_s, E_0 of O_s (the coupling to slab s + 1): per line l,
// column 6 l + b holds Y of component b and column 6 l + 3 + a the unit
// vector of row (a, k = 0); zero for the last slab.  With it the backward
// step x_s = Linv_s^T (y_s - Linv_s O_s x_{s+1}) = w_s - W_s v, v the six
// numbers per line x_{s+1}(b, N - 1) and X^T x_{s+1}.
__host__ __device__ constexpr int zp_ws(int G) { return pad4(6 * G); }
__host__ __device__ constexpr int zp_rec(int MG, int G) { return zlp(MG) + 8 * MG + MG * zp_ws(G); }

// FP64 solve.  The block O_{s-1} (rows: slab s - 1, columns: slab s, block
// diagonal over the lines) is nonzero only in the rows of the bottom-face
// nodes (k = 0) and the columns of the top-face nodes (k = N - 1) of each line
// (Eqs. (numflux), (penalty) on the zeta face), so O_{s-1} = U_{s-1} V_s^T
// with six columns per line l: U = [Y | E_0] (column 6 l + b: Y of component
// b; 6 l + 3 + a: the unit vector of row (a, k = 0)) and V = [E_{N-1} | X]
// (6 l + b: the unit vector of row (b, k = N - 1); 6 l + 3 + a: X of component
// a).  Only the zeta derivative couples away from the face node, so with D
// the derivative matrix
//   Y[(b, k)][b] = y_b D(0, k), k != 0;      X[(a, k)][a] = x_a D(N-1, k), k != N-1
// and X has a full 3 x 3 block in the rows k = N - 1 (all else zero): 15
// numbers per line.
//
// Elimination, S_s the slab's Schur complement, W_s = S_s^{-1} U_s and Q_s =
// S_s^{-1} V_s:
//   w_s = S_s^{-1} (r_s - V_s g_{s-1}),   g_s = U_s^T w_s
//   x_s = w_s - W_s f_{s+1},              f_s = V_s^T x_s
// As written (the FP32 solve) each slab waits for the full solve of the one
// above it (forward) or below it (backward): two chains of S dense products.
// But only the 6 g numbers g and f cross an interface:
//   a_s = S_s^{-1} r_s,   c_s = U_s^T a_s,   d_s = V_s^T a_s
//   g_s = c_s - K_s g_{s-1},   f_s = d_s - H_s g_{s-1} - K_s^T f_{s+1}
//   x_s = a_s - Q_s g_{s-1} - W_s f_{s+1}
// with K_s = W_s^T V_s and H_s = V_s^T Q_s (6 g x 6 g).  The dense products of
// all slabs are independent, and the chains run on 6 g numbers per step.
// The factors grow (12 g entries more per row, 72 g^2 more per slab) and the
// arithmetic shrinks: FP64 is bound by its arithmetic (an FP64 instruction
// occupies the pipe for 16 cycles whether 6 or 32 lanes are on, and the chain
// form spends most of them on packed triangles of few lanes), FP32 by the
// latency and bytes of the factors, so FP64 takes this form and FP32 the one
// above (FP64 | FP32, us: 2.0 M unknowns at p = 6: 669 -> 383 | 122 -> 176;
// p = 7, 11 slabs: 173 -> 156 | 48 -> 68; p = 4 box, 12288: 30 -> 19 | 13 -> 11).
//
// Factors of a group, three arrays in turn, every record padded to 16 bytes:
//   S_s^{-1}, s < S: by circulant diagonals, entry m MG + t = S^{-1}[t][(t + m)
//        mod MG], m = 0 .. MG / 2 (each entry of the symmetric matrix once, the
//        last diagonal of an even MG twice): a row reads two conflict-free
//        entries per diagonal.  Then 16 numbers per line of the coupling:
//        y_b of interface s, x_a of interface s - 1, X's 3 x 3 block [b][a]
//   (Q_s | W_s)^T, s < S: 12 g rows of pad4(MG) (Q_0 and W_{S-1} zero)
//   K_s | H_s, s < S: K by rows of odd stride 6 g + 1, H by rows of 6 g (used:
//        K_1 .. K_{S-2}, H_1 .. H_{S-1})
__host__ __device__ constexpr int zg_ld(int G) { return 6 * G + 1; }
__host__ __device__ constexpr int zg_circ(int MG) { return MG * (MG / 2 + 1); }
__host__ __device__ constexpr int zg_srec(int MG, int G) { return pad4(zg_circ(MG)) + 16 * G; }
__host__ __device__ constexpr int zg_qrec(int MG, int G) { return 12 * G * pad4(MG); }
__host__ __device__ constexpr int zg_kpart(int G) { return pad4(6 * G * zg_ld(G)); }
__host__ __device__ constexpr int zg_krec(int G) { return zg_kpart(G) + 36 * G * G; }
__host__ __device__ constexpr long long zg_qoff(int MG, int G, int S) { return (long long)S * zg_srec(MG, G); }
__host__ __device__ constexpr long long zg_koff(int MG, int G, int S) {
  return zg_qoff(MG, G, S) + (long long)S * zg_qrec(MG, G);
}
__host__ __device__ constexpr long long zg_entries(int MG, int G, int S) {
  return zg_koff(MG, G, S) + (long long)S * zg_krec(G);
}
