// fem_iso_mat.cuh -- the contraction of the non-affine Laplacian (Eqs. 17-19)
// and its adjoint, summed by the structure of K instead of entry by entry.
//
// With p_{k,a} = J^{-T}(vertex k) grad lambda_a (a = 0..D, zero sum over a)
// and lambda_k the projection's P1 basis,
//   A_ij = scale sum_{kl} (D+4)! int lambda_k lambda_l  D_i^k . D_j^l,
//   D_i^k = grad phi_i with p_{k,a} in the place of grad lambda_a.
// For a pair (x, y) of barycentric indices only the symmetric part over the
// vertices k, l counts: H_k = p_{k,x} . p_{k,y} and, for k < l,
// S_kl = p_{k,x} . p_{l,y} + p_{l,x} . p_{k,y}.  (D+4)! int of a monomial of
// degree four is the product of the factorials of its exponents, so the sums
// over k, l of (H, S) times int lambda_k lambda_l lambda_c lambda_d collapse to
//   q_c = 4 H_c + sum_{l != c} S_cl,   b = (sum_c q_c) / 2,
//   T_cd = b + q_c + q_d + S_cd,  T_cc = 2 (b + 2 q_c + 2 H_c),
//   with one lambda less:  (D+4) (b + q_c),  with two less:  (D+4)(D+3) b.
// Every entry of A is a short sum of these over the pairs that its basis
// functions' gradients hold (vertex function a: (4 lambda_a - 1) p_a; edge
// function (a, c): 4 (lambda_a p_c + lambda_c p_a)).  On P2 tetrahedra that is
// about 1100 operations an element where the entry-by-entry contraction takes
// 2538 FMAs and 78 dot products; on P1 an entry is (D+4)(D+3) b, five dot
// products.
#pragma once
#include "fem_iso.cuh"

namespace fem {

template <int D>
struct IsoMat {
  static constexpr int NV = D + 1, NB = (D + 1) * (D + 2) / 2;
  static constexpr float n1 = D + 4, n2 = (D + 4) * (D + 3);
  static constexpr __host__ __device__ int edge(int a, int c) {  // basis index of edge function (a, c)
    const int lo = a < c ? a : c, hi = a < c ? c : a;
    return NV + lo * (2 * NV - lo - 1) / 2 + (hi - lo - 1);
  }
  static constexpr __host__ __device__ int entry(int i, int j) {  // upper triangle of A, rows of NB
    return i < j ? pair_index(i, j, NB) : pair_index(j, i, NB);
  }
};

// p_{k,0} = -sum_{a>0} p_{k,a}; p_{k,a} = ji[k][a-1] for a > 0.
template <int D>
__device__ __forceinline__ void iso_p0(const float (&ji)[D + 1][D][D], float (&p0)[D + 1][D]) {
#pragma unroll
  for (int k = 0; k <= D; ++k)
#pragma unroll
    for (int al = 0; al < D; ++al) {
      float s = -ji[k][0][al];
#pragma unroll
      for (int a = 1; a < D; ++a) s -= ji[k][a][al];
      p0[k][al] = s;
    }
}

template <int D>
__device__ __forceinline__ float iso_dot(const float* u, const float* v) {
  float s = u[0] * v[0];
#pragma unroll
  for (int al = 1; al < D; ++al) s = fmaf(u[al], v[al], s);
  return s;
}

// P1: acc[(i, j)] = (D+4)(D+3) b of the pair (i, j), b = P_i . P_j + sum_k p_{k,i} . p_{k,j}
// with P_i = sum_k p_{k,i}.  Every pair directly, the small terms first: taking
// the entries of index 0 from the zero row sums doubles the largest error
// (8.0e-7 against 4.5e-7 of an element's largest entry, warped 128^3 cube).
template <int D>
__device__ __forceinline__ void iso_matrix_p1(const float (&ji)[D + 1][D][D], float* acc) {
  constexpr int NV = D + 1;
  float p0[NV][D], P[NV][D];
  iso_p0<D>(ji, p0);
#pragma unroll
  for (int a = 0; a < NV; ++a)
#pragma unroll
    for (int al = 0; al < D; ++al) {
      float s = a ? ji[0][a ? a - 1 : 0][al] : p0[0][al];
#pragma unroll
      for (int k = 1; k < NV; ++k) s += a ? ji[k][a ? a - 1 : 0][al] : p0[k][al];
      P[a][al] = s;
    }
#pragma unroll
  for (int x = 0; x < NV; ++x)
#pragma unroll
    for (int y = x; y < NV; ++y) {
      float b = 0.f;  // the small terms first, the large one last
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const float* kx = x ? ji[k][x ? x - 1 : 0] : p0[k];
        const float* ky = y ? ji[k][y ? y - 1 : 0] : p0[k];
#pragma unroll
        for (int al = 0; al < D; ++al) b = fmaf(kx[al], ky[al], b);
      }
      acc[pair_index(x, y, NV)] = IsoMat<D>::n2 * (b + iso_dot<D>(P[x], P[y]));
    }
}

// P2: acc[(i, j)] of the upper triangle, without the common factor.
template <int D>
__device__ __forceinline__ void iso_matrix_p2(const float (&ji)[D + 1][D][D], float* acc) {
  using M = IsoMat<D>;
  constexpr int NV = M::NV;
  constexpr float n1 = M::n1, n2 = M::n2;
  float p0[NV][D];
  iso_p0<D>(ji, p0);
#pragma unroll
  for (int t = 0; t < M::NB * (M::NB + 1) / 2; ++t) acc[t] = 0.f;
#pragma unroll
  for (int x = 0; x < NV; ++x)
#pragma unroll
    for (int y = x; y < NV; ++y) {
      float S[NV][NV], q[NV];  // S[c][c] holds H_c
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const float* kx = x ? ji[k][x ? x - 1 : 0] : p0[k];
        const float* ky = y ? ji[k][y ? y - 1 : 0] : p0[k];
        S[k][k] = iso_dot<D>(kx, ky);
#pragma unroll
        for (int l = k + 1; l < NV; ++l) {
          const float* lx = x ? ji[l][x ? x - 1 : 0] : p0[l];
          const float* ly = y ? ji[l][y ? y - 1 : 0] : p0[l];
          float s = iso_dot<D>(kx, ly);
          if (x == y) {
            s += s;
          } else {
#pragma unroll
            for (int al = 0; al < D; ++al) s = fmaf(lx[al], ky[al], s);
          }
          S[k][l] = s;
          S[l][k] = s;
        }
      }
      float b = 0.f;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        float s = 4.f * S[c][c];
#pragma unroll
        for (int l = 0; l < NV; ++l)
          if (l != c) s += S[c][l];
        q[c] = s;
        b += s;
      }
      b *= 0.5f;
      // vertex - vertex
      if (x == y)
        acc[M::entry(x, x)] = fmaf(32.f - 8.f * n1 + n2, b, fmaf(64.f - 8.f * n1, q[x], 64.f * S[x][x]));
      else
        acc[M::entry(x, y)] = fmaf(16.f - 8.f * n1 + n2, b, fmaf(16.f - 4.f * n1, q[x] + q[y], 16.f * S[x][y]));
      // vertex v of the pair - edge (u, c), u the other one
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 1 && x == y) continue;
        const int v = side ? y : x, u = side ? x : y;
        const float zv = fmaf(16.f, q[v], (16.f - 4.f * n1) * b);
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          if (c == u) continue;
          const float z = c == v ? fmaf(64.f - 4.f * n1, q[v], fmaf(32.f - 4.f * n1, b, 64.f * S[v][v]))
                                 : fmaf(16.f - 4.f * n1, q[c], fmaf(16.f, S[v][c], zv));
          acc[M::entry(v, M::edge(u, c))] += z;
        }
      }
      // edge (x, c) - edge (y, d): T_cd once per ordered choice of the two gradients
      float h[NV];
#pragma unroll
      for (int c = 0; c < NV; ++c) h[c] = fmaf(0.5f, b, q[c]);
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        if (c == x) continue;
#pragma unroll
        for (int d = 0; d < NV; ++d) {
          if (d == y || (x == y && d < c)) continue;
          const float t = c == d ? 4.f * (h[c] + S[c][c]) : h[c] + h[d] + S[c][d];
          const bool twice = x != y && c == y && d == x;  // the edge (x, y) with itself
          acc[M::entry(M::edge(x, c), M::edge(y, d))] += twice ? t + t : t;
        }
      }
    }
  // the edge - edge entries carry 4 * 4 from the basis functions
#pragma unroll
  for (int i = NV; i < M::NB; ++i)
#pragma unroll
    for (int j = i; j < M::NB; ++j) acc[M::entry(i, j)] *= 16.f;
}

// Adjoint: for s = sym(dA) over the upper triangle (s_ij = dA_ij + dA_ji off
// the diagonal), u[k][a-1] = d/dp_{k,a} of sum_T s_T acc_T (without the common
// factor), p_{k,0} already folded in.  acc is homogeneous of degree two in p,
// so sum_T s_T acc_T = sum u . p / 2 (Euler): the caller needs no acc.
template <int D>
__device__ __forceinline__ void iso_adjoint_p1(const float* s, const float (&ji)[D + 1][D][D],
                                                        float (&u)[D + 1][D][D]) {
  constexpr int NV = D + 1;
  constexpr float n2 = IsoMat<D>::n2;
  float P[D][D], w[D][D];  // w: weight of the pair (x, y) once index 0 is folded in
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int al = 0; al < D; ++al) {
      float t = ji[0][a][al];
#pragma unroll
      for (int k = 1; k < NV; ++k) t += ji[k][a][al];
      P[a][al] = t;
    }
#pragma unroll
  for (int x = 1; x < NV; ++x)
#pragma unroll
    for (int y = x; y < NV; ++y) {
      const float t = x == y ? 2.f * (s[pair_index(x, x, NV)] - s[pair_index(0, x, NV)] + s[0])
                             : s[pair_index(x, y, NV)] - s[pair_index(0, x, NV)] - s[pair_index(0, y, NV)] + 2.f * s[0];
      w[x - 1][y - 1] = n2 * t;
      w[y - 1][x - 1] = n2 * t;
    }
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int x = 0; x < D; ++x)
#pragma unroll
      for (int al = 0; al < D; ++al) {
        float t = w[x][0] * (P[0][al] + ji[k][0][al]);
#pragma unroll
        for (int y = 1; y < D; ++y) t = fmaf(w[x][y], P[y][al] + ji[k][y][al], t);
        u[k][x][al] = t;
      }
}

template <int D, class Sym>
__device__ __forceinline__ void iso_adjoint_p2(const Sym& s, const float (&ji)[D + 1][D][D],
                                                        float (&u)[D + 1][D][D]) {
  using M = IsoMat<D>;
  constexpr int NV = M::NV;
  constexpr float n1 = M::n1, n2 = M::n2;
  float p0[NV][D], u0[NV][D];
  iso_p0<D>(ji, p0);
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int al = 0; al < D; ++al) {
      u0[k][al] = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) u[k][a][al] = 0.f;
    }
#pragma unroll
  for (int x = 0; x < NV; ++x)
#pragma unroll
    for (int y = x; y < NV; ++y) {
      float gS[NV][NV], gq[NV], gb;  // gradients of S (k < l; H on the diagonal), q and b
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        gq[c] = 0.f;
#pragma unroll
        for (int d = c; d < NV; ++d) gS[c][d] = 0.f;
      }
      auto at = [&](int c, int d) -> float& { return gS[c < d ? c : d][c < d ? d : c]; };
      // vertex - vertex
      const float vv = s(M::entry(x, y));
      if (x == y) {
        gb = (32.f - 8.f * n1 + n2) * vv;
        gq[x] = (64.f - 8.f * n1) * vv;
        gS[x][x] = 64.f * vv;
      } else {
        gb = (16.f - 8.f * n1 + n2) * vv;
        gq[x] = (16.f - 4.f * n1) * vv;
        gq[y] = gq[x];
        gS[x][y] = 16.f * vv;
      }
      // vertex - edge
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 1 && x == y) continue;
        const int v = side ? y : x, o = side ? x : y;
        float zsum = 0.f;  // of the entries with c != v
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          if (c == o) continue;
          const float z = s(M::entry(v, M::edge(o, c)));
          if (c == v) {
            gq[v] = fmaf(64.f - 4.f * n1, z, gq[v]);
            gb = fmaf(32.f - 4.f * n1, z, gb);
            at(v, v) = fmaf(64.f, z, at(v, v));
          } else {
            gq[c] = fmaf(16.f - 4.f * n1, z, gq[c]);
            at(v, c) = fmaf(16.f, z, at(v, c));
            zsum += z;
          }
        }
        gq[v] = fmaf(16.f, zsum, gq[v]);
        gb = fmaf(16.f - 4.f * n1, zsum, gb);
      }
      // edge - edge
      float gh[NV];
#pragma unroll
      for (int c = 0; c < NV; ++c) gh[c] = 0.f;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        if (c == x) continue;
#pragma unroll
        for (int d = 0; d < NV; ++d) {
          if (d == y || (x == y && d < c)) continue;
          const bool twice = x != y && c == y && d == x;
          const float t = (twice ? 32.f : c == d ? 64.f : 16.f) * s(M::entry(M::edge(x, c), M::edge(y, d)));
          gh[c] += t;
          if (c != d) gh[d] += t;
          at(c, d) += t;
        }
      }
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        gq[c] += gh[c];
        gb = fmaf(0.5f, gh[c], gb);
      }
      gb *= 0.5f;  // b = (sum q) / 2
#pragma unroll
      for (int c = 0; c < NV; ++c) gq[c] += gb;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        gS[c][c] = fmaf(4.f, gq[c], gS[c][c]);
#pragma unroll
        for (int d = c + 1; d < NV; ++d) gS[c][d] += gq[c] + gq[d];
      }
      // S = products of p
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const float* kx = x ? ji[k][x ? x - 1 : 0] : p0[k];
        const float* ky = y ? ji[k][y ? y - 1 : 0] : p0[k];
        float* ukx = x ? u[k][x ? x - 1 : 0] : u0[k];
        float* uky = y ? u[k][y ? y - 1 : 0] : u0[k];
#pragma unroll
        for (int al = 0; al < D; ++al) {
          if (x == y) {
            ukx[al] = fmaf(2.f * gS[k][k], kx[al], ukx[al]);
          } else {
            ukx[al] = fmaf(gS[k][k], ky[al], ukx[al]);
            uky[al] = fmaf(gS[k][k], kx[al], uky[al]);
          }
        }
#pragma unroll
        for (int l = k + 1; l < NV; ++l) {
          const float* lx = x ? ji[l][x ? x - 1 : 0] : p0[l];
          const float* ly = y ? ji[l][y ? y - 1 : 0] : p0[l];
          float* ulx = x ? u[l][x ? x - 1 : 0] : u0[l];
          float* uly = y ? u[l][y ? y - 1 : 0] : u0[l];
          const float g = x == y ? 2.f * gS[k][l] : gS[k][l];
#pragma unroll
          for (int al = 0; al < D; ++al) {
            ukx[al] = fmaf(g, ly[al], ukx[al]);
            uly[al] = fmaf(g, kx[al], uly[al]);
            if (x != y) {
              ulx[al] = fmaf(g, ky[al], ulx[al]);
              uky[al] = fmaf(g, lx[al], uky[al]);
            }
          }
        }
      }
    }
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int al = 0; al < D; ++al) u[k][a][al] -= u0[k][al];
}

}  // namespace fem
