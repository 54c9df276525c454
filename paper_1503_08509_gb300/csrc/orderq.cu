// Screens of order q >= 2 (Sec. 2.1, Eq. moment1d) on the order p = q + 2 mesh
// (Sec. 2: p = q + 2): potentials and energy.
//
// The stages of Algorithm 1 for a general order:
//   coefficients  C[e][kappa] = sum_{j in e} Q_j c_kappa(delta_j) on the element's
//                 (q+1)^3 screen nodes (Eq. oned, Eq. moment1d; the weights are
//                 polynomials in delta / h made on the host);
//   density       r on the periodic order-q mesh (Eq. assign): the element lists
//                 added at the shared nodes;
//   load vector   b = 4 pi (Mpq (x) Mpq (x) Mpq) r, less its neutralising
//                 background (Sec. 2.2);
//   mesh solve    K phi = b, int phi = 0, by iterative refinement: the residual
//                 in FP64 (separable banded passes of the order-p matrices),
//                 the correction by the FP32 fast-diagonalisation solve of the
//                 order-p mesh (the tensor-core transform passes of the order-3
//                 mesh with the order-p eigenbasis);
//   screen field  S[e][m] = sum over the screen nodes o of e's block of the
//                 node's amplitude times the FE table of its type at node m of
//                 e (Eq. sc with the tables of the Remark of Sec. 4, in the
//                 node-regrouped layout), split by the tables' mirror
//                 symmetries into eight blocks, double-float arithmetic;
//   evaluation    Phi_t = sum_m (phi - S)[e_t][m] u_m(tau_t) + the singular sum
//                 over the block (Eq. evalsmooth, Sec. 2.4), and U (FP64).
// One-element screens (Sec. 5.3) are the same stages with weights on the
// element's interior nodes only.  Both precisions take this path in FP64 or
// double-float arithmetic, except the FP32 inner solve of the refinement and,
// in the mixed precision, the FP32 singular sums.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "df.cuh"
#include "gridsum.cuh"

namespace fep3m {

namespace {

constexpr int OT = 256;

__device__ __forceinline__ int wrapq(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

inline unsigned gsz(int64_t n, int t = OT) { return (unsigned)((n + t - 1) / t); }

// C[e][kappa], one thread per (element, screen node); kappa = i + (q+1)(j + (q+1) k).
// Here and in the density, the copy as float pairs for the screen contraction is times a
// power of two near the inverse mean charge, so that the pairs' low words stay normal.
template <class V4>
__global__ void k_oq_coeff(int64_t ne, OQParams prm, const int* __restrict__ start, const int* __restrict__ count,
                           const V4* __restrict__ part, double scale, double* __restrict__ C, df* __restrict__ Cp) {
  const int q = prm.q, Q1 = q + 1, nk = Q1 * Q1 * Q1;
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= ne * nk) return;
  const int64_t e = g / nk;
  const int kap = (int)(g - e * nk);
  const int ki[3] = {kap % Q1, (kap / Q1) % Q1, kap / (Q1 * Q1)};
  double acc = 0.0;
  const int s0 = start[e], cnt = count[e];
  for (int j = s0; j < s0 + cnt; ++j) {
    const V4 pj = part[j];
    const double t[3] = {(double)pj.x - 0.5, (double)pj.y - 0.5, (double)pj.z - 0.5};   // delta / h
    double w = (double)pj.w;
    for (int a = 0; a < 3; ++a) {
      const double* Wr = prm.W + ki[a] * Q1;
      double v = Wr[q];
      for (int l = q - 1; l >= 0; --l) v = fma(v, t[a], Wr[l]);   // Horner
      w *= v;
    }
    acc += w;
  }
  C[g] = acc;
  Cp[g] = df_split(acc * scale);
}

// r on the order-q mesh: node g of an axis is local node g mod q of element
// g / q, and for g mod q = 0 also local node q of the element before
__global__ void k_oq_density(int n, int q, const double* __restrict__ C, double scale, double* __restrict__ r,
                             df* __restrict__ rp) {
  const int Nq = q * n, Q1 = q + 1, nk = Q1 * Q1 * Q1;
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= (int64_t)Nq * Nq * Nq) return;
  const int gg[3] = {(int)(g % Nq), (int)((g / Nq) % Nq), (int)(g / ((int64_t)Nq * Nq))};
  int el[3][2], lo[3][2], cnt[3];
  for (int a = 0; a < 3; ++a) {
    el[a][0] = gg[a] / q;
    lo[a][0] = gg[a] - q * el[a][0];
    cnt[a] = 1;
    if (lo[a][0] == 0) {
      el[a][1] = wrapq(el[a][0] - 1, n);
      lo[a][1] = q;
      cnt[a] = 2;
    }
  }
  double acc = 0.0;
  for (int c = 0; c < cnt[2]; ++c)
    for (int b = 0; b < cnt[1]; ++b)
      for (int a = 0; a < cnt[0]; ++a) {
        const int64_t e = el[0][a] + (int64_t)n * (el[1][b] + (int64_t)n * el[2][c]);
        acc += C[e * nk + lo[0][a] + Q1 * (lo[1][b] + Q1 * lo[2][c])];
      }
  r[g] = acc;
  rp[g] = df_split(acc * scale);
}

// the screen nodes that order-p node g of an axis couples to, with the mixed
// mass weights: element g / p with local index g mod p, and for g mod p = 0
// also the element before with local index p
__device__ __forceinline__ int oq_mpq_row(int g, int n, const OQParams& prm, int node[10], double wgt[10]) {
  const int p = prm.p, q = prm.q, Q1 = q + 1, Nq = q * n;
  const int e = g / p, t = g - p * e;
  int k = 0;
  for (int j = 0; j <= q; ++j, ++k) {
    node[k] = wrapq(q * e + j, Nq);
    wgt[k] = prm.Mpq[t * Q1 + j];
  }
  if (t == 0)
    for (int j = 0; j <= q; ++j, ++k) {
      node[k] = wrapq(q * (e - 1) + j, Nq);
      wgt[k] = prm.Mpq[p * Q1 + j];
    }
  return k;
}

// One axis of b = 4 pi (Mpq (x) Mpq (x) Mpq) r, three separable passes (x, y,
// then z; the extents d are p n along the axes done, q n along the others, the
// input's q n along this one): up to 2 (q + 1) terms a node and pass instead
// of their cube (n = 15, q = 2: 136 -> 16 us)
__global__ void k_oq_load(int n, int axis, int d0, int d1, int d2, OQParams prm, const double* __restrict__ in,
                          double* __restrict__ out, double scale) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= (int64_t)d0 * d1 * d2) return;
  int idx[3] = {(int)(g % d0), (int)((g / d0) % d1), (int)(g / ((int64_t)d0 * d1))};
  int din[3] = {d0, d1, d2};
  din[axis] = prm.q * n;
  const int64_t st[3] = {1, din[0], (int64_t)din[0] * din[1]};
  int node[10];
  double w[10];
  const int k = oq_mpq_row(idx[axis], n, prm, node, w);
  idx[axis] = 0;
  const int64_t base = idx[0] + st[1] * idx[1] + st[2] * idx[2];
  double acc = 0.0;
  for (int j = 0; j < k; ++j) acc += w[j] * in[base + node[j] * st[axis]];
  out[g] = scale * acc;
}

__device__ __forceinline__ double oq_w3(int64_t g, int Np, const OQParams& prm) {
  const int p = prm.p;
  return prm.wn[(int)(g % Np) % p] * prm.wn[(int)((g / Np) % Np) % p] * prm.wn[(int)(g / ((int64_t)Np * Np)) % p];
}

// deterministic FP64 sum of v (weighted: of w3 v, w3 the node integrals) into *out
__global__ void __launch_bounds__(OT) k_oq_sum(int64_t len, int Np, OQParams prm, int weighted,
                                               const double* __restrict__ v, double* __restrict__ partial,
                                               unsigned int* __restrict__ counter, double* __restrict__ out) {
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)OT + threadIdx.x; i < len; i += (int64_t)gridDim.x * OT)
    acc += weighted ? oq_w3(i, Np, prm) * v[i] : v[i];
  double t;
  if (grid_sum256(acc, gridDim.x, blockIdx.x, partial, counter, t)) *out = t;
}

// out = in - s w3 (the load less its uniform background), s = *sum / n^3, with
// sum out^2 into *norm and the refinement's state
__global__ void __launch_bounds__(OT) k_oq_project(int Np, OQParams prm, const double* __restrict__ sum, double inv,
                                                   const double* __restrict__ in, double* __restrict__ out,
                                                   double* __restrict__ partial, unsigned int* __restrict__ counter,
                                                   double* __restrict__ norm, double rtol,
                                                   RefineState* __restrict__ st) {
  const int64_t len = (int64_t)Np * Np * Np;
  const double m = *sum * inv;
  double acc = 0.0;
  for (int64_t g = blockIdx.x * (int64_t)OT + threadIdx.x; g < len; g += (int64_t)gridDim.x * OT) {
    const double v = in[g] - m * oq_w3(g, Np, prm);
    out[g] = v;
    acc = fma(v, v, acc);
  }
  double t;
  if (grid_sum256(acc, gridDim.x, blockIdx.x, partial, counter, t)) {
    *norm = t;
    refine_begin(t, (double)len, rtol, st);
  }
}
// v -= *sum / n^3 (the mean)
__global__ void k_oq_mean(int64_t len, const double* __restrict__ sum, double inv, double* __restrict__ v) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < len) v[g] -= *sum * inv;
}

// The residual pb - K phi on the periodic order-p mesh in three separable
// banded passes, each reading its inputs once (rows by node type t = g mod p:
// an interior node couples to its element's p + 1 nodes only):
//   z:  a = M_z phi, b = K_z phi
//   y:  c = M_y a, f = K_y a + M_y b
//   x:  r = pb - (K_x c + M_x f), written as FP32 times the scale, with the sum
//       of its squares into *norm
// (n = 15, q = 2: 6 launches, 60 us -> 3 launches, 45 us.)
template <int AXIS>
__global__ void __launch_bounds__(OT) k_oq_band(int Np, OQParams prm, const double* __restrict__ in,
                                                const double* __restrict__ in2, double* __restrict__ o1,
                                                double* __restrict__ o2, const double* __restrict__ pb,
                                                RefineState* state, float* __restrict__ r32,
                                                double* __restrict__ partial, unsigned int* __restrict__ counter,
                                                double* __restrict__ norm) {
  const int64_t g = blockIdx.x * (int64_t)OT + threadIdx.x, len = (int64_t)Np * Np * Np;
  const int p = prm.p;
  double sq = 0.0;
  if (g < len) {
    const int64_t st = AXIS == 0 ? 1 : (AXIS == 1 ? Np : (int64_t)Np * Np);
    const int ga = AXIS == 0 ? (int)(g % Np) : (AXIS == 1 ? (int)((g / Np) % Np) : (int)(g / ((int64_t)Np * Np)));
    const int t = ga % p, lo = t == 0 ? 0 : p - t, hi = t == 0 ? 2 * p : 2 * p - t;
    const int64_t b0 = g - ga * st;
    const double *M = prm.bM[t], *K = prm.bK[t];
    double s1 = 0.0, s2 = 0.0;
    for (int o = lo; o <= hi; ++o) {
      int ja = ga + o - p;
      ja = ja < 0 ? ja + Np : (ja >= Np ? ja - Np : ja);
      const int64_t j = b0 + ja * st;
      const double v = in[j];
      if (AXIS == 2) {
        s1 = fma(M[o], v, s1);
        s2 = fma(K[o], v, s2);
      } else if (AXIS == 1) {
        s1 = fma(M[o], v, s1);
        s2 = fma(K[o], v, fma(M[o], in2[j], s2));
      } else {
        s1 = fma(K[o], v, fma(M[o], in2[j], s1));
      }
    }
    if (AXIS == 0) {
      const float r = (float)((pb[g] - s1) * (double)state->scale);
      r32[g] = r;
      sq = (double)r * (double)r;
    } else {
      o1[g] = s1;
      o2[g] = s2;
    }
  }
  if (AXIS == 0) {
    double total;
    if (grid_sum256(sq, gridDim.x, blockIdx.x, partial, counter, total)) {
      *norm = total;
      if (total <= state->limit) state->inv = 0.f;
    }
  }
}

__global__ void k_oq_round(int64_t n, const double* __restrict__ in, const RefineState* __restrict__ st,
                           float* __restrict__ out) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < n) out[g] = (float)(in[g] * (double)st->scale);
}
__global__ void k_oq_add(int64_t n, const float* __restrict__ x, const RefineState* __restrict__ st,
                         double* __restrict__ phi, int first) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const float inv = st->inv;   // a power of two, or zero: an earlier sweep reached the tolerance
  if (inv != 0.f && g < n) phi[g] = (first ? 0.0 : phi[g]) + (double)(x[g] * inv);
}

// ------------------------------------------------------------ screen field
// S[e][m] = sum_o A_e(o) H(o, m): the U^3 screen nodes o of e's block (per axis
// o = q (n_sr + 1) - u, U = (2 n_sr + 1) q + 1), their amplitudes A_e (the
// nodal density inside the block; at its boundary nodes the terms of the
// block's own elements) and the table at e's (p + 1)^3 nodes m.
//
// The block and the tables are symmetric under reflection of each axis about
// the element's centre, H(U - 1 - o, p - m) = H(o, m), so with the even and odd
// parts of A and of S per axis,
//   A+-(i) = A(i) +- A(U - 1 - i)  (the centre node of an odd U: even, once),
//   S(j) = S+(j) + S-(j),  S(p - j) = S+(j) - S-(j),
// the contraction falls into eight independent ones (b = sx + 2 sy + 4 sz),
// each with about half the nodes along every axis: 54 872 multiply-adds an
// element instead of 421 875 (q = 2, n_sr = 3; without the regrouping by
// nodes, 1.16 M).  S stays in its even and odd parts: the evaluation contracts
// them with the even and odd parts of the shape functions.
//
// Two launches per piece of elements (a piece's parts of A fit the L2 cache):
//   k_oq_amps  one CTA per element and parity along z: A gathered and split by
//              parity in shared memory
//   k_oq_gemm  per tile of elements and block b the product in double-float
//              arithmetic, eight elements and one node per thread, 32 nodes of
//              the block at a time in pairs and across them in three floats
//              (relative to sum |A H| about 1e-15; an FP64 multiply-add costs as
//              much as 64 FP32 operations, one in pairs 11).
// n = 15, q = 2 (3375 elements): 8917 -> 298 us.
struct ParityBlocks {
  int U, P1;
  int K[8], koff[9], M[8], moff[9];   // nodes of A and S per block and their offsets
};
__host__ __device__ inline int part_len(int len, int odd) { return odd ? len / 2 : (len + 1) / 2; }
inline ParityBlocks parity_blocks(int U, int P1) {
  ParityBlocks pb;
  pb.U = U;
  pb.P1 = P1;
  pb.koff[0] = pb.moff[0] = 0;
  for (int b = 0; b < 8; ++b) {
    pb.K[b] = part_len(U, b & 1) * part_len(U, (b >> 1) & 1) * part_len(U, b >> 2);
    pb.M[b] = part_len(P1, b & 1) * part_len(P1, (b >> 1) & 1) * part_len(P1, b >> 2);
    pb.koff[b + 1] = pb.koff[b] + pb.K[b];
    pb.moff[b + 1] = pb.moff[b] + pb.M[b];
  }
  return pb;
}

// grid (elements of the piece, parity along z): the half of the planes the
// parity keeps in shared memory (27 KB for q = 2; 208 KB for q = 4, n_sr = 4)
__global__ void __launch_bounds__(OT) k_oq_amps(int n, int n_sr, int q, ParityBlocks pb, int64_t e0,
                                                const int* __restrict__ count, const df* __restrict__ Cp,
                                                const df* __restrict__ rp, df* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  df* A = reinterpret_cast<df*>(smem);   // [part_len(U, sz)][U][U]
  __shared__ int node[3][40];            // the density's node of offset o per axis, times its stride
  const int64_t e = e0 + blockIdx.x;
  if (count[e] == 0) return;
  const int sz = blockIdx.y, U = pb.U, UU = U * U, nz = part_len(U, sz), tid = threadIdx.x;
  const int Nq = q * n, Q1 = q + 1, nk = Q1 * Q1 * Q1;
  const int E[3] = {(int)(e % n), (int)((e / n) % n), (int)(e / ((int64_t)n * n))};
  for (int i = tid; i < 3 * U; i += OT) {   // U <= 37
    const int a = i / U, o = i - a * U;
    node[a][o] = wrapq(q * E[a] + q * (n_sr + 1) - o, Nq) * (a == 0 ? 1 : (a == 1 ? Nq : Nq * Nq));
  }
  __syncthreads();
  auto amplitude = [&](int ox, int oy, int oz) -> df {
    if (ox > 0 && ox < U - 1 && oy > 0 && oy < U - 1 && oz > 0 && oz < U - 1)
      return rp[node[0][ox] + node[1][oy] + node[2][oz]];
    // the block's elements that hold the node: per axis floor(u / q), and for a
    // vertex also the element before, as far as they lie in the block
    const int o[3] = {ox, oy, oz};
    int el[3][2], lo[3][2], cnt[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int w = q * (2 * n_sr + 1) - o[a];   // u + q n_sr >= 0
      const int d = w / q, l = w - q * d;          // element d - n_sr of the block, local node l
      const bool first = d <= 2 * n_sr, second = l == 0 && d > 0;
      cnt[a] = (first ? 1 : 0) + (second ? 1 : 0);
      el[a][0] = wrapq(E[a] + (first ? d : d - 1) - n_sr, n);
      lo[a][0] = first ? l : q;
      el[a][1] = wrapq(E[a] + d - 1 - n_sr, n);
      lo[a][1] = q;
    }
    df v = {0.f, 0.f};
    for (int z = 0; z < cnt[2]; ++z)
      for (int y = 0; y < cnt[1]; ++y)
        for (int x = 0; x < cnt[0]; ++x)
          v = df_add(v, Cp[(el[0][x] + (int64_t)n * (el[1][y] + (int64_t)n * el[2][z])) * nk + lo[0][x] +
                           Q1 * (lo[1][y] + Q1 * lo[2][z])]);
    return v;
  };
  for (int i = tid; i < UU * nz; i += OT) {
    const int r = i / U, ox = i - r * U, oz = r / U, oy = r - oz * U;
    df v = amplitude(ox, oy, oz);
    if (2 * oz + 1 != U) {   // with its mirror image along z (the centre plane is its own)
      df w = amplitude(ox, oy, U - 1 - oz);
      if (sz) w = {-w.h, -w.l};
      v = df_add(v, w);
    }
    A[i] = v;
  }
  // sums and differences of mirrored nodes along x, then y
  const int half = U / 2;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    __syncthreads();
    for (int i = tid; i < half * U * nz; i += OT) {
      const int k = i % half, r = i / half;   // r: the row (y, z) for x, the column (x, z) for y
      const int base = a == 0 ? U * r : r % U + UU * (r / U), st = a == 0 ? 1 : U;
      df &x = A[base + k * st], &y = A[base + (U - 1 - k) * st];
      const df s = df_add(x, y), d = df_add(x, df{-y.h, -y.l});
      x = s;
      y = d;
    }
  }
  __syncthreads();
  df* dst = out + blockIdx.x * (int64_t)pb.koff[8];
  const int ke = part_len(U, 0), ko = part_len(U, 1);
  for (int i = tid; i < UU * nz; i += OT) {
    const int r = i / U, ox = i - r * U, kz = r / U, oy = r - kz * U;
    const int sx = ox >= ke, sy = oy >= ke;
    const int kx = sx ? U - 1 - ox : ox, ky = sy ? U - 1 - oy : oy;
    dst[pb.koff[sx + 2 * sy + 4 * sz] + kx + (sx ? ko : ke) * (ky + (sy ? ko : ke) * kz)] = A[i];
  }
}

// grid (tiles of elements, 8 blocks): S parts of elements e0 + [0, ne).  A
// thread takes eight elements and one node; where a block has few nodes, the
// contraction is dealt to several threads and added at the end.
// The next chunk of A is fetched into registers and that of the table copied
// to shared memory asynchronously while this one is multiplied (with the loads
// in the loop each step waited for the L2 cache: 651 -> 165 us for 3375 elements).
constexpr int GK = 32, GE = 8, GMAX = 64;   // contraction chunk, elements per thread, elements per tile
constexpr size_t GSMEM = 2 * GK * (GMAX + 2) * sizeof(df) + 2 * GK * 64 * sizeof(df);
__global__ void __launch_bounds__(OT, 2) k_oq_gemm(ParityBlocks pb, int64_t e0, int ne, const df* __restrict__ A,
                                                   const df* __restrict__ H, double* __restrict__ S) {
  extern __shared__ __align__(16) unsigned char smem[];
  df(*As)[GK][GMAX + 2] = reinterpret_cast<df(*)[GK][GMAX + 2]>(smem);            // [2]
  df(*Hs)[GK * 64] = reinterpret_cast<df(*)[GK * 64]>(smem + 2 * GK * (GMAX + 2) * sizeof(df));   // [2]
  double* red = reinterpret_cast<double*>(smem);                                  // OT GE / 2, at the end
  const int b = blockIdx.y, K = pb.K[b], M = pb.M[b], U3 = pb.koff[8], P3 = pb.moff[8], tid = threadIdx.x;
  int G = GMAX / GE;                      // groups of eight elements per tile
  while (G > 1 && G * M > OT) G >>= 1;
  const int TE = GE * G, t0 = blockIdx.x * TE;
  if (t0 >= ne) return;
  const int per = G * M;                  // threads per slice of the contraction; M <= 64, so per <= OT
  const int NS = OT / per, sl = tid / per, r = tid - sl * per, g = r / M, m = r - g * M;
  const bool on = sl < NS;
  const df* Hb = H;
  for (int k = 0; k < b; ++k) Hb += (int64_t)pb.K[k] * pb.M[k];
  const df* Ab = A + (int64_t)t0 * U3 + pb.koff[b];
  df pre[GMAX * GK / OT];
  auto fetch = [&](int k0) {   // A's chunk: lane = node, a warp's rows 32 consecutive nodes
#pragma unroll
    for (int j = 0; j < GMAX * GK / OT; ++j) {
      const int e = (tid >> 5) + (OT / 32) * j, k = k0 + (tid & 31);
      pre[j] = e < TE && t0 + e < ne && k < K ? Ab[(int64_t)e * U3 + k] : df{0.f, 0.f};
    }
  };
  auto store = [&](int c) {
#pragma unroll
    for (int j = 0; j < GMAX * GK / OT; ++j) As[c & 1][tid & 31][(tid >> 5) + (OT / 32) * j] = pre[j];
  };
  auto copyH = [&](int c) {   // eight bytes at a time: a block's table starts at any entry
    const int k0 = c * GK, len = min(GK, K - k0) * M;
    const unsigned dst = (unsigned)__cvta_generic_to_shared(&Hs[c & 1][0]);
    for (int i = tid; i < len; i += OT)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 8 * i), "l"(Hb + (int64_t)k0 * M + i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int nc = (K + GK - 1) / GK;
  tf tot[GE] = {};
  fetch(0);
  copyH(0);
  store(0);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int c = 0; c < nc; ++c) {
    const int nk = min(GK, K - c * GK);
    if (c + 1 < nc) {
      fetch((c + 1) * GK);
      copyH(c + 1);
    }
    if (on) {
      df acc[GE] = {};
#pragma unroll 2
      for (int k = sl; k < nk; k += NS) {
        const df h = Hs[c & 1][k * M + m];
        const float4* ap = reinterpret_cast<const float4*>(&As[c & 1][k][GE * g]);
#pragma unroll
        for (int j = 0; j < GE / 2; ++j) {
          const float4 v = ap[j];
          df_fma(acc[2 * j], df{v.x, v.y}, h);
          df_fma(acc[2 * j + 1], df{v.z, v.w}, h);
        }
      }
#pragma unroll
      for (int j = 0; j < GE; ++j) tf_add(tot[j], acc[j]);
    }
    if (c + 1 < nc) store(c + 1);   // the other buffer: last read before the previous barrier
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  if (NS > 1) {
    // slices 1 .. NS - 1 through shared memory, four elements at a time
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      __syncthreads();
      if (on && sl > 0)
#pragma unroll
        for (int j = 0; j < GE / 2; ++j) red[tid * (GE / 2) + j] = df_value(tot[h * (GE / 2) + j]);
      __syncthreads();
      if (sl == 0)
#pragma unroll
        for (int j = 0; j < GE / 2; ++j) {
          const int e = t0 + GE * g + h * (GE / 2) + j;
          double s = df_value(tot[h * (GE / 2) + j]);
          for (int q = 1; q < NS; ++q) s += red[(q * per + r) * (GE / 2) + j];
          if (e < ne) S[(e0 + e) * P3 + pb.moff[b] + m] = s;
        }
    }
  } else if (on) {
#pragma unroll
    for (int j = 0; j < GE; ++j) {
      const int e = t0 + GE * g + j;
      if (e < ne) S[(e0 + e) * P3 + pb.moff[b] + m] = df_value(tot[j]);
    }
  }
}

// Phi at each charge, one warp per charge: phi contracted with the order-p
// shape functions at the charge less the even and odd parts of S contracted
// with theirs (element units, FP64; inv_scale undoes the amplitudes' scale),
// plus the singular part already in phi_s.  4000 charges, q = 2: 108 -> 22 us
// against one thread per charge.
template <class V4>
__global__ void __launch_bounds__(OT) k_oq_eval(int64_t N, int n, OQParams prm, ParityBlocks pb, double inv_h,
                                                double inv_scale, const int* __restrict__ perm,
                                                const int* __restrict__ ecoord, const V4* __restrict__ part,
                                                const double* __restrict__ phi, const double* __restrict__ S,
                                                double* __restrict__ phi_s, double* __restrict__ phi_out) {
  __shared__ double lw[OT / 32][3][8], pw[OT / 32][3][8];   // shape functions, their even then odd parts
  __shared__ unsigned short dec[7 * 7 * 7];                 // a part's indices along the axes
  const int p = prm.p, P1 = p + 1, P3 = P1 * P1 * P1, Np = p * n, me = part_len(P1, 0);
  for (int b = 0; b < 8; ++b) {
    const int m0 = part_len(P1, b & 1), m1 = part_len(P1, (b >> 1) & 1);
    for (int i = threadIdx.x; i < pb.M[b]; i += OT) {
      const int x = i % m0 + (b & 1 ? me : 0), y = (i / m0) % m1 + (b & 2 ? me : 0), z = i / (m0 * m1) + (b & 4 ? me : 0);
      dec[pb.moff[b] + i] = (unsigned short)(x | y << 4 | z << 8);
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = blockIdx.x * (int64_t)(OT / 32) + warp;
  if (t >= N) return;
  const int ec = ecoord[t];
  const int ex = ec & 1023, ey = (ec >> 10) & 1023, ez = ec >> 20;
  const int64_t e = ex + (int64_t)n * (ey + (int64_t)n * ez);
  const V4 pt = part[t];
  if (lane < 3 * P1) {   // equispaced order-p Lagrange values, one per lane
    const int a = lane / P1, k = lane - a * P1;
    const double x = (a == 0 ? (double)pt.x : (a == 1 ? (double)pt.y : (double)pt.z)) * p;
    double v = prm.lden[k];
    for (int j = 0; j <= p; ++j)
      if (j != k) v *= x - j;
    lw[warp][a][k] = v;
  }
  __syncwarp();
  if (lane < 3 * P1) {
    const int a = lane / P1, k = lane - a * P1;
    const double* l = lw[warp][a];
    pw[warp][a][k] = k >= me ? l[k - me] - l[p - (k - me)] : (2 * k == p ? l[k] : l[k] + l[p - k]);
  }
  __syncwarp();
  double acc = 0.0, scr = 0.0;
  for (int r = lane; r < P1 * P1; r += 32) {
    const int my = r % P1, mz = r / P1;
    int gy = p * ey + my, gz = p * ez + mz;
    gy -= gy >= Np ? Np : 0;
    gz -= gz >= Np ? Np : 0;
    const double* row = phi + (int64_t)Np * (gy + (int64_t)Np * gz);
    double s = 0.0;
    for (int mx = 0; mx <= p; ++mx) {
      const int gx = p * ex + mx;
      s = fma(row[gx >= Np ? gx - Np : gx], lw[warp][0][mx], s);
    }
    acc = fma(s, lw[warp][1][my] * lw[warp][2][mz], acc);
  }
  for (int i = lane; i < P3; i += 32) {
    const int d = dec[i];
    scr = fma(S[e * P3 + i], pw[warp][0][d & 15] * pw[warp][1][(d >> 4) & 15] * pw[warp][2][d >> 8], scr);
  }
  acc -= scr * inv_scale;
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    const double val = acc * inv_h + phi_s[t];
    phi_s[t] = val;
    if (phi_out) phi_out[perm[t]] = val;
  }
}

// ---------------------------------------------------------------- host side
// o->red: partials of the sums from OQ_PART on (one per block), before them the
// sums' results: the refinement's state, then the norms of the right-hand side and of each sweep's residual
// (the sweeps past OQ_NORMS share the last)
constexpr int OQ_SUM = 0, OQ_STATE = 2, OQ_NORM = 4, OQ_PART = 36, OQ_NORMS = OQ_PART - OQ_NORM - 1;
inline int sum_blocks(int64_t len) { return (int)std::min<int64_t>(1024, std::max<int64_t>(1, len / (OT * 4))); }

void oq_sum(OrderQ* o, int64_t len, int weighted, const double* v, cudaStream_t s) {
  FEP3M_CL k_oq_sum<<<sum_blocks(len), OT, 0, s>>>(len, o->Np, o->prm, weighted, v, o->red + OQ_PART, o->counter,
                                                   o->red + OQ_SUM);
}

// K phi = pb (pb neutral, with its norm and scale: oq_project), int phi = 0:
// iterative refinement around the FP32 fast-diagonalisation solve.  The norms
// stay on the device and are read once after as many sweeps as the last solve
// took (and after each further one); sweeps past the first that reached the
// tolerance change nothing (RefineState)
cudaError_t oq_solve(fep3m_ctx* ctx, OrderQ* o, int max_sweeps) {
  const int n = ctx->n, Np = o->Np;
  const int64_t len = (int64_t)Np * Np * Np;
  cudaStream_t s = ctx->stream;
  RefineState* st = (RefineState*)(o->red + OQ_STATE);
  double *part = o->red + OQ_PART, *norm = o->red + OQ_NORM;
  o->sweeps = 0;
  o->relres = 0.0;
  FEP3M_CL k_oq_round<<<gsz(len), OT, 0, s>>>(len, o->pb, st, o->r32);
  const int read = std::max(1, std::min(o->plan, std::min(max_sweeps, OQ_NORMS)));
  for (int k = 0; k < max_sweeps; ++k) {
    const int at = std::min(k, OQ_NORMS - 1);
    cudaError_t e = fdm_apply(o->fdm, o->r32, o->x32, o->w1, o->w2, s);
    if (e != cudaSuccess) return e;
    FEP3M_CL k_oq_add<<<gsz(len), OT, 0, s>>>(len, o->x32, st, o->phi, k == 0);
    double *a = o->t[0], *b = o->t[1], *c = o->t[2], *f = o->t[3];
    FEP3M_CL k_oq_band<2><<<gsz(len), OT, 0, s>>>(Np, o->prm, o->phi, nullptr, a, b, nullptr, nullptr, nullptr,
                                                  nullptr, nullptr, nullptr);
    FEP3M_CL k_oq_band<1><<<gsz(len), OT, 0, s>>>(Np, o->prm, a, b, c, f, nullptr, nullptr, nullptr, nullptr, nullptr,
                                                  nullptr);
    FEP3M_CL k_oq_band<0><<<gsz(len), OT, 0, s>>>(Np, o->prm, c, f, nullptr, nullptr, o->pb, st, o->r32, part,
                                                  o->counter, norm + 1 + at);
    if (k + 1 < read) continue;
    cudaMemcpyAsync(o->host_red, o->red + OQ_STATE, (at + 4) * sizeof(double), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    const RefineState& hs = *(const RefineState*)o->host_red;
    const double nb = std::sqrt(o->host_red[2]), *nr = o->host_red + 3;
    if (!(nb > 0.0)) {
      cudaMemsetAsync(o->phi, 0, len * sizeof(double), s);
      return cudaGetLastError();
    }
    int j = 0;   // the first sweep that reached the tolerance (as the device decided), or the last one
    while (j < at && !(nr[j] <= hs.limit)) ++j;
    o->plan = j + 1;
    o->sweeps = j == at ? k + 1 : j + 1;
    o->relres = std::sqrt(nr[j]) / (hs.scale * nb);
    if (nr[j] <= hs.limit) break;
  }
  // int phi = 0: remove the node-integral weighted mean the FP32 corrections leave
  oq_sum(o, len, 1, o->phi, s);
  FEP3M_CL k_oq_mean<<<gsz(len), OT, 0, s>>>(len, o->red + OQ_SUM, 1.0 / ((double)n * n * n), o->phi);
  return cudaGetLastError();
}

size_t oq_amps_smem(int U) { return (size_t)U * U * part_len(U, 0) * sizeof(df); }

// the table of the eight parity blocks from the node-regrouped one: block b's
// K x M entries, the mean over the mirror images (which agree to rounding)
// with the parities' signs
std::vector<df> oq_parity_table(const ParityBlocks& pb, const std::vector<double>& H) {
  const int U = pb.U, P1 = pb.P1, P3 = pb.moff[8];
  std::vector<df> out;
  out.reserve((size_t)U * U * U * P3 / 7);
  for (int b = 0; b < 8; ++b) {
    const int odd[3] = {b & 1, (b >> 1) & 1, b >> 2};
    const int k0 = part_len(U, odd[0]), k1 = part_len(U, odd[1]), m0 = part_len(P1, odd[0]), m1 = part_len(P1, odd[1]);
    for (int k = 0; k < pb.K[b]; ++k)
      for (int m = 0; m < pb.M[b]; ++m) {
        const int kk[3] = {k % k0, (k / k0) % k1, k / (k0 * k1)}, mm[3] = {m % m0, (m / m0) % m1, m / (m0 * m1)};
        double v = 0.0;
        for (int f = 0; f < 64; ++f) {   // bit a: mirror node o along axis a; bit 3 + a: mirror node m
          int64_t o = 0, r = 0;
          int sign = 1;
          for (int a = 2; a >= 0; --a) {
            const int fo = (f >> a) & 1, fm = (f >> (3 + a)) & 1;
            o = o * U + (fo ? U - 1 - kk[a] : kk[a]);
            r = r * P1 + (fm ? P1 - 1 - mm[a] : mm[a]);
            if (odd[a] && fo != fm) sign = -sign;
          }
          v += sign * H[(size_t)o * P3 + r];
        }
        out.push_back(df_split(v / 64.0));
      }
  }
  return out;
}

void oq_params(const OrderQHost& h, OQParams& prm) {
  std::memset(&prm, 0, sizeof(prm));
  const int p = h.p, q = h.q, P1 = p + 1;
  prm.q = q;
  prm.p = p;
  for (size_t i = 0; i < h.W.size(); ++i) prm.W[i] = h.W[i];
  for (size_t i = 0; i < h.Mpq.size(); ++i) prm.Mpq[i] = h.Mpq[i];
  // global periodic rows: node type t = 0 (a vertex: local p of the element
  // before, local 0 of its own) or t (local t of its element)
  for (int t = 0; t < p; ++t) {
    auto add = [&](int local, int shift) {   // element whose local 0 sits at node g - shift
      for (int j = 0; j <= p; ++j) {
        const int o = j - shift + p;
        prm.bM[t][o] += h.Me[local * P1 + j];
        prm.bK[t][o] += h.Ke[local * P1 + j];
      }
    };
    if (t == 0) {
      add(p, p);
      add(0, 0);
    } else {
      add(t, t);
    }
    double wi = 0.0;
    const int li = t == 0 ? 0 : t;
    for (int j = 0; j <= p; ++j) wi += h.Me[li * P1 + j];   // int of the shape function (they sum to one)
    prm.wn[t] = t == 0 ? 2.0 * wi : wi;
  }
  for (int k = 0; k <= p; ++k) {
    double d = 1.0;
    for (int j = 0; j <= p; ++j)
      if (j != k) d *= k - j;
    prm.lden[k] = 1.0 / d;
  }
}

}  // namespace

int orderq_create(fep3m_ctx* c) {
  const int q = c->cfg.q, n = c->n;
  OrderQ* o = new (std::nothrow) OrderQ();
  if (!o) return FEP3M_ENOMEM;
  c->oq = o;
  const int pad = c->cfg.table_pad > 0 ? c->cfg.table_pad : 2;
  OrderQHost h;
  o->one_element = (c->cfg.flags & FEP3M_ONE_ELEMENT) != 0;
  if (!orderq_host(q, n, c->n_sr, pad, o->one_element, h)) return FEP3M_EINVAL;
  oq_params(h, o->prm);
  o->q = q;
  o->p = q + 2;
  o->Nq = q * n;
  o->Np = o->p * n;
  o->U = (2 * c->n_sr + 1) * q + 1;
  const int64_t ne = (int64_t)n * n * n, nq3 = (int64_t)o->Nq * o->Nq * o->Nq, np3 = (int64_t)o->Np * o->Np * o->Np;
  const int Q1 = q + 1, P1 = o->p + 1;
  cudaError_t e = cudaSuccess;
  auto al = [&](void** ptr, size_t bytes) {
    if (e == cudaSuccess) e = cudaMalloc(ptr, bytes);
  };
  al((void**)&o->C, ne * Q1 * Q1 * Q1 * sizeof(double));
  al((void**)&o->r, nq3 * sizeof(double));
  al((void**)&o->b, np3 * sizeof(double));
  al((void**)&o->pb, np3 * sizeof(double));
  al((void**)&o->phi, np3 * sizeof(double));
  for (int k = 0; k < 4; ++k) al((void**)&o->t[k], np3 * sizeof(double));
  al((void**)&o->r32, np3 * sizeof(float));
  al((void**)&o->x32, np3 * sizeof(float));
  al((void**)&o->w1, np3 * sizeof(float));
  al((void**)&o->w2, np3 * sizeof(float));
  al((void**)&o->S, ne * P1 * P1 * P1 * sizeof(double));
  const ParityBlocks pb = parity_blocks(o->U, P1);
  const std::vector<df> tab = oq_parity_table(pb, h.H);
  al((void**)&o->H, tab.size() * sizeof(df));
  al((void**)&o->Cp, ne * Q1 * Q1 * Q1 * sizeof(df));
  al((void**)&o->rp, nq3 * sizeof(df));
  // elements per piece of the screen contraction: amplitudes of about 96 MB, in the L2 cache
  // between the two launches (at least a tile)
  o->piece = (int)std::min<int64_t>(ne, std::max<int64_t>(GMAX, ((int64_t)96 << 20) / ((int64_t)pb.koff[8] * sizeof(df))));
  al((void**)&o->amps, (size_t)o->piece * pb.koff[8] * sizeof(df));
  al((void**)&o->red, (OQ_PART + std::max<int64_t>(1024, gsz(np3))) * sizeof(double));
  al((void**)&o->counter, sizeof(unsigned int));
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FEP3M_ENOMEM : FEP3M_ECUDA;
  if (cudaMallocHost(&o->host_red, (OQ_NORMS + 3) * sizeof(double)) != cudaSuccess) return FEP3M_ENOMEM;
  cudaMemcpy(o->H, tab.data(), tab.size() * sizeof(df), cudaMemcpyHostToDevice);
  cudaMemset(o->counter, 0, sizeof(unsigned int));
  e = fdm_setup(o->fdm, o->Np, h.lam, h.V, 1, !(c->cfg.flags & FEP3M_CUDA_CORES));
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FEP3M_ENOMEM : FEP3M_ECUDA;
  if (smem_limit((const void*)k_oq_amps, oq_amps_smem(o->U)) != cudaSuccess ||
      smem_limit((const void*)k_oq_gemm, GSMEM) != cudaSuccess)
    return FEP3M_ECUDA;
  return FEP3M_OK;
}

void orderq_destroy(fep3m_ctx* c) {
  OrderQ* o = c->oq;
  if (!o) return;
  void* p[] = {o->C, o->r, o->b, o->pb, o->phi, o->t[0], o->t[1], o->t[2], o->t[3], o->r32, o->x32,
               o->w1, o->w2, o->S, o->H, o->red, o->Cp, o->rp, o->amps, o->counter};
  for (void* x : p)
    if (x) cudaFree(x);
  if (o->host_red) cudaFreeHost(o->host_red);
  fdm_free(o->fdm);
  delete o;
  c->oq = nullptr;
}

static double oq_rtol(const fep3m_ctx* c) {
  return c->cfg.mg_rtol > 0 ? c->cfg.mg_rtol : (c->precision == FEP3M_FP64 ? 1e-13 : 1e-10);
}

// the load vector less its background, from b (device), with its norm and scale
static void oq_project(fep3m_ctx* c, OrderQ* o, cudaStream_t s) {
  const int n = c->n, Np = o->Np;
  const int64_t len = (int64_t)Np * Np * Np;
  oq_sum(o, len, 0, o->b, s);
  FEP3M_CL k_oq_project<<<sum_blocks(len), OT, 0, s>>>(Np, o->prm, o->red + OQ_SUM, 1.0 / ((double)n * n * n), o->b,
                                                       o->pb, o->red + OQ_PART, o->counter, o->red + OQ_NORM,
                                                       oq_rtol(c), (RefineState*)(o->red + OQ_STATE));
}

int orderq_compute(fep3m_ctx* c, double* phi_dev, double* U_dev) {
  OrderQ* o = c->oq;
  const int n = c->n, q = o->q, Q1 = q + 1, P1 = o->p + 1;
  const int64_t ne = (int64_t)n * n * n, N = c->N;
  const int64_t nq3 = (int64_t)o->Nq * o->Nq * o->Nq, np3 = (int64_t)o->Np * o->Np * o->Np;
  cudaStream_t s = c->stream;
  const int64_t nc = ne * Q1 * Q1 * Q1;
  if (c->precision == FEP3M_MIXED)
    FEP3M_CL k_oq_coeff<float4><<<gsz(nc), OT, 0, s>>>(ne, o->prm, c->start, c->count, (const float4*)c->part,
                                                        c->q_scale, o->C, (df*)o->Cp);
  else
    FEP3M_CL k_oq_coeff<vec4<double>::type><<<gsz(nc), OT, 0, s>>>(ne, o->prm, c->start, c->count,
                                                                     (const vec4<double>::type*)c->part, c->q_scale,
                                                                     o->C, (df*)o->Cp);
  FEP3M_CL k_oq_density<<<gsz(nq3), OT, 0, s>>>(n, q, o->C, c->q_scale, o->r, (df*)o->rp);
  {
    const int Np = o->Np, Nq = o->Nq;
    const int64_t n1 = (int64_t)Np * Nq * Nq, n2 = (int64_t)Np * Np * Nq;
    FEP3M_CL k_oq_load<<<gsz(n1), OT, 0, s>>>(n, 0, Np, Nq, Nq, o->prm, o->r, o->t[0], 1.0);
    FEP3M_CL k_oq_load<<<gsz(n2), OT, 0, s>>>(n, 1, Np, Np, Nq, o->prm, o->t[0], o->t[1], 1.0);
    FEP3M_CL k_oq_load<<<gsz(np3), OT, 0, s>>>(n, 2, Np, Np, Np, o->prm, o->t[1], o->b, 4.0 * M_PI);
  }
  oq_project(c, o, s);
  cudaError_t e = oq_solve(c, o, c->cfg.mg_max_cycles > 0 ? c->cfg.mg_max_cycles : 10);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FEP3M_ENOMEM : FEP3M_ECUDA;
  const ParityBlocks pb = parity_blocks(o->U, P1);
  for (int64_t e0 = 0; e0 < ne; e0 += o->piece) {
    const int m = (int)std::min<int64_t>(o->piece, ne - e0);
    FEP3M_CL k_oq_amps<<<dim3((unsigned)m, 2), OT, oq_amps_smem(o->U), s>>>(n, c->n_sr, q, pb, e0, c->count,
                                                                            (const df*)o->Cp, (const df*)o->rp,
                                                                            (df*)o->amps);
    // tiles of the block with most nodes (GE elements at least)
    int G = GMAX / GE;
    while (G > 1 && G * pb.M[0] > OT) G >>= 1;
    FEP3M_CL k_oq_gemm<<<dim3((unsigned)((m + GE * G - 1) / (GE * G)), 8), OT, GSMEM, s>>>(pb, e0, m, (const df*)o->amps,
                                                                                       (const df*)o->H, o->S);
  }
  if ((e = singular_sums(c, s)) != cudaSuccess) return FEP3M_ECUDA;
  if (c->precision == FEP3M_MIXED)
    FEP3M_CL k_oq_eval<float4><<<gsz(N, OT / 32), OT, 0, s>>>(N, n, o->prm, pb, c->inv_h, 1.0 / c->q_scale, c->perm,
                                                               c->ecoord,
                                                      (const float4*)c->part, o->phi, o->S, c->phi_s, phi_dev);
  else
    FEP3M_CL k_oq_eval<vec4<double>::type><<<gsz(N, OT / 32), OT, 0, s>>>(N, n, o->prm, pb, c->inv_h,
                                                                  1.0 / c->q_scale, c->perm, c->ecoord,
                                                                  (const vec4<double>::type*)c->part, o->phi, o->S,
                                                                  c->phi_s, phi_dev);
  if (U_dev && (e = energy(c, U_dev)) != cudaSuccess) return FEP3M_ECUDA;
  e = cudaGetLastError();
  if (e != cudaSuccess) return FEP3M_ECUDA;
  return o->relres <= 10 * oq_rtol(c) ? FEP3M_OK : FEP3M_ENOCONV;
}

int orderq_solve(fep3m_ctx* c, const double* b_dev, double* phi_dev) {
  OrderQ* o = c->oq;
  const int64_t np3 = (int64_t)o->Np * o->Np * o->Np;
  cudaStream_t s = c->stream;
  cudaMemcpyAsync(o->b, b_dev, np3 * sizeof(double), cudaMemcpyDeviceToDevice, s);
  oq_project(c, o, s);
  cudaError_t e = oq_solve(c, o, c->cfg.mg_max_cycles > 0 ? c->cfg.mg_max_cycles : 10);
  if (e != cudaSuccess) return FEP3M_ECUDA;
  cudaMemcpyAsync(phi_dev, o->phi, np3 * sizeof(double), cudaMemcpyDeviceToDevice, s);
  return o->relres <= 10 * oq_rtol(c) ? FEP3M_OK : FEP3M_ENOCONV;
}

}  // namespace fep3m
