// The box [0, L]^3 with Dirichlet data Phi = g or Neumann data dPhi/dn = g on
// its boundary (Sec. "Alternate boundary conditions"), screens of order q = 1
// on the order-3 mesh.
//
// The paper carries the periodic method over to a box by one change: the mesh
// problem's boundary data are the given data less what the short-range
// potential already carries there (Eq. bcadjust), Phi^sm = g - Phi^sr, so that
// Phi = Phi^sm + Phi^sr = g on the boundary (Algorithm 1 marks the step for
// the surface elements); for Neumann data the same holds for the normal
// derivatives, and in the Galerkin form the adjusted flux is a boundary load
// s_m = int (g - dPhi^sr/dn) v_m dS.  Here:
//   binning, screens, short-range sums, evaluation: the periodic path's
//     kernels, on a periodic grid of nb + n_sr elements per axis whose first
//     nb hold the box (the context's n).  The n_sr empty layers make the
//     block around every box element reach box elements and empty ones only,
//     and no image of a charge: the block cut off at the box faces;
//   load vector: b = 4 pi (Mpq (x) Mpq (x) Mpq) r with the open (box-only)
//     mixed mass on the (3 nb + 1)^3 box nodes: the parts of boundary
//     charges' screens outside the box are not loads of the box problem;
//   boundary values: h (g - Phi^sr) at each boundary node, from the singular
//     sum over the node's block and the screen field at the node (the
//     vertex-regrouped contraction of the pair kernel for the node's element),
//     in double-float arithmetic, one CTA per boundary element;
//   Neumann load: s at the face nodes, per face element by a tensor
//     Gauss-Legendre rule (BOX_NGL points per axis) of g less the normal
//     derivative of Phi^sr (singular sum over the point's block and the
//     screen field's gradient through the order-3 basis), one CTA per face
//     element, gathered per node in a fixed order;
//   mesh solve: K phi = b at the (3 nb - 1)^3 interior nodes with the
//     boundary values fixed (Dirichlet), or K phi = b + s less its component
//     along the node integrals (the constant null space) on all (3 nb + 1)^3
//     nodes with int phi = 0 (Neumann), by iterative refinement: the residual
//     in FP64 or, mixed, double-float arithmetic (the periodic solver's fused
//     apply on the open node grid), the
//     correction by the FP32 fast-diagonalisation solve of the solved nodes
//     with the box eigenbasis (Dirichlet: no null mode; the periodic solve's
//     transform passes, on the tensor cores unless FEP3M_CUDA_CORES);
//   evaluation: Phi_i = Phi^sm(x_i) + Phi^sr_i by the periodic evaluation
//     kernel on the box's node grid, and U = 1/2 sum_i Q_i Phi_i (FP64).
// Mesh values are in element units (h Phi), as on the periodic path.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "df.cuh"
#include "gridsum.cuh"

namespace fep3m {

void box_eigen(int p, int n, bool dirichlet, std::vector<double>& lam, std::vector<double>& V);

namespace {

constexpr int BT = 256;
static_assert(BOX_NGL == FEP3M_NEUMANN_NGL, "the face rule of the ABI");

inline unsigned gsz(int64_t n, int t = BT) { return (unsigned)((n + t - 1) / t); }

__device__ __forceinline__ int wrapb(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// the vertices (and weights) that order-3 node g of an axis takes on the
// open box mesh: the box elements containing g (node 0: element 0 only;
// node 3 nb: element nb - 1 only), each with its two vertices.  FP32: the
// weights times 120, exact integers (as the periodic path's load vector; the
// caller's scale divides by 120^3)
template <class T>
__device__ __forceinline__ int box_mpq_row(int g, int nb, const BoxBand& bd, int vtx[4], T wgt[4]) {
  const double s = sizeof(T) == 4 ? 120.0 : 1.0;
  const int e = g / 3, t = g - 3 * e;
  int k = 0;
  auto add = [&](int el, int local) {
    vtx[k] = el;
    wgt[k++] = sizeof(T) == 4 ? (T)rint(s * bd.Mpq[local][0]) : (T)bd.Mpq[local][0];
    vtx[k] = el + 1;
    wgt[k++] = sizeof(T) == 4 ? (T)rint(s * bd.Mpq[local][1]) : (T)bd.Mpq[local][1];
  };
  if (t != 0) {
    add(e, t);
  } else {
    if (e > 0) add(e - 1, 3);
    if (e < nb) add(e, 0);
  }
  return k;
}

// One axis of b = 4 pi (Mpq (x) Mpq (x) Mpq) r on the box: out (extents d[3])
// at order-3 node idx[axis] sums the input's vertices along the axis; the
// input is read with strides si[3] (the first pass reads the vertex density
// of the padded periodic grid, whose first nb + 1 vertices per axis are the
// box's)
template <class Tin, class Tout>
__global__ void k_box_load_axis(int nb, int axis, int d0, int d1, int d2, int64_t si0, int64_t si1, int64_t si2,
                                BoxBand bd, const Tin* __restrict__ in, Tout* __restrict__ out, double scale) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= (int64_t)d0 * d1 * d2) return;
  int idx[3] = {(int)(g % d0), (int)((g / d0) % d1), (int)(g / ((int64_t)d0 * d1))};
  const int64_t si[3] = {si0, si1, si2};
  int vtx[4];
  Tin w[4];
  const int k = box_mpq_row<Tin>(idx[axis], nb, bd, vtx, w);
  idx[axis] = 0;
  const int64_t base = idx[0] * si[0] + idx[1] * si[1] + idx[2] * si[2];
  Tin acc = Tin(0);
  for (int j = 0; j < k; ++j) acc += w[j] * in[base + vtx[j] * si[axis]];
  out[g] = (Tout)(scale * (double)acc);
}

// Short-range part at the boundary.  Both kernels below take one CTA of BT
// threads per boundary (or face) element and work on its block, the elements
// within n_sr of it that lie in the box: the block's charges are staged in
// shared memory a chunk at a time (a row of the block along x is one
// contiguous run of sorted charges), and the sums run in double-float
// arithmetic on the FP32 pipes (df.cuh) with FP64 totals.  The charges are
// scaled by a power of two near the inverse of their mean magnitude, so that
// the pairs' low words stay normal FP32 numbers whatever the charges' unit.
constexpr int BROWS = 81;   // rows (y, z) of a block, n_sr <= 4

// a thread's running sum: a pair, on the FP64 path three floats
template <class T> struct Sum {
  typedef typename std::conditional<sizeof(T) == 4, df, tf>::type type;
};

__device__ __forceinline__ void negate(df& s) { s = {-s.h, -s.l}; }
__device__ __forceinline__ void negate(tf& s) { s = {-s.h, -s.m, -s.l}; }
// s += a, running sums of two threads
__device__ __forceinline__ void add_part(df& s, df a) { s = df_add(s, a); }
__device__ __forceinline__ void add_part(tf& s, tf a) { tf_add(s, a); }

// the runs of the block's rows: j0[r] the first sorted charge of row r, pre[r]
// the charges of the rows before it; returns their number.  By the CTA.
__device__ int block_rows(int n, int nb, int n_sr, const int E[3], const int* __restrict__ start, int* j0, int* pre) {
  const int nbk = 2 * n_sr + 1, nrow = nbk * nbk;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const int x0 = max(E[0] - n_sr, 0), x1 = min(E[0] + n_sr, nb - 1);
    int carry = 0;
    for (int base = 0; base < nrow; base += 32) {
      const int r = base + lane;
      int first = 0, cnt = 0;
      if (r < nrow) {
        const int y = E[1] + r % nbk - n_sr, z = E[2] + r / nbk - n_sr;
        if (y >= 0 && z >= 0 && y < nb && z < nb) {
          // x1 + 1 <= nb is an element of the padded row: its start ends the run
          const int64_t row = (int64_t)n * (y + (int64_t)n * z);
          first = start[row + x0];
          cnt = start[row + x1 + 1] - first;
        }
      }
      int x = cnt;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += v;
      }
      if (r < nrow) {
        j0[r] = first;
        pre[r] = carry + x - cnt;
      }
      carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) pre[nrow] = carry;
  }
  __syncthreads();
  return pre[nrow];
}

// sorted index of the block's charge s (0 <= s < pre[nrow])
__device__ __forceinline__ int block_charge(int s, int nrow, const int* j0, const int* pre) {
  int lo = 0, hi = nrow;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pre[mid] <= s) lo = mid;
    else hi = mid;
  }
  return j0[lo] + (s - pre[lo]);
}

// Vertex amplitudes of element E's block as pairs: A[o] = the corner terms
// C[v - k][k] at vertex v = E - o of the block's elements, times scale
template <class T>
__device__ void block_amplitudes(int n, int n_sr, const int E[3], T scale, const T* __restrict__ Cv, df* A) {
  const int keep = n_sr + 1, noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  for (int o = threadIdx.x; o < no3; o += BT) {
    const int ox = o % noff - keep, oy = (o / noff) % noff - keep, oz = o / (noff * noff) - keep;
    const int64_t v = wrapb(E[0] - ox, n) + (int64_t)n * (wrapb(E[1] - oy, n) + (int64_t)n * wrapb(E[2] - oz, n));
    // the corner's element v - k is in the block: |o + k| <= n_sr per axis
    const unsigned mx = ox == -keep ? 0xAAu : (ox == n_sr ? 0x55u : 0xFFu);
    const unsigned my = oy == -keep ? 0xCCu : (oy == n_sr ? 0x33u : 0xFFu);
    const unsigned mz = oz == -keep ? 0xF0u : (oz == n_sr ? 0x0Fu : 0xFFu);
    const unsigned mask = mx & my & mz;
    typedef typename vec4<T>::type V4;
    const V4 a = reinterpret_cast<const V4*>(Cv + 8 * v)[0], b = reinterpret_cast<const V4*>(Cv + 8 * v)[1];
    const T c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    if constexpr (sizeof(T) == 4) {
      df s = {0.f, 0.f};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const df t = df_two_sum(s.h, ((mask >> k) & 1u) ? c[k] * scale : 0.f);
        s = {t.h, s.l + t.l};
      }
      A[o] = s;
    } else {
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k) s += ((mask >> k) & 1u) ? c[k] : 0.0;
      A[o] = df_split(s * scale);
    }
  }
}

// Boundary values of the mesh problem (Eq. bcadjust), element units:
//   phi[node] = h g[node] - sum_{j in block} Q_j / |x_node - x_j| (element
//   units) + sum_o A_e(o) H(o, m),
// the last term the screen field of the block's charges at node m of the
// node's element e (Hdf the absolute vertex table [offset][node] as pairs).
// The element writes the boundary nodes it owns (per axis local nodes 0 .. 2,
// and 3 on the last element: the binning rule min(i / 3, nb - 1)): 9 on a
// face element, up to 37 at a corner.  Thread (k, part) sums node k over the
// charges and the offsets part, part + nparts, ...: with M nodes, nparts =
// BT / M, so nearly all threads work whatever M is.  A charge at a boundary
// node makes that node's value infinite.  Bound by FP32 issue (about 80
// operations per node and charge, 11 per node and offset); rock salt in a
// 32^3 box: 1722 -> 132 us against FP64 sums with one lane per block element.
constexpr int BCH = 256;    // charges staged at once
struct BoxSrc {             // a staged charge at its largest (FP64 positions)
  tf x[3];
  df q;
};
template <class T>
__global__ void __launch_bounds__(BT) k_box_boundary(int n, int nb, int n_sr, double h, double scale,
                                                     double inv_scale, const int* __restrict__ bel, const int* __restrict__ start,
                                                     const int* __restrict__ ecoord,
                                                     const typename vec4<T>::type* __restrict__ part,
                                                     const T* __restrict__ Cv, const float2* __restrict__ Hdf,
                                                     const double* __restrict__ g, double* __restrict__ phi) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff, nrow = (2 * n_sr + 1) * (2 * n_sr + 1);
  df* A = reinterpret_cast<df*>(smem);                                  // no3
  // a charge's coordinates from E's corner: an FP32 one plus a whole number is a
  // pair exactly, an FP64 one takes three floats
  typedef typename std::conditional<sizeof(T) == 4, df, tf>::type X1;
  struct Src {
    X1 x[3];
    df q;
  };
  struct Part {
    typename Sum<T>::type s;
    double far;
  };
  Src* ch = reinterpret_cast<Src*>(A + no3);                            // [BCH]
  Part* red = reinterpret_cast<Part*>(smem + no3 * sizeof(df) + BCH * sizeof(BoxSrc));   // BT
  __shared__ int j0[BROWS], pre[BROWS + 1], list[64], nlist;
  const int e = bel[blockIdx.x];
  const int E[3] = {e % n, (e / n) % n, e / (n * n)};
  const int tid = threadIdx.x, Nn = 3 * nb + 1;
  if (tid < 32) {   // the boundary nodes E owns, in order
    int base = 0;
    for (int m = tid; m < 64; m += 32) {
      const int mm[3] = {m & 3, (m >> 2) & 3, m >> 4};
      bool own = true, bnd = false;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        own = own && (mm[d] < 3 || E[d] == nb - 1);
        const int gi = 3 * E[d] + mm[d];
        bnd = bnd || gi == 0 || gi == 3 * nb;
      }
      const unsigned b = __ballot_sync(0xffffffffu, own && bnd);
      if (own && bnd) list[base + __popc(b & ((1u << tid) - 1u))] = m;
      base += __popc(b);
    }
    if (tid == 0) nlist = base;
  }
  block_amplitudes<T>(n, n_sr, E, (T)scale, Cv, A);
  const int total = block_rows(n, nb, n_sr, E, start, j0, pre);   // ends with a barrier
  const int M = nlist, nparts = BT / M, k = tid % M, p = tid / M;
  const bool on = p < nparts;
  const int m = list[k], mm[3] = {m & 3, (m >> 2) & 3, m >> 4};
  X1 tn[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // (mm / 3 by selection: an FP64 division here costs as much as the sums)
    const int q = mm[a];
    constexpr float h1 = (float)(1.0 / 3.0), h2 = (float)(2.0 / 3.0);
    constexpr float m1 = (float)(1.0 / 3.0 - h1), m2 = (float)(2.0 / 3.0 - h2);
    constexpr float l1 = (float)(1.0 / 3.0 - h1 - m1), l2 = (float)(2.0 / 3.0 - h2 - m2);
    const float th = q == 0 ? 0.f : (q == 1 ? h1 : (q == 2 ? h2 : 1.f));
    const float tm = q == 1 ? m1 : (q == 2 ? m2 : 0.f);
    if constexpr (sizeof(T) == 4) tn[a] = df{-th, -tm};
    else tn[a] = tf{th, tm, q == 1 ? l1 : (q == 2 ? l2 : 0.f)};
  }
  auto diff = [&](const X1& x, int a) -> df {
    if constexpr (sizeof(T) == 4) return df_add(x, tn[a]);
    else return tf_diff(x, tn[a]);
  };
  typename Sum<T>::type acc = {};   // screen field
  double far = 0.0;      // terms outside the pairs' range
  if (on) {
#pragma unroll 4
    for (int o = p; o < no3; o += nparts) {
      const float2 hv = Hdf[(int64_t)o * 64 + m];
      df_fma(acc, A[o], df{hv.x, hv.y});
    }
  }
  typename Sum<T>::type sing = {};
  for (int c0 = 0; c0 < total; c0 += BCH) {
    const int nc = min(BCH, total - c0);
    if (c0) __syncthreads();
    if (tid < nc) {
      const int j = block_charge(c0 + tid, nrow, j0, pre);
      const typename vec4<T>::type pj = part[j];
      const int ec = ecoord[j];
      const int d[3] = {(ec & 1023) - E[0], ((ec >> 10) & 1023) - E[1], (ec >> 20) - E[2]};
      const T pp[3] = {pj.x, pj.y, pj.z};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if constexpr (sizeof(T) == 4) ch[tid].x[a] = df_two_sum((float)d[a], pp[a]);
        else ch[tid].x[a] = tf_split((double)d[a] + pp[a]);
      }
      if constexpr (sizeof(T) == 4) ch[tid].q = {pj.w * (float)scale, 0.f};
      else ch[tid].q = df_split(pj.w * scale);
    }
    __syncthreads();
    if (on) {
#pragma unroll 2
      for (int c = p; c < nc; c += nparts) {
        df r2 = df_sqr(diff(ch[c].x[0], 0));
        r2 = df_add(r2, df_sqr(diff(ch[c].x[1], 1)));
        r2 = df_add(r2, df_sqr(diff(ch[c].x[2], 2)));
        if (df_in_range(r2)) df_fma(sing, ch[c].q, df_rsqrt<sizeof(T) == 8>(r2));
        else far += df_value(ch[c].q) / sqrt(df_value(r2));
      }
    }
  }
  negate(sing);
  add_part(sing, acc);      // screen field less the singular sum
  red[tid] = {sing, far};   // threads off: zero
  __syncthreads();
  if (tid < M) {
    typename Sum<T>::type t = red[tid].s;
    double f = far;
    for (int q = 1; q < nparts; ++q) {
      add_part(t, red[q * M + tid].s);
      if (red[q * M + tid].far != 0.0) f += red[q * M + tid].far;   // also NaN
    }
    const double s = df_value(t) - f;
    const int gx = 3 * E[0] + mm[0], gy = 3 * E[1] + mm[1], gz = 3 * E[2] + mm[2];
    const int64_t node = gx + (int64_t)Nn * (gy + (int64_t)Nn * gz);
    phi[node] = h * g[node] + s * inv_scale;
  }
}

// Neumann face loads, element units (the mesh problem K phi = b + s):
//   s_m = int_face (g - dPhi^sr/dn) v_m dS
//       = sum_p w_p (h^2 g_p - D_p) l_i(t1_p) l_j(t2_p)
// over the BOX_NGL^2 Gauss-Legendre points p of a face element (weights w_p on
// the unit square), D_p the normal derivative of Phi^sr in element units:
// -sum_{j in block} Q_j (r . n) / |r|^3 (r the point less x_j) less the
// screen field's derivative there.  One CTA per face element fe = (face, e1,
// e2), face = 2 axis + side (side 1: the face at L, outward normal +axis), e1
// and e2 along the next two axes (e2 fastest); the point data g in the same
// order, points (i, j) with i along the first of those axes.  Writes the 16
// face-node sums (node i1 + 4 i2).
//
// On a face r . n is one number per charge and |r|^2 = (t_i - x1)^2 +
// ((t_j - x2)^2 + (r . n)^2) takes 8 + 8 values per charge over the 64
// points, so these are staged per charge and a (point, charge) pair costs
// one sum, the power -3/2 and one multiply-add: about 40 FP32 operations.
// The screen field's normal derivative needs the table contracted along the
// normal axis only once, on the host: Hface[face][offset][16 face nodes].
// Thread (point, group of four) walks every fourth charge.  Bound by FP32
// issue; rock salt in a 32^3 box (77 M pairs): 14603 -> 216 us against FP64
// terms with the 64 nodes' gradient at every point.
constexpr int FCH = 64;     // charges staged at once
template <class T>
__global__ void __launch_bounds__(BT) k_box_flux(int n, int nb, int n_sr, double h, double scale, double inv_scale, BoxQuad qd,
                                                 const int* __restrict__ start, const int* __restrict__ ecoord,
                                                 const typename vec4<T>::type* __restrict__ part,
                                                 const T* __restrict__ Cv, const float2* __restrict__ Hface,
                                                 const double* __restrict__ g, double* __restrict__ sface) {
  constexpr int NP = BOX_NGL * BOX_NGL, NG = BT / NP;
  static_assert(BOX_NGL == 8 && BT == 4 * FCH && NG == 4, "the thread mapping below");
  extern __shared__ __align__(16) unsigned char smem[];
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff, nrow = (2 * n_sr + 1) * (2 * n_sr + 1);
  df* A = reinterpret_cast<df*>(smem);   // no3
  __shared__ df sA[FCH][BOX_NGL + 1], sB[FCH][BOX_NGL + 1], sW[FCH];   // odd rows: no bank conflicts
  __shared__ double red[BT], G[16], fp[NP], half[32];
  __shared__ int j0[BROWS], pre[BROWS + 1];
  const int fe = blockIdx.x, face = fe / (nb * nb), e1 = (fe / nb) % nb, e2 = fe % nb;
  const int ax = face >> 1, side = face & 1, a1 = (ax + 1) % 3, a2 = (ax + 2) % 3;
  int E[3];
  E[0] = ax == 0 ? (side ? nb - 1 : 0) : (a1 == 0 ? e1 : e2);
  E[1] = ax == 1 ? (side ? nb - 1 : 0) : (a1 == 1 ? e1 : e2);
  E[2] = ax == 2 ? (side ? nb - 1 : 0) : (a1 == 2 ? e1 : e2);
  const int tid = threadIdx.x;
  const double sgn = side ? 1.0 : -1.0;   // outward normal along ax
  block_amplitudes<T>(n, n_sr, E, (T)scale, Cv, A);
  const int total = block_rows(n, nb, n_sr, E, start, j0, pre);   // ends with a barrier
  {
    // the screen field's slope along ax at the 16 face nodes, in 16 parts
    const int m = tid & 15, q = tid >> 4;
    const float2* Hf = Hface + (int64_t)face * no3 * 16;
    typename Sum<T>::type acc = {};
#pragma unroll 4
    for (int o = q; o < no3; o += BT / 16) {
      const float2 hv = Hf[o * 16 + m];
      df_fma(acc, A[o], df{hv.x, hv.y});
    }
    red[tid] = df_value(acc);
    __syncthreads();
    if (tid < 16) {
      double s = 0.0;
      for (int k = 0; k < BT / 16; ++k) s += red[16 * k + tid];
      G[tid] = s;
    }
  }
  const int p = tid & (NP - 1), pi = p >> 3, pj = p & 7, grp = tid / NP;
  typename Sum<T>::type acc = {};   // sum_j Q_j (r . n) / |r|^3, element units
  double far = 0.0;      // terms outside the pairs' range
  for (int c0 = 0; c0 < total; c0 += FCH) {
    const int nc = min(FCH, total - c0);
    __syncthreads();
    const int c = tid >> 2, sub = tid & 3;   // four threads per charge: two points of each axis
    if (c < nc) {
      const int j = block_charge(c0 + c, nrow, j0, pre);
      const typename vec4<T>::type q = part[j];
      const int ec = ecoord[j];
      const int d[3] = {(ec & 1023) - E[0], ((ec >> 10) & 1023) - E[1], (ec >> 20) - E[2]};
      const T x3[3] = {q.x, q.y, q.z};
      const int dn = ax == 0 ? d[0] : (ax == 1 ? d[1] : d[2]), d1 = a1 == 0 ? d[0] : (a1 == 1 ? d[1] : d[2]),
                d2 = a2 == 0 ? d[0] : (a2 == 1 ? d[1] : d[2]);
      const T xn = ax == 0 ? x3[0] : (ax == 1 ? x3[1] : x3[2]), x1 = a1 == 0 ? x3[0] : (a1 == 1 ? x3[1] : x3[2]),
              x2 = a2 == 0 ? x3[0] : (a2 == 1 ? x3[1] : x3[2]);
      if constexpr (sizeof(T) == 4) {
        // dn + xn etc. exactly as pairs; the point's coordinate less the charge's
        const df rn = df_two_sum((float)(side - dn), -xn), X1 = df_two_sum((float)(-d1), -x1),
                 X2 = df_two_sum((float)(-d2), -x2), rn2 = df_sqr(rn);
#pragma unroll
        for (int k = 2 * sub; k < 2 * sub + 2; ++k) {
          const df t = {qd.th[k], qd.tl[k]};
          sA[c][k] = df_sqr(df_add(t, X1));
          sB[c][k] = df_add(df_sqr(df_add(t, X2)), rn2);
        }
        if (sub == 0) {
          const float w = q.w * (float)scale, s = (float)sgn * w, ph = s * rn.h;
          sW[c] = {ph, fmaf(s, rn.l, fmaf(s, rn.h, -ph))};
        }
      } else {
        const double rn = side - (dn + xn), X1 = d1 + x1, X2 = d2 + x2;
#pragma unroll
        for (int k = 2 * sub; k < 2 * sub + 2; ++k) {
          const double u = qd.t[k] - X1, v = qd.t[k] - X2;
          sA[c][k] = df_split(u * u);
          sB[c][k] = df_split(fma(v, v, rn * rn));
        }
        if (sub == 0) sW[c] = df_split(q.w * scale * (sgn * rn));
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int k = grp; k < nc; k += NG) {
      const df a = sA[k][pi], b = sB[k][pj], s = df_two_sum(a.h, b.h);
      const df r2 = {s.h, s.l + (a.l + b.l)};
      if (df_in_range(r2)) {
        df_fma(acc, sW[k], df_rsqrt3<sizeof(T) == 8>(r2));
      } else {
        const double ir = 1.0 / sqrt(df_value(r2));
        far += df_value(sW[k]) * ir * ir * ir;
      }
    }
  }
  __syncthreads();
  red[tid] = df_value(acc) + far;
  __syncthreads();
  if (tid < NP) {
    double sg = 0.0, sd = 0.0;
#pragma unroll
    for (int k = 0; k < NG; ++k) sg += red[k * NP + p];
#pragma unroll
    for (int i2 = 0; i2 < 4; ++i2) {
      double row = 0.0;
#pragma unroll
      for (int i1 = 0; i1 < 4; ++i1) row = fma(G[i1 + 4 * i2], qd.l[pi][i1], row);
      sd = fma(row, qd.l[pj][i2], sd);
    }
    const double D = -(sg + sgn * sd) * inv_scale;
    fp[p] = qd.w[pi] * qd.w[pj] * (h * h * g[(int64_t)fe * NP + p] - D);
  }
  __syncthreads();
  if (tid < 32) {   // s_(i1, i2) = sum_i l_i1(t_i) sum_j l_i2(t_j) fp(i, j): first over i
    const int i1 = tid & 3, j = tid >> 2;
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < BOX_NGL; ++i) s = fma(fp[i * BOX_NGL + j], qd.l[i][i1], s);
    half[tid] = s;
    __syncwarp();
    if (tid < 16) {
      const int i2 = tid >> 2;
      s = 0.0;
#pragma unroll
      for (int k = 0; k < BOX_NGL; ++k) s = fma(half[i1 + 4 * k], qd.l[k][i2], s);
      sface[(int64_t)fe * 16 + tid] = s;
    }
  }
}

// rhs = b + s: every boundary node collects the loads of the face elements
// (of each face it lies on) that contain it, in a fixed order
__global__ void k_box_sgather(int nb, const double* __restrict__ b, const double* __restrict__ sface,
                              double* __restrict__ rhs) {
  const int Nn = 3 * nb + 1;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)Nn * Nn * Nn) return;
  const int c[3] = {(int)(i % Nn), (int)((i / Nn) % Nn), (int)(i / ((int64_t)Nn * Nn))};
  double s = 0.0;
  for (int ax = 0; ax < 3; ++ax)
    for (int side = 0; side < 2; ++side) {
      if (c[ax] != (side ? 3 * nb : 0)) continue;
      const int a1 = (ax + 1) % 3, a2 = (ax + 2) % 3, face = 2 * ax + side;
      for (int k1 = 0; k1 < 2; ++k1) {
        const int f1 = c[a1] / 3 - 1 + k1, i1 = c[a1] - 3 * f1;
        if (f1 < 0 || f1 >= nb || i1 > 3) continue;
        for (int k2 = 0; k2 < 2; ++k2) {
          const int f2 = c[a2] / 3 - 1 + k2, i2 = c[a2] - 3 * f2;
          if (f2 < 0 || f2 >= nb || i2 > 3) continue;
          s += sface[((int64_t)(face * nb + f1) * nb + f2) * 16 + i1 + 4 * i2];
        }
      }
    }
  rhs[i] = b[i] + s;
}

// phi = h g on the boundary nodes (no adjustment), 0 inside
__global__ void k_box_plain_bvals(int Nn, double h, const double* __restrict__ g, double* __restrict__ phi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)Nn * Nn * Nn) return;
  const int x = (int)(i % Nn), y = (int)((i / Nn) % Nn), z = (int)(i / ((int64_t)Nn * Nn));
  const bool bnd = x == 0 || y == 0 || z == 0 || x == Nn - 1 || y == Nn - 1 || z == Nn - 1;
  phi[i] = bnd ? h * g[i] : 0.0;
}

// node of solved index i: the Ns^3 solved nodes start at index off per axis
// (Dirichlet: the interior, off = 1; Neumann: all nodes, off = 0)
__device__ __forceinline__ int64_t solved_node(int64_t i, int Ns, int Nn, int off) {
  const int x = (int)(i % Ns) + off, y = (int)((i / Ns) % Ns) + off, z = (int)(i / ((int64_t)Ns * Ns)) + off;
  return x + (int64_t)Nn * (y + (int64_t)Nn * z);
}

// node integral (h = 1) of node g of an axis of the open mesh
__device__ __forceinline__ double box_w1(int g, int Nn, const BoxBand& bd) {
  return (g == 0 || g == Nn - 1) ? bd.wend : bd.wn[g % 3];
}

// deterministic FP64 sums: mode 0, sum of squares of v at the solved nodes
// into *out, with the refinement's state for it; mode 1, sum of v over all
// nodes; mode 2, sum of w3 v over all nodes (w3 the 3-D node integrals)
__global__ void __launch_bounds__(BT) k_box_sum(int mode, int Ns, int Nn, int off, BoxBand bd,
                                                const double* __restrict__ v, double* __restrict__ partial,
                                                unsigned int* __restrict__ counter, double* __restrict__ out,
                                                double rtol, RefineState* __restrict__ st) {
  static_assert(BT == 256, "grid_sum256");
  const int64_t len = mode == 0 ? (int64_t)Ns * Ns * Ns : (int64_t)Nn * Nn * Nn;
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    if (mode == 0) {
      const double x = v[solved_node(i, Ns, Nn, off)];
      acc = fma(x, x, acc);
    } else if (mode == 1) {
      acc += v[i];
    } else {
      const int x = (int)(i % Nn), y = (int)((i / Nn) % Nn), z = (int)(i / ((int64_t)Nn * Nn));
      acc = fma(box_w1(x, Nn, bd) * box_w1(y, Nn, bd) * box_w1(z, Nn, bd), v[i], acc);
    }
  }
  double s;
  if (grid_sum256(acc, gridDim.x, blockIdx.x, partial, counter, s)) {
    *out = s;
    if (mode == 0) refine_begin(s, (double)len, rtol, st);
  }
}

// the first residual at the solved nodes, scaled into FP32; the FP32
// correction added back (pairs: the new iterate as float pairs too)
__global__ void k_box_round(int Ns, int Nn, int off, const double* __restrict__ res,
                            const RefineState* __restrict__ st, float* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < (int64_t)Ns * Ns * Ns) out[i] = (float)(res[solved_node(i, Ns, Nn, off)] * (double)st->scale);
}
__global__ void k_box_add(int Ns, int Nn, int off, const float* __restrict__ x, const RefineState* __restrict__ st,
                          double* __restrict__ phi, df* __restrict__ pairs) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const float inv = st->inv;   // a power of two, or zero: an earlier sweep reached the tolerance
  if (inv != 0.f && i < (int64_t)Ns * Ns * Ns) {
    const int64_t j = solved_node(i, Ns, Nn, off);
    const double v = phi[j] + (double)(x[i] * inv);
    phi[j] = v;
    if (pairs) pairs[j] = df_split(v);
  }
}
__global__ void k_box_clear(int Ns, int Nn, int off, double* __restrict__ phi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < (int64_t)Ns * Ns * Ns) phi[solved_node(i, Ns, Nn, off)] = 0.0;
}

// out = in - s w3 (w3 the node integrals: the load of a constant density, the
// compatibility projection of a Neumann load) or, with constant, out = in - s;
// s = *sum * scale
__global__ void k_box_sub(int Nn, BoxBand bd, const double* __restrict__ sum, double scale, int constant,
                          const double* __restrict__ in, double* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)Nn * Nn * Nn) return;
  const int x = (int)(i % Nn), y = (int)((i / Nn) % Nn), z = (int)(i / ((int64_t)Nn * Nn));
  const double w = constant ? 1.0 : box_w1(x, Nn, bd) * box_w1(y, Nn, bd) * box_w1(z, Nn, bd);
  out[i] = in[i] - (*sum) * scale * w;
}

// box views of the padded grid: element counts and element ids of the charges
__global__ void k_box_counts(int n, int nb, const int* __restrict__ count, int* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)nb * nb * nb) return;
  const int x = (int)(i % nb), y = (int)((i / nb) % nb), z = (int)(i / ((int64_t)nb * nb));
  out[i] = count[x + (int64_t)n * (y + (int64_t)n * z)];
}
__global__ void k_box_cells(int64_t N, int n, int nb, const int* __restrict__ cell, int* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int e = cell[i];
  out[i] = e % n + nb * ((e / n) % n + nb * (e / (n * n)));
}
template <class T>
__global__ void k_box_coeffs(int n, int nb, const T* __restrict__ C, double* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)8 * nb * nb * nb) return;
  const int64_t e = i >> 3;
  const int x = (int)(e % nb), y = (int)((e / nb) % nb), z = (int)(e / ((int64_t)nb * nb));
  out[i] = (double)C[8 * (x + (int64_t)n * (y + (int64_t)n * z)) + (i & 7)];
}

double box_rtol(const fep3m_ctx* c) {
  return c->cfg.mg_rtol > 0 ? c->cfg.mg_rtol : (c->precision == FEP3M_FP64 ? 1e-13 : 1e-10);
}

// B->red: partials of the sums (1024) or of the fused applies from PART on
// (box_apply_blocks), and before them the sums' results and the refinement's state
constexpr int RED_SUM = 1024, RED_STATE = 1026, RED_NORM = 1028, PART = 1060;   // norms: the start's, one per sweep
constexpr int NORMS = PART - RED_NORM - 1;   // (the sweeps past them share the last)
static_assert(sizeof(RefineState) == 2 * sizeof(double), "RED_STATE");

void box_sum(Box* B, int mode, const double* v, double* dst, cudaStream_t s, double rtol = 0.0) {
  const int64_t len = (int64_t)B->Nn * B->Nn * B->Nn;
  const int nblk = (int)std::min<int64_t>(1024, std::max<int64_t>(1, len / (BT * 8)));
  FEP3M_CL k_box_sum<<<nblk, BT, 0, s>>>(mode, B->Ns, B->Nn, B->off, B->band, v, B->red, B->counter, dst,
                                         rtol, (RefineState*)(B->red + RED_STATE));
}

// K phi = rhs at the solved nodes (Dirichlet: the interior, phi's boundary
// values held; Neumann: all, rhs compatible; phi zero at the solved nodes):
// iterative refinement around the FP32 fast-diagonalisation solve, the
// residuals scaled by one power of two near the first one's inverse RMS.  In
// MIXED the residual is formed in double-float arithmetic (as the periodic
// solver's) from a copy of the iterate as float pairs, down to tolerances of
// BOX_PAIR_RTOL: the pairs' rounding leaves 1e-13 (8^3 elements) to 7e-13 (48^3)
// of the Dirichlet residual and 6e-13 to 3e-12 of the Neumann one, FP64 2e-15 and
// 2e-14 (8^3), so a tighter tolerance takes the FP64 residual.  So do values a
// pair cannot hold (an infinite boundary value, beside a charge on its node, is
// NaN as a pair): a NaN norm is looked at again in FP64, which tells an infinite
// residual from none.
// The norms stay on the device: they are read once after as many sweeps as
// the last solve took (and after each further one); sweeps past the first that
// reached the tolerance change nothing (RefineState).  Sets B->sweeps and
// B->relres (the residual relative to that of phi's starting values)
constexpr double BOX_PAIR_RTOL = 1e-11;
cudaError_t box_refine(fep3m_ctx* c, Box* B, const double* rhs, double* phi, bool mixed) {
  const int Ns = B->Ns, Nn = B->Nn;
  const int64_t len = (int64_t)Ns * Ns * Ns, nn3 = (int64_t)Nn * Nn * Nn;
  cudaStream_t s = c->stream;
  const double rtol = box_rtol(c);
  const int max_sweeps = c->cfg.mg_max_cycles > 0 ? c->cfg.mg_max_cycles : 10;
  df* pairs = mixed ? (df*)c->phi_hl : nullptr;
  RefineState* st = (RefineState*)(B->red + RED_STATE);
  double* norm = B->red + RED_NORM;
  cudaError_t e;
  if (mixed && (e = split_pairs(nn3, rhs, B->t[0], s)) != cudaSuccess) return e;
  if (mixed && (e = split_pairs(nn3, phi, pairs, s)) != cudaSuccess) return e;
  BoxApply ap;
  ap.N = Nn;
  ap.Ns = Ns;
  ap.off = B->off;
  ap.pairs = mixed;
  ap.x = mixed ? (const void*)pairs : phi;
  ap.b = mixed ? (const void*)B->t[0] : rhs;
  ap.partials = B->red + PART;
  ap.counter = B->counter;
  const double* r0 = rhs;   // Neumann: phi is zero
  if (!B->neumann) {
    ap.r64 = B->res;
    if ((e = box_apply(ap, s)) != cudaSuccess) return e;
    ap.r64 = nullptr;
    r0 = B->res;
  }
  box_sum(B, 0, r0, norm, s, rtol);
  FEP3M_CL k_box_round<<<gsz(len), BT, 0, s>>>(Ns, Nn, B->off, r0, st, B->r32);
  ap.state = st;
  ap.r = B->r32;
  B->sweeps = 0;
  B->relres = 0.0;
  const int read = std::max(1, std::min(B->plan, std::min(max_sweeps, NORMS)));   // sweeps before the norms are looked at
  for (int k = 0; k < max_sweeps; ++k) {
    if ((e = fdm_apply(B->fdm, B->r32, B->x32, B->w1, B->w2, s)) != cudaSuccess) return e;
    FEP3M_CL k_box_add<<<gsz(len), BT, 0, s>>>(Ns, Nn, B->off, B->x32, st, phi, pairs);
    const int at = std::min(k, NORMS - 1);
    ap.norm = norm + 1 + at;
    if ((e = box_apply(ap, s)) != cudaSuccess) return e;
    if (k + 1 < read) continue;
    // host_red: the state, then the norms
    cudaMemcpyAsync(B->host_red, B->red + RED_STATE, (at + 4) * sizeof(double), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    const RefineState& hs = *(const RefineState*)B->host_red;
    const double n0 = std::sqrt(B->host_red[2]), *nr = B->host_red + 3;
    if (!(n0 > 0.0)) {
      // a zero (or, for non-finite data, NaN) residual: nothing to solve
      FEP3M_CL k_box_clear<<<gsz(len), BT, 0, s>>>(Ns, Nn, B->off, phi);
      if (mixed && n0 != 0.0) return box_refine(c, B, rhs, phi, false);
      return cudaGetLastError();
    }
    int j = 0;   // the first sweep that reached the tolerance (as the device decided), or the last one
    while (j < at && nr[j] > hs.limit) ++j;
    B->plan = j + 1;
    B->sweeps = j == at ? k + 1 : j + 1;
    B->relres = std::sqrt(nr[j]) / (hs.scale * n0);
    if (!(nr[j] > hs.limit)) break;
  }
  return cudaGetLastError();
}
cudaError_t box_refine(fep3m_ctx* c, Box* B, const double* rhs, double* phi) {
  return box_refine(c, B, rhs, phi, c->precision == FEP3M_MIXED && box_rtol(c) >= BOX_PAIR_RTOL);
}

}  // namespace

int box_create(fep3m_ctx* c, int nb, bool neumann, const double* Hw) {
  Box* B = new (std::nothrow) Box();
  if (!B) return FEP3M_ENOMEM;
  c->box = B;
  B->nb = nb;
  B->Nn = 3 * nb + 1;
  B->NI = 3 * nb - 1;
  B->neumann = neumann;
  B->Ns = neumann ? B->Nn : B->NI;
  B->off = neumann ? 0 : 1;
  // mixed mass and node integrals (h = 1)
  double Me[4][4], Ke[4][4], Mpq[4][2];
  element_matrices_q3(Me, Ke, Mpq);
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 2; ++j) B->band.Mpq[i][j] = Mpq[i][j];
  double rs[4] = {0, 0, 0, 0};   // element row sums: the integrals of the shape functions
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) rs[i] += Me[i][j];
  B->band.wn[0] = rs[0] + rs[3];
  B->band.wn[1] = rs[1];
  B->band.wn[2] = rs[2];
  B->band.wend = rs[0];
  {
    std::vector<double> x, w;
    gauss_legendre01(BOX_NGL, x, w);
    for (int k = 0; k < BOX_NGL; ++k) {
      B->quad.t[k] = x[k];
      B->quad.w[k] = w[k];
      q3_values<double>(x[k], B->quad.l[k]);
      const df t = df_split(x[k]);
      B->quad.th[k] = t.h;
      B->quad.tl[k] = t.l;
    }
  }
  // the vertex table [offset][64 nodes] as pairs (Dirichlet), or contracted
  // along each face's normal axis with the shape functions' derivatives there:
  // [face][offset][16 face nodes] (Neumann)
  const int no3 = c->noff * c->noff * c->noff;
  std::vector<df> tab;
  if (!neumann) {
    tab.resize((size_t)no3 * 64);
    for (size_t i = 0; i < tab.size(); ++i) tab[i] = df_split(Hw[i]);
  } else {
    tab.resize((size_t)6 * no3 * 16);
    for (int face = 0; face < 6; ++face) {
      const int ax = face >> 1, st[3] = {1, 4, 16};
      double dv[4];
      q3_derivs<double>(face & 1, dv);
      for (int o = 0; o < no3; ++o)
        for (int m = 0; m < 16; ++m) {
          const double* Ho = Hw + (size_t)o * 64 + (m & 3) * st[(ax + 1) % 3] + (m >> 2) * st[(ax + 2) % 3];
          double v = 0.0;
          for (int k = 0; k < 4; ++k) v += dv[k] * Ho[k * st[ax]];
          tab[((size_t)face * no3 + o) * 16 + m] = df_split(v);
        }
    }
  }
  // boundary elements (padded-grid ids)
  std::vector<int> bel;
  const int n = c->n;
  for (int z = 0; z < nb; ++z)
    for (int y = 0; y < nb; ++y)
      for (int x = 0; x < nb; ++x)
        if (x == 0 || y == 0 || z == 0 || x == nb - 1 || y == nb - 1 || z == nb - 1)
          bel.push_back(x + n * (y + n * z));
  B->nbel = (int)bel.size();
  const int64_t nn3 = (int64_t)B->Nn * B->Nn * B->Nn, ns3 = (int64_t)B->Ns * B->Ns * B->Ns;
  cudaError_t e = cudaSuccess;
  auto al = [&](void** ptr, size_t bytes) {
    if (e == cudaSuccess) e = cudaMalloc(ptr, bytes);
  };
  al((void**)&B->g, box_data_size(c) * sizeof(double));
  al((void**)&B->gstage, box_data_size(c) * sizeof(double));
  al((void**)&B->b, nn3 * sizeof(double));
  al((void**)&B->rhs, nn3 * sizeof(double));
  al((void**)&B->res, nn3 * sizeof(double));
  for (double*& t : B->t) al((void**)&t, nn3 * sizeof(double));
  al((void**)&B->r32, ns3 * sizeof(float));
  al((void**)&B->x32, ns3 * sizeof(float));
  al((void**)&B->w1, ns3 * sizeof(float));
  al((void**)&B->w2, ns3 * sizeof(float));
  al((void**)&B->bel, bel.size() * sizeof(int));
  al((void**)&B->red, (PART + box_apply_blocks(B->Nn)) * sizeof(double));
  al((void**)&B->counter, sizeof(unsigned int));
  al((void**)&B->tab, tab.size() * sizeof(df));
  if (neumann) al((void**)&B->sface, (size_t)6 * nb * nb * 16 * sizeof(double));
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FEP3M_ENOMEM : FEP3M_ECUDA;
  if (cudaMallocHost(&B->host_red, (NORMS + 3) * sizeof(double)) != cudaSuccess) return FEP3M_ENOMEM;
  cudaMemset(B->counter, 0, sizeof(unsigned int));
  if ((e = box_apply_setup(c->st)) != cudaSuccess) return FEP3M_ECUDA;
  cudaMemset(B->g, 0, box_data_size(c) * sizeof(double));
  cudaMemcpy(B->bel, bel.data(), bel.size() * sizeof(int), cudaMemcpyHostToDevice);
  cudaMemcpy(B->tab, tab.data(), tab.size() * sizeof(df), cudaMemcpyHostToDevice);
  std::vector<double> lam, V;
  box_eigen(3, nb, !neumann, lam, V);
  e = fdm_setup(B->fdm, B->Ns, lam, V, 1, !(c->cfg.flags & FEP3M_CUDA_CORES), neumann);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FEP3M_ENOMEM : FEP3M_ECUDA;
  return FEP3M_OK;
}

void box_destroy(fep3m_ctx* c) {
  Box* B = c->box;
  if (!B) return;
  void* p[] = {B->g, B->gstage, B->b, B->rhs, B->res, B->r32, B->x32, B->w1, B->w2, B->bel, B->red, B->sface, B->tab, B->counter};
  for (void* x : p)
    if (x) cudaFree(x);
  for (double* t : B->t)
    if (t) cudaFree(t);
  if (B->host_red) cudaFreeHost(B->host_red);
  fdm_free(B->fdm);
  delete B;
  c->box = nullptr;
}

// values of the boundary data: the (3 nb + 1)^3 nodes (Dirichlet) or the
// 6 nb^2 BOX_NGL^2 face quadrature points (Neumann)
int64_t box_data_size(const fep3m_ctx* c) {
  const Box* B = c->box;
  if (B->neumann) return (int64_t)6 * B->nb * B->nb * BOX_NGL * BOX_NGL;
  return (int64_t)B->Nn * B->Nn * B->Nn;
}

int box_set_boundary(fep3m_ctx* c, const double* g_dev) {
  Box* B = c->box;
  return cudaMemcpyAsync(B->g, g_dev, box_data_size(c) * sizeof(double), cudaMemcpyDeviceToDevice, c->stream) ==
                 cudaSuccess
             ? FEP3M_OK
             : FEP3M_ECUDA;
}

// the load vector of the box (three separable passes; the first reads the
// padded grid's vertex density)
static void box_load(fep3m_ctx* c, Box* B, cudaStream_t s) {
  const int nb = B->nb, n = c->n, Nn = B->Nn, V1 = nb + 1;
  const int64_t n1 = (int64_t)Nn * V1 * V1, n2 = (int64_t)Nn * Nn * V1, n3 = (int64_t)Nn * Nn * Nn;
  if (c->precision == FEP3M_MIXED) {
    float *t1 = (float*)B->t[0], *t2 = (float*)B->t[1];
    FEP3M_CL k_box_load_axis<float, float><<<gsz(n1), BT, 0, s>>>(nb, 0, Nn, V1, V1, 1, n, (int64_t)n * n, B->band,
                                                                 (const float*)c->rv, t1, 1.0);
    FEP3M_CL k_box_load_axis<float, float><<<gsz(n2), BT, 0, s>>>(nb, 1, Nn, Nn, V1, 1, Nn, (int64_t)Nn * V1, B->band,
                                                                 t1, t2, 1.0);
    FEP3M_CL k_box_load_axis<float, double><<<gsz(n3), BT, 0, s>>>(nb, 2, Nn, Nn, Nn, 1, Nn, (int64_t)Nn * Nn, B->band,
                                                                  t2, B->b, 4.0 * M_PI / (120.0 * 120.0 * 120.0));
  } else {
    double *t1 = B->t[0], *t2 = B->t[1];
    FEP3M_CL k_box_load_axis<double, double><<<gsz(n1), BT, 0, s>>>(nb, 0, Nn, V1, V1, 1, n, (int64_t)n * n, B->band,
                                                                   (const double*)c->rv, t1, 1.0);
    FEP3M_CL k_box_load_axis<double, double><<<gsz(n2), BT, 0, s>>>(nb, 1, Nn, Nn, V1, 1, Nn, (int64_t)Nn * V1,
                                                                   B->band, t1, t2, 1.0);
    FEP3M_CL k_box_load_axis<double, double><<<gsz(n3), BT, 0, s>>>(nb, 2, Nn, Nn, Nn, 1, Nn, (int64_t)Nn * Nn,
                                                                   B->band, t2, B->b, 4.0 * M_PI);
  }
}

// Neumann: rhs less its component along the node integrals (compatible with
// the constant null space); after the solve, phi less its mean (int phi = 0)
static void box_project(Box* B, double* rhs, cudaStream_t s) {
  const int64_t nn3 = (int64_t)B->Nn * B->Nn * B->Nn;
  const double w3 = (double)B->nb * B->nb * B->nb;   // the box's volume, h = 1
  box_sum(B, 1, rhs, B->red + RED_SUM, s);
  FEP3M_CL k_box_sub<<<gsz(nn3), BT, 0, s>>>(B->Nn, B->band, B->red + RED_SUM, 1.0 / w3, 0, rhs, rhs);
}
static void box_zero_mean(Box* B, double* phi, cudaStream_t s) {
  const int64_t nn3 = (int64_t)B->Nn * B->Nn * B->Nn;
  const double w3 = (double)B->nb * B->nb * B->nb;
  box_sum(B, 2, phi, B->red + RED_SUM, s);
  FEP3M_CL k_box_sub<<<gsz(nn3), BT, 0, s>>>(B->Nn, B->band, B->red + RED_SUM, 1.0 / w3, 1, phi, phi);
}

int box_compute(fep3m_ctx* c, double* phi_dev, double* U_dev) {
  Box* B = c->box;
  cudaStream_t s = c->stream;
  const int64_t nn3 = (int64_t)B->Nn * B->Nn * B->Nn;
  cudaError_t e;
  if (cudaMemsetAsync(c->iflags + 2, 0, sizeof(int), s) != cudaSuccess) return FEP3M_ECUDA;
  if ((e = element_lists(c)) != cudaSuccess) return FEP3M_ECUDA;
  box_load(c, B, s);
  // singular sums and screen field of the targets (need no mesh solution)
  if ((e = pair_screen(c, 0, s, false)) != cudaSuccess) return FEP3M_ECUDA;
  if (cudaMemsetAsync(c->phi64, 0, nn3 * sizeof(double), s) != cudaSuccess) return FEP3M_ECUDA;
  const size_t asz = (size_t)c->noff * c->noff * c->noff * sizeof(df);
  const bool f32 = c->precision == FEP3M_MIXED;
  const double* rhs = B->b;
  if (!B->neumann) {
    // boundary values (Eq. bcadjust), then the interior solve
    const size_t smem = asz + BCH * sizeof(BoxSrc) + BT * (sizeof(double) + 2 * sizeof(df));
    if (f32)
      FEP3M_CL k_box_boundary<float><<<B->nbel, BT, smem, s>>>(c->n, B->nb, c->n_sr, c->h, c->q_scale,
                                                               1.0 / c->q_scale, B->bel, c->start,
                                                               c->ecoord, (const float4*)c->part, (const float*)c->Cv,
                                                               (const float2*)B->tab, B->g, c->phi64);
    else
      FEP3M_CL k_box_boundary<double><<<B->nbel, BT, smem, s>>>(c->n, B->nb, c->n_sr, c->h, c->q_scale,
                                                                1.0 / c->q_scale, B->bel,
                                                                c->start, c->ecoord, (const vec4<double>::type*)c->part,
                                                                (const double*)c->Cv, (const float2*)B->tab, B->g,
                                                                c->phi64);
  } else {
    // the adjusted flux as a boundary load, made compatible
    const unsigned nfe = (unsigned)(6 * B->nb * B->nb);
    if (f32)
      FEP3M_CL k_box_flux<float><<<nfe, BT, asz, s>>>(c->n, B->nb, c->n_sr, c->h, c->q_scale, 1.0 / c->q_scale, B->quad, c->start,
                                                      c->ecoord, (const float4*)c->part, (const float*)c->Cv,
                                                      (const float2*)B->tab, B->g, B->sface);
    else
      FEP3M_CL k_box_flux<double><<<nfe, BT, asz, s>>>(c->n, B->nb, c->n_sr, c->h, c->q_scale, 1.0 / c->q_scale, B->quad, c->start,
                                                       c->ecoord, (const vec4<double>::type*)c->part,
                                                       (const double*)c->Cv, (const float2*)B->tab, B->g, B->sface);
    FEP3M_CL k_box_sgather<<<gsz(nn3), BT, 0, s>>>(B->nb, B->b, B->sface, B->rhs);
    box_project(B, B->rhs, s);
    rhs = B->rhs;
  }
  if ((e = box_refine(c, B, rhs, c->phi64)) != cudaSuccess) return FEP3M_ECUDA;
  if (B->neumann) box_zero_mean(B, c->phi64, s);
  if ((e = pair_prepare(c)) != cudaSuccess) return FEP3M_ECUDA;
  if ((e = pair_eval(c, phi_dev, 0)) != cudaSuccess) return FEP3M_ECUDA;
  if (U_dev && (e = energy(c, U_dev)) != cudaSuccess) return FEP3M_ECUDA;
  if (cudaGetLastError() != cudaSuccess) return FEP3M_ECUDA;
  return B->relres <= 10 * box_rtol(c) ? FEP3M_OK : FEP3M_ENOCONV;
}

int box_solve(fep3m_ctx* c, double* rhs_dev, double* phi_dev) {
  Box* B = c->box;
  const int Nn = B->Nn;
  const int64_t nn3 = (int64_t)Nn * Nn * Nn;
  if (B->neumann) {
    box_project(B, rhs_dev, c->stream);
    cudaMemsetAsync(phi_dev, 0, nn3 * sizeof(double), c->stream);
  } else {
    FEP3M_CL k_box_plain_bvals<<<gsz(nn3), BT, 0, c->stream>>>(Nn, c->h, B->g, phi_dev);
  }
  if (box_refine(c, B, rhs_dev, phi_dev) != cudaSuccess) return FEP3M_ECUDA;
  if (B->neumann) box_zero_mean(B, phi_dev, c->stream);
  if (cudaGetLastError() != cudaSuccess) return FEP3M_ECUDA;
  return B->relres <= 10 * box_rtol(c) ? FEP3M_OK : FEP3M_ENOCONV;
}

// box views for the inspection entry points: counts (nb^3) and element ids
// (N) into device buffers, and the element lists as FP64 (8 nb^3)
cudaError_t box_binning(fep3m_ctx* c, int* count_out, int* cell_out) {
  const int nb = c->box->nb;
  if (count_out)
    FEP3M_CL k_box_counts<<<gsz((int64_t)nb * nb * nb), BT, 0, c->stream>>>(c->n, nb, c->count, count_out);
  if (cell_out) FEP3M_CL k_box_cells<<<gsz(c->N), BT, 0, c->stream>>>(c->N, c->n, nb, c->cell, cell_out);
  return cudaGetLastError();
}
cudaError_t box_coeffs(fep3m_ctx* c, double* out) {
  const int nb = c->box->nb;
  const int64_t len = (int64_t)8 * nb * nb * nb;
  if (c->precision == FEP3M_MIXED)
    FEP3M_CL k_box_coeffs<float><<<gsz(len), BT, 0, c->stream>>>(c->n, nb, (const float*)c->C, out);
  else
    FEP3M_CL k_box_coeffs<double><<<gsz(len), BT, 0, c->stream>>>(c->n, nb, (const double*)c->C, out);
  return cudaGetLastError();
}

}  // namespace fep3m
