// Short-range evaluation (Sec. 2.4-2.5) and the smooth-potential evaluation
// (Sec. 2.3, Eq. evalsmooth), and the reverse sweeps of the adjoint.
//
// For a target charge t in element e (local coordinate tau_t in [0,1]^3):
//   Phi_t = (1/h) sum_m G_e[m] u_m(tau_t) + sum_{j in block(e), j != t} Q_j / |x_j - x_t|
//   G_e[m] = phi[node(e, m)] - sum_{o} A_e(o) H(o, m)
// where the second term of G_e is the screen potential of every charge of the
// (2 n_sr + 1)^3 block around e (own charge included: the self term of
// Sec. 2.5), written at the 64 order-3 nodes of e.  It is the element-to-point
// evaluation of Sec. 3.1.2 (Eq. sc with per-element combined coefficients),
// regrouped by vertex: all screens are sums of vertex hats, every vertex hat
// has the same FE table H (Remark of Sec. 4), so the block's screens act
// through the vertex amplitudes
//   A_e(o) = sum over the corners k of block elements at vertex v = e - o of C[v - k][k]
// which equal the full vertex density r_v inside the block and partial sums on
// its boundary.  H(o, m) is the table value at node m of an element at offset
// o (element units) from the vertex.
//
// Two launches per evaluation: k_pair_screen (the screen field sum_o A_e(o)
// H(o, m) and the singular sums; it needs no mesh solution and runs while the
// mesh is solved) and k_pair_eval (G_e and the contraction with u_m(tau_t)
// after the solve).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "df.cuh"
#include "tc.cuh"

namespace fep3m {

namespace {

using namespace tc;
constexpr uint32_t UMMA_IDESC = umma_idesc(64, 64);   // the screen contraction: M = 64 elements, N = 64 nodes

constexpr int PT = 256;
constexpr int PTC = 512;   // threads of the tensor-core screen kernel

__device__ __forceinline__ int wrapn(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

template <class T> __device__ __forceinline__ T rsq(T x);
// 1 / sqrt(x) in FP64 from the FP32 hardware estimate y, refined by one
// third-order (Householder) step: with e = 1 - x y^2, 1 / sqrt(x) =
// y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2 / 8 + O(e^3)), and the dropped term is
// below 2^-64 (emulated worst case 0.9 ulp).  Outside [2^-100, 2^100), where
// the FP32 estimate could under- or overflow (including x = 0, coincident
// charges, and negative or NaN x), the FP64 division is used; the range test
// reads the exponent bits on the integer pipe.
template <> __device__ __forceinline__ double rsq<double>(double x) {
  const int bexp = __double2hiint(x) >> 20;   // sign and biased exponent
  if ((unsigned)(bexp - 923) >= 200u) return 1.0 / sqrt(x);
  const double y = (double)rsqrt_est((float)x);
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
// the hardware estimate refined by one Newton step, y (3 - x y^2) / 2 (for x
// = 0 the estimate is +inf and the step gives NaN: coincident charges)
template <> __device__ __forceinline__ float rsq<float>(float x) {
  const float y = rsqrt_est(x);
  return y * fmaf(-0.5f * x, y * y, 1.5f);
}

// fused multiply-add in the working precision
__device__ __forceinline__ float fmaw(float a, float b, float c) { return fmaf(a, b, c); }

// compensated (Kahan) accumulator; FP64 uses plain sums
template <class T> struct Acc {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T v) {
    if (sizeof(T) == 4) {
      T y = v - c;
      T t = s + y;
      c = (t - s) - y;
      s = t;
    } else {
      s += v;
    }
  }
  __device__ __forceinline__ T get() const { return s - c; }
};

// ----------------------------------------------------------- brick kernels
// k_pair_screen: one CTA per brick of BX x BY x BZ target elements:
//  (1) the brick's "extended vertex field" R in shared memory (below);
//  (2) the screen field of all brick elements at their 64 nodes,
//      sum_o A(e, o) H(o, m): on the tensor cores (split bf16 MMAs) or as 512
//      rank-1 updates of a 64 x 64 tile on the CUDA cores (4 x 4 register
//      tile per thread, A and H staged in chunks of OCH offsets);
//  (3) the charges of the brick's short-range halo, staged in shared memory
//      in element order (when they fit) with each charge's halo x index;
//  (4) a few threads per target, each summing some of the 49 element rows of
//      the target's block (one contiguous run of staged charges per row).
// k_pair_eval: one CTA per brick after the solve: G = phi - screen field at
// the nodes, contracted with the shape functions at each target.
constexpr int BX = 4, BY = 4, BZ = 4, BE = BX * BY * BZ;   // 64 elements per brick
constexpr int OCH = 32;                                      // offsets per chunk
constexpr int MAXROW = 81;                                   // rows (y, z) of the block (n_sr <= 4)

template <class T>
__device__ __forceinline__ void warp_sum(T& v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
}

// the rows (dy, dz) of a block, by the CTA; ends with a barrier
__device__ __forceinline__ void row_table(int n_sr, char2* rows /* MAXROW */) {
  const int nb = 2 * n_sr + 1;
  for (int r = threadIdx.x; r < nb * nb; r += blockDim.x) rows[r] = make_char2(r % nb - n_sr, r / nb - n_sr);
  __syncthreads();
}

// The rows (y, z) of a target's block: row r's charges are a run of consecutive
// sorted ones from rows[r].x on, and where the row wraps rows[r].y of them are
// followed by a second run from rows[r].z on; pre[r] the charges of the rows
// before it.  Returns (and pre[nrow] holds) their number.  By a warp.
__device__ __forceinline__ int warp_rows(int n, int n_sr, const char2* tab, int ex, int ey, int ez,
                                         const int* __restrict__ start, int4* rows /* MAXROW */,
                                         int* pre /* MAXROW + 1 */) {
  const int lane = threadIdx.x & 31, nb = 2 * n_sr + 1, nrow = nb * nb;
  int carry = 0;
  for (int r0 = 0; r0 < nrow; r0 += 32) {
    const int r = r0 + lane;
    int a0 = 0, a1 = 0, b0 = 0, b1 = 0;
    if (r < nrow) {
      const char2 d = tab[r];
      int yy = ey + d.x, zz = ez + d.y;
      yy += yy < 0 ? n : (yy >= n ? -n : 0);
      zz += zz < 0 ? n : (zz >= n ? -n : 0);
      const int64_t rowbase = (int64_t)n * (yy + (int64_t)n * zz);
      const int x0 = ex - n_sr, x1 = ex + n_sr;
      if (x0 < 0) {
        a0 = start[rowbase + x0 + n]; a1 = start[rowbase + n];        // x0+n .. n-1
        b0 = start[rowbase];          b1 = start[rowbase + x1 + 1];   // 0 .. x1
      } else if (x1 >= n) {
        a0 = start[rowbase + x0];     a1 = start[rowbase + n];        // x0 .. n-1
        b0 = start[rowbase];          b1 = start[rowbase + x1 - n + 1];
      } else {
        a0 = start[rowbase + x0];     a1 = start[rowbase + x1 + 1];
      }
    }
    const int cnt = a1 - a0 + b1 - b0;
    int x = cnt;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += v;
    }
    if (r < nrow) {
      rows[r] = make_int4(a0, a1 - a0, b0, 0);
      pre[r] = carry + x - cnt;
    }
    carry += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) pre[nrow] = carry;
  __syncwarp();
  return carry;
}

// the source's element less the target's, the nearest image
__device__ __forceinline__ int block_delta(int d, int n, int n_sr) {
  return d > n_sr ? d - n : (d < -n_sr ? d + n : d);
}

// Singular sum for one target over its block, lanes of one warp in parallel.
// w[j]: source weights; returns sum w/r and (GRAD) sum w (x_j - x_t)/r^3 in
// every lane, physical units, compensated per lane.
template <class T, bool GRAD>
__device__ __forceinline__ void warp_singular(int n, int n_sr, const char2* tab, T h, int ex, int ey, int ez, int slot,
                                              typename vec4<T>::type pt, const int* __restrict__ start,
                                              const typename vec4<T>::type* __restrict__ part,
                                              const int* __restrict__ ecoord, int4* rows, int* pre,
                                              const double* __restrict__ w, T out[4]) {
  const int total = warp_rows(n, n_sr, tab, ex, ey, ez, start, rows, pre);
  Acc<T> ps, fx, fy, fz;
  int k = 0;
  for (int f = threadIdx.x & 31; f < total; f += 32) {
    while (pre[k + 1] <= f) ++k;
    const int i = f - pre[k];
    const int4 r = rows[k];
    const int j = i < r.y ? r.x + i : r.z + (i - r.y);
    if (j == slot) continue;
    const typename vec4<T>::type pj = part[j];
    const int ec = ecoord[j];
    const int dx = block_delta((ec & 1023) - ex, n, n_sr), dy = block_delta(((ec >> 10) & 1023) - ey, n, n_sr),
              dz = block_delta((ec >> 20) - ez, n, n_sr);
    const T rx = (T(dx) + (pj.x - pt.x)) * h, ry = (T(dy) + (pj.y - pt.y)) * h, rz = (T(dz) + (pj.z - pt.z)) * h;
    const T ir = rsq<T>(rx * rx + ry * ry + rz * rz);
    const T wj = (T)w[j];
    ps.add(wj * ir);
    if (GRAD) {
      const T f3 = wj * ir * ir * ir;
      fx.add(f3 * rx);
      fy.add(f3 * ry);
      fz.add(f3 * rz);
    }
  }
  out[0] = ps.get();
  out[1] = fx.get();
  out[2] = fy.get();
  out[3] = fz.get();
  for (int i = 0; i < (GRAD ? 4 : 1); ++i) warp_sum(out[i]);
  __syncwarp();
}

// ---------------------------------------------------- FP64 singular sums
// An FP64 operation costs as much as 64 FP32 ones on this GPU, so the charges'
// own singular sums of an FP64 context run in float pairs.  A charge for them:
// per axis its local coordinate tau = a + b + c, a the multiple of 2^-20 nearest
// tau, b the multiple of 2^-42 nearest the rest and c what is left (below
// 2^-43), so that the differences of two coordinates' parts (a's plus a whole
// number) are exact in FP32, and a's difference is zero or larger than b's; and
// the charge times a power of two near the inverse mean charge
// (fep3m_ctx::q_scale), so that low words stay normal numbers.
struct __align__(16) PairCharge {
  float a[3], b[3], c[3];
  df q;
  float ex;   // the element's x coordinate
};
static_assert(sizeof(PairCharge) == FEP3M_PAIR_CHARGE_BYTES, "the context's allocation");

__global__ void k_pair_charges(int64_t N, const vec4<double>::type* __restrict__ part,
                               const int* __restrict__ ecoord, double scale,
                               PairCharge* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const vec4<double>::type p = part[i];
  const double x[3] = {p.x, p.y, p.z};
  PairCharge c;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double a = rint(x[k] * 1048576.0) * (1.0 / 1048576.0);
    const double r = x[k] - a, b = rint(r * 4398046511104.0) * (1.0 / 4398046511104.0);   // 2^42
    c.a[k] = (float)a;
    c.b[k] = (float)b;
    c.c[k] = (float)(r - b);
  }
  c.q = df_split(p.w * scale);
  c.ex = (float)(ecoord[i] & 1023);
  out[i] = c;
}

// the same in FP64 (as exact as the coordinates)
__device__ __forceinline__ double charge_diff64(const PairCharge& s, const PairCharge& t, int k, float d) {
  return (double)((s.a[k] - t.a[k]) + d) +
         ((double)(s.b[k] - t.b[k]) + (double)(s.c[k] - t.c[k]));
}
// x_s - x_t along axis k, the source's element d elements on
__device__ __forceinline__ df charge_diff(const PairCharge& s, const PairCharge& t, int k, float d) {
  const float A = (s.a[k] - t.a[k]) + d, B = s.b[k] - t.b[k];   // exact
  const float h = A + B;
  return {h, (B - (h - A)) + (s.c[k] - t.c[k])};
}

// One warp per target: sum Q / r into phi_s, (GRAD) sum Q (x_j - x_t) / r^3
// into E_s, and half of them to psi and gpsi when given (the singular adjoint
// for the energy's weights Q / 2).  A lane sums sixteen charges at a time in
// pairs (element units) and those sums in three floats.  A pair's term is good
// to a few 2^-48; the few charges within three quarters of an element, whose terms
// are the largest, take FP64 (as do distances outside df_in_range).  The sum keeps
// the terms' roundings, about 2^-48 of the root of the sum of their squares, where
// FP64 terms would leave a thirtieth of that (emulated: rock salt, two charges per
// element edge, 5e-14 against 2e-15 of potentials of 3.5).  What a potential as a
// whole is off the method by is more, the screens' table and its contraction: against
// a table solved in long double, with the mesh solved to rounding, neutral charges at
// 0.1 to 8 per element and n_sr 2 to 4 came out 0.4 to 1.03 times as far off as with
// FP64 terms and tables (potentials 3e-14 to 6e-13, forces 2e-15 to 5e-12), charges of
// one sign 1.0 (potentials) and 1.2 times (forces, n_sr = 4).  About 120 FP32 operations per pair;
// bound by FP32 issue and, for few targets, by the latency of the loads.
// 4000 charges, q = 2, potentials: 266 -> 42 us.
constexpr float NEAR2 = 0.5625f;   // three quarters of an element, squared
template <bool GRAD>
__global__ void __launch_bounds__(PT) k_singular64(int64_t N, int n, int n_sr, double u0, double u1,
                                                   const int* __restrict__ start, const PairCharge* __restrict__ ch,
                                                   const int* __restrict__ ecoord, double* __restrict__ phi_s,
                                                   double* __restrict__ E_s, double* __restrict__ psi,
                                                   double* __restrict__ gpsi) {
  constexpr int NS = GRAD ? 4 : 1;
  __shared__ int4 rows_all[PT / 32][MAXROW];
  __shared__ int pre_all[PT / 32][MAXROW + 1];
  __shared__ char2 tab[MAXROW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = blockIdx.x * (int64_t)(PT / 32) + warp;
  row_table(n_sr, tab);
  if (t >= N) return;
  int4* rows = rows_all[warp];
  int* pre = pre_all[warp];
  const int et = ecoord[t], ex = et & 1023, ey = (et >> 10) & 1023, ez = et >> 20;
  const PairCharge ct = ch[t];
  const int total = warp_rows(n, n_sr, tab, ex, ey, ez, start, rows, pre);
  // x displacement of a charge's element: its coordinate plus one of these (the period taken
  // off in the first run of a row that wraps below, or the second of one that wraps above)
  const float sx0 = (float)((ex - n_sr < 0 ? -n : 0) - ex), sx1 = (float)((ex - n_sr < 0 ? 0 : n) - ex);
  tf tot[NS] = {};
  double s64[NS] = {};
  bool met = false;   // some distance took FP64
  int k = 0;
  for (int f0 = lane; f0 < total; f0 += 32 * 16) {
    df s[NS] = {};
#pragma unroll 2
    for (int f = f0; f < min(total, f0 + 32 * 16); f += 32) {
      while (pre[k + 1] <= f) ++k;
      const int i = f - pre[k];
      const int4 r = rows[k];
      const bool first = i < r.y;
      const int j = first ? r.x + i : r.z + (i - r.y);
      if (j == (int)t) continue;
      const PairCharge cj = ch[j];
      const char2 d = tab[k];
      const float ddx = cj.ex + (first ? sx0 : sx1);
      const df dx = charge_diff(cj, ct, 0, ddx), dy = charge_diff(cj, ct, 1, (float)d.x),
               dz = charge_diff(cj, ct, 2, (float)d.y);
      const df x2 = df_sqr(dx), y2 = df_sqr(dy), z2 = df_sqr(dz);
      const df xy = df_two_sum(x2.h, y2.h), xyz = df_two_sum(xy.h, z2.h);
      const df r2 = {xyz.h, xyz.l + ((xy.l + x2.l) + (y2.l + z2.l))};
      if (r2.h >= NEAR2 && df_in_range(r2)) {
        const df ir = df_rsqrt<true>(r2);
        const df w = df_mul(cj.q, ir);
        df_acc(s[0], w);
        if constexpr (GRAD) {
          const df g = df_mul(w, df_sqr(ir));
          df_fma(s[1], g, dx);
          df_fma(s[2], g, dy);
          df_fma(s[3], g, dz);
        }
      } else {
        const double x = charge_diff64(cj, ct, 0, ddx), y = charge_diff64(cj, ct, 1, (float)d.x),
                     z = charge_diff64(cj, ct, 2, (float)d.y);
        met = true;
        const double ir = rsq<double>(x * x + y * y + z * z), w = df_value(cj.q) * ir;
        s64[0] += w;
        if constexpr (GRAD) {
          const double g = w * ir * ir;
          s64[1] += g * x;
          s64[2] += g * y;
          s64[3] += g * z;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) tf_add(tot[i], s[i]);
  }
  auto with = [&](tf a, int o) -> tf {   // a plus lane ^ o's
    tf_add(a, tf{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.m, o),
                 __shfl_xor_sync(0xffffffffu, a.l, o)});
    return a;
  };
  // the lanes' sums: with four, the lanes first split them, lane i (mod 4) adding up sum i
  tf sum = tot[0];
  if constexpr (GRAD) {
    const bool b1 = lane & 1, b2 = lane & 2;
    auto give = [&](const tf& keep, const tf& other, int o) -> tf {
      tf a = keep;
      tf_add(a, tf{__shfl_xor_sync(0xffffffffu, other.h, o), __shfl_xor_sync(0xffffffffu, other.m, o),
                   __shfl_xor_sync(0xffffffffu, other.l, o)});
      return a;
    };
    const tf e = give(b1 ? tot[1] : tot[0], b1 ? tot[0] : tot[1], 1), f = give(b1 ? tot[3] : tot[2], b1 ? tot[2] : tot[3], 1);
    sum = give(b2 ? f : e, b2 ? e : f, 2);
  } else {
    sum = with(with(sum, 1), 2);
  }
  sum = with(with(with(sum, 4), 8), 16);
  double out = df_value(sum);   // lane i's: sum i
  if (__any_sync(0xffffffffu, met)) {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      warp_sum(s64[i]);
      if (lane == i) out += s64[i];
    }
  }
  if (lane >= NS) return;
  out *= lane == 0 ? u0 : u1;   // physical units
  if (lane == 0) {
    phi_s[t] = out;
    if (psi) psi[t] = 0.5 * out;
  } else {
    E_s[3 * t + lane - 1] = out;
    if (gpsi) gpsi[3 * t + lane - 1] = 0.5 * out;
  }
}

// Extended vertex field: per axis SW = 3 BX + 2 n_sr - 1 slots, the first
// SF = BX + 2 n_sr - 1 the full vertex densities of the vertices interior
// offsets reach, then BX slots of corner-1-only sums (offset -(n_sr+1),
// vertex e + n_sr + 1) and BX of corner-0-only sums (offset n_sr, vertex
// e - n_sr).  A(e, o) is then the single value R[beta(o) + lambda(e)].
constexpr int STAGE_CAP = 1536;   // halo charges staged in shared memory

// CUDA-core layout (TC = false): region 1 holds R first, then the staged
// charges; A and H chunks follow.  Tensor-core layout (TC = true): 48 KB of
// operand tiles (1 KB aligned), then R, then the staged charges.  Both end with
// the index tables.
template <bool TC>
struct Pair3Smem {
  static constexpr int NT = TC ? PTC : PT;
  // bytes per R and chunk-operand entry: one float (tensor cores) or a hi + lo
  // float pair (the double-float CUDA-core contraction)
  static constexpr int ES = TC ? 4 : 8;
  __host__ __device__ static int SW(int n_sr) { return 3 * BX + 2 * n_sr - 1; }
  __host__ __device__ static int HW(int n_sr) { return BX + 2 * n_sr; }
  // R's strides: rows 4 modulo 16 entries and (tensor cores) planes 16 modulo 32, so that the 4 x 4
  // x 2 elements a warp reads fall on 32 different banks
  __host__ __device__ static int RS(int n_sr) { return TC ? SW(n_sr) + (20 - SW(n_sr) % 16) % 16 : SW(n_sr); }
  __host__ __device__ static int PS(int n_sr) {
    const int p = RS(n_sr) * SW(n_sr);
    return TC ? p + (48 - p % 32) % 32 : p;
  }
  __host__ __device__ static size_t rbytes(int n_sr) {
    return ((size_t)PS(n_sr) * SW(n_sr) * ES + 31) / 32 * 32;
  }
  __host__ __device__ static size_t region1(int n_sr) {
    const size_t r = rbytes(n_sr);
    const size_t stg = (size_t)STAGE_CAP * sizeof(float4);
    return r > stg ? r : stg;
  }
  __host__ __device__ static size_t ints(int n_sr) {
    const int hw = HW(n_sr);
    const int noff = 2 * n_sr + 2, nb = 2 * n_sr + 1, sw = SW(n_sr);
    return (size_t)hw * hw * hw + 1 + BE + 1 + 1 + NT / 32 + 1 + 3 + ((size_t)noff * noff * noff + 63) / 64 * 64 +
           (size_t)nb * nb + 3 * sw + 3 * hw + 32;
  }
  static constexpr size_t TILES = 6 * 8192;   // three bf16 pieces of A (64 x 64) and of B (64 x 64)
  // tensor cores: the staged charges in a region of their own (staged while the contraction runs)
  __host__ __device__ static size_t stgbytes() {
    return (size_t)STAGE_CAP * sizeof(float4) + ((size_t)STAGE_CAP + 15) / 16 * 16;
  }
  static size_t bytes(int n_sr) {
    if (TC) return 1024 + TILES + rbytes(n_sr) + stgbytes() + ints(n_sr) * sizeof(int) + 16;
    return region1(n_sr) + 2 * (size_t)OCH * 64 * ES + ints(n_sr) * sizeof(int) + (size_t)STAGE_CAP;
  }
};

// exclusive scan of one int per thread over the block (NT threads); returns the
// thread's prefix and writes the total to *total
template <int NT>
__device__ __forceinline__ int block_scan_excl(int v, int* wsum /* NT/32 + 1 */, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    int a = 0;
    for (int w = 0; w < NT / 32; ++w) {
      const int t = wsum[w];
      wsum[w] = a;
      a += t;
    }
    wsum[NT / 32] = a;
  }
  __syncthreads();
  const int res = wsum[wid] + x - v;
  *total = wsum[NT / 32];
  __syncthreads();
  return res;
}

// Named CTA barriers (bar.sync id, n): groups of whole warps synchronise
// among themselves (id 0 with the CTA's thread count is __syncthreads).
__device__ __forceinline__ void group_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// group_sync that also returns whether v was true in any thread of the group
__device__ __forceinline__ bool group_sync_or(int id, int n, bool v) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

// exclusive scan of one int per thread over a group of GN threads (gt its
// index in the group, whole warps; barrier id); returns the prefix, writes
// the total to *total
template <int GN>
__device__ __forceinline__ int group_scan_excl(int gt, int id, int v, int* wsum /* GN/32 + 1 */, int* total) {
  const int lane = gt & 31, wid = gt >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  group_sync(id, GN);
  if (gt == 0) {
    int a = 0;
    for (int w = 0; w < GN / 32; ++w) {
      const int t = wsum[w];
      wsum[w] = a;
      a += t;
    }
    wsum[GN / 32] = a;
  }
  group_sync(id, GN);
  const int res = wsum[wid] + x - v;
  *total = wsum[GN / 32];
  group_sync(id, GN);
  return res;
}

constexpr int SG = 256;   // threads of the short-range sums (the whole CTA on the CUDA cores, half of it
                          // beside the tensor-core contraction)

// How the halo's charges reach the singular sums: all staged in shared memory
// at once; staged tile by tile (consecutive runs of halo elements whose charges
// fit); or, when a single element holds more charges than fit, read from
// global memory.
enum HaloMode { HALO_STAGED = 0, HALO_TILED = 1, HALO_GLOBAL = 2 };

// the halo element id of halo index i (HW^3 elements, x fastest)
__device__ __forceinline__ int halo_gid(int i, int n, int HW, const int* __restrict__ we) {
  const int hx = i % HW, hy = (i / HW) % HW, hz = i / (HW * HW);
  return we[hx] + n * (we[HW + hy] + n * we[2 * HW + hz]);
}

// Prefix of the charges of the brick's short-range halo (HW^3 elements):
// hs[i] = the first slot of halo element i in halo order, hs[HW^3] = the total;
// the charges are staged in shared memory in that order (with each charge's
// halo x index) when they all fit (cap).  By SG threads (gt, barrier id).
// Returns the HaloMode.
__device__ int stage_halo(int gt, int id, int n, int HW, const int* __restrict__ we, const int* __restrict__ start,
                          const int* __restrict__ count, const float4* __restrict__ part, int cap, float4* stg,
                          unsigned char* sxb, int* hs, int* flag, int* wsum) {
  const int nh = HW * HW * HW;
  const int per = (nh + SG - 1) / SG, i0 = gt * per;
  int cnt[8], gid[8];   // per <= 7 for n_sr <= 4 (nh <= 1728)
  int sum = 0, big = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = i0 + k;
    cnt[k] = 0;
    gid[k] = 0;
    if (k < per && i < nh) {
      gid[k] = halo_gid(i, n, HW, we);
      cnt[k] = count[gid[k]];
    }
    sum += cnt[k];
    big |= cnt[k] > cap;
  }
  int total;
  int run = group_scan_excl<SG>(gt, id, sum, wsum, &total);
  const bool fits = total <= cap;
  const bool single = group_sync_or(id, SG, big != 0);   // an element over the cap: no tiling
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = i0 + k;
    if (k < per && i < nh) {
      hs[i] = run;
      if (fits) {
        const int j0 = start[gid[k]];
        const unsigned char hx = (unsigned char)(i % HW);
        for (int q = 0; q < cnt[k]; ++q) {
          stg[run + q] = part[j0 + q];
          sxb[run + q] = hx;
        }
      }
    }
    run += cnt[k];
  }
  if (gt == 0) {
    hs[nh] = total;
    flag[0] = fits ? HALO_STAGED : (single ? HALO_GLOBAL : HALO_TILED);
  }
  group_sync(id, SG);
  return flag[0];
}

// One thread's part of a target's singular sums with the charges read from global
// memory (crowded elements): the rows r = q, q + tpt, ... of the block, element by
// element (a row may wrap around the periodic box), each row's terms summed in
// order in FP32, the row sums with compensation; element units.  Bound by the
// latency of the loads, so eight (potentials alone: twelve) are in flight; a function
// of its own, so that its registers are not shared out with the kernel's.  20 000
// charges in a blob of 16^3 elements, with forces and without: inline, one charge
// at a time, 65.2 and 41.8 ms, now 49.4 and 35.6 (four in flight 64.0 and 46.2).
template <bool GRAD>
__device__ __noinline__ float4 global_target(int q, int tpt, int n, int n_sr, const int* wx, const int* wy, const int* wz,
                                             int slot, const int* __restrict__ start, const int* __restrict__ count,
                                             const float4* __restrict__ part) {
  constexpr int NB = GRAD ? 8 : 12;
  Acc<float> ps, fx, fy, fz;
  const int nb = 2 * n_sr + 1, nrow = nb * nb;
  const float4 pt = part[slot];
  for (int r = q; r < nrow; r += tpt) {
    const int ay = r % nb, az = r / nb;
    const int64_t rowg = (int64_t)n * (wy[ay] + (int64_t)n * wz[az]);
    const float ddy = (float)(ay - n_sr), ddz = (float)(az - n_sr);
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    for (int ax = 0; ax < nb; ++ax) {
      const int64_t g = rowg + wx[ax];
      const float ddx = (float)(ax - n_sr);
      const int j0 = start[g], j1 = j0 + count[g];
      auto term = [&](const float4& p, int j) {
        const float rx = ddx + (p.x - pt.x), ry = ddy + (p.y - pt.y), rz = ddz + (p.z - pt.z);
        const float ir = j == slot ? 0.f : rsq<float>(fmaw(rx, rx, fmaw(ry, ry, rz * rz)));
        const float qi = p.w * ir;
        s0 += qi;
        if (GRAD) {
          const float f3 = qi * (ir * ir);
          s1 = fmaw(f3, rx, s1);
          s2 = fmaw(f3, ry, s2);
          s3 = fmaw(f3, rz, s3);
        }
      };
      int j = j0;
      for (; j + NB <= j1; j += NB) {
        float4 p[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) p[k] = part[j + k];
#pragma unroll
        for (int k = 0; k < NB; ++k) term(p[k], j + k);
      }
#pragma unroll 1
      for (; j < j1; ++j) term(part[j], j);
    }
    ps.add(s0);
    if (GRAD) {
      fx.add(s1);
      fy.add(s2);
      fz.add(s3);
    }
  }
  return make_float4(ps.get(), fx.get(), fy.get(), fz.get());
}

// Singular sums of every target charge in the brick, by SG threads (gt), four
// per target: each walks the rows r = q, q + 4, ... of its target's block (a
// row (dy, dz) is 2 n_sr + 1 consecutive halo elements, so its staged charges
// are one run), two charges per step, each row's terms summed in order in
// FP32 and the row sums added with compensation; a shuffle tree combines the
// four.  Staged tile by tile (a dense halo): the tiles are consecutive runs of
// halo elements whose charges fit; each target takes the part of each row
// inside the tile, and its tile sums are added in FP64 in tile order (into
// phi_s / E_s, element units, scaled at the last tile).  Global (an element
// over the staging area): the same rows read from global memory, element by
// element.  Writes phi_s and E_s (and half of them to psi, gpsi).
template <bool GRAD>
__device__ void singular_targets(int gt, int id, int mode, int n, int n_sr, float h, int E0x, int E0y, int E0z, int HW,
                                 int ntarget, const int* __restrict__ epre, const int* __restrict__ hs,
                                 const int* __restrict__ rtab, const int* __restrict__ we,
                                 float4* stg, unsigned char* sxb, int cap, const int* __restrict__ start,
                                 const int* __restrict__ count, const float4* __restrict__ part,
                                 double* __restrict__ phi_s, double* __restrict__ E_s, double* __restrict__ psi,
                                 double* __restrict__ gpsi) {
  constexpr int TPT = 4;
  const int nb = 2 * n_sr + 1, nrow = nb * nb, nh = HW * HW * HW;
  const int q = gt & (TPT - 1);
  const double ih = 1.0 / (double)h;   // the sums are in element units
  int ta = 0, tz = nh;                 // the tile: halo elements [ta, tz)
  for (int tile = 0;; ++tile) {
    int c0 = 0;                        // the tile's first charge slot
    if (mode == HALO_TILED) {
      // the longest run of elements from ta whose charges fit (every element does)
      int lo = ta + 1, hi = nh;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (hs[mid] - hs[ta] <= cap) lo = mid;
        else hi = mid - 1;
      }
      tz = lo;
      c0 = hs[ta];
      for (int i = ta + gt; i < tz; i += SG) {
        const int j0 = start[halo_gid(i, n, HW, we)], k0 = hs[i] - c0, cnt = hs[i + 1] - hs[i];
        const unsigned char hx = (unsigned char)(i % HW);
        for (int k = 0; k < cnt; ++k) {
          stg[k0 + k] = part[j0 + k];
          sxb[k0 + k] = hx;
        }
      }
      group_sync(id, SG);
    }
    const bool last = tz >= nh;
    for (int tb = 0; tb < ntarget; tb += SG / TPT) {
      const int k = tb + gt / TPT;
      const bool valid = k < ntarget;
      float v4[4] = {0.f, 0.f, 0.f, 0.f};
      int slot = 0;
      if (valid) {
        int lo = 0, hi2 = BE;                 // element of target k: epre[l] <= k < epre[l + 1]
        while (hi2 - lo > 1) {
          const int mid = (lo + hi2) >> 1;
          if (epre[mid] <= k) lo = mid;
          else hi2 = mid;
        }
        const int l = lo;
        const int lx = l % BX, ly = (l / BX) % BY, lz = l / (BX * BY);
        const int ex = E0x + lx, ey = E0y + ly, ez = E0z + lz;
        const int kk = k - epre[l];
        slot = start[ex + (int64_t)n * (ey + (int64_t)n * ez)] + kk;
        const int base = lx + HW * (ly + HW * lz);          // halo index of block offset (-n_sr, -n_sr, -n_sr)
        const int cx = lx + n_sr;                           // the target's halo x index
        Acc<float> ps, fx, fy, fz;
        if (mode != HALO_GLOBAL) {
          const int selfh = base + n_sr * (1 + HW + HW * HW);   // the target's own halo element
          const int self = hs[selfh] + kk - c0;
          const float4 pt = mode == HALO_STAGED ? stg[self] : part[slot];
          const float cxf = (float)cx;
          float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, ddy = 0.f, ddz = 0.f;
          int r = q, j = 0, je = 0;
          for (;;) {
            if (j >= je) {
              ps.add(s0);
              if (GRAD) {
                fx.add(s1);
                fy.add(s2);
                fz.add(s3);
              }
              s0 = s1 = s2 = s3 = 0.f;
              if (r >= nrow) break;
              const int rt = rtab[r];
              const int h0 = base + (rt & 0xFFFF);
              const int ha = h0 > ta ? h0 : ta, hb = h0 + nb < tz ? h0 + nb : tz;   // the row's part in the tile
              j = ha < hb ? hs[ha] - c0 : 0;
              je = ha < hb ? hs[hb] - c0 : 0;
              ddy = (float)(((rt >> 16) & 0xFF) - n_sr);
              ddz = (float)((rt >> 24) - n_sr);
              r += TPT;
              continue;
            }
            const bool two = j + 1 < je;
            const int jb = two ? j + 1 : j;
            const float4 pa = stg[j], pb = stg[jb];
            // element units (1/h applied once per target, in FP64), fused r^2 and sums
            const float rxa = ((float)sxb[j] - cxf) + (pa.x - pt.x), rya = ddy + (pa.y - pt.y), rza = ddz + (pa.z - pt.z);
            const float rxb = ((float)sxb[jb] - cxf) + (pb.x - pt.x), ryb = ddy + (pb.y - pt.y), rzb = ddz + (pb.z - pt.z);
            const float ira = j == self ? 0.f : rsq<float>(fmaw(rxa, rxa, fmaw(rya, rya, rza * rza)));
            const float irb = (!two || jb == self) ? 0.f : rsq<float>(fmaw(rxb, rxb, fmaw(ryb, ryb, rzb * rzb)));
            const float qa = pa.w * ira, qb = pb.w * irb;
            s0 += qa;
            s0 += qb;
            if (GRAD) {
              const float f3a = qa * (ira * ira), f3b = qb * (irb * irb);
              s1 = fmaw(f3a, rxa, s1);
              s2 = fmaw(f3a, rya, s2);
              s3 = fmaw(f3a, rza, s3);
              s1 = fmaw(f3b, rxb, s1);
              s2 = fmaw(f3b, ryb, s2);
              s3 = fmaw(f3b, rzb, s3);
            }
            j += 2;
          }
          v4[0] = ps.get();
          v4[1] = fx.get();
          v4[2] = fy.get();
          v4[3] = fz.get();
        } else {
          const float4 g = global_target<GRAD>(q, TPT, n, n_sr, we + lx, we + HW + ly, we + 2 * HW + lz, slot, start,
                                               count, part);
          v4[0] = g.x;
          v4[1] = g.y;
          v4[2] = g.z;
          v4[3] = g.w;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 1; o < TPT; o <<= 1) v4[i] += __shfl_xor_sync(0xffffffffu, v4[i], o);
      if (valid && q == 0) {
        // element units; tile sums added in FP64 in tile order, scaled at the last tile
        double sum[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) sum[a] = (double)v4[a];
        if (tile > 0) {
          sum[0] += phi_s[slot];
          if (GRAD)
#pragma unroll
            for (int a = 0; a < 3; ++a) sum[1 + a] += E_s[3 * slot + a];
        }
        if (last) {
          const double ps0 = sum[0] * ih;
          phi_s[slot] = ps0;
          if (psi) psi[slot] = 0.5 * ps0;
          if (GRAD) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              const double e = sum[1 + a] * (ih * ih);
              E_s[3 * slot + a] = e;
              if (gpsi) gpsi[3 * slot + a] = 0.5 * e;
            }
          }
        } else {
          phi_s[slot] = sum[0];
          if (GRAD)
#pragma unroll
            for (int a = 0; a < 3; ++a) E_s[3 * slot + a] = sum[1 + a];
        }
      }
    }
    if (last) break;
    group_sync(id, SG);   // the next tile overwrites the staging area
    ta = tz;
  }
}

// One CTA per brick of BX x BY x BZ elements: the screen field of every brick
// element at its 64 nodes (written to Gscr, brick-major) and the singular sums
// of every target charge in the brick (written to phi_s and E_s; with psi,
// half of them to psi and gpsi as well: the singular adjoint for the weights
// Q / 2 of the energy, whose kernel 1/r is symmetric).  TC: the
// contraction on the tensor cores (Hb holds the table's bf16
// pieces in the tiles' layout, err receives a bounded wait that gave up),
// 512 threads and eight per target; otherwise CUDA cores, 256 threads and
// four per target.
template <bool GRAD, bool TC>
__global__ void __launch_bounds__(TC ? PTC : PT, 2) k_pair_screen(int n, int n_sr, float h, const int* __restrict__ start,
                                                             const int* __restrict__ count,
                                                             const float4* __restrict__ part,
                                                             const float* __restrict__ Vc,
                                                             const uint4* __restrict__ Hb, const float2* __restrict__ H0,
                                                             const float2* __restrict__ Hdf, float* __restrict__ Gscr,
                                                             double* __restrict__ phi_s, double* __restrict__ E_s,
                                                             double* __restrict__ psi, double* __restrict__ gpsi,
                                                             int* __restrict__ err) {
  static_assert(PT == SG && PTC == 2 * SG, "the short-range sums take the whole CUDA-core CTA, half the tensor-core one");
  constexpr int NT = TC ? PTC : PT;
  typedef Pair3Smem<TC> SM;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nbx = (n + BX - 1) / BX, nby = (n + BY - 1) / BY;
  const int E0x = (blockIdx.x % nbx) * BX, E0y = ((blockIdx.x / nbx) % nby) * BY, E0z = (blockIdx.x / (nbx * nby)) * BZ;
  const int keep = n_sr + 1, noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  const int SW = 3 * BX + 2 * n_sr - 1, SF = BX + 2 * n_sr - 1, HW = BX + 2 * n_sr;
  const int nb = 2 * n_sr + 1, nrow = nb * nb;
  float *R, *A_c = nullptr, *H_c = nullptr;
  float4* stg;
  unsigned char* tiles = nullptr;
  int* hs;                                                // halo element prefix, HW^3 + 1
  unsigned char* sxb;                                     // STAGE_CAP: halo x index of each staged charge
  if (TC) {
    tiles = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // swizzle atoms on 1 KB
    R = (float*)(tiles + SM::TILES);
    stg = (float4*)((unsigned char*)R + SM::rbytes(n_sr));
    sxb = (unsigned char*)(stg + STAGE_CAP);
    hs = (int*)((unsigned char*)stg + SM::stgbytes());
  } else {
    const size_t r1 = SM::region1(n_sr);
    R = (float*)smem_raw;                                     // region 1: R, later the staged charges
    stg = (float4*)smem_raw;
    A_c = (float*)(smem_raw + r1);                            // [OCH][64] chunks of A and H (float pairs)
    H_c = (float*)((unsigned char*)A_c + OCH * 64 * SM::ES);
    hs = (int*)((unsigned char*)H_c + OCH * 64 * SM::ES);
  }
  int* epre = hs + HW * HW * HW + 1;                      // BE + 1
  int* flag = epre + BE + 1;
  int* wsum = flag + 1;                                   // NT/32 + 1 scan scratch
  int* otab = (int*)(((uintptr_t)(wsum + NT / 32 + 1) + 15) & ~(uintptr_t)15);   // R base index of each offset, in
  const int no3p = (no3 + 63) / 64 * 64;                  //   whole chunks of 64
  int* rtab = otab + no3p;                                // nb^2 rows (dy, dz): halo offset | ay << 16 | az << 24
  int* wv = rtab + nrow;                                  // 3 x SW wrapped vertex coords times 1, n, n^2
  int* we = wv + 3 * SW;                                  // 3 x HW wrapped halo element coords
  if (!TC) sxb = (unsigned char*)(we + 3 * HW + 32);
  uint64_t* mbar = (uint64_t*)(((uintptr_t)(we + 3 * HW) + 7) & ~(uintptr_t)7);   // TC only
  uint32_t* tslot = (uint32_t*)(mbar + 1);
  const int tid = threadIdx.x;
  int ntarget;
  {
    int c0 = 0;
    if (tid < BE) {
      const int lx = E0x + (tid % BX), ly = E0y + (tid / BX) % BY, lz = E0z + tid / (BX * BY);
      if (lx < n && ly < n && lz < n) c0 = count[lx + (int64_t)n * (ly + (int64_t)n * lz)];
    }
    const int pre = block_scan_excl<NT>(c0, wsum, &ntarget);
    if (tid < BE) epre[tid] = pre;
    if (tid == 0) epre[BE] = ntarget;
  }
  if (ntarget == 0) return;
  // index tables (no divisions in the hot loops below)
  const int RS = SM::RS(n_sr), PS = SM::PS(n_sr);
  for (int o = tid; o < no3p; o += NT) {
    const int ox = o % noff - keep, oy = (o / noff) % noff - keep, oz = o / (noff * noff) - keep;
    const int bx = ox == -keep ? SF : (ox == n_sr ? SF + BX : n_sr - 1 - ox);
    const int by = oy == -keep ? SF : (oy == n_sr ? SF + BX : n_sr - 1 - oy);
    const int bz = oz == -keep ? SF : (oz == n_sr ? SF + BX : n_sr - 1 - oz);
    otab[o] = o < no3 ? bx + RS * by + PS * bz : 0;
  }
  for (int r = tid; r < nrow; r += NT) rtab[r] = HW * ((r % nb) + HW * (r / nb)) | (r % nb) << 16 | (r / nb) << 24;
  {
    const int E0[3] = {E0x, E0y, E0z};
    for (int i = tid; i < 3 * SW; i += NT) {
      const int a = i / SW, sa = i % SW;
      int v;
      if (sa < SF) v = E0[a] + sa - (n_sr - 1);
      else if (sa < SF + BX) v = E0[a] + (sa - SF) + keep;
      else v = E0[a] + (sa - SF - BX) - n_sr;
      // the term of axis a in the index of the class sums Vc: its vertex coordinate and its class
      const int cls = sa < SF ? 0 : (sa < SF + BX ? 1 : 2);
      wv[i] = wrapn(v, n) * (a == 0 ? 1 : (a == 1 ? n : n * n)) + cls * (a == 0 ? 1 : (a == 1 ? 3 : 9)) * n * n * n;
    }
    for (int i = tid; i < 3 * HW; i += NT) {
      const int a = i / HW, ha = i % HW;
      we[i] = wrapn(E0[a] - n_sr + ha, n);
    }
  }
  __syncthreads();
  // (1) extended vertex field (unrolled: the gathers of several entries in flight); the
  // coordinates of entries i = tid + k NT advanced without divisions
  const int dsx = NT % SW, dsy = (NT / SW) % SW, dsz = NT / (SW * SW);
  int sx = tid % SW, sy = (tid / SW) % SW, sz = tid / (SW * SW);
#pragma unroll 4
  for (int i = tid; i < SW * SW * SW; i += NT) {
    const float val = Vc[wv[sx] + wv[SW + sy] + wv[2 * SW + sz]];   // class and vertex: < 27 n^3 < 2^31
    if constexpr (!TC) {
      // the hi + lo floats of the double-float contraction (an FP32 value has lo = 0)
      reinterpret_cast<float2*>(R)[i] = make_float2(val, 0.f);
    } else {
      R[sx + RS * sy + PS * sz] = val;
    }
    sx += dsx;
    sy += dsy;
    sz += dsz;
    if (sx >= SW) {
      sx -= SW;
      ++sy;
    }
    if (sy >= SW) {
      sy -= SW;
      ++sz;
    }
  }
  // (2) screen field and (3) singular sums
  if constexpr (TC) {
    // Tensor cores: two groups of eight warps run side by side.  Group A
    // (warps 0 .. 7: two of each TMEM lane quarter) computes the screen field:
    // for each chunk of 64 offsets, the three bf16 pieces of A (64 brick
    // elements x 64 offsets, built from R) and of H (64 nodes x 64 offsets,
    // precomputed) in shared memory; one thread issues the six piece products
    // per K step of 16 (M = 64, N = 64) into two TMEM accumulators (hi: the
    // product of the leading pieces, lo: the other five).  The hi accumulator
    // holds one chunk at a time and is added into registers after each chunk,
    // so that no accumulation inside the tensor core spans more than 64 terms
    // of the leading product; the chunk sums are added with compensation.  In
    // the FP32 path the table is relative to each element's corners (see
    // pair_relative_table), so these sums carry no large smooth part.  Group
    // B (warps 8 .. 15) stages the halo charges in a region of their own and
    // computes the singular sums meanwhile.
    const uint32_t tl = smem_u32(tiles);
    if (tid < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_u32(tslot)));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) mbar_init(smem_u32(mbar));
    tc_fence_before();
    __syncthreads();   // R complete; TMEM address and barrier visible
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const int warp = tid >> 5;
    bool failed = false;
    if (tid < SG) {
      const int gt = tid;
      // The field at node 0 (the one absolute column of the relative table,
      // the element's potential level) is summed on the CUDA cores from the A
      // values each thread splits anyway, with the table's hi + lo floats (H0)
      // in two FP32 sums rounded to nearest (the tensor cores' accumulation
      // would round it alike in every element, and U adds that up); four
      // partial sums per element, combined in the epilogue.
      __shared__ float2 s0p[(SG / 64) * BE];
      float s0h = 0.f, s0l = 0.f;
      const int l = gt & 63, g = gt >> 6;   // this thread's A units: row l, chunk offsets 8 g .. and 8 (g + 4) ..
      const int lam = (l % BX) + RS * ((l / BX) % BY) + PS * (l / (BX * BY));
      const uint32_t aoff[2] = {sw128_off(l, 8 * g), sw128_off(l, 8 * (g + 4))};
      const int nch = (no3 + 63) / 64;
      // this thread's accumulator entries (tmem_ld16x64b): register jj holds element row
      // 16 qq + (lane / 4) + 8 (lane mod 2), node column 32 hh + 2 jj + (lane / 2) mod 2
      const int qq = warp & 3, hh = warp >> 2, lane = tid & 31;
      const int arow = 16 * qq + (lane >> 2) + 8 * (lane & 1), acol = 32 * hh + ((lane >> 1) & 1);
      const uint32_t ta = tmem + ((uint32_t)(32 * qq) << 16) + 32 * hh;
      float hsum[16], hcmp[16];   // compensated chunk sums of the hi accumulator
#pragma unroll
      for (int jj = 0; jj < 16; ++jj) hsum[jj] = hcmp[jj] = 0.f;
      for (int c = 0; c < nch; ++c) {
        for (int i = gt; i < 1536; i += SG) cp_async16(tl + 24576 + 16 * i, Hb + (size_t)c * 1536 + i);
        asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t p0[4], p1[4], p2[4];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int o = 64 * c + 8 * (g + 4 * hf) + 2 * jj;
            // (past the last offset any finite value does: the table is zero there)
            const int2 ot = *reinterpret_cast<const int2*>(otab + o);
            const float xa = R[ot.x + lam], xb = R[ot.y + lam];
            bf16_split2(xa, xb, p0[jj], p1[jj], p2[jj]);
            if (o + 1 < no3) {
              const float4 h2 = *reinterpret_cast<const float4*>(H0 + o);   // H0[o], H0[o + 1]
              s0h = fmaf(xa, h2.x, fmaf(xb, h2.z, s0h));
              s0l = fmaf(xa, h2.y, fmaf(xb, h2.w, s0l));
            }
          }
          sts128(tl + aoff[hf], p0);
          sts128(tl + 8192 + aoff[hf], p1);
          sts128(tl + 16384 + aoff[hf], p2);
        }
        cp_async_wait_all();
        fence_async_smem();
        group_sync(1, SG);
        if (gt == 0) {
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint32_t a = tl + 32 * kk, b = tl + 24576 + 32 * kk;
            const uint32_t acc = (c > 0 || kk > 0) ? 1u : 0u;
            umma_bf16(tmem, umma_desc(a), umma_desc(b), UMMA_IDESC, kk > 0 ? 1u : 0u);         // a0 b0
            umma_bf16(tmem + 64, umma_desc(a), umma_desc(b + 8192), UMMA_IDESC, acc);          // a0 b1
            umma_bf16(tmem + 64, umma_desc(a + 8192), umma_desc(b), UMMA_IDESC, 1u);           // a1 b0
            umma_bf16(tmem + 64, umma_desc(a), umma_desc(b + 16384), UMMA_IDESC, 1u);          // a0 b2
            umma_bf16(tmem + 64, umma_desc(a + 8192), umma_desc(b + 8192), UMMA_IDESC, 1u);   // a1 b1
            umma_bf16(tmem + 64, umma_desc(a + 16384), umma_desc(b), UMMA_IDESC, 1u);          // a2 b0
          }
          umma_commit(smem_u32(mbar));
        }
        // one warp polls the barrier; the group waits at its named barrier
        const bool done = warp == 0 ? mbar_wait(smem_u32(mbar), (uint32_t)(c & 1)) : true;
        if (group_sync_or(1, SG, !done)) {
          failed = true;
          break;
        }
        tc_fence_after();
        uint32_t vh[16];
        tmem_ld16x64b(ta, vh);
        tmem_wait_ld();
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
          const float y = __uint_as_float(vh[jj]) - hcmp[jj], t = hsum[jj] + y;
          hcmp[jj] = (t - hsum[jj]) - y;
          hsum[jj] = t;
        }
        tc_fence_before();   // the next chunk's MMAs overwrite hi after the next barrier
      }
      if (failed) {
        if (gt == 0) atomicExch(err, 1);
        // a last bounded wait on both phases for MMAs still in flight, and for the table copy
        (void)mbar_wait(smem_u32(mbar), 0u);
        (void)mbar_wait(smem_u32(mbar), 1u);
        cp_async_wait_all();
      }
      s0p[g * BE + l] = make_float2(s0h, s0l);
      group_sync(1, SG);
      tc_fence_after();
      if (!failed) {
        uint32_t vl[16];
        tmem_ld16x64b(ta + 64, vl);
        tmem_wait_ld();
        float* drow = (float*)Gscr + (int64_t)blockIdx.x * (BE * 64) + arow * 64 + acol;
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) drow[2 * jj] = (hsum[jj] - hcmp[jj]) + __uint_as_float(vl[jj]);
        if (acol == 0) {   // column 0 from the CUDA-core sums
          double sum = 0.0;
#pragma unroll
          for (int q = 0; q < SG / 64; ++q) {
            const float2 v = s0p[q * BE + arow];
            sum += (double)v.x + (double)v.y;
          }
          drow[0] = (float)sum;
        }
      }
      tc_fence_before();
    } else {
      const int gt = tid - SG;
      const int mode = stage_halo(gt, 2, n, HW, we, start, count, part, STAGE_CAP, stg, sxb, hs, flag, wsum);
      singular_targets<GRAD>(gt, 2, mode, n, n_sr, h, E0x, E0y, E0z, HW, ntarget, epre, hs, rtab, we, stg, sxb,
                                STAGE_CAP, start, count, part, phi_s, E_s, psi, gpsi);
    }
    __syncthreads();   // every TMEM read done
    if (tid < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem));
  } else {
    // CUDA cores: 4 x 4 register tile, per-chunk partial sums added into a
    // total, in double-float arithmetic on the FP32 pipes (FP64 issues at a
    // small fraction of the FP32 rate here): A and H are staged as hi + lo float pairs (the table's from FP64; an FP32 A has lo =
    // 0), each product keeps its exact leading part (fused two-product) and the
    // two cross terms, and the products are summed by two-sum into a hi + lo
    // accumulator; each chunk's sum goes into an FP64 total, which keeps the
    // relative error near 2^-48 of the chunk's sum of |A H| instead of growing
    // over all offsets.  The FP32 path's result is then rounded to FP32.
    const int eb = tid >> 4, mb = tid & 15;
    // this thread stages entries i = tid + k PT: element l = i & 63 is fixed per thread
    const int lst = tid & 63;
    const int lam = (lst % BX) + SW * (((lst / BX) % BY) + SW * (lst / (BX * BY)));
    constexpr int SPT = OCH * 64 / PT;   // staged entries per thread per chunk
    float* gb = Gscr + (int64_t)blockIdx.x * (BE * 64);
    {
      // the table's hi + lo floats come precomputed (Hdf); R was split in (1)
      float2 hpf[SPT];                   // next chunk's table values, fetched during this chunk
#pragma unroll
      for (int k = 0; k < SPT; ++k) {
        const int i = tid + k * PT, o = i >> 6;
        hpf[k] = o < no3 ? Hdf[(int64_t)o * 64 + (i & 63)] : make_float2(0.f, 0.f);
      }
      const float2* R2 = reinterpret_cast<const float2*>(R);
      float sh[4][4], sl[4][4];
      double tot[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) tot[i][j] = 0.0;
      float2* A2 = reinterpret_cast<float2*>(A_c);
      float2* H2 = reinterpret_cast<float2*>(H_c);
      for (int o0 = 0; o0 < no3; o0 += OCH) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < SPT; ++k) {
          const int i = tid + k * PT;
          const int o = o0 + (i >> 6);
          H2[i] = hpf[k];
          A2[i] = o < no3 ? R2[otab[o] + lam] : make_float2(0.f, 0.f);
        }
        __syncthreads();
        if (o0 + OCH < no3) {
#pragma unroll
          for (int k = 0; k < SPT; ++k) {
            const int i = tid + k * PT, o = o0 + OCH + (i >> 6);
            hpf[k] = o < no3 ? Hdf[(int64_t)o * 64 + (i & 63)] : make_float2(0.f, 0.f);
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) sh[i][j] = sl[i][j] = 0.f;
#pragma unroll 2
        for (int oi = 0; oi < OCH; ++oi) {
          const float4* ap = reinterpret_cast<const float4*>(A2 + oi * 64 + 4 * eb);
          const float4* hp = reinterpret_cast<const float4*>(H2 + oi * 64 + 4 * mb);
          const float4 a01 = ap[0], a23 = ap[1], h01 = hp[0], h23 = hp[1];
          const float ah[4] = {a01.x, a01.z, a23.x, a23.z}, al[4] = {a01.y, a01.w, a23.y, a23.w};
          const float hh[4] = {h01.x, h01.z, h23.x, h23.z}, hl[4] = {h01.y, h01.w, h23.y, h23.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float p = ah[i] * hh[j];
              float e = fmaf(ah[i], hh[j], -p);
              e = fmaf(ah[i], hl[j], e);
              e = fmaf(al[i], hh[j], e);
              const float t = sh[i][j] + p, z = t - sh[i][j];
              sl[i][j] += ((sh[i][j] - (t - z)) + (p - z)) + e;
              sh[i][j] = t;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) tot[i][j] += (double)sh[i][j] + (double)sl[i][j];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float4 v;
        v.x = (float)tot[i][0];
        v.y = (float)tot[i][1];
        v.z = (float)tot[i][2];
        v.w = (float)tot[i][3];
        *reinterpret_cast<float4*>(gb + (4 * eb + i) * 64 + 4 * mb) = v;
      }
    }
    // Region 1 (R) was last read before the chunk loop's final barrier, so the
    // staging may overwrite it without another one.
    const int mode = stage_halo(tid, 0, n, HW, we, start, count, part, STAGE_CAP, stg, sxb, hs, flag, wsum);
    singular_targets<GRAD>(tid, 0, mode, n, n_sr, h, E0x, E0y, E0z, HW, ntarget, epre, hs, rtab, we, stg, sxb,
                              STAGE_CAP, start, count, part, phi_s, E_s, psi, gpsi);
  }
}

// The screen field in an FP64 context.  The table is symmetric under reflection
// of each axis about the element's centre, H(noff - 1 - o, 3 - m) = H(o, m), so
// with the even and odd parts of the amplitudes and of the field along each axis
//   A+-(i) = A(i) +- A(noff - 1 - i),  S(j) = S+(j) + S-(j),  S(3 - j) = S+(j) - S-(j)
// the contraction falls into eight products (parities s = sx + 2 sy + 4 sz) of
// (n_sr + 1)^3 amplitudes with two nodes per axis: an eighth of the
// multiply-adds.  They run in float pairs on the FP32 pipes, 32 offsets at a
// time in pairs and across those in three floats (relative to sum |A H| about
// 1e-15).  One CTA per brick and parities (sy, sz), so that small meshes fill
// the GPU too; it forms both parities along x.  As in k_pair_screen the brick's
// extended vertex field R is in shared memory and A(e, o) = R[otab(o) +
// lambda(e)]; R comes as pairs, times a power of two (fep3m_ctx::q_scale).
// Gscr[brick][element][8 s + jx + 2 jy + 4 jz].  Bound by FP32 issue (about 105
// operations per pair of parts staged, 12 per multiply-add).  Rock salt 32^3:
// screen and singular sums took 2080 us in one kernel (the whole contraction in
// pairs, FP64 singular terms); now 164 us here and 165 us in k_singular64.
constexpr int SK = 32;   // offsets staged at once
// row stride of R: 4 modulo 16 pairs, so that the four rows of four elements a
// half-warp reads fall on different banks (even: the operands after R stay aligned)
__host__ __device__ constexpr int screen64_row(int sw) { return sw + (20 - sw % 16) % 16; }
static size_t screen64_smem(int n_sr) {
  const int sw = 3 * BX + 2 * n_sr - 1, kh = n_sr + 1, K = kh * kh * kh;
  return ((size_t)screen64_row(sw) * sw * sw + 2 * SK * (BE + 2) + 2 * K * 8) * sizeof(df) + (size_t)K * 8 * sizeof(int);
}
__global__ void __launch_bounds__(PT, 2) k_screen64(int n, int n_sr, const int* __restrict__ count,
                                                    const df* __restrict__ Vc, const df* __restrict__ HP, double inv_scale,
                                                    double* __restrict__ Gscr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nbx = (n + BX - 1) / BX, nby = (n + BY - 1) / BY;
  const int E0[3] = {(int)(blockIdx.x % nbx) * BX, (int)((blockIdx.x / nbx) % nby) * BY,
                     (int)(blockIdx.x / (nbx * nby)) * BZ};
  const int sy = blockIdx.y & 1, sz = blockIdx.y >> 1;
  const int kh = n_sr + 1, noff = 2 * kh, K = kh * kh * kh;
  const int SW = 3 * BX + 2 * n_sr - 1, SF = BX + 2 * n_sr - 1, SW3 = SW * SW * SW;
  const int RS = screen64_row(SW);
  df* R = reinterpret_cast<df*>(smem_raw);
  df(*As)[SK][BE + 2] = reinterpret_cast<df(*)[SK][BE + 2]>(R + RS * SW * SW);   // [2]: parity along x
  df* Hs = reinterpret_cast<df*>(As + 2);                                            // [2][K][8]
  int* otab = reinterpret_cast<int*>(Hs + 2 * K * 8);                                // [K][8] mirror images of an offset
  __shared__ int wv[3][3 * BX + 8];
  const int tid = threadIdx.x;
  bool any = false;
  if (tid < BE) {
    const int lx = E0[0] + tid % BX, ly = E0[1] + (tid / BX) % BY, lz = E0[2] + tid / (BX * BY);
    any = lx < n && ly < n && lz < n && count[lx + (int64_t)n * (ly + (int64_t)n * lz)] != 0;
  }
  if (!__syncthreads_or(any)) return;
  auto slot = [&](int o) {   // R's slot of offset index o (0 .. noff - 1) of an axis
    return o == 0 ? SF : (o == noff - 1 ? SF + BX : 2 * n_sr - o);
  };
  for (int i = tid; i < 3 * SW; i += PT) {
    const int a = i / SW, sa = i % SW;
    const int v = sa < SF ? E0[a] + sa - (n_sr - 1) : (sa < SF + BX ? E0[a] + (sa - SF) + kh : E0[a] + (sa - SF - BX) - n_sr);
    // the term of axis a in the index of the class sums Vc: its vertex coordinate and its class
    const int cls = sa < SF ? 0 : (sa < SF + BX ? 1 : 2);
    wv[a][sa] = wrapn(v, n) * (a == 0 ? 1 : (a == 1 ? n : n * n)) + cls * (a == 0 ? 1 : (a == 1 ? 3 : 9)) * n * n * n;
  }
  for (int i = tid; i < 8 * K; i += PT) {
    const int k = i >> 3, f = i & 7, kk[3] = {k % kh, (k / kh) % kh, k / (kh * kh)};
    int idx = 0;
    for (int a = 2; a >= 0; --a)
      idx += slot((f >> a) & 1 ? noff - 1 - kk[a] : kk[a]) * (a == 0 ? 1 : (a == 1 ? RS : RS * SW));
    otab[i] = idx;
  }
  for (int i = tid; i < 2 * K * 8; i += PT) Hs[i] = HP[(int64_t)(2 * sy + 4 * sz) * K * 8 + i];   // sx = 0, 1 follow
  __syncthreads();
#pragma unroll 4
  for (int i = tid; i < SW3; i += PT) {
    const int r = i / SW, x = i - r * SW, z = r / SW, y = r - z * SW;
    R[x + RS * r] = Vc[wv[0][x] + wv[1][y] + wv[2][z]];
  }
  const int el = tid & 63, k4 = tid >> 6;   // staging: this thread's element, and every fourth offset
  const int lam = (el % BX) + RS * (((el / BX) % BY) + SW * (el / (BX * BY)));
  const int m = tid & 7, g = (tid >> 3) & 15, sx = tid >> 7;   // product: node part, four elements, parity along x
  tf tot[4] = {};
  for (int k0 = 0; k0 < K; k0 += SK) {
    const int nk = min(SK, K - k0);
    __syncthreads();
#pragma unroll 2
    for (int kk = k4; kk < nk; kk += 4) {
      const int* o = otab + 8 * (k0 + kk);
      df t[2];
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const df a0 = R[o[f] + lam], a1 = R[o[f + 2] + lam], b0 = R[o[f + 4] + lam], b1 = R[o[f + 6] + lam];
        const df a = df_add(a0, sy ? df{-a1.h, -a1.l} : a1), b = df_add(b0, sy ? df{-b1.h, -b1.l} : b1);
        t[f] = df_add(a, sz ? df{-b.h, -b.l} : b);
      }
      As[0][kk][el] = df_add(t[0], t[1]);
      As[1][kk][el] = df_add(t[0], df{-t[1].h, -t[1].l});
    }
    __syncthreads();
    df acc[4] = {};
    const df* Hm = Hs + (int64_t)sx * K * 8 + (int64_t)k0 * 8 + m;
#pragma unroll 4
    for (int kk = 0; kk < nk; ++kk) {
      const df h = Hm[8 * kk];
      const float4* ap = reinterpret_cast<const float4*>(&As[sx][kk][4 * g]);
      const float4 v0 = ap[0], v1 = ap[1];
      df_fma(acc[0], df{v0.x, v0.y}, h);
      df_fma(acc[1], df{v0.z, v0.w}, h);
      df_fma(acc[2], df{v1.x, v1.y}, h);
      df_fma(acc[3], df{v1.z, v1.w}, h);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) tf_add(tot[j], acc[j]);
  }
  double* gb = Gscr + (int64_t)blockIdx.x * (BE * 64) + 8 * (sx + 2 * sy + 4 * sz) + m;
#pragma unroll
  for (int j = 0; j < 4; ++j) gb[(4 * g + j) * 64] = df_value(tot[j]) * inv_scale;
}

// One CTA per brick, after the mesh solve: G = mesh potential - screen field
// at the 64 nodes of each non-empty brick element, then four threads per
// target charge each contract 16 of the nodes with the order-3 shape
// functions (and their derivatives) at the charge; the mesh part is added to
// the singular part the screen kernel left in phi_s / E_s (FP64 contexts:
// k_pair_eval64).
//
// The screen field arrives relative to the element's corners (the
// field at node 0, corner fields relative to it, elsewhere the field less its
// trilinear interpolant; pair_relative_table), and G is split the same way:
// G0 and the corner values of G - G0 in FP64 (the mesh potential's hi + lo
// float pair added in FP64), and the remainder G - G0 - trilinear(corners) in
// FP32 (from the same pairs).  The trilinear part and its gradient at the
// charge are evaluated in FP64; only the small remainder goes through the FP32
// contraction.
template <bool GRAD>
__global__ void __launch_bounds__(PT) k_pair_eval(int n, int Nm, float inv_h, const int* __restrict__ start,
                                                  const int* __restrict__ count, const float4* __restrict__ part,
                                                  const float2* __restrict__ phi_hl, const float* __restrict__ Gscr,
                                                  const int* __restrict__ perm, double* __restrict__ phi_s,
                                                  double* __restrict__ E_s, double* __restrict__ phi_out) {
  typedef float T;
  typedef float4 V4;
  __shared__ __align__(32) T G[BE * 64];
  __shared__ double G0[BE];
  __shared__ double Gc[BE * 8];   // corner values of G - G0
  __shared__ int epre[BE + 1];
  __shared__ int wsum[PT / 32 + 1];
  const int nbx = (n + BX - 1) / BX, nby = (n + BY - 1) / BY;
  const int E0x = (blockIdx.x % nbx) * BX, E0y = ((blockIdx.x / nbx) % nby) * BY, E0z = (blockIdx.x / (nbx * nby)) * BZ;
  const int tid = threadIdx.x;
  int ntarget;
  {
    int c0 = 0;
    if (tid < BE) {
      const int lx = E0x + (tid % BX), ly = E0y + (tid / BX) % BY, lz = E0z + tid / (BX * BY);
      if (lx < n && ly < n && lz < n) c0 = count[lx + (int64_t)n * (ly + (int64_t)n * lz)];
    }
    const int pre = block_scan_excl<PT>(c0, wsum, &ntarget);
    if (tid < BE) epre[tid] = pre;
    if (tid == 0) epre[BE] = ntarget;
  }
  if (ntarget == 0) return;
  __syncthreads();
  const T* gb = Gscr + (int64_t)blockIdx.x * (BE * 64);
  const int N = Nm;
  // mesh node of node m of brick element l: on the periodic mesh (Nm = 3n
  // nodes per axis) wrapped, on a box's (Nm = 3 nb + 1, targets in the first
  // nb elements) never past the last node
  auto node = [&](int l, int m) -> int64_t {
    const int ex = E0x + l % BX, ey = E0y + (l / BX) % BY, ez = E0z + l / (BX * BY);
    const int gx = 3 * ex + (m & 3), gy = 3 * ey + ((m >> 2) & 3), gz = 3 * ez + (m >> 4);   // < 3n + 3
    return (gx >= N ? gx - N : gx) + (int64_t)N * ((gy >= N ? gy - N : gy) + (int64_t)N * (gz >= N ? gz - N : gz));
  };
  auto phd = [&](int64_t k) -> double {
    const float2 p = phi_hl[k];
    return (double)p.x + (double)p.y;
  };
  if (tid < BE && epre[tid + 1] != epre[tid]) {
    const double p00 = phd(node(tid, 0));
    G0[tid] = p00 - (double)gb[tid * 64];
    Gc[tid * 8] = 0.0;
#pragma unroll
    for (int c = 1; c < 8; ++c) {
      const int mc = 3 * (c & 1) + 12 * ((c >> 1) & 1) + 48 * (c >> 2);
      Gc[tid * 8 + c] = (phd(node(tid, mc)) - p00) - (double)gb[tid * 64 + mc];
    }
  }
  // node differences of the mesh potential from its hi + lo floats
  for (int i = tid; i < BE * 64; i += PT) {
    const int l = i >> 6, m = i & 63;
    if (epre[l + 1] == epre[l]) continue;   // empty (or outside the mesh): never read
    const float2 p = phi_hl[node(l, m)], p0 = phi_hl[node(l, 0)];
    G[i] = (p.x - p0.x) + (p.y - p0.y);
  }
  __syncthreads();
  // remainder: the difference less its trilinear interpolant, less the screen
  // remainder; zero at the corners
  constexpr int PER = BE * 64 / PT;
  float rem[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = tid + k * PT, l = i >> 6, m = i & 63;
    const int mx = m & 3, my = (m >> 2) & 3, mz = m >> 4;
    rem[k] = 0.f;
    if (epre[l + 1] == epre[l]) continue;
    if ((mx == 0 || mx == 3) && (my == 0 || my == 3) && (mz == 0 || mz == 3)) continue;
    const float* g = G + l * 64;
    const float tx = mx * (1.f / 3.f), ty = my * (1.f / 3.f), tz = mz * (1.f / 3.f);
    // corners (0,0,0) 0, (3,0,0) 3, (0,3,0) 12, (3,3,0) 15, z + 48
    const float x00 = fmaf(tx, g[3] - g[0], g[0]), x10 = fmaf(tx, g[15] - g[12], g[12]);
    const float x01 = fmaf(tx, g[51] - g[48], g[48]), x11 = fmaf(tx, g[63] - g[60], g[60]);
    const float y0 = fmaf(ty, x10 - x00, x00), y1 = fmaf(ty, x11 - x01, x01);
    rem[k] = (g[m] - fmaf(tz, y1 - y0, y0)) - gb[i];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PER; ++k) G[tid + k * PT] = rem[k];
  __syncthreads();
  const int q = tid & 3;   // nodes 16 q .. 16 q + 15: mz = q, (mx, my) over 4 x 4
  for (int tb = 0; tb < ntarget; tb += PT / 4) {
    const int k = tb + (tid >> 2);
    const bool valid = k < ntarget;
    T v4[4] = {T(0), T(0), T(0), T(0)};
    int slot = 0, l = 0;
    V4 pt;
    pt.x = pt.y = pt.z = pt.w = T(0);
    if (valid) {
      int lo = 0, hi2 = BE;
      while (hi2 - lo > 1) {
        const int mid = (lo + hi2) >> 1;
        if (epre[mid] <= k) lo = mid;
        else hi2 = mid;
      }
      l = lo;
      const int ex = E0x + l % BX, ey = E0y + (l / BX) % BY, ez = E0z + l / (BX * BY);
      slot = start[ex + (int64_t)n * (ey + (int64_t)n * ez)] + (k - epre[l]);
      pt = part[slot];
      T ux[4], uy[4], uz[4], dx4[4], dy4[4], dz4[4];
      q3_values<T>(pt.x, ux);
      q3_values<T>(pt.y, uy);
      q3_values<T>(pt.z, uz);
      if (GRAD) {
        q3_derivs<T>(pt.x, dx4);
        q3_derivs<T>(pt.y, dy4);
        q3_derivs<T>(pt.z, dz4);
      }
#pragma unroll
      for (int my = 0; my < 4; ++my) {
        const V4 gv = *reinterpret_cast<const V4*>(G + l * 64 + 16 * q + 4 * my);
        const T g4[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
        for (int mx = 0; mx < 4; ++mx) {
          const T g = g4[mx];
          const T wyz = uy[my] * uz[q];
          v4[0] += g * ux[mx] * wyz;
          if (GRAD) {
            v4[1] += g * dx4[mx] * wyz;
            v4[2] += g * ux[mx] * dy4[my] * uz[q];
            v4[3] += g * ux[mx] * uy[my] * dz4[q];
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v4[i] += __shfl_xor_sync(0xffffffffu, v4[i], 1);
      v4[i] += __shfl_xor_sync(0xffffffffu, v4[i], 2);
    }
    // The trilinear part of G - G0 and its gradient at the charge, in FP64: thread q takes the
    // corner pair q (cy + 2 cz) along x, the pairs meet along y, then z, by shuffles, and thread q
    // finishes sum q (an FP64 instruction takes its pipe for the whole warp, however few lanes are on)
    const double* g = Gc + l * 8;
    const double y = pt.y, z = pt.z;
    const double b = g[2 * q + 1] - g[2 * q], a = fma((double)pt.x, b, g[2 * q]);
    const double ao = __shfl_xor_sync(0xffffffffu, a, 1), bo = __shfl_xor_sync(0xffffffffu, b, 1);
    const bool q1 = q & 1, q2 = q & 2;
    const double a0 = q1 ? ao : a, b0 = q1 ? bo : b;
    const double ay = (q1 ? a : ao) - a0, A = fma(y, ay, a0), B = fma(y, (q1 ? b : bo) - b0, b0);
    const double Ao = __shfl_xor_sync(0xffffffffu, A, 2);
    const double A0 = q2 ? Ao : A, az = (q2 ? A : Ao) - A0;
    double t;   // sum q's trilinear part: the value, d/dx, d/dy, d/dz
    if (GRAD) {
      const double Bo = __shfl_xor_sync(0xffffffffu, B, 2), yo = __shfl_xor_sync(0xffffffffu, ay, 2);
      // value, d/dx, d/dy at z are lerps of their values on the two z faces
      const double lo = q == 0 ? A0 : (q == 1 ? (q2 ? Bo : B) : (q2 ? yo : ay));
      const double hi = q == 0 ? A0 + az : (q == 1 ? (q2 ? B : Bo) : (q2 ? ay : yo));
      t = q == 3 ? az : fma(z, q == 0 ? az : hi - lo, lo);
    } else {
      t = fma(z, az, A0);
    }
    if (valid && (GRAD || q == 0)) {
      const double v = (double)(q == 0 ? v4[0] : (q == 1 ? v4[1] : (q == 2 ? v4[2] : v4[3]))) + t;
      if (q == 0) {
        const double phi = (v + G0[l]) * (double)inv_h + phi_s[slot];
        phi_s[slot] = phi;
        if (phi_out) phi_out[perm[slot]] = phi;
      } else {
        double* E = E_s + 3 * slot + (q - 1);
        *E = v * ((double)inv_h * (double)inv_h) + *E;
      }
    }
  }
}

// The same in an FP64 context.  The screen field comes in its even and odd
// parts (k_screen64); its nodal values are formed in shared memory, three
// sums and differences each, and subtracted from the mesh potential.  They are held
// relative to node 0's (G0): the shape functions sum to one and their gradients to
// zero, so an element's level enters the potential alone and the rounding acts on
// the variation only (charges of one sign give a level of hundreds).  Four
// threads per target take the four z layers of nodes: each evaluates one shape
// function and derivative per axis (shared by shuffles) and contracts its
// layer along x, then y: about 400 FP64 operations per target where the terms
// one by one took 3000 (rock salt 32^3 with forces: 98 -> 79 us; an FP64
// operation costs as much as 64 FP32 ones here).
__device__ __forceinline__ void q3_one(double t, int i, double& v, double& d) {
  const double k = i == 0 ? -4.5 : (i == 1 ? 13.5 : (i == 2 ? -13.5 : 4.5));
  const double r0 = i == 0 ? 1.0 / 3.0 : 0.0, r1 = i < 2 ? 2.0 / 3.0 : 1.0 / 3.0, r2 = i == 3 ? 2.0 / 3.0 : 1.0;
  const double a = t - r0, b = t - r1, c = t - r2, ab = a * b;
  v = k * (ab * c);
  d = k * fma(c, a + b, ab);
}
template <bool GRAD>
__global__ void __launch_bounds__(PT) k_pair_eval64(int n, int Nm, double inv_h, const int* __restrict__ start,
                                                    const int* __restrict__ count,
                                                    const vec4<double>::type* __restrict__ part,
                                                    const double* __restrict__ phi64, const double* __restrict__ Gscr,
                                                    const int* __restrict__ perm, double* __restrict__ phi_s,
                                                    double* __restrict__ E_s, double* __restrict__ phi_out) {
  typedef vec4<double>::type V4;
  __shared__ __align__(32) double G[BE * 64];
  __shared__ double G0[BE];
  __shared__ int epre[BE + 1];
  __shared__ int wsum[PT / 32 + 1];
  const int nbx = (n + BX - 1) / BX, nby = (n + BY - 1) / BY;
  const int E0x = (blockIdx.x % nbx) * BX, E0y = ((blockIdx.x / nbx) % nby) * BY, E0z = (blockIdx.x / (nbx * nby)) * BZ;
  const int tid = threadIdx.x;
  int ntarget;
  {
    int c0 = 0;
    if (tid < BE) {
      const int lx = E0x + (tid % BX), ly = E0y + (tid / BX) % BY, lz = E0z + tid / (BX * BY);
      if (lx < n && ly < n && lz < n) c0 = count[lx + (int64_t)n * (ly + (int64_t)n * lz)];
    }
    const int pre = block_scan_excl<PT>(c0, wsum, &ntarget);
    if (tid < BE) epre[tid] = pre;
    if (tid == 0) epre[BE] = ntarget;
  }
  if (ntarget == 0) return;
  __syncthreads();
  const double* gb = Gscr + (int64_t)blockIdx.x * (BE * 64);
  constexpr int PER = BE * 64 / PT;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = tid + k * PT;
    G[i] = epre[(i >> 6) + 1] != epre[i >> 6] ? gb[i] : 0.0;
  }
  // part i = jx + 2 jy + 4 jz + 8 (sx + 2 sy + 4 sz): along each axis the even
  // part's place takes their sum (node j), the odd part's the difference (node 3 - j)
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER / 2; ++k) {
      const int i = tid + k * PT, bit = 8 << a;
      const int e = ((i & ~(bit - 1)) << 1) | (i & (bit - 1));   // bit 3 + a clear
      if (epre[(e >> 6) + 1] == epre[e >> 6]) continue;
      const double x = G[e], y = G[e | bit];
      G[e] = x + y;
      G[e | bit] = x - y;
    }
  }
  __syncthreads();
  double val[PER];
  int at[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int i = tid + k * PT, l = i >> 6;
    int m[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int j = (i >> a) & 1;
      m[a] = (i >> (3 + a)) & 1 ? 3 - j : j;
    }
    at[k] = l * 64 + m[0] + 4 * m[1] + 16 * m[2];
    val[k] = 0.0;
    if (epre[l + 1] == epre[l]) continue;   // empty (or outside the mesh): never read
    // the node on the periodic mesh (Nm = 3 n) wrapped, on a box's (Nm = 3 nb + 1) never past the last
    const int gx = 3 * (E0x + l % BX) + m[0], gy = 3 * (E0y + (l / BX) % BY) + m[1], gz = 3 * (E0z + l / (BX * BY)) + m[2];
    val[k] = phi64[(gx >= Nm ? gx - Nm : gx) +
                   (int64_t)Nm * ((gy >= Nm ? gy - Nm : gy) + (int64_t)Nm * (gz >= Nm ? gz - Nm : gz))] - G[i];
    if ((at[k] & 63) == 0) G0[l] = val[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PER; ++k) G[at[k]] = val[k] - G0[at[k] >> 6];
  __syncthreads();
  const int q = tid & 3, lane0 = (tid & 31) & ~3;
  for (int tb = 0; tb < ntarget; tb += PT / 4) {
    const int k = tb + (tid >> 2);
    const bool valid = k < ntarget;
    int slot = 0, l = 0;
    V4 pt;
    pt.x = pt.y = pt.z = pt.w = 0.0;
    if (valid) {
      int lo = 0, hi2 = BE;
      while (hi2 - lo > 1) {
        const int mid = (lo + hi2) >> 1;
        if (epre[mid] <= k) lo = mid;
        else hi2 = mid;
      }
      l = lo;
      const int ex = E0x + l % BX, ey = E0y + (l / BX) % BY, ez = E0z + l / (BX * BY);
      slot = start[ex + (int64_t)n * (ey + (int64_t)n * ez)] + (k - epre[l]);
      pt = part[slot];
    }
    double ux, uy, uz, dx, dy, dz;
    q3_one(pt.x, q, ux, dx);
    q3_one(pt.y, q, uy, dy);
    q3_one(pt.z, q, uz, dz);
    double X[4], DX[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      X[i] = __shfl_sync(0xffffffffu, ux, lane0 + i);
      if (GRAD) DX[i] = __shfl_sync(0xffffffffu, dx, lane0 + i);
    }
    double v = 0.0, vx = 0.0, vy = 0.0;   // this layer: value, d/dx, d/dy
#pragma unroll
    for (int my = 0; my < 4; ++my) {
      const V4 gv = *reinterpret_cast<const V4*>(G + l * 64 + 16 * q + 4 * my);
      const double Y = __shfl_sync(0xffffffffu, uy, lane0 + my);
      const double row = fma(gv.x, X[0], fma(gv.y, X[1], fma(gv.z, X[2], gv.w * X[3])));
      v = fma(row, Y, v);
      if (GRAD) {
        const double DY = __shfl_sync(0xffffffffu, dy, lane0 + my);
        vx = fma(fma(gv.x, DX[0], fma(gv.y, DX[1], fma(gv.z, DX[2], gv.w * DX[3]))), Y, vx);
        vy = fma(row, DY, vy);
      }
    }
    double v4[4] = {v * uz, vx * uz, vy * uz, v * dz};
#pragma unroll
    for (int i = 0; i < (GRAD ? 4 : 1); ++i) {
      v4[i] += __shfl_xor_sync(0xffffffffu, v4[i], 1);
      v4[i] += __shfl_xor_sync(0xffffffffu, v4[i], 2);
    }
    if (!valid) continue;
    // thread q writes sum q
    if (q == 0) {
      const double phi = (v4[0] + G0[l]) * inv_h + phi_s[slot];
      phi_s[slot] = phi;
      if (phi_out) phi_out[perm[slot]] = phi;
    } else if (GRAD) {
      double* E = E_s + 3 * slot + (q - 1);
      *E = (q == 1 ? v4[1] : (q == 2 ? v4[2] : v4[3])) * (inv_h * inv_h) + *E;
    }
  }
}

// ----------------------------------------------------------------- adjoint
__global__ void k_weights(int64_t N, double gU, const double* __restrict__ gphi, const int* __restrict__ perm,
                          const double* __restrict__ Qs, double* __restrict__ w, float* __restrict__ w32,
                          double scale, double* __restrict__ ws) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= N) return;
  const double v = 0.5 * gU * Qs[k] + (gphi ? gphi[perm[k]] : 0.0);
  w[k] = v;
  if (w32) w32[k] = (float)v;
  if (k == 0 && scale > 0.0) {
    ws[0] = scale;
    ws[1] = 1.0 / scale;
  }
}

// FP64: the power of two that takes the largest weight near 2^100, and its inverse, for
// weights that only the device knows (fep3m_vjp's gphi).  The screen adjoint's float pairs
// are of the scaled weights (the field they give is within 2^12 of them, n_sr <= 4), so that
// their low words stay normal FP32 numbers whatever the weights' unit; non-finite weights
// stay as they are.  One CTA: the weights are read once more, beside the mesh solve (76 800
// charges 8 us, 10^6 49 us).
__global__ void __launch_bounds__(1024) k_weight_scale(int64_t N, const double* __restrict__ w,
                                                       double* __restrict__ ws) {
  __shared__ int top[32];
  int hi = 0;   // the largest exponent, by the high words
  for (int64_t k = threadIdx.x; k < N; k += 1024) hi = max(hi, __double2hiint(w[k]) & 0x7fffffff);
  for (int o = 16; o > 0; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = hi;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = 1; i < 32; ++i) hi = max(hi, top[i]);
  const int e = (hi >> 20) - 1023, k = e == 1024 ? 0 : max(-900, min(900, 100 - e));
  ws[0] = ldexp(1.0, k);
  ws[1] = ldexp(1.0, -k);
}

// W[e][m] = sum_{t in e} w_t u_m(tau_t): the adjoint's point deposit, per
// element.  wsum (FP32 path): sum_{t in e} w_t in FP64 as hi + lo floats, the
// exact sum over m of W[e][m] (the shape functions sum to one).  wT: the
// weights in the working precision.  A warp takes 32 consecutive elements,
// whose charges are one run of the sorted arrays: it reads their starts and,
// 32 at a time, the charges in one load each, then hands them round by
// shuffles, two nodes per lane (with one thread per element and node each
// element waited for three dependent loads: 262 144 charges on 64^3, 146 ->
// 41 us, 10^6 on 128^3, 845 -> 145 us; FP64 rock salt 32^3, where every thread also evaluated twelve
// shape functions, 208 -> 34 us).  That takes some 290 cycles a charge in series,
// so rows of 32 elements with more than `run` charges are dealt by elements to the
// CTA's warps, which put the shape functions of eight charges at a time into shared
// memory and sum over them there (3 KB a CTA, 6 in FP64: with 32 at a time the CTAs
// did not fit beside the screen kernel's, and the FP64 step waited 40 us for that).
// 4096 charges in one row of 32^3 elements: 617 us in one warp, now 40; 20 000 in a blob
// of 16^3: 1165 -> 107.  A CTA takes eight rows.
//
// Dealing costs a row two dependent loads per element, but on a small mesh the rows in
// series leave the GPU idle: there (deposit_dealt) a CTA takes one row and deals it
// whatever it holds.  0.2 / 1 / 3 charges per element, in series and dealt (us), FP32:
// 12^3 8.7 / 17 / 34 and 6.5 / 7.7 / 8.9; 28^3 9.3 / 18 / 37 and 19 / 21 / 22; 32^3 10 /
// 18 / 35 and 23 / 24 / 25; 48^3 12 / 23 / 49 and 66 / 69 / 73.  FP64: 12^3 11 / 32 / 82
// and 8.9 / 12 / 16; 28^3 13 / 35 / 92 and 16 / 39 / 55; 32^3 14 / 37 / 91 and 20 / 50 /
// 77; 48^3 22 / 85 / 238 and 46 / 141 / 235.
constexpr int DEP_RUN = 160;   // (64^3, FP32: 4 charges per element 119 us in series, 165 dealt)
static bool deposit_dealt(int64_t ne, int64_t N) {
  const int64_t rows = (ne + 31) / 32, run = N * 32 / ne;
  return rows < 200 + 15 * run || run > DEP_RUN;
}
// order-3 shape function i at t as q3_values forms it: k (t - r0) (t - r1) (t - r2)
template <class T>
__device__ __forceinline__ T q3_value(T t, int i) {
  const T k = i == 0 ? T(-4.5) : (i == 1 ? T(13.5) : (i == 2 ? T(-13.5) : T(4.5)));
  const T r0 = i == 0 ? T(1) / T(3) : T(0), r1 = i < 2 ? T(2) / T(3) : T(1) / T(3), r2 = i == 3 ? T(2) / T(3) : T(1);
  return k * (t - r0) * (t - r1) * (t - r2);
}
template <class T>
__global__ void __launch_bounds__(PT) k_elem_deposit(int64_t ne, int nrows, int run, const int* __restrict__ start,
                                                     const int* __restrict__ count,
                                                     const typename vec4<T>::type* __restrict__ part,
                                                     const double* __restrict__ w, const T* __restrict__ wT,
                                                     T* __restrict__ W, float2* __restrict__ wsum) {
  __shared__ int crowded[PT / 32];
  __shared__ T shape[PT / 32][12][8];   // of eight of a warp's charges: x (times the weight), y, z
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t cta0 = blockIdx.x * (int64_t)nrows * 32, e0 = cta0 + 32 * warp;
  // this lane's nodes: m = lane and lane + 32 (the same x and y index, z index 2 on)
  const int mx = lane & 3, my = (lane >> 2) & 3, mz = lane >> 4;
  typename vec4<T>::type pc;   // charges held, one per lane
  T wc = T(0);
  pc.x = pc.y = pc.z = pc.w = T(0);
  bool crowd = false;
  if (warp < nrows && e0 < ne) {
    const int nel = (int)min((int64_t)32, ne - e0);
    const int s0 = lane < nel ? start[e0 + lane] : 0, cnt = lane < nel ? count[e0 + lane] : 0;
    const int first = __shfl_sync(0xffffffffu, s0, 0), end = __shfl_sync(0xffffffffu, s0 + cnt, nel - 1);
    crowd = end - first > run;
    if (!crowd) {
      if (wsum && lane < nel) {
        double ws = 0.0;
        for (int j = s0; j < s0 + cnt; ++j) ws += w[j];
        const float hi = (float)ws;
        wsum[e0 + lane] = make_float2(hi, (float)(ws - (double)hi));
      }
      int base = first;                 // the charges base .. base + 31 are held
      auto hold = [&]() {
        if (base + lane < end) {
          pc = part[base + lane];
          wc = wT[base + lane];
        }
      };
      hold();
      for (int i = 0; i < nel; ++i) {
        const int s = __shfl_sync(0xffffffffu, s0, i), c = __shfl_sync(0xffffffffu, cnt, i);
        T a0 = T(0), a1 = T(0);
        for (int j = s; j < s + c; ++j) {
          if (j >= base + 32) {
            base = j;
            hold();
          }
          const int src = j - base;
          const T x = __shfl_sync(0xffffffffu, pc.x, src), y = __shfl_sync(0xffffffffu, pc.y, src),
                  z = __shfl_sync(0xffffffffu, pc.z, src), wj = __shfl_sync(0xffffffffu, wc, src);
          if constexpr (sizeof(T) == 4) {
            const T xy = wj * q3_value(x, mx) * q3_value(y, my);
            a0 += xy * q3_value(z, mz);
            a1 += xy * q3_value(z, mz + 2);
          } else {
            // one shape function per lane (12 of them), then shuffles
            const T u = q3_value(lane < 4 ? x : (lane < 8 ? y : z), lane & 3);
            const T xy = wj * __shfl_sync(0xffffffffu, u, mx) * __shfl_sync(0xffffffffu, u, 4 + my);
            const T z0 = __shfl_sync(0xffffffffu, u, 8 + mz), z1 = __shfl_sync(0xffffffffu, u, 10 + mz);
            a0 = fma(xy, z0, a0);
            a1 = fma(xy, z1, a1);
          }
        }
        W[(e0 + i) * 64 + lane] = a0;
        W[(e0 + i) * 64 + lane + 32] = a1;
      }
    }
  }
  if (lane == 0) crowded[warp] = crowd;
  if (!__syncthreads_or(crowd)) return;
  T(*u)[8] = shape[warp];
  const int axis = lane >> 3;   // this lane's shape functions: along x, y or z (or none), of charge lane mod 8
  for (int r = 0; r < nrows; ++r) {
    if (!crowded[r]) continue;
    const int64_t e1 = min(cta0 + 32 * r + 32, ne);
    for (int64_t e = cta0 + 32 * r + warp; e < e1; e += PT / 32) {
      const int s = start[e], c = count[e];
      T a0 = T(0), a1 = T(0);
      double ws = 0.0;
      for (int base = 0; base < c; base += 32) {
        const int m = min(32, c - base);
        if (lane < m) {
          pc = part[s + base + lane];
          wc = wT[s + base + lane];
          if (wsum) ws += w[s + base + lane];
        }
        for (int b = 0; b < m; b += 8) {
          const int src = b + (lane & 7);   // (past the last charge: a stale one, not read below)
          const T x = __shfl_sync(0xffffffffu, pc.x, src), y = __shfl_sync(0xffffffffu, pc.y, src),
                  z = __shfl_sync(0xffffffffu, pc.z, src), wj = __shfl_sync(0xffffffffu, wc, src);
          const T t = axis == 0 ? x : (axis == 1 ? y : z);
          if (axis < 3)
#pragma unroll
            for (int i = 0; i < 4; ++i) u[4 * axis + i][lane & 7] = axis == 0 ? wj * q3_value(t, i) : q3_value(t, i);
          __syncwarp();
          const int e8 = min(8, m - b);
          if (e8 == 8) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const T xy = u[mx][k] * u[4 + my][k];
              a0 = fma(xy, u[8 + mz][k], a0);
              a1 = fma(xy, u[10 + mz][k], a1);
            }
          } else {
            for (int k = 0; k < e8; ++k) {
              const T xy = u[mx][k] * u[4 + my][k];
              a0 = fma(xy, u[8 + mz][k], a0);
              a1 = fma(xy, u[10 + mz][k], a1);
            }
          }
          __syncwarp();
        }
      }
      W[e * 64 + lane] = a0;
      W[e * 64 + lane + 32] = a1;
      if (wsum) {
        warp_sum(ws);
        const float hi = (float)ws;
        if (lane == 0) wsum[e] = make_float2(hi, (float)(ws - (double)hi));
      }
    }
  }
}

// g[node] = sum over (element, local node) pairs at the node of W: in FP64,
// or (T = float, the mixed solver's right-hand side) as a float pair h + l
// summed by two-sums.  Grid (y, z): a CTA takes a row of nodes, so that the
// elements along y and z are the CTA's and a node's own index costs one
// division (one thread per node of the whole mesh spent 227 instructions on
// the indices: 262 144 charges on 64^3, 100 -> 45 us)
template <class T>
__global__ void __launch_bounds__(PT) k_node_assemble(int n, const T* __restrict__ W, double* __restrict__ g) {
  const int N = 3 * n, iy = blockIdx.x, iz = blockIdx.y;
  // rows of W of the up to four elements that share the row: element row and local node offset
  int64_t row[4];
  int cnt = 0;
  {
    const int ey = iy / 3, ty = iy - 3 * ey, ez = iz / 3, tz = iz - 3 * ez;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if ((c && tz) || (b && ty)) continue;
        const int y = b ? (ey ? ey - 1 : n - 1) : ey, z = c ? (ez ? ez - 1 : n - 1) : ez;
        row[cnt++] = (int64_t)n * (y + (int64_t)n * z) * 64 + 4 * (b ? 3 : ty) + 16 * (c ? 3 : tz);
      }
  }
  const int64_t out = (int64_t)N * (iy + (int64_t)N * iz);
  for (int ix = threadIdx.x; ix < N; ix += PT) {
    const int e = ix / 3, t = ix - 3 * e, at = e * 64 + t, before = (e ? e - 1 : n - 1) * 64 + 3;
    if constexpr (sizeof(T) == 4) {
      float sh = 0.f, sl = 0.f;
      auto add = [&](float v) {
        const float u = sh + v, bv = u - sh;
        sl += (sh - (u - bv)) + (v - bv);
        sh = u;
      };
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (r >= cnt) break;
        add(W[row[r] + at]);
        if (t == 0) add(W[row[r] + before]);
      }
      const float h = sh + sl;
      reinterpret_cast<float2*>(g)[out + ix] = make_float2(h, sl - (h - sh));
    } else {
      double acc = 0.0;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (r >= cnt) break;
        acc += (double)W[row[r] + at];
        if (t == 0) acc += (double)W[row[r] + before];
      }
      g[out + ix] = acc;
    }
  }
}

// Screen part of the adjoint, as a GEMM and a gather (deterministic, no atomics):
//   D[o][e] = sum_m W[e][m] H(o, m)               (every element e, every vertex offset o)
//   A[s][k] = sum_{o : o + k in block} D[o][s + k + o]
// D[o][e] is the table field of element e's deposit seen from the vertex e - o
// (the tensor-core row GEMM in the FP32 path, or k_adj_gemm; k_adj64 in FP64;
// the gather is k_adj_vertex).
constexpr int GT = 64;   // GEMM tile: 64 elements x 64 offsets, K = 64 nodes
constexpr int ADJ_NT = 128;   // tensor-core column tile: offsets per tile

// CUDA cores (MIXED with FEP3M_CUDA_CORES): the products are summed in
// double-float arithmetic on the FP32 pipes (hi + lo float pairs in shared
// memory: the table's from FP64, the FP32 deposit has lo = 0; fused two-product
// with the cross terms, two-sum accumulation), in two halves of 32 nodes whose
// sums are added in FP64.
__global__ void __launch_bounds__(PT) k_adj_gemm(int64_t ne, int o0, int no, const float* __restrict__ W,
                                                 const double* __restrict__ Hw, float* __restrict__ D) {
  __shared__ float2 Ws2[64][GT + 1];   // [m][element]
  __shared__ float2 Hs2[64][GT + 1];   // [m][offset]
  const int64_t e0 = (int64_t)blockIdx.x * GT;
  const int oo0 = o0 + blockIdx.y * GT;
  for (int i = threadIdx.x; i < GT * 64; i += PT) {
    const int r = i >> 6, m = i & 63;
    const int64_t e = e0 + r;
    const int o = oo0 + r;
    const double w = e < ne ? (double)W[e * 64 + m] : 0.0;
    const double hv = (o < o0 + no) ? Hw[(int64_t)o * 64 + m] : 0.0;
    const float wh = (float)w, hh = (float)hv;
    Ws2[m][r] = make_float2(wh, (float)(w - (double)wh));
    Hs2[m][r] = make_float2(hh, (float)(hv - (double)hh));
  }
  __syncthreads();
  const int te = threadIdx.x & 15, to = threadIdx.x >> 4;   // 4 elements x 4 offsets per thread
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    float sh[4][4], sl[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sh[i][j] = sl[i][j] = 0.f;
#pragma unroll 4
    for (int m = 32 * half; m < 32 * half + 32; ++m) {
      float2 a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = Ws2[m][te + 16 * i];
        b[i] = Hs2[m][to + 16 * i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float p = a[i].x * b[j].x;
          float e = fmaf(a[i].x, b[j].x, -p);
          e = fmaf(a[i].x, b[j].y, e);
          e = fmaf(a[i].y, b[j].x, e);
          const float t = sh[i][j] + p, z = t - sh[i][j];
          sl[i][j] += ((sh[i][j] - (t - z)) + (p - z)) + e;
          sh[i][j] = t;
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += (double)sh[i][j] + (double)sl[i][j];
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int o = oo0 + to + 16 * j;
    if (o >= o0 + no) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t e = e0 + te + 16 * i;
      if (e < ne) D[(int64_t)(o - o0) * ne + e] = (float)acc[i][j];
    }
  }
}

// Double-float accumulator (hi + lo floats, summed by two-sum): the FP32
// path's screen adjoint sums, whose terms cancel to a small remainder.
struct dfacc {
  float h, l;
};
__device__ __forceinline__ void acc_add(dfacc& a, float b) {
  const float s = a.h + b, bb = s - a.h;
  a.l += (a.h - (s - bb)) + (b - bb);
  a.h = s;
}
__device__ __forceinline__ void acc_merge(dfacc& a, const dfacc& b) {
  const float s = a.h + b.h, bb = s - a.h;
  a.l += ((a.h - (s - bb)) + (b.h - bb)) + b.l;
  a.h = s;
}
__device__ __forceinline__ double acc_value(const dfacc& a) { return (double)a.h + (double)a.l; }
// the FP64 path's: three floats
__device__ __forceinline__ void acc_merge(tf& a, tf b) { tf_add(a, b); }
__device__ __forceinline__ double acc_value(tf a) { return df_value(a); }

// The FP64 path's D by parity (see k_screen64): with W+-(j) = W(j) +- W(3 - j)
// along each axis, D+-(i) = sum_j E+-(i, j) W+-(j) and D(i) = D+(i) + D-(i),
// D(noff - 1 - i) = D+(i) - D-(i): 4096 multiply-adds an element instead of 32
// 768 (n_sr = 3), in float pairs, and three sums and differences per value.  A
// CTA takes 32 consecutive elements, one per lane; a warp forms the eight
// parities of two offsets i at a time for them and writes their sixteen
// mirrored values of D as pairs (rows of 32 consecutive elements), times the
// weights' scale ws[0] (k_weight_scale).  HP: the table by parity, [s][i][j].
// Bound by FP32 issue; rock salt 32^3: 778 -> 146 us against the full product in pairs with D rounded to FP64.
constexpr int AE = 32;
static size_t adj64_smem(int n_sr) {
  const int kh = n_sr + 1;
  return (size_t)AE * 65 * sizeof(double) + (size_t)64 * AE * sizeof(df) + (size_t)kh * kh * kh * 64 * sizeof(df);
}
__global__ void __launch_bounds__(PT, 2) k_adj64(int64_t ne, int n_sr, int z0, int z1, const double* __restrict__ W,
                                                 const double* __restrict__ ws, const df* __restrict__ HP,
                                                 df* __restrict__ D) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int kh = n_sr + 1, noff = 2 * kh, K = kh * kh * kh, plane = noff * noff;
  double(*Wd)[65] = reinterpret_cast<double(*)[65]>(smem_raw);                                      // [AE]
  df(*Ws)[AE] = reinterpret_cast<df(*)[AE]>(smem_raw + AE * 65 * sizeof(double));                   // [64]: 8 s + j
  df* Hs = reinterpret_cast<df*>(smem_raw + AE * 65 * sizeof(double) + 64 * AE * sizeof(df));       // [8][K][8]
  const int64_t e0 = blockIdx.x * (int64_t)AE;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 64 * K; i += PT) Hs[i] = HP[i];
  for (int i = tid; i < AE * 64; i += PT) {
    const int e = i >> 6;
    Wd[e][i & 63] = e0 + e < ne ? W[(e0 + e) * 64 + (i & 63)] : 0.0;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    __syncthreads();
    for (int i = tid; i < AE * 32; i += PT) {
      // node pair: index j (0, 1) along axis a and its mirror image 3 - j
      const int e = i & 31, r = i >> 5, j = r & 1, o = r >> 1, o0 = o & 3, o1 = o >> 2;
      const int st = a == 0 ? 1 : (a == 1 ? 4 : 16);
      const int base = a == 0 ? 4 * o0 + 16 * o1 : (a == 1 ? o0 + 16 * o1 : o0 + 4 * o1);
      double &x = Wd[e][base + j * st], &y = Wd[e][base + (3 - j) * st];
      const double s = x + y, d = x - y;
      x = s;
      y = d;
    }
  }
  __syncthreads();
  const double scale = ws[0];
  for (int i = tid; i < AE * 64; i += PT) {
    const int e = i & 31, b = i >> 5, s = b >> 3, j = b & 7;
    int node = 0;
    for (int a = 2; a >= 0; --a) {
      const int ja = (j >> a) & 1;
      node = node * 4 + ((s >> a) & 1 ? 3 - ja : ja);
    }
    Ws[b][e] = df_split(Wd[e][node] * scale);
  }
  __syncthreads();
  for (int i0 = 2 * warp; i0 < K; i0 += 2 * (PT / 32)) {
    df v[2][8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      v[0][s] = v[1][s] = df{0.f, 0.f};
      // (an odd K: the last pair's second offset repeats the first, unused)
      const float4* h0 = reinterpret_cast<const float4*>(Hs + (s * K + i0) * 8);
      const float4* h1 = i0 + 1 < K ? h0 + 4 : h0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const df w0 = Ws[8 * s + 2 * j][lane], w1 = Ws[8 * s + 2 * j + 1][lane];
        const float4 a = h0[j], b = h1[j];
        df_fma(v[0][s], w0, df{a.x, a.y});
        df_fma(v[0][s], w1, df{a.z, a.w});
        df_fma(v[1][s], w0, df{b.x, b.y});
        df_fma(v[1][s], w1, df{b.z, b.w});
      }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int i = i0 + t;
      if (i >= K) break;
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          if ((s >> a) & 1) continue;
          const df x = v[t][s], y = v[t][s | (1 << a)];
          v[t][s] = df_add(x, y);
          v[t][s | (1 << a)] = df_add(x, df{-y.h, -y.l});
        }
      const int ix = i % kh, iy = (i / kh) % kh, iz = i / (kh * kh);
      if (e0 + lane >= ne) continue;
#pragma unroll
      for (int f = 0; f < 8; ++f) {
        const int ox = f & 1 ? noff - 1 - ix : ix, oy = f & 2 ? noff - 1 - iy : iy, oz = f & 4 ? noff - 1 - iz : iz;
        if (oz >= z0 && oz < z1) D[((int64_t)(oz - z0) * plane + oy * noff + ox) * ne + e0 + lane] = v[t][f];
      }
    }
  }
}

// Screen adjoint, gathered by vertex:
//   A[s][k] = sum over the offsets o with o + k inside the block of D(o, s + k + o).
// For the vertex v = s + k the terms are D(o, v + o) over the offsets that
// corner k's block holds: along each axis, o_a = -(n_sr + 1) only for k_a = 1,
// o_a = n_sr only for k_a = 0, the others for both.  A CTA takes 256 / AVZ
// consecutive vertices (consecutive lanes read consecutive elements of D) and
// deals the offset planes oz of the chunk [z0, z1) to AVZ threads per vertex.  A
// thread sums a plane's terms into nine classes (first, inner, last offset along
// x and along y); planes of one class along z add up there (AVZ = 1), then go to
// the corners' sums in shared memory, which are combined in order:
// deterministic.  The rows of D come by cp.async into a ring of the thread's own
// (av_ring rows of 2 n_sr + 2 values in flight), the weight sums a row ahead in
// registers.  FP32 path (H0 set): D holds the contraction with the
// node-0-relative table, and each term gains H(o, 0) Wsum(v + o)
// (pair_adjoint_table); terms and sums in double-float arithmetic (19 operations
// a term, of 36 instructions).  FP64 path: D is the whole contraction, as pairs,
// summed in three floats: the up to (2 n_sr)^3 terms of a class are of one sign
// where the weights are, and the low word of a pair's sum would round each of
// them at 2^-48 of the running sum (rock salt 32^3, 28 us with two floats, 35 with
// three).  Bound by instruction issue, at 2/3 of its rate.  10^6
// charges on 128^3: 3484 us with one warp per 32 vertices and row of offsets and 27
// class sums in shared memory, 2301 with a row ahead in registers and AVZ = 8, 1458
// now; 262 144 on 64^3: 439, 285 and 195 us.
//
// One thread per vertex (AVZ = 1) from 40 elements per axis on, eight below,
// where one leaves too few warps (8 / 1, us: 16^3 9.9 / 35, 32^3 37 / 39, 40^3
// 68 / 61, 48^3 110 / 92, 64^3 249 / 195).
// asynchronous copy of one value (4 or 8 bytes) to shared memory
template <class T>
__device__ __forceinline__ void cp_async_val(T* dst, const T* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(sizeof(T))
               : "memory");
}
// rows of D in flight per thread: a divisor of the rows of a plane (a row's place is the same in every plane)
template <int NSR>
constexpr int av_ring = NSR == 2 ? 3 : (NSR == 4 ? 5 : 4);
template <class T, int NSR, int AVZ>
struct AdjVertexSmem {
  static constexpr int NOFF = 2 * NSR + 2;
  T ring[av_ring<NSR>][NOFF][PT];
  typedef typename std::conditional<sizeof(T) == 4, dfacc, tf>::type Acc;   // (tf: three floats)
  Acc part[AVZ][8][PT / AVZ];
  float2 h0[sizeof(T) == 4 ? NOFF * NOFF * NOFF : 1];
  int live[PT / AVZ];
};
template <class T, int NSR, int AVZ>
__global__ void __launch_bounds__(PT, 2) k_adj_vertex(int n, int z0, int z1, int first, const int* __restrict__ count,
                                                      const T* __restrict__ D, int64_t ld, const float2* __restrict__ H0,
                                                      const float2* __restrict__ wsum, const double* __restrict__ ws,
                                                      double* __restrict__ A) {
  constexpr int KEEP = NSR + 1, NOFF = 2 * NSR + 2, PLANE = NOFF * NOFF, AVV = PT / AVZ, AV_RING = av_ring<NSR>;
  constexpr bool REL = sizeof(T) == 4;   // T: float, or df (FP64)
  typedef typename AdjVertexSmem<T, NSR, AVZ>::Acc Acc;
  extern __shared__ __align__(16) unsigned char av_smem[];
  AdjVertexSmem<T, NSR, AVZ>& S = *reinterpret_cast<AdjVertexSmem<T, NSR, AVZ>*>(av_smem);
  const int64_t ne = (int64_t)n * n * n;
  const int tid = threadIdx.x, vl = tid & (AVV - 1), zg = AVZ == 1 ? 0 : tid / AVV;
  const int64_t v = blockIdx.x * (int64_t)AVV + vl;
  const bool in = v < ne;
  const int vx = in ? (int)(v % n) : 0, vy = in ? (int)((v / n) % n) : 0, vz = in ? (int)(v / ((int64_t)n * n)) : 0;
  if (zg == 0) {
    bool any = false;   // the eight elements v - k; A is read only for non-empty ones
    if (in) {
      const int px = vx ? vx - 1 : n - 1, py = vy ? vy - 1 : n - 1, pz = vz ? vz - 1 : n - 1;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        any |= count[((k & 1) ? px : vx) + (int64_t)n * (((k & 2) ? py : vy) + (int64_t)n * ((k & 4) ? pz : vz))] != 0;
    }
    S.live[vl] = any;
  }
  if (REL)
    for (int i = tid; i < PLANE * NOFF; i += PT) S.h0[i] = H0[i];
  __syncthreads();
  const bool act = S.live[vl] != 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) S.part[zg][k][vl] = Acc{};   // corner sums, k = kx + 2 ky + 4 kz
  const int oz0 = z0 + zg;
  if (oz0 < z1 && __any_sync(0xffffffffu, act)) {
    int wx[NOFF];   // the elements' x coordinates vx + o - KEEP (n >= 2 n_sr + 1: one period at most)
#pragma unroll
    for (int i = 0; i < NOFF; ++i) {
      int x = vx + i - KEEP;
      x += x < 0 ? n : 0;
      wx[i] = x >= n ? x - n : x;
    }
    int ey0 = vy - KEEP;
    ey0 += ey0 < 0 ? n : 0;
    auto plane_row = [&](int oz) {   // the first element of the plane's elements (n <= 404: below 2^31)
      int ez = vz + oz - KEEP;
      ez += ez < 0 ? n : 0;
      ez = ez >= n ? ez - n : ez;
      return n * n * ez;
    };
    Acc P[3][3];   // [class along y][class along x]: first, inner, last
#pragma unroll
    for (int i = 0; i < 9; ++i) P[i / 3][i % 3] = Acc{};
    float2 w[REL ? 2 : 1][NOFF];   // the weight sums of the row being summed and of the next
    int eyd = ey0, eyw = ey0;      // element rows of the next fetch and the next load
    // row oy of plane oz of D into this thread's ring; called in order of the rows
    auto fetch = [&](int oz, int oy, int prow) {
      if (oz < z1) {
        const T* Dr = D + ((int64_t)(oz - z0) * PLANE + oy * NOFF) * ld;
        const int er = prow + n * eyd;
#pragma unroll
        for (int ox = 0; ox < NOFF; ++ox)
          cp_async_val(&S.ring[oy % AV_RING][ox][tid], Dr + ox * ld + (unsigned)(er + wx[ox]));
        eyd = eyd + 1 == n ? 0 : eyd + 1;
        if (oy == NOFF - 1) eyd = ey0;
      }
      tc::cp_async_commit();       // (past the last row an empty group, for the count below)
    };
    auto load = [&](int oy, int prow) {   // row oy's weight sums; called in order of the rows
      if constexpr (REL) {
        const int er = prow + n * eyw;
#pragma unroll
        for (int ox = 0; ox < NOFF; ++ox) w[oy & 1][ox] = wsum[(unsigned)(er + wx[ox])];
        eyw = eyw + 1 == n ? 0 : eyw + 1;
        if (oy == NOFF - 1) eyw = ey0;
      }
    };
    int prow = plane_row(oz0);
#pragma unroll
    for (int oy = 0; oy < AV_RING; ++oy) fetch(oz0, oy, prow);
    load(0, prow);
#pragma unroll 1
    for (int oz = oz0; oz < z1; oz += AVZ) {
      const int pnext = plane_row(oz + AVZ);
#pragma unroll
      for (int oy = 0; oy < NOFF; ++oy) {
        constexpr int L = NOFF - 1;
        const int cy = oy == 0 ? 0 : (oy == L ? 2 : 1);
        if (oy + 1 < NOFF) load(oy + 1, prow);
        else if (oz + AVZ < z1) load(0, pnext);
        asm volatile("cp.async.wait_group %0;" ::"n"(AV_RING - 1) : "memory");   // row oy (this thread's own copies)
        T d[NOFF];
#pragma unroll
        for (int ox = 0; ox < NOFF; ++ox) d[ox] = S.ring[oy % AV_RING][ox][tid];
        if (oy + AV_RING < NOFF) fetch(oz, oy + AV_RING, prow);   // into the row just read
        else fetch(oz + AVZ, oy + AV_RING - NOFF, pnext);
#pragma unroll
        for (int ox = 0; ox < NOFF; ++ox) {
          const int cx = ox == 0 ? 0 : (ox == L ? 2 : 1);
          if constexpr (REL) {
            const float2 h = S.h0[oz * PLANE + oy * NOFF + ox], u = w[oy & 1][ox];
            const float p = h.x * u.x;
            float r = fmaf(h.x, u.x, -p);
            r = fmaf(h.x, u.y, r);
            r = fmaf(h.y, u.x, r);
            acc_add(P[cy][cx], p);
            acc_add(P[cy][cx], d[ox] + r);
          } else {
            tf_add(P[cy][cx], d[ox]);
          }
        }
      }
      prow = pnext;
      // the inner planes of a thread count alike for both corners: their sums stay in P
      if (AVZ == 1 && oz > 0 && oz < NOFF - 2 && oz < z1 - 1) continue;
#pragma unroll
      for (int k = 0; k < 4; ++k) {   // corner (kx, ky): classes 0, 1 for 1, classes 1, 2 for 0
        const int x0 = k & 1 ? 0 : 1, y0 = k & 2 ? 0 : 1;
        Acc t = P[y0][x0];
        acc_merge(t, P[y0][x0 + 1]);
        acc_merge(t, P[y0 + 1][x0]);
        acc_merge(t, P[y0 + 1][x0 + 1]);
        if (oz != NOFF - 1) acc_merge(S.part[zg][k + 4][vl], t);
        if (oz != 0) acc_merge(S.part[zg][k][vl], t);
      }
#pragma unroll
      for (int i = 0; i < 9; ++i) P[i / 3][i % 3] = Acc{};
    }
  }
  __syncthreads();
  if (!in || !act) return;
#pragma unroll
  for (int t = 0; t < 8 / AVZ; ++t) {
    const int k = zg + AVZ * t, kx = k & 1, ky = (k >> 1) & 1, kz = k >> 2;
    Acc s = S.part[0][k][vl];
#pragma unroll
    for (int z = 1; z < AVZ; ++z) acc_merge(s, S.part[z][k][vl]);
    const int sx = vx - kx < 0 ? n - 1 : vx - kx, sy = vy - ky < 0 ? n - 1 : vy - ky, sz = vz - kz < 0 ? n - 1 : vz - kz;
    double* dst = A + (sx + (int64_t)n * (sy + (int64_t)n * sz)) * 8 + k;
    const double a = REL ? acc_value(s) : acc_value(s) * ws[1];
    *dst = first ? a : *dst + a;
  }
}

template <class T, bool GRAD>
__global__ void __launch_bounds__(PT) k_pair_adj_warp(int64_t N, int n, int n_sr, T h, const int* __restrict__ start,
                                                      const typename vec4<T>::type* __restrict__ part,
                                                      const int* __restrict__ ecoord, const double* __restrict__ w,
                                                      double* __restrict__ psi, double* __restrict__ gpsi) {
  __shared__ int4 rows_all[PT / 32][MAXROW];
  __shared__ int pre_all[PT / 32][MAXROW + 1];
  __shared__ char2 tab[MAXROW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = blockIdx.x * (int64_t)(PT / 32) + warp;
  row_table(n_sr, tab);
  if (t >= N) return;
  const typename vec4<T>::type pt = part[t];
  const int ec = ecoord[t];
  T sg[4];
  warp_singular<T, GRAD>(n, n_sr, tab, h, ec & 1023, (ec >> 10) & 1023, ec >> 20, (int)t, pt, start, part, ecoord,
                         rows_all[warp], pre_all[warp], w, sg);
  if (lane == 0) {
    psi[t] = (double)sg[0];
    if (GRAD) {
      gpsi[3 * t + 0] = (double)sg[1];
      gpsi[3 * t + 1] = (double)sg[2];
      gpsi[3 * t + 2] = (double)sg[3];
    }
  }
}

// per charge: dLf/dQ and dLf/dx from the pieces (see fep3m_vjp)
template <class T>
__global__ void k_final(int64_t N, int n, double inv_h, double gU, double sign,
                        const typename vec4<T>::type* __restrict__ part,
                        const int* __restrict__ perm, const int* __restrict__ cell, const double* __restrict__ w,
                        const double* __restrict__ phi_s, const double* __restrict__ E_s,
                        const double* __restrict__ psi, const double* __restrict__ gpsi, const double* __restrict__ mu,
                        const double* __restrict__ A, double* __restrict__ dpos, double* __restrict__ dQ) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= N) return;
  const int i = perm[t];
  const int e = cell[i];
  const int ex = e % n, ey = (e / n) % n, ez = e / (n * n);
  const typename vec4<T>::type p = part[t];
  const double tx = p.x, ty = p.y, tz = p.z, Q = p.w;
  const double wx[2] = {1.0 - tx, tx}, wy[2] = {1.0 - ty, ty}, wz[2] = {1.0 - tz, tz};
  const double sg[2] = {-1.0, 1.0};
  double sQ = 0, gx = 0, gy = 0, gz = 0;
  for (int k = 0; k < 8; ++k) {
    const int kx = k & 1, ky = (k >> 1) & 1, kz = k >> 2;
    const int64_t v = wrapn(ex + kx, n) + (int64_t)n * (wrapn(ey + ky, n) + (int64_t)n * wrapn(ez + kz, n));
    const double coef = (mu[v] - A[(int64_t)e * 8 + k]) * inv_h;
    sQ += wx[kx] * wy[ky] * wz[kz] * coef;
    gx += sg[kx] * wy[ky] * wz[kz] * coef;
    gy += wx[kx] * sg[ky] * wz[kz] * coef;
    gz += wx[kx] * wy[ky] * sg[kz] * coef;
  }
  const double wt = w[t];
  if (dQ) dQ[i] = 0.5 * gU * phi_s[t] + psi[t] + sQ;
  if (dpos) {
    dpos[3 * i + 0] = sign * (wt * E_s[3 * t + 0] + Q * (gpsi[3 * t + 0] + gx * inv_h));
    dpos[3 * i + 1] = sign * (wt * E_s[3 * t + 1] + Q * (gpsi[3 * t + 1] + gy * inv_h));
    dpos[3 * i + 2] = sign * (wt * E_s[3 * t + 2] + Q * (gpsi[3 * t + 2] + gz * inv_h));
  }
}

// deterministic sum of a per-charge product (FP64): out = 1/2 sum Q phi
__global__ void k_energy(int64_t N, const double* __restrict__ Qs, const double* __restrict__ phi,
                         double* __restrict__ partials, unsigned int* __restrict__ counter, double* __restrict__ out) {
  __shared__ double sh[PT / 32];
  __shared__ bool last;
  double acc = 0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < N; k += (int64_t)gridDim.x * blockDim.x)
    acc += Qs[k] * phi[k];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0;
    for (int k = 0; k < PT / 32; ++k) s += sh[k];
    partials[blockIdx.x] = s;
    __threadfence();
    last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    double s = 0;
    for (unsigned int k = 0; k < gridDim.x; ++k) s += ((volatile double*)partials)[k];
    *out = 0.5 * s;
    *counter = 0u;
  }
}

inline int gsz(int64_t n, int t = PT) { return (int)((n + t - 1) / t); }

}  // namespace

// ordered singular pairs, non-empty elements and the largest element population
// per non-empty element e with c0 charges and s charges in its block (nb
// non-empty block elements): singular pairs c0 s - c0, one non-empty element,
// the largest c0, nb (element pairs of the screen contraction) and c0 nb
// (charge-element pairs)
__device__ __forceinline__ void pair_count_one(int n, int n_sr, const int* __restrict__ count, int64_t e,
                                               unsigned long long v[5]) {
  const int c0 = count[e];
  if (c0 == 0) return;
  const int ex = (int)(e % n), ey = (int)((e / n) % n), ez = (int)(e / ((int64_t)n * n));
  long long s = 0, nb = 0;
  for (int dz = -n_sr; dz <= n_sr; ++dz)
    for (int dy = -n_sr; dy <= n_sr; ++dy)
      for (int dx = -n_sr; dx <= n_sr; ++dx) {
        const int cj = count[wrapn(ex + dx, n) + (int64_t)n * (wrapn(ey + dy, n) + (int64_t)n * wrapn(ez + dz, n))];
        s += cj;
        nb += cj > 0;
      }
  v[0] = (unsigned long long)((long long)c0 * s - c0);
  v[1] = 1ull;
  v[2] = (unsigned long long)c0;
  v[3] = (unsigned long long)nb;
  v[4] = (unsigned long long)((long long)c0 * nb);
}

// warp sums (and max) first: one atomic per warp and counter
__global__ void k_pair_count(int n, int n_sr, const int* __restrict__ count, unsigned long long* __restrict__ out) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned long long v[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
  if (e < (int64_t)n * n * n) pair_count_one(n, n_sr, count, e, v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    v[1] += __shfl_down_sync(0xffffffffu, v[1], o);
    const unsigned long long m = __shfl_down_sync(0xffffffffu, v[2], o);
    v[2] = m > v[2] ? m : v[2];
    v[3] += __shfl_down_sync(0xffffffffu, v[3], o);
    v[4] += __shfl_down_sync(0xffffffffu, v[4], o);
  }
  if ((threadIdx.x & 31) == 0 && v[1] != 0ull) {
    atomicAdd(&out[0], v[0]);
    atomicAdd(&out[1], v[1]);
    atomicMax(&out[2], v[2]);
    atomicAdd(&out[3], v[3]);
    atomicAdd(&out[4], v[4]);
  }
}

cudaError_t pair_counts(fep3m_ctx* c, unsigned long long* dev5, cudaStream_t s) {
  const int64_t ne = (int64_t)c->n * c->n * c->n;
  cudaMemsetAsync(dev5, 0, 5 * sizeof(unsigned long long), s);
  FEP3M_CL k_pair_count<<<gsz(ne), PT, 0, s>>>(c->n, c->n_sr, c->count, dev5);
  return cudaGetLastError();
}

static int pair_bricks(const fep3m_ctx* c) {
  const int n = c->n;
  return ((n + BX - 1) / BX) * ((n + BY - 1) / BY) * ((n + BZ - 1) / BZ);
}

size_t pair_screen_bytes(const fep3m_ctx* c) {
  return (size_t)pair_bricks(c) * BE * 64 * (c->precision == FEP3M_MIXED ? sizeof(float) : sizeof(double));
}

template <bool GRAD, bool TC>
static cudaError_t launch_pair_screen(fep3m_ctx* c, cudaStream_t s, bool half) {
  const size_t smem = Pair3Smem<TC>::bytes(c->n_sr);
  auto kern = k_pair_screen<GRAD, TC>;
  cudaError_t e = smem_limit((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  FEP3M_CL kern<<<(unsigned)pair_bricks(c), TC ? PTC : PT, smem, s>>>(
      c->n, c->n_sr, (float)c->h, c->start, c->count, (const float4*)c->part, (const float*)c->Vc,
      (const uint4*)c->Hb, (const float2*)c->H0df, (const float2*)c->Hdf, (float*)c->Gscr, c->phi_s, c->E_s,
      half ? c->psi_s : nullptr,
      half ? c->gpsi_s : nullptr, c->iflags + 2);
  return cudaGetLastError();
}

// nodes per axis of the mesh the evaluation reads: the periodic order-3 mesh,
// or a box's
static int mesh_nodes_per_axis(const fep3m_ctx* c) { return c->box ? c->box->Nn : 3 * c->n; }

// MIXED: the mesh potential as hi + lo floats: the periodic solver's output
// itself, a box's split by pair_prepare
static const float2* mesh_potential_pairs(const fep3m_ctx* c) {
  if (c->precision != FEP3M_MIXED) return nullptr;
  return c->box ? (const float2*)c->phi_hl : (const float2*)c->phi64;
}

template <bool GRAD>
static cudaError_t launch_pair_eval(fep3m_ctx* c, double* phi_out) {
  const unsigned g = (unsigned)pair_bricks(c);
  if (c->precision == FEP3M_MIXED)
    FEP3M_CL k_pair_eval<GRAD><<<g, PT, 0, c->stream>>>(
        c->n, mesh_nodes_per_axis(c), (float)c->inv_h, c->start, c->count, (const float4*)c->part,
        mesh_potential_pairs(c), (const float*)c->Gscr, c->perm, c->phi_s, c->E_s, phi_out);
  else
    FEP3M_CL k_pair_eval64<GRAD><<<g, PT, 0, c->stream>>>(
        c->n, mesh_nodes_per_axis(c), c->inv_h, c->start, c->count, (const vec4<double>::type*)c->part, c->phi64,
        (const double*)c->Gscr, c->perm, c->phi_s, c->E_s, phi_out);
  return cudaGetLastError();
}

static cudaError_t singular64(fep3m_ctx* c, bool grad, bool half, cudaStream_t s);

cudaError_t pair_screen(fep3m_ctx* c, int want_grad, cudaStream_t s, bool energy_adjoint) {
  const bool half = energy_adjoint && want_grad;
  if (c->precision == FEP3M_MIXED) {
    if (c->Hb)
      return want_grad ? launch_pair_screen<true, true>(c, s, half)
                       : launch_pair_screen<false, true>(c, s, half);
    return want_grad ? launch_pair_screen<true, false>(c, s, half)
                     : launch_pair_screen<false, false>(c, s, half);
  }
  const size_t smem = screen64_smem(c->n_sr);
  cudaError_t e = smem_limit((const void*)k_screen64, smem);
  if (e != cudaSuccess) return e;
  FEP3M_CL k_screen64<<<dim3((unsigned)pair_bricks(c), 4), PT, smem, s>>>(
      c->n, c->n_sr, c->count, (const df*)c->Vc, (const df*)c->HP, 1.0 / c->q_scale,
      (double*)c->Gscr);
  return singular64(c, want_grad != 0, half, s);
}

// Corner structure of an element's 64 order-3 nodes (m = mx + 4 my + 16 mz):
// corner c = cx + 2 cy + 4 cz sits at node 3 cx + 12 cy + 48 cz, and the
// trilinear interpolant of the eight corner values has weight
// prod_a (c_a ? m_a / 3 : 1 - m_a / 3) at node m.
static int corner_node(int c) { return 3 * (c & 1) + 12 * ((c >> 1) & 1) + 48 * (c >> 2); }
static bool is_corner_node(int m) {
  const int mx = m & 3, my = (m >> 2) & 3, mz = m >> 4;
  return (mx == 0 || mx == 3) && (my == 0 || my == 3) && (mz == 0 || mz == 3);
}
static double corner_weight(int c, int m) {
  const int mm[3] = {m & 3, (m >> 2) & 3, m >> 4};
  double w = 1.0;
  for (int a = 0; a < 3; ++a) w *= ((c >> a) & 1) ? mm[a] / 3.0 : 1.0 - mm[a] / 3.0;
  return w;
}

// The FP32 path's screen-field table, relative to each element's corners:
// column 0 is H(o, 0); the other corner columns H(o, c) - H(o, 0); every
// other column H(o, m) minus the trilinear interpolant of H(o, corners) at m.
// The contraction sum_o A(o) Hrel(o, m) then returns the field at node 0, the
// corner fields relative to it and, elsewhere, the field less its trilinear
// interpolant: the same field with its large smooth part taken out of the
// FP32 sums (its corner values enter the evaluation in FP64).
void pair_relative_table(int n_sr, const double* Hw, double* Hrel) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  for (int o = 0; o < no3; ++o) {
    const double* h = Hw + (size_t)o * 64;
    double* r = Hrel + (size_t)o * 64;
    for (int m = 0; m < 64; ++m) {
      if (m == 0) {
        r[m] = h[0];
      } else if (is_corner_node(m)) {
        r[m] = h[m] - h[0];
      } else {
        double t = 0.0;
        for (int c = 0; c < 8; ++c) t += corner_weight(c, m) * h[corner_node(c)];
        r[m] = h[m] - t;
      }
    }
  }
}

// The FP32 path's screen-adjoint table: Hd(o, m) = H(o, m) - H(o, 0), column 0
// zero.  With Wsum(e) = sum_m W[e][m] the contraction splits as
//   D(o, e) = H(o, 0) Wsum(e) + sum_m W[e][m] Hd(o, m):
// the tensor cores form the second part (small terms), the gather adds the
// first in double-float arithmetic (H0: hi + lo floats of H(o, 0)).
void pair_adjoint_table(int n_sr, const double* Hw, double* Hd, float* H0) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  for (int o = 0; o < no3; ++o) {
    const double h0 = Hw[(size_t)o * 64];
    for (int m = 0; m < 64; ++m) Hd[(size_t)o * 64 + m] = m == 0 ? 0.0 : Hw[(size_t)o * 64 + m] - h0;
    const float hi = (float)h0;
    H0[2 * o] = hi;
    H0[2 * o + 1] = (float)(h0 - (double)hi);
  }
}

// The table as the mean over its mirror images along each axis, H(noff - 1 - o, 3 - m) =
// H(o, m), which agree to the rounding of the solve that made them.  The FP64 path's
// contractions by parity are of this table, so whatever else the path forms from it (a
// box's boundary values and fluxes) takes it too: what a screen adds at the boundary and
// what it subtracts at a charge is then the same field.
void pair_mirror_table(int n_sr, double* Hw) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  for (int a = 0; a < 3; ++a) {
    const int so = a == 0 ? 1 : (a == 1 ? noff : noff * noff), sm = a == 0 ? 1 : (a == 1 ? 4 : 16);
    for (int o = 0; o < no3; ++o) {
      const int oa = (o / so) % noff;
      if (2 * oa >= noff) continue;   // with its image (noff is even)
      for (int m = 0; m < 64; ++m) {
        double &x = Hw[(size_t)o * 64 + m];
        double &y = Hw[(size_t)(o + (noff - 1 - 2 * oa) * so) * 64 + m + (3 - 2 * ((m / sm) & 3)) * sm];
        x = y = 0.5 * (x + y);
      }
    }
  }
}

// the FP64 path's table by parity: HP[s][k][j], s = sx + 2 sy + 4 sz, k the offsets
// 0 .. n_sr and j the nodes 0, 1 per axis (x fastest): the mean over the mirror
// images (which agree to rounding) with the parities' signs, as float pairs
void pair_parity_table(int n_sr, const double* Hw, float* out) {
  const int kh = n_sr + 1, noff = 2 * kh, K = kh * kh * kh;
  for (int s = 0; s < 8; ++s)
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < 8; ++j) {
        const int kk[3] = {k % kh, (k / kh) % kh, k / (kh * kh)};
        double v = 0.0;
        for (int f = 0; f < 64; ++f) {   // bit a: mirror the offset along axis a; bit 3 + a: the node
          int o = 0, m = 0, sign = 1;
          for (int a = 2; a >= 0; --a) {
            const int fo = (f >> a) & 1, fm = (f >> (3 + a)) & 1, ja = (j >> a) & 1;
            o = o * noff + (fo ? noff - 1 - kk[a] : kk[a]);
            m = m * 4 + (fm ? 3 - ja : ja);
            if (((s >> a) & 1) && fo != fm) sign = -sign;
          }
          v += sign * Hw[(size_t)o * 64 + m];
        }
        const df d = df_split(v / 64.0);
        out[2 * ((size_t)(s * K + k) * 8 + j)] = d.h;
        out[2 * ((size_t)(s * K + k) * 8 + j) + 1] = d.l;
      }
}

// the table's three bf16 pieces for the screen adjoint's contraction
// D[o][e] = sum_m W[e][m] H(o, m) on the tensor cores: B[o][m] = H(o, m) in
// column tiles of ADJ_NT offsets, one chunk of the 64 nodes
size_t pair_adj_table_bytes(int n_sr) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  return (size_t)((no3 + ADJ_NT - 1) / ADJ_NT) * 3 * ADJ_NT * 64 * 2;
}
void pair_adj_table(int n_sr, const double* Hw, uint16_t* out) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff, ntile = (no3 + ADJ_NT - 1) / ADJ_NT;
  std::memset(out, 0, pair_adj_table_bytes(n_sr));
  for (int t = 0; t < ntile; ++t)
    for (int ii = 0; ii < ADJ_NT; ++ii) {
      const int o = t * ADJ_NT + ii;
      if (o >= no3) continue;
      for (int m = 0; m < 64; ++m) {
        uint16_t pc[3];
        bf16_pieces(Hw[(size_t)o * 64 + m], pc);
        for (int p = 0; p < 3; ++p) out[((size_t)t * 3 + p) * ADJ_NT * 64 + sw128_off(ii, m) / 2] = pc[p];
      }
    }
}

// the table's three bf16 pieces per chunk of 64 offsets, in the swizzled
// K-major layout of the tensor-core tiles: [chunk][piece][node row][offset]
size_t pair_tc_table_bytes(int n_sr) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff;
  return (size_t)((no3 + 63) / 64) * 3 * 8192;
}
void pair_tc_table(int n_sr, const double* Hw, uint16_t* out) {
  const int noff = 2 * n_sr + 2, no3 = noff * noff * noff, nch = (no3 + 63) / 64;
  auto bits = [](double v) -> uint16_t {   // round to nearest even bf16 (finite v)
    const float f = (float)v;
    uint32_t u;
    std::memcpy(&u, &f, 4);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
  };
  auto val = [](uint16_t b) -> double {
    const uint32_t u = (uint32_t)b << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return (double)f;
  };
  std::memset(out, 0, pair_tc_table_bytes(n_sr));
  for (int ch = 0; ch < nch; ++ch)
    for (int m = 0; m < 64; ++m)
      for (int k = 0; k < 64; ++k) {
        const int o = 64 * ch + k;
        double r = o < no3 ? Hw[(size_t)o * 64 + m] : 0.0;
        for (int p = 0; p < 3; ++p) {
          const uint16_t b = bits(r);
          r -= val(b);
          out[((size_t)(ch * 3 + p) * 8192 + sw128_off(m, k)) / 2] = b;
        }
      }
}

// a box's FP64 mesh vectors as hi + lo floats
__global__ void k_phi_hilo(int64_t n, const double* __restrict__ phi, float2* __restrict__ out) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= n) return;
  const double v = phi[g];
  const float hi = (float)v;
  out[g] = make_float2(hi, (float)(v - (double)hi));
}

cudaError_t split_pairs(int64_t n, const double* v, void* out, cudaStream_t s) {
  FEP3M_CL k_phi_hilo<<<gsz(n), PT, 0, s>>>(n, v, (float2*)out);
  return cudaGetLastError();
}

cudaError_t pair_prepare(fep3m_ctx* c) {
  if (c->precision == FEP3M_MIXED && c->box) {   // the periodic solver writes float pairs itself
    const int64_t na = mesh_nodes_per_axis(c), nodes = na * na * na;
    FEP3M_CL k_phi_hilo<<<gsz(nodes), PT, 0, c->stream>>>(nodes, c->phi64, (float2*)c->phi_hl);
  }
  return cudaGetLastError();
}

cudaError_t pair_eval(fep3m_ctx* c, double* phi_out, int want_grad) {
  return want_grad ? launch_pair_eval<true>(c, phi_out) : launch_pair_eval<false>(c, phi_out);
}

// Potentials and their gradients at the charges, on stream s, after a forward
// without gradients: the mesh potential and the screens' class sums are there.
// FP64 keeps the screen field too; the FP32 screen kernel writes it again, as the
// singular sums are made there.
cudaError_t pair_fields(fep3m_ctx* c, cudaStream_t s) {
  cudaError_t e = c->precision == FEP3M_MIXED ? pair_screen(c, 1, s, false) : singular64(c, true, false, s);
  if (e != cudaSuccess) return e;
  const cudaStream_t keep = c->stream;
  c->stream = s;   // launch_pair_eval issues on c->stream
  e = pair_eval(c, nullptr, 1);
  c->stream = keep;
  return e;
}

cudaError_t energy(fep3m_ctx* c, double* U_dev, cudaStream_t s) {
  const int64_t N = c->N;
  const int nb = (int)std::min<int64_t>(std::max<int64_t>(gsz(N), 1), 1024);
  FEP3M_CL k_energy<<<nb, PT, 0, s ? s : c->stream>>>(N, c->Q_s, c->phi_s, (double*)c->red_tmp, c->red_counter, U_dev);
  return cudaGetLastError();
}

constexpr int AV_LARGE = 40;   // k_adj_vertex
template <class T, int NSR, int AVZ>
static void launch_adj_vertex_z(fep3m_ctx* c, int z0, int z1, const T* D, int64_t ld, double* A, cudaStream_t s) {
  const int64_t ne = (int64_t)c->n * c->n * c->n;
  const bool rel = sizeof(T) == 4;   // D relative to node 0 (FP32 path)
  const size_t smem = sizeof(AdjVertexSmem<T, NSR, AVZ>);
  (void)smem_limit((const void*)k_adj_vertex<T, NSR, AVZ>, smem);   // a failure shows as the launch's error
  constexpr int AVV = PT / AVZ;
  FEP3M_CL k_adj_vertex<T, NSR, AVZ><<<(unsigned)((ne + AVV - 1) / AVV), PT, smem, s>>>(
      c->n, z0, z1, z0 == 0, c->count, D, ld, rel ? (const float2*)c->H0df : nullptr,
      rel ? (const float2*)c->Wsum : nullptr, c->scal + kWeightScale, A);
}
template <class T, int NSR>
static void launch_adj_vertex(fep3m_ctx* c, int z0, int z1, const T* D, int64_t ld, double* A, cudaStream_t s) {
  if (c->n >= AV_LARGE) launch_adj_vertex_z<T, NSR, 1>(c, z0, z1, D, ld, A, s);
  else launch_adj_vertex_z<T, NSR, 8>(c, z0, z1, D, ld, A, s);
}

// D-GEMM + gather over chunks of whole offset planes (all offsets with one
// oz), sized so D stays within a memory budget
template <class T>
static cudaError_t screen_adjoint(fep3m_ctx* c, const T* W, double* A) {
  const int n = c->n;
  const int64_t ne = (int64_t)n * n * n;
  const int noff = c->noff, plane = noff * noff;
  // bytes of D held at once: a quarter of the device's memory (at least 2 GiB), so that on a
  // large GPU even the 256^3 mesh takes D in one piece (each further piece re-reads and
  // re-writes A and launches the gather again); sized at the context's first sweep
  if (c->adj_planes == 0) {
    size_t budget = (size_t)1 << 31;
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess) budget = std::max(budget, std::min(total_b / 4, free_b / 2));
    else (void)cudaGetLastError();
    c->adj_planes = (int)std::min<int64_t>(noff, std::max<int64_t>(1, (int64_t)(budget / ((size_t)ne * sizeof(T) * plane))));
  }
  // tensor cores (FP32 path, table pieces prepared): column tiles of ADJ_NT offsets
  const bool tcore = sizeof(T) == 4 && c->HbA != nullptr;
  // one CTA per SM (k_tc_sweep) where the sweep is not beside the mesh solve, whose short kernels on the
  // critical path would wait for it (run_forward); its stores take D's rows as whole 128-byte lines
  // (81^3 elements, rows unpadded: 406 us, padded 221; the gather 387 and 375)
  const bool sweep = tcore && mesh_solve_alone(&c->solv[0]);
  const int64_t ld = sweep ? (ne + 31) / 32 * 32 : ne;
  const int planes = c->adj_planes;
  const size_t need = (size_t)planes * plane * ld * sizeof(T);
  if (c->D_bytes < need) {
    if (c->D_adj) cudaFree(c->D_adj);
    c->D_adj = nullptr;
    c->D_bytes = 0;
    cudaError_t e = cudaMalloc(&c->D_adj, need);
    if (e != cudaSuccess) return e;
    c->D_bytes = need;
  }
  cudaStream_t s = c->stream;
  for (int z0 = 0; z0 < noff; z0 += planes) {
    const int z1 = std::min(noff, z0 + planes), o0 = z0 * plane, no = (z1 - z0) * plane;
    if (tcore) {
      cudaError_t e = sweep
                          ? tc_sweep_gemm(ne, ld, o0, o0 + no, (const float*)W, c->HbA, (float*)c->D_adj, c->iflags + 2, s)
                          : tc_rows_gemm(ne, 64, o0, o0 + no, ADJ_NT, (const float*)W, c->HbA, (float*)c->D_adj,
                                         c->iflags + 2, s);
      if (e != cudaSuccess) return e;
    } else if constexpr (sizeof(T) == 8) {
      const size_t smem = adj64_smem(c->n_sr);
      (void)smem_limit((const void*)k_adj64, smem);   // a failure shows as the launch's error
      FEP3M_CL k_adj64<<<(unsigned)((ne + AE - 1) / AE), PT, smem, s>>>(ne, c->n_sr, z0, z1, (const double*)W,
                                                                       c->scal + kWeightScale, (const df*)c->HP,
                                                                       (df*)c->D_adj);
    } else {
      dim3 grid((unsigned)((ne + GT - 1) / GT), (unsigned)((no + GT - 1) / GT));
      FEP3M_CL k_adj_gemm<<<grid, PT, 0, s>>>(ne, o0, no, W, c->Ha64, (float*)c->D_adj);
    }
    typedef typename std::conditional<sizeof(T) == 4, float, df>::type DT;
    const DT* D = (const DT*)c->D_adj;
    switch (c->n_sr) {
      case 1: launch_adj_vertex<DT, 1>(c, z0, z1, D, ld, A, s); break;
      case 2: launch_adj_vertex<DT, 2>(c, z0, z1, D, ld, A, s); break;
      case 3: launch_adj_vertex<DT, 3>(c, z0, z1, D, ld, A, s); break;
      default: launch_adj_vertex<DT, 4>(c, z0, z1, D, ld, A, s); break;
    }
  }
  return cudaGetLastError();
}

// weights w = gU Q / 2 + gphi (sorted order), element deposits, adjoint right-hand side g64
cudaError_t adjoint_pre(fep3m_ctx* c, double gU, const double* gphi, cudaStream_t s) {
  const int n = c->n;
  const int64_t ne = (int64_t)n * n * n, N = c->N;
  // FP64: the scale of the screen adjoint's pairs, for weights gU Q / 2 from the charges' (their
  // largest is below 2^31 times their mean), else from the weights (adjoint_sweeps)
  c->weights_given = gphi != nullptr;
  double scale = 0.0;   // (none given)
  if (!c->weights_given)
    scale = gU == 0.0 ? 1.0 : std::ldexp(1.0, std::max(-900, std::min(900, 64 - std::ilogb(gU) + std::ilogb(c->q_scale))));
  FEP3M_CL k_weights<<<gsz(N), PT, 0, s>>>(N, gU, gphi, c->perm, c->Q_s, c->w_s, c->w_s32, scale,
                                           c->scal + kWeightScale);
  const bool dealt = deposit_dealt(ne, N);
  const int nrows = dealt ? 1 : PT / 32, run = dealt ? 0 : DEP_RUN, per = 32 * nrows;   // rows of 32 elements per CTA
  if (c->precision == FEP3M_MIXED) {
    FEP3M_CL k_elem_deposit<float><<<gsz(ne, per), PT, 0, s>>>(ne, nrows, run, c->start, c->count, (const float4*)c->part, c->w_s,
                                                               c->w_s32, (float*)c->W_el, (float2*)c->Wsum);
    FEP3M_CL k_node_assemble<float><<<dim3(3 * n, 3 * n), PT, 0, s>>>(n, (const float*)c->W_el, c->g64);
  } else {
    FEP3M_CL k_elem_deposit<double><<<gsz(ne, per), PT, 0, s>>>(ne, nrows, run, c->start, c->count, (const vec4<double>::type*)c->part,
                                                                c->w_s, c->w_s, (double*)c->W_el, nullptr);
    FEP3M_CL k_node_assemble<double><<<dim3(3 * n, 3 * n), PT, 0, s>>>(n, (const double*)c->W_el, c->g64);
  }
  return cudaGetLastError();
}

// the screen sweep A and (with singular) the singular adjoint potential: they
// need the deposit of the weights (adjoint_pre) but not the adjoint mesh
// solution, so they run concurrently with the mesh solves
cudaError_t adjoint_sweeps(fep3m_ctx* c, cudaStream_t s, bool singular) {
  const int n = c->n;
  const int64_t N = c->N;
  cudaStream_t keep = c->stream;
  c->stream = s;   // screen_adjoint issues on c->stream
  cudaError_t e;
  if (c->precision == FEP3M_MIXED) {
    e = screen_adjoint<float>(c, (const float*)c->W_el, (double*)c->A_el);
    if (e == cudaSuccess && singular)
      FEP3M_CL k_pair_adj_warp<float, true><<<(unsigned)((N + 7) / 8), PT, 0, s>>>(N, n, c->n_sr, (float)c->h, c->start,
                                                         (const float4*)c->part, c->ecoord, c->w_s, c->psi_s, c->gpsi_s);
  } else {
    if (c->weights_given) FEP3M_CL k_weight_scale<<<1, 1024, 0, s>>>(N, c->w_s, c->scal + kWeightScale);
    e = screen_adjoint<double>(c, (const double*)c->W_el, (double*)c->A_el);
    if (e == cudaSuccess && singular)
      FEP3M_CL k_pair_adj_warp<double, true><<<(unsigned)((N + 7) / 8), PT, 0, s>>>(N, n, c->n_sr, c->h, c->start,
                                                          (const vec4<double>::type*)c->part, c->ecoord, c->w_s,
                                                          c->psi_s, c->gpsi_s);
  }
  c->stream = keep;
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// the part that needs lam: the vertex adjoint mu = 4 pi (Mpq^T)^3 lam
cudaError_t adjoint_vertex(fep3m_ctx* c, cudaStream_t s) {
  const fep3m::Level& L0 = c->solv[1].mg.lv[0];
  return vertex_adjoint(c, c->lam64, c->mu_v, L0.t1, L0.t2, s);
}

// the charges' singular sums of an FP64 context into phi_s (and, with grad, E_s;
// half: also half of them into psi_s and gpsi_s)
static cudaError_t singular64(fep3m_ctx* c, bool grad, bool half, cudaStream_t s) {
  const int64_t N = c->N;
  PairCharge* ch = (PairCharge*)c->part_pairs;
  FEP3M_CL k_pair_charges<<<gsz(N), PT, 0, s>>>(N, (const vec4<double>::type*)c->part, c->ecoord, c->q_scale, ch);
  double *psi = half ? c->psi_s : nullptr, *gpsi = half ? c->gpsi_s : nullptr;
  auto k = grad ? k_singular64<true> : k_singular64<false>;
  FEP3M_CL k<<<(unsigned)((N + 7) / 8), PT, 0, s>>>(N, c->n, c->n_sr, c->inv_h / c->q_scale,
                                                    c->inv_h * c->inv_h / c->q_scale, c->start, ch, c->ecoord,
                                                    c->phi_s, c->E_s, psi, gpsi);
  return cudaGetLastError();
}

cudaError_t singular_sums(fep3m_ctx* c, cudaStream_t s) {
  const int64_t N = c->N;
  if (c->precision == FEP3M_FP64) return singular64(c, false, false, s);
  FEP3M_CL k_pair_adj_warp<float, false><<<(unsigned)((N + 7) / 8), PT, 0, s>>>(
      N, c->n, c->n_sr, (float)c->h, c->start, (const float4*)c->part, c->ecoord, c->Q_s, c->phi_s, nullptr);
  return cudaGetLastError();
}

// per-charge dLf/dx (times sign) and dLf/dQ
cudaError_t adjoint_final(fep3m_ctx* c, double gU, double* dpos, double* dQ, double sign, cudaStream_t s) {
  const int64_t N = c->N;
  if (c->precision == FEP3M_MIXED)
    FEP3M_CL k_final<float><<<gsz(N), PT, 0, s>>>(N, c->n, c->inv_h, gU, sign, (const float4*)c->part, c->perm, c->cell,
                                         c->w_s, c->phi_s, c->E_s, c->psi_s, c->gpsi_s, (const double*)c->mu_v,
                                         (const double*)c->A_el, dpos, dQ);
  else
    FEP3M_CL k_final<double><<<gsz(N), PT, 0, s>>>(N, c->n, c->inv_h, gU, sign, (const vec4<double>::type*)c->part, c->perm,
                                          c->cell, c->w_s, c->phi_s, c->E_s, c->psi_s, c->gpsi_s,
                                          (const double*)c->mu_v, (const double*)c->A_el, dpos, dQ);
  return cudaGetLastError();
}

}  // namespace fep3m
