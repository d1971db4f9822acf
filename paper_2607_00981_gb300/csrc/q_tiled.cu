// RCCSDT(Q) for small o (2 <= o <= 8 in FP32; in FP64, whose tiles are twice the size in shared
// memory, 2 <= o <= 6, and o = 7 up to v = 86): the ABC-ordered sum of q_energy.cu (same equations and
// notation) with the products of one virtual quadruple as register-tiled GEMMs.
//
// Each of the four products of r = P(X + Y) is symmetric under one exchange of its
// columns -- x1, x2 under (r k)(s l), y1 under (q j)(r k), y2 under (p i)(q j) -- so the
// 24 joint permutations are 12 distinct ones counted twice (which cancels the 1/2 of
// X and Y): half the multiply-adds of the permutation-by-permutation form, which is what
// bounds FP64 (the pipe takes 2 per clock and SM).
//
// One CTA per quadruple (persistent, round robin), labels L[0] <= .. <= L[3]:
//   X  for each position pair r < s the values t^{e L_r L_s}_{ikl} are read once, straight
//      from the virtual-triangular T3 (o^3 contiguous values per e), by the thread
//      that owns the columns (i, k, l); both orders of the other two positions form the
//      rows (2 o of them), whose integrals are staged in shared memory: 2 o x 2 register
//      tiles, K = v, then x2 (K = o) into the same tile.
//   Y  for each position s the columns (i, l) of t^{e L_s}_{il} against the rows
//      (p, j, k) of the three Wbar slices of the other labels, both staged in chunks of
//      e: 2 o x 2 register tiles, K = v, then y2 (K = o).
// Rows come in runs of o (padded to even), so operands load as pairs and FP32 multiplies
// as fma.f32x2.  A tile is stored to a shared buffer of its own (no two writers per
// element) and every thread then adds, in a fixed order, the permuted elements of its
// occupied tuples into registers.  The spin sum t~ has coefficients +-2^n and is unrolled
// with the permuted offsets as sums of compile-time multiples; FP32 takes it as a
// sum of three floats (error-free additions, about 70 bits; 24 FP64 additions per tuple made
// o=6 v=48 74.6 ms); the quotients by the energy denominators and every sum of energies
// are FP64.  (In two floats, with the quotients, 62.9 ms; now 69.1.)
//
// FP64 is bound by its pipe (41 ms at o=5 v=29 against 84 ms for 24 permutations).  FP32
// is bound by shared memory (16-byte row loads feeding two columns each) and by the
// latency between its barriers at two CTAs per SM: o=6 v=48, 247596 quadruples, 63 ms
// (13.2 TFLOP/s executed) against 589 ms for the permutation-by-permutation kernel; the
// intermediates with it 5.4 ms against 32 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "elem.cuh"
#include "q_tiled.h"

namespace rcc {
namespace {

// Spin summation 2 (2 - P_c^d)(2 - P_b^c - P_b^d)(2 - P_a^b - P_a^c - P_a^d) as
// sum_pi coef_pi R(O o pi^-1): inverse maps of the 24 orderings and coefficients.
struct SpinTab {
  int inv[24][4] = {};
  int coef[24] = {};
};
constexpr SpinTab make_spin() {
  SpinTab t;
  int perm[24][4] = {}, n = 0;
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b)
      for (int c = 0; c < 4; ++c) {
        if (a == b || a == c || b == c) continue;
        perm[n][0] = a, perm[n][1] = b, perm[n][2] = c, perm[n][3] = 6 - a - b - c;
        ++n;
      }
  int g[24] = {};
  g[0] = 1;
  for (int first = 0; first < 3; ++first) {  // apply 2 - sum_{y > first} P_first^y
    int out[24] = {};
    for (int i = 0; i < 24; ++i) {
      out[i] += 2 * g[i];
      for (int y = first + 1; y < 4; ++y)
        for (int k = 0; k < 24; ++k) {
          bool same = true;
          for (int x = 0; x < 4; ++x) {
            const int z = perm[i][x], w = z == first ? y : (z == y ? first : z);
            same = same && perm[k][x] == w;
          }
          if (same) out[k] -= g[i];
        }
    }
    for (int i = 0; i < 24; ++i) g[i] = out[i];
  }
  for (int i = 0; i < 24; ++i) {
    t.coef[i] = 2 * g[i];
    for (int x = 0; x < 4; ++x) t.inv[i][perm[i][x]] = x;
  }
  return t;
}
constexpr SpinTab kSpin = make_spin();
// f(coefficient, inverse map) for the orderings PI .. 23, both compile-time
template <int PI = 0, class F>
__device__ __forceinline__ void each_ordering(F f) {
  if constexpr (PI < 24) {
    constexpr int c = kSpin.coef[PI], i0 = kSpin.inv[PI][0], i1 = kSpin.inv[PI][1], i2 = kSpin.inv[PI][2],
                  i3 = kSpin.inv[PI][3];
    f(c, i0, i1, i2, i3);
    each_ordering<PI + 1>(f);
  }
}

__host__ __device__ __forceinline__ i64 tri2(i64 b, i64 c) { return c * (c + 1) / 2 + b; }  // b <= c
__host__ __device__ __forceinline__ i64 tri3q(i64 a, i64 b, i64 c) { return c * (c + 1) * (c + 2) / 6 + tri2(a, b); }
__host__ __device__ __forceinline__ i64 tet4(i64 d) { return d * (d + 1) * (d + 2) * (d + 3) / 24; }

// largest x with f(x) <= idx, 0 <= x < n
template <class F>
__device__ __forceinline__ int largest(int n, i64 idx, F f) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (f(mid) <= idx) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void decode3(i64 idx, int v, int& a, int& b, int& c) {  // a <= b <= c, colex
  c = largest(v, idx, [](i64 x) { return x * (x + 1) * (x + 2) / 6; });
  idx -= (i64)c * (c + 1) * (c + 2) / 6;
  b = largest(c + 1, idx, [](i64 x) { return x * (x + 1) / 2; });
  a = (int)(idx - (i64)b * (b + 1) / 2);
}

// (pq|rs) = sum_P L[P][p][q] L[P][r][s] over p >= q, r >= s, pair >= pair; all images written
__global__ void __launch_bounds__(256) k_qt_eri(const double* __restrict__ L, int naux, int n, double* __restrict__ G) {
  const i64 n2 = (i64)n * n, np = (i64)n * (n + 1) / 2;
  const i64 row = blockIdx.y;  // pair p >= q
  for (i64 pq = row; pq < np; pq += gridDim.y) {
    const int p = largest(n, pq, [](i64 x) { return x * (x + 1) / 2; }), q = (int)(pq - tri2(0, p));
    for (i64 rs = blockIdx.x * (i64)blockDim.x + threadIdx.x; rs <= pq; rs += (i64)gridDim.x * blockDim.x) {
      const int r = largest(n, rs, [](i64 x) { return x * (x + 1) / 2; }), s = (int)(rs - tri2(0, r));
      const double* lp = L + (i64)p * n + q;
      const double* lr = L + (i64)r * n + s;
      double x = 0.0;
#pragma unroll 4
      for (int P = 0; P < naux; ++P) x += lp[P * n2] * lr[P * n2];
      const i64 a = (i64)p * n + q, b = (i64)q * n + p, c = (i64)r * n + s, d = (i64)s * n + r;
      G[a * n2 + c] = x;
      G[a * n2 + d] = x;
      G[b * n2 + c] = x;
      G[b * n2 + d] = x;
      G[c * n2 + a] = x;
      G[c * n2 + b] = x;
      G[d * n2 + a] = x;
      G[d * n2 + b] = x;
    }
  }
}

// virtual-triangular T3, [tri3(a <= b <= c)][i][j][k] = t^{abc}_{ijk}: a warp per block
template <typename S, typename T>
__global__ void __launch_bounds__(256) k_qt_t3v(const S* __restrict__ t3c, int o, int v, i64 nv3, T* __restrict__ out) {
  const int o3 = o * o * o, lane = threadIdx.x & 31;
  const i64 V3 = (i64)v * v * v;
  for (i64 blk = blockIdx.x * 8ll + (threadIdx.x >> 5); blk < nv3; blk += gridDim.x * 8ll) {
    int a0, b0, c0;
    decode3(blk, v, a0, b0, c0);
    for (int x = lane; x < o3; x += 32) {
      int k = x % o, j = (x / o) % o, i = x / (o * o), a = a0, b = b0, c = c0;
      if (i > j) { int t = i; i = j; j = t; t = a; a = b; b = t; }
      if (j > k) { int t = j; j = k; k = t; t = b; b = c; c = t; }
      if (i > j) { int t = i; i = j; j = t; t = a; a = b; b = t; }
      out[blk * o3 + x] = (T)t3c[tri3q(i, j, k) * V3 + ((i64)a * v + b) * v + c];
    }
  }
}

// Integral and t2 layouts (see QtArgs); kind 0 A1, 1 A2, 2 Vv, 3 T2e, 4 T2m
template <typename T>
__global__ void k_qt_layout(int kind, const double* __restrict__ G, const double* __restrict__ t2, int o, int v,
                            T* __restrict__ out, i64 tot) {
  const i64 n1 = o + v, n2 = n1 * n1, n3 = n2 * n1;
  for (i64 x = blockIdx.x * (i64)blockDim.x + threadIdx.x; x < tot; x += (i64)gridDim.x * blockDim.x) {
    double val;
    i64 r = x;
    if (kind == 0) {  // [p][q][e][j] = (pe|qj)
      const int j = (int)(r % o), e = (int)((r /= o) % v), q = (int)((r /= v) % v), p = (int)(r / v);
      val = G[(o + p) * n3 + (o + e) * n2 + (o + q) * n1 + j];
    } else if (kind == 1) {  // [p][i][m][j] = (pi|mj)
      const int j = (int)(r % o), m = (int)((r /= o) % o), i = (int)((r /= o) % o), p = (int)(r / o);
      val = G[(o + p) * n3 + i * n2 + m * n1 + j];
    } else if (kind == 2) {  // [p][q][i][j] = (pi|qj)
      const int j = (int)(r % o), i = (int)((r /= o) % o), q = (int)((r /= o) % v), p = (int)(r / v);
      val = G[(o + p) * n3 + i * n2 + (o + q) * n1 + j];
    } else if (kind == 3) {  // [s][e][(i,l), padded to even] = t_il^es
      const int rc = (o * o + 1) / 2 * 2, il = (int)(r % rc), e = (int)((r /= rc) % v), s = (int)(r / v);
      val = il < o * o ? t2[((i64)il * v + e) * v + s] : 0.0;
    } else {  // [r][s][m][l] = t_ml^rs
      const int l = (int)(r % o), m = (int)((r /= o) % o), s = (int)((r /= o) % v), rr = (int)(r / v);
      val = t2[(((i64)m * o + l) * v + rr) * v + s];
    }
    out[x] = (T)val;
  }
}

// W1[a][tri(b <= c)][e][j][k, padded to even] = Wbar^{abc}_{ejk}.  One CTA per (a, b <= c): the sum over f
// as a v x o^2 product with K = 2 v (both orders of b, c), 4 x 4 register tiles, operands
// staged in chunks of f; the four sums over m (K = o) per element from L1 / L2.
constexpr int kW1FC = 8;
template <typename T>
__global__ void __launch_bounds__(128) k_qt_wbar1(const T* __restrict__ G, const T* __restrict__ t2, int o, int v,
                                                  T* __restrict__ W1) {
  extern __shared__ __align__(16) unsigned char qt_smem[];
  const int o2 = o * o, vp = (v + 3) & ~3, op = (o2 + 3) & ~3;
  T* Gs = (T*)qt_smem;          // [kW1FC][vp]
  T* Ts = Gs + kW1FC * vp;      // [kW1FC][op]
  const i64 n1 = o + v, n2 = n1 * n1, n3 = n2 * n1, V2 = (i64)v * v;
  const int a = blockIdx.y;
  const i64 bc = blockIdx.x;
  const int c = largest(v, bc, [](i64 x) { return x * (x + 1) / 2; }), b = (int)(bc - tri2(0, c));
  const int ne = vp / 4, nj = op / 4;
  const int po = (o + 1) / 2 * 2, ro = o * po;
  T* out = W1 + ((i64)a * tri2(0, v) + bc) * (i64)v * ro;
  for (int it0 = 0; it0 < ne * nj; it0 += 128) {
    const int it = it0 + threadIdx.x, te = it % ne * 4, tj = it / ne * 4;
    const bool live = it < ne * nj;
    T acc[4][4] = {};
    for (int half = 0; half < 2; ++half) {  // (ae|bf) t_jk^fc, then (ae|cf) t_kj^fb
      const int x = half ? c : b, y = half ? b : c;
      for (int f0 = 0; f0 < v; f0 += kW1FC) {
        __syncthreads();
        for (int q = threadIdx.x; q < kW1FC * vp; q += 128) {
          const int f = q % kW1FC, e = q / kW1FC;  // f contiguous in G
          Gs[f * vp + e] = (e < v && f0 + f < v) ? G[(o + a) * n3 + (o + e) * n2 + (o + x) * n1 + o + f0 + f] : (T)0;
        }
        for (int q = threadIdx.x; q < kW1FC * op; q += 128) {
          const int f = q / op, jk = q % op, j = half ? jk % o : jk / o, k = half ? jk / o : jk % o;
          Ts[f * op + jk] = (jk < o2 && f0 + f < v) ? t2[((i64)j * o + k) * V2 + (i64)(f0 + f) * v + y] : (T)0;
        }
        __syncthreads();
        if (live)
#pragma unroll
          for (int f = 0; f < kW1FC; ++f) {
            T g[4], t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) g[u] = Gs[f * vp + te + u], t[u] = Ts[f * op + tj + u];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int w = 0; w < 4; ++w) acc[u][w] = fma(g[u], t[w], acc[u][w]);
          }
      }
    }
    if (!live) continue;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int jk = tj + w, j = jk / o, k = jk % o;
      if (jk >= o2) break;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = te + u;
        if (e >= v) break;
        T s = 0;
        for (int m = 0; m < o; ++m) {
          const i64 mk = ((i64)m * o + k) * V2, mj = ((i64)m * o + j) * V2;
          const T* gme = G + m * n3 + (o + e) * n2;              // (me|..)
          const T* gae = G + (o + a) * n3 + (o + e) * n2 + m * n1;  // (ae|m.)
          s = fma(gme[(o + b) * n1 + j], t2[mk + (i64)a * v + c], s);
          s = fma(gae[j], t2[mk + (i64)b * v + c], s);
          s = fma(gme[(o + c) * n1 + k], t2[mj + (i64)a * v + b], s);
          s = fma(gae[k], t2[mj + (i64)c * v + b], s);
        }
        out[(i64)e * ro + j * po + k] = (T)0.5 * acc[u][w] - s;
      }
    }
  }
}

// W2[tri(q <= r)][m][i][j][k] = Wbar^{qrm}_{jki} = -1/2 sum_n ((mi|nj) t_nk^qr + (mi|nk) t_nj^rq)
template <typename T>
__global__ void k_qt_wbar2(const T* __restrict__ G, const T* __restrict__ t2, int o, int v, T* __restrict__ W2) {
  const i64 n1 = o + v, n2 = n1 * n1, n3 = n2 * n1, V2 = (i64)v * v, o4 = (i64)o * o * o * o;
  const i64 tot = tri2(0, v) * o4;
  for (i64 x = blockIdx.x * (i64)blockDim.x + threadIdx.x; x < tot; x += (i64)gridDim.x * blockDim.x) {
    const i64 qr = x / o4;
    const int y = (int)(x - qr * o4);
    const int k = y % o, j = (y / o) % o, i = (y / (o * o)) % o, m = y / (o * o * o);
    const int r = largest(v, qr, [](i64 z) { return z * (z + 1) / 2; }), q = (int)(qr - tri2(0, r));
    T s = 0;
    for (int n = 0; n < o; ++n) {
      s = fma(G[m * n3 + i * n2 + n * n1 + j], t2[((i64)n * o + k) * V2 + (i64)q * v + r], s);
      s = fma(G[m * n3 + i * n2 + n * n1 + k], t2[((i64)n * o + j) * V2 + (i64)r * v + q], s);
    }
    W2[x] = (T)-0.5 * s;
  }
}

template <typename T>
struct QtArgs {
  i64 ntuple;       // sorted quadruples, the ones of zero weight included
  int v, nx;        // nx: X rounds staged ahead (3, or 1 where shared memory is short)
  const double* eps;
  const T* t3v;     // [tri3][o^3]
  const T* A1;      // [p][q][e][j]
  const T* A2;      // [p][i][m][j]
  const T* Vv;      // [p][q][i][j]
  const T* W1;      // [a][tri(b <= c)][e][j][k], k padded to even
  const T* W2;      // [tri(q <= r)][m][i][j][k]
  const T* T2e;     // [s][e][i][l], (i, l) padded to even
  const T* T2m;     // [r][s][m][l]
  double* partial;  // [grid]
};

// Threads per CTA: the items of one X round, 2 ceil(o^3 / 2), in whole warps; half of them for
// o = 8 (512), where 512 threads would leave 128 registers, less than the tiles take.  CTAs
// per SM that the registers are cut for: as many as their threads fill (FP32, o <= 4), then
// as many as shared memory takes (o = 5 four, o = 6 two, o >= 7 one; FP64 one from o = 5 on).
// Against a thread per tuple with 24 permutations: o = 2, v = 60 16.4 ms (463), o = 3, v = 20
// 0.54 (4.4), o = 4, v = 30 2.6 (27.1), o = 5, v = 30 6.1 (42.4), o = 7, v = 24 9.2 (43.4), o = 8,
// v = 20 6.5 (41.1); in FP64 o = 6, v = 20 16.4 (36.8).
constexpr int qt_threads(int O) { return O <= 3 ? 32 : O == 4 ? 64 : O == 5 ? 128 : O == 6 ? 224 : O == 7 ? 352 : 256; }
template <typename T>
constexpr int qt_min_ctas(int O) {
  return sizeof(T) == 8 ? (O <= 4 ? 4 : 1) : O <= 3 ? 16 : O == 4 ? 8 : O == 5 ? 4 : O == 6 ? 2 : 1;
}
constexpr int kQtEC = 16;  // e values staged at a time in phase Y

template <typename T, int O>
struct QtCfg {
  static constexpr int O2 = O * O, O3 = O2 * O, O4 = O2 * O2, OP = (O + 1) / 2 * 2, THREADS = qt_threads(O);
  static constexpr int CH = (O3 + 1) / 2;                      // X: columns c and c + CH per item
  static constexpr int RT = 2 * OP;                            // rows of an item: two runs
  static constexpr int RG = (3 * O + 1) / 2, CG = (O2 + 1) / 2;  // Y: run pairs, column pairs
  static constexpr int RW = RG * RT, RC = 2 * CG;
  // shared memory (elements): tile buffers | energies (2 per tuple) | X | Y | staged operands
  static constexpr int BUF = ((4 * O4 > RW * RC ? 4 * O4 : RW * RC) + 3) / 4 * 4;
  static constexpr int EPS = sizeof(T) == 4 ? (2 * O4 + 3) / 4 * 4 : (O4 + 3) / 4 * 4;
  static constexpr int O4P = (O4 + 3) / 4 * 4;                 // X and Y sums of the tuples
  static constexpr int RO = O * OP, YST = kQtEC * (3 * RO + RC);  // a slice's values per e; a staged chunk
  static constexpr int VST = (12 * O2 + 3) / 4 * 4, A2 = 4 * O2 * OP;
  // nx: staged X operands, of all three rounds (3) or of the current one (1)
  static size_t smem(int v, int nx) {
    return sizeof(T) * (size_t)(BUF + EPS + 2 * O4P + VST + A2 + 2 * YST + nx * 2 * v * RT) +
           2 * (size_t)v * sizeof(int);
  }
};

// Pairs of consecutive rows: FP32 multiply-adds two at a time (fma.f32x2), FP64 one by one.
template <typename T>
struct Pair;
template <>
struct Pair<float> {
  float2 v;
  __device__ __forceinline__ void fma(const Pair& w, const Pair& t) {
    unsigned long long a = *(unsigned long long*)&v, b = *(const unsigned long long*)&w.v,
                       c = *(const unsigned long long*)&t.v;
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a) : "l"(b), "l"(c));
    *(unsigned long long*)&v = a;
  }
};
template <>
struct Pair<double> {
  double2 v;
  __device__ __forceinline__ void fma(const Pair& w, const Pair& t) {
    v.x = ::fma(w.v.x, t.v.x, v.x);
    v.y = ::fma(w.v.y, t.v.y, v.y);
  }
};
template <typename T>
__device__ __forceinline__ Pair<T> both(T x) {
  Pair<T> p;
  p.v.x = x;
  p.v.y = x;
  return p;
}
// N pairs from p, aligned to the widest of 8 / 16 bytes that N allows
template <int N>
__device__ __forceinline__ void load_pairs(const float* p, Pair<float> (&x)[N]) {
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int q = 0; q < N / 2; ++q) {
      const float4 f = *(const float4*)(p + 4 * q);
      x[2 * q].v = make_float2(f.x, f.y);
      x[2 * q + 1].v = make_float2(f.z, f.w);
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) x[q].v = *(const float2*)(p + 2 * q);
  }
}
template <int N>
__device__ __forceinline__ void load_pairs(const double* p, Pair<double> (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) x[q].v = *(const double2*)(p + 2 * q);
}

// Asynchronous copies of N values (4, 8 or 16 bytes) into shared memory
template <int N, typename T>
__device__ __forceinline__ void copy_async(T* dst, const T* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(N * (int)sizeof(T))
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait(int pending) {  // at most `pending` groups still in flight
  if (pending >= 3) asm volatile("cp.async.wait_group 3;" ::: "memory");
  else if (pending == 2) asm volatile("cp.async.wait_group 2;" ::: "memory");
  else if (pending == 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
  else asm volatile("cp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ float two_sum(float& h, float x) {  // h += x; what its rounding leaves
  const float s = h + x, bp = s - h, e = (h - (s - bp)) + (x - bp);
  h = s;
  return e;
}

template <typename T, int O>
__global__ void __launch_bounds__(qt_threads(O), qt_min_ctas<T>(O)) k_qt_main(const QtArgs<T> a) {
  typedef QtCfg<T, O> C;
  constexpr int O2 = C::O2, O3 = C::O3, O4 = C::O4, OP = C::OP, HP = OP / 2, RT = C::RT, TH = C::THREADS;
  constexpr int CH = C::CH, RO = C::RO, RC = C::RC, RG = C::RG, CG = C::CG, EC = kQtEC;
  extern __shared__ __align__(16) unsigned char qt_smem[];
  const int v = a.v, tid = threadIdx.x;
  T* buf = (T*)qt_smem;
  double* seps = (double*)(buf + C::BUF);  // sum of the occupied energies of a tuple
  T* xs = buf + C::BUF + C::EPS;    // sums over the rounds, each tuple's by its own thread
  T* ys = xs + C::O4P;
  T* Vs = ys + C::O4P;              // [6][O2] integrals, [6][O2] t2
  T* A2s = Vs + C::VST;             // [4][i][m][OP]
  T* Yst = A2s + C::A2;             // two chunks of Wbar rows [EC][RW] and t2 columns [EC][RC]
  T* As = Yst + 2 * C::YST;         // [round][2][v][2][OP]
  int* sblk = (int*)(As + a.nx * 2 * v * RT);  // [2][v] block of sorted(e, r, s)
  __shared__ double red[32];
  __shared__ int slab[2][5];
  __shared__ i64 sqi[2];
  // the first quadruple qi, qi + grid, ... with a nonzero degeneracy factor: its labels
  auto next = [&](i64 qi, int w) {
    for (; qi < a.ntuple; qi += gridDim.x) {
      int L[4];
      L[3] = largest(v, qi, [](i64 x) { return tet4(x); });
      decode3(qi - tet4(L[3]), v, L[0], L[1], L[2]);
      const int eq = (L[0] == L[1]) + (L[1] == L[2]) + (L[2] == L[3]);
      const int fac = eq == 0 ? 24 : eq == 1 ? 12 : (eq == 2 && L[1] != L[2]) ? 6 : 0;
      if (!fac) continue;  // three or four equal labels
      for (int q = 0; q < 4; ++q) slab[w][q] = L[q];
      slab[w][4] = fac;
      break;
    }
    sqi[w] = qi;
  };
  constexpr int CN = O % 2 == 0 ? 2 : 1;  // values per copy
  // position pairs of X's rounds: (0,1) (2,3) | (0,2) (1,3) | (0,3) (1,2)
  auto pair_r = [](int round, int h) { return h == 0 ? 0 : (round == 0 ? 2 : 1); };
  auto pair_s = [](int round, int h) { return h == 0 ? round + 1 : (round == 2 ? 2 : 3); };
  auto stage_x = [&](const int* L, int round, T* dst) {  // [h][e][order][j] of the complementary pairs
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int p = L[pair_r(round, h ^ 1)], q = L[pair_s(round, h ^ 1)];
      const T* pq = a.A1 + ((i64)p * v + q) * v * O;
      const T* qp = a.A1 + ((i64)q * v + p) * v * O;
      for (int x = tid; x < v * O / CN; x += TH) {
        const int e = x * CN / O, j = x * CN % O;
        copy_async<CN>(dst + (h * v + e) * RT + j, pq + x * CN);
        copy_async<CN>(dst + (h * v + e) * RT + OP + j, qp + x * CN);
      }
    }
  };
  const int nch = (v + EC - 1) / EC, nc = 4 * nch;
  auto stage_y = [&](const int* L, int c) {  // chunk c: position c / nch, e from (c % nch) EC
    const int s = c / nch, e0 = c % nch * EC, ne = min(EC, v - e0);
    const int l0 = L[s == 0 ? 1 : 0], l1 = L[s <= 1 ? 2 : 1], l2 = L[s <= 2 ? 3 : 2];
    T* Ws = Yst + (c & 1) * C::YST;
    T* Ts = Ws + 3 * EC * RO;
    // (slices and columns are contiguous: flat copies of two values)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int p = q == 0 ? l0 : (q == 1 ? l1 : l2), b = q == 0 ? l1 : l0, cc = q == 2 ? l1 : l2;
      const T* w = a.W1 + (((i64)p * tri2(0, v) + tri2(b, cc)) * v + e0) * RO;
      for (int x = tid * 2; x < ne * RO; x += TH * 2) copy_async<2>(Ws + q * EC * RO + x, w + x);
    }
    const T* t2 = a.T2e + ((i64)L[s] * v + e0) * RC;
    for (int x = tid * 2; x < ne * RC; x += TH * 2) copy_async<2>(Ts + x, t2 + x);
  };
  // everything of a quadruple that can be under way before it starts
  auto prefetch = [&](int w) {
    const int L[4] = {slab[w][0], slab[w][1], slab[w][2], slab[w][3]};
    for (int x = tid; x < 4 * O3 / CN; x += TH) {
      const int y = x * CN, p = y / O3, z = y % O3;
      copy_async<CN>(A2s + (p * O2 + z / O) * OP + z % O, a.A2 + (i64)L[p] * O3 + z);
    }
    for (int r = 0; r < a.nx; ++r) {
      stage_x(L, r, As + r * 2 * v * RT);
      copy_commit();
    }
    stage_y(L, 0);
    copy_commit();
  };
  for (int el = tid; el < O4; el += TH) {
    const double e = a.eps[el / O3] + a.eps[el / O2 % O] + a.eps[el / O % O] + a.eps[el % O];
    seps[el] = e;
  }
  if (tid == 0) next(blockIdx.x, 0);
  __syncthreads();
  double total = 0.0;
  if (sqi[0] < a.ntuple) prefetch(0);
  for (int par = 0; sqi[par] < a.ntuple; par ^= 1) {
    const int L[4] = {slab[par][0], slab[par][1], slab[par][2], slab[par][3]};
    const int fac = slab[par][4];
    if (tid == 0) next(sqi[par] + gridDim.x, par ^ 1);
    // dst (+)= f(occupied indices) for this thread's tuples (rolled: the unrolled form kept
    // every tuple's offsets in registers across the whole quadruple and spilled)
    auto tuples = [&](T* dst, bool first, auto f) {
#pragma unroll 1
      for (int el = tid; el < O4; el += TH) {
        const int oc[4] = {el / O3, el / O2 % O, el / O % O, el % O};
        const T x = f(oc);
        dst[el] = first ? x : dst[el] + x;
      }
    };
    // ---- X: three rounds of two position pairs r < s; the others p < q
#pragma unroll 1
    for (int round = 0; round < 3; ++round) {
      const int pr[2] = {pair_r(round, 0), pair_r(round, 1)}, ps[2] = {pair_s(round, 0), pair_s(round, 1)};
      __syncthreads();  // the buffers of the previous phase are consumed
      if (a.nx == 1 && round) {
        stage_x(L, round, As);
        copy_commit();
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = L[pr[h]], s = L[ps[h]];
        for (int e = tid; e < v; e += TH)
          sblk[h * v + e] = (int)((e <= r ? tri3q(e, r, s) : (e <= s ? tri3q(r, e, s) : tri3q(r, s, e))) * O3);
      }
      copy_wait(a.nx == 3 ? 3 - round : (round ? 0 : 1));  // behind this round: later rounds, Y's first chunk
      __syncthreads();
      for (int it = tid; it < 2 * CH; it += TH) {
        const int h = it / CH, c0 = it % CH, c1 = min(c0 + CH, O3 - 1);
        const int p = h ? pr[0] : pr[1], q = h ? ps[0] : ps[1], r = L[h ? pr[1] : pr[0]], s = L[h ? ps[1] : ps[0]];
        const int i0 = c0 / O2, kl0 = c0 % O2, i1 = c1 / O2, kl1 = c1 % O2;
        Pair<T> acc[2][2][HP];  // [column][order][row pair]
#pragma unroll
        for (int x = 0; x < 2 * HP; ++x) acc[0][x / HP][x % HP] = acc[1][x / HP][x % HP] = both<T>((T)0);
        const int* bt = sblk + h * v;
        const T* Ah = As + ((a.nx == 3 ? round * 2 : 0) + h) * v * RT;
        // x1 = sum_e v^{pq}_{ej} t^{ers}_{ikl}; the stored order of (i, k, l) by the range of e
        auto sweep = [&](int e0, int e1, int f0, int f1) {
#pragma unroll 8
          for (int e = e0; e < e1; ++e) {
            const T* tb = a.t3v + bt[e];
            const Pair<T> t0 = both<T>(__ldg(tb + f0)), t1 = both<T>(__ldg(tb + f1));
            Pair<T> w[OP];
            load_pairs(Ah + e * RT, w);
#pragma unroll
            for (int x = 0; x < OP; ++x) {
              acc[0][x / HP][x % HP].fma(w[x], t0);
              acc[1][x / HP][x % HP].fma(w[x], t1);
            }
          }
        };
        const int k0 = kl0 / O, l0 = kl0 % O, k1 = kl1 / O, l1 = kl1 % O;
        sweep(0, r + 1, c0, c1);
        sweep(r + 1, s + 1, (k0 * O + i0) * O + l0, (k1 * O + i1) * O + l1);
        sweep(s + 1, v, kl0 * O + i0, kl1 * O + i1);
        // x2 = sum_m v^{pm}_{ij} t^{qrs}_{mkl}, and with p and q exchanged
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const int pp = w ? q : p, qq = L[w ? p : q];
          const int mst = qq <= r ? O2 : (qq <= s ? O : 1);  // stride of m in the sorted block
          const T* tb = a.t3v + bt[qq];
          const int b0 = qq <= r ? kl0 : (qq <= s ? k0 * O2 + l0 : kl0 * O);
          const int b1 = qq <= r ? kl1 : (qq <= s ? k1 * O2 + l1 : kl1 * O);
          const T* a0 = A2s + (pp * O + i0) * O * OP;
          const T* a1 = A2s + (pp * O + i1) * O * OP;
          T u0[O], u1[O];  // all loads before the products
#pragma unroll
          for (int m = 0; m < O; ++m) {
            u0[m] = -__ldg(tb + b0 + m * mst);
            u1[m] = -__ldg(tb + b1 + m * mst);
          }
#pragma unroll
          for (int m = 0; m < O; ++m) {
            const Pair<T> t0 = both<T>(u0[m]), t1 = both<T>(u1[m]);
            Pair<T> w0[HP], w1[HP];
            load_pairs(a0 + m * OP, w0);
            load_pairs(a1 + m * OP, w1);
#pragma unroll
            for (int x = 0; x < HP; ++x) {
              acc[0][w][x].fma(w0[x], t0);
              acc[1][w][x].fma(w1[x], t1);
            }
          }
        }
        // buffer (h, order)[j][ikl]
        T* bo = buf + h * 2 * O4 + c0;
        const bool two = c0 + CH < O3;
#pragma unroll
        for (int w = 0; w < 2; ++w)
#pragma unroll
          for (int j = 0; j < O; ++j) {
            const int at = w * O4 + j * O3;
            bo[at] = j & 1 ? acc[0][w][j / 2].v.y : acc[0][w][j / 2].v.x;
            if (two) bo[at + CH] = j & 1 ? acc[1][w][j / 2].v.y : acc[1][w][j / 2].v.x;
          }
      }
      __syncthreads();
      auto add = [&](auto P0, auto Q0, auto P1, auto Q1) {  // pair 0 = (P0, Q0), pair 1 = (P1, Q1)
        constexpr int p0 = decltype(P0)::value, q0 = decltype(Q0)::value, p1 = decltype(P1)::value,
                      q1 = decltype(Q1)::value;
        tuples(xs, round == 0, [&](const int* oc) {
          const int kl0 = oc[p0] * O + oc[q0], kl1 = oc[p1] * O + oc[q1];
          T s = buf[oc[q1] * O3 + oc[p1] * O2 + kl0];
          s += buf[O4 + oc[p1] * O3 + oc[q1] * O2 + kl0];
          s += buf[2 * O4 + oc[q0] * O3 + oc[p0] * O2 + kl1];
          s += buf[3 * O4 + oc[p0] * O3 + oc[q0] * O2 + kl1];
          return s;
        });
      };
      typedef std::integral_constant<int, 0> I0;
      typedef std::integral_constant<int, 1> I1;
      typedef std::integral_constant<int, 2> I2;
      typedef std::integral_constant<int, 3> I3;
      if (round == 0) add(I0{}, I1{}, I2{}, I3{});
      else if (round == 1) add(I0{}, I2{}, I1{}, I3{});
      else add(I0{}, I3{}, I1{}, I2{});
    }
    // ---- Y: position s; the others x0 < x1 < x2, each in turn the label p of t^{p ...}
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      const int x0 = s == 0 ? 1 : 0, x1 = s <= 1 ? 2 : 1, x2 = s <= 2 ? 3 : 2;
      const int l0 = L[x0], l1 = L[x1], l2 = L[x2];
      constexpr int NI = (RG * CG + TH - 1) / TH;
      Pair<T> acc[NI][2][2][HP];  // [item][column][run][row pair]
#pragma unroll
      for (int n = 0; n < NI; ++n)
#pragma unroll
        for (int x = 0; x < OP; ++x) acc[n][0][x / HP][x % HP] = acc[n][1][x / HP][x % HP] = both<T>((T)0);
      for (int c = s * nch; c < (s + 1) * nch; ++c) {
        const int ne = min(EC, v - (c - s * nch) * EC);
        const T* Ws = Yst + (c & 1) * C::YST;
        const T* Ts = Ws + 3 * EC * RO;
        __syncthreads();  // the other chunk buffer is consumed
        if (c + 1 < nc) {
          stage_y(L, c + 1);
          copy_commit();
        }
        copy_wait(c + 1 < nc ? 1 : 0);
        __syncthreads();
#pragma unroll
        for (int n = 0; n < NI; ++n) {
          const int it = tid + n * TH;
          if (it < RG * CG) {
            // runs (p, j), (p', j') of the item (for even O of one label, side by side)
            const int run0 = it / CG * 2, run1 = min(run0 + 1, 3 * O - 1);
            const T* wr0 = Ws + run0 / O * EC * RO + run0 % O * OP;
            const T* wr1 = Ws + run1 / O * EC * RO + run1 % O * OP;
            const T* tc = Ts + it % CG * 2;
#pragma unroll 2
            for (int e = 0; e < ne; ++e) {
              Pair<T> t[1], wv[OP];
              load_pairs(tc + e * RC, t);
              if constexpr (O % 2 == 0) {
                load_pairs(wr0 + e * RO, wv);
              } else {
                Pair<T> lo[HP], hi[HP];
                load_pairs(wr0 + e * RO, lo);
                load_pairs(wr1 + e * RO, hi);
#pragma unroll
                for (int x = 0; x < HP; ++x) wv[x] = lo[x], wv[HP + x] = hi[x];
              }
              const Pair<T> t0 = both<T>(t[0].v.x), t1 = both<T>(t[0].v.y);
#pragma unroll
              for (int x = 0; x < OP; ++x) {
                acc[n][0][x / HP][x % HP].fma(wv[x], t0);
                acc[n][1][x / HP][x % HP].fma(wv[x], t1);
              }
            }
          }
        }
      }
      // y2 = sum_m Wbar^{qrm}_{jki} t^{ps}_{ml}, runs (p, j), columns (i, l); then the
      // buffer [run][k][column]
#pragma unroll
      for (int n = 0; n < NI; ++n) {
        const int it = tid + n * TH;
        if (it < RG * CG) {
          const int run0 = it / CG * 2, col0 = it % CG * 2;
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const int run = min(run0 + g, 3 * O - 1), pi = run / O, j = run % O;
            const int lp = pi == 0 ? l0 : (pi == 1 ? l1 : l2), lq = pi == 0 ? l1 : l0, lr = pi == 2 ? l1 : l2;
            const T* w2 = a.W2 + tri2(lq, lr) * O4 + j * O;
            const T* tm = a.T2m + ((i64)lp * v + L[s]) * O2;
            const int ca = min(col0, O2 - 1), cb = min(col0 + 1, O2 - 1);
            T ua[O], ub[O];
#pragma unroll
            for (int m = 0; m < O; ++m) {
              ua[m] = -__ldg(tm + m * O + ca % O);
              ub[m] = -__ldg(tm + m * O + cb % O);
            }
            const T* wa = w2 + ca / O * O2;
            const T* wb = w2 + cb / O * O2;
            auto row = [&](const T* w, int x) {
              Pair<T> p;
              if constexpr (O % 2 == 0) {
                if constexpr (sizeof(T) == 4) p.v = __ldg((const float2*)(w + 2 * x));
                else p.v = __ldg((const double2*)(w + 2 * x));
              } else {
                p.v.x = __ldg(w + 2 * x);
                p.v.y = 2 * x + 1 < O ? __ldg(w + 2 * x + 1) : (T)0;
              }
              return p;
            };
#pragma unroll
            for (int m = 0; m < O; ++m) {
              const Pair<T> ta = both<T>(ua[m]), tb = both<T>(ub[m]);
#pragma unroll
              for (int x = 0; x < HP; ++x) {
                const Pair<T> p = row(wa + m * O3, x);
                acc[n][0][g][x].fma(p, ta);
                // (even O: both columns have one i)
                acc[n][1][g][x].fma(O % 2 == 0 ? p : row(wb + m * O3, x), tb);
              }
            }
            T* bo = buf + (run0 + g) * OP * RC + col0;
#pragma unroll
            for (int k = 0; k < O; ++k) {
              bo[k * RC] = k & 1 ? acc[n][0][g][k / 2].v.y : acc[n][0][g][k / 2].v.x;
              bo[k * RC + 1] = k & 1 ? acc[n][1][g][k / 2].v.y : acc[n][1][g][k / 2].v.x;
            }
          }
        }
      }
      __syncthreads();
      auto add = [&](auto X0, auto X1, auto X2) {
        constexpr int y0 = decltype(X0)::value, y1 = decltype(X1)::value, y2 = decltype(X2)::value, ss = 6 - y0 - y1 - y2;
        tuples(ys, s == 0, [&](const int* oc) {
          T x = buf[(oc[y1] * OP + oc[y2]) * RC + oc[y0] * O + oc[ss]];
          x += buf[((O + oc[y0]) * OP + oc[y2]) * RC + oc[y1] * O + oc[ss]];
          x += buf[((2 * O + oc[y0]) * OP + oc[y1]) * RC + oc[y2] * O + oc[ss]];
          return x;
        });
      };
      typedef std::integral_constant<int, 0> I0;
      typedef std::integral_constant<int, 1> I1;
      typedef std::integral_constant<int, 2> I2;
      typedef std::integral_constant<int, 3> I3;
      if (s == 0) add(I1{}, I2{}, I3{});
      else if (s == 1) add(I0{}, I2{}, I3{});
      else if (s == 2) add(I0{}, I1{}, I3{});
      else add(I0{}, I1{}, I2{});
      // (the next round stages after a barrier; its buffer stores come later still)
    }
    // ---- R to shared memory, Z = X + V, then f sum_O Z(O) t~(O)
    __syncthreads();
    for (int el = tid; el < O4; el += TH) buf[el] = xs[el] + ys[el];
    for (int x = tid; x < 6 * O2; x += TH) {  // the pairs p < q with v^{pq}_{ij} t^{rs}_{kl}
      const int pq = x / O2, p = pq < 3 ? 0 : (pq < 5 ? 1 : 2), q = pq < 3 ? pq + 1 : (pq < 5 ? pq - 1 : 3);
      const int r = p == 0 ? (q == 1 ? 2 : 1) : 0, s = 6 - p - q - r;
      Vs[x] = a.Vv[((i64)L[p] * v + L[q]) * O2 + x % O2];
      Vs[6 * O2 + x] = a.T2m[((i64)L[r] * v + L[s]) * O2 + x % O2];
    }
    if (sqi[par ^ 1] < a.ntuple) prefetch(par ^ 1);  // flies over the spin sum
    __syncthreads();
    const double ev = a.eps[O + L[0]] + a.eps[O + L[1]] + a.eps[O + L[2]] + a.eps[O + L[3]];
    double part = 0.0;
#pragma unroll 1
    for (int el = tid; el < O4; el += TH) {
      const int oc[4] = {el / O3, el / O2 % O, el / O % O, el % O};
      T z = xs[el];
#pragma unroll
      for (int pq = 0; pq < 6; ++pq) {
        const int p = pq < 3 ? 0 : (pq < 5 ? 1 : 2), q = pq < 3 ? pq + 1 : (pq < 5 ? pq - 1 : 3);
        const int r = p == 0 ? (q == 1 ? 2 : 1) : 0, s = 6 - p - q - r;
        z = fma(Vs[pq * O2 + oc[p] * O + oc[q]], Vs[(6 + pq) * O2 + oc[r] * O + oc[s]], z);
      }
      // offsets of the permuted tuples: sum over positions of occ O^k, k from the ordering
      int mu[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) mu[q][0] = oc[q], mu[q][1] = oc[q] * O, mu[q][2] = oc[q] * O2, mu[q][3] = oc[q] * O3;
      auto at = [&](int i0, int i1, int i2, int i3) { return buf[mu[i0][3] + mu[i1][2] + mu[i2][1] + mu[i3][0]]; };
      double s = 0.0;
      if constexpr (sizeof(T) == 8) {
        each_ordering([&](int c, int i0, int i1, int i2, int i3) { s = fma((double)c, at(i0, i1, i2, i3), s); });
        part += z * s / (seps[el] - ev);
      } else {  // (the coefficients are powers of two)
        float h = 0.f, m = 0.f, l = 0.f;
        each_ordering([&](int c, int i0, int i1, int i2, int i3) {
          l += two_sum(m, two_sum(h, (float)c * at(i0, i1, i2, i3)));
        });
        part += widen(z) * (widen(h) + (widen(m) + widen(l))) / (seps[el] - ev);
      }
    }
    total += (double)fac * part;
  }
#pragma unroll
  for (int x = 16; x > 0; x >>= 1) total += __shfl_xor_sync(0xffffffffu, total, x);
  __syncthreads();
  if ((tid & 31) == 0) red[tid >> 5] = total;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < TH / 32; ++w) t += red[w];
    a.partial[blockIdx.x] = t;
  }
}

// sum of the CTA partials (a fixed tree) / 24
__global__ void __launch_bounds__(256) k_qt_reduce(const double* __restrict__ partial, int n, double* __restrict__ out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += partial[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int x = 128; x > 0; x >>= 1) {
    if (threadIdx.x < x) red[threadIdx.x] += red[threadIdx.x + x];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0] / 24.0;
}

unsigned grid_of(i64 tot) { return (unsigned)std::max<i64>(1, std::min<i64>((tot + 255) / 256, 152 * 32)); }

template <typename T, int O>
int launch_main(QtArgs<T> a, int nsm, int smem_max, int* grid, cudaStream_t s) {
  // FP32: all rounds ahead while two CTAs fit an SM (FP64 waits for its pipe anyway)
  a.nx = sizeof(T) == 4 && QtCfg<T, O>::smem(a.v, 3) <= (size_t)smem_max / (qt_min_ctas<T>(O) > 1 ? 2 : 1) ? 3 : 1;
  const size_t smem = QtCfg<T, O>::smem(a.v, a.nx);
  if (smem + 2048 > (size_t)smem_max) return 1;
  int per_sm = 0;
  // (always: the static tables count against the 48 KB that need no opt-in)
  if (cudaFuncSetAttribute(k_qt_main<T, O>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_qt_main<T, O>, qt_threads(O), smem) != cudaSuccess ||
      per_sm < 1)
    return 1;
  *grid = (int)std::max<i64>(1, std::min<i64>(a.ntuple, std::min<i64>(*grid, (i64)nsm * per_sm)));
  ++g_launch_count;
  k_qt_main<T, O><<<*grid, qt_threads(O), smem, s>>>(a);
  return 0;
}

template <typename T>
size_t smem_of(int o, int v) {
  switch (o) {
    case 2: return QtCfg<T, 2>::smem(v, 1);
    case 3: return QtCfg<T, 3>::smem(v, 1);
    case 4: return QtCfg<T, 4>::smem(v, 1);
    case 5: return QtCfg<T, 5>::smem(v, 1);
    case 6: return QtCfg<T, 6>::smem(v, 1);
    case 7: return QtCfg<T, 7>::smem(v, 1);
    case 8:
      if constexpr (sizeof(T) == 4) return QtCfg<T, 8>::smem(v, 1);  // (FP64: 320 KB)
  }
  return (size_t)1 << 40;  // does not fit
}

}  // namespace

template <typename T>
bool qt_supported(int o, int v, int smem_max) {
  const i64 nv3 = tri3q(0, 0, v);
  return o >= 2 && o <= 8 && v <= 256 && nv3 * o * o * o < (1ll << 31) &&
         smem_of<T>(o, v) + 2048 <= (size_t)smem_max;
}
template bool qt_supported<float>(int, int, int);
template bool qt_supported<double>(int, int, int);

template <typename T>
QtSizes qt_sizes(int o, int v) {
  QtSizes z;
  const i64 o2 = (i64)o * o, V2 = (i64)v * v, n = o + v, op = (o + 1) / 2 * 2;
  const i64 el[9] = {tri3q(0, 0, v) * o2 * o, V2 * v * o, v * o2 * o, V2 * o2, (i64)v * tri2(0, v) * v * o * op,
                     tri2(0, v) * o2 * o2, V2 * ((o2 + 1) / 2 * 2), V2 * o2, sizeof(T) == 4 ? n * n * n * n + o2 * V2 : 0};
  size_t off = 0;
  for (int q = 0; q < 9; ++q) {
    z.off[q] = off;
    z.count[q] = el[q];
    off += (el[q] * sizeof(T) + 255) / 256 * 256;
  }
  z.eri = off;
  off += (size_t)(n * n * n * n * 8 + 255) / 256 * 256;
  z.partial = off;
  off += (size_t)kQtMaxGrid * 8;
  z.result = off;
  z.bytes = off + 256;
  return z;
}

template <typename T>
int qt_transpose(const QtInputs& in, T* out, cudaStream_t s) {
  const i64 nv3 = tri3q(0, 0, in.v);
  const unsigned g = (unsigned)std::min<i64>((nv3 + 7) / 8, 152 * 64);
  ++g_launch_count;
  if (in.t3_f32) k_qt_t3v<float, T><<<g, 256, 0, s>>>((const float*)in.t3, in.o, in.v, nv3, out);
  else k_qt_t3v<double, T><<<g, 256, 0, s>>>((const double*)in.t3, in.o, in.v, nv3, out);
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

template <typename T>
int qt_intermediates(const QtInputs& in, char* ws, const QtSizes& z, cudaStream_t s) {
  const int o = in.o, v = in.v, n = o + v;
  const i64 np = tri2(0, n), n4 = (i64)n * n * n * n;
  double* G = (double*)(ws + z.eri);
  auto P = [&](int q) { return (T*)(ws + z.off[q]); };
  g_launch_count += 8;
  k_qt_eri<<<dim3((unsigned)std::min<i64>((np + 255) / 256, 64), (unsigned)std::min<i64>(np, 65535)), 256, 0, s>>>(
      in.L, in.naux, n, G);
  const int kind_of[5] = {1, 2, 3, 6, 7};
  for (int k = 0; k < 5; ++k)
    k_qt_layout<T><<<grid_of(z.count[kind_of[k]]), 256, 0, s>>>(k, G, in.t2, o, v, P(kind_of[k]), z.count[kind_of[k]]);
  const T *g, *t2;
  if constexpr (sizeof(T) == 4) {
    float* gf = P(8);
    launch_convert<float, double>(gf, G, n4, s);
    launch_convert<float, double>(gf + n4, in.t2, (i64)o * o * v * v, s);
    g = gf;
    t2 = gf + n4;
  } else {
    g = G;
    t2 = in.t2;
  }
  const size_t sm = sizeof(T) * kW1FC * (size_t)(((v + 3) & ~3) + ((o * o + 3) & ~3));
  k_qt_wbar1<T><<<dim3((unsigned)tri2(0, v), v), 128, sm, s>>>(g, t2, o, v, P(4));
  k_qt_wbar2<T><<<grid_of(z.count[5]), 256, 0, s>>>(g, t2, o, v, P(5));
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

template <typename T>
int qt_main(const QtInputs& in, char* ws, const QtSizes& z, int nsm, int smem_max, int* grid, cudaStream_t s) {
  auto P = [&](int q) { return (const T*)(ws + z.off[q]); };
  QtArgs<T> a;
  a.ntuple = tet4(in.v);
  a.v = in.v;
  a.eps = in.e;
  a.t3v = P(0);
  a.A1 = P(1);
  a.A2 = P(2);
  a.Vv = P(3);
  a.W1 = P(4);
  a.W2 = P(5);
  a.T2e = P(6);
  a.T2m = P(7);
  a.partial = (double*)(ws + z.partial);
  *grid = kQtMaxGrid;
  int st = 1;
  switch (in.o) {
    case 2: st = launch_main<T, 2>(a, nsm, smem_max, grid, s); break;
    case 3: st = launch_main<T, 3>(a, nsm, smem_max, grid, s); break;
    case 4: st = launch_main<T, 4>(a, nsm, smem_max, grid, s); break;
    case 5: st = launch_main<T, 5>(a, nsm, smem_max, grid, s); break;
    case 6: st = launch_main<T, 6>(a, nsm, smem_max, grid, s); break;
    case 7: st = launch_main<T, 7>(a, nsm, smem_max, grid, s); break;
    case 8:
      if constexpr (sizeof(T) == 4) st = launch_main<T, 8>(a, nsm, smem_max, grid, s);
      break;
  }
  if (st) return 1;
  ++g_launch_count;
  k_qt_reduce<<<1, 256, 0, s>>>((const double*)(ws + z.partial), *grid, (double*)(ws + z.result));
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

template QtSizes qt_sizes<float>(int, int);
template QtSizes qt_sizes<double>(int, int);
template int qt_transpose<float>(const QtInputs&, float*, cudaStream_t);
template int qt_transpose<double>(const QtInputs&, double*, cudaStream_t);
template int qt_intermediates<float>(const QtInputs&, char*, const QtSizes&, cudaStream_t);
template int qt_intermediates<double>(const QtInputs&, char*, const QtSizes&, cudaStream_t);
template int qt_main<float>(const QtInputs&, char*, const QtSizes&, int, int, int*, cudaStream_t);
template int qt_main<double>(const QtInputs&, char*, const QtSizes&, int, int, int*, cudaStream_t);

}  // namespace rcc
