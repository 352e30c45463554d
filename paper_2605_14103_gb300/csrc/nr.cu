// Batched Newton-Raphson power flow for transmission grids (Sec. II-A).
//
// State x_b = [theta_Theta; |V|_Q] (angles of the PV and PQ buses, magnitudes
// of the PQ buses), mismatch F_b = [P_calc - P on Theta; Q_calc - Q on Q]
// with S_calc = V o conj(Y V) (eqs. 1-2), Newton step J dx = -F (eq. 3)
// solved by restarted GMRES on the left-preconditioned system
// M^-1 J dx = -M^-1 F.  J is never formed: GMRES uses the Jacobian-vector
// product dS = dV o conj(Y V) + V o conj(Y dV), dV = V o (j dtheta + d|V| / |V|).
// The preconditioner is the paper's block lower-triangular surrogate
// (eqs. 7-9):
//     z_Theta = (B' + eps I)^-1 diag(|V|_Theta)^-1 r_Theta
//     z_Q     = (B'' + eps I)^-1 diag(|V|_Q)^-1 (r_Q - G_Q,Theta z_Theta)
// with B' = -Im(Y)[Theta, Theta], B'' = -Im(Y)[Q, Q], G_Q,Theta = -Re(Y)[Q, Theta].
// The paper stores dense inverses of B' + eps I and B'' + eps I (its JAX
// stack lacks batched sparse direct solvers); here each is applied through
// its sparse LU factors (minimum-degree order, no pivoting: both matrices are
// diagonally dominant), whose triangular solves run level by level.  The
// operator is the same; a 2224-bus grid needs ~15 k factor entries and 35
// levels instead of a 40 MB dense inverse.
//
// GPU layout: one CTA solves one scenario at a time, from the flat start to
// the stop test, with every Newton and GMRES step inside the CTA (block-wide
// barriers only, no grid synchronisation, no host round trip); CTAs stride
// over the scenarios.  Per-CTA vectors and the Krylov basis live in a global
// scratch slice of the CTA (L1/L2 resident); the network (Y, G and the
// factors as tiles of rows, their levels) is shared read-only by all CTAs.
// Arnoldi uses classical Gram-Schmidt applied twice (the dot products of up
// to eight vectors in one block reduction), the Hessenberg matrix is reduced
// by Givens rotations as it grows and kept as its triangle.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <set>
#include <type_traits>
#include <vector>

#include "zbus_internal.cuh"

namespace zbus {
namespace nr {

constexpr int NR_THREADS = 128;
// CTAs per SM the register budget is sized for: 72 registers, so that the
// loads of a row and of several basis elements stay in flight (5 % over
// eight CTAs of 64).
constexpr int NR_MIN_CTAS = 7;
constexpr int NR_CHUNK = 8;       // dot products of one block reduction
constexpr int NR_MAX_RESTART_LEN = 60;
// Widest level left to one warp: a level of its own costs the CTA two barriers
// and its loads' latency (1500 cycles or so each way), one more in the warp's
// steps some 300 (2224 buses x 1000, FP64: 15.65 ms at 32, 15.25 at 128).
constexpr int NR_TAIL_ROWS = 128;
constexpr size_t NR_SMEM_MAX = 227 * 1024;
constexpr size_t NR_SMEM_DYN = NR_SMEM_MAX - 64;   // without the static words

// Sparse rows in tiles of 32, entry q of a tile's row i at 32 q + i behind the
// tile's first: a row's entries are found from its number alone (one load
// where row pointers need two in turn) and neighbouring rows load
// neighbouring words.  Shorter rows of a tile end in columns of -1.
struct Tiles {
  int ptr = 0;                // tab[ptr + t]: first entry of tile t, and one past the last
  int32_t* col = nullptr;
  double* val = nullptr;      // double2 for Y
  float* val_f = nullptr;     // FP32 copies (mixed form)
};

// The narrow end of a triangle as steps of one warp: in a step each of w <= 32
// rows takes up to four of its next entries, whatever its level, as long as
// their columns were finished before the step.  A row's entries are taken in
// their order, but it does not wait for all of them to start.  A step is two
// words of the index table, its first record and w - 1 | c << 8 with c the
// most entries a row of it takes; STEP_AHEAD + 1 copies of the last one follow.
// Missing entries of a record are zeros that meet the zero in y[N - 1].
struct Steps {
  int at = 0, n = 0;          // tab[at + 2 s], steps
  int2* row = nullptr;        // row | STEP_LAST (of its entries), perm
  int4* col = nullptr;
  double* val = nullptr;      // [records][4]
  double* dinv = nullptr;     // 1 / U_kk (U)
  float* val_f = nullptr;
  float* dinv_f = nullptr;
};
constexpr int STEP_LAST = 1 << 30;
constexpr int STEP_AHEAD = 3;    // one: 0.80 ms for 118 buses x 1000 mixed, two 0.77, three 0.73

// One factor P A P^T = L U of the preconditioner on the device.  Rows are
// stored level by level (a row's level is above that of every row its L or
// U entries couple it to), so the same contiguous ranges serve the forward
// solve upwards and the backward solve downwards.
struct Factor {
  int n = 0;
  // The levels from t_lev on, most with one or two rows, are one warp's
  // (narrow_walk), L's steps, then U's.
  int t_lev = 0, n_lev = 0;
  Steps TL, TU;
  int32_t* perm = nullptr;    // [n] row -> position in the block
  int lev_ptr = 0;            // tab[lev_ptr + l]: rows of level l, to the next level's
  int lev_tile = 0;           // tab[lev_tile + l]: a level's first tile
  Tiles L;                    // strictly lower entries, in elimination order
  Tiles U;                    // strictly upper entries
  double* dinv = nullptr;     // 1 / U_kk
  float* dinv_f = nullptr;
  int levels = 0;             // of both solves, each counted by itself
  int64_t nnz = 0;
};

// Everything the solve kernel reads, by value.
struct NrDev {
  int N, nt, nq, dim, m;
  const int32_t* tab;     // every lev_ptr, lev_tile and Tiles::ptr, one behind the other
  int tab_n;
  int tab_shared;         // the CTA keeps a copy of tab
  const int4* y_row;      // [N] k-th row of Y, longest first: bus, its rows of the factors
  Tiles Y;
  const int32_t* bus_type;
  const double* v_set;
  const int32_t* pos_t;   // [N] position in the angle block, -1 at the slack
  const int32_t* pos_q;   // [N] position in the magnitude block, -1 unless PQ
  const int32_t* row_t;   // [N] the bus's row of the factor of B', -1 at the slack
  const int32_t* row_q;   // [N] of the factor of B'', -1 unless PQ
  const int2* g_row;      // [nq] k-th row of G_Q,Theta, longest first: row of B''s factor, bus
  Tiles G;                // cols = Theta positions
  Factor Bp, Bpp;
  int tab_at;             // doubles of shared memory before the copy of tab
  double* scratch;
  int64_t stride;         // doubles of scratch per CTA
};

}  // namespace nr
}  // namespace zbus

struct zbus_nr_network_s {
  int device = 0;
  int N = 0, nt = 0, nq = 0;
  int slack = 0;
  zbus::nr::NrDev dev{};
  std::vector<void*> allocs;      // every device buffer of the network
  double* scratch = nullptr;
  int64_t scratch_size = 0;       // doubles
  bool smem_set[2] = {false, false};
  int sms = 1;
};

namespace zbus {
namespace nr {
namespace {

// ---------------------------------------------------------------------------
// Device helpers (block-wide; every thread of the CTA calls them).
// ---------------------------------------------------------------------------

struct SumOp {
  static __device__ __forceinline__ double f(double a, double b) { return a + b; }
};
struct MaxOp {   // NaN wins
  static __device__ __forceinline__ double f(double a, double b) {
    return (b > a || b != b) ? b : a;
  }
};

// The 128 partials p[] of one value: butterflies over 32 lanes (16, 8, 4, 2,
// 1), then the four results in order.  The four butterflies share their
// steps: after the first a lane holds two of them, after the second one.
template <class Op>
__device__ __forceinline__ double reduce_128(const double* p) {
  const int l = threadIdx.x & 31;
  const double a0 = p[l], a1 = p[l + 32], a2 = p[l + 64], a3 = p[l + 96];
  const bool b = l & 16, c = l & 8;
  const double x0 = Op::f(b ? a2 : a0, __shfl_xor_sync(0xffffffffu, b ? a0 : a2, 16));
  const double x1 = Op::f(b ? a3 : a1, __shfl_xor_sync(0xffffffffu, b ? a1 : a3, 16));
  double z = Op::f(c ? x1 : x0, __shfl_xor_sync(0xffffffffu, c ? x0 : x1, 8));
  for (int o = 4; o > 0; o >>= 1) z = Op::f(z, __shfl_xor_sync(0xffffffffu, z, o));
  const double q0 = __shfl_sync(0xffffffffu, z, 0), q1 = __shfl_sync(0xffffffffu, z, 8);
  const double q2 = __shfl_sync(0xffffffffu, z, 16), q3 = __shfl_sync(0xffffffffu, z, 24);
  return Op::f(Op::f(Op::f(q0, q1), q2), q3);
}

// Sum (or max) over the CTA of one value per thread; every thread gets it.
template <class Op>
__device__ double block_reduce(double v, double* red) {
  __syncthreads();
  red[threadIdx.x] = v;
  __syncthreads();
  return reduce_128<Op>(red);
}

// Values in the Krylov precision T: FP64 (the paper's solver) or FP32 (the
// mixed form, whose Newton direction is found in FP32 while the mismatch,
// the state and the stop test stay FP64).
template <class T> struct Cx;
template <> struct Cx<double> { using type = double2; };
template <> struct Cx<float> { using type = float2; };

__device__ __forceinline__ const double* vals(const Tiles& t, double) { return t.val; }
__device__ __forceinline__ const float* vals(const Tiles& t, float) { return t.val_f; }
__device__ __forceinline__ const double2* vals(const Tiles& t, double2) {
  return reinterpret_cast<const double2*>(t.val);
}
__device__ __forceinline__ const float2* vals(const Tiles& t, float2) {
  return reinterpret_cast<const float2*>(t.val_f);
}
__device__ __forceinline__ const double* dval(const Factor& f, double) { return f.dinv; }
__device__ __forceinline__ const float* dval(const Factor& f, float) { return f.dinv_f; }
__device__ __forceinline__ const double* vals(const Steps& t, double) { return t.val; }
__device__ __forceinline__ const float* vals(const Steps& t, float) { return t.val_f; }
__device__ __forceinline__ const double* dval(const Steps& t, double) { return t.dinv; }
__device__ __forceinline__ const float* dval(const Steps& t, float) { return t.dinv_f; }

// a b + c d, the first product unrounded.  Spelled out wherever the sum of
// two products occurs: the counts of Newton and Krylov steps amplify the last
// bit, so a compiler's choice of the product to round would show in them.
__device__ __forceinline__ double mul_add(double a, double b, double c, double d) {
  return fma(a, b, c * d);
}
__device__ __forceinline__ float mul_add(float a, float b, float c, float d) {
  return fmaf(a, b, c * d);
}

// A sparse row's entries 0 .. cnt, in order, U at a time: the loads of a batch
// (a column and its value, then what the column points at) are issued
// together, past the end at the last entry, so a short row waits for two
// loads and not for two per entry.  load(q) gives (column, value), at(column)
// the operand, mac(value, operand) takes it into the sum.
template <int U, class Load, class At, class Mac>
__device__ __forceinline__ void row_walk(int cnt, int n, uint32_t code, Load load, At at,
                                         Mac mac) {
  for (int e = 0; e < cnt; e += U) {
    decltype(load(0)) x[U];
#pragma unroll
    for (int q = 0; q < U; ++q) x[q] = load(min(e + q, cnt - 1));
    decltype(at(0)) v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) v[q] = at(x[q].col >= 0 && ZB_IN(x[q].col, n, code) ? x[q].col : 0);
#pragma unroll
    for (int q = 0; q < U; ++q)
      if (e + q < cnt && x[q].col >= 0 && ZB_IN(x[q].col, n, code)) mac(x[q].val, v[q]);
  }
}
template <class V> struct Entry {
  int col;
  V val;
};
// Row i of the tiles from tile t0 on.
template <class V, class At, class Mac>
__device__ __forceinline__ void tile_walk(const Tiles& m, const int32_t* tab, int t0, int i, int n,
                                          uint32_t code, At at, Mac mac) {
  const int t = m.ptr + t0 + (i >> 5);
  const int b = tab[t], cnt = (tab[t + 1] - b) >> 5;
  const int32_t* col = m.col + b + (i & 31);
  const V* val = vals(m, V()) + b + (i & 31);
  row_walk<4>(cnt, n, code,
              [&](int q) { return Entry<V>{__ldg(col + 32 * q), __ldg(val + 32 * q)}; }, at, mac);
}

__device__ __forceinline__ void load4(double* v, const double* p) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p));
  const double2 b = __ldg(reinterpret_cast<const double2*>(p) + 1);
  v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ void load4(float* v, const float* p) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}

// The narrow end of one triangle by one warp, a lane a record.  What it costs
// is a lone warp's dependent multiply-adds (64 cycles each in FP64) and its
// instructions, a few cycles each: so there are few steps (Steps), a step is
// some forty instructions, and its records come in vectors and are loaded
// STEP_AHEAD steps before their use (each buffer again right after it: a copy
// between buffers would wait for the load).  L, or UPPER: U, rows times
// 1 / U_kk and into out.
template <bool UPPER, class T>
__device__ __forceinline__ void narrow_walk(const Steps& st, const int32_t* tab, int n, int N,
                                            T* y, T* out) {
  [[maybe_unused]] constexpr uint32_t code = UPPER ? 0x405u : 0x403u;
  const int lane = threadIdx.x & 31;
  const T* val = vals(st, T());
  const T* dv = dval(st, T());
  const int2* step = reinterpret_cast<const int2*>(tab + st.at);
  struct Buffer {
    int w;
    int2 row;
    int4 col;
    T val[4], di;
  } x[STEP_AHEAD];
  int2 d = step[0];   // of the next step to load
  auto load = [&](Buffer& b, int s) {
    b.w = d.y;
    const int i = d.x + min(lane, d.y & 31);
    b.row = __ldg(st.row + i);
    b.col = __ldg(st.col + i);
    load4(b.val, val + 4 * i);
    if (UPPER) b.di = __ldg(dv + i);
    d = step[s + 1];
  };
  auto at = [&](int j) { return y[ZB_IN(j, N, code) ? j : 0]; };
#pragma unroll
  for (int i = 0; i < STEP_AHEAD; ++i) load(x[i], i);
  for (int s = 0; s < st.n; s += STEP_AHEAD) {
#pragma unroll
    for (int i = 0; i < STEP_AHEAD; ++i) {
      if (s + i >= st.n) break;
      Buffer& b = x[i];
      const int k = b.row.x & (STEP_LAST - 1), cnt = b.w >> 8;
      const T v0 = at(b.col.x), v1 = at(b.col.y), v2 = at(b.col.z), v3 = at(b.col.w);
      T a = at(k);
      if (sizeof(T) == 4 || cnt > 0) a -= b.val[0] * v0;   // in FP32 a branch costs more
      if (sizeof(T) == 4 || cnt > 1) a -= b.val[1] * v1;
      if (sizeof(T) == 4 || cnt > 2) a -= b.val[2] * v2;
      if (sizeof(T) == 4 || cnt > 3) a -= b.val[3] * v3;
      if (lane <= (b.w & 31)) {
        if (UPPER && (b.row.x & STEP_LAST)) {
          a *= b.di;
          if (ZB_IN(b.row.y, n, 0x406u)) out[b.row.y] = a;
        }
        if (ZB_IN(k, n, code)) y[k] = a;
      }
      __syncwarp();
      load(b, s + i + STEP_AHEAD);
    }
  }
}

// Solve (P A P^T) with its LU factors: out[perm[k]] = (U^-1 L^-1 y)_k.  y
// (shared, by factor row; y[N - 1] is 0) is overwritten; out is by block
// position.  Wide levels take the whole CTA and a barrier each; what the
// narrow ones at the end of the elimination hold is left to one warp, which
// only waits for itself.
template <class T>
__device__ void factor_solve(const Factor& f, const int32_t* tab, int N, T* y, T* out) {
  const int t = threadIdx.x;
  const T* dv = dval(f, T());
  for (int l = 1; l < f.t_lev; ++l) {   // level 0 has no lower entries
    const int k0 = tab[f.lev_ptr + l], k1 = tab[f.lev_ptr + l + 1];
    const int t0 = tab[f.lev_tile + l];
    for (int k = k0 + t; k < k1; k += NR_THREADS) {
      if (!ZB_IN(k, f.n, 0x402u)) continue;
      T a = y[k];
      tile_walk<T>(f.L, tab, t0, k - k0, f.n, 0x403u, [&](int j) { return y[j]; },
                   [&](T v, T x) { a -= v * x; });
      y[k] = a;
    }
    __syncthreads();
  }
  if (f.t_lev < f.n_lev) {
    if (t < 32) {
      if (f.TL.n > 0) narrow_walk<false, T>(f.TL, tab, f.n, N, y, out);
      narrow_walk<true, T>(f.TU, tab, f.n, N, y, out);
    }
    __syncthreads();
  }
  for (int l = f.t_lev - 1; l >= 0; --l) {
    const int k0 = tab[f.lev_ptr + l], k1 = tab[f.lev_ptr + l + 1];
    const int t0 = tab[f.lev_tile + l];
    for (int k = k0 + t; k < k1; k += NR_THREADS) {
      const int p = __ldg(f.perm + k);
      const T di = __ldg(dv + k);
      if (!ZB_IN(k, f.n, 0x404u) || !ZB_IN(p, f.n, 0x406u)) continue;
      T a = y[k];
      tile_walk<T>(f.U, tab, t0, k - k0, f.n, 0x405u, [&](int j) { return y[j]; },
                   [&](T v, T x) { a -= v * x; });
      a *= di;
      y[k] = a;
      out[p] = a;
    }
    __syncthreads();
  }
}

// z = M^-1 r (eqs. 8-9).  On entry, behind a barrier: y holds r_Theta / |V|
// by the rows of the factor of B', rq r_Q by those of B''.  ivm = 1 / |V|.
template <class T>
__device__ void precondition(const NrDev& d, const int32_t* tab, const T* ivm, T* y, const T* rq,
                             T* z) {
  factor_solve<T>(d.Bp, tab, d.N, y, z);
  if (d.nq > 0) {
    for (int k = threadIdx.x; k < d.nq; k += NR_THREADS) {
      const int2 row = __ldg(d.g_row + k);
      if (!ZB_IN(row.x, d.nq, 0x409u) || !ZB_IN(row.y, d.N, 0x409u)) continue;
      T a = rq[row.x];
      const T im = ivm[row.y];
      tile_walk<T>(d.G, tab, 0, k, d.nt, 0x408u, [&](int j) { return z[j]; },
                   [&](T v, T x) { a -= v * x; });
      y[row.x] = a * im;
    }
    __syncthreads();
    factor_solve<T>(d.Bpp, tab, d.N, y, z + d.nt);
  }
}

// acc += y v for one entry of Y.
template <class C> __device__ __forceinline__ void y_mac(C& acc, C y, C v) {
  acc.x += mul_add(y.x, v.x, -y.y, v.y);
  acc.y += mul_add(y.x, v.y, y.y, v.x);
}

// J u, the Jacobian of F at V (I = Y V) applied to u (dim), as the
// input of precondition: y and rq.  ivm = 1 / |V|.
template <class T>
__device__ void jvp(const NrDev& d, const int32_t* tab, const typename Cx<T>::type* V,
                    const typename Cx<T>::type* I, const T* ivm, const T* u,
                    typename Cx<T>::type* dV, T* y, T* rq) {
  using C = typename Cx<T>::type;
  const int t = threadIdx.x;
  for (int i = t; i < d.N; i += NR_THREADS) {
    const int pt = __ldg(d.pos_t + i), pq = __ldg(d.pos_q + i);
    const T dth = pt >= 0 ? u[pt] : T(0);
    const T a = pq >= 0 ? u[d.nt + pq] * ivm[i] : T(0);
    const C v = V[i];
    C x;
    x.x = mul_add(v.x, a, -v.y, dth);
    x.y = mul_add(v.y, a, v.x, dth);
    dV[i] = x;
  }
  __syncthreads();
  for (int k = t; k < d.N; k += NR_THREADS) {
    const int4 row = __ldg(d.y_row + k);
    const int i = row.x, kt = row.y, kq = row.z;
    if (!ZB_IN(i, d.N, 0x40au)) continue;
    if (kt < 0) y[d.N - 1] = T(0);   // the slack: no row, and its place the narrow walks' zero
    const C dv = dV[i], v = V[i], cur = I[i];
    const T im = ivm[i];
    C yd;
    yd.x = yd.y = T(0);
    tile_walk<C>(d.Y, tab, 0, k, d.N, 0x40au, [&](int j) { return dV[j]; },
                 [&](C y, C v) { y_mac(yd, y, v); });
    // dS = dV conj(I) + V conj(Y dV)
    const T sr = fma(v.y, yd.y, fma(v.x, yd.x, mul_add(dv.x, cur.x, dv.y, cur.y)));
    const T si = fma(-v.x, yd.y, fma(v.y, yd.x, mul_add(dv.y, cur.x, -dv.x, cur.y)));
    if (kt >= 0 && ZB_IN(kt, d.nt, 0x407u)) y[kt] = sr * im;
    if (kq >= 0 && ZB_IN(kq, d.nq, 0x407u)) rq[kq] = si;
  }
  __syncthreads();
}

// Gram-Schmidt over n basis vectors (compile-time, so that the loads of
// several elements are in flight: eight or so a thread).
template <class F>
__device__ __forceinline__ void for_count(int n, F f) {
  switch (n) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    default: f(std::integral_constant<int, 8>()); break;
  }
}
static_assert(NR_CHUNK == 8, "for_count covers a chunk");

// A thread's partial sums of v_q . w into red.
template <int NV, class T>
__device__ __forceinline__ void gs_dots(int dim, const T* Vk, const T* wv,
                                        double* red) {
  constexpr int U = NV <= 2 ? 4 : NV <= 4 ? 2 : 1;
  T acc[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = 0;
#pragma unroll U
  for (int e = threadIdx.x; e < dim; e += NR_THREADS) {
    const T we = wv[e];
#pragma unroll
    for (int q = 0; q < NV; ++q) acc[q] += Vk[q * dim + e] * we;
  }
#pragma unroll
  for (int q = 0; q < NV; ++q) red[q * NR_THREADS + threadIdx.x] = (double)acc[q];
}

// w -= sum of h_q v_q; then, FIRST, the partial sums of v_q . w into red,
// else w's own square into nw.
template <int NV, bool FIRST, class T>
__device__ __forceinline__ void gs_update(int dim, const T* __restrict__ Vk,
                                          T* __restrict__ wv, const T* hT, double* red, T& nw) {
  constexpr int U = NV <= 2 ? 4 : NV <= 4 ? 2 : 1;
  T acc[NV], h[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = 0, h[q] = hT[q];
#pragma unroll U
  for (int e = threadIdx.x; e < dim; e += NR_THREADS) {
    T we = wv[e], v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = Vk[q * dim + e];
#pragma unroll
    for (int q = 0; q < NV; ++q) we -= h[q] * v[q];
    wv[e] = we;
    if constexpr (FIRST) {
#pragma unroll
      for (int q = 0; q < NV; ++q) acc[q] += v[q] * we;
    } else {
      nw += we * we;
    }
  }
  if constexpr (FIRST) {
#pragma unroll
    for (int q = 0; q < NV; ++q) red[q * NR_THREADS + threadIdx.x] = (double)acc[q];
  }
}

// x += sum of h_q v_q.
template <int NV, class T>
__device__ __forceinline__ void gs_axpy(int dim, const T* __restrict__ Vk, T* __restrict__ x,
                                        const T* hT) {
  constexpr int U = NV <= 2 ? 4 : NV <= 4 ? 2 : 1;
  T h[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) h[q] = hT[q];
#pragma unroll U
  for (int e = threadIdx.x; e < dim; e += NR_THREADS) {
    T v = x[e];
#pragma unroll
    for (int q = 0; q < NV; ++q) v += h[q] * Vk[q * dim + e];
    x[e] = v;
  }
}

// ---------------------------------------------------------------------------
// The solve: one CTA per scenario at a time.
// ---------------------------------------------------------------------------
struct SolveArgs {
  int B;
  const double* P;        // [B][N]
  const double* Q;        // [B][N]
  double tol;
  int max_iter;
  double eta;             // GMRES relative tolerance on the preconditioned residual
  int max_restart;
  double2* V;             // [B][N]
  int32_t* iters;
  uint8_t* conv;
  int32_t* gmres;
};

// Scratch of one scenario: the FP64 state (V, I, F, |V|, angle, 1 / |V|),
// then the Krylov-precision arrays (FP32 copies of V, I, 1 / |V| for the
// mixed form; dV; right-hand side, solution, work vectors; the basis).
__host__ __device__ constexpr int64_t state_doubles(int64_t N) { return 9 * N; }
template <class T>
__host__ __device__ constexpr int64_t krylov_values(int64_t N, int64_t dim, int m) {
  return (sizeof(T) == 4 ? 5 * N : 0) + 1 + 2 * N + 4 * dim + (int64_t)(m + 1) * dim;
}
// Doubles of shared memory beside y: the triangle R of the Hessenberg matrix,
// the rotations, the right-hand side, a step's coefficients (new, in T,
// summed over the passes).
__host__ __device__ constexpr int shared_doubles(int m) {
  return m * (m + 1) / 2 + 2 * m + 4 * (m + 1);
}

// What bounds it: at a full batch the FP64 pipe (2 multiply-adds a clock and
// SM, 64 cycles for one that waits for the last; a warp instruction costs the
// same for one lane as for 32), for a few scenarios the chain of a scenario's
// loads, barriers and dependent multiply-adds.  Against both: rows of one
// length share a warp and are found without row pointers (Tiles), a row's
// loads are issued together, the index tables sit in shared memory, the
// narrow end of the factors is one warp's (narrow_walk), and Gram-Schmidt
// keeps several elements in flight and reads the basis once for the first
// pass's update and the second pass's products.  Every sum keeps its order.
// 1000 scenarios: 2224 buses FP64 22.4 -> 15.3 ms, mixed 11.3 -> 6.6 ms; 118
// buses mixed 1.14 -> 0.73 ms; one scenario of 2224 buses, FP64, 12.3 -> 6.3.
// Larger grids, to which NR_TAIL_ROWS and NR_MIN_CTAS were not fitted, 1 and 500
// scenarios of 5000 buses: FP64 33.2 -> 17.6 and 49.2 -> 33.6 ms, mixed 22.6 ->
// 10.3 and 31.9 -> 16.2; 1 and 200 of 13659 (20 steps, 1500 products): FP64 3.64
// -> 2.47 and 11.1 -> 7.86 s, mixed 2.34 -> 1.47 and 4.28 -> 3.19.
template <class T>
__global__ void __launch_bounds__(NR_THREADS, NR_MIN_CTAS) k_nr_solve(NrDev d, SolveArgs a) {
  constexpr bool MIXED = sizeof(T) == 4;
  using C = typename Cx<T>::type;
  extern __shared__ double sm[];
  const int m = d.m, N = d.N, nt = d.nt, dim = d.dim, t = threadIdx.x;
  double* R = sm;                            // column j at j (j + 1) / 2
  double* cs = R + m * (m + 1) / 2;          // [m]
  double* sn = cs + m;                       // [m]
  double* gv = sn + m;                       // [m + 1]
  double* hh = gv + m + 1;                   // [m + 1] this pass's Gram-Schmidt coefficients
  double* hc = hh + m + 1;                   // [m + 1] this step's column of the Hessenberg
  T* hT = reinterpret_cast<T*>(hc + m + 1);  // [m + 1] hh in T, converted once
  double* red = hc + 2 * (m + 1);            // partial sums, [NR_CHUNK][NR_THREADS] ...
  T* y = reinterpret_cast<T*>(red);          // ... or the factor work space, [N]
  int32_t* tab_s = reinterpret_cast<int32_t*>(sm + d.tab_at);
  if (d.tab_shared)
    for (int q = t; q < d.tab_n; q += NR_THREADS) tab_s[q] = __ldg(d.tab + q);
  const int32_t* tab = d.tab_shared ? tab_s : d.tab;
  __shared__ int s_flag, s_jd;

  double2* V = reinterpret_cast<double2*>(d.scratch + (int64_t)blockIdx.x * d.stride);
  double2* I = V + N;
  double2* F = I + N;                        // (P, Q) mismatch per bus
  double* vm = reinterpret_cast<double*>(F + N);
  double* va = vm + N;
  double* ivm = va + N;                      // 1 / |V| of the current iterate
  C *VT, *IT;                                // the state in the Krylov precision
  T *ivmT, *kb;
  if constexpr (MIXED) {
    VT = reinterpret_cast<C*>(ivm + N);
    IT = VT + N;
    ivmT = reinterpret_cast<T*>(IT + N);
    kb = ivmT + N;
  } else {
    VT = V, IT = I, ivmT = ivm;
    kb = ivm + N;
  }
  kb += N & 1;                               // dV is aligned to a C
  C* dV = reinterpret_cast<C*>(kb);
  T* bv = reinterpret_cast<T*>(dV + N);
  T* x = bv + dim;
  T* wv = x + dim;
  T* rq = wv + dim;                          // [nq]
  T* Vk = rq + dim;                          // basis, [m + 1][dim]

  // hh = (dot products of w with cnt basis vectors from i0), their partials
  // in red; hc accumulates them
  auto finish_dots = [&](int i0, int cnt) {
    __syncthreads();
    for (int p = t >> 5; p < cnt; p += NR_THREADS / 32) {
      const double v = reduce_128<SumOp>(red + p * NR_THREADS);
      if ((t & 31) == 0) {
        hh[i0 + p] = v;
        hT[i0 + p] = (T)v;
        hc[i0 + p] += v;
      }
    }
    __syncthreads();
  };

  for (int b = blockIdx.x; b < a.B; b += gridDim.x) {
    const double* P = a.P + (int64_t)b * N;
    const double* Q = a.Q + (int64_t)b * N;
    for (int i = t; i < N; i += NR_THREADS) {
      vm[i] = d.bus_type[i] == 0 ? 1.0 : d.v_set[i];
      va[i] = 0.0;
    }
    int gm_total = 0, it = 0, ok = 0;
    for (int k = 0;; ++k) {
      // V, I = Y V, mismatch F and its max (FP64)
      for (int i = t; i < N; i += NR_THREADS) {
        double si = 0.0, co = 1.0;
        if (k > 0) sincos(va[i], &si, &co);
        const double mag = vm[i];
        const double2 v = make_double2(mag * co, mag * si);
        const double im = 1.0 / mag;
        V[i] = v;
        ivm[i] = im;
        if constexpr (MIXED) {
          VT[i] = make_float2((float)v.x, (float)v.y);
          ivmT[i] = (T)im;
        }
      }
      __syncthreads();
      double fmax = 0.0;
      for (int q = t; q < N; q += NR_THREADS) {
        const int4 row = __ldg(d.y_row + q);
        const int i = row.x;
        if (!ZB_IN(i, N, 0x40bu)) continue;
        const double2 v = V[i];
        const double p_set = row.y >= 0 ? P[i] : 0.0, q_set = row.z >= 0 ? Q[i] : 0.0;
        double2 cur = make_double2(0.0, 0.0);
        tile_walk<double2>(d.Y, tab, 0, q, N, 0x40bu, [&](int j) { return V[j]; },
                           [&](double2 y, double2 v) { y_mac(cur, y, v); });
        const double ir = cur.x, ii = cur.y;
        I[i] = make_double2(ir, ii);
        if constexpr (MIXED) IT[i] = make_float2((float)ir, (float)ii);
        const double sr = mul_add(v.x, ir, v.y, ii);   // V conj(I)
        const double si = mul_add(v.y, ir, -v.x, ii);
        double2 f = make_double2(0.0, 0.0);
        if (row.y >= 0) {
          f.x = sr - p_set;
          fmax = MaxOp::f(fmax, fabs(f.x));
        }
        if (row.z >= 0) {
          f.y = si - q_set;
          fmax = MaxOp::f(fmax, fabs(f.y));
        }
        F[i] = f;
      }
      fmax = block_reduce<MaxOp>(fmax, red);
      it = k;
      if (!(fmax <= a.tol)) {
        if (fmax != fmax || isinf(fmax) || k == a.max_iter) break;
      } else {
        ok = 1;
        break;
      }
      // GMRES on M^-1 J dx = M^-1 (-F), x0 = 0
      __syncthreads();                       // red is y
      for (int e = t; e < dim; e += NR_THREADS) x[e] = T(0);
      for (int i = t; i < N; i += NR_THREADS) {
        const int kt = __ldg(d.row_t + i), kq = __ldg(d.row_q + i);
        const double2 f = F[i];
        if (kt >= 0 && ZB_IN(kt, nt, 0x407u)) y[kt] = (T)(-f.x) * ivmT[i];
        if (kt < 0) y[N - 1] = T(0);
        if (kq >= 0 && ZB_IN(kq, d.nq, 0x407u)) rq[kq] = (T)(-f.y);
      }
      __syncthreads();
      precondition<T>(d, tab, ivmT, y, rq, bv);
      T nb = 0;
#pragma unroll 4
      for (int e = t; e < dim; e += NR_THREADS) nb += bv[e] * bv[e];
      const double beta0 = sqrt(block_reduce<SumOp>((double)nb, red));
      bool done = !(beta0 > 0.0);
      for (int rs = 0; rs < a.max_restart && !done; ++rs) {
        // r = b - A x (x = 0 on the first pass)
        if (rs > 0) {
          jvp<T>(d, tab, VT, IT, ivmT, x, dV, y, rq);
          precondition<T>(d, tab, ivmT, y, rq, wv);
          for (int e = t; e < dim; e += NR_THREADS) Vk[e] = bv[e] - wv[e];
        } else {
          for (int e = t; e < dim; e += NR_THREADS) Vk[e] = bv[e];
        }
        T nr = 0;
#pragma unroll 4
        for (int e = t; e < dim; e += NR_THREADS) nr += Vk[e] * Vk[e];
        const double beta = sqrt(block_reduce<SumOp>((double)nr, red));
        if (!(beta > a.eta * beta0)) break;
        const T ib = (T)(1.0 / beta);
        for (int e = t; e < dim; e += NR_THREADS) Vk[e] *= ib;
        if (t == 0) {
          gv[0] = beta;
          s_jd = 0;
          s_flag = 0;
        }
        __syncthreads();
        for (int j = 0; j < m; ++j) {
          const T* vj = Vk + (int64_t)j * dim;
          jvp<T>(d, tab, VT, IT, ivmT, vj, dV, y, rq);
          for (int i = t; i <= j; i += NR_THREADS) hc[i] = 0.0;
          precondition<T>(d, tab, ivmT, y, rq, wv);
          // classical Gram-Schmidt, twice; products in T, sums across the
          // threads in FP64.  Up to NR_CHUNK vectors the first pass's
          // update and the second pass's products read the basis once.
          T nw = 0;
          const int nv = j + 1;
          if (nv <= NR_CHUNK) {
            for_count(nv, [&](auto n) {
              gs_dots<decltype(n)::value>(dim, Vk, wv, red);
            });
            finish_dots(0, nv);
            for_count(nv, [&](auto n) {
              gs_update<decltype(n)::value, true>(dim, Vk, wv, hT, red, nw);
            });
            finish_dots(0, nv);
            for_count(nv, [&](auto n) {
              gs_update<decltype(n)::value, false>(dim, Vk, wv, hT, red, nw);
            });
          } else {
            for (int pass = 0; pass < 2; ++pass) {
              for (int i0 = 0; i0 < nv; i0 += NR_CHUNK) {
                const int cnt = min(NR_CHUNK, nv - i0);
                for_count(cnt, [&](auto n) {
                  gs_dots<decltype(n)::value>(dim, Vk + i0 * dim, wv, red);
                });
                finish_dots(i0, cnt);
              }
              for (int i0 = 0; i0 < nv; i0 += NR_CHUNK) {
                nw = 0;
                for_count(min(NR_CHUNK, nv - i0), [&](auto n) {
                  gs_update<decltype(n)::value, false>(dim, Vk + i0 * dim, wv, hT + i0, red, nw);
                });
              }
            }
          }
          const double hn = sqrt(block_reduce<SumOp>((double)nw, red));
          T* vn = Vk + (int64_t)(j + 1) * dim;
          const T inv = hn > 0.0 ? (T)(1.0 / hn) : T(0);
#pragma unroll 4
          for (int e = t; e < dim; e += NR_THREADS) vn[e] = wv[e] * inv;
          ++gm_total;
          if (t == 0) {
            double* col = R + j * (j + 1) / 2;
            double h = hc[0];
            for (int i = 0; i < j; ++i) {   // earlier rotations
              const double h1 = hc[i + 1];
              const double r0 = mul_add(cs[i], h, sn[i], h1);
              h = mul_add(cs[i], h1, -sn[i], h);
              col[i] = r0;
            }
            const double den = hypot(h, hn);
            const double cj = den > 0.0 ? h / den : 1.0;
            const double sj = den > 0.0 ? hn / den : 0.0;
            cs[j] = cj;
            sn[j] = sj;
            col[j] = den;
            const double g = gv[j], res = fabs(-sj * g);
            gv[j + 1] = -sj * g;
            gv[j] = cj * g;
            s_jd = j + 1;
            s_flag = (res <= a.eta * beta0 || !(hn > 0.0) || res != res) ? 1 : 0;
          }
          __syncthreads();
          if (s_flag) break;
        }
        // y = R^-1 g (upper triangular), x += V y
        const int jd = s_jd;
        if (t == 0)
          for (int i = jd - 1; i >= 0; --i) {
            double v = gv[i];
            for (int q = i + 1; q < jd; ++q) v -= R[q * (q + 1) / 2 + i] * hh[q];
            hh[i] = v / R[i * (i + 1) / 2 + i];
            hT[i] = (T)hh[i];
          }
        if (s_flag) done = true;
        __syncthreads();
        for (int i = 0; i < jd; i += NR_CHUNK)
          for_count(min(NR_CHUNK, jd - i), [&](auto n) {
            gs_axpy<decltype(n)::value>(dim, Vk + (int64_t)i * dim, x, hT + i);
          });
        __syncthreads();
      }
      // Newton update (FP64 state)
      for (int i = t; i < N; i += NR_THREADS) {
        const int pt = __ldg(d.pos_t + i), pq = __ldg(d.pos_q + i);
        if (pt >= 0 && ZB_IN(pt, nt, 0x40cu)) va[i] += (double)x[pt];
        if (pq >= 0 && ZB_IN(pq, d.nq, 0x40du)) vm[i] += (double)x[nt + pq];
      }
      __syncthreads();
    }
    double2* Vo = a.V + (int64_t)b * N;
    for (int i = t; i < N; i += NR_THREADS) Vo[i] = V[i];
    if (t == 0) {
      a.iters[b] = it;
      a.conv[b] = (uint8_t)ok;
      if (a.gmres) a.gmres[b] = gm_total;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Host side: ordering, factorisation, level lists.
// ---------------------------------------------------------------------------

// Minimum-degree order of the symmetrised pattern of A (n x n, rows of
// (col, value) pairs), eliminating one node at a time and joining its
// neighbours; ties go to the lowest index.
std::vector<int> min_degree(int n, const std::vector<std::map<int, double>>& A) {
  std::vector<std::set<int>> adj(n);
  for (int i = 0; i < n; ++i)
    for (auto& kv : A[i])
      if (kv.first != i) {
        adj[i].insert(kv.first);
        adj[kv.first].insert(i);
      }
  std::vector<char> gone(n, 0);
  std::vector<int> order;
  order.reserve(n);
  for (int step = 0; step < n; ++step) {
    int best = -1;
    size_t bd = SIZE_MAX;
    for (int i = 0; i < n; ++i)
      if (!gone[i] && adj[i].size() < bd) {
        bd = adj[i].size();
        best = i;
      }
    gone[best] = 1;
    order.push_back(best);
    std::vector<int> nb(adj[best].begin(), adj[best].end());
    for (int u : nb) adj[u].erase(best);
    for (size_t p = 0; p < nb.size(); ++p)
      for (size_t q = p + 1; q < nb.size(); ++q) {
        adj[nb[p]].insert(nb[q]);
        adj[nb[q]].insert(nb[p]);
      }
    adj[best].clear();
  }
  return order;
}

struct HostFactor {
  int n = 0;
  int levels = 0;   // of the forward and of the backward solve, each by its own triangle
  std::vector<int32_t> perm, l_ptr, l_col, u_ptr, u_col, lev_ptr;
  std::vector<double> l_val, u_val, dinv;
  int t_lev = 0;   // first of the narrow levels at the end
};

// LU of P A P^T without pivoting (right-looking, sparse rows), the level
// lists of both triangular solves.  False if a pivot is not usable.
bool factorise(int n, const std::vector<std::map<int, double>>& A, HostFactor& hf,
               std::string& why) {
  hf = HostFactor();
  hf.n = n;
  hf.perm = min_degree(n, A);
  std::vector<int> inv(n);
  for (int i = 0; i < n; ++i) inv[hf.perm[i]] = i;
  std::vector<std::map<int, double>> R(n);            // rows of P A P^T
  std::vector<std::set<int>> below(n);                // rows i > k with an entry in column k
  double amax = 0.0;
  for (int i = 0; i < n; ++i)
    for (auto& kv : A[i]) {
      const int r = inv[i], c = inv[kv.first];
      R[r][c] += kv.second;
      if (r > c) below[c].insert(r);
      amax = std::max(amax, std::fabs(kv.second));
    }
  std::vector<std::vector<std::pair<int, double>>> Lrows(n);
  hf.dinv.assign(n, 0.0);
  std::vector<std::vector<std::pair<int, double>>> Urows(n);
  for (int k = 0; k < n; ++k) {
    auto itp = R[k].find(k);
    const double piv = itp == R[k].end() ? 0.0 : itp->second;
    if (!(std::fabs(piv) > 1e-13 * std::max(amax, 1e-300)) || !std::isfinite(piv)) {
      why = "zero or tiny pivot in the preconditioner factor at row " + std::to_string(k);
      return false;
    }
    hf.dinv[k] = 1.0 / piv;
    for (auto& kv : R[k])
      if (kv.first > k) Urows[k].push_back(kv);
    for (int i : below[k]) {
      auto e = R[i].find(k);
      if (e == R[i].end()) continue;
      const double lik = e->second / piv;
      R[i].erase(e);
      Lrows[i].push_back({k, lik});
      for (auto& kv : Urows[k]) {
        const int j = kv.first;
        auto f = R[i].find(j);
        if (f == R[i].end()) {
          R[i][j] = -lik * kv.second;
          if (i > j) below[j].insert(i);
        } else {
          f->second -= lik * kv.second;
        }
      }
    }
  }
  for (int i = 0; i < n; ++i) std::sort(Lrows[i].begin(), Lrows[i].end());
  // a row's level is above that of every earlier row it has an L or a U
  // entry with; rows are stored level by level, the longest L rows first
  std::vector<int> lev(n, 0), fwd(n, 0), bwd(n, 0);
  int nl = 0, nf = 0, nb = 0;
  for (int i = 0; i < n; ++i) {
    for (auto& kv : Lrows[i]) {
      lev[i] = std::max(lev[i], lev[kv.first] + 1);
      fwd[i] = std::max(fwd[i], fwd[kv.first] + 1);
    }
    for (auto& kv : Urows[i]) lev[kv.first] = std::max(lev[kv.first], lev[i] + 1);
    nl = std::max(nl, lev[i] + 1);
    nf = std::max(nf, fwd[i] + 1);
  }
  for (int i = n - 1; i >= 0; --i) {
    for (auto& kv : Urows[i]) bwd[i] = std::max(bwd[i], bwd[kv.first] + 1);
    nb = std::max(nb, bwd[i] + 1);
  }
  hf.levels = nf + nb;
  std::vector<int> order(n), row(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return lev[a] != lev[b] ? lev[a] < lev[b] : Lrows[a].size() > Lrows[b].size();
  });
  for (int k = 0; k < n; ++k) row[order[k]] = k;
  const std::vector<int32_t> perm = hf.perm;
  const std::vector<double> dinv = hf.dinv;
  hf.lev_ptr.assign(nl + 1, 0);
  hf.l_ptr.push_back(0);
  hf.u_ptr.push_back(0);
  for (int k = 0; k < n; ++k) {
    const int i = order[k];
    hf.perm[k] = perm[i];
    hf.dinv[k] = dinv[i];
    ++hf.lev_ptr[lev[i] + 1];
    for (auto& kv : Lrows[i]) {   // entries stay in elimination order
      hf.l_col.push_back(row[kv.first]);
      hf.l_val.push_back(kv.second);
    }
    for (auto& kv : Urows[i]) {
      hf.u_col.push_back(row[kv.first]);
      hf.u_val.push_back(kv.second);
    }
    hf.l_ptr.push_back((int32_t)hf.l_col.size());
    hf.u_ptr.push_back((int32_t)hf.u_col.size());
  }
  for (int l = 0; l < nl; ++l) hf.lev_ptr[l + 1] += hf.lev_ptr[l];
  hf.t_lev = nl;
  while (hf.t_lev > 0 && hf.lev_ptr[hf.t_lev] - hf.lev_ptr[hf.t_lev - 1] <= NR_TAIL_ROWS)
    --hf.t_lev;
  return true;
}

template <class T>
zbus_status upload(zbus_nr_network net, T** dst, const std::vector<T>& src, cudaStream_t st) {
  const size_t bytes = std::max<size_t>(1, src.size()) * sizeof(T);
  ZB_CUDA(cudaMalloc((void**)dst, bytes));
  net->allocs.push_back(*dst);
  if (!src.empty())
    ZB_CUDA(cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, st));
  return ZBUS_OK;
}

std::vector<float> to_float(const std::vector<double>& v) {
  return std::vector<float>(v.begin(), v.end());
}

// Appends v to the index table; returns where it starts.
int append(std::vector<int32_t>& tab, const std::vector<int32_t>& v) {
  const int at = (int)tab.size();
  tab.insert(tab.end(), v.begin(), v.end());
  return at;
}

// Rows first[g] .. first[g + 1) of a CSR matrix in tiles of 32, each group
// from a tile of its own; group_tile (may be null) gets its first.
template <class V, class F>
zbus_status upload_tiles(zbus_nr_network net, std::vector<int32_t>& tab,
                         const std::vector<int32_t>& first, const std::vector<int32_t>& ptr,
                         const std::vector<int32_t>& col, const std::vector<V>& val, F to_f,
                         Tiles& t, std::vector<int32_t>* group_tile, cudaStream_t st) {
  std::vector<int32_t> tp(1, 0), tc;
  std::vector<V> tv;
  if (group_tile) group_tile->clear();
  for (size_t g = 0; g + 1 < first.size(); ++g) {
    if (group_tile) group_tile->push_back((int32_t)tp.size() - 1);
    for (int k = first[g]; k < first[g + 1]; k += 32) {
      const int rows = std::min(32, first[g + 1] - k);
      int len = 0;
      for (int i = 0; i < rows; ++i) len = std::max(len, ptr[k + i + 1] - ptr[k + i]);
      for (int q = 0; q < len; ++q)
        for (int i = 0; i < 32; ++i) {
          const bool in = i < rows && ptr[k + i] + q < ptr[k + i + 1];
          tc.push_back(in ? col[ptr[k + i] + q] : -1);
          tv.push_back(in ? val[ptr[k + i] + q] : V());
        }
      tp.push_back((int32_t)tc.size());
    }
  }
  using W = decltype(to_f(V()));
  std::vector<W> tf;
  for (const V& v : tv) tf.push_back(to_f(v));
  t.ptr = append(tab, tp);
  ZB_CHECK(upload(net, &t.col, tc, st));
  ZB_CHECK(upload(net, reinterpret_cast<V**>(&t.val), tv, st));
  return upload(net, reinterpret_cast<W**>(&t.val_f), tf, st);
}
float real_f(double v) { return (float)v; }
float2 complex_f(double2 v) { return make_float2((float)v.x, (float)v.y); }

// Steps of the rows from hf.t_lev on: in each, the 32 rows with the longest
// way still to go among those that can take an entry or have taken all.
zbus_status upload_steps(zbus_nr_network net, std::vector<int32_t>& tab, const HostFactor& hf,
                         bool upper, Steps& s, cudaStream_t st) {
  const auto& ptr = upper ? hf.u_ptr : hf.l_ptr;
  const auto& col = upper ? hf.u_col : hf.l_col;
  const auto& val = upper ? hf.u_val : hf.l_val;
  const int r0 = hf.lev_ptr[hf.t_lev], t = hf.n - r0;
  // rounds from a row's start to the end of the longest chain through it;
  // every dependence of L points back, of U forward
  std::vector<int> way(t, 1), next(t), left;
  std::vector<char> done(t, 0);
  for (int i = 0; i < t; ++i) {
    const int k = upper ? i : t - 1 - i;   // users of a row come before it
    way[k] = std::max(way[k], 1);
    const int e0 = ptr[r0 + k], e1 = ptr[r0 + k + 1];
    for (int e = e0; e < e1; ++e) {
      const int j = col[e] - r0;
      if (j >= 0) way[j] = std::max(way[j], 1 + (e1 - e + 3) / 4 + way[k] - 1);
    }
  }
  for (int k = 0; k < t; ++k) {
    next[k] = ptr[r0 + k];
    if (!upper && ptr[r0 + k] == ptr[r0 + k + 1]) done[k] = 1;
    else left.push_back(k);
  }
  std::vector<int32_t> words;
  std::vector<int2> rows;
  std::vector<int4> c;
  std::vector<double> v, di;
  while (!left.empty()) {
    struct Cand {
      int way, k, cnt;
    };
    std::vector<Cand> cand;
    for (int k : left) {
      const int e1 = ptr[r0 + k + 1];
      int cnt = 0;
      while (cnt < 4 && next[k] + cnt < e1 &&
             (col[next[k] + cnt] < r0 || done[col[next[k] + cnt] - r0]))
        ++cnt;
      if (cnt > 0 || next[k] == e1) cand.push_back({way[k] + (e1 - next[k]) / 4, k, cnt});
    }
    std::stable_sort(cand.begin(), cand.end(),
                     [](const Cand& a, const Cand& b) { return a.way > b.way; });
    if (cand.size() > 32) cand.resize(32);
    int most = 0;
    for (const Cand& x : cand) most = std::max(most, x.cnt);
    words.push_back((int32_t)rows.size());
    words.push_back((int32_t)cand.size() - 1 | most << 8);
    for (const Cand& x : cand) {
      int32_t cc[4];
      for (int q = 0; q < 4; ++q) {
        cc[q] = q < x.cnt ? col[next[x.k] + q] : net->N - 1;
        v.push_back(q < x.cnt ? val[next[x.k] + q] : 0.0);
      }
      next[x.k] += x.cnt;
      const bool last = next[x.k] == ptr[r0 + x.k + 1];
      rows.push_back(make_int2((r0 + x.k) | (last ? STEP_LAST : 0), hf.perm[r0 + x.k]));
      c.push_back(make_int4(cc[0], cc[1], cc[2], cc[3]));
      di.push_back(hf.dinv[r0 + x.k]);
      done[x.k] = last;
    }
    left.erase(std::remove_if(left.begin(), left.end(), [&](int k) { return done[k]; }),
               left.end());
  }
  s.n = (int)words.size() / 2;
  for (int i = 0; i <= STEP_AHEAD && s.n > 0; ++i)
    words.insert(words.end(), {words[2 * s.n - 2], words[2 * s.n - 1]});
  if (tab.size() & 1) tab.push_back(0);   // a step is read as one pair
  s.at = append(tab, words);
  ZB_CHECK(upload(net, &s.row, rows, st));
  ZB_CHECK(upload(net, &s.col, c, st));
  ZB_CHECK(upload(net, &s.val, v, st));
  ZB_CHECK(upload(net, &s.val_f, to_float(v), st));
  ZB_CHECK(upload(net, &s.dinv, di, st));
  return upload(net, &s.dinv_f, to_float(di), st);
}

zbus_status upload_factor(zbus_nr_network net, std::vector<int32_t>& tab, const HostFactor& hf,
                          Factor& f, cudaStream_t st) {
  f.n = hf.n;
  const int n_lev = (int)hf.lev_ptr.size() - 1;
  f.t_lev = hf.t_lev;
  f.n_lev = n_lev;
  f.levels = hf.levels;
  std::vector<int32_t> lev_tile;
  ZB_CHECK(upload_tiles(net, tab, hf.lev_ptr, hf.l_ptr, hf.l_col, hf.l_val, real_f, f.L,
                        &lev_tile, st));
  ZB_CHECK(upload_tiles(net, tab, hf.lev_ptr, hf.u_ptr, hf.u_col, hf.u_val, real_f, f.U, nullptr,
                        st));
  ZB_CHECK(upload(net, &f.perm, hf.perm, st));
  f.lev_ptr = append(tab, hf.lev_ptr);
  f.lev_tile = append(tab, lev_tile);
  ZB_CHECK(upload(net, &f.dinv, hf.dinv, st));
  ZB_CHECK(upload(net, &f.dinv_f, to_float(hf.dinv), st));
  ZB_CHECK(upload_steps(net, tab, hf, false, f.TL, st));
  ZB_CHECK(upload_steps(net, tab, hf, true, f.TU, st));
  f.nnz = (int64_t)hf.l_val.size() + (int64_t)hf.u_val.size() + hf.n;
  return ZBUS_OK;
}

// The work space bound of a grid (part of the interface): one scenario's
// shared vectors in a full-square Hessenberg layout.
size_t work_space_bound(int m, int N, bool mixed) {
  return sizeof(double) * ((size_t)(m + 1) * m + 2 * m + 2 * (m + 1) + (size_t)(m + 1) * 4) +
         (mixed ? sizeof(float) : sizeof(double)) * ((size_t)N + m + 2);
}

// Shared memory: this and, in d, where the index table stands.  A grid near
// the bound keeps the table in global memory.
size_t smem_layout(NrDev& d, int m, bool mixed) {
  const size_t y = std::max((mixed ? sizeof(float) : sizeof(double)) * (size_t)d.N,
                            sizeof(double) * NR_CHUNK * NR_THREADS);
  d.tab_at = shared_doubles(m) + (int)((y + 7) / 8);
  const size_t bytes = sizeof(double) * (size_t)d.tab_at, tab = sizeof(int32_t) * (size_t)d.tab_n;
  d.tab_shared = bytes + tab <= NR_SMEM_DYN;
  return bytes + (d.tab_shared ? tab : 0);
}

int64_t scratch_doubles(const zbus_nr_network net, int m, bool mixed) {
  const int64_t N = net->N, dim = net->nt + net->nq;
  const int64_t kv = mixed ? (krylov_values<float>(N, dim, m) + 1) / 2
                           : krylov_values<double>(N, dim, m);
  const int64_t s = state_doubles(N) + kv;
  return (s + 31) / 32 * 32;
}

}  // namespace
}  // namespace nr

ZB_CHECK_WORD_ACCESSOR(check_word_nr)

}  // namespace zbus

using namespace zbus;
using namespace zbus::nr;

extern "C" {

void zbus_nr_opts_default(zbus_nr_opts* o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->gmres_restart = 30;
  o->gmres_max_restarts = 4;
  o->gmres_tol = 1e-6;
  o->precision = ZBUS_NR_FP64;
}

zbus_status zbus_nr_network_create(int32_t N, int64_t nnz, const int32_t* row,
                                   const int32_t* col, const double* val_reim,
                                   const int32_t* bus_type, const double* v_set, double eps,
                                   void* cuda_stream, zbus_nr_network* out) {
  NvtxRange nvtx_range("zbus_nr_network_create");
  set_error("");
  if (!out) return fail(ZBUS_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (N < 2) return fail(ZBUS_ERR_ARG, "N must be >= 2");
  if (nnz < 1) return fail(ZBUS_ERR_ARG, "nnz must be >= 1");
  if (!row || !col || !val_reim || !bus_type || !v_set)
    return fail(ZBUS_ERR_ARG, "a required host array is NULL");
  if (!(eps >= 0.0) || !std::isfinite(eps)) return fail(ZBUS_ERR_ARG, "eps must be finite, >= 0");
  int slack = -1;
  for (int i = 0; i < N; ++i) {
    if (bus_type[i] < 0 || bus_type[i] > 2) return fail(ZBUS_ERR_ARG, "bus_type must be 0, 1 or 2");
    if (bus_type[i] == 2) {
      if (slack >= 0) return fail(ZBUS_ERR_ARG, "exactly one slack bus (type 2) is required");
      slack = i;
    }
    if (bus_type[i] != 0 && !(v_set[i] > 0.0 && std::isfinite(v_set[i])))
      return fail(ZBUS_ERR_ARG, "v_set of a PV or slack bus must be finite and > 0");
  }
  if (slack < 0) return fail(ZBUS_ERR_ARG, "exactly one slack bus (type 2) is required");
  std::vector<std::map<int, std::pair<double, double>>> Yrows(N);
  for (int64_t t = 0; t < nnz; ++t) {
    if (row[t] < 0 || row[t] >= N || col[t] < 0 || col[t] >= N)
      return fail(ZBUS_ERR_ARG, "COO index out of range at entry " + std::to_string(t));
    if (!std::isfinite(val_reim[2 * t]) || !std::isfinite(val_reim[2 * t + 1]))
      return fail(ZBUS_ERR_ARG, "COO value not finite at entry " + std::to_string(t));
    auto& e = Yrows[row[t]][col[t]];
    e.first += val_reim[2 * t];
    e.second += val_reim[2 * t + 1];
  }
  auto* net = new zbus_nr_network_s();
  cudaError_t ce = cudaGetDevice(&net->device);
  if (ce != cudaSuccess) {
    delete net;
    return cuda_fail(ce, "cudaGetDevice", __FILE__, __LINE__);
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  auto bail = [&](zbus_status s) {
    std::string msg = zbus_last_error();
    cudaStreamSynchronize(st);
    zbus_nr_network_destroy(net);
    set_error(msg);
    return s;
  };
  net->N = N;
  net->slack = slack;
  std::vector<int32_t> pos_t(N, -1), pos_q(N, -1), t_bus, q_bus;
  for (int i = 0; i < N; ++i) {
    if (bus_type[i] != 2) {
      pos_t[i] = (int32_t)t_bus.size();
      t_bus.push_back(i);
    }
    if (bus_type[i] == 0) {
      pos_q[i] = (int32_t)q_bus.size();
      q_bus.push_back(i);
    }
  }
  net->nt = (int)t_bus.size();
  net->nq = (int)q_bus.size();
  // Y in CSR, its longest rows first; B' and B'' (+ eps I)
  std::vector<int32_t> yr(N), yp(1, 0), yc, gp(1, 0), gc;
  std::vector<double2> yv;
  std::vector<double> gval;
  std::vector<std::map<int, double>> Bp(net->nt), Bpp(net->nq);
  for (int i = 0; i < N; ++i) yr[i] = i;
  std::stable_sort(yr.begin(), yr.end(),
                   [&](int a, int b) { return Yrows[a].size() > Yrows[b].size(); });
  for (int i : yr) {
    for (auto& kv : Yrows[i]) {
      yc.push_back(kv.first);
      yv.push_back(make_double2(kv.second.first, kv.second.second));
      const int j = kv.first;
      if (pos_t[i] >= 0 && pos_t[j] >= 0) Bp[pos_t[i]][pos_t[j]] += -kv.second.second;
      if (pos_q[i] >= 0 && pos_q[j] >= 0) Bpp[pos_q[i]][pos_q[j]] += -kv.second.second;
    }
    yp.push_back((int32_t)yc.size());
  }
  for (int p = 0; p < net->nt; ++p) Bp[p][p] += eps;
  for (int p = 0; p < net->nq; ++p) Bpp[p][p] += eps;
  HostFactor fp, fpp;
  std::string why;
  if (!factorise(net->nt, Bp, fp, why)) return bail(fail(ZBUS_ERR_SINGULAR, "B': " + why));
  if (net->nq > 0 && !factorise(net->nq, Bpp, fpp, why))
    return bail(fail(ZBUS_ERR_SINGULAR, "B'': " + why));
  // G_Q,Theta, its longest rows first
  std::vector<int2> gr(net->nq);
  for (int k = 0; k < net->nq; ++k) gr[k] = make_int2(k, q_bus[fpp.perm[k]]);
  auto g_len = [&](int bus) {
    int n = 0;
    for (auto& kv : Yrows[bus]) n += pos_t[kv.first] >= 0;
    return n;
  };
  std::stable_sort(gr.begin(), gr.end(),
                   [&](const int2& a, const int2& b) { return g_len(a.y) > g_len(b.y); });
  for (const int2& row : gr) {
    for (auto& kv : Yrows[row.y])
      if (pos_t[kv.first] >= 0) {
        gc.push_back(pos_t[kv.first]);
        gval.push_back(-kv.second.first);
      }
    gp.push_back((int32_t)gc.size());
  }
  std::vector<int32_t> row_t(N, -1), row_q(N, -1);
  for (int k = 0; k < net->nt; ++k) row_t[t_bus[fp.perm[k]]] = k;
  for (int k = 0; k < net->nq; ++k) row_q[q_bus[fpp.perm[k]]] = k;
  std::vector<int4> yrow;
  for (int i : yr) yrow.push_back(make_int4(i, row_t[i], row_q[i], 0));
  NrDev& d = net->dev;
  d.N = N;
  d.nt = net->nt;
  d.nq = net->nq;
  d.dim = net->nt + net->nq;
  std::vector<int32_t> bt(bus_type, bus_type + N);
  std::vector<double> vs(v_set, v_set + N);
  zbus_status s = ZBUS_OK;
  int4* y_row;
  int2* g_row;
  int32_t *bt_d, *pt_d, *pq_d, *rt_d, *rq_d;
  double* vs_d;
  std::vector<int32_t> tab;
  if ((s = upload(net, &y_row, yrow, st)) || (s = upload(net, &g_row, gr, st)) ||
      (s = upload_tiles(net, tab, {0, N}, yp, yc, yv, complex_f, d.Y, nullptr, st)) ||
      (s = upload_tiles(net, tab, {0, net->nq}, gp, gc, gval, real_f, d.G, nullptr, st)) ||
      (s = upload(net, &bt_d, bt, st)) || (s = upload(net, &vs_d, vs, st)) ||
      (s = upload(net, &pt_d, pos_t, st)) || (s = upload(net, &pq_d, pos_q, st)) ||
      (s = upload(net, &rt_d, row_t, st)) || (s = upload(net, &rq_d, row_q, st)) ||
      (s = upload_factor(net, tab, fp, d.Bp, st)) ||
      (net->nq > 0 && (s = upload_factor(net, tab, fpp, d.Bpp, st))))
    return bail(s);
  int32_t* tab_d;
  if ((s = upload(net, &tab_d, tab, st))) return bail(s);
  d.tab = tab_d;
  d.tab_n = (int)tab.size();
  d.y_row = y_row;
  d.g_row = g_row;
  d.bus_type = bt_d;
  d.v_set = vs_d;
  d.pos_t = pt_d;
  d.pos_q = pq_d;
  d.row_t = rt_d;
  d.row_q = rq_d;
  ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return bail(cuda_fail(ce, "setup copies", __FILE__, __LINE__));
  int dev = net->device;
  cudaDeviceGetAttribute(&net->sms, cudaDevAttrMultiProcessorCount, dev);
  *out = net;
  return ZBUS_OK;
}

void zbus_nr_network_destroy(zbus_nr_network net) {
  if (!net) return;
  for (void* p : net->allocs) cudaFree(p);
  cudaFree(net->scratch);
  delete net;
}

zbus_status zbus_nr_network_info(zbus_nr_network net, int32_t* n_theta, int32_t* n_q,
                                 int64_t* factor_nnz, int32_t* factor_levels) {
  set_error("");
  if (!net) return fail(ZBUS_ERR_ARG, "network is NULL");
  if (n_theta) *n_theta = net->nt;
  if (n_q) *n_q = net->nq;
  if (factor_nnz) *factor_nnz = net->dev.Bp.nnz + net->dev.Bpp.nnz;
  if (factor_levels)
    *factor_levels = net->dev.Bp.levels + net->dev.Bpp.levels;
  return ZBUS_OK;
}

zbus_status zbus_nr_solve(zbus_nr_network net, int64_t B, const double* P, const double* Q,
                          double tol, int32_t max_iter, const zbus_nr_opts* opts, double* V_out,
                          int32_t* iters, uint8_t* converged, int32_t* gmres_iters,
                          void* cuda_stream) {
  NvtxRange nvtx_range("zbus_nr_solve");
  set_error("");
  if (!net) return fail(ZBUS_ERR_ARG, "network is NULL");
  if (B < 0 || B > INT32_MAX) return fail(ZBUS_ERR_ARG, "B out of range");
  if (!(tol >= 0.0) || !std::isfinite(tol)) return fail(ZBUS_ERR_ARG, "tol must be finite, >= 0");
  if (max_iter < 0) return fail(ZBUS_ERR_ARG, "max_iter must be >= 0");
  zbus_nr_opts o;
  zbus_nr_opts_default(&o);
  if (opts) o = *opts;
  if (o.gmres_restart < 1 || o.gmres_restart > NR_MAX_RESTART_LEN)
    return fail(ZBUS_ERR_ARG, "gmres_restart must be in 1 .. 60");
  if (o.gmres_max_restarts < 1) return fail(ZBUS_ERR_ARG, "gmres_max_restarts must be >= 1");
  if (!(o.gmres_tol > 0.0) || !(o.gmres_tol < 1.0))
    return fail(ZBUS_ERR_ARG, "gmres_tol must be in (0, 1)");
  if (o.precision != ZBUS_NR_FP64 && o.precision != ZBUS_NR_MIXED)
    return fail(ZBUS_ERR_ARG, "unknown NR precision");
  if (B == 0) return ZBUS_OK;
  if (!P || !Q || !V_out || !iters || !converged)
    return fail(ZBUS_ERR_ARG, "P, Q, V_out, iters and converged are required");
  int dev = -1;
  ZB_CUDA(cudaGetDevice(&dev));
  if (dev != net->device) return fail(ZBUS_ERR_ARG, "current CUDA device differs from the network's");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int m = o.gmres_restart;
  const bool mixed = o.precision == ZBUS_NR_MIXED;
  if (work_space_bound(m, net->N, mixed) > NR_SMEM_MAX)
    return fail(ZBUS_ERR_ARG, "grid too large for the per-CTA shared work space");
  NrDev d = net->dev;
  const size_t smem = smem_layout(d, m, mixed);
  const void* kern = mixed ? (const void*)k_nr_solve<float> : (const void*)k_nr_solve<double>;
  if (!net->smem_set[mixed]) {
    ZB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)NR_SMEM_DYN));
    net->smem_set[mixed] = true;
  }
  int per = 0;
  ZB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, NR_THREADS, smem));
  const int64_t ctas = std::min<int64_t>(B, (int64_t)net->sms * std::max(1, per));
  const int64_t stride = scratch_doubles(net, m, mixed);
  if (net->scratch_size < ctas * stride) {
    ZB_CUDA(cudaStreamSynchronize(st));
    cudaFree(net->scratch);
    net->scratch = nullptr;
    net->scratch_size = 0;
    ZB_CUDA(cudaMalloc((void**)&net->scratch, (size_t)ctas * stride * sizeof(double)));
    net->scratch_size = ctas * stride;
  }
  d.m = m;
  d.scratch = net->scratch;
  d.stride = stride;
  SolveArgs a;
  a.B = (int)B;
  a.P = P;
  a.Q = Q;
  a.tol = tol;
  a.max_iter = max_iter;
  a.eta = o.gmres_tol;
  a.max_restart = o.gmres_max_restarts;
  a.V = (double2*)V_out;
  a.iters = iters;
  a.conv = converged;
  a.gmres = gmres_iters;
  if (mixed)
    k_nr_solve<float><<<(int)ctas, NR_THREADS, smem, st>>>(d, a);
  else
    k_nr_solve<double><<<(int)ctas, NR_THREADS, smem, st>>>(d, a);
  ZB_CUDA(cudaGetLastError());
  return ZBUS_OK;
}

}  // extern "C"
