// The cycle below a level as one stored matrix.
//
// From x = 0, what Algorithm 1 does on level l and below (every sweep, transfer and the
// coarsest solve, nu times) is linear in the level's right-hand side: x_l = M b_l with a
// dense m x m matrix M, m the level's unknowns.  Run operation by operation it is a chain
// of about 2 x 30 colours and 5 other launches a level, each a few microseconds whatever
// the level's size (elasticity 32^3, FP32: 280 us of the 774 us preconditioner below
// level 1, for 8,538 unknowns; FP64 24^3: 690 us of 1317 us for 3,144).  M b instead reads
// m^2 values once.  M is filled at setup by running the cycle's own recorded operations on
// blocks of unit vectors, so it is the same operator, weights, smoother and cycle type, in the
// cycle's precision.  It follows the weights that a program sets before its first solve.  Under
// other weights later the cycle runs operation by operation, until M is filled for them
// (map_refresh); back under its own weights M is in use again.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "amg_internal.cuh"
#include "phase.cuh"
#include "vec.cuh"

namespace amgp2 {

namespace {

// ------------------------------------------------------------------- blocks of vectors

// A block of W vectors is stored entry by entry: entry k of vector c at k * W + c, so
// consecutive threads take consecutive vectors and every value of an operator is one
// broadcast load for a warp.  A thread holds 2 vectors (16 bytes an entry).
//
// FP64 handles build in FP64.  FP32 handles build in FP32 pairs (hi + lo) with the cycle's own
// FP32 (or BF16) operator values, to well below the rounding of M to FP32 that follows (mac
// below: not to the 2^-48 of the Krylov operator's pairs).  M b is then about as far from the
// FP64 cycle as the FP32 operations: 0.89 to 0.98 times for elasticity and the Laplacian,
// 0.94 to 1.10 for mixed elasticity (kMapMaxCond and kMapStokesFrom say where it is further).
// Built in plain FP32, M doubled that error (32^3: 7.1e-7 against 3.4e-7 relative).  FP64 would
// take the m nnz FMAs of three sweeps at 0.5e12 a second (87 ms at 32^3); the pairs issue at
// the FP32 rate.
constexpr int kColThreads = 128;
constexpr int kColN = 2;                             // vectors of a thread
constexpr int kColBlock = kColThreads * kColN;       // vectors of a CTA
constexpr int kColMax = 20 * kColBlock;              // vectors of one pass

struct Pair {
  float h, l;
};
__device__ __forceinline__ void mac(double& s, double a, double x) { s = fma(a, x, s); }
// s += a x: the rounded sum and its error, exact where |s| >= |a x| (FastTwoSum with the
// product unrounded); a step where the product is the larger one may lose its rounding
// error, as a plain FP32 step does, which the result, rounded to FP32, can bear
__device__ __forceinline__ void mac(Pair& s, float a, Pair x) {
  const float t = fmaf(a, x.h, s.h);
  const float e = fmaf(a, x.h, __fsub_rn(s.h, t));
  s.l = fmaf(a, x.l, s.l) + e;
  s.h = t;
}
__device__ __forceinline__ void add(double& s, double x) { s += x; }
__device__ __forceinline__ void add(Pair& s, Pair x) { pair_add(s.h, s.l, x.h, x.l); }
__device__ __forceinline__ double scaled(double om, double s, double d) { return om * s / d; }
__device__ __forceinline__ Pair scaled(float om, Pair s, float d) {   // om s / d
  Pair t{0.f, 0.f};
  mac(t, om, s);
  const float q = t.h / d;
  return {q, (fmaf(-q, d, t.h) + t.l) / d};
}
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(Pair x) { return (double)x.h + (double)x.l; }
__device__ __forceinline__ void narrow(double& x, double v) { x = v; }
__device__ __forceinline__ void narrow(Pair& x, double v) {
  x.h = (float)v;
  x.l = (float)(v - (double)x.h);
}
__device__ __forceinline__ double normal(double x) { return x; }
__device__ __forceinline__ Pair normal(Pair x) {   // |h| >= |l| (FastTwoSum)
  const float h = __fadd_rn(x.h, x.l);
  return {h, __fsub_rn(x.l, __fsub_rn(h, x.h))};
}
__device__ __forceinline__ double round_to(double, double x) { return x; }
__device__ __forceinline__ float round_to(float, Pair x) { return x.h; }

template <typename T>
struct alignas(16) Cell {   // an entry of neighbouring vectors
  T v[kColN];
};
template <typename T>
__device__ __forceinline__ Cell<T> ldc(const T* p) {
  union { float4 f; Cell<T> c; } u;
  u.f = *reinterpret_cast<const float4*>(p);
  return u.c;
}
template <typename T>
__device__ __forceinline__ void stc(T* p, const Cell<T>& c) {
  union { float4 f; Cell<T> c; } u;
#pragma unroll
  for (int q = 0; q < kColN; ++q) u.c.v[q] = normal(c.v[q]);
  *reinterpret_cast<float4*>(p) = u.f;
}
template <typename T>
__device__ __forceinline__ Cell<T> zero() {
  return Cell<T>{};
}
template <typename T, typename S>
__device__ __forceinline__ void axpy(Cell<T>& s, S a, const Cell<T>& x) {
#pragma unroll
  for (int q = 0; q < kColN; ++q) mac(s.v[q], a, x.v[q]);
}
template <typename T>
__device__ __forceinline__ void add(Cell<T>& s, const Cell<T>& x) {
#pragma unroll
  for (int q = 0; q < kColN; ++q) add(s.v[q], x.v[q]);
}
template <typename S, typename V>
__device__ __forceinline__ S value(const V* p) {
  if constexpr (std::is_same<S, V>::value) return __ldg(p);
  else return __bfloat162float(__ldg(p));
}
// unpadded unknown j -> entry of the padded layout
__device__ __forceinline__ int pad_index(int j, int n3) {
  return j < n3 ? 4 * (j / 3) + j % 3 : j + n3 / 3;
}

// block rows of A (rows_body of the cycle): CTA per row and column block.  T: entries of
// the vectors; S: operator scalars; V: storage of the block values.  L2 traffic of the
// gathered blocks and the pair operations bound it about equally: 14 ms of launches for
// m = 8,586 (12x13x14), within 10 % for CTAs of 32 to 128 threads and 2 or 4 sums.
template <typename T, typename S, typename V>
__global__ void __launch_bounds__(kColThreads) k_cols_rows(const Phase P, int W) {
  const int g = blockIdx.x;
  const int64_t c = (int64_t)blockIdx.y * kColBlock + threadIdx.x * kColN;
  const T* x = (const T*)P.x + c;
  const V* val = (const V*)P.val;
  const int i = P.rows ? __ldg(P.rows + g) : g;
  const int a = __ldg(P.rowptr + g), e = __ldg(P.rowend + g);
  // the row's columns and values staged in shared memory, kStage blocks at a time; A sums
  // of every A-th block each, whose loads are in flight together
  constexpr int A = 4, kStage = 64;
  __shared__ int sj[kStage];
  __shared__ S sv[kStage][9];
  Cell<T> s[A][3];
#pragma unroll
  for (int u = 0; u < A; ++u)
#pragma unroll
    for (int q = 0; q < 3; ++q) s[u][q] = zero<T>();
  if (P.crow) {   // saddle levels: with B^T p
    const S* bv = (const S*)P.cval;
    for (int t = P.crow[i]; t < P.crow[i + 1]; ++t) {
      const Cell<T> p = ldc((const T*)P.sd + c + (int64_t)P.ccol[t] * W);
#pragma unroll
      for (int q = 0; q < 3; ++q) axpy(s[1][q], __ldg(bv + (int64_t)q * P.n3 + t), p);
    }
  }
  for (int k0 = a; k0 < e; k0 += kStage) {
    const int n = min(kStage, e - k0);
    __syncthreads();
    for (int t = threadIdx.x; t < 9 * n; t += kColThreads)
      sv[t % n][t / n] = value<S>(val + (t / n) * P.nnz + k0 + t % n);
    for (int t = threadIdx.x; t < n; t += kColThreads) sj[t] = 4 * __ldg(P.col + k0 + t);
    __syncthreads();
    int k = 0;
    for (; k + A <= n; k += A) {
      Cell<T> xv[A][3];
#pragma unroll
      for (int u = 0; u < A; ++u)
#pragma unroll
        for (int q = 0; q < 3; ++q) xv[u][q] = ldc(x + (int64_t)(sj[k + u] + q) * W);
#pragma unroll
      for (int u = 0; u < A; ++u)
#pragma unroll
        for (int q = 0; q < 9; ++q) axpy(s[u][q / 3], sv[k + u][q], xv[u][q % 3]);
    }
    for (; k < n; ++k)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const Cell<T> v = ldc(x + (int64_t)(sj[k] + q) * W);
#pragma unroll
        for (int p = 0; p < 3; ++p) axpy(s[0][p], sv[k][3 * p + q], v);
      }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    add(s[0][q], s[1][q]);
    add(s[2][q], s[3][q]);
    add(s[0][q], s[2][q]);
  }
  T* y = (T*)P.y + c;
  const int64_t o = 4 * (int64_t)i * W;
  if (P.mode == kApply) {
#pragma unroll
    for (int q = 0; q < 3; ++q) stc(y + o + q * W, s[0][q]);
    return;
  }
  const T* b = (const T*)P.b + c;
  Cell<T> r[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    r[q] = ldc(b + o + q * W);
#pragma unroll
    for (int w = 0; w < kColN; ++w) s[0][q].v[w] = normal(s[0][q].v[w]);
    axpy(r[q], S(-1), s[0][q]);
    if (P.mode == kResid) stc(y + o + q * W, r[q]);
#pragma unroll
    for (int w = 0; w < kColN; ++w) r[q].v[w] = normal(r[q].v[w]);
  }
  if (P.mode == kResid) return;
  const S* wt = (const S*)P.wt;
  const S om = wt ? wt[0] : (S)P.omega;
  const S* d = (const S*)P.dinv + 12 * (int64_t)i;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    Cell<T> t = zero<T>(), xi = zero<T>();
    if (P.mode != kFirst) xi = ldc(x + o + q * W);
#pragma unroll
    for (int p = 0; p < 3; ++p) axpy(t, __ldg(d + 4 * q + p), r[p]);
    if (P.mode == kFirst && P.p) {
      Cell<T> u = zero<T>();
      axpy(u, S(1) - om, r[q]);
      stc((T*)P.p + c + o + q * W, u);
    }
#pragma unroll
    for (int w = 0; w < kColN; ++w) t.v[w] = normal(t.v[w]);
    axpy(xi, om, t);
    stc(y + o + q * W, xi);
  }
}

// the other operations of the cycle, CTA per item (row, node or entry) and column block
template <typename T, typename S>
__global__ void __launch_bounds__(kColThreads) k_cols_phase(const Phase P, int W) {
  const int i = blockIdx.x;
  const int64_t c = (int64_t)blockIdx.y * kColBlock + threadIdx.x * kColN;
  const T* x = (const T*)P.x + c;
  const T* b = (const T*)P.b + c;
  T* y = (T*)P.y + c;
  const S* val = (const S*)P.val;
  const S* wt = (const S*)P.wt;
  const int64_t o = (int64_t)i * W, o4 = 4 * (int64_t)i * W;
  auto norm = [](Cell<T> v) {
#pragma unroll
    for (int w = 0; w < kColN; ++w) v.v[w] = normal(v.v[w]);
    return v;
  };
  switch (P.type) {
    case PH_COPY: stc(y + o, ldc(x + o)); break;
    case PH_RESTRICT:
    case PH_PROLONG: {
      if (i >= P.n) {   // the pressure rows of a saddle level's transfer
        const int k = i - P.n;
        const int64_t d = (4 * (int64_t)P.n + k) * W;
        Cell<T> s = zero<T>();
        for (int t = P.crow[k]; t < P.crow[k + 1]; ++t)
          axpy(s, ((const S*)P.cval)[t], ldc(x + (4 * (int64_t)P.n3 + P.ccol[t]) * W));
        if (P.type == PH_PROLONG) {
          Cell<T> v = ldc(b + d);
          axpy(v, wt ? wt[1] : S(1), norm(s));
          s = v;
        }
        stc(y + d, s);
        break;
      }
      Cell<T> s[3] = {zero<T>(), zero<T>(), zero<T>()};
      for (int t = P.rowptr[i]; t < P.rowptr[i + 1]; ++t) {
        const int64_t j = 4 * (int64_t)P.col[t] * W;
#pragma unroll
        for (int q = 0; q < 3; ++q) axpy(s[q], val[t], ldc(x + j + q * W));
      }
      const S wc = wt ? wt[1] : S(1);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (P.type == PH_PROLONG) {
          Cell<T> v = ldc(b + o4 + q * W);
          axpy(v, wc, norm(s[q]));
          s[q] = v;
        }
        stc(y + o4 + q * W, s[q]);
      }
      break;
    }
    case PH_RESTRICT1:
    case PH_PROLONG1: {
      Cell<T> s = zero<T>();
      for (int t = P.rowptr[i]; t < P.rowptr[i + 1]; ++t)
        axpy(s, val[t], ldc(x + (int64_t)P.col[t] * W));
      if (P.type == PH_PROLONG1) {
        Cell<T> v = ldc(y + o);
        axpy(v, wt ? wt[1] : S(1), norm(s));
        s = v;
      }
      stc(y + o, s);
      break;
    }
    case PH_COARSE: {   // the generalised inverse in FP64, as in the cycle
      double s[kColN] = {};
      for (int j = 0; j < P.m; ++j) {
        const double X = P.X[(int64_t)i * P.m + j];
        const Cell<T> v = ldc(b + (int64_t)pad_index(j, P.n3) * W);
#pragma unroll
        for (int q = 0; q < kColN; ++q) s[q] = fma(X, wide(v.v[q]), s[q]);
      }
      Cell<T> t;
#pragma unroll
      for (int q = 0; q < kColN; ++q) narrow(t.v[q], s[q]);
      stc(y + (int64_t)pad_index(i, P.n3) * W, t);
      break;
    }
    case PH_BT_ADD: {
      Cell<T> s[3] = {zero<T>(), zero<T>(), zero<T>()};
      for (int t = P.rowptr[i]; t < P.rowptr[i + 1]; ++t) {
        const Cell<T> p = ldc(x + (int64_t)P.col[t] * W);
#pragma unroll
        for (int q = 0; q < 3; ++q) axpy(s[q], val[q * P.nnz + t], p);
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        Cell<T> v = ldc(y + o4 + q * W);
        axpy(v, (S)P.omega, norm(s[q]));
        stc(y + o4 + q * W, v);
      }
      break;
    }
    case PH_PROWS: {
      const T* p = (const T*)P.p + c;
      Cell<T> s = zero<T>(), cp = zero<T>();
      for (int t = P.rowptr[i]; t < P.rowptr[i + 1]; ++t) {
        const int64_t j = 4 * (int64_t)P.col[t] * W;
#pragma unroll
        for (int q = 0; q < 3; ++q) axpy(s, val[q * P.nnz + t], ldc(x + j + q * W));
      }
      if (P.mode != 3 && P.mode != 4)
        for (int t = P.crow[i]; t < P.crow[i + 1]; ++t)
          axpy(cp, ((const S*)P.cval)[t], ldc(p + (int64_t)P.ccol[t] * W));
      axpy(s, S(-1), norm(cp));                        // B u - C p
      if (P.mode == 1) {
        Cell<T> g = ldc(b + o);
        axpy(g, S(-1), norm(s));
        s = g;
      } else if (P.mode == 3) {
        axpy(s, S(-1), ldc(b + o));
      } else if (P.mode == 2 || P.mode == 4) {
        const S om = wt ? wt[3] : (S)P.omega;
        const S d = ((const S*)P.sd)[i];
        axpy(s, S(-1), ldc(b + o));
        s = norm(s);
        Cell<T> v = P.mode == 2 ? ldc(p + o) : zero<T>();
        if (d != S(0)) {
#pragma unroll
          for (int q = 0; q < kColN; ++q) add(v.v[q], scaled(om, s.v[q], d));
        }
        s = v;
      }
      stc(y + o, s);
      break;
    }
    case PH_SROWS: {
      Cell<T> s = ldc(b + o);
      for (int t = P.rowptr[i]; t < P.rowptr[i + 1]; ++t)
        axpy(s, -val[t], ldc(x + (int64_t)P.col[t] * W));
      if (P.mode == 1) {
        Cell<T> v = ldc(x + o);
        axpy(v, (S)P.omega * ((const S*)P.dinv)[i], norm(s));
        s = v;
      }
      stc(y + o, s);
      break;
    }
    case PH_VEC: {
      Cell<T> v = zero<T>();
      if (P.mode == 0) {
        axpy(v, (S)P.omega * ((const S*)P.dinv)[i], ldc(x + o));
      } else {
        v = ldc(y + o);
        add(v, ldc(x + o));
        if (P.mode == 2) axpy(v, -((const S*)P.dinv)[i], ldc(b + o));
      }
      stc(y + o, v);
      break;
    }
    default:
      break;
  }
}

// unit vectors first, first + 1, ... of the level's m unknowns (the block is zero before)
template <typename T>
__global__ void k_cols_unit(T* b, int first, int m, int n3, int W) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < W && first + c < m) narrow(b[(int64_t)pad_index(first + c, n3) * W + c], 1.0);
}

// columns first.. of M from the block's solution vectors
template <typename T, typename S>
__global__ void k_cols_store(const T* __restrict__ x, S* __restrict__ M, int first, int m, int ld,
                             int n3, int W) {
  const int j = blockIdx.x;
  for (int c = threadIdx.x; c < W && first + c < m; c += blockDim.x)
    M[(int64_t)j * ld + first + c] = round_to(S(0), x[(int64_t)pad_index(j, n3) * W + c]);
}

// The blocks of vectors that stand for the level work vectors while phases run on W
// columns: a phase's vector operand is found by the level vector that it points into.
template <typename T, typename S>
struct ColVectors {
  struct Range {
    const S* base;
    int64_t n;
    int64_t at;
  };
  std::vector<Range> ranges;
  int64_t total = 0;
  DBuf<T> mem;

  void add(const DBuf<S>& v) {
    if (v.p) ranges.push_back({v.p, (int64_t)v.n, -1});
  }
  Range* find(const void* p) {
    const S* q = static_cast<const S*>(p);
    for (Range& r : ranges)
      if (q >= r.base && q < r.base + r.n) return &r;
    return nullptr;
  }
  void use(const void* p) {   // gives the vector of p its place
    Range* r = p ? find(p) : nullptr;
    if (r && r->at < 0) {
      r->at = total;
      total += r->n;
    }
  }
  T* map(const void* p, int W) {
    Range* r = find(p);
    return r ? mem.p + (r->at + (static_cast<const S*>(p) - r->base)) * W : nullptr;
  }
};

void add_level(ColVectors<double, double>& v, const Level& l) {
  v.add(l.x64); v.add(l.b64); v.add(l.r64); v.add(l.t64);
  for (const auto& s : l.S) { v.add(s->x64); v.add(s->b64); v.add(s->r64); }
}
void add_level(ColVectors<Pair, float>& v, const Level& l) {
  v.add(l.x32); v.add(l.b32); v.add(l.r32); v.add(l.t32);
  for (const auto& s : l.S) { v.add(s->x32); v.add(s->b32); v.add(s->r32); }
}

template <typename T, typename S>
void run_cols(amg_handle* h, const Phase& P, int W) {
  cudaStream_t s = h->stream;
  if (P.type == PH_ZERO) {
    if (P.n > 0) AMG_CUDA(cudaMemsetAsync(P.y, 0, (size_t)P.n * W * sizeof(T), s));
    return;
  }
  const int items = P.type == PH_COARSE                              ? P.m
                    : P.type == PH_RESTRICT || P.type == PH_PROLONG ? P.n + P.m
                                                                     : P.n;
  if (items <= 0) return;
  const dim3 grid(items, W / kColBlock);
  if (P.type != PH_ROWS) {
    k_cols_phase<T, S><<<grid, kColThreads, 0, s>>>(P, W);
  } else if (P.vbf) {
    if constexpr (std::is_same<S, float>::value)
      k_cols_rows<T, float, __nv_bfloat16><<<grid, kColThreads, 0, s>>>(P, W);
  } else {
    k_cols_rows<T, S, S><<<grid, kColThreads, 0, s>>>(P, W);
  }
  h->launches++;
}

// M (the handle's precision S) from the cycle's operations on blocks of T vectors
template <typename T, typename S>
void build(amg_handle* h, const CoarseMap& map, S* M) {
  // all columns at once up to kColMax: a launch's CTAs go over the rows of a colour first,
  // so a block of 256 columns keeps its vectors in L2, and the small colours still fill the
  // chip (512 columns a pass at 32^3: 97 ms, all but a few launches waiting on latency)
  const int from = map.level, m = map.m;
  int W = div_up(div_up(m, div_up(m, kColMax)), kColBlock) * kColBlock;
  std::vector<Phase> ph;
  record_map_phases<S>(h, from, ph);
  ColVectors<T, S> v;
  for (size_t l = from; l < h->L.size(); ++l) add_level(v, *h->L[l]);
  const Level& lv = *h->L[from];
  constexpr bool f32 = std::is_same<S, float>::value;
  const void* lb = f32 ? (const void*)lv.b32.p : lv.b64.p;
  const void* lx = f32 ? (const void*)lv.x32.p : lv.x64.p;
  v.use(lb);
  v.use(lx);
  for (const Phase& P : ph)
    for (const void* q : {P.x, P.b, P.p, (const void*)P.y, P.type == PH_ROWS ? P.sd : nullptr})
      v.use(q);
  for (;;) {   // fewer columns a pass where the device has no room (1.6 GB at m = 8,538)
    try {
      v.mem.alloc((size_t)v.total * W);
      break;
    } catch (const Error& e) {
      if (e.code != AMG_ERR_NOMEM || W <= kColBlock) throw;
      W = std::max(kColBlock, W / 2 / kColBlock * kColBlock);
    }
  }
  T* b = v.map(lb, W);
  T* x = v.map(lx, W);
  for (Phase& P : ph) {
    for (const void** q : {&P.x, &P.b, &P.p})
      if (*q) *q = v.map(*q, W);
    P.y = v.map(P.y, W);
    if (P.type == PH_ROWS && P.sd) P.sd = v.map(P.sd, W);
  }
  AMG_CUDA(cudaMemsetAsync(v.mem.p, 0, v.mem.bytes(), h->stream));
  const int n3 = 3 * lv.n;
  for (int first = 0; first < m; first += W) {
    AMG_CUDA(cudaMemsetAsync(b, 0, (size_t)lv.dofs4() * W * sizeof(T), h->stream));
    k_cols_unit<T><<<div_up(W, 256), 256, 0, h->stream>>>(b, first, m, n3, W);
    for (const Phase& P : ph) run_cols<T, S>(h, P, W);
    k_cols_store<T, S><<<m, 256, 0, h->stream>>>(x, M, first, m, map.ld, n3, W);
    h->launches += 2;
  }
  AMG_LAUNCH_CHECK();
  AMG_CUDA(cudaStreamSynchronize(h->stream));   // the blocks are freed here
}

// ------------------------------------------------------------------- application

constexpr int kMapThreads = 256;

// the products of 16 bytes of a row, added to a running sum (FP32: with its rounding
// error, TwoSum, so that a row's sum of thousands of terms loses no more than the short
// sums of the cycle's sparse rows)
template <typename T> struct Stream16;
template <> struct Stream16<float> {
  using type = float4;
  struct Sum {
    float s = 0.f, e = 0.f;
    __device__ void add(float4 a, float4 b) {
      const float d = fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, __fmul_rn(a.x, b.x))));
      pair_add(s, e, d, 0.f);
    }
    __device__ void join(const Sum& o) { pair_add(s, e, o.s, o.e); }
    __device__ void lane(int o) {
      const float t = __shfl_xor_sync(0xffffffffu, s, o);
      const float u = __shfl_xor_sync(0xffffffffu, e, o);
      pair_add(s, e, t, u);
    }
    __device__ float value() const { return s + e; }
  };
};
template <> struct Stream16<double> {
  using type = double2;
  struct Sum {
    double s = 0.0;
    __device__ void add(double2 a, double2 b) { s = fma(a.y, b.y, fma(a.x, b.x, s)); }
    __device__ void join(const Sum& o) { s += o.s; }
    __device__ void lane(int o) { s += __shfl_xor_sync(0xffffffffu, s, o); }
    __device__ double value() const { return s; }
  };
};

// x = M b, padded vectors of IO converted to T (FP32 handles at level 0 take the outer
// FP64 vectors directly).  One warp a row at a time; b is staged unpadded in shared memory
// by every CTA; the row's values stream with U 16-byte loads in flight a lane.  STREAM:
// evict-first loads for a matrix beyond the L2 capacity, so that it does not push out the
// vectors; a smaller one is left to stay in L2 from one application to the next.  Memory
// bound in FP32 (m = 8,538: 292 MB in 52 us, 5.6 TB/s), by the FP64 issue rate in FP64
// (m = 2,187: 16 us, 9.5 us of it FMAs).
template <typename T, typename IO, bool STREAM>
__global__ void __launch_bounds__(kMapThreads) k_map_apply(int m, int ld, int n3,
                                                           const T* __restrict__ M,
                                                           const IO* __restrict__ b,
                                                           IO* __restrict__ x) {
  using V = typename Stream16<T>::type;
  constexpr int N = 16 / sizeof(T), U = 8;
  extern __shared__ __align__(16) unsigned char map_smem[];
  T* sb = reinterpret_cast<T*>(map_smem);
  for (int j = threadIdx.x; j < ld; j += kMapThreads)
    sb[j] = j < m ? (T)b[pad_index(j, n3)] : T(0);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (kMapThreads / 32);
  const V* sv = reinterpret_cast<const V*>(sb);
  const int nv = ld / N;
  for (int i = blockIdx.x * (kMapThreads / 32) + (threadIdx.x >> 5); i < m; i += nw) {
    const V* row = reinterpret_cast<const V*>(M + (int64_t)i * ld);
    typename Stream16<T>::Sum s[4];
    for (int k = lane; k < nv; k += 32 * U) {
      V a[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + 32 * u < nv) a[u] = STREAM ? __ldcs(row + k + 32 * u) : __ldg(row + k + 32 * u);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + 32 * u < nv) s[u & 3].add(a[u], sv[k + 32 * u]);
    }
    s[0].join(s[1]);
    s[2].join(s[3]);
    s[0].join(s[2]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[0].lane(o);
    if (lane == 0) {
      const int o = pad_index(i, n3);
      x[o] = (IO)s[0].value();
      if (i < n3 && (o & 3) == 2) x[o + 1] = IO(0);   // the node's padding
    }
  }
}

// X = M B for kRhs = 16 vectors in planes of four (map_plane).  A CTA takes R rows; its 8
// warps share the columns (32 a step), so a lane multiplies one column of R rows with the
// column's 16 entries of B: per step R coalesced 4-byte loads of M and 4 coalesced 16-byte
// loads of B for 16 R FMAs.  The lanes' sums are reduced by halving exchanges (lane L ends
// with R / 2 of the 16 R sums), then across the warps in shared memory.  FP32 issue bounds it
// (16 m^2 FMAs: 2 us at m = 2,048 with the chip to itself).
template <int R>
__global__ void __launch_bounds__(256, R == 8 ? 1 : 2) k_map_m(int m, int ld,
                                                               const float* __restrict__ M,
                                                               const float* __restrict__ B,
                                                               float* __restrict__ X) {
  constexpr int V = R * kRhs;
  __shared__ float red[8][V];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row0 = blockIdx.x * R;
  const float4* b4 = reinterpret_cast<const float4*>(B);
  float v[V];
#pragma unroll
  for (int i = 0; i < V; ++i) v[i] = 0.f;
#pragma unroll 2
  for (int k = w * 32 + lane; k < m; k += 256) {
    float a[R];
    float4 b[4];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = __ldg(M + (int64_t)min(row0 + r, m - 1) * ld + k);
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = __ldg(b4 + (int64_t)q * m + k);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float* s = v + r * kRhs + 4 * q;
        s[0] = fmaf(a[r], b[q].x, s[0]);
        s[1] = fmaf(a[r], b[q].y, s[1]);
        s[2] = fmaf(a[r], b[q].z, s[2]);
        s[3] = fmaf(a[r], b[q].w, s[3]);
      }
  }
  int first = 0;
#pragma unroll
  for (int o = 16, n = V / 2; o > 0; o >>= 1, n >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float other = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + n], o);
      v[i] = (up ? v[i + n] : v[i]) + other;
    }
    first += up ? n : 0;
  }
#pragma unroll
  for (int i = 0; i < V / 32; ++i) red[w][first + i] = v[i];
  __syncthreads();
  const int t = threadIdx.x, row = row0 + t / kRhs, r = t % kRhs;
  if (t < V && row < m) {
    float s = 0.f, e = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) pair_add(s, e, red[q][t], 0.f);
    X[map_plane(m, row, r)] = s + e;
  }
}

template <typename T>
const T* matrix(const CoarseMap& M) {
  if constexpr (std::is_same<T, float>::value) return M.m32.p;
  else return M.m64.p;
}

// The largest level stored as a matrix.  Below these sizes M b is faster than the chain
// of launches that it replaces: reading M takes 4 m^2 bytes at 5.6 TB/s in FP32 (75 us at
// 10,240; 52 us at 8,538, in place of 280 us) against 65 launches of 2 to 5 us and the levels
// below; in FP64 the m^2 FMAs take 75 us at 6,144 (0.5e12 a second on this GPU).  They also
// bound the memory (420 and 300 MB) and the time of the construction (20 ms at 8,538).
constexpr int kMapMax32 = 10240;
constexpr int kMapMax64 = 6144;
// A segregated Gauss-Seidel level is 7 launches, not 65, so a large map saves less beyond the
// next smaller one.  Mixed elasticity, an application with the map of the size given against
// the next smaller, and its construction:
//   FP32  3,065 (9^3) 70 against 117 us, 3.6 ms     4,159 (24^3) 251 against 295, 3.6 ms
//         6,371 (28^3) 353 against 388, 7.8 ms      8,706 (13x11x15) 122 against 130, 13 ms
//         9,267 (32^3) 485 against 499, 18 ms
//   FP64  3,065 108 against 172 us, 7.0 ms          4,159 525 against 579, 15 ms
// An FGMRES solve is 50 to 130 applications: up to 4,159 a solve repays it in FP32 (in FP64
// three do), at 6,371 two to four, beyond that ten and more.
constexpr int kMapMaxSgs = 4608;
// Applications operation by operation, under weights that M was not built with, after which
// it is filled for them: by then what M would have saved is about what filling it costs, so a
// program that changes weights often loses nothing and one that keeps them waits at most
// about twice.  Measured filling time over the time that an application saves: FP32 14 at
// 1,029 unknowns, 16 at 1,263, 35 at 2,793, 37 at 4,159, 90 at 8,538; FP64 15 at 828, 14 at
// 1,029, 40 at 2,793, 115 at 4,159 (Stokes, whose cycle saves least).
inline int64_t map_pays(const CoarseMap& M) { return 10 + M.m / (M.m32.p ? 100 : 60); }

// The worst conditioned diagonal block (row-sum norms) with which a cycle is stored.  M b
// cancels where the operations do not: a block with directions of very different stiffness,
// not along the axes, mixes them in every entry of M.  Against the cycle in FP64 (elasticity
// 12x11x13, its blocks D taken to Q S D S Q^T with S = diag(1, t, 1)), FP32:
//   t = 8    (condition 113)    operations 5.5e-7, stored 5.7e-7
//   t = 20   (condition 715)               3.4e-6         3.7e-6
//   t = 100  (condition 1.7e4)             1.1e-4         2.6e-4
//   t = 1000 (9x8x10)                      1.4e-2         2.1e-1: CG took 45 iterations with
//            the operations and did not converge with the matrix
// In FP64, whose M is built without low parts, the two differ by 1e-15, 2e-14 and 1.6e-11 at
// t = 8, 20 and 100.  Elasticity has 4 (nu = 0.3), 13 (0.45), 61 (0.49); stretched boxes and
// jumps of the coefficient 5; there M is as close as the operations.
constexpr float kMapMaxCond = 128.f;
// K of Stokes is singular: the constant pressure is in every column of M, and the response to
// it in every pressure column, and what is left of them after M b cancelled is the rounding of
// large entries.  Error of the projected result over 16 residuals K x, stored against
// operations: FP32 1.6 times on the average of 5^3 to 24^3 (9.8 at 5^3); FP64 5 to 9 times from
// level 0 (5^3), 1.0 to 1.9 from level 1 (6^3 to 9^3), 1.00 from level 2 (12^3 to 24^3).
// (Mixed elasticity: 0.94 to 1.10 in FP32, 1.0 to 1.4 in FP64; elasticity and the Laplacian at
// most 1 in FP32, in FP64 2 to 2.8 from level 0, at 5e-16, and 0.8 to 1.3 below.)
constexpr int kMapStokesFrom = 2;
// The share of the free device memory that a matrix may take: it is a gain in time only, and
// the Krylov vectors, further handles and the caller's data need the rest.  (Where they do not
// fit, the handle that asks gives its own matrices back: giving_maps_back.)
constexpr int kMapMemoryShare = 32;
// and the share of the coarsest solve (FP64) in the construction
constexpr int64_t kMapCoarseWork = 4000000000ll;

// Batched solves, FP32: M B takes 16 m^2 FMAs, 8 us of the whole chip at 4,096.  The chain
// that it replaces leaves most of the chip to the other problems, so no larger map is used.
constexpr int kMapMaxBatch = 4096;

// the first level of at most `most` unknowns, its matrix allocated and zero
void plan(amg_handle* h, CoarseMap& M, int most) {
  const bool f32 = h->opt.precision == AMG_FP32;
  for (const auto& lv : h->L)
    if (!(lv->block_cond <= kMapMaxCond)) return;
  const bool stokes = h->kind == AMG_STOKES;
  if (stokes && f32) return;
  for (int l = stokes ? kMapStokesFrom : 0; l + 1 < (int)h->L.size(); ++l) {
    const int m = h->L[l]->dofs();
    if (m > most || (int64_t)h->coarse_m * h->coarse_m * m > kMapCoarseWork) continue;
    M.m = m;
    M.ld = (m + 31) / 32 * 32;
    const size_t count = (size_t)m * M.ld;
    size_t free_bytes = 0, total_bytes = 0;
    AMG_CUDA(cudaMemGetInfo(&free_bytes, &total_bytes));
    if (count * (f32 ? sizeof(float) : sizeof(double)) > free_bytes / kMapMemoryShare) return;
    try {
      if (f32) M.m32.alloc(count);
      else M.m64.alloc(count);
    } catch (const Error& e) {
      if (e.code != AMG_ERR_NOMEM) throw;
      return;   // no room: the cycle runs operation by operation
    }
    // the padding of the rows stays 0
    if (f32) AMG_CUDA(cudaMemsetAsync(M.m32.p, 0, M.m32.bytes(), h->stream));
    else AMG_CUDA(cudaMemsetAsync(M.m64.p, 0, M.m64.bytes(), h->stream));
    M.level = l;
    return;
  }
}

// the weights of the levels that M holds (4 a level)
std::vector<double> own_weights(const amg_handle* h, const CoarseMap& M) {
  return {h->weights.begin() + 4 * M.level, h->weights.end()};
}

// M of the handle's current weights
void fill(amg_handle* h, CoarseMap& M) {
  if (M.level < 0) return;
  M.from = -1;
  M.w.clear();
  try {
    if (M.m32.p) build<Pair, float>(h, M, M.m32.p);
    else build<double, double>(h, M, M.m64.p);
  } catch (const Error& e) {
    M = CoarseMap{};   // the cycle runs operation by operation
    drop_loops(h);
    if (e.code != AMG_ERR_NOMEM) throw;
    return;
  }
  M.w = M.seen = own_weights(h, M);
  M.from = M.level;
}

// In use where the weights are those that it was built with.  The setup's matrix is filled
// again for weights that a program sets before it uses the handle: it would be of no use.
void follow(amg_handle* h, CoarseMap& M) {
  if (M.level < 0) return;
  const std::vector<double> now = own_weights(h, M);
  if (now != M.seen) M.waited = 0;
  M.seen = now;
  M.from = now == M.w ? M.level : -1;
  if (M.from < 0 && M.fresh) {
    M.fresh = false;
    fill(h, M);
  }
}

}  // namespace

void map_plan(amg_handle* h) {
  const amg_options& o = h->opt;
  // a launch variant that the caller forces keeps its levels; the Vanka phases are not recorded
  if (o.cluster_from != -1 || o.cycle_kernel != 0 || o.gs_cluster != -1 || o.gs_flow != -1 ||
      o.gs_stream != -1 || o.gs_tma != -1 || o.smoother == AMG_SMOOTHER_VANKA)
    return;
  plan(h, h->map,
       o.smoother == AMG_SMOOTHER_SGS ? kMapMaxSgs
       : o.precision == AMG_FP32      ? kMapMax32
                                      : kMapMax64);
}

CoarseMap* map_batch(amg_handle* h) {
  // the batched cycle reads the FP32 values of every level, also with BF16 storage
  if (h->map.level < 0 || !h->map.m32.p || h->bf16_coarse || h->opt.batch_tile != -1)
    return nullptr;
  CoarseMap& M = h->map.m <= kMapMaxBatch ? h->map : h->bmap;
  if (M.level < 0) {
    plan(h, M, kMapMaxBatch);
    fill(h, M);
    if (M.level < 0) return nullptr;
  }
  map_refresh(h, M);
  return &M;
}

void map_build(amg_handle* h) {
  if (h->map.from < 0) fill(h, h->map);
}

void map_follow(amg_handle* h) {
  follow(h, h->map);
  follow(h, h->bmap);
}

bool map_release(amg_handle* h) {
  if (h->map.level < 0 && h->bmap.level < 0) return false;
  AMG_CUDA(cudaStreamSynchronize(h->stream));
  drop_loops(h);
  h->map = CoarseMap{};
  h->bmap = CoarseMap{};
  h->batch_map = nullptr;
  return true;
}

void map_refresh(amg_handle* h, CoarseMap& M) {
  if (M.level >= 0 && M.from < 0 && M.waited >= map_pays(M)) fill(h, M);
}

void map_apply_m(amg_handle* h, const CoarseMap& M, const float* b, float* x) {
  // 4 rows a CTA where 8 would leave SMs idle
  if (M.m < 8 * 152) k_map_m<4><<<div_up(M.m, 4), 256, 0, h->stream>>>(M.m, M.ld, M.m32, b, x);
  else k_map_m<8><<<div_up(M.m, 8), 256, 0, h->stream>>>(M.m, M.ld, M.m32, b, x);
  h->launches++;
}

template <typename T, typename IO>
void map_apply(amg_handle* h, const IO* b, IO* x) {
  const int m = h->map.m, ld = h->map.ld, n3 = 3 * h->L[h->map.from]->n;
  const T* M = matrix<T>(h->map);
  const int smem = ld * (int)sizeof(T);
  const bool stream = (int64_t)m * ld * sizeof(T) > (64ll << 20);
  const auto k = stream ? k_map_apply<T, IO, true> : k_map_apply<T, IO, false>;
  max_dynamic_smem((const void*)k, (sizeof(T) == 4 ? kMapMax32 : kMapMax64) * (int)sizeof(T));
  // a warp a row where the rows allow it, at most four CTAs an SM
  const int grid = std::max(1, std::min(div_up(m, kMapThreads / 32), 4 * 152));
  k<<<grid, kMapThreads, smem, h->stream>>>(m, ld, n3, M, b, x);
  h->launches++;
}

template void map_apply<float, float>(amg_handle*, const float*, float*);
template void map_apply<float, double>(amg_handle*, const double*, double*);
template void map_apply<double, double>(amg_handle*, const double*, double*);

}  // namespace amgp2
