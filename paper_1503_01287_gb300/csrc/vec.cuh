// Node vectors of the cycle are stored 4 values per node (x, y, z, 0) so that a
// node is one aligned 16-byte (FP32) or 32-byte (FP64) access: the gather of
// x_j in a block row is a single vector load.  The pressure part (saddle
// systems) follows the 4n velocity entries as plain scalars.
#pragma once

#include <cuda_runtime.h>

namespace amgp2 {

__device__ __forceinline__ void ld3(const float* p, int j, float& a, float& b, float& c) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p) + j);
  a = v.x; b = v.y; c = v.z;
}

__device__ __forceinline__ void ld3(const double* p, int j, double& a, double& b, double& c) {
  double w;
  asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
      : "=d"(a), "=d"(b), "=d"(c), "=d"(w)
      : "l"(p + 4 * (size_t)j));
}

// coherent variant for vectors written earlier in the same kernel by other threads
__device__ __forceinline__ void ld3c(const float* p, int j, float& a, float& b, float& c) {
  const float4 v = reinterpret_cast<const float4*>(p)[j];
  a = v.x; b = v.y; c = v.z;
}

__device__ __forceinline__ void ld3c(const double* p, int j, double& a, double& b, double& c) {
  double w;
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(a), "=d"(b), "=d"(c), "=d"(w)
               : "l"(p + 4 * (size_t)j)
               : "memory");
}

// through L2 only.  A kernel under programmatic dependent launch may share an SM with the
// kernels before it while these still write: what they write it reads like this, after
// griddepcontrol.wait (an earlier load may have left the old line in L1, and ld.global.nc
// is defined for data that nothing writes while the kernel runs).
__device__ __forceinline__ void ld3g(const float* p, int j, float& a, float& b, float& c) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(p) + j);
  a = v.x; b = v.y; c = v.z;
}

__device__ __forceinline__ void ld3g(const double* p, int j, double& a, double& b, double& c) {
  double w;
  asm volatile("ld.global.cg.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(a), "=d"(b), "=d"(c), "=d"(w)
               : "l"(p + 4 * (size_t)j)
               : "memory");
}

__device__ __forceinline__ void st3(float* p, int j, float a, float b, float c) {
  reinterpret_cast<float4*>(p)[j] = make_float4(a, b, c, 0.f);
}

__device__ __forceinline__ void st3(double* p, int j, double a, double b, double c) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p + 4 * (size_t)j), "d"(a),
               "d"(b), "d"(c), "d"(0.0)
               : "memory");
}

// FP32-pair arithmetic of the Krylov operator: (S, s) += a x with a = (a.x, a.y)
// = hi + lo and x = xh + xl.  The product a.x xh is exact as the rounded product
// p plus its error fma(a.x, xh, -p); the cross terms a.x xl + a.y xh join the
// error, a.y xl (about 2^-48 of the product) is dropped; p is added to S with
// TwoSum (Knuth) and the sum's error with the product's error to s.  The _rn
// intrinsics keep the compiler from contracting any of these into an FMA.
__device__ __forceinline__ void pair_fma(float& S, float& s, float2 a, float xh, float xl) {
  const float p = __fmul_rn(a.x, xh);
  float e = fmaf(a.x, xh, -p);
  e = fmaf(a.x, xl, e);
  e = fmaf(a.y, xh, e);
  const float t = __fadd_rn(S, p);
  const float bp = __fsub_rn(t, S);
  const float err = __fadd_rn(__fsub_rn(S, __fsub_rn(t, bp)), __fsub_rn(p, bp));
  S = t;
  s = __fadd_rn(s, __fadd_rn(err, e));
}

// the same for x that is a float (its low part 0)
__device__ __forceinline__ void pair_fma(float& S, float& s, float2 a, float x) {
  const float p = __fmul_rn(a.x, x);
  float e = fmaf(a.x, x, -p);
  e = fmaf(a.y, x, e);
  const float t = __fadd_rn(S, p);
  const float bp = __fsub_rn(t, S);
  const float err = __fadd_rn(__fsub_rn(S, __fsub_rn(t, bp)), __fsub_rn(p, bp));
  S = t;
  s = __fadd_rn(s, __fadd_rn(err, e));
}

// (S, s) += (T, t) for the reduction across the lanes of a row
__device__ __forceinline__ void pair_add(float& S, float& s, float T, float t) {
  const float u = __fadd_rn(S, T);
  const float bp = __fsub_rn(u, S);
  const float err = __fadd_rn(__fsub_rn(S, __fsub_rn(u, bp)), __fsub_rn(T, bp));
  S = u;
  s = __fadd_rn(s, __fadd_rn(err, t));
}

// FP32 pair of an FP64 value (hi = fl32(d), lo = fl32(d - hi)) and back
__device__ __forceinline__ float2 to_pair(double d) {
  const float hi = __double2float_rn(d);
  return make_float2(hi, __double2float_rn(d - (double)hi));
}
__device__ __forceinline__ double from_pair(float2 p) { return (double)p.x + (double)p.y; }
// a leading sum S and a small error sum s as one normalised pair (FastTwoSum)
__device__ __forceinline__ float2 norm_pair(float S, float s) {
  const float hi = __fadd_rn(S, s);
  return make_float2(hi, __fsub_rn(s, __fsub_rn(hi, S)));
}

// Sums of (s0, s1, s2) over the G lanes of a row, left one component a lane: lane 0 of the
// group gets component 0, lane G/4 component 1, lane G/2 component 2 (first_of).  The first
// exchange splits the components over the halves of the group and the second over the
// quarters, so that 2 + 1 + 1 + ... additions replace 3 a stage, in the same summation tree:
// FP64 additions issue at 1/67 of the FP32 rate on this GPU whatever lanes need them, and
// the row update after it (r, D^{-1} r, x) takes one component a lane instead of three on
// one lane.
template <int G>
__device__ __forceinline__ int component_of(int gl) {
  return (gl & (G / 2)) ? 2 : ((gl & (G / 4)) ? 1 : 0);
}
template <int G>
__device__ __forceinline__ bool holds_component(int gl) {
  return gl == 0 || gl == G / 4 || gl == G / 2;
}
template <int G, typename T>
__device__ __forceinline__ T row_sum3(T s0, T s1, T s2, int gl) {
  const bool up = gl & (G / 2), odd = gl & (G / 4);
  T a = up ? s2 : s0;
  a += __shfl_xor_sync(0xffffffffu, up ? s0 : s2, G / 2);
  const T b = s1 + __shfl_xor_sync(0xffffffffu, s1, G / 2);
  const T keep = !up && odd ? b : a;
  T v = keep + __shfl_xor_sync(0xffffffffu, !up && !odd ? b : a, G / 4);
#pragma unroll
  for (int o = G / 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// the same for pairs (.x + .y)
template <int G>
__device__ __forceinline__ float2 row_sum3_pair(float2 s0, float2 s1, float2 s2, int gl) {
  const bool up = gl & (G / 2), odd = gl & (G / 4);
  auto joined = [](float2 a, float2 b, int o) {   // a + the partner's b
    const float T = __shfl_xor_sync(0xffffffffu, b.x, o);
    const float t = __shfl_xor_sync(0xffffffffu, b.y, o);
    pair_add(a.x, a.y, T, t);
    return a;
  };
  const float2 a = joined(up ? s2 : s0, up ? s0 : s2, G / 2);
  const float2 b = joined(s1, s1, G / 2);
  float2 v = joined(!up && odd ? b : a, !up && !odd ? b : a, G / 4);
#pragma unroll
  for (int o = G / 8; o > 0; o >>= 1) v = joined(v, v, o);
  return v;
}
// the three components of a value held as row_sum3 leaves it, in every lane of the group
template <int G, typename T>
__device__ __forceinline__ void spread3(T v, int lane, T& v0, T& v1, T& v2) {
  const int base = lane & ~(G - 1);
  v0 = __shfl_sync(0xffffffffu, v, base);
  v1 = __shfl_sync(0xffffffffu, v, base + G / 4);
  v2 = __shfl_sync(0xffffffffu, v, base + G / 2);
}

// The end of a block row's update, whose lanes hold the partial sums (s0, s1, s2) of A x:
// FP64 one component a lane as above; FP32 all three on the group's first lane (the spread
// costs a shuffle more than the saved instructions give: 32^3 level-0 sweep 103.7 against
// 98.9 us) unless SPLIT asks for it.  N: components of a lane that `holds` operands.
template <typename T, int G, bool SPLIT = false>
struct RowEnd {
  static constexpr bool kSplit = sizeof(T) == 8 || SPLIT;
  static constexpr int N = kSplit ? 1 : 3;
  static __device__ __forceinline__ bool holds(int gl) {
    return kSplit ? holds_component<G>(gl) : gl == 0;
  }
  // the lane's components of node i of a padded vector, loaded by `one` or `node`
  template <typename L>
  static __device__ __forceinline__ void load(const T* v, int i, int gl, T (&o)[N]) {
    if constexpr (kSplit) o[0] = L::one(v + 4 * (int64_t)i + component_of<G>(gl));
    else L::node(v, i, o[0], o[1], o[2]);
  }
  // its row q of the padded 3x3 inverse of node i
  static __device__ __forceinline__ void load_dinv_row(const T* d, int i, int gl, int q,
                                                       T (&o)[3]) {
    ld3(d + 12 * (int64_t)i, kSplit ? component_of<G>(gl) : q, o[0], o[1], o[2]);
  }
  static __device__ __forceinline__ void sum(T s0, T s1, T s2, int gl, T (&o)[N]) {
    if constexpr (kSplit) {
      o[0] = row_sum3<G>(s0, s1, s2, gl);
    } else {
#pragma unroll
      for (int q = G / 2; q > 0; q >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, q);
        s1 += __shfl_xor_sync(0xffffffffu, s1, q);
        s2 += __shfl_xor_sync(0xffffffffu, s2, q);
      }
      o[0] = s0; o[1] = s1; o[2] = s2;
    }
  }
  // the three components of r in the lanes that hold any; called by all lanes of the warp
  static __device__ __forceinline__ void all(const T (&r)[N], T& r0, T& r1, T& r2) {
    if constexpr (kSplit) {
      spread3<G>(r[0], threadIdx.x & 31, r0, r1, r2);
    } else {
      r0 = r[0]; r1 = r[1]; r2 = r[2];
    }
  }
  // stores the lane's components of node i; PAD: and the padding as 0 (an update in place
  // finds it 0)
  template <bool PAD>
  static __device__ __forceinline__ void store(T* y, int i, int gl, const T (&v)[N]) {
    if constexpr (kSplit) {
      if (holds(gl)) y[4 * (int64_t)i + component_of<G>(gl)] = v[0];
      if (PAD && gl == G - 1) y[4 * (int64_t)i + 3] = T(0);
    } else {
      if (holds(gl)) st3(y, i, v[0], v[1], v[2]);
    }
  }
};

}  // namespace amgp2
