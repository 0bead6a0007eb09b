// Plain doubles behind the interface of Wide (wide.cuh), for the complex double instantiation of
// the column kernel: a number is its 8 bytes, a sum is one double (its exponent and shifts do
// nothing), and every operation is the FP64 one.  At one limb the FP64 pipe is the cheaper one
// (two multiply-adds of 64 clocks a product pair against four times as many integer
// instructions); what the kernel's schedule saves is the chain between steps.
#pragma once

#include "wide.cuh"

namespace mgs {

template <>
struct Wide<1> {
  static constexpr int L = 1, W = 2, K = 2, S = 2, BIAS = 0, SUMBITS = 0;
  struct num {
    double v;
    static constexpr int e = 0;
  };
  struct sum {
    u32 a[2];
  };
  __device__ static __forceinline__ double get(const u32* w) { return __hiloint2double((int)w[1], (int)w[0]); }
  __device__ static __forceinline__ void put(double v, u32* w) {
    w[0] = (u32)__double2loint(v);
    w[1] = (u32)__double2hiint(v);
  }
  __device__ static __forceinline__ double signed_by(double v, u32 neg) {  // -v for neg = ~0
    return __hiloint2double(__double2hiint(v) ^ (int)(neg & 0x80000000u), __double2loint(v));
  }
  __device__ static __forceinline__ int biased_exp(const u32*) { return 0; }
  __device__ static __forceinline__ num unpack(const u32* w) { return num{get(w)}; }
  __device__ static __forceinline__ void pack(const num& v, u32, u32* w) { put(v.v, w); }
  __device__ static __forceinline__ void clear(sum& a) { a.a[0] = a.a[1] = 0u; }
  __device__ static __forceinline__ void add_sum(sum& a, const u32* b) { put(get(a.a) + get(b), a.a); }
  __device__ static __forceinline__ void mac(sum& a, int, const num& x, const num& y, u32 neg) {
    put(__fma_rn(signed_by(x.v, neg), y.v, get(a.a)), a.a);
  }
  __device__ static __forceinline__ void mac2(sum& a, int, const num& x1, const num& y1, u32 neg1, const num& x2,
                                              const num& y2, u32 neg2) {
    const double t = __fma_rn(signed_by(x1.v, neg1), y1.v, get(a.a));
    put(__fma_rn(signed_by(x2.v, neg2), y2.v, t), a.a);
  }
  __device__ static __forceinline__ void add(sum& a, int, const num& x, u32 neg) {
    put(get(a.a) + signed_by(x.v, neg), a.a);
  }
  __device__ static __forceinline__ void shift_sum(sum&, int) {}
  __device__ static __forceinline__ num normalize(const sum& a, int, u32&) { return num{get(a.a)}; }
  __device__ static __forceinline__ void store(const sum& a, int, u32* w) {
    w[0] = a.a[0];
    w[1] = a.a[1];
  }
  __device__ static __forceinline__ void update(const num& y, const num& x1, const num& y1, u32 neg1, const num& x2,
                                                const num& y2, u32 neg2, u32* w) {
    const double t = __fma_rn(signed_by(x1.v, neg1), y1.v, y.v);
    put(__fma_rn(signed_by(x2.v, neg2), y2.v, t), w);
  }
  __device__ static __forceinline__ num quotient(const num& n, const num& d, u32&) { return num{__ddiv_rn(n.v, d.v)}; }
  __device__ static __forceinline__ void div_words(const u32* x, const u32* d, u32* w) { put(__ddiv_rn(get(x), get(d)), w); }
  __device__ static __forceinline__ void mul_words(const u32* x, const u32* y, u32* w) { put(get(x) * get(y), w); }
  __device__ static __forceinline__ void sqrt_words(const u32* x, u32* w) { put(__dsqrt_rn(get(x)), w); }
  __device__ static __forceinline__ void of_limbs(const double* v, u32* w) { put(v[0], w); }
  __device__ static __forceinline__ void to_limbs(const u32* w, double* v) { v[0] = get(w); }
  __device__ static __forceinline__ bool positive(const u32* w) {
    const double v = get(w);
    return v > 0.0 && (w[1] & 0x7ff00000u) != 0x7ff00000u;
  }
};

}  // namespace mgs
