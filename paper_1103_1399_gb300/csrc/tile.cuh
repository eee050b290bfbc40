// Pieces of the evolvers that keep the state on chip (onchip.cu, team.cu):
// register windows of a CTA's tile, their shared-memory transposes, phase-row
// lookups and cp.async copies.
#pragma once

#include "device_common.cuh"

namespace qaa {

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Barrier over the NT threads that run an instance (the others of a batch
// CTA have left).
template <int NT>
__device__ __forceinline__ void team_sync() {
  if constexpr (NT <= 32)
    __syncwarp();
  else
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

// P rows of the kRowsTurn form hold z = e^(-i theta E) - 1: of a phase near 1 the
// FP32 pair (cos, sin) is off by up to 3e-8 in magnitude, the pair (cos - 1, sin) by
// next to nothing, and those errors are what the weights of the levels drift by.
// d + x z for complex x, z.
__device__ __forceinline__ float2 cmac(float2 d, float2 x, float2 z) {
  return make_float2(fmaf(-x.y, z.y, fmaf(x.x, z.x, d.x)), fmaf(x.x, z.y, fmaf(x.y, z.x, d.y)));
}
__device__ __forceinline__ float2 row_entry(const float2* prow, const unsigned* e, int r) {
  const unsigned off = (r & 1) ? e[r / 2] >> 16 : e[r / 2] & 0xffffu;
  return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(prow) + off);
}

// v <- (1 + prow[E]) v; E of register pairs packed as two byte offsets.
template <int N>
__device__ __forceinline__ void apply_rows(float2 (&v)[N], const unsigned (&e)[(N + 1) / 2], const float2* prow) {
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = add2(v[r], cmac(make_float2(0.f, 0.f), v[r], row_entry(prow, e, r)));
}
template <int N>
__device__ __forceinline__ void apply_rows(Inc<N>& x, const unsigned (&e)[(N + 1) / 2], const float2* prow) {
#pragma unroll
  for (int r = 0; r < N; ++r) x.d[r] = cmac(x.d[r], x.at(r), row_entry(prow, e, r));
}

// Turns and phases on a plain tile (R = 5: no registers for the increments) and on
// an Inc tile, by the same names.
template <int N, bool INC>
struct Tile;
template <int N>
struct Tile<N, false> {
  float2 v[N];
  __device__ __forceinline__ float2 at(int r) const { return v[r]; }
  template <int B0, int B1>
  __device__ __forceinline__ void turn(const RotCoef& c, bool = false) {
    reg_turn<B0, B1>(v, c);
  }
  __device__ __forceinline__ void phase(const unsigned (&e)[(N + 1) / 2], const float2* prow) { apply_rows<N>(v, e, prow); }
  __device__ __forceinline__ void carry() {}
  __device__ __forceinline__ void settle() {}
  __device__ __forceinline__ void zero() {}
  __device__ __forceinline__ void grow(float k) { scale_by<N>(v, k); }
  __device__ __forceinline__ void scale(float p) { scale_pow2<N>(v, p); }
};
template <int N>
struct Tile<N, true> : Inc<N> {
  __device__ __forceinline__ void phase(const unsigned (&e)[(N + 1) / 2], const float2* prow) { apply_rows<N>(*this, e, prow); }
};

// |x|^2 over a thread's N amplitudes (an Inc's as rounded) as a double-float: every
// square as its FP32 product and that product's exact error, the products summed by
// TwoSum.  A plain FP32 sum would be biased by up to 4e-7 on a uniform state (every
// thread adds the same numbers and rounds the same way), and with it the norm a run
// is held to.
template <int N, class X>
__device__ __forceinline__ DFloat norm_of(const X& x) {
  float s = 0.f, e = 0.f;
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const float2 v = x.at(r);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float a = k ? v.y : v.x;
      const float p = a * a, t = s + p, bb = t - s;
      e += ((s - (t - bb)) + (p - bb)) + fmaf(a, a, -p);
      s = t;
    }
  }
  return DFloat{s, e};
}
__device__ __forceinline__ DFloat warp_sum(DFloat t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t = df_add(t, df_shfl_xor(t, o));
  return t;
}

template <int T, int R>
struct CtaGeom {
  static_assert(2 * R < T && T <= 3 * R, "three windows");
  static constexpr int NT = 1 << (T - R);
  static constexpr int N = 1 << R;
  // Padded slot of index l, linear in disjoint bits.  Conflict-free for 8-byte
  // accesses along consecutive l and along strides of 2^R (R = 3: a two-way
  // conflict on a few lanes of the MID window).
  __host__ __device__ static constexpr int slot(int l) { return R >= 4 ? l + (l >> R) : l + 2 * (l >> 4) + (l >> 6); }
  static constexpr int SLOTS = slot((1 << T) - 1) + 1;
  static constexpr bool kTwoBuffers = T <= 13;  // one barrier per transpose instead of two
};

enum Window { kTop, kBot, kMid };

template <int T, int R, int W>
__device__ __forceinline__ int win_base(int tid) {
  if (W == kTop) return tid;
  if (W == kBot) return tid << R;
  return (tid & ((1 << R) - 1)) | ((tid >> R) << (2 * R));
}
template <int T, int R, int W>
__device__ __forceinline__ constexpr int win_step() {
  return W == kTop ? 1 << (T - R) : (W == kBot ? 1 : 1 << R);
}

template <int T, int R, int W>
__device__ __forceinline__ void put(const float2 (&v)[1 << R], float2* buf, int tid) {
  using G = CtaGeom<T, R>;
  float2* p = buf + G::slot(win_base<T, R, W>(tid));
#pragma unroll
  for (int r = 0; r < (1 << R); ++r) p[G::slot(r * win_step<T, R, W>())] = v[r];
}
template <int T, int R, int W>
__device__ __forceinline__ void get(float2 (&v)[1 << R], const float2* buf, int tid) {
  using G = CtaGeom<T, R>;
  const float2* p = buf + G::slot(win_base<T, R, W>(tid));
#pragma unroll
  for (int r = 0; r < (1 << R); ++r) v[r] = p[G::slot(r * win_step<T, R, W>())];
}
// A tile's transposes: the increments, where there are any, travel with the values
// (behind them in the buffer).  Rounding them into the values at every transpose
// instead (three or four roundings per step) made the error of <H_P> as large as that of
// turns rounded one by one: n = 16, 400 steps, 3.9e-7 rms over 8 instances; so 6e-8.
template <int T, int R, bool INC>
__host__ __device__ constexpr size_t tile_bytes() {
  return (INC ? 16u : 8u) * static_cast<size_t>(CtaGeom<T, R>::SLOTS);
}
template <int T, int R, int W, bool CARRY = true, bool INC>
__device__ __forceinline__ void put_tile(Tile<1 << R, INC>& x, float2* buf, int tid) {
  if (!CARRY) x.settle();
  put<T, R, W>(x.v, buf, tid);
  if constexpr (INC && CARRY) put<T, R, W>(x.d, buf + CtaGeom<T, R>::SLOTS, tid);
}
template <int T, int R, int W, bool CARRY = true, bool INC>
__device__ __forceinline__ void get_tile(Tile<1 << R, INC>& x, const float2* buf, int tid) {
  get<T, R, W>(x.v, buf, tid);
  if (!CARRY) x.zero();
  if constexpr (INC && CARRY) get<T, R, W>(x.d, buf + CtaGeom<T, R>::SLOTS, tid);
}

}  // namespace qaa
