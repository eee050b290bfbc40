// Device helpers shared by the kernels: packed FP32 butterflies, complex
// multiply, in-register Walsh-Hadamard stages, the per-tile clause fold and the
// bit-sliced violated-clause counter.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "qaa_internal.cuh"

namespace qaa {

// ---- packed FP32 arithmetic (sm_100+ f32x2) ---------------------------------
__device__ __forceinline__ unsigned long long f2_bits(float2 a) {
  return (static_cast<unsigned long long>(__float_as_uint(a.y)) << 32) | __float_as_uint(a.x);
}
__device__ __forceinline__ float2 bits_f2(unsigned long long u) {
  return make_float2(__uint_as_float(static_cast<unsigned>(u)), __uint_as_float(static_cast<unsigned>(u >> 32)));
}
__device__ __forceinline__ void butterfly(float2& u, float2& w) {
  unsigned long long a = f2_bits(u), b = f2_bits(w), s, d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(a), "l"(b));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  u = bits_f2(s);
  w = bits_f2(d);
}

// a * z for complex a, z (FP32, fused multiply-add in both components).
__device__ __forceinline__ float2 cmul(float2 a, float2 z) {
  return make_float2(fmaf(a.x, z.x, -a.y * z.y), fmaf(a.x, z.y, a.y * z.x));
}

// Butterflies over register-index bits [B0, B1) of a 32-entry register tile:
// for every bit b and every r with bit b clear, (v[r], v[r+2^b]) <- (v[r]+v[r+2^b], v[r]-v[r+2^b]).
template <int B0, int B1>
__device__ __forceinline__ void reg_wht(float2 (&v)[32]) {
#pragma unroll
  for (int b = B0; b < B1; ++b) {
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      if (!(r & (1 << b))) butterfly(v[r], v[r | (1 << b)]);
    }
  }
}

// ---- one-qubit rotations in the gauge i^popcount ------------------------------
// exp(-i theta H_B) = prod_i e^(-ih) (cos h + i sin h sigma^x_i), h = theta / 2
// (Sec. 2.1).  With phi_x = i^popcount(x) psi_x (an exact swap and negation of
// components) every factor is real: cos h times (u, w) <- (u + b w, w - b u), b = tan
// h, on the pair of amplitudes whose index differs in the bit (u: bit clear), so it
// acts on (re, im) as a packed pair: one packed FMA per amplitude and qubit, against
// the two additions and a fifth of a complex multiply of a Walsh-Hadamard sandwich,
// and one rounding.  Angles with |tan h| > 1 are taken in two turns of h / 2.  The
// norm is taken out by the scale (1 + b^2)^(-n/2) per turn of the rounded b, as (1 + r)
// 2^-e: 2^-e in every step, the product of the (1 + r) with the norm fold (TurnScale;
// the streaming low pass puts it into its P row), so rounding b changes the angle by
// less than 1e-7 of itself and the norm not at all; the phase e^(-inh), the same for
// every amplitude, is left out until the last P row of a launch.  (As a factor of
// every P row it would round the entry of E = 0, else exactly 1, in every step, and
// with it the weight of the ground state: 2.6e-6 instead of 5e-7 after 400 steps.)
struct RotCoef {
  unsigned long long b, nb;
  float r, pow2;
  bool twice;
};
// row: the B row's entries 0 and 1.
__device__ __forceinline__ RotCoef rot_coef(const float2* row) {
  const float2 tb = row[0], sc = row[1];
  RotCoef c;
  c.b = f2_bits(make_float2(tb.y, tb.y));
  c.nb = f2_bits(make_float2(-tb.y, -tb.y));
  c.r = sc.x;
  c.pow2 = sc.y;
  c.twice = tb.x == 2.0f;
  return c;
}
__device__ __forceinline__ float2 fma2(unsigned long long k, float2 x, float2 y) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(k), "l"(f2_bits(x)), "l"(f2_bits(y)));
  return bits_f2(d);
}
__device__ __forceinline__ float2 mul2(unsigned long long k, float2 x) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(k), "l"(f2_bits(x)));
  return bits_f2(d);
}
__device__ __forceinline__ float2 add2(float2 x, float2 y) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(x)), "l"(f2_bits(y)));
  return bits_f2(d);
}
__device__ __forceinline__ float2 sub2(float2 x, float2 y) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(x)), "l"(f2_bits(y)));
  return bits_f2(d);
}
// Turns of the register-index bits [B0, B1) of an N-entry tile.  PAIRS: two bits at
// a time; on the four amplitudes of two bits
//   (1 + bJ)(1 + bJ') v = v + b (Jv + J'v + b JJ'v),
// so an amplitude rounds once per two qubits (the inner sum's errors come times
// b) for 2.5 packed operations instead of 2, and a dozen more registers.
template <int B0, int B1, int N, bool PAIRS>
__device__ __forceinline__ void turn_once(float2 (&v)[N], const RotCoef& c) {
  if constexpr (PAIRS) {
#pragma unroll
    for (int b = B0; b + 1 < B1; b += 2) {
      const int p = 1 << b, q = 2 << b;
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (!(r & (p | q))) {
          const float2 v0 = v[r], v1 = v[r | p], v2 = v[r | q], v3 = v[r | p | q];
          const float2 s = add2(v1, v2), e = sub2(v3, v0);
          v[r] = fma2(c.b, fma2(c.b, v3, s), v0);
          v[r | p] = fma2(c.b, fma2(c.nb, v2, e), v1);
          v[r | q] = fma2(c.b, fma2(c.nb, v1, e), v2);
          v[r | p | q] = fma2(c.nb, fma2(c.nb, v0, s), v3);
        }
      }
    }
  }
#pragma unroll
  for (int b = PAIRS ? B1 - (B1 - B0) % 2 : B0; b < B1; ++b) {
#pragma unroll
    for (int r = 0; r < N; ++r) {
      if (!(r & (1 << b))) {
        const float2 u = v[r], w = v[r | (1 << b)];
        v[r] = fma2(c.b, w, u);
        v[r | (1 << b)] = fma2(c.nb, u, w);
      }
    }
  }
}
// (The second turn as its own code: a loop around one would make every load of v
// finish before it starts.)
template <int B0, int B1, int N, bool PAIRS = true>
__device__ __forceinline__ void reg_turn(float2 (&v)[N], const RotCoef& c) {
  turn_once<B0, B1, N, PAIRS>(v, c);
  if (c.twice) turn_once<B0, B1, N, PAIRS>(v, c);
}

template <int N>
__device__ __forceinline__ void scale_by(float2 (&v)[N], float k) {
  const unsigned long long kk = f2_bits(make_float2(k, k));
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = fma2(kk, v[r], v[r]);
}
template <int N>
__device__ __forceinline__ void scale_pow2(float2 (&v)[N], float p) {
  if (p == 1.0f) return;
  const unsigned long long pp = f2_bits(make_float2(p, p));
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = mul2(pp, v[r]);
}

// A register tile with the increments since its last rounding kept apart: the
// value is v + d.  A step's turns and phases are small changes, so d is computed to
// 2^-24 of itself, where rounding the amplitude in every turn and phase would round it
// to 2^-24 of itself each time.  Where most of the weight sits in a few amplitudes
// their rounding is the error of the ground-state probability and of <H_P>.
//
// What a rounding leaves out, at most 2^-24 of the value, is kept in 8 bits of itself (a
// bfloat16 pair).
__device__ __forceinline__ unsigned pack_rest(float2 e) {
  unsigned p;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p) : "f"(e.y), "f"(e.x));
  return p;
}
__device__ __forceinline__ float2 unpack_rest(unsigned p) {
  return make_float2(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u));
}
template <int N>
__device__ __forceinline__ void scale_rest(unsigned (&rest)[N], float f) {
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const float2 e = unpack_rest(rest[r]);
    rest[r] = pack_rest(make_float2(f * e.x, f * e.y));
  }
}
template <int N>
struct Inc {
  float2 v[N], d[N];
  __device__ __forceinline__ float2 at(int r) const { return add2(v[r], d[r]); }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int r = 0; r < N; ++r) d[r] = make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void settle() {
#pragma unroll
    for (int r = 0; r < N; ++r) v[r] = at(r);
    zero();
  }
  // v <- the rounded v + d, d <- what the rounding left out (exact for |d| <= |v|).
  __device__ __forceinline__ void carry() {
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const float2 t = at(r);
      d[r] = sub2(d[r], sub2(t, v[r]));
      v[r] = t;
    }
  }
  // Before v alone leaves the thread: v <- the rounded v + d + left, left <- what the
  // rounding left out, d <- 0.
  __device__ __forceinline__ void leave(unsigned (&left)[N]) {
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const float2 s = add2(d[r], unpack_rest(left[r])), t = add2(v[r], s);
      left[r] = pack_rest(sub2(s, sub2(t, v[r])));
      v[r] = t;
    }
    zero();
  }
  // The value times 1 + k.
  __device__ __forceinline__ void grow(float k) {
    const unsigned long long kk = f2_bits(make_float2(k, k));
#pragma unroll
    for (int r = 0; r < N; ++r) d[r] = fma2(kk, at(r), d[r]);
  }
  // The value times a power of two.
  __device__ __forceinline__ void scale(float p) {
    scale_pow2<N>(v, p);
    scale_pow2<N>(d, p);
  }
  // Turns of the register-index bits [B0, B1), two at a time as in turn_once; `fresh`:
  // d is zero.
  template <int B0, int B1>
  __device__ __forceinline__ void once(const RotCoef& c, bool fresh) {
#pragma unroll
    for (int b = B0; b + 1 < B1; b += 2) {
      const int p = 1 << b, q = 2 << b;
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (!(r & (p | q))) {
          const bool first = fresh && b == B0;
          const float2 a0 = first ? v[r] : at(r), a1 = first ? v[r | p] : at(r | p);
          const float2 a2 = first ? v[r | q] : at(r | q), a3 = first ? v[r | p | q] : at(r | p | q);
          const float2 s = add2(a1, a2), e = sub2(a3, a0);
          const float2 i0 = fma2(c.b, a3, s), i1 = fma2(c.nb, a2, e), i2 = fma2(c.nb, a1, e), i3 = fma2(c.nb, a0, s);
          d[r] = first ? mul2(c.b, i0) : fma2(c.b, i0, d[r]);
          d[r | p] = first ? mul2(c.b, i1) : fma2(c.b, i1, d[r | p]);
          d[r | q] = first ? mul2(c.b, i2) : fma2(c.b, i2, d[r | q]);
          d[r | p | q] = first ? mul2(c.nb, i3) : fma2(c.nb, i3, d[r | p | q]);
        }
      }
    }
#pragma unroll
    for (int b = B1 - (B1 - B0) % 2; b < B1; ++b) {
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (!(r & (1 << b))) {
          const int w = r | (1 << b);
          const bool first = fresh && b == B0;
          const float2 su = first ? v[r] : at(r), sw = first ? v[w] : at(w);
          d[r] = first ? mul2(c.b, sw) : fma2(c.b, sw, d[r]);
          d[w] = first ? mul2(c.nb, su) : fma2(c.nb, su, d[w]);
        }
      }
    }
  }
  template <int B0, int B1>
  __device__ __forceinline__ void turn(const RotCoef& c, bool fresh = false) {
    once<B0, B1>(c, fresh);
    if (c.twice) {
      settle();
      reg_turn<B0, B1, N, false>(v, RotCoef{c.b, c.nb, c.r, c.pow2, false});
    }
  }
};

// v <- i^k v (exact).
__device__ __forceinline__ float2 times_i(float2 v, int k) {
  const float2 s = (k & 1) ? make_float2(-v.y, v.x) : v;
  return (k & 2) ? make_float2(-s.x, -s.y) : s;
}

// Runtime-bounded variant (bits [b0, b1) with b0, b1 in [0, 5]).
__device__ __forceinline__ void reg_wht_rt(float2 (&v)[32], int b0, int b1) {
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    if (b >= b0 && b < b1) {
#pragma unroll
      for (int r = 0; r < 32; ++r) {
        if (!(r & (1 << b))) butterfly(v[r], v[r | (1 << b)]);
      }
    }
  }
}

// ---- clause fold for one 1024-amplitude tile (bits 0..9 vary) --------------
// For tile index T = x >> 10 every clause either
//   * has a literal on bits >= 10 that is true for the whole tile -> dropped,
//   * has all its literals on bits >= 10 and all false -> +1 for every x (nconst),
//   * otherwise stays active, reduced to its literals on bits 0..9.
// Active clauses are written (warp-cooperatively, in clause order) to `act` as
// {reg_pat, lane_pat}: the 32-bit truth tables over the register-held window and
// over the lane-held window.  The list is padded with zero entries to a multiple
// of 16 (a zero entry counts for nobody).
template <bool REG_IS_LOW>
__device__ __forceinline__ void fold_tile(const ClauseLP* __restrict__ s_cl, int m, unsigned tile_hi,
                                          int lane, uint2* __restrict__ act, int& nconst, int& npad) {
  int base = 0, cconst = 0;
  for (int c0 = 0; c0 < m; c0 += 32) {
    const int c = c0 + lane;
    bool is_act = false, is_const = false;
    uint2 e = make_uint2(0u, 0u);
    if (c < m) {
      const ClauseLP k = s_cl[c];
      const bool hi_false = ((tile_hi ^ k.hi_viol) & k.hi_mask) == 0u;
      const bool has_lo = (k.pat0 & k.pat5) != 0xffffffffu;
      is_act = hi_false && has_lo;
      is_const = hi_false && !has_lo;
      e = REG_IS_LOW ? make_uint2(k.pat0, k.pat5) : make_uint2(k.pat5, k.pat0);
    }
    const unsigned ba = __ballot_sync(0xffffffffu, is_act);
    const unsigned bc = __ballot_sync(0xffffffffu, is_const);
    if (is_act) act[base + __popc(ba & ((1u << lane) - 1u))] = e;
    base += __popc(ba);
    cconst += __popc(bc);
  }
  const int padded = (base + 15) & ~15;
  if (lane < padded - base) act[base + lane] = make_uint2(0u, 0u);
  __syncwarp();
  nconst = cconst;
  npad = padded;
}

// ---- bit-sliced counting ----------------------------------------------------
// Carry-save adder: (h, l) <- carry and sum of l + b + c (all bit-parallel).
__device__ __forceinline__ void csa(unsigned& h, unsigned& l, unsigned b, unsigned c) {
  const unsigned a = l;
  l = a ^ b ^ c;
  h = (a & b) | (a & c) | (b & c);
}

// Sum of `count` (a multiple of 16) 32-bit words get(0), get(1), ... bit by bit:
// pl[b] holds bit b of each of the 32 sums.  Harley-Seal carry-save tree over
// 16 words at a time, then a ripple add of the weight-16 carries.  Sums up to
// 1023 are exact.
template <class Get>
__device__ __forceinline__ void count_words(int count, Get&& get, unsigned (&pl)[kPlanes]) {
  unsigned ones = 0, twos = 0, fours = 0, eights = 0;
  unsigned hi[kPlanes - 4];
#pragma unroll
  for (int k = 0; k < kPlanes - 4; ++k) hi[k] = 0;
  for (int i = 0; i < count; i += 16) {
    unsigned d[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) d[j] = get(i + j);
    unsigned twosA, twosB, foursA, foursB, eightsA, eightsB, sixteens;
    csa(twosA, ones, d[0], d[1]);
    csa(twosB, ones, d[2], d[3]);
    csa(foursA, twos, twosA, twosB);
    csa(twosA, ones, d[4], d[5]);
    csa(twosB, ones, d[6], d[7]);
    csa(foursB, twos, twosA, twosB);
    csa(eightsA, fours, foursA, foursB);
    csa(twosA, ones, d[8], d[9]);
    csa(twosB, ones, d[10], d[11]);
    csa(foursA, twos, twosA, twosB);
    csa(twosA, ones, d[12], d[13]);
    csa(twosB, ones, d[14], d[15]);
    csa(foursB, twos, twosA, twosB);
    csa(eightsB, fours, foursA, foursB);
    csa(sixteens, eights, eightsA, eightsB);
    unsigned carry = sixteens;
#pragma unroll
    for (int k = 0; k < kPlanes - 4; ++k) {
      const unsigned t = hi[k] & carry;
      hi[k] ^= carry;
      carry = t;
    }
  }
  pl[0] = ones;
  pl[1] = twos;
  pl[2] = fours;
  pl[3] = eights;
#pragma unroll
  for (int k = 0; k < kPlanes - 4; ++k) pl[4 + k] = hi[k];
}

// For every register index r (0..31) count the active entries whose lane_pat
// has `lanebit` set and whose reg_pat has bit r set.  Result: pl[b] holds bit b
// of each of the 32 counts (bit r of pl[b] belongs to register r).
__device__ __forceinline__ void count_active(const uint2* __restrict__ act, int npad, unsigned lanebit,
                                             unsigned (&pl)[kPlanes]) {
  count_words(
      npad,
      [&](int i) {
        const uint2 e = act[i];
        return (e.y & lanebit) ? e.x : 0u;
      },
      pl);
}

// Stored per-tile counts (layout Y: registers hold bits 0..4).  E(x) never
// changes during a run, so the merged low passes (and the observables) read
// these instead of folding and counting the clauses again.  Layout, in 32-bit
// words:
//   [0] P, the number of bit planes stored: the bits of the largest count of
//       active (non-constant) violated clauses above its tile's smallest, so that
//       the planes above P are zero everywhere and not stored (P = 6 instead
//       of kPlanes = 10 for the 30-qubit benchmark instance: 0.75 instead of
//       1.25 bytes per amplitude for the low pass to read);
//   [1] the word offset of the planes, a multiple of 32 (128-byte rows);
//   [32 + t] the constant part of tile t (clauses violated on the whole tile, and
//       the smallest active count);
//   [planes + (t P + b) 32 + l] bit plane b < P of lane l's 32 counts in tile t.
constexpr int kCountHeaderWords = 32;

__device__ __forceinline__ void load_counts(const unsigned* __restrict__ counts, long long tile, int lane,
                                            unsigned (&pl)[kPlanes], int& nconst) {
  const int P = static_cast<int>(__ldg(counts));
  const unsigned* c = counts + __ldg(counts + 1) + static_cast<size_t>(tile) * (32 * P) + lane;
#pragma unroll
  for (int b = 0; b < kPlanes; ++b) pl[b] = b < P ? __ldg(c + 32 * b) : 0u;
  nconst = static_cast<int>(__ldg(counts + kCountHeaderWords + tile));
}

// Counts of registers R and R+16 packed as (count_R) | (count_{R+16} << 16).
template <int R>
__device__ __forceinline__ unsigned extract_pair(const unsigned (&pl)[kPlanes]) {
  unsigned w = 0;
#pragma unroll
  for (int b = 0; b < kPlanes; ++b) {
    const unsigned s = (R >= b) ? (pl[b] >> (R - b)) : (pl[b] << (b - R));
    w |= s & (0x00010001u << b);
  }
  return w;
}

// v + v z for complex v, z: four FMAs, as a multiplication takes.
__device__ __forceinline__ float2 cadd(float2 v, float2 z) {
  return make_float2(fmaf(-v.y, z.y, fmaf(v.x, z.x, v.x)), fmaf(v.x, z.y, fmaf(v.y, z.x, v.y)));
}

template <int R, bool MINUS1>
struct ApplyPhaseUnroll {
  __device__ __forceinline__ static void run(float2 (&v)[32], const unsigned (&pl)[kPlanes], int nconst,
                                             const float2* __restrict__ tab) {
    const unsigned w = extract_pair<R>(pl);
    const float2 z0 = tab[nconst + static_cast<int>(w & 0xffffu)], z1 = tab[nconst + static_cast<int>(w >> 16)];
    v[R] = MINUS1 ? cadd(v[R], z0) : cmul(v[R], z0);
    v[R + 16] = MINUS1 ? cadd(v[R + 16], z1) : cmul(v[R + 16], z1);
    ApplyPhaseUnroll<R + 1, MINUS1>::run(v, pl, nconst, tab);
  }
};
template <bool MINUS1>
struct ApplyPhaseUnroll<16, MINUS1> {
  __device__ __forceinline__ static void run(float2 (&)[32], const unsigned (&)[kPlanes], int, const float2*) {}
};

// v[r] <- exp(-i theta E(x_r)) v[r] where E = nconst + the bit-sliced count in
// pl and tab[E] holds the FP32-rounded FP64 phase (the P row of the step), minus 1
// with MINUS1 (kRowsTurn).
template <bool MINUS1 = false>
__device__ __forceinline__ void apply_p_phase(float2 (&v)[32], const unsigned (&pl)[kPlanes], int nconst,
                                              const float2* __restrict__ tab) {
  ApplyPhaseUnroll<0, MINUS1>::run(v, pl, nconst, tab);
}

template <int R>
struct StoreCountUnroll {
  __device__ __forceinline__ static void run(int (&e)[32], const unsigned (&pl)[kPlanes], int nconst) {
    const unsigned w = extract_pair<R>(pl);
    e[R] = nconst + static_cast<int>(w & 0xffffu);
    e[R + 16] = nconst + static_cast<int>(w >> 16);
    StoreCountUnroll<R + 1>::run(e, pl, nconst);
  }
};
template <>
struct StoreCountUnroll<16> {
  __device__ __forceinline__ static void run(int (&)[32], const unsigned (&)[kPlanes], int) {}
};

// E(x_r) for the 32 register-held amplitudes.
__device__ __forceinline__ void energies(int (&e)[32], const uint2* __restrict__ act, int npad, int nconst,
                                         unsigned lanebit) {
  unsigned pl[kPlanes];
  count_active(act, npad, lanebit, pl);
  StoreCountUnroll<0>::run(e, pl, nconst);
}


// Overlapped launches (launch_overlapped): let the next kernel's blocks in as soon as
// there is room, and wait until the kernel before this one is complete.
__device__ __forceinline__ void let_next_in() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The device's global nanosecond timer (the PTX special register %globaltimer).
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---- norm fold (see NormFold) ------------------------------------------------
// Sum of |v|^2 over a lane's 32 register-held amplitudes: packed FP32 FMAs in
// two interleaved chains of 16, then one FP32 add per component.
__device__ __forceinline__ float tile_norm(const float2 (&v)[32]) {
  unsigned long long a = 0ull, b = 0ull;
#pragma unroll
  for (int r = 0; r < 32; r += 2) {
    const unsigned long long x = f2_bits(v[r]), y = f2_bits(v[r + 1]);
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(a) : "l"(x));
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(b) : "l"(y));
  }
  const float2 fa = bits_f2(a), fb = bits_f2(b);
  return (fa.x + fb.x) + (fa.y + fb.y);
}

// Double-float sums for the norm fold: hi + lo with |lo| <= ulp(hi) / 2.
// df_add: Knuth's TwoSum of the leading parts, the trailing parts added to its
// error, then renormalised (about 44 significant bits for sums of positive
// terms); df_add1 adds one FP32 value.  No FMA contraction can apply (no
// products), and nvcc does not reassociate FP32 additions.
struct DFloat {
  float hi, lo;
};
__device__ __forceinline__ DFloat df_add(DFloat a, DFloat b) {
  const float s = a.hi + b.hi;
  const float bb = s - a.hi;
  const float e = (a.hi - (s - bb)) + (b.hi - bb);
  const float t = e + (a.lo + b.lo);
  const float h = s + t;
  return DFloat{h, t - (h - s)};
}
__device__ __forceinline__ DFloat df_add1(DFloat a, float b) {
  const float s = a.hi + b;
  const float bb = s - a.hi;
  const float t = ((a.hi - (s - bb)) + (b - bb)) + a.lo;
  const float h = s + t;
  return DFloat{h, t - (h - s)};
}
__device__ __forceinline__ DFloat df_shfl_xor(DFloat a, int o) {
  return DFloat{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

// d = c - 1 for c = sqrt(r / (s 2^k)), 2^k the power of two that brings s
// within a factor sqrt(2) of r (0 when either is not a positive finite normal
// number).  The scaling by 2^k is exact, r - s 2^k is exact in its leading
// part (Sterbenz: the two are within a factor 2), and with
// eps = (r - s 2^k) / (s 2^k), d = eps/2 - eps^2/8 to within eps^3 / 16 (1e-18
// at the eps ~ 1e-6 of a fold; sqrtf beyond |eps| = 0.01).  Kept as c - 1, d
// carries c to about 1e-13 (c itself rounded to FP32 would be off by up to
// 6e-8, a systematic norm error of 1.2e-7); a value x is scaled by
// fold_apply(x, d) = x + x d, one rounding.
__device__ __forceinline__ float fold_scale(DFloat r, DFloat s) {
  const int er = (__float_as_int(r.hi) >> 23) & 0xff, es = (__float_as_int(s.hi) >> 23) & 0xff;
  if (!(r.hi > 0.f) || !(s.hi > 0.f) || er == 0 || es == 0 || er == 0xff || es == 0xff) return 0.0f;
  const int k = er - es;
  if (k > 126 || k < -126) return 0.0f;
  const float p = __int_as_float((127 + k) << 23);
  float sh = s.hi * p, sl = s.lo * p;
  if (sh > r.hi * 1.41421356f) {
    sh *= 0.5f;
    sl *= 0.5f;
  } else if (sh < r.hi * 0.70710678f) {
    sh *= 2.0f;
    sl *= 2.0f;
  }
  const float eps = ((r.hi - sh) + (r.lo - sl)) / sh;
  return fabsf(eps) < 1e-2f ? eps * (0.5f - 0.125f * eps) : sqrtf(1.0f + eps) - 1.0f;
}
__device__ __forceinline__ float fold_apply(float x, float d) { return fmaf(x, d, x); }
__device__ __forceinline__ float2 fold_apply(float2 x, float d) { return make_float2(fmaf(x.x, d, x.x), fmaf(x.y, d, x.y)); }

// The correction of a low pass as d = c - 1 (0 when there is nothing to
// correct), valid in lane 0.  One whole warp calls it: lane i adds partials i, i + 32,
// ... of both slots (the loads of the two slots in flight together; L2 loads,
// since within a persistent kernel the slots were written by other CTAs since
// this SM last read them), then a shuffle tree in the same fixed order in
// every CTA.
__device__ __forceinline__ float fold_factor(const NormFold& f, int lane) {
  if (!f.ref || !f.prev) return 0.0f;
  const int cr = __float_as_int(__ldcg(&f.ref[0].x)), cp = __float_as_int(__ldcg(&f.prev[0].x));
  const int cnt = cr > cp ? cr : cp;
  DFloat r{0.f, 0.f}, s{0.f, 0.f};
  for (int i = lane; i < cnt; i += 32) {
    if (i < cr) {
      const float2 a = __ldcg(f.ref + 1 + i);
      r = df_add(r, DFloat{a.x, a.y});
    }
    if (i < cp) {
      const float2 b = __ldcg(f.prev + 1 + i);
      s = df_add(s, DFloat{b.x, b.y});
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    r = df_add(r, df_shfl_xor(r, o));
    s = df_add(s, df_shfl_xor(s, o));
  }
  return lane == 0 ? fold_scale(r, s) : 0.0f;
}

// Block-wide correction d = c - 1: warp 0 computes it, every thread gets it.
// Contains a __syncthreads: every thread of the block must call it.
__device__ __forceinline__ float fold_factor_block(const NormFold& f) {
  __shared__ float s_c;
  if (threadIdx.x < 32) {
    const float c = fold_factor(f, threadIdx.x);
    if (threadIdx.x == 0) s_c = c;
  }
  __syncthreads();
  return s_c;
}

// The scale the turns of the steps so far still owe, as R = prod (1 + r) - 1, and
// the norm fold.  Both are applied together, every fold_period steps and after the
// last of a launch (so that the result carries no drift of the steps since the
// last fold: up to 8e-7 with most of the weight in one amplitude): multiplying by
// 1 + r in every step (r ~ -1e-7 towards the end of a sweep) would round an amplitude
// that hardly changes the same way every time.
struct TurnScale {
  float R = 0.f;
  __device__ __forceinline__ void step(float r) { R = fmaf(R, r, R + r); }
  // The factor minus 1 that brings the measured sum s to ref, R included; R restarts.
  __device__ __forceinline__ float fold(DFloat ref, DFloat s) {
    const float q = fmaf(R, R, 2.0f * R), p = s.hi * q;  // s (1 + R)^2
    const float d = fold_scale(ref, df_add(s, DFloat{p, fmaf(s.hi, q, -p) + s.lo * q}));
    const float k = fmaf(R, d, R + d);
    R = 0.f;
    return k;
  }
};
// Write the block's partial: the double-float sum of one pair per thread in a
// fixed order; block 0 also writes the partial count.  Contains
// __syncthreads: every thread of the block must call it.
__device__ __forceinline__ void fold_store(const NormFold& f, DFloat v) {
  __shared__ DFloat s_w[32];
  if (!f.out) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) s_w[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    DFloat t = s_w[0];
    for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) t = df_add(t, s_w[w]);
    f.out[1 + blockIdx.x] = make_float2(t.hi, t.lo);
    if (f.out2) f.out2[1 + blockIdx.x] = make_float2(t.hi, t.lo);
    if (blockIdx.x == 0) {
      const float cnt = __int_as_float(static_cast<int>(gridDim.x));
      f.out[0] = make_float2(cnt, 0.f);
      if (f.out2) f.out2[0] = make_float2(cnt, 0.f);
    }
  }
}

}  // namespace qaa
