// Lanczos on H(s) = (1 - s) H_B + s H_P (Eq. (1)) for the lowest levels: the
// gap the adiabatic evolution of Sec. 2.1 must respect.
//
// H is real symmetric, so the Lanczos vectors are real; they are kept in FP64
// (8 bytes per amplitude, like a complex64 state), so loss of orthogonality
// and the end of the Krylov space show at the 1e-12 level.  No host
// synchronisation: the recurrence scalars live in device memory.  The vectors are
// stored unnormalised, u_j with v_j = u_j / beta_j, so one iteration is
//   y = H u_j, partials of <u_j, y>:  H_B u = (n/2) u - 1/2 sum_i u(x ^ 2^(i-1)) and
//     H_P u = E u from the exported diagonal
//   u_(j+1) = y / beta_j - (alpha_j / beta_j) u_j - (beta_j / beta_(j-1)) u_(j-1),
//     partials of |u_(j+1)|^2; every block adds up the previous partials itself
// in place of separate reductions and a normalising pass (five launches and 15 n
// more bytes per amplitude).
//
// What bounds it: GB300 does about two FP64 operations per clock and SM, and the n
// additions of the neighbour sum were two thirds of them (62 us at n = 20).  From
// kTileMinBits on the sum is taken in 64-bit integers instead, tile by tile: the
// tile's values as fixed-point numbers with 59 bits below the tile's largest
// exponent (rounding 2^-60 of the tile's largest value; an FP64 sum rounds each
// amplitude to 2^-53 of itself), added exactly, converted back once.  |error of H u| /
// |u| against extended precision, FP64 sums / this: ground state at s = 0.2 1.0e-15 /
// 0.9e-15, at s = 0.5 4.8e-16 / 3.0e-16, a Krylov residual at s = 0.2 1.0e-15 / 1.1e-15, random
// 8.2e-16 / 8.1e-16 (n = 18..20; amplitudes over up to 2^80).  A tile of
// 2^TB values in shared memory serves the TB bits it spans: a low pass for bits
// [0, TB) and strided passes of up to TB - 3 bits (64-byte runs) above, whose sums go
// through y.
#include <cstdint>

#include "qaa_internal.cuh"

namespace qaa {

namespace {

constexpr int kLzThreads = 256;

__device__ __forceinline__ double lz_block_sum(double v, double* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) s_red[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += s_red[w];
  return t;
}

// splitmix64: a counter-based generator (Steele, Lea, Flood 2014), used for a
// reproducible random start vector.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__global__ void __launch_bounds__(kLzThreads) lz_start_kernel(double* __restrict__ v, unsigned long long N, int random,
                                                              unsigned long long seed) {
  for (unsigned long long x = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; x < N;
       x += static_cast<unsigned long long>(gridDim.x) * blockDim.x) {
    double r = 1.0;
    if (random) {
      const unsigned long long h = splitmix64(seed ^ splitmix64(x));
      r = static_cast<double>(h >> 11) * 0x1.0p-53 * 2.0 - 1.0;
    }
    v[x] = r;
  }
}

// y = H u by direct gathers, for vectors too small to keep every SM busy with tiles.
__global__ void __launch_bounds__(kLzThreads)
    lz_apply_kernel(double* __restrict__ y, const double* __restrict__ u, const uint16_t* __restrict__ E, int n,
                    unsigned long long N, double a_hb, double a_hp, double* __restrict__ partials) {
  __shared__ double s_red[kLzThreads / 32];
  double acc = 0.0;
  for (unsigned long long x = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; x < N;
       x += static_cast<unsigned long long>(gridDim.x) * blockDim.x) {
    const double c = u[x];
    double sum = 0.0;
    for (int i = 0; i < n; ++i) sum += u[x ^ (1ull << i)];
    const double h = a_hb * (0.5 * n * c - 0.5 * sum) + a_hp * static_cast<double>(E[x]) * c;
    y[x] = h;
    acc += c * h;
  }
  const double t = lz_block_sum(acc, s_red);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// A value as a fixed-point integer, 59 bits below the exponent field `top` of the
// tile's largest value (e <= top, top > 0), rounded to nearest.
__device__ __forceinline__ long long to_fixed(double c, int top) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(c));
  const int e = static_cast<int>(bits >> 52) & 0x7ff;
  if (e == 0) return 0;  // zero, or a subnormal beside a normal maximum
  const unsigned long long m = ((bits & 0xfffffffffffffull) | 0x10000000000000ull) << 6;
  const int sh = top - e;
  const unsigned long long f = sh == 0 ? m : (sh > 60 ? 0ull : (m + (1ull << (sh - 1))) >> sh);
  return static_cast<long long>(bits) < 0 ? -static_cast<long long>(f) : static_cast<long long>(f);
}

// The fixed-point sum s back as a double, rounded to nearest, by integer
// operations (the conversion instruction runs at the FP64 rate and took as long as
// several additions).  NaN beside infinities; 0 where it would be subnormal.
__device__ __forceinline__ double from_fixed(long long s, int top) {
  if (top == 0x7ff) return __longlong_as_double(0x7ff8000000000000ll);
  const unsigned long long mag = static_cast<unsigned long long>(s < 0 ? -s : s);  // below 2^63
  const int lz = __clzll(static_cast<long long>(mag | 1ull));
  const unsigned long long r = ((mag << (lz - 1)) + 0x200ull) >> 10;  // 2^52 .. 2^53
  const int e = top - lz + 5;  // exponent field: 1023 + 63 - lz of mag, unit 2^(top - 1081)
  if (mag == 0 || e <= 0) return 0.0;
  const unsigned long long b = (static_cast<unsigned long long>(e - 1) << 52) + r;
  return __longlong_as_double(static_cast<long long>(b | (static_cast<unsigned long long>(s) & 0x8000000000000000ull)));
}

// One pass over tiles of 2^TB values, 8 per thread: thread = the low TB - 3 bits of
// the tile index, register = the top 3.  LOW: the tile is contiguous, the sum covers
// its TB bits, y = H u with the strided bits' sums taken from y (`more`) and the
// partials of <u, y>.  Otherwise the tile spans q bits of the index from bit a on,
// in runs of 2^(TB-q), and their sum goes to y (added to it with `more`).  The
// fixed-point values stay in shared memory only: with 8 doubles and what is loaded
// beside them a thread has 64 registers, 1024 threads per SM hide the loads (16 per
// thread and the values in registers too ran at 20 % occupancy, 1.4 times slower).
template <int TB, bool LOW>
__global__ void __launch_bounds__(1 << (TB - 3), (1024 >> (TB - 3)) > 0 ? (1024 >> (TB - 3)) : 1)
    lz_tile_kernel(double* __restrict__ y, const double* __restrict__ u, const uint16_t* __restrict__ E, int n, int m,
                   int a, int q, int more, long long ntiles, double a_hb, double a_hp, double* __restrict__ partials) {
  constexpr int NT = 1 << (TB - 3), N = 8;
  extern __shared__ __align__(16) unsigned char smem[];
  long long* s_f = reinterpret_cast<long long*>(smem);
  double* s_diag = reinterpret_cast<double*>(smem) + (1 << TB);  // LOW: the diagonal by E
  __shared__ int s_top[2];
  __shared__ double s_red[NT / 32];
  const int tid = threadIdx.x;
  const int C = TB - q;  // strided: run bits
  if (LOW) {
    for (int e = tid; e <= m; e += NT) s_diag[e] = a_hb * 0.5 * n + a_hp * static_cast<double>(e);
  }
  if (tid < 2) s_top[tid] = 0;
  __syncthreads();
  double acc = 0.0;
  int flip = 0;
  for (long long T = blockIdx.x; T < ntiles; T += gridDim.x, flip ^= 1) {
    const unsigned long long uT = static_cast<unsigned long long>(T);
    unsigned long long base, step;
    if (LOW) {
      base = (uT << TB) + tid;
      step = NT;
    } else {
      const int lo_bits = a - C;
      const int i0 = tid >> C;  // low bits of the strided index
      base = ((uT & ((1ull << lo_bits) - 1ull)) << C) | (tid & ((1 << C) - 1)) | (static_cast<unsigned long long>(i0) << a) |
             ((uT >> lo_bits) << (a + q));
      step = 1ull << (a + q - 3);  // the top 3 strided bits
    }
    double c[N], t[N];
    unsigned ev[N];
#pragma unroll
    for (int k = 0; k < N; ++k) c[k] = u[base + k * step];
#pragma unroll
    for (int k = 0; k < N; ++k) t[k] = more ? y[base + k * step] : 0.0;
    if (LOW) {
#pragma unroll
      for (int k = 0; k < N; ++k) ev[k] = E[base + k * step];
    }
    int top = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int e = (__double2hiint(c[k]) >> 20) & 0x7ff;
      top = e > top ? e : top;
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if ((tid & 31) == 0) atomicMax(&s_top[flip], top);
    __syncthreads();  // and every thread is done with the last tile's s_f
    top = s_top[flip];
#pragma unroll
    for (int k = 0; k < N; ++k) s_f[tid + k * NT] = to_fixed(c[k], top);
    __syncthreads();
    if (tid == 0) s_top[flip] = 0;  // next used two tiles on
#pragma unroll
    for (int k = 0; k < N; ++k) {
      long long s = 0;
#pragma unroll
      for (int b = 0; b < 3; ++b) s += s_f[tid + (k ^ (1 << b)) * NT];
#pragma unroll
      for (int b = 0; b < TB - 3; ++b)
        if (LOW || b >= C) s += s_f[(tid ^ (1 << b)) + k * NT];
      const double sum = from_fixed(s, top);
      const double v = more ? sum + t[k] : sum;
      if (LOW) {
        const double h = fma(-0.5 * a_hb, v, s_diag[ev[k]] * c[k]);
        y[base + k * step] = h;
        acc = fma(c[k], h, acc);
      } else {
        y[base + k * step] = v;
      }
    }
  }
  if (LOW) {
    const double t = lz_block_sum(acc, s_red);
    if (tid == 0) partials[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kLzThreads)
    lz_dot_kernel(const double* __restrict__ a, const double* __restrict__ b, unsigned long long N,
                  double* __restrict__ partials) {
  __shared__ double s_red[kLzThreads / 32];
  double acc = 0.0;
  for (unsigned long long x = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; x < N;
       x += static_cast<unsigned long long>(gridDim.x) * blockDim.x)
    acc += a[x] * b[x];
  const double t = lz_block_sum(acc, s_red);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// The sum of np partials in a fixed order, by one warp, in every lane.
__device__ __forceinline__ double lz_total(const double* __restrict__ partials, int np, int lane) {
  double t = 0.0;
  for (int i = lane; i < np; i += 32) t += partials[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// up <- u_(j+1) (the recurrence above), partials of its squared norm.  dots: the npa
// partials of <u_j, y>; norms: the npb partials of |u_j|^2; inverses: 1 / |u_j| by
// parity of j (0 after a breakdown).  beta_j is 0 for j = 0 (the norm of the start
// vector is no coefficient).  Block 0 writes alpha_j, beta_j and its inverse.  The
// scalars are one warp's work in every block, of two blocks per SM: in every thread of
// eight blocks per SM their FP64 operations took 30 us at n = 20.
constexpr int kUpThreads = 512;
__global__ void __launch_bounds__(kUpThreads, 2)
    lz_update_kernel(const double* __restrict__ y, const double* __restrict__ u, double* __restrict__ up,
                     const double* __restrict__ dots, int npa, const double* __restrict__ norms, int npb, int j,
                     double* __restrict__ alpha, double* __restrict__ beta, double* __restrict__ inverses,
                     unsigned long long N, double* __restrict__ partials) {
  __shared__ double s_red[kUpThreads / 32];
  __shared__ double s_c[3];
  if (threadIdx.x < 32) {
    const double s = lz_total(norms, npb, threadIdx.x), d = lz_total(dots, npa, threadIdx.x);
    if (threadIdx.x == 0) {
      double inv = s > 1e-300 ? rsqrt(s) : 0.0;  // |u| below 1e-150 counts as none
      const double norm = s * inv;
      const double al = d * inv * inv;
      s_c[0] = inv;
      s_c[1] = -al * inv;
      s_c[2] = j > 0 ? -norm * inverses[(j + 1) & 1] : 0.0;  // beta_j / |u_(j-1)|
      if (blockIdx.x == 0) {
        alpha[j] = al;
        beta[j] = j > 0 ? norm : 0.0;
        inverses[j & 1] = inv;
      }
    }
  }
  __syncthreads();
  const double c1 = s_c[0], c2 = s_c[1], c3 = s_c[2];
  double acc = 0.0;
  const unsigned long long stride = static_cast<unsigned long long>(gridDim.x) * kUpThreads;
  unsigned long long x = blockIdx.x * static_cast<unsigned long long>(kUpThreads) + threadIdx.x;
  // N is a power of two: from 4 strides on, four elements in flight per thread
  for (; x + 3 * stride < N; x += 4 * stride) {
    double p[4], v[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      p[k] = up[x + k * stride];
      v[k] = u[x + k * stride];
      w[k] = y[x + k * stride];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double r = fma(c3, p[k], fma(c2, v[k], c1 * w[k]));
      up[x + k * stride] = r;
      acc = fma(r, r, acc);
    }
  }
  for (; x < N; x += stride) {
    const double r = fma(c3, up[x], fma(c2, u[x], c1 * y[x]));
    up[x] = r;
    acc = fma(r, r, acc);
  }
  const double t = lz_block_sum(acc, s_red);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// beta_iters from the last partials.
__global__ void lz_last_kernel(const double* __restrict__ norms, int np, double* __restrict__ out) {
  const double t = lz_total(norms, np, threadIdx.x);
  if (threadIdx.x == 0) *out = sqrt(t > 0.0 ? t : 0.0);
}

// Tiles from n = 18 on (2^11 values at n = 18, 2^12 above, so that every SM has
// one): at n = 17 an iteration took 24.3 us with tiles of 2^10 and 23.3 with the gathers.
// us per iteration, before (five launches, gathers) and now: n = 10 about 20 / 16, n = 18
// 41 / 26, n = 20 92 / 46, n = 24 1308 / 477, n = 28 22700 / 7240, n = 30 98400 / 33000.
// What is left is bound by the FP64 operations again (8 to 10 per amplitude).
constexpr int kTileMinBits = 18;

template <int TB>
cudaError_t launch_tiles(const LaunchCtx& lc, const LanczosArgs& a, double* y, const double* u, int maxp, int* np) {
  const double a_hb = 1.0 - a.s;
  const long long ntiles = 1ll << (a.n - TB);
  const size_t s_strided = sizeof(long long) << TB;
  const size_t s_low = s_strided + sizeof(double) * (QAA_MAX_CLAUSES_DEV + 1);
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(lz_tile_kernel<TB, true>), s_low);
  if (e == cudaSuccess) e = allow_smem(reinterpret_cast<const void*>(lz_tile_kernel<TB, false>), s_strided);
  if (e != cudaSuccess) return e;
  long long grid = (1024 >> (TB - 3)) * 1ll * lc.num_sms;
  if (grid > maxp) grid = maxp;
  if (grid > ntiles) grid = ntiles;
  const int rest = a.n - TB, ng = (rest + TB - 4) / (TB - 3);
  int bit = TB;
  for (int g = 0; g < ng; ++g) {
    const int q = rest / ng + (g < rest % ng ? 1 : 0);  // 5 to 9: a thread's registers take three
    lz_tile_kernel<TB, false><<<static_cast<unsigned>(grid), 1 << (TB - 3), s_strided, lc.stream>>>(
        y, u, nullptr, a.n, a.m, bit, q, g > 0, ntiles, a_hb, a.s, nullptr);
    bit += q;
  }
  lz_tile_kernel<TB, true><<<static_cast<unsigned>(grid), 1 << (TB - 3), s_low, lc.stream>>>(
      y, u, a.E, a.n, a.m, 0, 0, ng > 0, ntiles, a_hb, a.s, a.partials);
  *np = static_cast<int>(grid);
  return cudaGetLastError();
}

}  // namespace

// Partials: <u, y>, |u|^2 of even and of odd iterations, and two inverse norms.
static int lanczos_blocks(int num_sms) { return 6 * num_sms; }
int lanczos_partials(int num_sms) { return 3 * lanczos_blocks(num_sms) + 2; }

cudaError_t launch_lanczos(const LaunchCtx& lc, const LanczosArgs& a, int* done_iters) {
  const unsigned long long N = 1ull << a.n;
  const int P = lanczos_blocks(lc.num_sms);
  double* norms[2] = {a.partials + P, a.partials + 2 * P};
  double* inverses = a.partials + 3 * P;
  auto blocks = [&](int threads, int per_sm) {
    const long long need = static_cast<long long>((N + threads - 1) / threads), most = 1ll * per_sm * lc.num_sms;
    return static_cast<unsigned>(need < most ? need : most);
  };
  const unsigned grid = blocks(kLzThreads, 4), ugrid = blocks(kUpThreads, 2);
  lz_start_kernel<<<grid, kLzThreads, 0, lc.stream>>>(a.v, N, a.random_start, a.seed);
  lz_dot_kernel<<<grid, kLzThreads, 0, lc.stream>>>(a.v, a.v, N, norms[0]);
  int npn = static_cast<int>(grid);
  cudaError_t e = cudaMemsetAsync(a.vp, 0, N * sizeof(double), lc.stream);
  if (e != cudaSuccess) return e;
  double *u = a.v, *up = a.vp;
  for (int j = 0; j < a.iters; ++j) {
    int npd = static_cast<int>(grid);
    if (a.n >= kTileMinBits) {
      e = a.n == 18 ? launch_tiles<11>(lc, a, a.w, u, P, &npd) : launch_tiles<12>(lc, a, a.w, u, P, &npd);
      if (e != cudaSuccess) return e;
    } else {
      lz_apply_kernel<<<grid, kLzThreads, 0, lc.stream>>>(a.w, u, a.E, a.n, N, 1.0 - a.s, a.s, a.partials);
    }
    lz_update_kernel<<<ugrid, kUpThreads, 0, lc.stream>>>(a.w, u, up, a.partials, npd, norms[j & 1], npn, j, a.alpha, a.beta,
                                                          inverses, N, norms[(j + 1) & 1]);
    npn = static_cast<int>(ugrid);
    // the previous vector's buffer has received the next one
    double* t = up;
    up = u;
    u = t;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  lz_last_kernel<<<1, 32, 0, lc.stream>>>(norms[a.iters & 1], npn, a.beta + a.iters);
  *done_iters = a.iters;
  return cudaGetLastError();
}

}  // namespace qaa
