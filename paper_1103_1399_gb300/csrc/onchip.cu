// Small-instance evolver (n <= 14): the whole complex64 state stays in one CTA for
// every step of a run, so HBM is touched once on entry and once on exit.
//
// Same Strang step as the streaming path (Eq. (1) frozen at s_k; H_P the
// violated-clause count, Sec. 4.3), with half phases of adjacent steps merged;
// exp(-i theta H_B) is applied as its n one-qubit factors in the gauge
// i^popcount (RotCoef): one packed FMA per amplitude and qubit.
//
// * n <= 8: one warp, the state in its registers (x = lane + 32 r): lane bits by
//   shuffles, no barrier and no shared-memory transpose in a step.
// * 9 <= n <= 14: one CTA of 2^(n-R) threads with 2^R amplitudes each.  A
//   thread's registers hold a window of R index bits: TOP [n-R, n), BOT [0, R) or
//   MID [R, 2R).  A step turns one window, moves the state through shared memory
//   to the next and ends with P: TOP BOT MID P, the next step MID BOT TOP P, so
//   two transposes per step.  E(x) of both P layouts stays in registers (16 bits
//   per amplitude, times 8: the byte offset in the phase row).
// Bound by shared memory (two transposes and the P row lookups) and, below
// n = 12, by the latency of a step's two barriers.  The earlier form (W B W in
// columns of 32 amplitudes, 24 butterfly levels, four shared-memory rounds and
// P rows from global memory) had 2^(n-5) threads busy.  Measured, us per step of
// a 400-step run, before and after: n = 6 1.76 / 0.33, n = 9 1.83 / 0.79, n = 11
// 3.00 / 1.36 (1.19 when the increments were rounded away at every window; from n =
// 12 on a single run takes a cluster, team.cu; batches keep one CTA per instance).
// Phase rows come through a ring of cp.async copies issued kCtaRing - 1 steps ahead.
#include "tile.cuh"

namespace qaa {

namespace {

constexpr int kBatchThreads = 512;

struct RunArgs {
  float2* psi;
  const ClauseMV* cl;
  const float2* ptab;
  const float2* btab;
  int n, m, nsteps;
  bool first_p, init;
  float init_val;
};

// Phase rows of step j (the P row that ends it, its rotation) into ring slot j.
// One commit group per call, empty beyond the last step.
template <int NT, int RING>
__device__ __forceinline__ void fetch_rows(const RunArgs& A, float2* s_p, float2* s_ab, int j, int tid) {
  if (j < A.nsteps) {
    const int mp1 = A.m + 1;
    float2* dst = s_p + (j % RING) * mp1;
    const float2* src = A.ptab + static_cast<size_t>(j + 1) * mp1;
    for (int i = tid; i < mp1; i += NT) cp_async8(dst + i, src + i);
    if (tid < 2) cp_async8(s_ab + 2 * (j % RING) + tid, A.btab + static_cast<size_t>(j) * (A.n + 1) + tid);
  }
  cp_async_commit();
}

// ------------------------------------------------------------ one warp ------
// A lane's entries of the phase rows depend on its energies only, so they are
// loaded straight into registers, kAhead steps before their use.
template <int N>
__device__ void warp_run(const RunArgs& A, unsigned char* smem) {
  constexpr int kAhead = N >= 8 ? 2 : 4;
  const int lane = threadIdx.x & 31;
  const int n = A.n, mp1 = A.m + 1;
  ClauseMV* s_cl = reinterpret_cast<ClauseMV*>(smem);
  for (int c = lane; c < A.m; c += 32) s_cl[c] = A.cl[c];
  const bool mine = lane < (1 << n);  // n < 5: the other lanes hold zeros
  Inc<N> x;
  auto& v = x.v;
#pragma unroll
  for (int r = 0; r < N; ++r)
    v[r] = !mine ? make_float2(0.f, 0.f) : (A.init ? make_float2(A.init_val, 0.f) : A.psi[lane + 32 * r]);
  __syncwarp();
  int ev[N];
#pragma unroll
  for (int r = 0; r < N; ++r) ev[r] = 0;
#pragma unroll 4
  for (int c = 0; c < A.m; ++c) {
    const unsigned mk = static_cast<unsigned>(s_cl[c].mask), vl = static_cast<unsigned>(s_cl[c].viol);
#pragma unroll
    for (int r = 0; r < N; ++r) ev[r] += (static_cast<unsigned>(lane + 32 * r) & mk) == vl;
  }
  float2 z[kAhead][N], row[kAhead][2];
  auto load = [&](int k, int j) {
    if (j >= A.nsteps) return;
    const float2* p = A.ptab + static_cast<size_t>(j + 1) * mp1;
    const float2* b = A.btab + static_cast<size_t>(j) * (n + 1);
#pragma unroll
    for (int r = 0; r < N; ++r) z[k][r] = __ldg(p + ev[r]);
    row[k][0] = __ldg(b);
    row[k][1] = __ldg(b + 1);
  };
#pragma unroll
  for (int k = 0; k < kAhead; ++k) load(k, k);
  auto warp_norm = [&]() { return warp_sum(norm_of<N>(x)); };
  x.zero();
  const DFloat nref = warp_norm();
  const int pc = __popc(lane);
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = times_i(v[r], pc + __popc(r));
  if (A.first_p) {
#pragma unroll
    for (int r = 0; r < N; ++r) x.d[r] = cmac(x.d[r], v[r], A.ptab[ev[r]]);
  }
  TurnScale ts;
  for (int j0 = 0; j0 < A.nsteps; j0 += kAhead) {
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int j = j0 + k;
      if (j >= A.nsteps) break;
      const RotCoef c = rot_coef(row[k]);
      if constexpr (N >= 2) x.template turn<0, (N >= 8 ? 3 : (N >= 4 ? 2 : 1))>(c);
      auto lanes = [&]() {
#pragma unroll
        for (int b = 0; b < 5; ++b) {
          if (b < n) {
            const unsigned long long kk = ((lane >> b) & 1) ? c.nb : c.b;
#pragma unroll
            for (int r = 0; r < N; ++r) {
              const float2 s = x.at(r);
              x.d[r] = fma2(kk, make_float2(__shfl_xor_sync(0xffffffffu, s.x, 1 << b), __shfl_xor_sync(0xffffffffu, s.y, 1 << b)),
                            x.d[r]);
            }
          }
        }
      };
      lanes();
      if (c.twice) {
        x.settle();
        lanes();
      }
#pragma unroll
      for (int r = 0; r < N; ++r) x.d[r] = cmac(x.d[r], x.at(r), z[k][r]);
      load(k, j + kAhead);
      x.carry();
      x.scale(c.pow2);
      // every fold_period(n)-th step and the last
      ts.step(c.r);
      if ((j + 1) % fold_period(1) == 0 || j + 1 == A.nsteps)
        x.grow(__shfl_sync(0xffffffffu, ts.fold(nref, warp_norm()), 0));
    }
  }
  if (mine) {
#pragma unroll
    for (int r = 0; r < N; ++r) A.psi[lane + 32 * r] = times_i(x.at(r), -(pc + __popc(r)));
  }
}

size_t warp_smem(int m) { return 16u * static_cast<size_t>(m); }

// ------------------------------------------------------------- one CTA ------
constexpr int kCtaRing = 4;

// Violated-clause counts of a thread's amplitudes (base xb, window bits
// [p, p+R)), packed as byte offsets: every clause becomes (fixed mask, fixed
// value, truth table over the window) in shared memory once, then each thread
// adds the tables of the clauses whose fixed literals are all false, bit-sliced.
template <int R, int NT>
__device__ void window_energies(const ClauseMV* __restrict__ cl, int m, uint4* s_ent, int p, unsigned xb, int tid,
                                unsigned (&e)[1 << (R - 1)]) {
  const unsigned win = ((1u << R) - 1u) << p;
  const int padded = (m + 15) & ~15;
  team_sync<NT>();
  for (int c = tid; c < padded; c += NT) {
    uint4 t = make_uint4(0u, 0u, 0u, 0u);
    if (c < m) {
      const unsigned mk = static_cast<unsigned>(cl[c].mask), vl = static_cast<unsigned>(cl[c].viol);
      unsigned pat = 0xffffffffu;
      const unsigned half[5] = {0xaaaaaaaau, 0xccccccccu, 0xf0f0f0f0u, 0xff00ff00u, 0xffff0000u};
#pragma unroll
      for (int b = 0; b < R; ++b)
        if ((mk >> (p + b)) & 1u) pat &= ((vl >> (p + b)) & 1u) ? half[b] : ~half[b];
      t = make_uint4(mk & ~win, vl & ~win, pat, 0u);
    }
    s_ent[c] = t;
  }
  team_sync<NT>();
  unsigned pl[kPlanes];
  count_words(
      padded,
      [&](int i) {
        const uint4 t = s_ent[i];
        return ((xb ^ t.y) & t.x) == 0u ? t.z : 0u;
      },
      pl);
#pragma unroll
  for (int r = 0; r < (1 << R); r += 2) {
    unsigned w = 0;
#pragma unroll
    for (int b = 0; b < kPlanes; ++b) w |= ((pl[b] >> r) & 1u) << (b + 3) | ((pl[b] >> (r + 1)) & 1u) << (b + 19);
    e[r / 2] = w;
  }
}

template <int T, int R>
__host__ __device__ inline size_t cta_smem(int m) {
  using G = CtaGeom<T, R>;
  const size_t buf = (tile_bytes<T, R, (R < 5)>() * (G::kTwoBuffers ? 2 : 1) + 15u) & ~static_cast<size_t>(15);
  const size_t ent = 16u * static_cast<size_t>((m + 15) & ~15);  // the buffers hold the clause tables first
  return (buf > ent ? buf : ent) + 8u * kCtaRing * static_cast<size_t>(m + 3);
}

// The sum over the threads of a double-float (fixed order); every thread gets it.
template <int NT>
__device__ DFloat cta_norm(DFloat v, DFloat* s_w, int tid) {
  v = warp_sum(v);
  team_sync<NT>();
  if ((tid & 31) == 0) s_w[tid >> 5] = v;
  team_sync<NT>();
  DFloat t{0.f, 0.f};
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) t = df_add(t, s_w[w]);
  return t;
}

template <int T, int R>
__device__ void cta_run(const RunArgs& A, unsigned char* smem) {
  using G = CtaGeom<T, R>;
  constexpr int NT = G::NT, N = G::N;
  __shared__ DFloat s_w[kBatchThreads / 32];
  const int tid = threadIdx.x;
  const int mp1 = A.m + 1;
  float2* s_buf = reinterpret_cast<float2*>(smem);
  float2* s_ab = reinterpret_cast<float2*>(smem + cta_smem<T, R>(A.m) - 8u * kCtaRing * static_cast<size_t>(A.m + 3));
  float2* s_p = s_ab + 2 * kCtaRing;
  for (int j = 0; j < kCtaRing - 1; ++j) fetch_rows<NT, kCtaRing>(A, s_p, s_ab, j, tid);
  const int xt = win_base<T, R, kTop>(tid), xm = win_base<T, R, kMid>(tid);
  Tile<N, (R < 5)> x;
  auto& v = x.v;
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = A.init ? make_float2(A.init_val, 0.f) : A.psi[xt + (r << (T - R))];
  unsigned et[N / 2], em[N / 2];
  window_energies<R, NT>(A.cl, A.m, reinterpret_cast<uint4*>(smem), T - R, xt, tid, et);
  window_energies<R, NT>(A.cl, A.m, reinterpret_cast<uint4*>(smem), R, xm, tid, em);
  x.zero();
  const DFloat nref = cta_norm<NT>(norm_of<N>(x), s_w, tid);  // also ends the use of s_buf as the clause tables
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = times_i(v[r], __popc(xt) + __popc(r));
  if (A.first_p) x.phase(et, A.ptab);
  float2* b0 = s_buf;
  float2* b1 = s_buf + (G::kTwoBuffers ? tile_bytes<T, R, (R < 5)>() / 8 : 0);
  TurnScale ts;
  cp_async_wait<1>();
  team_sync<NT>();  // the first rotation is in
  for (int j = 0; j < A.nsteps; ++j) {
    if (!G::kTwoBuffers && j > 0) team_sync<NT>();  // the buffer is free
    const RotCoef c = rot_coef(s_ab + 2 * (j % kCtaRing));
    const float2* prow = s_p + (j % kCtaRing) * mp1;
    const bool down = !(j & 1);
    if (down) {
      x.template turn<0, R>(c);
      put_tile<T, R, kTop>(x, b0, tid);
    } else {
      x.template turn<0, T - 2 * R>(c);
      put_tile<T, R, kMid>(x, b0, tid);
    }
    cp_async_wait<1>();  // rows up to step j + 1, visible to all beyond the barrier
    team_sync<NT>();
    fetch_rows<NT, kCtaRing>(A, s_p, s_ab, j + kCtaRing - 1, tid);  // into the slot of step j - 1, which all have left
    get_tile<T, R, kBot>(x, b0, tid);
    if (!G::kTwoBuffers) team_sync<NT>();
    x.template turn<0, R>(c);
    put_tile<T, R, kBot>(x, b1, tid);
    team_sync<NT>();
    if (down) {
      get_tile<T, R, kMid>(x, b1, tid);
      x.template turn<0, T - 2 * R>(c);
      x.phase(em, prow);
    } else {
      get_tile<T, R, kTop>(x, b1, tid);
      x.template turn<0, R>(c);
      x.phase(et, prow);
    }
    x.carry();
    if (c.pow2 != 1.0f) x.scale(c.pow2);
    ts.step(c.r);
    if ((j + 1) % fold_period(T) == 0 || j + 1 == A.nsteps)
      x.grow(ts.fold(nref, cta_norm<NT>(norm_of<N>(x), s_w, tid)));
  }
  if (A.nsteps & 1) {
#pragma unroll
    for (int r = 0; r < N; ++r) A.psi[xm + (r << R)] = times_i(x.at(r), -(__popc(xm) + __popc(r)));
  } else {
#pragma unroll
    for (int r = 0; r < N; ++r) A.psi[xt + (r << (T - R))] = times_i(x.at(r), -(__popc(xt) + __popc(r)));
  }
}

// Register bits per thread of the CTA form: 32 amplitudes from n = 13, 16 at n =
// 10..12, 8 at n = 9 (at least two warps).
#define QAA_ONCHIP_SIZES(X) X(9, 3) X(10, 4) X(11, 4) X(12, 4) X(13, 5) X(14, 5)

template <int T, int R>
__global__ void __launch_bounds__(CtaGeom<T, R>::NT) cta_kernel(const RunArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  cta_run<T, R>(A, smem);
}

__device__ void warp_dispatch(const RunArgs& A, unsigned char* smem) {
  if (A.n <= 5)
    warp_run<1>(A, smem);
  else if (A.n == 6)
    warp_run<2>(A, smem);
  else if (A.n == 7)
    warp_run<4>(A, smem);
  else
    warp_run<8>(A, smem);
}

__global__ void __launch_bounds__(32) warp_kernel(const RunArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  warp_dispatch(A, smem);
}

// A batch of independent instances of uneven size and length: one CTA each;
// the threads an instance does not use leave at once.
__global__ void __launch_bounds__(kBatchThreads) onchip_batch_kernel(const OnchipJob* __restrict__ jobs, int njobs) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (static_cast<int>(blockIdx.x) >= njobs) return;
  const OnchipJob jb = jobs[blockIdx.x];
  if (jb.stamp && threadIdx.x == 0) *jb.stamp = global_ns();
  const RunArgs A{jb.psi, jb.cl, jb.ptab, jb.btab, jb.n, jb.m, jb.nsteps, jb.first_p != 0, jb.init != 0, jb.init_val};
  switch (jb.n) {
#define QAA_CASE(T, R)                                                        \
  case T:                                                                     \
    if (threadIdx.x < static_cast<unsigned>(CtaGeom<T, R>::NT)) cta_run<T, R>(A, smem); \
    break;
    QAA_ONCHIP_SIZES(QAA_CASE)
#undef QAA_CASE
    default:
      if (threadIdx.x < 32) warp_dispatch(A, smem);
  }
}

template <int T, int R>
cudaError_t launch_cta(const LaunchCtx& lc, const RunArgs& A) {
  const cudaError_t e =
      allow_smem(reinterpret_cast<const void*>(cta_kernel<T, R>), cta_smem<T, R>(QAA_MAX_CLAUSES_DEV));
  if (e != cudaSuccess) return e;
  cta_kernel<T, R><<<1, CtaGeom<T, R>::NT, cta_smem<T, R>(A.m), lc.stream>>>(A);
  return cudaGetLastError();
}

}  // namespace

size_t onchip_smem_bytes(int n, int m) {
  switch (n) {
#define QAA_CASE(T, R) \
  case T:              \
    return cta_smem<T, R>(m);
    QAA_ONCHIP_SIZES(QAA_CASE)
#undef QAA_CASE
    default:
      return warp_smem(m);
  }
}

// The largest dynamic shared memory any on-chip instance needs.
static size_t onchip_smem_max() {
  size_t b = 0;
  for (int n = 1; n <= kOnchipMaxBits; ++n) {
    const size_t s = onchip_smem_bytes(n, QAA_MAX_CLAUSES_DEV);
    if (s > b) b = s;
  }
  return b;
}

cudaError_t launch_onchip_batch(const LaunchCtx& lc, const OnchipJob* jobs_dev, int njobs, size_t smem_bytes) {
  if (njobs <= 0) return cudaSuccess;
  cudaError_t err = allow_smem(reinterpret_cast<const void*>(onchip_batch_kernel), onchip_smem_max());
  if (err != cudaSuccess) return err;
  onchip_batch_kernel<<<njobs, kBatchThreads, smem_bytes, lc.stream>>>(jobs_dev, njobs);
  return cudaGetLastError();
}

cudaError_t launch_onchip(const LaunchCtx& lc, float2* psi, int n, int m, const ClauseMV* cl, const float2* ptab,
                          const float2* btab, int nsteps, bool first_p) {
  if (n < 1 || n > kOnchipMaxBits) return cudaErrorInvalidValue;
  const RunArgs A{psi, cl, ptab, btab, n, m, nsteps, first_p, false, 0.f};
  switch (n) {
#define QAA_CASE(T, R) \
  case T:              \
    return launch_cta<T, R>(lc, A);
    QAA_ONCHIP_SIZES(QAA_CASE)
#undef QAA_CASE
    default: {
      const cudaError_t e =
          allow_smem(reinterpret_cast<const void*>(warp_kernel), onchip_smem_bytes(8, QAA_MAX_CLAUSES_DEV));
      if (e != cudaSuccess) return e;
      warp_kernel<<<1, 32, onchip_smem_bytes(n, m), lc.stream>>>(A);
      return cudaGetLastError();
    }
  }
}

}  // namespace qaa
