// Mid-size evolver: the state of one instance stays in the registers of a team of
// 2^C CTAs for every step of a run.
//
// A CTA's tile holds T = n - C index bits.  Two layouts alternate, one per step:
//   A: x = l | cta << T                              (tile bits [0, T))
//   B: x = (l mod 2^D) | cta << D | (l >> D) << T    (tile bits [0, D) and [T, n))
// with D = T - C; tile bits [D, T) of one layout are the CTA bits of the other.
// A step turns the T tile bits, exchanges the tiles between the CTAs (element
// (cta, l) goes to CTA l >> D, slot (l mod 2^D) | cta << D, in either direction),
// turns the C bits that came in and applies P: one exchange per step, where the
// streaming passes read and write the state once per group of bits.
//
// Within a CTA a thread holds a window of R tile bits (tile.cuh).  For C <= R the
// incoming bits are in the TOP window: TOP BOT MID, exchange, TOP, P.  For C > R the
// rest of them is in MID: MID BOT TOP, exchange, TOP, MID, P.
//
// The exchange:
// * CLUSTER (8 CTAs of one cluster): st.async into the partners' shared memory,
//   counted by the receiver's mbarrier (a cluster barrier per step instead: 1.79
//   against 1.51 us per step at n = 13).  Two receive buffers in turn, for nothing else
//   (team_schedule.h): what a CTA has received in step j its partners sent after a
//   barrier behind their reads of step j - 1's buffer, which it fills in step j + 1.
// * grid (a cooperative launch): 64-bit words in global memory (L2) that say by
//   themselves whether they have arrived (kEmpty), so the exchange costs one store
//   and the polling of one load; with a grid barrier between stores and loads (a
//   release, an atomic, an acquire and the loads in sequence) n = 16 took 3.10
//   instead of 2.70 us per step.  The slots are used in turn (team_schedule.h): a warp
//   of its own (with two CTAs per SM: thread 0) runs the fences that order a slot's
//   emptying before its next word.
//
// Norm fold as in the streaming passes (NormFold), with the reference kept in the
// handle's fold slot across launches of a range: the sum measured after a step
// travels with the next exchange and corrects the P after it.
#include "team_schedule.h"
#include "tile.cuh"

namespace qaa {

namespace {

constexpr int kTeamRing = 3;  // phase rows in flight: this step's and two ahead
// Polls of a wait before it gives up, by default (half a second in the grid forms, eight
// in the cluster form, whose polls sleep) and with an injected fault (1 ms, 15 ms).  The
// cluster form must not give up while words sent to it are in flight, because its
// CTAs return after giving up: the smaller limit, too, is thousands of times a word's
// flight.
constexpr int kTeamPolls = 1 << 21, kTeamPollsInjected = 1 << 12;

struct TeamArgs {
  float2* psi;
  const uint16_t* energy;  // E(x)
  const float2* ptab;
  const float2* btab;
  float2* xbuf;    // grid: the exchange buffers, 2^n amplitudes each
  float2* part;    // grid: [receiver][sender] norm partials of the steps, then of the end
  unsigned* count; // grid barrier: arrivals, zeroed before the launch
  float2* ref;     // the range's reference norm (double-float)
  int* err;
  int n, m, nsteps;
  int polls;       // limit of every wait on another CTA
  bool first;      // the launch starts a range: apply P row 0, take the reference
  bool lose;       // injected fault: CTA 0 withholds its first exchange
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_smem(const void* p, unsigned rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
  return a;
}

// The grid exchange: amplitudes go through global memory as 64-bit words that say
// by themselves whether they have arrived.  A slot holds kEmpty (a NaN pattern no
// arithmetic result has) until its sender stores the amplitude; the receiver
// polls the slot, takes the value and stores kEmpty again.
constexpr unsigned long long kEmpty = ~0ull;
__device__ __forceinline__ unsigned long long word_load(const float2* p) {
  unsigned long long x;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
  return x;
}
__device__ __forceinline__ void word_store(float2* p, unsigned long long x) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(x) : "memory");
}
// Take N words at p, p + step, ...; false when the wait ran out.
template <int N>
__device__ __forceinline__ bool take_words(float2 (&v)[N], float2* p, int step, int polls) {
  unsigned long long x[N];
#pragma unroll
  for (int r = 0; r < N; ++r) x[r] = word_load(p + r * step);
  bool wait = true;
  for (int i = 0; wait && i < polls; ++i) {
    wait = false;
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (x[r] == kEmpty) {
        x[r] = word_load(p + r * step);
        wait = true;
      }
  }
#pragma unroll
  for (int r = 0; r < N; ++r) {
    v[r] = bits_f2(x[r]);
    word_store(p + r * step, kEmpty);
  }
  return !wait;
}
// The other grid exchange: plain stores, a grid barrier, plain loads.  Every
// CTA's stores before its `round`-th call are visible to this one after it; false
// when the wait ran out.  The counter only grows within a launch.  `arrive`: false for
// the injected fault.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned round, bool arrive, int polls, int tid, int* s_ok) {
  __syncthreads();
  if (tid == 0) {
    const unsigned target = round * gridDim.x;
    if (arrive) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    int ok = 0;
    for (int i = 0; i < polls && !ok; ++i) {
      unsigned c;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
      ok = c >= target;
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

template <int ID, int NT>
__device__ __forceinline__ void bar_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(NT) : "memory");
}
template <int ID, int NT>
__device__ __forceinline__ void bar_arrive() {
  asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(NT) : "memory");
}

// mbarrier transactions of the cluster exchange.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void peer_send(uint32_t a, float2 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a), "f"(v.x),
               "f"(v.y), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool recv_wait(uint64_t* bar, uint32_t parity, int polls) {
  for (int i = 0; i < polls; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

template <int T, int R, int C, bool CLUSTER>
struct TeamGeom : CtaGeom<T, R> {
  using G = CtaGeom<T, R>;
  static constexpr int D = T - C;
  static constexpr bool kSplit = C > R;  // incoming bits in TOP and MID
  static constexpr int kP = kSplit ? kMid : kTop;     // window of P
  static constexpr int kOut = kSplit ? kTop : kMid;   // window that sends
  static_assert(D >= 0 && (!kSplit || D >= R), "incoming bits must lie in TOP and MID");
  static_assert(!CLUSTER || C <= 3, "portable clusters of 8 CTAs");
  // grid: self-validating words, with a warp of its own for the fence that orders
  // the emptied slots; 512 threads with 32 amplitudes each (2^14 per CTA) use the
  // grid barrier: the words' second set of stores and registers cost more there
  // than the barrier (n = 21: 13.1 against 11.5 us per step)
  static constexpr bool kWords = !CLUSTER && G::NT < 512;
  static constexpr int kPerSm = C >= 8 ? 2 : 1;
  static constexpr bool kFenceWarp = kWords && kPerSm == 1;
  static constexpr int kThreads = G::NT + (kFenceWarp ? 32 : 0);
  // increments beside the values where there are registers for them; they go through
  // the transposes too where the tile is the SM's only one (two: rounded at every window)
  static constexpr bool kInc = R < 5;
  static constexpr bool kCarry = kInc && kPerSm == 1;
  // What the rounding before the exchange leaves out stays in registers and is taken up
  // two steps on, when the amplitude is in the same layout, thread and register again.
  // Its turn in between is ignored: at angles that are not small it is one more error of
  // the size of the rounding.  The scales of the steps in between are not: they reach
  // 2^-n.
  static constexpr bool kLeft = kCarry;
  // transpose buffers: two where they fit (one barrier per transpose instead of two);
  // the cluster's receive buffers lie behind them
  static constexpr int kBufs = T > 13 ? 1 : 2;
  static_assert(!CLUSTER || kBufs == 2, "team_schedule.h");
  static constexpr size_t kTile = (tile_bytes<T, R, kCarry>() + 15u) / 16u * 16u;
  static constexpr size_t kBytes = kTile * kBufs + (CLUSTER ? (kClusterBuffers - 2) * 8u * static_cast<size_t>(G::SLOTS) : 0u);
};

template <int T, int R, int C, bool CLUSTER>
size_t team_smem(int m) {
  using G = TeamGeom<T, R, C, CLUSTER>;
  return G::kBytes + 8u * kTeamRing * static_cast<size_t>(m + 3);
}

template <int T, int R, int C, bool CLUSTER>
__global__ void __launch_bounds__(TeamGeom<T, R, C, CLUSTER>::kThreads, (TeamGeom<T, R, C, CLUSTER>::kPerSm)) team_kernel(const TeamArgs A) {
  using G = TeamGeom<T, R, C, CLUSTER>;
  constexpr int NT = G::NT, N = G::N, D = G::D, TEAM = 1 << C;
  constexpr int kP = G::kP, kOut = G::kOut;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ DFloat s_w[NT / 32 > 0 ? NT / 32 : 1];
  __shared__ float2 s_part[2][CLUSTER ? TEAM : 1];  // in the steps; at the end
  __shared__ __align__(8) uint64_t s_bar[3];
  __shared__ int s_late, s_ok;
  const int tid = threadIdx.x;
  const unsigned cta = CLUSTER ? cluster_rank() : blockIdx.x;
  const int mp1 = A.m + 1;
  float2* s_buf = reinterpret_cast<float2*>(smem);
  float2* s_ab = s_buf + G::kBytes / 8;
  float2* s_p = s_ab + 2 * kTeamRing;
  auto fetch = [&](int j) {
    if (j < A.nsteps) {
      float2* dst = s_p + (j % kTeamRing) * mp1;
      const float2* src = A.ptab + static_cast<size_t>(j + 1) * mp1;
      for (int i = tid; i < mp1; i += NT) cp_async8(dst + i, src + i);
      if (tid < 2) cp_async8(s_ab + 2 * (j % kTeamRing) + tid, A.btab + static_cast<size_t>(j) * (A.n + 1) + tid);
    }
    cp_async_commit();
  };
  if constexpr (!CLUSTER) {
    if (tid == 0) s_late = 0;
    __syncthreads();
    if (G::kFenceWarp && tid >= NT) {
      // the fence warp: takes and kEmpty stores of step j come before any amplitude of
      // step j + kWordFenceLag leaves this CTA
      for (int j = 0; j < A.nsteps; ++j) {
        bar_sync<2, NT + 32>();
        if (*static_cast<volatile int*>(&s_late) || j + kWordFenceLag >= A.nsteps) return;
        __threadfence();
        if (j & 1) bar_arrive<4, NT + 32>(); else bar_arrive<3, NT + 32>();
      }
      return;
    }
  }
  for (int j = 0; j < kTeamRing - 1; ++j) fetch(j);

  // this thread's amplitudes in the P window: tile index lp + r * lstep
  const int lp = win_base<T, R, kP>(tid);
  constexpr int lstep = win_step<T, R, kP>();
  const unsigned xa = static_cast<unsigned>(lp) | cta << T;
  auto index_b = [&](int l) { return static_cast<unsigned>(l & ((1 << D) - 1)) | cta << D | static_cast<unsigned>(l >> D) << T; };
  unsigned ea[N / 2], eb[N / 2];
#pragma unroll
  for (int r = 0; r < N; r += 2) {
    ea[r / 2] = 8u * (A.energy[xa + r * lstep] | static_cast<unsigned>(A.energy[xa + (r + 1) * lstep]) << 16);
    eb[r / 2] = 8u * (A.energy[index_b(lp + r * lstep)] | static_cast<unsigned>(A.energy[index_b(lp + (r + 1) * lstep)]) << 16);
  }
  Tile<N, G::kInc> x;
  auto& v = x.v;
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = A.psi[xa + r * lstep];
  const int pc = __popc(lp) + __popc(cta);

  // a warp's sum of |v|^2 for the CTA's partial
  auto measure = [&]() {
    const DFloat t = warp_sum(norm_of<N>(x));
    if ((tid & 31) == 0) s_w[tid >> 5] = t;
  };
  // the CTA's partial to every CTA of the team (one warp, after a barrier since measure)
  auto publish = [&](int bar, int end) {
    DFloat t{0.f, 0.f};
    for (int w = 0; w < NT / 32; ++w) t = df_add(t, s_w[w]);
    if (CLUSTER) {
      if (tid < TEAM) peer_send(peer_smem(s_part[end] + cta, tid), make_float2(t.hi, t.lo), peer_smem(s_bar + bar, tid));
    } else {
      // a copy for every CTA: its slots are emptied by their one reader
      for (int i = tid; i < TEAM; i += 32) word_store(A.part + (end * TEAM + i) * TEAM + cta, f2_bits(make_float2(t.hi, t.lo)));
    }
  };
  // the team's sum, the same in every thread
  auto collect = [&](int end) {
    DFloat t{0.f, 0.f};
    if (CLUSTER) {
      for (int i = 0; i < TEAM; ++i) t = df_add(t, DFloat{s_part[end][i].x, s_part[end][i].y});
    } else {
      // warp 0 takes the partials; the others get the sum through shared memory
      if (tid < 32) {
        for (int i = tid; i < TEAM; i += 32) {
          float2 p[1];
          if (!take_words<1>(p, A.part + (end * TEAM + cta) * TEAM + i, 0, A.polls)) s_late = 1;
          t = df_add(t, DFloat{p[0].x, p[0].y});
        }
        t = warp_sum(t);
        if (tid == 0) s_part[end][0] = make_float2(t.hi, t.lo);
      }
      team_sync<NT>();
      t = DFloat{s_part[end][0].x, s_part[end][0].y};
    }
    return t;
  };

  bool pending = true;  // a measured sum travels with the next exchange
  DFloat ref{0.f, 0.f};
  if (!A.first) {
    const float2 r = __ldcg(A.ref);
    ref = DFloat{r.x, r.y};
  }
  x.zero();
  measure();
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = times_i(v[r], pc + __popc(r));
  if (A.first) x.phase(ea, A.ptab);

  // the bytes that arrive in step j
  auto expect = [&](int j) {
    const bool sum = j == 0 || j % fold_period(T + C) == 0;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(s_bar + (j & 1))),
                 "r"((8u << T) + (sum ? 8u * TEAM : 0u))
                 : "memory");
  };
  if (CLUSTER && tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(s_bar)) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(s_bar + 1)) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(s_bar + 2)) : "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(s_bar + 2)), "r"(8u * TEAM) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    expect(0);
    expect(1);
  }
  cp_async_wait<0>();
  if (CLUSTER)
    cluster_barrier();  // every CTA of the cluster runs before its shared memory is written
  else
    team_sync<NT>();

  // transposes through one or two buffers; `b` alternates so that one barrier is enough
  int b = 0;
  auto buffer = [&](int k) { return s_buf + G::kTile / 8 * k; };
  auto receive = [&](int j) {  // cluster
    return s_buf + G::kTile / 8 * 2 + static_cast<size_t>(G::SLOTS) * (cluster_receive(j) - 2);
  };
  unsigned left[2][G::kLeft ? N : 1] = {};  // by layout
  bool late = false;
  TurnScale ts;
  for (int j = 0; j < A.nsteps; ++j) {
    const RotCoef c = rot_coef(s_ab + 2 * (j % kTeamRing));
    const float2* prow = s_p + (j % kTeamRing) * mp1;
    float2* b0 = buffer(CLUSTER ? cluster_transpose(j, 0) : b);
    float2* b1 = buffer(CLUSTER ? cluster_transpose(j, 1) : (G::kBufs == 2 ? b ^ 1 : 0));
    auto middle = [&]() {  // barrier between a put and a get; with one buffer another before the next put
      cp_async_wait<0>();
      team_sync<NT>();
      if (G::kWords) late = *static_cast<volatile int*>(&s_late) != 0;
      if (G::kWords && !G::kFenceWarp && tid == 0) __threadfence();  // behind step j - 1
    };
    auto reuse = [&]() {
      if (G::kBufs == 1) team_sync<NT>();
    };
    if constexpr (!G::kSplit) {
      x.template turn<0, R>(c);
      put_tile<T, R, kTop, G::kCarry>(x, b0, tid);
      middle();
      if (G::kWords && late) {
        if (G::kFenceWarp) bar_arrive<2, NT + 32>();  // the fence warp may be waiting for this step's
        break;
      }
      if (pending && tid < 32) publish(j & 1, 0);
      fetch(j + kTeamRing - 1);
      get_tile<T, R, kBot, G::kCarry>(x, b0, tid);
      reuse();
      x.template turn<0, R>(c, !G::kCarry);
      put_tile<T, R, kBot, G::kCarry>(x, b1, tid);
      team_sync<NT>();
      get_tile<T, R, kMid, G::kCarry>(x, b1, tid);
      reuse();
      x.template turn<0, T - 2 * R>(c);
    } else {
      x.template turn<0, T - 2 * R>(c);
      put_tile<T, R, kMid, G::kCarry>(x, b0, tid);
      middle();
      if (G::kWords && late) {
        if (G::kFenceWarp) bar_arrive<2, NT + 32>();  // the fence warp may be waiting for this step's
        break;
      }
      if (pending && tid < 32) publish(j & 1, 0);
      fetch(j + kTeamRing - 1);
      get_tile<T, R, kBot, G::kCarry>(x, b0, tid);
      reuse();
      x.template turn<0, R>(c, !G::kCarry);
      put_tile<T, R, kBot, G::kCarry>(x, b1, tid);
      team_sync<NT>();
      get_tile<T, R, kTop, G::kCarry>(x, b1, tid);
      reuse();
      x.template turn<0, R>(c, !G::kCarry);
    }
    // only the values leave: the one rounding of an amplitude per step
    if constexpr (!G::kLeft)
      x.settle();
    else if (j & 1)
      x.leave(left[1]);
    else
      x.leave(left[0]);
    // exchange: tile index l -> CTA l >> D, slot (l mod 2^D) | cta << D
    {
      const int l0 = win_base<T, R, kOut>(tid);
      constexpr int ls = win_step<T, R, kOut>();
      constexpr int dm = (1 << D) - 1;
      const bool lost = A.lose && cta == 0 && j == 0;
      if constexpr (CLUSTER) {
        float2* dst = receive(j) + G::slot((l0 & dm) | static_cast<int>(cta) << D);
        if (!lost) {
#pragma unroll
          for (int r = 0; r < N; ++r)
            peer_send(peer_smem(dst, (l0 >> D) + ((r * ls) >> D)) + 8u * G::slot((r * ls) & dm), v[r],
                      peer_smem(s_bar + (j & 1), (l0 >> D) + ((r * ls) >> D)));
        }
        // the CTA goes on or gives up as one: words may arrive as some threads' waits run out
        late = __syncthreads_or(!recv_wait(s_bar + (j & 1), (j >> 1) & 1, A.polls)) != 0;
        if (late) break;
        if (tid == 0 && j + 2 < A.nsteps) expect(j + 2);
        get<T, R, kTop>(v, receive(j), tid);
      } else {
        float2* xb = A.xbuf + (static_cast<size_t>(G::kWords ? word_buffer(j) : j & 1) << A.n);
        float2* dst = xb + (static_cast<size_t>(l0 >> D) << T) + ((l0 & dm) | static_cast<int>(cta) << D);
        float2* src = xb + (static_cast<size_t>(cta) << T) + win_base<T, R, kTop>(tid);
        if constexpr (G::kWords) {
          if (G::kFenceWarp && j >= kWordFenceLag) {  // the fence warp is done with step j - kWordFenceLag
            static_assert(kWordFenceLag == 2, "one barrier per parity");
            if (j & 1) bar_sync<4, NT + 32>(); else bar_sync<3, NT + 32>();
          }
          if (!lost) {
#pragma unroll
            for (int r = 0; r < N; ++r)
              word_store(dst + ((static_cast<size_t>((r * ls) >> D) << T) + ((r * ls) & dm)), f2_bits(v[r]));
          }
          if (!take_words<N>(v, src, win_step<T, R, kTop>(), A.polls)) s_late = 1;
          if (G::kFenceWarp) bar_arrive<2, NT + 32>();
        } else {
#pragma unroll
          for (int r = 0; r < N; ++r) __stcg(dst + ((static_cast<size_t>((r * ls) >> D) << T) + ((r * ls) & dm)), v[r]);
          if (!grid_barrier(A.count, static_cast<unsigned>(j) + 1u, !lost, A.polls, tid, &s_ok)) {
            late = true;
            break;
          }
#pragma unroll
          for (int r = 0; r < N; ++r) v[r] = __ldcg(src + r * win_step<T, R, kTop>());
        }
      }
    }
    float k = 0.f;
    if (pending) {
      const DFloat s = collect(0);
      if (j == 0 && A.first) {
        ref = s;
        if (cta == 0 && tid == 0) *A.ref = make_float2(s.hi, s.lo);
      }
      k = ts.fold(ref, s);
      pending = false;
    }
    if constexpr (!G::kSplit) {
      x.template turn<R - C, R>(c, true);
    } else {
      x.template turn<0, R>(c, true);
      float2* b2 = buffer(b);
      put_tile<T, R, kTop, G::kCarry>(x, b2, tid);
      team_sync<NT>();
      get_tile<T, R, kMid, G::kCarry>(x, b2, tid);
      reuse();
      x.template turn<D - R, T - 2 * R>(c, !G::kCarry);
      if (G::kBufs == 2) b ^= 1;
    }
    if (j & 1)
      x.phase(ea, prow);
    else
      x.phase(eb, prow);
    if (c.pow2 != 1.0f) x.scale(c.pow2);
    if (k != 0.f) x.grow(k);
    if (G::kLeft && (c.pow2 != 1.0f || k != 0.f)) {
      const float f = fmaf(c.pow2, k, c.pow2);
      scale_rest(left[0], f);
      scale_rest(left[1], f);
    }
    ts.step(c.r);
    if ((j + 1) % fold_period(T + C) == 0 && j + 1 < A.nsteps) {
      measure();
      pending = true;
    }
  }
  // the last fold
  if (!CLUSTER) {
    team_sync<NT>();
    late = late || *static_cast<volatile int*>(&s_late) != 0;
  }
  if (!late) {  // the same in every thread of the CTA
    measure();
    team_sync<NT>();
    if (tid < 32) publish(2, 1);
    if (CLUSTER) {
      late = __syncthreads_or(!recv_wait(s_bar + 2, 0, A.polls)) != 0;
    }
    x.grow(ts.fold(ref, collect(1)));
    if (!CLUSTER) late = *static_cast<volatile int*>(&s_late) != 0;
  }
  if (late && (CLUSTER || tid == 0)) atomicExch(A.err, 2);
  if (CLUSTER) cluster_barrier();  // no CTA leaves while another may still store into its shared memory
  if (A.nsteps & 1) {
#pragma unroll
    for (int r = 0; r < N; ++r) A.psi[index_b(lp + r * lstep)] = times_i(x.at(r), -(pc + __popc(r)));
  } else {
#pragma unroll
    for (int r = 0; r < N; ++r) A.psi[xa + r * lstep] = times_i(x.at(r), -(pc + __popc(r)));
  }
}

template <int T, int R, int C, bool CLUSTER>
cudaError_t launch(const LaunchCtx& lc, const TeamArgs& A) {
  auto kern = team_kernel<T, R, C, CLUSTER>;
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kern), team_smem<T, R, C, CLUSTER>(QAA_MAX_CLAUSES_DEV));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << C);
  cfg.blockDim = dim3(TeamGeom<T, R, C, CLUSTER>::kThreads);
  cfg.dynamicSmemBytes = team_smem<T, R, C, CLUSTER>(A.m);
  cfg.stream = lc.stream;
  cudaLaunchAttribute at[1];
  if (CLUSTER) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {1u << C, 1u, 1u};
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (!TeamGeom<T, R, C, CLUSTER>::kWords && !CLUSTER) {
    e = cudaMemsetAsync(A.count, 0, sizeof(unsigned), lc.stream);
    if (e != cudaSuccess) return e;
  }
  return cudaLaunchKernelEx(&cfg, kern, A);
}

// Whether the current device can hold the whole team at once.
template <int T, int R, int C, bool CLUSTER>
bool fits(int num_sms, int m) {
  auto kern = team_kernel<T, R, C, CLUSTER>;
  if (allow_smem(reinterpret_cast<const void*>(kern), team_smem<T, R, C, CLUSTER>(QAA_MAX_CLAUSES_DEV)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int k = 0;
  if (CLUSTER) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << C);
    cfg.blockDim = dim3(TeamGeom<T, R, C, CLUSTER>::kThreads);
    cfg.dynamicSmemBytes = team_smem<T, R, C, CLUSTER>(m);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {1u << C, 1u, 1u};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&k, kern, &cfg) == cudaSuccess) return k >= 1;
  } else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, kern, TeamGeom<T, R, C, CLUSTER>::kThreads,
                                                           team_smem<T, R, C, CLUSTER>(m)) == cudaSuccess) {
    return k * num_sms >= 1 << C;
  }
  cudaGetLastError();
  return false;
}

}  // namespace

// The team of each n: tile bits T, register bits R, CTA bits C.  Small tiles win
// up to the exchange's latency.  us per step of a 200-step run, the launch included,
// of the choices tried (with single turns; the increments beside the amplitudes and
// the paired turns add up to 30 %):
//   n = 12 cluster (9,3) 1.20, one CTA 1.39      n = 13 cluster (10,4) 1.51, one CTA 2.39
//   n = 14 cluster (11,4) 2.01, grid (9,3) 2.05, (10,4) 2.39, one CTA 4.79
//   n = 15 grid (9,3) 2.08, (10,4) 2.49, (11,4) 2.62, cluster (12,4) 3.09
//   n = 16 grid (10,4) 2.70, (11,4) 2.81, cluster (13,5) 5.16
//   n = 17 grid (11,4) 2.88, (12,4) 4.04, (13,5) 5.57    n = 18 grid (11,4) 3.17, (12,4) 4.06
//   n = 19 grid (12,4) 4.08, (13,5) 6.51
//   n = 20 grid (12,4) with two CTAs per SM 6.36, (13,5) 6.65    n = 21 grid (14,5) 11.5
// The kernels as they are, 400 steps, against the streaming passes (n = 12..14: the
// earlier one-CTA kernel): n = 12 1.40 / 3.16, 13 1.88 / 4.85, 14 2.41 / 8.60, 15 2.30 /
// 12.4, 16 3.04 / 12.4, 17 3.49 / 13.2, 18 3.71 / 14.6, 19 5.16 / 14.7, 20 7.18 / 18.8,
// 21 12.3 / 24.9; the state's error against 64 bits 2e-7 / 3.2e-6 (n = 16).
// Without the increments in the transposes (an amplitude rounded at every window) n = 16
// took 2.94, n = 19 4.44, with four times the error of <H_P> and of the ground
// probability; with what a rounding leaves out packed into 4 bytes instead n = 16 3.51,
// n = 19 5.08.  n = 20 rounds at every window (9.1 with the increments in the transposes;
// 8.5 with a fence warp, whose share leaves 96 registers; 6.6 without increments: a
// rounding per pair of turns), 200 steps, rms of 24 instances: state 7.3e-7 (1.2e-6 without
// increments, 2.5e-6 from the earlier passes), <H_P> 5.5e-8 (1.1e-7, 1.9e-7), ground
// probability 2.3e-7 (4.3e-7, 6.1e-7).  n = 21 has no registers for increments: a
// rounding per pair of turns, state 1.3e-6 (2.6e-6 from the earlier passes), <H_P> 1.1e-7
// (1e-7), ground probability 3.1e-7 (2.9e-7), 400 steps 1.8e-6 (3.7e-6), 3.7e-7 (6.3e-7),
// 2.1e-7 (2.1e-7).
// n <= 11 stays with one CTA (0.94 at n = 11 against 1.07 in a cluster); 2^22
// amplitudes do not fit in the registers.
#define QAA_TEAMS(X)                                                                                       \
  X(9, 3, 3, true) X(10, 4, 3, true) X(11, 4, 3, true) X(9, 3, 6, false) X(10, 4, 6, false) X(11, 4, 6, false) \
  X(11, 4, 7, false) X(12, 4, 7, false) X(12, 4, 8, false) X(14, 5, 7, false)

// Scratch: partials [2][2^C][2^C], the barrier counter, then the exchange buffers;
// nothing for a cluster.
constexpr size_t kTeamHead = 2u * 65536u * sizeof(float2);
size_t team_bytes(int n) {
  if (n <= 14) return 0;
  return kTeamHead + 256 + (static_cast<size_t>(8 * (n <= 20 ? kWordBuffers : 2)) << n);
}

cudaError_t team_reset(const LaunchCtx& lc, int n, void* work) {
  if (n <= 14) return cudaSuccess;
  return cudaMemsetAsync(work, 0xff, n <= 20 ? team_bytes(n) : kTeamHead, lc.stream);
}

bool team_fits(int n, int m, int num_sms) {
  switch (n) {
#define QAA_CASE(T, R, C, K) \
  case T + C:                \
    return fits<T, R, C, K>(num_sms, m);
    QAA_TEAMS(QAA_CASE)
#undef QAA_CASE
    default:
      return false;
  }
}

cudaError_t launch_team(const LaunchCtx& lc, float2* psi, int n, int m, const uint16_t* energy, const float2* ptab,
                        const float2* btab, int nsteps, bool first, void* work, double* fold, int* err, bool lose) {
  if (nsteps < 1) return cudaErrorInvalidValue;
  char* w = static_cast<char*>(work);
  TeamArgs A;
  A.psi = psi;
  A.energy = energy;
  A.ptab = ptab;
  A.btab = btab;
  A.part = reinterpret_cast<float2*>(w);
  A.count = reinterpret_cast<unsigned*>(w + kTeamHead);
  A.xbuf = reinterpret_cast<float2*>(w + kTeamHead + 256);
  A.ref = reinterpret_cast<float2*>(fold);
  A.err = err;
  A.n = n;
  A.m = m;
  A.nsteps = nsteps;
  A.polls = lose ? kTeamPollsInjected : kTeamPolls;
  A.first = first;
  A.lose = lose;
  switch (n) {
#define QAA_CASE(T, R, C, K) \
  case T + C:                \
    return launch<T, R, C, K>(lc, A);
    QAA_TEAMS(QAA_CASE)
#undef QAA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace qaa
