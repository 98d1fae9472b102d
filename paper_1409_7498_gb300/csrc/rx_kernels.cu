// Reaction step (Sec. III, Table I) and observables.
//
// The three selection stages are atomic-free and independent of thread
// scheduling: every random choice is the minimum of Philox keys that depend
// only on (seed, step, particle ids), so the outcome is a function of the
// state alone.
//   rx_find      steps 1-5: each eligible A scans its 27 neighbour cells for
//                eligible T (type mask, state window, not yet bonded to A) with
//                r^2 < r_react^2 tested in FP64 on absolute positions (after an
//                FP32 prefilter that can only widen the set), accepts each with
//                u < k dt Theta (Eq. 4) and keeps the accepted T of smallest
//                key Philox(step, id_A, id_T): one T per A.
//   rx_select_T  steps 6-7: each A winner scans the cells around its T for the
//                other A's that picked the same T and keeps the pair only if
//                its key Philox(step, id_T, id_A) is the smallest: one A per T.
//   rx_select_apply  steps 6-9 fused: one A per T, then the bonds, both
//                adjacency rows and the states; the running populations per
//                (type, state) move with each bond, and the last block writes
//                the reaction's history record from them.
#include <cuda_runtime.h>

#include <type_traits>

#include "prx_internal.cuh"
#include "rx_device.cuh"

namespace prx {

namespace {

__device__ __forceinline__ long long block_sum_ll(long long v) {
  __shared__ long long part[RX_THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) part[wid] = v;
  __syncthreads();
  long long t = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < RX_THREADS / 32; ++w) t += part[w];
  return t;
}

// Work list of the eligible A's (their order does not matter: each A's
// result goes to its own slot), and win[] cleared for every slot.  Four slots
// per thread (one 4-byte load of types and one of states, one 16-byte clear
// of win), so a quarter of the blocks and of the block-level atomics on the
// work-list counter that one slot per thread takes.  b: the block's index
// among the blocks of 4 RX_THREADS slots.
__device__ __forceinline__ void rx_compact_body(const Sys& S, uint32_t b) {
  const RxParams& R = S.R;
  Ctl* ctl = S.ctl;
  const SoA B = ctl->set ? S.s1 : S.s0;
  const uint32_t i0 = (b * blockDim.x + threadIdx.x) * 4u;
  uint32_t bits = 0u;
  if (i0 + 3u < S.n) {
    const uchar4 t4 = *reinterpret_cast<const uchar4*>(B.type + i0);
    const char4 s4 = *reinterpret_cast<const char4*>(B.state + i0);
    *reinterpret_cast<uint4*>(S.win + i0) = make_uint4(NONE, NONE, NONE, NONE);
    const uint32_t tt[4] = {t4.x, t4.y, t4.z, t4.w};
    const int ss[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool el = R.nr > 1 ? rx_elig_A(R, tt[u], ss[u]) != 0u
                               : in_window(R.mask_A, R.a_lo, R.a_hi, tt[u], ss[u]);
      bits |= (el ? 1u : 0u) << u;
    }
  } else {
    for (uint32_t u = 0; u < 4u && i0 + u < S.n; ++u) {
      const uint32_t i = i0 + u;
      S.win[i] = NONE;
      const bool el = R.nr > 1 ? rx_elig_A(R, B.type[i], B.state[i]) != 0u
                               : in_window(R.mask_A, R.a_lo, R.a_hi, B.type[i], B.state[i]);
      bits |= (el ? 1u : 0u) << u;
    }
  }
  // warp inclusive scan of the counts, block prefix in shared memory, one
  // atomic per block
  const uint32_t c = __popc(bits);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  __shared__ uint32_t wcnt[RX_THREADS / 32];
  __shared__ uint32_t bbase;
  if (lane == 31) wcnt[wid] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < RX_THREADS / 32; ++w) {
      const uint32_t v = wcnt[w];
      wcnt[w] = t;
      t += v;
    }
    bbase = t ? atomicAdd(&ctl->n_active, t) : 0u;
  }
  __syncthreads();
  uint32_t pos = bbase + wcnt[wid] + x - c;
  for (uint32_t u = 0; u < 4u; ++u)
    if ((bits >> u) & 1u) S.tmp[pos++] = i0 + u;
}
__global__ void __launch_bounds__(RX_THREADS) k_rx_compact4(Sys S) { rx_compact_body(S, blockIdx.x); }

__global__ void __launch_bounds__(RX_THREADS)
    kb_rx_compact(const Sys* __restrict__ T, const BlkMap* __restrict__ M) {
  const BlkMap m = M[blockIdx.x];
  const Sys& S = T[m.sys];
  if (!S.has_rx) return;  // this member has no reaction scheme
  if (m.b & 3u) return;  // (the map's entries are blocks of RX_THREADS slots)
  rx_compact_body(S, m.b >> 2);
}

// KIND 0: one reaction by the random rule; 1: the nearest rule or concurrent
// reactions, with the lanes that suit their number of A's; 2: a batch's member,
// either of these (four lanes: the other members fill the GPU too).
template <bool NL16, int KIND>
__device__ __forceinline__ void rx_find_body(const Sys& S, const Blk blk, long long step_arg) {
  const RxParams& R = S.R;

  Ctl* ctl = S.ctl;
  const unsigned long long step = step_arg >= 0 ? (unsigned long long)step_arg : ctl->step;
  const SoA B = ctl->set ? S.s1 : S.s0;
  const uint4* P = ctl->phase ? S.P1 : S.P0;
  const uint32_t nact = ctl->n_active;
  // four lanes per eligible A (one reaction, random rule) or a group: blocks past them have nothing to do
  const bool four = KIND == 0 || (KIND == 2 && R.rule != PRX_SELECT_NEAREST && R.nr <= 1);
  const uint32_t lanes = KIND == 1 ? (uint32_t)rx_find_lanes(R, nact) : 4u;
  if (blk.b * (blockDim.x / lanes) >= nact) return;
  long long ncand = 0, nret = 0;
  if (four) {
    rx_find_random4<NL16>(S, blk, B, P, step, S.tmp, nact, ncand, nret);
  } else if constexpr (KIND != 0) {
    // the nearest rule and concurrent reactions: a group of lanes per eligible A
    auto groups = [&](auto g) {
      constexpr int G = decltype(g)::value;
      const uint32_t lane = threadIdx.x & 31u;
      for (uint32_t wb = (blk.b * blockDim.x + (threadIdx.x & ~31u)) / G; wb < nact; wb += blk.nb * blockDim.x / G) {
        const uint32_t w = wb + lane / G;
        const bool valid = w < nact;
        const uint32_t i = valid ? S.tmp[w] : 0u;
        uint32_t best = NONE, ch = 0u;
        if (R.rule == PRX_SELECT_NEAREST) best = nearest_partner<NL16, G>(S, B, P, i, valid, true, ncand);
        else best = rx_find_multi<NL16, G>(S, B, P, step, i, valid, ncand, nret, ch);
        if (valid && lane % G == 0u) {
          if (R.nr > 1) S.wch[i] = (uint8_t)ch;
          S.win[i] = best;
        }
      }
    };
    if (KIND == 2 || lanes == 4u) groups(std::integral_constant<int, 4>{});
    else if constexpr (KIND == 1) {
      if (lanes == 1u) groups(std::integral_constant<int, 1>{});
      else groups(std::integral_constant<int, RX_GROUP>{});
    }
  }
  const long long c = block_sum_ll(ncand);
  const long long r = block_sum_ll(nret);
  if (threadIdx.x == 0 && (c | r)) {
    atomicAdd((unsigned long long*)&ctl->trace[0], (unsigned long long)c);
    atomicAdd((unsigned long long*)&ctl->trace[1], (unsigned long long)r);
  }
}

template <bool NL16, int KIND>
__global__ void __launch_bounds__(RX_THREADS, 4) k_rx_find(Sys S, long long step_arg) {
  rx_find_body<NL16, KIND>(S, Blk{blockIdx.x, gridDim.x}, step_arg);
}
__global__ void __launch_bounds__(RX_THREADS, 4)
    kb_rx_find(const Sys* __restrict__ T, const BlkMap* __restrict__ M) {
  const BlkMap m = M[blockIdx.x];
  const Sys& S = T[m.sys];
  if (!S.has_rx) return;  // this member has no reaction scheme
  if (S.nl16) rx_find_body<true, 2>(S, Blk{m.b, m.nb}, -1LL);
  else rx_find_body<false, 2>(S, Blk{m.b, m.nb}, -1LL);
}

// Steps 6-7 for one A winner: every other A that picked the same T lies
// within r_react of T, hence in T's Verlet list.
template <bool NL16>
__device__ __forceinline__ void rx_find_T_body(const Sys& S, const Blk blk) {
  const RxParams& R = S.R;
  if (R.rule != PRX_SELECT_NEAREST) return;
  Ctl* ctl = S.ctl;
  const SoA B = ctl->set ? S.s1 : S.s0;
  const uint4* P = ctl->phase ? S.P1 : S.P0;
  const uint32_t i = blk.b * blockDim.x + threadIdx.x;
  if (i >= S.n || !in_window(R.mask_T, R.t_lo, R.t_hi, B.type[i], B.state[i])) return;
  long long unused = 0;
  S.win[i] = nearest_partner<NL16, 1>(S, B, P, i, true, false, unused);
}

template <bool NL16>
__global__ void __launch_bounds__(RX_THREADS) k_rx_find_T(Sys S) {
  rx_find_T_body<NL16>(S, Blk{blockIdx.x, gridDim.x});
}
__global__ void __launch_bounds__(RX_THREADS)
    kb_rx_find_T(const Sys* __restrict__ T, const BlkMap* __restrict__ M) {
  const BlkMap m = M[blockIdx.x];
  const Sys& S = T[m.sys];
  if (!S.has_rx) return;  // this member has no reaction scheme
  if (S.nl16) rx_find_T_body<true>(S, Blk{m.b, m.nb});
  else rx_find_T_body<false>(S, Blk{m.b, m.nb});
}

// Table I steps 6-9 in one pass over the eligible A's (the compacted list
// S.tmp): the T that an A picked keeps the A with the smallest key_T
// (random rule), or a mutual nearest pair is accepted with probability
// k dt Theta (nearest rule); an A that keeps its T forms the bond at once:
// adjacency of both, states, and a record in the bond list.  The decisions
// read only the choices (win) and ids, which no bond changes, and each A
// and each T take part in at most one bond, so forming bonds while other
// A's still decide changes nothing.  Bond-list positions come from one
// atomic per warp: the list's order may vary between runs (it is read back
// sorted), its content does not.
template <bool NL16>
__device__ __forceinline__ void rx_select_apply_body(const Sys& S, const Blk blk, long long step_arg) {
  const RxParams& R = S.R;
  Ctl* ctl = S.ctl;
  const unsigned long long step = step_arg >= 0 ? (unsigned long long)step_arg : ctl->step;
  const SoA B = ctl->set ? S.s1 : S.s0;
  const uint32_t nact = ctl->n_active;
  // blocks past the eligible A's have nothing to do; the last of the others
  // (of the first, when there is no A) writes the record
  const uint32_t lanes = (uint32_t)rx_select_lanes(R, nact);
  const uint32_t per = blockDim.x / lanes;  // A's per block and pass
  const uint32_t busy = max(1u, min(blk.nb, (nact + per - 1u) / per));
  if (blk.b >= busy) return;
  long long nwin = 0, nfin = 0;
  // population changes of this block's bonds, per (type, state)
  __shared__ int32_t dpop[PRX_MAX_TYPES * PRX_MAX_STATES];
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += blockDim.x) dpop[k] = 0;
  __syncthreads();
  // block-strided over the eligible A's (a group of lanes each), warp-uniform
  // trip count
  auto groups = [&](auto g) {
    constexpr uint32_t G = decltype(g)::value;
    for (uint32_t base = blk.b * per; base < nact; base += blk.nb * per) {
      const uint32_t w = base + threadIdx.x / G;
      const bool first = threadIdx.x % G == 0u;
      const uint32_t i = w < nact ? S.tmp[w] : 0u;
      bool winner;
      const uint32_t T = rx_decide<NL16, (int)G>(S, B, step, i, w < nact, winner);
      nwin += winner && first ? 1 : 0;
      nfin += rx_form(S, B, step, i, first ? T : NONE, dpop) ? 1 : 0;
    }
  };
  if (lanes == 4u) groups(std::integral_constant<uint32_t, 4>{});
  else groups(std::integral_constant<uint32_t, 1>{});
  const long long cw = block_sum_ll(nwin);
  const long long cf = block_sum_ll(nfin);
  if (threadIdx.x == 0) {
    if (R.rule == PRX_SELECT_NEAREST) {  // mutual pairs, accepted pairs
      if (cw) atomicAdd((unsigned long long*)&ctl->trace[1], (unsigned long long)cw);
      if (cf) atomicAdd((unsigned long long*)&ctl->trace[2], (unsigned long long)cf);
    } else if (cw) {
      atomicAdd((unsigned long long*)&ctl->trace[2], (unsigned long long)cw);
    }
    if (cf) atomicAdd((unsigned long long*)&ctl->trace[3], (unsigned long long)cf);
  }
  // the block's population changes into its replica of the running counts
  // (POP_REPLICAS copies, so that blocks do not all meet on the same few
  // counters); the last block sums the replicas into the reaction record
  // (populations, bonds, step)
  __syncthreads();
  int32_t* rep = S.pop + (size_t)(blk.b % POP_REPLICAS) * (PRX_MAX_TYPES * PRX_MAX_STATES);
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += blockDim.x)
    if (dpop[k]) atomicAdd(rep + k, dpop[k]);
  __threadfence();
  __shared__ bool is_last;
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(&ctl->done_rx, 1u) == busy - 1;
  __syncthreads();
  if (is_last) {
    if (threadIdx.x == 0) ctl->done_rx = 0u;
    rx_record(S, step_arg >= 0 ? step_arg : (long long)ctl->step);
  }
}

template <bool NL16>
__global__ void __launch_bounds__(RX_THREADS) k_rx_select_apply(Sys S, long long step_arg) {
  rx_select_apply_body<NL16>(S, Blk{blockIdx.x, gridDim.x}, step_arg);
}
__global__ void __launch_bounds__(RX_THREADS, 4)
    kb_rx_select_apply(const Sys* __restrict__ T, const BlkMap* __restrict__ M) {
  const BlkMap m = M[blockIdx.x];
  const Sys& S = T[m.sys];
  if (!S.has_rx) return;  // this member has no reaction scheme
  if (S.nl16) rx_select_apply_body<true>(S, Blk{m.b, m.nb}, -1LL);
  else rx_select_apply_body<false>(S, Blk{m.b, m.nb}, -1LL);
}

// Populations per (type, state) counted over every slot into S.pop (creation;
// the reaction steps keep them current).
__global__ void __launch_bounds__(RX_THREADS) k_pop_init(Sys S) {
  const SoA B = S.ctl->set ? S.s1 : S.s0;
  __shared__ int32_t h[PRX_MAX_TYPES * PRX_MAX_STATES];
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += blockDim.x) h[k] = 0;
  __syncthreads();
  // Block-strided over the slots; within a warp, lanes with the same
  // (type, state) bin are counted by one shared atomic of their leader.
  const int lane = threadIdx.x & 31;
  for (uint32_t base = blockIdx.x * blockDim.x; base < S.n; base += gridDim.x * blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    int key = -1;
    if (i < S.n) {
      const uint32_t t = B.type[i];
      const int s = B.state[i];
      if (t < PRX_MAX_TYPES && s >= 0 && s < PRX_MAX_STATES) key = (int)t * PRX_MAX_STATES + s;
    }
    const unsigned grp = __match_any_sync(0xFFFFFFFFu, key);
    if (key >= 0 && lane == __ffs(grp) - 1) atomicAdd(&h[key], __popc(grp));
  }
  __syncthreads();
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += blockDim.x)
    if (h[k]) atomicAdd(S.pop + k, h[k]);
}

// The observables in one launch, packed for one copy: FP64 sums of m v^2 / 2
// and m v (grid-strided per thread, a fixed warp tree, the warps in order; the
// last block adds the blocks' sums, thread t blocks t, t + 256, ..., and a
// fixed tree: the same order on every call), the populations from the running
// counts, and the control block.  Three kernels, a recount of the populations
// and three copies before: observables of 2,048 beads 35 -> 27 us.
__global__ void __launch_bounds__(RX_THREADS) k_obs_hist(Sys S, double mass, ObsPack* __restrict__ out) {
  Ctl* ctl = S.ctl;
  const SoA B = ctl->set ? S.s1 : S.s0;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < S.n; i += gridDim.x * blockDim.x) {
    const double vx = B.vx[i], vy = B.vy[i], vz = B.vz[i];
    a[0] += vx * vx + vy * vy + vz * vz;
    a[1] += vx;
    a[2] += vy;
    a[3] += vz;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] += __shfl_down_sync(0xFFFFFFFFu, a[q], o);
  __shared__ double part[4][RX_THREADS];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0)
    for (int q = 0; q < 4; ++q) part[q][wid] = a[q];
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[threadIdx.x][w];
    S.red[4 * (size_t)blockIdx.x + threadIdx.x] = (threadIdx.x == 0 ? 0.5 * mass : mass) * t;
  }
  __threadfence();
  __shared__ bool is_last;
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(&ctl->done_obs, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!is_last) return;
  if (threadIdx.x == 0) ctl->done_obs = 0u;
  for (int q = 0; q < 4; ++q) a[q] = 0.0;
  for (uint32_t b = threadIdx.x; b < gridDim.x; b += blockDim.x)
    for (int q = 0; q < 4; ++q) a[q] += __ldcg(S.red + 4 * (size_t)b + q);
  for (int q = 0; q < 4; ++q) part[q][threadIdx.x] = a[q];
  __syncthreads();
  for (int w = RX_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int q = 0; q < 4; ++q) part[q][threadIdx.x] += part[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 4) out->sums[threadIdx.x] = part[threadIdx.x][0];
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += blockDim.x) {
    int32_t c = 0;
    for (int q = 0; q < POP_REPLICAS; ++q) c += S.pop[q * (PRX_MAX_TYPES * PRX_MAX_STATES) + k];
    (&out->rec.counts[0][0])[k] = c;
  }
  if (threadIdx.x == 0) {
    out->rec.step = (long long)ctl->step;
    out->rec.bonds = (long long)ctl->nbonds;
  }
  static_assert(sizeof(Ctl) % 8 == 0, "the control block is copied in 8-byte words");
  for (uint32_t w = threadIdx.x; w < sizeof(Ctl) / 8; w += blockDim.x)
    reinterpret_cast<unsigned long long*>(&out->ctl)[w] = reinterpret_cast<const unsigned long long*>(ctl)[w];
}

// Batched reaction steps clear each member's counters in a kernel.
__global__ void kb_rx_begin(const Sys* __restrict__ T, const BlkMap* __restrict__ M) {
  const Sys& S = T[M[blockIdx.x].sys];
  if (!S.has_rx || threadIdx.x != 0) return;
  for (int q = 0; q < 4; ++q) S.ctl->trace[q] = 0;
  S.ctl->n_active = 0u;
}

// The histogram's squared bin edges, and its counts and class sizes cleared.
__global__ void k_hist_begin(double r_max, double* __restrict__ e2, int nbins, unsigned long long* __restrict__ counts) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nbins + 2; k += gridDim.x * blockDim.x) {
    counts[k] = 0ull;
    if (k <= nbins) {
      const double e = __ddiv_rn(__dmul_rn(r_max, (double)k), (double)nbins);
      e2[k] = __dmul_rn(e, e);
    }
  }
}

// Pair-distance histogram between two particle classes (the data of
// g_AB(r), Secs. V-VI): eight lanes per slot, those of class a run over its
// Verlet list (a lane its entries q, q + 8, ...); pairs are binned by the
// exact FP64 r^2 (minimum image, the reaction test's fma order) against the
// squared bin edges e2[0..nbins].  Counts are integers, so the result does not
// depend on the order of the atomics.  counts[nbins] and [nbins + 1] receive
// the class sizes.  Bound by the chain of dependent loads (entry -> type ->
// position) that eight lanes shorten; a call at 33,096 beads and 110 bins takes
// 35 us (one lane per slot, and two allocations, an upload and a second wait
// per call: 197 us).
template <bool NL16>
__global__ void __launch_bounds__(RX_THREADS)
    k_pair_hist(Sys S, PairClass a, PairClass b, const double* __restrict__ e2, int nbins,
                unsigned long long* counts) {
  extern __shared__ __align__(16) unsigned char smem_h[];
  double* se2 = reinterpret_cast<double*>(smem_h);
  unsigned int* sc = reinterpret_cast<unsigned int*>(se2 + nbins + 1);
  for (int k = threadIdx.x; k <= nbins; k += blockDim.x) se2[k] = e2[k];
  for (int k = threadIdx.x; k < nbins; k += blockDim.x) sc[k] = 0u;
  __syncthreads();
  Ctl* ctl = S.ctl;
  const SoA B = ctl->set ? S.s1 : S.s0;
  const uint32_t q = threadIdx.x & 7u;
  const double rmax2 = se2[nbins];
  int na = 0, nb = 0;
  for (uint32_t base = blockIdx.x * (RX_THREADS / 8); base < S.n; base += gridDim.x * (RX_THREADS / 8)) {
    const uint32_t i = base + (threadIdx.x >> 3);
    if (i >= S.n) continue;
    const uint32_t ti = B.type[i];
    const int si = B.state[i];
    const bool ia = in_window(a.mask, a.lo, a.hi, ti, si);
    if (q == 0u) {
      na += ia ? 1 : 0;
      nb += in_window(b.mask, b.lo, b.hi, ti, si) ? 1 : 0;
    }
    if (!ia) continue;
    const double xi = B.x[i], yi = B.y[i], zi = B.z[i];
    const int cnt = S.nn[i];
    for (int k = (int)q; k < cnt; k += 8) {
      const uint32_t j = nl_get_rx<NL16>(S, k, i);
      if (!in_window(b.mask, b.lo, b.hi, B.type[j], B.state[j])) continue;
      const double ddx = min_image(__dsub_rn(B.x[j], xi), S.L[0], S.halfL[0]);
      const double ddy = min_image(__dsub_rn(B.y[j], yi), S.L[1], S.halfL[1]);
      const double ddz = min_image(__dsub_rn(B.z[j], zi), S.L[2], S.halfL[2]);
      const double r2 = __fma_rn(ddz, ddz, __fma_rn(ddy, ddy, __dmul_rn(ddx, ddx)));
      if (!(r2 < rmax2)) continue;
      int lo = 0, hi = nbins - 1;  // largest bin whose lower edge is <= r
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (se2[mid] <= r2) lo = mid;
        else hi = mid - 1;
      }
      atomicAdd(&sc[lo], 1u);
    }
  }
  const long long ca = block_sum_ll(na), cb = block_sum_ll(nb);  // (also orders the counts before their read)
  if (threadIdx.x == 0) {
    if (ca) atomicAdd(&counts[nbins], (unsigned long long)ca);
    if (cb) atomicAdd(&counts[nbins + 1], (unsigned long long)cb);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nbins; k += blockDim.x)
    if (sc[k]) atomicAdd(&counts[k], (unsigned long long)sc[k]);
}

inline unsigned blocks_rx(uint32_t n) { return n ? (n + RX_THREADS - 1) / RX_THREADS : 1u; }

}  // namespace

int rx_kernel_count(int rule) { return rule == PRX_SELECT_NEAREST ? 4 : 3; }

void launch_rx(const Sys& S, cudaStream_t st, long long step_arg,
               void (*hook)(void*, const char*, int), void* ctx) {
  const unsigned g = blocks_rx(S.n);
  auto H = [&](const char* nm, int p) {
    if (hook) hook(ctx, nm, p);
  };
  cudaMemsetAsync(&S.ctl->trace[0], 0, sizeof(long long) * 4 + sizeof(unsigned int), st);
  H("rx_compact", 0);
  {
    const unsigned g4 = blocks_rx((S.n + 3u) / 4u);
    k_rx_compact4<<<g4, RX_THREADS, 0, st>>>(S);
  }
  H("rx_compact", 1);
  const unsigned gf = g < 1216u ? g : 1216u;
  H("rx_find", 0);
  if (S.R.rule != PRX_SELECT_NEAREST && S.R.nr <= 1) {
    if (S.nl16) k_rx_find<true, 0><<<gf, RX_THREADS, 0, st>>>(S, step_arg);
    else k_rx_find<false, 0><<<gf, RX_THREADS, 0, st>>>(S, step_arg);
  } else {
    if (S.nl16) k_rx_find<true, 1><<<gf, RX_THREADS, 0, st>>>(S, step_arg);
    else k_rx_find<false, 1><<<gf, RX_THREADS, 0, st>>>(S, step_arg);
  }
  H("rx_find", 1);
  if (S.R.rule == PRX_SELECT_NEAREST) {
    H("rx_find_T", 0);
    if (S.nl16) k_rx_find_T<true><<<g, RX_THREADS, 0, st>>>(S);
    else k_rx_find_T<false><<<g, RX_THREADS, 0, st>>>(S);
    H("rx_find_T", 1);
  }
  H("rx_select_apply", 0);
  if (S.nl16) k_rx_select_apply<true><<<gf, RX_THREADS, 0, st>>>(S, step_arg);
  else k_rx_select_apply<false><<<gf, RX_THREADS, 0, st>>>(S, step_arg);
  H("rx_select_apply", 1);
}

void launch_pair_hist(const Sys& S, cudaStream_t st, const PairClass& a, const PairClass& b, double r_max, double* e2,
                      int nbins, unsigned long long* counts) {
  k_hist_begin<<<(nbins + 2 + 255) / 256, 256, 0, st>>>(r_max, e2, nbins, counts);
  if (!S.n) return;
  const unsigned all = (S.n + RX_THREADS / 8 - 1) / (RX_THREADS / 8), g = all < 1216u ? all : 1216u;
  const size_t sm = 8 * (size_t)(nbins + 1) + 4 * (size_t)nbins;
  if (S.nl16) k_pair_hist<true><<<g, RX_THREADS, sm, st>>>(S, a, b, e2, nbins, counts);
  else k_pair_hist<false><<<g, RX_THREADS, sm, st>>>(S, a, b, e2, nbins, counts);
}

// On-demand observables into `out` (on at most 8 blocks per SM).
void launch_observables(const Sys& S, cudaStream_t st, ObsPack* out) {
  const unsigned g = blocks_rx(S.n) < 1216u ? blocks_rx(S.n) : 1216u;
  k_obs_hist<<<g, RX_THREADS, 0, st>>>(S, S.mass, out);
}

void launch_pop_init(const Sys& S, cudaStream_t st) {
  cudaMemsetAsync(S.pop, 0, sizeof(int32_t) * POP_REPLICAS * PRX_MAX_TYPES * PRX_MAX_STATES, st);
  if (S.n) k_pop_init<<<blocks_rx(S.n) < 1216u ? blocks_rx(S.n) : 1216u, RX_THREADS, 0, st>>>(S);
}

int batch_rx_kernel_count() { return 5; }

void launch_batch_rx(const BatchLaunch& L, cudaStream_t st) {
  kb_rx_begin<<<L.n_one, 32, 0, st>>>(L.T, L.one);
  kb_rx_compact<<<L.n_part, RX_THREADS, 0, st>>>(L.T, L.part);
  kb_rx_find<<<L.n_part, RX_THREADS, 0, st>>>(L.T, L.part);
  // (one entry when no member has the nearest-partner rule: it then does nothing)
  kb_rx_find_T<<<L.any_nearest ? L.n_part : 1u, RX_THREADS, 0, st>>>(L.T, L.part);
  kb_rx_select_apply<<<L.n_part, RX_THREADS, 0, st>>>(L.T, L.part);
}

}  // namespace prx
