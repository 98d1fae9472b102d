// Device functions of the reaction step that the one-phase kernels
// (rx_kernels.cu) and the persistent run kernels (engine.cu) share.
#pragma once
#include "prx_internal.cuh"

namespace prx {

namespace {

__device__ __forceinline__ bool in_window(uint32_t mask, int lo, int hi, uint32_t t, int s) {
  return ((mask >> t) & 1u) && s >= lo && s <= hi;
}

// One particle of type t moves from state s0 to s1 in the block's
// population changes (states outside 0..15 are not counted).
__device__ __forceinline__ void pop_move(int32_t* dpop, uint32_t t, int s0, int s1) {
  if (t >= PRX_MAX_TYPES) return;
  if (s0 >= 0 && s0 < PRX_MAX_STATES) atomicSub(&dpop[t * PRX_MAX_STATES + s0], 1);
  if (s1 >= 0 && s1 < PRX_MAX_STATES) atomicAdd(&dpop[t * PRX_MAX_STATES + s1], 1);
}

__device__ __forceinline__ unsigned long long key64(uint4 w) {
  return ((unsigned long long)w.x << 32) | w.y;
}

template <bool NL16>
__device__ __forceinline__ uint32_t nl_get_rx(const Sys& S, int k, uint32_t i) {
  if constexpr (NL16) return ((const uint16_t*)S.nl)[(size_t)k * S.n + i];
  else return ((const uint32_t*)S.nl)[(size_t)k * S.n + i];
}

// LAMMPS rule (Sec. IV.A): the eligible partner of the other kind (a T when
// want_T, else an A) within r_react of slot i, not bonded to it, of smallest
// exact r^2 (ties to the smaller id); `in_range` counts the pairs in range.
// The G lanes of a group share a slot, lane q its list entries q, q + G, ...:
// with RX_GROUP lanes the chain of dependent loads (entry -> position -> type)
// runs once per slot instead of once per entry.  Called by whole warps unless
// G = 1; lanes of a group without a slot pass valid = false.
constexpr int RX_GROUP = 16;
// Lanes per eligible A in the one-phase kernels.  While the groups fit the GPU
// at once, more lanes shorten the chain; beyond, the slot's own loads and draws
// of every group queue up.  us of the search with 16 / 4 / 1 lanes, nearest
// rule: 2,200 A's 14.7 / 16.9 / 34, 20,000 29.7 / 24.6 / 39, 67,000 72 / 50 / 54,
// 117,000 118 / 78 / 71; concurrent reactions: 11,000 22 / 25 / 46, 33,000 37 /
// 32 / 56, 116,000 104 / 79 / 93.  Of the selection: nearest rule (which walks no
// list), 2,200 A's 12.0 / 10.2 / 10.2, 117,000 30 / 21 / 14.3; random rule, 2,200
// 13.6 / 12.6 / 11.4, 11,000 14.3 / 13.8 / 14.0, 67,000 22 / 17.7 / 15.6.
__device__ __forceinline__ int rx_find_lanes(const RxParams& R, uint32_t nact) {
  const bool several = R.nr > 1;
  return nact <= (several ? 20000u : 5000u) ? RX_GROUP : nact <= (several ? 200000u : 90000u) ? 4 : 1;
}
__device__ __forceinline__ int rx_select_lanes(const RxParams& R, uint32_t nact) {
  return R.rule == PRX_SELECT_NEAREST || nact > 32768u ? 1 : 4;
}
template <bool NL16, int G>
__device__ __forceinline__ uint32_t nearest_partner(const Sys& S, const SoA& B, const uint4* P,
                                                    uint32_t i, bool valid, bool want_T, long long& in_range) {
  const RxParams& R = S.R;
  i = valid ? i : 0u;
  const uint4 pi = P[i];
  const double xi = B.x[i], yi = B.y[i], zi = B.z[i];
  const uint32_t nb = B.nadj[i];
  uint32_t best = NONE, bestid = 0u;
  double best_r2 = 0.0;
  const int cnt = valid ? S.nn[i] : 0;
  for (int k = (int)(threadIdx.x & (G - 1)); k < cnt; k += G) {
    const uint32_t j = nl_get_rx<NL16>(S, k, i);
    // distance prefilter first (as in the random rule's search)
    const uint4 pj = P[j];
    const float ex = __int2float_rn(pdiff(pj.x, pi.x)) * S.scale[0];
    const float ey = __int2float_rn(pdiff(pj.y, pi.y)) * S.scale[1];
    const float ez = __int2float_rn(pdiff(pj.z, pi.z)) * S.scale[2];
    if (!(fmaf(ez, ez, fmaf(ey, ey, ex * ex)) < R.rr2_pre)) continue;
    const bool ok = want_T ? in_window(R.mask_T, R.t_lo, R.t_hi, B.type[j], B.state[j])
                           : in_window(R.mask_A, R.a_lo, R.a_hi, B.type[j], B.state[j]);
    if (!ok) continue;
    const double ddx = min_image(__dsub_rn(B.x[j], xi), S.L[0], S.halfL[0]);
    const double ddy = min_image(__dsub_rn(B.y[j], yi), S.L[1], S.halfL[1]);
    const double ddz = min_image(__dsub_rn(B.z[j], zi), S.L[2], S.halfL[2]);
    const double r2 = __fma_rn(ddz, ddz, __fma_rn(ddy, ddy, __dmul_rn(ddx, ddx)));
    if (!(r2 < R.rr2)) continue;
    bool bonded = false;
    for (uint32_t b = 0; b < nb; ++b) bonded |= (B.adj[(size_t)i * S.cap + b] & SLOT_MASK) == j;
    if (bonded) continue;
    ++in_range;
    const uint32_t idj = B.id[j];
    if (best == NONE || r2 < best_r2 || (r2 == best_r2 && idj < bestid)) {
      best = j;
      best_r2 = r2;
      bestid = idj;
    }
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    const double r2 = __shfl_xor_sync(0xFFFFFFFFu, best_r2, o);
    const uint32_t id = __shfl_xor_sync(0xFFFFFFFFu, bestid, o), j = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    if (j != NONE && (best == NONE || r2 < best_r2 || (r2 == best_r2 && id < bestid))) {
      best = j;
      best_r2 = r2;
      bestid = id;
    }
  }
  return best;
}

// Table I steps 2 and 5 for one candidate pair (A = idi, T = slot j):
// retained when u < k dt Theta (Eq. 4), then the smallest selection key wins
// (ties to the smaller id).
__device__ __forceinline__ void rx_accept_and_key(const Sys& S, const SoA& B,
                                                  unsigned long long step, uint32_t idi, uint32_t j,
                                                  uint64_t p53, long long& nret, uint32_t& best,
                                                  unsigned long long& bestkey, uint32_t& bestid) {
  const uint32_t idj = B.id[j];
  const uint4 wa = keyed_draw(S.seed, step, idi, idj, TAG_ACCEPT);
  if (!u53_below(wa.x, wa.y, p53)) return;
  ++nret;
  const unsigned long long key = key64(keyed_draw(S.seed, step, idi, idj, TAG_SEL_A));
  if (best == NONE || key < bestkey || (key == bestkey && idj < bestid)) {
    best = j;
    bestkey = key;
    bestid = idj;
  }
}

// Steps 1-5 for one eligible A of a scheme of concurrent reactions: its
// candidate pairs, each with its set m of candidate reactions (A and T in the
// reaction's windows, exact FP64 r^2 below the reaction's cutoff, not
// bonded), one acceptance draw against the cumulative bounds of m, and the
// retained pair of smallest selection key.  `ch` receives the chosen pair's
// reaction.  A group of G lanes per A, as in nearest_partner.
template <bool NL16, int G>
__device__ __forceinline__ uint32_t rx_find_multi(const Sys& S, const SoA& B, const uint4* P,
                                                  unsigned long long step, uint32_t i, bool valid,
                                                  long long& ncand, long long& nret, uint32_t& ch) {
  const RxParams& R = S.R;
  i = valid ? i : 0u;
  const uint32_t elA = rx_elig_A(R, B.type[i], B.state[i]);
  const uint4 pi = P[i];
  const uint32_t idi = B.id[i];
  const uint32_t nb = B.nadj[i];
  uint32_t best = NONE, bestid = 0u;
  unsigned long long bestkey = 0ull;
  const int cnt = valid ? S.nn[i] : 0;
  for (int k = (int)(threadIdx.x & (G - 1)); k < cnt; k += G) {
    const uint32_t j = nl_get_rx<NL16>(S, k, i);
    const uint4 pj = P[j];
    const float ex = __int2float_rn(pdiff(pj.x, pi.x)) * S.scale[0];
    const float ey = __int2float_rn(pdiff(pj.y, pi.y)) * S.scale[1];
    const float ez = __int2float_rn(pdiff(pj.z, pi.z)) * S.scale[2];
    if (!(fmaf(ez, ez, fmaf(ey, ey, ex * ex)) < R.rr2_pre)) continue;  // beyond every cutoff
    const uint32_t el = elA & rx_elig_T(R, B.type[j], B.state[j]);
    if (!el) continue;
    const double ddx = min_image(__dsub_rn(B.x[j], B.x[i]), S.L[0], S.halfL[0]);
    const double ddy = min_image(__dsub_rn(B.y[j], B.y[i]), S.L[1], S.halfL[1]);
    const double ddz = min_image(__dsub_rn(B.z[j], B.z[i]), S.L[2], S.halfL[2]);
    const double r2 = __fma_rn(ddz, ddz, __fma_rn(ddy, ddy, __dmul_rn(ddx, ddx)));
    uint32_t m = 0u;
    for (int r = 0; r < R.nr; ++r)
      if (((el >> r) & 1u) && r2 < R.rr2r[r]) m |= 1u << r;
    if (!m) continue;
    bool bonded = false;
    for (uint32_t b = 0; b < nb; ++b) bonded |= (B.adj[(size_t)i * S.cap + b] & SLOT_MASK) == j;
    if (bonded) continue;
    ++ncand;
    const uint32_t idj = B.id[j];
    const uint4 wa = keyed_draw(S.seed, step, idi, idj, TAG_ACCEPT);
    const unsigned long long u53 = (((unsigned long long)wa.x << 32) | wa.y) >> 11;
    int c = -1, q = 0;
    for (int r = 0; r < R.nr && c < 0; ++r) {
      if (!((m >> r) & 1u)) continue;
      if (u53 < R.p53c[m][q]) c = r;
      ++q;
    }
    if (c < 0) continue;
    ++nret;
    const unsigned long long key = key64(keyed_draw(S.seed, step, idi, idj, TAG_SEL_A));
    if (best == NONE || key < bestkey || (key == bestkey && idj < bestid)) {
      best = j;
      bestkey = key;
      bestid = idj;
      ch = (uint32_t)c;
    }
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    const unsigned long long key = __shfl_xor_sync(0xFFFFFFFFu, bestkey, o);
    const uint32_t id = __shfl_xor_sync(0xFFFFFFFFu, bestid, o), j = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    const uint32_t c = __shfl_xor_sync(0xFFFFFFFFu, ch, o);
    if (j != NONE && (best == NONE || key < bestkey || (key == bestkey && id < bestid))) {
      best = j;
      bestkey = key;
      bestid = id;
      ch = c;
    }
  }
  return best;
}

// Steps 1-5 for the single-reaction random rule, over the work list of
// nact eligible A's (grid-stride).  An A's Verlet list holds every particle within
// the list cutoff, which includes r_react, hence every candidate.  Four lanes
// per eligible A:
// lane q of an A's group takes its list entries q, q + 4, ..., marks its
// candidates, draws for them, and keeps its retained pair of smallest
// (key, id); the group then takes the smallest of the four.  That pair is
// the unique minimum over all of the A's retained pairs, the same one the
// list walk of a single thread finds, so the choice does not depend on the
// split; four lanes per A shorten each A's chain of dependent list ->
// position -> type loads fourfold.  The loop's trip count is uniform over a
// warp (8 A's per warp and pass), so the group shuffles see every lane.
template <bool NL16>
__device__ __forceinline__ void rx_find_random4(const Sys& S, const Blk blk, const SoA& B,
                                                const uint4* P, unsigned long long step,
                                                const uint32_t* list, uint32_t nact,
                                                long long& ncand, long long& nret) {
  const RxParams& R = S.R;
  const uint32_t q = threadIdx.x & 3u;
  const uint32_t gstride = (blk.nb * blockDim.x) >> 2;
  for (uint32_t wb = (blk.b * blockDim.x + (threadIdx.x & ~31u)) >> 2; wb < nact; wb += gstride) {
    const uint32_t w = wb + ((threadIdx.x & 31u) >> 2);
    const bool valid = w < nact;
    uint32_t best = NONE, bestid = 0u;
    unsigned long long bestkey = 0ull;
    const uint32_t i = valid ? list[w] : 0u;
    if (valid) {
      const uint4 pi = P[i];
      const uint32_t idi = B.id[i];
      const uint32_t nb = B.nadj[i];
      const int cnt = S.nn[i];
      // pass 1 marks this lane's candidates (bit k / 4 for list entry k);
      // pass 2 draws for them
      unsigned long long mask = 0ull;
      for (int k0 = (int)q; k0 < cnt; k0 += 16) {
        // up to four of this lane's entries at once: their slots, then their
        // positions, then the types and states of those within the prefilter
        uint32_t jj[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) jj[u] = k0 + 4 * u < cnt ? nl_get_rx<NL16>(S, k0 + 4 * u, i) : i;
        float r2v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint4 pj = P[jj[u]];
          const float ex = __int2float_rn(pdiff(pj.x, pi.x)) * S.scale[0];
          const float ey = __int2float_rn(pdiff(pj.y, pi.y)) * S.scale[1];
          const float ez = __int2float_rn(pdiff(pj.z, pi.z)) * S.scale[2];
          r2v[u] = fmaf(ez, ez, fmaf(ey, ey, ex * ex));
        }
        uint32_t tw = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool near = k0 + 4 * u < cnt && r2v[u] < R.rr2_pre;
          if (near && in_window(R.mask_T, R.t_lo, R.t_hi, B.type[jj[u]], B.state[jj[u]])) tw |= 1u << u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (!((tw >> u) & 1u)) continue;
          const uint32_t j = jj[u];
          if (!(r2v[u] < R.rr2_in)) {  // near the cutoff: the exact FP64 test
            const double ddx = min_image(__dsub_rn(B.x[j], B.x[i]), S.L[0], S.halfL[0]);
            const double ddy = min_image(__dsub_rn(B.y[j], B.y[i]), S.L[1], S.halfL[1]);
            const double ddz = min_image(__dsub_rn(B.z[j], B.z[i]), S.L[2], S.halfL[2]);
            const double r2 = __fma_rn(ddz, ddz, __fma_rn(ddy, ddy, __dmul_rn(ddx, ddx)));
            if (!(r2 < R.rr2)) continue;
          }
          bool bonded = false;
          for (uint32_t b = 0; b < nb; ++b) bonded |= (B.adj[(size_t)i * S.cap + b] & SLOT_MASK) == j;
          if (bonded) continue;
          const int m = (k0 + 4 * u) >> 2;
          if (m < 64) {
            mask |= 1ull << m;
          } else {
            ++ncand;
            rx_accept_and_key(S, B, step, idi, j, R.p53, nret, best, bestkey, bestid);
          }
        }
      }
      while (mask) {
        const int m = __ffsll((long long)mask) - 1;
        mask &= mask - 1ull;
        ++ncand;
        rx_accept_and_key(S, B, step, idi, nl_get_rx<NL16>(S, 4 * m + (int)q, i), R.p53, nret,
                          best, bestkey, bestid);
      }
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      const unsigned long long ok = __shfl_xor_sync(0xFFFFFFFFu, bestkey, off);
      const uint32_t oid = __shfl_xor_sync(0xFFFFFFFFu, bestid, off);
      const uint32_t ob = __shfl_xor_sync(0xFFFFFFFFu, best, off);
      if (ob != NONE && (best == NONE || ok < bestkey || (ok == bestkey && oid < bestid))) {
        best = ob;
        bestkey = ok;
        bestid = oid;
      }
    }
    if (valid && q == 0u) S.win[i] = best;
  }
}

// Steps 6-7 for one eligible A (a group of G lanes, as in nearest_partner):
// the T it keeps (NONE: none), the same in every lane of the group; `winner`
// tells whether it had picked one (random rule) or its choice was mutual
// (nearest).  A lane alone takes four list entries of T at a time (independent
// loads go out together).
template <bool NL16, int G>
__device__ __forceinline__ uint32_t rx_decide(const Sys& S, const SoA& B, unsigned long long step,
                                              uint32_t i, bool valid, bool& winner) {
  const RxParams& R = S.R;
  const uint32_t T = valid ? S.win[i] : NONE;
  winner = false;
  if (R.rule == PRX_SELECT_NEAREST) {
    // LAMMPS rule: an A and the T it picked react when the T picked it too
    // and u < k dt Theta, drawn with the pair's smaller id first
    if (T == NONE || S.win[T] != i) return NONE;
    winner = true;
    const uint32_t ida = B.id[i], idt = B.id[T];
    const uint4 w = keyed_draw(S.seed, step, min(ida, idt), max(ida, idt), TAG_NEAREST);
    return u53_below(w.x, w.y, R.p53) ? T : NONE;
  }
  winner = T != NONE;
  // the other A's that picked T are in T's list
  bool lost = false;
  const int cnt = winner ? S.nn[T] : 0;
  uint32_t idi = 0u, idT = 0u;
  unsigned long long mine = 0ull;
  bool drawn = false;
  constexpr int U = G == 1 ? 4 : 1;
  for (int k = (int)(threadIdx.x & (G - 1)); k < cnt; k += G * U) {
    uint32_t aa[U], wa[U];
#pragma unroll
    for (int u = 0; u < U; ++u) aa[u] = k + u * G < cnt ? nl_get_rx<NL16>(S, k + u * G, T) : i;
#pragma unroll
    for (int u = 0; u < U; ++u) wa[u] = S.win[aa[u]];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (aa[u] == i || wa[u] != T) continue;
      if (!drawn) {
        idi = B.id[i], idT = B.id[T];
        mine = key64(keyed_draw(S.seed, step, idT, idi, TAG_SEL_T));
        drawn = true;
      }
      const uint32_t ida = B.id[aa[u]];
      const unsigned long long other = key64(keyed_draw(S.seed, step, idT, ida, TAG_SEL_T));
      lost |= other < mine || (other == mine && ida < idi);
    }
  }
  if constexpr (G > 1) {
    const unsigned any = __ballot_sync(0xFFFFFFFFu, lost);
    const unsigned group = ((1u << G) - 1u) << ((threadIdx.x & 31u) & ~(G - 1u));
    lost = (any & group) != 0u;
  }
  return winner && !lost ? T : NONE;
}

// Step 9 for the pairs (i, T) of a warp (T = NONE: none), called by the whole
// warp: both adjacency rows, the states and their populations (dpop, the
// block's changes), a record in the bond list at a place from one atomic per
// warp.  Returns whether the lane's pair survived the selection (its bond
// can still be refused by a valence limit, PRX_ECAPACITY).
__device__ __forceinline__ bool rx_form(const Sys& S, const SoA& B, unsigned long long step, uint32_t i,
                                        uint32_t T, int32_t* dpop) {
  const RxParams& R = S.R;
  Ctl* ctl = S.ctl;
  const int lane = threadIdx.x & 31;
  bool form = false;
  uint32_t na = 0, nt = 0, ch = 0;
  if (T != NONE) {
    const uint32_t ta = B.type[i], tt = B.type[T];
    // the pair's reaction sets the valence limits, increments and style
    ch = R.nr > 1 ? (uint32_t)S.wch[i] : 0u;
    const uint32_t mva = R.nr > 1 ? R.maxvalr[ch][ta] : R.maxval[ta];
    const uint32_t mvt = R.nr > 1 ? R.maxvalr[ch][tt] : R.maxval[tt];
    const uint32_t capA = mva < S.cap ? mva : S.cap;
    const uint32_t capT = mvt < S.cap ? mvt : S.cap;
    na = B.nadj[i];
    nt = B.nadj[T];
    form = na < capA && nt < capT;
    if (!form) set_status(ctl, PRX_ECAPACITY);
  }
  const unsigned bal = __ballot_sync(0xFFFFFFFFu, form);
  if (!bal) return T != NONE;
  unsigned long long first = 0ull;
  if (lane == __ffs(bal) - 1) first = atomicAdd(&ctl->nbonds, (unsigned long long)__popc(bal));
  first = __shfl_sync(0xFFFFFFFFu, first, __ffs(bal) - 1);
  if (!form) return T != NONE;
  const unsigned long long pos = first + __popc(bal & ((1u << lane) - 1u));
  if (pos >= S.bond_cap) {
    set_status(ctl, PRX_ECAPACITY);
    return true;
  }
  const uint32_t style = R.nr > 1 ? R.styler[ch] : R.style;
  const uint32_t sbit = style << 31;
  B.adj[(size_t)i * S.cap + na] = T | sbit;
  B.nadj[i] = (uint8_t)(na + 1);
  B.adj[(size_t)T * S.cap + nt] = i | sbit;
  B.nadj[T] = (uint8_t)(nt + 1);
  const int sa = B.state[i], stt = B.state[T];
  const int sa1 = (int8_t)(sa + (R.nr > 1 ? R.dAr[ch] : R.dA));
  const int st1 = (int8_t)(stt + (R.nr > 1 ? R.dTr[ch] : R.dT));
  B.state[i] = (int8_t)sa1;
  B.state[T] = (int8_t)st1;
  pop_move(dpop, B.type[i], sa, sa1);
  pop_move(dpop, B.type[T], stt, st1);
  BondRec rec;
  rec.a = B.id[i];
  rec.t = B.id[T];
  rec.step = (int64_t)step;
  rec.style = style;
  rec.reaction = ch;
  S.bonds[pos] = rec;
  return true;
}

// The reaction's record (populations, bonds, step) from the running counts,
// by one whole block after every block's changes have been added.
__device__ __forceinline__ void rx_record(const Sys& S, long long step) {
  Ctl* ctl = S.ctl;
  const unsigned long long slot = ctl->hist_count % S.hist_cap;
  HistRec* rec = &S.hist[slot];
  HistRec* latest = &S.hist[S.hist_cap + 1];
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += blockDim.x) {
    int32_t c = 0;
    for (int r = 0; r < POP_REPLICAS; ++r) c += __ldcg(S.pop + r * (PRX_MAX_TYPES * PRX_MAX_STATES) + k);
    (&rec->counts[0][0])[k] = c;
    (&latest->counts[0][0])[k] = c;
  }
  __syncthreads();  // every thread has read hist_count
  if (threadIdx.x == 0) {
    const long long nb = (long long)atomicAdd(&ctl->nbonds, 0ull);
    rec->step = latest->step = step;
    rec->bonds = latest->bonds = nb;
    ctl->hist_count += 1ull;
    ctl->reactions += 1ull;
  }
}

}  // namespace

}  // namespace prx
