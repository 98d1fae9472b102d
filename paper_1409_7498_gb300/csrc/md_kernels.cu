// MD kernels: the fused force + Langevin velocity-Verlet step, and the
// rebuild (deterministic counting sort of the slots by cell, then the Verlet
// neighbour lists from a shared-memory sweep of the neighbour cells).
//
// Step kernel, one thread per slot (FP32 force mode):
//   WCA (Sec. II.C, Eq. 15) over the Verlet list, displacements taken
//   exactly from the periodic fixed-point positions and rounded once to FP32;
//   FENE (Sec. II.C) or mirror LJ (Eq. 17) over the adjacency row; Langevin
//   random force keyed by (seed, step, id); then in FP64: v' = a v + b F (one
//   DFMA per component), x' = x + dt v' (one DFMA).  The new fixed-point
//   position comes from x' through integer operations on its binary64
//   fields, so the FP64 pipe (about 70x slower than FP32 on this part) sees
//   only the six DFMAs.
#include <mutex>
#include <type_traits>
#include <cuda_runtime.h>

#include "md_device.cuh"
#include "prx_internal.cuh"

namespace prx {

namespace {

// Last warp of a grid to finish, without a block barrier: each warp counts
// itself out of its block in shared memory, and the last warp of a block
// counts the block out of the grid.  `warps_left` is set to the block's warp
// count before the block's work starts.
// The only data the last warp reads is the rebuild flag, whose setters
// fence after setting it; warps therefore fence only once per block.
__device__ __forceinline__ bool last_warp(unsigned int* counter, unsigned int* warps_left,
                                          uint32_t nb) {
  __syncwarp();
  bool last = false;
  if ((threadIdx.x & 31) == 0) {
    if (atomicSub(warps_left, 1u) == 1u) {
      __threadfence();
      last = atomicAdd(counter, 1u) == nb - 1;
    }
  }
  return last;
}

// A particle moved more than skin/2: flag the system (and its batch).  Not a
// system whose persistent run timed out, which may have left its cell counters
// and positions in the middle of a rebuild: its lists, old or new, name slots
// below n and may be walked, but the next sort would place slots beyond n.
__device__ __forceinline__ void raise_rebuild(const Sys& S) {
  if (S.ctl->status == PRX_ETIMEOUT) return;
  atomicExch(&S.ctl->rebin_flag, 1);
  if (S.in_batch) atomicExch(&S.batch->any_rebuild, 1);
  __threadfence();
}

// End of a step, by the last thread of the system to finish: its step counter
// and buffer phase advance; for a single system the graph's rebuild condition
// is set, for a batch the last system to finish sets it for all.
__device__ __forceinline__ void step_done(const Sys& S, int ph, unsigned long long step,
                                          cudaGraphConditionalHandle cond, int use_cond) {
  Ctl* ctl = S.ctl;
  ctl->done_step = 0u;
  ctl->phase = ph ^ 1;
  ctl->step = step;
  if (!S.in_batch) {
    const int dg = ctl->dg_on;  // (loads side by side)
    const unsigned long long left = ctl->steps_left - 1ull;
    const unsigned int until = S.has_rx ? ctl->until_rx - 1u : 1u;
    const int flag = atomicAdd(&ctl->rebin_flag, 0);
    if (use_cond) cudaGraphSetConditional(cond, flag ? 1u : 0u);
    if (dg) {  // device-driven run (dg.cu): whether another step may follow at once
      ctl->steps_left = left;
      ctl->until_rx = until ? until : S.theta;
      ctl->rx_due = !until;
      ctl->hold = flag || !until || !left;
    }
  } else {
    __threadfence();
    if (atomicAdd(&S.batch->done_step, 1u) == S.n_members - 1) {
      S.batch->done_step = 0u;
      const int flag = atomicExch(&S.batch->any_rebuild, 0);
      if (flag) S.batch->rebuilds += 1ull;
      S.batch->rebuild_now = flag;  // for a device-driven run (dg.cu)
      if (use_cond) cudaGraphSetConditional(cond, flag ? 1u : 0u);
    }
  }
}
__device__ __forceinline__ void step_epilogue(const Sys& S, int ph, unsigned long long step,
                                              cudaGraphConditionalHandle cond, int use_cond,
                                              unsigned int* warps_left, uint32_t nb) {
  if (last_warp(&S.ctl->done_step, warps_left, nb)) step_done(S, ph, step, cond, use_cond);
}

// Single system: as many blocks as are resident at once (or the launch
// configuration's blocks per SM), each warp taking 32-slot chunks strided by
// the grid's warp count, so that every SM stays fully occupied to the end
// instead of running a partial last wave.  BT threads per block, with the
// register budget of 48 resident warps per SM for every BT; the block shape
// changes only the scheduling, not any particle's arithmetic.
template <bool NL16, bool FORCES_ONLY, bool CUBIC, bool CAP, int BT>
__global__ void __launch_bounds__(BT, 1536 / BT)
    k_step_nl(Sys S, cudaGraphConditionalHandle cond, int use_cond) {
  __shared__ unsigned int warps_left;
  Ctl* ctl = S.ctl;
  const int hold = ctl->hold, ph = ctl->phase;
  const unsigned long long step = ctl->step + 1ull;
  if (hold) return;  // (dg.cu; the same for every block)
  if (threadIdx.x == 0) warps_left = blockDim.x >> 5;
  __syncthreads();
  const uint4* __restrict__ P = ph ? S.P1 : S.P0;
  uint4* __restrict__ Pn = ph ? S.P0 : S.P1;
  const uint32_t W = gridDim.x * (blockDim.x >> 5);
  // one loop per SoA set (a uniform branch), so that the set's array
  // pointers are read from the kernel parameters where they are used
  // instead of occupying registers across the loop
  auto run = [&](const SoA& B) {
    for (uint32_t c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c * 32u < S.n; c += W) {
      const uint32_t i = c * 32u + (threadIdx.x & 31u);
      if (i < S.n && step_one<NL16, FORCES_ONLY, CUBIC, CAP>(S, ctl, B, P, Pn, i, step)) raise_rebuild(S);
    }
  };
  if (ctl->set) run(S.s1);
  else run(S.s0);
  if constexpr (!FORCES_ONLY) step_epilogue(S, ph, step, cond, use_cond, &warps_left, gridDim.x);
}
// The same step with four lanes per slot, for systems too small to fill the
// GPU with one thread per slot: a warp takes 8 consecutive slots; lane q of
// a slot's group sums its list entries q, q + 4, ... and bonds q, q + 4, ...;
// the four partial forces are combined by a fixed butterfly (the same order
// every step), and lanes 0-7 then integrate the 8 slots as in the one-lane
// kernel.  Four times as many warps per slot hide the dependent
// list -> position gathers that a small grid leaves exposed.  The sum order
// differs from the one-lane kernel's (FP32 rounding only).
template <bool NL16, bool FORCES_ONLY, bool CUBIC, int BT>
__global__ void __launch_bounds__(BT, 1536 / BT)
    k_step_nl4(Sys S, cudaGraphConditionalHandle cond, int use_cond) {
  __shared__ unsigned int warps_left;
  Ctl* ctl = S.ctl;
  const int hold = ctl->hold, ph = ctl->phase;
  const unsigned long long step = ctl->step + 1ull;
  if (hold) return;  // (dg.cu; the same for every block)
  if (threadIdx.x == 0) warps_left = blockDim.x >> 5;
  __syncthreads();
  const uint4* __restrict__ P = ph ? S.P1 : S.P0;
  uint4* __restrict__ Pn = ph ? S.P0 : S.P1;
  const uint32_t W = gridDim.x * (blockDim.x >> 5);
  const int lane = threadIdx.x & 31, q = lane & 3;
  auto run = [&](const SoA& B) {
    for (uint32_t c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c * 8u < S.n; c += W) {
      const uint32_t i = c * 8u + (uint32_t)(lane >> 2);
      float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f;
      uint32_t wref = 0u;
      bool ok = true;
      if (i < S.n) {
        const int cnt = __ldg(S.nn + i);
        const uint4 pi = __ldg(P + i);
        wref = pi.w;
        for (int k0 = q; k0 < cnt; k0 += 16) {
          uint32_t rn[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) rn[u] = k0 + 4 * u < cnt ? nl_raw<NL16>(S, k0 + 4 * u, i) : i;
          uint4 pj[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) pj[u] = __ldg(P + rn[u]);
#pragma unroll
          for (int u = 0; u < 4; ++u) pair32<CUBIC>(S, pj[u], pi, fx, fy, fz, e);
        }
        if constexpr (CUBIC) {
          fx *= S.scale[0];
          fy *= S.scale[0];
          fz *= S.scale[0];
        }
        const uint32_t nb = __ldg(B.nadj + i);
        for (uint32_t b = (uint32_t)q; b < nb; b += 4) {
          const uint32_t ent = __ldg(B.adj + (size_t)i * S.cap + b);
          const uint4 pj = __ldg(P + (ent & SLOT_MASK));
          float dx, dy, dz;
          disp(S, pj, pi, dx, dy, dz);
          ok = bond32(S, ent >> 31, dx, dy, dz, fx, fy, fz, e) && ok;
        }
      }
      if (!ok) set_status(ctl, PRX_EOVERSTRETCH);
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        fx += __shfl_xor_sync(0xFFFFFFFFu, fx, o);
        fy += __shfl_xor_sync(0xFFFFFFFFu, fy, o);
        fz += __shfl_xor_sync(0xFFFFFFFFu, fz, o);
        if constexpr (FORCES_ONLY) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
      }
      // lane g (< 8) takes slot c * 8 + g from the group's first lane
      const int src = (lane & 7) * 4;
      const float gx = __shfl_sync(0xFFFFFFFFu, fx, src);
      const float gy = __shfl_sync(0xFFFFFFFFu, fy, src);
      const float gz = __shfl_sync(0xFFFFFFFFu, fz, src);
      const float ge = __shfl_sync(0xFFFFFFFFu, e, src);
      const uint32_t gw = __shfl_sync(0xFFFFFFFFu, wref, src);
      const uint32_t ii = c * 8u + (uint32_t)lane;
      if (lane < 8 && ii < S.n) {
        if constexpr (FORCES_ONLY) {
          store_force(S, __ldg(B.id + ii), (double)gx, (double)gy, (double)gz, (double)ge);
        } else {
          const double xi = B.x[ii], yi = B.y[ii], zi = B.z[ii];
          const double vx = B.vx[ii], vy = B.vy[ii], vz = B.vz[ii];
          const uint32_t pid = __ldg(B.id + ii);
          if (integrate32(S, ctl, B, Pn, ii, pid, gw, step, gx, gy, gz, xi, yi, zi, vx, vy, vz)) raise_rebuild(S);
        }
      }
    }
  };
  if (ctl->set) run(S.s1);
  else run(S.s0);
  if constexpr (!FORCES_ONLY) step_epilogue(S, ph, step, cond, use_cond, &warps_left, gridDim.x);
}

// Members of a batch may differ in list width, box shape and force cap: the
// batch step runs one launch per variant present.  Like the single-system
// kernel it is a grid of the resident blocks: each takes a contiguous run of
// the variant's block map (256 slots per entry), so that it changes member
// rarely, and keeps the member's parameters in shared memory meanwhile.
// Read from the member table in global memory by one block per entry, they
// cost a load and an address at every use: 235 us per step of 256 replicas
// (3.4 M beads), 201 this way.
template <bool NL16, bool CUBIC, bool CAP>
__global__ void __launch_bounds__(256, 6)
    kb_step_nl(const Sys* __restrict__ T, const BlkMap* __restrict__ M, uint32_t n,
               cudaGraphConditionalHandle cond, int use_cond, uint32_t* act_n, BlkMap* act, uint4 act_off) {
  __shared__ int need;
  if (!act && blockIdx.x == 0 && threadIdx.x < 5) act_n[threadIdx.x] = 0u;  // for this step's rebuild plan
  __shared__ __align__(16) unsigned char sbuf[sizeof(Sys)];
  const Sys& S = *reinterpret_cast<const Sys*>(sbuf);
  static_assert(sizeof(Sys) % 8 == 0, "Sys is copied in 8-byte words");
  uint32_t e = (uint32_t)((unsigned long long)n * blockIdx.x / gridDim.x);
  const uint32_t e1 = (uint32_t)((unsigned long long)n * (blockIdx.x + 1u) / gridDim.x);
  while (e < e1) {
    const BlkMap m = M[e];
    const uint32_t cnt = min(e1 - e, m.nb - m.b);  // this member's entries of the block's run
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(T + m.sys);
    for (uint32_t w = threadIdx.x; w < sizeof(Sys) / 8; w += blockDim.x)
      reinterpret_cast<unsigned long long*>(sbuf)[w] = src[w];
    __syncthreads();
    Ctl* ctl = S.ctl;
    const int ph = ctl->phase;
    const unsigned long long step = ctl->step + 1ull;
    const SoA& B = ctl->set ? S.s1 : S.s0;
    const uint4* P = ph ? S.P1 : S.P0;
    uint4* Pn = ph ? S.P0 : S.P1;
    for (uint32_t k = 0; k < cnt; ++k) {
      const uint32_t i = (m.b + k) * 256u + threadIdx.x;
      if (i < S.n && step_one<NL16, false, CUBIC, CAP>(S, ctl, B, P, Pn, i, step)) raise_rebuild(S);
    }
    __syncthreads();  // the block's work on the member is done (and its parameters read)
    if (threadIdx.x == 0) {
      __threadfence();
      need = 0;
      if (atomicAdd(&ctl->done_step, cnt) + cnt == m.nb) {
        need = act && atomicAdd(&ctl->rebin_flag, 0) ? 1 : 0;
        if (!need) step_done(S, ph, step, cond, use_cond);
      }
    }
    __syncthreads();
    if (need) {  // the member's last block lists its blocks for the rebuild's kernels
      __shared__ uint32_t at[3];
      const uint32_t nb[3] = {m.nb, ((uint32_t)S.ncell + SCAN_TILE - 1) / SCAN_TILE, (uint32_t)(S.tiles_y * S.nc[2])};
      if (threadIdx.x == 0) {
        at[0] = act_off.x + atomicAdd(&act_n[0], nb[0]);
        atomicAdd(&act_n[1], nb[0]);
        at[1] = act_off.y + atomicAdd(&act_n[2], nb[1]);
        at[2] = act_off.z + atomicAdd(&act_n[3], nb[2]);
      }
      __syncthreads();
      for (int f = 0; f < 3; ++f)
        for (uint32_t q = threadIdx.x; q < nb[f]; q += blockDim.x) act[at[f] + q] = BlkMap{m.sys, q, nb[f], 0u};
      __syncthreads();
      if (threadIdx.x == 0) step_done(S, ph, step, cond, use_cond);
    }
    e += cnt;
    if (e < e1) __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// FP64 force mode (small systems): conservative forces per slot from the
// absolute positions over the same Verlet list, written to fout (for
// prx_compute_forces by particle, with the energies in eout); the integration runs as a second
// kernel so that no thread reads a position another thread updates.
// Arithmetic per pair in the order of the plain definitions.  FP64 issues
// at about 1/64 of the FP32 rate on this part, so the few particles of an
// FP64 system are spread over every SM: four lanes per slot (lane q takes
// the list entries and bonds q, q + 4, ...), one warp per block, and the
// four partial sums combined by a fixed butterfly (the same order every
// step).
// ---------------------------------------------------------------------------
constexpr int F64_LANES = 4;

template <bool NL16, bool ENERGY>
__global__ void __launch_bounds__(32) k_forces64(Sys S) {
  Ctl* ctl = S.ctl;
  const int hold = ctl->hold, set = ctl->set;
  if (hold) return;  // (dg.cu)
  const SoA B = set ? S.s1 : S.s0;
  const int lane = threadIdx.x & 31, q = lane & (F64_LANES - 1);
  const uint32_t i = blockIdx.x * (32 / F64_LANES) + (uint32_t)(lane / F64_LANES);
  double fx = 0.0, fy = 0.0, fz = 0.0, e = 0.0;
  bool ok = true;
  if (i < S.n) {
    const double xi = B.x[i], yi = B.y[i], zi = B.z[i];
    const int cnt = S.nn[i];
    for (int k = q; k < cnt; k += F64_LANES) {
      const uint32_t j = nl_get<NL16>(S, k, i);
      const double ddx = min_image(__dsub_rn(B.x[j], xi), S.L[0], S.halfL[0]);
      const double ddy = min_image(__dsub_rn(B.y[j], yi), S.L[1], S.halfL[1]);
      const double ddz = min_image(__dsub_rn(B.z[j], zi), S.L[2], S.halfL[2]);
      const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy)), __dmul_rn(ddz, ddz));
      if (r2 < S.rc2) wca64<ENERGY>(S, ddx, ddy, ddz, r2, fx, fy, fz, e);
    }
    const uint32_t nb = B.nadj[i];
    for (uint32_t b = (uint32_t)q; b < nb; b += F64_LANES) {
      const uint32_t ent = B.adj[(size_t)i * S.cap + b];
      const uint32_t j = ent & SLOT_MASK;
      const double ddx = min_image(__dsub_rn(B.x[j], xi), S.L[0], S.halfL[0]);
      const double ddy = min_image(__dsub_rn(B.y[j], yi), S.L[1], S.halfL[1]);
      const double ddz = min_image(__dsub_rn(B.z[j], zi), S.L[2], S.halfL[2]);
      ok = bond64<ENERGY>(S, ent >> 31, ddx, ddy, ddz, fx, fy, fz, e) && ok;
    }
  }
  if (!ok) set_status(ctl, PRX_EOVERSTRETCH);
#pragma unroll
  for (int o = 1; o < F64_LANES; o <<= 1) {
    fx = __dadd_rn(fx, __shfl_xor_sync(0xFFFFFFFFu, fx, o));
    fy = __dadd_rn(fy, __shfl_xor_sync(0xFFFFFFFFu, fy, o));
    fz = __dadd_rn(fz, __shfl_xor_sync(0xFFFFFFFFu, fz, o));
    if constexpr (ENERGY) e = __dadd_rn(e, __shfl_xor_sync(0xFFFFFFFFu, e, o));
  }
  if (q == 0 && i < S.n) {
    if constexpr (ENERGY) {
      store_force(S, B.id[i], fx, fy, fz, e);
    } else {
      S.fout[3 * (size_t)i + 0] = fx;
      S.fout[3 * (size_t)i + 1] = fy;
      S.fout[3 * (size_t)i + 2] = fz;
    }
  }
}

// FP64 integration in the oracle's order of operations:
//   F = F_c - gamma m v + R,  v' = v + (dt/m) F,  x' = x + dt v'.
__global__ void __launch_bounds__(STEP_THREADS)
    k_integrate64(Sys S, cudaGraphConditionalHandle cond, int use_cond) {
  __shared__ unsigned int warps_left;
  Ctl* ctl = S.ctl;
  const int hold = ctl->hold, set = ctl->set, ph = ctl->phase;
  const unsigned long long step = ctl->step + 1ull;
  if (hold) return;  // (dg.cu; the same for every block)
  if (threadIdx.x == 0) warps_left = blockDim.x >> 5;
  __syncthreads();
  const SoA B = set ? S.s1 : S.s0;
  const uint4* __restrict__ P = ph ? S.P1 : S.P0;
  uint4* __restrict__ Pn = ph ? S.P0 : S.P1;
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < S.n) {
    const uint32_t W = P[i].w;
    const uint32_t pid = B.id[i];
    double R[3] = {0.0, 0.0, 0.0};
    if (S.thermo) {
      const uint4 w = keyed_draw(S.seed, step, pid, 0u, TAG_THERMO);
      R[0] = __dmul_rn(S.cR, __dsub_rn(f2d_exact(u24f(w.x)), 0.5));
      R[1] = __dmul_rn(S.cR, __dsub_rn(f2d_exact(u24f(w.y)), 0.5));
      R[2] = __dmul_rn(S.cR, __dsub_rn(f2d_exact(u24f(w.z)), 0.5));
    }
    double* xs[3] = {B.x, B.y, B.z};
    double* vs[3] = {B.vx, B.vy, B.vz};
    uint32_t Xn[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double v = vs[d][i];
      const double F = __dadd_rn(__dsub_rn(S.fout[3 * (size_t)i + d], __dmul_rn(S.gm, v)), R[d]);
      const double vn = __dadd_rn(v, __dmul_rn(S.b_kick, F));
      const double xn = __dadd_rn(xs[d][i], __dmul_rn(S.dt, vn));
      if (!isfinite(vn) || !isfinite(xn)) set_status(ctl, PRX_ENONFINITE);
      vs[d][i] = vn;
      xs[d][i] = xn;
      Xn[d] = periodic_fx(xn, S.Lfx[d], S.M64[d]);
    }
    if (moved_beyond_skin(S, Xn[0], Xn[1], Xn[2], W)) raise_rebuild(S);
    Pn[i] = make_uint4(Xn[0], Xn[1], Xn[2], W);
  }
  step_epilogue(S, ph, step, cond, use_cond, &warps_left, gridDim.x);
}

// ---------------------------------------------------------------------------
// Rebuild.  Keys (wrapping x into [0, L)), counting sort with a stable
// (ascending old slot) order inside each cell, permutation of every
// per-particle array into the other SoA set with fresh fixed-point positions,
// adjacency remap, then the Verlet lists.
// ---------------------------------------------------------------------------
// Cell of every slot from the fixed-point position the last step wrote.
__device__ __forceinline__ void rebin_keys_body(const Sys& S, const Blk blk) {
  Ctl* ctl = S.ctl;
  const uint4* __restrict__ P = ctl->phase ? S.P1 : S.P0;
  const uint32_t i = blk.b * blockDim.x + threadIdx.x;
  if (i >= S.n) return;
  const uint4 q = P[i];
  const uint32_t cx = __umulhi(q.x, (uint32_t)S.nc[0]);
  const uint32_t cy = __umulhi(q.y, (uint32_t)S.nc[1]);
  const uint32_t cz = __umulhi(q.z, (uint32_t)S.nc[2]);
  const uint32_t k = (cz * (uint32_t)S.nc[1] + cy) * (uint32_t)S.nc[0] + cx;
  S.key[i] = k;
  atomicAdd(&S.count[k], 1u);
}

__global__ void k_rebin_keys(Sys S) { rebin_keys_body(S, Blk{blockIdx.x, gridDim.x}); }

// First binning of a system (no step has written fixed-point positions yet):
// cells from the FP64 positions, which are wrapped into the box in place.
__global__ void k_rebin_keys_x(Sys S) {
  Ctl* ctl = S.ctl;
  const SoA B = ctl->set ? S.s1 : S.s0;
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S.n) return;
  double* xs[3] = {B.x, B.y, B.z};
  uint32_t c[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double v0 = xs[d][i];
    const double v = wrap_into_box(v0, S.L[d]);
    if (v != v0) xs[d][i] = v;
    c[d] = __umulhi(periodic_fx(v, S.Lfx[d], S.M64[d]), (uint32_t)S.nc[d]);
  }
  const uint32_t k = (c[2] * (uint32_t)S.nc[1] + c[1]) * (uint32_t)S.nc[0] + c[0];
  S.key[i] = k;
  atomicAdd(&S.count[k], 1u);
}
__global__ void __launch_bounds__(256) kb_rebin_keys(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    rebin_keys_body(S, Blk{m.b, m.nb});
  }
}

// Restore: keys were uploaded (a checkpoint's cells); only count them.
__device__ __forceinline__ void count_keys_body(const Sys& S, const Blk blk) {
  const uint32_t i = blk.b * blockDim.x + threadIdx.x;
  if (i >= S.n) return;
  atomicAdd(&S.count[S.key[i]], 1u);
}

__global__ void k_count_keys(Sys S) { count_keys_body(S, Blk{blockIdx.x, gridDim.x}); }

// Exclusive scan of count[0..ncell) into cell_start[0..ncell], three passes.
__device__ __forceinline__ void scan_tiles_body(const Sys& S, const Blk blk) {
  __shared__ uint32_t red[256];
  const uint32_t* __restrict__ in = S.count;
  const uint32_t n = (uint32_t)S.ncell;
  const uint32_t base = blk.b * SCAN_TILE;
  uint32_t s = 0;
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    const uint32_t idx = base + k * 256 + threadIdx.x;
    if (idx < n) s += in[idx];
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) S.blk_off[blk.b] = red[0];
}
__global__ void k_scan_tiles(Sys S) { scan_tiles_body(S, Blk{blockIdx.x, gridDim.x}); }
__global__ void __launch_bounds__(256) kb_scan_tiles(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    scan_tiles_body(S, Blk{m.b, m.nb});
    __syncthreads();
  }
}

// Single block: exclusive scan of the tile sums in place.
__device__ __forceinline__ void scan_top_body(const Sys& S) {
  uint32_t* tsum = S.blk_off;
  const uint32_t ntiles = ((uint32_t)S.ncell + SCAN_TILE - 1) / SCAN_TILE;
  uint32_t carry = 0;
  for (uint32_t base = 0; base < ntiles; base += 256) {
    const uint32_t idx = base + threadIdx.x;
    const uint32_t v = idx < ntiles ? tsum[idx] : 0u;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan_256(v, total);
    if (idx < ntiles) tsum[idx] = carry + ex;
    carry += total;
  }
}
__global__ void k_scan_top(Sys S) { scan_top_body(S); }
__global__ void __launch_bounds__(256) kb_scan_top(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    scan_top_body(S);
    __syncthreads();
  }
}

__device__ __forceinline__ void scan_down_body(const Sys& S, const Blk blk) {
  const uint32_t* __restrict__ in = S.count;
  const uint32_t n = (uint32_t)S.ncell;
  uint32_t* __restrict__ out = S.cell_start;
  const uint32_t base = blk.b * SCAN_TILE + threadIdx.x * (SCAN_TILE / 256);
  uint32_t loc[SCAN_TILE / 256];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    loc[k] = (base + k < n) ? in[base + k] : 0u;
    s += loc[k];
  }
  uint32_t total;
  uint32_t run = S.blk_off[blk.b] + block_exclusive_scan_256(s, total);
  if (blk.b == 0 && threadIdx.x == 0) out[0] = 0u;
#pragma unroll
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    run += loc[k];
    if (base + k < n) out[base + k + 1] = run;
  }
}
// The same with the tile's offset summed from the tile sums by the block
// itself (no scan_top pass; for grids of at most 1,024 tiles).
__device__ __forceinline__ void scan_down_self_body(const Sys& S, const Blk blk) {
  const uint32_t* __restrict__ in = S.count;
  const uint32_t n = (uint32_t)S.ncell;
  uint32_t* __restrict__ out = S.cell_start;
  uint32_t part = 0;
  for (uint32_t t = threadIdx.x; t < blk.b; t += blockDim.x) part += S.blk_off[t];
  uint32_t off;
  (void)block_exclusive_scan_256(part, off);
  const uint32_t base = blk.b * SCAN_TILE + threadIdx.x * (SCAN_TILE / 256);
  uint32_t loc[SCAN_TILE / 256];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    loc[k] = (base + k < n) ? in[base + k] : 0u;
    s += loc[k];
  }
  uint32_t total;
  uint32_t run = off + block_exclusive_scan_256(s, total);
  if (blk.b == 0 && threadIdx.x == 0) out[0] = 0u;
#pragma unroll
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    run += loc[k];
    if (base + k < n) out[base + k + 1] = run;
  }
}
__global__ void k_scan_down(Sys S) { scan_down_body(S, Blk{blockIdx.x, gridDim.x}); }
__global__ void k_scan_down_self(Sys S) { scan_down_self_body(S, Blk{blockIdx.x, gridDim.x}); }
__global__ void __launch_bounds__(256) kb_scan_down(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    scan_down_body(S, Blk{m.b, m.nb});
    __syncthreads();
  }
}

// Cell counters of a batch's members cleared before its launch-by-launch
// rebuild.
__global__ void __launch_bounds__(256) kb_rebin_clear(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    const uint32_t c = m.b * blockDim.x + threadIdx.x;
    if (c < (uint32_t)S.ncell) {
      S.count[c] = 0u;
      S.fill[c] = 0u;
    }
  }
}

__device__ __forceinline__ void rebin_scatter_body(const Sys& S, const Blk blk) {
  const uint32_t i = blk.b * blockDim.x + threadIdx.x;
  if (i >= S.n) return;
  const uint32_t k = S.key[i];
  const uint32_t pos = atomicAdd(&S.fill[k], 1u);
  S.tmp[S.cell_start[k] + pos] = i;
}

__global__ void k_rebin_scatter(Sys S) { rebin_scatter_body(S, Blk{blockIdx.x, gridDim.x}); }
__global__ void __launch_bounds__(256) kb_rebin_scatter(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    rebin_scatter_body(S, Blk{m.b, m.nb});
  }
}

// Sorts each cell's members by old slot: the order inside a cell then does
// not depend on the order in which the scatter's atomics completed.  Then
// records every member's new slot (new_of_old), for the permutation.
__device__ __forceinline__ void cas_u32(uint32_t& a, uint32_t& b) {
  const uint32_t lo = min(a, b), hi = max(a, b);
  a = lo;
  b = hi;
}
__device__ __forceinline__ void rebin_cellsort_body(const Sys& S, const Blk blk) {
  const uint32_t c = blk.b * blockDim.x + threadIdx.x;
  if (c >= (uint32_t)S.ncell) return;
  const uint32_t s0 = S.cell_start[c], s1 = S.cell_start[c + 1];
  S.count[c] = 0u;  // for the next rebuild
  S.fill[c] = 0u;
  if (s1 - s0 <= 8u) {
    // the common case: an 8-input sorting network in registers (absent
    // members padded with the largest key)
    uint32_t v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = s0 + q < s1 ? S.tmp[s0 + q] : 0xFFFFFFFFu;
    cas_u32(v[0], v[1]); cas_u32(v[2], v[3]); cas_u32(v[4], v[5]); cas_u32(v[6], v[7]);
    cas_u32(v[0], v[2]); cas_u32(v[1], v[3]); cas_u32(v[4], v[6]); cas_u32(v[5], v[7]);
    cas_u32(v[1], v[2]); cas_u32(v[5], v[6]); cas_u32(v[0], v[4]); cas_u32(v[3], v[7]);
    cas_u32(v[1], v[5]); cas_u32(v[2], v[6]);
    cas_u32(v[1], v[4]); cas_u32(v[3], v[6]);
    cas_u32(v[2], v[4]); cas_u32(v[3], v[5]);
    cas_u32(v[3], v[4]);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (s0 + q < s1) {
        S.tmp[s0 + q] = v[q];
        S.new_of_old[v[q]] = s0 + q;
      }
    }
    return;
  }
  for (uint32_t a = s0 + 1; a < s1; ++a) {
    const uint32_t v = S.tmp[a];
    uint32_t b = a;
    while (b > s0 && S.tmp[b - 1] > v) {
      S.tmp[b] = S.tmp[b - 1];
      --b;
    }
    S.tmp[b] = v;
  }
  for (uint32_t a = s0; a < s1; ++a) S.new_of_old[S.tmp[a]] = a;
}

__global__ void k_rebin_cellsort(Sys S) { rebin_cellsort_body(S, Blk{blockIdx.x, gridDim.x}); }
__global__ void __launch_bounds__(256) kb_rebin_cellsort(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    rebin_cellsort_body(S, Blk{m.b, m.nb});
  }
}

// New slot s takes old slot tmp[s]: copies every per-particle array into the
// other set (bond partners renamed to their new slots) and writes the
// fixed-point position with a fresh displacement reference; tmp[s] then
// receives the cell the sort put the slot in (read by the list build).
__device__ __forceinline__ void rebin_permute_one(const Sys& S, uint32_t s, bool wrap) {
  Ctl* ctl = S.ctl;
  const int set = ctl->set;
  const SoA A = set ? S.s1 : S.s0;
  const SoA B = set ? S.s0 : S.s1;
  uint4* P = ctl->phase ? S.P1 : S.P0;
  const uint32_t o = S.tmp[s];
  // every load first: a store into set B could alias a later load from set A
  // as far as the compiler knows, and would hold that load back
  double x = __ldg(A.x + o), y = __ldg(A.y + o), z = __ldg(A.z + o);
  const double vx = __ldg(A.vx + o), vy = __ldg(A.vy + o), vz = __ldg(A.vz + o);
  const uint32_t pid = __ldg(A.id + o);
  const uint8_t ty = __ldg(A.type + o);
  const int8_t st = __ldg(A.state + o);
  const uint32_t nb = __ldg(A.nadj + o);
  const uint32_t key = __ldg(S.key + o);
  uint32_t e[4];  // partners renamed to their new slots (the first four at once)
#pragma unroll
  for (int b = 0; b < 4; ++b) e[b] = b < (int)nb ? __ldg(A.adj + (size_t)o * S.cap + b) : 0u;
#pragma unroll
  for (int b = 0; b < 4; ++b)
    if (b < (int)nb) e[b] = __ldg(S.new_of_old + (e[b] & SLOT_MASK)) | (e[b] & ~SLOT_MASK);
  // positions re-enter the box here (a checkpoint restore keeps them as
  // saved, so that the continued run wraps them at the same step as the
  // original run)
  if (wrap) {
    x = wrap_into_box(x, S.L[0]);
    y = wrap_into_box(y, S.L[1]);
    z = wrap_into_box(z, S.L[2]);
  }
  B.x[s] = x;
  B.y[s] = y;
  B.z[s] = z;
  B.vx[s] = vx;
  B.vy[s] = vy;
  B.vz[s] = vz;
  B.id[s] = pid;
  B.type[s] = ty;
  B.state[s] = st;
  B.nadj[s] = (uint8_t)nb;
#pragma unroll
  for (int b = 0; b < 4; ++b)
    if (b < (int)nb) B.adj[(size_t)s * S.cap + b] = e[b];
  for (uint32_t b = 4; b < nb; ++b) {
    const uint32_t f = A.adj[(size_t)o * S.cap + b];
    B.adj[(size_t)s * S.cap + b] = S.new_of_old[f & SLOT_MASK] | (f & ~SLOT_MASK);
  }
  const uint32_t X = periodic_fx(x, S.Lfx[0], S.M64[0]);
  const uint32_t Y = periodic_fx(y, S.Lfx[1], S.M64[1]);
  const uint32_t Z = periodic_fx(z, S.Lfx[2], S.M64[2]);
  P[s] = make_uint4(X, Y, Z, coarse_ref(X, Y, Z, S.wshift));
  reinterpret_cast<float4*>(S.fout)[s] = build_xyz(S, X, Y, Z, key, s);  // for the list build that follows
  S.tmp[s] = key;
}

__device__ __forceinline__ void rebin_permute_body(const Sys& S, const Blk blk, bool wrap) {
  const uint32_t s = blk.b * blockDim.x + threadIdx.x;
  if (s < S.n) rebin_permute_one(S, s, wrap);
}
// Single system: the resident blocks' warps take 32-slot chunks strided by
// the grid's warp count (no partial last wave, as in k_step_nl).
__global__ void k_rebin_permute(Sys S, int wrap) {
  const uint32_t W = gridDim.x * (blockDim.x >> 5);
  for (uint32_t c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c * 32u < S.n; c += W) {
    const uint32_t i = c * 32u + (threadIdx.x & 31u);
    if (i < S.n) rebin_permute_one(S, i, wrap != 0);
  }
}
__global__ void __launch_bounds__(256) kb_rebin_permute(const Sys* __restrict__ T, const BlkMap* __restrict__ M, const uint32_t* __restrict__ C) {
  for (uint32_t e = blockIdx.x; e < *C; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    rebin_permute_body(S, Blk{m.b, m.nb}, true);
  }
}

// ---------------------------------------------------------------------------
// Rebuild of a batch's members through buckets (all of them with at most
// BUCKET_CELLS cells that hold few particles): the keys' atomics give each
// slot's arrival rank in its cell, under which it is noted in the cell's
// bucket, or, beyond ENG_BUCKET members, linked to the cell's further ones (fill
// holds their heads, win the links; slots plus one, 0 the end); a scan of the counts gives the cells' first slots, and a slot's new
// place is its cell's first slot plus the number of the cell's members with a
// smaller old slot.  With the plan's work done by the step kernel, four
// kernels instead of ten: 256 replicas 377 -> 369 us per step.  (A single
// system keeps the seven kernels of launch_rebin: at a million beads the
// permutation by old slot, whose stores are scattered, takes 67 us instead of
// the 57 of scatter, sort and permutation.)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void keys_bucket_body(const Sys& S, const Blk blk) {
  Ctl* ctl = S.ctl;
  const uint4* P = ctl->phase ? S.P1 : S.P0;
  const uint32_t i = blk.b * blockDim.x + threadIdx.x;
  if (i >= S.n) return;
  const uint32_t k = cell_of_pos(S, P[i]);
  S.key[i] = k;
  const uint32_t rank = atomicAdd(&S.count[k], 1u);
  if (rank < ENG_BUCKET) S.bucket[(size_t)k * ENG_BUCKET + rank] = i;
  else S.win[i] = atomicExch(&S.fill[k], i + 1u);  // (win is free outside reaction steps)
}

// Scan tile blk.b with the counts before it summed by the block itself.
__device__ __forceinline__ void scan_direct_body(const Sys& S, const Blk blk) {
  const uint32_t n = (uint32_t)S.ncell, base = blk.b * SCAN_TILE;
  uint32_t part = 0, off;
#pragma unroll 16
  for (uint32_t c = threadIdx.x * 4u; c < base; c += 1024u) {
    const uint4 v = *reinterpret_cast<const uint4*>(S.count + c);
    part += v.x + v.y + v.z + v.w;
  }
  (void)block_exclusive_scan_256(part, off);
  const uint32_t c0 = base + threadIdx.x * (SCAN_TILE / 256);
  uint32_t loc[SCAN_TILE / 256];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    loc[k] = c0 + k < n ? S.count[c0 + k] : 0u;
    s += loc[k];
  }
  uint32_t total;
  uint32_t run = off + block_exclusive_scan_256(s, total);
  if (blk.b == 0 && threadIdx.x == 0) S.cell_start[0] = 0u;
#pragma unroll
  for (int k = 0; k < SCAN_TILE / 256; ++k) {
    run += loc[k];
    if (c0 + k < n) S.cell_start[c0 + k + 1] = run;
  }
}

// Old slots of block blk of 256, and the block's share of the counters back to
// zero.  In a cell with more members than a bucket holds (one in 10,000 to 100
// at four to six per cell on average) a lookup costs one load after another for
// each further member.  Counted from the keys of all slots instead, it cost the
// cell's every member and bond partner a walk over the system: two members of
// 200,000 particles, 4.3 per cell, 304 us per step; with the links 72.
__device__ __forceinline__ void permute_bucket_body(const Sys& S, const Blk blk) {
  Ctl* ctl = S.ctl;
  const SoA A = ctl->set ? S.s1 : S.s0, B = ctl->set ? S.s0 : S.s1;
  uint4* P = ctl->phase ? S.P1 : S.P0;
  auto start = [&](uint32_t k) { return S.cell_start[k]; };
  auto linked = [&](uint32_t j, uint32_t k, uint32_t first, uint32_t) {
    const uint32_t* b = S.bucket + (size_t)k * ENG_BUCKET;
    uint32_t r = first;
#pragma unroll 4
    for (uint32_t q = 0; q < ENG_BUCKET; ++q) r += b[q] < j ? 1u : 0u;
#pragma unroll 1
    for (uint32_t h = S.fill[k]; h; h = S.win[h - 1u]) r += h - 1u < j ? 1u : 0u;
    return r;
  };
  const uint32_t o = blk.b * 256u + threadIdx.x;
  if (o < S.n) permute_old<true>(S, A, B, P, S.tmp, o, start, false, linked);
  for (uint32_t c = o; c < (uint32_t)S.ncell; c += blk.nb * 256u) S.count[c] = 0u;
}

// The kernels over the members that need a rebuild.  Their blocks were listed
// by the step kernel as each member finished: act_n[0 .. 3] count the entries
// of the keys, the permutation, the scan and the list build.  A count is reset
// once its kernel is done: the keys' by the scan, the scan's by the
// permutation, the other two by the list build's last block.
__global__ void __launch_bounds__(256) kb_keys_bucket(const Sys* __restrict__ T, const BlkMap* __restrict__ M, uint32_t* act_n) {
  const uint32_t n = act_n[0];
  for (uint32_t e = blockIdx.x; e < n; e += gridDim.x) keys_bucket_body(T[M[e].sys], Blk{M[e].b, M[e].nb});
}
__global__ void __launch_bounds__(256) kb_scan_direct(const Sys* __restrict__ T, const BlkMap* __restrict__ M, uint32_t* act_n) {
  const uint32_t n = act_n[2];
  if (blockIdx.x == 0 && threadIdx.x == 0) act_n[0] = 0u;
  for (uint32_t e = blockIdx.x; e < n; e += gridDim.x) {
    scan_direct_body(T[M[e].sys], Blk{M[e].b, M[e].nb});
    __syncthreads();
  }
}
__global__ void __launch_bounds__(256, 4) kb_permute_bucket(const Sys* __restrict__ T, const BlkMap* __restrict__ M, uint32_t* act_n) {
  const uint32_t n = act_n[1];
  if (blockIdx.x == 0 && threadIdx.x == 0) act_n[2] = 0u;
  for (uint32_t e = blockIdx.x; e < n; e += gridDim.x) permute_bucket_body(T[M[e].sys], Blk{M[e].b, M[e].nb});
}

// One tile per block; the last warp of the system's tiles flips the SoA set
// and clears the flag (a warp count, not a block barrier: warps that finish
// early leave).
template <bool NL16>
__device__ __forceinline__ void build_nlist_body(const Sys& S, const Blk blk, unsigned char* smem) {
  __shared__ unsigned int warps_left;
  if (threadIdx.x == 0) warps_left = blockDim.x >> 5;
  Ctl* ctl = S.ctl;
  build_tile<NL16>(S, reinterpret_cast<const float4*>(S.fout), S.tmp, blk.b, smem);
  if (last_warp(&ctl->done_rebin, &warps_left, blk.nb)) {
    ctl->done_rebin = 0u;
    ctl->set ^= 1;
    ctl->rebin_flag = 0;
    ctl->rebins += 1ull;
  }
}

template <bool NL16>
__global__ void __launch_bounds__(256) k_build_nlist(Sys S) {
  extern __shared__ __align__(16) unsigned char smem_b[];
  build_nlist_body<NL16>(S, Blk{blockIdx.x, gridDim.x}, smem_b);
}
// (Four blocks per SM: 64 registers with 36 bytes of spills, 256 replicas 361.5 us
// per step; three blocks without spills 366.5.)
__global__ void __launch_bounds__(256, 4)
    kb_build_nlist(const Sys* __restrict__ T, const BlkMap* __restrict__ M, uint32_t* C, uint32_t* act_n) {
  extern __shared__ __align__(16) unsigned char smem_b[];
  const uint32_t n = *C;
  for (uint32_t e = blockIdx.x; e < n; e += gridDim.x) {
    const BlkMap m = M[e];
    const Sys& S = T[m.sys];
    if (act_n)  // bucket rebuilds: the links' heads back to zero
      for (uint32_t c = m.b * blockDim.x + threadIdx.x; c < (uint32_t)S.ncell; c += m.nb * blockDim.x) S.fill[c] = 0u;
    if (S.nl16) build_nlist_body<true>(S, Blk{m.b, m.nb}, smem_b);
    else build_nlist_body<false>(S, Blk{m.b, m.nb}, smem_b);
    __syncthreads();  // the buffers and the warp count are used again
  }
  // bucket rebuilds: the last block resets the counts still set (every block
  // has read C by then)
  if (act_n && threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&act_n[4], 1u) == gridDim.x - 1u) act_n[1] = act_n[3] = act_n[4] = 0u;
  }
}

inline unsigned blocks_for(uint64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Rebuild plan of a batch: the entries of the five block maps (stored one
// after the other: part, cell, tile, one, build) that belong to members
// whose rebuild flag is set, compacted into `act` at the same family offsets,
// with their counts in act_n.  The lanes of a warp that append to the same
// family reserve their places with one atomic; the order of the compacted
// entries does not matter (every block's work depends only on its entry).
__global__ void kb_rebuild_plan(const Sys* __restrict__ T, const BlkMap* __restrict__ maps,
                                uint4 off, uint32_t n_all, BlkMap* __restrict__ act,
                                uint32_t* __restrict__ act_n) {
  const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  int fam = -1;
  BlkMap m{};
  if (e < n_all) {
    m = maps[e];
    if (T[m.sys].ctl->rebin_flag)
      fam = e < off.x ? 0 : e < off.y ? 1 : e < off.z ? 2 : e < off.w ? 3 : 4;
  }
  const unsigned grp = __match_any_sync(0xFFFFFFFFu, fam);
  const int lane = threadIdx.x & 31, lead = __ffs(grp) - 1;
  uint32_t base = 0u;
  if (fam >= 0 && lane == lead) base = atomicAdd(&act_n[fam], (uint32_t)__popc(grp));
  base = __shfl_sync(0xFFFFFFFFu, base, lead);
  if (fam >= 0) {
    const uint32_t start = fam == 0 ? 0u : fam == 1 ? off.x : fam == 2 ? off.y : fam == 3 ? off.z : off.w;
    act[start + base + __popc(grp & ((1u << lane) - 1u))] = m;
  }
}

// Input staging for a plain creation (slot = particle index).  Positions are
// wrapped by at most one box edge (v >= L: v - L; v < 0: v + L, FP64), the
// same operations as the host-side restore path.
__global__ void k_stage_input(Sys S, const double* __restrict__ buf, int which) {
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S.n) return;
  const SoA& B = S.s0;
  double c[3];
  unsigned err = 0u;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double v = buf[3 * (size_t)s + k];
    if (which == 0) {
      if (!isfinite(v)) {
        err = max(err, 1u);
      } else {
        if (v >= S.L[k]) v = __dsub_rn(v, S.L[k]);
        if (v < 0.0) v = __dadd_rn(v, S.L[k]);
        if (!(v >= 0.0 && v < S.L[k])) err = max(err, 2u);
      }
    }
    c[k] = v;
  }
  if (which == 0) {
    B.x[s] = c[0];
    B.y[s] = c[1];
    B.z[s] = c[2];
    B.id[s] = s;
    if (B.type[s] >= PRX_MAX_TYPES) err = max(err, 3u);
    if (err) atomicMax(&S.ctl->input_err, err);
  } else {
    B.vx[s] = c[0];
    B.vy[s] = c[1];
    B.vz[s] = c[2];
  }
}

}  // namespace

// Read-back in particle order: slot s of the current set goes to index id[s]
// of `out` (device): 0 states (i8), 1 types (u8), 2 positions wrapped once
// into the box (the permutation's rule), [n][3], 3 velocities [n][3].
__global__ void k_gather_by_id(Sys S, int what, void* __restrict__ out) {
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S.n) return;
  const SoA B = S.ctl->set ? S.s1 : S.s0;
  const uint32_t p = B.id[s];
  if (what == 0) {
    ((int8_t*)out)[p] = B.state[s];
  } else if (what == 1) {
    ((uint8_t*)out)[p] = B.type[s];
  } else if (what == 2) {
    double* o = (double*)out + 3 * (size_t)p;
    o[0] = wrap_into_box(B.x[s], S.L[0]);
    o[1] = wrap_into_box(B.y[s], S.L[1]);
    o[2] = wrap_into_box(B.z[s], S.L[2]);
  } else {
    double* o = (double*)out + 3 * (size_t)p;
    o[0] = B.vx[s];
    o[1] = B.vy[s];
    o[2] = B.vz[s];
  }
}

void launch_gather_by_id(const Sys& S, cudaStream_t st, int what, void* out) {
  if (S.n) k_gather_by_id<<<blocks_for(S.n, 256), 256, 0, st>>>(S, what, out);
}

// Sum of the particles' energies (with the forces arranged by the kernel that
// computes them, a call at 262,144 beads takes 0.20 ms; arranged and summed on
// the host: 1.55 ms): per-block sums over a fixed assignment of
// particles, then one block adds them up, each in a fixed tree.
__global__ void __launch_bounds__(256) k_energy_sum(const double* __restrict__ v, uint32_t n, double* __restrict__ out) {
  __shared__ double part[256];
  double s = 0.0;
  for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) s += v[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = part[0];
}

const double* launch_energy_sum(const Sys& S, cudaStream_t st) {
  // (red holds four values per 256 particles and four more)
  const unsigned all = blocks_for(S.n, 256), g = all < 608u ? all : 608u;
  k_energy_sum<<<g, 256, 0, st>>>(S.eout, S.n, S.red);
  k_energy_sum<<<1, 256, 0, st>>>(S.red, g, S.red + 4 * (size_t)all);
  return S.red + 4 * (size_t)all;
}

void launch_stage_input(const Sys& S, cudaStream_t st, const double* buf, int which) {
  if (S.n) k_stage_input<<<blocks_for(S.n, 256), 256, 0, st>>>(S, buf, which);
}

// Blocks of `threads` threads of kernel `kern` resident on the whole current
// device at once (cached per device and kernel id: the step kernel's
// variants and block sizes).
// Multiprocessors of the current device (cached per device).
unsigned device_sms() {
  static unsigned cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1u;
  if (!cache[dev]) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
      cudaGetLastError();
      return 1u;
    }
    cache[dev] = (unsigned)sms;
  }
  return cache[dev];
}

unsigned resident_blocks(int variant, const void* kern, int threads) {
  static std::mutex mu;
  static unsigned cache[64][160];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1u;
  std::lock_guard<std::mutex> lk(mu);
  unsigned& c = cache[dev][variant];
  if (!c) {
    int sms = 0, per = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, 0) != cudaSuccess) {
      cudaGetLastError();
      return 1u;
    }
    c = sms * per > 0 ? (unsigned)(sms * per) : 1u;
  }
  return c;
}

void launch_step(const Sys& S, cudaStream_t st, int fp64, int forces_only,
                 cudaGraphConditionalHandle h, int use_cond) {
  if (fp64) {
    const unsigned gf = blocks_for(S.n, 32 / F64_LANES) > 0 ? blocks_for(S.n, 32 / F64_LANES) : 1;
    if (forces_only) {
      if (S.nl16) k_forces64<true, true><<<gf, 32, 0, st>>>(S);
      else k_forces64<false, true><<<gf, 32, 0, st>>>(S);
    } else {
      if (S.nl16) k_forces64<true, false><<<gf, 32, 0, st>>>(S);
      else k_forces64<false, false><<<gf, 32, 0, st>>>(S);
      const unsigned gi = blocks_for(S.n, 32) > 0 ? blocks_for(S.n, 32) : 1;
      k_integrate64<<<gi, 32, 0, st>>>(S, h, use_cond);
    }
  } else {
    // forces-only launches keep 256 threads; the step takes the launch
    // configuration's block size and blocks per SM; both take its lanes per
    // slot (so that prx_compute_forces sums as the step does)
    const int bt = forces_only ? 256 : S.step_bt;
    auto K = [&](auto nl16, auto fo, auto cub) {
      constexpr bool N16 = decltype(nl16)::value, FO = decltype(fo)::value, CU = decltype(cub)::value;
      constexpr int v = (N16 ? 4 : 0) + (FO ? 2 : 0) + (CU ? 1 : 0);
      auto go = [&](auto btc) {
        constexpr int BT = decltype(btc)::value;
        const bool four = S.step_lanes == 4;
        const bool cap = !FO && S.fcapf > 0.f;  // (the forces-only kernel tests for a cap itself)
        auto* kern = four ? k_step_nl4<N16, FO, CU, BT>
                          : (cap ? k_step_nl<N16, FO, CU, !FO, BT> : k_step_nl<N16, FO, CU, false, BT>);
        const unsigned per = four ? BT / 4 : BT;  // slots per block
        const unsigned g0 = blocks_for(S.n, per) > 0 ? blocks_for(S.n, per) : 1;
        unsigned r = resident_blocks(v + 8 * (BT == 128 ? 1 : (BT == 512 ? 2 : 0)) + (four ? 32 : 0) + (cap ? 64 : 0),
                                     (const void*)kern, BT);
        if (!FO && S.step_bpsm > 0) {
          const unsigned want = (unsigned)S.step_bpsm * (unsigned)device_sms();
          r = want < r ? want : r;
        }
        kern<<<(g0 < r ? g0 : r), BT, 0, st>>>(S, h, use_cond);
      };
      if constexpr (FO) {
        go(std::integral_constant<int, 256>{});
      } else {
        if (bt == 128) go(std::integral_constant<int, 128>{});
        else if (bt == 512) go(std::integral_constant<int, 512>{});
        else go(std::integral_constant<int, 256>{});
      }
    };
    using T_ = std::true_type;
    using F_ = std::false_type;
    if (S.cubic) {
      if (S.nl16) forces_only ? K(T_{}, T_{}, T_{}) : K(T_{}, F_{}, T_{});
      else forces_only ? K(F_{}, T_{}, T_{}) : K(F_{}, F_{}, T_{});
    } else {
      if (S.nl16) forces_only ? K(T_{}, T_{}, F_{}) : K(T_{}, F_{}, F_{});
      else forces_only ? K(F_{}, T_{}, F_{}) : K(F_{}, F_{}, F_{});
    }
  }
}

int step_kernel_count(int fp64) { return fp64 ? 2 : 1; }

size_t build_tile_smem(const Sys& S) {
  return 16 * (size_t)S.tile_cap + sizeof(BuildRow) * TILE_ROWS_MAX + 4 * (size_t)(3 * (S.tile_y + 2)) * (S.nc[0] + 1);
}

// The dynamic shared-memory limit is an attribute of the kernel (per device),
// shared by every system: it only ever grows, to the largest tile any system
// on the device has asked for, so that systems of different sizes coexist.
namespace {
std::mutex g_smem_mu;
size_t g_smem_set[2][64];  // [single, batched][device]
int raise_smem_limit(int which, size_t bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  std::lock_guard<std::mutex> lk(g_smem_mu);
  if (bytes <= g_smem_set[which][dev]) return 0;
  bool ok;
  if (which == 0) {
    ok = cudaFuncSetAttribute(k_build_nlist<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)bytes) == cudaSuccess &&
         cudaFuncSetAttribute(k_build_nlist<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)bytes) == cudaSuccess;
  } else {
    ok = cudaFuncSetAttribute(kb_build_nlist, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)bytes) == cudaSuccess;
  }
  if (!ok) return -1;
  g_smem_set[which][dev] = bytes;
  return 0;
}
}  // namespace

int configure_build_kernel(size_t smem_bytes) { return raise_smem_limit(0, smem_bytes); }

constexpr unsigned kScanSelfTiles = 1024;   // tiles up to which the scan has two passes

int rebin_kernel_count(const Sys& S) {
  return (S.ncell + SCAN_TILE - 1) / SCAN_TILE <= (int)kScanSelfTiles ? 7 : 8;
}

// Whole rebuild: keys and counts (mode 0: from the fixed-point positions of
// the last step; 1: from the FP64 positions; 2: given), scan, scatter,
// per-cell sort, permutation (with the adjacency renamed), Verlet lists.  `hook`
// (optional) is called before (0) and after (1) each launch with the
// kernel's name, for event timing.
void launch_rebin(const Sys& S, cudaStream_t st, int mode, void (*hook)(void*, const char*, int),
                  void* ctx) {
  const unsigned gp = blocks_for(S.n, 256) ? blocks_for(S.n, 256) : 1;
  const unsigned gc = blocks_for(S.ncell, 256);
  const unsigned tiles = blocks_for(S.ncell, SCAN_TILE);
  auto H = [&](const char* nm, int p) {
    if (hook) hook(ctx, nm, p);
  };
  auto build = [&] {
    const unsigned gt = (unsigned)(S.tiles_y * S.nc[2]);
    const size_t sm = build_tile_smem(S);
    H("build_nlist", 0);
    if (S.nl16) k_build_nlist<true><<<gt, S.tile_threads, sm, st>>>(S);
    else k_build_nlist<false><<<gt, S.tile_threads, sm, st>>>(S);
    H("build_nlist", 1);
  };
  H(mode == 2 ? "count_keys" : "rebin_keys", 0);
  if (mode == 2) k_count_keys<<<gp, 256, 0, st>>>(S);
  else if (mode == 1) k_rebin_keys_x<<<gp, 256, 0, st>>>(S);
  else k_rebin_keys<<<gp, 256, 0, st>>>(S);
  H(mode == 2 ? "count_keys" : "rebin_keys", 1);
  H("scan_tiles", 0);
  k_scan_tiles<<<tiles, 256, 0, st>>>(S);
  H("scan_tiles", 1);
  if (tiles <= kScanSelfTiles) {
    H("scan_down", 0);
    k_scan_down_self<<<tiles, 256, 0, st>>>(S);
    H("scan_down", 1);
  } else {
    H("scan_top", 0);
    k_scan_top<<<1, 256, 0, st>>>(S);
    H("scan_top", 1);
    H("scan_down", 0);
    k_scan_down<<<tiles, 256, 0, st>>>(S);
    H("scan_down", 1);
  }
  H("rebin_scatter", 0);
  k_rebin_scatter<<<gp, 256, 0, st>>>(S);
  H("rebin_scatter", 1);
  H("rebin_cellsort", 0);
  k_rebin_cellsort<<<gc, 256, 0, st>>>(S);
  H("rebin_cellsort", 1);
  H("rebin_permute", 0);
  {
    const unsigned r = resident_blocks(8, (const void*)k_rebin_permute, 256);
    k_rebin_permute<<<(gp < r ? gp : r), 256, 0, st>>>(S, mode != 2);
  }
  H("rebin_permute", 1);
  build();
}

void launch_batch_step(const BatchLaunch& L, cudaStream_t st, cudaGraphConditionalHandle h,
                       int use_cond) {
  auto go = [&](auto nl16, auto cub, auto cap) {
    constexpr bool N16 = decltype(nl16)::value, CU = decltype(cub)::value, CA = decltype(cap)::value;
    constexpr int v = (N16 ? 4 : 0) + (CU ? 2 : 0) + (CA ? 1 : 0);
    if (!L.step_n[v]) return;
    auto* kern = kb_step_nl<N16, CU, CA>;
    const unsigned r = resident_blocks(128 + v, (const void*)kern, 256);
    kern<<<L.step_n[v] < r ? L.step_n[v] : r, 256, 0, st>>>(
        L.T, L.part + L.step_off[v], L.step_n[v], h, use_cond, L.act_n, L.buckets ? L.act : nullptr,
        make_uint4(0u, L.n_part + L.n_cell, L.n_part + L.n_cell + L.n_tile + L.n_one, 0u));
  };
  using T_ = std::true_type;
  using F_ = std::false_type;
  go(F_{}, F_{}, F_{}), go(F_{}, F_{}, T_{}), go(F_{}, T_{}, F_{}), go(F_{}, T_{}, T_{});
  go(T_{}, F_{}, F_{}), go(T_{}, F_{}, T_{}), go(T_{}, T_{}, F_{}), go(T_{}, T_{}, T_{});
}

// The rebuild pipeline over the members whose flag is set: a plan kernel
// compacts their blocks, and each kernel's resident blocks take the entries of
// its family in turn.  (A block per entry of the full map, returning at once
// beyond the compacted count, costs ~18 us per kernel at 13,400 entries, most
// of what a rebuild of the few members that need one takes.)
//
// Where every member's cells have buckets the step kernel lists the blocks and
// four kernels follow; else the plan and nine.
void launch_batch_rebuild(const BatchLaunch& L, cudaStream_t st) {
  auto grid = [](int v, const void* k, unsigned n) {
    const unsigned r = resident_blocks(v, k, 256);
    return n < r ? n : r;
  };
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kb_build_nlist, L.build_threads, L.build_smem) != cudaSuccess ||
      per < 1) {
    cudaGetLastError();
    per = 1;
  }
  const unsigned rb = device_sms() * (unsigned)per, gb = L.n_build < rb ? L.n_build : rb;
  if (L.buckets) {
    const BlkMap *tile = L.act + L.n_part + L.n_cell, *build = tile + L.n_tile + L.n_one;
    kb_keys_bucket<<<grid(144, (const void*)kb_keys_bucket, L.n_part), 256, 0, st>>>(L.T, L.act, L.act_n);
    kb_scan_direct<<<grid(145, (const void*)kb_scan_direct, L.n_tile), 256, 0, st>>>(L.T, tile, L.act_n);
    kb_permute_bucket<<<grid(146, (const void*)kb_permute_bucket, L.n_part), 256, 0, st>>>(L.T, L.act, L.act_n);
    kb_build_nlist<<<gb, L.build_threads, L.build_smem, st>>>(L.T, build, L.act_n + 3, L.act_n);
    return;
  }
  const uint32_t o1 = L.n_part, o2 = o1 + L.n_cell, o3 = o2 + L.n_tile, o4 = o3 + L.n_one;
  const uint32_t n_all = o4 + L.n_build;
  kb_rebuild_plan<<<blocks_for(n_all, 256), 256, 0, st>>>(L.T, L.part, make_uint4(o1, o2, o3, o4), n_all,
                                                           L.act, L.act_n);
  const BlkMap *part = L.act, *cell = L.act + o1, *tile = L.act + o2, *one = L.act + o3, *build = L.act + o4;
  const uint32_t *c_part = L.act_n, *c_cell = L.act_n + 1, *c_tile = L.act_n + 2, *c_one = L.act_n + 3;
  kb_rebin_clear<<<grid(136, (const void*)kb_rebin_clear, L.n_cell), 256, 0, st>>>(L.T, cell, c_cell);
  kb_rebin_keys<<<grid(137, (const void*)kb_rebin_keys, L.n_part), 256, 0, st>>>(L.T, part, c_part);
  kb_scan_tiles<<<grid(138, (const void*)kb_scan_tiles, L.n_tile), 256, 0, st>>>(L.T, tile, c_tile);
  kb_scan_top<<<grid(139, (const void*)kb_scan_top, L.n_one), 256, 0, st>>>(L.T, one, c_one);
  kb_scan_down<<<grid(140, (const void*)kb_scan_down, L.n_tile), 256, 0, st>>>(L.T, tile, c_tile);
  kb_rebin_scatter<<<grid(141, (const void*)kb_rebin_scatter, L.n_part), 256, 0, st>>>(L.T, part, c_part);
  kb_rebin_cellsort<<<grid(142, (const void*)kb_rebin_cellsort, L.n_cell), 256, 0, st>>>(L.T, cell, c_cell);
  kb_rebin_permute<<<grid(143, (const void*)kb_rebin_permute, L.n_part), 256, 0, st>>>(L.T, part, c_part);
  kb_build_nlist<<<gb, L.build_threads, L.build_smem, st>>>(L.T, build, L.act_n + 4, nullptr);
}

int batch_rebuild_kernel_count() { return 10; }

int configure_batch_build_kernel(size_t smem_bytes) { return raise_smem_limit(1, smem_bytes); }

}  // namespace prx
