// Reaction step on caller-owned device arrays, with no device allocation.
//
// Some callers cannot call cudaMalloc at all: code that runs against a fixed
// memory budget handed out by a host framework, or inside an allocator hook
// where allocating again would re-enter the allocator.  prx_react_noalloc
// serves them: inputs and outputs are the caller's device buffers, and the
// only scratch (per-particle choices and a few counters) lives in one
// file-scope __device__ array of fixed size, held by every GPU that loads the
// library until the process exits.
//
// The candidate search is all-pairs (at most PRX_NOALLOC_MAX_N particles), so
// no cell list or neighbour list is needed: one kind of particle fits in an
// SM's shared memory as FP32 coordinates, which decide every pair that is
// clearly out of range; the few others take the exact FP64 test.  Both selection rules of
// prx_react_once are implemented with its keyed Philox draws, its FP64
// distance test and its tie-breaking, so the two agree bit for bit on the
// same state: Table I's random rule (one T per A, then one A per T, each the
// smallest selection key) and the LAMMPS nearest-partner rule of Sec. IV.A
// (mutual nearest A-T pairs, then the acceptance draw).
#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

#include "prx_internal.cuh"

namespace {

using namespace prx;

struct NaScratch {
  uint32_t win[PRX_NOALLOC_MAX_N];  // random rule: chosen T of each A (Table I step 5);
                                    // nearest rule: nearest partner of each A and T
  uint32_t fin[PRX_NOALLOC_MAX_N];  // surviving pairs (step 7), by A
  uint16_t list[PRX_NOALLOC_MAX_N]; // the A's that chose a T, in any order
  unsigned long long trace[4];
  unsigned int nbonds;
  int status;
  unsigned int nlist;
};

// The scratch.  Every call shares it and it keeps the last call's contents;
// the counters are cleared at the start of each call and win/fin are fully
// rewritten.  Calls whose work overlaps on the GPU race on it.
static __device__ __align__(256) NaScratch g_na_scratch;

struct NaArgs {
  uint32_t n, cap;
  double L[3], halfL[3];
  const double* pos;
  const uint8_t* type;
  int8_t* state;
  uint8_t* nadj;
  uint32_t* adj;
  prx_bond* bonds;
  uint32_t bonds_cap;
  uint32_t* nbonds_out;
  uint64_t seed;
  unsigned long long step;
  RxParams R;
  float Lf[3], invLf[3];
  float near2;  // FP32 r^2 from which a pair is out of range for sure (NaN: none is)
  NaScratch* sc;
};

__device__ __forceinline__ bool na_window(uint32_t mask, int lo, int hi, uint32_t t, int s) {
  return ((mask >> t) & 1u) && s >= lo && s <= hi;
}

__device__ __forceinline__ unsigned long long na_key64(uint4 w) {
  return ((unsigned long long)w.x << 32) | w.y;
}

// Exact FP64 test of Table I step 1 for the pair (i, j): the minimum-image
// separation x_j - x_i, r^2 = fma(dz, dz, fma(dy, dy, dx dx)), strict
// r^2 < r_react^2.  Returns r^2, or a negative value when out of range.
__device__ __forceinline__ double na_r2(const NaArgs& a, uint32_t i, uint32_t j, double xi,
                                        double yi, double zi) {
  const double dx = min_image(__dsub_rn(a.pos[3 * (size_t)j], xi), a.L[0], a.halfL[0]);
  const double dy = min_image(__dsub_rn(a.pos[3 * (size_t)j + 1], yi), a.L[1], a.halfL[1]);
  const double dz = min_image(__dsub_rn(a.pos[3 * (size_t)j + 2], zi), a.L[2], a.halfL[2]);
  const double r2 = __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx)));
  return r2 < a.R.rr2 ? r2 : -1.0;
}

__device__ __forceinline__ bool na_bonded(const NaArgs& a, uint32_t i, uint32_t j) {
  const uint32_t nb = a.nadj[i];
  bool bonded = false;
  for (uint32_t b = 0; b < nb; ++b) bonded |= (a.adj[(size_t)i * a.cap + b] & SLOT_MASK) == j;
  return bonded;
}

// The particles a block searches for: NA_BLOCKS blocks share them in ranges.
constexpr int NA_BLOCKS = 128, NA_THREADS = 1024, NA_WARPS = NA_THREADS / 32;
constexpr int NA_RANGE = (PRX_NOALLOC_MAX_N + NA_BLOCKS - 1) / NA_BLOCKS;
// strips of one particle per thread that a whole block takes in turn, a batch
// of them at a time
constexpr int NA_STRIPS = (PRX_NOALLOC_MAX_N + NA_THREADS - 1) / NA_THREADS, NA_BATCH = 4;
static_assert(NA_STRIPS <= 32 && NA_STRIPS % NA_BATCH == 0 && NA_BATCH % 2 == 0, "strip masks");

// binary64 -> binary32 towards zero on the integer pipe (error below 2^-23
// of the value; values below 2^-126 become 0, beyond 2^128 or not finite a
// NaN, which no later test rejects).
__device__ __forceinline__ float na_f32(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const uint32_t e = (uint32_t)(b >> 52) & 0x7FFu, sign = (uint32_t)(b >> 32) & 0x80000000u;
  if (e < 897u) return __uint_as_float(sign);
  if (e > 1150u) return __uint_as_float(0x7FC00000u);
  return __uint_as_float(sign | ((uint32_t)(b >> 29) & 0x7FFFFFu) | ((e - 896u) << 23));
}

// Steps 1-5.  Random rule: each eligible A's retained T of smallest selection
// key.  Nearest rule: each eligible A's nearest eligible T and, in a second
// pass, each eligible T's nearest eligible A (smallest exact r^2, ties to the
// smaller id).  Per pass every block stages all particles of the partner's
// kind (FP32 coordinates, 14 bytes each) and searches them for its own range
// of particles; the warps are shared out over the block's particles, so that
// a few A's among many T's still keep all of them busy.  Bound by the FP32
// instructions of the pair test (16 per pair) and the staging: a call with
// 8,192 particles, 11% of them A, takes 92 us (one thread per particle and
// FP64 tests of every pair: 11,900 us).  A coordinate more than a box edge outside the
// box sends every pair to the exact test.
__global__ void __launch_bounds__(NA_THREADS, 1) k_na_find(NaArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* sx = reinterpret_cast<float*>(smem);
  float *sy = sx + a.n, *sz = sy + a.n;
  uint16_t* sid = reinterpret_cast<uint16_t*>(sz + a.n);
  __shared__ uint16_t own[NA_RANGE];
  __shared__ unsigned long long ckey[NA_WARPS];
  __shared__ uint32_t cid[NA_WARPS];
  __shared__ uint32_t nstaged, nown;
  __shared__ int far;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool nearest = a.R.rule == PRX_SELECT_NEAREST;
  const uint32_t lo = (uint32_t)((unsigned long long)a.n * blockIdx.x / NA_BLOCKS);
  const uint32_t hi = (uint32_t)((unsigned long long)a.n * (blockIdx.x + 1u) / NA_BLOCKS);
  auto is_A = [&](uint32_t j) { return na_window(a.R.mask_A, a.R.a_lo, a.R.a_hi, a.type[j], a.state[j]); };
  auto is_T = [&](uint32_t j) { return na_window(a.R.mask_T, a.R.t_lo, a.R.t_hi, a.type[j], a.state[j]); };
  for (uint32_t i = lo + threadIdx.x; i < hi; i += NA_THREADS) a.sc->win[i] = a.sc->fin[i] = NONE;
  unsigned long long cand = 0, ret = 0;
  for (int pass = 0; pass < (nearest ? 2 : 1); ++pass) {
    __syncthreads();
    if (threadIdx.x == 0) nstaged = nown = 0u, far = 0;
    __syncthreads();
    // which of this thread's particles are of the partner's kind (types and
    // states of four strips on their way at once), then their positions, two
    // strips at a time
    uint32_t kind = 0u;
#pragma unroll 1
    for (uint32_t u = 0; u * NA_THREADS < a.n; u += NA_BATCH) {
#pragma unroll
      for (int q = 0; q < NA_BATCH; ++q) {
        const uint32_t j = (u + q) * NA_THREADS + threadIdx.x, jc = min(j, a.n - 1u);
        const bool is = pass ? is_A(jc) : is_T(jc);
        if (j < a.n && is) kind |= 1u << (u + q);
      }
    }
#pragma unroll 1
    for (uint32_t u = 0; u * NA_THREADS < a.n; u += 2) {
      const bool el[2] = {((kind >> u) & 1u) != 0u, ((kind >> (u + 1u)) & 1u) != 0u};
      double x[2][3];
      uint32_t bal[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const double* pj = a.pos + 3 * (size_t)((u + q) * NA_THREADS + threadIdx.x);
        if (el[q]) x[q][0] = pj[0], x[q][1] = pj[1], x[q][2] = pj[2];
        bal[q] = __ballot_sync(0xFFFFFFFFu, el[q]);
      }
      uint32_t at = 0u;
      if (lane == 0 && (bal[0] | bal[1])) at = atomicAdd(&nstaged, (uint32_t)(__popc(bal[0]) + __popc(bal[1])));
      at = __shfl_sync(0xFFFFFFFFu, at, 0);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (el[q]) {
          const uint32_t e = at + __popc(bal[q] & ((1u << lane) - 1u));
          sx[e] = na_f32(x[q][0]), sy[e] = na_f32(x[q][1]), sz[e] = na_f32(x[q][2]);
          sid[e] = (uint16_t)((u + q) * NA_THREADS + threadIdx.x);
          // (also true for values that are not numbers)
          if (!(fabsf(sx[e]) <= 2.f * a.Lf[0] && fabsf(sy[e]) <= 2.f * a.Lf[1] && fabsf(sz[e]) <= 2.f * a.Lf[2]))
            far = 1;
        }
        at += __popc(bal[q]);
      }
    }
    for (uint32_t i = lo + threadIdx.x; i < hi; i += NA_THREADS)
      if (pass ? is_T(i) : is_A(i)) own[atomicAdd(&nown, 1u)] = (uint16_t)i;
    __syncthreads();
    const uint32_t ns = nstaged, nq = nown;
    // W warps per particle of the block's own
    uint32_t W = NA_WARPS;
    while (W > 1u && (NA_WARPS / W) < nq) W >>= 1;
    const uint32_t groups = NA_WARPS / W, grp = (uint32_t)warp / W, part = (uint32_t)warp % W;
    for (uint32_t q0 = 0; q0 < nq; q0 += groups) {
      const bool has = q0 + grp < nq;
      const uint32_t i = has ? own[q0 + grp] : 0u;
      unsigned long long best = ~0ull;  // selection key, or the bits of r^2
      uint32_t bestid = NONE;
      if (has) {
        const double xi = a.pos[3 * (size_t)i], yi = a.pos[3 * (size_t)i + 1], zi = a.pos[3 * (size_t)i + 2];
        const float fx = na_f32(xi), fy = na_f32(yi), fz = na_f32(zi);
        const bool all = far || !(fabsf(fx) <= 2.f * a.Lf[0] && fabsf(fy) <= 2.f * a.Lf[1] && fabsf(fz) <= 2.f * a.Lf[2]);
        for (uint32_t e = part * 32u + (uint32_t)lane; e < ns; e += W * 32u) {
          // nearest image: adding and taking off 1.5 2^23 rounds to an integer
          float dx = sx[e] - fx, dy = sy[e] - fy, dz = sz[e] - fz;
          dx = fmaf(-a.Lf[0], __fsub_rn(fmaf(dx, a.invLf[0], 12582912.f), 12582912.f), dx);
          dy = fmaf(-a.Lf[1], __fsub_rn(fmaf(dy, a.invLf[1], 12582912.f), 12582912.f), dy);
          dz = fmaf(-a.Lf[2], __fsub_rn(fmaf(dz, a.invLf[2], 12582912.f), 12582912.f), dz);
          if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) >= a.near2 && !all) continue;
          const uint32_t j = sid[e];
          const double r2 = na_r2(a, i, j, xi, yi, zi);
          if (r2 < 0.0 || na_bonded(a, i, j)) continue;
          cand += pass ? 0u : 1u;
          unsigned long long key;
          if (nearest) {
            key = (unsigned long long)__double_as_longlong(r2);  // (r2 >= 0: ordered as the values)
          } else {
            const uint4 wa = keyed_draw(a.seed, a.step, i, j, TAG_ACCEPT);
            if (!u53_below(wa.x, wa.y, a.R.p53)) continue;
            ++ret;
            key = na_key64(keyed_draw(a.seed, a.step, i, j, TAG_SEL_A));
          }
          if (bestid == NONE || key < best || (key == best && j < bestid)) {
            best = key;
            bestid = j;
          }
        }
      }
      auto merge = [&](unsigned long long k2, uint32_t j2) {
        if (j2 != NONE && (bestid == NONE || k2 < best || (k2 == best && j2 < bestid))) {
          best = k2;
          bestid = j2;
        }
      };
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long k2 = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        const uint32_t j2 = __shfl_xor_sync(0xFFFFFFFFu, bestid, o);
        merge(k2, j2);
      }
      if (lane == 0) ckey[warp] = best, cid[warp] = bestid;
      __syncthreads();
      if (has && part == 0u && lane == 0) {
        for (uint32_t w = 1; w < W; ++w) merge(ckey[warp + w], cid[warp + w]);
        a.sc->win[i] = bestid;
        if (bestid != NONE && !pass) a.sc->list[atomicAdd(&a.sc->nlist, 1u)] = (uint16_t)i;
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    cand += __shfl_xor_sync(0xFFFFFFFFu, cand, o);
    ret += __shfl_xor_sync(0xFFFFFFFFu, ret, o);
  }
  if (lane == 0 && cand) atomicAdd(&a.sc->trace[0], cand);
  if (lane == 0 && ret) atomicAdd(&a.sc->trace[1], ret);
}

// Steps 6-7, one warp per A that chose a T (random rule): it keeps its T only
// if its key Philox(step, id_T, id_A) is the smallest among the A's that
// chose the same T, which are found in the list of those A's.  Nearest rule:
// an A and the T it picked react when the T picked it too and u < k dt Theta,
// drawn with the pair's smaller id first.
__global__ void __launch_bounds__(256) k_na_select(NaArgs a) {
  const int lane = threadIdx.x & 31;
  const uint32_t nl = a.sc->nlist;
  for (uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nl; w += (gridDim.x * blockDim.x) >> 5) {
    const uint32_t i = a.sc->list[w], T = a.sc->win[i];
    if (a.R.rule == PRX_SELECT_NEAREST) {
      if (lane != 0 || a.sc->win[T] != i) continue;
      atomicAdd(&a.sc->trace[1], 1ull);  // mutual pairs
      const uint4 d = keyed_draw(a.seed, a.step, min(i, T), max(i, T), TAG_NEAREST);
      if (u53_below(d.x, d.y, a.R.p53)) {
        atomicAdd(&a.sc->trace[2], 1ull);  // accepted pairs
        a.sc->fin[i] = T;
      }
      continue;
    }
    bool lost = false;
    unsigned long long mine = 0ull;
    bool drawn = false;
    for (uint32_t v = (uint32_t)lane; v < nl; v += 32u) {
      const uint32_t k = a.sc->list[v];
      if (k == i || a.sc->win[k] != T) continue;
      if (!drawn) mine = na_key64(keyed_draw(a.seed, a.step, T, i, TAG_SEL_T)), drawn = true;
      const unsigned long long other = na_key64(keyed_draw(a.seed, a.step, T, k, TAG_SEL_T));
      lost |= other < mine || (other == mine && k < i);
    }
    lost = __any_sync(0xFFFFFFFFu, lost);
    if (lane == 0) {
      atomicAdd(&a.sc->trace[2], 1ull);
      if (!lost) a.sc->fin[i] = T;
    }
  }
}

// Step 9 in one block: bonds appended in ascending id of A (counts per strip
// and warp, then their prefix sums), adjacency rows and states updated.  A pair
// that would exceed a particle's valence forms no bond and takes no place in the
// bond list (status PRX_ECAPACITY); the surviving pairs are all counted in
// the trace, as prx_react_once counts them.  Each A and each T is in at most
// one pair, so the valence reads see the rows as they were before this step.
// Bound by latency: strip by strip, each with its loads and three barriers, it
// took 23.4 us for 8,192 particles; with the loads of four strips in flight and
// one scan for them 12.7 us (all sixteen strips unrolled: 11.0, and 3 us
// more for 1,000 particles, which only fetch the longer code).
__global__ void __launch_bounds__(NA_THREADS, 1) k_na_apply(NaArgs a) {
  __shared__ uint32_t before[NA_BATCH][NA_WARPS], total[NA_BATCH], pairs[NA_WARPS];
  static_assert((PRX_MAX_TYPES & (PRX_MAX_TYPES - 1)) == 0, "a mask keeps the type in range");
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t np = 0u, carry = 0u;
#pragma unroll 1
  for (uint32_t base = 0; base < a.n; base += NA_BATCH * NA_THREADS) {
    uint32_t T[NA_BATCH];
    uint32_t bond[NA_BATCH];  // bit 31: forms; rank in the warp, the rows' lengths
#pragma unroll
    for (int u = 0; u < NA_BATCH; ++u) {
      const uint32_t i = base + u * NA_THREADS + threadIdx.x;
      T[u] = i < a.n ? a.sc->fin[i] : NONE;
    }
#pragma unroll
    for (int u = 0; u < NA_BATCH; ++u) {
      const bool pair = T[u] != NONE;
      const uint32_t i = min(base + u * NA_THREADS + threadIdx.x, a.n - 1u), j = pair ? T[u] : i;
      // (a pair's types are below 8; the others' values are not used)
      const uint32_t ta = a.type[i] & (PRX_MAX_TYPES - 1), tt = a.type[j] & (PRX_MAX_TYPES - 1);
      const uint32_t na = a.nadj[i], nt = a.nadj[j];
      const uint32_t capA = a.R.maxval[ta] < a.cap ? a.R.maxval[ta] : a.cap;
      const uint32_t capT = a.R.maxval[tt] < a.cap ? a.R.maxval[tt] : a.cap;
      const bool has = pair && na < capA && nt < capT;
      if (pair && !has) atomicCAS(&a.sc->status, 0, PRX_ECAPACITY);
      np += __popc(__ballot_sync(0xFFFFFFFFu, pair));
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, has);
      bond[u] = has ? 0x80000000u | (uint32_t)__popc(bal & ((1u << lane) - 1u)) << 16 | nt << 8 | na : 0u;
      if (lane == 0) before[u][wid] = __popc(bal);
    }
    __syncthreads();
    if (wid < NA_BATCH) {
      const uint32_t v = before[wid][lane];
      uint32_t s = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t w = __shfl_up_sync(0xFFFFFFFFu, s, o);
        if (lane >= o) s += w;
      }
      before[wid][lane] = s - v;
      if (lane == 31) total[wid] = s;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NA_BATCH; ++u) {
      if (bond[u]) {
        const uint32_t i = base + u * NA_THREADS + threadIdx.x, j = T[u];
        const uint32_t na = bond[u] & 0xFFu, nt = (bond[u] >> 8) & 0xFFu;
        const uint32_t pos = carry + before[u][wid] + ((bond[u] >> 16) & 0x7FFFu);
        if (pos >= a.bonds_cap) {
          atomicCAS(&a.sc->status, 0, PRX_ECAPACITY);
        } else {
          const uint32_t sbit = a.R.style << 31;
          a.adj[(size_t)i * a.cap + na] = j | sbit;
          a.nadj[i] = (uint8_t)(na + 1);
          a.adj[(size_t)j * a.cap + nt] = i | sbit;
          a.nadj[j] = (uint8_t)(nt + 1);
          a.state[i] = (int8_t)(a.state[i] + a.R.dA);
          a.state[j] = (int8_t)(a.state[j] + a.R.dT);
          prx_bond b;
          b.a = i;
          b.t = j;
          b.step = (int64_t)a.step;
          b.style = a.R.style;
          b.reaction = 0u;
          a.bonds[pos] = b;
        }
      }
      carry += total[u];
    }
    __syncthreads();  // (the counts' places serve the next batch)
  }
  if (lane == 0) pairs[wid] = np;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t surv = 0u;
    for (int w = 0; w < NA_WARPS; ++w) surv += pairs[w];
    const uint32_t formed = carry < a.bonds_cap ? carry : a.bonds_cap;
    a.sc->nbonds = formed;
    a.sc->trace[3] = surv;
    *a.nbonds_out = formed;
  }
}

std::mutex g_na_mutex;
NaScratch* g_na_addr[256];
bool g_na_ready[256];

// Device address of the scratch on the current device.  The first call on a
// device looks it up (with that device current); later calls reuse it.
int na_scratch(NaScratch** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return PRX_ECUDA;
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_ready[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || !p) return PRX_ECUDA;
    if (cudaFuncSetAttribute(k_na_find, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             PRX_NOALLOC_MAX_N * (3 * (int)sizeof(float) + (int)sizeof(uint16_t))) != cudaSuccess)
      return PRX_ECUDA;
    g_na_addr[dev] = static_cast<NaScratch*>(p);
    g_na_ready[dev] = true;
  }
  *out = g_na_addr[dev];
  return PRX_OK;
}

}  // namespace

extern "C" int prx_react_noalloc(const prx_reaction_desc* rx, const double* box, double dt,
                                 uint64_t seed, uint64_t step, uint32_t n, const double* d_pos,
                                 const uint8_t* d_type, int8_t* d_state, uint32_t adj_cap,
                                 uint8_t* d_nadj, uint32_t* d_adj, prx_bond* d_bonds_out,
                                 uint32_t bonds_cap, uint32_t* d_nbonds_out, void* cuda_stream,
                                 prx_rx_trace* trace) {
  if (n > PRX_NOALLOC_MAX_N) return PRX_ECAPACITY;  // beyond the static scratch
  if (!rx || !box || !d_nbonds_out || !(dt > 0.0)) return PRX_EINVAL;
  if (adj_cap < 1 || adj_cap > PRX_MAX_ADJ) return PRX_EINVAL;
  if (n && (!d_pos || !d_type || !d_state || !d_nadj || !d_adj || (bonds_cap && !d_bonds_out)))
    return PRX_EINVAL;
  if (rx->a_lo > rx->a_hi || rx->t_lo > rx->t_hi || rx->theta < 1 || !(rx->k >= 0.0) ||
      !(rx->r_react > 0.0) || (rx->bond_style != PRX_BOND_FENE && rx->bond_style != PRX_BOND_MIRROR_LJ) ||
      ((rx->type_mask_A | rx->type_mask_T) >> PRX_MAX_TYPES) ||
      (rx->selection != PRX_SELECT_RANDOM && rx->selection != PRX_SELECT_NEAREST) ||
      ((rx->type_mask_A & rx->type_mask_T) && !(rx->a_hi < rx->t_lo || rx->t_hi < rx->a_lo)))
    return PRX_EINVAL;
  for (int k = 0; k < 3; ++k)
    if (!(box[k] > 0.0)) return PRX_EINVAL;
  NaScratch* sc = nullptr;
  int rc = na_scratch(&sc);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;

  NaArgs a;
  a.R = RxParams{};
  a.R.nr = 1;
  a.n = n;
  a.cap = adj_cap;
  for (int k = 0; k < 3; ++k) {
    a.L[k] = box[k];
    a.halfL[k] = 0.5 * box[k];
  }
  a.pos = d_pos;
  a.type = d_type;
  a.state = d_state;
  a.nadj = d_nadj;
  a.adj = d_adj;
  a.bonds = d_bonds_out;
  a.bonds_cap = bonds_cap;
  a.nbonds_out = d_nbonds_out;
  a.seed = seed;
  a.step = step;
  a.R.mask_A = rx->type_mask_A;
  a.R.mask_T = rx->type_mask_T;
  a.R.a_lo = rx->a_lo;
  a.R.a_hi = rx->a_hi;
  a.R.t_lo = rx->t_lo;
  a.R.t_hi = rx->t_hi;
  a.R.dA = rx->dA;
  a.R.dT = rx->dT;
  a.R.p = rx->k * dt * (double)rx->theta;
  a.R.p53 = p53_of(a.R.p);
  a.R.rr2 = rx->r_react * rx->r_react;
  a.R.rr2_pre = 0.f;
  a.R.style = (uint32_t)rx->bond_style;
  a.R.rule = rx->selection;
  for (int t = 0; t < PRX_MAX_TYPES; ++t) a.R.maxval[t] = rx->max_valence[t];
  a.sc = sc;
  // bound on the FP32 search's distances for coordinates within two box edges
  // of the origin: 2^-23 of the value lost in each conversion, three roundings
  // of at most 2 L each: below 2e-6 L per distance
  const double Lmax = std::fmax(box[0], std::fmax(box[1], box[2]));
  const double reach = rx->r_react * (1.0 + 1e-5) + 4e-6 * Lmax;
  a.near2 = (float)(reach * reach * (1.0 + 1e-5));
  // beyond these lengths a square leaves the FP32 range at either end: a bound
  // that no distance is beyond sends every pair to the exact test
  if (!(Lmax < 1e18 && reach > 1e-18)) a.near2 = NAN;
  for (int k = 0; k < 3; ++k) {
    a.Lf[k] = (float)box[k];
    a.invLf[k] = (float)(1.0 / box[k]);
  }

  // counters and status start at zero on every call
  struct Result {
    unsigned long long trace[4];
    unsigned int nbonds;
    int status;
    unsigned int nlist;
  } got;
  if (cudaMemsetAsync(&sc->trace[0], 0, offsetof(Result, nlist) + sizeof(got.nlist), st) != cudaSuccess)
    return PRX_ECUDA;
  k_na_find<<<NA_BLOCKS, NA_THREADS, (size_t)n * (3 * sizeof(float) + sizeof(uint16_t)), st>>>(a);
  k_na_select<<<NA_BLOCKS, 256, 0, st>>>(a);
  k_na_apply<<<1, NA_THREADS, 0, st>>>(a);
  if (cudaGetLastError() != cudaSuccess) return PRX_ECUDA;
  if (cudaMemcpyAsync(&got, &sc->trace[0], sizeof(got), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return PRX_ECUDA;
  const unsigned long long* tr = got.trace;
  const int status = got.status;
  if (trace) {
    trace->candidates = (int64_t)tr[0];
    trace->retained = (int64_t)tr[1];
    trace->a_winners = (int64_t)tr[2];
    trace->formed = (int64_t)tr[3];
  }
  return status;
}
