// Persistent run kernels: many MD steps of a system in one cooperative launch.
//
// A run of the one-phase kernels is a chain of launches (step, then the
// rebuild's seven and the reaction's three when they are due), and for a
// system of some ten thousand particles that chain costs more than the work:
// 20 us per step, of which a few are the step itself.  Here the blocks of one
// grid, all resident, keep the system for the whole launch.  Each phase (the
// step; keys, scan, scatter, permutation and lists of a rebuild; search and
// selection of a reaction step) is spread over the grid's blocks and ends
// at a barrier of the grid, which also carries the "a particle moved more
// than skin/2" flag, so that a step costs one barrier.
//
// The phases do the arithmetic of the one-phase kernels in the same order
// per particle (the same device functions, the same slot and list order), so
// a run gives the same bits whichever kernels it goes through.
//
// Everything that a phase reads was written by an earlier phase of the same
// launch: plain loads only (no ld.global.nc), which the barrier's fences
// order.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "md_device.cuh"
#include "prx_internal.cuh"
#include "rx_device.cuh"

namespace prx {

namespace {

constexpr int ENG_THREADS = 512;
constexpr unsigned ENG_F64_MAX = 16384;  // particles of a persistent FP64 run
constexpr int ENG_UNITS = 1024;  // (slot, layer) pairs per tile of the list build

// Barrier of the grid's `nb` blocks.  Two words, used in turn: the low
// half counts arrivals, the high half the blocks that raised the flag.  A
// block reaches the word's next use only after every block has left the
// other word's barrier, hence this one, so a count beyond the target cannot
// be seen.  The words start a launch at zero.
//
// The arrival releases at GPU scope and every poll acquires, so that the wait
// ends with the load that sees the target: 8.95 -> 8.52 us per step (33,096
// beads), against relaxed polls with a fence after them (a second round trip),
// whether that fence is __threadfence or fence.acq_rel.
struct GridBar {
  unsigned long long* w;
  int* res;  // shared: thread 0's verdict for the block
  uint32_t nb, e, flags0, flags1;
  uint32_t polls;  // of a barrier before it gives up

  // Waits for the whole grid; 1 when a thread of any block raised `f`, 0
  // when none did, 2 when the wait ran out.
  __device__ __forceinline__ int sync(bool f) {
    const int any = __syncthreads_or(f);
    if (threadIdx.x == 0) {
      unsigned long long* p = w + (e & 1u) * 16u;
      asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(any ? 0x100000001ull : 1ull) : "memory");
      const uint32_t target = (e / 2u + 1u) * nb;
      unsigned long long v;
      unsigned left = polls;
      do {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
      } while ((uint32_t)v != target && --left);
      const uint32_t fl = (uint32_t)(v >> 32);
      const uint32_t before = (e & 1u) ? flags1 : flags0;
      *res = left ? (fl != before ? 1 : 0) : 2;
      if (e & 1u) flags1 = fl;
      else flags0 = fl;
    }
    ++e;
    __syncthreads();
    return *res;
  }
};

template <bool NL16>
__device__ __forceinline__ uint32_t nl_plain(const Sys& S, int k, uint32_t i) {
  if constexpr (NL16) return ((const uint16_t*)S.nl)[(size_t)k * S.n + i];
  else return ((const uint32_t*)S.nl)[(size_t)k * S.n + i];
}

// A slot that a thread keeps in registers from step to step: everything a step
// reads but its neighbours' positions.
struct Resident {
  double x, y, z, vx, vy, vz;
  uint4 p;
  uint32_t pid, nb, e0, e1;
  int cnt;
};
// Its list is in shared memory up to RES_LIST entries ([entry][thread]), and
// so are the neighbours' positions of a step.
constexpr int RES_LIST = 16;
constexpr size_t RES_SMEM = (size_t)RES_LIST * ENG_THREADS * (4 + 16);

__device__ __forceinline__ uint32_t* res_list(unsigned char* smem) { return reinterpret_cast<uint32_t*>(smem); }
__device__ __forceinline__ uint4* res_pos(unsigned char* smem) {
  return reinterpret_cast<uint4*>(smem + (size_t)RES_LIST * ENG_THREADS * 4);
}

__device__ __forceinline__ void res_load_bonds(const Sys& S, const SoA& B, uint32_t i, Resident& r) {
  const uint32_t* arow = B.adj + (size_t)i * S.cap;
  r.nb = B.nadj[i];
  r.e0 = arow[0];
  r.e1 = S.cap > 1 ? arow[1] : i;
}

template <bool NL16>
__device__ __forceinline__ void res_load(const Sys& S, const SoA& B, const uint4* P, uint32_t i, Resident& r,
                                         unsigned char* smem) {
  r.cnt = S.nn[i];
  r.p = P[i];
  r.x = B.x[i], r.y = B.y[i], r.z = B.z[i];
  r.vx = B.vx[i], r.vy = B.vy[i], r.vz = B.vz[i];
  r.pid = B.id[i];
  res_load_bonds(S, B, i, r);
  uint32_t* sl = res_list(smem) + threadIdx.x;
  uint32_t l[RES_LIST];
#pragma unroll
  for (int u = 0; u < RES_LIST; ++u) l[u] = nl_plain<NL16>(S, u, i);
  // (entries past the list's last whole four are never read)
#pragma unroll
  for (int u = 0; u < RES_LIST; ++u) sl[u * ENG_THREADS] = l[u];
}

__device__ __forceinline__ void res_store_x(const SoA& B, uint32_t i, const Resident& r) {
  B.x[i] = r.x, B.y[i] = r.y, B.z[i] = r.z;
}
__device__ __forceinline__ void res_store_v(const SoA& B, uint32_t i, const Resident& r) {
  B.vx[i] = r.vx, B.vy[i] = r.vy, B.vz[i] = r.vz;
}

// 16-byte copy global -> shared through L1 that does not wait for the data.
__device__ __forceinline__ void cp_async16_ca(void* smem_dst, const void* gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}

// One FP32 step of a resident slot: every neighbour position is on its way
// into shared memory before the first is used (one round trip per step,
// overlapped with the random force), then the arithmetic of step_one.
template <bool NL16, bool CUBIC>
__device__ __forceinline__ bool res_step(const Sys& S, Ctl* ctl, const SoA& B, const uint4* P, uint4* Pn, uint32_t i,
                                         unsigned long long step, Resident& r, unsigned char* smem) {
  const uint4 pi = r.p;
  const uint32_t n1 = S.n - 1u;
  const uint32_t* sl = res_list(smem) + threadIdx.x;
  uint4* sp = res_pos(smem) + threadIdx.x;
  const int near = min(r.cnt, RES_LIST);
#pragma unroll 1
  for (int k = 0; k < near; k += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) cp_async16_ca(sp + (k + u) * ENG_THREADS, P + sl[(k + u) * ENG_THREADS]);
  }
  uint4 p0 = pi, p1 = pi;
  if (r.nb > 0u) p0 = P[min(r.e0 & SLOT_MASK, n1)];
  if (r.nb > 1u) p1 = P[min(r.e1 & SLOT_MASK, n1)];
  const float3 R = random_force(S, step, r.pid);
  float fx = 0.f, fy = 0.f, fz = 0.f;
  cp_async_wait_all();
#pragma unroll 1
  for (int k = 0; k < near; k += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) pair32_flat<CUBIC>(S, sp[(k + u) * ENG_THREADS], pi, fx, fy, fz);
  }
#pragma unroll 1
  for (int k = RES_LIST; k < r.cnt; ++k) pair32_flat<CUBIC>(S, P[nl_plain<NL16>(S, k, i)], pi, fx, fy, fz);
  if constexpr (CUBIC) {
    fx *= S.scale[0];
    fy *= S.scale[0];
    fz *= S.scale[0];
  }
  bool ok = true;
  float e = 0.f;
  const uint32_t* arow = B.adj + (size_t)i * S.cap;
#pragma unroll 1
  for (uint32_t b = 0; b < r.nb; ++b) {
    const uint32_t a = b == 0u ? r.e0 : b == 1u ? r.e1 : arow[b];
    const uint4 q = b == 0u ? p0 : b == 1u ? p1 : P[a & SLOT_MASK];
    float dx, dy, dz;
    disp(S, q, pi, dx, dy, dz);
    ok = bond32(S, a >> 31, dx, dy, dz, fx, fy, fz, e) && ok;
  }
  if (!ok) set_status(ctl, PRX_EOVERSTRETCH);
  const bool moved = kick_drift32(S, ctl, pi.w, fx, fy, fz, R, r.x, r.y, r.z, r.vx, r.vy, r.vz, r.p);
  Pn[i] = r.p;
  return moved;
}

// min_image with the tests on the integer pipe (a 64-bit compare of the
// magnitudes' bit patterns has the outcome of the FP64 compare): the FP64
// pipe, which an SM of this part has two lanes of, sees only the rare shift.
__device__ __forceinline__ double min_image_int(double d, double L, double half) {
  const long long b = __double_as_longlong(d);
  if ((b & 0x7FFFFFFFFFFFFFFFll) > __double_as_longlong(half)) d = b < 0 ? __dadd_rn(d, L) : __dsub_rn(d, L);
  return d;
}

// Displacement x_j - x_i and its square in k_forces64's order.
__device__ __forceinline__ double eng_sep64(const Sys& S, double* const x[3], uint32_t j, const double xi[3],
                                            double d[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] = min_image_int(__dsub_rn(x[c][j], xi[c]), S.L[c], S.halfL[c]);
  return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}

// One FP64 step of the 4 slots of warp chunk c, eight lanes per slot: an SM
// issues an FP64 instruction of a warp over ~20 cycles, so a step is bound by
// the length of each warp's FP64 chain; eight lanes halve k_forces64's.  The
// sums keep its order: its lane p adds entries p, p + 4, p + 8, ... in turn,
// which here are lane p's and lane p + 4's terms alternately (a pair out of
// range gives the term 0, and f - 0 = f).  Lanes 0..2 of a slot then
// integrate one component each (k_integrate64's arithmetic), from the
// positions x to xn.
template <bool NL16>
__device__ __forceinline__ bool eng_step64(const Sys& S, Ctl* ctl, const SoA& B, double* const x[3],
                                           double* const xn[3], const uint4* P, uint4* Pn, uint32_t c,
                                           unsigned long long step) {
  const int lane = threadIdx.x & 31, q = lane & 7;
  const uint32_t i0 = c * 4u + (uint32_t)(lane >> 3);
  const bool act = i0 < S.n;
  const uint32_t i = act ? i0 : S.n - 1u;
  double f[3] = {0.0, 0.0, 0.0}, e = 0.0;
  double xi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) xi[d] = x[d][i];
  const int cnt = S.nn[i];
  const uint32_t nb = B.nadj[i];
  const uint32_t ent = B.adj[(size_t)i * S.cap + min((uint32_t)q, S.cap - 1u)];
  const uint32_t W = P[i].w, pid = B.id[i];
  const double v = q == 0 ? B.vx[i] : q == 1 ? B.vy[i] : B.vz[i];
  bool ok = true;
  // adds the lanes' terms t in the order of k_forces64's lanes
  auto add = [&](const double t[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double u = __shfl_down_sync(0xFFFFFFFFu, t[d], 4, 8);
      f[d] = __dsub_rn(__dsub_rn(f[d], t[d]), u);
    }
  };
  const int most = (int)__reduce_max_sync(0xFFFFFFFFu, (unsigned)cnt);
  uint32_t j = q < cnt ? nl_plain<NL16>(S, q, i) : i;
#pragma unroll 1
  for (int k = q; k - q < most; k += 8) {
    const uint32_t jn = k + 8 < cnt ? nl_plain<NL16>(S, k + 8, i) : i;
    double d[3], t[3] = {0.0, 0.0, 0.0};
    const double r2 = eng_sep64(S, x, j, xi, d);
    // (r2 >= 0: the bit patterns compare as the values do)
    if (k < cnt && __double_as_longlong(r2) < __double_as_longlong(S.rc2)) {
      double g[3] = {0.0, 0.0, 0.0};
      wca64<false>(S, d[0], d[1], d[2], r2, g[0], g[1], g[2], e);
#pragma unroll
      for (int a = 0; a < 3; ++a) t[a] = -g[a];
    }
    add(t);
    j = jn;
  }
  if (__any_sync(0xFFFFFFFFu, nb > 0u)) {
    double t[3] = {0.0, 0.0, 0.0};
    if ((uint32_t)q < nb) {
      double d[3], g[3] = {0.0, 0.0, 0.0};
      (void)eng_sep64(S, x, ent & SLOT_MASK, xi, d);
      ok = bond64<false>(S, ent >> 31, d[0], d[1], d[2], g[0], g[1], g[2], e);
#pragma unroll
      for (int a = 0; a < 3; ++a) t[a] = -g[a];
    }
    add(t);
  }
  if (!ok) set_status(ctl, PRX_EOVERSTRETCH);
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
    for (int d = 0; d < 3; ++d) f[d] = __dadd_rn(f[d], __shfl_xor_sync(0xFFFFFFFFu, f[d], o));
  }
  // lanes 0..2: component q
  double R = 0.0;
  if (S.thermo) {
    const uint4 w = keyed_draw(S.seed, step, pid, 0u, TAG_THERMO);
    R = __dmul_rn(S.cR, __dsub_rn(f2d_exact(u24f(q == 0 ? w.x : q == 1 ? w.y : w.z)), 0.5));
  }
  const int a = min(q, 2);
  const double fc = q == 0 ? f[0] : q == 1 ? f[1] : f[2];
  const double F = __dadd_rn(__dsub_rn(fc, __dmul_rn(S.gm, v)), R);
  const double vn = __dadd_rn(v, __dmul_rn(S.b_kick, F));
  const double p = __dadd_rn(q == 0 ? xi[0] : q == 1 ? xi[1] : xi[2], __dmul_rn(S.dt, vn));
  const uint32_t X = periodic_fx(p, S.Lfx[a], S.M64[a]);
  if (act && q < 3) {
    if (!isfinite(vn) || !isfinite(p)) set_status(ctl, PRX_ENONFINITE);
    double* const to = q == 0 ? B.vx : q == 1 ? B.vy : B.vz;
    to[i] = vn;
    xn[a][i] = p;
  }
  const uint32_t Y = __shfl_down_sync(0xFFFFFFFFu, X, 1, 8), Z = __shfl_down_sync(0xFFFFFFFFu, X, 2, 8);
  bool moved = false;
  if (act && q == 0) {
    moved = moved_beyond_skin(S, X, Y, Z, W);
    Pn[i] = make_uint4(X, Y, Z, W);
  }
  return moved;
}

// Entry k of slot i's list.
template <bool NL16>
__device__ __forceinline__ void nl_put(const Sys& S, int k, uint32_t i, uint32_t j) {
  if constexpr (NL16) ((uint16_t*)S.nl)[(size_t)k * S.n + i] = (uint16_t)j;
  else ((uint32_t*)S.nl)[(size_t)k * S.n + i] = j;
}
// The count of slot i's list (cnt hits, written up to the capacity) and its
// padding to a whole stage of four with the slot itself.
template <bool NL16>
__device__ __forceinline__ void nl_close(const Sys& S, uint32_t i, int cnt) {
  const int m = min(cnt, S.list_cap);
  S.nn[i] = (uint8_t)m;
  if (cnt > S.list_cap) set_status(S.ctl, PRX_ECAPACITY);
  for (int k = m; k < ((m + 3) & ~3); ++k) nl_put<NL16>(S, k, i, i);
}

// Lists of one slot straight from the cells (exact fixed-point distances, the
// order of the tiles' windows), for the rare tiles that the staged build below
// cannot hold.
template <bool NL16>
__device__ __noinline__ void eng_list_slow(const Sys& S, const uint4* P, uint32_t i, uint32_t kc) {
  const int nx = S.nc[0], ny = S.nc[1], nz = S.nc[2];
  const int cx = (int)(kc % (uint32_t)nx), cy = (int)(kc / (uint32_t)nx % (uint32_t)ny), cz = (int)(kc / (uint32_t)nx / (uint32_t)ny);
  const uint4 pi = P[i];
  int cnt = 0;
  for (int dz = -1; dz <= 1; ++dz)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx) {
        const int c = (wrap_cell(cz + dz, nz) * ny + wrap_cell(cy + dy, ny)) * nx + wrap_cell(cx + dx, nx);
        for (uint32_t j = S.cell_start[c]; j < S.cell_start[c + 1]; ++j) {
          if (j == i) continue;
          float ex, ey, ez;
          disp(S, P[j], pi, ex, ey, ez);
          if (!(fmaf(ez, ez, fmaf(ey, ey, ex * ex)) < S.rv2_build)) continue;
          if (cnt < S.list_cap) nl_put<NL16>(S, cnt, i, j);
          ++cnt;
        }
      }
  nl_close<NL16>(S, i, cnt);
}

struct RowInfo {
  int base;        // first staged index of the row
  int padL;        // particles of the left image cell (cell nx-1)
  int rowcount;    // particles of the row
  int tot;         // padL + rowcount + padR
  int row_lo;      // first slot of the row
  int left_start;  // first slot of cell nx-1
  int c1;          // first slot of cell 1 (end of cell 0)
  uint32_t yref;   // fixed-point lower edge of the (wrapped) row in y
  uint32_t zref;   // and in z
  float yoff;      // that edge's offset from the tile's lower edge, unwrapped
  float zoff;
  int pad;
};
// FP32 coordinates of a staged particle in the tile's frame: y and z relative
// to the tile's lower cell edges (each row's images unwrapped), x in [0, L)
// with the left and right image cells shifted by -L and +L.  A slot keyed to
// cell 0 (nx-1) whose position rounds to the far end of the box (possible by
// one rounding step after a restore) is taken back to the near side.  The
// values carry ~1e-5 sigma of rounding; the list radius has a margin for it.
__device__ __forceinline__ float4 build_coords(const uint4 p, const RowInfo& r, int kr,
                                               uint32_t slot, float sx, float sy, float sz,
                                               float Lx) {
  float xf = __uint2float_rn(p.x) * sx;
  if (slot < (uint32_t)r.c1 && p.x >= 0x80000000u) xf -= Lx;
  if (slot >= (uint32_t)r.left_start && p.x < 0x80000000u) xf += Lx;
  if (kr < r.padL) xf -= Lx;
  else if (kr >= r.padL + r.rowcount) xf += Lx;
  const float yf = fmaf(__int2float_rn(pdiff(p.y, r.yref)), sy, r.yoff);
  const float zf = fmaf(__int2float_rn(pdiff(p.z, r.zref)), sz, r.zoff);
  return make_float4(xf, yf, zf, __uint_as_float(slot));
}

// The lists of one tile (eng_ty cell rows at one cz) with three threads per
// slot, one per layer of neighbour cells: each marks its hits of the
// layer's three windows in bit masks (no store and no branch per candidate),
// the three counts give each its place in the list, and the marked
// candidates are written.  The lists differ from build_tile's at most in pairs
// at the edge of the list radius.
template <bool NL16>
__device__ __forceinline__ void eng_build_tile(const Sys& S, const uint4* P, const uint32_t* cell_of, uint32_t tile,
                                               unsigned char* smem) {
  const int CAP = S.eng_cap;
  float4* sX = reinterpret_cast<float4*>(smem);
  RowInfo* ri = reinterpret_cast<RowInfo*>(smem + 16 * (size_t)(CAP + 4));
  uint32_t* sCS = reinterpret_cast<uint32_t*>(ri + TILE_ROWS_MAX);
  uint32_t* sM = sCS + TILE_ROWS_MAX * (S.nc[0] + 1);                 // [3][ENG_UNITS] hit masks
  uint16_t* sLo = reinterpret_cast<uint16_t*>(sM + 3 * ENG_UNITS);    // [3][ENG_UNITS] first staged entries
  uint8_t* sCnt = reinterpret_cast<uint8_t*>(sLo + 3 * ENG_UNITS);    // [ENG_UNITS] hits
  __shared__ int sBad;
  const int nx = S.nc[0], ny = S.nc[1], nz = S.nc[2];
  const int ty = tile % S.eng_tiles_y, cz = tile / S.eng_tiles_y;
  const int cy0 = ty * S.eng_ty;
  const int TYb = min(S.eng_ty, ny - cy0);
  const int RY = TYb + 2, R = 3 * RY;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = ENG_THREADS / 32;
  // one warp per row: its cell offsets, then its description
  for (int sr = warp; sr < R; sr += nwarps) {
    const int dzi = sr / RY, yi = sr - dzi * RY;
    const int uy = cy0 - 1 + yi, uz = cz - 1 + dzi;  // unwrapped row indices
    const int qy = wrap_cell(uy, ny), qz = wrap_cell(uz, nz);
    const uint32_t* src = S.cell_start + (qz * ny + qy) * nx;
    uint32_t* cs = sCS + sr * (nx + 1);
    for (int c = lane; c <= nx; c += 32) cs[c] = src[c];
    __syncwarp();
    if (lane == 0) {
      RowInfo r;
      r.padL = (int)(cs[nx] - cs[nx - 1]);
      r.rowcount = (int)(cs[nx] - cs[0]);
      r.tot = r.padL + r.rowcount + (int)(cs[1] - cs[0]);
      r.row_lo = (int)cs[0];
      r.left_start = (int)cs[nx - 1];
      r.c1 = (int)cs[1];
      // qy 2^32 / ny to within one unit
      r.yref = (uint32_t)__umul64hi((unsigned long long)qy << 32, S.inv_nc64[0]);
      r.zref = (uint32_t)__umul64hi((unsigned long long)qz << 32, S.inv_nc64[1]);
      r.yoff = (float)(uy - cy0) * S.cell_edge_f[0];
      r.zoff = (float)(uz - cz) * S.cell_edge_f[1];
      ri[sr] = r;
    }
  }
  if (threadIdx.x == 0) sBad = 0;
  __syncthreads();
  if (warp == 0) {
    int v = lane < R ? ri[lane].tot : 0;
    const int own = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xFFFFFFFFu, v, o);
      if (lane >= o) v += u;
    }
    if (lane < R) ri[lane].base = v - own;
    if (lane == 31 && v > CAP) sBad = 1;
  }
  const uint32_t rs = S.cell_start[(cz * ny + cy0) * nx];
  const uint32_t re = S.cell_start[(cz * ny + cy0 + TYb - 1) * nx + nx];
  __syncthreads();
  const int ns = (int)(re - rs);
  if (sBad || ns > S.eng_slots) {
    for (uint32_t i = rs + threadIdx.x; i < re; i += ENG_THREADS) eng_list_slow<NL16>(S, P, i, cell_of[i]);
    return;
  }
  const float sx = S.scale[0], sy = S.scale[1], sz = S.scale[2], rv2 = S.rv2_build;
  const float Lx = (float)S.L[0];
  for (int sr = warp; sr < R; sr += nwarps) {
    const RowInfo r = ri[sr];
    for (int kr = lane; kr < r.tot; kr += 32) {
      const int slot = kr < r.padL ? r.left_start + kr
                                   : r.row_lo + (kr < r.padL + r.rowcount ? kr - r.padL : kr - r.padL - r.rowcount);
      sX[r.base + kr] = build_coords(P[slot], r, kr, (uint32_t)slot, sx, sy, sz, Lx);
    }
  }
  __syncthreads();
  // (slot, layer) pairs, layer-major
  const int units = 3 * ns;
#pragma unroll 1
  for (int v = threadIdx.x; v < units; v += ENG_THREADS) {
    const int dzi = v >= 2 * ns ? 2 : (v >= ns ? 1 : 0);
    const uint32_t i = rs + (uint32_t)(v - dzi * ns);
    const uint32_t kc = cell_of[i];
    const int cx = (int)(kc % (uint32_t)nx);
    const int yrel = (int)(kc / (uint32_t)nx % (uint32_t)ny) - cy0;
    const RowInfo& rc = ri[RY + yrel + 1];
    const int kself = rc.base + rc.padL + ((int)i - rc.row_lo);
    const float4 fi = sX[kself];
    int cnt = 0;
#pragma unroll 1
    for (int w = 0; w < 3; ++w) {
      const int sr = dzi * RY + yrel + w;
      const uint32_t* cs = sCS + sr * (nx + 1);
      const RowInfo& r = ri[sr];
      const int lo = r.base + (cx == 0 ? 0 : r.padL + (int)cs[cx - 1] - r.row_lo);
      const int hi = r.base + (cx + 2 > nx ? r.tot : r.padL + (int)cs[cx + 2] - r.row_lo);
      const int len = hi - lo;
      if (len > 32) sBad = 1;  // (the same value from every thread that stores it)
      uint32_t mm = 0u;
#pragma unroll 1
      for (int k = 0; k < min(len, 32); k += 4) {
        uint32_t h = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 c = sX[lo + k + u];  // (the buffer has four spare entries)
          const float dx = c.x - fi.x, dy = c.y - fi.y, dz = c.z - fi.z;
          if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < rv2) h |= 1u << u;
        }
        mm |= h << k;
      }
      if (len < 32) mm &= (1u << len) - 1u;
      if (dzi == 1 && w == 1) mm &= ~(1u << ((kself - lo) & 31));
      sM[w * ENG_UNITS + v] = mm;
      sLo[w * ENG_UNITS + v] = (uint16_t)lo;
      cnt += __popc(mm);
    }
    sCnt[v] = (uint8_t)cnt;
  }
  __syncthreads();
  if (sBad) {
    for (uint32_t i = rs + threadIdx.x; i < re; i += ENG_THREADS) eng_list_slow<NL16>(S, P, i, cell_of[i]);
    return;
  }
#pragma unroll 1
  for (int v = threadIdx.x; v < units; v += ENG_THREADS) {
    const int dzi = v >= 2 * ns ? 2 : (v >= ns ? 1 : 0);
    const int q = v - dzi * ns;
    const uint32_t i = rs + (uint32_t)q;
    int k = 0;
    if (dzi > 0) k += sCnt[q];
    if (dzi > 1) k += sCnt[ns + q];
#pragma unroll 1
    for (int w = 0; w < 3; ++w) {
      const float4* from = sX + sLo[w * ENG_UNITS + v];
      uint32_t mm = sM[w * ENG_UNITS + v];
#pragma unroll 1
      while (mm) {  // two hits at a time
        const int h0 = __ffs(mm) - 1;
        mm &= mm - 1u;
        const int h1 = mm ? __ffs(mm) - 1 : -1;
        mm &= mm - 1u;
        const uint32_t j0 = __float_as_uint(from[h0].w), j1 = __float_as_uint(from[max(h1, 0)].w);
        if (k < S.list_cap) nl_put<NL16>(S, k, i, j0);
        if (h1 >= 0 && k + 1 < S.list_cap) nl_put<NL16>(S, k + 1, i, j1);
        k += h1 >= 0 ? 2 : 1;
      }
    }
    if (dzi == 2) nl_close<NL16>(S, i, k);  // the last layer's thread knows the whole count
  }
}

// Rebuild (at most ENG_CELLS cells) in three phases: keys, with every slot put
// into its cell's bucket; the permutation, before which each block scans all
// cell counts for itself in shared memory; the lists.  The keys' atomics give
// each slot's arrival rank in its cell, which decides its place in the bucket
// only: its new slot is its cell's first slot plus the number of the cell's
// members with a smaller old slot, so the order in which the atomics
// completed does not matter.  When a cell has more members than a bucket
// holds, a phase more scatters the slots by rank into tmp, whose rows take
// the buckets' place.
template <bool NL16>
__device__ __forceinline__ int eng_rebuild(const Sys& S, const SoA& A, const SoA& B, uint4* P, uint32_t b,
                                                 GridBar& bar, unsigned char* smem) {
  const uint32_t nb = bar.nb, g = b * ENG_THREADS + threadIdx.x, stride = nb * ENG_THREADS;
  const uint32_t ncell = (uint32_t)S.ncell;
  bool over = false;
  for (uint32_t i = g; i < S.n; i += stride) {
    const uint32_t k = cell_of_pos(S, P[i]);
    S.key[i] = k;
    const uint32_t rank = atomicAdd(&S.count[k], 1u);
    S.new_of_old[i] = rank;
    if (rank < ENG_BUCKET) S.bucket[(size_t)k * ENG_BUCKET + rank] = i;
    else over = true;
  }
  const int over_any = bar.sync(over);
  if (over_any == 2) return 2;
  // scan: warp w of the block takes cells [w seg, (w + 1) seg), 512 at a
  // time (four loads in flight), then adds the earlier segments' total
  uint32_t* sCS = reinterpret_cast<uint32_t*>(smem);
  constexpr uint32_t WARPS = ENG_THREADS / 32;
  __shared__ uint32_t wtot[WARPS];
  const int lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5;
  const uint32_t seg = (ncell + WARPS * 128u - 1u) / (WARPS * 128u) * 128u;
  const uint32_t s0 = warp * seg + 4u * (uint32_t)lane, s1 = (warp + 1u) * seg;
  uint32_t carry = 0u;
#pragma unroll 1
  for (uint32_t c0 = s0; c0 < s1; c0 += 512u) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t c = c0 + (uint32_t)u * 128u;
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (c < s1 && c < ncell) v[u] = *reinterpret_cast<const uint4*>(S.count + c);  // (padded with zeros)
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t c = c0 + (uint32_t)u * 128u;
      const uint32_t t = v[u].x + v[u].y + v[u].z + v[u].w;
      uint32_t x = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
      }
      const uint32_t e = carry + x - t;
      carry += __shfl_sync(0xFFFFFFFFu, x, 31);
      if (c < s1)
        *reinterpret_cast<uint4*>(sCS + c) = make_uint4(e, e + v[u].x, e + v[u].x + v[u].y, e + v[u].x + v[u].y + v[u].z);
    }
  }
  if (lane == 0) wtot[warp] = carry;
  __syncthreads();
  {
    uint32_t off = 0u;
    for (uint32_t w = 0; w < warp; ++w) off += wtot[w];
    for (uint32_t c = s0; c < s1; c += 128u) {
      uint4 v = *reinterpret_cast<uint4*>(sCS + c);
      v.x += off, v.y += off, v.z += off, v.w += off;
      *reinterpret_cast<uint4*>(sCS + c) = v;
    }
  }
  __syncthreads();
  auto first = [&](uint32_t k) { return sCS[k]; };
  // this block's share of the offsets, for the lists (and checkpoints)
  for (uint32_t c = g; c < ncell; c += stride) S.cell_start[c] = first(c);
  if (g == 0u) S.cell_start[ncell] = S.n;
  if (over_any) {
    for (uint32_t i = g; i < S.n; i += stride) S.tmp[first(S.key[i]) + S.new_of_old[i]] = i;
    if (bar.sync(false) == 2) return 2;
  }
  auto start = [&](uint32_t k) { return k < ncell ? first(k) : S.n; };
  auto from_tmp = [&](uint32_t j, uint32_t, uint32_t s0, uint32_t c) {
    uint32_t r = s0;
#pragma unroll 4
    for (uint32_t q = 0; q < c; ++q) r += S.tmp[s0 + q] < j ? 1u : 0u;
    return r;
  };
  for (uint32_t o = g; o < S.n; o += stride) permute_old<false>(S, A, B, P, S.win, o, start, over_any != 0, from_tmp);
  if (bar.sync(false) == 2) return 2;
  for (uint32_t c = g; c < ncell; c += stride) S.count[c] = 0u;  // (zero outside rebuilds)
  const uint32_t nt = (uint32_t)(S.eng_tiles_y * S.nc[2]);
  for (uint32_t t = b; t < nt; t += nb) {
    eng_build_tile<NL16>(S, P, S.win, t, smem);
    __syncthreads();
  }
  return bar.sync(false);
}

// Reaction step: each block searches for the eligible A's of its own range
// of slots (compacted into the same range of tmp), then forms the bonds.
template <bool NL16>
__device__ __forceinline__ int eng_react(const Sys& S, const SoA& B, const uint4* P, uint32_t b, GridBar& bar,
                                         unsigned long long step, uint32_t* s_cnt, int32_t* dpop) {
  const RxParams& R = S.R;
  const uint32_t nb = bar.nb;
  const uint32_t lo = (uint32_t)((unsigned long long)S.n * b / nb);
  const uint32_t hi = (uint32_t)((unsigned long long)S.n * (b + 1u) / nb);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) *s_cnt = 0u;
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += ENG_THREADS) dpop[k] = 0;
  __syncthreads();
  for (uint32_t base = lo; base < hi; base += ENG_THREADS) {
    const uint32_t i = base + threadIdx.x;
    bool el = false;
    if (i < hi) {
      S.win[i] = NONE;
      const uint32_t t = B.type[i];
      const int s = B.state[i];
      el = R.nr > 1 ? rx_elig_A(R, t, s) != 0u : in_window(R.mask_A, R.a_lo, R.a_hi, t, s);
    }
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, el);
    if (!bal) continue;
    uint32_t at = 0u;
    if (lane == 0) at = atomicAdd(s_cnt, (uint32_t)__popc(bal));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (el) S.tmp[lo + at + __popc(bal & ((1u << lane) - 1u))] = i;
  }
  __syncthreads();
  const uint32_t nact = *s_cnt;
  const uint32_t* list = S.tmp + lo;
  long long unused = 0;
  if (R.rule != PRX_SELECT_NEAREST && R.nr <= 1) {
    rx_find_random4<NL16>(S, Blk{0u, 1u}, B, P, step, list, nact, unused, unused);
  } else {
    for (uint32_t wb = (threadIdx.x & ~31u) / RX_GROUP; wb < nact; wb += ENG_THREADS / RX_GROUP) {
      const uint32_t w = wb + (uint32_t)lane / RX_GROUP;
      const bool valid = w < nact;
      const uint32_t i = valid ? list[w] : 0u;
      uint32_t best = NONE, ch = 0u;
      if (R.rule == PRX_SELECT_NEAREST) best = nearest_partner<NL16, RX_GROUP>(S, B, P, i, valid, true, unused);
      else best = rx_find_multi<NL16, RX_GROUP>(S, B, P, step, i, valid, unused, unused, ch);
      if (valid && lane % RX_GROUP == 0) {
        if (R.nr > 1) S.wch[i] = (uint8_t)ch;
        S.win[i] = best;
      }
    }
    if (R.rule == PRX_SELECT_NEAREST) {
      for (uint32_t wb = lo + (threadIdx.x & ~31u) / RX_GROUP; wb < hi; wb += ENG_THREADS / RX_GROUP) {
        const uint32_t i = wb + (uint32_t)lane / RX_GROUP;
        const bool valid = i < hi && in_window(R.mask_T, R.t_lo, R.t_hi, B.type[i], B.state[i]);
        if (!__any_sync(0xFFFFFFFFu, valid)) continue;
        const uint32_t best = nearest_partner<NL16, RX_GROUP>(S, B, P, i, valid, false, unused);
        if (valid && lane % RX_GROUP == 0) S.win[i] = best;
      }
    }
  }
  if (bar.sync(false) == 2) return 2;
  for (uint32_t wb = (threadIdx.x & ~31u) / RX_GROUP; wb < nact; wb += ENG_THREADS / RX_GROUP) {
    const uint32_t w = wb + (uint32_t)lane / RX_GROUP;
    const uint32_t i = w < nact ? list[w] : 0u;
    bool unused_w;
    const uint32_t T = rx_decide<NL16, RX_GROUP>(S, B, step, i, w < nact, unused_w);
    (void)rx_form(S, B, step, i, lane % RX_GROUP == 0 ? T : NONE, dpop);
  }
  __syncthreads();
  int32_t* rep = S.pop + (size_t)(b % POP_REPLICAS) * (PRX_MAX_TYPES * PRX_MAX_STATES);
  for (int k = threadIdx.x; k < PRX_MAX_TYPES * PRX_MAX_STATES; k += ENG_THREADS)
    if (dpop[k]) atomicAdd(rep + k, dpop[k]);
  if (bar.sync(false) == 2) return 2;
  if (b == 0u) rx_record(S, (long long)step);
  return 0;
}

// nsteps steps of one system by block b of its grid.  theta: steps between
// reaction steps (0: no scheme).
template <bool NL16, bool CUBIC, bool F64>
__device__ __forceinline__ void eng_run(const Sys& S, uint32_t b, GridBar& bar, uint32_t nsteps, uint32_t theta,
                                        unsigned char* smem) {
  __shared__ uint32_t s_cnt;
  __shared__ int32_t dpop[PRX_MAX_TYPES * PRX_MAX_STATES];
  Ctl* ctl = S.ctl;
  int set = ctl->set, ph = ctl->phase;
  int xp = 0;  // F64: the live positions are in the other set's arrays
  unsigned long long step = ctl->step;
  uint32_t until = theta ? theta - (uint32_t)(step % theta) : 0u;
  unsigned int rebins = 0;
  const uint32_t warp = threadIdx.x >> 5;
  constexpr uint32_t per = F64 ? 4u : 32u;
  const uint32_t chunks = (S.n + per - 1u) / per;
  // contiguous chunks of slots per block, so that a block's neighbour gathers
  // share its L1; FP32: one chunk per warp, its slots in the lanes' registers
  const uint32_t c0 = (uint32_t)((unsigned long long)chunks * b / bar.nb);
  const uint32_t c1 = (uint32_t)((unsigned long long)chunks * (b + 1u) / bar.nb);
  [[maybe_unused]] Resident r;
  const uint32_t ri = (c0 + warp) * 32u + (threadIdx.x & 31u);
  const bool rv = !F64 && c0 + warp < c1 && ri < S.n;
  if (rv) res_load<NL16>(S, set ? S.s1 : S.s0, ph ? S.P1 : S.P0, ri, r, smem);
  int bad = 0;
#pragma unroll 1
  for (uint32_t q = 0; q < nsteps; ++q) {
    ++step;
    const uint4* P = ph ? S.P1 : S.P0;
    uint4* Pn = ph ? S.P0 : S.P1;
    bool moved = false;
    const bool reacts = until == 1u;
    if constexpr (F64) {
      const SoA B = set ? S.s1 : S.s0, O = set ? S.s0 : S.s1;
      double* const x[3] = {xp ? O.x : B.x, xp ? O.y : B.y, xp ? O.z : B.z};
      double* const xn[3] = {xp ? B.x : O.x, xp ? B.y : O.y, xp ? B.z : O.z};
#pragma unroll 1
      for (uint32_t c = c0 + warp; c < c1; c += ENG_THREADS / 32)
        moved |= eng_step64<NL16>(S, ctl, B, x, xn, P, Pn, c, step);
      xp ^= 1;
    } else if (rv) {
      const SoA B = set ? S.s1 : S.s0;
      moved = res_step<NL16, CUBIC>(S, ctl, B, P, Pn, ri, step, r, smem);
      if (reacts) res_store_x(B, ri, r);  // the search tests absolute positions
    }
    ph ^= 1;
    const int any = bar.sync(moved);
    if ((bad = any == 2)) break;
    if (any) {
      const SoA A = set ? S.s1 : S.s0, B = set ? S.s0 : S.s1;
      if (rv) {
        if (!reacts) res_store_x(A, ri, r);
        res_store_v(A, ri, r);
      }
      if (F64 && xp) {  // the permutation reads the current set and writes the other
        for (uint32_t i = b * ENG_THREADS + threadIdx.x; i < S.n; i += bar.nb * ENG_THREADS)
          A.x[i] = B.x[i], A.y[i] = B.y[i], A.z[i] = B.z[i];
        xp = 0;
      }
      uint4* Pc = ph ? S.P1 : S.P0;
      if ((bad = eng_rebuild<NL16>(S, A, B, Pc, b, bar, smem) == 2)) break;
      set ^= 1;
      ++rebins;
      if (rv) res_load<NL16>(S, B, Pc, ri, r, smem);
    }
    if (reacts) {
      SoA B = set ? S.s1 : S.s0;
      if (F64 && xp) {
        const SoA O = set ? S.s0 : S.s1;
        B.x = O.x, B.y = O.y, B.z = O.z;
      }
      if ((bad = eng_react<NL16>(S, B, ph ? S.P1 : S.P0, b, bar, step, &s_cnt, dpop) == 2)) break;
      if (rv) res_load_bonds(S, B, ri, r);
      until = theta;
    } else {
      until -= until ? 1u : 0u;
    }
  }
  if (rv && !bad) {
    const SoA B = set ? S.s1 : S.s0;
    res_store_x(B, ri, r);
    res_store_v(B, ri, r);
  }
  if (F64 && xp && !bad) {
    const SoA A = set ? S.s1 : S.s0, B = set ? S.s0 : S.s1;
    for (uint32_t i = b * ENG_THREADS + threadIdx.x; i < S.n; i += bar.nb * ENG_THREADS)
      A.x[i] = B.x[i], A.y[i] = B.y[i], A.z[i] = B.z[i];
  }
  if (threadIdx.x == 0) {
    // over any earlier status: what a rebuild left half done (counters that are
    // not zero, positions in the next set's order) must stop the later ones
    if (bad) atomicExch(&ctl->status, PRX_ETIMEOUT);
    if (b == 0u) {
      ctl->set = set;
      ctl->phase = ph;
      ctl->eng_steps += step - ctl->step;
      ctl->step = step;
      ctl->rebins += rebins;
    }
  }
}

// One system, every block of the grid.  bar: this launch's two
// words; bar_next: the next launch's, cleared here (launches of a system
// follow one another on its stream).  nsteps = 0: a launch of a run that the
// device drives (dg.cu), which has steps_left to go and clears the words itself.
template <bool NL16, bool CUBIC, bool F64>
__global__ void __launch_bounds__(ENG_THREADS, 1)
    k_engine(Sys S, uint32_t nsteps, uint32_t theta, unsigned long long* bar, unsigned long long* bar_next,
             uint32_t polls) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int res;
  // a wait of an earlier launch ran out: nothing may build on what it left.
  // (A block that reads the status of this launch's own timeout leaves early
  // where the others already have.)
  const bool marks = nsteps != 0u && blockIdx.x == 0 && threadIdx.x == 0;
  const int gone = S.ctl->status == PRX_ETIMEOUT;
  if (__syncthreads_or(gone)) {
    if (marks) mark_run(S.ctl);
    return;
  }
  if (bar_next && blockIdx.x == 0 && threadIdx.x < 2) bar_next[threadIdx.x * 16] = 0ull;
  if (nsteps == 0u) nsteps = (uint32_t)min((unsigned long long)ENG_STEPS, S.ctl->steps_left);
  GridBar gb{bar, &res, gridDim.x, 0u, 0u, 0u, polls};
  eng_run<NL16, CUBIC, F64>(S, blockIdx.x, gb, nsteps, theta, smem);
  if (marks) mark_run(S.ctl);
}

// The kernel that runs system S.
template <bool F64>
const void* engine_kernel(const Sys& S) {
  if (F64 || S.cubic) return S.nl16 ? (const void*)k_engine<true, true, F64> : (const void*)k_engine<false, true, F64>;
  if constexpr (!F64) return S.nl16 ? (const void*)k_engine<true, false, false> : (const void*)k_engine<false, false, false>;
  return nullptr;
}

std::mutex g_eng_mu;
struct EngSmem {
  const void* k;
  int dev;
  size_t bytes;
};
EngSmem g_eng_smem[64];

// Raises the kernel's dynamic shared-memory limit on the current device to
// at least `bytes` (it only grows, so that systems of different sizes coexist).
bool eng_raise_smem(const void* k, int dev, size_t bytes) {
  std::lock_guard<std::mutex> lk(g_eng_mu);
  for (EngSmem& e : g_eng_smem) {
    if (e.k && (e.k != k || e.dev != dev)) continue;
    if (e.k && e.bytes >= bytes) return true;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return false;
    e = EngSmem{k, dev, bytes};
    return true;
  }
  return false;
}

}  // namespace

// Dynamic shared memory of a system's persistent runs: the largest of the
// resident slots' lists and gathered positions, the list build's buffers and
// the block's own scan of the cell counts (one after the other).
static size_t engine_smem(const Sys& S) {
  const size_t scan = 4 * ((size_t)S.ncell + 4 * ENG_THREADS);  // (whole segments)
  const size_t lists = 16 * (size_t)(S.eng_cap + 4) + sizeof(RowInfo) * TILE_ROWS_MAX +
                       4 * (size_t)TILE_ROWS_MAX * (S.nc[0] + 1) + (3 * 6 + 1) * (size_t)ENG_UNITS;
  return std::max(std::max(scan, lists), RES_SMEM);
}

// Resident blocks of kernel k on the current device (0: it cannot be
// launched cooperatively with `sm` bytes of shared memory).
static unsigned engine_resident(const void* k, size_t sm) {
  int dev = 0, coop = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
      !eng_raise_smem(k, dev, sm) ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, ENG_THREADS, sm) != cudaSuccess || per < 1) {
    cudaGetLastError();
    return 0;
  }
  return device_sms() * (unsigned)per;
}

// Which runs go through the persistent kernel, by size (us per step, launch
// chain -> persistent, step growth at density 0.85 on a GB300):
//   FP32: 1,024 beads 18.8 -> 6.5, 16,384 21.1 -> 7.7, 33,000 21.3 -> 9.1,
//   60,000 23.7 -> 12.1, 77,000 24.3 -> 14.6 (the chain with four steps per
//   graph takes 20.0 at 100,000): up to one resident slot per thread of the
//   GPU (77,824 with 152 SMs).
//   FP64: 1,250 beads 30.1 -> 11.3, 5,000 34.5 -> 19.6, 10,000 40.2 -> 35.2,
//   20,000 53 -> 58 (by then the FP64 pipe bounds both): up to 16,384.
// Runs with a force cap (warm-ups) and four-lane runs keep the launch chain,
// as do boxes with more cells or longer rows than the rebuild holds.
//
// And by what else is under way (runtime.cu, runs_persistent): k systems at once,
// each on its own stream, take the sum of their persistent steps, about 5.8 us
// plus 0.086 per 1,000 beads each, divided by the grids that fit side by side
// (FP64: 9.5 plus 1.85 per 1,000), but as chains 17 us plus 0.05 per 1,000 beads
// of all together (FP64: 28 plus 1.0).  `load` is a system's share of where the
// two are equal.  us per step of all, persistent / chains:
//   1,250 beads: k = 3 5.9 / 20, 8 17 / 18, 16 35 / 19
//   2,048: k = 2 11.7 / 20, 3 17.6 / 17, 4 24 / 17, 8 48 / 18, 16 96 / 19
//   16,384: k = 2 13.9 / 21, 3 20.6 / 18, 4 28 / 19, 16 113 / 26
//   33,096: k = 2 16.6 / 23, 3 25.5 / 21, 4 34 / 22, 8 68 / 27, 16 136 / 40
//   70,000: k = 2 23.8 / 24, 3 36 / 25, 4 48 / 28, 8 96 / 43, 16 192 / 80
//   FP64: 1,000: k = 2 21.8 / 30, 3 33 / 30, 8 87 / 31; 5,000: k = 2 34 / 35,
//   3 51 / 40, 8 137 / 61; 10,000: k = 2 59 / 46; 16,000: k = 2 75 / 62, 8 301 / 172
EngPlan engine_plan(const Sys& S, int fp64) {
  EngPlan p;
  if (!S.n || !S.bucket || S.ncell > (int)ENG_CELLS || !S.eng_ty || S.fcapf > 0.f || S.step_lanes != 1) return p;
  if (fp64 && S.n > ENG_F64_MAX) return p;
  p.smem = engine_smem(S);
  const unsigned warps = ENG_THREADS / 32;
  const unsigned chunks = fp64 ? (S.n + 3u) / 4u : (S.n + 31u) / 32u;
  p.kernel = fp64 ? engine_kernel<true>(S) : engine_kernel<false>(S);
  const unsigned most = engine_resident(p.kernel, p.smem);
  if (!fp64 && chunks > most * warps) return p;
  // a block per chunk as far as they go (the phases are bound by latency),
  // and one per tile of the list build
  p.blocks = std::min(most, std::max(chunks, (unsigned)(S.eng_tiles_y * S.nc[2])));
  const double share = 1.0 / (most / p.blocks);  // of the GPU: grids that fit side by side run at once
  p.load = fp64 ? (9.5 * share + 0.85e-3 * S.n) / 28.0 : (5.8 * share + 3.6e-5 * S.n) / 17.0;
  return p;
}

cudaError_t launch_engine(const Sys& S, cudaStream_t st, const EngPlan& p, uint32_t nsteps, uint32_t theta,
                          unsigned long long* bar, unsigned long long* bar_next) {
  Sys s = S;
  uint32_t polls = p.polls;
  void* args[] = {&s, &nsteps, &theta, &bar, &bar_next, &polls};
  return cudaLaunchCooperativeKernel(p.kernel, dim3(p.blocks), dim3(ENG_THREADS), args, p.smem, st);
}

}  // namespace prx
