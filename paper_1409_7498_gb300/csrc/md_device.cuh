// Device functions of the MD step, the rebuild and the Verlet-list build that
// the one-phase kernels (md_kernels.cu) and the persistent run kernels
// (engine.cu) share.
#pragma once
#include "prx_internal.cuh"

namespace prx {

namespace {

// WCA pair term in FP32; d = x_j - x_i.  Adds -g d to f and V/2 to e.
// Reciprocals and quotients use the hardware approximation (relative error
// about 2^-22), well inside the FP32 force tolerance.
__device__ __forceinline__ void wca32(const Sys& S, float dx, float dy, float dz, float r2,
                                      float& fx, float& fy, float& fz, float& e) {
  const float r2i = __fdividef(1.0f, r2);
  const float sr2 = S.sig2f * r2i;
  const float sr6 = sr2 * sr2 * sr2;
  float g = S.eps24f * sr6 * (2.0f * sr6 - 1.0f) * r2i;
  if (S.fcapf > 0.0f) {
    const float r = sqrtf(r2);
    if (g * r > S.fcapf) g = __fdividef(S.fcapf, r);
  }
  fx -= g * dx;
  fy -= g * dy;
  fz -= g * dz;
  e += 0.5f * S.eps4f * (sr6 * sr6 - sr6 + 0.25f);
}

// Bond term in FP32 (FENE or mirror LJ by style); returns false on FENE overstretch.
__device__ __forceinline__ bool bond32(const Sys& S, uint32_t style, float dx, float dy, float dz,
                                       float& fx, float& fy, float& fz, float& e) {
  const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
  float g;
  if (style == 0u) {
    if (!(r2 < S.fr02f)) return false;
    const float q = 1.0f - r2 * S.fr02if;
    g = -__fdividef(S.fkf, q);
    e += 0.5f * (-0.5f * S.fkf * S.fr02f * logf(q));
  } else {
    const float r = sqrtf(r2);
    if (!(r > S.rcf && r < 2.0f * S.rcf)) return true;
    const float sd = 2.0f * S.rcf - r;
    const float ss2 = __fdividef(S.sig2f, sd * sd);
    const float ss6 = ss2 * ss2 * ss2;
    const float dVdr = __fdividef(S.eps24f * (2.0f * ss6 * ss6 - ss6), sd);
    g = -__fdividef(dVdr, r);
    e += 0.5f * S.eps4f * (ss6 * ss6 - ss6 + 0.25f);
  }
  fx -= g * dx;
  fy -= g * dy;
  fz -= g * dz;
  return true;
}

// FP64 versions, arithmetic written as in the plain definitions.
template <bool ENERGY = true>
__device__ __forceinline__ void wca64(const Sys& S, double dx, double dy, double dz, double r2,
                                      double& fx, double& fy, double& fz, double& e) {
  const double sr2 = __ddiv_rn(S.sig2, r2);
  const double sr6 = __dmul_rn(__dmul_rn(sr2, sr2), sr2);
  const double sr12 = __dmul_rn(sr6, sr6);
  double g = __ddiv_rn(__dmul_rn(S.eps24, __dsub_rn(__dmul_rn(2.0, sr12), sr6)), r2);
  if (S.fcap > 0.0) {
    const double r = __dsqrt_rn(r2);
    if (__dmul_rn(g, r) > S.fcap) g = __ddiv_rn(S.fcap, r);
  }
  fx = __dsub_rn(fx, __dmul_rn(g, dx));
  fy = __dsub_rn(fy, __dmul_rn(g, dy));
  fz = __dsub_rn(fz, __dmul_rn(g, dz));
  if constexpr (ENERGY)
    e = __dadd_rn(e, __dmul_rn(0.5, __dmul_rn(S.eps4, __dadd_rn(__dsub_rn(sr12, sr6), 0.25))));
}

template <bool ENERGY = true>
__device__ __forceinline__ bool bond64(const Sys& S, uint32_t style, double dx, double dy,
                                       double dz, double& fx, double& fy, double& fz, double& e) {
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  double g;
  if (style == 0u) {
    if (!(r2 < S.fr02)) return false;
    const double q = __dsub_rn(1.0, __ddiv_rn(r2, S.fr02));
    g = __ddiv_rn(-S.fk, q);
    if constexpr (ENERGY)
      e = __dadd_rn(e, __dmul_rn(0.5, __dmul_rn(__dmul_rn(__dmul_rn(-0.5, S.fk), S.fr02), log(q))));
  } else {
    const double r = __dsqrt_rn(r2);
    if (!(r > S.rc && r < 2.0 * S.rc)) return true;
    const double sd = __dsub_rn(2.0 * S.rc, r);
    const double ss2 = __ddiv_rn(S.sig2, __dmul_rn(sd, sd));
    const double ss6 = __dmul_rn(__dmul_rn(ss2, ss2), ss2);
    const double ss12 = __dmul_rn(ss6, ss6);
    const double dVdr = __ddiv_rn(__dmul_rn(S.eps24, __dsub_rn(__dmul_rn(2.0, ss12), ss6)), sd);
    g = __ddiv_rn(-dVdr, r);
    if constexpr (ENERGY)
      e = __dadd_rn(e, __dmul_rn(0.5, __dmul_rn(S.eps4, __dadd_rn(__dsub_rn(ss12, ss6), 0.25))));
  }
  fx = __dsub_rn(fx, __dmul_rn(g, dx));
  fy = __dsub_rn(fy, __dmul_rn(g, dy));
  fz = __dsub_rn(fz, __dmul_rn(g, dz));
  return true;
}

// k-th Verlet-list entry of slot i: the neighbour's slot (16-bit for systems
// of at most 65,535 particles).  Entries past a slot's count hold stale
// slots of some earlier list: still valid slots.
template <bool NL16>
__device__ __forceinline__ uint32_t nl_raw(const Sys& S, int k, uint32_t i) {
  if constexpr (NL16) return __ldg(((const uint16_t*)S.nl) + (size_t)k * S.n + i);
  else return __ldg(((const uint32_t*)S.nl) + (size_t)k * S.n + i);
}
template <bool NL16>
__device__ __forceinline__ uint32_t nl_get(const Sys& S, int k, uint32_t i) {
  return nl_raw<NL16>(S, k, i);
}

// Fetch the line holding *a into L2 (no register result).
__device__ __forceinline__ void prefetch_l2(const void* a) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
}

// Physical minimum-image displacement x_j - x_i: exact in fixed point,
// converted with one rounding, scaled by L / 2^32.
__device__ __forceinline__ void disp(const Sys& S, uint4 pj, uint4 pi, float& dx, float& dy,
                                     float& dz) {
  dx = __int2float_rn(pdiff(pj.x, pi.x)) * S.scale[0];
  dy = __int2float_rn(pdiff(pj.y, pi.y)) * S.scale[1];
  dz = __int2float_rn(pdiff(pj.z, pi.z)) * S.scale[2];
}

// Displacement since the last list build exceeds skin/2 (coarse reference in .w).
__device__ __forceinline__ bool moved_beyond_skin(const Sys& S, uint32_t X, uint32_t Y, uint32_t Z,
                                                  uint32_t W) {
  const int ax = (int)(((X >> S.wshift[0]) - W) << 22) >> 22;
  const int ay = (int)(((Y >> S.wshift[1]) - (W >> 10)) << 22) >> 22;
  const int az = (int)(((Z >> S.wshift[2]) - (W >> 20)) << 22) >> 22;
  const float ex = (float)ax * S.wunit[0], ey = (float)ay * S.wunit[1], ez = (float)az * S.wunit[2];
  return fmaf(ez, ez, fmaf(ey, ey, ex * ex)) > S.disp2_max;
}

// periodic_fx for the step kernel: the scaling by 2^32 added to the binary64
// exponent field (exact for normal x; zero and subnormals stay below 1) and
// the truncation done by the hardware FP64 -> s64 conversion, which costs
// one FP64-pipe instruction instead of fx32's variable 64-bit shifts.  The
// same value as periodic_fx for |x| < 2^29.
__device__ __forceinline__ uint32_t periodic_fx_cvt(double x, long long Lfx, unsigned long long M) {
  const double y = __longlong_as_double(__double_as_longlong(x) + (32LL << 52));
  const unsigned long long a = (unsigned long long)(__double2ll_rz(y) + Lfx);
  return (uint32_t)__umul64hi(a, M);
}

// Forces read-back: force and energy of particle p.
__device__ __forceinline__ void store_force(const Sys& S, uint32_t p, double fx, double fy, double fz, double e) {
  S.fout[3 * (size_t)p + 0] = fx;
  S.fout[3 * (size_t)p + 1] = fy;
  S.fout[3 * (size_t)p + 2] = fz;
  S.eout[p] = e;
}

// Random force of the Langevin step (zero without a thermostat).
__device__ __forceinline__ float3 random_force(const Sys& S, unsigned long long step, uint32_t pid) {
  float3 R = make_float3(0.f, 0.f, 0.f);
  if (S.thermo) {
    const uint4 w = keyed_draw(S.seed, step, pid, 0u, TAG_THERMO);
    R.x = S.cRf * (u24f(w.x) - 0.5f);
    R.y = S.cRf * (u24f(w.y) - 0.5f);
    R.z = S.cRf * (u24f(w.z) - 0.5f);
  }
  return R;
}

// End of an FP32-mode step for one slot: Langevin kick (friction applied
// exactly in FP64) and drift in place; pn receives the new fixed-point
// position (with the displacement reference W).  Returns whether the
// particle moved more than skin/2 since the last list build.
//   v' = a v + b (F_c + R),  x' = x + dt v'
__device__ __forceinline__ bool kick_drift32(const Sys& S, Ctl* ctl, uint32_t W, float fx, float fy, float fz,
                                             float3 R, double& x, double& y, double& z, double& vx, double& vy,
                                             double& vz, uint4& pn) {
  const float kx = S.b_kickf * (fx + R.x), ky = S.b_kickf * (fy + R.y), kz = S.b_kickf * (fz + R.z);
  if (!(fabsf(kx) + fabsf(ky) + fabsf(kz) < 1e30f)) set_status(ctl, PRX_ENONFINITE);
  vx = __fma_rn(vx, S.a_fric, f2d_exact(kx));
  vy = __fma_rn(vy, S.a_fric, f2d_exact(ky));
  vz = __fma_rn(vz, S.a_fric, f2d_exact(kz));
  x = __fma_rn(S.dt, vx, x);
  y = __fma_rn(S.dt, vy, y);
  z = __fma_rn(S.dt, vz, z);
  pn = make_uint4(periodic_fx_cvt(x, S.Lfx[0], S.M64[0]), periodic_fx_cvt(y, S.Lfx[1], S.M64[1]),
                  periodic_fx_cvt(z, S.Lfx[2], S.M64[2]), W);
  return moved_beyond_skin(S, pn.x, pn.y, pn.z, W);
}

// The same for slot i in memory.
__device__ __forceinline__ bool integrate32(const Sys& S, Ctl* ctl, const SoA& B, uint4* Pn, uint32_t i,
                                            uint32_t pid, uint32_t W, unsigned long long step, float fx, float fy,
                                            float fz, double x, double y, double z, double vx, double vy,
                                            double vz) {
  uint4 pn;
  const bool moved = kick_drift32(S, ctl, W, fx, fy, fz, random_force(S, step, pid), x, y, z, vx, vy, vz, pn);
  B.vx[i] = vx;
  B.vy[i] = vy;
  B.vz[i] = vz;
  B.x[i] = x;
  B.y[i] = y;
  B.z[i] = z;
  Pn[i] = pn;
  return moved;
}

// One list entry's contribution to the force on pi (in a cubic box in
// position units, scaled once per particle at the end); the slot itself
// (padding, r = 0) and pairs beyond the cutoff add nothing.
template <bool CUBIC>
__device__ __forceinline__ void pair32(const Sys& S, uint4 pj, uint4 pi, float& fx, float& fy, float& fz, float& e) {
  if constexpr (CUBIC) {
    const float ux = __int2float_rn(pdiff(pj.x, pi.x));
    const float uy = __int2float_rn(pdiff(pj.y, pi.y));
    const float uz = __int2float_rn(pdiff(pj.z, pi.z));
    const float r2u = fmaf(uz, uz, fmaf(uy, uy, ux * ux));
    if (r2u > 0.f && r2u < S.rc2u) wca32(S, ux, uy, uz, r2u * S.s2f, fx, fy, fz, e);
  } else {
    float dx, dy, dz;
    disp(S, pj, pi, dx, dy, dz);
    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    if (r2 > 0.f && r2 < S.rc2f) wca32(S, dx, dy, dz, r2, fx, fy, fz, e);
  }
}

// pair32 without a force cap and without a branch: a pair that adds nothing
// gets g = 0 (f - 0 d = f), so that four entries' chains overlap.
template <bool CUBIC>
__device__ __forceinline__ void pair32_flat(const Sys& S, uint4 pj, uint4 pi, float& fx, float& fy, float& fz) {
  float dx, dy, dz, r2;
  bool hit;
  if constexpr (CUBIC) {
    dx = __int2float_rn(pdiff(pj.x, pi.x));
    dy = __int2float_rn(pdiff(pj.y, pi.y));
    dz = __int2float_rn(pdiff(pj.z, pi.z));
    const float r2u = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    hit = r2u > 0.f && r2u < S.rc2u;
    r2 = r2u * S.s2f;
  } else {
    disp(S, pj, pi, dx, dy, dz);
    r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    hit = r2 > 0.f && r2 < S.rc2f;
  }
  const float r2i = __fdividef(1.0f, r2);
  const float sr2 = S.sig2f * r2i;
  const float sr6 = sr2 * sr2 * sr2;
  float g = S.eps24f * sr6 * (2.0f * sr6 - 1.0f) * r2i;
  g = hit ? g : 0.f;
  fx -= g * dx;
  fy -= g * dy;
  fz -= g * dz;
}

// ---------------------------------------------------------------------------
// FP32 step kernel: one thread per slot, WCA over the Verlet list.
// ---------------------------------------------------------------------------
// The step of slot i: forces over its list and bonds, then the integration
// (or, FORCES_ONLY, the forces written out by particle); returns the rebuild
// trigger.
template <bool NL16, bool FORCES_ONLY, bool CUBIC, bool CAP>
__device__ __forceinline__ bool step_one(const Sys& S, Ctl* ctl, const SoA& B,
                                         const uint4* __restrict__ P, uint4* __restrict__ Pn,
                                         uint32_t i, unsigned long long step) {
  // every load that does not depend on another goes out first
  const int cnt = __ldg(S.nn + i);
  uint32_t rn[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) rn[u] = nl_raw<NL16>(S, u, i);
  const uint4 pi = __ldg(P + i);
  // the bond count and adjacency row are read after the list loop; a
  // prefetch into L2 now hides their DRAM latency without holding
  // registers across the loop
  prefetch_l2(B.nadj + i);
  prefetch_l2(B.adj + (size_t)i * S.cap);
  float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f;
  // software pipeline over the list, four entries per stage: the next
  // stage's list entries (when this list has one) load while this stage's
  // four gathers complete.
  // The build pads every list to whole stages with the slot itself (r = 0,
  // skipped).  In a cubic box displacements stay in position units and the
  // neighbour force is scaled once at the end.
  for (int k = 0; k < cnt; k += 4) {
    uint4 pj[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) pj[u] = __ldg(P + rn[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) rn[u] = k + 4 < cnt ? nl_raw<NL16>(S, k + 4 + u, i) : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if constexpr (CAP || FORCES_ONLY) pair32<CUBIC>(S, pj[u], pi, fx, fy, fz, e);
      else pair32_flat<CUBIC>(S, pj[u], pi, fx, fy, fz);
    }
  }
  if constexpr (CUBIC) {
    fx *= S.scale[0];
    fy *= S.scale[0];
    fz *= S.scale[0];
  }
  bool ok = true;
  // bonds two at a time: both entries, then both partners' positions, in
  // flight together (half the dependent load chains).  The first pair's
  // entries load beside the bond count, and its gathers do not wait for it:
  // entries past the count (stale or never written) are clamped to a valid
  // slot and their terms skipped.
  const uint32_t* arow0 = B.adj + (size_t)i * S.cap;
  const uint32_t nb = __ldg(B.nadj + i);
  {
    const uint32_t e0 = __ldg(arow0), e1 = S.cap > 1 ? __ldg(arow0 + 1) : i;
    const uint32_t s0 = min(e0 & SLOT_MASK, S.n - 1u), s1 = min(e1 & SLOT_MASK, S.n - 1u);
    const uint4 p0 = __ldg(P + s0), p1 = __ldg(P + s1);
    float dx, dy, dz;
    if (nb > 0u) {
      disp(S, p0, pi, dx, dy, dz);
      ok = bond32(S, e0 >> 31, dx, dy, dz, fx, fy, fz, e) && ok;
    }
    if (nb > 1u) {
      disp(S, p1, pi, dx, dy, dz);
      ok = bond32(S, e1 >> 31, dx, dy, dz, fx, fy, fz, e) && ok;
    }
  }
  for (int b = 2; b < (int)nb; b += 2) {
    const uint32_t* arow = B.adj + (size_t)i * S.cap + b;
    const bool two = b + 1 < (int)nb;
    const uint32_t e0 = __ldg(arow), e1 = two ? __ldg(arow + 1) : i;
    const uint4 p0 = __ldg(P + (e0 & SLOT_MASK)), p1 = __ldg(P + (e1 & SLOT_MASK));
    float dx, dy, dz;
    disp(S, p0, pi, dx, dy, dz);
    ok = bond32(S, e0 >> 31, dx, dy, dz, fx, fy, fz, e) && ok;
    if (two) {
      disp(S, p1, pi, dx, dy, dz);
      ok = bond32(S, e1 >> 31, dx, dy, dz, fx, fy, fz, e) && ok;
    }
  }
  if (!ok) set_status(ctl, PRX_EOVERSTRETCH);
  if constexpr (FORCES_ONLY) {
    store_force(S, __ldg(B.id + i), (double)fx, (double)fy, (double)fz, (double)e);
    return false;
  } else {
    const double xi = B.x[i], yi = B.y[i], zi = B.z[i];
    const double vx = B.vx[i], vy = B.vy[i], vz = B.vz[i];
    const uint32_t pid = __ldg(B.id + i);
    return integrate32(S, ctl, B, Pn, i, pid, pi.w, step, fx, fy, fz, xi, yi, zi, vx, vy, vz);
  }
}

// v >= L: v - L; then v < 0: v + L.  The tests compare binary64 bit
// patterns on the integer pipe (for non-negative doubles the bit order is the
// numeric order; -0.0 counts as 0), so the FP64 pipe only sees the rare
// particle that left the box.
__device__ __forceinline__ double wrap_into_box(double v, double L) {
  if (__double_as_longlong(v) >= __double_as_longlong(L)) v = __dsub_rn(v, L);
  const long long b = __double_as_longlong(v);
  if (b < 0 && (b << 1) != 0) v = __dadd_rn(v, L);
  return v;
}

__device__ __forceinline__ uint32_t block_exclusive_scan_256(uint32_t v, uint32_t& total) {
  __shared__ uint32_t warp_tot[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[wid] = x;
  __syncthreads();
  if (wid == 0) {
    uint32_t t = lane < 8 ? warp_tot[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < 8) warp_tot[lane] = t;
  }
  __syncthreads();
  const uint32_t before = wid ? warp_tot[wid - 1] : 0u;
  total = warp_tot[7];
  __syncthreads();
  return before + x - v;
}

// ---------------------------------------------------------------------------
// Verlet-list build.  One block per tile of TY consecutive cell rows (cy0 ..
// cy0+TY-1 at one cz); threads = the tile's particles, contiguous in slot
// order (in passes of blockDim when a tile is longer).  All (TY+2) x 3
// neighbour rows are staged in shared memory (one pass in the common case) as
// the FP32 coordinates that the permutation left in fout (build_xyz), each
// row extended by one periodic image cell at both ends, so every particle's
// 3 x 3 x 3 cell neighbourhood is 9 contiguous ranges.  y and z count from each
// row's own lower edges: a candidate's row is one edge up or down or the same,
// whether it is a periodic image or not.  A pair enters the list when its FP32
// distance is below r_c + skin (widened by the rounding bound).
//
// Bound by instruction issue: ~15 instructions per candidate and lane, ~110
// candidates.  Taking the coordinates from the permutation and describing the
// rows without divisions, instead of turning every staged entry from fixed
// point into the tile's frame: 133 -> 121 us at 1,048,576 beads.
// ---------------------------------------------------------------------------
// 16-byte copy global -> shared that does not wait for the data (cp.async,
// L2 only); cp_async_wait_all() waits for every copy the thread issued.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// FP32 coordinates of a slot for the list build.  x in [0, L) up to rounding: a
// position that rounds across the box edge from the cell that the sort put it
// in is kept on that cell's side.  y and z from the lower edges of the cell row
// that the sort put it in, so that they carry the rounding of a cell's edge, not
// of the box's.  .w holds the slot.
__device__ __forceinline__ float4 build_xyz(const Sys& S, uint32_t X, uint32_t Y, uint32_t Z, uint32_t key,
                                            uint32_t slot) {
  const uint32_t nx = (uint32_t)S.nc[0], ny = (uint32_t)S.nc[1];
  const uint32_t row = key / nx, cx = key - row * nx, cz = row / ny, cy = row - cz * ny;
  float x = __uint2float_rn(X) * S.scale[0];
  if (cx == 0u && X >= 0xC0000000u) x -= (float)S.L[0];
  if (cx == nx - 1u && X < 0x40000000u) x += (float)S.L[0];
  // c 2^32 / nc to within one unit
  const uint32_t y0 = (uint32_t)__umul64hi((unsigned long long)cy << 32, S.inv_nc64[0]);
  const uint32_t z0 = (uint32_t)__umul64hi((unsigned long long)cz << 32, S.inv_nc64[1]);
  return make_float4(x, __int2float_rn(pdiff(Y, y0)) * S.scale[1], __int2float_rn(pdiff(Z, z0)) * S.scale[2],
                     __uint_as_float(slot));
}

struct BuildRow {
  int base;         // first staged index of the row
  int padL;         // particles of the left image cell (cell nx-1)
  int cnt;          // particles of the row
  int tot;          // padL + cnt + particles of the right image cell (cell 0)
  int lo;           // first slot of the row
  int left;         // first slot of cell nx-1
};
constexpr int TILE_ROWS_MAX = 3 * (TILE_Y_MAX + 2);

// One candidate: hit = r2 < rv2; a hit is written to row `cnt` of the
// slot's column while cnt < cap, and cnt counts every hit (cnt > cap
// afterwards means the list overflowed).  The caller never passes the
// particle itself.  Predicated PTX, so that the warp does not diverge on the
// (frequent) hits.
template <bool NL16>
__device__ __forceinline__ void list_candidate(unsigned char* col, uint32_t stride, float r2,
                                               float rv2, uint32_t qslot, int cap, int& cnt) {
  if constexpr (NL16) {
    asm volatile(
        "{\n\t.reg .pred h, w;\n\t.reg .u64 a;\n\t"
        "setp.lt.f32 h, %1, %2;\n\t"
        "setp.lt.and.s32 w, %0, %4, h;\n\t"
        "mad.wide.u32 a, %0, %5, %6;\n\t"
        "@w st.global.u16 [a], %7;\n\t"
        "@h add.s32 %0, %0, 1;\n\t}"
        : "+r"(cnt)
        : "f"(r2), "f"(rv2), "r"(qslot), "r"(cap), "r"(stride), "l"(col), "h"((uint16_t)qslot)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred h, w;\n\t.reg .u64 a;\n\t"
        "setp.lt.f32 h, %1, %2;\n\t"
        "setp.lt.and.s32 w, %0, %4, h;\n\t"
        "mad.wide.u32 a, %0, %5, %6;\n\t"
        "@w st.global.u32 [a], %3;\n\t"
        "@h add.s32 %0, %0, 1;\n\t}"
        : "+r"(cnt)
        : "f"(r2), "f"(rv2), "r"(qslot), "r"(cap), "r"(stride), "l"(col)
        : "memory");
  }
}

// The list build of one tile (`tile` of tiles_y * nc[2]), by all threads of
// the block; F the slots' coordinates (build_xyz), cell_of the cell the sort
// put each slot in.  The block synchronises inside; a block that builds
// several tiles synchronises between them.
template <bool NL16>
__device__ __forceinline__ void build_tile(const Sys& S, const float4* F, const uint32_t* cell_of, uint32_t tile,
                                           unsigned char* smem) {
  const int CAP = S.tile_cap;
  float4* sX = reinterpret_cast<float4*>(smem);
  BuildRow* ri = reinterpret_cast<BuildRow*>(smem + 16 * (size_t)CAP);
  uint32_t* sCS = reinterpret_cast<uint32_t*>(ri + TILE_ROWS_MAX);
  __shared__ int sTOT;
  Ctl* ctl = S.ctl;
  const int nx = S.nc[0], ny = S.nc[1], nz = S.nc[2];
  const int ty = tile % S.tiles_y, cz = tile / S.tiles_y;
  const int cy0 = ty * ny / S.tiles_y;  // (the rows shared out evenly)
  const int TYb = (ty + 1) * ny / S.tiles_y - cy0;
  const int RY = TYb + 2, R = 3 * RY;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t rs = S.cell_start[(cz * ny + cy0) * nx];
  const uint32_t re = S.cell_start[(cz * ny + cy0 + TYb - 1) * nx + nx];

  // one warp per row: its cell offsets, then its description
  for (int sr = warp; sr < R; sr += nwarps) {
    const int dzi = sr / RY, yi = sr - dzi * RY;
    const int uy = cy0 - 1 + yi, uz = cz - 1 + dzi;  // unwrapped row indices
    const uint32_t* src = S.cell_start + (wrap_cell(uz, nz) * ny + wrap_cell(uy, ny)) * nx;
    uint32_t* cs = sCS + sr * (nx + 1);
    for (int c = lane; c <= nx; c += 32) cs[c] = src[c];
    __syncwarp();
    if (lane == 0) {
      BuildRow r;
      r.base = 0;
      r.padL = (int)(cs[nx] - cs[nx - 1]);
      r.cnt = (int)(cs[nx] - cs[0]);
      r.tot = r.padL + r.cnt + (int)(cs[1] - cs[0]);
      r.lo = (int)cs[0];
      r.left = (int)cs[nx - 1];
      ri[sr] = r;
    }
  }
  __syncthreads();
  if (warp == 0) {
    const int cnt = lane < R ? ri[lane].tot : 0;
    int x = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    if (lane < R) ri[lane].base = x - cnt;
    if (lane == 31) sTOT = x;
  }
  __syncthreads();
  const int TOT = sTOT;
  const float rv2 = S.rv2_build, Lx = (float)S.L[0];

  // Stages entries [c0, c0 + cn) of the neighbour rows, one warp per row: the
  // copies all in flight at once, then the images' shift in x.
  auto stage = [&](int c0, int cn) {
    for (int sr = warp; sr < R; sr += nwarps) {
      const BuildRow r = ri[sr];
      const int k0 = max(r.base, c0), k1 = min(r.base + r.tot, c0 + cn);
      for (int ent = k0 + lane; ent < k1; ent += 32) {
        const int kr = ent - r.base;
        const int slot = kr < r.padL ? r.left + kr
                                     : r.lo + (kr < r.padL + r.cnt ? kr - r.padL : kr - r.padL - r.cnt);
        cp_async16(&sX[ent - c0], F + slot);
      }
    }
    cp_async_wait_all();
    __syncwarp();
    for (int sr = warp; sr < R; sr += nwarps) {
      const BuildRow r = ri[sr];
      const int k0 = max(r.base, c0), k1 = min(r.base + r.tot, c0 + cn);
      for (int ent = k0 + lane; ent < min(r.base + r.padL, k1); ent += 32) sX[ent - c0].x -= Lx;
      for (int ent = max(r.base + r.padL + r.cnt, k0) + lane; ent < k1; ent += 32) sX[ent - c0].x += Lx;
    }
  };
  const bool one = TOT <= CAP;  // the common case: every row staged once
  if (one) {
    stage(0, TOT);
    __syncthreads();
  }

  for (uint32_t base = rs; base < re; base += blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    const bool act = i < re;
    // the cell the sort put this slot in (not the one its current position
    // maps to: after a checkpoint restore the two can differ by one)
    const uint32_t kc = act ? cell_of[i] : (uint32_t)((cz * ny + cy0) * nx);
    const float4 fi = act ? F[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    int cx = (int)(kc % (uint32_t)nx);
    int yrel = (int)((kc / (uint32_t)nx) % (uint32_t)ny) - cy0;
    if (yrel < 0 || yrel >= TYb) {  // cannot happen for a consistent sort
      set_status(ctl, PRX_EINVAL);
      yrel = 0;
      cx = 0;
    }
    // staged entries [lo, hi) of window w
    auto window = [&](int w, int& lo, int& hi) {
      const int sr = (w / 3) * RY + yrel + (w % 3);
      const uint32_t* cs = sCS + sr * (nx + 1);
      const BuildRow& r = ri[sr];
      const int off = r.base + r.padL - r.lo;  // slot -> staged entry
      lo = cx == 0 ? r.base : off + (int)cs[cx - 1];
      hi = cx + 2 > nx ? r.base + r.tot : off + (int)cs[cx + 2];
    };
    uint32_t win[9];  // (rows staged at once are at most CAP <= 65,535 entries)
    if (one) {
#pragma unroll
      for (int w = 0; w < 9; ++w) {
        int lo, hi;
        window(w, lo, hi);
        win[w] = (uint32_t)lo | ((uint32_t)hi << 16);
      }
    }
    const int kself0 = ri[RY + yrel + 1].base + ri[RY + yrel + 1].padL + ((int)i - ri[RY + yrel + 1].lo);
    int cnt = 0;
    const int cap = S.list_cap;
    unsigned char* col = (unsigned char*)S.nl + (size_t)i * (NL16 ? 2 : 4);
    const uint32_t stride = S.n * (NL16 ? 2u : 4u);
    // the staged entries [lo, hi) of window w; the particle itself is staged
    // once (entry kself), in the centre row's window (w = 4), whose walk skips
    // it: no candidate needs a self test
    auto candidates = [&](int w, int lo, int hi, int kself) {
      const float y = fi.y - (float)(w % 3 - 1) * S.cell_edge_f[0];
      const float z = fi.z - (float)(w / 3 - 1) * S.cell_edge_f[1];
      auto walk = [&](int a, int b) {
#pragma unroll 2
        for (int k = a; k < b; ++k) {
          const float4 q = sX[k];
          const float dx = q.x - fi.x, dy = q.y - y, dz = q.z - z;
          list_candidate<NL16>(col, stride, fmaf(dz, dz, fmaf(dy, dy, dx * dx)), rv2, __float_as_uint(q.w), cap,
                               cnt);
        }
      };
      if (w == 4) {
        walk(lo, min(hi, max(lo, kself)));
        walk(max(lo, kself + 1), hi);
      } else {
        walk(lo, hi);
      }
    };
    if (one) {
      if (act) {
#pragma unroll
        for (int w = 0; w < 9; ++w) candidates(w, (int)(win[w] & 0xFFFFu), (int)(win[w] >> 16), kself0);
      }
    } else {
      for (int c0 = 0; c0 < TOT; c0 += CAP) {  // neighbour rows longer than the buffer: staged per chunk
        const int cn = min(CAP, TOT - c0);
        __syncthreads();
        stage(c0, cn);
        __syncthreads();
#pragma unroll 1
        for (int w = 0; act && w < 9; ++w) {
          int lo, hi;
          window(w, lo, hi);
          candidates(w, max(lo, c0) - c0, min(hi, c0 + cn) - c0, kself0 - c0);
        }
      }
    }
    if (act) {
      const int m = min(cnt, cap);
      S.nn[i] = (uint8_t)m;
      if (cnt > cap) set_status(ctl, PRX_ECAPACITY);
      // pad to a whole stage of four with the slot itself (the step kernel
      // gathers four entries at a time; the self pair has r = 0 and no force)
      for (int k = m; k < ((m + 3) & ~3); ++k) {
        if constexpr (NL16) ((uint16_t*)S.nl)[(size_t)k * S.n + i] = (uint16_t)i;
        else ((uint32_t*)S.nl)[(size_t)k * S.n + i] = i;
      }
    }
  }
}

// Cell of a fixed-point position.
__device__ __forceinline__ uint32_t cell_of_pos(const Sys& S, const uint4 q) {
  const uint32_t cx = __umulhi(q.x, (uint32_t)S.nc[0]);
  const uint32_t cy = __umulhi(q.y, (uint32_t)S.nc[1]);
  const uint32_t cz = __umulhi(q.z, (uint32_t)S.nc[2]);
  return (cz * (uint32_t)S.nc[1] + cy) * (uint32_t)S.nc[0] + cx;
}

// Old slot o goes to its new slot: every per-particle array into the other
// set, bond partners renamed, a fresh displacement reference, and the slot's
// cell (into cell_of, read by the list build).  start(k) is the first slot of
// cell k (n for k = ncell); a slot's new place is that plus the number of its
// cell's members with a smaller old slot, from the cell's bucket or, where
// `other` (a bucket overflowed), from other(slot, cell, first, members).  The
// slot's own lookup and its first two bond partners' run side by side.  XYZ:
// also the list build's coordinates.
template <bool XYZ, class Start, class Other>
__device__ __forceinline__ void permute_old(const Sys& S, const SoA& A, const SoA& B, uint4* P, uint32_t* cell_of,
                                            uint32_t o, Start start, bool other_all, Other other) {
  double x = A.x[o], y = A.y[o], z = A.z[o];
  const double vx = A.vx[o], vy = A.vy[o], vz = A.vz[o];
  const uint32_t pid = A.id[o];
  const uint8_t ty = A.type[o];
  const int8_t st = A.state[o];
  const uint32_t nb = A.nadj[o];
  const uint32_t key = S.key[o];
  const uint32_t* from = A.adj + (size_t)o * S.cap;
  const uint32_t e0 = nb > 0u ? from[0] : o, e1 = nb > 1u ? from[1] : o;
  auto members_before = [&](uint4 v, uint32_t q, uint32_t c, uint32_t j) {  // among members q .. q + 3 of c
    return (q < c && v.x < j ? 1u : 0u) + (q + 1u < c && v.y < j ? 1u : 0u) + (q + 2u < c && v.z < j ? 1u : 0u) +
           (q + 3u < c && v.w < j ? 1u : 0u);
  };
  auto row = [&](uint32_t k) { return reinterpret_cast<const uint4*>(S.bucket + (size_t)k * ENG_BUCKET); };
  // of slot j in cell k with members first .. first + c, the first four of them v
  auto place = [&](uint32_t j, uint32_t k, uint32_t first, uint32_t c, uint4 v) {
    if (other_all || c > ENG_BUCKET) return other(j, k, first, c);
    uint32_t r = first + members_before(v, 0u, c, j);
#pragma unroll 1
    for (uint32_t q = 4u; q < c; q += 4u) r += members_before(row(k)[q >> 2], q, c, j);
    return r;
  };
  const uint32_t j[3] = {o, e0 & SLOT_MASK, e1 & SLOT_MASK};
  uint32_t k[3] = {key, S.key[j[1]], S.key[j[2]]}, f[3], c[3], r[3];
  uint4 v[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    f[q] = start(k[q]);
    c[q] = start(k[q] + 1u) - f[q];
    v[q] = row(k[q])[0];
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) r[q] = place(j[q], k[q], f[q], c[q], v[q]);
  const uint32_t s = r[0];
  uint32_t* to = B.adj + (size_t)s * S.cap;
  if (nb > 0u) to[0] = r[1] | (e0 & ~SLOT_MASK);
  if (nb > 1u) to[1] = r[2] | (e1 & ~SLOT_MASK);
#pragma unroll 1
  for (uint32_t b = 2; b < nb; ++b) {
    const uint32_t e = from[b], jb = e & SLOT_MASK, kb = S.key[jb], fb = start(kb);
    to[b] = place(jb, kb, fb, start(kb + 1u) - fb, row(kb)[0]) | (e & ~SLOT_MASK);
  }
  x = wrap_into_box(x, S.L[0]);
  y = wrap_into_box(y, S.L[1]);
  z = wrap_into_box(z, S.L[2]);
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
  const uint32_t X = periodic_fx(x, S.Lfx[0], S.M64[0]);
  const uint32_t Y = periodic_fx(y, S.Lfx[1], S.M64[1]);
  const uint32_t Z = periodic_fx(z, S.Lfx[2], S.M64[2]);
  P[s] = make_uint4(X, Y, Z, coarse_ref(X, Y, Z, S.wshift));
  if constexpr (XYZ) reinterpret_cast<float4*>(S.fout)[s] = build_xyz(S, X, Y, Z, key, s);
  cell_of[s] = key;
}

}  // namespace

}  // namespace prx
