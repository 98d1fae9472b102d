// Canonical order of the bond list (step, a, t) on the device.
//
// The list's records stand in the order in which the warps of a reaction step
// reserved their places.  Sorted on the host (a stable sort of 24-byte records)
// a read-back of 460,000 bonds took 15 ms, as long as 170 steps of the million
// beads that hold them; here it takes well under 1 ms.  Tiles of 1,024 records by a bitonic network in
// shared memory, then merge passes in which every record finds its place by a
// binary search in the sibling run (~17 dependent L2 reads, hidden by the
// hundreds of thousands of records searching at once).  Both are stable: equal
// records keep their order.  Every pass writes a whole permutation of the list,
// so the list stays valid whichever buffer the last pass wrote.
#include <cuda_runtime.h>

#include "prx_internal.cuh"

namespace prx {

namespace {

constexpr int TILE = 1024;

struct Key {
  unsigned long long hi, lo;  // step (order of signed numbers), a:t
};
__device__ __forceinline__ Key key_of(const BondRec& r) {
  return Key{(unsigned long long)r.step ^ (1ull << 63), ((unsigned long long)r.a << 32) | r.t};
}
__device__ __forceinline__ bool less_key(const Key& x, const Key& y) {
  return x.hi < y.hi || (x.hi == y.hi && x.lo < y.lo);
}

// Sorts each tile of 1,024 records of `in` into `out`, by (key, place).
__global__ void __launch_bounds__(TILE / 2) k_bonds_tiles(const BondRec* __restrict__ in, BondRec* __restrict__ out,
                                                          uint32_t m) {
  __shared__ unsigned long long hi[TILE], lo[TILE];
  __shared__ uint16_t at[TILE];
  const uint32_t base = blockIdx.x * TILE;
  for (int q = threadIdx.x; q < TILE; q += TILE / 2) {
    Key k{~0ull, ~0ull};  // places past the list sort behind every record
    if (base + q < m) k = key_of(in[base + q]);
    hi[q] = k.hi, lo[q] = k.lo;
    at[q] = (uint16_t)q;
  }
  for (int size = 2; size <= TILE; size <<= 1) {
    for (int d = size >> 1; d > 0; d >>= 1) {
      __syncthreads();
      const int t = threadIdx.x;
      const int i = 2 * t - (t & (d - 1)), j = i + d;
      const bool up = (i & size) == 0;
      const Key x{hi[i], lo[i]}, y{hi[j], lo[j]};
      const uint16_t p = at[i], q = at[j];
      const bool gt = less_key(y, x) || (!less_key(x, y) && q < p);
      if (gt == up) {
        hi[i] = y.hi, lo[i] = y.lo, at[i] = q;
        hi[j] = x.hi, lo[j] = x.lo, at[j] = p;
      }
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < TILE; q += TILE / 2)
    if (base + q < m) out[base + q] = in[base + at[q]];
}

// Merges the sorted runs of w records of `in` in pairs: a record's place is
// its place in its own run plus the number of records of the sibling run
// that go before it (a smaller key, or an equal one from the first run).
__global__ void __launch_bounds__(256) k_bonds_merge(const BondRec* __restrict__ in, BondRec* __restrict__ out,
                                                     uint32_t m, uint32_t w) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const uint32_t run = i / w, first = run * w;
  const bool second = run & 1u;
  // the sibling run [s0, s1)
  const uint32_t s0 = second ? first - w : min(first + w, m), s1 = second ? first : min(first + 2u * w, m);
  const BondRec r = in[i];
  const Key k = key_of(r);
  uint32_t a = s0, b = s1;
  while (a < b) {
    const uint32_t mid = a + ((b - a) >> 1);
    const Key q = key_of(in[mid]);
    if (less_key(q, k) || (second && !less_key(k, q))) a = mid + 1u;
    else b = mid;
  }
  out[(second ? first - w : first) + (i - first) + (a - s0)] = r;
}

}  // namespace

// Sorts the first m records of `list`, with room for m records in `scratch`;
// returns the buffer that holds the sorted records.  `list` keeps all m
// records, in some order.
BondRec* launch_sort_bonds(BondRec* list, BondRec* scratch, uint32_t m, cudaStream_t st) {
  if (!m) return list;
  const unsigned tiles = (m + TILE - 1) / TILE;
  BondRec *from = list, *to = scratch;
  k_bonds_tiles<<<tiles, TILE / 2, 0, st>>>(from, to, m);
  for (uint64_t w = TILE; w < m; w *= 2u) {
    BondRec* t = from;
    from = to;
    to = t;
    k_bonds_merge<<<(m + 255u) / 256u, 256, 0, st>>>(from, to, m, (uint32_t)w);
  }
  return to;
}

}  // namespace prx
