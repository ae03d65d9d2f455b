// k_ising.cu -- checkerboard Metropolis half-sweeps of 2-D Ising lattices
// that consume the generators' draws (the Monte Carlo use the paper's
// generators serve; Section 3.5 cites RANMAR's earlier Ising simulations).
//
// Periodic L x L lattice, J = 1, h = 0, spins +1/-1 in int8, row-major.  A
// half-sweep visits the sites of one colour ((x + y) % 2); sites of one
// colour only neighbour the other colour, so they update independently.
// The site with colour rank k (k = y L/2 + x/2) takes draw k, whose 24-bit
// value r = draw >> shift decides the proposal with integer thresholds:
// accept when dE = 2 s (sum of neighbours) <= 0, or r < t4 (dE = 4), or
// r < t8 (dE = 8).  Thresholds are computed once on the host, so both the
// library and any checker take the same integer decision.
//
// Up to kIsingPerLaunch lattices go to one launch with their descriptors
// passed by value; a block works on one lattice (block ranges by prefix).
// Lattices whose rows split into 16-byte chunks (L a multiple of 16, both
// buffers 16-byte aligned, and a draw layout that keeps 8 consecutive
// ranks in one row) take the vector form: a thread owns 16 consecutive
// sites of four rows, 8 of them of the colour in each, and moves them as one
// 16-byte load and store per row (the rows above and below read too) and two
// 16-byte draw loads per row.  The others take the scalar form, a thread per site.
#include <cmath>

#include "../../include/prng.h"
#include "common.cuh"

namespace prng {

constexpr int kIsingPerLaunch = 96;
constexpr int kIsingThreads = 256;
constexpr int kIsingSitesPerThread = 4;

struct IsingLaunch {
  prng_ising_req r[kIsingPerLaunch];
  uint32_t block0[kIsingPerLaunch + 1];  // first block of each lattice
  uint32_t n;
};

__global__ void __launch_bounds__(kIsingThreads) k_ising_half_sweep(const __grid_constant__ IsingLaunch b) {
  // Lattice of this block: largest i with block0[i] <= blockIdx.x.
  uint32_t lo = 0, hi = b.n;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (b.block0[mid] <= blockIdx.x) lo = mid;
    else hi = mid;
  }
  const prng_ising_req& q = b.r[lo];
  const uint32_t L = q.L, half = L >> 1;
  const uint64_t sites = (uint64_t)L * half;
  const uint64_t base = (uint64_t)(blockIdx.x - b.block0[lo]) * kIsingThreads * kIsingSitesPerThread;
#pragma unroll
  for (int j = 0; j < kIsingSitesPerThread; j++) {
    const uint64_t k = base + (uint64_t)j * kIsingThreads + threadIdx.x;
    if (k >= sites) break;
    const uint32_t y = (uint32_t)(k / half);
    const uint32_t x = 2 * (uint32_t)(k - (uint64_t)y * half) + ((y + q.colour) & 1u);
    const uint32_t yu = y == 0 ? L - 1 : y - 1, yd = y + 1 == L ? 0 : y + 1;
    const uint32_t xl = x == 0 ? L - 1 : x - 1, xr = x + 1 == L ? 0 : x + 1;
    int8_t* row = q.d_spins + (uint64_t)y * L;
    const int s = row[x];
    const int nb = q.d_spins[(uint64_t)yu * L + x] + q.d_spins[(uint64_t)yd * L + x] + row[xl] + row[xr];
    const int dE = 2 * s * nb;
    uint64_t di = k;
    if (q.pitch != 0) {   // k < 2^31: 32-bit quotient, a shift when per is a power of two
      const uint32_t k32 = (uint32_t)k, per = q.per;
      const uint32_t row = (per & (per - 1)) == 0 ? k32 >> (__ffs(per) - 1) : k32 / per;
      di = (uint64_t)row * q.pitch + (k32 - row * per);
    }
    const uint32_t r = q.d_draws[di] >> q.shift;
    const bool accept = dE <= 0 || (dE == 4 ? r < q.t4 : r < q.t8);
    if (accept) row[x] = (int8_t)(-s);
  }
}

// Vector form: a thread owns kIsingRows rows of 16 consecutive sites and updates
// the 8 sites of the colour in each, four at a time as the bytes of a word.
//
// A spin byte is 0x01 or 0xFF, so two spins' XOR is 0x00 (aligned) or 0xFE, and
// with the four neighbours' XORs e the site's class is bit logic on whole words:
// two or more e set: dE <= 0, flip; exactly one: dE = 4; none: dE = 8.  The draw
// decides the last two by d < t << shift, which is (d >> shift) < t without the
// shift (always, when t << shift passes 32 bits).  A flip is XOR 0xFE.  The
// 16-byte store also rewrites the 8 sites of the other colour with the values it
// read: nothing changes them during the half-sweep, so readers of those
// neighbours see the same bytes.
//
// What bounds it is DRAM: per site updated 2 bytes of spins read and 2 written
// (both colours' bytes) and 4 of draws.  The site-by-site form it replaces
// (compare, multiply and select per site on bytes, one row per thread) ran 340
// instructions per 8 updates and was bound by their issue: 11 lattices of 4096^2
// 179 -> 135 us, 4 of them 58 -> 37, 16 of 1024^2 15 -> 11; smaller launches cost
// what a launch costs in both.
constexpr int kIsingVecThreads = 256;
constexpr int kIsingRows = 4;

__device__ __forceinline__ uint32_t ising_lattice_of(const IsingLaunch& b) {
  uint32_t lo = 0, hi = b.n;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (b.block0[mid] <= blockIdx.x) lo = mid;
    else hi = mid;
  }
  return lo;
}

// q = a / b, by a shift when b is a power of two.
__device__ __forceinline__ uint32_t div_pow2(uint32_t a, uint32_t b) {
  return (b & (b - 1)) == 0 ? a >> (31 - __clz(b)) : a / b;
}

__global__ void __launch_bounds__(kIsingVecThreads) k_ising_half_sweep_v(const __grid_constant__ IsingLaunch b) {
  const uint32_t lo = ising_lattice_of(b);
  const prng_ising_req& q = b.r[lo];
  const uint32_t L = q.L, cpr = L >> 4;                      // 16-site chunks per row
  const uint32_t unit = (blockIdx.x - b.block0[lo]) * kIsingVecThreads + threadIdx.x;
  if (unit >= L / kIsingRows * cpr) return;                  // L <= 65520: L * L / 64 < 2^26
  const uint32_t strip = div_pow2(unit, cpr);
  const uint32_t y0 = strip * kIsingRows, x0 = (unit - strip * cpr) << 4;
  const uint64_t w4 = (uint64_t)q.t4 << q.shift, w8 = (uint64_t)q.t8 << q.shift;
  const uint32_t t4 = (uint32_t)w4, t8 = (uint32_t)w8;
  const uint32_t always4 = w4 >> 32 ? 0xFEFEFEFEu : 0u, always8 = w8 >> 32 ? 0xFEFEFEFEu : 0u;
  int8_t* const col = q.d_spins + x0;

  uint4 row[kIsingRows + 2];   // rows y0 - 1 .. y0 + kIsingRows
#pragma unroll
  for (int i = 0; i < kIsingRows + 2; i++) {
    uint32_t y = y0 + i - 1;
    if (i == 0 && y0 == 0) y = L - 1;
    if (i == kIsingRows + 1 && y == L) y = 0;
    row[i] = *reinterpret_cast<const uint4*>(col + (uint64_t)y * L);
  }
  uint4 d[kIsingRows][2];
  uint32_t side[kIsingRows];   // the neighbour beside the chunk: before it, or behind it
#pragma unroll
  for (int i = 0; i < kIsingRows; i++) {
    const uint32_t y = y0 + i, par = (y + q.colour) & 1u;     // x parity of the colour in row y
    const uint32_t k0 = y * (L >> 1) + (x0 >> 1);              // colour rank of the first site
    uint64_t di = k0;
    if (q.pitch != 0) {   // 8 ranks never straddle a row of `per` (per % 8 == 0)
      const uint32_t pr = div_pow2(k0, q.per);
      di = (uint64_t)pr * q.pitch + (k0 - pr * q.per);
    }
    d[i][0] = __ldcs(reinterpret_cast<const uint4*>(q.d_draws + di));
    d[i][1] = __ldcs(reinterpret_cast<const uint4*>(q.d_draws + di + 4));
    const uint32_t xs = par ? (x0 + 16 == L ? 0 : x0 + 16) : (x0 == 0 ? L - 1 : x0 - 1);
    side[i] = (uint8_t)q.d_spins[(uint64_t)y * L + xs];
  }
#pragma unroll
  for (int i = 0; i < kIsingRows; i++) {
    const bool odd = ((y0 + i + q.colour) & 1u) != 0;
    const uint4 C = row[i + 1], U = row[i], D = row[i + 2];
    // Bytes of the colour (and, in the row itself, of the other one), in order.
    const uint32_t mine = odd ? 0x7531u : 0x6420u, other = odd ? 0x6420u : 0x7531u;
    const uint32_t c0 = __byte_perm(C.x, C.y, mine), c1 = __byte_perm(C.z, C.w, mine);
    const uint32_t o0 = __byte_perm(C.x, C.y, other), o1 = __byte_perm(C.z, C.w, other);
    // The other neighbour in the row: one place before (even sites) or behind (odd ones).
    const uint32_t s0 = __byte_perm(o0, odd ? o1 : side[i], odd ? 0x4321u : 0x2104u);
    const uint32_t s1 = __byte_perm(o1, odd ? side[i] : o0, odd ? 0x4321u : 0x2107u);
    const uint32_t f0 = ising_flips4(c0, __byte_perm(U.x, U.y, mine), __byte_perm(D.x, D.y, mine), o0, s0, d[i][0],
                                     t4, t8, always4, always8);
    const uint32_t f1 = ising_flips4(c1, __byte_perm(U.z, U.w, mine), __byte_perm(D.z, D.w, mine), o1, s1, d[i][1],
                                     t4, t8, always4, always8);
    const uint32_t lo2 = odd ? 0x1404u : 0x4140u, hi2 = odd ? 0x3424u : 0x4342u;
    uint4 O;
    O.x = C.x ^ __byte_perm(f0, 0, lo2);
    O.y = C.y ^ __byte_perm(f0, 0, hi2);
    O.z = C.z ^ __byte_perm(f1, 0, lo2);
    O.w = C.w ^ __byte_perm(f1, 0, hi2);
    *reinterpret_cast<uint4*>(col + (uint64_t)(y0 + i) * L) = O;
  }
}

// Whether a lattice can take the vector form.
static bool ising_vec_ok(const prng_ising_req& q) {
  return (q.L & 15u) == 0 && q.L <= 65520 && (reinterpret_cast<uintptr_t>(q.d_spins) & 15) == 0 &&
         (reinterpret_cast<uintptr_t>(q.d_draws) & 15) == 0 &&
         (q.pitch == 0 || ((q.per & 7u) == 0 && (q.pitch & 3u) == 0));
}

}  // namespace prng

using namespace prng;

extern "C" int prng_ising_half_sweep(const prng_ising_req* reqs, uint32_t n, void* stream) {
  if (n == 0) return PRNG_OK;
  if (reqs == nullptr) return PRNG_ENULL;
  for (uint32_t i = 0; i < n; i++) {
    const prng_ising_req& q = reqs[i];
    if (q.d_spins == nullptr || q.d_draws == nullptr) return PRNG_ENULL;
    if (q.L < 2 || (q.L & 1) != 0 || q.colour > 1 || q.shift > 8) return PRNG_ESIZE;
    if (q.pitch != 0 && (q.per == 0 || q.per > q.pitch)) return PRNG_ESIZE;
    if ((reinterpret_cast<uintptr_t>(q.d_draws) & 3) != 0) return PRNG_ESIZE;
  }
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  // Each group of up to kIsingPerLaunch lattices: the vector-form ones in one
  // launch, the rest in another (a thread per 4 x 16 sites / per 4 sites).
  for (int vec = 1; vec >= 0; vec--) {
    const uint64_t per_block = vec ? (uint64_t)kIsingVecThreads * 16 * kIsingRows
                                   : (uint64_t)kIsingThreads * kIsingSitesPerThread * 2;
    IsingLaunch b;
    b.n = 0;
    uint64_t blocks = 0;
    auto flush = [&]() -> bool {
      if (b.n == 0) return true;
      if (blocks > 0x7FFFFFFFull) return false;
      b.block0[b.n] = (uint32_t)blocks;
      if (vec) k_ising_half_sweep_v<<<(unsigned)blocks, kIsingVecThreads, 0, s>>>(b);
      else k_ising_half_sweep<<<(unsigned)blocks, kIsingThreads, 0, s>>>(b);
      b.n = 0;
      blocks = 0;
      return cudaGetLastError() == cudaSuccess;
    };
    for (uint32_t i = 0; i < n; i++) {
      if (ising_vec_ok(reqs[i]) != (vec == 1)) continue;
      b.r[b.n] = reqs[i];
      b.block0[b.n] = (uint32_t)blocks;
      blocks += ((uint64_t)reqs[i].L * reqs[i].L + per_block - 1) / per_block;   // L * L sites
      if (++b.n == (uint32_t)kIsingPerLaunch && !flush()) return blocks > 0x7FFFFFFFull ? PRNG_ESIZE : PRNG_ECUDA;
    }
    if (!flush()) return blocks > 0x7FFFFFFFull ? PRNG_ESIZE : PRNG_ECUDA;
  }
  return PRNG_OK;
}

extern "C" int prng_ising_thresholds(double beta, uint32_t* t4, uint32_t* t8) {
  if (t4 == nullptr || t8 == nullptr) return PRNG_ENULL;
  if (!(beta >= 0.0)) return PRNG_ESIZE;
  *t4 = (uint32_t)std::floor(16777216.0 * std::exp(-4.0 * beta));
  *t8 = (uint32_t)std::floor(16777216.0 * std::exp(-8.0 * beta));
  return PRNG_OK;
}
