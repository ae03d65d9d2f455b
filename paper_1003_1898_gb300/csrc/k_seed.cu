// k_seed.cu -- on-device seeding of every stream of a handle (the paper
// initialises its lag tables on the GPU too, Section 3.1).
//
// Stream i takes s = splitmix64(seed + i) and maps it into its generator's
// seed range, then runs the generator's own table initialisation:
//   GGL      x0 = 1 + s mod (2^31 - 2)
//   XOR128   (x, y, z, w) = 32-bit halves of s and of splitmix64(s)
//   RANECU   s1 = 1 + lo32(s) mod (m1 - 1), s2 = 1 + hi32(s) mod (m2 - 1)
//   RANMAR   RMARIN(ij = lo32(s) mod 31329, kl = hi32(s) mod 30082)
//   RANLUX   24 words from the MLCG 40014 mod 2147483563 started at
//            s mod 2147483563 (19780503 when that is 0), carry = (x_{-1} == 0)
//   MT19937  init_genrand(lo32(s))
//
// Also the host helpers the launchers share: the SM count, and the
// retained stream-ordered scratch pool of the jump fills.
#include <mutex>

#include "batch.cuh"
#include "scratch.cuh"

namespace prng {

// RMARIN (James 1988, cited by Section 3.5): 97 entries of 24 bits, most
// significant bit first, from the lagged product generator m <- i j k mod 179
// and the LCG l <- (53 l + 1) mod 169.  Written in canonical order V[k] = U[97 -
// k].
//
// Both sequences jump, so the entries need not wait for one another: 179 is
// prime and no term is 0, so with logarithms to the base 2 (a primitive root of
// 179) a term is i^A j^B k^C, the exponents a tribonacci sequence mod 178; and n
// LCG steps are l -> 53^n l + c mod 169.  kRmarin holds them for the start of
// every entry (24 steps each).  A thread takes `cnt` entries from entry e0 on:
// one thread for all of them (2,328 serial steps) took 76 us to re-seed up to 4,096
// streams and 328 for 131,072; now 7, 12 (4,096 streams) and 206, integer-bound.
struct Rmarin {
  uint8_t log[179], exp[178];
  uint8_t e[97][3][3];   // exponents of (i, j, k) for the three terms before entry e
  uint8_t a[97], c[97];  // LCG: l -> a l + c mod 169
};
constexpr Rmarin make_rmarin() {
  Rmarin t{};
  uint32_t x = 1;
  for (int n = 0; n < 178; n++) {
    t.exp[n] = (uint8_t)x;
    t.log[x] = (uint8_t)n;
    x = 2 * x % 179;
  }
  uint32_t w[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}}, a = 1, c = 0;
  for (int e = 0; e < 97; e++) {
    for (int r = 0; r < 3; r++)
      for (int v = 0; v < 3; v++) t.e[e][r][v] = (uint8_t)w[r][v];
    t.a[e] = (uint8_t)a;
    t.c[e] = (uint8_t)c;
    for (int k = 0; k < 24; k++) {
      for (int v = 0; v < 3; v++) {
        const uint32_t m = (w[0][v] + w[1][v] + w[2][v]) % 178;
        w[0][v] = w[1][v];
        w[1][v] = w[2][v];
        w[2][v] = m;
      }
      a = 53 * a % 169;
      c = (53 * c + 1) % 169;
    }
  }
  return t;
}
__device__ constexpr Rmarin kRmarin = make_rmarin();

__device__ void rmarin_entries(uint32_t ij, uint32_t kl, uint32_t* st, uint64_t n, uint64_t row, int e0, int cnt) {
  const uint32_t li = kRmarin.log[(ij / 177) % 177 + 2], lj = kRmarin.log[ij % 177 + 2],
                 lk = kRmarin.log[(kl / 169) % 178 + 1];
  uint32_t v[3];
#pragma unroll
  for (int r = 0; r < 3; r++)
    v[r] = kRmarin.exp[(kRmarin.e[e0][r][0] * li + kRmarin.e[e0][r][1] * lj + kRmarin.e[e0][r][2] * lk) % 178];
  uint32_t i = v[0], j = v[1], k = v[2], l = (kRmarin.a[e0] * (kl % 169) + kRmarin.c[e0]) % 169;
  for (int e = e0; e < e0 + cnt; e++) {
    uint32_t acc = 0;
#pragma unroll 8
    for (int b = 0; b < 24; b++) {
      const uint32_t m = i * j * k % 179;   // below 179^3: one reduction does
      i = j;
      j = k;
      k = m;
      l = (53 * l + 1) % 169;
      acc = 2 * acc + ((l * m >> 5) & 1u);
    }
    st[(uint64_t)(96 - e) * n + row] = acc;
  }
  if (e0 == 0) st[97 * n + row] = 362436u;  // C_0 = 362436 / 2^24
}

// Stream `row` of a RANMAR handle: its entries e0 .. e0 + cnt - 1.
__device__ void seed_ranmar(uint64_t seed, uint64_t n, uint32_t* st, uint64_t row, int e0, int cnt) {
  const uint64_t s = splitmix64(seed + row);
  rmarin_entries((uint32_t)s % 31329u, (uint32_t)(s >> 32) % 30082u, st, n, row, e0, cnt);
}

// Seed stream `row` of a handle of n streams (state layout in common.cuh).
__device__ void seed_stream(int gen, uint64_t seed, uint64_t n, uint32_t* st, uint64_t row) {
  const uint64_t s = splitmix64(seed + row);
  const uint32_t lo = (uint32_t)s, hi = (uint32_t)(s >> 32);
  switch (gen) {
    case GGL:
      st[row] = (uint32_t)(1 + s % 2147483646ull);
      break;
    case XOR128: {
      const uint64_t t = splitmix64(s);
      uint32_t z = (uint32_t)t, w = (uint32_t)(t >> 32);
      if ((lo | hi | z | w) == 0) w = 1;
      st[row] = lo;
      st[n + row] = hi;
      st[2 * n + row] = z;
      st[3 * n + row] = w;
      break;
    }
    case RANECU:
      st[row] = 1 + lo % 2147483562u;
      st[n + row] = 1 + hi % 2147483398u;
      break;
    case RANMAR:
      rmarin_entries(lo % 31329u, hi % 30082u, st, n, row, 0, 97);
      break;
    case RANLUX: {
      uint32_t x = (uint32_t)(s % 2147483563ull);
      if (x == 0) x = 19780503u;
      uint32_t last = 0;
      for (int k = 0; k < 24; k++) {
        x = mlcg_step<40014u, 85u>(x);
        last = x & 0xFFFFFFu;
        st[(uint64_t)k * n + row] = last;
      }
      st[24 * n + row] = (last == 0) ? 1u : 0u;
      break;
    }
    case MT19937: {
      uint4* mt = reinterpret_cast<uint4*>(st + row * 624);   // 16-byte stores: four words a step
      uint4 q;
      q.w = lo;
      for (uint32_t k = 0; k < 624; k += 4) {
        q.x = k == 0 ? lo : 1812433253u * (q.w ^ (q.w >> 30)) + k;
        q.y = 1812433253u * (q.x ^ (q.x >> 30)) + k + 1;
        q.z = 1812433253u * (q.y ^ (q.y >> 30)) + k + 2;
        q.w = 1812433253u * (q.z ^ (q.z >> 30)) + k + 3;
        mt[k / 4] = q;
      }
      break;
    }
  }
}

__global__ void k_seed(int gen, uint64_t seed, uint64_t n, uint32_t* st) {
  const uint64_t row = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row < n) seed_stream(gen, seed, n, st, row);
}

// RANMAR handles: a thread per stream and G entries (blockIdx.y counts them).
__global__ void __launch_bounds__(128) k_seed_ranmar(uint64_t seed, uint64_t n, uint32_t* st, int G) {
  const uint64_t row = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int e0 = blockIdx.y * G;
  if (row < n) seed_ranmar(seed, n, st, row, e0, e0 + G < 97 ? G : 97 - e0);
}

// Persistent seeding of every re-seeded request of a batch: an item is up
// to 256 consecutive streams of one request.
__global__ void __launch_bounds__(256) k_batch_seed(const BatchQueue q) {
  __shared__ uint32_t slot;
  for (;;) {
    const uint32_t it = pop_cta(q.counter, &slot);
    if (it >= q.n_items) break;
    const BatchItem I = q.items[it];
    const BatchReq& r = q.reqs[I.req];
    if (r.gen == RANMAR) {   // the fewer streams, the fewer entries per thread
      const uint32_t G = I.rows < 16 ? 1 : I.rows / 8, groups = (97 + G - 1) / G;
      for (uint32_t u = threadIdx.x; u < I.rows * groups; u += 256) {
        const uint32_t g = u / I.rows, e0 = g * G;
        seed_ranmar(r.seed, r.d.n_rows, r.d.state, I.row0 + (u - g * I.rows), (int)e0,
                    (int)(e0 + G < 97 ? G : 97 - e0));
      }
    } else if (threadIdx.x < I.rows) {
      seed_stream(r.gen, r.seed, r.d.n_rows, r.d.state, I.row0 + threadIdx.x);
    }
  }
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    n = (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0) ? v : 1;
  }
  return n;
}

namespace {
constexpr int kMaxPoolDevices = 64;
std::mutex g_pool_lock;
cudaMemPool_t g_pool[kMaxPoolDevices] = {};
}  // namespace

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxPoolDevices) return cudaErrorInvalidDevice;
  cudaMemPool_t pool;
  {
    std::lock_guard<std::mutex> guard(g_pool_lock);
    if (g_pool[dev] == nullptr) {
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      e = cudaMemPoolCreate(&pool, &props);
      if (e != cudaSuccess) return e;
      // Freed blocks stay for the next call up to 1 GiB (the largest MT19937 jump fill
      // takes 179 MB, a serving tick's RANLUX starts some 10 MB); more goes back to the
      // device at the next synchronisation.
      uint64_t keep = 1ull << 30;
      e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
      if (e != cudaSuccess) {
        cudaMemPoolDestroy(pool);
        return e;
      }
      g_pool[dev] = pool;
    }
    pool = g_pool[dev];
  }
  return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

cudaError_t scratch_free(void* p, cudaStream_t s) { return cudaFreeAsync(p, s); }

cudaError_t launch_batch_seed(const BatchQueue& q, cudaStream_t s) {
  if (q.n_items == 0) return cudaSuccess;
  const uint32_t cap = (uint32_t)sm_count() * 8;
  k_batch_seed<<<q.n_items < cap ? q.n_items : cap, 256, 0, s>>>(q);
  return cudaGetLastError();
}

cudaError_t launch_seed(int gen, int p, uint64_t seed, uint64_t n, uint32_t* state, cudaStream_t s) {
  (void)p;
  if (n == 0) return cudaSuccess;
  if (gen == RANMAR) {
    // Enough threads to fill the GPU; the jump to an entry costs about one entry.
    const uint64_t want = (uint64_t)sm_count() * 2048;
    int G = 97;
    while (G > 1 && n * ((97 + G - 1) / G) < want) G = (G + 1) / 2;
    k_seed_ranmar<<<dim3((unsigned)((n + 127) / 128), (unsigned)((97 + G - 1) / G)), 128, 0, s>>>(seed, n, state, G);
    return cudaGetLastError();
  }
  const int T = gen == MT19937 ? 64 : 256;
  k_seed<<<(unsigned)((n + T - 1) / T), T, 0, s>>>(gen, seed, n, state);
  return cudaGetLastError();
}

}  // namespace prng
