// k_simple.cu -- staged bulk fill of the register-state generators XOR128
// (Section 3.3), which has no cheap jump-ahead, and GGL (Section 3.2) and
// RANECU (Section 3.4), whose fills can also run lane-parallel (k_mlcg.cu;
// the launch tile selects which).
//
// One thread owns one stream (or one jump chunk) with its state in
// registers.  Output is stream-major, so a warp's 32 streams write 32
// different rows: each thread drafts K consecutive draws into its row of a
// shared-memory tile with 16-byte stores, then the CTA writes the tile out
// row by row (each 16-byte store instruction of a warp covers whole
// 128-byte runs of rows),
// which turns the per-thread sequences into coalesced HBM writes.  With S = 2
// tiles one barrier per tile suffices; S = 1 halves the shared memory per
// stream (two barriers per tile) so that every stream of a large handle can
// be resident at once instead of running a partial second wave.
#include <algorithm>

#include "batch.cuh"
#include "scratch.cuh"

namespace prng {

struct GglGen {
  static constexpr int SH = 7, WB = 31;
  static constexpr bool JUMPS = true;
  uint32_t x;
  // Row of a jump fill: x0 a^k mod m (Appendix A, eq. MLCG).
  __device__ __forceinline__ void jump_start(uint64_t x0, uint64_t k) {
    x = mulmod_pm<1u>(powmod_pm<1u>(16807u, k), (uint32_t)x0);
  }
  __device__ __forceinline__ void load(const uint32_t* st, uint64_t n, uint64_t row) { x = st[row]; }
  __device__ __forceinline__ void store(uint32_t* st, uint64_t n, uint64_t row) const { st[row] = x; }
  __device__ __forceinline__ void zero() { x = 1; }
  // x <- 16807 x mod (2^31 - 1)  (Section 3.2 constants).
  __device__ __forceinline__ uint32_t next() {
    x = mlcg_step<16807u, 1u>(x);
    return x;
  }
};

struct RanecuGen {
  static constexpr int SH = 7, WB = 31;
  static constexpr bool JUMPS = true;
  uint32_t s1, s2;
  // Row of a jump fill: each component jumped separately from x0 = s1 | s2 << 32.
  __device__ __forceinline__ void jump_start(uint64_t x0, uint64_t k) {
    s1 = mulmod_pm<85u>(powmod_pm<85u>(40014u, k), (uint32_t)(x0 & 0xFFFFFFFFu));
    s2 = mulmod_pm<249u>(powmod_pm<249u>(40692u, k), (uint32_t)(x0 >> 32));
  }
  __device__ __forceinline__ void load(const uint32_t* st, uint64_t n, uint64_t row) {
    s1 = st[row];
    s2 = st[n + row];
  }
  __device__ __forceinline__ void store(uint32_t* st, uint64_t n, uint64_t row) const {
    st[row] = s1;
    st[n + row] = s2;
  }
  __device__ __forceinline__ void zero() { s1 = s2 = 1; }
  // Section 3.4: m1 = 2147483563 = 2^31 - 85, m2 = 2147483399 = 2^31 - 249;
  // combination z = s1 - s2, plus m1 - 1 when z < 1 (Appendix A, "Multiple
  // recursive generators").
  __device__ __forceinline__ uint32_t next() {
    s1 = mlcg_step<40014u, 85u>(s1);
    s2 = mlcg_step<40692u, 249u>(s2);
    int32_t z = (int32_t)s1 - (int32_t)s2;
    z += (z < 1) ? 2147483562 : 0;
    return (uint32_t)z;
  }
};

struct Xor128Gen {
  static constexpr int SH = 8, WB = 32;
  static constexpr bool JUMPS = false;
  uint32_t x, y, z, w;
  __device__ __forceinline__ void load(const uint32_t* st, uint64_t n, uint64_t row) {
    x = st[row];
    y = st[n + row];
    z = st[2 * n + row];
    w = st[3 * n + row];
  }
  __device__ __forceinline__ void store(uint32_t* st, uint64_t n, uint64_t row) const {
    st[row] = x;
    st[n + row] = y;
    st[2 * n + row] = z;
    st[3 * n + row] = w;
  }
  __device__ __forceinline__ void zero() { x = y = z = 0; w = 1; }
  // Appendix A, "XORShift", scalar form of XOR128 with shifts 11, 19, 8.
  __device__ __forceinline__ uint32_t next() {
    const uint32_t t = x ^ (x << 11);
    x = y;
    y = z;
    z = w;
    w = (w ^ (w >> 19)) ^ (t ^ (t >> 8));
    return w;
  }
};

template <class G, int OM>
__device__ __forceinline__ uint32_t conv(uint32_t v) {
  if constexpr (OM == OUT_F32) return as_f32_bits<G::SH>(v);
  else return v;   // u32, or a raw draw paired at the copy-out
}

// Row-major tile, thread t's K staged draws in row t.  16-byte chunk ch of
// row t is stored at chunk slot ch ^ (t & 7): eight consecutive threads
// writing the same chunk, or eight lanes reading eight chunks of one row,
// touch eight different bank quads, without padding the rows.
template <int K>
__device__ __forceinline__ int swz(int row, int ch) { return ch ^ (row & 7); }

// Copy-out of a staged tile that is not plain: columns [c0, c0 + w) of rows
// [row0, row0 + T), with fewer columns than the tile's, unaligned rows, or rows
// that a batched request's or a jump fill's limit cuts.  Not inlined: inside the
// column loop it cost the plain copy-out 11 % (256 x 4,096 f32 70 -> 78 us).
template <class G, int T, int K, int OM>
__device__ __noinline__ void odd_tile(const FillDesc& d, const uint32_t* t, uint64_t row0, uint64_t c0, int w) {
  constexpr int CH = K / 4, RS = T / CH, NW = T / 32;
  __builtin_assume(__isShared(t));
  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const uint64_t pitch = d.pitch, limit = d.limit;
  const int rows = d.n_rows - row0 < (uint64_t)T ? (int)(d.n_rows - row0) : T;
  uint32_t* out = static_cast<uint32_t*>(d.out);
  const bool aligned = ((pitch & 3) == 0) && ((reinterpret_cast<uintptr_t>(out) & 15) == 0);
  const bool cut = (row0 + rows - 1) * pitch + c0 + w > limit;
  if (OM != OUT_ISING && (w & 3) == 0 && aligned) {   // whole 16-byte chunks, but for the cut one
    const int cch = tid % CH;
    if (4 * cch >= w) return;
#pragma unroll 4
    for (int r = tid / CH; r < rows; r += RS) {
      const uint64_t e = (row0 + r) * pitch + c0 + 4 * cch;
      const uint4 v = *reinterpret_cast<const uint4*>(t + r * K + 4 * swz<K>(r, cch));
      if (e + 4 <= limit) {
        st_chunk<OM, G::WB>(out + e, v);
      } else if constexpr (OM != OUT_F64) {           // doubles have no limit
        if (e < limit) st_out(out + e, v.x);
        if (e + 1 < limit) st_out(out + e + 1, v.y);
        if (e + 2 < limit) st_out(out + e + 2, v.z);
      }
    }
    return;
  }
  if constexpr (OM == OUT_ISING) {
    // Sites of the whole tile by rank, a thread per chunk of four or per site.  (A
    // warp per row, one lane per site, left most lanes idle in the rows of a few
    // sites that such tiles hold, each update waiting for the one before: a sweep of
    // 256^2 over 16,384 streams 37 us, here 14, the time of its two calls.)
    const bool quads = d.ising.vec4 && (w & 3) == 0 && (pitch & 3) == 0;   // c0 is a multiple of 32
    const int per = quads ? w >> 2 : w;
    for (int i = tid; i < rows * per; i += T) {
      const int r = i / per, c = quads ? 4 * (i - r * per) : i - r * per;
      const uint64_t e = (row0 + r) * pitch + c0 + c;
      const uint32_t* word = t + r * K + 4 * swz<K>(r, c >> 2) + (c & 3);
      if (quads) put4<OM, G::WB>(d, nullptr, e, *reinterpret_cast<const uint4*>(word));
      else if (e < limit) put1<OM>(d, nullptr, e, *word);
    }
    return;
  }
  // Word by word (or double by double), lanes on consecutive columns, eight rows of
  // a lane in flight.  (A row at a time, from a pointer not known to be in shared
  // memory, each cost about 1 us a tile: 256 x 61 doubles 23 us inside the column
  // loop as it once stood, 27 that way, here 10.)
  if constexpr (OM == OUT_F64) {   // w, the row starts and the limit are even
    constexpr int PR = K / 2, RW = 32 / PR;   // pairs per row, rows per warp and step
    const int c = 2 * (lane % PR), sub = lane / PR;
    for (int q0 = wi; q0 * RW < rows; q0 += 8 * NW) {
      uint2 v[8];
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int r = (q0 + i * NW) * RW + sub;
        v[i] = *reinterpret_cast<const uint2*>(t + r * K + 4 * swz<K>(r, c >> 2) + (c & 3));
      }
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int r = (q0 + i * NW) * RW + sub;
        const uint64_t e = (row0 + r) * pitch + c0 + c;
        if (r < rows && c < w && (!cut || e < limit)) st_pair<G::WB>(out + e, v[i].x, v[i].y);
      }
    }
  } else {
    for (int r0 = wi; r0 < rows; r0 += 8 * NW) {
      uint32_t v[8][K / 32];
#pragma unroll
      for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < K / 32; j++) {
          const int r = r0 + i * NW, c = lane + 32 * j;
          v[i][j] = t[r * K + 4 * swz<K>(r, c >> 2) + (c & 3)];
        }
      uint64_t e = (row0 + r0) * pitch + c0 + lane;
#pragma unroll
      for (int i = 0; i < 8; i++) {
#pragma unroll
        for (int j = 0; j < K / 32; j++)
          if (r0 + i * NW < rows && lane + 32 * j < w && (!cut || e + 32 * j < limit))
            st_out(out + e + 32 * j, v[i][j]);
        e += NW * pitch;
      }
    }
  }
}

// Streams [row0, row0 + T) of a fill, one per thread; smem holds S tiles of
// T * K words.  The n draws go to columns col0 .. col0 + n - 1; the states are
// read from d.state and left in `store_to` (nullptr: nowhere).
template <class G, int T, int K, int S, int OM>
__device__ __forceinline__ void simple_rows(const FillDesc& d, uint64_t row0, uint32_t* smem, uint64_t col0,
                                            uint64_t n, uint32_t* store_to) {
  static_assert(K % 32 == 0, "tile rows hold whole 8-chunk swizzle groups");
  constexpr int CH = K / 4;          // 16-byte chunks per row
  constexpr int RS = T / CH;         // rows one copy-out pass of the CTA covers
  static_assert(RS % 8 == 0, "copy-out rows of one thread must share a swizzle phase");
  const int tid = threadIdx.x;
  const uint64_t row = row0 + tid;
  const bool active = row < d.n_rows;

  G g;
  if (!active) {
    g.zero();
  } else if constexpr (G::JUMPS) {
    if (d.jump) g.jump_start(d.x0, row * d.pitch);   // chunk `row` of one sequence
    else g.load(d.state, d.n_rows, row);
  } else {
    g.load(d.state, d.n_rows, row);
  }

  uint32_t* out = static_cast<uint32_t*>(d.out);
  const bool vec_ok = ((d.pitch & 3) == 0) && ((reinterpret_cast<uintptr_t>(out) & 15) == 0);
  // Copy-out role of this thread: chunk `cch` of rows cr0 + RS k, k < CH.
  const int cch = tid % CH, cr0 = tid / CH;
  const int cslot = swz<K>(cr0, cch);           // (cr0 + RS k) & 7 == cr0 & 7
  uint32_t* cg = out + (row0 + cr0) * d.pitch + col0 + 4 * cch;
  const uint64_t cstep = (uint64_t)RS * d.pitch;
  const uint64_t left = d.n_rows > row0 + cr0 ? d.n_rows - (row0 + cr0) : 0;
  const int crows = left >= (uint64_t)RS * (CH - 1) + 1 ? CH : (int)((left + RS - 1) / RS);
  const uint64_t last_row = (row0 + T < d.n_rows ? row0 + T : d.n_rows) - 1;
  const int sw = tid & 7;

  int buf = 0;
  for (uint64_t c0 = 0; c0 < n; c0 += K) {
    const int w = (n - c0 < (uint64_t)K) ? (int)(n - c0) : K;
    uint32_t* const t = smem + buf * (T * K);
    uint32_t* my = t + tid * K;
    if (w == K) {
#pragma unroll
      for (int c = 0; c < CH; c++) {
        uint4 v;
        v.x = conv<G, OM>(g.next());
        v.y = conv<G, OM>(g.next());
        v.z = conv<G, OM>(g.next());
        v.w = conv<G, OM>(g.next());
        *reinterpret_cast<uint4*>(my + 4 * (c ^ sw)) = v;
      }
    } else {
      for (int c = 0; c < w; c++) my[4 * ((c >> 2) ^ sw) + (c & 3)] = conv<G, OM>(g.next());
    }
    __syncthreads();
    if (w == K && (vec_ok || OM == OUT_ISING) && last_row * d.pitch + col0 + c0 + K <= d.limit) {
      const uint32_t* src = t + cr0 * K + 4 * cslot;
      uint32_t* dst = cg + c0;
      const uint64_t edst = (row0 + cr0) * d.pitch + 4 * cch + col0 + c0;
#pragma unroll
      for (int k = 0; k < CH; k++)
        if (k < crows) {
          if constexpr (OM == OUT_ISING)
            put4<OM, G::WB>(d, nullptr, edst + k * cstep, *reinterpret_cast<const uint4*>(src + k * RS * K));
          else
            st_chunk<OM, G::WB>(dst + k * cstep, *reinterpret_cast<const uint4*>(src + k * RS * K));
        }
    } else {
      odd_tile<G, T, K, OM>(d, t, row0, col0 + c0, w);
    }
    if constexpr (S == 1) __syncthreads();
    else buf ^= 1;
  }
  if (active && store_to != nullptr) g.store(store_to, d.n_rows, row);
}

// (The descriptor stays in the parameter space: a plain parameter whose address
// odd_tile takes would be copied to every thread's stack first.)
template <class G, int T, int K, int S, int OM>
__global__ void __launch_bounds__(T) k_fill_simple(const __grid_constant__ FillDesc d) {
  extern __shared__ __align__(16) uint32_t smem[];
  simple_rows<G, T, K, S, OM>(d, (uint64_t)blockIdx.x * T, smem, 0, d.n_per, d.jump ? nullptr : d.state);
}

// Segment blockIdx.y of every stream: draws [seg L, seg L + L) of the call, from
// the states that `starts` holds for it ([segment][word][stream]); the last
// segment leaves the handle's states.  (Its descriptor is an ordinary parameter,
// copied to the stack once: as a grid constant the compiler kept fewer of the
// copy-out's loads in flight, 65,536 x 2,048 f64 215 -> 231 us.)
template <class G, int T, int K, int S, int OM>
__global__ void __launch_bounds__(T) k_fill_segments(FillDesc d, uint32_t* starts, uint64_t L) {
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* const state = d.state;
  const uint64_t seg = blockIdx.y, col0 = seg * L;
  const uint64_t n = d.n_per - col0 < L ? d.n_per - col0 : L;
  d.state = starts + seg * 4 * d.n_rows;
  simple_rows<G, T, K, S, OM>(d, (uint64_t)blockIdx.x * T, smem, col0, n, seg + 1 == gridDim.y ? state : nullptr);
}

// Batched XOR128 fills: a block pops an item (T streams of one request).
template <int T, int K, int S, bool F32>
__global__ void __launch_bounds__(T) k_batch_xor128(const BatchQueue q) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint32_t slot;
  for (;;) {
    const uint32_t it = pop_cta(q.counter, &slot);
    if (it >= q.n_items) break;
    const BatchItem si = q.items[it];
    __shared__ FillDesc sd;
    load_desc(&sd, q.reqs[si.req].d, threadIdx.x, T);
    __syncthreads();
    simple_rows<Xor128Gen, T, K, S, F32 ? OUT_F32 : OUT_U32>(sd, si.row0, smem, 0, sd.n_per, sd.state);
  }
}

template <int T, int K, int S, bool F32>
static cudaError_t launch_bx(const BatchQueue& q, cudaStream_t s) {
  constexpr size_t bytes = (size_t)S * T * K * sizeof(uint32_t);
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_batch_xor128<T, K, S, F32>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_xor128<T, K, S, F32>, T, bytes);
  const uint32_t cap = (uint32_t)sm_count() * (per_sm > 0 ? per_sm : 1);
  k_batch_xor128<T, K, S, F32><<<q.n_items < cap ? q.n_items : cap, T, bytes, s>>>(q);
  return cudaGetLastError();
}

template <int T, int K, int S>
static cudaError_t launch_bx2(const BatchQueue& q, bool f32, cudaStream_t s) {
  return f32 ? launch_bx<T, K, S, true>(q, s) : launch_bx<T, K, S, false>(q, s);
}

cudaError_t launch_batch_xor128(const BatchQueue& q, Tile t, bool f32, cudaStream_t s) {
  if (q.n_items == 0) return cudaSuccess;
  if (t.threads == 64 && t.cols == 32 && t.stages == 1) return launch_bx2<64, 32, 1>(q, f32, s);
  if (t.threads == 128 && t.cols == 32 && t.stages == 2) return launch_bx2<128, 32, 2>(q, f32, s);
  if (t.threads == 128 && t.cols == 64 && t.stages == 1) return launch_bx2<128, 64, 1>(q, f32, s);
  if (t.threads == 256 && t.cols == 32 && t.stages == 1) return launch_bx2<256, 32, 1>(q, f32, s);
  return launch_bx2<128, 32, 1>(q, f32, s);
}

// Skip without output for XOR128 (plain stepping).
template <class G>
__global__ void k_skip_step(const FillDesc d) {
  const uint64_t row = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= d.n_rows) return;
  G g;
  g.load(d.state, d.n_rows, row);
  for (uint64_t k = 0; k < d.n_per; k++) g.next();
  g.store(d.state, d.n_rows, row);
}

template <class G, int T, int K, int S, int OM>
static cudaError_t launch_tkf(const FillDesc& d, cudaStream_t s) {
  constexpr size_t bytes = (size_t)S * T * K * sizeof(uint32_t);
  static bool configured = false;  // attribute set once per instantiation
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_fill_simple<G, T, K, S, OM>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  const uint64_t grid = (d.n_rows + T - 1) / T;
  k_fill_simple<G, T, K, S, OM><<<(unsigned)grid, T, bytes, s>>>(d);
  return cudaGetLastError();
}

template <class G, int T, int K, int S>
static cudaError_t launch_tk(const FillDesc& d, cudaStream_t s) {
  return with_mode(d.mode, [&](auto m) { return launch_tkf<G, T, K, S, decltype(m)::value>(d, s); });
}

// Supported tiles: (threads, cols, stages).
template <class G>
static cudaError_t launch_g(const FillDesc& d, Tile t, cudaStream_t s) {
  if (t.threads == 128 && t.cols == 32 && t.stages == 2) return launch_tk<G, 128, 32, 2>(d, s);
  if (t.threads == 128 && t.cols == 64 && t.stages == 1) return launch_tk<G, 128, 64, 1>(d, s);
  if (t.threads == 256 && t.cols == 32 && t.stages == 1) return launch_tk<G, 256, 32, 1>(d, s);
  return launch_tk<G, 128, 32, 1>(d, s);
}

// Whether a plain XOR128 fill of these many streams and draws is faster cut into
// segments of 64-column tiles, by the time a draw of every stream takes (ps).
// Whole, a scheduler's warps decide: one per 19,456 streams, and the fullest
// schedulers set the pace while others idle.  Cut to 131,072 threads and more the
// schedulers are even and the stores run at their rate.  The starts and the
// second launch cost about 16 us.  us, whole / cut, u32 and f64 (as many draws):
// 32,768 x 4,096 97 / 108 and 184 / 124; 40,000 x 8,192 260 / 225 and 398 / 272;
// 50,000 x 2,048 79 / 89 and 110 / 115; 65,536 x 4,096 203 / 188 and 250 / 223;
// 65,536 x 16,384 759 / 662 and 956 / 818; 80,000 x 8,192 494 / 401 and 586 / 509;
// 40,000 x 8,190 (unaligned) 612 / 424 and 928 / 557.
static bool xor128_cut_pays(const FillDesc& d) {
  const uint64_t w = (d.n_rows + 19455) / 19456;
  uint64_t whole, cut;
  if (d.mode == OUT_F64) {
    whole = std::max<uint64_t>(41600, 14400 * w);
    cut = 760 * d.n_rows / 1000;
  } else if (d.mode == OUT_F32) {
    whole = 3600 + 11000 * w;
    cut = 630 * d.n_rows / 1000;
  } else {
    whole = 11400 * w;
    cut = 620 * d.n_rows / 1000;
  }
  return whole > cut && d.n_per >= 16000000 / (whole - cut);
}

// A plain XOR128 fill of few streams as segments of L = 2^k draws, each a thread
// of its own, whose starts T^(seg L) s come from xor128_starts first.  A thread
// makes a draw in about 17 ns whatever the number of streams while those leave
// the GPU idle, so a stream is cut until there are some 65,536 threads, into at
// most 64 segments of at least 64 draws.  The starts cost a second kernel (about
// the time of 800 draws) and, at 65,536 threads, that of some 460 more.  us, whole
// / cut: 256 x 4,096 u32 74 / 28, f64 (as many draws) 165 / 29; 256 x 8,192 135 /
// 28; 4,096 x 4,096 73 / 38; 1,000 x 4,095 (unaligned) 427 / 41; 16,384 x 4,096
// 73 / 71, f64 168 / 84; 4,096 x 1,024 26 / 33, which stays whole.
// From 120 M draws on the stores bound it, and it takes 64-column tiles, whose
// 256-byte row runs they like better, and up to 200,704 threads, as streams too
// many for the first form do where xor128_cut_pays.  us, 65,536 threads of 32
// columns / this: 4,096 x 65,536 u32 221 / 197, f64 271 / 238; 16,384 x 16,384
// 214 / 191, 265 / 230; 30,000 x 4,096 113 / 102; 25,000 x 4,096 90 / 92 and
// 12,000 x 8,192 89 / 104, below the line.
static cudaError_t launch_xor128_segments(const FillDesc& d, bool& done, cudaStream_t s) {
  done = false;
  if (d.n_rows >= 100352 || d.n_per < 900) return cudaSuccess;
  const bool few = d.n_rows < 32768;
  const bool wide = d.mode != OUT_ISING &&
                    (few ? d.n_rows >= 2048 && d.n_per >= 120000000 / d.n_rows : xor128_cut_pays(d));
  if (!few && !wide) return cudaSuccess;
  const uint64_t want = std::min<uint64_t>(64, (wide ? 200704 : 65536) / d.n_rows);
  int lg = 6;
  while (lg < 57 && ((d.n_per - 1) >> lg) + 1 > want) lg++;
  const uint64_t L = 1ull << lg, segs = ((d.n_per - 1) >> lg) + 1;
  if (lg > 56 || L >= d.n_per) return cudaSuccess;
  if (!wide && d.n_per - L < 800 + 460 * d.n_rows * segs / 65536) return cudaSuccess;
  if (capturing(s)) return cudaSuccess;
  uint32_t* starts = nullptr;
  cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&starts), segs * 4 * d.n_rows * sizeof(uint32_t), s);
  if (e != cudaSuccess) {   // no room: whole streams
    cudaGetLastError();
    return cudaSuccess;
  }
  done = true;
  e = launch_xor128_starts(d.state, starts, d.n_rows, (uint32_t)segs, lg, s);
  if (e == cudaSuccess)
    e = with_mode(d.mode, [&](auto m) {
      constexpr int OM = decltype(m)::value, T = 64, K = 32;
      if constexpr (OM != OUT_ISING)
        if (wide) {
          const dim3 grid((unsigned)((d.n_rows + 2 * T - 1) / (2 * T)), (unsigned)segs);
          k_fill_segments<Xor128Gen, 2 * T, 2 * K, 1, OM><<<grid, 2 * T, 4 * T * K * sizeof(uint32_t), s>>>(d, starts, L);
          return cudaGetLastError();
        }
      const dim3 grid((unsigned)((d.n_rows + T - 1) / T), (unsigned)segs);
      k_fill_segments<Xor128Gen, T, K, 1, OM><<<grid, T, T * K * sizeof(uint32_t), s>>>(d, starts, L);
      return cudaGetLastError();
    });
  const cudaError_t ef = scratch_free(starts, s);
  return e != cudaSuccess ? e : ef;
}

cudaError_t launch_fill_simple(int gen, const FillDesc& d, Tile t, cudaStream_t s) {
  if (d.n_rows == 0 || d.n_per == 0) return cudaSuccess;
  if (d.out == nullptr) {  // skip: plain stepping (the MLCG generators jump instead)
    if (gen != XOR128) return cudaErrorInvalidValue;
    k_skip_step<Xor128Gen><<<(unsigned)((d.n_rows + 127) / 128), 128, 0, s>>>(d);
    return cudaGetLastError();
  }
  switch (gen) {
    case GGL: return launch_g<GglGen>(d, t, s);
    case XOR128: {
      if (!tile_chosen(XOR128, 0) && !d.jump) {
        bool done = false;
        const cudaError_t e = launch_xor128_segments(d, done, s);
        if (done || e != cudaSuccess) return e;
      }
      return launch_g<Xor128Gen>(d, t, s);
    }
    case RANECU: return launch_g<RanecuGen>(d, t, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace prng
