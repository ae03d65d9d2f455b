// k_ranlux_tc.cu -- RANLUX fills on the tensor cores (Section 3.6; Appendix A,
// "AWC and SWB" and "RANLUX").
//
// A subtract-with-borrow generator is a linear congruential one in disguise
// (Tezuka, L'Ecuyer, Couture 1993; Luescher 1994).  With b = 2^24, m = b^24 -
// b^10 + 1 and the state's 24 words (oldest first) packed as the 576-bit
// integer R, X = R - (R >> 336) + carry satisfies b X_{n+1} = X_n + x_n m, so
// X_{n+1} = b^{-1} X_n mod m.  A whole luxury cycle, p steps of which p - 24
// are thrown away, is then one multiplication by the constant a = b^{-p} mod m,
// whatever p is (so skips RANLUX++ too, Sibidanov 2017).  And since b^24 X_{n+24} = X_n + m R_{n+24}, the 24 words that
// follow X_n are R_{n+24} = -X_n m^{-1} mod 2^576 with m^{-1} = 1 + 2^240 +
// 2^480 (mod 2^576): two shifted additions.
//
// The product is a contraction: with X in 72 bytes, a X = sum_k byte_k (256^k a
// mod m), 72 residues of 72 bytes that all streams share.  A CTA's 128 streams
// are the 128 rows of a 128 x 80 x 80 matrix product per cycle on the tensor
// cores: bytes as f16, sums in f32.  It is exact: a byte sits in the low bits of
// an f16 pattern, a subnormal that means byte x 2^-24; the residues' bytes are
// f16 integers; all sums are whole multiples of 2^-24 below 2^24 of them.  A
// constant row adds 2^23 x 2^-24 to every sum, so a sum's f32 pattern is
// 0x3F000000 + the sum and no conversion is needed.
//
// What is kept per stream is N = m - X + D with D = 2^240 - 1 (so N = D - X mod
// m, in [D, 2^576)): then N = -X mod 2^576 and the delivered words are N (1 +
// 2^240 + 2^480).  Thread t of the CTA owns row t: its A operand and its sums
// are its own TMEM lane, and carries, reduction and output are 32-bit integer
// work in its registers.  While the tensor core multiplies for the next cycle,
// the threads turn the current N into words and write them out, through the
// same per-row ring and warp-level 128-byte copy-outs as k_fill_ranlux_ring.
#include <algorithm>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "ranlux_tc.cuh"
#include "scratch.cuh"
#include "tc.cuh"

namespace prng {

namespace {

constexpr int kLevels = 6;   // p >= kLuxTcMinP
constexpr int kLevelP[kLevels] = {97, 223, 389, 120, 240, 408};
// Operands per level: 2^i luxury cycles, i < kLuxPowers (0: the fill's own; the
// others move a segment's start along its stream).
constexpr int kNK = 80;                       // K and N of the product: 72 bytes, constants, padding
constexpr int kTabBytes = kNK * kNK * 2;      // the f16 operand, in core-matrix order
constexpr uint32_t kKStep = (kNK / 8) * 128;  // bytes between core matrices along K
constexpr uint32_t kRStep = 128;              // and along the residue bytes
constexpr uint32_t kMagic = 0x3F000000u;      // pattern of 2^23 x 2^-24

constexpr int kTmemCols = 128, kColD = 0, kColA = 80;

// Filled on a device's first RANLUX handle (2.4 MB).
__device__ uint4 g_tab[kLevels][kLuxPowers][kTabBytes / 16];
// The device's word that a kernel sets when it gave up waiting for the tensor core
// (never seen): in mapped host memory, so that a later call sees it without a copy.
__device__ uint32_t* g_failed;
constexpr int kMaxDevices = 64;
uint32_t* g_failed_host[kMaxDevices] = {};

__device__ __forceinline__ void lux_give_up() {
  *static_cast<volatile uint32_t*>(g_failed) = 1u;
  __threadfence_system();
}

// ---------------------------------------------------------- host: the operands

struct Big {   // 576 bits, little endian
  uint32_t w[18];
};

Big mod_m(std::vector<uint32_t> v) {
  // v mod m: 2^576 = 2^240 - 1 (mod m), folded until nothing is left above.
  for (;;) {
    bool high = false;
    for (size_t i = 18; i < v.size(); i++) high |= v[i] != 0;
    if (!high) break;
    std::vector<uint32_t> r(v.begin(), v.begin() + 18);
    r.resize(v.size() + 2, 0);
    std::vector<uint32_t> h(v.begin() + 18, v.end());
    uint64_t c = 0;                              // + h << 240 (7 words and 16 bits)
    for (size_t i = 0; i + 7 < r.size(); i++) {
      const uint32_t lo = i < h.size() ? h[i] << 16 : 0, hi = i > 0 && i - 1 < h.size() ? h[i - 1] >> 16 : 0;
      c += (uint64_t)r[i + 7] + (lo | hi);
      r[i + 7] = (uint32_t)c;
      c >>= 32;
    }
    int64_t bw = 0;                              // - h
    for (size_t i = 0; i < r.size(); i++) {
      bw += (int64_t)r[i] - (i < h.size() ? (int64_t)h[i] : 0);
      r[i] = (uint32_t)bw;
      bw >>= 32;
    }
    v = r;
  }
  v.resize(18, 0);
  Big x;
  std::copy(v.begin(), v.begin() + 18, x.w);
  // once more if x >= m, i.e. x + D >= 2^576
  uint64_t c = 0;
  uint32_t t[18];
  for (int i = 0; i < 18; i++) {
    c += (uint64_t)x.w[i] + (i < 7 ? 0xFFFFFFFFu : i == 7 ? 0xFFFFu : 0u);
    t[i] = (uint32_t)c;
    c >>= 32;
  }
  if (c) std::copy(t, t + 18, x.w);
  return x;
}

Big mul_m(const Big& a, const Big& b) {
  std::vector<uint32_t> p(37, 0);
  for (int i = 0; i < 18; i++) {
    uint64_t c = 0;
    for (int j = 0; j < 18; j++) {
      c += (uint64_t)a.w[i] * b.w[j] + p[i + j];
      p[i + j] = (uint32_t)c;
      c >>= 32;
    }
    p[i + 18] = (uint32_t)c;
  }
  return mod_m(p);
}

Big neg_m(const Big& a) {   // -a mod m, for a != 0: m - a = 2^576 - D - a
  int64_t bw = 0;
  Big r;
  for (int i = 0; i < 18; i++) {
    bw -= (int64_t)a.w[i] + (i < 7 ? 0xFFFFFFFFll : i == 7 ? 0xFFFFll : 0ll);
    r.w[i] = (uint32_t)bw;
    bw >>= 32;
  }
  return r;
}

Big shl8_m(const Big& a) {   // 256 a mod m: the top byte t comes back as t 2^240 - t
  const int64_t t = a.w[17] >> 24;
  Big r;
  int64_t c = -t;
  for (int i = 0; i < 18; i++) {
    c += (int64_t)(uint32_t)(a.w[i] << 8 | (i > 0 ? a.w[i - 1] >> 24 : 0)) + (i == 7 ? t << 16 : 0);
    r.w[i] = (uint32_t)c;
    c >>= 32;
  }
  if (c == 0) return r;
  std::vector<uint32_t> v(r.w, r.w + 18);
  v.push_back((uint32_t)c);
  return mod_m(v);
}

uint16_t f16_int(uint32_t v) {   // f16 pattern of an integer below 2^11 (or a power of two below 2^16)
  if (v == 0) return 0;
  int e = 31 - __builtin_clz(v);
  return (uint16_t)(((e + 15) << 10) | (e <= 10 ? (v << (10 - e)) & 0x3FF : (v >> (e - 10)) & 0x3FF));
}

// The operand of multiplication by a: column k < 72 holds the bytes of 256^k a
// mod m; column 72 (A's constant 2^-14) 2^13 everywhere, for the 2^23 x 2^-24;
// column 73 (A's constant 2^-24) the bytes of the correction that takes out the
// magic patterns of the combined sums and the offset D of the kept N: the words
// of the sum P + (Q << 16), each 0x3F000000 too large, and a D.
void build_tab(const Big& a, uint16_t* tab) {
  std::fill(tab, tab + kTabBytes / 2, (uint16_t)0);
  auto at = [&](int n, int k) -> uint16_t& {
    return tab[((k / 8) * kKStep + (n / 8) * kRStep + (n % 8) * 16 + (k % 8) * 2) / 2];
  };
  Big r = a;
  for (int k = 0; k < 72; k++) {
    for (int n = 0; n < 72; n++) at(n, k) = f16_int((r.w[n / 4] >> (8 * (n % 4))) & 0xFFu);
    r = shl8_m(r);
  }
  Big D{};
  for (int i = 0; i < 8; i++) D.w[i] = i < 7 ? 0xFFFFFFFFu : 0xFFFFu;
  const Big aD = mul_m(a, D);
  std::vector<uint32_t> e(20, 0);   // E + a D, E = sum over words of magic (1 + 2^16)
  uint64_t c = 0;
  for (int i = 0; i < 20; i++) {
    c += i < 18 ? (uint64_t)aD.w[i] : 0;
    if (i < 18) c += (uint32_t)(kMagic + (kMagic << 16));
    if (i > 0 && i < 19) c += kMagic >> 16;
    e[i] = (uint32_t)c;
    c >>= 32;
  }
  const Big bias = neg_m(mod_m(e));
  for (int n = 0; n < 72; n++) {
    at(n, 72) = f16_int(8192);
    at(n, 73) = f16_int((bias.w[n / 4] >> (8 * (n % 4))) & 0xFFu);
  }
}

}  // namespace

// The operands of every level and power (bounded: one array, built once per
// process; the caller holds the lock of lux_tables_init).
const std::vector<uint16_t>& lux_host_tables() {
  static std::vector<uint16_t> host;
  if (host.empty()) {
    // (m - 1) / b = b^23 - b^9, so b (b^23 - b^9) = -1 and b^{-1} = m - b^23 + b^9 (mod m).
    Big one{};
    one.w[0] = 1;
    std::vector<uint32_t> v(19, 0);
    int64_t c = 0;
    // b^23 = 2^552, b^9 = 2^216, b^10 = 2^240, b^24 = 2^576
    for (int i = 0; i < 19; i++) {
      c += (i == 18 ? 1 : 0) - (i == 7 ? 65536 : 0) + (i == 0 ? 1 : 0) - (i == 17 ? (1 << 8) : 0) +
           (i == 6 ? (1 << 24) : 0);
      v[i] = (uint32_t)c;
      c >>= 32;
    }
    const Big binv = mod_m(v);
    std::vector<uint16_t> t((size_t)kLevels * kLuxPowers * kTabBytes / 2);
    for (int l = 0; l < kLevels; l++) {
      Big a = one, s = binv;
      for (int k = kLevelP[l]; k; k >>= 1) {
        if (k & 1) a = mul_m(a, s);
        s = mul_m(s, s);
      }
      for (int i = 0; i < kLuxPowers; i++) {
        build_tab(a, t.data() + (size_t)(l * kLuxPowers + i) * kTabBytes / 2);
        a = mul_m(a, a);
      }
    }
    host.swap(t);
  }
  return host;
}

// Fill the current device's operands once.
cudaError_t lux_tables_init() {
  static std::mutex lock;
  static bool done[kMaxDevices] = {};
  std::lock_guard<std::mutex> guard(lock);
  const std::vector<uint16_t>* host;
  try {
    host = &lux_host_tables();
  } catch (const std::bad_alloc&) {   // no exception leaves a C entry point
    return cudaErrorMemoryAllocation;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (done[dev]) return cudaSuccess;
  uint32_t *word = g_failed_host[dev], *at = nullptr;
  if (word == nullptr) {
    e = cudaHostAlloc(reinterpret_cast<void**>(&word), sizeof(*word), cudaHostAllocMapped | cudaHostAllocPortable);
    if (e != cudaSuccess) return e;
    *word = 0;
    g_failed_host[dev] = word;
  }
  e = cudaHostGetDevicePointer(reinterpret_cast<void**>(&at), word, 0);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_failed, &at, sizeof(at));
  if (e != cudaSuccess) return e;
  e = cudaMemcpyToSymbol(g_tab, host->data(), host->size() * 2);
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

uint32_t* lux_failed_word(int dev) { return dev >= 0 && dev < kMaxDevices ? g_failed_host[dev] : nullptr; }

bool lux_tc_failed(int dev) {
  const volatile uint32_t* w = lux_failed_word(dev);
  return w != nullptr && *w != 0;
}

// --------------------------------------------------------------------- device

namespace {

// x += y (+ y3 << 480 when that is given), 576 bits, as carry chains.
__device__ __forceinline__ uint32_t add18(uint32_t (&x)[18], const uint32_t (&y)[18]) {
  uint32_t c;
  asm("add.cc.u32 %0, %0, %19;\n\t"
      "addc.cc.u32 %1, %1, %20;\n\t"
      "addc.cc.u32 %2, %2, %21;\n\t"
      "addc.cc.u32 %3, %3, %22;\n\t"
      "addc.cc.u32 %4, %4, %23;\n\t"
      "addc.cc.u32 %5, %5, %24;\n\t"
      "addc.cc.u32 %6, %6, %25;\n\t"
      "addc.cc.u32 %7, %7, %26;\n\t"
      "addc.cc.u32 %8, %8, %27;\n\t"
      "addc.cc.u32 %9, %9, %28;\n\t"
      "addc.cc.u32 %10, %10, %29;\n\t"
      "addc.cc.u32 %11, %11, %30;\n\t"
      "addc.cc.u32 %12, %12, %31;\n\t"
      "addc.cc.u32 %13, %13, %32;\n\t"
      "addc.cc.u32 %14, %14, %33;\n\t"
      "addc.cc.u32 %15, %15, %34;\n\t"
      "addc.cc.u32 %16, %16, %35;\n\t"
      "addc.cc.u32 %17, %17, %36;\n\t"
      "addc.u32 %18, 0, 0;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]), "+r"(x[6]), "+r"(x[7]),
        "+r"(x[8]), "+r"(x[9]), "+r"(x[10]), "+r"(x[11]), "+r"(x[12]), "+r"(x[13]), "+r"(x[14]),
        "+r"(x[15]), "+r"(x[16]), "+r"(x[17]), "=r"(c)
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(y[8]),
        "r"(y[9]), "r"(y[10]), "r"(y[11]), "r"(y[12]), "r"(y[13]), "r"(y[14]), "r"(y[15]), "r"(y[16]),
        "r"(y[17]));
  return c;
}

// Word i of D = 2^240 - 1.
__device__ __forceinline__ constexpr uint32_t d_word(int i) {
  return i < 7 ? 0xFFFFFFFFu : i == 7 ? 0xFFFFu : 0u;
}

// The delivered words N (1 + 2^240 + 2^480) mod 2^576 (240 bits = 7 words and
// 16 bits, 480 = 15 words).
__device__ __forceinline__ void lux_words(const uint32_t (&N)[18], uint32_t (&R)[18]) {
#pragma unroll
  for (int i = 0; i < 18; i++) R[i] = N[i];
  uint32_t S[11];
  S[0] = N[0] << 16;
#pragma unroll
  for (int i = 1; i < 11; i++) S[i] = __funnelshift_l(N[i - 1], N[i], 16);
  asm("add.cc.u32 %0, %0, %11;\n\t"
      "addc.cc.u32 %1, %1, %12;\n\t"
      "addc.cc.u32 %2, %2, %13;\n\t"
      "addc.cc.u32 %3, %3, %14;\n\t"
      "addc.cc.u32 %4, %4, %15;\n\t"
      "addc.cc.u32 %5, %5, %16;\n\t"
      "addc.cc.u32 %6, %6, %17;\n\t"
      "addc.cc.u32 %7, %7, %18;\n\t"
      "addc.cc.u32 %8, %8, %19;\n\t"
      "addc.cc.u32 %9, %9, %20;\n\t"
      "addc.u32 %10, %10, %21;\n\t"
      "add.cc.u32 %8, %8, %22;\n\t"
      "addc.cc.u32 %9, %9, %23;\n\t"
      "addc.u32 %10, %10, %24;"
      : "+r"(R[7]), "+r"(R[8]), "+r"(R[9]), "+r"(R[10]), "+r"(R[11]), "+r"(R[12]), "+r"(R[13]), "+r"(R[14]),
        "+r"(R[15]), "+r"(R[16]), "+r"(R[17])
      : "r"(S[0]), "r"(S[1]), "r"(S[2]), "r"(S[3]), "r"(S[4]), "r"(S[5]), "r"(S[6]), "r"(S[7]), "r"(S[8]),
        "r"(S[9]), "r"(S[10]), "r"(N[0]), "r"(N[1]), "r"(N[2]));
}

// The new N from the 72 sums v (f32 patterns, see the file's head).  Four sums
// make a 32-bit word of P (bytes 0 and 1 of the word) and one of Q (bytes 2 and
// 3, 16 bits up); the value above 2^576, top, folds back as top 2^240 - top,
// which are one word of Q and one of P, and one more fold puts N at X' + D
// (X' = a (m - X) mod m's representative).  top is taken from the highest word
// without the carries from below, which is wrong once in about 2^32 times; then,
// or when the sum itself passes 2^576, N's highest word is 0 and N lacks D.
__device__ __forceinline__ void lux_reduce(const uint32_t (&v)[72], uint32_t (&N)[18]) {
  uint32_t Q[18];
#pragma unroll
  for (int i = 0; i < 18; i++) {
    N[i] = v[4 * i + 1] * 256u + v[4 * i];
    Q[i] = v[4 * i + 3] * 256u + v[4 * i + 2];
  }
  const uint32_t t17 = N[17] + __funnelshift_l(Q[16], Q[17], 16);
  const uint32_t carry = t17 < N[17] ? 1u : 0u;
  const uint32_t q = (Q[17] >> 16) + carry + 1u;
  N[0] -= q;          // P's words are at least the magic pattern: no borrow
  Q[7] += q;          // 2^240 is bit 16 of word 7; Q's words are below 2^32 - 2^17
  uint32_t S[18];
  S[0] = Q[0] << 16;
#pragma unroll
  for (int i = 1; i < 18; i++) S[i] = __funnelshift_l(Q[i - 1], Q[i], 16);
  const uint32_t over = add18(N, S) - carry;
  if (N[17] == 0 && over != 0) {
    uint32_t Dw[18];
#pragma unroll
    for (int i = 0; i < 18; i++) Dw[i] = d_word(i);
    add18(N, Dw);
  }
}

// N 24 steps back: X -> b^24 X = D X (mod m), that is N -> D N + D - D^2, as the
// representative in [D, 2^576).  (N lo << 240) + ~(N hi) are disjoint bits; the
// constants of the two complements and D - D^2 are one constant C24.
__device__ __forceinline__ void lux_back24(uint32_t (&N)[18]) {
  // C24 = D - D^2 + (1 - D) + (1 - 2^240) mod m, D^2 = 2^480 - 2^241 + 1:
  //     = 2^240 - 2^480 + 1  ->  m - 2^480 + 2^240 + 1 = 2^576 - 2^480 + 2
  uint32_t a[18], t[18];
  uint32_t top = 0;
#pragma unroll
  for (int i = 0; i < 18; i++) {   // (lo << 240) | (~hi, 240 bits); hi = N >> 336 (10 words and 16 bits)
    const uint32_t hi = i < 8 ? (i < 7 ? __funnelshift_r(N[i + 10], N[i + 11], 16) : N[17] >> 16) : 0u;
    const uint32_t lo = i >= 7 ? (i == 7 ? N[0] << 16 : __funnelshift_l(N[i - 8], N[i - 7], 16)) : 0u;
    a[i] = i < 7 ? ~hi : i == 7 ? (lo | (~hi & 0xFFFFu)) : lo;
  }
#pragma unroll
  for (int i = 0; i < 18; i++) t[i] = ~N[i];
  top += add18(a, t);
#pragma unroll
  for (int i = 0; i < 18; i++) {   // hi << 240: words 7 .. 14
    const uint32_t h0 = i >= 7 && i < 15 ? (i - 7 < 7 ? __funnelshift_r(N[i + 3], N[i + 4], 16) : N[17] >> 16) : 0u;
    const uint32_t h1 = i >= 8 && i < 16 ? (i - 8 < 7 ? __funnelshift_r(N[i + 2], N[i + 3], 16) : N[17] >> 16) : 0u;
    t[i] = h0 << 16 | h1 >> 16;
  }
  top += add18(a, t);
#pragma unroll
  for (int i = 0; i < 18; i++) t[i] = i == 0 ? 2u : i < 15 ? 0u : 0xFFFFFFFFu;
  top += add18(a, t);
  while (top != 0) {   // top 2^576 = top (2^240 - 1) = (top - 1) 2^240 + (2^240 - top), 0 < top < 2^16
#pragma unroll
    for (int i = 0; i < 18; i++)
      t[i] = i == 0 ? 0u - top : i < 7 ? 0xFFFFFFFFu : i == 7 ? (top - 1u) << 16 | 0xFFFFu : 0u;
    top = add18(a, t);
  }
  // below D: add m = 2^576 - D
  bool small = true;
#pragma unroll
  for (int i = 8; i < 18; i++) small = small && a[i] == 0;
  bool all = a[7] == 0xFFFFu;
#pragma unroll
  for (int i = 0; i < 7; i++) all = all && a[i] == 0xFFFFFFFFu;
  if (small && a[7] <= 0xFFFFu && !all) {
#pragma unroll
    for (int i = 0; i < 18; i++) t[i] = i == 0 ? 1u : i < 7 ? 0u : i == 7 ? 0xFFFF0000u : 0xFFFFFFFFu;
    add18(a, t);
  }
#pragma unroll
  for (int i = 0; i < 18; i++) N[i] = a[i];
}

// N of a block-end state: ring words V (oldest first) and carry, then 24 steps
// back.  zero: the all-zero state, whose X = 0 has the same N as X = m.
__device__ __forceinline__ void lux_load(const uint32_t (&V)[24], uint32_t c, uint32_t (&N)[18], bool& zero) {
  uint32_t R[18], t[18];
  uint32_t any = c;
#pragma unroll
  for (int g = 0; g < 6; g++) {
    const uint32_t w0 = V[4 * g], w1 = V[4 * g + 1], w2 = V[4 * g + 2], w3 = V[4 * g + 3];
    any |= w0 | w1 | w2 | w3;
    R[3 * g] = w0 | w1 << 24;
    R[3 * g + 1] = w1 >> 8 | w2 << 16;
    R[3 * g + 2] = w2 >> 16 | w3 << 8;
  }
  // -X = (R >> 336) - R - c = (R >> 336) + ~R + (1 - c)
#pragma unroll
  for (int i = 0; i < 18; i++) t[i] = i < 8 ? (i < 7 ? __funnelshift_r(R[i + 10], R[i + 11], 16) : R[17] >> 16) : 0u;
#pragma unroll
  for (int i = 0; i < 18; i++) N[i] = ~R[i];
  add18(N, t);
#pragma unroll
  for (int i = 0; i < 18; i++) t[i] = i == 0 ? 1u - c : 0u;
  add18(N, t);
  zero = any == 0;
  if (zero) {
#pragma unroll
    for (int i = 0; i < 18; i++) N[i] = d_word(i);
  }
  lux_back24(N);
}

// Carry of the state whose words N delivered: X_n + R >= 2^576, i.e. R >= N.
__device__ __forceinline__ uint32_t lux_carry(const uint32_t (&N)[18], const uint32_t (&R)[18]) {
  uint32_t ge = 1;   // compare from the lowest word up
#pragma unroll
  for (int i = 0; i < 18; i++) ge = R[i] > N[i] ? 1u : R[i] < N[i] ? 0u : ge;
  return ge;
}

// 24-bit word j of R.
template <int J>
__device__ __forceinline__ uint32_t lux_word(const uint32_t (&R)[18]) {
  constexpr int g = (J / 4) * 3;
  if constexpr (J % 4 == 0) return R[g] & 0xFFFFFFu;
  else if constexpr (J % 4 == 1) return __funnelshift_r(R[g], R[g + 1], 24) & 0xFFFFFFu;
  else if constexpr (J % 4 == 2) return __funnelshift_r(R[g + 1], R[g + 2], 16) & 0xFFFFFFu;
  else return R[g + 2] >> 8;
}

template <int... J>
__device__ __forceinline__ void lux_words24(const uint32_t (&R)[18], uint32_t (&V)[24],
                                            std::integer_sequence<int, J...>) {
  ((V[J] = lux_word<J>(R)), ...);
}

template <int OM>
__device__ __forceinline__ uint32_t tc_conv(uint32_t x) {
  if constexpr (OM == OUT_F32) return __float_as_uint(__uint2float_rn(x) * 0x1p-24f);
  else return x;
}

// Output word j of R.  A float is made of the word times 2^8, whose shift left
// by 8 both drops the next word's bits and is a multiply by a constant-bank 2^8
// on the FMA pipe, where the mask would be one more integer instruction
// (65,536 x 4096 f32: 242 -> 231 us; the same for u32, which then has to shift
// back, is slower: 224 -> 228 us).
__constant__ uint32_t c_shl8 = 256u;
template <int OM, int J>
__device__ __forceinline__ uint32_t lux_out_word(const uint32_t (&R)[18]) {
  if constexpr (OM == OUT_F32) {
    constexpr int g = (J / 4) * 3;
    uint32_t X;
    if constexpr (J % 4 == 0) X = R[g] * c_shl8;
    else if constexpr (J % 4 == 1) X = __byte_perm(R[g], R[g + 1], 0x6543) * c_shl8;
    else if constexpr (J % 4 == 2) X = __byte_perm(R[g + 1], R[g + 2], 0x5432) * c_shl8;
    else X = R[g + 2] & 0xFFFFFF00u;
    return lux_out<OM>(X);
  } else {
    return lux_word<J>(R);
  }
}

template <int OM, int Q>
__device__ __forceinline__ uint4 lux_quad(const uint32_t (&R)[18]) {
  return make_uint4(lux_out_word<OM, 4 * Q>(R), lux_out_word<OM, 4 * Q + 1>(R), lux_out_word<OM, 4 * Q + 2>(R),
                    lux_out_word<OM, 4 * Q + 3>(R));
}

constexpr int kRC = 14, kRowWords = 4 * kRC + 4;   // ring chunks of a row; row pitch (odd in chunks)
constexpr int kBox = 32;                           // tile stores: 32 rows x 32 words

struct TcTable {
  uint4 tab[kTabBytes / 16];   // the operand; after the last product, scratch (25 words per thread)
  uint64_t bar;
  uint32_t tmem;
};

// The digits of N as this thread's A operand (before the CTA barrier that
// precedes the product).
__device__ __forceinline__ void lux_digits(uint32_t tm, const uint32_t (&N)[18]) {
  uint32_t A[36];
#pragma unroll
  for (int i = 0; i < 18; i++) {
    A[2 * i] = __byte_perm(N[i], 0, 0x4140);
    A[2 * i + 1] = __byte_perm(N[i], 0, 0x4342);
  }
  tc::st36(tm + ((threadIdx.x >> 5) << 21) + kColA, A);   // this warp's TMEM lanes
  tc::fence_before_sync();
}

// Warp 0, after that barrier: the product of the CTA's 128 rows.
__device__ __forceinline__ void lux_product(TcTable& sh, uint32_t tm) {
  if (tc::elect_one()) {
    tc::fence_after_sync();
    const uint32_t b = tc::smem_addr(sh.tab);
#pragma unroll
    for (int s = 0; s < kNK / 16; s++)
      tc::mma_f16_ts(tm + kColD, tm + kColA + 8 * s, tc::smem_desc(b + 2 * s * kKStep, kKStep, kRStep),
                     tc::idesc_f16_f32(128, kNK), s > 0);
    tc::mma_commit(&sh.bar);
  }
  __syncwarp();
}

// Both, when no thread is `bad`; false when the CTA gives up.
__device__ __forceinline__ bool lux_issue(TcTable& sh, uint32_t tm, const uint32_t (&N)[18], bool bad) {
  lux_digits(tm, N);
  if (__syncthreads_or(bad)) return false;
  if (threadIdx.x < 32) lux_product(sh, tm);
  return true;
}

// Wait for the product and take the new N.
__device__ __forceinline__ bool lux_take(TcTable& sh, uint32_t tm, uint32_t parity, uint32_t (&N)[18]) {
  const bool ok = tc::mbar_wait(&sh.bar, parity);
  __syncwarp();
  tc::fence_after_sync();
  uint32_t v[72];
  tc::ld72(tm + ((threadIdx.x >> 5) << 21) + kColD, v);
  lux_reduce(v, N);
  return ok;
}

// A's constant columns: 2^-14 and 2^-24 at K = 72 and 73, zeros behind.
__device__ __forceinline__ void lux_constants(uint32_t tm) {
  tc::st4(tm + ((threadIdx.x >> 5) << 21) + kColA + 36, 0x00010400u, 0u, 0u, 0u);
}

// Staging and output of a warp's 32 rows as 32 x 32-word tiles that the tile
// engine stores: word e of a row goes to tile e / 32, two tiles in turn, at
// 128 bytes per row with the eight 16-byte chunks exchanged by row (the
// engine's 128-byte swizzle), so that eight rows storing the same chunk hit
// eight bank quads.  Needs 16-byte-aligned rows in device memory.
template <int OM>
struct TileOut {
  uint8_t* box;        // the warp's two tiles, 4 KB each, 1 KB-aligned
  uint32_t rowb;       // this lane's row in a tile, swizzle phase folded in
  const void* map;
  uint32_t wrow0;
  bool rows;           // the warp has rows
  uint32_t done;       // tiles stored

  __device__ __forceinline__ uint32_t at(uint32_t chunk) const {   // byte of 16-byte chunk `chunk` of the row
    return rowb ^ ((chunk & 7u) << 4) ^ ((chunk & 8u) << 9);
  }
  __device__ __forceinline__ void put4(uint32_t chunk, uint4 v) const {
    *reinterpret_cast<uint4*>(box + at(chunk)) = v;
  }
  __device__ __forceinline__ uint32_t* word(uint64_t e) const {
    return reinterpret_cast<uint32_t*>(box + at((uint32_t)(e >> 2))) + (e & 3);
  }
  // Before words of a tile are written again: the engine has read it.
  __device__ __forceinline__ void acquire() const {
    if ((threadIdx.x & 31) == 0) tc::tile_store_wait_read();
    __syncwarp();
  }
  // Store the tiles that the first `words` words of the rows complete.
  __device__ __forceinline__ void release(uint32_t tiles) {
    while (done < tiles) {
      tc::fence_smem_to_async();
      __syncwarp();
      if ((threadIdx.x & 31) == 0 && rows)
        tc::tile_store(map, tc::smem_addr(box) + (done & 1u) * 4096u, done * kBox, wrow0);
      done++;
    }
  }
};

// Staged words of a quad in output mode OM (doubles: two of them).
template <int OM, int Q>
__device__ __forceinline__ uint4 lux_chunk(const uint32_t (&R)[18]) {
  const uint4 v = lux_quad<OM, Q>(R);
  if constexpr (OM == OUT_F64) {
    const double a = pair_f64<24>(v.x, v.y), b = pair_f64<24>(v.z, v.w);
    return make_uint4(__double2loint(a), __double2hiint(a), __double2loint(b), __double2hiint(b));
  } else {
    return v;
  }
}

// This thread's stored state; past the last stream any ordinary one.  (Not zeros:
// every double of an all-zero row takes the slow conversion of pairs whose high
// part is 0, and the CTA with such rows sets the pace: 12,000 x 700 doubles at
// p = 389 118 us, 16,000 x 700, whole CTAs, 79.)
__device__ __forceinline__ void lux_state(const FillDesc& d, uint64_t row, bool active, uint32_t (&V)[24],
                                          uint32_t& c) {
#pragma unroll
  for (int j = 0; j < 24; j++) V[j] = active ? d.state[(uint64_t)j * d.n_rows + row] : 0xA5A5A5u + j;
  c = active ? d.state[24 * d.n_rows + row] : 0u;
}
__device__ __forceinline__ void lux_store(const FillDesc& d, uint64_t row, bool active, const uint32_t (&V)[24],
                                          uint32_t c) {
  if (!active) return;
#pragma unroll
  for (int j = 0; j < 24; j++) d.state[(uint64_t)j * d.n_rows + row] = V[j];
  d.state[24 * d.n_rows + row] = c;
}

// Operand `power` of the level into shared memory (visible to the tensor core
// after the next CTA barrier).
__device__ __forceinline__ void lux_operand(TcTable& sh, int level, int power) {
  for (int i = threadIdx.x; i < kTabBytes / 16; i += 128) sh.tab[i] = g_tab[level][power][i];
  tc::fence_smem_to_async();
}

// TMEM and barrier of the CTA (visible after the next CTA barrier).
__device__ __forceinline__ void lux_setup(TcTable& sh) {
  if (threadIdx.x < 32) tc::tmem_alloc(&sh.tmem, kTmemCols);
  if (threadIdx.x == 0) tc::mbar_init(&sh.bar, 1);
}
// All threads: release the TMEM after every product has been taken.
__device__ __forceinline__ void lux_teardown(uint32_t tm) {
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc::fence_after_sync();
    tc::tmem_free(tm, kTmemCols);
  }
}

// h steps on the state, through 24 words of shared scratch.
template <class Emit>
__device__ __forceinline__ void lux_head(uint32_t (&V)[24], uint32_t& c, int h, uint32_t* scratch, Emit emit) {
  if (h == 0) return;
#pragma unroll
  for (int j = 0; j < 24; j++) scratch[j] = V[j];
  int ph = 0;
  uint32_t prev = 0;
  for (int k = 0; k < h; k++) {
    uint32_t x;
    ph = swb_smem<OUT_U32>(scratch, ph, c, 1, &x, true);
    emit(k, prev, x);
    prev = x;
  }
  for (int j = 0; j < 24; j++) V[j] = scratch[j + ph < 24 ? j + ph : j + ph - 24];
}

struct LuxPlan : LuxPieces {
  __device__ __forceinline__ explicit LuxPlan(const FillDesc& d) : LuxPieces(d.n_per, d.pos) {}
};

// State of row `row` at a block's end, R and its carry, and what of it a tail of
// m draws leaves (scratch: 24 words of shared memory; draw k to emit(k, draw k - 1, draw k)).
template <class Emit>
__device__ __forceinline__ void lux_finish(const FillDesc& d, uint64_t row, bool active,
                                           const uint32_t (&N)[18], const uint32_t (&R)[18], int m,
                                           uint32_t* scratch, Emit emit) {
  uint32_t c = lux_carry(N, R);
  uint32_t V[24];
  lux_words24(R, V, std::make_integer_sequence<int, 24>{});
  lux_head(V, c, m, scratch, emit);
  lux_store(d, row, active, V, c);
}

// Streams [128 blockIdx.x, + 128) of a fill, one per thread, u32, f32 or f64,
// rows 16-byte aligned in device memory and a start that leaves a multiple of 4
// draws in the open block: output by 32 x 32-word tile stores.
//
// What bounds it: neither DRAM (0.73 of the copy peak) nor the tensor core (its
// pipe is busy 31 % of the time) but the integer work around the product, about
// 400 instructions per 24 words of a stream (ALU pipe 61 % busy, issue 61 %), and
// the grain of the work: 65,536 streams are 3.4 CTAs per SM, so some SMs run four
// and the rest three.  2^28 words over 65,536 streams, a u32 and an f32 fill
// together, borrow chain -> here: p = 223 816 -> 451 us, p = 389 1,284 -> 451 (f32
// alone 654 -> 219).  The same product with the rows copied out of a ring
// by the warps (k_fill_ranlux_tc below) took 320 us: 100 more instructions per
// block.  Moving the funnel shifts to the FMA pipe (multiplies by 2^16 and their
// high halves) was slower (224 -> 238 us).
template <int OM>
__global__ void __launch_bounds__(128, 4) k_fill_ranlux_tiles(const FillDesc d, int level,
                                                              const __grid_constant__ CUtensorMap map) {
  __shared__ __align__(1024) uint8_t boxes[4][2 * 4096];
  __shared__ __align__(128) TcTable sh;
  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const uint64_t nr = d.n_rows;
  const uint64_t row = (uint64_t)blockIdx.x * 128 + tid;
  const uint64_t wrow0 = (uint64_t)blockIdx.x * 128 + wi * 32;
  const bool active = row < nr;

  uint32_t V[24], c;
  lux_state(d, row, active, V, c);
  lux_setup(sh);
  lux_operand(sh, level, 0);

  const LuxPlan plan(d);
  TileOut<OM> to{boxes[wi], (uint32_t)(lane * 128 + ((lane & 7) << 4)), &map, (uint32_t)wrow0, wrow0 < nr, 0};
  // Draw k of a head or tail (the one before it given too: doubles are made of pairs).
  auto emit = [&](uint64_t e, uint32_t prev, uint32_t x) {
    if constexpr (OM == OUT_F64) {
      if (e & 1) {
        const double v = pair_f64<24>(prev, x);
        to.word(e - 1)[0] = __double2loint(v);
        to.word(e - 1)[1] = __double2hiint(v);
      }
    } else {
      *to.word(e) = tc_conv<OM>(x);
    }
  };

  uint32_t N[18], R[18];
  bool zero = false;
  lux_head(V, c, plan.h, reinterpret_cast<uint32_t*>(boxes[wi] + 4096) + 25 * lane, emit);   // in the second tile
  if (plan.nb == 0 && plan.m == 0) lux_store(d, row, active, V, c);   // ends inside the block that was open
  lux_load(V, c, N, zero);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tm = sh.tmem;
  lux_constants(tm);

  uint32_t chunk = (uint32_t)plan.h / 4;    // 16-byte chunk of the row that the next block starts at
  // The 24 words of N into the tiles; complete tiles are stored.
  auto deliver = [&]() {
    lux_words(N, R);
    if (zero) {
#pragma unroll
      for (int i = 0; i < 18; i++) R[i] = 0;
    }
    to.acquire();
    to.put4(chunk, lux_chunk<OM, 0>(R));
    to.put4(chunk + 1, lux_chunk<OM, 1>(R));
    to.put4(chunk + 2, lux_chunk<OM, 2>(R));
    to.put4(chunk + 3, lux_chunk<OM, 3>(R));
    to.put4(chunk + 4, lux_chunk<OM, 4>(R));
    to.put4(chunk + 5, lux_chunk<OM, 5>(R));
    chunk += 6;
    to.release(chunk >> 3);
  };

  bool ok = true;
  const uint64_t products = plan.nb + (plan.m > 0 ? 1 : 0);
  for (uint64_t it = 0; it < products; it++) {
    if (!lux_issue(sh, tm, N, !ok)) break;
    if (it > 0) deliver();                        // the previous block, while the product runs
    ok = lux_take(sh, tm, (uint32_t)it & 1u, N) && ok;
  }
  ok = !__syncthreads_or(!ok);                    // also: no product reads the table any more
  if (!ok) {
    if (tid == 0) lux_give_up();
  } else {
    if (products > 0) {
      if (plan.m == 0) {
        deliver();
      } else {
        lux_back24(N);                            // the state at the start of the open block
        lux_words(N, R);
        if (zero) {
#pragma unroll
          for (int i = 0; i < 18; i++) R[i] = 0;
        }
      }
      to.acquire();
      const uint64_t e0 = d.n_per - plan.m;
      lux_finish(d, row, active, N, R, plan.m, reinterpret_cast<uint32_t*>(sh.tab) + 25 * tid,
                     [&](uint64_t k, uint32_t prev, uint32_t x) { emit(e0 + k, prev, x); });
    }
    to.release((uint32_t)((d.n_per + kBox - 1) / kBox));
  }
  if (lane == 0) tc::tile_store_wait_read();
  lux_teardown(tm);
}

// The same for any output (unaligned rows, the fused half-sweep, host memory)
// through a per-row ring of 56 words that the warp copies out 32 words at a time.
// Unaligned rows are stored word by word (or double by double) from eight rows held
// in registers: a row at a time, each load waiting for the one before, took 311 us for
// 30,320 x 1,001 doubles at p = 223 and 222 for 131,072 x 1,001 words; now 147 and 219
// (the borrow chain 192 and 310).
template <int OM>
__global__ void __launch_bounds__(128, 4) k_fill_ranlux_tc(const FillDesc d, int level, bool vec) {
  __shared__ __align__(128) TcTable sh;
  __shared__ __align__(16) uint32_t rings[128 * kRowWords];
  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const uint64_t nr = d.n_rows;
  const uint64_t row = (uint64_t)blockIdx.x * 128 + tid;
  const uint64_t wrow0 = (uint64_t)blockIdx.x * 128 + wi * 32;
  const bool active = row < nr;
  uint32_t* out = static_cast<uint32_t*>(d.out);
  const bool store = out != nullptr;
  uint32_t* my = rings + tid * kRowWords;
  const uint32_t* wrows = rings + wi * 32 * kRowWords;

  uint32_t V[24], c;
  lux_state(d, row, active, V, c);
  lux_setup(sh);
  lux_operand(sh, level, 0);

  const LuxPlan plan(d);
  uint64_t fpos = 0;   // draws of the row written out
  int wc = 0, fc = 0;  // ring chunk of the next block / of the next copy-out
  int pend = 0;        // words in the ring not yet written out

  // Draw e of the row, straight to the output (heads and tails).
  auto emit = [&](uint64_t e, uint32_t prev, uint32_t x) {
    if (!active || !store) return;
    const uint64_t i = row * d.pitch + e;
    if constexpr (OM == OUT_F64) {
      if (e & 1) st_pair<24>(out + i - 1, prev, x);
    } else {
      put1<OM>(d, out + i, i, tc_conv<OM>(x));
    }
  };

  uint32_t N[18], R[18];
  bool zero = false;
  if (vec && (uint64_t)plan.h < d.n_per) {   // into the ring, with the first block
    lux_head(V, c, plan.h, my + 32, [&](uint64_t e, uint32_t, uint32_t x) { my[e] = lux_conv<OM>(x); });
    pend = plan.h;
    wc = plan.h / 4;
  } else {
    lux_head(V, c, plan.h, my + 32, emit);
    fpos = plan.h;
  }
  if (plan.nb == 0 && plan.m == 0) lux_store(d, row, active, V, c);   // ends inside the block that was open
  lux_load(V, c, N, zero);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tm = sh.tmem;
  lux_constants(tm);

  // k chunks (4 k words, k <= 8) of every row of the warp, from ring chunk fc to
  // row column fpos: a quarter-warp per row and 16 bytes per lane, or word by
  // word when the rows are not aligned.
  const int fq = lane & 7, fr = lane >> 3;
  auto copy_out = [&](int k) {
    __syncwarp();
    if (store) {
      if (vec) {
        if (fq < k) {
          int ch = fc + fq;
          if (ch >= kRC) ch -= kRC;
#pragma unroll
          for (int i = 0; i < 8; i++) {
            const uint64_t rr = wrow0 + fr + 4 * i;
            if (rr < nr)
              put4<OM, 24>(d, out + rr * d.pitch + fpos + 4 * fq, rr * d.pitch + fpos + 4 * fq,
                           *reinterpret_cast<const uint4*>(wrows + (fr + 4 * i) * kRowWords + 4 * ch));
          }
        }
      } else if (OM == OUT_ISING) {
        int w = 4 * fc + lane;
        if (w >= 4 * kRC) w -= 4 * kRC;
        for (int i = 0; lane < 4 * k && i < 32 && wrow0 + i < nr; i++) {
          const uint64_t e = (wrow0 + i) * d.pitch + fpos + lane;
          put1<OM>(d, out + e, e, wrows[i * kRowWords + w]);
        }
      } else if constexpr (OM == OUT_F64) {   // a half-warp per row, eight steps in flight
        const int c = 2 * (lane & 15), sub = lane >> 4;
        int w = 4 * fc + c;
        if (w >= 4 * kRC) w -= 4 * kRC;
        for (int i0 = 0; i0 < 32; i0 += 16) {
          uint2 v[8];
#pragma unroll
          for (int i = 0; i < 8; i++)
            v[i] = *reinterpret_cast<const uint2*>(wrows + (i0 + 2 * i + sub) * kRowWords + w);
          uint64_t rr = wrow0 + i0 + sub;
          uint32_t* p = out + rr * d.pitch + fpos + c;
#pragma unroll
          for (int i = 0; i < 8; i++) {
            if (c < 4 * k && rr < nr) st_pair<24>(p, v[i].x, v[i].y);
            rr += 2;
            p += 2 * d.pitch;
          }
        }
      } else {   // a warp per row, eight in flight
        int w = 4 * fc + lane;
        if (w >= 4 * kRC) w -= 4 * kRC;
        for (int i0 = 0; i0 < 32; i0 += 8) {
          uint32_t v[8];
#pragma unroll
          for (int i = 0; i < 8; i++) v[i] = wrows[(i0 + i) * kRowWords + w];
          uint64_t rr = wrow0 + i0;
          uint32_t* p = out + rr * d.pitch + fpos + lane;
#pragma unroll
          for (int i = 0; i < 8; i++) {
            if (lane < 4 * k && rr < nr) st_out(p, v[i]);
            rr++;
            p += d.pitch;
          }
        }
      }
    }
    __syncwarp();
    fpos += 4 * k;
    fc += k;
    if (fc >= kRC) fc -= kRC;
    pend -= 4 * k;
  };
  // The 24 words of N into the ring; out as soon as 32 are pending.
  auto deliver = [&]() {
    lux_words(N, R);
    if (zero) {
#pragma unroll
      for (int i = 0; i < 18; i++) R[i] = 0;
    }
    auto slot = [&](int q) {
      int ch = wc + q;
      if (ch >= kRC) ch -= kRC;
      return reinterpret_cast<uint4*>(my + 4 * ch);
    };
    *slot(0) = lux_quad<OM, 0>(R);
    *slot(1) = lux_quad<OM, 1>(R);
    *slot(2) = lux_quad<OM, 2>(R);
    *slot(3) = lux_quad<OM, 3>(R);
    *slot(4) = lux_quad<OM, 4>(R);
    *slot(5) = lux_quad<OM, 5>(R);
    wc += 6;
    if (wc >= kRC) wc -= kRC;
    pend += 24;
    if (pend >= 32) copy_out(8);
  };

  bool ok = true;
  const uint64_t products = plan.nb + (plan.m > 0 ? 1 : 0);
  for (uint64_t it = 0; it < products; it++) {
    if (!lux_issue(sh, tm, N, !ok)) break;
    if (it > 0) deliver();                        // the previous block, while the product runs
    ok = lux_take(sh, tm, (uint32_t)it & 1u, N) && ok;
  }
  ok = !__syncthreads_or(!ok);                    // also: no product reads the table any more
  if (!ok) {
    if (tid == 0) lux_give_up();
  } else if (products > 0) {
    if (plan.m == 0) {
      deliver();
    } else {
      lux_back24(N);                              // the state at the start of the open block
      lux_words(N, R);
      if (zero) {
#pragma unroll
        for (int i = 0; i < 18; i++) R[i] = 0;
      }
    }
    if (pend > 0) copy_out(pend / 4);
    lux_finish(d, row, active, N, R, plan.m, reinterpret_cast<uint32_t*>(sh.tab) + 25 * tid,
                   [&](uint64_t k, uint32_t prev, uint32_t x) { emit(fpos + k, prev, x); });
  }
  lux_teardown(tm);
}

// ------------------------------------------------- segments and batched fills
//
// A stream whose blocks one thread would walk for long is cut into segments of B
// = 2^lgb blocks, each a row of its own: k_lux_starts walks the segments' starts
// along their streams, B cycles per product, and k_lux_items fills the segments.
// The first kernel alone reads the streams' states and the second's last segments
// alone write them, so no row waits for another.  A work item is the 32 streams
// of one warp in one segment; the four warps of a CTA work on different items, of
// one request or several, and share each product.  A request's items lie segment
// after segment, all its streams in each.
//
// k_lux_starts takes the segments in groups of 16, each group's first start by
// products with 2^i x 16 B cycles for the bits of its number (a row keeps a
// product when its bit is set), the others one after the other: every segment's
// start by its own bits, with a state load, a head and an operand load per
// segment, took longer than it saved above 4,096 streams (65,536 x 256: 55 us
// against 31 uncut).

// What the second kernel needs of an item, in one place: the fill and where the
// item lies in it, then the words N[18] and the zero flag of its 32 streams side
// by side.
struct LuxHead {
  FillDesc d;
  uint64_t row0;
  const CUtensorMap* map;   // of a batched fill's output, or nullptr
  uint32_t seg, pad;
};
constexpr uint32_t kHeadWords = sizeof(LuxHead) / 4, kHeadPitch = 64;
static_assert(sizeof(LuxHead) % 4 == 0 && kHeadWords <= kHeadPitch, "copied as words by two lanes' turns");
constexpr uint32_t kStartWords = kHeadPitch + 19 * 32;

// Head of item `it`, by its warp.
__device__ __forceinline__ void lux_head_of(const LuxJob& job, uint32_t it, LuxHead* h) {
  const int lane = threadIdx.x & 31;
  uint32_t seg;
  uint64_t row0;
  const CUtensorMap* map;
  if (job.reqs != nullptr) {
    const BatchItem b = job.items[it];
    seg = b.rows;
    row0 = b.row0;
    map = job.reqs[b.req].tiles ? job.maps + b.req : nullptr;
    load_desc(&h->d, job.reqs[b.req].d, lane, 32);
  } else {
    seg = it / job.warps;
    row0 = 32ull * (it - seg * job.warps);
    map = nullptr;   // the job's own
    load_desc(&h->d, job.one, lane, 32);
  }
  if (lane == 0) {
    h->row0 = row0;
    h->map = map;
    h->seg = seg;
  }
  __syncwarp();
}

__global__ void __launch_bounds__(128, 4) k_lux_starts(const __grid_constant__ LuxJob job, int level) {
  __shared__ __align__(128) TcTable sh;
  __shared__ uint32_t scratch[128 * 25];
  __shared__ LuxHead heads[4];
  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const uint32_t g = blockIdx.x * 4 + wi;     // the groups' first items
  const bool have = g < job.n_groups;
  const uint32_t it = !have                 ? 0
                      : job.firsts != nullptr ? job.firsts[g]
                      : job.reqs != nullptr   ? g
                                              : lux_first_item(g, job.warps);
  lux_setup(sh);

  uint32_t N[18];
  uint32_t seg = 0, cnt = 0, warps = 0;   // first segment and segments of this group; items from one to the next
  bool zero = false;
  if (have) {
    lux_head_of(job, it, &heads[wi]);
    const FillDesc& d = heads[wi].d;
    const uint64_t row = heads[wi].row0 + lane;
    const bool active = row < d.n_rows;
    seg = heads[wi].seg;
    const LuxPlan plan(d);
    // As many as the host counted when it sized the items: from the same function.
    cnt = lux_group_size(job.max_seg > 0 ? lux_segments(d.n_per, job.lgb) : 1, seg);
    warps = (uint32_t)((d.n_rows + 31) / 32);
    uint32_t V[24], c;
    lux_state(d, row, active, V, c);
    uint32_t* out = static_cast<uint32_t*>(d.out);
    lux_head(V, c, plan.h, scratch + 25 * tid, [&](uint64_t k, uint32_t prev, uint32_t x) {
      const uint64_t e = row * d.pitch + k;
      if (seg != 0 || !active || e >= d.limit) return;   // the first group writes the head
      if (d.mode == OUT_F64) {
        if (k & 1) st_pair<24>(out + e - 1, prev, x);
      } else {
        st_out(out + e, d.mode == OUT_F32 ? tc_conv<OUT_F32>(x) : x);
      }
    });
    if (plan.nb == 0 && plan.m == 0) lux_store(d, row, active, V, c);   // ends inside the open block
    lux_load(V, c, N, zero);
  } else {
#pragma unroll
    for (int i = 0; i < 18; i++) N[i] = d_word(i);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tm = sh.tmem;
  lux_constants(tm);
  bool ok = true;
  uint32_t products = 0;
  // To the group's first segment, by the bits of its number.
  const uint32_t group = have ? seg / kLuxGroup : 0;
  for (int i = 0; __syncthreads_or((group >> i) != 0); i++) {
    const bool take = (group >> i) & 1u;
    if (!__syncthreads_or(take)) continue;          // also: the operand is not in use any more
    lux_operand(sh, level, job.lgb + kLgLuxGroup + i);
    if (!lux_issue(sh, tm, N, !ok)) break;
    uint32_t T[18];
    ok = lux_take(sh, tm, products & 1u, T) && ok;
    products++;
    if (take) {
#pragma unroll
      for (int k = 0; k < 18; k++) N[k] = T[k];
    }
  }
  // Segment after segment.
  if (__syncthreads_or(cnt > 1)) lux_operand(sh, level, job.lgb);
  // The head of segment seg + j, by its warp; its item's start, or nullptr past the items.
  auto head = [&](uint32_t j) -> uint32_t* {
    if (j >= cnt || it + j * warps >= job.n_items) return nullptr;
    uint32_t* st = job.starts + (uint64_t)(it + j * warps) * kStartWords;
    if (lane == 0) heads[wi].seg = seg + j;
    __syncwarp();
    const uint32_t* h = reinterpret_cast<const uint32_t*>(&heads[wi]);
    for (uint32_t k = lane; k < kHeadWords; k += 32) st[k] = h[k];
    return st + kHeadPitch + lane;
  };
  for (uint32_t j = 0;; j++) {
    if (uint32_t* st = head(j)) {
#pragma unroll
      for (int k = 0; k < 18; k++) st[32 * k] = N[k];
      st[32 * 18] = zero ? 1u : 0u;
    }
    if (!__syncthreads_or(j + 1 < cnt) || !lux_issue(sh, tm, N, !ok)) break;
    ok = lux_take(sh, tm, products & 1u, N) && ok;
    products++;
  }
  // A CTA that gave up leaves heads without draws, so that the items' kernel skips
  // its segments instead of reading starts that were never written.
  if (__syncthreads_or(!ok)) {
    if (lane == 0) heads[wi].d.n_per = 0;
    for (uint32_t j = 0; j < cnt; j++) head(j);
  }
  if (!ok) lux_give_up();
  lux_teardown(tm);
}

// A warp's 32 rows of one segment: staging tiles as TileOut's, but any range of
// a tile can leave on its own, word by word, when it is cut by the segment's
// ends or the request's limit, or when the rows are not 16-byte aligned.
struct SegOut {
  uint8_t* box;
  const CUtensorMap* map;   // of the limit's whole rows; nullptr: word by word
  uint32_t rowb;
  uint32_t off;             // element of the row at tile 0, word 0
  uint32_t lo;              // first word of the segment in its first tile
  uint64_t whole;           // rows before the one that the request's limit cuts
  uint64_t done, pos;       // tiles left behind / words staged, counted from `off`

  __device__ __forceinline__ uint32_t at(uint32_t chunk) const {
    return rowb ^ ((chunk & 7u) << 4) ^ ((chunk & 8u) << 9);
  }
  __device__ __forceinline__ void put4(uint32_t q, uint4 v) const {
    *reinterpret_cast<uint4*>(box + at((uint32_t)(pos >> 2) + q)) = v;
  }
  __device__ __forceinline__ void acquire() const {
    if ((threadIdx.x & 31) == 0) tc::tile_store_wait_read();
    __syncwarp();
  }
  // Words [from, to) of tile `done` of the rows [r0, r1) of the warp.
  __device__ __forceinline__ void words(const FillDesc& d, uint64_t row0, int r0, int r1, uint32_t from,
                                        uint32_t to) const {
    const uint32_t lane = threadIdx.x & 31;
    const uint8_t* b = box + (done & 1) * 4096 + (lane & 3) * 4;
    uint32_t* out = static_cast<uint32_t*>(d.out);
    if (lane < from || lane >= to) return;
    const uint64_t e0 = row0 * d.pitch + 32 * done + off + lane;
    auto at_row = [&](int r) {
      return *reinterpret_cast<const uint32_t*>(b + r * 128 + (((lane >> 2) ^ (r & 7)) << 4));
    };
    if (r1 - r0 == 32 && e0 + 31 * d.pitch < d.limit) {   // the usual case: eight rows in flight
      uint32_t* p = out + e0;
      const uint64_t pitch = d.pitch;
      for (int r = 0; r < 32; r += 8) {
        uint32_t v[8];
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = at_row(r + k);
#pragma unroll
        for (int k = 0; k < 8; k++) {
          st_out(p, v[k]);
          p += pitch;
        }
      }
      return;
    }
    for (int r = r0; r < r1; r++) {
      const uint64_t e = e0 + r * d.pitch;
      if (e < d.limit) st_out(out + e, at_row(r));
    }
  }
  // Tile `done`, words up to `to`, leaves.
  __device__ __forceinline__ void leave(const FillDesc& d, uint64_t row0, uint32_t to) {
    const uint64_t left = d.n_rows - row0;
    const int rows = left < 32 ? (int)left : 32;
    if (map != nullptr && lo == 0 && to == kBox) {
      tc::fence_smem_to_async();
      __syncwarp();
      if ((threadIdx.x & 31) == 0 && row0 < whole)
        tc::tile_store(map, tc::smem_addr(box) + (uint32_t)(done & 1) * 4096u, (uint32_t)done * kBox, (uint32_t)row0);
      if (whole >= row0 && whole < row0 + rows)
        words(d, row0, (int)(whole - row0), (int)(whole - row0) + 1, 0, kBox);
    } else {
      __syncwarp();
      words(d, row0, 0, rows, lo, to);
    }
    lo = 0;
    done++;
  }
};

// Segments of one luxury level's fills.
//
// Per warp and product as k_fill_ranlux_tiles; a CTA's four warps are at
// different places of different items and meet only at the products.
template <int OM>
__global__ void __launch_bounds__(128, 4) k_lux_items(const __grid_constant__ LuxJob job, int level) {
  __shared__ __align__(1024) uint8_t boxes[4][2 * 4096];
  __shared__ __align__(128) TcTable sh;
  __shared__ LuxHead heads[4];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  lux_setup(sh);
  lux_operand(sh, level, 0);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tm = sh.tmem;
  lux_constants(tm);

  const FillDesc& d = heads[wi].d;
  SegOut so{};
  so.box = boxes[wi];
  so.rowb = (uint32_t)(lane * 128 + ((lane & 7) << 4));
  // The next item, in lane 0: popped when the one before it starts, so that it is
  // there when it is wanted; the warps of a single fill take theirs in turn.
  uint32_t next = blockIdx.x * 4 + wi;
  if (job.counter != nullptr && lane == 0) next = atomicAdd(job.counter, 1u);
  bool have = false, dry = false, due = false, zero = false, last = false, ok = true;
  uint64_t row0 = 0, left = 0;
  int m = 0;
  uint32_t N[18], R[18];
#pragma unroll
  for (int i = 0; i < 18; i++) N[i] = d_word(i);

  auto words = [&]() {
    lux_words(N, R);
    if (zero) {
#pragma unroll
      for (int i = 0; i < 18; i++) R[i] = 0;
    }
  };
  auto deliver = [&]() {
    words();
    so.acquire();
    so.put4(0, lux_chunk<OM, 0>(R));
    so.put4(1, lux_chunk<OM, 1>(R));
    so.put4(2, lux_chunk<OM, 2>(R));
    so.put4(3, lux_chunk<OM, 3>(R));
    so.put4(4, lux_chunk<OM, 4>(R));
    so.put4(5, lux_chunk<OM, 5>(R));
    so.pos += 24;
    if ((so.pos >> 5) > so.done) so.leave(d, row0, kBox);
  };

  for (uint32_t it = 0;; it++) {
    while (!have && !dry && ok) {         // this warp's next item that needs a product
      const uint32_t i = __shfl_sync(0xFFFFFFFFu, next, 0);
      dry = i >= job.n_items;
      if (dry) break;
      if (job.counter == nullptr) next += gridDim.x * 4;
      else if (lane == 0) next = atomicAdd(job.counter, 1u);
      const uint32_t* st = job.starts + (uint64_t)i * kStartWords;
      uint32_t* h = reinterpret_cast<uint32_t*>(&heads[wi]);
      __syncwarp();
      for (uint32_t k = lane; k < kHeadWords; k += 32) h[k] = st[k];
      st += kHeadPitch + lane;
#pragma unroll
      for (int k = 0; k < 18; k++) N[k] = st[32 * k];
      zero = st[32 * 18] != 0;
      __syncwarp();
      const LuxPlan plan(d);
      const uint64_t b0 = (uint64_t)heads[wi].seg << job.lgb;
      if (b0 > 0 && plan.nb <= b0) continue;   // an empty last segment, or a start that was given up
      uint64_t nb = plan.nb - b0;
      last = true;
      if (job.max_seg > 0 && nb > 1ull << job.lgb) {
        nb = 1ull << job.lgb;
        last = false;
      }
      m = last ? plan.m : 0;
      left = nb + (m > 0 ? 1 : 0);
      if (left == 0) continue;            // all of it in the block that was open
      row0 = heads[wi].row0;
      const uint64_t e0 = plan.h + 24 * b0;
      so.off = (uint32_t)(e0 & 3);
      so.pos = e0 - so.off;
      so.done = so.pos >> 5;
      so.lo = (uint32_t)(so.pos & 31);
      so.map = so.off != 0 ? nullptr : job.reqs != nullptr ? heads[wi].map : job.tiles ? &job.map : nullptr;
      // A batch's maps are in memory that the host rewrites between launches; a
      // single fill's is a kernel parameter.  The lane that stores the tiles waits.
      if (so.map != nullptr && job.reqs != nullptr && lane == 0) tc::map_acquire(so.map);
      so.whole = d.limit / d.pitch;
      have = true;
    }
    lux_digits(tm, N);
    if (!__syncthreads_or(have)) break;
    if (wi == 0) lux_product(sh, tm);
    if (due) deliver();                   // the previous block, while the product runs
    due = false;
    // A warp whose wait gives up drops its item and takes no other.
    ok = __all_sync(0xFFFFFFFFu, lux_take(sh, tm, it & 1u, N)) && ok;
    have = have && ok;
    if (!have) continue;
    if (--left > 0) {
      due = true;
      continue;
    }
    if (m == 0) {
      deliver();
    } else {
      lux_back24(N);                      // the state at the start of the open block
      words();
    }
    if (so.pos & 31) so.leave(d, row0, (uint32_t)(so.pos & 31));
    so.acquire();                         // the tiles are free
    if (last) {
      const uint64_t row = row0 + lane;
      const bool active = row < d.n_rows;
      uint32_t* out = static_cast<uint32_t*>(d.out);
      lux_finish(d, row, active, N, R, m, reinterpret_cast<uint32_t*>(so.box) + 25 * lane,
                 [&](uint64_t k, uint32_t prev, uint32_t x) {
                   const uint64_t e = row * d.pitch + d.n_per - m + k;
                   if (!active || e >= d.limit) return;
                   if constexpr (OM == OUT_F64) {
                     if (k & 1) st_pair<24>(out + e - 1, prev, x);
                   } else {
                     st_out(out + e, tc_conv<OM>(x));
                   }
                 });
      __syncwarp();
    }
    have = false;
  }
  if (!ok && lane == 0) lux_give_up();
  if (lane == 0) tc::tile_store_wait_read();
  lux_teardown(tm);
}

int level_of(int p) {
  for (int i = 0; i < kLevels; i++)
    if (kLevelP[i] == p) return i;
  return -1;
}

}  // namespace

bool lux_out_map(void* out, uint64_t pitch, uint64_t rows, CUtensorMap* map) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<Encode>(f);
  }();
  if (encode == nullptr || out == nullptr || (reinterpret_cast<uintptr_t>(out) & 15) != 0 ||
      !lux_tiles_reach(pitch, rows))
    return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, out) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int dev = -1;
  cudaGetDevice(&dev);
  if (at.type != cudaMemoryTypeDevice || at.device != dev) return false;
  const cuuint64_t dim[2] = {pitch, rows}, stride[1] = {4 * pitch};
  const cuuint32_t box[2] = {(cuuint32_t)kBox, (cuuint32_t)kBox}, step[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, out, dim, stride, box, step,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

uint64_t lux_start_bytes(uint64_t items) { return items * kStartWords * sizeof(uint32_t); }

LuxSplit lux_split(uint64_t warp_blocks, uint64_t longest) {
  return lux_split(warp_blocks, longest, (uint64_t)sm_count());
}

cudaError_t launch_lux_job(const LuxJob& job, int p, int mode, cudaStream_t s) {
  if (job.n_items == 0) return cudaSuccess;
  const int level = level_of(p);
  if (level < 0) return cudaErrorInvalidValue;
  const uint32_t ctas = (job.n_items + 3) / 4, cap = 4 * (uint32_t)sm_count();
  k_lux_starts<<<(job.n_groups + 3) / 4, 128, 0, s>>>(job, level);
  const uint32_t grid = ctas < cap ? ctas : cap;
  switch (mode) {
    case OUT_U32: k_lux_items<OUT_U32><<<grid, 128, 0, s>>>(job, level); break;
    case OUT_F32: k_lux_items<OUT_F32><<<grid, 128, 0, s>>>(job, level); break;
    case OUT_F64: k_lux_items<OUT_F64><<<grid, 128, 0, s>>>(job, level); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// A plain fill cut into segments (scratch for their starts from the retained pool).
static cudaError_t launch_segments(const FillDesc& d, const LuxSplit& sp, cudaStream_t s) {
  LuxJob job{};
  const uint64_t warps = (d.n_rows + 31) / 32, segs = lux_segments(d.n_per, sp.lgb);
  if (warps * segs > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  job.one = d;
  job.warps = (uint32_t)warps;
  job.n_items = (uint32_t)(warps * segs);
  job.lgb = sp.lgb;
  job.max_seg = (uint32_t)segs - 1;
  job.n_groups = (uint32_t)lux_groups(segs, warps);
  job.tiles = lux_out_map(d.out, d.pitch, d.n_rows, &job.map) ? 1 : 0;
  cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&job.starts), lux_start_bytes(job.n_items), s);
  if (e != cudaSuccess) return e;
  e = launch_lux_job(job, d.p, d.mode, s);
  const cudaError_t ef = scratch_free(job.starts, s);
  return e != cudaSuccess ? e : ef;
}

cudaError_t launch_fill_ranlux_tc(const FillDesc& d, bool segments, cudaStream_t s) {
  const int level = level_of(d.p);
  if (level < 0) return cudaErrorInvalidValue;
  if (segments && d.out != nullptr && d.mode != OUT_ISING) {
    const LuxSplit sp = lux_split((d.n_rows + 31) / 32 * (d.n_per / 24), d.n_per / 24);
    if (sp.cut && !capturing(s)) {
      const cudaError_t e = launch_segments(d, sp, s);
      if (e != cudaErrorMemoryAllocation) return e;
      cudaGetLastError();
    }
  }
  const bool vec = (d.pos >= 24 || (d.pos & 3) == 0) && (d.pitch & 3) == 0 &&
                   (d.mode == OUT_ISING || (reinterpret_cast<uintptr_t>(d.out) & 15) == 0);
  const uint64_t grid = (d.n_rows + 127) / 128;
  CUtensorMap map;
  const bool tiles = vec && d.mode != OUT_ISING && lux_out_map(d.out, d.pitch, d.n_rows, &map);
  return with_mode(d.mode, [&](auto mode) {
    constexpr int OM = decltype(mode)::value;
    if constexpr (OM != OUT_ISING) {
      if (tiles) {
        k_fill_ranlux_tiles<OM><<<(unsigned)grid, 128, 0, s>>>(d, level, map);
        return cudaGetLastError();
      }
    }
    k_fill_ranlux_tc<OM><<<(unsigned)grid, 128, 0, s>>>(d, level, vec);
    return cudaGetLastError();
  });
}

}  // namespace prng
