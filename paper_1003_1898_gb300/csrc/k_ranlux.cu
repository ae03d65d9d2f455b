// k_ranlux.cu -- RANLUX entry points (Section 3.6; Appendix A, "RANLUX"):
// dispatch on the luxury p to the launchers compiled per level (the standard
// p = 24, 48, 97, 223, 389 and the planar scheme's p = 120, 240, 408).
#include <algorithm>

#include "ranlux.cuh"
#include "ranlux_tc.cuh"

namespace prng {

PRNG_RANLUX_DECLARE(24)
PRNG_RANLUX_DECLARE(48)
PRNG_RANLUX_DECLARE(97)
PRNG_RANLUX_DECLARE(223)
PRNG_RANLUX_DECLARE(389)
PRNG_RANLUX_DECLARE(120)
PRNG_RANLUX_DECLARE(240)
PRNG_RANLUX_DECLARE(408)

// The tensor-core form costs the same per block at every p, the borrow chain p
// steps.  Cycles per block of each on a busy SM, from fills of 256 to 131,072
// streams: the chain's latency (4.9 per step and about 590 for the block's
// output) while its warps have a scheduler each, 4.25 per step and 280 per warp
// of the busiest scheduler beyond; the product's round trip (1,250 and 365 per
// tile of 128 streams on the SM, four tiles at a time).  Setting the product up
// costs about 6,500 cycles more than starting a chain (and 300 per tile on the SM:
// 131,072 x 61 at p = 223 25.8 / 28.2), cutting streams into
// segments 30,000 (a second kernel, the segments' starts) plus a product per
// segment up to 16 and about four per segment filled.  Measured in us, chain /
// product / segments: 65,536 x 4,096 u32 at p = 97 230 / 234 / -, p = 120 258 /
// 233, 223 405 / 234, 389 640 / 233; 4,096 x 4,096 at p = 223 139 / 133 / 52;
// 16,384 x 4,096 143 / 136 / 99; 256 x 8,192 265 / 249 / 43; 16,384 x 1,024 47 /
// 46 / 48; 32,768 x 1,024 68 / 53 / 65; 1,024 x 1,024 45 / 45 / 37; 4,096 x 248
// 20 / 22 / 35.  Fused half-sweeps go through the ring form of the product,
// whose short rows pay off later (4096^2 over 65,536 streams, 128 draws each, p =
// 223: 50 / 55; over 4,096, 2,048 draws each, p = 389: 550 / 470).
//
// Long rows that are not 16-byte aligned are stored word by word (a double at a
// time), which bounds both forms once the SMs are busy: about 2,150 cycles a block and
// warp of the busiest scheduler for the chain (doubles 1,900), 1,540 a block and
// tile on the SM for the product (1,450); and the chain waits longer for its own
// copies below that.  Segments are as fast as of aligned rows until they take more
// than one round.  The product (not the chain) also stores so when the open block
// leaves no multiple of 4 draws.  us, chain / product / segments, p = 97: 131,072 x
// 1,001 u32 320 / 220 / 251; 30,320 x 1,001 66 / 52 / 67, f64 152 / 147 / 124;
// 4,096 x 1,001 42 / 41 / 29.  Short rows lie close together in memory and cost what
// aligned ones do (131,072 x 61 u32 25.5 / 28.3).
Tile ranlux_auto_tile(const FillDesc& d) {
  // The borrow chain's own tile.  The ring, or where rows are not aligned 48 staged
  // columns at p < 97 and 96 above; but 48 for short rows of many streams (p = 24,
  // ring / 48: 131,072 x 64 27 / 23, 30,320 x 64 6.3 / 5.5, x 160 8.5 / 8.0, x 248 9.5
  // / 10.1, 20,000 x 64 5.2 / 4.8; p = 97 40,000 x 100 10.1 / 9.5; 96 / 48 at p = 223,
  // 131,072 x 13 16 / 14, 4,096 x 127 10.3 / 11.9).
  // Long rows at p = 48 take wide CTAs (131,072 x 8,192 781 / 714, 4,096 x 4,096 70 /
  // 95), of about 100,000 streams at p = 24 CTAs of 128 (98,304 x 8,192 596 / 538,
  // 131,072 x 8,192 781 / 766, x 4,096 388 / 382; 200,000 x 4,096 549 / 549; 65,536 x
  // 4,096 205 / 213; doubles no faster).
  // A skip, which writes nothing, is faster without the ring (65,536 x 2,400 at p = 24
  // 48 / 37; at p = 223 203, the product 114).
  const bool ring = ranlux_ring_ok(d);
  Tile t = ring || d.p < 97 ? Tile{64, 56, 1} : Tile{64, 96, 1};
  if (d.out == nullptr) t = Tile{128, 48, 1};
  else if (d.n_rows >= 20000 && d.n_per < 200 && (d.n_per >= 32 || !ring)) t = Tile{64, 48, 1};
  else if (d.p < 97 && d.n_rows >= 36000 && d.n_per < 320) t = Tile{64, 48, 1};
  else if (d.p == 48 && d.n_rows >= 65536 && d.n_per >= 1024) t = Tile{256, 56, 1};
  else if (d.p == 24 && d.mode != OUT_F64 && d.n_rows >= 98304 && d.n_rows <= 131072 && d.n_per >= 4096)
    t = Tile{128, 56, 1};
  // Long unaligned rows at p < 97 leave through the staged tile: in CTAs of 128 where
  // the busiest SM holds no more threads that way (30,320 x 2,047 at p = 24 143 / 136,
  // 50,000 x 4,095 503 / 485; but 25,000 x 2,047 100 / 118, 65,536 x 4,095 at p = 48
  // 660 / 697, and below 28,000 streams, 16,384 x 2,047, 76 / 78).
  if (d.out != nullptr && d.p < 97 && !ring && (d.mode == OUT_U32 || d.mode == OUT_F32) &&
      d.n_rows >= 28000 && d.n_rows < 65536 && d.n_per >= 1000) {
    const uint64_t sms = (uint64_t)sm_count(), c64 = (d.n_rows + 63) / 64, c128 = (d.n_rows + 127) / 128;
    if ((c64 + sms - 1) / sms == 2 * ((c128 + sms - 1) / sms)) t = Tile{128, 48, 1};
  }
  if (d.p < kLuxTcMinP || d.n_per < 24) return t;
  const uint64_t nb = d.n_per / 24, p = (uint64_t)d.p, sms = (uint64_t)sm_count();
  const bool stored = d.out != nullptr && d.mode != OUT_ISING, f64 = d.mode == OUT_F64;
  const bool odd_rows = stored && d.n_per >= 192 && ((d.pitch & 3) != 0 || (reinterpret_cast<uintptr_t>(d.out) & 15) != 0);
  const bool words = odd_rows || (stored && d.n_per >= 192 && d.pos < 24 && (d.pos & 3) != 0);   // the product stores word by word
  auto per_sm = [&](uint64_t tiles) { return (tiles + sms - 1) / sms; };
  auto product = [&](uint64_t tiles) {   // cycles of a product with `tiles` tiles to run
    const uint64_t c = per_sm(tiles);
    return (c <= 4 ? 1250 + 365 * c : 675 * c) * 106 / 100;
  };
  const uint64_t warps = (d.n_rows + 31) / 32, tiles = (d.n_rows + 127) / 128, c = per_sm(tiles);
  const uint64_t per_sched = (warps + 4 * sms - 1) / (4 * sms);
  const uint64_t wait = odd_rows ? (f64 ? 5 * p + 2850 : 47 * p / 10 + 1640) : (49 * p + 5900) / 10;
  const uint64_t warp = std::max<uint64_t>((17 * p + 1120) / 4, odd_rows ? (f64 ? 1900 : 2150) : 0);
  uint64_t best = nb * std::max<uint64_t>(wait, per_sched * warp);
  auto offer = [&](uint64_t cycles, Tile tile) {
    if (cycles < best) {
      best = cycles;
      t = tile;
    }
  };
  if (words)
    offer(3000 + 300 * c + nb * (c <= 2 ? (f64 ? 2880 + 390 * c : 1500 + 550 * c) : (f64 ? 1450 : 1540) * c),
          Tile{128, 24, 1});
  else
    offer((d.mode == OUT_ISING ? 40000 : 6500 + 300 * c) + nb * product(tiles), Tile{128, 24, 1});
  const LuxSplit sp = lux_split(warps * nb, nb);
  if (sp.cut && stored && nb < 1ull << 40) {   // a skip has no segments
    const uint64_t B = 1ull << sp.lgb, segs = (nb + B - 1) / B, slots = 16 * sms;
    const uint64_t rounds = (warps * segs + slots - 1) / slots;
    const uint64_t fill = rounds * (B + 4) * product(std::min<uint64_t>((warps * segs + 3) / 4, 4 * sms));
    offer(30000 + std::min<uint64_t>(segs, 16) * product(std::min<uint64_t>(tiles, 4 * sms)) +
              (words && rounds > 1 ? fill * 3 / 2 : fill),
          Tile{128, 24, 2});
  }
  return t;
}

cudaError_t launch_fill_ranlux(const FillDesc& d, Tile t, cudaStream_t s) {
  if (d.n_rows == 0 || d.n_per == 0) return cudaSuccess;
  if (t.cols == 24 && d.p >= kLuxTcMinP) return launch_fill_ranlux_tc(d, t.stages == 2, s);
  switch (d.p) {
    case 24: return ranlux_fill_p<24>(d, t, s);
    case 48: return ranlux_fill_p<48>(d, t, s);
    case 97: return ranlux_fill_p<97>(d, t, s);
    case 223: return ranlux_fill_p<223>(d, t, s);
    case 389: return ranlux_fill_p<389>(d, t, s);
    case 120: return ranlux_fill_p<120>(d, t, s);
    case 240: return ranlux_fill_p<240>(d, t, s);
    case 408: return ranlux_fill_p<408>(d, t, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_batch_ranlux(const BatchQueue& q, int p, Tile t, bool f32, cudaStream_t s) {
  if (q.n_items == 0) return cudaSuccess;
  switch (p) {
    case 24: return ranlux_batch_p<24>(q, t, f32, s);
    case 48: return ranlux_batch_p<48>(q, t, f32, s);
    case 97: return ranlux_batch_p<97>(q, t, f32, s);
    case 223: return ranlux_batch_p<223>(q, t, f32, s);
    case 389: return ranlux_batch_p<389>(q, t, f32, s);
    case 120: return ranlux_batch_p<120>(q, t, f32, s);
    case 240: return ranlux_batch_p<240>(q, t, f32, s);
    case 408: return ranlux_batch_p<408>(q, t, f32, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace prng
