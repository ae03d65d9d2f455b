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
// costs about 6,500 cycles more than starting a chain, cutting streams into
// segments 30,000 (a second kernel, the segments' starts) plus a product per
// segment up to 16 and about four per segment filled.  Measured in us, chain /
// product / segments: 65,536 x 4,096 u32 at p = 97 230 / 234 / -, p = 120 258 /
// 233, 223 405 / 234, 389 640 / 233; 4,096 x 4,096 at p = 223 139 / 133 / 52;
// 16,384 x 4,096 143 / 136 / 99; 256 x 8,192 265 / 249 / 43; 16,384 x 1,024 47 /
// 46 / 48; 32,768 x 1,024 68 / 53 / 65; 1,024 x 1,024 45 / 45 / 37; 4,096 x 248
// 20 / 22 / 35.  Fused half-sweeps go through the ring form of the product,
// whose short rows pay off later (4096^2 over 65,536 streams, 128 draws each, p =
// 223: 50 / 55; over 4,096, 2,048 draws each, p = 389: 550 / 470).
Tile ranlux_auto_tile(const FillDesc& d) {
  // The borrow chain's own tile: the ring, but for short rows of many streams
  // (131,072 x 64 at p = 24 27 / 23 us without it, x 248 41 / 37), at p >= 97 of
  // unaligned rows too (96 columns / 48: 131,072 x 13 at p = 223 16 / 14, x 61 27.6 /
  // 25.8; 30,320 x 127 15.3 / 14.4, 4,096 x 127 10.3 / 11.9); in wide CTAs
  // for long rows at p = 48 (131,072 x 8,192 781 / 714, 4,096 x 4,096 70 / 95), in
  // CTAs of 128 for long rows of about 100,000 streams at p = 24 (98,304 x 8,192 596 /
  // 538, 131,072 x 8,192 781 / 766, x 4,096 388 / 382; 200,000 x 4,096 549 / 549;
  // 65,536 x 4,096 205 / 213; doubles no faster).
  // A skip, which writes nothing, is faster without the ring (65,536 x 2,400 at p = 24
  // 48 / 37; at p = 223 203, the product 114).
  Tile t = d.out == nullptr                   ? Tile{128, 48, 1}
           : ranlux_ring_ok(d) || d.p < 97    ? Tile{64, 56, 1}
           : d.n_rows >= 30000 && d.n_per < 192 ? Tile{64, 48, 1}
                                                : Tile{64, 96, 1};
  if (d.out != nullptr && d.p < 97 && d.n_rows >= 32768) {
    if (d.n_per < 320) t = Tile{64, 48, 1};
    else if (d.p == 48 && d.n_rows >= 65536 && d.n_per >= 1024) t = Tile{256, 56, 1};
    else if (d.p == 24 && d.mode != OUT_F64 && d.n_rows >= 98304 && d.n_rows <= 131072 && d.n_per >= 4096)
      t = Tile{128, 56, 1};
  }
  // Long unaligned rows at p < 97 leave through the staged tile: in CTAs of 128 where
  // the busiest SM holds no more threads that way (30,320 x 2,047 at p = 24 143 / 136,
  // 50,000 x 4,095 503 / 485; but 25,000 x 2,047 100 / 118, 65,536 x 4,095 at p = 48
  // 660 / 697, and below 28,000 streams, 16,384 x 2,047, 76 / 78).
  if (d.out != nullptr && d.p < 97 && !ranlux_ring_ok(d) && (d.mode == OUT_U32 || d.mode == OUT_F32) &&
      d.n_rows >= 28000 && d.n_rows < 65536 && d.n_per >= 1000) {
    const uint64_t sms = (uint64_t)sm_count(), c64 = (d.n_rows + 63) / 64, c128 = (d.n_rows + 127) / 128;
    if ((c64 + sms - 1) / sms == 2 * ((c128 + sms - 1) / sms)) t = Tile{128, 48, 1};
  }
  if (d.p < kLuxTcMinP || d.n_per < 24) return t;
  const uint64_t nb = d.n_per / 24, p = (uint64_t)d.p, sms = (uint64_t)sm_count();
  auto product = [&](uint64_t tiles) {   // cycles of a product with `tiles` tiles to run
    const uint64_t c = (tiles + sms - 1) / sms;
    return (c <= 4 ? 1250 + 365 * c : 675 * c) * 106 / 100;
  };
  const uint64_t warps = (d.n_rows + 31) / 32, tiles = (d.n_rows + 127) / 128;
  const uint64_t per_sched = (warps + 4 * sms - 1) / (4 * sms);
  uint64_t best = nb * std::max<uint64_t>((49 * p + 5900) / 10, per_sched * ((17 * p + 1120) / 4));
  auto offer = [&](uint64_t cycles, Tile tile) {
    if (cycles < best) {
      best = cycles;
      t = tile;
    }
  };
  offer((d.mode == OUT_ISING ? 40000 : 6500) + nb * product(tiles), Tile{128, 24, 1});
  const LuxSplit sp = lux_split(warps * nb, nb);
  if (sp.cut && d.mode != OUT_ISING && d.out != nullptr && nb < 1ull << 40) {   // a skip has no segments
    const uint64_t B = 1ull << sp.lgb, segs = (nb + B - 1) / B, slots = 16 * sms;
    const uint64_t rounds = (warps * segs + slots - 1) / slots;
    offer(30000 + std::min<uint64_t>(segs, 16) * product(std::min<uint64_t>(tiles, 4 * sms)) +
              rounds * (B + 4) * product(std::min<uint64_t>((warps * segs + 3) / 4, 4 * sms)),
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
