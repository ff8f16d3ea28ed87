// k_syrk_digits.cu -- partials of the P64 covariance call from exact integer
// products on the tensor cores.
//
// FP64 runs at 1/67 of the FP32 rate on this GPU (1.9 FMAs per clock and SM
// against 128), so that S2 = sum_n x_n x_n^T of 350 x 350 pixels of 188 bands costs
// 3.6 ms at its full rate.  Here x = y - s is held as a 56-bit fixed-point number per band
// and written as seven signed 8-bit digits D_0 .. D_6 (splitting into slices whose
// products are exact: Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).
// Digits are exact in FP16, a product of two is at most 2^14, and the sums over a chunk of
// 32 pixels of all pairs (i, j) of one level i + j stay below 2^22: exact in the FP32
// accumulators.  They are then added as integers of 64 bits in three units, and a
// partial is rounded at its end.  All levels, 0 .. 12, are formed: the scale follows the
// band's farthest value, so that beside a hot or no-data pixel the products of all others
// lie in the low levels (without levels 8 .. 12 one pixel of 9999 among 10^6 in [0, 1)
// cost the variance 2e-13 of itself).  Digits that are zero throughout a chunk are skipped:
// FP32 cubes have four to six that are not, 16-bit ones two to four.
//
//   k_band_range     largest and smallest value of every band (one pass)
//   k_syrk_digits    one CTA = one 64 x 64 band tile of one pixel range
// The fixed-point scale of a band comes from its range.  A band with a non-finite value
// or a spread too small for an FP32 scale sets hdr->fx_range, and the FP64 SIMT
// form (guarded by it) does the work.  So does a band of which more than lost_max values have
// bits below the scale's unit u, which is at most 2^-53 of the distance d of two of its
// values (2^-52 in slots of more than 2^26 pixels).  n such values, below 2^-30 of the farthest one,
// move a covariance by at most u sqrt(n) of sqrt(C_bb / (N - 1)), and C_aa (N - 1) >= d^2 / 2:
// 2^-52 sqrt(2 n) of sqrt(C_aa C_bb) for both factors.  lost_max = N / 4096 (16 at least) makes
// that sqrt(N / 2) 2^-57 at its worst (1.3e-15 at 16 values, 5e-15 at 10^6 pixels), and lets
// the few values near zero of a cube with no-data pixels pass.
//
// The covariance call, FP64 products -> these: 350 x 350 x 188 FP32 4.74 -> 0.68 ms,
// 610 x 340 x 103 2.88 -> 0.57, 512 x 512 x 224 BF16 13.7 -> 1.44, 10,000 x 50 0.189 -> 0.072.
// Its error against extended precision, over cubes of 28,000 to 10^6 pixels and 24 to 244
// bands, with and without a pixel of 300 to 65,535 among values of a lower range (relative to
// sqrt(C_aa C_bb), root mean square): FP64 products 1.3e-16 .. 1.3e-14, these 9e-17 .. 2.8e-16.
//
// Band B of the tiles is a constant band whose only digit is D_0, so that its products are
// the band sums S1.
//
// mma.sync rather than tcgen05: the sums of a level leave the accumulators after every
// 32 pixels, which in registers costs an FADD and an IMAD, while from TMEM they
// would all pass through tcgen05.ld behind a wait.
#include "common.cuh"

namespace gbpca {

namespace {

constexpr int kTile = 64;             // bands of a tile
constexpr int kPx = 32;               // pixels of a chunk
constexpr int kRow = kTile + 8;       // halves of a pixel's row: eight rows fall on all banks
constexpr int kThr = 256;             // 2 x 4 warps of 32 x 16 outputs

constexpr int kDigits = 7;
constexpr unsigned long long kBias = 0x80808080808080ull;   // digit = byte - 128
constexpr int kBlockHalves = kDigits * kPx * kRow;
constexpr size_t kBlockBytes = 2 * (size_t)kBlockHalves;

// A raw row: 64 values and one more 16-byte unit, for a start between units.
template <typename In>
constexpr int raw_row() { return kTile * (int)sizeof(In) + 16; }

struct FxSync {
  long long q0[2][kTile];    // fixed-point shift of every band of the two blocks
  int k[2][kTile];           // the exponent of its scale
  unsigned used[2][2];       // OR of the digits' bytes (without bias), low and high word, by chunk parity
  unsigned used_b[2][2];
  int bad;
};

// FP32 values as unsigned words of the same order; NaNs lie beyond the infinities.
__device__ __forceinline__ unsigned ordered(float x) {
  const unsigned u = __float_as_uint(x);
  return u ^ ((unsigned)((int)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float unordered(unsigned o) {
  return __uint_as_float(o & 0x80000000u ? o ^ 0x80000000u : ~o);
}

// ext[b] = max of ordered(y_b), ext[B + b] = max of ~ordered(y_b); ext[2 B + b], filled by
// k_syrk_digits, counts the values with lost bits.  All start at 0.
// Bound: the read of the cube.  Warp = pixel, lane = bands lane, lane + 32, ...
template <typename In>
__global__ void __launch_bounds__(256)
k_band_range(const In* __restrict__ cube, int64_t N, int B, unsigned* __restrict__ ext) {
  __shared__ unsigned red[2][kMaxB];
  for (int b = threadIdx.x; b < 2 * kMaxB; b += 256) (&red[0][0])[b] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * 8;
  unsigned hi[8], lo[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) hi[q] = lo[q] = 0u;
#pragma unroll 4
  for (int64_t n = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); n < N; n += step) {
    const In* row = cube + n * B;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int b = lane + 32 * q;
      if (b < B) {
        const unsigned o = ordered(to_f32<In>(row[b]));
        hi[q] = max(hi[q], o);
        lo[q] = max(lo[q], ~o);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int b = lane + 32 * q;
    if (b < B) {
      atomicMax(&red[0][b], hi[q]);
      atomicMax(&red[1][b], lo[q]);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < B; b += 256) {
    atomicMax(&ext[b], red[0][b]);
    atomicMax(&ext[B + b], red[1][b]);
  }
}

// The scale 2^k of a band about its shift s: |x| 2^k < 2^(top_bit + 1), and |y| 2^k < 2^61 (which
// only bands whose values all lie within 2^-7 of each other reach: their digits then end at
// D_2, so that nothing is left out).  False: no such scale (a non-finite value, or a spread
// too small).
__device__ __forceinline__ bool band_scale(unsigned max_o, unsigned min_o, float s, int top_bit,
                                           int* k) {
  const float top = unordered(max_o), bot = unordered(~min_o);
  *k = 0;
  if (!(fabsf(top) <= 3.4028234e38f) || !(fabsf(bot) <= 3.4028234e38f) ||
      !(fabsf(s) <= 3.4028234e38f))
    return false;
  const double d = fmax((double)top - (double)s, (double)s - (double)bot);
  const double a = fmax(fabs((double)top), fabs((double)bot));
  if (d == 0.0) {                                // every digit is zero
    if (a != 0.0) *k = min(60 - ilogb(a), 120);
    return true;
  }
  const int e = min(top_bit - ilogb(d), 60 - ilogb(a));
  if (e > 120) return false;
  *k = e;
  return true;
}

// y 2^k towards zero, |y| 2^k < 2^61: the significand from the word's top, shifted down.
// (cvt.s64.f32 runs on the FP64 pipe and held it for a third of the kernel's time.)
__device__ __forceinline__ long long to_fixed(float y, int k) {
  const unsigned u = __float_as_uint(y);
  const int down = min(189 - k - (int)((u >> 23) & 255u), 63);
  const unsigned top = ((u << 7) & 0x3fffffffu) | 0x40000000u;
  const long long q = (long long)(((unsigned long long)top << 32) >> down);
  return (int)u < 0 ? -q : q;
}

// Whether y has bits that to_fixed cuts off: its lowest set bit against the shift.
__device__ __forceinline__ bool loses_bits(float y, int k) {
  const unsigned u = __float_as_uint(y);
  const unsigned top = (u << 7) | 0x40000000u;
  return y != 0.f && 189 - k - (int)((u >> 23) & 255u) > 31 + __ffs((int)top);
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Two biased fixed-point values -> their digits as FP16 pairs, plane by plane.
// A byte u under the exponent byte 0x64 is the FP16 number 1024 + u.
__device__ __forceinline__ void store_digits(__half* dst, unsigned long long ua,
                                             unsigned long long ub) {
  const __half2 off = __floats2half2_rn(1152.f, 1152.f);   // 1024 + 128
  const unsigned a[2] = {(unsigned)ua, (unsigned)(ua >> 32)};
  const unsigned b[2] = {(unsigned)ub, (unsigned)(ub >> 32)};
#pragma unroll
  for (int d = 0; d < kDigits; ++d) {
    const int byte = kDigits - 1 - d;
    const unsigned p = __byte_perm(a[byte >> 2], b[byte >> 2],
                                   (unsigned)((byte & 3) | ((4 + (byte & 3)) << 8)));
    const unsigned w = (p & 0x00ff00ffu) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), off);
    *reinterpret_cast<__half2*>(dst + (size_t)d * kPx * kRow) = h;
  }
}

// Grid: x = partial slot (pixels N x / parts ..), y = tile of the upper block-triangle.
// Bound: issue (58% of the slots) and the latency of the shared-memory reads; the tensor
// pipe is active 26% of the time, the ALU (conversion, digits) 58%.  A chunk's rows come by
// asynchronous copies during the products of the one before, and 8 warps of 32 x 16 outputs
// (128 registers) hide more latency than 4 of 32 x 32 (237): 350 x 350 x 188, with loads
// into registers and 4 warps 1.02 ms, so 0.61 (levels 0 .. 7; 0.68 with all levels and the
// count of lost bits).
template <typename In>
__global__ void __launch_bounds__(kThr, 2)
k_syrk_digits(const In* __restrict__ cube, int64_t N, int B, int parts,
              unsigned* __restrict__ ext, unsigned lost_max, float* __restrict__ shift_out,
              double* __restrict__ s1_part, double* __restrict__ s2_part,
              DevHeader* __restrict__ hdr) {
  extern __shared__ __align__(128) unsigned char smem[];
  __half* blk = reinterpret_cast<__half*>(smem);                     // [2][kDigits][kPx][kRow]
  unsigned char* raw = smem + 2 * kBlockBytes;                  // [2][kPx][raw_row]
  FxSync* sy = reinterpret_cast<FxSync*>(raw + 2 * kPx * raw_row<In>());
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = blockIdx.x;
  int ti = 0, tj = blockIdx.y;                    // tile row by row
  const int nb = (B + kTile) / kTile;             // blocks that hold B + 1 bands
  while (tj >= nb - ti) { tj -= nb - ti; ++ti; }
  tj += ti;
  const bool diag = ti == tj;
  pdl_wait();

  // |x| < 2^54, or 2^53 where a slot has more than 2^26 pixels (up to 2^28 in 280 GB): the
  // sum of their squares, in units of 2^72, stays below 2^62
  const int top_bit = N / parts >= (int64_t)1 << 26 ? 52 : 53;
  // every CTA looks at every band, so that all take the same way
  int bad = 0;
  for (int b = tid; b < B; b += kThr) {
    const float s = to_f32<In>(cube[b]);
    int k;
    if (!band_scale(ext[b], ext[B + b], s, top_bit, &k)) bad = 1;
    // the shift as it is subtracted, without its own lost bits
    if (g == 0 && blockIdx.y == 0)
      shift_out[b] = ext[b] == ~ext[B + b] ? s : ldexpf((float)to_fixed(s, k), -k);
  }
  if (tid < 2 * kTile) {
    const int h = tid >> 6, p = tid & 63;         // block, position in it
    const int b = (h ? tj : ti) * kTile + (p >> 1) + 32 * (p & 1);
    int k = b == B ? top_bit + 1 : 0;      // the constant band: D_0 = 64 (32)
    long long q0 = 0;
    if (b < B) {
      const float s = to_f32<In>(cube[b]);
      band_scale(ext[b], ext[B + b], s, top_bit, &k);
      q0 = to_fixed(s, k);
    } else if (b == B) {
      q0 = -(1ll << (top_bit + 1));               // digits of 0 - q0
    }
    sy->q0[h][p] = q0;
    sy->k[h][p] = k;
    if (tid < 4) (&sy->used[0][0])[tid] = (&sy->used_b[0][0])[tid] = 0u;
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0 && g == 0 && blockIdx.y == 0) hdr->fx_range = 1;
    return;
  }

  const int64_t n0 = N * g / parts, n1 = N * (g + 1) / parts;
  const int m0 = (warp & 1) * 32, c0 = (warp >> 1) * 16;   // this warp's outputs
  unsigned long long hi[2][2][4], lo[2][2][4];    // signed sums, modulo 2^64
  unsigned long long hi_off = 0, lo_off = 0, ex_off = 0;   // what the magic numbers added
  // levels 8 .. 12, in units of 1: few chunks have them, so they stay in local memory
  // (volatile: the registers hold hi and lo)
  volatile unsigned long long ex[16];
  bool ex_used = false;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) hi[i][j][r] = lo[i][j][r] = ex[8 * i + 4 * j + r] = 0;

  // ldmatrix (transposed) addresses: A from [pixel][band] as 16 x 16, B as 16 x 16
  const uint32_t sA = (uint32_t)__cvta_generic_to_shared(blk) +
                      2u * (((lane & 7) + ((lane >> 4) & 1) * 8) * kRow + m0 + ((lane >> 3) & 1) * 8);
  const uint32_t sB = (uint32_t)__cvta_generic_to_shared(blk) + (diag ? 0u : (uint32_t)kBlockBytes) +
                      2u * (((lane & 7) + ((lane >> 3) & 1) * 8) * kRow + c0 + ((lane >> 4) & 1) * 8);

  const int nconv = diag ? 1 : 2;
  // the rows of a chunk, as the whole 16-byte units that hold them (the cube starts on one;
  // the last one may end beyond it)
  const int64_t cube_bytes = N * B * (int64_t)sizeof(In);
  auto fetch = [&](int64_t c) {
    constexpr int kUnits = raw_row<In>() / 16;
    for (int e = tid; e < nconv * kPx * kUnits; e += kThr) {
      const int h = e / (kPx * kUnits), p = e / kUnits % kPx, u = e % kUnits;
      const int b0 = (h ? tj : ti) * kTile, nbands = min(kTile, B - b0);
      if (c + p >= n1) continue;
      const int64_t at = ((c + p) * B + b0) * (int64_t)sizeof(In);
      const int64_t src = (at & ~(int64_t)15) + 16 * u;
      if (src >= at + nbands * (int)sizeof(In)) continue;
      const int bytes = cube_bytes - src < 16 ? (int)(cube_bytes - src) : 16;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(raw + (h * kPx + p) * raw_row<In>() + 16 * u)),
                   "l"(reinterpret_cast<const char*>(cube) + src), "r"(bytes)
                   : "memory");
    }
  };
  fetch(n0);
  // |ex| < 2^63: what is above its 40 low bits goes over to lo
  auto carry_ex = [&]() {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const unsigned long long e = ex[8 * i + 4 * j + r] - ex_off;
          lo[i][j][r] += (unsigned long long)((long long)e >> 40);
          ex[8 * i + 4 * j + r] = e & 0xffffffffffull;
        }
    ex_off = 0;
  };
  unsigned lost[2] = {0u, 0u};     // values with lost bits, bands lane and lane + 32 (diagonal tiles)
  int par = 0, since = 0;
  for (int64_t c = n0; c < n1; c += kPx, par ^= 1) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();               // the chunk has landed; the digits of the last one are read
    // conversion: warp = pixel, lane = bands lane and lane + 32 of the block
    for (int h = 0; h < nconv; ++h) {
      const int b0 = (h ? tj : ti) * kTile;
      const bool inA = b0 + lane < B, inB = b0 + lane + 32 < B;
      const int kA = sy->k[h][2 * lane], kB = sy->k[h][2 * lane + 1];
      const long long qA = sy->q0[h][2 * lane], qB = sy->q0[h][2 * lane + 1];
      unsigned long long used = 0;
#pragma unroll
      for (int u = 0; u < kPx / 8; ++u) {
        const int p = warp + 8 * u;
        unsigned long long ua = kBias, ub = kBias;
        if (c + p < n1) {
          const int skip = (int)((((c + p) * B + b0) * (int64_t)sizeof(In)) & 15);
          const In* row = reinterpret_cast<const In*>(raw + (h * kPx + p) * raw_row<In>() + skip) + lane;
          const float va = inA ? to_f32<In>(row[0]) : 0.f, vb = inB ? to_f32<In>(row[32]) : 0.f;
          if (diag) {
            lost[0] += loses_bits(va, kA);
            lost[1] += loses_bits(vb, kB);
          }
          ua += (unsigned long long)(to_fixed(va, kA) - qA);
          ub += (unsigned long long)(to_fixed(vb, kB) - qB);
        }
        used |= (ua ^ kBias) | (ub ^ kBias);
        store_digits(blk + h * kBlockHalves + p * kRow + 2 * lane, ua, ub);
      }
      const unsigned ul = __reduce_or_sync(kFull, (unsigned)used);
      const unsigned uh = __reduce_or_sync(kFull, (unsigned)(used >> 32));
      if (lane == 0) {
        unsigned* dst = h ? sy->used_b[par] : sy->used[par];
        atomicOr(&dst[0], ul);
        atomicOr(&dst[1], uh);
      }
    }
    __syncthreads();
    if (c + kPx < n1) fetch(c + kPx);   // beside the products
    auto digits = [](unsigned l, unsigned h) {   // how many digits, from the top, are not all zero
      return l ? kDigits - ((__ffs((int)l) - 1) >> 3) : (h ? 3 - ((__ffs((int)h) - 1) >> 3) : 0);
    };
    const int na = digits(sy->used[par][0], sy->used[par][1]);
    const int nbd = diag ? na : digits(sy->used_b[par][0], sy->used_b[par][1]);
    if (tid < 2) sy->used[par ^ 1][tid] = sy->used_b[par ^ 1][tid] = 0u;

    // one level: all pairs of digits, then the sums into the integers by add(i, j, r, bits)
    auto level = [&](int l, auto add) {
      const int ia = l - nbd + 1 > 0 ? l - nbd + 1 : 0, ib = l < na - 1 ? l : na - 1;
      if (ia > ib) return false;
      float acc[2][2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
#pragma unroll 1
      for (int i = ia; i <= ib; ++i) {
        const uint32_t pa = sA + (uint32_t)(i * kPx * kRow * 2);
        const uint32_t pb = sB + (uint32_t)((l - i) * kPx * kRow * 2);
#pragma unroll
        for (int ks = 0; ks < kPx / 16; ++ks) {
          uint32_t a0[4], a1[4], b0[4];
          const uint32_t o = (uint32_t)(ks * 16 * kRow * 2);
          ldsm4t(a0, pa + o);
          ldsm4t(a1, pa + o + 32);
          ldsm4t(b0, pb + o);
          mma16816(acc[0][0], a0, b0[0], b0[1]);
          mma16816(acc[0][1], a0, b0[2], b0[3]);
          mma16816(acc[1][0], a1, b0[0], b0[1]);
          mma16816(acc[1][1], a1, b0[2], b0[3]);
        }
      }
      // |sum| <= 2^22: as an integer, the bits of 1.5 * 2^23 + sum are a constant + sum
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r)
            add(i, j, r, (unsigned long long)__float_as_uint(__fadd_rn(acc[i][j][r], 12582912.f)));
      return true;
    };
    // levels 0 .. 3 in units of 2^72, 4 .. 7 in units of 2^40, 8 .. 12 in units of 1
#pragma unroll 1
    for (int l = 0; l < 4; ++l) {
      const unsigned w = 1u << (8 * (3 - l));
      if (level(l, [&](int i, int j, int r, unsigned long long b) { hi[i][j][r] += b * w; }))
        hi_off += 0x4B400000ull * w;
    }
#pragma unroll 1
    for (int l = 4; l < 8; ++l) {
      const unsigned w = 1u << (8 * (7 - l));
      if (level(l, [&](int i, int j, int r, unsigned long long b) { lo[i][j][r] += b * w; }))
        lo_off += 0x4B400000ull * w;
    }
#pragma unroll 1
    for (int l = 8; l < na + nbd - 1; ++l) {
      const int sh = 8 * (12 - l);
      level(l, [&](int i, int j, int r, unsigned long long b) {
        ex[8 * i + 4 * j + r] = ex[8 * i + 4 * j + r] + (b << sh);
      });
      ex_off += 0x4B400000ull << sh;
      ex_used = true;
    }
    ++since;
    if (ex_used && (since & 255) == 0) carry_ex();
    if (since == 1 << 16) {        // |lo| < 2^63: carried over into hi
      since = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            lo[i][j][r] -= lo_off;
            hi[i][j][r] += (unsigned long long)((long long)lo[i][j][r] >> 32);
            lo[i][j][r] &= 0xffffffffull;
          }
      lo_off = 0;
    }
  }

  // a band of one value has none: its deviations are zero
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int b = ti * kTile + lane + 32 * h;
    if (lost[h] != 0 && ext[b] != ~ext[B + b] && atomicAdd(&ext[2 * B + b], lost[h]) + lost[h] > lost_max)
      hdr->fx_range = 1;
  }

  if (ex_used) carry_ex();
  // pair sums, in units of 2^(-k_a - k_b); a sum with the constant band is S1
  const int s2_elems = B * (B + 1) / 2;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int pr = m0 + 16 * i + (lane >> 2) + 8 * (r >> 1);
        const int pc = c0 + 8 * j + 2 * (lane & 3) + (r & 1);
        const int br = ti * kTile + (pr >> 1) + 32 * (pr & 1);
        const int bc = tj * kTile + (pc >> 1) + 32 * (pc & 1);
        if (br > bc || bc > B || br >= B) continue;   // below the diagonal, padding, (B, B)
        const long long low = (long long)(lo[i][j][r] - lo_off);
        const long long top = (long long)(hi[i][j][r] - hi_off) + (low >> 32);
        // the magnitude of top 2^72 + low 2^40 + ex, rounded to FP64 twice at most
        unsigned long long t = (unsigned long long)top, m = (unsigned long long)low & 0xffffffffull;
        unsigned long long f = ex_used ? ex[8 * i + 4 * j + r] : 0ull;
        if (top < 0) {
          f = (0ull - f) & 0xffffffffffull;
          m = ((f != 0 ? ~m : 0ull - m)) & 0xffffffffull;
          t = (f | m) != 0 ? ~t : 0ull - t;
        }
        const double v = fma((double)t, 4294967296.0, fma((double)f, 0x1p-40, (double)m));
        const double x = ldexp(top < 0 ? -v : v, 40 - sy->k[0][pr] - sy->k[1][pc]);
        if (bc == B) s1_part[(size_t)g * B + br] = x;
        else s2_part[(size_t)g * s2_elems + packed_index(br, bc, B)] = x;
      }
}

template <typename In>
cudaError_t digits_typed(const In* cube, int64_t N, int B, float* shift, double* s1_part,
                         double* s2_part, int parts, unsigned* ext, DevHeader* hdr,
                         cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ext, 0, sizeof(unsigned) * 3 * B, st);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<int64_t>(4 * device_sms(), (N + 31) / 32);
  k_band_range<In><<<grid, 256, 0, st>>>(cube, N, B, ext);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t smem = 2 * kBlockBytes + 2 * kPx * raw_row<In>() + sizeof(FxSync);
  auto kern = k_syrk_digits<In>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int nb = (B + kTile) / kTile;
  const unsigned lost_max = (unsigned)std::max<int64_t>(16, N >> 12);
  return launch_after(kern, dim3(parts, nb * (nb + 1) / 2), kThr, smem, st, cube, N, B, parts, ext,
                      lost_max, shift, s1_part, s2_part, hdr);
}

}  // namespace

// Eight CTAs an SM, two at a time.  Few bands or pixels: as many slots as the FP64 sums
// have (one for 256 pixels, the workspace holds no more), less the start of a last round.
int syrk_digits_parts(int B, int num_sms, int max_parts) {
  const int nb = (B + kTile) / kTile, tiles = nb * (nb + 1) / 2;
  const int parts = std::max(1, 8 * num_sms / tiles);
  if (parts <= max_parts) return parts;
  const int rounds = max_parts * tiles / (2 * num_sms);
  return rounds > 0 ? std::max(1, rounds * 2 * num_sms / tiles) : max_parts;
}

cudaError_t launch_syrk_digits(const void* cube, pca_dtype dt, int64_t N, int B, float* shift,
                               double* s1_part, double* s2_part, int parts, unsigned* ext,
                               DevHeader* hdr, cudaStream_t st) {
  switch (dt) {
    case PCA_F32:
      return digits_typed((const float*)cube, N, B, shift, s1_part, s2_part, parts, ext, hdr, st);
    case PCA_BF16:
      return digits_typed((const __nv_bfloat16*)cube, N, B, shift, s1_part, s2_part, parts, ext,
                          hdr, st);
    case PCA_F16:
      return digits_typed((const __half*)cube, N, B, shift, s1_part, s2_part, parts, ext, hdr, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbpca
