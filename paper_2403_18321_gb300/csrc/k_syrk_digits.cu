// k_syrk_digits.cu -- partials of the P64 covariance call from exact integer
// products on the tensor cores.
//
// FP64 runs at about 1/67 of the FP32 rate on this GPU (1.9 FMAs per clock and
// SM), so that S2 = sum_n x_n x_n^T of 350 x 350 pixels of 188 bands costs
// 3.6 ms at its full rate.  Here x = y - s is held as a 56-bit fixed-point number per band
// and written as seven signed 8-bit digits D_0 .. D_6 (splitting into slices whose
// products are exact: Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).
// Digits are exact in FP16, a product of two is at most 2^14, and the sums over a chunk of
// 32 pixels of all pairs (i, j) of one level i + j stay below 2^22: exact in the FP32
// accumulators.  They are then added as 64-bit integers, and a partial is rounded once.
// Levels 0 .. 7 are formed; what is left out of a product is below 2^-57 of the largest
// |x_a| |x_b| (an FP64 sum rounds to 2^-53 of itself at every pixel).  Digits that
// are zero throughout a chunk are skipped: FP32 cubes have four to six that are not, 16-bit
// ones two to four.
//
//   k_band_range     largest and smallest value of every band (one pass)
//   k_syrk_digits    one CTA = one 64 x 64 band tile of one pixel range
// The fixed-point scale of a band comes from its range.  A band with a non-finite value
// or a spread too small for an FP32 scale sets hdr->fx_range, and the FP64 SIMT
// form (guarded by it) does the work.
//
// The covariance call, 350 x 350 x 188 FP32: 4.74 ms with the FP64 products, 1.02 ms with these.  The
// covariance's error against extended precision, over cubes of 28,000 to 57,000 pixels and
// 51 to 244 bands (relative to sqrt(C_aa C_bb), root mean square): FP64 products
// 8e-17 .. 1.1e-15, these 9e-17 .. 1.4e-16.
//
// Band B of the tiles is a constant band whose only digit is D_0 = 64, so that its
// products are the band sums S1.
//
// mma.sync rather than tcgen05: the sums of a level leave the accumulators after every
// 32 pixels, which in registers costs an FADD and an IMAD, while from TMEM they
// would all pass through tcgen05.ld behind a wait.
#include "common.cuh"

namespace gbpca {

namespace {

constexpr int kTile = 64;             // bands of a tile
constexpr int kPx = 32;               // pixels of a chunk
constexpr int kDigits = 7;
constexpr int kRow = kTile + 8;       // halves of a pixel's row: eight rows fall on all banks
constexpr int kThr = 128;             // 2 x 2 warps of 32 x 32 outputs
constexpr unsigned long long kBias = 0x80808080808080ull;   // digit = byte - 128
constexpr size_t kBlockBytes = (size_t)kDigits * kPx * kRow * 2;

struct FxSync {
  long long q0[2][kTile];    // fixed-point shift of every band of the two blocks
  float scale[2][kTile];     // its power-of-two scale
  int k[2][kTile];           // the exponent of the scale
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

// ext[b] = max of ordered(y_b), ext[B + b] = max of ~ordered(y_b); both start at 0.
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

// The scale 2^k of a band about its shift s: |x| 2^k < 2^54, |y| 2^k < 2^61.  False: no
// such scale (a non-finite value, or a spread too small).
__device__ __forceinline__ bool band_scale(unsigned max_o, unsigned min_o, float s, int* k) {
  const float top = unordered(max_o), bot = unordered(~min_o);
  *k = 0;
  if (!(fabsf(top) <= 3.4028234e38f) || !(fabsf(bot) <= 3.4028234e38f) ||
      !(fabsf(s) <= 3.4028234e38f))
    return false;
  const double d = fmax((double)top - (double)s, (double)s - (double)bot);
  const double a = fmax(fabs((double)top), fabs((double)bot));
  if (d == 0.0) return true;                     // every digit is zero whatever the scale (see q0)
  const int e = min(53 - ilogb(d), 60 - ilogb(a));
  if (e > 120) return false;
  *k = e;
  return true;
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Two biased fixed-point values -> their seven digits as FP16 pairs, plane by plane.
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
// Bound: the tensor cores and the ldmatrix reads that feed them (a warp's 32 x 32
// outputs: four reads of 512 bytes for eight MMAs).  Two CTAs share an SM, one's conversion
// beside the other's products.
template <typename In>
__global__ void __launch_bounds__(kThr, 2)
k_syrk_digits(const In* __restrict__ cube, int64_t N, int B, int parts,
              const unsigned* __restrict__ ext, float* __restrict__ shift_out,
              double* __restrict__ s1_part, double* __restrict__ s2_part,
              DevHeader* __restrict__ hdr) {
  extern __shared__ __align__(128) unsigned char smem[];
  __half* blk[2] = {reinterpret_cast<__half*>(smem), reinterpret_cast<__half*>(smem + kBlockBytes)};
  FxSync* sy = reinterpret_cast<FxSync*>(smem + 2 * kBlockBytes);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = blockIdx.x;
  int ti = 0, tj = blockIdx.y;                    // tile row by row
  const int nb = (B + kTile) / kTile;             // blocks that hold B + 1 bands
  while (tj >= nb - ti) { tj -= nb - ti; ++ti; }
  tj += ti;
  const bool diag = ti == tj;
  pdl_wait();

  // every CTA looks at every band, so that all take the same way
  int bad = 0;
  for (int b = tid; b < B; b += kThr) {
    const float s = to_f32<In>(cube[b]);
    int k;
    if (!band_scale(ext[b], ext[B + b], s, &k)) bad = 1;
    if (g == 0 && blockIdx.y == 0) shift_out[b] = s;
  }
  {
    const int h = tid >> 6, p = tid & 63;         // block, position in it
    const int b = (h ? tj : ti) * kTile + (p >> 1) + 32 * (p & 1);
    int k = b == B ? 54 : 0;                      // the constant band: 64 * 2^48
    float sc = 0.f;
    long long q0 = 0;
    if (b < B) {
      const float s = to_f32<In>(cube[b]);
      band_scale(ext[b], ext[B + b], s, &k);
      sc = ext[b] == ~ext[B + b] ? 0.f : scalbnf(1.f, k);
      q0 = __float2ll_rn(s * sc);
    } else if (b == B) {
      q0 = -(64ll << 48);                         // digits of 0 - q0
    }
    sy->scale[h][p] = sc;
    sy->q0[h][p] = q0;
    sy->k[h][p] = k;
    if (tid < 4) (&sy->used[0][0])[tid] = (&sy->used_b[0][0])[tid] = 0u;
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0 && g == 0 && blockIdx.y == 0) hdr->fx_range = 1;
    return;
  }

  const int64_t n0 = N * g / parts, n1 = N * (g + 1) / parts;
  const int m0 = (warp & 1) * 32, c0 = (warp >> 1) * 32;   // this warp's outputs
  long long hi[2][4][4], lo[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) hi[i][j][r] = lo[i][j][r] = 0;

  // ldmatrix (transposed) addresses: A from [pixel][band] as 16 x 16, B as 16 x 16
  const uint32_t sA = (uint32_t)__cvta_generic_to_shared(blk[0]) +
                      2u * (((lane & 7) + ((lane >> 4) & 1) * 8) * kRow + m0 + ((lane >> 3) & 1) * 8);
  const uint32_t sB = (uint32_t)__cvta_generic_to_shared(blk[diag ? 0 : 1]) +
                      2u * (((lane & 7) + ((lane >> 3) & 1) * 8) * kRow + c0 + ((lane >> 4) & 1) * 8);

  const int nconv = diag ? 1 : 2;
  int par = 0, since = 0;
  for (int64_t c = n0; c < n1; c += kPx, par ^= 1) {
    // conversion: warp = pixel, lane = bands lane and lane + 32 of the block
    for (int h = 0; h < nconv; ++h) {
      const int b = (h ? tj : ti) * kTile + lane;
      const bool inA = b < B, inB = b + 32 < B;
      const float scA = sy->scale[h][2 * lane], scB = sy->scale[h][2 * lane + 1];
      const long long qA = sy->q0[h][2 * lane], qB = sy->q0[h][2 * lane + 1];
      float va[kPx / 4], vb[kPx / 4];
#pragma unroll
      for (int u = 0; u < kPx / 4; ++u) {
        const int64_t n = c + warp + 4 * u;
        const In* row = cube + (n < n1 ? n : n0) * B + b;
        va[u] = inA ? to_f32<In>(row[0]) : 0.f;
        vb[u] = inB ? to_f32<In>(row[32]) : 0.f;
      }
      unsigned long long used = 0;
#pragma unroll
      for (int u = 0; u < kPx / 4; ++u) {
        const int p = warp + 4 * u;
        unsigned long long ua = kBias, ub = kBias;
        if (c + p < n1) {
          ua += (unsigned long long)(__float2ll_rn(va[u] * scA) - qA);
          ub += (unsigned long long)(__float2ll_rn(vb[u] * scB) - qB);
        }
        used |= (ua ^ kBias) | (ub ^ kBias);
        store_digits(blk[h] + (size_t)p * kRow + 2 * lane, ua, ub);
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
    auto digits = [](unsigned l, unsigned h) {   // how many digits, from the top, are not all zero
      return l ? kDigits - ((__ffs((int)l) - 1) >> 3) : (h ? 3 - ((__ffs((int)h) - 1) >> 3) : 0);
    };
    const int na = digits(sy->used[par][0], sy->used[par][1]);
    const int nbd = diag ? na : digits(sy->used_b[par][0], sy->used_b[par][1]);
    if (tid < 2) sy->used[par ^ 1][tid] = sy->used_b[par ^ 1][tid] = 0u;

    // one level: all pairs of digits, then the sums into the integers with weight w
    auto level = [&](int l, int w, long long (&tot)[2][4][4]) {
      const int ia = l - nbd + 1 > 0 ? l - nbd + 1 : 0, ib = l < na - 1 ? l : na - 1;
      if (ia > ib) return;
      float acc[2][4][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
#pragma unroll 1
      for (int i = ia; i <= ib; ++i) {
        const uint32_t pa = sA + (uint32_t)(i * kPx * kRow * 2);
        const uint32_t pb = sB + (uint32_t)((l - i) * kPx * kRow * 2);
#pragma unroll
        for (int ks = 0; ks < kPx / 16; ++ks) {
          uint32_t a0[4], a1[4], b0[4], b1[4];
          const uint32_t o = (uint32_t)(ks * 16 * kRow * 2);
          ldsm4t(a0, pa + o);
          ldsm4t(a1, pa + o + 32);
          ldsm4t(b0, pb + o);
          ldsm4t(b1, pb + o + 32);
          mma16816(acc[0][0], a0, b0[0], b0[1]);
          mma16816(acc[0][1], a0, b0[2], b0[3]);
          mma16816(acc[0][2], a0, b1[0], b1[1]);
          mma16816(acc[0][3], a0, b1[2], b1[3]);
          mma16816(acc[1][0], a1, b0[0], b0[1]);
          mma16816(acc[1][1], a1, b0[2], b0[3]);
          mma16816(acc[1][2], a1, b1[0], b1[1]);
          mma16816(acc[1][3], a1, b1[2], b1[3]);
        }
      }
      // |sum| <= 2^22: the low bits of 1.5 * 2^23 + sum are the integer
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r)
            tot[i][j][r] +=
                (long long)(__float_as_int(__fadd_rn(acc[i][j][r], 12582912.f)) - 0x4B400000) * w;
    };
    // levels 0 .. 3 in units of 2^72, levels 4 .. 7 in units of 2^40
#pragma unroll 1
    for (int l = 0; l < 4; ++l) level(l, 1 << (8 * (3 - l)), hi);
#pragma unroll 1
    for (int l = 4; l < 8; ++l) level(l, 1 << (8 * (7 - l)), lo);
    if (++since == 1 << 16) {      // |lo| < 2^62: carried over into hi
      since = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            hi[i][j][r] += lo[i][j][r] >> 32;
            lo[i][j][r] &= 0xffffffffll;
          }
    }
    __syncthreads();               // the digits are read; the next chunk may be written
  }

  // pair sums in units of 2^(40 - k_a - k_b); a sum with the constant band is S1
  const int s2_elems = B * (B + 1) / 2;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int pr = m0 + 16 * i + (lane >> 2) + 8 * (r >> 1);
        const int pc = c0 + 8 * j + 2 * (lane & 3) + (r & 1);
        const int br = ti * kTile + (pr >> 1) + 32 * (pr & 1);
        const int bc = tj * kTile + (pc >> 1) + 32 * (pc & 1);
        if (br > bc || bc > B || br >= B) continue;   // below the diagonal, padding, (B, B)
        const long long top = hi[i][j][r] + (lo[i][j][r] >> 32);
        const double v = fma((double)top, 4294967296.0, (double)(lo[i][j][r] & 0xffffffffll));
        const double x = ldexp(v, 40 - sy->k[0][pr] - sy->k[1][pc]);
        if (bc == B) s1_part[(size_t)g * B + br] = x;
        else s2_part[(size_t)g * s2_elems + packed_index(br, bc, B)] = x;
      }
}

template <typename In>
cudaError_t digits_typed(const In* cube, int64_t N, int B, float* shift, double* s1_part,
                         double* s2_part, int parts, unsigned* ext, DevHeader* hdr,
                         cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ext, 0, sizeof(unsigned) * 2 * B, st);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<int64_t>(4 * device_sms(), (N + 31) / 32);
  k_band_range<In><<<grid, 256, 0, st>>>(cube, N, B, ext);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t smem = 2 * kBlockBytes + sizeof(FxSync);
  auto kern = k_syrk_digits<In>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int nb = (B + kTile) / kTile;
  return launch_after(kern, dim3(parts, nb * (nb + 1) / 2), kThr, smem, st, cube, N, B, parts, ext,
                      shift, s1_part, s2_part, hdr);
}

}  // namespace

// Eight CTAs an SM (two at a time), a chunk of pixels at least.
int syrk_digits_parts(int64_t N, int B, int num_sms) {
  const int nb = (B + kTile) / kTile, tiles = nb * (nb + 1) / 2;
  const int64_t cap = std::max(1, 8 * num_sms / tiles);
  return (int)std::min<int64_t>(cap, std::max<int64_t>(1, (N + kPx - 1) / kPx));
}

cudaError_t launch_syrk_digits(const void* cube, pca_dtype dt, int64_t N, int B, float* shift,
                               double* s1_part, double* s2_part, int parts, unsigned* ext,
                               DevHeader* hdr, cudaStream_t st) {
  switch (dt) {
    case PCA_F32:
      return digits_typed((const float*)cube, N, B, shift, s1_part, s2_part, parts, ext, hdr, st);
    case PCA_BF16:
      return digits_typed((const __nv_bfloat16*)cube, N, B, shift, s1_part, s2_part, parts, ext, hdr,
                          st);
    case PCA_F16:
      return digits_typed((const __half*)cube, N, B, shift, s1_part, s2_part, parts, ext, hdr, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbpca
