// k_cov.cu -- band means and covariance (Algorithm 1 stages 2-3; Sec. 4.2
// stages 2 and 3) on SIMT cores, and the reduction of per-CTA partials.
//
// One pass over the cube.  Every partial slot g (a contiguous pixel range)
// accumulates, for x = y - s with s the first pixel of the cube (a per-band
// shift; any fixed s works),
//     S1_g = sum_n x_n            (FP64, per band)
//     S2_g = sum_n x_n x_n^T      (upper triangle, FP32 for P32 / FP64 for P64)
// and the finalisation turns the totals into the paper's quantities:
//     mu = s + S1/N,  C = (S2 - S1 S1^T / N) / (N - 1),
// which equals X^T X/(N-1) with X = Y - 1 mu^T exactly in real arithmetic.
// The shift keeps the summands centred near zero, so the correction term is
// of the order of one band variance (no catastrophic cancellation) and the
// cube is read once instead of twice (separate mean pass + covariance pass).
#include "common.cuh"

namespace gbpca {

namespace {

// Threads of a CTA at most; a slot's tiles take as many CTAs as they need, two
// or more of which share an SM, so that one's loads run beside the others'
// products.  FP64: the pipe is so slow that what counts is how often the CTAs
// of a slot repeat the conversion of its pixels.
template <typename Acc>
constexpr int max_threads() { return sizeof(Acc) == 8 ? 384 : 256; }
// Columns of a thread's tile (rows: TM = 8 in FP32, 4 in FP64): 8 x 4 rather than
// 8 x 8 gives a slot of 103 bands 6 warps instead of 3, and the SMs hold few slots.
template <typename Acc>
constexpr int tile_cols() { return 4; }
constexpr int kChunk = 32;  // pixels whose band sums are added in the accumulator's type before FP64
constexpr int kStage = 16;  // pixels staged in shared memory at a time
constexpr int kAhead = 4;   // raw stages: a stage's products take less time than its copy

template <typename In>
__device__ __forceinline__ float ld(const In* p) { return to_f32<In>(*p); }

// Asynchronous copy of a 16-byte unit, of which `bytes` exist.
__device__ __forceinline__ void copy_unit(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
               : "memory");
}
// 16-byte units of a raw stage: kStage pixels, one more for a start between units.
__host__ __device__ inline int raw_units(int B, int el) { return (kStage * B * el + 15) / 16 + 1; }

// One CTA: pixels [n0, n1) of the cube into partial slot g (S1 when grp is
// 0), band-tile group grp.  Each thread owns one TM x TN tile of the upper
// block-triangle of S2 and adds its products pixel by pixel.
//
// Bound: the FP32 (FP64) pipe and issue while an SM works, and the last round of CTAs
// (610 x 340 x 103 FP32: 320 CTAs, 304 resident, an SM active 54% of the launch; 2.6 of 4
// instructions issued a cycle).  The pixels come in by asynchronous copies, up to three
// stages ahead, and are centred once per CTA into a second buffer (loads into
// registers, a few at a time between two barriers, took 14 of every 15 us).
// Tile t holds TM / U units of U consecutive bands (16 bytes), unit u being
// bands u Bu + U t and on, so that the lanes of a warp -- consecutive tiles of
// a row of tiles -- read consecutive 16-byte words of a pixel.
// A slot's 8 x 4 tiles give the few slots an SM holds (two or three) enough warps.
// 610 x 340 x 103 FP32, the whole covariance call: 391 us with 8 x 8 tiles of
// consecutive bands and synchronous loads, 231 us with the copies, 213 us with
// the smaller tiles.  350 x 350 x 188 in FP64 (two CTAs an SM): the fit 6.38 -> 6.15
// ms, of which the FP64 pipe at its full rate takes 3.6.
template <typename In, typename Acc, int TM>
__device__ __forceinline__ void syrk_simt_cta(const In* __restrict__ cube, int B, int64_t n0,
                                              int64_t n1, int g, int grp,
                                              float* __restrict__ shift_out,
                                              double* __restrict__ s1_part,
                                              Acc* __restrict__ s2_part,
                                              int* __restrict__ escale, unsigned char* smem_raw) {
  constexpr int U = 16 / (int)sizeof(Acc), NU = TM / U;   // bands per unit, units per row tile
  constexpr int TN = tile_cols<Acc>(), NC = TN / U, HV = NU / NC;   // column units; column parts
  struct __align__(16) Unit { Acc v[U]; };
  const int Bt = (B + TM - 1) / TM, ntiles = HV * Bt * (Bt + 1) / 2;
  const int s2_elems = B * (B + 1) / 2;
  const int Bpad = Bt * TM, Bu = Bt * U;                  // unit u of tile t: bands u Bu + U t ..
  Acc* xs = reinterpret_cast<Acc*>(smem_raw);                   // [kStage][Bpad]
  float* sh = reinterpret_cast<float*>(xs + kStage * Bpad);     // [Bpad] shift
  float4* raw = reinterpret_cast<float4*>(sh + ((Bpad + 3) & ~3));   // [kAhead][raw_units]
  const int ru = raw_units(B, (int)sizeof(In));
  const int tid = threadIdx.x, nthr = blockDim.x;

  for (int b = tid; b < Bpad; b += nthr) sh[b] = b < B ? ld(cube + b) : 0.f;
  if (g == 0 && grp == 0)
    for (int b = tid; b < B; b += nthr) {
      shift_out[b] = ld(cube + b);
      if (escale != nullptr) escale[b] = 0;
    }

  // tile of this thread: enumerate the upper block-triangle row by row, a row's
  // column parts one after the other
  const int t = grp * nthr + tid;
  int ti = -1, tj = -1, part = 0;
  if (t < ntiles) {
    int rem = t;
    for (int r = 0; r < Bt; ++r) {
      const int len = Bt - r;
      if (rem < HV * len) { ti = r; part = rem / len; tj = r + rem - part * len; break; }
      rem -= HV * len;
    }
  }
  Acc acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = Acc(0);
  double s1[2] = {0.0, 0.0};  // bands tid and tid + nthr (group 0 only; B <= 2 nthr)
  Acc cs[2] = {Acc(0), Acc(0)};
  // stage at pixel c: the whole 16-byte units that hold its values (the cube
  // starts on one; the last one may end beyond the cube)
  auto fetch = [&](int64_t c, int buf) {
    const int cp = (int)((n1 - c) < kStage ? (n1 - c) : kStage);
    const int64_t b0 = c * B * (int64_t)sizeof(In);
    const int skip = (int)(b0 & 15), bytes = skip + cp * B * (int)sizeof(In);
    const char* src = reinterpret_cast<const char*>(cube) + (b0 - skip);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(raw + buf * ru);
    for (int u = tid * 16; u < bytes; u += nthr * 16)
      copy_unit(dst + (uint32_t)u, src + u, bytes - u < 16 ? bytes - u : 16);
  };
  for (int k = 0; k < kAhead - 1; ++k) {
    if (n0 + k * kStage < n1) fetch(n0 + k * kStage, k);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }

  int buf = 0;
  for (int64_t c0 = n0; c0 < n1; c0 += kStage, buf = (buf + 1) % kAhead) {
    const int cp = (int)((n1 - c0) < kStage ? (n1 - c0) : kStage);
    asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 2) : "memory");
    __syncthreads();   // this stage has landed; the previous one's products are done
    if (c0 + (kAhead - 1) * kStage < n1) fetch(c0 + (kAhead - 1) * kStage, (buf + kAhead - 1) % kAhead);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const In* rp = reinterpret_cast<const In*>(raw + buf * ru) +
                   (int)((c0 * B * (int64_t)sizeof(In)) & 15) / (int)sizeof(In);
    const bool sum_done = ((c0 - n0) / kStage) % (kChunk / kStage) == kChunk / kStage - 1;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int b = tid + h * nthr;
      if (b >= Bpad) continue;
      const Acc sb = Acc(sh[b]);
      const int bb = b < B ? b : 0;
      Acc sum = cs[h];
      constexpr int kV = sizeof(Acc) == 8 ? 4 : 16;   // values in flight
#pragma unroll
      for (int p0 = 0; p0 < kStage; p0 += kV) {
        Acc v[kV];
#pragma unroll
        for (int p = 0; p < kV; ++p) v[p] = Acc(ld(rp + (p0 + p < cp ? p0 + p : 0) * B + bb)) - sb;
#pragma unroll
        for (int p = 0; p < kV; ++p) {
          const bool in = p0 + p < cp && b < B;
          xs[(p0 + p) * Bpad + b] = in ? v[p] : Acc(0);
          // S1 is one CTA's of the slot; in FP32, where the addition is cheap, the test
          // itself cost more (610 x 340 x 103: 236 us with it, 205 without)
          if (in && (sizeof(Acc) == 4 || grp == 0)) sum += v[p];
        }
      }
      cs[h] = sum;
      if (sum_done || c0 + kStage >= n1) {
        s1[h] += (double)sum;
        cs[h] = Acc(0);
      }
    }
    __syncthreads();
    if (ti >= 0) {
      const Acc* xa = xs + ti * U;
      const Acc* xb = xs + part * Bu + tj * U;
#pragma unroll 2
      for (int p = 0; p < cp; ++p) {
        Acc a[TM], bv[TN];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
          const Unit x = *reinterpret_cast<const Unit*>(xa + p * Bpad + u * Bu);
#pragma unroll
          for (int i = 0; i < U; ++i) a[u * U + i] = x.v[i];
        }
#pragma unroll
        for (int u = 0; u < NC; ++u) {
          const Unit y = *reinterpret_cast<const Unit*>(xb + p * Bpad + u * Bu);
#pragma unroll
          for (int i = 0; i < U; ++i) bv[u * U + i] = y.v[i];
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], bv[j], acc[i][j]);
      }
    }
  }
  __syncthreads();

  if (grp == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (tid + h * nthr < B) s1_part[(size_t)g * B + tid + h * nthr] = s1[h];
  }
  if (ti >= 0) {
    Acc* out = s2_part + (size_t)g * s2_elems;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int r = (i / U) * Bu + ti * U + i % U;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int c = (part + j / U) * Bu + tj * U + j % U;
        // the tiles of ti = tj form every pair twice
        if (r < B && c < B && (ti != tj || r <= c))
          out[r <= c ? packed_index(r, c, B) : packed_index(c, r, B)] = acc[i][j];
      }
    }
  }
}

// Grid: x walks the partial slots g (pixel ranges N g / parts ..), y = band-tile
// group.  The guarded form (the re-computation after an out-of-range
// tensor-core pass) runs on a small grid that returns at once when the flag is
// clear, instead of one CTA per slot.
template <typename In, typename Acc, int TM, bool kGuarded>
__global__ void __launch_bounds__(max_threads<Acc>(), 2)
k_syrk_simt(const In* __restrict__ cube, int64_t N, int B, int parts, float* __restrict__ shift_out,
            double* __restrict__ s1_part, Acc* __restrict__ s2_part,
            const int* __restrict__ guard, int* __restrict__ escale) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if constexpr (kGuarded) {
    pdl_begin();
    if (*(volatile const int*)guard == 0) return;
    for (int g = blockIdx.x; g < parts; g += gridDim.x) {
      syrk_simt_cta<In, Acc, TM>(cube, B, N * g / parts, N * (g + 1) / parts, g, blockIdx.y,
                                 shift_out, s1_part, s2_part, escale, smem_raw);
      __syncthreads();   // the CTA's shared staging is reused by the next slot
    }
  } else {   // one slot per CTA
    const int g = blockIdx.x;
    syrk_simt_cta<In, Acc, TM>(cube, B, N * g / parts, N * (g + 1) / parts, g, blockIdx.y,
                               shift_out, s1_part, s2_part, nullptr, smem_raw);
  }
}

// Grid: x walks the items (item x, x + gridDim.x, ...), y = band-tile group
// (groups beyond an item's tile skip it).  The guarded form runs on a small
// grid whose CTAs first look at every tile's range flag together and return
// when none is set, so that the common case costs a few microseconds, not one
// CTA per item.
template <typename In, typename Acc, int TM, bool kGuarded>
__global__ void __launch_bounds__(max_threads<Acc>(), 2)
k_syrk_simt_grouped(const TileDesc* __restrict__ T, const CovItem* __restrict__ items, int nitems,
                    int ntiles) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if constexpr (kGuarded) {
    int any = 0;
    for (int i = threadIdx.x; i < ntiles; i += blockDim.x)
      any |= *(volatile const int*)&T[i].hdr->cov_range;
    if (!__syncthreads_or(any)) return;
    for (int x = blockIdx.x; x < nitems; x += gridDim.x) {
      const CovItem it = items[x];
      const TileDesc& t = T[it.tile];
      const int B = t.B, Bt = (B + TM - 1) / TM;
      if ((int)(blockIdx.y * blockDim.x) >= TM / tile_cols<Acc>() * Bt * (Bt + 1) / 2) continue;
      if (*(volatile const int*)&t.hdr->cov_range == 0) continue;
      syrk_simt_cta<In, Acc, TM>(static_cast<const In*>(t.cube), B, it.p0, it.p1, it.slot,
                                 blockIdx.y, t.shift, t.s1p, static_cast<Acc*>(t.s2p), t.escale,
                                 smem_raw);
      __syncthreads();   // the CTA's shared staging is reused by the next item
    }
  } else {   // one item per CTA
    const CovItem it = items[blockIdx.x];
    const TileDesc& t = T[it.tile];
    const int B = t.B, Bt = (B + TM - 1) / TM;
    if ((int)(blockIdx.y * blockDim.x) >= TM / tile_cols<Acc>() * Bt * (Bt + 1) / 2) return;
    syrk_simt_cta<In, Acc, TM>(static_cast<const In*>(t.cube), B, it.p0, it.p1, it.slot,
                               blockIdx.y, t.shift, t.s1p, static_cast<Acc*>(t.s2p), nullptr,
                               smem_raw);
  }
}

// Threads and CTAs of a slot.  Every scheduler of an SM has a quarter of its pipe, so a
// CTA takes ceil(warps / 4) times a tile's products of a pixel, plus the conversion of
// the pixel that each CTA of a slot repeats, and an SM the sum over its CTAs.  In pipe slots:
// FP64 16 products and 2 operations a value, FP32 about 44 (with the reads) and 6.  Few
// slots (a short cube) leave SMs idle with the fewest CTAs; too small ones repeat the conversion.
// FP32 keeps the fewest wherever they fill the chip twice over (its reads hide behind the
// other CTA's products).  At least 64 threads, and half the bands (a thread sums two).
// FP64 covariance of 4,090 x 234: 14 CTAs a slot 464 us, 7 (chosen) 329; against the
// fewest CTAs 10,000 x 128 287 -> 245 us, 40,000 x 100 780 -> 626, 90,000 x 100 1283 ->
// 1175, 122,500 x 188 unchanged (three CTAs a slot either way).
template <typename Acc>
void syrk_shape(int B, int TM, int slots, int* threads, int* groups) {
  constexpr bool kDouble = sizeof(Acc) == 8;
  constexpr int kProducts = kDouble ? 16 : 44, kConvert = kDouble ? 2 : 6;
  const int Bt = (B + TM - 1) / TM, n = TM / tile_cols<Acc>() * Bt * (Bt + 1) / 2;
  const int least = std::max(64, (Bt * TM / 2 + 31) & ~31), sms = device_sms();
  const int fewest = (n + max_threads<Acc>() - 1) / max_threads<Acc>();
  auto width = [&](int g) { return ((n + g - 1) / g + 31) & ~31; };
  int64_t best = INT64_MAX;
  for (int g = fewest; g == fewest || g <= n / least; ++g) {
    const int64_t ctas = ((int64_t)slots * g + sms - 1) / sms;
    const int64_t cost = ctas * ((width(g) + 127) / 128 * kProducts * 128 + kConvert * Bt * TM);
    if (cost < best) { best = cost; *groups = g; *threads = width(g); }
    if (!kDouble && slots * fewest >= 2 * sms) break;
  }
}

template <typename In>
cudaError_t syrk_simt_typed(const In* cube, int64_t N, int B, bool fp64, float* shift,
                            double* s1_part, void* s2_part, int partials, cudaStream_t st,
                            const int* guard, int* escale) {
  const int gx = guard != nullptr ? std::min(partials, 4 * device_sms()) : partials;
  if (fp64) {
    constexpr int TM = 4;
    const int Bt = (B + TM - 1) / TM;
    int threads, groups;
    syrk_shape<double>(B, TM, partials, &threads, &groups);
    const size_t smem = (size_t)kStage * Bt * TM * sizeof(double) + Bt * TM * sizeof(float) +
                        16 + kAhead * sizeof(float4) * (size_t)raw_units(Bt * TM, (int)sizeof(In));
    auto kern = guard != nullptr ? k_syrk_simt<In, double, TM, true> : k_syrk_simt<In, double, TM, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (guard != nullptr)
      return launch_after(kern, dim3(gx, groups), threads, smem, st, cube, N, B, partials, shift, s1_part,
                          (double*)s2_part, guard, escale);
    kern<<<dim3(gx, groups), threads, smem, st>>>(cube, N, B, partials, shift, s1_part,
                                                       (double*)s2_part, guard, escale);
  } else {
    constexpr int TM = 8;
    const int Bt = (B + TM - 1) / TM;
    int threads, groups;
    syrk_shape<float>(B, TM, partials, &threads, &groups);
    const size_t smem = (size_t)kStage * Bt * TM * sizeof(float) + Bt * TM * sizeof(float) +
                        16 + kAhead * sizeof(float4) * (size_t)raw_units(Bt * TM, (int)sizeof(In));
    auto kern = guard != nullptr ? k_syrk_simt<In, float, TM, true> : k_syrk_simt<In, float, TM, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (guard != nullptr)
      return launch_after(kern, dim3(gx, groups), threads, smem, st, cube, N, B, partials, shift, s1_part,
                          (float*)s2_part, guard, escale);
    kern<<<dim3(gx, groups), threads, smem, st>>>(cube, N, B, partials, shift, s1_part,
                                                       (float*)s2_part, guard, escale);
  }
  return cudaGetLastError();
}

template <typename In>
cudaError_t syrk_simt_grouped_typed(const TileDesc* T, const CovItem* items, int nitems, int maxB,
                                    int ntiles, bool fp64, bool guarded, cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  const int gx = guarded ? std::min(nitems, 4 * device_sms()) : nitems;
  if (fp64) {
    constexpr int TM = 4;
    const int Bt = (maxB + TM - 1) / TM;
    int threads, groups;
    syrk_shape<double>(maxB, TM, nitems, &threads, &groups);
    const size_t smem = (size_t)kStage * Bt * TM * sizeof(double) + Bt * TM * sizeof(float) +
                        16 + kAhead * sizeof(float4) * (size_t)raw_units(Bt * TM, (int)sizeof(In));
    auto kern = guarded ? k_syrk_simt_grouped<In, double, TM, true>
                        : k_syrk_simt_grouped<In, double, TM, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(gx, groups), threads, smem, st>>>(T, items, nitems, ntiles);
  } else {
    constexpr int TM = 8;
    const int Bt = (maxB + TM - 1) / TM;
    int threads, groups;
    syrk_shape<float>(maxB, TM, nitems, &threads, &groups);
    const size_t smem = (size_t)kStage * Bt * TM * sizeof(float) + Bt * TM * sizeof(float) +
                        16 + kAhead * sizeof(float4) * (size_t)raw_units(Bt * TM, (int)sizeof(In));
    auto kern = guarded ? k_syrk_simt_grouped<In, float, TM, true>
                        : k_syrk_simt_grouped<In, float, TM, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(gx, groups), threads, smem, st>>>(T, items, nitems, ntiles);
  }
  return cudaGetLastError();
}

// d[b] = (sum_g S1_g[b]) / N, one warp per band (FP64 adds spread over SMs).
__device__ __forceinline__ void s1_reduce_band(int b, const double* __restrict__ s1_part,
                                               int partials, int B, int64_t N,
                                               const float* __restrict__ shift,
                                               double* __restrict__ dvec, double* __restrict__ mu,
                                               float* __restrict__ mu_f,
                                               DevHeader* __restrict__ hdr) {
  const int lane = threadIdx.x;
  double s = 0.0;
  for (int g = lane; g < partials; g += 32) s += s1_part[(size_t)g * B + b];
  s = warp_sum(s);
  if (lane == 0) {
    const double d = s / (double)N;
    const double m = (double)shift[b] + d;
    dvec[b] = d;
    mu[b] = m;
    mu_f[b] = (float)m;
    if (!isfinite(m)) { atomicOr(&hdr->nonfinite, 1); set_status(hdr, PCA_ERR_NONFINITE); }
  }
}
__global__ void k_s1_reduce(const double* __restrict__ s1_part, int partials, int B, int64_t N,
                            const float* __restrict__ shift, double* __restrict__ dvec,
                            double* __restrict__ mu, float* __restrict__ mu_f,
                            DevHeader* __restrict__ hdr, const int* __restrict__ alt,
                            int alt_partials) {
  pdl_begin();
  if (alt != nullptr && *alt != 0) partials = alt_partials;
  s1_reduce_band(blockIdx.x, s1_part, partials, B, N, shift, dvec, mu, mu_f, hdr);
}
__global__ void k_s1_reduce_batched(const TileDesc* __restrict__ T) {
  const TileDesc& t = T[blockIdx.y];
  if ((int)blockIdx.x >= t.B) return;
  s1_reduce_band(blockIdx.x, t.s1p, t.parts, t.B, t.N, t.shift, t.dvec, t.mu, t.muf, t.hdr);
}

// C_ij = (S2_ij - N d_i d_j) / (N - 1), S2 summed over the partials.  One
// CTA per 32 consecutive packed entries: lane = entry (coalesced reads of
// every partial), warp w adds the partials w, w + 8, ...  FP32 partials are
// added as an unevaluated FP32 pair (hi, lo) with error-free TwoSum steps --
// FP64 arithmetic runs at a small fraction of the FP32 rate on this GPU --
// and the eight warp sums are added in FP64 in a fixed order.
constexpr int kFinWarps = 8;

template <typename Acc>
__device__ __forceinline__ void cov_finalize_block(int blk, const Acc* __restrict__ s2_part,
                                                   int partials, int s2_elems, int B, int64_t N,
                                                   const double* __restrict__ dvec,
                                                   double* __restrict__ C,
                                                   DevHeader* __restrict__ hdr,
                                                   const int* __restrict__ escale) {
  __shared__ double part[kFinWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t e = (int64_t)blk * 32 + lane;
  double sum = 0.0;
  if (e < s2_elems) {
    if constexpr (sizeof(Acc) == 4) {
      float hi = 0.f, lo = 0.f;
      auto add = [&](float v) {
        const float s = __fadd_rn(hi, v);          // TwoSum(hi, v)
        const float z = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(v, z)));
        hi = s;
      };
      // eight loads in flight, added in their order (one at a time, the chain of the
      // additions hid little of each load: the 256-tile batch 1.67 ms, 0.93 so)
      constexpr int kAhead8 = 8;
      int g = warp;
      for (; g + (kAhead8 - 1) * kFinWarps < partials; g += kAhead8 * kFinWarps) {
        float v[kAhead8];
#pragma unroll
        for (int u = 0; u < kAhead8; ++u)
          v[u] = __ldcs(reinterpret_cast<const float*>(s2_part) + (size_t)(g + u * kFinWarps) * s2_elems + e);
#pragma unroll
        for (int u = 0; u < kAhead8; ++u) add(v[u]);
      }
      for (; g < partials; g += kFinWarps) add((float)s2_part[(size_t)g * s2_elems + e]);
      sum = (double)hi + (double)lo;
    } else {
#pragma unroll 8
      for (int g = warp; g < partials; g += kFinWarps) sum += (double)s2_part[(size_t)g * s2_elems + e];
    }
  }
  part[warp][lane] = sum;
  __syncthreads();
  if (warp == 0 && e < s2_elems) {
    double S2 = 0.0;
#pragma unroll
    for (int w = 0; w < kFinWarps; ++w) S2 += part[w][lane];
    // (i, j) of packed entry e = j(j+1)/2 + i
    int j = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((int64_t)(j + 1) * (j + 2) / 2 <= e) ++j;
    while ((int64_t)j * (j + 1) / 2 > e) --j;
    const int i = (int)(e - (int64_t)j * (j + 1) / 2);
    if (escale != nullptr) S2 = ldexp(S2, -(escale[i] + escale[j]));  // exact power of two
    const double c = (S2 - (double)N * dvec[i] * dvec[j]) / (double)(N - 1);
    C[(size_t)i * B + j] = c;
    C[(size_t)j * B + i] = c;
    if (!isfinite(c)) { atomicOr(&hdr->nonfinite, 1); set_status(hdr, PCA_ERR_NONFINITE); }
  }
}
template <typename Acc>
__global__ void __launch_bounds__(kFinWarps * 32)
k_cov_finalize(const Acc* __restrict__ s2_part, int partials, int s2_elems, int B, int64_t N,
               const double* __restrict__ dvec, double* __restrict__ C,
               DevHeader* __restrict__ hdr, const int* __restrict__ escale,
               const int* __restrict__ alt, int alt_partials) {
  pdl_begin();
  if (alt != nullptr && *alt != 0) partials = alt_partials;
  cov_finalize_block<Acc>(blockIdx.x, s2_part, partials, s2_elems, B, N, dvec, C, hdr, escale);
}
template <typename Acc>
__global__ void __launch_bounds__(kFinWarps * 32)
k_cov_finalize_batched(const TileDesc* __restrict__ T, int escaled) {
  const TileDesc& t = T[blockIdx.y];
  const int s2_elems = t.B * (t.B + 1) / 2;
  if ((int)blockIdx.x * 32 >= s2_elems) return;
  cov_finalize_block<Acc>(blockIdx.x, static_cast<const Acc*>(t.s2p), t.parts, s2_elems, t.B, t.N,
                          t.dvec, t.C, t.hdr, escaled ? t.escale : nullptr);
}

}  // namespace

cudaError_t launch_syrk_simt(const void* cube, pca_dtype dt, int64_t N, int B, bool fp64,
                             float* shift, double* s1_part, void* s2_part, int partials,
                             cudaStream_t st, const int* guard, int* escale) {
  switch (dt) {
    case PCA_F32:
      return syrk_simt_typed((const float*)cube, N, B, fp64, shift, s1_part, s2_part, partials, st,
                             guard, escale);
    case PCA_BF16:
      return syrk_simt_typed((const __nv_bfloat16*)cube, N, B, fp64, shift, s1_part, s2_part,
                             partials, st, guard, escale);
    case PCA_F16:
      return syrk_simt_typed((const __half*)cube, N, B, fp64, shift, s1_part, s2_part, partials, st,
                             guard, escale);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cov_finalize(const float* shift, const double* s1_part, const void* s2_part,
                                bool fp64_partials, int partials, int64_t N, int B, double* mu,
                                double* C, float* mu_f, double* dvec, DevHeader* hdr,
                                cudaStream_t st, const int* escale, const int* alt,
                                int alt_partials) {
  const cudaError_t e = launch_after(k_s1_reduce, B, 32, 0, st, s1_part, partials, B, N, shift, dvec,
                                     mu, mu_f, hdr, alt, alt_partials);
  if (e != cudaSuccess) return e;
  const int s2_elems = B * (B + 1) / 2;
  const int grid = (s2_elems + 31) / 32;
  if (fp64_partials)
    return launch_after(k_cov_finalize<double>, grid, kFinWarps * 32, 0, st, (const double*)s2_part,
                        partials, s2_elems, B, N, dvec, C, hdr, escale, alt, alt_partials);
  return launch_after(k_cov_finalize<float>, grid, kFinWarps * 32, 0, st, (const float*)s2_part,
                      partials, s2_elems, B, N, dvec, C, hdr, escale, alt, alt_partials);
}

cudaError_t launch_syrk_simt_grouped(const TileDesc* T, const CovItem* items, int nitems,
                                     int maxB, int ntiles, pca_dtype dt, bool fp64, bool guarded,
                                     cudaStream_t st) {
  switch (dt) {
    case PCA_F32:
      return syrk_simt_grouped_typed<float>(T, items, nitems, maxB, ntiles, fp64, guarded, st);
    case PCA_BF16:
      return syrk_simt_grouped_typed<__nv_bfloat16>(T, items, nitems, maxB, ntiles, fp64, guarded,
                                                    st);
    case PCA_F16:
      return syrk_simt_grouped_typed<__half>(T, items, nitems, maxB, ntiles, fp64, guarded, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cov_finalize_batched(const TileDesc* T, int ntiles, int maxB, bool fp64,
                                        bool escaled, cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  k_s1_reduce_batched<<<dim3(maxB, ntiles), 32, 0, st>>>(T);
  const dim3 grid((maxB * (maxB + 1) / 2 + 31) / 32, ntiles);
  if (fp64)
    k_cov_finalize_batched<double><<<grid, kFinWarps * 32, 0, st>>>(T, escaled ? 1 : 0);
  else
    k_cov_finalize_batched<float><<<grid, kFinWarps * 32, 0, st>>>(T, escaled ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace gbpca
