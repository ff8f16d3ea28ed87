// k_jacobi_sm.cu -- the cyclic Jacobi eigen-solver (Sec. 2, Eqs. 2-10) for up to
// 128 bands, the matrix in the shared memory of one SM.
//
// The paper zeroes one element per host round trip (Sec. 4.2 stage 4) and
// notes that rotations on disjoint row/column pairs commute (Sec. 2, last
// paragraph).  Here every parallel step applies B'/2 disjoint rotations
// (B' = B rounded up to even, a zero padding index when B is odd), FP32.
//
// Ordering: odd-even.  Even steps rotate the position pairs (0,1),(2,3),...,
// odd steps (1,2),(3,4),...; after each rotation the two positions swap, so
// the rotation actually applied is G = R Pi with R = [[c, s], [-s, c]] the
// Eq. 1/Eq. 6 rotation and Pi the 2x2 swap, G = [[s, c], [c, -s]].  With the
// swap every index pair meets exactly once in B' steps (a valid cyclic
// sweep), and the pairs are always adjacent positions.  V receives the same G
// (V <- V G), so at the end eigenvalue diag(A)[j] belongs to column j of V.
//
// What bounds it is the chain of angles -- a pair's next angle needs the block
// beside its diagonal after this step's rotations, about 300 cycles with the
// barrier -- and, from about 80 bands on, the shared-memory traffic of the other
// blocks (12 wavefronts per 32 blocks).  An exchange between SMs on the chain
// costs more than the angle (a store that another CTA waits for takes about 450
// cycles, the pushes to 4 CTAs 170 more), so the matrix stays in one CTA:
//
//   * The matrix CTA: the first warps form the angles, one pair per thread, from
//     the blocks beside the diagonal; the others turn the rest of the step's
//     blocks, several per lane; one barrier per step.  The entries of row pair I and
//     column pair J >= I lie in four triangles, one per row and column parity, all
//     at word offset S(I) + J with S(I) the rows before, packed: the blocks that a
//     warp's lanes take one after the other then fall on consecutive words, in even
//     and odd steps and across the ends of rows.
//   * Vector CTAs, the rest of the cluster, hold the rows of V in registers (lane
//     l of a warp: positions [W l, W l + W)) and replay the (c, s) records, which
//     the matrix CTA sends them every kMsg steps.  Nothing waits for them within
//     kRing messages.
//
// Per step (FP32 form, whole solve over its steps), against k_jacobi_cluster.cu on
// 1 to 4 CTAs: 32 bands 0.34 us / 0.77, 64 bands 0.33 / 0.67, 100 bands 0.51 /
// 0.69, 128 bands 0.69 / 0.73; same bits.  Tried and slower: the matrix over several
// CTAs that form every angle themselves and exchange bands and edge rows every four
// steps (224 bands: 1.14 us against 0.82; the exchange takes 1.6 us), blocks one at a
// time (100 bands 0.58), 1024 threads (128 bands 0.75).  The matrix in registers, 8 x 4
// entries a lane, was slower up to about 120 bands (64 bands 0.46) and above 128 (188 bands
// 1.14) and a little faster at 128 (0.66): not worth a form of its own.
//
// Every mbarrier wait is bounded: a CTA that gives up stops waiting, and the
// sweep's stop test ends the solve with PCA_ERR_TIMEOUT.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "jacobi.cuh"

namespace cg = cooperative_groups;

namespace gbpca {

namespace {

constexpr int kMsg = 8;           // steps per record message (even)
constexpr int kRing = 4;          // messages in flight to the vector CTAs

struct ParamFields {
  const double* C;
  int B;
  float tol32;
  int sweeps_max;
  int relative_stop;
  int nV;                 // vector CTAs; one matrix CTA
  float* diag32;
  float* v32;
  DevHeader* hdr;
};
// An entry of a list: padded, not over-aligned (the host keeps lists in byte vectors).
struct Params : ParamFields {
  unsigned char pad[kJacobiParamsBytes - sizeof(ParamFields)];
};
static_assert(sizeof(Params) == kJacobiParamsBytes && alignof(Params) <= alignof(std::max_align_t));

struct Shared {
  uint64_t vfree[kRing];  // matrix CTA: its vector CTAs are done with a message
  uint64_t full[kRing];   // vector CTA: a message has arrived
  __align__(16) uint4 msg[kRing];   // vector CTA: header of a message (x: 1 = stop)
  // records of the current even / odd step as the chain reads them: (c, s, new
  // a_pp, new a_qq); the last two entries are the row rotation of the thread that
  // has row 0 and the column rotation of the one that has the last column
  __align__(16) float4 rec[2][kMaxB / 2 + 2];
  float zero[4];          // where those two threads find and leave the blocks' missing halves
  float dg[kMaxB];        // diagonal at the sweep boundary
  double wred[2][32];
  int wviol[32];
  int flag;
  int abort;
  double sum_o, sum_d;    // of the last stop test: squares above and on the diagonal
  int escale;             // the matrix is held scaled by 2^-escale
};

__device__ __forceinline__ float lds(uint32_t a) {
  float x;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ float2 lds2(uint32_t a) {
  float2 x;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x.x), "=f"(x.y) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 x;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(a) : "memory");
  return x;
}
__device__ __forceinline__ void sts(uint32_t a, float x) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}
__device__ __forceinline__ void sts2(uint32_t a, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void sts4(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z),
               "f"(v.w)
               : "memory");
}

// Where the record of pair J lies in a step's table of (c, s): in order, with
// the 16-byte units (two records) of every other group of eight swapped in
// pairs.  32 consecutive pairs (a block warp, 8 bytes a lane) and the H
// consecutive pairs of each lane of a V warp (16 bytes a load) are both read
// without bank conflicts.
__host__ __device__ inline int ridx(int J) { return ((((J >> 1) ^ ((J >> 4) & 1)) << 1) | (J & 1)); }
// A 16-byte store into a CTA of the cluster that completes its bytes on that
// CTA's mbarrier `bar` (both addresses in the receiver's window).
__device__ __forceinline__ void st_async(uint32_t a, float4 v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
               : "memory");
}
// Copy of a contiguous block into a CTA of the cluster (16-byte units), its
// bytes completing on that CTA's mbarrier.
__device__ __forceinline__ void bulk_s2c(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "r"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void remote_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait of one thread per CTA; the others wait for it at a barrier (a
// warp that polls takes issue slots from the warps that work: V warps polling
// on their own ran at half speed).
static __device__ __noinline__ void wait_cluster_slow(uint64_t* b, uint32_t parity, int* abort) {
  const unsigned long long t0 = gtimer();
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(b)), "r"(parity), "r"(1000000u)
        : "memory");
    if (ok) return;
    if (*(volatile int*)abort) return;
    if (gtimer() - t0 > kWaitNs) {
      atomicExch(abort, 1);
      return;
    }
  }
}
__device__ __forceinline__ void wait_cluster(uint64_t* b, uint32_t parity, int* abort) {
  if (!mbar_try_cluster(b, parity)) wait_cluster_slow(b, parity, abort);
}

__device__ __forceinline__ void bar_all() { asm volatile("bar.sync 0;" ::: "memory"); }

// Words from one triangle of the rows to the next: the largest of this width
// and the spare blocks (a constant, so that it folds into the addresses; half a
// row of banks off a multiple of 32, so that even and odd columns don't collide).
template <int W>
__host__ __device__ constexpr int tri_words() {
  static_assert(W == 2 || W == 4, "up to 128 bands");
  return W == 2 ? 592 : 2128;    // 32 * 33 / 2 = 528, 64 * 65 / 2 = 2080 and 33 spare
}

// Diagonal position x after an odd step (rec[1]) preceded by an even step
// (rec[0]): positions 0 and B'-1 sat out the odd step.
__device__ __forceinline__ float diag_after_odd(const float4 (*rec)[kMaxB / 2 + 2], int x, int Bp) {
  if (x == 0) return rec[0][0].z;
  if (x == Bp - 1) return rec[0][Bp / 2 - 1].w;
  return (x & 1) ? rec[1][(x - 1) >> 1].z : rec[1][(x - 2) >> 1].w;
}

// The parameters of this CTA's matrix, read in place (parameter space or global
// memory) at each use rather than held in registers.
__device__ __forceinline__ const Params& par(const Params& one, const Params* list) {
  return list != nullptr ? list[blockIdx.x / (1 + one.nV)] : one;
}

// A vector CTA: rows [V0, V1) of V, replaying the records of every message.
template <int W, int VR>
__device__ __forceinline__ void vector_cta(const Params& p, Shared& sh, const float2* ring, int q,
                                           int tid) {
  constexpr int H = W / 2, kRec = 32 * H;
  const int lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int Bp = round_even(p.B), nV = p.nV;
  const int V0 = (int)((long)Bp * q / nV), V1 = (int)((long)Bp * (q + 1) / nV);
  // this warp's rows: V0 + warp + nw k, k < nrow
  const int nrow = V0 + warp < V1 ? (V1 - V0 - warp + nw - 1) / nw : 0;
  float v[VR][W];
#pragma unroll
  for (int k = 0; k < VR; ++k)
#pragma unroll
    for (int c = 0; c < W; ++c) v[k][c] = (k < nrow && V0 + warp + nw * k == W * lane + c) ? 1.f : 0.f;
  auto load_g = [&](uint32_t slot, float2* g) {   // this lane's H records
    if constexpr (H == 1) {
      g[0] = lds2(slot + 8u * (uint32_t)ridx(lane));
    } else {
#pragma unroll
      for (int t = 0; t < H; t += 2) {
        const float4 x = lds4(slot + 8u * (uint32_t)ridx(H * lane + t));
        g[t] = make_float2(x.x, x.y);
        g[t + 1] = make_float2(x.z, x.w);
      }
    }
  };
  int step0 = 0;                           // position in the sweep
  for (int mm = 0;; ++mm) {
    const int s = mm % kRing;
    const int n = min(kMsg, Bp - step0);
    if (tid == 0) {
      mbar_expect_tx(&sh.full[s], 16u + (uint32_t)(n * kRec * 8));
      wait_cluster(&sh.full[s], (uint32_t)(mm / kRing) & 1u, &sh.abort);
    }
    bar_all();
    if (*(volatile int*)&sh.abort || *(volatile uint32_t*)&sh.msg[s].x) break;
    // Every lane turns all its positions: those past the matrix hold zeros, the
    // records past the pairs of an odd step are (0, 1), which leaves the last
    // position as it is, and lane 0 leaves position 0 with (0, -1).
    if (nrow > 0) {
      const uint32_t ra = su32(ring) + 8u * (uint32_t)(s * kMsg * kRec);
#pragma unroll 1
      for (int j = 0; j < n; j += 2) {
        float2 g[H];
        load_g(ra + 8u * (uint32_t)(j * kRec), g);
#pragma unroll
        for (int k = 0; k < VR; ++k) {
          if (k >= nrow) break;             // uniform over the warp
#pragma unroll
          for (int t = 0; t < H; ++t) {
            const float x = v[k][2 * t], y = v[k][2 * t + 1];
            v[k][2 * t] = fmaf(x, g[t].y, y * g[t].x);
            v[k][2 * t + 1] = fmaf(x, g[t].x, -y * g[t].y);
          }
        }
        load_g(ra + 8u * (uint32_t)((j + 1) * kRec), g);
        // the pair before this lane's first straddles this lane and the previous one
        float2 gp;
        gp.x = __shfl_up_sync(kFull, g[H - 1].x, 1);
        gp.y = __shfl_up_sync(kFull, g[H - 1].y, 1);
        if (lane == 0) gp = make_float2(0.f, -1.f);
#pragma unroll
        for (int k = 0; k < VR; ++k) {
          if (k >= nrow) break;
          const float xl = v[k][W - 1], y0 = v[k][0];
          float yn = __shfl_down_sync(kFull, y0, 1);           // next lane's first
          const float xp = __shfl_up_sync(kFull, xl, 1);       // previous lane's last
          if (lane == 31) yn = 0.f;
#pragma unroll
          for (int t = 0; t < H - 1; ++t) {
            const float x = v[k][2 * t + 1], y = v[k][2 * t + 2];
            v[k][2 * t + 1] = fmaf(x, g[t].y, y * g[t].x);
            v[k][2 * t + 2] = fmaf(x, g[t].x, -y * g[t].y);
          }
          v[k][W - 1] = fmaf(xl, g[H - 1].y, yn * g[H - 1].x);
          v[k][0] = fmaf(xp, gp.x, -y0 * gp.y);
        }
      }
    }
    __syncwarp();
    if (lane == 0) remote_arrive(mapa(su32(&sh.vfree[s]), 0));
    step0 += n;
    if (step0 >= Bp) step0 = 0;
  }
#pragma unroll
  for (int k = 0; k < VR; ++k) {
    if (k >= nrow) break;
#pragma unroll
    for (int c = 0; c < W; ++c) {
      const int pos = W * lane + c;
      if (pos < Bp) p.v32[(size_t)(V0 + warp + nw * k) * Bp + pos] = v[k][c];
    }
  }
}

// One matrix per cluster: `one` when list is null, else list[cluster index]
// (every entry of a list has the cluster shape and V width of `one`).  CTA 0 is
// the matrix CTA.  VR: rows of V per warp of a vector CTA (checked on the host).
// MI: pairs of blocks per lane and parity (checked on the host).  Dynamic shared memory:
// record ring, the four triangles.
template <int W, int MI, int VR, int kThr>
__global__ void __launch_bounds__(kThr, 1)
k_jacobi_sm(const __grid_constant__ Params one, const Params* __restrict__ list) {
  constexpr int H = W / 2, kRec = 32 * H;  // pairs per lane in a V row; records per step
  extern __shared__ __align__(16) float dyn[];
  __shared__ Shared sh;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
  const int nV = par(one, list).nV;
  const int B = par(one, list).B, Bp = B + (B & 1), P = Bp / 2;
  const double* C = par(one, list).C;
  float2* ring = reinterpret_cast<float2*>(dyn);       // [kRing][kMsg][kRec] (c, s)

  // ---- uniform early exit (every CTA reads the same header word)
  if (par(one, list).hdr->nonfinite) {
    const Params& p = par(one, list);
    if (rank == 0) {
      for (int i = tid; i < Bp; i += nthr) p.diag32[i] = 0.f;
      if (tid == 0) { p.hdr->sweeps = 0; p.hdr->steps = 0; p.hdr->tol_used = p.tol32; }
    }
    for (int e = tid + rank * nthr; e < Bp * Bp; e += (1 + nV) * nthr)
      p.v32[e] = (e / Bp == e % Bp) ? 1.f : 0.f;
    return;
  }
  if (tid == 0) {
    sh.flag = 0;
    sh.abort = 0;
    for (int k = 0; k < kRing; ++k) {
      mbar_init(&sh.vfree[k], nV * (nthr / 32));
      mbar_init(&sh.full[k], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  if (rank > 0) {
    cl.sync();   // every CTA's barriers are initialised before remote stores
    vector_cta<W, VR>(par(one, list), sh, ring, rank - 1, tid);
    if (*(volatile int*)&sh.abort && tid == 0) set_status(par(one, list).hdr, PCA_ERR_TIMEOUT);
  } else {
    // ================================================================ matrix CTA
    constexpr int kTri = tri_words<W>();
    float* rows = dyn + 2 * kRec * kRing * kMsg;               // [row parity][column parity][kTri]
    auto tri = [&](int I) { return I * P - I * (I - 1) / 2; };  // S(I) + I
    auto at = [&](int i, int j) {
      return ((i & 1) * 2 + (j & 1)) * kTri + tri(i >> 1) - (i >> 1) + (j >> 1);
    };

    // ---- the matrix is held scaled by 2^-E, with max_i |a_ii| in [2^(E-1), 2^E):
    //      squares and products of entries then stay inside the FP32 range whatever
    //      the covariance's scale (|a_ij| <= max a_ii for a covariance); the
    //      eigenvalues and the norm are scaled back on output, the rotations
    //      and eigenvectors do not depend on it
    {
      double m = 0.0;
      for (int i = tid; i < B; i += nthr) m = fmax(m, fabs(C[(size_t)i * B + i]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(kFull, m, o));
      if (lane == 0) sh.wred[0][warp] = m;
      __syncthreads();
      if (tid == 0) {
        double cm = 0.0;
        for (int w = 0; w < nthr / 32; ++w) cm = fmax(cm, sh.wred[0][w]);
        int E = 0;
        if (cm > 0.0 && isfinite(cm)) frexp(cm, &E);
        sh.escale = E;
      }
      __syncthreads();
    }
    const double dscale = ldexp(1.0, -sh.escale);
    auto a0 = [&](int i, int j) {
      return (i < B && j < B) ? (float)(C[(size_t)i * B + j] * dscale) : 0.f;
    };
    for (int i = warp; i < Bp; i += nthr / 32)
      for (int j = i + 1 + lane; j < Bp; j += 32) rows[at(i, j)] = a0(i, j);
    if (tid < 4) sh.zero[tid] = -0.f;
    // (0, 1) for pairs past the matrix, and records that reproduce the initial
    // diagonal as the state after a sweep
    for (int e = tid; e < kRec * kRing * kMsg; e += nthr) ring[e] = make_float2(0.f, 1.f);
    for (int J = tid; J < P; J += nthr) {
      sh.rec[0][J] = make_float4(1.f, 0.f, a0(2 * J, 2 * J), a0(2 * J + 1, 2 * J + 1));
      sh.rec[1][J] = make_float4(1.f, 0.f, a0(2 * J + 1, 2 * J + 1),
                                 J + 1 < P ? a0(2 * J + 2, 2 * J + 2) : 0.f);
    }
    if (tid < 2) {
      sh.rec[tid][kMaxB / 2] = make_float4(0.f, -1.f, 0.f, 0.f);
      sh.rec[tid][kMaxB / 2 + 1] = make_float4(0.f, 1.f, 0.f, 0.f);
    }

    // ---- work lists
    const int ncw = (P + 31) / 32;           // chain warps: one pair per thread
    const bool chain = warp < ncw;
    const int nl = nthr - 32 * ncw, lid = tid - 32 * ncw;   // block lanes
    // one register array for both roles.  Block lanes take their blocks two at a
    // time, (I, J) and (I + 1, J) with I even, J >= I + 3, which share the record of J
    // and one load of those of I and I + 1: reg[2 e MI + t] the address of the first
    // (even rows' even columns at its pairs for e = 0, odd rows' for e = 1), reg[(2 e
    // + 1) MI + t], by bytes: the records of I and J, the words from S(I) to S(I+1).
    // The blocks (I, I + 2), I even, are left over, one each for the last lanes.  A
    // lane without blocks in its warp's last round turns spare ones.
    constexpr int kRegs = 4 * MI > 16 ? 4 * MI : 16;
    uint32_t reg[kRegs];
    int rounds[2] = {0, 0};                  // of this warp
    uint32_t sa[2] = {0, 0}, sr = 0;         // the left-over block (0: none), as above
    uint32_t xa = 0, xb = 0;                 // odd steps: a row-0 or last-column block
    int xk = 0, xty = 0;                     // its pair; 1 row 0, 2 last column
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int np = P - e;
#pragma unroll
      for (int t = 0; t < MI; ++t) {
        if (chain) continue;
        uint32_t& la = reg[2 * e * MI + t];
        uint32_t& lr = reg[(2 * e + 1) * MI + t];
        la = su32(rows) + 4u * (uint32_t)(tri(P) + lane + e * 2 * kTri);
        lr = 1u << 16;
        int rem = lid + t * nl, I = 0;
        while (I < np && rem >= max(0, np - 3 - I)) { rem -= max(0, np - 3 - I); I += 2; }
        if (I < np) {
          const int J = I + 3 + rem;
          la = su32(rows) + 4u * (uint32_t)(tri(I) - I + J + e * 2 * kTri);
          lr = (uint32_t)ridx(I) | ((uint32_t)ridx(J) << 8) | ((uint32_t)(P - I - 1) << 16);
        }
        if (__any_sync(kFull, I < np)) rounds[e] = t + 1;
      }
      const int I = 2 * (nl - 1 - lid);
      if (!chain && I + 2 < np) {
        sa[e] = su32(rows) + 4u * (uint32_t)(tri(I) + 2 + e * 2 * kTri);
        sr = (uint32_t)ridx(I) | ((uint32_t)ridx(I + 2) << 8) | ((uint32_t)(P - I - 1) << 16);
      }
    }
    if (!chain) {
      // odd-step extras, from the last lanes on: row 0 against the odd pairs, and the
      // odd row pairs against the idle last column; the chain takes the two whose
      // result is the off-diagonal of a next pair
      const int nx = max(0, P - 2), x = nl - 33 - lid;   // (past the left-over blocks)
      if (x >= 0 && x < nx) {
        xk = x + 1;
        xty = 1;
        xa = su32(rows + at(0, 2 * xk + 1));
        xb = su32(rows + at(0, 2 * xk + 2));
      } else if (x >= 0 && x < 2 * nx) {
        xk = x - nx;
        xty = 2;
        xa = su32(rows + at(2 * xk + 1, Bp - 1));
        xb = su32(rows + at(2 * xk + 2, Bp - 1));
      }
    }
    // The chain thread's block beside the diagonal: reg[8 e + 0..3] its four entries,
    // + 4, 5 its two records, + 6 where the new record goes, + 7 that one's ring offset.
    // In odd steps two more threads take row 0 (a column rotation only) and the last
    // column (a row rotation only); the missing halves of their blocks are zeros and
    // the missing rotations constants, so that all run the same code.
    const bool xr = P >= 2 && tid == P - 2, xc = P >= 2 && tid == P - 1;
    if (chain) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int I = tid;
        const uint32_t z = su32(sh.zero);
        auto A = [&](int i, int j) { return su32(rows + at(i, j)); };
        uint32_t q0 = z, q1 = z + 4, q2 = z, q3 = z + 4;
        if (e == 1 && xr) {
          q2 = A(0, 1);
          q3 = A(0, 2);
        } else if (e == 1 && xc) {
          q0 = A(Bp - 3, Bp - 1);
          q1 = z + 8;
          q2 = A(Bp - 2, Bp - 1);
          q3 = z + 12;
        } else if (I < P - e - 1) {
          const int p = 2 * I + e;
          q0 = A(p, p + 2);
          q1 = A(p, p + 3);
          q2 = A(p + 1, p + 2);
          q3 = A(p + 1, p + 3);
        }
        const bool sr = e == 1 && xr, sc = e == 1 && xc;
        const int o = min(sr ? 0 : (sc ? P - 1 : I + e), P - 1);     // the pair of the next step
        reg[8 * e + 0] = q0;
        reg[8 * e + 1] = q1;
        reg[8 * e + 2] = q2;
        reg[8 * e + 3] = q3;
        reg[8 * e + 4] = su32(&sh.rec[e][sr ? kMaxB / 2 : (sc ? P - 2 : min(I, P - 1))]);
        reg[8 * e + 5] = su32(&sh.rec[e][sr ? 0 : (sc ? kMaxB / 2 + 1 : min(I + 1, P - 1))]);
        reg[8 * e + 6] = su32(&sh.rec[1 - e][o]);
        reg[8 * e + 7] = 8u * (uint32_t)ridx(o);
      }
    }
    float keep = 0.f;   // row 0's / the last column's thread: that position's diagonal value
    int sweep = 0, status = PCA_OK;
    int mm = 0;                    // messages; records in ring slot mm % kRing
    const float tol2 = par(one, list).tol32 * par(one, list).tol32;
    const uint32_t ring_a = su32(ring);
    constexpr uint32_t kSlotB = 8u * (uint32_t)kRec, kTriB = 4u * (uint32_t)kTri;
    // The records of message x (n steps) to the vector CTAs, with a header (1: stop
    // instead); one thread.
    auto send_records = [&](int x, int n, uint32_t stop) {
      fence_proxy_async();
      const uint32_t src = ring_a + kSlotB * (uint32_t)((x % kRing) * kMsg);
      for (int v = 1; v <= nV; ++v) {
        const uint32_t bar = mapa(su32(&sh.full[x % kRing]), v);
        st_async(mapa(su32(&sh.msg[x % kRing]), v), make_float4(__uint_as_float(stop), 0.f, 0.f, 0.f), bar);
        bulk_s2c(mapa(src, v), src, kSlotB * (uint32_t)n, bar);
      }
    };
    const bool sender = tid == nthr - 1;
    cl.sync();   // every CTA's barriers are initialised before remote stores

    for (;;) {
      // -------------- diagonal at the sweep boundary (after the last odd step)
      for (int x = tid; x < Bp; x += nthr) sh.dg[x] = diag_after_odd(sh.rec, x, Bp);
      bar_all();
      // -------------- stop test
      {
        float so2 = 0.f, sd = 0.f;
        int viol = 0;
        for (int i = warp; i < Bp; i += nthr / 32) {
          const float dii = sh.dg[i];
          if (lane == 0) sd = fmaf(dii, dii, sd);
          const float aii = fabsf(dii);
          for (int j = i + 1 + lane; j < Bp; j += 32) {
            const float a = rows[at(i, j)];
            so2 = fmaf(a, a, so2);
            viol |= (a * a > tol2 * aii * fabsf(sh.dg[j])) ? 1 : 0;
          }
        }
        so2 = warp_sum(so2);
        sd = warp_sum(sd);
        viol = __any_sync(kFull, viol);
        if (lane == 0) {
          sh.wred[0][warp] = (double)so2;
          sh.wred[1][warp] = (double)sd;
          sh.wviol[warp] = viol;
        }
        bar_all();
        if (warp == 0) {
          const bool has = lane < nthr / 32;
          const double o = warp_sum(has ? sh.wred[0][lane] : 0.0);
          const double d = warp_sum(has ? sh.wred[1][lane] : 0.0);
          const int v = __any_sync(kFull, has && sh.wviol[lane]);
          if (lane == 0) {
            // off <= tol ||A||_F on the squares, and by the roots themselves only
            // where the squares are too close to tell (FP64 roots are slow here)
            const double off2 = 2.0 * o, fro2 = 2.0 * o + d, tl = (double)par(one, list).tol32;
            const double lim = tl * tl * fro2;
            const bool conv = par(one, list).relative_stop ? !v
                              : off2 > 1.000001 * lim      ? false
                              : off2 < 0.999999 * lim      ? true
                                                           : sqrt(off2) <= tl * sqrt(fro2);
            int flag = 0;
            if (*(volatile int*)&sh.abort) flag = 3;
            else if (fro2 == 0.0 || conv) flag = 1;
            else if (sweep >= par(one, list).sweeps_max) flag = 2;
            sh.flag = flag;
            sh.sum_o = o;
            sh.sum_d = d;
          }
        }
        bar_all();
      }
      const int flag = sh.flag;
      if (flag) {
        status = flag == 1 ? PCA_OK : (flag == 2 ? PCA_ERR_NOCONV : PCA_ERR_TIMEOUT);
        break;
      }

      // -------------- the first (even) step's pairs
      if (tid < P) {
        float* x = rows + at(2 * tid, 2 * tid + 1);
        const float4 r = pair_record(sh.dg[2 * tid], sh.dg[2 * tid + 1], *x);
        *x = 0.f;
        ring[(mm % kRing) * kMsg * kRec + ridx(tid)] = make_float2(r.x, r.y);
        sh.rec[0][tid] = r;
      }
      bar_all();
      if (xr) keep = sh.rec[0][0].z;
      if (xc) keep = sh.rec[0][P - 1].w;

      for (int step0 = 0; step0 < Bp; step0 += kMsg, ++mm) {
        const int n = min(kMsg, Bp - step0);
        const uint32_t slot0 = ring_a + kSlotB * (uint32_t)((mm % kRing) * kMsg);
        const uint32_t slot1 = ring_a + kSlotB * (uint32_t)(((mm + 1) % kRing) * kMsg);
        if (chain) {
          auto chain_step = [&](auto E_, uint32_t dst, bool last) {
            constexpr int e = decltype(E_)::value;
            if (tid < P - e - 1 || (e == 1 && (xr || xc))) {
              const float4 gI = lds4(reg[8 * e + 4]), gJ = lds4(reg[8 * e + 5]);
              float m00 = lds(reg[8 * e]), m01 = lds(reg[8 * e + 1]);
              float m10 = lds(reg[8 * e + 2]), m11 = lds(reg[8 * e + 3]);
              const float app = (e == 1 && xr) ? keep : gI.w, aqq = (e == 1 && xc) ? keep : gJ.z;
              rot_block(make_float2(gI.x, gI.y), make_float2(gJ.x, gJ.y), m00, m01, m10, m11);
              const float4 r = pair_record(app, aqq, m10);
              sts(reg[8 * e], m00);
              sts(reg[8 * e + 1], m01);
              sts(reg[8 * e + 3], m11);
              sts(reg[8 * e + 2], last ? m10 : 0.f);   // the next step's rotation of this pair zeroes it
              if (!last) {
                sts4(reg[8 * e + 6], r);
                sts2(dst + reg[8 * e + 7], r.x, r.y);
                if (e == 1) keep = xr ? r.z : r.w;
              }
            }
            bar_all();
          };
          uint32_t dst = slot0 + kSlotB;
#pragma unroll 1
          for (int j = 0; j < n; j += 2) {
            chain_step(std::integral_constant<int, 0>{}, dst, false);
            dst = j + 2 < n ? dst + kSlotB : slot1;
            chain_step(std::integral_constant<int, 1>{}, dst, step0 + j + 2 == Bp);
            dst += kSlotB;
          }
        } else {
          // the records of the next message go into a slot its readers have left
          if (sender && mm + 1 >= kRing)
            wait_cluster(&sh.vfree[(mm + 1) % kRing], (uint32_t)((mm + 1) / kRing - 1) & 1u, &sh.abort);
          auto block_step = [&](auto E_, uint32_t rcb) {
            constexpr int e = decltype(E_)::value;
            // entries (p, 2J + e), (p, 2J + e + 1) from address a, those of row q from b
            constexpr uint32_t o0 = e == 0 ? 0u : kTriB, o1 = e == 0 ? kTriB : 4u;
            auto row_q = [&](uint32_t a, uint32_t d) { return e == 0 ? a + 2 * kTriB : a - 2 * kTriB + d; };
#pragma unroll
            for (int t = 0; t < MI; ++t) {
              if (t >= rounds[e]) break;     // uniform over the warp
              const uint32_t lr = reg[(2 * e + 1) * MI + t], d = 4u * __byte_perm(lr, 0, 0x4442);
              const uint32_t a0 = reg[2 * e * MI + t], b0 = row_q(a0, d);          // block (I, J)
              const uint32_t a1 = a0 + d, b1 = row_q(a1, d - 4u);                  // block (I + 1, J)
              const float4 gi = lds4(rcb + 8u * __byte_perm(lr, 0, 0x4440));
              const float2 gj = lds2(rcb + 8u * __byte_perm(lr, 0, 0x4441));
              float m[2][4] = {{lds(a0 + o0), lds(a0 + o1), lds(b0 + o0), lds(b0 + o1)},
                               {lds(a1 + o0), lds(a1 + o1), lds(b1 + o0), lds(b1 + o1)}};
              rot_block(make_float2(gi.x, gi.y), gj, m[0][0], m[0][1], m[0][2], m[0][3]);
              rot_block(make_float2(gi.z, gi.w), gj, m[1][0], m[1][1], m[1][2], m[1][3]);
              sts(a0 + o0, m[0][0]);
              sts(a0 + o1, m[0][1]);
              sts(b0 + o0, m[0][2]);
              sts(b0 + o1, m[0][3]);
              sts(a1 + o0, m[1][0]);
              sts(a1 + o1, m[1][1]);
              sts(b1 + o0, m[1][2]);
              sts(b1 + o1, m[1][3]);
            }
            if (sa[e] != 0) {
              const uint32_t a = sa[e], b = row_q(a, 4u * __byte_perm(sr, 0, 0x4442));
              const float2 gi = lds2(rcb + 8u * __byte_perm(sr, 0, 0x4440));
              const float2 gj = lds2(rcb + 8u * __byte_perm(sr, 0, 0x4441));
              float m00 = lds(a + o0), m01 = lds(a + o1), m10 = lds(b + o0), m11 = lds(b + o1);
              rot_block(gi, gj, m00, m01, m10, m11);
              sts(a + o0, m00);
              sts(a + o1, m01);
              sts(b + o0, m10);
              sts(b + o1, m11);
            }
            if (e && xty) {
              const float2 gg = lds2(rcb + 8u * (uint32_t)ridx(xk));
              const float x = lds(xa), y = lds(xb);
              if (xty == 1) {              // (0, p), (0, q) against a column pair
                sts(xa, fmaf(x, gg.y, y * gg.x));
                sts(xb, fmaf(x, gg.x, -y * gg.y));
              } else {                     // (p, L), (q, L) against a row pair
                sts(xa, fmaf(gg.y, x, gg.x * y));
                sts(xb, fmaf(gg.x, x, -gg.y * y));
              }
            }
            bar_all();
          };
          uint32_t rcb = slot0;
#pragma unroll 1
          for (int j = 0; j < n; j += 2) {
            block_step(std::integral_constant<int, 0>{}, rcb);
            block_step(std::integral_constant<int, 1>{}, rcb + kSlotB);
            rcb += 2 * kSlotB;
          }
          if (sender) send_records(mm, n, 0u);
        }
      }
      ++sweep;
    }

    {
      const Params& p = par(one, list);
      for (int x = tid; x < Bp; x += nthr)
        p.diag32[x] = ldexpf(diag_after_odd(sh.rec, x, Bp), sh.escale);
      if (tid == 0) {
        const double off = sqrt(2.0 * sh.sum_o), fro = sqrt(2.0 * sh.sum_o + sh.sum_d);
        p.hdr->sweeps = sweep;
        p.hdr->steps = sweep * Bp;
        p.hdr->tol_used = p.tol32;
        p.hdr->off_rel = fro == 0.0 ? 0.0 : off / fro;
        p.hdr->fro = ldexp(fro, sh.escale);
        if (status != PCA_OK) set_status(p.hdr, status);
      }
    }
    // the vector CTAs stop: a message of the expected size, marked
    if (sender) send_records(mm, min(kMsg, Bp), 1u);
  }
  if (*(volatile int*)&sh.abort) {
    // an abandoned wait may leave stores of other CTAs in flight: give them
    // time to land before any CTA of the cluster leaves
    const unsigned long long t0 = gtimer();
    while (gtimer() - t0 < 100000ull) {
    }
  }
  cl.sync();  // no CTA leaves while others may still write its shared memory
}

// Pairs of blocks per lane (MI): 225 of 64 bands on 512 - 32 lanes, 961 of 128 on
// 768 - 64; the 31 left-over blocks and 124 odd-step extras fit beside them.
constexpr int kThreads2 = 512, kThreads4 = 768;

size_t sm_smem(int w) {
  return sizeof(float) * (2 * 32 * (size_t)(w / 2) * kRing * kMsg +
                          4 * (size_t)(w == 2 ? tri_words<2>() : tri_words<4>()));
}

}  // namespace

bool jacobi_sm_supported(int B) { return round_even(B) <= 128; }
// One vector CTA holds V: 64 / 16 = 4 rows a warp (W 2), 128 / 24 = 6 (W 4).
int jacobi_sm_fewest(int) { return 2; }

size_t jacobi_sm_fill(void* dst, const double* C, int B, float tol32, int sweeps_max,
                         bool relative_stop, float* diag32, float* v32, DevHeader* hdr, int n) {
  Params p{};
  p.C = C;
  p.B = B;
  p.tol32 = tol32;
  p.sweeps_max = sweeps_max;
  p.relative_stop = relative_stop ? 1 : 0;
  p.nV = n - 1;
  p.diag32 = diag32;
  p.v32 = v32;
  p.hdr = hdr;
  *static_cast<Params*>(dst) = p;
  return sm_smem(jacobi_width(B));
}

// count clusters: the parameters of the first in host memory, all in device
// memory (dev_list; null: one cluster with the host parameters).
cudaError_t launch_jacobi_sm(const void* host_first, const void* dev_list, int count, size_t smem,
                                cudaStream_t st) {
  const Params& one = *static_cast<const Params*>(host_first);
  const int w = jacobi_width(one.B);
  auto kern = w == 2 ? k_jacobi_sm<2, 1, 4, kThreads2> : k_jacobi_sm<4, 2, 6, kThreads4>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((1 + one.nV) * count);
  cfg.blockDim = dim3(w == 2 ? kThreads2 : kThreads4);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1 + one.nV;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, one, static_cast<const Params*>(dev_list));
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace gbpca
