// forces_noalloc.cu -- Coulomb accelerations without any device allocation.
//
// iontrap_forces evaluates the force kernel on a handle, and a handle owns device
// buffers.  Some callers cannot allocate: a process that hands all of its device memory
// to its own pool up front and forbids allocations behind its back, a host application
// that loads this library as a plugin and owns every device buffer itself, or a
// latency-critical loop that must not pay for cudaMalloc's implicit synchronisation.  For
// them, iontrap_forces_noalloc takes the positions and the output in the caller's device
// memory and needs nothing else: one kernel, whose partial sums never leave the chip.
//
// A cluster of S <= 8 CTAs sums 32 or 64 ions (one per lane, or two packed), CTA s against the
// s-th of S equal j-ranges.  Warp w of a CTA takes the range's w-th chunk of 128 j: it splits the
// FP64 positions into hi/lo floats itself (integer operations: the FP64 pipe would take
// longer than the pairs at small n), and its plain FP32 chunk sums are Kahan-added in chunk
// order by the CTA, the CTAs' (sum, compensation) pairs merged in range order through
// distributed shared memory.  That is the summation order (and the bits) of the last-CTA step
// form with these j-ranges, without its scratch, counters and clears.
//
// Bound by the FP32 pipe at n = 8192 (half of its rate: few warps, the split of the positions
// in every CTA) and by the launch and one chunk's latency below ~2000.  Measured back to back on
// GB300, us per call, the previous two clears and two launches against this kernel: n = 64:
// 17 -> 8.3, 1000: 21 -> 8.3, 3000: 32 -> 14.4, 5000: 46 -> 24.6, 8192: 77 -> 52.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "iontrap_internal.cuh"

namespace cg = cooperative_groups;
using namespace it;

namespace {

constexpr long long kNoAllocMaxIons = 8192;
constexpr int kNoAllocMaxSplits = 8;
constexpr int kMaxChunks = (int)(kNoAllocMaxIons / kNoAllocMaxSplits / kSeg);  // warps per CTA: 8

struct ForcesArgs {
  int n, jsplit;
  const unsigned char* sp;
  const double* x;
  double* out;
  double coul[IONTRAP_MAX_SPECIES];
  float w[IONTRAP_MAX_SPECIES];
};

// I ions per lane: 1, or 2 packed.  M: CTAs of eight warps that the registers leave room for, at
// least.  Without that bound the compiler took 158 for the pair loop written in stages of 16 j and
// two CTAs of five warps shared an SM (n = 5000: 28.5 us a call, 24.6 with M = 1 and 95 registers);
// 64 registers (M = 4) take stages of 4 j, and with two ions and unit charges still one spilled word,
// which the fourth CTA outweighs (n = 7000: 45.9 -> 39.2 us).
template <int I, bool UNITW, int M>
__global__ void __launch_bounds__(32 * kMaxChunks, M) k_forces_cluster(const __grid_constant__ ForcesArgs A) {
  constexpr int kBlockIons = 32 * I, kStage = M == 1 ? 16 : 4;
  __shared__ __align__(16) float4 sh[kMaxChunks][kSeg], sl[kMaxChunks][kSeg];
  __shared__ float s_sum[kMaxChunks][3][kBlockIons];   // chunk sums; row 0 then the CTA's Kahan sum
  __shared__ float s_comp[3][kBlockIons];              // and compensation
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
  const int n = A.n, i0 = blockIdx.x * kBlockIons;
  const int j0 = blockIdx.y * A.jsplit, j1 = min(n, j0 + A.jsplit);
  const int chunks = (j1 - j0 + kSeg - 1) / kSeg;
  const int jc = j0 + warp * kSeg, jn = min(kSeg, j1 - jc);
  if (jn > 0) {
    // every load first (one trip to memory), then the conversions
    constexpr int Q = kSeg / 32;
    double x[Q + I][3];
    float w[Q];
    long long ii[I];
#pragma unroll
    for (int q = 0; q < Q + I; ++q) {
      const int e = q < Q ? jc + 32 * q + lane : i0 + 32 * (q - Q) + lane;
      const bool on = q < Q ? 32 * q + lane < jn : e < n;
      if (q >= Q) ii[q - Q] = e;
#pragma unroll
      for (int d = 0; d < 3; ++d) x[q][d] = on ? A.x[d * n + e] : 1.0;  // (unused)
      if (q < Q) w[q] = UNITW ? 1.0f : (on ? A.w[A.sp[e]] : 0.0f);
    }
    float2 nxh[1][3], nxl[1][3], acc[1][3];
#pragma unroll
    for (int q = 0; q < Q + I; ++q) {
      float h[3], l[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) split_hilo(x[q][d], h[d], l[d]);
      if (q < Q) {
        sh[warp][32 * q + lane] = make_float4(h[0], h[1], h[2], w[q]);
        sl[warp][32 * q + lane] = make_float4(l[0], l[1], l[2], 0.0f);
      } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (q == Q)
            nxh[0][d].x = -h[d], nxl[0][d].x = -l[d];
          else
            nxh[0][d].y = -h[d], nxl[0][d].y = -l[d];
          acc[0][d] = make_float2(0.f, 0.f);
        }
      }
    }
    __syncwarp();
    const bool diag = jc < i0 + kBlockIons && i0 < jc + jn;
    if constexpr (I == 1) {
      const float h1[1][3] = {{nxh[0][0].x, nxh[0][1].x, nxh[0][2].x}};
      const float l1[1][3] = {{nxl[0][0].x, nxl[0][1].x, nxl[0][2].x}};
      float a1[1][3] = {{0.f, 0.f, 0.f}};
      if (diag)
        segment_f32<1, true, UNITW>(sh[warp], sl[warp], jn, jc, h1, l1, ii, a1);
      else
        segment_f32<1, false, UNITW>(sh[warp], sl[warp], jn, jc, h1, l1, ii, a1);
#pragma unroll
      for (int d = 0; d < 3; ++d) acc[0][d].x = a1[0][d];
    } else {
      if (diag)
        segment_f32x2<I, true, UNITW, kStage>(sh[warp], sl[warp], jn, jc, nxh, nxl, ii, acc);
      else
        segment_f32x2<I, false, UNITW, kStage>(sh[warp], sl[warp], jn, jc, nxh, nxl, ii, acc);
    }
#pragma unroll
    for (int k = 0; k < I; ++k)
#pragma unroll
      for (int d = 0; d < 3; ++d) s_sum[warp][d][32 * k + lane] = k ? acc[0][d].y : acc[0][d].x;
  }
  __syncthreads();
  // the chunks' sums, Kahan-added in chunk order (the accumulators hold the negated sums)
  for (int k = tid; k < 3 * kBlockIons; k += threads) {
    float ks = 0.0f, kc = 0.0f;
    for (int c = 0; c < chunks; ++c) {
      const float y = (&s_sum[c][0][0])[k] - kc;
      const float t = ks + y;
      kc = (t - ks) - y;
      ks = t;
    }
    (&s_sum[0][0][0])[k] = ks;
    (&s_comp[0][0])[k] = kc;
  }
  cluster.sync();
  // CTA r finishes its share of the ions: the S partials in range order
  const int S = (int)gridDim.y, r = (int)cluster.block_rank(), per = (kBlockIons + S - 1) / S;
  for (int k = tid; k < 3 * per; k += threads) {
    const int c = k / per, q = r * per + (k - c * per), i = i0 + q;
    if (q >= kBlockIons || i >= n) continue;
    float su = 0.f, cu = 0.f, a[kNoAllocMaxSplits], b[kNoAllocMaxSplits];
#pragma unroll
    for (int p = 0; p < kNoAllocMaxSplits; ++p)
      if (p < S) {
        a[p] = *cluster.map_shared_rank(&s_sum[0][c][q], (unsigned)p);
        b[p] = *cluster.map_shared_rank(&s_comp[c][q], (unsigned)p);
      }
#pragma unroll
    for (int p = 0; p < kNoAllocMaxSplits; ++p)
      if (p < S) kahan_merge(su, cu, a[p], b[p]);
    A.out[(size_t)c * n + i] = A.coul[A.sp[i]] * (widen(cu) - widen(su));
  }
  cluster.sync();  // nobody leaves while others read its shared memory
}

}  // namespace

extern "C" int iontrap_forces_noalloc(const iontrap_species* species, int n_species,
                                      const uint8_t* d_species_of_ion, const double* d_x, int64_t n,
                                      double* d_acc, void* cuda_stream) {
  if (!species || n_species < 1 || n_species > IONTRAP_MAX_SPECIES || !d_species_of_ion || !d_x || !d_acc ||
      n < 1)
    return IONTRAP_EINVAL;
  for (int s = 0; s < n_species; ++s)
    if (!(species[s].mass_amu > 0) || !std::isfinite(species[s].mass_amu) || !std::isfinite(species[s].charge_e))
      return IONTRAP_EINVAL;
  if (n > kNoAllocMaxIons) return IONTRAP_ETOOLARGE;

  ForcesArgs A{};
  A.n = (int)n, A.sp = d_species_of_ion, A.x = d_x, A.out = d_acc;
  // equal j-ranges of at least 128 ions, at most 8
  const long long splits = std::min<long long>(kNoAllocMaxSplits, std::max<long long>(1, (n + 127) / 128));
  A.jsplit = (int)((n + splits - 1) / splits);
  const unsigned nsplit = (unsigned)((n + A.jsplit - 1) / A.jsplit);
  const double ke = 1.0 / (4.0 * kPi * kEps0);
  bool unitw = true;
  for (int s = 0; s < n_species; ++s) {
    const double M = species[s].mass_amu * kAmu, z = species[s].charge_e;
    A.coul[s] = ke * kE * kE * z / M;
    A.w[s] = (float)z;
    unitw = unitw && z == 1.0;
  }
  cudaLaunchConfig_t cfg{};
  // one ion per lane while the chip is short of warps (us per call, 1 / 2 ions per lane:
  // n = 2600: 12.3 / 14.4, 3201: 16.4 / 14.4, 4097: 22.6 / 18.5, 8192: 60 / 54); and from seven
  // warps a CTA on four CTAs per SM rather than three (M = 1 / 4: n = 5000: 24.6 / 26.7, 6000:
  // 32.8 / 32.8, 7000: 45.9 / 39.2, 8192: 53.8 / 52.1; with a doubly charged species 7000: 48.7 / 41.1)
  const int I = n <= 2800 ? 1 : 2;
  const bool four = A.jsplit > 6 * kSeg;
  cfg.gridDim = dim3((unsigned)((n + 32 * I - 1) / (32 * I)), nsplit);
  cfg.blockDim = dim3(32u * (unsigned)((A.jsplit + kSeg - 1) / kSeg));
  cfg.stream = static_cast<cudaStream_t>(cuda_stream);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = nsplit;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(
      &cfg, I == 1 ? (unitw ? k_forces_cluster<1, true, 1> : k_forces_cluster<1, false, 1>)
            : four ? (unitw ? k_forces_cluster<2, true, 4> : k_forces_cluster<2, false, 4>)
                   : (unitw ? k_forces_cluster<2, true, 1> : k_forces_cluster<2, false, 1>), A);
  return e == cudaSuccess ? IONTRAP_OK : IONTRAP_ECUDA;
}
