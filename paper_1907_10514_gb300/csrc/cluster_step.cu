// cluster_step.cu -- row-persistent steps of a small simulation by one thread-block cluster.
//
// The row-persistent form (fused = 5, persistent.cu) spreads n ions over every SM and pays a
// grid-wide counter per step, or holds them all in one CTA and pays that SM's FP64 pipe.  Up
// to kRpcMaxN ions one cluster of C CTAs does better: the positions travel between its CTAs
// by distributed shared memory, each store completing bytes on the receiver's mbarrier, so a
// step has no global memory access, no grid barrier and no polling of L2.
//
// What bounds a step: a chain of latencies (pair items, the Kahan merge of the parts at 16
// cycles a part, the FP64 update, the stores' flight).  The warps are specialised to keep
// everything else off it:
//   owner warps (4)  merge and integrate, a thread per ion component.  An FP64 instruction
//                    occupies its sub-partition's pipe for ~76 cycles whatever its active
//                    lanes, so each of these warps has a sub-partition to itself and the
//                    chain is five of them: the float/double conversions around it, which
//                    run at the FP64 rate, are done with integer operations.  Trap, drag,
//                    laser and kick of the next step are evaluated while the pairs run
//   noise warps (2)  the next step's normals, a thread per ion
//   pair warps (14)  the part sums; a thread keeps its ion and takes every G-th part, and
//                    each round of G parts is handed to the owners while the next one runs
//
// Measured (200 steps of 64 ions, GB300): 3.30 us per step in one CTA before, 1.21 here; 150
// ions 4.0 on the grid, 1.92 here.  Where the 2500 cycles of a step of 64 ions go: stores'
// flight and pair items 800, merge 300, FP64 update 700, stores 300, the next step's FP64
// terms 500.
//
// The bits are those of persistent.cu's kernel for the same (n, NP, JP): the same part sums
// (rp_chunk), the same merge order, the same FP64 operations.
#include <cooperative_groups.h>

#include "iontrap_internal.cuh"

namespace cg = cooperative_groups;

namespace it {

constexpr int kRpcOwners = 128, kRpcNoise = 64, kRpcPairs = 448;  // threads of each kind
constexpr int kRpcThreads = kRpcOwners + kRpcNoise + kRpcPairs;   // 20 warps: 5 per sub-partition
constexpr int kRpcNoiseWarp = 7;                                  // and the one before it: the sub-partitions of owner
                                                                  // warps 3 and 2, which own ions last
constexpr int kRpcMaxRc = 40;                                     // entries per CTA: 3 x 40 owner threads
constexpr int kRpcMaxN = 432;                                     // measured: see rpc_ctas
constexpr int kRpcGroups = 8;                                     // rounds are handed over in at most this many groups
// named barriers: 1 .. kRpcGroups the groups of rounds, then
constexpr int kRpcBarStep = 9, kRpcBarLaser = 10;
constexpr unsigned long long kRpcSettleNs = 20000;                // stores in flight land in ~1 us

struct RpcArgs {
  long long K;  // steps in this launch
  int Rc;       // entries per CTA at most, a multiple of 4 (stores of four ions)
  int JP;       // j entries per part of the row-persistent shape (<= 128: one chunk)
  int NPe;      // parts that hold an ion: ceil(n / JP)
  int nspecies;
};

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// Four floats into another CTA's shared memory, counted on that CTA's mbarrier.
__device__ __forceinline__ void st_async4(uint32_t dst, const float (&q)[4], uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
               "r"(__float_as_uint(q[0])), "r"(__float_as_uint(q[1])), "r"(__float_as_uint(q[2])),
               "r"(__float_as_uint(q[3])), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Wait for the positions, giving up after limit ns or when another warp of the CTA has (*given).
__device__ __forceinline__ bool rpc_wait(uint64_t* bar, uint32_t parity, unsigned long long limit,
                                         const volatile int* given) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity))
    if (*given || globaltimer_ns() - t0 > limit) return false;
  return true;
}

// Part sums are kept [part][kRpcOwners] by owner thread: constant offsets for the merge.

// The sums of one ion (global index i) against the parts first, first + G, ... below NPe, left
// in ps (this ion's x entry; y and z at stride row); a group's barrier is passed on after every
// `per` rounds.  Every part tests for the self pair: one copy of the loop in the instruction
// cache is worth more than its two selects.
template <bool UNITW>
__device__ __forceinline__ void rpc_parts(const float* sb, const float* wz, float* ps, int row, int JP, int NPe, int G,
                                          int per, int groups, int first, int i, bool on) {
  float2 nh[3], nl[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float h = on ? -sb[rpc_at(i, d)] : 0.f, l = on ? -sb[rpc_at(i, 3 + d)] : 0.f;
    nh[d] = make_float2(h, h), nl[d] = make_float2(l, l);
  }
  int p = on ? first : NPe;
  for (int g = 0; g < groups; ++g) {
    for (int k = 0; k < per; ++k, p += G)
      if (p < NPe) {
        float f[3];
        rec_part<UNITW>(sb, wz, p * JP, JP, i, nh, nl, f);
#pragma unroll
        for (int d = 0; d < 3; ++d) ps[p * kRpcOwners + d * row] = f[d];
      }
    bar_arrive(1 + g, kRpcOwners + kRpcPairs);
  }
}

template <bool UNITW>
__global__ void __launch_bounds__(kRpcThreads, 1) k_step_f32_rpc(const __grid_constant__ StepArgs A, const RpcArgs P) {
  // two position buffers of NPe JP / 4 records, the charges [NPe JP], part sums
  // [NPe][kRpcOwners], normals of two steps [2][3][Rc], the RF
  // phase of the K steps, drag velocities [3][Rc], spring constants of two steps
  // [2][species][3]
  extern __shared__ __align__(16) float4 s_dyn[];
  __shared__ __align__(8) uint64_t bar[2];  // positions of a buffer complete
  __shared__ volatile int s_bad[2];         // a wait of this CTA gave up in an even, an odd step
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x;
  const int n = (int)A.n, n4 = (n + 3) & ~3, K = (int)P.K;
  const int Rc = P.Rc, NPe = P.NPe, JP = P.JP;
  const int blen = NPe * 6 * JP;
  float* buf = reinterpret_cast<float*>(s_dyn);
  float* wz = buf + 2 * blen;
  float* ps = wz + NPe * JP;
  float* zb = ps + NPe * kRpcOwners;
  double* scos = reinterpret_cast<double*>(zb + 6 * Rc);  // every array before is a multiple of 16 bytes
  double* svd = scos + K;
  double* sspr = svd + 3 * Rc;
  // the groups of four ions spread evenly: every CTA owns at least one.  (One without ions
  // would not be held back by its own stores: its pair warps could pass the owners' barriers
  // a step ahead of them)
  const int quad0 = rank * (n4 / 4) / C;
  const int r0 = 4 * quad0;
  const int Rg4 = 4 * ((rank + 1) * (n4 / 4) / C - quad0);  // entries of this CTA, a multiple of 4
  const int Rg = min(Rg4, n - r0);                          // of which ions
  const uint32_t step_bytes = 24u * (uint32_t)n4;
  const TrapDev& tp = A.trap;
  const long long ns0 = *A.step;
  const bool rf = !(tp.flags & (IONTRAP_RF_OFF | IONTRAP_TRAP_OFF | IONTRAP_PSEUDO));
  const unsigned long long lim = A.wait_ns ? A.wait_ns : kWaitLimitNs;

  if (tid == 0) {
    s_bad[0] = s_bad[1] = 0;
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    for (int b = 0; b < 2; ++b) mbar_arrive_expect_tx(&bar[b], step_bytes);
  }
  // the K cosines shared out among the CTAs (one takes a warp ~2 us of its FP64 pipe)
  for (int k = rank + C * tid; k < K; k += C * kRpcThreads)
    scos[k] = rf ? cos(tp.Omega * ((double)(ns0 + k + 1) * tp.dt)) : 0.0;
  // positions x_{ns0+1} into buffer 0, the padding into both
  {
    const int rb = (int)((ns0 + 1) & 1);
    const float4* __restrict__ ghi = A.hi[rb];
    const float4* __restrict__ glo = A.lo[rb];
    for (int e = tid; e < NPe * JP; e += kRpcThreads) {
      float4 h = make_float4(1e30f, 1e30f, 1e30f, 0.0f), l = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < n) h = __ldcg(ghi + e), l = __ldcg(glo + e);
      float* d = buf + rpc_at(e, 0);
      d[0] = h.x, d[4] = h.y, d[8] = h.z, d[12] = l.x, d[16] = l.y, d[20] = l.z;
      wz[e] = h.w;
      if (e >= n) {
        d += blen;
        d[0] = d[4] = d[8] = 1e30f;
        d[12] = d[16] = d[20] = 0.f;
      }
    }
  }
  // noise threads: an ion each; the normals of the first step
  const int warp = tid >> 5, lane = tid & 31;
  const int zq = warp == kRpcNoiseWarp ? lane : warp == kRpcNoiseWarp - 1 ? 32 + lane : -1;
  const bool noisy = zq >= 0 && zq < Rg && A.spc[A.sp[r0 + zq]].sigma > 0.0;
  auto draw = [&](int t) {
    float zz[3];
    normals3_f32(tp.seed, ns0 + t + 1, r0 + zq, zz);
    float* z = zb + (t & 1) * 3 * Rc + zq;
    z[0] = zz[0], z[Rc] = zz[1], z[2 * Rc] = zz[2];
  };
  if (noisy) draw(0);
  cluster.sync();  // barriers armed and positions staged before the first remote store
  for (int k = tid; k < K; k += kRpcThreads)
    if (k % C != rank) scos[k] = *cluster.map_shared_rank(scos + k, (unsigned)(k % C));
  __syncthreads();
  // and the spring constants of a step, a lane per species and component
  auto springs = [&](int t) {
    for (int k = lane; k < 3 * P.nspecies; k += 32)
      sspr[(t & 1) * 3 * IONTRAP_MAX_SPECIES + k] = trap_spring_c(tp, A.spc[k / 3], scos[t], k % 3);
  };
  if (warp == kRpcNoiseWarp) springs(0);
  __syncthreads();

  // the parts are taken in rounds of G (one per pair thread of an ion)
  const int G = kRpcPairs / Rg;
  const int rounds = (NPe + G - 1) / G;
  const int per = (rounds + kRpcGroups - 1) / kRpcGroups, groups = (rounds + per - 1) / per;

  // A wait that gives up ends the launch for the whole CTA at one step: the warp sets the step's
  // s_bad before it passes on its groups, so the value is settled when the owners have merged and
  // when the 20 warps have met at kRpcBarStep, after which they leave by it.  No pair warp is in the
  // next step before that barrier, and that step has a flag of its own; the step after it, which
  // has this one again, begins when every warp has read it.  A launch's last step ends without the
  // barrier: nothing waits after it.  (That the pair warps come to the barrier costs nothing: the
  // positions that they wait for next are in flight for longer.  64 ions, 200 steps and the state:
  // 267 us with 6 warps at the barrier, 267 with 20.)
  if (warp > kRpcNoiseWarp || (warp >= kRpcOwners / 32 && warp < kRpcNoiseWarp - 1)) {  // -------- pair warps
    const int pt = tid - kRpcOwners - (warp > kRpcNoiseWarp ? kRpcNoise : 0);
    const int first = pt / Rg, s = pt - first * Rg;
    const bool on = first < G;
    const int i = r0 + s;
    for (int t = 0; t < K; ++t) {
      const int cur = t & 1;
      if (t > 0) {
        const bool ok = rpc_wait(&bar[cur], (uint32_t)(((t - 1) >> 1) & 1), lim, &s_bad[cur]);
        if (__any_sync(0xffffffffu, !ok)) {  // give up; the owners and the other warps follow
          s_bad[cur] = 1;
          __threadfence_block();
          for (int g = 0; g < groups; ++g) bar_arrive(1 + g, kRpcOwners + kRpcPairs);
          if (t + 1 < K) bar_sync(kRpcBarStep, kRpcThreads);
          break;
        }
        // armed again for the positions two steps on: their senders wait for this CTA's own
        // of this step, which its owners send after every pair thread has arrived
        if (pt == 0) mbar_arrive_expect_tx(&bar[cur], step_bytes);
      }
      rpc_parts<UNITW>(buf + cur * blen, wz, ps + s, Rg4, JP, NPe, G, per, groups, first, i, on);
      if (t + 1 == K) break;
      bar_sync(kRpcBarStep, kRpcThreads);
      if (s_bad[cur]) break;
    }
  } else if (tid >= kRpcOwners) {  // -------------------------------------------- noise warps
    for (int t = 0; t + 1 < K; ++t) {
      if (warp == kRpcNoiseWarp) springs(t + 1);
      if (noisy) draw(t + 1);
      bar_sync(kRpcBarStep, kRpcThreads);
      if (s_bad[t & 1]) break;
    }
  } else {  // ------------------------------------------------------------------- owner warps
    // thread k < 3 Rg4 integrates component k / Rg4 of ion r0 + k % Rg4 (a padding entry
    // only sends its constant position)
    const int oc = tid / Rg4, oq = tid - oc * Rg4;
    const bool owns = tid < 3 * Rg4, own = owns && oq < Rg;
    const unsigned quads = __ballot_sync(0xffffffffu, owns);  // whole groups of four lanes
    const int ie = r0 + oq;
    double xf = 0.0, vd = 0.0, ext = 0.0;
    double ngamma = 0.0, sigma = 0.0, coul = 0.0, lrate = 0.0, kdir = 0.0;
    const int spe = own ? A.sp[ie] : 0;
    if (own) {
      const SpeciesDev& sd = A.spc[spe];
      ngamma = -sd.gamma, sigma = sd.sigma, coul = sd.coul, lrate = sd.lrate, kdir = sd.kdir[oc];
      vd = half_kick(A.v[oc * A.n + ie], A.a[oc * A.n + ie], tp.hdt);
      xf = drift(A.x[oc * A.n + ie], vd, tp.dt);
    }
    // force-independent terms of step t (the operations and order of accel_ext); the laser
    // needs all three components of an ion
    auto ext_of = [&](int t) {
      if (own)
        ext = __fma_rn(ngamma, vd, __dmul_rn(-sspr[((t & 1) * IONTRAP_MAX_SPECIES + spe) * 3 + oc], xf));
      if (tp.laser) {
        if (own) svd[oc * Rc + oq] = vd;
        bar_sync(kRpcBarLaser, kRpcOwners);
        if (own && lrate != 0.0) {
          const double v3[3] = {svd[oq], svd[Rc + oq], svd[2 * Rc + oq]};
          ext = __fma_rn(-laser_proj(A.spc[spe], v3), kdir, ext);
        }
      }
      if (own && sigma > 0.0) ext = __fma_rn(sigma, widen(zb[((t & 1) * 3 + oc) * Rc + oq]), ext);
    };
    // the CTAs this thread stores to, (tid & 3) + 4 k: its four ions' entry in buffer 0 and
    // the buffer's mbarrier there
    uint32_t rdst[4], rbar[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t r = (uint32_t)min((tid & 3) + 4 * k, C - 1);
      rdst[k] = map_rank(smem_u32(buf + (owns ? rpc_at(ie & ~3, oc) : 0)), r);
      rbar[k] = map_rank(smem_u32(&bar[0]), r);
    }
    // the step after which a CTA that the failure test stalls keeps its positions to itself
    const int stall_t = A.stall_on && rank == A.stall_cta && A.stall_step < K ? (int)A.stall_step : -1;
    ext_of(0);
    for (int t = 0; t < K; ++t) {
      const int cur = t & 1;
      // merge in part order (Kahan; the parts' compensations are zero), a group of rounds
      // at a time, eight loads in flight.  The parts without
      // ions, whose sums are zero, are left out: adding zeros only moves the sum's low bits
      // between su and cu, and their difference below is the same
      float su = 0.f, cu = 0.f;
      const float* q = ps + tid;
      int p = 0;
      auto add = [&](float v) {
        const float y = v - cu;
        const float tt = su + y;
        cu = (tt - su) - y;
        su = tt;
      };
      for (int g = 0; g < groups; ++g) {
        bar_sync(1 + g, kRpcOwners + kRpcPairs);
        const int p1 = min(NPe, (g + 1) * per * G);
#pragma unroll 1
        for (; p + 8 <= p1; p += 8, q += 8 * kRpcOwners) {
          float v[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = q[k * kRpcOwners];
#pragma unroll
          for (int k = 0; k < 8; ++k) add(v[k]);
        }
        if (p + 4 <= p1) {
          float v[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = q[k * kRpcOwners];
#pragma unroll
          for (int k = 0; k < 4; ++k) add(v[k]);
          p += 4, q += 4 * kRpcOwners;
        }
#pragma unroll 1
        for (; p < p1; ++p, q += kRpcOwners) add(q[0]);
      }
      const bool bad = s_bad[cur] != 0;
      float h = 1e30f, l = 0.0f;
      if (own && !bad) {
        const double Sd = widen(cu) - widen(su);
        const double acc = __fma_rn(coul, Sd, ext);
        const double vn = half_kick(vd, acc, tp.hdt);
        const double vh = half_kick(vn, acc, tp.hdt);
        const double xn = drift(xf, vh, tp.dt);
        split_hilo(xn, h, l);
        if (t + 1 == K) {  // the launch's last step: FP64 state and the pair stream
          const int wb = (int)((ns0 + t) & 1);
          A.x[oc * A.n + ie] = xf;
          A.v[oc * A.n + ie] = vn;
          A.a[oc * A.n + ie] = acc;
          reinterpret_cast<float*>(A.hi[wb] + ie)[oc] = h;
          reinterpret_cast<float*>(A.lo[wb] + ie)[oc] = l;
          if (oc == 0) {
            reinterpret_cast<float*>(A.hi[wb] + ie)[3] = A.spc[spe].w;
            reinterpret_cast<float*>(A.lo[wb] + ie)[3] = 0.0f;
          }
        }
        if ((((unsigned)__double2hiint(xn) >> 20) & 0x7ffu) == 0x7ffu) atomicOr(A.err, ERR_NONFINITE);
        vd = vh;
        xf = xn;
      }
      if (t + 1 == K) break;
      if (owns && !bad && t != stall_t) {
        // four consecutive threads hold four consecutive ions: each collects the four and
        // stores them to every fourth CTA
        const int base = tid & 28;
        float h4[4], l4[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) h4[k] = __shfl_sync(quads, h, base + k), l4[k] = __shfl_sync(quads, l, base + k);
        const uint32_t to = (cur ^ 1) ? 4u * (uint32_t)blen : 0u, tb = (cur ^ 1) ? 8u : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((tid & 3) + 4 * k < C) {
            st_async4(rdst[k] + to, h4, rbar[k] + tb);
            st_async4(rdst[k] + to + 48u, l4, rbar[k] + tb);
          }
      }
      bar_sync(kRpcBarStep, kRpcThreads);  // the next step's normals are there
      if (bad) break;
      ext_of(t + 1);
    }
    if (tid == 0 && (s_bad[0] | s_bad[1])) atomicOr(A.err, ERR_TIMEOUT);
  }
  cluster.sync();  // every store has been sent, and has landed in the CTAs that did not give up
  if (s_bad[0] | s_bad[1]) {  // others' stores may be in flight to this one
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < kRpcSettleNs) {
    }
  }
  if (rank == 0 && tid == 0 && !(*(volatile int*)A.err & ERR_TIMEOUT)) *A.step = ns0 + P.K;
}

size_t rpc_smem_bytes(int Rc, int NPe, int JP, long long K) {
  return (13 * (size_t)NPe * JP + (size_t)NPe * kRpcOwners + 6 * (size_t)Rc) * sizeof(float) +
         ((size_t)K + 3 * (size_t)Rc + 6 * IONTRAP_MAX_SPECIES) * sizeof(double);
}

// CTAs of the cluster that steps n ions in parts of JP entries, or 0 where the grid is taken:
// above kRpcMaxN, or when a part is longer than one chunk.  More CTAs shorten the pair phase
// and lengthen nothing but the stores (a CTA needs four ions at least); us per step measured
// on GB300, default shapes, grid or single CTA / clusters of 1, 4, 8, 16:
//   n = 16: 2.84 / 1.15 1.07 - -      64: 3.30 / - 1.26 1.21 1.23    100: 4.97 / - 1.61 1.57 1.43
//   128: 5.69 / - 2.05 1.73 1.53     200: 4.09 / - - 2.50 2.14       256: 4.13 / - - 3.06 2.58
//   400: 3.49 / - - - 3.10           512: 3.51 / - - - 4.1
// Above 168 ions shapes of 8 warps are stepped by tagged_step.cu instead.
static int rpc_entries(long long n, int C) { return (int)(((n + 3) / 4 + C - 1) / C * 4); }
int rpc_ctas(long long n, int JP) {
  if (JP > kSeg || n > kRpcMaxN) return 0;
  const int C = n < 13 ? 1 : n < 29 ? 4 : n <= 84 ? 8 : 16;
  return rpc_entries(n, C) <= kRpcMaxRc ? C : 0;  // three owner threads an entry
}

cudaError_t launch_rpc(const StepArgs& a, int nspecies, int C, int JP, long long K, cudaStream_t st) {
  RpcArgs P{};
  P.K = K;
  P.JP = JP;
  P.nspecies = nspecies;
  P.NPe = (int)((a.n + JP - 1) / JP);
  P.Rc = rpc_entries(a.n, C);
  const size_t smem = rpc_smem_bytes(P.Rc, P.NPe, JP, K);
  const auto fn = a.unitw ? k_step_f32_rpc<true> : k_step_f32_rpc<false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3(kRpcThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, a, P);
}

}  // namespace it
