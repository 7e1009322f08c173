// minimize.cu -- the iterations of a minimisation (modes.cu states the method) in one launch.
//
// For handles in the row-persistent form.  modes.cu's kernels take a cooperative force launch
// and three more per iteration, ~30 us on GB300 whatever n.  Here CTAs that hold all positions in
// shared memory, as the row-persistent step does, run the iterations themselves: three
// barriers an iteration, for the force and power sums, the largest displacement and the new
// positions.  Up to kMinClusterN ions the CTAs are one thread-block cluster and the barriers
// the hardware's; above, the grid of the step form and a counter polled in L2.
//
// What bounds an iteration is its chain of FP64 instructions (~68 cycles each: the sum tree,
// two divisions, a root) and the three barriers; comparisons with the tolerance and the step
// limit are decided on integers, and in a cluster only the owner warps issue FP64 work.
// Measured (us per iteration, modes.cu's kernels against this launch): n = 20: 29 -> 2.6,
// 200: 32 -> 5.2, 432: 33 -> 5.7 (cluster), 1000: 34 -> 12, 4096: 46 -> 27 (grid).
//
// Bits: the force is the row-persistent form's (same part sums, same merge), every FP64
// expression is modes.cu's, and the sums over ions are its tree (256 ions by halves, blocks in
// order), evaluated by every CTA alike.
#include <cooperative_groups.h>

#include "iontrap_internal.cuh"

namespace cg = cooperative_groups;

namespace it {

constexpr int kMinWarps = 16, kMinT = 32 * kMinWarps;
constexpr int kMinClusterN = 432;
constexpr int kMinMaxBlocks = 32;  // blocks of 256 ions: n <= 8192

struct MinRpArgs {
  long long n;
  double* x;
  double* v;
  const unsigned char* sp;
  float4* hi;
  float4* lo;
  double2* ion;      // [n]: F.F and v.F of an ion
  double* dmax;      // [CTAs]: largest squared displacement of a CTA
  unsigned* sync;    // arrival counter (zero before a launch)
  int* err;
  MinResult* res;
  double dt, dmaxlim, ftol;
  long long iters;   // at most this many moves in this launch
  int final_eval;    // evaluate |F| after the last move
  int R, NP, JP, unitw;
  unsigned long long limit;  // of a barrier's wait, ns
  long long stall_at;        // the barrier (counted from 0) that CTA stall_cta does not arrive at; -1: none
  int stall_cta;
  TrapDev trap;
  SpeciesDev spc[IONTRAP_MAX_SPECIES];
};

// Sum of up to 256 ions' values in the order of modes.cu's block reduction: ion t takes t + 128,
// then t + 64, ...; a warp's lane holds the ions lane + 32 k.  Levels that only add the zeros
// past `left` ions are left out.  The sum in lane 0's f[0].
__device__ __forceinline__ void tree256(double (&f)[8], int left) {
  if (left > 128)
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] += f[k + 4];
  if (left > 64)
#pragma unroll
    for (int k = 0; k < 2; ++k) f[k] += f[k + 2];
  if (left > 32) f[0] += f[1];
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) f[0] += __shfl_down_sync(0xffffffffu, f[0], h);
}

// Largest of a warp's values (not negative), on the bits; what is not a number counts as zero,
// as fmax passes it over.
__device__ __forceinline__ double warp_max(double m) {
  const bool num = m == m;
  const unsigned hw = num ? (unsigned)__double2hiint(m) : 0u, lw = num ? (unsigned)__double2loint(m) : 0u;
  const unsigned hm = __reduce_max_sync(0xffffffffu, hw);
  const unsigned lm = __reduce_max_sync(0xffffffffu, hw == hm ? lw : 0u);
  return __hiloint2double((int)hm, (int)lm);
}

// sqrt(q) < lim, decided on the squares unless they are close: values that are not negative
// compare as integers, so the usual case costs no FP64 instruction (what is not a number is not
// below).
struct SquareLimit {
  double lim;
  unsigned long long lo, hi;  // bits of lim^2 (1 -+ 1e-9)
};

__device__ __forceinline__ unsigned long long bits_of(double q) { return (unsigned long long)__double_as_longlong(q); }
__device__ __forceinline__ SquareLimit square_limit(double lim) {
  return {lim, bits_of(lim * lim * (1.0 - 1e-9)), bits_of(lim * lim * (1.0 + 1e-9))};
}
__device__ __forceinline__ bool below(double q, const SquareLimit& L) {
  if (bits_of(q) < L.lo) return true;
  if (bits_of(q) > L.hi) return false;
  return sqrt(q) < L.lim;
}

// min(1, dmax / m) for the largest squared displacement m^2; well below the limit without the
// root and the division.
__device__ __forceinline__ double move_scale(double m2, const SquareLimit& dmax) {
  if (bits_of(m2) < dmax.lo) return 1.0;
  const double m = sqrt(m2);
  return (m > 0.0 && dmax.lim < m) ? dmax.lim / m : 1.0;
}

__global__ void __launch_bounds__(kMinT, 1) k_minimize_rp(const __grid_constant__ MinRpArgs A) {
  // all positions as in the row-persistent step, the part sums and compensations
  // [NP][3][R], per owned ion component: F (or displacement) and v [2][3][R]
  extern __shared__ __align__(16) float4 s_dyn[];
  __shared__ double s_blk[kMinMaxBlocks][2];
  __shared__ double s_w[kMinWarps];
  __shared__ double s_one[3];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = (int)A.n, R = A.R, NP = A.NP, JP = A.JP;
  const int r0 = blockIdx.x * R, Rg = max(0, min(R, n - r0));
  const int NPe = min(NP, (n + JP - 1) / JP);  // parts with ions; the others add zeros
  const unsigned G = gridDim.x;
  float* sall = reinterpret_cast<float*>(s_dyn);
  float* ps = sall + (size_t)NP * 7 * JP;
  float* pc = ps + NP * 3 * R;
  double* sF = reinterpret_cast<double*>(pc + NP * 3 * R);  // 28 NP JP + 24 NP R bytes in: 8-byte aligned
  double* sv = sF + 3 * R;
  unsigned arrived = 0;
  bool bad = false;
  // every CTA's writes before are visible to every CTA after
  auto barrier = [&]() {
    ++arrived;
    __syncthreads();
    if (tid == 0) {
      if (!((int)blockIdx.x == A.stall_cta && arrived == A.stall_at + 1)) arrive_release(A.sync);
      bad = !poll_wait<true>(A.sync, G * arrived, A.err, A.limit);
    }
    bad = __syncthreads_or(bad);
  };
  // owner thread k < 3 Rg: component k / Rg of ion r0 + k % Rg
  const int rq = max(Rg, 1), oc = tid / rq, oq = tid - oc * rq;
  const bool own = tid < 3 * Rg;
  const int ie = r0 + oq;
  int spe = 0;
  double x = 0.0, v = 0.0, a = 0.0, kx = 0.0, mass = 0.0, coul = 0.0;
  if (own) {
    spe = A.sp[ie];
    x = A.x[oc * (long long)n + ie], v = A.v[oc * (long long)n + ie];
    kx = trap_spring_c(A.trap, A.spc[spe], 0.0, oc);
    mass = A.spc[spe].mass, coul = A.spc[spe].coul;
  }
  const SquareLimit ftol = square_limit(A.ftol), dmax = square_limit(A.dmaxlim);
  long long it = 0;
  for (;; ++it) {
    const bool last = it == A.iters;
    if (last && !A.final_eval) break;
    // positions
    for (int e = tid; e < NP * JP; e += kMinT) {
      const int p = e / JP, q = e - p * JP;
      float4 h = make_float4(1e30f, 1e30f, 1e30f, 0.0f), l = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < n) h = __ldcg(A.hi + e), l = __ldcg(A.lo + e);
      float* d = sall + (size_t)p * 7 * JP + q;
      d[0] = h.x, d[JP] = h.y, d[2 * JP] = h.z, d[3 * JP] = l.x, d[4 * JP] = l.y, d[5 * JP] = l.z, d[6 * JP] = h.w;
    }
    __syncthreads();
    // pair items (ion s, part p)
    for (int m = tid; m < Rg * NPe; m += kMinT) {
      const int p = m / Rg, s = m - p * Rg, i = r0 + s, ip = i / JP;
      const float* si = sall + (size_t)ip * 7 * JP + (i - ip * JP);
      const float* sj = sall + (size_t)p * 7 * JP;
      const float2 nh[3] = {make_float2(-si[0], -si[0]), make_float2(-si[JP], -si[JP]),
                            make_float2(-si[2 * JP], -si[2 * JP])};
      const float2 nl[3] = {make_float2(-si[3 * JP], -si[3 * JP]), make_float2(-si[4 * JP], -si[4 * JP]),
                            make_float2(-si[5 * JP], -si[5 * JP])};
      float ks[3] = {0.f, 0.f, 0.f}, kc[3] = {0.f, 0.f, 0.f};
      for (int c0 = 0; c0 < JP; c0 += kSeg) {
        const int qn = min(kSeg, JP - c0), jc = p * JP + c0;
        float2 acc[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (A.unitw)
          rp_chunk<true, true>(sj + c0, sj + 6 * JP + c0, JP, qn, jc, i, nh, nl, acc);
        else
          rp_chunk<true, false>(sj + c0, sj + 6 * JP + c0, JP, qn, jc, i, nh, nl, acc);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float u = acc[d].x + acc[d].y;
          const float y = u - kc[d];
          const float t = ks[d] + y;
          kc[d] = (t - ks[d]) - y;
          ks[d] = t;
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) ps[(p * 3 + d) * R + s] = ks[d], pc[(p * 3 + d) * R + s] = kc[d];
    }
    __syncthreads();
    if (own) {
      float su = 0.f, cu = 0.f;
      for (int p = 0; p < NPe; ++p) kahan_merge(su, cu, ps[(p * 3 + oc) * R + oq], pc[(p * 3 + oc) * R + oq]);
      for (int p = NPe; p < min(NP, NPe + 2); ++p) kahan_merge(su, cu, 0.f, 0.f);  // further zeros change nothing
      a = __fma_rn(-kx, x, __dmul_rn(coul, widen(cu) - widen(su)));
      sF[oc * R + oq] = mass * a;
      sv[oc * R + oq] = v;
    }
    __syncthreads();
    if (tid < Rg) {
      const double f0 = sF[tid], f1 = sF[R + tid], f2 = sF[2 * R + tid];
      const double v0 = sv[tid], v1 = sv[R + tid], v2 = sv[2 * R + tid];
      const double ff = square3(f0, f1, f2);
      const double vf = __fma_rn(v2, f2, __fma_rn(v1, f1, __dmul_rn(v0, f0)));
      __stcg(A.ion + r0 + tid, make_double2(ff, vf));
    }
    barrier();
    if (bad) break;
    // sums of 256 ions: ion t takes t + 128, then t + 64, ...: a warp's lane holds the ions
    // lane + 32 k (levels that only add the zeros past n are left out); one warp for F.F, one
    // for v.F
    for (int u = warp; (u >> 1) * 256 < n; u += kMinWarps) {
      const int b = u >> 1, left = n - b * 256;
      double f[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int i = b * 256 + 32 * k + lane;
        f[k] = i < n ? __ldcg(reinterpret_cast<const double*>(A.ion + i) + (u & 1)) : 0.0;
      }
      tree256(f, left);
      if (lane == 0) s_blk[b][u & 1] = f[0];
    }
    __syncthreads();
    if (tid == 0) {
      double FF = 0.0, vF = 0.0;
      for (int b = 0; b * 256 < n; ++b) FF += s_blk[b][0], vF += s_blk[b][1];
      const bool conv = below(FF, ftol);
      s_one[0] = vF > 0.0 ? vF / FF : 0.0;
      s_one[1] = FF;
      s_one[2] = conv || last ? 1.0 : 0.0;
      if ((conv || last) && blockIdx.x == 0) A.res->converged = conv ? 1 : 0;
    }
    __syncthreads();
    if (s_one[2] != 0.0) break;
    // kick, and the largest displacement
    if (own) {
      const double scale = s_one[0];
      v = __fma_rn(scale, __dmul_rn(mass, a), __dmul_rn(A.dt, a));
      sF[oc * R + oq] = A.dt * v;
    }
    __syncthreads();
    double d2 = 0.0;
    if (tid < Rg) {
      const double d0 = sF[tid], d1 = sF[R + tid], e2 = sF[2 * R + tid];
      d2 = square3(d0, d1, e2);
    }
    // the square root is monotonic: the maximum is taken before it
    if (warp * 32 < Rg) {
      d2 = warp_max(d2);
      if (lane == 0) s_w[warp] = d2;
    }
    __syncthreads();
    if (tid == 0) {
      double m = 0.0;
      for (int w = 0; w * 32 < Rg; ++w) m = fmax(m, s_w[w]);
      __stcg(A.dmax + blockIdx.x, m);
    }
    barrier();
    if (bad) break;
    if (warp == 0) {
      double m = 0.0;
      for (unsigned c = lane; c < G; c += 32) m = fmax(m, __ldcg(A.dmax + c));
      m = warp_max(m);
      if (lane == 0) {
        s_one[0] = move_scale(m, dmax);
      }
    }
    __syncthreads();
    if (own) {
      const double s = s_one[0];
      x = __fma_rn(s, A.dt * v, x);
      v = s * v;
      float h, l;
      split_hilo(x, h, l);
      __stcg(reinterpret_cast<float*>(A.hi + ie) + oc, h);
      __stcg(reinterpret_cast<float*>(A.lo + ie) + oc, l);
    }
    barrier();
    if (bad) break;
  }
  if (own) {
    A.x[oc * (long long)n + ie] = x;
    A.v[oc * (long long)n + ie] = v;
  }
  if (blockIdx.x == 0 && tid == 0) {
    A.res->iters += it;
    A.res->fnorm = sqrt(s_one[1]);
    if (it == A.iters && !A.final_eval) A.res->converged = 0;
  }
}

// The same on one cluster.  The three components of an ion sit in one warp (owner thread 30 w + k
// of warp w: component k % 3 of ion 10 w + k / 3), so that an ion's sums are shuffles; the owners'
// values wait in their CTA's shared memory and the others fetch them after a cluster barrier.
constexpr int kMinOwnIons = 10;  // ions of an owner warp
constexpr int kMinOwnWarps = 4;  // one per sub-partition: an FP64 instruction holds its pipe for 76 cycles

template <bool UNITW>
__global__ void __launch_bounds__(kMinT, 1) k_minimize_cl(const __grid_constant__ MinRpArgs A) {
  // positions in records [NPe JP / 4], charges [NPe JP], part sums [NPe][kMinT / 4]
  extern __shared__ __align__(16) float4 s_dyn[];
  __shared__ double s_ion[2][kMinOwnWarps * kMinOwnIons];   // F.F and v.F of the owned ions
  __shared__ float s_pos[6][kMinOwnWarps * kMinOwnIons];    // their positions
  __shared__ double s_max[kMinOwnWarps];                    // largest squared displacements
  __shared__ double s_blk[2][2];
  __shared__ int s_stop;
  constexpr int ROW = kMinT / 4;  // 128: three components of at most 40 ions
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int n = (int)A.n, R = A.R, JP = A.JP, NPe = (n + JP - 1) / JP;
  const int r0 = rank * R, Rg = max(0, min(R, n - r0));
  float* sb = reinterpret_cast<float*>(s_dyn);
  float* wz = sb + NPe * 6 * JP;
  float* ps = wz + NPe * JP;
  for (int e = tid; e < NPe * JP; e += kMinT) {
    float4 h = make_float4(1e30f, 1e30f, 1e30f, 0.0f), l = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < n) h = __ldcg(A.hi + e), l = __ldcg(A.lo + e);
    float* d = sb + rpc_at(e, 0);
    d[0] = h.x, d[4] = h.y, d[8] = h.z, d[12] = l.x, d[16] = l.y, d[20] = l.z;
    wz[e] = h.w;
  }
  const bool owner_warp = warp < kMinOwnWarps;
  // thread e < n fetches ion e's position from its owner
  const float* from = nullptr;
  if (tid < n) from = cluster.map_shared_rank(&s_pos[0][tid % R], (unsigned)(tid / R));
  // warp u < 4 sums F.F (u even) or v.F (u odd) of the ions 256 (u / 2) ..
  const double* sums[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = (warp >> 1) * 256 + 32 * k + lane;
    sums[k] = warp < 4 && i < n ? cluster.map_shared_rank(&s_ion[warp & 1][i % R], (unsigned)(i / R)) : nullptr;
  }
  // and the owner warps' maxima of all CTAs
  auto maxima_of = [&](int c) -> const double* {
    return owner_warp && c < C * kMinOwnWarps
               ? cluster.map_shared_rank(&s_max[c & (kMinOwnWarps - 1)], (unsigned)(c / kMinOwnWarps))
               : nullptr;
  };
  const double *maxima = maxima_of(lane), *maxima2 = maxima_of(lane + 32);
  // pair thread: its ion, and every G-th part
  const int G = Rg > 0 ? kMinT / Rg : 1;
  const int first = Rg > 0 ? tid / Rg : NPe, ps_s = tid - first * Rg, pi = r0 + ps_s;
  const bool pairs = Rg > 0 && first < G;
  // owner thread: component oc of ion r0 + oq
  const int oc = lane % 3, oq = warp * kMinOwnIons + lane / 3;
  const bool own = owner_warp && lane < 3 * kMinOwnIons && oq < Rg;
  const int ie = r0 + oq;
  double x = 0.0, v = 0.0, a = 0.0, kx = 0.0, mass = 0.0, coul = 0.0;
  if (own) {
    const SpeciesDev& sd = A.spc[A.sp[ie]];
    x = A.x[oc * (long long)n + ie], v = A.v[oc * (long long)n + ie];
    kx = trap_spring_c(A.trap, sd, 0.0, oc);
    mass = sd.mass, coul = sd.coul;
  }
  double FF = 0.0;
  bool conv = false;
  const SquareLimit ftol = square_limit(A.ftol), dmax = square_limit(A.dmaxlim);
  long long it = 0;
  __syncthreads();
  for (;; ++it) {
    const bool last = it == A.iters;
    if (last && !A.final_eval) break;
    if (pairs) {
      float2 nh[3], nl[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float h = -sb[rpc_at(pi, d)], l = -sb[rpc_at(pi, 3 + d)];
        nh[d] = make_float2(h, h), nl[d] = make_float2(l, l);
      }
      for (int p = first; p < NPe; p += G) {
        float f[3];
        rec_part<UNITW>(sb, wz, p * JP, JP, pi, nh, nl, f);
#pragma unroll
        for (int d = 0; d < 3; ++d) ps[p * ROW + 3 * ps_s + d] = f[d];
      }
    }
    __syncthreads();
    if (owner_warp) {
      float su = 0.f, cu = 0.f;
      const float* q = ps + 3 * min(oq, R - 1) + oc;
      auto add = [&](float u) {  // Kahan; the parts' compensations are zero
        const float y = u - cu, t = su + y;
        cu = (t - su) - y;
        su = t;
      };
      int p = 0;
#pragma unroll 1
      for (; p + 8 <= NPe; p += 8, q += 8 * ROW) {
        float u[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) u[k] = q[k * ROW];
#pragma unroll
        for (int k = 0; k < 8; ++k) add(u[k]);
      }
#pragma unroll 1
      for (; p < NPe; ++p, q += ROW) add(q[0]);
      a = __fma_rn(-kx, x, __dmul_rn(coul, widen(cu) - widen(su)));
      const double F = mass * a;
      const double F1 = __shfl_down_sync(0xffffffffu, F, 1), F2 = __shfl_down_sync(0xffffffffu, F, 2);
      const double v1 = __shfl_down_sync(0xffffffffu, v, 1), v2 = __shfl_down_sync(0xffffffffu, v, 2);
      if (own && oc == 0) {
        s_ion[0][oq] = square3(F, F1, F2);
        s_ion[1][oq] = __fma_rn(v2, F2, __fma_rn(v1, F1, __dmul_rn(v, F)));
      }
    }
    cluster.sync();
    if (warp < 4 && (warp >> 1) * 256 < n) {
      double f[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) f[k] = sums[k] ? *sums[k] : 0.0;
      tree256(f, n - (warp >> 1) * 256);
      if (lane == 0) s_blk[warp >> 1][warp & 1] = f[0];
    }
    __syncthreads();
    // the owners decide (their sub-partitions' FP64 pipes are theirs); the others learn of it
    // at the next barrier
    if (owner_warp) {
      FF = n > 256 ? s_blk[0][0] + s_blk[1][0] : s_blk[0][0];
      conv = below(FF, ftol);
      if (tid == 0) s_stop = conv || last;
    }
    if (owner_warp && !(conv || last)) {
      const double vF = n > 256 ? s_blk[0][1] + s_blk[1][1] : s_blk[0][1];
      const double scale = vF > 0.0 ? vF / FF : 0.0;
      v = __fma_rn(scale, __dmul_rn(mass, a), __dmul_rn(A.dt, a));
      const double d = A.dt * v;
      const double d1 = __shfl_down_sync(0xffffffffu, d, 1), e2 = __shfl_down_sync(0xffffffffu, d, 2);
      const double m = warp_max(own && oc == 0 ? square3(d, d1, e2) : 0.0);
      if (lane == 0) s_max[warp] = m;
    }
    cluster.sync();
    if (s_stop) break;
    if (owner_warp) {
      double m = maxima ? *maxima : 0.0;
      if (maxima2) {
        const double m2 = *maxima2;
        if (bits_of(m2) > bits_of(m)) m = m2;
      }
      const double s = move_scale(warp_max(m), dmax);
      x = __fma_rn(s, A.dt * v, x);
      v = s * v;
      if (own) {
        float h, l;
        split_hilo(x, h, l);
        s_pos[oc][oq] = h, s_pos[3 + oc][oq] = l;
      }
    }
    cluster.sync();
    if (tid < n) {
      float* d = sb + rpc_at(tid, 0);
      float f[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) f[c] = from[c * kMinOwnWarps * kMinOwnIons];
#pragma unroll
      for (int c = 0; c < 6; ++c) d[4 * c] = f[c];
    }
    __syncthreads();
  }
  if (own) {  // the state, and the pair stream the next launch starts from
    A.x[oc * (long long)n + ie] = x;
    A.v[oc * (long long)n + ie] = v;
    float h, l;
    split_hilo(x, h, l);
    reinterpret_cast<float*>(A.hi + ie)[oc] = h;
    reinterpret_cast<float*>(A.lo + ie)[oc] = l;
  }
  cluster.sync();  // nobody leaves while others read its shared memory
  if (rank == 0 && tid == 0) {
    A.res->iters += it;
    A.res->fnorm = sqrt(FF);
    A.res->converged = conv ? 1 : 0;
  }
}

static size_t minimize_cl_smem_bytes(int NPe, int JP) { return (7 * (size_t)NPe * JP + (size_t)NPe * (kMinT / 4)) * sizeof(float); }

size_t minimize_smem_bytes(int R, int NP, int JP) {
  return (7 * (size_t)NP * JP + 6 * (size_t)NP * R) * sizeof(float) + 6 * (size_t)R * sizeof(double);
}

// CTAs and ions per CTA for n ions in NP parts of JP entries, whose step form has R ions per
// CTA.  False where the launch does not fit.
bool minimize_shape(long long n, int R, int NP, int JP, int sms, int* ctas, int* ions, bool* cluster) {
  if (n > 256LL * kMinMaxBlocks) return false;
  if (n <= kMinClusterN && JP <= kSeg) {
    *ctas = n < 32 ? 1 : n < 64 ? 4 : n < 128 ? 8 : 16;
    *ions = (int)((n + *ctas - 1) / *ctas);
    *cluster = true;
    const size_t smem = minimize_cl_smem_bytes((int)((n + JP - 1) / JP), JP);
    for (const void* fn : {(const void*)k_minimize_cl<true>, (const void*)k_minimize_cl<false>}) {
      if (smem > 200 * 1024 ||
          cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess ||
          cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return false;
    }
    return true;
  }
  *cluster = false;
  *ions = R;
  *ctas = (int)((n + R - 1) / R);
  const size_t smem = minimize_smem_bytes(R, NP, JP);
  if (smem > 224 * 1024 || 3 * R > kMinT) return false;
  const void* fn = (const void*)k_minimize_rp;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024) != cudaSuccess) return false;
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kMinT, smem) != cudaSuccess) return false;
  return per * sms >= *ctas;
}

// Scratch: the result, the ions' sums, the CTAs' displacements, the counter.
size_t minimize_scratch_bytes(long long n, int ctas) { return 256 + (size_t)n * sizeof(double2) + (size_t)ctas * sizeof(double); }

// Enqueue up to iters iterations from the handle's x and v (pair stream b); final_eval: then
// |F| at the last positions.
cudaError_t launch_minimize(const StepArgs& s, void* scratch, bool cluster, int ctas, int ions, int NP, int JP,
                            double dt, double dmax, double ftol, long long iters, int final_eval, int b,
                            cudaStream_t st) {
  MinRpArgs A{};
  char* p = static_cast<char*>(scratch);
  A.n = s.n, A.x = s.x, A.v = s.v, A.sp = s.sp, A.hi = s.hi[b], A.lo = s.lo[b], A.err = s.err;
  A.res = reinterpret_cast<MinResult*>(p);
  A.sync = reinterpret_cast<unsigned*>(p + 128);
  A.ion = reinterpret_cast<double2*>(p + 256);
  A.dmax = reinterpret_cast<double*>(p + 256 + (size_t)s.n * sizeof(double2));
  A.dt = dt, A.dmaxlim = dmax, A.ftol = ftol, A.iters = iters, A.final_eval = final_eval;
  A.R = ions, A.NP = NP, A.JP = JP, A.unitw = s.unitw;
  A.limit = s.wait_ns ? s.wait_ns : kWaitLimitNs;
  A.stall_cta = s.stall_cta, A.stall_at = s.stall_on ? s.stall_step : -1;
  A.trap = s.trap;
  for (int k = 0; k < IONTRAP_MAX_SPECIES; ++k) A.spc[k] = s.spc[k];
  cudaError_t e = cudaMemsetAsync(A.sync, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(kMinT);
  cfg.dynamicSmemBytes = cluster ? minimize_cl_smem_bytes((int)((s.n + JP - 1) / JP), JP) : minimize_smem_bytes(ions, NP, JP);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  if (cluster) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (!cluster) return cudaLaunchKernelEx(&cfg, k_minimize_rp, A);
  return cudaLaunchKernelEx(&cfg, A.unitw ? k_minimize_cl<true> : k_minimize_cl<false>, A);
}

}  // namespace it
