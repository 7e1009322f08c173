// tagged_step.cu -- row-persistent steps whose positions carry their own arrival.
//
// In the row-persistent form (fused = 5, persistent.cu) a step ends with every CTA counting
// itself on one counter, after its stores are visible, and begins with a poll of the counter
// and the copies of all positions: four trips to L2, one after the other.  Here an ion's next
// position goes out as two 16-byte entries (three floats and the step's tag, written and read
// in one access each), and the other CTAs read the entries until the tag is the one they wait
// for: a store and a load are the whole handover, and what has arrived is stored to shared
// memory while the rest is awaited.  Two buffers alternate: who writes tag t + 2 has read all of
// t + 1, whose writers had read all of t.
//
// What bounds a step (n = 1000, GB300, us: 3.88 before, 3.0 now): the handover, 0.9 from the last
// store to the last arrival, of which the 32 n bytes that each of the G CTAs reads from L2 are
// half (0.7 at n = 500, 1.25 at 2047); the pairs 1.0; the merge of the parts 0.35 (a Kahan
// addition is a chain of four); the FP64 update and its stores 0.4.  Everything else is off the
// chain:
//   owner warps    (3 R threads) pairs as all the others, then merge and integrate; trap, drag,
//                  laser and kick of the next step while the entries fly.  The conversions
//                  between float and double run at the FP64 rate and are done with integers
//   other warps    pairs; the next step's normals while the owners merge; then the entries.
//                  They begin only when their own CTA has published: reading before that
//                  delayed the others' stores (n = 1000: 3.37 -> 3.20 us, 1500: 3.78 -> 3.63)
// Entries hold an ion's two halves side by side, 32 bytes: with the halves apart two CTAs' ions
// shared a sector whenever R was odd (n = 1000, R = 7: 3.68 -> 3.37).
//
// us per step (5 handles, K = 1000 steps a launch, this kernel / the counter and bulk copies;
// below 432 ions / one cluster): n = 150: 2.01 / 1.92, 176: 2.02 / 2.04, 224: 2.16 / 2.31, 321:
// 2.53 / 3.27, 432: 2.24 / 3.26, 500: 2.30 / 3.50, 800: 2.5 / 3.86, 1000: 3.0 / 3.89, 1500:
// 3.54 / 4.39, 2047: 5.08 / 5.64.  With 16 warps a CTA (n > 2047) there was no gain: 2500: 7.70 /
// 7.53, 3000: 8.5 / 8.6.
//
// The bits are those of persistent.cu's kernel for the same (n, NP, JP): the same part sums
// (rp_chunk), the same merge order, the same FP64 operations.  Parts without ions, whose sums
// are zero, are left out, and zeros fill the merge's last group: adding zeros only moves the
// sum's low bits between its two halves, whose difference is the same.
#include "iontrap_internal.cuh"

namespace it {

constexpr int kTagBarOwners = 1, kTagBarPublished = 2, kTagBarNoise = 3;  // named barriers
constexpr int kTagThreads = 256, kTagMinN = 168, kTagMaxN = 2176;
constexpr int kTagHeader = 128;  // bytes before the entries: the tag of the last published step

// Part sums: rows of kTagRow floats, kTagBatch rows read ahead of the ones being merged (rows
// past the last part hold zeros).
constexpr int kTagRow = 128, kTagBatch = 4;
__host__ __device__ constexpr int tag_rows(int NP) { return (NP + kTagBatch - 1) / kTagBatch * kTagBatch; }

struct TagArgs {
  unsigned* sync;   // arrivals at the launch's end (zero between launches)
  unsigned* tags;   // last tag; entries at tags + kTagHeader bytes: [2 buffers][n][hi, lo] of 16 bytes
  long long K;      // steps in this launch
  int R;            // ions per CTA
  int NP;           // j-parts that hold an ion: ceil(n / JP)
  int JP;           // j entries per part
  unsigned magic;   // floor(2^32 / JP) + 1: e / JP = umulhi(e, magic) for e < n
};

// 16 bytes in one access: a reader sees all of an entry or nothing of it.
__device__ __forceinline__ void st_entry(void* p, float x, float y, float z, unsigned tag) {
  const unsigned long long a = (unsigned long long)__float_as_uint(y) << 32 | __float_as_uint(x);
  const unsigned long long b = (unsigned long long)tag << 32 | __float_as_uint(z);
  asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "l"(a), "l"(b)
               : "memory");
}
__device__ __forceinline__ uint4 ld_entry(const void* p) {
  unsigned long long a, b;
  asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
  return make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Given up on a wait: the limit has passed, or another thread has given up.
__device__ __forceinline__ unsigned long long tag_limit(const StepArgs& A) { return A.wait_ns ? A.wait_ns : kWaitLimitNs; }
static __device__ __noinline__ bool tag_late(unsigned long long& t0, const StepArgs& A) {
  if (*(volatile int*)A.err & ERR_TIMEOUT) return true;
  const unsigned long long now = globaltimer_ns();
  if (!t0) t0 = now;
  if (now - t0 <= tag_limit(A)) return false;
  atomicOr(A.err, ERR_TIMEOUT);
  return true;
}

// Items first, first + stride, ... of the entries (item m: half m & 1 of ion m / 2; the half is
// the thread's own, stride being even), into the part-major arrays at dst as each arrives.  U
// reads are in flight.  False if the wait was given up.
template <int U>
static __device__ __forceinline__ bool tag_fetch(const uint4* src, int items, int first, int stride, unsigned tag,
                                                 float* dst, int JP, unsigned magic, const StepArgs& A) {
  unsigned long long late = 0;
  unsigned it = 0;
  for (int m0 = first; m0 < items; m0 += U * stride) {
    unsigned pend = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) pend |= (m0 + u * stride < items ? 1u : 0u) << u;
    for (;;) {
      uint4 a[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (pend >> u & 1u) a[u] = ld_entry(src + m0 + u * stride);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if ((pend >> u & 1u) && a[u].w == tag) {
          pend &= ~(1u << u);
          const int e = (m0 + u * stride) >> 1;
          float* d = dst + e + 6 * JP * (int)__umulhi((unsigned)e, magic);
          d[0] = __uint_as_float(a[u].x), d[JP] = __uint_as_float(a[u].y), d[2 * JP] = __uint_as_float(a[u].z);
        }
      if (!pend) break;
      if ((++it & 63u) == 0 && tag_late(late, A)) return false;
    }
  }
  return true;
}

template <int IPT, int U>
__global__ void __launch_bounds__(kTagThreads, 1) k_step_f32_tag(const __grid_constant__ StepArgs A, const TagArgs P) {
  extern __shared__ __align__(16) float4 s_dyn[];
  const int tid = threadIdx.x;
  const int n = (int)A.n;
  const int R = P.R, NP = P.NP, JP = P.JP, K = (int)P.K;
  const int r0 = (int)blockIdx.x * R;
  const int Rg = min(R, n - r0);
  float* sall = reinterpret_cast<float*>(s_dyn);
  float* ps = sall + (size_t)NP * 7 * JP;
  float* sself = ps + tag_rows(NP) * kTagRow;
  float* szz = sself + 6 * R;
  double* scos = reinterpret_cast<double*>(szz + 3 * R + (R & 1));
  double* svd = scos + K;
  const TrapDev& tp = A.trap;
  const long long ns0 = *A.step;
  const unsigned tag0 = *(volatile unsigned*)P.tags;
  uint4* const ent = reinterpret_cast<uint4*>(reinterpret_cast<char*>(P.tags) + kTagHeader);
  const bool rf = !(tp.flags & (IONTRAP_RF_OFF | IONTRAP_TRAP_OFF | IONTRAP_PSEUDO));
  // the step after which a CTA that the failure test stalls publishes nothing
  const int stall_t = A.stall_on && (int)blockIdx.x == A.stall_cta && A.stall_step < K ? (int)A.stall_step : -1;
  for (int k = tid; k < K; k += kTagThreads) scos[k] = rf ? cos(tp.Omega * ((double)(ns0 + k + 1) * tp.dt)) : 0.0;

  // pair work: ion slot (slots slot and slot + RT with two ions per thread) and j-part
  const int RT = (R + IPT - 1) / IPT;
  const int part = tid / RT, slot = tid - part * RT;
  const bool works = part < NP;
  const int ii = r0 + slot, ib = r0 + slot + RT;
  const int jc = part * JP;
  // the self pair can only sit in a part that overlaps the CTA's own ions; the loop's variant
  // is chosen per warp (its lanes may belong to several parts)
  const bool diag = __any_sync(0xffffffffu, works && jc < r0 + Rg && r0 < jc + JP);
  // owned items: thread k < 3 Rg integrates component k / Rg of ion r0 + k % Rg
  const int oc = tid / Rg, oq = tid - oc * Rg;
  const bool own = tid < 3 * Rg;
  const int ow = 32 * ((3 * Rg + 31) / 32);  // threads of the owner warps; the others fetch
  const long long ie = r0 + oq;
  const SpeciesDev& sd = A.spc[own ? A.sp[ie] : 0];
  double xf = 0.0, vd = 0.0, ext = 0.0;
  const double ngamma = -sd.gamma, sigma = sd.sigma, coul = sd.coul;
  if (own) {
    vd = half_kick(A.v[oc * A.n + ie], A.a[oc * A.n + ie], tp.hdt);
    xf = drift(A.x[oc * A.n + ie], vd, tp.dt);
  }
  // the normals of an owned ion: by a thread of the other warps, in shared memory
  const int nq = tid - ow, nw = 32 * ((Rg + 31) / 32);
  const bool noisy = nq >= 0 && nq < Rg && A.spc[A.sp[r0 + nq]].sigma > 0.0;
  auto draw = [&](long long counter) {
    if (noisy) {
      float zz[3];
      normals3_f32(tp.seed, counter, r0 + nq, zz);
#pragma unroll
      for (int d = 0; d < 3; ++d) szz[d * R + nq] = zz[d];
    }
    if (nq < nw) bar_arrive(kTagBarNoise, ow + nw);
  };
  // force-independent terms of step t (the operations and order of accel_ext): trap and drag,
  // laser (all three components of an ion's velocity), kick
  auto ext_of = [&](int t) {
    if (own) ext = __fma_rn(ngamma, vd, __dmul_rn(-trap_spring_c(tp, sd, scos[t], oc), xf));
    if (tp.laser) {
      if (own) svd[oc * Rg + oq] = vd;
      bar_sync(kTagBarOwners, ow);
      if (own && sd.lrate != 0.0) {
        const double v3[3] = {svd[oq], svd[Rg + oq], svd[2 * Rg + oq]};
        ext = __fma_rn(-laser_proj(sd, v3), sd.kdir[oc], ext);
      }
    }
    bar_sync(kTagBarNoise, ow + nw);
    if (own && sigma > 0.0) ext = __fma_rn(sigma, widen(szz[oc * R + oq]), ext);
  };
  for (int k = NP * kTagRow + tid; k < tag_rows(NP) * kTagRow; k += kTagThreads) ps[k] = 0.f;
  {  // the launch's first positions and the charges, from the pair stream
    const int rb = (int)((ns0 + 1) & 1);
    const float4* __restrict__ ghi = A.hi[rb];
    const float4* __restrict__ glo = A.lo[rb];
    for (int e = tid; e < NP * JP; e += kTagThreads) {
      float4 h = make_float4(1e30f, 1e30f, 1e30f, 0.0f), l = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < n) {
        h = __ldcg(ghi + e);
        l = __ldcg(glo + e);
      }
      float* d = sall + e + 6 * JP * (e / JP);
      d[0] = h.x, d[JP] = h.y, d[2 * JP] = h.z;
      d[3 * JP] = l.x, d[4 * JP] = l.y, d[5 * JP] = l.z;
      d[6 * JP] = h.w;
      if (e >= r0 && e < r0 + Rg) {
        float* s = sself + (e - r0);
        s[0] = h.x, s[R] = h.y, s[2 * R] = h.z, s[3 * R] = l.x, s[4 * R] = l.y, s[5 * R] = l.z;
      }
    }
  }
  __syncthreads();
  if (tid >= ow)
    draw(ns0 + 1);
  else
    ext_of(0);

  bool bad = false;
  for (int t = 0; t < K; ++t) {
    if (t > 0 && tid >= ow) {  // positions x_{ns + 1} of every ion
      const unsigned tag = tag0 + (unsigned)t;
      const uint4* src = ent + (size_t)(tag & 1) * 2 * n;
      const int PT = kTagThreads - ow, half = tid & 1;
      float* const base = sall + 3 * half * JP;
      bar_sync(kTagBarPublished, kTagThreads);
      bad = !tag_fetch<U>(src, 2 * n, tid - ow, PT, tag, base, JP, P.magic, A);
    }
    if (__syncthreads_or(bad)) {
      bad = true;
      break;
    }
    // optional phase timestamps (iontrap_trace_step): 4 per CTA and step
    const long long tslot = ((long long)blockIdx.x * K + t) * 4;
    trace_mark(A.trace, tslot + 0);
    trace_mark(A.trace, tslot + 1);
    if (works) {
      float2 nh[IPT][3], nl[IPT][3], acc[IPT][3];
#pragma unroll
      for (int k = 0; k < IPT; ++k) {
        const int s = slot + k * RT;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float h = s < Rg ? -sself[d * R + s] : 0.f, l = s < Rg ? -sself[(3 + d) * R + s] : 0.f;
          nh[k][d] = make_float2(h, h), nl[k][d] = make_float2(l, l);
          acc[k][d] = make_float2(0.f, 0.f);
        }
      }
      const float* sj = sall + (size_t)part * 7 * JP;
      if constexpr (IPT == 1) {
        if (A.unitw) {
          if (diag)
            rp_chunk<true, true, 4>(sj, sj + 6 * JP, JP, JP, jc, ii, nh[0], nl[0], acc[0]);
          else
            rp_chunk<false, true, 4>(sj, sj + 6 * JP, JP, JP, jc, ii, nh[0], nl[0], acc[0]);
        } else {
          if (diag)
            rp_chunk<true, false, 4>(sj, sj + 6 * JP, JP, JP, jc, ii, nh[0], nl[0], acc[0]);
          else
            rp_chunk<false, false, 4>(sj, sj + 6 * JP, JP, JP, jc, ii, nh[0], nl[0], acc[0]);
        }
      } else {
        if (A.unitw) {
          if (diag)
            rp_chunk_i2<true, true>(sj, sj + 6 * JP, JP, JP, jc, ii, ib, nh, nl, acc);
          else
            rp_chunk_i2<false, true>(sj, sj + 6 * JP, JP, JP, jc, ii, ib, nh, nl, acc);
        } else {
          if (diag)
            rp_chunk_i2<true, false>(sj, sj + 6 * JP, JP, JP, jc, ii, ib, nh, nl, acc);
          else
            rp_chunk_i2<false, false>(sj, sj + 6 * JP, JP, JP, jc, ii, ib, nh, nl, acc);
        }
      }
#pragma unroll
      for (int k = 0; k < IPT; ++k)
        if (slot + k * RT < R)
#pragma unroll
          for (int d = 0; d < 3; ++d) ps[part * kTagRow + d * R + slot + k * RT] = acc[k][d].x + acc[k][d].y;
    }
    __syncthreads();
    trace_mark(A.trace, tslot + 2);

    if (tid >= ow) {
      if (t + 1 < K) draw(ns0 + t + 2);  // the next step's normals, while the owners merge
    } else {  // merge in part order (Kahan; a part is one chunk: no compensation), finish the step
      if (own) {
        float su = 0.f, cu = 0.f;
        const float* q = ps + oc * R + oq;
        float v[kTagBatch];
#pragma unroll
        for (int k = 0; k < kTagBatch; ++k) v[k] = q[k * kTagRow];
#pragma unroll 1
        for (int p = kTagBatch;; p += kTagBatch) {
          float nx[kTagBatch];
          if (p < NP) {
            q += kTagBatch * kTagRow;
#pragma unroll
            for (int k = 0; k < kTagBatch; ++k) nx[k] = q[k * kTagRow];
          }
#pragma unroll
          for (int k = 0; k < kTagBatch; ++k) {
            const float y = v[k] - cu;
            const float tt = su + y;
            cu = (tt - su) - y;
            su = tt;
          }
          if (p >= NP) break;
#pragma unroll
          for (int k = 0; k < kTagBatch; ++k) v[k] = nx[k];
        }
        const double Sd = widen(cu) - widen(su);
        const double acc = __fma_rn(coul, Sd, ext);
        const double vn = half_kick(vd, acc, tp.hdt);
        const double vh = half_kick(vn, acc, tp.hdt);
        const double xn = drift(xf, vh, tp.dt);
        float h, l;
        split_hilo(xn, h, l);
        if (t + 1 == K) {  // the launch's last step: FP64 state and the pair stream
          const int wb = (int)((ns0 + t) & 1);
          A.x[oc * A.n + ie] = xf;
          A.v[oc * A.n + ie] = vn;
          A.a[oc * A.n + ie] = acc;
          reinterpret_cast<float*>(A.hi[wb] + ie)[oc] = h;
          reinterpret_cast<float*>(A.lo[wb] + ie)[oc] = l;
          if (oc == 0) {
            reinterpret_cast<float*>(A.hi[wb] + ie)[3] = sd.w;
            reinterpret_cast<float*>(A.lo[wb] + ie)[3] = 0.0f;
          }
        } else {
          sself[oc * R + oq] = h;
          sself[(3 + oc) * R + oq] = l;
        }
        // a non-finite acceleration or velocity reaches xn = xf + dt (vn + dt/2 acc)
        if ((((unsigned)__double2hiint(xn) >> 20) & 0x7ffu) == 0x7ffu) atomicOr(A.err, ERR_NONFINITE);
        vd = vh;
        xf = xn;
      }
      if (t + 1 < K) {
        bar_sync(kTagBarOwners, ow);
        if (tid < 2 * Rg && t != stall_t) {  // publish: half hf of ion q
          const int q = tid >> 1, hf = tid & 1;
          const unsigned tag = tag0 + (unsigned)t + 1u;
          const float* s = sself + 3 * hf * R + q;
          st_entry(ent + 2 * ((size_t)(tag & 1) * n + r0) + tid, s[0], s[R], s[2 * R], tag);
        }
        bar_arrive(kTagBarPublished, kTagThreads);
        ext_of(t + 1);  // while the other CTAs finish
      }
    }
    trace_mark(A.trace, tslot + 3);
  }

  // Once every CTA has read its last positions: clear the counter, advance the step index
  // and the tag.  A launch that gave up on a wait leaves all three alone, and the handle's sticky
  // timeout status retires them.  Its FP64 state is still the one it started from, unless the wait
  // was for the launch's last step: CTAs that received its positions have written theirs.
  __syncthreads();
  if (tid == 0) {
    if (!bad && stall_t != K - 1) arrive_release(P.sync);
    if (blockIdx.x == 0 && poll_wait<true>(P.sync, gridDim.x, A.err, tag_limit(A))) {
      *P.sync = 0u;
      *P.tags = tag0 + (unsigned)(K - 1);
      *A.step = ns0 + K;
      __threadfence();
    }
  }
}

size_t tag_smem_bytes(int R, int NP, int JP, long long K) {
  return ((size_t)NP * 7 * JP + (size_t)tag_rows(NP) * kTagRow + 9 * (size_t)R + 1) * sizeof(float) +
         ((size_t)K + 3 * (size_t)R) * sizeof(double);
}

// Bytes of the entries of n ions, or 0 above the size this form takes.
size_t tag_bytes(long long n) { return n <= kTagMaxN ? kTagHeader + 64 * (size_t)n : 0; }

const void* tag_kernel(int I, int U) {
  if (I == 1)
    return U <= 8 ? (const void*)k_step_f32_tag<1, 8>
                  : U <= 16 ? (const void*)k_step_f32_tag<1, 16> : (const void*)k_step_f32_tag<1, 24>;
  return U <= 8 ? (const void*)k_step_f32_tag<2, 8>
                : U <= 16 ? (const void*)k_step_f32_tag<2, 16> : (const void*)k_step_f32_tag<2, 24>;
}

// Whether a row-persistent shape is stepped here: CTAs of 8 warps (the default below 2048 ions;
// above, the reads outweigh the handover), parts of one chunk, one CTA per SM at most (the
// kernel's registers), half the warps free to fetch; and above kTagMinN ions where the shape
// could run on one cluster (figures above).
bool tag_takes(long long n, int W, int R, int JP, int G, int sms, bool cluster) {
  return n > (cluster ? kTagMinN : 0) && n <= kTagMaxN && 32 * W == kTagThreads && JP <= kSeg && G > 1 && G <= sms &&
         6 * R <= kTagThreads;
}

cudaError_t launch_tag(const StepArgs& a, unsigned* sync, unsigned* tags, int R, int JP, int I, int G,
                       long long K, cudaStream_t st) {
  const int fetchers = kTagThreads - 32 * ((3 * R + 31) / 32);
  // reads in flight per thread: what it takes to fetch all entries in one go, as far as the
  // registers allow (n = 500: 2.44 with 16, 2.29 with 8; 1000: 3.09 and 3.43; 2047: 5.68 with 16,
  // 5.40 with 24)
  const void* fn = tag_kernel(I, (int)((2 * a.n + fetchers - 1) / fetchers));
  TagArgs P{sync, tags, K, R, (int)((a.n + JP - 1) / JP), JP, (unsigned)((1ull << 32) / (unsigned)JP) + 1u};
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)G);
  cfg.blockDim = dim3((unsigned)(kTagThreads));
  cfg.dynamicSmemBytes = tag_smem_bytes(R, P.NP, JP, K);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  StepArgs ac = a;
  void* params[] = {&ac, &P};
  return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace it
