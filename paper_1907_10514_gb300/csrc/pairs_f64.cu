// pairs_f64.cu -- the plain FP64 form (IONTRAP_PREC_FP64): every unordered pair once.
//
// The FP64 pipe bounds this form (GB300: a warp instruction occupies its sub-partition's pipe
// for ~76 cycles), so it is designed to issue few FP64 instructions and lets everything else
// ride along.  A warp holds a row block of 32 I ions, I per lane, and takes the columns in
// blocks of 32: at rotation k lane l meets column (l + k) % 32, adds the pair to its own ions'
// sums and subtracts it from the column's, whose three sums move on to the next lane by
// shuffles (Newton's third law).  A pair costs 16 FP64 instructions for both its ions
// instead of 2 x 19:
//   3 differences, 3 for r^2, 4 for r^-3, 6 to accumulate.
// r^-3: y = the hardware's 21-bit r^-1 approximation; y^2, whose 42 bits fit a double, by
// integer instructions; e = 1 - r^2 y^2; r^-3 = y^2 y (1 - e)^(-3/2) with the series to e^2
// (|e| < 2^-19 measured, the next term is 35/16 e^3 < 2^-55),
// its e^2 term in FP32.
//
// The triangle of (row block, column block, rotation) is one line of equal units, cut evenly
// over all warps of the GPU by a table the host lays out once per handle (above 16384 ions one per
// band of kF64BandRows row blocks, each summed and folded into three sums per ion before the next:
// the column slots would grow with n^2 and now take 1.5 KB an ion).  The force-independent
// terms that are long FP64 chains (logarithm and square root of the noise, its sine and cosine,
// cos(Omega t)) are units of the same line, so that they run beside the pairs.  Sums go to fixed
// slots; k_finish_f64 adds an ion's slots in a fixed order, and integrates after the last band.  The
// result is a function of n, the SM count and the inputs only.
//
// Measured on GB300 (us per step, the form that summed every ordered pair with rsqrt(double)
// against this one): n = 64: 19.3 -> 11.9, 321: 26.1 -> 16.4, 1000: 53.4 -> 29.3, 2500:
// 216 -> 107, 4096: 534 -> 263, which is 95% of the FP64 pipe's rate.  r^-3 is within 2.3e-16
// of the exact value over 2^21 draws of r^2 (the cube of rsqrt(double): 5.4e-16).
#include <algorithm>
#include <cstring>
#include <vector>

#include "iontrap_internal.cuh"

namespace it {

// One warp's share of the line: where its pair units begin and how many there are, and its
// noise units.  A unit is one rotation of one (row block, column block) tile.
struct F64Share {
  int a, c, k;     // first row block, column block, rotation
  int tile;        // slot of that tile's column sums; the line's next tile has the next slot
  int units;       // rotations taken, crossing tiles and rows
  int flush;       // slot of the first row block's sums; the next row block's is flush + 1
  int first_main;  // the first tile is begun here (its column sums go to the main slot)
  int noise, nnoise;  // first noise unit and their number
};

struct F64Band {
  int row0 = 0, rows = 0, flushes = 0;
  std::vector<F64Share> share;
  std::vector<int> row_flush;  // [rows + 1]: slots of a row block
  std::vector<int> col_extra;  // [cols + 1]: warps that continue a tile of a column block, below
  std::vector<int> extra;      // their numbers
};

// Device view: a band's tables, and the slots, in the handle's scratch.
struct F64Args {
  const F64Share* share;
  const int* row_flush;
  const int* col_extra;
  const int* extra;
  double* row_sum;   // [flushes][I][3][32]
  double* col_sum;   // [tiles][3][32]: main column sums, the tiles of a row block side by side
  double* ext_sum;   // [warps][3][32]: column sums of continued tiles
  double* noise;     // [5][n16]: r1, r2, cos 1, sin 1, cos 2 (n16: n rounded up to 16)
  double* springs;   // [species][3] at the force time
  double* fold;      // [3][32 cols]: the sums of the bands before
  int row0, rows;    // the band's row blocks
  int cols, warps, nspecies, bath;
  int first, last;   // of the bands
};

// The tile (row block row0 + r of I sub-blocks, column block c) of a band: row block r has
// cols - (row0 + r) I of them.
__host__ __device__ __forceinline__ int f64_tile_slot(int row0, int r, int I, int cols, int c) {
  return r * (cols - row0 * I) - I * (r * (r - 1) / 2) + c - (row0 + r) * I;
}

constexpr int kF64Threads = 128;
constexpr int kF64NoiseIons = 16;  // ions of a noise unit (32 lanes: two numbers each)

// Rotations k0 <= k < k1 of one tile.  Row sub-block s starts at ion 32 (a I + s); the column
// block is col.  d = col - a I: the sub-block s < d meets every column, s == d is the block
// itself (rotations 1 .. 16, the last one by half of the lanes), s > d was met before as a
// column.  cj: x, y, z (and charge) of the columns, twice in a row.
template <int I, bool UNITW>
__device__ __forceinline__ void f64_tile(const double* cj, int lane, int d, int k0, int k1, const double (&xi)[I][3],
                                         const double (&zi)[I], double (&ai)[I][3], double (&aj)[3]) {
  for (int k = k0; k < k1; ++k) {
    const double xj = cj[lane + k], yj = cj[64 + lane + k], zj = cj[128 + lane + k];
    const double wj = UNITW ? 1.0 : cj[192 + lane + k];
#pragma unroll
    for (int s = 0; s < I; ++s) {
      if (s > d) break;
      const bool met = s < d || (k >= 1 && k <= 16);
      if (!met) continue;
      const bool on = s < d || k < 16 || lane < 16;
      const double dx = xi[s][0] - xj, dy = xi[s][1] - yj, dz = xi[s][2] - zj;
      double g = inv_cube(__fma_rn(dx, dx, __fma_rn(dy, dy, dz * dz)));
      if (!on) g = 0.0;
      const double gi = UNITW ? g : g * wj, gj = UNITW ? -g : -(g * zi[s]);
      ai[s][0] = __fma_rn(gi, dx, ai[s][0]);
      ai[s][1] = __fma_rn(gi, dy, ai[s][1]);
      ai[s][2] = __fma_rn(gi, dz, ai[s][2]);
      aj[0] = __fma_rn(gj, dx, aj[0]);
      aj[1] = __fma_rn(gj, dy, aj[1]);
      aj[2] = __fma_rn(gj, dz, aj[2]);
    }
    // the columns' sums move on with their columns
#pragma unroll
    for (int c = 0; c < 3; ++c) aj[c] = __shfl_sync(0xffffffffu, aj[c], (lane + 1) & 31);
  }
}

// Noise unit: the two logarithms or the two angles of 16 ions (the operations of normals3_f64,
// one per lane).  Units [0, m): logarithms, [m, 2 m): angles; 2 m: cos(Omega t) and the springs.
__device__ __forceinline__ void f64_noise(const StepArgs& A, const F64Args& F, long long ns, int u, int lane) {
  const int m = (int)((A.n + kF64NoiseIons - 1) / kF64NoiseIons);
  const long long n16 = (long long)m * kF64NoiseIons;
  const long long nf = A.mode == MODE_STEP ? ns + 1 : ns;
  if (u == 2 * m) {
    const double cosv = force_time_cos(A, ns);
    for (int s = lane; s < F.nspecies; s += 32) trap_springs(A.trap, A.spc[s], cosv, F.springs + 3 * s);
    return;
  }
  if (!F.bath) return;
  const bool angles = u >= m;
  const long long i = (long long)(angles ? u - m : u) * kF64NoiseIons + (lane >> 1);
  if (i >= A.n) return;
  const int q = lane & 1;
  unsigned long long c[4] = {(unsigned long long)nf, (unsigned long long)i, 0ull, 0ull};
  philox4x64_10(c, A.trap.seed, 0ull);
  const unsigned long long b = angles ? (q ? c[3] : c[1]) : (q ? c[2] : c[0]);
  const double v = ((double)(b >> 41) + 0.5) * 0x1p-23;
  if (!angles) {
    F.noise[q * n16 + i] = sqrt(-2.0 * log(v));
  } else {
    double s1, c1;
    sincospi(2.0 * v, &s1, &c1);
    F.noise[(q ? 4 : 2) * n16 + i] = c1;
    if (!q) F.noise[3 * n16 + i] = s1;
  }
}

template <int I, bool UNITW>
__global__ void __launch_bounds__(kF64Threads) k_pairs_f64(const __grid_constant__ StepArgs A, const __grid_constant__ F64Args F) {
  __shared__ double s_cj[kF64Threads / 32][4][64];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const int w = blockIdx.x * (kF64Threads / 32) + wl;
  if (w >= F.warps) return;
  const long long n = A.n, ns = *A.step;
  const F64Share sh = F.share[w];
  if (A.mode != MODE_FORCES)
    for (int u = 0; u < sh.nnoise; ++u) f64_noise(A, F, ns, sh.noise + u, lane);
  const double4_32a* __restrict__ pos = A.p64[(A.mode == MODE_STEP) ? (int)((ns + 1) & 1) : (int)(ns & 1)];
  // ions past n sit far away: r^-3 underflows to zero
  auto load = [&](long long i) { return i < n ? pos[i] : make_double4_32a(1e150, 1e150, 1e150, 0.0); };
  double* cj = &s_cj[wl][0][0];
  int a = sh.a, c = sh.c, k = sh.k, tile = sh.tile, flush = sh.flush;
  int left = (A.trap.flags & IONTRAP_COULOMB_OFF) ? 0 : sh.units;
  bool main = sh.first_main != 0;
  double xi[I][3], zi[I], ai[I][3];
  bool fresh = true;
  while (left > 0) {
    if (fresh) {
#pragma unroll
      for (int s = 0; s < I; ++s) {
        const double4_32a p = load(32LL * (a * I + s) + lane);
        xi[s][0] = p.x, xi[s][1] = p.y, xi[s][2] = p.z, zi[s] = p.w;
        ai[s][0] = ai[s][1] = ai[s][2] = 0.0;
      }
      fresh = false;
    }
    {
      const double4_32a p = load(32LL * c + lane);
      __syncwarp();
      cj[lane] = cj[lane + 32] = p.x, cj[64 + lane] = cj[96 + lane] = p.y, cj[128 + lane] = cj[160 + lane] = p.z;
      if (!UNITW) cj[192 + lane] = cj[224 + lane] = p.w;
      __syncwarp();
    }
    const int k1 = min(32, k + left);
    double aj[3] = {0.0, 0.0, 0.0};
    f64_tile<I, UNITW>(cj, lane, c - a * I, k, k1, xi, zi, ai, aj);
    left -= k1 - k;
    // lane l now holds the sums of column (l + k1) % 32
    const int col = (lane + k1) & 31;
    double* out = (main ? F.col_sum + 96LL * tile : F.ext_sum + 96LL * w) + col;
    ++tile;
#pragma unroll
    for (int q = 0; q < 3; ++q) __stcg(out + 32 * q, aj[q]);
    main = true;
    k = 0;
    if (++c == F.cols || left == 0) {
#pragma unroll
      for (int s = 0; s < I; ++s)
#pragma unroll
        for (int q = 0; q < 3; ++q) __stcg(F.row_sum + (((long long)flush * I + s) * 3 + q) * 32 + lane, ai[s][q]);
      ++flush;
      if (c == F.cols) ++a, c = a * I, fresh = true;
    }
  }
}

// An ion's sums over a band, and after the last one the rest of the step: a CTA per column block, kF64Slices warps per
// component, each adding every kF64Slices-th slot of a kind with eight loads in flight (the
// slots are ~60 at n = 4096: one warp's loads in turn would be the longest chain of the step).
constexpr int kF64Slices = 4;

template <int I>
__global__ void __launch_bounds__(96 * kF64Slices)
    k_finish_f64(const __grid_constant__ StepArgs A, const __grid_constant__ F64Args F) {
  __shared__ double s_v[3][32];
  __shared__ double s_sum[kF64Slices][3][32];
  const int lane = threadIdx.x & 31, q = (threadIdx.x >> 5) % 3, z = threadIdx.x / 96;
  const int c = blockIdx.x, a = c / I, r = a - F.row0;  // r: the block's row in the band, if there
  const long long n = A.n, i = 32LL * c + lane;
  const long long ns = *A.step;
  const bool on = i < n, step = A.mode == MODE_STEP;
  if (r < 0 && !F.last) return;
  if (!(A.trap.flags & IONTRAP_COULOMB_OFF)) {
    double S = 0.0;
    auto add = [&](auto slot, int m) {
      double t[4] = {0.0, 0.0, 0.0, 0.0};
      int u = z;
      for (; u + 7 * kF64Slices < m; u += 8 * kF64Slices) {
        double g[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) g[k] = __ldcg(slot(u + k * kF64Slices));
#pragma unroll
        for (int k = 0; k < 8; ++k) t[k & 3] += g[k];
      }
      double g[7];
#pragma unroll
      for (int k = 0; k < 7; ++k) g[k] = u + k * kF64Slices < m ? __ldcg(slot(u + k * kF64Slices)) : 0.0;
#pragma unroll
      for (int k = 0; k < 7; ++k) t[k & 3] += g[k];
      S += (t[0] + t[1]) + (t[2] + t[3]);
    };
    const bool row = r >= 0 && r < F.rows;
    const int f0 = row ? F.row_flush[r] : 0, e0 = F.col_extra[c];
    add([&](int u) { return F.row_sum + (((f0 + u) * (long long)I + (c - a * I)) * 3 + q) * 32 + lane; },
        row ? F.row_flush[r + 1] - f0 : 0);
    add([&](int u) { return F.col_sum + 96LL * f64_tile_slot(F.row0, u, I, F.cols, c) + 32 * q + lane; },
        max(0, min(r + 1, F.rows)));
    add([&](int u) { return F.ext_sum + 96LL * F.extra[e0 + u] + 32 * q + lane; }, F.col_extra[c + 1] - e0);
    s_sum[z][q][lane] = S;
  } else {
    s_sum[z][q][lane] = 0.0;
  }
  double* fold = F.fold + 32LL * F.cols * q + i;
  if (!F.last) {
    __syncthreads();
    if (z == 0) {
      double S = s_sum[0][q][lane];
#pragma unroll
      for (int k = 1; k < kF64Slices; ++k) S += s_sum[k][q][lane];
      __stcg(fold, F.first ? S : __ldcg(fold) + S);
    }
    return;
  }
  const SpeciesDev& sd = A.spc[on ? A.sp[i] : 0];
  double v = 0.0, vd = 0.0, xf = 0.0, ext = 0.0;
  if (on && z == 0 && A.mode != MODE_FORCES) {  // force-independent terms (the operations of accel_ext)
    const double x = A.x[q * n + i];
    v = A.v[q * n + i];
    const double vh = half_kick(v, A.a[q * n + i], A.trap.hdt);
    vd = step ? vh : v;
    xf = step ? drift(x, vh, A.trap.dt) : x;
    ext = __fma_rn(-sd.gamma, vd, __dmul_rn(-F.springs[3 * A.sp[i] + q], xf));
    s_v[q][lane] = vd;
  }
  __syncthreads();
  if (z == 0 && on) {
    double S = s_sum[0][q][lane];
#pragma unroll
    for (int k = 1; k < kF64Slices; ++k) S += s_sum[k][q][lane];
    if (!F.first) S += __ldcg(fold);
    if (A.mode == MODE_FORCES) {
      A.out[q * n + i] = sd.coul * S;
    } else {
      if (sd.lrate != 0.0) {
        const double v3[3] = {s_v[0][lane], s_v[1][lane], s_v[2][lane]};
        ext = __fma_rn(-laser_proj(sd, v3), sd.kdir[q], ext);
      }
      if (sd.sigma > 0.0) {
        const long long n16 = (n + kF64NoiseIons - 1) / kF64NoiseIons * kF64NoiseIons;
        const double r = F.noise[(q == 2 ? n16 : 0) + i], t = F.noise[(2 + q) * n16 + i];
        ext = __fma_rn(sd.sigma, r * t, ext);
      }
      const double acc = __fma_rn(sd.coul, S, ext);
      const double vn = step ? half_kick(vd, acc, A.trap.hdt) : v;
      const double xn = drift(xf, half_kick(vn, acc, A.trap.hdt), A.trap.dt);
      if (step) A.x[q * n + i] = xf, A.v[q * n + i] = vn;
      A.a[q * n + i] = acc;
      double* p = reinterpret_cast<double*>(A.p64[step ? (int)(ns & 1) : (int)((ns + 1) & 1)] + i);
      p[q] = xn;
      if (q == 0) p[3] = (double)sd.w;
      if (!(isfinite(acc) && isfinite(vn) && isfinite(xn))) atomicOr(A.err, ERR_NONFINITE);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(A.done, 1u);
    if (prev == gridDim.x - 1u) {
      *A.done = 0u;
      if (step) *A.step = ns + 1;
      __threadfence();
    }
  }
}

// ------------------------------------------------------------------ host side

// Ions per lane: row blocks of 32 I ions, so that an ion has few column slots (at most 64 up
// to 16384 ions) and small n still has rows to spread.
static int f64_rows(long long n) { return n <= 2048 ? 1 : n <= 4096 ? 2 : n <= 8192 ? 4 : 8; }

// The line: every tile (a, c >= a I) has 32 rotations; a rotation's cost is the sub-blocks
// that take part.  Warps: two per sub-partition (one already keeps the FP64 pipe 90% busy),
// fewer where that would leave a warp less than kF64MinCost (us per step with 2, 3, 4, 8:
// n = 64: 11.5 11.9 12.4 15.4; 321: 17.8 16.4 15.9 17.8; 1000: 29.3 29.3 29.3 29.3).
constexpr long long kF64NoiseCost = 5;  // of a noise unit, in rotations of one sub-block (16 FP64 instructions)
constexpr long long kF64MinCost = 3;
// Row blocks of a band: all of them up to 16384 ions.  A further band costs the end of its launch,
// where warps finish at different times, and the fold (all row blocks in one band / in bands, and
// the handle's memory: n = 32768: 15.09 / 15.13 ms per step, 116 / 53 MB; 100000: 140.1 / 140.4 ms,
// 967 / 171 MB).
constexpr int kF64BandRows = 64;

// The shape of n ions' bands; without the pair term there are noise units only.
struct F64Shape {
  int I, rows, cols, bands, units, warps;
  long long tile_cost(int d) const { return 32LL * std::min(d, I) + (d < I ? 16 : 0); }  // d: columns from its row block
  int band_rows(int b) const { return std::min(kF64BandRows, rows - b * kF64BandRows); }
  long long cost(int b) const {
    long long t = b == 0 ? kF64NoiseCost * units : 0;
    for (int a = b * kF64BandRows; a < b * kF64BandRows + band_rows(b); ++a)
      for (int c = a * I; c < cols; ++c) {
        const int d = c - a * I;
        if (d >= I) {
          t += tile_cost(d) * (cols - c);
          break;
        }
        t += tile_cost(d);
      }
    return t;
  }
};

static F64Shape f64_shape(long long n, int sms, bool coulomb) {
  F64Shape S{};
  S.I = f64_rows(n);
  S.cols = (int)((n + 31) / 32);
  S.rows = coulomb ? (S.cols + S.I - 1) / S.I : 0;
  S.bands = std::max(1, (S.rows + kF64BandRows - 1) / kF64BandRows);
  S.units = 2 * (int)((n + kF64NoiseIons - 1) / kF64NoiseIons) + 1;
  S.warps = (int)std::max<long long>(1, std::min<long long>(8LL * sms, S.cost(0) / kF64MinCost));
  return S;
}

static F64Band f64_band(const F64Shape& S, int b) {
  F64Band B;
  B.row0 = b * kF64BandRows, B.rows = S.band_rows(b);
  const int I = S.I, cols = S.cols, end_row = B.row0 + B.rows, units = b == 0 ? S.units : 0;
  // cost of rotation k of a tile at distance d = c - a I from its row block
  auto cost = [&](int d, int k) -> long long { return std::min(d, I) + (d < I && k >= 1 && k <= 16 ? 1 : 0); };
  const long long total = S.cost(b);
  B.share.resize(S.warps);
  B.row_flush.assign(B.rows + 1, 0);
  std::vector<std::vector<int>> extra(cols);
  int a = B.row0, c = a * I, k = 0;
  long long done = 0;
  int u = 0;
  for (int w = 0; w < S.warps; ++w) {
    // the cost line up to this warp's end; noise first (it is the longest chain)
    const long long end = total * (w + 1) / S.warps;
    F64Share& s = B.share[w];
    s.noise = u;
    while (u < units && done < end) ++u, done += kF64NoiseCost;
    s.nnoise = u - s.noise;
    s.a = a, s.c = c, s.k = k, s.tile = f64_tile_slot(B.row0, a - B.row0, I, cols, c), s.units = 0, s.flush = B.flushes, s.first_main = k == 0;
    const bool last = w + 1 == S.warps;
    if (a < end_row && (done < end || last) && k != 0) extra[c].push_back(w);
    bool open = false;
    while (a < end_row && (done < end || last)) {
      open = true;
      const int d = c - a * I;
      if (k == 0 && d >= I && !last && done + S.tile_cost(d) <= end) {  // whole tiles at once
        const long long m = std::min<long long>(cols - c, (end - done) / S.tile_cost(d));
        s.units += 32 * (int)m, done += m * S.tile_cost(d), k = 32, c += (int)m - 1;
      } else {
        ++s.units, done += cost(d, k), ++k;
      }
      if (k == 32) {
        k = 0;
        if (++c == cols) {
          ++B.flushes;
          open = false;
          ++a, c = a * I;
          B.row_flush[a - B.row0] = B.flushes;
        }
      }
    }
    if (open) ++B.flushes;
  }
  B.col_extra.assign(cols + 1, 0);
  for (int q = 0; q < cols; ++q) {
    for (int w : extra[q]) B.extra.push_back(w);
    B.col_extra[q + 1] = (int)B.extra.size();
  }
  return B;
}

// Scratch layout in bytes: the bands' tables, then the slots that they share.  Sizes follow from
// the shape: a warp leaves one row block's sums open at most and continues one tile.
struct F64Layout {
  size_t share, row_flush, col_extra, extra, band;  // a band's tables, and the bytes from one to the next
  size_t row_sum, col_sum, ext_sum, noise, springs, fold, bytes;
};

static F64Layout f64_layout(const F64Shape& S, long long n) {
  F64Layout L{};
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t p = at;
    at += (bytes + 255) / 256 * 256;
    return p;
  };
  const int rows = S.band_rows(0);
  const size_t tiles = rows ? (size_t)(f64_tile_slot(0, rows - 1, S.I, S.cols, S.cols - 1) + 1) : 0;
  L.share = take(S.warps * sizeof(F64Share));
  L.row_flush = take((rows + 1) * sizeof(int));
  L.col_extra = take((S.cols + 1) * sizeof(int));
  L.extra = take(S.warps * sizeof(int));
  L.band = at;
  at *= S.bands;
  const size_t warps = S.rows ? S.warps : 0;
  L.row_sum = take((warps + rows) * S.I * 96 * sizeof(double));
  L.col_sum = take(tiles * 96 * sizeof(double));
  L.ext_sum = take(warps * 96 * sizeof(double));
  L.noise = take(5 * (size_t)((n + 15) / 16 * 16) * sizeof(double));
  L.springs = take(3 * IONTRAP_MAX_SPECIES * sizeof(double));
  L.fold = take(S.bands > 1 ? 96 * (size_t)S.cols * sizeof(double) : 0);
  L.bytes = at;
  return L;
}

size_t f64_scratch_bytes(long long n, int sms, bool coulomb) {
  return f64_layout(f64_shape(n, sms, coulomb), n).bytes;
}

// Lay out a handle's scratch: its tables are written (synchronously, the host copy goes away)
// and *v is what the launches need.
cudaError_t f64_prepare(long long n, int sms, bool coulomb, void* scratch, cudaStream_t st, F64View* v) {
  const F64Shape S = f64_shape(n, sms, coulomb);
  const F64Layout L = f64_layout(S, n);
  v->base = scratch;
  v->I = S.I, v->rows = S.rows, v->cols = S.cols, v->warps = S.warps, v->bands = S.bands;
  const size_t off[10] = {L.share, L.row_flush, L.col_extra, L.extra, L.row_sum,
                          L.col_sum, L.ext_sum, L.noise, L.springs, L.fold};
  std::memcpy(v->off, off, sizeof(off));
  v->band_bytes = L.band;
  std::vector<unsigned char> h(L.band * S.bands);
  for (int b = 0; b < S.bands; ++b) {
    const F64Band B = f64_band(S, b);
    unsigned char* t = h.data() + L.band * b;
    std::memcpy(t + L.share, B.share.data(), B.share.size() * sizeof(F64Share));
    std::memcpy(t + L.row_flush, B.row_flush.data(), B.row_flush.size() * sizeof(int));
    std::memcpy(t + L.col_extra, B.col_extra.data(), B.col_extra.size() * sizeof(int));
    if (!B.extra.empty()) std::memcpy(t + L.extra, B.extra.data(), B.extra.size() * sizeof(int));
  }
  const cudaError_t e = cudaMemcpyAsync(scratch, h.data(), h.size(), cudaMemcpyHostToDevice, st);
  return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

cudaError_t launch_f64(const StepArgs& a, const F64View& v, int nspecies, cudaStream_t st) {
  char* b = static_cast<char*>(v.base);
  F64Args F{};
  F.row_sum = reinterpret_cast<double*>(b + v.off[4]);
  F.col_sum = reinterpret_cast<double*>(b + v.off[5]);
  F.ext_sum = reinterpret_cast<double*>(b + v.off[6]);
  F.noise = reinterpret_cast<double*>(b + v.off[7]);
  F.springs = reinterpret_cast<double*>(b + v.off[8]);
  F.fold = reinterpret_cast<double*>(b + v.off[9]);
  F.cols = v.cols, F.warps = v.warps, F.nspecies = nspecies;
  for (int s = 0; s < nspecies; ++s) F.bath |= a.spc[s].sigma > 0.0;
  const void* pairs = nullptr;
  const void* finish = nullptr;
  switch (v.I) {
    case 1: pairs = a.unitw ? (const void*)k_pairs_f64<1, true> : (const void*)k_pairs_f64<1, false>, finish = (const void*)k_finish_f64<1>; break;
    case 2: pairs = a.unitw ? (const void*)k_pairs_f64<2, true> : (const void*)k_pairs_f64<2, false>, finish = (const void*)k_finish_f64<2>; break;
    case 4: pairs = a.unitw ? (const void*)k_pairs_f64<4, true> : (const void*)k_pairs_f64<4, false>, finish = (const void*)k_finish_f64<4>; break;
    default: pairs = a.unitw ? (const void*)k_pairs_f64<8, true> : (const void*)k_pairs_f64<8, false>, finish = (const void*)k_finish_f64<8>; break;
  }
  StepArgs ac = a;
  void* params[] = {&ac, &F};
  const int per = kF64Threads / 32;
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < v.bands && e == cudaSuccess; ++k) {
    char* t = b + v.band_bytes * k;
    F.share = reinterpret_cast<const F64Share*>(t + v.off[0]);
    F.row_flush = reinterpret_cast<const int*>(t + v.off[1]);
    F.col_extra = reinterpret_cast<const int*>(t + v.off[2]);
    F.extra = reinterpret_cast<const int*>(t + v.off[3]);
    F.row0 = k * kF64BandRows, F.rows = std::min(kF64BandRows, v.rows - F.row0);
    F.first = k == 0, F.last = k + 1 == v.bands;
    e = cudaLaunchKernel(pairs, dim3((unsigned)((v.warps + per - 1) / per)), dim3(kF64Threads), params, 0, st);
    if (e == cudaSuccess) e = cudaLaunchKernel(finish, dim3((unsigned)v.cols), dim3(96 * kF64Slices), params, 0, st);
  }
  return e;
}

}  // namespace it
