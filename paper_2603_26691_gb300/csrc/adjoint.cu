// Hand-written adjoint of the Lagrangian step (FP64 handles in FP64, mixed FP32-velocity handles in
// FP32), run backward through checkpointed segments with recomputation.
//
// For a loss L(Jtot) of the time-summed per-cell source, with
// lam = dL/dJtot given per cell, one reverse step of one particle runs the
// chain rule backward through the forward step
//   c0 = cell(x);  u_p = sum_corners W(f) U;  a = 18 mu alpha / (rho_p d^2)
//   E = e^{-a dt};  E1 = 1 - E;  Q = E1 / a;  w = u_p + g / a
//   v' = w E1 + v E;  x' = x + w (dt - Q) + v Q
//   J = -m (v' - v - g dt),  m = mult rho_p pi d^3 / 6,  Jtot[c0] += J
// with the deposit cell held fixed (its derivative is zero almost everywhere)
// and the periodic wrap a translation.  With the cloud-in-cell deposit
// (Jtot[corner] += W(f) J over the gather's stencil) the adjoint of J is the
// W-weighted sum of lam over the corners, and the weights' derivatives add
// lam_corner . J to the stencil-fraction adjoint beside the gather's term.  Per particle it carries the adjoints
// of x and v between steps and accumulates dL/dd; dL/dalpha is reduced
// per block in a fixed order; dL/dU is scattered through the transposed
// trilinear weights into an exact carry-save fixed-point accumulator, so
// every output is independent of thread scheduling.
#include "fix_gather.cuh"
#include "st_common.cuh"

namespace st {
namespace {

constexpr int kAdjThreads = 256;

struct AdjArgs {
  const double* __restrict__ x[3];   // state at the start of the step (tape)
  const double* __restrict__ v[3];
  const double* __restrict__ d;
  double* __restrict__ xb[3];        // adjoint of the state after the step (in), before it (out)
  double* __restrict__ vb[3];
  double* __restrict__ db;           // accumulated dL/dd
  double* __restrict__ ab_part;      // [gridDim.x] dL/dalpha partial sums, accumulated over steps
  const D4* __restrict__ U;
  const double* __restrict__ lam;    // [3][ncell]
  long long* __restrict__ Uw;        // [ncell][3][kWideWords] carry-save dL/dU
  int64_t n, ncell;
  int nx, ny, nz;
  double inv_h[3];
  double dt, ca, mcoef, alpha, g[3];
  double inv_ca, inv_alpha;  // 1 / ca, 1 / alpha
};

__device__ __forceinline__ D4 ld_cell(const D4* __restrict__ U, int64_t c) {
  const double2* p = reinterpret_cast<const double2*>(U + c);
  double2 a = __ldg(p), b = __ldg(p + 1);
  return D4{a.x, a.y, b.x, b.y};
}

// CIC: the cloud-in-cell deposit (else the containing cell)
template <bool CIC>
__global__ void __launch_bounds__(kAdjThreads) adjoint_step_kernel(const AdjArgs a) {
  const int n3[3] = {a.nx, a.ny, a.nz};
  double alphab_sum = 0.0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n; p += (int64_t)gridDim.x * blockDim.x) {
    double x[3], v[3], xb[3], vb[3];
    for (int q = 0; q < 3; ++q) {
      x[q] = a.x[q][p];
      v[q] = a.v[q][p];
      xb[q] = a.xb[q][p];
      vb[q] = a.vb[q][p];
    }
    const double d = a.d[p];
    // recompute the forward intermediates
    int c0[3], i0[3], i1[3];
    double f[3];
    for (int q = 0; q < 3; ++q) {
      const double sx = x[q] * a.inv_h[q];
      c0[q] = min(max((int)floor(sx), 0), n3[q] - 1);
      const double s2 = sx - 0.5;
      const double fl = floor(s2);
      const int ii = (int)fl;
      f[q] = s2 - fl;
      i0[q] = ii < 0 ? ii + n3[q] : ii;
      i1[q] = ii + 1 >= n3[q] ? ii + 1 - n3[q] : ii + 1;
    }
    const int64_t key = c0[0] + (int64_t)a.nx * (c0[1] + (int64_t)a.ny * c0[2]);
    int64_t corner[8];
    D4 Uc[8];
    for (int k = 0; k < 8; ++k) {
      const int di = k & 1, dj = (k >> 1) & 1, dk = (k >> 2) & 1;
      corner[k] = (di ? i1[0] : i0[0]) + (int64_t)a.nx * ((dj ? i1[1] : i0[1]) + (int64_t)a.ny * (dk ? i1[2] : i0[2]));
      Uc[k] = ld_cell(a.U, corner[k]);
    }
    double up[3] = {0.0, 0.0, 0.0};
    double W[8];
    for (int k = 0; k < 8; ++k) {
      const int di = k & 1, dj = (k >> 1) & 1, dk = (k >> 2) & 1;
      W[k] = (di ? f[0] : 1.0 - f[0]) * (dj ? f[1] : 1.0 - f[1]) * (dk ? f[2] : 1.0 - f[2]);
      up[0] += W[k] * Uc[k].x;
      up[1] += W[k] * Uc[k].y;
      up[2] += W[k] * Uc[k].z;
    }
    const double dd = d * d;
    // the reciprocals once (GB300 divides in FP64 by iteration): 1/a, 1/a^2, 1/d
    const double inv_ra = dd * a.inv_ca;
    const double ra = 1.0 / inv_ra;
    const double inv_ra2 = inv_ra * inv_ra;
    const double inv_d = 1.0 / d;
    const double E1 = -expm1(-ra * a.dt);
    const double E = 1.0 - E1;  // e^{-a dt} as the complement of expm1, as in the forward step
    const double Q = E1 * inv_ra;
    const double m = a.mcoef * dd * d;
    double wt[3], vn[3];
    for (int q = 0; q < 3; ++q) {
      wt[q] = up[q] + a.g[q] * inv_ra;
      vn[q] = wt[q] + (v[q] - wt[q]) * E;
    }
    // reverse sweep
    double Jb[3];
    double lj[CIC ? 8 : 1];  // cloud in cell: lam at each corner dotted with J
    if constexpr (CIC) {
      double J[3];
      for (int q = 0; q < 3; ++q) J[q] = -m * (vn[q] - v[q] - a.g[q] * a.dt);
      Jb[0] = Jb[1] = Jb[2] = 0.0;
      for (int k = 0; k < 8; ++k) {
        const double l0 = a.lam[corner[k]], l1 = a.lam[a.ncell + corner[k]], l2 = a.lam[2 * a.ncell + corner[k]];
        Jb[0] += W[k] * l0;
        Jb[1] += W[k] * l1;
        Jb[2] += W[k] * l2;
        lj[k] = l0 * J[0] + l1 * J[1] + l2 * J[2];
      }
    } else {
      Jb[0] = a.lam[key];
      Jb[1] = a.lam[a.ncell + key];
      Jb[2] = a.lam[2 * a.ncell + key];
    }
    double mb = 0.0, Eb = 0.0, E1b = 0.0, Qb = 0.0, ab = 0.0;
    double ub[3], vsb[3];
    for (int q = 0; q < 3; ++q) {
      const double vnb = vb[q] - m * Jb[q];
      vsb[q] = m * Jb[q] + vnb * E + xb[q] * Q;
      mb -= (vn[q] - v[q] - a.g[q] * a.dt) * Jb[q];
      const double wtb = vnb * E1 + xb[q] * (a.dt - Q);
      E1b += vnb * wt[q];
      Eb += vnb * v[q];
      Qb += xb[q] * (v[q] - wt[q]);
      ub[q] = wtb;
      ab -= wtb * a.g[q] * inv_ra2;
    }
    E1b += Qb * inv_ra;
    ab -= Qb * E1 * inv_ra2;
    ab += a.dt * E * (E1b - Eb);
    alphab_sum += ab * ra * a.inv_alpha;
    double dbv = a.db[p] + ab * (-2.0 * ra * inv_d) + mb * 3.0 * m * inv_d;
    a.db[p] = dbv;
    // transposed trilinear weights: dL/dU (each corner's weight times ub) and dL/df, the
    // derivative of the trilinear form of the corner values' dot products with ub (plus, for the
    // cloud-in-cell deposit, lam . J at the corner), taken separably (differences along one
    // axis, interpolated along the other two)
    double dot[8];
    for (int k = 0; k < 8; ++k) {
      dot[k] = Uc[k].x * ub[0] + Uc[k].y * ub[1] + Uc[k].z * ub[2];
      if constexpr (CIC) dot[k] += lj[k];
      long long* w = a.Uw + corner[k] * 3 * kWideWords;
      wide_add(w, W[k] * ub[0]);
      wide_add(w + kWideWords, W[k] * ub[1]);
      wide_add(w + 2 * kWideWords, W[k] * ub[2]);
    }
    // corner k = di + 2 dj + 4 dk; lerp(p, q, t) = p + t (q - p)
    auto lerp = [](double p0, double p1, double t) { return p0 + t * (p1 - p0); };
    double fb[3];
    {
      // d/df_x: x-differences at the four (dj, dk) edges, interpolated in y then z
      const double e00 = dot[1] - dot[0], e10 = dot[3] - dot[2], e01 = dot[5] - dot[4], e11 = dot[7] - dot[6];
      fb[0] = lerp(lerp(e00, e10, f[1]), lerp(e01, e11, f[1]), f[2]);
      // d/df_y: y-differences, interpolated in x then z
      const double g00 = dot[2] - dot[0], g10 = dot[3] - dot[1], g01 = dot[6] - dot[4], g11 = dot[7] - dot[5];
      fb[1] = lerp(lerp(g00, g10, f[0]), lerp(g01, g11, f[0]), f[2]);
      // d/df_z: z-differences, interpolated in x then y
      const double h00 = dot[4] - dot[0], h10 = dot[5] - dot[1], h01 = dot[6] - dot[2], h11 = dot[7] - dot[3];
      fb[2] = lerp(lerp(h00, h10, f[0]), lerp(h01, h11, f[0]), f[1]);
    }
    for (int q = 0; q < 3; ++q) {
      a.xb[q][p] = xb[q] + fb[q] * a.inv_h[q];
      a.vb[q][p] = vsb[q];
    }
  }
  // fixed-order block reduction of dL/dalpha
  __shared__ double sh[kAdjThreads / 32];
  double s = alphab_sum;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kAdjThreads / 32; ++w) t += sh[w];
    a.ab_part[blockIdx.x] += t;
  }
}

// ---- a whole segment of the default physics (cell deposit) in one launch ----
//
// The same reverse sweep, bound by what is left on the FP64 pipe (one warp instruction in 64 cycles there):
//   * the interpolation and its derivatives by the position run on integers (fix_gather.cuh);
//   * what the diameter decides is computed once per particle, and the adjoints of position, velocity and
//     diameter stay in registers over the segment;
//   * dL/dU: a particle's products of weight and adjoint velocity are formed on integers too, each with a relative
//     error below 2^-53 whatever the weight's size.  They are summed over the steps it stays in one stencil (96-bit
//     sums in shared memory) and each sum is added to the carry-save accumulator when the particle leaves the stencil
//     or the segment ends: 24 global commits of three or four 64-bit reductions per stencil instead of per step,
//     which bound the sweep.  These sums are exact, and the diameter's run on over the segments, so the gradients do
//     not depend on how the steps are cut into segments.
// 69 FP64 instructions (109 operations) are left per particle and step in segments of 20, what is done once per segment
// included, against 349 operations.  2e6 particles on 64^3, 40 steps: 21.9 ms against 44.4 ms step by step; of these some
// 16 ms are the sweep without the sums, and the sums and their commits take about as much as each other.  (With products
// and sums of 64 bits, which kept fewer bits of small weights than FP64 does, 20.6 ms.)  16 warps per SM at 128
// registers: 12 at 168 take 0.9 ms more.  The loop over the components that adds the products is not unrolled: the kernel
// is as large as the instruction cache likes (1.1 ms more unrolled).
constexpr int kSegThreads = 128;
// stencils in a warp up to which its lanes are summed before the commits at a segment's end (sorted particles,
// 1e7 on 64^3: 22.9 ms with the line at 12 against 24.4 ms without sums across lanes; unsorted particles lie above
// any such line)
constexpr int kSharedStencils = 12;

// A thread's 24 running sums of products of corner weight k and adjoint velocity component q, integers in units
// of 2^(eb[q] - bits), of the stencil with base cell c0 and steps sx, sy, sz to the next cells.  WIDE: of 96 bits.
template <bool WIDE>
struct StencilSums {
  unsigned long long v[24][kSegThreads + 1];  // [3 k + q][thread]; padded: a commit reads columns
  int h[WIDE ? 24 : 1][kSegThreads + 1];      // bits 64 .. 95
  int e[3][kSegThreads];                      // eb, read by the lanes that commit
  // units that lanes may differ by to be summed first: their sums, aligned, have to fit 128 bits
  static constexpr int kNear = WIDE ? 13 : 28;

  __device__ __forceinline__ void clear(int t) {
#pragma unroll
    for (int i = 0; i < 24; ++i) {
      v[i][t] = 0;
      if (WIDE) h[i][t] = 0;
    }
  }
  __device__ __forceinline__ __int128 take(int i, int t) {
    const unsigned long long lo = v[i][t];
    v[i][t] = 0;
    if (!WIDE) return (long long)lo;
    const long long hi = h[i][t];
    h[i][t] = 0;
    return (__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo);
  }
};

// The sums of a lane's component q, and the stencil they belong to, for the commits below.
struct SumRef {
  int c0, sx, sy, sz;  // base cell, steps to the next cells
  int e;               // eb[q]
};

// Adds component q's sums of the lanes `who` to dL/dU, all lanes of the warp together: four lanes' sums at a time,
// one corner per lane.  (Few lanes leave their stencil in one step; each by itself would hold up the
// others for its eight corners.)
template <bool WIDE>
__device__ __noinline__ void commit_component(StencilSums<WIDE>& s, long long* __restrict__ Uw, unsigned who, int q, SumRef r,
                                              int bits) {
  const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31, k = lane & 7;
  __syncwarp();
  while (who) {
    int src = -1;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      if (who && (lane >> 3) == g) src = __ffs(who) - 1;
      who &= who - 1;  // stays 0
    }
    const int from = src < 0 ? lane : src;
    const int c0 = __shfl_sync(0xffffffffu, r.c0, from), sx = __shfl_sync(0xffffffffu, r.sx, from),
              sy = __shfl_sync(0xffffffffu, r.sy, from), sz = __shfl_sync(0xffffffffu, r.sz, from),
              e = __shfl_sync(0xffffffffu, r.e, from);
    if (src >= 0) {
      const __int128 v = s.take(3 * k + q, w0 + src);
      const int c = c0 + ((k & 1) ? sx : 0) + ((k & 2) ? sy : 0) + ((k & 4) ? sz : 0);
      long long* w = Uw + ((int64_t)c * 3 + q) * kWideWords;
      if (WIDE)
        wide_add_int128(w, v, e - bits);
      else
        wide_add_int(w, (long long)v, e - bits);
    }
  }
  __syncwarp();
}

// The same for all lanes and components where many lanes share few stencils (sorted particles at the end of a
// segment): the lanes of one stencil whose units are near enough are summed first.  The sums are exact, so
// their order does not matter.
template <bool WIDE>
__device__ __noinline__ void commit_shared(StencilSums<WIDE>& s, long long* __restrict__ Uw, unsigned who, int c0, int sx,
                                           int sy, int sz, int e0, int e1, int e2, int bits) {
  constexpr int kNear = StencilSums<WIDE>::kNear;
  const int t = threadIdx.x, lane = t & 31, w0 = t & ~31;
  const bool need = (who >> lane) & 1u;
  s.e[0][t] = e0;
  s.e[1][t] = e1;
  s.e[2][t] = e2;
  __syncwarp();
  while (who) {
    const int src = __ffs(who) - 1;
    const int b0 = __shfl_sync(0xffffffffu, c0, src), bx = __shfl_sync(0xffffffffu, sx, src),
              by = __shfl_sync(0xffffffffu, sy, src), bz = __shfl_sync(0xffffffffu, sz, src);
    const bool same = need && ((who >> lane) & 1u) && c0 == b0 && abs(e0 - s.e[0][w0 + src]) <= kNear &&
                      abs(e1 - s.e[1][w0 + src]) <= kNear && abs(e2 - s.e[2][w0 + src]) <= kNear;
    const unsigned grp = __ballot_sync(0xffffffffu, same);
    who &= ~grp;
    if (lane < 24) {
      const int k = lane / 3, q = lane - 3 * k;
      const int low = s.e[q][w0 + src] - kNear;
      __int128 sum = 0;
      for (unsigned g = grp; g; g &= g - 1u) {
        const int m = w0 + __ffs(g) - 1;
        sum += s.take(lane, m) << (s.e[q][m] - low);
      }
      const int c = b0 + ((k & 1) ? bx : 0) + ((k & 2) ? by : 0) + ((k & 4) ? bz : 0);
      wide_add_int128(Uw + ((int64_t)c * 3 + q) * kWideWords, sum, low - bits);
    }
  }
  __syncwarp();
}

// every lane's sums that hold anything (added), at the end of a segment
template <bool WIDE>
__device__ __forceinline__ void commit_all(StencilSums<WIDE>& s, long long* __restrict__ Uw, const int (&added)[3], int c0,
                                           int sx, int sy, int sz, const int (&eb)[3], int bits) {
  const bool need = added[0] || added[1] || added[2];
  const unsigned who = __ballot_sync(0xffffffffu, need);
  const unsigned peers = __match_any_sync(0xffffffffu, need ? c0 : -1);
  const int stencils = __popc(__ballot_sync(0xffffffffu, (peers & ((1u << (threadIdx.x & 31)) - 1u)) == 0u));
  if (stencils <= kSharedStencils) {
    commit_shared(s, Uw, who, c0, sx, sy, sz, eb[0], eb[1], eb[2], bits);
  } else {
#pragma unroll 1
    for (int q = 0; q < 3; ++q) commit_component(s, Uw, who, q, SumRef{c0, sx, sy, sz, q == 0 ? eb[0] : q == 1 ? eb[1] : eb[2]}, bits);
  }
}

constexpr int kSumSteps = 32;  // products one sum takes
// Products are integers below 2^57 (FP64) or 2^24 (FP32), shifted up by 0 .. window, so kSumSteps of them fit 96 or 64
// bits; a sum starts with `below` of the window below its first adjoint velocity's exponent (small weights, components
// that cross zero).  (FP64's shifts stay below a word's 32.)
template <bool WIDE>
struct Window {
  static constexpr int kWindow = WIDE ? 31 : 33, kBelow = WIDE ? 26 : 28;
};

// The trilinear weights with a relative error below 2^-58 each, whatever their size (the integers of fix::weights have 58
// below the point): corner k = dx + 2 dy + 4 dz has the weight m[k] 2^(-46 - c[k]).
// a b / 2^64, up to three units low (the product of the low halves is not formed)
__device__ __forceinline__ unsigned long long mul_high(unsigned long long a, unsigned long long b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (unsigned long long)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}
struct FloatWeights {
  unsigned long long m[8];
  int c[8];
};
// the largest c of a weight that is not zero
__device__ __forceinline__ int smallest_weight(const int64_t (&f)[3]) {
  int c = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int64_t m = min(f[q], fix::kOne - f[q]);
    c += m > 0 ? __clzll(m) : 63 - fix::kFrac;
  }
  return c;
}
__device__ __forceinline__ void float_weights(const int64_t (&f)[3], FloatWeights& w) {
  unsigned long long g[3][2];
  int c[3][2];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const unsigned long long a = (unsigned long long)(fix::kOne - f[q]), b = (unsigned long long)f[q];  // a > 0
    c[q][0] = __clzll((long long)a);
    c[q][1] = b ? __clzll((long long)b) : 63 - fix::kFrac;  // a zero stays zero
    g[q][0] = a << c[q][0];
    g[q][1] = b << c[q][1];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned long long xy = mul_high(g[0][k & 1], g[1][k >> 1]);
    w.m[k] = mul_high(xy, g[2][0]);
    w.m[4 + k] = mul_high(xy, g[2][1]);
    w.c[k] = c[0][k & 1] + c[1][k >> 1] + c[2][0];
    w.c[4 + k] = c[0][k & 1] + c[1][k >> 1] + c[2][1];
  }
}
// |u| = m 2^(e - 1086), m at least 2^63, for u != 0
__device__ __forceinline__ void float_value(double u, unsigned long long& m, int& e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(u);
  e = (int)((b >> 52) & 0x7ff);
  m = (b << 11) | 0x8000000000000000ull;
  if (__builtin_expect(e == 0, 0)) {  // subnormal
    const int z = __clzll((long long)(b << 1 >> 1));
    m = b << z;
    e = 12 - z;
  }
}
// their product: a whole number of at most 57 bits (53 at least), times 2^(e - c[k] - kProductBits), off by less than
// 2^-53 of itself
constexpr int kProductBits = 1061;
__device__ __forceinline__ unsigned long long product(unsigned long long w, unsigned long long u) {
  return (mul_high(w, u) + 64) >> 7;
}

// The products of the components `which` (a bit each), some of which a sum cannot hold (rare: weights below about
// 2^-26), each straight to dL/dU.
__device__ __noinline__ void commit_products(long long* __restrict__ Uw, unsigned which, SumRef r, int64_t f0, int64_t f1,
                                             int64_t f2, double ub0, double ub1, double ub2) {
  const int64_t f[3] = {f0, f1, f2};
  FloatWeights w;
  float_weights(f, w);
#pragma unroll 1
  for (; which; which &= which - 1) {
    const int q = __ffs(which) - 1;
    const double ub = q == 0 ? ub0 : q == 1 ? ub1 : ub2;
    unsigned long long u;
    int e;
    float_value(ub, u, e);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int c = r.c0 + ((k & 1) ? r.sx : 0) + ((k & 2) ? r.sy : 0) + ((k & 4) ? r.sz : 0);
      const long long p = (long long)product(w.m[k], u);
      wide_add_int(Uw + ((int64_t)c * 3 + q) * kWideWords, ub < 0.0 ? -p : p, e - w.c[k] - kProductBits);
    }
  }
}

constexpr int kWeightOne = 3 * (63 - fix::kFrac);  // FloatWeights::c of a weight of one
static_assert(Window<true>::kWindow + 57 + 5 < 96 && Window<true>::kWindow < 32, "kSumSteps products fit 96 bits");

// the 96-bit sum (v, h) plus (x2, x1, x0), or minus it (neg: all ones)
__device__ __forceinline__ void add96(unsigned long long& v, int& h, uint32_t x0, uint32_t x1, uint32_t x2, int neg) {
  uint32_t s0 = (uint32_t)v, s1 = (uint32_t)(v >> 32), s2 = (uint32_t)h, carry;
  asm("add.cc.u32 %3, %7, 1;\n\taddc.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.u32 %2, %2, %6;"
      : "+r"(s0), "+r"(s1), "+r"(s2), "=&r"(carry)
      : "r"(x0 ^ neg), "r"(x1 ^ neg), "r"(x2 ^ neg), "r"(neg));
  v = ((unsigned long long)s1 << 32) | s0;
  h = (int)s2;
}

struct SegArgs {
  const double* __restrict__ tape;  // [len][6][n]
  const double* __restrict__ d;
  double* __restrict__ xb[3];
  double* __restrict__ vb[3];
  double* __restrict__ ab;  // sums over the segments so far for dL/da and dL/dm; after the last one ab is dL/dd
  double* __restrict__ mb;
  double* __restrict__ ab_part;
  const fix::FixCell* __restrict__ U;
  const double* __restrict__ lam;
  long long* __restrict__ Uw;
  int64_t n, ncell;
  int nx, ny, nz, len, last;
  fix::Scale scale;
  double dt, mcoef, g[3];
  double inv_ca, inv_alpha;
};

__global__ void __launch_bounds__(kSegThreads, 4) adjoint_segment_kernel(const SegArgs a) {
  __shared__ StencilSums<true> sums;
  const int n3[3] = {a.nx, a.ny, a.nz};
  const int t = threadIdx.x;
  double alphab_sum = 0.0;
  sums.clear(t);
  for (int64_t wbase = blockIdx.x * (int64_t)blockDim.x + (t & ~31); wbase < a.n;
       wbase += (int64_t)gridDim.x * blockDim.x) {
    __syncwarp();
    const int64_t p = min(wbase + (t & 31), a.n - 1);
    // lanes past the end go along with the last particle and change nothing
    const bool valid = wbase + (t & 31) < a.n;
    const double d = a.d[p];
    const double dd = d * d;
    const double inv_ra = dd * a.inv_ca;
    const double ra = 1.0 / inv_ra;
    const double inv_ra2 = inv_ra * inv_ra;
    const double inv_d = 1.0 / d;
    const double E1 = -expm1(-ra * a.dt);
    const double E = 1.0 - E1;  // e^{-a dt} as the complement of expm1, as in the forward step
    const double Q = E1 * inv_ra;
    const double dtQ = a.dt - Q;
    const double m = a.mcoef * dd * d;
    const double c1 = a.dt * E, c2 = inv_ra * (c1 - Q);
    double xb[3], vb[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      xb[q] = a.xb[q][p];
      vb[q] = a.vb[q][p];
    }
    double ab_sum = a.ab[p], mb_sum = a.mb[p];
    int corner0 = -1, c1x = 0, c1y = 0, c1z = 0;  // the stencil of the sums: its base cell, steps to the next cells
    int eb[3] = {0, 0, 0}, added[3] = {0, 0, 0};
#pragma unroll 1
    for (int step = a.len - 1; step >= 0; --step) {
      __syncwarp();
      const double* slot = a.tape + (int64_t)step * 6 * a.n;
      double x[3], v[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        x[q] = slot[q * a.n + p];
        v[q] = slot[(3 + q) * a.n + p];
      }
      const fix::Stencil st = fix::stencil(x, a.scale, n3);
      const int key = st.c0[0] + a.nx * (st.c0[1] + a.ny * st.c0[2]);
      const double Jb[3] = {a.lam[key], a.lam[a.ncell + key], a.lam[2 * a.ncell + key]};
      const int base = st.i0[0] + a.nx * (st.i0[1] + a.ny * st.i0[2]);
      fix::Corners u;
      fix::load_corners(a.U, st, a.nx, a.ny, u);
      int64_t W[8];
      fix::weights(st.f, W);
      double ub[3], dvw[3];
      double mb = 0.0, S = 0.0, Qb = 0.0, gs = 0.0;
      {
        double up[3];
        fix::interpolate(u, W, up);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double wt = up[q] + a.g[q] * inv_ra;
          dvw[q] = v[q] - wt;
          const double mJ = m * Jb[q];
          const double vnb = vb[q] - mJ;
          // -(v' - v - g dt) = (v - w) (1 - E) + g dt
          mb += (dvw[q] * E1 + a.g[q] * a.dt) * Jb[q];
          S += vnb * dvw[q];
          Qb += xb[q] * dvw[q];
          ub[q] = vnb * E1 + xb[q] * dtQ;
          gs += ub[q] * a.g[q];
          vb[q] = vnb * E + (xb[q] * Q + mJ);
        }
      }
      // a's adjoint: through w (gravity), Q = E1 / a, and E, E1 (dE1/da = dt E)
      const double ab = c2 * Qb - c1 * S - gs * inv_ra2;
      ab_sum += ab;
      mb_sum += mb;
      // dL/df, the derivatives of the interpolated velocity dotted with its adjoint
      {
        double g[3];
        fix::derivative<0>(u, st.f, g);
        xb[0] += (g[0] * ub[0] + g[1] * ub[1] + g[2] * ub[2]) * a.scale.inv_h[0];
        fix::derivative<1>(u, st.f, g);
        xb[1] += (g[0] * ub[0] + g[1] * ub[1] + g[2] * ub[2]) * a.scale.inv_h[1];
        fix::derivative<2>(u, st.f, g);
        xb[2] += (g[0] * ub[0] + g[1] * ub[1] + g[2] * ub[2]) * a.scale.inv_h[2];
      }
      // dL/dU: sums of another stencil, or whose unit does not suit the products (too large, or too small as the adjoint
      // velocity decays within a cell: 24.9 against 31.9 ms with such products committed by themselves), are committed
      // and started anew; lone: components with a product that a new sum cannot hold either, summed: those with any for
      // the sums
      const bool moved = base != corner0;
      const int cmax = smallest_weight(st.f);
      unsigned lone = 0, summed = 0;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(ub[q]);
        const int e = (int)((b >> 52) & 0x7ff), fresh = e - kWeightOne - Window<true>::kBelow;
        const bool some = valid && (b << 1) != 0;
        const bool suits = !some || (e - kWeightOne - eb[q] <= Window<true>::kWindow && (e - cmax >= eb[q] || fresh >= eb[q]));
        const bool full = valid && added[q] && (moved || added[q] >= kSumSteps || !suits);
        const unsigned who = __ballot_sync(0xffffffffu, full);
        if (who) commit_component(sums, a.Uw, who, q, SumRef{corner0, c1x, c1y, c1z, eb[q]}, kProductBits);
        if (full) added[q] = 0;
        if (some) {
          if (added[q] == 0) eb[q] = fresh;
          ++added[q];
          (e != 0 && e - cmax >= eb[q] ? summed : lone) |= 1u << q;
        }
      }
      if (moved) {
        corner0 = base;
        c1x = st.i1[0] - st.i0[0];
        c1y = a.nx * (st.i1[1] - st.i0[1]);
        c1z = a.nx * a.ny * (st.i1[2] - st.i0[2]);
      }
      if (__any_sync(0xffffffffu, lone != 0u))
        commit_products(a.Uw, lone, SumRef{corner0, c1x, c1y, c1z, 0}, st.f[0], st.f[1], st.f[2], ub[0], ub[1], ub[2]);
      __syncwarp();
      FloatWeights w;
      float_weights(st.f, w);
#pragma unroll 1
      for (int q = 0; q < 3; ++q) {
        const double ubq = q == 0 ? ub[0] : q == 1 ? ub[1] : ub[2];
        const int ebq = q == 0 ? eb[0] : q == 1 ? eb[1] : eb[2];
        const unsigned long long b = (unsigned long long)__double_as_longlong(ubq);
        const int e = (int)((b >> 52) & 0x7ff);
        const unsigned long long u = (summed >> q) & 1u ? (b << 11) | 0x8000000000000000ull : 0ull;
        const int neg = (int)((long long)b >> 63), up = e - ebq;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const unsigned long long p = product(w.m[k], u);
          const uint32_t p0 = (uint32_t)p, p1 = (uint32_t)(p >> 32);
          const int sh = up - w.c[k];  // 0 .. kWindow where the product is not zero
          add96(sums.v[3 * k + q][t], sums.h[3 * k + q][t], p0 << (sh & 31), __funnelshift_l(p0, p1, sh),
                __funnelshift_l(p1, 0u, sh), neg);
        }
      }
    }
    if (!valid) added[0] = added[1] = added[2] = 0;
    commit_all(sums, a.Uw, added, corner0, c1x, c1y, c1z, eb, kProductBits);
    if (!valid) continue;
    if (a.last) {
      alphab_sum += ab_sum * ra * a.inv_alpha;
      a.ab[p] = ab_sum * (-2.0 * ra * inv_d) + mb_sum * (3.0 * m * inv_d);
    } else {
      a.ab[p] = ab_sum;
      a.mb[p] = mb_sum;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      a.xb[q][p] = xb[q];
      a.vb[q][p] = vb[q];
    }
  }
  // fixed-order block reduction of dL/dalpha
  __shared__ double sh[kSegThreads / 32];
  double s = alphab_sum;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((t & 31) == 0) sh[t >> 5] = s;
  __syncthreads();
  if (t == 0) {
    double r = 0.0;
    for (int w = 0; w < kSegThreads / 32; ++w) r += sh[w];
    a.ab_part[blockIdx.x] += r;
  }
}

// ---- the FP32 adjoint of the mixed-precision step ----
//
// The same reverse sweep in FP32 on the mixed state, a segment of steps per launch: the tape gives each
// start-of-step cell, the offsets in it and the velocity; the trilinear stencil is the forward kernel's (base
// cell and fractions from the offset, corners read from the ghost-padded FP32 field), the deposit cell the
// start cell.  Position adjoints are per metre, as in the FP64 adjoint (the periodic wrap and the
// whole-cell carry are translations); they and the velocity's stay in registers over the segment.  Each
// step's dL/dd and dL/dalpha contributions are FP32 and accumulate in FP64, per particle and in the steps'
// order.  dL/dU: the FP32 products of the adjoint velocity and the corners' weights are integers in a unit that
// reaches from 2^28 times below the first of them to 32 times above; they are summed over the steps a particle stays in
// one stencil (commit_component) and then over the warp's lanes of the same stencil (commit_shared), all exactly, so
// dL/dU is the same however the steps are cut into segments.  1e7 particles on 64^3 sorted once, 40 steps: 20.2 ms
// against 39.5 ms with warp sums and commits in every step, and 21.3 ms with weights of 26 bits, which lost small ones
// and could hold fewer adjoint velocities in a sum.  Half of it is the sweep with its sums, the rest the commits of the
// particles that leave a stencil, bound by L2's 1.9e11 64-bit reductions a second.

struct AdjMixedArgs {
  const char* __restrict__ tape;     // [len] states of 28 tape_n bytes
  int64_t tape_n;
  int len;
  const float* __restrict__ d;
  float* __restrict__ xb[3];
  float* __restrict__ vb[3];
  double* __restrict__ db;
  double* __restrict__ ab;
  const float4* __restrict__ Up;     // ghost-padded field
  const float* __restrict__ lam;     // [3][ncell]
  long long* __restrict__ Uw;
  int64_t n, ncell;
  int nx, ny, nz;
  float inv_h[3];
  float dt, cadt, inv_ca, mcoef, g[3], gdt[3];
};

// the weight of corner k = dx + 2 dy + 4 dz
__device__ __forceinline__ float corner_weight(const float (&f)[3], int k) {
  return (k & 1 ? f[0] : 1.0f - f[0]) * (k & 2 ? f[1] : 1.0f - f[1]) * (k & 4 ? f[2] : 1.0f - f[2]);
}

// The products of the components `which` (a bit each), some of which a sum cannot hold (rare: weights below about
// 2^-28), each straight to dL/dU.
__device__ __noinline__ void commit_products(long long* __restrict__ Uw, unsigned which, SumRef r, float f0, float f1,
                                             float f2, float ub0, float ub1, float ub2) {
  const float f[3] = {f0, f1, f2};
#pragma unroll 1
  for (; which; which &= which - 1) {
    const int q = __ffs(which) - 1;
    const float ub = q == 0 ? ub0 : q == 1 ? ub1 : ub2;
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
      const int c = r.c0 + ((k & 1) ? r.sx : 0) + ((k & 2) ? r.sy : 0) + ((k & 4) ? r.sz : 0);
      const float p = __fmul_rn(corner_weight(f, k), ub);
      if (p != 0.0f) add_f32_words(Uw + ((int64_t)c * 3 + q) * kWideWords, kWideWords, p, -kWideBase);
    }
  }
}

__global__ void __launch_bounds__(kSegThreads, 4) adjoint_segment_mixed_kernel(const AdjMixedArgs a) {
  __shared__ StencilSums<false> sums;
  const int n3[3] = {a.nx, a.ny, a.nz};
  const int row = a.nx + 2 * kFluidPad, slab = row * (a.ny + 2 * kFluidPad);
  const int t = threadIdx.x;
  sums.clear(t);
  for (int64_t wbase = blockIdx.x * (int64_t)blockDim.x + (t & ~31); wbase < a.n;
       wbase += (int64_t)gridDim.x * blockDim.x) {
    __syncwarp();
    const int64_t p = min(wbase + (t & 31), a.n - 1);
    // lanes past the end go along with the last particle and change nothing
    const bool valid = wbase + (t & 31) < a.n;
    float xb[3], vb[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      xb[q] = a.xb[q][p];
      vb[q] = a.vb[q][p];
    }
    const float d = a.d[p];
    const float dd = d * d;
    const float adt = a.cadt / dd;     // a dt
    const float inv_ra = dd * a.inv_ca;  // 1 / a
    const float ra = 1.0f / inv_ra;
    const float inv_ra2 = inv_ra * inv_ra;
    const float inv_d = 1.0f / d;
    const float E1 = -expm1f(-adt);
    const float E = 1.0f - E1;
    const float Q = E1 * inv_ra;
    const float m = a.mcoef * dd * d;
    double db = a.db[p], ab_sum = a.ab[p];
    int corner0 = -1, c1x = 0, c1y = 0, c1z = 0;  // the stencil of the sums: its base cell, steps to the next cells
    int eb[3] = {0, 0, 0}, added[3] = {0, 0, 0};
#pragma unroll 1
    for (int step = a.len - 1; step >= 0; --step) {
      __syncwarp();
      const float* slot = reinterpret_cast<const float*>(a.tape + (int64_t)step * 28 * a.tape_n);
      if (step > 0) {  // ask L2 for the next step's state: 22.9 -> 21.3 ms at 1e7 particles x 40 steps
#pragma unroll
        for (int q = 0; q < 7; ++q) asm volatile("prefetch.global.L2 [%0];" ::"l"(slot - (7 - q) * a.tape_n + p));
      }
      const int c = __float_as_int(slot[p]);
      const int ci[3] = {cell_i(c), cell_j(c), cell_k(c)};
      float v[3], f[3];
      int i0[3], lo[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float o = slot[(1 + q) * a.tape_n + p];
        v[q] = slot[(4 + q) * a.tape_n + p];
        const bool up_half = o >= 0.5f;
        i0[q] = ci[q] - (up_half ? 0 : 1);  // -1 .. n - 1
        f[q] = o + (up_half ? -0.5f : 0.5f);
        lo[q] = i0[q] < 0 ? i0[q] + n3[q] : i0[q];
      }
      const int64_t cell_key = ci[0] + (int64_t)a.nx * (ci[1] + (int64_t)a.ny * ci[2]);
      const float Jb[3] = {a.lam[cell_key], a.lam[a.ncell + cell_key], a.lam[2 * a.ncell + cell_key]};
      const int base = lo[0] + a.nx * (lo[1] + a.ny * lo[2]);
      const float4* b = a.Up + (i0[0] + kFluidPad) + (int64_t)row * (i0[1] + kFluidPad) + (int64_t)slab * (i0[2] + kFluidPad);
      float4 Uc[8];
      float up[3] = {0.0f, 0.0f, 0.0f}, W[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        Uc[k] = __ldg(b + (k & 1) + row * ((k >> 1) & 1) + slab * (k >> 2));
        W[k] = corner_weight(f, k);
        up[0] = fmaf(W[k], Uc[k].x, up[0]);
        up[1] = fmaf(W[k], Uc[k].y, up[1]);
        up[2] = fmaf(W[k], Uc[k].z, up[2]);
      }
      float wt[3], vn[3], ub[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        wt[q] = fmaf(a.g[q], inv_ra, up[q]);
        vn[q] = fmaf(v[q] - wt[q], E, wt[q]);
      }
      float mb = 0.0f, Eb = 0.0f, E1b = 0.0f, Qb = 0.0f, ab = 0.0f;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float vnb = vb[q] - m * Jb[q];
        vb[q] = fmaf(m, Jb[q], fmaf(vnb, E, xb[q] * Q));
        mb -= ((vn[q] - v[q]) - a.gdt[q]) * Jb[q];
        const float wtb = fmaf(vnb, E1, xb[q] * (a.dt - Q));
        E1b = fmaf(vnb, wt[q], E1b);
        Eb = fmaf(vnb, v[q], Eb);
        Qb = fmaf(xb[q], v[q] - wt[q], Qb);
        ub[q] = wtb;
        ab -= wtb * a.g[q] * inv_ra2;
      }
      E1b = fmaf(Qb, inv_ra, E1b);
      ab -= Qb * E1 * inv_ra2;
      ab = fmaf(a.dt * E, E1b - Eb, ab);
      ab_sum += widen(ab * ra);
      db += widen(ab * (-2.0f * ra * inv_d) + mb * 3.0f * m * inv_d);
      float dot[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) dot[k] = fmaf(Uc[k].x, ub[0], fmaf(Uc[k].y, ub[1], Uc[k].z * ub[2]));
      auto lerp = [](float p0, float p1, float u) { return fmaf(u, p1 - p0, p0); };
      {
        const float e00 = dot[1] - dot[0], e10 = dot[3] - dot[2], e01 = dot[5] - dot[4], e11 = dot[7] - dot[6];
        xb[0] = fmaf(lerp(lerp(e00, e10, f[1]), lerp(e01, e11, f[1]), f[2]), a.inv_h[0], xb[0]);
        const float g00 = dot[2] - dot[0], g10 = dot[3] - dot[1], g01 = dot[6] - dot[4], g11 = dot[7] - dot[5];
        xb[1] = fmaf(lerp(lerp(g00, g10, f[0]), lerp(g01, g11, f[0]), f[2]), a.inv_h[1], xb[1]);
        const float h00 = dot[4] - dot[0], h10 = dot[5] - dot[1], h01 = dot[6] - dot[2], h11 = dot[7] - dot[3];
        xb[2] = fmaf(lerp(lerp(h00, h10, f[0]), lerp(h01, h11, f[0]), f[1]), a.inv_h[2], xb[2]);
      }
      // dL/dU: sums of another stencil, or whose units cannot hold the adjoint velocity, are committed and started anew
      const bool moved = base != corner0;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int eu = max((int)((__float_as_uint(ub[q]) >> 23) & 0xffu), 1);
        const bool full = valid && added[q] && (moved || added[q] >= kSumSteps || eu - eb[q] > Window<false>::kWindow);
        const unsigned who = __ballot_sync(0xffffffffu, full);
        if (who) commit_component(sums, a.Uw, who, q, SumRef{corner0, c1x, c1y, c1z, eb[q]}, 150);
        if (full || added[q] == 0) {
          added[q] = 0;
          eb[q] = max(eu - Window<false>::kBelow, 1);
        }
        ++added[q];
      }
      if (moved) {
        corner0 = base;
        c1x = (lo[0] + 1 == a.nx ? 0 : lo[0] + 1) - lo[0];
        c1y = a.nx * ((lo[1] + 1 == a.ny ? 0 : lo[1] + 1) - lo[1]);
        c1z = a.nx * a.ny * ((lo[2] + 1 == a.nz ? 0 : lo[2] + 1) - lo[2]);
      }
      // the smallest weight that is not zero (rounding keeps the order of products)
      float least[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float m = fminf(f[q], 1.0f - f[q]);
        least[q] = m > 0.0f ? m : 1.0f;
      }
      const float Wmin = least[0] * least[1] * least[2];
      // components with a product that their sums cannot hold, and those with any for the sums
      unsigned lone = 0, summed = 0;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int emin = (int)(__float_as_uint(Wmin * fabsf(ub[q])) >> 23);  // 0: subnormal
        if (valid && ub[q] != 0.0f) (emin >= eb[q] ? summed : lone) |= 1u << q;
      }
      if (__any_sync(0xffffffffu, lone != 0u))
        commit_products(a.Uw, lone, SumRef{corner0, c1x, c1y, c1z, 0}, f[0], f[1], f[2], ub[0], ub[1], ub[2]);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        // a shift of 64 or more leaves nothing: of zeros (exponent 0 below eb >= 1), and of all where none is to be added
        const int e0 = (summed >> q) & 1u ? eb[q] : 1 << 16;
        const long long neg = ub[q] < 0.0f ? -1ll : 0ll;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t bits = __float_as_uint(__fmul_rn(W[k], fabsf(ub[q])));
          unsigned long long x = (bits & 0x7fffffu) | 0x800000u;
          asm("shl.b64 %0, %0, %1;" : "+l"(x) : "r"((int)(bits >> 23) - e0));
          sums.v[3 * k + q][t] += ((long long)x ^ neg) - neg;
        }
      }
    }
    if (!valid) added[0] = added[1] = added[2] = 0;
    commit_all(sums, a.Uw, added, corner0, c1x, c1y, c1z, eb, 150);
    if (!valid) continue;
    a.db[p] = db;
    a.ab[p] = ab_sum;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      a.xb[q][p] = xb[q];
      a.vb[q][p] = vb[q];
    }
  }
}

// partial sums of n doubles, one per block of kAdjBlocks: the order depends on n only
__global__ void __launch_bounds__(kAdjThreads) ordered_sum_kernel(const double* __restrict__ in, int64_t n,
                                                                  double* __restrict__ part) {
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) s += in[i];
  __shared__ double sh[kAdjThreads / 32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kAdjThreads / 32; ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

__global__ void f64_to_f32_kernel(const double* __restrict__ in, float* __restrict__ out, int64_t m) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

// value of each carry-save accumulator in FP64: out[c][q]
// carry propagation: digits in [0, 2^32) below a signed top word
__device__ __forceinline__ void wide_carry(long long* v) {
  long long c = 0;
  for (int k = 0; k < kWideWords - 1; ++k) {
    const long long t = v[k] + c;
    v[k] = t & 0xffffffffll;
    c = t >> 32;
  }
  v[kWideWords - 1] += c;
}

__global__ void wide_to_f64_kernel(const long long* __restrict__ Uw, double* __restrict__ out, int64_t m) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    // sign and magnitude first: summing signed words (a normalised negative value is words near 2^32
    // below a top word of -1) would cancel
    long long v[kWideWords];
    for (int k = 0; k < kWideWords; ++k) v[k] = Uw[i * kWideWords + k];
    wide_carry(v);
    const bool neg = v[kWideWords - 1] < 0;
    if (neg) {
      for (int k = 0; k < kWideWords; ++k) v[k] = -v[k];
      wide_carry(v);
    }
    // non-negative terms, smallest first
    double s = 0.0;
    for (int k = 0; k < kWideWords; ++k) s += ldexp((double)v[k], 32 * k + kWideBase);
    out[i] = neg ? -s : s;
  }
}

}  // namespace

cudaError_t launch_adjoint_step(st_ctx* h, const AdjointStepArgs& s) {
  AdjArgs a;
  for (int q = 0; q < 3; ++q) {
    a.x[q] = s.x[q];
    a.v[q] = s.v[q];
    a.xb[q] = s.xb[q];
    a.vb[q] = s.vb[q];
    a.inv_h[q] = h->geo.inv_h[q];
    a.g[q] = h->g[q];
  }
  a.d = s.d;
  a.db = s.db;
  a.ab_part = s.ab_part;
  a.U = (const D4*)h->fluid.p;
  a.lam = s.lam;
  a.Uw = s.Uw;
  a.n = h->np;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  a.dt = s.dt;
  a.ca = 18.0 * h->mu * h->alpha / h->rho_p;
  a.mcoef = h->mult * h->rho_p * 3.14159265358979323846 / 6.0;
  a.alpha = h->alpha;
  a.inv_ca = 1.0 / a.ca;
  a.inv_alpha = 1.0 / h->alpha;
  if (h->phys_deposit == ST_DEPOSIT_CIC)
    adjoint_step_kernel<true><<<kAdjBlocks, kAdjThreads, 0, h->stream>>>(a);
  else
    adjoint_step_kernel<false><<<kAdjBlocks, kAdjThreads, 0, h->stream>>>(a);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_adjoint_segment(st_ctx* h, const AdjointStepArgs& s, int len) {
  if (!h->fluid_fix.p) return cudaErrorInvalidValue;
  SegArgs a;
  a.tape = s.x[0];
  a.d = s.d;
  for (int q = 0; q < 3; ++q) {
    a.xb[q] = s.xb[q];
    a.vb[q] = s.vb[q];
    a.g[q] = h->g[q];
  }
  a.scale = fix::make_scale(h->geo.inv_h);
  a.ab = s.db;
  a.mb = s.mb;
  a.last = s.last;
  a.ab_part = s.ab_part;
  a.U = (const fix::FixCell*)h->fluid_fix.p;
  a.lam = s.lam;
  a.Uw = s.Uw;
  a.n = h->np;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  a.len = len;
  a.dt = s.dt;
  a.inv_ca = h->rho_p / (18.0 * h->mu * h->alpha);
  a.mcoef = h->mult * h->rho_p * 3.14159265358979323846 / 6.0;
  a.inv_alpha = 1.0 / h->alpha;
  const int64_t blocks = std::min<int64_t>((h->np + kSegThreads - 1) / kSegThreads, kAdjBlocks);
  adjoint_segment_kernel<<<(int)std::max<int64_t>(blocks, 1), kSegThreads, 0, h->stream>>>(a);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_adjoint_segment_mixed(st_ctx* h, const AdjointMixedArgs& s) {
  AdjMixedArgs a;
  a.tape = (const char*)s.tape;
  a.tape_n = s.tape_n;
  a.len = s.len;
  a.d = s.d;
  for (int q = 0; q < 3; ++q) {
    a.xb[q] = s.xb[q];
    a.vb[q] = s.vb[q];
    a.inv_h[q] = (float)h->geo.inv_h[q];
    a.g[q] = (float)h->g[q];
    a.gdt[q] = (float)(h->g[q] * s.dt);
  }
  a.db = s.db;
  a.ab = s.ab;
  a.Up = (const float4*)h->fluid_pad.p;
  a.lam = s.lam32;
  a.Uw = s.Uw;
  a.n = h->np;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  const double ca = 18.0 * h->mu * h->alpha / h->rho_p;
  a.dt = (float)s.dt;
  a.cadt = (float)(ca * s.dt);
  a.inv_ca = (float)(1.0 / ca);
  a.mcoef = (float)(h->mult * h->rho_p * 3.14159265358979323846 / 6.0);
  const int64_t blocks = std::min<int64_t>((h->np + kSegThreads - 1) / kSegThreads, 152 * 64);
  adjoint_segment_mixed_kernel<<<(int)std::max<int64_t>(blocks, 1), kSegThreads, 0, h->stream>>>(a);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_ordered_sum(st_ctx* h, const double* in, int64_t n, double* part) {
  ordered_sum_kernel<<<kAdjBlocks, kAdjThreads, 0, h->stream>>>(in, n, part);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_f64_to_f32(st_ctx* h, const double* in, float* out, int64_t m) {
  int64_t b = (m + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  f64_to_f32_kernel<<<(int)b, 256, 0, h->stream>>>(in, out, m);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_wide_to_f64(st_ctx* h, const long long* Uw, double* out, int64_t m) {
  int64_t b = (m + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  wide_to_f64_kernel<<<(int)b, 256, 0, h->stream>>>(Uw, out, m);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace st
