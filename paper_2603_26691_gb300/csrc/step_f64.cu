// Plain FP64 Lagrangian step: one particle per lane, 32 consecutive particles
// per warp.  Gather -> exponential integrator -> wrap/relocate -> impulse,
// then a warp-segmented reduction of the impulses over runs of equal
// start-of-step cell in storage order, committed to the exact fixed-point
// source accumulator.  The physics variants (nearest-grid-point gather,
// semi-implicit Euler, Schiller-Naumann drag, cloud-in-cell deposit) are
// uniform branches on the step's parameters.  GB300's FP64 rate is low, so this kernel is bound by
// FP64 arithmetic rather than by HBM.
#include "fix_gather.cuh"
#include "st_common.cuh"

namespace st {
namespace {

struct F64Args {
  F64State s;
  const D4* __restrict__ U;
  long long* __restrict__ acc;
  int64_t n;
  int64_t ncell;
  int nx, ny, nz;
  double L[3], invL[3], inv_h[3];
  double inv_ca;  // 1 / ca = rho_p / (18 mu alpha)
  StepParams p;
};

__device__ __forceinline__ double wrap_pos(double x, double L, double invL) {
  double y = x - L * floor(x * invL);
  if (y < 0.0) y += L;
  if (y >= L) y = 0.0;
  return y;
}

__device__ __forceinline__ D4 ld_cell(const D4* __restrict__ U, int64_t c) {
  const double2* p = reinterpret_cast<const double2*>(U + c);
  double2 a = __ldg(p), b = __ldg(p + 1);
  return D4{a.x, a.y, b.x, b.y};
}

__device__ __forceinline__ void lerp3(D4 a, D4 b, double f, double r[3]) {
  r[0] = fma(f, b.x - a.x, a.x);
  r[1] = fma(f, b.y - a.y, a.y);
  r[2] = fma(f, b.z - a.z, a.z);
}

// Schiller-Naumann drag factor f = C_D Re / 24: 1 + 0.15 Re^0.687 up to Re = 1000, 0.44 Re / 24 above
__device__ __forceinline__ double sn_factor(double re) {
  return re <= 1000.0 ? 1.0 + 0.15 * pow(re, 0.687) : (0.44 / 24.0) * re;
}

// Warp-segmented sum of J over runs of equal key (lanes in storage order), one commit per run.
__device__ __forceinline__ void deposit_runs(const F64Args& a, int lane, int key, double j0, double j1, double j2) {
  const int prev = __shfl_up_sync(0xffffffffu, key, 1);
  const bool head = (lane == 0) || (prev != key);
  const unsigned heads = __ballot_sync(0xffffffffu, head);
  const unsigned above = lane == 31 ? 0u : (heads & ~((2u << lane) - 1u));
  const int end = above ? (__ffs(above) - 2) : 31;
  for (int off = 1; off < 32; off <<= 1) {
    double t0 = __shfl_down_sync(0xffffffffu, j0, off);
    double t1 = __shfl_down_sync(0xffffffffu, j1, off);
    double t2 = __shfl_down_sync(0xffffffffu, j2, off);
    if (lane + off <= end) {
      j0 += t0;
      j1 += t1;
      j2 += t2;
    }
  }
  if (a.acc && head && key >= 0) {
    acc_add_f64(a.acc + kAccWords * key, j0, a.p.E);
    acc_add_f64(a.acc + kAccWords * (a.ncell + key), j1, a.p.E);
    acc_add_f64(a.acc + kAccWords * (2 * a.ncell + key), j2, a.p.E);
  }
}

__global__ void __launch_bounds__(256) step_f64_kernel(const F64Args a) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int n3[3] = {a.nx, a.ny, a.nz};
  const int64_t row = a.nx, slab = (int64_t)a.nx * a.ny;
  for (int64_t base = warp * 32; base < a.n; base += nwarp * 32) {
    const int64_t p = base + lane;
    int key = -1;
    double J[3] = {0.0, 0.0, 0.0};
    int i0[3] = {0, 0, 0}, i1[3] = {0, 0, 0};
    double f[3] = {0.0, 0.0, 0.0};
    if (p < a.n) {
      double x[3], v[3];
      for (int q = 0; q < 3; ++q) {
        x[q] = a.s.x[q][p];
        v[q] = a.s.v[q][p];
      }
      const double d = a.s.d[p];
      // start-of-step cell and trilinear stencil on cell centres
      int c0[3];
      for (int q = 0; q < 3; ++q) {
        double sx = x[q] * a.inv_h[q];
        int i = (int)floor(sx);
        c0[q] = min(max(i, 0), n3[q] - 1);
        double s2 = sx - 0.5;
        double fl = floor(s2);
        int ii = (int)fl;
        f[q] = s2 - fl;
        i0[q] = ii < 0 ? ii + n3[q] : ii;
        i1[q] = ii + 1 >= n3[q] ? ii + 1 - n3[q] : ii + 1;
      }
      key = c0[0] + a.nx * (c0[1] + a.ny * c0[2]);
      double up[3];
      if (a.p.ngp) {
        // nearest grid point: the value of the cell holding the particle
        const D4 Uc = ld_cell(a.U, key);
        up[0] = Uc.x;
        up[1] = Uc.y;
        up[2] = Uc.z;
      } else {
        D4 U000 = ld_cell(a.U, i0[0] + row * i0[1] + slab * i0[2]);
        D4 U100 = ld_cell(a.U, i1[0] + row * i0[1] + slab * i0[2]);
        D4 U010 = ld_cell(a.U, i0[0] + row * i1[1] + slab * i0[2]);
        D4 U110 = ld_cell(a.U, i1[0] + row * i1[1] + slab * i0[2]);
        D4 U001 = ld_cell(a.U, i0[0] + row * i0[1] + slab * i1[2]);
        D4 U101 = ld_cell(a.U, i1[0] + row * i0[1] + slab * i1[2]);
        D4 U011 = ld_cell(a.U, i0[0] + row * i1[1] + slab * i1[2]);
        D4 U111 = ld_cell(a.U, i1[0] + row * i1[1] + slab * i1[2]);
        double r00[3], r10[3], r01[3], r11[3];
        lerp3(U000, U100, f[0], r00);
        lerp3(U010, U110, f[0], r10);
        lerp3(U001, U101, f[0], r01);
        lerp3(U011, U111, f[0], r11);
        for (int q = 0; q < 3; ++q) {
          const double r0 = fma(f[1], r10[q] - r00[q], r00[q]);
          const double r1 = fma(f[1], r11[q] - r01[q], r01[q]);
          up[q] = fma(f[2], r1 - r0, r0);
        }
      }
      // drag rate a = alpha f(Re) / tau, f = 1 for Stokes drag
      const double dd = d * d;
      // 1/a first (one division per particle: GB300 divides in FP64 by iteration), then a from it
      double inv_ra = dd * a.inv_ca;
      if (a.p.sn) {
        const double r0 = up[0] - v[0], r1 = up[1] - v[1], r2 = up[2] - v[2];
        inv_ra /= sn_factor(a.p.re_coef * sqrt(r0 * r0 + r1 * r1 + r2 * r2) * d);
      }
      const double ra = 1.0 / inv_ra;
      const double adt = ra * a.p.dt;
      const double m = a.p.mcoef * dd * d;
      if (a.p.semi) {
        // semi-implicit Euler: v' = (v + dt (a u_p + g)) / (1 + a dt), x' = x + dt v'
        const double inv_den = 1.0 / (1.0 + adt);
        for (int q = 0; q < 3; ++q) {
          const double vn = (v[q] + a.p.dt * (ra * up[q] + a.p.g[q])) * inv_den;
          const double xn = x[q] + a.p.dt * vn;
          J[q] = -m * ((vn - v[q]) - a.p.g[q] * a.p.dt);
          a.s.x[q][p] = wrap_pos(xn, a.L[q], a.invL[q]);
          a.s.v[q][p] = vn;
        }
      } else {
        // exponential integrator
        // 1 - e^{-a dt} from expm1; e^{-a dt} as its complement (absolute error ~1e-16, which is what
        // multiplies v - w), one FP64 exponential instead of two
        const double E1 = -expm1(-adt);
        const double E = 1.0 - E1;
        const double Qd = E1 * inv_ra;
        for (int q = 0; q < 3; ++q) {
          const double wt = up[q] + a.p.g[q] * inv_ra;
          const double vn = wt + (v[q] - wt) * E;
          const double xn = x[q] + (wt * a.p.dt + (v[q] - wt) * Qd);
          J[q] = -m * ((vn - v[q]) - a.p.g[q] * a.p.dt);
          a.s.x[q][p] = wrap_pos(xn, a.L[q], a.invL[q]);
          a.s.v[q][p] = vn;
        }
      }
    }
    if (!a.p.cic) {
      deposit_runs(a, lane, key, J[0], J[1], J[2]);
    } else {
      // cloud in cell: the eight cells of the start-of-step trilinear stencil, each its own pass of
      // runs over the warp (sorted particles share corners, so runs stay long)
      for (int c = 0; c < 8; ++c) {
        const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
        const double w = (dx ? f[0] : 1.0 - f[0]) * (dy ? f[1] : 1.0 - f[1]) * (dz ? f[2] : 1.0 - f[2]);
        const int kc = key < 0 ? -1 : (dx ? i1[0] : i0[0]) + a.nx * ((dy ? i1[1] : i0[1]) + a.ny * (dz ? i1[2] : i0[2]));
        deposit_runs(a, lane, kc, w * J[0], w * J[1], w * J[2]);
      }
    }
  }
}

// The default physics (trilinear gather, exponential integrator, Stokes drag, cell deposit), nsteps steps per
// launch, bound by what is left on the FP64 pipe.  There an FP64 instruction costs 64 issue cycles, so:
//   * the gather runs on integers (fix_gather.cuh): about 400 issue cycles instead of 45 FP64 instructions;
//   * what the diameter alone decides (the exponential and the division) is computed once per launch: the
//     field is frozen, so a launch takes the steps up to the next sort one particle after the other, with
//     the state in registers;
//   * positions inside the box, told by their bits, need no wrap;
//   * the impulses are converted to the accumulator's integers at once and summed as 128-bit integers, over
//     the steps a particle stays in a cell and then over the warp's lanes of equal cell: exact, so the
//     sources do not depend on the storage order or on how steps are split over launches.
// 21 to 24 FP64 instructions are left per particle and step (2 to 3 per axis for the position and cell, 5 for the
// motion and the impulse; 59 in a launch of a single step, with what the diameter decides), against 134.  3e7 particles
// on 128^3, ten steps: 17.7 ms against 84.7 ms.
struct FixArgs {
  const double* in[6];              // position and velocity before the steps
  F64State s;                       // after them (the same arrays, or others); diameters
  double* __restrict__ tape;        // null, or where the state before step tape_first goes (x, v: 6 n values), the
  int tape_first, tape_every;       // one tape_every steps later 6 n values behind it, and so on
  const fix::FixCell* __restrict__ U;
  long long* __restrict__ acc;  // null: no deposit (the adjoint's recomputation)
  int64_t n, ncell;
  int nx, ny, nz, nsteps, E;
  double L[3], invL[3];
  fix::Scale scale;
  double dt, inv_ca, mcoef, g[3];
};

// a += round(x 2^E), |x| 2^E < 2^100
__device__ __forceinline__ void add_fixed(__int128& a, double x, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long man = b & 0xfffffffffffffull;
  if (ex != 0) man |= 1ull << 52;
  const int s = (ex == 0 ? 1 : ex) - 1075 + E;
  unsigned long long lo, hi = 0;
  if (__builtin_expect(s < 0, 0)) {
    lo = s > -64 ? (man + ((1ull << -s) >> 1)) >> -s : 0ull;
  } else {
    const int k = min(s, 63);
    lo = man << k;
    hi = k ? man >> (64 - k) : 0ull;
  }
  const __int128 t = (__int128)(((unsigned __int128)hi << 64) | lo);
  a += (b >> 63) ? -t : t;
}

// an integer in units of 2^-E to a cell's words: its magnitude's digits with its sign
__device__ __forceinline__ void commit_fixed(long long* p, __int128 v) {
  const bool neg = v < 0;
  const unsigned __int128 m = neg ? -(unsigned __int128)v : (unsigned __int128)v;
#pragma unroll
  for (int k = 0; k < kAccWords; ++k) {
    const long long d = (long long)(uint32_t)(m >> (32 * k));
    if (d) atomicAdd((unsigned long long*)&p[k], (unsigned long long)(neg ? -d : d));
  }
}

__device__ __forceinline__ __int128 shfl_down(__int128 v, int off) {
  const unsigned long long lo = __shfl_down_sync(0xffffffffu, (unsigned long long)v, off);
  const unsigned long long hi = __shfl_down_sync(0xffffffffu, (unsigned long long)((unsigned __int128)v >> 64), off);
  return (__int128)(((unsigned __int128)hi << 64) | lo);
}

__global__ void __launch_bounds__(256, 2) step_f64_fixed_kernel(const FixArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int n3[3] = {a.nx, a.ny, a.nz};
  for (int64_t base = warp * 32; base < a.n; base += nwarp * 32) {
    const int64_t p = base + lane;
    const unsigned lanes = __ballot_sync(0xffffffffu, p < a.n);
    int key = -1;
    __int128 J[3] = {0, 0, 0};
    if (p < a.n) {
      double x[3], v[3];
      for (int q = 0; q < 3; ++q) {
        x[q] = a.in[q][p];
        v[q] = a.in[3 + q][p];
      }
      const double d = a.s.d[p];
      const double dd = d * d;
      const double inv_ra = dd * a.inv_ca;
      const double ra = 1.0 / inv_ra;
      // 1 - e^{-a dt} from expm1; e^{-a dt} as its complement (absolute error ~1e-16, which is what
      // multiplies v - w)
      const double E1 = -expm1(-ra * a.dt);
      const double E = 1.0 - E1;
      const double Q = E1 * inv_ra;
      const double m = a.mcoef * dd * d;
      const double mE1 = m * E1;
      double gi[3], mg[3];
      for (int q = 0; q < 3; ++q) {
        gi[q] = a.g[q] * inv_ra;
        mg[q] = m * (a.g[q] * a.dt);
      }
      double* slot = a.tape;
      int next = a.tape ? a.tape_first : a.nsteps;
#pragma unroll 1
      for (int step = 0; step < a.nsteps; ++step) {
        if (step == next) {
          for (int q = 0; q < 3; ++q) {
            slot[q * a.n + p] = x[q];
            slot[(3 + q) * a.n + p] = v[q];
          }
          slot += 6 * a.n;
          next += a.tape_every;
        }
        const fix::Stencil st = fix::stencil(x, a.scale, n3);
        const int k = st.c0[0] + a.nx * (st.c0[1] + a.ny * st.c0[2]);
        if (k != key) {
          if (key >= 0 && a.acc) {
            for (int q = 0; q < 3; ++q) {
              commit_fixed(a.acc + kAccWords * (q * a.ncell + key), J[q]);
              J[q] = 0;
            }
          }
          key = k;
        }
        __syncwarp(lanes);
        double up[3];
        fix::gather(a.U, st, a.nx, a.ny, up);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double wt = up[q] + gi[q];
          const double dvw = v[q] - wt;
          const double xn = x[q] + (wt * a.dt + dvw * Q);
          v[q] = wt + dvw * E;
          // m [(v - w)(1 - E) + g dt] = -m [(v' - v) - g dt]
          if (a.acc) add_fixed(J[q], dvw * mE1 + mg[q], a.E);
          // inside [0, L): the bits of non-negative doubles are ordered like the values
          x[q] = (unsigned long long)__double_as_longlong(xn) < (unsigned long long)__double_as_longlong(a.L[q])
                     ? xn
                     : wrap_pos(xn, a.L[q], a.invL[q]);
        }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        a.s.x[q][p] = x[q];
        a.s.v[q][p] = v[q];
      }
    }
    if (!a.acc) continue;
    // the impulses since each particle's last change of cell: runs of equal cell over the warp
    const int prev = __shfl_up_sync(0xffffffffu, key, 1);
    const bool head = (lane == 0) || (prev != key);
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    if (heads != 0xffffffffu) {
      const unsigned above = lane == 31 ? 0u : (heads & ~((2u << lane) - 1u));
      const int end = above ? (__ffs(above) - 2) : 31;
#pragma unroll 1
      for (int off = 1; off < 32; off <<= 1) {
        const __int128 t0 = shfl_down(J[0], off), t1 = shfl_down(J[1], off), t2 = shfl_down(J[2], off);
        if (lane + off <= end) {
          J[0] += t0;
          J[1] += t1;
          J[2] += t2;
        }
      }
    }
    if (head && key >= 0)
      for (int q = 0; q < 3; ++q) commit_fixed(a.acc + kAccWords * (q * a.ncell + key), J[q]);
  }
}

}  // namespace

cudaError_t launch_step_f64(st_ctx* h, const StepParams& p) {
  return launch_step_f64_state(h, carve_f64(h->state.p, h->cap), (long long*)h->acc.p, p);
}

bool fixed_step_supported(const st_ctx* h) {
  return h->prec == ST_FP64 && h->fluid_fix.p && !h->micro_on && default_physics(h);
}

cudaError_t launch_step_f64_tape(st_ctx* h, const double* const (&in)[6], const F64State& s, long long* acc,
                                 const StepParams& p, double* tape, int first, int every) {
  if (!h->fluid_fix.p) return cudaErrorInvalidValue;
  FixArgs a;
  for (int k = 0; k < 6; ++k) a.in[k] = in[k];
  a.s = s;
  a.tape = tape;
  a.tape_first = first;
  a.tape_every = every;
  a.U = (const fix::FixCell*)h->fluid_fix.p;
  a.acc = acc;
  a.n = h->np;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  a.nsteps = p.nsteps;
  a.E = p.E;
  for (int q = 0; q < 3; ++q) {
    a.L[q] = h->geo.L[q];
    a.invL[q] = 1.0 / h->geo.L[q];
    a.g[q] = p.g[q];
  }
  a.scale = fix::make_scale(h->geo.inv_h);
  a.dt = p.dt;
  a.inv_ca = 1.0 / p.ca;
  a.mcoef = p.mcoef;
  const int64_t blocks = std::min<int64_t>((h->np + 255) / 256, 152 * 32);
  step_f64_fixed_kernel<<<(int)std::max<int64_t>(blocks, 1), 256, 0, h->stream>>>(a);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_step_f64_state(st_ctx* h, const F64State& s, long long* acc, const StepParams& p) {
  if (fixed_step_supported(h)) {
    const double* in[6] = {s.x[0], s.x[1], s.x[2], s.v[0], s.v[1], s.v[2]};
    return launch_step_f64_tape(h, in, s, acc, p, nullptr, 0, 1);
  }
  if (p.nsteps != 1) return cudaErrorInvalidValue;
  F64Args a;
  a.s = s;
  a.U = (const D4*)h->fluid.p;
  a.acc = acc;
  a.n = h->np;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  for (int q = 0; q < 3; ++q) {
    a.L[q] = h->geo.L[q];
    a.invL[q] = 1.0 / h->geo.L[q];
    a.inv_h[q] = h->geo.inv_h[q];
  }
  a.p = p;
  a.inv_ca = 1.0 / p.ca;
  int64_t warps = (h->np + 31) / 32;
  int64_t blocks = (warps * 32 + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (blocks < 1) blocks = 1;
  step_f64_kernel<<<(int)blocks, 256, 0, h->stream>>>(a);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace st
