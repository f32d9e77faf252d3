// Mixed-precision Lagrangian step: int32 packed cell + FP32 in-cell offset,
// FP32 (or BF16) velocity, FP32 diameter; FP32 arithmetic.  Each lane owns 4
// consecutive particles (2 where nothing is deposited), so every particle array is read and
// written with wide coalesced accesses; a warp covers 128
// particles.  Impulses are reduced over runs of equal start-of-step cell in
// storage order (lane-local suffix sums, then a segmented suffix scan across
// lanes) and each run is committed once to the exact fixed-point accumulator.
// The physics variants (nearest-grid-point gather, semi-implicit Euler,
// Schiller-Naumann drag) are uniform branches; the cloud-in-cell deposit is a
// template instance that runs the run-sum once per stencil corner.
// The field is frozen over a call and particles do not act on each other, so a launch takes the steps up to
// the next sort for one set of particles after the other, their state in registers; each step's runs are
// those of one step per launch, so the results do not depend on how the steps are split over launches.
// 2e6 particles on 100 x 84 x 60, ten steps: 0.49 ms against 0.68 ms.
// Bound by the latency of the gathers (from L1 and L2) and of the deposit's reductions at 16 warps an SM (126
// registers; 24 and 32 warps with spills: 0.52 and 0.59 ms).  Two particles per lane in 64 registers take 0.44 ms, but
// would sum in another order: the last bit of a sum, and through a coupled fluid of the velocities, would change.
// Without a deposit, as the adjoint recomputes its segments, there is no order to keep: two per lane (1e7 particles on
// 64^3, 40 steps forward and 38 recomputed: 11.05 ms against 11.7 ms).
#include <cstring>

#include "st_common.cuh"

namespace st {
namespace {

struct MixedArgs {
  MixedState in, s;   // the state before and after the steps (the same arrays, or others); diameters in `in`
  char* tape;         // null, or where the state before step tape_first goes (cells, offsets, velocities at a
  int64_t tape_n;     // stride of tape_n particles), the one tape_every steps later behind it, and so on
  int tape_first, tape_every, nsteps;
  const float4* __restrict__ U;
  long long* __restrict__ acc;
  int64_t n;
  int64_t ncell;
  int nx, ny, nz;
  float inv_h[3];
  float dt, cadt, inv_ca, mcoef;
  float g[3], gdt[3];
  int E;
  int ngp, semi, sn;  // nearest-grid-point gather, semi-implicit Euler, Schiller-Naumann drag
  float re_coef;      // rho_f / mu
};

__device__ __forceinline__ void lerp3(float4 a, float4 b, float f, float r[3]) {
  r[0] = fmaf(f, b.x - a.x, a.x);
  r[1] = fmaf(f, b.y - a.y, a.y);
  r[2] = fmaf(f, b.z - a.z, a.z);
}

__device__ __forceinline__ void commit(const MixedArgs& a, int key, float j0, float j1, float j2) {
  acc_add_f32(a.acc + kAccWords * key, j0, a.E);
  acc_add_f32(a.acc + kAccWords * (a.ncell + key), j1, a.E);
  acc_add_f32(a.acc + kAccWords * (2 * a.ncell + key), j2, a.E);
}

// particles per lane
template <bool DEP>
constexpr int kPerLane = DEP ? 4 : 2;

// P values of a lane, one access, streaming
template <int P, class T>
__device__ __forceinline__ void ld(const T* p, T (&v)[P]) {
  if constexpr (P == 4) {
    const float4 r = __ldcs((const float4*)p);
    memcpy(v, &r, sizeof(r));
  } else {
    const float2 r = __ldcs((const float2*)p);
    memcpy(v, &r, sizeof(r));
  }
}
template <int P, class T>
__device__ __forceinline__ void st(T* p, const T (&v)[P]) {
  if constexpr (P == 4) {
    float4 r;
    memcpy(&r, v, sizeof(r));
    __stcs((float4*)p, r);
  } else {
    float2 r;
    memcpy(&r, v, sizeof(r));
    __stcs((float2*)p, r);
  }
}

template <bool BF16, int P>
__device__ __forceinline__ void load_v(const MixedArgs& a, int q, int64_t p0, float (&v)[P]) {
  if constexpr (BF16) {
    __nv_bfloat162 r[P / 2];
    if constexpr (P == 4) {
      const uint2 u = __ldcs((const uint2*)((const __nv_bfloat16*)a.in.v[q] + p0));
      memcpy(r, &u, sizeof(u));
    } else {
      const unsigned u = __ldcs((const unsigned*)((const __nv_bfloat16*)a.in.v[q] + p0));
      memcpy(r, &u, sizeof(u));
    }
#pragma unroll
    for (int i = 0; i < P / 2; ++i) {
      const float2 f = __bfloat1622float2(r[i]);
      v[2 * i] = f.x;
      v[2 * i + 1] = f.y;
    }
  } else {
    ld((const float*)a.in.v[q] + p0, v);
  }
}

template <bool BF16, int P>
__device__ __forceinline__ void store_v(const MixedArgs& a, int q, int64_t p0, const float (&v)[P]) {
  if constexpr (BF16) {
    __nv_bfloat162 r[P / 2];
#pragma unroll
    for (int i = 0; i < P / 2; ++i) r[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    if constexpr (P == 4) {
      uint2 u;
      memcpy(&u, r, sizeof(u));
      __stcs((uint2*)((__nv_bfloat16*)a.s.v[q] + p0), u);
    } else {
      unsigned u;
      memcpy(&u, r, sizeof(u));
      __stcs((unsigned*)((__nv_bfloat16*)a.s.v[q] + p0), u);
    }
  } else {
    st((float*)a.s.v[q] + p0, v);
  }
}

// round a velocity to its stored precision
template <bool BF16>
__device__ __forceinline__ float stored(float v) {
  if (BF16) return __bfloat162float(__float2bfloat16_rn(v));
  return v;
}

// periodic index for a particle that moved more than a box length in one step (rare)
__device__ __noinline__ int wrap_index_slow(int ii, int n) {
  ii %= n;
  return ii < 0 ? ii + n : ii;
}

// cell index after a move of 2^22 cells or more in one step (rare); the offset is set here too
__device__ __noinline__ int relocate_far(float& o, int ci, int n) {
  const float fl = floorf(o);
  o = fmaxf(fminf(o - fl, 0.99999994f), 0.0f);
  long long k = ((long long)ci + (long long)fl) % n;
  return (int)(k < 0 ? k + n : k);
}

// Sums J over runs of equal key in the warp's particles (kP consecutive per lane) and commits
// each run once to the fixed-point accumulator: lane-local suffix sums, then a segmented suffix
// scan across lanes.  Negative keys are skipped.
template <int kP>
__device__ __forceinline__ void deposit_runs(const MixedArgs& a, int lane, const int (&key)[kP], const float (&J)[kP][3]) {
  // lane-local suffix sums S_j over the run that starts at j
  float S[kP][3];
#pragma unroll
  for (int q = 0; q < 3; ++q) S[kP - 1][q] = J[kP - 1][q];
  int tail = kP - 1;  // first element of the run that ends the lane (the lane's tail run)
#pragma unroll
  for (int j = kP - 2; j >= 0; --j) {
    const bool same = key[j] == key[j + 1];
    if (same && tail == j + 1) tail = j;
#pragma unroll
    for (int q = 0; q < 3; ++q) S[j][q] = J[j][q] + (same ? S[j + 1][q] : 0.0f);
  }
  // the lanes whose trailing run goes on in the next lane's leading run, and those that are one run
  const int nk0 = __shfl_down_sync(0xffffffffu, key[0], 1);
  const unsigned links = __ballot_sync(0xffffffffu, lane < 31 && nk0 == key[kP - 1] && key[kP - 1] >= 0);
  const unsigned whole = __ballot_sync(0xffffffffu, tail == 0);
  float A[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float t = __shfl_down_sync(0xffffffffu, S[0][q], 1);
    A[q] = (links >> lane) & 1u ? t : 0.0f;
  }
  // segmented suffix scan R_l = A_l + B_l R_{l+1}; through: the lanes from which the next `off` lanes are one run (the
  // scan ends with the last of them)
  unsigned through = links & (whole >> 1);
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    if (through == 0u) break;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float t = __shfl_down_sync(0xffffffffu, A[q], off);
      if ((through >> lane) & 1u) A[q] += t;
    }
    through &= through >> off;
  }
  const bool head_lane = lane == 0 || !((links >> (lane - 1)) & 1u);
#pragma unroll
  for (int j = 0; j < kP; ++j) {
    const bool start = (j == 0) ? head_lane : (key[j] != key[j - 1]);
    if (start && key[j] >= 0) {
      const bool to_end = j == tail;  // only the tail run continues into the next lane
      commit(a, key[j], S[j][0] + (to_end ? A[0] : 0.0f), S[j][1] + (to_end ? A[1] : 0.0f),
             S[j][2] + (to_end ? A[2] : 0.0f));
    }
  }
}

// Schiller-Naumann drag factor f = C_D Re / 24: 1 + 0.15 Re^0.687 up to Re = 1000, 0.44 Re / 24 above
__device__ __forceinline__ float sn_factor(float re) {
  return re <= 1000.0f ? fmaf(0.15f, powf(re, 0.687f), 1.0f) : (0.44f / 24.0f) * re;
}

// the coefficients of a step at drag rate a = alpha f(Re) / tau (f = 1 for Stokes drag), from a dt and 1 / a;
// both integrators take the form v' = w + (v - w) E, x' = x + w dt + (v - w) Q with w = u_p + g / a:
//   exponential:         E = e^{-a dt},       Q = (1 - E) / a
//   semi-implicit Euler: E = 1 / (1 + a dt),  Q = E dt  (x' = x + dt v')
__device__ __forceinline__ void drag(const MixedArgs& a, float adt, float inv_a, float& E, float& Q) {
  if (a.semi) {
    E = 1.0f / (1.0f + adt);
    Q = E * a.dt;
  } else {
    const float E1 = -expm1f(-adt);  // 1 - e^{-a dt}
    E = 1.0f - E1;
    Q = E1 * inv_a;
  }
}

// DEP: the impulses are deposited (CIC: cloud in cell); ONE: one step and no tape, without the loop
// (ten single steps of 2e7 particles on 100 x 84 x 60: 5.08 -> 4.93 ms, of 2e6 0.73 -> 0.71)
template <bool BF16, bool CIC, bool DEP, bool ONE>
__global__ void __launch_bounds__(256, DEP ? 2 : 4) step_mixed_kernel(const MixedArgs a) {
  constexpr int kP = kPerLane<DEP>, kPW = 32 * kP;  // particles per lane, per warp
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int n3[3] = {a.nx, a.ny, a.nz};
  for (int64_t base = warp * kPW; base < a.n; base += nwarp * kPW) {
    const int64_t p0 = base + lane * kP;
    {
      // pull the next iteration's particle lines towards L2 while this one computes
      const int64_t pn = p0 + nwarp * kPW;
      if (pn < a.n) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.in.cell + pn));
        for (int q = 0; q < 3; ++q) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.in.xi[q] + pn));
        for (int q = 0; q < 3; ++q)
          asm volatile("prefetch.global.L2 [%0];" ::"l"((const char*)a.in.v[q] + pn * (BF16 ? 2 : 4)));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.in.d + pn));
      }
    }
    int cell[kP];
    float xi[3][kP], v[3][kP], dv[kP];
    const int nvalid = (int)max((int64_t)0, min((int64_t)kP, a.n - p0));
    if (nvalid > 0) {
      ld(a.in.cell + p0, cell);
      for (int q = 0; q < 3; ++q) ld(a.in.xi[q] + p0, xi[q]);
      for (int q = 0; q < 3; ++q) load_v<BF16>(a, q, p0, v[q]);
      ld(a.in.d + p0, dv);
    }
    // Stokes drag is decided by the diameter alone
    float Ec[kP], Qc[kP];
    if (!a.sn && nvalid > 0) {
#pragma unroll
      for (int j = 0; j < kP; ++j) {
        const float dd = dv[j] * dv[j];
        drag(a, a.cadt / dd, dd * a.inv_ca, Ec[j], Qc[j]);
      }
    }
    char* slot = a.tape;
    int next = ONE ? -1 : a.tape ? a.tape_first : a.nsteps;
#pragma unroll 1
    for (int step = 0; step < (ONE ? 1 : a.nsteps); ++step) {
      int key[kP];
      float J[kP][3];
#pragma unroll
      for (int j = 0; j < kP; ++j) {
        key[j] = -1;
        J[j][0] = J[j][1] = J[j][2] = 0.0f;
      }
      // cloud-in-cell deposit: the start-of-step stencil's lower corner (periodic) and weights
      int sb[CIC ? kP : 1][3];
      float sf[CIC ? kP : 1][3];
      if (!ONE && step == next) {
        if (nvalid > 0) {
          float* f = (float*)slot;
          st((int*)slot + p0, cell);
          for (int q = 0; q < 3; ++q) {
            st(f + (1 + q) * a.tape_n + p0, xi[q]);
            st(f + (4 + q) * a.tape_n + p0, v[q]);
          }
        }
        slot += 28 * a.tape_n;
        next += a.tape_every;
      }
      if (nvalid > 0) {
#pragma unroll
        for (int j = 0; j < kP; ++j) {
          if (j < nvalid) {
            const int ci[3] = {cell_i(cell[j]), cell_j(cell[j]), cell_k(cell[j])};
            key[j] = ci[0] + a.nx * (ci[1] + a.ny * ci[2]);
            // trilinear stencil from (cell, offset): centres at offset 1/2; the field carries
            // kFluidPad ghost layers, so corner indices ii and ii + 1 (ii in [-1, n-1]) need no wrap
            int i0[3];
            float f[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const float o = xi[q][j];
              const bool hi = o >= 0.5f;
              i0[q] = ci[q] - (hi ? 0 : 1) + kFluidPad;
              f[q] = o + (hi ? -0.5f : 0.5f);
              if (CIC) {
                const int lo = i0[q] - kFluidPad;
                sb[CIC ? j : 0][q] = lo < 0 ? lo + n3[q] : lo;
                sf[CIC ? j : 0][q] = f[q];
              }
            }
            const int64_t row = a.nx + 2 * kFluidPad, slab = row * (a.ny + 2 * kFluidPad);
            float up[3];
            if (a.ngp) {
              // nearest grid point: the value of the cell holding the particle
              const float4 Uc = __ldg(a.U + (ci[0] + kFluidPad) + row * (ci[1] + kFluidPad) + slab * (ci[2] + kFluidPad));
              up[0] = Uc.x;
              up[1] = Uc.y;
              up[2] = Uc.z;
            } else {
              const float4* b = a.U + i0[0] + row * i0[1] + slab * i0[2];
              const float4 U000 = __ldg(b);
              const float4 U100 = __ldg(b + 1);
              const float4 U010 = __ldg(b + row);
              const float4 U110 = __ldg(b + row + 1);
              const float4 U001 = __ldg(b + slab);
              const float4 U101 = __ldg(b + slab + 1);
              const float4 U011 = __ldg(b + slab + row);
              const float4 U111 = __ldg(b + slab + row + 1);
              float r00[3], r10[3], r01[3], r11[3];
              lerp3(U000, U100, f[0], r00);
              lerp3(U010, U110, f[0], r10);
              lerp3(U001, U101, f[0], r01);
              lerp3(U011, U111, f[0], r11);
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                const float r0 = fmaf(f[1], r10[q] - r00[q], r00[q]);
                const float r1 = fmaf(f[1], r11[q] - r01[q], r01[q]);
                up[q] = fmaf(f[2], r1 - r0, r0);
              }
            }
            const float dd = dv[j] * dv[j];
            float inv_a = dd * a.inv_ca;   // 1 / a
            float E = Ec[j], Q = Qc[j];
            if (a.sn) {
              const float r0 = up[0] - v[0][j], r1 = up[1] - v[1][j], r2 = up[2] - v[2][j];
              const float fac = sn_factor(a.re_coef * sqrtf(fmaf(r0, r0, fmaf(r1, r1, r2 * r2))) * dv[j]);
              inv_a /= fac;
              drag(a, a.cadt / dd * fac, inv_a, E, Q);
            }
            const float m = a.mcoef * dd * dv[j];
            int cn[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const float wt = fmaf(a.g[q], inv_a, up[q]);
              const float dvw = v[q][j] - wt;
              const float vn = stored<BF16>(fmaf(dvw, E, wt));
              const float dx = fmaf(wt, a.dt, dvw * Q);
              // relocate: offset in cell units, carry whole cells into the index (k = round(o - 1/2)
              // by the 1.5 * 2^23 shift: no rounding or conversion instructions)
              float o = fmaf(dx, a.inv_h[q], xi[q][j]);
              int ii;
              if (__builtin_expect(fabsf(o) < 4194304.0f, 1)) {
                const float t = (o - 0.5f) + 12582912.0f;
                ii = ci[q] + (__float_as_int(t) - 0x4B400000);
                o = o - (t - 12582912.0f);
                if (o >= 1.0f) {  // on the upper face: offset 0 of the next cell
                  o = 0.0f;
                  ii += 1;
                }
                o = fmaxf(o, 0.0f);
                if (ii >= n3[q]) ii -= n3[q];
                else if (ii < 0) ii += n3[q];
                if (__builtin_expect((unsigned)ii >= (unsigned)n3[q], 0)) ii = wrap_index_slow(ii, n3[q]);
              } else {
                ii = relocate_far(o, ci[q], n3[q]);
              }
              cn[q] = ii;
              xi[q][j] = o;
              J[j][q] = -m * ((vn - v[q][j]) - a.gdt[q]);
              v[q][j] = vn;
            }
            cell[j] = pack_cell(cn[0], cn[1], cn[2]);
          }
        }
      }
      // ---- deposit: runs of equal key over the warp's 128 particles ----
      if (!DEP) {
      } else if (!CIC) {
        deposit_runs(a, lane, key, J);
      } else {
        // cloud in cell: one pass of runs per stencil corner (sorted particles share corners)
#pragma unroll 1
        for (int c = 0; c < 8; ++c) {
          const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
          int kc[kP];
          float Jc[kP][3];
#pragma unroll
          for (int j = 0; j < kP; ++j) {
            const float* fj = sf[CIC ? j : 0];
            const int* bj = sb[CIC ? j : 0];
            const float w = (dx ? fj[0] : 1.0f - fj[0]) * (dy ? fj[1] : 1.0f - fj[1]) * (dz ? fj[2] : 1.0f - fj[2]);
            int ix = bj[0] + dx, iy = bj[1] + dy, iz = bj[2] + dz;
            ix = ix >= a.nx ? ix - a.nx : ix;
            iy = iy >= a.ny ? iy - a.ny : iy;
            iz = iz >= a.nz ? iz - a.nz : iz;
            kc[j] = key[j] < 0 ? -1 : ix + a.nx * (iy + a.ny * iz);
#pragma unroll
            for (int q = 0; q < 3; ++q) Jc[j][q] = w * J[j][q];
          }
          deposit_runs(a, lane, kc, Jc);
        }
      }
    }
    if (nvalid > 0) {
      st(a.s.cell + p0, cell);
      for (int q = 0; q < 3; ++q) st(a.s.xi[q] + p0, xi[q]);
      for (int q = 0; q < 3; ++q) store_v<BF16>(a, q, p0, v[q]);
    }
  }
}

}  // namespace

cudaError_t launch_step_mixed(st_ctx* h, const StepParams& p) {
  const MixedState s = carve_mixed(h->state.p, h->cap, h->prec == ST_MIXED_BF16V);
  return launch_step_mixed_tape(h, s, s, h->np, (long long*)h->acc.p, p, nullptr, 0, 0, 1);
}

cudaError_t launch_step_mixed_tape(st_ctx* h, const MixedState& in, const MixedState& s, int64_t n, long long* acc,
                                   const StepParams& p, void* tape, int64_t tape_n, int first, int every) {
  MixedArgs a;
  bool bf = h->prec == ST_MIXED_BF16V;
  a.in = in;
  a.s = s;
  a.tape = (char*)tape;
  a.tape_n = tape_n;
  a.tape_first = first;
  a.tape_every = every;
  a.nsteps = p.nsteps;
  a.U = (const float4*)h->fluid_pad.p;
  a.acc = acc;
  a.n = n;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  for (int q = 0; q < 3; ++q) {
    a.inv_h[q] = (float)h->geo.inv_h[q];
    a.g[q] = (float)p.g[q];
    a.gdt[q] = (float)(p.g[q] * p.dt);
  }
  a.dt = (float)p.dt;
  a.cadt = (float)(p.ca * p.dt);
  a.inv_ca = (float)(1.0 / p.ca);
  a.mcoef = (float)p.mcoef;
  a.E = p.E;
  a.ngp = p.ngp;
  a.semi = p.semi;
  a.sn = p.sn;
  a.re_coef = (float)p.re_coef;
  const int per_warp = 32 * (acc ? kPerLane<true> : kPerLane<false>);
  const int64_t warps = (n + per_warp - 1) / per_warp;
  int64_t blocks = (warps * 32 + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  const bool one = p.nsteps == 1 && !tape;
  static void (*const dep[8])(const MixedArgs) = {
      step_mixed_kernel<false, false, true, false>, step_mixed_kernel<true, false, true, false>,
      step_mixed_kernel<false, true, true, false>,  step_mixed_kernel<true, true, true, false>,
      step_mixed_kernel<false, false, true, true>,  step_mixed_kernel<true, false, true, true>,
      step_mixed_kernel<false, true, true, true>,   step_mixed_kernel<true, true, true, true>};
  void (*kern)(const MixedArgs) = acc  ? dep[(int)bf + 2 * (int)(p.cic != 0) + 4 * (int)one]
                                  : bf ? step_mixed_kernel<true, false, false, false>
                                       : step_mixed_kernel<false, false, false, false>;
  kern<<<(int)blocks, 256, 0, h->stream>>>(a);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace st
