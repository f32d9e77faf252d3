// What the two kernels for sorted particles share (step_mixed_tma.cu: several steps per launch, one step of few
// particles; step_mixed_tma_single.cu: one step of many): units and their tiles, the arithmetic of a step, the deposit
// tile's digits, commits outside it, the sort's gather, and the launch arguments.  The two agree to the bit, so whatever
// rounds is here or, in the step itself, written in operations that the compiler does not contract.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "st_common.cuh"
#include "st_ptx.cuh"

namespace st {
namespace {

using namespace ptx;

constexpr int kU = 8;                       // unit edge (cells)
constexpr int kG = 3;                       // fluid halo = padding of the field
constexpr int kTE = kU + 2 * kG;            // fluid tile edge (14)
constexpr int kR = 2;                       // deposit halo
constexpr int kDE = kU + 2 * kR;            // deposit tile edge (12)
constexpr int kDepositCells = kDE * kDE * kDE;  // 1728
constexpr int kDigits = 3;                  // 15-bit digits per value in the shared deposit tile
constexpr int kDigitBits = 15;
constexpr int kDepShift = 51;               // shared tile units = global units * 2^kDepShift
constexpr int kFluidBytes = kTE * kTE * kTE * 16;               // 43904
constexpr int kDepositBytes = kDepositCells * 3 * kDigits * 4;  // 62208

__device__ __forceinline__ void tma_load_tile(void* dst, const CUtensorMap* map, int c1, int c2, int c3,
                                              uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(sptr(dst)),
      "l"(map), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(sptr(bar))
      : "memory");
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

struct TmaArgs {
  MixedState s;
  const float4* __restrict__ Up;      // ghost-padded field [nz+2G][ny+2G][nx+2G]
  long long* __restrict__ acc;
  const uint32_t* __restrict__ cell_start;
  int* __restrict__ err;
  unsigned* __restrict__ unit_ctr;    // next unit to hand out, CTAs that found none left (zero between launches)
  int64_t ncell;
  int nx, ny, nz;
  int nunits;                         // units of kU^3 cells in key order
  int logB, ncx, ncy;                 // chunk geometry for decoding a unit's origin
  float inv_h[3];
  float dt, cadt, inv_ca, mcoef;
  float g[3], gdt[3];
  int nsteps;                         // steps to take (1 .. kMaxFusedSteps)
  float s1, s2;                       // factors of the impulses on their way to deposit-tile units, 2^(kDepShift - E) of
                                      // the accumulator's (see the kernels)
  float4* __restrict__ rec;           // record output: two float4 per particle (see st_common.cuh)
  const uint32_t* __restrict__ perm;  // GATHER: storage index (old order) of each sorted position
  const float4* __restrict__ grec;    // GATHER: the records in the old order
  const uint32_t* __restrict__ ids_in;   // GATHER: ids in the old order
  uint32_t* __restrict__ ids_out;        // GATHER: ids in sorted order
  int ngp, semi, sn, cic;             // physics variants (the PHYS instances): nearest grid point, semi-implicit Euler,
  float re_coef;                      // Schiller-Naumann drag (Re = re_coef |u-v| d), cloud-in-cell deposit (the
                                      // multi-step kernel's alone)
};

// de-interleave 3 bits per level (local x bit lowest)
__device__ __forceinline__ uint32_t compact3(uint32_t v) {
  v &= 0x09249249u;
  v = (v | (v >> 2)) & 0x030c30c3u;
  v = (v | (v >> 4)) & 0x0300f00fu;
  v = (v | (v >> 8)) & 0xff0000ffu;
  v = (v | (v >> 16)) & 0x000003ffu;
  return v;
}

__device__ __forceinline__ void unit_origin(const TmaArgs& a, int u, int& ox, int& oy, int& oz) {
  const uint32_t key = (uint32_t)u * (kU * kU * kU);
  const uint32_t chunk = key >> (3 * a.logB);
  const uint32_t m = key & ((1u << (3 * a.logB)) - 1u);
  const int B = 1 << a.logB;
  const int cx = (int)(chunk % (uint32_t)a.ncx);
  const int cy = (int)((chunk / (uint32_t)a.ncx) % (uint32_t)a.ncy);
  const int cz = (int)(chunk / ((uint32_t)a.ncx * (uint32_t)a.ncy));
  ox = cx * B + (int)compact3(m);
  oy = cy * B + (int)compact3(m >> 1);
  oz = cz * B + (int)compact3(m >> 2);
}

template <bool BF16>
__device__ __forceinline__ int stage_bytes(int cnt) {
  return cnt * (BF16 ? 26 : 32);
}

// cell and offset of a coordinate that the fast relocation cannot take (rare): a move of 2^22 cells
// or more, or of more than one box length, in one step; the cell carried is floor(o) reduced
// periodically (fmodf is exact), the offset o - floor(o)
struct Relocated {
  int cell;
  float offset;
};
__device__ __noinline__ Relocated relocate_general(float o, int ci, int n) {
  if (!(fabsf(o) <= 3.0e38f)) return Relocated{ci, 0.5f};  // non-finite: keep the cell
  const float fl = floorf(o);
  int k = (ci + (int)fmodf(fl, (float)n)) % n;
  return Relocated{k < 0 ? k + n : k, fmaxf(fminf(o - fl, 0.99999994f), 0.0f)};
}

// two-lane FP32 arithmetic (one instruction for a register pair; round-to-nearest, no flush to
// zero, so each lane rounds exactly as the scalar operation would)
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long add_rm2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long dup2(float a) { return pack2(a, a); }
// lerp c0 + w (c1 - c0) on the (x, y) pair
__device__ __forceinline__ unsigned long long lerp2(unsigned long long w, unsigned long long c0, unsigned long long c1) {
  return fma2(w, sub2(c1, c0), c0);
}

// 1 - e^{-x} for a pair of arguments x >= 0 (*E = e^{-x}): the degree-5 Taylor polynomial in
// Horner form for x < 1/8 (truncation below 5e-8 relative), else 1 - 2^(-x log2 e); the polynomial
// as pair operations, the exponentials and the choice per lane
__device__ __forceinline__ unsigned long long one_minus_exp2(unsigned long long X, unsigned long long* E) {
  float x0, x1, a0, a1;
  unpack2(mul2(X, dup2(-1.4426950408889634f)), a0, a1);
  float ex0, ex1;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex0) : "f"(a0));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex1) : "f"(a1));
  unsigned long long S = fma2(X, dup2(1.0f / 120.0f), dup2(-1.0f / 24.0f));
  S = fma2(X, S, dup2(1.0f / 6.0f));
  S = fma2(X, S, dup2(-0.5f));
  S = fma2(X, S, dup2(1.0f));
  float s0, s1;
  unpack2(mul2(X, S), s0, s1);
  unpack2(X, x0, x1);
  const float r0 = x0 < 0.125f ? s0 : 1.0f - ex0;
  const float r1 = x1 < 0.125f ? s1 : 1.0f - ex1;
  *E = pack2(x0 < 0.125f ? 1.0f - r0 : ex0, x1 < 0.125f ? 1.0f - r1 : ex1);
  return pack2(r0, r1);
}

// trilinear interpolation of the 8 corner velocities (corner c_xyz, x fastest) at weights f: the
// x and y components as register pairs, z alone; the same operations and rounding per component
// as c0 + f (c1 - c0) applied along x, then y, then z
__device__ __forceinline__ void trilerp(const float4& c000, const float4& c100, const float4& c010,
                                        const float4& c110, const float4& c001, const float4& c101,
                                        const float4& c011, const float4& c111, float fx, float fy, float fz,
                                        float* up) {
  const unsigned long long FX = pack2(fx, fx), FY = pack2(fy, fy), FZ = pack2(fz, fz);
  const unsigned long long a = lerp2(FX, pack2(c000.x, c000.y), pack2(c100.x, c100.y));
  const unsigned long long b = lerp2(FX, pack2(c010.x, c010.y), pack2(c110.x, c110.y));
  const unsigned long long c = lerp2(FX, pack2(c001.x, c001.y), pack2(c101.x, c101.y));
  const unsigned long long d = lerp2(FX, pack2(c011.x, c011.y), pack2(c111.x, c111.y));
  const unsigned long long e = lerp2(FY, a, b), g = lerp2(FY, c, d);
  unpack2(lerp2(FZ, e, g), up[0], up[1]);
  const float az = fmaf(fx, c100.z - c000.z, c000.z), bz = fmaf(fx, c110.z - c010.z, c010.z);
  const float cz = fmaf(fx, c101.z - c001.z, c001.z), dz = fmaf(fx, c111.z - c011.z, c011.z);
  const float ez = fmaf(fy, bz - az, az), gz = fmaf(fy, dz - cz, cz);
  up[2] = fmaf(fz, gz - ez, ez);
}

// fluid velocity of a particle outside its unit's tile, from the ghost-padded field (L2); the same
// stencil and arithmetic as the tile path
__device__ __noinline__ float3 gather_padded(const float4* __restrict__ Up, int px, int pxy, int cell, float o0,
                                             float o1, float o2) {
  const int ci[3] = {cell_i(cell), cell_j(cell), cell_k(cell)};
  const float o[3] = {o0, o1, o2};
  int i0[3];
  float f[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const bool hi2 = o[q] >= 0.5f;
    i0[q] = ci[q] - (hi2 ? 0 : 1);
    f[q] = o[q] + (hi2 ? -0.5f : 0.5f);
  }
  const float4* g = Up + (i0[0] + kG) + (int64_t)px * (i0[1] + kG) + (int64_t)pxy * (i0[2] + kG);
  float up[3];
  trilerp(__ldg(g), __ldg(g + 1), __ldg(g + px), __ldg(g + px + 1), __ldg(g + pxy), __ldg(g + pxy + 1),
          __ldg(g + pxy + px), __ldg(g + pxy + px + 1), f[0], f[1], f[2], up);
  return make_float3(up[0], up[1], up[2]);
}

// nearest-grid-point value of a particle outside its unit's tile, from the ghost-padded field
__device__ __noinline__ float3 ngp_padded(const float4* __restrict__ Up, int px, int pxy, int cell) {
  const float4 u = __ldg(Up + (cell_i(cell) + kG) + (int64_t)px * (cell_j(cell) + kG) + (int64_t)pxy * (cell_k(cell) + kG));
  return make_float3(u.x, u.y, u.z);
}

// Schiller-Naumann drag factor f = C_D Re / 24: 1 + 0.15 Re^0.687 up to Re = 1000 (the power from
// the hardware base-2 logarithm and exponential), 0.44 Re / 24 above
__device__ __forceinline__ float sn_factor(float re) {
  float l, p;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(re));
  const float y = 0.687f * l;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"(y));
  return re <= 1000.0f ? fmaf(0.15f, p, 1.0f) : (0.44f / 24.0f) * re;
}

// One cell's value in the shared deposit tile: three signed digits in int32 words (w[0] + 2^15 w[kDepositCells] +
// 2^30 w[2 kDepositCells], the components kDigits kDepositCells words apart).  digits1 and digits2 split a value t in
// tile units, |t| < 2^45, exactly into balanced digits of round(t) by round-to-nearest additions of 1.5 * 2^(23+b),
// which leave the nearest multiple of 2^b: t = 2^30 d2 + 2^15 d1 + d0 + (t - round(t)) with |d0|, |d1| <= 2^14 and
// |d2| <= 2^15; digits2 a register pair.  Integer atomics make the sums exact and independent of the order of the adds.
__device__ __forceinline__ void digits1(float t, int& d0, int& d1, int& d2) {
  const float h = __fsub_rn(__fadd_rn(t, 0x1.8p53f), 0x1.8p53f);  // multiple of 2^30
  const float l = __fsub_rn(t, h);                                  // |l| <= 2^29, exact
  const float m = __fsub_rn(__fadd_rn(l, 0x1.8p38f), 0x1.8p38f);  // multiple of 2^15
  const float l2 = __fsub_rn(l, m);                                 // |l2| <= 2^14, exact
  d2 = __float_as_int(__fmaf_rn(h, 0x1p-30f, 12582912.0f)) - 0x4B400000;
  d1 = __float_as_int(__fmaf_rn(m, 0x1p-15f, 12582912.0f)) - 0x4B400000;
  d0 = __float_as_int(__fadd_rn(l2, 12582912.0f)) - 0x4B400000;
}
__device__ __forceinline__ void digits2(unsigned long long t, int* d0, int* d1, int* d2) {
  const unsigned long long C53 = pack2(0x1.8p53f, 0x1.8p53f), C38 = pack2(0x1.8p38f, 0x1.8p38f);
  const unsigned long long C23 = pack2(12582912.0f, 12582912.0f);
  const unsigned long long h = sub2(add2(t, C53), C53);
  const unsigned long long l = sub2(t, h);
  const unsigned long long m = sub2(add2(l, C38), C38);
  const unsigned long long l2 = sub2(l, m);
  float a, b;
  unpack2(fma2(h, pack2(0x1p-30f, 0x1p-30f), C23), a, b);
  d2[0] = __float_as_int(a) - 0x4B400000;
  d2[1] = __float_as_int(b) - 0x4B400000;
  unpack2(fma2(m, pack2(0x1p-15f, 0x1p-15f), C23), a, b);
  d1[0] = __float_as_int(a) - 0x4B400000;
  d1[1] = __float_as_int(b) - 0x4B400000;
  unpack2(add2(l2, C23), a, b);
  d0[0] = __float_as_int(a) - 0x4B400000;
  d0[1] = __float_as_int(b) - 0x4B400000;
}
// A commit outside the deposit tile, straight to the global accumulator.  A CTA's first kFarFree of a launch are plain
// reductions that nothing waits for; the count of adds allows for them.  Nothing bounds how many more one word gets
// in a launch, so these look at it: a word found beyond 2^60 passes 2^34 of its value on to the next
// word: each such add then takes more off than it put on, and the adds in flight on a GPU (fewer than
// 2^19 of less than 2^32) cannot carry a word from there to 2^62.  The sum over the words is unchanged.  (All of
// them waiting for the word: a call of ten steps of 5e8 particles on 256^3, with its
// export, 62.6 ms against 61.2 ms.)
__device__ __forceinline__ int* far_count() {  // the CTA's commits of this launch, up to about kFarFree
  __shared__ int n;
  return &n;
}
__device__ __forceinline__ bool far_free() {
  volatile int* n = far_count();
  return *n < kFarFree && atomicAdd(far_count(), 1) < kFarFree;
}
__device__ __forceinline__ void far_digit(long long* p, int k, long long d, bool free) {
  if (d == 0 || k >= kAccWords) return;
  if (free) {
    atomicAdd((unsigned long long*)&p[k], (unsigned long long)d);
    return;
  }
  const long long old = (long long)atomicAdd((unsigned long long*)&p[k], (unsigned long long)d);
  constexpr long long lim = 1ll << 60;
  if (k + 1 < kAccWords && (old > lim || old < -lim)) {
    const long long c = old > 0 ? 4ll : -4ll;
    atomicAdd((unsigned long long*)&p[k], (unsigned long long)(-c * (1ll << 32)));
    atomicAdd((unsigned long long*)&p[k + 1], (unsigned long long)c);
  }
}
// t (in deposit-tile units, an FP32 number) rounded to global units, as a commit outside the tile
__device__ __forceinline__ void add_far(long long* p, float t, bool free) {
  const uint32_t b = __float_as_uint(t);
  const uint32_t ex = (b >> 23) & 0xffu;
  uint32_t man = (b & 0x7fffffu) | (ex != 0 ? 0x800000u : 0u);
  int s = (int)max(ex, 1u) - 150 + kDepShift;
  if (s < 0) {
    const int k = -s;
    man = k < 32 ? (man + ((1u << k) >> 1)) >> k : 0u;
    s = 0;
  }
  const unsigned long long lo = (unsigned long long)man << (s & 31);  // man < 2^24: below 2^55
  const long long sg = (b >> 31) ? -1ll : 1ll;
  far_digit(p, s >> 5, sg * (long long)(lo & 0xffffffffull), free);
  far_digit(p, (s >> 5) + 1, sg * (long long)(lo >> 32), free);
}

// the deposit tile of the unit at uo into the global accumulator, cleared; by `threads` threads, this one the ctid-th
__device__ __forceinline__ void flush_tile(const TmaArgs& a, int* dep, const int (&uo)[3], int ctid, int threads) {
  for (int t = ctid; t < kDepositCells; t += threads) {
    const int li = t % kDE, lj = (t / kDE) % kDE, lk = t / (kDE * kDE);
    int gi = uo[0] - kR + li, gj = uo[1] - kR + lj, gk = uo[2] - kR + lk;
    gi = gi < 0 ? gi + a.nx : (gi >= a.nx ? gi - a.nx : gi);
    gj = gj < 0 ? gj + a.ny : (gj >= a.ny ? gj - a.ny : gj);
    gk = gk < 0 ? gk + a.nz : (gk >= a.nz ? gk - a.nz : gk);
    const int64_t gc = gi + (int64_t)a.nx * (gj + (int64_t)a.ny * gk);
    for (int q = 0; q < 3; ++q) {
      int* w = dep + q * kDigits * kDepositCells + t;
      const long long val = (long long)w[0] + ((long long)w[kDepositCells] << kDigitBits) +
                            ((long long)w[2 * kDepositCells] << (2 * kDigitBits));
      if (val != 0) {
        w[0] = 0;
        w[kDepositCells] = 0;
        w[2 * kDepositCells] = 0;
        acc_add_mag(a.acc + kAccWords * (q * a.ncell + gc), (unsigned long long)(val < 0 ? -val : val), kDepShift,
                    val < 0);
      }
    }
  }
}

// a lane's P (2 or 4) consecutive 32-bit values as one access
template <int P>
struct alignas(4 * P) Vec32 {
  uint32_t w[P];
};
__device__ __forceinline__ void stcs(void* p, const Vec32<2>& v) {
  __stcs(reinterpret_cast<uint2*>(p), make_uint2(v.w[0], v.w[1]));
}
__device__ __forceinline__ void stcs(void* p, const Vec32<4>& v) {
  __stcs(reinterpret_cast<uint4*>(p), make_uint4(v.w[0], v.w[1], v.w[2], v.w[3]));
}
template <int P>
__device__ __forceinline__ Vec32<P> ldcs(const void* p) {
  Vec32<P> v;
  if constexpr (P == 4) {
    const uint4 q = __ldcs(reinterpret_cast<const uint4*>(p));
    v = Vec32<P>{q.x, q.y, q.z, q.w};
  } else {
    const uint2 q = __ldcs(reinterpret_cast<const uint2*>(p));
    v = Vec32<P>{q.x, q.y};
  }
  return v;
}
template <int P>
__device__ __forceinline__ Vec32<P> vec(const float (&f)[P]) {
  Vec32<P> v;
#pragma unroll
  for (int j = 0; j < P; ++j) v.w[j] = __float_as_uint(f[j]);
  return v;
}

// GATHER: the permutation entries of a lane's sorted positions p0 .. p0 + P - 1 (p0 a multiple of
// P), zeros when it owns none of them within [S, E) (then p0 may lie past the buffer)
template <int P>
__device__ __forceinline__ Vec32<P> gather_perm(const TmaArgs& a, int64_t p0, int64_t S, int64_t E) {
  return p0 + P > S && p0 < E ? ldcs<P>(a.perm + p0) : Vec32<P>{};
}
// GATHER: the ids of the owned positions among p0 .. p0 + P - 1 through the permutation (0 elsewhere)
template <int P>
__device__ __forceinline__ Vec32<P> gather_ids(const TmaArgs& a, const Vec32<P>& pp, int64_t p0, int64_t S, int64_t E) {
  Vec32<P> id;
#pragma unroll
  for (int j = 0; j < P; ++j) id.w[j] = (p0 + j >= S && p0 + j < E) ? __ldg(a.ids_in + pp.w[j]) : 0u;
  return id;
}
// GATHER: store ids gathered for positions p0 .. p0 + P - 1 (the owned ones)
template <int P>
__device__ __forceinline__ void store_ids(const TmaArgs& a, const Vec32<P>& id, int64_t p0, int64_t S, int64_t E) {
  if (p0 >= S && p0 + P <= E) {
    stcs(a.ids_out + p0, id);
  } else {
#pragma unroll
    for (int j = 0; j < P; ++j)
      if (p0 + j >= S && p0 + j < E) a.ids_out[p0 + j] = id.w[j];
  }
}
// GATHER: ask L2 for the records of the owned positions among p0 .. p0 + P - 1 (a stage before their
// loads)
template <int P>
__device__ __forceinline__ void gather_prefetch(const TmaArgs& a, const Vec32<P>& pp, int64_t p0, int64_t S, int64_t E) {
#pragma unroll
  for (int j = 0; j < P; ++j)
    if (p0 + j >= S && p0 + j < E) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.grec + 2 * (int64_t)pp.w[j]));
}
// GATHER: the diameters of the owned positions among p0 .. p0 + P - 1, stored in sorted order as soon as
// their records arrive (a step does not change them)
template <int P>
__device__ __forceinline__ void store_d(const TmaArgs& a, const Rec32 (&r)[P], int64_t p0, int64_t S, int64_t E) {
  if (p0 >= S && p0 + P <= E) {
    Vec32<P> d;
#pragma unroll
    for (int j = 0; j < P; ++j) d.w[j] = __float_as_uint(r[j].d);
    stcs(a.s.d + p0, d);
  } else {
#pragma unroll
    for (int j = 0; j < P; ++j)
      if (p0 + j >= S && p0 + j < E) a.s.d[p0 + j] = r[j].d;
  }
}

inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

// the ghost-padded field as a tensor map of fluid tiles
inline cudaError_t field_map(const st_ctx* h, CUtensorMap* map) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const int nx = h->geo.n[0], ny = h->geo.n[1], nz = h->geo.n[2];
  cuuint64_t dims[4] = {4, (cuuint64_t)(nx + 2 * kG), (cuuint64_t)(ny + 2 * kG), (cuuint64_t)(nz + 2 * kG)};
  cuuint64_t strides[3] = {16, (cuuint64_t)16 * (nx + 2 * kG), (cuuint64_t)16 * (nx + 2 * kG) * (ny + 2 * kG)};
  cuuint32_t box[4] = {4, kTE, kTE, kTE};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, h->fluid_pad.p, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// the arguments of a launch but for mcoef, s1 and s2
inline TmaArgs tma_args(const st_ctx* h, const StepParams& p, bool records, bool gather) {
  TmaArgs a;
  a.s = carve_mixed(h->state.p, h->cap, h->prec == ST_MIXED_BF16V);
  // records written by steps that gather go where the stale state was, their cells apart
  a.rec = records ? (float4*)(gather ? h->state.p : h->state_alt.p) : nullptr;
  if (records && gather) a.s.cell = (int32_t*)h->rec_cell.p;
  // the deferred gather of the last sort: permutation, records (old order) and ids in, ids out
  a.perm = gather ? (const uint32_t*)h->vals[0].p : nullptr;
  a.grec = gather ? (const float4*)h->state_alt.p : nullptr;
  a.ids_in = gather ? (const uint32_t*)h->ids.p : nullptr;
  a.ids_out = gather ? (uint32_t*)h->ids_alt.p : nullptr;
  a.ngp = p.ngp;
  a.semi = p.semi;
  a.sn = p.sn;
  a.cic = p.cic;
  a.re_coef = (float)p.re_coef;
  a.Up = (const float4*)h->fluid_pad.p;
  a.acc = (long long*)h->acc.p;
  a.cell_start = (const uint32_t*)h->cell_start.p;
  a.err = (int*)h->flags.p;
  a.unit_ctr = (unsigned*)((char*)h->flags.p + kUnitCounterOffset);
  a.nsteps = p.nsteps;
  a.ncell = h->geo.ncell;
  a.nx = h->geo.n[0];
  a.ny = h->geo.n[1];
  a.nz = h->geo.n[2];
  a.nunits = (int)(h->nkeys / (kU * kU * kU));
  int logB = 0;
  while ((1 << logB) < h->geo.B) ++logB;
  a.logB = logB;
  a.ncx = a.nx / h->geo.B;
  a.ncy = a.ny / h->geo.B;
  for (int q = 0; q < 3; ++q) {
    a.inv_h[q] = (float)h->geo.inv_h[q];
    a.g[q] = (float)p.g[q];
    a.gdt[q] = (float)(p.g[q] * p.dt);
  }
  a.dt = (float)p.dt;
  a.cadt = (float)(p.ca * p.dt);
  a.inv_ca = (float)(1.0 / p.ca);
  return a;
}

// a persistent CTA per SM, as far as there are units (and far commits are counted for)
inline int tma_grid(const st_ctx* h, int nunits) {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->dev);
  return std::min(std::min(sms > 0 ? sms : 152, nunits), kFarCtas);
}

// the kernels' dynamic shared memory.  A kernel attribute is per device; atomic because handles may be driven from
// several host threads (setting an attribute twice is harmless)
constexpr int kAttrDevices = 64;
template <class Kern>
cudaError_t allow_smem(std::atomic<bool>* set, int dev, Kern kern, int bytes) {
  if (dev < 0 || dev >= kAttrDevices) return cudaErrorInvalidDevice;
  if (set[dev].load(std::memory_order_acquire)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) set[dev].store(true, std::memory_order_release);
  return e;
}

}  // namespace
}  // namespace st
