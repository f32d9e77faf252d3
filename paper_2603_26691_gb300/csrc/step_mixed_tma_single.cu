// One mixed-precision step of many sorted particles.
//
// A launch of one step is bound by the particles' 60 B of HBM traffic, not by what happens on the chip, and
// nothing it computes once per particle is used twice.  This kernel is the multi-step one
// (step_mixed_tma.cu: units, tiles, stages and their barriers are described there) laid out for
// that: 4 consecutive particles per lane and 15 consumer warps at 128 registers, larger stages, whole-lane
// 128-bit stores ahead of the deposit, coefficients in registers.  What the two share is in tma_common.cuh; the step's
// arithmetic and the order of its sums are those of the multi-step kernel too, so the results are the same to the bit
// whichever takes a step.  1e9 particles on
// 256^3: 12.5 ms a step against 14.9 ms there; 6e7 on 128^3 9.0 against 9.9 ms for ten, the paper's physics 9.8
// against 11.6 ms.  The cloud-in-cell deposit, bound by its adds, is faster there (9.6 against 13.6 ms at 2e7).
// A unit of more particles than the tile's digit words take (the multi-step kernel flushes the tile in between) sends
// its sums to the global accumulator.
// The first step after a sort may also do that sort's payload gather (the GATHER instance): the sort
// leaves a permutation and the previous step's 32-byte records {cell, offsets | velocity, diameter}
// in the old order, and each consumer thread loads its own particles' records through the
// permutation with one 256-bit load each, asked of L2 by a prefetch one stage ahead (their ids come
// a stage ahead into registers and are stored in sorted order at the start of the stage they belong
// to; the diameters are stored as soon as the records arrive), then stores the new state in sorted
// order.  The separate gather would write the sorted arrays only for this step to read them back.
// Every wait is bounded: a wait that gives up sets an error flag and the CTA
// returns.
#include "tma_common.cuh"

namespace st {
namespace {

constexpr int kP = 4;                      // consecutive particles per lane
constexpr int kConsumerWarps = 15;
constexpr int kT = kConsumerWarps * 32 * kP;  // particles per stage (1920)
constexpr int kStages = 2;
constexpr int kScanLanes = 8;              // runs are chained across at most this many lanes
constexpr int kDirectRecords = 16;         // more run records than this per warp: commit in place
constexpr int64_t kDepMaxCount = 65535;    // per-unit particles for which no digit word can overflow
constexpr int kThreads = (kConsumerWarps + 1) * 32;

constexpr int kStageBytes = kT * 32;       // 61440 (FP32 layout; BF16 uses less)
constexpr int kSmemBytes = kFluidBytes + kDepositBytes + kStages * kStageBytes + 16 * 8;  // 229128

// add round(r_q * 2^Es), q = 0, 1, 2, to the shared deposit-tile values of one cell; s1 * s2 = 2^Es
__device__ __forceinline__ void dep_add3(int* w, float r0, float r1, float r2, float s1, float s2) {
  int d0[3], d1[3], d2[3];
  digits2(mul2(mul2(pack2(r0, r1), pack2(s1, s1)), pack2(s2, s2)), d0, d1, d2);
  digits1(__fmul_rn(__fmul_rn(r2, s1), s2), d0[2], d1[2], d2[2]);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int* wq = w + q * (kDigits * kDepositCells);
    if (d0[q]) atomicAdd(wq, d0[q]);
    if (d1[q]) atomicAdd(wq + kDepositCells, d1[q]);
    if (d2[q]) atomicAdd(wq + 2 * kDepositCells, d2[q]);
  }
}

// `big`: the unit holds more particles than the tile takes; its sums are rounded to the tile's units all the same where
// the cell lies in the tile, so that they are those of the multi-step kernel
__device__ __noinline__ void commit_far(const TmaArgs& a, int3 uo, bool big, int c, float r0, float r1, float r2) {
  const int n[3] = {a.nx, a.ny, a.nz}, g[3] = {c % a.nx, c / a.nx % a.ny, c / (a.nx * a.ny)}, o[3] = {uo.x, uo.y, uo.z};
  bool in = big;
  for (int q = 0; q < 3; ++q) in = in && (g[q] - o[q] + kR + 2 * n[q]) % n[q] < kDE;
  const float r[3] = {r0, r1, r2};
  const bool free = far_free();
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    float t = r[q] * a.s1 * a.s2;  // tile units, exact
    if (in) t = rintf(t);
    add_far(a.acc + kAccWords * ((int64_t)q * a.ncell + c), t, free);
  }
}

// one run's sums: into the shared deposit tile, or (start cell outside the tile, or a big unit) straight to the global
// accumulator
__device__ __forceinline__ void commit_record(const TmaArgs& a, int* dep, int3 uo, bool big, int kk, float r0,
                                              float r1, float r2) {
  if (__builtin_expect(kk < kDepositCells, 1))
    dep_add3(dep + kk, r0, r1, r2, a.s1, a.s2);
  else
    commit_far(a, uo, big, kk - kDepositCells, r0, r1, r2);
}

template <bool BF16, bool PW2, bool REC, bool PHYS, bool GATHER>
__global__ void __maxnreg__(128) step_mixed_tma_single_kernel(const __grid_constant__ CUtensorMap fluid_map,
                                                                      const __grid_constant__ TmaArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  float4* fluid = reinterpret_cast<float4*>(smem);                               // [kTE^3]
  int* dep = reinterpret_cast<int*>(smem + kFluidBytes);                         // [3][kDigits][kDE^3]
  unsigned char* ring = smem + kFluidBytes + kDepositBytes;                      // [kStages][kStageBytes]
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + kStages * kStageBytes);
  uint64_t* full = bars;                    // [kStages]   producer -> consumers (bytes landed)
  uint64_t* empty = bars + kStages;         // [kStages]   consumers -> producer (stage free)
  uint64_t* tile_full = bars + 2 * kStages;  // [1]        fluid tile landed
  uint64_t* tile_empty = tile_full + 1;      // [1]        consumers done with a fluid tile
  uint64_t* dep_done = tile_empty + 1;       // [1]        every consumer warp finished a unit's deposits
  uint64_t* flush_done = dep_done + 1;       // [1]        deposit tile flushed and cleared
  volatile int* unit_slot = reinterpret_cast<volatile int*>(flush_done + 1);  // unit of the fluid tile

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *far_count() = 0;
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kConsumerWarps);
    }
    mbar_init(tile_full, 1);
    mbar_init(tile_empty, kConsumerWarps);
    mbar_init(dep_done, kConsumerWarps);
    mbar_init(flush_done, kConsumerWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < 3 * kDigits * kDepositCells; i += blockDim.x) dep[i] = 0;
  __syncthreads();

  if (warp == kConsumerWarps) {
    // ================= producer =================
    if (lane == 0) {
      int loaded = 0;    // non-empty units whose fluid tile was issued
      int64_t gt = 0;    // particle stages issued
      // units are handed out one at a time from a global counter, so a CTA that starts late (its SM
      // busy with other work) simply takes fewer units
      for (;;) {
        const int u = (int)atomicAdd(a.unit_ctr, 1u);
        if (u >= a.nunits) break;
        const int64_t S = a.cell_start[(int64_t)u * (kU * kU * kU)];
        const int64_t E = a.cell_start[(int64_t)(u + 1) * (kU * kU * kU)];
        if (E <= S) continue;
        if (loaded >= 1 && !mbar_wait(tile_empty, (loaded - 1) & 1)) {
          atomicOr(a.err, 1);
          return;
        }
        *unit_slot = u;  // published to the consumers by the tile barrier's arrive
        int ox, oy, oz;
        unit_origin(a, u, ox, oy, oz);
        mbar_expect_tx(tile_full, kFluidBytes);
        tma_load_tile(fluid, &fluid_map, ox, oy, oz, tile_full);
        ++loaded;
        const int64_t A = S & ~int64_t(7);
        const int64_t Z = (E + 7) & ~int64_t(7);
        for (int64_t t0 = A; t0 < Z; t0 += kT) {
          const int cnt = (int)min((int64_t)kT, Z - t0);
          const int st = (int)(gt % kStages);
          if (gt >= kStages && !mbar_wait(&empty[st], ((gt / kStages) - 1) & 1)) {
            atomicOr(a.err, 2);
            return;
          }
          unsigned char* dst = ring + st * kStageBytes;
          if (GATHER) {
            // the consumers load their particles themselves; the stage only serves as their scratch
            mbar_arrive(&full[st]);
            ++gt;
            continue;
          }
          mbar_expect_tx(&full[st], stage_bytes<BF16>(cnt));
          bulk_load(dst, a.s.cell + t0, cnt * 4, &full[st]);
          for (int q = 0; q < 3; ++q) bulk_load(dst + (1 + q) * kT * 4, a.s.xi[q] + t0, cnt * 4, &full[st]);
          const int vb = BF16 ? 2 : 4;
          for (int q = 0; q < 3; ++q)
            bulk_load(dst + 4 * kT * 4 + q * kT * vb, (const char*)a.s.v[q] + t0 * vb, cnt * vb, &full[st]);
          bulk_load(dst + 4 * kT * 4 + 3 * kT * vb, a.s.d + t0, cnt * 4, &full[st]);
          ++gt;
        }
      }
      // the last CTA to find no unit left makes the two counters ready for the next launch
      if (atomicInc(a.unit_ctr + 1, gridDim.x - 1) == gridDim.x - 1) atomicExch(a.unit_ctr, 0u);
      // no more units: a tile phase without a copy, unit -1
      {
        if (loaded >= 1 && !mbar_wait(tile_empty, (loaded - 1) & 1)) {
          atomicOr(a.err, 1);
          return;
        }
        *unit_slot = -1;
        mbar_arrive(tile_full);
      }
      // let the last copies land before the CTA can exit
      const int64_t first = gt > kStages ? gt - kStages : 0;
      for (int64_t k = first; k < gt; ++k) mbar_wait(&empty[k % kStages], (k / kStages) & 1);
    }
    return;
  }

  // ================= consumers =================
  const int ctid = threadIdx.x;  // 0 .. 32 kConsumerWarps - 1
  const int n3[3] = {a.nx, a.ny, a.nz};
  const int px = a.nx + 2 * kG, pxy = (a.nx + 2 * kG) * (a.ny + 2 * kG);
  int loaded = 0;
  int64_t gt = 0;
  for (;;) {
    if (!mbar_wait(tile_full, loaded & 1)) {
      atomicOr(a.err, 4);
      return;
    }
    const int u = *unit_slot;
    if (u < 0) break;
    const int64_t S = a.cell_start[(int64_t)u * (kU * kU * kU)];
    const int64_t E = a.cell_start[(int64_t)(u + 1) * (kU * kU * kU)];
    int uo[3];
    unit_origin(a, u, uo[0], uo[1], uo[2]);
    const bool use_tile = (E - S) <= kDepMaxCount;  // every digit word stays below 2^31
    const int64_t A = S & ~int64_t(7);
    const int64_t Z = (E + 7) & ~int64_t(7);
    const int L = kP * ctid;
    // GATHER: the permutation entries of this stage and of the next, and this stage's ids, are
    // held in registers a stage ahead
    Vec32<kP> pcur{}, pnext{}, gid{};
    if constexpr (GATHER) {
      pcur = gather_perm<kP>(a, A + L, S, E);
      gid = gather_ids(a, pcur, A + L, S, E);
      pnext = gather_perm<kP>(a, A + kT + L, S, E);
    }
    for (int64_t t0 = A; t0 < Z; t0 += kT) {
      const int st = (int)(gt % kStages);
      if (!mbar_wait(&full[st], (gt / kStages) & 1)) {
        atomicOr(a.err, 8);
        return;
      }
      const unsigned char* src = ring + st * kStageBytes;
      const int64_t p0 = t0 + L;
      int cell[4];
      float xi[3][4], v[3][4], dv[4];
      if constexpr (GATHER) {
        // this stage's records through the permutation, one 256-bit load each (asked of L2 a stage
        // ago); positions outside the unit get harmless values and are neither stored nor deposited
        const int glo = (int)max((int64_t)0, min((int64_t)4, S - p0));
        const int ghi = (int)max((int64_t)0, min((int64_t)4, E - p0));
        Rec32 r[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          r[j] = (j >= glo && j < ghi) ? ld_rec32(a.grec + 2 * (int64_t)pcur.w[j])
                                       : Rec32{0.0f, 0.5f, 0.5f, 0.5f, 0.0f, 0.0f, 0.0f, 1e-5f};
        // this stage's ids (loaded a stage ago) go out now; the next stage's come in, and its records
        // are asked for
        store_ids(a, gid, p0, S, E);
        if (t0 + kT < Z) {
          gather_prefetch(a, pnext, p0 + kT, S, E);
          gid = gather_ids(a, pnext, p0 + kT, S, E);
          pcur = pnext;
          pnext = gather_perm<kP>(a, p0 + 2 * kT, S, E);
        }
        store_d(a, r, p0, S, E);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          cell[j] = __float_as_int(r[j].c);
          xi[0][j] = r[j].x0;
          xi[1][j] = r[j].x1;
          xi[2][j] = r[j].x2;
          v[0][j] = r[j].v0;
          v[1][j] = r[j].v1;
          v[2][j] = r[j].v2;
          dv[j] = r[j].d;
        }
      } else {
        int4 c4 = *reinterpret_cast<const int4*>(src + L * 4);
        cell[0] = c4.x;
        cell[1] = c4.y;
        cell[2] = c4.z;
        cell[3] = c4.w;
        for (int q = 0; q < 3; ++q) {
          float4 x4 = *reinterpret_cast<const float4*>(src + (1 + q) * kT * 4 + L * 4);
          xi[q][0] = x4.x;
          xi[q][1] = x4.y;
          xi[q][2] = x4.z;
          xi[q][3] = x4.w;
        }
        if (BF16) {
          for (int q = 0; q < 3; ++q) {
            uint2 r = *reinterpret_cast<const uint2*>(src + 4 * kT * 4 + q * kT * 2 + L * 2);
            float2 l = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&r.x));
            float2 h = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&r.y));
            v[q][0] = l.x;
            v[q][1] = l.y;
            v[q][2] = h.x;
            v[q][3] = h.y;
          }
          float4 d4 = *reinterpret_cast<const float4*>(src + 4 * kT * 4 + 3 * kT * 2 + L * 4);
          dv[0] = d4.x;
          dv[1] = d4.y;
          dv[2] = d4.z;
          dv[3] = d4.w;
        } else {
          for (int q = 0; q < 3; ++q) {
            float4 r = *reinterpret_cast<const float4*>(src + 4 * kT * 4 + q * kT * 4 + L * 4);
            v[q][0] = r.x;
            v[q][1] = r.y;
            v[q][2] = r.z;
            v[q][3] = r.w;
          }
          float4 d4 = *reinterpret_cast<const float4*>(src + 7 * kT * 4 + L * 4);
          dv[0] = d4.x;
          dv[1] = d4.y;
          dv[2] = d4.z;
          dv[3] = d4.w;
        }
      }
      ++gt;

      // owned particles of this lane: [lo, hi) of 0..3 (the rest belong to neighbouring units
      // or lie past the unit); the others are computed too, without branches, from the unit's
      // origin cell so that every tile read stays in bounds, and neither stored nor deposited
      const int lo = (int)max((int64_t)0, min((int64_t)4, S - p0));
      const int hi = (int)max((int64_t)0, min((int64_t)4, E - p0));
      const int ucell = pack_cell(uo[0], uo[1], uo[2]);
      bool own[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        own[j] = (j >= lo) && (j < hi);
        if (!own[j]) cell[j] = ucell;
      }
      // ---- per particle: start cell relative to the unit, deposit key, fluid gather; then drag and
      // gravity (exponential integrator), relocation and exchanged momentum for two particles at
      // a time as FP32 register pairs.  A start cell within kR cells of the unit (the deposit tile)
      // has its whole stencil inside the fluid tile; the rest ("far" particles, rare) read the
      // padded field and commit to the global accumulator.
      int key[4];
      float J[4][3];
      unsigned vpk[3][2];  // BF16: the new velocities as packed pairs (particles 0-1, 2-3)
#pragma unroll
      for (int jp = 0; jp < 4; jp += 2) {
        int ci[2][3];
        float up[2][3];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = jp + e;
          ci[e][0] = cell_i(cell[j]);
          ci[e][1] = cell_j(cell[j]);
          ci[e][2] = cell_k(cell[j]);
          int rc[3], rb[3];
          float f[3];
          bool in_dep = true;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float o = xi[q][j];
            const bool hi2 = o >= 0.5f;
            f[q] = o + (hi2 ? -0.5f : 0.5f);
            int r = ci[e][q] - uo[q];  // periodic offset from the unit origin, valid within the tile
            if (PW2) {
              r = ((r + kR) & (n3[q] - 1)) - kR;
            } else {
              if (r >= n3[q] - kR) r -= n3[q];
              else if (r < kDE - kR - n3[q]) r += n3[q];
            }
            in_dep = in_dep && ((unsigned)(r + kR) < (unsigned)kDE);
            rc[q] = r;
            rb[q] = r - (hi2 ? 0 : 1);  // stencil base relative to the unit origin
          }
          const int tofs = in_dep ? (rb[0] + kG) + kTE * ((rb[1] + kG) + kTE * (rb[2] + kG)) : 0;
          key[j] = !own[j]                ? -1
                   : (in_dep && use_tile) ? (rc[0] + kR) + kDE * ((rc[1] + kR) + kDE * (rc[2] + kR))
                                          : kDepositCells + ci[e][0] + a.nx * (ci[e][1] + a.ny * ci[e][2]);
          if (PHYS && a.ngp) {
            // nearest grid point: the value of the start cell (inside the tile when in_dep)
            const float4 c = fluid[in_dep ? (rc[0] + kG) + kTE * ((rc[1] + kG) + kTE * (rc[2] + kG)) : 0];
            up[e][0] = c.x;
            up[e][1] = c.y;
            up[e][2] = c.z;
            if (__builtin_expect(!in_dep, 0)) {
              const float3 g = ngp_padded(a.Up, px, pxy, cell[j]);
              up[e][0] = g.x;
              up[e][1] = g.y;
              up[e][2] = g.z;
            }
          } else {
            const float4* bb = fluid + tofs;
            trilerp(bb[0], bb[1], bb[kTE], bb[kTE + 1], bb[kTE * kTE], bb[kTE * kTE + 1], bb[kTE * kTE + kTE],
                    bb[kTE * kTE + kTE + 1], f[0], f[1], f[2], up[e]);
            if (__builtin_expect(!in_dep, 0)) {
              const float3 g = gather_padded(a.Up, px, pxy, cell[j], xi[0][j], xi[1][j], xi[2][j]);
              up[e][0] = g.x;
              up[e][1] = g.y;
              up[e][2] = g.z;
            }
          }
        }
        // the integrator on the pair
        const unsigned long long D = pack2(dv[jp], dv[jp + 1]);
        const unsigned long long DD = mul2(D, D);
        float dd0, dd1;
        unpack2(DD, dd0, dd1);
        unsigned long long ADT = mul2(dup2(a.cadt), pack2(rcp_approx(dd0), rcp_approx(dd1)));
        unsigned long long INV_A = mul2(DD, dup2(a.inv_ca));
        unsigned long long EE, E1, Q;
        if (PHYS) {
          // drag rate a = alpha f(Re) / tau (f = 1 for Stokes drag), f from the start-of-step
          // relative velocity; both integrators take the form v' = w + (v - w) E,
          // x' = x + w dt + (v - w) Q with w = u_p + g / a:
          //   exponential:         E = e^{-a dt},       Q = (1 - E) / a
          //   semi-implicit Euler: E = 1 / (1 + a dt),  Q = E dt  (x' = x + dt v')
          if (a.sn) {
            float fac[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float r0 = up[e][0] - v[0][jp + e], r1 = up[e][1] - v[1][jp + e], r2 = up[e][2] - v[2][jp + e];
              fac[e] = sn_factor(a.re_coef * sqrtf(fmaf(r0, r0, fmaf(r1, r1, r2 * r2))) * dv[jp + e]);
            }
            ADT = mul2(ADT, pack2(fac[0], fac[1]));
            INV_A = mul2(INV_A, pack2(rcp_approx(fac[0]), rcp_approx(fac[1])));
          }
          if (a.semi) {
            float x0, x1;
            unpack2(ADT, x0, x1);
            const float e0 = rcp_approx(1.0f + x0), e1 = rcp_approx(1.0f + x1);
            EE = pack2(e0, e1);
            E1 = pack2(x0 * e0, x1 * e1);  // 1 - E = a dt / (1 + a dt)
            Q = mul2(EE, dup2(a.dt));
          } else {
            E1 = one_minus_exp2(ADT, &EE);
            Q = mul2(E1, INV_A);
          }
        } else {
          E1 = one_minus_exp2(ADT, &EE);
          Q = mul2(E1, INV_A);
        }
        const unsigned long long M = mul2(mul2(dup2(a.mcoef), DD), D);
        float oraw[2][3];
        int ii[2][3];
        bool bad[2] = {false, false};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const unsigned long long WT = fma2(dup2(a.g[q]), INV_A, pack2(up[0][q], up[1][q]));
          const unsigned long long V = pack2(v[q][jp], v[q][jp + 1]);
          const unsigned long long DVW = sub2(V, WT);
          float vn[2];
          unpack2(fma2(DVW, EE, WT), vn[0], vn[1]);
          if (BF16) {
            // the stored (rounded) velocity change, so that the deposit balances the particles'
            // momentum; the pair is rounded by one packing conversion, kept packed for the store (the product
            // is rounded before the run sums, as in the multi-step kernel)
            float m0, m1;
            unpack2(M, m0, m1);
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(vn[0], vn[1]);
            vpk[q][jp >> 1] = *reinterpret_cast<const unsigned*>(&b2);
            vn[0] = __low2float(b2);
            vn[1] = __high2float(b2);
            J[jp][q] = __fmul_rn(-m0, (vn[0] - v[q][jp]) - a.gdt[q]);
            J[jp + 1][q] = __fmul_rn(-m1, (vn[1] - v[q][jp + 1]) - a.gdt[q]);
          } else {
            // v' - v = -(v - w) (1 - E), without the cancellation of subtracting the rounded v'
            unpack2(mul2(M, fma2(DVW, E1, dup2(a.gdt[q]))), J[jp][q], J[jp + 1][q]);
          }
          const unsigned long long DXV = fma2(WT, dup2(a.dt), mul2(DVW, Q));
          const unsigned long long O = fma2(DXV, dup2(a.inv_h[q]), pack2(xi[q][jp], xi[q][jp + 1]));
          // whole cells carried: floor(o) from an add of 1.5 * 2^23 rounded toward -inf (exact for
          // |o| < 2^22), so no conversion instructions; the offset o - floor(o) lies in [0, 1]
          const unsigned long long T = add_rm2(O, dup2(12582912.0f));
          float o[2], t[2], x[2];
          unpack2(O, o[0], o[1]);
          unpack2(T, t[0], t[1]);
          unpack2(sub2(O, sub2(T, dup2(12582912.0f))), x[0], x[1]);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            oraw[e][q] = o[e];
            int k = (int)((unsigned)ci[e][q] + (unsigned)(__float_as_int(t[e]) - 0x4B400000));
            if (PW2) {
              k &= n3[q] - 1;  // any whole-cell move of fewer than 2^22 cells
              bad[e] = bad[e] || !(fabsf(o[e]) < 4194304.0f);
            } else {
              if (k >= n3[q]) k -= n3[q];
              else if (k < 0) k += n3[q];
              bad[e] = bad[e] || !(fabsf(o[e]) < 4194304.0f) || ((unsigned)k >= (unsigned)n3[q]);
            }
            ii[e][q] = k;
            xi[q][jp + e] = fminf(x[e], 0.99999994f);
            v[q][jp + e] = vn[e];
          }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (__builtin_expect(bad[e], 0)) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const Relocated rl = relocate_general(oraw[e][q], ci[e][q], n3[q]);
              ii[e][q] = rl.cell;
              xi[q][jp + e] = rl.offset;
            }
          }
          cell[jp + e] = pack_cell(ii[e][0], ii[e][1], ii[e][2]);
        }
      }
      // ---- store the owned particles (128-bit when the lane owns all four) ----
      const bool all_own = own[0] && own[1] && own[2] && own[3];
      if (REC) {
        // the step before a sort: the cells to the structure of arrays (the sort's keys), the whole
        // state as 32-byte records {cell, offsets | velocity, diameter}, one 256-bit store per
        // particle (a full sector; the sort's gather then reads one sector per particle).  The
        // diameters are read again from the stage.  BF16 handles store the (BF16-exact) velocities
        // as FP32 in the record.
        const float4 d4 =
            *reinterpret_cast<const float4*>(src + (BF16 ? 4 * kT * 4 + 3 * kT * 2 : 7 * kT * 4) + L * 4);
        const float dj[4] = {d4.x, d4.y, d4.z, d4.w};
        if (all_own) __stcs((int4*)(a.s.cell + p0), make_int4(cell[0], cell[1], cell[2], cell[3]));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (!own[j]) continue;
          if (!all_own) a.s.cell[p0 + j] = cell[j];
          st_rec32(a.rec + 2 * (p0 + j),
                   Rec32{__int_as_float(cell[j]), xi[0][j], xi[1][j], xi[2][j], v[0][j], v[1][j], v[2][j], dj[j]});
        }
      } else if (all_own) {
        __stcs((int4*)(a.s.cell + p0), make_int4(cell[0], cell[1], cell[2], cell[3]));
        for (int q = 0; q < 3; ++q)
          __stcs((float4*)(a.s.xi[q] + p0), make_float4(xi[q][0], xi[q][1], xi[q][2], xi[q][3]));
        if (BF16) {
          for (int q = 0; q < 3; ++q) __stcs((uint2*)((__nv_bfloat16*)a.s.v[q] + p0), make_uint2(vpk[q][0], vpk[q][1]));
        } else {
          for (int q = 0; q < 3; ++q)
            __stcs((float4*)((float*)a.s.v[q] + p0), make_float4(v[q][0], v[q][1], v[q][2], v[q][3]));
        }
      } else {
        for (int j = 0; j < 4; ++j) {
          if (!own[j]) continue;
          a.s.cell[p0 + j] = cell[j];
          for (int q = 0; q < 3; ++q) {
            a.s.xi[q][p0 + j] = xi[q][j];
            if (BF16)
              ((__nv_bfloat16*)a.s.v[q])[p0 + j] = __float2bfloat16_rn(v[q][j]);
            else
              ((float*)a.s.v[q])[p0 + j] = v[q][j];
          }
        }
      }
      // ---- deposit: runs of equal key over the warp's 128 particles (lane-local suffix sums, then a
      // segmented suffix scan across lanes chains runs that span lanes). ----
      auto deposit = [&](const int (&key)[4], const float (&J)[4][3]) {
        float Sx[4][3];
#pragma unroll
        for (int q = 0; q < 3; ++q) Sx[3][q] = J[3][q];
#pragma unroll
        for (int j = 2; j >= 0; --j) {
          const bool same = key[j] == key[j + 1];
#pragma unroll
          for (int q = 0; q < 3; ++q) Sx[j][q] = J[j][q] + (same ? Sx[j + 1][q] : 0.0f);
        }
        const int tail = (key[2] != key[3]) ? 3 : (key[1] != key[2]) ? 2 : (key[0] != key[1]) ? 1 : 0;
        const int nk0 = __shfl_down_sync(0xffffffffu, key[0], 1);
        const int nall = __shfl_down_sync(0xffffffffu, (int)(tail == 0), 1);
        float R[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) R[q] = __shfl_down_sync(0xffffffffu, Sx[0][q], 1);
        const int glane = lane & (kScanLanes - 1);
        const bool link = (glane < kScanLanes - 1) && (nk0 == key[3]) && (key[3] >= 0);
        int Bl = (link && nall) ? 1 : 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) R[q] = link ? R[q] : 0.0f;
        // the scan only matters where a run passes through a whole lane (often nowhere after drift)
        if (__any_sync(0xffffffffu, Bl)) {
#pragma unroll
          for (int off = 1; off < kScanLanes; off <<= 1) {
            float t0v = __shfl_down_sync(0xffffffffu, R[0], off);
            float t1v = __shfl_down_sync(0xffffffffu, R[1], off);
            float t2v = __shfl_down_sync(0xffffffffu, R[2], off);
            int tb = __shfl_down_sync(0xffffffffu, Bl, off);
            if (glane + off > kScanLanes - 1) {
              tb = 0;
              t0v = t1v = t2v = 0.0f;
            }
            if (Bl) {
              R[0] += t0v;
              R[1] += t1v;
              R[2] += t2v;
            }
            Bl &= tb;
          }
        }
        const int pk3 = __shfl_up_sync(0xffffffffu, key[3], 1);
        const bool head_lane = (glane == 0) || (pk3 != key[0]);
        // the run sums, one {J, key} record per run.  Few runs (after a sort): the records are packed
        // in (j, lane) order into the warp's own (already consumed) part of the stage - J in the cell
        // and first two offset arrays, the key in the third - and each lane takes one record at a
        // time, so the whole deposit is one pass.  Many runs (particles drifted away from their
        // sort-time cells): each lane commits its runs where they are, one pass per particle slot,
        // without the round trip through shared memory.
        bool starts[4];
        unsigned hms[4];
        int nh = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          starts[j] = ((j == 0) ? head_lane : (key[j] != key[j - 1])) && key[j] >= 0;
          hms[j] = __ballot_sync(0xffffffffu, starts[j]);
          nh += __popc(hms[j]);
        }
        const bool direct = nh > kDirectRecords;
        if (direct) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (starts[j]) {
              const bool to_end = j == tail;
              const float r0 = Sx[j][0] + (to_end ? R[0] : 0.0f);
              const float r1 = Sx[j][1] + (to_end ? R[1] : 0.0f);
              const float r2 = Sx[j][2] + (to_end ? R[2] : 0.0f);
              commit_record(a, dep, make_int3(uo[0], uo[1], uo[2]), !use_tile, key[j], r0, r1, r2);
            }
          }
        } else {
          int* rj0 = reinterpret_cast<int*>(const_cast<unsigned char*>(src)) + warp * 128;
          int* rj1 = rj0 + kT;
          int* rj2 = rj0 + 2 * kT;
          int* rk = rj0 + 3 * kT;
          const unsigned lt_mask = (1u << lane) - 1u;
          int base = 0;
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (starts[j]) {
              const bool to_end = j == tail;
              const int slot = base + __popc(hms[j] & lt_mask);
              rj0[slot] = __float_as_int(Sx[j][0] + (to_end ? R[0] : 0.0f));
              rj1[slot] = __float_as_int(Sx[j][1] + (to_end ? R[1] : 0.0f));
              rj2[slot] = __float_as_int(Sx[j][2] + (to_end ? R[2] : 0.0f));
              rk[slot] = key[j];
            }
            base += __popc(hms[j]);
          }
          __syncwarp();
          for (int e = lane; e < nh; e += 32) {
            commit_record(a, dep, make_int3(uo[0], uo[1], uo[2]), !use_tile, rk[e], __int_as_float(rj0[e]), __int_as_float(rj1[e]), __int_as_float(rj2[e]));
          }
          // the records were written through the generic proxy; order them before the producer's
          // next bulk copy into this stage
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
      };
      deposit(key, J);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
    }
    // all gathers of this unit are done: the producer may reuse its fluid buffer
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(tile_empty);
      mbar_arrive(dep_done);
    }
    // flush the deposit tile once every consumer warp has finished this unit
    if (!mbar_wait(dep_done, loaded & 1)) {
      atomicOr(a.err, 16);
      return;
    }
    flush_tile(a, dep, uo, ctid, kConsumerWarps * 32);
    __syncwarp();
    if (lane == 0) mbar_arrive(flush_done);
    if (!mbar_wait(flush_done, loaded & 1)) {
      atomicOr(a.err, 32);
      return;
    }
    ++loaded;
  }
}

}  // namespace

cudaError_t launch_step_mixed_tma_single(st_ctx* h, const StepParams& p, bool records, bool gather) {
  const bool bf = h->prec == ST_MIXED_BF16V;
  const bool phys = p.ngp || p.semi || p.sn;
  if ((records || gather) && phys) return cudaErrorInvalidValue;
  if (records && gather) return cudaErrorInvalidValue;
  bool pw2 = true;
  for (int q = 0; q < 3; ++q) pw2 = pw2 && (h->geo.n[q] & (h->geo.n[q] - 1)) == 0;
  using Kern = void (*)(const CUtensorMap, const TmaArgs);
  static const Kern table[16] = {
      step_mixed_tma_single_kernel<false, false, false, false, false>, step_mixed_tma_single_kernel<false, true, false, false, false>,
      step_mixed_tma_single_kernel<false, false, false, true, false>,  step_mixed_tma_single_kernel<false, true, false, true, false>,
      step_mixed_tma_single_kernel<true, false, false, false, false>,  step_mixed_tma_single_kernel<true, true, false, false, false>,
      step_mixed_tma_single_kernel<true, false, false, true, false>,   step_mixed_tma_single_kernel<true, true, false, true, false>,
      step_mixed_tma_single_kernel<false, false, true, false, false>,  step_mixed_tma_single_kernel<false, true, true, false, false>,
      step_mixed_tma_single_kernel<true, false, true, false, false>,   step_mixed_tma_single_kernel<true, true, true, false, false>,
      step_mixed_tma_single_kernel<false, false, false, false, true>,  step_mixed_tma_single_kernel<false, true, false, false, true>,
      step_mixed_tma_single_kernel<true, false, false, false, true>,   step_mixed_tma_single_kernel<true, true, false, false, true>};
  static std::atomic<bool> attr_set[16][kAttrDevices];
  const int variant = gather    ? 12 + 2 * (int)bf + (int)pw2
                      : records ? 8 + 2 * (int)bf + (int)pw2
                                : 4 * (int)bf + 2 * (int)phys + (int)pw2;
  const Kern kern = table[variant];
  CUtensorMap map;
  cudaError_t e = allow_smem(attr_set[variant], h->dev, kern, kSmemBytes);
  if (e == cudaSuccess) e = field_map(h, &map);
  if (e != cudaSuccess) return e;
  TmaArgs a = tma_args(h, p, records, gather);
  a.mcoef = (float)p.mcoef;
  {
    // 2^(E - kDepShift) as two representable factors; beyond +-250 every scaled impulse is 0 or
    // overflows the bound the exponent was chosen for, so clamping changes nothing
    const int Es = std::min(std::max(p.E - kDepShift, -250), 250);
    a.s1 = std::ldexp(1.0f, Es / 2);
    a.s2 = std::ldexp(1.0f, Es - Es / 2);
  }
  kern<<<tma_grid(h, a.nunits), kThreads, kSmemBytes, h->stream>>>(map, a);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace st
