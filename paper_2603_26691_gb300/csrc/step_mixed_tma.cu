// Mixed-precision Lagrangian step for sorted particles: a persistent,
// warp-specialised kernel fed by the Tensor Memory Accelerator.
//
// After the counting sort the particles of every aligned U^3 block of cells
// (U = min(B, 8); the Morton order inside a chunk makes each such block a
// contiguous key range) are contiguous in storage.  Each CTA owns a sequence of
// these units.  Per unit:
//   * a producer warp loads the unit's fluid tile - the U^3 cells plus a halo
//     of G cells - from the ghost-padded field with one 4-D TMA tensor copy,
//     once the consumers are done with the unit before it, and streams the
//     unit's particle arrays through a ring of shared-memory stages with 1-D
//     bulk copies (cp.async.bulk), signalling completion on mbarriers;
//   * consumer warps take kP consecutive particles per lane from the stage,
//     gather the fluid velocity from the shared tile (8 LDS.128 with immediate
//     offsets; particles that drifted out of the tile read the padded field
//     from L2), advance and relocate them, reduce their impulses over runs of equal
//     start-of-step cell across the warp, and store the new state with wide
//     streaming stores;
//   * each run is added once to the unit's deposit tile with integer shared atomics (exact and
//     independent of the order of the adds), which is flushed to the global carry-save fixed-point
//     accumulator.
// The field is frozen over a call and particles do not act on each other, so a launch takes all the steps
// up to the next sort on a stage before the next one (nsteps): the state, the diameter's coefficients, the
// fluid tile and the deposit tile stay on the chip between them, and a step costs its arithmetic and its
// deposit instead of 60 B of HBM traffic per particle.  The arithmetic and the grouping of the sums are those
// of one step per launch, so the results do not depend on how the steps are split over calls.
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

constexpr int kP = 2;                       // consecutive particles per lane
constexpr int kWarpParts = 32 * kP;
constexpr int kStages = 2;
constexpr int kScanPairs = 8;              // runs are chained across at most this many pairs of lanes
constexpr unsigned kPairLinks = 0x15551555u;  // the pairs that have a next one in their group, at their even lane
// adds to one cell's digit words between flushes: the two lower digits are at most 2^14, and the top one at
// most 1 + 2^8 per particle of the run (one particle's impulse is below 2^38 tile units)
constexpr int kDepMaxAdds = 131071;
// particles from which a launch of one step goes to step_mixed_tma_single.cu (ten single steps, there / here: 3e5 on
// 64^3 0.36 / 0.34 ms, 2e6 0.69 / 0.67, 2e7 on 128^3 4.54 / 4.72, 6e7 9.0 / 9.9)
constexpr int64_t kSingleParticles = 1 << 23;
constexpr unsigned kNoKey = 0xffffffffu;   // no cell: neither a tile-form nor a far one

// The shape of an instance.  The steps run on what the registers let run at once: two particles per lane and 23
// consumer warps at 80 registers hide more of the latency than four per lane and 15 warps at 128 (4e8
// particles on 256^3, ten steps: 44.1 against 48.2 ms when the shape was chosen, 36.8 ms since).  The physics
// variants need more registers: 19 warps at 96 (cloud-in-cell at 2e7 on 128^3: 8.9 ms, with four per lane 10.7; 6.6 ms
// since).  Swapped, 19 warps for the default and 23 for the variants: 39.9 against 37.3 ms and 8.8 against 7.3 ms.
template <bool PHYS>
struct Shape {
  static constexpr int kConsumerWarps = PHYS ? 19 : 23;
  static constexpr int kT = kConsumerWarps * kWarpParts;  // particles per stage
  static constexpr int kThreads = (kConsumerWarps + 1) * 32;
  static constexpr int kRegs = 65536 / kThreads / 8 * 8;
  static constexpr int kStageBytes = kT * 32;             // the FP32 layout; BF16 uses less
  static constexpr int kSmemBytes = kFluidBytes + kDepositBytes + kStages * kStageBytes + 16 * 8;
  static_assert(kSmemBytes + 16 <= 232448, "shared memory of a block");
  static_assert(kT * kMaxFusedSteps <= kDepMaxAdds, "a stage's deposits fit the digit words");
};

// add round(t_q), q = 0, 1, 2 (in tile units), to the shared deposit-tile values of one cell.  The top digit is zero up
// to 2^29, where nearly all values lie (the unit is 2^-45 of a bound on 128 of the largest particles): two digits then.
// The two lower digits alone, |t| <= 2^29
__device__ __forceinline__ void low_digits1(float t, int& d0, int& d1) {
  const float m = __fsub_rn(__fadd_rn(t, 0x1.8p38f), 0x1.8p38f);
  d1 = __float_as_int(__fmaf_rn(m, 0x1p-15f, 12582912.0f)) - 0x4B400000;
  d0 = __float_as_int(__fadd_rn(__fsub_rn(t, m), 12582912.0f)) - 0x4B400000;
}
__device__ __forceinline__ void low_digits2(unsigned long long t, int* d0, int* d1) {
  const unsigned long long C38 = pack2(0x1.8p38f, 0x1.8p38f), C23 = pack2(12582912.0f, 12582912.0f);
  const unsigned long long m = sub2(add2(t, C38), C38);
  float a, b;
  unpack2(fma2(m, pack2(0x1p-15f, 0x1p-15f), C23), a, b);
  d1[0] = __float_as_int(a) - 0x4B400000;
  d1[1] = __float_as_int(b) - 0x4B400000;
  unpack2(add2(sub2(t, m), C23), a, b);
  d0[0] = __float_as_int(a) - 0x4B400000;
  d0[1] = __float_as_int(b) - 0x4B400000;
}
__device__ __forceinline__ void dep_add3(int* w, float t0, float t1, float t2) {
  if (__builtin_expect(fmaxf(fmaxf(fabsf(t0), fabsf(t1)), fabsf(t2)) <= 0x1p29f, 1)) {
    int d0[3], d1[3];
    low_digits2(pack2(t0, t1), d0, d1);
    low_digits1(t2, d0[2], d1[2]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      int* wq = w + q * (kDigits * kDepositCells);
      // not asked whether they are zero: they rarely are (38.8 ms with the tests, 37.3 ms without)
      atomicAdd(wq, d0[q]);
      atomicAdd(wq + kDepositCells, d1[q]);
    }
    return;
  }
  int d0[3], d1[3], d2[3];
  digits2(pack2(t0, t1), d0, d1, d2);
  digits1(t2, d0[2], d1[2], d2[2]);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int* wq = w + q * (kDigits * kDepositCells);
    if (d0[q]) atomicAdd(wq, d0[q]);
    if (d1[q]) atomicAdd(wq + kDepositCells, d1[q]);
    if (d2[q]) atomicAdd(wq + 2 * kDepositCells, d2[q]);
  }
}

// In the step loop a particle's cell is kept relative to its unit: field q of c = offset from the unit's
// origin + kBias, three 10-bit fields.  Whole-cell moves add to the fields (signed moves borrow across
// fields and cancel, as long as every field ends up in 0 .. 1023), and one test covers the three axes:
// a cell of the deposit tile (offsets -kR .. kU + kR - 1) has fields kCellLo .. kCellLo + kDE - 1, that is
// bit 5 set, bits 6-9 clear, and bit 6 still clear after adding 64 - kCellLo - kDE.  Any other cell is kept as
// the global packed cell with bit 31 set (kFarCell).
constexpr int kCellLo = 32, kBias = kCellLo + kR;
constexpr unsigned kOnes = 1u | (1u << 10) | (1u << 20);
constexpr unsigned kFarCell = 0x80000000u;
static_assert(kCellLo == 32 && kCellLo + kDE <= 64, "the tile test below");

__device__ __forceinline__ bool in_tile(unsigned c) {
  constexpr unsigned high = 0xc0000000u | (0x3e0u * kOnes), want = 0x20u * kOnes;
  return (((c & high) ^ want) | ((c + (unsigned)(64 - kCellLo - kDE) * kOnes) & (0x40u * kOnes))) == 0u;
}
// index of a tile-form cell in the deposit tile
__device__ __forceinline__ int dep_index(unsigned c) {
  return (int)((c & 1023u) + kDE * ((c >> 10) & 1023u) + (kDE * kDE) * (c >> 20)) - kCellLo * (1 + kDE + kDE * kDE);
}
// the tile form of the global cell (i, j, k), or its far form
__device__ __forceinline__ unsigned local_cell(const int (&uo)[3], const int (&n3)[3], int32_t cell) {
  const int g[3] = {cell_i(cell), cell_j(cell), cell_k(cell)};
  unsigned c = 0;
  bool in = true;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int r = g[q] - uo[q];  // periodic offset from the unit origin, valid within the tile
    if (r >= n3[q] - kR) r -= n3[q];
    else if (r < kDE - kR - n3[q]) r += n3[q];
    in = in && (unsigned)(r + kR) < (unsigned)kDE;
    c += (unsigned)(r + kBias) << (10 * q);
  }
  return in ? c : ((unsigned)cell | kFarCell);
}
// the global packed cell of either form
__device__ __forceinline__ int32_t global_cell(const int (&uo)[3], const int (&n3)[3], unsigned c) {
  int g[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int r = uo[q] + (int)((c >> (10 * q)) & 1023u) - kBias;
    r = r < 0 ? r + n3[q] : r;
    g[q] = r >= n3[q] ? r - n3[q] : r;
  }
  return (c & kFarCell) ? (int32_t)(c & ~kFarCell) : pack_cell(g[0], g[1], g[2]);
}

__device__ __noinline__ void commit_far(const TmaArgs& a, unsigned cell, float r0, float r1, float r2) {
  const int64_t c = cell_i((int32_t)cell) + (int64_t)a.nx * (cell_j((int32_t)cell) + (int64_t)a.ny * cell_k((int32_t)cell));
  const float r[3] = {r0, r1, r2};
  const bool free = far_free();
#pragma unroll 1
  for (int q = 0; q < 3; ++q) add_far(a.acc + kAccWords * (q * a.ncell + c), r[q], free);
}

// one sum of impulses of the start cell c (either form): into the shared deposit tile or to the global
// accumulator
__device__ __forceinline__ void commit_record(const TmaArgs& a, int* dep, unsigned c, float r0, float r1, float r2) {
  if (__builtin_expect((int)c >= 0, 1))
    dep_add3(dep + dep_index(c), r0, r1, r2);
  else
    commit_far(a, c & ~kFarCell, r0, r1, r2);
}

template <bool BF16, bool REC, bool PHYS, bool GATHER>
__global__ void __maxnreg__(Shape<PHYS>::kRegs) step_mixed_tma_kernel(const __grid_constant__ CUtensorMap fluid_map,
                                                       const __grid_constant__ TmaArgs a) {
  constexpr int kConsumerWarps = Shape<PHYS>::kConsumerWarps, kT = Shape<PHYS>::kT;
  constexpr int kStageBytes = Shape<PHYS>::kStageBytes;
  extern __shared__ __align__(128) unsigned char smem[];
  float4* fluid = reinterpret_cast<float4*>(smem);                               // [kTE^3]
  int* dep = reinterpret_cast<int*>(smem + kFluidBytes);                         // [3][kDigits][kDE^3]
  unsigned char* ring = smem + kFluidBytes + kDepositBytes;                      // [kStages][kStageBytes]
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + kStages * kStageBytes);
  uint64_t* full = bars;                    // [kStages]   producer -> consumers (bytes landed)
  uint64_t* empty = bars + kStages;         // [kStages]   consumers -> producer (stage free)
  uint64_t* tile_full = bars + 2 * kStages;  // [1]        fluid tile landed
  uint64_t* tile_empty = tile_full + 1;      // [1]        consumers done with a fluid tile
  uint64_t* dep_done = tile_empty + 1;       // [1]        every consumer warp is done with the deposits before a flush
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
  // stages whose deposits no digit word can overflow (a particle adds to a word at most once a step)
  const int flush_stages = kDepMaxAdds / (kT * a.nsteps);
  // tile index of a cell by its fields
  auto tile_index = [](unsigned c) {
    return (int)((c & 1023u) + kTE * ((c >> 10) & 1023u) + (kTE * kTE) * (c >> 20)) -
           (kBias - kG) * (1 + kTE + kTE * kTE);
  };
  int loaded = 0;
  unsigned flushes = 0;
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
    const int64_t A = S & ~int64_t(7);
    const int64_t Z = (E + 7) & ~int64_t(7);
    const int L = kP * ctid;
    // cloud in cell: lanes take their corners in different orders where a warp's particles share few cells, or they would
    // all add to the same words (1e9 particles on 256^3, ten steps 416 against 624 ms, one at a time 500 against 700;
    // 2e7 on 128^3 7.0 against 7.7).  Up to four particles per cell neighbouring cells' words lie side by side and one
    // order is as good or better (8.4e6 on 128^3 3.16 either way, 4.2e6 1.81 against 1.90).
    const int rot = E - S >= 4 * kU * kU * kU ? (lane ^ (lane >> 3)) & 7 : 0;
    // the deposit tile into the global accumulator, once every consumer warp has made its deposits
    auto flush = [&]() -> bool {
      __syncwarp();
      if (lane == 0) mbar_arrive(dep_done);
      if (!mbar_wait(dep_done, flushes & 1)) {
        atomicOr(a.err, 16);
        return false;
      }
      flush_tile(a, dep, uo, ctid, kConsumerWarps * 32);
      __syncwarp();
      if (lane == 0) mbar_arrive(flush_done);
      if (!mbar_wait(flush_done, flushes & 1)) {
        atomicOr(a.err, 32);
        return false;
      }
      ++flushes;
      return true;
    };
    // GATHER: the permutation entries of this stage and of the next, and this stage's ids, are
    // held in registers a stage ahead
    Vec32<kP> pcur{}, pnext{}, gid{};
    if constexpr (GATHER) {
      pcur = gather_perm<kP>(a, A + L, S, E);
      gid = gather_ids(a, pcur, A + L, S, E);
      pnext = gather_perm<kP>(a, A + kT + L, S, E);
    }
    int deposited = 0;  // stages since the last flush
    for (int64_t t0 = A; t0 < Z; t0 += kT) {
      if (deposited == flush_stages) {
        if (!flush()) return;
        deposited = 0;
      }
      ++deposited;
      const int st = (int)(gt % kStages);
      if (!mbar_wait(&full[st], (gt / kStages) & 1)) {
        atomicOr(a.err, 8);
        return;
      }
      ++gt;
      const int64_t w0 = t0 + kWarpParts * warp;  // a warp none of whose particles the unit owns has nothing to do
      if (w0 >= E || w0 + kWarpParts <= S) {
        if (lane == 0) mbar_arrive(&empty[st]);
        continue;
      }
      unsigned char* src = ring + st * kStageBytes;
      const int64_t p0 = t0 + L;
      // owned particles of this lane: [lo, hi) of 0 .. kP - 1 (the rest belong to neighbouring units
      // or lie past the unit); the others are computed too, without branches, as harmless particles of the
      // unit's first cell without mass, and not stored
      const int lo = (int)max((int64_t)0, min((int64_t)kP, S - p0));
      const int hi = (int)max((int64_t)0, min((int64_t)kP, E - p0));
      const bool all_own = lo == 0 && hi == kP;
      int cell[kP];
      float xi[3][kP], v[3][kP], dv[kP];
      if constexpr (GATHER) {
        // this stage's records through the permutation, one 256-bit load each (asked of L2 a stage
        // ago)
        Rec32 r[kP];
#pragma unroll
        for (int j = 0; j < kP; ++j)
          r[j] = (j >= lo && j < hi) ? ld_rec32(a.grec + 2 * (int64_t)pcur.w[j])
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
        if (REC) {
          // the diameters into the stage, from where the records take them
          Vec32<kP> d;
#pragma unroll
          for (int j = 0; j < kP; ++j) d.w[j] = __float_as_uint(r[j].d);
          *reinterpret_cast<Vec32<kP>*>(src + (BF16 ? 4 * kT * 4 + 3 * kT * 2 : 7 * kT * 4) + L * 4) = d;
        } else {
          store_d(a, r, p0, S, E);
        }
#pragma unroll
        for (int j = 0; j < kP; ++j) {
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
        const Vec32<kP> c = *reinterpret_cast<const Vec32<kP>*>(src + L * 4);
        const Vec32<kP> dd = *reinterpret_cast<const Vec32<kP>*>(src + (BF16 ? 4 * kT * 4 + 3 * kT * 2 : 7 * kT * 4) + L * 4);
#pragma unroll
        for (int j = 0; j < kP; ++j) {
          cell[j] = (int)c.w[j];
          dv[j] = __uint_as_float(dd.w[j]);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const Vec32<kP> x = *reinterpret_cast<const Vec32<kP>*>(src + (1 + q) * kT * 4 + L * 4);
#pragma unroll
          for (int j = 0; j < kP; ++j) xi[q][j] = __uint_as_float(x.w[j]);
          if (BF16) {
#pragma unroll
            for (int j = 0; j < kP; j += 2) {
              const float2 f = __bfloat1622float2(
                  *reinterpret_cast<const __nv_bfloat162*>(src + 4 * kT * 4 + q * kT * 2 + (L + j) * 2));
              v[q][j] = f.x;
              v[q][j + 1] = f.y;
            }
          } else {
            const Vec32<kP> w = *reinterpret_cast<const Vec32<kP>*>(src + 4 * kT * 4 + q * kT * 4 + L * 4);
#pragma unroll
            for (int j = 0; j < kP; ++j) v[q][j] = __uint_as_float(w.w[j]);
          }
        }
      }
      if (!all_own) {
#pragma unroll
        for (int j = 0; j < kP; ++j) {
          if (j >= lo && j < hi) continue;
          cell[j] = pack_cell(uo[0], uo[1], uo[2]);
          dv[j] = 1e-5f;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            xi[q][j] = 0.5f;
            v[q][j] = 0.0f;
          }
        }
      }
      unsigned cl[kP];  // the particles' cells in the form of local_cell()
#pragma unroll
      for (int j = 0; j < kP; ++j) cl[j] = local_cell(uo, n3, cell[j]);
      // What the diameter alone decides is computed once and kept in the lane's own part of the stage (its
      // offsets and velocities, which are in registers now): e^{-a dt}, 1 - e^{-a dt}, 1 / a and the
      // mass; in the PHYS instance a dt, the diameter, 1 / a of Stokes drag and the mass.  (BF16
      // velocities leave no 16 bytes per lane in one piece; their stages end in unused bytes.)
      float* coef = reinterpret_cast<float*>(src) + kT + L;  // [3][kT]
      float* mass = reinterpret_cast<float*>(src + (BF16 ? 26 : 16) * kT) + L;
#pragma unroll
      for (int jp = 0; jp < kP; jp += 2) {
        const unsigned long long D = pack2(dv[jp], dv[jp + 1]);
        const unsigned long long DD = mul2(D, D);
        float dd0, dd1, m[2];
        unpack2(DD, dd0, dd1);
        const unsigned long long ADT = mul2(dup2(a.cadt), pack2(rcp_approx(dd0), rcp_approx(dd1)));
        const unsigned long long INV_A = mul2(DD, dup2(a.inv_ca));
        unpack2(mul2(mul2(dup2(a.mcoef), DD), D), m[0], m[1]);
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (jp + e < lo || jp + e >= hi) m[e] = 0.0f;
        unsigned long long EE, E1;
        if (PHYS) {
          EE = ADT;
          E1 = D;
        } else {
          E1 = one_minus_exp2(ADT, &EE);
        }
        *reinterpret_cast<unsigned long long*>(coef + jp) = EE;
        *reinterpret_cast<unsigned long long*>(coef + kT + jp) = E1;
        *reinterpret_cast<unsigned long long*>(coef + 2 * kT + jp) = INV_A;
        *reinterpret_cast<unsigned long long*>(mass + jp) = pack2(m[0], m[1]);
      }
      // ---- the steps: fluid gather, drag and gravity (exponential integrator), relocation and exchanged
      // momentum for two particles at a time as FP32 register pairs.  A particle in a cell of the
      // deposit tile has its whole stencil inside the fluid tile; the rest ("far" particles, rare) read
      // the padded field and commit to the global accumulator.
#pragma unroll 1
      for (int step = 0; step < a.nsteps; ++step) {
        unsigned key[kP];  // the step's start cells
        float J[kP][3];
#pragma unroll
        for (int jp = 0; jp < kP; jp += 2) {
          float up[2][3], f[2][3];
          unsigned bs[2];  // the stencil's base cell
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = jp + e;
            const bool far = (int)cl[j] < 0;
            unsigned c = far ? kCellLo * kOnes : cl[j];
            if (PHYS && a.ngp) {
              // nearest grid point: the value of the start cell
              const float4 t = fluid[tile_index(c)];
              up[e][0] = t.x;
              up[e][1] = t.y;
              up[e][2] = t.z;
              if (__builtin_expect(far, 0)) {
                const float3 g = ngp_padded(a.Up, px, pxy, (int32_t)(cl[j] & ~kFarCell));
                up[e][0] = g.x;
                up[e][1] = g.y;
                up[e][2] = g.z;
              }
            }
            if (!(PHYS && a.ngp) || (PHYS && a.cic)) {
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                const float o = xi[q][j];
                const bool hi2 = o >= 0.5f;
                f[e][q] = o + (hi2 ? -0.5f : 0.5f);
                c -= hi2 ? 0u : 1u << (10 * q);
              }
              bs[e] = c;
            }
            if (!(PHYS && a.ngp)) {
              const float4* bb = fluid + tile_index(c);
              trilerp(bb[0], bb[1], bb[kTE], bb[kTE + 1], bb[kTE * kTE], bb[kTE * kTE + 1], bb[kTE * kTE + kTE],
                      bb[kTE * kTE + kTE + 1], f[e][0], f[e][1], f[e][2], up[e]);
              if (__builtin_expect(far, 0)) {
                const float3 g = gather_padded(a.Up, px, pxy, (int32_t)(cl[j] & ~kFarCell), xi[0][j], xi[1][j], xi[2][j]);
                up[e][0] = g.x;
                up[e][1] = g.y;
                up[e][2] = g.z;
              }
            }
          }
          // the integrator on the pair
          unsigned long long EE = *reinterpret_cast<const unsigned long long*>(coef + jp);
          unsigned long long E1 = *reinterpret_cast<const unsigned long long*>(coef + kT + jp);
          unsigned long long INV_A = *reinterpret_cast<const unsigned long long*>(coef + 2 * kT + jp);
          const unsigned long long M = *reinterpret_cast<const unsigned long long*>(mass + jp);
          unsigned long long Q;
          if (PHYS) {
            // drag rate a = alpha f(Re) / tau (f = 1 for Stokes drag), f from the start-of-step
            // relative velocity; both integrators take the form v' = w + (v - w) E,
            // x' = x + w dt + (v - w) Q with w = u_p + g / a:
            //   exponential:         E = e^{-a dt},       Q = (1 - E) / a
            //   semi-implicit Euler: E = 1 / (1 + a dt),  Q = E dt  (x' = x + dt v')
            unsigned long long ADT = EE;
            if (a.sn) {
              float fac[2], dd[2];
              unpack2(E1, dd[0], dd[1]);
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const float r0 = up[e][0] - v[0][jp + e], r1 = up[e][1] - v[1][jp + e], r2 = up[e][2] - v[2][jp + e];
                fac[e] = sn_factor(a.re_coef * sqrtf(fmaf(r0, r0, fmaf(r1, r1, r2 * r2))) * dd[e]);
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
            Q = mul2(E1, INV_A);
          }
          float o[2][3], t[2][3];
          unsigned long long JP[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const unsigned long long WT = fma2(dup2(a.g[q]), INV_A, pack2(up[0][q], up[1][q]));
            const unsigned long long V = pack2(v[q][jp], v[q][jp + 1]);
            const unsigned long long DVW = sub2(V, WT);
            float vn[2];
            unpack2(fma2(DVW, EE, WT), vn[0], vn[1]);
            if (BF16) {
              // the stored (rounded) velocity change, so that the deposit balances the particles'
              // momentum; the pair is rounded by one packing conversion
              float m0, m1;
              unpack2(M, m0, m1);
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(vn[0], vn[1]);
              vn[0] = __low2float(b2);
              vn[1] = __high2float(b2);
              JP[q] = pack2(__fmul_rn(-m0, __fmul_rn((vn[0] - v[q][jp]) - a.gdt[q], a.s2)),
                            __fmul_rn(-m1, __fmul_rn((vn[1] - v[q][jp + 1]) - a.gdt[q], a.s2)));
            } else {
              // v' - v = -(v - w) (1 - E), without the cancellation of subtracting the rounded v'
              unsigned long long X = fma2(DVW, E1, dup2(a.gdt[q]));
              if (a.s2 != 1.0f) X = mul2(X, dup2(a.s2));
              JP[q] = mul2(M, X);  // in tile units
            }
            const unsigned long long DXV = fma2(WT, dup2(a.dt), mul2(DVW, Q));
            const unsigned long long O = fma2(DXV, dup2(a.inv_h[q]), pack2(xi[q][jp], xi[q][jp + 1]));
            // whole cells carried: floor(o) from an add of 1.5 * 2^23 rounded toward -inf (exact for
            // |o| < 2^22), so no conversion instructions; the offset o - floor(o) lies in [0, 1]
            const unsigned long long T = add_rm2(O, dup2(12582912.0f));
            float x[2];
            unpack2(O, o[0][q], o[1][q]);
            unpack2(T, t[0][q], t[1][q]);
            unpack2(sub2(O, sub2(T, dup2(12582912.0f))), x[0], x[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              xi[q][jp + e] = fminf(x[e], 0.99999994f);
              v[q][jp + e] = vn[e];
            }
          }
          if (PHYS && a.cic) {
            // cloud in cell: J spread over the eight cells of the start-of-step trilinear stencil with its
            // weights, each corner straight into the tile (the adds are exact, so their order does not matter)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              float j3[3], d[2];
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                unpack2(JP[q], d[0], d[1]);
                j3[q] = d[e];
              }
              const unsigned c0 = cl[jp + e];
#pragma unroll 1
              for (int i = 0; i < 8; ++i) {
                const int k = i ^ rot;
                float w = (k & 1) ? f[e][0] : 1.0f - f[e][0];
                w *= (k & 2) ? f[e][1] : 1.0f - f[e][1];
                w *= (k & 4) ? f[e][2] : 1.0f - f[e][2];
                unsigned c = bs[e] + (k & 1) + ((k & 2) << 9) + ((k & 4) << 18);
                if (__builtin_expect((int)c0 < 0 || !in_tile(c), 0)) {
                  // outside the tile: the periodic corner cell in the global accumulator
                  const int32_t g0 = global_cell(uo, n3, c0);
                  const unsigned off = (int)c0 < 0 ? c - kCellLo * kOnes : c - c0;  // corner less start cell
                  int g[3];
#pragma unroll
                  for (int q = 0; q < 3; ++q) {
                    const int s = (int)((off + kOnes) >> (10 * q) & 1023u) - 1;
                    g[q] = ((g0 >> (10 * q)) & 1023) + s;
                    g[q] = g[q] < 0 ? g[q] + n3[q] : (g[q] >= n3[q] ? g[q] - n3[q] : g[q]);
                  }
                  c = (unsigned)pack_cell(g[0], g[1], g[2]) | kFarCell;
                }
                if (jp + e >= lo && jp + e < hi) commit_record(a, dep, c, w * j3[0], w * j3[1], w * j3[2]);
              }
            }
          } else {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              float j0, j1;
              unpack2(JP[q], j0, j1);
              J[jp][q] = j0;
              J[jp + 1][q] = j1;
            }
          }
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int j = jp + e;
            const unsigned c0 = cl[j];
            unsigned c = c0 + __float_as_uint(t[e][0]) + (__float_as_uint(t[e][1]) << 10) +
                         (__float_as_uint(t[e][2]) << 20) - 0x4B400000u * kOnes;
            // moves of fewer than 16 cells from a cell of the tile keep every field in 0 .. 1023
            const bool ok = fabsf(o[e][0]) < 16.0f && fabsf(o[e][1]) < 16.0f && fabsf(o[e][2]) < 16.0f &&
                            (int)c0 >= 0 && in_tile(c);
            if (__builtin_expect(!ok, 0)) {
              const int32_t g0 = global_cell(uo, n3, c0);
              int g[3];
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                const Relocated rl = relocate_general(o[e][q], (g0 >> (10 * q)) & 1023, n3[q]);
                g[q] = rl.cell;
                xi[q][j] = rl.offset;
              }
              c = local_cell(uo, n3, pack_cell(g[0], g[1], g[2]));
            }
            key[j] = (j >= lo && j < hi) ? c0 : kNoKey;
            cl[j] = c;
          }
        }
        if (!(PHYS && a.cic)) {
          // ---- deposit: runs of equal key over the warp's particles: suffix sums within pairs of lanes (four
          // particles), then a segmented suffix scan over the pairs, chains runs in groups of kScanPairs of them.  (The
          // order of the sums is that of four particles per lane, whose results these are to the bit.) ----
          static_assert(kP == 2, "two lanes hold the four particles of a pair");
          const bool even = (lane & 1) == 0;
          const unsigned nk0 = __shfl_down_sync(0xffffffffu, key[0], 1);
          // this lane's particles are of one run; its last one's goes on in the next lane
          const bool same = key[0] == key[1], cont = nk0 == key[1];
          const unsigned sames = __ballot_sync(0xffffffffu, same), conts = __ballot_sync(0xffffffffu, cont);
          // the pairs whose last run goes on in the next pair, at their even lane; those that are one run
          const unsigned links = (__ballot_sync(0xffffffffu, cont && key[1] != kNoKey) >> 1) & kPairLinks;
          const unsigned whole = sames & conts & (sames >> 1) & 0x55555555u;
          float Sx[kP][3];
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            Sx[0][q] = J[0][q] + (same ? J[1][q] : 0.0f);
            const float r = __shfl_down_sync(0xffffffffu, Sx[0][q], 1);
            Sx[1][q] = J[1][q] + (even && cont ? r : 0.0f);
            Sx[0][q] = J[0][q] + (same ? Sx[1][q] : 0.0f);
          }
          const int pair = lane & ~1;
          const bool link = (links >> pair) & 1u;
          float R[3];  // of the pair, in both lanes: the sum of its last run beyond it
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float r = __shfl_sync(0xffffffffu, Sx[0][q], (pair + 2) & 31);
            R[q] = link ? r : 0.0f;
          }
          // through: the pairs from which the next `off` pairs are one run; the scan ends with the last of them
          // (after drift soon)
          unsigned through = links & (whole >> 2);
#pragma unroll
          for (int off = 1; off < kScanPairs; off <<= 1) {
            if (through == 0u) break;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const float r = __shfl_down_sync(0xffffffffu, R[q], 2 * off);
              if ((through >> pair) & 1u) R[q] += r;
            }
            through &= through >> (2 * off);
          }
          const bool head_lane = even ? lane % (2 * kScanPairs) == 0 || !((links >> (lane - 2)) & 1u)
                                      : !((conts >> (lane - 1)) & 1u);
          // a run that starts at the second particle, or the first, goes on to the end of the pair
          const bool to_end1 = !even || (cont && ((sames >> (lane + 1)) & 1u)), to_end0 = to_end1 && same;
          // each lane commits its run sums where they are, one pass per particle slot.  (Packing the sums of
          // few runs, fresh after a sort, into one pass through shared memory gained nothing: ten steps of 6e7
          // particles on 128^3, now 5.5 ms, took 7.01 ms with it and 6.93 ms without.)
#pragma unroll
          for (int j = 0; j < kP; ++j) {
            const bool start = ((j == 0) ? head_lane : (key[j] != key[j - 1])) && key[j] != kNoKey;
            if (start) {
              const bool to_end = j == 0 ? to_end0 : to_end1;
              commit_record(a, dep, key[j], Sx[j][0] + (to_end ? R[0] : 0.0f), Sx[j][1] + (to_end ? R[1] : 0.0f),
                            Sx[j][2] + (to_end ? R[2] : 0.0f));
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kP; ++j) cell[j] = global_cell(uo, n3, cl[j]);
      // ---- store the owned particles (one wide store per array when the lane owns all) ----
      if (REC) {
        // the step before a sort: the cells to the structure of arrays (the sort's keys), the whole
        // state as 32-byte records {cell, offsets | velocity, diameter}, one 256-bit store per
        // particle (a full sector; the sort's gather then reads one sector per particle).  The
        // diameters are read again from the stage.  BF16 handles store the (BF16-exact) velocities
        // as FP32 in the record.
        const Vec32<kP> d = *reinterpret_cast<const Vec32<kP>*>(src + (BF16 ? 4 * kT * 4 + 3 * kT * 2 : 7 * kT * 4) + L * 4);
        if (all_own) {
          Vec32<kP> c;
#pragma unroll
          for (int j = 0; j < kP; ++j) c.w[j] = (uint32_t)cell[j];
          stcs(a.s.cell + p0, c);
        }
#pragma unroll
        for (int j = 0; j < kP; ++j) {
          if (j < lo || j >= hi) continue;
          if (!all_own) a.s.cell[p0 + j] = cell[j];
          st_rec32(a.rec + 2 * (p0 + j), Rec32{__int_as_float(cell[j]), xi[0][j], xi[1][j], xi[2][j], v[0][j], v[1][j],
                                               v[2][j], __uint_as_float(d.w[j])});
        }
      } else if (all_own) {
        Vec32<kP> c;
#pragma unroll
        for (int j = 0; j < kP; ++j) c.w[j] = (uint32_t)cell[j];
        stcs(a.s.cell + p0, c);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          stcs(a.s.xi[q] + p0, vec(xi[q]));
          if (BF16) {
            // exact: the velocities are BF16 values
#pragma unroll
            for (int j = 0; j < kP; j += 2) {
              const __nv_bfloat162 b = __floats2bfloat162_rn(v[q][j], v[q][j + 1]);
              __stcs((unsigned*)((__nv_bfloat16*)a.s.v[q] + p0 + j), *reinterpret_cast<const unsigned*>(&b));
            }
          } else {
            stcs((float*)a.s.v[q] + p0, vec(v[q]));
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < kP; ++j) {
          if (j < lo || j >= hi) continue;
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
      // the coefficients and records were written through the generic proxy; order them before the producer's
      // next bulk copy into this stage
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
    }
    // all gathers of this unit are done: the producer may reuse its fluid buffer
    __syncwarp();
    if (lane == 0) mbar_arrive(tile_empty);
    if (!flush()) return;
    ++loaded;
  }
}

}  // namespace

bool tma_step_supported(const st_ctx* h) {
  if (h->prec == ST_FP64) return false;
  if (h->geo.B < kU) return false;
  for (int q = 0; q < 3; ++q)
    if (h->geo.n[q] % h->geo.B != 0 || h->geo.n[q] < kTE) return false;
  return h->fluid_pad.p != nullptr;
}

cudaError_t launch_step_mixed_tma(st_ctx* h, const StepParams& p, bool records, bool gather) {
  const bool bf = h->prec == ST_MIXED_BF16V;
  const bool phys = p.ngp || p.semi || p.sn || p.cic;
  if (p.nsteps < 1 || p.nsteps > kMaxFusedSteps) return cudaErrorInvalidValue;
  // a single step of many particles is bound by HBM: a kernel of its own, with the same results
  if (p.nsteps == 1 && h->np >= kSingleParticles && !p.cic && !(records && gather) && !(phys && (records || gather)))
    return launch_step_mixed_tma_single(h, p, records, gather);
  using Kern = void (*)(const CUtensorMap, const TmaArgs);
  static const Kern table[16] = {
      step_mixed_tma_kernel<false, false, false, false>, step_mixed_tma_kernel<true, false, false, false>,
      step_mixed_tma_kernel<false, true, false, false>,  step_mixed_tma_kernel<true, true, false, false>,
      step_mixed_tma_kernel<false, false, true, false>,  step_mixed_tma_kernel<true, false, true, false>,
      step_mixed_tma_kernel<false, true, true, false>,   step_mixed_tma_kernel<true, true, true, false>,
      step_mixed_tma_kernel<false, false, false, true>,  step_mixed_tma_kernel<true, false, false, true>,
      step_mixed_tma_kernel<false, true, false, true>,   step_mixed_tma_kernel<true, true, false, true>,
      step_mixed_tma_kernel<false, false, true, true>,   step_mixed_tma_kernel<true, false, true, true>,
      step_mixed_tma_kernel<false, true, true, true>,    step_mixed_tma_kernel<true, true, true, true>};
  static std::atomic<bool> attr_set[16][kAttrDevices];
  const int variant = (int)bf + 2 * (int)records + 4 * (int)phys + 8 * (int)gather;
  const Kern kern = table[variant];
  const int threads = phys ? Shape<true>::kThreads : Shape<false>::kThreads;
  const int smem = phys ? Shape<true>::kSmemBytes : Shape<false>::kSmemBytes;
  CUtensorMap map;
  cudaError_t e = allow_smem(attr_set[variant], h->dev, kern, smem);
  if (e == cudaSuccess) e = field_map(h, &map);
  if (e != cudaSuccess) return e;
  TmaArgs a = tma_args(h, p, records, gather);
  {
    // tile units: 2^(E - kDepShift) in the mass coefficient as far as it stays an FP32 number (a power of two: the
    // impulses' bits do not change), the rest in s2, which is 1 unless the impulses are tiny; beyond +-250 every scaled impulse is 0 or overflows the
    // bound the exponent was chosen for, so clamping changes nothing
    const int Es = std::min(std::max(p.E - kDepShift, -250), 250);
    const int k1 = std::min(Es, 100 - std::ilogb(std::max(p.mcoef, 1e-300)));
    a.mcoef = (float)std::ldexp(p.mcoef, k1);
    a.s1 = 1.0f;
    a.s2 = std::ldexp(1.0f, Es - k1);
  }
  kern<<<tma_grid(h, a.nunits), threads, smem, h->stream>>>(map, a);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace st
