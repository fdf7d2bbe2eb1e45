// Step (b) on the 5th-generation tensor cores: the per-layer mode contraction
//   S_l = W_l C_l,   W_l in C^{3M x 4M},  C_l[j][f] = c_j(z_f)          (Eq. 34, Sec. 4.1)
// written as one real GEMM. A = W viewed as interleaved reals (3M x 8M: the
// complex64 memory layout itself), B = [[Re C, Im C], [-Im C, Re C]] in the
// same interleaving (8M x NB, NB = 2 F_pad), D = [Re S | Im S] (3M x NB).
//
// Precision modes:
//   split-BF16: A = A_hi + A_lo, B = B_hi + B_lo (BF16 each); the three products
//               A_hi B_hi + A_hi B_lo + A_lo B_hi accumulate in one FP32 TMEM tile.
//   FP16:       A in FP16, B = B_hi + B_lo (FP16); two products.
//
// Persistent, warp-specialised kernel. Work is a list of tasks (item, unit,
// 128-row tile, K split), grouped per CTA on the host longest-first; every role
// walks the same list:
//   warp 0          producer: contiguous cp.async.bulk copies (no multicast) of
//                   the pre-swizzled tile-major A tiles (L2 evict-first: W is
//                   streamed once) and B chunks (evict-last: re-read by every row
//                   tile) into a ring of shared-memory stages (full/empty mbarriers)
//   warp 1          tcgen05.mma issuer (M = 128, N = NB, K = 16 per instruction)
//                   into one of two TMEM accumulators (acc_full/acc_empty)
//   warps 2-5       epilogue: tcgen05.ld 32 lanes x 8 columns of the other
//                   accumulator, coalesced stores of S_part[split][plane][row]
// so loads, MMAs and the previous task's epilogue overlap. Both issuing roles run warp-converged with
// one elected lane (ptx::elect_one). Every wait is bounded
// by a %globaltimer deadline; a timeout sets the error word and all roles stop.
#include "scw_internal.cuh"
#include "scw_ptx.cuh"

namespace scw {

template <int NB, bool SPLIT>
struct TcCfg {
  static constexpr uint32_t A_BYTES = 128u * 64u * 2u;
  static constexpr uint32_t B_BYTES = (uint32_t)NB * 64u * 2u;
  static constexpr int NA = SPLIT ? 2 : 1;
  static constexpr uint32_t STAGE_BYTES = NA * A_BYTES + 2 * B_BYTES;
  // two CTAs per SM while at least three stages fit in ~110 KB, else one CTA with up to ~220 KB
  static constexpr int STAGES_2 = (int)(110u * 1024u / STAGE_BYTES);
  static constexpr int CTAS_PER_SM = STAGES_2 >= 3 ? 2 : 1;
  static constexpr int STAGES_RAW = CTAS_PER_SM == 2 ? STAGES_2 : (int)(220u * 1024u / STAGE_BYTES);
  static constexpr int STAGES = STAGES_RAW > 8 ? 8 : STAGES_RAW;
  static constexpr uint32_t SMEM = STAGES * STAGE_BYTES + 1024u;
  static constexpr uint32_t ACC_COLS = NB <= 32 ? 32u : (NB <= 64 ? 64u : (NB <= 128 ? 128u : 256u));
  static constexpr uint32_t TMEM_COLS = 2 * ACC_COLS;
};

struct TaskGeom {
  int kb, kcount, layer, unit, tile, split, f0, nf, rt;
};

__device__ __forceinline__ TaskGeom task_geom(const int4 tk, const ItemDev& it) {
  TaskGeom g;
  const LayerUnit u = it.units[tk.y];
  const int ks = u.ks > 0 ? u.ks : it.k_split;
  const int per = (it.nk + ks - 1) / ks;
  g.kb = tk.w * per;
  g.kcount = max(0, min(it.nk, g.kb + per) - g.kb);
  g.layer = u.layer;
  g.unit = tk.y;
  g.tile = tk.z;
  g.split = tk.w;
  g.f0 = u.f0;
  g.nf = u.nf;
  g.rt = min(it.rows_tile, 3 * it.M - it.rows_tile * tk.z);  // rows of this tile that exist
  return g;
}

template <int NB, bool SPLIT, bool BATCH>
__global__ void __launch_bounds__(192) contract_tc_kernel(const __grid_constant__ ItemDev one,
                                                          const ItemDev* __restrict__ items,
                                                          const int4* __restrict__ tasks,
                                                          const int* __restrict__ cta_off, int* err,
                                                          uint64_t timeout_ns, int inject_stall) {
  using Cfg = TcCfg<NB, SPLIT>;
  constexpr int STAGES = Cfg::STAGES;
  constexpr int FP = NB / 2;  // plane slots
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES];
  __shared__ __align__(8) uint64_t empty_bar[STAGES];
  __shared__ __align__(8) uint64_t accf_bar[2];
  __shared__ __align__(8) uint64_t acce_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t_begin = cta_off[blockIdx.x], t_end = cta_off[blockIdx.x + 1];
  const uint64_t deadline = ptx::globaltimer() + timeout_ns;
  ptx::griddep_launch_dependents();  // the recomposition may be scheduled as CTAs of this grid finish
  trace_begin(one.trace, TRACE_CONTRACT);

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) {
      ptx::mbar_init(ptx::smem_u32(&full_bar[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&empty_bar[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(ptx::smem_u32(&accf_bar[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&acce_bar[i]), 4);  // one arrival per epilogue warp
    }
    ptx::mbar_init(ptx::smem_u32(&drain_bar), 1);
    abort_s = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(&tmem_base_s), Cfg::TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = tmem_base_s;

  if (warp == 0) {
    // ---------------- bulk-copy producer ----------------
    const uint32_t leader = ptx::elect_one();
    const uint64_t pol_a = ptx::policy_evict_first(), pol_b = ptx::policy_evict_last();
    int st = 0;
    uint32_t ph = 0;
    int issued = 0, skipped = -1;
    // W does not depend on the phase kernel that precedes this grid (programmatic launch): the first
    // ring of stages gets its A copies at once, their B copies follow once that kernel has finished
    bool dep_done = false;
    int npend = 0;
    uint32_t pend_sb[STAGES], pend_fb[STAGES];
    const uint16_t* pend_bh[STAGES];
    const uint16_t* pend_bl[STAGES];
    auto flush_pending = [&]() {
      ptx::griddep_wait();
      for (int q = 0; q < npend; ++q) {
        ptx::bulk_load(pend_sb[q], pend_bh[q], Cfg::B_BYTES, pend_fb[q], pol_b, leader);
        ptx::bulk_load(pend_sb[q] + Cfg::B_BYTES, pend_bl[q], Cfg::B_BYTES, pend_fb[q], pol_b, leader);
      }
      npend = 0;
      dep_done = true;
    };
    for (int t = t_begin; t < t_end && !ptx::warp_any(abort_s); ++t) {
      const int4 tk = tasks[t];
      const ItemDev& it = BATCH ? items[tk.x] : one;
      const TaskGeom g = task_geom(tk, it);
      const int R = 3 * it.M;
      // element offsets of this tile's first chunk in A and of the unit's first chunk in B
      const size_t a0 = (size_t)g.layer * R * it.nk * 64 + (size_t)g.tile * it.rows_tile * it.nk * 64;
      const size_t b0 = (size_t)g.unit * it.nk * NB * 64;
      const uint32_t a_bytes = (uint32_t)g.rt * 128u;
      const uint32_t tx = Cfg::NA * a_bytes + 2u * Cfg::B_BYTES;
      const uint16_t* Ah = static_cast<const uint16_t*>(it.Ahi);
      const uint16_t* Al = static_cast<const uint16_t*>(it.Alo);
      const uint16_t* Bh = static_cast<const uint16_t*>(it.Bhi);
      const uint16_t* Bl = static_cast<const uint16_t*>(it.Blo);
      for (int i = 0; i < g.kcount; ++i) {
        if (!ptx::mbar_wait_warp(ptx::smem_u32(&empty_bar[st]), ph ^ 1u, deadline)) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_EMPTY);
          abort_s = 1;
          break;
        }
        const uint32_t fb = ptx::smem_u32(&full_bar[st]);
        if (inject_stall && blockIdx.x == 0 && issued == 0) {
          skipped = 0;  // failure injection (scw_plan_inject_stall): this stage is never filled
        } else {
          ptx::mbar_arrive_expect_tx(fb, tx, leader);
          const int kc = g.kb + i;
          const uint32_t sa = ptx::smem_u32(smem + (size_t)st * Cfg::STAGE_BYTES);
          const size_t ao = a0 + (size_t)kc * g.rt * 64;
          ptx::bulk_load(sa, Ah + ao, a_bytes, fb, pol_a, leader);
          if (SPLIT) ptx::bulk_load(sa + Cfg::A_BYTES, Al + ao, a_bytes, fb, pol_a, leader);
          const uint32_t sb = sa + Cfg::NA * Cfg::A_BYTES;
          const size_t bo = b0 + (size_t)kc * NB * 64;
          if (dep_done) {
            ptx::bulk_load(sb, Bh + bo, Cfg::B_BYTES, fb, pol_b, leader);
            ptx::bulk_load(sb + Cfg::B_BYTES, Bl + bo, Cfg::B_BYTES, fb, pol_b, leader);
          } else {
            pend_sb[npend] = sb;
            pend_fb[npend] = fb;
            pend_bh[npend] = Bh + bo;
            pend_bl[npend] = Bl + bo;
            if (++npend == STAGES) flush_pending();
          }
        }
        ++issued;
        if (++st == STAGES) {
          st = 0;
          ph ^= 1u;
        }
      }
    }
    if (!dep_done) flush_pending();  // fewer stages than the ring, or an early stop
    if (ptx::warp_any(abort_s)) {
      // let the last issued copies land before the CTA's shared memory goes away
      const uint64_t d2 = ptx::drain_deadline(timeout_ns);
      for (int back = 1; back <= STAGES && back <= issued; ++back) {
        const int i = issued - back;
        if (i == skipped) continue;  // nothing was sent to that stage
        if (!ptx::mbar_wait_warp(ptx::smem_u32(&full_bar[i % STAGES]), (uint32_t)(i / STAGES) & 1u, d2)) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_DRAIN);
          break;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- tcgen05.mma issuer ----------------
    const uint32_t leader = ptx::elect_one();
    constexpr uint32_t idesc = ptx::idesc_f16(SPLIT, 128, NB);
    int st = 0;
    uint32_t ph = 0;
    int lt = 0;
    for (int t = t_begin; t < t_end && !ptx::warp_any(abort_s); ++t, ++lt) {
      const int4 tk = tasks[t];
      const ItemDev& it = BATCH ? items[tk.x] : one;
      const TaskGeom g = task_geom(tk, it);
      const int acc = lt & 1;
      if (!ptx::mbar_wait_warp(ptx::smem_u32(&acce_bar[acc]), ((uint32_t)(lt >> 1) & 1u) ^ 1u, deadline)) {
        if (leader) atomicOr(err, DEV_ERR_TIMEOUT_ACCUM);
        abort_s = 1;
        break;
      }
      ptx::tc_fence_after();
      const uint32_t d_tmem = tmem + (uint32_t)acc * Cfg::ACC_COLS;
      for (int i = 0; i < g.kcount; ++i) {
        if (!ptx::mbar_wait_warp(ptx::smem_u32(&full_bar[st]), ph, deadline)) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_FULL);
          abort_s = 1;
          break;
        }
        ptx::tc_fence_after();
        const uint32_t a_hi = ptx::smem_u32(smem + (size_t)st * Cfg::STAGE_BYTES);
        const uint32_t a_lo = a_hi + Cfg::A_BYTES;
        const uint32_t b_hi = a_hi + Cfg::NA * Cfg::A_BYTES;
        const uint32_t b_lo = b_hi + Cfg::B_BYTES;
        const uint64_t dah = ptx::sw128_desc(a_hi), dal = ptx::sw128_desc(a_lo);
        const uint64_t dbh = ptx::sw128_desc(b_hi), dbl = ptx::sw128_desc(b_lo);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          // K advance of 16 elements = 32 bytes inside the 128-byte swizzle row
          const uint64_t o = (uint64_t)(2 * kk);
          ptx::mma_f16(d_tmem, dah + o, dbh + o, idesc, (i > 0 || kk > 0) ? 1u : 0u, leader);
          ptx::mma_f16(d_tmem, dah + o, dbl + o, idesc, 1u, leader);
          if (SPLIT) ptx::mma_f16(d_tmem, dal + o, dbh + o, idesc, 1u, leader);
        }
        ptx::mma_commit(ptx::smem_u32(&empty_bar[st]), leader);
        if (++st == STAGES) {
          st = 0;
          ph ^= 1u;
        }
      }
      ptx::mma_commit(ptx::smem_u32(&accf_bar[acc]), leader);
    }
    if (ptx::warp_any(abort_s)) {
      // issued MMAs must finish before the tensor memory is released
      ptx::mma_commit(ptx::smem_u32(&drain_bar), leader);
      if (!ptx::mbar_wait_warp(ptx::smem_u32(&drain_bar), 0u, ptx::drain_deadline(timeout_ns)))
        if (leader) atomicOr(err, DEV_ERR_TIMEOUT_DRAIN);
    }
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int grp = warp & 3;  // TMEM lanes 32*grp .. 32*grp+31
    // partial spectra are read back right after this kernel: keep them in L2 while W streams through
    const uint64_t pol_s = ptx::policy_evict_last();
    int lt = 0;
    for (int t = t_begin; t < t_end && !abort_s; ++t, ++lt) {
      const int4 tk = tasks[t];
      const ItemDev& it = BATCH ? items[tk.x] : one;
      const TaskGeom g = task_geom(tk, it);
      const int acc = lt & 1;
      const bool ok = ptx::mbar_wait(ptx::smem_u32(&accf_bar[acc]), (uint32_t)(lt >> 1) & 1u, deadline);
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) atomicOr(err, DEV_ERR_TIMEOUT_ACCUM);
        abort_s = 1;
        break;
      }
      ptx::tc_fence_after();
      const int rows = 3 * it.M;
      const int rl = grp * 32 + lane;  // row within the tile
      const int row = g.tile * it.rows_tile + rl;
      float2* dst = it.S_part + ((size_t)g.split * it.Fz + g.f0) * rows;
      const uint32_t lane_addr = tmem + (uint32_t)acc * Cfg::ACC_COLS + ((uint32_t)(grp * 32) << 16);
#pragma unroll 1
      for (int f0 = 0; f0 < FP; f0 += 8) {
        uint32_t re[8], im[8];
        if (g.kcount > 0) {
          ptx::tmem_ld_x8(lane_addr + (uint32_t)f0, re);
          ptx::tmem_ld_x8(lane_addr + (uint32_t)(FP + f0), im);
          ptx::tmem_wait_ld();
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) re[q] = im[q] = 0u;
        }
        if (rl < g.rt) {
          const size_t d0 = ((size_t)g.split * it.Fz + g.f0) * rows + row;
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (f0 + q < g.nf && in_bounds(it, BND_S_PART, d0 + (size_t)(f0 + q) * rows))
              ptx::st_global_hint(dst + (size_t)(f0 + q) * rows + row,
                                  make_float2(__uint_as_float(re[q]), __uint_as_float(im[q])), pol_s);
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&acce_bar[acc]));
    }
  }

  // ---------------- teardown ----------------
  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  trace_end(one.trace, TRACE_CONTRACT);
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, Cfg::TMEM_COLS);
  }
}

// ---- 128 plane slots per unit (NB = 256) ----------------------------------------------------------------
// A K chunk of B takes 64 KB of shared memory here, against 32 KB of A, and as one stage with A only two
// fit: a chunk's B could be requested no earlier than one chunk ahead and took 1.2 us where its MMAs take
// 0.8. So A and B have rings of their own, and B's is cut into halves of 128 columns, multiplied one after
// the other (N = 128): four half chunks of B and three chunks of A (from memory) are in flight, and a half is
// requested again as soon as its own MMAs are done. The same products in the same order. 16 illuminations
// at 21 x 21 orders, 32 layers of 8 planes: 174 -> 161 us, 1425 TFLOP/s of the three products, 0.84 of the tensor
// cores' rate under the power cap (0.91 with padded rows and K counted). (Two row tiles per task, so that a B chunk
// is used twice, leave no tensor memory for a second set of accumulators: 191 us.)
template <bool SPLIT>
struct RingCfg {
  static constexpr int NB = 256, HB = 128;
  static constexpr uint32_t A_TILE = 128u * 64u * 2u;
  static constexpr int NA = SPLIT ? 2 : 1;
  static constexpr uint32_t A_STAGE = NA * A_TILE;
  static constexpr uint32_t B_HALF = (uint32_t)HB * 64u * 2u;  // hi or lo of half a chunk
  static constexpr uint32_t B_STAGE = 2 * B_HALF;
  static constexpr int BS = 4;
  static constexpr int AS = SPLIT ? 3 : 6;
  static constexpr uint32_t SMEM = BS * B_STAGE + AS * A_STAGE + 1024u;
  static constexpr uint32_t TMEM_COLS = 512u;  // two accumulators
};
constexpr int kRingThreads = 320;

template <bool SPLIT, bool BATCH>
__global__ void __launch_bounds__(kRingThreads) contract_ring_kernel(const __grid_constant__ ItemDev one,
                                                                     const ItemDev* __restrict__ items,
                                                                     const int4* __restrict__ tasks,
                                                                     const int* __restrict__ cta_off, int* err,
                                                                     uint64_t timeout_ns, int inject_stall) {
  using Cfg = RingCfg<SPLIT>;
  constexpr int AS = Cfg::AS, BS = Cfg::BS, NB = Cfg::NB, NACC = 2;
  constexpr int FP = NB / 2;  // plane slots
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t afull[AS], aempty[AS], bfull[BS], bempty[BS], accf_bar[NACC], acce_bar[NACC], drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smem_a = smem + BS * Cfg::B_STAGE;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t_begin = cta_off[blockIdx.x], t_end = cta_off[blockIdx.x + 1];
  const uint64_t deadline = ptx::globaltimer() + timeout_ns;
  ptx::griddep_launch_dependents();
  trace_begin(one.trace, TRACE_CONTRACT);

  if (threadIdx.x == 0) {
    for (int i = 0; i < AS; ++i) {
      ptx::mbar_init(ptx::smem_u32(&afull[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&aempty[i]), 1);
    }
    for (int i = 0; i < BS; ++i) {
      ptx::mbar_init(ptx::smem_u32(&bfull[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&bempty[i]), 1);
    }
    for (int i = 0; i < NACC; ++i) {
      ptx::mbar_init(ptx::smem_u32(&accf_bar[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&acce_bar[i]), 8);  // one arrival per epilogue warp
    }
    ptx::mbar_init(ptx::smem_u32(&drain_bar), 1);
    abort_s = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(&tmem_base_s), Cfg::TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = tmem_base_s;

  if (warp == 0) {
    // ---------------- bulk-copy producer ----------------
    const uint32_t leader = ptx::elect_one();
    const uint64_t pol_a = ptx::policy_evict_first(), pol_b = ptx::policy_evict_last();
    int as = 0, bs = 0, a_issued = 0, b_issued = 0;
    uint32_t aph = 0, bph = 0;
    bool stalled = false, dep_done = false;  // stalled: failure injection, the first A chunk is never sent
    for (int t = t_begin; t < t_end && !ptx::warp_any(abort_s); ++t) {
      const int4 tk = tasks[t];
      const ItemDev& it = BATCH ? items[tk.x] : one;
      const TaskGeom g = task_geom(tk, it);
      const size_t a0 = ((size_t)g.layer * 3 * it.M + (size_t)g.tile * it.rows_tile) * it.nk * 64;
      const size_t b0 = (size_t)g.unit * it.nk * NB * 64;
      const uint32_t a_bytes = (uint32_t)g.rt * 128u;
      const uint16_t* Ah = static_cast<const uint16_t*>(it.Ahi);
      const uint16_t* Al = static_cast<const uint16_t*>(it.Alo);
      const uint16_t* Bh = static_cast<const uint16_t*>(it.Bhi);
      const uint16_t* Bl = static_cast<const uint16_t*>(it.Blo);
      for (int i = 0; i < g.kcount; ++i) {
        const int kc = g.kb + i;
        bool ok = ptx::mbar_wait_warp(ptx::smem_u32(&aempty[as]), aph ^ 1u, deadline);
        if (ok) {
          if (inject_stall && blockIdx.x == 0 && a_issued == 0) {
            stalled = true;
          } else {
            const uint32_t fb = ptx::smem_u32(&afull[as]);
            const uint32_t sa = ptx::smem_u32(smem_a + (size_t)as * Cfg::A_STAGE);
            const size_t ao = a0 + (size_t)kc * g.rt * 64;
            ptx::mbar_arrive_expect_tx(fb, Cfg::NA * a_bytes, leader);
            ptx::bulk_load(sa, Ah + ao, a_bytes, fb, pol_a, leader);
            if (SPLIT) ptx::bulk_load(sa + Cfg::A_TILE, Al + ao, a_bytes, fb, pol_a, leader);
          }
          ++a_issued;
          if (++as == AS) {
            as = 0;
            aph ^= 1u;
          }
        }
        // W does not depend on the phase kernel that precedes this grid (programmatic launch), B does
        if (!dep_done) ptx::griddep_wait();
        dep_done = true;
        for (int h = 0; ok && h < 2; ++h) {
          ok = ptx::mbar_wait_warp(ptx::smem_u32(&bempty[bs]), bph ^ 1u, deadline);
          if (!ok) break;
          const uint32_t fb = ptx::smem_u32(&bfull[bs]);
          const uint32_t sb = ptx::smem_u32(smem + (size_t)bs * Cfg::B_STAGE);
          const size_t bo = b0 + ((size_t)kc * NB + h * Cfg::HB) * 64;
          ptx::mbar_arrive_expect_tx(fb, Cfg::B_STAGE, leader);
          ptx::bulk_load(sb, Bh + bo, Cfg::B_HALF, fb, pol_b, leader);
          ptx::bulk_load(sb + Cfg::B_HALF, Bl + bo, Cfg::B_HALF, fb, pol_b, leader);
          ++b_issued;
          if (++bs == BS) {
            bs = 0;
            bph ^= 1u;
          }
        }
        if (!ok) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_EMPTY);
          abort_s = 1;
          break;
        }
      }
    }
    if (!dep_done) ptx::griddep_wait();
    if (ptx::warp_any(abort_s)) {
      // let the last issued copies land before the CTA's shared memory goes away
      const uint64_t d2 = ptx::drain_deadline(timeout_ns);
      bool ok = true;
      for (int back = 1; ok && back <= AS && back <= a_issued; ++back) {
        const int i = a_issued - back;
        if (stalled && i == 0) continue;  // nothing was sent to that stage
        ok = ptx::mbar_wait_warp(ptx::smem_u32(&afull[i % AS]), (uint32_t)(i / AS) & 1u, d2);
      }
      for (int back = 1; ok && back <= BS && back <= b_issued; ++back) {
        const int i = b_issued - back;
        ok = ptx::mbar_wait_warp(ptx::smem_u32(&bfull[i % BS]), (uint32_t)(i / BS) & 1u, d2);
      }
      if (!ok && leader) atomicOr(err, DEV_ERR_TIMEOUT_DRAIN);
    }
  } else if (warp == 1) {
    // ---------------- tcgen05.mma issuer ----------------
    const uint32_t leader = ptx::elect_one();
    constexpr uint32_t idesc = ptx::idesc_f16(SPLIT, 128, Cfg::HB);
    int as = 0, bs = 0, lt = 0;
    uint32_t aph = 0, bph = 0;
    for (int t = t_begin; t < t_end && !ptx::warp_any(abort_s); ++t, ++lt) {
      const int4 tk = tasks[t];
      const ItemDev& it = BATCH ? items[tk.x] : one;
      const TaskGeom g = task_geom(tk, it);
      const int acc = lt % NACC;
      if (!ptx::mbar_wait_warp(ptx::smem_u32(&acce_bar[acc]), ((uint32_t)(lt / NACC) & 1u) ^ 1u, deadline)) {
        if (leader) atomicOr(err, DEV_ERR_TIMEOUT_ACCUM);
        abort_s = 1;
        break;
      }
      ptx::tc_fence_after();
      bool ok = true;
      for (int i = 0; i < g.kcount && ok; ++i) {
        ok = ptx::mbar_wait_warp(ptx::smem_u32(&afull[as]), aph, deadline);
        const uint32_t a_hi = ptx::smem_u32(smem_a + (size_t)as * Cfg::A_STAGE);
        const uint64_t dah = ptx::sw128_desc(a_hi), dal = ptx::sw128_desc(a_hi + Cfg::A_TILE);
        for (int h = 0; ok && h < 2; ++h) {
          ok = ptx::mbar_wait_warp(ptx::smem_u32(&bfull[bs]), bph, deadline);
          if (!ok) break;
          ptx::tc_fence_after();
          const uint32_t d_tmem = tmem + (uint32_t)(acc * NB + h * Cfg::HB);
          const uint32_t b_hi = ptx::smem_u32(smem + (size_t)bs * Cfg::B_STAGE);
          const uint64_t dbh = ptx::sw128_desc(b_hi), dbl = ptx::sw128_desc(b_hi + Cfg::B_HALF);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint64_t o = (uint64_t)(2 * kk);
            ptx::mma_f16(d_tmem, dah + o, dbh + o, idesc, (i > 0 || kk > 0) ? 1u : 0u, leader);
            ptx::mma_f16(d_tmem, dah + o, dbl + o, idesc, 1u, leader);
            if (SPLIT) ptx::mma_f16(d_tmem, dal + o, dbh + o, idesc, 1u, leader);
          }
          ptx::mma_commit(ptx::smem_u32(&bempty[bs]), leader);
          if (++bs == BS) {
            bs = 0;
            bph ^= 1u;
          }
        }
        if (!ok) break;
        ptx::mma_commit(ptx::smem_u32(&aempty[as]), leader);
        if (++as == AS) {
          as = 0;
          aph ^= 1u;
        }
      }
      if (!ok) {
        if (leader) atomicOr(err, DEV_ERR_TIMEOUT_FULL);
        abort_s = 1;
        break;
      }
      ptx::mma_commit(ptx::smem_u32(&accf_bar[acc]), leader);
    }
    if (ptx::warp_any(abort_s)) {
      // issued MMAs must finish before the tensor memory is released
      ptx::mma_commit(ptx::smem_u32(&drain_bar), leader);
      if (!ptx::mbar_wait_warp(ptx::smem_u32(&drain_bar), 0u, ptx::drain_deadline(timeout_ns)))
        if (leader) atomicOr(err, DEV_ERR_TIMEOUT_DRAIN);
    }
  } else {
    // ---------------- epilogue: two warps per 32-lane quadrant, one per half of the planes ----------------
    const int grp = warp & 3, h = (warp - 2) >> 2;  // TMEM lanes 32 grp .. 32 grp + 31
    const uint64_t pol_s = ptx::policy_evict_last();
    int lt = 0;
    for (int t = t_begin; t < t_end; ++t, ++lt) {
      const int4 tk = tasks[t];
      const ItemDev& it = BATCH ? items[tk.x] : one;
      const TaskGeom g = task_geom(tk, it);
      const int acc = lt % NACC;
      bool ok = true;
      for (;;) {
        if (ptx::mbar_try_wait(ptx::smem_u32(&accf_bar[acc]), (uint32_t)(lt / NACC) & 1u)) break;
        if (abort_s || ptx::globaltimer() > deadline) {
          ok = false;
          break;
        }
      }
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0 && !abort_s) atomicOr(err, DEV_ERR_TIMEOUT_ACCUM);
        abort_s = 1;
        break;
      }
      ptx::tc_fence_after();
      const int rows = 3 * it.M;
      const int rl = grp * 32 + lane;  // row within the tile
      const int row = g.tile * it.rows_tile + rl;
      const size_t d0 = ((size_t)g.split * it.Fz + g.f0) * rows + row;
      float2* dst = it.S_part + d0;
      const uint32_t lane_addr = tmem + (uint32_t)(acc * NB) + ((uint32_t)(grp * 32) << 16);
#pragma unroll 1
      for (int f0 = h * (FP / 2); f0 < (h + 1) * (FP / 2) && f0 < g.nf; f0 += 8) {
        uint32_t re[8], im[8];
        if (g.kcount > 0) {
          ptx::tmem_ld_x8(lane_addr + (uint32_t)f0, re);
          ptx::tmem_ld_x8(lane_addr + (uint32_t)(FP + f0), im);
          ptx::tmem_wait_ld();
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) re[q] = im[q] = 0u;
        }
        if (rl < g.rt) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (f0 + q < g.nf && in_bounds(it, BND_S_PART, d0 + (size_t)(f0 + q) * rows))
              ptx::st_global_hint(dst + (size_t)(f0 + q) * rows,
                                  make_float2(__uint_as_float(re[q]), __uint_as_float(im[q])), pol_s);
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&acce_bar[acc]));
    }
  }

  // ---------------- teardown ----------------
  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  trace_end(one.trace, TRACE_CONTRACT);
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, Cfg::TMEM_COLS);
  }
}

// ---------------------------------------------------------------- host side ---
template <int NB, bool SPLIT>
static cudaError_t launch_tc_t(const ItemDev& one, const ItemDev* items, const TcSchedule& s, int* err,
                               uint64_t timeout_ns, int inject, cudaStream_t st) {
  using Cfg = TcCfg<NB, SPLIT>;
  cudaError_t e;
  if (items) {
    e = allow_max_smem(reinterpret_cast<const void*>(contract_tc_kernel<NB, SPLIT, true>));
    if (e != cudaSuccess) return e;
    e = launch_pdl(contract_tc_kernel<NB, SPLIT, true>, dim3(s.grid), dim3(192), Cfg::SMEM, st, one, items,
                   (const int4*)s.d_tasks, (const int*)s.d_cta_off, err, timeout_ns, inject);
  } else {
    e = allow_max_smem(reinterpret_cast<const void*>(contract_tc_kernel<NB, SPLIT, false>));
    if (e != cudaSuccess) return e;
    e = launch_pdl(contract_tc_kernel<NB, SPLIT, false>, dim3(s.grid), dim3(192), Cfg::SMEM, st, one,
                   (const ItemDev*)nullptr, (const int4*)s.d_tasks, (const int*)s.d_cta_off, err, timeout_ns, inject);
  }
  return e;
}

template <bool SPLIT>
static cudaError_t launch_ring_t(const ItemDev& one, const ItemDev* items, const TcSchedule& s, int* err,
                                 uint64_t timeout_ns, int inject, cudaStream_t st) {
  auto fn = items ? contract_ring_kernel<SPLIT, true> : contract_ring_kernel<SPLIT, false>;
  cudaError_t e = allow_max_smem(reinterpret_cast<const void*>(fn));
  if (e != cudaSuccess) return e;
  return launch_pdl(fn, dim3(s.grid), dim3(kRingThreads), RingCfg<SPLIT>::SMEM, st, one, items,
                    (const int4*)s.d_tasks, (const int*)s.d_cta_off, err, timeout_ns, inject);
}

template <bool SPLIT>
static cudaError_t launch_tc_nb(int NB, const ItemDev& one, const ItemDev* items, const TcSchedule& s, int* err,
                                uint64_t timeout_ns, int inject, cudaStream_t st) {
  switch (NB) {
    case 16: return launch_tc_t<16, SPLIT>(one, items, s, err, timeout_ns, inject, st);
    case 32: return launch_tc_t<32, SPLIT>(one, items, s, err, timeout_ns, inject, st);
    case 48: return launch_tc_t<48, SPLIT>(one, items, s, err, timeout_ns, inject, st);
    case 64: return launch_tc_t<64, SPLIT>(one, items, s, err, timeout_ns, inject, st);
    case 128: return launch_tc_t<128, SPLIT>(one, items, s, err, timeout_ns, inject, st);
    case 256: return launch_ring_t<SPLIT>(one, items, s, err, timeout_ns, inject, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_contract_tc(const ItemDev& one, const ItemDev* items, const TcSchedule& s, int NB, bool bf16,
                               int* err, uint64_t timeout_ns, int inject, cudaStream_t st) {
  if (s.n_tasks == 0 || s.grid == 0) return cudaSuccess;
  return bf16 ? launch_tc_nb<true>(NB, one, items, s, err, timeout_ns, inject, st)
              : launch_tc_nb<false>(NB, one, items, s, err, timeout_ns, inject, st);
}

int tc_ctas_per_sm(int NB, bool bf16) {
  switch (NB) {
    case 16: return bf16 ? TcCfg<16, true>::CTAS_PER_SM : TcCfg<16, false>::CTAS_PER_SM;
    case 32: return bf16 ? TcCfg<32, true>::CTAS_PER_SM : TcCfg<32, false>::CTAS_PER_SM;
    case 48: return bf16 ? TcCfg<48, true>::CTAS_PER_SM : TcCfg<48, false>::CTAS_PER_SM;
    case 64: return bf16 ? TcCfg<64, true>::CTAS_PER_SM : TcCfg<64, false>::CTAS_PER_SM;
    case 128: return bf16 ? TcCfg<128, true>::CTAS_PER_SM : TcCfg<128, false>::CTAS_PER_SM;
    default: return 1;
  }
}

}  // namespace scw
