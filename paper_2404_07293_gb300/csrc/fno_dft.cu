// Truncated DFTs of the surrogate on the 5th-generation tensor cores (BF16 mode), the backward one
// fused with the weight gradient of the 1x1 convolution:
//   Vh[b][i][k] = alpha sum_p V[b][i][p] exp(-2 pi i (kx x + ky y) / N)     on the kept modes
// as D = A B^T over K = pixels: A = activations channel-first (rows (b, i), 128 per tile), B = the DFT
// table (rows (mode, re / im)), both K-major BF16 read by TMA with 128-byte swizzle.
//
// The activations are real, so the modes k and -k are complex conjugates, and the table's values are
// exact mirror images (its angles are reduced in integers): only one mode of each pair is multiplied
// and the epilogue stores its conjugate too. For m = 16 that is 288 columns instead of 512 (the modes
// with kx = -m/2 or ky = -m/2 have no kept partner). Every product and every sum that is left is the
// one that was computed before, in the same order.
//
// What bounds these kernels is the chain of one tile's 256 MMAs (K = 4096 pixels, 16 per instruction;
// each about 50 clocks up to N = 96, N / 2 clocks above): K is never split, so that the order of each
// sum is the same for every batch size. The tile width BN is chosen per batch size (dft_tile): wide
// when the row tiles alone nearly fill the machine, narrow when few samples would leave SMs idle. Both
// role loops run warp-converged (ptx::elect_one), and narrow tiles put two K blocks in a stage, so
// that the waits and commits do not add to the chain.
//   warp 0          TMA producer (full / empty mbarriers per stage)
//   warp 1          tcgen05.mma issuer (M = 128, N = BN, K = 16)
//   warps 2-13      epilogue: 16 columns (8 modes) at a time, three warps per 32-lane quadrant
// The forward form keeps two accumulators, so one tile's epilogue runs under the next tile's MMAs. The
// fused form (DW) also loads, on its first two column tiles and for one half of K each, the same 128
// rows of V beside dZ and accumulates dZ V^T (N = 128) in TMEM columns 256-383; the diagonal 32 x 32
// blocks are the four samples' dW partials, so dZ is read once.
// Every wait is bounded by a %globaltimer deadline; on timeout the CTA sets the error word, lets issued
// copies and MMAs land, frees its tensor memory and exits.
#include <algorithm>

#include "fno_internal.cuh"
#include "scw_ptx.cuh"

namespace scw {
namespace fno {

constexpr int kDftEpiWarps = 12;
constexpr int kDftThreads = 32 * (2 + kDftEpiWarps);

template <int BN, bool DW>
struct DftCfg {
  static constexpr int KS = BN <= 48 && !DW ? 2 : 1;  // K blocks per stage
  static constexpr uint32_t A_BYTES = 128u * 128u, B_BYTES = (uint32_t)BN * 128u;
  static constexpr uint32_t BLOCK = A_BYTES + B_BYTES;  // A, then B, per K block
  static constexpr uint32_t STAGE = KS * BLOCK + (DW ? A_BYTES : 0u);
  static constexpr int ST_RAW = (int)(212u * 1024u / STAGE);
  static constexpr int STAGES = ST_RAW > 10 ? 10 : ST_RAW;
  static constexpr uint32_t SMEM = STAGES * STAGE + 1024u;
  static constexpr uint32_t ACC = BN <= 32 ? 32u : (BN <= 64 ? 64u : (BN <= 128 ? 128u : 256u));
  static constexpr uint32_t DW_COL = 256u;
  static constexpr uint32_t TMEM = DW ? 512u : 2u * ACC;
};

template <int BN, bool DW>
__global__ void __launch_bounds__(kDftThreads, 1) dft_modes_kernel(const __grid_constant__ CUtensorMap mA,
                                                                  const __grid_constant__ CUtensorMap mB,
                                                                  const __grid_constant__ CUtensorMap mV,
                                                                  const __grid_constant__ EpiArgs ea,
                                                                  const __grid_constant__ EpiArgs ew, int K,
                                                                  int m_tiles, int n_tiles, int* err,
                                                                  uint64_t timeout_ns) {
  using Cfg = DftCfg<BN, DW>;
  constexpr int STAGES = Cfg::STAGES, NACC = DW ? 1 : 2;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES];
  __shared__ __align__(8) uint64_t empty_bar[STAGES];
  __shared__ __align__(8) uint64_t accf_bar[NACC];
  __shared__ __align__(8) uint64_t acce_bar[NACC];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_s;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tasks = m_tiles * n_tiles;
  const int nkb = K / 64, half = nkb / 2;  // K blocks; the dW half of column tile n < 2: [n half, (n + 1) half)
  const uint64_t deadline = ptx::globaltimer() + timeout_ns;
  // column tiles fastest: the tiles of a row tile run side by side and share its rows in L2
  auto tile_m0 = [&](int t) { return (t / n_tiles) * 128; };
  auto tile_n = [&](int t) { return t % n_tiles; };

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) {
      ptx::mbar_init(ptx::smem_u32(&full_bar[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&empty_bar[i]), 1);
    }
    for (int i = 0; i < NACC; ++i) {
      ptx::mbar_init(ptx::smem_u32(&accf_bar[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&acce_bar[i]), kDftEpiWarps);  // one arrival per epilogue warp
    }
    ptx::mbar_init(ptx::smem_u32(&drain_bar), 1);
    abort_s = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tensormap(&mA);
    ptx::prefetch_tensormap(&mB);
    if (DW) ptx::prefetch_tensormap(&mV);
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(&tmem_base_s), Cfg::TMEM);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = tmem_base_s;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const uint32_t leader = ptx::elect_one();
    pdl_sync();  // every result is stored behind loads issued after this
    int st = 0, issued = 0;
    uint32_t ph = 0;
    for (int t = blockIdx.x; t < n_tasks && !ptx::warp_any(abort_s); t += gridDim.x) {
      const int m0 = tile_m0(t), n = tile_n(t);
      for (int i = 0; i < nkb && !ptx::warp_any(abort_s); i += Cfg::KS) {
        if (!ptx::mbar_wait_warp(ptx::smem_u32(&empty_bar[st]), ph ^ 1u, deadline)) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_EMPTY);
          abort_s = 1;
          break;
        }
        const bool dw = DW && n < 2 && i >= n * half && i < (n + 1) * half;
        const uint32_t fb = ptx::smem_u32(&full_bar[st]);
        const uint32_t sa = ptx::smem_u32(smem + (size_t)st * Cfg::STAGE);
        ptx::mbar_arrive_expect_tx(fb, Cfg::KS * Cfg::BLOCK + (dw ? Cfg::A_BYTES : 0u), leader);
#pragma unroll
        for (int h = 0; h < Cfg::KS; ++h) {
          ptx::tma_load_2d(sa + h * Cfg::BLOCK, &mA, (i + h) * 64, m0, fb, leader);
          ptx::tma_load_2d(sa + h * Cfg::BLOCK + Cfg::A_BYTES, &mB, (i + h) * 64, n * BN, fb, leader);
        }
        if (dw) ptx::tma_load_2d(sa + Cfg::BLOCK, &mV, i * 64, m0, fb, leader);
        ++issued;
        if (++st == STAGES) {
          st = 0;
          ph ^= 1u;
        }
      }
    }
    if (ptx::warp_any(abort_s)) {
      const uint64_t d2 = ptx::drain_deadline(timeout_ns);
      for (int back = 1; back <= STAGES && back <= issued; ++back) {
        const int i = issued - back;
        if (!ptx::mbar_wait_warp(ptx::smem_u32(&full_bar[i % STAGES]), (uint32_t)(i / STAGES) & 1u, d2)) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_DRAIN);
          break;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- tcgen05.mma issuer ----------------
    const uint32_t leader = ptx::elect_one();
    constexpr uint32_t idesc = ptx::idesc_f16(true, 128, BN);
    constexpr uint32_t idesc_dw = ptx::idesc_f16(true, 128, 128);
    int st = 0, lt = 0;
    uint32_t ph = 0;
    for (int t = blockIdx.x; t < n_tasks && !ptx::warp_any(abort_s); t += gridDim.x, ++lt) {
      const int n = tile_n(t);
      const int acc = lt % NACC;
      // the epilogue has read the accumulator's previous tile
      if (!ptx::mbar_wait_warp(ptx::smem_u32(&acce_bar[acc]), ((uint32_t)(lt / NACC) & 1u) ^ 1u, deadline)) {
        if (leader) atomicOr(err, DEV_ERR_TIMEOUT_ACCUM);
        abort_s = 1;
        break;
      }
      ptx::tc_fence_after();
      const uint32_t d_tmem = tmem + (uint32_t)acc * Cfg::ACC;
      for (int i = 0; i < nkb; i += Cfg::KS) {
        if (!ptx::mbar_wait_warp(ptx::smem_u32(&full_bar[st]), ph, deadline)) {
          if (leader) atomicOr(err, DEV_ERR_TIMEOUT_FULL);
          abort_s = 1;
          break;
        }
        ptx::tc_fence_after();
        const uint32_t sa = ptx::smem_u32(smem + (size_t)st * Cfg::STAGE);
#pragma unroll
        for (int h = 0; h < Cfg::KS; ++h) {
          const uint64_t da = ptx::sw128_desc(sa + h * Cfg::BLOCK);
          const uint64_t db = ptx::sw128_desc(sa + h * Cfg::BLOCK + Cfg::A_BYTES);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)  // 16 elements = 32 bytes, in 16-byte units
            ptx::mma_f16(d_tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                         (i > 0 || h > 0 || kk > 0) ? 1u : 0u, leader);
        }
        const int j = i - n * half;  // position in this tile's dW half of K
        if (DW && n < 2 && j >= 0 && j < half) {
          const uint64_t da = ptx::sw128_desc(sa), dv = ptx::sw128_desc(sa + Cfg::BLOCK);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            ptx::mma_f16(tmem + Cfg::DW_COL, da + (uint64_t)(2 * kk), dv + (uint64_t)(2 * kk), idesc_dw,
                         (j > 0 || kk > 0) ? 1u : 0u, leader);
        }
        ptx::mma_commit(ptx::smem_u32(&empty_bar[st]), leader);
        if (++st == STAGES) {
          st = 0;
          ph ^= 1u;
        }
      }
      if (ptx::warp_any(abort_s)) break;
      ptx::mma_commit(ptx::smem_u32(&accf_bar[acc]), leader);
    }
    if (ptx::warp_any(abort_s)) {
      ptx::mma_commit(ptx::smem_u32(&drain_bar), leader);
      if (!ptx::mbar_wait_warp(ptx::smem_u32(&drain_bar), 0u, ptx::drain_deadline(timeout_ns)) && leader)
        atomicOr(err, DEV_ERR_TIMEOUT_DRAIN);
    }
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int grp = warp & 3;           // TMEM lanes 32 grp .. 32 grp + 31
    const int third = (warp - 2) >> 2;  // column chunks third, third + 3, ...; third 0 also takes dW
    int lt = 0;
    for (int t = blockIdx.x; t < n_tasks; t += gridDim.x, ++lt) {
      const int m0 = tile_m0(t), n = tile_n(t);
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
      const int row = m0 + grp * 32 + lane;
      const uint32_t lane_addr = tmem + ((uint32_t)(grp * 32) << 16);
#pragma unroll 1
      for (int c = third; c < BN / 16; c += 3) {
        const int j0 = (n * BN + 16 * c) / 2;  // the chunk's first independent mode
        if (2 * j0 >= ea.cols) break;          // warp-uniform
        uint32_t r[2][8];
        ptx::tmem_ld_x8(lane_addr + (uint32_t)acc * Cfg::ACC + (uint32_t)(16 * c), r[0]);
        ptx::tmem_ld_x8(lane_addr + (uint32_t)acc * Cfg::ACC + (uint32_t)(16 * c + 8), r[1]);
        ptx::tmem_wait_ld();
        if (row < ea.rows) {
          float2* o = reinterpret_cast<float2*>(ea.out) + row;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (2 * (j0 + j) < ea.cols) {
              const int2 md = __ldg(ea.modes + j0 + j);
              const float2 v = make_float2(ea.alpha * __uint_as_float(r[j >> 2][2 * (j & 3)]),
                                           ea.alpha * __uint_as_float(r[j >> 2][2 * (j & 3) + 1]));
              o[(size_t)md.x * ea.ld] = v;
              if (md.y >= 0) o[(size_t)md.y * ea.ld] = make_float2(v.x, -v.y);
            }
          }
        }
      }
      if (DW && third == 0 && n < 2) {  // the diagonal block of this quadrant's sample: dW_b partial, K half n
        float a[32];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t r[8];
          ptx::tmem_ld_x8(lane_addr + Cfg::DW_COL + (uint32_t)(32 * grp + 8 * q), r);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e) a[8 * q + e] = __uint_as_float(r[e]);
        }
        epilogue<EPI_DW, __nv_bfloat16, true>(ew, nullptr, nullptr, row, 32 * grp, n, a);
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
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, Cfg::TMEM);
  }
}

// ---------------------------------------------------------------- host side ---
int dft_independent_modes(int m, std::vector<int2>& modes) {
  modes.clear();
  const int h = m / 2;
  for (int ky = -h; ky < h; ++ky)
    for (int kx = -h; kx < h; ++kx) {
      const int k = (ky + h) * m + kx + h;
      const bool paired = ky > -h && kx > -h && (ky != 0 || kx != 0);
      const int mirror = paired ? (h - ky) * m + h - kx : -1;
      if (paired && mirror < k) continue;  // stored by its partner
      modes.push_back(make_int2(k, mirror));
    }
  return (int)modes.size();
}

// Index into kDftTiles of the tile width for M = rows and N = table rows: the one with the shortest MMA
// chain per SM, ceil(tiles / SMs) waves of max(200, 2 BN) clocks per K block, the narrowest among equals.
// m = 16 (288 columns), us per launch, profiled with cold caches, 512 columns in tiles of 256 -> now:
// 5 samples 28.4 -> 12.3 (BN = 16), 256 samples 29.4 -> 22.3 (BN = 144), with dW 39.2 -> 33.2.
int dft_tile(int M, int N, int sms) {
  const int m_tiles = (M + 127) / 128;
  int best = 0;
  long long best_cost = 0;
  for (int i = 0; i < kDftTileCount; ++i) {
    const int bn = kDftTiles[i];
    const long long tiles = (long long)m_tiles * ((N + bn - 1) / bn);
    const long long cost = ((tiles + sms - 1) / sms) * std::max(200, 2 * bn);
    if (i > 0 && N <= bn) continue;  // at least two column tiles (the fused form splits dW over them)
    if (i == 0 || cost < best_cost) {
      best = i;
      best_cost = cost;
    }
  }
  return best;
}

template <int BN, bool DW>
static cudaError_t launch_dft_t(const CUtensorMap& mA, const CUtensorMap& mB, const CUtensorMap& mV,
                                const EpiArgs& ea, const EpiArgs& ew, int M, int N, int K, int sms, int* err,
                                uint64_t timeout_ns, cudaStream_t st) {
  using Cfg = DftCfg<BN, DW>;
  cudaError_t e = allow_max_smem(reinterpret_cast<const void*>(dft_modes_kernel<BN, DW>));
  if (e != cudaSuccess) return e;
  const int m_tiles = (M + 127) / 128, n_tiles = (N + BN - 1) / BN;
  const int grid = std::max(1, std::min(m_tiles * n_tiles, sms));
  return launch_pdl(dft_modes_kernel<BN, DW>, dim3(grid), dim3(kDftThreads), Cfg::SMEM, st, mA, mB, mV, ea, ew, K,
                    m_tiles, n_tiles, err, timeout_ns);
}

cudaError_t launch_dft_tc(const CUtensorMap& mA, const CUtensorMap* mB, const CUtensorMap* mV, const EpiArgs& ea,
                          const EpiArgs* ew, int M, int N, int K, int* err, uint64_t timeout_ns, cudaStream_t st) {
  if (K % 128 != 0 || ea.modes == nullptr || (ew != nullptr && ew->splits != 2)) return cudaErrorInvalidValue;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int i = dft_tile(M, N, sms);
#define SCW_DFT(BN)                                                                                              \
  (ew ? launch_dft_t<BN, true>(mA, mB[i], *mV, ea, *ew, M, N, K, sms, err, timeout_ns, st)                       \
      : launch_dft_t<BN, false>(mA, mB[i], mB[i], ea, ea, M, N, K, sms, err, timeout_ns, st))
  switch (kDftTiles[i]) {
    case 16: return SCW_DFT(16);
    case 32: return SCW_DFT(32);
    case 48: return SCW_DFT(48);
    case 96: return SCW_DFT(96);
    case 144: return SCW_DFT(144);
    default: return cudaErrorInvalidValue;
  }
#undef SCW_DFT
}

}  // namespace fno
}  // namespace scw
