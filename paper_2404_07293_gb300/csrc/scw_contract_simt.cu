// Step (b), plain FP32 path: S_l = W_l C_l as a SIMT complex GEMM
// (Eq. 34 with the per-layer precompute of Sec. 4.1).
//
// W is consumed transposed (Wt[l][j][r], rows r contiguous, made once by
// scw_plan_set_layers) so that a warp's 32 lanes load 32 consecutive rows of
// one mode j in a single coalesced request, while that mode's weights
// C[j][f0..f0+FCH) are a shared-memory broadcast. Each thread accumulates two
// rows x FCH planes in registers; the 4M modes are split across CTAs and the
// partial spectra are summed by the recompose step.
#include <algorithm>

#include "scw_internal.cuh"
#include "scw_ptx.cuh"

namespace scw {

// The product is bound by streaming W^T (FCH complex MACs per 8-byte element): each thread keeps the next
// kBatch modes' elements of both its rows in flight while it multiplies the current ones. With four modes
// loaded just before their use, 16 layers of 15 x 15 orders took 51 us (78 MB: 1.5 TB/s), 35 us more of the step than now. For many planes
// it is bound by instruction issue instead, so the planes are multiplied in pairs with the packed FP32x2
// instructions: C sits in shared memory as (Re, Re', Im, Im') of two planes. Each sum keeps the
// order of its terms: Im then Re part of mode after mode.
constexpr int kBatch = 8;

template <int FCH>
__global__ void __launch_bounds__(128, FCH == 8 ? 4 : 3)
    contract_fp32_kernel(const float2* __restrict__ Wt, const float2* __restrict__ C, const LayerUnit* __restrict__ units,
                         int n_rblk, int ksplit, int M, int F_pad, int Fz, float2* __restrict__ S_part,
                         unsigned long long* trace, const __grid_constant__ ItemDev chk) {
  extern __shared__ float4 cs4[];  // [k][FCH / 2]
  ptx::griddep_launch_dependents();
  const int split = blockIdx.x % ksplit;
  const int rest = blockIdx.x / ksplit;
  const int rblk = rest % n_rblk;
  const int ui = rest / n_rblk;
  const LayerUnit u = units[ui];
  const int fc0 = blockIdx.y * FCH;
  const int K = 4 * M, rows = 3 * M;
  const int per = (K + ksplit - 1) / ksplit;
  const int kb = min(K, split * per);
  const int ke = min(K, kb + per);
  const int kc = ke - kb;
  const bool active = fc0 < u.nf;

  const int r0 = rblk * 256 + threadIdx.x;
  const int r1 = r0 + 128;
  // W^T rows (layer, mode) and columns r: the loop's largest index, checked once (indices grow with k)
  const bool wt_ok = kc == 0 || in_bounds(chk, BND_WT, ((size_t)u.layer * K + kb + kc - 1) * rows + min(r1, rows - 1));
  const bool v0 = r0 < rows && wt_ok && active, v1 = r1 < rows && wt_ok && active;
  const float2* w = Wt + ((size_t)u.layer * K + kb) * rows + r0;
  float2 w0[2][kBatch], w1[2][kBatch];
  auto load = [&](int buf, int k0) {
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const bool in = k0 + q < kc;
      w0[buf][q] = (in && v0) ? __ldg(w + (size_t)(k0 + q) * rows) : make_float2(0.f, 0.f);
      w1[buf][q] = (in && v1) ? __ldg(w + (size_t)(k0 + q) * rows + 128) : make_float2(0.f, 0.f);
    }
  };
  load(0, 0);             // W^T does not depend on the phase kernel that precedes this grid
  ptx::griddep_wait();    // the mode weights C do
  trace_begin(trace, TRACE_CONTRACT);
  if (!active) return;
  // (modes up to the next multiple of kBatch stay zero)
  const int kpad = (kc + kBatch - 1) / kBatch * kBatch;
  for (int i = threadIdx.x; i < kpad * (FCH / 2); i += blockDim.x) {
    const int k = i / (FCH / 2), f = 2 * (i - k * (FCH / 2));
    const size_t ci = ((size_t)ui * K + kb + k) * F_pad + fc0 + f;
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < kc && fc0 + f < F_pad && in_bounds(chk, BND_C, ci + 1)) c = *reinterpret_cast<const float4*>(C + ci);
    cs4[i] = make_float4(c.x, c.z, c.y, c.w);
  }
  __syncthreads();

  // accumulators of plane pairs: row 0 and row 1, real and imaginary parts
  float2 re0[FCH / 2], im0[FCH / 2], re1[FCH / 2], im1[FCH / 2];
#pragma unroll
  for (int q = 0; q < FCH / 2; ++q) re0[q] = im0[q] = re1[q] = im1[q] = make_float2(0.f, 0.f);
  auto mac = [&](int buf, int k0) {
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const float4* c = cs4 + (size_t)(k0 + q) * (FCH / 2);
      const float2 a = w0[buf][q], b = w1[buf][q];
      const float2 ax = make_float2(a.x, a.x), ay = make_float2(a.y, a.y), an = make_float2(-a.y, -a.y);
      const float2 bx = make_float2(b.x, b.x), by = make_float2(b.y, b.y), bn = make_float2(-b.y, -b.y);
#pragma unroll
      for (int h = 0; h < FCH / 2; ++h) {
        const float4 cc = c[h];
        const float2 cr = make_float2(cc.x, cc.y), ci = make_float2(cc.z, cc.w);
        re0[h] = __ffma2_rn(ax, cr, __ffma2_rn(an, ci, re0[h]));
        im0[h] = __ffma2_rn(ax, ci, __ffma2_rn(ay, cr, im0[h]));
        re1[h] = __ffma2_rn(bx, cr, __ffma2_rn(bn, ci, re1[h]));
        im1[h] = __ffma2_rn(bx, ci, __ffma2_rn(by, cr, im1[h]));
      }
    }
  };
#pragma unroll 1
  for (int k0 = 0; k0 < kpad; k0 += 2 * kBatch) {
    load(1, k0 + kBatch);
    mac(0, k0);
    if (k0 + kBatch >= kpad) break;
    load(0, k0 + 2 * kBatch);
    mac(1, k0 + kBatch);
  }

  const size_t d0 = ((size_t)split * Fz + u.f0 + fc0) * rows;
  float2* dst = S_part + d0;
#pragma unroll
  for (int f = 0; f < FCH; ++f) {
    if (fc0 + f < u.nf) {
      const int h = f >> 1;
      const float2 a = (f & 1) ? make_float2(re0[h].y, im0[h].y) : make_float2(re0[h].x, im0[h].x);
      const float2 b = (f & 1) ? make_float2(re1[h].y, im1[h].y) : make_float2(re1[h].x, im1[h].x);
      if (v0 && in_bounds(chk, BND_S_PART, d0 + (size_t)f * rows + r0)) dst[(size_t)f * rows + r0] = a;
      if (v1 && in_bounds(chk, BND_S_PART, d0 + (size_t)f * rows + r1)) dst[(size_t)f * rows + r1] = b;
    }
  }
  trace_end(trace, TRACE_CONTRACT);
}

// Modes in which W^T is split over CTAs: the split with the shortest schedule, rounds of resident CTAs (four
// per SM up to 8 planes, three above) of K / ks modes each plus about 24 modes' worth of start and end. At
// most kMaxChain modes are summed in one FP32 chain: longer ones saved 5 us of 213 at 21 x 21 orders and
// 32 layers, but raised the field's error against 64 bits from 4.4e-7 to 6.7e-7. The partial spectra grow with the
// splits: 64 x 64 orders, 2 layers of 16 planes take 64 (201 MB beside 6.4 GB of W and W^T) where chains of 768 modes
// took 22; writing and adding them is part of that step's 1046 us (2795 with the chains and without loads in flight).
constexpr int kMaxChain = 256;

int fp32_split(int n_units, int M, int F_pad, int sms) {
  const int K = 4 * M, fch = F_pad >= 16 ? 16 : 8;
  const long long tiles = (long long)n_units * ((3 * M + 255) / 256) * ((F_pad + fch - 1) / fch);
  const long long slots = (long long)sms * (fch == 8 ? 4 : 3);
  int best = 1;
  long long best_cost = 0;
  for (int ks = 1; ks <= std::max(1, std::min(64, K / 32)); ++ks) {
    const int per = (K + ks - 1) / ks;
    if (per > kMaxChain && ks < std::min(64, K / 32)) continue;
    if ((size_t)(per + kBatch) * fch * sizeof(float2) > 48 * 1024) continue;  // the slice of C in shared memory
    const long long cost = ((tiles * ks + slots - 1) / slots) * (per + 24);
    if (best_cost == 0 || cost < best_cost) {
      best = ks;
      best_cost = cost;
    }
  }
  return best;
}

cudaError_t launch_contract_fp32(const Plan& p, cudaStream_t st) {
  if (p.units.empty()) return cudaSuccess;
  const int n_rblk = (3 * p.M + 255) / 256;
  const int K = 4 * p.M;
  const int per = (K + p.k_split - 1) / p.k_split;
  const bool wide = p.F_pad >= 16;
  const int FCH = wide ? 16 : 8;
  dim3 grid((unsigned)(p.units.size() * n_rblk * p.k_split), (unsigned)((p.F_pad + FCH - 1) / FCH));
  const size_t smem = (size_t)(per + kBatch - 1) / kBatch * kBatch * FCH * sizeof(float2);
  cudaError_t e;
  if (wide) {
    e = allow_max_smem(reinterpret_cast<const void*>(contract_fp32_kernel<16>));
    if (e != cudaSuccess) return e;
    e = launch_pdl(contract_fp32_kernel<16>, grid, dim3(128), smem, st, (const float2*)p.Wt,
                   (const float2*)p.Cf, (const LayerUnit*)p.d_units, n_rblk, p.k_split, p.M, p.F_pad, p.Fz, p.S_part,
                   p.item.trace, p.item);
    if (e != cudaSuccess) return e;
  } else {
    e = allow_max_smem(reinterpret_cast<const void*>(contract_fp32_kernel<8>));
    if (e != cudaSuccess) return e;
    e = launch_pdl(contract_fp32_kernel<8>, grid, dim3(128), smem, st, (const float2*)p.Wt,
                   (const float2*)p.Cf, (const LayerUnit*)p.d_units, n_rblk, p.k_split, p.M, p.F_pad, p.Fz, p.S_part,
                   p.item.trace, p.item);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace scw
