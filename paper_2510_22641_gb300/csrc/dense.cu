// Launchers of the dense projections (ssd_dense_kernel) and of the operand split.
#include <atomic>
#include <initializer_list>

#include "dense.cuh"

namespace ssd {

// ------------------------------------------------------------------ operand parts from fp32 rows

// Row r of hi / lo (bf16 [rows][K]) = the parts of x[r] * gain (gain null: x[r]); rs[r] =
// 1/sqrt(mean(x[r]^2) + eps) with gain, 1 without.  For rows that no dense projection produced.
__global__ void __launch_bounds__(256) ssd_split_act_kernel(const float* __restrict__ x, int x_stride, int K,
                                                            const __nv_bfloat16* __restrict__ gain, float eps,
                                                            __nv_bfloat16* __restrict__ hi,
                                                            __nv_bfloat16* __restrict__ lo, float* __restrict__ rs) {
  __shared__ float red[8];
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.x, t = threadIdx.x, lane = t & 31;
  const float4* xr = reinterpret_cast<const float4*>(x + static_cast<size_t>(r) * x_stride);
  uint4* hr = reinterpret_cast<uint4*>(hi + static_cast<size_t>(r) * K);
  uint4* lr = reinterpret_cast<uint4*>(lo + static_cast<size_t>(r) * K);
  float ss = 0.f;
  for (int i = t; i < (K >> 3); i += 256) {
    const float4 a0 = __ldcg(xr + 2 * i), a1 = __ldcg(xr + 2 * i + 1);
    float v[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) ss = fmaf(v[e], v[e], ss);
    if (gain) {
      const uint4 gv = __ldg(reinterpret_cast<const uint4*>(gain) + i);
      const float2 g0 = bf16x2_to_float2(gv.x), g1 = bf16x2_to_float2(gv.y), g2 = bf16x2_to_float2(gv.z),
                   g3 = bf16x2_to_float2(gv.w);
      v[0] *= g0.x; v[1] *= g0.y; v[2] *= g1.x; v[3] *= g1.y;
      v[4] *= g2.x; v[5] *= g2.y; v[6] *= g3.x; v[7] *= g3.y;
    }
    uint32_t hw[4], lw[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * e]), h1 = __float2bfloat16_rn(v[2 * e + 1]);
      hw[e] = pack_bf16x2(h0, h1);
      lw[e] = pack_bf16x2(__float2bfloat16_rn(v[2 * e] - __bfloat162float(h0)),
                          __float2bfloat16_rn(v[2 * e + 1] - __bfloat162float(h1)));
    }
    hr[i] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    lr[i] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
  if (lane == 0) red[t >> 5] = ss;
  __syncthreads();
  if (t == 0) {
    float s = 0.f;
    for (int w = 0; w < 8; ++w) s += red[w];
    rs[r] = gain ? rsqrtf(s / static_cast<float>(K) + eps) : 1.0f;
  }
}

namespace {

std::atomic<int> g_max_clusters[kDnMaxSplit + 1] = {};  // clusters of 2 * split CTAs that run at once

template <Epi EPI>
cudaError_t launch_e(const CUtensorMap* w, const CUtensorMap* b, const DenseParams& p, int clusters, int smem,
                     cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * 2 * p.split);
  cfg.blockDim = dim3(kDnThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2 * p.split;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, p.apart ? ssd_dense_kernel<EPI, true> : ssd_dense_kernel<EPI, false>, w[0], w[1], w[2],
                            b[0], b[1], p);
}

template <Epi EPI>
cudaError_t attr_e() {
  for (auto* k : {ssd_dense_kernel<EPI, false>, ssd_dense_kernel<EPI, true>})
    if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, DnSmem::kMax)) return e;
  return cudaSuccess;
}

}  // namespace

// How a launch of M rows over n_rt weight tiles and `steps` K steps is cut up (dense.cuh): tokens per tile and
// CTA pairs per tile.  The cost that it compares, in clocks (measured, 1.92 GHz):
//  * a K step of nt tokens takes 4 nt clocks of MMA (hi and lo parts) and at least 350 (its loads: 0.18 us
//    at 64 tokens, 0.21 at 96, 0.27 at 128, 0.34 at 160, 0.47 at 224);
//  * a wave of tiles costs about 1000 on top (accumulator hand-over), and the last one's epilogue, which
//    nothing hides, about 75 per token (6.4 us at 160);
//  * sharing a tile's K steps among `split` pairs (only when every tile has a cluster of its own) costs two
//    exchanges through distributed shared memory, about 3000, and divides K steps and epilogue: 4096 x
//    11008 at 77 rows takes 24 us with split 3, 78 us without.
// max_split = 1 keeps a tile's K steps together at every M: then a row's sums do not depend on M (the tokens per
// tile change which MMA column a row takes, not the order of its products).
void dense_plan(int M, int n_rt, int steps, int pairs, int max_split, int* nt_out, int* split_out) {
  const int n_rp = (n_rt + 1) / 2;
  long long best = -1;
  for (int t = (M + kDnMaxTok - 1) / kDnMaxTok; t <= (M + 31) / 32; ++t) {
    const int nt = ((M + t - 1) / t + 31) / 32 * 32;
    const int tiles = n_rp * ((M + nt - 1) / nt);
    const long long step = 4 * nt + 16 > 350 ? 4 * nt + 16 : 350;
    for (int split = 1; split <= max_split && split <= steps; ++split) {
      if (split > 1 && tiles > g_max_clusters[split].load()) break;
      const long long waves = split > 1 ? 1 : (tiles + pairs - 1) / pairs;
      const long long cost = waves * ((steps + split - 1) / split * step + 1000) + 75ll * nt / split + (split > 1 ? 3000 : 0);
      if (best < 0 || cost < best) {
        best = cost;
        *nt_out = nt;
        *split_out = split;
      }
    }
  }
}

// p.apart (a batched verification's rows, at most kMaxMidRows, so nt <= 128 and two accumulators of 2 nt columns fit
// TMEM): hi and lo products accumulate apart, as in the GEMV: one accumulator for both is cut off to its own last
// bit twice per 16 columns instead of once.  13B verification, logits against 64 bits: 2.67e-5 with one
// accumulator, 2.49e-5 with two, in the same time (27.2 ms for 16 requests' 24 tokens either way).
// w: the site's weight maps; b: hi / lo maps of the rows' parts with p.nt / 2-row boxes (p.nt and p.split
// from dense_plan).  Fills in the tile counts.
cudaError_t dense_launch(Epi e, const CUtensorMap* w, const CUtensorMap* b, DenseParams p, int num_sms,
                         cudaStream_t s, bool pdl) {
  if (p.M < 1 || p.nt < 32 || p.nt > kDnMaxTok || p.nt % 32 || p.K % kTileK || p.n_rt < 1 || p.split < 1 ||
      p.split > kDnMaxSplit || p.split * kTileK > p.K || (e == Epi::ARGMAX && p.M > kMaxMidRows) ||
      (p.apart && 2 * p.nt > kDnMaxTok))
    return cudaErrorInvalidValue;
  p.tok_tiles = (p.M + p.nt - 1) / p.nt;
  p.stages = dense_stages(p.nt);
  const int ring = p.stages * (static_cast<int>(kWTileBytes) + p.nt * 128);
  if (dense_land_bytes(p.nt, p.split) > ring) return cudaErrorInvalidValue;
  const int tiles = (p.n_rt + 1) / 2 * p.tok_tiles, pairs = num_sms / 2;
  const int clusters = p.split > 1 || tiles < pairs ? tiles : pairs;
  const int smem = 1024 + DnSmem::kRing + ring;
  switch (e) {
    case Epi::QKV: return launch_e<Epi::QKV>(w, b, p, clusters, smem, s, pdl);
    case Epi::GATE_SILU: return launch_e<Epi::GATE_SILU>(w, b, p, clusters, smem, s, pdl);
    case Epi::RESID: return launch_e<Epi::RESID>(w, b, p, clusters, smem, s, pdl);
    case Epi::ARGMAX: return launch_e<Epi::ARGMAX>(w, b, p, clusters, smem, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t dense_attrs() {
  cudaError_t e;
  if ((e = attr_e<Epi::QKV>()) || (e = attr_e<Epi::GATE_SILU>()) || (e = attr_e<Epi::RESID>()) ||
      (e = attr_e<Epi::ARGMAX>()))
    return e;
  for (int split = 2; split <= kDnMaxSplit; ++split) {  // the same on every device of this kind
    if (g_max_clusters[split].load() > 0) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * split);
    cfg.blockDim = dim3(kDnThreads);
    cfg.dynamicSmemBytes = DnSmem::kMax;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2 * split;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&n, ssd_dense_kernel<Epi::RESID, false>, &cfg))) return e;
    g_max_clusters[split].store(n);
  }
  return cudaSuccess;
}

cudaError_t split_act_launch(const float* x, int x_stride, int K, const __nv_bfloat16* gain, float eps,
                             __nv_bfloat16* hi, __nv_bfloat16* lo, float* rs, int rows, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(rows);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ssd_split_act_kernel, x, x_stride, K, gain, eps, hi, lo, rs);
}

}  // namespace ssd
