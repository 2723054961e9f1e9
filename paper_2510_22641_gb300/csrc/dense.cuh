// Dense projections on the 5th-generation tensor cores: every projection over more than 16 rows --
// the prefill of a prompt (decoder-only prompts, the encoder of the encoder-decoder model) and the
// verification rows of batched requests.
//
//   out[m][n] = rs[m] * sum_k W[n][k] * v[m][k],   v = x * gain, rs[m] = 1/rms(x[m]) (1 without a norm)
//
// The rows arrive as bf16 parts v = hi + lo (2^-17 relative), written by whichever kernel produced
// them; both parts meet the bf16 weights with fp32 accumulation in TMEM, so a row keeps fp32-class
// accuracy at bf16 tensor-core rate.
//
// What bounds it, and the shape that follows:
//  * The weights are the MMA's M side (128 rows per CTA, 256 per CTA pair, cta_group::2), the rows
//    ("tokens") its N side, a tile of NT = 32..256 tokens chosen per launch (dense_plan) so that the
//    last wave of tiles is nearly full: 640 tokens x 4096 outputs are 64 pair tiles of 160 tokens on
//    76 pairs, where 128 x 128 tiles left 8 of 160 tiles to a second wave.
//  * Per 64-column K step a CTA reads its own 16 KB of weights and half of the token tile's hi and lo
//    parts (NT * 128 bytes); the pair shares the other half, so shared memory serves about 112 bytes
//    per clock at NT = 256.  One CTA alone would need 160 of the 128 it has: measured, that form ran
//    at half of the tensor rate.
//  * The issuing warps run their loops as whole warps and elect a lane only around the TMA and MMA
//    instructions, so that descriptors and addresses stay in uniform registers: as single-lane loops they
//    took 0.41 us per K step at every tile up to 192 tokens, against 0.18 us at 64 and 0.27 us at 128
//    tokens now (0.27 us is the MMAs' own time at 128).
//  * A launch with few tiles splits each tile's K steps over up to 4 pairs of a cluster (dense_plan).
//  * Outputs lie with 32 consecutive output columns across a warp's lanes (TMEM lane = weight row),
//    so every store of the epilogue is a full line; rotation and gate/up partners, which sit in other
//    warps' lanes, are exchanged through shared memory.  (Token rows on the lanes cost 32 sectors per
//    store: 17 us per 128 x 128 tile.)
//  * The epilogue writes what the next kernel reads -- bf16 parts of q, K, V^T for the attention, of h
//    for the down projection, of x * gain with the rows' sums of squares for the next normed
//    projection -- so no launch only converts.
//  Roles: warp 0 loads the weights by TMA (from before the upstream wait on), warp 10 the tokens' parts,
//  warp 1 of the pair's first CTA issues the MMAs of both CTAs, each as a whole warp with one lane
//  elected; warps 2..9 drain the double-buffered accumulator in two groups of four (16 tokens at a
//  time, alternating) while the next tile runs.
#pragma once

#include "gemv.cuh"

namespace ssd {

constexpr int kDnThreads = 352;      // warp 0 weight TMA, warp 1 MMA + TMEM, warps 2..9 epilogue, warp 10 token TMA
constexpr int kDnEpiThreads = 256;
constexpr int kDnMaxTok = 256;       // tokens per tile (the MMA's N)
constexpr int kDnMaxStages = 8;
constexpr int kDnXsLd = 12;          // exchange rows of 8 floats, padded so that 16-byte accesses of 8 lanes hit all banks
constexpr int kDnChunk = 16;         // tokens per epilogue chunk
constexpr int kDnMaxSplit = 4;       // CTA pairs of one cluster (8 CTAs)
constexpr int kDnLandLd = 20;        // landing rows of 16 floats of another pair's chunk, padded the same way

struct DnSmem {
  static constexpr int kRs = 0;                                       // [2][kDnMaxTok] row scales (tile parity)
  static constexpr int kPos = kRs + 2 * kDnMaxTok * 4;                // [2][kDnMaxTok] positions
  static constexpr int kReq = kPos + 2 * kDnMaxTok * 4;               // [2][kDnMaxTok] requests
  static constexpr int kKvr = kReq + 2 * kDnMaxTok * 4;               // [2][kDnMaxTok] rows of the K / V^T parts
  static constexpr int kKey = kKvr + 2 * kDnMaxTok * 4;               // [2 groups][4 warps][16] argmax keys
  static constexpr int kFlag = kKey + 2 * 4 * kDnChunk * 8;           // [2] last-tile flags
  static constexpr int kBar = (kFlag + 8 + 7) & ~7;                   // full, empty [stages]; tfull, tempty [2]
  static constexpr int kTmemSlot = kBar + (2 * kDnMaxStages + 4) * 8;
  static constexpr int kXs = (kTmemSlot + 16 + 127) & ~127;           // [2 groups][2][128][kDnXsLd] floats
  static constexpr int kRing = (kXs + 4 * kTileN * kDnXsLd * 4 + 1023) & ~1023;  // stages
  static constexpr int kMax = 232448;                                 // one CTA's limit
};
constexpr int kDnRing = (DnSmem::kMax - 1024 - DnSmem::kRing) / 1024 * 1024;  // most stage bytes
constexpr int dense_stages(int nt) {
  const int n = kDnRing / (static_cast<int>(kWTileBytes) + nt * 128);
  return n < kDnMaxStages ? n : kDnMaxStages;
}

// Landing bytes (over the ring) of one CTA for `split` pairs and nt tokens: a slot per chunk it owns and pair.
constexpr int dense_land_bytes(int nt, int split) {
  return split > 1 ? (nt / kDnChunk + split - 1) / split * split * kTileN * kDnLandLd * 4 : 0;
}

struct DenseParams {
  int M, N, K;              // rows (tokens), valid output columns (GATE_SILU: d_ff), reduction
  int n_rt;                 // 128-row weight tiles (GATE_SILU: 64 gate + 64 up rows each)
  int tok_tiles, nt;        // token tiles of nt tokens
  int split;                // CTA pairs that share one tile's reduction (the cluster holds `split` pairs)
  int stages;
  int whole;                // 1: a tile's K steps stay with one CTA pair, whatever M (dense_plan)
  int apart;                // 1: hi and lo products accumulate apart (nt <= 128)
  int seg_rows, seg_base;   // QKV: rows per source matrix, segment of the site's first matrix (0 q, 1 k, 2 v)
  float eps;
  DevState* st;             // error word, argmax keys; kv_len of one request
  // row scales: rs[m] = 1/sqrt(sum(ssq[m][0 .. ssq_n)) / K + eps), or rs_in[m], or 1
  const float* ssq;
  int ssq_n;                // a multiple of 4
  const float* rs_in;
  // positions: row m of one request sits at pos_off + m (+ st->kv_len unless abs_pos); with
  // batch_rows = R row m is request m / R, at req_st[b].kv_len + pos_off + m % R, cache slot b * req_kv
  // with row_map row m is {position, request, row in the K / V^T parts, -}; request < 0: padding, not stored
  int pos_off, abs_pos, batch_rows;
  const int4* row_map;
  const DevState* req_st;
  long long req_kv;
  // QKV
  float* q_out;             // fp32 q rows, or null
  int q_stride;
  float* k_cache;           // this layer's [H][max_seq][head_dim] (+ request slot), fp32
  float* v_cache;
  int head_dim, max_seq;
  const float2* rope_cs;    // [max_seq][head_dim/2] (cos, sin), or null: no rotation
  __nv_bfloat16 *qs_hi, *qs_lo;   // or null; prefill attention operands: q [row][qs_ld],
  int qs_ld;
  __nv_bfloat16 *ks_hi, *ks_lo;   // K [H][s_pad][head_dim],
  __nv_bfloat16 *vt_hi, *vt_lo;   // V transposed [H][head_dim][s_pad], at the row's position (or row_map's)
  int s_pad;
  int act;                  // GATE_SILU: 0 = SiLU(gate) * up, 1 = GELU_tanh(gate) * up
  // RESID: dst[m][n] = base[m][n] + (*scale) * out[m][n]
  const float* base;
  int base_stride;
  float* dst;
  int dst_stride;
  const float* scale;
  // the next projection's operand: parts of h (GATE_SILU) or of x * nx_gain (RESID), [row][nx_ld], and
  // RESID rows' sums of squares per 32 columns, nx_ssq[row][4 * n_rt] (null: not written)
  __nv_bfloat16 *nx_hi, *nx_lo;
  int nx_ld;
  const __nv_bfloat16* nx_gain;
  float* nx_ssq;
  int late_trigger;  // as GemvParams: dependents start only once the upstream grid has completed
  // ARGMAX (as GemvParams)
  int* tok_dst;
  int tok_stride;
  float* logits;
  int logits_rows, logits_step_rows;
};

// ------------------------------------------------------------------ cluster / pair PTX

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of `saddr` (a shared::cta address) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_cluster(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// TMA load into this CTA's shared memory that completes on a barrier of the pair (cluster address)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3}], [%4];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, float a, float b, float c, float d) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait with cluster-scope acquire: gives up after 2 s, or once a wait anywhere in the decode has
// given up (the error word), so that the launches after a timeout end at once.
__device__ __forceinline__ bool dense_wait(uint64_t* bar, uint32_t parity, const DevState* st) {
  const uint32_t a = smem_u32(bar);
  uint64_t t0 = 0;
  for (uint32_t i = 0;; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
        "p;\n}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if (i == 0) t0 = globaltimer_ns();
    if ((i & 255u) == 255u && (globaltimer_ns() - t0 > 2000000000ull || (__ldcg(&st->error) & DERR_TIMEOUT)))
      return false;
  }
}
// The same for a whole warp, with a warp-uniform result.
__device__ __forceinline__ bool dense_wait_warp(uint64_t* bar, uint32_t parity, const DevState* st) {
  return __all_sync(0xffffffffu, dense_wait(bar, parity, st));
}
__device__ __forceinline__ void umma_f16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Completion of the pair's MMAs issued so far, on the same barrier of both CTAs (`both`: their rank bits).
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar, uint16_t both) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"(both)
      : "memory");
}

// ------------------------------------------------------------------ epilogue helpers

// Sums of 16 values over a warp's lanes, each in a fixed tree: lanes 2i and 2i + 1 return value i's sum.
__device__ __forceinline__ float warp_sum16(const float (&v)[kDnChunk], int lane) {
  float a[8], b[4], c[2], d;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float keep = (lane & 16) ? v[i + 8] : v[i], send = (lane & 16) ? v[i] : v[i + 8];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float keep = (lane & 8) ? a[i + 4] : a[i], send = (lane & 8) ? a[i] : a[i + 4];
    b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float keep = (lane & 4) ? b[i + 2] : b[i], send = (lane & 4) ? b[i] : b[i + 2];
    c[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  {
    const float keep = (lane & 2) ? c[1] : c[0], send = (lane & 2) ? c[0] : c[1];
    d = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  return d + __shfl_xor_sync(0xffffffffu, d, 1);
}

__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}
// The same reduction with max over 64-bit keys.
__device__ __forceinline__ unsigned long long warp_max16(unsigned long long (&v)[kDnChunk], int lane) {
#pragma unroll
  for (int w = 8, bit = 16; w >= 1; w >>= 1, bit >>= 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i >= w) break;
      const unsigned long long keep = (lane & bit) ? v[i + w] : v[i], send = (lane & bit) ? v[i] : v[i + w];
      v[i] = max_u64(keep, __shfl_xor_sync(0xffffffffu, send, bit));
    }
  }
  return max_u64(v[0], __shfl_xor_sync(0xffffffffu, v[0], 1));
}

__device__ __forceinline__ void store_parts(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t i, float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  hi[i] = h;
  lo[i] = __float2bfloat16_rn(v - __bfloat162float(h));
}

// The parts of two consecutive rows' values v0, v1 of this lane's column, whole warp: lane pairs swap, so
// that the even lane stores both columns of the first row and the odd lane those of the second, 4 bytes
// each.  hi / lo: at the first row and the even lane's column; ld: the rows' distance (even).
__device__ __forceinline__ void store_parts2(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t ld, float v0, float v1,
                                             int lane) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
  const __nv_bfloat162 l = __floats2bfloat162_rn(v0 - __low2float(h), v1 - __high2float(h));
  const uint32_t hw = *reinterpret_cast<const uint32_t*>(&h), lw = *reinterpret_cast<const uint32_t*>(&l);
  const uint32_t ho = __shfl_xor_sync(0xffffffffu, hw, 1), lx = __shfl_xor_sync(0xffffffffu, lw, 1);
  const bool odd = lane & 1;
  const size_t o = odd ? ld : 0;
  *reinterpret_cast<uint32_t*>(hi + o) = odd ? __byte_perm(ho, hw, 0x7632) : __byte_perm(hw, ho, 0x5410);
  *reinterpret_cast<uint32_t*>(lo + o) = odd ? __byte_perm(lx, lw, 0x7632) : __byte_perm(lw, lx, 0x5410);
}

// Barrier among the 128 threads of epilogue group g.
__device__ __forceinline__ void group_sync(int g) { named_bar_sync(1 + g, 128); }

// Rows that pair up across the lanes of a weight tile -- a head's rotation pairs (j, j + head_dim/2) and a
// tile's gate and up rows -- share a chunk: the thread of the first row finishes tokens 0..7 of both, the
// thread of the second tokens 8..15, each sending the other its half through xs.  The caller alternates
// two xs buffers, so one barrier per chunk is enough.
__device__ __forceinline__ void exchange8(const float (&v)[kDnChunk], float (&w)[8], bool second, int partner,
                                          float* xs, int g, int row) {
  float4* mine = reinterpret_cast<float4*>(xs + row * kDnXsLd);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float4 a = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    const float4 b = make_float4(v[8 + 4 * i], v[9 + 4 * i], v[10 + 4 * i], v[11 + 4 * i]);
    mine[i] = second ? a : b;
  }
  group_sync(g);
  const float4* theirs = reinterpret_cast<const float4*>(xs + partner * kDnXsLd);
  const float4 t0 = theirs[0], t1 = theirs[1];
  w[0] = t0.x; w[1] = t0.y; w[2] = t0.z; w[3] = t0.w;
  w[4] = t1.x; w[5] = t1.y; w[6] = t1.z; w[7] = t1.w;
}

// The global inputs of one chunk's epilogue, fetched one chunk ahead (the first before the accumulator is
// complete): RESID the base rows' values, QKV the (cos, sin) of this thread's 8 tokens.
template <Epi EPI>
__device__ __forceinline__ void chunk_inputs(const DenseParams& p, int rt, int m0, int nv, const int* pos, int row,
                                             float (&in)[kDnChunk]) {
  if constexpr (EPI == Epi::RESID) {
    const int n = rt * kTileN + row;
#pragma unroll
    for (int i = 0; i < kDnChunk; ++i)
      in[i] = n < p.N && i < nv ? __ldcg(p.base + static_cast<size_t>(m0 + i) * p.base_stride + n) : 0.f;
  } else if constexpr (EPI == Epi::QKV) {
    const int seg = rt * kTileN / p.seg_rows, half = p.head_dim >> 1, j = row & (p.head_dim - 1);
    if (p.rope_cs && seg + p.seg_base < 2) {
      const int i0 = j < half ? 0 : 8, jj = j & (half - 1);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int ps = i0 + i < nv ? pos[i0 + i] : -1;
        const float2 cs = ps >= 0 && ps < p.max_seq ? __ldg(p.rope_cs + static_cast<size_t>(ps) * half + jj)
                                                    : make_float2(1.f, 0.f);
        in[2 * i] = cs.x;
        in[2 * i + 1] = cs.y;
      }
    }
  }
}

// One 16-token chunk of weight tile rt: v[i] is the raw product of this thread's weight row `row`
// (0..127 of the tile) and token m0 + i, of which the first nv are rows of the launch.  rs / pos / req
// are the chunk's scales, positions and requests, kvr its rows in the K / V^T parts, `in` its inputs
// (chunk_inputs), xs the exchange buffer.
// FULL: all 16 tokens, every column and position valid -- straight-line code whose stores overlap (one
// branch per token kept a chunk at 2 us) and operand parts stored 4 bytes at a time.
template <Epi EPI, bool FULL>
__device__ __forceinline__ void dense_chunk(const DenseParams& p, int rt, int m0, int nv, float (&v)[kDnChunk],
                                            const float (&in)[kDnChunk], const float* rs, const int* pos,
                                            const int* req, const int* kvr, float* xs, int g, int row,
                                            uint8_t* smem) {
  const int lane = row & 31;
  if constexpr (EPI == Epi::QKV) {
    const int r0 = rt * kTileN, seg = r0 / p.seg_rows, mat = seg + p.seg_base;
    const int Dh = p.head_dim, half = Dh >> 1;       // 64 or 128: a power of two
    const int n0 = r0 - seg * p.seg_rows, j = row & (Dh - 1), h = (n0 + row - j) / Dh;
#pragma unroll
    for (int i = 0; i < kDnChunk; ++i) v[i] *= rs[i];
    float* cache = mat == 1 ? p.k_cache : p.v_cache;
    // output column (h, jo) of token i in fp32: a q row, or a cache row
    auto put = [&](int i, int jo, float o) {
      if (!FULL && (pos[i] < 0 || pos[i] >= p.max_seq)) {
        set_error(p.st, DERR_POS);
        return;
      }
      if (mat == 0) {
        if (p.q_out) p.q_out[static_cast<size_t>(m0 + i) * p.q_stride + h * Dh + jo] = o;
        if (!FULL && p.qs_hi) store_parts(p.qs_hi, p.qs_lo, static_cast<size_t>(m0 + i) * p.qs_ld + h * Dh + jo, o);
      } else {
        cache[req[i] * p.req_kv + (static_cast<size_t>(h) * p.max_seq + pos[i]) * Dh + jo] = o;
        if (!FULL && mat == 1 && p.ks_hi)
          store_parts(p.ks_hi, p.ks_lo, (static_cast<size_t>(h) * p.s_pad + kvr[i]) * Dh + jo, o);
      }
    };
    // the same columns' operand parts of tokens i, i + 1 (q or K), consecutive rows of one request
    auto put_parts2 = [&](int i, int jo, float o0, float o1) {
      const int je = jo & ~1;
      if (mat == 0) {
        const size_t o = static_cast<size_t>(m0 + i) * p.qs_ld + h * Dh + je;
        if (p.qs_hi) store_parts2(p.qs_hi + o, p.qs_lo + o, p.qs_ld, o0, o1, lane);
      } else if (p.ks_hi) {
        const size_t o = (static_cast<size_t>(h) * p.s_pad + kvr[i]) * Dh + je;
        store_parts2(p.ks_hi + o, p.ks_lo + o, Dh, o0, o1, lane);
      }
    };
    if (mat < 2 && p.rope_cs) {
      const bool second = j >= half;
      const int i0 = second ? 8 : 0, jj = j & (half - 1);
      float w[8];
      exchange8(v, w, second, row ^ half, xs, g, row);
      float ra[8], rb[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float a = second ? w[i] : v[i], b = second ? v[8 + i] : w[i], c = in[2 * i], sn = in[2 * i + 1];
        ra[i] = a * c - b * sn;
        rb[i] = a * sn + b * c;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (!FULL && i0 + i >= nv) break;
        put(i0 + i, jj, ra[i]);
        put(i0 + i, jj + half, rb[i]);
      }
      if (FULL) {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
          put_parts2(i0 + i, jj, ra[i], ra[i + 1]);
          put_parts2(i0 + i, jj + half, rb[i], rb[i + 1]);
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < kDnChunk; ++i) {
        if (!FULL && i >= nv) break;
        put(i, j, v[i]);
      }
      if (mat < 2) {
        if (FULL) {
#pragma unroll
          for (int i = 0; i < kDnChunk; i += 2) put_parts2(i, j, v[i], v[i + 1]);
        }
      } else if (p.vt_hi && nv > 0 && pos[0] >= 0 && pos[0] + nv <= p.max_seq) {  // consecutive rows of one request
        const size_t o = (static_cast<size_t>(h) * Dh + j) * p.s_pad + kvr[0];
        if (nv == kDnChunk && (kvr[0] & 7) == 0) {
          uint32_t hw[8], lw[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * e]), h1 = __float2bfloat16_rn(v[2 * e + 1]);
            hw[e] = pack_bf16x2(h0, h1);
            lw[e] = pack_bf16x2(__float2bfloat16_rn(v[2 * e] - __bfloat162float(h0)),
                                __float2bfloat16_rn(v[2 * e + 1] - __bfloat162float(h1)));
          }
          uint4* dh = reinterpret_cast<uint4*>(p.vt_hi + o);
          uint4* dl = reinterpret_cast<uint4*>(p.vt_lo + o);
          dh[0] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
          dh[1] = make_uint4(hw[4], hw[5], hw[6], hw[7]);
          dl[0] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
          dl[1] = make_uint4(lw[4], lw[5], lw[6], lw[7]);
        } else {
#pragma unroll
          for (int i = 0; i < kDnChunk; ++i) {
            if (i >= nv) break;
            store_parts(p.vt_hi, p.vt_lo, o + i, v[i]);
          }
        }
      }
    }
  } else if constexpr (EPI == Epi::GATE_SILU) {  // rows 0..63 hold gate, 64..127 the same columns' up
    const bool up = row >= kHalfN;
    float w[8];
    exchange8(v, w, up, row ^ kHalfN, xs, g, row);
    const int n = rt * kHalfN + (row & (kHalfN - 1)), i0 = up ? 8 : 0;
    float hv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float s = FULL || i0 + i < nv ? rs[i0 + i] : 0.f;
      const float gt = (up ? w[i] : v[i]) * s, ut = (up ? v[8 + i] : w[i]) * s;
      hv[i] = (p.act ? gelu_tanh_f(gt) : silu_f(gt)) * ut;
    }
    if (FULL) {
      const size_t o = static_cast<size_t>(m0 + i0) * p.nx_ld + (n & ~1);
#pragma unroll
      for (int i = 0; i < 8; i += 2)
        store_parts2(p.nx_hi + o + static_cast<size_t>(i) * p.nx_ld, p.nx_lo + o + static_cast<size_t>(i) * p.nx_ld,
                     p.nx_ld, hv[i], hv[i + 1], lane);
    } else if (n < p.N) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (i0 + i >= nv) break;
        store_parts(p.nx_hi, p.nx_lo, static_cast<size_t>(m0 + i0 + i) * p.nx_ld + n, hv[i]);
      }
    }
  } else if constexpr (EPI == Epi::RESID) {
    const int n = rt * kTileN + row;
    const bool ok = FULL || n < p.N;
    const float s = __ldg(p.scale);
    const float gn = ok && p.nx_gain ? __bfloat162float(p.nx_gain[n]) : 1.0f;
    float* dst = p.dst + static_cast<size_t>(m0) * p.dst_stride + n;
#pragma unroll
    for (int i = 0; i < kDnChunk; ++i) {
      v[i] = FULL || (ok && i < nv) ? in[i] + s * (v[i] * rs[i]) : 0.f;
      if (FULL || (ok && i < nv)) dst[static_cast<size_t>(i) * p.dst_stride] = v[i];
    }
    if (p.nx_hi) {
      if (FULL) {
        const size_t o = static_cast<size_t>(m0) * p.nx_ld + (n & ~1);
#pragma unroll
        for (int i = 0; i < kDnChunk; i += 2)
          store_parts2(p.nx_hi + o + static_cast<size_t>(i) * p.nx_ld, p.nx_lo + o + static_cast<size_t>(i) * p.nx_ld,
                       p.nx_ld, v[i] * gn, v[i + 1] * gn, lane);
      } else if (ok) {
#pragma unroll
        for (int i = 0; i < kDnChunk; ++i) {
          if (i >= nv) break;
          store_parts(p.nx_hi, p.nx_lo, static_cast<size_t>(m0 + i) * p.nx_ld + n, v[i] * gn);
        }
      }
    }
    if (p.nx_ssq) {
#pragma unroll
      for (int i = 0; i < kDnChunk; ++i) v[i] *= v[i];
      const float q = warp_sum16(v, lane);
      const int i = lane >> 1;
      if (!(lane & 1) && i < nv) p.nx_ssq[static_cast<size_t>(m0 + i) * (4 * p.n_rt) + rt * 4 + (row >> 5)] = q;
    }
  } else {  // ARGMAX
    const int n = rt * kTileN + row;
    const bool ok = n < p.N;
    unsigned long long* wkeys = reinterpret_cast<unsigned long long*>(smem + DnSmem::kKey) + g * 4 * kDnChunk;
    int* last = reinterpret_cast<int*>(smem + DnSmem::kFlag) + g;
    unsigned long long key[kDnChunk];
#pragma unroll
    for (int i = 0; i < kDnChunk; ++i) {
      const float logit = v[i] * rs[i];
      key[i] = ok && i < nv ? argmax_key(logit, static_cast<uint32_t>(n)) : 0ull;
      if (p.logits && ok && i < nv) {
        const int m = m0 + i, b = req[i];
        const DevState* s = p.batch_rows ? p.req_st + b : p.st;
        const int lr = p.logits_step_rows > 0
                           ? __ldcg(&s->steps) * p.logits_step_rows + p.pos_off + m - (p.batch_rows ? b * p.batch_rows : 0)
                           : pos[i] + 1 - __ldcg(&s->prompt_len);
        if (lr >= 0 && lr < p.logits_rows)
          p.logits[(static_cast<size_t>(b) * p.logits_rows + lr) * p.N + n] = logit;
      }
    }
    const unsigned long long km = warp_max16(key, lane);
    if (!(lane & 1)) wkeys[(row >> 5) * kDnChunk + (lane >> 1)] = km;
    group_sync(g);
    if (row < nv) {
      unsigned long long k = wkeys[row];
#pragma unroll
      for (int w = 1; w < 4; ++w) k = max_u64(k, wkeys[w * kDnChunk + row]);
      atomicMax(&p.st->am_key[(m0 + row) * kAmKeyStride], k);
    }
    // one acq_rel ticket per (weight tile, chunk); the tile that completes a chunk's count reads and
    // resets its keys and writes the tokens (-1 once a bounded wait has given up)
    group_sync(g);
    unsigned int* count = &p.st->am_count[(m0 / kDnChunk) * kAmCountStride];
    if (row == 0) *last = atom_add_acq_rel_gpu(count, 1u) == static_cast<unsigned>(p.n_rt - 1);
    group_sync(g);
    if (*last) {
      const bool stopped = (__ldcg(&p.st->error) & DERR_TIMEOUT) != 0;
      if (row < nv) {
        const int m = m0 + row;
        const unsigned long long k = atomicExch(&p.st->am_key[m * kAmKeyStride], 0ull);
        const int tok = stopped ? -1 : static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(k & 0xFFFFFFFFull));
        if (p.batch_rows) {
          const int b = m / p.batch_rows;
          p.tok_dst[b * p.tok_stride + (m - b * p.batch_rows)] = tok;
        } else {
          p.tok_dst[m * (p.tok_stride ? p.tok_stride : 1)] = tok;
        }
      }
      if (row == 0) atomicExch(count, 0u);
    }
    group_sync(g);
  }
}

// ------------------------------------------------------------------ kernel
// map0..2: the site's weight matrices, 128-row (GATE_SILU: 64-row) x 64-column boxes; map_hi / map_lo:
// the rows' parts [rows][K], (nt / 2)-row x 64-column boxes.  Launched in clusters of 2 * split CTAs.
//
// split > 1 (a launch with fewer tiles than CTA pairs, one tile per cluster): pair s of the cluster takes
// the s-th part of the K steps.  The pairs' accumulators meet through distributed shared memory: 16-token
// chunk c belongs to pair c mod split, the others store their chunk into its (by then idle) stage ring, and
// the owner adds them in pair order and runs the chunk's epilogue.
// APART: hi and lo products accumulate apart, the lo accumulator nt columns after the hi one (dense_launch).
template <Epi EPI, bool APART>
__global__ void __launch_bounds__(kDnThreads, 1)
    ssd_dense_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
                     const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap map_hi,
                     const __grid_constant__ CUtensorMap map_lo, const DenseParams p) {
  using S = DnSmem;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);  // the same offset in every CTA of the cluster
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::kBar);  // used in the pair's first CTA
  uint64_t* empty = full + kDnMaxStages;
  uint64_t* tfull = empty + kDnMaxStages;
  uint64_t* tempty = tfull + 2;  // used in the pair's first CTA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + S::kTmemSlot);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int crank = static_cast<int>(cluster_rank()), rank = crank & 1, sp = crank >> 1;
  const uint32_t lead = static_cast<uint32_t>(crank & ~1);  // cluster rank of the pair's first CTA
  const int csize = 2 * p.split, first_tile = blockIdx.x / csize, tile_step = gridDim.x / csize;
  const int n_rp = (p.n_rt + 1) >> 1, tiles = n_rp * p.tok_tiles;
  const int all_steps = p.K / kTileK, k0 = all_steps * sp / p.split, k1 = all_steps * (sp + 1) / p.split;
  const int k_steps = k1 - k0, stages = p.stages, nt = p.nt;
  const uint32_t half_part = static_cast<uint32_t>(nt) * 64;  // bytes of this CTA's hi (or lo) rows of a stage
  const uint32_t stage_bytes = kWTileBytes + 2 * half_part;
  int tmem_cols = 32;
  while (tmem_cols < (APART ? 4 : 2) * nt) tmem_cols <<= 1;
  const uint32_t acc_stride = static_cast<uint32_t>(tmem_cols) >> 1;
  uint8_t* ring = smem + S::kRing;

  if (!p.late_trigger) pdl_trigger();
  if (tid == 0) {
    for (int s = 0; s < kDnMaxStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 16);  // 8 epilogue warps of each CTA of the pair
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tmem_fence_before();
  __syncthreads();
  cluster_sync_all();  // every CTA's barriers exist before another signals them
  tmem_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 || warp == 10) {
    // ---------------------------------------------------------------- TMA producers (every CTA)
    // warp 0: the weights (the first stages before the upstream grid's end) and the stage's expected bytes;
    // warp 10: the tokens' parts.  Everything but the column is fixed along a tile's K steps.
    const bool weights = warp == 0;
    const uint32_t full0 = map_cluster(smem_u32(full), lead);  // the pair's full barriers
    const uint32_t dst0 = smem_u32(ring) + (weights ? 0u : kWTileBytes);
    if (weights) {
      if (elect_one()) prefetch_tensormap(&map0);
    } else {
      if (elect_one()) prefetch_tensormap(&map_hi);
      pdl_wait();
      if (p.late_trigger && elect_one()) pdl_trigger();
    }
    int s = 0, filled = 0;
    uint32_t ph = 1;  // parity to wait for before a fill; the first round of fills does not wait
    bool ok = true;
    for (int t = first_tile; ok && t < tiles; t += tile_step) {
      const int rp = t / p.tok_tiles, rt = 2 * rp + rank;
      const bool have = rt < p.n_rt;  // odd tile count: the last pair's second half has no weights
      const uint32_t bytes = kWTileBytes * (2 * rp + 1 < p.n_rt ? 2u : 1u) + 4 * half_part;
      const CUtensorMap* wm = &map0;
      int y = EPI == Epi::GATE_SILU ? rt * kHalfN : rt * kTileN;
      if constexpr (EPI == Epi::QKV) {
        const int mat = y / p.seg_rows;
        wm = mat == 0 ? &map0 : (mat == 1 ? &map1 : &map2);
        y -= mat * p.seg_rows;
      }
      if (!weights) y = (t - rp * p.tok_tiles) * nt + rank * (nt >> 1);
      for (int ks = k0, x = k0 * kTileK; ks < k1; ++ks, x += kTileK, ++filled) {
        if (filled >= stages && !dense_wait_warp(&empty[s], ph, p.st)) {
          set_error(p.st, DERR_TIMEOUT);
          ok = false;
          break;
        }
        const uint32_t dst = dst0 + s * stage_bytes, bar = full0 + s * 8;
        if (weights) {
          if (elect_one()) {
            if (rank == 0) mbar_arrive_expect_tx(&full[s], bytes);
            if (have) {
              if constexpr (EPI == Epi::GATE_SILU) {
                tma_load_2d_pair(dst, &map0, bar, x, y);
                tma_load_2d_pair(dst + kWTileBytes / 2, &map1, bar, x, y);
              } else {
                tma_load_2d_pair(dst, wm, bar, x, y);
              }
            }
          }
        } else if (elect_one()) {
          tma_load_2d_pair(dst, &map_hi, bar, x, y);
          tma_load_2d_pair(dst + half_part, &map_lo, bar, x, y);
        }
        __syncwarp();
        if (++s == stages) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    // No CTA leaves with a copy in flight, even if a wait gives up only now.  As drain_ring, without its divisions:
    // stages before s were last filled in the ring's current pass (parity ph ^ 1), the others in the one before it (or
    // never: that parity has passed).
    if (weights && rank == 0 && lane == 0)
      for (int q = 0; q < stages; ++q) mbar_wait_for(&full[q], q < s ? ph ^ 1 : ph, 100000000ull);
    __syncwarp();
    if (p.split > 1) {  // the epilogue's two exchanges
      cluster_sync_all();
      cluster_sync_all();
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (the pair's first CTA)
    if (rank == 0) {
      const uint32_t idesc = umma_idesc_bf16(2 * kTileN, nt);
      const uint16_t both = static_cast<uint16_t>(3u << lead);
      const uint64_t w0 = umma_desc_sw128(smem_u32(ring)), h0 = umma_desc_sw128(smem_u32(ring) + kWTileBytes),
                     l0 = umma_desc_sw128(smem_u32(ring) + kWTileBytes + half_part);
      int s = 0, it = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = first_tile; ok && t < tiles; t += tile_step, ++it) {
        const int b = it & 1;
        if (!dense_wait_warp(&tempty[b], static_cast<uint32_t>(((it >> 1) & 1) ^ 1), p.st)) {
          set_error(p.st, DERR_TIMEOUT);
          break;
        }
        tmem_fence_after();
        const uint32_t d = tmem + static_cast<uint32_t>(b) * acc_stride, dl = APART ? d + static_cast<uint32_t>(nt) : d;
        for (int ks = 0; ks < k_steps; ++ks) {
          if (!dense_wait_warp(&full[s], ph, p.st)) {
            set_error(p.st, DERR_TIMEOUT);
            ok = false;
            break;
          }
          tmem_fence_after();
          const uint64_t so = static_cast<uint64_t>((s * stage_bytes) >> 4);  // descriptor units of the stage
          const uint32_t more = ks > 0 ? 1u : 0u, more_lo = APART ? more : 1u;
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < kTileK / 16; ++kk) {
              // +32 bytes (2 descriptor units) per 16-element K slice inside the swizzled row
              umma_f16_pair(d, w0 + so + 2 * kk, h0 + so + 2 * kk, idesc, kk > 0 ? 1u : more);
              umma_f16_pair(dl, w0 + so + 2 * kk, l0 + so + 2 * kk, idesc, kk > 0 ? 1u : more_lo);
            }
            umma_commit_pair(&empty[s], both);  // both CTAs' stage s may be refilled once these MMAs have read it
            if (ks == k_steps - 1) umma_commit_pair(&tfull[b], both);  // accumulator b is complete in both CTAs
          }
          __syncwarp();
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
    }
    __syncwarp();
    if (p.split > 1) {
      cluster_sync_all();
      cluster_sync_all();
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 2..9)
    const int et = tid - 64, ew = et >> 5, g = ew >> 2;  // group 0: warps 2..5, group 1: warps 6..9
    const int q = warp & 3;                              // TMEM lane quadrant this warp may access
    const int row = q * 32 + lane;
    float* xs = reinterpret_cast<float*>(smem + S::kXs) + g * 2 * kTileN * kDnXsLd;
    int xbuf = 0;
    const uint32_t tempty0 = map_cluster(smem_u32(&tempty[0]), lead);
    pdl_wait();
    int it = 0;
    bool ok = true;
    for (int t = first_tile; t < tiles; t += tile_step, ++it) {
      const int b = it & 1;
      const int tt = t % p.tok_tiles, rt = 2 * (t / p.tok_tiles) + rank;
      const int mb = tt * nt, n_tok = min(nt, p.M - mb);
      float* rs = reinterpret_cast<float*>(smem + S::kRs) + b * kDnMaxTok;
      int* pos = reinterpret_cast<int*>(smem + S::kPos) + b * kDnMaxTok;
      int* req = reinterpret_cast<int*>(smem + S::kReq) + b * kDnMaxTok;
      int* kvr = reinterpret_cast<int*>(smem + S::kKvr) + b * kDnMaxTok;
      // the tile's row scales, positions and requests (buffers by tile parity: a group is at most one
      // tile ahead of the other)
      if (p.ssq) {
        for (int i0 = ew * 4; i0 < n_tok; i0 += 32) {
          float a[4] = {0.f, 0.f, 0.f, 0.f};
          for (int f = lane; f < (p.ssq_n >> 2); f += 32) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int m = min(mb + i0 + i, p.M - 1);
              const float4 x = __ldcg(reinterpret_cast<const float4*>(p.ssq + static_cast<size_t>(m) * p.ssq_n) + f);
              a[i] += (x.x + x.y) + (x.z + x.w);
            }
          }
#pragma unroll
          for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] += __shfl_xor_sync(0xffffffffu, a[i], off);
          if (lane < 4 && i0 + lane < n_tok)
            rs[i0 + lane] = rsqrtf((lane == 0 ? a[0] : lane == 1 ? a[1] : lane == 2 ? a[2] : a[3]) /
                                       static_cast<float>(p.K) +
                                   p.eps);
        }
      } else {
        for (int i = et; i < n_tok; i += kDnEpiThreads) rs[i] = p.rs_in ? __ldcg(p.rs_in + mb + i) : 1.0f;
      }
      if constexpr (EPI == Epi::QKV || EPI == Epi::ARGMAX) {
        const int base = (p.abs_pos || p.batch_rows ? 0 : __ldcg(&p.st->kv_len)) + p.pos_off;
        for (int i = et; i < n_tok; i += kDnEpiThreads) {
          const int m = mb + i;
          int4 rm = make_int4(base + m, 0, base + m, 0);
          if (p.row_map) {
            rm = __ldcg(p.row_map + m);
          } else if (p.batch_rows) {
            rm.y = m / p.batch_rows;
            rm.x = rm.z = __ldcg(&p.req_st[rm.y].kv_len) + p.pos_off + m - rm.y * p.batch_rows;
          }
          pos[i] = rm.x;
          req[i] = rm.y;
          kvr[i] = rm.z;
        }
      }
      named_bar_sync(3, kDnEpiThreads);
      const bool have = rt < p.n_rt;
      // this group's chunks: every (2 * split)-th, starting at the pair's own
      const int cstep = 2 * p.split * kDnChunk, cfirst = (g * p.split + sp) * kDnChunk;
      float in[kDnChunk];
      if (have && cfirst < n_tok) chunk_inputs<EPI>(p, rt, mb + cfirst, min(kDnChunk, n_tok - cfirst), pos + cfirst, row, in);
      // after a wait that gave up the loop goes on without waiting (its results are invalid), so that
      // every thread keeps meeting the barriers
      if (ok && !dense_wait(&tfull[b], static_cast<uint32_t>((it >> 1) & 1), p.st)) {
        set_error(p.st, DERR_TIMEOUT);
        ok = false;
      }
      tmem_fence_after();
      const uint32_t acc = tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(b) * acc_stride;
      auto load_chunk = [&](int col, float (&v)[kDnChunk]) {  // 16 tokens of this thread's weight row
        tmem_ld16(acc + col, v);
        if constexpr (APART) {
          float lo[kDnChunk];
          tmem_ld16(acc + nt + col, lo);
#pragma unroll
          for (int i = 0; i < kDnChunk; ++i) v[i] += lo[i];
        }
      };
      float* land = reinterpret_cast<float*>(ring);  // [chunk / split][pair][128][kDnLandLd], over the stage ring
      if (p.split > 1) {
        __syncwarp();
        cluster_sync_all();  // every pair's MMAs are complete: the rings are idle
        int k = 0;
        for (int c = 0; c * kDnChunk < n_tok; ++c) {
          const int own = c % p.split;
          if (own == sp || (k++ & 1) != g || !have) continue;  // the two groups share the other pairs' chunks
          float v[kDnChunk];
          load_chunk(c * kDnChunk, v);
          const uint32_t dst = map_cluster(
              smem_u32(land + ((c / p.split * p.split + sp) * kTileN + row) * kDnLandLd), static_cast<uint32_t>(2 * own + rank));
#pragma unroll
          for (int i = 0; i < 4; ++i) st_cluster_v4(dst + 16 * i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
        __syncwarp();
        cluster_sync_all();  // every chunk has arrived at its owner
      }
      if (have) {
        for (int c0 = cfirst; c0 < n_tok; c0 += cstep) {
          float v[kDnChunk], cur[kDnChunk];
          __syncwarp();
          load_chunk(c0, v);
          if (p.split > 1) {  // the pairs' shares in pair order
            const int base = c0 / kDnChunk / p.split * p.split;
            float sum[kDnChunk];
            for (int s2 = 0; s2 < p.split; ++s2) {
              const float4* l = reinterpret_cast<const float4*>(land + ((base + s2) * kTileN + row) * kDnLandLd);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                float4 x = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                if (s2 != sp) x = l[i];
                sum[4 * i] = s2 ? sum[4 * i] + x.x : x.x;
                sum[4 * i + 1] = s2 ? sum[4 * i + 1] + x.y : x.y;
                sum[4 * i + 2] = s2 ? sum[4 * i + 2] + x.z : x.z;
                sum[4 * i + 3] = s2 ? sum[4 * i + 3] + x.w : x.w;
              }
            }
#pragma unroll
            for (int i = 0; i < kDnChunk; ++i) v[i] = sum[i];
          }
#pragma unroll
          for (int i = 0; i < kDnChunk; ++i) cur[i] = in[i];
          const int c1 = c0 + cstep;
          if (c1 < n_tok) chunk_inputs<EPI>(p, rt, mb + c1, min(kDnChunk, n_tok - c1), pos + c1, row, in);
          int nv = min(kDnChunk, n_tok - c0);
          bool whole = nv == kDnChunk;
          if constexpr (EPI == Epi::QKV) {
            // padding rows (request < 0) end a request's last chunk: only the rows before them are stored
            nv = __popc(__ballot_sync(0xffffffffu, lane < nv && req[c0 + lane] >= 0));
            const int ps = lane < nv ? pos[c0 + lane] : 0;
            whole = nv == kDnChunk && __all_sync(0xffffffffu, ps >= 0 && ps < p.max_seq);
          } else if constexpr (EPI != Epi::ARGMAX) {
            constexpr int kCols = EPI == Epi::GATE_SILU ? kHalfN : kTileN;
            whole = whole && (rt + 1) * kCols <= p.N;
          }
          float* x = xs + xbuf * kTileN * kDnXsLd;
          if (EPI != Epi::ARGMAX && whole)
            dense_chunk<EPI, true>(p, rt, mb + c0, nv, v, cur, rs + c0, pos + c0, req + c0, kvr + c0, x, g, row, smem);
          else
            dense_chunk<EPI, false>(p, rt, mb + c0, nv, v, cur, rs + c0, pos + c0, req + c0, kvr + c0, x, g, row, smem);
          xbuf ^= 1;
        }
      }
      tmem_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty0 + b * 8);  // this warp has read accumulator b
    }
  }
  tmem_fence_before();
  __syncthreads();
  cluster_sync_all();  // no CTA leaves while another may still signal it or read its shared memory
  if (warp == 1) {
    tmem_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
  }
}

}  // namespace ssd
