// Projections of small matrices over up to 16 rows: the latency form of the weight-streaming GEMV.
//
//   out[m][n] = sum_k W[n][k] * a[m][k],   W bf16 [N][K] (nn.Linear layout), a fp32
//
// A matrix that fits the shared memory of the chip (two CTAs of at most 113 KB on every SM: about 30 MB)
// streams in 1..4 us, less than the GEMV's chain of hand-overs costs: operand conversion, MMA, TMEM
// drain, partial sums, ticket, the owner's sum -- 5.7 us for 2048 x 2048 even with the weights in L2.
// Here a CTA owns whole output rows, so nothing is split between CTAs:
//   * before the upstream kernel has finished it brings its rows into shared memory, one bulk copy each
//     (programmatic dependent launch: the copy runs behind the previous kernel);
//   * then every warp loads its slice of K of the activation rows straight into registers, times the
//     norm's gain, as bf16 hi + lo parts (the GEMV's split), and multiplies them with all the CTA's rows by
//     warp-level MMAs (m16n8k16: the activation rows are M, padded to 16, the weight rows N): a lane's
//     fragments of both are 8 consecutive columns, so they need no shuffles, no layout change and, with rows
//     64 bytes apart in the banks, no bank conflicts;
//   * the K slices meet in shared memory and the GEMV's epilogue follows, with 1/rms from the same loads.
// The tensor pipe is far from its limit either way (0.7 us of MMAs at 30 MB); tcgen05 would bring back the
// TMEM and commit hand-overs.  fp32 products on the CUDA cores were measured too: the same at 1 row, but
// 1.7 us more for each further row at 25 MB.
//
// Every sum's order depends on K only, and a row's MMA results do not depend on the other rows, so a row's
// result is bitwise the same at every row count.
#pragma once

#include "gemv.cuh"

namespace ssd {

constexpr int kSmThreads = 256;
constexpr int kSmWarps = kSmThreads / 32;
constexpr int kSmRows = 8;            // weight rows of one MMA
constexpr int kSmCols = 32;           // columns of a lane group's fragments (two K steps of 16)
constexpr int kSmMaxSmem = 115712;    // per CTA with two on an SM
constexpr int kSmMaxK = 4096;         // longest K (small_plan)

struct SmallParams {
  const __nv_bfloat16* w[3];  // the site's matrices, [seg_rows][K] each (GATE_SILU: gate, up)
  int rows;                   // rows per CTA, a multiple of kSmRows
  int total;                  // rows in all (GATE_SILU: gate and up)
};

// Bytes between weight rows in shared memory: two rows 64 bytes apart modulo the banks' 128.
__host__ __device__ constexpr int small_ld(int K) { return K * 2 + 64; }
// Shared memory of one CTA: weights (and over them, once used, the K-slice sums [8][rows][M]), the norm's
// gain, sums of squares [8][kMaxRows], barrier, flag.
__host__ __device__ constexpr int small_smem(int rows, int K) {
  const int w = rows * small_ld(K), red = kSmWarps * rows * kMaxRows * 4;
  return (w > red ? w : red) + K * 2 + kSmWarps * kMaxRows * 4 + 16;
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 8 fp32 values (times 8 bf16 gains) as packed bf16 hi and lo parts; adds their squares (before the gain) to ss.
__device__ __forceinline__ void split8(const float4& a, const float4& b, bool gain, const uint4& gv, uint32_t (&hi)[4],
                                       uint32_t (&lo)[4], float& ss) {
  float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  if (gain) {
    const float2 g0 = bf16x2_to_float2(gv.x), g1 = bf16x2_to_float2(gv.y), g2 = bf16x2_to_float2(gv.z),
                 g3 = bf16x2_to_float2(gv.w);
#pragma unroll
    for (int e = 0; e < 8; ++e) ss = fmaf(v[e], v[e], ss);
    v[0] *= g0.x; v[1] *= g0.y; v[2] *= g1.x; v[3] *= g1.y;
    v[4] *= g2.x; v[5] *= g2.y; v[6] *= g3.x; v[7] *= g3.y;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
    const __nv_bfloat162 l = __floats2bfloat162_rn(v[2 * e] - __low2float(h), v[2 * e + 1] - __high2float(h));
    hi[e] = *reinterpret_cast<const uint32_t*>(&h);
    lo[e] = *reinterpret_cast<const uint32_t*>(&l);
  }
}

// The CTA-order row vr of the site: its matrix and row.  Rows that an epilogue combines are neighbours:
// GATE_SILU gate and up of a column; QKV with rotation the pair (j, j + head_dim / 2) of a head.
template <Epi EPI>
__device__ __forceinline__ void small_row(const GemvParams& p, int vr, int& mat, int& row) {
  if constexpr (EPI == Epi::GATE_SILU) {
    mat = vr & 1;
    row = vr >> 1;
  } else if constexpr (EPI == Epi::QKV) {
    mat = vr / p.seg_rows;
    row = vr - mat * p.seg_rows;
    if (p.rope_cs && mat + p.seg_base < 2) {
      const int j = row & (p.head_dim - 1);
      row = row - j + (j >> 1) + (j & 1) * (p.head_dim >> 1);
    }
  } else {
    mat = 0;
    row = vr;
  }
}

// MH: halves of the MMA's 16 activation rows in use (1: M <= 8, 2: M <= 16).
template <Epi EPI, int MH>
__global__ void __launch_bounds__(kSmThreads, 2) ssd_small_kernel(const SmallParams sp, const GemvParams p, int M) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int R = sp.rows, K = p.K, ld = small_ld(K);
  float* red = reinterpret_cast<float*>(smem);                               // [8][R][M], over the weights
  const int wbytes = max(R * ld, kSmWarps * R * kMaxRows * 4);
  const uint8_t* gs = smem + wbytes;                                         // [K] bf16 gain
  float* sq = reinterpret_cast<float*>(smem + wbytes + K * 2);               // [8][kMaxRows]
  uint64_t* bar = reinterpret_cast<uint64_t*>(sq + kSmWarps * kMaxRows);
  int* stop = reinterpret_cast<int*>(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int v0 = blockIdx.x * R, nr = min(R, sp.total - v0);  // this CTA's rows

  if (!p.late_trigger) pdl_trigger();
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    *stop = (*reinterpret_cast<volatile int*>(&p.st->error) & DERR_TIMEOUT) != 0;
  }
  __syncthreads();
  if (*stop) return;  // a timed-out wait earlier in the decode: nothing was requested yet
  if (warp == 0) {    // the rows do not depend on the previous kernel
    if (lane == 0) {
      mbar_arrive_expect_tx(bar, static_cast<uint32_t>(nr + (p.gain ? 1 : 0)) * K * 2);
      if (p.gain) bulk_load(smem + wbytes, p.gain, K * 2, bar);
    }
    __syncwarp();
    for (int i = lane; i < nr; i += 32) {
      int mat, row;
      small_row<EPI>(p, v0 + i, mat, row);
      const __nv_bfloat16* w = mat == 0 ? sp.w[0] : (mat == 1 ? sp.w[1] : sp.w[2]);
      bulk_load(smem + i * ld, w + static_cast<size_t>(row) * K, K * 2, bar);
    }
  }
  pdl_wait();
  if (p.late_trigger && tid == 0) pdl_trigger();

  // RESID: this thread's base values, fetched now
  constexpr int kItems = 2;
  float base_v[kItems] = {0.f, 0.f};
  if constexpr (EPI == Epi::RESID) {
#pragma unroll
    for (int t = 0; t < kItems; ++t) {
      const int it = tid + t * kSmThreads, m = it / R, n = v0 + it - m * R;
      if (m < M && n < p.N) base_v[t] = __ldcg(p.base + static_cast<size_t>(m) * p.base_stride + n);
    }
  }

  // this warp's 32-column blocks of K; lane (g, t): activation rows g and g + 8, weight row g of a block of 8,
  // columns 8 t .. 8 t + 7 of a 32-column block (the two K steps' fragments, in the same order for both)
  const int g = lane >> 2, t = lane & 3;
  const int nb = K / kSmCols, b0 = nb * warp / kSmWarps, b1 = nb * (warp + 1) / kSmWarps;
  constexpr int kMaxBlocks = 2 * kSmThreads / kMaxRows / kSmRows;  // R <= 32
  float acc[kMaxBlocks][4];
#pragma unroll
  for (int r = 0; r < kMaxBlocks; ++r)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[r][e] = 0.f;
  float ss[MH];
#pragma unroll
  for (int h = 0; h < MH; ++h) ss[h] = 0.f;
  constexpr int kChunk = 8 / MH;  // 32-column blocks whose activations are loaded together (64 registers)
  float4 raw[kChunk][MH][2];
  auto fetch = [&](int c, int blk) {  // block blk's activations
#pragma unroll
    for (int h = 0; h < MH; ++h) {
      const int m = g + 8 * h;
      const bool ok = m < M && blk < b1;
      const float4* x = reinterpret_cast<const float4*>(p.x + static_cast<size_t>(m) * p.x_stride + blk * kSmCols + 8 * t);
      raw[c][h][0] = ok ? __ldcg(x) : make_float4(0.f, 0.f, 0.f, 0.f);
      raw[c][h][1] = ok ? __ldcg(x + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
#pragma unroll
  for (int c = 0; c < kChunk; ++c) fetch(c, b0 + c);
  // The usual 2 s, and the 0.1 s that other kernels wait for their copies after giving up: these copies are all
  // there is to wait for, and the sums lie over them.  One wait, as the kernel has no registers to spare (two cost
  // 0.7 % of a 256-wide model's decode).
  if (!mbar_wait_for(bar, 0, 2100000000ull)) set_error(p.st, DERR_TIMEOUT);
  for (int c0 = b0; c0 < b1; c0 += kChunk) {
#pragma unroll
    for (int c = 0; c < kChunk; ++c) {
      if (c0 + c >= b1) break;
      uint4 gv = make_uint4(0, 0, 0, 0);
      if (p.gain) gv = *reinterpret_cast<const uint4*>(gs + ((c0 + c) * kSmCols + 8 * t) * 2);
      uint32_t hi[MH][4], lo[MH][4];
#pragma unroll
      for (int h = 0; h < MH; ++h) split8(raw[c][h][0], raw[c][h][1], p.gain != nullptr, gv, hi[h], lo[h], ss[h]);
      fetch(c, c0 + kChunk + c);  // the next chunk's block, behind this one's MMAs
      const uint8_t* wc = smem + g * ld + ((c0 + c) * kSmCols + 8 * t) * 2;
#pragma unroll
      for (int r = 0; r < kMaxBlocks; ++r) {
        if (r * kSmRows >= nr) break;  // rows past nr in the last block: sums that nobody reads
        const uint4 w = *reinterpret_cast<const uint4*>(wc + r * kSmRows * ld);
        const uint32_t z = 0;
        mma_bf16(acc[r], hi[0][0], MH > 1 ? hi[MH - 1][0] : z, hi[0][1], MH > 1 ? hi[MH - 1][1] : z, w.x, w.y);
        mma_bf16(acc[r], lo[0][0], MH > 1 ? lo[MH - 1][0] : z, lo[0][1], MH > 1 ? lo[MH - 1][1] : z, w.x, w.y);
        mma_bf16(acc[r], hi[0][2], MH > 1 ? hi[MH - 1][2] : z, hi[0][3], MH > 1 ? hi[MH - 1][3] : z, w.z, w.w);
        mma_bf16(acc[r], lo[0][2], MH > 1 ? lo[MH - 1][2] : z, lo[0][3], MH > 1 ? lo[MH - 1][3] : z, w.z, w.w);
      }
    }
  }
  __syncthreads();  // every warp has read its weights
  // this K slice's sums: acc[r] holds rows m = g (and g + 8) at weight rows 8 r + 2 t, + 1
#pragma unroll
  for (int r = 0; r < kMaxBlocks; ++r) {
    if (r * kSmRows >= nr) break;
    float* d = red + (warp * R + r * kSmRows + 2 * t) * M;
#pragma unroll
    for (int h = 0; h < MH; ++h)
      if (g + 8 * h < M) {
        d[g + 8 * h] = acc[r][2 * h];
        d[M + g + 8 * h] = acc[r][2 * h + 1];
      }
  }
  if (p.gain) {
#pragma unroll
    for (int h = 0; h < MH; ++h) {
      ss[h] += __shfl_xor_sync(0xffffffffu, ss[h], 1);
      ss[h] += __shfl_xor_sync(0xffffffffu, ss[h], 2);
      if (t == 0 && g + 8 * h < M) sq[warp * kMaxRows + g + 8 * h] = ss[h];
    }
  }
  __syncthreads();

  // out[m] of CTA row r (K slices in order, times 1/rms)
  auto value = [&](int m, int r) {
    float s = 0.f, q = 0.f;
#pragma unroll
    for (int k = 0; k < kSmWarps; ++k) s += red[(k * R + r) * M + m];
    if (p.gain) {
#pragma unroll
      for (int k = 0; k < kSmWarps; ++k) q += sq[k * kMaxRows + m];
      s *= rsqrtf(q / static_cast<float>(K) + p.eps);
    }
    return s;
  };
  // position and cache offset of row m
  auto place = [&](int m, long long& kv) {
    if (p.batch_rows) {
      const int b = m / p.batch_rows;
      kv = b * p.req_kv;
      return __ldcg(&p.req_st[b].kv_len) + batch_offset(p, m, b);
    }
    kv = 0;
    return (p.abs_pos ? 0 : __ldcg(&p.st->kv_len)) + p.pos_off + m;
  };
  if constexpr (EPI == Epi::RESID) {
    const float s = __ldg(p.scale);
#pragma unroll
    for (int t = 0; t < kItems; ++t) {
      const int it = tid + t * kSmThreads, m = it / R, r = it - m * R, n = v0 + r;
      if (m < M && r < nr) p.dst[static_cast<size_t>(m) * p.dst_stride + n] = base_v[t] + s * value(m, r);
    }
  } else if constexpr (EPI == Epi::SILU) {
    for (int it = tid; it < M * R; it += kSmThreads) {
      const int m = it / R, r = it - m * R;
      if (r < nr) p.h_out[static_cast<size_t>(m) * p.h_stride + v0 + r] = silu_f(value(m, r));
    }
  } else if constexpr (EPI == Epi::GATE_SILU) {
    const int half = R >> 1;
    for (int it = tid; it < M * half; it += kSmThreads) {
      const int m = it / half, r = 2 * (it - m * half);
      if (r >= nr) continue;
      const float g = value(m, r), u = value(m, r + 1);
      p.h_out[static_cast<size_t>(m) * p.h_stride + ((v0 + r) >> 1)] = (p.act ? gelu_tanh_f(g) : silu_f(g)) * u;
    }
  } else {  // QKV: rows in neighbouring pairs (with rotation: (j, j + head_dim / 2))
    const int half = R >> 1, Dh = p.head_dim;
    for (int it = tid; it < M * half; it += kSmThreads) {
      const int m = it / half, r = 2 * (it - m * half);
      if (r >= nr) continue;
      long long kv;
      const int pos = place(m, kv);
      if (pos < 0 || pos >= p.max_seq) {
        set_error(p.st, DERR_POS);
        continue;
      }
      int mat, row, row2;
      small_row<EPI>(p, v0 + r, mat, row);
      small_row<EPI>(p, v0 + r + 1, mat, row2);
      const int which = mat + p.seg_base;
      float a = value(m, r), b = value(m, r + 1);
      if (p.rope_cs && which < 2) {
        const float2 cs = __ldg(p.rope_cs + static_cast<size_t>(pos) * (Dh >> 1) + (row & (Dh - 1)));
        const float t = a * cs.x - b * cs.y;
        b = a * cs.y + b * cs.x;
        a = t;
      }
      if (which == 0) {
        p.q_out[static_cast<size_t>(m) * p.q_stride + row] = a;
        p.q_out[static_cast<size_t>(m) * p.q_stride + row2] = b;
      } else {
        float* cache = (which == 1 ? p.k_cache : p.v_cache) + kv;
        const int h = row / Dh, j = row - h * Dh, j2 = row2 - h * Dh;
        float* cr = cache + (static_cast<size_t>(h) * p.max_seq + pos) * Dh;
        cr[j] = a;
        cr[j2] = b;
      }
    }
  }
}

}  // namespace ssd
