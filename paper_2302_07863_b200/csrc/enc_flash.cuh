// Self-attention of the encoder (set-up step, d_kv = 64) on the 5th-generation tensor cores: softmax(Q K^T + bias) V per head over all
// encoder positions, bias by signed relative position.
// One block per (head, 128 query rows).  Queries, keys and values arrive as bf16 heads and remainders, written in that form by the epilogue
// of the projection GEMM (values transposed: [channel][position]), so tiles of 64 keys go from memory to tcgen05.mma by TMA with nothing
// in between; three products of each pair are kept (head x head, remainder x head, head x remainder: ~16 mantissa bits).
//   * warp 9 issues the MMAs: scores M128 N64 into one of two accumulators, weighted values M128 N64 (the probabilities from shared
//     memory) into another two; warp 8 feeds the ring of key / value tiles;
//   * two groups of four warps take the even and the odd tiles, thread <-> query row: 64 scores from tensor memory, bias, running
//     maximum, exponentials, probabilities as head and remainder into the group's operand tile, then the tile's weighted values are
//     added to 64 registers with the running soft-max's factor (no accumulator is rescaled in tensor memory); while one group is at its
//     exponentials the tensor pipe works for the other; their results are merged in shared memory at the end.
// Bound by the instruction stream of the soft-max (about 600 instructions a tile and thread) and the 768 tensor-pipe cycles a tile; per layer
// and head at 1024 positions 12 k cycles.  T5-large shapes, 512 positions, from kernel to kernel: the mma.sync kernel 20-23 us, this one
// 14-17; an encode of both models of 1024 ids 3974 -> 2954 us.
#pragma once
#include "enc_attention.cuh"
#include "enc_gemm.cuh"

namespace bild {

constexpr int EF_THREADS = 320, EF_ROWS = 128, EF_KEYS = 64, EF_STAGES = 3;
constexpr int EF_STAGE = 4 * 8192;                // key heads, key remainders, value heads, value remainders of a tile
constexpr int EF_P = 2 * 16384;                   // probabilities of a group's tile: heads, remainders
inline size_t ef_smem_bytes(int max_keys) {
  return 1024 + 2 * 16384 + (size_t)EF_STAGES * EF_STAGE + 2 * EF_P + (size_t)((max_keys + EF_ROWS + 3) & ~3) * 4 + 256;
}
// bf16 x bf16 -> fp32, A and B K-major, M = 128, N = 64
constexpr uint32_t EF_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void ef_mma(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(umma_desc_sw128(a)), "l"(umma_desc_sw128(b)), "r"(EF_IDESC), "r"(accumulate) : "memory");
}
// D = A B^T over 64 columns: Ah Bh + Al Bh + Ah Bl (tiles of 128-byte rows, 128-byte swizzle)
__device__ __forceinline__ void ef_product(uint32_t d, uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) ef_mma(d, ah + kk * 32, bh + kk * 32, kk ? 1u : 0u);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) ef_mma(d, al + kk * 32, bh + kk * 32, 1u);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) ef_mma(d, ah + kk * 32, bl + kk * 32, 1u);
}
__device__ __forceinline__ void ef_ld64(uint32_t taddr, uint32_t (&r)[64]) {   // 64 columns of this warp's lanes
  uint32_t (&lo)[32] = reinterpret_cast<uint32_t (&)[32]>(r[0]);
  uint32_t (&hi)[32] = reinterpret_cast<uint32_t (&)[32]>(r[32]);
  tmem_ld32_issue(taddr, lo);
  tmem_ld32_issue(taddr + 32, hi);
  tmem_ld_wait();
  tmem_ld_pin(lo);
  tmem_ld_pin(hi);
}

// two fp32 operations an instruction
__device__ __forceinline__ float2 ef_fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{.reg .b64 a, b, c, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; mov.b64 c, {%6, %7}; fma.rn.f32x2 d, a, b, c; mov.b64 {%0, %1}, d;}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 ef_add2(float2 a, float2 b) {
  float2 d;
  asm("{.reg .b64 a, b, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; add.rn.f32x2 d, a, b; mov.b64 {%0, %1}, d;}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float ef_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct EncFlashArgs {
  const float* bias;          // [H][bias_ld], entry bias_off + key - query
  int bias_ld, bias_off;
  const int* n_keys_dev;
  int M, H;                   // positions (rows of the launch), heads
  __nv_bfloat16 *oh, *ol;     // [M][H * 64] output as head and remainder
  int* err;
};

// tmQh .. tmKl: [positions][H * 64], boxes of 128 (queries) and 64 (keys) rows x 64 columns; tmVh, tmVl: [H * 64][positions], 64 x 64
template <int CS>   // blocks (a cluster) that share a query tile, each an equal part of the key tiles
__global__ void __launch_bounds__(EF_THREADS, 1) enc_flash_kernel(const EncFlashArgs a, const __grid_constant__ CUtensorMap tmQh,
                                                                   const __grid_constant__ CUtensorMap tmQl, const __grid_constant__ CUtensorMap tmKh,
                                                                   const __grid_constant__ CUtensorMap tmKl, const __grid_constant__ CUtensorMap tmVh,
                                                                   const __grid_constant__ CUtensorMap tmVl) {
  extern __shared__ unsigned char ef_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)ef_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sQ = base;                                   // heads, remainders
  unsigned char* sKV = sQ + 2 * 16384;
  unsigned char* sP = sKV + EF_STAGES * EF_STAGE;             // [group][heads, remainders]
  float* sBias = reinterpret_cast<float*>(sP + 2 * EF_P);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, h = blockIdx.x / CS, r0 = blockIdx.y * EF_ROWS, rank = CS > 1 ? (int)cluster_rank() : 0;
  __shared__ uint64_t kv_full[EF_STAGES], kv_free[EF_STAGES], q_full, s_full[2], p_full[2], o_full[2];
  __shared__ uint32_t tmem_slot;
  if (tid == 0) {
    for (int i = 0; i < EF_STAGES; ++i) { mbar_init(&kv_full[i], 1); mbar_init(&kv_free[i], 1); }
    mbar_init(&q_full, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 1); mbar_init(&o_full[i], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "n"(256) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int E = min(a.M, *a.n_keys_dev), all = (E + EF_KEYS - 1) / EF_KEYS;   // (the count was written before the encoder began)
  const int tile0 = rank * all / CS, tiles = (rank + 1) * all / CS - tile0;   // (rank 0 may have none: one tile, two blocks)
  for (int i = tid; i < E + EF_ROWS - 1; i += EF_THREADS) {   // entry i: key - query = i - (r0 + 127)
    const int idx = a.bias_off + i - (r0 + EF_ROWS - 1);
    sBias[i] = (idx >= 0 && idx < a.bias_ld) ? __ldg(a.bias + (size_t)h * a.bias_ld + idx) : 0.f;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;   // columns: scores of the two groups 0, 64; weighted values 128, 192
  pdl_launch_dependents();
  pdl_wait();
  if (tid == 256) {   // producer
    asm volatile("fence.proxy.async;" ::: "memory");   // rows written with ordinary stores, read by the copy engine
    mbar_expect_tx(&q_full, 2 * 16384);
    tma_load_2d(sQ, &tmQh, h * 64, r0, &q_full);
    tma_load_2d(sQ + 16384, &tmQl, h * 64, r0, &q_full);
    for (int t = 0; t < tiles; ++t) {
      const int st = t % EF_STAGES;
      if (t >= EF_STAGES && !mbar_wait(&kv_free[st], ((t / EF_STAGES) - 1) & 1)) *a.err = BILD_ERR_TIMEOUT;
      unsigned char* s = sKV + st * EF_STAGE;
      mbar_expect_tx(&kv_full[st], EF_STAGE);
      tma_load_2d(s, &tmKh, h * 64, (tile0 + t) * EF_KEYS, &kv_full[st]);
      tma_load_2d(s + 8192, &tmKl, h * 64, (tile0 + t) * EF_KEYS, &kv_full[st]);
      tma_load_2d(s + 16384, &tmVh, (tile0 + t) * EF_KEYS, h * 64, &kv_full[st]);
      tma_load_2d(s + 24576, &tmVl, (tile0 + t) * EF_KEYS, h * 64, &kv_full[st]);
    }
  } else if (tid == 288) {   // MMA issuer
    const uint32_t q = smem_u32(sQ);
    auto scores = [&](int t) {
      const int st = t % EF_STAGES;
      if (!mbar_wait(&kv_full[st], (t / EF_STAGES) & 1)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t k = smem_u32(sKV + st * EF_STAGE);
      ef_product(tmem + (t & 1) * 64, q, q + 16384, k, k + 8192);
      umma_commit(&s_full[t & 1]);
    };
    if (!mbar_wait(&q_full, 0)) *a.err = BILD_ERR_TIMEOUT;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tiles > 0) scores(0);
    if (tiles > 1) scores(1);
    for (int t = 0; t < tiles; ++t) {
      const int g = t & 1, st = t % EF_STAGES;
      if (!mbar_wait(&p_full[g], (t >> 1) & 1)) *a.err = BILD_ERR_TIMEOUT;   // (and the group has taken its scores: their accumulator is free)
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t p = smem_u32(sP + g * EF_P), v = smem_u32(sKV + st * EF_STAGE) + 16384;
      ef_product(tmem + 128 + g * 64, p, p + 16384, v, v + 8192);
      umma_commit(&o_full[g]);
      umma_commit(&kv_free[st]);
      if (t + 2 < tiles) scores(t + 2);
    }
  }
  __syncwarp();
  float o[64], m = -INFINITY, l = 0.f;
  const int g = warp >> 2, row = (warp & 3) * 32 + lane;   // (warps 8, 9: unused)
  if (warp < 8) {
#pragma unroll
    for (int j = 0; j < 64; ++j) o[j] = 0.f;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    unsigned char* ph = sP + g * EF_P + row * 128;
    const float* brow = sBias + EF_ROWS - 1 - row;   // entry of key 0 for this thread's query
#pragma unroll 1
    for (int t = g; t < tiles; t += 2) {
      const unsigned par = (t >> 1) & 1;
      if (!mbar_wait(&s_full[g], par)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t sr[64];
      ef_ld64(tl + g * 64, sr);
      const int k0 = (tile0 + t) * EF_KEYS;
      float mq[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};   // (four chains: one would wait for itself)
      if (k0 + EF_KEYS <= E) {
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          const float s = __uint_as_float(sr[j]) + brow[k0 + j];
          sr[j] = __float_as_uint(s);
          mq[j & 3] = fmaxf(mq[j & 3], s);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          const float s = k0 + j < E ? __uint_as_float(sr[j]) + brow[k0 + j] : -INFINITY;
          sr[j] = __float_as_uint(s);
          mq[j & 3] = fmaxf(mq[j & 3], s);
        }
      }
      const float mx = fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3]));
      constexpr float LOG2E = 1.4426950408889634f;
      const float nw = fmaxf(m, mx), sc = ef_exp2((m - nw) * LOG2E), nl = -nw * LOG2E;   // (first tile: 0)
      m = nw;
      float2 sum[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      // probabilities as head and remainder, eight keys (16 bytes) a store, into the swizzled operand tile
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 x = ef_fma2(make_float2(__uint_as_float(sr[8 * c + 2 * i]), __uint_as_float(sr[8 * c + 2 * i + 1])), make_float2(LOG2E, LOG2E),
                                   make_float2(nl, nl));
          const float2 p = make_float2(ef_exp2(x.x), ef_exp2(x.y));
          sum[i] = ef_add2(sum[i], p);
          hi[i] = ea_pack(p.x, p.y);
          const float2 q = ef_fma2(make_float2(__uint_as_float(hi[i] << 16), __uint_as_float(hi[i] & 0xffff0000u)), make_float2(-1.f, -1.f), p);
          lo[i] = ea_pack(q.x, q.y);
        }
        const int at = (c ^ (row & 7)) << 4;
        *reinterpret_cast<uint4*>(ph + at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4*>(ph + 16384 + at) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      }
      const float2 s2 = ef_add2(ef_add2(sum[0], sum[1]), ef_add2(sum[2], sum[3]));
      l = l * sc + (s2.x + s2.y);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the MMAs
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      ea_group_sync(g);
      if ((tid & 127) == 0) mbar_arrive(smem_u32(&p_full[g]));
      __syncwarp();   // (the arrival before its siblings poll)
      if (!mbar_wait(&o_full[g], par)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      ef_ld64(tl + 128 + g * 64, sr);
#pragma unroll
      for (int j = 0; j < 64; j += 2) {
        const float2 v = ef_fma2(make_float2(o[j], o[j + 1]), make_float2(sc, sc), make_float2(__uint_as_float(sr[j]), __uint_as_float(sr[j + 1])));
        o[j] = v.x; o[j + 1] = v.y;
      }
    }
  }
  // the odd tiles' results meet the even tiles' (thread to thread: the same row), in the place of the queries and key tiles; then the
  // second block's the first's
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  float* sM = reinterpret_cast<float*>(base);   // [66][128]
  if (warp >= 4 && warp < 8) {
#pragma unroll
    for (int j = 0; j < 64; ++j) sM[j * 128 + row] = o[j];
    sM[64 * 128 + row] = m; sM[65 * 128 + row] = l;
  }
  __syncthreads();
  auto merge = [&](const float* p) {
    const float m1 = p[64 * 128 + row], l1 = p[65 * 128 + row], gm = fmaxf(m, m1);
    const float w0 = m == -INFINITY ? 0.f : __expf(m - gm), w1 = m1 == -INFINITY ? 0.f : __expf(m1 - gm);
#pragma unroll
    for (int j = 0; j < 64; ++j) o[j] = o[j] * w0 + p[j * 128 + row] * w1;
    l = l * w0 + l1 * w1;
    m = gm;
  };
  if (warp < 4) merge(sM);
  if (CS > 1) {
    float* sR = sM + 66 * 128;   // (behind the block's own exchange area: queries and key tiles are done with in both blocks)
    __syncwarp();
    cluster_sync_all();
    if (rank == 1 && warp < 4) {
#pragma unroll
      for (int j = 0; j < 64; ++j) st_cluster_f1(smem_u32(sR + j * 128 + row), 0, o[j]);
      st_cluster_f1(smem_u32(sR + 64 * 128 + row), 0, m);
      st_cluster_f1(smem_u32(sR + 65 * 128 + row), 0, l);
    }
    __syncwarp();
    cluster_sync_all();
    if (rank == 0 && warp < 4) merge(sR);
  }
  if (rank == 0 && warp < 4 && r0 + row < E) {
    const float inv = 1.f / l;
    uint4* ph = reinterpret_cast<uint4*>(a.oh + (size_t)(r0 + row) * a.H * 64 + h * 64);
    uint4* pl = reinterpret_cast<uint4*>(a.ol + (size_t)(r0 + row) * a.H * 64 + h * 64);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) ea_split(o[8 * c + 2 * i] * inv, o[8 * c + 2 * i + 1] * inv, hi[i], lo[i]);
      ph[c] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      pl[c] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
  __syncthreads();
  if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(256) : "memory");
}

}  // namespace bild
