// Self-attention of the encoder (set-up step, d_kv = 64) on the 5th-generation tensor cores: softmax(Q K^T + bias) V per head over all
// encoder positions, bias by signed relative position.
// One block per (head, 128 query rows).  Queries, keys and values arrive as bf16 heads and remainders, written in that form by the epilogue
// of the projection GEMM (values transposed: [channel][position]), so tiles of 64 keys go from memory to tcgen05.mma by TMA with nothing
// in between; three products of each pair are kept (head x head, remainder x head, head x remainder: ~16 mantissa bits).
//   * warp 9 issues the MMAs, operand A always from tensor memory (queries: copied there once; probabilities: written over the scores they
//     come from), so that shared memory serves the key and value tiles alone: scores M128 N64 of up to four tiles ahead, weighted
//     values M128 N64 into one accumulator a group; warp 8 feeds the rings of key and of value tiles;
//   * two groups of four warps take the even and the odd tiles, thread <-> query row: 64 scores from tensor memory, bias, maximum,
//     exponentials, probabilities as head and remainder back.  The weighted values stay in tensor memory from tile to tile: the
//     exponentials refer to the first tile's maximum until one is more than 2^8 above it, and only then is the accumulator rescaled.
//     So a group goes from tile to tile without waiting for the tensor pipe; the groups' results are merged in shared memory
//     at the end.
// Takes 9.5 us a layer for one key tile, 17.5 for 512 and 36 for 1024 positions (T5-large shapes; an encode with it less one without).  Of the
// 36: 10 for the second and third products of each pair (an M128 N64 K16 MMA takes about 75 cycles, whichever memory A comes from and
// with two accumulators in turn as well), 3 for the merge and the output; exponentials and bias cost nothing on top.
// With the probabilities in shared memory and the products awaited tile by tile: encode of 389 / 512 ids, T5 pair, 1720 / 1746 us, now
// 1660 / 1699; mT5 pair, 300 ids 1735, now 1673; 1024 ids 2861 and 2853; up to 64 ids 1107 and 1110.
#pragma once
#include "enc_attention.cuh"
#include "enc_gemm.cuh"

namespace bild {

constexpr int EF_THREADS = 320, EF_ROWS = 128, EF_KEYS = 64, EF_STAGES = 4;
constexpr int EF_STAGE = 4 * 8192;                // key heads, key remainders, value heads, value remainders of a tile
constexpr int EF_Q = 384;                         // tensor memory: scores of tile t from 64 (t % 4), weighted values of the groups from 256, queries
inline size_t ef_smem_bytes(int max_keys) {
  return 1024 + 2 * 16384 + (size_t)EF_STAGES * EF_STAGE + (size_t)((max_keys + EF_ROWS + 3) & ~3) * 4 + 256;
}
// bf16 x bf16 -> fp32, M = 128, N = 64: A from tensor memory (a lane <-> a row, two columns of the row in 32 bits), B K-major in shared memory
constexpr uint32_t EF_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void ef_mma(uint32_t d_tmem, uint32_t a_tmem, uint32_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(umma_desc_sw128(b)), "r"(EF_IDESC), "r"(accumulate) : "memory");
}
// D = A B^T over 64 columns: Ah Bh + Al Bh + Ah Bl (A: 32 columns of heads, 32 of remainders; B: tiles of 128-byte rows, 128-byte swizzle;
// add: on top of what D holds)
__device__ __forceinline__ void ef_product(uint32_t d, uint32_t a, uint32_t bh, uint32_t bl, bool add) {
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) ef_mma(d, a + kk * 8, bh + kk * 32, kk || add ? 1u : 0u);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) ef_mma(d, a + 32 + kk * 8, bh + kk * 32, 1u);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) ef_mma(d, a + kk * 8, bl + kk * 32, 1u);
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

__device__ __forceinline__ void ef_st32(uint32_t taddr, const uint32_t* r) {   // 32 columns of this warp's lanes
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,"
      "%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),
      "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
      "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory");
}

__device__ __forceinline__ void ef_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
               "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
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
  float* sBias = reinterpret_cast<float*>(sKV + EF_STAGES * EF_STAGE);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, h = blockIdx.x / CS, r0 = blockIdx.y * EF_ROWS, rank = CS > 1 ? (int)cluster_rank() : 0;
  __shared__ uint64_t k_full[EF_STAGES], k_free[EF_STAGES], v_full[EF_STAGES], v_free[EF_STAGES], q_full, q_there, s_full[4], p_full[4], o_full[4], o_done;
  __shared__ uint32_t tmem_slot;
  if (tid == 0) {
    for (int i = 0; i < EF_STAGES; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_free[i], 1); mbar_init(&v_full[i], 1); mbar_init(&v_free[i], 1); }
    mbar_init(&q_full, 1);
    mbar_init(&q_there, 4);
    mbar_init(&o_done, 1);
    for (int i = 0; i < 4; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 1); mbar_init(&o_full[i], 1); }   // by tile: a group may be two ahead of the products
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "n"(512) : "memory");
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
  const uint32_t tmem = tmem_slot;
  pdl_launch_dependents();
  pdl_wait();
  if (tid == 256) {   // producer
    asm volatile("fence.proxy.async;" ::: "memory");   // rows written with ordinary stores, read by the copy engine
    mbar_expect_tx(&q_full, 2 * 16384);
    tma_load_2d(sQ, &tmQh, h * 64, r0, &q_full);
    tma_load_2d(sQ + 16384, &tmQl, h * 64, r0, &q_full);
    auto load = [&](int t, bool v) {   // key or value tile t: heads, then remainders
      const int st = t % EF_STAGES;
      uint64_t *full = v ? &v_full[st] : &k_full[st], *free = v ? &v_free[st] : &k_free[st];
      if (t >= EF_STAGES && !mbar_wait(free, ((t / EF_STAGES) - 1) & 1)) *a.err = BILD_ERR_TIMEOUT;
      unsigned char* s = sKV + st * EF_STAGE + (v ? 16384 : 0);
      const int x = v ? (tile0 + t) * EF_KEYS : h * 64, y = v ? h * 64 : (tile0 + t) * EF_KEYS;
      mbar_expect_tx(full, EF_STAGE / 2);
      tma_load_2d(s, v ? &tmVh : &tmKh, x, y, full);
      tma_load_2d(s + 8192, v ? &tmVl : &tmKl, x, y, full);
    };
    // the next tile's keys ahead of a tile's values: the scores run ahead, and a value tile's place is free only behind the products of
    // the tile three before
    if (tiles > 0) load(0, false);
    for (int t = 0; t < tiles; ++t) {
      if (t + 1 < tiles) load(t + 1, false);
      load(t, true);
    }
  } else if (tid == 288) {   // MMA issuer
    auto scores = [&](int t) {
      const int st = t % EF_STAGES;
      if (!mbar_wait(&k_full[st], (t / EF_STAGES) & 1)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t k = smem_u32(sKV + st * EF_STAGE);
      ef_product(tmem + (t & 3) * 64, tmem + EF_Q, k, k + 8192, false);
      umma_commit(&s_full[t & 3]);
      umma_commit(&k_free[st]);
    };
    if (!mbar_wait(&q_there, 0)) *a.err = BILD_ERR_TIMEOUT;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    for (int t = 0; t < 4 && t < tiles; ++t) scores(t);
    for (int t = 0; t < tiles; ++t) {
      const int g = t & 1, st = t % EF_STAGES;
      if (!mbar_wait(&p_full[t & 3], (t >> 2) & 1)) *a.err = BILD_ERR_TIMEOUT;
      if (!mbar_wait(&v_full[st], (t / EF_STAGES) & 1)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t v = smem_u32(sKV + st * EF_STAGE) + 16384;
      ef_product(tmem + 256 + g * 64, tmem + (t & 3) * 64, v, v + 8192, t >= 2);   // (the probabilities lie where the scores were)
      umma_commit(&o_full[t & 3]);
      umma_commit(&v_free[st]);
      if (t + 4 < tiles) scores(t + 4);   // (behind the products that read the probabilities there: MMAs run in order)
    }
    umma_commit(&o_done);
  }
  __syncwarp();
  float o[64], m = -INFINITY, l = 0.f;   // m: what the row's exponentials refer to
  const int g = warp >> 2, row = (warp & 3) * 32 + lane;   // (warps 8, 9: unused)
  if (warp < 8) {
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16), to = tl + 256 + g * 64;
    if (g == 0) {   // the queries into tensor memory: as the MMAs' operand they would be read from shared memory anew for every tile
      if (!mbar_wait(&q_full, 0)) *a.err = BILD_ERR_TIMEOUT;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t r[32];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint4 v = *reinterpret_cast<const uint4*>(sQ + half * 16384 + row * 128 + ((c ^ (row & 7)) << 4));
          r[4 * c] = v.x; r[4 * c + 1] = v.y; r[4 * c + 2] = v.z; r[4 * c + 3] = v.w;
        }
        ef_st32(tl + EF_Q + half * 32, r);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&q_there));
      __syncwarp();
    }
    const float* brow = sBias + EF_ROWS - 1 - row;   // entry of key 0 for this thread's query
#pragma unroll 1
    for (int t = g; t < tiles; t += 2) {
      if (!mbar_wait(&s_full[t & 3], (t >> 2) & 1)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t sr[64];
      ef_ld64(tl + (t & 3) * 64, sr);
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
      if (t >= 2) {
        // The exponentials refer to an earlier tile's maximum while that is at most 2^8 too low (a factor that cancels in the end);
        // only beyond are the sums brought to the new one.
        const bool far = !((mx - m) * LOG2E <= 8.f);
        if (__any_sync(0xffffffffu, far)) {
          // (the products of this group's tile before; those of tile t - 6, the barrier's phase before, are long behind these scores)
          if (!mbar_wait(&o_full[(t - 2) & 3], ((t - 2) >> 2) & 1)) *a.err = BILD_ERR_TIMEOUT;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const float nw = far ? fmaxf(m, mx) : m, sc = m == nw ? 1.f : ef_exp2((m - nw) * LOG2E);
          m = nw;
          l *= sc;
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            uint32_t r[32];
            tmem_ld32_issue(to + half * 32, r);
            tmem_ld_wait();
            tmem_ld_pin(r);
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) * sc);
            ef_st32(to + half * 32, r);
          }
        }
      } else {
        m = mx;
      }
      const float nl = -m * LOG2E;
      float2 sum[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      // probabilities as head and remainder, two keys in 32 bits, over the scores
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float2 x = ef_fma2(make_float2(__uint_as_float(sr[32 * c + 2 * i]), __uint_as_float(sr[32 * c + 2 * i + 1])), make_float2(LOG2E, LOG2E),
                                   make_float2(nl, nl));
          const float2 p = make_float2(ef_exp2(x.x), ef_exp2(x.y));
          sum[i & 3] = ef_add2(sum[i & 3], p);
          hi[i] = ea_pack(p.x, p.y);
          const float2 q = ef_fma2(make_float2(__uint_as_float(hi[i] << 16), __uint_as_float(hi[i] & 0xffff0000u)), make_float2(-1.f, -1.f), p);
          lo[i] = ea_pack(q.x, q.y);
        }
        ef_st16(tl + (t & 3) * 64 + c * 16, hi);
        ef_st16(tl + (t & 3) * 64 + 32 + c * 16, lo);
      }
      const float2 s2 = ef_add2(ef_add2(sum[0], sum[1]), ef_add2(sum[2], sum[3]));
      l += s2.x + s2.y;
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      ea_group_sync(g);
      if ((tid & 127) == 0) mbar_arrive(smem_u32(&p_full[t & 3]));
      __syncwarp();   // (the arrival before its siblings poll)
    }
    if (g < tiles) {
      if (!mbar_wait(&o_done, 0)) *a.err = BILD_ERR_TIMEOUT;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t sr[64];
      ef_ld64(to, sr);
#pragma unroll
      for (int j = 0; j < 64; ++j) o[j] = __uint_as_float(sr[j]);
    } else {
#pragma unroll
      for (int j = 0; j < 64; ++j) o[j] = 0.f;
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
  if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512) : "memory");
}

}  // namespace bild
