// Decoder sub-layers as ONE kernel each (bf16 weights, up to 8 token rows a launch), so that a layer
// of a decoder pass is three dependent kernels instead of eight:
//   * attn_sub_kernel: x_out = x_in + W_o * Attention(W_q|k|v * rms_norm(x_in))   (steps S1-S3 / L1-L3
//     for self-attention, S4-S6 / L4-L6 for cross-attention).  A cluster of C blocks owns one head:
//     rank r multiplies its share of the head's q|k|v rows (weights fetched by bulk copies BEFORE
//     the dependency wait of the programmatic launch), the cluster exchanges the k x 3 x d_kv results
//     through distributed shared memory (asynchronous stores that an mbarrier counts), rank r then attends over its share of the keys, the
//     per-rank (max, sum, weighted values) records are exchanged the same way, and every rank
//     multiplies the merged head output with its share of the rows of W_o's column slice; while a head has few keys
//     (they fit one staged chunk) every rank attends over all of them instead and the second exchange falls away;
//     the first kernel of a pass takes its rows from the embedding table (S0 / L0);
//   * ffn_sub_kernel: x_out = x_in + W_fo * act(W_i * rms_norm(x_in))   (S7-S8 / L7-L8).  Block b owns a
//     slice of d_ff (a multiple of 8 rows): the rows of W_i (and of the gate matrix) and the matching columns of W_fo
//     (from a copy laid out in load order), so the hidden activations never leave the block.
// Both kernels produce partial sums over heads / slices of d_ff of the d_model outputs.  They are added
// into x_out with vector reductions at the L2 (red.global.add); x_out was zeroed by the kernel before the
// previous one, one designated block adds x_in (the residual term), and every kernel zeroes the buffer
// the next kernel accumulates into: three buffers rotate through the pass.  The order of the floating-
// point additions at the L2 is not fixed, so logits may differ in the last bits from run to run.
#pragma once
#include "slice_linear.cuh"

namespace bild {

constexpr int SUB_THREADS = 256;
constexpr int SUB_RECPAD = 4;       // record of a rank and row = [max, sum, -, -, values[d_kv]]
constexpr int SUB_MAX_ROWS = 48;             // weight rows of one block and phase: three 16-row tiles
constexpr int SUB_FO_REGS = 32;              // most rows of d_ff a block takes: its columns of W_fo fill 64 registers of a thread
constexpr int SUB_HALF_SM = 113 * 1024;      // shared memory of a block that leaves room for a second one on the SM
constexpr int SUB_MB = 8;                    // token rows of the block variant (one 8-token tile of the tensor-core instruction)

struct SubShared {
  unsigned long long wbar;      // weight copies
  unsigned long long xbar[2];   // exchanges within the cluster
  float ssq[8][SUB_MB];         // the warps' sums of squares of the token rows
  int failed;
};

// Optional cycle stamps (build with -DBILD_STAMPS), summed per kernel kind and phase boundary: [0] block 0, [1] every
// block, [2] the longest a block took ([..][23]: how many blocks were added).
#ifdef BILD_STAMPS
__device__ unsigned long long g_sub_stamps[3][4][24];
#define SUB_STAMP_BEGIN() long long st_t[20]; int st_n = 0; st_t[st_n++] = clock64()
#define SUB_STAMP() st_t[st_n++] = clock64()
#define SUB_STAMP_END(kind)                                                                                \
  if (threadIdx.x == 0) {                                                                                 \
    for (int i_ = 1; i_ < st_n; ++i_) {                                                                   \
      const unsigned long long dt_ = (unsigned long long)(st_t[i_] - st_t[i_ - 1]);                      \
      if (blockIdx.x == 0) atomicAdd(&g_sub_stamps[0][kind][i_ - 1], dt_);                                \
      atomicAdd(&g_sub_stamps[1][kind][i_ - 1], dt_);                                                     \
      atomicMax(&g_sub_stamps[2][kind][i_ - 1], dt_);                                                     \
    }                                                                                                     \
    if (blockIdx.x == 0) atomicAdd(&g_sub_stamps[0][kind][23], 1ull);                                     \
    atomicAdd(&g_sub_stamps[1][kind][23], 1ull);                                                          \
  }
#else
#define SUB_STAMP_BEGIN()
#define SUB_STAMP()
#define SUB_STAMP_END(kind)
#endif

__host__ __device__ inline int sub_up16(int v) { return (v + 15) & ~15; }
// row stride (floats) of staged keys / values: 16 mod 32, so the four channel quarters of two keys hit 32 distinct banks
__host__ __device__ inline int sub_kv_stride(int dkv) { return ((dkv + 15) / 32) * 32 + 16; }

// Bounded wait for the weight copies: after `spin` unsuccessful polls the block records BILD_ERR_TIMEOUT for the host
// and goes on (with whatever the shared memory holds), so that every block of the kernel still leaves.
__device__ __forceinline__ void sub_wait(SubShared* sh, int* err, unsigned long long* bar, uint32_t parity, unsigned spin) {
  __syncwarp();   // (a lane that polls must not keep a sibling from issuing a copy)
  const uint32_t b = smem_u32(bar);
  if (mbar_try(b, parity)) return;
  if (*(volatile int*)&sh->failed) return;
  for (unsigned it = 0; it < spin; ++it)
    if (mbar_try(b, parity)) return;
  sh->failed = 1;
  atomicExch(err, (int)BILD_ERR_TIMEOUT);
}

// (nothing to publish: does not wait for the loads in flight)
__device__ __forceinline__ void sub_cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void sub_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void sub_cp16(void* dst_smem, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void sub_cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ bool sub_try_cluster(uint32_t bar, uint32_t parity) {   // (what the cluster's other blocks wrote is visible after it)
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Wait for the values the cluster's blocks store into this one (sub_push).  Every block sends its part after bounded waits of
// its own, so the limit here is only a last bound, above theirs.
// (The warp meets first: a lane that polls must not keep a sibling from sending what the others wait for.)
__device__ __forceinline__ void sub_wait_exchange(SubShared* sh, int* err, unsigned long long* bar, unsigned spin) {
  __syncwarp();
  const uint32_t b = smem_u32(bar);
  const unsigned lim = (spin > SPIN_LIMIT ? spin : SPIN_LIMIT) * 4u;
  for (unsigned it = 0; it < lim; ++it)
    if (sub_try_cluster(b, 0)) return;
  sh->failed = 1;
  atomicExch(err, (int)BILD_ERR_TIMEOUT);
}
// Stores into the shared memory of block `rank` of the cluster that count down the bytes its mbarrier `bar` expects: the
// receiver waits for the bytes, nobody for a cluster-wide barrier with its release of everything written before (which cost
// 883 cycles per exchange against 510 of these stores, eight blocks, 192 values each to everyone).
__device__ __forceinline__ void sub_push(const float* dst, const unsigned long long* bar, uint32_t rank, float v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
               ::"r"(cluster_map(smem_u32(dst), rank)), "r"(__float_as_uint(v)), "r"(cluster_map(smem_u32(bar), rank)) : "memory");
}
__device__ __forceinline__ void sub_push4(const float* dst, const unsigned long long* bar, uint32_t rank, float4 v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(cluster_map(smem_u32(dst), rank)), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
               "r"(__float_as_uint(v.w)), "r"(cluster_map(smem_u32(bar), rank)) : "memory");
}

__device__ __forceinline__ void sub_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void sub_mma8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(b0));
}
// two fp32 values as a pair of bf16 heads and a pair of bf16 remainders
__device__ __forceinline__ void sub_split(float x, float y, uint32_t& h, uint32_t& l) {
  h = sl_pack_bf16(x, y);
  l = sl_pack_bf16(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xffff0000u));
}
// ... and as three (24 mantissa bits: the fp32 values themselves)
__device__ __forceinline__ void sub_split3(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = sl_pack_bf16(x, y);
  const float rx = x - __uint_as_float(h << 16), ry = y - __uint_as_float(h & 0xffff0000u);
  m = sl_pack_bf16(rx, ry);
  l = sl_pack_bf16(rx - __uint_as_float(m << 16), ry - __uint_as_float(m & 0xffff0000u));
}

// ------------------------------------------------------------------------------------------------
// Products of a block's weight rows with the token rows
// ------------------------------------------------------------------------------------------------
// Warp w owns the columns [w CW, (w + 1) CW) of every row (CW = 32 x sub_chunks(d), 128 for d = 1024): it fetches that slice of
// the token rows from the L2, multiplies it with the norm gain, splits it into bf16 parts in its own piece of shared memory
// and multiplies it with its slice of the weight rows on mma.sync m16n8k16 -- no block barrier between the token rows and the
// products; the one barrier behind the products covers the eight warps' partial sums and their sums of squares (1 / rms is a
// factor of the sums).  Within a chunk of 32 columns the instruction's column positions are dealt so that a lane's 16-byte load
// holds the operands of two instructions (position 2 t, 2 t + 1 | 2 t + 8, 2 t + 9 of instruction i <-> columns
// 8 t + 4 i + 0, 1 | 2, 3), weights and token rows alike.
// A single token row is three columns of the right operand: its bf16 head, remainder and second remainder, so the products are
// those of the fp32 row at one instruction per 16 x 16 weights (multiply-adds with a warp reduction took twice the time of
// rows + norm + products together: 2.2 -> 1.1 us per attention kernel of the large model).
// A block of token rows is multiplied twice, heads and remainders, into two accumulator chains.
__host__ __device__ inline int sub_chunks(int d) { return ((d + 31) / 32 + 7) / 8; }                 // 32-column chunks per warp: 1..4
__host__ __device__ inline int sub_wst(int d) { return (d * 2 + 127) / 128 * 128 + 64; }            // bytes from weight row to weight row: 64 mod 128
__host__ __device__ inline int sub_xst(int d) { return (d / 2 + 31) / 32 * 32 + 16; }               // words from token row to token row: 16 mod 32
__host__ __device__ inline int sub_pst(int rows, bool half = false) {   // floats of partial sums per token: 2 p = 8 (half a tile: 24) mod 32
  return half ? 12 : (rows + 15) / 16 * 16 + 4;
}
__host__ __device__ inline int sub_xs_bytes(int d, int mb) { return (mb == 1 ? 3 : 2 * SUB_MB) * sub_xst(d) * 4; }
__host__ __device__ inline int sub_psum_bytes(int rows, int mb, bool half = false) { return 8 * (mb == 1 ? 1 : SUB_MB) * sub_pst(rows, half) * 4; }

template <bool ONE>
struct SubRows { float4 v[ONE ? 1 : SUB_MB]; };

// this lane's four columns of the token rows (after the dependency wait)
template <bool ONE>
__device__ __forceinline__ void sub_rows_issue(const float* __restrict__ x_in, int rows, int d, int col, bool on, SubRows<ONE>& rw) {
#pragma unroll
  for (int i = 0; i < (ONE ? 1 : SUB_MB); ++i)
    if (on && i < rows) rw.v[i] = __ldcg(reinterpret_cast<const float4*>(x_in + (size_t)i * d + col));
}

// The first sub-layer of a pass takes its rows from the embedding table (S0 / L0): row i = E[token_i], bf16.
template <bool ONE>
__device__ __forceinline__ void sub_rows_embed(const __nv_bfloat16* __restrict__ E, const int* __restrict__ tokens, int vocab, int rows,
                                               int d, int col, bool on, SubRows<ONE>& rw) {
#pragma unroll
  for (int i = 0; i < (ONE ? 1 : SUB_MB); ++i)
    if (on && i < rows) {
      int t = tokens[i];
      t = t < 0 ? 0 : (t >= vocab ? vocab - 1 : t);
      const uint2 w = __ldg(reinterpret_cast<const uint2*>(E + (size_t)t * d + col));
      rw.v[i] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                            __uint_as_float(w.y & 0xffff0000u));
    }
}

// Splits x * gain into the warp's slice of Xs and leaves the warp's sums of squares in sh->ssq.  Xs: [part][row] rows of
// sub_xst(d) words; `stores`: this lane's columns lie in the warp's slice, `on`: and inside the rows.  The raw values of the
// columns [seed0, seed1) go to sSeed[m][column - seed0]: the residual term the block adds.
template <bool ONE>
__device__ __forceinline__ void sub_rows_split(const SubRows<ONE>& rw, int k, int col, bool stores, bool on, float4 g, uint32_t* Xs, int xst,
                                               SubShared* sh, float* sSeed, int seed0, int seed1, int lane, int warp) {
  const bool sd = on && col >= seed0 && col < seed1;
  float q[ONE ? 1 : SUB_MB];
#pragma unroll
  for (int i = 0; i < (ONE ? 1 : SUB_MB); ++i) {
    q[i] = 0.f;
    if (stores && i < k) {
      float4 w = on ? rw.v[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      q[i] = w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
      if (sd) *reinterpret_cast<float4*>(sSeed + (size_t)i * (seed1 - seed0) + (col - seed0)) = w;
      w.x *= g.x; w.y *= g.y; w.z *= g.z; w.w *= g.w;
      uint32_t h0, h1, l0, l1, m0, m1;
      if (ONE) {
        sub_split3(w.x, w.y, h0, m0, l0); sub_split3(w.z, w.w, h1, m1, l1);
        *reinterpret_cast<uint2*>(Xs + xst + (col >> 1)) = make_uint2(m0, m1);
        *reinterpret_cast<uint2*>(Xs + 2 * xst + (col >> 1)) = make_uint2(l0, l1);
      } else {
        sub_split(w.x, w.y, h0, l0); sub_split(w.z, w.w, h1, l1);
        *reinterpret_cast<uint2*>(Xs + (size_t)(SUB_MB + i) * xst + (col >> 1)) = make_uint2(l0, l1);
      }
      *reinterpret_cast<uint2*>(Xs + (size_t)i * xst + (col >> 1)) = make_uint2(h0, h1);
    }
  }
  if (ONE) {
    const float s = warp_sum(q[0]);
    if (lane == 0) sh->ssq[warp][0] = s;
  } else {
    float qq[SUB_MB];
#pragma unroll
    for (int i = 0; i < SUB_MB; ++i) qq[i] = q[ONE ? 0 : i];
    const float r8 = treduce<SUB_MB>(qq, lane);   // lanes 4 i hold the warp's sum of row i
    if ((lane & 3) == 0) sh->ssq[warp][lane >> 2] = r8;
  }
  __syncwarp();
}
// 1 / x of a soft-max's sum (1 to the number of keys), relative error at most 2^-23: the hardware's approximation (its error, 2^-23, is
// squared) and a Newton step of two roundings; a full division is a chain several times as long.  Not for 0 and infinity.
__device__ __forceinline__ float sub_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r * fmaf(-x, r, 2.f);
}
__global__ void sub_rcp_kernel(const float* x, float* y, int n) {   // (for its test)
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = sub_rcp(x[i]);
}
// 1 / rms of token row m from the warps' sums of squares (after the barrier behind the products)
__device__ __forceinline__ float sub_inv(const SubShared* sh, int m, float inv_d, float eps) {
  float s[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) s[w] = sh->ssq[w][m];
  return rsqrtf((((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]))) * inv_d + eps);
}

// the left operands of this warp's slice of half a 16-row tile (chunks past the end of the rows: zero; rows past the last one: the last one
// again, their sums are not read)
__device__ __forceinline__ void sub_frags8(const unsigned char* sW, int wst, int nrows, int d, int half, int col0, int nch, int lane, uint4 (&f)[4]) {
  const int g = lane >> 2, t = lane & 3;
  const unsigned char* p0 = sW + (size_t)min(half * 8 + g, nrows - 1) * wst + (col0 + 8 * t) * 2;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    const bool in = ch < nch && col0 + ch * 32 + 8 * t < d;
    f[ch] = in ? *reinterpret_cast<const uint4*>(p0 + ch * 64) : make_uint4(0u, 0u, 0u, 0u);
  }
}
// the right operands: the warp's slice of the token rows
template <bool ONE> struct SubB { uint4 h[4], l[ONE ? 1 : 4]; };
template <bool ONE>
__device__ __forceinline__ void sub_bfrags(const uint32_t* Xs, int xst, int k, int col0, int nch, int lane, SubB<ONE>& b) {
  const int g = lane >> 2, t = lane & 3;
  const uint32_t* p = Xs + (size_t)min(g, (ONE ? 3 : k) - 1) * xst + (col0 >> 1) + 4 * t;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch)
    if (ch < nch) {
      b.h[ch] = *reinterpret_cast<const uint4*>(p + ch * 16);
      if (!ONE) b.l[ONE ? 0 : ch] = *reinterpret_cast<const uint4*>(p + (size_t)SUB_MB * xst + ch * 16);
    }
}
// one 16-row tile, its halves' operands f0 and f1 (`both`: the second one exists); the warp's partial sums go to psum [warp][token][sub_pst(rows)]
// HALF: of a block variant with up to 8 weight rows
template <bool ONE, bool HALF = false>
__device__ __forceinline__ void sub_tile(const uint4 (&f0)[4], const uint4 (&f1)[4], bool both, const SubB<ONE>& b, int nch, int nrows, int mt, float* psum, int warp, int lane) {
  const int g = lane >> 2, t = lane & 3, pst = sub_pst(nrows, HALF), row = mt * 16 + g;
  float c[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int ch = 0; ch < 4; ++ch)
    if (ch < nch) {
      const uint4 a0 = f0[ch], a1 = both ? f1[ch] : make_uint4(0u, 0u, 0u, 0u);
      sub_mma(c, a0.x, a1.x, a0.y, a1.y, b.h[ch].x, b.h[ch].y);
      if (ONE) {
        sub_mma(e, a0.z, a1.z, a0.w, a1.w, b.h[ch].z, b.h[ch].w);
      } else {
        sub_mma(e, a0.x, a1.x, a0.y, a1.y, b.l[ONE ? 0 : ch].x, b.l[ONE ? 0 : ch].y);
        sub_mma(c, a0.z, a1.z, a0.w, a1.w, b.h[ch].z, b.h[ch].w);
        sub_mma(e, a0.z, a1.z, a0.w, a1.w, b.l[ONE ? 0 : ch].z, b.l[ONE ? 0 : ch].w);
      }
    }
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] += e[i];
  if (ONE) {   // accumulator columns 0, 1 (lane t = 0) and 2 (lane t = 1): the three parts of the token row
    const float z0 = __shfl_down_sync(0xffffffffu, c[0], 1), z2 = __shfl_down_sync(0xffffffffu, c[2], 1);
    if (t == 0) {
      psum[(size_t)warp * pst + row] = c[0] + c[1] + z0;
      psum[(size_t)warp * pst + row + 8] = c[2] + c[3] + z2;
    }
  } else {
    float* p = psum + (size_t)(warp * SUB_MB + 2 * t) * pst + row;
    p[0] = c[0]; p[pst] = c[1];
    if (!HALF) { p[8] = c[2]; p[pst + 8] = c[3]; }
  }
}
// dot product (weight row, token row) over all warps, in a fixed order
template <bool ONE>
__device__ __forceinline__ float sub_total(const float* psum, int row, int m, int pst) {
  const float* p = psum + (size_t)m * pst + row;
  float v[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) v[w] = p[w * (ONE ? 1 : SUB_MB) * pst];   // (a warp without columns left zeros)
  return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
}

// ------------------------------------------------------------------------------------------------
// Attention sub-layer
// ------------------------------------------------------------------------------------------------
// What a kernel of a single-row pass asks into the L2 of the LM head's weights: chunks c0 .. c1 - 1, one every `stride` bytes, dealt to the
// blocks.  Block passes leave it out: no gain there, and the block kernels have no register for it.
struct HeadAhead { const unsigned char* base; size_t total, stride; unsigned len; int c0, c1; };
__device__ __forceinline__ void head_ahead(const HeadAhead& p) {   // one thread
  for (int i = p.c0 + (int)blockIdx.x; i < p.c1; i += (int)gridDim.x) {
    const size_t at = (size_t)i * p.stride;
    if (at < p.total)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.base + at), "r"((unsigned)min((size_t)p.len, p.total - at)) : "memory");
  }
}

struct AttnSubLayout { int wq, kv, kv2_k, kv2_v, kv_late, xs, rec, rrec, qkv, psum, sa, out, bias, seed, sh, total; };

struct AttnSubArgs {
  const CallDesc* desc;
  const float* x_in;    // [rows of the pass][d] residual stream (complete)
  const __nv_bfloat16* emb;  // not null: the first sub-layer of a pass, its rows are E[tokens[i]] instead of x_in (S0 / L0)
  const int* tokens;
  int vocab;
  float* x_out;         // [MAXB][d] zero on entry; receives x_in + the sub-layer's output
  float* x_zero;        // [MAXB][d] cleared for the kernel after this one
  const float* gain;
  float eps, inv_d;          // inv_d: 1 / d
  const __nv_bfloat16* Wp;   // self: [3 I][d] (q rows, then k, then v); cross: [I][d]
  const __nv_bfloat16* Wo;   // [d][I]
  float* kc;                 // [H][cap][dkv] keys of this layer (self: rows pos0.. are appended; cross: read only)
  float* vc;
  int cap;
  const float* bias;         // self: [H][bias_ld] relative-position bias by distance; cross: unused
  int bias_ld;
  const int* n_keys_dev;     // cross: encoder positions
  int self;
  int d, I, H, dkv, dkv_shift, C, c_shift;
  int kc_keys;               // keys per staged chunk
  int kc_main;               // WIDE: of them in the main area (the rest where the weight rows were)
  int red_keys;              // up to this many keys every rank attends over ALL keys of the head (no second exchange)
  int bias_len;              // floats reserved for the staged bias
  int mb;                    // token rows the shared memory is sized for
  unsigned spin;             // polls of the weight barrier before the kernel gives up
  int skip_copies;           // test of the time-out path: the weight copies are announced but not issued
  int early;                 // 1: the next kernel may start at once, 0: once this kernel has its token rows
  int* err;
  AttnSubLayout L;
  HeadAhead ahead;           // AHEAD
};

// Shared memory is kept under half an SM's (113 KB) where possible, so that the next kernel's blocks can sit beside
// this kernel's and run their prologue and weight fetch in its shadow (and so that 16 clusters of 8 are resident at
// once: above that size an SM takes one block, and a B200 then holds only 15 such clusters).
// late: the keys / values are staged where the projection's weight rows were, once those wait in registers.
// kc_main < kc: the keys from there on are.  kvst: floats from key to key.
inline AttnSubLayout attn_sub_layout(int d, int dkv, int P, int C, int mb, int kc, int bias_len, int late, int kc_main, int kvst) {
  AttnSubLayout L;
  const int npr = (P * dkv + C - 1) / C, no = (d + C - 1) / C, rec = dkv + SUB_RECPAD;
  const int wq_b = sub_up16(std::max(npr * sub_wst(d), (kc - kc_main) * (kvst + dkv + 4) * 4)), kv_b = sub_up16(kc_main * (kvst + dkv + 4) * 4);
  int off = 0;
  L.kv_late = late;
  L.wq = off; off += late ? std::max(wq_b, kv_b) : wq_b;
  L.kv = late ? L.wq : off; off += late ? 0 : kv_b;
  // floats from where a key / value past kc_main would follow the others to where it is: behind L.wq, keys first
  L.kv2_k = (L.wq - L.kv) / 4 - kc_main * kvst;
  L.kv2_v = (L.wq - L.kv) / 4 + (kc - kc_main) * kvst - kc_main * (dkv + 4) - kc_main * kvst;
  // token rows; afterwards the warps' records and the ranks' records
  L.xs = off; L.rec = off; L.rrec = off + sub_up16(8 * mb * rec * 4);
  off += std::max(sub_up16(sub_xs_bytes(d, mb)), sub_up16(8 * mb * rec * 4) + sub_up16(C * mb * rec * 4));
  L.qkv = off; off += sub_up16(mb * (P * dkv + 16) * 4);
  // partial sums of the products; afterwards the merged head output (block variant)
  L.psum = off; L.sa = off; L.out = L.rec;   // (the output tile: the records are merged by then)
  static_assert(SUB_MB * (SUB_THREADS / 2 + 4) * 4 <= 8 * SUB_MB * (16 + SUB_RECPAD) * 4, "at most 128 outputs a block, records of 16 channels and more");
  off += std::max(sub_up16(sub_psum_bytes(npr, mb, kc_main < kc)), mb == 1 ? 0 : sub_up16(mb * (dkv + 4) * 4));
  L.bias = off; off += sub_up16(bias_len * 4);
  L.seed = off; off += sub_up16(mb * no * 4);
  L.sh = off; off += sub_up16((int)sizeof(SubShared));
  L.total = off;
  return L;
}

// Chunk size, bias room and the key count up to which the ranks attend redundantly, for a cache of keys_cap keys.
// `all_keys` > 0 asks for a chunk that holds up to that many keys so that short caches need no second exchange; the
// chunk shrinks until the layout for passes of `mb` rows (1: the single-row kernel, SUB_MB: the block kernel; each has a plan
// of its own) stays under `prefer` bytes (half an SM), else under `limit`.
struct AttnSubPlan {
  int kc, bias_len, red_keys, late;
  bool ok;
  int kc_main, kvst;   // keys of a chunk in the main area, floats from key to key
  bool wide() const { return kc_main < kc; }
};
inline AttnSubPlan attn_sub_plan(int d, int dkv, int P, int C, int keys_cap, int all_keys, int prefer, int limit, int mb) {
  AttnSubPlan pl;
  const int per_rank = (keys_cap + C - 1) / C;
  const int need = std::min(64, sub_up16(per_rank)), want = std::min(128, sub_up16(std::max(per_rank, std::min(all_keys, keys_cap))));
  auto blen = [&](int kc) { return P == 3 ? (std::max(per_rank, kc) + MAXB + 8 + 3) / 4 * 4 : 4; };
  auto fits = [&](int kc, int lim) {
    for (pl.late = 0; pl.late < (P == 3 && (P * dkv + C - 1) / C <= 24 ? 2 : 1); ++pl.late)   // (cross-attention: its keys are requested first
      // thing, into an area of their own; more than 24 weight rows do not all wait in registers)
      if (attn_sub_layout(d, dkv, P, C, mb, kc, blen(kc), pl.late, kc, sub_kv_stride(dkv)).total <= lim) return true;
    pl.late = 0;
    return false;
  };
  int kc = std::max(need, want);
  while (kc > need && !fits(kc, prefer)) kc -= 16;
  while (kc > 16 && !fits(kc, limit)) kc -= 16;
  pl.kc = kc; pl.bias_len = blen(kc); pl.ok = fits(kc, limit);
  if (fits(kc, prefer)) pl.ok = true;
  else fits(kc, limit);
  pl.kc_main = kc; pl.kvst = sub_kv_stride(dkv);
  // Cross-attention of many keys: closer rows (two-way bank conflicts on the keys) and the room of the weight rows for the last keys hold a
  // rank's whole share of up to 1024 encoder keys in one chunk (a second one is staged and waited for inside the chain:
  // T5-large, 1024 ids, 200 cached rows, 2 / 5 / 8 rows 537 / 574 / 650 -> 509 / 544 / 620 us a pass, 800 ids 515 / 552 / 620 -> 492 / 527 / 593).
  if (P == 1 && mb > 1 && per_rank > kc && all_keys > 0 && (dkv + C - 1) / C <= 8) {
    const int st = dkv + 4, row_b = (st + dkv + 4) * 4, rest = sub_up16(((dkv + C - 1) / C) * sub_wst(d)) / row_b, wide = std::min(128, per_rank), main = wide - rest;
    if (wide > kc && main >= 16 && rest > 0 && attn_sub_layout(d, dkv, P, C, mb, wide, blen(wide), 0, main, st).total <= prefer) {
      kc = pl.kc = wide; pl.kc_main = main; pl.kvst = st; pl.late = 0; pl.bias_len = blen(wide); pl.ok = true;
    }
  }
  pl.red_keys = all_keys > 0 ? kc : 0;
  return pl;
}

// (max, sum, values) records of one token row added up, channels [4 u, 4 u + 4), and their sum; u < 0: the merged (max, sum, -, -)
template <bool EIGHT>   // n is 8
__device__ __forceinline__ float4 sub_merge_t(const float* rec, int stride, int n, int u, float& sum) {
  float m[8], l[8];
  const int uo = u < 0 ? 0 : SUB_RECPAD + 4 * u;
#pragma unroll
  for (int i = 0; i < 8; ++i) {   // (loads side by side; past the last record: the last one again, with weight 0)
    const float2 ml = *reinterpret_cast<const float2*>(rec + (EIGHT ? i : min(i, n - 1)) * stride);
    m[i] = ml.x; l[i] = EIGHT || i < n ? ml.y : 0.f;
  }
  const float gm = fmaxf(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])), fmaxf(fmaxf(m[4], m[5]), fmaxf(m[6], m[7])));
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  sum = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 v = *reinterpret_cast<const float4*>(rec + (EIGHT ? i : min(i, n - 1)) * stride + uo);
    const float w = l[i] > 0.f ? __expf(m[i] - gm) : 0.f;
    sum += w * l[i];
    o.x += w * v.x; o.y += w * v.y; o.z += w * v.z; o.w += w * v.w;
  }
  return u < 0 ? make_float4(gm, sum, 0.f, 0.f) : o;
}
__device__ __forceinline__ float4 sub_merge(const float* rec, int stride, int n, int u, float& sum) {
  return n == 8 ? sub_merge_t<true>(rec, stride, 8, u, sum) : sub_merge_t<false>(rec, stride, n, u, sum);
}

// One token row: this warp's keys of the chunk, eight at a time, two eights side by side.  Lane (key, channel quarter) scores,
// lane <-> two channels (one, with d_kv = 32 or 16) of the weighted values; everything stays in the warp.
struct SubAtt1 { float run, sum; float2 acc; };
template <typename KP, typename VP>
__device__ __forceinline__ void sub_attend_one(const float4 (&q)[4], int dq4, int dkv, int nk, KP kp, VP vp, const float* sBias, int bias0, bool biased,
                                               SubAtt1& st, int warp, int lane) {
  const int key = lane >> 2, qt = lane & 3, cw = dkv >= 64 ? 2 : 1, ch = min(lane * cw, dkv - cw);
#pragma unroll 1
  for (int t0 = warp * 8; t0 < nk; t0 += 128) {
    const bool two = t0 + 64 < nk;
    float s[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = t0 + 64 * h + key;
      s[h] = -INFINITY;
      if (h == 0 || two) {
        const float* p = kp(min(j, nk - 1));
        float a = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (u < dq4) {
            const float4 k4 = *reinterpret_cast<const float4*>(p + (u * 4 + qt) * 4);
            a += q[u].x * k4.x + q[u].y * k4.y + q[u].z * k4.z + q[u].w * k4.w;
          }
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (j < nk) s[h] = biased ? a + sBias[bias0 - j] : a;
      }
    }
    float mx = fmaxf(s[0], s[1]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float nw = fmaxf(st.run, mx), sc = st.run == -INFINITY ? 0.f : __expf(st.run - nw);
    const float p0 = __expf(s[0] - nw), p1 = __expf(s[1] - nw);   // (a key that is not there: 0)
    st.run = nw;
    st.sum = st.sum * sc + p0 + p1;          // per lane: the keys of its quad
    st.acc.x *= sc; st.acc.y *= sc;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (h == 0 || two) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float w = __shfl_sync(0xffffffffu, h ? p1 : p0, i * 4);
          const float* v = vp(min(t0 + 64 * h + i, nk - 1)) + ch;
          if (cw == 2) {
            const float2 v2 = *reinterpret_cast<const float2*>(v);
            st.acc.x += w * v2.x; st.acc.y += w * v2.y;
          } else {
            st.acc.x += w * v[0];
          }
        }
      }
  }
}

// Up to 8 token rows: this warp's keys of the chunk, eight at a time, on mma.sync: scores (token rows x keys, 16 channels per
// m16n8k16) leave a lane (token g; keys 2 t, 2 t + 1) with just the left operand of the weighted values (token rows x channels,
// eight keys per m16n8k8), so soft-max and both products stay in the warp, without a barrier.  Queries, keys, probabilities and
// values each as a bf16 head and remainder, three of the four products kept.  Channels are dealt to the instruction's positions so that
// keys and values arrive with 16-byte loads: score step i, positions (2 t, 2 t + 1 | 2 t + 8, 2 t + 9) <-> channels
// 16 i + 4 t + 0, 1 | 2, 3; value column g of tile n <-> channel 32 (n / 4) + 4 g + n % 4 (d_kv = 16: 2 g + n).
struct SubAtt8 { float run, sum; float o[8][4]; };
struct SubQ8 { uint32_t h[4][2], l[4][2]; };
template <typename KP, typename VP>
__device__ __forceinline__ void sub_attend_block(const SubQ8& q, int dkv, int nk, KP kp, VP vp, const float* sBias, int bias0, bool biased, int limit,
                                                 SubAtt8& st, int warp, int lane) {
  // bias0 - j: index of the bias of key j for this lane's token; limit: the last key this lane's token sees
  const int g = lane >> 2, t = lane & 3;
#pragma unroll 1
  for (int t0 = warp * 8; t0 < nk; t0 += 64) {
    float c[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f}, f[4] = {0.f, 0.f, 0.f, 0.f};
    const float* k0 = kp(min(t0 + g, nk - 1)) + 4 * t;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i * 16 < dkv) {
        const float4 k4 = *reinterpret_cast<const float4*>(k0 + i * 16);
        uint32_t h0, h1, l0, l1;
        sub_split(k4.x, k4.y, h0, l0); sub_split(k4.z, k4.w, h1, l1);
        sub_mma(c, q.h[i][0], 0u, q.h[i][1], 0u, h0, h1);
        sub_mma(e, q.l[i][0], 0u, q.l[i][1], 0u, h0, h1);
        sub_mma(f, q.h[i][0], 0u, q.h[i][1], 0u, l0, l1);
      }
    float s0 = c[0] + (e[0] + f[0]), s1 = c[1] + (e[1] + f[1]);
    const int ja = t0 + 2 * t, jb = ja + 1;
    if (biased) {
      s0 += sBias[max(0, bias0 - ja)]; s1 += sBias[max(0, bias0 - jb)];
    }
    if (ja > limit) s0 = -INFINITY;
    if (jb > limit) s1 = -INFINITY;
    float mx = fmaxf(s0, s1);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float nw = fmaxf(st.run, mx);
    const float sc = st.run == -INFINITY ? 0.f : __expf(st.run - nw);
    const float p0 = s0 == -INFINITY ? 0.f : __expf(s0 - nw), p1 = s1 == -INFINITY ? 0.f : __expf(s1 - nw);
    st.run = nw;
    st.sum = st.sum * sc + p0 + p1;   // per lane: its two keys
    uint32_t ph, pl;
    sub_split(p0, p1, ph, pl);
    const float* va = vp(min(ja, nk - 1));
    const float* vb = vp(min(jb, nk - 1));
#pragma unroll
    for (int n4 = 0; n4 < 2; ++n4)
      if (n4 * 32 < dkv) {
        float4 x, y;
        if (dkv >= 32) {
          x = *reinterpret_cast<const float4*>(va + n4 * 32 + 4 * g); y = *reinterpret_cast<const float4*>(vb + n4 * 32 + 4 * g);
        } else {
          const float2 x2 = *reinterpret_cast<const float2*>(va + 2 * g), y2 = *reinterpret_cast<const float2*>(vb + 2 * g);
          x = make_float4(x2.x, x2.y, 0.f, 0.f); y = make_float4(y2.x, y2.y, 0.f, 0.f);
        }
        const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          float (&o)[4] = st.o[n4 * 4 + n];
          o[0] *= sc; o[1] *= sc;
          uint32_t vh, vl;
          sub_split(xs[n], ys[n], vh, vl);
          sub_mma8(o, ph, 0u, vh);
          sub_mma8(o, pl, 0u, vh);
          sub_mma8(o, ph, 0u, vl);
        }
      }
  }
}

// ONE: a single token row (the small model's step, the large model's single-row pass); else 2 to 8 rows.
// Bound by the latency of its dependent chain (5 rows: 8 % of the memory's rate, 6-8 % of the tensor pipe while it runs): token rows from the L2,
// products, exchange of q | k | v within the head's cluster, attention, [exchange of the ranks' records], output products, reductions
// at the L2.  What is off the chain is done before the dependency wait: the weight rows wait as operands in registers, W_o's too,
// the cached keys and values in shared memory.  Between barriers each warp works alone: three (four) block barriers and one
// (two) waits for the cluster per kernel.
// Measured, T5-large shapes, pass of 24 layers, cache 32, 512 encoder keys, before -> after this form of the kernels (both
// sub-layer kernels; before: token rows and norm for the whole block, then products from shared memory, cluster barriers, scores,
// soft-max and values with a block barrier each): 1 row 473 -> 355 us, 5 rows 632 -> 550 us, 8 rows 691 -> 597 us, 16 rows
// 1080 -> 831 us; T5-small 100 -> 83 us.  With the steps noted at their places since: 311, 500, 552, 740 and 72 us.
// WIDE: cross-attention of a block whose last keys of a chunk lie where the weight rows were (attn_sub_plan); a kernel of its own, since the
// others would spill registers for it.
// AHEAD (single rows): asks for some of the LM head's weights on the way (head_share); instances of their own, since the few instructions cost
// a pass of 73 kernels 1.3 %.
// FIX (single rows): a kernel for self- or cross-attention (KIND) over heads of 64 channels in clusters of eight, all of which the compiler then knows.
// DQ (single rows, here and in the feed-forward kernel): rows of 256 DQ columns, so that every warp has all of its 32 DQ columns and every stride and
// trip count is a constant; the widths of 512, 768 and 1024, others go by DQ = 0.  These kernels are a chain of a few instructions at a time, so the index
// arithmetic and the branches that go are time.  General kernels -> FIX -> with DQ: a step of the T5-small shapes 78.1 -> 74.0 -> 71.9 us, mT5-small
// 117.9 -> 113.4 -> 109.2, single-row pass of T5-large 336.6 -> 327.2 -> 311.3, mT5-large 397.0 -> 392.8 -> 373.7.  The block kernels, at the limit of their
// registers, spill some with FIX, head width and cluster size
// together (5 rows 502 -> 522 us; DQ or KIND by itself was not tried there but for WIDE), and take every shape.
constexpr int SUB_CROSS = 0, SUB_SELF = 1, SUB_EITHER = 2;
template <bool ONE, bool WIDE = false, bool AHEAD = false, bool FIX = false, int KIND = SUB_EITHER, int DQ = 0>
__global__ void __launch_bounds__(SUB_THREADS, 2) attn_sub_kernel(const AttnSubArgs a) {
  extern __shared__ __align__(1024) unsigned char sub_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool self = KIND == SUB_EITHER ? a.self != 0 : KIND == SUB_SELF;
  const int C = FIX ? 8 : a.C, c_shift = FIX ? 3 : a.c_shift, d = DQ ? 256 * DQ : a.d, dkv = FIX ? 64 : a.dkv, dkv_shift = FIX ? 6 : a.dkv_shift;
  const int P = self ? 3 : 1, R = P * dkv;
  const int h = blockIdx.x >> c_shift, r = (int)cluster_rank();
  const int pr0 = (r * R) >> c_shift, npr = (((r + 1) * R) >> c_shift) - pr0;   // rows of the head's q|k|v projection
  const int no = d >> c_shift, o0 = r * no;                                         // output rows of W_o
  const int wst = sub_wst(d), xst = sub_xst(d), kvst = WIDE ? dkv + 4 : sub_kv_stride(dkv), qst = R + 16, recst = dkv + SUB_RECPAD;
  const int vst = dkv + 4;   // row stride of the staged values: the rows 2 t and channels 4 g of a tile hit 32 banks
  unsigned char* sWq = sub_smem + a.L.wq;
  uint32_t* Xs = reinterpret_cast<uint32_t*>(sub_smem + a.L.xs);
  float* sRec = reinterpret_cast<float*>(sub_smem + a.L.rec);     // [8 warps][mb][recst]
  float* sRrec = reinterpret_cast<float*>(sub_smem + a.L.rrec);   // [C ranks][mb][recst]
  float* sK = reinterpret_cast<float*>(sub_smem + a.L.kv);
  float* sV = sK + (size_t)(WIDE ? a.kc_main : a.kc_keys) * kvst;
  float* sQKV = reinterpret_cast<float*>(sub_smem + a.L.qkv);     // [mb][qst]
  float* psum = reinterpret_cast<float*>(sub_smem + a.L.psum);
  float* sBias = reinterpret_cast<float*>(sub_smem + a.L.bias);
  float* sSeed = reinterpret_cast<float*>(sub_smem + a.L.seed);
  float* sA = reinterpret_cast<float*>(sub_smem + a.L.sa);        // [mb][dkv + 4]
  SubShared* sh = reinterpret_cast<SubShared*>(sub_smem + a.L.sh);
  const int cpw = sub_chunks(d), col0 = warp * 32 * cpw, nch = DQ ? cpw : max(0, min(cpw, (d - col0 + 31) >> 5));
  const int col = col0 + lane * 4;
  const bool stores = lane * 4 < 32 * nch, on = stores && (DQ || col < d);   // this lane's four columns of the token rows
  SUB_STAMP_BEGIN();

  if (tid == 0) {
    mbar_init(smem_u32(&sh->wbar), 1);
    mbar_init(smem_u32(&sh->xbar[0]), 1);
    mbar_init(smem_u32(&sh->xbar[1]), 1);
    sh->failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect(smem_u32(&sh->wbar), (uint32_t)(npr * d * 2));
  }
  __syncthreads();
  if (a.early) pdl_launch_dependents();
  // weights depend on nothing: requested before the dependency wait.  Row i is copied by lane i / 8 of warp i % 8:
  // the copies a warp issues go out one after the other (about 25 ns each), the warps issue side by side
  {
    const int i = ((tid & 31) << 3) | (tid >> 5);
    if (i < npr && !a.skip_copies) {
      const int j = pr0 + i, part = j >> dkv_shift, ch = j & (dkv - 1);
      bulk_g2s(smem_u32(sWq + (size_t)i * wst), a.Wp + ((size_t)part * a.I + h * dkv + ch) * d, (uint32_t)(d * 2), smem_u32(&sh->wbar));
    }
  }
  if (AHEAD && tid == SUB_THREADS - 1) head_ahead(a.ahead);
  // output projection: warp w owns rows 16 w .. 16 w + 15 of this rank's share of W_o's column slice.  Thread (g, t) of the
  // warp keeps, of rows g and g + 8, the channels [t d_kv / 4, (t + 1) d_kv / 4), two per register: as it stands the left
  // operand of mma.sync m16n8k16 with the channels of a 16-channel step dealt out four to a thread
  const int og = lane >> 2, ot = lane & 3, cpt = dkv >> 2;
  uint32_t wr[2][8];
#pragma unroll
  for (int rr = 0; rr < 2; ++rr) {
#pragma unroll
    for (int i = 0; i < 8; ++i) wr[rr][i] = 0u;
    if (warp * 16 < no) {
      const __nv_bfloat16* p = a.Wo + (size_t)(o0 + min(warp * 16 + og + 8 * rr, no - 1)) * a.I + h * dkv + ot * cpt;
      if (cpt == 4) {
        asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(wr[rr][0]), "=r"(wr[rr][1]) : "l"(p));
      } else {
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(wr[rr][0]), "=r"(wr[rr][1]), "=r"(wr[rr][2]), "=r"(wr[rr][3]) : "l"(p));
        if (cpt == 16)
          asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(wr[rr][4]), "=r"(wr[rr][5]), "=r"(wr[rr][6]), "=r"(wr[rr][7]) : "l"(p + 8));
      }
    }
  }
  float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (on) g4 = __ldg(reinterpret_cast<const float4*>(a.gain + col));
  const float* Kh = a.kc + (size_t)h * a.cap * dkv;
  const float* Vh = a.vc + (size_t)h * a.cap * dkv;
  // places of a chunk's key jj
  auto k_at = [&](int jj) { return sK + ((size_t)jj * kvst + (WIDE && jj >= a.kc_main ? a.L.kv2_k : 0)); };
  auto v_at = [&](int jj) { return sV + ((size_t)jj * vst + (WIDE && jj >= a.kc_main ? a.L.kv2_v : 0)); };
  // stages keys / values [c0 + r0, c1) of the cache into the places r0.. (asynchronous 16-byte copies)
  auto stage_cached = [&](int c0, int c1, int r0 = 0) {
    const int up_sh = dkv_shift - 2, units = (c1 - c0) << up_sh;
#pragma unroll 1
    for (int i = tid + (r0 << up_sh); i < units; i += SUB_THREADS) {
      const int jj = i >> up_sh, u = (i & ((1 << up_sh) - 1)) * 4;
      sub_cp16(k_at(jj) + u, Kh + (size_t)(c0 + jj) * dkv + u);
      sub_cp16(v_at(jj) + u, Vh + (size_t)(c0 + jj) * dkv + u);
    }
  };
  // Few keys: every rank attends over all of them (the keys of the cache come from the L2, those of this pass from the
  // first exchange anyway), which costs a fraction of a microsecond and saves the exchange of the records and their merge.
  int n_keys = 0, j0 = 0, j1 = 0;
  bool red = false;
  if (!self) {   // the encoder keys are static: the first chunk is requested before the wait as well
    n_keys = min(*a.n_keys_dev, a.cap);
    red = n_keys <= a.red_keys;
    j0 = red ? 0 : (r * n_keys) >> c_shift; j1 = red ? n_keys : ((r + 1) * n_keys) >> c_shift;
    stage_cached(j0, min(j1, j0 + (WIDE ? a.kc_main : a.kc_keys)));
    // a share of more than one chunk: the later chunks are asked into the L2 now (they are staged when the first is used up)
    const int later = (j1 - j0 - a.kc_keys) * dkv / 32;   // 128-byte lines of keys (as many again of values)
#pragma unroll 1
    for (int i = tid; i < later; i += SUB_THREADS) {
      const size_t o = (size_t)(j0 + a.kc_keys) * dkv + (size_t)i * 32;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(Kh + o));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(Vh + o));
    }
  }
  // The call descriptor (row count, cache position) is written by kernels that have finished before the first kernel of a
  // pass starts (the head of the pass before, or a set-up kernel; that first kernel is a plain launch), never by a kernel
  // of the pass that this one may overlap: it is read before the dependency wait, and with it the cached keys and values (rows below the
  // cache position, written by earlier passes; a second chunk of a block is launched only when the first chunk's rows
  // of this layer are complete) and the bias by distance.
  const int k = ONE ? 1 : min(a.desc->k, a.mb), pos0 = a.desc->pos0;
  if (self) {
    n_keys = min(pos0 + k, a.cap);
    red = n_keys <= a.red_keys;
    j0 = red ? 0 : (r * n_keys) >> c_shift; j1 = red ? n_keys : ((r + 1) * n_keys) >> c_shift;
    if (!a.L.kv_late) stage_cached(j0, min(min(j1, pos0), j0 + a.kc_keys));
  }
  if (tid == 0) {   // what the exchanges bring: the head's q | k | v of every row, one record per rank and row
    mbar_expect(smem_u32(&sh->xbar[0]), (uint32_t)(R * k * 4));
    if (!red) mbar_expect(smem_u32(&sh->xbar[1]), (uint32_t)(C * k * recst * 4));
  }
  // relative-position bias of the distances this rank meets
  const int dist_lo = max(0, pos0 - (j1 - 1));
  const int bias_cnt = self ? min(pos0 + k - j0 - dist_lo, a.bias_len) : 0;
#pragma unroll 1
  for (int i = tid; i < bias_cnt; i += SUB_THREADS) sBias[i] = __ldg(a.bias + (size_t)h * a.bias_ld + dist_lo + i);
  SubRows<ONE> rw;
  if (a.emb) sub_rows_embed<ONE>(a.emb, a.tokens, a.vocab, k, d, col, on, rw);   // (tokens: part of the descriptor; the table: weights)
  __syncwarp();
  sub_cluster_arrive_relaxed();   // (0) this block is up: its shared memory may be written by the cluster
  SUB_STAMP();            // 0: requests
  // the weight rows become operands (two 16-row tiles in registers), then the keys may take their place
  const int mt = (npr + 15) >> 4;
  // (24 rows: 3 d_kv / 8 for d_kv = 64.  Half tiles, not whole ones: with 16 registers more the block variant spilled, and every pass of a
  // block was slower for it: T5-large, 5 rows, 539 -> 517 us, 16 rows 824 -> 753; mT5-large, 4 to 5 rows, 637 -> 579)
  uint4 hf[3][4];
  sub_wait(sh, a.err, &sh->wbar, 0, a.spin);
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (i * 8 < npr) sub_frags8(sWq, wst, npr, d, i, col0, nch, lane, hf[i]);
  if (a.L.kv_late) {
    __syncthreads();
    stage_cached(j0, min(min(j1, pos0), j0 + a.kc_keys));
  }
  if (WIDE && j1 - j0 > a.kc_main) {   // the last keys of the first chunk
    __syncthreads();
    stage_cached(j0, min(j1, j0 + a.kc_keys), a.kc_main);
  }
  SUB_STAMP();            // 1: weights in registers
  pdl_wait();
  SUB_STAMP();            // 2: dependency wait
  if (!a.emb) sub_rows_issue<ONE>(a.x_in, k, d, col, on, rw);
  {   // clear the buffer the next kernel accumulates into
    const int n4 = k * (d >> 2);
#pragma unroll 1
    for (int i = blockIdx.x * SUB_THREADS + tid; i < n4; i += gridDim.x * SUB_THREADS)
      reinterpret_cast<float4*>(a.x_zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  sub_rows_split<ONE>(rw, k, col, stores, on, g4, Xs, xst, sh, sSeed, h == 0 ? o0 : 0, h == 0 ? o0 + no : 0, lane, warp);
  if (!a.early) pdl_launch_dependents();
  SUB_STAMP();            // 3: token rows
  const int pst = sub_pst(npr, WIDE);
  // ---- phase A: this rank's q|k|v rows for all token rows -----------------------------------
  {
    SubB<ONE> b;
    sub_bfrags<ONE>(Xs, xst, k, col0, nch, lane, b);
    sub_tile<ONE, WIDE>(hf[0], hf[1], !WIDE && npr > 8, b, nch, npr, 0, psum, warp, lane);
    if (!WIDE && mt > 1) {   // (rows 24 and up: heads over fewer than eight blocks; never with kv_late)
      if (npr > 24) sub_frags8(sWq, wst, npr, d, 3, col0, nch, lane, hf[0]);
      sub_tile<ONE>(hf[2], hf[0], npr > 24, b, nch, npr, 1, psum, warp, lane);
    }
    if (!WIDE && mt > 2) {
      sub_frags8(sWq, wst, npr, d, 4, col0, nch, lane, hf[0]);
      if (npr > 40) sub_frags8(sWq, wst, npr, d, 5, col0, nch, lane, hf[1]);
      sub_tile<ONE>(hf[0], hf[1], npr > 40, b, nch, npr, 2, psum, warp, lane);
    }
  }
  sub_cp_wait();          // (first chunk of keys / values)
  __syncthreads();
  SUB_STAMP();            // 4: q|k|v products
  sub_cluster_wait();     // (0) every block of the cluster is up
  if (!ONE && ((npr | pr0) & 3) == 0 && npr <= 32) {   // warp <-> token row: values in lanes, then four at a time to every rank
    const int m = warp, n4 = npr >> 2, tot = n4 << c_shift;
    if (m < k) {
      float v = 0.f;
      if (lane < npr) {
        v = sub_total<ONE>(psum, lane, m, pst) * sub_inv(sh, m, a.inv_d, a.eps);
        const int j = pr0 + lane;
        if (self && j >= dkv && pos0 + m < a.cap)
          (j < 2 * dkv ? a.kc : a.vc)[((size_t)h * a.cap + pos0 + m) * dkv + (j & (dkv - 1))] = v;
      }
#pragma unroll 1
      for (int i0 = 0; i0 < tot; i0 += 32) {
        const int i = i0 + lane, q = i >> c_shift, rk = i & (C - 1);
        float4 o;
        o.x = __shfl_sync(0xffffffffu, v, (4 * q) & 31); o.y = __shfl_sync(0xffffffffu, v, (4 * q + 1) & 31);
        o.z = __shfl_sync(0xffffffffu, v, (4 * q + 2) & 31); o.w = __shfl_sync(0xffffffffu, v, (4 * q + 3) & 31);
        if (i < tot) sub_push4(sQKV + (size_t)m * qst + pr0 + 4 * q, &sh->xbar[0], (uint32_t)rk, o);
      }
    }
  } else {   // one (value, destination rank) pair per thread and turn
    const int tot = (npr * k) << c_shift;
#pragma unroll 1
    for (int idx = tid; idx < tot; idx += SUB_THREADS) {
      const int rk = idx & (C - 1), rest = idx >> c_shift, m = ONE ? 0 : rest / npr, i = rest - m * npr;
      const float v = sub_total<ONE>(psum, i, m, pst) * sub_inv(sh, m, a.inv_d, a.eps);
      const int j = pr0 + i;
      sub_push(sQKV + (size_t)m * qst + j, &sh->xbar[0], (uint32_t)rk, v);
      if (self && rk == r && j >= dkv && pos0 + m < a.cap)
        (j < 2 * dkv ? a.kc : a.vc)[((size_t)h * a.cap + pos0 + m) * dkv + (j & (dkv - 1))] = v;
    }
  }
  SUB_STAMP();            // 5: exchange stores
  sub_wait_exchange(sh, a.err, &sh->xbar[0], a.spin);   // q, new keys and new values of the head are complete
  SUB_STAMP();            // 6: exchange 1
  // ---- phase B: attention of the k rows over the keys [j0, j1), every warp on keys of its own -----------------
  constexpr int MBC = ONE ? 1 : SUB_MB;
  const int og_k = min(og, k - 1);
  SubAtt1 s1;
  SubAtt8 s8;
  float4 q1[4];
  SubQ8 q8;
  if (ONE) {
    s1.run = -INFINITY; s1.sum = 0.f; s1.acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u * 16 < dkv) q1[u] = *reinterpret_cast<const float4*>(sQKV + (u * 4 + ot) * 4);
  } else {
    s8.run = -INFINITY; s8.sum = 0.f;
#pragma unroll
    for (int n = 0; n < 8; ++n) { s8.o[n][0] = 0.f; s8.o[n][1] = 0.f; s8.o[n][2] = 0.f; s8.o[n][3] = 0.f; }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i * 16 < dkv) {
        float4 q4 = *reinterpret_cast<const float4*>(sQKV + (size_t)og_k * qst + i * 16 + 4 * ot);
        if (og >= k) q4 = make_float4(0.f, 0.f, 0.f, 0.f);
        sub_split(q4.x, q4.y, q8.h[i][0], q8.l[i][0]);
        sub_split(q4.z, q4.w, q8.h[i][1], q8.l[i][1]);
      }
  }
#pragma unroll 1
  for (int c0 = j0; c0 < j1; c0 += a.kc_keys) {
    const int c1 = min(j1, c0 + a.kc_keys), nk = c1 - c0;
    if (c0 > j0) {   // later chunks: staged now (the first one is on its way since the prologue)
      __syncthreads();
      stage_cached(c0, self ? min(c1, pos0) : c1);
      sub_cp_wait();
      __syncthreads();
    }
    // keys of this pass come from the exchange buffer
    const int own0 = self ? pos0 - c0 : nk;
    auto kp = [&](int j) { return j >= own0 ? sQKV + (size_t)(j - own0) * qst + dkv : k_at(j); };
    auto vp = [&](int j) { return j >= own0 ? sQKV + (size_t)(j - own0) * qst + 2 * dkv : v_at(j); };
    if (ONE) sub_attend_one(q1, dkv >> 4, dkv, nk, kp, vp, sBias, pos0 - c0 - dist_lo, self, s1, warp, lane);
    else sub_attend_block(q8, dkv, nk, kp, vp, sBias, pos0 + og - c0 - dist_lo, self, self ? min(nk - 1, pos0 + og_k - c0) : nk - 1, s8, warp, lane);
  }
  // the warp's record of every row: max, sum, weighted values
  if (ONE) {
    float l = s1.sum;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    float* rp = sRec + (size_t)warp * recst;
    if (lane == 0) *reinterpret_cast<float4*>(rp) = make_float4(s1.run, l, 0.f, 0.f);
    if (dkv >= 64) *reinterpret_cast<float2*>(rp + SUB_RECPAD + 2 * lane) = s1.acc;
    else if (lane < dkv) rp[SUB_RECPAD + lane] = s1.acc.x;
  } else {
    float l = s8.sum;
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    if (og < k) {
      float* rp = sRec + (size_t)(warp * MBC + og) * recst;
      if (ot == 0) *reinterpret_cast<float4*>(rp) = make_float4(s8.run, l, 0.f, 0.f);
      rp += SUB_RECPAD;
      if (dkv == 16) {
        *reinterpret_cast<float4*>(rp + 4 * ot) = make_float4(s8.o[0][0], s8.o[1][0], s8.o[0][1], s8.o[1][1]);
      } else {
#pragma unroll
        for (int n4 = 0; n4 < 2; ++n4)
          if (n4 * 32 < dkv) {
            *reinterpret_cast<float4*>(rp + n4 * 32 + 8 * ot) = make_float4(s8.o[4 * n4][0], s8.o[4 * n4 + 1][0], s8.o[4 * n4 + 2][0], s8.o[4 * n4 + 3][0]);
            *reinterpret_cast<float4*>(rp + n4 * 32 + 8 * ot + 4) = make_float4(s8.o[4 * n4][1], s8.o[4 * n4 + 1][1], s8.o[4 * n4 + 2][1], s8.o[4 * n4 + 3][1]);
          }
      }
    }
  }
  __syncthreads();
  SUB_STAMP();            // 7: attention over this rank's keys
  const float* rec = sRec;
  int nrec = 8;
  if (!red) {   // the ranks hold different keys: the block's merged records go to every rank
    const int nu = 1 + (dkv >> 2);   // 16-byte pieces of a record
    float sum;
    if (ONE) {
#pragma unroll 1
      for (int idx = tid; idx < nu << c_shift; idx += SUB_THREADS) {
        const int rk = idx & (C - 1), u = idx >> c_shift;
        sub_push4(sRrec + (size_t)r * recst + 4 * u, &sh->xbar[1], (uint32_t)rk, sub_merge(sRec, recst, 8, u - 1, sum));
      }
    } else {
#pragma unroll 1
      for (int m = warp; m < k; m += SUB_THREADS / 32)
        if (lane < nu) {
          const float4 v = sub_merge(sRec + (size_t)m * recst, MBC * recst, 8, lane - 1, sum);
#pragma unroll 1
          for (int rk = 0; rk < C; ++rk) sub_push4(sRrec + (size_t)(r * MBC + m) * recst + 4 * lane, &sh->xbar[1], (uint32_t)rk, v);
        }
    }
    SUB_STAMP();          // 8: records merged and sent
    sub_wait_exchange(sh, a.err, &sh->xbar[1], a.spin);
    rec = sRrec; nrec = C;
    SUB_STAMP();          // 9: exchange 2
  } else {
    SUB_STAMP(); SUB_STAMP();
  }
  // ---- phase C: this rank's rows of the output projection ---------------
  if (ONE) {
    // one row: the up to eight records are the columns of the right operand, each scaled by its weight in the merged soft-max
    // (fp32 as three bf16 parts); the sum over the columns is the output
    const float* rg = rec + (size_t)min(og, nrec - 1) * recst;
    const float2 ml = *reinterpret_cast<const float2*>(rg);
    float gm = og < nrec ? ml.x : -INFINITY;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    const float w = og < nrec && ml.y > 0.f ? __expf(ml.x - gm) : 0.f;
    float den = w * ml.y;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    const float sc = w * sub_rcp(den);
    float c[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f}, f[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int st = 0; st < 4; ++st)
      if (st * 16 < dkv) {
        float4 v = *reinterpret_cast<const float4*>(rg + SUB_RECPAD + ot * cpt + 4 * st);
        if (!(sc > 0.f)) v = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t h0, h1, m0, m1, l0, l1;
        sub_split3(v.x * sc, v.y * sc, h0, m0, l0);
        sub_split3(v.z * sc, v.w * sc, h1, m1, l1);
        sub_mma(c, wr[0][2 * st], wr[1][2 * st], wr[0][2 * st + 1], wr[1][2 * st + 1], h0, h1);
        sub_mma(e, wr[0][2 * st], wr[1][2 * st], wr[0][2 * st + 1], wr[1][2 * st + 1], m0, m1);
        sub_mma(f, wr[0][2 * st], wr[1][2 * st], wr[0][2 * st + 1], wr[1][2 * st + 1], l0, l1);
      }
    // accumulators: rows g and g + 8 of the tile, columns 2 t and 2 t + 1
    float v0 = (c[0] + c[1]) + ((e[0] + e[1]) + (f[0] + f[1])), v1 = (c[2] + c[3]) + ((e[2] + e[3]) + (f[2] + f[3]));
    v0 += __shfl_xor_sync(0xffffffffu, v0, 1); v1 += __shfl_xor_sync(0xffffffffu, v1, 1);
    v0 += __shfl_xor_sync(0xffffffffu, v0, 2); v1 += __shfl_xor_sync(0xffffffffu, v1, 2);
    const int row = warp * 16 + og + 8 * ot;
    if (ot < 2 && row < no) {
      const float v = ot ? v1 : v0;
      atomicAdd(a.x_out + o0 + row, h == 0 ? v + sSeed[row] : v);   // residual term once per column
    }
  } else {
    // merged head output of every row, then rows of W_o x token rows on mma.sync m16n8k16 (the right operand: each value as a
    // bf16 head and a bf16 remainder), 16 channels per step
    const int ast = dkv + 4;
#pragma unroll 1
    for (int idx = tid; idx < k << (dkv_shift - 2); idx += SUB_THREADS) {
      const int m = idx >> (dkv_shift - 2), u = idx & ((dkv >> 2) - 1);
      float sum;
      float4 v = sub_merge(rec + (size_t)m * recst, MBC * recst, nrec, u, sum);
      const float is = sub_rcp(sum);
      *reinterpret_cast<float4*>(sA + (size_t)m * ast + 4 * u) = make_float4(v.x * is, v.y * is, v.z * is, v.w * is);
    }
    __syncthreads();
    SUB_STAMP();          // 10: merge
    float* sOut = reinterpret_cast<float*>(sub_smem + a.L.out);
    const int ost = no + 4;
    if (warp * 16 < no) {
      float c[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};   // (heads | remainders: two chains)
#pragma unroll
      for (int st = 0; st < 4; ++st)
        if (st * 16 < dkv) {
          float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
          if (og < k) b4 = *reinterpret_cast<const float4*>(sA + (size_t)og * ast + ot * cpt + 4 * st);
          uint32_t h0, h1, l0, l1;
          sub_split(b4.x, b4.y, h0, l0); sub_split(b4.z, b4.w, h1, l1);
          sub_mma(c, wr[0][2 * st], wr[1][2 * st], wr[0][2 * st + 1], wr[1][2 * st + 1], h0, h1);
          sub_mma(e, wr[0][2 * st], wr[1][2 * st], wr[0][2 * st + 1], wr[1][2 * st + 1], l0, l1);
        }
#pragma unroll
      for (int i = 0; i < 4; ++i) c[i] += e[i];
      // accumulators: rows g and g + 8 of the tile, token rows 2 t and 2 t + 1
      const int row = warp * 16 + og;
      if (row < no) { sOut[(size_t)(2 * ot) * ost + row] = c[0]; sOut[(size_t)(2 * ot + 1) * ost + row] = c[1]; }
      if (row + 8 < no) { sOut[(size_t)(2 * ot) * ost + row + 8] = c[2]; sOut[(size_t)(2 * ot + 1) * ost + row + 8] = c[3]; }
    }
    __syncthreads();
    const int n4 = no >> 2;
#pragma unroll 1
    for (int idx = tid; idx < k * n4; idx += SUB_THREADS) {   // added four columns at a time
      const int m = idx / n4, q = idx - m * n4;
      float4 v = *reinterpret_cast<const float4*>(sOut + (size_t)m * ost + q * 4);
      if (h == 0) {   // residual term once per column
        const float4 xr = *reinterpret_cast<const float4*>(sSeed + (size_t)m * no + q * 4);
        v.x += xr.x; v.y += xr.y; v.z += xr.z; v.w += xr.w;
      }
      asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a.x_out + (size_t)m * d + o0 + q * 4), "f"(v.x), "f"(v.y), "f"(v.z),
                   "f"(v.w) : "memory");
    }
  }
  SUB_STAMP();            // 11: output projection + reductions issued
  SUB_STAMP_END(self ? 0 : 1);
}

// ------------------------------------------------------------------------------------------------
// Feed-forward sub-layer
// ------------------------------------------------------------------------------------------------
// W_fo [d][F] in the order the feed-forward kernels load it, in units of 8 columns (16 bytes of a row).  Unit u holds
//   one: [i < 4][tid < d / 4]            the piece of row 4 tid + i                  (d pieces)
//   blk: [i][rr < 2][w < 8][g < 8]       the piece of row (w + 8 i) 16 + g + 8 rr    (pack_wfo_dpad(d) pieces, zero past d)
// so that the threads of a warp read neighbouring pieces.  Built once, when the context is created.
__host__ __device__ inline int pack_wfo_dpad(int d) { return (d + 127) / 128 * 128; }
__global__ void pack_wfo_kernel(const __nv_bfloat16* __restrict__ W, uint4* __restrict__ one, uint4* __restrict__ blk, int d, int F) {
  const int u = blockIdx.x, d4 = d >> 2, dpad = pack_wfo_dpad(d);
  for (int p = threadIdx.x; p < d; p += blockDim.x) {
    const int i = p / d4, tt = p - i * d4;
    one[(size_t)u * d + p] = *reinterpret_cast<const uint4*>(W + (size_t)(4 * tt + i) * F + 8 * u);
  }
  for (int p = threadIdx.x; p < dpad; p += blockDim.x) {
    const int g = p & 7, w = (p >> 3) & 7, rr = (p >> 6) & 1, i = p >> 7, n = (w + 8 * i) * 16 + g + 8 * rr;
    blk[(size_t)u * dpad + p] = n < d ? *reinterpret_cast<const uint4*>(W + (size_t)n * F + 8 * u) : make_uint4(0u, 0u, 0u, 0u);
  }
}

struct FfnSubLayout { int wi, wi2, xs, psum, u, seed, sh, total; };

struct FfnSubArgs {
  const CallDesc* desc;
  const float* x_in;
  float* x_out;
  float* x_zero;             // nullptr: nothing to clear (second part of a split launch)
  const float* gain;
  float eps, inv_d;          // inv_d: 1 / d
  const __nv_bfloat16* Wi0;  // [F][d]
  const __nv_bfloat16* Wi1;  // [F][d] gate matrix (gated GELU) or nullptr
  const uint4* Wfo1;         // W_fo in the load order of the single-row variant (pack_wfo_kernel)
  const uint4* Wfo8;         // ... and of the block variant
  int d, F, gated;
  int part, nparts;          // this launch covers the slices blockIdx.x * nparts + part of gridDim.x * nparts
  int early;                 // when the next kernel may start: 2 ahead of this one's dependency wait, 1 behind it, 0 once this kernel has its token rows
  int seed;                  // 1: the blocks add x_in for their share of the columns
  int mb;
  unsigned spin;             // polls of the weight barrier before the kernel gives up
  int* err;
  FfnSubLayout L;
  HeadAhead ahead;           // AHEAD
};

// most rows of a slice when F (a multiple of 8) is dealt out in units of 8 rows
inline int ffn_sub_rows(int F, int slices) { return 8 * ((F / 8 + slices - 1) / slices); }
inline FfnSubLayout ffn_sub_layout(int d, int F, int gated, int slices, int grid, int mb) {
  FfnSubLayout L;
  const int nf = ffn_sub_rows(F, slices), nmat = gated ? 2 : 1;
  int off = 0;
  // weight rows of W_i (and the gate); once they wait in registers (the first 32), the slice's units of W_fo take their place
  const int fo_b = nf / 8 * (pack_wfo_dpad(d) * 16 + 32);
  L.wi = off; L.wi2 = sub_up16(std::max(std::min(nf * nmat, 32) * sub_wst(d), fo_b)); off += L.wi2 + sub_up16(std::max(nf * nmat - 32, 0) * sub_wst(d));
  L.xs = off; off += std::max(sub_up16(sub_xs_bytes(d, mb)), mb == 1 ? 0 : sub_up16(mb * (d + 4) * 4));   // token rows; later the block variant's output tile
  L.psum = off; off += sub_up16(sub_psum_bytes(nf * nmat, mb));
  L.u = off; off += sub_up16(mb * (SUB_FO_REGS + 4) * 4);
  L.seed = off; off += sub_up16(mb * 4 * ((d / 4 + grid - 1) / grid + 1) * 4);
  L.sh = off; off += sub_up16((int)sizeof(SubShared));
  L.total = off;
  return L;
}

// Bound as the attention kernels by its dependent chain: token rows, products, activation, output products, reductions at the L2
// (every block adds a partial sum to every output: 148 additions per address).  Times: see attn_sub_kernel.
template <bool ONE, bool AHEAD = false, int DQ = 0>
__global__ void __launch_bounds__(SUB_THREADS, 2) ffn_sub_kernel(const FfnSubArgs a) {
  extern __shared__ __align__(1024) unsigned char sub_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int d = DQ ? 256 * DQ : a.d, F = a.F, G = gridDim.x, S = G * a.nparts, s = blockIdx.x * a.nparts + a.part;
  const int f0 = 8 * (int)(((long long)s * (F >> 3)) / S), f1 = 8 * (int)(((long long)(s + 1) * (F >> 3)) / S), nf = f1 - f0;
  const int nmat = a.gated ? 2 : 1, nrows = nf * nmat;
  const int wst = sub_wst(d), xst = sub_xst(d);
  unsigned char* sWi = sub_smem + a.L.wi;
  unsigned char* sWi2 = sWi + a.L.wi2 - 32 * wst;   // rows 32 and up
  uint32_t* Xs = reinterpret_cast<uint32_t*>(sub_smem + a.L.xs);
  float* psum = reinterpret_cast<float*>(sub_smem + a.L.psum);
  float* sU = reinterpret_cast<float*>(sub_smem + a.L.u);
  float* sSeed = reinterpret_cast<float*>(sub_smem + a.L.seed);
  SubShared* sh = reinterpret_cast<SubShared*>(sub_smem + a.L.sh);
  constexpr int ust = SUB_FO_REGS + 4;
  const int cpw = sub_chunks(d), col0 = warp * 32 * cpw, nch = DQ ? cpw : max(0, min(cpw, (d - col0 + 31) >> 5));
  const int col = col0 + lane * 4;
  const bool stores = lane * 4 < 32 * nch, on = stores && (DQ || col < d);   // this lane's four columns of the token rows
  // columns whose residual term this block adds: units of four columns, spread over the grid
  const int d4 = d >> 2;
  const int su0 = a.seed ? (int)(((long long)blockIdx.x * d4) / G) : 0, su1 = a.seed ? (int)(((long long)(blockIdx.x + 1) * d4) / G) : 0;
  SUB_STAMP_BEGIN();

  if (tid == 0) {
    mbar_init(smem_u32(&sh->wbar), 1);
    sh->failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect(smem_u32(&sh->wbar), (uint32_t)(nrows * d * 2));
  }
  __syncthreads();
  {   // row i is copied by lane i / 8 of warp i % 8 (the copies of one warp are issued one after the other)
    const int i = ((tid & 31) << 3) | (tid >> 5);
    if (i < nrows) {
      const __nv_bfloat16* W = i < nf ? a.Wi0 : a.Wi1;
      const int rr = i < nf ? i : i - nf;
      bulk_g2s(smem_u32(i < 32 ? sWi + (size_t)i * wst : sWi2 + (size_t)i * wst), W + (size_t)(f0 + rr) * d, (uint32_t)(d * 2), smem_u32(&sh->wbar));
    }
  }
  if (AHEAD && tid == SUB_THREADS - 1) head_ahead(a.ahead);
  float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (on) g4 = __ldg(reinterpret_cast<const float4*>(a.gain + col));
  const int k = ONE ? 1 : min(a.desc->k, a.mb);   // (written before the pass began: see the attention kernel)
  SUB_STAMP();            // 0: requests
  // The rows of W_i become operands in registers; then the block's columns [f0, f1) of W_fo are fetched into their place, as units of
  // 8 columns from the copies of W_fo that pack_wfo_kernel lays out (8 columns of a row in place are 16 bytes every 2 F bytes: a
  // fraction of the memory's rate).  Both by bulk copies: 64 KB a block through the load units held up the shared-memory
  // accesses of the kernel in front on the same SM (5-row pass 594 -> 551 us without them).
  const int ust_fo = (ONE ? d : pack_wfo_dpad(d)) * 16 + 32;   // bytes from unit to unit: the lanes (row g, unit t) hit 32 banks
  uint4 fr[4][4];
  if (nf > 0) {
    sub_wait(sh, a.err, &sh->wbar, 0, a.spin);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i * 8 < nrows) sub_frags8(sWi, wst, nrows, d, i, col0, nch, lane, fr[i]);
    __syncthreads();
    const uint32_t ub = (uint32_t)(ust_fo - 32);
    if (tid == 0) mbar_expect(smem_u32(&sh->wbar), ub * (uint32_t)(nf >> 3));
    if (tid < (nf >> 3)) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_g2s(smem_u32(sWi + (size_t)tid * ust_fo), reinterpret_cast<const unsigned char*>(ONE ? a.Wfo1 : a.Wfo8) + (size_t)((f0 >> 3) + tid) * ub, ub,
               smem_u32(&sh->wbar));
    }
  }
  SUB_STAMP();            // 1: weights
  if (a.early == 2) pdl_launch_dependents();
  pdl_wait();
  if (a.early == 1) pdl_launch_dependents();
  SUB_STAMP();            // 2: dependency wait
  SubRows<ONE> rw;
  sub_rows_issue<ONE>(a.x_in, k, d, col, on, rw);
  if (a.x_zero) {
    const int n4 = k * d4;
#pragma unroll 1
    for (int i = blockIdx.x * SUB_THREADS + tid; i < n4; i += G * SUB_THREADS)
      reinterpret_cast<float4*>(a.x_zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  sub_rows_split<ONE>(rw, k, col, stores, on, g4, Xs, xst, sh, sSeed, su0 * 4, su1 * 4, lane, warp);
  if (!a.early) pdl_launch_dependents();
  SUB_STAMP();            // 3: token rows
  if (nf > 0) {   // hidden activations of the slice
    SubB<ONE> b;
    sub_bfrags<ONE>(Xs, xst, k, col0, nch, lane, b);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (i * 16 < nrows) sub_tile<ONE>(fr[2 * i], fr[2 * i + 1], i * 16 + 8 < nrows, b, nch, nrows, i, psum, warp, lane);
    if (nrows > 32) {
      sub_frags8(sWi2, wst, nrows, d, 4, col0, nch, lane, fr[0]);
      if (nrows > 40) sub_frags8(sWi2, wst, nrows, d, 5, col0, nch, lane, fr[1]);
      sub_tile<ONE>(fr[0], fr[1], nrows > 40, b, nch, nrows, 2, psum, warp, lane);
    }
  }
  // W_fo into registers while the sums go round.  ONE: thread <-> the four output rows 4 tid .. 4 tid + 3, chunk q = columns 8 q .. 8 q + 7.
  // Block variant: warp w owns the output tiles w, w + 8, ... (16 rows each); thread (g, t) takes, of rows g and g + 8 of a tile, the
  // columns 8 t .. 8 t + 7: read as the left operand of mma.sync m16n8k16 they are two steps of 16 slice rows, with the slice rows
  // dealt to the steps' positions so that one 16-byte load fills them (the right operand, the hidden activations, follows the same order).
  uint4 wf[8][2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) wf[i][j] = make_uint4(0u, 0u, 0u, 0u);
  if (nf > 0) sub_wait(sh, a.err, &sh->wbar, 1, a.spin);
  if (ONE) {
    if (tid * 4 < d) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (8 * q < nf) {
          const uint4* p = reinterpret_cast<const uint4*>(sWi + (size_t)q * ust_fo) + tid;
#pragma unroll
          for (int i = 0; i < 4; ++i) wf[i * 2 + (q >> 1)][q & 1] = p[i * (d >> 2)];
        }
    }
  } else {
    const int g = lane >> 2, t = lane & 3;
    if (8 * t < nf) {
      const uint4* p = reinterpret_cast<const uint4*>(sWi + (size_t)t * ust_fo) + warp * 8 + g;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((warp + 8 * i) * 16 < d) {
          wf[i][0] = p[i * 128]; wf[i][1] = p[i * 128 + 64];
        }
    }
  }
  __syncthreads();
  SUB_STAMP();            // 4: products
  const int pst = sub_pst(nrows);
  if (ONE) {
    if (tid < nf) {
      const float inv = sub_inv(sh, 0, a.inv_d, a.eps), v0 = sub_total<true>(psum, tid, 0, pst) * inv;
      sU[tid] = a.gated ? gelu_tanh(v0) * (sub_total<true>(psum, nf + tid, 0, pst) * inv) : fmaxf(v0, 0.f);
    }
  } else {   // warp <-> token row, lane <-> slice row of the 8 x 32 tile the output products read; what lies outside is zero
    float uv = 0.f;
    if (warp < k && lane < nf) {
      const float inv = sub_inv(sh, warp, a.inv_d, a.eps), v0 = sub_total<false>(psum, lane, warp, pst) * inv;
      uv = a.gated ? gelu_tanh(v0) * (sub_total<false>(psum, nf + lane, warp, pst) * inv) : fmaxf(v0, 0.f);
    }
    sU[(size_t)warp * ust + lane] = uv;
  }
  __syncthreads();
  SUB_STAMP();            // 5: hidden activations
  if (ONE) {
    // this slice's share of all d outputs: thread <-> four output rows, their columns of W_fo from its registers
    if (tid < d4) {
      const bool seeds = tid >= su0 && tid < su1;
      float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (8 * q < nf) {
          const float4 u0 = *reinterpret_cast<const float4*>(sU + 8 * q), u1 = *reinterpret_cast<const float4*>(sU + 8 * q + 4);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 w = wf[i * 2 + (q >> 1)][q & 1];
            o[i] += __uint_as_float(w.x << 16) * u0.x + __uint_as_float(w.x & 0xffff0000u) * u0.y + __uint_as_float(w.y << 16) * u0.z +
                    __uint_as_float(w.y & 0xffff0000u) * u0.w + __uint_as_float(w.z << 16) * u1.x + __uint_as_float(w.z & 0xffff0000u) * u1.y +
                    __uint_as_float(w.w << 16) * u1.z + __uint_as_float(w.w & 0xffff0000u) * u1.w;
          }
        }
      if (seeds) {
        const float4 xr = *reinterpret_cast<const float4*>(sSeed + (tid - su0) * 4);
        o[0] += xr.x; o[1] += xr.y; o[2] += xr.z; o[3] += xr.w;
      }
      if (nf > 0 || seeds)
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a.x_out + tid * 4), "f"(o[0]), "f"(o[1]), "f"(o[2]), "f"(o[3]) : "memory");
    }
  } else {
    // out[column][token] = sum_i W_fo[column][f0 + i] * u[token][i] on mma.sync m16n8k16: 16 output columns are the rows of
    // the left operand (from the registers), the token rows the columns of the right one, each activation as a bf16 head and
    // a bf16 remainder.  Step s of thread (g, t) covers the slice rows 8 t + 4 s .. 8 t + 4 s + 3.
    const int g = lane >> 2, t = lane & 3;
    uint32_t bh[2][2], bl[2][2];
#pragma unroll
    for (int st = 0; st < 2; ++st) {
      const float4 u4 = *reinterpret_cast<const float4*>(sU + (size_t)g * ust + 8 * t + 4 * st);
      bh[st][0] = sl_pack_bf16(u4.x, u4.y); bh[st][1] = sl_pack_bf16(u4.z, u4.w);
      bl[st][0] = sl_pack_bf16(u4.x - __uint_as_float(bh[st][0] << 16), u4.y - __uint_as_float(bh[st][0] & 0xffff0000u));
      bl[st][1] = sl_pack_bf16(u4.z - __uint_as_float(bh[st][1] << 16), u4.w - __uint_as_float(bh[st][1] & 0xffff0000u));
    }
    float* sOut = reinterpret_cast<float*>(Xs);   // [token][column]: the token rows are done with
    const int ost = d + 4;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int n0 = (warp + 8 * i) * 16;
      if (n0 < d) {
        float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
#define SUB_MMA(A0, A1, A2, A3, B0, B1)                                                                                          \
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};" \
                     : "+f"(c0), "+f"(c1), "+f"(c2), "+f"(c3) : "r"(A0), "r"(A1), "r"(A2), "r"(A3), "r"(B0), "r"(B1))
        SUB_MMA(wf[i][0].x, wf[i][1].x, wf[i][0].y, wf[i][1].y, bh[0][0], bh[0][1]);
        SUB_MMA(wf[i][0].x, wf[i][1].x, wf[i][0].y, wf[i][1].y, bl[0][0], bl[0][1]);
        SUB_MMA(wf[i][0].z, wf[i][1].z, wf[i][0].w, wf[i][1].w, bh[1][0], bh[1][1]);
        SUB_MMA(wf[i][0].z, wf[i][1].z, wf[i][0].w, wf[i][1].w, bl[1][0], bl[1][1]);
#undef SUB_MMA
        // accumulators: columns n0 + g and n0 + g + 8, token rows 2 t and 2 t + 1
        sOut[(size_t)(2 * t) * ost + n0 + g] = c0; sOut[(size_t)(2 * t + 1) * ost + n0 + g] = c1;
        sOut[(size_t)(2 * t) * ost + n0 + g + 8] = c2; sOut[(size_t)(2 * t + 1) * ost + n0 + g + 8] = c3;
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int un = tid; un < d4; un += SUB_THREADS)   // added four columns at a time
#pragma unroll 2   // (two rows' reads side by side: blocks of 16 rows 757 -> 749 us)
    for (int m = 0; m < k; ++m) {
      const bool seeds = un >= su0 && un < su1;
      if (nf > 0 || seeds) {
        float4 v = *reinterpret_cast<const float4*>(sOut + (size_t)m * ost + un * 4);
        if (seeds) {
          const float4 xr = *reinterpret_cast<const float4*>(sSeed + (size_t)m * (su1 - su0) * 4 + (un - su0) * 4);
          v.x += xr.x; v.y += xr.y; v.z += xr.z; v.w += xr.w;
        }
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a.x_out + (size_t)m * d + un * 4), "f"(v.x), "f"(v.y), "f"(v.z),
                     "f"(v.w) : "memory");
      }
    }
  }
  SUB_STAMP();            // 6: output products + reductions issued
  SUB_STAMP_END(2);
}

}  // namespace bild
