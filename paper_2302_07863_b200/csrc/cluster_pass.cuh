// All layers of a decoder pass of a small fp32 model (d_model <= 256, at most 2 MB a layer) in one kernel: a single cluster of eight
// blocks goes through the layers, the residual stream kept in every block's shared memory, the blocks' partial sums exchanged through
// distributed shared memory (steps S0-S8 / L0-L8; the LM head follows as a kernel of its own).
//   * self- and cross-attention: block c takes the heads c, c + 8, ...: its rows of q | k | v, the attention of all token rows, and the
//     head's columns of W_o, i.e. a partial sum of all d outputs;
//   * feed-forward: block c takes a slice of d_ff (units of 8 rows): hidden activations and the slice's columns of W_fo, again a
//     partial sum of all d outputs;
//   * behind each sub-layer every block sends its partial sums to all eight (asynchronous stores that the receiver's mbarrier counts)
//     and adds what it received to its copy of the residual stream, in block order: three exchanges a layer, no other traffic;
//   * the operands of the next sub-layer (gain, weights, cached keys and values) arrive by bulk copies while this one is computed.
// Such a layer is a few thousand multiply-adds per token row: a pass is bound by the latency of its instruction stream and of the
// kernels in a row (eight a layer with one kernel per operation), not by bytes.  Eight blocks: the portable cluster size, and the
// heads and slices of such models do not fill more.  Measured against one kernel per operation, 4 layers of 128 columns, 4 heads, d_ff
// 512, passes with LM head: 1 row 72 -> 53 us, 2 rows 137 -> 72, 5 rows 158 -> 90, 8 rows 177 -> 98; 2 layers of 64 columns, 1 row 39 -> 29.
// bf16 models of this size stay on the sub-layer kernels, whose tensor-core tiles are faster still (3 layers of 128 columns, 5 rows:
// 55 us there, 82 us with this kernel on bf16 weights).
// Sums run in a fixed order, so results do not depend on timing.
#pragma once
#include "sublayer.cuh"

namespace bild {

constexpr int CP_THREADS = 512, CP_WARPS = CP_THREADS / 32, CP_C = 8;

struct CPassArgs {
  const CallDesc* desc;           // rows and cache position (of a chunk, where a pass of 9 to 16 rows is cut in two)
  const int* tokens;              // this chunk's tokens
  const bild_dec_layer* layers;   // DEVICE array [n_layers]
  const void *wo_pack, *wfo_pack; // W_o [layer][self, cross][head][d][dkv] and W_fo [layer][block's slice][d][slice rows] (cp_pack_kernel)
  int n_layers, d, I, H, dkv, dkv_shift, F, gated, vocab;
  float eps, inv_d;
  const void* emb;
  float *selfK, *selfV;           // [layer][head][cap][dkv]
  const float *crossK, *crossV;   // [layer][head][ecap][dkv]
  int cap, ecap;
  const float* bias;              // [H][cap] by distance
  const int* n_keys_dev;          // encoder positions
  float* x_out;                   // [rows][d] residual stream behind the last layer
  int mb;                         // token rows the shared memory is sized for
  int kv_keys;                    // cached keys per head that are staged in shared memory (the others are read where they lie)
  unsigned spin;
  int* err;
};

inline int cp_slice_max(int F) { return 8 * ((F / 8 + CP_C - 1) / CP_C); }
// Bytes of the operands of one sub-layer as they wait in shared memory: gain, the head's (or slice's) weights, cached keys / values.
__host__ __device__ inline int cp_kv_stride(int dkv) { return dkv + 4; }   // floats: eight keys side by side hit 32 banks
struct CPassLayout { int tab, x, h, qkv, att, rec, u, ploc, recv, buf, buf_bytes, total; };
__host__ __device__ inline CPassLayout cp_layout(int d, int dkv, int fs, int gated, int wb, int mb, int layers, int kv_keys) {
  CPassLayout L;
  int off = 64;   // barrier, error flag
  L.tab = off; off += (layers * (int)sizeof(bild_dec_layer) + 15) & ~15;
  L.x = off; off += mb * d * 4;
  L.h = off; off += mb * d * 4;
  L.qkv = off; off += mb * 3 * dkv * 4;
  L.att = off; off += mb * dkv * 4;
  L.rec = off; off += CP_WARPS * (dkv + 4) * 4;
  L.u = off; off += mb * (fs + 8) * 4;
  L.ploc = off; off += mb * d * 4;
  L.recv = off; off += CP_C * mb * d * 4;
  const int attn = d * 4 + 4 * dkv * d * wb + 2 * kv_keys * cp_kv_stride(dkv) * 4, ffn = d * 4 + (2 + gated) * fs * d * wb;
  L.buf_bytes = ((attn > ffn ? attn : ffn) + 15) & ~15;
  L.buf = off; off += 2 * L.buf_bytes;   // the sub-layer at hand and the next one
  L.total = off;
  return L;
}

// out(i, m, sum over K of W[i][.] * X[m][.]) for all rows i < n and token rows m < k; W [n][K] and X [k][xst] in shared memory.  Eight
// lanes share a weight row (16 bytes each, neighbouring), the four groups of a warp take neighbouring rows, two each, and MR token rows at a
// time; then one transposed reduction over the eight lanes for all of them.  (Token rows past the last repeat it, nobody reads their sums.)
template <int MR, typename OutF>
__device__ __forceinline__ void cp_rows_t(const float* W, int n, int K, const float* X, int xst, int k, int warp, int lane, OutF out) {
  constexpr int N = 2 * MR;
  const int chunks = K >> 2, li = lane & 7, g = lane >> 3;
#pragma unroll 1
  for (int b0 = warp * 8; b0 < n; b0 += CP_WARPS * 8) {
#pragma unroll 1
    for (int m0 = 0; m0 < k; m0 += MR) {
      float acc[N];
#pragma unroll
      for (int i = 0; i < N; ++i) acc[i] = 0.f;
      const float* w0 = W + min(b0 + g, n - 1) * K;
      const float* w1 = W + min(b0 + 4 + g, n - 1) * K;
#pragma unroll 2
      for (int c = li; c < chunks; c += 8) {
        const float4 wa = *reinterpret_cast<const float4*>(w0 + 4 * c), wb = *reinterpret_cast<const float4*>(w1 + 4 * c);
#pragma unroll
        for (int m = 0; m < MR; ++m) {
          const float4 x = *reinterpret_cast<const float4*>(X + (MR == 1 ? 0 : min(m0 + m, k - 1) * xst) + 4 * c);
          acc[m] += wa.x * x.x + wa.y * x.y + wa.z * x.z + wa.w * x.w;
          acc[MR + m] += wb.x * x.x + wb.y * x.y + wb.z * x.z + wb.w * x.w;
        }
      }
      // lane bit b picks a half of what is left: the sum of value i + sum_b bit_b (N >> (b + 1)) ends up in acc[i]
      int at = 0;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int left = N >> b;
        if (left > 1) {
          const bool up = (lane >> b) & 1;
#pragma unroll
          for (int i = 0; i < left / 2; ++i) {
            const float send = up ? acc[i] : acc[i + left / 2], keep = up ? acc[i + left / 2] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1 << b);
          }
          at += up ? left / 2 : 0;
        } else {
          acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1 << b);
        }
      }
      constexpr int NV = N >= 8 ? N / 8 : 1;   // values a lane holds
      if (N >= 8 || li < N) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int v = at + i, m = m0 + (v & (MR - 1)), row = b0 + g + (v >= MR ? 4 : 0);
          if (row < n && m < k) out(row, m, acc[i]);
        }
      }
    }
  }
}
template <int MR, typename OutF>
__device__ __forceinline__ void cp_rows(const float* W, int n, int K, const float* X, int xst, int k, int warp, int lane, OutF out) {
  if (MR == 1) cp_rows_t<1>(W, n, K, X, xst, 1, warp, lane, out);
  else if (k <= 4) cp_rows_t<4>(W, n, K, X, xst, k, warp, lane, out);
  else cp_rows_t<8>(W, n, K, X, xst, k, warp, lane, out);
}

// Attention of the k token rows over one head: a row has up to 16 / (rows rounded up to a power of two) warps, each a share of the keys
// (at least 32); scores: lane <-> key; values: lane <-> (key of a group, four channels), so a step takes 128 / d_kv keys; the warps'
// records meet in shared memory.
// Keys below sn are staged (sk / sv, row stride kvst), up to own0 in the cache (K / V), from own0 on rows of this pass (kn / vn, row
// stride nst); bias: row m sees keys up to own0 + m, with bias by distance.
__device__ __forceinline__ void cp_attend(const float* q, int qst, const float* sk, const float* sv, int kvst, int sn, const float* K, const float* V,
                                          int n_keys, int own0, const float* kn, const float* vn, int nst, const float* bias, int k, int dkv, int dkv_shift,
                                          float* rec, float* att, int tid, int lane, int warp) {
  const int ksh = k <= 1 ? 0 : k <= 2 ? 1 : k <= 4 ? 2 : k <= 8 ? 3 : 4;
  int wsh = 0;
  while (wsh + 1 + ksh <= 4 && (32 << wsh) < n_keys) ++wsh;
  const int wpr = 1 << wsh, m = warp >> wsh, part = warp & (wpr - 1), rst = dkv + 4;
  if (m < k) {
    const int n = bias ? min(n_keys, own0 + m + 1) : n_keys;
    const int j0 = (part * n) >> wsh, j1 = ((part + 1) * n) >> wsh;
    float run = -INFINITY, sum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const int csh = dkv_shift - 2, ch = (lane & ((dkv >> 2) - 1)) * 4, sub = lane >> csh, nsub = 32 >> csh;
    const float* qm = q + m * qst;
#pragma unroll 1
    for (int b = j0; b < j1; b += 32) {
      const int cnt = min(32, j1 - b), j = b + min(lane, cnt - 1);
      const float* kr = j < sn ? sk + j * kvst : j < own0 ? K + (size_t)j * dkv : kn + (j - own0) * nst;
      float s = bias ? __ldg(bias + own0 + m - j) : 0.f, s2 = 0.f;
#pragma unroll 2
      for (int c = 0; c < dkv; c += 8) {
        const float4 a = *reinterpret_cast<const float4*>(kr + c), x = *reinterpret_cast<const float4*>(qm + c);
        const float4 e = *reinterpret_cast<const float4*>(kr + c + 4), y = *reinterpret_cast<const float4*>(qm + c + 4);
        s += a.x * x.x + a.y * x.y + a.z * x.z + a.w * x.w;
        s2 += e.x * y.x + e.y * y.y + e.z * y.z + e.w * y.w;
      }
      s = lane < cnt ? s + s2 : -INFINITY;
      const float nw = fmaxf(run, warp_max(s)), sc = run == -INFINITY ? 0.f : __expf(run - nw), p = __expf(s - nw);   // (no key: 0)
      run = nw;
      sum = sum * sc + p;
      acc.x *= sc; acc.y *= sc; acc.z *= sc; acc.w *= sc;
#pragma unroll 4
      for (int i0 = 0; i0 < cnt; i0 += nsub) {
        const int i = i0 + sub, jj = b + min(i, cnt - 1);
        const float* vr = jj < sn ? sv + jj * kvst : jj < own0 ? V + (size_t)jj * dkv : vn + (jj - own0) * nst;
        const float w = __shfl_sync(0xffffffffu, p, i & 31);   // (past the end: 0)
        const float4 v = *reinterpret_cast<const float4*>(vr + ch);
        acc.x += w * v.x; acc.y += w * v.y; acc.z += w * v.z; acc.w += w * v.w;
      }
    }
    sum = warp_sum(sum);
    for (int o = 1 << csh; o < 32; o <<= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    if (sub == 0) {
      if (wsh == 0) {
        const float is = sub_rcp(sum);
        *reinterpret_cast<float4*>(att + m * dkv + ch) = make_float4(acc.x * is, acc.y * is, acc.z * is, acc.w * is);
      } else {
        float* rp = rec + warp * rst;
        if (lane == 0) { rp[0] = run; rp[1] = sum; }
        *reinterpret_cast<float4*>(rp + 4 + ch) = acc;
      }
    }
  }
  __syncthreads();
  if (wsh) {
    for (int i = tid; i < k << dkv_shift; i += CP_THREADS) {
      const float* rp = rec + ((i >> dkv_shift) << wsh) * rst;
      const int c = i & (dkv - 1);
      float gm = -INFINITY, num = 0.f, den = 0.f;
#pragma unroll 4
      for (int p = 0; p < wpr; ++p) gm = fmaxf(gm, rp[p * rst]);
#pragma unroll 4
      for (int p = 0; p < wpr; ++p) {
        const float w = __expf(rp[p * rst] - gm);
        den += w * rp[p * rst + 1]; num += w * rp[p * rst + 4 + c];
      }
      att[i] = num * sub_rcp(den);
    }
    __syncthreads();
  }
}

// The columns of W_o by head and of W_fo by slice, contiguous, so that a block fetches its share with one copy each (64 to 256 small
// ones cost 1.5 us of issue).  grid.x: layers; built once, when the context is created.
__global__ void cp_pack_kernel(const bild_dec_layer* layers, int d, int I, int dkv, int F, float* wo_pack, float* wfo_pack) {
  const int l = blockIdx.x;
  const bild_dec_layer w = layers[l];
  for (int i = threadIdx.x; i < d * I; i += blockDim.x) {
    const int r = i / I, cc = i - r * I, h = cc / dkv;
    const size_t o = ((size_t)h * d + r) * dkv + (cc - h * dkv);
    wo_pack[(size_t)(2 * l) * d * I + o] = reinterpret_cast<const float*>(w.wo)[i];
    wo_pack[(size_t)(2 * l + 1) * d * I + o] = reinterpret_cast<const float*>(w.wco)[i];
  }
  const int fu = F >> 3;
  for (int c = 0; c < CP_C; ++c) {
    const int f0 = 8 * ((c * fu) / CP_C), fs = 8 * (((c + 1) * fu) / CP_C) - f0;
    for (int i = threadIdx.x; i < d * fs; i += blockDim.x)
      wfo_pack[((size_t)l * F + f0) * d + i] = reinterpret_cast<const float*>(w.wfo)[(size_t)(i / fs) * F + f0 + i % fs];
  }
}

template <int MR>   // MR: token rows in registers at a time (1: single-row passes)
__global__ void __cluster_dims__(CP_C, 1, 1) __launch_bounds__(CP_THREADS, 1) cluster_pass_kernel(const CPassArgs a) {
  extern __shared__ __align__(1024) unsigned char cp_smem[];
  constexpr int WB = 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = (int)cluster_rank();
  const int d = a.d, dkv = a.dkv, F = a.F, H = a.H, I = a.I, d4 = d >> 2;
  const int fu = F >> 3, f0 = 8 * ((c * fu) / CP_C), fs = 8 * (((c + 1) * fu) / CP_C) - f0, fsm = 8 * ((fu + CP_C - 1) / CP_C);
  const CPassLayout L = cp_layout(d, dkv, fsm, a.gated, WB, a.mb, a.n_layers, a.kv_keys);
  unsigned long long* xbar = reinterpret_cast<unsigned long long*>(cp_smem);        // exchanges
  unsigned long long* wbar = reinterpret_cast<unsigned long long*>(cp_smem + 8);    // [0], [1] operands of the sub-layers, two buffers; [2] a block's further heads
  int* failed = reinterpret_cast<int*>(cp_smem + 32);
  bild_dec_layer* tab = reinterpret_cast<bild_dec_layer*>(cp_smem + L.tab);
  float* xs = reinterpret_cast<float*>(cp_smem + L.x);         // [k][d] residual stream
  float* hs = reinterpret_cast<float*>(cp_smem + L.h);         // [k][d] normalised
  float* qkv = reinterpret_cast<float*>(cp_smem + L.qkv);      // [k][3 dkv] of the head at hand
  float* att = reinterpret_cast<float*>(cp_smem + L.att);      // [k][dkv]
  float* rec = reinterpret_cast<float*>(cp_smem + L.rec);
  float* us = reinterpret_cast<float*>(cp_smem + L.u);         // [k][slice]
  float* ploc = reinterpret_cast<float*>(cp_smem + L.ploc);    // [k][d] this block's partial sums
  float* recv = reinterpret_cast<float*>(cp_smem + L.recv);    // [8][k][d] everybody's
  const int k = MR == 1 ? 1 : min(a.desc->k, a.mb), pos0 = a.desc->pos0;   // (written before the pass began: see attn_sub_kernel)
  if (k <= 0) return;   // an empty second chunk
  const int ust = fsm + 8, qst = 3 * dkv, kvst = cp_kv_stride(dkv);
  if (tid == 0) {
    mbar_init(smem_u32(xbar), 1);
    mbar_init(smem_u32(&wbar[0]), 1);
    mbar_init(smem_u32(&wbar[1]), 1);
    mbar_init(smem_u32(&wbar[2]), 1);
    *failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < a.n_layers * (int)(sizeof(bild_dec_layer) / 8); i += CP_THREADS)
    reinterpret_cast<unsigned long long*>(tab)[i] = __ldg(reinterpret_cast<const unsigned long long*>(a.layers) + i);
  const int n_enc = min(*a.n_keys_dev, a.ecap);
  __syncthreads();
  sub_cluster_arrive_relaxed();
  pdl_launch_dependents();
  const unsigned lim = (a.spin > SPIN_LIMIT ? a.spin : SPIN_LIMIT) * 4u;
  auto wait = [&](unsigned long long* bar, unsigned parity) {   // bounded; after a time-out nothing is waited for any more
    __syncwarp();   // (a lane that polls must not keep a sibling from issuing a copy or a store)
    if (sub_try_cluster(smem_u32(bar), parity) || *(volatile int*)failed) return;
    for (unsigned it = 0; it < lim; ++it)
      if (sub_try_cluster(smem_u32(bar), parity)) return;
    *failed = 1;
    atomicExch(a.err, (int)BILD_ERR_TIMEOUT);
  };
  // operands of head h of an attention sub-layer in a buffer: gain | W_q (k, v) rows | W_o columns | keys | values
  const int o_wp = d * 4, o_wo = o_wp + 3 * dkv * d * WB, o_k = o_wo + d * dkv * WB, o_v = o_k + a.kv_keys * kvst * 4;
  // ... and of a slice of a feed-forward sub-layer: gain | W_i | gate | W_fo columns
  const int o_g = o_wp + fsm * d * WB, o_f = o_g + a.gated * fsm * d * WB;
  auto fetch_head = [&](unsigned char* b, unsigned long long* bar, bool self, int l, int h) {
    const bild_dec_layer& w = tab[l];
    const unsigned char* Wp = reinterpret_cast<const unsigned char*>(self ? w.wqkv : w.wcq);
    const unsigned char* Wo = reinterpret_cast<const unsigned char*>(a.wo_pack) + ((size_t)(2 * l + (self ? 0 : 1)) * H + h) * d * dkv * WB;
    const int np = self ? 3 : 1, cap = self ? a.cap : a.ecap, n = min(self ? pos0 : n_enc, a.kv_keys);
    const size_t kv = ((size_t)l * H + h) * cap * dkv;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (tid == 0) {
      mbar_expect(smem_u32(bar), (uint32_t)(d * 4 + np * dkv * d * WB + d * dkv * WB + n * dkv * 8));
      bulk_g2s(smem_u32(b), self ? w.ln1 : w.ln2, (uint32_t)(d * 4), smem_u32(bar));
    }
    if (tid >= 32 && tid < 32 + np)
      bulk_g2s(smem_u32(b + o_wp + (tid - 32) * dkv * d * WB), Wp + ((size_t)(tid - 32) * I + h * dkv) * d * WB, (uint32_t)(dkv * d * WB), smem_u32(bar));
    if (tid == 64) bulk_g2s(smem_u32(b + o_wo), Wo, (uint32_t)(d * dkv * WB), smem_u32(bar));
    // (the copies a warp issues go out one after the other: dealt to all warps)
    for (int i = lane * CP_WARPS + warp; i < 2 * n; i += CP_THREADS)
      bulk_g2s(smem_u32(b + ((i & 1) ? o_v : o_k) + (i >> 1) * kvst * 4),
               ((i & 1) ? (self ? a.selfV : a.crossV) : (self ? a.selfK : a.crossK)) + kv + (size_t)(i >> 1) * dkv, (uint32_t)(dkv * 4), smem_u32(bar));
  };
  auto fetch = [&](int s) {   // operands of sub-layer s (three a layer)
    const int l = s / 3, kind = s - 3 * l;
    unsigned char* b = cp_smem + L.buf + (s & 1) * L.buf_bytes;
    unsigned long long* bar = &wbar[s & 1];
    if (kind < 2) {
      if (c < H) { fetch_head(b, bar, kind == 0, l, c); return; }
      if (tid == 0) {   // a block without a head takes the gain only
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect(smem_u32(bar), (uint32_t)(d * 4));
        bulk_g2s(smem_u32(b), kind == 0 ? tab[l].ln1 : tab[l].ln2, (uint32_t)(d * 4), smem_u32(bar));
      }
      return;
    }
    const bild_dec_layer& w = tab[l];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (tid == 0) {
      mbar_expect(smem_u32(bar), (uint32_t)(d * 4 + (2 + a.gated) * fs * d * WB));
      bulk_g2s(smem_u32(b), w.ln3, (uint32_t)(d * 4), smem_u32(bar));
      if (fs > 0) {
        bulk_g2s(smem_u32(b + o_wp), reinterpret_cast<const unsigned char*>(w.wi0) + (size_t)f0 * d * WB, (uint32_t)(fs * d * WB), smem_u32(bar));
        if (a.gated) bulk_g2s(smem_u32(b + o_g), reinterpret_cast<const unsigned char*>(w.wi1) + (size_t)f0 * d * WB, (uint32_t)(fs * d * WB), smem_u32(bar));
      }
    }
    if (fs > 0 && tid == 32)
      bulk_g2s(smem_u32(b + o_f), reinterpret_cast<const unsigned char*>(a.wfo_pack) + ((size_t)l * F + f0) * d * WB, (uint32_t)(fs * d * WB), smem_u32(bar));
  };
  fetch(0);
  for (int i = tid; i < k * d; i += CP_THREADS) {
    const int m = i / d, cc = i - m * d;
    int t = a.tokens[m];
    t = t < 0 ? 0 : (t >= a.vocab ? a.vocab - 1 : t);
    xs[i] = reinterpret_cast<const float*>(a.emb)[(size_t)t * d + cc];
  }
  __syncthreads();
  pdl_wait();
  sub_cluster_wait();
  // residual stream + what the blocks 0 .. nsrc - 1 sent (in block order), then its norm with the gain of sub-layer s: warp <-> token row
  auto rows = [&](int nsrc, int s) {
    if (warp < k) {
      float4 v[2];
      float ss = 0.f;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i = lane + 32 * j;
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < d4) {
          float* p = xs + warp * d + 4 * i;
          v[j] = *reinterpret_cast<const float4*>(p);
          float4 q[CP_C];
#pragma unroll
          for (int b = 0; b < CP_C; ++b)
            q[b] = b < nsrc ? *reinterpret_cast<const float4*>(recv + (b * k + warp) * d + 4 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int b = 0; b < CP_C; ++b) { v[j].x += q[b].x; v[j].y += q[b].y; v[j].z += q[b].z; v[j].w += q[b].w; }
          *reinterpret_cast<float4*>(p) = v[j];
          ss += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
        }
      }
      if (s >= 0) {
        const float inv = rsqrtf(warp_sum(ss) * a.inv_d + a.eps);
        wait(&wbar[s & 1], (s >> 1) & 1);
        const float* g = reinterpret_cast<const float*>(cp_smem + L.buf + (s & 1) * L.buf_bytes);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int i = lane + 32 * j;
          if (i < d4) {
            const float4 gv = *reinterpret_cast<const float4*>(g + 4 * i);
            *reinterpret_cast<float4*>(hs + warp * d + 4 * i) = make_float4(v[j].x * inv * gv.x, v[j].y * inv * gv.y, v[j].z * inv * gv.z, v[j].w * inv * gv.w);
          }
        }
      }
    }
    __syncwarp();
  };
  rows(0, 0);
  const int ns = 3 * a.n_layers;
  unsigned xpar = 0, hpar = 0;
#pragma unroll 1
  for (int s = 0; s < ns; ++s) {
    const int l = s / 3, kind = s - 3 * l;
    unsigned char* b = cp_smem + L.buf + (s & 1) * L.buf_bytes;
    __syncthreads();   // normalised rows complete; the other buffer is no longer read
    if (s + 1 < ns) fetch(s + 1);
    wait(&wbar[s & 1], (s >> 1) & 1);
    int nsrc = CP_C;
    if (kind < 2) {
      const bool self = kind == 0;
      const int cap = self ? a.cap : a.ecap, n = self ? min(pos0 + k, cap) : n_enc, own = self ? pos0 : n;
      nsrc = min(H, CP_C);
#pragma unroll 1
      for (int h = c; h < H; h += CP_C) {
        if (h != c) {   // one more head for this block: its operands replace the last one's
          __syncthreads();
          fetch_head(b, &wbar[2], self, l, h);
          wait(&wbar[2], hpar);
          hpar ^= 1u;
        }
        const size_t kv = ((size_t)l * H + h) * cap * dkv;
        cp_rows<MR>(reinterpret_cast<const float*>(b + o_wp), (self ? 3 : 1) * dkv, d, hs, d, k, warp, lane, [&](int i, int m, float v) {
          qkv[m * qst + i] = v;
          if (i >= dkv && pos0 + m < cap) (i < 2 * dkv ? a.selfK : a.selfV)[kv + (size_t)(pos0 + m) * dkv + (i & (dkv - 1))] = v;
        });
        __syncthreads();
        const float* sk = reinterpret_cast<const float*>(b + o_k);
        const float* sv = reinterpret_cast<const float*>(b + o_v);
        const int sn = min(self ? pos0 : n_enc, a.kv_keys);
        const float* K = (self ? a.selfK : a.crossK) + kv;
        const float* V = (self ? a.selfV : a.crossV) + kv;
        const float* bias = self ? a.bias + (size_t)h * a.cap : nullptr;
        cp_attend(qkv, qst, sk, sv, kvst, sn, K, V, n, own, qkv + dkv, qkv + 2 * dkv, qst, bias, k, dkv, a.dkv_shift, rec, att, tid, lane, warp);
        cp_rows<MR>(reinterpret_cast<const float*>(b + o_wo), d, dkv, att, dkv, k, warp, lane,
                            [&](int i, int m, float v) { if (h == c) ploc[m * d + i] = v; else ploc[m * d + i] += v; });
      }
    } else {
      cp_rows<MR>(reinterpret_cast<const float*>(b + o_wp), fs, d, hs, d, k, warp, lane,
                          [&](int i, int m, float v) { us[m * ust + i] = a.gated ? gelu_tanh(v) : fmaxf(v, 0.f); });
      if (a.gated)   // (the same thread owns the same element)
        cp_rows<MR>(reinterpret_cast<const float*>(b + o_g), fs, d, hs, d, k, warp, lane, [&](int i, int m, float v) { us[m * ust + i] *= v; });
      __syncthreads();
      if (fs > 0) {
        cp_rows<MR>(reinterpret_cast<const float*>(b + o_f), d, fs, us, ust, k, warp, lane, [&](int i, int m, float v) { ploc[m * d + i] = v; });
      } else {
        for (int i = tid; i < k * d; i += CP_THREADS) ploc[i] = 0.f;
      }
    }
    // this block's partial sums to every block
    __syncthreads();
    if (tid == 0) mbar_expect(smem_u32(xbar), (uint32_t)(nsrc * k * d * 4));
    if (s > 0) sub_cluster_wait();   // every block has used what it received last
    if (c < nsrc)
      for (int i = tid; i < k * d4 * CP_C; i += CP_THREADS)
        sub_push4(recv + c * k * d + 4 * (i >> 3), xbar, (uint32_t)(i & (CP_C - 1)), *reinterpret_cast<const float4*>(ploc + 4 * (i >> 3)));
    wait(xbar, xpar);
    xpar ^= 1u;
    rows(nsrc, s + 1 < ns ? s + 1 : -1);
    sub_cluster_arrive_relaxed();
  }
  __syncthreads();
  for (int i = c * CP_THREADS + tid; i < k * d; i += CP_C * CP_THREADS) a.x_out[i] = xs[i];
  __syncwarp();
  sub_cluster_wait();
}

}  // namespace bild
