// Scoring kernel for lists of few parents: the levels of an fp32 expansion (a small model decoding a request or a handful)
// and short lists given to the stand-alone call, in fp32 and bf16.
//
// With a handful of parents the low-rank bias [parents x r] . [r x V] is no dense contraction, and the tile kernel -- one
// parent per lane, every lane over the whole tile -- would leave most lanes idle while it walks the vocabulary.  Here the
// mapping is turned round: one warp = one (parent, 256-token tile), one lane = eight consecutive tokens.
// The lane forms its eight logits with fused multiply-adds (U + sum_k A[x_p][k] W[k][v], k ascending),
// every token gets its exact Gumbel key (no bounds: a tile is over before any could arrive), and the
// warp's K best logits and K best keys come out of K rounds of a warp-wide arg-max.  The whole grid works
// on every parent at once.  W is read through L1 (the eight warps of a CTA share a tile and its lines).
// One parent at V = 32,000, r = 16: 61 us with the tile kernel, about 10 us here (a four-level tree: 217 us of scoring before, 47 us now).
//
// Records have the layout of the tile kernel's (header (max, sum0, sumT, counts), then K logits,
// K tokens, K keys, K tokens, K logits), one per (tile, parent) at rec[(tile * few_cap + p) * rec_words];
// the merge kernel is told which kernel ran.  The host sends a level here when it knows that the level
// cannot have more than few_cap parents (B * K^depth and B * Nmax bound it); few_cap is what 4 MiB of records hold, 256 at most.
#include "ts_internal.h"
#include "ts_scan.cuh"

namespace ts {

// eight consecutive elements
__device__ __forceinline__ void load8(const float* p, float* out) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w; out[4] = b.x; out[5] = b.y; out[6] = b.z; out[7] = b.w;
}

__device__ __forceinline__ void load8(const __nv_bfloat16* p, float* out) { unpack_bf16x8(__ldg(reinterpret_cast<const uint4*>(p)), out); }

constexpr int FEW_THREADS = 256;
constexpr int FEW_WARPS = FEW_THREADS / 32;
constexpr int FEW_TILE = 256;   // tokens per tile: eight per lane
// bf16 lists that the one-launch kernel (ts_tree.cu) would score too: at most so many parents, (parent, tile) pairs and ranks.
// That kernel takes 30 to 50 us for one parent as for 32 (its set-up, seed bounds and grid barriers); here a list costs 22 us
// and grows with its pairs.  Cold caches, T = 1, here / there (us): V = 32,000, r = 64: 36 / 44 for 1 parent, 36 / 46 for 16,
// 42 / 48 for 32, 56 / 52 for 64; V = 151,936: 36 / 50 for 1, 40 / 50 for 4, 48 / 52 for 8, 71 / 52 for 16; V = 1,000: 32 / 56
// for 64.  r = 128, K = 16, V = 128,256: 60 / 71 for 4, 71 / 73 for 8.  r = 256, V = 32,000: 65 / 58 for 1 (warm 34 / 40).
constexpr int FEW_TREE_MAX = 64, FEW_TREE_ITEMS = 3000, FEW_TREE_RANK = 128;

// (value desc, token asc) arg-max over the warp; every lane gets the winner (two reductions of integers: the value's
// order-preserving image, then the lowest token among those that have it)
__device__ __forceinline__ void warp_best(float& v, int& tok) {
  const unsigned e = enc_f(v), m = __reduce_max_sync(0xFFFFFFFFu, e);
  tok = (int)__reduce_min_sync(0xFFFFFFFFu, e == m ? (unsigned)tok : 0x7FFFFFFFu);
  v = dec_f(m);
}

template <typename TIn>
__global__ void __launch_bounds__(FEW_THREADS) score_few_kernel(const ScoreArgs a) {
  __shared__ float s_a[FEW_WARPS][256];   // head row A[x_p] of each warp's parent (r <= 256)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_wait();                // the parent list and its length come from the kernel before
  pdl_launch_dependents();
  const int P = a.P_dev ? *a.P_dev : a.P;
  if (P <= 0 || P > a.few_cap) return;   // an empty level (the host never sends a longer list here)
  const int p = blockIdx.y * FEW_WARPS + warp;
  if (p >= P) return;                  // no block-wide barrier below
  const int V = a.V, r = a.r, K = a.K;
  const int tile = blockIdx.x, v = tile * FEW_TILE + lane * 8;
  const bool in = v < V;               // V is a multiple of 8: a lane's eight tokens are all inside or all outside
  const TIn* Wg = reinterpret_cast<const TIn*>(a.W);
  const TIn* Ug = reinterpret_cast<const TIn*>(a.U);
  const TIn* Ag = reinterpret_cast<const TIn*>(a.A);
  const int req = a.p_req[p], dep = a.p_depth[p], ptok = a.p_token[p];
  const uint64_t hash = a.p_hash[p];
  for (int k = lane; k < r; k += 32) s_a[warp][k] = Elem<TIn>::to_f(Ag[(size_t)ptok * r + k]);
  __syncwarp();

  // ---- logits of the lane's eight tokens -------------------------------------------------------------
  float l[8];
  if (in) {
    load8(Ug + ((size_t)req * a.D + dep) * V + v, l);
#pragma unroll 16
    for (int k = 0; k < r; ++k) {
      float w[8];
      load8(Wg + (size_t)k * V + v, w);
      const float ak = s_a[warp][k];
#pragma unroll
      for (int i = 0; i < 8; ++i) l[i] = fmaf(ak, w[i], l[i]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) l[i] = -INFINITY;
  }

  // ---- max and sums of exponentials over the tile -----------------------------------------------------
  const float T = a.T, invT = T > 0.f ? 1.f / T : 1.f;
  const bool two = (T > 0.f) && (T != 1.f);
  float m = l[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) m = fmaxf(m, l[i]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
  float s0 = 0.f, sT = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float d = l[i] - m;   // -inf for tokens outside V: contributes 0
    s0 += __expf(d);
    if (two) sT += __expf(d * invT);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, off);
    sT += __shfl_xor_sync(0xFFFFFFFFu, sT, off);
  }
  if (!two) sT = s0;

  // ---- K best logits: K rounds of arg-max, lane j keeps the j-th ---------------------------------------
  float topv = -INFINITY; int topi = -1;
  {
    uint32_t taken = 0;
    for (int j = 0; j < K; ++j) {
      float bv = -INFINITY; int bi = 0x7FFFFFFF;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (!((taken >> i) & 1u) && l[i] > bv) { bv = l[i]; bi = v + i; }   // first maximum: lowest token
      warp_best(bv, bi);
      if (bv > -INFINITY && bi >= v && bi < v + 8) taken |= 1u << (bi - v);
      if (lane == j) { topv = bv; topi = bv > -INFINITY ? bi : -1; }
    }
  }

  // ---- K best Gumbel keys (without-replacement draws in order) -----------------------------------------
  float keyv = -INFINITY, keyl = 0.f; int keyi = -1;
  if (T > 0.f) {
    float key[8];
    if (in) {
      const uint4 cw = stream_words(a.seed, req, hash, STREAM_GUMBEL_COARSE, (uint32_t)v >> 3);
      const uint4 fw = stream_words(a.seed, req, hash, STREAM_GUMBEL_FINE, (uint32_t)v >> 3);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t c16 = (word_of(cw, i >> 1) >> (16 * (i & 1))) & 0xFFFFu;
        const uint32_t f16 = (word_of(fw, i >> 1) >> (16 * (i & 1))) & 0xFFFFu;
        key[i] = l[i] * invT + gumbel_from_bits((c16 << 16) | f16);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) key[i] = -INFINITY;
    }
    uint32_t taken = 0;
    for (int j = 0; j < K; ++j) {
      float bv = -INFINITY; int bi = 0x7FFFFFFF;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (!((taken >> i) & 1u) && key[i] > bv) { bv = key[i]; bi = v + i; }
      warp_best(bv, bi);
      const bool mine = bv > -INFINITY && bi >= v && bi < v + 8;
      float lg = 0.f;
      if (mine) {
        taken |= 1u << (bi - v);
#pragma unroll
        for (int i = 0; i < 8; ++i) lg = (bi - v == i) ? l[i] : lg;
      }
      // the winner's logit travels to lane j (exactly one lane holds it)
      const unsigned who = __ballot_sync(0xFFFFFFFFu, mine);
      const float wl = who ? __shfl_sync(0xFFFFFFFFu, lg, __ffs(who) - 1) : 0.f;
      if (lane == j) { keyv = bv; keyi = bv > -INFINITY ? bi : -1; keyl = wl; }
    }
  }

  // ---- publish the piece's best values (the merge filters the records with the resulting bounds) -----
  {
    const float bestL = __shfl_sync(0xFFFFFFFFu, topv, 0), bestK = __shfl_sync(0xFFFFFFFFu, keyv, 0);
    if (lane == 0) {
      const SharedThr gl{a.slots + (size_t)p * K * SLOT_STRIDE, tile % K};
      const SharedThr gk{a.slots + ((size_t)a.cap + p) * K * SLOT_STRIDE, tile % K};
      if (bestL > -INFINITY) publish(gl, bestL);
      if (T > 0.f && bestK > -INFINITY) publish(gk, bestK);
    }
  }

  // ---- record ----------------------------------------------------------------------------------------------
  const int rw = rec_words(K);
  float* rec = a.rec + ((size_t)tile * a.few_cap + p) * rw;
  const int nt = __popc(__ballot_sync(0xFFFFFFFFu, lane < K && topi >= 0));
  const int nk = __popc(__ballot_sync(0xFFFFFFFFu, lane < K && keyi >= 0));
  if (lane == 0) *reinterpret_cast<float4*>(rec) = make_float4(m, s0, sT, __int_as_float(nt | (nk << 8)));
  if (lane < K) {
    float* f = rec + 4; int* ii = reinterpret_cast<int*>(rec) + 4;
    f[lane] = topv; ii[K + lane] = topi; f[2 * K + lane] = keyv; ii[3 * K + lane] = keyi; f[4 * K + lane] = keyl;
  }
}

int few_tiles(const ts_config& c) { return (c.V + FEW_TILE - 1) / FEW_TILE; }

// parents a launch may hold (0: the kernel does not serve this configuration)
int few_capacity(const ts_config& c, bool use_tree) {
  if (c.V % 8 != 0 || (c.dt_U != TS_DTYPE_F32 && !use_tree)) return 0;
  if (use_tree && c.r > FEW_TREE_RANK) return 0;
  if (use_tree) return FEW_TREE_ITEMS / few_tiles(c) < FEW_TREE_MAX ? FEW_TREE_ITEMS / few_tiles(c) : FEW_TREE_MAX;
  const size_t per = (size_t)few_tiles(c) * rec_words(c.K) * 4, cap = ((size_t)4 << 20) / per;
  return cap > 256 ? 256 : (int)cap;
}

cudaError_t launch_score_few(const ts_ctx* ctx, const ScoreArgs& a, int p_bound, cudaStream_t st) {
  const dim3 grid(few_tiles(ctx->cfg), (p_bound + FEW_WARPS - 1) / FEW_WARPS > 0 ? (p_bound + FEW_WARPS - 1) / FEW_WARPS : 1);
  const cudaError_t e = ctx->cfg.dt_U == TS_DTYPE_F32 ? launch_kernel(score_few_kernel<float>, grid, dim3(FEW_THREADS), 0, st, a.pdl != 0, a)
                                                      : launch_kernel(score_few_kernel<__nv_bfloat16>, grid, dim3(FEW_THREADS), 0, st, a.pdl != 0, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace ts
