// Parent-conditioned scoring (Eq. 1) fused with logsumexp at temperature 1 and T, top-K logits and
// Gumbel top-K sibling draws (Eq. 2), one pass over the vocabulary.
//
// score_tile_kernel: fp32 FMA, any dtype, rank and vocabulary size.  The vocabulary is split into tiles, one CTA
// per tile with its W tile resident in shared memory for all parents of the launch, one parent per thread.
// merge_kernel folds the records of each parent.  Serves fp32 inputs (with ts_score_few.cu for short lists) and
// bf16 ranks that are no multiple of 8; the other bf16 shapes run on the tensor cores (ts_tree.cu).
#include "ts_internal.h"
#include "ts_scan.cuh"
#include "ts_merge.cuh"

namespace ts {

template <typename TIn, class Lists>
__global__ void __launch_bounds__(SCORE_THREADS, 1) score_tile_kernel(ScoreArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int r = a.r, TV = a.TV, V = a.V;
  TIn* Ws = reinterpret_cast<TIn*>(smem_raw);                              // [r][TV]
  float* as = reinterpret_cast<float*>(smem_raw + (size_t)r * TV * sizeof(TIn));  // [r][SCORE_THREADS]
  float* ghi = as + (size_t)r * SCORE_THREADS;                             // [512]
  const int tid = threadIdx.x;
  const int tile = blockIdx.x;
  const int t0 = tile * TV;
  const int tlen = min(TV, V - t0);
  const TIn* Wg = reinterpret_cast<const TIn*>(a.W);
  const TIn* Ug = reinterpret_cast<const TIn*>(a.U);
  const TIn* Ag = reinterpret_cast<const TIn*>(a.A);
  constexpr int VEC = Elem<TIn>::VEC;
  const bool vec_ok = (V % VEC) == 0;
  pdl_wait();
  pdl_launch_dependents();
  const int P = a.P_dev ? *a.P_dev : a.P;
  if (P <= 0) return;  // an empty level: nothing to stage

  // stage the W tile
  if (vec_ok) {
    const int per_row = TV / VEC;
    for (int i = tid; i < r * per_row; i += SCORE_THREADS) {
      const int k = i / per_row, c = (i % per_row) * VEC;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (c < tlen) v = __ldg(reinterpret_cast<const uint4*>(Wg + (size_t)k * V + t0 + c));
      *reinterpret_cast<uint4*>(Ws + (size_t)k * TV + c) = v;
    }
  } else {
    for (int i = tid; i < r * TV; i += SCORE_THREADS) {
      const int k = i / TV, c = i % TV;
      Ws[(size_t)k * TV + c] = c < tlen ? Wg[(size_t)k * V + t0 + c] : TIn(0.f);
    }
  }
  fill_gumbel_bounds(ghi, tid, SCORE_THREADS);
  __syncthreads();

  const float T = a.T, invT = T > 0.f ? 1.f / T : 1.f;
  const int K = a.K;
  const int rw = rec_words(K);

  for (int pg = 0; pg < P; pg += SCORE_THREADS) {
    const int p = pg + tid;
    if (p >= P) continue;  // no block-wide barrier below
    const int req = a.p_req[p], dep = a.p_depth[p], ptok = a.p_token[p];
    const uint64_t hash = a.p_hash[p];
    for (int k = 0; k < r; ++k) as[k * SCORE_THREADS + tid] = Elem<TIn>::to_f(Ag[(size_t)ptok * r + k]);
    const TIn* Urow = Ug + ((size_t)req * a.D + dep) * V + t0;
    RowScan<Lists> st;
    st.init(K);
    float gL = -INFINITY, gK = -INFINITY;
    const SharedThr gl{a.slots + (size_t)p * K * SLOT_STRIDE, tile % K};
    const SharedThr gk{a.slots + ((size_t)a.cap + p) * K * SLOT_STRIDE, tile % K};
    for (int c0 = 0; c0 < tlen; c0 += CHUNK) {
      const int valid = min(CHUNK, tlen - c0);
      float l[CHUNK];
      load16<TIn>(Urow + c0, vec_ok, valid, l);
      for (int k = 0; k < r; ++k) {
        const float ak = as[k * SCORE_THREADS + tid];
        float w[CHUNK];
        if (sizeof(TIn) == 2) {
          const uint4 w0 = *reinterpret_cast<const uint4*>(Ws + (size_t)k * TV + c0);
          const uint4 w1 = *reinterpret_cast<const uint4*>(Ws + (size_t)k * TV + c0 + 8);
          unpack_bf16x8(w0, w);
          unpack_bf16x8(w1, w + 8);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(Ws) + (size_t)k * TV + c0 + 4 * i);
            w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
          }
        }
#pragma unroll
        for (int i = 0; i < CHUNK; ++i) l[i] = fmaf(ak, w[i], l[i]);
      }
      if ((c0 & (4 * CHUNK - 1)) == 0) {  // refresh the launch-wide bounds every fourth chunk
        gL = fmaxf(gL, dec_f(slots_min(gl, K)));
        if (T > 0.f) gK = fmaxf(gK, dec_f(slots_min(gk, K)));
      }
      scan_chunk(st, l, t0 + c0, valid, T, invT, a.seed, req, hash, ghi, gL, gK, gl, gk);
    }
    gL = fmaxf(gL, dec_f(slots_min(gl, K)));
    if (T > 0.f) gK = fmaxf(gK, dec_f(slots_min(gk, K)));
    st.store(a.rec + ((size_t)tile * a.cap + p) * rw, gL, gK);  // piece = (tile, 0), slot = p
  }
}

// merge_kernel: one CTA of MERGE_THREADS threads per parent (body in ts_merge.cuh)
template <int KR>
__global__ void __launch_bounds__(MERGE_THREADS) merge_kernel(MergeArgs a) {
  __shared__ MergeSmem sm;
  pdl_wait();               // the scoring launch's records and the level's parent count
  pdl_launch_dependents();
  const int P = a.P_dev ? *a.P_dev : a.P;
  for (int p = blockIdx.x; p < P; p += gridDim.x) merge_parent<KR>(a, p, sm, (int)threadIdx.x, [] { __syncthreads(); });
}

// ------------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------------
size_t score_scratch_bytes(const ts_ctx* ctx, int P, int* cap_out) {
  int cap = (P + 7) / 8 * 8;
  if (cap_out) *cap_out = cap;
  // records, then the pruning state
  return record_bytes(ctx, cap) + align_up(thr_bytes(ctx, cap), 256);
}

unsigned* thr_base(const ts_ctx* ctx, float* rec, int cap) {
  return (unsigned*)((char*)rec + record_bytes(ctx, cap));
}

// pruning slots [2][cap][K] (one 128-byte line each); must be zero before a launch
size_t thr_bytes(const ts_ctx* ctx, int cap) { return 2 * (size_t)cap * (size_t)ctx->cfg.K * SLOT_STRIDE * sizeof(unsigned); }

cudaError_t launch_score(const ts_ctx* ctx, float* rec, int cap, const void* U, const void* A, const void* W,
                         int P, const int* P_dev, const int* p_req, const int* p_depth, const int* p_token,
                         const uint64_t* p_hash, float T, uint64_t seed, float* lse0, float* lseT, int* top_tok,
                         float* top_logit, int* draw_tok, float* draw_logit, cudaStream_t st, bool pdl,
                         int p_bound) {
  const ts_config& c = ctx->cfg;
  ScoreArgs a{};
  a.U = U; a.A = A; a.W = W; a.V = c.V; a.D = c.D; a.r = c.r; a.K = c.K; a.T = T; a.seed = seed;
  a.TV = ctx->tile.TV; a.ntiles = ctx->tile.ntiles; a.cap = cap; a.rec = rec;
  a.slots = thr_base(ctx, rec, cap);
  a.pdl = pdl ? 1 : 0;
  a.P = P; a.P_dev = P_dev;
  a.p_req = p_req; a.p_depth = p_depth; a.p_token = p_token; a.p_hash = p_hash;
  cudaError_t e = cudaSuccess;
  // Which kernel scores the level: the few-parents kernel when the host knows that the list cannot hold
  // more than few_cap parents (its own P, or a bound of the device-side count), the tile kernel otherwise.
  const int bound = P_dev ? p_bound : P;
  const bool run_few = bound >= 0 && bound <= ctx->few_cap;
  a.few_cap = ctx->few_cap;
  if (!run_few) {
    ProfScope ps(ctx, K_SCORE, st);
    if (c.dt_U == TS_DTYPE_BF16) {
      if (c.K <= 8) e = launch_kernel(score_tile_kernel<__nv_bfloat16, RegLists<8>>, a.ntiles, SCORE_THREADS, ctx->tile.smem, st, pdl, a);
      else e = launch_kernel(score_tile_kernel<__nv_bfloat16, MemLists>, a.ntiles, SCORE_THREADS, ctx->tile.smem, st, pdl, a);
    } else {
      if (c.K <= 8) e = launch_kernel(score_tile_kernel<float, RegLists<8>>, a.ntiles, SCORE_THREADS, ctx->tile.smem, st, pdl, a);
      else e = launch_kernel(score_tile_kernel<float, MemLists>, a.ntiles, SCORE_THREADS, ctx->tile.smem, st, pdl, a);
    }
    if (e != cudaSuccess) return e;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (run_few) {
    ProfScope ps(ctx, K_SCORE_FEW, st);
    e = launch_score_few(ctx, a, bound, st);
    if (e != cudaSuccess) return e;
  }
  MergeArgs m{};
  m.pdl = a.pdl;
  m.few_ntiles = run_few ? few_tiles(c) : 0; m.few_cap = ctx->few_cap;
  m.P = P; m.P_dev = P_dev; m.K = c.K; m.ntiles = a.ntiles; m.cap = cap; m.T = T;
  m.rec = rec; m.slots = a.slots;
  m.lse0 = lse0; m.lseT = lseT; m.top_tok = top_tok; m.top_logit = top_logit; m.draw_tok = draw_tok; m.draw_logit = draw_logit;
  int blocks = P_dev ? cap : P;
  if (blocks > 2 * ctx->num_sms) blocks = 2 * ctx->num_sms;   // parents beyond that are looped over
  if (blocks < 1) blocks = 1;
  {
    ProfScope ps(ctx, K_MERGE, st);
    if (c.K <= 8) e = launch_kernel(merge_kernel<8>, blocks, MERGE_THREADS, 0, st, pdl, m);
    else e = launch_kernel(merge_kernel<16>, blocks, MERGE_THREADS, 0, st, pdl, m);
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t score_setup(ts_ctx* ctx) {
  // never launched here: a tensor-core context needs its tile only to score ragged vocabularies without a workspace
  if (ctx->use_tree && ctx->cfg.V % 8 == 0) return cudaSuccess;
  cudaError_t e = allow_all_smem(score_tile_kernel<__nv_bfloat16, RegLists<8>>, ctx->max_smem);
  if (e == cudaSuccess) e = allow_all_smem(score_tile_kernel<__nv_bfloat16, MemLists>, ctx->max_smem);
  if (e == cudaSuccess) e = allow_all_smem(score_tile_kernel<float, RegLists<8>>, ctx->max_smem);
  if (e == cudaSuccess) e = allow_all_smem(score_tile_kernel<float, MemLists>, ctx->max_smem);
  return e;
}

}  // namespace ts

extern "C" int32_t ts_score_parents(ts_ctx* ctx, const void* U, const void* A, const void* W, int32_t P,
                                    const int32_t* parent_req, const int32_t* parent_depth,
                                    const int32_t* parent_token, const uint64_t* parent_hash, float T, uint64_t seed,
                                    float* lse0, float* lseT, int32_t* top_tok, float* top_logit, int32_t* draw_tok,
                                    float* draw_logit, void* ws, size_t ws_bytes, void* stream) {
  using namespace ts;
  if (!ctx) return set_error(TS_ERR_INVALID, "ts_score_parents: null context");
  const void* ptrs[] = {U, A, W, parent_req, parent_depth, parent_token, parent_hash, lse0, lseT,
                        top_tok, top_logit, draw_tok, draw_logit, ws};
  for (const void* p : ptrs)
    if (!p || ((uintptr_t)p & 15u)) return set_error(TS_ERR_INVALID, "ts_score_parents: null or misaligned pointer");
  const WsLayout L = make_layout(ctx, ctx->cfg.max_batch);
  if (P < 0 || P > L.Pcap)
    return set_error(TS_ERR_INVALID, "ts_score_parents: P out of range");
  if (!(T >= 0.f)) return set_error(TS_ERR_INVALID, "ts_score_parents: T must be >= 0");
  if (ws_bytes < L.total) return set_error(TS_ERR_WORKSPACE, "ts_score_parents: workspace too small");
  if (P == 0) return TS_OK;
  const cudaStream_t st = (cudaStream_t)stream;
  if (ctx->use_tree && P > ctx->few_cap) {
    const cudaError_t et = tree_score(ctx, (char*)ws + L.tree, U, A, W, P, parent_req, parent_depth, parent_token, parent_hash, T, seed, lse0, lseT, top_tok,
                                      top_logit, draw_tok, draw_logit, ctx->cfg.max_batch * ctx->cfg.D, st);
    return et == cudaSuccess ? TS_OK : set_cuda_error("ts_score_parents", et);
  }
  float* rec = (float*)((char*)ws + (ctx->use_tree ? L.tree : L.rec));
  int cap = L.rec_cap;
  if (ctx->use_tree) (void)score_scratch_bytes(ctx, P, &cap);
  cudaError_t e = cudaMemsetAsync(thr_base(ctx, rec, cap), 0, thr_bytes(ctx, cap), st);
  if (e != cudaSuccess) return set_cuda_error("ts_score_parents(memset)", e);
  e = launch_score(ctx, rec, cap, U, A, W, P, nullptr, parent_req, parent_depth, parent_token, parent_hash, T, seed, lse0, lseT, top_tok,
                   top_logit, draw_tok, draw_logit, st);
  if (e != cudaSuccess) return set_cuda_error("ts_score_parents", e);
  return TS_OK;
}
