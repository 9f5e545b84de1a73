// The one-launch expansion (ts_tree.cu): arguments, shared-memory plan and small device pieces.
#pragma once
#include "ts_internal.h"
#include "ts_level.cuh"
#include "ts_scan.cuh"
#include "ts_tc.cuh"

namespace ts {

constexpr int TX_SCAN_WARPS = 16;          // warps that scan accumulators: 4 tensor-memory lane quarters x 4 splits
constexpr int TX_SPLIT = TX_SCAN_WARPS / 4;
constexpr int TX_ISSUERS = 2;
constexpr int TX_MMA = TX_SCAN_WARPS;      // this and the next issue the MMAs
constexpr int TX_REFRESH = TX_MMA + TX_ISSUERS;   // requests W, keeps the rows' launch-wide bounds current
constexpr int TX_SELECT = TX_REFRESH + 1;       // evaluates queued candidates exactly
constexpr int TX_WARPS = TX_SELECT + 1;
constexpr int TX_THREADS = TX_WARPS * 32;
constexpr int TX_ROWS = 128;               // parent rows of one MMA tile
constexpr int TX_QCAP = 256;               // candidate queue entries (power of two)
constexpr int TX_PLACE_BITS = 17;          // of a queued candidate's place in the CTA's range
constexpr int TX_STAGE_MAX = 8;            // stages of the W ring
constexpr int TX_USTAGES = 4;              // stages of the base-logit ring (two: the chain of 128 requests 674 us, four: 581)
constexpr int TX_RING_MIN = TX_ROWS / 2 + 1;   // smallest batch that takes it: from here on a root level fills a tile's 128 rows alone
                                              // (direct / ring, us, V = 151,936, r = 64: 64 requests 280 / 296, chains 353 / 382; 80: 327 / 304,
                                              // 572 / 458; 128: 458 / 429, 763 / 556; r = 256: 80 452 / 468, 128 646 / 655; V = 32,000: equal)
constexpr int TX_SOLO = 16;                // new parents whose seed bounds an owner makes itself (8: up to 6 % slower, 384 -> 409 us at 32 requests, Nmax 128; 32: within 1 %)
constexpr int TX_PIECE = 1024;             // tokens of one scouting item

// Everything the scan needs to know about one parent.
struct __align__(16) ParentEntry {
  int row;              // base-logit row: request * D + depth
  int token;
  uint64_t hash;
  float thrL, thrK;     // seed bounds: the parent's K best logits / keys are not below these (-inf: none known)
  float mref;           // reference of the sums of exponentials (an exact logit of the parent; -inf: none known)
  int req;
};
static_assert(sizeof(ParentEntry) == 32, "two 16-byte loads");

struct OwnerLayout { uint32_t pool, lse, toks, cand, flags, lists, seeds, total; };

struct TreeArgs {
  OwnerLayout own;
  const void *U, *A, *W;
  const void *Uscan, *Wscan;   // base logits and W as the scan reads them (a ragged vocabulary: copies with padded rows)
  int V, Vs;             // vocabulary; row stride of Uscan and Wscan
  int D, r, K, N, B;
  float T; uint64_t seed;
  int score_P;           // > 0: score this many given parents and stop (ts_score_parents)
  const int *p_req, *p_depth, *p_token; const uint64_t* p_hash;      // the given parents
  float *o_lse0, *o_lseT; int* o_top_tok; float* o_top_logit; int* o_draw_tok; float* o_draw_logit;
  // plan
  int wide_u;            // base-logit rows start on 32 bytes
  int TV, ntiles, BN, nW, npiece, w_over, use_tma, no_seed, ragged;
  int tail_copies;       // the last group of a list may hold its rows in copies
  int lstride;           // words between two rows' lists
  int rowsU;             // requests a stage of the base-logit ring holds
  uint32_t oL, oW, oX, oU;   // byte offsets of the selection state, the W ring, the fixed part and the base-logit ring
  uint32_t rk[20];       // round keys of the sampling generator
  // workspace
  ParentEntry* ent[2]; int* ent_slot[2];
  int *lvl_count, *seed_need; unsigned* barrier; int* err;   // seed_need[d]: some owner left the seed bounds of its parents of depth d to all CTAs
  float4* sums;                                    // [cap][ntiles]: max reference, sum, tempered sum of every tile
  int* cand_cnt[2]; uint2 *cand_top, *cand_key; float* cand_lg;   // candidates per parent: (value, token), and the keys' logits
                                                                 // (counts by level parity: an owner clears the next level's while others still read this one's)
  float2* res_lse; uint4* res_cand;                // merged results of a level with many parents: [cap], [cap][KMAX] (top token, logit, draw, logit)
  unsigned *thr, *slots; int cap;
  uint2* utop;                                     // [2][B][npiece] (given parents: [P][npiece]): best base logit of every piece of a row
  unsigned char* pool; size_t pool_stride;         // per request: PoolView
  int *req_npar, *req_base, *req_nscored; float* root_lseT; double2* req_caps;
  // expansion inputs and outputs
  const int* anchor; const float* theta; DevCalib calib; int calib_qT;
  int *n_nodes, *tok, *parent, *depth, *sib_rank; float *logS, *q0, *logqT, *logkey; int* pop_rank;
  uint64_t* node_hash; float* node_lseT; uint64_t* mask; int *n_scored, *status;
  int words;
  uint32_t wait_limit; int lost_arrival;
};

// A request's pool of admitted nodes, structure of arrays in one block (global memory between levels, shared memory
// while its owner works on it).
struct PoolView {
  double *key, *logS; uint64_t *hash, *path; float *q0, *logqT, *lseT; int *tok, *parent, *meta;   // meta = alive << 16 | depth << 8 | sibling rank
};
__host__ __device__ inline size_t pool_bytes(int N) { const size_t n = (size_t)((N + 1) & ~1); return n * 56; }
__device__ __forceinline__ PoolView pool_view(unsigned char* p, int N) {
  const size_t n = (size_t)((N + 1) & ~1);
  PoolView v;
  v.key = reinterpret_cast<double*>(p); v.logS = v.key + n;
  v.hash = reinterpret_cast<uint64_t*>(v.logS + n); v.path = v.hash + n;
  v.q0 = reinterpret_cast<float*>(v.path + n); v.logqT = v.q0 + n; v.lseT = v.logqT + n;
  v.tok = reinterpret_cast<int*>(v.lseT + n); v.parent = v.tok + n; v.meta = v.parent + n;
  return v;
}

// Rows of a parent's K candidates are padded to a power of two (no divisions on the owner's chain of instructions).
__host__ __device__ inline int slot_log2(int K) { return K <= 8 ? 3 : 4; }

// Bytes of shared memory the owner of a request works in (pool, merged results, candidates, seed columns).
// tokens evaluated for a parent's seed bounds: at least 2K (K <= 16), a power of two
__host__ __device__ inline int seed_log2(int K) { return K <= 4 ? 3 : (K <= 8 ? 4 : 5); }
__host__ __device__ inline int seed_count(int K) { return 1 << seed_log2(K); }
__host__ __device__ inline OwnerLayout owner_layout(int N, int K, int r) {
  OwnerLayout o; uint32_t at = 0;
  auto take = [&](size_t bytes) { uint32_t x = at; at = (uint32_t)((at + bytes + 15) & ~(size_t)15); return x; };
  o.pool = take(pool_bytes(N));
  o.lse = take((size_t)N * 3 * 4);              // lse0, lseT, pool slot of every parent
  const size_t KP = (size_t)1 << slot_log2(K);
  o.toks = take((size_t)N * KP * 4 * 4);        // top tokens, draw tokens, top logits, draw logits
  const size_t cand = (size_t)N * KP * 16, res = (size_t)N * seed_count(K) * 8;
  o.cand = take(cand > res ? cand : res);       // key, logS of every slot; later the seed values of the new parents
  o.flags = take((size_t)N * KP * 2);           // valid, index of the best unused token
  o.lists = take(256 * 4 * 5);                  // histogram / free slots, new slots, trip counts and offsets, new parents
  o.seeds = take((size_t)seed_count(K) * (r + 1) * 4 + 32 * 8);   // words of W holding the seed tokens' columns; tokens and base logits
  o.total = at;
  return o;
}

}  // namespace ts
