// Host-side declarations shared by the translation units of the library.
#pragma once

#include <vector>

#include <cuda.h>

#include "ts_common.cuh"
#include "ts_launch.h"

namespace ts {

int32_t set_error(int32_t code, const char* msg);
int32_t set_cuda_error(const char* where, cudaError_t e);

cudaError_t score_setup(ts_ctx* ctx);
cudaError_t verify_setup(ts_ctx* ctx);
cudaError_t expand_setup(ts_ctx* ctx);
cudaError_t walk_setup(ts_ctx* ctx);
size_t level_smem_bytes(const ts_config& c);

struct ScoreArgs {
  const void *U, *A, *W;
  int V, D, r, K;
  int P; const int* P_dev;
  int pdl;                 // host side: launch with programmatic stream serialization
  int few_cap;             // parents the few-parents kernel's records have room for
  const int *p_req, *p_depth, *p_token; const uint64_t* p_hash;
  float T; uint64_t seed;
  int TV, ntiles, cap;
  float* rec;
  unsigned* slots;  // [2][cap][K]: launch-wide lower bounds (logit, key) per parent, order-preserving encoding
};

struct MergeArgs {
  int P; const int* P_dev; int K, ntiles, cap; float T;
  int pdl;   // host side: launch with programmatic stream serialization
  int few_ntiles, few_cap;   // few_ntiles > 0: the level was scored by the few-parents kernel over this many tiles
  const float* rec; unsigned* slots;
  float *lse0, *lseT; int* top_tok; float* top_logit; int* draw_tok; float* draw_logit;
};

// Bytes of record scratch a scoring pass over up to P parents needs, and the slot capacity it implies.
size_t score_scratch_bytes(const ts_ctx* ctx, int P, int* cap_out);
// The pruning slots sit behind the records; they must be zero before a launch and
// the merge kernel leaves them zero again.
unsigned* thr_base(const ts_ctx* ctx, float* rec, int cap);
size_t thr_bytes(const ts_ctx* ctx, int cap);

// Scoring pass + merge for a parent list whose length is P (host) or *P_dev (device) when P_dev is set;
// p_bound: an upper bound of *P_dev the host knows (-1: none).  A list that cannot exceed few_cap parents
// goes to the few-parents kernel where the context has one.
// rec: record scratch of score_scratch_bytes(ctx, max parents) bytes with slot capacity cap.
cudaError_t launch_score(const ts_ctx* ctx, float* rec, int cap, const void* U, const void* A, const void* W,
                         int P, const int* P_dev, const int* p_req, const int* p_depth, const int* p_token,
                         const uint64_t* p_hash, float T, uint64_t seed, float* lse0, float* lseT, int* top_tok,
                         float* top_logit, int* draw_tok, float* draw_logit, cudaStream_t st,
                         bool pdl = false, int p_bound = -1);

// Kernel launch, optionally with programmatic stream serialization: the kernel may then start while the
// kernel before it in the stream is still running, and must execute pdl_wait() before it touches anything
// that kernel (or, transitively, an earlier one) wrote.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                                 Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Cooperative launch (grid barriers: every CTA resident), chained to the kernel before it where the driver takes both
// attributes.
inline cudaError_t launch_cooperative(int& refused, const void* kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t st, void** kargs) {
  return launch_chained(refused, [&](bool chained) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative; attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization; attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = chained ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, kargs);
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
  });
}

// Lets a kernel ask for all the dynamic shared memory that its static arrays leave.  The limit is the process's, not a
// context's: a context's own plan as the limit would lower it for the contexts made before.
template <typename... KArgs>
inline cudaError_t allow_all_smem(void (*kernel)(KArgs...), int max_smem) {
  cudaFuncAttributes fa;
  const cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem - (int)fa.sharedSizeBytes);
}

// the few-parents kernel (ts_score_few.cu)
int few_tiles(const ts_config& c);
int few_capacity(const ts_config& c, bool use_tree);
cudaError_t launch_score_few(const ts_ctx* ctx, const ScoreArgs& a, int p_bound, cudaStream_t st);
// tensor maps (ts_tmap.cu), encoded or found cached in the context; false: not available.  Of W [r][V] for the walk
// and of the one-launch kernel's [r][stride] matrix: boxes of 64 tokens x r rows rounded up to 16.
bool w_tensor_map(ts_ctx* ctx, const void* W);
bool tree_tensor_map(ts_ctx* ctx, const void* W, int stride, CUtensorMap* out);
// of base logits [B][D][stride], boxes of 64 tokens x one depth x `rows` requests
bool u_tensor_map(ts_ctx* ctx, const void* U, int stride, int B, int rows, CUtensorMap* out);

// the one-launch expansion and scoring (ts_tree.cu)
struct TreeOut {
  int *n_nodes, *tok, *parent, *depth, *sib_rank; float *logS, *q0, *logqT, *logkey; int* pop_rank;
  uint64_t* node_hash; float* node_lseT; uint64_t* mask; int *n_scored, *status;
};
bool tree_plan(const ts_config& c, int num_sms, int max_smem, TreePlan* out);
cudaError_t tree_setup(ts_ctx* ctx);
size_t tree_score_bytes(const ts_ctx* ctx, int P);
cudaError_t tree_score(ts_ctx* ctx, char* scratch, const void* U, const void* A, const void* W, int P, const int* p_req, const int* p_depth, const int* p_token,
                       const uint64_t* p_hash, float T, uint64_t seed, float* lse0, float* lseT, int* top_tok, float* top_logit, int* draw_tok,
                       float* draw_logit, int rows, cudaStream_t st);
cudaError_t tree_expand(ts_ctx* ctx, char* ws, const TreeOut& o, const void* U, const void* A, const void* W, int B, const int* anchor, const float* theta,
                        float T, uint64_t seed, cudaStream_t st);

enum KernelId { K_INIT, K_SCORE, K_MERGE, K_LEVEL, K_FINAL, K_ZROWS, K_GREEDY, K_WALK, K_SCORE_FEW, K_ALLOC_SELECT, K_ALLOC_CUT, K_CALIB_ACC, K_CALIB_FIT, K_ATTN_INPUTS, K_PERSIST, K_COUNT };

struct Prof {
  bool on = false;
  std::vector<cudaEvent_t> ev;  // pairs: start, stop
  std::vector<int> ids;
  size_t used = 0;
  int64_t launches[K_COUNT] = {};
};

// Brackets one kernel launch with an event pair when instrumentation is on; always counts it.
struct ProfScope {
  Prof* p; cudaStream_t st; size_t slot; bool rec;
  ProfScope(const ts_ctx* ctx, int id, cudaStream_t s) : p((Prof*)ctx->prof), st(s), slot(0), rec(false) {
    if (!p) return;
    p->launches[id]++;
    if (p->on && p->used < p->ids.size()) {
      slot = p->used++; p->ids[slot] = id; rec = true;
      cudaEventRecord(p->ev[2 * slot], st);
    }
  }
  ~ProfScope() { if (rec) cudaEventRecord(p->ev[2 * slot + 1], st); }
};

inline bool bad_ptr(const void* p) { return !p || ((uintptr_t)p & 15u); }

}  // namespace ts
