// Arguments of the tensor-core walk (ts_walk.cu).
#pragma once
#include "ts_internal.h"
#include "ts_scan.cuh"
#include "ts_tc.cuh"
#include "ts_zrow.cuh"

namespace ts {

// What a reduction at a node needs: its target row, its base-logit row, its token, the offsets of the two exponents (base 2).
struct __align__(16) NodeDesc { int64_t zrow; int urow, tok; float zoff, qoff, zmax, zlogs; };
static_assert(sizeof(NodeDesc) == 32, "two 16-byte loads");
constexpr int WK_COLS = 8;   // residual coefficients that one reduction evaluates at a node (ts_walk.cu says why several)
// An owner's request for a reduction: the node's record, the residual coefficients, and the step it is for (0: none).
struct __align__(16) WalkRec { NodeDesc node; float C[WK_COLS]; int nC, stamp, pad[2]; };
static_assert(sizeof(WalkRec) == 80, "five 16-byte loads");
struct __align__(16) WalkEdge { double px, qx, u; int x, pad; };   // accept test of one edge: target and draft probability, uniform, token
static_assert(sizeof(WalkEdge) == 32, "two 16-byte loads");

struct WalkArgs {
  const __nv_bfloat16 *U, *A, *W, *Z; const int64_t* z_row_off;
  int B, V, D, r, N; float T; uint64_t seed;
  const int *anchor, *n_nodes, *tok, *parent, *depth; const uint64_t* node_hash;
  const float *logqT, *node_lseT; const ZPart* z_part; int z_np;
  int *acc_len, *acc_node, *acc_tok, *bonus; float* edge_stat; uint32_t* flags; int* status;
  NodeDesc* node; int2* child; WalkEdge* edge; WalkRec* rec;
  float* part;   // [B][2 * WK_COLS][vt_n]: range sums of the residual at every coefficient, then of the proposal where the residual is positive
  unsigned* barrier;
  int vt_TV, vt_n, max_steps, ring, use_tma, req, cols, tr, lsets; uint32_t oB, oT, oP, oS;   // offsets of the head rows, the staged rows, the partial sums and the rest; ring > 0: blocks of 128 tokens of W stream through that many slots
  uint32_t wait_limit; int lost_arrival;
};

// A pass: `req` requests on `cols` accumulator columns; 2^`lsets` sets of four warps share a range's tiles, up to `tr` of a set in tensor memory together,
// and the parts that makes of all four the requests.
struct WalkPlan { int ring, req, cols, tr, lsets; uint32_t oB, oT, oP, oS; size_t smem; };
bool walk_plan(const ts_ctx* ctx, int B, bool tma, WalkPlan* out);
cudaError_t launch_walk_mma(ts_ctx* ctx, WalkArgs& a, char* ws, const WalkPlan& p, cudaStream_t st);

}  // namespace ts
