// The recursive-rejection walk of the verification at T > 0 (Section 3.3) on the 5th-generation tensor cores: one
// cooperative launch, one CTA per vocabulary range.
//
// A request's walk is a scalar sequence (see ts_verify.cu for the algebra): sibling tests until one is accepted or a
// rejection needs Z = sum_w max(p(w) - C q(w), 0).  A step of the kernel is
//   advance   the CTA that owns a request adds up its range sums, and one of its warps runs the scalar sequence on state in
//             shared memory and publishes what its next reduction needs (80 bytes a request, no list and no counter);
//   barrier
//   reduce    every CTA reads those records and sums its range for all requests that asked: the draft logits are one MMA
//             tile per 128 tokens with the TOKENS on the 128 rows (W is the A operand, as it lies in memory) and the
//             requests on the columns, so that a thread holds one token and the work is in proportion to the requests.
//             (With the requests on the rows a step with three of them cost as much as one with 32; late steps have few.)
//   barrier
// When no request asks any more, every owner draws its requests' bonus tokens by itself: the range from the stored
// range sums, then the token inside it.  Two barriers a step and none at the start and the end.
//
// Measured at 32 requests, V = 151,936, r = 64 (several of them reject eight siblings): 106 us in five steps; with one coefficient a
// reduction it was nine steps and 146.  A step: sums and advance 3 to 7 (predictions), barriers 1.1 and 1.5, operands 2, the pass 18 (all
// requests, grid), 12 and 10 (a few, eight coefficients), 3 (one request, one coefficient).  Set-up 6, bonus draws 11.
#include <math.h>
#include <string.h>

#include "ts_walk.cuh"

namespace ts {

constexpr int WK_EPI = 16;                 // warps that read accumulators: 4 lane quarters x 4 sets of tiles
constexpr int WK_LOAD = WK_EPI;            // tensor memory; in the streaming form it requests W and issues the MMAs
constexpr int WK_THREADS = (WK_EPI + 1) * 32;
constexpr int WK_TR = 3;                   // tiles of a set in tensor memory together at most: WalkArgs::tr of them; a round is four sets' (512 columns)
constexpr int WK_ROUND = 4 * WK_TR;
constexpr int WK_VALS = 2 * WK_COLS;       // sums of a request: residual and proposal mass at every coefficient
constexpr int WK_GRID = 16;                // beside the number of coefficients: all but the first are guesses from the grid
__host__ __device__ constexpr int wk_seg(bool aligned) { return aligned ? 64 : 80; }   // bytes of a staged segment: 32 tokens that, unaligned, may start anywhere in a 16-byte chunk
constexpr int WK_STATIC = 2048;            // static shared memory at most
constexpr int WK_CHUNK = 1088;             // tokens of one step of the bonus rescan: 8 tokens x 136 places x 4 slices of the rank
constexpr size_t WK_DOT = 4 * WK_CHUNK * sizeof(float);   // shared memory of the rescan
constexpr double WK_TOL = 9.5367431640625e-7;   // 2^-20: a coefficient this close (relative) to an evaluated one counts as evaluated
constexpr double WK_REL = 6.103515625e-5;       // 2^-14: and the step to it times the proposal mass may be this much of the residual

// A request of a pass.  b: its number; rows that may start anywhere: and where in a 16-byte chunk the two do (bits 28, 24).
struct __align__(16) RedDesc { const __nv_bfloat16 *z, *u; float zoff, qoff; int b, nC; float C[WK_COLS]; };
static_assert(sizeof(RedDesc) == 64, "four 16-byte loads");

// The walk of one request.
struct WalkState {
  int cur, j, acc, nf, npass, phase;       // phase: 0 walking, 1 waits for the sum after a rejection, 2 waits for the sum of the bonus draw, 3 walk over, 4 not walked
  int cfirst, ccnt;
  int nC, pcol;                            // coefficients of the last reduction (| WK_GRID); the one that the bonus draw's range sums belong to
  float col[WK_COLS];
  double C, Zj, Qused, passC, partsC;      // partsC: the C that the stored range sums were computed for (-1: none)
  double S[WK_VALS];                       // the last reduction's sums
  double fC[KMAX];                         // residual coefficients that the siblings tested so far keep
};

struct WalkSm {
  unsigned char *Ws, *Bs, *stage; float* part; RedDesc* desc; int* tok; WalkState* st;
  uint64_t *t_full, *t_empty, *w_full, *w_free; uint32_t* tmem; volatile int* abort;
};

__device__ __forceinline__ bool wk_wait(uint64_t* bar, uint32_t parity, const WalkArgs& a, volatile int* abort) {
  return mbar_try_wait(bar, parity) || mbar_wait(bar, parity, abort, nullptr, a.wait_limit);
}
// instruction descriptor: D = f32, A = B = bf16, A MN-major (tokens contiguous), B K-major, M = 128, N = n
__device__ __forceinline__ uint32_t wk_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}

// ---- set-up of one request, by the whole CTA: child ranges, accept-test inputs of every edge, what a reduction at a node needs ----
__device__ __forceinline__ void wk_setup(const WalkArgs& a, WalkState& st, const int b, int* s_par, int* s_tok, float2* s_z) {
  const int tid = threadIdx.x, N = a.N;
  const size_t nb = (size_t)b * N, cb = (size_t)b * (N + 1);
  const int n = a.n_nodes[b];
  const bool okn = n >= 0 && n <= N;
  const int64_t row0 = a.z_row_off[b];
  const float invT = 1.f / a.T;
  constexpr float LOG2E = 1.4426950408889634f;
  const int64_t zq = zrow_piece(a.z_row_off[a.B] * a.V, a.V, a.z_np);
  // non-finite inputs: a target row with a NaN (its maximum is NaN), without finite mass, or a node whose proposal
  // log-probability is NaN (its expansion was reported TS_ERR_NUMERIC) -- the request is not walked
  int bad = 0;
  if (okn) {
    for (int i = tid; i <= n; i += WK_THREADS) {
      const int par = i ? a.parent[nb + i - 1] : -1, dep = i ? a.depth[nb + i - 1] : 0, tok = i ? a.tok[nb + i - 1] : a.anchor[b];
      const float ls = a.node_lseT[cb + i], lq = i ? a.logqT[nb + i - 1] : 0.f;
      const ZRow zr = zrow_fold(a.z_part, row0 + i, a.V, zq, a.z_np, a.T);
      const float zm = zr.m, zl = zr.logs;
      s_z[i] = make_float2(zm, zl);
      bad |= (zm != zm || isinf(zm) || zl != zl || isinf(zl) || lq != lq) ? 1 : 0;
      if (i) { s_par[i - 1] = par; s_tok[i - 1] = tok; }
      NodeDesc nd;
      nd.zrow = row0 + i; nd.urow = b * a.D + min(dep, a.D - 1);   // (a leaf at depth D asks only for its target row: keep the base row inside U)
      nd.tok = tok; nd.zoff = (-zm * invT - zl) * LOG2E; nd.qoff = -ls * LOG2E; nd.zmax = zm; nd.zlogs = zl;
      const uint4* src = reinterpret_cast<const uint4*>(&nd); uint4* dst = reinterpret_cast<uint4*>(a.node + cb + i);
      dst[0] = src[0]; dst[1] = src[1];
      a.child[cb + i] = make_int2(-1, 0);
    }
  }
  if (tid == 0) { st.cfirst = -1; st.ccnt = 0; }
  bad = __syncthreads_or(bad);
  for (int i = tid; okn && i < n; i += WK_THREADS) {
    if (bad) { if (a.edge_stat) a.edge_stat[nb + i] = 0.f; continue; }
    const int par = s_par[i];
    int j = 0;   // place among the siblings (they are contiguous)
    while (i - j - 1 >= 0 && s_par[i - j - 1] == par) ++j;
    if (j == 0) {
      int m = 1;
      while (i + m < n && s_par[i + m] == par) ++m;
      a.child[cb + par + 1] = make_int2(i, m);
      if (par < 0) { st.cfirst = i; st.ccnt = m; }
    }
    const int64_t row = row0 + par + 1;
    const int x = s_tok[i];
    const double lp = ((double)__bfloat162float(a.Z[row * a.V + x]) - (double)s_z[par + 1].x) / (double)a.T - (double)s_z[par + 1].y;
    const double lq = (double)a.logqT[nb + i];
    WalkEdge e;
    e.px = exp(lp); e.qx = exp(lq); e.x = x; e.pad = 0;
    e.u = u01(stream_words(a.seed, b, a.node_hash[cb + par + 1], STREAM_ACCEPT, (uint32_t)j).x);
    const uint4* src = reinterpret_cast<const uint4*>(&e); uint4* dst = reinterpret_cast<uint4*>(a.edge + nb + i);
    dst[0] = src[0]; dst[1] = src[1];
    if (a.edge_stat) a.edge_stat[nb + i] = (float)exp(fmin(lp - lq, 0.0));
  }
  for (int i = tid; i < a.D; i += WK_THREADS) { a.acc_node[(size_t)b * a.D + i] = -1; a.acc_tok[(size_t)b * a.D + i] = -1; }
  __syncthreads();
  if (tid == 0) {
    st.cur = -1; st.j = 0; st.acc = 0; st.nf = 0; st.npass = 0; st.phase = 0;
    st.C = 0.0; st.Zj = 1.0; st.Qused = 0.0; st.passC = 0.0; st.partsC = -1.0;
    st.nC = 0; st.pcol = 0;
    a.flags[b] = 0u;
    a.status[b] = !okn ? TS_ERR_INVALID : (bad ? TS_ERR_NUMERIC : TS_OK);
    if (!okn || bad) { st.phase = 4; a.acc_len[b] = 0; a.bonus[b] = -1; }
  }
  __syncthreads();
}

// ---- one request's scalar sequence, by one warp ------------------------------------------------------------------------
// Everything it may need -- the reduction's sums, the current node's children, the record of the current node -- is
// requested together: one memory round trip a step, and one more for every node it descends to.
//
// Several coefficients a reduction.  Rejecting sibling after sibling at one node needs F(C) = sum_w max(p - C q, 0) at
// C_1 = 1 < C_2 < ..., and C_(i+1) follows from F(C_i): one reduction after the other, 8 (K = 8) or 16 steps for a request
// that rejects all children, and the slowest request sets the length of the launch.  But F is convex with slope -G(C),
// G = the proposal mass where the residual is positive, and nothing in the sequence depends on the uniforms.  So a reduction evaluates
// F and G at several coefficients: the one that is needed, and guesses of the ones after it.  At first the guesses are a
// fixed grid (there the sums are of |p - C q|, two instructions a token and coefficient: F = (1 - C + sum |p - C q|) / 2, good
// enough for guesses); from its values (cubic interpolation of what the node's other tokens give; the children's own terms are known
// exactly) the rest of the sequence is predicted, evaluated, and where a prediction was within 2^-20 of what its
// predecessors turn out to give, F there is F and G at the prediction, to first order.  The term left out is at most the step times the
// proposal mass whose ratio p / q lies inside the step: some per cent of G where a tie of logits lies there, all of it only where no more than the step
// times G is left of F.  So the step times G may be 2^-14 of F at most, which keeps the term below the rounding of the
// exponentials.  (2^-20 costs 32 requests 5 us of 140.  A grid's slopes come from a parabola: its coefficients stand for themselves only, as
// does one that was evaluated alone.)  Where the prediction was not close enough, the next reduction evaluates the corrected
// predictions (errors go down quadratically).  A node's eight rejections take three reductions, sixteen take four or five.
__device__ __forceinline__ double wk_lanes_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}
__device__ __forceinline__ void wk_advance(const WalkArgs& a, WalkState& st, const int b, const int lane, const int stamp) {
  const int N = a.N;
  const size_t nb = (size_t)b * N, cb = (size_t)b * (N + 1);
  WalkRec* rec = a.rec + b;
  if (st.phase >= 3) { if (lane == 0) rec->stamp = 0; return; }
  int v = st.cur, first = st.cfirst, m = st.ccnt;
  WalkEdge e;
  auto fetch = [&]() {
    e.px = 0.0; e.qx = 1.0; e.u = 0.0; e.x = -1;
    if (lane < m) { const uint4* s = reinterpret_cast<const uint4*>(a.edge + nb + first + lane); uint4* d = reinterpret_cast<uint4*>(&e); d[0] = __ldcg(s); d[1] = __ldcg(s + 1); }
  };
  fetch();
  uint4 nd = make_uint4(0u, 0u, 0u, 0u);
  if (lane < 2) nd = __ldcg(reinterpret_cast<const uint4*>(a.node + cb + v + 1) + lane);
  const bool grid = (st.nC & WK_GRID) != 0;
  int kind = st.phase, have = kind ? st.nC & (WK_GRID - 1) : 0;
  bool fresh = true;   // the first coefficient is passC's own, whatever its value
  // lane k: the k-th coefficient of the reduction that just ran, and its sums over all tokens but the children
  double ck = 0.0, Fk = 0.0, Gk = 0.0;
  if (have) {
    if (lane < have) { ck = (double)st.col[lane]; Fk = st.S[lane]; Gk = st.S[WK_COLS + lane]; }
    if (grid && lane > 0 && lane < have) Fk = 0.5 * (1.0 - ck + Fk);   // (both distributions sum to one)
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
      const double p = __shfl_sync(0xFFFFFFFFu, e.px, i), q = __shfl_sync(0xFFFFFFFFu, e.qx, i), t = p - ck * q;
      if (t > 0.0) { Fk -= t; Gk -= q; }
    }
    if (have == 1) Gk = 0.0;   // (not computed: the step is the rounding of one coefficient to fp32)
    else if (grid) {           // slopes by the parabola through a coefficient and its neighbours
      const int k0 = min(max(lane - 1, 0), have - 3);
      const double c0 = __shfl_sync(0xFFFFFFFFu, ck, k0), c1 = __shfl_sync(0xFFFFFFFFu, ck, k0 + 1), c2 = __shfl_sync(0xFFFFFFFFu, ck, k0 + 2);
      const double f0 = __shfl_sync(0xFFFFFFFFu, Fk, k0), f1 = __shfl_sync(0xFFFFFFFFu, Fk, k0 + 1), f2 = __shfl_sync(0xFFFFFFFFu, Fk, k0 + 2);
      const double d01 = (f1 - f0) / (c1 - c0), d12 = (f2 - f1) / (c2 - c1);
      Gk = fmax(-(d01 + (d12 - d01) / (c2 - c0) * (2.0 * ck - c0 - c1)), 0.0);
    }
  }
  for (;;) {
    if (kind) {   // ---- the sum at passC: from the reduction that just ran, or by another one ----
      const double C = st.passC;
      const int nf = st.nf;
      const double off = fabs(C - ck);
      const unsigned hit = __ballot_sync(0xFFFFFFFFu, lane < have && ((lane == 0 && fresh) || (have > 1 && !grid && off <= WK_TOL * C && off * Gk <= WK_REL * fmax(Fk, 0.0))));
      fresh = false;
      // a child's own term: the residual it had when it was tested, or the one it has
      double own = lane < m ? fmax(e.px - (lane < nf && lane < KMAX ? st.fC[lane] : C) * e.qx, 0.0) : 0.0;
      if (!hit) {
        int nC = 1;
        float mine = (float)C;   // lane k: coefficient k
        const int need = kind == 2 ? 1 : m - nf + 1;   // sums that this node can still ask for
        if (need > 2 && have <= 1) {   // (of two sums the second's coefficient follows from the first)
          nC = WK_COLS | WK_GRID;
          constexpr float places[WK_COLS] = {1.f, 1.2f, 1.45f, 1.75f, 2.15f, 2.7f, 3.6f, 5.5f};
          float g = 1.f;
#pragma unroll
          for (int k = 1; k < WK_COLS; ++k) g = lane == k ? places[k] : g;
          mine = (float)C * g;
        } else if (need > 1 && have > 1) {
          // what does not depend on the sequence, by all lanes at once: lane i's 1 / (1 - proposal mass of the siblings before
          // it), lane k's 1 / (width of interval k)
          double Q = e.qx;
          if (lane >= m) Q = 0.0;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) { const double x = __shfl_up_sync(0xFFFFFFFFu, Q, o); if (lane >= o) Q += x; }
          Q = __shfl_up_sync(0xFFFFFFFFu, Q, 1);
          if (lane == 0) Q = 0.0;
          const float inv = Q < 1.0 ? (float)(1.0 / (1.0 - Q)) : 0.f, ckf = (float)ck, Fkf = (float)Fk, Gkf = (float)Gk;
          const float next = __shfl_down_sync(0xFFFFFFFFu, ckf, 1), rh = lane + 1 < have && next > ckf ? 1.f / (next - ckf) : 0.f;
          // (guesses in fp32, the sum of the steps in double: some 2e-7 of rounding, a quarter of what WK_TOL allows)
          const float pf = lane < m ? (float)e.px : 0.f, qf = lane < m ? (float)e.qx : 1.f;
          float mass = (float)own;
          double c = C;
#pragma unroll 1
          for (int i = nf; i < m && nC < WK_COLS; ++i) {
            // the other tokens' share at c: between two evaluated coefficients by Hermite's cubic, beyond the last by the decay there
            const float cf = (float)c;
            const int n = __popc(__ballot_sync(0xFFFFFFFFu, lane < have && ckf <= cf));
            const int k0 = n > 0 ? n - 1 : 0, k1 = n < have ? n : have - 1;
            const float c0 = __shfl_sync(0xFFFFFFFFu, ckf, k0), f0 = __shfl_sync(0xFFFFFFFFu, Fkf, k0), g0 = __shfl_sync(0xFFFFFFFFu, Gkf, k0);
            const float c1 = __shfl_sync(0xFFFFFFFFu, ckf, k1), f1 = __shfl_sync(0xFFFFFFFFu, Fkf, k1), g1 = __shfl_sync(0xFFFFFFFFu, Gkf, k1);
            const float w = __shfl_sync(0xFFFFFFFFu, rh, k0), scale = __shfl_sync(0xFFFFFFFFu, inv, i);
            float sum = mass;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
            const float dc = (float)(c - (double)c0);
            float f;
            if (n == 0) f = f0 - dc * g0;
            else if (n == have) f = f0 > 1e-30f ? f0 * __expf(-dc * g0 / f0) : 0.f;
            else {
              const float h = c1 - c0, t = dc * w, r = 1.f - t;
              f = r * r * (f0 * (1.f + 2.f * t) - g0 * h * t) + t * t * (f1 * (3.f - 2.f * t) + g1 * h * r);
            }
            const float z = fmaxf(f, 0.f) + sum;
            if (!(z > 1e-30f) || scale == 0.f) break;   // uniform
            c += (double)(z * scale);
            if (lane < m && lane >= i) mass = fmaxf(fmaf(-(float)c, qf, pf), 0.f);   // (sibling i keeps this from now on)
            if (lane == nC) mine = (float)c;
            ++nC;
          }
        }
        const int cols = nC & (WK_GRID - 1);
        if (lane < 2) reinterpret_cast<uint4*>(rec)[lane] = nd;
        if (lane < WK_COLS) { const float x = lane < cols ? mine : 0.f; rec->C[lane] = x; st.col[lane] = x; }
        if (lane == 0) { rec->nC = nC; rec->stamp = stamp; st.nC = nC; st.phase = kind; }
        __syncwarp();
        return;
      }
      const int k = __ffs(hit) - 1;
      const double c0 = __shfl_sync(0xFFFFFFFFu, ck, k), f0 = __shfl_sync(0xFFFFFFFFu, Fk, k), g0 = __shfl_sync(0xFFFFFFFFu, Gk, k);
      const double Cf = (double)(float)C;   // (sums are of the coefficient as fp32 holds it, by whichever way they come)
      const double step = fabs(Cf - c0) <= 2.0 * WK_TOL * Cf ? Cf - c0 : 0.0;   // (one beyond what fp32 holds: no step)
      const double f = f0 - step * g0 + wk_lanes_sum(own);
      __syncwarp();
      if (lane == 0) {
        st.npass++;
        if (kind == 1) {
          if (f <= 1e-30 * st.Zj) {   // the residual lost its mass: keep the previous one
            a.flags[b] |= TS_FLAG_ZERO_MASS;
            st.fC[st.nf - 1] = st.C;
            st.partsC = -1.0;
          } else { st.C = C; st.Zj = f; st.partsC = C; st.pcol = k; }
        } else { st.Zj = f; st.partsC = C; st.pcol = k; }
        st.phase = 0;
      }
      kind = 0;
      __syncwarp();
    }
    // the sibling chain at node v until one is accepted, a sum is needed, or they run out; all lanes follow it together
    const int j = st.j;
    const double C = st.C, c0 = st.Zj, Q = st.Qused;
    if (j < m && st.acc < a.D) {
      const double px = __shfl_sync(0xFFFFFFFFu, e.px, j), qx = __shfl_sync(0xFFFFFFFFu, e.qx, j), u = __shfl_sync(0xFFFFFFFFu, e.u, j);
      const int x = __shfl_sync(0xFFFFFFFFu, e.x, j);
      const double cj = c0 / (1.0 - Q);
      const double rho = fmin(1.0, fmax(px / qx - C, 0.0) / cj);
      __syncwarp();
      if (u < rho) {   // descend
        if (lane == 0) {
          a.acc_node[(size_t)b * a.D + st.acc] = first + j; a.acc_tok[(size_t)b * a.D + st.acc] = x;
          st.acc++; st.cur = first + j; st.j = 0; st.C = 0.0; st.Zj = 1.0; st.Qused = 0.0; st.nf = 0; st.partsC = -1.0;
        }
        v = first + j;
        const int2 c = __ldcg(a.child + cb + v + 1);
        first = c.x; m = c.y; have = 0;
        if (lane < 2) nd = __ldcg(reinterpret_cast<const uint4*>(a.node + cb + v + 1) + lane);
        if (lane == 0) { st.cfirst = first; st.ccnt = m; }
        fetch();
      } else {
        if (lane == 0) {
          const int k = st.nf;
          st.fC[k] = C + cj; st.nf = k + 1;
          st.Qused = Q + qx; st.j = j + 1; st.passC = C + cj;
        }
        kind = 1;
      }
    } else if (st.partsC != C) {
      __syncwarp();
      if (lane == 0) st.passC = C;
      kind = 2;
    } else {
      __syncwarp();
      if (lane == 0) { st.phase = 3; rec->stamp = 0; }
      __syncwarp();
      return;
    }
    __syncwarp();
  }
}

// ---- one reduction pass: sums over this CTA's tokens for up to WK_REQ requests ------------------------------------------------
// The MMAs of one tile into accumulator place `slot` of the round, W from slab pair `ws`; an elected lane of the calling warp.
// Issuing costs about 70 cycles an instruction (400 a tile of rank 64; 600 from a branch on the lane instead of an elected one,
// and 1200 beside busy warps): one warp for all nine tiles of a pass took longer than the sums, so where W is resident the
// first warp of every set issues its set's tiles.
__device__ __forceinline__ void wk_mma(const WalkArgs& a, const WalkSm& sm, const int ncol, const uint32_t ws, const uint32_t slot, const uint32_t tmem_base) {
  const int ksteps = (a.r + 15) / 16;
  const uint32_t slab = (uint32_t)ksteps * 2048u;
  tc_fence_after();
  if (elect_one()) {
    const uint64_t ad = smem_desc(smem_u32(sm.Ws) + 2u * ws * slab, slab, 1024u), bd = smem_desc(smem_u32(sm.Bs), 16u, 1024u);
    const uint32_t idesc = wk_idesc(ncol), d = tmem_base + slot * (uint32_t)a.cols;
#pragma unroll 4
    for (int ks = 0; ks < ksteps; ++ks)
      mma_bf16(d, ad + (uint64_t)(ks * 128), bd + (uint64_t)((ks >> 2) * (a.cols * 8) + (ks & 3) * 2), idesc, ks > 0 ? 1u : 0u);
    mma_commit(sm.t_full + slot);
    if (a.ring) mma_commit(sm.w_free + ws);
  }
  __syncwarp();
}
// the accumulators are free for round `rnd` (counted over all passes) when all warps are done with the round before
__device__ __forceinline__ bool wk_drained(const WalkArgs& a, const WalkSm& sm, const uint32_t rnd) {
  return rnd == 0u || __all_sync(0xFFFFFFFFu, wk_wait(sm.t_empty, (rnd - 1u) & 1u, a, sm.abort));
}
// Streaming form, one warp: blocks of 128 tokens of W through the ring, one after the other round the range and on into the next
// pass (W does not depend on which requests that sums), and the tiles in the same order.  (In order, and by one warp: a wait
// for a parity tells a slot's turns apart only while the waiter follows every one of them.)
__device__ __forceinline__ void wk_stream(const WalkArgs& a, const WalkSm& sm, const CUtensorMap* tm, const int ncol, const int t0, const int tlen, const uint32_t pass,
                                          uint32_t& wreq, uint32_t& rnd, const uint32_t tmem_base) {
  const int ntile = (tlen + 127) / 128, round = a.tr << a.lsets;
  const uint32_t slab = (uint32_t)((a.r + 15) / 16) * 2048u, ring = (uint32_t)a.ring, w0 = pass * (uint32_t)ntile;
  for (int t = 0; t <= ntile; ++t) {
    for (const uint32_t upto = w0 + (uint32_t)t + ring; wreq < upto; ++wreq) {
      const uint32_t slot = wreq % ring, use = wreq / ring;
      if (use >= 1 && !__all_sync(0xFFFFFFFFu, wk_wait(sm.w_free + slot, (use - 1) & 1, a, sm.abort))) return;
      const int nb = (int)(wreq % (uint32_t)ntile), ns = (tlen - nb * 128 > 64) ? 2 : 1;
      if (elect_one()) {
        mbar_expect_tx(sm.w_full + slot, (uint32_t)ns * slab);
        for (int h = 0; h < ns; ++h) tma_load_box(sm.Ws + (size_t)(2 * slot + h) * slab, tm, t0 + nb * 128 + h * 64, 0, sm.w_full + slot);
      }
      __syncwarp();
    }
    if (t == ntile) break;
    const uint32_t x = w0 + (uint32_t)t;
    const int i = t % round;
    if (i == 0 && t > 0) ++rnd;
    if (i == 0 && !wk_drained(a, sm, rnd)) return;
    if (!__all_sync(0xFFFFFFFFu, wk_wait(sm.w_full + x % ring, (x / ring) & 1, a, sm.abort))) return;
    wk_mma(a, sm, ncol, x % ring, (uint32_t)i, tmem_base);
  }
  ++rnd;
}

// Of the four sets of warps, how many (as a power of two) share the tiles: the plan's, or more for one pair of requests or two; the rest share the requests.
__device__ __forceinline__ int wk_sets(const WalkArgs& a, const int nreq) { return nreq > 4 ? a.lsets : (nreq > 2 ? max(a.lsets, 1) : 2); }

// Sums of N values over the lanes: halve the values while halving the lanes; lane (32 / N) v ends with value v.
template <int N>
__device__ __forceinline__ float wk_fold(float* x, const int lane) {
#pragma unroll
  for (int h = N / 2, o = 16; o > 0; h >>= 1, o >>= 1) {
    if (h >= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < N / 2; ++k)
        if (k < h) {
          const float give = up ? x[k] : x[k + h], keep = up ? x[k + h] : x[k];
          x[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
        }
    } else x[0] += __shfl_xor_sync(0xFFFFFFFFu, x[0], o);
  }
  return x[0];
}

// Number of sums of a request with so many coefficients (values 0 .. WK_COLS-1: residuals, or on the grid absolute differences;
// from WK_COLS on: proposal masses).
__device__ __forceinline__ bool wk_has(const int nC, const int val) {
  const int cols = nC & (WK_GRID - 1);
  return val < WK_COLS ? val < cols : (cols > 1 && !(nC & WK_GRID) && val - WK_COLS < cols);
}

// The scanning warps.  A warp holds the accumulators of 32 tokens in each of its set's tiles, up to three, and goes through the requests two
// at a time: a request's chain of waits, loads and exponentials is some 600 cycles, so two go through it together, and what does not depend on
// the request is worked out before the loop.  Their rows come through shared memory by 16-byte copies (AL: rows start on 16 bytes),
// requested when the pair before has been read: one and two pairs further ahead cost 12 to 30 KB each and were no faster, the four warps
// of a scheduler cover for one another.  One request at a time, with the copies' addresses and sizes worked out for every one, a pass of 32 requests
// and one coefficient took 23 us instead of 14; two-byte loads by every token's thread 18.
// A request's several coefficients cost a warp a sum over its lanes each, so the tiles are shared by as few sets of four warps as hold them, and
// the sets that are left take every second or all but every fourth pair instead; with one pair (two pairs) the tiles go to all sets (two).
template <bool AL>
__device__ __forceinline__ void wk_epilogue(const WalkArgs& a, const WalkSm& sm, const int nreq, const int ncol, const int t0, const int tlen,
                                            const uint32_t tmem_base, uint32_t& used, uint32_t& rnd, const bool first_pass) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = warp & 3, ls = wk_sets(a, nreq), sets = 1 << ls, set = (warp >> 2) & (sets - 1), part = warp >> (2 + ls), nparts = 4 >> ls;
  const int ntile = (tlen + 127) / 128;
  const float zs = (1.f / a.T) * 1.4426950408889634f;   // exponentials as powers of two
  float* mine = sm.part + (size_t)warp * a.req * WK_VALS;
  constexpr int CPS = AL ? 4 : 5;                       // 16-byte copies of a segment
  constexpr uint32_t SEG = wk_seg(AL);
  const uint32_t SLOT = 2u * (uint32_t)a.tr * SEG;      // a request's segments
  const uint32_t dbase = smem_u32(sm.desc), place = smem_u32(sm.stage) + (uint32_t)warp * 2u * SLOT;
  const int seg = lane / CPS, ch = lane - seg * CPS;    // lane's copy of a request: 16 bytes of one segment (tile, row)
  bool alive = true;
  const int round = a.tr << a.lsets, step = 128 << ls;   // (a round is the plan's, however many sets share it)
  for (int r0 = 0; r0 < ntile; r0 += round, ++rnd) {
    const int left = min(ntile - r0, round) - set, ntl = left > 0 ? (left + sets - 1) >> ls : 0;   // the set's tiles: r0 + set + sets i
    const int tok = (r0 + set) * 128 + q * 32;                                              // the warp's first token in the first of them; then + step i
    int nt = 0;                                                                             // its tiles with any token
#pragma unroll
    for (int i = 0; i < WK_TR; ++i) if (i < ntl && tok + step * i < tlen) nt = i + 1;
    const bool tail = nt > 0 && tok + step * (nt - 1) + 32 > tlen;                          // (uniform) the last of them is cut short
    const int o = tok + step * (seg >> 1), nv = min(32, tlen - o);
    const bool act = seg < 2 * nt && (!AL || 8 * ch < nv);
    const uint64_t off = 2ull * (uint64_t)(uint32_t)(t0 + o) + 16u * (uint32_t)ch;
    const int bytes = 2 * nv - 16 * ch;                                                     // of the segment from the lane's chunk on
    const uint32_t from = dbase + (uint32_t)(seg & 1) * 8u, to = place + (uint32_t)seg * SEG + (uint32_t)ch * 16u;
    auto stage = [&](int j) {   // requests j and j + 1
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (act && j + h < nreq) {
          uint64_t row;
          asm volatile("ld.shared.u64 %0, [%1];" : "=l"(row) : "r"(from + (uint32_t)(j + h) * (uint32_t)sizeof(RedDesc)));
          const uint32_t dst = to + (uint32_t)h * SLOT;
          if (AL) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(row + off) : "memory");
          else {   // 32 tokens that start anywhere: up to five whole chunks, cut at the last token's end (segments are whole 64 bytes into the row)
            const int shift = (int)((uint32_t)row & 15u), n = min(16, bytes + shift);
            if (n > 0) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(row + off - (uint64_t)shift), "r"(n) : "memory");
          }
        }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(2 * part);
    if (q == 0 && !a.ring) {   // (the parts share a set's tiles)
      if (alive) alive = wk_drained(a, sm, rnd);
      for (int i = part; i < ntl && alive; i += nparts) {
        const int t = r0 + set + sets * i;
        if (first_pass && a.use_tma) alive = __all_sync(0xFFFFFFFFu, wk_wait(sm.w_full + t, 0, a, sm.abort));
        if (alive) wk_mma(a, sm, ncol, (uint32_t)t, (uint32_t)(set + sets * i), tmem_base);
      }
    }
    for (int i = 0; i < ntl; ++i) {
      const uint32_t slot = (uint32_t)(set + sets * i);
      if (alive) alive = __all_sync(0xFFFFFFFFu, wk_wait(sm.t_full + slot, (used >> slot) & 1u, a, sm.abort));
    }
    used ^= (1u << min(ntile - r0, round)) - 1u;
    tc_fence_after();
    const uint32_t tcol = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(set * a.cols);
#pragma unroll 1
    for (int j = 2 * part; j < nreq && alive; j += 2 * nparts) {
      uint32_t acc[2 * WK_TR];
#pragma unroll
      for (int i = 0; i < WK_TR; ++i)
        if (i < nt) asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(acc[2 * i]), "=r"(acc[2 * i + 1]) : "r"(tcol + (uint32_t)(sets * i * a.cols + j)) : "memory");
      float p[2 * WK_TR], qq[2 * WK_TR], c0[2]; int b[2], nC[2];
      const int two = j + 1 < nreq ? 1 : 0;
      const uint32_t dj = dbase + (uint32_t)j * (uint32_t)sizeof(RedDesc);
      float zoff[2], qoff[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t dh = dj + (uint32_t)(h * two) * (uint32_t)sizeof(RedDesc);   // (a lone request stands in for its partner)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=f"(zoff[h]), "=f"(qoff[h]), "=r"(b[h]), "=r"(nC[h]) : "r"(dh + 16u));
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(c0[h]) : "r"(dh + 32u));
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncwarp();   // the lanes' copies of this pair are all there
      tmem_ld_wait();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t zr = place + (uint32_t)h * SLOT + (uint32_t)lane * 2u, ur = zr + SEG;
        if (!AL) { zr += (uint32_t)b[h] >> 28; ur += ((uint32_t)b[h] >> 24) & 15u; }
#pragma unroll
        for (int i = 0; i < WK_TR; ++i) {
          const int e = h * WK_TR + i;
          p[e] = qq[e] = 0.f;
          if (i < nt && h <= two) {
            uint32_t z, u;
            asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(z) : "r"(zr + 2u * (uint32_t)i * SEG));
            asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(u) : "r"(ur + 2u * (uint32_t)i * SEG));
            p[e] = ex2_approx(fmaf(__uint_as_float(z << 16), zs, zoff[h]));
            qq[e] = ex2_approx(fmaf(__uint_as_float(acc[2 * i + h]) + __uint_as_float(u << 16), zs, qoff[h]));   // C == 0: qoff = -huge, the term vanishes
          }
        }
      }
      __syncwarp();   // nobody reads this pair's places any more
      stage(j + 2 * nparts);
      if (tail) {
#pragma unroll
        for (int e = 0; e < 2 * WK_TR; ++e) if (tok + step * (e % WK_TR) + lane >= tlen) { p[e] = 0.f; qq[e] = 0.f; }   // (the accumulator may hold anything)
      }
      float* to_part = mine + j * WK_VALS;
      if (nC[0] == 1 && nC[1] == 1) {
        // a tile's lanes first, then the tiles in order (the bits of the bonus draw's range sums hang on it)
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = (e & 3) < WK_TR ? fmaxf(fmaf(-c0[e >> 2], qq[(e >> 2) * WK_TR + ((e & 3) < WK_TR ? (e & 3) : 0)], p[(e >> 2) * WK_TR + ((e & 3) < WK_TR ? (e & 3) : 0)]), 0.f) : 0.f;
        const float v0 = wk_fold<8>(x, lane), v1 = __shfl_down_sync(0xFFFFFFFFu, v0, 4), v2 = __shfl_down_sync(0xFFFFFFFFu, v0, 8);
        if ((lane & 15) == 0 && (lane >> 4) <= two) { float* d = to_part + (lane >> 4) * WK_VALS; *d = r0 == 0 ? (v0 + v1) + v2 : ((*d + v0) + v1) + v2; }
        continue;
      }
#pragma unroll 1
      for (int h = 0; h <= two; ++h, to_part += WK_VALS) {
        float ph[WK_TR], qh[WK_TR];
#pragma unroll
        for (int i = 0; i < WK_TR; ++i) { ph[i] = h ? p[WK_TR + i] : p[i]; qh[i] = h ? qq[WK_TR + i] : qq[i]; }
        const int n = h ? nC[1] : nC[0];
        if (n == 1) {
          const float c = h ? c0[1] : c0[0];
          float x[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = i < WK_TR ? fmaxf(fmaf(-c, qh[i < WK_TR ? i : 0], ph[i < WK_TR ? i : 0]), 0.f) : 0.f;
          const float v0 = wk_fold<4>(x, lane), v1 = __shfl_sync(0xFFFFFFFFu, v0, 8), v2 = __shfl_sync(0xFFFFFFFFu, v0, 16);
          if (lane == 0) *to_part = r0 == 0 ? (v0 + v1) + v2 : ((*to_part + v0) + v1) + v2;
          continue;
        }
        float c[WK_COLS];
        const uint32_t dc = dj + (uint32_t)h * (uint32_t)sizeof(RedDesc) + 32u;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(dc));
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(c[4]), "=f"(c[5]), "=f"(c[6]), "=f"(c[7]) : "r"(dc + 16u));
        if (n & WK_GRID) {
          float x[WK_COLS];
#pragma unroll
          for (int k = 0; k < WK_COLS; ++k) x[k] = 0.f;
#pragma unroll
          for (int i = 0; i < WK_TR; ++i)
            if (i < nt) {
              x[0] += fmaxf(fmaf(-c[0], qh[i], ph[i]), 0.f);
#pragma unroll
              for (int k = 1; k < WK_COLS; ++k) x[k] += fabsf(fmaf(-c[k], qh[i], ph[i]));
            }
          const float v = wk_fold<WK_COLS>(x, lane);
          if ((lane & 3) == 0) { float* d = to_part + (lane >> 2); *d = r0 == 0 ? v : *d + v; }
        } else {
          float x[WK_VALS];
#pragma unroll
          for (int k = 0; k < WK_VALS; ++k) x[k] = 0.f;
#pragma unroll
          for (int i = 0; i < WK_TR; ++i)
            if (i < nt) {
#pragma unroll
              for (int k = 0; k < WK_COLS; ++k) {
                const float t = fmaf(-c[k], qh[i], ph[i]);
                if (t > 0.f) { x[k] += t; x[WK_COLS + k] += qh[i]; }
              }
            }
          const float v = wk_fold<WK_VALS>(x, lane);
          if ((lane & 1) == 0) { float* d = to_part + (lane >> 1); *d = r0 == 0 ? v : *d + v; }
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(sm.t_empty);
  }
}

// ---- the bonus token of one request whose walk is over, by the CTA that owns it ----------------------------------------------
__device__ __forceinline__ void wk_bonus(const WalkArgs& a, const WalkState& st, const int b, float* s_dot) {
  __shared__ float s_a[RMAX];
  __shared__ double s_scan[WK_EPI + 1], s_target, s_before;
  __shared__ int s_tile, s_found, s_last, s_fx[KMAX];   // the tested siblings: token, target and draft probability
  __shared__ double s_fp[KMAX], s_fq[KMAX];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t cb = (size_t)b * (a.N + 1);
  const int v = st.cur, nf = st.nf;
  const double C = st.C;
  const NodeDesc nd = a.node[cb + v + 1];
  const uint64_t hv = a.node_hash[cb + v + 1];
  if (tid < nf) { const WalkEdge e = a.edge[(size_t)b * a.N + st.cfirst + tid]; s_fx[tid] = e.x; s_fp[tid] = e.px; s_fq[tid] = e.qx; }
  // the range that holds the token: cumulative range sums at C (to first order from the coefficient they were evaluated at),
  // corrected for the tested siblings, which keep the residual they had when tested
  double* s_pt = reinterpret_cast<double*>(s_dot);
  {
    const float col = st.col[st.pcol];
    const double Ce = (double)col, Cf = (double)(float)C, step = st.nC > 1 && !(st.nC & WK_GRID) && fabs(Cf - Ce) <= 2.0 * WK_TOL * Cf ? Cf - Ce : 0.0;
    const float* part = a.part + ((size_t)b * WK_VALS + st.pcol) * a.vt_n;
    const int t = tid;   // (a range each: there are no more than SMs)
    double pt = t < a.vt_n ? (double)__ldcg(part + t) : 0.0;
    if (step != 0.0 && t < a.vt_n) pt -= step * (double)__ldcg(part + (size_t)WK_COLS * a.vt_n + t);
    __syncthreads();
    if (t < a.vt_n) {
      for (int i = 0; i < nf; ++i)
        if (s_fx[i] >= t * a.vt_TV && s_fx[i] < (t + 1) * a.vt_TV) pt += fmax(s_fp[i] - st.fC[i] * s_fq[i], 0.0) - fmax(s_fp[i] - Ce * s_fq[i], 0.0) + (s_fp[i] > Ce * s_fq[i] ? step * s_fq[i] : 0.0);
      s_pt[t] = fmax(pt, 0.0);
    }
  }
  for (int k = tid; k < a.r; k += WK_THREADS) s_a[k] = __bfloat162float(a.A[(size_t)nd.tok * a.r + k]);
  __syncthreads();
  if (warp == 0) {
    const double u = u01(stream_words(a.seed, b, hv, STREAM_BONUS, 0u).x);
    // a lane adds up neighbouring ranges, the warp scans the lanes, the lane with the crossing looks closer
    const double target = u * st.Zj;
    const int per = (a.vt_n + 31) / 32, r0 = min(a.vt_n, lane * per), r1 = min(a.vt_n, r0 + per);
    double sum = 0.0; int last = -1;
    for (int t = r0; t < r1; ++t) { const double p = s_pt[t]; sum += p; if (p > 0.0) last = t; }
    double inc = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) { const double o = __shfl_up_sync(0xFFFFFFFFu, inc, off); if (lane >= off) inc += o; }
    last = __reduce_max_sync(0xFFFFFFFFu, last);
    int found = -1; double before = inc - sum;
    if (inc > target)
      for (int t = r0; t < r1 && found < 0; ++t) { const double p = s_pt[t]; if (before + p > target) found = t; else before += p; }
    const unsigned who = __ballot_sync(0xFFFFFFFFu, found >= 0);
    if (lane == (who ? __ffs(who) - 1 : 0)) {
      if (!who) { found = last >= 0 ? last : 0; before = -1.0; }   // rounding: take the last range with mass
      s_tile = found; s_target = target; s_before = before; s_found = 0x7FFFFFFF; s_last = -1;
    }
  }
  __syncthreads();
  const int s_lo = s_tile * a.vt_TV, s_hi = min(a.V, s_lo + a.vt_TV);
  const double want = s_before >= 0.0 ? s_target - s_before : 1e300;
  const __nv_bfloat16 *zr = a.Z + nd.zrow * a.V, *ur = a.U + (size_t)nd.urow * a.V;
  const bool need_q = C != 0.0 || nf > 0, vec = (a.V & 7) == 0;
  const double lseT = need_q ? (double)a.node_lseT[cb + v + 1] : 0.0;
  double carry = 0.0;
  for (int c0 = s_lo; c0 < s_hi; c0 += WK_CHUNK) {
    const int len = min(WK_CHUNK, s_hi - c0);
    float zv[2] = {0.f, 0.f}, uv[2] = {0.f, 0.f};   // requested before the low-rank part, used after it
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (2 * tid + h < len) { zv[h] = __bfloat162float(zr[c0 + 2 * tid + h]); if (need_q) uv[h] = __bfloat162float(ur[c0 + 2 * tid + h]); }
    // low-rank part of the draft logits, rank in four slices (one when rows are not aligned): loads of eight rows together
    if (need_q) {
      if (vec) {
        const int g = tid % (WK_CHUNK / 8), ks = tid / (WK_CHUNK / 8);
        float acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0.f;
        if (g * 8 < len) {
          const uint4* wp = reinterpret_cast<const uint4*>(a.W + c0 + g * 8);
          const size_t pitch = (size_t)a.V / 8;
#pragma unroll 1
          for (int k0 = ks; k0 < a.r; k0 += 32) {
            uint4 w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = k0 + 4 * u < a.r ? __ldg(wp + (size_t)(k0 + 4 * u) * pitch) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const float ak = k0 + 4 * u < a.r ? s_a[k0 + 4 * u] : 0.f;
              float f[8];
              unpack_bf16x8(w[u], f);
#pragma unroll
              for (int i = 0; i < 8; ++i) acc[i] = fmaf(ak, f[i], acc[i]);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) s_dot[ks * WK_CHUNK + g * 8 + i] = acc[i];
      } else
        for (int o = tid; o < len; o += WK_THREADS) {
          float acc = 0.f;
          int k = 0;
          for (; k + 8 <= a.r; k += 8) {
            __nv_bfloat16 w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = a.W[(size_t)(k + u) * a.V + c0 + o];
#pragma unroll
            for (int u = 0; u < 8; ++u) acc = fmaf(s_a[k + u], __bfloat162float(w[u]), acc);
          }
          for (; k < a.r; ++k) acc = fmaf(s_a[k], __bfloat162float(a.W[(size_t)k * a.V + c0 + o]), acc);
          s_dot[o] = acc; s_dot[WK_CHUNK + o] = 0.f; s_dot[2 * WK_CHUNK + o] = 0.f; s_dot[3 * WK_CHUNK + o] = 0.f;
        }
      __syncthreads();
    }
    // residuals of two neighbouring tokens a thread, prefix sums in token order
    double rw[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int o = 2 * tid + h, w = c0 + o;
      rw[h] = 0.0;
      if (o < len) {
        double Cw = C;
        for (int f = 0; f < nf; ++f) if (s_fx[f] == w) Cw = st.fC[f];
        const double p = exp(((double)zv[h] - (double)nd.zmax) / (double)a.T - (double)nd.zlogs);
        double q = 0.0;
        if (Cw != 0.0) {
          const float lg = uv[h] + ((s_dot[o] + s_dot[WK_CHUNK + o]) + (s_dot[2 * WK_CHUNK + o] + s_dot[3 * WK_CHUNK + o]));
          q = exp((double)lg / (double)a.T - lseT);
        }
        rw[h] = fmax(p - Cw * q, 0.0);
      }
    }
    double inc = rw[0] + rw[1];
    const double own = inc;
    for (int off = 1; off < 32; off <<= 1) { const double t = __shfl_up_sync(0xFFFFFFFFu, inc, off); if (lane >= off) inc += t; }
    if (lane == 31) s_scan[warp] = inc;
    __syncthreads();
    double base = carry, total = 0.0;
    for (int w2 = 0; w2 <= WK_EPI; ++w2) { if (w2 < warp) base += s_scan[w2]; total += s_scan[w2]; }
    const double c1 = base + (inc - own) + rw[0], c2 = base + inc;
    const int o = c0 - s_lo + 2 * tid;
    if (rw[1] > 0.0) atomicMax(&s_last, o + 1); else if (rw[0] > 0.0) atomicMax(&s_last, o);
    if (2 * tid < len && c1 > want) atomicMin(&s_found, o); else if (2 * tid + 1 < len && c2 > want) atomicMin(&s_found, o + 1);
    carry += total;
    __syncthreads();
    if (s_found != 0x7FFFFFFF) break;   // uniform: read after the barrier
  }
  if (tid == 0) {
    int o = s_found;
    if (o == 0x7FFFFFFF) o = s_last >= 0 ? s_last : s_hi - s_lo - 1;   // rounding pushed the crossing past the range
    a.bonus[b] = s_lo + o;
    a.acc_len[b] = st.acc;
    a.flags[b] |= (uint32_t)min(st.npass, 0xFFFF) << 8;   // bits 8..23: sums this walk used
  }
  __syncthreads();
}

template <bool AL>
__global__ void __launch_bounds__(WK_THREADS, 1) walk_mma_kernel(const __grid_constant__ WalkArgs a, const __grid_constant__ CUtensorMap tmW) {
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ int s_cnt[WK_EPI + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = (int)blockIdx.x, ncta = (int)gridDim.x;
  const int rp = (a.r + 63) / 64 * 64, rw = (a.r + 15) / 16 * 16, t0 = cta * a.vt_TV, tlen = min(a.vt_TV, a.V - t0), ntile = (tlen + 127) / 128;
  const uint32_t slab = (uint32_t)rw * 128u;
  unsigned char* base = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
  WalkSm sm;
  sm.Ws = base; sm.Bs = base + a.oB; sm.stage = base + a.oT; sm.part = reinterpret_cast<float*>(base + a.oP);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + a.oS);
  sm.t_full = bars; sm.t_empty = bars + WK_ROUND; sm.w_full = bars + WK_ROUND + 4; sm.w_free = sm.w_full + 32;
  sm.tmem = reinterpret_cast<uint32_t*>(sm.w_free + 8); sm.abort = reinterpret_cast<volatile int*>(sm.tmem + 1);
  sm.desc = reinterpret_cast<RedDesc*>(bars + 64); sm.tok = reinterpret_cast<int*>(sm.desc + a.req); sm.st = reinterpret_cast<WalkState*>(sm.tok + a.req);
  if (warp == WK_LOAD) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(sm.tmem)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < WK_ROUND; ++i) mbar_init(sm.t_full + i, 1);
    mbar_init(sm.t_empty, WK_EPI);
    for (int i = 0; i < (a.ring ? a.ring : ntile); ++i) mbar_init(sm.w_full + i, 1);
    for (int i = 0; i < a.ring; ++i) mbar_init(sm.w_free + i, 1);
    *sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!a.ring && a.use_tma)
      for (int nb = 0; nb < ntile; ++nb) {
        const int ns = (tlen - nb * 128 > 64) ? 2 : 1;
        mbar_expect_tx(sm.w_full + nb, (uint32_t)ns * slab);
        for (int h = 0; h < ns; ++h) tma_load_box(sm.Ws + (size_t)(2 * nb + h) * slab, &tmW, t0 + (2 * nb + h) * 64, 0, sm.w_full + nb);
      }
  }
  if (!a.use_tma) {   // no tensor map, or rows that are not whole 16 bytes: plain loads into the same swizzled places
    const bool vec = (a.V & 7) == 0;
    const unsigned short* Wg = reinterpret_cast<const unsigned short*>(a.W);
    for (int idx = tid; idx < a.vt_TV / 64 * rw * 8; idx += WK_THREADS) {
      const int sl = idx / (rw * 8), rem = idx - sl * rw * 8, k = rem >> 3, j = rem & 7, v = t0 + sl * 64 + j * 8;
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      if (k < a.r) {
        const unsigned short* src = Wg + (size_t)k * a.V + v;
        if (vec) { if (v < a.V) *reinterpret_cast<uint4*>(w) = __ldg(reinterpret_cast<const uint4*>(src)); }
        else
#pragma unroll
          for (int i = 0; i < 8; ++i) if (v + i < a.V) w[i >> 1] |= (uint32_t)__ldg(src + i) << (16 * (i & 1));
      }
      *reinterpret_cast<uint4*>(sm.Ws + (size_t)sl * slab + k * 128 + ((j ^ (k & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  for (int i = tid; i < rp / 64 * a.cols * 8; i += WK_THREADS) reinterpret_cast<uint4*>(sm.Bs)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *sm.tmem;
  pdl_wait();   // row statistics and the tree come from earlier kernels; W (loaded above) does not
  pdl_launch_dependents();

  const int nown = a.B > cta ? (a.B - cta + ncta - 1) / ncta : 0;   // requests cta, cta + ncta, ...
  {   // (parents, tokens, and maximum and log-sum-exp of a request's rows, where the passes put their sums later)
    float2* z = reinterpret_cast<float2*>(sm.part); int* par = reinterpret_cast<int*>(z + 257);
    for (int i = 0; i < nown; ++i) wk_setup(a, sm.st[i], cta + i * ncta, par, par + 256, z);
  }
  unsigned gen = 0;
  const unsigned nexpect = (unsigned)ncta + (a.lost_arrival ? 1u : 0u);
  bool dead = false, finished = false;
  uint32_t used = 0u, rnd = 0u, wreq = 0u, pass = 0u;   // parities of the accumulator places, rounds and W blocks requested, over all passes
  for (int step = 0; !dead && step < a.max_steps; ++step) {
    // the sums that the owners' requests asked for, a warp each: range sums in a fixed order
    for (int x = warp; x < nown * WK_VALS; x += WK_THREADS / 32) {
      WalkState& st = sm.st[x / WK_VALS];
      const int val = x % WK_VALS;
      if ((st.phase == 1 || st.phase == 2) && wk_has(st.nC, val)) {
        const float* part = a.part + ((size_t)(cta + x / WK_VALS * ncta) * WK_VALS + val) * a.vt_n;
        double f = 0.0;
        for (int r0 = 0; r0 < a.vt_n; r0 += 5 * 32) {
          float pv[5];
#pragma unroll
          for (int k = 0; k < 5; ++k) pv[k] = (r0 + k * 32 + lane < a.vt_n) ? __ldcg(part + r0 + k * 32 + lane) : 0.f;
#pragma unroll
          for (int k = 0; k < 5; ++k) f += (double)pv[k];
        }
        f = wk_lanes_sum(f);
        if (lane == 0) st.S[val] = f;
      }
    }
    if (nown > 0) __syncthreads();   // (uniform)
    if (warp < WK_EPI)
      for (int i = warp; i < nown; i += WK_EPI) wk_advance(a, sm.st[i], cta + i * ncta, lane, step + 1);
    if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) { dead = true; break; }
    int nwk = 0;
    for (int sb = 0; sb == 0 || sb < nwk; sb += a.req) {
      // the requests that asked, in order of their numbers: the sb-th to the (sb + req - 1)-th of them
      nwk = 0;
      for (int c0 = 0; c0 < a.B; c0 += WK_EPI * 32) {
        const int b = c0 + tid;
        uint4 r0 = make_uint4(0u, 0u, 0u, 0u), r1 = r0, r2 = r0, r3 = r0, r4 = r0;
        if (tid < WK_EPI * 32 && b < a.B) {
          const uint4* src = reinterpret_cast<const uint4*>(a.rec + b);
          r0 = __ldcg(src); r1 = __ldcg(src + 1); r2 = __ldcg(src + 2); r3 = __ldcg(src + 3); r4 = __ldcg(src + 4);
        }
        const bool want = (int)r4.y == step + 1;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, want);
        if (lane == 0) s_cnt[warp] = __popc(bal);
        __syncthreads();
        int off = nwk;
        for (int w = 0; w < WK_EPI; ++w) { if (w < warp) off += s_cnt[w]; nwk += s_cnt[w]; }
        const int at = off + __popc(bal & ((1u << lane) - 1u)) - sb;
        if (want && at >= 0 && at < a.req) {
          RedDesc d;
          const int64_t zrow = (int64_t)(((uint64_t)r0.y << 32) | r0.x);
          d.z = a.Z + zrow * a.V; d.u = __uint_as_float(r2.x) != 0.f ? a.U + (size_t)(int)r0.z * a.V : d.z;   // (no proposal in the sum: its base row is not touched)
          d.zoff = __uint_as_float(r1.x); d.qoff = __uint_as_float(r2.x) != 0.f ? __uint_as_float(r1.y) : -1e30f;   // (lseT may be NaN where it is not needed)
          d.b = b; d.nC = (int)r4.x;
          if (!AL) d.b |= (int)(((uint32_t)(uintptr_t)d.z & 15u) << 28 | ((uint32_t)(uintptr_t)d.u & 15u) << 24);   // (where in a 16-byte chunk the rows start)
          RedDesc& o = sm.desc[at];
          o.z = d.z; o.u = d.u; o.zoff = d.zoff; o.qoff = d.qoff; o.b = d.b; o.nC = d.nC;
          reinterpret_cast<uint4*>(o.C)[0] = r2; reinterpret_cast<uint4*>(o.C)[1] = r3;
          sm.tok[at] = (int)r0.w;
        }
        __syncthreads();
      }
      if (nwk == 0) break;
      const int nreq = min(a.req, nwk - sb), ncol = (nreq + 15) & ~15;
      // head rows of the requests' nodes: the B operand, K-major with the 128-byte swizzle
      for (int idx = tid; idx < nreq * (a.r / 8); idx += WK_THREADS) {
        const int g = idx / (a.r / 8), ck = idx - g * (a.r / 8);
        *reinterpret_cast<uint4*>(sm.Bs + (ck >> 3) * (a.cols * 128) + g * 128 + (((ck & 7) ^ (g & 7)) << 4)) =
            __ldg(reinterpret_cast<const uint4*>(a.A + (size_t)sm.tok[g] * a.r + ck * 8));
      }
      // ask L2 for this range of the rows that will be read
      for (int x = warp; x < 2 * nreq; x += WK_THREADS / 32) {
        const RedDesc& d = sm.desc[x >> 1];
        const __nv_bfloat16* src = ((x & 1) ? d.u : d.z) + t0;
        if (!(x & 1) || d.u != d.z)
          for (int l = lane * 64; l < tlen; l += 32 * 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + l));
      }
      fence_async_smem();
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (warp < WK_EPI) wk_epilogue<AL>(a, sm, nreq, ncol, t0, tlen, tmem_base, used, rnd, pass == 0u);
      if (warp == WK_LOAD && a.ring) wk_stream(a, sm, &tmW, ncol, t0, tlen, pass, wreq, rnd, tmem_base);
      ++pass;
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (*sm.abort) { dead = true; break; }
      for (int x = tid; x < nreq * WK_VALS; x += WK_THREADS) {
        const RedDesc& d = sm.desc[x / WK_VALS];
        const int val = x % WK_VALS;
        if (wk_has(d.nC, val)) {
          const int ls = wk_sets(a, nreq), nw = 4 << ls, w0 = ((x / (2 * WK_VALS)) & ((4 >> ls) - 1)) << (2 + ls);   // the warps that had the request
          const float* from = sm.part + (size_t)w0 * (a.req * WK_VALS) + x;
          float s = 0.f;
#pragma unroll
          for (int w = 0; w < WK_EPI; ++w) s += w < nw ? from[w * a.req * WK_VALS] : 0.f;
          a.part[((size_t)(d.b & 0xFFFFFF) * WK_VALS + val) * a.vt_n + cta] = s;
        }
      }
      __syncthreads();
    }
    if (dead) { if (tid == 0) atomicExch(a.barrier + 1, 1u); break; }
    if (nwk == 0) { finished = true; break; }   // uniform over the grid: no request asked, every walk is over
    if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) { dead = true; break; }
  }
  // ---- no bulk load may still be writing this CTA's shared memory (waits bounded) -----------------------------------------
  if (warp == WK_LOAD && lane == 0 && a.use_tma) {
    const uint32_t lo = a.ring ? (wreq > (uint32_t)a.ring ? wreq - (uint32_t)a.ring : 0u) : 0u, hi = a.ring ? wreq : (uint32_t)ntile;
    for (uint32_t x = lo; x < hi; ++x) {
      uint64_t* bar = sm.w_full + (a.ring ? x % (uint32_t)a.ring : x);
      const uint32_t par = a.ring ? (x / (uint32_t)a.ring) & 1u : 0u;
      bool landed = false;
      for (uint32_t i = 0; i < WAIT_LIMIT && !landed; ++i) { landed = mbar_test_wait(bar, par); if (!landed) __nanosleep(100); }
    }
  }
  __syncthreads();
  for (int i = 0; i < nown; ++i) {
    if (sm.st[i].phase == 4) continue;
    if (finished) wk_bonus(a, sm.st[i], cta + i * ncta, reinterpret_cast<float*>(base));
    else if (tid == 0) a.status[cta + i * ncta] = TS_ERR_TIMEOUT;   // a wait ran out, or the steps did
  }
  tc_fence_before();
  __syncthreads();
  if (warp == WK_LOAD) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// ------------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------------
// What a plan takes of shared memory; false: too much, or more accumulators than tensor memory has.
static bool walk_fit(const ts_ctx* ctx, int B, int req, int sets, int tr, bool stream, WalkPlan* out) {
  const ts_config& c = ctx->cfg;
  const int ntile = (ctx->vt_TV + 127) / 128;
  WalkPlan p{};
  p.req = req; p.cols = req < 16 ? 16 : req; p.tr = tr; p.lsets = sets == 4 ? 2 : sets - 1;
  if (sets * tr * p.cols > 512) return false;
  const size_t slab = (size_t)(c.r + 15) / 16 * 2048, avail = (size_t)ctx->max_smem - WK_STATIC;
  const size_t head = (size_t)((c.r + 63) / 64) * p.cols * 128, stage = (size_t)WK_EPI * tr * 4 * wk_seg(c.V % 8 == 0);
  const size_t part = (size_t)WK_EPI * req * WK_VALS * 4, states = (size_t)((B + ctx->vt_n - 1) / ctx->vt_n) * sizeof(WalkState);
  const size_t fixed = head + stage + part + 64 * 8 + (size_t)req * (sizeof(RedDesc) + 4) + states + 1024;
  if (fixed > avail) return false;
  size_t w = (size_t)(ctx->vt_TV / 64) * slab;
  const size_t tiles = (size_t)ntile * 2 * slab + 1024;   // (the MMAs of a last tile of 64 tokens read the slab behind it too)
  if (stream) {
    p.ring = (int)((avail - fixed) / (2 * slab));
    p.ring = p.ring > 8 ? 8 : p.ring;
    if (p.ring < 2) return false;
    w = (size_t)p.ring * 2 * slab;
  } else if (ctx->vt_TV / 128 >= 32) return false;   // (barriers)
  if (w < WK_DOT) w = (WK_DOT + 1023) & ~(size_t)1023;   // (where the bonus draws work)
  p.smem = w + fixed;
  if (!stream && p.smem < tiles) p.smem = tiles;
  if (p.smem > avail) return false;
  p.oB = (uint32_t)w; p.oT = (uint32_t)(w + head); p.oP = (uint32_t)(p.oT + stage); p.oS = (uint32_t)(p.oP + part);
  *out = p;
  return true;
}

// Shared-memory plan.  (Verification, us, prepared rounds of the given batch; "before": the plan that went from 64 requests to 32 and then gave W up.)
//   Tiles.  As few sets of warps as hold them: what several coefficients cost is a sum over the lanes per request, set and quarter.
//     V = 50,257, 128 requests: 190 to 205 (three tiles in one set), 235 to 260 (in three); V = 100,000: 225 to 257, before 265 to 315.
//   W resident before W streamed, passes of fewer requests (not fewer tiles) where that takes room: V = 200,064, r = 64, 32 requests:
//     172 and 158 (16 a pass), 214 and 204 (32, a third of the tiles), 192 and 181 (32, streamed).  Eight a pass pay up to 32 requests (V = 230,000: 32:
//     220 and 214 against 230 and 223 streamed; 48: 295 and 320 against 272 and 315).
//   Streamed passes take 64 requests only if that costs no round of tiles more: r = 96, V = 151,936, 48 requests: 221 and 234 by 32, 245 and 259 by 64.
//   Without a tensor map (rows that are not whole 16 bytes) W has to be resident, whatever becomes of the rest: else the walk runs on fused
//     multiply-adds.  V = 151,643, r = 64, 32 requests: 161 and 166, without a plan 735 and 717; the last size, V = 230,003: 314 and 257.
bool walk_plan(const ts_ctx* ctx, int B, bool tma, WalkPlan* out) {
  const int ntile = (ctx->vt_TV + 127) / 128, sets = ntile <= WK_TR ? 1 : (ntile <= 2 * WK_TR ? 2 : 4), full = ntile <= sets * WK_TR ? (ntile + sets - 1) / sets : WK_TR;
  const int most = B <= 16 ? 16 : (B <= 32 || (ntile + 7) / 8 != (ntile + 11) / 12 ? 32 : 64);
  auto tiles = [&](int req) { return sets * full * req > 512 ? 512 / (sets * req) : full; };
  for (int req = most; req >= 8; req /= 2)
    if ((req > 8 || B <= 32 || !tma) && walk_fit(ctx, B, req, sets, tiles(req), false, out)) return true;
  if (!tma || B <= 8)
    for (int n = sets, tr = full;;) {
      if (n < 4) { n *= 2; tr = (ntile + n - 1) / n; } else --tr;
      if (tr < 1) break;
      if (walk_fit(ctx, B, 8, n, tr, false, out)) return true;
    }
  if (tma)
    for (int req = most; req >= 8; req /= 2)
      if (walk_fit(ctx, B, req, sets, tiles(req), true, out)) return true;
  return false;
}

size_t walk_ws_bytes(const ts_ctx* ctx, int B) {
  const size_t b = (size_t)B, n = (size_t)ctx->cfg.Nmax;
  return align_up(b * (n + 1) * sizeof(NodeDesc), 256) + align_up(b * (n + 1) * 8, 256) + align_up(b * n * sizeof(WalkEdge), 256) + align_up(b * sizeof(WalkRec), 256) +
         align_up(b * WK_VALS * (size_t)ctx->vt_n * 4, 256);
}

cudaError_t walk_setup(ts_ctx* ctx) {
  cudaFuncAttributes fa;
  for (const void* fn : {(const void*)walk_mma_kernel<true>, (const void*)walk_mma_kernel<false>}) {
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess && fa.sharedSizeBytes > WK_STATIC) e = cudaErrorInvalidConfiguration;   // (the plan counts on no more)
    if (e != cudaSuccess) return e;
  }
  const cudaError_t e = allow_all_smem(walk_mma_kernel<true>, ctx->max_smem);
  return e != cudaSuccess ? e : allow_all_smem(walk_mma_kernel<false>, ctx->max_smem);
}

cudaError_t launch_walk_mma(ts_ctx* ctx, WalkArgs& a, char* ws, const WalkPlan& p, cudaStream_t st) {
  const size_t b = (size_t)a.B, n = (size_t)a.N;
  a.node = (NodeDesc*)ws; ws += align_up(b * (n + 1) * sizeof(NodeDesc), 256);
  a.child = (int2*)ws; ws += align_up(b * (n + 1) * 8, 256);
  a.edge = (WalkEdge*)ws; ws += align_up(b * n * sizeof(WalkEdge), 256);
  a.rec = (WalkRec*)ws; ws += align_up(b * sizeof(WalkRec), 256);
  a.part = (float*)ws;
  a.ring = p.ring; a.req = p.req; a.cols = p.cols; a.tr = p.tr; a.lsets = p.lsets; a.oB = p.oB; a.oT = p.oT; a.oP = p.oP; a.oS = p.oS;
  CUtensorMap tm;
  memset(&tm, 0, sizeof(tm));
  if (a.use_tma) memcpy(&tm, ctx->tmapW, sizeof(tm));
  ProfScope ps(ctx, K_WALK, st);
  // (chained to the row statistics: the W load and the tensor-memory allocation run beside them)
  void* kargs[] = {(void*)&a, (void*)&tm};
  return launch_cooperative(ctx->walk_unchained, a.V % 8 == 0 ? (const void*)walk_mma_kernel<true> : (const void*)walk_mma_kernel<false>, dim3(a.vt_n), dim3(WK_THREADS), p.smem, st, kargs);
}

}  // namespace ts
