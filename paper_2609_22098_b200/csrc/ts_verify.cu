// Lossless tree verification (Section 3.2 item 3, Section 3.3).
//
// Stage 1 (all rows, fully parallel): max, arg-max and log-sum-exp at temperature T of every target
//   row, in equal pieces of the array of rows.  With these, the first-sibling accept ratio of every edge is a scalar
//   expression, so per-edge statistics and greedy walks need no further vocabulary pass.
// Stage 2, T == 0: pointer chase along arg-max matches.
// Stage 2, T > 0: one persistent cooperative kernel (bf16: ts_walk.cu; here the form for fp32, ranks that are no multiple
//   of 8 and ranges of W that fit neither shared memory nor a tensor map).  The recursive-rejection walk is run as a
//   scalar sequence: with R(w) = max(p(w) - C q(w), 0) the unnormalised residual after rejections,
//   sibling j is accepted with probability min(1, max(p(x)/q(x) - C, 0) / c_j), c_j = Z_j / (1 - Q),
//   and a rejection moves C to C + c_j and needs Z_{j+1} = sum_w R(w), one reduction over the
//   vocabulary (tokens already tested keep the residual they had when tested).  Every grid step
//   runs that reduction for all requests that just rejected, each CTA owning a vocabulary range;
//   q is recomputed from U, A, W, no per-node vocabulary vector is stored.  The bonus token is the
//   inverse CDF of the final residual in token order: range sums locate the range, one CTA rescans it.
#include <math.h>

#include "ts_internal.h"
#include "ts_scan.cuh"
#include "ts_tc.cuh"
#include "ts_walk.cuh"
#include "ts_zrow.cuh"

namespace ts {

// 2^x by the hardware approximation (the library exp2f costs several times more in the hot loops here)
__device__ __forceinline__ float fast_ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// maximum that returns NaN when either operand is NaN (fmaxf drops NaNs)
__device__ __forceinline__ float max_nan(float a, float b) { float y; asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b)); return y; }

// ------------------------------------------------------------------------------------------------
// Stage 1: row statistics
// ------------------------------------------------------------------------------------------------
// 32 bytes of a row (32-byte aligned), still packed; read once, so not kept in L1
template <typename TIn> struct ZVec {
  static constexpr int N = 32 / (int)sizeof(TIn);
  uint32_t q[8];
  __device__ __forceinline__ void load(const TIn* p) {
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]) : "l"(p));
  }
  __device__ __forceinline__ float at(int i) const {   // (i: a constant)
    if (sizeof(TIn) == 4) return __uint_as_float(q[i]);
    return __uint_as_float((i & 1) ? q[i >> 1] & 0xFFFF0000u : q[i >> 1] << 16);
  }
  __device__ __forceinline__ static uint32_t max2(uint32_t a, uint32_t b) {
    uint32_t y;
    if (sizeof(TIn) == 4) y = __float_as_uint(max_nan(__uint_as_float(a), __uint_as_float(b)));
    else asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(y) : "r"(a), "r"(b));
    return y;
  }
  __device__ __forceinline__ float max() const {   // NaN when one of them is
    const uint32_t m = max2(max2(max2(q[0], q[1]), max2(q[2], q[3])), max2(max2(q[4], q[5]), max2(q[6], q[7])));
    if (sizeof(TIn) == 4) return __uint_as_float(m);
    return max_nan(__uint_as_float(m << 16), __uint_as_float(m & 0xFFFF0000u));
  }
};

// One CTA per piece of the array of target rows (ts_zrow.cuh says how it is cut).  Bound by memory, with the one ex2 per
// element close behind (18 us of a B200's special-function units for the 175 MB of a serving batch of 32, 27 us of its
// memory).  Per element there is one fused multiply-add, one ex2 and one add, and per 32 bytes a packed maximum; what
// would be work per new maximum is kept out of the loop: the position inside the vector is looked up once at the end,
// and the sums keep the reference of the thread's first vectors until a maximum leaves it by 2^32 (a running maximum
// per thread made some lane of nearly every warp rescale and search in nearly every vector).  Two CTAs of 64 registers
// with the next 64 bytes of every thread in flight beat three of 40 without (2,000 rows: 121 us, not 126).
// One CTA per row took (V = 151,936, launch included) 21 us for the 15 rows of one request, 47 us for 575 rows, 144 us
// for 2,000; now 11, 42 and 121 us.  Finer pieces (4 and 8 per SM, dealt by the hardware) were slower: 45 and 49 us.
template <typename TIn, bool SUMS>
__global__ void __launch_bounds__(ZT, ZCTAS) zrow_stats_kernel(const TIn* Z, const int64_t* z_row_off, int B, int V, float T, ZPart* part, unsigned* walk_barrier) {
  __shared__ unsigned s_m[2][ZT / 32], s_c[2][ZT / 32]; __shared__ float s_ref[2][ZT / 32], s_s[2][ZT / 32]; __shared__ int s_nan[2][ZT / 32];
  pdl_wait();   // the target logits (and the tree) may come from the kernel just before this one
  pdl_launch_dependents();
  // the walk's barrier words start at zero (done here rather than by a memset, which would sit between
  // this kernel and the walk in the stream and keep the walk from starting its preamble early)
  if (walk_barrier && blockIdx.x == 0 && threadIdx.x < 16) walk_barrier[threadIdx.x] = 0u;
  const int64_t total = z_row_off[B] * V, q = zrow_piece(total, V, gridDim.x);
  const int64_t e0 = blockIdx.x * q, e1 = e0 + q < total ? e0 + q : total;
  if (e0 >= e1) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int VEC = ZVec<TIn>::N, UNR = 2;
  const float sc = SUMS ? 1.4426950408889634f / T : 1.f, reach = 32.f / sc;
  int par = 0;
  int64_t row = e0 / V;
  for (int64_t s0 = e0; s0 < e1; ++row, par ^= 1) {
    // the piece's share [s0, s1) of this row, as token numbers [lo, hi); [al, be) of it is whole aligned vectors (a row
    // starts wherever the vocabulary and the caller's pointer put it)
    const int64_t base = row * V, s1 = base + V < e1 ? base + V : e1;
    const TIn* z = Z + base;
    const int lo = (int)(s0 - base), hi = (int)(s1 - base), mis = (int)((uintptr_t)z / sizeof(TIn) % VEC);
    const int al = min(hi, lo + (VEC - (lo + mis) % VEC) % VEC), be = max(al, hi - (hi + mis) % VEC);
    float bv = -INFINITY, ref = -INFINITY, lim = -INFINITY, boff = 0.f, sum = 0.f;   // lim = ref + reach, boff = -ref * sc once ref is finite
    int bc = 0x7FFFFFFF;                                                             // first token of the vector that holds bv
    auto top = [&](float vm, int c) {
      if (vm > bv) bc = c;   // first maximum wins: a thread's tokens increase
      bv = max_nan(bv, vm);  // a NaN stays
      if (SUMS && vm > lim) { sum *= fast_ex2((ref - vm) * sc); ref = vm; lim = vm + reach; boff = -vm * sc; }
    };
    auto one = [&](int c) { const float x = Elem<TIn>::to_f(z[c]); top(x, c); if (SUMS) sum += fast_ex2(fmaf(x, sc, boff)); };
    auto vec = [&](const ZVec<TIn>& v, int c) {
      top(v.max(), c);
      if (SUMS) {
        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < VEC; ++i) s4[i & 3] += fast_ex2(fmaf(v.at(i), sc, boff));
        sum += (s4[0] + s4[1]) + (s4[2] + s4[3]);
      }
    };
    if (tid < al - lo) one(lo + tid);
    // the next vectors are requested before the present ones are worked on
    constexpr int STEP = UNR * ZT * VEC, SPAN = (UNR - 1) * ZT * VEC;
    int c = al + tid * VEC;
    ZVec<TIn> v[UNR];
    if (c + SPAN < be)
#pragma unroll
      for (int u = 0; u < UNR; ++u) v[u].load(z + c + u * ZT * VEC);
    for (; c + SPAN < be; c += STEP) {
      ZVec<TIn> nx[UNR];
      if (c + STEP + SPAN < be)
#pragma unroll
        for (int u = 0; u < UNR; ++u) nx[u].load(z + c + STEP + u * ZT * VEC);
#pragma unroll
      for (int u = 0; u < UNR; ++u) vec(v[u], c + u * ZT * VEC);
#pragma unroll
      for (int u = 0; u < UNR; ++u) v[u] = nx[u];
    }
    for (; c < be; c += ZT * VEC) { v[0].load(z + c); vec(v[0], c); }
    if (tid < hi - be) one(be + tid);
    // fold: value descending (-0 equals 0), ties to the lowest token; sums to the largest reference
    auto fold = [&](unsigned& m, unsigned& cc, float& r, float& s, int& nan) {
      const unsigned wm = __reduce_max_sync(0xFFFFFFFFu, m);
      cc = __reduce_min_sync(0xFFFFFFFFu, m == wm ? cc : 0x7FFFFFFFu);
      m = wm;
      nan = __any_sync(0xFFFFFFFFu, nan);
      const float wr = dec_f(__reduce_max_sync(0xFFFFFFFFu, enc_f(r)));
      s = r > -INFINITY ? s * fast_ex2((r - wr) * sc) : 0.f;
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      r = wr;
    };
    int nan = bv != bv ? 1 : 0;
    unsigned m = enc_f((nan ? -INFINITY : bv) + 0.f), cc = (unsigned)bc;
    fold(m, cc, ref, sum, nan);
    if (lane == 0) { s_m[par][warp] = m; s_c[par][warp] = cc; s_ref[par][warp] = ref; s_s[par][warp] = sum; s_nan[par][warp] = nan; }
    __syncthreads();   // (the arrays of the share before last are free: warp 0 has come through this barrier twice since)
    if (warp == 0) {
      const bool in = lane < ZT / 32;
      m = in ? s_m[par][lane] : 0u; cc = in ? s_c[par][lane] : 0x7FFFFFFFu; ref = in ? s_ref[par][lane] : -INFINITY; sum = in ? s_s[par][lane] : 0.f;
      nan = in ? s_nan[par][lane] : 0;
      fold(m, cc, ref, sum, nan);
      const float gv = dec_f(m);
      // the first token of the winning vector that has the maximum
      const unsigned t = cc + (unsigned)lane;
      const unsigned hit = __ballot_sync(0xFFFFFFFFu, lane < VEC && cc != 0x7FFFFFFFu && t < (unsigned)hi && Elem<TIn>::to_f(z[t]) == gv);
      if (lane == 0) {
        ZPart o;
        o.m = nan ? nanf("") : gv; o.arg = hit ? (int)cc + __ffs(hit) - 1 : 0x7FFFFFFF; o.ref = ref; o.sum = sum;
        part[row + blockIdx.x] = o;
      }
    }
    s0 = s1;
  }
}

struct VerifyArgs {
  const void *U, *A, *W, *Z; const int64_t* z_row_off;
  int B, V, D, r, K, N; float T; uint64_t seed;
  const int *anchor, *n_nodes, *tok, *parent, *depth, *sib; const uint64_t* node_hash;
  const float *logqT, *node_lseT;
  float* z_max; int* z_arg; float* z_logs;   // per row, folded from its pieces by the CTA that owns the request
  const ZPart* z_part; int z_np;             // the row statistics and the number of pieces they were cut into
  int *acc_len, *acc_node, *acc_tok, *bonus; float* edge_stat; uint32_t* flags; int* status;
  double *edge_px, *edge_qx, *edge_u;   // per edge: target and draft probability of its token, its accept uniform
  VerifyState* state; float* part; unsigned* barrier;
  int* child_first; int* child_cnt;   // [B][N+1], slot 0 = root
  int* wk_list; int* sc_list;         // [2][B] requests that asked for a reduction / a range rescan, by step parity
  int* ctr;                           // [0..1] reduction counts, [2..3] rescan counts (by parity), [4] unfinished requests
  int vt_TV, vt_n, max_steps;
  uint32_t wait_limit;   // polls before a bounded wait (grid barrier, mbarrier) gives up
  int lost_arrival;      // test switch: grid barriers expect one arrival more than will come
  int w_smem;   // 1: the kernel keeps its range of W in dynamic shared memory
  };

// ------------------------------------------------------------------------------------------------
// Stage 2, T == 0
// ------------------------------------------------------------------------------------------------
__global__ void verify_greedy_kernel(VerifyArgs a) {
  pdl_wait();   // the row statistics
  const int b = blockIdx.x, N = a.N;
  const int n_in = a.n_nodes[b];
  const bool okn = n_in >= 0 && n_in <= N;
  const int n = okn ? n_in : 0;
  const int64_t row0 = a.z_row_off[b];
  const size_t nb = (size_t)b * N;
  // a target row that holds a NaN (its maximum is NaN) or nothing finite has no arg-max
  int bad = 0;
  const int64_t zq = zrow_piece(a.z_row_off[a.B] * a.V, a.V, a.z_np);
  for (int i = threadIdx.x; okn && i <= n; i += blockDim.x) {
    const ZRow z = zrow_fold(a.z_part, row0 + i, a.V, zq, a.z_np, a.T);
    a.z_arg[row0 + i] = z.arg;
    bad |= (z.m != z.m || z.m == -INFINITY) ? 1 : 0;
  }
  bad = __syncthreads_or(okn ? bad : 0);
  if (a.edge_stat)
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      a.edge_stat[nb + i] = (!bad && a.tok[nb + i] == a.z_arg[row0 + a.parent[nb + i] + 1]) ? 1.f : 0.f;
  if (threadIdx.x == 0) {
    int cur = -1, acc = 0;
    if (!okn || bad) a.bonus[b] = -1;
    else
      for (;;) {
        const int g = a.z_arg[row0 + cur + 1];
        int hit = -1;
        for (int i = cur + 1; i < n; ++i)  // children come after their parent in canonical order
          if (a.parent[nb + i] == cur && a.tok[nb + i] == g) { hit = i; break; }
        if (hit < 0 || acc >= a.D) { a.bonus[b] = g; break; }
        a.acc_node[(size_t)b * a.D + acc] = hit; a.acc_tok[(size_t)b * a.D + acc] = g; ++acc; cur = hit;
      }
    for (int i = acc; i < a.D; ++i) { a.acc_node[(size_t)b * a.D + i] = -1; a.acc_tok[(size_t)b * a.D + i] = -1; }
    a.acc_len[b] = acc; a.flags[b] = 0u; a.status[b] = !okn ? TS_ERR_INVALID : (bad ? TS_ERR_NUMERIC : TS_OK);
  }
}

// ------------------------------------------------------------------------------------------------
// Stage 2, T > 0
// ------------------------------------------------------------------------------------------------
template <typename TIn>
__device__ __forceinline__ float z_elem(const VerifyArgs& a, int64_t row, int w) {
  return Elem<TIn>::to_f(reinterpret_cast<const TIn*>(a.Z)[row * a.V + w]);
}

// Scalar state machine of one request, run by one warp of the request's owner CTA.
// need: 0 walking, 1 reduction after a rejection, 4 reduction for the bonus draw, 5 walk over (bonus token
// still to be drawn), 2 range rescan, 3 finished.  The bonus draws of all requests are left to the end of
// the kernel (closing == true): locating the range and rescanning it would otherwise hold up, at every
// step, the requests that are still walking.
// Lane 0 decides; at every visited node the lanes fetch the accept-test inputs of all its children at
// once (one memory round trip per node), and the warp folds range sums together.
template <typename TIn>
__device__ void advance(const VerifyArgs& a, int b, int lane, int parity, bool closing) {
  VerifyState* gst = a.state + b;
  const int N = a.N;
  const size_t nb = (size_t)b * N;
  const int need_in = gst->need;
  const int cur0 = gst->cur, cf0 = gst->cfirst, cc0 = gst->ccnt;
  if (need_in == 3 || (need_in == 5 && !closing)) return;
  // accept-test inputs of the current node's children, requested together with everything else this step
  // needs (the range sums, the state): one memory round trip instead of a chain of three
  int x0 = -1; double px0 = 0.0, qx0 = 1.0, ux0 = 0.0;
  if ((need_in == 0 || need_in == 1 || need_in == 4) && lane < cc0) {
    x0 = a.tok[nb + cf0 + lane];
    px0 = a.edge_px[nb + cf0 + lane]; qx0 = a.edge_qx[nb + cf0 + lane]; ux0 = a.edge_u[nb + cf0 + lane];
  }
  // ---- fold in the reduction that just ran -------------------------------------------------
  double fsum = 0.0;
  if (need_in == 1 || need_in == 4) {
    float pv[8];   // the first 256 range sums in one memory round trip
#pragma unroll
    for (int k = 0; k < 8; ++k) pv[k] = (k * 32 + lane < a.vt_n) ? __ldcg(a.part + (size_t)b * a.vt_n + k * 32 + lane) : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) if (k * 32 + lane < a.vt_n) fsum += (double)pv[k];
    for (int t = 256 + lane; t < a.vt_n; t += 32) fsum += (double)__ldcg(a.part + (size_t)b * a.vt_n + t);
    for (int off = 16; off > 0; off >>= 1) fsum += __shfl_xor_sync(0xFFFFFFFFu, fsum, off);
  }
  VerifyState st;   // working copy (written back once at the end)
  if (lane == 0) st = *gst;
  int go_scan = 0;
  if (lane == 0) {
    if (need_in == 1 || need_in == 4) {
      double zn = fsum;  // the pass used passC for every token; tested siblings keep their own C_i
      for (int i = 0; i < st.nf; ++i)
        zn += fmax(st.fp[i] - st.fC[i] * st.fq[i], 0.0) - fmax(st.fp[i] - st.passC * st.fq[i], 0.0);
      if (need_in == 1) {
        if (zn <= 1e-30 * st.Zj) {  // residual lost its mass: keep the previous one
          a.flags[b] |= TS_FLAG_ZERO_MASS;
          st.fC[st.nf - 1] = st.C;
          st.partsC = -1.0;
        } else { st.C = st.passC; st.Zj = zn; st.partsC = st.passC; }
      } else { st.Zj = zn; st.partsC = st.passC; }
      st.need = 0;
    }
    if (st.need == 2) {  // the rescan wrote its token
      a.bonus[b] = st.result;
      a.acc_len[b] = st.acc;
      a.flags[b] |= (uint32_t)min(st.npass, 0xFFFF) << 8;   // bits 8..23: sums this walk used (a reduction each)
      st.need = 3;
    }
    if (st.need == 5) go_scan = 1;   // closing: draw the bonus token now
  }
  int walking = __shfl_sync(0xFFFFFFFFu, lane == 0 ? (st.need == 0) : 0, 0);
  bool at_start = true;   // still at the node the step began at: its children were fetched above
  while (walking) {
    // inputs of every child's accept test at the current node, one child per lane
    const int v = __shfl_sync(0xFFFFFFFFu, st.cur, 0);
    int first = cf0, m = cc0;
    double px = px0, qx = qx0; int x = x0;
    double ux = ux0;
    if (!at_start || v != cur0) {
      first = a.child_first[(size_t)b * (N + 1) + v + 1]; m = a.child_cnt[(size_t)b * (N + 1) + v + 1];
      px = 0.0; qx = 1.0; x = -1; ux = 0.0;
      if (lane < m) {   // computed for every edge when the walk was set up
        x = a.tok[nb + first + lane];
        px = a.edge_px[nb + first + lane]; qx = a.edge_qx[nb + first + lane]; ux = a.edge_u[nb + first + lane];
      }
      if (lane == 0) { st.cfirst = first; st.ccnt = m; }
    }
    at_start = false;
    // lane 0 runs the sibling chain at this node until it accepts, needs a reduction, or runs out
    int again = 0;
    for (int j = __shfl_sync(0xFFFFFFFFu, st.j, 0); j < 32; ++j) {   // m <= K <= 16; earlier siblings were tested in earlier steps
      const double pxj = __shfl_sync(0xFFFFFFFFu, px, j), qxj = __shfl_sync(0xFFFFFFFFu, qx, j);
      const int xj = __shfl_sync(0xFFFFFFFFu, x, j);
      const double uj = __shfl_sync(0xFFFFFFFFu, ux, j);
      int stop = 0;
      if (lane == 0) {
        if (st.j != j) { }   // siblings before st.j were tested in an earlier step
        else if (st.j < m && st.acc < a.D) {
          const double cj = st.Zj / (1.0 - st.Qused);
          const double num = fmax(pxj / qxj - st.C, 0.0);
          const double rho = fmin(1.0, num / cj);
          if (uj < rho) {
            a.acc_node[(size_t)b * a.D + st.acc] = first + j; a.acc_tok[(size_t)b * a.D + st.acc] = xj;
            st.acc++; st.cur = first + j; st.j = 0; st.C = 0.0; st.Zj = 1.0; st.Qused = 0.0; st.nf = 0; st.partsC = -1.0;
            stop = 1; again = 1;          // descend: next node
          } else {
            st.fx[st.nf] = xj; st.fp[st.nf] = pxj; st.fq[st.nf] = qxj; st.fC[st.nf] = st.C + cj; st.nf++;
            st.Qused += qxj; st.j++;
            st.passC = st.C + cj; st.row_node = v; st.need = 1;
            stop = 1;                      // wait for the reduction
          }
        } else {
          if (st.partsC != st.C) { st.passC = st.C; st.row_node = v; st.need = 4; }
          else go_scan = 1;
          stop = 1;
        }
      }
      stop = __shfl_sync(0xFFFFFFFFu, stop, 0);
      if (stop) break;
    }
    walking = __shfl_sync(0xFFFFFFFFu, again, 0);
  }
  go_scan = __shfl_sync(0xFFFFFFFFu, go_scan, 0);
  if (go_scan && !closing) {
    if (lane == 0) { st.need = 5; atomicSub(a.ctr + 4, 1); }   // one walker fewer
  } else if (go_scan) {
    // locate the vocabulary range holding the bonus token: cumulative corrected range sums
    const int cur = __shfl_sync(0xFFFFFFFFu, st.cur, 0), nf = __shfl_sync(0xFFFFFFFFu, st.nf, 0);
    const double C = __shfl_sync(0xFFFFFFFFu, st.C, 0), Zj = __shfl_sync(0xFFFFFFFFu, st.Zj, 0);
    const uint64_t hv = a.node_hash[(size_t)b * (N + 1) + cur + 1];
    const double u = u01(stream_words(a.seed, b, hv, STREAM_BONUS, 0u).x);
    const double target = u * Zj;
    double carry = 0.0; int found = -1; double before = 0.0; int last_pos = -1;
    // correction of tested sibling i (lane i): its range, and the difference between the residual it kept
    // and the one the last reduction gave it (the state in global memory is current: this runs in a later
    // step than the one that wrote it)
    int f_tile = -1; double f_delta = 0.0;
    if (lane < nf) {
      const int fxi = gst->fx[lane];
      const double fpi = gst->fp[lane], fqi = gst->fq[lane], fCi = gst->fC[lane];
      f_tile = fxi / a.vt_TV;
      f_delta = fmax(fpi - fCi * fqi, 0.0) - fmax(fpi - C * fqi, 0.0);
    }
    // the first 256 range sums are requested together (one memory round trip for the usual grid sizes)
    float pre[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) pre[k] = (k * 32 + lane < a.vt_n) ? __ldcg(a.part + (size_t)b * a.vt_n + k * 32 + lane) : 0.f;
    for (int t0 = 0; t0 < a.vt_n && found < 0; t0 += 32) {
      const int t = t0 + lane;
      double pt = 0.0;
      if (t0 < 256) {
        float pv = pre[0];
#pragma unroll
        for (int k = 1; k < 8; ++k) pv = (t0 >> 5) == k ? pre[k] : pv;
        pt = (double)pv;
      } else if (t < a.vt_n) pt = (double)__ldcg(a.part + (size_t)b * a.vt_n + t);
      for (int i = 0; i < nf; ++i) {   // tested siblings keep the residual they had when tested
        const int ti = __shfl_sync(0xFFFFFFFFu, f_tile, i);
        const double di = __shfl_sync(0xFFFFFFFFu, f_delta, i);
        if (t == ti) pt += di;
      }
      if (pt < 0.0) pt = 0.0;
      double inc = pt;
      for (int off = 1; off < 32; off <<= 1) { const double o = __shfl_up_sync(0xFFFFFFFFu, inc, off); if (lane >= off) inc += o; }
      const bool cross = (t < a.vt_n) && (carry + inc > target);
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, cross);
      const unsigned pos = __ballot_sync(0xFFFFFFFFu, pt > 0.0);
      if (pos) last_pos = t0 + 31 - __clz(pos);
      if (bal) {
        const int src = __ffs(bal) - 1;
        found = t0 + src;
        before = carry + __shfl_sync(0xFFFFFFFFu, inc - pt, src);
      }
      carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) {
      if (found < 0) { found = last_pos >= 0 ? last_pos : 0; before = -1.0; }  // rounding: take the last range with mass
      st.scan_tile = found; st.target = target; st.before = before; st.need = 2;
    }
  }
  if (lane == 0) {
    *gst = st;   // made visible to the other CTAs by the fence of the grid barrier that follows
    if (st.need == 1 || st.need == 4) a.wk_list[parity * a.B + atomicAdd(a.ctr + parity, 1)] = b;
    if (st.need == 1 || st.need == 4) gst->npass = st.npass + 1;
    else if (st.need == 2) a.sc_list[parity * a.B + atomicAdd(a.ctr + 2 + parity, 1)] = b;
  }
  __syncwarp();
}

template <typename TIn>
__device__ __forceinline__ float logit_scalar(const VerifyArgs& a, int req, int dep, int ptok, int w) {
  const TIn* Wg = reinterpret_cast<const TIn*>(a.W);
  const TIn* Ug = reinterpret_cast<const TIn*>(a.U);
  const TIn* Ag = reinterpret_cast<const TIn*>(a.A);
  float acc = Elem<TIn>::to_f(Ug[((size_t)req * a.D + dep) * a.V + w]);
  for (int k = 0; k < a.r; ++k)
    acc = fmaf(Elem<TIn>::to_f(Ag[(size_t)ptok * a.r + k]), Elem<TIn>::to_f(Wg[(size_t)k * a.V + w]), acc);
  return acc;
}

constexpr int VG = 4;  // requests sharing one sweep over the W columns

// One work item of a reduction step: NG requests of one group over tokens [c_lo, c_hi) of the CTA's range.
template <typename TIn>
struct SweepCtx {
  const TIn *Z, *U, *Wsrc; size_t wstride; int wshift; int V, D, r; float invT;
  const float* a; const int *req, *dep; const long long* row; const float *C, *zmax, *zlogs, *lseT;
};

template <typename TIn, int NG>
__device__ __forceinline__ void sweep_item(const SweepCtx<TIn>& c, int g0, int c_lo, int c_hi, int lane, float* out) {
  constexpr int VEC = Elem<TIn>::VEC;
  float sum[NG];
  bool need_q = false;
#pragma unroll
  for (int g = 0; g < NG; ++g) { sum[g] = 0.f; need_q |= (c.C[g0 + g] != 0.f); }
  for (int v = c_lo + lane * VEC; v < c_hi; v += 32 * VEC) {
    float z[NG][8], acc[NG][8];
#pragma unroll
    for (int g = 0; g < NG; ++g) {   // every load of the step first: target rows, base rows
      const TIn* zp = c.Z + c.row[g0 + g] * c.V + v;
      const TIn* up = c.U + ((size_t)c.req[g0 + g] * c.D + c.dep[g0 + g]) * c.V + v;
      const bool ldq = need_q && c.C[g0 + g] != 0.f;   // a member with C = 0 needs no proposal: its base row is not touched
      if (sizeof(TIn) == 2) {
        unpack_bf16x8(__ldg(reinterpret_cast<const uint4*>(zp)), z[g]);
        if (ldq) unpack_bf16x8(__ldg(reinterpret_cast<const uint4*>(up)), acc[g]);
      } else {
        const float4 x = __ldg(reinterpret_cast<const float4*>(zp)); z[g][0] = x.x; z[g][1] = x.y; z[g][2] = x.z; z[g][3] = x.w;
        if (ldq) { const float4 y = __ldg(reinterpret_cast<const float4*>(up)); acc[g][0] = y.x; acc[g][1] = y.y; acc[g][2] = y.z; acc[g][3] = y.w; }
      }
      if (need_q && !ldq) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) acc[g][i] = 0.f;
      }
    }
    if (need_q) {
      const TIn* wp = c.Wsrc + (v + c.wshift);
#pragma unroll 4
      for (int k = 0; k < c.r; ++k) {
        float w[8];
        if (sizeof(TIn) == 2) unpack_bf16x8(*reinterpret_cast<const uint4*>(wp + (size_t)k * c.wstride), w);
        else { const float4 x = *reinterpret_cast<const float4*>(wp + (size_t)k * c.wstride); w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w; }
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          const float ak = c.a[(g0 + g) * RMAX + k];
#pragma unroll
          for (int i = 0; i < VEC; ++i) acc[g][i] = fmaf(ak, w[i], acc[g][i]);
        }
      }
    }
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      const float Cg = c.C[g0 + g], zm = c.zmax[g0 + g], zl = c.zlogs[g0 + g], lt = c.lseT[g0 + g];
#pragma unroll
      for (int i = 0; i < VEC; ++i) {
        const float p = __expf((z[g][i] - zm) * c.invT - zl);
        const float q = Cg != 0.f ? __expf(acc[g][i] * c.invT - lt) : 0.f;
        sum[g] += fmaxf(p - Cg * q, 0.f);
      }
    }
  }
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    float sg = sum[g];
    for (int off = 16; off > 0; off >>= 1) sg += __shfl_xor_sync(0xFFFFFFFFu, sg, off);
    if (lane == 0) out[(size_t)g * 16] = sg;
  }
}


constexpr int SB = 32; // requests whose head rows are staged together
constexpr int WT = 288;       // threads of the walk kernel

// The walk proper.  Returns false when a bounded wait ran out (every thread of the CTA returns the same).
template <typename TIn>
__device__ __forceinline__ bool walk_body(const VerifyArgs& a, unsigned char* w_raw) {
  __shared__ int s_req[VG], s_dep[VG], s_node[VG];
  __shared__ float s_C[VG], s_zmax[VG], s_zlogs[VG], s_lseT[VG];
  __shared__ float s_red[VG][WT / 32];
  __shared__ double s_scan[WT];
  __shared__ int s_found, s_last;
  __shared__ float sb_a[SB * RMAX];
  __shared__ int sb_req[SB], sb_dep[SB], sb_tok[SB];
  __shared__ long long sb_row[SB];
  __shared__ float sb_C[SB], sb_zmax[SB], sb_zlogs[SB], sb_lseT[SB], sb_part[SB * 16];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned nblocks = gridDim.x;
  const unsigned nexpect = nblocks + (a.lost_arrival ? 1u : 0u);   // arrivals a grid barrier waits for
  unsigned gen = 0;
  constexpr int VEC = Elem<TIn>::VEC;
  const bool vec_ok = (a.V % VEC) == 0;
  const float invT = 1.f / a.T;
  const int v_lo = blockIdx.x * a.vt_TV, v_hi = min(a.V, v_lo + a.vt_TV);
  const TIn* Zg = reinterpret_cast<const TIn*>(a.Z);
  const TIn* Ag = reinterpret_cast<const TIn*>(a.A);
  const TIn* Wg = reinterpret_cast<const TIn*>(a.W);
  const int N = a.N;
  TIn* Ws = reinterpret_cast<TIn*>(w_raw);   // [r][vt_TV] when a.w_smem
  if (a.w_smem && vec_ok) {
    const int per_row = a.vt_TV / VEC;
    for (int i = tid; i < a.r * per_row; i += WT) {
      const int k = i / per_row, c = (i % per_row) * VEC;
      uint4 x = make_uint4(0, 0, 0, 0);
      if (v_lo + c < a.V) x = __ldg(reinterpret_cast<const uint4*>(Wg + (size_t)k * a.V + v_lo + c));
      *reinterpret_cast<uint4*>(Ws + (size_t)k * a.vt_TV + c) = x;
    }
  }
  const bool ws_ok = a.w_smem && vec_ok;

  // ---- per-edge statistics, child ranges and state initialisation (owner CTA of each request) ------
  const int64_t zq = zrow_piece(a.z_row_off[a.B] * a.V, a.V, a.z_np);
  if (blockIdx.x == 0 && tid < 5) a.ctr[tid] = tid == 4 ? a.B : 0;
  for (int b = blockIdx.x; b < a.B; b += nblocks) {
    const int n = a.n_nodes[b];
    const bool okn = n >= 0 && n <= N;
    const size_t nb = (size_t)b * N, cbase = (size_t)b * (N + 1);
    const int64_t row0 = a.z_row_off[b];
    for (int i = tid; i <= N; i += WT) { a.child_first[cbase + i] = -1; a.child_cnt[cbase + i] = 0; }
    // non-finite inputs: a target row with a NaN (its maximum is NaN), without finite mass, or a node whose
    // proposal log-probability is NaN (its expansion was reported TS_ERR_NUMERIC) -- the request is not walked
    int bad = 0;
    if (okn) {
      for (int i = tid; i <= n; i += WT) {
        const ZRow z = zrow_fold(a.z_part, row0 + i, a.V, zq, a.z_np, a.T);
        a.z_max[row0 + i] = z.m; a.z_logs[row0 + i] = z.logs;
        bad |= (z.m != z.m || isinf(z.m) || z.logs != z.logs || isinf(z.logs)) ? 1 : 0;
      }
      for (int i = tid; i < n; i += WT) { const float lq = a.logqT[nb + i]; bad |= (lq != lq) ? 1 : 0; }
    }
    bad = __syncthreads_or(bad);
    if (bad && a.edge_stat)
      for (int i = tid; i < n; i += WT) a.edge_stat[nb + i] = 0.f;
    if (okn && !bad)
      for (int i = tid; i < n; i += WT) {
        const int par = a.parent[nb + i];
        if (i == 0 || a.parent[nb + i - 1] != par) a.child_first[cbase + par + 1] = i;   // siblings are contiguous
        atomicAdd(&a.child_cnt[cbase + par + 1], 1);
        {
          // what the accept test of this edge needs, off the walk's critical path: p(x), q(x) and the uniform
          // of sibling j at its parent (j = place among the contiguous siblings)
          const int64_t row = row0 + par + 1;
          int j = 0;
          while (i - j - 1 >= 0 && a.parent[nb + i - j - 1] == par) ++j;
          a.edge_px[nb + i] = exp(((double)z_elem<TIn>(a, row, a.tok[nb + i]) - (double)a.z_max[row]) / (double)a.T - (double)a.z_logs[row]);
          a.edge_qx[nb + i] = exp((double)a.logqT[nb + i]);
          a.edge_u[nb + i] = u01(stream_words(a.seed, b, a.node_hash[(size_t)b * (N + 1) + par + 1], STREAM_ACCEPT, (uint32_t)j).x);
        }
        if (a.edge_stat) {
          const int64_t row = row0 + par + 1;
          const double lr = ((double)z_elem<TIn>(a, row, a.tok[nb + i]) - (double)a.z_max[row]) / (double)a.T -
                            (double)a.z_logs[row] - (double)a.logqT[nb + i];
          a.edge_stat[nb + i] = (float)exp(fmin(lr, 0.0));
        }
      }
    __syncthreads();   // the root's child range is read below
    if (tid == 0) {
      VerifyState& st = a.state[b];
      st.cur = -1; st.j = 0; st.acc = 0; st.need = 0; st.nf = 0; st.scan_tile = -1; st.row_node = -1; st.result = -1;
      st.C = 0.0; st.Zj = 1.0; st.Qused = 0.0; st.target = 0.0; st.before = 0.0; st.passC = 0.0; st.partsC = -1.0;
      st.npass = 0; st.pad_ = 0;
      st.cfirst = a.child_first[cbase]; st.ccnt = a.child_cnt[cbase];   // children of the root
      a.flags[b] = 0u;
      a.status[b] = !okn ? TS_ERR_INVALID : (bad ? TS_ERR_NUMERIC : TS_OK);
      if (!okn || bad) { st.need = 3; a.acc_len[b] = 0; a.bonus[b] = -1; }
      for (int i = 0; i < a.D; ++i) { a.acc_node[(size_t)b * a.D + i] = -1; a.acc_tok[(size_t)b * a.D + i] = -1; }
    }
    __syncthreads();
  }
  __threadfence();
  if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) return false;
  // requests rejected at set-up leave the count of unfinished ones
  for (int b = blockIdx.x; b < a.B; b += nblocks)
    if (tid == 0 && a.state[b].need == 3) atomicSub(a.ctr + 4, 1);

  // stage 0: walk steps until every request's walk is over; stage 1: one step that locates and rescans the
  // range of every bonus token; stage 2: the owners commit the results
  int stage = 0;
  for (int step = 0; step < a.max_steps; ++step) {
    const int par = step & 1;
    // ---- phase A: scalar walks of the requests this CTA owns, one warp each ----------------------
    for (int b = blockIdx.x + warp * (int)nblocks; b < a.B; b += (WT / 32) * (int)nblocks) advance<TIn>(a, b, lane, par, stage > 0);
    if (stage == 2) return true;
    if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) return false;
    // ---- phase B: vocabulary work requested by the walks -----------------------------------------
    const int nwk = __ldcg(a.ctr + par), nsc = __ldcg(a.ctr + 2 + par), left = __ldcg(a.ctr + 4);
    if (blockIdx.x == 0 && tid < 2) a.ctr[2 * tid + (par ^ 1)] = 0;   // next step's counters
    if (vec_ok) {
      // Reductions sum_w max(p(w) - C q(w), 0) over this CTA's vocabulary range, for up to SB requests
      // at a time.  Work item = (group of VG requests, chunk of the range); items are dealt to the warps,
      // so a single request still uses several warps and many requests run side by side.  Partial sums
      // are combined in a fixed order.
      const int len = v_hi - v_lo;
      const int chunk = max(256, ((len + 15) / 16 + 255) / 256 * 256);   // at most 16 chunks
      const int nchunk = (len + chunk - 1) / chunk;
      for (int sb0 = 0; sb0 < nwk; sb0 += SB) {
        const int nreq = min(SB, nwk - sb0);
        if (tid < nreq) {
          const int b = __ldcg(a.wk_list + par * a.B + sb0 + tid);
          const VerifyState* st = a.state + b;
          const int v = st->row_node;
          const int64_t row = a.z_row_off[b] + v + 1;
          sb_req[tid] = b; sb_row[tid] = row; sb_dep[tid] = v < 0 ? 0 : min(a.depth[(size_t)b * N + v], a.D - 1);   // a leaf at depth D asks only for its target row (C = 0): keep the base-row index inside U
          sb_tok[tid] = v < 0 ? a.anchor[b] : a.tok[(size_t)b * N + v];
          sb_C[tid] = (float)st->passC; sb_zmax[tid] = a.z_max[row]; sb_zlogs[tid] = a.z_logs[row];
          sb_lseT[tid] = a.node_lseT[(size_t)b * (N + 1) + v + 1];
        }
        __syncthreads();
        for (int i = tid; i < nreq * a.r; i += WT) {
          const int g = i / a.r, k = i % a.r;
          sb_a[g * RMAX + k] = Elem<TIn>::to_f(Ag[(size_t)sb_tok[g] * a.r + k]);
        }
        __syncthreads();
        const int ngrp = (nreq + VG - 1) / VG;
        for (int item = warp; item < ngrp * nchunk; item += WT / 32) {
          const int grp = item / nchunk, ch = item % nchunk;
          const int g0 = grp * VG, ng = min(VG, nreq - g0);
          const int c_lo = v_lo + ch * chunk, c_hi = min(v_hi, c_lo + chunk);
          const SweepCtx<TIn> sc{Zg, reinterpret_cast<const TIn*>(a.U), ws_ok ? Ws : Wg, ws_ok ? (size_t)a.vt_TV : (size_t)a.V,
                                 ws_ok ? -v_lo : 0, a.V, a.D, a.r, invT, sb_a, sb_req, sb_dep, sb_row, sb_C, sb_zmax, sb_zlogs, sb_lseT};
          float* out = sb_part + (size_t)g0 * 16 + ch;
          switch (ng) {
            case 1: sweep_item<TIn, 1>(sc, g0, c_lo, c_hi, lane, out); break;
            case 2: sweep_item<TIn, 2>(sc, g0, c_lo, c_hi, lane, out); break;
            case 3: sweep_item<TIn, 3>(sc, g0, c_lo, c_hi, lane, out); break;
            default: sweep_item<TIn, 4>(sc, g0, c_lo, c_hi, lane, out); break;
          }
        }
        __syncthreads();
        if (tid < nreq) {
          float t = 0.f;
          for (int ch = 0; ch < nchunk; ++ch) t += sb_part[tid * 16 + ch];
          a.part[(size_t)sb_req[tid] * a.vt_n + blockIdx.x] = t;
        }
        __syncthreads();
      }
    } else
    for (int w0 = 0; w0 < nwk; w0 += VG) {
      const int ng = min(VG, nwk - w0);
      if (tid < ng) {
        const int b = __ldcg(a.wk_list + par * a.B + w0 + tid);
        const VerifyState* st = a.state + b;
        const int v = st->row_node;
        const int64_t row = a.z_row_off[b] + v + 1;
        s_req[tid] = b; s_node[tid] = v; s_dep[tid] = v < 0 ? 0 : min(a.depth[(size_t)b * N + v], a.D - 1);
        s_C[tid] = (float)st->passC; s_zmax[tid] = a.z_max[row]; s_zlogs[tid] = a.z_logs[row];
        s_lseT[tid] = a.node_lseT[(size_t)b * (N + 1) + v + 1];
      }
      __syncthreads();
      float sum[VG];
#pragma unroll
      for (int g = 0; g < VG; ++g) sum[g] = 0.f;
      for (int v = v_lo + tid; v < v_hi; v += WT) {
        for (int g = 0; g < ng; ++g) {
          const int b = s_req[g];
          const int64_t row = a.z_row_off[b] + s_node[g] + 1;
          const float p = __expf((z_elem<TIn>(a, row, v) - s_zmax[g]) * invT - s_zlogs[g]);
          float q = 0.f;
          if (s_C[g] != 0.f) {
            const int ptok = s_node[g] < 0 ? a.anchor[b] : a.tok[(size_t)b * N + s_node[g]];
            q = __expf(logit_scalar<TIn>(a, b, s_dep[g], ptok, v) * invT - s_lseT[g]);
          }
          sum[g] += fmaxf(p - s_C[g] * q, 0.f);
        }
      }
#pragma unroll
      for (int g = 0; g < VG; ++g) {
        float sg = sum[g];
        for (int off = 16; off > 0; off >>= 1) sg += __shfl_xor_sync(0xFFFFFFFFu, sg, off);
        if (lane == 0) s_red[g][warp] = sg;
      }
      __syncthreads();
      if (tid < ng) {
        float t = 0.f;
        for (int w = 0; w < WT / 32; ++w) t += s_red[tid][w];
        a.part[(size_t)s_req[tid] * a.vt_n + blockIdx.x] = t;
      }
      __syncthreads();
    }
    // range rescans for bonus tokens that fall into this CTA's range: the residual of every token of
    // the range is evaluated once (tokens dealt round-robin to the threads: row i of the range holds
    // tokens i*WT .. i*WT+WT-1), then prefix sums in token order locate the crossing
    // Rescans are dealt round-robin to the CTAs (several bonus tokens often fall into one range, and a
    // rescan needs nothing of the CTA that owns the range except its columns of W, which any CTA can read
    // from global memory).
    for (int si = blockIdx.x; si < nsc; si += (int)nblocks) {
      const int b = __ldcg(a.sc_list + par * a.B + si);
      const VerifyState& st = a.state[b];
      const int s_lo = st.scan_tile * a.vt_TV, s_hi = min(a.V, s_lo + a.vt_TV);
      const bool own = st.scan_tile == (int)blockIdx.x;   // this CTA's own range: W is in shared memory
      const int v = st.cur;
      const int64_t row = a.z_row_off[b] + v + 1;
      const int dep = v < 0 ? 0 : a.depth[(size_t)b * N + v];
      const int ptok = v < 0 ? a.anchor[b] : a.tok[(size_t)b * N + v];
      const double C = st.C;
      const double zmax = a.z_max[row], zlogs = a.z_logs[row];
      const double lseT = C != 0.0 ? (double)a.node_lseT[(size_t)b * (N + 1) + v + 1] : 0.0;
      const int nf = st.nf;
      const double want = st.before >= 0.0 ? st.target - st.before : 1e300;
      for (int k = tid; k < a.r; k += WT) sb_a[k] = Elem<TIn>::to_f(Ag[(size_t)ptok * a.r + k]);
      if (tid == 0) { s_found = 0x7FFFFFFF; s_last = -1; }
      __syncthreads();
      const int len = s_hi - s_lo;
      const int nrow = (len + WT - 1) / WT;
      double carry = 0.0;
      for (int i = 0; i < nrow; ++i) {
        const int o = i * WT + tid, w = s_lo + o;
        double rw = 0.0;
        if (o < len) {
          double Cw = C;
          for (int f = 0; f < nf; ++f) if (st.fx[f] == w) Cw = st.fC[f];
          const double p = exp(((double)z_elem<TIn>(a, row, w) - zmax) / (double)a.T - zlogs);
          double q = 0.0;
          if (Cw != 0.0) {
            float acc = Elem<TIn>::to_f(reinterpret_cast<const TIn*>(a.U)[((size_t)b * a.D + dep) * a.V + w]);
            if (ws_ok && own) { for (int k = 0; k < a.r; ++k) acc = fmaf(sb_a[k], Elem<TIn>::to_f(Ws[(size_t)k * a.vt_TV + o]), acc); }
            else {
              // another CTA's range: the column of W comes from global memory, eight rows requested at a time
              // (same order of the multiply-adds as above, so the same bits)
              int k = 0;
              for (; k + 8 <= a.r; k += 8) {
                TIn wv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) wv[u] = Wg[(size_t)(k + u) * a.V + w];
#pragma unroll
                for (int u = 0; u < 8; ++u) acc = fmaf(sb_a[k + u], Elem<TIn>::to_f(wv[u]), acc);
              }
              for (; k < a.r; ++k) acc = fmaf(sb_a[k], Elem<TIn>::to_f(Wg[(size_t)k * a.V + w]), acc);
            }
            q = exp((double)acc / (double)a.T - lseT);
          }
          rw = fmax(p - Cw * q, 0.0);
        }
        // inclusive prefix over the row in thread (= token) order
        double inc = rw;
        for (int off = 1; off < 32; off <<= 1) { const double t = __shfl_up_sync(0xFFFFFFFFu, inc, off); if (lane >= off) inc += t; }
        if (lane == 31) s_scan[warp] = inc;
        __syncthreads();
        double wbase = 0.0, rowsum = 0.0;
        for (int w2 = 0; w2 < WT / 32; ++w2) { if (w2 < warp) wbase += s_scan[w2]; rowsum += s_scan[w2]; }
        const double cum = carry + wbase + inc;
        if (o < len && rw > 0.0) atomicMax(&s_last, o);
        if (o < len && cum > want) atomicMin(&s_found, o);
        carry += rowsum;
        __syncthreads();
        if (s_found != 0x7FFFFFFF) break;   // uniform: read after the barrier
      }
      if (tid == 0) {
        int o = s_found;
        if (o == 0x7FFFFFFF) o = s_last >= 0 ? s_last : len - 1;   // rounding pushed the crossing past the range
        a.state[b].result = s_lo + o;
      }
      __syncthreads();
    }
    __threadfence();
    if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) return false;
    if (stage == 1) stage = 2;
    else if (left == 0 && nwk == 0) stage = 1;   // uniform over the grid: both were read after the step's first barrier
  }
  // steps ran out
  for (int b = blockIdx.x; b < a.B; b += nblocks)
    if (tid == 0 && a.state[b].need != 3) a.status[b] = TS_ERR_TIMEOUT;
  return true;
}

template <typename TIn>
__global__ void __launch_bounds__(WT, 1) verify_walk_kernel(const VerifyArgs a) {
  extern __shared__ __align__(16) unsigned char w_raw[];
  pdl_wait();   // row statistics and the tree come from earlier kernels
  if (walk_body<TIn>(a, w_raw)) return;
  // a barrier gave up: the owners mark what they had not finished
  for (int b = blockIdx.x; b < a.B; b += gridDim.x)
    if (threadIdx.x == 0 && a.state[b].need != 3) a.status[b] = TS_ERR_TIMEOUT;
}

cudaError_t verify_setup(ts_ctx* ctx) {
  // the walk kernel may keep its range of W in shared memory
  const cudaError_t e = allow_all_smem(verify_walk_kernel<__nv_bfloat16>, ctx->max_smem);
  return e != cudaSuccess ? e : allow_all_smem(verify_walk_kernel<float>, ctx->max_smem);
}

}  // namespace ts

extern "C" int32_t ts_verify_tree(ts_ctx* ctx, const void* U, const void* A, const void* W, const void* Z,
                                  const int64_t* z_row_off, int32_t B, const int32_t* anchor_tok,
                                  const int32_t* n_nodes, const int32_t* tok, const int32_t* parent,
                                  const int32_t* depth, const int32_t* sib_rank, const uint64_t* node_hash,
                                  const float* logqT, const float* node_lseT, float T, uint64_t seed,
                                  int32_t* acc_len, int32_t* acc_node, int32_t* acc_tok, int32_t* bonus_tok,
                                  float* edge_stat, uint32_t* flags, int32_t* status, void* ws_v, size_t ws_bytes,
                                  void* stream) {
  using namespace ts;
  if (!ctx) return set_error(TS_ERR_INVALID, "ts_verify_tree: null context");
  const void* req[] = {U, A, W, Z, z_row_off, anchor_tok, n_nodes, tok, parent, depth, sib_rank, node_hash,
                       acc_len, acc_node, acc_tok, bonus_tok, flags, status, ws_v};
  for (const void* p : req)
    if (bad_ptr(p)) return set_error(TS_ERR_INVALID, "ts_verify_tree: null or misaligned pointer");
  if (edge_stat && ((uintptr_t)edge_stat & 15u)) return set_error(TS_ERR_INVALID, "ts_verify_tree: misaligned edge_stat");
  const ts_config& c = ctx->cfg;
  if (B < 1 || B > c.max_batch) return set_error(TS_ERR_INVALID, "ts_verify_tree: B out of range");
  if (!(T >= 0.f)) return set_error(TS_ERR_INVALID, "ts_verify_tree: T must be >= 0");
  if (T > 0.f && (bad_ptr(logqT) || bad_ptr(node_lseT)))
    return set_error(TS_ERR_INVALID, "ts_verify_tree: logqT and node_lseT are required when T > 0");
  const WsLayout L = make_layout(ctx, B);
  if (ws_bytes < L.total) return set_error(TS_ERR_WORKSPACE, "ts_verify_tree: workspace too small");
  char* ws = (char*)ws_v;
  cudaStream_t st = (cudaStream_t)stream;

  VerifyArgs a{};
  a.U = U; a.A = A; a.W = W; a.Z = Z; a.z_row_off = z_row_off; a.B = B; a.V = c.V; a.D = c.D; a.r = c.r; a.K = c.K;
  a.N = c.Nmax; a.T = T; a.seed = seed; a.anchor = anchor_tok; a.n_nodes = n_nodes; a.tok = tok; a.parent = parent;
  a.depth = depth; a.sib = sib_rank; a.node_hash = node_hash; a.logqT = logqT; a.node_lseT = node_lseT;
  a.z_max = (float*)(ws + L.z_max); a.z_arg = (int*)(ws + L.z_arg); a.z_logs = (float*)(ws + L.z_lse);
  ZPart* z_part = (ZPart*)(ws + L.z_part);
  a.z_part = z_part; a.z_np = L.z_np;
  a.acc_len = acc_len; a.acc_node = acc_node; a.acc_tok = acc_tok; a.bonus = bonus_tok; a.edge_stat = edge_stat;
  a.flags = flags; a.status = status;
  a.state = (VerifyState*)(ws + L.vf_state); a.part = (float*)(ws + L.vf_part); a.barrier = (unsigned*)(ws + L.vf_barrier);
  a.child_first = (int*)(ws + L.vf_child); a.child_cnt = a.child_first + (size_t)B * (c.Nmax + 1);
  a.edge_px = (double*)(ws + L.vf_edge); a.edge_qx = a.edge_px + (size_t)B * c.Nmax; a.edge_u = a.edge_qx + (size_t)B * c.Nmax;
  a.wk_list = (int*)(ws + L.vf_lists); a.sc_list = a.wk_list + 2 * (size_t)B; a.ctr = a.sc_list + 2 * (size_t)B;
  a.vt_TV = ctx->vt_TV; a.vt_n = ctx->vt_n; a.max_steps = 2 * (c.Nmax + c.D) + 10;
  a.wait_limit = ctx->wait_limit; a.lost_arrival = (ctx->test_mode & TS_TEST_LOST_ARRIVAL) ? 1 : 0;

  cudaError_t ez;
  {
    ProfScope ps(ctx, K_ZROWS, st);
    unsigned* bar = T > 0.f ? a.barrier : (unsigned*)nullptr;
    auto stats = [&](auto* kernel, auto* z) { return launch_kernel(kernel, L.z_np, ZT, 0, st, true, z, z_row_off, B, c.V, T, z_part, bar); };
    if (c.dt_Z == TS_DTYPE_BF16) ez = stats(T > 0.f ? zrow_stats_kernel<__nv_bfloat16, true> : zrow_stats_kernel<__nv_bfloat16, false>, (const __nv_bfloat16*)Z);
    else ez = stats(T > 0.f ? zrow_stats_kernel<float, true> : zrow_stats_kernel<float, false>, (const float*)Z);
  }
  cudaError_t e = ez != cudaSuccess ? ez : cudaGetLastError();
  if (e != cudaSuccess) return set_cuda_error("ts_verify_tree(rows)", e);
  if (T == 0.f) {
    { ProfScope ps(ctx, K_GREEDY, st); e = launch_kernel(verify_greedy_kernel, B, 128, 0, st, true, a); }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error("ts_verify_tree(greedy)", e);
    return TS_OK;
  }
  if (ctx->use_walk) {
    const bool tma = c.V % 8 == 0 && w_tensor_map(ctx, W);
    WalkPlan wp;
    if (walk_plan(ctx, B, tma, &wp)) {
      WalkArgs w{};
      w.U = (const __nv_bfloat16*)U; w.A = (const __nv_bfloat16*)A; w.W = (const __nv_bfloat16*)W; w.Z = (const __nv_bfloat16*)Z; w.z_row_off = z_row_off;
      w.B = B; w.V = c.V; w.D = c.D; w.r = c.r; w.N = c.Nmax; w.T = T; w.seed = seed;
      w.anchor = anchor_tok; w.n_nodes = n_nodes; w.tok = tok; w.parent = parent; w.depth = depth; w.node_hash = node_hash;
      w.logqT = logqT; w.node_lseT = node_lseT; w.z_part = a.z_part; w.z_np = a.z_np;
      w.acc_len = acc_len; w.acc_node = acc_node; w.acc_tok = acc_tok; w.bonus = bonus_tok; w.edge_stat = edge_stat; w.flags = flags; w.status = status;
      w.barrier = a.barrier; w.vt_TV = a.vt_TV; w.vt_n = a.vt_n; w.max_steps = a.max_steps;
      w.wait_limit = a.wait_limit; w.lost_arrival = a.lost_arrival; w.use_tma = tma ? 1 : 0;
      e = launch_walk_mma(ctx, w, ws + L.walk, wp, st);
      return e == cudaSuccess ? TS_OK : set_cuda_error("ts_verify_tree(walk)", e);
    }
  }
  const size_t w_bytes = (size_t)c.r * ctx->vt_TV * (c.dt_W == TS_DTYPE_BF16 ? 2 : 4);
  a.w_smem = (w_bytes + 40 * 1024 <= (size_t)ctx->max_smem) ? 1 : 0;
  void* kargs[] = {(void*)&a};
  const void* fn = c.dt_Z == TS_DTYPE_BF16 ? (const void*)verify_walk_kernel<__nv_bfloat16> : (const void*)verify_walk_kernel<float>;
  {
    ProfScope ps(ctx, K_WALK, st);
    e = launch_cooperative(ctx->walk_unchained, fn, dim3(a.vt_n), dim3(WT), a.w_smem ? w_bytes : 0, st, kargs);
  }
  if (e != cudaSuccess) return set_cuda_error("ts_verify_tree(walk)", e);
  return TS_OK;
}
