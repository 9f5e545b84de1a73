// The recursive-rejection walk of the verification at T > 0 (Section 3.3) on the 5th-generation tensor cores: one
// cooperative launch, one CTA per vocabulary range.
//
// A request's walk is a scalar sequence (see ts_verify.cu for the algebra): sibling tests until one is accepted or a
// rejection needs Z = sum_w max(p(w) - C q(w), 0).  A step of the kernel is
//   advance   one warp per request, in the CTA that owns it, runs the scalar sequence on state in shared memory and
//             publishes what its next reduction needs (48 bytes a request, no list and no counter);
//   barrier
//   reduce    every CTA reads those records and sums its range for all requests that asked: the draft logits are one MMA
//             tile per 128 tokens with the TOKENS on the 128 rows (W is the A operand, as it lies in memory) and the
//             requests on the columns, so that a thread holds one token and the work is in proportion to the requests.
//             (With the requests on the rows a step with three of them cost as much as one with 32; late steps have few.)
//   barrier
// When no request asks any more, every owner draws its requests' bonus tokens by itself: the range from the stored
// range sums, then the token inside it.  Two barriers a step and none at the start and the end.
//
// Measured at 32 requests, V = 151,936, r = 64 (11 to 12 steps): 11.5 us a step -- advance 2 to 3, barriers 1.1 and 1.5,
// operands 1.5, the pass about 5.
#include <math.h>
#include <string.h>

#include "ts_walk.cuh"

namespace ts {

constexpr int WK_EPI = 16;                 // warps that read accumulators: 4 lane quarters x 4 sets of tiles
constexpr int WK_LOAD = WK_EPI;            // tensor memory; in the streaming form it requests W and issues the MMAs
constexpr int WK_THREADS = (WK_EPI + 1) * 32;
constexpr int WK_REQ = 64;                 // requests of one reduction pass (columns of a tile)
constexpr int WK_BUF = 8;                  // accumulator buffers of WK_REQ columns: two per set of tiles
constexpr int WK_CHUNK = 1088;             // tokens of one step of the bonus rescan: 8 tokens x 136 places x 4 slices of the rank

struct RedDesc { const __nv_bfloat16 *z, *u; float C, zoff, qoff; int b; };
static_assert(sizeof(RedDesc) == 32, "two 16-byte loads");

// The walk of one request.
struct WalkState {
  int cur, j, acc, nf, npass, phase;       // phase: 0 walking, 1 waits for the sum after a rejection, 2 waits for the sum of the bonus draw, 3 walk over, 4 not walked
  int cfirst, ccnt;
  double C, Zj, Qused, passC, partsC;      // partsC: the C that the stored range sums were computed for (-1: none)
  int fx[KMAX]; double fC[KMAX], fp[KMAX], fq[KMAX];
};

struct WalkSm {
  unsigned char *Ws, *Bs; WalkState* st;
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
__device__ __forceinline__ void wk_setup(const WalkArgs& a, WalkState& st, const int b, int* s_par, float2* s_z) {
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
      if (i) s_par[i - 1] = par;
      NodeDesc nd;
      nd.zrow = row0 + i; nd.urow = b * a.D + min(dep, a.D - 1);   // (a leaf at depth D asks only for its target row: keep the base row inside U)
      nd.tok = tok; nd.zoff = (-zm * invT - zl) * LOG2E; nd.qoff = -ls * LOG2E; nd.zmax = zm; nd.zlogs = zl;
      const uint4* src = reinterpret_cast<const uint4*>(&nd); uint4* dst = reinterpret_cast<uint4*>(a.node + cb + i);
      dst[0] = src[0]; dst[1] = src[1];
      a.child[cb + i] = make_int2(-1, 0);
    }
  }
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
    }
    const int64_t row = row0 + par + 1;
    const int x = a.tok[nb + i];
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
    st.cfirst = -1; st.ccnt = 0;
    if (okn && !bad) { const int2 c = a.child[cb]; st.cfirst = c.x; st.ccnt = c.y; }
    a.flags[b] = 0u;
    a.status[b] = !okn ? TS_ERR_INVALID : (bad ? TS_ERR_NUMERIC : TS_OK);
    if (!okn || bad) { st.phase = 4; a.acc_len[b] = 0; a.bonus[b] = -1; }
  }
  __syncthreads();
}

// ---- one request's scalar sequence, by one warp ------------------------------------------------------------------------
// Everything it may need -- the range sums, the current node's children, the record of the current node -- is requested
// together: one memory round trip a step, and one more for every node it descends to.
__device__ __forceinline__ void wk_advance(const WalkArgs& a, WalkState& st, const int b, const int lane, const int stamp) {
  const int N = a.N;
  const size_t nb = (size_t)b * N, cb = (size_t)b * (N + 1);
  WalkRec* rec = a.rec + b;
  if (st.phase >= 3) { if (lane == 0) rec->stamp = 0; return; }
  int v = st.cur, first = st.cfirst, m = st.ccnt;
  WalkEdge e; e.px = 0.0; e.qx = 1.0; e.u = 0.0; e.x = -1;
  auto fetch = [&]() {
    if (lane < m) { const uint4* s = reinterpret_cast<const uint4*>(a.edge + nb + first + lane); uint4* d = reinterpret_cast<uint4*>(&e); d[0] = __ldcg(s); d[1] = __ldcg(s + 1); }
  };
  fetch();
  uint4 nd = make_uint4(0u, 0u, 0u, 0u);
  if (lane < 2) nd = __ldcg(reinterpret_cast<const uint4*>(a.node + cb + v + 1) + lane);
  const int phase = st.phase;
  if (phase) {   // ---- fold in the sum that just ran ----
    double f = 0.0;
    const float* part = a.part + (size_t)b * a.vt_n;
    for (int t0 = 0; t0 < a.vt_n; t0 += 5 * 32) {
      float pv[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) pv[k] = (t0 + k * 32 + lane < a.vt_n) ? __ldcg(part + t0 + k * 32 + lane) : 0.f;
#pragma unroll
      for (int k = 0; k < 5; ++k) f += (double)pv[k];
    }
    // the pass used passC for every token; tested siblings keep the residual they had when tested
    if (lane < st.nf) f += fmax(st.fp[lane] - st.fC[lane] * st.fq[lane], 0.0) - fmax(st.fp[lane] - st.passC * st.fq[lane], 0.0);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) f += __shfl_xor_sync(0xFFFFFFFFu, f, off);
    __syncwarp();
    if (lane == 0) {
      if (phase == 1) {
        if (f <= 1e-30 * st.Zj) {   // the residual lost its mass: keep the previous one
          a.flags[b] |= TS_FLAG_ZERO_MASS;
          st.fC[st.nf - 1] = st.C;
          st.partsC = -1.0;
        } else { st.C = st.passC; st.Zj = f; st.partsC = st.passC; }
      } else { st.Zj = f; st.partsC = st.passC; }
      st.phase = 0;
    }
    __syncwarp();
  }
  for (;;) {
    // the sibling chain at node v until one is accepted, a sum is needed, or they run out; all lanes follow it together
    int j = st.j;
    const double C = st.C, c0 = st.Zj, Q = st.Qused;
    int out = 0;   // 1 accepted, 2 sum after a rejection, 3 sum for the bonus draw, 4 walk over
    if (j < m && st.acc < a.D) {
      const double px = __shfl_sync(0xFFFFFFFFu, e.px, j), qx = __shfl_sync(0xFFFFFFFFu, e.qx, j), u = __shfl_sync(0xFFFFFFFFu, e.u, j);
      const int x = __shfl_sync(0xFFFFFFFFu, e.x, j);
      const double cj = c0 / (1.0 - Q);
      const double rho = fmin(1.0, fmax(px / qx - C, 0.0) / cj);
      __syncwarp();
      if (u < rho) {
        out = 1;
        if (lane == 0) {
          a.acc_node[(size_t)b * a.D + st.acc] = first + j; a.acc_tok[(size_t)b * a.D + st.acc] = x;
          st.acc++; st.cur = first + j; st.j = 0; st.C = 0.0; st.Zj = 1.0; st.Qused = 0.0; st.nf = 0; st.partsC = -1.0;
        }
      } else {
        out = 2;
        if (lane == 0) {
          const int k = st.nf;
          st.fx[k] = x; st.fp[k] = px; st.fq[k] = qx; st.fC[k] = C + cj; st.nf = k + 1;
          st.Qused = Q + qx; st.j = j + 1; st.passC = C + cj;
        }
      }
    } else {
      out = st.partsC != C ? 3 : 4;
      __syncwarp();
      if (lane == 0) { if (out == 3) st.passC = C; else st.phase = 3; }
    }
    __syncwarp();
    if (out != 1) {
      if (out == 4) { if (lane == 0) rec->stamp = 0; }
      else {
        if (lane < 2) reinterpret_cast<uint4*>(rec)[lane] = nd;
        if (lane == 0) { rec->C = (float)st.passC; rec->stamp = stamp; st.npass++; st.phase = out == 2 ? 1 : 2; }
      }
      __syncwarp();
      return;
    }
    // descend
    v = st.cur;
    const int2 c = __ldcg(a.child + cb + v + 1);
    first = c.x; m = c.y;
    if (lane < 2) nd = __ldcg(reinterpret_cast<const uint4*>(a.node + cb + v + 1) + lane);
    if (lane == 0) { st.cfirst = first; st.ccnt = m; }
    fetch();
    __syncwarp();
  }
}

// ---- one reduction pass: sums of max(p - C q, 0) over this CTA's tokens for up to WK_REQ requests ---------------------------
// The MMAs of one tile into accumulator buffer `buf`, W from slab pair `ws`; an elected lane of the calling warp.
// Issuing costs about 70 cycles an instruction (400 a tile of rank 64; 600 from a branch on the lane instead of an elected one,
// and 1200 beside busy warps): one warp for all nine tiles of a pass took longer than the sums, so where W is resident the
// first warp of every set issues its set's tiles.
__device__ __forceinline__ void wk_mma(const WalkArgs& a, const WalkSm& sm, const int ncol, const uint32_t ws, const uint32_t buf, const uint32_t tmem_base) {
  const int ksteps = (a.r + 15) / 16;
  const uint32_t slab = (uint32_t)((a.r + 63) / 64 * 64) * 128u;
  tc_fence_after();
  if (elect_one()) {
    const uint64_t ad = smem_desc(smem_u32(sm.Ws) + 2u * ws * slab, slab, 1024u), bd = smem_desc(smem_u32(sm.Bs), 16u, 1024u);
    const uint32_t idesc = wk_idesc(ncol), d = tmem_base + buf * (uint32_t)WK_REQ;
#pragma unroll 4
    for (int ks = 0; ks < ksteps; ++ks)
      mma_bf16(d, ad + (uint64_t)(ks * 128), bd + (uint64_t)((ks >> 2) * (WK_REQ * 128 / 16) + (ks & 3) * 2), idesc, ks > 0 ? 1u : 0u);
    mma_commit(sm.t_full + buf);
    if (a.ring) mma_commit(sm.w_free + ws);
  }
  __syncwarp();
}
// a set's tile number `nt` (counted over all passes) waits until the buffer's tile before last is drained
__device__ __forceinline__ bool wk_drained(const WalkArgs& a, const WalkSm& sm, const uint32_t buf, const uint32_t nt) {
  return nt < 2u || __all_sync(0xFFFFFFFFu, wk_wait(sm.t_empty + buf, ((nt >> 1) - 1u) & 1u, a, sm.abort));
}
__device__ __forceinline__ bool wk_issue(const WalkArgs& a, const WalkSm& sm, const int ncol, const int t, const int set, const uint32_t nt, const bool first_pass, const uint32_t tmem_base) {
  const uint32_t buf = (uint32_t)set * 2u + (nt & 1u);
  if (first_pass && a.use_tma && !__all_sync(0xFFFFFFFFu, wk_wait(sm.w_full + t, 0, a, sm.abort))) return false;
  if (!wk_drained(a, sm, buf, nt)) return false;
  wk_mma(a, sm, ncol, (uint32_t)t, buf, tmem_base);
  return true;
}
// Streaming form, one warp: blocks of 128 tokens of W through the ring, one after the other round the range and on into the next
// pass (W does not depend on which requests that sums), and the tiles in the same order.  (In order, and by one warp: a wait
// for a parity tells a slot's turns apart only while the waiter follows every one of them.)
__device__ __forceinline__ void wk_stream(const WalkArgs& a, const WalkSm& sm, const CUtensorMap* tm, const int ncol, const int t0, const int tlen, const uint32_t pass,
                                          uint32_t& wreq, const uint32_t tmem_base) {
  const int ntile = (tlen + 127) / 128;
  const uint32_t slab = (uint32_t)((a.r + 63) / 64 * 64) * 128u, ring = (uint32_t)a.ring, w0 = pass * (uint32_t)ntile;
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
    const uint32_t x = w0 + (uint32_t)t, set = (uint32_t)t & 3u, nt = pass * (uint32_t)((ntile - (int)set + 3) / 4) + (uint32_t)(t >> 2), buf = set * 2u + (nt & 1u);
    if (!__all_sync(0xFFFFFFFFu, wk_wait(sm.w_full + x % ring, (x / ring) & 1, a, sm.abort))) return;
    if (!wk_drained(a, sm, buf, nt)) return;
    wk_mma(a, sm, ncol, x % ring, buf, tmem_base);
  }
}

// The scanning warps.  Per tile and eight requests a thread loads its token's target and base logit of every request (a
// warp reads 64 contiguous bytes of each row), requested one group ahead.
__device__ __forceinline__ void wk_epilogue(const WalkArgs& a, const WalkSm& sm, const int nreq, const int ncol, const int t0, const int tlen,
                                            const uint32_t tmem_base, uint32_t& nt, const bool first_pass, const RedDesc* desc, float* s_part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = warp & 3, set = warp >> 2;
  const int ntile = (tlen + 127) / 128, ng = (nreq + 7) / 8;
  const float zs = (1.f / a.T) * 1.4426950408889634f;   // exponentials as powers of two
  float* mine = s_part + warp * WK_REQ;
  for (int j = lane; j < WK_REQ; j += 32) mine[j] = 0.f;
  __syncwarp();
  unsigned short nz[8], nu[8];
  auto load = [&](int t, int g) {
    const int o = t * 128 + q * 32 + lane;
    const bool in = o < tlen;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int j = g * 8 + i;
      nz[i] = 0xFF80; nu[i] = 0;   // -inf: p = 0 and the term vanishes
      if (in && j < nreq) {
        const RedDesc& d = desc[j];
        nz[i] = __ldg(reinterpret_cast<const unsigned short*>(d.z) + t0 + o);
        if (d.C != 0.f) nu[i] = __ldg(reinterpret_cast<const unsigned short*>(d.u) + t0 + o);
      }
    }
  };
  bool alive = true;
  const bool issues = q == 0 && !a.ring;
  if (issues) for (int k = 0; k < 2 && alive; ++k) if (set + 4 * k < ntile) alive = wk_issue(a, sm, ncol, set + 4 * k, set, nt + (uint32_t)k, first_pass, tmem_base);
  if (set < ntile) load(set, 0);
  for (int t = set; t < ntile && alive; t += 4, ++nt) {
    const uint32_t buf = (uint32_t)set * 2u + (nt & 1u);
    if (!__all_sync(0xFFFFFFFFu, wk_wait(sm.t_full + buf, (nt >> 1) & 1u, a, sm.abort))) { alive = false; break; }
    tc_fence_after();
    for (int g = 0; g < ng; ++g) {
      uint32_t acc[8];
      __syncwarp();   // (the tensor-memory load is a warp-wide instruction)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(acc[0]), "=r"(acc[1]), "=r"(acc[2]), "=r"(acc[3]), "=r"(acc[4]), "=r"(acc[5]), "=r"(acc[6]), "=r"(acc[7])
                   : "r"(tmem_base + ((uint32_t)(q * 32) << 16) + buf * (uint32_t)WK_REQ + (uint32_t)(g * 8)) : "memory");
      float z[8], u[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) { z[i] = __uint_as_float((uint32_t)nz[i] << 16); u[i] = __uint_as_float((uint32_t)nu[i] << 16); }
      if (g + 1 < ng) load(t, g + 1); else if (t + 4 < ntile) load(t + 4, 0);
      tmem_ld_wait();
      float s[8];
      const bool upper = nreq - g * 8 > 4;   // (late steps have a few requests: half a group)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (i >= 4 && !upper) { s[i] = 0.f; continue; }
        const int j = min(g * 8 + i, nreq - 1);
        const float p = ex2_approx(fmaf(z[i], zs, desc[j].zoff));
        const float qq = ex2_approx(fmaf(__uint_as_float(acc[i]) + u[i], zs, desc[j].qoff));   // C == 0: qoff = -huge, the term vanishes
        s[i] = fmaxf(fmaf(-desc[j].C, qq, p), 0.f);
        if (z[i] == -INFINITY) s[i] = 0.f;   // (outside the range the accumulator may hold anything)
      }
      // sums over the lanes: halve the eight values three times, then two plain steps; lane 4i ends with value i
#pragma unroll
      for (int h = 4, off = 16; h >= 1; h >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < h) {
            const float give = up ? s[i] : s[i + h], keep = up ? s[i + h] : s[i];
            s[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, off);
          }
      }
      float v = s[0];
      v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
      v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
      if ((lane & 3) == 0) mine[g * 8 + (lane >> 2)] += v;
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(sm.t_empty + buf);
    if (issues && t + 8 < ntile) alive = wk_issue(a, sm, ncol, t + 8, set, nt + 2u, first_pass, tmem_base);
  }
}

// ---- the bonus token of one request whose walk is over, by the CTA that owns it ----------------------------------------------
__device__ __forceinline__ void wk_bonus(const WalkArgs& a, const WalkState& st, const int b, float* s_dot) {
  __shared__ float s_a[RMAX];
  __shared__ double s_scan[WK_EPI + 1], s_target, s_before;
  __shared__ int s_tile, s_found, s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t cb = (size_t)b * (a.N + 1);
  const int v = st.cur, nf = st.nf;
  const double C = st.C;
  if (warp == 0) {
    // the range that holds the token: cumulative range sums, corrected for the tested siblings
    const double u = u01(stream_words(a.seed, b, a.node_hash[cb + v + 1], STREAM_BONUS, 0u).x);
    const double target = u * st.Zj;
    int f_tile = -1; double f_delta = 0.0;
    if (lane < nf) { f_tile = st.fx[lane] / a.vt_TV; f_delta = fmax(st.fp[lane] - st.fC[lane] * st.fq[lane], 0.0) - fmax(st.fp[lane] - C * st.fq[lane], 0.0); }
    double carry = 0.0, before = 0.0; int found = -1, last_pos = -1;
    const float* part = a.part + (size_t)b * a.vt_n;
    for (int t1 = 0; t1 < a.vt_n && found < 0; t1 += 5 * 32) {
      float pre[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) pre[k] = (t1 + k * 32 + lane < a.vt_n) ? __ldcg(part + t1 + k * 32 + lane) : 0.f;
#pragma unroll 1
      for (int k = 0; k < 5 && found < 0; ++k) {
        const int t = t1 + k * 32 + lane;
        double pt = (double)pre[0];
#pragma unroll
        for (int e = 1; e < 5; ++e) pt = k == e ? (double)pre[e] : pt;
        for (int i = 0; i < nf; ++i) {   // tested siblings keep the residual they had when tested
          const int ti = __shfl_sync(0xFFFFFFFFu, f_tile, i);
          const double di = __shfl_sync(0xFFFFFFFFu, f_delta, i);
          if (t == ti) pt += di;
        }
        if (pt < 0.0) pt = 0.0;
        double inc = pt;
        for (int off = 1; off < 32; off <<= 1) { const double o = __shfl_up_sync(0xFFFFFFFFu, inc, off); if (lane >= off) inc += o; }
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, t < a.vt_n && carry + inc > target);
        const unsigned pos = __ballot_sync(0xFFFFFFFFu, pt > 0.0);
        if (pos) last_pos = t1 + k * 32 + 31 - __clz(pos);
        if (bal) { const int src = __ffs(bal) - 1; found = t1 + k * 32 + src; before = carry + __shfl_sync(0xFFFFFFFFu, inc - pt, src); }
        carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
      }
    }
    if (lane == 0) {
      if (found < 0) { found = last_pos >= 0 ? last_pos : 0; before = -1.0; }   // rounding: take the last range with mass
      s_tile = found; s_target = target; s_before = before; s_found = 0x7FFFFFFF; s_last = -1;
    }
  }
  const NodeDesc nd = a.node[cb + v + 1];
  for (int k = tid; k < a.r; k += WK_THREADS) s_a[k] = __bfloat162float(a.A[(size_t)nd.tok * a.r + k]);
  __syncthreads();
  const int s_lo = s_tile * a.vt_TV, s_hi = min(a.V, s_lo + a.vt_TV);
  const double want = s_before >= 0.0 ? s_target - s_before : 1e300;
  const __nv_bfloat16 *zr = a.Z + nd.zrow * a.V, *ur = a.U + (size_t)nd.urow * a.V;
  const bool need_q = C != 0.0 || nf > 0, vec = (a.V & 7) == 0;
  const double lseT = need_q ? (double)a.node_lseT[cb + v + 1] : 0.0;
  double carry = 0.0;
  for (int c0 = s_lo; c0 < s_hi; c0 += WK_CHUNK) {
    const int len = min(WK_CHUNK, s_hi - c0);
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
        for (int f = 0; f < nf; ++f) if (st.fx[f] == w) Cw = st.fC[f];
        const double p = exp(((double)__bfloat162float(zr[w]) - (double)nd.zmax) / (double)a.T - (double)nd.zlogs);
        double q = 0.0;
        if (Cw != 0.0) {
          const float lg = __bfloat162float(ur[w]) + ((s_dot[o] + s_dot[WK_CHUNK + o]) + (s_dot[2 * WK_CHUNK + o] + s_dot[3 * WK_CHUNK + o]));
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
    a.flags[b] |= (uint32_t)min(st.npass, 0xFFFF) << 8;   // bits 8..23: reductions this walk needed
  }
  __syncthreads();
}

__global__ void __launch_bounds__(WK_THREADS, 1) walk_mma_kernel(const __grid_constant__ WalkArgs a, const __grid_constant__ CUtensorMap tmW) {
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ RedDesc s_desc[WK_REQ];
  __shared__ int s_tok[WK_REQ], s_par[256], s_cnt[WK_EPI + 1];
  __shared__ float s_part[WK_EPI * WK_REQ];
  __shared__ float2 s_z[257];   // (maximum, log-sum-exp) of a request's rows
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = (int)blockIdx.x, ncta = (int)gridDim.x;
  const int rp = (a.r + 63) / 64 * 64, t0 = cta * a.vt_TV, tlen = min(a.vt_TV, a.V - t0), ntile = (tlen + 127) / 128;
  const uint32_t slab = (uint32_t)rp * 128u;
  unsigned char* base = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
  WalkSm sm;
  sm.Ws = base; sm.Bs = base + a.oB;
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + a.oS);
  sm.t_full = bars; sm.t_empty = bars + WK_BUF; sm.w_full = bars + 2 * WK_BUF; sm.w_free = sm.w_full + 32;
  sm.tmem = reinterpret_cast<uint32_t*>(sm.w_free + 8); sm.abort = reinterpret_cast<volatile int*>(sm.tmem + 1);
  sm.st = reinterpret_cast<WalkState*>(bars + 64);
  if (warp == WK_LOAD) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(sm.tmem)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < WK_BUF; ++i) { mbar_init(sm.t_full + i, 1); mbar_init(sm.t_empty + i, 4); }
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
    for (int idx = tid; idx < a.vt_TV / 64 * rp * 8; idx += WK_THREADS) {
      const int sl = idx / (rp * 8), rem = idx - sl * rp * 8, k = rem >> 3, j = rem & 7, v = t0 + sl * 64 + j * 8;
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
  for (int i = tid; i < (int)slab / 16; i += WK_THREADS) reinterpret_cast<uint4*>(sm.Bs)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *sm.tmem;
  pdl_wait();   // row statistics and the tree come from earlier kernels; W (loaded above) does not
  pdl_launch_dependents();

  const int nown = a.B > cta ? (a.B - cta + ncta - 1) / ncta : 0;   // requests cta, cta + ncta, ...
  for (int i = 0; i < nown; ++i) wk_setup(a, sm.st[i], cta + i * ncta, s_par, s_z);
  unsigned gen = 0;
  const unsigned nexpect = (unsigned)ncta + (a.lost_arrival ? 1u : 0u);
  bool dead = false, finished = false;
  uint32_t nt = 0u, wreq = 0u, pass = 0u;   // tiles of this warp's set and W blocks requested, over all passes
  for (int step = 0; !dead && step < a.max_steps; ++step) {
    if (warp < WK_EPI)
      for (int i = warp; i < nown; i += WK_EPI) wk_advance(a, sm.st[i], cta + i * ncta, lane, step + 1);
    if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) { dead = true; break; }
    int nwk = 0;
    for (int sb = 0; sb == 0 || sb < nwk; sb += WK_REQ) {
      // the requests that asked, in order of their numbers: the sb-th to the (sb + WK_REQ - 1)-th of them
      nwk = 0;
      for (int c0 = 0; c0 < a.B; c0 += WK_EPI * 32) {
        const int b = c0 + tid;
        uint4 r0 = make_uint4(0u, 0u, 0u, 0u), r1 = r0, r2 = r0;
        if (tid < WK_EPI * 32 && b < a.B) { const uint4* src = reinterpret_cast<const uint4*>(a.rec + b); r0 = __ldcg(src); r1 = __ldcg(src + 1); r2 = __ldcg(src + 2); }
        const bool want = (int)r2.y == step + 1;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, want);
        if (lane == 0) s_cnt[warp] = __popc(bal);
        __syncthreads();
        int off = nwk;
        for (int w = 0; w < WK_EPI; ++w) { if (w < warp) off += s_cnt[w]; nwk += s_cnt[w]; }
        const int at = off + __popc(bal & ((1u << lane) - 1u)) - sb;
        if (want && at >= 0 && at < WK_REQ) {
          RedDesc d;
          const int64_t zrow = (int64_t)(((uint64_t)r0.y << 32) | r0.x);
          d.z = a.Z + zrow * a.V; d.u = a.U + (size_t)(int)r0.z * a.V;
          d.C = __uint_as_float(r2.x); d.zoff = __uint_as_float(r1.x); d.qoff = d.C != 0.f ? __uint_as_float(r1.y) : -1e30f;   // (lseT may be NaN where it is not needed)
          d.b = b;
          s_desc[at] = d; s_tok[at] = (int)r0.w;
        }
        __syncthreads();
      }
      if (nwk == 0) break;
      const int nreq = min(WK_REQ, nwk - sb), ncol = (nreq + 15) & ~15;
      // head rows of the requests' nodes: the B operand, K-major with the 128-byte swizzle
      for (int idx = tid; idx < nreq * (a.r / 8); idx += WK_THREADS) {
        const int g = idx / (a.r / 8), ck = idx - g * (a.r / 8);
        *reinterpret_cast<uint4*>(sm.Bs + (ck >> 3) * (WK_REQ * 128) + g * 128 + (((ck & 7) ^ (g & 7)) << 4)) =
            __ldg(reinterpret_cast<const uint4*>(a.A + (size_t)s_tok[g] * a.r + ck * 8));
      }
      // ask L2 for this range of the rows that will be read
      for (int x = warp; x < 2 * nreq; x += WK_THREADS / 32) {
        const RedDesc& d = s_desc[x >> 1];
        const __nv_bfloat16* src = ((x & 1) ? d.u : d.z) + t0;
        if (!(x & 1) || d.C != 0.f)
          for (int l = lane * 64; l < tlen; l += 32 * 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + l));
      }
      fence_async_smem();
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (warp < WK_EPI) wk_epilogue(a, sm, nreq, ncol, t0, tlen, tmem_base, nt, pass == 0u, s_desc, s_part);
      else if (a.ring) wk_stream(a, sm, &tmW, ncol, t0, tlen, pass, wreq, tmem_base);
      ++pass;
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (*sm.abort) { dead = true; break; }
      if (tid < nreq) {
        float s = 0.f;
        for (int w = 0; w < WK_EPI; ++w) s += s_part[w * WK_REQ + tid];
        a.part[(size_t)s_desc[tid].b * a.vt_n + cta] = s;
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
// Shared-memory plan: the range of W resident where it fits, else a ring of 128-token blocks (that needs the tensor map).
bool walk_plan(const ts_ctx* ctx, int B, bool tma, WalkPlan* out) {
  const ts_config& c = ctx->cfg;
  const size_t rp = (size_t)(c.r + 63) / 64 * 64, slab = rp * 128;
  const size_t fixed = slab + 64 * 8 + (size_t)((B + ctx->vt_n - 1) / ctx->vt_n) * sizeof(WalkState) + 1024;
  const size_t avail = (size_t)ctx->max_smem - 16 * 1024;   // static shared memory
  const size_t dot = 4 * WK_CHUNK * sizeof(float);
  WalkPlan p{};
  size_t w = (size_t)(ctx->vt_TV / 64) * slab;
  if (w + fixed > avail || ctx->vt_TV / 128 >= 32) {
    if (!tma) return false;
    p.ring = (int)((avail - (fixed < avail ? fixed : avail)) / (2 * slab));
    p.ring = p.ring > 8 ? 8 : p.ring;
    if (p.ring < 2) return false;
    w = (size_t)p.ring * 2 * slab;
  }
  if (w < dot) w = (dot + 1023) & ~(size_t)1023;
  if (w + fixed > avail) return false;
  p.oB = (uint32_t)w; p.oS = (uint32_t)(w + slab); p.smem = w + fixed;
  *out = p;
  return true;
}

size_t walk_ws_bytes(const ts_ctx* ctx, int B) {
  const size_t b = (size_t)B, n = (size_t)ctx->cfg.Nmax;
  return align_up(b * (n + 1) * sizeof(NodeDesc), 256) + align_up(b * (n + 1) * 8, 256) + align_up(b * n * sizeof(WalkEdge), 256) + align_up(b * sizeof(WalkRec), 256);
}

cudaError_t walk_setup(ts_ctx* ctx) { return allow_all_smem(walk_mma_kernel, ctx->max_smem); }

cudaError_t launch_walk_mma(ts_ctx* ctx, WalkArgs& a, char* ws, const WalkPlan& p, cudaStream_t st) {
  const size_t b = (size_t)a.B, n = (size_t)a.N;
  a.node = (NodeDesc*)ws; ws += align_up(b * (n + 1) * sizeof(NodeDesc), 256);
  a.child = (int2*)ws; ws += align_up(b * (n + 1) * 8, 256);
  a.edge = (WalkEdge*)ws; ws += align_up(b * n * sizeof(WalkEdge), 256);
  a.rec = (WalkRec*)ws;
  a.ring = p.ring; a.oB = p.oB; a.oS = p.oS;
  CUtensorMap tm;
  memset(&tm, 0, sizeof(tm));
  if (a.use_tma) memcpy(&tm, ctx->tmapW, sizeof(tm));
  ProfScope ps(ctx, K_WALK, st);
  // (chained to the row statistics: the W load and the tensor-memory allocation run beside them)
  void* kargs[] = {(void*)&a, (void*)&tm};
  return launch_cooperative(ctx->walk_unchained, (const void*)walk_mma_kernel, dim3(a.vt_n), dim3(WK_THREADS), p.smem, st, kargs);
}

}  // namespace ts
