// The whole expansion of a batch in one cooperative launch (bf16 inputs on the 5th-generation tensor cores).
//
// One CTA per SM holds one vocabulary range for the whole launch.  A level of the trees is two phases, each
// closed by a bounded grid barrier:
//   scan   every CTA scores all of the level's parents on its range: the low-rank bias [128 parents x r].[r x BN
//          tokens] is a tcgen05 tile per block of BN tokens, W streams through a ring of bulk-tensor loads (and runs
//          ahead across levels: it does not depend on them), and 16 warps read the accumulators (one tensor-memory
//          lane = one parent), add the base logits (from L2, where a prefetch of the group's rows put them, or from a
//          ring of their own), and keep (max reference, sums) and the few tokens that can be among a parent's K best.
//   owner  the CTA that owns a request merges the request's parents (one warp each), runs the level step and makes
//          the next level's parent list with its seed bounds; the CTAs without a request meanwhile sweep the base
//          logits of the level after (best token of every 1024: where the next seed bounds come from).
// Before this, a level was three dependent launches (scan with its own set-up, merge of fixed-size records, level
// step on global-memory state): about 70 us per level at 32 requests, V = 151,936, r = 64, of which the arithmetic
// needs less than ten.  Now (serve shape: 32 requests, 16 nodes): 12 to 30 us of scan, 11 to 19 us of owner phase and two
// grid barriers of 1.2 to 2.3 us per level, 192 us for the expansion and 6 for its set-up launch (365 with three launches a level).
//
// Bounds.  Per parent K slots in global memory, slot j = best value published by the pieces (range, split, replica)
// whose number is j mod K; pieces hold disjoint tokens, so the minimum over the slots is a lower bound of the K-th
// best value and a token strictly below it is skipped.  The scan starts from the parent's seed bounds: the K-th
// best exact value among the tokens with the largest base logits, less a rounding margin.
#include <math.h>
#include <string.h>

#include "ts_tree.cuh"

namespace ts {

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// sixteen consecutive bf16 (32-byte aligned when `wide`): read once, so not kept in L1; hi = false: only the first eight exist
__device__ __forceinline__ void load16_bf16(const __nv_bfloat16* p, const bool wide, const bool hi, uint4& a, uint4& b) {
  if (wide) {
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
  } else {
    a = __ldcg(reinterpret_cast<const uint4*>(p));
    if (hi) b = __ldcg(reinterpret_cast<const uint4*>(p) + 1);
  }
}
// Shared-memory state of a CTA.
struct TxSm {
  unsigned char *As, *Ws, *Us;
  unsigned long long* q;       // [TX_QCAP] queued candidates (QEntry)
  float* lists;                // [128][lstride]: topv, topi, keyv, keyi, keyl of every row, sorted (value desc, token asc)
  int* ln;                     // [2][128] entries in use
  volatile float* lthr;        // [2][128] K-th best of the row's own list (-inf until it is full)
  volatile float* best;        // [2][TX_SPLIT][128] best value published by the piece (row, split)
  float* part;                 // [3][TX_SPLIT][128] reference, sum, tempered sum of every (split, row)
  float* ghi;                  // [512] noise bounds
  volatile float* thr;         // [2][128] launch-wide bounds of the rows' parents
  ParentEntry* ent;            // [128] the group's parents by tile row
  uint64_t *a_full, *t_full, *t_empty, *w_full, *w_free, *u_full, *u_free;
  uint32_t* tmem;
  volatile int *abort, *done;
  volatile unsigned* q_head; unsigned* q_tail;
};

// words between two rows' lists: no multiple of four, so that at most two of the threads of neighbouring rows read the same bank
constexpr int list_stride(int K) { return 5 * K + (K % 4 == 0 ? 1 : 0); }
constexpr size_t tx_select_bytes(int K) {
  return (size_t)TX_QCAP * 8 + (size_t)TX_ROWS * list_stride(K) * 4 + 2 * TX_ROWS * 4 + 2 * TX_ROWS * 4 + 2 * TX_SPLIT * TX_ROWS * 4 + 3 * TX_SPLIT * TX_ROWS * 4;
}
constexpr size_t TX_FIXED_BYTES = 512 * 4 + 2 * TX_ROWS * 4 + TX_ROWS * sizeof(ParentEntry) + (1 + 4 * TX_STAGE_MAX + 2 * TX_USTAGES) * 8 + 64;

__device__ __forceinline__ TxSm tx_carve(unsigned char* sm, const TreeArgs& a) {
  TxSm s;
  s.As = sm; s.Ws = sm + a.oW; s.Us = sm + a.oU;
  s.q = reinterpret_cast<unsigned long long*>(sm + a.oL);
  s.lists = reinterpret_cast<float*>(s.q + TX_QCAP);
  s.ln = reinterpret_cast<int*>(s.lists + (size_t)TX_ROWS * a.lstride);
  s.lthr = reinterpret_cast<float*>(s.ln + 2 * TX_ROWS);
  s.best = s.lthr + 2 * TX_ROWS;
  s.part = const_cast<float*>(s.best) + 2 * TX_SPLIT * TX_ROWS;
  s.ent = reinterpret_cast<ParentEntry*>(sm + a.oX);
  s.ghi = reinterpret_cast<float*>(s.ent + TX_ROWS);
  s.thr = s.ghi + 512;
  uint64_t* bars = reinterpret_cast<uint64_t*>(const_cast<float*>(s.thr) + 2 * TX_ROWS);
  s.a_full = bars; s.t_full = bars + 1; s.t_empty = s.t_full + TX_STAGE_MAX; s.w_full = s.t_empty + TX_STAGE_MAX; s.w_free = s.w_full + TX_STAGE_MAX;
  s.u_full = s.w_free + TX_STAGE_MAX; s.u_free = s.u_full + TX_USTAGES;
  s.tmem = reinterpret_cast<uint32_t*>(s.u_free + TX_USTAGES);
  s.abort = reinterpret_cast<volatile int*>(s.tmem + 1);
  s.done = reinterpret_cast<volatile int*>(s.tmem + 2);
  s.q_head = reinterpret_cast<volatile unsigned*>(s.tmem + 3);
  s.q_tail = s.tmem + 4;
  return s;
}

// A queued candidate in one 64-bit word, so that a plain store publishes it whole: logit in the high half; below it a tag
// that changes with every turn of the queue (4 bits), kind (2), split (2), row (7), place in the range (TX_PLACE_BITS).  (With the tag
// in a word of its own a fence had to stand between the two stores, and the fence waited for the scanning thread's
// base-logit loads in flight: two microseconds a candidate.)
__device__ __forceinline__ uint32_t q_tag(unsigned idx) { return (idx / TX_QCAP) % 15u + 1u; }   // never 0: 0 = nothing written
__device__ __forceinline__ unsigned long long q_pack(float lg, unsigned idx, uint32_t kind, int split, int row, int off) {
  return ((unsigned long long)__float_as_uint(lg) << 32) | (q_tag(idx) << 28) | (kind << 26) | ((uint32_t)split << 24) | ((uint32_t)row << TX_PLACE_BITS) | (uint32_t)off;
}

// insertion into one sorted list of at most K entries (value desc, token asc); returns the K-th value (-inf: not full)
__device__ __forceinline__ float tx_insert(float* v, int* t, float* aux, int& n, int K, float val, int tok, float lg) {
  int pos = n < K ? n : K - 1;
  if (n == K && !(val > v[pos] || (val == v[pos] && (unsigned)tok < (unsigned)t[pos]))) return v[pos];
  while (pos > 0 && (val > v[pos - 1] || (val == v[pos - 1] && (unsigned)tok < (unsigned)t[pos - 1]))) {
    v[pos] = v[pos - 1]; t[pos] = t[pos - 1];
    if (aux) aux[pos] = aux[pos - 1];
    --pos;
  }
  v[pos] = val; t[pos] = tok;
  if (aux) aux[pos] = lg;
  n = n < K ? n + 1 : K;
  return n == K ? v[K - 1] : -INFINITY;
}

// The sampling key of one token, exactly (both generator streams).
__device__ __forceinline__ float exact_key(uint64_t seed, int req, uint64_t hash, int tok, float lg, float invT) {
  const uint4 cw = stream_words(seed, req, hash, STREAM_GUMBEL_COARSE, (uint32_t)tok >> 3);
  const uint4 fw = stream_words(seed, req, hash, STREAM_GUMBEL_FINE, (uint32_t)tok >> 3);
  const uint32_t c16 = (word_of(cw, (tok & 7) >> 1) >> (16 * (tok & 1))) & 0xFFFFu;
  const uint32_t f16 = (word_of(fw, (tok & 7) >> 1) >> (16 * (tok & 1))) & 0xFFFFu;
  return lg * invT + gumbel_from_bits((c16 << 16) | f16);
}

// Coarse words of the sampling uniforms, with everything that is fixed per parent worked out once: of the generator's
// counter only the index changes from call to call, and it reaches the other lane pair one round later, so one of the
// two products of the first round and one of the second are constants of the parent.
struct CoarseGen {
  uint32_t x0, y2, y3, c3;
  __device__ __forceinline__ void init(const uint32_t* rk, int req, uint64_t hash) {
    c3 = (((uint32_t)req & 0xFFFFFFu) | ((uint32_t)STREAM_GUMBEL_COARSE << 24)) ^ rk[1];
    const uint32_t c1 = (uint32_t)hash, c2 = (uint32_t)(hash >> 32);
    const uint32_t n0 = __umulhi(0xCD9E8D57u, c2) ^ c1 ^ rk[0];   // round 1, word 0
    y2 = __umulhi(0xD2511F53u, n0) ^ rk[3];                        // round 2, word 2 = y2 ^ (word 3 of round 1)
    y3 = 0xD2511F53u * n0;                                         // round 2, word 3
    x0 = (0xCD9E8D57u * c2) ^ rk[2];                               // round 2, word 0 = hi(M1 * word 2 of round 1) ^ x0
  }
  // rk: the twenty round keys (kernel parameters: an exclusive-or takes one as its constant operand)
  __device__ __forceinline__ uint4 words(const uint32_t* rk, uint32_t index) const {
    const uint64_t pi = mul_wide(0xD2511F53u, index);
    const uint32_t a2 = (uint32_t)(pi >> 32) ^ c3, a3 = (uint32_t)pi;
    const uint64_t pa = mul_wide(0xCD9E8D57u, a2);
    uint32_t c0 = (uint32_t)(pa >> 32) ^ x0, c1 = (uint32_t)pa, c2 = y2 ^ a3, cc3 = y3;
#pragma unroll
    for (int i = 2; i < 10; ++i) {
      const uint64_t p0 = mul_wide(0xD2511F53u, c0), p1 = mul_wide(0xCD9E8D57u, c2);
      c0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk[2 * i]; c1 = (uint32_t)p1; c2 = (uint32_t)(p0 >> 32) ^ cc3 ^ rk[2 * i + 1]; cc3 = (uint32_t)p0;
    }
    return make_uint4(c0, c1, c2, cc3);
  }
};

// One candidate, handled by one lane of the selecting warp: exact key, insertion, publication.
__device__ __forceinline__ void tx_select(const TreeArgs& a, const TxSm& sm, const unsigned long long e, float invT, int tile, int R, int g) {
  const int K = a.K, tok = tile * a.TV + (int)((uint32_t)e & ((1u << TX_PLACE_BITS) - 1u));
  const float lg = __uint_as_float((uint32_t)(e >> 32));
  const int row = (int)((uint32_t)e >> TX_PLACE_BITS) & 127, s = (int)((uint32_t)e >> 24) & 3;
  const uint32_t kind = ((uint32_t)e >> 26) & 3u;
  const int per = TX_ROWS / R;
  const int prow = R > 1 ? row % per : row, rho = R > 1 ? row / per : 0;
  const int p = g * TX_ROWS + prow;
  const int pid = ((tile * TX_SPLIT + s) * R + rho) % K;
  float* L = sm.lists + (size_t)row * a.lstride;
  if (kind & 1u) {
    if (lg >= sm.thr[prow] && lg >= sm.lthr[row]) {
      sm.lthr[row] = tx_insert(L, reinterpret_cast<int*>(L) + K, nullptr, sm.ln[row], K, lg, tok, 0.f);
      volatile float* b = sm.best + s * TX_ROWS + row;
      if (lg > *b) { *b = lg; atomicMax(a.slots + ((size_t)p * K + pid) * SLOT_STRIDE, enc_f(lg)); }
    }
  }
  if (kind & 2u) {
    const float thr = fmaxf(sm.thr[TX_ROWS + prow], sm.lthr[TX_ROWS + row]);
    const ParentEntry& pe = sm.ent[row];
    const uint4 cw = stream_words(a.seed, pe.req, pe.hash, STREAM_GUMBEL_COARSE, (uint32_t)tok >> 3);
    const uint32_t c16 = (word_of(cw, (tok & 7) >> 1) >> (16 * (tok & 1))) & 0xFFFFu;
    if (lg * invT + sm.ghi[noise_bound_index(c16)] >= thr) {   // the bounds have often risen since the candidate was queued
      const uint4 fw = stream_words(a.seed, pe.req, pe.hash, STREAM_GUMBEL_FINE, (uint32_t)tok >> 3);
      const uint32_t f16 = (word_of(fw, (tok & 7) >> 1) >> (16 * (tok & 1))) & 0xFFFFu;
      const float key = lg * invT + gumbel_from_bits((c16 << 16) | f16);
      if (key >= thr) {
        sm.lthr[TX_ROWS + row] = tx_insert(L + 2 * K, reinterpret_cast<int*>(L) + 3 * K, L + 4 * K, sm.ln[TX_ROWS + row], K, key, tok, lg);
        volatile float* b = sm.best + (TX_SPLIT + s) * TX_ROWS + row;
        if (key > *b) { *b = key; atomicMax(a.slots + (((size_t)a.cap + p) * K + pid) * SLOT_STRIDE, enc_f(key)); }
      }
    }
  }
}

__device__ __noinline__ bool tx_wait_slow(uint64_t* bar, uint32_t parity, volatile int* abort, int* err, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
    if (i > 64) __nanosleep(64);
  }
  *abort = 1;
  atomicExch(err, 1);
  return false;
}
__device__ __forceinline__ bool tx_wait(uint64_t* bar, uint32_t parity, const TxSm& sm, const TreeArgs& a) {
  return mbar_try_wait(bar, parity) || tx_wait_slow(bar, parity, sm.abort, a.err, a.wait_limit);
}
// the same by a whole warp, one answer for all its lanes
__device__ __forceinline__ bool tx_wait_warp(uint64_t* bar, uint32_t parity, const TxSm& sm, const TreeArgs& a) {
  return __all_sync(0xFFFFFFFFu, tx_wait(bar, parity, sm, a));
}

// a polling loop that ran out: the scan is given up and the call reports it
__device__ __forceinline__ void tx_give_up(const TxSm& sm, const TreeArgs& a) { *sm.abort = 1; atomicExch(a.err, 1); }

// ---- scanning warps: one group of up to 128 parents over this CTA's range ---------------------------------
// Cost: two generator calls (76 multiply-xor steps), 16 ex2 and about 100 other instructions per 16 tokens and
// parent; a warp owns every (4R)-th chunk of 16 tokens, so with few parents (R = 2, 4 replicas of the rows) the
// copies share the range.
template <bool RING>
__device__ __forceinline__ void tx_scan(const TreeArgs& a, const TxSm& sm, const int R, const int P, const int g, const int t0, const int tlen,
                                        const uint32_t tmem_base, BlockPos& pos, const int nst, const uint32_t ub0) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q = warp & 3, s = warp >> 2;
  const int per = TX_ROWS / R, K = a.K;
  (void)K;
  {
    const int cpr = (a.r + 63) / 64 * 8;          // 16-byte chunks per A row
    const __nv_bfloat16* Ag = reinterpret_cast<const __nv_bfloat16*>(a.A);
    for (int idx = tid; idx < TX_ROWS * cpr; idx += TX_SCAN_WARPS * 32) {
      const int rr = idx / cpr, ck = idx % cpr;
      const ParentEntry& pe = sm.ent[rr];
      const bool in = pe.row >= 0 && ck * 8 < a.r;
      cp_async16(sm.As + (size_t)(ck >> 3) * (TX_ROWS * 128) + rr * 128 + (((ck & 7) ^ (rr & 7)) << 4), in ? Ag + (size_t)pe.token * a.r + ck * 8 : Ag, in);
    }
    cp_async_wait_all();
    fence_async_smem();
    mbar_arrive(sm.a_full);
  }
  const int row = q * 32 + lane;
  const ParentEntry& me = sm.ent[row];
  const bool active = me.row >= 0;
  const int prow = R > 1 ? row % per : row, rho = R > 1 ? row / per : 0;   // rho is uniform within a warp
  const float T = a.T, invT = T > 0.f ? 1.f / T : 1.f;
  const bool keys = T > 0.f, two = keys && T != 1.f;
  const float slack = 8.f * fminf(1.f, T > 0.f ? T : 1.f);   // how far a logit may exceed the sums' reference
  CoarseGen gen; gen.init(a.rk, me.req, me.hash);
  float m = me.mref, s0 = 0.f, sT = 0.f;
  const int CB = a.BN / 16, nblk = (tlen + a.BN - 1) / a.BN, stride = R * TX_SPLIT, own = rho * TX_SPLIT + s;
  const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16);
  // Base logits, straight from L2: 32 bytes of its parent's row per lane and chunk (a scan reads each once; lanes whose
  // parents share a row read the same sector).  A copying warp could not keep up with 128 different rows: 3 us per block
  // of 128 tokens by 16-byte cp.async, 6 us by one bulk copy per row.
  // RING: by bulk-tensor boxes of 64 tokens of every request at the level's depth, swizzled so that lanes of any eight
  // neighbouring requests read different banks.  A warp whose lanes read 32 different rows touches 32 pages with every
  // load: a scan of 128 parents on 128 rows took 50 us in the median CTA and 72 us in the slowest, against 34 and 36 when
  // all lanes read one row; the box costs about 33 cycles a row, 40 us a scan of the same level.  Batches of 32 were
  // slower this way (383 -> 396 us a round), a batch of 128 with three groups of parents a level the same.
  const __nv_bfloat16* urow = reinterpret_cast<const __nv_bfloat16*>(a.Uscan) + (size_t)max(me.row, 0) * a.Vs + t0;
  const int vleft = a.Vs - t0;   // tokens of the row from t0 on (whole 16 bytes)
  int o = own * 16;              // the next chunk to request
  uint4 nx0 = make_uint4(0u, 0u, 0u, 0u), nx1 = nx0;
  const bool wide = a.wide_u != 0;
  if (!RING && o < tlen) load16_bf16(urow + o, wide, o + 8 < vleft, nx0, nx1);
  const uint32_t uoff = (uint32_t)me.req * 128u, usw = (uint32_t)me.req & 7u, uslab = (uint32_t)a.rowsU * 128u;
  bool alive = true;
  for (int nb = 0; nb < nblk; ++nb, pos.next(nst)) {
    const int slot = pos.slot;
    if (!tx_wait_warp(sm.t_full + slot, pos.full(), sm, a)) { alive = false; break; }
    const uint32_t ust = RING ? (ub0 + (uint32_t)nb) & (uint32_t)(TX_USTAGES - 1) : 0u;
    if (RING && !tx_wait_warp(sm.u_full + ust, ((ub0 + (uint32_t)nb) / TX_USTAGES) & 1u, sm, a)) { alive = false; break; }
    const unsigned char* ublk = sm.Us + (size_t)ust * (a.BN / 64) * uslab + uoff;
    tc_fence_after();
    const int nch = min(CB, (tlen - nb * a.BN + 15) / 16);
    for (int c = (own - nb * CB) & (stride - 1); c < nch; c += stride) {
      uint32_t ra[16];
      __syncwarp();   // (the tensor-memory load is a warp-wide instruction)
      tmem_ld16_issue(trow + (uint32_t)(slot * a.BN + c * 16), ra);
      uint4 u0 = nx0, u1 = nx1;   // requested one owned chunk ago; the next one's are requested now
      if (RING) {
        const unsigned char* up = ublk + (uint32_t)(c >> 2) * uslab;
        const uint32_t j = (uint32_t)(c & 3) * 2u;
        u0 = *reinterpret_cast<const uint4*>(up + ((j ^ usw) << 4)); u1 = *reinterpret_cast<const uint4*>(up + (((j + 1u) ^ usw) << 4));
      }
      o += stride * 16;
      if (!RING && o < tlen) load16_bf16(urow + o, wide, o + 8 < vleft, nx0, nx1);
      const int v0 = t0 + nb * a.BN + c * 16, valid = min(16, a.V - v0);
      // high halves of the sixteen uniforms: issued first, their long dependent chains overlap the rest
      uint4 cw0 = make_uint4(0, 0, 0, 0), cw1 = cw0;
      if (keys) { cw0 = gen.words(a.rk, (uint32_t)v0 >> 3); cw1 = gen.words(a.rk, ((uint32_t)v0 >> 3) + 1u); }
      tmem_ld_wait();
      if (!active) continue;
      float acc[16];
      unpack_bf16x8(u0, acc); unpack_bf16x8(u1, acc + 8);
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[i] += __uint_as_float(ra[i]);
      if (valid < 16) {   // warp-uniform: the vocabulary's last chunk
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = (i < valid) ? acc[i] : -INFINITY;
      }
      const float thrL = sm.thr[prow], thrK = sm.thr[TX_ROWS + prow];
      float gmax[4], cm = -INFINITY;
#pragma unroll
      for (int sg = 0; sg < 4; ++sg) {
        gmax[sg] = fmaxf(fmaxf(acc[4 * sg], acc[4 * sg + 1]), fmaxf(acc[4 * sg + 2], acc[4 * sg + 3]));
        cm = fmaxf(cm, gmax[sg]);
      }
      if (cm > m + slack) {   // rare: the reference is an exact logit of one of the parent's best tokens
        const float d = m == -INFINITY ? 0.f : m - cm;
        s0 *= __expf(d); sT *= __expf(d * invT);
        m = cm;
      }
      {
        // exp(l - m) as ex2(l log2(e) - m log2(e)); while nothing finite has been seen every l is -inf and adds 0
        constexpr float LOG2E = 1.4426950408889634f;
        const float off0 = m == -INFINITY ? 0.f : -m * LOG2E, scT = LOG2E * invT, offT = off0 * invT;
        float a0 = 0.f, a1 = 0.f, aT = 0.f, aU = 0.f;
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          a0 += ex2_approx(fmaf(acc[i], LOG2E, off0));
          a1 += ex2_approx(fmaf(acc[i + 1], LOG2E, off0));
          if (two) { aT += ex2_approx(fmaf(acc[i], scT, offT)); aU += ex2_approx(fmaf(acc[i + 1], scT, offT)); }
        }
        a0 += a1;
        s0 += a0;
        sT += two ? aT + aU : a0;
      }
      uint32_t mkK = 0, mkL = 0;
      if (cm >= thrL) {
#pragma unroll
        for (int i = 0; i < 16; ++i) mkL |= (uint32_t)(acc[i] >= thrL && acc[i] > -INFINITY) << i;
      }
      if (keys) {
        // the whole chunk first: its best logit plus the noise bound of the largest leading bits bounds every key
        // in it; then four tokens at a time, then singly
        const uint32_t m8 = __vmaxu2(__vmaxu2(__vmaxu2(cw0.x, cw0.y), __vmaxu2(cw0.z, cw0.w)),
                                     __vmaxu2(__vmaxu2(cw1.x, cw1.y), __vmaxu2(cw1.z, cw1.w)));
        const uint32_t c16all = max(m8 & 0xFFFFu, m8 >> 16);
        if (cm * invT + sm.ghi[noise_bound_index(c16all)] >= thrK && cm > -INFINITY) {
#pragma unroll
          for (int sg = 0; sg < 4; ++sg) {
            const uint4& cw = sg < 2 ? cw0 : cw1;
            const uint32_t wa = (sg & 1) ? cw.z : cw.x, wb = (sg & 1) ? cw.w : cw.y;
            const uint32_t m2 = __vmaxu2(wa, wb);
            const uint32_t c16m = max(m2 & 0xFFFFu, m2 >> 16);
            if (gmax[sg] * invT + sm.ghi[noise_bound_index(c16m)] >= thrK && gmax[sg] > -INFINITY) {
#pragma unroll
              for (int i = 4 * sg; i < 4 * sg + 4; ++i) {
                const uint32_t word = word_of(i < 8 ? cw0 : cw1, (i & 7) >> 1);
                const uint32_t c16 = (word >> (16 * (i & 1))) & 0xFFFFu;
                mkK |= (uint32_t)(acc[i] * invT + sm.ghi[noise_bound_index(c16)] >= thrK && acc[i] > -INFINITY) << i;
              }
            }
          }
        }
      }
      uint32_t mk = mkK | mkL;
#pragma unroll 1
      while (mk) {   // rare: hand the token to the selecting warp
        const int i = __ffs(mk) - 1;
        mk &= mk - 1;
        const uint32_t kind = ((mkL >> i) & 1u) | ((mkK >> i) & 1u) << 1;
        const unsigned idx = atomicAdd(sm.q_tail, 1u);
        uint32_t spin = 0;
        while ((int)(idx - *sm.q_head) >= TX_QCAP) {   // queue full: the selecting warp is behind
          if (*sm.abort) break;
          if (++spin > a.wait_limit) { *sm.abort = 1; atomicExch(a.err, 1); break; }
          __nanosleep(64);
        }
        *reinterpret_cast<volatile unsigned long long*>(sm.q + (idx & (TX_QCAP - 1))) = q_pack(pick16(acc, i), idx, kind, s, row, v0 + i - t0);
      }
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) { mbar_arrive(sm.t_empty + slot); if (RING) mbar_arrive(sm.u_free + ust); }
  }
  sm.part[(0 * TX_SPLIT + s) * TX_ROWS + row] = m; sm.part[(1 * TX_SPLIT + s) * TX_ROWS + row] = s0; sm.part[(2 * TX_SPLIT + s) * TX_ROWS + row] = sT;
  __threadfence_block();
  __syncwarp();
  if (lane == 0) atomicAdd((int*)sm.done, alive ? 1 : (1 << 20));   // one tick per warp per group (a large one releases the others after a failed wait)
}

// ---- W blocks into their ring (by the refreshing warp) ----------------------------------------------------------------
// `upto`: blocks of the whole launch that may be requested while this group runs.  Requests run on into the next scan (W
// does not depend on which parents that will score) except where the owners work in the ring.  Not the issuing warp's
// business: a request costs its thread most of a microsecond of instruction latency, which held up the MMAs.
struct WLoad { BlockPos pos; int nb; uint32_t requested; };
template <bool BLOCKING>
__device__ __forceinline__ void tx_load(const TreeArgs& a, const TxSm& sm, const CUtensorMap* tm, const int t0, const int tlen, WLoad& w, const uint32_t upto) {
  const int nblk = (tlen + a.BN - 1) / a.BN, rw = (a.r + 15) / 16 * 16;
  const uint32_t slab = (uint32_t)rw * 128u;
  for (; w.requested < upto; ++w.requested, w.pos.next(a.nW)) {
    if (w.pos.reused()) {
      if (BLOCKING) { if (!tx_wait_warp(sm.w_free + w.pos.slot, w.pos.empty(), sm, a)) return; }
      else if (!__all_sync(0xFFFFFFFFu, mbar_test_wait(sm.w_free + w.pos.slot, w.pos.empty()))) return;
    }
    if (!a.use_tma) {   // no tensor map: 16-byte copies into the same swizzled places
      const int CB8 = a.BN / 8, sh = a.BN == 128 ? 4 : 3, lane = threadIdx.x & 31;
      const int ck = lane & (CB8 - 1), r0 = lane >> sh, rstep = 32 >> sh, v = t0 + w.nb * a.BN + ck * 8;
      const __nv_bfloat16* Wg = reinterpret_cast<const __nv_bfloat16*>(a.Wscan);
      unsigned char* wd = sm.Ws + (size_t)(w.pos.slot * (a.BN / 64)) * slab;
      for (int k = r0; k < rw; k += rstep) {
        const bool in = v < a.Vs && k < a.r;
        cp_async16(wd + (size_t)(ck >> 3) * slab + k * 128 + (((ck & 7) ^ (k & 7)) << 4), in ? Wg + (size_t)k * a.Vs + v : Wg, in);
      }
      cp_async_wait_all();
      fence_async_smem();
      mbar_arrive(sm.w_full + w.pos.slot);
    } else if (elect_one()) {
      const int ns = min(a.BN / 64, (tlen - w.nb * a.BN + 63) / 64);
      mbar_expect_tx(sm.w_full + w.pos.slot, (uint32_t)ns * slab);
      unsigned char* dst = sm.Ws + (size_t)(w.pos.slot * (a.BN / 64)) * slab;
      for (int h = 0; h < ns; ++h) tma_load_box(dst + (size_t)h * slab, tm, t0 + w.nb * a.BN + h * 64, 0, sm.w_full + w.pos.slot);
    }
    __syncwarp();
    if (++w.nb == nblk) w.nb = 0;
  }
}

// ---- base logits of a block of tokens, of every request at the level's depth, into their ring (by the same warp) --------
// `uend`: blocks of the whole launch up to the end of the group's.
struct ULoad { uint32_t requested; };
__device__ __forceinline__ void tx_load_u(const TreeArgs& a, const TxSm& sm, const CUtensorMap* tm, const int t0, const int tlen, const int depth, ULoad& u, const uint32_t uend) {
  const uint32_t nblk = (uint32_t)((tlen + a.BN - 1) / a.BN), uslab = (uint32_t)a.rowsU * 128u;
  for (; u.requested < uend; ++u.requested) {
    const uint32_t st = u.requested & (uint32_t)(TX_USTAGES - 1), use = u.requested / TX_USTAGES;
    if (use > 0u && !__all_sync(0xFFFFFFFFu, mbar_test_wait(sm.u_free + st, (use - 1u) & 1u))) return;
    if (elect_one()) {
      const int off = (int)(nblk - (uend - u.requested)) * a.BN, ns = min(a.BN / 64, (tlen - off + 63) / 64);
      mbar_expect_tx(sm.u_full + st, (uint32_t)ns * uslab);
      for (int h = 0; h < ns; ++h) tma_load_box3(sm.Us + ((size_t)st * (a.BN / 64) + h) * uslab, tm, t0 + off + h * 64, depth, 0, sm.u_full + st);
    }
    __syncwarp();
  }
}

// ---- the issuing warps: one tile of MMAs per block, in turn ---------------------------------------------------------------
// (Waiting, issuing and committing a block of four MMAs takes a warp 0.75 us, of sixteen 0.9: one warp for the nine blocks of 128 tokens,
// or the seventeen of 64 at rank 256, was what scans of few parents waited for.  An accumulator stage may change hands: who
// issues block j has waited, at most three blocks earlier, until a block after j - 2 stages was drained, so that its parity is never two turns off.)
__device__ __forceinline__ void tx_issue(const TreeArgs& a, const TxSm& sm, const int which, const int tlen, const uint32_t tmem_base, BlockPos& pos, BlockPos& wpos, const int group_no, const int nst) {
  const int nblk = (tlen + a.BN - 1) / a.BN, ksteps = (a.r + 15) / 16;
  const uint32_t slab = (uint32_t)ksteps * 2048u;
  const uint64_t adesc0 = smem_desc(smem_u32(sm.As), 16u, 1024u), bdesc0 = smem_desc(smem_u32(sm.Ws), slab, 1024u);
  if (!tx_wait_warp(sm.a_full, group_no & 1, sm, a)) return;
  for (int nb = 0; nb < nblk; ++nb, pos.next(nst), wpos.next(a.nW)) {
    if (wpos.slot % TX_ISSUERS != which) continue;   // (by the ring's slots: a wait for a parity is right only for who follows every turn of a slot)
    if (!tx_wait_warp(sm.w_full + wpos.slot, wpos.full(), sm, a)) return;
    if (pos.reused() && !tx_wait_warp(sm.t_empty + pos.slot, pos.empty(), sm, a)) return;
    tc_fence_after();
    if (elect_one()) {
      const int n = min(a.BN, (tlen - nb * a.BN + 63) / 64 * 64);   // whole 64-token slabs
      const uint32_t idesc = instr_desc(n), d = tmem_base + (uint32_t)(pos.slot * a.BN);
      const uint64_t bd = bdesc0 + (uint64_t)((uint32_t)(wpos.slot * (a.BN / 64)) * (slab >> 4));
#pragma unroll 4
      for (int ks = 0; ks < ksteps; ++ks)
        mma_bf16(d, adesc0 + (uint64_t)((ks >> 2) * (TX_ROWS * 128 / 16) + (ks & 3) * 2), bd + (uint64_t)(ks * 128), idesc, ks > 0 ? 1u : 0u);
      mma_commit(sm.t_full + pos.slot);
      mma_commit(sm.w_free + wpos.slot);
    }
    __syncwarp();
  }
}

// ---- the refreshing warp -----------------------------------------------------------------------------------------
// Condenses the slots of the parents this CTA is responsible for (parent p belongs to range p mod ntiles) into two
// words per parent and copies the condensed words of its rows into shared memory, until the scan is over.
template <bool RING>
__device__ __forceinline__ void tx_refresh(const TreeArgs& a, const TxSm& sm, const int R, const int P, const int g, const int tile, const int done_target,
                                           const CUtensorMap* tm, const int t0, const int tlen, WLoad& w, const uint32_t upto,
                                           const CUtensorMap* tmU, const int depth, ULoad& u, const uint32_t uend) {
  const int lane = threadIdx.x & 31, per = TX_ROWS / R, K = a.K;
  const int p_lo = g * TX_ROWS, p_hi = min(P, p_lo + per), nt = a.ntiles;
  const int p_own = p_lo + ((tile - p_lo % nt + nt) % nt);
  const int which = lane >> 4, j = lane & 15;
  for (uint32_t spin = 0; spin < a.wait_limit; ++spin) {
    if (RING) tx_load_u(a, sm, tmU, t0, tlen, depth, u, uend);
    tx_load<false>(a, sm, tm, t0, tlen, w, upto);
    if (*sm.done >= done_target || *sm.abort) break;
    // (a pass is a memory round trip: steady at first, while the bounds rise, every eighth turn later, so that the end of
    // the scan is seldom waited for)
    if (spin >= 12u && (spin & 7u)) { __nanosleep(100); continue; }
    unsigned v = 0xFFFFFFFFu;
    if (p_own < p_hi && j < K) v = __ldcg(a.slots + (((size_t)which * a.cap + p_own) * K + j) * SLOT_STRIDE);
    unsigned rL[4], rK[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int rr = lane + 32 * k, p = p_lo + rr;
      const bool in = rr < per && p < P;
      rL[k] = in ? __ldcg(a.thr + p) : 0u;
      rK[k] = in ? __ldcg(a.thr + (size_t)a.cap + p) : 0u;
    }
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v = min(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
    if (p_own < p_hi && j == 0) __stcg(a.thr + (size_t)which * a.cap + p_own, v);
    for (int p = p_own + nt; p < p_hi; p += nt) {
      unsigned w = 0xFFFFFFFFu;
      if (j < K) w = __ldcg(a.slots + (((size_t)which * a.cap + p) * K + j) * SLOT_STRIDE);
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) w = min(w, __shfl_xor_sync(0xFFFFFFFFu, w, off));
      if (j == 0) __stcg(a.thr + (size_t)which * a.cap + p, w);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int rr = lane + 32 * k, p = p_lo + rr;
      if (rr < per && p < P) {   // never below the seed bounds
        sm.thr[rr] = fmaxf(dec_f(rL[k]), sm.ent[rr].thrL);
        sm.thr[TX_ROWS + rr] = fmaxf(dec_f(rK[k]), sm.ent[rr].thrK);
      }
    }
  }
  __syncwarp();
  if (lane == 0 && *sm.done < done_target && !*sm.abort) tx_give_up(sm, a);
  __syncwarp();
  if (!*sm.abort) tx_load<true>(a, sm, tm, t0, tlen, w, upto);
}

// ---- the selecting warp: drains the queue until the scan is over ----------------------------------------------------
__device__ __forceinline__ void tx_drain(const TreeArgs& a, const TxSm& sm, const int R, const int g, const int tile, const int done_target) {
  const int lane = threadIdx.x & 31;
  const float invT = a.T > 0.f ? 1.f / a.T : 1.f;
  unsigned head = *sm.q_head;
  for (uint32_t spin = 0;; ++spin) {
    if (*sm.abort) break;
    if (spin >= a.wait_limit) { if (lane == 0) tx_give_up(sm, a); break; }
    const bool finished = *sm.done >= done_target;   // read before the tail: pushes precede the tick
    const unsigned tail = *reinterpret_cast<volatile unsigned*>(sm.q_tail);
    const int avail = (int)(tail - head);
    if (avail <= 0) {
      if (finished) break;
      __nanosleep(100);
      continue;
    }
    spin = 0;
    const int n = min(avail, 32);
    unsigned long long e = 0ull;
    bool have = false;
    if (lane < n) {
      volatile unsigned long long* slot = sm.q + ((head + lane) & (TX_QCAP - 1));
      const uint32_t tag = q_tag(head + lane);
      for (uint32_t t = 0; t < a.wait_limit; ++t) {   // the producer writes right after claiming: a few cycles
        e = *slot;
        have = (((uint32_t)e >> 28) & 15u) == tag;
        if (have || *sm.abort) break;
      }
    }
    __threadfence_block();
    if (__any_sync(0xFFFFFFFFu, lane < n && !have)) { if (lane == 0) tx_give_up(sm, a); break; }   // (or given up elsewhere)
    head += (unsigned)n;
    if (lane == 0) *sm.q_head = head;   // the slots may be reused
    // candidates of one row are inserted one after the other (lanes of a row take turns)
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, have ? (int)((uint32_t)e >> TX_PLACE_BITS) & 127 : -1 - lane);
    const int turn = __popc(peers & ((1u << lane) - 1u));
    const int turns = __reduce_max_sync(0xFFFFFFFFu, have ? turn + 1 : 0);
    for (int t = 0; t < turns; ++t) {
      if (have && turn == t) tx_select(a, sm, e, invT, tile, R, g);
      __syncwarp();
    }
  }
}

// Copies of the rows in group g.  The copies decide which chunks of the range a partial sum covers, so a parent's sums may have
// copies only by what is the same on every run.  Lists of one group: their length.  Given parents also by group (the place in the list is
// the caller's): the last one may hold few (150 parents: its 22 took as long as the 128 before them, 26 us); not without room for
// the copies' candidates (a.tail_copies).  An expansion's parents come to the list in the order their owners are done.
__device__ __forceinline__ int group_replicas(const TreeArgs& a, const int P, const int g) { return g == 0 || a.tail_copies ? mma_replicas(P - g * TX_ROWS) : 1; }
// where the candidates of parent p start
__device__ __forceinline__ size_t cand_base(const TreeArgs& a, const int P, const int p) {
  const int g = p / TX_ROWS;
  return (size_t)(g * TX_ROWS + (p - g * TX_ROWS) * group_replicas(a, P, g)) * a.ntiles * a.K;
}

// ---- end of a group: the range's sums and surviving candidates of every parent -------------------------------------
// A row's sums, best logits and best keys by three threads side by side (one after the other, with the lists' atomics behind
// the sums, it took 2 us a group).
__device__ __forceinline__ void tx_publish(const TreeArgs& a, const TxSm& sm, const int R, const int P, const int g, const int tile, int* cnt) {
  const int role = (int)threadIdx.x / TX_ROWS, row = (int)threadIdx.x % TX_ROWS, per = TX_ROWS / R, K = a.K;
  if (role > 2) return;
  const int prow = R > 1 ? row % per : row, p = g * TX_ROWS + prow;
  if (p >= P) return;
  if (role == 0) {
    if (row >= per) return;
    const float T = a.T, invT = T > 0.f ? 1.f / T : 1.f;
    // the pieces' sums in a fixed order: the same bits on every run
    float m = -INFINITY, lo = INFINITY, s0 = 0.f, sT = 0.f;
#pragma unroll 1
    for (int rho = 0; rho < R; ++rho)
#pragma unroll
      for (int s = 0; s < TX_SPLIT; ++s) { const float hm = sm.part[(0 * TX_SPLIT + s) * TX_ROWS + rho * per + row]; m = fmaxf(m, hm); lo = fminf(lo, hm); }
    if (lo == m) {   // nearly always (no piece left the parent's reference): plain sums (a running reference takes four copies of a row 1.1 us longer)
#pragma unroll 1
      for (int rho = 0; rho < R; ++rho)
#pragma unroll
        for (int s = 0; s < TX_SPLIT; ++s) { s0 += sm.part[(1 * TX_SPLIT + s) * TX_ROWS + rho * per + row]; sT += sm.part[(2 * TX_SPLIT + s) * TX_ROWS + rho * per + row]; }
      if (m == -INFINITY) sT = 0.f;   // (nothing finite: the sums are 0, or NaN if a piece met one)
    } else {
      m = -INFINITY;
#pragma unroll 1
      for (int rho = 0; rho < R; ++rho)
#pragma unroll
        for (int s = 0; s < TX_SPLIT; ++s) {
          const int rr = rho * per + row;
          const float hm = sm.part[(0 * TX_SPLIT + s) * TX_ROWS + rr], h0 = sm.part[(1 * TX_SPLIT + s) * TX_ROWS + rr], hT = sm.part[(2 * TX_SPLIT + s) * TX_ROWS + rr];
          if (hm == -INFINITY) { s0 += h0; continue; }
          if (hm > m) { const float d = m == -INFINITY ? 0.f : m - hm; s0 *= __expf(d); sT *= __expf(d * invT); m = hm; }
          const float d = hm - m;
          s0 += h0 * __expf(d); sT += hT * __expf(d * invT);
        }
    }
    a.sums[(size_t)p * a.ntiles + tile] = make_float4(m, s0, sT, 0.f);
    return;
  }
  const size_t base = cand_base(a, P, p);
  const float* L = sm.lists + (size_t)row * a.lstride + (role == 2 ? 2 * K : 0);
  const float bound = sm.thr[(role == 2 ? TX_ROWS : 0) + prow];
  const int n = sm.ln[(role == 2 ? TX_ROWS : 0) + row];
  int k = 0;
#pragma unroll 4
  for (int j = 0; j < K; ++j) k += (j < n && L[j] >= bound) ? 1 : 0;   // (sorted: the first k)
  if (k == 0) return;
  const int at = atomicAdd(cnt + (role == 2 ? a.cap : 0) + p, k);
  const int* Li = reinterpret_cast<const int*>(L) + K;
  uint2* out = (role == 2 ? a.cand_key : a.cand_top) + base + at;
#pragma unroll 2
  for (int j = 0; j < k; ++j) {
    out[j] = make_uint2(__float_as_uint(L[j]), (unsigned)Li[j]);
    if (role == 2) a.cand_lg[base + at + j] = L[2 * K + j];
  }
}

// ---- merge of one parent, by one warp --------------------------------------------------------------------------------
// The K best of n (value, token) pairs (value desc, token asc): lane j < K gets the j-th in (tok, val, lg).  The first 96
// entries are picked by rounds of two warp-wide maxima (the value's order-preserving image, then the inverted token among its
// ties) and one removal; of what follows only the few that beat the K-th so far are inserted, one by one.  (Rounds for every
// 96 entries: crowded levels hold several hundred per parent, 24 to 28 us for a parent's three merges at K = 16.)
__device__ __noinline__ float3 warp_topk(const uint2* cand, const float* lgs, const int* count, int K, int lane) {
  uint32_t wv = 0u, wt = 0u; float wl = 0.f;   // winner `lane` so far: 0 = none
  // the first 64 entries are requested together with the count (past a short segment they are a neighbour's, and past the
  // last one's another array of the workspace: not used, and always inside it)
  const int n = __ldcg(count);
  const uint2 pre0 = __ldcg(cand + lane), pre1 = __ldcg(cand + 32 + lane);
  const float pl0 = lgs ? __ldcg(lgs + lane) : 0.f, pl1 = lgs ? __ldcg(lgs + 32 + lane) : 0.f;
#pragma unroll 1
  for (int base = 0; base < n; base += 3 * 32) {
    uint32_t ev[3], et[3]; float el[3];
    const int used = min(3, (n - base + 31) / 32);   // (warp-uniform) slots of 32 entries in this batch
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int i = base + u * 32 + lane;
      ev[u] = 0u; et[u] = 0u; el[u] = 0.f;
      if (u < used && i < n) {
        const uint2 c = (u == 0 && base == 0) ? pre0 : ((u == 1 && base == 0) ? pre1 : __ldcg(cand + i));
        ev[u] = enc_f(__uint_as_float(c.x)); et[u] = ~c.y;
        el[u] = !lgs ? __uint_as_float(c.x) : ((u == 0 && base == 0) ? pl0 : ((u == 1 && base == 0) ? pl1 : __ldcg(lgs + i)));
      }
    }
    if (base == 0) {
#pragma unroll 1
      for (int j = 0; j < K; ++j) {
        uint32_t bv = ev[0], bt = et[0]; float bl = el[0];
#pragma unroll
        for (int u = 1; u < 3; ++u)
          if (u < used && (ev[u] > bv || (ev[u] == bv && et[u] > bt))) { bv = ev[u]; bt = et[u]; bl = el[u]; }
        const uint32_t mv = __reduce_max_sync(0xFFFFFFFFu, bv);
        if (mv == 0u) break;   // warp-uniform
        const uint32_t mt = __reduce_max_sync(0xFFFFFFFFu, bv == mv ? bt : 0u);
        const bool mine = bv == mv && bt == mt;
        const unsigned who = __ballot_sync(0xFFFFFFFFu, mine);
        const float l = __shfl_sync(0xFFFFFFFFu, bl, __ffs(who) - 1);
        if (mine) {
#pragma unroll
          for (int u = 0; u < 3; ++u) if (ev[u] == mv && et[u] == mt) { ev[u] = 0u; et[u] = 0u; }
        }
        if (lane == j) { wv = mv; wt = mt; wl = l; }
      }
      continue;
    }
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      uint32_t tv = __shfl_sync(0xFFFFFFFFu, wv, K - 1), tt = __shfl_sync(0xFFFFFFFFu, wt, K - 1);
      unsigned todo = __ballot_sync(0xFFFFFFFFu, ev[u] > tv || (ev[u] == tv && et[u] > tt));
#pragma unroll 1
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t v = __shfl_sync(0xFFFFFFFFu, ev[u], src), t = __shfl_sync(0xFFFFFFFFu, et[u], src);
        const float l = __shfl_sync(0xFFFFFFFFu, el[u], src);
        const int pos = __popc(__ballot_sync(0xFFFFFFFFu, lane < K && (wv > v || (wv == v && wt > t))));   // (K: beaten by now)
        const uint32_t pv = __shfl_up_sync(0xFFFFFFFFu, wv, 1), pt = __shfl_up_sync(0xFFFFFFFFu, wt, 1);
        const float pl = __shfl_up_sync(0xFFFFFFFFu, wl, 1);
        if (lane < K && lane > pos) { wv = pv; wt = pt; wl = pl; }
        if (lane < K && lane == pos) { wv = v; wt = t; wl = l; }
      }
    }
  }
  return make_float3(__int_as_float(wv ? (int)~wt : -1), wv ? dec_f(wv) : 0.f, wv ? wl : 0.f);   // token (as bits), value, logit
}

// Log-normalisers of a parent from its ranges' sums; every lane gets them.
__device__ __noinline__ float2 warp_lse(const float4* h, const int nt, const float T, int lane) {
  const float invT = T > 0.f ? 1.f / T : 1.f;
  float m = -INFINITY, s0 = 0.f, sT = 0.f;
#pragma unroll 1
  for (int t0 = 0; t0 < nt; t0 += 5 * 32) {
    float4 x[5];
#pragma unroll
    for (int u = 0; u < 5; ++u) { const int t = t0 + u * 32 + lane; x[u] = t < nt ? __ldcg(h + t) : make_float4(-INFINITY, 0.f, 0.f, 0.f); }
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      if (x[u].x == -INFINITY) { s0 += x[u].y; continue; }
      if (x[u].x > m) { const float d = m == -INFINITY ? 0.f : m - x[u].x; s0 *= __expf(d); sT *= __expf(d * invT); m = x[u].x; }
      const float d = x[u].x - m;
      s0 += x[u].y * __expf(d); sT += x[u].z * __expf(d * invT);
    }
  }
  float gm = m;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) gm = fmaxf(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, off));
  if (m > -INFINITY) { s0 *= __expf(m - gm); sT *= __expf((m - gm) * invT); }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) { s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, off); sT += __shfl_xor_sync(0xFFFFFFFFu, sT, off); }
  const float lse0 = gm + logf(s0);
  return make_float2(lse0, T > 0.f ? gm * invT + logf(sT) : lse0);
}

// ---- seed bounds ------------------------------------------------------------------------------------------------------
// Best base logit (and its token) of one piece of one row, by one warp; a ragged vocabulary's rows are copied to
// their padded places on the way.
__device__ __forceinline__ void scout_piece(const TreeArgs& a, int row, int piece, int piece_len, uint2* out, int lane) {
  const int lo = piece * piece_len, hi = min(a.V, lo + piece_len);
  const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(a.U) + (size_t)row * a.V;
  float bv = -INFINITY; int bi = 0x7FFFFFFF;
  uint4 x[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int v = lo + (u * 32 + lane) * 8;
    x[u] = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);   // -inf
    if (v < hi) {
      if (!a.ragged) x[u] = __ldg(reinterpret_cast<const uint4*>(src + v));
      else {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t e0 = v + 2 * i < a.V ? __ldg(reinterpret_cast<const unsigned short*>(src) + v + 2 * i) : 0xFF80u;
          const uint32_t e1 = v + 2 * i + 1 < a.V ? __ldg(reinterpret_cast<const unsigned short*>(src) + v + 2 * i + 1) : 0xFF80u;
          w[i] = e0 | (e1 << 16);
        }
        x[u] = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(const_cast<__nv_bfloat16*>(reinterpret_cast<const __nv_bfloat16*>(a.Uscan)) + (size_t)row * a.Vs + v) = x[u];
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    float f[8];
    unpack_bf16x8(x[u], f);
#pragma unroll
    for (int i = 0; i < 8; ++i) if (f[i] > bv) { bv = f[i]; bi = lo + (u * 32 + lane) * 8 + i; }
  }
  const unsigned e = bi == 0x7FFFFFFF ? 0u : enc_f(bv);
  const unsigned mv = __reduce_max_sync(0xFFFFFFFFu, e);
  const unsigned mt = __reduce_min_sync(0xFFFFFFFFu, (e == mv && e != 0u) ? (unsigned)bi : 0x7FFFFFFFu);
  if (lane == 0) *out = make_uint2(mv, mt);   // (0: nothing above -inf in the piece)
}

// The seed tokens of one row, by one warp: a lane's best of the pieces it reads, ranked among the lanes' by counting (any
// tokens give valid bounds, so the second best of a lane is not missed; picking the best 16 of all pieces one after the
// other took 3.5 us and was what the owner's other warps waited for).
__device__ __forceinline__ void pick_seeds(const int npiece, const uint2* ut, int NS, int* stok, float* sval, int lane) {
  uint32_t bv = 0u, bt = 0u;
#pragma unroll 1
  for (int i0 = 0; i0 < npiece; i0 += 160) {
    uint2 e[5];
#pragma unroll
    for (int u = 0; u < 5; ++u) { const int i = i0 + u * 32 + lane; e[u] = i < npiece ? __ldcg(ut + i) : make_uint2(0u, 0u); }
#pragma unroll
    for (int u = 0; u < 5; ++u) if (e[u].x > bv) { bv = e[u].x; bt = e[u].y; }
  }
  int rank = 0;
#pragma unroll
  for (int l = 0; l < 32; ++l) { const uint32_t o = __shfl_sync(0xFFFFFFFFu, bv, l); rank += (o > bv || (o == bv && l < lane)) ? 1 : 0; }
  if (rank < NS) { stok[rank] = bv ? (int)bt : -1; sval[rank] = bv ? dec_f(bv) : -INFINITY; }
}

// Shared-memory pieces of an owner (offsets of OwnerLayout).
struct OwnerSm {
  PoolView pv; float *lse0, *lseT; int* pslot; int *ttok, *dtok; float *tlog, *dlog; double *ckey, *clogS;
  unsigned char *valid, *best; int *hist, *newl, *tcnt, *toff, *npl; uint32_t* Wc; int* stok; float* sval; float* res;
};
__device__ __forceinline__ OwnerSm owner_carve(unsigned char* sm, const TreeArgs& a) {
  const int N = a.N, NK = a.N << slot_log2(a.K);
  OwnerSm s;
  s.pv = pool_view(sm + a.own.pool, N);
  s.lse0 = reinterpret_cast<float*>(sm + a.own.lse); s.lseT = s.lse0 + N; s.pslot = reinterpret_cast<int*>(s.lseT + N);
  s.ttok = reinterpret_cast<int*>(sm + a.own.toks); s.dtok = s.ttok + NK; s.tlog = reinterpret_cast<float*>(s.dtok + NK); s.dlog = s.tlog + NK;
  s.ckey = reinterpret_cast<double*>(sm + a.own.cand); s.clogS = s.ckey + NK; s.res = reinterpret_cast<float*>(sm + a.own.cand);
  s.valid = sm + a.own.flags; s.best = s.valid + NK;
  s.hist = reinterpret_cast<int*>(sm + a.own.lists); s.newl = s.hist + 256; s.tcnt = s.newl + 256; s.toff = s.tcnt + 256; s.npl = s.toff + 256;
  s.Wc = reinterpret_cast<uint32_t*>(sm + a.own.seeds);
  s.stok = reinterpret_cast<int*>(s.Wc + (size_t)seed_count(a.K) * (a.r + 1)); s.sval = reinterpret_cast<float*>(s.stok + 32);
  return s;
}

// The seed tokens' columns of W (words of two tokens; rows of r + 1 words in shared memory: the threads that later read one
// k of different tokens hit different banks).  All threads; every word is a sector of its own, so a thread requests its
// words together, and keeps them in registers while other work goes on (cp.async of 4 bytes took 5 us for 1024 of them).
constexpr int SEED_REGS = 4;
__device__ __forceinline__ void load_seed_columns(const TreeArgs& a, const OwnerSm& s, int NS, int e0, uint32_t* w) {
  const uint32_t* Wg = reinterpret_cast<const uint32_t*>(a.Wscan);
#pragma unroll
  for (int u = 0; u < SEED_REGS; ++u) {
    const int e = e0 + u * TX_THREADS + (int)threadIdx.x;
    w[u] = 0u;
    if (e < NS * a.r) {
      const int j = e & (NS - 1), k = e >> seed_log2(a.K), tok = s.stok[j];
      if (tok >= 0) w[u] = __ldcg(Wg + (((size_t)k * a.Vs + tok) >> 1));   // (a ragged vocabulary's padded W is written by this launch: not the read-only path)
    }
  }
}
__device__ __forceinline__ void store_seed_columns(const TreeArgs& a, const OwnerSm& s, int NS, int e0, const uint32_t* w) {
#pragma unroll
  for (int u = 0; u < SEED_REGS; ++u) {
    const int e = e0 + u * TX_THREADS + (int)threadIdx.x;
    if (e < NS * a.r) s.Wc[(e & (NS - 1)) * (a.r + 1) + (e >> seed_log2(a.K))] = w[u];
  }
}

// Seed bounds and list entries of `cnt` parents of one row (all threads; the columns have landed).  Parent i: token
// ptok[i], hash phash[i], pool slot s.npl[i]; its place in the level's list is li0 + i * step (place != null: *place, known after the first barrier).
__device__ __forceinline__ void make_parents(const TreeArgs& a, const OwnerSm& s, const int cnt, int li0, const int* place, const int step, const int req, const int row, const int NS,
                                             const int* ptok, const uint64_t* phash, ParentEntry* ent, int* ent_slot, int* cnt_next) {
  const int tid = threadIdx.x, r = a.r, K = a.K, lg = seed_log2(K);
  const float invT = a.T > 0.f ? 1.f / a.T : 1.f;
  const __nv_bfloat16* Ag = reinterpret_cast<const __nv_bfloat16*>(a.A);
  // every (parent, seed token) pair exactly: eight lanes a pair, 16 bytes of the head row a lane and step
  const int sub = tid & 7;
#pragma unroll 1
  for (int e0 = 0; e0 < cnt * NS; e0 += TX_THREADS / 8) {
    const int e = e0 + (tid >> 3);
    const bool have = e < cnt * NS;
    const int i = have ? e >> lg : 0, j = e & (NS - 1), tok = s.stok[j];
    float dot = 0.f;
    if (have && tok >= 0) {
      const uint32_t* wc = s.Wc + (size_t)j * (r + 1);
      const int hi = tok & 1;
#pragma unroll 1
      for (int k = sub * 8; k < r; k += 64) {
        float av[8];
        unpack_bf16x8(__ldg(reinterpret_cast<const uint4*>(Ag + (size_t)ptok[i] * r + k)), av);
#pragma unroll
        for (int u = 0; u < 8; ++u) { const uint32_t w = wc[k + u]; dot = fmaf(av[u], __uint_as_float(hi ? (w & 0xFFFF0000u) : (w << 16)), dot); }
      }
    }
    dot += __shfl_xor_sync(0xFFFFFFFFu, dot, 1); dot += __shfl_xor_sync(0xFFFFFFFFu, dot, 2); dot += __shfl_xor_sync(0xFFFFFFFFu, dot, 4);
    if (have && sub == 0) {
      float lo = -INFINITY, key = -INFINITY;
      if (tok >= 0) {
        lo = s.sval[j] + dot;
        key = a.T > 0.f ? exact_key(a.seed, req, phash[i], tok, lo, invT) : lo;
      }
      s.res[2 * e] = lo; s.res[2 * e + 1] = key;
    }
  }
  float* bL = reinterpret_cast<float*>(s.tcnt); float* bK = reinterpret_cast<float*>(s.toff); float* bM = reinterpret_cast<float*>(s.hist);
#pragma unroll 1
  for (int i = tid; i < cnt; i += TX_THREADS) { bL[i] = -INFINITY; bK[i] = -INFINITY; bM[i] = -INFINITY; }
  __syncthreads();
  if (place) li0 = *place;
  // the parents' pruning state and candidate counts start clean
#pragma unroll 1
  for (int e = tid; e < cnt * 2 * K; e += TX_THREADS) {
    const int i = e / (2 * K), w = (e / K) & 1, j = e % K;
    a.slots[(((size_t)w * a.cap + li0 + i * step) * K + j) * SLOT_STRIDE] = 0u;
  }
#pragma unroll 1
  for (int e = tid; e < cnt * 2; e += TX_THREADS) {
    a.thr[(size_t)(e & 1) * a.cap + li0 + (e >> 1) * step] = 0u;
    cnt_next[(size_t)(e & 1) * a.cap + li0 + (e >> 1) * step] = 0;
  }
#pragma unroll 1
  for (int e = tid; e < 2 * cnt * NS; e += TX_THREADS) {
    // one thread per value: the one with exactly K - 1 values before it (ties broken by place) is the K-th best
    const int j = e & (NS - 1), which = (e >> lg) & 1, i = e >> (lg + 1);
    const float* val = s.res + (size_t)i * NS * 2 + which;
    const float mine = val[2 * j];
    int before = 0;
#pragma unroll 1
    for (int t = 0; t < NS; ++t) before += (val[2 * t] > mine || (val[2 * t] == mine && t < j)) ? 1 : 0;
    const bool fin = mine == mine && fabsf(mine) < INFINITY;
    if (before == K - 1 && fin && !a.no_seed) {
      // rounding of an r-term fp32 sum in another order, of the division by T and of the fast logarithms
      const float margin = (2e-4f + 4e-5f * fabsf(mine)) * (which == 0 ? 1.f : fmaxf(invT, 1.f)) + (which == 0 ? 0.f : 2e-4f);
      (which ? bK : bL)[i] = mine - margin;
    }
    if (before == 0 && which == 0 && fin) bM[i] = mine;
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < cnt; i += TX_THREADS) {
    ParentEntry pe;
    pe.row = row; pe.token = ptok[i]; pe.hash = phash[i]; pe.thrL = bL[i]; pe.thrK = a.T > 0.f ? bK[i] : -INFINITY; pe.mref = bM[i]; pe.req = req;
    const uint4* src = reinterpret_cast<const uint4*>(&pe);
    uint4* dst = reinterpret_cast<uint4*>(ent + li0 + i * step);
    dst[0] = src[0]; dst[1] = src[1];
    if (ent_slot) ent_slot[li0 + i * step] = s.npl[i];
  }
}

// The calibrated estimate as one copy of code, so that one warp can bring it into the instruction caches while the others sweep: met
// for the first time in the first owner phase it took 5 us instead of 1.6.
__device__ __noinline__ double tx_estimate(const DevCalib& c, int d, double lx, double lse0) { return log_phat(c, d, lx, lse0); }

// One level of one request: merge of its parents, slots and cut of Algorithm 1, the next level's parents.
// d = depth of the parents just scanned; d = -1: the start of request b (an empty pool and the root as the only parent of
// level 0) or, for ts_score_parents, the list entry of given parent b.
// (Inlined, once: behind a call the arguments would be read through generic addresses, some 40 cycles each.)
// share >= 0: not the level step, but the seed bounds of every `step`-th of the new parents of request b, from the share-th
// on (a request with many leaves them to the CTAs that own none); spread: the merge was done by all CTAs.
template <bool MANY>
__device__ __forceinline__ void tx_owner(const TreeArgs& a, unsigned char* sm, const int b, const int d, const int share_, const int step, const bool spread_, const int P) {
  const int share = MANY ? share_ : -1;
  const bool spread = MANY && spread_;
  const OwnerSm s = owner_carve(sm, a);
  __shared__ int sh[8];
  __shared__ int own[3];   // of request blockIdx.x: parents of its current level, their base in the list, status fine (kept here: a memory round trip less)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = a.N, K = a.K, lk = slot_log2(K), cur = d & 1, nxt = cur ^ 1, NS = seed_count(K);
  int* ptok = s.ttok; uint64_t* phash = reinterpret_cast<uint64_t*>(s.tlog);   // the new parents (merged results are done with by then)
  int cnt = 1, li0 = b, req = b, row = b * a.D + d + 1;
  bool more = true;
  int npar = 0, base = 0, K_eff = 0, N_eff = 0, pslot = -1;
  double2 caps = make_double2(0.0, 0.0);
  int place = 0;
  unsigned char* gpool = a.pool + (size_t)b * a.pool_stride;
  if (share >= 0) {
    const int np = __ldcg(a.req_npar + nxt * a.B + b);
    cnt = np > TX_SOLO ? (np - share + step - 1) / step : 0;
    if (cnt <= 0) return;   // uniform
    li0 = __ldcg(a.req_base + b) + share;
#pragma unroll 1
    for (int i = tid; i < cnt; i += TX_THREADS) {
      const uint4 e = __ldcg(reinterpret_cast<const uint4*>(a.ent[nxt] + li0 + i * step));
      ptok[i] = (int)e.y; phash[i] = ((uint64_t)e.w << 32) | e.z;
    }
  } else if (d < 0) {
    const bool given = a.score_P > 0;
    if (given) { req = a.p_req[b]; row = req * a.D + a.p_depth[b]; }
    else {
      PoolView g = pool_view(gpool, N);
#pragma unroll 1
      for (int i = tid; i < N; i += TX_THREADS) g.meta[i] = 0;
    }
    if (tid == 0) {
      if (given) { ptok[0] = a.p_token[b]; phash[0] = a.p_hash[b]; }
      else {
        const int t = a.anchor[b];
        const bool ok = t >= 0 && t < a.V && a.theta[b] == a.theta[b];
        a.status[b] = ok ? TS_OK : TS_ERR_INVALID;
        ptok[0] = ok ? t : 0; phash[0] = 0ull;
        a.req_npar[b] = 1; a.req_base[b] = b; a.req_nscored[b] = 0;
        if (b == (int)blockIdx.x) { own[0] = 1; own[1] = b; own[2] = ok ? 1 : 0; }
        a.root_lseT[b] = nanf("");
        const float th = a.theta[b];   // (>= 1: the chain member of the price ladder)
        a.req_caps[b] = make_double2(th >= 1.f || !(th > 0.f) ? -INFINITY : log((double)th), th >= 1.f ? 1.0 : 0.0);
      }
      s.npl[0] = -1;
    }
  } else {
    bool fine;
    if (b == (int)blockIdx.x) { npar = own[0]; base = own[1]; fine = own[2] != 0; }
    else { npar = __ldcg(a.req_npar + cur * a.B + b); base = __ldcg(a.req_base + b); fine = __ldcg(a.status + b) == TS_OK; }
    if (npar == 0 || !fine) {   // uniform: nothing below has run yet
      if (tid == 0) a.req_npar[nxt * a.B + b] = 0;
      return;   // (own[] stays: no parents, or not fine)
    }
    caps = __ldcg(a.req_caps + b);   // log theta (-inf on the chain member), 1 on the chain member (not looked at before the merge)
    more = d + 1 < a.D;
    uint4* dst = reinterpret_cast<uint4*>(s.pv.key); const uint4* src = reinterpret_cast<const uint4*>(gpool);
#pragma unroll 1
    for (int i = tid; i < (int)(pool_bytes(N) / 16); i += TX_THREADS) cp_async16(dst + i, src + i, true);   // (lands while the merge runs)
    if (tid < npar) pslot = __ldcg(a.ent_slot[cur] + base + tid);   // (at most 256 parents)
    if (tid < 8) sh[tid] = 0;
  }
  // ---- merge: a warp each for a parent's log-normalisers, its best logits and its best keys: each is one or two memory
  // round trips, side by side (the last warp picks the next row's seed tokens meanwhile) ----
  if (warp == TX_WARPS - 1) {
    if (more) pick_seeds(a.npiece, a.utop + ((size_t)nxt * a.B + b) * a.npiece, NS, s.stok, s.sval, lane);
  } else if (spread && share < 0) {
#pragma unroll 1
    for (int t = tid; t < npar << lk; t += TX_THREADS - 32) {
      const int i = t >> lk, j = t & ((1 << lk) - 1);
      const size_t at = (size_t)(base + i) * KMAX + j;
      if (j < K) {
        const uint4 e = __ldcg(a.res_cand + at);
        s.ttok[t] = (int)e.x; s.tlog[t] = __uint_as_float(e.y); s.dtok[t] = (int)e.z; s.dlog[t] = __uint_as_float(e.w);
      }
      if (j == 0) { const float2 l = __ldcg(a.res_lse + base + i); s.lse0[i] = l.x; s.lseT[i] = l.y; }
    }
  } else if (d >= 0 && share < 0) {
#pragma unroll 1
    for (int task = warp; task < npar * 3; task += TX_WARPS - 1) {
      const int i = task / 3, kind = task - 3 * i, p = base + i;
      if (kind == 2 && !(a.T > 0.f)) continue;
      if (kind == 0) {
        const float2 l = warp_lse(a.sums + (size_t)p * a.ntiles, a.ntiles, a.T, lane);
        if (lane == 0) { s.lse0[i] = l.x; s.lseT[i] = l.y; }
      } else {
        const size_t cb = cand_base(a, P, p);
        const float3 w = warp_topk(kind == 1 ? a.cand_top + cb : a.cand_key + cb, kind == 1 ? nullptr : a.cand_lg + cb, a.cand_cnt[cur] + (kind == 1 ? 0 : a.cap) + p, K, lane);
        if (lane < K) {
          if (kind == 1) { s.ttok[(i << lk) + lane] = __float_as_int(w.x); s.tlog[(i << lk) + lane] = w.y; }
          if (kind == 2 || !(a.T > 0.f)) { s.dtok[(i << lk) + lane] = __float_as_int(w.x); s.dlog[(i << lk) + lane] = w.z; }
        }
      }
    }
  }
  if (tid < npar) s.pslot[tid] = pslot;
  cp_async_wait_all();
  __syncthreads();
  const double log_theta = caps.x;
  K_eff = caps.y != 0.0 ? 1 : min(K, a.V); N_eff = caps.y != 0.0 ? min(a.D, N) : N;
  uint32_t wcol[SEED_REGS];
  if (more) load_seed_columns(a, s, NS, 0, wcol);   // on their way while the draws are ranked
  if (d >= 0 && share < 0) {
  // the best token of q0 not among the first j draws, for every j: places of the draws in the top list, or-ed up
#pragma unroll 1
  for (int i = warp; i < npar; i += TX_WARPS) {
    unsigned used = 0u;
    if (!(a.T > 0.f)) used = lane < K ? 1u << lane : 0u;
    else if (lane < K) {
      const int x = s.dtok[(i << lk) + lane];
#pragma unroll 4
      for (int t = 0; t < K; ++t) if (x >= 0 && s.ttok[(i << lk) + t] == x) used |= 1u << t;
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) { const unsigned u = __shfl_up_sync(0xFFFFFFFFu, used, o); if (lane >= o) used |= u; }
    const unsigned prior = __shfl_up_sync(0xFFFFFFFFu, used, 1);
    if (lane < K) { const unsigned fr = ~(lane ? prior : 0u) & ((1u << K_eff) - 1u); s.best[(i << lk) + lane] = fr ? (unsigned char)(__ffs(fr) - 1) : 255u; }
  }
  __syncthreads();
  if (more) store_seed_columns(a, s, NS, 0, wcol);
  // ---- slots of every scored parent: two threads per (parent, sibling rank), one for the key (the best unused token's
  // estimate), one for the survival of the token drawn ----
#pragma unroll 1
  for (int t2 = tid; t2 < 2 * npar << lk; t2 += TX_THREADS) {
    const int t = t2 >> 1, which = t2 & 1, i = t >> lk, j = t & ((1 << lk) - 1);
    const double lse0 = s.lse0[i], lseT = s.lseT[i];
    const int slot = s.pslot[i];
    const bool bad = !(lse0 == lse0) || isinf(lse0);
    if (j == 0 && which == 0) {
      if (slot < 0) a.root_lseT[b] = (float)lseT; else s.pv.lseT[slot] = (float)lseT;
      if (bad) { a.status[b] = TS_ERR_NUMERIC; if (b == (int)blockIdx.x) own[2] = 0; }
    }
    int ok = 0;
    if (j < K_eff && !bad) {
      const int bi = s.best[t], x = s.dtok[t];
      if (bi < K_eff && s.ttok[(i << lk) + bi] >= 0 && x >= 0) {
        const double logS_v = slot < 0 ? 0.0 : s.pv.logS[slot];
        // the calibrator's input: the untempered conditional, or (ablation) the tempered one
        const bool tempered = a.calib_qT && a.T > 0.f;
        const double lsc = tempered ? 1.0 / (double)a.T : 1.0, lsn = tempered ? lseT : lse0;
        const double v = logS_v + tx_estimate(a.calib, d, (double)(which ? s.dlog[t] : s.tlog[(i << lk) + bi]) * lsc, lsn);
        if (which) s.clogS[t] = v;
        else { s.ckey[t] = v; ok = !(v < log_theta); }
      }
    }
    if (which == 0) s.valid[t] = (unsigned char)ok;
  }
  __syncthreads();
  // a sibling slot exists only if the one before it was admitted (keys are non-increasing in j)
  {
    int nv = 0, np = 0;
#pragma unroll 1
    for (int i = tid; i < npar; i += TX_THREADS) {
      bool open = true;
#pragma unroll 1
      for (int j = 0; j < K; ++j) { if (!s.valid[(i << lk) + j]) open = false; if (open) ++nv; else s.valid[(i << lk) + j] = 0; }
    }
#pragma unroll 1
    for (int i = tid; i < N; i += TX_THREADS) np += s.pv.meta[i] >> 16;
    nv = __reduce_add_sync(0xFFFFFFFFu, nv); np = __reduce_add_sync(0xFFFFFFFFu, np);
    if (lane == 0) { if (np) atomicAdd(&sh[0], np); if (nv) atomicAdd(&sh[1], nv); }
  }
  __syncthreads();
  const int ncand = npar << lk, shift = 60 - 4 * d;
  auto skey = [](double k) -> uint64_t {
    if (k == 0.0) k = 0.0;   // -0 and +0 compare equal: one pattern
    const uint64_t u = (uint64_t)__double_as_longlong(k);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
  };
  // entry e: a pool slot (e < N) or a candidate
  const int M = N + ncand;
  auto live = [&](int e) -> bool { return e < N ? (s.pv.meta[e] >> 16) != 0 : s.valid[e - N] != 0; };
  auto key_of = [&](int e) -> double { return e < N ? s.pv.key[e] : s.ckey[e - N]; };
  auto depth_of = [&](int e) -> int { return e < N ? (s.pv.meta[e] >> 8) & 255 : d + 1; };
  auto path_of = [&](int e) -> uint64_t {
    if (e < N) return s.pv.path[e];
    const int c = e - N, slot = s.pslot[c >> lk];
    return (slot < 0 ? 0ull : s.pv.path[slot]) | ((uint64_t)(c & ((1 << lk) - 1)) << shift);
  };
  if (sh[0] + sh[1] > N_eff) {
    // The N_eff-th largest key by radix selection over the keys' order-preserving bit patterns (eight bits a pass);
    // entries above it stay, entries below it go, and those that tie with it are ranked among themselves by
    // (depth, path) for the places that are left.
    uint64_t prefix = 0;
    int need = N_eff;
#pragma unroll 1
    for (int sh8 = 56; sh8 >= 0; sh8 -= 8) {
      if (tid < 256) s.hist[tid] = 0;
      __syncthreads();
#pragma unroll 1
      for (int e = tid; e < M; e += TX_THREADS) {
        if (!live(e)) continue;
        const uint64_t k = skey(key_of(e));
        if (sh8 == 56 || (k >> (sh8 + 8)) == (prefix >> (sh8 + 8))) {
          const int bin = (int)((k >> sh8) & 255u);
          if (MANY) {   // one addition per bin and warp: the first pass, over sign and exponent, has two or three bins for 1,700 keys
            const unsigned peers = __match_any_sync(__activemask(), bin);
            if (lane == __ffs(peers) - 1) atomicAdd(&s.hist[bin], __popc(peers));
          } else atomicAdd(&s.hist[bin], 1);
        }
      }
      __syncthreads();
      if (warp == 0) {
        // lane l owns bins 255 - 8l .. 248 - 8l (descending); the bin where the running count reaches `need`
        int mine = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) mine += s.hist[255 - 8 * lane - j];
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (lane >= o) incl += v; }
        const unsigned reach = __ballot_sync(0xFFFFFFFFu, incl >= need);
        if (lane == __ffs(reach) - 1) {   // reach != 0: at least `need` entries match the prefix
          int cum = incl - mine, bin = 255 - 8 * lane;
          for (int j = 0; j < 8; ++j) {
            const int h = s.hist[255 - 8 * lane - j];
            if (cum + h >= need) { bin = 255 - 8 * lane - j; break; }
            cum += h;
          }
          sh[2] = bin; sh[3] = need - cum; sh[7] = s.hist[bin] == need - cum ? 1 : 0;
        }
      }
      __syncthreads();
      prefix |= (uint64_t)sh[2] << sh8;
      need = sh[3];
      if (sh[7]) break;   // the whole bin stays: its lower end is the threshold, nothing ties with it from below
    }
    const bool whole = sh[7] != 0;   // (thousands of distinct keys: after three or four passes)
    if (tid == 0) sh[4] = 0;
    __syncthreads();
    if (!whole)
#pragma unroll 1
    for (int e = tid; e < M; e += TX_THREADS)
      if (live(e) && skey(key_of(e)) == prefix) { const int at = atomicAdd(&sh[4], 1); if (at < 256) s.newl[at] = e; }
    __syncthreads();
    const int ntie = whole ? 0 : sh[4];
    unsigned drop = 0u;   // bit per trip: M <= 17 * 256 entries, at most 8 trips
#pragma unroll 1
    for (int e = tid, it = 0; e < M; e += TX_THREADS, ++it) {
      if (!live(e)) continue;
      const double ke = key_of(e);
      const uint64_t k = skey(ke);
      bool out = k < prefix;
      if (k == prefix && ntie > need) {
        int rank = 0;
        const int de = depth_of(e); const uint64_t pe = path_of(e);
        const int nn = ntie <= 256 ? ntie : M;
#pragma unroll 1
        for (int t = 0; t < nn; ++t) {
          const int f = ntie <= 256 ? s.newl[t] : t;
          if (f == e || (ntie > 256 && !(live(f) && skey(key_of(f)) == prefix))) continue;
          if (before(key_of(f), depth_of(f), path_of(f), ke, de, pe)) ++rank;
        }
        out = rank >= need;
      }
      drop |= (out ? 1u : 0u) << it;
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid, it = 0; e < M; e += TX_THREADS, ++it)
      if ((drop >> it) & 1u) { if (e < N) s.pv.meta[e] &= 0xFFFF; else s.valid[e - N] = 0; }
    __syncthreads();
  }
  // ---- placement: the t-th surviving candidate (in candidate order) takes the t-th free slot (in slot order) ----
  {
    const bool fr = tid < N && (s.pv.meta[tid] >> 16) == 0;
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, fr);
    if (lane == 0 && warp < 8) s.npl[warp] = __popc(bal);
    const int ntrip = (ncand + TX_THREADS - 1) / TX_THREADS;   // <= 7
    unsigned vm = 0;
#pragma unroll 1
    for (int it = 0; it < ntrip; ++it) {
      const int c = it * TX_THREADS + tid;
      const bool v = c < ncand && s.valid[c];
      const unsigned vb = __ballot_sync(0xFFFFFFFFu, v);
      vm |= (v ? 1u : 0u) << it;
      if (lane == 0) s.tcnt[it * TX_WARPS + warp] = __popc(vb);
    }
    __syncthreads();
    int off = 0, nfree = 0;
#pragma unroll 1
    for (int w = 0; w < 8; ++w) { if (w < warp) off += s.npl[w]; nfree += s.npl[w]; }
    if (fr) s.hist[off + __popc(bal & ((1u << lane) - 1u))] = tid;
    const int ne = ntrip * TX_WARPS;
    if (warp == 0) {   // exclusive prefix over (trip, warp)
      int run = 0;
#pragma unroll 1
      for (int e0 = 0; e0 < ne; e0 += 32) {
        const int e = e0 + lane, c = e < ne ? s.tcnt[e] : 0;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (lane >= o) incl += v; }
        if (e < ne) s.toff[e] = run + incl - c;
        run += __shfl_sync(0xFFFFFFFFu, incl, 31);
      }
      if (lane == 0) sh[5] = min(run, nfree);
      if (lane == 0 && run > nfree) { a.status[b] = TS_ERR_OVERFLOW; if (b == (int)blockIdx.x) own[2] = 0; }
    }
    __syncthreads();
#pragma unroll 1
    for (int it = 0; it < ntrip; ++it) {
      const bool v = (vm >> it) & 1u;
      const unsigned vb = __ballot_sync(0xFFFFFFFFu, v);
      if (!v) continue;
      const int c = it * TX_THREADS + tid, t = s.toff[it * TX_WARPS + warp] + __popc(vb & ((1u << lane) - 1u));
      if (t >= nfree) continue;
      const int sl = s.hist[t], i = c >> lk, j = c & ((1 << lk) - 1), slot = s.pslot[i], x = s.dtok[c];
      if (more) asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const __nv_bfloat16*>(a.A) + (size_t)x * a.r));   // (its head row is needed soon)
      const double lx = s.dlog[c], lse0 = s.lse0[i], lseT = s.lseT[i];
      s.pv.meta[sl] = (1 << 16) | ((d + 1) << 8) | j; s.pv.parent[sl] = slot; s.pv.tok[sl] = x;
      s.pv.key[sl] = s.ckey[c]; s.pv.logS[sl] = s.clogS[c];
      s.pv.q0[sl] = (float)exp(lx - lse0);
      s.pv.logqT[sl] = a.T > 0.f ? (float)(lx / (double)a.T - lseT) : (float)(lx - lse0);
      s.pv.lseT[sl] = nanf("");
      s.pv.hash[sl] = path_hash(slot < 0 ? 0ull : s.pv.hash[slot], x);
      s.pv.path[sl] = (slot < 0 ? 0ull : s.pv.path[slot]) | ((uint64_t)j << shift);
      s.newl[t] = sl;
    }
  }
  __syncthreads();
  const int nnew = sh[5];
  // ---- next level's parents: new nodes that can still have admissible children ----
  {
    const bool par = more && tid < nnew && !(s.pv.logS[s.newl[tid]] < log_theta);
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, par);
    if (lane == 0 && warp < 8) s.tcnt[warp] = __popc(bal);
    uint64_t ph = 0; int pt = 0, sl = 0;
    if (par) { sl = s.newl[tid]; ph = s.pv.hash[sl]; pt = s.pv.tok[sl]; }
    __syncthreads();
    int off = 0;
    cnt = 0;
#pragma unroll 1
    for (int w = 0; w < 8; ++w) { if (w < warp) off += s.tcnt[w]; cnt += s.tcnt[w]; }
    if (tid == 0) {
      if (cnt > 0) place = atomicAdd(a.lvl_count + d + 1, cnt);   // (asked for here, waited for after the seed products)
      if (b == (int)blockIdx.x) own[0] = cnt;
      a.req_npar[nxt * a.B + b] = cnt; a.req_nscored[b] += npar;
    }
    if (par) { const int i = off + __popc(bal & ((1u << lane) - 1u)); s.npl[i] = sl; ptok[i] = pt; phash[i] = ph; }
  }
  uint4* gdst = reinterpret_cast<uint4*>(gpool); const uint4* psrc = reinterpret_cast<const uint4*>(s.pv.key);
#pragma unroll 1
  for (int i = tid; i < (int)(pool_bytes(N) / 16); i += TX_THREADS) gdst[i] = psrc[i];
  }
  // ---- seed bounds and list entries ----
  if (more && (d < 0 || share >= 0)) store_seed_columns(a, s, NS, 0, wcol);
  if (more)
#pragma unroll 1
    for (int e0 = SEED_REGS * TX_THREADS; e0 < NS * a.r; e0 += SEED_REGS * TX_THREADS) { load_seed_columns(a, s, NS, e0, wcol); store_seed_columns(a, s, NS, e0, wcol); }
  __syncthreads();
  const bool placed = d >= 0 && share < 0;
  if (placed && tid == 0) { sh[6] = place; a.req_base[b] = place; if (b == (int)blockIdx.x) own[1] = place; }   // (visible after the barrier in make_parents, or the one here)
  if (MANY && more && share < 0 && cnt > TX_SOLO) {   // many parents: entries without bounds; all CTAs make those after the next barrier
    __syncthreads();
    if (placed) li0 = sh[6];
#pragma unroll 1
    for (int i = tid; i < cnt; i += TX_THREADS) {
      uint4* dst = reinterpret_cast<uint4*>(a.ent[nxt] + li0 + i);
      dst[0] = make_uint4((unsigned)row, (unsigned)ptok[i], (unsigned)phash[i], (unsigned)(phash[i] >> 32));
      dst[1] = make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, (unsigned)req);
      a.ent_slot[nxt][li0 + i] = s.npl[i];
    }
    if (tid == 0) a.seed_need[d + 1] = 1;
  } else if (more && cnt > 0) make_parents(a, s, cnt, li0, placed ? sh + 6 : nullptr, share >= 0 ? step : 1, req, row, NS, ptok, phash, a.ent[nxt], share >= 0 ? nullptr : a.ent_slot[nxt], a.cand_cnt[nxt]);
  __syncthreads();
}

// Canonical (BFS) renumbering, outputs and ancestor bitmasks of one request, out of shared memory.
// (MANY: rounds of the counting loop together, 18 us at 256 nodes without; in the forms for small trees it cost the chain of 128 requests 2 %.)
template <bool MANY>
__device__ __forceinline__ void tx_finalize(const TreeArgs& a, unsigned char* sm, const int b, const bool timed_out) {
  constexpr int UNROLL = MANY ? 4 : 1;
  const OwnerSm s = owner_carve(sm, a);
  const int tid = threadIdx.x, N = a.N;
  const size_t pb = (size_t)b * N;
  int* canon = s.ttok; int* cpar = s.dtok;
  __shared__ int n_sh;
  {
    uint4* dst = reinterpret_cast<uint4*>(s.pv.key); const uint4* src = reinterpret_cast<const uint4*>(a.pool + (size_t)b * a.pool_stride);
#pragma unroll 1
    for (int i = tid; i < (int)(pool_bytes(N) / 16); i += TX_THREADS) dst[i] = __ldcg(src + i);
  }
  if (tid == 0) n_sh = 0;
  __syncthreads();
  // a node's places by counting; G neighbouring lanes share a node's comparisons
  const int G = N <= 80 ? 8 : (N <= 160 ? 4 : 2);
#pragma unroll 1
  for (int q0 = 0; q0 < N; q0 += TX_THREADS / G) {
    const int x = q0 + tid / G, sub = tid % G;
    const bool have = x < N && (s.pv.meta[x] >> 16) != 0;
    int cr = 0, pr = 0;
    if (have) {
      const int dx = (s.pv.meta[x] >> 8) & 255; const uint64_t px = s.pv.path[x]; const double kx = s.pv.key[x];
#pragma unroll UNROLL
      for (int t = sub; t < N; t += G) {
        const int mt = s.pv.meta[t], dt = (mt >> 8) & 255;   // (no branches: the loads of several rounds go out together)
        const uint64_t pt = s.pv.path[t]; const double kt = s.pv.key[t];
        const bool other = t != x && (mt >> 16) != 0, first = dt < dx || (dt == dx && pt < px);
        cr += other && first ? 1 : 0;
        pr += other && (kt > kx || (kt == kx && first)) ? 1 : 0;
      }
    }
    for (int o = 1; o < G; o <<= 1) { cr += __shfl_xor_sync(0xFFFFFFFFu, cr, o); pr += __shfl_xor_sync(0xFFFFFFFFu, pr, o); }
    if (x < N && sub == 0) canon[x] = have ? cr : -1;
    if (have && sub == 0) {
      atomicAdd(&n_sh, 1);
      const size_t o = pb + cr;
      a.tok[o] = s.pv.tok[x]; a.depth[o] = (s.pv.meta[x] >> 8) & 255; a.sib_rank[o] = s.pv.meta[x] & 255;
      a.logS[o] = (float)s.pv.logS[x]; a.q0[o] = s.pv.q0[x]; a.logqT[o] = s.pv.logqT[x];
      if (a.logkey) a.logkey[o] = (float)s.pv.key[x];
      if (a.pop_rank) a.pop_rank[o] = pr;
      a.node_hash[(size_t)b * (N + 1) + cr + 1] = s.pv.hash[x];
      if (a.node_lseT) a.node_lseT[(size_t)b * (N + 1) + cr + 1] = s.pv.lseT[x];
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int x = tid; x < N; x += TX_THREADS) {
    const int c = canon[x];
    if (c < 0) continue;
    const int px = s.pv.parent[x], cp = px < 0 ? -1 : canon[px];
    cpar[c] = cp;
    a.parent[pb + c] = cp;
  }
  if (tid == 0) {
    if (timed_out && a.status[b] == TS_OK) a.status[b] = TS_ERR_TIMEOUT;
    a.n_nodes[b] = n_sh;
    a.node_hash[(size_t)b * (N + 1)] = 0ull;
    if (a.node_lseT) a.node_lseT[(size_t)b * (N + 1)] = a.root_lseT[b];
    if (a.n_scored) a.n_scored[b] = a.req_nscored[b];
  }
  __syncthreads();
  // a node's mask row: its own bit and its ancestors', up the (short) chain of parents
  const int n = n_sh;
#pragma unroll 1
  for (int e = tid; e < n * a.words; e += TX_THREADS) {
    const int i = e / a.words, w = e % a.words;
    uint64_t m = 0ull;
#pragma unroll 1
    for (int x = i; x >= 0; x = cpar[x]) if ((x >> 6) == w) m |= 1ull << (x & 63);
    a.mask[pb * a.words + e] = m;
  }
  __syncthreads();
}

// MANY: owners share the work on crowded levels with the CTAs that own no request (a second instantiation: the code costs
// the scan of the other one's launches 4 %).
template <bool MANY, bool RING>
__global__ void __launch_bounds__(TX_THREADS, 1) tree_kernel(const __grid_constant__ TreeArgs a, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmU) {
  extern __shared__ unsigned char raw[];
  unsigned char* base_sm = raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u);
  const TxSm sm = tx_carve(base_sm, a);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = (int)blockIdx.x, ncta = (int)gridDim.x;
  const int t0 = cta * a.TV, tlen = min(a.TV, a.V - t0);     // this CTA's vocabulary range (empty for the last CTAs of some vocabularies)
  // ---- set-up: nothing here reads what an earlier kernel wrote -----------------------------------------------------
  if (warp == TX_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(sm.tmem)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(sm.a_full, TX_SCAN_WARPS * 32 + (a.lost_arrival ? 1 : 0));
    for (int i = 0; i < TX_STAGE_MAX; ++i) {
      mbar_init(sm.t_full + i, 1); mbar_init(sm.t_empty + i, TX_SCAN_WARPS);
      mbar_init(sm.w_full + i, a.use_tma ? 1 : 32); mbar_init(sm.w_free + i, 1);
    }
    for (int i = 0; i < TX_USTAGES; ++i) { mbar_init(sm.u_full + i, 1); mbar_init(sm.u_free + i, TX_SCAN_WARPS); }
    *sm.abort = 0; *sm.done = 0; *sm.q_head = 0u; *sm.q_tail = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fill_gumbel_bounds(sm.ghi, tid, TX_THREADS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *sm.tmem;
  pdl_wait();                 // inputs, workspace and the words the kernel before cleared
  pdl_launch_dependents();

  unsigned gen = 0;
  const unsigned nexpect = (unsigned)ncta + (a.lost_arrival ? 1u : 0u);
  bool dead = false;
  WLoad wl{{0, 0u, 0u}, 0, 0u};
  ULoad ul{0u};
  uint32_t ub0 = 0u;          // blocks that went through the base-logit ring
  BlockPos pos{0, 0u, 0u}, wpos{0, 0u, 0u};
  int groups = 0;
  const int nreq = a.score_P > 0 ? a.score_P : a.B;

  if (a.ragged) {   // W with padded rows (the bulk-tensor loads need rows of whole 16 bytes)
    const unsigned short* src = reinterpret_cast<const unsigned short*>(a.W);
    const int cpr = a.Vs / 8;
    for (int e = cta * TX_THREADS + tid; e < a.r * cpr; e += ncta * TX_THREADS) {
      const int k = e / cpr, v = (e % cpr) * 8;
      uint32_t w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t e0 = v + 2 * i < a.V ? __ldg(src + (size_t)k * a.V + v + 2 * i) : 0u, e1 = v + 2 * i + 1 < a.V ? __ldg(src + (size_t)k * a.V + v + 2 * i + 1) : 0u;
        w[i] = e0 | (e1 << 16);
      }
      *reinterpret_cast<uint4*>(const_cast<unsigned short*>(reinterpret_cast<const unsigned short*>(a.Wscan)) + (size_t)k * a.Vs + v) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    asm volatile("fence.proxy.async;" ::: "memory");   // the bulk-tensor loads of W read these through the other proxy
  }
  // Phases: d = -2 sweeps the depth-0 rows (given parents: theirs); d = -1 starts the requests; d >= 0 scans the parents of
  // depth d and runs their level step.
  int d = -2;
  if (tid == 0 && a.score_P == 0)   // the anchors' head rows: on their way while the first rows are swept
    for (int b = cta; b < a.B; b += ncta) {
      const int t = a.anchor[b];
      if (t >= 0 && t < a.V) asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const __nv_bfloat16*>(a.A) + (size_t)t * a.r));
    }
  if (warp == TX_REFRESH && a.score_P == 0 && cta < a.B) { const double x = tx_estimate(a.calib, 0, -1.0, 0.5); asm volatile("" ::"d"(x)); }   // (for the instruction caches)
  for (;; ++d) {
    int P = nreq;
    if (d >= 0) {
    if (d > 0) P = __ldcg(a.lvl_count + d);
    if (P <= 0) break;
    // ---- scan ---------------------------------------------------------------------------------------------------------
    if (tlen > 0) {
      const int ngroups = (P + TX_ROWS - 1) / TX_ROWS;
      for (int g = 0; g < ngroups; ++g, ++groups) {
        const int R = group_replicas(a, P, g), per = TX_ROWS / R;
        if (tid < TX_ROWS) {
          const int p = g * TX_ROWS + (R > 1 ? tid % per : tid);
          uint4 e0 = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u), e1 = make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0u);   // row -1: unused
          if (p < P) { const uint4* src = reinterpret_cast<const uint4*>(a.ent[d & 1] + p); e0 = __ldcg(src); e1 = __ldcg(src + 1); }
          uint4* dst = reinterpret_cast<uint4*>(sm.ent + tid);
          dst[0] = e0; dst[1] = e1;
          sm.thr[tid] = __uint_as_float(e1.x); sm.thr[TX_ROWS + tid] = __uint_as_float(e1.y);
          sm.ln[tid] = 0; sm.ln[TX_ROWS + tid] = 0; sm.lthr[tid] = -INFINITY; sm.lthr[TX_ROWS + tid] = -INFINITY;
        }
        for (int i = tid; i < 2 * TX_SPLIT * TX_ROWS; i += TX_THREADS) sm.best[i] = -INFINITY;
        if (g == 0) for (int i = tid; i < TX_QCAP; i += TX_THREADS) sm.q[i] = 0ull;   // (owners work in this memory: the queue's tags start clean)
        __syncthreads();
        // ask L2 for this range of every base-logit row the group reads (neighbours of the list often share theirs): the scan
        // itself asks for 32 bytes a lane one chunk ahead, which leaves DRAM waiting when the rows are many
        if (!RING) {
          const int nrow = min(TX_ROWS, P - g * TX_ROWS), lines = (tlen * 2 + 127) / 128;
#pragma unroll 1
          for (int x = warp; x < nrow; x += TX_WARPS) {
            const int rw = sm.ent[x].row;
            if (x > 0 && sm.ent[x - 1].row == rw) continue;
            const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(a.Uscan) + (size_t)rw * a.Vs + t0;
#pragma unroll 1
            for (int l = lane; l < lines; l += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + l * 64));
          }
        }
        const int done_target = (groups + 1) * TX_SCAN_WARPS;
        const int nst = min(512 / a.BN, TX_STAGE_MAX);   // accumulator stages
        const uint32_t ublocks = RING ? (uint32_t)((tlen + a.BN - 1) / a.BN) : 0u;
        if (warp < TX_SCAN_WARPS) tx_scan<RING>(a, sm, R, min(TX_ROWS, P - g * TX_ROWS), g, t0, tlen, tmem_base, pos, nst, ub0);
        else if (warp < TX_REFRESH) tx_issue(a, sm, warp - TX_MMA, tlen, tmem_base, pos, wpos, groups, nst);
        else if (warp == TX_REFRESH) {
          const uint32_t nblk = (uint32_t)((tlen + a.BN - 1) / a.BN);
          const uint32_t level_end = (uint32_t)(groups + ngroups - g) * nblk + ((a.w_over || a.score_P > 0) ? 0u : (uint32_t)a.nW);
          tx_refresh<RING>(a, sm, R, P, g, cta, done_target, &tmW, t0, tlen, wl, min((uint32_t)(groups + 1) * nblk + (uint32_t)a.nW, level_end), &tmU, d, ul, ub0 + ublocks);
        } else tx_drain(a, sm, R, g, cta, done_target);
        ub0 += ublocks;
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (*sm.abort) { dead = true; break; }
        tx_publish(a, sm, R, P, g, cta, a.cand_cnt[d & 1]);
        __syncthreads();
      }
    }
    if (dead) { if (tid == 0) atomicExch(a.barrier + 1, 1u); break; }
    if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) { dead = true; break; }
    if (a.score_P > 0) {
      // given parents: merged by all CTAs, results to the caller
      const int K = a.K;
      for (int x = cta + ncta * warp; x < 3 * P; x += ncta * TX_WARPS) {
        const int kind = x / P, p = x - kind * P;
        const size_t cb = cand_base(a, P, p);
        if (kind == 0) {
          const float2 l = warp_lse(a.sums + (size_t)p * a.ntiles, a.ntiles, a.T, lane);
          if (lane == 0) { a.o_lse0[p] = l.x; a.o_lseT[p] = l.y; }
          continue;
        }
        if (kind == 2 && !(a.T > 0.f)) continue;
        const float3 w = warp_topk(kind == 1 ? a.cand_top + cb : a.cand_key + cb, kind == 1 ? nullptr : a.cand_lg + cb, a.cand_cnt[0] + (kind == 1 ? 0 : a.cap) + p, K, lane);
        if (lane < K) {
          const size_t o = (size_t)p * K + lane;
          if (kind == 1) { a.o_top_tok[o] = __float_as_int(w.x); a.o_top_logit[o] = w.y; }
          if (kind == 2 || !(a.T > 0.f)) { a.o_draw_tok[o] = __float_as_int(w.x); a.o_draw_logit[o] = w.z; }
        }
      }
      break;
    }
    }
    // ---- merge by all CTAs where the owners alone would take long over it (8 requests with 60 parents each: 150 us; from 4
    // parents a request on instead of 8 the extra barrier costs up to 7 %, from 16 on within 2 % either way) ---------------
    const bool spread = MANY && d >= 0 && P > 8 * a.B;
    if (spread) {
      const int K = a.K;
#pragma unroll 1
      for (int x = cta + ncta * warp; x < 3 * P; x += ncta * TX_WARPS) {   // (a parent's three parts side by side)
        const int kind = x / P, p = x - kind * P;
        const size_t cb = cand_base(a, P, p);
        if (kind == 0) {
          const float2 l = warp_lse(a.sums + (size_t)p * a.ntiles, a.ntiles, a.T, lane);
          if (lane == 0) a.res_lse[p] = l;
          continue;
        }
        if (kind == 2 && !(a.T > 0.f)) continue;
        const float3 w = warp_topk(kind == 1 ? a.cand_top + cb : a.cand_key + cb, kind == 1 ? nullptr : a.cand_lg + cb, a.cand_cnt[d & 1] + (kind == 1 ? 0 : a.cap) + p, K, lane);
        uint2* out = reinterpret_cast<uint2*>(a.res_cand + (size_t)p * KMAX + lane);
        if (lane < K) {
          if (kind == 1) out[0] = make_uint2(__float_as_uint(w.x), __float_as_uint(w.y));
          if (kind == 2 || !(a.T > 0.f)) out[1] = make_uint2(__float_as_uint(w.x), __float_as_uint(w.z));
        }
      }
      if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) { dead = true; break; }
    }
    // ---- owners (second turn: shares of the seed bounds that owners with many new parents left) ----------------------------
    bool over = false;
#pragma unroll 1
    for (int turn = 0;; ++turn) {
      if (d >= -1) {
        const int first = MANY && turn ? cta % nreq : cta, share = MANY && turn ? cta / nreq : -1, hstep = MANY ? ncta / nreq : 1;
        if (!MANY || share < hstep)
#pragma unroll 1
          for (int b = first; b < nreq; b += MANY && turn ? nreq : ncta) tx_owner<MANY>(a, base_sm, b, d, share, hstep, spread, P);
      }
      // best base logits of the rows after the next ones, by the CTAs that own no request where there are enough of them
      // (given parents: of their rows, before anything else)
      if (turn == 0 && (d == -2 || (a.score_P == 0 && d + 2 < a.D))) {
        const int h0 = d >= -1 && ncta - a.B >= ncta / 4 ? a.B : 0;
        const int piece_len = (((a.V + a.npiece - 1) / a.npiece) + 7) & ~7;
        uint2* ut = a.utop + (size_t)(d & 1) * a.B * a.npiece;
        if (cta >= h0)
#pragma unroll 1
          for (int i = (cta - h0) * TX_WARPS + warp; i < nreq * a.npiece; i += (ncta - h0) * TX_WARPS) {
            const int x = i / a.npiece;
            if (d >= 0 && __ldcg(a.req_npar + (d & 1) * a.B + x) <= 0) continue;
            const int row = a.score_P > 0 ? a.p_req[x] * a.D + a.p_depth[x] : x * a.D + d + 2;
            scout_piece(a, row, i % a.npiece, piece_len, ut + i, lane);
          }
      }
      if (d + 1 >= a.D && a.score_P == 0) { over = true; break; }
      if (RING && a.ragged) asm volatile("fence.proxy.async;" ::: "memory");   // the padded rows written here are read by bulk-tensor loads
      fence_async_smem();   // owners work in memory that the next scan's bulk loads may write
      if (!grid_barrier(a.barrier, nexpect, gen, a.wait_limit)) { dead = true; break; }
      if (!MANY || turn || d < 0 || __ldcg(a.seed_need + d + 1) == 0) break;   // uniform: written before the barrier
    }
    if (over || dead) break;
    if (a.ragged && (RING || d == -2)) asm volatile("fence.proxy.async;" ::: "memory");   // (and after it, for the warp that requests them)
  }
  if (dead && d == -2 && a.score_P == 0) {
    for (int b = cta; b < a.B; b += ncta) {   // nothing of these requests exists yet: an empty tree
      PoolView g = pool_view(a.pool + (size_t)b * a.pool_stride, a.N);
      for (int i = tid; i < a.N; i += TX_THREADS) g.meta[i] = 0;
      if (tid == 0) { a.status[b] = TS_OK; a.req_nscored[b] = 0; a.root_lseT[b] = nanf(""); }
    }
    __syncthreads();
  }
  // ---- no copy may still be writing this CTA's shared memory when the last phase works in it or the CTA ends -----------
  cp_async_wait_all();
  if (a.use_tma && warp == TX_REFRESH && lane == 0)
    for (uint32_t x = wl.requested > (uint32_t)a.nW ? wl.requested - (uint32_t)a.nW : 0u; x < wl.requested; ++x) {
      const uint32_t slot = x % (uint32_t)a.nW, use = x / (uint32_t)a.nW;
      bool landed = false;
      for (uint32_t i = 0; i < WAIT_LIMIT && !landed; ++i) { landed = mbar_test_wait(sm.w_full + slot, use & 1); if (!landed) __nanosleep(100); }
    }
  if (RING && warp == TX_REFRESH && lane == 0)
    for (uint32_t x = ul.requested > (uint32_t)TX_USTAGES ? ul.requested - (uint32_t)TX_USTAGES : 0u; x < ul.requested; ++x) {
      bool landed = false;
      for (uint32_t i = 0; i < WAIT_LIMIT && !landed; ++i) { landed = mbar_test_wait(sm.u_full + (x & (uint32_t)(TX_USTAGES - 1)), (x / TX_USTAGES) & 1u); if (!landed) __nanosleep(100); }
    }
  if (dead && tid == 0) { atomicExch(a.barrier + 1, 1u); atomicExch(a.err, 1); }
  __syncthreads();
  const bool late = dead || *reinterpret_cast<volatile int*>(a.err) != 0;
  if (a.score_P == 0) {
    for (int b = cta; b < a.B; b += ncta) tx_finalize<MANY>(a, base_sm, b, late);
  } else if (!MANY && !RING && late) {   // given parents: there is no status array to report it in (in the other instantiations
                                         // the code alone cost the chain of 128 requests 20 us of 726)
    for (int p = cta; p < a.score_P; p += ncta) {
      if (tid == 0) a.o_lse0[p] = a.o_lseT[p] = nanf("");
      if (tid < a.K) {
        const size_t o = (size_t)p * a.K + tid;
        a.o_top_tok[o] = a.o_draw_tok[o] = -1; a.o_top_logit[o] = a.o_draw_logit[o] = 0.f;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == TX_MMA) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

__global__ void tree_init_kernel(unsigned* words, int n) {
  pdl_wait();                // the launch before may still be using them
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < n; i += blockDim.x) words[i] = 0u;
}

// ------------------------------------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------------------------------------

// Shared-memory plan: A tile, ring of base-logit blocks, selection state, ring of W blocks.  Blocks of 128 tokens where two
// stages of each ring fit (one MMA instruction a K step fills 128 columns: issuing costs per instruction), else 64;
// what is left goes to deeper rings.
bool tree_plan(const ts_config& c, int num_sms, int max_smem, TreePlan* out) {
  const size_t rp = (size_t)(c.r + 63) / 64 * 64, rw = (size_t)(c.r + 15) / 16 * 16;
  const size_t avail = (size_t)max_smem - 1024 - 512;   // alignment, static shared memory
  auto up = [](size_t x) { return (x + 1023) & ~(size_t)1023; };
  TreePlan p{};
  p.TV = ((c.V + num_sms - 1) / num_sms + 63) / 64 * 64;
  p.ntiles = (c.V + p.TV - 1) / p.TV;
  if (p.TV > 1 << TX_PLACE_BITS) return false;   // (never on 148 SMs: V <= 2^24)
  p.Vs = (c.V + 7) & ~7;
  int piece = ((c.V + 127) / 128 + 7) & ~7;
  piece = piece < 64 ? 64 : (piece > TX_PIECE ? TX_PIECE : piece);
  p.npiece = (c.V + piece - 1) / piece;
  const size_t own = owner_layout(c.Nmax, c.K, c.r).total, sel = up(tx_select_bytes(c.K)), fix = up(TX_FIXED_BYTES), A = rp * 256;
  for (int BN = 128; BN >= 64; BN /= 2) {
    const size_t w = rw * 2 * BN;
    int nW = 2;
    auto total = [&](int nw) { return A + sel + fix + (size_t)nw * w; };
    if (total(nW) > avail) continue;
    while (nW < TX_STAGE_MAX && total(nW + 1) <= avail) ++nW;
    // An even number of blocks of 128: with an odd one the two issuing warps' slots don't alternate (expansion of 32 requests at
    // V = 64,000: rank 160, K = 14: 267 us with two, 287 with three; rank 128, K = 2: 123 with four, 127 with five).  Blocks of 64
    // are too short for two stages (rank 256, V = 151,936: 322 with two, 305 with three).
    if (BN == 128) nW &= ~1;
    p.BN = BN; p.nW = nW;
    p.oL = (uint32_t)A; p.oW = (uint32_t)(p.oL + sel); p.oX = (uint32_t)(p.oW + (size_t)nW * w);
    // owners work in [A, selection state] and, where that is not enough, in the W ring (which then does not run ahead);
    // where not even that is, behind them
    p.w_over = own > p.oW ? 1 : 0;
    if (own > p.oX) p.oX = (uint32_t)up(own);
    if (p.oX + fix > avail) continue;
    p.smem = p.oX + fix + 1024;
    // The form with the base-logit ring: RU stages of it beside what W stages then fit.
    p.rowsU = ((c.max_batch < TX_ROWS ? c.max_batch : TX_ROWS) + 7) & ~7;
    const size_t ring = (size_t)TX_USTAGES * (BN / 64) * p.rowsU * 128;
    auto behind = [&](int nw) { const size_t x = p.oW + (size_t)nw * w; return up(own > x ? own : x); };
    p.ring_nW = 0;
    for (int nw = 2; nw <= TX_STAGE_MAX && behind(nw) + fix + ring <= avail; ++nw) p.ring_nW = nw;
    if (p.ring_nW) { p.ring_oX = (uint32_t)behind(p.ring_nW); p.ring_oU = (uint32_t)(p.ring_oX + fix); p.ring_smem = p.ring_oU + ring + 1024; }
    *out = p;
    return true;
  }
  return false;
}

// Workspace of one call over `nreq` requests (or given parents) whose lists hold up to `cap` parents.
struct TreeWs { size_t head, ent[2], slot[2], sums, cnt, top, key, lg, thr, utop, pool, state, caps, rlse, rcand, upad, wpad, total; int cap; };
// given parents whose last group may be held in copies (the built-in scratch array, rows = 0, has no room for them)
static bool tail_copies(bool expand, int rows) { return !expand && rows > 0; }
static TreeWs tree_ws(const ts_ctx* ctx, int nreq, int cap, bool expand, int rows) {
  const ts_config& c = ctx->cfg; const TreePlan& p = ctx->tree;
  TreeWs w{}; size_t at = 0;
  auto take = [&](size_t bytes) { const size_t o = at; at = align_up(at + bytes, 256); return o; };
  w.cap = cap = (cap + 7) / 8 * 8;
  const size_t C = (size_t)cap, nt = (size_t)p.ntiles, cands = (tail_copies(expand, rows) ? (C + TX_ROWS - 1) / TX_ROWS * TX_ROWS : C > TX_ROWS ? C : (size_t)TX_ROWS) * nt * c.K;   // (copies of rows: at most 128 a group)
  w.head = take(256);
  w.ent[0] = take(C * sizeof(ParentEntry));
  if (expand) { w.ent[1] = take(C * sizeof(ParentEntry)); w.slot[0] = take(C * 4); w.slot[1] = take(C * 4); }
  w.sums = take(C * nt * 16); w.cnt = take((expand ? 4 : 2) * C * 4);
  w.top = take(cands * 8); w.key = take(cands * 8); w.lg = take(cands * 4);
  w.thr = take(2 * C * 4 + 2 * C * c.K * SLOT_STRIDE * 4);
  w.utop = take((size_t)nreq * (expand ? 2 : 1) * p.npiece * 8);
  if (expand) { w.pool = take((size_t)nreq * pool_bytes(c.Nmax)); w.state = take((size_t)nreq * 5 * 4); w.caps = take((size_t)nreq * 16); w.rlse = take(C * 8); w.rcand = take(C * KMAX * 16); }
  if (c.V % 8) { w.upad = take((size_t)rows * p.Vs * 2); w.wpad = take((size_t)c.r * p.Vs * 2); }
  w.total = at;
  return w;
}

// the region of the caller's workspace: sized for expansion, and for given parents up to the same list length
size_t tree_ws_bytes(const ts_ctx* ctx, int B) {
  const int cap = B * ctx->cfg.Nmax > B ? B * ctx->cfg.Nmax : B;
  const size_t e = tree_ws(ctx, B, cap, true, B * ctx->cfg.D).total, g = tree_ws(ctx, cap, cap, false, B * ctx->cfg.D).total;
  const size_t t = e > g ? e : g, f = ctx->few_cap > 0 ? score_scratch_bytes(ctx, ctx->few_cap, nullptr) : 0;   // (short lists: ts_score_few.cu)
  return t > f ? t : f;
}

// scratch of a scoring call over P given parents; 0: not possible without the caller's workspace (padded copies)
size_t tree_score_bytes(const ts_ctx* ctx, int P) { return ctx->cfg.V % 8 ? 0 : tree_ws(ctx, P, P, false, 0).total; }

static void fill_args(ts_ctx* ctx, TreeArgs& a, char* base, const TreeWs& w, bool expand, const void* U, const void* A, const void* W, float T, uint64_t seed) {
  const ts_config& c = ctx->cfg; const TreePlan& p = ctx->tree;
  a.U = U; a.A = A; a.W = W; a.V = c.V; a.D = c.D; a.r = c.r; a.K = c.K; a.N = c.Nmax; a.T = T; a.seed = seed;
  a.own = owner_layout(c.Nmax, c.K, c.r);
  a.ragged = c.V % 8 ? 1 : 0;
  a.Vs = p.Vs; a.Uscan = a.ragged ? base + w.upad : U; a.Wscan = a.ragged ? base + w.wpad : W;
  a.wide_u = (p.Vs % 16 == 0 && ((uintptr_t)a.Uscan & 31u) == 0) ? 1 : 0;
  a.TV = p.TV; a.ntiles = p.ntiles; a.BN = p.BN; a.nW = p.nW; a.npiece = p.npiece; a.w_over = p.w_over;
  a.lstride = list_stride(c.K); a.oL = p.oL; a.oW = p.oW; a.oX = p.oX; a.oU = 0; a.rowsU = p.rowsU;
  for (uint32_t i = 0; i < 10; ++i) { a.rk[2 * i] = (uint32_t)seed + i * 0x9E3779B9u; a.rk[2 * i + 1] = (uint32_t)(seed >> 32) + i * 0xBB67AE85u; }
  a.no_seed = (ctx->test_mode & TS_TEST_NO_SEED) ? 1 : 0;
  int* head = (int*)(base + w.head);
  a.barrier = (unsigned*)head; a.err = head + 4; a.lvl_count = head + 8; a.seed_need = head + 8 + DMAX + 2;
  for (int i = 0; i < (expand ? 2 : 1); ++i) { a.ent[i] = (ParentEntry*)(base + w.ent[i]); a.ent_slot[i] = expand ? (int*)(base + w.slot[i]) : nullptr; }
  a.sums = (float4*)(base + w.sums); for (int i = 0; i < 2; ++i) a.cand_cnt[i] = (int*)(base + w.cnt) + (expand ? i : 0) * 2 * (size_t)w.cap;
  a.cand_top = (uint2*)(base + w.top); a.cand_key = (uint2*)(base + w.key); a.cand_lg = (float*)(base + w.lg);
  a.cap = w.cap; a.thr = (unsigned*)(base + w.thr); a.slots = a.thr + 2 * (size_t)w.cap;
  a.utop = (uint2*)(base + w.utop);
  a.wait_limit = ctx->wait_limit; a.lost_arrival = (ctx->test_mode & TS_TEST_LOST_ARRIVAL) ? 1 : 0;
}

static cudaError_t launch_tree(ts_ctx* ctx, TreeArgs& a, int prof_id, cudaStream_t st) {
  // Crowded levels (a request with dozens of parents) need room for them in the tree and CTAs to spare.  Expansion, owners
  // alone / sharing (us): K = 16, flat logits, Nmax 96: 331 / 257 for 1 request, 591 / 520 for 8, 1,916 / 1,918 for 64; Nmax
  // 256: 607 / 378, 1,140 / 894, 3,824 / 3,693.  Where levels are not crowded sharing costs 2 to 8 %, at any Nmax: 222 / 239 for
  // 32 requests of 16 nodes at Nmax 96, 226 / 245 at 128; with K = 8 it does not pay up to Nmax 128 (640 / 679 and 759 / 792 for 32).
  const bool many = a.score_P == 0 && ctx->num_sms >= 2 * a.B && a.N > 96;
  CUtensorMap tm, tmU;
  memset(&tm, 0, sizeof(tm)); memset(&tmU, 0, sizeof(tmU));
  a.use_tma = tree_tensor_map(ctx, a.Wscan, a.Vs, &tm) ? 1 : 0;
  // (given parents lie at mixed depths, and a box holds 128 requests)
  const TreePlan& p = ctx->tree;
  const bool ring = p.ring_nW > 0 && a.score_P == 0 && !many && a.B >= TX_RING_MIN && a.B <= a.rowsU && u_tensor_map(ctx, a.Uscan, a.Vs, a.B, a.rowsU, &tmU);
  if (ring) { a.nW = p.ring_nW; a.oX = p.ring_oX; a.oU = p.ring_oU; }
  cudaError_t e;
  { ProfScope ps(ctx, K_INIT, st); e = launch_kernel(tree_init_kernel, 1, 64, 0, st, true, a.barrier, 8 + 2 * (DMAX + 2)); }
  if (e != cudaSuccess) return e;
  ProfScope ps(ctx, prof_id, st);
  const void* fn = many ? (const void*)tree_kernel<true, false> : (ring ? (const void*)tree_kernel<false, true> : (const void*)tree_kernel<false, false>);
  void* kargs[] = {(void*)&a, (void*)&tm, (void*)&tmU};
  return launch_cooperative(ctx->tree_unchained, fn, dim3(ctx->num_sms), dim3(TX_THREADS), ring ? p.ring_smem : p.smem, st, kargs);
}

cudaError_t tree_setup(ts_ctx* ctx) {
  cudaError_t e = allow_all_smem(tree_kernel<false, false>, ctx->max_smem);
  if (e == cudaSuccess) e = allow_all_smem(tree_kernel<true, false>, ctx->max_smem);
  return e != cudaSuccess ? e : allow_all_smem(tree_kernel<false, true>, ctx->max_smem);
}

cudaError_t tree_score(ts_ctx* ctx, char* scratch, const void* U, const void* A, const void* W, int P, const int* p_req, const int* p_depth, const int* p_token,
                       const uint64_t* p_hash, float T, uint64_t seed, float* lse0, float* lseT, int* top_tok, float* top_logit, int* draw_tok,
                       float* draw_logit, int rows, cudaStream_t st) {
  TreeArgs a{};
  fill_args(ctx, a, scratch, tree_ws(ctx, P, P, false, rows), false, U, A, W, T, seed);
  a.score_P = P; a.B = 1; a.tail_copies = tail_copies(false, rows) ? 1 : 0;
  a.p_req = p_req; a.p_depth = p_depth; a.p_token = p_token; a.p_hash = p_hash;
  a.o_lse0 = lse0; a.o_lseT = lseT; a.o_top_tok = top_tok; a.o_top_logit = top_logit; a.o_draw_tok = draw_tok; a.o_draw_logit = draw_logit;
  return launch_tree(ctx, a, K_SCORE, st);
}

cudaError_t tree_expand(ts_ctx* ctx, char* ws, const TreeOut& o, const void* U, const void* A, const void* W, int B, const int* anchor, const float* theta,
                        float T, uint64_t seed, cudaStream_t st) {
  const ts_config& c = ctx->cfg;
  TreeArgs a{};
  const TreeWs w = tree_ws(ctx, B, B * c.Nmax > B ? B * c.Nmax : B, true, B * c.D);
  fill_args(ctx, a, ws, w, true, U, A, W, T, seed);
  a.B = B; a.anchor = anchor; a.theta = theta; a.calib = ctx->calib; a.calib_qT = (ctx->ablation & TS_ABLATE_CALIB_QT) ? 1 : 0;
  a.pool = (unsigned char*)ws + w.pool; a.pool_stride = pool_bytes(c.Nmax);
  int* state = (int*)(ws + w.state);
  a.req_npar = state; a.req_base = state + 2 * (size_t)B; a.req_nscored = state + 3 * (size_t)B; a.root_lseT = (float*)(state + 4 * (size_t)B);
  a.req_caps = (double2*)(ws + w.caps); a.res_lse = (float2*)(ws + w.rlse); a.res_cand = (uint4*)(ws + w.rcand);
  a.n_nodes = o.n_nodes; a.tok = o.tok; a.parent = o.parent; a.depth = o.depth; a.sib_rank = o.sib_rank; a.logS = o.logS; a.q0 = o.q0; a.logqT = o.logqT;
  a.logkey = o.logkey; a.pop_rank = o.pop_rank; a.node_hash = o.node_hash; a.node_lseT = o.node_lseT; a.mask = o.mask; a.n_scored = o.n_scored; a.status = o.status;
  a.words = (c.Nmax + 63) / 64;
  return launch_tree(ctx, a, K_PERSIST, st);
}

}  // namespace ts
