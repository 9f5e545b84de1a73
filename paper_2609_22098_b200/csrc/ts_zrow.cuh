// Statistics of the target rows (maximum, its first position, log-sum-exp at temperature T) by pieces: the split that
// zrow_stats_kernel (ts_verify.cu) works by, and the fold of a row's pieces by whoever reads the row next.
#pragma once
#include "ts_common.cuh"

namespace ts {

constexpr int ZT = 512;        // threads per piece
constexpr int ZSPLIT = 8;      // a row is cut into at most this many pieces by length ...
constexpr int ZPIECES = ZSPLIT + 2;   // ... and so lies in at most this many

// Elements per piece.  The rows are one array of `total` elements, cut into equal pieces without regard to the rows: 15
// rows of one request occupy 120 SMs and 500 rows leave no last wave.  Below an eighth of a row (or 4096 elements, eight
// per thread) a piece would cost more in its fold than in its loads.
__device__ __forceinline__ int64_t zrow_piece(int64_t total, int V, int npiece) {
  int64_t q = (total + npiece - 1) / npiece;
  const int64_t least = (V + ZSPLIT - 1) / ZSPLIT > 4096 ? (V + ZSPLIT - 1) / ZSPLIT : 4096;
  if (q < least) q = least;
  return (q + 7) & ~(int64_t)7;
}

// One piece's share of a row: maximum (NaN: the share holds one), its first position, sum of exp((z - ref) / T).
struct __align__(16) ZPart { float m; int arg; float ref, sum; };
struct ZRow { float m; int arg; float logs; };

// The share of piece c in `row` is part[row + c] (along the array, either the row or the piece changes from share to share).
__device__ __forceinline__ ZRow zrow_fold(const ZPart* part, int64_t row, int V, int64_t q, int npiece, float T) {
  int64_t c0 = row * V / q, c1 = ((row + 1) * V - 1) / q;
  if (c1 > npiece - 1) c1 = npiece - 1;
  const int n = (int)(c1 - c0) + 1;
  ZPart v[ZPIECES];
#pragma unroll
  for (int i = 0; i < ZPIECES; ++i) {
    v[i].m = -INFINITY; v[i].arg = 0x7FFFFFFF; v[i].ref = -INFINITY; v[i].sum = 0.f;
    if (i < n) *reinterpret_cast<float4*>(&v[i]) = __ldcg(reinterpret_cast<const float4*>(part + row + c0 + i));
  }
  ZRow o; o.m = -INFINITY; o.arg = 0x7FFFFFFF;
  bool nan = false;
#pragma unroll
  for (int i = 0; i < ZPIECES; ++i) {
    nan |= v[i].m != v[i].m;
    if (v[i].m > o.m || (v[i].m == o.m && v[i].arg < o.arg)) { o.m = v[i].m; o.arg = v[i].arg; }
  }
  const float invT = T > 0.f ? 1.f / T : 1.f;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < ZPIECES; ++i)
    if (v[i].ref > -INFINITY) s += v[i].sum * __expf((v[i].ref - o.m) * invT);
  o.logs = logf(s);
  if (nan) o.m = nanf("");
  return o;
}

}  // namespace ts
