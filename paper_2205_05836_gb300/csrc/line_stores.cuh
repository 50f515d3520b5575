// Bit-deposit stores in whole lines, shared by the tensor-core epilogues.
//
// A 32 x 32 block of C (rows m0 .., columns n0 .., both multiples of 32) goes
// to out[pdep(m, mask_m) | pdep(n, mask_n)].  Each of the five lowest output
// bits belongs to one of the two masks: cm of them to m (its cm lowest bits)
// and cn = 5 - cm to n.  The 32 floats of one 128-byte line are therefore the
// elements whose low cm row bits and low cn column bits take every value
// while the other bits stay fixed, and the block is 32 such lines.  The warp
// stages the block in shared memory (lane = row) and walks it line by line,
// lane l holding the element at offset l of the line, so that every store
// instruction writes one full line.  (One row at a time, lane = column, the
// 32 floats went to up to 32 sectors: 4 bytes of each.)
// Element (r, c) is staged at r * 32 + (c ^ rotl5(r, cn)): distinct banks for
// the writes (r = lane, c fixed) and for the reads (below).
#pragma once

#include "internal.cuh"

namespace cutqc {

struct LineStores {
  int cm, cn;            // low output bits held by m and by n; cm + cn < 5: fewer than 32 outputs
  uint64_t line_off[32]; // offset of line i: row bits from cm up take i's low cn bits, column bits from cn up the rest
};

inline LineStores line_stores(uint64_t mask_m, uint64_t mask_n) {
  LineStores s{};
  s.cm = __builtin_popcountll(mask_m & 31);
  s.cn = __builtin_popcountll(mask_n & 31);
  if (s.cm + s.cn == 5)
    for (int i = 0; i < 32; ++i)
      s.line_off[i] = pdep64((uint64_t)(i & ((1 << s.cn) - 1)) << s.cm, mask_m) |
                      pdep64((uint64_t)(i >> s.cn) << s.cn, mask_n);
  return s;
}

// v: this lane's row (m0 + lane) of the block; base: the output offset of
// element (m0, n0).  stored(value) is called for every element this lane
// stores.  (The callers know the base from a warp-wide deposit; depositing m0
// and n0 bit by bit here took 800 cycles a block: 2^26 outputs of 16 terms 274
// us.)
template <class F>
__device__ __forceinline__ void store_block_lines(const float (&v)[32], float* stg, const LineStores& s, int lane,
                                                  int64_t m0, int64_t n0, int64_t M, int64_t N, uint64_t mask_m,
                                                  uint64_t mask_n, uint64_t base, float* out, int streaming,
                                                  F&& stored) {
  const int cm = s.cm, cn = s.cn;
  const int rot = ((lane << cn) | (lane >> (5 - cn))) & 31;
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 32; ++c) stg[lane * 32 + (c ^ rot)] = v[c];
  __syncwarp();
  if (cm + cn < 5) {
    // fewer than 32 outputs in all
    for (int r = 0; r < 32; ++r) {
      const int64_t m = m0 + r, n = n0 + lane;
      if (m < M && n < N) {
        const float val = stg[r * 32 + (lane ^ (((r << cn) | (r >> (5 - cn))) & 31))];
        out[pdep64((uint64_t)m, mask_m) | pdep64((uint64_t)n, mask_n)] = val;
        stored(val);
      }
    }
    return;
  }
  // the lane's low row and column bits: bit j of the lane is output bit j
  int mp = 0, np = 0;
  {
    int im = 0, in = 0;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int b = (lane >> j) & 1;
      if ((mask_n >> j) & 1) np |= b << in++;
      else mp |= b << im++;
    }
  }
  const int swz = np ^ (mp << cn);
  float* dst = out + (base | (uint64_t)lane);
  const bool full = m0 + 32 <= M && n0 + 32 <= N;
  const float* src = stg + mp * 32;
#pragma unroll 8
  for (int i = 0; i < 32; ++i) {
    const int mh = i & ((1 << cn) - 1), nh = i >> cn;
    // rotl5(mp | mh << cm, cn) = mp << cn | mh, so the column of the element
    // is (np | nh << cn) ^ (mp << cn | mh) = swz ^ i
    const float val = src[(mh << (cm + 5)) + (swz ^ i)];
    if (full || (m0 + (mp | (mh << cm)) < M && n0 + (np | (nh << cn)) < N)) {
      float* p = dst + s.line_off[i];
      if (streaming) __stcs(p, val);
      else *p = val;
      stored(val);
    }
  }
}

}  // namespace cutqc
