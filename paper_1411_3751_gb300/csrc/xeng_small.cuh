// Parts of the X-engine that reads the packed samples itself (no operand in HBM, xeng_small.cu). Operand encoding and
// the sums that undo it: f8_common.cuh.
#pragma once

#include "f8_common.cuh"

namespace corr {
namespace xd {

constexpr int MAX_BLOCKS = 16;  // blocks of one launch: one tensor map each

struct Args {
  CUtensorMap map[MAX_BLOCKS];  // block b as [T][C ld] bytes
  long long* cross;
  long long* autos;
  long long* s1;  // offset sums [C][N][2], both cadences
  long long* s2;
  long long Bs;
  int N, C, npol, T;
  int ld;               // inputs a row and channel as stored: N, or more (repacked rows)
  int n_kb, n_k;        // 128-sample stages of a block (the last one may be short) and of all blocks
  int chunk_k;          // stages per in-chip partial sum
  int splits, kps;      // the stages of an item are divided over `splits` items of kps stages
  int n_units, g, ub;   // 64-input units, channels and bytes of one
  long long n_items;
  int* err;
};

// One 32-column chunk of an accumulator (16 a-inputs: columns k and 16 + k = Re and Im of a_k) as complex products: the
// lanes holding Re c and Im c of one c-input are 16 apart, exchange half of their columns and own 8 a-inputs
// each, the Re lane the even, the Im lane the odd ones. Combining first halves the words a thread holds, and
// leaves registers for eight cells in flight.
__device__ __forceinline__ void combine_chunk(const uint32_t (&v)[32], bool im_lane, int (&re)[8], int (&im)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    // columns of the even input; the odd one's follow
    const int jr = 2 * k, ji = jr + 16;
    const int own_r = f8::to_int(__uint_as_float(im_lane ? v[jr + 1] : v[jr]));
    const int own_i = f8::to_int(__uint_as_float(im_lane ? v[ji + 1] : v[ji]));
    const int recv_r = f8::to_int(__shfl_xor_sync(0xffffffffu, __uint_as_float(im_lane ? v[jr] : v[jr + 1]), 16));
    const int recv_i = f8::to_int(__shfl_xor_sync(0xffffffffu, __uint_as_float(im_lane ? v[ji] : v[ji + 1]), 16));
    // Re lane: own row Re c, partner Im c; Im lane the other way round
    re[k] = im_lane ? recv_r + own_i : own_r + recv_i;
    im[k] = im_lane ? recv_i - own_r : own_i - recv_r;
  }
}

// Cells as 32-bit offsets from the channel's first (a channel has less than 2^31 of them): half the registers of pointers.
template <bool ADD>
__device__ __forceinline__ void add_cells(longlong2* __restrict__ base, const uint32_t (&cell)[8], uint32_t valid,
                                          const int (&re)[8], const int (&im)[8]) {
  if (ADD) {
#pragma unroll
    for (int m = 0; m < 8; ++m)
      if (valid & (1u << m)) {
        atomicAdd(reinterpret_cast<unsigned long long*>(base + cell[m]), (unsigned long long)(long long)re[m]);
        atomicAdd(reinterpret_cast<unsigned long long*>(base + cell[m]) + 1, (unsigned long long)(long long)im[m]);
      }
  } else {
    longlong2 old[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) old[m] = base[cell[m]];
#pragma unroll
    for (int m = 0; m < 8; ++m)
      if (valid & (1u << m)) base[cell[m]] = make_longlong2(old[m].x + re[m], old[m].y + im[m]);
  }
}

// Adds a combined chunk of a-inputs from a_base (the lane's own a_base + im_lane + 2 k) to cross[f] and, on the
// diagonal, autos[f]. ADD: 64-bit reductions (items that share cells), else load, add, store.
// lp = log2(n_pol): station n >> lp, polarisation n & lp (n_pol is 1 or 2).
template <bool ADD>
__device__ __forceinline__ void add_chunk(const int (&re)[8], const int (&im)[8], bool im_lane, int c, int a_base, int N,
                                          int lp, long long* __restrict__ cross_f, long long* __restrict__ autos_f) {
  const unsigned sc = (unsigned)c >> lp, pc = (unsigned)c & (unsigned)lp;
  uint32_t cell[8];
  uint32_t valid = 0u;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int a = a_base + (im_lane ? 1 : 0) + 2 * k;
    cell[k] = 0u;  // in-bounds placeholder for skipped cells (loaded, never stored)
    if (a >= 0 && a < N && c >= 0 && c < N) {
      const unsigned sa = (unsigned)a >> lp;
      if (sa >= sc) {
        const unsigned b = sa * (sa + 1) / 2 + sc;
        cell[k] = (b << (2 * lp)) + ((((unsigned)a & (unsigned)lp) << lp) + pc);
        valid |= 1u << k;
        if (a == c) {
          if (ADD)
            atomicAdd(reinterpret_cast<unsigned long long*>(autos_f + a), (unsigned long long)(long long)re[k]);
          else
            autos_f[a] += re[k];
        }
      }
    }
  }
  add_cells<ADD>(reinterpret_cast<longlong2*>(cross_f), cell, valid, re, im);
}

// Stage k of an item's blocks: block k / n_kb, sample 128 (k % n_kb).
struct StagePos {
  int blk, kb;
  __device__ __forceinline__ StagePos(int k, int n_kb) : blk(k / n_kb), kb(k - (k / n_kb) * n_kb) {}
  __device__ __forceinline__ void next(int n_kb, int step = 1) {
    kb += step;
    while (kb >= n_kb) {
      kb -= n_kb;
      ++blk;
    }
  }
};

}  // namespace xd

// Blocks of T samples that one launch takes: a tensor map each, and at most 2^28 samples (the offset sums of a
// converter thread are 32-bit).
inline int direct_max_blocks(int T) {
  const long long k = (1LL << 28) / T;
  return k < 1 ? 1 : (k < xd::MAX_BLOCKS ? (int)k : xd::MAX_BLOCKS);
}

// One launch's work: `n` blocks of T_blk samples of one array.
struct DirectJob {
  Shape s;
  const uint8_t* const* blocks;  // [T_blk][C][ld]
  int n, T_blk, ld, flush_len;
  long long *cross, *autos, *s1, *s2;
  int* err;
};

}  // namespace corr
