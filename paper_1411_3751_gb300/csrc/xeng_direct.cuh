// Shared by the two X-engines that read the packed samples themselves (no operand in HBM): xeng_direct.cu
// (SM pairs, more than 64 inputs) and xeng_small.cu (at most 64 inputs). Operand encoding and the sums
// that undo it: f8_common.cuh.
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
  int n_units, g, ub;   // xeng_small: 64-input units, channels and bytes of one
  int nb, n_tiles;      // xeng_direct: 128-input blocks, tiles of the triangle
  long long n_items;
  int* err;
};

// Adds one 32-column chunk of an accumulator (16 a-inputs from a_base: column 8 (k / 4) + k % 4 = Re a_k, + 4 =
// Im a_k) to cross[f] and, on the diagonal, autos[f]. The lanes holding Re c and Im c of one c-input are
// XOR apart; they exchange half of their columns and own 8 a-inputs each. ADD: 64-bit reductions (items
// that share cells), else load, add, store, G (4 or 8) cells in flight.
template <int XOR, bool ADD, int G>
__device__ __forceinline__ void add_chunk(const uint32_t (&v)[32], bool im_lane, int c, int a_base, int N, int lp,
                                          long long* __restrict__ cross_f, long long* __restrict__ autos_f) {
  // lp = log2(n_pol): station n >> lp, polarisation n & lp (n_pol is 1 or 2)
  const unsigned sc = (unsigned)c >> lp, pc = (unsigned)c & (unsigned)lp;
#pragma unroll
  for (int k0 = 0; k0 < 8; k0 += G) {
    int re[G], im[G];
    long long* cell[G];
    uint32_t valid = 0u;
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int k = k0 + m, jr = 8 * (k >> 2) + (k & 3), ji = jr + 4;  // columns of a_k within the 16 kept
      const float own_r = __uint_as_float(im_lane ? v[16 + jr] : v[jr]);
      const float own_i = __uint_as_float(im_lane ? v[16 + ji] : v[ji]);
      const float recv_r = __shfl_xor_sync(0xffffffffu, __uint_as_float(im_lane ? v[jr] : v[16 + jr]), XOR);
      const float recv_i = __shfl_xor_sync(0xffffffffu, __uint_as_float(im_lane ? v[ji] : v[16 + ji]), XOR);
      // Re lane: own row Re c, partner Im c; Im lane the other way round
      re[m] = im_lane ? f8::to_int(recv_r) + f8::to_int(own_i) : f8::to_int(own_r) + f8::to_int(recv_i);
      im[m] = im_lane ? f8::to_int(recv_i) - f8::to_int(own_r) : f8::to_int(own_i) - f8::to_int(recv_r);
      const int a = a_base + (im_lane ? 8 : 0) + k;
      cell[m] = cross_f;  // in-bounds placeholder for skipped cells (loaded, never stored)
      if (a >= 0 && a < N && c >= 0 && c < N) {
        const unsigned sa = (unsigned)a >> lp;
        if (sa >= sc) {
          const unsigned b = sa * (sa + 1) / 2 + sc;
          cell[m] = cross_f + 2 * (((long long)b << (2 * lp)) + ((((unsigned)a & (unsigned)lp) << lp) + pc));
          valid |= 1u << m;
          if (a == c) {
            if (ADD)
              atomicAdd(reinterpret_cast<unsigned long long*>(autos_f + a), (unsigned long long)(long long)re[m]);
            else
              autos_f[a] += re[m];
          }
        }
      }
    }
    if (ADD) {
#pragma unroll
      for (int m = 0; m < G; ++m)
        if (valid & (1u << m)) {
          atomicAdd(reinterpret_cast<unsigned long long*>(cell[m]), (unsigned long long)(long long)re[m]);
          atomicAdd(reinterpret_cast<unsigned long long*>(cell[m]) + 1, (unsigned long long)(long long)im[m]);
        }
    } else {
      longlong2 old[G];
#pragma unroll
      for (int m = 0; m < G; ++m) old[m] = *reinterpret_cast<const longlong2*>(cell[m]);
#pragma unroll
      for (int m = 0; m < G; ++m)
        if (valid & (1u << m)) *reinterpret_cast<longlong2*>(cell[m]) = make_longlong2(old[m].x + re[m], old[m].y + im[m]);
    }
  }
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

// Items' stages are divided by direct_splits() where whole items leave SMs idle: the division of n_k stages that
// minimises waves x (stages + overhead), `slots` items running at once.
int direct_splits(long long items, int slots, int n_k, int overhead);
// The kernels' common arguments; boxes of box_bytes x 128 samples.
cudaError_t direct_args(const DirectJob& j, int box_bytes, bool swizzle, xd::Args* a);

}  // namespace corr
