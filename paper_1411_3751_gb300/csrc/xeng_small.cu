// X-engine for arrays of at most 64 inputs that builds its operand on the chip: tcgen05.mma (kind::f8f6f4, M = N
// = 128, K = 32) of a 64-input tile with itself, the tile made in shared memory from the packed samples
// that TMA brings in. HBM-bound: the samples are read once (the two-pass path wrote two operand bytes a
// sample and read them back, five times the traffic).
//
// A unit is 64 neighbouring sample bytes of a time, the MMA's 128 operand rows: one channel of up to 64
// inputs, or g channels of N inputs with g N <= 64 (their products are the diagonal blocks; those across
// channels are not used). With 33 to 63 inputs the unit runs into the next channel, whose rows are not
// used either. An item is two neighbouring units, so that TMA boxes are 128 bytes x 128 samples, and a
// range of stages of 128 samples. A unit that starts between 16-byte boundaries takes the columns from the
// boundary below on, and the rows of the unit before are not used: g leaves room for them. (Without that, such
// counts were repacked first: 20 inputs x 1200 channels x 4096 samples 91 us, 52 in place; 31 inputs 115 and 94.)
//
// A and B of a unit's MMA are the same rows. With both read from one shared-memory tile a stage moved 128 KB
// through shared memory (MMA reads 64, conversion 48, TMA 16) and took 660 ns, 1.3 times what HBM needs; so A
// comes from TMEM: ldmatrix.trans.b8 brings the samples into registers transposed (four samples of an input a
// word), a shift and logic operations make the operand words, and these go both to TMEM (A, tcgen05.st) and to
// the K-major, 128-byte swizzled tile (B): 96 KB a stage.
//
// Roles (one CTA per SM): warp 0 TMA producer; warp 1 TMEM allocation and MMA issuer; warps 4-19 converters, two
// sets that take the stages in turn, a warp for a TMEM lane quarter (16 inputs) of one unit, that also form the
// inputs' offset sums; warps 20-27 epilogue, likewise. The accumulators (256 columns) and the A ring (192) fill
// TMEM, so there is one accumulator a unit: the epilogue takes it into registers before it adds to the int64
// sums. The registers are split by setmaxnreg: 128 x 32 + 512 x 56 + 256 x 120 of the 896 x 72 of the launch.
// 32 inputs x 2400 channels x 4 x 8192 samples: 677 us with both operands in shared memory and one converter set,
// 705 with A in TMEM, 622 with a second set as well, 598 with the units' MMAs in turn (370 at the measured copy
// bandwidth). With a quarter of the MMAs it takes 530, without the B stores 25 us less.
// Every wait is bounded (f8::WAIT_NS).
#include <algorithm>
#include <cstring>

#include "corr_internal.cuh"
#include "xeng_small.cuh"

namespace corr {
namespace {

using namespace f8;

constexpr int S_SETS = 2;                 // sets of eight converter warps that take the stages in turn
constexpr int S_THREADS = 128 + 256 * S_SETS + 256;
constexpr int S_EPI_WARP = 4 + 8 * S_SETS;
constexpr int S_RAW = 6, S_OP = 3;        // ring stages: raw samples, operand tiles
constexpr int S_RAW_BYTES = 128 * KT;     // two units
constexpr int S_TILE = 128 * KT;          // one unit's operand
constexpr int S_OP_BYTES = 2 * S_TILE;
constexpr int S_OP_OFF = S_RAW * S_RAW_BYTES;
constexpr int S_BAR_OFF = S_OP_OFF + S_OP * S_OP_BYTES;
constexpr int S_SMEM = S_BAR_OFF + 512 + 1024;
constexpr int S_CONV_WARPS = 8;           // of a set
constexpr int S_A_COL = 256;               // first TMEM column of the A ring, 32 columns a unit and stage
static_assert(S_A_COL + 64 * S_OP <= 512, "TMEM columns");
static_assert(S_SMEM <= 227 * 1024, "shared memory");

struct SmallItem {
  long long p;  // unit pair
  int k0, k1;
  __device__ __forceinline__ SmallItem(const xd::Args& a, long long w, long long n_pairs) {
    const int sp = (int)(w / n_pairs);
    p = w - sp * n_pairs;
    k0 = sp * a.kps;
    k1 = min(a.n_k, k0 + a.kps);
  }
};

template <bool ADD>
__global__ void __launch_bounds__(S_THREADS, 1) xeng_small_kernel(const __grid_constant__ xd::Args args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* raw_full = reinterpret_cast<uint64_t*>(smem + S_BAR_OFF);
  uint64_t* raw_empty = raw_full + S_RAW;
  uint64_t* op_full = raw_empty + S_RAW;
  uint64_t* op_empty = op_full + S_OP;
  uint64_t* tfull = op_empty + S_OP;
  uint64_t* tempty = tfull + 1;
  uint64_t* drain = tempty + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long total = args.n_items, n_pairs = (args.n_units + 1) / 2;
  const int chunk_k = args.chunk_k;
  int* err = args.err;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S_RAW; ++s) {
      ptx::mbar_init(&raw_full[s], 1);
      ptx::mbar_init(&raw_empty[s], S_CONV_WARPS);
    }
    for (int s = 0; s < S_OP; ++s) {
      ptx::mbar_init(&op_full[s], S_CONV_WARPS);
      ptx::mbar_init(&op_empty[s], 1);
    }
    ptx::mbar_init(tfull, 1);
    ptx::mbar_init(tempty, 8);
    ptx::mbar_init(drain, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  __syncwarp();
  if (warp == 1) {
    ptx::tmem_alloc(tslot, TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tbase = *tslot;

  if (warp < 4) {
    ptx::setmaxnreg_dec<32>();
    if (warp == 0 && lane == 0) {
      // ---------------- TMA producer ----------------
      int slot = 0;
      uint32_t phase = 0, n_issued = 0;
      for (long long w = blockIdx.x; w < total && !*abort_flag; w += gridDim.x) {
        const SmallItem it(args, w, n_pairs);
        const int x = (int)(it.p * 2 * args.ub) & ~15;
        xd::StagePos p(it.k0, args.n_kb);
        for (int k = it.k0; k < it.k1; ++k, p.next(args.n_kb)) {
          if (!ptx::mbar_wait(&raw_empty[slot], phase ^ 1, WAIT_NS)) {
            record_error(err, abort_flag, 1);
            break;
          }
          ptx::mbar_arrive_expect_tx(&raw_full[slot], S_RAW_BYTES);
          ptx::tma_load_2d(smem + slot * S_RAW_BYTES, &args.map[p.blk], &raw_full[slot], x, p.kb * KT);
          ++n_issued;
          if (++slot == S_RAW) {
            slot = 0;
            phase ^= 1;
          }
        }
      }
      // copies still in flight must land before the CTA exits: the last use of every slot
      for (int s = 0; s < S_RAW; ++s) {
        const uint32_t uses = n_issued / S_RAW + ((uint32_t)s < n_issued % S_RAW ? 1u : 0u);
        if (uses > 0) ptx::mbar_wait(&raw_full[s], (uses - 1) & 1, WAIT_NS);
      }
    } else if (warp == 1 && lane == 0) {
      // ---------------- MMA issuer ----------------
      const uint32_t idesc = ptx::idesc_f8_e4m3(128, 128, 0, 0);
      // K-major, 128-byte swizzle: 8 rows x 128 samples per 1024 bytes (SBO); 32 samples on = 32 bytes
      const uint64_t desc0 = ptx::smem_desc(ptx::smem_u32(smem + S_OP_OFF), 16, 1024, 2);
      int slot = 0;
      uint32_t phase = 0, use = 0;
      bool ok = true;
      for (long long w = blockIdx.x; w < total && ok && !*abort_flag; w += gridDim.x) {
        const SmallItem it(args, w, n_pairs);
        const bool two = 2 * it.p + 1 < args.n_units;
        for (int k0 = it.k0; k0 < it.k1 && ok; k0 += chunk_k) {
          const int k1 = min(k0 + chunk_k, it.k1);
          if (!ptx::mbar_wait(tempty, (use & 1) ^ 1, WAIT_NS)) {
            record_error(err, abort_flag, 2);
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          for (int k = k0; k < k1; ++k) {
            if (!ptx::mbar_wait(&op_full[slot], phase, WAIT_NS)) {
              record_error(err, abort_flag, 3);
              ok = false;
              break;
            }
            ptx::tc_fence_after();
            const uint64_t bd = desc0 + (uint64_t)((slot * S_OP_BYTES) >> 4);
            const uint32_t at = tbase + S_A_COL + 64 * slot;
            // the units in turn: two MMAs into one accumulator wait for each other
#pragma unroll
            for (int kk = 0; kk < KT / 32; ++kk) {
              ptx::mma_f8f6f4_ts(tbase, at + 8 * kk, bd + 2 * kk, idesc, (k > k0 || kk > 0) ? 1u : 0u);
              if (two)
                ptx::mma_f8f6f4_ts(tbase + 128, at + 32 + 8 * kk, bd + (S_TILE >> 4) + 2 * kk, idesc,
                                   (k > k0 || kk > 0) ? 1u : 0u);
            }
            ptx::mma_commit(&op_empty[slot]);
            if (++slot == S_OP) {
              slot = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
          ptx::mma_commit(tfull);
          ++use;
        }
      }
      // all issued MMAs complete before TMEM is released
      ptx::mma_commit(drain);
      ptx::mbar_wait(drain, 0, WAIT_NS);
    }
  } else if (warp < S_EPI_WARP) {
    // ---------------- converters: lane quarter q of unit h, every S_SETS-th stage ----------------
    ptx::setmaxnreg_dec<56>();
    const int q = warp & 3, h = ((warp - 4) >> 2) & 1, set = (warp - 4) >> 3;
    const uint32_t raw0 = ptx::smem_u32(smem) + (uint32_t)lane * 128;
    const uint32_t a_tmem = tbase + S_A_COL + 32 * h + ((uint32_t)(32 * q) << 16);
    // B row 32 q + lane / 4 (Re; + 8, and + 16 for Im), samples 16 j + 4 (lane % 4) ..: 16-byte chunk j of the row
    const int br = lane >> 2;
    uint8_t* b_dst = smem + S_OP_OFF + h * S_TILE + (32 * q + br) * 128 + 4 * (lane & 3);
    int rs = set, os = set;
    uint32_t rph = 0, oph = 0;
    int ahead = set;  // stages until the set's next one
    bool ok = true;
    for (long long w = blockIdx.x; w < total && ok; w += gridDim.x) {
      if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
      const SmallItem it(args, w, n_pairs);
      // lane l addresses sample row l (+ 32 kk) of the 16-byte column of the quarter's inputs (128-byte swizzle)
      const int x0 = (int)(it.p * 2 * args.ub) & 15, col = ((x0 + h * args.ub) >> 4) + q, shift = (x0 + h * args.ub) & 15;
      const uint32_t a_off = raw0 + (uint32_t)((col ^ (lane & 7)) << 4);
      xd::StagePos p(it.k0 + ahead, args.n_kb);
      uint32_t sum[4] = {0u, 0u, 0u, 0u};  // Re, Im of inputs lane / 4 and lane / 4 + 8 of the quarter's 16
      for (int k = it.k0 + ahead; k < it.k1; k += S_SETS, p.next(args.n_kb, S_SETS)) {
        const int n_valid = args.T - p.kb * KT;  // samples of this stage (at most 128)
        const bool got = ptx::mbar_wait(&raw_full[rs], rph, WAIT_NS) && ptx::mbar_wait(&op_empty[os], oph ^ 1, WAIT_NS);
        // together again: the lanes leave their waits one by one, and ldmatrix and tcgen05.st are for whole warps
        if (!__all_sync(0xffffffffu, got)) {
          record_error(err, abort_flag, 5);
          ok = false;
          break;
        }
        ptx::tc_fence_after();  // the MMAs that read this A slot have completed
        const uint32_t raw = a_off + (uint32_t)(rs * S_RAW_BYTES);
        uint8_t* dst = b_dst + os * S_OP_BYTES;
        uint32_t x[16];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          ptx::ldmatrix_b8_x2_trans(raw + kk * 4096, x[4 * kk], x[4 * kk + 1], x[4 * kk + 2], x[4 * kk + 3]);
#pragma unroll
        for (int half = 0; half < 2; ++half) {  // 64 samples at a time
          uint32_t y[8], z[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            y[i] = flip_hi(x[8 * half + i]);
            z[i] = flip_lo(x[8 * half + i]);
          }
          if (n_valid < KT) {  // samples past the block: zeros
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const uint32_t m = byte_mask(n_valid - (64 * half + 16 * (i >> 1) + 4 * (lane & 3)));
              y[i] &= m;
              z[i] &= m;
            }
          }
          ptx::tmem_st_16x128b_x4(a_tmem + 64 * os + 16 * half, y);
          ptx::tmem_st_16x128b_x4(a_tmem + (16u << 16) + 64 * os + 16 * half, z);
#pragma unroll
          for (int i = 0; i < 8; ++i) {  // word 2 j + r: chunk 4 half + j, row + 8 r
            uint8_t* o = dst + (i & 1) * 1024 + (((4 * half + (i >> 1)) ^ br) << 4);
            *reinterpret_cast<uint32_t*>(o) = y[i];
            *reinterpret_cast<uint32_t*>(o + 2048) = z[i];
            sum[2 * (i & 1)] = __dp4a(y[i], 0x01010101u, sum[2 * (i & 1)]);
            sum[2 * (i & 1) + 1] = __dp4a(z[i], 0x01010101u, sum[2 * (i & 1) + 1]);
          }
        }
        ptx::tmem_st_wait();
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          ptx::mbar_arrive(&op_full[os]);
          // the stores above needed the loaded samples, so the loads are done (an arrival right behind them
          // may overtake them, and the next box would land under them)
          ptx::mbar_arrive(&raw_empty[rs]);
        }
        rs += S_SETS;
        if (rs >= S_RAW) {
          rs -= S_RAW;
          rph ^= 1;
        }
        os += S_SETS;
        if (os >= S_OP) {
          os -= S_OP;
          oph ^= 1;
        }
      }
      if (!ok) break;
      ahead = (ahead - (it.k1 - it.k0)) % S_SETS;
      if (ahead < 0) ahead += S_SETS;
      const long long u = 2 * it.p + h;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // a thread saw a quarter of at most 2^28 samples (direct_max_blocks) of at most 15
        unsigned long long s = sum[i];
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        const int in = 16 * q + br + 8 * (i >> 1) - shift;  // input row of the unit
        const int ch = in / args.ld, n = in - ch * args.ld;
        const long long f = u * args.g + ch;
        if ((lane & 3) == 0 && in >= 0 && ch < args.g && n < args.N && u < args.n_units && f < args.C) {
          const long long idx = (f * args.N + n) * 2 + (i & 1);
          atomicAdd(reinterpret_cast<unsigned long long*>(args.s1 + idx), s);
          atomicAdd(reinterpret_cast<unsigned long long*>(args.s2 + idx), s);
        }
      }
    }
  } else {
    // ---------------- epilogue: lane quarter q of unit h ----------------
    ptx::setmaxnreg_inc<120>();
    const int q = warp & 3, h = (warp - S_EPI_WARP) >> 2;
    const bool im_lane = (lane & 16) != 0;
    const int lp = args.npol >> 1;
    uint32_t use = 0;
    bool ok = true;
    for (long long w = blockIdx.x; w < total && ok; w += gridDim.x) {
      const SmallItem it(args, w, n_pairs);
      const long long u = 2 * it.p + h;
      const int shift = (int)(u * args.ub) & 15;
      const int ic = 16 * q + (lane & 15) - shift;  // c-input of the unit
      const int ch = ic / args.ld, c = ic - ch * args.ld;
      // the chunks (16 a-inputs) that hold this warp's channels, from the diagonal on
      const int last = min(64, ((16 * q + 15 - shift) / args.ld + 1) * args.ld + shift);
      const int cc_end = (last + 15) / 16;
      const long long f = u * args.g + ch;
      const bool live = ic >= 0 && ch < args.g && u < args.n_units && f < args.C;
      long long* cross_f = args.cross + (live ? f : 0) * args.Bs * args.npol * args.npol * 2;
      long long* autos_f = args.autos + (live ? f : 0) * args.N;
      for (int k0 = it.k0; k0 < it.k1; k0 += chunk_k) {
        if (__any_sync(0xffffffffu, *abort_flag != 0)) {
          ok = false;
          break;
        }
        const bool got = ptx::mbar_wait(tfull, use & 1, WAIT_NS);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) record_error(err, abort_flag, 4);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint32_t t = tbase + 128 * h + ((uint32_t)(32 * q) << 16);
        int re[4][8], im[4][8];
#pragma unroll
        for (int j = 0; j < 2; ++j) {  // two chunks at a time
          uint32_t v[2][32];
          ptx::tmem_ld_32x32b_x32(t + 64 * j, v[0]);
          ptx::tmem_ld_32x32b_x32(t + 64 * j + 32, v[1]);
          ptx::tmem_ld_wait();
          xd::combine_chunk(v[0], im_lane, re[2 * j], im[2 * j]);
          xd::combine_chunk(v[1], im_lane, re[2 * j + 1], im[2 * j + 1]);
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(tempty);
        ++use;
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
          if (u < args.n_units && cc >= q && cc < cc_end)
            xd::add_chunk<ADD>(re[cc], im[cc], im_lane, live ? c : -1, 16 * cc - shift - ch * args.ld, args.N, lp, cross_f, autos_f);
      }
    }
  }
  __syncwarp();  // the roles ran on single lanes: what follows is for whole warps
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  if (warp == 1) ptx::tmem_dealloc(tbase, TMEM_COLS);
}

// Channels (of ld stored inputs) per 64-input unit: as many as fit behind the inputs that a unit's first 16-byte
// column may hold of the one before (16 - gcd(16, unit) at most); 0 if not even one does.
int small_group(int ld) {
  for (int g = 64 / ld; g >= 1; --g)
    if (g * ld + ((16 - (g * ld & -(g * ld))) & 15) <= 64) return g;
  return 0;
}

// Items' stages are divided where whole items leave SMs idle: the division of n_k stages that minimises waves x (stages
// + overhead), `slots` items running at once.
int direct_splits(long long items, int slots, int n_k, int overhead) {
  int best = 1;
  double best_t = 1e300;
  for (int s = 1; s <= n_k && s <= 256; ++s) {
    const int kps = (n_k + s - 1) / s;
    if ((n_k + kps - 1) / kps != s) continue;  // the same division as a smaller s
    const double waves = (double)((items * s + slots - 1) / slots);
    const double t = waves * (kps + overhead + (s > 1 ? 1 : 0));
    if (t < 0.97 * best_t) {
      best = s;
      best_t = t;
    }
    if (items * s >= 8LL * slots) break;
  }
  return best;
}

cudaError_t direct_args(const DirectJob& j, xd::Args* a) {
  std::memset(a, 0, sizeof(*a));
  if (j.n > xd::MAX_BLOCKS) return cudaErrorInvalidValue;
  for (int b = 0; b < j.n; ++b) {
    std::string err;
    if (encode_raw_tensor_map(&a->map[b], j.blocks[b], (long long)j.s.C * j.ld, j.T_blk, &err) != 0) {
      set_last_error(err);
      return cudaErrorInvalidValue;
    }
  }
  a->cross = j.cross;
  a->autos = j.autos;
  a->s1 = j.s1;
  a->s2 = j.s2;
  a->Bs = j.s.Bs;
  a->N = j.s.N;
  a->ld = j.ld;
  a->C = j.s.C;
  a->npol = j.s.npol;
  a->T = j.T_blk;
  a->n_kb = (j.T_blk + KT - 1) / KT;
  a->n_k = a->n_kb * j.n;
  a->chunk_k = j.flush_len / KT;
  a->err = j.err;
  return cudaSuccess;
}

}  // namespace

bool xeng_small_supported(const Shape& s, int ld, const void* d_in) {
  const long long row = (long long)ld * s.C;
  return s.N <= 64 && small_group(ld) > 0 && row % 16 == 0 && row < (1LL << 31) && reinterpret_cast<uintptr_t>(d_in) % 16 == 0;
}

cudaError_t launch_xeng_small(const DirectJob& j, int num_sms, cudaStream_t st) {
  if (j.n == 0 || j.T_blk == 0) return cudaSuccess;
  xd::Args a;
  cudaError_t e = direct_args(j, &a);
  if (e != cudaSuccess) return e;
  a.g = small_group(j.ld);
  a.ub = a.g * j.ld;
  a.n_units = (j.s.C + a.g - 1) / a.g;
  const long long pairs = (a.n_units + 1) / 2;
  a.splits = direct_splits(pairs, num_sms, a.n_k, 4);
  a.kps = (a.n_k + a.splits - 1) / a.splits;
  a.n_items = pairs * a.splits;
  const unsigned grid = (unsigned)std::min<long long>(num_sms, a.n_items);
  e = set_smem_limit(a.splits > 1 ? reinterpret_cast<const void*>(xeng_small_kernel<true>)
                                  : reinterpret_cast<const void*>(xeng_small_kernel<false>), S_SMEM);
  if (e != cudaSuccess) return e;
  if (a.splits > 1)
    xeng_small_kernel<true><<<grid, S_THREADS, S_SMEM, st>>>(a);
  else
    xeng_small_kernel<false><<<grid, S_THREADS, S_SMEM, st>>>(a);
  return cudaGetLastError();
}

}  // namespace corr
