// X-engine on pairs of SMs that builds its operand on the chip: tcgen05.mma.cta_group::2 (kind::f8f6f4, M =
// 256, N = 256, K = 32) with A in TMEM and B in shared memory, both made from the packed 4+4-bit samples
// that TMA brings in. Nothing but the samples and the int64 sums crosses HBM (the two-pass path writes
// two operand bytes a sample and reads them back). For more than 64 inputs.
//
// Work item = (channel, 128 c-inputs C0 .., 128 a-inputs A0 >= C0, a range of stages). CTA rank r of the
// pair holds the c-side rows of inputs C0 + 64 r .. + 63 (A, its 128 TMEM lanes) and the a-side rows of
// inputs A0 + 64 r .. + 63 (half of B); its TMEM gets its c-side rows times all 256 a-side rows.
//
// A stage is 128 samples: 8 KB of samples a side, fetched as boxes of 64 bytes x 128 samples (64-byte
// swizzle, so that both readers below touch all banks).
//   A: rows are TMEM lanes and samples run along the columns, i.e. the samples are needed transposed.
//      ldmatrix.trans.b8 transposes 16 inputs x 16 samples on the way into the registers, as four samples
//      of an input a word; a shift and two logic operations split and flip the nibbles, and the fragment
//      is tcgen05.st's 16x128b shape as it stands. Lanes 32 q .. + 15 of a quarter are Re of 16 inputs,
//      + 16 .. + 31 Im of the same.
//   B: a thread turns 16 samples of one time (16 bytes) into 32 operand bytes of the MN-major, 128-byte
//      swizzled tile, row groups of 4 Re and 4 Im.
// Why A in TMEM: with both operands in shared memory a stage moves 48 KB through the load/store path in the
// 512 clocks of its MMAs; so it is 32 KB, and the MMAs read only B from shared memory.
//
// Rows of any length: a TMA box starts on a 16-byte boundary, so channel f's tiles start at the boundary at or
// below its first byte, (f N) mod 16 inputs before input 0. Both sides are shifted alike; the rows that belong
// to the neighbouring channel give products that the epilogue leaves out, as it does those past N.
//
// Roles: warp 0 TMA producer; warp 1 TMEM allocation and, in the even CTA, the MMA issuer; warps 4-11
// converters (two sets of four warps, one TMEM lane quarter each, that take the stages in turn); warps
// 12-19 epilogue. The accumulator takes 256 of the 512 columns and the A ring 192, so there is one
// accumulator: the epilogue takes all of it into registers, combined to complex products on the way (64 a
// thread), before it adds to the int64 sums, and the MMAs wait for those loads only, about 1000 clocks an
// item. The register file is split by setmaxnreg: 128 x 24 + 256 x 80 + 256 x 144 of the 640 x 96 of the
// launch. (80 and 144, 512 inputs x 109 channels x 8000 samples: 388 us; 88 and 136: 393, 96 and 128: 397.)
//
// What bounds it: 512 inputs x 128 channels x 4 blocks of 8192 samples take 1.60 ms a launch (the two passes:
// 1.245 + 4 x 0.253), 370 ns a stage. The MMAs alone need 62 x 4, with every barrier and copy but no conversion
// the stage takes 311; the rest is the converters' shared-memory traffic beside the MMAs' operand reads: without
// the ldmatrix 340, without the B stores 332. A third set of converter warps, separate A and B warps and other
// ring depths (5 + 8, 6 + 7) measured the same or slower.
//
// Offset sums: diagonal items (C0 == A0) see every input once; their A converters add up each word's four
// samples with dp4a.
// Every wait is bounded (f8::WAIT_NS); a timeout sets the error word and both CTAs' abort flags.
#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>

#include "corr_internal.cuh"
#include "xeng_direct.cuh"

namespace corr {
namespace {

using namespace f8;

constexpr int D_SETS = 2;                // sets of four converter warps
constexpr int D_THREADS = 128 + 128 * D_SETS + 256;
constexpr int D_EPI_WARP = 4 + 4 * D_SETS;  // first epilogue warp
constexpr int D_RAW = 7, D_OP = 6;       // ring stages: raw samples; operands (A in TMEM, B in shared memory)
constexpr int D_BOX = 64 * KT;           // raw bytes of one side and stage
constexpr int D_RAW_BYTES = 2 * D_BOX;
constexpr int D_A_COL = 256;             // first TMEM column of the A ring, 32 columns a stage
constexpr int D_OP_OFF = D_RAW * D_RAW_BYTES;
constexpr int D_BAR_OFF = D_OP_OFF + D_OP * B_ATOM;
constexpr int D_SMEM = D_BAR_OFF + 512 + 1024;
constexpr int D_EPI_WARPS = 8;
static_assert(D_A_COL + 32 * D_OP <= 512, "TMEM columns");
static_assert(D_SMEM <= 227 * 1024, "shared memory");

__device__ __forceinline__ void direct_error(int* err, volatile int* abort_flag, uint32_t peer_abort, int code) {
  *abort_flag = 1;
  ptx::st_shared_cluster_u32(peer_abort, 1u);
  atomicCAS(err, 0, code);
}

// Inputs of the channel before that the first tile of channel f starts with.
__device__ __forceinline__ int tile_shift(const xd::Args& a, int f) { return (int)((unsigned)f * (unsigned)a.ld & 15u); }

struct Item {
  int f, c0, a0, k0, k1;  // c0, a0: rows of the channel's tiles
  // From tile rows to inputs, -15 .. N - 1.
  __device__ __forceinline__ void to_inputs(const xd::Args& a) {
    const int shift = tile_shift(a, f);
    c0 -= shift;
    a0 -= shift;
  }
  __device__ __forceinline__ Item(const xd::Args& a, long long w) {
    int t = (int)(w % a.n_tiles);
    const long long r = w / a.n_tiles;
    const int sp = (int)(r % a.splits);
    f = (int)(r / a.splits);
    int ci = 0;
    while (t >= a.nb - ci) {
      t -= a.nb - ci;
      ++ci;
    }
    c0 = 128 * ci;
    a0 = 128 * (ci + t);
    k0 = sp * a.kps;
    k1 = min(a.n_k, k0 + a.kps);
  }
};

// The item's cells of this CTA into L2 while its MMAs run: for each a-station one run of the 64 c-inputs' products,
// so that the loads of the old sums wait for L2 and not for DRAM. Short integrations are bound by the epilogue:
// 512 inputs x 2400 channels x 240 samples 2.63 ms without the prefetch, 2.44 with it; x 109 x 8000 397 and 389 us.
__device__ __forceinline__ void prefetch_cells(const xd::Args& a, const Item& it, uint32_t rank, int w, int lane, int lp,
                                               const long long* cross_f) {
  const int c0 = (it.c0 + 64 * (int)rank) >> lp, sc0 = max(c0, 0), S = a.N >> lp;
  for (int i = 32 * w + lane; i < 128 >> lp; i += 32 * D_EPI_WARPS) {
    const int sa = (it.a0 >> lp) + i;
    const int end = min(min(c0 + (64 >> lp), sa + 1), S);
    if (sa < S && sc0 < end) {
      const unsigned b = (unsigned)sa * (unsigned)(sa + 1) / 2 + (unsigned)sc0;
      ptx::prefetch_l2(cross_f + 2 * ((long long)b << (2 * lp)), (uint32_t)(end - sc0) << (4 + 2 * lp));
    }
  }
}

template <bool ADD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(D_THREADS, 1)
    xeng_direct_kernel(const __grid_constant__ xd::Args args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* raw_full = reinterpret_cast<uint64_t*>(smem + D_BAR_OFF);
  uint64_t* raw_empty = raw_full + D_RAW;
  uint64_t* op_full = raw_empty + D_RAW;
  uint64_t* op_empty = op_full + D_OP;
  uint64_t* tfull = op_empty + D_OP;
  uint64_t* tempty = tfull + 1;
  uint64_t* drain = tempty + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const bool leader = rank == 0;
  const long long pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const long long total = args.n_items;
  const int chunk_k = args.chunk_k;
  int* err = args.err;

  if (threadIdx.x == 0) {
    for (int s = 0; s < D_RAW; ++s) {
      ptx::mbar_init(&raw_full[s], 1);
      ptx::mbar_init(&raw_empty[s], 4);  // the warps of the converter set that read the stage
    }
    for (int s = 0; s < D_OP; ++s) {
      ptx::mbar_init(&op_full[s], 8);    // four converter warps of each CTA (the even CTA's barrier is used)
      ptx::mbar_init(&op_empty[s], 1);   // the pair's commit
    }
    ptx::mbar_init(tfull, 1);
    ptx::mbar_init(tempty, 2 * D_EPI_WARPS);
    ptx::mbar_init(drain, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(tslot, TMEM_COLS);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // both CTAs' barriers initialised before any remote arrival
  ptx::tc_fence_after();
  const uint32_t tbase = *tslot;
  const uint32_t peer_abort = ptx::mapa_shared(const_cast<int*>(abort_flag), rank ^ 1u);

  if (warp < 4) {
    ptx::setmaxnreg_dec<24>();
    if (warp == 0 && lane == 0) {
      // ---------------- TMA producer (both CTAs) ----------------
      int slot = 0;
      uint32_t phase = 0, n_issued = 0;
      for (long long w = pair; w < total && !*abort_flag; w += n_pairs) {
        Item it(args, w);
        it.to_inputs(args);
        const int xc = it.f * args.ld + it.c0 + 64 * (int)rank, xa = it.f * args.ld + it.a0 + 64 * (int)rank;
        const bool diag = it.c0 == it.a0;  // A and B are of the same inputs: one box
        xd::StagePos p(it.k0, args.n_kb);
        for (int k = it.k0; k < it.k1; ++k, p.next(args.n_kb)) {
          if (!ptx::mbar_wait(&raw_empty[slot], phase ^ 1, WAIT_NS)) {
            direct_error(err, abort_flag, peer_abort, 1);
            break;
          }
          uint8_t* dst = smem + slot * D_RAW_BYTES;
          ptx::mbar_arrive_expect_tx(&raw_full[slot], diag ? D_BOX : D_RAW_BYTES);
          ptx::tma_load_2d(dst, &args.map[p.blk], &raw_full[slot], xc, p.kb * KT);
          if (!diag) ptx::tma_load_2d(dst + D_BOX, &args.map[p.blk], &raw_full[slot], xa, p.kb * KT);
          ++n_issued;
          if (++slot == D_RAW) {
            slot = 0;
            phase ^= 1;
          }
        }
      }
      // copies still in flight must land before the CTA exits: the last use of every slot
      for (int s = 0; s < D_RAW; ++s) {
        const uint32_t uses = n_issued / D_RAW + ((uint32_t)s < n_issued % D_RAW ? 1u : 0u);
        if (uses > 0) ptx::mbar_wait(&raw_full[s], (uses - 1) & 1, WAIT_NS);
      }
    } else if (warp == 1 && lane == 0) {
      if (leader) {
        // ---------------- MMA issuer (even CTA) ----------------
        const uint32_t idesc = ptx::idesc_f8_e4m3(256, 256, 0, 1);
        const uint64_t b_desc0 = ptx::smem_desc(ptx::smem_u32(smem + D_OP_OFF), B_ATOM, 1024, 2);
        int slot = 0;
        uint32_t phase = 0, use = 0;
        bool ok = true;
        for (long long w = pair; w < total && ok && !*abort_flag; w += n_pairs) {
          const Item it(args, w);
          for (int k0 = it.k0; k0 < it.k1 && ok; k0 += chunk_k) {
            const int k1 = min(k0 + chunk_k, it.k1);
            if (!ptx::mbar_wait(tempty, (use & 1) ^ 1, WAIT_NS)) {
              direct_error(err, abort_flag, peer_abort, 2);
              ok = false;
              break;
            }
            ptx::tc_fence_after();
            for (int k = k0; k < k1; ++k) {
              if (!ptx::mbar_wait(&op_full[slot], phase, WAIT_NS)) {
                direct_error(err, abort_flag, peer_abort, 3);
                ok = false;
                break;
              }
              ptx::tc_fence_after();
              const uint64_t b_desc = b_desc0 + (uint64_t)((slot * B_ATOM) >> 4);
              const uint32_t a_tmem = tbase + D_A_COL + 32 * slot;
#pragma unroll
              for (int kk = 0; kk < KT / 32; ++kk)
                ptx::mma_f8f6f4_pair_ts(tbase, a_tmem + 8 * kk, b_desc + kk * 256, idesc, (k > k0 || kk > 0) ? 1u : 0u);
              ptx::mma_commit_pair(&op_empty[slot], 3);
              if (++slot == D_OP) {
                slot = 0;
                phase ^= 1;
              }
            }
            if (!ok) break;
            ptx::mma_commit_pair(tfull, 3);
            ++use;
          }
        }
        // all issued MMAs (into both CTAs' TMEM) complete before either CTA releases it
        ptx::mma_commit_pair(drain, 3);
        ptx::mbar_wait(drain, 0, WAIT_NS);
      } else {
        ptx::mbar_wait(drain, 0, WAIT_NS);  // odd CTA: the even CTA's last commit
      }
    }
  } else if (warp < D_EPI_WARP) {
    // ---------------- converters ----------------
    ptx::setmaxnreg_dec<80>();
    const int q = warp & 3, set = (warp - 4) >> 2;
    const uint32_t raw0 = ptx::smem_u32(smem);
    // A: lane l addresses sample row l (+ 32 kk) of the warp's 16-byte column of inputs
    const uint32_t a_off = (uint32_t)lane * 64 + (uint32_t)((q ^ ((lane >> 1) & 3)) << 4);
    const uint32_t a_tmem = tbase + D_A_COL + ((uint32_t)(32 * q) << 16);
    // B: lane -> 16-byte column c, sample rows 32 q + 8 i + kr
    const int c = lane & 3, kr = lane >> 2;
    const uint32_t b_off = (uint32_t)(32 * q + kr) * 64 + (uint32_t)((c ^ ((kr >> 1) & 3)) << 4);
    const uint32_t o_off = (uint32_t)D_OP_OFF + (uint32_t)(4 * q) * 1024 + (uint32_t)kr * 128;
    const uint32_t o0_off = o_off + (uint32_t)(((2 * c) ^ kr) << 4), o1_off = o_off + (uint32_t)(((2 * c + 1) ^ kr) << 4);
    int rs = set, os = set;
    uint32_t rph = 0, oph = 0;
    int ahead = set;  // stages until the set's next one (the sets take the CTA's stages in turn)
    bool ok = true;
    for (long long w = pair; w < total && ok && !*abort_flag; w += n_pairs) {
      const Item it(args, w);
      const bool diag = it.c0 == it.a0;
      uint32_t sum[4] = {0u, 0u, 0u, 0u};  // Re, Im of inputs lane / 4 and lane / 4 + 8 of the quarter's 16
      const int kfirst = it.k0 + ahead;
      xd::StagePos p(kfirst, args.n_kb);
      for (int k = kfirst; k < it.k1; k += D_SETS, p.next(args.n_kb, D_SETS)) {
        const int n_valid = min(KT, args.T - p.kb * KT);  // samples of this stage
        if (!ptx::mbar_wait(&raw_full[rs], rph, WAIT_NS) || !ptx::mbar_wait(&op_empty[os], oph ^ 1, WAIT_NS)) {
          direct_error(err, abort_flag, peer_abort, 5);
          ok = false;
          break;
        }
        ptx::tc_fence_after();  // the MMAs that read this A slot have completed
        const uint32_t raw = raw0 + (uint32_t)(rs * D_RAW_BYTES);
        // all loads first
        uint32_t x[16];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          ptx::ldmatrix_b8_x2_trans(raw + a_off + kk * 2048, x[4 * kk], x[4 * kk + 1], x[4 * kk + 2], x[4 * kk + 3]);
        const uint8_t* b_src = smem + rs * D_RAW_BYTES + (diag ? 0 : D_BOX) + b_off;
        uint4 r[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) r[i] = *reinterpret_cast<const uint4*>(b_src + i * 512);
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // 64 samples at a time
          uint32_t y[8], z[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = flip_hi(x[8 * h + i]);
          ptx::tmem_st_16x128b_x4(a_tmem + 32 * os + 16 * h, y);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[i] = flip_lo(x[8 * h + i]);
          ptx::tmem_st_16x128b_x4(a_tmem + (16u << 16) + 32 * os + 16 * h, z);
          if (diag) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              sum[2 * (i & 1)] = __dp4a(y[i], 0x01010101u, sum[2 * (i & 1)]);
              sum[2 * (i & 1) + 1] = __dp4a(z[i], 0x01010101u, sum[2 * (i & 1) + 1]);
            }
          }
        }
        if (n_valid < KT) {
          // samples past the block read as 0, i.e. offset 8: out of the sums, and B rows of zeros
          if ((lane & 3) == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[i] -= 8u * (uint32_t)(KT - n_valid);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (32 * q + 8 * i + kr >= n_valid) r[i] = make_uint4(0x88888888u, 0x88888888u, 0x88888888u, 0x88888888u);
        }
        uint8_t* b_dst = smem + os * B_ATOM;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          *reinterpret_cast<uint4*>(b_dst + o0_off + i * 1024) =
              make_uint4(flip_hi(r[i].x), flip_lo(r[i].x), flip_hi(r[i].y), flip_lo(r[i].y));
          *reinterpret_cast<uint4*>(b_dst + o1_off + i * 1024) =
              make_uint4(flip_hi(r[i].z), flip_lo(r[i].z), flip_hi(r[i].w), flip_lo(r[i].w));
        }
        ptx::tmem_st_wait();
        ptx::fence_proxy_async_smem();
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          ptx::mbar_arrive_remote(ptx::mapa_shared(&op_full[os], 0));
          // the stores above needed the loaded samples, so the loads are done (an arrival right behind them
          // may overtake them, and the next box would land under them)
          ptx::mbar_arrive(&raw_empty[rs]);
        }
        rs += D_SETS;
        if (rs >= D_RAW) {
          rs -= D_RAW;
          rph ^= 1;
        }
        os += D_SETS;
        if (os >= D_OP) {
          os -= D_OP;
          oph ^= 1;
        }
      }
      ahead = (ahead - (it.k1 - it.k0)) % D_SETS;
      if (ahead < 0) ahead += D_SETS;
      if (diag && ok) {
        // anew, not from `it`: the shift kept over the loop above slows the conversion down (1.640 ms a launch, 1.620)
        long long wl = w;
        asm volatile("" : "+l"(wl));
        Item d(args, wl);
        d.to_inputs(args);
        unsigned long long s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // a thread saw at most 2^28 / 8 samples (launch_xeng_direct), its last stages' correction included
          s[i] = (unsigned long long)(long long)(int)sum[i];
          s[i] += __shfl_xor_sync(0xffffffffu, s[i], 1);
          s[i] += __shfl_xor_sync(0xffffffffu, s[i], 2);
        }
        if ((lane & 3) == 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int n = d.c0 + 64 * (int)rank + 16 * q + (lane >> 2) + 8 * (i >> 1);
            if (n >= 0 && n < args.N && s[i] != 0) {
              const long long idx = ((long long)d.f * args.N + n) * 2 + (i & 1);
              atomicAdd(reinterpret_cast<unsigned long long*>(args.s1 + idx), s[i]);
              atomicAdd(reinterpret_cast<unsigned long long*>(args.s2 + idx), s[i]);
            }
          }
        }
      }
    }
  } else {
    // ---------------- epilogue (both CTAs) ----------------
    ptx::setmaxnreg_inc<144>();
    const int q = warp & 3, half = (warp - D_EPI_WARP) >> 2;  // lane quarter; a-inputs 64 half .. + 63
    const bool im_lane = (lane & 16) != 0;
    const int lp = args.npol >> 1;
    uint32_t use = 0;
    bool ok = true;
    for (long long w = pair; w < total && ok; w += n_pairs) {
      Item it(args, w);
      it.to_inputs(args);
      const int c = it.c0 + 64 * (int)rank + 16 * q + (lane & 15);
      long long* cross_f = args.cross + (long long)it.f * args.Bs * args.npol * args.npol * 2;
      long long* autos_f = args.autos + (long long)it.f * args.N;
      prefetch_cells(args, it, rank, warp - 12, lane, lp, cross_f);
      for (int k0 = it.k0; k0 < it.k1; k0 += chunk_k) {
        if (__any_sync(0xffffffffu, *abort_flag != 0)) {
          ok = false;
          break;
        }
        const bool got = ptx::mbar_wait(tfull, use & 1, WAIT_NS);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) direct_error(err, abort_flag, peer_abort, 4);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        int re[4][8], im[4][8];
        const uint32_t t = tbase + ((uint32_t)(32 * q) << 16) + 128 * half;
#pragma unroll
        for (int j = 0; j < 4; j += 2) {  // all four at once: 128 words, and spills
          uint32_t v[2][32];
          ptx::tmem_ld_32x32b_x32(t + 32 * j, v[0]);
          ptx::tmem_ld_32x32b_x32(t + 32 * j + 32, v[1]);
          ptx::tmem_ld_wait();
          xd::combine_chunk<16>(v[0], im_lane, re[j], im[j]);
          xd::combine_chunk<16>(v[1], im_lane, re[j + 1], im[j + 1]);
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_remote(ptx::mapa_shared(tempty, 0));
        ++use;
        const int c_min = it.c0 + 64 * (int)rank + 16 * q, c_max = c_min + 15;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int a_base = it.a0 + 64 * half + 16 * j;
          if (lp == 1 && c_min >= 0 && a_base > c_max && a_base + 16 <= args.N)
            xd::add_chunk_full<ADD>(re[j], im[j], im_lane, c, a_base, cross_f);
          else if (a_base + 15 >= c_min - lp && a_base < args.N && c_min < args.N)  // not all above the diagonal or past N
            xd::add_chunk<ADD>(re[j], im[j], im_lane, c, a_base, args.N, lp, cross_f, autos_f);
        }
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // no CTA leaves while its peer may still signal its barriers or read its operands
  ptx::tc_fence_after();
  if (warp == 1) ptx::tmem_dealloc_pair(tbase, TMEM_COLS);
}

// Clusters of this kernel that fit on the device at once (cached per device).
int direct_max_pairs() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  const auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2 * (unsigned)sm_count(), 1, 1);
  cfg.blockDim = dim3(D_THREADS, 1, 1);
  cfg.dynamicSmemBytes = D_SMEM;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, xeng_direct_kernel<false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  cache[dev] = n;
  return n;
}

}  // namespace

// Whole rows of 16 bytes (TMA's stride). Where channels start between 16-byte boundaries the first tile holds up to
// 16 - gcd(N, 16) inputs of the channel before; that may not take one more row of tiles (repack.cu takes those).
bool xeng_direct_supported(const Shape& s, int ld, const void* d_in) {
  const long long row = (long long)ld * s.C;
  const int shift = (16 - (ld & -ld)) & 15;  // the largest of any channel
  return s.N > 64 && row % 16 == 0 && reinterpret_cast<uintptr_t>(d_in) % 16 == 0 && row < (1LL << 31) &&
         (s.N + shift + 127) / 128 == (s.N + 127) / 128;
}

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

cudaError_t direct_args(const DirectJob& j, int box_bytes, xd::Args* a) {
  std::memset(a, 0, sizeof(*a));
  if (j.n > xd::MAX_BLOCKS) return cudaErrorInvalidValue;
  for (int b = 0; b < j.n; ++b) {
    std::string err;
    if (encode_raw_tensor_map(&a->map[b], j.blocks[b], (long long)j.s.C * j.ld, j.T_blk, box_bytes, &err) != 0) {
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

cudaError_t launch_xeng_direct(const DirectJob& j, int num_sms, cudaStream_t st) {
  if (j.n == 0 || j.T_blk == 0) return cudaSuccess;
  xd::Args a;
  cudaError_t e = direct_args(j, 64, &a);
  if (e == cudaSuccess) e = set_smem_limit(reinterpret_cast<const void*>(xeng_direct_kernel<false>), D_SMEM);
  if (e != cudaSuccess) return e;
  int pairs = std::max(1, num_sms / 2);
  const int fit = direct_max_pairs();
  if (fit > 0) pairs = std::min(pairs, fit);
  a.nb = (j.s.N + 127) / 128;
  a.n_tiles = a.nb * (a.nb + 1) / 2;
  const long long items = (long long)a.n_tiles * j.s.C;
  // an item's fixed cost (ring start, drain) is about six stages' time
  a.splits = direct_splits(items, pairs, a.n_k, 6);
  a.kps = (a.n_k + a.splits - 1) / a.splits;
  a.n_items = items * a.splits;
  const unsigned grid = 2u * (unsigned)std::min<long long>(pairs, a.n_items);
  if (a.splits > 1) {
    e = set_smem_limit(reinterpret_cast<const void*>(xeng_direct_kernel<true>), D_SMEM);
    if (e != cudaSuccess) return e;
    xeng_direct_kernel<true><<<grid, D_THREADS, D_SMEM, st>>>(a);
  } else {
    xeng_direct_kernel<false><<<grid, D_THREADS, D_SMEM, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace corr
