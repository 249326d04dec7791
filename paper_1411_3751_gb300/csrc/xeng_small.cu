// X-engine for arrays of at most 64 inputs that builds its operand on the chip: tcgen05.mma (kind::f8f6f4, M = N
// = 128, K = 32) of a 64-input tile with itself, the tile made in shared memory from the packed samples
// that TMA brings in. HBM-bound: the samples are read once (the two-pass path wrote two operand bytes a
// sample and read them back, five times the traffic).
//
// A unit is 64 neighbouring sample bytes of a time, the MMA's 128 operand rows: one channel of up to 64
// inputs, or g channels of N inputs with g N <= 64 (their products are the diagonal blocks; those across
// channels are not used). With 33 to 63 inputs the unit runs into the next channel, whose rows are not
// used either. An item is two neighbouring units, so that TMA boxes are 128 bytes x 128 samples, and a
// range of stages of 128 samples.
//
// Roles (one CTA per SM): warp 0 TMA producer; warp 1 TMEM allocation and MMA issuer (each unit has two of
// the four 128-column accumulators); warps 2-9 converters: 16 bytes of one time -> 32 operand bytes of the
// MN-major, 128-byte swizzled tile, and the inputs' offset sums; warps 10-17 epilogue, four a unit.
// Every wait is bounded (f8::WAIT_NS).
#include <algorithm>
#include <cstring>

#include "corr_internal.cuh"
#include "xeng_direct.cuh"

namespace corr {
namespace {

using namespace f8;

constexpr int S_THREADS = 576;
constexpr int S_RAW = 6, S_OP = 3;        // ring stages: raw samples, operand tiles
constexpr int S_RAW_BYTES = 128 * KT;     // two units
constexpr int S_TILE = 128 * KT;          // one unit's operand
constexpr int S_OP_BYTES = 2 * S_TILE;
constexpr int S_OP_OFF = S_RAW * S_RAW_BYTES;
constexpr int S_BAR_OFF = S_OP_OFF + S_OP * S_OP_BYTES;
constexpr int S_SMEM = S_BAR_OFF + 512 + 1024;
constexpr int S_CONV_WARPS = 8;
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
  uint64_t* tfull = op_empty + S_OP;  // [2]
  uint64_t* tempty = tfull + 2;       // [2]
  uint64_t* drain = tempty + 2;
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
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], 8);
    }
    ptx::mbar_init(drain, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(tslot, TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tbase = *tslot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      int slot = 0;
      uint32_t phase = 0, n_issued = 0;
      for (long long w = blockIdx.x; w < total && !*abort_flag; w += gridDim.x) {
        const SmallItem it(args, w, n_pairs);
        const int x = (int)(it.p * 2 * args.ub);
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
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      const uint32_t idesc = ptx::idesc_f8_e4m3(128, 128, 1, 1);
      const uint64_t desc0 = ptx::smem_desc(ptx::smem_u32(smem + S_OP_OFF), 16, 1024, 2);
      int slot = 0, acc = 0;
      uint32_t phase = 0, use[2] = {0u, 0u};
      bool ok = true;
      for (long long w = blockIdx.x; w < total && ok && !*abort_flag; w += gridDim.x) {
        const SmallItem it(args, w, n_pairs);
        const bool two = 2 * it.p + 1 < args.n_units;
        for (int k0 = it.k0; k0 < it.k1 && ok; k0 += chunk_k) {
          const int k1 = min(k0 + chunk_k, it.k1);
          if (!ptx::mbar_wait(&tempty[acc], (use[acc] & 1) ^ 1, WAIT_NS)) {
            record_error(err, abort_flag, 2);
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          const uint32_t d = tbase + 256 * acc;
          for (int k = k0; k < k1; ++k) {
            if (!ptx::mbar_wait(&op_full[slot], phase, WAIT_NS)) {
              record_error(err, abort_flag, 3);
              ok = false;
              break;
            }
            ptx::tc_fence_after();
            const uint64_t dd = desc0 + (uint64_t)((slot * S_OP_BYTES) >> 4);
#pragma unroll
            for (int kk = 0; kk < KT / 32; ++kk) ptx::mma_f8f6f4(d, dd + kk * 256, dd + kk * 256, idesc, (k > k0 || kk > 0) ? 1u : 0u);
            if (two) {
              const uint64_t d2 = dd + (S_TILE >> 4);
#pragma unroll
              for (int kk = 0; kk < KT / 32; ++kk)
                ptx::mma_f8f6f4(d + 128, d2 + kk * 256, d2 + kk * 256, idesc, (k > k0 || kk > 0) ? 1u : 0u);
            }
            ptx::mma_commit(&op_empty[slot]);
            if (++slot == S_OP) {
              slot = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
          ptx::mma_commit(&tfull[acc]);
          ++use[acc];
          acc ^= 1;
        }
      }
      // all issued MMAs complete before TMEM is released
      ptx::mma_commit(drain);
      ptx::mbar_wait(drain, 0, WAIT_NS);
    }
  } else if (warp < 2 + S_CONV_WARPS) {
    // ---------------- converters ----------------
    // Lane -> 16-byte column c of unit h, sample rows: eight neighbouring lanes read four columns of unit 0
    // and, a row on, of unit 1, which touches every bank (as the swizzled stores do); in the second
    // phase of a step the rows swap.
    const int cw = warp - 2;
    const int c = lane & 3, h = (lane >> 2) & 1, pr = lane >> 3;  // row pairs 8 i + pr ... of the warp's 16 rows
    const uint32_t r_col = (uint32_t)(16 * c + h * args.ub);
    int rs = 0, os = 0;
    uint32_t rph = 0, oph = 0;
    bool ok = true;
    for (long long w = blockIdx.x; w < total && ok; w += gridDim.x) {
      const SmallItem it(args, w, n_pairs);
      xd::StagePos p(it.k0, args.n_kb);
      for (int k0 = it.k0; k0 < it.k1 && ok; k0 += chunk_k) {
        const int k1 = min(k0 + chunk_k, it.k1);
        // packed sums of the thread's 16 inputs: bytes over a stage's 4 samples, 16-bit lanes over the chunk
        // (at most 15 x 4 x 512 stages)
        uint32_t sre[4][2] = {{0u, 0u}, {0u, 0u}, {0u, 0u}, {0u, 0u}};
        uint32_t sim[4][2] = {{0u, 0u}, {0u, 0u}, {0u, 0u}, {0u, 0u}};
        for (int k = k0; k < k1; ++k, p.next(args.n_kb)) {
          if (*abort_flag) {
            ok = false;
            break;
          }
          const int n_valid = min(KT, args.T - p.kb * KT);
          if (!ptx::mbar_wait(&raw_full[rs], rph, WAIT_NS)) {
            record_error(err, abort_flag, 5);
            ok = false;
            break;
          }
          const uint8_t* src = smem + rs * S_RAW_BYTES + r_col;
          uint4 r[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {  // step i >> 1, phase i & 1
            const int row = 16 * cw + 8 * (i >> 1) + 2 * pr + (h ^ (i & 1));
            r[i] = *reinterpret_cast<const uint4*>(src + row * 128);
          }
          if (!ptx::mbar_wait(&op_empty[os], oph ^ 1, WAIT_NS)) {
            record_error(err, abort_flag, 6);
            ok = false;
            break;
          }
          uint8_t* dst = smem + S_OP_OFF + os * S_OP_BYTES + h * S_TILE;
          uint32_t bre[4] = {0u, 0u, 0u, 0u}, bim[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = 16 * cw + 8 * (i >> 1) + 2 * pr + (h ^ (i & 1));
            uint4 o0 = make_uint4(flip_hi(r[i].x), flip_lo(r[i].x), flip_hi(r[i].y), flip_lo(r[i].y));
            uint4 o1 = make_uint4(flip_hi(r[i].z), flip_lo(r[i].z), flip_hi(r[i].w), flip_lo(r[i].w));
            if (row >= n_valid) o0 = o1 = make_uint4(0u, 0u, 0u, 0u);
            uint8_t* rowp = dst + (row >> 3) * 1024 + (row & 7) * 128;
            *reinterpret_cast<uint4*>(rowp + (((2 * c) ^ (row & 7)) << 4)) = o0;
            *reinterpret_cast<uint4*>(rowp + (((2 * c + 1) ^ (row & 7)) << 4)) = o1;
            bre[0] += o0.x;
            bim[0] += o0.y;
            bre[1] += o0.z;
            bim[1] += o0.w;
            bre[2] += o1.x;
            bim[2] += o1.y;
            bre[3] += o1.z;
            bim[3] += o1.w;
          }
          ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            ptx::mbar_arrive(&op_full[os]);
            // the stores above needed the loaded samples, so the loads are done; an arrival right behind the
            // loads overtook them, and the next box landed under them
            ptx::mbar_arrive(&raw_empty[rs]);
          }
          if (++rs == S_RAW) {
            rs = 0;
            rph ^= 1;
          }
          if (++os == S_OP) {
            os = 0;
            oph ^= 1;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            sre[i][0] += bre[i] & 0x00FF00FFu;
            sre[i][1] += (bre[i] >> 8) & 0x00FF00FFu;
            sim[i][0] += bim[i] & 0x00FF00FFu;
            sim[i][1] += (bim[i] >> 8) & 0x00FF00FFu;
          }
        }
        if (!ok) break;
        // the sums of this chunk over the four lanes of a column; each of them adds 4 of its 16 inputs
        const long long u = 2 * it.p + h;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int re = (int)((sre[i][b & 1] >> (16 * (b >> 1))) & 0xFFFF), im = (int)((sim[i][b & 1] >> (16 * (b >> 1))) & 0xFFFF);
            re += __shfl_xor_sync(0xffffffffu, re, 8);
            im += __shfl_xor_sync(0xffffffffu, im, 8);
            re += __shfl_xor_sync(0xffffffffu, re, 16);
            im += __shfl_xor_sync(0xffffffffu, im, 16);
            const int in = 16 * c + 4 * i + b;  // input row of the unit
            const int ch = in / args.ld, n = in - ch * args.ld;
            const long long f = u * args.g + ch;
            if (pr == i && ch < args.g && n < args.N && u < args.n_units && f < args.C) {
              const long long idx = (f * args.N + n) * 2;
              atomicAdd(reinterpret_cast<unsigned long long*>(args.s1 + idx), (unsigned long long)re);
              atomicAdd(reinterpret_cast<unsigned long long*>(args.s1 + idx + 1), (unsigned long long)im);
              atomicAdd(reinterpret_cast<unsigned long long*>(args.s2 + idx), (unsigned long long)re);
              atomicAdd(reinterpret_cast<unsigned long long*>(args.s2 + idx + 1), (unsigned long long)im);
            }
          }
      }
    }
  } else {
    // ---------------- epilogue (warps 10..17): four warps, one TMEM lane quarter each, a unit ----------------
    const int q = warp & 3, h = (warp - 10) >> 2;
    const bool im_lane = (lane & 4) != 0;
    const int lp = args.npol >> 1;
    const int row = 32 * q + lane;
    const int ic = 4 * (row >> 3) + (row & 3);  // c-input of the unit
    const int ch = ic / args.ld, c = ic - ch * args.ld;
    // the chunks (16 a-inputs) that hold this warp's channels, from the diagonal on
    const int last = min(64, ((16 * q + 15) / args.ld + 1) * args.ld);
    const int cc_end = (last + 15) / 16;
    uint32_t use[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (long long w = blockIdx.x; w < total && ok; w += gridDim.x) {
      const SmallItem it(args, w, n_pairs);
      const long long u = 2 * it.p + h, f = u * args.g + ch;
      const bool live = ch < args.g && u < args.n_units && f < args.C;
      long long* cross_f = args.cross + (live ? f : 0) * args.Bs * args.npol * args.npol * 2;
      long long* autos_f = args.autos + (live ? f : 0) * args.N;
      for (int k0 = it.k0; k0 < it.k1; k0 += chunk_k) {
        if (__any_sync(0xffffffffu, *abort_flag != 0)) {
          ok = false;
          break;
        }
        const bool got = ptx::mbar_wait(&tfull[acc], use[acc] & 1, WAIT_NS);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) record_error(err, abort_flag, 4);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        if (u < args.n_units) {
          for (int cc = q; cc < cc_end; ++cc) {
            uint32_t v[32];
            ptx::tmem_ld_32x32b_x32(tbase + 256 * acc + 128 * h + ((uint32_t)(32 * q) << 16) + 32 * cc, v);
            ptx::tmem_ld_wait();
            int re[8], im[8];
            xd::combine_chunk<4>(v, im_lane, re, im);
            xd::add_chunk<ADD>(re, im, im_lane, live ? c : -1, 16 * cc - ch * args.ld, args.N, lp, cross_f, autos_f);
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&tempty[acc]);
        ++use[acc];
        acc ^= 1;
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  if (warp == 1) ptx::tmem_dealloc(tbase, TMEM_COLS);
}

// Channels (of ld stored inputs) per 64-input unit: as many as fit with a unit of whole 16-byte columns; 0 if none.
int small_group(int ld) {
  if (ld > 64) return 0;
  for (int g = 64 / ld; g >= 1; --g)
    if (g * ld % 16 == 0) return g;
  return 0;
}

}  // namespace

bool xeng_small_supported(const Shape& s, int ld, const void* d_in) {
  const long long row = (long long)ld * s.C;
  return s.N <= 64 && small_group(ld) > 0 && row % 16 == 0 && row < (1LL << 31) && reinterpret_cast<uintptr_t>(d_in) % 16 == 0;
}

cudaError_t launch_xeng_small(const DirectJob& j, int num_sms, cudaStream_t st) {
  if (j.n == 0 || j.T_blk == 0) return cudaSuccess;
  cudaError_t e = set_smem_limit(reinterpret_cast<const void*>(xeng_small_kernel<false>), S_SMEM);
  if (e == cudaSuccess) e = set_smem_limit(reinterpret_cast<const void*>(xeng_small_kernel<true>), S_SMEM);
  xd::Args a;
  if (e == cudaSuccess) e = direct_args(j, 128, false, &a);
  if (e != cudaSuccess) return e;
  a.g = small_group(j.ld);
  a.ub = a.g * j.ld;
  a.n_units = (j.s.C + a.g - 1) / a.g;
  const long long pairs = (a.n_units + 1) / 2;
  a.splits = direct_splits(pairs, num_sms, a.n_k, 4);
  a.kps = (a.n_k + a.splits - 1) / a.splits;
  a.n_items = pairs * a.splits;
  const unsigned grid = (unsigned)std::min<long long>(num_sms, a.n_items);
  if (a.splits > 1)
    xeng_small_kernel<true><<<grid, S_THREADS, S_SMEM, st>>>(a);
  else
    xeng_small_kernel<false><<<grid, S_THREADS, S_SMEM, st>>>(a);
  return cudaGetLastError();
}

}  // namespace corr
