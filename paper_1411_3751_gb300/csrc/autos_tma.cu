// Total power A[f][n] += sum_t |x_{f,n}(t)|^2 (Sec. 2.6: total power at a high cadence) of blocks whose rows TMA
// takes: HBM-bound, the samples are read once. (autos_kernel does the others; its byte-lane squares take more
// issue slots than HBM leaves: 512 inputs x 2400 channels x 240 samples 77 us, 54 us so, 5.4 TB/s; 64 inputs x 6000
// samples 212 and 140 us, 6.6 TB/s.)
//
// A row t is M = C N neighbouring bytes; an item is 128 of them (128 cells) and a run of rows, fetched as boxes of
// 128 bytes x 128 samples into a ring by one thread. Warp w takes the 16-byte column w of a box: ldmatrix.trans.b8
// brings it into registers transposed, four samples of an input a word, and the high nibbles (16 Re as signed
// bytes) and, shifted, the low ones (16 Im) meet themselves in dp4a: five instructions for four samples. The sums
// are 256 |x|^2; rows past the block read as 0 and add nothing. Every wait is bounded (f8::WAIT_NS).
#include <algorithm>
#include <cstring>

#include "corr_internal.cuh"
#include "f8_common.cuh"

namespace corr {
namespace {

using namespace f8;

constexpr int AT_THREADS = 288;             // 8 consumer warps, 1 producer warp
constexpr int AT_RING = 6;                  // 96 KB; two CTAs an SM
constexpr int AT_BOX = 128 * KT;
constexpr int AT_SMEM = AT_RING * AT_BOX + 256 + 1024;
constexpr int AT_MAX_STAGES = 1024;         // of an item: 2^15 samples a lane of at most 2^15 in an int32

struct AutosArgs {
  CUtensorMap map;  // [T][M] bytes
  long long* autos;
  long long M, n_items, n_cols;  // cells; items; 128-byte columns
  int n_k, kps;                  // stages of the block, of an item
  int* err;
};

__global__ void __launch_bounds__(AT_THREADS, 2) autos_tma_kernel(const __grid_constant__ AutosArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + AT_RING * AT_BOX);
  uint64_t* empty = full + AT_RING;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + AT_RING);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < AT_RING; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 8);
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  __syncthreads();
  int slot = 0;
  uint32_t phase = 0;
  if (warp == 8) {
    if (lane == 0) {
      uint32_t n_issued = 0;
      for (long long w = blockIdx.x; w < a.n_items && !*abort_flag; w += gridDim.x) {
        const int run = (int)(w / a.n_cols);
        const int x = (int)(w - run * a.n_cols) * 128, k1 = min(a.n_k, (run + 1) * a.kps);
        for (int k = run * a.kps; k < k1; ++k) {
          if (!ptx::mbar_wait(&empty[slot], phase ^ 1, WAIT_NS)) {
            record_error(a.err, abort_flag, 7);
            break;
          }
          ptx::mbar_arrive_expect_tx(&full[slot], AT_BOX);
          ptx::tma_load_2d(smem + slot * AT_BOX, &a.map, &full[slot], x, k * KT);
          ++n_issued;
          if (++slot == AT_RING) {
            slot = 0;
            phase ^= 1;
          }
        }
      }
      // copies still in flight must land before the CTA exits: the last use of every slot
      for (int s = 0; s < AT_RING; ++s) {
        const uint32_t uses = n_issued / AT_RING + ((uint32_t)s < n_issued % AT_RING ? 1u : 0u);
        if (uses > 0) ptx::mbar_wait(&full[s], (uses - 1) & 1, WAIT_NS);
      }
    }
    return;
  }
  // lane l addresses sample row l (+ 32 kk) of the warp's column (128-byte swizzle)
  const uint32_t src = ptx::smem_u32(smem) + (uint32_t)lane * 128 + (uint32_t)((warp ^ (lane & 7)) << 4);
  for (long long w = blockIdx.x; w < a.n_items; w += gridDim.x) {
    if (__any_sync(0xffffffffu, *abort_flag != 0)) return;
    const int run = (int)(w / a.n_cols);
    const long long x = (w - run * a.n_cols) * 128;
    const int k1 = min(a.n_k, (run + 1) * a.kps);
    int acc[2] = {0, 0};  // inputs lane / 4 and lane / 4 + 8 of the column
    for (int k = run * a.kps; k < k1; ++k) {
      // all lanes out of their waits: ldmatrix is for whole warps
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(&full[slot], phase, WAIT_NS))) {
        record_error(a.err, abort_flag, 8);
        return;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        uint32_t v[4];
        ptx::ldmatrix_b8_x2_trans(src + slot * AT_BOX + kk * 4096, v[0], v[1], v[2], v[3]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int re = (int)(v[i] & 0xF0F0F0F0u), im = (int)((v[i] << 4) & 0xF0F0F0F0u);
          acc[i & 1] = __dp4a(re, re, __dp4a(im, im, acc[i & 1]));
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&empty[slot]);  // the sums needed the loaded samples, so the loads are done
      if (++slot == AT_RING) {
        slot = 0;
        phase ^= 1;
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      long long s = acc[i];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      const long long cell = x + 16 * warp + (lane >> 2) + 8 * i;
      if ((lane & 3) == 0 && cell < a.M)
        atomicAdd(reinterpret_cast<unsigned long long*>(a.autos + cell), (unsigned long long)(s >> 8));
    }
  }
}

}  // namespace

bool autos_tma_supported(const Shape& s, const void* d_in) {
  const long long M = (long long)s.C * s.N;
  return M % 16 == 0 && M < (1LL << 31) && reinterpret_cast<uintptr_t>(d_in) % 16 == 0;
}

cudaError_t launch_autos_tma(const Shape& s, const uint8_t* d_in, int T_blk, long long* d_autos, int* d_err, cudaStream_t st) {
  if (T_blk == 0) return cudaSuccess;
  AutosArgs a;
  std::memset(&a, 0, sizeof(a));
  a.M = (long long)s.C * s.N;
  std::string err;
  if (encode_raw_tensor_map(&a.map, d_in, a.M, T_blk, &err) != 0) {
    set_last_error(err);
    return cudaErrorInvalidValue;
  }
  a.autos = d_autos;
  a.err = d_err;
  a.n_cols = (a.M + 127) / 128;
  a.n_k = (T_blk + KT - 1) / KT;
  // runs of the rows: the whole block while the columns fill the GPU several times over
  const long long ctas = 2LL * sm_count();
  const long long want = std::max<long long>(1, (4 * ctas + a.n_cols - 1) / a.n_cols);
  a.kps = (int)std::min<long long>(AT_MAX_STAGES, std::max<long long>(1, (a.n_k + want - 1) / want));
  a.n_items = a.n_cols * ((a.n_k + a.kps - 1) / a.kps);
  const cudaError_t e = set_smem_limit(reinterpret_cast<const void*>(autos_tma_kernel), AT_SMEM);
  if (e != cudaSuccess) return e;
  autos_tma_kernel<<<(unsigned)std::min(ctas, a.n_items), AT_THREADS, AT_SMEM, st>>>(a);
  return cudaGetLastError();
}

}  // namespace corr
