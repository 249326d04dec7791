// Corner turn between GPUs (paper Sec. 2.3 and Fig. 2: each F-engine board holds every channel of its
// own antennas, each X-engine GPU needs every antenna of its own channels, and the network turns the
// data from one grouping to the other). With one process per GPU the exchange is an all-to-all; these
// two kernels are its local halves, byte permutations with no arithmetic:
//  * pack:   this rank's inputs [T][C][n_local] -> one contiguous block [T][C_d][n_local] per
//            destination d, in destination order (C_d = chan_bounds[d + 1] - chan_bounds[d]);
//  * unpack: the blocks received from every source s, [T][C][n_s] each in source order ->
//            [T][C][N], source s's inputs at columns input_bounds[s] .. input_bounds[s + 1] - 1.
// Both move whole granules, the largest of 16, 8, 4, 2 and 1 bytes that divides every row, part and pointer.
#include <string>
#include <vector>

#include "corr_internal.cuh"

namespace corr {
namespace {

constexpr int kMaxParts = 1024;

struct Bounds {
  long long b[kMaxParts + 1];
  int n;
};

__device__ __forceinline__ int find_part(const Bounds& bd, long long x) {
  int lo = 0, hi = bd.n - 1;  // largest p with b[p] <= x
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (bd.b[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// HBM-bound (1000 samples x 2398 channels x 32 inputs, then 16 sources of 32 inputs x 109 channels: one
// warp per 32-byte row, two of its lanes busy and a 64-bit division and a search a row, took 367 + 182 us).
//
// Pack: the channels of destination d are neighbours in every input row t, and stay neighbours in its
// block, so (t, d) is one contiguous run of C_d n_local bytes on both sides. A warp copies pieces of
// at most PIECE bytes of such a run, four loads in flight a lane: 367 -> 25 us.
constexpr int CT_PIECE = 4096;
constexpr int CT_NT = 256;

template <typename V>
__global__ void __launch_bounds__(CT_NT) ct_pack_kernel(const uint8_t* __restrict__ in, int T, int C, int n_local,
                                                        const __grid_constant__ Bounds chans, int pieces,
                                                        uint8_t* __restrict__ out) {
  constexpr int U = 4, VP = CT_PIECE / (int)sizeof(V);  // granules per piece
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (CT_NT / 32);
  const long long items = (long long)T * chans.n * pieces;
  for (long long w = blockIdx.x * (long long)(CT_NT / 32) + (threadIdx.x >> 5); w < items; w += warps) {
    const long long td = w / pieces;
    const int piece = (int)(w - td * pieces);
    const long long t = td / chans.n;
    const int d = (int)(td - t * chans.n);
    const long long c0 = chans.b[d], cd = chans.b[d + 1] - c0;
    const long long v0 = (long long)piece * VP, run = cd * n_local / (int)sizeof(V);  // granules of the run
    if (v0 >= run) continue;
    const int n = (int)(run - v0 < VP ? run - v0 : VP);
    const V* src = reinterpret_cast<const V*>(in + (t * C + c0) * n_local) + v0;
    V* dst = reinterpret_cast<V*>(out + ((long long)T * c0 + t * cd) * n_local) + v0;
    for (int i = lane; i < n; i += 32 * U) {
      V x[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i + 32 * u < n) x[u] = src[i + 32 * u];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i + 32 * u < n) dst[i + 32 * u] = x[u];
    }
  }
}

// Unpack: a thread keeps one granule column of the output rows, so it looks its source up once, and
// walks down the rows, eight loads in flight; neighbouring threads write neighbouring granules.
// `cols` columns a block (threadIdx.x % cols; blockIdx.x counts blocks of columns), CT_NT / cols rows a
// step: 182 -> 23 us.
template <typename V>
__global__ void __launch_bounds__(CT_NT) ct_unpack_kernel(const uint8_t* __restrict__ in, long long rows, int N, int cols,
                                                          const __grid_constant__ Bounds inputs,
                                                          uint8_t* __restrict__ out) {
  constexpr int U = 8;
  const int rpb = CT_NT / cols;  // rows a block step
  const int sub = (int)threadIdx.x / cols;
  const long long n = ((long long)blockIdx.x * cols + ((int)threadIdx.x - sub * cols)) * (int)sizeof(V);  // first input
  if (sub >= rpb || n >= N) return;
  const int s = find_part(inputs, n);
  const long long n0 = inputs.b[s], ns = inputs.b[s + 1] - n0;
  const uint8_t* src = in + rows * n0 + (n - n0);
  uint8_t* dst = out + n;
  const long long step = (long long)gridDim.y * rpb;
  for (long long r = (long long)blockIdx.y * rpb + sub; r < rows; r += U * step) {
    V x[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r + u * step < rows) x[u] = *reinterpret_cast<const V*>(src + (r + u * step) * ns);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r + u * step < rows) *reinterpret_cast<V*>(dst + (r + u * step) * N) = x[u];
  }
}

template <typename V>
void launch_pack(const uint8_t* in, int T, int C, int n_local, const Bounds& bd, uint8_t* out, cudaStream_t st) {
  long long widest = 0;
  for (int d = 0; d < bd.n; ++d) widest = bd.b[d + 1] - bd.b[d] > widest ? bd.b[d + 1] - bd.b[d] : widest;
  const long long pieces = (widest * n_local + CT_PIECE - 1) / CT_PIECE;
  long long blocks = ((long long)T * bd.n * pieces + CT_NT / 32 - 1) / (CT_NT / 32);
  const long long cap = (long long)sm_count() * 16;
  if (blocks > cap) blocks = cap;
  ct_pack_kernel<V><<<(unsigned)blocks, CT_NT, 0, st>>>(in, T, C, n_local, bd, (int)pieces, out);
}

template <typename V>
void launch_unpack(const uint8_t* in, long long rows, int N, const Bounds& bd, uint8_t* out, cudaStream_t st) {
  const int all = N / (int)sizeof(V), cols = all < CT_NT ? all : CT_NT;
  const unsigned gx = (unsigned)((all + cols - 1) / cols);
  const int rpb = CT_NT / cols;
  long long gy = (rows + 8 * rpb - 1) / (8 * rpb);
  const long long cap = ((long long)sm_count() * 16 + gx - 1) / gx;
  if (gy > cap) gy = cap;
  ct_unpack_kernel<V><<<dim3(gx, (unsigned)gy), CT_NT, 0, st>>>(in, rows, N, cols, bd, out);
}

// Largest granule (16, 8, 4, 2 or 1 bytes) that divides everything or-ed into x.
int granule(unsigned long long x) {
  int g = 16;
  while (x & (unsigned long long)(g - 1)) g /= 2;
  return g;
}

int ct_fail(int code, const std::string& m) {
  set_last_error(m);
  return code;
}

bool read_bounds(const int* h, int n, long long end, Bounds* bd) {
  if (!h || n < 1 || n > kMaxParts) return false;
  if (h[0] != 0 || h[n] != end) return false;
  for (int i = 0; i < n; ++i)
    if (h[i + 1] < h[i]) return false;
  for (int i = 0; i <= n; ++i) bd->b[i] = h[i];
  bd->n = n;
  return true;
}

}  // namespace
}  // namespace corr

using namespace corr;

extern "C" int corr_corner_turn_pack(const void* d_in, int n_time, int n_chans, int n_local, const int* chan_bounds,
                                     int n_dest, void* d_out, void* cuda_stream) {
  if (n_time < 0 || n_chans < 0 || n_local < 0)
    return ct_fail(CORR_ERR_ARG, "corr_corner_turn_pack: need n_time, n_chans, n_local >= 0");
  Bounds bd;
  if (!read_bounds(chan_bounds, n_dest, n_chans, &bd))
    return ct_fail(CORR_ERR_ARG, "corr_corner_turn_pack: chan_bounds must run 0 = b[0] <= ... <= b[n_dest] = n_chans, "
                                 "1 <= n_dest <= 1024");
  const long long rows = (long long)n_time * n_chans;
  if (rows == 0 || n_local == 0) return CORR_OK;  // nothing to move (an empty shard)
  if (!d_in || !d_out) return ct_fail(CORR_ERR_ARG, "corr_corner_turn_pack: NULL buffer");
  const uint8_t* in = static_cast<const uint8_t*>(d_in);
  uint8_t* out = static_cast<uint8_t*>(d_out);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  switch (granule((unsigned long long)n_local | reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out))) {
    case 16: launch_pack<uint4>(in, n_time, n_chans, n_local, bd, out, st); break;
    case 8: launch_pack<uint2>(in, n_time, n_chans, n_local, bd, out, st); break;
    case 4: launch_pack<uint32_t>(in, n_time, n_chans, n_local, bd, out, st); break;
    case 2: launch_pack<uint16_t>(in, n_time, n_chans, n_local, bd, out, st); break;
    default: launch_pack<uint8_t>(in, n_time, n_chans, n_local, bd, out, st); break;
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return ct_fail(CORR_ERR_CUDA, std::string("corr_corner_turn_pack: ") + cudaGetErrorString(e));
  return CORR_OK;
}

extern "C" int corr_corner_turn_unpack(const void* d_in, int n_time, int n_chans, int n_inputs, const int* input_bounds,
                                       int n_src, void* d_out, void* cuda_stream) {
  if (n_time < 0 || n_chans < 0 || n_inputs < 0)
    return ct_fail(CORR_ERR_ARG, "corr_corner_turn_unpack: need n_time, n_chans, n_inputs >= 0");
  Bounds bd;
  if (!read_bounds(input_bounds, n_src, n_inputs, &bd))
    return ct_fail(CORR_ERR_ARG, "corr_corner_turn_unpack: input_bounds must run 0 = b[0] <= ... <= b[n_src] = "
                                 "n_inputs, 1 <= n_src <= 1024");
  const long long rows = (long long)n_time * n_chans;
  if (rows == 0 || n_inputs == 0) return CORR_OK;  // nothing to move (an empty shard)
  if (!d_in || !d_out) return ct_fail(CORR_ERR_ARG, "corr_corner_turn_unpack: NULL buffer");
  const uint8_t* in = static_cast<const uint8_t*>(d_in);
  uint8_t* out = static_cast<uint8_t*>(d_out);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  unsigned long long x = reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out);
  for (int s = 0; s <= n_src; ++s) x |= (unsigned long long)input_bounds[s];
  switch (granule(x)) {
    case 16: launch_unpack<uint4>(in, rows, n_inputs, bd, out, st); break;
    case 8: launch_unpack<uint2>(in, rows, n_inputs, bd, out, st); break;
    case 4: launch_unpack<uint32_t>(in, rows, n_inputs, bd, out, st); break;
    case 2: launch_unpack<uint16_t>(in, rows, n_inputs, bd, out, st); break;
    default: launch_unpack<uint8_t>(in, rows, n_inputs, bd, out, st); break;
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return ct_fail(CORR_ERR_CUDA, std::string("corr_corner_turn_unpack: ") + cudaGetErrorString(e));
  return CORR_OK;
}
