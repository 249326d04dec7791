// Samples with rows of any length to rows of whole 16-byte columns, for the X-engine that reads the samples with
// TMA (xeng_small.cu): in[rows][N] -> out[rows][Np], Np = N rounded up to 16, zeros behind the last input. Taken where
// a sample of all channels is not a multiple of 16 bytes (TMA's stride) or the block starts between 16-byte
// boundaries. Reads one byte a sample and writes little more (the two-pass path writes two and reads them back):
// with the X-engine behind it 20 inputs x 1201 channels x 4096 samples 91 us (two passes 163), 63 x 601 118 (172).
//
// HBM-bound. A thread keeps one 16-byte column of the output rows and walks down them, several rows in flight. The
// input rows start at any byte: where rows and buffer are not multiples of 8 or 4 bytes a column is the five
// aligned words around it, shifted together (the neighbours' words come from L1), or single bytes where those
// words would leave the buffer.
#include "corr_internal.cuh"

namespace corr {
namespace {

constexpr int RP_NT = 256;
// rows in flight: 8, or 4 of the five-word columns (63 inputs x 601 channels x 4096: 64 us, with 8 rows 80)
constexpr int RP_WIDE = 8, RP_NARROW = 4;

// The 16 bytes at p, nv of them inputs, zeros behind. ALIGN 8 or 4: rows and buffer are multiples of it, whole pieces.
template <int ALIGN>
__device__ __forceinline__ uint4 load_column(const uint8_t* p, int nv, const uint8_t* in, const uint8_t* end) {
  if (ALIGN == 8) {
    const uint2 lo = __ldg(reinterpret_cast<const uint2*>(p));
    const uint2 hi = nv > 8 ? __ldg(reinterpret_cast<const uint2*>(p) + 1) : make_uint2(0u, 0u);
    return make_uint4(lo.x, lo.y, hi.x, hi.y);
  }
  uint32_t x[5] = {0u, 0u, 0u, 0u, 0u};
  if (ALIGN == 4) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (nv > 4 * k) x[k] = __ldg(reinterpret_cast<const uint32_t*>(p) + k);
    return make_uint4(x[0], x[1], x[2], x[3]);
  }
  const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3);
  const uint8_t* q = p - sh;
  if (q >= in && q + 20 <= end) {
#pragma unroll
    for (int k = 0; k < 5; ++k) x[k] = __ldg(reinterpret_cast<const uint32_t*>(q) + k);
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = __funnelshift_r(x[k], x[k + 1], 8 * sh);
    if (nv < 16) {  // the next row's bytes behind the last input
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int n = nv - 4 * k;
        x[k] &= n >= 4 ? 0xFFFFFFFFu : n <= 0 ? 0u : 0xFFFFFFFFu >> (32 - 8 * n);
      }
    }
  } else {
    for (int k = 0; k < nv; ++k) {
      const uint32_t b = (uint32_t)p[k] << (8 * (k & 3));
      if (k < 4) x[0] |= b; else if (k < 8) x[1] |= b; else if (k < 12) x[2] |= b; else x[3] |= b;
    }
  }
  return make_uint4(x[0], x[1], x[2], x[3]);
}

// A block step takes RP_NT / cols rows of cols = Np / 16 columns (at most four, so a few threads idle at three).
template <int ALIGN>
__global__ void __launch_bounds__(RP_NT) repack_kernel(const uint8_t* __restrict__ in, long long rows, int N, int Np,
                                                       uint8_t* __restrict__ out) {
  constexpr int RP_U = ALIGN > 1 ? RP_WIDE : RP_NARROW;
  const int cols = Np / 16, rpb = RP_NT / cols, sub = (int)threadIdx.x / cols;
  const int n0 = 16 * ((int)threadIdx.x - sub * cols);
  if (sub >= rpb) return;
  const int nv = min(16, N - n0);
  const uint8_t* end = in + rows * N;
  const long long step = (long long)gridDim.x * rpb;
  for (long long r = (long long)blockIdx.x * rpb + sub; r < rows; r += RP_U * step) {
    uint4 v[RP_U];
#pragma unroll
    for (int u = 0; u < RP_U; ++u)
      if (r + u * step < rows) v[u] = load_column<ALIGN>(in + (r + u * step) * N + n0, nv, in, end);
#pragma unroll
    for (int u = 0; u < RP_U; ++u)
      if (r + u * step < rows) *reinterpret_cast<uint4*>(out + (r + u * step) * Np + n0) = v[u];
  }
}

}  // namespace

cudaError_t launch_repack(const uint8_t* d_in, long long rows, int N, int Np, uint8_t* d_out, cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
  if (Np > 64) return cudaErrorInvalidValue;
  const int rpb = RP_NT / (Np / 16);
  const uintptr_t x = reinterpret_cast<uintptr_t>(d_in) | (uintptr_t)N;
  const int rows_step = rpb * (x % 4 == 0 ? RP_WIDE : RP_NARROW);
  const long long want = (rows + rows_step - 1) / rows_step, cap = (long long)sm_count() * 16;
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  if (x % 8 == 0)
    repack_kernel<8><<<grid, RP_NT, 0, st>>>(d_in, rows, N, Np, d_out);
  else if (x % 4 == 0)
    repack_kernel<4><<<grid, RP_NT, 0, st>>>(d_in, rows, N, Np, d_out);
  else
    repack_kernel<1><<<grid, RP_NT, 0, st>>>(d_in, rows, N, Np, d_out);
  return cudaGetLastError();
}

}  // namespace corr
