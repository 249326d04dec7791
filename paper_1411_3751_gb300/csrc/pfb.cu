// Polyphase filterbank (PFB) F-engine (Sec. 2.2): each input's real 8-bit ADC stream is split into
// frames of M = 8192 samples; spectrum t weights the P = n_taps frames t .. t + P - 1 by the
// prototype filter (FIR, exact in integers: 8-bit samples x 18-bit coefficients), sums them, and
// takes an M-point real DFT, keeping channels 0 .. M/2 - 1 (24.0 kHz apart at a 196.608 MHz clock).
// The paper's fixed-point FFT halves at each of its log2(M) = 13 stages; here the FFT runs in FP32
// and the result is scaled by the same 2^-13 once (an exact power of two).
//
//   y_t[m] = sum_p h[p M + m] x[(t + p) M + m]                       (int32, exact)
//   X_t[k] = 2^-13 sum_m y_t[m] exp(-2 pi i k m / M),  k < M / 2      (FP32)
//
// One CTA of 256 threads per (input, two spectra). The real DFT is a 4096-point complex FFT of
// z[j] = y[2j] + i y[2j+1] followed by the split step that separates the even and odd halves:
//   X[k] = (Z[k] + conj Z[-k]) / 2 - i W^k (Z[k] - conj Z[-k]) / 2,  W = exp(-2 pi i / M).
// The complex FFT is a Stockham autosort FFT (no bit reversal) of three radix-16 passes. What bounded it
// was shared memory (four exchanges of 64 KB a spectrum) and load latency, so data leave the registers
// only twice: the FIR sums are formed by the threads whose first pass takes them, and in the last pass a
// thread of a spectrum's 128 holds columns u and 256 - u, whose outputs are each other's mirror images
// k and 4096 - k, so that the split step needs no exchange either. Twiddles come from tables computed on
// the host in double precision. 512 inputs x 64 spectra, 4 taps: 753 us before, 573 us so
// (2 CTAs of 8 warps an SM. At 588 us, with the split factors as products: without the FIR's loads 465, without the
// output stores 489; with 80 registers and a third CTA 686, with the samples staged through shared memory by
// 16-byte loads 613).
#include "corr_internal.cuh"

#include <cmath>
#include <mutex>

namespace corr {
namespace {

constexpr int PFB_M = 8192;          // real FFT length
constexpr int PFB_H = PFB_M / 2;     // complex FFT length / output channels
constexpr int PFB_NT = 256;
constexpr float PFB_SCALE = 1.0f / 8192.0f;  // 2^-13

__device__ float2 g_w4096[PFB_H];  // exp(-2 pi i j / 4096)
__device__ __align__(16) float2 g_w8192[PFB_H / 2];  // exp(-2 pi i k / 8192), k < 2048

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }  // a * (-i)

// shared-memory index with one pad element per 16 (breaks the stride-16 bank pattern of pass 0)
__device__ __forceinline__ int sidx(int i) { return i + (i >> 4); }

// In-register forward 16-point DFT, X[q] = sum_r v[r] exp(-2 pi i r q / 16), as 4 x 4: 4-point DFTs
// over a (r = 4 a + b), twiddles exp(-2 pi i b k1 / 16), 4-point DFTs over b; output X[k1 + 4 k2].
__device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3) {
  const float2 s02 = cadd(a0, a2), d02 = csub(a0, a2), s13 = cadd(a1, a3), d13 = mul_mi(csub(a1, a3));
  a0 = cadd(s02, s13);
  a2 = csub(s02, s13);
  a1 = cadd(d02, d13);
  a3 = csub(d02, d13);
}

__device__ __forceinline__ void dft16(float2 (&v)[16]) {
  constexpr float C1 = 0.92387953251128674f;  // cos(pi / 8)
  constexpr float S1 = 0.38268343236508978f;  // sin(pi / 8)
  constexpr float R2 = 0.70710678118654752f;  // cos(pi / 4)
#pragma unroll
  for (int b = 0; b < 4; ++b) dft4(v[b], v[b + 4], v[b + 8], v[b + 12]);  // now v[4 k1 + b] = A[b][k1]
  // twiddles exp(-2 pi i b k1 / 16) for b, k1 in 1..3
  v[5] = cmul(v[5], make_float2(C1, -S1));    // b=1,k1=1: m=1
  v[9] = cmul(v[9], make_float2(R2, -R2));    // b=1,k1=2: m=2
  v[13] = cmul(v[13], make_float2(S1, -C1));  // b=1,k1=3: m=3
  v[6] = cmul(v[6], make_float2(R2, -R2));    // b=2,k1=1: m=2
  v[10] = mul_mi(v[10]);                      // b=2,k1=2: m=4
  v[14] = cmul(v[14], make_float2(-R2, -R2)); // b=2,k1=3: m=6
  v[7] = cmul(v[7], make_float2(S1, -C1));    // b=3,k1=1: m=3
  v[11] = cmul(v[11], make_float2(-R2, -R2)); // b=3,k1=2: m=6
  v[15] = cmul(v[15], make_float2(-C1, S1));  // b=3,k1=3: m=9
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
  // now v[4 k1 + k2] = X[k1 + 4 k2]; reorder to natural order
  float2 t[16];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) t[k1 + 4 * k2] = v[4 * k1 + k2];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = t[q];
}

constexpr int PFB_SPB = 2;                    // spectra per block (share the coefficient and frame loads)
constexpr int PFB_ZLEN = PFB_H + PFB_H / 16;  // padded complex buffer per spectrum

// Rows q < 8 of the split step's factors W^(u + 256 q), u <= 128, beside the buffers (the others are -i times these).
// From the table, each rounded once: as products W^u W^(256 q) their error is 2.4 times as large (the spectrum's 1.44e-7
// instead of 1.39e-7, relative, 4 taps). They come with cp.async while the FIR runs: at the size above 573 us, as
// products 588, loaded where they are used 628, all 16 rows so 716.
constexpr int PFB_WLD = 130;  // row stride
constexpr int PFB_SMEM = (PFB_SPB * PFB_ZLEN + 8 * PFB_WLD) * (int)sizeof(float2);

__device__ __forceinline__ void fetch_split_factors(float2* ws, int tid) {
  const int q = tid >> 5, u = 4 * (tid & 31);
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ws + q * PFB_WLD + u);
  const float2* src = g_w8192 + 256 * q + u;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16), "l"(src + 2) : "memory");
  if (u == 0) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 128 * 8), "l"(src + 128) : "memory");
}

// v[r] *= w^r for r = 1 .. 15 from w1 = w, w4 = w^4, w8, w12, as w^(4a + b) = w^(4a) w^b, for each of S columns.
template <int S>
__device__ __forceinline__ void twiddle16(float2 (&v)[S][16], float2 w1, float2 w4, float2 w8, float2 w12) {
  const float2 w2 = cmul(w1, w1), w3 = cmul(w2, w1);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const float2 wa = a == 1 ? w4 : a == 2 ? w8 : w12;
    const float2 t1 = a ? cmul(wa, w1) : w1, t2 = a ? cmul(wa, w2) : w2, t3 = a ? cmul(wa, w3) : w3;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      if (a) v[s][4 * a] = cmul(v[s][4 * a], wa);
      v[s][4 * a + 1] = cmul(v[s][4 * a + 1], t1);
      v[s][4 * a + 2] = cmul(v[s][4 * a + 2], t2);
      v[s][4 * a + 3] = cmul(v[s][4 * a + 3], t3);
    }
  }
}
__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }

// X[k] and X[4096 - k] from a = Z[k], b = Z[4096 - k] and w = W^k, scaled:
//   E = (a + conj b) / 2, O = (a - conj b) / 2, X[k] = E - i w O, X[4096 - k] = conj(E + i w O).
__device__ __forceinline__ void split_pair(float2 a, float2 b, float2 w, float2& xk, float2& xm) {
  const float h = 0.5f * PFB_SCALE;
  const float2 e = make_float2(h * (a.x + b.x), h * (a.y - b.y));
  const float2 od = make_float2(h * (a.x - b.x), h * (a.y + b.y));
  const float2 wo = mul_mi(cmul(w, od));
  xk = cadd(e, wo);
  xm = make_float2(e.x - wo.x, wo.y - e.y);
}

// Two samples of one frame (2-byte aligned) as a word, the second one in the high half.
__device__ __forceinline__ int load2(const int8_t* __restrict__ p) {
  return (int)__ldg(reinterpret_cast<const unsigned short*>(p));
}
__device__ __forceinline__ int byte0(int w) { return (int)(int8_t)(uint8_t)w; }
__device__ __forceinline__ int byte1(int w) { return (int)(int8_t)(uint8_t)(w >> 8); }

// PT > 0 fixes the tap count at compile time; PT == 0 takes it from P.
template <int PT>
__global__ void __launch_bounds__(PFB_NT, 2) pfb_kernel(const int8_t* __restrict__ adc, long long stride, int T,
                                                        int P, const int* __restrict__ h, float2* __restrict__ out) {
  extern __shared__ __align__(16) float2 zs[];  // PFB_SPB buffers of PFB_ZLEN, the split factors
  float2* ws = zs + PFB_SPB * PFB_ZLEN;
  const int t0 = blockIdx.x * PFB_SPB, n = blockIdx.y, tid = threadIdx.x;
  const int ns = T - t0 < PFB_SPB ? T - t0 : PFB_SPB;
  fetch_split_factors(ws, tid);
  float2 v[PFB_SPB][16];
  // FIR: the thread's column of the first pass, points tid + 256 r, i.e. samples 2 tid + 512 r and the next,
  // of both spectra: frames t0 .. t0 + P (the last one only if there is a second spectrum)
  const int8_t* x = adc + (size_t)n * stride + (size_t)t0 * PFB_M + 2 * tid;
  const int* hc = h + 2 * tid;
  if (PT > 0) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      int y[PFB_SPB][2] = {{0, 0}, {0, 0}};
      int fr[PT + 1];
      int2 c[PT > 0 ? PT : 1];
#pragma unroll
      for (int q = 0; q <= PT; ++q) fr[q] = q < PT || ns > 1 ? load2(x + (size_t)q * PFB_M + 512 * r) : 0;
#pragma unroll
      for (int p = 0; p < PT; ++p) c[p] = __ldg(reinterpret_cast<const int2*>(hc + p * PFB_M + 512 * r));
#pragma unroll
      for (int p = 0; p < PT; ++p)
#pragma unroll
        for (int s = 0; s < PFB_SPB; ++s) {
          y[s][0] += c[p].x * byte0(fr[p + s]);
          y[s][1] += c[p].y * byte1(fr[p + s]);
        }
#pragma unroll
      for (int s = 0; s < PFB_SPB; ++s) v[s][r] = make_float2((float)y[s][0], (float)y[s][1]);
    }
  } else {
    // any tap count: four points at a time, four taps of each in flight. (A tap of all 16 points at a time was slower:
    // 512 inputs x 8 spectra, 16 taps 180 us, 155 so, and with few spectra, where each step's latency shows, slower than
    // the shared-memory FIR that it replaced: 64 inputs x 1 spectrum, 16 taps 16.4 us, 14.5 that one, 14.4 so. Between
    // one and three waves of blocks it was the faster one: 128 x 8, 9 taps 31 and 35 us, the shared-memory FIR 47.)
#pragma unroll
    for (int r0 = 0; r0 < 16; r0 += 4) {
      int y[4][PFB_SPB][2] = {};
#pragma unroll 1
      for (int p0 = 0; p0 < P; p0 += 4) {
        int f[4][5];
        int2 c[4][4];
#pragma unroll
        for (int j = 0; j < 5; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const size_t at = (size_t)(p0 + j) * PFB_M + 512 * (r0 + i);
            f[i][j] = p0 + j < P + ns - 1 ? load2(x + at) : 0;
            if (j < 4) c[i][j] = p0 + j < P ? __ldg(reinterpret_cast<const int2*>(hc + at)) : make_int2(0, 0);
          }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int s = 0; s < PFB_SPB; ++s) {
              y[i][s][0] += c[i][j].x * byte0(f[i][j + s]);
              y[i][s][1] += c[i][j].y * byte1(f[i][j + s]);
            }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int s = 0; s < PFB_SPB; ++s) v[s][r0 + i] = make_float2((float)y[i][s][0], (float)y[i][s][1]);
    }
  }
  // pass 1 (span 1): outputs 16 tid + q
#pragma unroll
  for (int s = 0; s < PFB_SPB; ++s) {
    dft16(v[s]);
#pragma unroll
    for (int q = 0; q < 16; ++q) zs[s * PFB_ZLEN + sidx(16 * tid + q)] = v[s][q];
  }
  __syncthreads();
  // pass 2 (span 16): points tid + 256 r -> 16 (tid - k) + k + 16 q, k = tid mod 16
  {
    const int k = tid & 15, e = 16 * k;
    const float2 w1 = g_w4096[e], w4 = g_w4096[4 * e], w8 = g_w4096[8 * e], w12 = g_w4096[12 * e];
#pragma unroll
    for (int s = 0; s < PFB_SPB; ++s)
#pragma unroll
      for (int r = 0; r < 16; ++r) v[s][r] = zs[s * PFB_ZLEN + sidx(tid + 256 * r)];
    twiddle16<PFB_SPB>(v, w1, w4, w8, w12);
    __syncthreads();
    const int base = (tid - k) * 16 + k;
#pragma unroll
    for (int s = 0; s < PFB_SPB; ++s) {
      dft16(v[s]);
#pragma unroll
      for (int q = 0; q < 16; ++q) zs[s * PFB_ZLEN + sidx(base + 16 * q)] = v[s][q];
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // pass 3 (span 256) and split step: threads 128 s .. + 127 take spectrum s, thread u columns u and 256 - u
  // (thread 0: columns 0 and 128, each its own mirror image)
  const int s = tid >> 7, u = tid & 127;
  if (s >= ns) return;
  const int cb = u ? 256 - u : 128, eb = u ? u : 128;
  const float2* z = zs + s * PFB_ZLEN;
  float2 c2[1][16], d2[1][16];
  float2(&za)[16] = c2[0];
  float2(&zb)[16] = d2[0];
  {
    const float2 w1 = g_w4096[u], w4 = g_w4096[4 * u], w8 = g_w4096[8 * u], w12 = g_w4096[12 * u];
#pragma unroll
    for (int r = 0; r < 16; ++r) za[r] = z[sidx(u + 256 * r)];
    twiddle16<1>(c2, w1, w4, w8, w12);
    dft16(za);  // za[q] = Z[u + 256 q]
  }
  {
    // column 256 - u: exp(-2 pi i (256 - u) r / 4096) = W16^r conj(w^r); the factor W16^r advances the outputs
    // by one: zb[q] = Z[cb + 256 ((q + 15) mod 16)] (also with eb = 128 for column 128)
    const float2 w1 = conjf2(g_w4096[eb]), w4 = conjf2(g_w4096[4 * eb]), w8 = conjf2(g_w4096[8 * eb]),
                 w12 = conjf2(g_w4096[12 * eb]);
#pragma unroll
    for (int r = 0; r < 16; ++r) zb[r] = z[sidx(cb + 256 * r)];
    twiddle16<1>(d2, w1, w4, w8, w12);
    dft16(zb);
  }
  float2* o = out + ((size_t)n * T + t0 + s) * PFB_H;
  if (u != 0) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {  // k = u + 256 q, 4096 - k = 256 - u + 256 (15 - q)
      float2 xk, xm;
      const float2 w = ws[(q & 7) * PFB_WLD + u];
      split_pair(za[q], zb[(16 - q) & 15], q < 8 ? w : mul_mi(w), xk, xm);
      o[u + 256 * q] = xk;
      o[PFB_H - u - 256 * q] = xm;
    }
  } else {
    o[0] = make_float2((za[0].x + za[0].y) * PFB_SCALE, 0.f);  // DC; the Nyquist bin (x - y) is not kept
    o[PFB_H / 2] = make_float2(za[8].x * PFB_SCALE, -za[8].y * PFB_SCALE);  // k = 2048: W^2048 = -i
#pragma unroll
    for (int q = 1; q < 8; ++q) {  // k = 256 q, 4096 - k = 256 (16 - q)
      float2 xk, xm;
      split_pair(za[q], za[16 - q], ws[q * PFB_WLD], xk, xm);
      o[256 * q] = xk;
      o[PFB_H - 256 * q] = xm;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {  // k = 128 + 256 q, 4096 - k = 128 + 256 (15 - q)
      float2 xk, xm;
      split_pair(zb[q + 1], zb[(16 - q) & 15], ws[q * PFB_WLD + 128], xk, xm);
      o[128 + 256 * q] = xk;
      o[PFB_H - 128 - 256 * q] = xm;
    }
  }
}

std::once_flag g_tw_once[64];
cudaError_t g_tw_err[64];

cudaError_t ensure_twiddles(int dev) {
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::call_once(g_tw_once[dev], [dev]() {
    float2 w1[PFB_H], w2[PFB_H / 2];
    for (int j = 0; j < PFB_H; ++j) {
      const double a1 = -2.0 * M_PI * j / 4096.0, a2 = -2.0 * M_PI * j / 8192.0;
      w1[j] = make_float2((float)std::cos(a1), (float)std::sin(a1));
      if (j < PFB_H / 2) w2[j] = make_float2((float)std::cos(a2), (float)std::sin(a2));
    }
    cudaError_t e = cudaMemcpyToSymbol(g_w4096, w1, sizeof(w1));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_w8192, w2, sizeof(w2));
    g_tw_err[dev] = e;
  });
  return g_tw_err[dev];
}

template <int PT>
cudaError_t launch_taps(const int8_t* d_adc, long long stride, int T, int P, const int* d_h, float2* d_out, dim3 grid,
                        cudaStream_t st) {
  const cudaError_t e = set_smem_limit(reinterpret_cast<const void*>(pfb_kernel<PT>), PFB_SMEM);
  if (e == cudaSuccess) pfb_kernel<PT><<<grid, PFB_NT, PFB_SMEM, st>>>(d_adc, stride, T, P, d_h, d_out);
  return e;
}

}  // namespace

cudaError_t launch_pfb(const int8_t* d_adc, long long stride, int N, int T, int P, const int* d_h, float2* d_out,
                       cudaStream_t st) {
  if ((long long)N * T == 0) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = ensure_twiddles(dev);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((T + PFB_SPB - 1) / PFB_SPB), (unsigned)N);
  // up to eight taps unrolled, every load of a point in flight at once (512 inputs x 8 spectra: 4 taps 82 us, 8 taps
  // 100); in the loop over taps 9 take 125, 16 take 155
  switch (P) {
    case 1: e = launch_taps<1>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 2: e = launch_taps<2>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 3: e = launch_taps<3>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 4: e = launch_taps<4>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 5: e = launch_taps<5>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 6: e = launch_taps<6>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 7: e = launch_taps<7>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    case 8: e = launch_taps<8>(d_adc, stride, T, P, d_h, d_out, grid, st); break;
    default: e = launch_taps<0>(d_adc, stride, T, P, d_h, d_out, grid, st);
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace corr
