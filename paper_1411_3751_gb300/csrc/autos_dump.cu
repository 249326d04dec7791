// Total-power (autocorrelation) kernel and the dump/format kernel.
#include "corr_internal.cuh"

namespace corr {
namespace {

// Autocorrelations A[f][n] += sum_t |x_{f,n}(t)|^2 (Sec. 2.6: total power of selected inputs at a high
// cadence) of blocks whose rows TMA does not take (the others: autos_tma.cu). A row t is M = C N neighbouring
// bytes; a thread keeps 16 of them (16 cells) and walks down t, four rows' loads in flight while four are added
// up, the 8 warps of a block taking every eighth row of the same 512 bytes; the warps' sums meet in shared memory and
// are added to the int64 sums by one thread a cell. Block b takes columns b % gx and run b / gx of the rows: t is
// split where the columns alone leave SMs idle and into runs whose 16-bit sums hold (the sums then meet in
// 64-bit atomics, exact in any order).
//
// A square of a 4-bit component x = m - 8 s (s the sign bit, m the low three) is m^2 or (8 - m)^2: a byte
// permute with the nibbles as selectors looks four of them up at once, the selectors' top bit making
// the other sign's entries zero (the permute then repeats the entry's top bit, clear in every entry). Two
// rows' squares (at most 64 each) fit a byte lane; then the halves of a sample are added into 16-bit lanes.
// (A dp4a a sample for the sums runs at a quarter of the other instructions' rate: 85 us at 512 inputs x 2400
// channels x 240 aligned samples, 77 so, 358 with one byte a load.)
constexpr int AU_NT = 256, AU_W = AU_NT / 32, AU_U = 4;

// squares of the four components in the low 16 bits of w (wx = w ^ 0x88888888), one byte each
__device__ __forceinline__ uint32_t squares4(uint32_t w, uint32_t wx) {
  uint32_t p, q;  // prmt's default mode; the intrinsic leaves the selectors' top bits undocumented
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(p) : "r"(0x09040100u), "r"(0x31241910u), "r"(w));
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(q) : "r"(0x19243140u), "r"(0x01040910u), "r"(wx));
  return p | q;
}

// acc[0], acc[1] (16-bit lanes, samples 0, 1 and 2, 3 of the words) += |x|^2 over the same word of two rows.
__device__ __forceinline__ void add_power4(uint32_t (&acc)[2], uint32_t w0, uint32_t w1) {
  const uint32_t x0 = w0 ^ 0x88888888u, x1 = w1 ^ 0x88888888u;
  const uint32_t lo = squares4(w0, x0) + squares4(w1, x1), hi = squares4(w0 >> 16, x0 >> 16) + squares4(w1 >> 16, x1 >> 16);
  acc[0] += (lo & 0x00FF00FFu) + ((lo >> 8) & 0x00FF00FFu);
  acc[1] += (hi & 0x00FF00FFu) + ((hi >> 8) & 0x00FF00FFu);
}
constexpr int AU_ROWS = AU_W * 504;  // rows a block takes at most: 504 samples of at most 128 a 16-bit lane

// The 16 bytes at any address p: the five aligned words around them, shifted together, or byte by byte where those
// words would leave the buffer [in, end).
__device__ __forceinline__ uint4 autos_load(const uint8_t* p, int nv, const uint8_t* in, const uint8_t* end) {
  const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3);
  const uint8_t* q = p - sh;
  uint32_t x[5] = {0u, 0u, 0u, 0u, 0u};
  if (nv == 16 && q >= in && q + 20 <= end) {
#pragma unroll
    for (int k = 0; k < 5; ++k) x[k] = __ldg(reinterpret_cast<const uint32_t*>(q) + k);
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = __funnelshift_r(x[k], x[k + 1], 8 * sh);
  } else {
    for (int k = 0; k < nv; ++k) x[k >> 2] |= (uint32_t)p[k] << (8 * (k & 3));
  }
  return make_uint4(x[0], x[1], x[2], x[3]);
}

__global__ void __launch_bounds__(AU_NT) autos_kernel(const uint8_t* __restrict__ in, long long M, int T, int rows,
                                                      unsigned gx, bool split, long long* __restrict__ autos) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned run = blockIdx.x / gx, bx = blockIdx.x - run * gx;
  const long long col = bx * 512LL + 16 * lane;
  const int nv = M - col >= 16 ? 16 : (M > col ? (int)(M - col) : 0);
  const int t_end = (int)min((long long)T, (run + 1LL) * rows);
  const uint8_t* end = in + (size_t)T * M;
  uint32_t acc[4][2] = {{0u, 0u}, {0u, 0u}, {0u, 0u}, {0u, 0u}};  // word k: its samples' sums in 16-bit lanes
  if (nv > 0) {
    // the next four rows' loads are in flight while four are added up
    // (long: the last steps of a row count near 2^31 would overflow an int)
    auto load = [&](uint4 (&w)[AU_U], long long t0) {
#pragma unroll
      for (int u = 0; u < AU_U; ++u) {
        const long long t = t0 + AU_W * u;
        w[u] = t < t_end ? autos_load(in + (size_t)t * M + col, nv, in, end) : make_uint4(0u, 0u, 0u, 0u);
      }
    };
    long long t0 = (long long)run * rows + warp;
    uint4 w[AU_U], nx[AU_U];
    load(w, t0);
    while (t0 < t_end) {
      t0 += AU_W * AU_U;
      load(nx, t0);
#pragma unroll
      for (int u = 0; u < AU_U; u += 2) {
        add_power4(acc[0], w[u].x, w[u + 1].x);
        add_power4(acc[1], w[u].y, w[u + 1].y);
        add_power4(acc[2], w[u].z, w[u + 1].z);
        add_power4(acc[3], w[u].w, w[u + 1].w);
      }
#pragma unroll
      for (int u = 0; u < AU_U; ++u) w[u] = nx[u];
    }
  }
  __shared__ __align__(16) int part[AU_W][512];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    *reinterpret_cast<int4*>(&part[warp][16 * lane + 4 * k]) =
        make_int4((int)(acc[k][0] & 0xFFFFu), (int)(acc[k][0] >> 16), (int)(acc[k][1] & 0xFFFFu), (int)(acc[k][1] >> 16));
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = threadIdx.x + AU_NT * h;
    const long long cell = bx * 512LL + i;
    if (cell >= M) break;
    long long sum = 0;
#pragma unroll
    for (int v = 0; v < AU_W; ++v) sum += part[v][i];
    if (!split)
      autos[cell] += sum;
    else
      atomicAdd(reinterpret_cast<unsigned long long*>(autos + cell), (unsigned long long)sum);
  }
}

// Dump: out[k] = fmt(acc[k]). CI64 copies, CF32 rounds to nearest float, CF32_NORM divides by the
// sample count in double and rounds to float. Contributions of the tensor path are held in the
// offset domain (u = x + 8 + 8i) and are mapped back here:
//   V = Vu - (8 - 8i) s_a - (8 + 8i) conj(s_c) + 128 T_off,   A = Au - 16 (Re s + Im s) + 128 T_off
// (s = per-input offset sums and T_off = samples accumulated through that path, per cadence).

// float((double)v / (double)n), the definition of CF32_NORM.
__device__ __forceinline__ float norm_exact(long long v, long long n) {
  return n > 0 ? __double2float_rn(__ddiv_rn(__ll2double_rn(v), (double)n)) : 0.f;
}

// v as a sum of two floats, hi = v rounded to nearest: the 16-bit halves enter as mantissas of 2^23, so there are
// no conversion instructions (with three of them a value the 512-input, 109-channel normalised dump took 165 us, not
// 97, which is what the plain float dump takes).
__device__ __forceinline__ void split32(int v, float& hi, float& lo) {
  const unsigned u = (unsigned)v ^ 0x80000000u;
  const float h = __fsub_rn(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7432)), 8388608.f + 32768.f);  // v >> 16
  const float l = __fsub_rn(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7410)), 8388608.f);            // v & 65535
  hi = __fmaf_rn(h, 65536.f, l);
  lo = __fsub_rn(l, __fmaf_rn(h, -65536.f, hi));
}

// The same value without FP64 arithmetic (a GB300 SM does about 2 FP64 operations per clock: with the
// FP64 division the 109-channel, 512-input normalised dump took 553 us, eight times its HBM time): v
// and 1 / n as sums of two floats, the product to about 2^-46 relative. If adding +-2^-44 to it does
// not change the rounded float, that float is the rounded exact quotient (and so the one the double
// division rounds to, whose error is 2^-53); else, about one value in 2^18, divide as defined.
__device__ __forceinline__ bool norm_quotient(float hi, float lo, float rh, float rl, float& q) {
  const float p = __fmul_rn(hi, rh);
  const float e = __fmaf_rn(lo, rh, __fmaf_rn(hi, rl, __fmaf_rn(hi, rh, -p)));
  const float d = __fmul_rn(fabsf(p), 5.6843418860808015e-14f);  // 2^-44
  q = __fadd_rn(p, __fadd_rn(e, d));
  return q == __fadd_rn(p, __fsub_rn(e, d));
}
__device__ __forceinline__ float norm_fast(long long v, long long n, float rh, float rl) {
  const float hi = __ll2float_rn(v), lo = __ll2float_rn(v - __float2ll_rn(hi));
  float q;
  return norm_quotient(hi, lo, rh, rl, q) ? q : norm_exact(v, n);
}
// Values that are 32-bit numbers, no fallback: false if the quotient is not certain or v is larger.
__device__ __forceinline__ bool norm_32(long long v, float rh, float rl, float& q) {
  float hi, lo;
  split32((int)v, hi, lo);
  return norm_quotient(hi, lo, rh, rl, q) && v == (long long)(int)v;
}

// float(v)
__device__ __forceinline__ float nearest(long long v) {
  return v == (long long)(int)v ? __int2float_rn((int)v) : __ll2float_rn(v);
}

// Sample count of a normalised dump: n for every cell with rh + rl = 1 / n, or (cells reset
// selectively) n - base[...] each.
struct DumpNorm {
  long long n;
  float rh, rl;
};

DumpNorm dump_norm(long long n) {
  const double inv = n > 0 ? 1.0 / (double)n : 0.0;
  DumpNorm d;
  d.n = n;
  d.rh = (float)inv;
  d.rl = (float)(inv - (double)d.rh);
  return d;
}

// One value in format FMT (CI64: long long, else float); ns = the cell's own count if HAS_BASE.
template <bool HAS_BASE>
__device__ __forceinline__ float as_float(long long v, int fmt, const DumpNorm& dn, long long ns) {
  if (fmt == CORR_FMT_CF32) return nearest(v);
  if (HAS_BASE) return norm_exact(v, ns);
  if (dn.n <= 0) return 0.f;
  float q;
  return norm_32(v, dn.rh, dn.rl, q) ? q : norm_fast(v, dn.n, dn.rh, dn.rl);
}

template <typename T>
__device__ __forceinline__ void put(void* out, long long k, long long v, int fmt, long long n_samples) {
  if (fmt == CORR_FMT_CI64) {
    static_cast<long long*>(out)[k] = v;
  } else if (fmt == CORR_FMT_CF32) {
    static_cast<float*>(out)[k] = __ll2float_rn(v);
  } else {
    static_cast<float*>(out)[k] = norm_exact(v, n_samples);
  }
}

// station pair index b -> (a, c) with b = a (a + 1) / 2 + c, a >= c; b < 2^31 - 2^15 (a <= 65534), so
// that (a + 1) (a + 2) < 2^32
__device__ __forceinline__ void pair_of(int b, int& sa, int& sc) {
  unsigned a = (unsigned)((sqrtf(8.0f * (float)b + 1.0f) - 1.0f) * 0.5f);
  while (a * (a + 1) / 2 > (unsigned)b) --a;
  while ((a + 1) * (a + 2) / 2 <= (unsigned)b) ++a;
  sa = (int)a;
  sc = b - (int)(a * (a + 1) / 2);
}

// Corrected value of cross cell `cell` (= f * B_s * P + b * P + pidx) from its raw int64 sums.
__device__ __forceinline__ void cross_value(const long long* __restrict__ acc, long long cell, long long f, int b,
                                            int pidx, const Shape2& g, long long& re, long long& im) {
  const longlong2 v2 = reinterpret_cast<const longlong2*>(acc)[cell];
  re = v2.x;
  im = v2.y;
  if (g.soff != nullptr && g.t_off != 0) {
    int sa, sc;
    pair_of(b, sa, sc);
    const long long a = (long long)sa * g.npol + pidx / g.npol;
    const long long c = (long long)sc * g.npol + pidx % g.npol;
    const longlong2 s_a = reinterpret_cast<const longlong2*>(g.soff)[f * g.N + a];
    const longlong2 s_c = reinterpret_cast<const longlong2*>(g.soff)[f * g.N + c];
    re += -8 * (s_a.x + s_a.y + s_c.x + s_c.y) + 128 * g.t_off;
    im += -8 * (s_a.y - s_a.x + s_c.x - s_c.y);
  }
}

__device__ __forceinline__ long long auto_value(const long long* __restrict__ acc, long long k, const Shape2& g) {
  long long v = acc[k];
  if (g.soff != nullptr && g.t_off != 0) {
    const longlong2 s = reinterpret_cast<const longlong2*>(g.soff)[k];
    v += -16 * (s.x + s.y) + 128 * g.t_off;  // A = Au - 16 (Re s + Im s) + 128 T
  }
  return v;
}

// NPOL neighbouring cells (16 bytes each) as one access: at NPOL = 2 the 256-bit forms, a whole 32-byte
// sector a thread. (Two 16-byte stores a thread write half sectors, which the L2 has to merge: the
// 200-input, 300-channel float dump took 205 us so, latency-bound at 0.9 TB/s.)
template <int NPOL>
__device__ __forceinline__ void load_cells(const longlong2* p, longlong2 (&v)[NPOL]) {
  if constexpr (NPOL == 2)
    asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(v[0].x), "=l"(v[0].y), "=l"(v[1].x), "=l"(v[1].y)
                 : "l"(p)
                 : "memory");
  else
    v[0] = *p;
}
template <int NPOL>
__device__ __forceinline__ void store_cells(longlong2* p, const longlong2 (&v)[NPOL]) {
  if constexpr (NPOL == 2)
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(v[0].x), "l"(v[0].y), "l"(v[1].x), "l"(v[1].y)
                 : "memory");
  else
    *p = v[0];
}

// Cross dump. A thread takes a unit = the NPOL products of one station pair and a-polarisation, i.e.
// NPOL neighbouring cells (one s_a and NPOL neighbouring s_c serve them; NPOL = 2: 32 bytes in, 32 or
// 16 out). blockIdx.y is the channel f0 + blockIdx.y, whose units are divided over gridDim.x blocks;
// [u0, u1) are the units dumped, numbered over all channels, the output indexed from u0 (vec: a unit's
// values leave in one store, the output is aligned to that). With ZERO the
// dumped cells restart from zero in the same pass (a separate memset wrote them once more and cost
// its launch), and if zero_soff the block, alone on its channel, zeroes the channel's offset sums too.
constexpr int DUMP_NT = 256;

template <int NPOL, bool ZERO, bool HAS_BASE>
__global__ void __launch_bounds__(DUMP_NT) dump_cross_kernel(long long* __restrict__ acc, long long u0, long long u1,
                                                             long long f0, void* __restrict__ out, int fmt, DumpNorm dn,
                                                             bool vec, Shape2 g, long long* zero_soff) {
  const long long f = f0 + blockIdx.y;
  const long long upc = g.Bs * NPOL;  // units per channel
  const long long first = f * upc;
  const unsigned r_begin = (unsigned)(u0 > first ? u0 - first : 0);
  const unsigned r_end = (unsigned)(u1 - first < upc ? u1 - first : upc);
  const bool corr = g.soff != nullptr && g.t_off != 0;
  const longlong2* s = reinterpret_cast<const longlong2*>(g.soff) + f * g.N;
  for (unsigned r = r_begin + blockIdx.x * DUMP_NT + threadIdx.x; r < r_end; r += gridDim.x * DUMP_NT) {
    const int b = (int)(NPOL == 2 ? r >> 1 : r);
    longlong2* cell = reinterpret_cast<longlong2*>(acc) + (first + r) * NPOL;
    longlong2 v[NPOL];
    load_cells<NPOL>(cell, v);
    if (corr) {
      int sa, sc;
      pair_of(b, sa, sc);
      const longlong2 s_a = s[NPOL * sa + (NPOL == 2 ? (int)(r & 1) : 0)];
#pragma unroll
      for (int q = 0; q < NPOL; ++q) {
        const longlong2 s_c = s[NPOL * sc + q];
        v[q].x += 128 * g.t_off - 8 * (s_a.x + s_a.y + s_c.x + s_c.y);
        v[q].y -= 8 * (s_a.y - s_a.x + s_c.x - s_c.y);
      }
    }
    const long long o = (first + r - u0) * NPOL;
    if (fmt == CORR_FMT_CI64) {
      if (vec) {
        store_cells<NPOL>(static_cast<longlong2*>(out) + o, v);
      } else {
#pragma unroll
        for (int q = 0; q < NPOL; ++q) {
          static_cast<long long*>(out)[2 * (o + q)] = v[q].x;
          static_cast<long long*>(out)[2 * (o + q) + 1] = v[q].y;
        }
      }
    } else {
      const long long ns = HAS_BASE ? dn.n - g.base[b] : dn.n;
      float w[2 * NPOL];
      // a unit's quotients together, one branch for all (a branch a value: 107 us instead of 97 as above)
      bool done = !HAS_BASE && fmt == CORR_FMT_CF32_NORM && dn.n > 0;
      if (done) {
#pragma unroll
        for (int q = 0; q < NPOL; ++q) {
          const bool re = norm_32(v[q].x, dn.rh, dn.rl, w[2 * q]), im = norm_32(v[q].y, dn.rh, dn.rl, w[2 * q + 1]);
          done = done && re && im;
        }
      }
      if (!done) {
#pragma unroll
        for (int q = 0; q < NPOL; ++q) {
          w[2 * q] = as_float<HAS_BASE>(v[q].x, fmt, dn, ns);
          w[2 * q + 1] = as_float<HAS_BASE>(v[q].y, fmt, dn, ns);
        }
      }
      if (!vec) {
#pragma unroll
        for (int q = 0; q < 2 * NPOL; ++q) static_cast<float*>(out)[2 * o + q] = w[q];
      } else if constexpr (NPOL == 2) {
        *reinterpret_cast<float4*>(static_cast<float*>(out) + 2 * o) = make_float4(w[0], w[1], w[2], w[3]);
      } else {
        *reinterpret_cast<float2*>(static_cast<float*>(out) + 2 * o) = make_float2(w[0], w[1]);
      }
    }
    if (ZERO) {
      // last, when the cells have arrived: zeroes stored behind loads still in flight made the pass
      // latency-bound (205 us instead of 40 at 200 inputs x 300 channels)
      longlong2 z[NPOL];
#pragma unroll
      for (int q = 0; q < NPOL; ++q) z[q] = make_longlong2(0, 0);
      store_cells<NPOL>(cell, z);
    }
  }
  if (ZERO && zero_soff) {
    __syncthreads();  // every thread has read the sums
    longlong2* z = reinterpret_cast<longlong2*>(zero_soff) + f * g.N;
    for (int i = threadIdx.x; i < g.N; i += DUMP_NT) z[i] = make_longlong2(0, 0);
  }
}

// Autos dump of elements [k0, k0 + n); with zero_soff (the offset sums of g) the dumped inputs' sums and
// offset sums restart from zero.
__global__ void dump_autos_kernel(long long* __restrict__ acc, long long k0, long long n, void* __restrict__ out,
                                  int fmt, DumpNorm dn, Shape2 g, long long* zero_soff) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
    const long long v = auto_value(acc, k0 + k, g);
    if (fmt == CORR_FMT_CI64)
      static_cast<long long*>(out)[k] = v;
    else if (g.base)
      static_cast<float*>(out)[k] = as_float<true>(v, fmt, dn, dn.n - g.base[(k0 + k) % g.N]);
    else
      static_cast<float*>(out)[k] = as_float<false>(v, fmt, dn, dn.n);
    if (zero_soff) {
      acc[k0 + k] = 0;
      reinterpret_cast<longlong2*>(zero_soff)[k0 + k] = make_longlong2(0, 0);
    }
  }
}

// Selective dump (Sec. 2.6: selected cells are dumped and zeroed at their own cadence). Cross: unit =
// (channel, list pair k >= l, product p q) -> sum x_{st[k] p} conj(x_{st[l] q}); the stored cell is
// (st[k] p, st[l] q) when st[k] >= st[l], else its conjugate (st[l] q, st[k] p). Autos: unit =
// (channel, list position k, pol p) -> input st[k] n_pol + p. A reset stores minus the corrected
// value's offset-domain correction, acc := acc - value, so the corrected value restarts from zero
// while the shared offset sums keep integrating (the correction is affine in them).
__global__ void dump_select_kernel(long long* __restrict__ acc, const int* __restrict__ st, int n_st, int f0, int nf,
                                   void* __restrict__ out, int fmt, long long n_samples, int reset, Shape2 g) {
  if (g.autos) {
    const long long per = (long long)n_st * g.npol;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < (long long)nf * per;
         u += (long long)gridDim.x * blockDim.x) {
      const long long fl = u / per;
      const int r = (int)(u - fl * per);
      const int i = st[r / g.npol] * g.npol + r % g.npol;
      const long long k = (f0 + fl) * g.N + i;
      const long long v = auto_value(acc, k, g);
      put<void>(out, u, v, fmt, g.base ? n_samples - g.base[i] : n_samples);
      if (reset) acc[k] -= v;
    }
    return;
  }
  const long long npairs = (long long)n_st * (n_st + 1) / 2;
  const long long per = npairs * g.P;
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < (long long)nf * per;
       u += (long long)gridDim.x * blockDim.x) {
    const long long fl = u / per;
    const int r = (int)(u - fl * per);
    const int pr = r / g.P, pidx = r % g.P;
    int k, l;
    pair_of(pr, k, l);
    const int a = st[k], c = st[l], p = pidx / g.npol, q = pidx % g.npol;
    const bool swap = a < c;
    const int sa = swap ? c : a, sc = swap ? a : c;
    const int sp = swap ? q * g.npol + p : pidx;  // stored product index
    const int b = sa * (sa + 1) / 2 + sc;
    const long long f = f0 + fl;
    const long long cell = (f * g.Bs + b) * g.P + sp;
    long long re, im;
    cross_value(acc, cell, f, b, sp, g, re, im);
    const long long ns = g.base ? n_samples - g.base[b] : n_samples;
    put<void>(out, 2 * u, re, fmt, ns);
    put<void>(out, 2 * u + 1, swap ? -im : im, fmt, ns);
    if (reset) {
      acc[2 * cell] -= re;
      acc[2 * cell + 1] -= im;
    }
  }
}

__global__ void set_base_kernel(long long* __restrict__ base, const int* __restrict__ st, int n_st, long long value,
                                int npol, int autos) {
  const long long n = autos ? (long long)n_st * npol : (long long)n_st * (n_st + 1) / 2;
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x) {
    if (autos) {
      base[st[u / npol] * npol + u % npol] = value;
    } else {
      int k, l;
      pair_of((int)u, k, l);
      const int a = st[k] > st[l] ? st[k] : st[l], c = st[k] > st[l] ? st[l] : st[k];
      base[a * (a + 1) / 2 + c] = value;
    }
  }
}

}  // namespace

cudaError_t launch_autos(const Shape& s, const uint8_t* d_in, int T_blk, long long* d_autos, cudaStream_t st) {
  if (T_blk == 0) return cudaSuccess;
  const long long M = (long long)s.C * s.N;
  const long long gx = (M + 511) / 512;
  // rows per block: all of them while the columns fill the GPU (four blocks an SM), else at least 64 (8 a
  // warp, one step of loads); at most AU_ROWS
  const long long want = (4LL * sm_count() + gx - 1) / gx;
  long long rows = ((long long)T_blk + want - 1) / want;
  if (rows < 64) rows = 64;
  if (rows > AU_ROWS) rows = AU_ROWS;
  if (rows > T_blk) rows = T_blk;
  const long long runs = (T_blk + rows - 1) / rows;
  const unsigned grid = (unsigned)(gx * runs);
  autos_kernel<<<grid, AU_NT, 0, st>>>(d_in, M, T_blk, (int)rows, (unsigned)gx, runs > 1, d_autos);
  return cudaGetLastError();
}

cudaError_t launch_dump_select(long long* d_acc, const int* d_st, int n_st, int f0, int nf, void* d_out, int fmt,
                               long long n_samples, int reset, const Shape2& g, cudaStream_t st) {
  const long long units = (long long)nf * (g.autos ? (long long)n_st * g.npol : (long long)n_st * (n_st + 1) / 2 * g.P);
  if (units == 0) return cudaSuccess;
  long long blocks = (units + 255) / 256;
  if (blocks > (long long)sm_count() * 32) blocks = (long long)sm_count() * 32;
  dump_select_kernel<<<(unsigned)blocks, 256, 0, st>>>(d_acc, d_st, n_st, f0, nf, d_out, fmt, n_samples, reset, g);
  return cudaGetLastError();
}

cudaError_t launch_set_base(long long* d_base, const int* d_st, int n_st, long long value, const Shape2& g,
                            cudaStream_t st) {
  const long long n = g.autos ? (long long)n_st * g.npol : (long long)n_st * (n_st + 1) / 2;
  long long blocks = (n + 255) / 256;
  if (blocks > (long long)sm_count() * 8) blocks = (long long)sm_count() * 8;
  if (blocks == 0) return cudaSuccess;
  set_base_kernel<<<(unsigned)blocks, 256, 0, st>>>(d_base, d_st, n_st, value, g.npol, g.autos);
  return cudaGetLastError();
}

cudaError_t launch_dump(long long* d_acc, long long n_elems, void* d_out, int fmt, long long n_samples, long long k_base,
                        const Shape2& g, long long* zero_soff, bool zero, bool* soff_zeroed, cudaStream_t st) {
  *soff_zeroed = false;
  if (n_elems == 0) return cudaSuccess;
  const DumpNorm dn = dump_norm(n_samples);
  if (g.autos) {
    long long blocks = (n_elems + 255) / 256;
    if (blocks > (long long)sm_count() * 32) blocks = (long long)sm_count() * 32;
    dump_autos_kernel<<<(unsigned)blocks, 256, 0, st>>>(d_acc, k_base, n_elems, d_out, fmt, dn, g, zero ? zero_soff : nullptr);
    *soff_zeroed = zero;
    return cudaGetLastError();
  }
  const long long upc = g.Bs * g.npol, u0 = k_base / 2 / g.npol, u1 = u0 + n_elems / 2 / g.npol;
  const long long f0 = u0 / upc, f1 = (u1 - 1) / upc;
  // blocks per channel: one (which may then zero the channel's offset sums) up to 16 units a thread,
  // else 4 units a thread
  const bool whole = upc <= 16 * DUMP_NT;
  const long long bx = whole ? 1 : (upc + 4 * DUMP_NT - 1) / (4 * DUMP_NT);
  const dim3 grid((unsigned)bx, (unsigned)(f1 - f0 + 1));
  const bool zs = zero && whole && u0 == f0 * upc && u1 == (f1 + 1) * upc;
  long long* z = zs ? zero_soff : nullptr;
  *soff_zeroed = zs;
  const bool base = g.base != nullptr;
  const bool vec = reinterpret_cast<uintptr_t>(d_out) % ((fmt == CORR_FMT_CI64 ? 16 : 8) * g.npol) == 0;
#define DUMP_CROSS(NP, ZE, BA) dump_cross_kernel<NP, ZE, BA><<<grid, DUMP_NT, 0, st>>>(d_acc, u0, u1, f0, d_out, fmt, dn, vec, g, z)
  if (g.npol == 2) {
    if (zero) {
      if (base) DUMP_CROSS(2, true, true); else DUMP_CROSS(2, true, false);
    } else {
      if (base) DUMP_CROSS(2, false, true); else DUMP_CROSS(2, false, false);
    }
  } else {
    if (zero) {
      if (base) DUMP_CROSS(1, true, true); else DUMP_CROSS(1, true, false);
    } else {
      if (base) DUMP_CROSS(1, false, true); else DUMP_CROSS(1, false, false);
    }
  }
#undef DUMP_CROSS
  return cudaGetLastError();
}

}  // namespace corr
