// Kernels of the dedispersion + single-pulse-search path (sm_103a), except the tiled
// dedispersion kernel (dd_dedisp.cu).
//
//   k_shift_table : FP64 delay table, one IEEE operation at a time (Sec. 3 DM plan)
//   k_corner_turn : time-major uint8 spectra -> channel-major ring (Sec. 1 time chunks)
//   k_decimate    : exact x2 time decimation levels, uint8/uint16 -> uint16
//   k_dedisp_naive: one thread per output sample (reference-shaped; testing aid)
//   k_moments     : exact S1 / 128-bit S2 of each series window (Sec. 2.2)
//   k_sps         : boxcar SNR over prefix sums + block peak finding (Sec. 2.2)
#include <math.h>

#include <algorithm>
#include <climits>
#include <type_traits>

#include "dd_internal.h"

namespace ddk {

// ------------------------------------------------------------------ delay table

__constant__ ShiftRange c_ranges[kMaxRanges];

__global__ void k_shift_table(const double* __restrict__ freqs, int32_t nchans, int32_t cpad,
                              double fref, double tsamp, int32_t nranges, int32_t total_rows,
                              int32_t* __restrict__ shifts, int32_t* __restrict__ err) {
  const int64_t total = (int64_t)total_rows * cpad;
  // k_DM = 4.148808e3 s MHz^2 pc^-1 cm^3 (textbook cold-plasma constant).
  const double kdm = 4.148808e3;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t row = (int32_t)(e / cpad);
    const int32_t c = (int32_t)(e - (int64_t)row * cpad);
    int r = 0;
    while (r + 1 < nranges && row >= c_ranges[r + 1].row0) ++r;
    const ShiftRange R = c_ranges[r];
    int32_t s = 0;
    {
      // Padding channels (c >= nchans, all-zero data) repeat the last channel's delay, so they
      // add no delay classes of their own to the last channel group.
      const int32_t cc = c < nchans ? c : nchans - 1;
      // dm = start + i*step; a = 1/(f*f); b = 1/(fref*fref); tau = (k*dm)*(a-b);
      // x = tau/(tsamp*d) + 0.5; s = floor(x).  Explicit round-to-nearest intrinsics: no FMA.
      const double dm = __dadd_rn(R.dm_start, __dmul_rn((double)(row - R.row0), R.dm_step));
      const double f = freqs[cc];
      const double a = __ddiv_rn(1.0, __dmul_rn(f, f));
      const double b = __ddiv_rn(1.0, __dmul_rn(fref, fref));
      const double tau = __dmul_rn(__dmul_rn(kdm, dm), __dsub_rn(a, b));
      const double x = __dadd_rn(__ddiv_rn(tau, __dmul_rn(tsamp, (double)R.decimation)), 0.5);
      const double fl = floor(x);
      if (!(fl >= 0.0 && fl <= 2147483647.0)) {
        atomicOr(err, 1);
        s = 0;
      } else {
        s = (int32_t)fl;
      }
    }
    shifts[e] = s;
  }
}

cudaError_t launch_shift_table(const double* freqs, int32_t nchans, int32_t cpad, double fref,
                               double tsamp, const ShiftRange* ranges, int32_t nranges,
                               int32_t total_rows, int32_t* shifts, int32_t* err,
                               cudaStream_t st) {
  cudaError_t e = cudaMemcpyToSymbolAsync(c_ranges, ranges, sizeof(ShiftRange) * nranges, 0,
                                          cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  const int64_t total = (int64_t)total_rows * cpad;
  int64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (blocks < 1) blocks = 1;
  k_shift_table<<<(unsigned)blocks, 256, 0, st>>>(freqs, nchans, cpad, fref, tsamp, nranges,
                                                  total_rows, shifts, err);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ corner turn

// 64 samples x 64 channels per CTA: 16 channels of one spectrum per thread into shared memory, a
// 4x4 byte transpose in registers (PRMT), 4-byte stores of channel rows. ALIGNED: every spectrum
// starts 16-byte aligned (nchans a multiple of 16), one 16-byte load per thread. Otherwise five
// aligned words and funnel shifts, or single bytes where a word would leave the chunk. Bound by
// memory; one byte per thread, which any layout took before, wrote single bytes a row apart
// (1001 channels x 49984 samples, with the other small launches: 3.7 -> 3.0 ms a chunk).
template <bool ALIGNED>
__global__ void __launch_bounds__(256) k_corner_turn(const uint8_t* __restrict__ in, int64_t n,
                                                     int32_t nchans, uint8_t* __restrict__ ring,
                                                     int64_t stride, int64_t col0) {
  __shared__ uint32_t S[64][17];
  const int tid = threadIdx.x;
  const int64_t t0 = (int64_t)blockIdx.x * 64;
  const int32_t c0 = blockIdx.y * 64;
  {
    const int r = tid >> 2, q = tid & 3;
    const int64_t t = t0 + r;
    const int32_t c = c0 + 16 * q;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (t < n && c < nchans) {
      if (ALIGNED) {
        v = __ldg(reinterpret_cast<const uint4*>(in + t * nchans + c));
      } else {
        const uint8_t* p = in + t * nchans + c;
        const uint32_t ph = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 3);
        const uint8_t* w = p - ph;
        if (w >= in && w + 20 <= in + n * nchans) {
          const uint32_t* x = reinterpret_cast<const uint32_t*>(w);
          const uint32_t x0 = __ldg(x), x1 = __ldg(x + 1), x2 = __ldg(x + 2), x3 = __ldg(x + 3),
                         x4 = __ldg(x + 4);
          v.x = __funnelshift_r(x0, x1, 8 * ph);
          v.y = __funnelshift_r(x1, x2, 8 * ph);
          v.z = __funnelshift_r(x2, x3, 8 * ph);
          v.w = __funnelshift_r(x3, x4, 8 * ph);
        } else {
          uint32_t o[4] = {0, 0, 0, 0};
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if (c + k < nchans) o[k / 4] |= (uint32_t)p[k] << (8 * (k % 4));
          v = make_uint4(o[0], o[1], o[2], o[3]);
        }
      }
    }
    S[r][4 * q + 0] = v.x;
    S[r][4 * q + 1] = v.y;
    S[r][4 * q + 2] = v.z;
    S[r][4 * q + 3] = v.w;
  }
  __syncthreads();
  const int tb = tid & 15, cw = tid >> 4;
  const uint32_t w0 = S[4 * tb + 0][cw], w1 = S[4 * tb + 1][cw];
  const uint32_t w2 = S[4 * tb + 2][cw], w3 = S[4 * tb + 3][cw];
  const uint32_t a0 = __byte_perm(w0, w1, 0x5140), a1 = __byte_perm(w0, w1, 0x7362);
  const uint32_t a2 = __byte_perm(w2, w3, 0x5140), a3 = __byte_perm(w2, w3, 0x7362);
  uint32_t o[4];
  o[0] = __byte_perm(a0, a2, 0x5410);
  o[1] = __byte_perm(a0, a2, 0x7632);
  o[2] = __byte_perm(a1, a3, 0x5410);
  o[3] = __byte_perm(a1, a3, 0x7632);
  const int64_t t = t0 + 4 * tb;
  if (t >= n) return;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int32_t c = c0 + 4 * cw + j;
    if (c < nchans)
      *reinterpret_cast<uint32_t*>(ring + (int64_t)c * stride + col0 + t) = o[j];
  }
}

// The ring's rows and the column of the first sample are 4-byte aligned (both 256-byte aligned
// in every plan); the last word of a chunk may write up to 3 zeros past it, into row slack.
cudaError_t launch_corner_turn(const uint8_t* in, int64_t n, int32_t nchans, uint8_t* ring,
                               int64_t ring_stride, int64_t col0, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (ring_stride % 4 || col0 % 4 || ((uintptr_t)ring & 3)) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((n + 63) / 64), (unsigned)((nchans + 63) / 64));
  if (nchans % 16 == 0 && ((uintptr_t)in & 15) == 0)
    k_corner_turn<true><<<grid, 256, 0, st>>>(in, n, nchans, ring, ring_stride, col0);
  else
    k_corner_turn<false><<<grid, 256, 0, st>>>(in, n, nchans, ring, ring_stride, col0);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ decimation

// Levels x2 .. x2^LEVELS of the uint8 ring in one pass: 16 samples per thread, 8, 4, 2 and 1 sums
// of them stored. Bound by memory: the ring is read once and each level written once, 2.9 bytes
// per sample with four levels against 4.6 when every level read the one before. Channels c =
// blockIdx.y, blockIdx.y + gridDim.y, ... (a grid dimension holds at most 65535 of them). The
// last thread of a row may read and write past the data, into the rows' slack.
struct DecimateArgs {
  const uint8_t* in;
  int64_t in_stride;
  uint16_t* out[4];
  int64_t out_stride[4];
  int64_t n;  // samples
  int32_t cpad;
};

template <int LEVELS>
__global__ void __launch_bounds__(256) k_decimate_u8(const DecimateArgs a) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (16 * k >= a.n) return;
  for (int64_t c = blockIdx.y; c < a.cpad; c += gridDim.y) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(a.in + c * a.in_stride + 16 * k));
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t p[4];  // level 1: two 16-bit sums a word
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = (w[i] & 0x00FF00FFu) + ((w[i] >> 8) & 0x00FF00FFu);
    *reinterpret_cast<uint4*>(a.out[0] + c * a.out_stride[0] + 8 * k) =
        make_uint4(p[0], p[1], p[2], p[3]);
    if (LEVELS < 2) continue;
    uint32_t q[2];  // level 2: four sums (below 2^10) in two words
#pragma unroll
    for (int i = 0; i < 2; ++i)
      q[i] = ((p[2 * i] & 0xFFFFu) + (p[2 * i] >> 16)) |
             ((p[2 * i + 1] & 0xFFFFu) + (p[2 * i + 1] >> 16)) << 16;
    *reinterpret_cast<uint2*>(a.out[1] + c * a.out_stride[1] + 4 * k) = make_uint2(q[0], q[1]);
    if (LEVELS < 3) continue;
    const uint32_t r = ((q[0] & 0xFFFFu) + (q[0] >> 16)) | ((q[1] & 0xFFFFu) + (q[1] >> 16)) << 16;
    *reinterpret_cast<uint32_t*>(a.out[2] + c * a.out_stride[2] + 2 * k) = r;
    if (LEVELS < 4) continue;
    a.out[3][c * a.out_stride[3] + k] = (uint16_t)((r & 0xFFFFu) + (r >> 16));
  }
}

// out[c][m] = in[c][2m] + in[c][2m+1] of a uint16 level (beyond x16), four outputs per thread.
__global__ void k_decimate_u16(const uint16_t* __restrict__ in, int64_t in_stride,
                               uint16_t* __restrict__ out, int64_t out_stride, int64_t n_out,
                               int32_t cpad) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (4 * k >= n_out) return;
  for (int64_t c = blockIdx.y; c < cpad; c += gridDim.y) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(in + c * in_stride + 8 * k));
    const uint32_t s0 = (v.x & 0xFFFFu) + (v.x >> 16), s1 = (v.y & 0xFFFFu) + (v.y >> 16);
    const uint32_t s2 = (v.z & 0xFFFFu) + (v.z >> 16), s3 = (v.w & 0xFFFFu) + (v.w >> 16);
    uint2 o;
    o.x = s0 | (s1 << 16);
    o.y = s2 | (s3 << 16);
    *reinterpret_cast<uint2*>(out + c * out_stride + 4 * k) = o;
  }
}

cudaError_t launch_decimate(const uint8_t* in, int64_t in_stride, uint16_t* const* out,
                            const int64_t* out_stride, int levels, int32_t cpad, int64_t n,
                            cudaStream_t st, int* launches) {
  *launches = 0;
  if (n <= 0 || levels < 1) return cudaSuccess;
  DecimateArgs a;
  a.in = in;
  a.in_stride = in_stride;
  const int first = std::min(levels, 4);
  for (int l = 0; l < 4; ++l) {
    a.out[l] = l < first ? out[l] : nullptr;
    a.out_stride[l] = l < first ? out_stride[l] : 0;
  }
  a.n = n;
  a.cpad = cpad;
  const dim3 grid((unsigned)((n + 16 * 256 - 1) / (16 * 256)), (unsigned)std::min(cpad, 65535));
  if (first == 1) k_decimate_u8<1><<<grid, 256, 0, st>>>(a);
  else if (first == 2) k_decimate_u8<2><<<grid, 256, 0, st>>>(a);
  else if (first == 3) k_decimate_u8<3><<<grid, 256, 0, st>>>(a);
  else k_decimate_u8<4><<<grid, 256, 0, st>>>(a);
  *launches = 1;
  for (int l = 4; l < levels; ++l) {
    const int64_t n_out = n >> (l + 1);
    if (n_out <= 0) break;
    const dim3 g((unsigned)(((n_out + 3) / 4 + 255) / 256), (unsigned)std::min(cpad, 65535));
    k_decimate_u16<<<g, 256, 0, st>>>(out[l - 1], out_stride[l - 1], out[l], out_stride[l], n_out,
                                      cpad);
    *launches += 1;
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------ naive dedispersion

template <typename T>
__global__ void k_dedisp_naive(const T* __restrict__ xd, int64_t stride, int32_t cpad, int64_t m0,
                               int64_t nout, const int32_t* __restrict__ shifts,
                               int32_t* __restrict__ y, int64_t y_stride) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t i = blockIdx.y;
  if (j >= nout) return;
  const int32_t* s = shifts + (int64_t)i * cpad;
  int32_t acc = 0;
  for (int32_t c = 0; c < cpad; ++c) acc += (int32_t)xd[(int64_t)c * stride + m0 + j + s[c]];
  y[(int64_t)i * y_stride + j] = acc;
}

cudaError_t launch_dedisp_naive(const DedispRange& r, int32_t cpad, cudaStream_t st) {
  if (r.nout <= 0 || r.n_trials <= 0) return cudaSuccess;
  dim3 grid((unsigned)((r.nout + 255) / 256), (unsigned)r.n_trials);
  if (r.is_u16)
    k_dedisp_naive<uint16_t><<<grid, 256, 0, st>>>(static_cast<const uint16_t*>(r.xd), r.xd_stride,
                                                   cpad, r.m0, r.nout, r.shifts, r.y, r.y_stride);
  else
    k_dedisp_naive<uint8_t><<<grid, 256, 0, st>>>(static_cast<const uint8_t*>(r.xd), r.xd_stride,
                                                  cpad, r.m0, r.nout, r.shifts, r.y, r.y_stride);
  return cudaGetLastError();
}

// Direct kernel: for ranges the tiled kernel cannot take (delay classes beyond its tables, as with
// coarse channels, or decimation above x16) whose delays also spread too far over 64 trials for
// the staged kernel's shared memory (dd_dedisp.cu). A CTA of 8 warps owns 16
// consecutive trials x 512 outputs; a warp takes 2 trials, lane l the 4-sample groups
// 4l + 128g (g = 0..3) of both. Per channel a lane reads, through the read-only cache, the two
// aligned 32-bit words holding its 4 samples and funnel-shifts them into place (the shift is
// the same in every lane of the warp: it depends only on m0 + delay). uint8 samples are added
// in 16-bit SWAR lanes (even / odd samples), flushed to 32-bit sums every 256 channels
// (256 x 255 < 2^16); uint16 samples (up to 255 x 256) are added to 32-bit sums directly.
constexpr int kDirectTrials = 16;
constexpr int kDirectTile = 512;

template <typename T>
__global__ void __launch_bounds__(256) k_dedisp_direct(const T* __restrict__ xd, int64_t stride,
                                                       int32_t cpad, int64_t m0, int64_t nout,
                                                       int32_t n_trials,
                                                       const int32_t* __restrict__ shifts,
                                                       int32_t* __restrict__ y, int64_t y_stride) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t tbase = blockIdx.x * kDirectTrials + 2 * warp;
  if (tbase >= n_trials) return;  // whole warp
  const int ntr = min(2, n_trials - tbase);
  const int64_t j0 = (int64_t)blockIdx.y * kDirectTile;
  uint32_t acc[2][4][4];  // [trial][group g][sample e]
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[q][g][e] = 0;
  const char* base = reinterpret_cast<const char*>(xd);
  const int64_t row_bytes = stride * (int64_t)sizeof(T);
  for (int32_t c0 = 0; c0 < cpad; c0 += 256) {
    uint32_t ev[2][4], od[2][4];  // uint8 path: packed 16-bit sums of samples (0,2) and (1,3)
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int g = 0; g < 4; ++g) ev[q][g] = od[q][g] = 0;
    const int32_t c1 = min(cpad, c0 + 256);
    for (int32_t c = c0; c < c1; ++c) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q < ntr) {
          const int64_t s = __ldg(shifts + (int64_t)(tbase + q) * cpad + c);
          // byte address of this lane's first sample of group 0
          const int64_t b = (int64_t)c * row_bytes + (m0 + j0 + s + 4 * lane) * (int64_t)sizeof(T);
          const uint32_t sh = (uint32_t)(b & 3) * 8u;
          const uint32_t* wp = reinterpret_cast<const uint32_t*>(base + (b & ~(int64_t)3));
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            if (sizeof(T) == 1) {
              const uint32_t* p = wp + 32 * g;  // 128 samples further per group
              const uint32_t v = __funnelshift_r(__ldg(p), __ldg(p + 1), sh);
              ev[q][g] += v & 0x00FF00FFu;
              od[q][g] += __byte_perm(v, 0, 0x4341);
            } else {
              const uint32_t* p = wp + 64 * g;
              const uint32_t w0 = __ldg(p), w1 = __ldg(p + 1), w2 = __ldg(p + 2);
              const uint32_t v0 = __funnelshift_r(w0, w1, sh), v1 = __funnelshift_r(w1, w2, sh);
              acc[q][g][0] += v0 & 0xFFFFu;
              acc[q][g][1] += v0 >> 16;
              acc[q][g][2] += v1 & 0xFFFFu;
              acc[q][g][3] += v1 >> 16;
            }
          }
        }
      }
    }
    if (sizeof(T) == 1) {
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          acc[q][g][0] += ev[q][g] & 0xFFFFu;
          acc[q][g][2] += ev[q][g] >> 16;
          acc[q][g][1] += od[q][g] & 0xFFFFu;
          acc[q][g][3] += od[q][g] >> 16;
        }
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (q < ntr) {
      int32_t* yr = y + (int64_t)(tbase + q) * y_stride;
#pragma unroll
      for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int64_t j = j0 + 128 * g + 4 * lane + e;
          if (j < nout) yr[j] = (int32_t)acc[q][g][e];
        }
    }
  }
}

cudaError_t launch_dedisp_direct(const DedispRange& r, int32_t cpad, cudaStream_t st) {
  if (r.nout <= 0 || r.n_trials <= 0) return cudaSuccess;
  dim3 grid((unsigned)((r.n_trials + kDirectTrials - 1) / kDirectTrials),
            (unsigned)((r.nout + kDirectTile - 1) / kDirectTile));
  if (r.is_u16)
    k_dedisp_direct<uint16_t><<<grid, 256, 0, st>>>(static_cast<const uint16_t*>(r.xd),
                                                    r.xd_stride, cpad, r.m0, r.nout, r.n_trials,
                                                    r.shifts, r.y, r.y_stride);
  else
    k_dedisp_direct<uint8_t><<<grid, 256, 0, st>>>(static_cast<const uint8_t*>(r.xd), r.xd_stride,
                                                   cpad, r.m0, r.nout, r.n_trials, r.shifts, r.y,
                                                   r.y_stride);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ moments

struct U128 {
  unsigned long long lo, hi;
};

__device__ __forceinline__ U128 add128(U128 a, U128 b) {
  U128 r;
  r.lo = a.lo + b.lo;
  r.hi = a.hi + b.hi + (r.lo < a.lo ? 1ull : 0ull);
  return r;
}

// One CTA per trial; 16-byte loads, four in flight per thread (one int a load when the row is not
// 16-byte aligned). The squares of two int32 values sum below 2^64 before the 128-bit add.
__global__ void __launch_bounds__(256) k_moments(const int32_t* __restrict__ y, int64_t n,
                                                 int64_t stride, Moments* __restrict__ mom) {
  const int32_t i = blockIdx.x;
  const int32_t* yi = y + (int64_t)i * stride;
  unsigned long long s1 = 0;
  U128 s2 = {0, 0};
  auto add2 = [&](int32_t p, int32_t q) {
    s1 += (unsigned long long)((int64_t)p + q);
    s2 = add128(s2, U128{(unsigned long long)((int64_t)p * p) + (unsigned long long)((int64_t)q * q), 0});
  };
  int64_t j = 0;  // the first sample left to the one-int loop
  if ((reinterpret_cast<uintptr_t>(yi) & 15) == 0) {
    const int4* v = reinterpret_cast<const int4*>(yi);
    const int64_t n4 = n / 4;
    int64_t k = threadIdx.x;
    for (; k + 768 < n4; k += 1024) {
      const int4 a = __ldg(v + k), b = __ldg(v + k + 256), c = __ldg(v + k + 512),
                 d = __ldg(v + k + 768);
      add2(a.x, a.y), add2(a.z, a.w), add2(b.x, b.y), add2(b.z, b.w);
      add2(c.x, c.y), add2(c.z, c.w), add2(d.x, d.y), add2(d.z, d.w);
    }
    for (; k < n4; k += 256) {
      const int4 a = __ldg(v + k);
      add2(a.x, a.y), add2(a.z, a.w);
    }
    j = 4 * n4;
  }
  for (j += threadIdx.x; j < n; j += blockDim.x) add2(__ldg(yi + j), 0);
  __shared__ unsigned long long sh[3][8];
  for (int off = 16; off > 0; off >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, off);
    U128 o;
    o.lo = __shfl_xor_sync(0xffffffffu, s2.lo, off);
    o.hi = __shfl_xor_sync(0xffffffffu, s2.hi, off);
    s2 = add128(s2, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    sh[0][w] = s1;
    sh[1][w] = s2.lo;
    sh[2][w] = s2.hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = 0;
    U128 b = {0, 0};
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
      a += sh[0][k];
      b = add128(b, U128{sh[1][k], sh[2][k]});
    }
    mom[i].s1 = a;
    mom[i].s2lo = b.lo;
    mom[i].s2hi = b.hi;
    mom[i].pad = 0;
  }
}

cudaError_t launch_moments(const int32_t* y, int32_t ntr, int64_t n, int64_t stride, Moments* mom,
                           cudaStream_t st) {
  if (ntr <= 0) return cudaSuccess;
  k_moments<<<ntr, 256, 0, st>>>(y, n, stride, mom);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ single pulse search

// Correctly rounded unsigned 128-bit -> double: the top 64 significant bits with a sticky bit
// for everything below, converted with round-to-nearest-even, then scaled by a power of two.
__device__ __forceinline__ double u128_to_f64(unsigned long long hi, unsigned long long lo) {
  if (hi == 0) return __ull2double_rn(lo);
  const int lz = __clzll((long long)hi);
  const int sh = 64 - lz;  // 1..64
  unsigned long long top, sticky;
  if (sh == 64) {
    top = hi;
    sticky = lo != 0;
  } else {
    top = (hi << lz) | (lo >> sh);
    sticky = (lo << lz) != 0;
  }
  return ldexp(__ull2double_rn(top | sticky), sh);
}

// sqrt(n*S2 - S1^2) of a window's moments, V = n*S2 - S1^2 formed exactly in 128 bits (S1 >= 0
// because every series value is a sum of non-negative samples) and rounded once to FP64; 0 for a
// constant series.
__device__ __forceinline__ double window_sqrt_var(const Moments& m, long long n) {
  const unsigned long long un = (unsigned long long)n, us1 = m.s1;
  const unsigned long long p_lo = un * m.s2lo;
  const unsigned long long p_hi = __umul64hi(un, m.s2lo) + un * m.s2hi;
  const unsigned long long q_lo = us1 * us1, q_hi = __umul64hi(us1, us1);
  const unsigned long long v_lo = p_lo - q_lo;
  const unsigned long long v_hi = p_hi - q_hi - (p_lo < q_lo ? 1ull : 0ull);
  if (v_lo == 0 && v_hi == 0) return 0.0;
  return sqrt(u128_to_f64(v_hi, v_lo));
}

// SNR >= thr  <=>  B >= (w*S1 + thr*den) / n. The bound keeps a margin of 2 + 1e-9 relative so
// that rounding in this estimate can never reject a boxcar sum the exact test accepts; as a
// uint32 bound on boxcar sums (< 2^31): at or below 0 every sum passes, above 2^32 - 1 none.
__device__ __forceinline__ uint32_t window_bound(int w, long long s1, double thr, double den,
                                                 long long n) {
  const double t = ((double)w * (double)s1 + thr * den) / (double)n;
  const double tl = t - 2.0 - 1e-9 * fabs(t);
  return tl <= 0.0 ? 0u : (tl >= 4294967295.0 ? 0xFFFFFFFFu : (uint32_t)floor(tl));
}

constexpr int kSpsThreads = 256;
constexpr int kSpsWarps = kSpsThreads / 32;
constexpr int kSpsPass = 512;                     // window samples per warp and pass
constexpr int kSpsPad = 3;                        // aligns P[1 + hist + 4k] to 16 bytes
constexpr int kMaxHist = 1024;                    // widths up to 1024, rounded up to 256

// Exact argmax over the block of B lanes: the largest v among its valid lanes and its lowest lane
// (`off`, within the block); false when the block has no valid lane.
__device__ __forceinline__ bool block_argmax(uint32_t v, bool valid, int B, int lane,
                                             uint32_t& best, int& off) {
  uint32_t mx = valid ? v : 0u;
  if (B == 32) {
    mx = __reduce_max_sync(0xffffffffu, mx);
  } else {
    for (int o = B >> 1; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  const uint32_t bm = B == 32 ? 0xffffffffu : ((1u << B) - 1u);
  const uint32_t at = (__ballot_sync(0xffffffffu, valid && v == mx) >> (lane & ~(B - 1))) & bm;
  best = mx;
  off = __ffs(at) - 1;
  return at != 0;
}

// Prefix sums through window samples q - w .. q + 3 - w of the pass, i.e. entries
// P[idx - w .. idx - w + 3] with idx 16-byte aligned: one aligned 16-byte load when w is a
// multiple of 4, else two, from which the four entries are picked (w is the same in every lane,
// so the pick is a uniform branch). Lanes take consecutive 16-byte units: no bank conflicts.
__device__ __forceinline__ uint4 prefix4(const uint32_t* P, int idx, int w) {
  const int m = (-w) & 3;
  const uint4* q = reinterpret_cast<const uint4*>(P + idx - w - m);
  const uint4 a = q[0];
  if (m == 0) return a;
  const uint4 b = q[1];
  if (m == 1) return make_uint4(a.y, a.z, a.w, b.x);
  if (m == 2) return make_uint4(a.z, a.w, b.x, b.y);
  return make_uint4(a.w, b.x, b.y, b.z);
}

// A width's alignment, decided once per width (it is the same in every lane) instead of per load:
// M = -w mod 4 entries into the aligned chunk; OWN: w < 4 with M > 0, where the second chunk is the
// lane's own four prefix sums. f takes both as integral constants.
template <typename F>
__device__ __forceinline__ void by_alignment(int w, F&& f) {
  const int m = (-w) & 3;
  if (m == 0) f(std::integral_constant<int, 0>(), std::bool_constant<false>());
  else if (w == 1) f(std::integral_constant<int, 3>(), std::bool_constant<true>());
  else if (w == 2) f(std::integral_constant<int, 2>(), std::bool_constant<true>());
  else if (m == 1) f(std::integral_constant<int, 1>(), std::bool_constant<false>());
  else if (m == 2) f(std::integral_constant<int, 2>(), std::bool_constant<false>());
  else f(std::integral_constant<int, 3>(), std::bool_constant<false>());
}

// Entries P[idx - w .. idx - w + 3] (q: P + idx, v: the lane's own entries P[idx .. idx + 3]).
template <int M, bool OWN>
__device__ __forceinline__ uint4 earlier4(const uint32_t* q, int w, const uint4& v) {
  const uint4* c = reinterpret_cast<const uint4*>(q - w - M);
  const uint4 a = c[0];
  if (M == 0) return a;
  const uint4 b = OWN ? v : c[1];
  if (M == 1) return make_uint4(a.y, a.z, a.w, b.x);
  if (M == 2) return make_uint4(a.z, a.w, b.x, b.y);
  return make_uint4(a.w, b.x, b.y, b.z);
}

// A warp's view of one series. The search kernels give each warp a segment of consecutive
// samples of one trial, taken in passes of kSpsPass samples: lane l owns the 4-sample chunks
// 4l + 128 g (g = 0..3) of the pass. The warp's own shared-memory row P holds uint32 prefix sums
// of the pass and of the H samples before it (entry 1 + H + q = sum through sample q of the pass;
// the sums wrap, but every boxcar sum is < 2^31, so the difference of two prefixes is exact). The
// history is built once per segment from the H samples before it and then carried from pass to
// pass, so warps never wait for one another: against one CTA per trial with four barriers per
// 4096-sample pass, a warp's loads of the next pass overlap this pass's boxcars, and a trial's
// window spreads over as many warps as the chip has room for.
struct SpsRow {
  const int32_t* y;
  uint32_t* P;
  long long n;
  int H, lane;
  bool vec;

  // chunk at sample j: zero outside the window
  __device__ __forceinline__ uint4 load(long long j) const {
    if (vec && j >= 0 && j + 4 <= n) {
      const int4 t = __ldg(reinterpret_cast<const int4*>(y + j));
      return make_uint4((uint32_t)t.x, (uint32_t)t.y, (uint32_t)t.z, (uint32_t)t.w);
    }
    uint4 v = make_uint4(0, 0, 0, 0);
    if (j >= 0 && j < n) v.x = (uint32_t)__ldg(y + j);
    if (j + 1 >= 0 && j + 1 < n) v.y = (uint32_t)__ldg(y + j + 1);
    if (j + 2 >= 0 && j + 2 < n) v.z = (uint32_t)__ldg(y + j + 2);
    if (j + 3 >= 0 && j + 3 < n) v.w = (uint32_t)__ldg(y + j + 3);
    return v;
  }
  // inclusive prefix sums of G x 128 samples in place, continuing from `run`; returns the sum
  // through their last sample
  template <int G>
  __device__ __forceinline__ uint32_t scan(uint4 (&v)[G], uint32_t run) const {
    uint32_t incl[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      v[g].y += v[g].x;
      v[g].z += v[g].y;
      v[g].w += v[g].z;
      incl[g] = v[g].w;
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl[g], off);
        if (lane >= off) incl[g] += o;
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint32_t pre = run + incl[g] - v[g].w;
      run += __shfl_sync(0xffffffffu, incl[g], 31);
      v[g].x += pre;
      v[g].y += pre;
      v[g].z += pre;
      v[g].w += pre;
    }
    return run;
  }
  // P[0 .. H] for a segment starting at sample s0; returns P[H]
  __device__ __forceinline__ uint32_t history(long long s0) const {
    if (lane == 0) P[0] = 0;
    uint32_t run = 0;
    for (int q = 0; q < H; q += 256) {
      uint4 v[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
      if (s0 > 0) {  // before the window every sample is zero
        v[0] = load(s0 - H + q + 4 * lane);
        v[1] = load(s0 - H + q + 128 + 4 * lane);
        run = scan(v, run);
      }
      *reinterpret_cast<uint4*>(P + 1 + q + 4 * lane) = v[0];
      *reinterpret_cast<uint4*>(P + 1 + q + 128 + 4 * lane) = v[1];
    }
    return run;
  }
  __device__ __forceinline__ void load_pass(long long j0, uint4 (&v)[4]) const {
#pragma unroll
    for (int g = 0; g < 4; ++g) v[g] = load(j0 + 4 * lane + 128 * g);
  }
  __device__ __forceinline__ void store_pass(const uint4 (&v)[4]) const {
#pragma unroll
    for (int g = 0; g < 4; ++g)
      *reinterpret_cast<uint4*>(P + 1 + H + 4 * lane + 128 * g) = v[g];
  }
  // the last H + 1 entries become the next pass's history
  __device__ __forceinline__ void carry() const {
    if (lane == 0) P[0] = P[kSpsPass];
    for (int q = 0; q < H; q += 128) {
      const uint4 t = *reinterpret_cast<const uint4*>(P + 1 + kSpsPass + q + 4 * lane);
      *reinterpret_cast<uint4*>(P + 1 + q + 4 * lane) = t;
      __syncwarp();  // at H > 512 a later write lands where an earlier read came from
    }
    __syncwarp();
  }
};

__host__ __device__ constexpr int sps_row_words(int hist) { return kSpsPad + 1 + hist + kSpsPass; }

// Samples of a warp's segment: 8 passes (their history re-read is 6% at H = 256), 16 with wide
// boxcars (H >= 512), fewer while the launch has less than 24 warps per SM and a segment stays
// at least four times its history.
constexpr int kSegSms = 152;  // a GB300's SMs; only the split depends on it, no result
inline int64_t sps_segment(int n_trials, int64_t n, int hist) {
  int64_t seg = kSpsPass * (hist >= 512 ? 16 : 8);
  while (seg > 2 * kSpsPass && seg / 2 >= 4 * hist &&
         n_trials * ((n + seg - 1) / seg) < kSegSms * 24)
    seg /= 2;
  // a chip nearly idle: single passes, so that a bright pulse's groups spread over more warps
  while (seg > kSpsPass && n_trials * ((n + seg - 1) / seg) < kSegSms * 4) seg /= 2;
  while ((n + seg * kSpsWarps - 1) / (seg * kSpsWarps) > 65535) seg *= 2;  // grid rows
  return seg;
}

// CTA (trial, 8 segments): warp v takes segment 8 * blockIdx.y + v. Every boxcar sum is compared
// with an integer bound per width below which the SNR cannot reach the threshold; a 32-sample
// group where one passes is searched exactly by its warp (lane = sample): per width the group's
// largest boxcar sum (earliest sample) per peak block, then the FP64 SNRs in the oracle's
// evaluation order. Bound by instruction issue in the filter (one aligned 16-byte prefix load,
// four subtractions, a three-way maximum and a compare per four boxcar sums).
__global__ void __launch_bounds__(kSpsThreads, 3) k_sps(const SpsArgs a, const long long seg) {
  extern __shared__ __align__(16) uint32_t Ps[];
  __shared__ double den[kMaxWidths];
  __shared__ long long ca[kMaxWidths], cb[kMaxWidths];
  __shared__ uint32_t bthr[kMaxWidths];

  const int32_t i = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const long long n = a.n;
  const double thr = (double)a.threshold;
  // Per width k: SNR = (ca[k] * B - cb[k]) / den[k]. Window statistics: ca = n, cb = w * S1,
  // den = sqrt(w) * sqrt(n * S2 - S1^2). Clipped per-width statistics (a.wst): ca = N_k,
  // cb = T1_k, den = sqrt(N_k * T2_k - T1_k^2). A width with den 0 gives no candidates.
  // One warp works them out (FP64 is slow here, and eight warps would share its pipe).
  __shared__ int constant;  // a constant series has no candidates
  if (wid > 0) {
  } else if (a.wst == nullptr) {
    const Moments m = a.mom[i];
    const long long s1 = (long long)m.s1;
    const double sq = window_sqrt_var(m, n);
    if (tid == 0) constant = sq == 0.0;
    if (tid < a.nw && sq != 0.0) {
      const int w = a.wd[tid];
      den[tid] = sqrt((double)w) * sq;
      ca[tid] = n;
      cb[tid] = (long long)w * s1;
      bthr[tid] = window_bound(w, s1, thr, den[tid], n);
    }
  } else if (tid < a.nw) {
    if (tid == 0) constant = 0;
    const WidthStats st = a.wst[(int64_t)i * a.nw + tid];
    const unsigned long long un = (unsigned long long)st.n, ut1 = (unsigned long long)st.t1;
    const unsigned long long p_lo = un * st.t2lo;
    const unsigned long long p_hi = __umul64hi(un, st.t2lo) + un * st.t2hi;
    const unsigned long long q_lo = ut1 * ut1, q_hi = __umul64hi(ut1, ut1);
    const unsigned long long v_lo = p_lo - q_lo;
    const unsigned long long v_hi = p_hi - q_hi - (p_lo < q_lo ? 1ull : 0ull);
    const bool live = st.n > 0 && (v_lo | v_hi) != 0;
    den[tid] = live ? sqrt(u128_to_f64(v_hi, v_lo)) : 0.0;
    ca[tid] = st.n;
    cb[tid] = st.t1;
    // SNR >= thr  <=>  B >= (T1 + thr*den) / N, with the margin above
    const double t = live ? ((double)st.t1 + thr * den[tid]) / (double)st.n : 0.0;
    const double tl = t - 2.0 - 1e-9 * fabs(t);
    bthr[tid] = !live ? 0xFFFFFFFFu
                      : (tl <= 0.0 ? 0u : (tl >= 4294967295.0 ? 0xFFFFFFFFu : (uint32_t)floor(tl)));
  }
  __syncthreads();  // the only CTA barrier: the widths' statistics
  if (constant) return;
  const long long s0 = ((long long)blockIdx.y * kSpsWarps + wid) * seg;
  if (s0 >= n) return;
  const long long s1 = s0 + seg < n ? s0 + seg : n;
  const int H = a.hist, nw = a.nw;
  const int wmax = a.wd[nw - 1];
  const int B = a.block;
  SpsRow R;
  R.y = a.y + (int64_t)i * a.stride;
  R.P = Ps + (size_t)wid * sps_row_words(H) + kSpsPad;
  R.n = n;
  R.H = H;
  R.lane = lane;
  R.vec = (reinterpret_cast<uintptr_t>(R.y) & 15) == 0;
  const uint32_t* P = R.P;

  uint4 nv[4];
  R.load_pass(s0, nv);
  uint32_t run = R.history(s0);
  for (long long j0 = s0; j0 < s1; j0 += kSpsPass) {
    uint4 v[4] = {nv[0], nv[1], nv[2], nv[3]};
    run = R.scan(v, run);
    R.store_pass(v);
    __syncwarp();
    if (j0 + kSpsPass < s1) R.load_pass(j0 + kSpsPass, nv);  // in flight during the boxcars

    // ---- filter: every boxcar sum of this lane's samples against the bounds
    const bool interior = j0 >= wmax - 1 && j0 + kSpsPass <= n;  // every (sample, width) valid
    bool hot[4] = {false, false, false, false};
    const uint32_t* Pq = P + 1 + H + 4 * lane;
    if (interior) {
      // sums are below 2^31 (a wrapped one, from negative input, is passed over by the exact
      // search): the largest sum less the bound, over the widths
      int over[4] = {INT_MIN, INT_MIN, INT_MIN, INT_MIN};
#pragma unroll 1
      for (int k = 0; k < nw; ++k) {
        const int w = a.wd[k];
        const int t = (int)min(bthr[k], 0x7FFFFFFFu);
        by_alignment(w, [&](auto m, auto own) {
          constexpr int M = decltype(m)::value;
          constexpr bool OWN = decltype(own)::value;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const uint4 st = earlier4<M, OWN>(Pq + 128 * g, w, v[g]);
            const int mx = max(max((int)(v[g].x - st.x), (int)(v[g].y - st.y)),
                               max((int)(v[g].z - st.z), (int)(v[g].w - st.w)));
            over[g] = max(over[g], max(mx, 0) - t);
          }
        });
      }
#pragma unroll
      for (int g = 0; g < 4; ++g) hot[g] = over[g] >= 0;
    } else {
#pragma unroll 1
      for (int k = 0; k < nw; ++k) {
        const int w = a.wd[k];
        const uint32_t t = bthr[k];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const uint4 st = prefix4(P, 1 + H + 4 * lane + 128 * g, w);
          const long long j = j0 + 4 * lane + 128 * g;
          hot[g] |= (j < n && j >= w - 1 && v[g].x - st.x >= t) |
                    (j + 1 < n && j + 1 >= w - 1 && v[g].y - st.y >= t) |
                    (j + 2 < n && j + 2 >= w - 1 && v[g].z - st.z >= t) |
                    (j + 3 < n && j + 3 >= w - 1 && v[g].w - st.w >= t);
        }
      }
    }
    // lanes 8c .. 8c + 7 of chunk row g cover the pass's 32-sample group 4g + c
    unsigned groups = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const unsigned hm = __ballot_sync(0xffffffffu, hot[g]);
#pragma unroll
      for (int c = 0; c < 4; ++c) groups |= ((hm >> (8 * c)) & 0xFFu) ? (1u << (4 * g + c)) : 0u;
    }

    // ---- exact search of the hot groups, lane = sample
    while (groups) {
      const int c = __ffs(groups) - 1;
      groups &= groups - 1;
      const int q = c * 32 + lane;  // pass sample
      const long long j = j0 + q;
      const uint32_t pj = P[1 + H + q];
      // A width whose largest sum stays below its bound cannot reach the threshold and is left
      // out before the FP64 division.
      bool leader = (lane & (B - 1)) == 0;
      double bs = 0.0;
      long long bj = 0;
      int bwid = 0;
      bool have = false;
      if (B == 32) {
        // lane k takes width k, so the widths' divisions run at once
        uint32_t mine = 0;
        int moff = 0;
        for (int k = 0; k < nw; ++k) {
          const int w = a.wd[k];
          const bool valid = (j < n) && (j >= w - 1) && den[k] != 0.0;
          uint32_t best;
          int off;
          const bool any = block_argmax(valid ? pj - P[1 + H + q - w] : 0u, valid, 32, lane, best,
                                        off);
          if (lane == k) {
            have = any && (int32_t)best >= 0 && best >= bthr[k];
            mine = best;
            moff = off;
          }
        }
        int kw = lane;
        if (have) bs = (double)(ca[lane] * (long long)mine - cb[lane]) / den[lane];
        // The best width: largest SNR, then the earliest sample, then the smallest width. In
        // FP32 first (a double's rounding to float is monotone, so the largest double is among
        // the lanes holding the largest float); FP64 compares only where that leaves several.
        const float fs = have ? (float)bs : -INFINITY;
        float fm = fs;
        for (int o = 8; o > 0; o >>= 1) fm = fmaxf(fm, __shfl_xor_sync(0xffffffffu, fm, o));
        const unsigned top = __ballot_sync(0xffffffffu, have && fs == fm) & 0xFFFFu;
        if (__popc(top) > 1) {
          for (int o = 8; o > 0; o >>= 1) {
            const double os = __shfl_xor_sync(0xffffffffu, bs, o);
            const int oj = __shfl_xor_sync(0xffffffffu, moff, o);
            const int ok = __shfl_xor_sync(0xffffffffu, kw, o);
            const bool oh = __shfl_xor_sync(0xffffffffu, have ? 1 : 0, o) != 0;
            if (oh && (!have || os > bs || (os == bs && (oj < moff || (oj == moff && ok < kw))))) {
              have = true;
              bs = os;
              moff = oj;
              kw = ok;
            }
          }
          leader = lane == 0;
        } else {
          leader = lane < 16 && ((top >> lane) & 1u) != 0;  // the winner writes
        }
        bj = j0 + c * 32 + moff;
        bwid = a.wd[kw & (kMaxWidths - 1)];
      } else {
        for (int k = 0; k < nw; ++k) {
          const int w = a.wd[k];
          const bool valid = (j < n) && (j >= w - 1) && den[k] != 0.0;
          uint32_t best;
          int off;
          const bool any = block_argmax(valid ? pj - P[1 + H + q - w] : 0u, valid, B, lane, best,
                                        off);
          if (leader && any && (int32_t)best >= 0 && best >= bthr[k]) {
            const double snr = (double)(ca[k] * (long long)best - cb[k]) / den[k];
            const long long jk = j + off;  // the leader holds the block's first sample
            if (!have || snr > bs || (snr == bs && jk < bj)) {
              have = true;
              bs = snr;
              bj = jk;
              bwid = w;
            }
          }
        }
      }
      if (leader && have && bs >= thr) {
        const unsigned long long idx = atomicAdd(a.count, 1ull);
        if ((long long)idx < a.cap) {
          dd_cand_t cd;
          cd.trial = i;
          cd.range = a.range;
          cd.t_start = (a.J0 + bj - bwid + 1) * (long long)a.d;
          cd.width = bwid * a.d;
          cd.pad = 0;
          cd.snr = bs;
          a.cands[idx] = cd;
        }
      }
    }
    __syncwarp();  // every read of this pass's P is done
    if (j0 + kSpsPass < s1) R.carry();
  }
}

// The search's last step on a range whose block maxima the fused dedispersion kernel recorded:
// one CTA per trial, one thread per peak block. The block's candidate is, over the widths, the
// recorded largest boxcar sum's SNR (the SNR grows with the sum at a fixed width, and the
// recorded sample is the earliest holding it), with k_sps's statistics, evaluation order and
// tie rules, so the candidates are the ones k_sps finds on the same series.
__global__ void __launch_bounds__(kSpsThreads) k_sps_fused(const SpsFusedArgs a) {
  __shared__ double den[kMaxWidths];
  __shared__ long long ca[kMaxWidths], cb[kMaxWidths];
  __shared__ uint32_t kthr[kMaxWidths];
  const int32_t i = blockIdx.x;
  const int tid = threadIdx.x;
  const long long n = a.n;
  if (n <= 0) return;
  __shared__ int constant;  // a constant series has no candidates
  const double thr = (double)a.threshold;
  if (tid < 32) {  // one warp's FP64, as in k_sps
    const Moments m = a.mom[i];
    const double sq = window_sqrt_var(m, n);
    if (tid == 0) constant = sq == 0.0;
    if (tid < a.nw && sq != 0.0) {
      const int w = a.wd[tid];
      den[tid] = sqrt((double)w) * sq;
      ca[tid] = n;
      cb[tid] = (long long)w * (long long)m.s1;
      // a record can reach the threshold only if its sum passes k_sps's integer bound (key =
      // sum + 1, so key > bound); the others are skipped before the FP64 SNR
      kthr[tid] = window_bound(w, (long long)m.s1, thr, den[tid], n);
    }
  }
  __syncthreads();
  if (constant) return;
  const int64_t row = (int64_t)i * a.nw;
  for (int64_t b = tid; b < a.nblk; b += kSpsThreads) {
    double bs = 0.0;
    long long bj = 0;
    int bwid = 0;
    bool have = false;
    for (int k = 0; k < a.nw; ++k) {
      const uint32_t key = a.key[(row + k) * a.nblk + b];
      if (key == 0 || key <= kthr[k]) continue;  // no sample, or below the bound
      const long long best = (long long)(key - 1u);
      const long long jk = b * a.block + a.off[(row + k) * a.nblk + b];
      const long long num = ca[k] * best - cb[k];
      const double snr = (double)num / den[k];
      if (!have || snr > bs || (snr == bs && jk < bj)) {
        have = true;
        bs = snr;
        bj = jk;
        bwid = a.wd[k];
      }
    }
    if (have && bs >= thr) {
      const unsigned long long idx = atomicAdd(a.count, 1ull);
      if ((long long)idx < a.cap) {
        dd_cand_t cd;
        cd.trial = i;
        cd.range = a.range;
        cd.t_start = (a.J0 + bj - bwid + 1) * (long long)a.d;
        cd.width = bwid * a.d;
        cd.pad = 0;
        cd.snr = bs;
        a.cands[idx] = cd;
      }
    }
  }
}

// Clipped statistics of every boxcar series of one trial (one CTA per trial): for each width w,
// the values B_w[j] (window samples j >= w - 1) are summed over the whole window (step 0:
// count, sum, 128-bit sum of squares), then, for up to `iters` steps, again over the values
// within ceil(mu - kappa*sd) .. floor(mu + kappa*sd) of the previous step's mean and population
// deviation (FP64, one rounding per operation, as the oracle). A width whose previous step has no
// values or no variance keeps its statistics.
//
// Each step sweeps the series once, each warp over its own eighth of the window (SpsRow). The
// bounds are whole numbers, so a value is tested and summed as x = B - lo <= hi - lo in 32-bit
// integers, and the sums of B and B^2 follow exactly from the count and the sums of x and x^2. A
// lane's sums of a width wait in shared memory between passes, so the width loop stays rolled:
// unrolled over widths with the sums in registers it outgrew the instruction cache and took 18
// instructions a value (4.2 ms for the 1024-channel beam's three ranges, 9 widths x 4 sweeps, 2.9 so; in
// FP64 it was bound by the FP64 pipe, 44 ms).
struct ClipSum {
  unsigned long long c1, c2;  // sums of x and (low half) of x^2
};

__global__ void __launch_bounds__(kSpsThreads, 3) k_clip_stats(const ClipArgs a) {
  extern __shared__ __align__(16) uint32_t Ps[];
  __shared__ uint32_t lo_b[kMaxWidths], span_b[kMaxWidths];  // values lo .. lo + span
  __shared__ int live[kMaxWidths];                           // 0: statistics final
  __shared__ int some[kMaxWidths];  // 0: the bounds hold no value; 1; 2: 64-bit sums suffice
  __shared__ WidthStats st[kMaxWidths];
  __shared__ unsigned long long red[kMaxWidths][4][kSpsWarps];

  const int32_t i = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const long long n = a.n;
  const int nw = a.nw, H = a.hist;
  const int wmax = a.wd[nw - 1];
  SpsRow R;
  R.y = a.y + (int64_t)i * a.stride;
  R.P = Ps + (size_t)wid * sps_row_words(H) + kSpsPad;
  R.n = n;
  R.H = H;
  R.lane = lane;
  R.vec = (reinterpret_cast<uintptr_t>(R.y) & 15) == 0;
  const uint32_t* P = R.P;
  // this lane's sums of width k: sums[32 k], cnts[32 k] (count; carries of c2 in cnts[32 (nw + k)])
  ClipSum* sums = reinterpret_cast<ClipSum*>(Ps + (size_t)kSpsWarps * sps_row_words(H)) +
                  (size_t)wid * nw * 32 + lane;
  uint32_t* cnts = reinterpret_cast<uint32_t*>(
                       reinterpret_cast<ClipSum*>(Ps + (size_t)kSpsWarps * sps_row_words(H)) +
                       (size_t)kSpsWarps * nw * 32) +
                   (size_t)wid * nw * 64 + lane;
  const long long per = ((n + kSpsWarps - 1) / kSpsWarps + 127) / 128 * 128;
  const long long s0 = min(n, wid * per), s1 = min(n, s0 + per);
  // a lane's sums of squares over its part of a sweep stay below 2^64, its sums over a pass
  // below 2^32
  const double lane_values = 16.0 * (double)((per + kSpsPass - 1) / kSpsPass);
  auto narrow = [&](uint32_t span) {
    return (double)span * (double)span * lane_values < 1.8e19 && span < (1u << 28);
  };
  if (tid < kMaxWidths) {
    lo_b[tid] = 0u;  // step 0: every value (all boxcar sums are >= 0)
    span_b[tid] = tid < nw ? (uint32_t)a.wd[tid] * a.vmax : 0u;
    live[tid] = tid < nw ? 1 : 0;
    some[tid] = narrow(span_b[tid]) ? 2 : 1;
    st[tid] = WidthStats{0, 0, 0, 0};
  }
  __syncthreads();
  for (int step = 0; step <= a.iters; ++step) {
    bool any = false;
    for (int k = 0; k < nw; ++k) any |= live[k] != 0;
    if (!any) break;  // uniform: every thread reads the same flags
    for (int k = 0; k < nw; ++k) {
      sums[32 * k] = ClipSum{0, 0};
      cnts[32 * k] = cnts[32 * (nw + k)] = 0;
    }
    if (s0 < s1) {
      uint4 nv[4];
      R.load_pass(s0, nv);
      uint32_t run = R.history(s0);
      for (long long j0 = s0; j0 < s1; j0 += kSpsPass) {
        uint4 v[4] = {nv[0], nv[1], nv[2], nv[3]};
        run = R.scan(v, run);
        R.store_pass(v);
        __syncwarp();
        if (j0 + kSpsPass < s1) R.load_pass(j0 + kSpsPass, nv);
        const bool interior = j0 >= wmax - 1 && j0 + kSpsPass <= s1;
#pragma unroll 1
        for (int k = 0; k < nw; ++k) {
          const int how = live[k] ? some[k] : 0;
          if (how == 0) continue;  // uniform
          const int w = a.wd[k];
          const uint32_t lo = lo_b[k], span = span_b[k];
          ClipSum c = sums[32 * k];
          uint32_t cn = cnts[32 * k];
          if (how == 2 && interior) {
            uint32_t sum = 0;
            by_alignment(w, [&](auto m, auto own) {
              constexpr int M = decltype(m)::value;
              constexpr bool OWN = decltype(own)::value;
#pragma unroll
              for (int g = 0; g < 4; ++g) {
                const uint4 s4 = earlier4<M, OWN>(P + 1 + H + 4 * lane + 128 * g, w, v[g]);
                const uint32_t x[4] = {v[g].x - s4.x - lo, v[g].y - s4.y - lo,
                                       v[g].z - s4.z - lo, v[g].w - s4.w - lo};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const bool in = x[e] <= span;
                  const uint32_t xm = in ? x[e] : 0u;
                  cn += in ? 1u : 0u;
                  sum += xm;
                  c.c2 += (unsigned long long)xm * xm;
                }
              }
            });
            c.c1 += sum;
          } else {
            uint32_t carry = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const uint4 s4 = prefix4(P, 1 + H + 4 * lane + 128 * g, w);
              const uint32_t x[4] = {v[g].x - s4.x - lo, v[g].y - s4.y - lo, v[g].z - s4.z - lo,
                                     v[g].w - s4.w - lo};
              const long long j = j0 + 4 * lane + 128 * g;
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const bool in = x[e] <= span && j + e < s1 && j + e >= w - 1;
                const uint32_t m = in ? x[e] : 0u;
                const unsigned long long sq = (unsigned long long)m * m;
                if (in) ++cn;
                c.c1 += m;
                c.c2 += sq;
                carry += c.c2 < sq ? 1u : 0u;
              }
            }
            if (carry) cnts[32 * (nw + k)] += carry;
          }
          sums[32 * k] = c;
          cnts[32 * k] = cn;
        }
        __syncwarp();  // every read of this pass's P is done
        if (j0 + kSpsPass < s1) R.carry();
      }
    }
    // CTA sums of the widths: warp butterflies, then one thread per width
#pragma unroll 1
    for (int k = 0; k < nw; ++k) {
      unsigned long long x0 = cnts[32 * k], x1 = sums[32 * k].c1, lo = sums[32 * k].c2;
      unsigned long long hi = cnts[32 * (nw + k)];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        x0 += __shfl_xor_sync(0xffffffffu, x0, off);
        x1 += __shfl_xor_sync(0xffffffffu, x1, off);
        const unsigned long long olo = __shfl_xor_sync(0xffffffffu, lo, off);
        const unsigned long long ohi = __shfl_xor_sync(0xffffffffu, hi, off);
        const unsigned long long nlo = lo + olo;
        hi = hi + ohi + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
      }
      if (lane == 0) {
        red[k][0][wid] = x0;
        red[k][1][wid] = x1;
        red[k][2][wid] = lo;
        red[k][3][wid] = hi;
      }
    }
    __syncthreads();
    if (tid < nw && live[tid]) {
      unsigned long long c = 0, x1 = 0, lo = 0, hi = 0;
      for (int q = 0; q < kSpsWarps; ++q) {
        c += red[tid][0][q];
        x1 += red[tid][1][q];
        const unsigned long long nlo = lo + red[tid][2][q];
        hi = hi + red[tid][3][q] + (nlo < lo ? 1ull : 0ull);
        lo = nlo;
      }
      // sums of B = x + l over c values: T1 = X1 + c l, T2 = X2 + 2 l X1 + c l^2 (128 bits)
      const unsigned long long l = lo_b[tid];
      const unsigned long long t1 = x1 + c * l;
      const unsigned long long a0 = 2 * l * x1, a1 = __umul64hi(2 * l, x1);
      const unsigned long long b0 = l * l * c, b1 = __umul64hi(l * l, c);
      unsigned long long r0 = lo + a0, r1 = hi + a1 + (r0 < lo ? 1ull : 0ull);
      r1 += b1 + (r0 + b0 < r0 ? 1ull : 0ull);
      r0 += b0;
      const WidthStats s = WidthStats{(long long)c, (long long)t1, r0, r1};
      st[tid] = s;
      // bounds of the next step from this step's statistics
      if (step < a.iters) {
        const unsigned long long un = c, ut1 = t1;
        const unsigned long long p_lo = un * s.t2lo;
        const unsigned long long p_hi = __umul64hi(un, s.t2lo) + un * s.t2hi;
        const unsigned long long q_lo = ut1 * ut1, q_hi = __umul64hi(ut1, ut1);
        const unsigned long long v_lo = p_lo - q_lo;
        const unsigned long long v_hi = p_hi - q_hi - (p_lo < q_lo ? 1ull : 0ull);
        if (s.n == 0 || (v_lo | v_hi) == 0) {
          live[tid] = 0;
        } else {
          const double dn = __ll2double_rn(s.n);
          const double mu = __ddiv_rn(__ll2double_rn(s.t1), dn);
          const double sd = __ddiv_rn(__dsqrt_rn(u128_to_f64(v_hi, v_lo)), dn);
          const double ks = __dmul_rn(a.kappa, sd);
          const double lo = ceil(__dsub_rn(mu, ks)), hi = floor(__dadd_rn(mu, ks));
          // the whole-number bounds on values 0 .. 2^31 - 1
          const double top = 2147483647.0;
          const uint32_t l2 = lo <= 0.0 ? 0u : (lo <= top ? (uint32_t)lo : 0u);
          lo_b[tid] = l2;
          span_b[tid] =
              hi >= top ? 0x7FFFFFFFu - l2 : (hi >= (double)l2 ? (uint32_t)hi - l2 : 0u);
          some[tid] = lo <= top && hi >= 0.0 && lo <= hi ? (narrow(span_b[tid]) ? 2 : 1) : 0;
        }
      }
    }
    __syncthreads();
  }
  if (tid < nw) a.out[(int64_t)i * nw + tid] = st[tid];
}

// Dynamic shared memory of k_clip_stats: a prefix-sum row and the lanes' sums per warp.
static size_t clip_smem(int nw, int hist) {
  return (sizeof(uint32_t) * (size_t)sps_row_words(hist) +
          32 * (size_t)nw * (sizeof(ClipSum) + 2 * sizeof(uint32_t))) *
         kSpsWarps;
}

cudaError_t launch_clip_stats(const ClipArgs& a, cudaStream_t st) {
  if (a.n <= 0 || a.n_trials <= 0 || a.nw <= 0) return cudaSuccess;
  if (a.nw > kMaxWidths || a.hist < 0 || a.hist % 256 || a.hist > kMaxHist || a.iters < 0 ||
      !(a.kappa > 0))
    return cudaErrorInvalidValue;
  // The limit is state of the function on the device, shared by every plan and host thread: always
  // the largest a launch can need, so that no thread lowers it between another's set and launch.
  const cudaError_t e =
      cudaFuncSetAttribute(k_clip_stats, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)clip_smem(kMaxWidths, kMaxHist));
  if (e != cudaSuccess) return e;
  const size_t smem = clip_smem(a.nw, a.hist);
  k_clip_stats<<<a.n_trials, kSpsThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sps(const SpsArgs& a, cudaStream_t st) {
  if (a.n <= 0 || a.n_trials <= 0 || a.nw <= 0) return cudaSuccess;
  if (a.hist < 0 || a.hist % 256 || a.hist > kMaxHist || a.block < 1 || a.block > 32)
    return cudaErrorInvalidValue;
  const size_t smem = sizeof(uint32_t) * (size_t)sps_row_words(a.hist) * kSpsWarps;
  if (smem > 48 * 1024) {  // the largest history only: the limit set is always the same
    const cudaError_t e =
        cudaFuncSetAttribute(k_sps, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int64_t seg = sps_segment(a.n_trials, a.n, a.hist);
  const int64_t rows = (a.n + seg * kSpsWarps - 1) / (seg * kSpsWarps);
  k_sps<<<dim3((unsigned)a.n_trials, (unsigned)rows), kSpsThreads, smem, st>>>(a, seg);
  return cudaGetLastError();
}

cudaError_t launch_sps_fused(const SpsFusedArgs& a, cudaStream_t st) {
  if (a.n <= 0 || a.n_trials <= 0 || a.nw <= 0) return cudaSuccess;
  if (a.block < 1 || a.block > 32 || a.nblk != (a.n + a.block - 1) / a.block)
    return cudaErrorInvalidValue;
  k_sps_fused<<<a.n_trials, kSpsThreads, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace ddk
