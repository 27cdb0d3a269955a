// dump.cu -- end of integration: visibilities, full-Stokes, reset; and the
// pitch copy used when block_len is not a multiple of 16 bytes.
//
// Full-Stokes (abstract, Sec. 1) per antenna pair p >= q, inputs 2p+pol:
//   XX = V[2p][2q], YY = V[2p+1][2q+1], XY = V[2p][2q+1], YX = V[2p+1][2q]
//   (p == q: XY = conj(V[2p+1][2p]), the element above the diagonal)
//   I = XX + YY, Q = XX - YY, U = XY + YX, V = -j (XY - YX)
// Each lower-triangle element belongs to exactly one antenna pair, so one
// thread per pair reads its 3 or 4 elements, writes them to the visibility
// output, zeroes them in the integration buffer and writes the four Stokes
// products -- one pass over HBM with no cross-thread hazards.  Consecutive
// threads take consecutive q, so the 32-byte (XX, XY) and (YX, YY) element
// pairs they touch are contiguous across the warp.  Bound by HBM: 192 inputs,
// 1024 channels, 1.2 GB in 209 us (5.8 TB/s; 271 us before the pair's row came
// from a single-precision root and the Stokes products left in whole sectors).

#include "xe_internal.h"

namespace xe {

namespace {

// The largest p with p(p+1)/2 <= a, for a < 2^27 (4096 antennas have 2^23
// pairs): a single-precision square root is within one of it, and two integer
// steps settle it.  (Double precision runs at 1/64 of the rate here; its root
// for every pair took most of the kernel's time.)
__device__ __forceinline__ int tri_row(int a) {
  int p = (int)((sqrtf(8.0f * (float)a + 1.0f) - 1.0f) * 0.5f);
  while ((p + 1) * (p + 2) / 2 <= a) ++p;
  while (p * (p + 1) / 2 > a) --p;
  return p;
}

// A 32-byte store of two 16-byte values (one full sector).
__device__ __forceinline__ void store32(longlong2 *p, longlong2 a, longlong2 b) {
  asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a.x), "l"(a.y), "l"(b.x),
               "l"(b.y)
               : "memory");
}

// WIDE: the Stokes output is 32-byte aligned and its products leave in two
// full-sector stores.
template <bool WIDE>
__global__ void dump_dual_kernel(int64_t *__restrict__ acc, int64_t *__restrict__ vis,
                                 int64_t *__restrict__ stokes, int n_ant, int n_chan,
                                 int *status) {
  const long long n_in = 2LL * n_ant;
  const long long P = n_in * (n_in + 1) / 2;
  const int A = n_ant * (n_ant + 1) / 2;
  const long long total = (long long)A * n_chan;
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  // channel and pair of idx, advanced without further divisions
  int c = (int)(idx / A), a = (int)(idx - (long long)c * A);
  const int c_step = (int)(stride / A), a_step = (int)(stride - (long long)c_step * A);
  for (; idx < total; idx += stride) {
    const int p = tri_row(a), q = a - p * (p + 1) / 2;
    const long long base = c * P;
    // element offsets (in pairs) of XX, XY (p > q only), YX, YY
    const long long e_xx = base + p * (2 * p + 1) + 2 * q, e_xy = e_xx + 1;
    const long long e_yx = base + (2 * p + 1) * (p + 1) + 2 * q, e_yy = e_yx + 1;
    a += a_step;
    c += c_step;
    if (a >= A) a -= A, ++c;
#ifdef CORR_DEBUG
    // every element this thread touches lies in channel c's part of the buffer
    if (p >= n_ant || q > p || e_xx < base || e_yy >= base + P) {
      atomicOr(status, kStatusBounds);
      continue;
    }
#endif
    longlong2 *a2 = reinterpret_cast<longlong2 *>(acc);
    const longlong2 zero = make_longlong2(0, 0);
    const longlong2 xx = a2[e_xx], yx = a2[e_yx], yy = a2[e_yy];
    longlong2 xy;
    if (p > q) {
      xy = a2[e_xy];
    } else {
      xy = make_longlong2(yx.x, -yx.y);
    }
    if (vis) {
      longlong2 *v2 = reinterpret_cast<longlong2 *>(vis);
      v2[e_xx] = xx;
      if (p > q) v2[e_xy] = xy;
      v2[e_yx] = yx;
      v2[e_yy] = yy;
    }
    a2[e_xx] = zero;
    if (p > q) a2[e_xy] = zero;
    a2[e_yx] = zero;
    a2[e_yy] = zero;
    if (stokes) {
      longlong2 *s2 = reinterpret_cast<longlong2 *>(stokes) + idx * 4;
      const longlong2 si = make_longlong2(xx.x + yy.x, xx.y + yy.y);
      const longlong2 sq = make_longlong2(xx.x - yy.x, xx.y - yy.y);
      const longlong2 su = make_longlong2(xy.x + yx.x, xy.y + yx.y);
      const longlong2 sv = make_longlong2(xy.y - yx.y, -(xy.x - yx.x));  // -j (XY - YX)
      if (WIDE) {
        store32(s2, si, sq);
        store32(s2 + 2, su, sv);
      } else {
        s2[0] = si;
        s2[1] = sq;
        s2[2] = su;
        s2[3] = sv;
      }
    }
  }
}

__global__ void dump_single_kernel(int64_t *__restrict__ acc, int64_t *__restrict__ vis,
                                   long long n_elems2) {
  longlong2 *a2 = reinterpret_cast<longlong2 *>(acc);
  longlong2 *v2 = reinterpret_cast<longlong2 *>(vis);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n_elems2;
       idx += (long long)gridDim.x * blockDim.x) {
    const longlong2 v = a2[idx];
    if (v2) v2[idx] = v;
    a2[idx] = make_longlong2(0, 0);
  }
}

// Debug builds: one block compares both guard bands with kGuardByte.
__global__ void guard_check_kernel(const unsigned char *__restrict__ before,
                                   const unsigned char *__restrict__ after, size_t bytes,
                                   int *status) {
  const uint32_t want = 0x01010101u * kGuardByte;
  bool bad = false;
  for (size_t w = threadIdx.x; w < bytes / 4; w += blockDim.x)
    bad |= reinterpret_cast<const uint32_t *>(before)[w] != want ||
           reinterpret_cast<const uint32_t *>(after)[w] != want;
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kStatusBounds);
}

// dst[row][0..pitch) = src[row][0..T) followed by zeros.  A thread makes 16
// output bytes from the five aligned source words that hold them (the words
// come from L1 for all but one lane).  A row's last bytes, and the source's
// last ones, whose fifth word would lie past its end, are put together from
// bytes.  src is 4-byte aligned and pitch a multiple of 16.  (45 MB in 15 us;
// byte by byte 75 us, a word a thread 27 us.)
__global__ void pitch_kernel(const uint8_t *__restrict__ src, uint8_t *__restrict__ dst,
                             long long rows, int T, int pitch) {
  const int quads = pitch >> 4;  // 16-byte pieces of a row
  const long long n_quads = rows * quads;
  const long long src_bytes = rows * (long long)T;
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  long long row = k / quads;
  int w = (int)(k - row * quads);
  const long long row_step = stride / quads;
  const int w_step = (int)(stride - row_step * quads);
#pragma unroll 2
  for (; k < n_quads; k += stride) {
    const long long at = row * T + 16 * w;  // first source byte of the piece
    const int left = T - 16 * w;            // bytes of the row from there on
    uint32_t v[4] = {0u, 0u, 0u, 0u};
    if (left >= 16 && (at | 3) + 16 < src_bytes) {
      const uint32_t *s = reinterpret_cast<const uint32_t *>(src + (at & ~3LL));
      uint32_t x[5];
#pragma unroll
      for (int e = 0; e < 5; ++e) x[e] = __ldg(s + e);
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = __funnelshift_r(x[e], x[e + 1], 8 * (int)(at & 3));
    } else {
#pragma unroll
      for (int b = 0; b < 16; ++b)
        if (b < left) v[b >> 2] |= (uint32_t)__ldg(src + at + b) << (8 * (b & 3));
    }
    reinterpret_cast<uint4 *>(dst)[k] = make_uint4(v[0], v[1], v[2], v[3]);
    row += row_step;
    w += w_step;
    if (w >= quads) w -= quads, ++row;
  }
}

}  // namespace

cudaError_t launch_dump(int64_t *acc, int64_t *vis, int64_t *stokes, int n_ant, int n_pol,
                        int n_chan, cudaStream_t stream, int grid, int *status) {
  if (n_pol == 2) {
    if ((reinterpret_cast<uintptr_t>(stokes) & 31u) == 0)
      dump_dual_kernel<true><<<grid, 256, 0, stream>>>(acc, vis, stokes, n_ant, n_chan, status);
    else
      dump_dual_kernel<false><<<grid, 256, 0, stream>>>(acc, vis, stokes, n_ant, n_chan, status);
  } else {
    const long long n_in = n_ant;
    dump_single_kernel<<<grid, 256, 0, stream>>>(acc, vis, n_in * (n_in + 1) / 2 * n_chan);
  }
  return cudaGetLastError();
}

cudaError_t launch_guard_check(const unsigned char *before, const unsigned char *after,
                               size_t bytes, int *status, cudaStream_t stream) {
  guard_check_kernel<<<1, 256, 0, stream>>>(before, after, bytes, status);
  return cudaGetLastError();
}

cudaError_t launch_pitch(const uint8_t *src, uint8_t *dst, long long rows, int T, int pitch,
                         cudaStream_t stream, int grid) {
  pitch_kernel<<<grid, 256, 0, stream>>>(src, dst, rows, T, pitch);
  return cudaGetLastError();
}

}  // namespace xe
