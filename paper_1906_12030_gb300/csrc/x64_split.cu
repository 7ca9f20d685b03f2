// Digit images of the binary64 operands that x64_gemm_kernel multiplies.
//
// Every row of an operand is cut into blocks of 256 along K.  With 2^e the
// exponent of the row's largest entry and 2^b that of the block's (raised to
// 2^(e-24) where it is smaller, so that every digit product stays a normal
// binary32 number), an entry x is rounded to a multiple X of 2^(b-62) and X
// written as eight balanced digits to the base 2^8,
//   x 2^-e ~ sum_p d_p 2^(b-e-6-8p),   d_0 in [-128, 128], else [-128, 127],
// each stored as the BF16 value d_p 2^(b-e-6-8p), which is exact.  Entries
// within a factor 2^10 of the block's largest are represented exactly.
// Adding 128 (256^0 + ... + 256^7) to X makes the balanced digits plain
// bytes, so a digit costs one byte permute and one FMA.
// A ninth plane holds |x| 2^-e itself, cut to a BF16 value (below 2^-60, but
// not zero: 2^-60), from which the GEMM sums the magnitudes of its terms.
//
// Image: tiles of `tile` rows (128 for the GEMM's A, 64 for B); per tile and
// 16 of K, per digit, groups of eight rows, the two 8-wide halves of the 16
// as 8 x 16-byte core matrices; after all digits of the tile its magnitudes,
// likewise.  A GEMM stage is then one contiguous piece.
// Columns K .. 16 ceil(K / 16) - 1 are zero; rows beyond the operand's are
// not written (they only meet outputs that are not stored).
//
// Bound: memory, 8 bytes read and 18 written per entry (65536 x 4096: 7.0 GB
// in 1.35 ms, 5.2 TB/s).  A block of threads
// holds 8192 entries (whole rows) in registers between finding the exponents
// and writing the digits, so each entry is read once; rows of more than 8192
// entries get their exponents from a pass of their own.
#include "common.cuh"
#include "kernels.h"
#include "launch.h"

namespace mera {
namespace {

constexpr int kThreadsX = 256;
constexpr int kItems = 4;                        // groups of 8 entries per thread
constexpr int kCap = kThreadsX * kItems * 8;     // entries per block of threads

struct SplitArgs {
  const double* src;
  int64_t ld, rows, K, seg_rows, tiles_per_seg;
  uint8_t* img;
  int* rowexp;
  int tile, nk;        // rows per tile, 16-wide steps of K
  int R, G;            // rows and groups of 8 entries per block of threads
  int known;           // rowexp holds the rows' exponents already
  int gx;              // blocks of threads along the rows
  int pairs;           // entries of a row may be read two at a time
};
struct SplitGroup {
  int n;
  int end[kGroup];     // blocks of the jobs up to and including each
  int rend[kGroup];    // rows whose exponents need a pass of their own, likewise
  SplitArgs job[kGroup];
};

// High word of |x|, at least 1 unless x is zero: orders entries by magnitude
// up to the exponent and the leading bits.
__device__ __forceinline__ int mag_word(double x) {
  const int hi = __double2hiint(x) & 0x7FFFFFFF;
  return hi == 0 && __double2loint(x) != 0 ? 1 : hi;
}

// Exponent of a row from its largest magnitude word.
__device__ __forceinline__ int row_exponent(int w) {
  const int e = (w >> 20) - 1023;
  if (w == 0) return 0;  // all zeros: every digit is zero
  return (e > kX64MaxExp || e < -kX64MaxExp) ? kX64Bad : e;
}

__global__ void __launch_bounds__(512) x64_rowexp_kernel(const __grid_constant__ SplitGroup g) {
  pdl_begin();
  __shared__ int sm[16];
  for (int64_t rg = blockIdx.x; rg < g.rend[g.n - 1]; rg += gridDim.x) {
    int i = 0;
    while (rg >= g.rend[i]) ++i;
    const SplitArgs& a = g.job[i];
    const int64_t r = rg - (i > 0 ? g.rend[i - 1] : 0);
    const double* p = a.src + r * a.ld;
    int w = 0;
    for (int64_t k = threadIdx.x; k < a.K; k += blockDim.x) w = max(w, mag_word(p[k]));
    w = __reduce_max_sync(0xffffffffu, w);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < 16; ++k) w = max(w, sm[k]);
      a.rowexp[r] = row_exponent(w);
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kThreadsX, 2) x64_split_kernel(const __grid_constant__ SplitGroup gr) {
  pdl_begin();
  int job = 0;
  while (int(blockIdx.x) >= gr.end[job]) ++job;
  const int block = int(blockIdx.x) - (job > 0 ? gr.end[job - 1] : 0);
  const SplitArgs& a = gr.job[job];
  extern __shared__ int s_max[];  // [R][blocks of 256]: magnitude words, then [R] row exponents
  const int nb = (a.G * 8 + kX64Block - 1) / kX64Block;
  int* s_row = s_max + a.R * nb;
  const int64_t r0 = int64_t(block % a.gx) * a.R;
  const int kbase = block / a.gx * a.G * 8;
  const int rlow = min(a.R, 8);  // rows run fastest over the threads: stores fill whole core matrices
  for (int i = threadIdx.x; i < a.R * nb; i += kThreadsX) s_max[i] = 0;
  __syncthreads();

  double x[kItems][8];
  int rr[kItems], gg[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const int id = threadIdx.x + kThreadsX * i;
    const int q = id / rlow;
    const int g = q % a.G;
    const int r = id % rlow + rlow * (q / a.G);
    rr[i] = (r < a.R && r0 + r < a.rows && kbase / 16 + g / 2 < a.nk) ? r : -1;
    gg[i] = g;
#pragma unroll
    for (int j = 0; j < 8; ++j) x[i][j] = 0.0;
    if (rr[i] < 0) continue;
    const int64_t k = kbase + g * 8;
    const double* s = a.src + (r0 + r) * a.ld + k;
    if (a.pairs && k + 8 <= a.K) {
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        const double2 d = *reinterpret_cast<const double2*>(s + j);
        x[i][j] = d.x;
        x[i][j + 1] = d.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (k + j < a.K) x[i][j] = s[j];
    }
  }
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    if (rr[i] < 0) continue;
    int w = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) w = max(w, mag_word(x[i][j]));
    atomicMax(&s_max[rr[i] * nb + gg[i] * 8 / kX64Block], w);
  }
  __syncthreads();
  for (int r = threadIdx.x; r < a.R; r += kThreadsX) {
    if (r0 + r >= a.rows) continue;
    int e;
    if (a.known) {
      e = a.rowexp[r0 + r];
    } else {
      int w = 0;
      for (int b = 0; b < nb; ++b) w = max(w, s_max[r * nb + b]);
      e = row_exponent(w);
      a.rowexp[r0 + r] = e;
    }
    s_row[r] = e;
  }
  __syncthreads();

#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    if (rr[i] < 0) continue;
    const int e = s_row[rr[i]];
    const int w = s_max[rr[i] * nb + gg[i] * 8 / kX64Block];
    const int b = max((w >> 20) - 1023, e - 24);  // exponent of the block's grid
    const bool zero = w == 0 || e == kX64Bad;
    uint32_t lo[8], hi[8], mag[8], top = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x[i][j]));
      const int ex = int(u >> 52) & 0x7FF;
      long long X = static_cast<long long>((u & 0xFFFFFFFFFFFFFull) | (ex ? 0x10000000000000ull : 0ull));
      const int sh = ex - 1023 - b + 10;  // X 2^sh multiples of 2^(b-62), below 2^63
      if (sh >= 0)
        X <<= sh;  // at most 10, ex - 1023 <= b
      else
        X = sh < -54 ? 0 : (X + (1ll << (-sh - 1))) >> -sh;
      if (static_cast<long long>(u) < 0) X = -X;
      if (zero) X = 0;
      const unsigned long long Y = static_cast<unsigned long long>(X) + 0x8080808080808080ull;
      lo[j] = uint32_t(Y);
      hi[j] = uint32_t(Y >> 32);
      // the top digit of a positive X may be 128: its byte has wrapped to 0
      if (X >= 0 && static_cast<long long>(Y) >= 0) top |= 1u << j;
      const int em = max(ex - 1023 - e, -60);
      const uint32_t v = (uint32_t(em + 127) << 7) | (em > -60 ? uint32_t(u >> 45) & 0x7Fu : 0u);
      mag[j] = zero || (u << 1) == 0 ? 0u : v;
    }
    const int64_t r = r0 + rr[i];
    const int64_t seg = r / a.seg_rows, rs = r - seg * a.seg_rows;
    const int64_t t = seg * a.tiles_per_seg + rs / a.tile;
    const int ri = int(rs % a.tile);
    const int g = kbase / 8 + gg[i];
    const int plane = a.tile * 32;
    uint8_t* d = a.img + t * a.nk * int64_t(kX64Planes * plane) + (ri / 8) * 256 + (g & 1) * 128 + (ri % 8) * 16;
    *reinterpret_cast<uint4*>(d + (int64_t(a.nk) * kX64Digits + g / 2) * plane) =
        make_uint4(mag[0] | mag[1] << 16, mag[2] | mag[3] << 16, mag[4] | mag[5] << 16, mag[6] | mag[7] << 16);
    d += int64_t(g / 2) * (kX64Digits * plane);
#pragma unroll
    for (int p = 0; p < kX64Digits; ++p) {
      const float sc = zero ? 0.0f : __int_as_float((b - e - 6 - 8 * p + 127) << 23);
      const float off = -8388736.0f * sc;  // -(2^23 + 128) sc
      uint32_t f[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t u = __byte_perm(p <= 3 ? hi[j] : lo[j], 0x4B000000u, 0x7440u + uint32_t(p <= 3 ? 3 - p : 7 - p));
        if (p == 0) u += (top >> j & 1u) << 8;
        f[j] = __float_as_uint(__fmaf_rn(__uint_as_float(u), sc, off));
      }
      uint4 o;  // BF16 pairs: the values are exact in the upper halves
      o.x = __byte_perm(f[0], f[1], 0x7632);
      o.y = __byte_perm(f[2], f[3], 0x7632);
      o.z = __byte_perm(f[4], f[5], 0x7632);
      o.w = __byte_perm(f[6], f[7], 0x7632);
      *reinterpret_cast<uint4*>(d + p * plane) = o;
    }
  }
}

}  // namespace

static cudaError_t launch_group(const X64SplitJob* jobs, int n, cudaStream_t stream) {
  SplitGroup g;
  g.n = 0;
  int64_t blocks = 0, rows_known = 0;
  size_t smem = 0;
  for (int i = 0; i < n; ++i) {
    const X64SplitJob& j = jobs[i];
    if (j.rows <= 0 || j.K <= 0) continue;
    if (j.K > (1 << 30) || j.seg_rows <= 0 || j.rows % j.seg_rows) return cudaErrorInvalidValue;
    SplitArgs& a = g.job[g.n];
    a.src = j.src;
    a.ld = j.ld;
    a.pairs = (j.ld & 1) == 0 && (reinterpret_cast<uintptr_t>(j.src) & 15) == 0;
    a.rows = j.rows;
    a.K = j.K;
    a.seg_rows = j.seg_rows;
    a.tiles_per_seg = (j.seg_rows + j.tile - 1) / j.tile;
    a.img = static_cast<uint8_t*>(j.img);
    a.rowexp = j.rowexp;
    a.tile = j.tile;
    a.nk = int((j.K + 15) / 16);
    const int kp = a.nk * 16;
    int64_t ksegs = 1;
    if (kp <= kCap) {
      a.known = 0;
      a.G = kp / 8;
      int R = 1;
      while (2 * R * kp <= kCap && R < 256) R *= 2;
      // at least two blocks of threads per SM where the rows allow it
      while (R > 8 && (j.rows + R - 1) / R < 2 * 152) R /= 2;
      a.R = R;
    } else {
      a.known = 1;
      a.R = 8;
      a.G = kCap / 8 / 8;  // 1024 of K: four blocks of 256
      ksegs = (kp + a.G * 8 - 1) / (a.G * 8);
      rows_known += j.rows;
    }
    const int64_t gx = (j.rows + a.R - 1) / a.R;
    blocks += gx * ksegs;
    if (blocks > 0x7fffffff || rows_known > 0x7fffffff) return cudaErrorInvalidValue;
    a.gx = int(gx);
    g.end[g.n] = int(blocks);
    g.rend[g.n] = int(rows_known);
    const int nb = (a.G * 8 + kX64Block - 1) / kX64Block;
    smem = std::max(smem, size_t(a.R) * (nb + 1) * sizeof(int));
    ++g.n;
  }
  if (g.n == 0) return cudaSuccess;
  if (rows_known > 0) {
    count_launch();
    launch(x64_rowexp_kernel, rows_known <= 304, unsigned(std::min<int64_t>(rows_known, 152 * 16)), 512, 0, stream, g);
  }
  count_launch();
  launch(x64_split_kernel, blocks <= 304, unsigned(blocks), kThreadsX, smem, stream, g);
  return cudaGetLastError();
}

cudaError_t launch_x64_split(const X64SplitJob* jobs, int n, cudaStream_t stream) {
  for (int i = 0; i < n; i += kGroup) {
    const cudaError_t e = launch_group(jobs + i, std::min(kGroup, n - i), stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mera
