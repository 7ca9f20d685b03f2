// Binary64 kernels: operand permute/cast, FP64 GEMM with scattered epilogue,
// deterministic reductions (trace, Hilbert-Schmidt products, norms) and the
// elementwise parts of the polar iteration (quintic Newton-Schulz).
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"

namespace mera {

// ---------------------------------------------------------------------------
// Input tensor -> operand layout, cast to the operand precision.
//
// The copy is a permutation of the tensor's legs.  The legs are grouped into
// A (those of smallest destination stride, up to kTile elements), B (those of
// smallest source stride among the rest, up to kTile elements) and the outer
// legs; a leg is split in two where that makes a group fill exactly.  Each
// block moves TA x TB tiles through shared memory: reads run along B (or
// along A when A is also contiguous in the source), writes along A, so both
// sides move runs of up to kTile elements.  The in-tile offsets come from
// tables in shared memory and the outer offsets are decoded once per tile.
// ---------------------------------------------------------------------------
constexpr int kTile = 64;

struct PermuteArgs {
  int n_other;
  int64_t dim[2 * kMaxLeg], src_stride[2 * kMaxLeg], dst_stride[2 * kMaxLeg];  // outer legs
  int ta, tb;              // tile extents (products of the A and B legs)
  int read_a;              // A is contiguous in the source too: read along A
  int64_t outer;           // number of tiles (product of the outer legs)
  int64_t a_src[kTile], a_dst[kTile], b_src[kTile], b_dst[kTile];  // in-tile offsets
};

// o < 2^31 (checked at launch), so the decode divides in 32 bits.
__device__ __forceinline__ void decode_other(const PermuteArgs& p, uint32_t o, int64_t& so, int64_t& dof) {
  so = 0;
  dof = 0;
#pragma unroll 1
  for (int i = p.n_other - 1; i >= 0; --i) {
    const uint32_t d = uint32_t(p.dim[i]);
    const uint32_t q = o / d;
    const int64_t x = int64_t(o - q * d);
    so += x * p.src_stride[i];
    dof += x * p.dst_stride[i];
    o = q;
  }
}

struct PermuteJobArgs {
  const double* src;
  void* dst;
  int64_t plane;
  PermuteArgs p;
};
template <int G>
struct PermuteGroup {
  int n;
  int64_t end[G];  // tiles of the jobs up to and including each
  PermuteJobArgs job[G];
};

// Tiles of every job one after another; a block reloads its offset tables
// when its next tile belongs to another job.  A launch of one job has its
// parameters at fixed addresses and its tables and divisors made once: looked
// up per tile, the copies took 7 to 8 % longer (chi = 24 BF16X3 descend 0.79 ms
// instead of 0.74, chi = 20 TF32 env_w 2.42 instead of 2.23).
template <int PREC, int G>
__global__ void __launch_bounds__(256) permute_tile_kernel(const __grid_constant__ PermuteGroup<G> g) {
  pdl_begin();
  __shared__ double tile[kTile * (kTile + 1)];
  __shared__ int64_t s_as[kTile], s_ad[kTile], s_bs[kTile], s_bd[kTile];
  const int tid = threadIdx.x;
  auto load_tables = [&](const PermuteArgs& p) {
    if (tid < kTile) {
      s_as[tid] = tid < p.ta ? p.a_src[tid] : 0;
      s_ad[tid] = tid < p.ta ? p.a_dst[tid] : 0;
      s_bs[tid] = tid < p.tb ? p.b_src[tid] : 0;
      s_bd[tid] = tid < p.tb ? p.b_dst[tid] : 0;
    }
    __syncthreads();
  };
  // x / d for x < 2^13 by a float reciprocal: (x + 0.5) / d is at least
  // 0.5 / d away from an integer, far more than the float rounding error
  auto copy_tile = [&](const PermuteArgs& p, const double* __restrict__ src, void* dst, int64_t plane, int ta, int tb,
                       float inv_ta, float inv_tb, int64_t t) {
    const int count = ta * tb;
    const int pitch = tb + 1;  // tile[ia * pitch + ib]
    int64_t so, dof;
    decode_other(p, uint32_t(t), so, dof);
    // reads: 8 independent loads per thread in flight before any shared store
    for (int e0 = 0; e0 < count; e0 += 256 * 8) {
      double v[8];
      int slot[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int e = e0 + tid + 256 * k;
        slot[k] = -1;
        v[k] = 0.0;
        if (e < count) {
          int ia, ib;
          if (p.read_a) {
            ib = int((float(e) + 0.5f) * inv_ta);
            ia = e - ib * ta;
          } else {
            ia = int((float(e) + 0.5f) * inv_tb);
            ib = e - ia * tb;
          }
          v[k] = src[so + s_as[ia] + s_bs[ib]];
          slot[k] = ia * pitch + ib;
        }
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (slot[k] >= 0) tile[slot[k]] = v[k];
    }
    __syncthreads();
    // writes along A (contiguous in the destination)
    for (int e = tid; e < count; e += 256) {
      const int ib = int((float(e) + 0.5f) * inv_ta), ia = e - ib * ta;
      OperandStore<PREC>::store(dst, dof + s_ad[ia] + s_bd[ib], plane, tile[ia * pitch + ib]);
    }
    __syncthreads();
  };
  const int64_t total = g.end[g.n - 1];
  if constexpr (G == 1) {
    const PermuteArgs& p = g.job[0].p;
    const int ta = p.ta, tb = p.tb;
    const float inv_ta = 1.0f / float(ta), inv_tb = 1.0f / float(tb);
    load_tables(p);
    for (int64_t t = blockIdx.x; t < total; t += gridDim.x)
      copy_tile(p, g.job[0].src, g.job[0].dst, g.job[0].plane, ta, tb, inv_ta, inv_tb, t);
  } else {
    int cur = -1;
    for (int64_t tg = blockIdx.x; tg < total; tg += gridDim.x) {
      int i = 0;
      while (tg >= g.end[i]) ++i;
      const PermuteArgs& p = g.job[i].p;
      if (i != cur) {
        cur = i;
        load_tables(p);
      }
      copy_tile(p, g.job[i].src, g.job[i].dst, g.job[i].plane, p.ta, p.tb, 1.0f / float(p.ta), 1.0f / float(p.tb),
                tg - (i > 0 ? g.end[i - 1] : 0));
    }
  }
}

namespace {

struct Leg {
  int64_t dim, ss, ds;
};

// Take legs from `pool` in order of `key` into a group of at most kTile
// elements; the first leg that does not fit whole is split when a divisor
// of its size fills the group further.  Returns the group's legs, inner first.
template <typename Key>
std::vector<Leg> take_group(std::vector<Leg>& pool, Key key) {
  std::stable_sort(pool.begin(), pool.end(), [&](const Leg& x, const Leg& y) { return key(x) < key(y); });
  std::vector<Leg> g;
  int64_t prod = 1;
  while (!pool.empty()) {
    Leg l = pool.front();
    if (prod * l.dim <= kTile) {
      g.push_back(l);
      prod *= l.dim;
      pool.erase(pool.begin());
      continue;
    }
    int64_t q = kTile / prod;
    while (q > 1 && l.dim % q) --q;
    if (q > 1) {  // inner part (q values) joins the group, outer part stays
      g.push_back({q, l.ss, l.ds});
      pool.front() = {l.dim / q, l.ss * q, l.ds * q};
      prod *= q;
    }
    break;
  }
  return g;
}

// In-tile offsets of a group: index i = sum over legs of x_leg * (product
// of the inner legs' sizes), inner leg fastest.
int fill_table(const std::vector<Leg>& g, int64_t* src_off, int64_t* dst_off) {
  int n = 1;
  src_off[0] = dst_off[0] = 0;
  for (const Leg& l : g) {
    for (int64_t x = 1; x < l.dim; ++x)
      for (int i = 0; i < n; ++i) {
        src_off[x * n + i] = src_off[i] + x * l.ss;
        dst_off[x * n + i] = dst_off[i] + x * l.ds;
      }
    n *= int(l.dim);
  }
  return n;
}

}  // namespace

namespace {

// Tile description of one copy; false where its tile indices exceed 32 bits.
bool permute_args(const PermuteStep& st, PermuteArgs& p) {
  // Every leg with its source and destination strides (size-1 legs dropped).
  std::vector<Leg> pool;
  int64_t acc = st.ld;
  for (int i = st.row_src.n - 1; i >= 0; --i) {
    if (st.row_src.dim[i] > 1) pool.push_back({st.row_src.dim[i], st.row_src.stride[i], acc});
    acc *= st.row_src.dim[i];
  }
  acc = 1;
  for (int i = st.col_src.n - 1; i >= 0; --i) {
    if (st.col_src.dim[i] > 1) pool.push_back({st.col_src.dim[i], st.col_src.stride[i], acc});
    acc *= st.col_src.dim[i];
  }
  // Ls: the leg contiguous in the source, Ld: the one contiguous in the
  // destination.  When they differ, Ls is kept out of A so that it leads B;
  // when they coincide, A leads with it and the reads run along A.
  p = PermuteArgs{};
  std::vector<Leg> ga, gb;
  if (!pool.empty()) {
    size_t is = 0, id = 0;
    for (size_t i = 1; i < pool.size(); ++i) {
      if (pool[i].ss < pool[is].ss) is = i;
      if (pool[i].ds < pool[id].ds) id = i;
    }
    if (is == id) {
      p.read_a = 1;
      ga = take_group(pool, [](const Leg& l) { return l.ds; });
      gb = take_group(pool, [](const Leg& l) { return l.ss; });
    } else {
      const Leg ls = pool[is];
      pool.erase(pool.begin() + long(is));
      ga = take_group(pool, [](const Leg& l) { return l.ds; });
      pool.push_back(ls);
      gb = take_group(pool, [](const Leg& l) { return l.ss; });
    }
  }
  p.ta = fill_table(ga, p.a_src, p.a_dst);
  p.tb = fill_table(gb, p.b_src, p.b_dst);
  if (int(pool.size()) > 2 * kMaxLeg) return false;
  p.outer = 1;
  p.n_other = 0;
  for (const Leg& l : pool) {  // outer legs (order is irrelevant for correctness)
    p.dim[p.n_other] = l.dim;
    p.src_stride[p.n_other] = l.ss;
    p.dst_stride[p.n_other] = l.ds;
    p.outer *= l.dim;
    ++p.n_other;
  }
  return p.outer < (int64_t(1) << 31);
}

template <int G>
cudaError_t launch_permute_group(const PermuteJob* jobs, int n, int prec, cudaStream_t stream) {
  static thread_local PermuteGroup<G> g;  // up to 15 KB
  g.n = 0;
  int64_t total = 0;
  for (int i = 0; i < n; ++i) {
    if (jobs[i].step->rows <= 0 || jobs[i].step->cols <= 0) continue;
    PermuteJobArgs& a = g.job[g.n];
    if (!permute_args(*jobs[i].step, a.p)) return cudaErrorInvalidValue;
    a.src = jobs[i].src;
    a.dst = jobs[i].dst;
    a.plane = jobs[i].plane;
    total += a.p.outer;
    g.end[g.n++] = total;
  }
  if (g.n == 0) return cudaSuccess;
  count_launch();
  const unsigned grid = unsigned(std::max<int64_t>(1, std::min<int64_t>(total, 152 * 8)));
#define MERA_PERMUTE_LAUNCH(P) launch(permute_tile_kernel<P, G>, total <= 152 * 6, grid, 256, 0, stream, g);
  switch (prec) {
    case PREC_F64: MERA_PERMUTE_LAUNCH(PREC_F64) break;
    case PREC_TF32: MERA_PERMUTE_LAUNCH(PREC_TF32) break;
    case PREC_BF16: MERA_PERMUTE_LAUNCH(PREC_BF16) break;
    case PREC_BF16X3: MERA_PERMUTE_LAUNCH(PREC_BF16X3) break;
    case PREC_BF16X6: MERA_PERMUTE_LAUNCH(PREC_BF16X6) break;
    case PREC_OZ3:
    case PREC_OZ4:  // into the raw hi + lo planes; the split step follows
    case PREC_RAW: MERA_PERMUTE_LAUNCH(PREC_RAW) break;
    default: return cudaErrorInvalidValue;
  }
#undef MERA_PERMUTE_LAUNCH
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_permute(const PermuteJob* jobs, int n, int prec, cudaStream_t stream) {
  for (int i = 0; i < n; i += kGroup) {
    const int m = std::min(kGroup, n - i);
    const cudaError_t e = m == 1 ? launch_permute_group<1>(jobs + i, m, prec, stream)
                                 : launch_permute_group<kGroup>(jobs + i, m, prec, stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// FP64 GEMM.  (16 T) x (16 T) tile per block of 256 threads, T x T outputs per
// thread at stride 16 (conflict-free shared-memory reads), K in steps of 16.
// T = 4 for large problems; T = 2 or 1 when the tile count would leave most
// of the 152 SMs idle (the small square products of the polar iteration), and
// gemm_f64_small_kernel below that.
// ---------------------------------------------------------------------------
constexpr int kBK = 16;

struct GemmF64Group {
  int n;
  int end[kGroup];  // blocks of the jobs up to and including each
  GemmF64Args job[kGroup];
};

// Job of a block, and the block's index within it.
__device__ __forceinline__ int job_of(const int* end, int b, int& local) {
  int i = 0;
  while (b >= end[i]) ++i;
  local = b - (i > 0 ? end[i - 1] : 0);
  return i;
}

// 8 x 8 tile per block of 256 threads, four threads per output, each with a
// quarter of every 64-wide stage of K; their sums meet in a fixed order.
// Products of this size are bound by latency and by the FP64 pipe of the SMs
// they reach (two FMAs per clock): small tiles reach more of them, one stage
// covers K <= 64 with one round trip to memory, and the next stage is in
// flight while this one is summed.  256 x 64 x 64: 6.0 us with 16 x 16 tiles.
__global__ void __launch_bounds__(256) gemm_f64_small_kernel(const __grid_constant__ GemmF64Group g) {
  pdl_begin();
  constexpr int R = 8, KS = 64, P = KS + 2;
  __shared__ double As[R * P], Bs[R * P];
  __shared__ double part[3][R * R];
  int tile;
  const GemmF64Args& p = g.job[job_of(g.end, int(blockIdx.x), tile)];
  if (p.skip_if && *p.skip_if) return;
  const int tid = threadIdx.x;
  const int tiles_n = int((p.N + R - 1) / R);
  const int64_t m0 = int64_t(tile / tiles_n) * R, n0 = int64_t(tile % tiles_n) * R;
  // two elements of each operand per thread and stage, along its unit stride
  int ra[2], ka[2], rb[2], kb[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int e = tid + 256 * i;
    if (p.a_k == 1) { ra[i] = e / KS; ka[i] = e % KS; } else { ra[i] = e % R; ka[i] = e / R; }
    if (p.b_k == 1) { rb[i] = e / KS; kb[i] = e % KS; } else { rb[i] = e % R; kb[i] = e / R; }
  }
  double va[2], vb[2];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int64_t gm = m0 + ra[i], ga = k0 + ka[i], gn = n0 + rb[i], gb = k0 + kb[i];
      va[i] = (gm < p.M && ga < p.K) ? p.A[gm * p.a_m + ga * p.a_k] : 0.0;
      vb[i] = (gn < p.N && gb < p.K) ? p.B[gn * p.b_n + gb * p.b_k] : 0.0;
    }
  };
  const int o = tid % (R * R), q = tid / (R * R);  // output, quarter of K
  const int r = o / R, c = o % R;
  double acc = 0.0;
  load(0);
  for (int64_t k0 = 0; k0 < p.K; k0 += KS) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      As[ra[i] * P + ka[i]] = va[i];
      Bs[rb[i] * P + kb[i]] = vb[i];
    }
    __syncthreads();
    if (k0 + KS < p.K) load(k0 + KS);
    const int left = int(min(int64_t(KS), p.K - k0));
    const int lo = q * (KS / 4), hi = min(left, lo + KS / 4);
    if (p.ordered) {
      if (q == 0) {
#pragma unroll 16
        for (int k = 0; k < left; ++k) acc = fma(As[r * P + k], Bs[c * P + k], acc);
      }
    } else if (hi - lo == KS / 4) {
#pragma unroll
      for (int k = 0; k < KS / 4; ++k) acc = fma(As[r * P + lo + k], Bs[c * P + lo + k], acc);
    } else {
      for (int k = lo; k < hi; ++k) acc = fma(As[r * P + k], Bs[c * P + k], acc);
    }
    __syncthreads();
  }
  if (q > 0) part[q - 1][o] = acc;
  __syncthreads();
  if (q > 0 || m0 + r >= p.M || n0 + c >= p.N) return;
  const double v = p.alpha * (p.ordered ? acc : ((acc + part[0][o]) + part[1][o]) + part[2][o]);
  double* dst = p.C + legmap_offset32(p.m_dst, uint32_t(m0 + r)) + legmap_offset32(p.n_dst, uint32_t(n0 + c));
  *dst = p.accumulate ? (*dst + v) : v;
}

template <int T>
__global__ void __launch_bounds__(256) gemm_f64_kernel(const __grid_constant__ GemmF64Group g) {
  pdl_begin();
  constexpr int R = 16 * T;
  __shared__ double As[kBK][R + 1];
  __shared__ double Bs[kBK][R + 1];
  __shared__ int64_t offm[R];
  __shared__ int64_t offn[R];
  int tile;
  const GemmF64Args& p = g.job[job_of(g.end, int(blockIdx.x), tile)];
  if (p.skip_if && *p.skip_if) return;

  // the K loop's operands in registers: the job's index is not a constant
  const double* __restrict__ const pa = p.A;
  const double* __restrict__ const pb = p.B;
  const int64_t a_m = p.a_m, a_k = p.a_k, b_n = p.b_n, b_k = p.b_k, M = p.M, N = p.N, K = p.K;
  const int tid = threadIdx.x;
  const int64_t tiles_n = (N + R - 1) / R;
  const int64_t m0 = (tile / tiles_n) * R;
  const int64_t n0 = (tile % tiles_n) * R;
  const int tx = tid % 16, ty = tid / 16;

  double acc[T][T];
#pragma unroll
  for (int i = 0; i < T; ++i)
#pragma unroll
    for (int j = 0; j < T; ++j) acc[i][j] = 0.0;

  const bool a_kfast = (a_k == 1);
  const bool b_kfast = (b_k == 1);

  for (int64_t k0 = 0; k0 < K; k0 += kBK) {
    // R rows x 16 k per operand, T elements per thread, along the unit stride.
#pragma unroll
    for (int i = 0; i < T; ++i) {
      int r, k;
      if (a_kfast) {
        k = tid % 16;
        r = tid / 16 + 16 * i;
      } else {
        r = tid % R;
        k = tid / R + (256 / R) * i;
      }
      const int64_t gm = m0 + r, gk = k0 + k;
      As[k][r] = (gm < M && gk < K) ? pa[gm * a_m + gk * a_k] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < T; ++i) {
      int r, k;
      if (b_kfast) {
        k = tid % 16;
        r = tid / 16 + 16 * i;
      } else {
        r = tid % R;
        k = tid / R + (256 / R) * i;
      }
      const int64_t gn = n0 + r, gk = k0 + k;
      Bs[k][r] = (gn < N && gk < K) ? pb[gn * b_n + gk * b_k] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
      double a[T], b[T];
#pragma unroll
      for (int i = 0; i < T; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < T; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

  for (int t = tid; t < 2 * R; t += 256) {
    if (t < R) {
      const int64_t gm = m0 + t;
      offm[t] = gm < p.M ? legmap_offset32(p.m_dst, uint32_t(gm)) : 0;
    } else {
      const int64_t gn = n0 + t - R;
      offn[t - R] = gn < p.N ? legmap_offset32(p.n_dst, uint32_t(gn)) : 0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < T; ++i) {
    const int r = ty + 16 * i;
    if (m0 + r >= p.M) continue;
#pragma unroll
    for (int j = 0; j < T; ++j) {
      const int c = tx + 16 * j;
      if (n0 + c >= p.N) continue;
      double* dst = p.C + offm[r] + offn[c];
      const double v = p.alpha * acc[i][j];
      *dst = p.accumulate ? (*dst + v) : v;
    }
  }
}

constexpr int64_t kFill = 2 * 152;  // enough blocks to occupy every SM twice

// Whether a product goes to gemm_f64_small_kernel.  It alone sums in another
// order, so this is for each product by its own size and not by its group's:
// the result does not depend on what else runs in the launch.
static bool gemm_f64_is_small(const GemmF64Args& a) { return ((a.M + 15) / 16) * ((a.N + 15) / 16) < kFill; }

// Jobs that are all small, or all not.
static cudaError_t launch_gemm_f64_group(GemmF64Group& g, cudaStream_t stream) {
  if (g.n == 0) return cudaSuccess;
  const bool small = gemm_f64_is_small(g.job[0]);
  auto blocks = [&](int64_t r) {
    int64_t t = 0;
    for (int i = 0; i < g.n; ++i) {
      t += ((g.job[i].M + r - 1) / r) * ((g.job[i].N + r - 1) / r);
      g.end[i] = int(std::min<int64_t>(t, 0x7fffffff));
    }
    return t;
  };
  int64_t r = small ? 8 : 16;
  for (int64_t q : {64, 32})
    if (r == 16 && (blocks(q) >= kFill || blocks(q / 2) > 0x7fffffff)) r = q;
  const int64_t nb = blocks(r);
  if (nb > 0x7fffffff) return cudaErrorInvalidValue;
  count_launch();
  switch (r) {
    case 64: launch(gemm_f64_kernel<4>, nb <= 304, unsigned(nb), 256, 0, stream, g); break;
    case 32: launch(gemm_f64_kernel<2>, nb <= 304, unsigned(nb), 256, 0, stream, g); break;
    case 16: launch(gemm_f64_kernel<1>, nb <= 304, unsigned(nb), 256, 0, stream, g); break;
    default: launch(gemm_f64_small_kernel, nb <= 304, unsigned(nb), 256, 0, stream, g); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_gemm_f64(const GemmF64Args* args, int n, cudaStream_t stream) {
  GemmF64Group g[2];
  g[0].n = g[1].n = 0;
  for (int i = 0; i < n; ++i) {
    if (args[i].M <= 0 || args[i].N <= 0) continue;
    if (args[i].M > 0x7fffffff || args[i].N > 0x7fffffff) return cudaErrorInvalidValue;  // 32-bit row/column decode
    GemmF64Group& to = g[gemm_f64_is_small(args[i]) ? 1 : 0];
    to.job[to.n++] = args[i];
    if (to.n < kGroup) continue;
    const cudaError_t e = launch_gemm_f64_group(to, stream);
    if (e != cudaSuccess) return e;
    to.n = 0;
  }
  const cudaError_t e = launch_gemm_f64_group(g[0], stream);
  return e != cudaSuccess ? e : launch_gemm_f64_group(g[1], stream);
}

__global__ void __launch_bounds__(256) ordered_sum_kernel(const double* parts, int n,
                                                          double* out, int64_t count) {
  pdl_begin();
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x) {
    double v = parts[i];
    for (int k = 1; k < n; ++k) v += parts[k * count + i];
    out[i] = v;
  }
}

cudaError_t launch_ordered_sum(const double* parts, int n, double* out, int64_t count, cudaStream_t stream) {
  if (count <= 0) return cudaSuccess;
  count_launch();
  launch(ordered_sum_kernel, count <= 152 * 256, unsigned(std::min<int64_t>((count + 255) / 256, 152 * 8)), 256, 0, stream, parts, n, out, count);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Deterministic reductions: each block writes one partial, one block sums the
// partials in a fixed order.
// ---------------------------------------------------------------------------
template <int NT>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[NT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = (threadIdx.x < NT / 32) ? sh[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;  // valid in thread 0
}

// mode 0: out = sum; mode 1: out = sqrt(sum)
__global__ void __launch_bounds__(1024) reduce_partials_kernel(const double* partials, int np,
                                                               double* out, int mode) {
  pdl_begin();
  double v = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) v += partials[i];
  v = block_sum<1024>(v);
  if (threadIdx.x == 0) *out = mode == 1 ? sqrt(v) : v;
}

// 32 x 32 tiles of an n x n matrix, block (32, 8).  tile (ti, tj) covers rows
// [32 ti, 32 ti + 32) and columns [32 tj, ...).  The transposed tile of B is
// staged through shared memory so both reads are coalesced.
__global__ void __launch_bounds__(256) dot_t_kernel(const double* A, const double* B,
                                                    int64_t n, double* partials) {
  pdl_begin();
  __shared__ double bt[32][33];
  const int64_t nt = (n + 31) / 32;
  double v = 0.0;
  for (int64_t t = blockIdx.x; t < nt * nt; t += gridDim.x) {
    const int64_t i0 = (t / nt) * 32, j0 = (t % nt) * 32;
    // bt[c][r] = B[j0 + r][i0 + c]
    for (int r = threadIdx.y; r < 32; r += 8) {
      const int64_t gj = j0 + r, gi = i0 + threadIdx.x;
      bt[threadIdx.x][r] = (gj < n && gi < n) ? B[gj * n + gi] : 0.0;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8) {
      const int64_t gi = i0 + r, gj = j0 + threadIdx.x;
      if (gi < n && gj < n) v += A[gi * n + gj] * bt[r][threadIdx.x];
    }
    __syncthreads();
  }
  const int tid = threadIdx.y * 32 + threadIdx.x;
  // reuse block_sum with a flat thread index
  __shared__ double sh[8];
  double s = v;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) sh[threadIdx.y] = s;
  __syncthreads();
  if (tid == 0) {
    double tot = 0.0;
    for (int w = 0; w < 8; ++w) tot += sh[w];
    partials[blockIdx.x] = tot;
  }
}

static int reduction_blocks(int64_t tiles) { return int(std::min<int64_t>(std::max<int64_t>(tiles, 1), 4096)); }

cudaError_t launch_dot_transposed(const double* A, const double* B, int64_t n, double* partials, double* out,
                                  cudaStream_t stream) {
  const int64_t nt = (n + 31) / 32;
  const int nb = reduction_blocks(nt * nt);
  count_launch(2);
  launch(dot_t_kernel, nb <= 304, nb, dim3(32, 8), 0, stream, A, B, n, partials);
  launch(reduce_partials_kernel, true, 1, 1024, 0, stream, partials, nb, out, 0);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(1024) trace_kernel(const double* X, int64_t n, double* out) {
  pdl_begin();
  double v = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) v += X[i * n + i];
  v = block_sum<1024>(v);
  if (threadIdx.x == 0) *out = v;
}

// rho = (X + X^T) / (2 tr X) over pairs of 32 x 32 tiles (I, J), I <= J:
// both tiles are read once and both written once, so X is read once in all,
// and each pair of entries is summed and scaled once (the sum commutes): at
// two binary64 operations per entry the FP64 pipe, not memory, set the pace
// (chi = 16, 268 MB: 96 us with both sums, 70 with one).  Blocks walk the pairs row by row of tiles.
template <bool RESID>
__global__ void __launch_bounds__(256) sym_normalize_kernel(const double* X, double* rho, int64_t n,
                                                            const double* trace, double* partials) {
  pdl_begin();
  __shared__ double sa[32][33], sb[32][33];
  const double inv2t = 0.5 / *trace;
  const int64_t nt = (n + 31) / 32;
  double v = 0.0;
  // pair t of the upper triangle: row I holds nt - I of them
  int64_t I = 0, base = 0;
  const int64_t pairs = nt * (nt + 1) / 2;
  for (int64_t t = blockIdx.x; t < pairs; t += gridDim.x) {
    while (t >= base + (nt - I)) {
      base += nt - I;
      ++I;
    }
    const int64_t J = I + (t - base);
    const int64_t i0 = I * 32, j0 = J * 32;
    for (int r = threadIdx.y; r < 32; r += 8) {
      const int64_t ga = i0 + r, gb = j0 + threadIdx.x;  // tile (I, J)
      sa[r][threadIdx.x] = (ga < n && gb < n) ? X[ga * n + gb] : 0.0;
      const int64_t gc = j0 + r, gd = i0 + threadIdx.x;  // tile (J, I)
      sb[r][threadIdx.x] = (gc < n && gd < n) ? X[gc * n + gd] : 0.0;
    }
    __syncthreads();
    double nv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = threadIdx.y + 8 * q;
      const int64_t gi = i0 + r, gj = j0 + threadIdx.x;
      nv[q] = (sa[r][threadIdx.x] + sb[threadIdx.x][r]) * inv2t;
      if (gi < n && gj < n) {
        if constexpr (RESID) {
          const double d = nv[q] - rho[gi * n + gj];
          v += d * d;
        }
        rho[gi * n + gj] = nv[q];
      }
    }
    if (I != J) {
      // the mirrored tile, through shared memory (each entry of sa is read
      // above by the thread that overwrites it here)
#pragma unroll
      for (int q = 0; q < 4; ++q) sa[threadIdx.y + 8 * q][threadIdx.x] = nv[q];
      __syncthreads();
      for (int r = threadIdx.y; r < 32; r += 8) {
        const int64_t gi = j0 + r, gj = i0 + threadIdx.x;
        if (gi < n && gj < n) {
          const double x = sa[threadIdx.x][r];
          if constexpr (RESID) {
            const double d = x - rho[gi * n + gj];
            v += d * d;
          }
          rho[gi * n + gj] = x;
        }
      }
    }
    __syncthreads();
  }
  if constexpr (RESID) {
    __shared__ double sh[8];
    double s = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) sh[threadIdx.y] = s;
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      double tot = 0.0;
      for (int w = 0; w < 8; ++w) tot += sh[w];
      partials[blockIdx.x] = tot;
    }
  }
}

cudaError_t launch_sym_normalize(const double* X, double* rho, int64_t n, double* partials, double* scalars,
                                 double* resid, cudaStream_t stream) {
  launch(trace_kernel, true, 1, 1024, 0, stream, X, n, scalars);
  const int64_t nt = (n + 31) / 32;
  const int nb = reduction_blocks(nt * (nt + 1) / 2);
  if (resid) {
    count_launch(3);
    launch(sym_normalize_kernel<true>, nb <= 304, nb, dim3(32, 8), 0, stream, X, rho, n, scalars, partials);
    launch(reduce_partials_kernel, true, 1, 1024, 0, stream, partials, nb, resid, 1);
  } else {
    count_launch(2);
    launch(sym_normalize_kernel<false>, nb <= 304, nb, dim3(32, 8), 0, stream, X, rho, n, scalars, partials);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Polar (quintic Newton-Schulz) helpers.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) sumsq_kernel(const double* x, int64_t count, double* partials) {
  pdl_begin();
  double v = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x)
    v += x[i] * x[i];
  v = block_sum<256>(v);
  if (threadIdx.x == 0) partials[blockIdx.x] = v;
}

__global__ void __launch_bounds__(256) scale_by_inverse_kernel(const double* src, double* dst,
                                                               int64_t count, const double* norm) {
  pdl_begin();
  const double s = 1.0 / *norm;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x)
    dst[i] = src[i] * s;
}

// Gershgorin rescale of the first Newton-Schulz step: with G = X^T X and
// c = max_i sum_j |G_ij| >= lambda_max(G), X / sqrt(c) has every singular
// value in (0, 1] and the same polar factor, usually much closer to 1 than
// the Frobenius scaling leaves them.  The largest sum is kept by its bit
// pattern (non-negative binary64 values order like integers), so *c starts at
// zero.  One thread per column (G is symmetric), its sum in order.
__global__ void __launch_bounds__(64) ns_gershgorin_kernel(const double* G, int64_t n, double* c) {
  pdl_begin();
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double r = 0.0;
#pragma unroll 8
  for (int64_t j = 0; j < n; ++j) r += fabs(G[j * n + i]);
  atomicMax(reinterpret_cast<unsigned long long*>(c), static_cast<unsigned long long>(__double_as_longlong(r)));
}

__global__ void __launch_bounds__(256) ns_prescale_kernel(double* G, int64_t gcount, double* X, int64_t xcount,
                                                          const double* c) {
  pdl_begin();
  const double ig = 1.0 / *c, ix = 1.0 / sqrt(*c);
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < gcount + xcount;
       i += int64_t(gridDim.x) * blockDim.x) {
    if (i < gcount)
      G[i] *= ig;
    else
      X[i - gcount] *= ix;
  }
}

cudaError_t launch_ns_prescale(double* G, double* X, int64_t m, int64_t n, double* c, cudaStream_t stream) {
  count_launch(2);
  launch(ns_gershgorin_kernel, true, unsigned((n + 63) / 64), 64, 0, stream, G, n, c);
  const int64_t total = n * n + m * n;
  const int nb = int(std::min<int64_t>((total + 255) / 256, 1024));
  launch(ns_prescale_kernel, nb <= 304, nb, 256, 0, stream, G, n * n, X, m * n, c);
  return cudaGetLastError();
}

cudaError_t launch_frob_scale(const double* src, double* dst, int64_t count, double* partials, double* scalars,
                              cudaStream_t stream) {
  const int nb = int(std::min<int64_t>((count + 255) / 256, 1024));
  count_launch(3);
  launch(sumsq_kernel, nb <= 304, nb, 256, 0, stream, src, count, partials);
  launch(reduce_partials_kernel, true, 1, 1024, 0, stream, partials, nb, scalars, 1);
  launch(scale_by_inverse_kernel, nb <= 304, nb, 256, 0, stream, src, dst, count, scalars);
  return cudaGetLastError();
}

// The step X <- X p(X^T X) with the odd quintic x p(x^2),
//   p(g) = 5/2 - (5/2) g + g^2,  so that x p(x^2) = (5/2) x - (5/2) x^3 + x^5:
// it fixes 1 with zero slope (x p(x^2) - 1 ~ (5/2) (x - 1)^2: quadratic
// convergence, like the cubic (3 x - x^3) / 2), maps [0, 1] into
// [0, 1.061], below its repelling fixed point sqrt(3/2) = 1.225, and grows a
// small singular value 2.5-fold per step where the cubic grows it 1.5-fold.
// At three products per step against two that is 1.36 against 1.22 per
// product; the point is the reach of a step budget: 100 steps bring a
// singular value of 1e-38 of the largest to 1, the cubic's 1e-17.
// Bm = p(G) = (5/2)(I - G) + G2 (G2 = G G) and partial sums of ||G - I||_F^2.
__global__ void __launch_bounds__(256) ns_combine_kernel(const double* G, const double* G2,
                                                         double* Bm, int64_t n, double* partials, const int* skip_if) {
  pdl_begin();
  if (skip_if && *skip_if) return;
  double v = 0.0;
  const int64_t count = n * n;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x) {
    const bool diag = (i / n) == (i % n);
    const double d = G[i] - (diag ? 1.0 : 0.0);
    v += d * d;
    Bm[i] = fma(-2.5, d, G2[i]);
  }
  v = block_sum<256>(v);
  if (threadIdx.x == 0) partials[blockIdx.x] = v;
}

// state[0] = done, state[1] = iterations executed, state[2] = converged after
// this iteration; resid = ||X^T X - I||_F of the iterate entering it.
__global__ void __launch_bounds__(1024) ns_check_kernel(const double* partials, int np, double* resid,
                                                        double tol, int* state) {
  pdl_begin();
  if (state[0]) return;
  double v = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) v += partials[i];
  v = block_sum<1024>(v);
  if (threadIdx.x == 0) {
    const double r = sqrt(v);
    *resid = r;
    state[2] = (r <= tol || !(r == r)) ? 1 : 0;  // converged, or NaN: stop after this step
  }
}

__global__ void ns_finish_kernel(int* state) {
  pdl_begin();
  if (state[0]) return;
  state[1] += 1;
  if (state[2]) state[0] = 1;
}

cudaError_t launch_ns_step(const double* G, const double* G2, double* Bm, int64_t n, double* partials,
                           double* resid, double tol, int* state, cudaStream_t stream) {
  const int nb = int(std::min<int64_t>((n * n + 255) / 256, 1024));
  count_launch(2);
  launch(ns_combine_kernel, nb <= 304, nb, 256, 0, stream, G, G2, Bm, n, partials, state);
  launch(ns_check_kernel, true, 1, 1024, 0, stream, partials, nb, resid, tol, state);
  return cudaGetLastError();
}

cudaError_t launch_ns_finish(int* state, cudaStream_t stream) {
  count_launch();
  launch(ns_finish_kernel, true, 1, 1, 0, stream, state);
  return cudaGetLastError();
}


// One Newton-Schulz step of a small matrix in three launches: G^2 with the
// polynomial, its residual and the convergence check in the epilogue; X B
// (gemm_f64); X^T X, which also closes the step and, in the last step of a
// loop body, decides whether to go on.  G and G^2 are symmetric, so only the
// 8 x 8 tiles on and above the diagonal are summed (tile pairs), which takes a
// third off the FP64 work of a step.  Tiles as in gemm_f64_small_kernel, each
// output one chain of FMAs in the order of K (four chains were 2 % faster, but
// their rounding changed the path of long optimisations).  A step of a
// 256 x 256 matrix was seven launches and 127 us and is 86 us now.
constexpr int kNsR = 8, kNsK = 64, kNsP = kNsK + 2;

// Tile pair t of the upper triangle, row by row: (i, j), i <= j < nt.
__device__ __forceinline__ void tile_pair(int t, int nt, int& i, int& j) {
  i = 0;
  for (int len = nt; t >= len; --len) {
    t -= len;
    ++i;
  }
  j = i + t;
}

// Sum over k of A[i][k] B[j][k] for this thread's output of the tile pair,
// complete in threads 0..63.  KFAST: rows of `x` run along k (x[i * ld + k]);
// else along the outputs (x[k * ld + i]).
template <bool KFAST>
__device__ __forceinline__ double ns_tile(const double* __restrict__ x, int64_t ld, int n, int K, int i0, int j0,
                                          double* As, double* Bs) {
  const int tid = threadIdx.x;
  int r[2], k[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + 256 * q;
    r[q] = KFAST ? e / kNsK : e % kNsR;
    k[q] = KFAST ? e % kNsK : e / kNsR;
  }
  double va[2], vb[2];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int kk = k0 + k[q], gi = i0 + r[q], gj = j0 + r[q];
      va[q] = (gi < n && kk < K) ? x[KFAST ? gi * ld + kk : kk * ld + gi] : 0.0;
      vb[q] = (gj < n && kk < K) ? x[KFAST ? gj * ld + kk : kk * ld + gj] : 0.0;
    }
  };
  const double* a = As + tid / kNsR % kNsR * kNsP;
  const double* b = Bs + tid % kNsR * kNsP;
  const bool sums = tid < kNsR * kNsR;
  double acc = 0.0;
  load(0);
  for (int k0 = 0; k0 < K; k0 += kNsK) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      As[r[q] * kNsP + k[q]] = va[q];
      Bs[r[q] * kNsP + k[q]] = vb[q];
    }
    __syncthreads();
    if (k0 + kNsK < K) load(k0 + kNsK);
    if (sums) {  // in the order of K: an optimisation's path does not depend on the kernel
      const int terms = min(kNsK, K - k0);
      if (terms == kNsK) {
#pragma unroll 16
        for (int t = 0; t < kNsK; ++t) acc = fma(a[t], b[t], acc);
      } else {
        for (int t = 0; t < terms; ++t) acc = fma(a[t], b[t], acc);
      }
    }
    __syncthreads();
  }
  return acc;
}

// Bm = (5/2)(I - G) + G^2; the last block to finish sums the tiles' shares of
// ||G - I||_F^2 in their order and sets state[2].  state[3] counts the blocks
// and is left at zero.
__global__ void __launch_bounds__(256) ns_square_kernel(const double* G, double* Bm, int n,
                                                        double* partials, double* resid, double tol,
                                                        int* state) {
  pdl_begin();
  __shared__ double As[kNsR * kNsP], Bs[kNsR * kNsP];
  __shared__ int last;
  if (state[0]) return;
  int ti, tj;
  tile_pair(int(blockIdx.x), (n + kNsR - 1) / kNsR, ti, tj);
  const int i0 = ti * kNsR, j0 = tj * kNsR;
  const double g2 = ns_tile<true>(G, n, n, n, i0, j0, As, Bs);
  const int tid = threadIdx.x;
  double v = 0.0;
  if (tid < kNsR * kNsR) {
    const int i = i0 + tid / kNsR, j = j0 + tid % kNsR;
    if (i < n && j < n) {
      const double d = G[int64_t(i) * n + j] - (i == j ? 1.0 : 0.0);
      const double b = fma(-2.5, d, g2);
      Bm[int64_t(i) * n + j] = b;
      if (ti != tj) Bm[int64_t(j) * n + i] = b;
      v = ti == tj ? d * d : 2.0 * (d * d);
    }
  }
  v = block_sum<256>(v);
  if (tid == 0) {
    partials[blockIdx.x] = v;
    __threadfence();
    last = atomicAdd(&state[3], 1) == int(gridDim.x) - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  v = 0.0;
  for (int i = tid; i < int(gridDim.x); i += 256) v += __ldcg(partials + i);
  v = block_sum<256>(v);
  if (tid == 0) {
    const double r = sqrt(v);
    *resid = r;
    state[2] = (r <= tol || !(r == r)) ? 1 : 0;  // converged, or NaN: stop after this step
    state[3] = 0;
  }
}

// G = X^T X (m x n, row-major X).  `close`: ends a step (state[1] += 1; done
// if it converged, and then G is not needed).  `cond`: the loop's condition.
__global__ void __launch_bounds__(256) ns_gram_kernel(const double* X, double* G, int m,
                                                      int n, int* state, int close, int set_cond,
                                                      cudaGraphConditionalHandle cond, int max_iter) {
  pdl_begin();
  __shared__ double As[kNsR * kNsP], Bs[kNsR * kNsP];
  // block 0 alone writes state[0] and state[1], and what it writes is the
  // same early return for every block that reads it
  const int done = state[0], stop = close ? state[2] : 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int it = state[1];
    if (close && !done) {
      state[1] = ++it;
      if (stop) state[0] = 1;
    }
    if (set_cond) cudaGraphSetConditional(cond, (!done && !stop && it < max_iter) ? 1u : 0u);
  }
  if (done || stop) return;
  int ti, tj;
  tile_pair(int(blockIdx.x), (n + kNsR - 1) / kNsR, ti, tj);
  const double g = ns_tile<false>(X, n, n, m, ti * kNsR, tj * kNsR, As, Bs);
  const int tid = threadIdx.x;
  if (tid >= kNsR * kNsR) return;
  const int i = ti * kNsR + tid / kNsR, j = tj * kNsR + tid % kNsR;
  if (i >= n || j >= n) return;
  G[int64_t(i) * n + j] = g;
  if (ti != tj) G[int64_t(j) * n + i] = g;
}

static unsigned ns_pairs(int64_t n) {
  const int64_t nt = (n + kNsR - 1) / kNsR;
  return unsigned(nt * (nt + 1) / 2);
}

cudaError_t launch_ns_square(const double* G, double* Bm, int64_t n, double* partials, double* resid, double tol,
                             int* state, cudaStream_t stream) {
  count_launch();
  launch(ns_square_kernel, ns_pairs(n) <= 304, ns_pairs(n), 256, 0, stream, G, Bm, int(n), partials, resid, tol, state);
  return cudaGetLastError();
}

cudaError_t launch_ns_gram(const double* X, double* G, int64_t m, int64_t n, int* state, bool close,
                           const cudaGraphConditionalHandle* cond, int max_iter, cudaStream_t stream) {
  count_launch();
  launch(ns_gram_kernel, ns_pairs(n) <= 304, ns_pairs(n), 256, 0, stream, X, G, int(m), int(n), state, close ? 1 : 0, cond ? 1 : 0,
                                                  cond ? *cond : cudaGraphConditionalHandle{}, max_iter);
  return cudaGetLastError();
}

// out = -X with X the iterate the Newton-Schulz state points at (buffer
// state[1] & 1), chosen on the device so that no host read is needed.  The
// sign flip is a bit operation (exact, off the FP64 pipe).
__global__ void __launch_bounds__(256) ns_output_kernel(const double* x0, const double* x1,
                                                        const int* state, double* out, int64_t count) {
  pdl_begin();
  const double* src = (state[1] & 1) ? x1 : x0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = __longlong_as_double(__double_as_longlong(src[i]) ^ (1ll << 63));
}

cudaError_t launch_ns_output(const double* x0, const double* x1, const int* state, double* out, int64_t count,
                             cudaStream_t stream) {
  const int nb = int(std::min<int64_t>((count + 255) / 256, 1024));
  if (nb <= 0) return cudaSuccess;
  count_launch();
  launch(ns_output_kernel, nb <= 304, nb, 256, 0, stream, x0, x1, state, out, count);
  return cudaGetLastError();
}

// Riemannian gradient step on the Stiefel manifold (embedded metric):
// with A = X^T G, S = (A + A^T) / 2 and T = X S, the step direction is
// G - T; the kernel writes Yneg = -(X - eta (G - T)) for the polar retraction
// (the polar update returns -polar(-Y) = polar(Y)).
__global__ void __launch_bounds__(256) stiefel_sym_kernel(const double* A, double* S, int64_t n) {
  pdl_begin();
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n * n; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / n, c = i - r * n;
    S[i] = 0.5 * (A[i] + A[c * n + r]);
  }
}

__global__ void __launch_bounds__(256) stiefel_combine_kernel(const double* X, const double* G,
                                                              const double* T, double* Yneg, int64_t count,
                                                              double eta) {
  pdl_begin();
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x)
    Yneg[i] = eta * (G[i] - T[i]) - X[i];
}

cudaError_t launch_stiefel_sym(const double* A, double* S, int64_t n, cudaStream_t stream) {
  const int nb = int(std::min<int64_t>((n * n + 255) / 256, 1024));
  count_launch();
  launch(stiefel_sym_kernel, nb <= 304, nb, 256, 0, stream, A, S, n);
  return cudaGetLastError();
}

cudaError_t launch_stiefel_combine(const double* X, const double* G, const double* T, double* Yneg, int64_t count,
                                   double eta, cudaStream_t stream) {
  const int nb = int(std::min<int64_t>((count + 255) / 256, 1024));
  count_launch();
  launch(stiefel_combine_kernel, nb <= 304, nb, 256, 0, stream, X, G, T, Yneg, count, eta);
  return cudaGetLastError();
}

// Last kernel of a recorded Newton-Schulz loop body: go on while not
// converged and fewer than max_iter steps have run.
__global__ void ns_continue_kernel(const int* state, cudaGraphConditionalHandle h, int max_iter) {
  pdl_begin();
  cudaGraphSetConditional(h, (state[0] == 0 && state[1] < max_iter) ? 1u : 0u);
}

cudaError_t launch_ns_continue(const int* state, cudaGraphConditionalHandle h, int max_iter, cudaStream_t stream) {
  count_launch();
  launch(ns_continue_kernel, true, 1, 1, 0, stream, state, h, max_iter);
  return cudaGetLastError();
}


// out = g * (a + b) elementwise (b may be null), g a device scalar: the
// energy adjoint's sum of the two environment halves times the upstream
// gradient.
__global__ void __launch_bounds__(256) scaled_sum_kernel(const double* a, const double* b,
                                                         const double* g, double* out,
                                                         int64_t n) {
  pdl_begin();
  const double gv = *g;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    out[i] = gv * (b ? a[i] + b[i] : a[i]);
}

cudaError_t launch_scaled_sum(const double* a, const double* b, const double* g, double* out, int64_t n,
                              cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const unsigned grid = unsigned(std::min<int64_t>((n + 255) / 256, 152 * 8));
  count_launch();
  launch(scaled_sum_kernel, grid <= 304, grid, 256, 0, stream, a, b, g, out, n);
  return cudaGetLastError();
}

}  // namespace mera
