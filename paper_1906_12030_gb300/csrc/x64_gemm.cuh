// Binary64 GEMM on the BF16 tensor cores (the large products of MERA_PREC_F64).
// Included by tc_gemm.cu inside its anonymous namespace: it shares that
// file's PTX wrappers (mbarrier, tcgen05) and its device status word.
//
// What bounds a binary64 product on this GPU is the FP64 pipe (two FMAs per
// clock and SM, 1.25 TFLOP/s); the BF16 tensor cores do 1500 times as many
// products.  So each operand entry is cut into eight signed 8-bit digits
// (x64_split.cu), and the product is the sum of the 36 digit products whose
// orders p + q are at most 7.  This is the error-free splitting of Ozaki,
// Ogita, Oishi and Rump (Numer. Algorithms 59, 2012), with one exponent per
// row and block of 256 along K.
//
// Exactness.  With 2^E the product of the two block scales, every product of
// order d is an integer multiple of 2^(E-12-8d) of magnitude at most 2^14
// units, so a block's sum of order d stays below (d+1) 2^22 units: at most
// 2^24, what an FP32 accumulator holds exactly, for d <= 3 whatever the data,
// and for d >= 4 unless nearly all products are extreme and of one sign
// (then off by a unit of 2^-44 or less, 2^-52 of such a result).  Each order
// therefore has an accumulator of its own.
//
// Accuracy.  What is left out of a term, the orders from 8 up, is at most
// 2^-59 of the product of the two rows' scales 2^E and 2^-62 of it at random
// (the bits below the eighth digit are less).  Against the sum's own size
// S = sum |a_k b_k| that is nothing where the rows hold entries of one scale,
// but not where an entry far above the others meets a zero or a small one.
// So S is summed too, from one more plane of magnitudes, and an output is
// taken from the digits only where S >= 2^-8 sqrt(K) 2^E (and >= 2^-6 2^E):
// its error is then below K 2^-53 S, the bound of a chain of binary64 FMAs,
// whatever the operands, and 2^-54 S or less at random, what such a chain has.
// S = 0 leaves an exact zero.  The others are left to the FP64 units.  With
// seven digits and 2^6 times the limit, a tenth to most of the outputs of
// ordinary maps were below it; with eight 0 to 0.2 % of a map's are (chi = 4
// to 9 of random isometries, chi = 6 after 3 and 60 sweeps).
//
// Tile 128 x 64: eight accumulators of 64 columns fill tensor memory.  (A
// wider tile has no room for eight; a narrower one needs more shared-memory
// reads of A per product than the tensor cores take time for.)  The digits of
// B lie next to each other in a stage and the accumulators next to each
// other in tensor memory, so one MMA of width 256 meets a digit of A with
// four digits of B and adds into four orders: 12 MMAs per 16 of K for the 36
// products.  Per 16 of K the MMAs take 1184 clocks, the shared-memory reads
// of their operands 1008 and the writes of the copies 432 (magnitudes
// included): shared-memory bandwidth sets the pace.
//
// A stage is 16 of K of all digits, stored by the split kernel as the very
// image that the MMA reads (8 x 16-byte core matrices, no swizzle), so a
// stage is two contiguous bulk copies and four stages fit in shared memory.
// The magnitudes come after the last block of a work item, 128 of K to a
// stage, into the first accumulator once the epilogue has taken the digits'
// sums out: before the first block, they would have had to wait for the
// stores of the item before.
//
// Warp roles as in tc_gemm_kernel: warp 0 copies, warp 1 MMA, warps 2..17
// epilogue, four per tensor-memory lane quarter with 16 columns each.  There
// is one set of accumulators, so the MMAs wait while the epilogue folds the
// eight sums of a block into a triple hi + mid + lo of binary32 values per
// output and hands them back; everything after that runs beside the next
// tile's MMAs.  The result is rounded once to binary64 by integer operations
// (an FP64 add per output and part would cost as much as the MMAs of a short
// K).
//
// Measured (chi = 16 descend, the pair of chi^9 products): 65536 x 4096 x 256
// 110 ms on the FP64 pipe, 3.11 ms here (44 TFLOP/s); 65536 x 256 x 4096 110 ->
// 3.03 ms (45 TFLOP/s, 0.89 of the burst BF16 rate / 37); with seven unchecked
// digits 3.0 and 2.66.  The whole map 497 -> 17.9 ms, its error against 64 bits
// 1.8e-15 -> 1.5e-15.
//
// Rows of A or B that the digits cannot represent (a NaN, an infinity, or a
// largest entry beyond 2^+-kX64MaxExp) carry the exponent kX64Bad.  Outputs
// that touch one, and those below the limit on S, are left to
// x64_exact_kernel, which sums them from the binary64 operands on the FP64
// units: each tile has a mask of them, 64 bits per row.  (Summed here, by the
// epilogue, a column of K = 331776 would keep the copy and MMA warps waiting
// past the limit of their waits.)

constexpr int kXBN = 64;
constexpr int kXDigits = kX64Digits;
constexpr int kXOrders = 8;
constexpr int kXAPlane = kBM * 32, kXBPlane = kXBN * 32;  // 16 of K, one plane
constexpr int kXABytes = kXDigits * kXAPlane;             // all digits
constexpr int kXBBytes = kXDigits * kXBPlane;
constexpr int kXATile = kXABytes + kXAPlane;              // and the magnitudes: bytes of a tile's image per 16 of K
constexpr int kXBTile = kXBBytes + kXBPlane;
constexpr int kXMagSteps = kXDigits;                      // 16-wide steps of magnitudes that fill a stage
constexpr int kXStageBytes = kXABytes + kXBBytes;
constexpr int kXStages = 4;
constexpr int kXEpiWarps = 16;
constexpr int kXEpiThreads = 32 * kXEpiWarps;
constexpr int kXThreads = 64 + kXEpiThreads;
constexpr int kXCols = kXBN / (kXEpiWarps / 4);  // columns per epilogue thread
constexpr int kXTmemCols = kXOrders * kXBN;
constexpr size_t kXSmem = 1024 + size_t(kXStages) * kXStageBytes + 1024 + kXBN * (sizeof(int64_t) + sizeof(int));
static_assert(kXTmemCols == 512, "all of tensor memory");

struct X64Params {
  const uint8_t* A;  // digit images
  const uint8_t* B;
  const int* ea;     // row exponents
  const int* eb;
  const double* A64;  // binary64 operands (rows with exponent kX64Bad)
  const double* B64;
  int64_t lda, ldb;
  int64_t M, N, K;
  double* C;
  LegMap m_dst, n_dst;
  double alpha;
  int alpha_exp;      // alpha == 2^alpha_exp
  int accumulate;
  int nk;             // 16-wide steps of K
  int split, kc;      // K split: steps per split
  float least;        // an output whose scaled magnitudes sum to less, but not to zero, is left to the FP64 units
  float* partial;     // split > 1: hi, mid, lo and magnitude planes [split][N][M]
  int64_t p_plane;
  unsigned long long* mask;  // outputs left to x64_exact_kernel: [tile][kBM], bit c for column c
  int tiles_m, tiles_n, group_m;  // work items (fewer than 2^31) and their order, as in Epilogue
};

struct X64Group {
  int n;
  int end[kGroup];  // work items of the jobs up to and including each
  X64Params job[kGroup];
};

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, the
// two of a 16-wide K step 128 bytes apart, groups of eight rows 256 bytes.
__device__ __forceinline__ uint64_t x64_desc(uint32_t saddr) {
  return uint64_t((saddr & 0x3FFFFu) >> 4) | (uint64_t(128 >> 4) << 16) | (uint64_t(256 >> 4) << 32) |
         (uint64_t(1) << 46);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}

// s + e = a + b exactly (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// The same where a is a multiple of ulp(b) (FastTwoSum under its relaxed
// condition).
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

// (h, m, l) += (x, y, z), each an unevaluated sum of decreasing magnitude.
__device__ __forceinline__ void triple_add(float& h, float& m, float& l, float x, float y, float z) {
  float c1, c2, c3;
  two_sum(h, x, h, c1);
  two_sum(m, y, m, c2);
  two_sum(m, c1, m, c3);
  l = __fadd_rn(l, __fadd_rn(z, __fadd_rn(c2, c3)));
}

// (h + m + l) 2^e rounded to binary64 with integer operations: h gives the
// bit pattern, m + l the number of its last places to add, found with two
// rounding constants (conversions run at a fraction of the FP32 rate).  The
// exponent stays normal (|e| <= 2 kX64MaxExp + 1).
__device__ __forceinline__ double triple_to_f64(float h, float m, float l, int e) {
  two_sum(h, m, h, m);
  two_sum(m, l, m, l);
  two_sum(h, m, h, m);
  const uint32_t u = __float_as_uint(h);
  const int eh = int((u >> 23) & 0xFFu);
  // below 2^-70 of the scale there is nothing under h that the digits resolve
  const float sc = eh < 127 - 70 ? 0.0f : __int_as_float((52 + 127 + 127 - eh) << 23);
  const float mp = __fmul_rn(m, sc);                      // |mp| <= 2^28
  const float t1 = __fadd_rn(mp, 0x1.8p29f);                  // its multiples of 64
  const float rem = __fsub_rn(mp, __fsub_rn(t1, 0x1.8p29f));  // exact, |rem| <= 32
  const float t2 = __fadd_rn(__fmaf_rn(l, sc, rem), 0x1.8p23f);
  int q = (__float_as_int(t1) - 0x4E400000) * 64 + (__float_as_int(t2) - 0x4B400000);
  if (int(u) < 0) q = -q;  // towards larger magnitude
  if (q < 0 && (u & 0x7FFFFFu) == 0) q *= 2;  // below a power of two the places are half as large
  // 24-bit significand of h over 29 more places
  const long long mag = (static_cast<long long>(eh + (1023 - 127) + e) << 52) +
                        (static_cast<long long>(u & 0x7FFFFFu) << 29) + q;
  const uint32_t hi = (uint32_t(static_cast<unsigned long long>(mag) >> 32) & 0x7FFFFFFFu) | (u & 0x80000000u);
  return eh == 0 ? 0.0 : __hiloint2double(int(hi), int(uint32_t(mag)));
}

// Mask word of row `row` of a tile.
__device__ __forceinline__ unsigned long long* x64_mask(const X64Params& p, int row_t, int col_t, int row) {
  return p.mask + (int64_t(row_t) * p.tiles_n + col_t) * kBM + row;
}

__device__ __forceinline__ void x64_store(const X64Params& p, int64_t off, double x) {
  double* d = p.C + off;
  *d = p.accumulate ? *d + x : x;
}

// MULTI: a work item may span several blocks of K.
template <bool MULTI>
__global__ void __launch_bounds__(kXThreads, 1) x64_gemm_kernel(const __grid_constant__ X64Group g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* aux = smem + size_t(kXStages) * kXStageBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(aux);
  uint64_t* empty = full + kXStages;
  uint64_t* acc_full = empty + kXStages;  // MMA -> epilogue, one phase per block
  uint64_t* acc_empty = acc_full + 1;     // epilogue -> MMA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* abort_snapshot = abort_flag + 1;
  volatile int* never = abort_flag + 2;
  int64_t* off_n = reinterpret_cast<int64_t*>(aux + 1024);
  int* exp_n = reinterpret_cast<int*>(off_n + kXBN);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kXStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, kXEpiWarps);
    *abort_flag = 0;
    *abort_snapshot = 0;
    *never = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(uint32_t(kXTmemCols))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();
  const int items = g.end[g.n - 1];

  if (warp == 0) {
    if (lane == 0) {
      // ---- producer: all digits of 16 of K per stage ----------------------
      uint32_t it = 0;
      bool alive = true;
      for (int tg = int(blockIdx.x); tg < items && alive; tg += gridDim.x) {
        int t;
        const X64Params& p = g.job[item_of(g.end, tg, t)];
        const int k0 = split_of(t, p.tiles_m * p.tiles_n, p.split) * p.kc, k1 = min(k0 + p.kc, p.nk);
        int row_t, col_t;
        tile_of(t, p.tiles_m, p.tiles_n, p.group_m, row_t, col_t);
        const uint8_t* a = p.A + int64_t(row_t) * p.nk * kXATile;
        const uint8_t* b = p.B + int64_t(col_t) * p.nk * kXBTile;
        auto stage = [&](const uint8_t* sa, uint32_t na, const uint8_t* sb, uint32_t nb) {
          const uint32_t s = it % kXStages;
          if (it >= uint32_t(kXStages) && !mbar_wait(&empty[s], ((it / kXStages) & 1) ^ 1, abort_flag)) {
            alive = false;
            return;
          }
          uint8_t* st = smem + size_t(s) * kXStageBytes;
          mbar_arrive_expect_tx(&full[s], na + nb);
          bulk_load(st, sa, na, &full[s]);
          bulk_load(st + kXABytes, sb, nb, &full[s]);
          ++it;
        };
        for (int k = k0; k < k1 && alive; ++k)
          stage(a + k * int64_t(kXABytes), kXABytes, b + k * int64_t(kXBBytes), kXBBytes);
        a += int64_t(p.nk) * kXABytes;  // the magnitudes
        b += int64_t(p.nk) * kXBBytes;
        for (int k = k0; k < k1 && alive; k += kXMagSteps) {
          const uint32_t c = uint32_t(min(kXMagSteps, k1 - k));
          stage(a + k * int64_t(kXAPlane), c * kXAPlane, b + k * int64_t(kXBPlane), c * kXBPlane);
        }
      }
      for (uint32_t j = (it > uint32_t(kXStages) ? it - kXStages : 0); j < it; ++j)
        mbar_wait(&full[j % kXStages], (j / kXStages) & 1, never);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---- MMA issuer ---------------------------------------------------------
      uint32_t it = 0, bc = 0;  // stages consumed, blocks issued
      bool alive = true;
      for (int tg = int(blockIdx.x); tg < items && alive; tg += gridDim.x) {
        int t;
        const X64Params& p = g.job[item_of(g.end, tg, t)];
        const int k0 = split_of(t, p.tiles_m * p.tiles_n, p.split) * p.kc, k1 = min(k0 + p.kc, p.nk);
        for (int k = k0; k < k1 && alive; ++bc) {
          const int ke = min(k1, (k / kX64BlockSteps + 1) * kX64BlockSteps);
          if (bc >= 1 && !mbar_wait(acc_empty, (bc - 1) & 1, abort_flag)) {
            alive = false;
            break;
          }
          tc_fence_after();
          bool first = true;
          for (; k < ke; ++k, ++it, first = false) {
            const uint32_t s = it % kXStages;
            if (!mbar_wait(&full[s], (it / kXStages) & 1, abort_flag)) {
              alive = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + size_t(s) * kXStageBytes), sb = sa + kXABytes;
#pragma unroll
            for (int pa = 0; pa < kXDigits; ++pa) {
              const uint64_t da = x64_desc(sa + pa * kXAPlane);
              const int nq = min(kXDigits, kXOrders - pa);  // digits of B that this digit of A meets
#pragma unroll
              for (int q = 0; q < nq; q += 4) {
                const int cnt = min(4, nq - q);
                const uint64_t db = x64_desc(sb + q * kXBPlane);
                const uint32_t d = tmem + uint32_t((pa + q) * kXBN);
                tc_mma<PREC_BF16>(d, da, db, make_idesc(1u, kBM, cnt * kXBN), (pa == 0 && first) ? 0u : 1u);
              }
            }
            tc_commit(&empty[s]);
          }
          tc_commit(acc_full);  // also after an abort, so that no epilogue warp waits forever
        }
        if (!alive) break;
        // the magnitudes, as one more block
        if (!mbar_wait(acc_empty, (bc - 1) & 1, abort_flag)) break;
        tc_fence_after();
        for (int k = k0; k < k1; k += kXMagSteps, ++it) {
          const uint32_t s = it % kXStages;
          if (!mbar_wait(&full[s], (it / kXStages) & 1, abort_flag)) {
            alive = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + size_t(s) * kXStageBytes), sb = sa + kXABytes;
          for (int j = 0; j < min(kXMagSteps, k1 - k); ++j)
            tc_mma<PREC_BF16>(tmem, x64_desc(sa + j * kXAPlane), x64_desc(sb + j * kXBPlane),
                              make_idesc(1u, kBM, kXBN), k > k0 || j > 0 ? 1u : 0u);
          tc_commit(&empty[s]);
        }
        tc_commit(acc_full);
        ++bc;
      }
    }
  } else {
    // ---- epilogue (warps 2..17) --------------------------------------------------
    const int et = threadIdx.x - 64;
    const int quarter = warp % 4;
    const int c0 = ((warp - 2) / 4) * kXCols;  // first column of this warp's share
    const int row = quarter * 32 + lane;
    uint32_t bc = 0;
    for (int tg = int(blockIdx.x); tg < items; tg += gridDim.x) {
      int t;
      const X64Params& p = g.job[item_of(g.end, tg, t)];
      const int64_t ks = split_of(t, p.tiles_m * p.tiles_n, p.split);
      int row_t, col_t;
      tile_of(t, p.tiles_m, p.tiles_n, p.group_m, row_t, col_t);
      const int64_t m0 = int64_t(row_t) * kBM, n0 = int64_t(col_t) * kXBN;
      const int k0 = int(ks) * p.kc, k1 = min(k0 + p.kc, p.nk);
      asm volatile("bar.sync 1, %0;" ::"n"(kXEpiThreads) : "memory");
      if (et == 0) *abort_snapshot = *abort_flag;
      for (int c = et; c < kXBN; c += kXEpiThreads) {
        const int64_t n = n0 + c;
        off_n[c] = n < p.N ? legmap_offset32(p.n_dst, uint32_t(n)) : 0;
        exp_n[c] = n < p.N ? p.eb[n] : 0;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kXEpiThreads) : "memory");
      if (*abort_snapshot) break;
      const int64_t m = m0 + row;
      const bool row_ok = m < p.M;
      float h[kXCols], mid[kXCols], lo[kXCols];
      if constexpr (MULTI) {
#pragma unroll
        for (int j = 0; j < kXCols; ++j) h[j] = mid[j] = lo[j] = 0.0f;
      }
      bool ok = true;
      for (int k = k0; k < k1; k = min(k1, (k / kX64BlockSteps + 1) * kX64BlockSteps), ++bc) {
        ok = __all_sync(0xffffffffu, mbar_wait(acc_full, bc & 1, abort_flag) ? 1 : 0) != 0;
        tc_fence_after();
        if (!ok) break;  // the next tile's snapshot sees the abort flag
        const uint32_t ta = tmem + uint32_t(c0) + (uint32_t(quarter * 32) << 16);
#pragma unroll
        for (int g = 0; g < kXCols; g += 4) {
          uint32_t v[kXOrders][4];
#pragma unroll
          for (int d = 0; d < kXOrders; ++d) tmem_ld4(ta + uint32_t(d * kXBN + g), v[d]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // VecSum from the smallest order up.  v[d] is a multiple of its
            // order's unit, at least 2^6 ulps of the sum of what is below.
            float s = __uint_as_float(v[7][j]), c, r = 0.0f;
#pragma unroll
            for (int d = 6; d >= 1; --d) {
              fast_two_sum(__uint_as_float(v[d][j]), s, s, c);
              r = __fadd_rn(r, c);
            }
            fast_two_sum(__uint_as_float(v[0][j]), s, s, c);
            if constexpr (MULTI) {
              triple_add(h[g + j], mid[g + j], lo[g + j], s, c, r);
            } else {
              h[g + j] = s;
              mid[g + j] = c;
              lo[g + j] = r;
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
        if constexpr (!MULTI) {
          ++bc;
          break;
        }
      }
      // sums of the magnitudes
      uint32_t sum[kXCols];
      ok = ok && __all_sync(0xffffffffu, mbar_wait(acc_full, bc & 1, abort_flag) ? 1 : 0) != 0;
      if (!ok) continue;  // the next tile's snapshot sees the abort flag
      tc_fence_after();
      tmem_ld16(tmem + uint32_t(c0) + (uint32_t(quarter * 32) << 16), sum);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
      ++bc;
      uint16_t* const mask = reinterpret_cast<uint16_t*>(x64_mask(p, row_t, col_t, row)) + c0 / kXCols;
      if (p.split > 1) {  // partial triple, summed by x64_reduce_kernel
        if (ks == 0) *mask = 0;
        if (!row_ok) continue;
        float* q = p.partial + (ks * p.N + n0 + c0) * p.M + m;
#pragma unroll
        for (int j = 0; j < kXCols; ++j, q += p.M)
          if (n0 + c0 + j < p.N) {
            q[0] = h[j];
            q[p.p_plane] = mid[j];
            q[2 * p.p_plane] = lo[j];
            q[3 * p.p_plane] = __uint_as_float(sum[j]);
          }
        continue;
      }
      const int ra = row_ok ? p.ea[m] : 0;
      uint32_t todo = 0, skip = 0;  // columns that exist, and those left to x64_exact_kernel
#pragma unroll
      for (int j = 0; j < kXCols; ++j) {
        if (row_ok && n0 + c0 + j < p.N) todo |= 1u << j;
        const float s = __uint_as_float(sum[j]);
        if (ra == kX64Bad || exp_n[c0 + j] == kX64Bad || (s < p.least && s > 0.0f)) skip |= 1u << j;
      }
      skip &= todo;
      todo &= ~skip;
      *mask = uint16_t(skip);
      if (todo == 0) continue;
      const int64_t off_m = legmap_offset32(p.m_dst, uint32_t(m));
      if (!p.accumulate) {
#pragma unroll
        for (int j = 0; j < kXCols; ++j) {
          const int c = c0 + j;
          const int rb = exp_n[c];
          if (!(todo >> j & 1u)) continue;
          p.C[off_m + off_n[c]] = triple_to_f64(h[j], mid[j], lo[j], ra + rb + p.alpha_exp);
        }
      } else {
        // bound by the latency of the reads: four go out together
#pragma unroll
        for (int j = 0; j < kXCols; j += 4) {
          double y[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) y[k] = (todo >> (j + k) & 1u) ? p.C[off_m + off_n[c0 + j + k]] : 0.0;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int c = c0 + j + k;
            const int rb = exp_n[c];
            if (!(todo >> (j + k) & 1u)) continue;
            p.C[off_m + off_n[c]] = y[k] + triple_to_f64(h[j + k], mid[j + k], lo[j + k], ra + rb + p.alpha_exp);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(uint32_t(kXTmemCols))
                 : "memory");
  }
}

// Sum of the K-split partial triples and magnitudes in a fixed order, then the
// GEMM's output.  One thread per row m over a chunk of columns.
__global__ void __launch_bounds__(128) x64_reduce_kernel(const __grid_constant__ X64Group g) {
  pdl_begin();
  const X64Params& p = g.job[blockIdx.z];
  const int64_t m = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (m >= p.M) return;
  const int64_t off_m = legmap_offset32(p.m_dst, uint32_t(m));
  const int ra = p.ea[m];
  const int64_t n_per = (p.N + gridDim.y - 1) / gridDim.y;
  const int64_t n_lo = int64_t(blockIdx.y) * n_per, n_hi = min(p.N, n_lo + n_per);
  for (int64_t n = n_lo; n < n_hi; ++n) {
    float h = 0.0f, mid = 0.0f, lo = 0.0f, sum = 0.0f;
    for (int s = 0; s < p.split; ++s) {
      const float* q = p.partial + (int64_t(s) * p.N + n) * p.M + m;
      triple_add(h, mid, lo, q[0], q[p.p_plane], q[2 * p.p_plane]);
      sum += q[3 * p.p_plane];
    }
    const int rb = p.eb[n];
    if (ra == kX64Bad || rb == kX64Bad || (sum < p.least && sum > 0.0f)) {  // (the mask was cleared by the GEMM)
      atomicOr(x64_mask(p, int(m / kBM), int(n / kXBN), int(m % kBM)), 1ull << (n % kXBN));
      continue;
    }
    x64_store(p, off_m + legmap_offset32(p.n_dst, uint32_t(n)), triple_to_f64(h, mid, lo, ra + rb + p.alpha_exp));
  }
}

// The outputs that the tiles' masks name, from the binary64 operands.  Bound:
// the FP64 pipe where many are named; where none is, the reading of the masks
// (a bit per output); in between latency: a map of ordinary operands names a
// few outputs of every thousand.  So each block looks through its units (eight
// rows of a tile; they go round the blocks, so that even a single tile meets
// sixteen SMs) and gathers what they name.  From units that name little, a
// warp takes an output at a time, 128 terms in flight.  A unit that names much
// is summed by the whole block through shared memory, one chain of FMAs in the
// order of K per output, as the FP64 kernels sum it, bit for bit; so is any
// output of a row that the digits cannot represent.  `end` counts units.
// (Everything through shared memory: chi = 8 sweep 10.8 ms.)
constexpr int kExRows = 8, kExUnits = kBM / kExRows;  // rows per unit, units per tile
__global__ void __launch_bounds__(256) x64_exact_kernel(const __grid_constant__ X64Group g) {
  pdl_begin();
  constexpr int KC = 32, P = KC + 1;        // of K at a time, and the pitch of its rows
  constexpr int kFew = 16;                  // outputs of a unit that warps take one by one
  __shared__ double As[kExRows * P], Bs[kXBN * P];
  __shared__ int many[256], n_many, n_few, n_out;
  __shared__ int few[256 * kFew];           // thread that looked at the unit, output in it
  __shared__ uint16_t outs[kExRows * kXBN];
  static_assert(kExRows * kXBN == 1 << 9, "outputs of a unit");
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t units = g.end[g.n - 1];
  // job of a unit, and where its tile lies
  auto place = [&](int unit, int& local, int64_t& m0, int64_t& n0) -> const X64Params& {
    const X64Params& p = g.job[item_of(g.end, unit, local)];
    const int tile = local / kExUnits;
    m0 = int64_t(tile / p.tiles_n) * kBM + local % kExUnits * kExRows;
    n0 = int64_t(tile % p.tiles_n) * kXBN;
    return p;
  };
  auto store = [](const X64Params& p, int64_t m, int64_t n, double v) {
    x64_store(p, legmap_offset32(p.m_dst, uint32_t(m)) + legmap_offset32(p.n_dst, uint32_t(n)), p.alpha * v);
  };
  for (int64_t base = 0; base < units; base += 256 * int64_t(gridDim.x)) {
    if (tid == 0) n_many = n_few = 0;
    __syncthreads();
    const int64_t u = base + int64_t(tid) * gridDim.x + blockIdx.x;
    if (u < units) {
      int local;
      int64_t m0, n0;
      const X64Params& p = place(int(u), local, m0, n0);
      const ulonglong2* w = reinterpret_cast<const ulonglong2*>(p.mask + int64_t(local) * kExRows);
      unsigned long long bits[kExRows];
      int count = 0;
#pragma unroll
      for (int q = 0; q < kExRows; q += 2) {
        const ulonglong2 v = w[q / 2];
        bits[q] = v.x;
        bits[q + 1] = v.y;
        count += __popcll(v.x) + __popcll(v.y);
      }
      if (count > 0) {
        bool chain = count > kFew;
        if (!chain) {
#pragma unroll
          for (int q = 0; q < kExRows; ++q)
            for (unsigned long long b = bits[q]; b; b &= b - 1) {
              const int64_t n = n0 + __ffsll(static_cast<long long>(b)) - 1;
              if (m0 + q < p.M && n < p.N && (p.ea[m0 + q] == kX64Bad || p.eb[n] == kX64Bad)) chain = true;
            }
        }
        if (chain) {
          many[atomicAdd(&n_many, 1)] = int(u);
        } else {
          int i = atomicAdd(&n_few, count);
#pragma unroll
          for (int q = 0; q < kExRows; ++q)
            for (unsigned long long b = bits[q]; b; b &= b - 1)
              few[i++] = tid << 9 | (q * kXBN + __ffsll(static_cast<long long>(b)) - 1);
        }
      }
    }
    __syncthreads();
    for (int i = tid / 32; i < n_few; i += 8) {
      int local;
      int64_t m, n;
      const X64Params& p = place(int(base + int64_t(few[i] >> 9) * gridDim.x + blockIdx.x), local, m, n);
      m += few[i] % (kExRows * kXBN) / kXBN;
      n += few[i] % kXBN;
      if (m >= p.M || n >= p.N) continue;
      const double* a = p.A64 + m * p.lda;
      const double* b = p.B64 + n * p.ldb;
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      int64_t k = lane;
      for (; k + 96 < p.K; k += 128) {
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = fma(a[k + 32 * q], b[k + 32 * q], s[q]);
      }
      for (; k < p.K; k += 32) s[0] = fma(a[k], b[k], s[0]);
      double v = (s[0] + s[1]) + (s[2] + s[3]);
      __syncwarp();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) store(p, m, n, v);
    }
    for (int i = 0; i < n_many; ++i) {
      int local;
      int64_t m0, n0;
      const X64Params& p = place(many[i], local, m0, n0);
      if (tid == 0) n_out = 0;
      __syncthreads();
      for (int e = tid; e < kExRows * kXBN; e += 256)
        if ((p.mask[int64_t(local) * kExRows + e / kXBN] >> (e % kXBN) & 1) && m0 + e / kXBN < p.M &&
            n0 + e % kXBN < p.N)
          outs[atomicAdd(&n_out, 1)] = uint16_t(e);
      __syncthreads();
      const int total = n_out;
      const int e0 = tid < total ? outs[tid] : 0, e1 = tid + 256 < total ? outs[tid + 256] : 0;
      const double* const a0 = As + e0 / kXBN * P;
      const double* const b0 = Bs + e0 % kXBN * P;
      const double* const a1 = As + e1 / kXBN * P;
      const double* const b1 = Bs + e1 % kXBN * P;
      double s0 = 0.0, s1 = 0.0;
      const int kk = tid % KC, rr = tid / KC;  // this thread's column and first row of the loads
      for (int64_t k0 = 0; k0 < p.K; k0 += KC) {
        const bool in = k0 + kk < p.K;
        As[rr * P + kk] = in && m0 + rr < p.M ? p.A64[(m0 + rr) * p.lda + k0 + kk] : 0.0;
#pragma unroll
        for (int q = 0; q < kXBN; q += 256 / KC)
          Bs[(rr + q) * P + kk] = in && n0 + rr + q < p.N ? p.B64[(n0 + rr + q) * p.ldb + k0 + kk] : 0.0;
        __syncthreads();
        const int terms = int(min(int64_t(KC), p.K - k0));
        if (tid < total) {
#pragma unroll 8
          for (int k = 0; k < terms; ++k) s0 = fma(a0[k], b0[k], s0);
        }
        if (tid + 256 < total) {
#pragma unroll 8
          for (int k = 0; k < terms; ++k) s1 = fma(a1[k], b1[k], s1);
        }
        __syncthreads();
      }
      if (tid < total) store(p, m0 + e0 / kXBN, n0 + e0 % kXBN, s0);
      if (tid + 256 < total) store(p, m0 + e1 / kXBN, n0 + e1 % kXBN, s1);
    }
    __syncthreads();
  }
}
