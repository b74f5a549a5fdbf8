// Binary64 products on the tensor cores, by exact slices of the operands (Sec. 5.5's Down path).
// Part of gemm_tc.cu (included there, inside its namespace, after the PTX wrappers).
//
// What bounds the FP64 pipe: it does 2 multiply-adds a cycle and SM (1.25 TFLOP/s), and a conversion from
// fp32 costs as much as one, so 128 rows of 8192 by 3072 take at least 5.2 ms there (7.4 ms measured).  The
// fp16 tensor rate is 1500 times that, and the product is exact on it if the operands are cut into digits
// that it multiplies and adds without rounding (the scheme of Ozaki, Ogita, Oishi, Rump, Numer. Algorithms
// 59 (2012)):
//   * every row of X~ and of W is taken in fixed point below its largest exponent E, v = x 2^(53 - E) rounded to
//     an integer below 2^54, and v as 7 digits of 8 bits, v = sum_p d_p 2^(8 p), |d_p| <= 128, each exact in
//     fp16;
//   * the products of digits p of W and s of X~ with p + s >= 5 (34 of the 49; the rest is below 2^-57 of
//     the largest terms) go into 8 accumulators, one per p + s.  A sum over 128 of K is at most
//     7 x 128 x 2^14 < 2^24 in magnitude, so every fp32 accumulator holds an exact integer;
//   * after 128 of K the accumulators are added into one 96-bit integer per output, exactly.
// So the only errors are the roundings to fixed point (2^-54 of the row's largest entry each), the dropped
// products and the conversion of the result.  Against gamma_K S (S the sum of the terms' magnitudes) that
// is small unless S is far below the rows' largest entries, which f64_finish_kernel checks for every output
// (by samples of K, then by more of it): an output that fails, or whose rows hold an infinity or NaN, is summed again
// in binary64, by the same kernel.
//
// Kernel: one CTA per 128 rows of W (the MMA's rows) x TN tokens (its columns) over a K range.  16 worker
// warps load the fp32 / binary64 tiles (cp.async, a stage ahead, each thread its own groups of 4 entries),
// cut them into digits in registers and store these into the stage (64-byte rows, 64-byte swizzle); warp 0
// issues the MMAs, a digit of W against several of X~ at once; every 4 stages of 32 of K the workers read
// the 8 accumulators and add them up while they fill the ring again.
// What bounds it now (128 rows, 8192 by 3072: 195 us of the call's 238): shared memory, which a stage of 32 of K
// asks for about 380 KB (3000 cycles), then the conversions of the accumulators (58 us), which nothing overlaps.
// 8 worker warps and integer digits for W took 265 us; a digit against one other digit per MMA as much as now.

constexpr int F64_WORKERS = 16, F64_WT = 32 * F64_WORKERS, F64_THREADS = 32 * (F64_WORKERS + 1), F64_CHUNK = 128;
constexpr int kDigits = 7, kDiags = 8, kMinDiag = 5;

template <int TN, class TX>
struct F64Cfg {
  static_assert(TN == 16 || TN == 32 || TN == 64, "8 accumulators of TN columns in 512");
  static constexpr uint32_t W_SLICE = BM * 64, X_SLICE = TN * 64;
  static constexpr uint32_t X_OFF = kDigits * W_SLICE, STAGE = X_OFF + kDigits * X_SLICE;
  static constexpr int STAGES = 2;
  // raw tiles of one stage: 16-byte units, unit u of worker thread t at (u * F64_WT + t); a thread holds groups
  // of 4 entries, 8 threads to a row
  static constexpr int ROWS_AT_ONCE = F64_WT / 8;
  static constexpr int W_GROUPS = BM / ROWS_AT_ONCE, X_UNITS = (int)sizeof(TX) / 4;
  static constexpr int RAW_UNITS = W_GROUPS + X_UNITS;
  static_assert(BM % ROWS_AT_ONCE == 0 && TN <= ROWS_AT_ONCE, "one group of X~ a thread at most");
  static constexpr uint32_t RAW_OFF = STAGES * STAGE, AUX_OFF = RAW_OFF + RAW_UNITS * F64_WT * 16;
  static constexpr uint32_t EXP_OFF = AUX_OFF + 256;  // row exponents: 128 of W, TN of X~
  static constexpr uint32_t SMEM = EXP_OFF + (BM + TN) * 4 + 1024;
  static constexpr uint32_t TMEM_COLS = kDiags * TN;
  static_assert(STAGE % 1024 == 0 && X_SLICE % 1024 == 0 && SMEM <= 232448, "shared memory of the CTA");
};

// The digits of 4 consecutive entries into their places in the 7 slices (8 bytes each).
// fp32 entries, on the FP32 pipe, two at a time: with y = x 2^-E below 2, t_7 = 2^-3 y and from the top digit
// down r = 256 t + M rounds to the digit (M = 1.5 2^23), d = r - M, t' = 256 t - d: every step but the
// rounding to d is exact (t' is a multiple of t's last place), so the last remainder, at most half of the
// last digit's unit, is all that is lost.
__device__ __forceinline__ uint32_t half_pair(unsigned long long v) {
  float a, b;
  up2(v, a, b);
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void store_digits(uint8_t* dst, uint32_t slice, const float4& x, int emax) {
  // 2^-E: E = emax - 127, so the field is 254 - emax; 2^-127 (a denormal) for E = 127
  const float down = emax < 254 ? __int_as_float((254 - emax) << 23) : __int_as_float(0x400000);
  // p2 of equal halves; y 2^-3 so that the first digit comes out of the same step: 256 y 2^-3 = 32 y, below 64
  unsigned long long t0 = p2((x.x * down) * 0.125f, (x.y * down) * 0.125f);
  unsigned long long t1 = p2((x.z * down) * 0.125f, (x.w * down) * 0.125f);
  const unsigned long long k256 = p2(256.f, 256.f), magic = p2(12582912.f, 12582912.f),
                           unmagic = p2(-12582912.f, -12582912.f), minus = p2(-1.f, -1.f);
#pragma unroll
  for (int p = kDigits - 1; p >= 0; --p) {
    const unsigned long long d0 = add2(fma2(t0, k256, magic), unmagic), d1 = add2(fma2(t1, k256, magic), unmagic);
    *reinterpret_cast<uint2*>(dst + p * slice) = make_uint2(half_pair(d0), half_pair(d1));
    t0 = fma2(t0, k256, fma2(d0, minus, p2(-0.f, -0.f)));
    t1 = fma2(t1, k256, fma2(d1, minus, p2(-0.f, -0.f)));
  }
}
// Binary64 entries, in integers: v = rint(x 2^(53 - E)) from the bits, its bytes plus 0x80..80 being the digits
// plus 128.
__device__ __forceinline__ unsigned long long fixed_digits(double x, int emax) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(u >> 52) & 2047;
  const unsigned long long m = (u & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
  const unsigned long long t = (((m << 2) >> min(emax - max(e, 1), 63)) + 1ull) >> 1;  // below 2^54, to nearest
  return ((long long)u < 0 ? 0ull - t : t) + 0x0080808080808080ull;
}
// Byte p of a, b as the fp16 pair (digit, digit): 0x6400 + byte is 1024 + byte in fp16.
template <int P>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long a, unsigned long long b) {
  const uint32_t wa = P < 4 ? (uint32_t)a : (uint32_t)(a >> 32), wb = P < 4 ? (uint32_t)b : (uint32_t)(b >> 32);
  constexpr uint32_t sel = (uint32_t)(P & 3) | ((uint32_t)(4 + (P & 3)) << 4);
  const uint32_t bytes = __byte_perm(__byte_perm(wa, wb, sel), 0x64u, 0x4140);  // [byte a, 0x64, byte b, 0x64]
  const __half2 h = *reinterpret_cast<const __half2*>(&bytes);
  const __half2 r = __hsub2(h, __half2half2(__ushort_as_half((unsigned short)0x6480)));  // - 1152, exact
  return *reinterpret_cast<const uint32_t*>(&r);
}
template <int P>
__device__ __forceinline__ void store_bytes(uint8_t* dst, uint32_t slice, const unsigned long long (&v)[4]) {
  if constexpr (P < kDigits) {
    *reinterpret_cast<uint2*>(dst + P * slice) = make_uint2(digit_pair<P>(v[0], v[1]), digit_pair<P>(v[2], v[3]));
    store_bytes<P + 1>(dst, slice, v);
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool in) {
  const int bytes = in ? 16 : 0;  // 0: the 16 bytes are zero-filled and src is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// 32 lanes x 4 columns, no wait (tmem_wait_ld before the values are used).
__device__ __forceinline__ void tmem_ld_32x4_nowait(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
// Waits for the loads above; the registers pass through, so no use of them can move before the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&a)[4], uint32_t (&b)[4], uint32_t (&c)[4], uint32_t (&d)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]),
                 "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])::"memory");
}

// What the slices need of a row: its largest biased exponent field (at least 1; kRowNonFinite with an
// infinity or NaN; 0 for a row of zeros) and the mean magnitude in units of 2^E.
template <class TX>
struct F64Pair;
template <>
struct F64Pair<float> {
  using type = float2;
};
template <>
struct F64Pair<double> {
  using type = double2;
};
struct F64Row {
  int e;
  float mean;
};
constexpr int kRowNonFinite = -1;

// One block per row: rows 0..N-1 of W, then the M rows of X~.
template <class TX>
__global__ void __launch_bounds__(256) f64_rows_kernel(F64Row* __restrict__ rows, const float* __restrict__ W,
                                                       const TX* __restrict__ X, int64_t K, int64_t N) {
  pdl_wait();
  pdl_trigger();
  __shared__ uint32_t s_max[8];
  __shared__ float s_sum[8];
  const int64_t r = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool w_row = r < N;
  uint32_t top = 0u;  // largest magnitude, as the ordered high word
  float sum = 0.f;
  if (w_row) {
    const float4* p = reinterpret_cast<const float4*>(W + r * K);
    for (int64_t i = threadIdx.x; i < (K >> 2); i += 256) {
      const float4 v = __ldg(p + i);
      top = max(max(top, max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu)),
                max(__float_as_uint(v.z) & 0x7FFFFFFFu, __float_as_uint(v.w) & 0x7FFFFFFFu));
      sum += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
    }
  } else if constexpr (sizeof(TX) == 4) {
    const float4* p = reinterpret_cast<const float4*>(X + (r - N) * K);
    for (int64_t i = threadIdx.x; i < (K >> 2); i += 256) {
      const float4 v = __ldg(p + i);
      top = max(max(top, max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu)),
                max(__float_as_uint(v.z) & 0x7FFFFFFFu, __float_as_uint(v.w) & 0x7FFFFFFFu));
      sum += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
    }
  } else {
    const uint4* p = reinterpret_cast<const uint4*>(X + (r - N) * K);
    for (int64_t i = threadIdx.x; i < (K >> 1); i += 256) {
      const uint4 v = __ldg(p + i);
      // a denormal's or zero's high word may be 0 while its low word is not: at least 1 then
      top = max(top, max((v.y & 0x7FFFFFFFu) | (v.x ? 1u : 0u), (v.w & 0x7FFFFFFFu) | (v.z ? 1u : 0u)));
    }
  }
  const bool wide = !w_row && sizeof(TX) == 8;
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (lane == 0) s_max[warp] = top;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) top = max(top, s_max[w]);
  const int bits = wide ? 20 : 23, last = wide ? 2047 : 255, bias = wide ? 1023 : 127;
  int e = (int)(top >> bits);
  const bool finite = e < last;
  if (e == 0 && top != 0u) e = 1;
  if (wide && finite) {  // magnitudes relative to 2^E, from the bits (E known now)
    const uint4* p = reinterpret_cast<const uint4*>(X + (r - N) * K);
    for (int64_t i = threadIdx.x; i < (K >> 1); i += 256) {
      const uint4 v = __ldg(p + i);
      const uint32_t hw[2] = {v.y & 0x7FFFFFFFu, v.w & 0x7FFFFFFFu};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int ex = (int)(hw[h] >> 20) - e + 127;
        if (ex > 0) sum += __uint_as_float(((uint32_t)ex << 23) | ((hw[h] & 0xFFFFFu) << 3));
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < 8; ++w) t += s_sum[w];
    if (!wide) t = ldexpf(t, bias - max(e, 1));
    rows[r] = F64Row{finite ? e : kRowNonFinite, t / (float)K};
  }
}

// Partial sums of the K range of split blockIdx.y as 96-bit integers: hi (bits 32..95) and lo, [split][m][n].
template <int TN, class TX>
__global__ void __launch_bounds__(F64_THREADS, 1)
tc_f64_kernel(long long* __restrict__ hi, uint32_t* __restrict__ lo, const F64Row* __restrict__ rows,
              const float* __restrict__ W, const TX* __restrict__ X, int64_t M, int64_t K, int64_t N,
              int64_t k_per_split) {
  using L = F64Cfg<TN, TX>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* aux = smem + L::AUX_OFF;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(aux + 64);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(aux + 72);
  int* s_exp = reinterpret_cast<int*>(smem + L::EXP_OFF);
  const uint32_t bar_base = smem_u32(aux);
  auto full_bar = [&](int st) { return bar_base + 8u * st; };         // a stage's digits are stored
  auto empty_bar = [&](int st) { return bar_base + 8u * (2 + st); };  // its MMAs are done
  const uint32_t acc_full = bar_base + 32u, acc_free = bar_base + 40u, drain_bar = bar_base + 48u;

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int64_t n0 = (int64_t)blockIdx.x * BM, m0 = (int64_t)blockIdx.z * TN;
  const int64_t kbeg = (int64_t)blockIdx.y * k_per_split, kend = std::min<int64_t>(K, kbeg + k_per_split);
  const int n_stages = kend > kbeg ? (int)ceil_div(kend - kbeg, 32) : 0;
  constexpr int SPC = F64_CHUNK / 32;  // stages per chunk
  const int n_chunks = (n_stages + SPC - 1) / SPC;

  if (threadIdx.x == 0) {
    for (int st = 0; st < 2; ++st) {
      mbar_init(full_bar(st), F64_WORKERS);
      mbar_init(empty_bar(st), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_free, F64_WORKERS);
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), L::TMEM_COLS);
  pdl_wait();  // the rows' exponents come from the kernel before this one
  for (int i = threadIdx.x; i < BM + TN; i += F64_THREADS) {
    const int64_t r = i < BM ? n0 + i : m0 + (i - BM);
    const bool in = i < BM ? r < N : r < M;
    s_exp[i] = in ? max(rows[i < BM ? r : N + r].e, 1) : 1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == 0) {
    // ---------------- MMA issuer ----------------
    bool ok = true;
    const uint32_t leader = elect_one();
    const uint32_t sd0 = sdesc_lo(smem_u32(smem));
    for (int t = 0; t < n_stages && ok; ++t) {
      const int st = t & 1, c = t / SPC;
      if (t % SPC == 0 && c > 0) {  // the workers have read the chunk before
        ok = __all_sync(0xffffffffu, mbar_wait(acc_free, (uint32_t)(c - 1) & 1u, kWaitNs, abort_flag));
        if (!ok) break;
      }
      ok = __all_sync(0xffffffffu, mbar_wait(full_bar(st), (uint32_t)(t >> 1) & 1u, kWaitNs, abort_flag));
      if (!ok) break;
      tc_fence_after();
      const uint32_t sd = sd0 + (uint32_t)st * (L::STAGE >> 4);
      const uint32_t later = t % SPC == 0 ? 0u : 1u;  // 0: the chunk's first products overwrite
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
        for (int p = kDigits - 1; p >= 0; --p) {
          // W's digit p against the digits s0..6 of X~: consecutive slices of X~ are consecutive rows in shared
          // memory and their accumulators p + s consecutive columns, so one MMA takes up to 256 / TN of them
          constexpr int kAtOnce = 256 / TN;
          const int s0 = kMinDiag - p > 0 ? kMinDiag - p : 0;
          int s = s0;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            if (s >= kDigits) continue;
            // the chunk's first products of an accumulator overwrite: those of W's top digit, then (5, 0)
            const bool opens = kk == 0 && (p == kDigits - 1 || (p == kMinDiag && s == 0));
            const int cnt = p == kMinDiag && s == 0 ? 1 : (kDigits - s < kAtOnce ? kDigits - s : kAtOnce);
            mma_of<Fp16x3>(make_idesc(0, BM, cnt * TN), tmem + (uint32_t)((p + s - kMinDiag) * TN),
                           sd + (uint32_t)((p * (int)L::W_SLICE) >> 4) + kk * 2u,
                           sd + (uint32_t)(((int)L::X_OFF + s * (int)L::X_SLICE) >> 4) + kk * 2u, kSdescHi64,
                           opens ? later : 1u, leader);
            s += cnt;
          }
        }
      }
      if (leader) {
        mma_commit(empty_bar(st));
        if (t % SPC == SPC - 1 || t == n_stages - 1) mma_commit(acc_full);
      }
      __syncwarp();
    }
    pdl_trigger();
    if (leader) {
      if (!ok) {
        *abort_flag = 1;
        atomicOr(&g_device_status, kStatusTimeout);
      }
      mma_commit(drain_bar);  // issued MMAs finish before TMEM is released
    }
    __syncwarp();
    // on the normal path too: the arrival must not land in the shared memory of a CTA that follows this one
    mbar_wait(drain_bar, 0u, kDrainNs, nullptr);
  } else {
    // ---------------- workers: digits of the tiles into the ring, accumulators into 96-bit sums ----------
    const int tid = (int)threadIdx.x - 32;  // 0 .. F64_WT - 1
    constexpr int CW = TN / (F64_WORKERS / 4);  // this warp's columns (tokens)
    const int q = warp & 3, part = (warp - 1) >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(part * CW);
    uint8_t* raw = smem + L::RAW_OFF;
    const uint32_t raw_addr = smem_u32(raw) + 16u * (uint32_t)tid;
    const int j = tid & 7, row0 = tid >> 3;  // 4 entries j of rows row0, row0 + ROWS_AT_ONCE of W, row0 of X~
    const bool x_on = row0 < TN;
    uint32_t run_lo[CW], run_mid[CW], run_hi[CW];  // the 96-bit sums
#pragma unroll
    for (int i = 0; i < CW; ++i) run_lo[i] = run_mid[i] = run_hi[i] = 0u;

    auto fetch = [&](int t) {  // stage t's raw entries of this thread
      const int64_t k = kbeg + 32 * (int64_t)t + 4 * j;
      const bool k_in = k < kend;  // whole groups of 4
#pragma unroll
      for (int i = 0; i < L::W_GROUPS; ++i) {
        const int64_t n = n0 + row0 + L::ROWS_AT_ONCE * i;
        const bool in = k_in && n < N;
        cp_async16(raw_addr + 16u * F64_WT * i, in ? W + n * K + k : W, in);
      }
      if (x_on) {
        const int64_t m = m0 + row0;
        const bool in = k_in && m < M;
#pragma unroll
        for (int h = 0; h < L::X_UNITS; ++h)
          cp_async16(raw_addr + 16u * F64_WT * (L::W_GROUPS + h), in ? X + m * K + k + (16 / (int)sizeof(TX)) * h : X,
                     in);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto cut = [&](int t) {  // this thread's entries of stage t: raw -> digits in the ring
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      uint8_t* stage = smem + (size_t)(t & 1) * L::STAGE;
      const uint8_t* mine = raw + 16 * (size_t)tid;
      auto dst_of = [&](uint32_t base, int row) {  // 64-byte swizzle
        return stage + base + row * 64 + (((j >> 1) ^ ((row >> 1) & 3)) << 4) + (j & 1) * 8;
      };
#pragma unroll
      for (int i = 0; i < L::W_GROUPS; ++i) {
        const int row = row0 + L::ROWS_AT_ONCE * i;
        store_digits(dst_of(0, row), L::W_SLICE, *reinterpret_cast<const float4*>(mine + 16 * F64_WT * i), s_exp[row]);
      }
      if (x_on) {
        const int e = s_exp[BM + row0];
        const uint8_t* xs = mine + 16 * F64_WT * L::W_GROUPS;
        if constexpr (sizeof(TX) == 4) {
          store_digits(dst_of(L::X_OFF, row0), L::X_SLICE, *reinterpret_cast<const float4*>(xs), e);
        } else {
          const double2 x = *reinterpret_cast<const double2*>(xs);
          const double2 y = *reinterpret_cast<const double2*>(xs + 16 * F64_WT);
          const unsigned long long v[4] = {fixed_digits(x.x, e), fixed_digits(x.y, e), fixed_digits(y.x, e),
                                           fixed_digits(y.y, e)};
          store_bytes<0>(dst_of(L::X_OFF, row0), L::X_SLICE, v);
        }
      }
    };
    bool ok = true;
    auto gather = [&](int c) {  // chunk c's accumulators into the sums
      ok = __all_sync(0xffffffffu, mbar_wait(acc_full, (uint32_t)c & 1u, kWaitNs * 2, abort_flag)) && !*abort_flag;
      if (!ok) return;
      tc_fence_after();
#pragma unroll
      for (int b = 0; b < CW / 4; ++b) {
        const uint32_t base = lane_base + 4u * b;
        uint32_t r[4][4];
        long long sum[2][4];  // accumulators 7..4 and 3..0, weights 2^24 .. 1 (units of 2^32 and of 1)
#pragma unroll
        for (int g = 0; g < 2; ++g) {
#pragma unroll
          for (int d = 0; d < 4; ++d) tmem_ld_32x4_nowait(base + (uint32_t)((7 - 4 * g - d) * TN), r[d]);
          tmem_wait_ld(r[0], r[1], r[2], r[3]);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            sum[g][i] = (long long)__float2int_rn(__uint_as_float(r[0][i])) * (1 << 24) +
                        (long long)__float2int_rn(__uint_as_float(r[1][i])) * (1 << 16) +
                        (long long)__float2int_rn(__uint_as_float(r[2][i])) * (1 << 8) +
                        (long long)__float2int_rn(__uint_as_float(r[3][i]));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const long long top = sum[0][i] + (sum[1][i] >> 32);  // >> rounds down: the low word stays unsigned
          const int o = 4 * b + i;
          asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
              : "+r"(run_lo[o]), "+r"(run_mid[o]), "+r"(run_hi[o])
              : "r"((uint32_t)sum[1][i]), "r"((uint32_t)top), "r"((uint32_t)((unsigned long long)top >> 32)));
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_free);
    };

    if (n_stages > 0) fetch(0);
    for (int t = 0; t < n_stages; ++t) {
      const int st = t & 1;
      if (t >= 2) {
        ok = __all_sync(0xffffffffu, mbar_wait(empty_bar(st), ((uint32_t)(t >> 1) & 1u) ^ 1u, kWaitNs, abort_flag));
        if (!ok) break;
      }
      cut(t);
      if (t + 1 < n_stages) fetch(t + 1);  // into the slots this thread has just read
      fence_proxy_async_smem();            // the digits before the MMAs that read them
      __syncwarp();
      if (lane == 0) mbar_arrive(full_bar(st));
      if (t % SPC == 0 && t > 0) {  // the chunk before, while its successor's first stage is ready
        gather(t / SPC - 1);
        if (!ok) break;
      }
    }
    if (ok && n_chunks > 0) gather(n_chunks - 1);
    pdl_trigger();
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (ok) {
      const int64_t n = n0 + 32 * q + lane;
#pragma unroll
      for (int i = 0; i < CW; ++i) {
        const int64_t m = m0 + part * CW + i;
        if (n < N && m < M) {
          const int64_t o = ((int64_t)blockIdx.y * M + m) * N + n;
          hi[o] = (long long)(((unsigned long long)run_hi[i] << 32) | run_mid[i]);
          lo[o] = run_lo[i];
        }
      }
    } else if (lane == 0) {
      *abort_flag = 1;
      atomicOr(&g_device_status, kStatusTimeout);
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, L::TMEM_COLS);
  }
}

// Outputs of 32 columns n x 32 rows m per block: the splits' sums added, scaled and finished.
// Guard: in units of 2^(E_x + E_w) the slices' error is at most 2^-54 (sum|w| + sum|x|) (the roundings to
// fixed point) + K 2^-57.6 (the dropped products), and the conversion adds 2 x 2^-53 S, so everything stays
// inside gamma_K S while S (1 - 2 / K) >= (mean|w| + mean|x|) / 2 + 0.04.  S is bounded from below by up to
// 128 of its terms, 8 runs of 16 of K (1.3 to 8 there for noise-masked rows, against 0.2 to 0.5).
constexpr int kGuardK = 128;
__device__ __forceinline__ float relative(float v, int e) {  // |v| 2^-E, below 2, rounded down; 0 if tiny
  const uint32_t u = __float_as_uint(v) & 0x7FFFFFFFu;
  const int ex = (int)(u >> 23) - e + 127;
  return ex > 0 && (u >> 23) ? __uint_as_float(((uint32_t)ex << 23) | (u & 0x7FFFFFu)) : 0.f;
}
__device__ __forceinline__ float relative(double v, int e) {
  const uint32_t u = (uint32_t)((unsigned long long)__double_as_longlong(v) >> 32) & 0x7FFFFFFFu;
  const int ex = (int)(u >> 20) - e + 127;
  return ex > 0 && (u >> 20) ? __uint_as_float(((uint32_t)ex << 23) | ((u & 0xFFFFFu) << 3)) : 0.f;
}

// Shared memory of a block of 32 x 32 outputs.
constexpr int kSumRow = 33;
struct F64Block {
  alignas(16) float ws[32][kGuardK + 4], xs[32][kGuardK + 4];  // sampled entries; once read, ws holds sums
  F64Row wr[32], xr[32];
  uint32_t soft[32], hard[32], done[32];  // by row, a bit a column: not cleared by the samples; not finite; summed again
  __device__ double* sums() { return reinterpret_cast<double*>(&ws[0][0]); }
};
static_assert(sizeof(double) * 32 * kSumRow <= sizeof(float) * 32 * (kGuardK + 4), "the block's sums");

// The V values of each lane summed over the warp: a lane gets the total of value lane / (32 / V) (halves exchanged while
// more than one is left: V - 1 sums and then log2(32 / V), not 5 V; in binary64 each costs 16 cycles of the SM's pipe).
template <int V, class T>
__device__ __forceinline__ T warp_totals(T (&v)[V], int lane) {
  int o = 16;
#pragma unroll
  for (int c = V; c >= 2; c /= 2, o /= 2) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < c / 2; ++i) {
      const T send = up ? v[i] : v[i + c / 2], keep = up ? v[i + c / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}
// Cells of a 32 x 32 block that the sampled bound does not clear, R rows (mr, mr + 1, ...) by 4 columns (nc, ...) a warp:
// those in `soft` (bit 4 r + c) are cleared when S over more of K, then all of it, does it; the others and those in
// `hard` are summed in binary64, each lane 2 of K at a time.  Returns the cells summed, their sums in res.
// The whole call, us, at 8192 by 3072 and 1, 16, 128 rows; last what the FP64 pipe's kernel (fp64.cu) takes of any rows:
//   all cleared by the samples             104   107   247
//   an entry a row 1000 times the others   109   142   401   (each summed again by a warp of its own: 692, 1985, 4660)
//   10000 times                            126   644  4628   (700, 2197, 6992)
//   an infinity in one row                 252   256   533   (1991, 2059, 2434)
//   every output summed again              316  1924  9013   (1967, 7041, 19080)
//   FP64 pipe                              129   958  7421
// Bound there by the FP64 pipe of the SMs that hold the blocks (96 of them up to 32 rows); small outputs have few: 16 x
// 512 by 512, an entry of 1000 a row, 69 us (117; 39 on the pipe).
template <int R, class TX>
__device__ __forceinline__ uint32_t f64_again(const float* __restrict__ W, const TX* __restrict__ X, int64_t M,
                                              int64_t K, int64_t N, int64_t mr, int64_t nc, const F64Row* xr,
                                              const F64Row* wr, uint32_t soft, uint32_t hard, float part, double* res) {
  using X2 = typename F64Pair<TX>::type;
  constexpr int V = 4 * R, LPV = 32 / V;  // cells, lanes a cell
  constexpr int64_t kRun = 512;           // of K between two looks at S
  const int lane = threadIdx.x & 31, cell = lane / LPV;
  const int r_max = (int)std::min<int64_t>(R - 1, M - 1 - mr), c_max = (int)std::min<int64_t>(3, N - 1 - nc);
  const float* w0 = W + nc * K + 2 * lane;
  const TX* x0 = X + mr * K + 2 * lane;
  if (soft != 0u) {
    float S[V];
#pragma unroll
    for (int i = 0; i < V; ++i) S[i] = 0.f;
    const float mean = wr[std::min(cell & 3, c_max)].mean + xr[std::min(cell >> 2, r_max)].mean;
    for (int64_t k0 = 0; k0 < K && soft != 0u; k0 += kRun) {
      const int64_t k1 = std::min(K, k0 + kRun) - 2 * lane;
#pragma unroll(R == 1 ? 4 : 1)
      for (int64_t k = k0; k < k1; k += 64) {
        float2 w[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) w[c] = __ldg(reinterpret_cast<const float2*>(w0 + std::min(c, c_max) * K + k));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int e = max(wr[std::min(c, c_max)].e, 1);
          w[c] = make_float2(relative(w[c].x, e), relative(w[c].y, e));
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const X2 x = __ldg(reinterpret_cast<const X2*>(x0 + std::min(r, r_max) * K + k));
          const int e = max(xr[std::min(r, r_max)].e, 1);
          const float xa = relative(x.x, e), xb = relative(x.y, e);
#pragma unroll
          for (int c = 0; c < 4; ++c) S[4 * r + c] = fmaf(w[c].x, xa, fmaf(w[c].y, xb, S[4 * r + c]));
        }
      }
      float t[V];
#pragma unroll
      for (int i = 0; i < V; ++i) t[i] = S[i];
      const bool clear = warp_totals<V>(t, lane) * part >= 0.51f * mean + 0.041f;
      soft &= ~__reduce_or_sync(0xffffffffu, clear ? 1u << cell : 0u);
    }
  }
  const uint32_t need = soft | hard;
  if (need == 0u) return 0u;
  double v[V];
#pragma unroll
  for (int i = 0; i < V; ++i) v[i] = 0.0;
#pragma unroll(R == 1 ? 4 : 1)
  for (int64_t k = 0; k < K - 2 * lane; k += 64) {
    float2 w[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) w[c] = __ldg(reinterpret_cast<const float2*>(w0 + std::min(c, c_max) * K + k));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const X2 x = __ldg(reinterpret_cast<const X2*>(x0 + std::min(r, r_max) * K + k));
      const double xa = (double)x.x, xb = (double)x.y;
#pragma unroll
      for (int c = 0; c < 4; ++c) v[4 * r + c] = fma(xb, (double)w[c].y, fma(xa, (double)w[c].x, v[4 * r + c]));
    }
  }
  const double t = warp_totals<V>(v, lane);
  if (lane % LPV == 0 && (need >> cell & 1u)) res[(cell >> 2) * kSumRow + (cell & 3)] = t;
  return need;
}

// The block's flagged cells, 4 rows x 4 columns a task, tasks dealt out to the 8 warps.  Not inlined: the kernel's own
// registers stay those of the common case.
template <class TX>
__device__ __noinline__ void f64_again_block(F64Block* blk, const float* __restrict__ W, const TX* __restrict__ X,
                                             int64_t M, int64_t K, int64_t N, int64_t m0, int64_t n0, float part) {
  double* res = blk->sums();
  for (int t = threadIdx.x >> 5; t < 64; t += 8) {
    const int g = 4 * (t >> 3), q = 4 * (t & 7);
    uint32_t sb = 0u, hb = 0u;
    int rows_in = 0, last = 0;
    for (int r = 0; r < 4; ++r) {
      const uint32_t a = blk->soft[g + r] >> q & 15u, b = blk->hard[g + r] >> q & 15u;
      sb |= a << (4 * r);
      hb |= b << (4 * r);
      if (a | b) {
        ++rows_in;
        last = r;
      }
    }
    if (rows_in == 0) continue;
    uint32_t done;
    if (rows_in == 1)
      done = f64_again<1, TX>(W, X, M, K, N, m0 + g + last, n0 + q, blk->xr + g + last, blk->wr + q, sb >> (4 * last),
                              hb >> (4 * last), part, res + (g + last) * kSumRow + q)
             << (4 * last);
    else
      done = f64_again<4, TX>(W, X, M, K, N, m0 + g, n0 + q, blk->xr + g, blk->wr + q, sb, hb, part,
                              res + g * kSumRow + q);
    if ((threadIdx.x & 31) == 0)
      for (int r = 0; r < 4; ++r) atomicOr(&blk->done[g + r], (done >> (4 * r) & 15u) << q);
  }
}

template <class TX>
__global__ void __launch_bounds__(256, 3) f64_finish_kernel(double* __restrict__ out64, float* __restrict__ out32,
                                                         const long long* __restrict__ hi,
                                                         const uint32_t* __restrict__ lo,
                                                         const F64Row* __restrict__ rows,
                                                         const float* __restrict__ W, const TX* __restrict__ X,
                                                         const double* __restrict__ c, int splits, int64_t M, int64_t K,
                                                         int64_t N, int mode) {
  __shared__ F64Block blk;
  auto& ws = blk.ws;
  auto& xs = blk.xs;
  auto& wr = blk.wr;
  auto& xr = blk.xr;
  pdl_wait();
  pdl_trigger();
  const int64_t n0 = (int64_t)blockIdx.x * 32, m0 = (int64_t)blockIdx.y * 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < 64) {
    const int i = threadIdx.x & 31;
    const bool isw = threadIdx.x < 32;
    const bool in = isw ? n0 + i < N : m0 + i < M;
    const F64Row r = in ? rows[isw ? n0 + i : N + m0 + i] : F64Row{0, 0.f};
    (isw ? wr : xr)[i] = r;
  }
  __syncthreads();
  const int64_t nb = std::max<int64_t>(1, std::min<int64_t>(kGuardK / 16, K / 16));  // disjoint runs of 16 of K
  const int64_t step = K / nb / 16 * 16;
  const float part = 0.999f * (float)(K - 2) / (float)K;
  {  // a thread takes one of the sampled columns, rows threadIdx.x / kGuardK, + 2, ...: all its loads in flight
    const int s = threadIdx.x % kGuardK;
    const int64_t k = (s / 16) * step + s % 16;
    const bool k_in = s / 16 < nb && k < K;
    float wv[16];
    TX xv[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int r = threadIdx.x / kGuardK + 2 * i;
      wv[i] = k_in && n0 + r < N ? __ldg(W + (n0 + r) * K + k) : 0.f;
      xv[i] = k_in && m0 + r < M ? __ldg(X + (m0 + r) * K + k) : (TX)0;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int r = threadIdx.x / kGuardK + 2 * i;
      ws[r][s] = relative(wv[i], max(wr[r].e, 1));
      xs[r][s] = relative(xv[i], max(xr[r].e, 1));
    }
  }
  __syncthreads();
  float S[4] = {0.f, 0.f, 0.f, 0.f};  // rows m0 + 4 warp + 0..3, column n0 + lane
  for (int s = 0; s < kGuardK; s += 4) {
    const float4 w4 = *reinterpret_cast<const float4*>(&ws[lane][s]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 x4 = *reinterpret_cast<const float4*>(&xs[4 * warp + i][s]);
      S[i] = fmaf(w4.x, x4.x, fmaf(w4.y, x4.y, fmaf(w4.z, x4.z, fmaf(w4.w, x4.w, S[i]))));
    }
  }
  const int64_t n = n0 + lane;
  const F64Row rw = wr[lane];
  long long h[4] = {0, 0, 0, 0}, l[4] = {0, 0, 0, 0};
  for (int sp = 0; sp < splits; ++sp)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t m = m0 + 4 * warp + i, o = ((int64_t)sp * M + m) * N + n;
      if (m < M && n < N) {
        h[i] += __ldcg(hi + o);
        l[i] += (long long)__ldcg(lo + o);
      }
    }
  double out[4];
  uint32_t flagged = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t m = m0 + 4 * warp + i;
    const F64Row rx = xr[4 * warp + i];
    bool soft = false, hard = false;
    out[i] = 0.0;
    if (m < M && n < N) {
      const long long top = h[i] + (l[i] >> 32), low = l[i] & 0xFFFFFFFFll;
      // value (top 2^32 + low) 2^(40 - 106 + E_w + E_x), E = e - 127 or e - 1023
      const int sc = 40 - 106 + (max(rw.e, 1) - 127) + (max(rx.e, 1) - (sizeof(TX) == 8 ? 1023 : 127));
      const int s1 = sc / 2, s2 = sc - s1;  // in two exact steps, each a normal power of two
      out[i] = fma((double)top, 4294967296.0, (double)low) * __hiloint2double((s1 + 1023) << 20, 0) *
               __hiloint2double((s2 + 1023) << 20, 0);
      hard = rw.e == kRowNonFinite || rx.e == kRowNonFinite;
      const bool zero = rw.e == 0 || rx.e == 0;  // a row of zeros (with a finite one): exactly 0
      soft = !hard && !zero && !(S[i] * part >= 0.51f * (rw.mean + rx.mean) + 0.041f);
    }
    const uint32_t sm = __ballot_sync(0xffffffffu, soft), hm = __ballot_sync(0xffffffffu, hard);
    if (lane == 0) {
      blk.soft[4 * warp + i] = sm;
      blk.hard[4 * warp + i] = hm;
      blk.done[4 * warp + i] = 0u;
    }
    flagged |= sm | hm;
  }
  if (__syncthreads_or((int)flagged) != 0) {
    f64_again_block<TX>(&blk, W, X, M, K, N, m0, n0, part);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (blk.done[4 * warp + i] >> lane & 1u) out[i] = blk.sums()[(4 * warp + i) * kSumRow + lane];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t m = m0 + 4 * warp + i;
    if (m < M && n < N) finish_f64(out64, out32, m * N + n, out[i], c, mode);
  }
}

// ---- host side ----
// Plan of a product: tokens per tile, K range of a split, splits; 0 tokens: the FP64 pipe's kernel takes it.
struct F64TcPlan {
  int tn;
  int64_t k_per_split;
  int splits;
  int64_t rows_bytes, hi_bytes;
  size_t bytes;  // after the counters
};

F64TcPlan plan_f64_tc(int64_t M, int64_t K, int64_t N) {
  F64TcPlan p{};
  const int cc = device_cc();
  if ((cc != 100 && cc != 103) || !f64_on_tensor_cores(M, K, N)) return p;
  p.tn = M <= 16 ? 16 : M <= 32 ? 32 : 64;
  const int64_t tiles = ceil_div(N, (int64_t)BM) * ceil_div(M, (int64_t)p.tn), chunks = ceil_div(K, (int64_t)F64_CHUNK);
  const int64_t sms = device_sm_count();
  double best = 1e300;
  for (int64_t s = 1; s <= std::min<int64_t>(chunks, 64); ++s) {  // a CTA's fixed time is about that of 2 chunks
    const double c = (double)ceil_div(tiles * s, sms) * ((double)ceil_div(chunks, s) + 2.0) + 0.02 * (double)s;
    if (c < best * (1.0 - 1e-9)) {
      best = c;
      p.k_per_split = ceil_div(chunks, s) * F64_CHUNK;
    }
  }
  p.splits = (int)ceil_div(K, p.k_per_split);
  p.rows_bytes = round_up((N + M) * (int64_t)sizeof(F64Row), 256);
  p.hi_bytes = round_up((int64_t)p.splits * M * N * 8, 256);
  p.bytes = (size_t)(p.rows_bytes + p.hi_bytes + round_up((int64_t)p.splits * M * N * 4, 256));
  return p;
}

template <int TN, class TX>
spl_status launch_f64_tc(const F64TcPlan& p, double* out64, float* out32, const TX* A, const float* W, const double* c,
                         int64_t M, int64_t K, int64_t N, char* ws, cudaStream_t stream, int mode) {
  using L = F64Cfg<TN, TX>;
  static bool done[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPL_ECUDA;
  if (!done[dev]) {
    if (cudaFuncSetAttribute(tc_f64_kernel<TN, TX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM) !=
        cudaSuccess)
      return SPL_ECUDA;
    done[dev] = true;
  }
  F64Row* rows = reinterpret_cast<F64Row*>(ws);
  long long* hi = reinterpret_cast<long long*>(ws + p.rows_bytes);
  uint32_t* lo = reinterpret_cast<uint32_t*>(ws + p.rows_bytes + p.hi_bytes);
  spl_status st = launch_pdl(f64_rows_kernel<TX>, dim3((unsigned)(N + M)), dim3(256), 0, stream, rows, W, A, K, N);
  if (st != SPL_OK) return st;
  const dim3 grid((unsigned)ceil_div(N, (int64_t)BM), (unsigned)p.splits, (unsigned)ceil_div(M, (int64_t)TN));
  st = launch_pdl(tc_f64_kernel<TN, TX>, grid, dim3(F64_THREADS), L::SMEM, stream, hi, lo, (const F64Row*)rows, W, A, M,
                  K, N, p.k_per_split);
  if (st != SPL_OK) return st;
  return launch_pdl(f64_finish_kernel<TX>, dim3((unsigned)ceil_div(N, (int64_t)32), (unsigned)ceil_div(M, (int64_t)32)),
                    dim3(256), 0, stream, out64, out32, (const long long*)hi, (const uint32_t*)lo, (const F64Row*)rows,
                    W, A, c, p.splits, M, K, N, mode);
}
