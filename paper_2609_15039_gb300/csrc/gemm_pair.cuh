// FP16X3 products on SM pairs (tcgen05 cta_group::2): the form the prefill-sized products take.
// Part of gemm_tc.cu (included there, inside its namespace, after the PTX wrappers).
//
// What bounds the one-SM tiles: a 128 x 256 x 16 MMA takes 128 cycles and reads 4 KB of A and 8 KB of W
// from shared memory (96 B per cycle), while TMA writes 48 KB per k-block of 32 -- 150 B per cycle in all
// at full rate, over the 128 the SM's shared memory moves, so the tensor pipe waits (1044 cycles per
// k-block measured against 768 of MMAs).  Here two CTAs of a cluster, one per SM, compute one 256 x BN
// tile: each holds its own 128 rows of A and half of the tile's W rows, and the hardware gives both SMs
// the whole W tile, so an MMA reads 4 + 4 KB per SM, a k-block loads 32 KB per SM instead of 48, and A_hi,
// an operand of two of the three products, is kept in the tensor core between them (collector::a).
//
// Persistent: one pair per two SMs loops over the tiles pair, pair + pairs, ... (M fastest).  Warps:
//   warp 0      TMA producer (both CTAs): own 128 rows of A, own half of W; every copy signals the
//               leader's (cluster rank 0) full barrier.
//   warp 1      TMEM allocator (both), MMA issuer (leader): three products per k-step into one of two
//               accumulators of 128 lanes x BN columns in each SM; commits are multicast to both CTAs.
//   warps 2-9   epilogue: two warpgroups, each half of the columns of the SM's 128 rows.
// The K range is cut into segments of `chain` k-blocks of 32 (see kChainBlocks); segments alternate between
// the two accumulators.  The epilogue keeps the tile's running sum in registers (up to 128 per thread):
// the first segment is read, later ones are added with round-to-nearest (R = fl(R + P)), the same sums in
// the same order as tc_gemm_kernel's unsplit segmented form, so the result equals it bit for bit.  An
// accumulator is handed back as soon as it is read, so folding, C and the stores overlap the MMAs of the
// next segments.  C comes in and the result goes out by TMA, 32 rows x 32 columns per warp at a time
// through 4 KB of shared memory of the warp's own (rows and columns past the tensor are clipped); where
// an output row is not a whole number of 16-byte units (N % 4 != 0) the warp writes the 4 KB out row by row.
//
// Hand-over: every segment of the CTA's tiles, numbered g = 0, 1, ..., uses accumulator g % 2; its sums are
// complete at completion g / 2 of buf_full[g % 2] (in each CTA, one multicast commit) and the accumulator
// is free for segment g + 2 at completion g / 2 of buf_free[g % 2] (the leader's; 16 arrivals, one per
// epilogue warp of both CTAs).  Every wait is bounded; a role that gives up raises its CTA's abort flag and
// the device status word, copies and MMAs already issued are waited for, and the two CTAs leave together.

constexpr int PAIR_THREADS = 320, PAIR_EPI_WARPS = 8;

template <int BN>
struct PairCfg {
  static_assert(BN % 32 == 0 && BN >= 128 && BN <= 256, "cta_group::2, M = 256: N a multiple of 32 up to 256");
  static constexpr int BK = 64;  // fp16 elements of K per stage: 128-byte rows, 128-byte swizzle (two k-blocks)
  static constexpr uint32_t A_HALF = 128 * BK * 2, W_HALF = (BN / 2) * BK * 2;
  static constexpr uint32_t A_HI = 0, A_LO = A_HALF, W_HI = 2 * A_HALF, W_LO = W_HI + W_HALF;
  static constexpr uint32_t STAGE = W_LO + W_HALF;  // bytes TMA brings per stage and CTA
  static constexpr uint32_t STAGING = PAIR_EPI_WARPS * 4096;
  static constexpr uint32_t TOTAL = 224u * 1024u;
  static constexpr int STAGES = (int)((TOTAL - STAGING) / STAGE);
  static constexpr uint32_t STAGING_OFF = STAGES * STAGE, AUX_OFF = STAGING_OFF + STAGING;
  static constexpr uint32_t SCALE_OFF = AUX_OFF + 1024;    // per epilogue warp: 2^-e of 32 rows of W
  static constexpr uint32_t SMEM = SCALE_OFF + PAIR_EPI_WARPS * 128 + 1024;  // + alignment slack
  static constexpr uint32_t IDESC = make_idesc(0, 256, BN);
  static constexpr uint32_t ACC_COLS = 256, TMEM_COLS = 512;
  static constexpr int CHUNKS = BN / 32, G0 = (CHUNKS + 1) / 2;  // column chunks; those of warpgroup 0
  // full[S], empty[S], buf_full[2], buf_free[2], drain, c_load[8], then the TMEM slot and the abort flag
  static constexpr uint32_t AUX_BARS = 8 * (2 * STAGES + 5 + PAIR_EPI_WARPS);
  static_assert(W_HALF % 1024 == 0 && W_HI % 1024 == 0 && STAGE % 1024 == 0, "swizzle atoms aligned");
  static_assert(STAGES >= 3 && AUX_BARS + 16 <= 1024 && SMEM <= 232448, "shared memory of the CTA");
};

__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t leader_bar, int x,
                                                 int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(leader_bar), "l"(policy)
      : "memory");
}
// The MMAs issued so far arrive, once done, on the barrier at this offset in both CTAs.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// mbar_wait for a barrier that the other CTA of the pair arrives on.
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, unsigned long long budget_ns,
                                                  volatile int* abort) {
  if (mbar_try_cluster(bar, parity)) return true;
  const unsigned long long deadline = now_ns() + budget_ns;
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_cluster(bar, parity)) return true;
    if ((it & 63u) == 0u && ((abort && *abort) || now_ns() > deadline)) return false;
  }
}

template <int BN>
__global__ void __launch_bounds__(PAIR_THREADS, 1)
tc_pair_kernel(const __grid_constant__ TcMaps maps, float* __restrict__ out, const float* __restrict__ C,
               const int* __restrict__ a_exp, const int* __restrict__ w_exp, int64_t M, int64_t K, int64_t N, int tiles,
               int m_tiles, int chain, int64_t c_rows) {
  using L = PairCfg<BN>;
  constexpr int STAGES = L::STAGES, BK = L::BK;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* aux = smem + L::AUX_OFF;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(aux + L::AUX_BARS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(aux + L::AUX_BARS + 8);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);
  const int my_tiles = tiles > pair ? (tiles - 1 - pair) / pairs + 1 : 0;
  const int nk = (int)ceil_div(K, 32), ns = (int)ceil_div(K, BK);  // k-blocks and stages of a tile
  const int seg_len = chain > 0 && chain < nk ? chain : nk;        // k-blocks per segment
  const int nseg = (int)ceil_div(nk, seg_len);
  const uint32_t bar_base = smem_u32(aux);
  auto full_bar = [&](int st) { return bar_base + 8u * st; };
  auto empty_bar = [&](int st) { return bar_base + 8u * (STAGES + st); };
  auto buf_full = [&](int b) { return bar_base + 8u * (2 * STAGES + b); };
  auto buf_free = [&](int b) { return bar_base + 8u * (2 * STAGES + 2 + b); };
  const uint32_t drain_bar = bar_base + 8u * (2 * STAGES + 4);
  auto c_bar = [&](int w) { return bar_base + 8u * (2 * STAGES + 5 + w); };
  // this CTA's 128 rows of A and of the output, and the tile's first column
  auto tile_origin = [&](int i, int64_t& m0, int64_t& n0) {
    const int tile = pair + i * pairs;
    m0 = (int64_t)(tile % m_tiles) * 256 + 128 * (int64_t)rank;
    n0 = (int64_t)(tile / m_tiles) * BN;
  };

  if (threadIdx.x == 0) {
    for (int st = 0; st < STAGES; ++st) {
      mbar_init(full_bar(st), 1);
      mbar_init(empty_bar(st), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(buf_full(b), 1);
      mbar_init(buf_free(b), 2 * PAIR_EPI_WARPS);
    }
    mbar_init(drain_bar, 1);
    for (int w = 0; w < PAIR_EPI_WARPS; ++w) mbar_init(c_bar(w), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_slot))),
                 "r"(L::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers are set up before either signals the other's
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs): the ring runs on across the pair's tiles ----------------
    // The leader's full barrier expects both CTAs' bytes; a stage is free in both once the leader's
    // commit arrives on each CTA's empty barrier.  W does not depend on the kernel before this one: the
    // first stages' W tiles are issued before the wait for it.
    bool ok = true;
    const uint64_t pol_w = l2_evict_first(), pol_a = l2_evict_last();
    const uint32_t lead_full = map_to_rank(bar_base, 0);  // the leader's full[0]
    auto load_w = [&](int st, int kb, int64_t n0) {
      const uint32_t sa = smem_u32(smem + (size_t)st * L::STAGE);
      const int y = (int)(n0 + (int64_t)rank * (BN / 2));
      tma_load_2d_pair(sa + L::W_HI, &maps.w_hi, lead_full + 8u * st, kb * BK, y, pol_w);
      tma_load_2d_pair(sa + L::W_LO, &maps.w_lo, lead_full + 8u * st, kb * BK, y, pol_w);
    };
    auto load_a = [&](int st, int kb, int64_t m0) {
      const uint32_t sa = smem_u32(smem + (size_t)st * L::STAGE);
      tma_load_2d_pair(sa + L::A_HI, &maps.a_hi, lead_full + 8u * st, kb * BK, (int)m0, pol_a);
      tma_load_2d_pair(sa + L::A_LO, &maps.a_lo, lead_full + 8u * st, kb * BK, (int)m0, pol_a);
    };
    const int pre = my_tiles > 0 ? (ns < STAGES ? ns : STAGES) : 0;  // stages filled before any is freed
    if (pre > 0 && lane == 0) {
      int64_t m0, n0;
      tile_origin(0, m0, n0);
      for (int kb = 0; kb < pre; ++kb) {
        if (rank == 0) mbar_expect_tx(full_bar(kb), 2 * L::STAGE);
        load_w(kb, kb, n0);
      }
    }
    __syncwarp();
    pdl_wait();  // A comes from the kernel before this one
    if (pre > 0 && lane == 0) {
      int64_t m0, n0;
      tile_origin(0, m0, n0);
      for (int kb = 0; kb < pre; ++kb) load_a(kb, kb, m0);
    }
    __syncwarp();
    uint32_t it = (uint32_t)pre;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int64_t m0, n0;
      tile_origin(i, m0, n0);
      for (int kb = i == 0 ? pre : 0; kb < ns; ++kb, ++it) {
        const int st = (int)(it % STAGES);
        if (it >= (uint32_t)STAGES) {
          ok = __all_sync(0xffffffffu, mbar_wait(empty_bar(st), ((it / STAGES) & 1u) ^ 1u, kWaitNs, abort_flag));
          if (!ok) break;
        }
        if (lane == 0) {
          if (rank == 0) mbar_expect_tx(full_bar(st), 2 * L::STAGE);
          load_a(st, kb, m0);
          load_w(st, kb, n0);
        }
        __syncwarp();
      }
    }
    pdl_trigger();
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicOr(&g_device_status, kStatusTimeout);
      }
      // copies already issued land well within this time (their barrier may be in the other CTA)
      const unsigned long long until = now_ns() + kDrainNs;
      while (now_ns() < until) {
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader): segments alternate between the accumulators ----------------
    bool ok = true;
    const uint32_t leader = elect_one();
    if (rank == 0) {
      const uint32_t sd0 = sdesc_lo(smem_u32(smem));
      int st = 0;
      uint32_t ph = 0u, g = 0;
      for (int i = 0; i < my_tiles && ok; ++i) {
        for (int sg = 0; sg < nseg && ok; ++sg, ++g) {
          const uint32_t b = g & 1u;
          if (g >= 2) {
            ok = __all_sync(0xffffffffu,
                            mbar_wait_cluster(buf_free(b), ((g >> 1) - 1u) & 1u, kWaitNs * 4, abort_flag));
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t acc = tmem + b * L::ACC_COLS;
          const int kb0 = sg * seg_len, kb1 = std::min(nk, kb0 + seg_len);
          for (int kb = kb0; kb < kb1; ++kb) {  // even blocks open a stage, odd ones (or the tile's last) free it
            if ((kb & 1) == 0 || kb == kb0) {
              ok = __all_sync(0xffffffffu, mbar_wait(full_bar(st), ph, kWaitNs, abort_flag));
              if (!ok) break;
              tc_fence_after();
            }
            const uint32_t sd = sd0 + (uint32_t)st * (L::STAGE >> 4) + (uint32_t)(kb & 1) * 4u;
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
              const uint32_t k = sd + kk * 2u;  // one instruction's K is 32 bytes of the swizzled row
              const uint32_t first = (kb == kb0 && kk == 0) ? 0u : 1u;
              mma<Fp16x3, L::IDESC, 2>(acc, k + (L::A_LO >> 4), k + (L::W_HI >> 4), kSdescHi128, first,
                                                  leader);
              mma<Fp16x3, L::IDESC, 2, kCollFill>(acc, k + (L::A_HI >> 4), k + (L::W_LO >> 4), kSdescHi128, 1u,
                                                  leader);
              mma<Fp16x3, L::IDESC, 2, kCollUse>(acc, k + (L::A_HI >> 4), k + (L::W_HI >> 4), kSdescHi128, 1u,
                                                 leader);
            }
            if ((kb & 1) != 0 || kb == nk - 1) {
              if (leader) mma_commit_pair(empty_bar(st));
              if (++st == STAGES) {
                st = 0;
                ph ^= 1u;
              }
            }
            __syncwarp();
          }
          if (!ok) break;
          if (leader) mma_commit_pair(buf_full(b));  // the segment's sums are complete once these MMAs are
          __syncwarp();
        }
      }
    }
    pdl_trigger();
    if (!ok) {
      if (leader) {
        *abort_flag = 1;
        atomicOr(&g_device_status, kStatusTimeout);
        mma_commit_pair(drain_bar);  // MMAs already issued finish before TMEM is released
      }
      __syncwarp();
      mbar_wait(drain_bar, 0u, kDrainNs, nullptr);
    }
  } else {
    // ---------------- warps 2..9: the running sum in registers, then C and the result ----------------
    const int q = warp & 3;           // TMEM lane quarter this warp may access
    const int grp = (warp - 2) >> 2;  // warpgroup: its column chunks are [c_lo, c_lo + nc)
    const int c_lo = grp ? L::G0 : 0, nc = grp ? L::CHUNKS - L::G0 : L::G0;
    const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * c_lo);
    uint8_t* stage_out = smem + L::STAGING_OFF + (size_t)(warp - 2) * 4096;  // 32 rows x 32 fp32, 128-byte swizzle
    const uint32_t stage_addr = smem_u32(stage_out);
    float* col_scale = reinterpret_cast<float*>(smem + L::SCALE_OFF) + 32 * (warp - 2);
    const uint32_t my_cbar = c_bar(warp - 2);
    const uint32_t lead_free = map_to_rank(buf_free(0), 0);
    const uint64_t pol_c = l2_evict_first();
    pdl_wait();  // C and the row exponents of A come from before this kernel
    bool ok = true;
    uint32_t g = 0, c_loads = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      int64_t m0, n0;
      tile_origin(i, m0, n0);
      const int64_t mw = m0 + 32 * q;  // the warp's first row
      const int64_t m = mw + lane;
      const float sr = m < M ? pow2f(-__ldg(a_exp + m)) : 1.0f;
      const bool tma_epi = (N & 3) == 0;
      const bool rows_in = mw < M, has_c = tma_epi && rows_in && mw < c_rows;
      // C's chunk c of this warp into the staging rows, once the last result has been copied out of them
      auto fetch_c = [&](int c) {
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          mbar_expect_tx(my_cbar, 4096);
          tma_load_2d(stage_addr, &maps.c, my_cbar, (int)(n0 + 32 * (c_lo + c)), (int)mw, pol_c);
        }
        __syncwarp();
      };
      if (has_c && nc > 0 && n0 + 32 * c_lo < N) fetch_c(0);  // in flight during the tile's mainloop
      if (!tma_epi && m < c_rows)  // the warp's rows of C into L2 meanwhile
        for (int64_t n = n0 + 32 * c_lo; n < n0 + 32 * (c_lo + nc) && n < N; n += 32) prefetch_l2(C + m * N + n);
      float run[L::G0][32];
      // segment g's sums are complete: its accumulator (false: gave up)
      auto take = [&](uint32_t& base) {
        const int b = (int)(g & 1u);
        ok = __all_sync(0xffffffffu, mbar_wait(buf_full(b), (g >> 1) & 1u, kWaitNs * 4, abort_flag)) && !*abort_flag;
        base = lane_base + (uint32_t)b * L::ACC_COLS;
        tc_fence_after();
        return ok;
      };
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(lead_free + 8u * (g & 1u));
        ++g;
      };
      uint32_t base;
      if (!take(base)) break;
#pragma unroll
      for (int c = 0; c < L::G0; ++c)
        if (c < nc) tmem_ld_32x32(base + (uint32_t)(32 * c), run[c]);
      release();
#pragma unroll 1
      for (int sg = 1; sg < nseg; ++sg) {
        if (!take(base)) break;
#pragma unroll
        for (int c = 0; c < L::G0; ++c)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (c >= nc) continue;
            float p[16];
            tmem_ld_32x16(base + (uint32_t)(32 * c + 16 * h), p);
#pragma unroll
            for (int j = 0; j < 16; ++j) run[c][16 * h + j] = __fadd_rn(run[c][16 * h + j], p[j]);
          }
        release();
      }
      if (!ok) break;
#pragma unroll
      for (int c = 0; c < L::G0; ++c) {
        const int64_t nc0 = n0 + 32 * (c_lo + c);
        if (c < nc && rows_in && nc0 < N) {  // the same for the whole warp
          col_scale[lane] = pow2f(-(nc0 + lane < N ? __ldg(w_exp + nc0 + lane) : 0));
          __syncwarp();
          if (has_c) {
            if (c > 0) fetch_c(c);
            ok = ok && __all_sync(0xffffffffu, mbar_wait(my_cbar, c_loads & 1u, kWaitNs, abort_flag));
            ++c_loads;
          } else if (tma_epi) {
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
          }
          float4* row = reinterpret_cast<float4*>(stage_out + (size_t)lane * 128);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 sc = *reinterpret_cast<const float4*>(col_scale + 4 * j);
            float4 o = make_float4((run[c][4 * j] * sr) * sc.x, (run[c][4 * j + 1] * sr) * sc.y,
                                   (run[c][4 * j + 2] * sr) * sc.z, (run[c][4 * j + 3] * sr) * sc.w);
            float4* dst = row + (j ^ (lane & 7));
            if (has_c) {
              const float4 cc = *dst;
              o = make_float4(__fsub_rn(o.x, cc.x), __fsub_rn(o.y, cc.y), __fsub_rn(o.z, cc.z), __fsub_rn(o.w, cc.w));
            }
            *dst = o;
          }
          if (tma_epi) {
            fence_proxy_async_smem();  // these writes before the copy that reads them
            __syncwarp();
            if (lane == 0) {
              if (ok) tma_store_2d(&maps.y, stage_addr, (int)nc0, (int)mw);
              asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
          } else {
            // output rows of no whole 16-byte units: lanes along a row, all 32 rows of C in flight at once
            // (one row after the other: 469 us at 952 by 80 by 26301, 143 so)
            const bool col = nc0 + lane < N;
            const int64_t o0 = mw * N + nc0 + lane;
            const int live = col ? (int)std::min<int64_t>(32, M - mw) : 0;
            const int c_end = col && mw < c_rows ? (int)std::min<int64_t>(32, c_rows - mw) : 0;
            float cc[32];
#pragma unroll
            for (int r = 0; r < 32; ++r) cc[r] = r < c_end ? __ldcs(C + o0 + r * N) : 0.f;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 32; ++r) {
              const float v = reinterpret_cast<const float*>(stage_out)[32 * r + 4 * ((lane >> 2) ^ (r & 7)) + (lane & 3)];
              if (r < live) out[o0 + r * N] = r < c_end ? __fsub_rn(v, cc[r]) : v;
            }
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    pdl_trigger();
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicOr(&g_device_status, kStatusTimeout);
      const unsigned long long until = now_ns() + kDrainNs;  // a copy of C still in flight lands
      while (now_ns() < until) {
      }
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the other CTA's MMAs, signals and reads of this one are done
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(L::TMEM_COLS) : "memory");
  }
  cluster_sync_all();
}
