// fp32 tap convolution on the tensor cores.  Included by dc_f32_kernels.cu inside its anonymous namespace.
//
// An fp32 number is the exact sum of three bf16 numbers (8 + 8 + 8 bits of significand): x = h + m + l with h = bf16(x),
// m = bf16(x - h), l = x - h - m.  The product of two such sums keeps the six terms down to 2^-16 of the leading one,
//   a b = ah bh + (ah bm + am bh) + (ah bl + am bm + al bh),
// and drops three below 2^-24, the size of an fp32 rounding.  tcgen05 multiplies bf16 exactly and accumulates in fp32; the three
// magnitudes have accumulators of their own, so that the small terms are not rounded to the large one's grid, and the epilogue adds
// them smallest first.  Six bf16 products still run at several times the rate of the FP32 pipe: the batched 64-channel residual
// block of the vocoder (192,000 frames) went from 213 us, 22 TFLOP/s, on FFMA tiles (4 x 4 per thread, bound by shared-memory
// operand latency) to what the conversion and the fp32 rows' traffic cost.
//
// One CTA: M (128 or 64) frames x BN channels of one phase.  Ten warps: 0..7 read the fp32 input rows (ring, or the caller's chunk), split
// them and write the three bf16 planes as swizzled operand tiles, and later run the epilogue; 8 issues the products; 9 streams the
// weights, split and packed as swizzled tiles at create.
// A panel holds 64 channels of the tile's frames and of the up to 8 in front of them: a tap is a row offset of the operand
// descriptor, so a row is read and split once for all its taps.  (Dilations above 4 fill the panel once per tap.)
// Per 64 channels and tap: 4 reduction steps of ah x bh, ah x [bm bl], am x [bh bm], al x bh.

constexpr int TC_H = 8;                           // left-context rows in front of a tile's frames
constexpr int tc_panel(int M) { return 3 * (M + TC_H) * 128; }   // bytes of a panel (64 channels): three bf16 planes
constexpr int TC_THREADS = 320, TC_CONV = 256;     // converting / epilogue threads
constexpr int TC_MAX_A = 2, TC_MAX_B = 4;
constexpr int TC_BARS = 1024;                      // barriers (and alignment slack: the base is declared 1024-byte aligned)

__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, int* s_fail, int* err, int code) {
  const uint32_t a = ptx::smem_u32(bar);
#pragma unroll 1
  for (uint32_t i = 0; i < (1u << 20); ++i) {
    if (__all_sync(0xffffffffu, ptx::mbar_try_wait_s(a, parity))) return true;
    if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(s_fail) != 0)) return false;
  }
  *reinterpret_cast<volatile int*>(s_fail) = 1;
  atomicCAS(err, 0, code);
  __syncwarp();
  return false;
}

// Two fp32 values -> their h, m and l parts as bf16 pairs.
__device__ __forceinline__ void split2(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
  __nv_bfloat162 b = __floats2bfloat162_rn(x, y);
  h = *reinterpret_cast<const uint32_t*>(&b);
  x -= __uint_as_float(h << 16);
  y -= __uint_as_float(h & 0xFFFF0000u);
  b = __floats2bfloat162_rn(x, y);
  m = *reinterpret_cast<const uint32_t*>(&b);
  x -= __uint_as_float(m << 16);
  y -= __uint_as_float(m & 0xFFFF0000u);
  b = __floats2bfloat162_rn(x, y);
  l = *reinterpret_cast<const uint32_t*>(&b);
}

// The random excitation of four channels of one output frame.  A call: inlined into the epilogue's unrolled loop the generator and its
// logarithms and sines are most of the kernel's code, which every CTA then fetches past.
__device__ __noinline__ float4 excite4(float4 v, long long t, int n, int rng_id, float std_dev, uint32_t seed_lo, uint32_t seed_hi) {
  uint32_t w[4];
  float e[4];
  philox4x32_10((uint32_t)(unsigned long long)t, (uint32_t)((unsigned long long)t >> 32), (uint32_t)(n >> 2), 0x80000000u + (uint32_t)rng_id, seed_lo,
                seed_hi, w);
  normals4(w, e);
  return make_float4(fmaf(std_dev, e[0], v.x), fmaf(std_dev, e[1], v.y), fmaf(std_dev, e[2], v.z), fmaf(std_dev, e[3], v.w));
}

// The tensor cores truncate when they add to an accumulator, which over a long reduction is a bias (7.6e-5 of RMS at the vocoder's end
// with one accumulator, 2.1e-5 with one per panel).  So the leading term of every (panel, tap) - four additions - has an accumulator of
// its own, which the epilogue threads add up in registers, rounded to nearest.  DRAIN (inputs of more than one panel): two sets of three, a
// panel's taps each, one set added up while the next panel is multiplied.  One panel: one set.  At 64 columns, where two CTAs share the SM's
// tensor memory: two accumulators that the taps take in turn (TURN).  (64 frames and several panels as well: a launch alone has one such tile per SM at most, but
// launches of other sessions lie beside it.  Three models of 2, 3 and 5 streams each 182, 272 and 325 us, with room for one CTA per SM 190, 275 and 331; one
// model 101.5, 133.5 and 155.3 against 101.1, 133.4 and 153.8.)  (A single one for the three taps, twelve additions: ten layers of 64 channels
// end at 4.3e-6 of their norm, against 2.0e-6 for sums of the FP32 pipe.)
//
// PACK (batches; chunks of up to TC_PACK frames at the layer's rate): a tile holds two slots, the second one's rows 64 behind the
// first one's, so that the panel's rows 64 .. 71 are its left context.  Alone, a chunk of 50 frames at the vocoder's first rate left 61 %
// of every product to padding.
constexpr int TC_SEG = 64, TC_PACK = TC_SEG - TC_H;
struct TcSlot {       // one stream's share of a launch
  int          T;     // frames at the layer's rate
  long long    pos;
  const float* in_direct;
  float*       out_direct;
  const float* in_ring;
  float*       out_ring;
  float*       save_ring;
  int          rng_id;
};

//
// M: frames of a tile.  64 where tiles of 128 would leave SMs without one (launch_tapconv_tc has the rule and the figures).  A 64-row product lies in sixteen
// TMEM lanes of each quarter, so that the epilogue's eight warps all have rows: a thread holds 8 columns of each 16.
template <int BN, bool DRAIN, bool PACK, int M>
__global__ void __launch_bounds__(TC_THREADS, DRAIN && M == 128 ? 1 : 2) tapconv_tc_kernel(const __grid_constant__ TapConvF32 p, const __grid_constant__ TapConvTc tc) {
  // per-call values: from the device-side call record of the stream or of the slot (captured graphs), or by value
  const int plane = (p.batch != nullptr ? blockIdx.z / p.n_phase : 0), phase = blockIdx.z - plane * p.n_phase;
  auto record = [&](int slot) {
    TcSlot a{p.T_in, p.pos_in, p.in_direct, p.out_direct, p.in_ring, p.out_ring, p.save_ring, p.exc_rng_id};
    F32Call c{};
    if (p.batch != nullptr) {   // (the count, the call and the rings are requested together: two L2 latencies less in front of the rows.  Through the slot's pointer to its table: 8 streams 219 us against 212, 32 streams 641 against 622)
      const F32StreamPtrs& ptrs = p.batch->ptrs[slot];
      c = p.batch->b.s[slot].call;
      a.in_ring = ptrs.ring[p.layer];
      a.out_ring = p.last_layer ? nullptr : ptrs.ring[p.layer + 1];
      a.save_ring = p.first_layer ? ptrs.ring[p.layer] : nullptr;
      if (slot >= p.batch->b.n) {
        a.T = 0;
        return a;
      }
    } else if (p.call != nullptr) {
      c = *p.call;
    }
    if (p.batch != nullptr || p.call != nullptr) {
      a.rng_id = c.rng_id;
      a.T = c.T * p.rate_in;
      a.pos = c.frames * p.rate_in;
      a.in_direct = p.first_layer ? c.feats : nullptr;
      a.out_direct = p.last_layer ? c.out : nullptr;
    }
    return a;
  };
  static_assert(M == 128 || (M == 64 && !PACK), "frames of a tile");
  constexpr int ROWS = M + TC_H, PLANE = ROWS * 128, PANEL = 3 * PLANE;
  constexpr int ITEMS = (ROWS * 8 + TC_CONV - 1) / TC_CONV;   // 8-channel pieces per thread and panel
  const TcSlot s0 = record(PACK ? 2 * plane : plane);
  TcSlot s1 = s0;
  if (PACK) s1 = record(2 * plane + 1);
  const int m0 = PACK ? 0 : blockIdx.x * M, n0 = blockIdx.y * BN;
  if (PACK ? s0.T <= 0 : m0 >= s0.T) return;   // the grid is sized for the longest chunk

  extern __shared__ __align__(1024) uint8_t tc_smem[];
  constexpr int B_TILE = 3 * BN * 128;
  uint8_t* sA = tc_smem;
  uint8_t* sB = sA + tc.n_a * PANEL;
  uint64_t* full_a = reinterpret_cast<uint64_t*>(sB + tc.n_b * B_TILE);
  uint64_t* empty_a = full_a + TC_MAX_A;
  uint64_t* full_b = empty_a + TC_MAX_A;
  uint64_t* empty_b = full_b + TC_MAX_B;
  uint64_t* accum = empty_b + TC_MAX_B;           // [2]: products of a panel (with TURN: of a tap) done
  uint64_t* drained = accum + 2;                  // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drained + 2);
  int* s_fail = reinterpret_cast<int*>(tmem_slot + 1);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  if ((ptx::smem_u32(tc_smem) & 1023u) != 0u) {   // would corrupt the swizzled tiles: refuse (uniform)
    if (tid == 0) atomicExch(tc.err, 14);
    return;
  }
  // Row numbers in 32-bit arithmetic (a ring index needs only the low bits of the clock; in 64 bits, with its branches, the
  // address of a row cost more instructions than its arithmetic), the element offset widened: frame m0 + i, i possibly negative.
  const int C_in = p.C_in, in_mask = p.in_mask;
  auto in_row = [&](const TcSlot& a, int i) -> const float* {
    const bool direct = a.in_direct != nullptr && i >= 0;
    const uint32_t r = direct ? (uint32_t)i : ((uint32_t)a.pos + (uint32_t)i) & (uint32_t)in_mask;
    return (direct ? a.in_direct : a.in_ring) + (size_t)r * (uint32_t)C_in;
  };
  const int c8 = (tid & 7) * 8, row0 = tid >> 3;          // this thread's pieces: channels c8 .. c8 + 7 of rows row0, row0 + 32, ...
  float4 xa[ITEMS], xb[ITEMS];
  auto load = [&](int u) {
    const int blk = tc.per_tap ? u / p.n_taps : u, tap = tc.per_tap ? u - blk * p.n_taps : 0;
    const int c = blk * 64 + c8;
    const int i0 = m0 - TC_H - (tc.per_tap ? p.shift[tap] : 0);
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const int row = row0 + 32 * i, seg = PACK && i >= TC_SEG / 32 ? TC_SEG : 0;   // (with PACK the tile starts at frame 0)
      const TcSlot& a = seg ? s1 : s0;
      xa[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      xb[i] = xa[i];
      if (row < ROWS && m0 + row - seg - TC_H < a.T && c < C_in && (!PACK || a.T > 0)) {   // (an odd batch's last tile has no second slot)
        const float* src = in_row(a, i0 + row - seg) + c;
        xa[i] = *reinterpret_cast<const float4*>(src);
        if (c + 4 < C_in) xb[i] = *reinterpret_cast<const float4*>(src + 4);
      }
    }
  };
  // The set-up beside the first latency: the converting warps request their rows while another makes the barriers.  (Rows behind the block's barrier: one
  // stream of the vocoder 99.7 us per chunk against 97.5, 8 streams 218 against 212, 32 streams 641 against 622.  The first weights in front of it as well,
  // which only hold the rows up: 99.6, 32 streams 630 against 624, and a layer of few frames slower than without either.)
  if (warp < 8) {
    load(0);
  } else if (warp == 9 && lane == 0) {
#pragma unroll 1
    for (int i = 0; i < TC_MAX_A; ++i) {
      ptx::mbar_init(&full_a[i], TC_CONV);
      ptx::mbar_init(&empty_a[i], 1);
    }
#pragma unroll 1
    for (int i = 0; i < TC_MAX_B; ++i) {
      ptx::mbar_init(&full_b[i], 1);
      ptx::mbar_init(&empty_b[i], 1);
    }
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&accum[i], 1);
      ptx::mbar_init(&drained[i], TC_CONV);
    }
    *s_fail = 0;
    ptx::fence_barrier_init();
  }
  __syncwarp();
  // columns: leading term (see above), then the 2^-8 and the 2^-16 terms
  constexpr bool TURN = BN > 32 && (!DRAIN || M == 64);
  constexpr uint32_t S_COL = TURN ? 2 * BN : (DRAIN ? 6 * BN : 3 * BN);
  constexpr uint32_t TMEM_COLS = S_COL + 2 * BN <= 128 ? 128 : (S_COL + 2 * BN <= 256 ? 256 : 512);
  if (warp == 8) ptx::tmem_alloc(tmem_slot, TMEM_COLS);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  const int n_units = tc.n_blocks * (tc.per_tap ? p.n_taps : 1), taps_u = tc.per_tap ? 1 : p.n_taps;

  if (warp == 9) {
    // ---------------- weight stream: one tile of three planes per (block, tap) ----------------
    const size_t plane = (size_t)tc.C_pad * 128;
    const uint8_t* src = tc.W + (size_t)phase * tc.n_blocks * p.n_taps * 3 * plane + (size_t)n0 * 128;
    const int n = tc.n_blocks * p.n_taps;
    int st = 0;
    uint32_t ph = 1;
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i < n && ok; ++i, src += 3 * plane) {
      if (i >= tc.n_b) ok = tc_wait(&empty_b[st], ph, s_fail, tc.err, 0x201);
      if (ok && ptx::elect_one()) {
        ptx::mbar_expect_tx(&full_b[st], B_TILE);
#pragma unroll 1
        for (int q = 0; q < 3; ++q) ptx::bulk_load(sB + st * B_TILE + q * BN * 128, src + q * plane, BN * 128, &full_b[st]);
      }
      __syncwarp();
      if (++st == tc.n_b) { st = 0; ph ^= 1u; }
    }
  } else if (warp == 8) {
    // ---------------- products ----------------
    // One (panel, tap) after the other; the loop is a chain of one thread's instructions, so addresses advance on 32-bit values and
    // the next barriers are polled ahead of this step's products (with a wait in front of every step it took 1,700 cycles, the
    // products alone 900).
    const uint32_t id2 = ptx::umma_idesc_bf16(M, 2 * BN, 0, 0), id1 = ptx::umma_idesc_bf16(M, BN, 0, 0);
    constexpr uint32_t DESC_HI = (uint32_t)((((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61)) >> 32);
    const uint32_t a_lo = ((ptx::smem_u32(sA) & 0x3FFFF) >> 4) | (1u << 16), b_lo = ((ptx::smem_u32(sB) & 0x3FFFF) >> 4) | (1u << 16);
    const uint32_t bar_b = ptx::smem_u32(full_b), bar_eb = ptx::smem_u32(empty_b), bar_a = ptx::smem_u32(full_a), bar_ea = ptx::smem_u32(empty_a);
    const uint32_t off0 = (uint32_t)(tc.per_tap ? TC_H : TC_H - p.shift[0]) * 8u, off1 = (uint32_t)(TC_H - p.shift[1]) * 8u, off2 = (uint32_t)(TC_H - p.shift[2]) * 8u;
    uint32_t sa = 0, pa = 0, sb = 0, pb = 0;
    bool ok = true, ready_a = ptx::mbar_try_wait_s(bar_a, 0), ready_b = ptx::mbar_try_wait_s(bar_b, 0);
    int u = 0, j = 0, v = 0;                       // panel, its tap, taps so far
#pragma unroll 1
    while (u < n_units && ok) {
      if (j == 0) {
        if (DRAIN && !TURN && u >= 2) ok = tc_wait(&drained[u & 1], ((u >> 1) - 1) & 1, s_fail, tc.err, 0x206);
        if (!__all_sync(0xffffffffu, ready_a)) ok &= tc_wait(&full_a[sa], pa, s_fail, tc.err, 0x202);
      }
      if (TURN && v >= 2) ok &= tc_wait(&drained[v & 1], ((v >> 1) - 1) & 1, s_fail, tc.err, 0x206);
      if (!__all_sync(0xffffffffu, ready_b)) ok &= tc_wait(&full_b[sb], pb, s_fail, tc.err, 0x203);
      if (!ok) break;
      ptx::tc_fence_after();
      const bool last = j + 1 == taps_u, first = u == 0 && j == 0;
      const uint32_t al0 = a_lo + sa * (uint32_t)(PANEL >> 4) + (j == 0 ? off0 : (j == 1 ? off1 : off2)), bl0 = b_lo + sb * (uint32_t)(B_TILE >> 4);
      const uint64_t ah = ((uint64_t)DESC_HI << 32) | al0, am = ah + (PLANE >> 4), al = am + (PLANE >> 4), b = ((uint64_t)DESC_HI << 32) | bl0;
      const uint32_t eb = bar_eb + 8u * sb, ea = bar_ea + 8u * sa, d_main = tmem_base + (uint32_t)(TURN ? v & 1 : (u & 1) * 3 + j) * BN;
      uint64_t* done = &accum[(TURN ? v : u) & 1];
      ++v;
      if (++sb == (uint32_t)tc.n_b) { sb = 0; pb ^= 1u; }
      if (last) {
        if (++sa == (uint32_t)tc.n_a) { sa = 0; pa ^= 1u; }
        ++u;
        j = 0;
        ready_a = u < n_units && ptx::mbar_try_wait_s(bar_a + 8u * sa, pa);
      } else {
        ++j;
      }
      ready_b = u < n_units && ptx::mbar_try_wait_s(bar_b + 8u * sb, pb);
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          ptx::umma_bf16(d_main, ah + 2 * k, b + 2 * k, id1, k != 0);
          ptx::umma_bf16(tmem_base + S_COL, ah + 2 * k, b + (BN * 128 >> 4) + 2 * k, id2, k == 0 ? (uint32_t)!first : 1u);
          ptx::umma_bf16(tmem_base + S_COL, am + 2 * k, b + 2 * k, id2, 1);
          ptx::umma_bf16(tmem_base + S_COL + BN, al + 2 * k, b + 2 * k, id1, 1);
        }
        ptx::umma_commit_s(eb);
        if (last) ptx::umma_commit_s(ea);
        if (TURN || last) ptx::umma_commit(done);
      }
      __syncwarp();
    }
  } else {
    // ---------------- input rows -> bf16 planes ----------------
    const int q = warp & 3, col0 = (warp >> 2) * (BN / 2);   // epilogue: TMEM lane quarter; columns col0 .. col0 + BN / 2 - 1
    const uint32_t lanes = tmem_base + ((uint32_t)(q * 32) << 16);
    constexpr int NC = BN / 32, W = M / 8;                   // a thread's columns: W of each 16
    float sum[NC][W], panel_sum[TURN ? NC : 1][W];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int i = 0; i < W; ++i) sum[c][i] = 0.f;
    auto drain = [&](int u, int j) {                         // panel u (with TURN: the u-th tap, tap j of its panel)
      const bool got = tc_wait(&accum[u & 1], (u >> 1) & 1, s_fail, tc.err, 0x205);
      ptx::tc_fence_after();
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const uint32_t col = lanes + (uint32_t)((u & 1) * (TURN ? 1 : 3) * BN + col0 + 16 * c);
        uint32_t z[2 * W];
        float s[W];
        ptx::tmem_ld_rows_issue<W>(col, z);
        if (TURN || taps_u == 1) {
          ptx::tmem_ld_wait<W>(z);
#pragma unroll
          for (int i = 0; i < W; ++i) s[i] = __uint_as_float(z[i]);
        } else {
          ptx::tmem_ld_rows_issue<W>(col + BN, z + W);
          ptx::tmem_ld_wait<2 * W>(z);
#pragma unroll
          for (int i = 0; i < W; ++i) s[i] = __uint_as_float(z[i]) + __uint_as_float(z[W + i]);
          if (taps_u == 3) {
            ptx::tmem_ld_rows_issue<W>(col + 2 * BN, z);
            ptx::tmem_ld_wait<W>(z);
#pragma unroll
            for (int i = 0; i < W; ++i) s[i] += __uint_as_float(z[i]);
          }
        }
        if (TURN) {                                          // (a panel's taps are added up first, as below)
#pragma unroll
          for (int i = 0; i < W; ++i) panel_sum[c][i] = s[i] = j == 0 ? s[i] : panel_sum[c][i] + s[i];
        }
        if (!TURN || j + 1 == taps_u) {
#pragma unroll
          for (int i = 0; i < W; ++i) sum[c][i] += s[i];
        }
      }
      ptx::tc_fence_before();
      ptx::mbar_arrive(&drained[u & 1]);
      return got;
    };
    int sa = 0;
    uint32_t ph = 1;
    bool ok = true;
#pragma unroll 1
    for (int u = 0; u < n_units; ++u) {
      if (u >= tc.n_a) ok &= tc_wait(&empty_a[sa], ph, s_fail, tc.err, 0x204);
      uint8_t* dst = sA + sa * PANEL;
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const int row = row0 + 32 * i;
        if (row < ROWS) {
          uint4 h, m, l;
          split2(xa[i].x, xa[i].y, h.x, m.x, l.x);
          split2(xa[i].z, xa[i].w, h.y, m.y, l.y);
          split2(xb[i].x, xb[i].y, h.z, m.z, l.z);
          split2(xb[i].z, xb[i].w, h.w, m.w, l.w);
          uint8_t* d = dst + row * 128 + (((tid & 7) ^ (row & 7)) << 4);
          *reinterpret_cast<uint4*>(d) = h;
          *reinterpret_cast<uint4*>(d + PLANE) = m;
          *reinterpret_cast<uint4*>(d + 2 * PLANE) = l;
        }
      }
      ptx::fence_proxy_async_smem();
      ptx::mbar_arrive(&full_a[sa]);
      if (++sa == tc.n_a) { sa = 0; ph ^= 1u; }
      if (u + 1 < n_units) load(u + 1);
      if (DRAIN && u > 0) {
        if (TURN) {
#pragma unroll 1
          for (int j = 0; j < taps_u; ++j) ok &= drain((u - 1) * taps_u + j, j);
        } else {
          ok &= drain(u - 1, 0);
        }
      }
    }

    // Carry update of the first layer: its left context for the next chunk is the tail of the caller's chunk, written into ring
    // rows that no CTA of this launch reads (distinct logical frames map to distinct rows: the ring holds f_chunk + halo frames).
    auto save = [&](const TcSlot& a) {
      const int first = a.T > p.save_rows ? a.T - p.save_rows : 0;
      const int c4 = C_in >> 2;
#pragma unroll 1
      for (int i = tid; i < (a.T - first) * c4; i += TC_CONV) {
        const int r = first + i / c4, c = (i - (i / c4) * c4) * 4;
        const float4 v = *reinterpret_cast<const float4*>(a.in_direct + (long long)r * C_in + c);
        *reinterpret_cast<float4*>(a.save_ring + (long long)((int)((a.pos + r) & (long long)in_mask)) * C_in + c) = v;
      }
    };
    if (p.first_layer && blockIdx.x == 0 && blockIdx.y == 0 && phase == 0) {
      if (s0.save_ring != nullptr) save(s0);
      if (PACK && s1.T > 0) save(s1);
    }

    // ---------------- epilogue ----------------
    // A thread's accumulator row crosses to row-wise order through shared memory (the panel is idle by then), so that a warp reads the
    // residual and writes the result in whole 64- or 128-byte pieces of rows: a thread per row took 32 wavefronts per access, half
    // of the load/store pipe's time.
    constexpr int LPR = BN / 8;                    // lanes that share a row, 4 channels each
    constexpr int LD = BN / 2 + 4;                 // floats between rows of the staging tile (no bank conflicts)
    constexpr int RW = M / 4, NP = RW * LPR / 32;   // rows of a warp; pieces of a thread
    float* stage = reinterpret_cast<float*>(sA) + warp * RW * LD;
    const int g = lane % LPR, rr = lane / LPR, n = n0 + col0 + 4 * g;
    const bool n_ok = n < p.C_out;
    // the warp's slot and its first frame there
    const TcSlot& a = PACK && q >= TC_SEG / 32 ? s1 : s0;
    const int first = m0 + q * RW + rr - (PACK && q >= TC_SEG / 32 ? TC_SEG : 0);
    const bool direct = a.out_direct != nullptr;
    float* const out = direct ? a.out_direct : a.out_ring;
    const uint32_t out0 = direct ? 0u : (uint32_t)(p.n_phase * a.pos), out_mask = direct ? ~0u : (uint32_t)p.out_mask;
    const int T_out = PACK ? min(a.T, TC_SEG) : a.T;
    if (TURN) {
#pragma unroll 1
      for (int j = 0; j + 1 < taps_u; ++j) ok &= drain((n_units - 1) * taps_u + j, j);
    }
    float4 x[NP];                                 // the residual rows, fetched under the products (with TURN half of them: registers)
    auto residual = [&](int i) {
      const int row = first + i * (32 / LPR);
      x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (p.residual_silu && row < T_out && n_ok) x[i] = *reinterpret_cast<const float4*>(in_row(a, row) + n);
    };
    constexpr int X_EARLY = TURN ? NP / 2 : NP;
#pragma unroll
    for (int i = 0; i < X_EARLY; ++i) residual(i);
    const float4 bias = n_ok ? *reinterpret_cast<const float4*>(p.bias + n) : make_float4(0.f, 0.f, 0.f, 0.f);
    ok &= TURN ? drain(n_units * taps_u - 1, taps_u - 1) : drain(n_units - 1, 0);
    ok = ok && *reinterpret_cast<volatile int*>(s_fail) == 0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      uint32_t z[2 * W];
      float z0[W];
      ptx::tmem_ld_rows_issue<W>(lanes + (uint32_t)(S_COL + col0 + 16 * c), z);
      ptx::tmem_ld_rows_issue<W>(lanes + (uint32_t)(S_COL + BN + col0 + 16 * c), z + W);
      ptx::tmem_ld_wait<2 * W>(z);
#pragma unroll
      for (int i = 0; i < W; ++i) z0[i] = sum[c][i] + (__uint_as_float(z[i]) + __uint_as_float(z[W + i]));
      float* d = stage + (M == 64 ? lane & 15 : lane) * LD + 16 * c + (M == 64 ? 8 * (lane >> 4) : 0);
#pragma unroll
      for (int i = 0; i < W / 4; ++i) *reinterpret_cast<float4*>(d + 4 * i) = make_float4(z0[4 * i], z0[4 * i + 1], z0[4 * i + 2], z0[4 * i + 3]);
    }
#pragma unroll
    for (int i = X_EARLY; i < NP; ++i) residual(i);
    __syncwarp();
    // (one pass per step over all of the thread's pieces: the options cost one branch each, and the pieces' latencies overlap)
    float4 v[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      v[i] = *reinterpret_cast<const float4*>(stage + (rr + i * (32 / LPR)) * LD + 4 * g);
      v[i] = make_float4(v[i].x + bias.x, v[i].y + bias.y, v[i].z + bias.z, v[i].w + bias.w);
    }
    if (p.residual_silu) {
#pragma unroll
      for (int i = 0; i < NP; ++i)
        v[i] = make_float4(x[i].x + silu_f(v[i].x), x[i].y + silu_f(v[i].y), x[i].z + silu_f(v[i].z), x[i].w + silu_f(v[i].w));
    }
    if (p.post_silu) {
#pragma unroll
      for (int i = 0; i < NP; ++i) v[i] = make_float4(silu_f(v[i].x), silu_f(v[i].y), silu_f(v[i].z), silu_f(v[i].w));
    }
    if (p.exc_std != 0.f) {   // the stream's clock at this layer's output rate is the generator's offset
#pragma unroll
      for (int i = 0; i < NP; ++i)
        v[i] = excite4(v[i], (long long)p.n_phase * (a.pos + first + i * (32 / LPR)) + phase, n, a.rng_id, p.exc_std, p.exc_seed_lo, p.exc_seed_hi);
    }
    if (n_ok && ok) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int row = first + i * (32 / LPR);
        const uint32_t ro = (out0 + (uint32_t)(p.n_phase * row + phase)) & out_mask;
        if (row < T_out) *reinterpret_cast<float4*>(out + (size_t)ro * (uint32_t)p.C_out + n) = v[i];
      }
    }
    ptx::tc_fence_before();
  }
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(s_fail) != 0) ptx::pause_for_copies();
  if (warp == 8) ptx::tmem_dealloc(tmem_base, TMEM_COLS);
}

// W of (phase, tap), [C_in][C_out] fp32 -> planes of swizzled tiles (see TapConvTc::W).
__global__ void tapconv_pack_kernel(const float* W, long long w_phase_stride, long long w_tap_stride, int C_in, int C_out, int C_pad, int n_blocks, int n_taps,
                                    uint8_t* dst) {
  const int blk = blockIdx.y, tap = blockIdx.z % n_taps, phase = blockIdx.z / n_taps;
  const float* w = W + phase * w_phase_stride + tap * w_tap_stride;
  uint8_t* d = dst + ((size_t)(phase * n_blocks + blk) * n_taps + tap) * 3 * C_pad * 128;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < C_pad * 32; i += gridDim.x * blockDim.x) {
    const int n = i % C_pad, k = 2 * (i / C_pad), c = blk * 64 + k;   // two input channels of one output channel
    const float x = n < C_out && c < C_in ? w[(size_t)c * C_out + n] : 0.f, y = n < C_out && c + 1 < C_in ? w[(size_t)(c + 1) * C_out + n] : 0.f;
    uint32_t s[3];
    split2(x, y, s[0], s[1], s[2]);
    for (int q = 0; q < 3; ++q)
      *reinterpret_cast<uint32_t*>(d + (size_t)q * C_pad * 128 + (size_t)n * 128 + (((k >> 3) ^ (n & 7)) << 4) + (k & 7) * 2) = s[q];
  }
}
