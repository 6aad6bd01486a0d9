// The chunk step as one kernel of clusters for batches of more than two slots per cluster.  Included by dc_flow.cu behind dc_flow_cluster.cuh.
//
// A cluster keeps up to four slots as two tiles of 128 rows (two slots each) and walks them in turn through every stage, so that the hand-over of
// one tile - the epilogue, the rows' way through L2, the other CTAs' arrivals - lies under the products of the others.  With one tile per cluster nothing does:
// a stage of 5,700 cycles has 1,900 of products.  Hence no barrier over the cluster here: a CTA that has stored its columns of a tile arrives at that tile's
// barrier in every CTA, the loaders wait for sixteen arrivals, and all else is local to the CTA.
//   * Weights: a stage's tiles fill the ring once (it holds a whole stage) and are released by the last tile's products.
//   * Activations: a ring of four blocks of 64 channels runs ahead across tiles and stages.
//   * Accumulators: two sets, so that the products of a tile run under the epilogue of the one before.
//   * The residual stream (bf16, the thread's row and columns) waits in tensor memory for the tile's next turn.
// The arithmetic - reduction order, accumulators per issuer, key blocks, rescaling - is that of the other forms: the same bytes.

constexpr int TIL_MAX = 2;                           // tiles of a cluster
// Register split: with the other kernels' 104 the loader spills, and a spilled value comes from L2.
constexpr int TIL_REGS_CTRL = 120, TIL_REGS_EPI = 192;
static_assert(128 * TIL_REGS_CTRL + CLU_EPI * TIL_REGS_EPI == 128 * CLU_REGS_CTRL + CLU_EPI * CLU_REGS_EPI, "the registers that the block is launched with");
constexpr int TIL_RA = 4;                            // activation ring (even: a slot belongs to one issuer)
constexpr int TIL_A = 128 * 128;                     // one block: 128 rows x 64 channels
constexpr int TIL_XCH = TIL_RA * TIL_A;              // the taps' exchange
constexpr int TIL_STG = TIL_XCH + 32 * 1024;         // two staging buffers: a tile's rows of 32 channels and their partial sums of squares
constexpr int TIL_STG_BYTES = 128 * 64 + 2 * 2 * SLOT_ROWS * 4;
constexpr int TIL_HR = TIL_STG + 2 * TIL_STG_BYTES;  // the carried rows on their way: [slot][two halves][8 rows][32 B]
constexpr int TIL_W = CLU_PANEL;                     // weight ring
constexpr int TIL_SX = 48 * 1024;                    // attention: exchange of maxima and sums, behind Q and the P buffers
constexpr int TIL_ACC = 96, TIL_RES = 4 * TIL_ACC;   // TMEM columns: accumulator (set, issuer) at (2 set + issuer) TIL_ACC, then the residuals
static_assert(TIL_HR % 16 == 0 && TIL_HR + 2 * 2 * HALO * 32 <= TIL_W && TIL_W + CLU_RS * CLU_SLOT + CLU_TAIL == (int)CLU_SMEM, "one CTA's shared memory");
static_assert(TIL_RES >= CLU_O_COL + 128 && TIL_RES + 16 * TIL_MAX <= 512, "tensor memory");
static_assert(ATT_Q_BYTES + 2 * ATT_P_BYTES <= TIL_SX && TIL_SX + 1024 <= CLU_PANEL - (int)CLU_KVS * CLU_KV_BYTES, "attention's share");

struct TileSlot {      // what the epilogues need of a slot
  bf16 *halo, *kv;
  int   T, Tc, kv_head, n_prompt0, pass, tau_off;
};
static_assert(8 * (3 * TIL_RA + 2 * CLU_RS + 2 * (int)CLU_KVS + TIL_MAX + 20) + 2 * TIL_MAX * ((int)sizeof(CluJob) + (int)sizeof(TileSlot)) + 8 +
                      4 * (96 + 32 * 2 * TIL_MAX) + 16 <= CLU_TAIL, "barriers and constants");

// The same bounded wait on a barrier that other CTAs of the cluster arrive at: what they stored before is visible behind it.
__device__ __forceinline__ bool clu_wait_cluster(uint64_t* bar, uint32_t parity, int* s_fail, int* err, int code) {
  const uint32_t a = ptx::smem_u32(bar);
#pragma unroll 1
  for (uint32_t i = 0; i < (1u << 20); ++i) {
    if (__all_sync(0xffffffffu, ptx::mbar_try_wait_cluster(a, parity))) return true;
    if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(s_fail) != 0)) return false;
  }
  *reinterpret_cast<volatile int*>(s_fail) = 1;
  atomicCAS(err, 0, code);
  __syncwarp();
  return false;
}

template <bool ROUNDED>
__global__ void __launch_bounds__(CLU_THREADS, 1) flow_tiles_kernel(const __grid_constant__ CluParams p) {
  constexpr int BN = CLU_BN, RS = CLU_RS;
  extern __shared__ __align__(1024) uint8_t clu_smem[];
  uint8_t* aring = clu_smem;
  uint8_t* xch = clu_smem + TIL_XCH;
  uint8_t* wring = clu_smem + TIL_W;
  uint8_t* sQ = clu_smem;
  uint8_t* sP = sQ + ATT_Q_BYTES;
  uint8_t* kvring = clu_smem + CLU_PANEL - CLU_KVS * CLU_KV_BYTES;
  uint64_t* full_a = reinterpret_cast<uint64_t*>(wring + RS * CLU_SLOT);   // [TIL_RA] each
  uint64_t* empty_a = full_a + TIL_RA;
  uint64_t* normed = empty_a + TIL_RA;
  uint64_t* full_w = normed + TIL_RA;    // [RS]
  uint64_t* empty_w = full_w + RS;       // [RS]
  uint64_t* full_kv = empty_w + RS;      // [CLU_KVS]
  uint64_t* empty_kv = full_kv + CLU_KVS;
  uint64_t* ready = empty_kv + CLU_KVS;  // [TIL_MAX]: every CTA has stored its part of the tile's stage
  uint64_t* accum = ready + TIL_MAX;     // [2]
  uint64_t* drained = accum + 2;         // [2]: the epilogue has read the accumulator set
  uint64_t* att_done = drained + 2;
  uint64_t* staged = att_done + 1;       // the epilogue has written its part of an item (of a tile's stage) ...
  uint64_t* stage_free = staged + 2;     // ... and may write the one after the next; [2] each
  uint64_t* bar_q = stage_free + 2;
  uint64_t* bar_s = bar_q + 1;           // [2] each, by stream (key block parity)
  uint64_t* bar_sfree = bar_s + 2;
  uint64_t* bar_p = bar_sfree + 2;
  uint64_t* bar_pv = bar_p + 2;
  CluJob* s_job = reinterpret_cast<CluJob*>(bar_pv + 2);                   // [2 TIL_MAX]
  TileSlot* s_slot = reinterpret_cast<TileSlot*>(s_job + 2 * TIL_MAX);     // [2 TIL_MAX]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_slot + 2 * TIL_MAX);
  int* s_fail = reinterpret_cast<int*>(tmem_slot + 1);
  float* s_bias = reinterpret_cast<float*>(wring + RS * CLU_SLOT + CLU_TAIL - 4 * (96 + 32 * 2 * TIL_MAX));   // [3 BN]
  float* s_tau = s_bias + 96;                              // [slot][32]
  float* s_m = s_tau;                                      // attention: [2][64], references of the streams
  float* s_x = reinterpret_cast<float*>(clu_smem + TIL_SX);   // attention: [2][2][64]
  float* s_rs = s_tau;                                     // norm: the rows' scales, [128] (the ring of keys and values may already land in the exchange's place)

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int rank = (int)ptx::cluster_ctarank();
  const int n0 = rank * BN;
  const int slot0 = (int)(blockIdx.x / (unsigned)p.CL) * p.spc, ns = min(p.spc, p.n_slots - slot0), nt = (ns + 1) >> 1;
  const int nkb_c = p.C / KBLK, nkb_in = p.Kin / KBLK;
  const int n_out = p.mel / 16;
  const int nch_out = rank < n_out ? (n_out - rank + p.CL - 1) / p.CL : 0;

  if ((ptx::smem_u32(clu_smem) & 1023u) != 0u) {   // the swizzled tiles need it (the same for every CTA of the grid)
    if (tid == 0) atomicExch(p.err, 14);
    return;
  }
  if (p.tick) {   // a wavefront pass: a cluster whose slots are all holes has nothing to do
    ptx::pdl_wait();
    bool any = false;
#pragma unroll 1
    for (int i = 0; i < ns; ++i) any |= p.slots[slot0 + i].T > 0;
    if (!any) return;
  }
  if (tid == 0) {
#pragma unroll 1
    for (int i = 0; i < TIL_RA; ++i) {
      ptx::mbar_init(&full_a[i], 1);
      ptx::mbar_init(&empty_a[i], 1);
      ptx::mbar_init(&normed[i], CLU_EPI);
    }
#pragma unroll 1
    for (int i = 0; i < RS; ++i) {
      ptx::mbar_init(&full_w[i], 1);
      ptx::mbar_init(&empty_w[i], 1);
    }
#pragma unroll 1
    for (int i = 0; i < (int)CLU_KVS; ++i) {
      ptx::mbar_init(&full_kv[i], 1);
      ptx::mbar_init(&empty_kv[i], 1);
    }
#pragma unroll 1
    for (int i = 0; i < TIL_MAX; ++i) ptx::mbar_init(&ready[i], (uint32_t)p.CL);
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&accum[i], 2);
      ptx::mbar_init(&drained[i], CLU_EPI);
      ptx::mbar_init(&staged[i], CLU_EPI);
      ptx::mbar_init(&stage_free[i], 1);
      ptx::mbar_init(&bar_s[i], 1);
      ptx::mbar_init(&bar_sfree[i], 128);
      ptx::mbar_init(&bar_p[i], 128);
      ptx::mbar_init(&bar_pv[i], 1);
    }
    ptx::mbar_init(att_done, CLU_EPI);
    ptx::mbar_init(bar_q, 1);
    *s_fail = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 1) ptx::tmem_alloc(tmem_slot, 512);
  if (tid >= 128 && tid < 128 + 2 * TIL_MAX) {       // the slots' table
    ptx::pdl_wait();
    const int i = tid - 128;
    SlotInfo si{};
    if (i < ns) si = p.slots[slot0 + i];
    s_slot[i] = TileSlot{si.halo, si.kv, si.T, si.Tc, si.kv_head, si.n_prompt0, si.pass, si.tau_off};
    CluJob jb;
    jb.kv = si.kv;
    jb.T = si.T;
    jb.k.set(si, p.P, p.Rk);
    s_job[i] = jb;
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  ptx::cluster_arrive();                             // (the other CTAs' barriers exist behind it)
  ptx::cluster_wait();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  auto rows_of = [&](int t) { return 2 * t + 1 < ns ? 128 : 64; };
  auto blocks = [&](int nkb) { return (nkb + 1) & ~1; };   // ring slots of a tile's operand: even, so that a slot belongs to one issuer
  const long long kv_plane = (long long)(p.P + p.Rk) * p.C;
  const int dh = 1 << p.dh_shift;

  if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TIL_REGS_CTRL));
  else asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(TIL_REGS_EPI));

  if (warp == 2) {
    // ---------------- weight stream, and the hand-over of what the epilogue has written ----------------
    // One warp polls for both, so that the epilogue goes on with the next item at once: 1,000 cycles for a fence, 500 for a bulk copy.
    ptx::pdl_wait();
    const uint8_t* src0 = p.wstream + (long long)rank * p.wstream_bytes;
    const uint32_t bar_staged = ptx::smem_u32(staged), bar_e0 = ptx::smem_u32(empty_w);
    CluStage w, hs;                                // stage of the next weight tile; of the next item
    long long off = 0;
    int w_kb = 0, ht = 0, xi = 0;
    uint32_t t = 0, slot = 0, ph = 1, h = 0, spins = 0;
    bool more_w = true;
#pragma unroll 1
    while (more_w || hs.s < p.n_steps) {
      bool did = false;
      if (hs.s < p.n_steps && __all_sync(0xffffffffu, ptx::mbar_test_wait_s(bar_staged + 8u * (h & 1u), (h >> 1) & 1u))) {
        did = true;
        const int rows = rows_of(ht);
        const uint8_t* const stg = clu_smem + TIL_STG + (h & 1u) * TIL_STG_BYTES;
        if (hs.kind == CLU_IN || hs.kind == CLU_CONV || hs.kind == CLU_OPROJ) {
          if (ptx::elect_one()) {
            const bool feeds_norm = (hs.kind == CLU_CONV && hs.j + 1 == p.cpa) || (hs.kind == CLU_OPROJ && hs.g + 1 == p.n_attn);
            bf16* const out = p.X[hs.kind == CLU_IN ? 0 : xi ^ 1];
            ptx::bulk_store(out + (long long)(slot0 + 2 * ht) * nkb_c * CLU_SLOT_KB + (long long)rank * (rows * 32), stg, (uint32_t)rows * 64u);
            if (feeds_norm) {
              float* dst = p.ssq + ((long long)(slot0 + 2 * ht) * (p.C >> 4) + 2 * rank) * SLOT_ROWS;
              const uint8_t* ssq_out = stg + 128 * 64;
              ptx::bulk_store(dst, ssq_out, 512u);
              if (rows == 128) ptx::bulk_store(dst + (long long)(p.C >> 4) * SLOT_ROWS, ssq_out + 512, 512u);
            }
            ptx::bulk_store_wait_read();
            ptx::mbar_arrive(&stage_free[h & 1u]);
            ptx::bulk_store_wait();
          }
          __syncwarp();
          ptx::fence_proxy_async_global();
        } else {
          if (ptx::elect_one()) ptx::mbar_arrive(&stage_free[h & 1u]);
          __syncwarp();
          asm volatile("fence.acq_rel.gpu;" ::: "memory");   // (covers what the epilogue's threads stored before they arrived)
        }
        if (lane < p.CL) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_u32(&ready[ht]), (uint32_t)lane));
        __syncwarp();
        ++h;
        if (++ht == nt) {
          ht = 0;
          if (hs.kind == CLU_IN) xi = 0;
          if (hs.kind == CLU_CONV || hs.kind == CLU_OPROJ) xi ^= 1;
          hs.next(p);
        }
      }
      if (more_w) {
        const int n = w.kind == CLU_ATT || (w.kind == CLU_OUT && nch_out == 0) ? 0 : (w.kind == CLU_IN ? nkb_in : nkb_c);
        if (w_kb >= n) {
          if (w.kind == CLU_OUT) off = 0;
          w.next(p);
          w_kb = 0;
          more_w = w.s < p.n_steps;
          did = true;
        } else if (t < RS || __all_sync(0xffffffffu, ptx::mbar_test_wait_s(bar_e0 + 8u * slot, ph))) {
          const uint32_t bytes = w.kind == CLU_CONV || w.kind == CLU_QKV ? 3u * BN * 128u : (w.kind == CLU_OUT ? (uint32_t)nch_out * 2048u : BN * 128u);
          if (ptx::elect_one()) {
            ptx::mbar_expect_tx(&full_w[slot], bytes);
            ptx::bulk_load(wring + slot * CLU_SLOT, src0 + off, bytes, &full_w[slot]);
          }
          __syncwarp();
          off += bytes;
          ++w_kb;
          ++t;
          if (++slot == RS) { slot = 0; ph ^= 1u; }
          did = true;
        }
      }
      if (did) {
        spins = 0;
      } else {
        if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(s_fail) != 0)) more_w = false;   // (the epilogue runs through to its end)
        if (++spins == (1u << 24)) {
          *reinterpret_cast<volatile int*>(s_fail) = 1;
          atomicCAS(p.err, 0, 0x301);
          break;
        }
      }
    }
  } else if (warp == 0) {
    // ---------------- activations, Q, K/V blocks ----------------
    ptx::pdl_wait();
    int xi = 0;
    uint32_t k = 0;                                // stages so far
    uint32_t ab = 0, as = 0, ap = 1;               // activation blocks so far, ring position
    uint32_t n_g = 0, n_att = 0;                   // GEMM items with products, attention stages so far
    uint32_t it0 = 0, pre = 0;                     // K/V items of earlier jobs; items of the next job already requested
    bool ok = true;
    auto item_fetch = [&](const CluJob& jb, const bf16* planes, int item) {
      bool is_v;
      int b;
      clu_item(item, jb.k.nkb, &is_v, &b);
      const uint32_t gi = it0 + (uint32_t)item, ks = gi % CLU_KVS, use = gi / CLU_KVS;
      if (use > 0 && !clu_wait(&empty_kv[ks], (use - 1) & 1u, s_fail, p.err, 0x302)) return false;
      uint8_t* dst = kvring + ks * CLU_KV_BYTES;
      const int n = min(ATT_KB, jb.k.L - b * ATT_KB);   // key rows of this block
      if (is_v && n < ATT_KB) {                    // rows behind the last key must be finite up to the next UMMA step
        const int n16 = min(ATT_KB, (n + 15) & ~15);
#pragma unroll 1
        for (int i = lane; i < (n16 - n) << (p.dh_shift - 3); i += 32) *reinterpret_cast<uint4*>(dst + n * 2 * dh + i * 16) = make_uint4(0u, 0u, 0u, 0u);
        ptx::fence_proxy_async_smem();
        __syncwarp();
      }
      if (ptx::elect_one()) jb.k.fetch(planes + (is_v ? kv_plane : 0), b, n, p.P, p.Rk, p.dh_shift, dst, &full_kv[ks]);
      __syncwarp();
      return true;
    };
#pragma unroll 1
    for (CluStage st; st.s < p.n_steps && ok; st.next(p), ++k) {
      if (st.kind != CLU_ATT) {
        const bool skip = st.kind == CLU_OUT && nch_out == 0;
        const int nkb = st.kind == CLU_IN ? nkb_in : nkb_c;
        if (!skip) {
          if (st.kind == CLU_OPROJ) ok = clu_wait(att_done, (n_att - 1) & 1u, s_fail, p.err, 0x303);   // (attention works in the ring's memory)
          const bf16* x = st.kind == CLU_IN ? p.Ain : (st.kind == CLU_OPROJ ? p.O : p.X[xi]);
#pragma unroll 1
          for (int t = 0; t < nt && ok; ++t) {
            if (k > 0 && !(ok = clu_wait_cluster(&ready[t], (k - 1) & 1u, s_fail, p.err, 0x304))) break;
            ptx::fence_proxy_async_global();
            const int rows = rows_of(t);
            const bf16* src = x + (long long)(slot0 + 2 * t) * nkb * CLU_SLOT_KB;
#pragma unroll 1
            for (int kb = 0; kb < blocks(nkb); ++kb) {
              if (ab >= TIL_RA && !(ok = clu_wait(&empty_a[as], ap, s_fail, p.err, 0x305))) break;
              if (ptx::elect_one()) {
                uint8_t* dst = aring + as * TIL_A;
                if (kb >= nkb) {
                  ptx::mbar_arrive(&full_a[as]);
                } else if (st.kind == CLU_IN) {    // (from another kernel: a slot's blocks are its own)
                  ptx::mbar_expect_tx(&full_a[as], (uint32_t)rows * 128u);
                  ptx::bulk_load(dst, src + kb * CLU_SLOT_KB, 8192u, &full_a[as]);
                  if (rows == 128) ptx::bulk_load(dst + 8192, src + (nkb + kb) * CLU_SLOT_KB, 8192u, &full_a[as]);
                } else {
                  ptx::mbar_expect_tx(&full_a[as], (uint32_t)rows * 128u);
                  ptx::bulk_load(dst, src + (long long)kb * rows * 64, (uint32_t)rows * 128u, &full_a[as]);
                }
              }
              __syncwarp();
              ++ab;
              if (++as == TIL_RA) { as = 0; ap ^= 1u; }
            }
          }
          n_g += (uint32_t)nt;
        } else {
          // (every stage's phase is waited for: a parity cannot tell a phase from the one before the last)
#pragma unroll 1
          for (int t = 0; t < nt && ok; ++t) ok = clu_wait_cluster(&ready[t], (k - 1) & 1u, s_fail, p.err, 0x31c);
        }
        if (st.kind == CLU_IN) xi = 0;
        if (st.kind == CLU_CONV || st.kind == CLU_OPROJ) xi ^= 1;
        if (st.kind == CLU_QKV && ok) {
          // once the stage's products are done, the ring's memory is attention's: the carried blocks of the first job
          ok = clu_wait(&accum[(n_g - 1) & 1u], ((n_g - 1) >> 1) & 1u, s_fail, p.err, 0x306);
          const int jl = rank;
          if (ok && jl < min(ns, 2) * p.n_heads) {
            const CluJob jb = s_job[jl / p.n_heads];
            const bf16* planes = jb.kv + (long long)(st.s * p.n_attn + st.g) * 2 * kv_plane + (long long)(jl % p.n_heads) * p.kv_hs;
            pre = 0;
            if (jb.T > 0) {
              int item = 0;
#pragma unroll 1
              for (; item < 2 * jb.k.nkb && item < (int)CLU_KVS && ok; ++item) {
                bool is_v;
                int b;
                clu_item(item, jb.k.nkb, &is_v, &b);
                if (b >= jb.k.n_early) break;
                ok = item_fetch(jb, planes, item);
              }
              pre = (uint32_t)item;
              if (ptx::elect_one()) {
#pragma unroll 1
                for (; item < 2 * jb.k.nkb; ++item) {
                  bool is_v;
                  int b;
                  clu_item(item, jb.k.nkb, &is_v, &b);
                  if (b < jb.k.n_early) jb.k.prefetch(planes + (is_v ? kv_plane : 0), b, p.P, p.Rk, p.dh_shift);
                }
              }
              __syncwarp();
            }
          }
        }
      } else {
        bool first = true;
        uint32_t last_k = 0;
#pragma unroll 1
        for (int t = 0; t < nt && ok; ++t) {
          if (!(ok = clu_wait_cluster(&ready[t], (k - 1) & 1u, s_fail, p.err, 0x307))) break;
          ptx::fence_proxy_async_global();
#pragma unroll 1
          for (int jl = rank; jl < (rows_of(t) >> 6) * p.n_heads && ok; jl += p.CL) {
            const int sl = 2 * t + jl / p.n_heads, head = jl % p.n_heads;
            const CluJob jb = s_job[sl];
            if (jb.T == 0) continue;
            // the previous job's scores are done when its last K slot is released
            if (!first && !(ok = clu_wait(&empty_kv[last_k % CLU_KVS], (last_k / CLU_KVS) & 1u, s_fail, p.err, 0x308))) break;
            if (ptx::elect_one()) {
              const bf16* src = p.Q + ((long long)(slot0 + sl) * nkb_c + (head << p.dh_shift >> 6)) * CLU_SLOT_KB + HALO * 64;
              ptx::mbar_expect_tx(bar_q, 2u * (SLOT_ROWS - HALO) * 128u);
              ptx::bulk_load(sQ, src, (SLOT_ROWS - HALO) * 128u, bar_q);
              ptx::bulk_load(sQ + 8192, src, (SLOT_ROWS - HALO) * 128u, bar_q);
            }
            __syncwarp();
            const bf16* planes = jb.kv + (long long)(st.s * p.n_attn + st.g) * 2 * kv_plane + (long long)head * p.kv_hs;
#pragma unroll 1
            for (int item = first ? (int)pre : 0; item < 2 * jb.k.nkb && ok; ++item) ok = item_fetch(jb, planes, item);
            last_k = it0 + (uint32_t)clu_item_k(jb.k.nkb - 1);
            it0 += 2u * (uint32_t)jb.k.nkb;
            first = false;
          }
        }
        pre = 0;
        ++n_att;
      }
    }
  } else if (warp < 4) {
    // ---------------- warps 1, 3: UMMA issuers (attention: scores, P V) ----------------
    const int me = warp >> 1;
    uint32_t ab = 0, wt = 0, n_g = 0;              // activation blocks and weight tiles of earlier items / stages; items
    uint32_t it0 = 0, n_q = 0, n_s0 = 0, n_s1 = 0;
    uint32_t norm_ph = 0;                          // bit s: parity of the next normalised block in ring slot s
    bool ok = true;
#pragma unroll 1
    for (CluStage st; st.s < p.n_steps && ok; st.next(p)) {
      if (st.kind != CLU_ATT) {
        const bool skip = st.kind == CLU_OUT && nch_out == 0;
        if (skip) continue;
        const int nkb = st.kind == CLU_IN ? nkb_in : nkb_c;
        const bool norm = ROUNDED && (st.kind == CLU_QKV || st.kind == CLU_OUT);
        const int N = st.kind == CLU_CONV || st.kind == CLU_QKV ? 3 * BN : (st.kind == CLU_OUT ? 16 * nch_out : BN);
        const uint32_t idesc = ptx::umma_idesc_bf16(TILE_M, N, 0, 0);
        constexpr uint32_t HI128 = (uint32_t)((((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61)) >> 32);
        constexpr uint32_t HI64 = (uint32_t)((((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)4 << 61)) >> 32);
        const uint32_t a_hi = st.kind == CLU_IN ? HI128 : HI64;
        const uint32_t a_lo0 = ((ptx::smem_u32(aring) & 0x3FFFF) >> 4) | (1u << 16), w_lo = ((ptx::smem_u32(wring) & 0x3FFFF) >> 4) | (1u << 16);
#pragma unroll 1
        for (int t = 0; t < nt && ok; ++t, ++n_g) {
          const uint32_t a_k2 = st.kind == CLU_IN ? 4u : (uint32_t)(rows_of(t) * 64) >> 4;
          const uint32_t d_acc = tmem_base + (2u * (n_g & 1u) + (uint32_t)me) * TIL_ACC;
          if (n_g >= 2) ok = clu_wait(&drained[n_g & 1u], ((n_g >> 1) - 1) & 1u, s_fail, p.err, 0x309);
          uint32_t as = (ab + (uint32_t)me) % TIL_RA, ap = ((ab + (uint32_t)me) / TIL_RA) & 1u;
          uint32_t ws = (wt + (uint32_t)me) % RS, wp = ((wt + (uint32_t)me) / RS) & 1u, acc = 0;
          ptx::tc_fence_after();
#pragma unroll 1
          for (int kb = me; kb < blocks(nkb) && ok; kb += 2) {
            if (kb < nkb) ok = clu_wait(&full_w[ws], wp, s_fail, p.err, 0x30a);
            if (norm) {
              ok = ok && clu_wait(&normed[as], (norm_ph >> as) & 1u, s_fail, p.err, 0x30b);
              norm_ph ^= 1u << as;
            } else {
              ok = ok && clu_wait(&full_a[as], ap, s_fail, p.err, 0x30c);
            }
            if (!ok) break;
            ptx::tc_fence_after();
            const uint32_t a_lo = a_lo0 + as * (uint32_t)(TIL_A >> 4);
            const uint64_t da = ((uint64_t)a_hi << 32) | a_lo, da2 = ((uint64_t)a_hi << 32) | (a_lo + a_k2), db = ((uint64_t)HI128 << 32) | (w_lo + ws * (uint32_t)(CLU_SLOT >> 4));
            if (ptx::elect_one()) {
              if (kb < nkb) {
                ptx::umma_bf16(d_acc, da, db, idesc, acc);
                ptx::umma_bf16(d_acc, da + 2, db + 2, idesc, 1);
                ptx::umma_bf16(d_acc, da2, db + 4, idesc, 1);
                ptx::umma_bf16(d_acc, da2 + 2, db + 6, idesc, 1);
                if (t + 1 == nt) ptx::umma_commit(&empty_w[ws]);
              }
              ptx::umma_commit(&empty_a[as]);
            }
            __syncwarp();
            acc = 1;
            as += 2;
            if (as >= TIL_RA) { as -= TIL_RA; ap ^= 1u; }
            ws += 2;
            if (ws >= RS) { ws -= RS; wp ^= 1u; }
          }
          if (ptx::elect_one()) ptx::umma_commit(&accum[n_g & 1u]);   // (an issuer without products arrives at once)
          __syncwarp();
          ab += (uint32_t)blocks(nkb);
        }
        wt += (uint32_t)nkb;
      } else if (warp == 1) {
        // ---- scores ----
        const uint32_t idesc_s = ptx::umma_idesc_bf16(128, ATT_KB, 0, 0);
        auto kv_desc = [&](uint32_t ks) { return p.dh_shift == 6 ? att_kv_desc<64>(ptx::smem_u32(kvring + ks * CLU_KV_BYTES)) : att_kv_desc<32>(ptx::smem_u32(kvring + ks * CLU_KV_BYTES)); };
        // the scores take the accumulators' place
        ok = clu_wait(&drained[(n_g - 1) & 1u], ((n_g - 1) >> 1) & 1u, s_fail, p.err, 0x30d);
        if (n_g >= 2) ok = ok && clu_wait(&drained[n_g & 1u], ((n_g >> 1) - 1) & 1u, s_fail, p.err, 0x30e);
#pragma unroll 1
        for (int t = 0; t < nt && ok; ++t) {
#pragma unroll 1
          for (int jl = rank; jl < (rows_of(t) >> 6) * p.n_heads && ok; jl += p.CL) {
            const int sl = 2 * t + jl / p.n_heads, head = jl % p.n_heads, nkb = s_job[sl].k.nkb;
            if (s_job[sl].T == 0) continue;
            const uint64_t dq = ptx::umma_desc_sw128(ptx::smem_u32(sQ)) + (uint64_t)(((head << p.dh_shift) & 63) >> 3);
#pragma unroll 1
            for (int b = 0; b < nkb && ok; ++b) {
              const int w = b & 1;
              const uint32_t gi = it0 + (uint32_t)clu_item_k(b), ks = gi % CLU_KVS;
              ok = clu_wait(&full_kv[ks], (gi / CLU_KVS) & 1u, s_fail, p.err, 0x30f);
              if (b == 0) ok = ok && clu_wait(bar_q, n_q++ & 1u, s_fail, p.err, 0x310);
              const uint32_t n = w ? n_s1++ : n_s0++;
              if (n > 0) ok = ok && clu_wait(&bar_sfree[w], (n - 1) & 1u, s_fail, p.err, 0x311);
              if (!ok) break;
              ptx::tc_fence_after();
              const uint64_t dk = kv_desc(ks);
              const uint32_t d_s = tmem_base + (uint32_t)w * ATT_KB;
              if (ptx::elect_one()) {
                ptx::umma_bf16(d_s, dq, dk, idesc_s, 0);
                ptx::umma_bf16(d_s, dq + 2, dk + 2, idesc_s, 1);
                if (p.dh_shift == 6) {
                  ptx::umma_bf16(d_s, dq + 4, dk + 4, idesc_s, 1);
                  ptx::umma_bf16(d_s, dq + 6, dk + 6, idesc_s, 1);
                }
                ptx::umma_commit(&bar_s[w]);
                ptx::umma_commit(&empty_kv[ks]);
              }
              __syncwarp();
            }
            it0 += 2u * (uint32_t)nkb;
          }
        }
      } else {
        // ---- O_w += P(b) V(b) ----
        const uint32_t idesc_pv = ptx::umma_idesc_bf16(128, dh, 0, 1);   // B = V, MN-major
        const uint64_t dp = ptx::umma_desc_sw128(ptx::smem_u32(sP));
        auto kv_desc = [&](uint32_t ks) { return p.dh_shift == 6 ? att_kv_desc<64>(ptx::smem_u32(kvring + ks * CLU_KV_BYTES)) : att_kv_desc<32>(ptx::smem_u32(kvring + ks * CLU_KV_BYTES)); };
        const uint32_t v_step = 2u << p.dh_shift;
#pragma unroll 1
        for (int t = 0; t < nt && ok; ++t) {
#pragma unroll 1
          for (int jl = rank; jl < (rows_of(t) >> 6) * p.n_heads && ok; jl += p.CL) {
            const int sl = 2 * t + jl / p.n_heads, L = s_job[sl].k.L, nkb = s_job[sl].k.nkb;
            if (s_job[sl].T == 0) continue;
#pragma unroll 1
            for (int b = 0; b < nkb && ok; ++b) {
              const int w = b & 1;
              const uint32_t gi = it0 + (uint32_t)clu_item_v(b, nkb), vs = gi % CLU_KVS;
              ok = clu_wait(&full_kv[vs], (gi / CLU_KVS) & 1u, s_fail, p.err, 0x312);
              ok = ok && clu_wait(&bar_p[w], (w ? n_s1++ : n_s0++) & 1u, s_fail, p.err, 0x313);
              if (!ok) break;
              ptx::tc_fence_after();
              const uint64_t dpb = dp + (uint64_t)(w * (ATT_P_BYTES >> 4)), dv = kv_desc(vs);
              const uint32_t d_o = tmem_base + CLU_O_COL + (uint32_t)w * 64u;
              const int ksteps = min(ATT_KB / 16, (L - b * ATT_KB + 15) >> 4);
              if (ptx::elect_one()) {
#pragma unroll
                for (int i = 0; i < ATT_KB / 16; ++i)
                  if (i < ksteps)
                    ptx::umma_bf16(d_o, dpb + (uint64_t)((i >> 2) * (8192 >> 4) + (i & 3) * 2), dv + (uint64_t)((uint32_t)i * v_step), idesc_pv, (b >> 1 | i) != 0);
                ptx::umma_commit(&bar_pv[w]);
                ptx::umma_commit(&empty_kv[vs]);
              }
              __syncwarp();
            }
            it0 += 2u * (uint32_t)nkb;
          }
        }
      }
    }
  } else {
    // ---------------- epilogue: a thread owns one row of every tile and 16 columns; attention: warps 4..7 even, 8..11 odd key blocks ----------------
    ptx::pdl_wait();
    const int et = tid - 128;
    const int q = warp & 3, cg = (warp - 4) >> 2;
    const int row_t = q * 32 + lane, rho = row_t & 63, f = rho - HALO;
    const int c0 = 16 * cg;
    uint8_t* const hr = clu_smem + TIL_HR + (((row_t >> 6) * 2 + cg) * HALO + (rho & 7)) * 32;   // a left-context thread's carried row
    const uint32_t lanes = tmem_base + ((uint32_t)(q * 32) << 16);
    const int aq = q & 1, ah = q >> 1;              // softmax: query quarter, key half
    uint32_t k = 0, n_g = 0, n_blk = 0;             // stages, GEMM items, key blocks of this thread's stream so far
    uint32_t ab = 0;                                // activation blocks of earlier items (rounded norm)
    int xi = 0;

    uint32_t h = 0;                                 // items so far
    // The item before the last has left (so all threads are done with that one).
    auto free_wait = [&]() {
      if (h > 1) clu_wait(&stage_free[h & 1u], ((h >> 1) - 1) & 1u, s_fail, p.err, 0x31d);
    };
    auto hand_over = [&]() {
      ptx::mbar_arrive(&staged[h & 1u]);
      ++h;
    };
    // A stage's constants: requested a stage ahead, into registers.
    float cb = 0.f, ct = 0.f;
    auto request_consts = [&](const CluStage& s) {
      if (s.kind == CLU_ATT || s.s >= p.n_steps) return;
      const int gbase = p.C + s.g * (p.cpa + 4) * p.C;     // biases in blob order: input, then per group conv..., Q, K, V, O
      if (s.kind == CLU_OUT) {
        if (et < 16 * nch_out) cb = p.fc[p.o_bout + (rank + (et >> 4) * p.CL) * 16 + (et & 15)];
      } else {
        const int ob = s.kind == CLU_IN ? 0 : (s.kind == CLU_CONV ? gbase + s.j * p.C : gbase + (p.cpa + (s.kind == CLU_OPROJ ? 3 : 0)) * p.C);
        if (et < (s.kind == CLU_QKV ? 3 * BN : BN)) cb = p.fc[ob + (et / BN) * p.C + n0 + et % BN];
      }
      if (s.kind == CLU_CONV && et < ns * BN) ct = p.fc[p.o_tau + (s.s * p.n_conv + s.l) * p.C + s_slot[et / BN].tau_off + n0 + et % BN];
    };
    request_consts(CluStage());

#pragma unroll 1
    for (CluStage st; st.s < p.n_steps; st.next(p), ++k) {
      CluStage nx = st;
      nx.next(p);
      if (st.kind == CLU_ATT) {
        request_consts(nx);
#pragma unroll 1
        for (int t = 0; t < nt; ++t) {
          clu_wait(&ready[t], (k - 1) & 1u, s_fail, p.err, 0x31a);   // (an arrival of this stage must not count for the one before)
#pragma unroll 1
          for (int jl = rank; jl < (rows_of(t) >> 6) * p.n_heads; jl += p.CL) {
            const int sl = 2 * t + jl / p.n_heads, head = jl % p.n_heads;
            const CluJob jb = s_job[sl];
            if (jb.T == 0) continue;
            const int nkb = jb.k.nkb;
            const int row = aq * 32 + lane, w = cg;
            float* sx = s_x + w * 128;
            float m_ref = -INFINITY, lsum = 0.f;
            bool ok = true;
#pragma unroll 1
            for (int b = w; b < nkb; b += 2, ++n_blk) {
              ok &= clu_wait(&bar_s[w], n_blk & 1u, s_fail, p.err, 0x314);
              ptx::tc_fence_after();
              float v[64];
              ptx::tmem_ld64(lanes + (uint32_t)(w * ATT_KB + ah * 64), v);
              ptx::tc_fence_before();
              ptx::mbar_arrive(&bar_sfree[w]);
              const int col0 = b * ATT_KB + ah * 64;
              float mx = att_mask_max(v, jb.k.L - col0, jb.k.g0 - col0, jb.k.g1 - col0);
              sx[ah * 64 + row] = mx * p.scale_log2e;
              ptx::named_bar_sync(4 + w, 128);
              mx = fmaxf(sx[row], sx[64 + row]);
              ptx::named_bar_sync(4 + w, 128);
              if (b >= 2) ok &= clu_wait(&bar_pv[w], (n_blk - 1) & 1u, s_fail, p.err, 0x315);
              if (b < 2) {
                m_ref = mx;
              } else {
                const bool need = mx > m_ref + ATT_RESCALE_LOG2;
                if (__any_sync(0xffffffffu, need)) {
                  ptx::tc_fence_after();
                  const float alpha = need ? exp2f(m_ref - mx) : 1.0f;
                  if (need) m_ref = mx;
                  lsum *= alpha;
                  if (ah == 0) att_rescale(lanes + (uint32_t)(CLU_O_COL + w * 64), alpha, dh);
                  ptx::tc_fence_before();
                }
              }
              lsum += att_exp_store(v, p.scale_log2e, m_ref, sP + w * ATT_P_BYTES + ah * 8192 + row * 128, row);
              ptx::fence_proxy_async_smem();
              ptx::tc_fence_before();
              ptx::mbar_arrive(&bar_p[w]);
            }
            sx[ah * 64 + row] = lsum;
            if (ah == 0) s_m[w * 64 + row] = m_ref;
            if (w < nkb) ok &= clu_wait(&bar_pv[w], (n_blk - 1) & 1u, s_fail, p.err, 0x316);
            ptx::named_bar_sync(1, CLU_EPI);
            ptx::tc_fence_after();
            ok = ok && *reinterpret_cast<volatile int*>(s_fail) == 0;
            if (ah == 0) {                           // O rows 0..63 live in lanes 0..63; each group of warps stores half of the columns
              float w0, w1;
              att_combine(nkb, s_m[row], s_x[row] + s_x[64 + row], s_m[64 + row], s_x[128 + row] + s_x[192 + row], &w0, &w1);
              const int rows = rows_of(t), orow = (sl & 1) * 64 + HALO + row, perm = (orow >> 1) & 3;
              bf16* oblk = p.O + (long long)(slot0 + 2 * t) * nkb_c * CLU_SLOT_KB + orow * 32;
#pragma unroll 1
              for (int c = w * (dh >> 1); c < (w + 1) * (dh >> 1); c += 16) {
                float o16[16], q16[16];
                ptx::tmem_ld16x2(lanes + (uint32_t)(CLU_O_COL + c), lanes + (uint32_t)(CLU_O_COL + 64 + c), o16, q16);
                if (row < jb.T && ok) {
#pragma unroll
                  for (int i = 0; i < 16; ++i) o16[i] = nkb > 1 ? fmaf(q16[i], w1, o16[i] * w0) : o16[i] * w0;
                  uint4 a, b;
                  pack16_bf16(o16, a, b);
                  const int ch = (head << p.dh_shift) + c;
                  store16(oblk + (long long)(ch >> 5) * (rows * 32) + ((((ch & 31) >> 3) ^ perm) & ~1) * 8, (perm & 1) ? b : a, (perm & 1) ? a : b);
                }
              }
            }
            ptx::tc_fence_before();
            ptx::named_bar_sync(1, CLU_EPI);         // (the next job overwrites the exchange and the accumulators)
          }
          free_wait();
          hand_over();
        }
        ptx::mbar_arrive(att_done);
        continue;
      }

      const int kind = st.kind, nkb = kind == CLU_IN ? nkb_in : nkb_c;
      const bool skip = kind == CLU_OUT && nch_out == 0;
      const bool two_iss = nkb >= 2;
      const bool next_conv = kind == CLU_IN || (kind == CLU_CONV && st.j + 1 < p.cpa) || (kind == CLU_OPROJ && st.g + 1 < p.n_attn);
      const int l_next = kind == CLU_CONV ? st.l + 1 : (kind == CLU_OPROJ ? st.l : 0);
      const bool feeds_norm = (kind == CLU_CONV && st.j + 1 == p.cpa) || (kind == CLU_OPROJ && st.g + 1 == p.n_attn);
      const bool norm = (kind == CLU_QKV || kind == CLU_OUT) && !skip;
      const int d = kind == CLU_CONV ? p.dil[st.l] : 0;
      ptx::named_bar_sync(1, CLU_EPI);               // everybody has read the last stage's constants
      if (et < 3 * BN) s_bias[et] = cb;
      if (kind == CLU_CONV && et < ns * BN) s_tau[et] = ct;
      request_consts(nx);

#pragma unroll 1
      for (int t = 0; t < nt; ++t) {
        const TileSlot& si = s_slot[2 * t + (row_t >> 6)];
        const int slot = slot0 + 2 * t + (row_t >> 6), T = si.T, new_row = rho - si.Tc;
        const bool in_range = T > 0, halo_row = in_range && rho < HALO, chunk_row = in_range && f >= 0 && f < T;
        const bool moves = (halo_row || chunk_row) && new_row >= 0 && new_row < HALO;
        bf16* const carry = next_conv && in_range ? si.halo + ((long long)st.s * p.n_conv + l_next) * HALO * p.C : nullptr;
        const int rows = rows_of(t);

        // ---- what does not depend on the accumulator, under the main loop ----
        uint32_t xr[8];                              // the residual stream: this thread's row and columns
        float rs = 1.f;
        if (norm) {
          // partial sums of squares of the row, 16 channels each, added in chunk order: the first half by the threads of the first 16 columns, the second by the others
          clu_wait(&ready[t], (k - 1) & 1u, s_fail, p.err, 0x317);
          const float* src = p.ssq + ((long long)slot * (p.C >> 4) + cg * (p.C >> 5)) * SLOT_ROWS + rho;
          float part[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) part[j] = chunk_row && j < p.C >> 5 ? __ldcg(src + j * SLOT_ROWS) : 0.f;
          float ss = 0.f;
          if (cg == 0) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (j < p.C >> 5) ss += part[j];
            s_rs[row_t] = ss;
          }
          ptx::named_bar_sync(1, CLU_EPI);
          if (cg == 1) {
            ss = s_rs[row_t];
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (j < p.C >> 5) ss += part[j];
            rs = rsqrtf(ss * p.inv_C + p.eps);
            s_rs[row_t] = ROUNDED && !chunk_row ? -1.f : rs;   // (-1: a row that stays as it is)
          }
        } else {
          if (carry != nullptr && halo_row) {          // (from memory, 1,000 cycles and more: nobody waits for it here)
            cp_async16(hr, carry + rho * p.C + n0 + c0);
            cp_async16(hr + 16, carry + rho * p.C + n0 + c0 + 8);
          }
          if (kind == CLU_CONV || kind == CLU_OPROJ) ptx::tmem_ld8_issue(lanes + (uint32_t)(TIL_RES + 16 * t + 8 * cg), xr);
        }
        free_wait();
        if (t == 0 || norm) ptx::named_bar_sync(1, CLU_EPI);   // constants (and the rows' scales) are in place
        if (norm) rs = s_rs[row_t];
        if (ROUNDED && norm) {
          const int half = rows == 64;
          float kk[4];
          kk[0] = s_rs[et >> 2];
          kk[1] = half ? kk[0] : s_rs[64 + (et >> 2)];
          kk[2] = half ? -1.f : kk[0];
          kk[3] = half ? -1.f : kk[1];
#pragma unroll 1
          for (int kb = 0; kb < nkb; ++kb) {
            const uint32_t a = ab + (uint32_t)kb, as = a % TIL_RA;
            clu_wait(&full_a[as], (a / TIL_RA) & 1u, s_fail, p.err, 0x318);
            uint4* px = reinterpret_cast<uint4*>(aring + as * TIL_A) + et;
            uint4 x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (i < 2 || !half) x[i] = px[256 * i];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (i < 2 || !half) {
                const uint32_t w[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
                uint32_t o[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(w[j] << 16) * kk[i], __uint_as_float(w[j] & 0xFFFF0000u) * kk[i]);
                  o[j] = *reinterpret_cast<const uint32_t*>(&b2);
                }
                if (!(kk[i] < 0.f)) px[256 * i] = make_uint4(o[0], o[1], o[2], o[3]);
              }
            }
            ptx::fence_proxy_async_smem();
            ptx::mbar_arrive(&normed[as]);
          }
          rs = 1.f;
        }
        bool got = true;
        const uint32_t acc0 = 2u * (n_g & 1u) * TIL_ACC, acc1 = acc0 + TIL_ACC;
        if (!skip) got = clu_wait(&accum[n_g & 1u], (n_g >> 1) & 1u, s_fail, p.err, 0x319);
        else clu_wait(&ready[t], (k - 1) & 1u, s_fail, p.err, 0x31b);   // (no products that would have waited)
        ptx::tc_fence_after();
        if (kind == CLU_CONV || kind == CLU_OPROJ) ptx::tmem_ld_wait<8>(xr);
        const bool ok = got && *reinterpret_cast<volatile int*>(s_fail) == 0;
        const bool is_chunk = chunk_row && ok;
        auto load_pair = [&](uint32_t col, float* v) {  // even blocks + odd blocks, always in this order
          if (two_iss) {
            uint32_t z[32];
            ptx::tmem_ld_rows_issue<16>(lanes + acc0 + col, z);
            ptx::tmem_ld_rows_issue<16>(lanes + acc1 + col, z + 16);
            ptx::tmem_ld_wait<32>(z);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(z[i]) + __uint_as_float(z[16 + i]);
          } else {
            ptx::tmem_ld16(lanes + acc0 + col, v);
          }
        };
        auto release = [&]() {                         // the accumulators have been read
          ptx::tc_fence_before();
          ptx::mbar_arrive(&drained[n_g & 1u]);
        };

        if (kind == CLU_OUT) {
#pragma unroll 1
          for (int kc = cg; kc < nch_out; kc += 2) {
            const int n = (rank + kc * p.CL) * 16;
            float acc[16];
            load_pair((uint32_t)(16 * kc), acc);
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = fmaf(acc[i], rs, s_bias[16 * kc + i]);
            if (p.cfg_w > 0.f) {
              // guided step: rows 64.. are the unconditional pass; they hand their velocity over through shared memory
              float4* xv4 = reinterpret_cast<float4*>(xch) + kc * 256;
              if (q >= 2) {
#pragma unroll
                for (int j = 0; j < 4; ++j) xv4[j * 64 + (q - 2) * 32 + lane] = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
              }
              ptx::named_bar_sync(2 + cg, 128);
              if (q < 2) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float4 u = xv4[j * 64 + q * 32 + lane];
                  acc[4 * j] = fmaf(1.f + p.cfg_w, acc[4 * j], -p.cfg_w * u.x);
                  acc[4 * j + 1] = fmaf(1.f + p.cfg_w, acc[4 * j + 1], -p.cfg_w * u.y);
                  acc[4 * j + 2] = fmaf(1.f + p.cfg_w, acc[4 * j + 2], -p.cfg_w * u.z);
                  acc[4 * j + 3] = fmaf(1.f + p.cfg_w, acc[4 * j + 3], -p.cfg_w * u.w);
                }
              }
            }
            if (is_chunk && si.pass == 0) {
              float* xs = p.xstate + ((long long)slot * SLOT_ROWS + rho) * p.mel + n;
              float xv[16];
#pragma unroll
              for (int i = 0; i < 16; i += 4) {
                const float4 x4 = *reinterpret_cast<const float4*>(xs + i);
                xv[i] = x4.x; xv[i + 1] = x4.y; xv[i + 2] = x4.z; xv[i + 3] = x4.w;
              }
#pragma unroll
              for (int i = 0; i < 16; ++i) xv[i] = xv[i] + acc[i] * p.inv_n;
#pragma unroll
              for (int i = 0; i < 16; i += 4) *reinterpret_cast<float4*>(xs + i) = make_float4(xv[i], xv[i + 1], xv[i + 2], xv[i + 3]);
              uint4 a, b;
              pack16_bf16(xv, a, b);
              bf16* blk = p.Ain + ((long long)slot * nkb_in + (n >> 6)) * CLU_SLOT_KB;
              clu_store16(blk, rho, n & 63, a, b);
              if (p.cfg_w > 0.f) clu_store16(blk + (long long)nkb_in * CLU_SLOT_KB, rho, n & 63, a, b);   // the unconditional pass starts from the same x
              const SlotInfo& so = p.slots[slot];      // (read again: only here, once per chunk)
              if ((p.tick ? (so.flags & SLOT_LAST) != 0 : st.s == p.n_steps - 1) && f < so.Tc) {
                float* o = so.out + (long long)f * p.mel + n;
#pragma unroll
                for (int i = 0; i < 16; i += 4) *reinterpret_cast<float4*>(o + i) = make_float4(xv[i], xv[i + 1], xv[i + 2], xv[i + 3]);
              }
            }
          }
          if (!skip) release();
          hand_over();
        } else if (kind == CLU_QKV) {
          const long long kv_off = ((long long)st.s * p.n_attn + st.g) * 2 * kv_plane;
          const int col = n0 + c0, hh = col >> p.dh_shift, wi = col - (hh << p.dh_shift);
          const int tp = min(T, p.P - si.n_prompt0);   // the chunk's first tp frames complete the prompt
          int kv_row = si.n_prompt0 + f;               // K/V plane row of this thread's frame
          if (f >= tp) {
            kv_row = si.kv_head + f - tp;
            if (kv_row >= p.Rk) kv_row -= p.Rk;
            kv_row += p.P;
          }
          const int perm = kv_perm(kv_row, p.dh_shift);
          bf16* kvp = si.kv + kv_off + (long long)hh * p.kv_hs + ((long long)kv_row << p.dh_shift) + ((((wi >> 3) ^ perm) & ~1) << 3);
#pragma unroll
          for (int which = 0; which < 3; ++which) {
            float acc[16];
            load_pair((uint32_t)(which * BN + c0), acc);
            if (which == 2) release();
            const float4* bias4 = reinterpret_cast<const float4*>(s_bias + which * BN + c0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 b4 = bias4[i];
              acc[4 * i] = fmaf(acc[4 * i], rs, b4.x);
              acc[4 * i + 1] = fmaf(acc[4 * i + 1], rs, b4.y);
              acc[4 * i + 2] = fmaf(acc[4 * i + 2], rs, b4.z);
              acc[4 * i + 3] = fmaf(acc[4 * i + 3], rs, b4.w);
            }
            uint4 a, b;
            pack16_bf16(acc, a, b);
            if (is_chunk) {
              if (which == 0) clu_store16(p.Q + ((long long)slot * nkb_c + (col >> 6)) * CLU_SLOT_KB, rho, col & 63, a, b);
              else store16(kvp + (which - 1) * kv_plane, (perm & 1) ? b : a, (perm & 1) ? a : b);
            }
          }
          hand_over();
        } else {
          // ---- a new residual row: input projection, conv block, attention output projection ----
          float2 acc[8];
          if (kind == CLU_CONV) {
            // y[r] = Z_0[r - 2 d] + Z_1[r - d] + Z_2[r]: rows change lanes through shared memory
            float2 z[8], z2[8];
            const uint32_t col = lanes + (uint32_t)c0;
            auto sum = [&](const uint32_t* s, float2* v) {
#pragma unroll
              for (int i = 0; i < 8; ++i) v[i] = add2(pair2(s[2 * i], s[2 * i + 1]), pair2(s[16 + 2 * i], s[17 + 2 * i]));
            };
            uint32_t ra[32], rb[32];
            ptx::tmem_ld_rows_issue<16>(col + acc0, ra);
            ptx::tmem_ld_rows_issue<16>(col + acc1, ra + 16);
            ptx::tmem_ld_rows_issue<16>(col + acc0 + BN, rb);
            ptx::tmem_ld_rows_issue<16>(col + acc1 + BN, rb + 16);
            ptx::tmem_ld_wait<32>(ra);
            ptx::tmem_ld_wait<32>(rb);
            sum(ra, acc);
            sum(rb, z);
            ptx::tmem_ld_rows_issue<16>(col + acc0 + 2 * BN, ra);
            ptx::tmem_ld_rows_issue<16>(col + acc1 + 2 * BN, ra + 16);
            float4* xz = reinterpret_cast<float4*>(xch) + cg * (2 * 4 * TILE_M);
            if (t > 0) ptx::named_bar_sync(2 + cg, 128);   // (the tile before has read its rows)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              xz[j * TILE_M + row_t] = make_float4(acc[2 * j].x, acc[2 * j].y, acc[2 * j + 1].x, acc[2 * j + 1].y);
              xz[(4 + j) * TILE_M + row_t] = make_float4(z[2 * j].x, z[2 * j].y, z[2 * j + 1].x, z[2 * j + 1].y);
            }
            ptx::tmem_ld_wait<32>(ra);
            sum(ra, z2);
            release();
            asm volatile("cp.async.wait_all;" ::: "memory");   // (the carried rows have been read behind the barrier: they are overwritten below)
            ptx::named_bar_sync(2 + cg, 128);
            const int r0 = max(row_t - 2 * d, 0), r1 = max(row_t - d, 0);
            const float4* bias4 = reinterpret_cast<const float4*>(s_bias + c0);
            const float4* tau4 = reinterpret_cast<const float4*>(s_tau + (2 * t + (row_t >> 6)) * BN + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 a0 = xz[j * TILE_M + r0], a1 = xz[(4 + j) * TILE_M + r1], b4 = bias4[j], t4 = tau4[j];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const float2 q0 = h ? make_float2(a0.z, a0.w) : make_float2(a0.x, a0.y), q1 = h ? make_float2(a1.z, a1.w) : make_float2(a1.x, a1.y);
                const float2 bb = h ? make_float2(b4.z, b4.w) : make_float2(b4.x, b4.y), tt = h ? make_float2(t4.z, t4.w) : make_float2(t4.x, t4.y);
                const int i = 2 * j + h;
                const float2 y = add2(add2(add2(add2(q0, q1), z2[i]), bb), tt);
                acc[i] = add2(unpack2(xr[i]), silu2(y));
              }
            }
          } else {
            load_pair((uint32_t)c0, reinterpret_cast<float*>(acc));
            release();
            const float4* bias4 = reinterpret_cast<const float4*>(s_bias + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 b4 = bias4[j];
              acc[2 * j] = add2(acc[2 * j], make_float2(b4.x, b4.y));
              acc[2 * j + 1] = add2(acc[2 * j + 1], make_float2(b4.z, b4.w));
            }
            if (kind == CLU_OPROJ) {
#pragma unroll
              for (int i = 0; i < 8; ++i) acc[i] = add2(acc[i], unpack2(xr[i]));
            }
          }
          uint32_t w[8];
          pack_row<16>(reinterpret_cast<const float*>(acc), w);
          ptx::tmem_st8(lanes + (uint32_t)(TIL_RES + 16 * t + 8 * cg), w);
          uint4 va = make_uint4(w[0], w[1], w[2], w[3]), vb = make_uint4(w[4], w[5], w[6], w[7]);
          if (rho < HALO) {                            // a left-context row hands the carried row on
            if (kind != CLU_CONV) asm volatile("cp.async.wait_all;" ::: "memory");
            va = *reinterpret_cast<const uint4*>(hr);
            vb = *reinterpret_cast<const uint4*>(hr + 16);
          }
          uint8_t* const stg = clu_smem + TIL_STG + (h & 1u) * TIL_STG_BYTES;
          bf16* const rows_out = reinterpret_cast<bf16*>(stg);
          float* const ssq_out = reinterpret_cast<float*>(stg + 128 * 64);   // [slot][2][SLOT_ROWS]
          *reinterpret_cast<uint4*>(rows_out + clu_at32(row_t, c0)) = va;
          *reinterpret_cast<uint4*>(rows_out + clu_at32(row_t, c0 + 8)) = vb;
          if (feeds_norm) {                            // sum of squares of the 16 stored values, fixed order
            float ss = 0.f;
            if (is_chunk) {
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xFFFF0000u);
                ss = fmaf(lo, lo, ss);
                ss = fmaf(hi, hi, ss);
              }
            }
            ssq_out[(row_t >> 6) * 128 + cg * SLOT_ROWS + rho] = ss;
          }
          ptx::fence_proxy_async_smem();
          hand_over();
          // shift the carry by the committed frames: nobody in this launch reads it again
          if (kind != CLU_CONV) ptx::named_bar_sync(1, CLU_EPI);   // (every carried row has been read)
          if (carry != nullptr && moves && ok) store16(carry + new_row * p.C + n0 + c0, va, vb);
        }
        if (!skip) {
          ++n_g;
          ab += (uint32_t)blocks(nkb);
        }
      }
      if (kind == CLU_IN) xi = 0;
      if (kind == CLU_CONV || kind == CLU_OPROJ) xi ^= 1;
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(s_fail) != 0) ptx::pause_for_copies();
  ptx::cluster_arrive();                             // (no CTA leaves before the others' last arrivals at its barriers)
  ptx::cluster_wait();
  if (warp == 1) ptx::tmem_dealloc(tmem_base, 512);
}
