// The whole chunk step of the flow decoder (every Euler step, every layer) as ONE kernel, for batches whose slots fit the
// thread-block clusters that the GPU keeps resident.  Included by dc_flow.cu inside its anonymous namespace.
//
// A stage of the network (one GEMM, or attention) for a few slots is far too little work to fill the GPU; what it costs as
// a kernel of its own is latency: launch boundary, set-up, the wait for the whole previous grid, the first operand tiles
// through L2.  Here a cluster of CL CTAs keeps one or two slots (64 or 128 rows) for the whole step: CTA r owns the columns
// [32 r, 32 r + 32) of every layer, the activations pass from stage to stage through L2, and the hardware cluster barrier and
// signals from CTA to CTA stand where the launch boundary was.
//   * Measured for the hand-over alone (16 CTAs write 4 KB each, everybody reads the 64 KB; cycles until it is released / the
//     first operand block has landed / all of them): bulk copies and signals (clu_arrive_bulk) 950 / 1,500 / 2,020, thread stores
//     and a fence (clu_arrive_release) 1,380 / 1,940 / 2,460; through global counters instead of the barrier 3,460 / 4,940 /
//     5,660; pushed through distributed shared memory 3,760 for all (17 bytes per cycle and SM).
//   * Weights do not depend on the activations: one warp streams the CTA's share of every layer (packed at create in the
//     order and the shared-memory image in which it is consumed) through a ring that runs up to RS reduction blocks ahead,
//     across stage and step boundaries.
//   * The residual stays in the registers of the thread that computes it (a thread keeps its row and columns throughout).
// The arithmetic - reduction order, accumulators per issuer, key blocks, rescaling - is that of the stand-alone kernels, so
// that results do not depend on which of the two a batch size takes.

constexpr int CLU_THREADS = 384;     // warps: 0 activations / K/V loader, 1 and 3 UMMA issuers, 2 weight stream, 4..11 epilogue / softmax
constexpr int CLU_EPI = 256;
// Register split: the 227 KB of shared memory leave no L1 to speak of, so a spilled value comes from L2; the control warps hand
// registers over.  128 x 104 + 256 x 200 = 384 x 168, which the host checks.
constexpr int CLU_REGS_CTRL = 104, CLU_REGS_EPI = 200;
constexpr int CLU_PANEL = 128 * 1024;                // activations [block][64 spc rows][128 B] (hidden <= 512); attention: Q, two P buffers, K/V ring
constexpr int CLU_KV_BYTES = ATT_KB * 128;           // one K or V block
constexpr int CLU_ACC2 = 256;                        // TMEM column of the odd issuer's accumulator
constexpr int CLU_O_COL = 256;                       // attention: S of even / odd blocks at columns 0 / 128, O of the two streams at 256 / 320
constexpr int CLU_TAIL = 3072;                       // barriers and constants behind the rings
constexpr int CLU_CONST_FLOATS = 3 * 64 + 128 + 256;

// 32 columns per CTA.  (64 columns, i.e. clusters half as large and twice as many resident, were slower than the kernels of their
// own wherever 32 do not fit: 16 streams 1,822 us against 1,667.)
constexpr int CLU_BN = 32;
constexpr int CLU_SLOT = 3 * CLU_BN * 128;           // bytes of the largest weight tile (three taps / Q, K, V)
// Weight ring: the tiles of a whole stage, so that a stage's last products do not wait for slots that its first ones free, 1,000 cycles of
// latency later.  (Six slots: 2,325 cycles from a conv stage's first product to its last one's end, eight: 2,000.  One stream 916 -> 895 us per
// chunk, seven 960 -> 911, fourteen 1,097 -> 1,032.)  Even: within a stage a ring slot belongs to one issuer.
constexpr int CLU_RS = 8;
constexpr size_t CLU_SMEM = (size_t)CLU_PANEL + CLU_RS * CLU_SLOT + CLU_TAIL;
static_assert(CLU_SMEM <= 227 * 1024, "one CTA's shared memory");

struct CluParams {
  const SlotInfo* slots;
  int             n_slots;             // slots of the launch
  int             CL;                  // CTAs of a cluster
  int             C, mel, Kin, n_heads;
  int             n_conv, n_attn, cpa, n_steps;
  int             tick;                // one pass, every slot at the Euler step of its table entry (wavefront)
  int             dil[DC_MAX_CONV];
  const float*    fc;                  // biases and the timestep-bias table, in blob order
  int             o_bout, o_tau;
  const uint8_t*  wstream;             // [CL] streams of wstream_bytes
  long long       wstream_bytes;
  bf16 *          X[2], *O;            // activations between GEMMs, blocks of 32 channels (clu_at32): [cluster][C / 32][rows of its slots][32]
  bf16 *          Q, *Ain;             // queries, input of the network: blocks of 64 channels (clu_row16): [slot][C or Kin / 64][64 rows][64]
  float*          xstate;
  float*          ssq;                 // [slot][C / 16][SLOT_ROWS] partial sums of squares of the rows that feed an RMS norm
  float           inv_C, eps, inv_n, cfg_w;
  int             P, Rk, kv_hs, dh_shift;
  float           scale_log2e;
  int*            err;
};

enum CluKind { CLU_IN = 0, CLU_CONV = 1, CLU_QKV = 2, CLU_ATT = 3, CLU_OPROJ = 4, CLU_OUT = 5 };

// Every role walks the same sequence of stages.
struct CluStage {
  int kind = CLU_IN, s = 0, l = 0, g = 0, j = 0;
  __device__ __forceinline__ void next(const CluParams& p) {
    switch (kind) {
      case CLU_IN: kind = CLU_CONV; l = 0; g = 0; j = 0; break;
      case CLU_CONV: ++l; if (++j == p.cpa) kind = p.n_attn > 0 ? CLU_QKV : CLU_OUT; break;
      case CLU_QKV: kind = CLU_ATT; break;
      case CLU_ATT: kind = CLU_OPROJ; break;
      case CLU_OPROJ: if (++g < p.n_attn) { kind = CLU_CONV; j = 0; } else kind = CLU_OUT; break;
      default: kind = CLU_IN; ++s; break;
    }
  }
};

// A row's 16-byte chunks lie in global memory where the swizzled shared-memory tile has them, so that a block of a slot is one untiled bulk copy (no tensor
// map to fetch: 800 cycles less until the first tile is there): in blocks of 64 channels chunk c of a row at c ^ (row & 7), in blocks of 32 at c ^ ((row >> 1) & 3).
constexpr int CLU_SLOT_KB = SLOT_ROWS * KBLK;
__device__ __forceinline__ int clu_row16(int rho, int c) { return rho * KBLK + ((((c >> 3) ^ (rho & 7)) & ~1) << 3); }   // the 32 bytes of columns c .. c + 15
template <int NC>
__device__ __forceinline__ void pack_row(const float* v, uint32_t* w) {
#pragma unroll
  for (int i = 0; i < NC / 2; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
}

// The stage's stores become visible to the cluster, then the epilogue's threads arrive: a barrier among them and ONE warp's fence,
// which covers what the others wrote before the barrier; their arrivals need not wait for it.  (A fence in each of the eight warps took
// 1,600 cycles of a conv stage's 7,060: one stream 1,017 -> 968 us.  The release form of the arrive costs 1,600 behind a store in flight.)
__device__ __forceinline__ void clu_arrive_release(int warp) {
  ptx::named_bar_sync(1, CLU_EPI);
  if (warp == 4) asm volatile("fence.acq_rel.gpu;" ::: "memory");
  ptx::cluster_arrive_relaxed();
}

// A stage's rows leave the CTA as one piece, [64 or 128 rows][32 channels] (clu_at32), which one thread copies out of shared memory in bulk, and a signal to every
// CTA of the cluster tells that they are there.  What orders the rows in front of the other CTAs' reads: the copying thread waits for its copies to
// complete, which makes their writes visible to it; behind that its warp stores one word into every CTA with st.async, whose complete-tx on the CTA's `hand`
// barrier has release semantics at cluster scope; who reads the rows or the row statistics has waited on `hand` with acquire at cluster scope.  The cluster
// barrier, whose arrivals are relaxed here, orders no rows: it tells that the buffers are free again.
// Measured for the hand-over alone (16 CTAs, 4 KB each, cycles from the staging until it is released / until the first operand block is there): behind thread stores and a
// fence 1,385 / 1,945, the copies with a fence behind them 1,670 / 2,228, with the signals 948 / 1,500, with nothing but the relaxed barrier, which orders nothing,
// 828 / 1,387.  One stream 764 us per chunk at the time, 747 now (thread stores and a fence 801, a fence behind the copies 829, the relaxed barrier alone 743), hidden 256 289 (298, -,
// 275), fourteen streams 944 (990, -, 931).  The request of the next operand behind the cluster barrier AND the signals: 771, hidden 256 286, fourteen 949.
__device__ __forceinline__ int clu_at32(int rho, int c) { return rho * 32 + (((c >> 3) ^ ((rho >> 1) & 3)) << 3); }   // element of channel c of a block: the 64-byte swizzle
struct CluPiece {
  void*       dst;
  const void* src;
  uint32_t    bytes;
};
template <int N>
__device__ __forceinline__ void clu_arrive_bulk(int warp, int lane, const CluPiece (&piece)[N], uint32_t hand, uint32_t word, int CL) {
  ptx::fence_proxy_async_smem();
  ptx::named_bar_sync(1, CLU_EPI);
  if (warp == 4) {
    const uint32_t to = lane < CL ? lane : 0, bar_to = ptx::map_to_cta(hand, to), word_to = ptx::map_to_cta(word, to);
    if (ptx::elect_one()) {
#pragma unroll
      for (int i = 0; i < N; ++i)
        if (piece[i].bytes > 0) ptx::bulk_store(piece[i].dst, piece[i].src, piece[i].bytes);
      ptx::bulk_store_wait();
    }
    __syncwarp();
    ptx::fence_proxy_async_global();
    if (lane < CL) ptx::st_async(word_to, 0u, bar_to);
    __syncwarp();
  }
  ptx::cluster_arrive_relaxed();
}

// Bounded wait of a whole warp that gives up at once after any wait of this CTA has given up: the step then runs through without
// waiting, the copying warps request nothing more, and the CTA pauses before it exits.  The vote keeps the warp together: lanes that leave a polling loop one by one go on as separate groups, and everything
// up to the next warp-wide instruction is then executed several times (an issue loop took 600 cycles per block instead of 260).
template <bool CLUSTER = false>   // phases that other CTAs complete: acquire at cluster scope
__device__ __forceinline__ bool clu_wait(uint64_t* bar, uint32_t parity, int* s_fail, int* err, int code) {
  const uint32_t a = ptx::smem_u32(bar);
#pragma unroll 1
  for (uint32_t i = 0; i < (1u << 20); ++i) {
    if (__all_sync(0xffffffffu, CLUSTER ? ptx::mbar_try_wait_cluster_s(a, parity) : ptx::mbar_try_wait_s(a, parity))) return true;
    if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(s_fail) != 0)) return false;
  }
  *reinterpret_cast<volatile int*>(s_fail) = 1;
  atomicCAS(err, 0, code);
  __syncwarp();
  return false;
}

struct CluJob {     // what the heads of a slot attend
  const bf16* kv;
  int         T;
  AttKeys     k;
};

static_assert(8 * (16 + 2 * CLU_RS + 3 * (int)CLU_KVS + 12) + 2 * (int)sizeof(CluJob) + 12 + 4 * CLU_CONST_FLOATS <= CLU_TAIL, "barriers and constants");

// RING (a wavefront pass): fewer clusters than slots, the live slots are those from slot slots[0].first_live on, circularly.  (An instantiation of its
// own: with the choice at run time every other call was 2 to 5 us slower.)
// ROUNDED (DC_OPT_ROUNDED_NORM): the normalised activations are rounded to bf16 before the GEMM that reads them.  (As a choice at run time its code, which
// grew with the rewrite by all threads, cost the models without it 2 % and hidden 64, the shortest stages, 4 %: one stream 854 us against 837, fourteen
// 975 against 956, hidden 64 260 against 249.)
// SPC: slots per cluster.  With one slot the products have 64 rows, which tensor memory holds in sixteen lanes of each quarter: all eight epilogue warps
// have rows and a thread has 8 columns of one (lane l of a quarter: row l & 15, columns 8 (l >> 4) ..), where products of 128 rows leave the warps of
// the upper quarters idle and give the others 16 - and an epilogue is a chain of instructions, five cycles each.  The products get shorter, too: 48.5
// cycles for 64 x 96 x 16 against 56.5 for 128 x 96 x 16.  One stream 862 -> 801 us per chunk, hidden 256 317 -> 298, seven streams 872 -> 813, prompt and
// look-ahead 832 -> 762; the same bytes.
template <bool RING, bool ROUNDED, int SPC>
__global__ void __launch_bounds__(CLU_THREADS, 1) flow_cluster_kernel(const __grid_constant__ CluParams p) {
  constexpr int BN = CLU_BN, RS = CLU_RS;
  constexpr bool ONE = SPC == 1;
  constexpr int NC = ONE ? 8 : 16;         // columns of a thread's row piece
  constexpr int ROWS = SLOT_ROWS * SPC;    // rows of a GEMM stage's products
  extern __shared__ __align__(1024) uint8_t clu_smem[];
  uint8_t* panel = clu_smem;
  uint8_t* wring = panel + CLU_PANEL;
  // attention's share of the panel.  With one slot per cluster the activations take only its first half, and the K/V ring has
  // the other half to itself: the carried key blocks of the next attention stage are fetched stages ahead.
  constexpr int kb_bytes = SPC * 8192;
  uint8_t* sQ = panel;
  uint8_t* sP = sQ + ATT_Q_BYTES;
  uint8_t* kvring = panel + CLU_PANEL - CLU_KVS * CLU_KV_BYTES;
  uint64_t* full_a = reinterpret_cast<uint64_t*>(wring + RS * CLU_SLOT);   // [8]
  uint64_t* normed = full_a + 8;         // [8]
  uint64_t* full_w = normed + 8;         // [RS]
  uint64_t* empty_w = full_w + RS;       // [RS]
  uint64_t* full_kv = empty_w + RS;      // [2 CLU_KVS]: clu_kv_full
  uint64_t* empty_kv = full_kv + 2 * CLU_KVS;
  uint64_t* accum = empty_kv + CLU_KVS;
  uint64_t* bar_q = accum + 1;
  uint64_t* bar_s = bar_q + 1;           // [2] each, by stream (key block parity)
  uint64_t* bar_sfree = bar_s + 2;
  uint64_t* bar_p = bar_sfree + 2;
  uint64_t* bar_pv = bar_p + 2;
  uint64_t* hand = bar_pv + 2;           // [2], in turn: a stage's rows of every CTA of the cluster are there
  CluJob* s_job = reinterpret_cast<CluJob*>(hand + 2);                    // [2], one per slot
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_job + 2);
  int* s_fail = reinterpret_cast<int*>(tmem_slot + 1);
  uint32_t* s_word = tmem_slot + 2;      // what the signals store: nobody reads it
  float* s_bias = reinterpret_cast<float*>(wring + RS * CLU_SLOT + CLU_TAIL - 4 * CLU_CONST_FLOATS);   // [3 BN], 16-byte aligned
  float* s_tau = s_bias + 3 * 64;                          // [2][64]
  float* s_x = s_tau + 128;                                // [2][2][64]: per stream, exchange between the column halves
  float* s_m = s_tau;                                      // attention: [2][64], references of the streams

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (known to be the same for the whole warp)
  const int rank = (int)ptx::cluster_ctarank();
  const int n0 = rank * BN;
  int slot_0 = (int)(blockIdx.x / (unsigned)p.CL) * SPC;
  if (RING) {
    ptx::pdl_wait();
    slot_0 += p.slots[0].first_live;
    if (slot_0 >= p.n_slots) slot_0 -= p.n_slots;
  }
  const int slot0 = slot_0, m0 = slot0 * SLOT_ROWS;
  const int nkb_c = p.C / KBLK, nkb_in = p.Kin / KBLK;
  const int n_out = p.mel / 16;
  const int nch_out = rank < n_out ? (n_out - rank + p.CL - 1) / p.CL : 0;   // 16-column chunks rank, rank + CL, ... of the output projection

  if ((ptx::smem_u32(clu_smem) & 1023u) != 0u) {   // the swizzled tiles need it (the same for every CTA of the grid)
    if (tid == 0) atomicExch(p.err, 14);
    return;
  }
  if (p.tick) {   // a wavefront pass: a cluster whose slots are all holes has nothing to do
    ptx::pdl_wait();
    bool any = false;
#pragma unroll 1
    for (int i = 0; i < SPC; ++i) any |= slot0 + i < p.n_slots && p.slots[slot0 + i].T > 0;
    if (!any) return;
  }
  if (tid == 0) {
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
      ptx::mbar_init(&full_a[i], 1);
      ptx::mbar_init(&normed[i], CLU_EPI);
    }
#pragma unroll 1
    for (int i = 0; i < RS; ++i) {
      ptx::mbar_init(&full_w[i], 1);
      ptx::mbar_init(&empty_w[i], 1);
    }
#pragma unroll 1
    for (int i = 0; i < (int)CLU_KVS; ++i) {
      ptx::mbar_init(&full_kv[clu_kv_full(false, i)], 1);
      ptx::mbar_init(&full_kv[clu_kv_full(true, i)], 1);
      ptx::mbar_init(&empty_kv[i], 1);
    }
    ptx::mbar_init(accum, 2);
    ptx::mbar_init(bar_q, 1);
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&bar_s[i], 1);
      ptx::mbar_init(&bar_sfree[i], 128);
      ptx::mbar_init(&bar_p[i], 128);
      ptx::mbar_init(&bar_pv[i], 1);
      ptx::mbar_init(&hand[i], 1);
    }
    *s_fail = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 1) ptx::tmem_alloc(tmem_slot, 512);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  ptx::cluster_arrive_relaxed();         // (the other CTAs signal on this one's barriers; fence_barrier_init is the release)
  ptx::cluster_wait();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  auto issuers = [&](int nkb) { return nkb >= 2 ? 2 : 1; };
  // Descriptor of K/V slot ks.  With two slots per cluster made anew for every block: fourteen streams 995 -> 938 us against one made in front of the loop and
  // advanced, which keeps it out of the uniform registers that a product takes it from; with one slot 745 -> 751.
  auto kv_base = [&](uint32_t a) { return p.dh_shift == 6 ? att_kv_desc<64>(a) : att_kv_desc<32>(a); };
  auto kv_desc = [&](uint64_t first, uint32_t ks) { return ONE ? first + (uint64_t)(ks * (CLU_KV_BYTES >> 4)) : kv_base(ptx::smem_u32(kvring + ks * CLU_KV_BYTES)); };
  const int n_jobs = SPC * p.n_heads;            // (slot, head) pairs of the cluster; CTA r takes r, r + CL, ...
  const bool one_job = ONE || n_jobs <= p.CL;    // at most one of a CTA: its rows leave in bulk
  auto in_bulk = [&](int kind) { return kind == CLU_ATT ? one_job : kind != CLU_QKV && kind != CLU_OUT; };
  const long long kv_plane = (long long)(p.P + p.Rk) * p.C;
  const int dh = 1 << p.dh_shift;

  if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(CLU_REGS_CTRL));
  else asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(CLU_REGS_EPI));

  if (warp == 2) {
    // ---------------- weight stream ----------------
    const uint8_t* src0 = p.wstream + (long long)rank * p.wstream_bytes;
    CluStage w;                                    // stage of the next tile to request
    int w_kb = 0;
    long long off = 0;
    uint32_t t = 0, end = 0, slot = 0, ph = 1;     // tiles requested; tiles of all stages up to the current one; ring position
    auto tiles = [&](int kind) { return kind == CLU_ATT || (kind == CLU_OUT && nch_out == 0) ? 0 : (kind == CLU_IN ? nkb_in : nkb_c); };
#pragma unroll 1
    for (CluStage st; st.s < p.n_steps; st.next(p)) {
      end += (uint32_t)tiles(st.kind);
      // as far as RS tiles behind this stage's: their ring slots are free at the latest when this stage's products are done
#pragma unroll 1
      while (t < end + RS && w.s < p.n_steps) {
        if (w_kb >= tiles(w.kind)) {
          if (w.kind == CLU_OUT) off = 0;
          w.next(p);
          w_kb = 0;
          continue;
        }
        const uint32_t bytes = w.kind == CLU_CONV || w.kind == CLU_QKV ? 3u * BN * 128u : (w.kind == CLU_OUT ? (uint32_t)nch_out * 2048u : BN * 128u);
        if (t >= RS && !clu_wait(&empty_w[slot], ph, s_fail, p.err, 0x101)) break;
        if (ptx::elect_one()) {
          ptx::mbar_expect_tx(&full_w[slot], bytes);
          ptx::bulk_load(wring + slot * CLU_SLOT, src0 + off, bytes, &full_w[slot]);
        }
        __syncwarp();
        off += bytes;
        ++w_kb;
        ++t;
        if (++slot == RS) { slot = 0; ph ^= 1u; }
      }
      ptx::cluster_arrive_relaxed();
      ptx::cluster_wait();
    }
  } else if (warp < 4) {
    // ---------------- warp 0: activation panel, Q, K/V blocks; warps 1, 3: UMMA issuers (attention: scores, P V) ----------------
    ptx::pdl_wait();
    const int me = warp >> 1;                      // issuer 0 or 1
    int xi = 0;                                    // X[xi] holds the residual stream
    uint32_t n_g = 0, n_gc = 0, n_gi = 0, n_norm = 0;   // GEMM stages so far: all, on hidden channels, input projections, normalised ones
    uint32_t wt = 0;                               // weight tiles of earlier stages
    uint32_t it0 = 0, pre = 0, n_q = 0;            // K/V items of earlier jobs; items of the next job already requested; Q tiles so far
    uint32_t n_s0 = 0, n_s1 = 0;                   // key blocks of the two streams in earlier jobs
    CluKvPhases kv_phases;                         // warp 1: of the K barriers, warp 3: of the V barriers
    uint32_t n_hand = 0;                           // warp 0: stages whose rows left in bulk so far
    const bool two = !ONE && slot0 + 1 < p.n_slots;   // (an odd batch's last cluster has one slot: the other's rows are anything)
    // (the input projection's operand comes from another kernel: a slot's blocks are its own)
    auto request = [&](const bf16* src, int nkb, bool in) {
      ptx::fence_proxy_async_global();
      if (ptx::elect_one()) {
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb) {
          ptx::mbar_expect_tx(&full_a[kb], two ? 16384u : 8192u);
          if (!ONE && in) {
            ptx::bulk_load(panel + kb * kb_bytes, src + kb * CLU_SLOT_KB, 8192u, &full_a[kb]);
            if (two) ptx::bulk_load(panel + kb * kb_bytes + 8192, src + (nkb + kb) * CLU_SLOT_KB, 8192u, &full_a[kb]);
          } else {
            ptx::bulk_load(panel + kb * kb_bytes, src + kb * (two ? 2 : 1) * CLU_SLOT_KB, two ? 16384u : 8192u, &full_a[kb]);
          }
        }
      }
      __syncwarp();
    };
    if (warp == 0) request(p.Ain + (long long)slot0 * nkb_in * CLU_SLOT_KB, nkb_in, true);
#pragma unroll 1
    for (CluStage st; st.s < p.n_steps; st.next(p)) {
      bool fetch = false;
      if (st.kind != CLU_ATT) {
        const int nkb = st.kind == CLU_IN ? nkb_in : nkb_c;
        const bool skip = st.kind == CLU_OUT && nch_out == 0;   // no output columns for this CTA
        if (skip || warp == 0) {
        } else {
          const int n_iss = issuers(nkb);
          const bool norm = ROUNDED && (st.kind == CLU_QKV || st.kind == CLU_OUT);
          if (me < n_iss) {
            const int N = st.kind == CLU_CONV || st.kind == CLU_QKV ? 3 * BN : (st.kind == CLU_OUT ? 16 * nch_out : BN);
            const uint32_t idesc = ptx::umma_idesc_bf16(ROWS, N, 0, 0);
            const uint32_t d_acc = tmem_base + (uint32_t)me * CLU_ACC2;
            // The loop is a chain of instructions of one thread, and every address it has to make costs as much as a product: ring
            // slot, phases and descriptors advance incrementally on 32-bit values, and the next block's barriers are polled ahead
            // of this block's products (a wait that finds its barrier complete costs as much as a product, too).
            constexpr uint32_t DESC_HI = (uint32_t)((((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61)) >> 32);
            const bool b32 = st.kind != CLU_IN;    // blocks of 32 channels in the 64-byte swizzle
            const uint32_t a_hi = b32 ? (uint32_t)((((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)4 << 61)) >> 32) : DESC_HI;
            const uint32_t a_k2 = b32 ? (two ? 8192u : 4096u) >> 4 : 4u;
            const uint32_t w_lo = ((ptx::smem_u32(wring) & 0x3FFFF) >> 4) | (1u << 16), a_step = (uint32_t)(n_iss * (kb_bytes >> 4));
            const uint32_t bar_w0 = ptx::smem_u32(full_w), bar_e0 = ptx::smem_u32(empty_w), a_bstep = 8u * (uint32_t)n_iss;
            uint32_t slot = (wt + (uint32_t)me) % RS, pw = ((wt + (uint32_t)me) / RS) & 1u, acc = 0;
            uint32_t a_lo = (((ptx::smem_u32(panel) & 0x3FFFF) >> 4) | (1u << 16)) + (uint32_t)(me * (kb_bytes >> 4));
            uint32_t bar_a = ptx::smem_u32(norm ? normed : full_a) + 8u * (uint32_t)me;
            // parity of each activation block's barrier: blocks that every stage has, and those beyond
            const uint32_t n_lo = norm ? n_norm : n_gc + n_gi, n_hi = norm ? n_norm : (nkb_c > nkb_in ? n_gc : n_gi);
            const uint32_t lo_mask = (1u << min(nkb_c, nkb_in)) - 1u;
            uint32_t pa = (((n_lo & 1u) ? ~0u : 0u) & lo_mask) | (((n_hi & 1u) ? ~0u : 0u) & ~lo_mask);
            pa >>= me;
            bool ok_w = ptx::mbar_try_wait_s(bar_w0 + 8u * slot, pw), ok_a = ptx::mbar_try_wait_s(bar_a, pa & 1u);
            ptx::tc_fence_after();                 // the epilogue's loads of the previous accumulator (cluster barrier)
#pragma unroll 1
            for (int kb = me; kb < nkb; kb += n_iss) {
              if (!__all_sync(0xffffffffu, ok_w && ok_a)) {
                clu_wait(&full_w[slot], pw, s_fail, p.err, 0x103);
                clu_wait(&(norm ? normed : full_a)[kb], pa & 1u, s_fail, p.err, 0x105);
              }
              const uint64_t da = ((uint64_t)a_hi << 32) | a_lo, da2 = ((uint64_t)a_hi << 32) | (a_lo + a_k2), db = ((uint64_t)DESC_HI << 32) | (w_lo + slot * (uint32_t)(CLU_SLOT >> 4));
              const uint32_t empty = bar_e0 + 8u * slot;
              slot += (uint32_t)n_iss;
              if (slot >= RS) { slot -= RS; pw ^= 1u; }
              a_lo += a_step;
              bar_a += a_bstep;
              pa >>= n_iss;
              if (kb + n_iss < nkb) {
                ok_w = ptx::mbar_try_wait_s(bar_w0 + 8u * slot, pw);
                ok_a = ptx::mbar_try_wait_s(bar_a, pa & 1u);
              }
              if (ptx::elect_one()) {
                ptx::umma_bf16(d_acc, da, db, idesc, acc);
                ptx::umma_bf16(d_acc, da + 2, db + 2, idesc, 1);
                ptx::umma_bf16(d_acc, da2, db + 4, idesc, 1);
                ptx::umma_bf16(d_acc, da2 + 2, db + 6, idesc, 1);
                ptx::umma_commit_s(empty);
              }
              __syncwarp();
              acc = 1;
            }
          }
          wt += (uint32_t)nkb;
        }
        if (warp != 0) {
          if (ptx::elect_one()) ptx::umma_commit(accum);   // (an issuer without products of its own arrives at once)
          __syncwarp();
        }
        // one slot per cluster: the K/V ring is its own, the next attention's carried blocks are requested in the first conv block
        // (s_job is there from the second stage on); two: the panel is free once the projection's products are done
        fetch = p.n_attn > 0 && (ONE ? st.kind == CLU_CONV : st.kind == CLU_QKV);
        if (fetch && warp == 0 && !ONE && !clu_wait(accum, n_g & 1u, s_fail, p.err, 0x106)) fetch = false;
        ++n_g;
        if (st.kind == CLU_IN) { ++n_gi; xi = 0; } else if (!skip) ++n_gc;
        if (!skip && (st.kind == CLU_QKV || st.kind == CLU_OUT)) ++n_norm;
        if (st.kind == CLU_CONV || st.kind == CLU_OPROJ) xi ^= 1;
      }
      const bool att = st.kind == CLU_ATT;
      if (warp == 0 && (att || (fetch && pre == 0))) {
        // ---- Q and the K/V items of this CTA's jobs; ahead of the stage (fetch): the first job's items whose blocks hold only rows
        // of earlier chunks, at most the ring's size, so that nothing here depends on products of a coming stage ----
        bool first = true;
        uint32_t last_k = 0;                       // the previous job's last K item
        if (att) ptx::fence_proxy_async_global();
#pragma unroll 1
        for (int jid = rank; jid < n_jobs; jid += p.CL) {
          const CluJob jb = s_job[jid / p.n_heads];
          if (jb.T == 0) {
            if (!att) break;
            continue;
          }
          const int head = jid % p.n_heads, slot = slot0 + jid / p.n_heads;
          if (att) {
            // S of the previous job's last block has been computed when its K slot is released (the slot's earlier phases
            // have all been waited for when it was filled)
            if (!first && !clu_wait(&empty_kv[last_k % CLU_KVS], (last_k / CLU_KVS) & 1u, s_fail, p.err, 0x107)) break;
            // the slot's 56 chunk rows of the head's 64-column block (rows T.. are never stored; with head_dim 32 the block
            // holds two heads), twice: see flow_attn_kernel
            if (ptx::elect_one()) {
              const bf16* src = p.Q + ((long long)slot * nkb_c + (head << p.dh_shift >> 6)) * CLU_SLOT_KB + HALO * 64;
              ptx::mbar_expect_tx(bar_q, 2u * (SLOT_ROWS - HALO) * 128u);
              ptx::bulk_load(sQ, src, (SLOT_ROWS - HALO) * 128u, bar_q);
              ptx::bulk_load(sQ + 8192, src, (SLOT_ROWS - HALO) * 128u, bar_q);
            }
            __syncwarp();
          }
          const bf16* planes = jb.kv + (long long)(st.s * p.n_attn + st.g) * 2 * kv_plane + (long long)head * p.kv_hs;
          int item = att && first ? (int)pre : 0;
#pragma unroll 1
          for (; item < 2 * jb.k.nkb; ++item) {
            bool is_v;
            int b;
            clu_item(item, jb.k.nkb, &is_v, &b);
            if (!att && (item == (int)CLU_KVS || b >= jb.k.n_early)) break;
            const uint32_t gi = it0 + (uint32_t)item, ks = gi % CLU_KVS, k = gi / CLU_KVS;
            if (k > 0 && !clu_wait(&empty_kv[ks], (k - 1) & 1u, s_fail, p.err, 0x102)) break;
            uint8_t* dst = kvring + ks * CLU_KV_BYTES;
            const int n = min(ATT_KB, jb.k.L - b * ATT_KB);   // key rows of this block
            if (is_v && n < ATT_KB) {              // rows behind the last key must be finite up to the next UMMA step
              const int n16 = min(ATT_KB, (n + 15) & ~15);
#pragma unroll 1
              for (int i = lane; i < (n16 - n) << (p.dh_shift - 3); i += 32) *reinterpret_cast<uint4*>(dst + n * 2 * dh + i * 16) = make_uint4(0u, 0u, 0u, 0u);
              ptx::fence_proxy_async_smem();
              __syncwarp();
            }
            if (ptx::elect_one()) jb.k.fetch(planes + (is_v ? kv_plane : 0), b, n, p.P, p.Rk, p.dh_shift, dst, &full_kv[clu_kv_full(is_v, ks)]);
            __syncwarp();
          }
          if (!att) {
            pre = (uint32_t)item;
            // the carried rows behind the ring's: asked into L2, so that their copies take an L2 round trip when a slot is free and
            // not one to memory (3,500 cycles, half of the sweep's time)
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
            break;
          }
          last_k = it0 + (uint32_t)clu_item_k(jb.k.nkb - 1);
          it0 += 2u * (uint32_t)jb.k.nkb;
          first = false;
        }
        if (att) pre = 0;
      } else if (att && warp == 1) {
        // ---- scores: S(b) as soon as its stream's previous scores have been read.  (Scores and P V from one warp: 2,000 cycles of
        // waits and issue per block, which paced the sweep; a warp for each halves that.) ----
        const uint32_t idesc_s = ptx::umma_idesc_bf16(128, ATT_KB, 0, 0);
        const uint64_t dkv = ONE ? kv_base(ptx::smem_u32(kvring)) : 0ull;
#pragma unroll 1
        for (int jid = rank; jid < n_jobs; jid += p.CL) {
          const int nkb = s_job[jid / p.n_heads].k.nkb, head = jid % p.n_heads;
          if (s_job[jid / p.n_heads].T == 0) continue;
          const uint64_t dq = ptx::umma_desc_sw128(ptx::smem_u32(sQ)) + (uint64_t)(((head << p.dh_shift) & 63) >> 3);
#pragma unroll 1
          for (int b = 0; b < nkb; ++b) {
            const int w = b & 1;
            const uint32_t gi = it0 + (uint32_t)clu_item_k(b), ks = gi % CLU_KVS;
            clu_wait(&full_kv[clu_kv_full(false, ks)], kv_phases.next(ks), s_fail, p.err, 0x108);
            if (b == 0) clu_wait(bar_q, n_q++ & 1u, s_fail, p.err, 0x10a);
            const uint32_t k = w ? n_s1++ : n_s0++;
            if (k > 0) clu_wait(&bar_sfree[w], (k - 1) & 1u, s_fail, p.err, 0x109);   // the stream's previous scores have been read
            ptx::tc_fence_after();
            const uint64_t dk = kv_desc(dkv, ks);
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
      } else if (att && warp == 3) {
        // ---- O_w += P(b) V(b) ----
        const uint32_t idesc_pv = ptx::umma_idesc_bf16(128, dh, 0, 1);   // B = V, MN-major
        const uint64_t dp = ptx::umma_desc_sw128(ptx::smem_u32(sP));
        const uint64_t dkv = ONE ? kv_base(ptx::smem_u32(kvring)) : 0ull;
        const uint32_t v_step = 2u << p.dh_shift;
#pragma unroll 1
        for (int jid = rank; jid < n_jobs; jid += p.CL) {
          const int L = s_job[jid / p.n_heads].k.L, nkb = s_job[jid / p.n_heads].k.nkb;
          if (s_job[jid / p.n_heads].T == 0) continue;
#pragma unroll 1
          for (int b = 0; b < nkb; ++b) {
            const int w = b & 1;
            const uint32_t gi = it0 + (uint32_t)clu_item_v(b, nkb), vs = gi % CLU_KVS;
            clu_wait(&full_kv[clu_kv_full(true, vs)], kv_phases.next(vs), s_fail, p.err, 0x10d);
            clu_wait(&bar_p[w], (w ? n_s1++ : n_s0++) & 1u, s_fail, p.err, 0x10c);
            ptx::tc_fence_after();
            const uint64_t dpb = dp + (uint64_t)(w * (ATT_P_BYTES >> 4)), dv = kv_desc(dkv, vs);
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
      // The next stage's operand, if that is a GEMM: requested right behind the barrier, from an address made in front of it, where nobody waits.
      // (One stream 895.8 -> 883.3 us, fourteen 1,034 -> 1,014, the small decoder 333.6 -> 322.9.)  X[xi] by now is what this stage writes.
      CluStage nx = st;
      nx.next(p);
      const bool wants = warp == 0 && nx.s < p.n_steps && nx.kind != CLU_ATT && !(nx.kind == CLU_OUT && nch_out == 0);
      const int nx_nkb = nx.kind == CLU_IN ? nkb_in : nkb_c;
      const bf16* nx_src = (nx.kind == CLU_IN ? p.Ain : (nx.kind == CLU_OPROJ ? p.O : p.X[xi])) + (long long)slot0 * nx_nkb * CLU_SLOT_KB;
      // (this barrier's previous phase is complete: warp 0 has waited for it, two stages in bulk ago)
      const bool bulk = warp == 0 && in_bulk(st.kind);
      uint64_t* const bar_h = &hand[clu_hand(n_hand)];
      const uint32_t ph_h = clu_hand_parity(n_hand);
      if (bulk) {
        if (ptx::elect_one()) ptx::mbar_expect_tx(bar_h, 4u * (uint32_t)p.CL);
        __syncwarp();
        ++n_hand;
      }
      ptx::cluster_arrive_relaxed();
      // (read here, where nobody waits for it: a wait takes so long to give up that what it left behind one stage earlier has landed)
      bool failed = warp == 0 && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(s_fail) != 0);
      // The rows of a stage in bulk: this CTA's own signal tells that its panel is free, so the request need not wait for the cluster barrier as well.
      if (bulk && !failed) failed = !clu_wait<true>(bar_h, ph_h, s_fail, p.err, 0x115);
      if (!bulk) ptx::cluster_wait();
      if (wants && !failed) request(nx_src, nx_nkb, nx.kind == CLU_IN);
      if (bulk) ptx::cluster_wait();
      if (failed) {
#pragma unroll 1
        for (st.next(p); st.s < p.n_steps; st.next(p)) {
          ptx::cluster_arrive_relaxed();
          ptx::cluster_wait();
        }
        break;
      }
    }
  } else {
    // ---------------- epilogue: a thread owns one row and NC columns; attention: warps 4..7 even, 8..11 odd key blocks ----------------
    ptx::pdl_wait();
    const int et = tid - 128;
    const int q = warp & 3, cg = (warp - 4) >> 2;
    const int row_t = ONE ? q * 16 + (lane & 15) : q * 32 + lane, r = m0 + row_t;
    const int c0 = 16 * cg + (ONE ? 8 * (lane >> 4) : 0);   // the thread's first column of the CTA's 32
    const int slot = r / SLOT_ROWS, rho = r % SLOT_ROWS, f = rho - HALO;
    const bool own = slot < p.n_slots;
    const SlotInfo si = own ? p.slots[slot] : SlotInfo{0, 0, 0, 0, nullptr, nullptr, nullptr, nullptr, 0, 0, 0, 0, 0, 0, 0};
    if (et < SPC) {                               // (read by the control warps behind the first cluster barrier)
      const SlotInfo sj = slot0 + et < p.n_slots ? p.slots[slot0 + et] : SlotInfo{0, 0, 0, 0, nullptr, nullptr, nullptr, nullptr, 0, 0, 0, 0, 0, 0, 0};
      CluJob jb;
      jb.kv = sj.kv;
      jb.T = sj.T;
      jb.k.set(sj, p.P, p.Rk);
      s_job[et] = jb;
    }
    bf16* const s_halo = si.halo;
    bf16* const s_kv = si.kv;
    const bool is_out = si.pass == 0;
    const int tau0 = p.slots[slot0].tau_off, tau1 = !ONE && slot0 + 1 < p.n_slots ? p.slots[slot0 + 1].tau_off : 0;
    const int rows = !ONE && slot0 + 1 < p.n_slots ? 2 * SLOT_ROWS : SLOT_ROWS;   // of the cluster's blocks (an odd batch's last cluster has one slot)
    const bool in_range = si.T > 0;
    const bool halo_row = in_range && rho < HALO, chunk_row = in_range && f >= 0 && f < si.T;
    const int new_row = rho - si.Tc;                // carry row this thread's value moves to
    const bool moves = (halo_row || chunk_row) && new_row >= 0 && new_row < HALO;
    const uint32_t lanes = tmem_base + ((uint32_t)(q * 32) << 16);
    const float* tau_s = s_tau + (ONE ? 0 : (q >> 1) & 1) * 64;
    const int aq = q & 1, ah = q >> 1;              // softmax: query quarter, key half
    const int tp = min(si.T, p.P - si.n_prompt0);   // the chunk's first tp frames complete the prompt
    int kv_row = 0;                                 // K/V plane row of this thread's frame
    if (f < tp) {
      kv_row = si.n_prompt0 + f;
    } else {
      kv_row = si.kv_head + f - tp;
      if (kv_row >= p.Rk) kv_row -= p.Rk;
      kv_row += p.P;
    }
    uint32_t xr[NC / 2];                          // the residual stream: this thread's row and columns, bf16 pairs
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) xr[i] = 0u;
    int xi = 0;
    uint32_t n_g = 0, n_gc = 0, n_gi = 0;
    uint32_t n_hand = 0;                            // stages whose rows left in bulk so far
    uint32_t n_blk = 0;                             // key blocks of this thread's stream so far
#pragma unroll 1
    for (CluStage st; st.s < p.n_steps; st.next(p)) {
      if (st.kind == CLU_ATT) {
#pragma unroll 1
        for (int jid = rank; jid < n_jobs; jid += p.CL) {
          const CluJob jb = s_job[jid / p.n_heads];
          if (jb.T == 0) continue;
          const int nkb = jb.k.nkb, head = jid % p.n_heads;
          const int row = aq * 32 + lane, w = cg;
          float* sx = s_x + w * 128;
          float m_ref = -INFINITY, lsum = 0.f;
          bool ok = true;
#pragma unroll 1
          for (int b = w; b < nkb; b += 2, ++n_blk) {
            const uint32_t k = n_blk;
            ok &= clu_wait(&bar_s[w], k & 1u, s_fail, p.err, 0x10e);
            ptx::tc_fence_after();
            float v[64];
            ptx::tmem_ld64(lanes + (uint32_t)(w * ATT_KB + ah * 64), v);
            ptx::tc_fence_before();
            ptx::mbar_arrive(&bar_sfree[w]);       // S(b) has been read: the stream's next scores may overwrite it
            const int col0 = b * ATT_KB + ah * 64;
            float mx = att_mask_max(v, jb.k.L - col0, jb.k.g0 - col0, jb.k.g1 - col0);
            sx[ah * 64 + row] = mx * p.scale_log2e;
            ptx::named_bar_sync(4 + w, 128);
            mx = fmaxf(sx[row], sx[64 + row]);
            ptx::named_bar_sync(4 + w, 128);
            if (b >= 2) ok &= clu_wait(&bar_pv[w], (k - 1) & 1u, s_fail, p.err, 0x110);   // the stream's P buffer and O are quiescent
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
          // (each group waits for its own stream, whose phases it has followed; the barrier tells the other group)
          if (w < nkb) ok &= clu_wait(&bar_pv[w], (n_blk - 1) & 1u, s_fail, p.err, 0x111);
          ptx::named_bar_sync(1, CLU_EPI);
          ptx::tc_fence_after();
          ok = ok && *reinterpret_cast<volatile int*>(s_fail) == 0;
          if (ah == 0) {                           // O rows 0..63 live in lanes 0..63; each group of warps stores half of the columns
            float c0, c1;
            att_combine(nkb, s_m[row], s_x[row] + s_x[64 + row], s_m[64 + row], s_x[128 + row] + s_x[192 + row], &c0, &c1);
            const int orow = (ONE ? 0 : (jid / p.n_heads) * SLOT_ROWS) + HALO + row;
#pragma unroll 1
            for (int c = w * (dh >> 1); c < (w + 1) * (dh >> 1); c += 16) {
              float o16[16], q16[16];
              ptx::tmem_ld16x2(lanes + (uint32_t)(CLU_O_COL + c), lanes + (uint32_t)(CLU_O_COL + 64 + c), o16, q16);   // (O_1 is anything with one block)
              if (row < jb.T && ok) {
#pragma unroll
                for (int i = 0; i < 16; ++i) o16[i] = nkb > 1 ? fmaf(q16[i], c1, o16[i] * c0) : o16[i] * c0;
                uint4 a, bq;
                pack16_bf16(o16, a, bq);
                if (one_job) {                     // (the queries' tile is idle by now)
                  bf16* d = reinterpret_cast<bf16*>(sQ) + (c >> 5) * (SLOT_ROWS * 32);
                  *reinterpret_cast<uint4*>(d + clu_at32(row + HALO, c & 31)) = a;
                  *reinterpret_cast<uint4*>(d + clu_at32(row + HALO, (c & 31) + 8)) = bq;
                } else {
                  const int ch = (head << p.dh_shift) + c, perm = (orow >> 1) & 3;
                  store16(p.O + (long long)slot0 * nkb_c * CLU_SLOT_KB + (long long)(ch >> 5) * (rows * 32) + orow * 32 + ((((ch & 31) >> 3) ^ perm) & ~1) * 8,
                          (perm & 1) ? bq : a, (perm & 1) ? a : bq);
                }
              }
            }
          }
          ptx::tc_fence_before();
          if (!one_job) ptx::named_bar_sync(1, CLU_EPI);   // (the next job overwrites the exchange and the accumulators)
        }
        if (one_job) {
          // the 56 rows of its slot in the head's one or two blocks of 32 channels
          const int head = ONE ? rank : rank % p.n_heads, sl = ONE ? 0 : rank / p.n_heads;
          const bool has = rank < n_jobs && slot0 + sl < p.n_slots && s_job[sl].T > 0;
          const uint32_t bytes = has ? (SLOT_ROWS - HALO) * 64u : 0u;
          bf16* dst = p.O + (long long)slot0 * nkb_c * CLU_SLOT_KB + ((head << p.dh_shift) >> 5) * (rows * 32) + (sl * SLOT_ROWS + HALO) * 32;
          const uint8_t* src = sQ + HALO * 64;
          const CluPiece piece[2] = {{dst, src, bytes}, {dst + rows * 32, src + SLOT_ROWS * 64, p.dh_shift == 6 ? bytes : 0u}};
          clu_arrive_bulk(warp, lane, piece, ptx::smem_u32(&hand[clu_hand(n_hand++)]), ptx::smem_u32(s_word), p.CL);
        } else {
          clu_arrive_release(warp);
        }
        ptx::cluster_wait();
        continue;
      }

      const int kind = st.kind, nkb = kind == CLU_IN ? nkb_in : nkb_c;
      const int n_iss = issuers(nkb);
      const bool next_conv = kind == CLU_IN || (kind == CLU_CONV && st.j + 1 < p.cpa) || (kind == CLU_OPROJ && st.g + 1 < p.n_attn);
      const int l_next = kind == CLU_CONV ? st.l + 1 : (kind == CLU_OPROJ ? st.l : 0);
      bf16* carry = next_conv && in_range ? s_halo + ((long long)st.s * p.n_conv + l_next) * HALO * p.C : nullptr;
      const bool feeds_norm = (kind == CLU_CONV && st.j + 1 == p.cpa) || (kind == CLU_OPROJ && st.g + 1 == p.n_attn);
      const bool skip = kind == CLU_OUT && nch_out == 0;
      const bool norm = (kind == CLU_QKV || kind == CLU_OUT) && !skip;

      // ---- what does not depend on the accumulator, under the main loop ----
      float4 part[8];                                // partial sums of squares of the row, 16 channels each (first: their loads take longest)
      if (norm) clu_wait<true>(&hand[clu_hand(n_hand - 1u)], clu_hand_parity(n_hand - 1u), s_fail, p.err, 0x116);   // (the statistics of the stage before, of every CTA)
      if (norm && chunk_row) {
        const float* src = p.ssq + (long long)slot * (p.C >> 4) * SLOT_ROWS + rho;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < p.C >> 6)
            part[j] = make_float4(__ldcg(src + 4 * j * SLOT_ROWS), __ldcg(src + (4 * j + 1) * SLOT_ROWS), __ldcg(src + (4 * j + 2) * SLOT_ROWS), __ldcg(src + (4 * j + 3) * SLOT_ROWS));
      }
      {
        const int gbase = p.C + st.g * (p.cpa + 4) * p.C;     // biases in blob order: input, then per group conv..., Q, K, V, O
        if (kind == CLU_OUT) {
          if (et < 16 * nch_out) s_bias[et] = p.fc[p.o_bout + (rank + (et >> 4) * p.CL) * 16 + (et & 15)];
        } else {
          const int ob = kind == CLU_IN ? 0 : (kind == CLU_CONV ? gbase + st.j * p.C : gbase + (p.cpa + (kind == CLU_OPROJ ? 3 : 0)) * p.C);
          const int nb = kind == CLU_QKV ? 3 * BN : BN;
          if (et < nb) s_bias[et] = p.fc[ob + (et / BN) * p.C + n0 + et % BN];
        }
        if (kind == CLU_CONV && et < SPC * BN) {
          const int sl = et / BN, c = et % BN;
          s_tau[sl * 64 + c] = p.fc[p.o_tau + (st.s * p.n_conv + st.l) * p.C + (sl ? tau1 : tau0) + n0 + c];
        }
      }
      // The carried row for the next conv block.  Where none follows, a left-context row stays as it is (one slot per cluster) or is zeros (two); no row reads it.
      // (Each the form that took less: one stream 747 us per chunk against 757 with zeros, fourteen 933 against 947 without.)
      uint4 hr[NC / 8];
#pragma unroll
      for (int i = 0; i < NC / 8; ++i)
        if (!ONE) hr[i] = make_uint4(0u, 0u, 0u, 0u);
      if (carry != nullptr && halo_row) {
        const uint4* src = reinterpret_cast<const uint4*>(carry + rho * p.C + n0 + c0);
#pragma unroll
        for (int i = 0; i < NC / 8; ++i) hr[i] = src[i];
      }
      float rs = 1.f;
      if (norm) {
        float ss = 0.f;
        if (chunk_row) {                             // added in chunk order
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (j < p.C >> 6) ss = (((ss + part[j].x) + part[j].y) + part[j].z) + part[j].w;
        }
        rs = rsqrtf(ss * p.inv_C + p.eps);
      }
      if (ROUNDED && norm && c0 == 0) s_x[row_t] = chunk_row ? rs : -1.f;   // (-1: a row that stays as it is)
      ptx::named_bar_sync(1, CLU_EPI);               // constants are in place; every carried row has been read
      if (ROUNDED && norm) {
        // The normalised activations as rounded bf16 values: the panel is rewritten in place, block by block ahead of the issuer, 16 bytes of every 32nd
        // row by a thread (a warp's accesses are whole rows: no bank conflicts), all of them requested before the first is used.  Rows outside the chunk are
        // read and not written: a branch around every piece cost more than the pieces.
        // (32 bytes of each slot's row in turn, with a wait in between: 14 streams 1,140 us, one guided stream 1,105, one stream 960; pieces in branches of
        // their own 1,110, 1,079 and 956; so 1,086, 1,054 and 934.)
        const bool two = !ONE && rows == 2 * SLOT_ROWS;
        float k[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) k[i] = s_x[(rows == SLOT_ROWS ? 0 : (i & 1) * SLOT_ROWS) + (et >> 2)];   // (16 bytes of a slot's row in either block of 32 channels)
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb) {
          clu_wait(&full_a[kb], ((kb < nkb_c ? n_gc : 0u) + (kb < nkb_in ? n_gi : 0u)) & 1u, s_fail, p.err, 0x114);
          uint4* px = reinterpret_cast<uint4*>(panel + kb * kb_bytes) + et;
          uint4 x[4];
          x[0] = px[0];
          x[1] = px[256];
          if (two) {
            x[2] = px[512];
            x[3] = px[768];
          }
          auto put = [&](int i) {
            const uint32_t w[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
            uint32_t o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(w[j] << 16) * k[i], __uint_as_float(w[j] & 0xFFFF0000u) * k[i]);
              o[j] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            if (!(k[i] < 0.f)) px[256 * i] = make_uint4(o[0], o[1], o[2], o[3]);
          };
          put(0);
          put(1);
          if (two) {
            put(2);
            put(3);
          }
          ptx::fence_proxy_async_smem();
          ptx::mbar_arrive(&normed[kb]);
        }
        rs = 1.f;
      }
      const bool got = clu_wait(accum, n_g & 1u, s_fail, p.err, 0x113);
      ptx::tc_fence_after();
      const bool ok = got && *reinterpret_cast<volatile int*>(s_fail) == 0;
      const bool is_chunk = chunk_row && ok;

      auto load_pair = [&](uint32_t col, float* v) {  // NC columns of the 16 from `col` on; even blocks + odd blocks, always in this order
        if (n_iss == 2) {
          uint32_t t[2 * NC];
          ptx::tmem_ld_rows_issue<NC>(lanes + col, t);
          ptx::tmem_ld_rows_issue<NC>(lanes + CLU_ACC2 + col, t + NC);
          ptx::tmem_ld_wait<2 * NC>(t);
#pragma unroll
          for (int i = 0; i < NC; ++i) v[i] = __uint_as_float(t[i]) + __uint_as_float(t[NC + i]);
        } else {
          uint32_t t[NC];
          ptx::tmem_ld_rows_issue<NC>(lanes + col, t);
          ptx::tmem_ld_wait<NC>(t);
#pragma unroll
          for (int i = 0; i < NC; ++i) v[i] = __uint_as_float(t[i]);
        }
      };
      // A row's 16 columns as one 32-byte store, the halves swapped where the row's place in the swizzle is odd.  (ONE: the two lanes of a row bring
      // them together in the lower one.)
      auto put_row = [&](bool pred, bf16* d, bool swap, const uint32_t* w) {
        uint4 a = make_uint4(w[0], w[1], w[2], w[3]), b;
        if (ONE) {
          b.x = __shfl_xor_sync(0xffffffffu, a.x, 16);
          b.y = __shfl_xor_sync(0xffffffffu, a.y, 16);
          b.z = __shfl_xor_sync(0xffffffffu, a.z, 16);
          b.w = __shfl_xor_sync(0xffffffffu, a.w, 16);
          pred = pred && lane < 16;
        } else {
          b = make_uint4(w[NC / 2 - 4], w[NC / 2 - 3], w[NC / 2 - 2], w[NC / 2 - 1]);
        }
        if (pred) store16(d, swap ? b : a, swap ? a : b);
      };

      if (kind == CLU_OUT) {
#pragma unroll 1
        for (int k = cg; k < nch_out; k += 2) {
          const int n = (rank + k * p.CL) * 16 + c0 - 16 * cg;
          float acc[NC];
          load_pair((uint32_t)(16 * k), acc);
#pragma unroll
          for (int i = 0; i < NC; ++i) acc[i] = fmaf(acc[i], rs, s_bias[16 * k + c0 - 16 * cg + i]);
          if (!ONE && p.cfg_w > 0.f) {
            // guided step: rows 64.. are the unconditional pass; they hand their velocity over through shared memory
            float4* xv4 = reinterpret_cast<float4*>(panel) + k * 256;
            if (q >= 2) {
#pragma unroll
              for (int j = 0; j < NC / 4; ++j) xv4[j * 64 + (q - 2) * 32 + lane] = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
            }
            ptx::named_bar_sync(2 + cg, 128);
            if (q < 2) {
#pragma unroll
              for (int j = 0; j < NC / 4; ++j) {
                const float4 u = xv4[j * 64 + q * 32 + lane];
                acc[4 * j] = fmaf(1.f + p.cfg_w, acc[4 * j], -p.cfg_w * u.x);
                acc[4 * j + 1] = fmaf(1.f + p.cfg_w, acc[4 * j + 1], -p.cfg_w * u.y);
                acc[4 * j + 2] = fmaf(1.f + p.cfg_w, acc[4 * j + 2], -p.cfg_w * u.z);
                acc[4 * j + 3] = fmaf(1.f + p.cfg_w, acc[4 * j + 3], -p.cfg_w * u.w);
              }
            }
          }
          const bool advances = is_chunk && is_out;
          uint32_t w[NC / 2];
#pragma unroll
          for (int i = 0; i < NC / 2; ++i) w[i] = 0u;
          if (advances) {
            float* xs = p.xstate + (long long)r * p.mel + n;
            float xv[NC];
#pragma unroll
            for (int i = 0; i < NC; i += 4) {
              const float4 t = *reinterpret_cast<const float4*>(xs + i);
              xv[i] = t.x; xv[i + 1] = t.y; xv[i + 2] = t.z; xv[i + 3] = t.w;
            }
#pragma unroll
            for (int i = 0; i < NC; ++i) xv[i] = xv[i] + acc[i] * p.inv_n;
#pragma unroll
            for (int i = 0; i < NC; i += 4) *reinterpret_cast<float4*>(xs + i) = make_float4(xv[i], xv[i + 1], xv[i + 2], xv[i + 3]);
            pack_row<NC>(xv, w);
            const SlotInfo& so = p.slots[slot];      // (read again: only here, once per chunk)
            if ((p.tick ? (so.flags & SLOT_LAST) != 0 : st.s == p.n_steps - 1) && f < so.Tc) {
              float* o = so.out + (long long)f * p.mel + n;
#pragma unroll
              for (int i = 0; i < NC; i += 4) *reinterpret_cast<float4*>(o + i) = make_float4(xv[i], xv[i + 1], xv[i + 2], xv[i + 3]);
            }
          }
          bf16* d = p.Ain + ((long long)slot * nkb_in + (n >> 6)) * CLU_SLOT_KB + clu_row16(rho, n & 63);
          put_row(advances, d, rho & 1, w);
          if (!ONE && p.cfg_w > 0.f) put_row(advances, d + (long long)nkb_in * CLU_SLOT_KB, rho & 1, w);   // the unconditional pass starts from the same x
        }
        if (!ONE && p.cfg_w > 0.f) ptx::fence_proxy_async_smem();   // (the exchange above: the next stage's bulk copies overwrite it)
        ptx::tc_fence_before();
        clu_arrive_release(warp);
      } else if (kind == CLU_QKV) {
        const long long kv_off = ((long long)st.s * p.n_attn + st.g) * 2 * kv_plane;
        const int col = n0 + 16 * cg;
        const int hh = col >> p.dh_shift, wi = col - (hh << p.dh_shift);
        const int perm = kv_perm(kv_row, p.dh_shift);
        bf16* kvp = s_kv + kv_off + (long long)hh * p.kv_hs + ((long long)kv_row << p.dh_shift) + ((((wi >> 3) ^ perm) & ~1) << 3);
#pragma unroll
        for (int which = 0; which < 3; ++which) {
          float acc[NC];
          load_pair((uint32_t)(which * BN + 16 * cg), acc);
          const float4* bias4 = reinterpret_cast<const float4*>(s_bias + which * BN + c0);
#pragma unroll
          for (int i = 0; i < NC / 4; ++i) {
            const float4 b4 = bias4[i];
            acc[4 * i] = fmaf(acc[4 * i], rs, b4.x);
            acc[4 * i + 1] = fmaf(acc[4 * i + 1], rs, b4.y);
            acc[4 * i + 2] = fmaf(acc[4 * i + 2], rs, b4.z);
            acc[4 * i + 3] = fmaf(acc[4 * i + 3], rs, b4.w);
          }
          uint32_t w[NC / 2];
          pack_row<NC>(acc, w);
          if (which == 0) put_row(is_chunk, p.Q + ((long long)slot * nkb_c + (col >> 6)) * CLU_SLOT_KB + clu_row16(rho, col & 63), rho & 1, w);
          else put_row(is_chunk, kvp + (which - 1) * kv_plane, perm & 1, w);
        }
        ptx::tc_fence_before();
        clu_arrive_release(warp);
      } else {
        // ---- a new residual row: input projection, conv block, attention output projection ----
        bf16* out = p.X[kind == CLU_IN ? 0 : xi ^ 1];
        float2 acc[NC / 2];
        if (kind == CLU_CONV) {
          // y[r] = Z_0[r - 2 d] + Z_1[r - d] + Z_2[r]: rows change lanes through shared memory (the panel is idle by now)
          float2 z[NC / 2], z2[NC / 2];
          const uint32_t col = lanes + (uint32_t)(16 * cg);
          auto sum = [&](const uint32_t* t, float2* v) {
#pragma unroll
            for (int i = 0; i < NC / 2; ++i) v[i] = add2(pair2(t[2 * i], t[2 * i + 1]), pair2(t[NC + 2 * i], t[NC + 2 * i + 1]));
          };
          if (n_iss == 2) {
            uint32_t ra[2 * NC], rb[2 * NC];     // even blocks + odd blocks, two taps behind one wait (ONE: all three)
            ptx::tmem_ld_rows_issue<NC>(col, ra);
            ptx::tmem_ld_rows_issue<NC>(col + CLU_ACC2, ra + NC);
            ptx::tmem_ld_rows_issue<NC>(col + BN, rb);
            ptx::tmem_ld_rows_issue<NC>(col + CLU_ACC2 + BN, rb + NC);
            if (ONE) {
              uint32_t rc[2 * NC];
              ptx::tmem_ld_rows_issue<NC>(col + 2 * BN, rc);
              ptx::tmem_ld_rows_issue<NC>(col + CLU_ACC2 + 2 * BN, rc + NC);
              ptx::tmem_ld_wait<2 * NC>(ra);
              ptx::tmem_ld_wait<2 * NC>(rb);
              ptx::tmem_ld_wait<2 * NC>(rc);
              sum(ra, acc);
              sum(rb, z);
              sum(rc, z2);
            } else {
              ptx::tmem_ld_wait<2 * NC>(ra);
              ptx::tmem_ld_wait<2 * NC>(rb);
              sum(ra, acc);
              sum(rb, z);
              ptx::tmem_ld_rows_issue<NC>(col + 2 * BN, ra);
              ptx::tmem_ld_rows_issue<NC>(col + CLU_ACC2 + 2 * BN, ra + NC);
              ptx::tmem_ld_wait<2 * NC>(ra);
              sum(ra, z2);
            }
          } else {
            load_pair((uint32_t)(16 * cg), reinterpret_cast<float*>(acc));
            load_pair((uint32_t)(BN + 16 * cg), reinterpret_cast<float*>(z));
            load_pair((uint32_t)(2 * BN + 16 * cg), reinterpret_cast<float*>(z2));
          }
          // [column group][tap][four columns][row]
          float4* xz = reinterpret_cast<float4*>(panel) + (c0 / NC) * (2 * (NC / 4) * ROWS);
#pragma unroll
          for (int j = 0; j < NC / 4; ++j) {
            xz[j * ROWS + row_t] = make_float4(acc[2 * j].x, acc[2 * j].y, acc[2 * j + 1].x, acc[2 * j + 1].y);
            xz[(NC / 4 + j) * ROWS + row_t] = make_float4(z[2 * j].x, z[2 * j].y, z[2 * j + 1].x, z[2 * j + 1].y);
          }
          ptx::named_bar_sync(2 + cg, 128);
          const int d = p.dil[st.l], r0 = max(row_t - 2 * d, 0), r1 = max(row_t - d, 0);
          const float4* bias4 = reinterpret_cast<const float4*>(s_bias + c0);
          const float4* tau4 = reinterpret_cast<const float4*>(tau_s + c0);
#pragma unroll
          for (int j = 0; j < NC / 4; ++j) {
            const float4 a0 = xz[j * ROWS + r0], a1 = xz[(NC / 4 + j) * ROWS + r1], b4 = bias4[j], t4 = tau4[j];
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
          load_pair((uint32_t)(16 * cg), reinterpret_cast<float*>(acc));
          const float4* bias4 = reinterpret_cast<const float4*>(s_bias + c0);
#pragma unroll
          for (int j = 0; j < NC / 4; ++j) {
            const float4 b4 = bias4[j];
            acc[2 * j] = add2(acc[2 * j], make_float2(b4.x, b4.y));
            acc[2 * j + 1] = add2(acc[2 * j + 1], make_float2(b4.z, b4.w));
          }
          if (kind == CLU_OPROJ) {
#pragma unroll
            for (int i = 0; i < NC / 2; ++i) acc[i] = add2(acc[i], unpack2(xr[i]));
          }
        }
        pack_row<NC>(reinterpret_cast<const float*>(acc), xr);
        uint32_t w[NC / 2];
#pragma unroll
        for (int i = 0; i < NC / 2; ++i) w[i] = xr[i];
        if (rho < HALO && (!ONE || carry != nullptr)) {   // a left-context row hands the carried row on
#pragma unroll
          for (int i = 0; i < NC / 8; ++i) { w[4 * i] = hr[i].x; w[4 * i + 1] = hr[i].y; w[4 * i + 2] = hr[i].z; w[4 * i + 3] = hr[i].w; }
        }
        // Staged in the panel behind the taps' exchange.  (Rows that are neither the chunk's nor its left context go along; no row reads one behind it.)
        bf16* const rows_out = reinterpret_cast<bf16*>(panel + SPC * 16384);
        float* const ssq_out = reinterpret_cast<float*>(panel + SPC * 16384 + ROWS * 64);   // [slot][2][SLOT_ROWS]
#pragma unroll
        for (int i = 0; i < NC / 8; ++i)
          *reinterpret_cast<uint4*>(rows_out + clu_at32(row_t, c0 + 8 * i)) = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
        if (feeds_norm && in_range) {              // sum of squares of the row's 16 stored values, fixed order (ONE: the upper lane goes on from the lower one's)
          float ss = 0.f;
#pragma unroll
          for (int part16 = 0; part16 < 16 / NC; ++part16) {
            if (part16) ss = __shfl_xor_sync(0xffffffffu, ss, 16);
            if (is_chunk) {
#pragma unroll
              for (int i = 0; i < NC / 2; ++i) {
                const float lo = __uint_as_float(xr[i] << 16), hi = __uint_as_float(xr[i] & 0xFFFF0000u);
                ss = fmaf(lo, lo, ss);
                ss = fmaf(hi, hi, ss);
              }
            }
          }
          if (!ONE || lane >= 16) ssq_out[(row_t >> 6) * 2 * SLOT_ROWS + cg * SLOT_ROWS + rho] = ss;
        }
        ptx::tc_fence_before();
        const long long ssq_slot = (long long)(p.C >> 4) * SLOT_ROWS;
        float* const ssq = p.ssq + (long long)slot0 * ssq_slot + 2 * rank * SLOT_ROWS;
        const uint32_t ssq_bytes = feeds_norm ? 2u * SLOT_ROWS * 4u : 0u;
        const CluPiece rows_piece = {out + (long long)slot0 * nkb_c * CLU_SLOT_KB + rank * (rows * 32), rows_out, (uint32_t)rows * 64u};
        const uint32_t hand_now = ptx::smem_u32(&hand[clu_hand(n_hand++)]);
        if (ONE) {
          const CluPiece piece[2] = {rows_piece, {ssq, ssq_out, ssq_bytes}};
          clu_arrive_bulk(warp, lane, piece, hand_now, ptx::smem_u32(s_word), p.CL);
        } else {
          const CluPiece piece[3] = {rows_piece, {ssq, ssq_out, ssq_bytes}, {ssq + ssq_slot, ssq_out + 2 * SLOT_ROWS, rows == 2 * SLOT_ROWS ? ssq_bytes : 0u}};
          clu_arrive_bulk(warp, lane, piece, hand_now, ptx::smem_u32(s_word), p.CL);
        }
        // shift the carry by the committed frames: nobody in this launch reads it again
        if (carry != nullptr && moves && ok) {
          bf16* d = carry + new_row * p.C + n0 + c0;
          if (ONE) *reinterpret_cast<uint4*>(d) = make_uint4(w[0], w[1], w[2], w[3]);
          else store16(d, make_uint4(w[0], w[1], w[2], w[3]), make_uint4(w[NC / 2 - 4], w[NC / 2 - 3], w[NC / 2 - 2], w[NC / 2 - 1]));
        }
      }
      ++n_g;
      if (kind == CLU_IN) { ++n_gi; xi = 0; } else if (!skip) ++n_gc;
      if (kind == CLU_CONV || kind == CLU_OPROJ) xi ^= 1;
      ptx::cluster_wait();
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (*reinterpret_cast<volatile int*>(s_fail) != 0) ptx::pause_for_copies();
  if (warp == 1) ptx::tmem_dealloc(tmem_base, 512);
}

// The weight streams: CTA r's tiles in the order of the stages, each tile [rows][64 channels] as the 128-byte-swizzled
// shared-memory image.  Row j RJ + n of a tile is matrix row r rs_rank + j rs_j + n, channels cs_j j + 64 kb ...
struct CluPack {
  const bf16* src;
  long long   dst_off;       // byte offset of the stage in a CTA's stream
  int         ldk, J, RJ, rs_rank, rs_j, cs_j, n_valid;   // n_valid: matrix rows (the last CTAs of the output projection have fewer chunks)
};
__global__ void clu_pack_kernel(const CluPack c, uint8_t* stream, long long stream_bytes) {
  const int rank = blockIdx.y, kb = blockIdx.z;
  int J = c.J;                                       // (the sub-blocks that fall outside the matrix are the last ones: left out)
  while (J > 0 && rank * c.rs_rank + (J - 1) * c.rs_j >= c.n_valid) --J;
  const int rows = J * c.RJ;
  uint8_t* dst = stream + rank * stream_bytes + c.dst_off + (long long)kb * rows * 128;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows * 8; i += gridDim.x * blockDim.x) {
    const int row = i >> 3, ch = i & 7, j = row / c.RJ, n = row - j * c.RJ;
    const bf16* s = c.src + (long long)(rank * c.rs_rank + j * c.rs_j + n) * c.ldk + (long long)j * c.cs_j + kb * KBLK + ch * 8;
    *reinterpret_cast<uint4*>(dst + row * 128 + ((ch ^ (row & 7)) << 4)) = *reinterpret_cast<const uint4*>(s);
  }
}
