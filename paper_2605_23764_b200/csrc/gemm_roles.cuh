// Warp roles of the CTA-pair grouped GEMMs as device functions: TMA producers, tcgen05.mma issuer and
// epilogue warps of the token-column row-space operators and of the strip-wise weight gradients.
//
// Every function here handles ONE work item (a token tile x column tile of a row-space operator, or a
// strip of a weight gradient), already decoded, for one role: decoding an item takes a chain of dependent
// global loads (two or three microseconds), so callers decode the NEXT item while the current one runs.  The one-launch-per-operator kernels (gemm_tc3.cu,
// gemm_wgrad.cu) walk an operator's items in a static order with no event counters; the persistent
// launch (fused.cu) takes items of all operators of a pass from one ticket queue, carries the pipeline
// state (stage ring position, barrier parities, end of TMEM in turn) from item to item and orders
// tiles by event counters (the dependent and trigger events of Section 4.3).  Both use exactly this
// code, so they produce the same bits.
#pragma once

#include "gemm_swap.cuh"

namespace moe {

constexpr int WG_A_SLOTS = 5;    // weight gradients: 16 KB slots of the strip's A operand
constexpr int WG_B_STAGES = 7;   // weight gradients: 16 KB stages of the streamed B operand
constexpr int MAX_STAGES = 12;   // row-space operators: see plan_ring
constexpr size_t WGRAD_STAGING_AT = (size_t)WG_A_SLOTS * A_STAGE_BYTES + (size_t)WG_B_STAGES * HALF_B_BYTES;   // behind both

// Warps of a GEMM CTA: 0 weight loader, 1 MMA issuer, 2-5 and 8-11 epilogue, 6 token loader, 7 left to the kernel (scheduler).
// TMEM lanes 32 (w % 4) .. are what warp w can read.
constexpr int GEMM_ROLE_WARPS = 12;
__device__ __forceinline__ bool is_epilogue_warp(int warp) { return (warp >= 2 && warp < 6) || (warp >= 8 && warp < 12); }
__device__ __forceinline__ int epilogue_index(int warp) { return (warp & 3) + (warp >= 8 ? 4 : 0); }

// Accumulators.  An item has 32 to 256 TMEM columns, a merged one 128 + 160 or 128 + 192; items take the two ends of the 512
// columns in turn, so that an item's products run beside the epilogue of the one before.  Where the two overlap -- behind or before
// merged items -- the item begins when the tile in the middle is drained: that tile is the larger one, and its epilogue comes
// first.  The overlap never reaches the tile behind it: two items have 320 columns at most.  Four slots: end, tile.
constexpr int ACC_SLOTS = 4;
static_assert(2 * MERGED_TOKENS_MAX - TMEM_COLS <= BLOCK_M + TOK_GRAIN, "a merged item's first tile is at least as wide as any overlap");
static_assert(MERGED_TOKENS_MAX + 2 * BLOCK_M - TMEM_COLS <= 2 * BLOCK_M, "an item of one tile as well");
// first column of tile `part` (0: the one towards the middle) of an item of n0 + n1 columns
__device__ __forceinline__ int acc_column(int end, int part, int n0, int n1) {
  return part == 0 ? (end ? TMEM_COLS - n0 - n1 : n1) : (end ? TMEM_COLS - n1 : 0);
}

struct __align__(8) PipeBarriers {
  uint64_t full[MAX_STAGES];      // used in the even CTA: bytes of both CTAs' loads of the stage
  uint64_t empty[MAX_STAGES];     // in each CTA: the stage's MMAs are complete
  uint64_t a_empty[WG_A_SLOTS];  // weight gradients, in each CTA: every MMA that reads the A slot's content is complete
  uint64_t tmem_full[ACC_SLOTS];  // in each CTA: accumulator ready
  uint64_t tmem_empty[ACC_SLOTS]; // used in the even CTA: the epilogue warps of the pair have drained it
  uint64_t drain;
  uint32_t tmem_base;
  int epi_phase[EPI_WARPS];       // in each CTA: the phase each epilogue warp is in (its stores of earlier phases have read shared memory)
  int epi_done[ACC_SLOTS];        // in each CTA, per accumulator: epilogue warps whose stores of the tile are under way
  int pad;
};

// Pipeline state of a role, carried from item to item (the barriers persist).  The parity to wait for is kept per
// stage, so operators with rings of different depth can follow one another in one launch (the ring position
// restarts at 0 at such a boundary, where every stage has been consumed).
struct LoaderState {
  uint32_t s = 0, empty_par = (1u << MAX_STAGES) - 1, a_s = 0, a_ph = (1u << WG_A_SLOTS) - 1;
  int guard = 0;   // != 0: the phase whose epilogue warps must all have arrived before a stage above WGRAD_STAGING_AT is loaded
};
struct IssuerState {
  uint32_t s = 0, full_par = 0, a_s = 0;
  int end = 0;                    // of the TMEM columns, for the next item
  uint32_t busy = 0, acc_par = 0; // by slot: not seen drained; parity of the next drain
  int before_n = 0;               // columns of the item before
};
struct EpiState { int end = 0; uint32_t full_par = 0; };

__device__ __forceinline__ void pipe_init(PipeBarriers* bars) {   // one thread
  for (int s = 0; s < MAX_STAGES; ++s) {
    mbar_init(&bars->full[s], 1);
    mbar_init(&bars->empty[s], 1);
  }
  for (int s = 0; s < WG_A_SLOTS; ++s) mbar_init(&bars->a_empty[s], 1);
  for (int s = 0; s < ACC_SLOTS; ++s) {
    mbar_init(&bars->tmem_full[s], 1);
    mbar_init(&bars->tmem_empty[s], 2 * EPI_WARPS);
    bars->epi_done[s] = 0;
  }
  mbar_init(&bars->drain, 1);
  for (int w = 0; w < EPI_WARPS; ++w) bars->epi_phase[w] = 0;
}
// Phase boundaries of the persistent launch.  The shared memory of a phase (operand ring, staging) is carved per operator.
// Operand rings start at the bottom, staging lies at the top (staging_at), so the loads of a phase start as soon as the
// MMAs of the phase before are complete (loader_enter_phase) while its epilogue is still at work.  Who writes what another
// warp's staging of an earlier phase may occupy -- epilogue warps, and loaders above WGRAD_STAGING_AT -- first waits until
// every epilogue warp of the CTA has entered the phase.  A word per warp rather than an mbarrier: a pair may pass several
// phases at once.
__device__ __forceinline__ void epi_enter_phase(PipeBarriers* bars, int ew, int phase) {   // one lane
  __threadfence_block();
  *reinterpret_cast<volatile int*>(&bars->epi_phase[ew]) = phase;
}
__device__ __forceinline__ bool phase_wait(PipeBarriers* bars, int phase, const WaitCtl& wc) {   // one lane
  volatile int* c = bars->epi_phase;
  uint64_t t0 = 0;
  auto behind = [&]() {
    int least = phase;
#pragma unroll
    for (int w = 0; w < EPI_WARPS; ++w) least = min(least, c[w]);
    return least < phase;
  };
  for (uint32_t spin = 1; behind(); ++spin) {
    __nanosleep(100);
    if ((spin & 63u) == 0) {
      if (*reinterpret_cast<volatile int*>(&wc.status->abort)) return false;
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > wc.budget_ns) {
        report(wc.status, /*MOE_ERR_TIMEOUT*/ 2, (SITE_EMPTY << 24) | 0xFFFF00 | (phase & 0xFF));
        return false;
      }
    }
  }
  __threadfence_block();
  return true;
}

// A loader warp enters a phase with another ring: every stage of the old one has been multiplied (the commit that frees a
// stage also covers the A slots of a weight gradient).  Stages the old ring did not use pass at once.
__device__ __forceinline__ bool loader_enter_phase(PipeBarriers* bars, LoaderState& ls, int phase, const WaitCtl& wc) {
#pragma unroll 1
  for (int s = 0; s < MAX_STAGES; ++s)
    if (!mbar_wait_warp(&bars->empty[s], (ls.empty_par >> s) & 1, wc, SITE_EMPTY, phase, 50)) return false;
  ls.s = ls.a_s = 0;
  ls.guard = phase;
  return true;
}

// After a failed or aborted launch: let the tensor core finish what was issued before TMEM is freed.
__device__ __forceinline__ void issuer_drain(PipeBarriers* bars, DevStatus* status) {   // the issuing warp
  tc_commit_pair(&bars->drain);
  const WaitCtl shortwc{status, 20ull * 1000 * 1000};
  mbar_wait_warp(&bars->drain, 0, shortwc, SITE_DRAIN, 0);
}

// ---------------------------------------------------------------- per-tile trace (optional)
// One 32-byte record per traced interval: {t0, t1} in globaltimer ns, {role | phase << 8, item, CTA,
// ns from t0 until the dependencies were met}.
struct TraceCtl {
  uint4* buf;     // NULL: tracing off
  int cap;        // records
  int* cursor;
};
enum TraceRole : int { TR_SCHED = 0, TR_MMA = 1, TR_EPI = 2, TR_VEC = 3 };
__device__ __forceinline__ void trace_put(const TraceCtl& tr, int role, int phase, int item, uint64_t t0, uint64_t t_dep,
                                          uint64_t t1) {
  const int i = atomicAdd(tr.cursor, 1);
  if (i >= tr.cap) return;   // the cursor keeps counting: the host sees how many records were dropped
  tr.buf[2 * i] = make_uint4((uint32_t)t0, (uint32_t)(t0 >> 32), (uint32_t)t1, (uint32_t)(t1 >> 32));
  tr.buf[2 * i + 1] = make_uint4((uint32_t)(role | (phase << 8)), (uint32_t)item, blockIdx.x, (uint32_t)(t_dep - t0));
}

// ---------------------------------------------------------------- event policies
// No events: the one-launch-per-operator kernels (the kernel boundary orders the operators).
struct NoDeps {
  static constexpr bool kOn = false;
  __device__ __forceinline__ void signal(int, int) const {}
  __device__ __forceinline__ bool tracing() const { return false; }
  __device__ __forceinline__ void trace(int, int, uint64_t, uint64_t, uint64_t) const {}
};
// Event counters per M-block with static thresholds.
struct ChainDeps {
  static constexpr bool kOn = true;
  int* ctr;
  int wait_kind;             // dependent event of the phase's items
  const ChainParams* cp;     // (its thresholds)
  int trig_kind;             // trigger event (CTR_NONE: nothing consumes the phase's output inside the launch)
  int phase;
  WaitCtl wc;
  TraceCtl tr;
  // All lanes of a warp: wait until the counters of M-blocks [first, first + count), the first of them M-block `rel` of its
  // expert with `rows` rows, reach their thresholds.
  __device__ __forceinline__ bool wait(int first, int count, int rows, int rel, int lane, int item) const {
    int ok = 1;
    for (int q = lane; q < count; q += 32)
      if (!counter_wait(ctr + ctr_index(first + q, wait_kind), phase_wait_thr(*cp, phase, rows, rel + q), wc, item)) ok = 0;
    return __all_sync(0xffffffffu, ok) != 0;
  }
  // The same without waiting, by a group of `lanes` lanes of which this is lane `sub`: has this lane found its counters there?
  __device__ __forceinline__ bool met(int first, int count, int rows, int rel, int sub, int lanes) const {
    bool ok = true;
    for (int q = sub; q < count; q += lanes) {
      int v;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(ctr + ctr_index(first + q, wait_kind)) : "memory");
      if (v < phase_wait_thr(*cp, phase, rows, rel + q)) ok = false;
    }
    return ok;
  }
  // One lane, after its warp's stores of the tile are complete and ordered (see the epilogue roles).
  __device__ __forceinline__ void signal(int first, int count) const {
    if (trig_kind < 0) return;
    asm volatile("fence.acq_rel.gpu;" ::: "memory");   // one for all of them
    for (int q = 0; q < count; ++q)
      asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(ctr + ctr_index(first + q, trig_kind)) : "memory");
  }
  __device__ __forceinline__ bool tracing() const { return tr.buf != nullptr; }
  __device__ __forceinline__ void trace(int role, int item, uint64_t t0, uint64_t t_dep, uint64_t t1) const {
    trace_put(tr, role, phase, item, t0, t_dep, t1);
  }
};

// =====================================================================================================
// Token-column row-space operators (gemm_swap.cuh)
// =====================================================================================================
// Shared memory of an operator, from the 1024-byte aligned base: weights [stages][16 KB] | tokens [stages][tok_bytes], and at
// the end of LAYOUT_BYTES the staging.  What the token stages do not need goes into more stages: the products of a k-block of a
// small tile are over long before the loads of one are, so that the stages in flight bound the tile; and a
// pass over few tokens is a stream of weights from HBM (32 tokens: eleven stages, 198 KB in flight instead of 80).  The rings
// come from the host (schedule.h, ring_rows); the layout leaves the rows of the largest expert in meta[7] and what merges in
// meta[3], meta[4], and every role finds the same one.  (Worked out in the kernel for every item, passes of short items took 1-3 % longer; stages as large as their own tile,
// in a ring of bytes, cost the loaders more than the depth gave.)
// Against five stages in all of these, forward, medians of 12 runs in turn in three processes each, within 1 % of one another: 2048
// tokens x 8, 128 experts, 7168 x 2048: 2373 -> 2323 us (six); 2048 x 4, 128 experts, 4096 x 1536: 904 -> 864 (eight, no expert above
// 128 rows); 512 x 6 + 2, 64 experts, 2048 x 1408: 241 -> 233 (six).  One merged item takes a launch back to
// five.
constexpr size_t PIPE_BARRIER_BYTES = 384;
constexpr size_t TICKET_RING_BYTES = 640;   // of the persistent launch
constexpr size_t LAYOUT_BYTES = 227 * 1024 - 1024 - PIPE_BARRIER_BYTES - TICKET_RING_BYTES;
__host__ __device__ constexpr size_t swap_staging_bytes(GemmMode mode) { return EPI_WARPS * (size_t)sw_staging_bytes(mode); }
__host__ __device__ constexpr size_t staging_at(GemmMode mode) { return (LAYOUT_BYTES - swap_staging_bytes(mode)) & ~size_t(127); }
// The same for every role and item of a launch: the layout is complete before them.
__device__ __forceinline__ GemmArgs::Ring which_ring(const GemmArgs& a) {
  const int tiles = a.meta[3], items = a.meta[4], largest = a.meta[7];
  return a.ring[uniform(ring_choice(largest, a.ring_rows[0], a.ring_rows[1], tiles != items))];
}
// does stage s (its weights or its tokens) reach above WGRAD_STAGING_AT?
__device__ __forceinline__ bool above_guard(const GemmArgs::Ring& r, uint32_t s) {
  return (size_t)r.stages * W_STAGE_BYTES + (size_t)(s + 1) * r.tok_bytes > WGRAD_STAGING_AT ||
         (size_t)(s + 1) * W_STAGE_BYTES > WGRAD_STAGING_AT;
}
// TMA producers (both CTAs) of item t.  tok_warp = false: the weights and the stage's byte count; true: the
// tokens.
template <class DEP>
__device__ __forceinline__ bool swap_load_item(GemmMode mode, const GemmArgs& a, const GemmArgs::Ring ring, uint8_t* smem,
                                               PipeBarriers* bars, LoaderState& ls, bool tok_warp, int rank, int lane, const SwapWork& wk, int t,
                                               const WaitCtl& wc, const DEP& dep) {
  const int stages = ring.stages, tokb = ring.tok_bytes;
  uint8_t* sW = smem;                              // [stages][16 KB] weights
  uint8_t* sT = smem + stages * W_STAGE_BYTES;     // [stages][tokb] tokens (this CTA's half)
  // with events: the tokens are there (acquired by the scheduler and handed on through the ticket ring, or by the caller);
  // what the producers wrote must be seen by the TMA loads
  if (DEP::kOn && tok_warp) fence_proxy_async_global();
  const int nkb = uniform(wk.nkb), e = uniform(wk.e), n0 = uniform(wk.n0);
  const int row_a = uniform(wk.row0), half_a = uniform(wk.ntok) >> 1;
  const int row_b = row_a + 2 * half_a, half_b = uniform(wk.ntok_b) >> 1;
  for (int kb = 0; kb < nkb; ++kb) {
    if (!mbar_wait_warp(&bars->empty[ls.s], (ls.empty_par >> ls.s) & 1, wc, SITE_EMPTY, t, 50)) return false;
    ls.empty_par ^= 1u << ls.s;
    if (DEP::kOn && ls.guard && above_guard(ring, ls.s)) {   // a weight gradient's staging may still be in use there
      if (!uniform(lane == 0 ? (int)phase_wait(bars, ls.guard, wc) : 1)) return false;
      ls.guard = 0;
    }
    if (!tok_warp) {
      load_weights_swap(mode, a, e, n0, kb, rank, sW + ls.s * W_STAGE_BYTES, &bars->full[ls.s], 2 * (half_a + half_b));
    } else {
      load_tokens_swap(a, row_a, half_a, kb, rank, sT + ls.s * tokb, &bars->full[ls.s]);
      if (half_b)   // the second token tile, behind the first in the stage
        load_tokens_swap(a, row_b, half_b, kb, rank, sT + ls.s * tokb + half_a * (BK * 2), &bars->full[ls.s]);
    }
    if (++ls.s == (uint32_t)stages) ls.s = 0;
  }
  return true;
}

// The issuer takes columns for an item of n0 (+ n1) columns: what they overlap has been drained when this returns.  Its slots are
// 2 * is.end and, for the second tile, the one behind; the caller flips is.end.
__device__ __forceinline__ bool acc_claim(PipeBarriers* bars, IssuerState& is, int n0, int n1, const WaitCtl& wc, int t) {
  uint32_t need = 3u << (2 * is.end);   // the item before the last, at the same end
  if (is.before_n + n0 + n1 > TMEM_COLS) need |= 1u << (2 * (is.end ^ 1));   // and the tile in the middle of the last
  need &= is.busy;
#pragma unroll 1
  while (need) {
    const int slot = __ffs(need) - 1;
    if (!mbar_wait_warp(&bars->tmem_empty[slot], (is.acc_par >> slot) & 1, wc, SITE_TMEM_EMPTY, t)) return false;
    is.acc_par ^= 1u << slot;
    is.busy &= ~(1u << slot);
    need &= need - 1;
  }
  is.busy |= (n1 ? 3u : 1u) << (2 * is.end);
  is.before_n = n0 + n1;
  return true;
}

// MMA issuer: warp 1 of the even CTA.  The whole warp walks the loop with uniform control flow and operands; one elected
// lane issues (common.cuh).
template <bool W_MN, class DEP>
__device__ __forceinline__ bool swap_issue_item(const GemmArgs::Ring ring, uint8_t* smem, PipeBarriers* bars, uint32_t tmem_base,
                                                IssuerState& is, const SwapWork& wk, int t, const WaitCtl& wc,
                                                const DEP& dep) {
  const uint32_t stages = ring.stages, t_step = ring.tok_bytes >> 4;
  const uint32_t w_lo0 = swap_w_desc_lo<W_MN>(smem_u32(smem));
  const uint32_t t_lo0 = smem_desc_lo(smem_u32(smem + stages * W_STAGE_BYTES), 16);
  uint32_t w_lo = w_lo0 + is.s * (W_STAGE_BYTES >> 4), t_lo = t_lo0 + is.s * t_step;
  const int nkb = uniform(wk.nkb), ntok = uniform(wk.ntok), ntok_b = uniform(wk.ntok_b);
  // a merged item's second tile is the larger one: the first in the accumulators
  const int n0 = ntok_b ? ntok_b : ntok, n1 = ntok_b ? ntok : 0;
  if (!acc_claim(bars, is, n0, n1, wc, t)) return false;
  tc_fence_after_sync();
  const uint32_t d_first = uniform(tmem_base + acc_column(is.end, 0, n0, n1));
  const uint32_t d_tmem = uniform(ntok_b ? tmem_base + acc_column(is.end, 1, n0, n1) : d_first);
  const uint32_t idesc = swap_idesc<W_MN>(ntok), idesc_b = swap_idesc<W_MN>(ntok_b ? ntok_b : TOK_GRAIN);
  const uint32_t t_off_b = (uint32_t)((ntok >> 1) * (BK * 2)) >> 4;
  uint64_t t0 = 0;
  for (int kb = 0; kb < nkb; ++kb) {
    if (!mbar_wait_warp(&bars->full[is.s], (is.full_par >> is.s) & 1, wc, SITE_FULL, t)) return false;
    is.full_par ^= 1u << is.s;
    if (DEP::kOn && kb == 0 && dep.tracing()) t0 = globaltimer_ns();
    tc_fence_after_sync();
    mma_kblock_swap<W_MN>(d_tmem, w_lo, t_lo, idesc, kb == 0);
    if (ntok_b) mma_kblock_swap<W_MN>(d_first, w_lo, t_lo + t_off_b, idesc_b, kb == 0);
    tc_commit_pair(&bars->empty[is.s]);   // frees the stage in both CTAs
    if (++is.s == stages) {
      is.s = 0; w_lo = w_lo0; t_lo = t_lo0;
    } else {
      w_lo += W_STAGE_BYTES >> 4; t_lo += t_step;
    }
  }
  tc_commit_pair(&bars->tmem_full[2 * is.end]);  // accumulator slices ready in both CTAs
  if (ntok_b) tc_commit_pair(&bars->tmem_full[2 * is.end + 1]);
  is.end ^= 1;
  if (DEP::kOn && dep.tracing() && (threadIdx.x & 31) == 0) dep.trace(TR_MMA, t, t0, t0, globaltimer_ns());
  return true;
}

// Epilogue warps (both CTAs, own features).  With events: the CTA's last warp to finish a tile signals its M-blocks.  Its
// release at GPU scope covers what the other warps stored before they counted themselves; the consumer's fence.proxy.async
// makes it visible to its TMA loads.  When every warp released its own stores, each waited 4-6 us for all of the SM's to
// drain, longer than the work on the tile (1777 tokens: 10 us a gate+up tile, 3 of them work).
template <int MODE, class DEP>
__device__ __forceinline__ bool swap_epilogue_item(const GemmArgs& a, uint8_t* smem, PipeBarriers* bars,
                                                   uint32_t tmem_base, EpiState& es, int rank, int ew, int lane,
                                                   const SwapWork& wk, int t, const WaitCtl& wc, const DEP& dep) {
  uint8_t* staging = smem + staging_at((GemmMode)MODE) + ew * sw_staging_bytes((GemmMode)MODE);
  const bool merged = wk.ntok_b != 0;
  for (int part = 0; part < (merged ? 2 : 1); ++part) {   // a merged item is two tiles here, the larger one -- the second -- first
    SwapTile st{wk.row0, wk.ntok, wk.n0, wk.nb};
    int acc = acc_column(es.end, 0, st.ntok, 0);
    if (merged) {
      acc = acc_column(es.end, part, wk.ntok_b, wk.ntok);
      if (part == 0) { st.row0 += wk.ntok; st.ntok = wk.ntok_b; }
    }
    const int as = 2 * es.end + part;
    uint64_t t0 = 0;
    auto ready = [&]() {
      if (!mbar_wait_warp(&bars->tmem_full[as], (es.full_par >> as) & 1, wc, SITE_TMEM_FULL, t, 200)) return false;
      if (DEP::kOn && ew == 0 && lane == 0 && dep.tracing()) t0 = globaltimer_ns();
      __syncwarp();
      tc_fence_after_sync();
      return true;
    };
    if (!epilogue_swap<MODE>(a, st, tmem_base + acc, rank, ew, lane, staging, ready)) return false;
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) {
      bool last = false;
      if (DEP::kOn) {
        // counted before the accumulator is given back: the next tile of the slot, which uses this counter again, follows
        int before;
        asm volatile("atom.acq_rel.cta.shared::cta.add.s32 %0, [%1], 1;" : "=r"(before) : "r"(smem_u32(&bars->epi_done[as])) : "memory");
        last = before == EPI_WARPS - 1;
        if (last) *reinterpret_cast<volatile int*>(&bars->epi_done[as]) = 0;
      }
      mbar_arrive_leader(&bars->tmem_empty[as]);
      if (DEP::kOn) {
        if (last) dep.signal(st.row0 / BLOCK_M, mblocks_of(st.ntok));
        if (ew == 0 && dep.tracing()) dep.trace(TR_EPI, t, t0, t0, globaltimer_ns());
      }
    }
    es.full_par ^= 1u << as;
    __syncwarp();
  }
  es.end ^= 1;
  return true;
}

// =====================================================================================================
// Weight gradients, strip by strip, the strip's A operand resident in shared memory
// =====================================================================================================
// dW[e] (M x N) = P_e^T . Q_e with K = the expert's rows: at a few hundred rows per expert a 256 x 256
// tile reads 320 KB of operands for 128 KB of output.  A pair therefore takes a whole strip (its 256
// rows of dW across all column tiles) and loads the strip's A operand (this CTA's 128 columns of P_e,
// all K rows) once: when the expert has at most A_RES_KB k-blocks it stays in the five 16 KB A slots for
// every column tile of the strip, and only the B operand streams through the stage ring.  Longer
// experts stream A through the same slots stage by stage.  An A slot is refilled only after the MMAs
// that read its previous content have completed (a_empty, one commit per content).
//
// With K of only four or five k-blocks a column tile lasts about as long as the latency of its B loads, so the
// B ring is deeper than one tile (WG_B_STAGES): the loads of tile i + 1 are in flight while tile i multiplies.
// The staging of the epilogue is what pays for it: one 4 KB box of 32 rows x 64 columns per warp.
constexpr int A_RES_KB = WG_A_SLOTS;         // k-blocks of A that can stay resident
constexpr size_t WGRAD_LAYOUT_BYTES = WGRAD_STAGING_AT + EPI_WARPS * OUT_BOX_BYTES;
// the weight gradients' operands never touch the staging of a row-space operator in front of them
static_assert(WGRAD_STAGING_AT <= staging_at(GEMM_ACT_GRAD) && WGRAD_STAGING_AT <= staging_at(GEMM_GATE_GRAD), "phase overlap");

// Epilogue of one 128 x 256 accumulator slice of a weight gradient (or zeros for an expert without rows): warps `quad`
// and `quad + 4` store 32 rows, 64 columns at a time in turn, each through a staging box of its own.
__device__ __forceinline__ void epilogue_wgrad_tile(const GemmArgs& a, const Tile& tl, uint32_t tmem_acc, int ew, int lane,
                                                    uint8_t* box) {
  const int quad = ew & 3;
  const uint32_t trow = tmem_acc + (static_cast<uint32_t>(quad * 32) << 16);
  const int y0 = tl.m0 + quad * 32;
  if (y0 >= a.M) return;
#pragma unroll 1
  for (int c0 = (ew >> 2) * 64; c0 < BN; c0 += 128) {
    if (tl.n0 + c0 >= a.N) break;
    float v[64];
    if (tl.nkb == 0) {
#pragma unroll
      for (int i = 0; i < 64; ++i) v[i] = 0.f;
    } else {
      // 64 columns per TMEM round trip (one wait per box)
#pragma unroll
      for (int q = 0; q < 4; ++q) tmem_ld16(trow + c0 + 16 * q, v + 16 * q);
      tmem_ld_wait();
    }
    if (lane == 0) tma_store_wait_read();   // the box's previous store has read it
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 64; h += 8) stage8(box, lane, h >> 3, v + h);
    staging_release();
    if (lane == 0) {
      tma_store_3d(&a.tmOut0, tl.n0 + c0, y0, tl.e, box);
      tma_store_commit();
    }
  }
}

struct Strip {
  int e, mp, row0, nkb, rows;   // expert, 256-row block of dW, first padded row, k-blocks, rows of the expert
  int nb0, nb1;                 // column tiles
  __device__ __forceinline__ int m0(int rank) const { return (2 * mp + rank) * BLOCK_M; }   // this CTA's 128 rows
};
__device__ __forceinline__ int wgrad_strips(const GemmArgs& a) {
  return strip_items(a.Ep, (a.n_tiles_m + 1) / 2, a.n_tiles_n, a.split, a.meta[6]);
}
// Item s of the operator (schedule.h).  Strips are expert-major, so the pairs working at the same time share the expert's
// B operand in L2.
__device__ __forceinline__ Strip decode_strip(const GemmArgs& a, int s) {
  const StripItem it = decode_strip_item(s, (a.n_tiles_m + 1) / 2, a.n_tiles_n, a.split, a.meta[6], a.wg_order);
  Strip st;
  st.e = it.e;
  st.mp = it.strip;
  st.nb0 = it.nb0;
  st.nb1 = it.nb1;
  st.row0 = a.mb_start[st.e] * BLOCK_M;
  st.rows = a.counts[st.e];
  st.nkb = (st.rows + BK - 1) / BK;
  return st;
}

// TMA producers (both CTAs) of strip sp.  b_warp = false: A (and the stage's byte count); true: B.
template <class DEP>
__device__ __forceinline__ bool wgrad_load_strip(const GemmArgs& a, uint8_t* smem, PipeBarriers* bars, LoaderState& ls,
                                                 bool b_warp, int rank, int lane, const Strip& st, int sp,
                                                 const WaitCtl& wc, const DEP& dep) {
  uint8_t* sA = smem;                                   // [WG_A_SLOTS][16 KB] A slots
  uint8_t* sB = smem + WG_A_SLOTS * A_STAGE_BYTES;     // [WG_B_STAGES][16 KB] B stages
  const int m0 = uniform(st.m0(rank)), row0 = uniform(st.row0), nkb = uniform(st.nkb);
  const bool resident = nkb <= A_RES_KB;
  if (DEP::kOn) fence_proxy_async_global();   // as in swap_load_item
  const int nb0 = uniform(st.nb0), nb1 = uniform(st.nb1);
  for (int nb = nb0; nb < nb1; ++nb) {
    const bool load_a = !resident || nb == nb0;
    for (int kb = 0; kb < nkb; ++kb) {
      const int slot = resident ? kb : (int)ls.a_s;
      if (!mbar_wait_warp(&bars->empty[ls.s], (ls.empty_par >> ls.s) & 1, wc, SITE_EMPTY, sp, 50)) return false;
      if (!b_warp && load_a && !mbar_wait_warp(&bars->a_empty[slot], (ls.a_ph >> slot) & 1, wc, SITE_EMPTY, sp, 50)) return false;
      const int k0 = row0 + kb * BK;
      if (!b_warp) {
        if (rank == 0) mbar_expect_tx_elect(&bars->full[ls.s], 2 * (HALF_B_BYTES + (load_a ? A_STAGE_BYTES : 0)));
        if (load_a) {
          tma_load_2d_pair(sA + slot * A_STAGE_BYTES, &a.tmA, m0, k0, &bars->full[ls.s]);
          tma_load_2d_pair(sA + slot * A_STAGE_BYTES + MN_BOX_BYTES, &a.tmA, m0 + 64, k0, &bars->full[ls.s]);
        }
      } else {
        tma_load_2d_pair(sB + ls.s * HALF_B_BYTES, &a.tmB, nb * BN + 2 * rank * 64, k0, &bars->full[ls.s]);
        tma_load_2d_pair(sB + ls.s * HALF_B_BYTES + MN_BOX_BYTES, &a.tmB, nb * BN + (2 * rank + 1) * 64, k0, &bars->full[ls.s]);
      }
      ls.empty_par ^= 1u << ls.s;
      if (load_a) ls.a_ph ^= 1u << slot;
      if (!resident && ++ls.a_s == WG_A_SLOTS) ls.a_s = 0;
      if (++ls.s == WG_B_STAGES) ls.s = 0;
    }
  }
  return true;
}

template <class DEP>
__device__ __forceinline__ bool wgrad_issue_strip(const GemmArgs& a, uint8_t* smem, PipeBarriers* bars, uint32_t tmem_base,
                                                  IssuerState& is, const Strip& st, int sp, const WaitCtl& wc,
                                                  const DEP& dep) {
  const uint32_t a_lo0 = smem_desc_lo(smem_u32(smem), MN_BOX_BYTES);
  const uint32_t b_lo0 = smem_desc_lo(smem_u32(smem + WG_A_SLOTS * A_STAGE_BYTES), MN_BOX_BYTES);
  constexpr uint32_t idesc = make_idesc_bf16(2 * BLOCK_M, BN, 1, 1), hi = smem_desc_hi(1024);
  constexpr int KSTEP = 2048 >> 4;   // 16 k-rows of an MN-major box
  const int nkb = uniform(st.nkb), rows = uniform(st.rows);
  const bool resident = nkb <= A_RES_KB;
  if (nkb == 0) return true;
  uint64_t t0 = 0;
  const int nb0 = uniform(st.nb0), nb1 = uniform(st.nb1);
  for (int nb = nb0; nb < nb1; ++nb) {
    if (!acc_claim(bars, is, BN, 0, wc, sp)) return false;
    tc_fence_after_sync();
    const uint32_t d_tmem = uniform(tmem_base + acc_column(is.end, 0, BN, 0));
    const bool last_use = !resident || nb == nb1 - 1;
    for (int kb = 0; kb < nkb; ++kb) {
      if (!mbar_wait_warp(&bars->full[is.s], (is.full_par >> is.s) & 1, wc, SITE_FULL, sp)) return false;
      is.full_par ^= 1u << is.s;
      if (DEP::kOn && nb == nb0 && kb == 0 && dep.tracing()) t0 = globaltimer_ns();
      tc_fence_after_sync();
      const int slot = resident ? kb : (int)is.a_s;
      const uint32_t a_lo = a_lo0 + slot * (A_STAGE_BYTES >> 4), b_lo = b_lo0 + is.s * (HALF_B_BYTES >> 4);
      // the last k-block may hold fewer than 64 rows of the expert: the 16-row steps that would only multiply
      // zero padding are not issued
      const int steps = k16_steps_of(rows, kb);
      if (steps == BK / 16) {
        tc_mma4_bf16_pair<KSTEP, KSTEP>(d_tmem, a_lo, b_lo, hi, idesc, kb != 0);
      } else {
        for (int k16 = 0; k16 < steps; ++k16)
          tc_mma1_bf16_pair(d_tmem, a_lo + k16 * KSTEP, b_lo + k16 * KSTEP, hi, idesc, kb != 0 || k16 != 0);
      }
      tc_commit_pair(&bars->empty[is.s]);
      if (last_use) tc_commit_pair(&bars->a_empty[slot]);
      if (!resident && ++is.a_s == WG_A_SLOTS) is.a_s = 0;
      if (++is.s == WG_B_STAGES) is.s = 0;
    }
    tc_commit_pair(&bars->tmem_full[2 * is.end]);
    is.end ^= 1;
  }
  if (DEP::kOn && dep.tracing() && (threadIdx.x & 31) == 0) dep.trace(TR_MMA, sp, t0, t0, globaltimer_ns());
  return true;
}

template <class DEP>
__device__ __forceinline__ bool wgrad_epilogue_strip(const GemmArgs& a, uint8_t* smem, PipeBarriers* bars,
                                                     uint32_t tmem_base, EpiState& es, int rank, int ew, int lane,
                                                     const Strip& st, int sp, const WaitCtl& wc, const DEP& dep) {
  uint8_t* box = smem + WGRAD_STAGING_AT + ew * OUT_BOX_BYTES;
  Tile tl;
  tl.e = st.e; tl.m0 = st.m0(rank); tl.nkb = st.nkb;
  const bool idle = tl.m0 >= a.M;   // the strip's second half lies outside dW: nothing to store
  bool ok = true;
  uint64_t t0 = 0;
  if (DEP::kOn && ew == 0 && lane == 0 && dep.tracing()) t0 = globaltimer_ns();
  for (int nb = st.nb0; nb < st.nb1; ++nb) {
    tl.n0 = nb * BN;
    if (st.nkb == 0) {
      if (!idle) epilogue_wgrad_tile(a, tl, 0, ew, lane, box);  // an expert without rows: zeros
      continue;
    }
    const int as = 2 * es.end;
    if (!mbar_wait(&bars->tmem_full[as], (es.full_par >> as) & 1, wc, SITE_TMEM_FULL, sp, 200)) { ok = false; break; }
    tc_fence_after_sync();
    if (!idle) epilogue_wgrad_tile(a, tl, tmem_base + acc_column(es.end, 0, BN, 0), ew, lane, box);
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive_leader(&bars->tmem_empty[as]);
    es.full_par ^= 1u << as;
    es.end ^= 1;
  }
  if (DEP::kOn && ew == 0 && lane == 0 && dep.tracing()) dep.trace(TR_EPI, sp, t0, t0, globaltimer_ns());
  return ok;
}

}  // namespace moe
