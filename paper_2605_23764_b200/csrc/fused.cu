// The single persistent, dependency-driven launch of the forward (and of the backward) layer.
//
// One grid of one CTA per SM in clusters of two runs the whole operator chain.  Per CTA:
//   warp 0      TMA producer of the weights (weight gradients: of the A operand)
//   warp 1      tcgen05.mma issuer (even CTA) and TMEM owner
//   warps 2-5, 8-11  epilogue: TMEM -> fused element-wise math -> global memory, then the tile's trigger event
//   warp 6      TMA producer of the tokens (weight gradients: of the B operand)
//   warp 7      even CTA: scheduler of the pair -- takes the next tickets of the matrix queue, looks at the
//               items' dependent events and publishes the items to the other roles, met or not; odd CTA: vector worker
//   warps 12-15 vector workers: tickets of the vector queue (permute-gather, routing-weight
//               gradient, combine); the matrix-role warps join them once the matrix queue is empty.
// The matrix roles are the ones of the one-launch-per-operator kernels (gemm_roles.cuh); here they
// take the items of all operators of the pass from one ticket queue (schedule.h) with the pipeline
// state carried from item to item, so that no SM waits at an operator boundary for the others, the
// permutes run beside the GEMMs, and what orders tiles are event counters with static thresholds --
// the paper's unified runtime (Sections 4.3, 4.4) restated for one SM, where "matrix core" and
// "vector core" are warp roles of the same CTA.
#include "gemm_roles.cuh"
#include "launch_pairs.cuh"
#include "schedule.h"
#include "topk.cuh"

namespace moe {

constexpr int SCHED_WARP = 7;   // even CTA: scheduler of the pair; odd CTA: a vector worker
constexpr int VEC_WARPS = 4;
constexpr int FUSED_THREADS = 32 * (GEMM_ROLE_WARPS + VEC_WARPS);

static_assert(GATHER_ROWS == 4, "vec_gather");
constexpr size_t FUSED_SMEM_BYTES = 1024 + LAYOUT_BYTES + PIPE_BARRIER_BYTES + TICKET_RING_BYTES;
static_assert(WGRAD_LAYOUT_BYTES <= LAYOUT_BYTES && FUSED_SMEM_BYTES <= 227 * 1024, "shared memory budget");

// ---------------------------------------------------------------- vector work (one warp per task)
__device__ __forceinline__ uint4 ldg_nc_v4(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
// data written earlier in this launch by other SMs: read at L2
__device__ __forceinline__ uint4 ldg_cg_v4(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Dispatch / backward Dispatch: GATHER_ROWS rows of one 32-row group of an expert.  The rows' slots and place are two
// independent loads by group; then the rows are copied together: 16 independent 16-byte loads in flight per lane.
// Returns the rows' M-block.
__device__ __forceinline__ int vec_gather(const FusedArgs& fa, int task, int lane) {
  const int g = task / GATHER_SUB, sub = (task - g * GATHER_SUB) * GATHER_ROWS;
  const LayoutView& lv = fa.lv;
  const int4 sl = *reinterpret_cast<const int4*>(lv.group_slot + (size_t)g * GROUP_ROWS + sub);
  const int p0 = lv.group_row[g] + sub;
  const int slots[GATHER_ROWS] = {sl.x, sl.y, sl.z, sl.w};
  const int nvec = fa.d >> 3;
  const int k = fa.cp.k;
  const uint4* in[GATHER_ROWS];
#pragma unroll
  for (int r = 0; r < GATHER_ROWS; ++r) {
    in[r] = nullptr;
    if (slots[r] >= 0) in[r] = reinterpret_cast<const uint4*>(fa.gather_src + (size_t)(slots[r] / fa.kp) * fa.d);
  }
  float w = 0.0f;   // routing weight, a lane per row (padding rows: 0); stored behind the rows, nothing waits for the load
  if (fa.prow_w && lane < GATHER_ROWS) {
    const int slot = lane == 0 ? slots[0] : lane == 1 ? slots[1] : lane == 2 ? slots[2] : slots[3];
    if (slot >= 0) {
      const int t = slot / fa.kp, j = slot - t * fa.kp;
      w = j < k ? fa.topk_w[(size_t)t * k + j] : 1.0f;
    }
  }
  const int ldv = row_ld(fa.d) >> 3;
  uint4* out = reinterpret_cast<uint4*>(fa.gather_dst) + (size_t)p0 * ldv;
  constexpr int U = 16 / GATHER_ROWS;
  for (int v = lane; v < nvec; v += 32 * U) {
    uint4 q[GATHER_ROWS][U];
#pragma unroll
    for (int r = 0; r < GATHER_ROWS; ++r)
#pragma unroll
      for (int u = 0; u < U; ++u)
        q[r][u] = (in[r] && v + 32 * u < nvec) ? ldg_nc_v4(in[r] + v + 32 * u) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int r = 0; r < GATHER_ROWS; ++r)
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (v + 32 * u < nvec) out[(size_t)r * ldv + v + 32 * u] = q[r][u];   // padding rows are zero-filled
  }
  if (fa.prow_w && lane < GATHER_ROWS) fa.prow_w[p0 + lane] = w;
  return p0 / BLOCK_M;
}

// Combine / backward Combine of one token, or of one of its column chunks.  Dependent events: `done` of every M-block that
// holds one of the token's rows (many-to-many, Section 4.3): each lane polls the counter of one row.
__device__ __forceinline__ bool vec_combine(const FusedArgs& fa, int task, int lane, const WaitCtl& wc) {
  const int kp = fa.kp, split = fa.cp.combine_split;
  const int thr = thr_done(fa.cp);
  const int i = task / split, chunk = task - i * split;
  const int per = (((fa.d >> 3) + split - 1) / split + 31) & ~31;   // vectors of a chunk
  const int v0 = chunk * per, nvec = min(fa.d >> 3, v0 + per);
  {
    const int t = fa.lv.combine_order ? fa.lv.combine_order[i] : i;   // tokens in the order in which their last row is produced
    const int* prow = fa.lv.prow_of + (size_t)t * kp;
    if (fa.d_topk_w && chunk == 0)   // a slot dropped for an invalid expert id has no row: its weight's gradient is zero
      for (int j = lane; j < fa.cp.k; j += 32)
        if (prow[j] < 0) fa.d_topk_w[(size_t)t * fa.cp.k + j] = 0.f;
    // dependent events: `done` of every M-block that holds one of the token's rows
    int ok = 1;
    for (int j = lane; j < kp; j += 32) {
      const int p = prow[j];
      if (p >= 0 && !counter_wait(fa.ctr + ctr_index(p / BLOCK_M, CTR_DONE), thr, wc, task, 2048)) ok = 0;
    }
    if (!__all_sync(0xffffffffu, ok)) return false;
    // two vector positions per lane and step: sixteen independent row loads in flight (a warp alone is latency-bound)
    for (int v = v0 + lane; v < nvec; v += 64) {
      const bool two = v + 32 < nvec;
      float acc[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[q] = 0.f;
      for (int j0 = 0; j0 < kp; j0 += 8) {
        uint4 r[8], r2[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int j = j0 + u;
          const int p = j < kp ? prow[j] : -1;
          const uint4* row = reinterpret_cast<const uint4*>(fa.combine_rows + (size_t)(p >= 0 ? p : 0) * row_ld(fa.d));
          r[u] = p >= 0 ? ldg_cg_v4(row + v) : make_uint4(0, 0, 0, 0);
          r2[u] = (p >= 0 && two) ? ldg_cg_v4(row + v + 32) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          acc[0] += bf16lo(r[u].x); acc[1] += bf16hi(r[u].x);
          acc[2] += bf16lo(r[u].y); acc[3] += bf16hi(r[u].y);
          acc[4] += bf16lo(r[u].z); acc[5] += bf16hi(r[u].z);
          acc[6] += bf16lo(r[u].w); acc[7] += bf16hi(r[u].w);
          acc[8] += bf16lo(r2[u].x); acc[9] += bf16hi(r2[u].x);
          acc[10] += bf16lo(r2[u].y); acc[11] += bf16hi(r2[u].y);
          acc[12] += bf16lo(r2[u].z); acc[13] += bf16hi(r2[u].z);
          acc[14] += bf16lo(r2[u].w); acc[15] += bf16hi(r2[u].w);
        }
      }
      uint4 o;
      o.x = pack_bf16x2(acc[0], acc[1]);
      o.y = pack_bf16x2(acc[2], acc[3]);
      o.z = pack_bf16x2(acc[4], acc[5]);
      o.w = pack_bf16x2(acc[6], acc[7]);
      reinterpret_cast<uint4*>(fa.combine_out + (size_t)t * fa.d)[v] = o;
      if (two) {
        o.x = pack_bf16x2(acc[8], acc[9]);
        o.y = pack_bf16x2(acc[10], acc[11]);
        o.z = pack_bf16x2(acc[12], acc[13]);
        o.w = pack_bf16x2(acc[14], acc[15]);
        reinterpret_cast<uint4*>(fa.combine_out + (size_t)t * fa.d)[v + 32] = o;
      }
    }
  }
  return true;
}

// Routing-weight gradient of the rows of one M-block: the act_grad epilogues left partial dot products
// per (row, column tile, CTA, warp); summed here in a fixed order.  Dependent event: `activated`.
__device__ __forceinline__ bool vec_dw(const FusedArgs& fa, int mb, int lane, const WaitCtl& wc) {
  int ok = 1;
  if (lane == 0) ok = counter_wait(fa.ctr + ctr_index(mb, CTR_ACTIVATED), thr_activated(fa.cp), wc, mb, 4096) ? 1 : 0;
  if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
  const LayoutView& lv = fa.lv;
  const int e = lv.mblk_expert[mb];
  const int cnt = lv.counts[e], local0 = mb * BLOCK_M - lv.pad_off[e], off0 = lv.offsets[e];
  const int k = fa.cp.k;
  for (int r = lane; r < BLOCK_M; r += 32) {
    const int local = local0 + r;
    if (local >= cnt) continue;
    const int slot = lv.src_of[off0 + local];
    const int t = slot / fa.kp, j = slot - t * fa.kp;
    if (j >= k) continue;   // a shared expert's row: its weight is the constant 1
    const float* part = fa.dw_partial + (size_t)(mb * BLOCK_M + r) * fa.dw_nparts;
    float s = 0.f;
    for (int q = 0; q < fa.dw_nparts; ++q) s += __ldcg(part + q);
    fa.d_topk_w[(size_t)t * k + j] = s;
  }
  return true;
}

// Vector workers.  The first gather_fast_tasks() gather tasks -- what the first matrix items of every
// pair wait for -- are taken by every worker; after that fa.gatherers warps per CTA keep gathering,
// a few M-blocks' worth of traffic at a time, well ahead of the matrix queue but far below the bandwidth the
// GEMMs need: a gather at full speed takes its bytes from the loads of the matrix tiles and slows them by more
// than it saves.  The other workers go on to the second queue and sleep on its dependent events.
__device__ __forceinline__ void vector_worker_loop(const FusedArgs& fa, const WaitCtl& wc, const TraceCtl& tr, int M,
                                                   int lane, bool background_gatherer) {
  if (*reinterpret_cast<volatile int*>(&fa.status->abort)) return;
  const int ngather = gather_total(fa.lv.meta[5]), fast = gather_fast_tasks(fa.d);
  // with shared experts the gather starts at their first row, like the matrix queue (schedule.h, rotate_index)
  const int S = fa.cp.kp - fa.cp.k;
  const int gather_first = S > 0 ? fa.lv.group_start[fa.cp.Ep - S] * GATHER_SUB : 0;
  while (true) {
    int t = ngather;
    if (lane == 0) {
      const int seen = *reinterpret_cast<volatile int*>(&fa.ctr[CTR_VEC_TICKET]);
      if (seen < ngather && (background_gatherer || seen < fast)) t = atomicAdd(&fa.ctr[CTR_VEC_TICKET], 1);
    }
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= ngather) break;
    t = rotate_index(t, gather_first, ngather);
    uint64_t t0 = 0;
    if (tr.buf && lane == 0) t0 = globaltimer_ns();
    const int mb = vec_gather(fa, t, lane);
    __syncwarp();
    if (lane == 0) {
      counter_signal(fa.ctr + ctr_index(mb, CTR_GATHERED), 1);
      if (tr.buf) trace_put(tr, TR_VEC, VEC_GATHER, t, t0, t0, globaltimer_ns());
    }
  }
  const int npost = post_total(fa.cp, M), dw_first = S > 0 ? fa.lv.mb_start[fa.cp.Ep - S] : 0;
  while (true) {
    int t = 0;
    if (lane == 0) t = atomicAdd(&fa.ctr[CTR_POST_TICKET], 1);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= npost) break;
    VecTask v = decode_post_ticket(fa.cp, t, M);
    if (v.op == VEC_DW) v.idx = rotate_index(v.idx, dw_first, M);   // in the order act_grad produces them
    uint64_t t0 = 0;
    if (tr.buf && lane == 0) t0 = globaltimer_ns();
    const bool ok = v.op == VEC_COMBINE ? vec_combine(fa, v.idx, lane, wc) : vec_dw(fa, v.idx, lane, wc);
    if (tr.buf && lane == 0) trace_put(tr, TR_VEC, v.op, v.idx, t0, t0, globaltimer_ns());
    if (!ok) break;
    if (fa.announce_out && v.op == VEC_COMBINE) {
      // Host-buffer calls: the result may leave for the host as soon as its last row is written, while the
      // launch still computes weight gradients.  The warp's stores, then a device-wide fence, then the count;
      // whoever finishes the last task publishes the word the copy-out stream waits for.
      __syncwarp();
      if (lane == 0) {
        __threadfence();
        if (atomicAdd(&fa.ctr[CTR_COMBINE_DONE], 1) + 1 == combine_total(fa.cp)) {
          __threadfence_system();
          *reinterpret_cast<volatile int*>(&fa.ctr[CTR_OUT_READY]) = 1;
        }
      }
    }
  }
}

// ---------------------------------------------------------------- matrix queue: tickets of a CTA pair
// The matrix queue is the concatenation of the phases' item lists (schedule.h); pairs take tickets with
// one atomic counter.  Tickets are handed out in time order, so the ~74 items in flight are always a
// contiguous window of the queue: items that share an operand (the token tiles of one expert and
// column tile share its weight slab, the strips of one expert share its rows) start within
// microseconds of each other and meet in L2, however the pairs' speeds differ -- a static deal of
// items to pairs loses that as soon as gather or combine traffic makes the pairs drift apart.
// The scheduler warp of the even CTA takes the pair's tickets -- a few items ahead of the epilogue (sched_hold) --
// looks at the items' dependent events and publishes the items to every role of both CTAs through a small ring in shared
// memory: ticket, decode and look hide behind the loads of the items before.  If the events are not met yet, whoever loads what they stand for waits for
// them (the token loader; both loaders of a weight gradient): the weights, which depend on nothing, are under way meanwhile.
constexpr int TK_RING = 8;
// A published item: the ticket and the decoded work (decoding takes a chain of dependent global loads; the
// scheduler does it once, ahead of time, for every role of both CTAs).
struct __align__(16) WorkDesc {
  int ticket;                                  // -1: the queue is empty
  int phase, item, flags;                      // WD_READY
  int e, n0, nb, nkb;                          // strips: nb = 256-row block of dW, n0 = first column tile
  int row0, ntok, ntok_b, nb1;                 // strips: ntok = rows of the expert, ntok_b = 0, nb1 = end of the column tiles
  __device__ __forceinline__ int mb_first() const { return row0 / BLOCK_M; }              // M-blocks of the item's rows
  __device__ __forceinline__ int mb_count() const { return mblocks_of(ntok + ntok_b); }
};
constexpr int WD_READY = 1;   // the dependent events were met when the item was published
constexpr int WD_PIECES = 3;
static_assert(sizeof(WorkDesc) == 16 * WD_PIECES, "published as 16-byte stores");
struct __align__(16) TicketRing {
  WorkDesc work[TK_RING];
  uint64_t full[TK_RING];    // in each CTA: the slot holds an item
  uint64_t empty[TK_RING];   // used in the even CTA: every consumer of both CTAs has read the slot
};
// consumers: in each CTA both loaders and the epilogue warps, plus the MMA issuer of the even CTA
constexpr int TK_CONSUMERS = 2 * (2 + EPI_WARPS) + 1;

// The scheduler's `batch` groups of lanes (32 / batch lanes each) publish an item each, item n + group, as their slots come
// free; `mine`: this group has an item.  Three lanes store to each of the two CTAs, one releases.
__device__ __forceinline__ bool ring_publish(TicketRing* r, uint32_t n, const WorkDesc& wd, bool mine, int group, int sub,
                                             uint32_t own /* the group's lanes */, const WaitCtl& wc) {
  const uint32_t it = n + group, slot = it % TK_RING;
  const uint4* src = reinterpret_cast<const uint4*>(&wd);
  const uint4 piece = (sub & 3) == 0 ? src[0] : (sub & 3) == 1 ? src[1] : src[2];
  uint64_t t0 = 0;
  for (uint32_t spin = 1;; ++spin) {
    const uint32_t free = __ballot_sync(0xffffffffu, mine && mbar_try_wait_cluster(&r->empty[slot], ((it / TK_RING) & 1) ^ 1));
    const bool go = (free & own) == own;   // every lane of the group has seen it
    if (go && sub < 8 && (sub & 3) < WD_PIECES) st_cluster_v4(map_to_rank(smem_u32(&r->work[slot]), sub >> 2) + 16 * (sub & 3), piece);
    __syncwarp();
    if (go && sub == 0) {
      mbar_arrive_cluster_addr(map_to_rank(smem_u32(&r->full[slot]), 0));
      mbar_arrive_cluster_addr(map_to_rank(smem_u32(&r->full[slot]), 1));
    }
    if (go) mine = false;
    if (!__any_sync(0xffffffffu, mine)) return true;
    __nanosleep(50);
    if ((spin & 63u) == 0) {
      int gone = *reinterpret_cast<volatile int*>(&wc.status->abort);
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > wc.budget_ns) {
        report(wc.status, /*MOE_ERR_TIMEOUT*/ 2, (SITE_EMPTY << 24) | 0xFFFFF9);
        gone = 1;
      }
      if (__any_sync(0xffffffffu, gone)) return false;
    }
  }
}
// All lanes of a consumer warp; returns false on a failed wait.
__device__ __forceinline__ bool ring_take(TicketRing* r, uint32_t n, WorkDesc* wd, int lane, const WaitCtl& wc) {
  const int slot = n % TK_RING;
  int ok = 1;
  if (lane == 0) ok = mbar_wait_cluster(&r->full[slot], (n / TK_RING) & 1, wc, SITE_FULL, -8, 100) ? 1 : 0;
  if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
  *wd = r->work[slot];
  __syncwarp();
  if (lane == 0) mbar_arrive_leader(&r->empty[slot]);
  return true;
}
__device__ __forceinline__ SwapWork desc_swap_work(const WorkDesc& wd) {
  return SwapWork{wd.e, wd.n0, wd.nb, wd.nkb, wd.row0, wd.ntok, wd.ntok_b};
}
__device__ __forceinline__ Strip desc_strip(const WorkDesc& wd) {
  Strip st;
  st.e = wd.e; st.mp = wd.nb; st.row0 = wd.row0; st.rows = wd.ntok; st.nkb = wd.nkb;
  st.nb0 = wd.n0; st.nb1 = wd.nb1;
  return st;
}
// Decode item `item` of phase `phase` (scheduler).
template <bool BWD>
__device__ __forceinline__ void decode_item(const FusedArgs& fa, int phase, int item, WorkDesc& wd) {
  const bool strip = BWD && (phase == 1 || phase == 3);
  if (strip) {
    const GemmArgs& a = fa.op[phase];
    const Strip st = decode_strip(a, item);
    wd.e = st.e; wd.n0 = st.nb0; wd.nb = st.mp; wd.nkb = st.nkb;
    wd.row0 = st.row0; wd.ntok = st.rows; wd.ntok_b = 0; wd.nb1 = st.nb1;   // all rows of the expert
    return;
  }
  SwapWork w;
  if (!BWD) w = phase == 0 ? decode_swap_work<GEMM_GATE_UP>(fa.op[0], item) : decode_swap_work<GEMM_DOWN>(fa.op[1], item);
  else w = phase == 0 ? decode_swap_work<GEMM_ACT_GRAD>(fa.op[0], item) : decode_swap_work<GEMM_GATE_GRAD>(fa.op[2], item);
  wd.e = w.e; wd.n0 = w.n0; wd.nb = w.nb; wd.nkb = w.nkb;
  wd.row0 = w.row0; wd.ntok = w.ntok; wd.ntok_b = w.ntok_b; wd.nb1 = 0;
}

// Items of each phase and their prefix sums: ticket t belongs to phase p iff start[p] <= t < start[p + 1].
struct PhaseTable {
  int start[SCHED_MAX_SEG + 1];
};
template <bool BWD>
__device__ __forceinline__ PhaseTable make_phase_table(const FusedArgs& fa) {
  PhaseTable pt;
  pt.start[0] = 0;
  if (!BWD) {
    pt.start[1] = total_swap_work(fa.op[0]);
    pt.start[2] = pt.start[1] + total_swap_work(fa.op[1]);
    pt.start[3] = pt.start[4] = pt.start[2];
  } else {
    pt.start[1] = total_swap_work(fa.op[0]);
    pt.start[2] = pt.start[1] + wgrad_strips(fa.op[1]);
    pt.start[3] = pt.start[2] + total_swap_work(fa.op[2]);
    pt.start[4] = pt.start[3] + wgrad_strips(fa.op[3]);
  }
  return pt;
}
// Where each row-space phase's item list starts when there are shared experts (schedule.h, rotate_index): at the
// first item of the first shared expert.  `first[p]` = 0: no rotation (no shared experts, or a weight-gradient phase).
__device__ __forceinline__ int swap_first_item(const GemmArgs& a, int first_shared) {
  return a.work_start[first_shared] * a.n_tiles_n;
}
template <bool BWD>
__device__ __forceinline__ PhaseTable make_rotation_table(const FusedArgs& fa) {
  PhaseTable r;
  for (int p = 0; p <= SCHED_MAX_SEG; ++p) r.start[p] = 0;
  const int S = fa.cp.kp - fa.cp.k, E = fa.cp.Ep - S;
  if (S == 0) return r;
  if (!BWD) {
    r.start[0] = swap_first_item(fa.op[0], E);
    r.start[1] = swap_first_item(fa.op[1], E);
  } else {
    r.start[0] = swap_first_item(fa.op[0], E);
    r.start[2] = swap_first_item(fa.op[2], E);
  }
  return r;
}
__device__ __forceinline__ int phase_of(const PhaseTable& pt, int t) {
  int p = 0;
  while (p + 1 < SCHED_MAX_SEG && t >= pt.start[p + 1]) ++p;
  return p;
}

__device__ __forceinline__ ChainDeps phase_deps(const FusedArgs& fa, int phase, const WaitCtl& wc, const TraceCtl& tr) {
  ChainDeps d;
  d.ctr = fa.ctr;
  d.wait_kind = phase_wait_kind(fa.cp, phase);
  d.cp = &fa.cp;
  d.trig_kind = phase_trigger_kind(fa.cp, phase);
  d.phase = phase;
  d.wc = wc;
  d.tr = tr;
  return d;
}

// ---------------------------------------------------------------- one item, by role
template <bool BWD>
__device__ __forceinline__ bool load_item(const FusedArgs& fa, const GemmArgs::Ring ring, const WorkDesc& wd, uint8_t* smem, PipeBarriers* bars,
                                          LoaderState& ls, bool second_warp, int rank, int lane, const WaitCtl& wc,
                                          const ChainDeps& dep) {
  const int phase = wd.phase, t = wd.item;
  const bool strip = BWD && (phase == 1 || phase == 3);
  if (!(wd.flags & WD_READY) && (second_warp || strip)) {   // the item's dependent events (Section 4.3)
    const int first = wd.mb_first();
    if (!dep.wait(first, wd.mb_count(), fa.lv.counts[wd.e], first - fa.lv.mb_start[wd.e], lane, t)) return false;
  }
  if (strip)
    return wgrad_load_strip(fa.op[phase], smem, bars, ls, second_warp, rank, lane, desc_strip(wd), t, wc, dep);
  const SwapWork wk = desc_swap_work(wd);
  // act_grad's and gate_grad's weights lie alike: one copy of the code serves both.  The forward's loaders know their operator when
  // compiled: chosen per k-block, passes that stream weights take 1-2.5 % longer (4096 tokens x 4, 128 experts, 7168 x 2048: 2334 us
  // against 2397).
  if (BWD) return swap_load_item(GEMM_ACT_GRAD, fa.op[phase], ring, smem, bars, ls, second_warp, rank, lane, wk, t, wc, dep);
  if (phase == 0) return swap_load_item(GEMM_GATE_UP, fa.op[0], ring, smem, bars, ls, second_warp, rank, lane, wk, t, wc, dep);
  return swap_load_item(GEMM_DOWN, fa.op[1], ring, smem, bars, ls, second_warp, rank, lane, wk, t, wc, dep);
}
template <bool BWD>
__device__ __forceinline__ bool issue_item(const FusedArgs& fa, const GemmArgs::Ring ring, const WorkDesc& wd, uint8_t* smem, PipeBarriers* bars,
                                           uint32_t tmem_base, IssuerState& is, const WaitCtl& wc,
                                           const ChainDeps& dep) {
  const int phase = wd.phase, t = wd.item;
  if (BWD && (phase == 1 || phase == 3))
    return wgrad_issue_strip(fa.op[phase], smem, bars, tmem_base, is, desc_strip(wd), t, wc, dep);
  const SwapWork wk = desc_swap_work(wd);
  return swap_issue_item<BWD>(ring, smem, bars, tmem_base, is, wk, t, wc, dep);
}
template <bool BWD>
__device__ __forceinline__ bool epilogue_item(const FusedArgs& fa, const WorkDesc& wd, uint8_t* smem, PipeBarriers* bars,
                                              uint32_t tmem_base, EpiState& es, int rank, int ew, int lane,
                                              const WaitCtl& wc, const ChainDeps& dep) {
  const int phase = wd.phase, t = wd.item;
  if (BWD && (phase == 1 || phase == 3))
    return wgrad_epilogue_strip(fa.op[phase], smem, bars, tmem_base, es, rank, ew, lane, desc_strip(wd), t, wc, dep);
  const SwapWork wk = desc_swap_work(wd);
  if (!BWD) {
    if (phase == 0)
      return swap_epilogue_item<GEMM_GATE_UP>(fa.op[0], smem, bars, tmem_base, es, rank, ew, lane, wk, t, wc, dep);
    return swap_epilogue_item<GEMM_DOWN>(fa.op[1], smem, bars, tmem_base, es, rank, ew, lane, wk, t, wc, dep);
  }
  if (phase == 0)
    return swap_epilogue_item<GEMM_ACT_GRAD>(fa.op[0], smem, bars, tmem_base, es, rank, ew, lane, wk, t, wc, dep);
  return swap_epilogue_item<GEMM_GATE_GRAD>(fa.op[2], smem, bars, tmem_base, es, rank, ew, lane, wk, t, wc, dep);
}

// A matrix role's walk over the pair's items in ticket order; `enter` at each phase boundary of the backward (gemm_roles.cuh): the
// new phase's ring, of its own depth, starts at stage 0.  (The forward's two operators have one layout: the ring and the staging run
// on.)  The backward has a loop for each role: in one for all of them every warp carries all roles' state, 14 registers of which
// act_grad's epilogue has none to spare (1056 tokens, 32 + 1 experts, 1024 x 512: 90 us, in three loops 84).  The forward has
// registers left, and one loop: in three, 4096 tokens x 8, 256 experts, 7168 x 2048 take 4569 us for 4520.
template <bool BWD, class ENTER, class WORK>
__device__ __forceinline__ bool walk_items(const FusedArgs& fa, TicketRing* ring, int lane, const WaitCtl& wc, const TraceCtl& tr,
                                           ENTER enter, WORK work) {
  int cur_phase = 0;
  for (uint32_t n = 0;; ++n) {
    WorkDesc wd;
    if (!ring_take(ring, n, &wd, lane, wc)) return false;
    if (wd.ticket < 0) return true;
    if (BWD && wd.phase != cur_phase) {
      cur_phase = wd.phase;
      if (!enter(cur_phase)) return false;
    }
    if (!work(wd, phase_deps(fa, wd.phase, wc, tr))) return false;
  }
}

// ---------------------------------------------------------------- the kernel
template <bool BWD>
__global__ void __launch_bounds__(FUSED_THREADS, 1) fused_chain_kernel(const __grid_constant__ FusedArgs fa) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  PipeBarriers* bars = reinterpret_cast<PipeBarriers*>(smem + LAYOUT_BYTES);
  static_assert(sizeof(PipeBarriers) <= PIPE_BARRIER_BYTES && sizeof(TicketRing) <= TICKET_RING_BYTES, "shared-memory bookkeeping");
  TicketRing* ring = reinterpret_cast<TicketRing*>(reinterpret_cast<uint8_t*>(bars) + PIPE_BARRIER_BYTES);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const WaitCtl wc{fa.status, fa.budget_ns};
  const TraceCtl tr{fa.trace, fa.trace_cap, fa.ctr + CTR_TRACE_CURSOR};

  if (threadIdx.x == 0) {
    pipe_init(bars);
    for (int s = 0; s < TK_RING; ++s) {
      mbar_init(&ring->full[s], 1);
      mbar_init(&ring->empty[s], TK_CONSUMERS);
    }
    mbar_fence_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc_pair(&bars->tmem_base, TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers exist before anyone signals across the pair
  tc_fence_after_sync();
  const uint32_t tmem_base = uniform(bars->tmem_base);
  // (No trigger for the next launch: a router that takes the SMs as this launch's CTAs leave them is 2-3 % slower.)
  pdl_wait();   // the layout's tables, and everything else in front of this launch
  const int M = fa.lv.meta[0];
  const bool loader = warp == 0 || warp == 6, issuer = warp == 1 && rank == 0, epilogue = is_epilogue_warp(warp);

  if (warp == SCHED_WARP && rank == 0) {
    // ------------------------------------------------ scheduler of the pair (even CTA)
    // the first ticket is on its way while the tables are read
    int first_ticket = 0;
    if (lane == 0) first_ticket = atomicAdd(&fa.ctr[CTR_MAT_TICKET], 1);
    const PhaseTable pt = make_phase_table<BWD>(fa);
    const PhaseTable rot = make_rotation_table<BWD>(fa);   // first item of the first shared expert in each row-space phase
    const int total = pt.start[SCHED_MAX_SEG];
    int batches = 0;   // two bits a phase: log2
#pragma unroll
    for (int p = 0; p < SCHED_MAX_SEG; ++p)
      batches |= phase_batch_log2(pt.start[p + 1] - pt.start[p], fa.cp.batch[p], (int)gridDim.x) << (2 * p);
    int batch = 1, phase = 0;   // of the last ticket
    bool more = true;
    for (uint32_t n = 0; more;) {
      // the item sched_hold() before the batch's last has been taken first, then the tickets
      int ok = 1;
      const uint32_t hold = sched_hold(batch, fa.cp.strips[phase] != 0), next = n + batch;
      if (lane == 0 && next > hold)
        ok = mbar_wait_cluster(&ring->empty[(next - 1 - hold) % TK_RING], ((next - 1 - hold) / TK_RING) & 1, wc, SITE_EMPTY, -7, 100) ? 1 : 0;
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      int t = first_ticket;
      if (lane == 0 && n > 0) t = atomicAdd(&fa.ctr[CTR_MAT_TICKET], batch);
      t = __shfl_sync(0xffffffffu, t, 0);
      // `batch` groups of lanes decode a ticket each; a group's lanes share the look at its item's events
      const int lanes = 32 / batch, group = lane / lanes, sub = lane - group * lanes;
      t += group;
      uint64_t t0 = 0;
      if (tr.buf) t0 = globaltimer_ns();
      WorkDesc wd;
      wd.ticket = t < total ? t : -1;
      bool met = true;
      if (t < total) {
        wd.phase = phase_of(pt, t);
        wd.item = t - pt.start[wd.phase];
        if (rot.start[wd.phase]) wd.item = rotate_index(wd.item, rot.start[wd.phase], pt.start[wd.phase + 1] - pt.start[wd.phase]);
        wd.flags = 0;
        decode_item<BWD>(fa, wd.phase, wd.item, wd);
        const int first = wd.mb_first();
        met = phase_deps(fa, wd.phase, wc, tr).met(first, wd.mb_count(), fa.lv.counts[wd.e], first - fa.lv.mb_start[wd.e], sub, lanes);
      } else {
        wd.phase = wd.item = wd.flags = wd.e = wd.n0 = wd.nb = wd.nkb = 0;
        wd.row0 = wd.ntok = wd.ntok_b = wd.nb1 = 0;
      }
      const uint32_t unmet = __ballot_sync(0xffffffffu, !met), own = (lanes == 32 ? ~0u : (1u << lanes) - 1u) << (group * lanes);
      if (wd.ticket >= 0 && (unmet & own) == 0) wd.flags |= WD_READY;
      const uint64_t td = tr.buf ? globaltimer_ns() : 0;
      const bool mine = t < total || group == 0 || t - 1 < total;   // the end of the queue is published once
      if (!ring_publish(ring, n, wd, mine, group, sub, own, wc)) break;
      if (tr.buf && sub == 0 && wd.ticket >= 0) phase_deps(fa, wd.phase, wc, tr).trace(TR_SCHED, wd.item, t0, td, globaltimer_ns());
      more = !__any_sync(0xffffffffu, wd.ticket < 0);
      n += batch;
      phase = __shfl_sync(0xffffffffu, wd.phase, 31);
      batch = 1 << ((batches >> (2 * phase)) & 3);
    }
  } else if (loader || issuer || epilogue) {
    // ------------------------------------------------ matrix roles: the pair's items in ticket order
    const int ew = epilogue_index(warp);
    GemmArgs::Ring op_ring{};
    if (!epilogue) op_ring = which_ring(fa.op[0]);   // the operators of a pass have the same staging, and the same rings
    LoaderState ls;
    IssuerState is;
    EpiState es;
    auto load = [&](const WorkDesc& wd, const ChainDeps& dep) {
      return load_item<BWD>(fa, op_ring, wd, smem, bars, ls, warp == 6, rank, lane, wc, dep);
    };
    auto issue = [&](const WorkDesc& wd, const ChainDeps& dep) {
      return issue_item<BWD>(fa, op_ring, wd, smem, bars, tmem_base, is, wc, dep);
    };
    auto finish = [&](const WorkDesc& wd, const ChainDeps& dep) {
      return epilogue_item<BWD>(fa, wd, smem, bars, tmem_base, es, rank, ew, lane, wc, dep);
    };
    bool ok;
    if (!BWD) {
      ok = walk_items<BWD>(fa, ring, lane, wc, tr, [](int) { return true; }, [&](const WorkDesc& wd, const ChainDeps& dep) {
        return loader ? load(wd, dep) : issuer ? issue(wd, dep) : finish(wd, dep);
      });
    } else if (loader) {
      ok = walk_items<BWD>(fa, ring, lane, wc, tr, [&](int phase) { return loader_enter_phase(bars, ls, phase, wc); }, load);
    } else if (issuer) {
      ok = walk_items<BWD>(fa, ring, lane, wc, tr, [&](int) { is.s = is.a_s = 0; return true; }, issue);
    } else {
      auto enter = [&](int phase) {
        int go = 1;
        if (lane == 0) {
          tma_store_wait_read();
          epi_enter_phase(bars, ew, phase);
          go = phase_wait(bars, phase, wc) ? 1 : 0;
        }
        return __shfl_sync(0xffffffffu, go, 0) != 0;
      };
      ok = walk_items<BWD>(fa, ring, lane, wc, tr, enter, finish);
    }
    if (epilogue && lane == 0) {
      tma_store_wait_all();
      epi_enter_phase(bars, ew, SCHED_MAX_SEG);   // nothing of this warp is left in shared memory
    }
    if (issuer && uniform(!ok || *reinterpret_cast<volatile int*>(&fa.status->abort) ? 1 : 0)) issuer_drain(bars, fa.status);
  }

  // ------------------------------------------------ vector workers: the dedicated warps from the start, the
  // matrix-role warps once the matrix queue is empty (the tail of the vector queue -- combine -- runs on the
  // whole SM)
  __syncwarp();
  vector_worker_loop(fa, wc, tr, M, lane, warp >= GEMM_ROLE_WARPS && warp < GEMM_ROLE_WARPS + fa.gatherers);

  // ---------------------------------------------------------------- teardown
  if (*reinterpret_cast<volatile int*>(&fa.status->abort)) __nanosleep(200000);
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // neither CTA leaves while its partner may still read its shared memory or signal it
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
}

int vector_warps() { return VEC_WARPS; }

cudaError_t launch_fused(bool bwd, const FusedArgs& fa, int num_sms, cudaStream_t s, int* launches) {
  ++*launches;
  static PairLaunchState st_fwd, st_bwd;
  if (bwd)
    return launch_on_pairs(st_bwd, fused_chain_kernel<true>, fa, FUSED_THREADS, FUSED_SMEM_BYTES, num_sms, s, true);
  return launch_on_pairs(st_fwd, fused_chain_kernel<false>, fa, FUSED_THREADS, FUSED_SMEM_BYTES, num_sms, s, true);
}

}  // namespace moe
