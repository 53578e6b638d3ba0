// The tile schedule of the single persistent launch: one ticket-ordered matrix queue (the counterpart
// of the paper's matrix-core task queue, Section 4.3), two ticket-ordered vector queues, and the
// dependent / trigger event counters of every tile with their static thresholds.  Plain host/device
// code without CUDA calls, so the same functions drive the kernels and the CPU-side simulation that
// checks the schedule for coverage and deadlock freedom.
//
// Matrix queue.  The operators of a pass are phases in dependency order -- forward: gate+up, down;
// backward: act_grad, w2_grad, gate_grad, w1_grad -- and phase p's work items are numbered
// expert-major (column tile slow, token tile fast).  The queue is the concatenation of the phases'
// item lists, fixed before the launch; CTA pairs take its tickets in order.  The order of the queue
// is static (the paper's statically ordered task lists); which pair runs which item is decided by
// arrival, which keeps the items in flight a contiguous window of the queue: items that share an
// operand (the token tiles of one expert and column tile share its weight slab, the strips of one
// expert share its rows) start within microseconds of each other and meet in L2 however the pairs'
// speeds differ.  A pair that reaches phase p+1 early starts on it while others still finish phase p.
//
// Events (Section 4.3).  Per M-block (128 rows of the padded expert-ordered row space) three
// counters with static thresholds:
//   gathered   += 1 per gather task (4 rows)                      threshold: its rows up to the expert's last 32-row group / 4
//   activated  += 1 per CTA and column tile of phase 0            threshold SIG * column tiles
//   done       += 1 per CTA and column tile of the last row-space phase (down / gate_grad)
// A phase-0 item depends on `gathered` of its M-blocks, a down / gate_grad item and a w1_grad
// strip on `activated`, a w2_grad strip on `gathered`; a combine task depends on `done` of the
// M-blocks that hold its token's rows (many-to-many: up to k+S counters per token), the
// routing-weight-gradient task of an M-block on its `activated`.
//
// Deadlock freedom: every item's producers have smaller tickets (an earlier phase) or are vector
// tasks that never wait for matrix items of the same or a later phase; tickets are taken in order
// and only by CTAs that are running, so the holder of the smallest unfinished ticket always finds its dependent events
// met in finite time -- with any number of CTAs resident, as when another stream's launch holds some of the SMs: a CTA
// that has not started holds nothing.  Vector tasks alike: a worker that waits in the second queue is not one of the
// background gatherers, which empty the first.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MOE_HD __host__ __device__ __forceinline__
#else
#define MOE_HD inline
#endif

namespace moe {

constexpr int SCHED_MAX_SEG = 4;       // phases of a pass
constexpr int GROUP_ROWS = 32;         // an expert's rows are gathered (and multiplied) up to a multiple of this
constexpr int GATHER_ROWS = 4;         // rows of a gather task: the first M-blocks of a launch, which every CTA pair
                                       // waits for, are complete after a few microseconds
constexpr int GATHER_SUB = GROUP_ROWS / GATHER_ROWS;   // gather tasks per row group
constexpr int EPI_WARPS = 8;           // epilogue warps per CTA: two per quarter of the accumulator rows
constexpr int SIG = 2;                 // signals per (M-block, column tile): the last epilogue warp of each CTA of the pair

enum VecOp : int { VEC_GATHER = 0, VEC_DW = 2, VEC_COMBINE = 3 };

// Token-column tiles: the ceil(mc / 2) row-space units of an expert with mc M-blocks.  An odd count
// does not leave a lone M-block at the end (a tile of a few tokens still streams the whole weight
// tile): the single block sits before the last unit, which takes the last full block and the tail.
MOE_HD void balanced_unit(int mc, int u, int* first, int* count) {
  const int uc = (mc + 1) >> 1;
  *first = 2 * u;
  *count = 2;
  if ((mc & 1) == 0) return;
  if (u == uc - 1) {
    if (mc == 1) { *first = 0; *count = 1; }
    else *first = 2 * u - 1;
  } else if (u == uc - 2) {
    *count = 1;
  }
}

// Which experts merge their last two units, in every row-space phase: an odd count of three or more M-blocks whose
// last block is mostly padding (at most MERGE_TAIL_MAX rows).  Then the last unit (block + tail) is small, staging the
// weights once for both units saves the larger half of the shared-memory traffic, and what the next item waits for, the epilogue
// of the larger of the two tiles (gemm_roles.cuh, acc_claim), is short.  With a full last block (e.g. 384 rows) that costs
// as much as the second weight pass or more: down was 5 % faster unmerged there, 257..320-row experts 6 % slower.
constexpr int MERGE_TAIL_MAX = 64;
// Merged against two items in gate+up (forward) and act_grad (backward), 64 experts of 300 rows, F = 1408, medians of 14 runs in
// turn, us: d = 64 125 -> 107 forward; 256 132 -> 111 and 227 -> 207; 512 159 -> 136 and 313 -> 293; 1024 235 -> 217 and 473 -> 470;
// 1536 even backward; 2048 428 -> 382 and 809 -> 801; 4096 1558 -> 1509 backward (quartiles of one side 1-2 % of these).  Experts
// of 288 +- 17 rows, almost all of which merge, gain alike.
// A shared expert does not merge: one merged item takes a stage from every other (ring_choice), and a shared expert with a short
// last block is there at a quarter of all token counts; where items are few to a pair, a merged one is also the longest.  Merged
// against two items, us: 300 tokens, 8 x 2 + 1 experts, 2048 x 1408, forward 62.2 against 56.4, a step 174 against 161; 2060 x 4 + 1,
// 128 experts, 4096 x 1536, forward 975 against 945; 4100 x 4 + 1, 128 experts, 7168 x 2048 2640 against 2551.  Of 14 shapes with more
// shared experts than usual (2 to 16) two lose, 300 tokens, 2048 x 1408, forward: 16 x 2 + 4 87.7 against 91.6, 8 x 1 + 8 87.7 against 89.8.
MOE_HD bool expert_merges(int rows, int mblocks, bool shared) {
  return !shared && (mblocks & 1) && mblocks >= 3 && rows - (mblocks - 1) * 128 <= MERGE_TAIL_MAX;
}

constexpr int MERGED_TOKENS_MAX = 256 + MERGE_TAIL_MAX;   // of one item

// The operand rings of a call of T tokens (gemm_tc3.cu, plan_ring), by the rows of the largest expert: a ring for tiles of at most
// rows[0] tokens, of at most rows[1], of 256, and for merged items.  Distinct ids give an expert T rows at most, so that the
// second ring holds what a call of 129 to 224 tokens needs (a shared expert has T rows always): seven stages for six up to 192.
// Forward over 130 tokens x 8 + 1, 256 experts, 7168 x 2048: 3350 -> 3253 us; a step over 160 x 2 + 1, 8 experts, 4096 x 1536: 243 -> 234.
MOE_HD int ring_rows(int T, int ring) {
  const int rows = (T + GROUP_ROWS - 1) / GROUP_ROWS * GROUP_ROWS, most = ring == 0 ? 128 : 256;
  return rows < most ? rows : most;
}
MOE_HD int ring_choice(int largest, int rows0, int rows1, bool merged) {
  return largest <= rows0 ? 0 : largest <= rows1 ? 1 : merged ? 3 : 2;
}

// One work item of a row-space phase: a token tile (unit) of an expert and a column tile, or -- for an expert that merges
// (expert_merges) -- its last two units under one k-loop.  `start[e]` = first item of a column tile of expert e, `blk_expert[i]` =
// expert of item i (both from the layout kernels).
struct SwapItem {
  int e, nb;            // expert, column tile
  int unit;             // first unit of the item
  int merged;           // 1: units `unit` and `unit + 1`
  int mb_first;         // first M-block (absolute) of the item
  int mb_count;         // M-blocks of the item (both units): 1..3, contiguous
  int mb_count_a;       // M-blocks of the first unit
};
MOE_HD SwapItem decode_swap_item(int t, int n_tiles_n, const int* start, const int* blk_expert, const int* mb_start) {
  SwapItem it;
  const int e = blk_expert[t / n_tiles_n];
  const int ws = start[e];
  const int wcount = start[e + 1] - ws;
  const int local = t - ws * n_tiles_n;
  it.nb = local / wcount;
  const int wi = local - it.nb * wcount;
  const int mc = mb_start[e + 1] - mb_start[e];
  it.e = e;
  it.unit = wi;
  // the item table has one entry fewer than the expert has units exactly when the expert merges
  it.merged = (wcount == ((mc + 1) >> 1) - 1 && wi == wcount - 1) ? 1 : 0;
  int f, c;
  balanced_unit(mc, wi, &f, &c);
  it.mb_first = mb_start[e] + f;
  it.mb_count_a = c;
  it.mb_count = c;
  if (it.merged) {
    int f2, c2;
    balanced_unit(mc, wi + 1, &f2, &c2);
    it.mb_count += c2;
  }
  return it;
}

// Items of a weight-gradient phase.  A strip is 256 rows of dW[e] across all column tiles, its A operand resident in shared
// memory -- for an expert of up to 320 rows.  Longer experts stream A anyway; from WG_LONG_KB k-blocks (961 rows) on, a
// column tile is long enough (5 us) to be an item of its own, and these items come first: a shared expert of 1777 rows, last
// in expert order with three or five tiles to a strip, kept single pairs busy for 50 us after everyone else had finished.
// Behind them the other experts' strips, shared experts first as in the row-space phases.  order[]: the experts in that
// order, the n_long long ones in front.  With few strips to a CTA pair (strip_split) a strip is cut into `split` ranges of
// column tiles, whose A operand is loaded again: 8 experts of 192 x 6328 left 58 of 74 pairs without a strip.
constexpr int WG_LONG_KB = 16;
MOE_HD int strip_long(int rows) { return (rows + 63) / 64 >= WG_LONG_KB ? 1 : 0; }
struct StripItem { int e, strip, nb0, nb1; };   // expert, 256-row block of dW, column tiles [nb0, nb1)
MOE_HD int strip_split(int Ep, int strips, int ntn, int pairs) {
  const int n = Ep * strips;
  int split = (8 * pairs + n - 1) / n;          // about eight items for each pair, of at least four tiles
  if (split > ntn / 4) split = ntn / 4;
  if (split < 1) split = 1;
  if (n * split < pairs) {                      // fewer than one: of any size
    split = (pairs + n - 1) / n;
    if (split > ntn) split = ntn;
  }
  return split;
}
MOE_HD int strip_items(int Ep, int strips, int ntn, int split, int n_long) { return strips * ((Ep - n_long) * split + n_long * ntn); }
MOE_HD StripItem decode_strip_item(int t, int strips, int ntn, int split, int n_long, const int* order) {
  StripItem it;
  const int per = strips * ntn;
  if (t < n_long * per) {
    it.e = order[t / per];
    const int r = t % per;
    it.strip = r / ntn;
    it.nb0 = r - it.strip * ntn;
    it.nb1 = it.nb0 + 1;
  } else {
    t -= n_long * per;
    const int piece = t % split, st = t / split;
    it.e = order[n_long + st / strips];
    it.strip = st % strips;
    it.nb0 = piece * ntn / split;
    it.nb1 = (piece + 1) * ntn / split;
  }
  return it;
}
// Place of expert e in order[] given the number of long experts before it (long_before), before the first shared expert E
// (long_before_E) and in all.
MOE_HD int strip_order(int e, int rows, int E, int Ep, int long_before, int long_before_E, int n_long) {
  if (strip_long(rows)) return long_before;
  const int nl = e - long_before, nl_E = E - long_before_E, total = Ep - n_long;
  return n_long + (e >= E ? nl - nl_E : nl + total - nl_E);
}

// What a pass consists of (filled on the host from the layer's shape).
struct ChainParams {
  int is_bwd;
  int Ep, T, k, kp;
  int n_phases;                 // 2 (forward) or 4 (backward)
  int ntn[SCHED_MAX_SEG];       // column tiles per item (row-space phases) / per strip (weight gradients)
  int strips[SCHED_MAX_SEG];    // weight-gradient phases: strips (256 rows of dW) per expert; else 0
  int dep_extra;                // test hook: added to the `activated` threshold (> 0 = never reached)
  int want_dw;                  // backward: routing-weight-gradient tasks are part of the vector queue
  int combine_split;            // combine tasks per token (column chunks)
  int split[SCHED_MAX_SEG];     // weight-gradient phases: ranges of column tiles per strip
  int batch[SCHED_MAX_SEG];     // items a pair's scheduler takes and decodes together (1, 2 or 4)
};
// Ticket, decode and the look at the dependent events are a chain of four or five accesses to L2, 3 us; one at a time that is
// the pace of a pair whose items are shorter (down with F = 192: 0.7 us of MMAs, 4 us an item).  Items of a few k-blocks are
// therefore taken two or four at a time.  Not longer ones: the last items of a launch would lie with few pairs.
MOE_HD int sched_batch(int kblocks) { return kblocks <= 8 ? 4 : kblocks <= 16 ? 2 : 1; }
// Batches pay with many items to a pair; with few, the last ones would lie with some of the pairs.  log2 of the batch of a phase
// of `items` items, of at most `most`: 16 and 8 items for each pair of the launch's `ctas`.
MOE_HD int phase_batch_log2(int items, int most, int ctas) {
  return items >= 8 * ctas && most == 4 ? 2 : items >= 4 * ctas && most >= 2 ? 1 : 0;
}
// Items a pair holds at most that its epilogue has not begun: enough to hide the 3 us (with one fewer than four row-space
// items the passes over few tokens were 2-6 % slower).  Strips of a weight gradient are tens of microseconds long and of
// unequal length, four and a half to a pair in a step of 3400 tokens: what a pair holds beyond the next two nobody else can take.
MOE_HD int sched_hold(int batch, bool strips) { return batch == 4 ? 8 : batch == 1 && strips ? 2 : 4; }
// Vector warps per CTA that keep gathering after the first tasks.  Two gather 1.4 TB/s in and out; below the F where gate+up (or
// act_grad, half as long) takes that pace the matrix items wait for the rows, above it more gatherers only take from the
// bandwidth of their loads.  Two against all four, us forward / backward: 16384 tokens x 8 rows, d = 1024, 32 experts, F = 512
// 833 -> 530 / 1113 -> 837, F = 1024 913 -> 802 / 1552 -> 1500, F = 1280 even, F = 1536 1047 -> 1175 / 2112 -> 2370; 8192 tokens,
// d = 2048, 64 experts, F = 512 503 -> 447 / 821 -> 771, F = 1280 925 -> 858 / 1924 -> 1753, even from 1536 on; 4096 tokens,
// d = 4096, 590 -> 578 / 995 -> 917 at F = 512, even from 1024 on.  Where they part depends on d and the experts' rows, and the
// runs differ by 5-10 % under the power cap: the lines lie within the band, not at a sharp point.
MOE_HD int background_gatherers(int is_bwd, int F, int all) { return F <= (is_bwd ? 1536 : 1024) ? all : 2; }

// Gather tasks of M-block `rel` (relative to its expert's first) of an expert with `rows` rows.
MOE_HD int thr_gathered(int rows, int rel) {
  const int left = ((rows + GROUP_ROWS - 1) & ~(GROUP_ROWS - 1)) - rel * 128;
  return (left < 128 ? left : 128) / GATHER_ROWS;
}
MOE_HD int thr_activated(const ChainParams& cp) { return SIG * cp.ntn[0] + cp.dep_extra; }
MOE_HD int thr_done(const ChainParams& cp) { return SIG * cp.ntn[cp.is_bwd ? 2 : 1]; }

// Queue order with shared experts: every queue of the persistent launch (gather tasks, the items of the row-space
// phases) starts at the first shared expert and wraps around.  Every token has a row in every shared expert, and those
// experts come last in expert order: taken in expert order, no token would be complete before the very end and the
// whole combine would be a tail.  Started first, the shared rows are done early and a token is complete with its last
// ROUTED row, as without shared experts.  Dependencies are unchanged (an item still follows its producers in every
// queue, all queues being rotated alike); only the order among independent tasks changes (Section 4.5).
MOE_HD int rotate_index(int i, int first, int n) {
  const int j = i + first;
  return j >= n ? j - n : j;
}

// ---------------------------------------------------------------- counters (ints in device memory)
// 700 warps and more poll these words.  By the times, about 1 KB of consecutive addresses is served by one part of L2: where all of
// a small pass's counters lay in one such block -- a matter of where the workspace began -- signals and tickets queued behind
// the polls.  The three tickets therefore have a block each and the counters of an M-block 64 bytes.  1024 tokens x 4, 32 experts,
// 1024 x 512, forward: 57.6 us in one block, 51.7 in two, 49.2 so; 1777 x 3 + 1, 24 experts, 1160 x 712, a step: 217 -> 205; 256 x 2, 8
// experts, 256 x 128, a step: 49.3 -> 46.2.  32 or 128 bytes an M-block: even to 2 % slower.
constexpr int CTR_VEC_TICKET = 0, CTR_TRACE_CURSOR = 1, CTR_MAT_TICKET = 256, CTR_POST_TICKET = 512, CTR_PER_MB = 768, CTR_STRIDE = 16;
// combine tasks finished, and the word that turns 1 when all of them are (a copy-out stream may wait on it)
constexpr int CTR_COMBINE_DONE = 4, CTR_OUT_READY = 5;
enum CtrKind : int { CTR_GATHERED = 0, CTR_ACTIVATED = 1, CTR_DONE = 2, CTR_NONE = -1 };
MOE_HD int ctr_index(int mb, int kind) { return CTR_PER_MB + CTR_STRIDE * mb + kind; }
MOE_HD int ctr_ints(int cap_mblocks) { return CTR_PER_MB + CTR_STRIDE * cap_mblocks; }
static_assert(CTR_PER_MB % 4 == 0 && CTR_STRIDE % 4 == 0, "cleared 16 bytes at a time");

// dependent / trigger counter kind of each phase
MOE_HD int phase_wait_kind(const ChainParams& cp, int phase) {
  if (!cp.is_bwd) return phase == 0 ? CTR_GATHERED : CTR_ACTIVATED;
  return (phase == 0 || phase == 1) ? CTR_GATHERED : CTR_ACTIVATED;
}
// threshold of M-block `rel` of an expert with `rows` rows
MOE_HD int phase_wait_thr(const ChainParams& cp, int phase, int rows, int rel) {
  return phase_wait_kind(cp, phase) == CTR_GATHERED ? thr_gathered(rows, rel) : thr_activated(cp);
}
MOE_HD int phase_trigger_kind(const ChainParams& cp, int phase) {
  if (!cp.is_bwd) return phase == 0 ? CTR_ACTIVATED : CTR_DONE;
  return phase == 0 ? CTR_ACTIVATED : (phase == 2 ? CTR_DONE : CTR_NONE);
}

// ---------------------------------------------------------------- vector queues (ticket order)
// Two queues: the gather tasks in row order, and behind them the tasks that consume matrix tiles
// (backward: the routing-weight gradient per M-block; then the combine tasks).  A worker leaves the first
// queue for the second only when the first is empty -- or earlier, when it is not one of the few workers
// that keep gathering in the background (see fused.cu).
// Gather tasks every vector worker helps with at the start of a launch: the first M-blocks, which every CTA pair waits for,
// and at least GATHER_FAST_BYTES of rows.  A pass with no more rows than that is bound by the latency of its tasks, not by the
// bytes they take from the matrix tiles' loads: 1777 tokens x 4 rows of 2320 bytes took 48 us when 1024 tasks were
// everybody's (now 24), and every second matrix item waited.
constexpr int GATHER_FAST_TASKS = 1024, GATHER_FAST_BYTES = 24 << 20;
MOE_HD int gather_fast_tasks(int d) {
  const int n = GATHER_FAST_BYTES / (GATHER_ROWS * 2 * d);
  return n > GATHER_FAST_TASKS ? n : GATHER_FAST_TASKS;
}
struct VecTask {
  int op;       // VecOp
  int idx;      // gather: row group * GATHER_SUB + sub-task; dw: M-block; combine: token position * combine_split + column chunk
};
MOE_HD int gather_total(int groups) { return GATHER_SUB * groups; }
MOE_HD int combine_total(const ChainParams& cp) { return cp.T * cp.combine_split; }
MOE_HD int post_total(const ChainParams& cp, int M) {
  int n = combine_total(cp);
  if (cp.is_bwd && cp.want_dw) n += M;
  return n;
}
// Column chunks of a combine task: one warp sums a token's rows of 14 KB in 15-20 us, most of it latency.  With many tokens
// the warps hide each other's; with few, a token is cut into chunks of 64 16-byte vectors as long as no more than about two
// tasks fall on each of the launch's vector warps.
MOE_HD int combine_split_of(int T, int d) {
  const int chunks = (d / 8 + 63) / 64, room = T > 0 ? 1024 / T : 1;
  const int s = chunks < room ? chunks : room;
  return s > 1 ? s : 1;
}
// From this many tokens on combine tasks are taken in the order in which the tokens are completed.  With fewer about every
// task has a warp of its own that waits for it, and the sort only makes the layout longer (1-2 us of 7-10).
constexpr int COMBINE_ORDER_TOKENS = 512;
MOE_HD VecTask decode_post_ticket(const ChainParams& cp, int t, int M) {
  VecTask v;
  if (cp.is_bwd && cp.want_dw) {
    if (t < M) { v.op = VEC_DW; v.idx = t; return v; }
    t -= M;
  }
  v.op = VEC_COMBINE; v.idx = t;
  return v;
}

}  // namespace moe
