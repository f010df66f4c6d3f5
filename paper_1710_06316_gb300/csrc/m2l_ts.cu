// m2l_ts.cu -- compressed list-2 translations accumulated per target box on the 5th-
// generation tensor cores (precision mode 1, compressed ranks <= 112).
//
// The M2L of a level sums, for every target box b,   Lc[b] += sum_o C_o Mc[src(b, o)]
// over the offsets o of its list 2 (paper Sec. 3: the V-list translations of the FMM).
// Here a work item is a block of up to 128 target boxes of one level and one kernel
// (Laplace or Yukawa) with a range of its offsets (each offset's pairs form one run).  For each offset the source vectors of
// the targets that have a source there are gathered into the rows of the A operand (absent
// targets get zero rows), the translation C_o is the B operand, and
//      D[target, :] += A[target, :] C_o^T            (M = 128 targets, N = K = r)
// accumulates in tensor memory across all the offsets of the item (tcgen05.mma kind::f16,
// BF16 hi/lo split into hi*hi + hi*lo + lo*hi, FP32 accumulation).  The accumulator is
// read once per item and added into the targets' compressed local vectors: one write per
// target and item instead of one per translated pair.
//
// Blocks: a list-2 source of a child in octant (cx, cy, cz) of its parent lies at -3 .. 2 or
// -2 .. 3 along each axis, by the octant, so boxes of one octant share 189 of the 316
// offsets.  On levels of many boxes a block therefore takes boxes of one octant (in box
// order), which leaves fewer runs with more pairs each.
//
// Warp roles (288 threads): warps 0-3 gather the A operand of the next runs (16-byte
// cp.async) while one thread brings C_o by bulk asynchronous
// copy; warp 8 issues the MMAs; warps 4-7 read the accumulator (tcgen05.ld, one target
// per lane) and add it into Lc.  Two operand stages and two accumulators let the gather of
// offset k + 1, the MMAs of offset k and the epilogue of the previous item overlap.  A stage
// belongs to two of the gather warps, so that one run's copies are in flight while the other
// two warps issue the next run's (with all four on every run and a barrier of theirs before
// and after it, the kernel's time was that of its ~1.3 us chain of issue, latency and MMAs
// per run: 122 us on the 163,842-node sphere, 94 now; 4.90 -> 2.76 ms on 5.03M nodes).  Every mbarrier wait is bounded: on expiry the
// warp records the handle's error flag, the CTA's MMAs drain (bounded), its tensor memory is
// freed and it returns.
#include <cuda_bf16.h>

#include <cub/cub.cuh>

#include <algorithm>

#include "internal.cuh"
#include "tcgen05.cuh"

namespace afmpb {

constexpr int kTsRows = 128;                   // target boxes per block (MMA M, TMEM lanes)
constexpr int kTsThreads = 288;                // 4 gather warps, 4 epilogue warps, 1 MMA warp
constexpr int kTsMaxR = 112;                   // largest compressed rank this kernel takes
// Operand stages: two, so that two CTAs fit an SM at rank 64 (94 us on the 163,842-node sphere
// against 122 us with four stages, a warp to each, on one CTA per SM).
constexpr int kTsStages = 2;
constexpr int kTsItemRuns = 32;                // most runs (offsets) in one item
constexpr int kTsItemEnt = 768;                // most entries (translated pairs) in one item
// Levels with at least this many boxes are blocked by octant: eight part-filled blocks of
// 189 offsets replace six full ones of 316.
constexpr int kTsOctantBoxes = 6 * kTsRows;

// B operand tiles: C_o split into BF16 hi / lo in the canonical K-major layout with R rows.
// out: [table][slot][hi, lo][R x R]
__global__ void k_ts_tables(int R, int ntables, const float *__restrict__ C, __nv_bfloat16 *__restrict__ out) {
  const int64_t per = (int64_t)R * R;
  const int64_t total = (int64_t)ntables * kNumOffsets * per;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t tile = e / per;
    const int within = (int)(e % per);
    const int n = within / R, k = within % R;          // C_o[n][k]: output n, input k
    __nv_bfloat16 hi, lo;
    split_bf16(C[e], hi, lo);
    const uint32_t off = canon_off(n, k, R) >> 1;
    out[tile * 2 * per + off] = hi;
    out[tile * 2 * per + per + off] = lo;
  }
}

// Block group of every box: level * 8 + octant on levels blocked by octant, level * 8 else.
__global__ void k_ts_groups(int nbox, const int4 *__restrict__ anchor, const int *__restrict__ lvl_start,
                            uint32_t *__restrict__ group, int32_t *__restrict__ box) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbox) return;
  const int4 a = anchor[b];
  const bool split = lvl_start[a.w + 1] - lvl_start[a.w] >= kTsOctantBoxes;
  group[b] = (uint32_t)(8 * a.w + (split ? 4 * (a.x & 1) + 2 * (a.y & 1) + (a.z & 1) : 0));
  box[b] = b;
}

// start[g] = first slot (position in the order by group) of group g, start[ngroup] = nbox;
// slot_of[box] = its slot
__global__ void k_ts_slots(int nbox, int ngroup, const uint32_t *__restrict__ group, const int32_t *__restrict__ box,
                           int *__restrict__ start, int32_t *__restrict__ slot_of) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nbox) slot_of[box[i]] = i;
  if (i <= ngroup) {
    int lo = 0, hi = nbox;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (group[mid] < (uint32_t)i) lo = mid + 1;
      else hi = mid;
    }
    start[i] = lo;
  }
}

// (block, offset) key and (row, source) entry of every list-2 pair: key = global block *
// kNumOffsets + offset slot, entry = row << 32 | source box.
__global__ void k_ts_keys(const M2LGroup *__restrict__ groups, const int2 *__restrict__ pairs,
                          const uint32_t *__restrict__ group, const int32_t *__restrict__ slot_of,
                          const int *__restrict__ grp_start, const int *__restrict__ grp_block,
                          uint32_t *__restrict__ key, uint64_t *__restrict__ ent) {
  const M2LGroup g = groups[blockIdx.x];
  for (int j = threadIdx.x; j < g.count; j += blockDim.x) {
    const int2 pr = pairs[g.start + j];
    const int slot = slot_of[pr.x];
    const int q = (int)group[slot], rel = slot - grp_start[q];
    const int blk = grp_block[q] + rel / kTsRows;
    key[g.start + j] = (uint32_t)blk * kNumOffsets + (uint32_t)g.offset;
    ent[g.start + j] = ((uint64_t)(uint32_t)(rel % kTsRows) << 32) | (uint32_t)pr.y;
  }
}

// The rows present in each run, as a 128-bit mask.
__global__ void k_ts_masks(int nruns, const int4 *__restrict__ runs, const uint64_t *__restrict__ ent,
                           uint4 *__restrict__ mask) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nruns) return;
  uint32_t m[4] = {0, 0, 0, 0};
  for (int e = runs[r].y; e < runs[r].z; ++e) {
    const int row = (int)(ent[e] >> 32);
#pragma unroll
    for (int w = 0; w < 4; ++w) m[w] |= row >> 5 == w ? 1u << (row & 31) : 0u;
  }
  mask[r] = make_uint4(m[0], m[1], m[2], m[3]);
}

__device__ __forceinline__ void ts_producer_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
__device__ __forceinline__ void red_add_v4(float *addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

// With kBatch the items of several problems share the launch: item.req names the problem
// whose runs, entries, multipoles, tables and local expansions (reqs[item.req]) it uses,
// and the item count is read from *d_nitems (a list compacted to the running problems).
template <bool kBatch>
__global__ void __launch_bounds__(kTsThreads) k_m2l_ts(int R, int nitems_arg, const TSItem *__restrict__ items,
                                                      const int4 *__restrict__ runs_1,
                                                      const uint4 *__restrict__ masks_1,
                                                      const uint64_t *__restrict__ ent_1,
                                                      const int32_t *__restrict__ box_1,
                                                      const __nv_bfloat16 *__restrict__ Mc16_1,
                                                      const __nv_bfloat16 *__restrict__ tiles_1,
                                                      float *__restrict__ Lc_1, int *__restrict__ err_flag,
                                                      const int *__restrict__ d_nitems,
                                                      const TSReq *__restrict__ reqs) {
  constexpr int NS = kTsStages;
  extern __shared__ __align__(128) uint8_t smem[];
  after_previous();
  const int nitems = kBatch ? *d_nitems : nitems_arg;
  auto runs_of = [&](const TSItem &it) -> const int4 * { return kBatch ? reqs[it.req].runs : runs_1; };
  auto masks_of = [&](const TSItem &it) -> const uint4 * { return kBatch ? reqs[it.req].masks : masks_1; };
  auto box_of = [&](const TSItem &it) -> const int32_t * { return kBatch ? reqs[it.req].box : box_1; };
  auto ent_of = [&](const TSItem &it) -> const uint64_t * { return kBatch ? reqs[it.req].ent : ent_1; };
  auto mc_of = [&](const TSItem &it) -> const __nv_bfloat16 * {
    return kBatch ? reinterpret_cast<const __nv_bfloat16 *>(reqs[it.req].Mc16) : Mc16_1;
  };
  auto tiles_of = [&](const TSItem &it) -> const __nv_bfloat16 * {
    return kBatch ? reinterpret_cast<const __nv_bfloat16 *>(reqs[it.req].tiles) : tiles_1;
  };
  auto lc_of = [&](const TSItem &it) -> float * { return kBatch ? reqs[it.req].Lc : Lc_1; };
  // stage s: A hi, A lo (kTsRows x R each), B hi, B lo (R x R each)
  const uint32_t a_bytes = (uint32_t)(kTsRows * R * 2), b_bytes = (uint32_t)(R * R * 2);
  const uint32_t stage_bytes = 2 * a_bytes + 2 * b_bytes;
  const uint32_t s_base = cvta_smem(smem);
  __shared__ __align__(8) uint64_t bar_full[NS], bar_empty[NS], bar_accf[2], bar_acce[2];
  __shared__ uint32_t tmem_base;
  __shared__ __align__(16) int4 s_runs[2][kTsItemRuns];   // the runs, their row masks and the entries of
  __shared__ __align__(16) uint4 s_mask[2][kTsItemRuns];  // two items, brought in by bulk copy one item
  __shared__ __align__(16) uint64_t s_ent[2][kTsItemEnt + 2];   // ahead
  __shared__ __align__(8) uint64_t bar_item[2], bar_ifree[2];
  __shared__ int s_last;                                 // runs whose MMAs were committed (failure drain)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // The items are ordered by cost (few to a CTA) or by block (many): round k of the CTAs
  // takes the next gridDim.x items, in alternating direction.
  const int G = (int)gridDim.x;
  auto item_at = [&](int k) { return k * G + ((k & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x); };
  int nk = 0;                                            // this CTA's items: item_at(0 .. nk - 1)
  while (nk * G < nitems && item_at(nk) < nitems) ++nk;
  if (nk == 0) return;                                   // uniform per CTA
  uint32_t mb_full[NS], mb_empty[NS], mb_accf[2], mb_acce[2];
  for (int b = 0; b < NS; ++b) {
    mb_full[b] = cvta_smem(&bar_full[b]);
    mb_empty[b] = cvta_smem(&bar_empty[b]);
  }
  for (int b = 0; b < 2; ++b) {
    mb_accf[b] = cvta_smem(&bar_accf[b]);
    mb_acce[b] = cvta_smem(&bar_acce[b]);
  }
  // two accumulators of R FP32 columns each, rounded up to a power of two >= 32
  uint32_t ncols = 32;
  while (ncols < (uint32_t)(2 * R)) ncols <<= 1;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(cvta_smem(&tmem_base)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int b = 0; b < NS; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb_full[b]), "r"(4 / NS + 1));   // its warps, and C_o
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb_empty[b]));
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb_accf[b]));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(mb_acce[b]));   // one arrival per epilogue warp
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cvta_smem(&bar_item[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(cvta_smem(&bar_ifree[b])));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_last = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  bool failed = false;

  if (warp < 4) {
    // ---- gather -------------------------------------------------------------------------
    // Each run has at most one entry per target row (a target has one source per offset).  A
    // stage keeps the rows of its last run: a row that was present and is not now is
    // cleared by the row's thread, so rows that stay absent cost nothing.
    const uint32_t mb_item[2] = {cvta_smem(&bar_item[0]), cvta_smem(&bar_item[1])};
    const uint32_t mb_ifree[2] = {cvta_smem(&bar_ifree[0]), cvta_smem(&bar_ifree[1])};
    auto load_item = [&](int k) {                        // thread 0: item k's runs and entries -> buffer k & 1
      const TSItem it = items[item_at(k)];
      const int b = k & 1;
      const uint32_t rb = (uint32_t)(it.run1 - it.run0) * 16;
      const int a0 = it.ent0 & ~1;                       // 16-byte aligned start (entries are 8 bytes)
      const uint32_t eb = (uint32_t)(((it.ent1 - a0) + 1) & ~1) * 8;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // earlier reads of the buffer done
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb_item[b]), "r"(2 * rb + eb) : "memory");
      auto copy = [&](const void *dst, const void *src, uint32_t bytes) {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         cvta_smem(dst)),
                     "l"(src), "r"(bytes), "r"(mb_item[b])
                     : "memory");
      };
      copy(&s_runs[b][0], runs_of(it) + it.run0, rb);
      copy(&s_mask[b][0], masks_of(it) + it.run0, rb);
      copy(&s_ent[b][0], ent_of(it) + a0, eb);
    };
    int issued = -1, waited = -1;                        // item positions loaded / waited for (thread 0 issues)
    if (threadIdx.x == 0)
      for (; issued < 1 && issued + 1 < nk; ++issued) load_item(issued + 1);
    // the stages start all zero (no row present)
    for (uint32_t o = threadIdx.x * 16; o < NS * stage_bytes; o += 128 * 16)
      asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(s_base + o), "r"(0u) : "memory");
    ts_producer_sync();
    // a stage belongs to 4 / NS of the warps, which gather every NS-th run: the copies of
    // one run are in flight while the next run's are issued and the previous one's MMAs run
    constexpr int kStageThreads = 128 / NS;
    const int s = threadIdx.x / kStageThreads, ts = threadIdx.x % kStageThreads;
    const uint32_t st = s_base + (uint32_t)s * stage_bytes;
    uint32_t was = 0;                                    // bit i: row ts + i kStageThreads is present
    int use = 0;
    for (int k = 0; k < nk && !failed; ++k) {
      const TSItem item = items[item_at(k)];
      const int b = k & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(mb_item[b], (uint32_t)((k >> 1) & 1)))) {
        failed = true;
        break;
      }
      waited = k;
      const __nv_bfloat16 *mc = mc_of(item) + (size_t)item.kt * 2 * R;
      const __nv_bfloat16 *tl = tiles_of(item) + (size_t)item.table * kNumOffsets * 2 * R * R;
      const int kg = item.rank / 8;                      // 16-byte groups along K that the MMAs read
      for (int r = 0; r < item.run1 - item.run0; ++r, ++use) {
        if (use % NS != s) continue;
        // the MMAs of the run that this stage held are done
        if (use >= NS && !__all_sync(0xffffffffu, mbar_wait(mb_empty[s], (uint32_t)((use / NS - 1) & 1)))) {
          failed = true;
          break;
        }
        const int4 run = s_runs[b][r];                   // (offset slot, first entry, end entry, -)
        if (ts == 0) {
          // C_o of the item's table: hi and lo tiles (consecutive), counted on the full barrier
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb_full[s]), "r"(2 * b_bytes)
                       : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  st + 2 * a_bytes),
              "l"(tl + (size_t)run.x * 2 * R * R), "r"(2 * b_bytes), "r"(mb_full[s])
              : "memory");
        }
        // eight entries to a warp at a time, four lanes to an entry
        const uint64_t *ent = &s_ent[b][(item.ent0 & 1) + (run.y - item.ent0)];
        for (int e = ts >> 2; e < run.z - run.y; e += kStageThreads / 4) {
          const uint64_t v = ent[e];
          const int prow = (int)(v >> 32);
          const __nv_bfloat16 *g = mc + (size_t)(uint32_t)v * 4 * R;
          for (int k8 = ts & 3; k8 < kg; k8 += 4) {
            const uint32_t off = canon_off(prow, k8 * 8, kTsRows);
            cp_async16_zfill(st + off, g + k8 * 8, true);
            cp_async16_zfill(st + a_bytes + off, g + R + k8 * 8, true);
          }
        }
        const uint32_t *mask = reinterpret_cast<const uint32_t *>(&s_mask[b][r]);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
          const int row = ts + i * kStageThreads;
          const bool now = (mask[row >> 5] >> (row & 31)) & 1u;
          if (((was >> i) & 1u) && !now) {
            for (int k8 = 0; k8 < R / 8; ++k8) {
              const uint32_t off = canon_off(row, k8 * 8, kTsRows);
              asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(st + off), "r"(0u) : "memory");
              asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(st + a_bytes + off), "r"(0u) : "memory");
            }
          }
          was = (was & ~(1u << i)) | ((now ? 1u : 0u) << i);
        }
        // this warp's rows have landed: make them visible to the tensor core
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb_full[s]) : "memory");
      }
      if (failed) break;
      // this warp has read item k's buffer; when all four have, it takes item k + 2
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb_ifree[b]) : "memory");
      if (warp == 0 && k + 2 < nk) {
        if (!__all_sync(0xffffffffu, mbar_wait(mb_ifree[b], (uint32_t)((k >> 1) & 1)))) {
          failed = true;
          break;
        }
        if (lane == 0) {
          load_item(k + 2);
          issued = k + 2;
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (threadIdx.x == 0)                                // after a failure: let issued item copies land (bounded)
      for (int k = waited + 1; k <= issued; ++k) mbar_wait(mb_item[k & 1], (uint32_t)((k >> 1) & 1));
  } else if (warp == 8) {
    // ---- MMA issue (one thread) ----------------------------------------------------------
    if (lane == 0) {
      int use = 0, committed = 0;
      const uint32_t lbo_a = (kTsRows / 8) * 128, lbo_b = (uint32_t)(R / 8) * 128, sbo = 128;
      for (int k = 0; k < nk && !failed; ++k) {
        const TSItem item = items[item_at(k)];
        const int a = k & 1;
        if (k >= 2 && !mbar_wait(mb_acce[a], (uint32_t)(((k >> 1) - 1) & 1))) {   // epilogue of item k - 2 read it
          failed = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t acc = tmem + (uint32_t)(a * R);
        const uint32_t idesc = instr_desc(kTsRows, R);
        for (int r = item.run0; r < item.run1; ++r, ++use) {
          const int s = use % NS;
          if (!mbar_wait(mb_full[s], (uint32_t)((use / NS) & 1))) {
            failed = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t st = s_base + (uint32_t)s * stage_bytes;
          const uint32_t sa_hi = st, sa_lo = st + a_bytes, sb_hi = st + 2 * a_bytes, sb_lo = sb_hi + b_bytes;
          for (int q = 0; q < item.rank / 16; ++q) {
            const uint32_t ka = 2 * q * lbo_a, kb = 2 * q * lbo_b;
            const uint64_t dah = smem_desc(sa_hi + ka, lbo_a, sbo), dal = smem_desc(sa_lo + ka, lbo_a, sbo);
            const uint64_t dbh = smem_desc(sb_hi + kb, lbo_b, sbo), dbl = smem_desc(sb_lo + kb, lbo_b, sbo);
            const uint32_t first = (r == item.run0 && q == 0) ? 0u : 1u;      // 0: overwrite the accumulator
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc),
                "l"(dah), "l"(dbh), "r"(idesc), "r"(first));
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc),
                "l"(dah), "l"(dbl), "r"(idesc), "r"(1u));
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc),
                "l"(dal), "l"(dbh), "r"(idesc), "r"(1u));
          }
          // the stage is free once these MMAs have read it
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              mb_empty[s]));
          committed = use + 1;
        }
        if (failed) break;
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            mb_accf[a]));
      }
      s_last = committed;
    }
    failed = __shfl_sync(0xffffffffu, failed, 0);
  } else {
    // ---- epilogue: one target box per lane ------------------------------------------------
    const int ew = warp - 4;
    const int row = 32 * ew + lane;
    for (int k = 0; k < nk; ++k) {
      const TSItem item = items[item_at(k)];
      const int a = k & 1;
      const bool valid = item.base + row < item.end;
      const int box = valid ? box_of(item)[item.base + row] : 0;
      const bool ok = __all_sync(0xffffffffu, mbar_wait(mb_accf[a], (uint32_t)((k >> 1) & 1)));
      if (!ok) {
        failed = true;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      float *out = lc_of(item) + ((size_t)box * 2 + item.kt) * R;
      for (int c0 = 0; c0 < item.rank; c0 += 16) {
        uint32_t v[16];
        const uint32_t taddr = tmem + ((uint32_t)(32 * ew) << 16) + (uint32_t)(a * R + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        if (valid) {
          const float sc = item.scale;
#pragma unroll
          for (int q = 0; q < 16; q += 4)
            red_add_v4(out + c0 + q, __uint_as_float(v[q]) * sc, __uint_as_float(v[q + 1]) * sc,
                       __uint_as_float(v[q + 2]) * sc, __uint_as_float(v[q + 3]) * sc);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb_acce[a]) : "memory");
    }
  }
  if (failed && lane == 0) atomicExch(err_flag, 1);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (threadIdx.x == 0) {
    // bounded: the last committed MMA group has read its stage before the memory goes
    const int last = s_last;
    if (last > 0) mbar_wait(mb_empty[(last - 1) % NS], (uint32_t)(((last - 1) / NS) & 1));
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

namespace {
int ts_stage_bytes(int R) { return 2 * kTsRows * R * 2 + 2 * R * R * 2; }   // A hi, lo + B hi, lo
int ts_smem_bytes(int R) { return kTsStages * ts_stage_bytes(R); }
}  // namespace

bool m2l_ts_applies(const afmpb_t *h) { return h->m2l_rank > 0 && h->m2l_rank <= kTsMaxR && h->d_Mc16; }

// Work of the kernel: the list-2 entries re-sorted by (target block, offset) on the device,
// the runs of equal keys, and items of at most `per_item` runs of one block and one kernel.
Err build_m2l_ts(afmpb_t *h) {
  const std::vector<int> &level_table = h->h_level_table;
  const int R = h->m2l_rank;
  auto &A = h->arena;
  cudaStream_t s = h->stream;
  const auto &T = h->shape;
  const int64_t np = h->n_m2l_pairs;
  h->ts_nitems = 0;
  if (np == 0 || h->m2l_groups.empty()) return Err{};
  // target boxes by block group (level, octant); blocks of kTsRows within each group
  const int ngroup = 8 * T.nlevel;
  int *d_lvl = nullptr, *d_gstart = nullptr, *d_gblk = nullptr;
  uint32_t *grp = nullptr, *grp_sorted = nullptr;
  int32_t *ids = nullptr, *slot_of = nullptr;
  AFMPB_TRY(A.alloc(&d_lvl, T.lvl_start.size(), "ts level start"));
  AFMPB_TRY(A.alloc(&d_gstart, ngroup + 1, "ts group start"));
  AFMPB_TRY(A.alloc(&d_gblk, ngroup + 1, "ts group block"));
  AFMPB_TRY(A.alloc(&grp, T.nbox, "ts groups"));
  AFMPB_TRY(A.alloc(&grp_sorted, T.nbox, "ts groups sorted"));
  AFMPB_TRY(A.alloc(&ids, T.nbox, "ts box ids"));
  AFMPB_TRY(A.alloc(&slot_of, T.nbox, "ts slots"));
  AFMPB_TRY(A.alloc(&h->d_ts_box, T.nbox, "ts boxes by slot"));
  AFMPB_CUDA(cudaMemcpyAsync(d_lvl, T.lvl_start.data(), sizeof(int) * T.lvl_start.size(), cudaMemcpyHostToDevice, s));
  k_ts_groups<<<div_up(T.nbox, 256), 256, 0, s>>>(T.nbox, h->d_box_anchor, d_lvl, grp, ids);
  AFMPB_TRY(check_launch("k_ts_groups"));
  {
    int bits = 1;
    while ((1 << bits) < ngroup) ++bits;
    size_t bytes = 0;
    AFMPB_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, bytes, grp, grp_sorted, ids, h->d_ts_box, T.nbox, 0, bits, s));
    uint8_t *tmp = nullptr;
    AFMPB_TRY(A.alloc(&tmp, std::max<size_t>(bytes, 16), "ts group sort scratch"));
    AFMPB_CUDA(cub::DeviceRadixSort::SortPairs(tmp, bytes, grp, grp_sorted, ids, h->d_ts_box, T.nbox, 0, bits, s));
    A.release(tmp);
  }
  k_ts_slots<<<div_up(std::max(T.nbox, ngroup + 1), 256), 256, 0, s>>>(T.nbox, ngroup, grp_sorted, h->d_ts_box,
                                                                       d_gstart, slot_of);
  AFMPB_TRY(check_launch("k_ts_slots"));
  std::vector<int> gstart(ngroup + 1), gblk(ngroup + 1, 0);
  AFMPB_CUDA(cudaMemcpyAsync(gstart.data(), d_gstart, sizeof(int) * (ngroup + 1), cudaMemcpyDeviceToHost, s));
  AFMPB_CUDA(cudaStreamSynchronize(s));
  h->ts_blocks.clear();
  for (int g = 0; g < ngroup; ++g) {
    for (int i = gstart[g]; i < gstart[g + 1]; i += kTsRows)
      h->ts_blocks.push_back({i, std::min(i + kTsRows, gstart[g + 1]), g / 8});
    gblk[g + 1] = (int)h->ts_blocks.size();
  }
  const int nblocks = (int)h->ts_blocks.size();
  AFMPB_CUDA(cudaMemcpyAsync(d_gblk, gblk.data(), sizeof(int) * (ngroup + 1), cudaMemcpyHostToDevice, s));
  uint32_t *key = nullptr, *key_sorted = nullptr, *uniq = nullptr;
  uint64_t *ent = nullptr;
  int32_t *cnt = nullptr, *d_nruns = nullptr;
  AFMPB_TRY(A.alloc(&key, np, "ts keys"));
  AFMPB_TRY(A.alloc(&key_sorted, np, "ts keys sorted"));
  AFMPB_TRY(A.alloc(&ent, np, "ts entries unsorted"));
  AFMPB_TRY(A.alloc(&h->d_ts_ent, np + 2, "ts entries"));   // +2: 16-byte rounded item copies
  AFMPB_TRY(A.alloc(&uniq, np, "ts run keys"));
  AFMPB_TRY(A.alloc(&cnt, np, "ts run sizes"));
  AFMPB_TRY(A.alloc(&d_nruns, 1, "ts run count"));
  k_ts_keys<<<(unsigned)h->m2l_groups.size(), 256, 0, s>>>(h->d_m2l_groups, h->d_m2l_pairs, grp_sorted, slot_of,
                                                          d_gstart, d_gblk, key, ent);
  AFMPB_TRY(check_launch("k_ts_keys"));
  int bits = 1;
  while (((uint64_t)1 << bits) < (uint64_t)nblocks * kNumOffsets) ++bits;
  {
    size_t bytes = 0;
    AFMPB_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, bytes, key, key_sorted, ent, h->d_ts_ent, np, 0, bits, s));
    uint8_t *tmp = nullptr;
    AFMPB_TRY(A.alloc(&tmp, std::max<size_t>(bytes, 16), "ts sort scratch"));
    AFMPB_CUDA(cub::DeviceRadixSort::SortPairs(tmp, bytes, key, key_sorted, ent, h->d_ts_ent, np, 0, bits, s));
    AFMPB_CUDA(cudaStreamSynchronize(s));
    A.release(tmp);
    bytes = 0;
    AFMPB_CUDA(cub::DeviceRunLengthEncode::Encode(nullptr, bytes, key_sorted, uniq, cnt, d_nruns, np, s));
    AFMPB_TRY(A.alloc(&tmp, std::max<size_t>(bytes, 16), "ts encode scratch"));
    AFMPB_CUDA(cub::DeviceRunLengthEncode::Encode(tmp, bytes, key_sorted, uniq, cnt, d_nruns, np, s));
    AFMPB_CUDA(cudaStreamSynchronize(s));
    A.release(tmp);
  }
  int32_t nruns = 0;
  AFMPB_CUDA(cudaMemcpyAsync(&nruns, d_nruns, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  AFMPB_CUDA(cudaStreamSynchronize(s));
  std::vector<uint32_t> rkey(nruns);
  std::vector<int32_t> rcnt(nruns);
  AFMPB_CUDA(cudaMemcpyAsync(rkey.data(), uniq, sizeof(uint32_t) * nruns, cudaMemcpyDeviceToHost, s));
  AFMPB_CUDA(cudaMemcpyAsync(rcnt.data(), cnt, sizeof(int32_t) * nruns, cudaMemcpyDeviceToHost, s));
  AFMPB_CUDA(cudaStreamSynchronize(s));
  for (void *q : {(void *)d_lvl, (void *)d_gstart, (void *)d_gblk, (void *)grp, (void *)grp_sorted, (void *)ids,
                  (void *)slot_of, (void *)key, (void *)key_sorted, (void *)ent, (void *)uniq,
                  (void *)cnt, (void *)d_nruns})
    A.release(q);
  h->ts_rkey = std::move(rkey);
  h->ts_rcnt = std::move(rcnt);
  {
    // runs (offset slot, first entry, end entry)
    std::vector<int4> runs(nruns);
    int64_t e0 = 0;
    for (int r = 0; r < nruns; ++r) {
      runs[r] = make_int4((int)(h->ts_rkey[r] % kNumOffsets), (int)e0, (int)(e0 + h->ts_rcnt[r]), 0);
      e0 += h->ts_rcnt[r];
    }
    AFMPB_TRY(A.alloc(&h->d_ts_runs, std::max<size_t>(1, runs.size()), "ts runs"));
    AFMPB_CUDA(cudaMemcpyAsync(h->d_ts_runs, runs.data(), sizeof(int4) * runs.size(), cudaMemcpyHostToDevice, s));
    AFMPB_TRY(A.alloc(&h->d_ts_masks, std::max<size_t>(1, runs.size()), "ts row masks"));
    k_ts_masks<<<div_up(std::max(nruns, 1), 128), 128, 0, s>>>(nruns, h->d_ts_runs, h->d_ts_ent, h->d_ts_masks);
    AFMPB_TRY(check_launch("k_ts_masks"));
    AFMPB_CUDA(cudaStreamSynchronize(s));
  }
  AFMPB_TRY(cut_m2l_ts_items(h));
  // B tiles from the compressed FP32 tables
  const size_t elems = (size_t)h->m2l_ntables * kNumOffsets * 2 * R * R;
  AFMPB_TRY(A.alloc(&h->d_ts_tiles, elems, "ts translation tiles"));
  k_ts_tables<<<2048, 256, 0, s>>>(R, h->m2l_ntables, h->d_C, reinterpret_cast<__nv_bfloat16 *>(h->d_ts_tiles));
  AFMPB_TRY(check_launch("k_ts_tables"));
  AFMPB_TRY(alloc_wait_flag(h));
  AFMPB_TRY(raise_smem_limit((const void *)k_m2l_ts<false>, ts_smem_bytes(R)));
  AFMPB_TRY(raise_smem_limit((const void *)k_m2l_ts<true>, ts_smem_bytes(R)));
  AFMPB_CUDA(cudaStreamSynchronize(s));
  return Err{};
}

// Items over the stored runs: consecutive runs of one target block and one kernel, at most
// h->ts_runs_per_item runs (0: about four items per SM, at most kTsItemRuns) and kTsItemEnt
// entries each.  Replaces earlier items; the tile tuner calls it with other sizes.
Err cut_m2l_ts_items(afmpb_t *h) {
  auto &A = h->arena;
  cudaStream_t s = h->stream;
  const auto &T = h->shape;
  const std::vector<uint32_t> &rkey = h->ts_rkey;
  const std::vector<int32_t> &rcnt = h->ts_rcnt;
  const int nruns = (int)rkey.size();
  const std::vector<int> &level_table = h->h_level_table;
  std::vector<int64_t> rstart(nruns + 1, 0);
  for (int r = 0; r < nruns; ++r) rstart[r + 1] = rstart[r] + rcnt[r];
  int dev = 0, sms = 0;
  AFMPB_CUDA(cudaGetDevice(&dev));
  AFMPB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int per_item = h->ts_runs_per_item > 0 ? std::min(kTsItemRuns, h->ts_runs_per_item)
                                                : std::min(kTsItemRuns, std::max(8, nruns / std::max(1, 4 * sms)));
  std::vector<TSItem> items;
  for (int kt = 0; kt < 2; ++kt) {
    for (int r = 0; r < nruns;) {
      const int blk = (int)(rkey[r] / kNumOffsets);
      int rend = r;
      while (rend < nruns && (int)(rkey[rend] / kNumOffsets) == blk) ++rend;
      const TSBlock &B = h->ts_blocks[blk];
      const int l = B.level;
      const bool use = kt == 0 || (l >= h->m2l_yuk_levels && !h->laplace_only);
      if (use) {
        const int table = kt == 0 ? 0 : level_table[l];
        // consecutive runs of the block, at most per_item runs and kTsItemEnt entries each
        for (int q0 = r; q0 < rend;) {
          int q1 = q0, ne = 0;
          while (q1 < rend && q1 - q0 < per_item && ne + rcnt[q1] <= kTsItemEnt) ne += rcnt[q1++];
          TSItem it{};
          it.base = B.begin;
          it.end = B.end;
          it.run0 = q0;
          it.run1 = q1;
          it.ent0 = (int)rstart[q0];
          it.ent1 = (int)rstart[q1];
          it.kt = kt;
          it.table = table;
          it.rank = h->h_table_rank[table];
          // Laplace tables are for the unit box: scale by 1 / w of the level
          it.scale = kt == 0 ? (float)(1.0 / std::ldexp(T.w0, -l)) : 1.0f;
          items.push_back(it);
          q0 = q1;
        }
      }
      r = rend;
    }
  }
  // few items to a CTA: by cost, so that the CTAs' shares differ by less than one small item
  if ((int64_t)items.size() <= 32 * (int64_t)sms)
    std::stable_sort(items.begin(), items.end(), [](const TSItem &x, const TSItem &y) {
      return (x.run1 - x.run0) * x.rank > (y.run1 - y.run0) * y.rank;
    });
  h->ts_nitems = (int)items.size();
  if (h->d_ts_items) A.release(h->d_ts_items);
  AFMPB_TRY(A.alloc(&h->d_ts_items, std::max<size_t>(1, items.size()), "ts items"));
  if (!items.empty())
    AFMPB_CUDA(cudaMemcpyAsync(h->d_ts_items, items.data(), sizeof(TSItem) * items.size(), cudaMemcpyHostToDevice, s));
  AFMPB_CUDA(cudaStreamSynchronize(s));
  return Err{};
}

Err enqueue_m2l_ts(afmpb_t *h, cudaStream_t s) {
  if (h->ts_nitems == 0) return Err{};
  int dev = 0, sms = 0;
  AFMPB_CUDA(cudaGetDevice(&dev));
  AFMPB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int R = h->m2l_rank;
  const int per_sm = std::max(1, std::min(2, (227 * 1024) / (ts_smem_bytes(R) + 16 * 1024)));
  const unsigned grid = (unsigned)std::min(h->ts_nitems, per_sm * sms);
  const auto *mc = reinterpret_cast<const __nv_bfloat16 *>(h->d_Mc16);
  const auto *tl = reinterpret_cast<const __nv_bfloat16 *>(h->d_ts_tiles);
  return launch_next(true, "k_m2l_ts", k_m2l_ts<false>, grid, kTsThreads, ts_smem_bytes(R), s, R, h->ts_nitems, h->d_ts_items,
                       h->d_ts_runs, h->d_ts_masks, h->d_ts_ent, h->d_ts_box, mc, tl, h->d_Lc, h->d_tc_flag, nullptr, nullptr);
}

// The items of the running problems of a batch, in their order: one block scans the
// flags 1024 items at a time.
__global__ void __launch_bounds__(1024) k_ts_compact(int n, const TSItem *__restrict__ in, const TSReq *__restrict__ reqs,
                                                     TSItem *__restrict__ out, int *__restrict__ count) {
  __shared__ int s_warp[32];
  __shared__ int s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_base = 0;
  __syncthreads();
  for (int c0 = 0; c0 < n; c0 += 1024) {
    const int i = c0 + (int)threadIdx.x;
    TSItem it{};
    int keep = 0;
    if (i < n) {
      it = in[i];
      const int *a = reqs[it.req].active;
      keep = (a == nullptr || *a != 0) ? 1 : 0;
    }
    int v = keep;                                        // inclusive scan within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    if (lane == 31) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
      int w = s_warp[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += u;
      }
      s_warp[lane] = w;                                  // inclusive over warps
    }
    __syncthreads();
    const int before = s_base + (warp > 0 ? s_warp[warp - 1] : 0) + v - keep;
    if (keep) out[before] = it;
    __syncthreads();
    if (threadIdx.x == 0) s_base += s_warp[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) *count = s_base;
}

Err enqueue_m2l_ts_batch(const TSReq *d_reqs, const TSItem *d_items, int nitems, TSItem *d_items_run, int *d_count,
                         int R, int *err_flag, cudaStream_t s) {
  if (nitems == 0) return Err{};
  int dev = 0, sms = 0;
  AFMPB_CUDA(cudaGetDevice(&dev));
  AFMPB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  k_ts_compact<<<1, 1024, 0, s>>>(nitems, d_items, d_reqs, d_items_run, d_count);
  AFMPB_TRY(check_launch("k_ts_compact"));
  const int per_sm = std::max(1, std::min(2, (227 * 1024) / (ts_smem_bytes(R) + 16 * 1024)));
  const unsigned grid = (unsigned)std::min(nitems, per_sm * sms);
  k_m2l_ts<true><<<grid, kTsThreads, ts_smem_bytes(R), s>>>(R, 0, d_items_run, nullptr, nullptr, nullptr, nullptr, nullptr,
                                                            nullptr, nullptr, err_flag, d_count, d_reqs);
  return check_launch("k_m2l_ts batch");
}

}  // namespace afmpb
