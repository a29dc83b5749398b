// echo_overlap.cu -- the validator's overlap test (Sec. 3: compose, then adjust the
// kernels that overlap communication; Sec. 2.3: their slowdown factor).  This file
// is compiled once for each (ECHO_OV_LAUNCH, ECHO_OV_PROP) pair, so that the four
// families of variants build in parallel; each object defines one entry point.
#include <cuda_runtime.h>

#include <cstdint>

#include "echo_internal.h"
#include "echo_bounds.h"
#include "echo_slowdown.cuh"

#if !defined(ECHO_OV_LAUNCH) || !defined(ECHO_OV_PROP)
#error "compile with -DECHO_OV_LAUNCH=0|1 -DECHO_OV_PROP=0|1"
#endif

namespace echo {
namespace {

using dev::slowed;

// Blocks per SM the register budget allows (kOvWarps warps each); wide cursor sets, and
// the variants that load launch conditions, keep their registers instead of spilling.
constexpr int overlap_min_blocks(int ncmax, bool launch) {
  return ncmax <= 2 ? (launch ? 6 : 8) : ncmax <= 4 ? (launch ? 5 : 6) : ncmax <= 8 ? 4 : 2;
}

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ int64_t s_ld64(uint32_t a) {
  int64_t v;
  asm volatile("ld.shared.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint4 s_ld128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}

// debug bounds: the launch conditions of cq entry e are nodes of the graph
__device__ __noinline__ bool lq_ok(const OverlapArgs &a, int32_t e) {
  bool ok = true;
  for (int32_t k = a.lq_off[e]; k < a.lq_off[e + 1]; ++k) ok &= in_range(a.lq_ops[k], a.rows);
  return ok;
}

// When rank r launched the comm op of cq entry e: the latest finish among its
// launch conditions on r (out of line: the cursor loads are unrolled many times).
__device__ __noinline__ int64_t launch_time(const int32_t *__restrict__ lq_off, const int32_t *__restrict__ lq_ops,
                                            const int64_t *__restrict__ f, int sh, int32_t e) {
  int64_t t = 0;
  for (int32_t k = lq_off[e]; k < lq_off[e + 1]; ++k) t = max(t, f[(int64_t)lq_ops[k] << sh]);
  return t;
}

// The validator's overlap test, as a walk over each rank's candidates.  A warp takes a
// piece of a rank's candidate list (in issue order) for one scenario block (of at most 32):
// 32 / block lanes-wide teams share the piece, team k taking its candidates k, k + teams,
// ..., so that the warp's loads and stores of a step are neighbouring rows of the block
// whatever its width.  Every timeline of a rank runs its ops one after the other, so
// on each comm timeline the intervals are sorted and the candidates' starts only
// grow: the lane keeps, per comm timeline, a cursor at the first comm op of
// positive length that finishes after the current candidate starts, with that
// op's interval in registers.  The candidate overlaps this timeline iff that
// interval starts before the candidate finishes (later comm ops start after the
// cursor op ends).  A piece places its cursors by binary search.  The cursor lists hold
// only the comm ops that can overlap a compute op of the rank, so moves are rare,
// and the smallest cursor end and start decide most candidates with two
// comparisons.  The candidates' records, then their finish times, durations and factors
// come through a ring in shared memory (cp.async), kOvBatch steps at a time, while the
// batch before them is tested: nothing in flight is held in a register that moves.  An
// overlapped compute op of positive length gets rint(d * slowdown) or the proportional
// form for the next composition (cd_next, compact); the decisions themselves are stored
// only when `ov` is given.
// What bounds it: instructions (issue slots half busy and more); with blocks of 1 and 2 each
// team's own search and cursor moves, which the warp runs one after the other.  (Starts and
// finishes in compact matrices of their own: 316 against 306 us on GPT-175B x 250, and the
// composition that writes them 1212 against 1062.)  Measured, before -> now (us):
// GPT-1.3B x 1 80 -> 20, x 256 99 (blocks of 32; 123 in blocks of 2) -> 69, x 500 folded
// 330 -> 35 (its pieces are now cut by the longest rank's list, not the mean of all ranks);
// GPT-175B x 250 338 (blocks of 32; 535 in blocks of 2) -> 306, x 1024 1050 -> 780; 1024
// ranks x 64 1000 -> 678.
// LAUNCH: a comm op's interval on the rank opens at the rank's launch of it
// (a.lq_off), else at its start.  PROP: the proportional slowdown model.
template <int NCMAX, bool LAUNCH, bool PROP>
__global__ void __launch_bounds__(kOvWarps * 32, overlap_min_blocks(NCMAX, LAUNCH)) overlap_kernel(OverlapArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int32_t S = a.S;
  const int lane = threadIdx.x & 31;
  // element (i, s) of a matrix sits at base + (i << sh); blocks of at most 32 scenarios
  const int sh = a.lay.slog2, teams = 32 >> sh, team = lane >> sh;
  const int64_t wid = (int64_t)blockIdx.x * kOvWarps + (threadIdx.x >> 5);
  const int64_t G = (S + (1 << sh) - 1) >> sh;
  if (wid >= (int64_t)a.n_ranks * G * a.parts) return;  // uniform over the warp
  const int32_t part = (int32_t)(wid % a.parts);
  const int32_t r = (int32_t)(wid / a.parts % a.n_ranks);
  const int32_t s = (int32_t)(wid / a.parts / a.n_ranks << sh) + (lane & ((1 << sh) - 1));
  const bool act = s < S;  // (padding lanes of the last block copy and store nothing)
  const int32_t sl = act ? s : S - 1;
  const int nc = a.n_cq;
  // this piece of the rank's list, cut at multiples of the batch
  const int32_t r0 = (int32_t)a.cand_off[r], r1 = (int32_t)a.cand_off[r + 1];
  const int32_t per = teams * kOvBatch, nb = (r1 - r0 + per - 1) / per;
  const int32_t c0 = min(r1, r0 + (int32_t)((int64_t)nb * part / a.parts) * per);
  const int32_t c1 = min(r1, r0 + (int32_t)((int64_t)nb * (part + 1) / a.parts) * per);
  if (c0 >= c1) return;
  const int64_t base = a.lay.at(0, sl);
  const int64_t *__restrict__ f = a.f + base;
  const int64_t *__restrict__ du = a.dur + base;  // comm ops' durations (never slowed)
  // the candidates' durations in the pass that produced f: the original ones, or the
  // previous validator pass's (compact [candidate][scenario] rows)
  const int64_t *__restrict__ cu = a.cd_used ? a.cd_used + a.lay_c.at(0, sl) : nullptr;
  int64_t *__restrict__ cn = a.cd_next ? a.cd_next + a.lay_c.at(0, sl) : nullptr;
  const double *__restrict__ sf = a.sf + sl;
  // per warp: records [3 batches][kOvBatch][teams] of 16 bytes, then values [2
  // batches][kOvBatch][finish, duration, factor][32 lanes]
  const uint32_t recs = (uint32_t)__cvta_generic_to_shared(smem) + (threadIdx.x >> 5) * (uint32_t)overlap_warp_bytes(teams);
  const uint32_t vals = recs + 3 * kOvBatch * 16 * teams + lane * 8;
  const uint32_t row = 8u << sh, rec_step = 16 * teams, rec_batch = kOvBatch * rec_step;
  constexpr uint32_t kValStep = 3 * 256, kValBatch = kOvBatch * kValStep;
  // row x of a matrix from its scenario's first element on
  auto at = [&](const void *m, uint32_t x) { return static_cast<const char *>(m) + (uint64_t)x * row; };
  const int32_t last = act ? c1 : c0;  // this lane's candidates end here
  // per comm timeline: position, end, and interval of the cursor op; the cursor op
  // always has positive length and finishes after the current op's start (or the
  // cursor is at the end, with an interval that never overlaps)
  // (nid: the node of the cursor's next position, loaded one move ahead so that a
  // move waits for the interval's loads only)
  int32_t cur[NCMAX] = {}, end[NCMAX] = {}, nid[NCMAX] = {};
  int64_t sw[NCMAX], fw[NCMAX];
  auto fetch = [&](int j, int64_t w) {  // node w's interval as cursor j's op
    if (a.dbg && !(in_range(w, a.rows) && (!LAUNCH || lq_ok(a, cur[j])))) {  // debug bounds
      atomicCAS(a.status, 0, (int32_t)kDevBounds);
      sw[j] = fw[j] = INT64_MAX;
      return;
    }
    fw[j] = f[w << sh];
    if (LAUNCH) {  // from the rank's launch: its launch conditions' latest finish
      sw[j] = launch_time(a.lq_off, a.lq_ops, f, sh, cur[j]);
    } else {
      sw[j] = fw[j] - du[w << sh];
    }
  };
  auto advance = [&](int j) {  // cursor j one position on
    ++cur[j];
    if (cur[j] < end[j]) {
      const int64_t w = nid[j];
      nid[j] = cur[j] + 1 < end[j] ? a.cq_ops[cur[j] + 1] : 0;
      fetch(j, w);
    } else {
      sw[j] = fw[j] = INT64_MAX;
    }
  };
  // records of the batch whose first candidate is i0, into `to`: one lane of each team
  // copies its own
  auto copy_recs = [&](int32_t i0, uint32_t to) {
    if ((lane & ((1 << sh) - 1)) == 0) {
#pragma unroll
      for (int u = 0; u < kOvBatch; ++u) {
        const int32_t i = i0 + u * teams + team;
        if (i < c1) cp_async<16>(to + team * 16 + u * rec_step, a.cand_rec + i);
      }
    }
  };
  bool bad = false;  // debug bounds: a record with an index out of range
  const void *const d_of = cu ? (const void *)cu : (const void *)du;
  auto copy_vals = [&](int32_t i0, uint32_t rec, uint32_t to) {
#pragma unroll
    for (int u = 0; u < kOvBatch; ++u) {
      if (i0 + u * teams + team < last) {
        const uint4 q = s_ld128(rec + team * 16 + u * rec_step);
        if (a.dbg && !(in_range(q.x, a.rows) && in_range(q.y, a.c_rows) && in_range(q.z, a.n_kclass))) {
          bad = true;
          atomicCAS(a.status, 0, (int32_t)kDevBounds);
        } else {
          cp_async<8>(to + u * kValStep, at(f, q.x));
          cp_async<8>(to + u * kValStep + 256, at(d_of, cu ? q.y : q.x));
          cp_async<8>(to + u * kValStep + 512, sf + (uint64_t)q.z * (uint32_t)S);
        }
      }
    }
  };
  // rings: records of this batch, of the next, of the one after it; values of this batch, of the next
  uint32_t rec0 = recs, rec1 = recs + rec_batch, rec2 = recs + 2 * rec_batch, val0 = vals, val1 = vals + kValBatch;
  copy_recs(c0, rec0);
  copy_recs(c0 + per, rec1);
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
  __syncwarp();
  copy_vals(c0, rec0, val0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  // the cursors of this lane's first candidate
  {
    int64_t sv0 = 0;
    if (part > 0 || team > 0) {
      const int32_t i = min(c0 + team, c1 - 1);  // (a team without a candidate looks for nothing)
      const uint4 q = a.cand_rec[i];
      if (a.dbg && !(in_range(q.x, a.rows) && in_range(q.y, a.c_rows))) {  // debug bounds
        atomicCAS(a.status, 0, (int32_t)kDevBounds);
        bad = true;
      } else {
        sv0 = f[(int64_t)q.x << sh] - (cu ? cu[(int64_t)q.y << sh] : du[(int64_t)q.x << sh]);
      }
    }
    // binary searches (first comm op finishing after sv0; finishes are sorted): of many
    // timelines side by side, so that a round waits for memory twice and not twice a timeline
    // (1024 ranks x 64: 767 -> 709 us); of few one after the other, which
    // needs fewer registers (GPT-1.3B x 45, launch intervals: 47 us, side by side 51)
    constexpr bool kTogether = NCMAX > 4;
    const bool inner = part > 0 || team > 0;
    int32_t hi[NCMAX];
#pragma unroll
    for (int j = 0; j < NCMAX; ++j) {
      cur[j] = j < nc ? (int32_t)a.cq_off[r * nc + j] : 0;
      end[j] = j < nc ? (int32_t)a.cq_off[r * nc + j + 1] : 0;
      hi[j] = inner ? end[j] : cur[j];
      sw[j] = fw[j] = INT64_MAX;
    }
    auto search = [&](int j) { return cur[j] < hi[j]; };
#pragma unroll
    for (int j = 0; j < NCMAX; ++j)
      while (!kTogether && search(j)) {
        const int32_t mid = (cur[j] + hi[j]) >> 1, w = a.cq_ops[mid];
        if (a.dbg && !in_range(w, a.rows)) {  // debug bounds: stop searching
          atomicCAS(a.status, 0, (int32_t)kDevBounds);
          hi[j] = cur[j];
        } else if (f[(int64_t)w << sh] > sv0) {
          hi[j] = mid;
        } else {
          cur[j] = mid + 1;
        }
      }
    while (kTogether) {
      bool any = false;
#pragma unroll
      for (int j = 0; j < NCMAX; ++j)
        if (search(j)) {
          any = true;
          nid[j] = a.cq_ops[(cur[j] + hi[j]) >> 1];
          if (a.dbg && !in_range(nid[j], a.rows)) {  // debug bounds: stop searching
            atomicCAS(a.status, 0, (int32_t)kDevBounds);
            hi[j] = cur[j];
          }
        }
      if (!any) break;
#pragma unroll
      for (int j = 0; j < NCMAX; ++j)
        if (search(j)) fw[j] = f[(int64_t)nid[j] << sh];
#pragma unroll
      for (int j = 0; j < NCMAX; ++j)
        if (search(j)) {
          const int32_t mid = (cur[j] + hi[j]) >> 1;
          if (fw[j] > sv0)
            hi[j] = mid;
          else
            cur[j] = mid + 1;
        }
    }
#pragma unroll
    for (int j = 0; j < NCMAX; ++j)
      if (cur[j] < end[j]) nid[j] = a.cq_ops[cur[j]];
#pragma unroll
    for (int j = 0; j < NCMAX; ++j) {
      if (cur[j] < end[j])
        fetch(j, nid[j]);
      else
        sw[j] = fw[j] = INT64_MAX;
    }
#pragma unroll
    for (int j = 0; j < NCMAX; ++j) nid[j] = cur[j] + 1 < end[j] ? a.cq_ops[cur[j] + 1] : 0;
#pragma unroll
    for (int j = 0; j < NCMAX; ++j)
      while (cur[j] < end[j] && sw[j] >= fw[j]) advance(j);  // zero-length ops never overlap
  }
  // The smallest cursor end and start over the timelines: while every cursor op
  // ends after a candidate starts (fmin > sv), no cursor moves, and the candidate
  // overlaps iff some cursor op starts before it ends (smin < fv).
  // (Up to four timelines are compared one by one: as many instructions, and none a move.)
  constexpr bool kDirect = NCMAX <= 4;
  int64_t fmin, smin;
  auto bounds = [&]() {
    if (kDirect) return;
    fmin = smin = INT64_MAX;
#pragma unroll
    for (int j = 0; j < NCMAX; ++j)
      if (j < nc) {
        fmin = min(fmin, fw[j]);
        smin = min(smin, sw[j]);
      }
  };
  bounds();
#pragma unroll 1
  for (int32_t i0 = c0; i0 < c1; i0 += per) {
    // one wait a batch: the records of the next batch and the values of this one, both
    // asked for a batch ago
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncwarp();  // (records are read by the lanes of the team that did not copy them)
    copy_recs(i0 + 2 * per, rec2);
    copy_vals(i0 + per, rec1, val1);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (a.dbg && __any_sync(0xffffffffu, bad)) break;  // (the copies in flight land below)
    uint32_t rec = rec0 + team * 16, val = val0;
#pragma unroll 1
    for (int32_t i = i0 + team, u = 0; u < kOvBatch && i < last; ++u, i += teams, rec += rec_step, val += kValStep) {
      const int64_t fv = s_ld64(val), dv = s_ld64(val + 256), sv = fv - dv;
      const uint4 q = s_ld128(rec);
      bool move = !kDirect && fmin <= sv;
      if (kDirect) {
#pragma unroll
        for (int j = 0; j < NCMAX; ++j) move |= fw[j] <= sv;
      }
      if (move) {
#pragma unroll
        for (int j = 0; j < NCMAX; ++j) {
          if (fw[j] <= sv) {  // the cursor op ended before this op starts: move on
            do {
              advance(j);
            } while (cur[j] < end[j] && (fw[j] <= sv || sw[j] >= fw[j]));
          }
        }
        bounds();
      }
      bool hit = !kDirect && smin < fv;
      if (kDirect) {
#pragma unroll
        for (int j = 0; j < NCMAX; ++j) hit |= sw[j] < fv;
      }
      hit &= sv < fv;
      int64_t len = 0;
      if (PROP && hit && cn) {
        // proportional model: the length of [sv, fv) covered by the union of the
        // comm intervals, swept in start order across the timelines.  Later
        // candidates start no earlier than fv, so a cursor moves past every
        // interval that ends by fv; one reaching beyond fv stays.
        int64_t covered = sv;
        uint32_t held = 0;  // timelines whose cursor interval reaches beyond fv
        while (true) {
          int jb = -1;
          int64_t first = fv;
#pragma unroll
          for (int j = 0; j < NCMAX; ++j)
            if (j < nc && !((held >> j) & 1) && sw[j] < first) {
              first = sw[j];
              jb = j;
            }
          if (jb < 0) break;
#pragma unroll
          for (int j = 0; j < NCMAX; ++j) {  // (j == jb, in registers)
            if (j != jb) continue;
            const int64_t lo = max(sw[j], covered), hi = min(fw[j], fv);
            if (hi > lo) {
              len += hi - lo;
              covered = hi;
            }
            if (fw[j] > fv) {
              held |= 1u << j;
            } else {
              do {
                advance(j);
              } while (cur[j] < end[j] && sw[j] >= fw[j]);
            }
          }
        }
        bounds();
      }
      if (a.ov) a.ov[base + ((int64_t)q.x << sh)] = hit;
      if (cn) {
        const int64_t d0 = cu ? *reinterpret_cast<const int64_t *>(at(du, q.x)) : dv;  // the original duration
        int64_t dn = d0;
        if (hit) {
          const int64_t factor = s_ld64(val + 512);  // (its bits)
          dn = PROP ? dev::slowed_proportional(d0, __longlong_as_double(factor), len) : slowed(d0, factor);
        }
        *reinterpret_cast<int64_t *>(const_cast<char *>(at(cn, q.y))) = dn;
      }
    }
    const uint32_t r = rec0, v = val0;
    rec0 = rec1;
    rec1 = rec2;
    rec2 = r;
    val0 = val1;
    val1 = v;
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

}  // namespace

#define ECHO_OV_CAT(l, p) launch_overlap_l##l##_p##p
#define ECHO_OV_NAME(l, p) ECHO_OV_CAT(l, p)

cudaError_t ECHO_OV_NAME(ECHO_OV_LAUNCH, ECHO_OV_PROP)(const OverlapArgs &a, dim3 grid, int tx, cudaStream_t st) {
  const size_t smem = kOvWarps * overlap_warp_bytes(32 >> a.lay.slog2);  // (at most 48 KB)
  constexpr bool L = ECHO_OV_LAUNCH != 0, P = ECHO_OV_PROP != 0;
  if (a.n_cq <= 1)
    overlap_kernel<1, L, P><<<grid, tx, smem, st>>>(a);
  else if (a.n_cq <= 2)
    overlap_kernel<2, L, P><<<grid, tx, smem, st>>>(a);
  else if (a.n_cq <= 3)
    overlap_kernel<3, L, P><<<grid, tx, smem, st>>>(a);
  else if (a.n_cq <= 4)
    overlap_kernel<4, L, P><<<grid, tx, smem, st>>>(a);
  else if (a.n_cq <= 6)
    overlap_kernel<6, L, P><<<grid, tx, smem, st>>>(a);
  else if (a.n_cq <= 8)
    overlap_kernel<8, L, P><<<grid, tx, smem, st>>>(a);
  else
    overlap_kernel<kMaxStreams, L, P><<<grid, tx, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace echo
