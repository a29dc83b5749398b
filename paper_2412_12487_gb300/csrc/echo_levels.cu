// echo_levels.cu -- the levelled composer (Sec. 4.2, 5.2): the max-plus pass over the
// multi-rank execution graph, batched over scenario blocks, as a pipeline of warp
// roles inside one thread block per scenario block.
//
// Along a segment (a serial chain) an op's finish is the segment's start plus the
// running sum of its durations, and the sums need nothing from the rest of the graph.
// So only one addition per segment is serial along the critical path of levels;
// everything else is done ahead of it or behind it, by other warps, each at its own
// pace:
//   copy warps   one level after another, as far ahead as the shared-memory ring
//                allows, by the bulk-copy engine: records, duration rows and the
//                candidates' rows, and one warp the heads' programs;
//   sum warps    every segment's sum (a candidate's duration taken from the validator's
//                rows);
//   head warps   the only serial part: start = max over the head's inputs, finish of
//                the tail = start + the segment's sum, one barrier per level;
//   store warps  finish = start + running sum, for every row or only those a later
//                step reads.
// Stage l % kLvStages has a barrier after each role: full -> summed -> headed ->
// stored -> (the ring space is free).
//
// What bounds it: with few scenarios a block (1 and 2) the head warps, about 500 cycles a
// level; with 8 the shared-memory pipe and instruction issue (60-77% and 59% busy, the
// same time with 16 blocks on the device as with 128, so not memory).  One set of
// warps doing all of this between two barriers took 1.1 us a level.
// Measured, first / final composition (us), before -> now:
//   GPT-1.3B x 1      415 / 453   ->  138 / 143   (dataflow composer before)
//   GPT-1.3B x 256    415 / 461   ->  159 / 180   (dataflow composer before)
//   GPT-175B x 250   2895 / 3099  -> 1060 / 1200  (dataflow composer before)
//   GPT-175B x 1024  3362 / 3731  -> 2110 / 3100
#include <cuda_runtime.h>

#include <cstdint>

#include "echo_bounds.h"
#include "echo_internal.h"

namespace echo {
namespace {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// addresses 16-byte aligned, size a multiple of 16; completes `bytes` on the mbarrier
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// orders this thread's shared-memory accesses before later bulk copies into the same space
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

// N consecutive int64 of shared memory at byte address a (a 16-byte vector for N == 2)
template <int N>
__device__ __forceinline__ void s_load(uint32_t a, int64_t (&v)[N]) {
  if constexpr (N == 2)
    asm("ld.shared.v2.s64 {%0, %1}, [%2];\n" : "=l"(v[0]), "=l"(v[1]) : "r"(a) : "memory");
  else
    asm("ld.shared.s64 %0, [%1];\n" : "=l"(v[0]) : "r"(a) : "memory");
}
template <int N>
__device__ __forceinline__ void s_store(uint32_t a, const int64_t (&v)[N]) {
  if constexpr (N == 2)
    asm volatile("st.shared.v2.s64 [%0], {%1, %2};\n" ::"r"(a), "l"(v[0]), "l"(v[1]) : "memory");
  else
    asm volatile("st.shared.s64 [%0], %1;\n" ::"r"(a), "l"(v[0]) : "memory");
}
template <int N>
__device__ __forceinline__ void g_store(int64_t *p, const int64_t (&v)[N]) {
  if constexpr (N == 2)
    *reinterpret_cast<longlong2 *>(p) = make_longlong2(v[0], v[1]);
  else
    *p = v[0];
}
__device__ __forceinline__ uint32_t s_ld32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t s_ld16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];\n" : "=h"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint4 s_ld128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a)
               : "memory");
  return v;
}

// What one thread block shares: barriers, counts and places (byte addresses in shared
// memory).
struct Shared {
  uint64_t *full, *summed, *headed, *stored;  // [kLvStages] each
  uint64_t *heads;                            // [kLvStages / kLvGroup] head programs landed
  uint32_t counts, out;                       // [kLvStages] sum (store) warps that are done with the stage's levels, ever
  uint32_t chunk;                             // [kLvStages] address of the level's chunk (its descriptor)
  uint32_t prog;                              // [kLvStages] head programs, a.prog_bytes each
  uint32_t base, ring;
  volatile int32_t *abort;
};
constexpr uint32_t kStageMask = kLvStages - 1;
__device__ __forceinline__ uint32_t desc_of(const Shared &sh, int32_t l) {
  return s_ld32(sh.chunk + 4 * (l & kStageMask));
}

// Give up a wait once the limit passes or another warp of the block gave up (every role
// then leaves its walk).
__device__ __noinline__ bool lv_expired(volatile int32_t *abort, long long t0, long long limit, int32_t *status) {
  if (*abort) return true;
  if (clock64() - t0 <= limit) return false;
  *abort = 1;
  atomicCAS(status, (int32_t)kDevOk, (int32_t)kDevTimeout);
  return true;
}
// Wait for use n of a barrier; false when the wait gave up.
__device__ __forceinline__ bool lv_wait(uint64_t *bar, uint32_t n, const Shared &sh, const LevelArgs &a) {
  if (mbar_try_wait(bar, n & 1)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, n & 1))
    if (lv_expired(sh.abort, t0, a.wait_limit_cycles, a.status)) return false;
  return true;
}
// Wait until a stage's count (a word at `count` that the warps of a level add to) reaches
// `want`.  The level's phase of `bar` is what the warp sleeps on, the count decides: it
// also tells of a level that is long past.
__device__ __forceinline__ uint32_t ld_count(uint32_t count) {
  uint32_t n;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(n) : "r"(count) : "memory");
  return n;
}
__device__ __noinline__ bool lv_wait_count(uint32_t count, uint32_t want, uint64_t *bar, uint32_t n, volatile int32_t *abort,
                                           long long limit, int32_t *status) {
  const long long t0 = clock64();
#pragma unroll 1
  while (ld_count(count) < want) {
    if (*abort) return false;
    if (!mbar_try_wait(bar, n & 1) && lv_expired(abort, t0, limit, status)) return false;
  }
  return true;
}
__device__ __forceinline__ void lv_bad(const Shared &sh, const LevelArgs &a) {  // a debug-bounds check failed
  *sh.abort = 1;
  atomicCAS(a.status, (int32_t)kDevOk, (int32_t)kDevBounds);
}

// Debug bounds: what a step's descriptor places (records and masks, duration rows, starts,
// candidates' rows and the row list) lies in the ring, at the alignment that it is read
// with, and its rows in the matrix.  (Out of line: the checking variant only.)
template <int SIGMA>
__device__ __noinline__ bool desc_ok(const LevelArgs &a, const uint4 &m, const uint4 &m2) {
  constexpr uint32_t kRow = SIGMA * 8, kVec = SIGMA >= 2 ? 16 : 8;
  const int64_t segs = m.y & 0xFFFF, rows = m.y >> 16, cands = m2.x >> 16, R = a.ring_bytes;
  const int64_t recs = cands ? ((4 * segs + 15) & ~15) + 16 * segs : 4 * segs;
  return place_ok(m.x, recs, 16, R) && place_ok(m.z, rows * kRow, kVec, R) && place_ok(m.w, segs * kRow, kVec, R) &&
         (!cands || place_ok(m2.z, cands * kRow, kVec, R)) && (level_walks(SIGMA) || place_ok(m2.w, 2 * rows, 2, R)) &&
         range_ok(m2.y, m2.y + rows, a.pitch);
}

// ---- copy warps: kLvCopyWarps of them take the levels in turn ------------------------
// A bulk copy costs its issuing thread about 220 cycles and each further one right after
// it 50, and the fence 250 while other warps store to global memory (measured apart from
// the rest), so one warp would copy a level every 700 cycles.
// `plan`: for every level the copies of its records, durations and candidates' durations,
// {byte offset in the ring, last level that must have been stored, first unit of the
// source, units} each.  The whole warp waits (a lone lane would spin instead of
// sleeping), one lane issues.
template <int SIGMA, bool ALL, bool DBG>
__device__ void copy_role(const LevelArgs &a, const Shared &sh, int c, int lane) {
  const uint4 *plan = reinterpret_cast<const uint4 *>(a.meta);
  const uint4 *recs = reinterpret_cast<const uint4 *>(ALL ? a.recs_all : a.recs_kept);
  const int64_t n_recs = ALL ? a.n_recs_all : a.n_recs_kept;
  const int64_t *dur = a.dur + (int64_t)blockIdx.x * a.pitch * SIGMA;
  const int64_t *cdur = a.cdur ? a.cdur + (int64_t)blockIdx.x * a.c_pitch * SIGMA : nullptr;
  // (registers that a load is still to fill are never moved, only indexed by the unrolled
  // loop: a move would wait for the load, about 700 cycles)
  uint4 m[2][3];
  auto load = [&](uint4 (&x)[3], int32_t l) {
    l = min(l, a.L - 1);
    x[0] = __ldg(plan + (ALL ? 0 : 1) * (int64_t)a.L + l);
    x[1] = __ldg(plan + 2 * (int64_t)a.L + l);
    x[2] = __ldg(plan + 3 * (int64_t)a.L + l);
  };
  load(m[0], c);
  load(m[1], c + kLvCopyWarps);
  int32_t done = 0;  // every level < done has been stored
  int32_t last = -1; // the last level this warp has armed
  bool ok = true;
#pragma unroll 1
  for (int32_t l0 = c; l0 < a.L && ok; l0 += 2 * kLvCopyWarps) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int32_t l = l0 + i * kLvCopyWarps;
      ok = ok && l < a.L && (a.skip_level < 0 || l < a.skip_level);  // failure injection: skip_level never arrives
      if (!ok) break;
      const uint4 r = m[i][0], d = m[i][1], q = m[i][2];
      const uint32_t b_rec = r.w * 16, b_dur = d.w * (SIGMA * 8), b_cand = a.cdur ? q.w * (SIGMA * 8) : 0;
      const int32_t dep = max((int32_t)r.y, l - kLvStages);
      if (DBG && !(range_ok(r.z, (int64_t)r.z + r.w, n_recs) && range_ok(d.z, (int64_t)d.z + d.w, a.pitch) &&
                   (!a.cdur || range_ok(q.z, (int64_t)q.z + q.w, a.c_pitch)) &&
                   range_ok(r.x, (int64_t)r.x + b_rec, a.ring_bytes) && range_ok(d.x, (int64_t)d.x + b_dur, a.ring_bytes) &&
                   range_ok(q.x, (int64_t)q.x + b_cand, a.ring_bytes) && (r.x | d.x | (b_cand ? q.x : 0)) % 16 == 0 &&
                   (d.z | d.w | (a.cdur ? q.z | q.w : 0)) * SIGMA % 2 == 0 && dep < l)) {
        lv_bad(sh, a);
        ok = false;
        break;
      }
      // the ring space and the stage are free once every level <= dep has been stored: at
      // most kLvStages levels in doubt, a lane for each
#pragma unroll 1
      while (ok && done <= dep) {
        const int32_t x = done + lane;
        auto want = [&](int32_t y) { return (uint32_t)a.store_team * ((uint32_t)y / kLvStages + 1); };
        const bool out = lane >= kLvStages || x > dep || ld_count(sh.out + 4 * (x & kStageMask)) >= want(x);
        const uint32_t open = __ballot_sync(0xffffffffu, !out);
        if (!open) {
          done = min(done + kLvStages, dep + 1);
        } else {
          done += __ffs(open) - 1;
          ok = __all_sync(0xffffffffu, lv_wait_count(sh.out + 4 * (done & kStageMask), want(done), sh.stored + (done & kStageMask), done / kLvStages, sh.abort, a.wait_limit_cycles, a.status));
        }
      }
      if (!ok) break;
      if (lane == 0) {
        fence_async();  // the other roles' accesses to the space come before the copies into it
        uint64_t *bar = &sh.full[l & kStageMask];
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(sh.chunk + 4 * (l & kStageMask)), "r"(sh.ring + r.x) : "memory");
        mbar_arrive_expect_tx(bar, b_rec + b_dur + b_cand);
        bulk_g2s(sh.ring + r.x, recs + r.z, b_rec, bar);
        bulk_g2s(sh.ring + d.x, dur + (int64_t)d.z * SIGMA, b_dur, bar);
        if (b_cand) bulk_g2s(sh.ring + q.x, cdur + (int64_t)q.z * SIGMA, b_cand, bar);
      }
      __syncwarp();
      last = l;
      load(m[i], l + 2 * kLvCopyWarps);
    }
  }
  // let the copies this warp started land before the block exits
  const long long t0 = clock64();
#pragma unroll 1
  for (int32_t l = last; l >= 0 && l > last - kLvStages; l -= kLvCopyWarps)
    while (!mbar_try_wait(&sh.full[l & kStageMask], ((uint32_t)l / kLvStages) & 1))
      if (clock64() - t0 > a.wait_limit_cycles) {
        atomicCAS(a.status, (int32_t)kDevOk, (int32_t)kDevTimeout);
        break;
      }
}

// ---- copy warp of the head programs: kLvGroup levels a copy ---------------------------
template <bool DBG>
__device__ void head_copy_role(const LevelArgs &a, const Shared &sh, int lane) {
  constexpr int kG = kLvStages / kLvGroup;  // groups in flight
  const int32_t n = (a.L + kLvGroup - 1) / kLvGroup;
  const uint32_t bytes = a.prog_bytes * kLvGroup;
  int32_t g = 0;
#pragma unroll 1
  for (; g < n; ++g) {
    if (g >= kG) {  // every level of the group before it in the same place has been headed
      const int32_t top = (g - kG + 1) * kLvGroup - 1;
      if (!__all_sync(0xffffffffu, lv_wait(sh.headed + (top & kStageMask), top / kLvStages, sh, a))) break;
    }
    if (lane == 0) {
      fence_async();
      uint64_t *bar = &sh.heads[g % kG];
      mbar_arrive_expect_tx(bar, bytes);
      bulk_g2s(sh.prog + g % kG * bytes, reinterpret_cast<const char *>(a.heads) + (int64_t)g * bytes, bytes, bar);
    }
    __syncwarp();
  }
  const long long t0 = clock64();  // (its copies land before the block exits)
#pragma unroll 1
  for (int32_t x = max(0, g - kG); x < g; ++x)
    while (!mbar_try_wait(&sh.heads[x % kG], (x / kG) & 1))
      if (clock64() - t0 > a.wait_limit_cycles) {
        atomicCAS(a.status, (int32_t)kDevOk, (int32_t)kDevTimeout);
        break;
      }
}

// ---- sum warps ------------------------------------------------------------------------
// Teams of warps take the levels in turn: what a warp spends on a level besides its
// segments (the wait, the descriptor, the loop: about 60 instructions) is paid once per
// level and not by every warp.  A thread takes a segment for LV scenarios.
//
// Blocks of 4 scenarios and more (level_walks) only add the chain up here, and the store
// warps walk it again from its start: shared memory is what bounds such a block (80% of
// its cycles busy when every running sum was written and read back), and this reads each
// row twice where the other way reads it twice and writes it once.  Narrower blocks write
// the running sums in place: their store warps then run over rows and not over segments,
// so that the lanes of a warp store to consecutive addresses.
//
// Running sums in place: four rows at a time, the next four in flight (past the segment's
// end it loads rows that it does not use; the block's shared memory has room for them).
template <int SIGMA, bool CANDS>
__device__ __forceinline__ void sum_segment(uint32_t p, uint32_t n, uint32_t q, uint64_t mask) {
  constexpr int LV = SIGMA >= 2 ? 2 : 1;
  constexpr uint32_t kRow = SIGMA * 8;
  int64_t d[4][LV], e[4][LV], acc[LV];
#pragma unroll
  for (int i = 0; i < LV; ++i) acc[i] = 0;
  uint32_t at = p;
  auto load4 = [&](int64_t (&x)[4][LV]) {  // the next four rows; a candidate's comes from its own row
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      if (CANDS) {
        const bool c = mask & 1;
        s_load<LV>(c ? q : at + u * kRow, x[u]);
        q += c ? kRow : 0;
        mask >>= 1;
      } else {
        s_load<LV>(at + u * kRow, x[u]);
      }
    }
    at += 4 * kRow;
  };
  auto put = [&](uint32_t u) {
#pragma unroll
    for (int i = 0; i < LV; ++i) acc[i] += d[u][i];
    s_store<LV>(p + u * kRow, acc);
  };
  load4(d);
#pragma unroll 1
  for (; n >= 4; n -= 4) {
    load4(e);
    put(0);
    put(1);
    put(2);
    put(3);
    p += 4 * kRow;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int i = 0; i < LV; ++i) d[u][i] = e[u][i];
  }
  if (n > 0) put(0);
  if (n > 1) put(1);
  if (n > 2) put(2);
}

// The rows [t, t + R) of a chain at p, 0 past its end; a candidate's row (a bit of mask)
// comes from q on, one after another.
template <int SIGMA, int R>
__device__ __forceinline__ void load_rows(int64_t (&x)[R][2], uint32_t p, uint32_t t, uint32_t len, uint32_t &q,
                                          uint64_t &mask) {
  constexpr uint32_t kRow = SIGMA * 8;
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const bool c = mask & 1;
    x[u][0] = x[u][1] = 0;
    if (t + u < len) s_load<2>(c ? q : p + (t + u) * kRow, x[u]);
    q += c ? kRow : 0;
    mask >>= 1;
  }
}

template <int SIGMA, bool DBG>
__device__ void sum_role(const LevelArgs &a, const Shared &sh, int team, int teams, int w, int nw, int lane) {
  constexpr int LV = SIGMA >= 2 ? 2 : 1, TPS = SIGMA / LV, SPW = 32 / TPS;  // segments per warp
  constexpr uint32_t kRow = SIGMA * 8;
  const uint32_t j = (lane % TPS) * LV * 8, sw = w * SPW + lane / TPS;
#pragma unroll 1
  for (int32_t l = team; l < a.L; l += teams) {
    if (!__all_sync(0xffffffffu, lv_wait(sh.full + (l & kStageMask), l / kLvStages, sh, a))) return;
    const uint32_t ds = desc_of(sh, l);
    const uint4 m = s_ld128(ds);
    uint32_t nseg = m.y & 0xFFFF;
    const uint32_t recs = sh.ring + m.x, dur = sh.ring + m.z + j;
    if (DBG && !desc_ok<SIGMA>(a, m, s_ld128(ds + 16))) {
      lv_bad(sh, a);
      nseg = 0;
    }
#pragma unroll 1
    for (uint32_t k = sw; k < nseg; k += (uint32_t)nw * SPW) {
      const uint32_t h = s_ld32(recs + 4 * k);
      const uint32_t len = (h >> 16) & 0xFF;
      if (DBG && !(len > 0 && range_ok(h & 0xFFFF, (int64_t)(h & 0xFFFF) + len, m.y >> 16))) {
        lv_bad(sh, a);
        continue;
      }
      const uint32_t p = dur + (h & 0xFFFF) * kRow;
      uint64_t mask = 0;
      uint32_t q = 0;
      if (a.cdur && (h >> 24)) {  // the segment holds candidates: mask of their chain positions, first row
        const uint4 m2 = s_ld128(ds + 16), c = s_ld128(recs + ((4 * nseg + 15) & ~15u) + 16 * k);
        mask = (uint64_t)c.x | ((uint64_t)c.y << 32);
        q = sh.ring + m2.z + j + c.z * kRow;
        if (DBG && !masked_row_ok(c.z, mask, m2.x >> 16)) {
          lv_bad(sh, a);
          continue;
        }
      }
      if constexpr (level_walks(SIGMA)) {
        int64_t acc[2] = {0, 0};
        uint32_t t = 0, p1 = p;
        if (!mask)  // (whole groups of rows, without a test for each: half the instructions)
#pragma unroll 1
          for (; t + 8 <= len; t += 8, p1 += 8 * kRow) {
            int64_t x[8][2];
#pragma unroll
            for (int u = 0; u < 8; ++u) s_load<2>(p1 + u * kRow, x[u]);
#pragma unroll
            for (int i = 0; i < 2; ++i)
              acc[i] += ((x[0][i] + x[1][i]) + (x[2][i] + x[3][i])) + ((x[4][i] + x[5][i]) + (x[6][i] + x[7][i]));
          }
#pragma unroll 1
        for (; t < len; t += 4) {
          int64_t x[4][2];
          load_rows<SIGMA, 4>(x, p, t, len, q, mask);
#pragma unroll
          for (int i = 0; i < 2; ++i) acc[i] += (x[0][i] + x[1][i]) + (x[2][i] + x[3][i]);
        }
        s_store<2>(sh.ring + m.w + j + k * kRow, acc);  // the head replaces it by the start
      } else if (mask) {
        sum_segment<SIGMA, true>(p, len, q, mask);
      } else {
        sum_segment<SIGMA, false>(p, len, 0, 0);
      }
    }
    __syncwarp();
    if (lane == 0) {
      asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(sh.counts + 4 * (l & kStageMask)) : "memory");
      mbar_arrive(&sh.summed[l & kStageMask]);
    }
  }
}

// ---- head warps: the serial part ----------------------------------------------------
// A thread takes a segment for LV scenarios, as the level's head program says: 16 bytes a
// segment, eight 16-bit places in shared memory in units of 8 bytes: the segment's sum
// (its last row), its start, the slot of its finish, four inputs, and a list of further
// ones (0: none).  Unused inputs name a slot that holds 0, unused outputs one that nobody
// reads, and a level's program has an entry for every thread, so no thread has to ask
// whether it has a segment.  The program is loaded two levels ahead, so the path from one
// barrier to the next is one round of loads (sum and inputs), the maxima, an addition, a
// store.  A head thread whose wait gave up stays in the barriers and does nothing else.
// (Two groups of head warps with half of the scenarios and a barrier each: 3.0 against 2.8
// ms on GPT-175B x 1024, as the instructions of all warps together limit such blocks.)
// Puts the largest tail finishes into mk_s.
template <int SIGMA, bool DBG>
__device__ void head_role(const LevelArgs &a, const Shared &sh, int t, int nt, int64_t *mk_s) {
  constexpr int LV = SIGMA >= 4 ? 2 : 1, TPS = SIGMA / LV;
  constexpr int kG = kLvStages / kLvGroup;
  const int j = t % TPS * LV;                     // this thread's first scenario
  const uint32_t at = sh.base + j * 8;            // it in the row at place 0
  const uint32_t prog = sh.prog + t / TPS * 16;
  int64_t mk[LV];
#pragma unroll
  for (int i = 0; i < LV; ++i) mk[i] = 0;
  bool ok = true;
  // debug bounds: a place of `n` values in shared memory, aligned as it is read
  auto inside = [&](uint32_t place, int64_t n, uint32_t align) {
    return place_ok(place, n, align, a.smem_bytes / 8);
  };
  constexpr uint32_t kZero = kLvFixedBytes / 8;  // slot 0
  auto row = [&](uint32_t place, int64_t (&x)[LV]) {
    if (DBG && !inside(place, SIGMA, LV)) {
      lv_bad(sh, a);
      place = kZero;
    }
    s_load<LV>(at + place * 8, x);
  };
  auto top = [&](int64_t (&x)[LV], const int64_t (&y)[LV]) {
#pragma unroll
    for (int i = 0; i < LV; ++i) x[i] = max(x[i], y[i]);
  };
  auto two = [&](uint32_t w, int64_t (&x)[LV]) {  // the larger of the two inputs of a word
    int64_t y[LV];
    row(w & 0xFFFF, x);
    row(w >> 16, y);
    top(x, y);
  };
  auto step = [&](const uint4 &h) {
    int64_t sum[LV], s[LV], v[LV], u[LV], w[LV];
    row(h.x & 0xFFFF, sum);
    row(h.y >> 16, s);
    row(h.z & 0xFFFF, u);
    row(h.z >> 16, v);
    row(h.w & 0xFFFF, w);
    top(s, u);
    top(v, w);
    top(s, v);
    uint32_t more = h.w >> 16;
    if (DBG && more && !inside(more, 2, 2)) {  // (its first piece, before that is read)
      lv_bad(sh, a);
      more = 0;
    }
    if (more) {  // a list: pieces of 16 bytes, the first {pieces, six inputs}, the others eight inputs
      uint32_t e = sh.base + more * 8;
      uint4 y = s_ld128(e);
      uint32_t n = y.x;
      y.x = 0;
      if (DBG && !(n > 0 && inside(more, 2 * (int64_t)n, 2))) {
        lv_bad(sh, a);
        n = 1;
      }
#pragma unroll 1
      while (true) {
        if (y.x) {
          two(y.x, u);
          top(s, u);
        }
        two(y.y, u);
        two(y.z, v);
        two(y.w, w);
        top(u, v);
        top(s, w);
        top(s, u);
        if (--n == 0) break;
        e += 16;
        y = s_ld128(e);
      }
    }
    int64_t f[LV];
#pragma unroll
    for (int i = 0; i < LV; ++i) f[i] = s[i] + sum[i];
    if (DBG && !(inside(h.x >> 16, SIGMA, LV) && inside(h.y & 0xFFFF, SIGMA, LV))) {
      lv_bad(sh, a);
      return;
    }
    s_store<LV>(at + (h.y & 0xFFFF) * 8, f);
    s_store<LV>(at + (h.x >> 16) * 8, s);
    top(mk, f);
  };
  auto program = [&](int32_t l) {
    if (l % kLvGroup == 0 && l < a.L && ok) ok = lv_wait(sh.heads + l / kLvGroup % kG, l / kLvStages, sh, a);
    return s_ld128(prog + (l & kStageMask) * a.prog_bytes);
  };
  auto count = [&](int32_t l) { return sh.counts + 4 * (l & kStageMask); };
  uint4 h0 = program(0), h1 = program(1);
  uint32_t c = ld_count(count(0));
#pragma unroll 2
  for (int32_t l = 0; l < a.L; ++l) {
    const uint32_t want = (uint32_t)a.sum_team * ((uint32_t)l / kLvStages + 1);
    if (c < want && ok)
      ok = lv_wait_count(count(l), want, sh.summed + (l & kStageMask), l / kLvStages, sh.abort, a.wait_limit_cycles, a.status);
    const uint4 h2 = program(l + 2);
    c = ld_count(count(l + 1));
    if (ok) step(h0);
    named_barrier(1, nt);
    if (t == 0 && ok) mbar_arrive(&sh.headed[l & kStageMask]);
    h0 = h1;
    h1 = h2;
  }
#pragma unroll
  for (int i = 0; i < LV; ++i)
    atomicMax(reinterpret_cast<unsigned long long *>(&mk_s[j + i]), (unsigned long long)mk[i]);
}

// ---- store warps: finish = start + running sum (teams as above) ----------------------
// The walk: the segment's rows again, from its start.  `mask` of the kept rows (all of
// them in the final composition).
template <int SIGMA, bool ALL, bool DBG>
__device__ void walk_role(const LevelArgs &a, const Shared &sh, int team, int teams, int w, int nw, int lane) {
  constexpr int TPS = SIGMA / 2, SPW = 32 / TPS;
  constexpr uint32_t kRow = SIGMA * 8;
  const uint32_t j = (lane % TPS) * 16, sw = w * SPW + lane / TPS;
  int64_t *fb = a.f + (int64_t)blockIdx.x * a.pitch * SIGMA + (lane % TPS) * 2;
#pragma unroll 1
  for (int32_t l = team; l < a.L; l += teams) {
    if (!__all_sync(0xffffffffu, lv_wait(sh.headed + (l & kStageMask), l / kLvStages, sh, a))) return;
    const uint32_t ds = desc_of(sh, l);
    const uint4 m = s_ld128(ds), m2 = s_ld128(ds + 16);
    const uint32_t nseg = m.y & 0xFFFF, recs = sh.ring + m.x, dur = sh.ring + m.z + j;
    uint32_t n = ALL ? nseg : m2.x & 0xFFFF;
    if (DBG && !desc_ok<SIGMA>(a, m, m2)) {
      lv_bad(sh, a);
      n = 0;
    }
#pragma unroll 1
    for (uint32_t x = sw; x < n; x += (uint32_t)nw * SPW) {
      uint32_t k = x, len, h;
      uint64_t keep = ~0ull;
      if (ALL) {
        h = s_ld32(recs + 4 * k);
        len = (h >> 16) & 0xFF;
      } else {  // a segment with kept rows: {segment | last kept row + 1 << 16, 0, mask of the kept rows}
        const uint4 e = s_ld128(sh.ring + m2.w + 16 * x);
        k = e.x & 0xFFFF;
        len = e.x >> 16;
        keep = (uint64_t)e.z | ((uint64_t)e.w << 32);
        if (DBG && !in_range(k, nseg)) {
          lv_bad(sh, a);
          continue;
        }
        h = s_ld32(recs + 4 * k);
      }
      uint64_t mask = 0;
      uint32_t q = 0;
      if (a.cdur && (h >> 24)) {
        const uint4 c = s_ld128(recs + ((4 * nseg + 15) & ~15u) + 16 * k);
        mask = (uint64_t)c.x | ((uint64_t)c.y << 32);
        q = sh.ring + m2.z + j + c.z * kRow;
        if (DBG && !masked_row_ok(c.z, mask, m2.x >> 16)) {
          lv_bad(sh, a);
          continue;
        }
      }
      if (DBG && !range_ok(h & 0xFFFF, (int64_t)(h & 0xFFFF) + len, m.y >> 16)) {
        lv_bad(sh, a);
        continue;
      }
      int64_t f[2];
      s_load<2>(sh.ring + m.w + j + k * kRow, f);
      const uint32_t p = dur + (h & 0xFFFF) * kRow;
      int64_t *g = fb + (int64_t)(m2.y + (h & 0xFFFF)) * SIGMA;
      uint32_t t = 0;
      if (ALL && !mask) {
        uint32_t p1 = p;
#pragma unroll 1
        for (; t + 4 <= len; t += 4, p1 += 4 * kRow, g += 4 * SIGMA) {
          int64_t d[4][2];
#pragma unroll
          for (int u = 0; u < 4; ++u) s_load<2>(p1 + u * kRow, d[u]);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            f[0] += d[u][0];
            f[1] += d[u][1];
            g_store<2>(g + u * SIGMA, f);
          }
        }
      }
#pragma unroll 1
      for (; t < len; t += 4) {
        int64_t d[4][2];
        load_rows<SIGMA, 4>(d, p, t, len, q, mask);
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
          f[0] += d[u][0];
          f[1] += d[u][1];
          if (t + u < len && (ALL || (keep >> u & 1))) g_store<2>(g + u * SIGMA, f);
        }
        g += 4 * SIGMA;
        keep >>= 4;
      }
    }
    __syncwarp();
    if (lane == 0) {
      asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(sh.out + 4 * (l & kStageMask)) : "memory");
      mbar_arrive(&sh.stored[l & kStageMask]);
    }
  }
}

// Row order, over running sums.
template <int SIGMA, bool ALL, bool DBG>
__device__ void store_role(const LevelArgs &a, const Shared &sh, int team, int teams, int w, int nw, int lane) {
  constexpr int LV = SIGMA >= 2 ? 2 : 1, VPR = SIGMA / LV;  // vectors per row
  constexpr uint32_t kRow = SIGMA * 8;
  int64_t *fb = a.f + (int64_t)blockIdx.x * a.pitch * SIGMA;
#pragma unroll 1
  for (int32_t l = team; l < a.L; l += teams) {
    if (!__all_sync(0xffffffffu, lv_wait(sh.headed + (l & kStageMask), l / kLvStages, sh, a))) return;
    const uint32_t ds = desc_of(sh, l);
    const uint4 m = s_ld128(ds), m2 = s_ld128(ds + 16);
    const uint32_t counts = m.y, row0 = m2.y, map = sh.ring + m2.w, start = sh.ring + m.w, dur = sh.ring + m.z;
    uint32_t n = (ALL ? counts >> 16 : m2.x & 0xFFFF) * VPR;  // vectors
    if (DBG && !desc_ok<SIGMA>(a, m, m2)) {
      lv_bad(sh, a);
      n = 0;
    }
    int64_t *fl = fb + (int64_t)row0 * SIGMA;
    // vector x: its row of the level and its segment; the loads of 4 vectors are in flight together
#pragma unroll 1
    for (uint32_t x0 = (uint32_t)w * 32 + lane; x0 < n; x0 += (uint32_t)nw * 128) {
      uint32_t row[4], seg[4];
      int64_t d[4][LV], s[4][LV];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t x = x0 + u * nw * 32;
        if (x < n) {
          if (ALL) {
            row[u] = x / VPR;
            seg[u] = s_ld16(map + 2 * row[u]);
          } else {
            const uint32_t e = s_ld32(map + 4 * (x / VPR));
            row[u] = e & 0xFFFF;
            seg[u] = e >> 16;
          }
          if (DBG && !(in_range(row[u], counts >> 16) && in_range(seg[u], counts & 0xFFFF))) {
            lv_bad(sh, a);
            n = 0;  // (row and segment 0 need not exist)
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t x = x0 + u * nw * 32, c = (x % VPR) * (LV * 8);
        if (x < n) {
          s_load<LV>(dur + row[u] * kRow + c, d[u]);
          s_load<LV>(start + seg[u] * kRow + c, s[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t x = x0 + u * nw * 32;
        if (x < n) {
#pragma unroll
          for (int i = 0; i < LV; ++i) d[u][i] += s[u][i];
          g_store<LV>(fl + (int64_t)row[u] * SIGMA + (x % VPR) * LV, d[u]);
        }
      }
    }
    __syncwarp();
    if (lane == 0) {
      asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(sh.out + 4 * (l & kStageMask)) : "memory");
      mbar_arrive(&sh.stored[l & kStageMask]);
    }
  }
}

template <int SIGMA, bool ALL, bool DBG>
__global__ void __launch_bounds__(kLvMaxWarps * 32, 1) compose_levels_kernel(LevelArgs a) {
  extern __shared__ __align__(16) unsigned char sbuf[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  Shared sh;
  int64_t *mk_s = reinterpret_cast<int64_t *>(sbuf);  // [16]
  sh.abort = reinterpret_cast<volatile int32_t *>(sbuf + 128);
  sh.full = reinterpret_cast<uint64_t *>(sbuf + 144);
  sh.summed = sh.full + kLvStages;
  sh.headed = sh.summed + kLvStages;
  sh.stored = sh.headed + kLvStages;
  sh.heads = sh.stored + kLvStages;
  sh.counts = smem_u32(sh.heads + kLvStages / kLvGroup);
  sh.out = sh.counts + kLvStages * 4;
  sh.chunk = sh.out + kLvStages * 4;
  sh.base = smem_u32(sbuf);
  sh.prog = sh.base + a.prog_at;
  sh.ring = sh.base + a.ring_at;
  if (tid < 16) mk_s[tid] = 0;
  if (tid < 2 * kLvStages) asm volatile("st.shared.u32 [%0], 0;" ::"r"(sh.counts + 4 * tid) : "memory");
  if (tid < SIGMA) reinterpret_cast<int64_t *>(sbuf + kLvFixedBytes)[tid] = 0;  // slot 0: no input
  if (tid == 0) {
    *sh.abort = 0;
    for (int b = 0; b < kLvStages; ++b) {
      mbar_init(&sh.full[b], 1);  // the copy warp's arrive.expect_tx
      mbar_init(&sh.summed[b], a.sum_team);
      mbar_init(&sh.headed[b], 1);
      mbar_init(&sh.stored[b], a.store_team);
    }
    for (int b = 0; b < kLvStages / kLvGroup; ++b) mbar_init(&sh.heads[b], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  fence_async();
  __syncthreads();
  const int nh = a.head_warps, ns = a.sum_warps, nst = a.store_warps;
  if (warp < nh) {
    head_role<SIGMA, DBG>(a, sh, tid, nh * 32, mk_s);
  } else if (warp < nh + ns) {
    const int w = warp - nh;
    sum_role<SIGMA, DBG>(a, sh, w / a.sum_team, ns / a.sum_team, w % a.sum_team, a.sum_team, lane);
  } else if (warp < nh + ns + nst) {
    const int w = warp - nh - ns;
    if constexpr (level_walks(SIGMA))
      walk_role<SIGMA, ALL, DBG>(a, sh, w / a.store_team, nst / a.store_team, w % a.store_team, a.store_team, lane);
    else
      store_role<SIGMA, ALL, DBG>(a, sh, w / a.store_team, nst / a.store_team, w % a.store_team, a.store_team, lane);
  } else if (warp == nh + ns + nst) {
    head_copy_role<DBG>(a, sh, lane);
  } else {
    copy_role<SIGMA, ALL, DBG>(a, sh, warp - nh - ns - nst - 1, lane);
  }
  __syncthreads();
  const int32_t s = blockIdx.x * SIGMA + tid;
  if (tid < SIGMA && s < a.S) a.makespan[s] = mk_s[tid];
}

template <int SIGMA>
cudaError_t launch_levels_t(const LevelArgs &a, cudaStream_t st) {
  // debug bounds runs the checking variant, which stores every finish
  auto k = a.dbg ? compose_levels_kernel<SIGMA, true, true>
                 : a.store_all ? compose_levels_kernel<SIGMA, true, false> : compose_levels_kernel<SIGMA, false, false>;
  const size_t smem = a.smem_bytes;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((a.S + SIGMA - 1) / SIGMA);
  k<<<grid, (a.head_warps + a.sum_warps + a.store_warps + 1 + kLvCopyWarps) * 32, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_compose_levels(const LevelArgs &a, int sigma, cudaStream_t st) {
  if (a.S == 0) return cudaSuccess;
  switch (sigma) {
    case 1: return launch_levels_t<1>(a, st);
    case 2: return launch_levels_t<2>(a, st);
    case 4: return launch_levels_t<4>(a, st);
    case 8: return launch_levels_t<8>(a, st);
    case 16: return launch_levels_t<16>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace echo
