// echo_kernels.cu -- sm_103a kernels of the CC estimator, the validator and the
// readbacks.  All floating point that decides an integer is written with explicit
// round-to-nearest intrinsics (no contraction), so results do not depend on -fmad.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <functional>
#include <mutex>
#include <vector>

#include "echo.h"
#include "echo_internal.h"

namespace echo {

namespace {

constexpr int kAR = 0, kAG = 1, kSR = 3;  // reduce-scatter (2) takes the generic ring path
constexpr int kRing = 0, kTree = 1;

// ceil(a / b), a >= 0, b > 0.  Quotients of the estimator (chunk rounds) are small, and a
// 64-bit division takes about 100 instructions: an estimate in fp32 is off by at most
// q * 2^-21 + 1 < 2 below 2^20, which the remainder puts right.  (b is a product and may
// have wrapped below 0, like a sum n: both take the division.)
__device__ __forceinline__ int64_t cdiv64(int64_t a, int64_t b) {
  const int64_t n = a + b - 1;
  const float q0 = __fdividef((float)n, (float)b);
  if (!(q0 < 1048576.0f) || n < 0 || (uint64_t)b >= (1ull << 40)) return n / b;
  int32_t q = (int32_t)q0;
  int64_t r = n - (int64_t)q * b;
  if (r < 0) { --q; r += b; }
  if (r < 0) { --q; r += b; }
  if (r >= b) { ++q; r -= b; }
  if (r >= b) ++q;
  return q;
}

__device__ __forceinline__ int64_t chunk_for(int64_t nbytes, const ChunkTable &t) {
  for (int i = 0; i < t.n; ++i)
    if (nbytes <= t.max_bytes[i]) return t.chunk[i];
  return t.chunk[t.n - 1];
}

// x as a double, 0 <= x, rounded to nearest even: below 2^53 the bits are put together in
// integers, as a conversion occupies the fp64 pipe (527 G operations/s on this part, a
// seventieth of its integer rate) like an addition.
__device__ __forceinline__ double to_double(int64_t x) {
  if ((uint64_t)x >> 53) return (double)x;
  const int up = __clzll(x) - 11;  // puts the highest bit at bit 52
  const uint64_t bits = (((uint64_t)x << (up & 63)) & ((1ull << 52) - 1)) | ((uint64_t)(1075 - up) << 52);
  return __longlong_as_double(x ? (int64_t)bits : 0);
}
// The product of two such doubles: exact in integers when it stays below 2^53.
__device__ __forceinline__ double product(int64_t x, int64_t y) {
  if (((uint64_t)x | (uint64_t)y) >> 31 || (x * y) >> 53) return __dmul_rn(to_double(x), to_double(y));
  return to_double(x * y);
}

// Eqs. 2-4 (Sec. 5.3): eta chunk rounds, eta*(N-1) ring steps (twice that for
// all-reduce), each L + p/B with p = S/(N*eta); inter-node link once M > 1.  Send/recv takes
// the same operations: eta chunk transfers of S/eta over the pair's link.  One code path
// for all of them, so that a warp of mixed queries runs it once.
__device__ __forceinline__ double linear_ns(int type, int64_t S, int N, int M, double alpha, double Ba, double La,
                                            double Be, double Le, double delta, int64_t C) {
  const bool pair = type == kSR;
  int64_t eta = cdiv64(S, pair ? C : (int64_t)N * C);
  if (eta < 1) eta = 1;
  const double size = to_double(S);
  const double p = __ddiv_rn(size, pair ? to_double(eta) : product(N, eta));
  const double L = M > 1 ? Le : La;
  const double B = M > 1 ? Be : Ba;
  const double t = __dadd_rn(L, __ddiv_rn(p, B));
  const int64_t steps = pair ? eta : (type == kAR ? 2 : 1) * eta * (int64_t)(N - 1);
  const double T = __dadd_rn(alpha, __dmul_rn(to_double(steps), t));
  return type == kAG || pair ? T : __dadd_rn(T, __dmul_rn(delta, size));
}

// Eq. 5 (Sec. 5.3): tree all-reduce; eta chunks, K-1 intra-node hops (beta) and
// log2(M) inter-node levels (gamma) up and down.
__device__ __forceinline__ double tree_ns(int64_t S, int M, int K, double lg, double alpha, double Ba, double La,
                                          double Be, double Le, double delta, int64_t C) {
  int64_t eta = cdiv64(S, C);
  if (eta < 1) eta = 1;
  const double size = to_double(S);
  double pt = __ddiv_rn(size, to_double(eta));
  double beta = __dadd_rn(La, __ddiv_rn(pt, Ba));
  double gamma = M > 1 ? __dadd_rn(Le, __ddiv_rn(pt, Be)) : beta;
  double T = __dadd_rn(alpha, __dmul_rn(gamma, to_double(eta - 1)));
  T = __dadd_rn(T, __dmul_rn(__dmul_rn(2.0, beta), to_double(K - 1)));
  T = __dadd_rn(T, __dmul_rn(__dmul_rn(2.0, gamma), lg));
  T = __dadd_rn(T, __dmul_rn(delta, size));
  return T;
}

__device__ double cc_ns_of(int type, int algo, int64_t S, int N, int M, int K, double lg,
                           double alpha, double Ba, double La, double Be, double Le, double delta,
                           const ChunkTable &tbl) {
  if (N <= 1 || S <= 0) return 0.0;
  int64_t C = chunk_for(S, tbl);
  const bool ring = type != kAR || algo != kTree, tree = type == kAR && algo != kRing;
  const double r = ring ? linear_ns(type, S, N, M, alpha, Ba, La, Be, Le, delta, C) : 0.0;
  const double t = tree ? tree_ns(S, M, K, lg, alpha, Ba, La, Be, Le, delta, C) : 0.0;
  return !tree ? r : !ring || t < r ? t : r;
}

__device__ __forceinline__ void set_status(int32_t *status, int32_t code) {
  atomicCAS(status, 0, code);
}

// ---------------------------------------------------------------------------------
// B1: CC estimate over [signature x scenario]
// ---------------------------------------------------------------------------------
__global__ void cc_estimate_kernel(const CcSig *__restrict__ sig, int32_t G, ScenParams p, int32_t S,
                                   ChunkTable tbl, const int32_t *__restrict__ sig_count,
                                   double *__restrict__ cc_ns, int64_t *__restrict__ cc_dur,
                                   double *__restrict__ comm_sum, int32_t *status, int model, int ar_policy) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)G * S) return;
  int32_t g = (int32_t)(idx / S), s = (int32_t)(idx % S);
  CcSig q = sig[g];
  double T;
  if (model == 1) {
    // alpha-beta comparison model (Sec. 2.3): size over bandwidth plus latency on
    // the bottleneck link
    T = (q.N <= 1 || q.nbytes <= 0)
            ? 0.0
            : __dadd_rn(q.M > 1 ? p.late[s] : p.lata[s], __ddiv_rn((double)q.nbytes, q.M > 1 ? p.bwe[s] : p.bwa[s]));
  } else {
    const int algo = q.type == kAR && ar_policy > 0 ? ar_policy - 1 : q.algo;  // a policy for every all-reduce
    T = cc_ns_of(q.type, algo, q.nbytes, q.N, q.M, q.K, q.lg, p.alpha[s], p.bwa[s], p.lata[s], p.bwe[s],
                 p.late[s], p.delta[s], tbl);
  }
  int64_t d = 0;
  if (T >= 0.0 && T < 2305843009213693952.0) {  // 2^61
    d = __double2ll_rn(T);
  } else {
    set_status(status, kDevCcOverflow);
  }
  cc_ns[idx] = T;
  cc_dur[idx] = d;
  atomicAdd(&comm_sum[s], (double)d * (double)sig_count[g]);
}

// every comm node takes its signature's duration row
__global__ void cc_scatter_kernel(const int32_t *__restrict__ comm_node, const int32_t *__restrict__ comm_sig,
                                  int64_t n_comm, const int64_t *__restrict__ cc_dur, int32_t S, MatLayout lay,
                                  int64_t *__restrict__ dur) {
  int64_t total = n_comm * S;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t c = idx / S;
    int32_t s = (int32_t)(idx - c * S);
    dur[lay.at(comm_node[c], s)] = cc_dur[(int64_t)comm_sig[c] * S + s];
  }
}

// The link parameters and slowdown factors of a batch, read where the caller has them:
// blockIdx.y is the array.  Seven copies of a few KB took 2 to 9 us each.
struct HostParams {
  const double *link[6], *slowdown;
};
__global__ void load_params_kernel(HostParams h, int32_t S, int64_t n_sf, double *__restrict__ prm,
                                   double *__restrict__ sf) {
  const int k = blockIdx.y;
  const double *src = k < 6 ? h.link[k] : h.slowdown;
  double *dst = k < 6 ? prm + (int64_t)k * S : sf;
  const int64_t n = k < 6 ? S : n_sf;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) dst[i] = src[i];
}

// A block's queries.  Every thread takes one as far as it is linear (send/recv and rings),
// then the trees (a sixth of a mixed sweep) are gathered, so that two warps and not eight
// run their code.  What bounds it is the fp64 pipe (divisions run at 73 G/s on this part):
// two or three divisions a query.  With a branch per form, every warp of a mixed sweep ran
// them all, some twelve divisions (a call with 10^6 queries on the device: 297 us, now 105;
// with the fields loaded where they are used, one after the other, 205).
// A query's inputs are read before its own result is written, and by no other thread
// after that, so the output may be one of the input arrays.
constexpr int kQueryThreads = 256;
struct QueryShared {
  int32_t n;                    // trees
  uint16_t who[kQueryThreads];  // their threads
  double ring[kQueryThreads];   // by thread: a ring's time that a tree's is to be compared with
};
struct Queries {
  const uint8_t *type, *algo;
  const int64_t *nbytes;
  const int32_t *N, *M;
  const double *lg;  // log2(M): by query, or by M
  bool lg_by_m;
  ScenParams p;
};
__device__ __forceinline__ void query_block(int64_t i, bool mine, const Queries &q, const ChunkTable &tbl, double *out,
                                            QueryShared &sh) {
  if (threadIdx.x == 0) sh.n = 0;
  __syncthreads();
  if (mine) {
    // (all fields are asked for before the first is looked at)
    const int type = q.type[i], algo = q.algo[i], N = q.N[i], M = q.M[i];
    const int64_t S = q.nbytes[i];
    const double alpha = q.p.alpha[i], bwa = q.p.bwa[i], lata = q.p.lata[i], bwe = q.p.bwe[i], late = q.p.late[i],
                 delta = q.p.delta[i];
    const bool some = N > 1 && S > 0;
    const bool tree = some && type == kAR && algo != kRing;
    double T = 0.0;
    if (some && !(tree && algo == kTree))
      T = linear_ns(type, S, N, M, alpha, bwa, lata, bwe, late, delta, chunk_for(S, tbl));
    if (tree) {
      sh.ring[threadIdx.x] = T;
      sh.who[atomicAdd(&sh.n, 1)] = (uint16_t)threadIdx.x;
    } else {
      out[i] = T;
    }
  }
  __syncthreads();
  if ((int)threadIdx.x < sh.n) {
    const int w = sh.who[threadIdx.x];
    const int64_t k = i - threadIdx.x + w;
    const int algo = q.algo[k], N = q.N[k], M = q.M[k];
    const int64_t S = q.nbytes[k];
    const double alpha = q.p.alpha[k], bwa = q.p.bwa[k], lata = q.p.lata[k], bwe = q.p.bwe[k], late = q.p.late[k],
                 delta = q.p.delta[k];
    const double t = tree_ns(S, M, (N + M - 1) / M, q.lg[q.lg_by_m ? M : k], alpha, bwa, lata, bwe, late, delta,
                             chunk_for(S, tbl));
    const double r = sh.ring[w];
    out[k] = algo == kTree || t < r ? t : r;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kQueryThreads) cc_query_kernel(int64_t n, Queries q, ChunkTable tbl, double *out) {
  __shared__ QueryShared sh;
  for (int64_t i0 = (int64_t)blockIdx.x * kQueryThreads; i0 < n; i0 += (int64_t)gridDim.x * kQueryThreads)
    query_block(i0 + threadIdx.x, i0 + threadIdx.x < n, q, tbl, out, sh);
}

// ---------------------------------------------------------------------------------
// load: caller-order rows -> internal order and blocked layout, with validation
// and per-scenario sums
// ---------------------------------------------------------------------------------
// What bounds it is memory.  Three things had to go for that (GPT-1.3B x 256, int64):
//   - an fp64 conversion and addition per element for the sums (140 us by the part's fp64
//     rate of 527 G/s): they are exact integers, in halves of 32 bits, until the end;
//   - an fp64 atomic per thread at the end (2 M of them): one per column and block;
//   - rows of 8 to 128 bytes stored one by one in narrow blocks: a tile of kTileOps rows x
//     kTileCols scenarios goes through shared memory, so that neighbouring rows of a block
//     are stored together; the next tile is loaded meanwhile (185 us without that, 97 with).
// 158 us before in blocks of 32 scenarios, 270 us in blocks of 2; 97 us in both (6.1 of the
// 6.8 TB/s of a copy).
constexpr int kTileLog = 5, kTileOps = 1 << kTileLog, kTileCols = 64;
template <typename T>
__global__ void __launch_bounds__(256, 6) permute_rows_kernel(const T *__restrict__ raw, const int32_t *__restrict__ int2ext,
                                                              const uint8_t *__restrict__ local, int64_t V, int32_t S,
                                                              MatLayout lay, int64_t *__restrict__ dur,
                                                              double *__restrict__ sums, int32_t *status) {
  constexpr int kGroups = 256 / kTileCols, kEach = kTileOps / kGroups;  // rows a thread loads of a tile
  __shared__ T tile[kTileOps][kTileCols + 1];
  // the caller's row, -1: a comm op's (0 until the collectives are estimated)
  __shared__ int32_t from[2][kTileOps];
  const int col = threadIdx.x % kTileCols, grp = threadIdx.x / kTileCols;
  const int32_t c0 = blockIdx.x * kTileCols, s = c0 + col;
  const int sl = lay.slog2, pl = kTileLog + sl;  // (log2 of) a row's scenarios in a block, the tile's elements in one
  uint64_t lo = 0;
  int64_t hi = 0;
  bool neg = false;
  // while a tile is stored, the next one's elements are on their way, and the places of
  // the one after that (two dependent loads)
  const int64_t step = (int64_t)gridDim.y * kTileOps, first = (int64_t)blockIdx.y * kTileOps;
  auto rows = [&](int64_t i0, int b) {
    if (threadIdx.x < kTileOps) {
      const int64_t i = i0 + threadIdx.x;
      from[b][threadIdx.x] = i < V && local[i] ? int2ext[i] : -1;
    }
  };
  T x[kEach];
  auto load = [&](int b) {
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      const int32_t e = from[b][k * kGroups + grp];
      x[k] = s < S && e >= 0 ? raw[(int64_t)e * S + s] : 0;
    }
  };
  rows(first, 0);
  __syncthreads();
  load(0);
  rows(first + step, 1);
  __syncthreads();
  int b = 1;
  for (int64_t i0 = first; i0 < V; i0 += step, b ^= 1) {
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      neg |= x[k] < 0;
      lo += (uint32_t)x[k];
      if (sizeof(T) == 8) hi += (int64_t)x[k] >> 32;
      tile[k * kGroups + grp][col] = x[k];
    }
    load(b);
    rows(i0 + 2 * step, b ^ 1);
    __syncthreads();
    const int n = (int)min((int64_t)kTileOps, V - i0);
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      const int e = k * 256 + threadIdx.x, blk = e >> pl, y = e & ((1 << pl) - 1);
      const int o = y >> sl, c = (blk << sl) + (y & ((1 << sl) - 1));
      if (o < n && c0 + c < S) dur[lay.at(i0 + o, c0 + c)] = (int64_t)tile[o][c];
    }
    __syncthreads();
  }
  if (neg) set_status(status, kDevNegativeDuration);
  // one atomic per column and block
  __shared__ uint64_t lo_s[256];
  __shared__ int64_t hi_s[256];
  lo_s[threadIdx.x] = lo;
  hi_s[threadIdx.x] = hi;
  __syncthreads();
  if (grp == 0 && s < S) {
    for (int k = kTileCols; k < 256; k += kTileCols) {
      lo += lo_s[k + col];
      hi += hi_s[k + col];
    }
    atomicAdd(&sums[s], (double)lo + (double)hi * 4294967296.0);
  }
}

// ---------------------------------------------------------------------------------
// readback: internal order and blocked layout -> caller order, [op][scenario]
// ---------------------------------------------------------------------------------
// start = finish - the duration the op had in the last composition: d, or for an
// overlap candidate its row of the compact cd when given
__global__ void readback_kernel(const int32_t *__restrict__ ext2int, int64_t op0, int64_t op1, int32_t s0,
                                int32_t s1, MatLayout lay, const int64_t *__restrict__ f,
                                const int64_t *__restrict__ d, const int32_t *__restrict__ cidx, MatLayout lay_c,
                                const int64_t *__restrict__ cd, int64_t *__restrict__ start,
                                int64_t *__restrict__ finish) {
  const int32_t Sr = s1 - s0;
  int64_t total = (op1 - op0) * Sr;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = idx / Sr;
    int32_t s = s0 + (int32_t)(idx - o * Sr);
    const int32_t i = ext2int[op0 + o];
    int64_t at = lay.at(i, s);
    int64_t fv = f[at];
    if (start) {
      const int32_t ci = cd ? cidx[i] : -1;
      start[idx] = fv - (ci >= 0 ? cd[lay_c.at(ci, s)] : d[at]);
    }
    if (finish) finish[idx] = fv;
  }
}

// The same for whole batches (32 scenarios and more) in narrow blocks, where a row of one
// block is only 8 to 128 bytes.  What bounds it is memory: a tile of kTileOps ops x
// kReadCols scenarios goes through shared memory, so that the loads take neighbouring rows
// of a block together (ops of a chain are neighbours in both orders) and the stores whole
// rows of the caller's; a tile is loaded while the one before it is stored.
constexpr int kReadCols = 32;
__global__ void __launch_bounds__(256, 4) readback_tile_kernel(
    const int32_t *__restrict__ ext2int, int64_t op0, int64_t op1, int32_t s0, int32_t s1, MatLayout lay,
    const int64_t *__restrict__ f, const int64_t *__restrict__ d, const int32_t *__restrict__ cidx, MatLayout lay_c,
    const int64_t *__restrict__ cd, int64_t *__restrict__ start, int64_t *__restrict__ finish) {
  constexpr int kEach = kTileOps * kReadCols / 256;
  // (rows padded by one element: a warp's column of them falls into different banks)
  __shared__ int64_t ft[kTileOps][kReadCols + 1], st[kTileOps][kReadCols + 1];
  __shared__ int32_t row[2][kTileOps], crow[2][kTileOps];
  const int32_t c0 = (s0 & ~(kReadCols - 1)) + blockIdx.y * kReadCols;  // first scenario of the tile
  const int sl = lay.slog2, pl = kTileLog + sl;  // (log2 of) a row's scenarios in a block, the tile's elements in one
  const int64_t step = (int64_t)gridDim.x * kTileOps, first = op0 + (int64_t)blockIdx.x * kTileOps;
  auto rows = [&](int64_t o0, int b) {
    if (threadIdx.x < kTileOps) {
      const int64_t o = o0 + threadIdx.x;
      const int32_t i = o < op1 ? ext2int[o] : -1;
      row[b][threadIdx.x] = i;
      crow[b][threadIdx.x] = cd && i >= 0 ? cidx[i] : -1;
    }
  };
  int64_t fv[kEach], dv[kEach];
  auto load = [&](int b) {
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      const int e = k * 256 + threadIdx.x, blk = e >> pl, y = e & ((1 << pl) - 1);
      const int o = y >> sl, s = c0 + (blk << sl) + (y & ((1 << sl) - 1));
      const int32_t i = row[b][o], ci = crow[b][o];
      fv[k] = dv[k] = 0;
      if (i >= 0 && s >= s0 && s < s1) {
        const int64_t at = lay.at(i, s);
        fv[k] = f[at];
        if (start) dv[k] = ci >= 0 ? cd[lay_c.at(ci, s)] : d[at];
      }
    }
  };
  rows(first, 0);
  __syncthreads();
  load(0);
  rows(first + step, 1);
  __syncthreads();
  const int64_t Sr = s1 - s0;
  int b = 1;
  for (int64_t o0 = first; o0 < op1; o0 += step, b ^= 1) {
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      const int e = k * 256 + threadIdx.x, blk = e >> pl, y = e & ((1 << pl) - 1);
      const int o = y >> sl, c = (blk << sl) + (y & ((1 << sl) - 1));
      ft[o][c] = fv[k];
      st[o][c] = fv[k] - dv[k];
    }
    load(b);
    rows(o0 + 2 * step, b ^ 1);
    __syncthreads();
    const int n = (int)min((int64_t)kTileOps, op1 - o0);
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      const int e = k * 256 + threadIdx.x, o = e / kReadCols, c = e % kReadCols, s = c0 + c;
      if (o < n && s >= s0 && s < s1) {
        const int64_t to = (o0 - op0 + o) * Sr + (s - s0);
        if (finish) finish[to] = ft[o][c];
        if (start) start[to] = st[o][c];
      }
    }
    __syncthreads();
  }
}

// The same when every op is asked for, of blocks of two scenarios and more, in columns of
// kRingMinCols scenarios and more.  What bounds it is memory, and how whole the pieces are
// that it is read and written in: tiles follow the internal order, so that a block's rows
// come in pieces of 256 bytes and more, and leave as up to 2 KB of a caller's row each.  A
// tile of both matrices comes into a ring in shared memory as it lies there (cp.async of 16
// bytes, two tiles ahead); a block's part is padded by one row, so that a row of the tile is
// read without bank conflicts.  Measured, all times of GPT-175B, tiles of 32 x 32 as above ->
// this (us): x 200 1563 -> 1335, x 250 1880 -> 1502 (6.4 TB/s in the kernel), x 600 (three
// columns of 200) 4180 -> 3999, x 1024 6795 -> 5802; columns of 176 (x 352) 2401 -> 2439,
// of 150 (x 300) 2296 -> 2441.
// Other tiles, x 250, kernel alone: 32 x 64 1787, 32 x 128 1514, 8 x 256 1695, 16 x 256 1380.
// Blocks of one scenario (8-byte copies: x 100 891 -> 927) and ranges of ops (in the caller's
// order a chain's few rows start and end inside a piece: x 250 1874 -> 1908) stay with the
// kernel above.
constexpr int kRingOps = 16, kRingCols = 256, kRingMinCols = 192, kRingStages = 3;
constexpr int kRingTile = (kRingOps + 1) * kRingCols;  // elements of a padded tile of one matrix
constexpr size_t kRingSmem = (size_t)kRingStages * 2 * kRingTile * sizeof(int64_t);
// (blockIdx.y: `width` scenarios, a multiple of the block, from scenario c0 on)
__global__ void __launch_bounds__(256) readback_all_kernel(const int32_t *__restrict__ int2ext, int64_t V, int32_t s0,
                                                           int32_t s_end, int32_t width, MatLayout lay, const int64_t *__restrict__ f,
                                                           const int64_t *__restrict__ d,
                                                           const int32_t *__restrict__ cidx, MatLayout lay_c,
                                                           const int64_t *__restrict__ cd, int64_t *__restrict__ start,
                                                           int64_t *__restrict__ finish) {
  constexpr int kCopies = kRingOps * kRingCols / 2 / 256, kEach = kRingOps * kRingCols / 256;
  extern __shared__ __align__(16) int64_t tile[];  // [kRingStages][f, d][blocks][kRingOps + 1][block's scenarios]
  __shared__ int32_t crow[4][kRingOps], to_row[4][kRingOps];  // candidate's row, caller's (-1: none)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sl = lay.slog2, ul = sl - 1;  // (log2 of) a row's elements and copies
  const int32_t c0 = (s0 >> sl << sl) + blockIdx.y * width, s1 = min(s_end, c0 + width);
  const int64_t step = (int64_t)gridDim.x * kRingOps, first = (int64_t)blockIdx.x * kRingOps;
  // this thread's copies of a tile: op (-1: none), place in the padded tile, scenario
  int32_t op[kCopies], at[kCopies], scen[kCopies];
#pragma unroll
  for (int k = 0; k < kCopies; ++k) {
    const int x = k * 256 + (int)threadIdx.x, blk = x / kRingOps >> ul, y = x & ((kRingOps << ul) - 1);
    op[k] = y >> ul;
    at[k] = (blk * (kRingOps + 1) << sl) + y * 2;
    scen[k] = c0 + (blk << sl) + (y & ((1 << ul) - 1)) * 2;
    if (scen[k] + 2 <= s0 || scen[k] >= s1) op[k] = -1;
  }
  // rows of tile t, by the first lanes of one warp
  auto in = [&](int64_t t) { return lane < kRingOps && first + t * step + lane < V; };
  auto cand = [&](int64_t t) { return cd && in(t) ? cidx[first + t * step + lane] : -1; };
  auto outer = [&](int64_t t) { return in(t) ? int2ext[first + t * step + lane] : -1; };
  auto put = [&](int64_t t, int32_t c, int32_t o) {
    if (lane < kRingOps) crow[t & 3][lane] = c, to_row[t & 3][lane] = o;
  };
  auto load = [&](int64_t t) {
    int64_t *const to = tile + (t % kRingStages) * 2 * kRingTile;
#pragma unroll
    for (int k = 0; k < kCopies; ++k) {
      const int64_t i = first + t * step + op[k];
      if (op[k] < 0 || i >= V) continue;
      const int32_t ci = crow[t & 3][op[k]];
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(to + at[k]);
      const int64_t from = lay.at(i, scen[k]);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(f + from) : "memory");
      if (start)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + kRingTile * 8),
                     "l"(ci >= 0 ? cd + lay_c.at(ci, scen[k]) : d + from)
                     : "memory");
    }
  };
  const int64_t tiles = first < V ? (V - first + step - 1) / step : 0;
  int32_t c3 = -1, o3 = -1;  // rows of the tile three ahead
  if (warp == 0) {
    for (int t = 0; t < 3; ++t) put(t, cand(t), outer(t));
    c3 = cand(3), o3 = outer(3);
  }
  __syncthreads();
  for (int t = 0; t < kRingStages - 1; ++t) {
    if (t < tiles) load(t);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int64_t Sr = s_end - s0;
  const int32_t col = threadIdx.x, s = c0 + col;  // this thread's scenario
  static_assert(kRingCols == 256, "a thread stores one column");
  const bool mine = s >= s0 && s < s1;
  const int from = ((col >> sl) * (kRingOps + 1) << sl) + (col & ((1 << sl) - 1));  // element (0, s) of a tile
#pragma unroll 1
  for (int64_t t = 0; t < tiles; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kRingStages - 2) : "memory");
    __syncthreads();  // tile t is here for all, and tile t - 1 has been read by all
    if (t + kRingStages - 1 < tiles) load(t + kRingStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (warp == 0) {
      put(t + 3, c3, o3);
      c3 = cand(t + 4), o3 = outer(t + 4);
    }
    const int64_t *const ft = tile + (t % kRingStages) * 2 * kRingTile + from, *const dt = ft + kRingTile;
#pragma unroll
    for (int o = 0; o < kEach; ++o) {
      const int32_t r = to_row[t & 3][o];
      if (r < 0 || !mine) continue;
      const int64_t fv = ft[o << sl], to = r * Sr + (s - s0);
      if (finish) finish[to] = fv;
      if (start) start[to] = fv - dt[o << sl];
    }
  }
}

// Full validator durations for the direct composer: the
// candidates' rows of the compact cd into dst (which holds the original durations).
__global__ void scatter_candidates_kernel(const int32_t *__restrict__ cand_node, int64_t n_cand, int32_t S,
                                          MatLayout lay, MatLayout lay_c, const int64_t *__restrict__ cd,
                                          int64_t *__restrict__ dst) {
  const int64_t total = n_cand * S;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = idx / S;
    const int32_t s = (int32_t)(idx - k * S);
    dst[lay.at(cand_node[k], s)] = cd[lay_c.at(k, s)];
  }
}

__global__ void read_cc_kernel(const int32_t *__restrict__ ext2int, int64_t op0, int64_t op1, int32_t S,
                               const int32_t *__restrict__ node_sig, const double *__restrict__ cc_ns,
                               double *__restrict__ out) {
  int64_t total = (op1 - op0) * S;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = idx / S;
    int32_t s = (int32_t)(idx - o * S);
    int32_t g = node_sig[ext2int[op0 + o]];
    out[idx] = g >= 0 ? cc_ns[(int64_t)g * S + s] : __longlong_as_double(0x7ff8000000000000LL);
  }
}

__global__ void read_ov_kernel(const int32_t *__restrict__ ext2int, int64_t op0, int64_t op1, int32_t S,
                               MatLayout lay, const uint8_t *__restrict__ ov, const uint8_t *__restrict__ cand,
                               uint8_t *__restrict__ out) {
  int64_t total = (op1 - op0) * S;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    int64_t o = idx / S;
    int32_t s = (int32_t)(idx - o * S);
    int64_t i = ext2int[op0 + o];
    out[idx] = (ov && cand[i]) ? ov[lay.at(i, s)] : 0;  // only the candidates are tested
  }
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 152 * 32) b = 152 * 32;
  return (int)b;
}

}  // namespace

cudaError_t launch_cc_estimate(const CcSig *sig, int32_t G, ScenParams p, int32_t S, const ChunkTable &tbl,
                               const int32_t *sig_count, double *cc_ns, int64_t *cc_dur, double *comm_sum,
                               int32_t *status, int model, int ar_policy, cudaStream_t st) {
  int64_t n = (int64_t)G * S;
  if (n == 0) return cudaSuccess;
  int threads = 256;
  int64_t blocks = (n + threads - 1) / threads;
  cc_estimate_kernel<<<(unsigned)blocks, threads, 0, st>>>(sig, G, p, S, tbl, sig_count, cc_ns, cc_dur,
                                                          comm_sum, status, model, ar_policy);
  return cudaGetLastError();
}

cudaError_t launch_cc_scatter(const int32_t *comm_node, const int32_t *comm_sig, int64_t n_comm,
                              const int64_t *cc_dur, int32_t S, MatLayout lay, int64_t *dur, cudaStream_t st) {
  if (n_comm == 0) return cudaSuccess;
  cc_scatter_kernel<<<grid_for(n_comm * S, 256), 256, 0, st>>>(comm_node, comm_sig, n_comm, cc_dur, S, lay, dur);
  return cudaGetLastError();
}

cudaError_t launch_cc_query(int64_t n, const uint8_t *type, const uint8_t *algo, const int64_t *nbytes,
                            const int32_t *N, const int32_t *M, const double *lg, bool lg_by_m, ScenParams p,
                            const ChunkTable &tbl, double *out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  cc_query_kernel<<<grid_for(n, kQueryThreads), kQueryThreads, 0, st>>>(n, Queries{type, algo, nbytes, N, M, lg, lg_by_m, p}, tbl, out);
  return cudaGetLastError();
}

cudaError_t launch_load_params(const double *const src[6], const double *slowdown, int32_t S, int32_t C, double *prm,
                               double *sf, cudaStream_t st) {
  const HostParams h{{src[0], src[1], src[2], src[3], src[4], src[5]}, slowdown};
  const dim3 grid((unsigned)std::min<int64_t>(((int64_t)std::max(1, C) * S + 255) / 256, 152), 7);
  load_params_kernel<<<grid, 256, 0, st>>>(h, S, (int64_t)C * S, prm, sf);
  return cudaGetLastError();
}

cudaError_t launch_permute_rows(const void *raw, int bits, const int32_t *int2ext, const uint8_t *local, int64_t V,
                                int32_t S, MatLayout lay, int64_t *dur, double *sums, int32_t *status,
                                cudaStream_t st) {
  if (V == 0 || S == 0) return cudaSuccess;
  // one wave of blocks: 6 of 256 threads on an SM
  const int64_t cols = (S + kTileCols - 1) / kTileCols, tiles = (V + kTileOps - 1) / kTileOps;
  const dim3 grid((unsigned)cols, (unsigned)std::min<int64_t>(tiles, std::max<int64_t>(1, 152 * 6 / cols)));
  if (bits == 32)
    permute_rows_kernel<int32_t><<<grid, 256, 0, st>>>(static_cast<const int32_t *>(raw), int2ext, local, V, S, lay, dur,
                                                       sums, status);
  else
    permute_rows_kernel<int64_t><<<grid, 256, 0, st>>>(static_cast<const int64_t *>(raw), int2ext, local, V, S, lay, dur,
                                                       sums, status);
  return cudaGetLastError();
}

// Are the rows of a replica and of its representative equal?  One stream over all rows;
// HBM bounds it, so a row is compared in the widest words that its length and start allow
// (16 bytes, else the durations' own), by a team of lanes with eight loads in flight each.
// 143491 pairs of 500 durations of 32 bits: 308 us element by element with a 64-bit
// division each, 61 us now.
__device__ __forceinline__ uint32_t differ(uint32_t a, uint32_t b) { return a ^ b; }
__device__ __forceinline__ uint32_t differ(uint64_t a, uint64_t b) { return a != b; }
__device__ __forceinline__ uint32_t differ(uint4 a, uint4 b) {
  return (a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w);
}
template <typename U>
__global__ void replica_check_kernel(const U *__restrict__ raw, const int2 *__restrict__ pairs, int64_t n_pairs,
                                     int32_t n, int32_t team_log2, int32_t *flag) {
  const int32_t team = 1 << team_log2, lane = threadIdx.x & (team - 1);
  uint32_t diff = 0;
  for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> team_log2; p < n_pairs;
       p += ((int64_t)gridDim.x * blockDim.x) >> team_log2) {
    const int2 pr = __ldg(pairs + p);
    const U *a = raw + (int64_t)pr.x * n, *b = raw + (int64_t)pr.y * n;
    for (int32_t i = lane; i < n; i += 4 * team) {
      U x[4], y[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k * team < n) x[k] = __ldg(a + i + k * team), y[k] = __ldg(b + i + k * team);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k * team < n) diff |= differ(x[k], y[k]);
    }
  }
  if (__any_sync(0xffffffffu, diff != 0) && (threadIdx.x & 31) == 0) *flag = 1;
}
template <typename U>
void replica_check_rows(const void *raw, const int32_t *pairs, int64_t n_pairs, int64_t row_bytes, int32_t *flag,
                        cudaStream_t st) {
  const int32_t n = (int32_t)(row_bytes / (int64_t)sizeof(U));
  int32_t team_log2 = 0;  // a lane takes four words of a row at a time
  while (team_log2 < 5 && (4 << team_log2) < n) ++team_log2;
  const int64_t blocks = std::min<int64_t>(((n_pairs << team_log2) + 255) / 256, 152 * 8);
  replica_check_kernel<U><<<(unsigned)blocks, 256, 0, st>>>(
      static_cast<const U *>(raw), reinterpret_cast<const int2 *>(pairs), n_pairs, n, team_log2, flag);
}

cudaError_t launch_replica_check(const void *raw, int bits, const int32_t *pairs, int64_t n_pairs, int32_t S,
                                 int32_t *flag, cudaStream_t st) {
  if (n_pairs == 0 || S == 0) return cudaSuccess;
  const int64_t row_bytes = (int64_t)S * (bits / 8);
  if (row_bytes % 16 == 0)
    replica_check_rows<uint4>(raw, pairs, n_pairs, row_bytes, flag, st);
  else if (bits == 64)
    replica_check_rows<uint64_t>(raw, pairs, n_pairs, row_bytes, flag, st);
  else
    replica_check_rows<uint32_t>(raw, pairs, n_pairs, row_bytes, flag, st);
  return cudaGetLastError();
}

cudaError_t launch_overlap(const OverlapArgs &a, cudaStream_t st) {
  const int64_t warps = (int64_t)a.n_ranks * ((a.S + (1 << a.lay.slog2) - 1) >> a.lay.slog2) * a.parts;
  if (a.S == 0 || warps == 0) return cudaSuccess;
  if (a.n_cq < 0 || a.n_cq > kMaxStreams || a.parts < 1 || a.lay.slog2 > 5) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((warps + kOvWarps - 1) / kOvWarps));
  const int tx = kOvWarps * 32;
  // the variants are compiled in four translation units (echo_overlap.cu)
  const bool prop = a.model == 1 && a.cd_next;
  if (a.lq_off)
    return prop ? launch_overlap_l1_p1(a, grid, tx, st) : launch_overlap_l1_p0(a, grid, tx, st);
  return prop ? launch_overlap_l0_p1(a, grid, tx, st) : launch_overlap_l0_p0(a, grid, tx, st);
}

cudaError_t launch_readback(const int32_t *ext2int, const int32_t *int2ext, int64_t V, int64_t op0, int64_t op1, int32_t s0, int32_t s1, MatLayout lay,
                            const int64_t *f, const int64_t *d, const int32_t *cidx, MatLayout lay_c,
                            const int64_t *cd, int64_t *start, int64_t *finish, cudaStream_t st) {
  int64_t n = (op1 - op0) * (s1 - s0);
  if (n <= 0) return cudaSuccess;
  constexpr int64_t kMaxCols = 65535;  // columns of the tiled kernels (the grid's second dimension)
  // columns of one width, so that the blocks have the same to do; one wave of blocks, one on an SM
  const int32_t sig = 1 << lay.slog2, S = s1 - (s0 & ~(sig - 1));
  const int64_t cols = (S + kRingCols - 1) / kRingCols;
  const int32_t width = (int32_t)((S + cols - 1) / cols + sig - 1) & ~(sig - 1);
  if (op0 == 0 && op1 == V && width >= kRingMinCols && cols <= kMaxCols && lay.slog2 >= 1 && lay.slog2 < 5) {
    const int64_t tiles = (V + kRingOps - 1) / kRingOps;
    const dim3 grid((unsigned)std::min<int64_t>(tiles, std::max<int64_t>(1, 152 / cols)), (unsigned)cols);
    const cudaError_t e = cudaFuncSetAttribute(readback_all_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRingSmem);
    if (e != cudaSuccess) return e;
    readback_all_kernel<<<grid, 256, kRingSmem, st>>>(int2ext, V, s0, s1, width, lay, f, d, cidx, lay_c, cd, start, finish);
    return cudaGetLastError();
  }
  // (about two million scenarios at most: with that many an op's row is long enough for any kernel)
  const int32_t first = s0 & ~(kReadCols - 1);
  const int64_t tile_cols = ((int64_t)s1 - first + kReadCols - 1) / kReadCols;
  if (s1 - s0 >= kReadCols && lay.slog2 < 5 && tile_cols <= kMaxCols) {
    const int64_t tiles = (op1 - op0 + kTileOps - 1) / kTileOps;
    // one wave of blocks: 4 of 256 threads on an SM
    const dim3 grid((unsigned)std::min<int64_t>(tiles, std::max<int64_t>(1, 152 * 4 / tile_cols)), (unsigned)tile_cols);
    readback_tile_kernel<<<grid, 256, 0, st>>>(ext2int, op0, op1, s0, s1, lay, f, d, cidx, lay_c, cd, start, finish);
    return cudaGetLastError();
  }
  readback_kernel<<<grid_for(n, 256), 256, 0, st>>>(ext2int, op0, op1, s0, s1, lay, f, d, cidx, lay_c, cd, start,
                                                    finish);
  return cudaGetLastError();
}

cudaError_t launch_scatter_candidates(const int32_t *cand_node, int64_t n_cand, int32_t S, MatLayout lay,
                                      MatLayout lay_c, const int64_t *cd, int64_t *dst, cudaStream_t st) {
  if (n_cand == 0 || S == 0) return cudaSuccess;
  scatter_candidates_kernel<<<grid_for(n_cand * S, 256), 256, 0, st>>>(cand_node, n_cand, S, lay, lay_c, cd, dst);
  return cudaGetLastError();
}

cudaError_t launch_read_cc(const int32_t *ext2int, int64_t op0, int64_t op1, int32_t S, const int32_t *node_sig,
                           const double *cc_ns, double *out, cudaStream_t st) {
  int64_t n = (op1 - op0) * S;
  if (n <= 0) return cudaSuccess;
  read_cc_kernel<<<grid_for(n, 256), 256, 0, st>>>(ext2int, op0, op1, S, node_sig, cc_ns, out);
  return cudaGetLastError();
}

cudaError_t launch_read_ov(const int32_t *ext2int, int64_t op0, int64_t op1, int32_t S, MatLayout lay,
                           const uint8_t *ov, const uint8_t *cand, uint8_t *out, cudaStream_t st) {
  int64_t n = (op1 - op0) * S;
  if (n <= 0) return cudaSuccess;
  read_ov_kernel<<<grid_for(n, 256), 256, 0, st>>>(ext2int, op0, op1, S, lay, ov, cand, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------
// fp64 rates of this device (measurement support): each thread keeps 8 independent
// chains of one operation (add, multiply or divide with round-to-nearest, as the
// CC estimator uses them), so the pipe, not the dependence latency, sets the rate.
// The result feeds a kernel in the sink so nothing is optimized away.
// ---------------------------------------------------------------------------------
constexpr int kFp64Chains = 8;
template <int OP>
__global__ void fp64_rate_kernel(int iters, double y, double *sink) {
  double x[kFp64Chains];
#pragma unroll
  for (int k = 0; k < kFp64Chains; ++k) x[k] = 1.0 + (threadIdx.x + k) * 1e-9;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int k = 0; k < kFp64Chains; ++k)
      x[k] = OP == 0 ? __dadd_rn(x[k], y) : OP == 1 ? __dmul_rn(x[k], y) : __ddiv_rn(x[k], y);
  }
  double t = 0.0;
#pragma unroll
  for (int k = 0; k < kFp64Chains; ++k) t = __dadd_rn(t, x[k]);
  if (t == 12345.0) sink[0] = t;  // never true for these inputs
}

}  // namespace echo

extern "C" int echo_measure_fp64(int device, double *rates) {
  using namespace echo;
  if (!rates) return ECHO_E_INVALID_ARG;
  int prev = 0;
  if (cudaGetDevice(&prev) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) return ECHO_E_CUDA;
  struct Restore {
    int dev;
    ~Restore() { cudaSetDevice(dev); }
  } restore{prev};
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  double *sink = nullptr;
  if (cudaMalloc(&sink, sizeof(double)) != cudaSuccess) return ECHO_E_OOM;
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  const int threads = 256, blocks = sms * 8;
  int rc = ECHO_OK;
  for (int op = 0; op < 3 && rc == ECHO_OK; ++op) {
    const int iters = op == 2 ? 256 : 4096;
    const double y = op == 1 ? 1.0000000001 : op == 2 ? 0.9999999999 : 1e-12;
    auto launch = [&]() {
      if (op == 0) fp64_rate_kernel<0><<<blocks, threads>>>(iters, y, sink);
      else if (op == 1) fp64_rate_kernel<1><<<blocks, threads>>>(iters, y, sink);
      else fp64_rate_kernel<2><<<blocks, threads>>>(iters, y, sink);
    };
    launch();  // warm-up
    float best = 0.f;
    for (int rep = 0; rep < 5; ++rep) {
      cudaEventRecord(a);
      launch();
      cudaEventRecord(b);
      if (cudaEventSynchronize(b) != cudaSuccess) {
        rc = ECHO_E_CUDA;
        break;
      }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, a, b);
      if (rep == 0 || ms < best) best = ms;
    }
    rates[op] = (double)blocks * threads * iters * kFp64Chains / (best * 1e-3);
  }
  if (cudaGetLastError() != cudaSuccess && rc == ECHO_OK) rc = ECHO_E_CUDA;
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(sink);
  return rc;
}

// ---------------------------------------------------------------------------------
// Allocation-free CC queries.
//
// Some callers cannot call cudaMalloc: a process whose device memory is owned by a
// framework's memory pool (a stray allocation would fail or fragment that pool), or
// one that runs under a fixed per-process memory budget.  echo_cc_query_noalloc
// serves them: the caller passes device arrays in and out, and the only other
// device memory the kernel touches is the file-scope array below, which every GPU
// that loads this library holds until the process exits.
//
// Layout of the array: bytes [0, 4) hold a status word (one bit per kind of bad
// query), cleared at the start of every call; from byte 256 on, log2(m) for m = 0..kNoallocMaxNodes, computed on
// the host with the same libm log2 the allocating path uses, so both paths give
// identical estimates.  Node counts above kNoallocMaxNodes are rejected.
// ---------------------------------------------------------------------------------
namespace echo {
namespace {
constexpr int32_t kNoallocMaxNodes = 65536;
constexpr size_t kNoallocLgOffset = 256;
constexpr size_t kNoallocScratchBytes = kNoallocLgOffset + sizeof(double) * (kNoallocMaxNodes + 1);
constexpr int kNoallocMaxDevices = 64;
// status bits: a batch may hold both kinds of bad query, so each sets its own bit
// and the host ranks them (a malformed query before an unsupported size)
enum : int32_t { kNoallocOk = 0, kNoallocTooManyNodes = 1, kNoallocBadQuery = 2 };
}  // namespace
}  // namespace echo

static __device__ __align__(256) unsigned char g_noalloc_scratch[echo::kNoallocScratchBytes];

namespace echo {
namespace {

struct NoallocDevice {
  std::once_flag once;
  unsigned char *ptr = nullptr;  // device address of g_noalloc_scratch on this device
  cudaError_t err = cudaSuccess;
};
NoallocDevice g_noalloc_devices[kNoallocMaxDevices];

// Once per device, with that device current: look up the array's device address
// (host code cannot use the symbol itself) and fill the log2 table.
void noalloc_setup(NoallocDevice &d) {
  void *p = nullptr;
  d.err = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (d.err != cudaSuccess) return;
  std::vector<double> lg(kNoallocMaxNodes + 1, 0.0);
  for (int32_t m = 1; m <= kNoallocMaxNodes; ++m) lg[m] = std::log2((double)m);
  unsigned char *base = static_cast<unsigned char *>(p);
  d.err = cudaMemcpy(base + kNoallocLgOffset, lg.data(), lg.size() * sizeof(double), cudaMemcpyHostToDevice);
  if (d.err != cudaSuccess) return;
  d.ptr = base;
}

// (by their bits: a comparison of doubles occupies the fp64 pipe)
__device__ __forceinline__ bool nonneg_finite(double x) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  return (u >> 52 & 0x7ff) != 0x7ff && (!(u >> 63) || !(u << 1));
}
__device__ __forceinline__ bool pos_finite(double x) {
  const uint64_t u = (uint64_t)__double_as_longlong(x);
  return (u >> 52) < 0x7ff && u != 0;
}

// Same estimate as cc_query_kernel; log2(M) comes from the table in the static
// array and each query is checked on the device, since its fields live there.
__global__ void __launch_bounds__(kQueryThreads) cc_query_noalloc_kernel(int64_t n, Queries q, ChunkTable tbl,
                                                                         int32_t *status, double *out) {
  __shared__ QueryShared sh;
  const ScenParams &p = q.p;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int64_t i0 = (int64_t)blockIdx.x * kQueryThreads; i0 < n; i0 += (int64_t)gridDim.x * kQueryThreads) {
    const int64_t i = i0 + threadIdx.x;
    bool mine = i < n;
    if (mine) {
      const int t = q.type[i], a = q.algo[i], n_r = q.N[i], m = q.M[i];
      const bool ok = (t <= kSR) & ((t != kAR) | (a <= 2)) & (q.nbytes[i] >= 0) & (n_r >= 1) & (m >= 1) & (m <= n_r) &
                      nonneg_finite(p.alpha[i]) & nonneg_finite(p.lata[i]) & nonneg_finite(p.late[i]) &
                      nonneg_finite(p.delta[i]) & pos_finite(p.bwa[i]) & pos_finite(p.bwe[i]);
      if (!ok || m > kNoallocMaxNodes) {
        out[i] = nan;
        atomicOr(status, ok ? kNoallocTooManyNodes : kNoallocBadQuery);
        mine = false;
      }
    }
    query_block(i, mine, q, tbl, out, sh);
  }
}

}  // namespace
}  // namespace echo

extern "C" int echo_cc_query_noalloc(const echo_cc_query_desc *q, double *out_ns, void *cuda_stream) {
  using namespace echo;
  if (!q || q->n < 0) return ECHO_E_INVALID_ARG;
  if (q->n == 0) return ECHO_OK;
  if (!out_ns || !q->cc_type || !q->cc_algo || !q->nbytes || !q->n_ranks || !q->n_nodes || !q->alpha_ns ||
      !q->bw_intra || !q->lat_intra || !q->bw_inter || !q->lat_inter || !q->delta)
    return ECHO_E_INVALID_ARG;
  // the chunk table is a few host values passed by value to the kernel
  ChunkTable tbl;
  std::memset(&tbl, 0, sizeof tbl);
  if (q->n_chunk == 0) {
    const int64_t mx[5] = {4LL << 20, 8LL << 20, 64LL << 20, 128LL << 20, INT64_MAX};
    const int64_t cb[5] = {18000, 36000, 72000, 144000, 288000};
    tbl.n = 5;
    for (int i = 0; i < 5; ++i) {
      tbl.max_bytes[i] = mx[i];
      tbl.chunk[i] = cb[i];
    }
  } else {
    if (q->n_chunk < 0 || q->n_chunk > kMaxChunk) return ECHO_E_UNSUPPORTED;
    if (!q->chunk_max_bytes || !q->chunk_bytes) return ECHO_E_INVALID_ARG;
    tbl.n = q->n_chunk;
    for (int i = 0; i < q->n_chunk; ++i) {
      if (q->chunk_bytes[i] <= 0 || (i > 0 && q->chunk_max_bytes[i] < q->chunk_max_bytes[i - 1]))
        return ECHO_E_INVALID_ARG;
      tbl.max_bytes[i] = q->chunk_max_bytes[i];
      tbl.chunk[i] = q->chunk_bytes[i];
    }
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return ECHO_E_CUDA;
  NoallocDevice &d = g_noalloc_devices[dev];
  std::call_once(d.once, noalloc_setup, std::ref(d));
  if (d.err != cudaSuccess || !d.ptr) return ECHO_E_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemsetAsync(d.ptr, 0, sizeof(int32_t), st) != cudaSuccess) return ECHO_E_CUDA;
  ScenParams p{q->alpha_ns, q->bw_intra, q->lat_intra, q->bw_inter, q->lat_inter, q->delta};
  const Queries dq{q->cc_type, q->cc_algo, q->nbytes, q->n_ranks, q->n_nodes,
                   reinterpret_cast<const double *>(d.ptr + kNoallocLgOffset), true, p};
  cc_query_noalloc_kernel<<<grid_for(q->n, kQueryThreads), kQueryThreads, 0, st>>>(
      q->n, dq, tbl, reinterpret_cast<int32_t *>(d.ptr), out_ns);
  if (cudaGetLastError() != cudaSuccess) return ECHO_E_CUDA;
  int32_t status = 0;
  if (cudaMemcpyAsync(&status, d.ptr, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return ECHO_E_CUDA;
  if (status & kNoallocBadQuery) return ECHO_E_INVALID_ARG;
  if (status & kNoallocTooManyNodes) return ECHO_E_UNSUPPORTED;
  return ECHO_OK;
}
