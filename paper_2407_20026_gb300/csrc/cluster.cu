// Batched FP32 CG with FP64 refinement, one thread-block cluster per system, or
// one team of CTAs over a whole, a half or a quarter of the chip.
//
// What bounds it: the latency of an iteration.  The two-kernel engine (pcg.cu)
// streams every system's K from HBM in every iteration and pays two launches'
// ramps and tails (16 to 23 us an iteration, however small the systems are).
// Here a cluster of C CTAs keeps one system for many iterations: its vectors
// live in the CTAs' shared memory, K in their tensor and shared memory as far
// as it fits and behind that in L2 (64 bytes a clock and SM, about 20 TB/s in
// all, three times HBM, while the systems in flight fit its 126 MB), and the
// CTAs meet at two cluster barriers an iteration (about 0.25 us each).
// Measured, 64 x 64 shells (25,350 DOF) to 1e-6, two-kernel engine -> here:
// one system 16.1 -> 6.5 us an iteration (208.8 -> 82.8 ms a solve; on 16 SMs),
// 48 systems 1.58 -> 0.61 us a system-iteration (945 -> 377 ms); two-level
// preconditioner, one 28.8 -> 14.2 us, 128 systems 403 -> 256 ms.
//
// Larger systems (and a few middle-sized ones together) take teams of 152, 76
// or 38 CTAs of a cooperative launch: more room for K on chip and more SMs to
// stream the rest, but z goes through global memory and the barriers too
// (team_sync: 4,000 to 6,000 clocks an iteration more than a cluster's).
// Measured, us an iteration, two-kernel engine -> team: 256 x 256 shell
// (396,294 DOF, K 85 MB, 57 MB of it streamed) 36 -> 12.5, 128 x 128 shell
// 28 -> 8.2, 100 x 100 grid shell 25 -> 7.6 (on a cluster of 16: 13.8).  The
// coarse correction needs a cluster: two-level systems do not take teams.
//
// The arithmetic is the two-kernel engine's, so every result is the same bits
// and the two engines can follow one another on a system at any step:
//   - a row is the fma chain over its blocks in column order, p = z + beta p;
//   - p^T q: the exact products of a 5-node group's 30 rows in the fixed tree
//     of a warp (double-float), one partial per group;
//   - r^T z, r^T r: six terms per node in order, then the tree over the tile's
//     30 nodes, one partial per tile;
//   - the scalars: the floats that the FP64 sums of the partials lead to (see
//     below), or those sums themselves, with the same trees and orders.
// Every CTA receives all partials (stores into its shared memory) and forms the
// scalars itself, so that control flow is uniform over the cluster.
//
// Data layout (cluster_pack_kernel, once per solve): K by tiles of 30 nodes,
// [block position][float4 0..8][lane]: lane n holds node n's whole block at that
// position as pairs of rows, (K[2a][c], K[2a+1][c]), so that a warp's loads are
// 512 contiguous bytes, one read of p serves six rows, and two rows share a
// packed FP32 multiply-add (each half rounds as a scalar one).  Rows of fewer
// blocks than the tile's longest are padded; the padding is read and not used.
// (A lane per row, three lanes a node with two rows each, issued three times
// the instructions and shared-memory reads: 128 ms for the one system above.)
// Each warp works on tiles of its own.
//
// Two things cost more here than elsewhere: a spilled register (each barrier's
// acquire drops L1, so that local memory is an L2 round trip: variants with
// 300 bytes of spills ran at half the speed, and the last 12 bytes cost 4 %), and code (a warp walks through
// the whole iteration once, so that instructions come from the outer levels of
// the instruction caches: loops are kept rolled, rare paths are functions).
#include <math.h>

#include <algorithm>
#include <climits>
#include <map>
#include <mutex>

#include "rounding.h"
#include "sso_internal.cuh"

namespace sso {
namespace {

constexpr int CL_POS_F4 = 9 * 32;  // float4 per block position of a tile
constexpr uint16_t kNoBlock = 0xffff;  // column slot past a row's end

// ---------------------------------------------------------------------------
// Cluster primitives.
__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cl_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Barrier over every thread of the cluster; orders shared (own and remote) and
// global memory accesses of the threads on both sides.
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_sync() {
  cl_arrive();
  cl_wait();
}
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, unsigned rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_st(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_st2(uint32_t addr, float x, float y) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// float -> double with integer operations for normal values and zero (the
// conversion instruction runs on the FP64 pipe: 64 clocks of a warp).
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned e = m >> 23;
  if (e >= 1u && e <= 254u) {
    const unsigned hi = (b & 0x80000000u) | ((m >> 3) + (896u << 20));
    return __hiloint2double((int)hi, (int)(m << 29));
  }
  if (m == 0u) return __hiloint2double((int)b, 0);
  return (double)x;
}
__device__ __forceinline__ double df_to_f64(DF x) { return f32_to_f64(x.hi) + f32_to_f64(x.lo); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
// Tensor memory as a store of K: each warp reads the 32 TMEM lanes of its
// quadrant (warp % 4), one lane per thread, 36 columns a position.
__device__ __forceinline__ void tm_alloc(uint32_t* out, int cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_addr(out)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tm_free(uint32_t base, int cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tm_st(uint32_t a, ulonglong2 v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a),
               "r"((uint32_t)v.x), "r"((uint32_t)(v.x >> 32)), "r"((uint32_t)v.y),
               "r"((uint32_t)(v.y >> 32))
               : "memory");
}
__device__ __forceinline__ void tm_ld36(uint32_t a, uint32_t (&r)[36]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
      "%30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(a)
      : "memory");
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35])
               : "r"(a + 32)
               : "memory");
}
__device__ __forceinline__ void tm_ld24(uint32_t a, uint32_t (&r)[24]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(a)
      : "memory");
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23])
      : "r"(a + 16)
      : "memory");
}
__device__ __forceinline__ void tm_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// Registers of a load may be read after the wait only: makes the compiler see
// them written here.
template <int N>
__device__ __forceinline__ void tm_loaded(uint32_t (&r)[N]) {
  static_assert(N % 12 == 0, "");
#pragma unroll
  for (int i = 0; i < N; i += 12)
    asm volatile(""
                 : "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), "+r"(r[i + 4]),
                   "+r"(r[i + 5]), "+r"(r[i + 6]), "+r"(r[i + 7]), "+r"(r[i + 8]),
                   "+r"(r[i + 9]), "+r"(r[i + 10]), "+r"(r[i + 11]));
}
__device__ __forceinline__ void tm_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// One node's block at a position: rows 2a and 2a + 1, columns c as the pair
// 6a + c (registers 2 (6a + c) and the next).
struct KPos {
  uint32_t r[36];
};
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// acc += K p for the node's six rows, columns in order
__device__ __forceinline__ void fma_pos(const KPos& k, const float* p,
                                        unsigned long long (&acc)[3]) {
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const unsigned long long pp = pack2(p[c], p[c]);
#pragma unroll
    for (int a = 0; a < 3; ++a)
      acc[a] = fma2(pack2(__uint_as_float(k.r[2 * (6 * a + c)]),
                          __uint_as_float(k.r[2 * (6 * a + c) + 1])),
                    pp, acc[a]);
  }
}

// A partial of a CG sum, or several, on an integer grid (below).
struct Fix {
  long long s;    // on the grid
  unsigned a;     // magnitude >> 38, rounded up
  unsigned bad;   // not finite, or 2 times the previous sum and more
};
// A positive value (h + l) 2^e, h in [1, 2), to about 2^-47.
struct Apx {
  float h, l;
  int e;
};
// What every thread of the CTA shares.  The pointers are for the rare paths
// (functions of their own, so that the iteration keeps its registers).
struct ClShared {
  SysScalars sc;       // parity, iters and inner of a CG iteration: in registers
  SysDesc sys;         // (a barrier's acquire drops L1: global copies would be L2 round trips)
  int n_done;          // 1 until the scalar updates report the system finished
  int lo, hi;          // node window of the CTA's columns
  int wlo[16], whi[16];  // the windows of every CTA of the cluster
  uint32_t tmem;       // base of the CTA's tensor memory
  int tm_m;            // the preconditioner's columns in a warp's share
  float2* gA;          // this CTA's partials as double-floats: p^T q per 5-node group,
  float4* tB;          // (r^T z, r^T r) per tile, two iterations
  Fix *fixA, *fixB, *fixR, *fixC;  // partials on the grids, of every CTA
  float *yS, *wS;      // two-level: y and w, two iterations
  const int* aptr;     // members of this CTA's aggregates
  const float4* member;
  const float4* rfw;   // offsets of the window's nodes
  const float4* Ms;    // preconditioner
  int T0, nt, n_ow, n_mine;
  double rz_known, thr;
  float beta;          // warps 0 and 1 to the others: beta, whether it and the
  int ok, rr_ok, end;  // comparison are certain, the end of the sweep
  int e_rr;
  Apx rz;
  double ex_pq, ex_rz, ex_rr;  // exact_sums
  double red[2 * CL_MAX_VWARPS];
  // teams without a cluster: the next barrier's set of words, whether a barrier
  // gave up, the words and their last values, the warps' sums and the team's
  unsigned epoch;
  int lost, team, copy;
  unsigned long long *slots, before[2][6];
  int* flags;
  unsigned long long words[16][6];
  Fix tot[2];
};

// finite / positive and finite, by the bits (FP64 compares cost 64 clocks)
__device__ __forceinline__ bool f64_finite(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ bool f64_positive(double x) {
  return __double_as_longlong(x) > 0 && f64_finite(x);
}

// ---------------------------------------------------------------------------
// The CG scalars without FP64.  alpha = r^T z / p^T q and beta enter the
// vectors as floats, and the sweep's end is one comparison, so the FP64 sums
// themselves are not needed in an iteration: only those roundings.  GB300
// issues one FP64 add of a warp per 64 clocks and a division takes 565; the
// chains of the FP64 sums took about a third of an iteration.  Each partial
// (a double-float) is instead rounded to a 64-bit integer on a grid of 2^-50
// of the previous iteration's sum; the integers are added exactly, in any
// order, and the quotient is formed to about 2^-41 with a bound on everything
// that separates it from the FP64 result: the grid (at most 1.25 2^-49 of the
// sum per partial: a high part is truncated only where the low part is less
// than a quarter of the grid; 2^-34.5 for p^T q's 18,432 partials of twelve
// chunks, 2^-37.1 for r^T z), the rounding of the FP64 chains (at most 24 2^-53
// of the sum of magnitudes, which may be 2^10 times the sum), the quotient's
// own: 0.93 2^-34 together.
// When a float's rounding (or the comparison) is the same anywhere within
// 2^-34 of the quotient, it is the two-kernel engine's; else, and where a sum
// leaves the grid's range, the exact sums are formed (exact_sums): each of an
// iteration's two quotients fails the test once in 512 times; with a sweep's
// first iterations, exact sums are formed once in 50 (a few hundred iterations a
// sweep) to 100 iterations.
constexpr int kGrid = 50;

__device__ __forceinline__ long long fix_part(float x, int k, unsigned& bad) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  const unsigned m = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
  const int sh = (int)(e ? e : 1u) - 150 + k;
  if (e == 0xffu || (sh > 27 && m)) bad = 1u;
  const long long q = sh >= 0 ? (long long)m << min(sh, 27) : (long long)(m >> min(-sh, 31));
  return (int)b < 0 ? -q : q;
}
__device__ __forceinline__ Fix to_fix(DF x, int k) {
  Fix f;
  f.bad = 0u;
  f.s = fix_part(x.hi, k, f.bad) + fix_part(x.lo, k, f.bad);
  f.a = (unsigned)((f.s < 0 ? -f.s : f.s) >> 38) + 1u;  // (at most 2^14: no sum overflows)
  return f;
}
// Sum over the warp, in every lane.
__device__ __forceinline__ Fix fix_warp_sum(Fix f) {
  const unsigned l0 = (unsigned)f.s & 0x3fffffu, l1 = (unsigned)(f.s >> 22) & 0x3fffffu;
  const long long s0 = __reduce_add_sync(0xffffffffu, l0), s1 = __reduce_add_sync(0xffffffffu, l1);
  const long long s2 = __reduce_add_sync(0xffffffffu, (int)(f.s >> 44));
  f.s = s0 + (s1 << 22) + (s2 << 44);
  f.a = __reduce_add_sync(0xffffffffu, f.a);
  f.bad = __any_sync(0xffffffffu, f.bad) ? 1u : 0u;
  return f;
}
__device__ __forceinline__ void push_fix(const Fix* slot, const Fix& f, unsigned rank) {
  asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(cl_map(smem_addr(slot), rank)),
               "l"(f.s), "l"((unsigned long long)f.bad << 32 | f.a)
               : "memory");
}
__device__ __noinline__ Fix fix_total(const Fix* slot, int n, int lane) {
  Fix t{0, 0u, 0u};
#pragma unroll 1
  for (int i = lane; i < n; i += 128) {
    ulonglong2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = i + 32 * u < n ? reinterpret_cast<const ulonglong2*>(slot)[i + 32 * u]
                            : make_ulonglong2(0ull, 0ull);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      t.s += (long long)v[u].x;
      t.a += (unsigned)v[u].y;
      t.bad |= (unsigned)(v[u].y >> 32);
    }
  }
  return fix_warp_sum(t);
}

// ---------------------------------------------------------------------------
// The barrier of a team of CTAs that is not a cluster (a cooperative launch's,
// all resident at once), with up to two sums over the warps of all CTAs: every
// warp calls team_add for each, then all call team_sync, which leaves them in
// sh.tot.  A sum goes as three words of integers, which add up in any order.
// Each CTA adds its six words, with 1 in the upper 16 bits, to each of
// CL_TEAM_COPIES lines, and polls one of these (a line that all SMs poll serves
// late adds late, and its readers unevenly).  Words are never reset: a word's
// growth since the last barrier of its set is the team's sum once it holds the
// team's count, so that a sum costs no round trip beyond the barrier's own.
// Two sets alternate, as a CTA may be one barrier ahead of a slow reader.
// data: global stores before are visible to the team after (else only the sums
// are).  Measured in a loop of barriers alone, 152 CTAs: one counter 2,000
// clocks (3,000 with data's fences), this 1,800 to 2,200; a slot per CTA that
// all poll 6,200, a mailbox per CTA that all store into 4,700, clusters of 4
// and their mailboxes 3,700.  256 x 256 shell, us an iteration: slots 21,
// mailboxes 15.9, this 13.6 (12.5 since K streams through registers).
// A CTA that waits for ten seconds gives up: it sets the error flag, and its
// later barriers do not wait.
constexpr int kTeamPolls = 1 << 25;  // of about 700 clocks: ten seconds (other kernels may go first)
constexpr int kTeamBias = 1 << 24;             // keeps the upper halves positive

// The warp's share of sum k (one lane).
__device__ __forceinline__ void team_add(ClShared& sh, int k, Fix f) {
  if (f.s >= (1ll << 55) || f.s <= -(1ll << 55)) f = Fix{0, f.a, 1u};
  unsigned long long* w = sh.words[threadIdx.x >> 5] + 3 * k;
  w[0] = (unsigned)f.s;
  w[1] = (unsigned long long)((f.s >> 32) + kTeamBias);
  w[2] = ((unsigned long long)f.bad << 34) | f.a;
}
__device__ __forceinline__ void fence_gpu() {
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
}
__device__ __noinline__ void team_sync(ClShared& sh, bool data) {
  const int lane = threadIdx.x & 31;
  __syncthreads();
  // (a team of one CTA, in FP64 alone and without sums, has met by now: 256 10 x
  // 10 grid shells 11.7 -> 10.3 ms)
  if (threadIdx.x < 32 && sh.team > 1) {
    const int W = blockDim.x >> 5, word = lane % 6, part = lane / 6;
    // (rows of warps that the CTA does not have are zero; no loops: the code
    // comes from outer caches, and a branch stalls where it goes on)
    const unsigned long long* mine = sh.words[part] + word;
    const unsigned long long v = mine[0] + mine[5 * 6] + mine[10 * 6] + (part ? 0ull : mine[15 * 6]);
    unsigned long long add = 1ull << 48;
#pragma unroll
    for (int p = 0; p < 5; ++p) add += __shfl_sync(0xffffffffu, v, word + 6 * p);
    const unsigned set = sh.epoch;
    unsigned long long* line = sh.slots + 16 * CL_TEAM_COPIES * set;
    if (data) fence_gpu();
    if (lane < 30) {
#pragma unroll
      for (int c = 0; c < CL_TEAM_COPIES; c += 5)
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(line + 16 * (c + part) +
                                                                      word),
                     "l"(add)
                     : "memory");
    }
    // the first six lanes' words (the others read them too)
    const unsigned long long* p = line + 16 * sh.copy + word;
    const unsigned long long before = sh.before[set][word];
    unsigned long long now;
    int polls = sh.lost ? 1 : kTeamPolls;
    do {
      asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(now) : "l"(p) : "memory");
    } while (!__all_sync(0xffffffffu, (int)((now - before) >> 48) == sh.team) && --polls);
    if (polls == 0 && lane == 0) {
      sh.lost = 1;
      atomicExch(sh.flags + 1, WAIT_TEAM);
    }
    if (data) fence_gpu();
    if (lane < 6) sh.before[set][word] = now;
    now = (now - before) & ((1ull << 48) - 1ull);
    const unsigned long long hi = __shfl_down_sync(0xffffffffu, now, 1);
    const unsigned long long ab = __shfl_down_sync(0xffffffffu, now, 2);
    if (lane == 0 || lane == 3)
      sh.tot[lane / 3] =
          Fix{(long long)now + (((long long)hi - (long long)sh.team * W * kTeamBias) << 32),
              (unsigned)ab, (unsigned)(ab >> 34)};
    if (lane == 0) sh.epoch = set ^ 1u;
  }
  __syncthreads();
}
// Barrier after global stores that the other CTAs read.
template <bool GRID>
__device__ __forceinline__ void all_sync(ClShared& sh) {
  if (GRID)
    team_sync(sh, true);
  else
    cl_sync();
}

__device__ __forceinline__ Apx apx_bits(unsigned long long m, int e) {  // m: bit 63 set
  return Apx{__uint_as_float(0x3f800000u | ((unsigned)(m >> 40) & 0x7fffffu)),
             (float)((unsigned)(m >> 16) & 0xffffffu) * 0x1p-47f, e};
}
__device__ __forceinline__ Apx apx_f64(double x) {  // positive and finite (a subnormal: e off,
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);  // and refused)
  return apx_bits((b << 11) | 0x8000000000000000ull, (int)(b >> 52) - 1023);
}
// The sum on the grid 2^-k; false where its bound does not hold.
__device__ __forceinline__ bool apx_fix(const Fix& f, int k, Apx& out) {
  if (f.bad || f.s < (1ll << (kGrid - 1)) || f.s >= (1ll << (kGrid + 3)) ||
      (long long)f.a > f.s >> 28)
    return false;
  const int lz = __clzll(f.s);
  out = apx_bits((unsigned long long)f.s << lz, 63 - lz - k);
  return true;
}
// The float nearest a / b; false where 2^-34 of it more or less would change it.  A
// reciprocal, its product, and one remainder step (to 2^-41); then Ziv's test.
__device__ __forceinline__ bool apx_quotient(const Apx& a, const Apx& b, float& out) {
  float rb;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rb) : "f"(b.h));
  const float q0 = __fmul_rn(a.h, rb);
  const float r = __fadd_rn(__fmaf_rn(-q0, b.h, a.h), __fmaf_rn(-q0, b.l, a.l));
  const float q1 = __fmul_rn(r, rb);
  const float f = __fadd_rn(q0, q1);
  const float rest = __fsub_rn(q1, __fsub_rn(f, q0));  // q0 + q1 - f, exactly
  const unsigned fb = __float_as_uint(f);
  const int e = a.e - b.e;
  out = __uint_as_float(fb + ((unsigned)e << 23));
  return e > -100 && e < 100 && a.e > -900 && b.e > -900 && (fb & 0x7fffffu) != 0u &&
         quotient_certain(f, rest);
}
// value <= thr for the sum f on the grid 2^-k; sets *clear where the bounds
// leave no doubt (the sum's own is 2^-33 of it).
__device__ __forceinline__ bool fix_le(const Fix& f, int k, double thr, bool& clear) {
  const long long b = __double_as_longlong(thr);
  const int sh = (int)(b >> 52) - 1075 + k;  // thr = m 2^(sh - k)
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (1ull << 52);
  clear = !f.bad && f.s >= (1ll << (kGrid - 1)) && f.s < (1ll << (kGrid + 3)) && b > (1ll << 52);
  if (sh > 10) return true;  // the threshold is above the grid's range
  const long long t = sh >= 0 ? (long long)(m << sh) : (long long)(m >> min(-sh, 63));
  const long long d = f.s - t;
  clear = clear && (d < 0 ? -d : d) > (f.s >> 30);
  return d <= 0;
}
__device__ __forceinline__ int f64_exp(double x) {
  return (int)((__double2hiint(x) >> 20) & 0x7ff) - 1023;
}

// Sum of the FP64 partials buf[0 .. n) as kernel A forms it: virtual warp v
// takes partials [256 v, 256 v + 256), eight contiguous ones per lane.
__device__ __noinline__ double vwarp_sum(const double* buf, int v, int n, int lane) {
  const int e0 = 256 * v + CHUNK_PER_THREAD * lane;
  double x[CHUNK_PER_THREAD];
#pragma unroll
  for (int u = 0; u < CHUNK_PER_THREAD; ++u) x[u] = e0 + u < n ? __ldcg(buf + e0 + u) : 0.0;
  double a = x[0];
#pragma unroll
  for (int u = 1; u < CHUNK_PER_THREAD; ++u) a += x[u];
  return warp_sum(a);
}

// Sum of the chunk sums x[0 .. n) by one thread: the tree of a warp.
__device__ __noinline__ double chunk_tree(const double* x, int n) {
  double t[16];
  static_assert(CL_MAX_CHUNKS <= 16, "");
#pragma unroll
  for (int k = 0; k < 16; ++k) t[k] = k < n ? x[k] : 0.0;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < o; ++k) t[k] += t[k + o];
  return t[0];
}

// One thread: the total of kernel A's partials from the virtual warps' sums
// (six per chunk, added in order; then the chunks).
__device__ __noinline__ double total_a(double* red, int n_vw, int n_chunks) {
  if (n_chunks == 1) {
    double s = red[0];
#pragma unroll 1
    for (int k = 1; k < n_vw; ++k) s += red[k];
    return s;
  }
  for (int c = 0; c < n_chunks; ++c) {
    double s = red[WARPS * c];
    for (int k = WARPS * c + 1; k < min(n_vw, WARPS * (c + 1)); ++k) s += red[k];
    red[c] = s;  // chunk c's own sums are read
  }
  return chunk_tree(red, n_chunks);
}
// One warp: the total of kernel B's partials (in lane 0).
__device__ __noinline__ double total_b(const double* buf, int n_tiles, int n_chunks, int lane,
                                          double* scratch) {
  if (n_chunks == 1) return vwarp_sum(buf, 0, n_tiles, lane);
  for (int c = 0; c < n_chunks; ++c) {
    const double s = vwarp_sum(buf, c, n_tiles, lane);
    if (lane == 0) scratch[c] = s;
  }
  __syncwarp();
  return lane == 0 ? chunk_tree(scratch, n_chunks) : 0.0;
}

// w^T y of the coarse solve as its kernel forms it (one thread).
__device__ __noinline__ double coarse_dot(const float* y, const float* w, int nc) {
  double wy = 0.0;
#pragma unroll 1
  for (int r0 = 0; r0 < nc; r0 += COARSE_ROWS_PER_BLOCK) {
    double part = 0.0;
#pragma unroll 1
    for (int r = r0; r < r0 + COARSE_ROWS_PER_BLOCK; r += 2) {
      double dot = 0.0;
      if (r < nc) dot += (double)y[r] * (double)w[r];
      if (r + 1 < nc) dot += (double)y[r + 1] * (double)w[r + 1];
      part += dot;
    }
    wy += part;
  }
  return wy;
}

// The FP64 sums themselves, by every CTA from all partials (through global
// memory): r^T z and r^T r of
// the iteration in buffer `par` (ex_rz, ex_rr) and, with_a, p^T q (ex_pq).
template <bool TWO, bool GRID>
__device__ __noinline__ void exact_sums(ClShared& sh, int par, bool with_a) {
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, W = blockDim.x >> 5;
  const int n_tiles = sh.sys.n_tiles, n_ow = sh.n_ow, n_chunks = sh.sys.n_chunks;
  const int n_vw = (n_ow + 255) / 256;
  // (a buffer of r^T z and r^T r per parity: the sums of the previous iteration
  // and of this one are formed one after the other, with no barrier between)
  double *bufA = sh.sys.part_a, *bufB = sh.sys.part_b + 2 * (size_t)n_tiles * par;
#pragma unroll 1
  for (int t = tid; t < sh.nt; t += blockDim.x) {
    const float4 v = sh.tB[par * sh.nt + t];
    bufB[sh.T0 + t] = df_to_f64(DF{v.x, v.y});
    bufB[n_tiles + sh.T0 + t] = df_to_f64(DF{v.z, v.w});
  }
  if (with_a) {
#pragma unroll 1
    for (int g = tid; g < WARPS * sh.nt; g += blockDim.x) {
      const float2 v = sh.gA[g];
      bufA[WARPS * sh.T0 + g] = df_to_f64(DF{v.x, v.y});
    }
  }
  all_sync<GRID>(sh);
  if (w < 2) {
    const double s = total_b(bufB + (size_t)w * n_tiles, n_tiles, n_chunks, lane,
                             sh.red + CL_MAX_VWARPS + CL_MAX_CHUNKS * w);
    if (lane == 0) {
      if (w == 0)
        sh.ex_rz = TWO ? s + coarse_dot(sh.yS + par * COARSE_MAX_N, sh.wS + par * COARSE_MAX_N,
                                        6 * sh.sys.n_agg)
                       : s;
      else
        sh.ex_rr = s;
    }
  }
  if (with_a) {
#pragma unroll 1
    for (int v = w; v < n_vw; v += W) {
      const double s = vwarp_sum(bufA, v, n_ow, lane);
      if (lane == 0) sh.red[v] = s;
    }
    __syncthreads();
    if (tid == 0) sh.ex_pq = total_a(sh.red, n_vw, n_chunks);
  }
  __syncthreads();
}

// z = z_b + P y at a node (the rule of coarse_prolong_kernel): o its offset
// from its aggregate's centroid, o.w the aggregate and the fixed DOFs (<< 8).
__device__ __forceinline__ void prolong_node(float4 o, const float* yS, const float zb[6],
                                             float z[6]) {
  const unsigned info = __float_as_uint(o.w);
  const float* y = yS + 6 * (info & 0xffu);
  const float t0 = y[0], t1 = y[1], t2 = y[2], w0 = y[3], w1 = y[4], w2 = y[5];
  const float c[6] = {fmaf(w1, o.z, fmaf(-w2, o.y, t0)), fmaf(w2, o.x, fmaf(-w0, o.z, t1)),
                      fmaf(w0, o.y, fmaf(-w1, o.x, t2)), w0, w1, w2};
#pragma unroll
  for (int d = 0; d < 6; ++d) z[d] = zb[d] + ((info >> (8 + d)) & 1u ? 0.f : c[d]);
}
__device__ __forceinline__ void ldcg6(const float* p, float v[6]) {
  const float2* q = reinterpret_cast<const float2*>(p);
  const float2 a = __ldcg(q), b = __ldcg(q + 1), c = __ldcg(q + 2);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y; v[4] = c.x; v[5] = c.y;
}
__device__ __forceinline__ void lds6(const float* p, float* v) {
  const float2* q = reinterpret_cast<const float2*>(p);
  const float2 a = q[0], b = q[1], c = q[2];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y; v[4] = c.x; v[5] = c.y;
}
__device__ __forceinline__ void sts6(float* p, const float v[6]) {
  float2* q = reinterpret_cast<float2*>(p);
  q[0] = make_float2(v[0], v[1]);
  q[1] = make_float2(v[2], v[3]);
  q[2] = make_float2(v[4], v[5]);
}

// K of every listed system in the layout above; one warp per tile.  Rows past
// the system's end and positions past a row's end are written as zeros.
__global__ void __launch_bounds__(128) cluster_pack_kernel(const SysDesc* __restrict__ sys,
                                                           const int* __restrict__ list) {
  const SysDesc& S = sys[list[blockIdx.y]];
  const int t = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= S.n_tiles) return;
  const int node = TILE * t + lane;
  const bool act = lane < TILE && node < S.n_nodes;
  const int j0 = act ? S.row_ptr[node] : 0, j1 = act ? S.row_ptr[node + 1] : 0;
  const int a = S.toff[t], m = S.toff[t + 1] - a;
  float4* out = reinterpret_cast<float4*>(S.klo) + (size_t)a * CL_POS_F4 + lane;
  for (int k = 0; k < m; ++k) {
    float v[36];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const float4 x = j0 + k < j1 ? __ldg(reinterpret_cast<const float4*>(
                                               S.K32 + (size_t)(j0 + k) * 36) + i)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
      v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {  // pairs 2i and 2i + 1: rows 2a, 2a + 1, columns c, c + 1
      const int r = 2 * (2 * i / 6), c = 2 * i % 6;
      out[(size_t)k * CL_POS_F4 + 32 * i] =
          make_float4(v[6 * r + c], v[6 * r + 6 + c], v[6 * r + c + 1], v[6 * r + 7 + c]);
    }
  }
}

// INIT and RESID, phase A: r64 = b - K64 x of the CTA's rows in FP64, the
// partials of ||r64||^2 and ||b||^2 to global memory (once per sweep, a few
// microseconds: kept out of the iteration's registers).
__device__ __noinline__ void residual_phase(const SysDesc& S, int state, int g0, int g1, int n1,
                                            int n_ow) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
  for (int g = g0 + w; g < g1; g += W) {
    const int node = NODES_PER_WARP * g + lane / 6, r = lane % 6, i = 6 * node + r;
    double part = 0.0, part_b = 0.0;
    if (lane < 6 * NODES_PER_WARP && node < n1) {
      const double bi = __ldg(S.b + i);
      double acc = bi;
      part_b = bi * bi;
      if (state == ST_RESID) {
        double dot = 0.0;
        const int j1 = __ldg(S.row_ptr + node + 1);
        for (int j = __ldg(S.row_ptr + node); j < j1; ++j) {
          const double2* kv = reinterpret_cast<const double2*>(S.K64 + (size_t)j * 36 + 6 * r);
          const double2* xv = reinterpret_cast<const double2*>(S.x + 6 * (size_t)__ldg(S.col + j));
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const double2 kk = __ldg(kv + q), xx = __ldcg(xv + q);
            dot = fma(kk.x, xx.x, dot);
            dot = fma(kk.y, xx.y, dot);
          }
        }
        acc -= dot;
      }
      S.r64[i] = acc;
      part = acc * acc;
    }
    part = warp_sum(part);
    part_b = warp_sum(part_b);
    if (lane == 0) {
      S.part_a[g] = part;
      S.part_a[n_ow + g] = part_b;
    }
  }
}

// INIT and RESID, phase B: r = r64 / ||r64|| of the CTA's rows.
__device__ __noinline__ void scale_residual(const SysDesc& S, double rr64, int n0, int nown,
                                            float* R) {
  const double inv_norm = 1.0 / ::sqrt(rr64);
  for (int i = threadIdx.x; i < 6 * nown; i += blockDim.x)
    R[i] = (float)(__ldcg(S.r64 + 6 * (size_t)n0 + i) * inv_norm);
  __syncthreads();
}

// The scalar update after the residual pass, and after phase B outside a CG
// iteration (one thread).
__device__ __noinline__ void residual_scalars(ClShared& sh, int state, int n_vw, int n_chunks) {
  const double a = total_a(sh.red, n_vw, n_chunks);
  finish_a_scalars(&sh.sc, state, a, total_a(sh.red + CL_MAX_VWARPS, n_vw, n_chunks), &sh.n_done);
}
__device__ __noinline__ void sweep_scalars(ClShared& sh, int state, double s1, double s2) {
  finish_b(&sh.sc, state, s1, s2, &sh.n_done, true);
}

// A system's CG on one cluster, up to max_steps steps (an A and a B phase
// each) from the state in its SysScalars, which it leaves ready for more.
template <bool TWO, bool JAC, int KREG, bool GRID>
__global__ void __launch_bounds__(KREG ? CL_REG_THREADS : CL_MAX_THREADS, 1) cluster_cg_kernel(
    const SysDesc* __restrict__ sys, const int* __restrict__ list, int* __restrict__ flags,
    int max_steps, int smem_bytes, int tm_cols, int m_tm, int team, unsigned long long* slots) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  __shared__ ClShared sh;
  static_assert(!(TWO && GRID), "the coarse correction exchanges through a cluster");
  const unsigned C = GRID ? (unsigned)team : cl_size();
  const unsigned rank = GRID ? blockIdx.x % C : cl_rank();
  const int tid = threadIdx.x, nth = blockDim.x, w = tid >> 5, lane = tid & 31;
  {
    const SysDesc& G = sys[list[blockIdx.x / C]];
    if (*(volatile const int*)&G.sc->state == ST_DONE) return;  // alike in every CTA
    if (!GRID) cl_arrive();  // waited for before the first store to another CTA
#pragma unroll 1
    for (int i = tid; i < (int)(sizeof(SysDesc) / 4); i += nth)
      reinterpret_cast<int*>(&sh.sys)[i] = reinterpret_cast<const int*>(&G)[i];
#pragma unroll 1
    for (int i = tid; i < (int)(sizeof(SysScalars) / 4); i += nth)
      reinterpret_cast<int*>(&sh.sc)[i] = __ldcg(reinterpret_cast<const int*>(G.sc) + i);
  }
  if (tid == 0) {
    sh.n_done = 1;
    sh.lo = INT_MAX;
    sh.hi = 0;
    if (GRID) {
      sh.epoch = 0u;
      sh.lost = 0;
      sh.team = team;
      sh.copy = (int)rank % CL_TEAM_COPIES;
      sh.slots = slots + CL_TEAM_WORDS * (blockIdx.x / C);
      sh.flags = flags;
    }
  }
  if (GRID && tid < 12) sh.before[tid / 6][tid % 6] = 0ull;
  if (GRID)
    for (int i = tid; i < 96; i += nth) sh.words[i / 6][i % 6] = 0ull;
  __syncthreads();
  const SysDesc& S = sh.sys;
  const int n = S.n_nodes, n_tiles = S.n_tiles, n_ow = WARPS * n_tiles;
  const int T0 = n_tiles * (int)rank / (int)C, T1 = n_tiles * ((int)rank + 1) / (int)C;
  // W: warps that own tiles, the system's own number (a launch may have more,
  // for another system of its list: the plan counts slots of K for this many)
  const int nt = T1 - T0;
  const int W = min(min(nth >> 5, cluster_warps((n_tiles + (int)C - 1) / (int)C)), max(nt, 1));
  const int n0 = min(n, TILE * T0), n1 = min(n, TILE * T1), nown = n1 - n0;
  const int U0 = __ldg(S.toff + T0), U1 = __ldg(S.toff + T1);
  {  // the nodes that this CTA's rows read
    int lo = INT_MAX, hi = 0;
#pragma unroll 1
    for (int i = n0 + tid; i < n1; i += nth) {
      lo = min(lo, __ldg(S.col + __ldg(S.row_ptr + i)));
      hi = max(hi, __ldg(S.col + __ldg(S.row_ptr + i + 1) - 1) + 1);
    }
    if (hi > lo) {
      atomicMin(&sh.lo, lo);
      atomicMax(&sh.hi, hi);
    }
  }
  __syncthreads();
  const int lo = nown ? sh.lo : 0, wn = nown ? sh.hi - sh.lo : 0;

  // shared memory (cluster_smem_bytes is the same sum)
  unsigned char* sp = cl_smem;
  auto take = [&sp](size_t bytes) {
    unsigned char* p = sp;
    sp += (bytes + 15) & ~(size_t)15;
    return p;
  };
  // first what other CTAs store into, at the same place in each
  Fix* fixA = reinterpret_cast<Fix*>(take(GRID ? 0 : 16 * (size_t)n_tiles));  // p^T q per tile
  Fix* fixB = reinterpret_cast<Fix*>(take(GRID ? 0 : 16 * (size_t)n_tiles));  // r^T z per tile
  Fix* fixR = reinterpret_cast<Fix*>(take(GRID ? 0 : 16 * (size_t)n_tiles));  // r^T r per tile
  Fix* fixC = reinterpret_cast<Fix*>(take(TWO ? 16 * 8 * COARSE_ROW_BLOCKS : 0));  // w^T y
  float* wS = reinterpret_cast<float*>(take(TWO ? 8 * COARSE_MAX_N : 0));  // two iterations
  float* yS = reinterpret_cast<float*>(take(TWO ? 8 * COARSE_MAX_N : 0));
  int* aptr = reinterpret_cast<int*>(take(TWO ? 4 * (COARSE_MAX_AGG + 1) : 0));
  float* Zw = reinterpret_cast<float*>(take(GRID ? 0 : 24 * (size_t)wn));  // z (two-level: z_b) of the window
  float* P = reinterpret_cast<float*>(take(24 * (size_t)wn));
  float* Q = reinterpret_cast<float*>(take(24 * (size_t)nown));
  float* R = reinterpret_cast<float*>(take(24 * (size_t)nown));
  float* D = reinterpret_cast<float*>(take(24 * (size_t)nown));
  float2* gA = reinterpret_cast<float2*>(take(8 * WARPS * (size_t)nt));
  float4* tB = reinterpret_cast<float4*>(take(32 * (size_t)nt));
  // the preconditioner in shared memory, or (m_tm) in the last of the warp's
  // columns of tensor memory, 24 a tile
  const int tm_share = tm_cols / ((W + 3) / 4);
  const int tm_m = m_tm ? M32_PACK * ((nt + W - 1) / W) : 0;
  float4* Ms = reinterpret_cast<float4*>(take(m_tm ? 0 : (JAC ? 768 : 3072) * (size_t)nt));
  // two-level: offsets of the window's nodes; members of this CTA's aggregates
  // (rank, rank + C, ...), offset and node index
  float4* rfw = reinterpret_cast<float4*>(take(TWO ? 16 * (size_t)wn : 0));
  const int n_mine = TWO && S.n_agg > (int)rank ? (S.n_agg - (int)rank + (int)C - 1) / (int)C : 0;
  if (TWO) {
    if (tid == 0) {
      int at = 0;
#pragma unroll 1
      for (int k = 0; k < n_mine; ++k) {
        const int a = (int)(rank + C * k);
        aptr[k] = at;
        at += __ldg(S.agg_ptr + a + 1) - __ldg(S.agg_ptr + a);
      }
      aptr[n_mine] = at;
    }
    __syncthreads();
  }
  float4* member = reinterpret_cast<float4*>(take(TWO ? 16 * (size_t)aptr[n_mine] : 0));
  uint16_t* slot = reinterpret_cast<uint16_t*>(take(64 * (size_t)(U1 - U0)));  // [position][lane]
  int* toffS = reinterpret_cast<int*>(take(4 * (size_t)(nt + 1)));
  sp = cl_smem + (((sp - cl_smem) + 127) & ~(size_t)127);
  ulonglong2* Kres = reinterpret_cast<ulonglong2*>(sp);
  const int left = smem_bytes - (int)(sp - cl_smem);
  // positions of K per warp in shared memory
  const int cap = left > 0 ? left / (CL_POS_BYTES * W) : 0;
  if (tid == 0) {
    sh.fixA = fixA;
    sh.fixB = fixB;
    sh.fixR = fixR;
    sh.fixC = fixC;
    sh.gA = gA;
    sh.tB = tB;
    sh.yS = yS;
    sh.wS = wS;
    sh.aptr = aptr;
    sh.member = member;
    sh.rfw = rfw;
    sh.Ms = Ms;
    sh.T0 = T0;
    sh.nt = nt;
    sh.n_ow = n_ow;
    sh.n_mine = n_mine;
    sh.rz_known = sh.sc.rz;
    sh.thr = sh.sc.inner_thr;
  }

  // columns as window slots; kNoBlock past a row's end, where the sum skips
  // them (the two idle lanes read slot 0)
#pragma unroll 1
  for (int t = T0 + w; t < T1; t += nth >> 5) {
    const int a = __ldg(S.toff + t), e = __ldg(S.toff + t + 1), i = TILE * t + lane;
    const bool act = lane < TILE && i < n;
    const int j0 = act ? __ldg(S.row_ptr + i) : 0, c = act ? __ldg(S.row_ptr + i + 1) - j0 : 0;
#pragma unroll 1
    for (int k = 0; k < e - a; ++k)
      slot[32 * (a - U0 + k) + lane] = k < c ? (uint16_t)(__ldg(S.col + j0 + k) - lo)
                                     : lane < TILE ? kNoBlock : (uint16_t)0;
  }
#pragma unroll 1
  for (int t = tid; t <= nt; t += nth) toffS[t] = __ldg(S.toff + T0 + t);
  if (TWO) {
    const float4* rf = reinterpret_cast<const float4*>(S.node_rf);
#pragma unroll 1
    for (int i = tid; i < wn; i += nth) {
      float4 o = __ldg(rf + lo + i);
      unsigned info = (unsigned)__ldg(S.agg_of + lo + i);
#pragma unroll 1
      for (int d = 0; d < 6; ++d)
        info |= (__ldg(S.fixed + 6 * (size_t)(lo + i) + d) ? 1u : 0u) << (8 + d);
      o.w = __uint_as_float(info);
      rfw[i] = o;
    }
#pragma unroll 1
    for (int k = w; k < n_mine; k += nth >> 5) {
      const int b = __ldg(S.agg_ptr + rank + C * k), c = aptr[k + 1] - aptr[k];
#pragma unroll 1
      for (int q = lane; q < c; q += 32) {
        const int i = __ldg(S.agg_nodes + b + q);
        float4 o = __ldg(rf + i);
        o.w = __int_as_float(i);
        member[aptr[k] + q] = o;
      }
    }
  }
  // preconditioner: [tile][float4 0..5][lane = node] (Jacobi: six floats a node)
  if (m_tm) {
  } else if (!JAC) {
    const float4* m4 = reinterpret_cast<const float4*>(S.M32) + 6 * (size_t)n0;
#pragma unroll 1
    for (int i = tid; i < 6 * nown; i += nth) {
      const int l = i / 6, c = i - 6 * l;
      Ms[192 * (l / TILE) + 32 * c + l % TILE] = __ldg(m4 + i);
    }
  } else {
    const float2* m2 = reinterpret_cast<const float2*>(S.M32 + 6 * (size_t)n0);
#pragma unroll 1
    for (int i = tid; i < 3 * nown; i += nth) reinterpret_cast<float2*>(Ms)[i] = __ldg(m2 + i);
  }
  // This warp's tiles are contiguous, so its K is one run of m positions: the
  // first nkr in registers (CTAs of few warps), the next ntm in tensor memory
  // (the warp's share of its quadrant's columns), the next ns in its share of
  // shared memory, and the others come from L2 in every iteration, by plain
  // loads that run three thirds of a position ahead of the products (the
  // registers of a third are loaded again as soon as it has been used).  (A
  // ring of slots in shared memory that bulk copies refill waited for each copy
  // in turn: 48 systems 421 ms against 393, 256 x 256 shell 13.8 us an iteration
  // against 12.5; slots of a third of a position: 509 ms, 15.1 us.)
  const int ta = w < W ? T0 + nt * w / W : T1, tb = w < W ? T0 + nt * (w + 1) / W : T1;
  const int pa = __ldg(S.toff + ta), m = __ldg(S.toff + tb) - pa;
  if (tm_cols && w == 0) tm_alloc(&sh.tmem, tm_cols);
  __syncthreads();
  const ulonglong2* Kg = reinterpret_cast<const ulonglong2*>(S.klo) + (size_t)pa * CL_POS_F4;
  KPos kr[KREG ? KREG : 1];
#pragma unroll
  for (int i = 0; i < KREG; ++i)
    if (i < m) {
      const uint4* k4 = reinterpret_cast<const uint4*>(Kg + (size_t)i * CL_POS_F4) + lane;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const uint4 v = __ldg(k4 + 32 * q);
        kr[i].r[4 * q] = v.x; kr[i].r[4 * q + 1] = v.y;
        kr[i].r[4 * q + 2] = v.z; kr[i].r[4 * q + 3] = v.w;
      }
    }
  const int nkr = min(m, KREG), ntm = min(m - nkr, (tm_share - tm_m) / 36);
  const int ns = min(cap, m - nkr - ntm), ng = m - nkr - ntm - ns;
  Kg += (size_t)nkr * CL_POS_F4;
  const uint32_t tmw =
      tm_cols ? sh.tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((w >> 2) * tm_share) : 0u;
#pragma unroll 1
  for (int i = 0; i < 9 * ntm; ++i) tm_st(tmw + 4 * i, __ldg(Kg + lane + 32 * i));
  const uint32_t tmm = tmw + tm_share - tm_m;
  if (tid == 0) sh.tm_m = tm_share - tm_m;
  if (m_tm)
#pragma unroll 1
    for (int t = ta; t < tb; ++t) {
      const int node = TILE * t + lane;
      const bool act = lane < TILE && node < n;
      const ulonglong2* m2 = reinterpret_cast<const ulonglong2*>(S.M32) + 6 * (size_t)(act ? node : n0);
#pragma unroll 1
      for (int c = 0; c < 6; ++c) tm_st(tmm + M32_PACK * (t - ta) + 4 * c, __ldg(m2 + c));
    }
  tm_wait_st();
  ulonglong2* Kw = Kres + (size_t)w * cap * CL_POS_F4;
  Kg += (size_t)ntm * CL_POS_F4;
#pragma unroll 4
  for (int i = lane; i < ns * CL_POS_F4; i += 32) Kw[i] = __ldg(Kg + i);
  const int streamed = pa + nkr + ntm + ns;  // the first position that streams
  // the vectors of a sweep under way
  {
    const float2* r2 = reinterpret_cast<const float2*>((const float*)S.r + 6 * (size_t)n0);
    const float2* d2 = reinterpret_cast<const float2*>((const float*)S.dx + 6 * (size_t)n0);
    const float2* p2 = reinterpret_cast<const float2*>(
        (const float*)(sh.sc.parity ? S.p1 : S.p0) + 6 * (size_t)lo);
    const float2* z2 = reinterpret_cast<const float2*>((const float*)S.z + 6 * (size_t)lo);
#pragma unroll 1
    for (int i = tid; i < 3 * nown; i += nth) {
      reinterpret_cast<float2*>(R)[i] = __ldcg(r2 + i);
      reinterpret_cast<float2*>(D)[i] = __ldcg(d2 + i);
    }
#pragma unroll 1
    for (int i = tid; i < 3 * wn; i += nth) {
      reinterpret_cast<float2*>(P)[i] = __ldcg(p2 + i);
      if (!GRID) reinterpret_cast<float2*>(Zw)[i] = __ldcg(z2 + i);
    }
  }
  bool z_alt = false;   // teams without a cluster: z is in S.zb, not S.z
  bool zdirect = true;  // Zw holds z itself (two-level: until this launch's first z_b)
  int state = sh.sc.state, parity = sh.sc.parity, iters = sh.sc.iters, inner = sh.sc.inner;
  // scalars of the iteration, alike in every thread: r^T z (exact while known),
  // beta, grids of the three sums, the buffer of the last phase B
  bool known = true;
  Apx rz = apx_f64(sh.sc.rz);
  float beta = (float)sh.sc.beta;
  int kA = 0, kB = kGrid - f64_exp(sh.sc.rz), kR = kGrid - f64_exp(sh.sc.rr), par = 0;
  bool have_kA = false;
  // Every CTA has started by now (one that has not must not be stored to: the
  // CTAs of a cluster are placed together, but an SM that has to drain another
  // kernel first starts its own late) ...
  if (!GRID) cl_wait();
  if (!GRID && tid < (int)C) {
    cl_st(cl_map(smem_addr(&sh.wlo[rank]), tid), lo);
    cl_st(cl_map(smem_addr(&sh.whi[rank]), tid), lo + wn);
  }
  if (!GRID) cl_sync();  // ... and has read the system's state and set up its windows
  // (a launch may begin in the fold, which reads D by other threads than loaded it;
  // nothing else separates a team's copies from its first step)
  if (GRID) __syncthreads();
  unsigned dest = 0u;  // CTAs whose windows reach this warp's nodes
#pragma unroll 1
  for (unsigned c = 0; !GRID && c < C; ++c)
    if (sh.wlo[c] < min(n, TILE * tb) && sh.whi[c] > TILE * ta && tb > ta) dest |= 1u << c;

#pragma unroll 1
  for (int step = 0; step < max_steps && state != ST_DONE && !(GRID && sh.lost); ++step) {
    float alpha = 0.f;
    // ------------------------------------------------------------- phase A
    if (state == ST_PCG) {
      const bool first = inner == 0;
      if (GRID) {
        const float b = first ? 0.f : beta;
        float2* P2 = reinterpret_cast<float2*>(P);
        const float2* Z2 = reinterpret_cast<const float2*>((const float*)(z_alt ? S.zb : S.z) +
                                                           6 * (size_t)lo);
#pragma unroll 1
        for (int i = tid; i < 3 * wn; i += 4 * nth) {
          float2 z[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (i + u * nth < 3 * wn) z[u] = __ldcg(Z2 + i + u * nth);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (i + u * nth < 3 * wn) {
              const float2 p = first ? z[u] : P2[i + u * nth];
              P2[i + u * nth] = make_float2(fmaf(b, p.x, z[u].x), fmaf(b, p.y, z[u].y));
            }
        }
      } else if (!TWO || zdirect) {
        const float b = first ? 0.f : beta;
        float2* P2 = reinterpret_cast<float2*>(P);
        const float2* Z2 = reinterpret_cast<const float2*>(Zw);
#pragma unroll 1
        for (int i = tid; i < 3 * wn; i += nth) {
          const float2 z = Z2[i], p = first ? z : P2[i];
          P2[i] = make_float2(fmaf(b, p.x, z.x), fmaf(b, p.y, z.y));
        }
      } else {
        const float b = first ? 0.f : beta;
        const float* y = sh.yS + par * COARSE_MAX_N;
        const float4* rfw = sh.rfw;
#pragma unroll 1
        for (int i = tid; i < wn; i += nth) {
          float zb[6], z[6], p[6];
          lds6(Zw + 6 * i, zb);
          prolong_node(rfw[i], y, zb, z);
          lds6(P + 6 * i, p);
#pragma unroll
          for (int d = 0; d < 6; ++d) p[d] = fmaf(b, first ? z[d] : p[d], z[d]);
          sts6(P + 6 * i, p);
        }
      }
      __syncthreads();
      {  // q = K p over this warp's tiles
        int t = ta, left = m ? toffS[ta - T0 + 1] - toffS[ta - T0] : 0;  // positions of the tile
        const uint16_t* sl = slot + 32 * (pa - U0) + lane;
        unsigned long long acc[3] = {0ull, 0ull, 0ull};
        auto row_end = [&] {
          if (--left) return;  // else the tile's rows are done
          const int l = TILE * t + lane - n0;
          if (lane < TILE && l < n1 - n0) {
            float q[6];
#pragma unroll
            for (int a = 0; a < 3; ++a) unpack2(acc[a], q[2 * a], q[2 * a + 1]);
            sts6(Q + 6 * l, q);
          }
          acc[0] = acc[1] = acc[2] = 0ull;
          if (++t < tb) left = toffS[t - T0 + 1] - toffS[t - T0];
        };
        auto column = [&](float (&p)[6]) {  // p at the next position's column
          const int at = *sl;
          sl += 32;
          lds6(P + (at == kNoBlock ? 0 : 6 * at), p);
          return at != kNoBlock;
        };
        // the positions in registers, then the others
#pragma unroll
        for (int i = 0; i < KREG; ++i)
          if (i < nkr) {
            float p[6];
            if (column(p)) fma_pos(kr[i], p, acc);
            row_end();
          }
        __syncwarp();
#pragma unroll 1
        for (int i = 0; i < ntm + ns; ++i) {
          KPos K;
          float p[6];
          if (i < ntm) {
            tm_ld36(tmw + 36 * i, K.r);
          } else {
            const uint4* kp = reinterpret_cast<const uint4*>(Kw + (size_t)(i - ntm) * CL_POS_F4) + lane;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
              const uint4 v = kp[32 * q];
              K.r[4 * q] = v.x; K.r[4 * q + 1] = v.y; K.r[4 * q + 2] = v.z; K.r[4 * q + 3] = v.w;
            }
          }
          const bool real = column(p);
          if (i < ntm) tm_wait_ld();
          tm_loaded(K.r);
          if (real) fma_pos(K, p, acc);
          row_end();
          __syncwarp();
        }
        if (ng > 0) {
          const ulonglong2* kp = reinterpret_cast<const ulonglong2*>(S.klo) +
                                 (size_t)streamed * CL_POS_F4 + lane;
          ulonglong2 k[9];
#pragma unroll
          for (int q = 0; q < 9; ++q) k[q] = __ldg(kp + 32 * q);
#pragma unroll 1
          for (int i = 1; i <= ng; ++i) {
            float p[6];
            const bool real = column(p);
            if (i < ng) kp += CL_POS_F4;  // (the last position is loaded again, and not used)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              unsigned long long s = acc[a];
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                s = fma2(k[3 * a + q].x, pack2(p[2 * q], p[2 * q]), s);
                s = fma2(k[3 * a + q].y, pack2(p[2 * q + 1], p[2 * q + 1]), s);
              }
              if (real) acc[a] = s;
#pragma unroll
              for (int q = 0; q < 3; ++q) k[3 * a + q] = __ldg(kp + 32 * (3 * a + q));
            }
            row_end();
            __syncwarp();
          }
        }
      }
      // p^T q: four lanes per 5-node group (six groups a tile): lane j forms the
      // levels 16, 8 and 4 of the tree over the rows l = j mod 4 of the group's
      // 30 (lanes 30 and 31 of that tree hold zero), two shuffles the last two
      __syncwarp();
      Fix pq_sum{0, 0u, 0u};
#pragma unroll 1
      for (int t = ta; t < tb; ++t) {
        const int g = WARPS * t + (lane >> 2), j = lane & 3;
        DF v = {0.f, 0.f};
        if (lane < 4 * WARPS) {
          const float* gp = P + 30 * g - 6 * lo + j;
          const float* gq = Q + 30 * g - 6 * n0 + j;
          const int rows = 6 * n1 - 30 * g - j;  // rows of the group from row j on
          DF x[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            x[k] = (k < 7 || j < 2) && 4 * k < rows ? df_prod(gp[4 * k], gq[4 * k]) : DF{0.f, 0.f};
#pragma unroll
          for (int k = 0; k < 4; ++k) x[k] = df_add(x[k], x[k + 4]);
          x[0] = df_add(x[0], x[2]);
          x[1] = df_add(x[1], x[3]);
          v = df_add(x[0], x[1]);
        }
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) {
          DF y;
          y.hi = __shfl_down_sync(0xffffffffu, v.hi, o);
          y.lo = __shfl_down_sync(0xffffffffu, v.lo, o);
          v = df_add(v, y);
        }
        Fix f{0, 0u, 0u};
        if (lane < 4 * WARPS && j == 0) {
          sh.gA[g - WARPS * T0] = make_float2(v.hi, v.lo);
          f = to_fix(v, kA);
        }
        if (GRID) {
          pq_sum = Fix{pq_sum.s + f.s, pq_sum.a + f.a, pq_sum.bad | f.bad};
        } else {
          f = fix_warp_sum(f);
          if (lane < (int)C) push_fix(sh.fixA + t, f, lane);
        }
      }
      if (GRID) {
        pq_sum = fix_warp_sum(pq_sum);
        if (lane == 0) team_add(sh, 0, pq_sum);
        team_sync(sh, false);
      } else {
        cl_sync();
      }
      // alpha = r^T z / p^T q, by every warp
      Apx pq;
      const Fix fa = GRID ? sh.tot[0] : fix_total(sh.fixA, S.n_tiles, lane);
      if (have_kA && apx_fix(fa, kA, pq) && apx_quotient(rz, pq, alpha)) {
        kA = kGrid - pq.e;
      } else {
        exact_sums<TWO, GRID>(sh, par, true);
        const double s = sh.ex_pq;
        if (!f64_positive(s)) {
          if (tid == 0) sh.sc.status = SSO_ERR_SINGULAR;
          state = ST_DONE;
          break;
        }
        alpha = (float)((known ? sh.rz_known : sh.ex_rz) / s);
        kA = kGrid - f64_exp(s);
        have_kA = true;
      }
      parity ^= 1;
    } else if (state != ST_FOLD) {  // INIT, RESID
      const int n_ow = sh.n_ow, n_vw = (n_ow + 255) / 256;
      residual_phase(S, state, WARPS * T0, WARPS * T1, n1, n_ow);
      all_sync<GRID>(sh);
#pragma unroll 1
      for (int v = w; v < 2 * n_vw; v += nth >> 5) {
        const bool second = v >= n_vw;
        const int k = second ? v - n_vw : v;
        const double s = vwarp_sum(S.part_a + (second ? n_ow : 0), k, n_ow, lane);
        if (lane == 0) sh.red[(second ? CL_MAX_VWARPS : 0) + k] = s;
      }
      __syncthreads();
      if (tid == 0) residual_scalars(sh, state, n_vw, S.n_chunks);
      __syncthreads();
    }
    // ------------------------------------------------------------- phase B
    if (state == ST_FOLD) {
      const double scale = sh.sc.scale;
      double* x = S.x + 6 * (size_t)n0;
#pragma unroll 1
      for (int i = tid; i < 6 * nown; i += nth) {
        x[i] = fma(scale, (double)D[i], __ldcg(x + i));
        D[i] = 0.f;
      }
      state = ST_RESID;
      all_sync<GRID>(sh);  // the other CTAs read x next
      continue;
    }
    if (state != ST_PCG) {
      const double rr64 = sh.sc.rr64;
      if (!(f64_finite(rr64) && !(rr64 <= sh.sc.rtol2 * sh.sc.ff))) {
        // converged or not finite: no new sweep
        __syncthreads();
        if (tid == 0) sweep_scalars(sh, state, 0.0, 0.0);
        __syncthreads();
        state = sh.sc.state;
        continue;
      }
      scale_residual(S, rr64, n0, nown, R);
    }
    par ^= 1;
    // z goes to the buffer that no CTA still reads
    float* zn = GRID ? (float*)(z_alt ? S.z : S.zb) : nullptr;
    Fix b_sum{0, 0u, 0u};
    __syncwarp();
#pragma unroll 1
    for (int t = ta; t < tb; ++t) {
      const int node = TILE * t + lane, l = node - n0;
      DF d1 = {0.f, 0.f}, d2 = {0.f, 0.f};
      float rv[6], zv[6], mm[JAC ? 6 : M32_PACK];
      if (m_tm) {
        if constexpr (!JAC) {
          uint32_t r[M32_PACK];
          tm_ld24(tmw + sh.tm_m + M32_PACK * (t - ta), r);
          tm_wait_ld();
          tm_loaded(r);
#pragma unroll
          for (int c = 0; c < M32_PACK; ++c) mm[c] = __uint_as_float(r[c]);
        }
      }
      if (lane < TILE && node < n1) {
        lds6(R + 6 * l, rv);
        if (state == ST_PCG) {
          float pv[6], qv[6], dv[6];
          lds6(P + 6 * (node - lo), pv);
          lds6(Q + 6 * l, qv);
          lds6(D + 6 * l, dv);
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            dv[c] = fmaf(alpha, pv[c], dv[c]);
            rv[c] = fmaf(-alpha, qv[c], rv[c]);
          }
          sts6(D + 6 * l, dv);
          sts6(R + 6 * l, rv);
        }
        if (TWO) sts6((float*)S.r + 6 * (size_t)node, rv);  // restricted by any CTA
        if (!JAC) {
          if (!m_tm) {
            const float4* mp = sh.Ms + 192 * (t - T0) + lane;
#pragma unroll
            for (int c = 0; c < M32_PACK / 4; ++c) {
              const float4 v = mp[32 * c];
              mm[4 * c] = v.x; mm[4 * c + 1] = v.y; mm[4 * c + 2] = v.z; mm[4 * c + 3] = v.w;
            }
          }
#pragma unroll
          for (int a = 0; a < 6; ++a) {
            float acc = 0.f;
#pragma unroll
            for (int c = 0; c < 6; ++c) acc = fmaf(mm[sym6(a, c)], rv[c], acc);
            zv[a] = acc;
          }
        } else {
          lds6(reinterpret_cast<const float*>(sh.Ms) + 6 * l, mm);
#pragma unroll
          for (int a = 0; a < 6; ++a) zv[a] = mm[a] * rv[a];
        }
      }
      // z (z_b) into every window that holds the node
#pragma unroll 1
      for (unsigned left = dest; left; left &= left - 1) {
        const int c = __ffs(left) - 1, wl = sh.wlo[c];
        if (lane < TILE && node < n1 && node >= wl && node < sh.whi[c]) {
          const uint32_t a = cl_map(smem_addr(Zw + 6 * (node - wl)), c);
          cl_st2(a, zv[0], zv[1]);
          cl_st2(a + 8, zv[2], zv[3]);
          cl_st2(a + 16, zv[4], zv[5]);
        }
      }
      if (GRID && lane < TILE && node < n1) sts6(zn + 6 * (size_t)node, zv);
      if (lane < TILE && node < n1) {
        d1 = df_prod(rv[0], zv[0]);
        d2 = df_prod(rv[0], rv[0]);
#pragma unroll
        for (int a = 1; a < 6; ++a) {
          d1 = df_add(d1, df_prod(rv[a], zv[a]));
          d2 = df_add(d2, df_prod(rv[a], rv[a]));
        }
      }
      // both trees at once: the first level leaves r^T z in lanes 0-15 and
      // r^T r in lanes 16-31 (the pair's sum does not depend on its order)
      DF v = lane < 16 ? d1 : d2, y = lane < 16 ? d2 : d1;
      y.hi = __shfl_xor_sync(0xffffffffu, y.hi, 16);
      y.lo = __shfl_xor_sync(0xffffffffu, y.lo, 16);
      v = df_add(v, y);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        y.hi = __shfl_down_sync(0xffffffffu, v.hi, o, 16);
        y.lo = __shfl_down_sync(0xffffffffu, v.lo, o, 16);
        v = df_add(v, y);
      }
      if ((lane & 15) == 0)
        reinterpret_cast<float2*>(sh.tB + par * sh.nt + t - T0)[lane >> 4] = make_float2(v.hi, v.lo);
      v.hi = __shfl_sync(0xffffffffu, v.hi, lane & 16);
      v.lo = __shfl_sync(0xffffffffu, v.lo, lane & 16);
      const Fix f = to_fix(v, lane < 16 ? kB : kR);
      if (GRID)
        b_sum = Fix{b_sum.s + f.s, b_sum.a + f.a, b_sum.bad | f.bad};
      else if ((lane & 15) < (int)C)
        push_fix((lane < 16 ? sh.fixB : sh.fixR) + t, f, lane & 15);
    }
    if (GRID) {
      if ((lane & 15) == 0) team_add(sh, lane >> 4, b_sum);
      z_alt = !z_alt;
    }
    all_sync<GRID>(sh);
    if (TWO) {
      // coarse correction: w = P^T r, y = A_c^-1 w, r^T z = r^T z_b + w^T y
      const int nc = 6 * S.n_agg;
      const int n_rb = (nc + COARSE_ROWS_PER_BLOCK - 1) / COARSE_ROWS_PER_BLOCK;
      const int my_rb = n_rb > (int)rank ? (n_rb - (int)rank + (int)C - 1) / (int)C : 0;
      float* ws = sh.wS + par * COARSE_MAX_N;
      float* ys = sh.yS + par * COARSE_MAX_N;
      // rows ra, ra + 1 of the coarse inverse, eight columns a lane
      constexpr int CPL = (COARSE_MAX_N + 31) / 32;
      float xa[CPL], xb[CPL];
      auto load_rows = [&](int it) {
        const int ra = COARSE_ROWS_PER_BLOCK * ((int)rank + (int)C * (it >> 3)) + 2 * (it & 7);
        const float* A = S.Aci + (size_t)ra * nc;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          const int c = lane + 32 * k;
          xa[k] = (ra < nc && c < nc) ? __ldg(A + c) : 0.f;
          xb[k] = (ra + 1 < nc && c < nc) ? __ldg(A + nc + c) : 0.f;
        }
      };
#pragma unroll 1
      for (int k0 = w; k0 < sh.n_mine; k0 += nth >> 5) {
        const float4* mb = sh.member + sh.aptr[k0];
        const int e = sh.aptr[k0 + 1] - sh.aptr[k0], a = (int)rank + (int)C * k0;
        const float* r = (const float*)S.r;
        float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        // (one member of a lane at a time: loads of several in flight cost
        // registers, and a spilled register is an L2 round trip here, where
        // every barrier's acquire drops L1; measured 256 ms for 128 shells of
        // 64 x 64, 262 with two members in flight, 307 with four)
#pragma unroll 1
        for (int q = lane; q < e; q += 32) {
          const float4 o = mb[q];
          float v[6];
          ldcg6(r + 6 * (size_t)__float_as_int(o.w), v);
          acc[0] += v[0];
          acc[1] += v[1];
          acc[2] += v[2];
          acc[3] += fmaf(o.y, v[2], fmaf(-o.z, v[1], v[3]));
          acc[4] += fmaf(o.z, v[0], fmaf(-o.x, v[2], v[4]));
          acc[5] += fmaf(o.x, v[1], fmaf(-o.y, v[0], v[5]));
        }
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int d = 0; d < 6; ++d) acc[d] += __shfl_down_sync(0xffffffffu, acc[d], o);
#pragma unroll
        for (int d = 0; d < 6; ++d) {
          const float s = __shfl_sync(0xffffffffu, acc[d], 0);
          if (lane < (int)C) cl_st(cl_map(smem_addr(ws + 6 * a + d), lane), s);
        }
      }
      cl_sync();
#pragma unroll 1
      for (int it = w; it < 8 * my_rb; it += nth >> 5) {
        load_rows(it);
        const int rb = (int)rank + (int)C * (it >> 3);
        const int ra = COARSE_ROWS_PER_BLOCK * rb + 2 * (it & 7), rbb = ra + 1;
        float aa = 0.f, ab = 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          const int c = lane + 32 * k;
          const float wc = c < nc ? ws[c] : 0.f;
          aa = fmaf(xa[k], wc, aa);
          ab = fmaf(xb[k], wc, ab);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          aa += __shfl_down_sync(0xffffffffu, aa, o);
          ab += __shfl_down_sync(0xffffffffu, ab, o);
        }
        aa = __shfl_sync(0xffffffffu, aa, 0);
        ab = __shfl_sync(0xffffffffu, ab, 0);
        DF v = {0.f, 0.f};
        if (ra < nc) v = df_prod(aa, ws[ra]);
        if (rbb < nc) v = df_add(v, df_prod(ab, ws[rbb]));
        const Fix f = to_fix(v, kB);
        if (lane < (int)C) {
          if (ra < nc) cl_st(cl_map(smem_addr(ys + ra), lane), aa);
          if (rbb < nc) cl_st(cl_map(smem_addr(ys + rbb), lane), ab);
          push_fix(sh.fixC + 8 * rb + (it & 7), f, lane);
        }
      }
      cl_sync();
      zdirect = false;
    }
    if (state == ST_PCG) {
      ++iters;
      ++inner;
      if (w == 0) {
        Fix f = GRID ? sh.tot[0] : fix_total(sh.fixB, S.n_tiles, lane);
        if (TWO) {
          const int n_rb = (6 * S.n_agg + COARSE_ROWS_PER_BLOCK - 1) / COARSE_ROWS_PER_BLOCK;
          const Fix g = fix_total(sh.fixC, 8 * n_rb, lane);
          f = Fix{f.s + g.s, f.a + g.a, f.bad | g.bad};
        }
        Apx rz_new{1.f, 0.f, 0};
        float b;
        const bool ok = apx_fix(f, kB, rz_new) & apx_quotient(rz_new, rz, b);
        if (lane == 0) {
          sh.ok = ok;
          sh.beta = b;
          sh.rz = rz_new;
        }
      }
      if (w == 1) {
        const Fix f = GRID ? sh.tot[1] : fix_total(sh.fixR, S.n_tiles, lane);
        Apx rr{1.f, 0.f, 0};
        bool clear;
        const bool end = fix_le(f, kR, sh.thr, clear);
        const bool ok = apx_fix(f, kR, rr);
        if (lane == 0) {
          sh.rr_ok = clear && ok;
          sh.end = end;
          sh.e_rr = rr.e;
        }
      }
      __syncthreads();
      bool end = sh.end;
      int e_rr = sh.e_rr;
      beta = sh.beta;
      if (sh.ok && sh.rr_ok) {
        rz = sh.rz;
        known = false;
      } else {
        double rz_old = sh.rz_known;
        if (!known) {
          exact_sums<TWO, GRID>(sh, par ^ 1, false);
          rz_old = sh.ex_rz;
        }
        exact_sums<TWO, GRID>(sh, par, false);
        const double s1 = sh.ex_rz, s2 = sh.ex_rr;
        if (!(f64_finite(s1) && f64_finite(s2))) {
          if (tid == 0) sh.sc.status = SSO_ERR_SINGULAR;
          state = ST_DONE;
          break;
        }
        beta = (float)(s1 / rz_old);
        end = s2 <= sh.thr;
        if (tid == 0) sh.rz_known = s1;
        __syncthreads();
        known = true;
        rz = apx_f64(s1);
        e_rr = f64_exp(s2);
        if (!f64_positive(s1)) rz.e = -2000;  // refused by the quotient test
      }
      kB = kGrid - rz.e;
      kR = kGrid - e_rr;
      if (end || iters >= sh.sc.max_iter) state = ST_FOLD;
    } else {
      exact_sums<TWO, GRID>(sh, par, false);
      if (tid == 0) {
        sh.sc.iters = iters;
        sweep_scalars(sh, state, sh.ex_rz, sh.ex_rr);
      }
      __syncthreads();
      state = sh.sc.state;
      inner = sh.sc.inner;
      known = true;
      rz = apx_f64(sh.sc.rz);
      if (!f64_positive(sh.sc.rz)) rz.e = -2000;
      kB = kGrid - f64_exp(sh.sc.rz);
      kR = kGrid - f64_exp(sh.sc.rr);
      if (tid == 0) {
        sh.rz_known = sh.sc.rz;
        sh.thr = sh.sc.inner_thr;
      }
      __syncthreads();
      have_kA = false;
    }
  }
  // leave the system as the two-kernel engine would: r, dx, p and z in global
  // memory, the scalars written by one thread
  if (state == ST_PCG && !known) exact_sums<TWO, GRID>(sh, par, false);
  const bool lost = GRID && sh.lost;  // a barrier gave up: the run has failed
  if (state != ST_DONE && !lost) {
    float2* r2 = reinterpret_cast<float2*>((float*)S.r + 6 * (size_t)n0);
    float2* d2 = reinterpret_cast<float2*>((float*)S.dx + 6 * (size_t)n0);
    float2* p2 = reinterpret_cast<float2*>((float*)(parity ? S.p1 : S.p0) + 6 * (size_t)n0);
#pragma unroll 1
    for (int i = tid; i < 3 * nown; i += nth) {
      r2[i] = reinterpret_cast<const float2*>(R)[i];
      d2[i] = reinterpret_cast<const float2*>(D)[i];
      p2[i] = reinterpret_cast<const float2*>(P + 6 * (n0 - lo))[i];
    }
#pragma unroll 1
    for (int i = n0 + tid; GRID && z_alt && i < n1; i += nth) {
      float z[6];
      ldcg6((const float*)S.zb + 6 * (size_t)i, z);
      sts6((float*)S.z + 6 * (size_t)i, z);
    }
#pragma unroll 1
    for (int i = n0 + tid; !GRID && i < n1; i += nth) {
      float z[6];
      lds6(Zw + 6 * (i - lo), z);
      if (TWO && !zdirect) {
        float zb[6];
#pragma unroll
        for (int d = 0; d < 6; ++d) zb[d] = z[d];
        prolong_node(sh.rfw[i - lo], sh.yS + par * COARSE_MAX_N, zb, z);
      }
      sts6((float*)S.z + 6 * (size_t)i, z);
    }
  }
  if (tm_cols && w == 0) tm_free(sh.tmem, tm_cols);
  if (!GRID) cl_sync();  // no CTA leaves while another may still store into it
  if (rank == 0 && tid == 0 && !lost) {
    sh.sc.state = state;
    sh.sc.parity = parity;
    sh.sc.iters = iters;
    sh.sc.inner = inner;
    if (state == ST_PCG) sh.sc.rz = known ? sh.rz_known : sh.ex_rz;
    sh.sc.beta = (double)beta;  // the vectors use the rounded value alone
    *S.sc = sh.sc;
    if (state == ST_DONE) atomicSub(flags, 1);
  }
}

// The FP64 CG of a system on one team of CTAs (cooperative launch), up to
// max_steps steps from the state in its SysScalars, as cluster_cg_kernel for
// the FP32 one and with the arithmetic and trees of the two-kernel engine
// (pcg_a_kernel<double>, pcg_b_kernel<double>): the same bits.
//
// What bounds it: the FP64 pipe, two multiply-adds a clock and SM, and the
// latency of two barriers and the FP64 sums after each.  The two-kernel engine
// forms p = z + beta p again for every block of every row, which doubles the
// pipe's work; here a CTA updates its window of p once, in shared memory, with
// its rows of the other vectors, M and (where it fits) K.  A CTA has few tiles,
// six warps on each: a lane per row (five nodes a warp) for the products and
// the updates, a lane per node for the dot products' trees.
// Measured, us an iteration, two kernels -> here: 41 x 41 grid shell (10,086 DOF)
// 26.8 -> 11.6, 100 x 100 39 -> 22.2, 24 x 24 shell 26 -> 12.5, 64 grid shells of
// 41 x 41 134 -> 112.  Teams of any sizes share a launch: list holds its systems,
// then their first CTAs (a launch per size: 32 grid shells of sides 8 to 60 185
// ms; 40 together, 71 with two kernels).
template <bool JAC>
__global__ void __launch_bounds__(TEAM64_THREADS, 1) team64_kernel(
    const SysDesc* __restrict__ sys, const int* __restrict__ list, int* __restrict__ flags,
    int n_list, int max_steps, int smem_bytes, unsigned long long* slots) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  __shared__ ClShared sh;
  __shared__ int entry;  // of the list: this CTA's system
  const int tid = threadIdx.x, nth = blockDim.x, w = tid >> 5, lane = tid & 31, W = nth >> 5;
  const int* first = list + n_list;
  for (int i = tid; i < n_list; i += nth)
    if (__ldg(first + i) <= (int)blockIdx.x && (int)blockIdx.x < __ldg(first + i + 1)) entry = i;
  __syncthreads();
  const int C = __ldg(first + entry + 1) - __ldg(first + entry);
  const int rank = (int)blockIdx.x - __ldg(first + entry);
  {
    const SysDesc& G = sys[list[entry]];
    if (*(volatile const int*)&G.sc->state == ST_DONE) return;  // alike in every CTA
    for (int i = tid; i < (int)(sizeof(SysDesc) / 4); i += nth)
      reinterpret_cast<int*>(&sh.sys)[i] = reinterpret_cast<const int*>(&G)[i];
    for (int i = tid; i < (int)(sizeof(SysScalars) / 4); i += nth)
      reinterpret_cast<int*>(&sh.sc)[i] = __ldcg(reinterpret_cast<const int*>(G.sc) + i);
  }
  if (tid == 0) {
    sh.n_done = 1;
    sh.lo = INT_MAX;
    sh.hi = 0;
    sh.epoch = 0u;
    sh.lost = 0;
    sh.team = C;
    sh.copy = rank % CL_TEAM_COPIES;
    sh.slots = slots + CL_TEAM_WORDS * entry;
    sh.flags = flags;
  }
  if (tid < 12) sh.before[tid / 6][tid % 6] = 0ull;
  for (int i = tid; i < 96; i += nth) sh.words[i / 6][i % 6] = 0ull;
  __syncthreads();
  const SysDesc& S = sh.sys;
  const int n = S.n_nodes, n_tiles = S.n_tiles, n_ow = WARPS * n_tiles, n_vw = (n_ow + 255) / 256;
  const int T0 = n_tiles * rank / C, T1 = n_tiles * (rank + 1) / C, nt = T1 - T0;
  const int n0 = min(n, TILE * T0), n1 = min(n, TILE * T1), nown = n1 - n0;
  const int j0 = __ldg(S.row_ptr + n0), nb = __ldg(S.row_ptr + n1) - j0;
  {
    int lo = INT_MAX, hi = 0;
    for (int i = n0 + tid; i < n1; i += nth) {
      lo = min(lo, __ldg(S.col + __ldg(S.row_ptr + i)));
      hi = max(hi, __ldg(S.col + __ldg(S.row_ptr + i + 1) - 1) + 1);
    }
    if (hi > lo) {
      atomicMin(&sh.lo, lo);
      atomicMax(&sh.hi, hi);
    }
  }
  __syncthreads();
  const int lo = nown ? sh.lo : 0, wn = nown ? sh.hi - sh.lo : 0;
  // shared memory (team64_smem_bytes is the same sum)
  double* P = reinterpret_cast<double*>(cl_smem);      // the window's p
  double* Q = P + 6 * (size_t)wn;                      // own rows
  double* R = Q + 6 * (size_t)nown;
  double* X = R + 6 * (size_t)nown;
  double* Z = X + 6 * (size_t)nown;
  double* Ms = Z + 6 * (size_t)nown;
  double* Ks = Ms + (JAC ? 6 : 36) * (size_t)nown;
  const size_t used = (size_t)((unsigned char*)Ks - cl_smem) + 4 * ((size_t)nb + nown + 2);
  const bool k_in = used + 288 * (size_t)nb <= (size_t)smem_bytes;
  int* slot = reinterpret_cast<int*>(Ks + (k_in ? 36 * (size_t)nb : 0));  // 6 x window slot
  int* rp = slot + nb;
  const double* Mg = S.M64 + (JAC ? 6 : 36) * (size_t)n0;
  for (int i = tid; i < (JAC ? 6 : 36) * nown; i += nth) Ms[i] = __ldg(Mg + i);
  const double* Kg = S.K64 + 36 * (size_t)j0;
  if (k_in)
    for (int i = tid; i < 18 * nb; i += nth)
      reinterpret_cast<double2*>(Ks)[i] = __ldg(reinterpret_cast<const double2*>(Kg) + i);
  const double* K = k_in ? Ks : Kg;
  for (int i = tid; i < nb; i += nth) slot[i] = 6 * (__ldg(S.col + j0 + i) - lo);
  for (int i = tid; i <= nown; i += nth) rp[i] = __ldg(S.row_ptr + n0 + i) - j0;
  for (int i = tid; i < 6 * nown; i += nth) {
    R[i] = __ldcg((const double*)S.r + 6 * (size_t)n0 + i);
    X[i] = __ldcg(S.x + 6 * (size_t)n0 + i);
  }
  {
    const double* pg = (const double*)(sh.sc.parity ? S.p1 : S.p0) + 6 * (size_t)lo;
    for (int i = tid; i < 6 * wn; i += nth) P[i] = __ldcg(pg + i);
  }
  bool z_alt = false;  // z is in S.zb, not S.z
  // this lane's row within a group of five nodes
  const int ln = lane / 6, rr = lane % 6;
  __syncthreads();

  int state = sh.sc.state;
  for (int step = 0; step < max_steps && state != ST_DONE && !sh.lost; ++step) {
    if (state == ST_PCG) {
      const bool first = sh.sc.inner == 0;
      const double beta = first ? 0.0 : sh.sc.beta;
      const double* z = (const double*)(z_alt ? S.zb : S.z) + 6 * (size_t)lo;
      for (int i = tid; i < 6 * wn; i += 4 * nth) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * nth < 6 * wn) v[u] = __ldcg(z + i + u * nth);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * nth < 6 * wn)
            P[i + u * nth] = fma(beta, first ? v[u] : P[i + u * nth], v[u]);
      }
      __syncthreads();
      for (int g = w; g < WARPS * nt; g += W) {
        const int l = NODES_PER_WARP * g + ln;
        double part = 0.0;
        if (lane < 6 * NODES_PER_WARP && l < nown) {
          double acc = 0.0;
          const int e = rp[l + 1];
          for (int j = rp[l]; j < e; ++j) {
            const double2* kv = reinterpret_cast<const double2*>(K + 36 * (size_t)j + 6 * rr);
            const double2* pv = reinterpret_cast<const double2*>(P + slot[j]);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const double2 a = kv[q], b = pv[q];
              acc = fma(a.x, b.x, acc);
              acc = fma(a.y, b.y, acc);
            }
          }
          Q[6 * l + rr] = acc;
          part = P[6 * (n0 - lo + l) + rr] * acc;
        }
        part = warp_sum(part);
        if (lane == 0) S.part_a[WARPS * T0 + g] = part;
      }
      team_sync(sh, true);
      for (int v = w; v < n_vw; v += W) {
        const double a = vwarp_sum(S.part_a, v, n_ow, lane);
        if (lane == 0) sh.red[v] = a;
      }
      __syncthreads();
      if (tid == 0)
        finish_a_scalars(&sh.sc, ST_PCG, total_a(sh.red, n_vw, S.n_chunks), 0.0, &sh.n_done);
      __syncthreads();
      if (sh.sc.state == ST_DONE) {
        state = ST_DONE;
        break;
      }
    } else {  // INIT, RESID
      residual_phase(S, state, WARPS * T0, WARPS * T1, n1, n_ow);
      team_sync(sh, true);
      for (int v = w; v < 2 * n_vw; v += W) {
        const bool second = v >= n_vw;
        const int k = second ? v - n_vw : v;
        const double a = vwarp_sum(S.part_a + (second ? n_ow : 0), k, n_ow, lane);
        if (lane == 0) sh.red[(second ? CL_MAX_VWARPS : 0) + k] = a;
      }
      __syncthreads();
      if (tid == 0) residual_scalars(sh, state, n_vw, S.n_chunks);
      __syncthreads();
      const double rr64 = sh.sc.rr64;
      if (!(f64_finite(rr64) && !(rr64 <= sh.sc.rtol2 * sh.sc.ff))) {
        __syncthreads();
        if (tid == 0) finish_b(&sh.sc, state, 0.0, 0.0, &sh.n_done, false);
        __syncthreads();
        state = sh.sc.state;
        continue;
      }
    }
    const double alpha = sh.sc.alpha, ua = alpha * sh.sc.scale;
    const double inv_norm = state == ST_PCG ? 0.0 : 1.0 / ::sqrt(sh.sc.rr64);
    double* zn = (double*)(z_alt ? S.z : S.zb) + 6 * (size_t)n0;
    for (int g = w; g < WARPS * nt; g += W) {
      const int l = NODES_PER_WARP * g + ln, i = 6 * l + rr;
      const bool act = lane < 6 * NODES_PER_WARP && l < nown;
      if (act) {
        if (state == ST_PCG) {
          X[i] = fma(ua, P[6 * (n0 - lo) + i], X[i]);
          R[i] = fma(-alpha, Q[i], R[i]);
        } else {
          R[i] = __ldcg(S.r64 + 6 * (size_t)n0 + i) * inv_norm;
        }
      }
      __syncwarp();
      if (act) {
        double z;
        if (JAC) {
          z = Ms[i] * R[i];
        } else {
          z = 0.0;
#pragma unroll
          for (int c = 0; c < 6; ++c) z = fma(Ms[36 * l + 6 * rr + c], R[6 * l + c], z);
        }
        Z[i] = z;
        zn[i] = z;
      }
    }
    __syncthreads();
    // r^T z and r^T r of a tile: a warp each
    for (int k = w; k < 2 * nt; k += W) {
      const int l = TILE * (k >> 1) + lane;
      double v = 0.0;
      if (lane < TILE && l < nown) {
        const double* b = k & 1 ? R : Z;
#pragma unroll
        for (int a = 0; a < 6; ++a) v = fma(R[6 * l + a], b[6 * l + a], v);
      }
      v = warp_sum(v);
      if (lane == 0) S.part_b[(k & 1) * n_tiles + T0 + (k >> 1)] = v;
    }
    z_alt = !z_alt;
    team_sync(sh, true);
    if (w < 2) {
      const double v = total_b(S.part_b + (size_t)w * n_tiles, n_tiles, S.n_chunks, lane,
                               sh.red + CL_MAX_VWARPS + CL_MAX_CHUNKS * w);
      if (lane == 0) (w == 0 ? sh.ex_rz : sh.ex_rr) = v;
    }
    __syncthreads();
    if (tid == 0) finish_b(&sh.sc, state, sh.ex_rz, sh.ex_rr, &sh.n_done, false);
    __syncthreads();
    state = sh.sc.state;
    if (state == ST_RESID) {  // the other CTAs read x next
      for (int i = tid; i < 6 * nown; i += nth) S.x[6 * (size_t)n0 + i] = X[i];
      team_sync(sh, true);
    }
  }
  if (sh.lost) return;  // a barrier gave up: the run has failed
  if (state == ST_PCG || state == ST_DONE)
    for (int i = tid; i < 6 * nown; i += nth) S.x[6 * (size_t)n0 + i] = X[i];
  if (state == ST_PCG) {
    double* pg = (double*)(sh.sc.parity ? S.p1 : S.p0) + 6 * (size_t)n0;
    for (int i = tid; i < 6 * nown; i += nth) {
      ((double*)S.r)[6 * (size_t)n0 + i] = R[i];
      ((double*)S.z)[6 * (size_t)n0 + i] = Z[i];
      pg[i] = P[6 * (n0 - lo) + i];
    }
  }
  if (rank == 0 && tid == 0) {
    *S.sc = sh.sc;
    if (state == ST_DONE) atomicSub(flags, 1);
  }
}

}  // namespace

// Shared memory of one CTA before resident K (the kernel carves the same sum).
size_t cluster_smem_bytes(const ClusterShare& c, int precond, bool m_tm, bool team) {
  auto a = [](size_t b) { return (b + 15) & ~(size_t)15; };
  const size_t own = (size_t)TILE * c.own_tiles, nt = c.own_tiles;
  size_t s = team ? 0 : 3 * 16 * (size_t)c.n_tiles;
  if (precond == SSO_TWO_LEVEL)
    s += 16 * 8 * COARSE_ROW_BLOCKS + 2 * a(8 * COARSE_MAX_N) + a(4 * (COARSE_MAX_AGG + 1)) +
         16 * (size_t)c.window + 16 * (size_t)c.members;
  s += (team ? 1 : 2) * a(24 * (size_t)c.window) + 3 * a(24 * own) + 8 * WARPS * nt + 32 * nt;
  if (!m_tm) s += (precond == SSO_JACOBI ? 768 : 3072) * nt;
  s += 64 * (size_t)c.positions + a(4 * (nt + 1));
  return s + 128;
}

// Columns of tensor memory for a CTA of `smem` bytes of dynamic shared memory:
// more for larger CTAs, by thresholds that keep the sum over any CTAs of this
// kernel that fit one SM's shared memory together within its 512 columns
// (171.5 + 57 KB and 113 + 113 + 57 KB exceed the SM's 228 KB), so that no
// allocation ever waits for another.
static int cluster_tm_cols(int smem) {
  const int all = smem + (int)sizeof(ClShared) + 1024;
  return all >= 175616 ? 512 : all >= 115712 ? 256 : all >= 58368 ? 128 : 0;
}
int cluster_tm_positions(int smem, int own_tiles, int warps, bool m_tm) {
  const int share = cluster_tm_cols(smem) / ((warps + 3) / 4);
  const int m = m_tm ? M32_PACK * ((own_tiles + warps - 1) / warps) : 0;
  return share < m ? -1 : (share - m) / 36;
}

// Sets the kernels' attributes on the current device, once (they are the
// device's own); the dynamic shared memory of a CTA there.
static cudaError_t cluster_attributes(int* max_smem) {
  static std::mutex mu;
  static std::map<int, int> limits;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  int& limit = limits[dev];
  if (!limit) {
    const void* fns[11] = {(const void*)team64_kernel<false>, (const void*)team64_kernel<true>,
                          (const void*)cluster_cg_kernel<false, false, 0, false>,
                          (const void*)cluster_cg_kernel<false, true, 0, false>,
                          (const void*)cluster_cg_kernel<true, false, 0, false>,
                          (const void*)cluster_cg_kernel<false, false, CL_KREG, false>,
                          (const void*)cluster_cg_kernel<false, true, CL_KREG, false>,
                          (const void*)cluster_cg_kernel<false, false, 0, true>,
                          (const void*)cluster_cg_kernel<false, true, 0, true>,
                          (const void*)cluster_cg_kernel<false, false, CL_KREG, true>,
                          (const void*)cluster_cg_kernel<false, true, CL_KREG, true>};
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    int room = optin;
    for (const void* f : fns) {
      cudaFuncAttributes at;
      if ((e = cudaFuncGetAttributes(&at, f)) != cudaSuccess) return e;
      room = std::min(room, optin - (int)at.sharedSizeBytes);
    }
    room &= ~15;
    for (const void* f : fns) {
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
    limit = room;
  }
  *max_smem = limit;
  return cudaSuccess;
}

static void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int clusters, int size,
                           int threads, int smem, cudaStream_t s) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)(clusters * size));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)size;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

cudaError_t cluster_limits(int* max_smem, int slots[CL_SIZES], int* max_ctas) {
  cudaError_t e = cluster_attributes(max_smem);
  int dev = 0, coop = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *max_ctas = coop ? sms : 0;
  for (int k = 0; k < CL_SIZES && e == cudaSuccess; ++k) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, 1, cl_size_of(k), CL_MAX_THREADS, *max_smem, nullptr);
    slots[k] = 0;
    e = cudaOccupancyMaxActiveClusters(&slots[k], cluster_cg_kernel<false, false, 0, false>, &cfg);
  }
  return e;
}

cudaError_t launch_cluster_pack(const SysDesc* sys, const int* list, int n_list, int max_nodes,
                                cudaStream_t s) {
  if (n_list <= 0) return cudaSuccess;
  if (n_list > 65535) return cudaErrorInvalidValue;
  const int tiles = (max_nodes + TILE - 1) / TILE;
  cluster_pack_kernel<<<dim3((unsigned)((tiles + 3) / 4), (unsigned)n_list), 128, 0, s>>>(sys,
                                                                                         list);
  return cudaGetLastError();
}

cudaError_t launch_cluster_cg(const SysDesc* sys, const int* list, int n_list, int size,
                              int threads, int smem, int precond, bool m_tm, bool team,
                              unsigned long long* slots, int* flags, int max_steps,
                              cudaStream_t s) {
  if (n_list <= 0) return cudaSuccess;
  int limit = 0;
  cudaError_t e = cluster_attributes(&limit);
  if (e != cudaSuccess) return e;
  if (smem > limit) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cluster_config(cfg, at, n_list, size, threads, smem, s);
  const int cols = cluster_tm_cols(smem);
  auto run = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, sys, list, flags, max_steps, smem, cols, (int)m_tm,
                              team ? size : 0, slots);
  };
  if (team) {
    if (precond == SSO_TWO_LEVEL || n_list > CL_MAX_TEAMS) return cudaErrorInvalidValue;
    e = cudaMemsetAsync(slots, 0, 8 * (size_t)CL_TEAM_WORDS * n_list, s);
    if (e != cudaSuccess) return e;
    at[0] = cudaLaunchAttribute{};
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    if (threads <= CL_REG_THREADS)
      return precond == SSO_JACOBI ? run(cluster_cg_kernel<false, true, CL_KREG, true>)
                                   : run(cluster_cg_kernel<false, false, CL_KREG, true>);
    return precond == SSO_JACOBI ? run(cluster_cg_kernel<false, true, 0, true>)
                                 : run(cluster_cg_kernel<false, false, 0, true>);
  }
  if (precond == SSO_TWO_LEVEL) return run(cluster_cg_kernel<true, false, 0, false>);
  if (threads <= CL_REG_THREADS)
    return precond == SSO_JACOBI ? run(cluster_cg_kernel<false, true, CL_KREG, false>)
                                 : run(cluster_cg_kernel<false, false, CL_KREG, false>);
  return precond == SSO_JACOBI ? run(cluster_cg_kernel<false, true, 0, false>)
                               : run(cluster_cg_kernel<false, false, 0, false>);
}

// The shared memory of a CTA of the FP64 engine without K, and all of K's.
size_t team64_smem_bytes(const ClusterShare& c, bool jacobi, size_t* k_bytes) {
  const size_t own = (size_t)TILE * c.own_tiles;
  *k_bytes = 288 * (size_t)c.members;
  return 48 * (size_t)c.window + 48 * 4 * own + 8 * (jacobi ? 6 : 36) * own +
         4 * ((size_t)c.members + own + 2);
}

cudaError_t launch_team64(const SysDesc* sys, const int* list, int n_list, int ctas, int threads,
                          int smem, bool jacobi, unsigned long long* slots, int* flags,
                          int max_steps, cudaStream_t s) {
  if (n_list <= 0) return cudaSuccess;
  int limit = 0;
  cudaError_t e = cluster_attributes(&limit);
  if (e != cudaSuccess) return e;
  if (smem > limit || n_list > CL_MAX_TEAMS || threads > TEAM64_THREADS)
    return cudaErrorInvalidValue;
  e = cudaMemsetAsync(slots, 0, 8 * (size_t)CL_TEAM_WORDS * n_list, s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cluster_config(cfg, at, 1, ctas, threads, smem, s);
  at[0] = cudaLaunchAttribute{};
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  return cudaLaunchKernelEx(&cfg, jacobi ? team64_kernel<true> : team64_kernel<false>, sys, list,
                            flags, n_list, max_steps, smem, slots);
}

}  // namespace sso
